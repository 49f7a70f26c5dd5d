// energy.cu -- full energies of production bcc configurations (Sec. 3, Eq. 1): every few exchange intervals
// the sum over all bonds replaces the walkers' running energies, so that rounding never builds up.
#include "walker_common.cuh"

namespace rewl {

constexpr int kEnergyThreads = 512;

// E = -sum over the forward half of every shell of J S_i.S_n of one configuration, by one CTA.
//
// Float-float throughout: with nearly parallel spins every site has nearly the same field, so plain FP32
// rounding errors would add up coherently over the sites.  The order of the sum is the one of a walker of
// `nt` threads whose thread t adds the sites t, t + nt, ... in turn: the sites' terms are independent, so all
// threads of the CTA compute them, a tile of kEnergyThreads sites at a time, and its first nt threads add
// them up from shared memory while the others are at the next tile.
//
// What bounds it: the arithmetic (25 bonds per site at four shells, about 48 instructions each: decode
// 14, three float-float products and sums 30).  Inside the walker kernels, by the walker's own 128
// threads with run-time shell offsets, it took 3.9 ms at bcc L = 32, 512 walkers; here 1.8 ms (bcc L = 16, 2 shells, 64 walkers:
// 72 -> 25 us).  Two CTAs of 512 threads per SM (64 registers): 512 walkers are two waves.
template <int NSH>
__device__ __forceinline__ void energy_update(const WalkerArgs& a, const int slot, const int nt) {
  constexpr ShellTable T = make_shells(NSH);
  __shared__ float term[2][6][kEnergyThreads];
  __shared__ double red[4];
  const int tid = threadIdx.x;
  const int N = a.geo.N, L = a.geo.L;
  const int twoL = 2 * L, LL = L * L;
  const auto lat = GlobalLattice<false>::of(a.st.spins, a.st.perm[slot], N);
  float Jsh[4];
#pragma unroll
  for (int s = 0; s < 4; ++s) Jsh[s] = a.geo.Jsh_f[s];
  float hi = 0.0f, lo = 0.0f;
  const int tiles = (N + kEnergyThreads - 1) / kEnergyThreads;
  for (int tile = 0; tile < tiles; ++tile) {
    const int i = tile * kEnergyThreads + tid;
    float (*out)[kEnergyThreads] = term[tile & 1];
    if (i < N) {
      int X, Y, Z;
      bcc_coords(i, L, a.geo.divL, X, Y, Z);
      int xw[7], yw[7], zw[7];
#pragma unroll
      for (int d = -3; d <= 3; ++d) {
        int x = X + d, y = Y + d, z = Z + d;
        x += (x < 0) ? twoL : 0;
        x -= (x >= twoL) ? twoL : 0;
        y += (y < 0) ? twoL : 0;
        y -= (y >= twoL) ? twoL : 0;
        z += (z < 0) ? twoL : 0;
        z -= (z >= twoL) ? twoL : 0;
        xw[d + 3] = x;
        yw[d + 3] = L * y;
        zw[d + 3] = LL * z;
      }
      // site = x' + L y' + L^2 z' - s' (L + L^2), s' the neighbour's sublattice
      const int s = X & 1;
      const int par_same = s * (L + LL), par_flip = (s ^ 1) * (L + LL);
      float hxh = 0.f, hxl = 0.f, hyh = 0.f, hyl = 0.f, hzh = 0.f, hzl = 0.f;
      int j0 = 0;
#pragma unroll
      for (int sh = 0; sh < NSH; ++sh) {
        const int count = sh == 0 ? 8 : (sh == 1 ? 6 : (sh == 2 ? 12 : 24));
        const float J = Jsh[sh];
#pragma unroll
        for (int k = 0; k < count / 2; ++k) {
          const int j = j0 + k;
          const int n = xw[T.dx[j] + 3] + yw[T.dy[j] + 3] + zw[T.dz[j] + 3] - ((T.dx[j] & 1) ? par_flip : par_same);
          float vx, vy, vz;
          lat.get(n, vx, vy, vz);
          float p, pe;
          two_prod(J, vx, p, pe);
          ff_add(hxh, hxl, p, pe);
          two_prod(J, vy, p, pe);
          ff_add(hyh, hyl, p, pe);
          two_prod(J, vz, p, pe);
          ff_add(hzh, hzl, p, pe);
        }
        j0 += count;
      }
      float six, siy, siz, p, pe;
      lat.get(i, six, siy, siz);
      two_prod(six, hxh, p, pe);
      out[0][tid] = p;
      out[1][tid] = fmaf(six, hxl, pe);
      two_prod(siy, hyh, p, pe);
      out[2][tid] = p;
      out[3][tid] = fmaf(siy, hyl, pe);
      two_prod(siz, hzh, p, pe);
      out[4][tid] = p;
      out[5][tid] = fmaf(siz, hzl, pe);
    }
    // the tile's terms are complete; the buffer of the tile before is free (its sums were added before
    // this barrier)
    __syncthreads();
    if (tid < nt)
      for (int k = tid; k < kEnergyThreads && tile * kEnergyThreads + k < N; k += nt) {
        ff_add(hi, lo, out[0][k], out[1][k]);
        ff_add(hi, lo, out[2][k], out[3][k]);
        ff_add(hi, lo, out[4][k], out[5][k]);
      }
  }
  if (tid < nt) {                          // whole warps: nt is 64 or 128
    double v = (double)hi + (double)lo;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFullMask, v, o);
    if ((tid & 31) == 0) red[tid >> 5] = v;
  }
  __syncthreads();
  if (tid == 0) {
    double tot = 0.0;
    for (int w = 0; w < (nt >> 5); ++w) tot += red[w];
    const int wlo = a.win.starts[global_slot(a.st, slot) / a.win.m];
    replace_energy(a, slot, wlo, -(double)a.geo.energy_weight * tot);
  }
}

template <int NSH>
__global__ void __launch_bounds__(kEnergyThreads, 2) energy_update_kernel(const WalkerArgs a) {
  energy_update<NSH>(a, blockIdx.x, kWalkerThreads);
}

template <int NSH>
__global__ void __launch_bounds__(kEnergyThreads, 2)
    energy_update_batch_kernel(const WalkerArgs* __restrict__ jobs, const int2* __restrict__ items, int walk_threads) {
  const int2 it = items[blockIdx.x];
  energy_update<NSH>(jobs[it.x], it.y, walk_threads);
}

cudaError_t launch_energy_update(const WalkerArgs& a, int n_slots, cudaStream_t stream) {
  static_assert(kWalkerThreads <= 128 && kEnergyThreads % kWalkerThreads == 0, "order of the sum");
  switch (a.geo.n_shells) {
    case 1: energy_update_kernel<1><<<n_slots, kEnergyThreads, 0, stream>>>(a); break;
    case 2: energy_update_kernel<2><<<n_slots, kEnergyThreads, 0, stream>>>(a); break;
    case 3: energy_update_kernel<3><<<n_slots, kEnergyThreads, 0, stream>>>(a); break;
    case 4: energy_update_kernel<4><<<n_slots, kEnergyThreads, 0, stream>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_energy_update_batch(const WalkerArgs* jobs, const int2* items, int n_items, int n_shells,
                                       int walk_threads, cudaStream_t stream) {
  if (walk_threads < 32 || walk_threads > 128 || kEnergyThreads % walk_threads != 0) return cudaErrorInvalidValue;
  switch (n_shells) {
    case 1: energy_update_batch_kernel<1><<<n_items, kEnergyThreads, 0, stream>>>(jobs, items, walk_threads); break;
    case 2: energy_update_batch_kernel<2><<<n_items, kEnergyThreads, 0, stream>>>(jobs, items, walk_threads); break;
    case 3: energy_update_batch_kernel<3><<<n_items, kEnergyThreads, 0, stream>>>(jobs, items, walk_threads); break;
    case 4: energy_update_batch_kernel<4><<<n_items, kEnergyThreads, 0, stream>>>(jobs, items, walk_threads); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace rewl
