// walker.cu -- the persistent Wang-Landau walker kernel (Sec. 4.2, Eq. 4; trial move Sec. 4.4).
//
// One CTA per walker slot (window k, walker a).  The CTA stages the slot's ln g / H tables and,
// when it fits, the whole spin lattice of its configuration in shared memory; warp 0 then runs
// `moves` trial moves.  The walk is a strict Markov chain, so it is advanced in speculative
// batches of K = 32 / G moves, G lanes per move:
//   - the local field h_i = sum_j J_ij S_j as a G-lane reduction, dE = -(S'-S).h, and a bitmask of the
//     earlier moves in the batch whose site is the same site or one of its neighbours;
//   - the moves are resolved in order: a move is re-evaluated if an earlier accepted move in the
//     batch touched its neighbourhood, then accepted with min[1, g(E)/g(E')] (reject outside the
//     window), and ln g += ln f, H += 1 at the resulting state.
// The result is the sequential walk exactly: in trajectory mode (FP64, no contraction) it
// reproduces the FP64 reference walk bit for bit.
//
// Production mode keeps FP64 out of the per-move chain (FP64 has a 64-cycle latency on this
// GPU): spins and dE in FP32; the energy as int64 in 2^-32 bin units (bin = high word); ln g,
// ln f and ln u as int64 in 2^-40 units, so ln g accumulates ln f increments exactly.  Its draws come
// from a second warp, and its moves are resolved per accepted move (walk_units).
#include <cstdio>

#include "walker_common.cuh"

namespace rewl {

// Trajectory, warp 0: the walk.  All state below is warp-uniform unless named per-lane.
template <class Lat>
__device__ void walk(const WalkerArgs& a, int slot, int wlo, double* lng_s, uint32_t* H_s, const uint32_t* off_s,
                     const double* J_s, const Lat& lat) {
  const int lane = threadIdx.x & 31;
  const int G = a.G, K = 32 / G;
  const int g = lane / G, sub = lane % G;
  const unsigned gmask = (G == 32) ? kFullMask : (((1u << G) - 1u) << (g * G));
  const int N = a.geo.N, W = a.win.W;
  const bool bcc = a.geo.kind == 0;
  const bool init = a.init != 0;
  const uint2 key = make_uint2((uint32_t)global_slot(a.st, slot), a.key1);

  // ---- uniform walker state ----
  double E = a.st.E[slot];
  int bcur = a.st.bin[slot];
  const double lnf = a.st.lnf[slot];
  const bool frozen = !(lnf >= a.lnf_final);
  if (!init && (unsigned)(bcur - wlo) >= (unsigned)W) {
    if (lane == 0) atomicExch(a.st.ctrl + 0, kErrOutOfWindow);
    return;
  }
  // initial drive: target = window centre
  const double c_traj = __dadd_rn(a.win.e_min, __dmul_rn(__dadd_rn((double)wlo, __dmul_rn((double)W, 0.5)), a.win.dE));

  double lng_cur = 0.0;
  uint32_t h_cur = 0;
  if (!init) {
    lng_cur = lng_s[bcur - wlo];
    h_cur = H_s[bcur - wlo];
  }
  long long t = init ? 0 : a.st.steps[slot];
  long long remaining = init ? a.init_cap : a.moves;
  long long n_acc = 0, n_rec = 0;
  bool done = false;

  while (remaining > 0 && !done) {
    const int nvalid = (int)(remaining < (long long)K ? remaining : (long long)K);

    // ---------------- phase A: K moves in parallel ----------------
    int site, X = 0, Y = 0, Z = 0;
    double nx, ny, nz, u;
    draw_traj(key, (unsigned long long)(t + g), init, N, site, u, nx, ny, nz);
    if (bcc) bcc_coords(site, a.geo.L, a.geo.divL, X, Y, Z);
    const double dE = delta_energy<true>(a, off_s, J_s, lat, site, X, Y, Z, nx, ny, nz, sub, G, kFullMask);

    // conflicts with earlier moves of the batch: same site or a neighbour of it
    uint32_t conf = 0;
    if (bcc) {
      const uint32_t packed = (uint32_t)X | ((uint32_t)Y << 10) | ((uint32_t)Z << 20);
      const int L = a.geo.L, twoL = 2 * a.geo.L;
      for (int j = 0; j + 1 < K; ++j) {
        const uint32_t pj = __shfl_sync(kFullMask, packed, j * G);
        if (j < g) {
          int ex = X - (int)(pj & 1023u), ey = Y - (int)((pj >> 10) & 1023u), ez = Z - (int)(pj >> 20);
          ex -= (ex > L) ? twoL : 0;
          ex += (ex <= -L) ? twoL : 0;
          ey -= (ey > L) ? twoL : 0;
          ey += (ey <= -L) ? twoL : 0;
          ez -= (ez > L) ? twoL : 0;
          ez += (ez <= -L) ? twoL : 0;
          if (ex * ex + ey * ey + ez * ez <= a.geo.r2max) conf |= 1u << j;
        }
      }
    } else {
      const int z = a.geo.z;
      for (int j = 0; j + 1 < K; ++j) {
        const int sj = __shfl_sync(kFullMask, site, j * G);
        bool hit = false;
        if (j < g) {
          if (sj == site) hit = true;
          for (int s = sub; s < z; s += G)
            if (__ldg(a.geo.tab_nbr + (size_t)s * N + site) == sj) hit = true;
        }
        const uint32_t bal = __ballot_sync(kFullMask, hit);
        if (j < g && (bal & gmask)) conf |= 1u << j;
      }
    }

    // ---------------- phase B: resolve in order ----------------
    uint32_t acc_mask = 0;
    int k = 0;
    for (; k < nvalid; ++k) {
      if (init && (unsigned)(bcur - wlo) < (unsigned)W) {
        done = true;
        break;
      }
      const int src = k * G;
      const uint32_t cm = __shfl_sync(kFullMask, conf, src);
      bool acc;
      double dE_k = __shfl_sync(kFullMask, dE, src);
      const double u_k = __shfl_sync(kFullMask, u, src);
      if (cm & acc_mask) {
        double dn = 0.0;
        if (g == k) dn = delta_energy<true>(a, off_s, J_s, lat, site, X, Y, Z, nx, ny, nz, sub, G, gmask);
        dE_k = __shfl_sync(kFullMask, dn, src);
        ++n_rec;
      }
      const double Ep = __dadd_rn(E, dE_k);
      if (init) {
        acc = fabs(__dsub_rn(Ep, c_traj)) <= fabs(__dsub_rn(E, c_traj));
        if (acc) {
          E = Ep;
          bcur = bin_fp64(E, a.win);
        }
      } else {
        const int bp = bin_fp64(Ep, a.win);
        const int rel = bp - wlo;
        const bool inw = (unsigned)rel < (unsigned)W;
        acc = false;
        if (inw) {
          const double lngp = (bp == bcur) ? lng_cur : lng_s[rel];
          const double d = __dsub_rn(lng_cur, lngp);
          acc = (d >= 0.0) || (u_k < exp_fp64(d, a.ex));
          if (acc) {
            if (bp != bcur) {
              lng_s[bcur - wlo] = lng_cur;
              H_s[bcur - wlo] = h_cur;
              lng_cur = lngp;
              h_cur = H_s[rel];
              bcur = bp;
            }
            E = Ep;
          }
        }
      }
      if (acc) {
        acc_mask |= 1u << k;
        ++n_acc;
        if (lane == src) lat.set(site, nx, ny, nz);
        __syncwarp();
      }
      if (!init && !frozen) {
        lng_cur = __dadd_rn(lng_cur, lnf);
        ++h_cur;
      }
    }
    t += k;
    remaining -= k;
    __syncwarp();
  }
  if (init && !done && (unsigned)(bcur - wlo) < (unsigned)W) done = true;

  if (lane == 0) {
    a.st.E[slot] = E;
    a.st.bin[slot] = bcur;
    if (init) {
      a.st.init_moves[slot] = t;
      if (!done) atomicExch(a.st.ctrl + 0, kErrInitCap);
    } else {
      lng_s[bcur - wlo] = lng_cur;
      H_s[bcur - wlo] = h_cur;
      a.st.steps[slot] = t;
      a.st.accepts[slot] += n_acc;
      a.st.recomputes[slot] += n_rec;
    }
  }
  __syncwarp();
}

// Production draws of 32 trial moves, prepared by warp 1 a lane per move while warp 0 walks the 32 before.
// (Small enough for the 1 KB that the kernel's shared memory leaves beside the tables and the lattice.)
struct DrawBatch {
  float2 code[32];       // octahedral code of the proposed spin
  uint32_t place[32];    // bcc: half-unit coordinates X | Y << 10 | Z << 20; else the site
  float ln_u[32];
  uint32_t conf[32];     // earlier moves of the batch of K on the same site or a neighbour of it
  long long last;        // chunk in which the walk ended
};
constexpr int kBarDrawn = 1, kBarTaken = 2;   // named barriers of warps 0 and 1
__device__ __forceinline__ void pair_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void pair_arrive(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }

// Warp 1: chunk c holds moves 32 c .. 32 c + 31 of this call.  A chunk is drawn in registers while the one
// before is walked, and handed over when that one has been taken, unless the walk ended in it.
__device__ __forceinline__ void draw_moves(const WalkerArgs& a, int slot, DrawBatch& buf) {
  const int lane = threadIdx.x & 31;
  const int N = a.geo.N, K = 32 / a.G;
  const bool bcc = a.geo.kind == 0, init = a.init != 0;
  const uint2 key = make_uint2((uint32_t)global_slot(a.st, slot), a.key1);
  const unsigned long long t0 = init ? 0ULL : (unsigned long long)a.st.steps[slot];
  const int first = lane / K * K;             // the batch's first move
  for (long long c = 0;; ++c) {
    int site;
    float ln_u, nx, ny, nz;
    draw_prod(key, t0 + 32ULL * (unsigned long long)c + (unsigned)lane, init, N, site, ln_u, nx, ny, nz);
    const float2 code = oct_encode(nx, ny, nz);
    uint32_t conf = 0, place = (uint32_t)site;
    if (bcc) {
      int X, Y, Z;
      bcc_coords(site, a.geo.L, a.geo.divL, X, Y, Z);
      place = (uint32_t)X | ((uint32_t)Y << 10) | ((uint32_t)Z << 20);
      const int L = a.geo.L, twoL = 2 * a.geo.L;
      for (int j = 0; j + 1 < K; ++j) {
        const uint32_t pj = __shfl_sync(kFullMask, place, first + j);
        int ex = X - (int)(pj & 1023u), ey = Y - (int)((pj >> 10) & 1023u), ez = Z - (int)(pj >> 20);
        ex -= (ex > L) ? twoL : 0;
        ex += (ex <= -L) ? twoL : 0;
        ey -= (ey > L) ? twoL : 0;
        ey += (ey <= -L) ? twoL : 0;
        ez -= (ez > L) ? twoL : 0;
        ez += (ez <= -L) ? twoL : 0;
        conf |= first + j < lane && ex * ex + ey * ey + ez * ez <= a.geo.r2max ? 1u << j : 0u;
      }
    } else {
      for (int s = -1; s < a.geo.z; ++s) {
        const int n = s < 0 ? site : __ldg(a.geo.tab_nbr + (size_t)s * N + site);
        for (int j = 0; j + 1 < K; ++j)
          conf |= n == __shfl_sync(kFullMask, site, first + j) && first + j < lane ? 1u << j : 0u;
      }
    }
    __syncwarp();                             // (the draws may have diverged)
    if (c > 0) {
      pair_sync(kBarTaken);                   // chunk c-1
      if (c > *(volatile long long*)&buf.last) return;
    }
    buf.code[lane] = code;
    buf.place[lane] = place;
    buf.ln_u[lane] = ln_u;
    buf.conf[lane] = conf;
    __syncwarp();
    pair_arrive(kBarDrawn);
  }
}

// dE of a move in 2^-32 bins: its FP64 product with `scale`, rounded to an integer.  FP64 conversions take 93
// cycles each and additions 62, so the FP32 number is widened by its bits and the product rounded by an addition
// that leaves no place for the fraction; |dE| < limit keeps the product below 2^50.
__device__ __forceinline__ long long to_units(float dE, double scale, float limit) {
  if (!(fabsf(dE) < limit)) return __double2ll_rn(__dmul_rn((double)dE, scale));
  const uint32_t b = __float_as_uint(dE), m = b & 0x7fffffffu;
  const double wide = __hiloint2double((int)(m < 0x00800000u ? 0u : (b & 0x80000000u) | ((m >> 3) + 0x38000000u)),
                                       (int)(m < 0x00800000u ? 0u : b << 29));   // (below 2^-126: no unit at all)
  const double magic = 6755399441055744.0;    // 1.5 2^52
  return __double_as_longlong(__dadd_rn(__dmul_rn(wide, scale), magic)) - __double_as_longlong(magic);
}

// The slots of a lane of a group of G on a bcc lattice, slots sub, sub + G, .. of the canonical order, held in
// registers.  The sum of delta_energy, without its loop: the loads of all slots are in flight together.  (The
// initial drive of bcc L = 12, 2 shells, 64 walkers, one lane per move: 640 us with the loop, 470 us so.)
template <int kG, int kSlots, bool kHeld>     // kHeld: in registers, else read from shared memory for each move
struct LaneSlots {
  int dx[kHeld ? kSlots : 1], dy[kHeld ? kSlots : 1], dz[kHeld ? kSlots : 1];
  float J[kHeld ? kSlots : 1];
  const uint32_t* off_at;                       // slot q: off_at[kG q], J_at[kG q] (of kMaxSlotsPerSite entries)
  const float* J_at;
  uint32_t have = 0, opens = 0;               // slots that exist; that begin another shell
  __device__ __forceinline__ LaneSlots(const uint32_t* off_s, const float* J_s, int sub, int z) : off_at(off_s + (sub < z ? sub : 0)), J_at(J_s + sub) {
    uint32_t shell = 0xffffffffu;
#pragma unroll
    for (int q = 0; q < kSlots; ++q) {
      const int j = sub + q * kG;
      const uint32_t o = off_s[j < z ? j : 0];
      if constexpr (kHeld) {
        unpack_offset(o, dx[q], dy[q], dz[q]);
        J[q] = J_s[j < z ? j : 0];
      }
      if (j < z) {
        have |= 1u << q;
        opens |= (o >> 24) != shell ? 1u << q : 0u;
        shell = o >> 24;
      }
    }
  }
  template <class Lat>
  __device__ __forceinline__ float delta(const Lat& lat, int site, uint32_t place, float nx, float ny, float nz, int L) const {
    float vx[kSlots], vy[kSlots], vz[kSlots];
#pragma unroll
    for (int q = 0; q < kSlots; ++q) {
      int ox, oy, oz;
      if constexpr (kHeld) {
        ox = dx[q];
        oy = dy[q];
        oz = dz[q];
      } else {
        unpack_offset(((have >> q) & 1u) != 0u ? off_at[kG * q] : off_at[0], ox, oy, oz);
      }
      lat.get(bcc_offset_site((int)(place & 1023u), (int)((place >> 10) & 1023u), (int)(place >> 20), ox, oy, oz, L), vx[q],
              vy[q], vz[q]);
    }
    float ox, oy, oz;
    lat.get(site, ox, oy, oz);
    float hx = 0.0f, hy = 0.0f, hz = 0.0f, tx = 0.0f, ty = 0.0f, tz = 0.0f, Jc = 0.0f;
#pragma unroll
    for (int q = 0; q < kSlots; ++q) {
      const bool open = ((opens >> q) & 1u) != 0u, add = ((have >> q) & 1u) != 0u;
      const float ux = fmaf(Jc, tx, hx), uy = fmaf(Jc, ty, hy), uz = fmaf(Jc, tz, hz);
      hx = open ? ux : hx;
      hy = open ? uy : hy;
      hz = open ? uz : hz;
      tx = open ? 0.0f : tx;
      ty = open ? 0.0f : ty;
      tz = open ? 0.0f : tz;
      if constexpr (kHeld)
        Jc = open ? J[q] : Jc;
      else
        Jc = open ? J_at[kG * q] : Jc;
      const float sx = tx + vx[q], sy = ty + vy[q], sz = tz + vz[q];
      tx = add ? sx : tx;
      ty = add ? sy : ty;
      tz = add ? sz : tz;
    }
    hx = fmaf(Jc, tx, hx);
    hy = fmaf(Jc, ty, hy);
    hz = fmaf(Jc, tz, hz);
#pragma unroll
    for (int o = kG >> 1; o > 0; o >>= 1) {
      hx += __shfl_xor_sync(kFullMask, hx, o);
      hy += __shfl_xor_sync(kFullMask, hy, o);
      hz += __shfl_xor_sync(kFullMask, hz, o);
    }
    const float dx0 = nx - ox, dy0 = ny - oy, dz0 = nz - oz;
    return -fmaf(dz0, hz, fmaf(dy0, hy, dx0 * hx));
  }
};
template <int kG, bool kHeld>
struct LaneSlots<kG, 0, kHeld> {
  __device__ __forceinline__ LaneSlots(const uint32_t*, const float*, int, int) {}
};

// Production, warp 0: batches of K = 32 / G moves, a group of G lanes per move.  A round finds the first move
// of the batch that is accepted with the walker where it is; the moves before it are rejected.  The moves that
// it touches are evaluated again on the new lattice, all of them at once.  Everything but dE is integer.
// One warp's chain of dependent instructions bounds it (of 227 KB of shared memory 10 KB are in use, and one walker
// cannot be split).  bcc L = 4, 2 shells, G = 8, 8 walkers, the walker that accepts most (2.6 of a batch of 4), per
// batch: 220 cycles for the draws and places, 620 per evaluation (1.4), 400 per round (2.9).  Before, with each
// warp's draws in line, a move resolved at a time and the slots in a loop: 1,400 cycles per move, 6.8 ms per 10^4
// moves; with draws by warp 1 and rounds 4.9 ms; slots in registers 3.8 ms; G known when compiled 2.9 ms.
template <bool kInit, int kG, int kSlots, class Lat>
__device__ __forceinline__ void walk_units(const WalkerArgs& a, int slot, int wlo, long long* lng_s, uint32_t* H_s, const uint32_t* off_s,
                           const float* J_s, const Lat& lat, DrawBatch& buf) {
  const int lane = threadIdx.x & 31;
  const int G = kG ? kG : a.G, K = 32 / G;
  const int g = lane / G, sub = lane % G;
  const int W = a.win.W;
  const bool bcc = kSlots > 0 || a.geo.kind == 0;
  constexpr bool init = kInit;
  long long Efx = a.st.efx[slot];
  int bcur = fx_bin(Efx);
  const long long lnf_fx = a.st.lnf_fx[slot];
  const bool frozen = !((double)lnf_fx * kLngUnit >= a.lnf_final);
  const long long lnf = init || frozen ? 0 : lnf_fx;
  const long long c_fx = ((long long)(2 * wlo + W)) << 31;       // initial drive: target = window centre
  const bool outside = (unsigned)(bcur - wlo) >= (unsigned)W;
  if (!init && outside && lane == 0) atomicExch(a.st.ctrl + 0, kErrOutOfWindow);
  bool done = init ? !outside : outside;      // the walk has ended (or cannot begin)
  const bool bad = !init && outside;
  long long lng0 = init || bad ? 0 : lng_s[bcur - wlo];          // ln g of the bin at the batch's first move
  long long t = init ? 0 : a.st.steps[slot];
  long long remaining = init ? a.init_cap : a.moves;
  long long n_acc = 0, n_rec = 0;
  const long long g_lnf = (long long)g * lnf;
  const float limit = (float)(0x1.0p49 / a.win.dq_scale64);
  const LaneSlots<kG, kSlots, !kInit || kSlots <= 2> slots(off_s, J_s, sub, a.geo.z);

  for (long long c = 0;; ++c) {
    __syncwarp();
    pair_sync(kBarDrawn);
    for (int first = 0; first < 32 && remaining > 0 && !done; first += K) {
      const int nvalid = (int)(remaining < (long long)K ? remaining : (long long)K);
      const uint32_t place = buf.place[first + g];
      const float2 code = buf.code[first + g];
      const uint32_t conf = buf.conf[first + g];
      // accepted if ln g(target) <= ln g(now), or below ln g(now) - ln u
      const long long lu = __float2ll_rn(buf.ln_u[first + g] * 0x1.0p40f);
      const long long margin = g_lnf - (lu < 0 ? lu + 1 : 0);
      float nx, ny, nz;
      oct_decode(code, nx, ny, nz);           // the proposal is the spin its code decodes to
      const int X = (int)(place & 1023u), Y = (int)((place >> 10) & 1023u), Z = (int)(place >> 20);
      const int site = bcc ? bcc_offset_site(X, Y, Z, 0, 0, 0, a.geo.L) : (int)place;
      const uint32_t touched = __reduce_or_sync(kFullMask, conf);   // moves that touch a later one
      long long dq = 0;
      uint32_t acc_mask = 0, again = 0xffffffffu;   // again: which moves to evaluate, by the moves they touch
      int rb = bcur - wlo;                    // bin after this lane's move
      bool live = g < nvalid;
      int k = 0;                              // moves resolved
      while (true) {
        if (again) {
          __syncwarp();
          const bool mine = (conf & again) != 0u || acc_mask == 0u;
          float dE = 0.0f;
          if constexpr (kSlots > 0) {
            // (one lane per move and a lattice in global memory: only the moves in question load their neighbours)
            if (kG > 1 || std::is_same<Lat, CodePlanes>::value || mine) dE = slots.delta(lat, site, place, nx, ny, nz, a.geo.L);
          } else if (G == 1) {
            if (mine) dE = delta_energy<false>(a, off_s, J_s, lat, site, X, Y, Z, nx, ny, nz, 0, 1, 0u);
            __syncwarp();
          } else {
            dE = delta_energy<false>(a, off_s, J_s, lat, site, X, Y, Z, nx, ny, nz, sub, G, kFullMask);
          }
          const long long units = to_units(dE, a.win.dq_scale64, limit);
          dq = mine ? units : dq;
          again = 0u;
        }
        const long long Ep = Efx + dq;
        const int bp = fx_bin(Ep);
        bool acc;
        long long lt = 0;
        if (init) {
          const long long d0 = Efx - c_fx, d1 = Ep - c_fx;
          acc = (d1 < 0 ? -d1 : d1) <= (d0 < 0 ? -d0 : d0);
        } else {
          const int rel = bp - wlo;
          lt = lng_s[min((unsigned)rel, (unsigned)W - 1u)];
          acc = (unsigned)rel < (unsigned)W && (bp == bcur || lt <= lng0 + margin);
        }
        const int e = (int)__reduce_min_sync(kFullMask, live && acc ? (unsigned)g : 32u);
        if (e == 32) break;                   // every move left is rejected
        const int src = e * G;
        const long long Enew = shfl_ll(Ep, src);
        const long long l0 = shfl_ll(lt - g_lnf, src);
        const int bnew = fx_bin(Enew);
        if (lane == src) put_spin(lat, site, nx, ny, nz, code);
        Efx = Enew;
        acc_mask |= 1u << e;
        if (bnew != bcur) {
          if (!init) lng_s[bcur - wlo] = lng0 + (long long)e * lnf;
          lng0 = l0;
          bcur = bnew;
        }
        rb = g >= e ? bcur - wlo : rb;
        live = live && g > e;
        if (init && (unsigned)(bcur - wlo) < (unsigned)W) {
          done = true;
          k = e + 1;
          break;
        }
        if (e + 1 >= nvalid) break;
        if ((touched >> e) & 1u) again = 1u << e;
      }
      if (!done) k = nvalid;
      lng0 += (long long)nvalid * lnf;
      if (!init) {
        if (!frozen && sub == 0 && g < nvalid) atomicAdd(&H_s[rb], 1u);
        n_rec += __popc(__ballot_sync(kFullMask, sub == 0 && g < nvalid && (conf & acc_mask) != 0u));
      }
      n_acc += __popc(acc_mask);
      t += k;
      remaining -= k;
      __syncwarp();
    }
    const bool ended = remaining <= 0 || done;
    if (ended && lane == 0) *(volatile long long*)&buf.last = c;
    __syncwarp();
    pair_arrive(kBarTaken);
    if (ended) break;
  }
  if (lane == 0 && !bad) {
    a.st.efx[slot] = Efx;
    if (init) {
      a.st.init_moves[slot] = t;
      if (!done) atomicExch(a.st.ctrl + 0, kErrInitCap);
    } else {
      lng_s[bcur - wlo] = lng0;
      a.st.steps[slot] = t;
      a.st.accepts[slot] += n_acc;
      a.st.recomputes[slot] += n_rec;
    }
  }
  __syncwarp();
}

// Walkers that an SM is to hold (production): seven in the initial drive, which starts all of them at once, and with
// up to two slots per lane (2048 walkers of bcc L = 4: 586 us per 1000 moves, 733 us with six); four with more slots,
// held in registers (512 walkers of bcc L = 8: 264 us; 311 us with six and the slots in shared memory).
template <bool kTraj, bool kSmem, bool kInit, int kG, int kSlots>
__global__ void __launch_bounds__(kWalkerThreads, kTraj ? 1 : kInit || kSlots <= 2 ? 7 : 4)
    walker_kernel(const WalkerArgs a) {
  using Real = typename Mode<kTraj>::Real;
  using Lng = typename Mode<kTraj>::Lng;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[kWalkerThreads / 32];
  __shared__ DrawBatch draws;               // production

  const int slot = blockIdx.x;
  const int tid = threadIdx.x;
  const int N = a.geo.N, W = a.win.W;
  const int wlo = a.win.starts[global_slot(a.st, slot) / a.win.m];
  const int rep = a.st.perm[slot];

  Lng* lng_s = reinterpret_cast<Lng*>(smem_raw);
  uint32_t* H_s = reinterpret_cast<uint32_t*>(smem_raw + sizeof(Lng) * (size_t)W);
  uint32_t* off_s = reinterpret_cast<uint32_t*>(smem_raw + sizeof(Lng) * (size_t)W + (((size_t)W * 4 + 15) & ~(size_t)15));
  Real* J_s = reinterpret_cast<Real*>(off_s + kMaxSlotsPerSite);
  Real* spin_s = J_s + kMaxSlotsPerSite;

  const auto glat = GlobalLattice<kTraj>::of(a.st.spins, rep, N);
  typename WalkLattice<kTraj, kSmem>::T lat;
  if constexpr (kSmem)
    lat = typename WalkLattice<kTraj, true>::T(spin_s, N);
  else
    lat = glat;

  // stage tables and lattice
  const size_t lbase = (size_t)slot * W;
  if (!a.init) {
    for (int w = tid; w < W; w += blockDim.x) {
      if (kTraj)
        lng_s[w] = (Lng)a.st.lng[lbase + w];
      else
        lng_s[w] = (Lng)a.st.lng_fx[lbase + w];
      H_s[w] = a.st.H[lbase + w];
    }
  }
  for (int j = tid; j < kMaxSlotsPerSite; j += blockDim.x) {
    off_s[j] = a.geo.off[j];
    J_s[j] = kTraj ? (Real)a.geo.Jd[j] : (Real)a.geo.Jf[j];
  }
  if constexpr (kSmem) copy_lattice(lat, glat, N, tid, blockDim.x);
  if (!kTraj && tid == 0) draws.last = 0x7fffffffffffffffLL;
  __syncthreads();

  if constexpr (kTraj) {
    if (tid < 32) walk(a, slot, wlo, lng_s, H_s, off_s, J_s, lat);
  } else {
    if (tid < 32)
      walk_units<kInit, kG, kSlots>(a, slot, wlo, lng_s, H_s, off_s, J_s, lat, draws);
    else if (tid < 64)
      draw_moves(a, slot, draws);
  }
  __syncthreads();

  if constexpr (kSmem) copy_lattice(glat, lat, N, tid, blockDim.x);
  if (!a.init) {
    for (int w = tid; w < W; w += blockDim.x) {
      if (kTraj)
        a.st.lng[lbase + w] = (double)lng_s[w];
      else
        a.st.lng_fx[lbase + w] = (long long)lng_s[w];
      a.st.H[lbase + w] = H_s[w];
    }
  }
  // bcc production lattices: energy_update_kernel, after the walk
  if (a.recompute && !a.init && (kTraj || a.geo.kind != 0)) {
    const double Ef = full_energy<kTraj>(a, off_s, lat, red, threadIdx.x, blockDim.x, 0);
    if (tid == 0) {
      if (kTraj) {
        const double d = fabs(Ef - a.st.E[slot]);
        if (d > a.st.drift[slot]) a.st.drift[slot] = d;
      } else {
        replace_energy(a, slot, wlo, Ef);
      }
    }
  }
}

// FP64 energy of every configuration (one CTA each), spins read from global memory.
template <bool kTraj>
__global__ void __launch_bounds__(kWalkerThreads) energies_kernel(const WalkerArgs a, double* out) {
  __shared__ double red[kWalkerThreads / 32];
  __shared__ uint32_t off_s[kMaxSlotsPerSite];
  for (int j = threadIdx.x; j < kMaxSlotsPerSite; j += blockDim.x) off_s[j] = a.geo.off[j];
  __syncthreads();
  const int N = a.geo.N;
  const auto lat = GlobalLattice<kTraj>::of(a.st.spins, blockIdx.x, N);
  const double e = full_energy<kTraj>(a, off_s, lat, red, threadIdx.x, blockDim.x, 0);
  if (threadIdx.x == 0) out[blockIdx.x] = e;
}

cudaError_t launch_energies(const WalkerArgs& a, int n_replicas, bool traj, double* out, cudaStream_t stream) {
  if (traj)
    energies_kernel<true><<<n_replicas, kWalkerThreads, 0, stream>>>(a, out);
  else
    energies_kernel<false><<<n_replicas, kWalkerThreads, 0, stream>>>(a, out);
  return cudaGetLastError();
}

// The neighbour table exactly as the walker kernel computes it: [z][N] indices and couplings.
__global__ void neighbour_dump_kernel(const Geometry g, int32_t* nbr, double* J) {
  const long long total = (long long)g.z * g.N;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(t / g.N), i = (int)(t % g.N);
    if (g.kind == 0) {
      int X, Y, Z, dx, dy, dz;
      bcc_coords(i, g.L, g.divL, X, Y, Z);
      unpack_offset(g.off[j], dx, dy, dz);
      nbr[t] = bcc_offset_site(X, Y, Z, dx, dy, dz, g.L);
      J[t] = g.Jd[j];
    } else {
      nbr[t] = g.tab_nbr[t];
      J[t] = g.tab_Jd[t];
    }
  }
}

cudaError_t launch_neighbour_dump(const Geometry& g, int32_t* nbr, double* J, cudaStream_t stream) {
  neighbour_dump_kernel<<<256, 256, 0, stream>>>(g, nbr, J);
  return cudaGetLastError();
}

size_t walker_smem_bytes(bool traj, bool smem_lattice, int N, int W) {
  const size_t lng = (traj ? sizeof(double) : sizeof(long long)) * (size_t)W;
  const size_t h = ((size_t)W * 4 + 15) & ~(size_t)15;
  const size_t real = traj ? sizeof(double) : sizeof(float);
  size_t bytes = lng + h + 4 * kMaxSlotsPerSite + real * kMaxSlotsPerSite;
  if (smem_lattice) bytes += smem_site_bytes(traj) * (size_t)N;
  return bytes;
}

template <bool kTraj, bool kSmem, bool kInit, int kG, int kSlots>
static cudaError_t launch_walker_kernel(const WalkerArgs& a, int n_slots, size_t smem, cudaStream_t stream) {
  const auto kernel = walker_kernel<kTraj, kSmem, kInit, kG, kSlots>;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kernel<<<n_slots, kWalkerThreads, smem, stream>>>(a);
  return cudaGetLastError();
}

template <bool kSmem, bool kInit>
static cudaError_t launch_units(const WalkerArgs& a, int n_slots, size_t smem, cudaStream_t stream) {
  // bcc: lanes per move and slots per lane, for the couplings of 1 to 4 shells (8, 14, 26, 50 slots) and the
  // groups that the size rule picks for them; one lane per move only for the initial drive, as the pipelined
  // walker walks such lattices.  Other groups, and lattices given as tables, run the loop.
  const int n = a.geo.kind == 0 ? (a.geo.z + a.G - 1) / a.G : 99;
  if (a.G == 16 && n <= 4) return launch_walker_kernel<false, kSmem, kInit, 16, 4>(a, n_slots, smem, stream);
  if (a.G == 8 && n <= 2) return launch_walker_kernel<false, kSmem, kInit, 8, 2>(a, n_slots, smem, stream);
  if (a.G == 8 && n <= 7) return launch_walker_kernel<false, kSmem, kInit, 8, 7>(a, n_slots, smem, stream);
  if (a.G == 4 && n <= 7) return launch_walker_kernel<false, kSmem, kInit, 4, 7>(a, n_slots, smem, stream);
  if constexpr (kInit) {
    if (a.G == 1 && n <= 14) return launch_walker_kernel<false, kSmem, true, 1, 14>(a, n_slots, smem, stream);
  }
  return launch_walker_kernel<false, kSmem, kInit, 0, 0>(a, n_slots, smem, stream);
}

cudaError_t launch_walkers(const WalkerArgs& a, int n_slots, bool traj, bool smem_lattice, size_t smem,
                           cudaStream_t stream) {
  cudaError_t e;
  if (traj)
    e = smem_lattice ? launch_walker_kernel<true, true, false, 0, 0>(a, n_slots, smem, stream)
                     : launch_walker_kernel<true, false, false, 0, 0>(a, n_slots, smem, stream);
  else if (a.init)
    e = smem_lattice ? launch_units<true, true>(a, n_slots, smem, stream) : launch_units<false, true>(a, n_slots, smem, stream);
  else
    e = smem_lattice ? launch_units<true, false>(a, n_slots, smem, stream) : launch_units<false, false>(a, n_slots, smem, stream);
  if (e == cudaSuccess && a.recompute && !a.init && !traj && a.geo.kind == 0)
    e = launch_energy_update(a, n_slots, stream);
  return e;
}

}  // namespace rewl
