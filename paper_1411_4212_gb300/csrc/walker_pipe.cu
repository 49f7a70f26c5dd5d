// walker_pipe.cu -- warp-specialised Wang-Landau walker for bcc lattices, one lane per trial move
// (Sec. 4.2, Eq. 4; trial move Sec. 4.4).
//
// One CTA per walker slot.  Warp 1 (producer) prepares batch b+1 of 32 trial moves while warp 0
// (resolver) resolves batch b strictly in order, so the walk is the sequential Markov chain:
//   producer: Philox draws, the local field h_i = sum_j J_ij S_j over the coupling shells (bcc
//     offsets known at compile time, the neighbour loads in one unrolled loop), dE = -(S'-S).h, and
//     two conflict masks read from a shared-memory owner table -- the moves of batch b (still being
//     resolved while batch b+1 reads the lattice) and the earlier moves of batch b+1 that sit on the
//     same site or a neighbouring one;
//   resolver: a move whose mask meets a move accepted since the lattice was read is corrected
//     exactly (production: from the move batches; trajectory: summed again on the current lattice);
//     then accept with min[1, g(E)/g(E')] (reject outside the window) and add ln f to ln g and 1 to
//     H at the resulting state.
// The owner table may alias sites (hashed): an alias names a move that cannot change the field; the
// producer sorts such bits out by the distance of the sites.  Two record buffers alternate; named barriers
// READY(b mod 2) and DONE(b mod 2) order the hand-over, so the producer reads the lattice for batch b after every
// move of batch b-2 has been written; what batch b-1 changes is corrected.
#include "walker_common.cuh"

namespace rewl {

constexpr int kPairThreads = 64;   // resolver warp + producer warp
constexpr int kWorkerThreads = 64;     // batched walker: threads per worker (one pair)

__host__ __device__ constexpr size_t align16(size_t n) { return (n + 15) & ~(size_t)15; }

__device__ __forceinline__ void named_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(kPairThreads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(kPairThreads) : "memory");
}

// Production: one batch of 32 trial moves as the producer hands it over, one entry per move.  Every
// section is an array of 16-byte words, so the resolver's reads (lane = move, or any other move of the
// batch) are conflict-free 16-byte loads.  A move touches another when it sits on the other's site or on
// one of its neighbours; the masks hold the moves that touch this one, by the shell they sit on.
struct alignas(16) MoveBatch {
  int4 head[32];         // energy increment (2^-24 bins) | ln u (2^-20 units) | moves of batch b-1 touching
                         // this one | earlier moves of this batch touching it (both as they are counted)
  int4 place[32];        // site | octahedral code (u, v) of the proposed spin, what the lattice stores | half-unit
                         // coordinates X | Y << 10 | Z << 20 (here, where the resolver writes nothing, because the
                         // producer reads them of the batch that is being resolved)
  float4 n[32];          // proposed spin | earlier moves of this batch on this site
  float4 h[32];          // local field (snapshot) | moves of batch b-1 on this site (bits reversed: move j
                         // is bit 31 - j, so that count-leading-zeros walks them in order)
  float4 ds[32];         // new - old spin: the move's change to the lattice if accepted (kept current by
                         // the resolver)
  int4 cur[32];          // earlier moves of this batch on a neighbour, by shell
  int4 prev[32];         // moves of batch b-1 on a neighbour, by shell (bits reversed)
  int4 all;              // moves that touch a later one | moves on a later one's site | moves whose
                         // increment is a bin or more (count)
};

// Trajectory: one batch of 32 trial moves, an array per quantity.
struct alignas(16) TrajBatch {
  double dE[32], u[32];
  double nx[32], ny[32], nz[32];
  int4 move[32];         // site | half-unit coordinates X | Y << 10 | Z << 20 | ln u to 4e-6 (1 where u is too small
                         // for it) | dE in 2^-24 bins
  int4 marks[32];        // moves of batch b-1, earlier moves of this batch that touch this one; the same as the
                         // owner table has them (with the aliases), for the count of recomputed moves
};

// Bytes of the two move batches in flight.
__host__ __device__ constexpr size_t batch_bytes(bool traj) {
  return traj ? 2 * sizeof(TrajBatch) : 2 * sizeof(MoveBatch);
}

// Local field of (X, Y, Z) by one lane over all slots in canonical order, with the owner-table
// words of the site's neighbours OR-ed into touch[shell] (trajectory: touch[0]).
template <bool kTraj, int NSH, class Lat>
__device__ __forceinline__ void field_one_lane(const Lat& lat, int X, int Y, int Z, int L, const typename Mode<kTraj>::Real (&Jsh)[4],
                                               typename Mode<kTraj>::Real& hx, typename Mode<kTraj>::Real& hy,
                                               typename Mode<kTraj>::Real& hz, const uint2* own, uint32_t omask,
                                               uint2 (&touch)[4]) {
  using Real = typename Mode<kTraj>::Real;
  constexpr ShellTable T = make_shells(NSH);
  const int twoL = 2 * L, LL = L * L;
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
  hx = Real(0);
  hy = Real(0);
  hz = Real(0);
  // production: per-shell spin sums first, then one coupling per shell -- fewer roundings, and
  // none at all for aligned spins (whose dE would otherwise carry the same rounding every move)
  Real tx[4] = {Real(0), Real(0), Real(0), Real(0)}, ty[4] = {Real(0), Real(0), Real(0), Real(0)},
       tz[4] = {Real(0), Real(0), Real(0), Real(0)};
#pragma unroll
  for (int j = 0; j < T.z; ++j) {
    const int n = xw[T.dx[j] + 3] + yw[T.dy[j] + 3] + zw[T.dz[j] + 3] - ((T.dx[j] & 1) ? par_flip : par_same);
    Real vx, vy, vz;
    lat.get(n, vx, vy, vz);
    if constexpr (kTraj) {
      const Real J = Jsh[T.sh[j]];
      hx = __dadd_rn(hx, __dmul_rn(J, vx));
      hy = __dadd_rn(hy, __dmul_rn(J, vy));
      hz = __dadd_rn(hz, __dmul_rn(J, vz));
    } else {
      tx[T.sh[j]] += vx;
      ty[T.sh[j]] += vy;
      tz[T.sh[j]] += vz;
    }
    const uint2 o = own[n & omask];
    touch[kTraj ? 0 : T.sh[j]].x |= o.x;
    touch[kTraj ? 0 : T.sh[j]].y |= o.y;
  }
  if constexpr (!kTraj) {
#pragma unroll
    for (int s2 = 0; s2 < NSH; ++s2) {
      hx = fmaf(Jsh[s2], tx[s2], hx);
      hy = fmaf(Jsh[s2], ty[s2], hy);
      hz = fmaf(Jsh[s2], tz[s2], hz);
    }
  }
}

// Uniform in [1, 2) from the top 23 bits of a word (no integer-to-float conversion).
__device__ __forceinline__ float one_to_two(uint32_t x) { return __uint_as_float(0x3f800000u | (x >> 9)); }

// dE (FP32) -> int32 in 2^-24 bins: dE * (hi + lo) with the product of the head exact (fmaf).
__device__ __forceinline__ int dq24_of(float dE, const Windows& w) {
  const float p = dE * w.dq24_hi;
  const float e = fmaf(dE, w.dq24_hi, -p) + dE * w.dq24_lo;
  return __float2int_rn(p) + __float2int_rn(e);
}

// Trajectory mode.  dE in 2^-24 bins, at most kFarUnits = 64 bins either way (NaN: kFarUnits).
constexpr int kFarUnits = 1 << 30;
__device__ __forceinline__ int traj_units(double dE, double bin_units) {
  const int q = __double2int_rn(dE * bin_units);
  return dE == dE ? max(-kFarUnits, min(kFarUnits, q)) : kFarUnits;
}
// dE = -(S' - S) . h, one rounding per operation.
__device__ __forceinline__ double traj_energy(double nx, double ny, double nz, double ox, double oy, double oz, double hx,
                                              double hy, double hz) {
  const double dx = __dsub_rn(nx, ox), dy = __dsub_rn(ny, oy), dz = __dsub_rn(nz, oz);
  return -__dadd_rn(__dadd_rn(__dmul_rn(dx, hx), __dmul_rn(dy, hy)), __dmul_rn(dz, hz));
}
// dE of a move on the lattice as it is by a whole warp, in the producer's order: a product per lane, then the
// component of the field per lane (the sums are as long as by one lane, the FP64 issue a fifth).
template <int NSH>
__device__ __forceinline__ double traj_again(const SpinPlanes<double>& lat, const uint32_t* off_s, const double* J_s,
                                             int site, uint32_t coords, double nx, double ny, double nz, int L, int lane) {
  constexpr int z = make_shells(NSH).z, kParts = (3 * z + 31) / 32;
  double prod[kParts];
#pragma unroll
  for (int q = 0; q < kParts; ++q) {
    const int i = min(q * 32 + lane, 3 * z - 1), j = i / 3;
    int dx, dy, dz;
    unpack_offset(off_s[j], dx, dy, dz);
    const int n = bcc_offset_site((int)(coords & 1023u), (int)((coords >> 10) & 1023u), (int)(coords >> 20), dx, dy, dz, L);
    prod[q] = __dmul_rn(J_s[j], lat.component(n, i - 3 * j));
  }
  const int c = lane % 3;
  const double d = __dsub_rn(c == 0 ? nx : c == 1 ? ny : nz, lat.component(site, c));
  double h = 0.0;
#pragma unroll
  for (int j = 0; j < z; ++j) {
    // product 3 j + c: part (3 j + c) / 32 of lane (3 j + c) % 32
    const int q0 = 3 * j / 32, q1 = (3 * j + 2) / 32;
    double v = __shfl_sync(kFullMask, prod[q0], (3 * j + c) & 31);
    if (q1 != q0) {
      const double v1 = __shfl_sync(kFullMask, prod[q1], (3 * j + c) & 31);
      v = 3 * j + c >= 32 * q1 ? v1 : v;
    }
    h = __dadd_rn(h, v);
  }
  const double p = __dmul_rn(d, h);
  return -__dadd_rn(__dadd_rn(__shfl_sync(kFullMask, p, 0), __shfl_sync(kFullMask, p, 1)), __shfl_sync(kFullMask, p, 2));
}
// Order key of an entry of the ln g table; NaN above every number.
__device__ __forceinline__ long long traj_key(double v) { return order_key(v == v ? v : fabs(v)); }

// One exchange interval of walker slot `slot` by a group of nt threads (tid = 0..nt-1, nt a multiple
// of 32, at least 64): warp 0 resolves, warp 1 produces, every warp loads and stores.  smem_raw is
// the group's shared-memory arena (walker_pipe_smem_bytes), red holds nt/32 doubles.  Barrier
// bar_sync spans the group; bar_pair .. bar_pair+3 are READY(0), READY(1), DONE(0), DONE(1) of the
// resolver/producer pair.
template <bool kTraj, bool kSmem, int NSH>
__device__ __forceinline__ void pipe_walk_slot(const WalkerArgs& a, const int slot, const long long moves,
                                               const int recompute, unsigned char* smem_raw, double* red,
                                               const int tid, const int nt, const int bar_sync,
                                               const int bar_pair) {
  using Real = typename Mode<kTraj>::Real;
  using Lng = long long;   // production: 2^-40 units; trajectory: the order key of the FP64 value
  const int kBarReady = bar_pair, kBarDone = bar_pair + 2;
  const int warp = tid >> 5, lane = tid & 31;
  const int N = a.geo.N, W = a.win.W, L = a.geo.L;
  const int wlo = a.win.starts[global_slot(a.st, slot) / a.win.m];
  const int rep = a.st.perm[slot];
  const uint32_t omask = (uint32_t)a.own_mask;

  // shared layout: ln g | H | offsets | J per slot | move batches [2] | owner table | lattice (in shared
  // memory only); every section starts on a 16-byte boundary
  unsigned char* p = smem_raw;
  Lng* lng_s = reinterpret_cast<Lng*>(p);
  p += align16(sizeof(Lng) * (size_t)W);
  uint32_t* H_s = reinterpret_cast<uint32_t*>(p);
  p += align16((size_t)W * 4);
  uint32_t* off_s = reinterpret_cast<uint32_t*>(p);
  p += 4 * kMaxSlotsPerSite;
  Real* J_s = reinterpret_cast<Real*>(p);
  p += sizeof(Real) * kMaxSlotsPerSite;
  TrajBatch* rec = reinterpret_cast<TrajBatch*>(p);        // trajectory: [2]
  MoveBatch* mb = reinterpret_cast<MoveBatch*>(p);         // production: [2]
  p += batch_bytes(kTraj);
  uint2* own = reinterpret_cast<uint2*>(p);
  p += sizeof(uint2) * ((size_t)omask + 1);
  Real* spin_s = reinterpret_cast<Real*>(p);

  const auto glat = GlobalLattice<kTraj>::of(a.st.spins, rep, N);
  typename WalkLattice<kTraj, kSmem>::T lat;
  if constexpr (kSmem)
    lat = typename WalkLattice<kTraj, true>::T(spin_s, N);
  else
    lat = glat;

  const size_t lbase = (size_t)slot * W;
  for (int w = tid; w < W; w += nt) {
    if constexpr (kTraj)
      lng_s[w] = traj_key(a.st.lng[lbase + w]);
    else
      lng_s[w] = a.st.lng_fx[lbase + w];
    H_s[w] = a.st.H[lbase + w];
  }
  for (int j = tid; j < kMaxSlotsPerSite; j += nt) {
    off_s[j] = a.geo.off[j];
    J_s[j] = kTraj ? (Real)a.geo.Jd[j] : (Real)a.geo.Jf[j];
  }
  for (uint32_t i = tid; i <= omask; i += nt) own[i] = make_uint2(0u, 0u);
  if constexpr (kSmem) copy_lattice(lat, glat, N, tid, nt);
  group_sync(bar_sync, nt);

  const int nb = (int)((moves + 31) / 32);
  const long long t0 = a.st.steps[slot];
  const uint2 key = make_uint2((uint32_t)global_slot(a.st, slot), a.key1);

  const double bin_units = kTraj ? 16777216.0 / a.win.dE : 0.0;   // 2^-24 bins per unit of energy

  if (warp == 1) {
    // ------------------------------- producer -------------------------------
    Real Jsh[4];
#pragma unroll
    for (int s2 = 0; s2 < 4; ++s2) Jsh[s2] = kTraj ? (Real)a.geo.Jsh_d[s2] : (Real)a.geo.Jsh_f[s2];
    int site_prev = 0;
    bool valid_prev = false;
    const bool aliased = (long long)omask + 1 < (long long)N;   // several sites share an owner entry
    for (int b = 0; b < nb; ++b) {
      const int cur = b & 1;
      const bool valid = (long long)b * 32 + lane < moves;
      const unsigned long long t = (unsigned long long)(t0 + (long long)b * 32 + lane);
      int site;
      Real nx, ny, nz;
      double u = 0.0;
      int lu = 0;
      float2 code = make_float2(0.0f, 0.0f);
      if constexpr (kTraj) {
        double dnx, dny, dnz;
        draw_traj(key, t, false, N, site, u, dnx, dny, dnz);
        nx = (Real)dnx;
        ny = (Real)dny;
        nz = (Real)dnz;
      } else {
        const uint4 x = philox10(make_uint4((uint32_t)t, (uint32_t)(t >> 32), 0u, 0u), key);
        site = (int)__umulhi(x.x, (uint32_t)N);
        const float uf = (one_to_two(x.y) - 1.0f) + 0x1.0p-24f;                // (0, 1)
        lu = __float2int_rn(__logf(uf) * 1048576.0f);
        const float zc = (2.0f * one_to_two(x.z) - 3.0f) + 0x1.0p-23f;          // (-1, 1), cos(theta)
        float sn, cs;
        __sincosf((one_to_two(x.w) - 1.5f) * 6.28318530717958648f, &sn, &cs);  // azimuth in [-pi, pi)
        const float q = fmaxf(fmaf(-zc, zc, 1.0f), 0x1.0p-46f);
        const float r = q * rsqrtf(q);                                          // sin(theta)
        // the proposal is the spin its code decodes to
        code = oct_encode(r * cs, r * sn, zc);
        float fx, fy, fz;
        oct_decode(code, fx, fy, fz);
        nx = (Real)fx;
        ny = (Real)fy;
        nz = (Real)fz;
      }
      int X, Y, Z;
      bcc_coords(site, L, a.geo.divL, X, Y, Z);
      uint32_t* own32 = reinterpret_cast<uint32_t*>(own);
      if (valid) atomicOr(own32 + 2 * (site & omask) + cur, 1u << lane);
      __syncwarp();
      uint2 touch[4] = {};
      Real hx, hy, hz;
      // the draws and the owner-table insert above do not touch the lattice, so they overlap the
      // resolver's publication of batch b-2; the lattice holds every batch up to b-2 after DONE
      if (b >= 2) named_sync(kBarDone + (b & 1));
      field_one_lane<kTraj, NSH>(lat, X, Y, Z, L, Jsh, hx, hy, hz, own, omask, touch);
      const uint2 oself = own[site & omask];
      Real ox, oy, oz;
      lat.get(site, ox, oy, oz);
      // moves on this site and on the neighbours of each shell: earlier ones of this batch, and those of
      // batch b-1
      const uint32_t below = (1u << lane) - 1u, any_prev = b > 0 ? 0xffffffffu : 0u;
      uint32_t scur = (cur ? oself.y : oself.x) & below, sprev = (cur ? oself.x : oself.y) & any_prev;
      uint32_t tcur[4], tprev[4], ccur = scur, cprev = sprev;
#pragma unroll
      for (int s2 = 0; s2 < 4; ++s2) {
        tcur[s2] = (cur ? touch[s2].y : touch[s2].x) & below;
        tprev[s2] = (cur ? touch[s2].x : touch[s2].y) & any_prev;
        ccur |= tcur[s2];
        cprev |= tprev[s2];
      }
      if constexpr (kTraj) {
        TrajBatch& m = rec[cur];
        const double dE = traj_energy(nx, ny, nz, ox, oy, oz, hx, hy, hz);
        const float lu = u > 0x1.0p-100 ? logf(__double2float_rn(u)) : 1.0f;
        m.dE[lane] = dE;
        m.u[lane] = u;
        m.nx[lane] = nx;
        m.ny[lane] = ny;
        m.nz[lane] = nz;
        m.move[lane] = make_int4(site, X | (Y << 10) | (Z << 20), __float_as_int(lu), traj_units(dE, bin_units));
        __syncwarp();
        // the table's bits without the aliases: moves on this site or on a neighbour
        auto touching = [&](const TrajBatch& other, uint32_t bits) -> uint32_t {
          uint32_t real = 0u;
          for (; bits; bits &= bits - 1u) {
            const int j = __ffs(bits) - 1;
            const uint32_t q = (uint32_t)other.move[j].y;
            int ex = abs((int)(q & 1023u) - X), ey = abs((int)((q >> 10) & 1023u) - Y), ez = abs((int)(q >> 20) - Z);
            ex = min(ex, 2 * L - ex);
            ey = min(ey, 2 * L - ey);
            ez = min(ez, 2 * L - ez);
            const int r2 = ex * ex + ey * ey + ez * ez;
            real |= r2 == 0 || r2 == 3 || (NSH > 1 && r2 == 4) || (NSH > 2 && r2 == 8) || (NSH > 3 && r2 == 11) ? 1u << j : 0u;
          }
          return real;
        };
        m.marks[lane] = make_int4((int)(aliased ? touching(rec[cur ^ 1], cprev) : cprev),
                                  (int)(aliased ? touching(m, ccur) : ccur), (int)cprev, (int)ccur);
      } else {
        MoveBatch& m = mb[cur];
        // (rounded subtractions: a plain one could fuse with the product that decoded the old spin)
        const float dx = __fsub_rn(nx, ox), dy = __fsub_rn(ny, oy), dz = __fsub_rn(nz, oz);
        const float dE = -fmaf(dz, hz, fmaf(dy, hy, dx * hx));
        const int dq = dq24_of(dE, a.win);
        m.ds[lane] = make_float4(dx, dy, dz, 0.0f);
        m.place[lane] = make_int4(site, __float_as_int(code.x), __float_as_int(code.y), X | (Y << 10) | (Z << 20));
        if (aliased) {
          // An owner table smaller than the lattice is hashed: a bit may name a move whose site is neither
          // this move's site nor one of its neighbours, or name a shell that it does not sit on.  Sort the
          // bits by the distance of the sites.  With the lattice in global memory only real conflicts
          // count.  (At bcc L = 32 with 2048 entries, 92 % of the flagged moves were aliases.)
          __syncwarp();
          // Both masks in one loop: their moves' words are in flight together (64 runs in a batch 30.6 -> 30.1 ms).
          uint32_t bc = ccur, bp = cprev;
          const MoveBatch& before = mb[cur ^ 1];
          scur = sprev = 0u;
#pragma unroll
          for (int s2 = 0; s2 < 4; ++s2) tcur[s2] = tprev[s2] = 0u;
          auto sort_bit = [&](const uint32_t q, const uint32_t bit, uint32_t& same, uint32_t (&sh)[4]) {
            // every offset component of a neighbour is below L half-units, so the wrapped displacement
            // is the offset; squared distances 3, 4, 8, 11 are the shells 1..4
            int ex = abs((int)(q & 1023u) - X), ey = abs((int)((q >> 10) & 1023u) - Y), ez = abs((int)(q >> 20) - Z);
            ex = min(ex, 2 * L - ex);
            ey = min(ey, 2 * L - ey);
            ez = min(ez, 2 * L - ez);
            const int r2 = ex * ex + ey * ey + ez * ez;
            // (a shell without coupling changes nothing either)
            same |= r2 == 0 ? bit : 0u;
            sh[0] |= r2 == 3 && Jsh[0] != Real(0) ? bit : 0u;
            sh[1] |= NSH > 1 && r2 == 4 && Jsh[1] != Real(0) ? bit : 0u;
            sh[2] |= NSH > 2 && r2 == 8 && Jsh[2] != Real(0) ? bit : 0u;
            sh[3] |= NSH > 3 && r2 == 11 && Jsh[3] != Real(0) ? bit : 0u;
          };
          while (bc | bp) {
            const uint32_t bit_c = bc & (0u - bc), bit_p = bp & (0u - bp);   // 0: none left
            const uint32_t qc = (uint32_t)m.place[(__ffs(bc) - 1) & 31].w, qp = (uint32_t)before.place[(__ffs(bp) - 1) & 31].w;
            sort_bit(qc, bit_c, scur, tcur);
            sort_bit(qp, bit_p, sprev, tprev);
            bc ^= bit_c;
            bp ^= bit_p;
          }
          if constexpr (!kSmem) {
            ccur = scur | tcur[0] | tcur[1] | tcur[2] | tcur[3];
            cprev = sprev | tprev[0] | tprev[1] | tprev[2] | tprev[3];
          }
        }
        m.head[lane] = make_int4(dq, lu, (int)cprev, (int)ccur);
        m.n[lane] = make_float4(nx, ny, nz, __uint_as_float(scur));
        m.h[lane] = make_float4(hx, hy, hz, __uint_as_float(__brev(sprev)));
        m.cur[lane] = make_int4((int)tcur[0], (int)tcur[1], (int)tcur[2], (int)tcur[3]);
        m.prev[lane] = make_int4((int)__brev(tprev[0]), (int)__brev(tprev[1]), (int)__brev(tprev[2]),
                                 (int)__brev(tprev[3]));
        const uint32_t touched = __reduce_or_sync(kFullMask, valid ? scur | tcur[0] | tcur[1] | tcur[2] | tcur[3] : 0u);
        const uint32_t on_site = __reduce_or_sync(kFullMask, valid ? scur : 0u);
        const int n_long = __popc(__ballot_sync(kFullMask, (unsigned)(dq + (1 << 24)) >= (1u << 25)));
        if (lane == 0) m.all = make_int4((int)touched, (int)on_site, n_long, 0);
      }
      __syncwarp();
      named_arrive(kBarReady + cur);
      // batch b+1 inserts into the other slot, which still holds batch b-1's bits
      if (valid_prev) own32[2 * (site_prev & omask) + (cur ^ 1)] = 0u;
      __syncwarp();   // every clear lands before any lane inserts batch b+1
      site_prev = site;
      valid_prev = valid;
    }
    for (int b = nb - 2 > 0 ? nb - 2 : 0; b < nb; ++b) named_sync(kBarDone + (b & 1));
  } else if (warp == 0) {
   if constexpr (kTraj) {
    // ------------------------ resolver (trajectory mode) ------------------------
    // The walk in FP64 exactly as specified, one rounding per operation; but an FP64 operation takes 62 cycles,
    // a division 550 and the specified exponential 34 operations in a row, so none of them sits on the chain
    // from one accepted move to the next.  Lane k holds move k; a round finds the first move that is accepted,
    // as in the production resolver below, from quantities that decide all but a few moves in 1e5:
    //   - the walker's position to 2^-24 bins in integers (taken afresh from E every batch, off by at most one
    //     unit, then half a unit per accepted move): its bin is certain unless it lies within kEdge units of a
    //     bin's edge;
    //   - ln g(now) - ln u to kTol (ln u is good to 4e-6, the sums below 1e9 to 1e-6): the move is accepted if
    //     ln g(target) is below, rejected if above by more.
    // A move that this leaves open, or whose dE is of an older lattice, is taken when its turn comes: its dE is
    // summed again, and the specified operations decide.  E and the exact ln g are carried beside the chain.  A
    // bin's ln g grows by a rounded addition of ln f per move; where no sum of this call can round (grid) that is
    // one product and sum, else the additions are made when the walker leaves the bin.  The table holds order
    // keys, so comparisons are integer ones.
    // Measured, bcc L = 16, 2 shells, 64 walkers: 18.3 ms per 10^4 moves with every move decided in turn, 2.8 ms
    // so (slowest walker, 30 of 32 moves accepted: 17,500 cycles per batch, 370 per accepted move and 2,100 per dE
    // summed again; the producer's 12,600, mostly FP64 issue at 17 cycles per warp instruction, come next).
    constexpr int kBin = 1 << 24, kEdge = 64;
    constexpr double kTol = 1e-5;
    constexpr uint32_t kNoKey = 0xffffffffu, kRare = 0x07fffffeu, kPayload = 0x07ffffffu;
    double E = a.st.E[slot];
    int r = a.st.bin[slot] - wlo;
    const double lnf0 = a.st.lnf[slot];
    const bool frozen = !(lnf0 >= a.lnf_final);
    const double lnf = frozen ? 0.0 : lnf0;
    const bool bad = (unsigned)r >= (unsigned)W;
    if (bad) {
      if (lane == 0) atomicExch(a.st.ctrl + 0, kErrOutOfWindow);
      r = 0;                                  // no move is made
    }
    const double lane_lnf = (double)lane * lnf;
    const uint32_t lane_key = (uint32_t)lane << 27;
    // grid: every sum that ln g can reach in this call is exact, as all entries and ln f are multiples of 2^low
    // and nothing gets as large as 2^(low + 53)
    bool grid;
    {
      // exponent and lowest set bit (both biased) of an entry; 0 takes no part, what is not a plain number none
      int high = 0, low = 4096;
      auto note = [&](double v) {
        const unsigned long long m = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL;
        const int ex = (int)(m >> 52);
        const unsigned long long f = m & 0xfffffffffffffULL;
        high = max(high, ex);
        low = m == 0ULL ? low : ex == 0 || ex == 2047 ? -4096 : min(low, f ? ex - 53 + __ffsll((long long)f) : ex);
      };
      for (int w = lane; w < W; w += 32) note(order_value(lng_s[w]));
      high = __reduce_max_sync(kFullMask, high);
      low = __reduce_min_sync(kFullMask, low);
      note(lnf);
      // |ln g| < 2^(high - 1022) + moves ln f; twice the larger one is a bound
      const int rise = ((__double2hiint((double)moves * lnf) & 0x7fffffff) >> 20) + 1;
      grid = !frozen && max(high + 1, rise) + 1 - low <= 53 && low > 0;
    }
    // ln g after n more moves in the same bin: n rounded additions of ln f
    auto advance = [&](double v, int n) -> double {
      for (; n > 0 && !frozen; --n) v = __dadd_rn(v, lnf);
      return v;
    };
    const bool wild = !(fabs(lnf) < 1e6);
    double entry = order_value(lng_s[r]);     // ln g of the bin at move e_in; grid: drawn back to the batch's first move
    uint32_t acc_prev = 0;
    long long n_acc = 0, n_rec = 0;
    for (int b = 0; b < nb; ++b) {
      const int cur = b & 1;
      named_sync(kBarReady + cur);
      const int nvalid = bad ? 0 : (int)(moves - (long long)b * 32 < 32 ? moves - (long long)b * 32 : 32);
      const bool valid = lane < nvalid;
      const TrajBatch& B = rec[cur];
      const int4 move = B.move[lane], marks = B.marks[lane];
      const int site = move.x;
      const float lu = __int_as_float(move.z);
      double dE = B.dE[lane];
      const double nx = B.nx[lane], ny = B.ny[lane], nz = B.nz[lane];
      int dq = move.w;
      const uint32_t cc = (uint32_t)marks.y;
      bool stale = valid && ((uint32_t)marks.x & acc_prev) != 0u;       // dE is of an older lattice
      // dE of moves `todo` again, on the lattice as it is
      auto refresh = [&](uint32_t todo) {
        __syncwarp();
        for (; todo; todo &= todo - 1u) {
          const int k = __ffs(todo) - 1;
          const int4 mk = B.move[k];
          const double v = traj_again<NSH>(lat, off_s, J_s, mk.x, (uint32_t)mk.y, B.nx[k], B.ny[k], B.nz[k], L, lane);
          if (lane == k) {
            dE = v;
            dq = traj_units(v, bin_units);
            stale = false;
          }
        }
        __syncwarp();
      };
      refresh(__ballot_sync(kFullMask, stale && cc == 0u));    // (the others may go stale again before their turn)
      // position of E above the bottom of bin r0, 2^-24 bins; lost: nowhere near (the state was set from outside)
      int at, r0;
      bool lost;
      auto locate = [&]() {
        r0 = r;
        const double q = (E - a.win.e_min) * bin_units - (double)(wlo + r) * 16777216.0;
        lost = !(fabs(q) < 16.0 * kBin);
        at = lost ? 0 : __double2int_rn(q);
      };
      locate();
      // ln g(target) up to klo: accepted; from khi: rejected; between, or where |ln g| is beyond what they are good
      // for: open
      const double from_lo = lane_lnf - (double)lu - kTol, from_hi = lane_lnf - (double)lu + kTol;
      long long klo, khi;
      bool far;
      auto thresholds = [&](double L0) {      // L0: ln g of the bin drawn back to the batch's first move
        far = (__double2hiint(L0) & 0x7fffffff) >= 0x41cdcd65 || wild || lu > 0.0f;      // 1e9
        klo = order_key(L0 + from_lo);
        khi = order_key(L0 + from_hi);
      };
      thresholds(entry);
      // ln g of the bin at move k
      int e_in = 0;
      auto lng_at = [&](int k) -> double {
        if (grid) return entry + (double)k * lnf;
        return advance(entry, k - e_in);
      };
      uint32_t acc_cur = 0;
      int rb = r;                             // bin after this lane's move
      bool live = valid;
      while (true) {
        const int pos = at + dq, db = pos >> 24;
        const int rel = r0 + db;
        const int fr = pos & (kBin - 1);
        const bool inw = (unsigned)rel < (unsigned)W;
        const long long lt = lng_s[min((unsigned)rel, (unsigned)W - 1u)];
        const bool sure = !stale && !far && !lost && (unsigned)(dq + kFarUnits - 1) < 2u * kFarUnits - 1u &&
                          (unsigned)(fr - kEdge) < (unsigned)(kBin - 2 * kEdge);
        const bool same_bin = rel == r;
        const bool yes = inw && (same_bin || lt <= klo);
        const bool no = !inw || (!same_bin && lt >= khi);
        const double cand = order_value(lt) - lane_lnf;
        const uint32_t code = (uint32_t)(dq + 4 * kBin);
        const uint32_t m = __reduce_min_sync(
            kFullMask, live && !(sure && no) ? lane_key | (sure && yes && code < kRare ? code : kRare) : kNoKey);
        const int e = (int)(m >> 27);
        live = live && lane > e;
        const double E_step = __shfl_sync(kFullMask, dE, e);
        int re, seen;                         // bin of the move; the bin that the integers gave it
        if ((m & kPayload) < kRare) {
          at += (int)(m & kPayload) - 4 * kBin;
          re = seen = r0 + (at >> 24);
        } else {
          if (m == kNoKey) break;             // every move left is rejected
          // stale, uncertain or long
          if (__shfl_sync(kFullMask, (int)stale, e)) {
            refresh(1u << e);
            live = live || (lane == e);
            continue;
          }
          const int de = __shfl_sync(kFullMask, dq, e);
          re = seen = __shfl_sync(kFullMask, rel, e);
          if (__shfl_sync(kFullMask, (int)!(sure && yes), e)) {
            // the specified operations
            re = bin_fp64(__dadd_rn(E, E_step), a.win) - wlo;
            bool accept = false;
            if ((unsigned)re < (unsigned)W) {
              const double L = lng_at(e);
              const double d = __dsub_rn(L, re == r ? L : order_value(lng_s[re]));
              accept = (d >= 0.0) || (B.u[e] < exp_fp64(d, a.ex));
            }
            if (!accept) continue;
          }
          at += de;
        }
        if (re != r) {
          double L0 = __shfl_sync(kFullMask, cand, e);
          if (seen != re) L0 = order_value(lng_s[re]) - __shfl_sync(kFullMask, lane_lnf, e);
          thresholds(L0);
          if (grid) {
            lng_s[r] = order_key(entry + __shfl_sync(kFullMask, lane_lnf, e));
            entry = L0;
          } else {
            lng_s[r] = traj_key(advance(entry, e - e_in));
            entry = order_value(lng_s[re]);
          }
          e_in = e;
          r = re;
          rb = lane >= e ? r : rb;
        }
        E = __dadd_rn(E, E_step);
        acc_cur |= 1u << e;
        if (lane == e) lat.set(site, nx, ny, nz);
        stale = stale || ((cc >> e) & 1u) != 0u;
        if (lost || !((unsigned)(at + 16 * kBin) < 32u * kBin)) locate();   // positions are relative to bin r0
      }
      entry = lng_at(nvalid);
      if (!frozen && valid) atomicAdd(&H_s[rb], 1u);
      n_rec += __popc(__ballot_sync(kFullMask, valid && (((uint32_t)marks.z & acc_prev) | ((uint32_t)marks.w & acc_cur)) != 0u));
      n_acc += __popc(acc_cur);
      acc_prev = acc_cur;
      __syncwarp();
      named_arrive(kBarDone + cur);
    }
    if (lane == 0 && !bad) {
      a.st.E[slot] = E;
      a.st.bin[slot] = r + wlo;
      lng_s[r] = traj_key(entry);
      a.st.steps[slot] = t0 + moves;
      a.st.accepts[slot] += n_acc;
      a.st.recomputes[slot] += n_rec;
    }
   } else {
    // ------------------------ resolver (production mode) ------------------------
    // The lattice holds every batch up to b-2 while batch b is resolved: batch b-1's accepted spins
    // are written at the start of batch b, after the producer has read the lattice for batch b.  A
    // move's energy change then follows exactly from the producer's snapshot (field h, old spin o)
    // and the accepted moves of batch b-1 and of batch b before it that touch it: each adds
    // J (S' - S) to h, or replaces o when it sits on the move's own site, in the order of the moves.
    // Lane k holds move k throughout: it pulls the corrections from batch b-1 at the start, and when a
    // move of this batch is accepted, every later lane that it touches takes its correction at once
    // (push), all lanes together.
    // The walker's state is its bin r of the window and the fraction of the bin below its energy, in
    // 2^-24 bins (the eight lowest bits of the fixed-point energy never change during a walk: increments
    // are whole 2^-24 bins).  ln g of the current bin at move k is A + k ln f; it goes back to the table
    // only when the walker leaves the bin.
    const long long efx0 = a.st.efx[slot];
    int r = fx_bin(efx0) - wlo;
    int frac = (int)((uint32_t)efx0 >> 8);
    const uint32_t frac_low = (uint32_t)efx0 & 0xffu;
    // shell couplings as four scalars: an indexed read of the parameter array would be a
    // constant-memory load whose lanes take different indexes, serialised lane by lane
    const float J0 = a.geo.Jsh_f[0], J1 = NSH > 1 ? a.geo.Jsh_f[1] : 0.0f, J2 = NSH > 2 ? a.geo.Jsh_f[2] : 0.0f,
                J3 = NSH > 3 ? a.geo.Jsh_f[3] : 0.0f;
    const long long lnf_fx = a.st.lnf_fx[slot];
    const bool frozen = !((double)lnf_fx * kLngUnit >= a.lnf_final);
    const long long lnf_eff = frozen ? 0 : lnf_fx;
    const bool bad = (unsigned)r >= (unsigned)W;
    if (bad) {
      if (lane == 0) atomicExch(a.st.ctrl + 0, kErrOutOfWindow);
      r = 0;                                // no move is made
    }
    long long A = lng_s[r];
    const long long lane_lnf = (long long)lane * lnf_eff;
    constexpr int kBin = 1 << 24;
    constexpr uint32_t kNoKey = 0xffffffffu;
    constexpr int kDense = 14;
    const uint32_t lane_key = (uint32_t)lane << 27;
    // Three ways through a batch, all with the same decisions; each batch takes the cheapest for the
    // counts of the batch before it:
    //   scan       -- a run of moves that stay in the bin is accepted together; one round per move that
    //                 leaves it: few exits (high-energy windows);
    //   blocks     -- one round per accepted move, steps to a neighbouring bin decided by two pass bits
    //                 per move: few accepted moves, few bin changes (low-energy windows, where most
    //                 proposals are rejected exits);
    //   sequential -- one round per accepted move, every lane looking up ln g at its own target bin: any
    //                 accepted move may change bin (bins as narrow as the temperature).
    // What bounds it: the chain from one accepted move to the next, latency alone (one warp, every
    // instruction waits for the one before).  So a round costs as few dependent steps as possible, and
    // rejected moves cost nothing.  Resolving one move after the other, or blocks of 8 with a restart at
    // every event, took 90-350 cycles per move; now (ms per 10^4 moves, GB300) bcc L = 16, 2 shells,
    // [E_gs, 0], 64 walkers: 0.69 -> 0.46; bcc L = 8, 3 shells, converging (4000 moves): 1.03 -> 0.50;
    // 576 walkers of bcc L = 4, 5, 6, converging (4000 moves): 3.1 -> 0.67.
    // A round finds the first move that counts, and what it does, with one warp minimum (24 cycles; a
    // vote, a find-first-set and a shuffle take 100): key = lane << 27 | payload, all ones for lanes
    // with nothing to say and for decided moves.  One branch per round tells the rare payloads apart.
    enum { kScan = 0, kBlocks = 1, kSequential = 2 };
    const int forced = a.resolver - 1;      // -1: per-batch choice
    int path = kBlocks, n_in = 0, n_exit = 32, n_chg = 0;
    int n_scan = 0, n_blocks = 0, n_seq = 0;   // batches per path
    uint32_t acc_prev = 0, acc_prev_rev = 0, pub_prev = 0;
    int4 place_prev = make_int4(0, 0, 0, 0);
    long long n_acc = 0;
    unsigned n_rec = 0;                        // this lane's corrected moves
    for (int b = 0; b < nb; ++b) {
      const int cur = b & 1;
      named_sync(kBarReady + cur);
      const int nvalid = bad ? 0 : (int)(moves - (long long)b * 32 < 32 ? moves - (long long)b * 32 : 32);
      const bool valid = lane < nvalid;
      MoveBatch& C = mb[cur];
      const MoveBatch& P = mb[cur ^ 1];
      const int4 all = C.all;
      const int4 hd = C.head[lane];
      const float4 n4 = C.n[lane];
      float4 h4 = C.h[lane], d4 = C.ds[lane];
      const int4 tc = C.cur[lane], tp = C.prev[lane];
      const uint32_t touched = (uint32_t)all.x;     // moves that touch a later one
      const uint32_t sc = __float_as_uint(n4.w);
      const int4 place = C.place[lane];
      int dq = hd.x;
      auto increment = [&]() { dq = dq24_of(-fmaf(d4.z, h4.z, fmaf(d4.y, h4.y, d4.x * h4.x)), a.win); };
      // coupling of the shell whose mask has this bit
      auto coupling = [&](const int4& t, uint32_t bit) -> float {
        float J = (uint32_t)t.x & bit ? J0 : 0.0f;
        if constexpr (NSH > 1) J = (uint32_t)t.y & bit ? J1 : J;
        if constexpr (NSH > 2) J = (uint32_t)t.z & bit ? J2 : J;
        if constexpr (NSH > 3) J = (uint32_t)t.w & bit ? J3 : J;
        return J;
      };
      // an accepted move with proposed spin v sits on this lane's site
      auto replace = [&](const float4 v) {
        d4.x = n4.x - v.x;
        d4.y = n4.y - v.y;
        d4.z = n4.z - v.z;
        C.ds[lane] = d4;
      };
      // ---- corrections from batch b-1 ----
      {
        const uint32_t sp = __float_as_uint(h4.w);
        uint32_t t = valid ? (sp | (uint32_t)tp.x | (uint32_t)tp.y | (uint32_t)tp.z | (uint32_t)tp.w) & acc_prev_rev : 0u;
        n_rec += valid && ((uint32_t)hd.z & acc_prev) != 0u ? 1u : 0u;
        if (t) {
          do {
            const int j = __clz((int)t);
            const uint32_t bit = 0x80000000u >> j;
            t ^= bit;
            const float4 dj = P.ds[j];
            if (sp & bit) {
              replace(P.n[j]);
            } else {
              const float J = coupling(tp, bit);
              h4.x = fmaf(J, dj.x, h4.x);
              h4.y = fmaf(J, dj.y, h4.y);
              h4.z = fmaf(J, dj.z, h4.z);
            }
          } while (t);
          increment();
        }
      }
      // batch b-1's spins go to the lattice now that the producer has read it for batch b: accepted
      // moves, minus those superseded on their site
      if (b > 0) {
        if ((pub_prev >> lane) & 1u)
          lat.set_code(place_prev.x, make_float2(__int_as_float(place_prev.y), __int_as_float(place_prev.z)));
        __syncwarp();
        named_arrive(kBarDone + (cur ^ 1));
      }
      place_prev = place;
      // ---- the batch in order ----
      // Measured (cycles per batch): blocks 350 + 95 per accepted move + 350 per bin change (and per move
      // of a bin or more, if undecided by the pass bits), scan 450 + 100 per rejected exit + 300 per other
      // event, sequential 300 + 160 per accepted move (250 where every accepted move is pushed).  So two
      // bin changes, or two moves that may reach beyond the next bin, make the sequential path cheaper than
      // blocks; than scan only where few moves are accepted between such events (at the beginning of a run nearly
      // all are: the first 3 x 1000 moves of bcc L = 16, 1 shell, 500 bins took 125 us each without this comparison,
      // 81 with it, those of L = 24, 2 shells, 2000 bins 125 and 89).  It asks for a third more than break-even:
      // counts of the batch before say only so much about this one.  Between scan and blocks the counts of exits and
      // of accepted moves decide.
      path = n_chg >= 2 || all.z >= 2 ? kSequential : (n_exit + 2 < n_in ? kScan : kBlocks);
      const int events = n_chg + __popc(touched) + all.z;
      if (path == kSequential && 150 + 100 * (n_exit - n_chg) + 300 * events < 110 * n_in) path = kScan;
      if (forced >= 0) path = forced;
      uint32_t same = 0u;                  // accepted moves of this batch on this lane's site
      uint32_t acc_cur = 0u;
      int rb = r;                          // bin before this lane's move
      n_chg = 0;                           // bin changes
      // A move is accepted iff ln g(now) - ln g(target) >= T, T = min(0, (ln u + 1) 2^20): with
      // d = ln g(now) - ln g(target) in 2^-40 units this is d >= 0 or ln u < floor(d / 2^20).  With
      // ln g(now) = A + lane ln f: ln g(target) <= A + Q.
      const long long Q = lane_lnf - (hd.y < 0 ? (long long)(hd.y + 1) * 1048576LL : 0LL);
      // (it reads what an earlier push of the batch may have written in another lane: the warp is ordered before it,
      // with nothing to wait for there; after the store the same barrier cost 2 % of a batch, 7 % in the dense form)
      auto push = [&](const int e) {
        const uint32_t bit = 1u << e;
        const float4 de = C.ds[e];
        const float J = coupling(tc, bit);
        h4.x = fmaf(J, de.x, h4.x);        // J = 0: unchanged
        h4.y = fmaf(J, de.y, h4.y);
        h4.z = fmaf(J, de.z, h4.z);
        const float4 v = C.n[e];
        const bool own = (sc & bit) != 0u;   // it sits on this lane's site
        d4.x = own ? n4.x - v.x : d4.x;
        d4.y = own ? n4.y - v.y : d4.y;
        d4.z = own ? n4.z - v.z : d4.z;
        if (own) C.ds[lane] = d4;
        same |= sc & bit;
        increment();
      };
      // the accepted move e leaves the bin for bin r + db
      auto change_bin = [&](const int e, const int db) {
        const long long el = (long long)e * lnf_eff;
        lng_s[r] = (A + el);
        r += db;
        A = lng_s[r] - el;
        rb = lane > e ? r : rb;
        ++n_chg;
      };
      // Would a step to bin r + 1 / r - 1 be accepted at this lane's move: positions [lo, lo + span)
      // (2^-24 bins from the bottom of bin r) are accepted, those inside the bin among them.
      int lo = 0;
      uint32_t span = 0;
      auto pass = [&]() {
        const bool up = r + 1 < W && lng_s[min(r + 1, W - 1)] <= A + Q;
        const bool down = r > 0 && lng_s[max(r - 1, 0)] <= A + Q;
        lo = down ? -kBin : 0;
        span = (uint32_t)(kBin + (up ? kBin : 0) - lo);
      };
      // the target bin r + db of move e, looked up
      auto admits = [&](const int e, const int db) -> bool {
        return (unsigned)(r + db) < (unsigned)W && lng_s[r + db] <= A + shfl_ll(Q, e);
      };
      if (path == kSequential && __popc(touched) >= kDense) {
        // Many moves touch a later one (small lattices): every round pushes, without asking.  Measured,
        // ms per 10^4 moves with and without this form: 1.03 and 1.36 at bcc L = 4 (about 27 of 32 moves
        // touch a later one), 1.26 and 1.21 at L = 8 (11 of 32).
        // payload: the increment, -4..4 bins; kRare (-4 bins) stands for a longer one, and for -1 (whose
        // key would be kNoKey in lane 31).
        constexpr uint32_t kRare = 0x04000000u, kPayload = 0x07ffffffu;
        bool live = valid;
        while (true) {
          const int pos = frac + dq, rel = r + (pos >> 24);
          const long long lt = lng_s[min((unsigned)rel, (unsigned)W - 1u)];
          const bool plain = (unsigned)(dq + 4 * kBin - 1) < 8u * kBin - 1u && dq != -1;
          const uint32_t key = lane_key | (plain ? (uint32_t)dq & kPayload : kRare);
          // ln g of the walker's own bin in the table is at most its present value, so a move that
          // stays passes the test too
          const bool ok = live && (unsigned)rel < (unsigned)W && lt <= A + Q;
          const uint32_t m = __reduce_min_sync(kFullMask, ok ? key : kNoKey);
          __syncwarp();                    // for push, below
          const int e = (int)(m >> 27);
          const long long A2 = shfl_ll(rel == r ? A : lt - lane_lnf, e);   // ln g after the move, less e ln f
          int pe = frac + ((int)(m << 5) >> 5);
          if ((m & kPayload) == kRare || m == kNoKey) {
            if (m == kNoKey) break;        // every move left is rejected
            pe = __shfl_sync(kFullMask, pos, e);
          }
          lng_s[r] = (A + (long long)e * lnf_eff);
          n_chg += (pe >> 24) != 0 ? 1 : 0;
          r += pe >> 24;
          frac = pe & (kBin - 1);
          A = A2;
          acc_cur |= 1u << e;
          live = live && lane > e;
          rb = lane > e ? r : rb;
          push(e);
        }
      } else if (path == kSequential) {
        // payload: the increment, -4..4 bins; kRare (-4 bins) stands for a longer one, for -1 (whose key
        // would be kNoKey in lane 31) and for a move that touches a later one.
        // pos, at: positions relative to bin r0, which follows the walker when it is 16 bins away (sums
        // stay below 128 bins).
        constexpr uint32_t kRare = 0x04000000u, kPayload = 0x07ffffffu;
        int r0 = r, at = frac;
        auto make_key = [&]() -> uint32_t {
          const bool plain = (unsigned)(dq + 4 * kBin - 1) < 8u * kBin - 1u && dq != -1 && !((touched >> lane) & 1u);
          return lane_key | (plain ? (uint32_t)dq & kPayload : kRare);
        };
        uint32_t key = valid ? make_key() : kNoKey;
        int pos, rel;
        long long lt;
        auto look = [&]() {
          pos = at + dq;
          rel = r0 + (pos >> 24);
          lt = lng_s[min((unsigned)rel, (unsigned)W - 1u)];
        };
        look();
        bool away = false;
        while (true) {
          // ln g of the walker's own bin in the table is at most its present value, so a move that
          // stays passes the test too
          const bool ok = (unsigned)rel < (unsigned)W && lt <= A + Q;
          const uint32_t m = __reduce_min_sync(kFullMask, ok ? key : kNoKey);
          const int e = (int)(m >> 27);
          const long long A2 = shfl_ll(rel == r ? A : lt - lane_lnf, e);   // ln g after the move, less e ln f
          const bool rare = (m & kPayload) == kRare || m == kNoKey || away;
          const int at2 = at + ((int)(m << 5) >> 5);
          if (!rare) lng_s[r] = (A + (long long)e * lnf_eff);
          const int pos2 = at2 + dq, rel2 = r0 + (pos2 >> 24);
          const long long lt2 = lng_s[min((unsigned)rel2, (unsigned)W - 1u)];
          int rn;
          if (rare) {
            if (m == kNoKey) break;        // every move left is rejected
            const int pe = __shfl_sync(kFullMask, pos, e);
            lng_s[r] = (A + (long long)e * lnf_eff);
            r0 += pe >> 24;
            at = pe & (kBin - 1);
            rn = r0;
            key = lane > e ? key : kNoKey;
            if ((touched >> e) & 1u) {
              __syncwarp();
              push(e);
              key = key == kNoKey ? kNoKey : make_key();
            }
            look();
          } else {
            at = at2;
            pos = pos2;
            rel = rel2;
            lt = lt2;
            rn = r0 + (at >> 24);
            key = lane > e ? key : kNoKey;
          }
          A = A2;
          away = (unsigned)(at + 16 * kBin) >= 32u * kBin;
          n_chg += rn != r ? 1 : 0;
          r = rn;
          acc_cur |= 1u << e;
          rb = lane > e ? r : rb;
        }
        frac = at & (kBin - 1);
      } else if (path == kBlocks) {
        // payload: bit 24 the move leaves the bin, bit 25 it touches a later one or may reach further than
        // the next bin (looked up on its own), else the new fraction
        constexpr uint32_t kRare = 0x03000000u;
        uint32_t kc;
        bool live = valid;
        auto arm = [&]() {                 // after a bin change or a correction
          pass();
          const bool far = (unsigned)(dq + kBin) >= 2u * kBin;
          kc = lane_key | (far || ((touched >> lane) & 1u) ? 0x02000000u : 0u);
          if (far) {                       // a candidate wherever it lands
            lo = (int)0x80000000u;
            span = 0xffffffffu;
          }
          if (!live) span = 0u;
        };
        arm();
        while (true) {
          const int pos = frac + dq;
          const uint32_t m = __reduce_min_sync(
              kFullMask, (uint32_t)pos - (uint32_t)lo < span ? ((uint32_t)pos & 0x01ffffffu) | kc : kNoKey);
          const int e = (int)(m >> 27);
          if (m & kRare) {
            if (m == kNoKey) break;        // every move left is rejected
            const int pe = __shfl_sync(kFullMask, pos, e);
            const int de = pe >> 24;
            live = live && lane > e;
            span = live ? span : 0u;
            if (de != 0) {
              if (!admits(e, de)) continue;
              change_bin(e, de);
            }
            acc_cur |= 1u << e;
            frac = pe & (kBin - 1);
            if ((touched >> e) & 1u) {
              __syncwarp();
              push(e);
            }
            arm();
          } else {
            live = live && lane > e;
            span = live ? span : 0u;
            acc_cur |= 1u << e;
            frac = (int)(m & 0xffffffu);
          }
        }
      } else if (nvalid > 0) {
        // Prefix sums S of the increments give every undecided move's position if all of them before it
        // are accepted in the bin (which they are until one leaves the bin or meets an accepted move
        // of this batch); sums wrap modulo 2^32, but up to the first exit they stay within 101 bins.
        // payload: the increment of a rejected exit; kRare: an accepted one, one that may reach further
        // than the next bin, or a move that meets an accepted one and takes its corrections when its turn
        // comes (then every earlier move in `need` is an accepted one); no increment beside kRare, so that
        // no key of lane 31 is kNoKey
        constexpr uint32_t kRare = 0x04000000u;
        const uint32_t every = nvalid >= 32 ? 0xffffffffu : ((1u << nvalid) - 1u);
        uint32_t need = sc | (uint32_t)tc.x | (uint32_t)tc.y | (uint32_t)tc.z | (uint32_t)tc.w;
        uint32_t rej = 0u;                   // rejected moves
        uint32_t S = valid ? (uint32_t)dq : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t t = __shfl_up_sync(kFullMask, S, o);
          if (lane >= o) S += t;
        }
        uint32_t base = (uint32_t)frac;
        pass();
        bool live = valid;
        bool far;
        uint32_t kc;
        auto arm = [&]() {                   // after a correction
          far = (unsigned)(dq + kBin) >= 2u * kBin;
          kc = lane_key | ((uint32_t)dq & 0x03ffffffu);
        };
        arm();
        while (true) {
          const int pos = (int)(base + S);
          const bool meet = need != 0u;
          const uint32_t m = __reduce_min_sync(
              kFullMask, live && (meet || (unsigned)pos >= (unsigned)kBin)
                             ? (meet || far || (uint32_t)pos - (uint32_t)lo < span ? lane_key | kRare : kc) : kNoKey);
          const int e = (int)(m >> 27);
          const uint32_t bit = 1u << e;
          if (m & kRare) {
            if (m == kNoKey) {               // the rest of the batch stays in the bin
              frac = __shfl_sync(kFullMask, pos, nvalid - 1);
              break;
            }
            uint32_t fix = __shfl_sync(kFullMask, need, e);
            if (fix) {                       // move e takes its corrections
              const float4 h0 = h4, d0 = d4;
              const int dq0 = dq;
              for (; fix; fix &= fix - 1u) {
                const int j = __ffs(fix) - 1;
                const uint32_t bj = 1u << j;
                const float4 dj = C.ds[j];
                const float J = coupling(tc, bj);
                h4.x = fmaf(J, dj.x, h4.x);
                h4.y = fmaf(J, dj.y, h4.y);
                h4.z = fmaf(J, dj.z, h4.z);
                if (lane == e && (sc & bj)) {
                  replace(C.n[j]);
                  same |= bj;
                }
              }
              increment();
              if (lane != e) {               // the others wait for their turn
                h4 = h0;
                d4 = d0;
                dq = dq0;
              } else {
                need = 0u;
              }
              __syncwarp();
              const int more = __shfl_sync(kFullMask, dq - dq0, e);
              S += lane >= e ? (uint32_t)more : 0u;
              arm();
              continue;
            }
            const int pe = __shfl_sync(kFullMask, pos, e), de = __shfl_sync(kFullMask, dq, e);
            live = live && lane > e;
            if (admits(e, pe >> 24)) {
              const int db = pe >> 24;
              change_bin(e, db);
              pass();
              base -= (uint32_t)(db * kBin);
            } else {
              rej |= bit;
              need &= ~bit;
              base -= (uint32_t)de;
            }
          } else {
            rej |= bit;
            need &= ~bit;
            live = live && lane > e;
            base -= (uint32_t)((int)(m << 6) >> 6);
          }
        }
        acc_cur = every & ~rej;
      }
      // histogram: every move counts at the bin it leaves the walker in, i.e. the bin before the next move
      if (!frozen && valid) atomicAdd(&H_s[lane == 0 ? r : rb], 1u);
      n_rec += valid && ((uint32_t)hd.w & acc_cur) != 0u ? 1u : 0u;
      pub_prev = acc_cur;
      if ((uint32_t)all.y & acc_cur)       // moves superseded on their site by a later accepted one
        pub_prev &= ~__reduce_or_sync(kFullMask, (acc_cur >> lane) & 1u ? same : 0u);
      if (nvalid > 0) {
        n_scan += path == kScan ? 1 : 0;
        n_blocks += path == kBlocks ? 1 : 0;
        n_seq += path == kSequential ? 1 : 0;
      }
      n_in = __popc(acc_cur);
      n_exit = nvalid - n_in + n_chg;      // moves that left the bin, accepted or not
      A += (long long)nvalid * lnf_eff;
      n_acc += n_in;
      acc_prev = acc_cur;
      acc_prev_rev = __brev(acc_cur);
    }
    // the last batch's spins
    if (nb > 0) {
      if ((pub_prev >> lane) & 1u)
        lat.set_code(place_prev.x, make_float2(__int_as_float(place_prev.y), __int_as_float(place_prev.z)));
      __syncwarp();
      named_arrive(kBarDone + ((nb - 1) & 1));
    }
    const unsigned corrected = __reduce_add_sync(kFullMask, n_rec);
    if (lane == 0 && !bad) {
      a.st.efx[slot] = ((long long)(r + wlo) << 32) | (long long)(((uint32_t)frac << 8) | frac_low);
      lng_s[r] = A;
      a.st.steps[slot] = t0 + moves;
      a.st.accepts[slot] += n_acc;
      a.st.recomputes[slot] += corrected;
      a.st.path_batches[3 * (size_t)slot + 0] += n_scan;
      a.st.path_batches[3 * (size_t)slot + 1] += n_blocks;
      a.st.path_batches[3 * (size_t)slot + 2] += n_seq;
    }
   }
  }
  group_sync(bar_sync, nt);

  if constexpr (kSmem) copy_lattice(glat, lat, N, tid, nt);
  for (int w = tid; w < W; w += nt) {
    if constexpr (kTraj)
      a.st.lng[lbase + w] = order_value(lng_s[w]);
    else
      a.st.lng_fx[lbase + w] = lng_s[w];
    a.st.H[lbase + w] = H_s[w];
  }
  if constexpr (kTraj) {       // production: energy_update_kernel, after the walk
    if (recompute) {
      const double Ef = full_energy<kTraj>(a, off_s, lat, red, tid, nt, bar_sync);
      if (tid == 0) {
        const double d = fabs(Ef - a.st.E[slot]);
        if (d > a.st.drift[slot]) a.st.drift[slot] = d;
      }
    }
  }
}

// One CTA per slot; barrier 0 spans the CTA, 1..4 serve the pair.  Lattice in shared memory,
// arguments as kernel parameters.  The arena holds the lattice, so at bcc L = 16 one CTA fills an
// SM's shared memory; the register budget is left open (minimum one block per SM): bcc L = 16, 2 shells over its full
// range 3.86 ms with the 109 registers that it takes, 4.16 with the 79 of the default budget; L = 8, 3 shells
// converging 8.4 and 9.5 (127, 80).  (Small lattices fit 3 or 4 CTAs per SM by registers at this budget.)
template <bool kTraj, int NSH>
__global__ void __launch_bounds__(kWalkerThreads, 1) walker_pipe_kernel(const WalkerArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[kWalkerThreads / 32];
  pipe_walk_slot<kTraj, true, NSH>(a, blockIdx.x, a.moves, a.recompute, smem_raw, red, threadIdx.x, blockDim.x, 0, 1);
}

// The same over a lattice in global memory, with the arguments read from a device copy (through
// L1) and the per-launch moves and recompute flag as parameters.  On GB300 the bcc L = 32
// four-shell walker ran 25 % faster this way than with parameter arguments, while the
// shared-memory walker ran 3 % slower, so each keeps its own form.  Register budget: four blocks
// per SM (at most 128 registers), the residency that runs 512 walkers in one wave at 2048-entry tables.  (With four
// shells the default budget gives 128 as well, 9.97 against 9.96 ms of the full range; 96 with fewer.)
template <bool kTraj, int NSH>
__global__ void __launch_bounds__(kWalkerThreads, 4)
    walker_pipe_global_kernel(const WalkerArgs* __restrict__ ap, long long moves, int recompute) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[kWalkerThreads / 32];
  pipe_walk_slot<kTraj, false, NSH>(*ap, blockIdx.x, moves, recompute, smem_raw, red, threadIdx.x, blockDim.x, 0, 1);
}

// Persistent walker over many jobs: every 64-thread worker (resolver warp + producer warp) takes
// (job, slot) items from the work list until it is exhausted; a CTA holds `workers` workers, each
// with its own shared-memory arena and barriers (1 + 5w .. 5 + 5w).  A job's lattice sits in the
// arena or stays in global memory (L2) as its smem_lattice flag says.
// Register budget: at least two blocks of the largest shape per SM (at most 170 registers per
// thread; production spills nothing).  64 runs in a batch, 3 shells, three CTAs of two workers per SM: 30.2 ms with
// 168 registers, 30.0 with the 136 of the default budget, 33.5 with the 198 of an open one (two CTAs per SM); runs of
// L = 4, 5, 6 converging 12.3, 12.4 and 12.3.
template <bool kTraj, int NSH>
__global__ void __launch_bounds__(kBatchMaxWorkers * kWorkerThreads, 2)
    walker_batch_kernel(const WalkerArgs* __restrict__ jobs, const int2* __restrict__ items, int n_items, int* head,
                        long long moves, int recompute, unsigned arena) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[kBatchMaxWorkers][kWorkerThreads / 32];
  __shared__ int next[kBatchMaxWorkers];
  const int w = threadIdx.x / kWorkerThreads, wt = threadIdx.x % kWorkerThreads;
  const int bar_sync = 1 + 5 * w, bar_pair = 2 + 5 * w;
  unsigned char* mine = smem_raw + (size_t)w * arena;
  for (;;) {
    // every thread has read next[w] before the first barrier inside the walk, so the next write
    // cannot overtake a read
    if (wt == 0) next[w] = atomicAdd(head, 1);
    group_sync(bar_sync, kWorkerThreads);
    const int it = next[w];
    if (it >= n_items) break;
    const int2 js = items[it];
    const WalkerArgs& a = jobs[js.x];
    if (a.smem_lattice)
      pipe_walk_slot<kTraj, true, NSH>(a, js.y, moves, recompute, mine, red[w], wt, kWorkerThreads, bar_sync,
                                       bar_pair);
    else
      pipe_walk_slot<kTraj, false, NSH>(a, js.y, moves, recompute, mine, red[w], wt, kWorkerThreads, bar_sync,
                                        bar_pair);
  }
}

template <bool kTraj, int NSH>
static cudaError_t batch_kernel_setup(int workers, size_t arena, int* blocks_per_sm) {
  const size_t smem = (size_t)workers * arena;
  cudaError_t e = cudaFuncSetAttribute(walker_batch_kernel<kTraj, NSH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, walker_batch_kernel<kTraj, NSH>,
                                                       workers * kWorkerThreads, smem);
}

cudaError_t setup_walkers_batch(bool traj, int n_shells, int workers, size_t arena, int* blocks_per_sm) {
  if (workers < 1 || workers > kBatchMaxWorkers) return cudaErrorInvalidValue;
  switch (n_shells * 2 + (traj ? 1 : 0)) {
    case 2: return batch_kernel_setup<false, 1>(workers, arena, blocks_per_sm);
    case 3: return batch_kernel_setup<true, 1>(workers, arena, blocks_per_sm);
    case 4: return batch_kernel_setup<false, 2>(workers, arena, blocks_per_sm);
    case 5: return batch_kernel_setup<true, 2>(workers, arena, blocks_per_sm);
    case 6: return batch_kernel_setup<false, 3>(workers, arena, blocks_per_sm);
    case 7: return batch_kernel_setup<true, 3>(workers, arena, blocks_per_sm);
    case 8: return batch_kernel_setup<false, 4>(workers, arena, blocks_per_sm);
    case 9: return batch_kernel_setup<true, 4>(workers, arena, blocks_per_sm);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_walkers_batch(const BatchLaunch& b, cudaStream_t stream) {
  if (b.workers < 1 || b.workers > kBatchMaxWorkers || b.grid < 1) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(b.head, 0, sizeof(int), stream);
  if (e != cudaSuccess) return e;
  const dim3 grid(b.grid), block(b.workers * kWorkerThreads);
  const size_t smem = (size_t)b.workers * b.arena;
  const unsigned arena = (unsigned)b.arena;
#define REWL_BATCH_LAUNCH(T, S) \
  walker_batch_kernel<T, S><<<grid, block, smem, stream>>>(b.jobs, b.items, b.n_items, b.head, b.moves, b.recompute, arena)
  switch (b.n_shells * 2 + (b.traj ? 1 : 0)) {
    case 2: REWL_BATCH_LAUNCH(false, 1); break;
    case 3: REWL_BATCH_LAUNCH(true, 1); break;
    case 4: REWL_BATCH_LAUNCH(false, 2); break;
    case 5: REWL_BATCH_LAUNCH(true, 2); break;
    case 6: REWL_BATCH_LAUNCH(false, 3); break;
    case 7: REWL_BATCH_LAUNCH(true, 3); break;
    case 8: REWL_BATCH_LAUNCH(false, 4); break;
    case 9: REWL_BATCH_LAUNCH(true, 4); break;
    default: return cudaErrorInvalidValue;
  }
#undef REWL_BATCH_LAUNCH
  e = cudaGetLastError();
  if (e == cudaSuccess && b.recompute && !b.traj)
    e = launch_energy_update_batch(b.jobs, b.items, b.n_items, b.n_shells, kWorkerThreads, stream);
  return e;
}

size_t walker_pipe_smem_bytes(bool traj, bool smem_lattice, int N, int W, int own_entries) {
  const size_t lng = align16((traj ? sizeof(double) : sizeof(long long)) * (size_t)W);
  const size_t h = align16((size_t)W * 4);
  const size_t real = traj ? sizeof(double) : sizeof(float);
  size_t bytes = lng + h + 4 * kMaxSlotsPerSite + real * kMaxSlotsPerSite + batch_bytes(traj) + 8 * (size_t)own_entries;
  if (smem_lattice) bytes += smem_site_bytes(traj) * (size_t)N;
  return bytes;
}

bool walker_pipe_fits(bool traj, bool smem_lattice, int N, int W, int own_entries, size_t limit) {
  const size_t kRecordBytes = traj ? 5120 : 6144;
  return walker_pipe_smem_bytes(traj, smem_lattice, N, W, own_entries) - batch_bytes(traj) + kRecordBytes <= limit;
}

int walker_pipe_table(bool traj, bool smem_lattice, int N, int W, int own_entries, size_t limit) {
  static_assert(batch_bytes(true) <= 5120 && batch_bytes(false) <= 6144 + 8 * (256 - 64), "a table of 256 entries gives way");
  while (own_entries > 64 && walker_pipe_smem_bytes(traj, smem_lattice, N, W, own_entries) > limit) own_entries /= 2;
  return own_entries;
}

template <bool kTraj, int NSH>
static cudaError_t launch_pipe_t(const WalkerArgs& a, const WalkerArgs* d_args, int n_slots, size_t smem,
                                 cudaStream_t stream) {
  if (d_args) {
    cudaError_t e = cudaFuncSetAttribute(walker_pipe_global_kernel<kTraj, NSH>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    walker_pipe_global_kernel<kTraj, NSH><<<n_slots, kWalkerThreads, smem, stream>>>(d_args, a.moves, a.recompute);
  } else {
    cudaError_t e = cudaFuncSetAttribute(walker_pipe_kernel<kTraj, NSH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    walker_pipe_kernel<kTraj, NSH><<<n_slots, kWalkerThreads, smem, stream>>>(a);
  }
  return cudaGetLastError();
}

template <bool kTraj>
static cudaError_t launch_pipe_shells(const WalkerArgs& a, const WalkerArgs* d_args, int n_slots, size_t smem,
                                      cudaStream_t stream) {
  switch (a.geo.n_shells) {
    case 1: return launch_pipe_t<kTraj, 1>(a, d_args, n_slots, smem, stream);
    case 2: return launch_pipe_t<kTraj, 2>(a, d_args, n_slots, smem, stream);
    case 3: return launch_pipe_t<kTraj, 3>(a, d_args, n_slots, smem, stream);
    case 4: return launch_pipe_t<kTraj, 4>(a, d_args, n_slots, smem, stream);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_walkers_pipe(const WalkerArgs& a, const WalkerArgs* d_args, int n_slots, bool traj, size_t smem,
                                cudaStream_t stream) {
  if (a.smem_lattice == (d_args != nullptr)) return cudaErrorInvalidValue;
  if (traj) return launch_pipe_shells<true>(a, d_args, n_slots, smem, stream);
  const cudaError_t e = launch_pipe_shells<false>(a, d_args, n_slots, smem, stream);
  return e == cudaSuccess && a.recompute ? launch_energy_update(a, n_slots, stream) : e;
}

}  // namespace rewl
