// Colour passes of the FP64 multigrid with the neighbour sums on the integer pipe
// (the fixed-point form and its unit: fixed.cuh), for the larger levels.
//
// One kernel for the passes of a Gauss-Seidel sweep and those that follow it:
//   FC_SWEEP  phi = x_GS on one colour, in place (its neighbours have other colours)
//   FC_OPEN   the same on colour 0, opening a step
//   FC_LAG    the same on colour 0, keeping the old values (packed at index / 2) and
//             the sum of delta^2, delta = x_GS - x_old: the lagged convergence check
//   FC_RESID  delta on every colour but the last, zero on the last (after a sweep)
//   FC_NORM   the sum of delta^2 over those colours
// 7-point (two colours, equal or unequal spacings) and 13-point (three colours,
// equal spacings).  Planes of phi (with a halo of G) and of fs come through a TMA
// ring; an arriving plane of phi is turned into units in a ring of 2 G + 2 work
// planes, and each lane takes the group of 2 (3) consecutive nodes of its row and
// updates the member of the pass's colour from the work planes around.  FP64 is
// left with one FMA per update (three for unequal spacings) instead of 5 or 10.
// x_GS = c S + fs with S the exact sum, delta from the second differences
// (S - 6 C and the like): both are nearer the exact values than the FP64 chains.
//
// A pass reads phi and fs once and writes a part of phi: on 256^3, 134 + 134 MB in
// and 134 out (whole lines), 59 us at the copy rate.  Measured (us a pass under ncu;
// FP64 diagonal walks before): 256^3 88 -> 75, with the lag 131 -> 102, residual
// 104 -> 79; 160 x 112 x 208 unequal spacings 32.7 -> 27.7; 13-point 192^3 54.7 -> 36.8,
// residual 113 -> 51, norm 131 -> 55; 96^3 sweeps 11.1 (walks 10.2), with the lag
// 15.5, residual 11.5, its solve 1920 -> 1879.  Bound by the memory system at 78 % of
// the copy rate on the largest levels (half of the issue slots busy, 4 us of it for
// rounding the values to nearest), on the smallest by the chain of TMA wait,
// barrier and update from plane to plane.
//
// Bounds.  H: the largest of |phi| as last tracked, the boundary data and |fs|,
// below 2^57 units (13-point 2^56).  A 7-point update is a mean of its neighbours
// plus fs, so a pass adds at most H to the largest value: 7 H after the three sweeps
// that fx_sweeps_fit allows between two trackings, sums of six below 42 H < 2^63.
// The 13-point weights' magnitudes add up to 102 / 90: after two sweeps (six passes)
// values are below 10.6 H, sums of six and S1 - 6 C below 127.2 H < 2^63.
// The 7-point S - 6 C has a closer bound, because residuals are formed after a sweep
// at least: C = S' / 6 + fs with S' the neighbours' sum of the time, so S - 6 C =
// (S - S') - 6 fs.  In its first pass after the tracking a node changes by at most
// 3 H (first colour) or 4 H (second), in a later one by the mean of its
// neighbours' last changes, 4 H again: |S - S'| <= 24 H, |S - 6 C| <= 30 H < 2^62.  Unequal
// spacings form u(-1) + u(1) - 2 C per axis, below 28 H.
#include "fixed.cuh"

#include "cart_kernels.cuh"
#include "fixed_sweeps.cuh"
#include "stencil.cuh"

namespace ps {

template <int KIND, int RR, int NSS>
struct FcGeom {
  static constexpr int G = KIND == FX13 ? 2 : 1, NCOL = G + 1;
  static constexpr int NW = 8, R = RR;   // warps, rows per warp
  static constexpr int TX = 32 * NCOL, TY = NW * R, NT = 32 * NW;
  static constexpr int WX = TX + 2 * G, WY = TY + 2 * G, NEL = WX * WY, NLD = (NEL + NT - 1) / NT;
  static constexpr int XC = KIND == FX13 ? 1 : 0;          // binades of the unit above fixed.cuh's
  static constexpr int ND = 2 * G + 2, NS = NSS;             // work planes, TMA stages
  static constexpr int UB = align_up(NEL * 8, 128), BB = align_up(WX * TY * 8, 128);
  static constexpr int SMEM = NS * (UB + BB) + ND * UB + NS * 8;
};

// v in units of 2^(eb - 1079 + C), for values up to 2^C times 16 H, rounded to
// nearest, ties away from zero: an update keeps the sum of its neighbours, so a
// one-sided rounding of the values below H / 16 (those above are exact) is a source
// all over the faint part of a field, which the coarse levels sum up.
// R.m.s. error of one V-cycle from a peak of 10^4 over values of 1 (96 x 112 x 80,
// 7- / 13-point): 2.6e-11 / 4.8e-11 truncated, 4.6e-13 / 7.1e-13 as here, 1.3e-12 /
// 2.6e-12 of the FP64 passes.
template <int C>
__device__ __forceinline__ long long fx_from_wide(double v, int eb) {
  const int hi = __double2hiint(v);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned long long m =
      ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(v)) << 9;
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(eb + 4 + C - e));   // shifts past 63 give 0
  const long long s = (long long)(hi >> 31);
  return ((long long)((r + 1) >> 1) ^ s) - s;
}

// The same from three bits below the unit, where three to five eighths go to the even
// neighbour: as often up as down for values in general and for exact ties.  Where
// fs is zero a 7-point mean on equal spacings is a whole number of sixths of a unit,
// every sixth a tie.
__device__ __forceinline__ long long fx_from_even(double v, int eb) {
  const int hi = __double2hiint(v);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned long long m =
      ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(v)) << 11;
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(eb + 4 - e));
  const long long s = (long long)(hi >> 31);
  return ((long long)((r + 3u + ((unsigned)r >> 2 & 2u)) >> 3) ^ s) - s;
}

// 16 a - b as a double (the sum may exceed 64 bits)
__device__ __forceinline__ double fx_sum13(long long a, long long b) {
  return fx_two_limbs(((a >> 32) << 4) - (b >> 32), ((long long)(unsigned)a << 4) - (long long)(unsigned)b);
}

template <int KIND, bool ISO, int MODE, typename W, typename Gm>
__device__ __forceinline__ bool fc_march(const CUtensorMap& mU, const CUtensorMap& mB, const Dims& d, double cx, double cy,
                                         double cz, const FxScale& sc, int zc, int colour, double* phi, double* out,
                                         unsigned char* smem, double& s2, unsigned& hmax) {
  constexpr int G = Gm::G, NCOL = Gm::NCOL, R = Gm::R, WX = Gm::WX, NEL = Gm::NEL, NLD = Gm::NLD, NT = Gm::NT;
  constexpr int NS = Gm::NS, ND = Gm::ND, UE = Gm::UB / 8, BE = Gm::BB / 8;
  constexpr bool FX = !std::is_same<W, double>::value;
  constexpr int NC = MODE == FC_RESID || MODE == FC_NORM ? NCOL - 1 : 1;   // colours evaluated
  double* const ring = reinterpret_cast<double*>(smem);
  double* const bring = reinterpret_cast<double*>(smem + NS * Gm::UB);
  W* const work = reinterpret_cast<W*>(smem + NS * (Gm::UB + Gm::BB));
  unsigned long long* const bar = reinterpret_cast<unsigned long long*>(smem + NS * (Gm::UB + Gm::BB) + ND * Gm::UB);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i0 = blockIdx.x * Gm::TX + G, j0 = blockIdx.y * Gm::TY + G;
  const int k0 = blockIdx.z * zc + G, k1 = min(k0 + zc, G + d.nk());
  const int zl = k0 - G, zh = k1 - 1 + G;
  if (tid == 0) {
    for (int q = 0; q < NS; q++) mbar_init(&bar[q], 1);
    fence_mbar_init();
  }
  __syncthreads();
  auto issue = [&](int z, int q) {   // thread 0: stage q <- phi(z) and fs(z - G)
    if (z > zh) return;
    const bool withb = z - G >= k0;
    mbar_expect_tx(&bar[q], NEL * 8 + (withb ? WX * Gm::TY * 8 : 0));
    tma_load_3d(ring + q * UE, &mU, i0 - G, j0 - G, z, &bar[q]);
    if (withb) tma_load_3d(bring + q * BE, &mB, i0 - G, j0, z - G, &bar[q]);
  };
  if (tid == 0)
    for (int q = 0; q < NS; q++) issue(zl + q, q);
  if constexpr (FX) {
    const double u = sc.unit() * (1 << Gm::XC);
    cx *= u;
    cy *= u;
    cz *= u;
  }
  bool ok = true;
  int wq = 0, cw = ND - 1;   // stage and work plane of the plane that arrived last
  unsigned wph = 0;
  const int jr = j0 + warp * R;   // array row of the warp's first row
  // bit q: the thread's q-th staged node is interior in x and y (boundary nodes are
  // bounded by themselves, and some are read by no stencil) / has colour 1 in the
  // planes of even z (the colour-0 nodes may be written meanwhile; they are tracked
  // as they are written)
  unsigned inner = 0u, black = 0u;
  if constexpr (MODE == FC_LAG || MODE == FC_NORM) {
#pragma unroll
    for (int q = 0; q < NLD; q++) {
      const int el = tid + q * NT, x = i0 - G + el % WX, y = j0 - G + el / WX;
      inner |= (unsigned)(x >= G && x < G + d.ni() && y >= G && y < G + d.nj()) << q;
      black |= (unsigned)((x + y) & 1) << q;
    }
  }
  for (int z = zl; z <= zh; z++) {
    const int k = z - G;
    const bool active = k >= k0;
    // the old values of this step's nodes, in flight during the wait
    double old[R];
    if constexpr (MODE == FC_LAG) {
#pragma unroll
      for (int r = 0; r < R; r++) {
        const int j = jr + r, m = ((colour - (i0 - G + 1) - (j - G + 1) - (k - G + 1)) % NCOL + NCOL) % NCOL;
        const int i = i0 + NCOL * lane + m;
        old[r] = active && j < G + d.nj() && i < G + d.ni() ? phi[d.at(i, j, k)] : 0.0;
      }
    }
    mbar_wait(&bar[wq], wph, ok);
    cw = cw + 1 == ND ? 0 : cw + 1;
    {
      const double* raw = ring + wq * UE;
      W* w = work + cw * UE;
#pragma unroll
      for (int q = 0; q < NLD; q++)
        if ((q + 1) * NT <= NEL || tid + q * NT < NEL) {
          const double v = raw[tid + q * NT];
          if constexpr (FX && KIND == FX7 && ISO) w[tid + q * NT] = fx_from_even(v, sc.eb);
          else if constexpr (FX) w[tid + q * NT] = fx_from_wide<Gm::XC>(v, sc.eb);
          else w[tid + q * NT] = v;
          if ((MODE == FC_NORM || (MODE == FC_LAG && ((black >> q ^ z) & 1))) && (inner >> q & 1u) && z >= G && z < G + d.nk())
            hmax = max(hmax, (unsigned)__double2hiint(v) & 0x7fffffffu);
        }
    }
    __syncthreads();
    if (tid == 0 && ok && z > zl) {   // after a failed wait no new copy is issued
      fence_proxy_async();
      issue(z - 1 + NS, wq == 0 ? NS - 1 : wq - 1);
    }
    const double* fb = bring + wq * BE;
    if (++wq == NS) {
      wq = 0;
      wph ^= 1u;
    }
    if (!active) continue;
    auto plane = [&](int back) { return work + (cw - back < 0 ? cw - back + ND : cw - back) * UE; };
    const W* P = plane(G);
    const W* A1 = plane(G - 1);
    const W* B1 = plane(G + 1);
    const W* A2 = G == 2 ? plane(0) : nullptr;
    const W* B2 = G == 2 ? plane(4) : nullptr;
    double x[R][NC], dl[R][NC];
    int at[R][NC];
    long long node[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int j = jr + r;
      node[r] = d.at(i0 + NCOL * lane, j, k);
#pragma unroll
      for (int q = 0; q < NC; q++) {
        const int c = MODE == FC_RESID || MODE == FC_NORM ? q : colour;
        const int m = ((c - (i0 - G + 1) - (j - G + 1) - (k - G + 1)) % NCOL + NCOL) % NCOL;   // uniform over the warp
        at[r][q] = m;
        const int a = (j - j0 + G) * WX + G + NCOL * lane + m;
        const double f = fb[(j - j0) * WX + G + NCOL * lane + m];
        const W C = P[a];
        const W ew = P[a + 1] + P[a - 1], ns = P[a + WX] + P[a - WX], ud = A1[a] + B1[a];
        if constexpr (!FX) {   // residuals as x_GS - x: zero where a sweep would change nothing
          const W S = (ew + ns) + ud;
          if constexpr (KIND == FX13) {
            const W S2 = ((P[a + 2] + P[a - 2]) + (P[a + 2 * WX] + P[a - 2 * WX])) + (A2[a] + B2[a]);
            x[r][q] = fma(fma(16.0, S, -S2), cx, f);
          } else if constexpr (ISO) {
            x[r][q] = fma(S, cx, f);
          } else {
            x[r][q] = fma(ew, cx, fma(ns, cy, fma(ud, cz, f)));
          }
          dl[r][q] = x[r][q] - C;
        } else if constexpr (KIND == FX13) {
          const W S1 = (ew + ns) + ud;
          const W S2 = ((P[a + 2] + P[a - 2]) + (P[a + 2 * WX] + P[a - 2 * WX])) + (A2[a] + B2[a]);
          if (MODE == FC_SWEEP || MODE == FC_OPEN || MODE == FC_LAG) x[r][q] = fma(fx_sum13(S1, S2), cx, f);
          if (MODE != FC_SWEEP && MODE != FC_OPEN) dl[r][q] = fma(fx_sum13(S1 - C * 6, S2 - C * 6), cx, f);
        } else if constexpr (ISO) {
          const W S = (ew + ns) + ud;
          if (MODE == FC_SWEEP || MODE == FC_OPEN || MODE == FC_LAG) x[r][q] = fma(fx_double(S), cx, f);
          if (MODE != FC_SWEEP && MODE != FC_OPEN) dl[r][q] = fma(fx_double(S - C * 6), cx, f);
        } else {
          if (MODE == FC_SWEEP || MODE == FC_OPEN || MODE == FC_LAG)
            x[r][q] = fma(fx_double(ew), cx, fma(fx_double(ns), cy, fma(fx_double(ud), cz, f)));
          if (MODE != FC_SWEEP && MODE != FC_OPEN) {
            const W c2 = C + C;
            dl[r][q] = fma(fx_double(ew - c2), cx, fma(fx_double(ns - c2), cy, fma(fx_double(ud - c2), cz, f)));
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; r++) {
      if (jr + r >= G + d.nj()) continue;
#pragma unroll
      for (int q = 0; q < NC; q++) {
        const int i = i0 + NCOL * lane + at[r][q];
        if (i >= G + d.ni()) continue;
        const long long p = node[r] + at[r][q];
        if (MODE == FC_SWEEP || MODE == FC_OPEN || MODE == FC_LAG) phi[p] = x[r][q];
        if (MODE == FC_LAG) {
          out[p >> 1] = old[r];
          hmax = max(hmax, (unsigned)__double2hiint(x[r][q]) & 0x7fffffffu);
        }
        if (MODE == FC_RESID) out[p] = dl[r][q];
        if (MODE == FC_LAG || MODE == FC_NORM) s2 = fma(dl[r][q], dl[r][q], s2);
      }
      if (MODE == FC_RESID) {   // the last colour's member
        const int m = ((NCOL - 1 - (i0 - G + 1) - (jr + r - G + 1) - (k - G + 1)) % NCOL + NCOL) % NCOL;
        if (i0 + NCOL * lane + m < G + d.ni()) out[node[r] + m] = 0.0;
      }
    }
  }
  return ok;
}

template <int KIND, bool ISO, int MODE, typename Gm>
__global__ void __launch_bounds__(256, 227 * 1024 / (Gm::SMEM + 1024) > 4 ? 4 : 227 * 1024 / (Gm::SMEM + 1024))
    k_fc_pass(const __grid_constant__ CUtensorMap mU, const __grid_constant__ CUtensorMap mB, Dims d, double cx, double cy,
              double cz, int zc, int colour, double* phi, double* out, DevState* __restrict__ st,
              const unsigned* __restrict__ h1, const unsigned* __restrict__ h2, const unsigned* __restrict__ h3,
              unsigned* __restrict__ track, double* __restrict__ partials) {
  extern __shared__ __align__(128) unsigned char fc_smem[];
  if ((MODE == FC_LAG || MODE == FC_OPEN) && st->done) return;   // uniform over the grid
  if (MODE == FC_OPEN && block_linear_id() == 0 && threadIdx.x == 0) st->lag_pending = 1;
  // the pass that opens a step forms the values of the lagged pass again, in its arithmetic
  const FxScale sc(max(*h1, max(*h2, *h3)), MODE == FC_OPEN ? st->lexact : st->exact);
  double s2 = 0.0;
  unsigned hmax = 0u;
  const bool ok =
      sc.fx ? fc_march<KIND, ISO, MODE, long long, Gm>(mU, mB, d, cx, cy, cz, sc, zc, colour, phi, out, fc_smem, s2, hmax)
            : fc_march<KIND, ISO, MODE, double, Gm>(mU, mB, d, cx, cy, cz, sc, zc, colour, phi, out, fc_smem, s2, hmax);
  if (!ok) atomicExch(&st->fault, 1);
  if constexpr (MODE == FC_LAG || MODE == FC_NORM) {
    __shared__ double sh[256];
    if (track != nullptr) atomic_max_group(hmax, track);
    s2 = block_sum_warp0(s2, threadIdx.x, 256, sh);
    if (threadIdx.x == 0) {
      const int b = block_linear_id();
      partials[2 * b] = s2;
      partials[2 * b + 1] = 0.0;
    }
  }
}

template <int KIND, bool ISO, int MODE, typename Gm>
static cudaError_t fc_v(const Dims& d, const Coef<double>& cf, int colour, double* phi, const double* fs, double* out,
                        DevState* st, const FcBounds& b, double* partials, int* nblocks, cudaStream_t s) {
  static PerDevice cached;
  int occ = 0, zc = 0;
  const cudaError_t e = resident_blocks(k_fc_pass<KIND, ISO, MODE, Gm>, 256, Gm::SMEM, cached, &occ);
  if (e != cudaSuccess) return e;
  CUtensorMap mU, mB;
  if (!encode_level_map(&mU, DT_F64, phi, d, Gm::WX, Gm::WY) || !encode_level_map(&mB, DT_F64, fs, d, Gm::WX, Gm::TY))
    return cudaErrorInvalidValue;
  const dim3 grid = fx_chunks((d.ni() + Gm::TX - 1) / Gm::TX, (d.nj() + Gm::TY - 1) / Gm::TY, d.nk(), occ, 4, &zc);
  if (nblocks) *nblocks = (int)(grid.x * grid.y * grid.z);
  // 13-point: c1 = 16 c, c2 = -c
  const double cx = KIND == FX13 ? cf.c1[0] / 16.0 : cf.c1[0];
  k_fc_pass<KIND, ISO, MODE, Gm><<<grid, 256, Gm::SMEM, s>>>(mU, mB, d, cx, cf.c1[1], cf.c1[2], zc, colour, phi, out, st,
                                                          b.phi, b.boundary, b.fs, b.track, partials);
  return cudaGetLastError();
}

template <int KIND, bool ISO, int MODE>
static cudaError_t fc_t(const Dims& d, const Coef<double>& cf, int colour, double* phi, const double* fs, double* out,
                        DevState* st, const FcBounds& b, double* partials, int* nblocks, cudaStream_t s) {
  // 7-point, more than 3 10^6 nodes: 64 x 16 tiles (halo 1.16 instead of 1.29 of the
  // nodes; 256^3: 70.5 us against 72.1, with the lag 92 against 104); below, and
  // 13-point: tiles of 8 rows and one more stage (128^3 12.9 us against 13.7, 96^3
  // 9.3 against 11.1; 13-point 192^3 33.5 against 43.9 with two stages, 50 with 16 rows;
  // all of these with truncated values, 4 to 10 % below the passes' present times)
  if (KIND == FX7 && (long long)d.ni() * d.nj() * d.nk() > 3000000)
    return fc_v<KIND, ISO, MODE, FcGeom<KIND, 2, 2>>(d, cf, colour, phi, fs, out, st, b, partials, nblocks, s);
  return fc_v<KIND, ISO, MODE, FcGeom<KIND, 1, 3>>(d, cf, colour, phi, fs, out, st, b, partials, nblocks, s);
}

int fc_partials(const Dims& d) {   // at least the blocks of any pass
  const long long tiles = (d.ni() + 63) / 64 * (long long)((d.nj() + 7) / 8);
  return (int)(8LL * device_sm_count() + (d.nk() + 95) / 96 * tiles);
}

bool fc_level(const Dims& d, int order, const double h[3]) {
  return fx_level(d) && (order == 2 || (h[0] == h[1] && h[1] == h[2]));
}

cudaError_t launch_fc_pass(const Dims& d, int order, const double h[3], int mode, int colour, double* phi,
                           const double* fs, double* out, DevState* st, const FcBounds& b, double* partials, int* nblocks,
                           cudaStream_t s) {
  if (!fc_level(d, order, h) || d.g != order / 2) return cudaErrorInvalidValue;
  const Coef<double> cf = make_coef<double>(d, h, order);
  const bool iso = h[0] == h[1] && h[1] == h[2];
#define PS_FC(MODE)                                                                                          \
  case MODE:                                                                                                 \
    if (order == 4) return fc_t<FX13, true, MODE>(d, cf, colour, phi, fs, out, st, b, partials, nblocks, s); \
    return iso ? fc_t<FX7, true, MODE>(d, cf, colour, phi, fs, out, st, b, partials, nblocks, s)             \
               : fc_t<FX7, false, MODE>(d, cf, colour, phi, fs, out, st, b, partials, nblocks, s);
  switch (mode) {
    PS_FC(FC_SWEEP)
    PS_FC(FC_RESID)
    PS_FC(FC_NORM)
    case FC_OPEN:
      if (order != 2 || !iso) return cudaErrorInvalidValue;
      return fc_t<FX7, true, FC_OPEN>(d, cf, 0, phi, fs, out, st, b, partials, nblocks, s);
    case FC_LAG:
      if (order != 2 || !iso || (d.sy() & 1) || (d.sz() & 1)) return cudaErrorInvalidValue;
      return fc_t<FX7, true, FC_LAG>(d, cf, 0, phi, fs, out, st, b, partials, nblocks, s);
  }
#undef PS_FC
  return cudaErrorInvalidValue;
}

}  // namespace ps
