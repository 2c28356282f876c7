// FP64 stencil values with the sums over neighbours on the integer pipe.
//
// GB300 issues about 1.7 FP64 instructions a cycle and SM against 128 integer
// ones, so a residual pass that adds 6, 12 or 26 neighbours in FP64 is bound by
// that pipe at a fraction of the memory bandwidth.  Here each value is turned
// once, as its plane is staged in shared memory, into a 64-bit fixed-point
// number with one unit for the whole pass, and the neighbours are added
// exactly: per node two FP64 instructions are left (the sum converted back, and
// one FMA with the weight and the right-hand side).
//
// The unit.  With H the largest |u| of the pass (its high word, kept in the
// solver state by the kernels that write u), values are below 2^57 units, so a
// unit is 2^-4 of the last place of H's binade: 1/8 of the largest rounding
// error of one FP64 addition near H.  The 7- and 13-point operators annihilate
// constants, and their sums are formed as second differences,
//   7-point   T = S1 - 6 C
//   13-point  T = 16 (S1 - 6 C) - (S2 - 6 C)      (S1, S2: distance 1, 2)
// each group of which is below 12 H < 2^61 units.  The weighted sum may not be
// for a field that changes by more than H from node to node; then (a test on the
// high words) the groups are converted and weighted in FP64 one by one.  The
// 27-point sums
//   T = w0 C + w1 faces + w2 edges + w3 corners   (integer weights)
// are formed exactly in two limbs, low and high words multiplied apart (wide
// 32-bit multiply-adds), and the leading 62 bits converted.  What is lost is
// the part of a value below a unit: against the roundings of an FP64 sum of
// values of size |u| the error is smaller wherever |u| > H / 16, and over a field
// whenever its r.m.s. is (potentials of extended sources are; a source of a few
// nodes has its peak 100 r.m.s. high, and its faint parts keep that many fewer bits).
//
// The floor.  What the units leave in a residual bounds how far a solve can
// converge, at 1e-14 relative for a point source on 256^3, where FP64 sums reach
// 6e-16.  So the norm finisher compares each residual norm with the units' share
// (fx_noise of the operator, times H) and, from FX_FLOOR times that share on, the passes
// run the same march in FP64 (st->exact): no convergence factor is lost on the
// way, and the accuracy that can be reached is that of the FP64 sums.  Passes whose H
// is infinite, NaN or near the ends of the exponent range do so as well.
#pragma once
#include <type_traits>

#include "per_device.cuh"
#include "tma.cuh"

namespace ps {

// Exponent field of the pass's largest |u| from its high word; fx: the range in
// which the fixed-point form is used.
struct FxScale {
  int eb;
  bool fx;
  __device__ __forceinline__ explicit FxScale(unsigned hmax, int exact) {
    eb = (int)(hmax >> 20);
    fx = !exact && (hmax == 0u || (eb >= 200 && eb <= 0x7f0));
    if (hmax == 0u) eb = 1023;   // every value is zero
  }
  // one unit as a binary64: 2^(eb - 1079)
  __device__ __forceinline__ double unit() const { return __longlong_as_double((long long)(eb - 56) << 52); }
};

// v in units of 2^(eb - 1079), truncated towards zero: the significand (with its
// implicit bit) shifted left by 4 and right by the distance of the exponents.
// Zeros and subnormals are more than 64 binades below and become 0 or -1.
__device__ __forceinline__ long long fx_from(double v, int eb) {
  const int hi = __double2hiint(v);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned long long m =
      ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(v)) << 4;
  long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(eb - e));   // shifts past 63 give 0
  const int s = hi >> 31;
  const unsigned long long x = (unsigned long long)r ^ ((unsigned long long)(unsigned)s << 32 | (unsigned)s);
  return (long long)x;   // one's complement of a negative value: half a unit at most from its negation
}

// The binary64 of an integer, rounded to nearest (half away from zero), on the
// integer pipe: the conversion instruction takes a slot of the FP64 pipe and
// its latency.
__device__ __forceinline__ double fx_double(long long v) {
  const int s = (int)(v >> 63);
  const unsigned long long a = (unsigned long long)((v ^ (long long)s) - (long long)s);
  const int lz = __clzll((long long)a);   // 1 .. 64
  const unsigned long long m = ((a << (lz - 1)) + 512u) >> 10;   // implicit bit at 52 (53 after a carry)
  const unsigned hi = (unsigned)(m >> 32) + ((unsigned)(1085 - lz) << 20);
  return a == 0 ? 0.0 : __hiloint2double((int)(hi | ((unsigned)s & 0x80000000u)), (int)(unsigned)m);
}

// H 2^32 + L, up to 2^93 in size, as a double: exact up to its 62 leading bits.
__device__ __forceinline__ double fx_two_limbs(long long H, long long L) {
  H += L >> 32;
  // shifted right by 11 unless it fits 63 bits
  const bool big = (unsigned long long)(H + (1LL << 30)) >= (1ull << 31);
  const unsigned low = (unsigned)L;
  const long long t = big ? (long long)((unsigned long long)H << 21 | low >> 11)
                          : (long long)((unsigned long long)H << 32 | low);
  const double v = fx_double(t);
  return __hiloint2double(__double2hiint(v) + (big ? 11 << 20 : 0), __double2loint(v));
}

// |x| < 2^(32 + b), from the high word
__device__ __forceinline__ bool fx_below(long long x, int b) {
  return (unsigned)((int)(x >> 32) + (1 << b)) < (2u << b);
}

// y[r] = x[r] * 2^e rounded to FP32 (f64_to_f32_pow2), without branches for
// values whose result is normal or zero.
template <int R>
__device__ __forceinline__ void fx_to_f32(const double (&x)[R], int e, float (&y)[R]) {
  bool plain = true;
#pragma unroll
  for (int r = 0; r < R; r++) {
    const unsigned hi = (unsigned)__double2hiint(x[r]), lo = (unsigned)__double2loint(x[r]);
    const int ex = (int)(hi >> 20) & 0x7ff, fe = ex + (127 - 1023 + e);
    const unsigned m = __funnelshift_r(lo, hi, 29) & 0x7fffffu;
    // ties to even: the 29 dropped bits plus just under half, plus one where the kept part is odd
    const unsigned up = ((lo & 0x1fffffffu) + 0x0fffffffu + (m & 1u)) >> 29;
    const unsigned mag = ex == 0 ? 0u : ((unsigned)fe << 23) + m + up;
    plain &= ex == 0 || (unsigned)(fe - 1) < 254u;
    y[r] = __uint_as_float((hi & 0x80000000u) | mag);
  }
  if (!plain)
    for (int r = 0; r < R; r++) y[r] = f64_to_f32_pow2(x[r], e);
}

enum { FX7 = 7, FX13 = 13, FX27 = 27 };

// Operator of a pass: value = base + c T.  27-point: integer weights of T, w1 to
// w3 >= 0, with |w0| + 6 w1 + 12 w2 + 8 w3 <= FX_WSUM.
constexpr int FX_WSUM = 65536;
struct FxOp {
  double c;
  int w0, w1, w2, w3;
};

template <int KIND>
struct FxGeom {
  static constexpr int G = KIND == FX13 ? 2 : 1;
  static constexpr int TX = 64, TROWS = 4, R = 4;   // a thread owns R rows of one column
  static constexpr int TY = TROWS * R, NT = TX * TROWS;
  static constexpr int WX = TX + 2 * G, WY = TY + 2 * G, NEL = WX * WY;   // staged plane of u
  static constexpr int NLD = (NEL + NT - 1) / NT;
  static constexpr int NS = 3;                                           // stages of the TMA ring
  static constexpr int UB = align_up(NEL * 8, 128), BB = align_up(WX * TY * 8, 128);
  static constexpr int SMEM = NS * (UB + BB) + 2 * UB + NS * 8;
};

// A pass over the interior nodes: FP64 planes of u (with a halo of G) and of the
// right-hand side come through a TMA ring, the plane of u that has arrived is
// turned into units in one of two work buffers, and each thread forms the
// in-plane groups of its R rows from there and keeps the groups of the planes
// around in registers.  Per plane epi(offset, pitch, inside, values, bases) takes
// the thread's R nodes, node r at offset + r pitch, interior where inside[r].
// One barrier a plane: it separates the writes of a work buffer from its reads
// two planes earlier, and hands the stage of the previous plane back to the
// copy engine.
// Epi::LAYERS: epi.layer[r] says whether node r lies on the first or last layer of an axis.
// Epi::TRACK: epi.hmax takes the high word of the largest |u| of the interior nodes
// staged (the tile's own and their neighbours; not the boundary's, some of which
// no stencil reads).
template <int KIND, typename W, typename Epi>
__device__ __forceinline__ bool fx_march(const CUtensorMap& mU, const CUtensorMap& mB, const Dims& d, const FxOp& op,
                                         const FxScale& sc, int zc, unsigned char* smem, Epi& epi) {
  using Gm = FxGeom<KIND>;
  constexpr int G = Gm::G, R = Gm::R, WX = Gm::WX, NEL = Gm::NEL, NLD = Gm::NLD, NT = Gm::NT, NS = Gm::NS;
  constexpr bool FX = !std::is_same<W, double>::value;
  constexpr int UE = Gm::UB / 8, BE = Gm::BB / 8;
  double* const ring = reinterpret_cast<double*>(smem);
  double* const bring = reinterpret_cast<double*>(smem + NS * Gm::UB);
  W* const work = reinterpret_cast<W*>(smem + NS * (Gm::UB + Gm::BB));
  unsigned long long* const bar = reinterpret_cast<unsigned long long*>(smem + NS * (Gm::UB + Gm::BB) + 2 * Gm::UB);
  const int tid = threadIdx.x, tx = tid & (Gm::TX - 1), ty = tid / Gm::TX;
  const int i0 = blockIdx.x * Gm::TX + G, j0 = blockIdx.y * Gm::TY + G;
  const int k0 = blockIdx.z * zc + G, k1 = min(k0 + zc, G + d.nk());
  const int zl = k0 - G, zh = k1 - 1 + G;   // planes of u
  if (tid == 0) {
    for (int q = 0; q < NS; q++) mbar_init(&bar[q], 1);
    fence_mbar_init();
  }
  __syncthreads();
  auto issue = [&](int z, int q) {   // thread 0: stage q <- u(z) and base(z - G)
    if (z > zh) return;
    const bool withb = z - G >= k0;
    mbar_expect_tx(&bar[q], NEL * 8 + (withb ? WX * Gm::TY * 8 : 0));
    tma_load_3d(ring + q * UE, &mU, i0 - G, j0 - G, z, &bar[q]);
    if (withb) tma_load_3d(bring + q * BE, &mB, i0 - G, j0, z - G, &bar[q]);
  };
  if (tid == 0)
    for (int q = 0; q < NS; q++) issue(zl + q, q);
  bool ok = true;
  int wq = 0, wb = 0;
  unsigned wph = 0;
  const int jr = j0 + ty * R;
  bool in[R];
#pragma unroll
  for (int r = 0; r < R; r++) in[r] = i0 + tx < G + d.ni() && jr + r < G + d.nj();
  long long at = d.at(i0 + tx, jr, k0);
  unsigned inner = 0u;   // bit q: the thread's q-th staged node is interior in x and y
  if constexpr (Epi::TRACK) {
#pragma unroll
    for (int q = 0; q < NLD; q++) {
      const int el = tid + q * NT, x = i0 + el % WX, y = j0 + el / WX;   // + G
      inner |= (unsigned)(x >= 2 * G && x < 2 * G + d.ni() && y >= 2 * G && y < 2 * G + d.nj()) << q;
    }
  }
  // in-plane groups of a staged plane: C centre; F the four faces; E the four
  // diagonals (27-point) or the four nodes at distance 2 (13-point)
  auto sums = [&](const W* b, W (&C)[R], W (&F)[R], W (&E)[R]) {
    const W* s = b + (ty * R) * WX + tx + G;   // row jr - G, the thread's column
    W m[R + 2 * G];
#pragma unroll
    for (int q = 0; q < R + 2 * G; q++) m[q] = s[q * WX];
    if constexpr (KIND == FX27) {
      W a[R + 2];
#pragma unroll
      for (int q = 0; q < R + 2; q++) a[q] = s[q * WX - 1] + s[q * WX + 1];
#pragma unroll
      for (int r = 0; r < R; r++) {
        C[r] = m[r + 1];
        F[r] = a[r + 1] + (m[r] + m[r + 2]);
        E[r] = a[r] + a[r + 2];
      }
    } else {
#pragma unroll
      for (int r = 0; r < R; r++) {
        const W* c = s + (r + G) * WX;
        C[r] = m[r + G];
        F[r] = (c[-1] + c[1]) + (m[r + G - 1] + m[r + G + 1]);
        if constexpr (KIND == FX13) E[r] = (c[-2] + c[2]) + (m[r] + m[r + 4]);
      }
    }
  };
  // the next plane: z = its index; its stage and the groups of the thread's rows
  int z = zl;
  auto arrive = [&](W (&C)[R], W (&F)[R], W (&E)[R]) -> const double* {
    mbar_wait(&bar[wq], wph, ok);
    const double* raw = ring + wq * UE;
    W* w = work + wb * UE;
#pragma unroll
    for (int q = 0; q < NLD; q++)
      if ((q + 1) * NT <= NEL || tid + q * NT < NEL) {
        const double v = raw[tid + q * NT];
        if constexpr (FX) w[tid + q * NT] = fx_from(v, sc.eb);
        else w[tid + q * NT] = v;
        if constexpr (Epi::TRACK)
          if ((inner >> q & 1u) && z >= G && z < G + d.nk()) epi.hmax = max(epi.hmax, (unsigned)__double2hiint(v) & 0x7fffffffu);
      }
    __syncthreads();
    if (tid == 0 && ok && z > zl) {   // after a failed wait no new copy is issued
      fence_proxy_async();
      issue(z - 1 + NS, wq == 0 ? NS - 1 : wq - 1);
    }
    const double* b = bring + wq * BE;
    if (++wq == NS) {
      wq = 0;
      wph ^= 1u;
    }
    wb ^= 1;
    z++;
    sums(w, C, F, E);
    return b;
  };
  const double cu = FX ? op.c * sc.unit() : op.c;
  // values of the thread's R nodes from their groups (27-point: centre, faces,
  // edges, corners; others: second differences at distance 1 and 2, in FP64 the sums)
  auto values = [&](const W (&c0)[R], const W (&g1)[R], const W (&g2)[R], const W (&g3)[R], const double (&f)[R],
                    double (&x)[R]) {
    if constexpr (!FX && KIND != FX27) {   // x_GS - x, with x_GS as the FP64 sweeps form it
#pragma unroll
      for (int r = 0; r < R; r++) x[r] = fma(KIND == FX7 ? g1[r] : fma(16.0, g1[r], -g2[r]), cu, f[r]) - c0[r];
    } else if constexpr (KIND == FX7) {
#pragma unroll
      for (int r = 0; r < R; r++) x[r] = fma(fx_double(g1[r]), cu, f[r]);
    } else if constexpr (KIND == FX27 && FX) {
#pragma unroll
      for (int r = 0; r < R; r++) {
        // |T| < 2^73: low words' products below 2^48, high words' below 2^46
        auto lo = [](long long v) { return (unsigned long long)(unsigned)v; };
        auto hi = [](long long v) { return (long long)(int)(v >> 32); };
        const unsigned long long lc = lo(c0[r]) * (unsigned)abs(op.w0);
        const long long L = (long long)(lo(g1[r]) * (unsigned)op.w1 + lo(g2[r]) * (unsigned)op.w2 +
                                        lo(g3[r]) * (unsigned)op.w3 + (op.w0 < 0 ? 0ull - lc : lc));
        const long long H = hi(c0[r]) * op.w0 + hi(g1[r]) * op.w1 + hi(g2[r]) * op.w2 + hi(g3[r]) * op.w3;
        x[r] = fma(fx_two_limbs(H, L), cu, f[r]);
      }
    } else if constexpr (KIND == FX27) {
#pragma unroll
      for (int r = 0; r < R; r++)
        x[r] = fma(fma((double)op.w0, c0[r], fma((double)op.w1, g1[r], fma((double)op.w2, g2[r], op.w3 * g3[r]))), cu, f[r]);
    } else {
      bool fits = true;   // one test for all nodes, so that their chains run interleaved
#pragma unroll
      for (int r = 0; r < R; r++) fits &= fx_below(g1[r], 26) && fx_below(g2[r], 29);   // 16 2^58 + 2^61 < 2^63
      if (fits) {
#pragma unroll
        for (int r = 0; r < R; r++) x[r] = fma(fx_double(g1[r] * 16 - g2[r]), cu, f[r]);
      } else {
#pragma unroll
        for (int r = 0; r < R; r++) x[r] = fma(fx_double(g1[r]), 16.0 * cu, fma(fx_double(g2[r]), -cu, f[r]));
      }
    }
  };
  auto finish = [&](const double* b, const W (&c0)[R], const W (&g1)[R], const W (&g2)[R], const W (&g3)[R]) {
    double f[R], x[R];
#pragma unroll
    for (int r = 0; r < R; r++) f[r] = b[(ty * R + r) * WX + tx + G];
    values(c0, g1, g2, g3, f, x);
    if constexpr (Epi::LAYERS) {
      const int k = z - 1 - G, i = i0 + tx;   // the plane that arrived last is z - 1
      const bool l = i == G || i == G + d.ni() - 1 || k == G || k == G + d.nk() - 1;
#pragma unroll
      for (int r = 0; r < R; r++) epi.layer[r] = l || jr + r == G || jr + r == G + d.nj() - 1;
    }
    epi(at, d.px, in, x, f);
    at += d.sz();
  };
  W c0[R], g1[R], g2[R], g3[R];
  if constexpr (G == 1) {
    W Cm[R], Fm[R], Em[R], Cc[R], Fc[R], Ec[R], Cn[R], Fn[R], En[R];
    arrive(Cm, Fm, Em);
    arrive(Cc, Fc, Ec);
    for (int k = k0; k < k1; k++) {
      const double* b = arrive(Cn, Fn, En);
#pragma unroll
      for (int r = 0; r < R; r++) {
        c0[r] = Cc[r];
        g1[r] = Fc[r] + (Cm[r] + Cn[r]);
        if constexpr (KIND == FX27) {
          g2[r] = Ec[r] + (Fm[r] + Fn[r]);
          g3[r] = Em[r] + En[r];
        } else if constexpr (FX) {
          g1[r] -= Cc[r] * 6;
        }
        Cm[r] = Cc[r];
        Fm[r] = Fc[r];
        Em[r] = Ec[r];
        Cc[r] = Cn[r];
        Fc[r] = Fn[r];
        Ec[r] = En[r];
      }
      finish(b, c0, g1, g2, g3);
    }
  } else {
    W C2m[R], C1m[R], Cc[R], Cp[R], Cn[R], Fc[R], Fp[R], Fn[R], Ec[R], Ep[R], En[R];
    arrive(C2m, Fn, En);
    arrive(C1m, Fn, En);
    arrive(Cc, Fc, Ec);
    arrive(Cp, Fp, Ep);
    for (int k = k0; k < k1; k++) {
      const double* b = arrive(Cn, Fn, En);
#pragma unroll
      for (int r = 0; r < R; r++) {
        const W c6 = FX ? Cc[r] * (W)6 : (W)0;
        c0[r] = Cc[r];
        g1[r] = Fc[r] + (C1m[r] + Cp[r]) - c6;
        g2[r] = Ec[r] + (C2m[r] + Cn[r]) - c6;
        C2m[r] = C1m[r];
        C1m[r] = Cc[r];
        Cc[r] = Cp[r];
        Cp[r] = Cn[r];
        Fc[r] = Fp[r];
        Fp[r] = Fn[r];
        Ec[r] = Ep[r];
        Ep[r] = En[r];
      }
      finish(b, c0, g1, g2, g3);
    }
  }
  return ok;
}

// The pass in the arithmetic that its scale (and the residual reached) allows.
template <int KIND, typename Epi>
__device__ __forceinline__ void fx_pass(const CUtensorMap& mU, const CUtensorMap& mB, const Dims& d, const FxOp& op,
                                        unsigned hmax, int zc, DevState* __restrict__ st, Epi& epi) {
  extern __shared__ __align__(128) unsigned char fx_smem[];
  const FxScale sc(hmax, st->exact);
  const bool ok = sc.fx ? fx_march<KIND, long long>(mU, mB, d, op, sc, zc, fx_smem, epi)
                        : fx_march<KIND, double>(mU, mB, d, op, sc, zc, fx_smem, epi);
  if (!ok) atomicExch(&st->fault, 1);
}

// Levels a pass runs on: rows at 16-byte multiples (TMA), and tiles enough to
// fill the device (below, one node per thread has the shorter chain).
constexpr long long FX_MIN_NODES = 700000;   // about 90^3
inline bool fx_level(const Dims& d) {
  return d.px % 2 == 0 && (long long)d.ni() * d.nj() * d.nk() >= FX_MIN_NODES;
}

// Tensor maps of a pass over a level: planes of u with their halo, planes of the right-hand side.
template <int KIND>
inline bool fx_maps(const Dims& d, const double* u, const double* base, CUtensorMap* mU, CUtensorMap* mB) {
  return encode_level_map(mU, 0, u, d, FxGeom<KIND>::WX, FxGeom<KIND>::WY) &&
         encode_level_map(mB, 0, base, d, FxGeom<KIND>::WX, FxGeom<KIND>::TY);
}

// Launch geometry: as many z-chunks as fill the resident blocks of whole waves
// (blocks_per_sm of the kernel), of `least` to 96 planes each (a chunk stages 2 G
// planes that it does not write).
inline dim3 fx_chunks(int gx, int gy, int nk, int blocks_per_sm, int least, int* zc) {
  const long long slots = (long long)device_sm_count() * blocks_per_sm, tiles = (long long)gx * gy;
  long long n = slots / tiles;                             // one wave
  if (n < (nk + 95) / 96) n = ((nk + 95) / 96 * tiles + slots - 1) / slots * slots / tiles;
  n = n < 1 ? 1 : n;
  const int most = nk < least ? 1 : nk / least;
  if (n > most) n = most;
  *zc = (int)((nk + n - 1) / n);
  return dim3(gx, gy, (nk + *zc - 1) / *zc);
}
template <int KIND>
inline dim3 fx_grid(const Dims& d, int blocks_per_sm, int* zc) {
  using Gm = FxGeom<KIND>;
  return fx_chunks((d.ni() + Gm::TX - 1) / Gm::TX, (d.nj() + Gm::TY - 1) / Gm::TY, d.nk(), blocks_per_sm, 8, zc);
}

}  // namespace ps
