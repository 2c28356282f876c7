// Colour passes of FP32 and BF16 levels (omega = 1) over staged planes.
//
// One colour of the three of the 13-point operator, in place (the 7-point levels
// have fused sweeps).
// A pass that loads the neighbours of a node from global memory, two or four
// bytes at a time and three nodes apart, is bound by the L1 cache.  Here planes
// of phi (with a halo of G) and of fs come through a TMA ring; BF16 planes are
// widened once to FP32 in a ring of 2 G + 2 work planes, FP32 planes are read
// where they land.  A lane owns the G + 1 consecutive nodes of its rows that hold
// one member of each colour, so a warp reads its operands G + 1 words apart,
// without bank conflicts.  The value is formed in the order of gs_value: the
// stored bits are those of the per-node pass.  No node of another colour changes
// during the pass, so what a neighbour tile stages meanwhile is not ambiguous
// where it is used.  Measured (us a pass, per-node pass before): 256^3 FP32
// 42.6 -> 29.4 (200 MB, 30 at the copy rate), 128^3 FP32 9.8 -> 8.3; 512^3 BF16
// 181.7 -> 177.7 (800 MB, 118 at the copy rate; bound by issue and the L1 data
// path: 2.4 instructions a cycle, L1 at 84 % of its peak).  64^3 FP32 is slower (5.5 against 3.6: a few tiles, a
// chain from plane to plane), hence SS_MIN_NODES.  Two rows a lane: with one, 196
// on 512^3 (more halo to stage).
#include <algorithm>

#include "cart_kernels.cuh"
#include "fixed.cuh"
#include "staged_sweeps.cuh"

namespace ps {

namespace {

template <typename T, int G, int RR>
struct SsGeom {
  static constexpr bool WIDE = sizeof(T) == 2;              // widened into work planes
  static constexpr int NC = G + 1, NW = 8, NT = 32 * NW, R = RR;
  static constexpr int TX = 32 * NC, TY = NW * R;
  static constexpr int WX = align_up(TX + 2 * G, 16 / (int)sizeof(T)), WY = TY + 2 * G;
  // stages of phi: the planes on the way, and where they are read in place the
  // 2 G + 1 planes in use; stages of fs; work planes
  static constexpr int NS = WIDE ? 3 : 2 * G + 4, NF = 4, ND = WIDE ? 2 * G + 2 : 0;
  static constexpr int UB = align_up(WX * WY * (int)sizeof(T), 128), FB = align_up(WX * TY * (int)sizeof(T), 128);
  static constexpr int DB = align_up(WX * WY * 4, 128);
  static constexpr int SMEM = NS * UB + NF * FB + ND * DB + NS * 8;
};

template <typename T, int G, bool ISO, int R>
__global__ void __launch_bounds__(256, 227 * 1024 / (SsGeom<T, G, R>::SMEM + 1024) > 4 ? 4 : 227 * 1024 / (SsGeom<T, G, R>::SMEM + 1024))
    k_colour_staged(const __grid_constant__ CUtensorMap mP, const __grid_constant__ CUtensorMap mF, Dims d, Coef<float> cf,
                    int zc, int colour, T* phi, int* __restrict__ fault) {
  using Gm = SsGeom<T, G, R>;
  using S = St<T>;
  constexpr int NS = Gm::NS, NF = Gm::NF, ND = Gm::ND, NC = Gm::NC, WX = Gm::WX, WY = Gm::WY, NT = Gm::NT;
  constexpr int AHEAD = Gm::WIDE ? NS : NS - 2 * G - 1;   // planes on the way
  constexpr int UE = Gm::UB / (int)sizeof(T), FE = Gm::FB / (int)sizeof(T), DE = Gm::DB / 4;
  extern __shared__ __align__(128) unsigned char ss_smem[];
  T* const ring = reinterpret_cast<T*>(ss_smem);
  T* const fring = reinterpret_cast<T*>(ss_smem + NS * Gm::UB);
  float* const work = reinterpret_cast<float*>(ss_smem + NS * Gm::UB + NF * Gm::FB);
  unsigned long long* const bar = reinterpret_cast<unsigned long long*>(ss_smem + NS * Gm::UB + NF * Gm::FB + ND * Gm::DB);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i0 = blockIdx.x * Gm::TX + G, j0 = blockIdx.y * Gm::TY + G;
  const int k0 = blockIdx.z * zc + G, k1 = min(k0 + zc, G + d.nk());
  const int zl = k0 - G, zh = k1 - 1 + G;
  if (tid == 0) {
    for (int q = 0; q < NS; q++) mbar_init(&bar[q], 1);
    fence_mbar_init();
  }
  __syncthreads();
  auto issue = [&](int z) {   // thread 0: phi(z) and fs(z - G)
    if (z > zh) return;
    const int q = (z - zl) % NS, qf = (z - zl) % NF;
    const bool withf = z - G >= k0;
    mbar_expect_tx(&bar[q], (WX * WY + (withf ? WX * Gm::TY : 0)) * (int)sizeof(T));
    tma_load_3d(ring + q * UE, &mP, i0 - G, j0 - G, z, &bar[q]);
    if (withf) tma_load_3d(fring + qf * FE, &mF, i0 - G, j0, z - G, &bar[q]);
  };
  if (tid == 0)
    for (int q = 0; q < AHEAD; q++) issue(zl + q);
  bool ok = true;
  int wq = 0, wf = 0, cw = 0;   // stage, fs stage and (widened) work plane of plane z
  unsigned wph = 0;
  const int jr = j0 + warp * R;
  const int left = G + d.ni() - (i0 + NC * lane);   // the lane's interior nodes: the first `left`
  int m = ((colour - (i0 - G + 1) - (jr - G + 1) - (k0 - G + 1)) % NC + NC) % NC;   // member of row jr, plane k0
  T* out = phi + d.at(i0 + NC * lane, jr, k0);
  for (int z = zl; z <= zh; z++) {
    mbar_wait(&bar[wq], wph, ok);
    if constexpr (Gm::WIDE) {
      const uint4* raw = reinterpret_cast<const uint4*>(ring + wq * UE);
      float4* w = reinterpret_cast<float4*>(work + cw * DE);
      for (int q = tid; q < WX * WY / 8; q += NT) {
        const uint4 v = raw[q];
        w[2 * q] = make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                               __uint_as_float(v.y & 0xffff0000u));
        w[2 * q + 1] = make_float4(__uint_as_float(v.z << 16), __uint_as_float(v.z & 0xffff0000u),
                                   __uint_as_float(v.w << 16), __uint_as_float(v.w & 0xffff0000u));
      }
    }
    __syncthreads();   // the step before has been read; the work plane is complete
    // the stage of plane z (widened) or z - 2 G - 1, and the fs stage of the step before, are free
    if (tid == 0 && ok) {   // after a failed wait no new copy is issued
      fence_proxy_async();
      issue(z + AHEAD);
    }
    const int cq = Gm::WIDE ? cw : wq;
    constexpr int NP = Gm::WIDE ? ND : NS, PE = Gm::WIDE ? DE : UE;
    const float* base = Gm::WIDE ? work : reinterpret_cast<const float*>(ring);
    const T* fp = fring + wf * FE;
    if (++wq == NS) {
      wq = 0;
      wph ^= 1u;
    }
    if (++wf == NF) wf = 0;
    if constexpr (Gm::WIDE) {
      if (++cw == ND) cw = 0;
    }
    if (z - G < k0) continue;
    auto plane = [&](int back) { return base + (cq - back < 0 ? cq - back + NP : cq - back) * PE; };
    const int a0 = (warp * R + G) * WX + G + NC * lane;
    const float* P = plane(G) + a0;
    const float* A1 = plane(G - 1) + a0;
    const float* B1 = plane(G + 1) + a0;
    const float* A2 = plane(0) + a0;
    const float* B2 = plane(2 * G) + a0;
    float v[R];
    int mr = m;
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int a = r * WX + mr;
      const float f = S::ld(fp + (warp * R + r) * WX + G + NC * lane + mr);
      const float ax = P[a + 1] + P[a - 1], ay = P[a + WX] + P[a - WX], az = A1[a] + B1[a];
      if (ISO) v[r] = fma((ax + ay) + az, cf.c1[0], f);
      else v[r] = fma(ax, cf.c1[0], fma(ay, cf.c1[1], fma(az, cf.c1[2], f)));
      if constexpr (G == 2) {
        const float bx = P[a + 2] + P[a - 2], by = P[a + 2 * WX] + P[a - 2 * WX], bz = A2[a] + B2[a];
        if (ISO) v[r] = fma((bx + by) + bz, cf.c2[0], v[r]);
        else v[r] = fma(bx, cf.c2[0], fma(by, cf.c2[1], fma(bz, cf.c2[2], v[r])));
      }
      mr = mr == 0 ? NC - 1 : mr - 1;
    }
    mr = m;
#pragma unroll
    for (int r = 0; r < R; r++) {
      if (mr < left && jr + r < G + d.nj()) S::st(out + r * d.sy() + mr, v[r]);
      mr = mr == 0 ? NC - 1 : mr - 1;
    }
    out += d.sz();
    m = m == 0 ? NC - 1 : m - 1;
  }
  if (!ok) atomicExch(fault, 1);
}

template <typename T, int G, bool ISO, int R>
cudaError_t ss_t(const Dims& d, const double h[3], int dt, int colour, void* phi, const void* fs, int* fault, cudaStream_t s) {
  using Gm = SsGeom<T, G, R>;
  static PerDevice cached;
  int occ = 0, zc = 0;
  auto kern = k_colour_staged<T, G, ISO, R>;
  const cudaError_t e = resident_blocks(kern, 256, Gm::SMEM, cached, &occ);
  if (e != cudaSuccess) return e;
  CUtensorMap mP, mF;
  if (!encode_level_map(&mP, dt, phi, d, Gm::WX, Gm::WY) || !encode_level_map(&mF, dt, fs, d, Gm::WX, Gm::TY))
    return cudaErrorInvalidValue;
  const dim3 grid = fx_chunks((d.ni() + Gm::TX - 1) / Gm::TX, (d.nj() + Gm::TY - 1) / Gm::TY, d.nk(), occ, 4, &zc);
  kern<<<grid, Gm::NT, Gm::SMEM, s>>>(mP, mF, d, make_coef<float>(d, h, 2 * G), zc, colour, (T*)phi, fault);
  return cudaGetLastError();
}

}  // namespace

bool colour_staged_level(const Dims& d, int order, int dt) {
  const size_t es = dt == DT_F32 ? 4 : 2;
  return dt != DT_F64 && order == 4 && d.g == 2 && (d.px * es) % 16 == 0 &&
         (long long)d.ni() * d.nj() * d.nk() >= SS_MIN_NODES;
}

cudaError_t launch_colour_staged(const Dims& d, int order, const double h[3], int dt, int colour, void* phi, const void* fs,
                                 int* fault, cudaStream_t s) {
  if (!colour_staged_level(d, order, dt) || fault == nullptr) return cudaErrorInvalidValue;
  const bool iso = h[0] == h[1] && h[1] == h[2];
  if (dt == DT_F32)
    return iso ? ss_t<float, 2, true, 2>(d, h, dt, colour, phi, fs, fault, s)
               : ss_t<float, 2, false, 2>(d, h, dt, colour, phi, fs, fault, s);
  return iso ? ss_t<__nv_bfloat16, 2, true, 2>(d, h, dt, colour, phi, fs, fault, s)
             : ss_t<__nv_bfloat16, 2, false, 2>(d, h, dt, colour, phi, fs, fault, s);
}

}  // namespace ps
