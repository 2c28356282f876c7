// Device code shared by the per-solve kernels (cart_kernels.cu) and the
// batched kernels (batch.cu): the Gauss-Seidel value of a node, the
// coarsest-level CG of one thread block, and the residual-norm finisher.
#pragma once
#include "ps_common.cuh"

namespace ps {

// ------------------------------------------------------------------ stencil core
// phi_GS without the diagonal: sum of weighted neighbours plus fs.
template <int G, bool ISO, typename T, typename C>
__device__ __forceinline__ C gs_value(const T* __restrict__ phi, long long p, long long sy,
                                      long long sz, const Coef<C>& cf, C fs) {
  using S = St<T>;
  C ax = S::ld(phi + p + 1) + S::ld(phi + p - 1);
  C v;
  if constexpr (ISO && G == 1 && sizeof(C) == 8) {
    // FP64 7-point on equal spacings: the order of the diagonal colour pass
    // (k_sweep_diag), (E + W) + (S + D) + (N + U), so that residuals after a
    // sweep repeat its arithmetic exactly
    const C sd = S::ld(phi + p - sy) + S::ld(phi + p - sz);
    const C nu = S::ld(phi + p + sy) + S::ld(phi + p + sz);
    return fma((ax + sd) + nu, cf.c1[0], fs);
  }
  if constexpr (ISO && G == 2 && sizeof(C) == 8) {
    // FP64 13-point on equal spacings: the order of the diagonal colour pass
    // (k_sweep_diag13), (E + W) + (S + U) + (N + D) at distance 1, then the
    // same at distance 2
    const C su1 = S::ld(phi + p - sy) + S::ld(phi + p + sz);
    const C nd1 = S::ld(phi + p + sy) + S::ld(phi + p - sz);
    const C v1 = fma((ax + su1) + nd1, cf.c1[0], fs);
    const C ew2 = S::ld(phi + p + 2) + S::ld(phi + p - 2);
    const C su2 = S::ld(phi + p - 2 * sy) + S::ld(phi + p + 2 * sz);
    const C nd2 = S::ld(phi + p + 2 * sy) + S::ld(phi + p - 2 * sz);
    return fma((ew2 + su2) + nd2, cf.c2[0], v1);
  }
  C ay = S::ld(phi + p + sy) + S::ld(phi + p - sy);
  C az = S::ld(phi + p + sz) + S::ld(phi + p - sz);
  if (ISO) {
    v = fma((ax + ay) + az, cf.c1[0], fs);
  } else {
    v = fma(ax, cf.c1[0], fma(ay, cf.c1[1], fma(az, cf.c1[2], fs)));
  }
  if (G == 2) {
    C bx = S::ld(phi + p + 2) + S::ld(phi + p - 2);
    C by = S::ld(phi + p + 2 * sy) + S::ld(phi + p - 2 * sy);
    C bz = S::ld(phi + p + 2 * sz) + S::ld(phi + p - 2 * sz);
    if (ISO) {
      v = fma((bx + by) + bz, cf.c2[0], v);
    } else {
      v = fma(bx, cf.c2[0], fma(by, cf.c2[1], fma(bz, cf.c2[2], v)));
    }
  }
  return v;
}

// Set the enclosing graph's while-condition (chunk > 0 marks a graph body):
// continue while not done and below the iteration budget of this step, so
// every graph launch ends after a bounded number of iterations.
__device__ __forceinline__ void set_loop(const DevState* st, unsigned long long cond, int chunk) {
  if (chunk > 0) {
    const unsigned int more = (st->done == DONE_NO && st->iter < st->chunk_end) ? 1u : 0u;
    cudaGraphSetConditional((cudaGraphConditionalHandle)cond, more);
  }
}

// Sum a residual pass's per-block partials {sum delta^2, max |delta|} in block
// order, record the norm in the state and decide convergence (one block).
// mode: 0 = reference norm, 1 = initial residual, 2 = iteration check, 3 =
// iteration check that calls only a non-finite norm divergence (SOR on graded
// spherical grids: its non-normal iteration grows the residual a
// hundred-to-thousandfold before it converges), 4 = initial residual whose
// pass returned early on a zero guess (st->guess_nonzero == 0): the residual
// is then the reference vector, and its norm and max are those of mode 0.
// The block is a serial stretch of every iteration, so it is kept short: 256
// threads, one reduction through shared memory, the maxima and the scale on
// the integer pipe (10.8 us under ncu with 1024 threads, FP64 maxima, log2 and
// exp2, most of it in the SM's FP64 pipe).
constexpr int FINISH_THREADS = 256;
// Residual norms below this many times the share of the fixed-point units turn the
// passes to FP64: a V-cycle's factor (refinement step's: 100) above the share.
constexpr double FX_FLOOR = 64.0;
__device__ __forceinline__ void finish_norm_block(const double* __restrict__ partials, int nblocks,
                                                  double dscale, int mode, DevState* __restrict__ st,
                                                  unsigned long long cond, int chunk) {
  __shared__ double red[FINISH_THREADS];
  __shared__ double mx[32];
  const bool from_ref = mode == 4 && st->guess_nonzero == 0;
  if (mode == 4) mode = 1;
  double s = 0.0;
  AbsMax am;   // the maxima are magnitudes: compared by their bits
#pragma unroll 4
  for (int b = threadIdx.x; b < nblocks; b += FINISH_THREADS) {
    s += partials[2 * b];
    am.take(partials[2 * b + 1]);
  }
  const double wm = warp_absmax(am.value());
  if ((threadIdx.x & 31) == 0) mx[threadIdx.x >> 5] = wm;
  const double S = block_sum_warp0(s, threadIdx.x, FINISH_THREADS, red);
  if (threadIdx.x >= 32) return;
  double m = warp_absmax(threadIdx.x < FINISH_THREADS / 32 ? mx[threadIdx.x] : 0.0);
  if (threadIdx.x != 0) return;
  const double rr = from_ref ? st->rr : dscale * dscale * S;
  if (from_ref) m = st->amax;
  if (mode == 0) {
    st->rr = rr;
    double ref = sqrt(rr);
    st->ref = ref > 0.0 ? ref : 1.0;
    st->amax = m;
    st->scale_next = m > 0.0 ? pow2_scale(m) : 1.0;
    return;
  }
  if (st->done && mode >= 2) {
    set_loop(st, cond, chunk);
    return;
  }
  if (st->fault) {
    st->done = DONE_FAULT;
    set_loop(st, cond, chunk);
    return;
  }
  st->rr = rr;
  st->amax = m;
  // the residual pass that used these has run; what it read is the potential of
  // the next iteration
  const unsigned vb = max(st->bmax, st->fmax);
  st->vmax = mode == 1 ? max(st->umax, st->bmax) : st->vnext;
  st->lmax = max(mode == 1 ? st->umax : st->hu[0], vb);
  // what the units of this residual's passes may leave of it (fixed.cuh)
  const unsigned eb = max(max(max(st->umax, st->unext), st->vmax), vb) >> 20;
  st->lexact = st->exact;
  st->exact = eb < 0x7ffu && sqrt(rr) <= FX_FLOOR * st->fx_noise * __longlong_as_double((long long)eb << 52);
  if (mode == 1) st->lexact = st->exact;
  st->vnext = 0u;
  st->umax = st->unext;
  st->unext = 0u;
#pragma unroll
  for (int l = 0; l < 8; l++) st->hu[l] = st->hr[l] = 0u;
  const double rel = sqrt(rr) / st->ref;
  st->rel = rel;
  // IR: the scale of the next stored inner right-hand side (power of two)
  st->scale_cur = st->scale_next;
  st->scale_next = m > 0.0 ? pow2_scale(m) : 1.0;
  if (mode == 1) {
    st->iter = 0;
    st->rel0 = rel;
    st->done = rel <= st->tol ? DONE_CONVERGED : (st->max_iter <= 0 ? DONE_MAXITER : DONE_NO);
    if (!isfinite(rel)) st->done = DONE_DIVERGED;
    return;
  }
  st->iter += 1;
  if (!isfinite(rel) || (mode == 2 && rel > 1e3 * fmax(st->rel0, 1.0))) st->done = DONE_DIVERGED;
  else if (rel <= st->tol) st->done = DONE_CONVERGED;
  else if (st->iter >= st->max_iter) st->done = DONE_MAXITER;
  set_loop(st, cond, chunk);
}

// 1 / x for normal x with 1 / x normal: PTX's approximate reciprocal, then two steps
// of Newton's iteration y += y (1 - x y) for the root of 1 / y - x, each of which
// squares the relative error, and fused, so that the last rounding alone is left
// (4 FP64 instructions; a division takes about 10, 76 cycles each per warp).  Within
// one unit in the last place (ps_probe_recip).
__device__ __forceinline__ double recip(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(y, fma(-x, y, 1.0), y);
  return fma(y, fma(-x, y, 1.0), y);
}

// ------------------------------------------------------------------ grid barrier
// Barrier over the blocks of a cooperative launch (all resident at once):
// *bar counts arrivals, target = blocks times the barriers passed so far.  What
// any block wrote before it is visible after it (to loads that go to L2: the L1
// caches are not coherent, so data that other blocks write are read with
// __ldcg).  The count may pass 2^32 (very long launches): it is compared by its
// distance from the target.  The wait is bounded (2 s): past it ok turns false
// in the block, which sets *fault (the result is invalid even if the other
// blocks went on) and then stops, and so do the others in turn.
__device__ __forceinline__ void grid_barrier(unsigned* bar, unsigned target, int* fault, bool& ok) {
  __shared__ int alive;
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    unsigned v, spins = 0;
    unsigned long long t0 = 0;
    int good = 1;
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if ((int)(v - target) >= 0) break;
      if ((++spins & 255u) == 0) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t0 == 0) t0 = t;
        if (t - t0 > 2000000000ull) {
          good = 0;
          atomicExch(fault, 1);
          break;
        }
      }
    }
    alive = good;
  }
  __syncthreads();
  ok = ok && alive != 0;
}

// ------------------------------------------------------------------ thread-block cluster
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// Barrier over the cluster's threads; shared-memory writes before it, remote
// ones included, are visible after it.
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Store v at the address that p (in this CTA's shared memory) has in CTA `rank`.
__device__ __forceinline__ void store_remote(double* p, unsigned rank, double v) {
  unsigned a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// ------------------------------------------------------------------ coarsest-level CG
// One cluster solves -A e = d * fs (zero boundary, e0 = 0) by CG (Sec. 2.1.3:
// the coarsest level is solved with CG) until ||r|| <= tol ||r0|| or max_iter
// iterations.  GB300's FP64 pipe is narrow (about 1.7 instructions a cycle and
// SM, 63 cycles from one to the next that needs it), so one SM spends most of
// a solve issuing FP64: the level is cut into slabs along its longest axis, one
// slab per CTA, and the work runs on up to 16 SMs.  What is left is the chain
// of an iteration's sums and exchanges, so the recurrences are those of
// pipelined CG (P. Ghysels, W. Vanroose, Parallel Computing 40, 2014): with
// w = A r kept beside r, gamma = r.r and delta = w.r are summed together and
// n = A w does not wait for them,
//   beta = gamma / gamma', den = delta - beta^2 den', alpha = gamma / den,
//   z = n + beta z, s = w + beta s, p = r + beta p,
//   x += alpha p, r -= alpha s, w -= alpha z,
// the iterates of CG with one cluster barrier an iteration instead of three
// (den = p.A p).  The barrier hands round each warp's partial sums and the
// values of w next to the slab edges; w is kept twice, so that the next values
// are written while a slower CTA still reads the last ones.  A thread owns
// in-plane positions over the slab's planes, all vectors but w in registers.
// All CTAs add the same partials in the same order and therefore take the same
// alpha, beta and decision to stop.  Solve times: see launch_coarse_cg.
struct CgSlab {
  int s, a0, a1;      // slab axis (the longest, z first) and the in-plane axes
  int m0, m1, m2;     // unknowns along a0, a1, s
  int np;             // planes per CTA
  __host__ __device__ CgSlab(const Dims& d, int nc) {
    const int n[3] = {d.ni(), d.nj(), d.nk()};
    s = 2;
    if (n[1] > n[s]) s = 1;
    if (n[0] > n[s]) s = 0;
    a0 = s == 0 ? 1 : 0;
    a1 = s == 2 ? 1 : 2;
    m0 = n[a0];
    m1 = n[a1];
    m2 = n[s];
    np = (m2 + nc - 1) / nc;
  }
  __host__ __device__ int smem_doubles(int g) const {
    return 2 * (np + 2 * g) * (m0 + 2 * g) * (m1 + 2 * g);   // w, twice
  }
  // in-plane positions per thread and register slots (positions x planes) for at most maxt threads
  __host__ __device__ int positions(int maxt) const { return (m0 * m1 + maxt - 1) / maxt; }
};
constexpr int CG_MAXT = 128;      // threads per CTA: one warp per SM sub-partition and FP64 unit
constexpr int CG_MAXNC = 16;      // CTAs per cluster
constexpr int CG_MAX_SLOTS = 24;  // register slots per thread of the largest variant

template <int G, bool ISO, typename TF, typename TE, int PPT>
__device__ __forceinline__ void coarse_cg_cluster(const Dims& d, const Coef<double>& cf0,
                                                  const TF* __restrict__ fs, TE* __restrict__ e,
                                                  double tol, int max_iter, DevState* __restrict__ st,
                                                  double* sm) {
  __shared__ double part[2][2][CG_MAXNC * (CG_MAXT / 32)];   // [set][gamma, delta][rank, warp]
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nthr >> 5;
  const int rank = (int)cluster_rank(), NC = (int)cluster_size();
  const CgSlab L(d, NC);
  const int m0 = L.m0, m1 = L.m1, m2 = L.m2, np = L.np, area = m0 * m1;
  const int w0 = m0 + 2 * G, plane = w0 * (m1 + 2 * G);
  const int k0 = rank * np, nown = max(0, min(np, m2 - k0)), nsl = np + 2 * G;
  const int wsz = nsl * plane;   // w is kept at sm and sm + wsz: [nsl][m1 + 2G][m0 + 2G] each
  Coef<double> cf = cf0;
  // along the slab's axes (selects: an index would put the arrays in local memory)
  auto along = [](int a, auto v0, auto v1, auto v2) { return a == 0 ? v0 : (a == 1 ? v1 : v2); };
  auto permute = [&](const double (&v)[3], double (&o)[3]) {
    o[0] = along(L.a0, v[0], v[1], v[2]);
    o[1] = along(L.a1, v[0], v[1], v[2]);
    o[2] = along(L.s, v[0], v[1], v[2]);
  };
  permute(cf0.c1, cf.c1);
  permute(cf0.c2, cf.c2);
  const int t0 = (int)along(L.a0, 1LL, d.sy(), d.sz()), t1 = (int)along(L.a1, 1LL, d.sy(), d.sz()),
            t2 = (int)along(L.s, 1LL, d.sy(), d.sz());   // strides in fs and e (dense, small)
  const int Q = (area + nthr - 1) / nthr;   // in-plane positions per thread
  for (int u = tid; u < 2 * wsz; u += nthr) sm[u] = 0.0;
  __syncthreads();
  // b = d fs on every plane of the slab and its neighbours (in the second array: w takes its place after the first step)
  for (int q = 0; q < Q; q++) {
    const int f = tid + q * nthr;
    if (f >= area) break;
    const int j = f / m0, i = f - j * m0;
    for (int l = 0; l < nsl; l++) {
      const int k = k0 - G + l;
      if (k < 0 || k >= m2) continue;
      sm[wsz + l * plane + (j + G) * w0 + i + G] =
          cf.d * (double)St<TF>::ld(fs + (i + G) * t0 + (j + G) * t1 + (k + G) * t2);
    }
  }
  cluster_sync();   // b complete here, and every CTA runs before its memory is written
  // slot k = (q, l): position tid + q * nthr of the slab's plane l
  int gofs[PPT];   // offset in fs and e, -1 where the slot is empty
  int c[PPT];      // offset in w
  int up[PPT];     // ranks that have the slot's plane among their neighbours (G below, G above; a byte each, 255 = none)
  double x[PPT], r[PPT], p[PPT], s[PPT], z[PPT], w[PPT];
  // (A v) at a slot: d v - sum of d c times the neighbours
  const double cd = cf.d;
#pragma unroll
  for (int a = 0; a < 3; a++) {
    cf.c1[a] *= -cd;
    cf.c2[a] *= -cd;
  }
  auto apply = [&](const double* v, int at) -> double {
    return gs_value<G, ISO>(v, (long long)at, (long long)w0, (long long)plane, cf, cd * v[at]);
  };
#pragma unroll
  for (int k = 0; k < PPT; k++) {
    const int q = k / np, l = k - q * np, f = tid + q * nthr;
    const bool own = q < Q && f < area && l < nown;
    const int j = own ? f / m0 : 0, i = own ? f - j * m0 : 0;
    gofs[k] = own ? (i + G) * t0 + (j + G) * t1 + (k0 + l + G) * t2 : -1;
    c[k] = own ? (l + G) * plane + (j + G) * w0 + i + G : 0;
    unsigned to = 0xffffffffu;
    int last = rank;
#pragma unroll
    for (int o = -G, b = 0; o <= G; o++) {
      if (o == 0) continue;
      const int kz = k0 + l + o, tr = kz >= 0 ? kz / np : 0;
      if (own && kz >= 0 && kz < m2 && tr != rank && tr != last) {
        to = (to & ~(0xffu << (8 * b))) | ((unsigned)tr << (8 * b));
        last = tr;
      }
      b++;
    }
    up[k] = (int)to;
    x[k] = p[k] = s[k] = z[k] = 0.0;
    r[k] = own ? sm[wsz + c[k]] : 0.0;
    w[k] = own ? apply(sm + wsz, c[k]) : 0.0;
  }
  // w of the slots into buffer bsel, here and in the CTAs that read it
  auto publish = [&](int bsel) {
#pragma unroll
    for (int k = 0; k < PPT; k++) {
      if (gofs[k] < 0) continue;
      double* at = sm + (bsel ? wsz : 0) + c[k];
      *at = w[k];
      if (up[k] == -1) continue;
#pragma unroll
      for (int b = 0; b < 2 * G; b++) {
        const int to = (up[k] >> (8 * b)) & 0xff;
        // the plane's place in that CTA's slab: shifted by the distance of the slabs
        if (to != 0xff) store_remote(at + (rank - to) * np * plane, to, w[k]);
      }
    }
  };
  double igamma = 0.0, den = 0.0, stop2 = 0.0;
  int it = 0;
  publish(0);
  for (;; it++) {
    const int b = it & 1;
    double ga = 0.0, da = 0.0;
#pragma unroll
    for (int k = 0; k < PPT; k++) {   // empty slots hold zeros
      ga = fma(r[k], r[k], ga);
      da = fma(w[k], r[k], da);
    }
    // both sums in one tree: lanes 0-15 add gamma, 16-31 delta (a warp-wide
    // FP64 instruction holds its sub-partition for 76 cycles)
    const bool hi = lane >= 16;
    double v = (hi ? da : ga) + __shfl_xor_sync(0xffffffffu, hi ? ga : da, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((lane & 15) < NC) store_remote(&part[b][hi][rank * nw + warp], lane & 15, v);
    cluster_sync();
    v = 0.0;
    for (int i = lane & 15; i < NC * nw; i += 16) v += part[b][hi][i];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const double g = __shfl_sync(0xffffffffu, v, 0), dl = __shfl_sync(0xffffffffu, v, 16);
    double n[PPT];   // A w: independent of the sums
#pragma unroll
    for (int k = 0; k < PPT; k++) n[k] = gofs[k] >= 0 ? apply(sm + (b ? wsz : 0), c[k]) : 0.0;
    if (it == 0) {
      stop2 = tol * tol * g;   // on squared norms
      if (!(g > 0.0) || max_iter <= 0) break;
    } else if (g <= stop2 || it >= max_iter) {
      break;
    }
    const double beta = g * igamma;   // 0 in the first step
    den = fma(-beta * beta, den, dl);
    // alpha = g / den and 1 / g (for the next beta) from one reciprocal, within a few
    // units in the last place: x and r move by the same alpha, so their agreement,
    // and with it the accuracy reached, does not depend on these (divisions: 32^3
    // solve 694 -> 721 us)
    const double gd = g * den;
    double alpha;
    if (fabs(gd) > 1e-280 && fabs(gd) < 1e280) {
      const double inv = recip(gd);
      alpha = g * (g * inv);
      igamma = den * inv;
    } else {
      alpha = g / den;
      igamma = 1.0 / g;
    }
#pragma unroll
    for (int k = 0; k < PPT; k++) {
      s[k] = fma(beta, s[k], w[k]);
      z[k] = fma(beta, z[k], n[k]);
      w[k] = fma(-alpha, z[k], w[k]);
    }
    publish(b ^ 1);
#pragma unroll
    for (int k = 0; k < PPT; k++) {
      p[k] = fma(beta, p[k], r[k]);
      x[k] = fma(alpha, p[k], x[k]);
      r[k] = fma(-alpha, s[k], r[k]);
    }
  }
  // (no remote write follows the last barrier, so every CTA may leave)
#pragma unroll
  for (int k = 0; k < PPT; k++)
    if (gofs[k] >= 0) St<TE>::st(e + gofs[k], (typename St<TE>::C)x[k]);
  if (rank == 0 && tid == 0 && st != nullptr) {
    st->coarse_iter_last = it;
    st->coarse_iter_total += it;
  }
}

}  // namespace ps
