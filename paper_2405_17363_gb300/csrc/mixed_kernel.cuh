// FP32-inner / FP64-outer iterative refinement, warp-packed layout (see
// warp_kernel.cuh for the lane/segment arrangement).  Per cell and sweep: the
// FP64 true residual r = b - A x and its norm decide convergence; otherwise an
// FP32 right-Jacobi BiCGSTAB solves A32 d = r / ||r|| to a relative inner
// tolerance (or an inner iteration cap) and x += ||r|| d in FP64.  The FP64
// pipe only sees the residual products, norms and updates; the inner
// iterations run on the FP32 pipe.
//
// Shared memory per cell: A in FP32 [segA] and, when a.a64_smem is set, in
// FP64 [segA] (otherwise the FP64 residual product reads A through L1 from
// the cell's row in global memory, which the staging has just brought into
// L2: it runs two or three times per cell, against tens of FP32 products, and
// the smaller footprint lets more warps run), and the FP64 product's input and
// output vectors [segV each], whose space the inner iteration's three FP32
// vectors take in turn.
#pragma once
#include "warp_common.cuh"

namespace camp {

template <int E, int LC>
__device__ __forceinline__ void mixed_body(const MixedArgs &a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SchedWord *sch_s = reinterpret_cast<SchedWord *>(smem_raw);
  const int nsch = a.L * a.Lc;
  for (int i = threadIdx.x; i < nsch; i += blockDim.x) sch_s[i] = a.sched[i];

  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int Lc = LC ? LC : a.Lc;  // lanes per cell (compile-time when LC > 0)
  const int seg = LC ? lane / LC : lane >> a.log2Lc;
  const int sl = lane & (Lc - 1);
  const int n = a.n, nnz = a.nnz;
  const size_t cellBytes = mixed_cell_bytes(a.segA, a.segV, a.a64_smem, Lc);
  unsigned char *wb = smem_raw + sched_smem_bytes(nsch) +
                      ((size_t)warp * a.k + seg) * cellBytes;
  double *As = reinterpret_cast<double *>(wb);
  double *g64 = As + (a.a64_smem ? a.segA : 0);
  double *o64 = g64 + a.segV;
  float *As32 = reinterpret_cast<float *>(o64 + a.segV);
  float *g32 = reinterpret_cast<float *>(g64);  // the inner iteration's vectors
  float *o1 = g32 + a.segV;
  float *o2 = o1 + a.segV;
  // in-launch difficulty ordering first: it borrows the start of the warp
  // regions (and ends with a block barrier)
  if (a.ord_ws)
    order_prologue<false>(a, reinterpret_cast<int *>(smem_raw + sched_smem_bytes(nsch)));
  __syncthreads();
  const SchedWord *sch = sch_s;
  const unsigned g64a = smem_addr(g64), o64a = smem_addr(o64), g32a = smem_addr(g32),
                 o1a = smem_addr(o1), o2a = smem_addr(o2);
  const int warps_total = gridDim.x * (blockDim.x >> 5);
  constexpr int K = LC ? 32 / LC : 0;  // cells per warp (0: a.k)

  auto refine_group = [&](int g) {
    const int pos = g * (K ? K : a.k) + seg;
    const bool has = pos < a.cells;
    // the order may have been written earlier in this launch (cell + 1 from
    // the in-launch ordering): read it through L2, clamped in range
    const int c = (has && a.order)
                      ? (int)min((unsigned)(__ldcg(a.order + pos) - (a.ord_ws ? 1 : 0)),
                                 (unsigned)a.cells - 1u)
                      : pos;
    const double *Ac = a.A + (size_t)(has ? c : 0) * nnz;
    if (a.a64_smem) {  // stage A in slot order, FP64 and its FP32 rounding
      stage_scatter(Ac, a.dst, nnz, sl, Lc, has, [&](int t, double v) { As[t] = v; });
      zero_padding(As, a.pads, a.npads, a.L, sl, Lc);
    }
    stage_scatter(Ac, a.dst32, nnz, sl, Lc, has, [&](int t, double v) { As32[t] = d2f_rn(v); });
    zero_padding(As32, a.pads32, a.npads, a.L, sl, Lc);
    __syncwarp();
    double xv[E];
    float dinv[E];
    double bb;
    {
      double acc[1] = {0.0};
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int i = sl + e * Lc;
        const bool v = has && i < n;
        const double bi = v ? __ldg(a.b + (size_t)c * n + i) : 0.0;
        const float d = v ? As32[__ldg(a.dslot32 + i)] : 0.0f;
        dinv[e] = v ? (d != 0.0f ? 1.0f / d : 1.0f) : 0.0f;
        xv[e] = 0.0;
        acc[0] = fma(bi, bi, acc[0]);
      }
      bb = seg_sum_x<LC>(acc[0], Lc);
    }
    const double thr = (a.tol * a.tol) * bb;  // (tol ||b||)^2
    int st = -1, sweeps = 0, inner = 0;
    double resid = 0.0;
    bool done = !has;
    if (has && !is_finite_bits(bb)) {
      st = CAMP_CELL_NONFINITE;
      resid = __longlong_as_double(0x7ff8000000000000ll);
      done = true;
    } else if (has && is_zero_bits(bb)) {
      st = CAMP_CELL_CONVERGED;
      done = true;
    }
    for (int pass = 0;; ++pass) {
      // ---- FP64 true residual r = b - A x (x = 0 on the first pass)
      double r[E];
      if (pass > 0) {
        __syncwarp();  // the inner vectors' last reads
#pragma unroll
        for (int e = 0; e < E; ++e) g64[sl + e * Lc] = xv[e];
        __syncwarp();
        if (a.a64_smem) flat_spmv(sch, a.L, Lc, sl, As, g64a, o64a);
        else flat_spmv_gather(sch, a.src, a.L, Lc, sl, Ac, g64a, o64a);
        __syncwarp();
      }
      double rr[1] = {0.0};
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int i = sl + e * Lc;
        const double bi = (has && i < n) ? __ldg(a.b + (size_t)c * n + i) : 0.0;
        r[e] = pass > 0 && i < n ? bi - o64[i] : bi;
      }
      if (pass > 0) {
#pragma unroll
        for (int e = 0; e < E; ++e) rr[0] = fma(r[e], r[e], rr[0]);
        rr[0] = seg_sum_x<LC>(rr[0], Lc);
      } else {
        rr[0] = bb;  // r = b: the same chain and exact sum
      }
      if (!done) {
        // ||r|| <= tol ||b|| on the bit patterns; the relative residual itself
        // (a square root and a division) is formed once, at the end
        if (!is_finite_bits(rr[0])) {
          st = CAMP_CELL_NONFINITE;
          done = true;
        } else if (le_nonneg(rr[0], thr)) {
          st = CAMP_CELL_CONVERGED;
          done = true;
        } else if (sweeps >= a.max_sweeps) {
          st = CAMP_CELL_MAXIT;
          done = true;
        }
        if (done) resid = sqrt(rr[0] * recip64(bb));
      }
      if (!__any_sync(kFull, !done)) break;
      // ---- FP32 inner solve of A d = r / ||r||.  The scale only sets the
      // size of the FP32 right-hand side, so it is formed in FP32 (FP64 when
      // ||r||^2 is outside the FP32 range).
      float rn32, rinv32;
      bool wide = false;
      {
        const int ex = (int)(((unsigned long long)__double_as_longlong(rr[0]) >> 52) & 0x7ffull) - 1023;
        wide = ex < -120 || ex > 120;
        const float rr32 = d2f_rn(rr[0]);
        rinv32 = rsqrtf(rr32);
        rn32 = rr32 * rinv32;
      }
      const double rn64 = wide ? sqrt(rr[0]) : 0.0;
      const double sc64 = wide ? 1.0 / rn64 : 0.0;
      float rf[E], rh[E], p[E], d[E];  // rf also holds s = r - alpha v
      float cc[1] = {0.0f};
      __syncwarp();  // the FP64 product's last reads
      // pad rows of the product vectors are never written by the products
      for (int i = n + sl; i < E * Lc; i += Lc) {
        o1[i] = 0.0f;
        o2[i] = 0.0f;
      }
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const float ce = done ? 0.0f : (wide ? d2f_rn(r[e] * sc64) : d2f_rn(r[e]) * rinv32);
        rf[e] = ce;
        rh[e] = ce;
        p[e] = 0.0f;
        d[e] = 0.0f;
        cc[0] = fmaf(ce, ce, cc[0]);
      }
      seg_sumf<1>(cc, Lc);
      const float thr = a.tol_in * a.tol_in * cc[0];
      float rho = cc[0], rho_prev = 1.0f, alpha = 1.0f, omega = 1.0f;
      bool act = !done && cc[0] > 0.0f && isfinite(cc[0]);
      int it = 0;
      bool head = true;  // first iteration: p = r
      while (__any_sync(kFull, act)) {
        if (act) {
          if (it >= a.maxit_in || !isfinite(rho) || fabsf(rho) < 1e-37f) act = false;
        }
        // p = r + beta (p - omega v), v of the iteration before
        if (head) {
          head = false;
#pragma unroll
          for (int e = 0; e < E; ++e) p[e] = rf[e];
        } else {
          const float beta = (rho / rho_prev) * (alpha / omega);
#pragma unroll
          for (int e = 0; e < E; ++e)
            p[e] = fmaf(beta, fmaf(-omega, o1[sl + e * Lc], p[e]), rf[e]);
        }
#pragma unroll
        for (int e = 0; e < E; ++e) g32[sl + e * Lc] = dinv[e] * p[e];
        __syncwarp();
        flat_spmvf(sch, a.L, Lc, sl, As32, g32a, o1a);
        __syncwarp();
        if (act) ++it;
        float sg[1] = {0.0f};
#pragma unroll
        for (int e = 0; e < E; ++e) sg[0] = fmaf(rh[e], o1[sl + e * Lc], sg[0]);
        seg_sumf<1>(sg, Lc);
        if (act && (!isfinite(sg[0]) || fabsf(sg[0]) < 1e-37f)) act = false;
        alpha = rho / sg[0];
        float q0[1] = {0.0f};
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int i = sl + e * Lc;
          if (act) d[e] = fmaf(alpha, g32[i], d[e]);
          rf[e] = fmaf(-alpha, o1[i], rf[e]);  // s
          q0[0] = fmaf(rf[e], rf[e], q0[0]);
        }
        seg_sumf<1>(q0, Lc);
        // converged on the half step: tested before the second product
        if (act && q0[0] <= thr) act = false;
        if (!__any_sync(kFull, act)) break;
#pragma unroll
        for (int e = 0; e < E; ++e) g32[sl + e * Lc] = dinv[e] * rf[e];
        __syncwarp();
        flat_spmvf(sch, a.L, Lc, sl, As32, g32a, o2a);
        __syncwarp();
        float qt[2] = {0.0f, 0.0f};
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const float t = o2[sl + e * Lc];
          qt[0] = fmaf(t, rf[e], qt[0]);
          qt[1] = fmaf(t, t, qt[1]);
        }
        seg_sumf<2>(qt, Lc);
        bool full = false;
        if (act) {
          if (!isfinite(qt[0]) || !isfinite(qt[1]) || qt[1] == 0.0f)
            act = false;
          else
            full = true;
        }
        omega = qt[0] / qt[1];
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int i = sl + e * Lc;
          if (full) d[e] = fmaf(omega, g32[i], d[e]);
          rf[e] = fmaf(-omega, o2[i], rf[e]);
        }
        float q2[2] = {0.0f, 0.0f};
#pragma unroll
        for (int e = 0; e < E; ++e) {
          q2[0] = fmaf(rh[e], rf[e], q2[0]);
          q2[1] = fmaf(rf[e], rf[e], q2[1]);
        }
        seg_sumf<2>(q2, Lc);
        if (full) {
          if (q2[1] <= thr || omega == 0.0f) act = false;
        }
        rho_prev = rho;
        rho = q2[0];
      }
      if (!done) {
        inner += it;
        ++sweeps;
#pragma unroll
        for (int e = 0; e < E; ++e)
          xv[e] += wide ? rn64 * f2d_exact(d[e]) : f2d_exact(rn32 * d[e]);
      }
    }
    if (has) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int i = sl + e * Lc;
        if (i < n) a.x[(size_t)c * n + i] = xv[e];
      }
      if (sl == 0) {
        a.iters[c] = inner;
        if (a.sweeps) a.sweeps[c] = sweeps;
        a.resid[c] = resid;
        if (a.status) a.status[c] = st;
      }
    }
    __syncwarp();
  };

  if (!a.queue) {
    for (int g = blockIdx.x * (blockDim.x >> 5) + warp; g < a.ngroups; g += warps_total)
      refine_group(g);
    return;
  }
  // dynamic assignment (an ordered launch first gives every warp one group
  // of a stratified wave)
  bool first = true;
  unsigned g = 0;
  while (take_group(a, warp, lane, first, g)) {
    const bool mine = await_order_entries(a, g, K ? K : a.k, lane);
    refine_group((int)g);
    if (mine) a.ord_out[g * (K ? K : a.k) + lane] = 0;
  }
  finish_queue(a, true, warps_total, lane);
}

// FP32 and FP64 issue and shared memory are each about half busy, so resident
// warps hide the rest: 20 per SM (96 registers), and 24 (80 registers) with up
// to 3 rows per lane on 32 lanes, where 4 bytes spill and A in FP64 is not read
// through L1; 16 (128 registers) beyond 5 rows per lane.  16 / 20 / 24 warps:
// 150 species x 100,000 cells 1,919 / 1,858 / 2,273 us, 80 x 10,000 117 / 112 /
// 105, 40 x 20,000 (16 lanes) 114 / 113 / 123.
template <int E, int LC>
constexpr bool kMixedMany = E <= 3 && LC == 32;
template <int E, int LC>
__global__ void __launch_bounds__(kMixedMany<E, LC> || E > 5 ? 256 : 320, kMixedMany<E, LC> ? 3 : 2)
    mixed_refine_kernel(const __grid_constant__ MixedArgs a) {
  mixed_body<E, LC>(a);
}

}  // namespace camp
