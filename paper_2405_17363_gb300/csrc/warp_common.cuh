// Device helpers shared by the warp-packed kernels (FP64 solve and FP32-inner
// refinement): bit-pattern tests that avoid the FP64 pipe, segment-local
// shuffle sums and the schedule-driven SpMV.
#pragma once
#include "camp_internal.h"

namespace camp {

constexpr unsigned kFull = 0xffffffffu;

// Difficulty class of a cell from the high word of its estimate (a
// non-negative double, so its high words order as integers): the half-octave
// index (exponent and first fraction bit), largest first, 32 octaves down from
// TOP.  max_i |A_ii - 1| takes TOP 2^19 (estimates from 3/2 2^19 share class 0,
// those below 2^-12, which converge in an iteration or two, the last one): the
// stiff cells of a long step have estimates of 10^2 to 10^5 and 15 to 300
// iterations, and with 12 and above in one class they came in no order at all
// (80 species, pairs: 4,000 such cells 2,454 us, 2,235 in order; 6,000 cells
// 3,549 and 3,012).
// |gamma| takes TOP 2^3.
constexpr int kTopDeparture = 19, kTopGamma = 3;
template <int TOP>
__device__ __forceinline__ int difficulty_class(unsigned hi) {
  const int idx = (int)(hi >> 19);  // 2 * biased exponent + top fraction bit
  const int top = ((1023 + TOP) << 1) | 1;
  const int c = top - idx;
  return c < 0 ? 0 : (c >= kOrdClasses ? kOrdClasses - 1 : c);
}
__device__ __forceinline__ unsigned diag_departure_hi(double aii) {
  return (unsigned)((unsigned long long)__double_as_longlong(fabs(aii - 1.0)) >> 32);
}
// The same key from gamma itself (its magnitude, on the integer pipe).
__device__ __forceinline__ unsigned magnitude_hi(double v) {
  return (unsigned)(((unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull) >> 32);
}

__device__ __forceinline__ bool is_finite_bits(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  return ((u >> 52) & 0x7ffull) != 0x7ffull;
}
// |v| < 1e-300, on the bit pattern (no FP64 instruction)
__device__ __forceinline__ bool abs_tiny(double v) {
  const unsigned long long u =
      (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
  return u < 0x01a56e1fc2f8f359ull;  // bit pattern of 1e-300
}
// a <= b for a, b >= +0 (or NaN a: false), on the bit pattern
__device__ __forceinline__ bool le_nonneg(double a, double b) {
  return __double_as_longlong(a) <= __double_as_longlong(b);
}

// Sum NV values over the Lc lanes of each segment (xor butterfly; every lane
// of the segment ends with the same bits).
template <int NV>
__device__ __forceinline__ void seg_sum(double (&v)[NV], int Lc) {
  for (int off = Lc >> 1; off > 0; off >>= 1) {
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] += __shfl_xor_sync(kFull, v[q], off);
  }
}

// Two sums over the segment with log2(Lc) FP64 additions instead of
// 2 log2(Lc): at the first level each lane pair exchanges the value the other
// keeps (the lower lane keeps a, the upper keeps b), then one value is summed;
// a final exchange gives every lane both totals.
__device__ __forceinline__ void seg_sum2(double &a, double &b, int Lc) {
  if (Lc == 1) return;
  const int half = Lc >> 1;
  const bool up = (threadIdx.x & half) != 0;
  double keep = up ? b : a;
  const double send = up ? a : b;
  keep += __shfl_xor_sync(kFull, send, half);
  for (int off = half >> 1; off > 0; off >>= 1) keep += __shfl_xor_sync(kFull, keep, off);
  const double other = __shfl_xor_sync(kFull, keep, half);
  a = up ? other : keep;
  b = up ? keep : other;
}

__device__ __forceinline__ double fma_t(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fma_t(float a, float b, float c) { return fmaf(a, b, c); }

// Shared-memory accesses by 32-bit address (byte offset in the CTA's window).
__device__ __forceinline__ unsigned smem_addr(const void *p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void lds(double &v, unsigned a) {
  asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a));
}
__device__ __forceinline__ void lds(float &v, unsigned a) {
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
}
__device__ __forceinline__ void sts(unsigned a, double v) {
  asm volatile("st.shared.f64 [%0], %1;" :: "r"(a), "d"(v) : "memory");
}
// *a = v when flag != 0, as one predicated store (no branch)
__device__ __forceinline__ void sts_if(unsigned flag, unsigned a, double v) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q st.shared.f64 [%1], %2;\n\t}"
               :: "r"(flag), "r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void sts_if(unsigned flag, unsigned a, float v) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q st.shared.f32 [%1], %2;\n\t}"
               :: "r"(flag), "r"(a), "f"(v) : "memory");
}

// The gathered vector's address of a slot (a word holds 4 * column above 4 *
// row and the lane's end flag).
template <class T>
__device__ __forceinline__ unsigned slot_col_addr(unsigned w, unsigned gs) {
  return gs + (w >> (sizeof(T) == 8 ? 15 : 16));
}
// A slot in which some lane ends a row: those lanes store their sum and
// start from zero (a predicated store and a select).
template <class T>
__device__ __forceinline__ void slot_end(unsigned w, T &acc, unsigned os) {
  sts_if(w & kSlotEnd, os + (w & kSlotRowMask) * (sizeof(T) == 8 ? 2u : 1u), acc);
  acc = (w & kSlotEnd) ? T(0) : acc;
}

// os[row] = sum over this lane's slots of A_slot * gs[col] (gs, os: shared
// addresses; sch: the schedule's words; ends: the launch's row-end mask, a
// kernel parameter, so the tests on it are uniform branches).  lo(b, ..) and
// hi(b, ..) give the A values of the lane's slots 4b, 4b+1 and 4b+2, 4b+3;
// last(j, av), those of the slots j .. L-1 past the last whole block.
// FP64: the chain of dependent multiply-adds (64 cycles each for one warp,
// which is also the sub-partition's issue interval) bounds both a lone warp
// and a full SM, so everything else runs under it: the gathers and A values
// of a half block are issued two multiply-adds ahead, the words a block
// ahead, and only the slots of the end mask (8 to 11 of 36 at 80 rows on 16
// lanes) put a select on the chain.  Measured at 80 rows, 564 entries, 16
// lanes, in isolation: 95 cycles per slot for a lone warp against 100 with a
// conditional store and select in every slot, in 520 instructions against 915;
// 65 per slot and warp with three or four warps per sub-partition either way.
// (Two word sets and an unrolled pair of blocks: 81 alone, but the kernels
// around it spilled: 183 us against 180 at 80 species x 10,000 cells.)
// A pattern without an aligned layout (align.h finds none: dense ones, above
// some 250 rows; and camp_solve_noalloc) runs it on the schedule as built, with
// the mask set wherever rows end: in nearly every slot of a sparse pattern,
// where spmv_flat below would be a little faster, in a few of a dense one, where
// it would be slower (us a solve, this and spmv_flat: 400 species, 2,880
// entries, 5,000 cells 666 and 646; 512, 3,997, 4,000 cells 900 and 870; 107,
// 7,653, 2,000 cells 2,074 and 2,301; 40, 1,235, 5,000 cells 397 and 424).
template <class T, class Lo, class Hi, class Last>
__device__ __forceinline__ void spmv_slots(const SchedWord *__restrict__ sch,
                                           const unsigned *__restrict__ ends, int L, int Lc, int sl,
                                           Lo lo, Hi hi, Last last, unsigned gs, unsigned os) {
  static_assert(kSlotBlock == 4, "word blocks are 16 bytes");
  const uint4 *s4 = reinterpret_cast<const uint4 *>(sch) + sl;
  T acc = T(0);
  const int nb = L >> 2;
  unsigned mk = 0;
  if (nb > 0) {
    uint4 w = *s4;
    T x0, x1, x2, x3, a0, a1, a2, a3;
    lds(x0, slot_col_addr<T>(w.x, gs));
    lds(x1, slot_col_addr<T>(w.y, gs));
    lo(0, a0, a1);
#pragma unroll 1
    for (int b = 0;;) {
      if ((b & 7) == 0) mk = b < 8 * kEndWords ? ends[b >> 3] : ~0u;
      lds(x2, slot_col_addr<T>(w.z, gs));
      lds(x3, slot_col_addr<T>(w.w, gs));
      hi(b, a2, a3);
      uint4 wn = w;
      const bool more = ++b < nb;
      if (more) wn = s4[b * Lc];
      acc = fma_t(a0, x0, acc);
      if (mk & 1u) slot_end(w.x, acc, os);
      acc = fma_t(a1, x1, acc);
      if (mk & 2u) slot_end(w.y, acc, os);
      if (more) {
        lds(x0, slot_col_addr<T>(wn.x, gs));
        lds(x1, slot_col_addr<T>(wn.y, gs));
        lo(b, a0, a1);
      }
      acc = fma_t(a2, x2, acc);
      if (mk & 4u) slot_end(w.z, acc, os);
      acc = fma_t(a3, x3, acc);
      if (mk & 8u) slot_end(w.w, acc, os);
      mk >>= 4;
      if (!more) break;
      w = wn;
    }
  }
  if (L & 3) {
    if ((nb & 7) == 0) mk = nb < 8 * kEndWords ? ends[nb >> 3] : ~0u;
    SchedWord w[3];
    T av[3], xv[3];
#pragma unroll
    for (int u = 0; u < 3; ++u) w[u] = (L & 3) > u ? sch[(4 * nb + u) * Lc + sl] : 0u;
#pragma unroll
    for (int u = 0; u < 3; ++u) lds(xv[u], slot_col_addr<T>(w[u], gs));
    last(4 * nb, av);
#pragma unroll
    for (int u = 0; u < 3; ++u)
      if ((L & 3) > u) {
        acc = fma_t(av[u], xv[u], acc);
        if (mk & (1u << u)) slot_end(w[u], acc, os);
      }
  }
}

// o[row] = sum over this lane's slots of A_slot * g[col], A in slot order in
// shared memory (As: the cell's block, pair_pos places).
__device__ __forceinline__ void seg_spmv(const SchedWord *__restrict__ sch,
                                         const unsigned *__restrict__ ends, int L, int Lc, int sl,
                                         const double *__restrict__ As, unsigned gs, unsigned os) {
  const double2 *A2 = reinterpret_cast<const double2 *>(As) + sl;
  auto pair = [&](int p, double &a, double &b) {
    const double2 v = A2[p * Lc];
    a = v.x;
    b = v.y;
  };
  spmv_slots<double>(
      sch, ends, L, Lc, sl, [&](int b, double &u, double &v) { pair(2 * b, u, v); },
      [&](int b, double &u, double &v) { pair(2 * b + 1, u, v); },
      [&](int j, double *av) {
        if (L - j > 1) pair(j >> 1, av[0], av[1]);
        else av[0] = As[j * Lc + sl];
        if (L - j > 2) av[2] = As[(j + 2) * Lc + sl];
      },
      gs, os);
}

// Same with A read from global memory through the slots' source entries.
__device__ __forceinline__ void seg_spmv_gather(const SchedWord *__restrict__ sch,
                                                const unsigned *__restrict__ ends,
                                                const int *__restrict__ src, int L, int Lc, int sl,
                                                const double *__restrict__ Ag, unsigned gs,
                                                unsigned os) {
  const int2 *s2 = reinterpret_cast<const int2 *>(src) + 2 * sl;
  auto value = [&](int k) { return k >= 0 ? __ldg(Ag + k) : 0.0; };
  auto pair = [&](int p, double &a, double &b) {
    const int2 k = __ldg(s2 + (p >> 1) * 2 * Lc + (p & 1));
    a = value(k.x);
    b = value(k.y);
  };
  spmv_slots<double>(
      sch, ends, L, Lc, sl, [&](int b, double &u, double &v) { pair(2 * b, u, v); },
      [&](int b, double &u, double &v) { pair(2 * b + 1, u, v); },
      [&](int j, double *av) {
#pragma unroll
        for (int u = 0; u < 3; ++u)
          if (L - j > u) av[u] = value(__ldg(src + (j + u) * Lc + sl));
      },
      gs, os);
}

// Coalesced, vectorised read of one cell's A row (CSR order), handed to
// put(place, value) with the place from the dst map.  The row is read in
// 16-byte pairs from its first 16-byte boundary (lane sl reads pairs sl,
// sl + Lc, ...); an entry before that boundary and an odd entry at the end
// are read alone by lane 0.  The map is kept twice, the copy at odd shifted by
// one int, so that the pairs' places are 8-byte loads at either boundary.  The
// loads of P pairs are issued before any store, so a lane waits for memory
// once per batch rather than once per entry.
constexpr int kStagePairs = 8;
template <int P = kStagePairs, class Put>
__device__ __forceinline__ void stage_scatter(const double *__restrict__ Ac,
                                              const int *__restrict__ dst, int nnz,
                                              int sl, int Lc, bool live, Put put) {
  const int h = (int)((reinterpret_cast<size_t>(Ac) >> 3) & 1);  // entries before the boundary
  const int np = (nnz - h) >> 1;                                  // whole pairs
  const double2 *A2 = reinterpret_cast<const double2 *>(Ac + h);
  const int2 *d2 = reinterpret_cast<const int2 *>(dst + (h ? dst_odd(nnz) + 1 : 0));
  for (int p0 = sl; p0 < np; p0 += P * Lc) {
    double2 v[P];
    int2 d[P];
#pragma unroll
    for (int u = 0; u < P; ++u) {
      const int p = p0 + u * Lc;
      const bool in = p < np;
      d[u] = in ? __ldg(d2 + p) : make_int2(-1, -1);
      v[u] = (live && in) ? __ldg(A2 + p) : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int u = 0; u < P; ++u)
      if (d[u].x >= 0) {
        put(d[u].x, v[u].x);
        put(d[u].y, v[u].y);
      }
  }
  if (sl == 0) {
    if (h) put(__ldg(dst), live ? __ldg(Ac) : 0.0);
    if ((nnz - h) & 1) put(__ldg(dst + nnz - 1), live ? __ldg(Ac + nnz - 1) : 0.0);
  }
}

// Zero a slot-ordered A's padding slots (never scatter targets): the places
// pads[0 .. npads), or with npads < 0 every lane's slots from pads[lane] on.
template <class T>
__device__ __forceinline__ void zero_padding(T *__restrict__ Abase, const int *__restrict__ pads,
                                             int npads, int L, int sl, int Lc) {
  for (int i = sl; i < npads; i += Lc) Abase[__ldg(pads + i)] = T(0);
  if (npads < 0)
    for (int j = __ldg(pads + sl); j < L; ++j) Abase[pair_pos(j, sl, L, Lc)] = T(0);
}

// float variant of the segment sum
template <int NV>
__device__ __forceinline__ void seg_sumf(float (&v)[NV], int Lc) {
  for (int off = Lc >> 1; off > 0; off >>= 1) {
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] += __shfl_xor_sync(kFull, v[q], off);
  }
}

// The same product with a row end in every slot (a predicated store and a
// select, no branch), as the refinement kernel runs it on the schedule as
// built: an FP32 chain is short, so issue slots and shared-memory wavefronts
// bound that kernel, and the branches of spmv_slots and the bank conflicts of
// aligned rows cost it more than they save (150 species x 100,000 cells:
// 1,983 us against 2,195).  block(b, av): the A values of slots 4b .. 4b+3;
// one(j): that of slot j past the last whole block.
template <class T, class Block, class One>
__device__ __forceinline__ void spmv_flat(const SchedWord *__restrict__ sch, int L, int Lc, int sl,
                                          Block block, One one, unsigned gs, unsigned os) {
  const uint4 *s4 = reinterpret_cast<const uint4 *>(sch) + sl;
  T acc = T(0);
  const int nb = L >> 2;
  auto step = [&](unsigned w, T av, T xv) {
    acc = fma_t(av, xv, acc);
    slot_end(w, acc, os);
  };
  if (nb > 0) {
    uint4 w = *s4;
#pragma unroll 1
    for (int b = 0;;) {
      T av[4], x0, x1, x2, x3;
      lds(x0, slot_col_addr<T>(w.x, gs));
      lds(x1, slot_col_addr<T>(w.y, gs));
      lds(x2, slot_col_addr<T>(w.z, gs));
      lds(x3, slot_col_addr<T>(w.w, gs));
      block(b, av);
      uint4 wn = w;
      if (++b < nb) wn = s4[b * Lc];
      step(w.x, av[0], x0);
      step(w.y, av[1], x1);
      step(w.z, av[2], x2);
      step(w.w, av[3], x3);
      if (b == nb) break;
      w = wn;
    }
  }
#pragma unroll
  for (int u = 0; u < 3; ++u)
    if ((L & 3) > u) {
      const unsigned w = sch[(4 * nb + u) * Lc + sl];
      T x;
      lds(x, slot_col_addr<T>(w, gs));
      step(w, one(4 * nb + u), x);
    }
}

// FP32, A32 in slot order in shared memory (word_pos places).
__device__ __forceinline__ void flat_spmvf(const SchedWord *__restrict__ sch, int L, int Lc, int sl,
                                           const float *__restrict__ As, unsigned gs, unsigned os) {
  const float4 *A4 = reinterpret_cast<const float4 *>(As) + sl;
  spmv_flat<float>(
      sch, L, Lc, sl,
      [&](int b, float *av) {
        const float4 p = A4[b * Lc];
        av[0] = p.x; av[1] = p.y; av[2] = p.z; av[3] = p.w;
      },
      [&](int j) { return As[j * Lc + sl]; }, gs, os);
}
// FP64, A in shared memory (pair_pos places), or read from global memory
// through the slots' source entries.
__device__ __forceinline__ void flat_spmv(const SchedWord *__restrict__ sch, int L, int Lc, int sl,
                                          const double *__restrict__ As, unsigned gs, unsigned os) {
  const double2 *A2 = reinterpret_cast<const double2 *>(As) + sl;
  spmv_flat<double>(
      sch, L, Lc, sl,
      [&](int b, double *av) {
        const double2 p = A2[(2 * b) * Lc], q = A2[(2 * b + 1) * Lc];
        av[0] = p.x; av[1] = p.y; av[2] = q.x; av[3] = q.y;
      },
      [&](int j) { return As[pair_pos(j, sl, L, Lc)]; }, gs, os);
}
__device__ __forceinline__ void flat_spmv_gather(const SchedWord *__restrict__ sch,
                                                 const int *__restrict__ src, int L, int Lc, int sl,
                                                 const double *__restrict__ Ag, unsigned gs,
                                                 unsigned os) {
  const int4 *s4 = reinterpret_cast<const int4 *>(src) + sl;
  auto value = [&](int k) { return k >= 0 ? __ldg(Ag + k) : 0.0; };
  spmv_flat<double>(
      sch, L, Lc, sl,
      [&](int b, double *av) {
        const int4 k = __ldg(s4 + b * Lc);
        av[0] = value(k.x); av[1] = value(k.y); av[2] = value(k.z); av[3] = value(k.w);
      },
      [&](int j) { return value(__ldg(src + j * Lc + sl)); }, gs, os);
}

// FP64 -> FP32 conversion, round to nearest even, entirely on the integer
// pipe (on this GPU a hardware F2F conversion occupies the FP64 pipe).  IEEE
// 754 rounding written from its definition: keep 23 of the 52 fraction bits
// and round on the 29 dropped bits, ties to even; a carry out of the fraction
// increments the exponent (and reaches infinity at the top of the range).
// Results below the FP32 normal range are flushed to a signed zero; Inf and
// NaN map to Inf and a quiet NaN.
__device__ __forceinline__ float d2f_rn(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  const unsigned sign = (unsigned)(u >> 32) & 0x80000000u;
  const int ed = (int)((u >> 52) & 0x7ffull);
  const unsigned long long frac = u & 0xfffffffffffffull;
  const int ef = ed - 1023 + 127;
  unsigned m = (unsigned)(frac >> 29);
  const unsigned rem = (unsigned)(frac & 0x1fffffffull);
  m += (rem > 0x10000000u || (rem == 0x10000000u && (m & 1u))) ? 1u : 0u;
  unsigned bits = ((unsigned)ef << 23) + m;          // valid for 1 <= ef <= 254
  bits = (ef >= 255) ? 0x7f800000u : bits;            // overflow -> Inf
  bits = (ef <= 0) ? 0u : bits;                       // underflow -> 0
  bits = (ed == 0x7ff) ? (frac ? 0x7fc00000u : 0x7f800000u) : bits;
  return __uint_as_float(sign | bits);
}

// Exact FP32 -> FP64 widening on the integer pipe (FP32 subnormals, which
// d2f_rn never produces, are read as zero).
__device__ __forceinline__ double f2d_exact(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned ef = (b >> 23) & 0xffu;
  const unsigned long long sign = (unsigned long long)(b >> 31) << 63;
  const unsigned long long mant = (unsigned long long)(b & 0x7fffffu) << 29;
  unsigned long long u = sign | ((unsigned long long)(ef - 127 + 1023) << 52) | mant;
  u = (ef == 0u) ? sign : u;
  u = (ef == 0xffu) ? (sign | (0x7ffull << 52) | mant) : u;
  return __longlong_as_double((long long)u);
}

// x == 0 (either sign) on the bit pattern
__device__ __forceinline__ bool is_zero_bits(double v) {
  return ((unsigned long long)__double_as_longlong(v) << 1) == 0ull;
}

// 1/d in FP64 by Newton-Raphson iteration y <- y + y (1 - d y).  d = m 2^k
// with m in [1, 2) (m and k read from the bit pattern); an FP32
// rcp.approx of m (relative error about 2^-22) seeds STEPS Newton steps on m,
// each squaring the relative error (one step: about 2^-44; two: FP64
// rounding); the exponent of the result is then lowered by k on the bit
// pattern.  Only the 2*STEPS Newton FMAs use the FP64 pipe (a division costs
// about seven).  Zero gives Inf, Inf gives zero, NaN
// stays NaN; results that would leave the normal FP64 range (|d| above
// 2^1022 or below 2^-1022) are returned as zero or Inf.
template <int STEPS>
__device__ __forceinline__ double recip64n(double d) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(d);
  const unsigned long long sign = u & 0x8000000000000000ull;
  const int ed = (int)((u >> 52) & 0x7ffull);
  const unsigned long long frac = u & 0xfffffffffffffull;
  const double m = __longlong_as_double((long long)(frac | (1023ull << 52)));
  float yf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf)
      : "f"(__uint_as_float(0x3f800000u | (unsigned)(frac >> 29))));
  double y = __longlong_as_double((long long)(((unsigned long long)(__float_as_uint(yf) & 0x7fffffu) << 29) |
                                              ((unsigned long long)(((__float_as_uint(yf) >> 23) & 0xffu) - 127 + 1023) << 52)));
#pragma unroll
  for (int s = 0; s < STEPS; ++s) {
    const double r = fma(-m, y, 1.0);
    y = fma(y, r, y);                     // 1/m in (0.5, 1]
  }
  const unsigned long long yu = (unsigned long long)__double_as_longlong(y);
  const int ey = (int)((yu >> 52) & 0x7ffull) - (ed - 1023);
  unsigned long long out = sign | ((unsigned long long)ey << 52) | (yu & 0xfffffffffffffull);
  out = (ey <= 0) ? sign : out;                                   // underflow
  out = (ey >= 0x7ff || ed == 0) ? (sign | (0x7ffull << 52)) : out;  // overflow, 1/0
  out = (ed == 0x7ff) ? (frac ? 0x7ff8000000000000ull : sign) : out;  // NaN, 1/Inf
  return __longlong_as_double((long long)out);
}

// Full-precision reciprocal (two Newton steps): the Jacobi preconditioner.
__device__ __forceinline__ double recip64(double d) { return recip64n<2>(d); }
// Scalars of the iteration (alpha, beta, omega): one step, relative error
// about 2^-44; x and r are updated with the same scalar, so they stay
// consistent and the true-residual test still decides convergence.
__device__ __forceinline__ double recip64s(double d) { return recip64n<1>(d); }

// A high word H such that every v whose |v| has a larger one satisfies
// v^2 > thr, also after rounding: the high word of an upper bound of
// sqrt(thr) (the fraction rounded up to FP32, an approximate FP32 square root,
// 2^-18 on top for its error).  Then a sum of squares that contains v^2, as a
// chain of multiply-adds from zero and the exact sum of the chains, is above
// thr too (each only grows, and rounding is monotone), so the convergence test
// ||r||^2 <= thr needs neither while one entry of r stands out: near
// convergence alone it is evaluated.  Saves 10 of 153 FP64 instructions and
// two of six exact sums per iteration.  thr outside [2^-900, 2^900]: no v.
__device__ __forceinline__ unsigned sqrt_bound_hi(double thr) {
  const unsigned hi = (unsigned)__double2hiint(thr), lo = (unsigned)__double2loint(thr);
  const int ed = (int)(hi >> 20);
  const int e = ed - 1023, odd = e & 1;
  float t = __uint_as_float((0x3f800000u | (hi & 0xfffffu) << 3 | lo >> 29) + 1u);
  t = odd ? t + t : t;
  asm("sqrt.approx.ftz.f32 %0, %0;" : "+f"(t));
  t = fmaf(t, 0x1p-18f, t);
  const unsigned tb = __float_as_uint(t);
  const unsigned H = (unsigned)(1023 + (e - odd) / 2 + (int)(tb >> 23) - 127) << 20 |
                     ((tb >> 3) & 0xfffffu);
  return ed >= 123 && ed <= 1923 ? H : 0x7fffffffu;
}
__device__ __forceinline__ unsigned abs_hi(double v) {
  return (unsigned)__double2hiint(v) & 0x7fffffffu;
}

// Sum of v over the Lc lanes of each segment on the integer pipe.  Every
// term m 2^(e-1075) (53-bit integer m) is aligned to the segment's largest
// exponent as a signed 64-bit fixed-point number with 5 guard bits (room for
// 32 terms), the integers are summed exactly with xor shuffles, and the total
// is rounded once to FP64 (nearest, ties to even).  The error is at most one
// rounding plus 2^-57 of the largest term per term, every lane gets the same
// bits, and no FP64 instruction is issued.  Any NaN or Inf gives NaN; totals
// below the normal FP64 range flush to zero.
__device__ __forceinline__ double seg_sum_exact(double v, int Lc) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  const int e = (int)((u >> 52) & 0x7ffull);
  const unsigned long long frac = u & 0xfffffffffffffull;
  const unsigned long long m = e ? (frac | (1ull << 52)) : frac;
  const int ee = e ? e : 1;
  int emax = ee;
  for (int off = Lc >> 1; off > 0; off >>= 1) emax = max(emax, __shfl_xor_sync(kFull, emax, off));
  const int sh = emax - ee;
  long long f = sh >= 58 ? 0ll : (long long)((m << 5) >> sh);
  f = (u >> 63) ? -f : f;
  for (int off = Lc >> 1; off > 0; off >>= 1) f += __shfl_xor_sync(kFull, f, off);
  const unsigned long long neg = f < 0 ? 1ull : 0ull;
  const unsigned long long a = (unsigned long long)(f < 0 ? -f : f);
  const int lz = __clzll((long long)a);
  const unsigned long long an = a << (lz & 63);
  unsigned long long mant = an >> 11;
  const unsigned rem = (unsigned)(an & 0x7ffull);
  mant += (rem > 0x400u || (rem == 0x400u && (mant & 1ull))) ? 1ull : 0ull;
  int E = (63 - lz) + emax - 57;
  E += (mant >> 53) ? 1 : 0;                 // rounding carried into a new bit
  mant = (mant >> 53) ? (mant >> 1) : mant;
  unsigned long long out = (neg << 63) | ((unsigned long long)E << 52) | (mant & 0xfffffffffffffull);
  out = (E <= 0 || a == 0ull) ? (neg << 63) : out;            // zero / flush
  out = (E >= 0x7ff) ? ((neg << 63) | (0x7ffull << 52)) : out;  // overflow
  out = (emax == 0x7ff) ? 0x7ff8000000000000ull : out;         // NaN or Inf present
  return __longlong_as_double((long long)out);
}

// The same sum with the segment reductions done by full-warp redux.sync (one
// instruction per reduction, all lanes taking part): for each of the K =
// 32/Lc segments, the lanes of that segment contribute and the others add
// the neutral element.  The exponent maximum is reduced directly and the
// 64-bit fixed-point total as three 32-bit sums of its 20-bit digits (at
// most 32 lanes of 20-bit digits cannot overflow 32 bits), recombined
// exactly, so the result is bit-identical to seg_sum_exact.
template <int K>
__device__ __forceinline__ double seg_sum_exact_redux(double v) {
  constexpr int Lc = 32 / K;
  const int seg = (threadIdx.x & 31) / Lc;
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  const int e = (int)((u >> 52) & 0x7ffull);
  const unsigned long long frac = u & 0xfffffffffffffull;
  const unsigned long long m = e ? (frac | (1ull << 52)) : frac;
  const int ee = e ? e : 1;
  int emax = 0;
#pragma unroll
  for (int s = 0; s < K; ++s) {
    const int r = (int)__reduce_max_sync(kFull, seg == s ? (unsigned)ee : 0u);
    emax = seg == s ? r : emax;
  }
  const int sh = emax - ee;
  long long f = sh >= 58 ? 0ll : (long long)((m << 5) >> sh);
  f = (u >> 63) ? -f : f;
  const unsigned d0 = (unsigned)(f & 0xfffffll);
  const unsigned d1 = (unsigned)((f >> 20) & 0xfffffll);
  const int d2 = (int)(f >> 40);
  unsigned s0 = 0, s1 = 0;
  int s2 = 0;
#pragma unroll
  for (int s = 0; s < K; ++s) {
    const bool mine = seg == s;
    const unsigned r0 = __reduce_add_sync(kFull, mine ? d0 : 0u);
    const unsigned r1 = __reduce_add_sync(kFull, mine ? d1 : 0u);
    const int r2 = __reduce_add_sync(kFull, mine ? d2 : 0);
    s0 = mine ? r0 : s0;
    s1 = mine ? r1 : s1;
    s2 = mine ? r2 : s2;
  }
  f = ((long long)s2 << 40) + ((long long)s1 << 20) + (long long)s0;
  const unsigned long long neg = f < 0 ? 1ull : 0ull;
  const unsigned long long a = (unsigned long long)(f < 0 ? -f : f);
  const int lz = __clzll((long long)a);
  const unsigned long long an = a << (lz & 63);
  unsigned long long mant = an >> 11;
  const unsigned rem = (unsigned)(an & 0x7ffull);
  mant += (rem > 0x400u || (rem == 0x400u && (mant & 1ull))) ? 1ull : 0ull;
  int E = (63 - lz) + emax - 57;
  E += (mant >> 53) ? 1 : 0;
  mant = (mant >> 53) ? (mant >> 1) : mant;
  unsigned long long out = (neg << 63) | ((unsigned long long)E << 52) | (mant & 0xfffffffffffffull);
  out = (E <= 0 || a == 0ull) ? (neg << 63) : out;
  out = (E >= 0x7ff) ? ((neg << 63) | (0x7ffull << 52)) : out;
  out = (emax == 0x7ff) ? 0x7ff8000000000000ull : out;
  return __longlong_as_double((long long)out);
}

// Exact segment sum.  With Lc known at compile time (LC > 0) and at most two
// cells per warp, the reductions run as full-warp redux.sync (one instruction
// each; a redux over part of a warp measured several times slower than
// shuffles); otherwise the shuffle form.  Both give the same bits.
template <int LC>
__device__ __forceinline__ double seg_sum_x(double v, int Lc) {
  if constexpr (LC >= 16) return seg_sum_exact_redux<32 / LC>(v);
  else return seg_sum_exact(v, Lc);
}

// A bounded wait ran out: raise the launch's time-out flag (device memory,
// read by the launch's last warp) and the host-mapped error word.
__device__ __forceinline__ void wait_timed_out(int *flag, int *err) {
  atomicExch(flag, 1);
  if (err) {
    *(volatile int *)err = 1;
    __threadfence_system();
  }
}

// Grid barrier of a cooperative launch, bounded in time: the CTA's threads
// meet, thread 0 publishes the CTA's writes and counts it in, then waits
// until the counter reaches target.  A wait longer than `limit` clocks (by
// default about a second; the CTAs of a cooperative launch are all resident,
// so a legitimate wait is microseconds) raises the time-out flags and goes on.
__device__ __forceinline__ void grid_barrier_bounded(unsigned *ctr, unsigned target,
                                                     int *flag, int *err, long long limit) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(ctr, 1u);
    const long long t0 = clock64();
    for (;;) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
      if (v >= target) break;
      if (clock64() - t0 > limit) {
        wait_timed_out(flag, err);
        break;
      }
      __nanosleep(64);
    }
    __threadfence();
  }
  __syncthreads();
}

// In-launch difficulty ordering (run by every CTA of a cooperative solve
// launch before it solves; Args: WarpArgs or MixedArgs).  The estimate, the classes and the hardest-first
// order are those of the separate ordering pass: max_i |A_ii - 1| binned on
// half octaves, here over the sampled diagonal rows (or of |gamma_c|, see
// BY_GAMMA).  Each CTA classifies a contiguous share of the cells, counts them per class in shared memory and
// reserves its range inside each class with one global atomic per class;
// after a grid barrier it turns the class totals into class starts and
// writes its cells' order entries (cell + 1).  A warp that takes a group
// waits for the group's entries (written by whichever CTAs own those cells,
// all resident and past the barrier) and clears them once it has read them,
// so the order is all zero again for the next launch.
// sm: kOrdSmemBytes of this CTA's shared memory not yet in use.
// BY_GAMMA: classify by |gamma_c| instead (the fused assembly and Newton
// launches, whose matrices do not exist before a cell is assembled; gamma
// scales the off-identity part of A = I - gamma J, so it ranks the cells as
// the diagonal estimate does).
__device__ __forceinline__ const double *ord_gamma_of(const WarpArgs &a) { return a.gamma; }
__device__ __forceinline__ const double *ord_gamma_of(const MixedArgs &) { return nullptr; }
template <bool BY_GAMMA, class Args>
__device__ __forceinline__ void order_prologue(const Args &a, int *sm) {
  int *hist = sm;                       // per class: count, then class start
  int *base = sm + kOrdClasses;         // per class: this CTA's offset inside it
  unsigned long long *bkey = reinterpret_cast<unsigned long long *>(sm + 2 * kOrdClasses);
  // per cell of a pass: (estimate high word << 32 | sampled row), then its class word
  unsigned long long *key =
      reinterpret_cast<unsigned long long *>(reinterpret_cast<char *>(sm) + kOrdKeyOffset);
  unsigned *ctr = reinterpret_cast<unsigned *>(a.ord_ws + kOrdClasses);
  const int per = (a.cells + gridDim.x - 1) / gridDim.x;
  const int c0 = min(a.cells, (int)blockIdx.x * per), c1 = min(a.cells, c0 + per);
  const int nr = BY_GAMMA ? 1 : a.ord_nrows;
  // a share of one pass keeps its class words in shared memory
  const bool one_piece = c1 - c0 <= kOrdPiece;
  for (int i = threadIdx.x; i < kOrdClasses; i += blockDim.x) hist[i] = 0;
  if (threadIdx.x == 0) *bkey = 0ull;
  for (int p0 = c0; p0 < c1; p0 += kOrdPiece) {
    const int pc = min(kOrdPiece, c1 - p0);
    for (int i = threadIdx.x; i < pc; i += blockDim.x) key[i] = 0ull;
    __syncthreads();
    // the pass's sampled diagonal entries, flattened; each thread issues a
    // batch of independent loads before it folds them in
    const int m = pc * nr;
    for (int j0 = threadIdx.x; j0 < m; j0 += kOrdBatch * blockDim.x) {
      double v[kOrdBatch];
      int cl[kOrdBatch], q[kOrdBatch];
#pragma unroll
      for (int u = 0; u < kOrdBatch; ++u) {
        const int j = j0 + u * blockDim.x;
        cl[u] = j < m ? j / nr : -1;
        q[u] = j - cl[u] * nr;
        if (cl[u] >= 0)
          v[u] = BY_GAMMA ? __ldg(ord_gamma_of(a) + p0 + cl[u])
                          : __ldg(a.A + (size_t)(p0 + cl[u]) * a.nnz + __ldg(a.ord_rows + q[u]));
      }
#pragma unroll
      for (int u = 0; u < kOrdBatch; ++u)
        if (cl[u] >= 0)
          atomicMax(key + cl[u], (unsigned long long)(BY_GAMMA ? magnitude_hi(v[u])
                                                               : diag_departure_hi(v[u]))
                                         << 32 |
                                     (unsigned)q[u]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < pc; i += blockDim.x) {
      const unsigned long long kk = key[i];
      const int k = difficulty_class<BY_GAMMA ? kTopGamma : kTopDeparture>((unsigned)(kk >> 32));
      const int w = k | atomicAdd(hist + k, 1) << 6;
      if (a.ord_hits) atomicMax(bkey, kk);
      if (one_piece) key[i] = (unsigned)w;
      else a.ord_cls[p0 + i] = w;
    }
    __syncthreads();
  }
  // where the CTA's hardest cell peaked (the host picks the rows to sample)
  if (a.ord_hits && threadIdx.x == 0 && c1 > c0) atomicAdd(a.ord_hits + (unsigned)*bkey, 1u);
  for (int k = threadIdx.x; k < kOrdClasses; k += blockDim.x)
    base[k] = hist[k] ? atomicAdd(a.ord_ws + k, hist[k]) : 0;
  grid_barrier_bounded(ctr, gridDim.x, a.ord_ws + kOrdFlag, a.ord_err, a.ord_wait);
  if (threadIdx.x < 32) {
    // exclusive prefix of the class totals, two classes per lane
    const int l = threadIdx.x;
    const int ta = __ldcg(a.ord_ws + 2 * l), tb = __ldcg(a.ord_ws + 2 * l + 1);
    int s = ta + tb;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(kFull, s, o);
      if (l >= o) s += t;
    }
    hist[2 * l] = s - ta - tb;
    hist[2 * l + 1] = s - tb;
  }
  __syncthreads();
  for (int c = c0 + threadIdx.x; c < c1; c += blockDim.x) {
    const int w = one_piece ? (int)key[c - c0] : __ldcg(a.ord_cls + c);
    const int k = w & (kOrdClasses - 1);
    const int pos = hist[k] + base[k] + (w >> 6);
    if (pos < a.cells) __stcg(a.ord_out + pos, c + 1);  // in range unless the barrier timed out
  }
  __syncthreads();  // the warps' solve regions overlap the shared memory used here
}

// Wait, bounded in time as the barrier, until the in-launch ordering has
// written the order entries *p of the lanes with `mine`.  The entry is the only
// datum passed, so a relaxed load suffices (an acquire would also invalidate
// the SM's L1 each time).  Every lane stays in the loop until all entries are
// there: with the waiting lanes alone in it the warp could go on split, each
// part issuing the whole solve by itself, and which code did so changed with
// register allocation (180 or 204 us at 80 species x 10,000 cells, 95 or 176 at
// 57 x 4,001).
__device__ __forceinline__ void wait_order_entries(const int *p, bool mine, int *flag, int *err,
                                                   long long limit) {
  const long long t0 = clock64();
  for (;;) {
    int v = 1;
    if (mine) asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    if (__all_sync(kFull, v != 0)) return;
    const bool late = clock64() - t0 > limit;
    if (__any_sync(kFull, late)) {
      if (v == 0) wait_timed_out(flag, err);
      break;
    }
    __nanosleep(32);
  }
  __syncwarp();
}

// Next group of this warp in a launch with the dynamic queue (false when none
// is left).  An ordered launch (a.order set) first gives every warp one group
// of a stratified wave, or spreads the tickets over the order when there are
// fewer groups than warps (WarpArgs::ord_wave); `first` starts true.
template <class Args>
__device__ __forceinline__ bool take_group(const Args &a, int warp, int lane, bool &first,
                                           unsigned &g) {
  const bool strat = a.order && a.ord_stride == 0 && a.ord_wave > 0;
  if (first && strat) {
    first = false;
    const unsigned B = gridDim.x, b = blockIdx.x, w = (unsigned)warp;
    g = w * B + ((w & 1u) ? B - 1u - b : b);
    return true;
  }
  first = false;
  unsigned t = 0;
  if (lane == 0) t = atomicAdd(a.queue, 1u);
  t = __shfl_sync(kFull, t, 0);
  if (strat) t += (unsigned)a.ord_wave;
  if (t >= (unsigned)a.ngroups) return false;
  if (a.order && a.ord_stride && t < (unsigned)a.ord_wave)
    t = (unsigned)((unsigned long long)t * (unsigned)a.ord_stride % (unsigned)a.ord_wave);
  g = t;
  return true;
}

// In-launch ordering: lanes 0 .. k-1 wait for the order entries of group g's
// k cells; returns whether this lane owns one (to clear it after the solve).
template <class Args>
__device__ __forceinline__ bool await_order_entries(const Args &a, unsigned g, int k, int lane) {
  if (!a.ord_ws) return false;
  const int p = (int)g * k + lane;
  const bool mine = lane < k && p < a.cells;
  wait_order_entries(a.order + p, mine, a.ord_ws + kOrdFlag, a.ord_err, a.ord_wait);
  return mine;
}

// End of a launch with the dynamic queue, called by every lane of every
// warp once it has no group left: the last warp to finish (every other warp
// has taken its last group before counting itself done, so every CTA is past
// its ordering prologue) resets the queue pair and, after an in-launch
// ordering, the ordering's workspace, so both are ready for the next launch
// in stream order.  If a wait of the ordering ran out, the order may have
// sent some cells to no warp and others to two: that warp then marks every
// cell of the launch CAMP_CELL_INVALID (status, when given) with a NaN
// residual and clears the order entries the launch left set.
template <class Args>
__device__ __forceinline__ void finish_queue(const Args &a, bool ordered, int warps_total,
                                             int lane) {
  unsigned last = 0;
  if (lane == 0) {
    __threadfence();
    last = atomicAdd(a.queue + 1, 1u) == (unsigned)warps_total - 1u ? 1u : 0u;
  }
  last = __shfl_sync(kFull, last, 0);
  if (!last) return;
  __threadfence();
  if (ordered && a.ord_ws && __ldcg(a.ord_ws + kOrdFlag) != 0) {
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    for (int c = lane; c < a.cells; c += 32) {
      a.ord_out[c] = 0;
      a.resid[c] = nan;
      if (a.status) a.status[c] = CAMP_CELL_INVALID;
    }
  }
  if (lane == 0) {
    atomicExch(a.queue, 0u);
    atomicExch(a.queue + 1, 0u);
    if (ordered && a.ord_ws)
      for (int i = 0; i < kOrdWords; ++i) atomicExch(a.ord_ws + i, 0);
  }
}

}  // namespace camp
