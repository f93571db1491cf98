// Device helpers shared by the kernels of the EREM library: warp and block
// reductions, deterministic cross-block partial sums, vector loads and
// stores of the padded layout, exact float -> double conversion, the Leja
// stopping test and the control-block bookkeeping of one Leja substep.
//
// Included by kernels.cu (one translation unit); everything sits in an
// anonymous namespace inside erem.
#pragma once

#include "erem_internal.h"

namespace erem {
namespace {

constexpr int NT = kThreads;

// ---------------------------------------------------------------------------
// small device helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_min(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Sum over 256 threads, valid in tid 0, with the pairs of the butterflies of
// block_reduce_t (a warp's 16, 8, 4, 2, 1, then the warps' 4, 2, 1) and so their
// bits.  A butterfly adds in every lane of every warp: 45 FP64 instructions to a
// block, more than the terms of the sum in a pass with one cell per thread, and
// the FP64 pipe (two results a clock and SM) is what bounds these passes.  One
// warp that reads the 256 terms from shared memory, four lanes to a warp's
// terms, needs 12.  Which warp differs from block to block, since a warp's index
// picks the quarter of the SM whose pipe it uses.  128^3 pressure: A d
// 40.6 -> 38.4 us, the last sweep with (z, r) and (z, Ad) 26.1 -> 22.2, and 19.9
// with both sums together.
// The NV sums of a pass go together: one wait for shared memory, each summed by a
// warp of its own.  The results are valid in every thread.
template <int NV>
__device__ void block_sums256(double (&v)[NV], int tid) {
  __shared__ double all[NV][8 * 36], res[NV];   // pitch 36: the four lanes of eight warps take different banks
  const int warp = ((tid >> 5) + (int)((blockIdx.x * 0x9E3779B1u) >> 29)) & 7;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) all[k][(tid >> 5) * 36 + (tid & 31)] = v[k];
  __syncthreads();
  if (warp < NV) {
    const double* p = all[warp] + ((tid & 31) >> 2) * 36 + (tid & 3);
    double a = ((p[0] + p[16]) + (p[8] + p[24])) + ((p[4] + p[20]) + (p[12] + p[28]));
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    a += __shfl_xor_sync(0xffffffffu, a, 16);
    a += __shfl_xor_sync(0xffffffffu, a, 8);
    a += __shfl_xor_sync(0xffffffffu, a, 4);
    if ((tid & 31) == 0) res[warp] = a;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = res[k];
}

// Block-wide reduction over BS threads with linear index tid; the result is
// valid in tid 0.  OP 0 = sum, 1 = min, 2 = max.  Safe to call repeatedly
// (syncs before reusing smem).
template <int OP, int BS>
__device__ double block_reduce_t(double v, double* sh, int tid) {
  if (OP == 0 && BS == 256) {
    double s[1] = {v};
    block_sums256<1>(s, tid);
    return s[0];
  }
  v = OP == 0 ? warp_sum(v) : (OP == 1 ? warp_min(v) : warp_max(v));
  __syncthreads();
  if ((tid & 31) == 0) sh[tid >> 5] = v;
  __syncthreads();
  if (tid < 32) {
    double w = tid < (BS / 32) ? sh[tid] : (OP == 0 ? 0.0 : (OP == 1 ? INFINITY : -INFINITY));
    w = OP == 0 ? warp_sum(w) : (OP == 1 ? warp_min(w) : warp_max(w));
    v = w;
  }
  return v;
}
template <int OP>
__device__ double block_reduce(double v, double* sh) {
  return block_reduce_t<OP, NT>(v, sh, threadIdx.x);
}

// Publish this block's partials (block bid of nblocks); returns true in every
// thread of the last block to arrive.  part has kRedSlots doubles per block.
__device__ bool publish_partials_t(double* part, unsigned* cnt, const double* vals, int nv,
                                   int tid, int bid, int nblocks) {
  __shared__ int s_last;
  if (tid == 0) {
    for (int k = 0; k < nv; ++k) part[bid * kRedSlots + k] = vals[k];
    __threadfence();
    const unsigned t = atomicAdd(cnt, 1u);
    s_last = (t == (unsigned)nblocks - 1u);
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last != 0;
}
__device__ bool publish_partials(double* part, unsigned* cnt, const double* vals, int nv) {
  return publish_partials_t(part, cnt, vals, nv, threadIdx.x, blockIdx.x, gridDim.x);
}

// Sum (or min/max) of partial k over all blocks, in block order; tid 0.
template <int OP, int BS>
__device__ double gather_partials_t(const double* part, int k, double* sh, int tid, int nblocks) {
  double v = OP == 0 ? 0.0 : (OP == 1 ? INFINITY : -INFINITY);
  for (int b = tid; b < nblocks; b += BS) {
    const double x = __ldcg(part + b * kRedSlots + k);
    v = OP == 0 ? v + x : (OP == 1 ? fmin(v, x) : fmax(v, x));
  }
  return block_reduce_t<OP, BS>(v, sh, tid);
}

// The sums of partials 0 .. NV - 1 over all blocks, in block order, in every
// thread.  The only block that still runs waits here: a thread's loads go out
// together, not one after the other's addition.
template <int NV>
__device__ void gather_sums(const double* part, double (&out)[NV]) {
  constexpr int kBatch = 4;
  const int tid = threadIdx.x, nblocks = gridDim.x;
#pragma unroll
  for (int k = 0; k < NV; ++k) out[k] = 0.0;
  for (int b0 = tid; b0 < nblocks; b0 += kBatch * NT) {
    double x[kBatch][NV];
#pragma unroll
    for (int q = 0; q < kBatch; ++q)
      if (b0 + q * NT < nblocks) {
#pragma unroll
        for (int k = 0; k < NV; ++k) x[q][k] = __ldcg(part + (b0 + q * NT) * kRedSlots + k);
      }
#pragma unroll
    for (int q = 0; q < kBatch; ++q)
      if (b0 + q * NT < nblocks) {
#pragma unroll
        for (int k = 0; k < NV; ++k) out[k] += x[q][k];
      }
  }
  block_sums256<NV>(out, tid);
}
template <int OP>
__device__ double gather_partials(const double* part, int k, double* sh) {
  return gather_partials_t<OP, NT>(part, k, sh, threadIdx.x, gridDim.x);
}

// Arm the control block for a new Leja substep.
__device__ __forceinline__ void arm_ctrl(Ctrl* c, const StopParams& sp) {
  c->done = 0;
  c->degree = 0;
  c->fail = 0;
  c->nonfinite = 0;
  c->m_last = 0;
  c->stop_m = 0x3fffffff;
  c->err = 0.0;
  c->sp = sp;
}

// ---------------------------------------------------------------------------
// vector access to the padded layout
// ---------------------------------------------------------------------------
template <typename Tq, int VEC> struct VecT;
template <> struct VecT<float, 4> { using V = float4; };
template <> struct VecT<float, 2> { using V = float2; };
template <> struct VecT<double, 2> { using V = double2; };

template <typename Tq, int VEC>
__device__ __forceinline__ void ldv(Tq (&r)[VEC], const Tq* p) {
  using V = typename VecT<Tq, VEC>::V;
  const V v = *reinterpret_cast<const V*>(p);
  const Tq* s = reinterpret_cast<const Tq*>(&v);
#pragma unroll
  for (int k = 0; k < VEC; ++k) r[k] = s[k];
}
template <typename Tq, int VEC>
__device__ __forceinline__ void ldv_stream(Tq (&r)[VEC], const Tq* p) {
  using V = typename VecT<Tq, VEC>::V;
  const V v = __ldcs(reinterpret_cast<const V*>(p));
  const Tq* s = reinterpret_cast<const Tq*>(&v);
#pragma unroll
  for (int k = 0; k < VEC; ++k) r[k] = s[k];
}
template <typename Tq, int VEC>
__device__ __forceinline__ void stv(Tq* p, const Tq (&r)[VEC]) {
  using V = typename VecT<Tq, VEC>::V;
  V v;
  Tq* d = reinterpret_cast<Tq*>(&v);
#pragma unroll
  for (int k = 0; k < VEC; ++k) d[k] = r[k];
  *reinterpret_cast<V*>(p) = v;
}
// VEC doubles of P, streamed (read once, written once per term)
template <int VEC>
__device__ __forceinline__ void ldP(double (&r)[VEC], const double* p) {
#pragma unroll
  for (int k = 0; k < VEC; k += 2) {
    const double2 v = __ldcs(reinterpret_cast<const double2*>(p + k));
    r[k] = v.x;
    r[k + 1] = v.y;
  }
}
template <int VEC>
__device__ __forceinline__ void stP(double* p, const double (&r)[VEC]) {
#pragma unroll
  for (int k = 0; k < VEC; k += 2) __stcs(reinterpret_cast<double2*>(p + k), make_double2(r[k], r[k + 1]));
}

// float -> double, exact, from the bit fields with integer instructions
// only (the FP64 pipe of GB300 is the scarce unit in the FP32-bulk sweep, and
// a hardware conversion kept for rare inputs is if-converted into one that
// every call executes): normal numbers, infinities and NaNs by widening the
// fields, zeros by their sign, and a subnormal f through 2^24 f (an exact
// FP32 product, and a normal number) with 24 taken off the exponent.
__device__ __forceinline__ double f2d_fast(float f) {
  const unsigned e0 = (__float_as_uint(f) >> 23) & 0xffu;
  const float g = e0 == 0u ? f * 16777216.0f : f;
  const unsigned u = __float_as_uint(g);
  const unsigned e = (u >> 23) & 0xffu;
  const unsigned E = e == 0xffu ? 0x7ffu : e + (e0 == 0u ? 872u : 896u);
  const unsigned hi = e == 0u ? (u & 0x80000000u)
                              : (u & 0x80000000u) | (E << 20) | ((u & 0x7fffffu) >> 3);
  const unsigned lo = e == 0u ? 0u : u << 29;
  return __hiloint2double((int)hi, (int)lo);
}

// |x| as ordered bits (for |x| the order of the bits is the order of the
// values) and a finiteness test on them: integer operations only.
__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffULL;
}
__device__ __forceinline__ bool bits_finite(unsigned long long b) {
  return (b >> 52) != 0x7ffULL;
}

// sqrt(x) for x >= 0 (infinities, NaNs and negative x give what sqrt gives): the
// FP32 reciprocal root of the significand scaled to [1, 4), then two Newton
// steps for the root in FP64 (each squares the relative error: 2^-22, 2^-43,
// 2^-53), 7 FP64 operations.  An FP64 operation holds a scheduler's FP64 unit
// for 64 cycles on this part, and the library's sqrt() is a chain of many.
__device__ __forceinline__ double sqrt_newton(double x) {
  const unsigned long long b = abs_bits(x);
  const int e = (int)(b >> 52);
  if (x < 0.0 || e == 0 || e == 0x7ff) return sqrt(x);   // zeros, subnormals, infinities, NaNs
  const int h = (e - 1023) >> 1;                         // x = m 4^h, 1 <= m < 4
  const double m = __longlong_as_double((long long)(b - ((unsigned long long)(2 * h) << 52)));
  const double y = f2d_fast(rsqrtf(__double2float_rn(m)));
  const double hy = 0.5 * y;
  double s = m * y;
  s = fma(fma(-s, s, m), hy, s);
  s = fma(fma(-s, s, m), hy, s);
  return __longlong_as_double(__double_as_longlong(s) + ((long long)h << 52));
}

// n / d by Newton's method: the reciprocal of d's significand from FP32 (2^-22
// after rounding d to 24 bits), one Newton step for it in FP64 (2^-44), and
// the residual correction of the quotient, q + (n - d q) y, which is exact up to
// its last rounding and 2^-88 of the quotient: the correctly rounded quotient
// but for one in about 10^10 operand pairs, and then one unit in the last
// place off.  Five FP64 operations, the rest on integers and FP32.  Operands
// outside 2^+-500 (zero numerators apart) take the ordinary division.
__device__ __forceinline__ double div_newton(double n, double d) {
  const unsigned dh = (unsigned)__double2hiint(d), dl = (unsigned)__double2loint(d);
  const unsigned nh = (unsigned)__double2hiint(n);
  const unsigned ed = (dh >> 20) & 0x7ffu, en = (nh >> 20) & 0x7ffu;
  const bool zero_n = abs_bits(n) == 0ULL;
  if (ed - 523u > 1000u || (en - 523u > 1000u && !zero_n)) return n / d;
  // |d| = m 2^(ed - 1023), m rounded to a float in [1, 2]
  const unsigned mb = 0x3f800000u + ((((dh & 0xfffffu) << 3) | (dl >> 29)) + ((dl >> 28) & 1u));
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(mb)));
  const unsigned rb = __float_as_uint(r);
  const unsigned er = ((rb >> 23) & 0xffu) + 896u + 1023u - ed;   // exponent of y 2^-(ed - 1023)
  double y = __hiloint2double((int)((dh & 0x80000000u) | (er << 20) | ((rb & 0x7fffffu) >> 3)),
                              (int)(rb << 29));
  y = fma(fma(-d, y, 1.0), y, y);
  const double q = n * y;
  return fma(fma(-d, q, n), y, q);
}

// Compensated FP32 sum of squares, hi + lo, with the range of FP64: from 2^100 on
// (by a square or by the sum) it is kept times 2^-64, so that only a square that
// is itself infinite makes it so.  Newton vectors of converging interpolations
// reach ||q||^2 of 10^50 and more, and FP32 ends at 3.4e38.  What a scaled sum
// loses of its small terms (below 2^-62) is beyond FP64's precision of a sum above
// 2^100.  With sc = 1 every operation has the bits of the plain pair, and the
// range costs a maximum, a comparison and a branch that is not taken.
constexpr float kSquareBig = 0x1p100f, kSquareDown = 0x1p-64f;
struct SquareSum {
  float hi = 0.f, lo = 0.f, sc = 1.f;
  __device__ __forceinline__ void down() {
    if (sc != 1.f) return;
    sc = kSquareDown;
    hi *= kSquareDown;
    lo *= kSquareDown;
  }
  __device__ __forceinline__ void add(float sq) {
    if (fmaxf(hi, sq) > kSquareBig) down();
    const float s = fmaf(sq, sc, hi);
    const float bp = s - hi;
    lo += (hi - (s - bp)) + fmaf(sq, sc, -bp);
    hi = s;
  }
};
// The same for a thread that adds at most 1 / sc squares: all of them times sc, a
// power of two, so that the sum stays in range as long as each square does, with
// no test and no further register.  The bits are those of the plain pair unless a
// square is below 2^-126 / sc.
__device__ __forceinline__ void add_square(float sq, float sc, float& hi, float& lo) {
  const float s = fmaf(sq, sc, hi);
  const float bp = s - hi;
  lo += (hi - (s - bp)) + fmaf(sq, sc, -bp);
  hi = s;
}

// The Leja copy of J is interleaved per warp tile of T = 32 VEC cells: the
// tile's NC coefficient arrays D W E S N (B T) follow one another, T values
// each.  A warp whose lanes own 32 consecutive VEC-cell vectors reads each
// coefficient as one contiguous 512-byte run, and the NC runs of a tile are
// adjacent in memory (one stream instead of NC).  c[k] points at coefficient
// k of tile 0; the vector starting at cell i reads c[k] + leja_off(i).
template <typename Tq>
struct LejaCoef {
  const Tq* c[7];
  int nc;
  // diagonal-free copy (c[0] unused): the row sum of each x = 0 cell, one per
  // (y, z) row; every other row of J sums to zero (a uniform temperature is
  // transported nowhere in the interior)
  const Tq* r0;
};
template <int T>
__device__ __forceinline__ size_t leja_off(int i, int nc) {
  return (size_t)i + (size_t)(i / T) * (size_t)(nc - 1) * T;
}

// Stopping test of §4.2 on the estimate of term m (thread 0 of the last block).
__device__ void stop_test(Ctrl* c, int m, double dm, double S) {
  const StopParams sp = c->sp;
  const double scal = sp.tol_a + sp.tol_r * c->yinf;
  // one thread on the critical path of a launch: the library's division and
  // root are chains of a thousand cycles and more
  const double e = div_newton(fabs(sp.delta * dm), scal) * sqrt_newton(div_newton(S, sp.ncells));
  c->e[m] = e;
  c->m_last = m;
  if (!bits_finite(abs_bits(e))) {
    c->nonfinite = 1;
    c->done = 1;
    return;
  }
  const int lo = max(1, m - sp.window + 1);
  double mean = 0.0;
  for (int k = lo; k <= m; ++k) mean += c->e[k];
  mean = div_newton(mean, (double)(m - lo + 1));
  c->err = mean;
  if (sp.replay) return;
  if (sp.pow10 * mean < 1.0) {
    c->done = 1;
    c->degree = m;
  } else if (m >= sp.m_max) {
    c->fail = 1;
    c->done = 1;
  }
}

template <typename Tq>
__device__ __forceinline__ double to_f64_fast(Tq v) {
  if constexpr (sizeof(Tq) == 4) return f2d_fast(v);
  else return v;
}

}  // namespace
}  // namespace erem
