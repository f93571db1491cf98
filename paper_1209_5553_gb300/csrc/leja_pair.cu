// Two Leja terms in one pass over a large 3D grid (FP32-bulk).
//
// A term moves 24 bytes of couplings per cell and, averaged over odd and even
// terms, 16 of vectors and running sum; two terms in one pass read the
// couplings once and never write the vector between them: 48 bytes per cell
// and pair instead of 80 (diagonal-free copy).
//
// One CTA per SM owns a block of whole rows, [y0, y1) x [z0, z1), and marches
// through its planes.  Step k forms q_m on plane z (the block's rows and one
// row on either side, formed again by the neighbour) from three planes of
// q_{m-1} in shared memory, and q_{m+1} on plane z - 1 from three planes of q_m
// in shared memory; the couplings of a plane, read once, stay in the
// registers of the thread that owns the cells from the first use to the
// second.  q_{m+1} on plane z - 1 needs its neighbours' q_m of that plane only, formed
// a step ago: a warp announces its part of plane z and waits for the others'
// plane z - 1, so warps run up to a step apart and the FP64 operations of P (half
// of a step's time on their pipe) run beside other warps' stencils.  Planes of
// couplings, of q_{m-1} and of P arrive by bulk copies (the tile-interleaved copy
// of J makes the rows of a plane one contiguous range) two steps ahead of their
// use, and are fetched into L2 two planes before that.
//
// Every cell takes the operations of k_leja_term in the same order (the same
// bits), also in the rows and planes that two blocks form.  P receives
// d_{m-1} q_{m-1} + d_m q_m, as at an odd term of the single form; a substep that
// stops at m + 1 has P short of d_{m+1} q_{m+1}, which its consumer adds.
//
// What bounds it: DRAM moves the 48 bytes and no more (256^3: 796 MB a pair,
// 5.7 TB/s); a step's instructions (FP64 pipe 46 %, issue 56 %, with 19 warps of
// 96 registers) take longer than its copies.  Measured per term, against
// k_leja_term and k_leja_term_lag: 256^3 70 us (107), 224^3 53 (75), 192^3 38 (48),
// 128^3 14.6 (17.3), 96 x 400 x 100 23 (27); with the diagonal 224^3 56 (84),
// 128^3 16.0 (18.3).  An earlier form took 82 us at 256^3 with one block barrier per
// step, 95 without the fetch into L2.
#include <algorithm>

#include "erem_internal.h"
#include "device_common.cuh"

namespace erem {
namespace {

constexpr int kPairThreads = 608;    // at most: 576 vectors of a plane and the copying warp
constexpr int kPairAhead = 2;        // planes fetched into L2 before their copies
constexpr int kPairPolls = 1 << 18;   // polls of a barrier before a wait gives up (about a second: a poll in
                                     // vain took 3.8 us)

struct PairArgs {
  const float* qi;     // q_{m-1}
  float* qo;           // q_{m+1}
  double* P;
  const double* p0;    // m = 1: P starts from d_0 p0
  const float* jl;
  const float* r0;
  const double* xi;
  const double* dd;
  double cg;
  int m, m_end;        // terms m and m + 1; tests up to term m_end
  int px, ny, nz, rows, zc, nby;   // block: rows x zc planes; blocks in y
  int cf_bytes, q0_bytes, q1_bytes, p_bytes;   // shared memory of one plane of each
  float sq_scale;      // 2^-k, at least as many squares as a thread adds up to (planes)
  int polls;           // of a wait for a step's copies or vectors before it gives up
  double* part;
  unsigned* cnt;
  Ctrl* ctrl;
};

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_load(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void bulk_prefetch(const void* src, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
// Wait (bounded) for the phase of the given parity; false when the limit ran out.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, int polls) {
  for (int k = 0; k < polls; ++k) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

__device__ __forceinline__ void lds4(float (&r)[4], unsigned p) {
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]) : "r"(p));
}
__device__ __forceinline__ float lds1(unsigned p) {
  float r;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(r) : "r"(p));
  return r;
}
__device__ __forceinline__ double2 lds2d(unsigned p) {
  double2 r;
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(r.x), "=d"(r.y) : "r"(p));
  return r;
}
__device__ __forceinline__ void sts4(unsigned p, const float (&r)[4]) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(p), "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3])
               : "memory");
}

// float -> double, exact, four at a time: where all four are zeros or normal
// numbers (the usual case) the fields are widened in six instructions each,
// otherwise by f2d_fast
__device__ __forceinline__ void widen4(double (&d)[4], const float (&f)[4]) {
  unsigned small = 0xffffffffu, big = 0u;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const unsigned w = __float_as_uint(f[k]) & 0x7fffffffu;
    small = min(small, w - 1u);   // a zero counts as the largest
    big = max(big, w);
  }
  if (small >= 0x007fffffu && big < 0x7f800000u) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int u = __float_as_int(f[k]);
      const int hi = ((u >> 3) & 0x8fffffff) + 0x38000000;
      d[k] = __hiloint2double(f[k] == 0.0f ? u : hi, u << 29);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k] = f2d_fast(f[k]);
  }
}

// The stencil of one vector: c holds (D) W E S N B T in turn.
template <bool ND>
__device__ __forceinline__ void pair_stencil(float (&out)[4], const float (&c)[ND ? 6 : 7][4],
                                             const float (&qc)[4], float ql, float qr,
                                             const float (&qs)[4], const float (&qn)[4],
                                             const float (&qb)[4], const float (&qt)[4], float r0,
                                             float sh) {
  constexpr int o = ND ? 0 : 1;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float west = k == 0 ? ql : qc[k - 1];
    const float east = k == 3 ? qr : qc[k + 1];
    float a;
    if constexpr (ND) {
      a = ((k == 0 ? r0 : 0.0f) - sh) * qc[k];
      a = fmaf(c[o][k], west - qc[k], a);
      a = fmaf(c[o + 1][k], east - qc[k], a);
      a = fmaf(c[o + 2][k], qs[k] - qc[k], a);
      a = fmaf(c[o + 3][k], qn[k] - qc[k], a);
      a = fmaf(c[o + 4][k], qb[k] - qc[k], a);
      a = fmaf(c[o + 5][k], qt[k] - qc[k], a);
    } else {
      a = (c[0][k] - sh) * qc[k];
      a = fmaf(c[o][k], west, a);
      a = fmaf(c[o + 1][k], east, a);
      a = fmaf(c[o + 2][k], qs[k], a);
      a = fmaf(c[o + 3][k], qn[k], a);
      a = fmaf(c[o + 4][k], qb[k], a);
      a = fmaf(c[o + 5][k], qt[k], a);
    }
    out[k] = a;
  }
}

// a vector's squares, times sc
__device__ __forceinline__ void add_squares(const float (&a)[4], float sc, float& hi, float& lo) {
  float sq = 0.0f;
#pragma unroll
  for (int k = 0; k < 4; ++k) sq = fmaf(a[k], a[k], sq);
  add_square(sq, sc, hi, lo);
}

template <bool ND, bool FIRST>
__global__ void __launch_bounds__(kPairThreads, 1) k_leja_pair(const PairArgs a) {
  constexpr int NC = ND ? 6 : 7;
  extern __shared__ __align__(128) unsigned char smem[];
  // [0, 1]: the copies of even and odd steps; [2, 3]: q_m formed, even and odd steps
  __shared__ __align__(8) unsigned long long s_bar[4];
  __shared__ double s_red[2][kPairThreads / 32];
  __shared__ int s_last, s_late;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int nwarp = blockDim.x >> 5;
  const bool copy_warp = wid == nwarp - 1, copier = copy_warp && lane == 0;
  const int y0 = (blockIdx.x % a.nby) * a.rows, y1 = min(y0 + a.rows, a.ny);
  const int z0 = (blockIdx.x / a.nby) * a.zc, z1 = min(z0 + a.zc, a.nz);
  const int plane = a.px * a.ny;
  unsigned char* const s_cf = smem;                                  // 2 planes of couplings
  unsigned char* const s_q0 = s_cf + 2 * (size_t)a.cf_bytes;         // 4 planes of q_{m-1}
  unsigned char* const s_q1 = s_q0 + 4 * (size_t)a.q0_bytes;         // 4 planes of q_m
  unsigned char* const s_P = s_q1 + 4 * (size_t)a.q1_bytes;          // 2 planes of P
  const unsigned bar0 = smem_u32(&s_bar[0]);
  const int zf = max(z0 - 1, 0), zl = min(z1, a.nz - 1);   // planes of q_m
  const int K = zl - zf + 1;

  // plane p of q_{m-1}: rows [y0 - 2, y1 + 2), slot (p - zf + 1) & 3
  const int qa = max(y0 - 2, 0), qb_ = min(y1 + 2, a.ny);
  const unsigned q0b = (unsigned)(qb_ - qa) * a.px * 4u;
  auto load_q0 = [&](int p, unsigned bar) {
    bulk_load(smem_u32(s_q0) + ((p - zf + 1) & 3) * a.q0_bytes + (unsigned)(qa - (y0 - 2)) * a.px * 4u,
              a.qi + (size_t)p * plane + (size_t)qa * a.px, q0b, bar);
  };
  // couplings of plane p: rows [y0 - 1, y1 + 1), the tiles of 128 cells that hold them
  const int ca = max(y0 - 1, 0), cb = min(y1 + 1, a.ny);
  auto tile0 = [&](int p) { return (p * plane + ca * a.px) >> 7; };   // cells fit 31 bits
  auto tiles = [&](int p) { return ((p * plane + cb * a.px + 127) >> 7) - tile0(p); };
  auto load_cf = [&](int p, unsigned bar) {
    bulk_load(smem_u32(s_cf) + ((p - zf) & 1) * a.cf_bytes, a.jl + (size_t)tile0(p) * (128 * NC),
              (unsigned)tiles(p) * (128u * NC * 4u), bar);
  };
  // the block's rows of P (m = 1: of p0) on plane p, where P is updated
  const double* Pin = FIRST ? a.p0 : a.P;
  const unsigned pb = (unsigned)(y1 - y0) * a.px * 8u;
  auto p_bytes = [&](int p) { return p >= z0 && p < z1 ? pb : 0u; };
  auto load_P = [&](int p, unsigned bar) {
    if (p >= z0 && p < z1)
      bulk_load(smem_u32(s_P) + ((p - zf) & 1) * a.p_bytes, Pin + (size_t)p * plane + (size_t)y0 * a.px, pb,
                bar);
  };
  // the block's own rows of plane p on their way into L2 (its neighbours
  // fetch theirs): two planes of copies in flight do not cover the latency of
  // DRAM under load
  auto ahead = [&](int p) {
    if (p < a.nz && p <= z1) {
      const size_t r = (size_t)p * plane + (size_t)y0 * a.px;
      const size_t e = (size_t)p * plane + (size_t)y1 * a.px;
      const size_t t0 = r / 128, t1 = (e + 127) / 128;
      bulk_prefetch(a.jl + t0 * (128 * NC), (unsigned)(t1 - t0) * (128u * NC * 4u));
      bulk_prefetch(a.qi + r, (unsigned)(e - r) * 4u);
      bulk_prefetch(Pin + r, (unsigned)(e - r) * 8u);
    }
  };
  if (tid == 0) {
    mbar_init(bar0, 1);
    mbar_init(bar0 + 8, 1);
    mbar_init(bar0 + 16, nwarp - 1);
    mbar_init(bar0 + 24, nwarp - 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_late = 0;
  }
  __syncthreads();
  // The couplings do not depend on the launch before: their first planes are
  // on the way while its last blocks finish.
  if (copier) {
    const unsigned n0 = (zf > 0 ? 1 : 0) + 1 + (zf + 1 < a.nz ? 1 : 0);
    mbar_expect(bar0, (unsigned)tiles(zf) * (128u * NC * 4u) + n0 * q0b + p_bytes(zf));
    load_cf(zf, bar0);
    if (K > 1) {
      mbar_expect(bar0 + 8, (unsigned)tiles(zf + 1) * (128u * NC * 4u) + (zf + 2 < a.nz ? q0b : 0u) +
                                p_bytes(zf + 1));
      load_cf(zf + 1, bar0 + 8);
    }
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  // every copy announced above is also started: the block may only leave with
  // none in flight
  if (copier) {
    if (zf > 0) load_q0(zf - 1, bar0);
    load_q0(zf, bar0);
    if (zf + 1 < a.nz) load_q0(zf + 1, bar0);
    if (K > 1 && zf + 2 < a.nz) load_q0(zf + 2, bar0 + 8);
    load_P(zf, bar0);
    if (K > 1) load_P(zf + 1, bar0 + 8);
  }
  if (copier)
    for (int d = 2; d < 2 + kPairAhead; ++d) ahead(zf + d);
  if (*(volatile int*)&a.ctrl->done) {
    if (!mbar_wait(bar0, 0, kPairPolls) || (K > 1 && !mbar_wait(bar0 + 8, 0, kPairPolls)))
      atomicOr(&a.ctrl->flags, FLAG_TIMEOUT);
    return;
  }

  const int m = a.m;
  const float sh1 = (float)(a.cg + a.xi[m - 1]), sh2 = (float)(a.cg + a.xi[m]);
  const double dm = a.dd[m], dm1 = a.dd[m - 1];
  // the thread's vector: row y (from y0 - 1), cells ix ..
  const int vrow = a.px / 4;
  const int y = y0 - 1 + tid / vrow;
  const int ix = (tid - (tid / vrow) * vrow) * 4;
  const bool own1 = y >= 0 && y < a.ny && y <= y1;   // forms q_m here
  const bool own2 = y >= y0 && y < y1;               // ... and q_{m+1}, P, the norms
  const bool has_w = ix > 0, has_e = ix + 4 < a.px;
  const int oS = y > 0 ? -4 * a.px : 0, oN = y < a.ny - 1 ? 4 * a.px : 0;
  const int cell = y * a.px + ix;                                          // in its plane
  const unsigned cf0 = smem_u32(s_cf);
  const unsigned q00 = smem_u32(s_q0) + 4u * ((y - (y0 - 2)) * a.px + ix);   // in a plane of q_{m-1}
  const unsigned q10 = smem_u32(s_q1) + 4u * ((y - (y0 - 1)) * a.px + ix);   // in a plane of q_m
  const unsigned p00 = smem_u32(s_P) + 8u * ((y - y0) * a.px + ix);          // in a plane of P
  float h1 = 0.f, l1 = 0.f, h2 = 0.f, l2 = 0.f;
  float cp[NC][4];       // couplings of plane z - 1
  float rp = 0.f;        // ... and its row sum at x = 0
  bool late = false;
  float rn = 0.f;        // ... of plane z, read one step ahead
  const bool col0 = ND && own1 && ix == 0;
  if (col0) rn = a.r0[zf * a.ny + y];

  if (copy_warp) {
    // once q_m is formed on plane z, the couplings' buffer of this step and
    // plane z - 1 of q_{m-1} are free for the copies of the step after the next.
    // (The step's own copies have landed then, unless a wait for them ran out: its
    // barrier may only be announced again when they have.)
    if (copier) {
      int issued = min(K, 2);   // steps whose copies were started
      for (int k = 0; k + 2 < K; ++k) {
        const int z = zf + k;
        const unsigned bar = bar0 + 8 * (k & 1), phase = (k >> 1) & 1;
        if (!mbar_wait(bar0 + 16 + 8 * (k & 1), phase, a.polls) || !mbar_wait(bar, phase, a.polls)) {
          late = true;
          break;
        }
        const bool more = z + 3 < a.nz;
        mbar_expect(bar, (unsigned)tiles(z + 2) * (128u * NC * 4u) + (more ? q0b : 0u) + p_bytes(z + 2));
        load_cf(z + 2, bar);
        if (more) load_q0(z + 3, bar);
        load_P(z + 2, bar);
        ahead(z + 2 + kPairAhead);
        issued = k + 3;
      }
      // the block leaves with no copy in flight, also where waits ran out
      for (int k = max(issued - 2, 0); k < issued; ++k)
        if (!mbar_wait(bar0 + 8 * (k & 1), (k >> 1) & 1, kPairPolls)) late = true;
    }
    __syncwarp();
  }
  for (int k = 0; k <= K && !copy_warp; ++k) {
    const int z = zf + k;
    float cn[NC][4];
    float rz = 0.f;
    if (k < K) {
      rz = rn;
      if (col0 && k + 1 < K) rn = a.r0[(z + 1) * a.ny + y];
      if (!late && !mbar_wait(bar0 + 8 * (k & 1), (k >> 1) & 1, a.polls)) late = true;
      float qc[4], out[4];
      if (own1) {
        {
          const int i = z * plane + cell;
          const unsigned cf = cf0 + (unsigned)((k & 1) * a.cf_bytes) +
                              4u * (unsigned)(((i >> 7) - tile0(z)) * (128 * NC) + (i & 127));
#pragma unroll
          for (int j = 0; j < NC; ++j) lds4(cn[j], cf + j * 512);
        }
        const unsigned c0 = q00 + (unsigned)(((k + 1) & 3) * a.q0_bytes);
        const unsigned b0 = q00 + (unsigned)((k & 3) * a.q0_bytes);
        const unsigned t0 = q00 + (unsigned)(((k + 2) & 3) * a.q0_bytes);
        float qs[4], qn[4], qb[4], qt[4];
        lds4(qc, c0);
        lds4(qs, c0 + oS);
        lds4(qn, c0 + oN);
        lds4(qb, z > 0 ? b0 : c0);
        lds4(qt, z < a.nz - 1 ? t0 : c0);
        const float ql = has_w ? lds1(c0 - 4) : 0.f, qr = has_e ? lds1(c0 + 16) : 0.f;
        pair_stencil<ND>(out, cn, qc, ql, qr, qs, qn, qb, qt, rz, sh1);
        sts4(q10 + (unsigned)((k & 3) * a.q1_bytes), out);
      }
      const bool sum = own2 && z >= z0 && z < z1;
      double p[4];
      if (sum) {
        const double2 u = lds2d(p00 + (unsigned)((k & 1) * a.p_bytes));
        const double2 v = lds2d(p00 + (unsigned)((k & 1) * a.p_bytes) + 16);
        p[0] = u.x; p[1] = u.y; p[2] = v.x; p[3] = v.y;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar0 + 16 + 8 * (k & 1));
      if (sum) {
        double w1[4];
        widen4(w1, out);
        if constexpr (FIRST) {
#pragma unroll
          for (int j = 0; j < 4; ++j) p[j] = fma(dm, w1[j], dm1 * p[j]);
        } else {
          double w0[4];
          widen4(w0, qc);
#pragma unroll
          for (int j = 0; j < 4; ++j) p[j] = fma(dm, w1[j], fma(dm1, w0[j], p[j]));
        }
        stP<4>(a.P + z * plane + cell, p);
        add_squares(out, a.sq_scale, h1, l1);
      }
    }
    if (k > 0 && !late && !mbar_wait(bar0 + 16 + 8 * ((k - 1) & 1), ((k - 1) >> 1) & 1, a.polls))
      late = true;
    const int zb = z - 1;   // q_{m+1}
    if (own2 && zb >= z0 && zb < z1) {
      const unsigned c1 = q10 + (unsigned)(((k + 3) & 3) * a.q1_bytes);
      const unsigned b1 = q10 + (unsigned)(((k + 2) & 3) * a.q1_bytes);
      const unsigned t1 = q10 + (unsigned)((k & 3) * a.q1_bytes);
      float qc[4], qs[4], qn[4], qb[4], qt[4], out[4];
      lds4(qc, c1);
      lds4(qs, c1 + oS);
      lds4(qn, c1 + oN);
      lds4(qb, zb > 0 ? b1 : c1);
      lds4(qt, zb < a.nz - 1 ? t1 : c1);
      const float ql = has_w ? lds1(c1 - 4) : 0.f, qr = has_e ? lds1(c1 + 16) : 0.f;
      pair_stencil<ND>(out, cp, qc, ql, qr, qs, qn, qb, qt, rp, sh2);
      stv<float, 4>(a.qo + zb * plane + cell, out);
      add_squares(out, a.sq_scale, h2, l2);
    }
#pragma unroll
    for (int j = 0; j < NC; ++j)
#pragma unroll
      for (int v = 0; v < 4; ++v) cp[j][v] = cn[j][v];
    rp = rz;
  }
  if (late) s_late = 1;

  // ||q_m||^2 and ||q_{m+1}||^2, in a fixed order
  const double n1 = warp_sum(f2d_fast(h1) + f2d_fast(l1));
  const double n2 = warp_sum(f2d_fast(h2) + f2d_fast(l2));
  if (lane == 0) {
    s_red[0][wid] = n1;
    s_red[1][wid] = n2;
  }
  __syncthreads();
  if (wid == 0) {
    const double b1 = warp_sum(lane < nwarp ? s_red[0][lane] : 0.0);
    const double b2 = warp_sum(lane < nwarp ? s_red[1][lane] : 0.0);
    if (lane == 0) {
      if (s_late) atomicOr(&a.ctrl->flags, FLAG_TIMEOUT);
      a.part[(size_t)blockIdx.x * kRedSlots] = b1;
      a.part[(size_t)blockIdx.x * kRedSlots + 1] = b2;
      __threadfence();
      s_last = atomicAdd(a.cnt, 1u) == gridDim.x - 1u;
      if (s_last) __threadfence();
    }
    __syncwarp();
    if (s_last) {
      double S1 = 0.0, S2 = 0.0;
      for (int b = lane; b < (int)gridDim.x; b += 32) {
        S1 += __ldcg(a.part + (size_t)b * kRedSlots);
        S2 += __ldcg(a.part + (size_t)b * kRedSlots + 1);
      }
      S1 = warp_sum(S1);
      S2 = warp_sum(S2);
      if (lane == 0) {
        *a.cnt = 0;
        const double back = 1.0 / (double)a.sq_scale;   // a power of two
        stop_test(a.ctrl, m, dm, S1 * back);
        if (!a.ctrl->done && m + 1 <= a.m_end) stop_test(a.ctrl, m + 1, a.dd[m + 1], S2 * back);
      }
    }
  }
}

struct PairShape {
  int rows = 0, zc = 0, nby = 0, grid = 0, threads = 0;
  int cf = 0, q0 = 0, q1 = 0, pl = 0;
  size_t smem = 0;
};

// The block shape: at most one block per SM, the shortest march.  A step takes
// about 0.9 us + 2.6 ns per vector of its rows (the rows formed for neighbours
// included), 2.1 us at 256^3, and there are two steps more than planes.
PairShape pair_shape(const erem_ctx* c) {
  PairShape best;
  const int nc = c->jl_nodiag ? 6 : 7, vrow = c->px / 4;
  long long cost = -1;
  for (int rows = 1; rows <= c->ny; ++rows) {
    PairShape s;
    if ((rows + 2) * vrow > kPairThreads - 32) break;
    s.rows = rows;
    s.nby = (c->ny + rows - 1) / rows;
    if (s.nby > c->sm_count) continue;
    const int nbz = std::min(c->nz, c->sm_count / s.nby);
    s.zc = (c->nz + nbz - 1) / nbz;
    s.grid = s.nby * ((c->nz + s.zc - 1) / s.zc);
    s.threads = ((rows + 2) * vrow + 31) / 32 * 32 + 32;
    const int edge = (rows + 2) * c->px;   // a plane's rows need not start on a tile
    s.cf = (c->px % 128 == 0 ? edge / 128 : (edge + 127) / 128 + 1) * 128 * nc * 4;
    s.q0 = (rows + 4) * c->px * 4;
    s.q1 = (rows + 2) * c->px * 4;
    s.pl = rows * c->px * 8;
    s.smem = 2 * (size_t)(s.cf + s.pl) + 4 * (size_t)(s.q0 + s.q1);
    if (s.smem + 2048 > (size_t)c->smem_optin) break;
    const long long t = (long long)((rows + 2) * vrow + 350) * (s.zc + 2);
    if (cost < 0 || t < cost) {
      cost = t;
      best = s;
    }
  }
  return best;
}

}  // namespace

// Whether the terms run in pairs: FP32-bulk in 3D, at least four rows to a
// block (fewer, and a block forms half of its rows for its neighbours: rows of
// up to 384 cells).  At four rows a pair was still 8 % faster than two terms
// (384 x 160 x 160: 60.4 against 65.9 us a term), at every other size tried from
// 1.5 million cells up (smaller grids are resident) 5 to 35 %.  FP64 terms are
// bound by the FP64 pipe, which rows formed twice would load more.
bool leja_pair_fits(const erem_ctx* c) {
  if (!c->pair_ok || c->dim != 3 || c->prec != EREM_FP32_BULK) return false;
  return pair_shape(c).rows >= std::min(4, c->ny);
}

// Terms m (odd) and m + 1 from q[qin]; tests up to term m_end.
cudaError_t launch_leja_pair(const erem_ctx* c, int m, int m_end, int qin, double cg, cudaStream_t s) {
  const PairShape sh = pair_shape(c);
  PairArgs a{};
  a.qi = (const float*)c->q[qin];
  a.qo = (float*)c->q[qin ^ 1];
  a.P = c->P;
  a.p0 = c->p0;
  a.jl = (const float*)c->jl_all;
  a.r0 = c->jl_r0;
  a.xi = c->xi_dev;
  a.dd = c->dd_dev;
  a.cg = cg;
  a.m = m;
  a.m_end = m_end;
  a.px = c->px;
  a.ny = c->ny;
  a.nz = c->nz;
  a.rows = sh.rows;
  a.zc = sh.zc;
  a.nby = sh.nby;
  a.cf_bytes = sh.cf;
  a.q0_bytes = sh.q0;
  a.q1_bytes = sh.q1;
  a.p_bytes = sh.pl;
  a.sq_scale = 1.f;
  while (a.sq_scale * (float)sh.zc > 1.f) a.sq_scale *= 0.5f;
  a.polls = c->wait_polls >= 0 ? c->wait_polls : kPairPolls;
  a.part = c->red_part;
  a.cnt = c->red_cnt;
  a.ctrl = c->ctrl;
  void (*kern)(PairArgs) = c->jl_nodiag ? (m == 1 ? k_leja_pair<true, true> : k_leja_pair<true, false>)
                                        : (m == 1 ? k_leja_pair<false, true> : k_leja_pair<false, false>);
  cudaError_t e = cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)c->smem_optin - 2048);
  if (e != cudaSuccess) return e;
  ++c->launches;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(sh.grid);
  cfg.blockDim = dim3(sh.threads);
  cfg.dynamicSmemBytes = sh.smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = (c->pdl && m > 1) ? 1 : 0;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

}  // namespace erem
