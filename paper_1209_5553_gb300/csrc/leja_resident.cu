// Resident Leja interpolation: every Newton term of a substep in one
// cooperative launch, for grids whose Leja working set fits on the chip.
//
// One CTA per SM owns a block of (y, z) rows.  It keeps its part of the Leja
// copy of J and both Newton vectors in shared memory and its part of the
// running sum P in registers from the first term to the last, so a term moves
// only the block's outermost rows and one partial sum per CTA through L2.
//
// Arithmetic: every cell takes the operations of k_leja_term_lag in the same
// order, so q_m and P have its bits; only the order in which the squares
// enter ||q_m||^2 differs.
//
// Messages.  Rows and partial sums travel as 64-bit words, 32 bits of data
// and the 32-bit number of the term: a reader polls the words it needs until
// they carry the number it expects, so neither side fences or waits for a
// flag.  Two buffers per row, by the parity of the term, are enough: a CTA
// overwrites its word of term m when it publishes term m + 2, which it
// computes from its neighbours' words of term m + 1, and a neighbour wrote
// those after it had read the word of term m (the reader of a word owns the
// same x position in the neighbouring row, and its own word is read back).
//
// The stopping test of term m - 2 is taken while term m is computed: one warp
// of every CTA publishes the CTA's partial of term m - 1, sums the CTAs'
// partials of term m - 2 in CTA order (the same bits, so the same decision
// everywhere) and never waits long.  Term m adds d_{m-2} q_{m-2} to P (m = 1,
// 2: nothing; P starts as d_0 p0), so the second term after the stopping one
// completes P.  Partials have a ring of four slots: a CTA publishes term m + 4
// after its test of term m + 2, for which every CTA had published that term,
// i.e. had ended the pass that tests term m.
//
// What bounds it: on the smallest grids the chain of one term (the block
// barrier, the messages, 480 to 870 cycles one way, and about 25 FP64
// operations of the test, 64 cycles each), 1.45 us; on larger ones the FP64
// pipe (2 operations per clock and SM: one per cell and term for P in
// FP32-bulk, 8 to 10 in FP64) and the latency of shared memory with four
// warps per scheduler.  Measured per term, against one launch per term
// (k_leja_term_lag): FP32-bulk 64^2 1.45 us (4.4), 512^2 1.9 (6.4), 1024^2
// 4.2 (10.3), 64^3 3.0 (6.5), 96^3 5.5 (10.7); FP64 64^2 1.5 (4.5), 517 x 389
// 4.2 (9.1; FP64 pipe 3.0), 101 x 77 x 59 10.6 (16.5; FP64 pipe 8.7).
//
// All CTAs are co-resident (cooperative launch, at most one per SM), and
// every wait has an iteration limit, after which the CTA raises FLAG_TIMEOUT
// and leaves.
#include <algorithm>

#include "erem_internal.h"
#include "device_common.cuh"

namespace erem {
namespace {

constexpr int kResThreads = 512;             // 14 compute warps, a sum warp and a test warp
constexpr int kResWork = kResThreads - 64;
constexpr int kResWarps = kResWork / 32;
constexpr int kResMaxKV = 4;                 // vectors per thread, at most
constexpr int kResRing = 4;                  // partials kept per CTA
constexpr int kResTab = 256;                 // Leja points and differences staged per launch, at most
constexpr int kResStatic = 16 * 1024;         // static shared memory, at most
constexpr int kResPolls = 1 << 21;           // polls before a wait gives up (about a second)

struct ResArgs {
  const void* jl;      // Leja copy of J (tile-interleaved)
  const void* r0;      // diagonal-free copy: x = 0 row sums
  char* q;             // tape: q_m at q + m qstride up to q_{tape_to}, all of them written
  size_t qstride;
  int tape_to;         // (0 without a tape)
  void* qb[2];         // other q_m that are kept: qb[m & 1]
  int nxi, ndd;        // entries of the tables
  double* P;
  const double* p0;    // m = 1: P = d_0 p0
  const double* xi;
  const double* dd;
  double cg;
  int px, ny, nz;
  int hy, hz, nby;     // rows of a block in y and z; blocks in y
  int m0, m1;          // terms m0 .. m1
  int keep_q;          // q of the last term is written (for a continuation)
  unsigned base;       // number that marks term m's messages: base + m
  ulonglong2* msg;     // rows: [parity][vector][2] words pairs
  ulonglong2* part;    // partials: [CTA][kResRing]
  int polls;           // of a wait for a message before it gives up
  Ctrl* ctrl;
};

// two words, each read or written at once (64-bit accesses are)
__device__ __forceinline__ ulonglong2 ld_words(const ulonglong2* p) {
  ulonglong2 v;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_words(ulonglong2* p, unsigned a, unsigned b, unsigned tag) {
  const unsigned long long t = (unsigned long long)tag << 32;
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(t | a), "l"(t | b) : "memory");
}
__device__ __forceinline__ bool tagged(const ulonglong2& v, unsigned tag) {
  return (unsigned)(v.x >> 32) == tag && (unsigned)(v.y >> 32) == tag;
}

// A vector (16 bytes) as a message of four words, and back (bounded wait;
// false when the limit ran out).
template <typename Tq, int VEC>
__device__ __forceinline__ void put_msg(ulonglong2* p, const Tq (&r)[VEC], unsigned tag) {
  uint4 u;
  Tq* d = reinterpret_cast<Tq*>(&u);
#pragma unroll
  for (int k = 0; k < VEC; ++k) d[k] = r[k];
  st_words(p, u.x, u.y, tag);
  st_words(p + 1, u.z, u.w, tag);
}
template <typename Tq, int VEC>
__device__ __forceinline__ bool get_msg(Tq (&r)[VEC], const ulonglong2* p, unsigned tag, int polls) {
  ulonglong2 a, b;
  int k = 0;
  do {
    a = ld_words(p);
    b = ld_words(p + 1);
  } while (!(tagged(a, tag) && tagged(b, tag)) && ++k < polls);
  const uint4 u = make_uint4((unsigned)a.x, (unsigned)a.y, (unsigned)b.x, (unsigned)b.y);
  const Tq* d = reinterpret_cast<const Tq*>(&u);
#pragma unroll
  for (int j = 0; j < VEC; ++j) r[j] = d[j];
  return k < polls;
}

template <typename Tq>
__device__ __forceinline__ Tq* q_of(const ResArgs& a, int m) {
  return a.q && m <= a.tape_to ? (Tq*)(a.q + (size_t)m * a.qstride) : (Tq*)a.qb[m & 1];
}

template <typename Tq, int VEC>
__device__ __forceinline__ void ldv_cg(Tq (&r)[VEC], const Tq* p) {
  using V = typename VecT<Tq, VEC>::V;
  const V v = __ldcg(reinterpret_cast<const V*>(p));
  const Tq* s = reinterpret_cast<const Tq*>(&v);
#pragma unroll
  for (int k = 0; k < VEC; ++k) r[k] = s[k];
}

// neighbour sources of a vector (bits of its mask)
enum : int {
  RS_OWN = 1,              // the thread owns this vector
  RS_W = 2, RS_E = 4,      // x neighbours exist
  RS_SS = 8, RS_SG = 16,   // south row: in the block / in another CTA's
  RS_NS = 32, RS_NG = 64,
  RS_BS = 128, RS_BG = 256,
  RS_TS = 512, RS_TG = 1024,
  RS_PUB = 2048,           // another CTA reads this row
  RS_X0 = 4096,            // first vector of its row
  RS_REMOTE = RS_SG | RS_NG | RS_BG | RS_TG
};

template <typename Tq, int VEC, int DIM, bool ND, int KV>
__global__ void __launch_bounds__(kResThreads, 1) k_leja_res(const ResArgs a) {
  constexpr int NCF = DIM == 3 ? 7 : 5;          // coefficients D W E S N (B T)
  constexpr int NC = ND ? NCF - 1 : NCF;         // stored ones
  constexpr bool DREG = sizeof(Tq) == 8;         // FP64: the diagonal in registers, more rows fit
  constexpr int NCS = DREG ? NC - 1 : NC;        // coefficients in shared memory
  constexpr float kSq = 1.f / KV;                // of a thread's squares (add_square)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // squares per thread, by the parity of the term: a double, or the float pair
  // of the compensated FP32 sum, times kSq
  __shared__ double s_red[2][kResWork];
  // shifts c/gamma + xi_m, divided differences d_m and |delta d_m| / (scale sqrt(N))
  // from m = m0 - 2 on
  __shared__ Tq s_sh[kResTab];
  __shared__ double s_dd[kResTab], s_f[kResTab];
  __shared__ double s_e[64];                     // the last estimates, a ring
  __shared__ int s_stop[2];                      // decision of the test taken in pass parity
  __shared__ int s_abort;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const bool sum_warp = wid == kResWarps, test_warp = wid == kResWarps + 1;
  const bool work = wid < kResWarps;
  const int vrow = a.px / VEC;
  // the CTA's rows: [y0, y0 + ly) x [z0, z0 + lz)
  const int y0 = (blockIdx.x % a.nby) * a.hy, z0 = (blockIdx.x / a.nby) * a.hz;
  const int ly = min(a.hy, a.ny - y0), lz = min(a.hz, a.nz - z0);
  const int nr = ly * lz;
  const int nv = nr * vrow;
  const int nvb = a.hy * a.hz * vrow;
  const int nw = min(kResWarps, (nv + 31) / 32);   // warps that own vectors
  Tq* const coef = reinterpret_cast<Tq*>(smem_raw);            // NCS x nvb vectors
  Tq* const qs = coef + (size_t)NCS * nvb * VEC;               // 2 x nvb vectors
  // vector v of the CTA lies at vector gvec(v) of the padded layout
  auto gvec = [&](int v) {
    const int rl = v / vrow;
    return (y0 + rl % ly + a.ny * (z0 + rl / ly)) * vrow + (v - rl * vrow);
  };
  if (tid == 0) {
    s_abort = 0;
    s_stop[0] = s_stop[1] = 0;
  }
  const StopParams& sp = a.ctrl->sp;
  const int window = sp.window, m_max = sp.m_max, replay = sp.replay;
  const double pow10 = sp.pow10;
  const int t0 = max(a.m0 - 2, 0);               // first staged index
  {
    const double fs = fabs(sp.delta) / ((sp.tol_a + sp.tol_r * a.ctrl->yinf) * sqrt(sp.ncells));
    for (int k = tid; k <= a.m1 - t0; k += kResThreads) {
      s_sh[k] = (Tq)(a.cg + a.xi[min(t0 + k, a.nxi - 1)]);  // past the table: a term after the decision
      const double d = a.dd[min(t0 + k, a.ndd - 1)];
      s_dd[k] = d;
      s_f[k] = fs * fabs(d);
    }
  }
  if (test_warp && a.m0 > 1)  // continuing: the estimates of the terms before
    for (int k = max(1, a.m0 - 64) + lane; k < a.m0; k += 32) s_e[k & 63] = a.ctrl->e[k];
  // the block's coefficients, q_{m0-1} and P
  int mask[KV], vv[KV], gv[KV];
  Tq qc[KV][VEC];
  Tq cd[DREG ? KV : 1][VEC];
  double P[KV][VEC];
  if (work) {
    const Tq* jl = (const Tq*)a.jl;
    const Tq* q0 = q_of<Tq>(a, a.m0 - 1);
    for (int v = tid; v < nv; v += kResWork) {
      const int i = gvec(v) * VEC;
      const size_t off = leja_off<32 * VEC>(i, NC);
#pragma unroll
      for (int k = 0; k < NCS; ++k) {
        Tq c[VEC];
        ldv_stream<Tq, VEC>(c, jl + (k + NC - NCS) * 32 * VEC + off);
        stv<Tq, VEC>(coef + ((size_t)k * nvb + v) * VEC, c);
      }
    }
#pragma unroll
    for (int k = 0; k < KV; ++k) {
      const int t = tid + k * kResWork;
      mask[k] = 0;
      vv[k] = gv[k] = 0;
      if (t < nv) {
        // 2D: the first and last row come last, so that the rows that wait for
        // other CTAs start after the inner ones
        int v = t;
        if (DIM == 2) {
          v += vrow;
          if (v >= nv) v -= nv;
        }
        vv[k] = v;
        gv[k] = gvec(v);
        const int rl = v / vrow;
        const int jy = rl % ly, jz = rl / ly;
        const int ix = (v - rl * vrow) * VEC;
        int m = RS_OWN;
        if (ix > 0) m |= RS_W;
        else m |= RS_X0;
        if (ix + VEC < a.px) m |= RS_E;
        if (jy > 0) m |= RS_SS;
        else if (y0 > 0) m |= RS_SG;
        if (jy < ly - 1) m |= RS_NS;
        else if (y0 + ly < a.ny) m |= RS_NG;
        if (DIM == 3) {
          if (jz > 0) m |= RS_BS;
          else if (z0 > 0) m |= RS_BG;
          if (jz < lz - 1) m |= RS_TS;
          else if (z0 + lz < a.nz) m |= RS_TG;
        }
        if (m & RS_REMOTE) m |= RS_PUB;  // who is read from there reads there
        mask[k] = m;
        const size_t i = (size_t)gv[k] * VEC;
        if constexpr (DREG) ldv_stream<Tq, VEC>(cd[k], jl + leja_off<32 * VEC>((int)i, NC));
        ldv_cg<Tq, VEC>(qc[k], q0 + i);
        stv<Tq, VEC>(qs + ((size_t)((a.m0 - 1) & 1) * nvb + v) * VEC, qc[k]);
        if (a.m0 > 1) {  // continuing: q_{m0-2}
          Tq qp[VEC];
          ldv_cg<Tq, VEC>(qp, q_of<Tq>(a, a.m0 - 2) + i);
          stv<Tq, VEC>(qs + ((size_t)(a.m0 & 1) * nvb + v) * VEC, qp);
        }
        ldP<VEC>(P[k], (a.m0 == 1 ? a.p0 : a.P) + i);
        if (a.m0 == 1) {
          const double d0 = a.dd[0];
#pragma unroll
          for (int j = 0; j < VEC; ++j) P[k][j] *= d0;
        }
      }
    }
  }
  __syncthreads();

  // the CTA's sum of the squares of term mt (control warp): the threads' sums
  // in a fixed order
  auto publish_norm = [&](int mt) {
    double v;
    if constexpr (sizeof(Tq) == 4) {
      // the low parts, at most 2^-22 of their pairs, are summed in FP32 (2^-42 of
      // the sum)
      const float2* r = reinterpret_cast<const float2*>(s_red[mt & 1]) + lane;
      v = f2d_fast(r[0].x);
      float lo = r[0].y;
      for (int k = 1; k < nw; ++k) {
        v += f2d_fast(r[k * 32].x);
        lo += r[k * 32].y;
      }
      v = (v + f2d_fast(lo)) * (double)(1.f / kSq);
    } else {
      const double* r = s_red[mt & 1] + lane;
      v = r[0];
      for (int k = 1; k < nw; ++k) v += r[k * 32];
    }
    v = warp_sum(v);
    if (lane == 0)
      st_words(a.part + (size_t)blockIdx.x * kResRing + (mt & (kResRing - 1)),
               (unsigned)__double2hiint(v), (unsigned)__double2loint(v), a.base + (unsigned)mt);
  };

  int m = a.m0;
  for (;; ++m) {
    if (work) {
      const Tq sh_m = s_sh[m - 1 - t0];
      const double dprev = m > 2 ? s_dd[m - 2 - t0] : 0.0;
      const Tq* qi = qs + (size_t)((m - 1) & 1) * nvb * VEC;
      Tq* qo = qs + (size_t)(m & 1) * nvb * VEC;
      const Tq* q0g = q_of<Tq>(a, m - 1);          // m = m0
      Tq* qgo = q_of<Tq>(a, m);
      const size_t nvg = (size_t)a.ny * a.nz * vrow;
      const ulonglong2* mi = a.msg + 2 * (size_t)((m - 1) & 1) * nvg;
      ulonglong2* mo = a.msg + 2 * (size_t)(m & 1) * nvg;
      const unsigned tag = a.base + (unsigned)m;
      const bool first = m == a.m0;                // q_{m0-1} was complete before the launch
      bool ok = true;
      // a neighbour row of another CTA
      auto remote = [&](Tq (&r)[VEC], int v) {
        if (first) ldv_cg<Tq, VEC>(r, q0g + (size_t)v * VEC);
        else ok &= get_msg<Tq, VEC>(r, mi + 2 * (size_t)v, tag - 1u, a.polls);
      };
      float s_hi = 0.f, s_lo = 0.f;
      double acc = 0.0;
#pragma unroll
      for (int k = 0; k < KV; ++k) {
        const int mk = mask[k];
        if (!(mk & RS_OWN)) continue;
        const int v = vv[k], g = gv[k];
        const int o = v * VEC;
        const int orow = a.px, opl = a.px * ly;
        Tq qsv[VEC], qnv[VEC], qb[VEC], qt[VEC];
        if (mk & RS_SG) remote(qsv, g - vrow);
        else ldv<Tq, VEC>(qsv, qi + o - (mk & RS_SS ? orow : 0));
        if (mk & RS_NG) remote(qnv, g + vrow);
        else ldv<Tq, VEC>(qnv, qi + o + (mk & RS_NS ? orow : 0));
        if (DIM == 3) {
          if (mk & RS_BG) remote(qb, g - vrow * a.ny);
          else ldv<Tq, VEC>(qb, qi + o - (mk & RS_BS ? opl : 0));
          if (mk & RS_TG) remote(qt, g + vrow * a.ny);
          else ldv<Tq, VEC>(qt, qi + o + (mk & RS_TS ? opl : 0));
        }
        const Tq ql = mk & RS_W ? qi[o - 1] : Tq(0);
        const Tq qr = mk & RS_E ? qi[o + VEC] : Tq(0);
        Tq out[VEC], c[VEC];
        Tq sq = Tq(0);
        const Tq* cv = coef + o;
        const size_t cs = (size_t)nvb * VEC;
        Tq rs = Tq(0);
        if constexpr (ND) {
          if (mk & RS_X0) rs = ((const Tq*)a.r0)[g / vrow];
#pragma unroll
          for (int j = 0; j < VEC; ++j) out[j] = ((j == 0 ? rs : Tq(0)) - sh_m) * qc[k][j];
        } else {
          if constexpr (DREG) {
#pragma unroll
            for (int j = 0; j < VEC; ++j) c[j] = cd[k][j];
          } else {
            ldv<Tq, VEC>(c, cv);
            cv += cs;
          }
#pragma unroll
          for (int j = 0; j < VEC; ++j) out[j] = (c[j] - sh_m) * qc[k][j];
        }
        // couplings W E S N (B T), one at a time: sum_j J_ij (q_j - q_i) with
        // the implied diagonal, J_ij q_j otherwise
        auto add = [&](const Tq (&nb)[VEC]) {
          ldv<Tq, VEC>(c, cv);
          cv += cs;
#pragma unroll
          for (int j = 0; j < VEC; ++j) out[j] = fma(c[j], ND ? nb[j] - qc[k][j] : nb[j], out[j]);
        };
        {
          Tq nb[VEC];
#pragma unroll
          for (int j = 0; j < VEC; ++j) nb[j] = j == 0 ? ql : qc[k][j - 1];
          add(nb);
#pragma unroll
          for (int j = 0; j < VEC; ++j) nb[j] = j == VEC - 1 ? qr : qc[k][j + 1];
          add(nb);
        }
        add(qsv);
        add(qnv);
        if (DIM == 3) {
          add(qb);
          add(qt);
        }
        if ((mk & RS_PUB) && m < a.m1) put_msg<Tq, VEC>(mo + 2 * (size_t)g, out, tag);
        if (m <= a.tape_to) stv<Tq, VEC>(qgo + (size_t)g * VEC, out);
        Tq qp[VEC];  // q_{m-2}, in the buffer q_m takes
        ldv<Tq, VEC>(qp, qo + o);
        stv<Tq, VEC>(qo + o, out);
        if (m > 2) {
#pragma unroll
          for (int j = 0; j < VEC; ++j) P[k][j] = fma(dprev, to_f64_fast(qp[j]), P[k][j]);
        }
#pragma unroll
        for (int j = 0; j < VEC; ++j) {
          if constexpr (sizeof(Tq) == 4) sq = fmaf(out[j], out[j], sq);
          else acc = fma(out[j], out[j], acc);
          qc[k][j] = out[j];
        }
        if constexpr (sizeof(Tq) == 4) add_square(sq, kSq, s_hi, s_lo);
      }
      if constexpr (sizeof(Tq) == 4) reinterpret_cast<float2*>(s_red[m & 1])[tid] = make_float2(s_hi, s_lo);
      else s_red[m & 1][tid] = acc;
      if (!ok) {
        s_abort = 1;
        atomicOr(&a.ctrl->flags, FLAG_TIMEOUT);
      }
    } else if (sum_warp) {
      if (m > a.m0) publish_norm(m - 1);
    } else {
      const int mt = m - 2;                        // the stopping test of term m - 2
      if (mt >= 1) {
        // the partials of term mt: messages of this launch, or the ring's
        // values where the launch before ended with that term.  They were
        // sent a term ago: all are asked for at once, and again where one is late
        constexpr int NB = kResSms / 32;
        const unsigned tag = a.base + (unsigned)mt;
        const ulonglong2* pp = a.part + (mt & (kResRing - 1));
        ulonglong2 w[NB];
#pragma unroll
        for (int j = 0; j < NB; ++j)
          if (lane + 32 * j < (int)gridDim.x) w[j] = ld_words(pp + (size_t)(lane + 32 * j) * kResRing);
        const int lo = max(1, mt - window + 1);
        double part = 0.0;
        for (int k = lo; k < mt; ++k) part += s_e[k & 63];
        double S = 0.0;
        bool ok = true;
#pragma unroll
        for (int j = 0; j < NB; ++j)
          if (lane + 32 * j < (int)gridDim.x) {
            if (mt >= a.m0)
              for (int k = 0; !tagged(w[j], tag); w[j] = ld_words(pp + (size_t)(lane + 32 * j) * kResRing))
                if (++k >= a.polls) {
                  ok = false;
                  break;
                }
            S += __hiloint2double((int)(unsigned)w[j].x, (int)(unsigned)w[j].y);
          }
        S = warp_sum(S);
        if (!__all_sync(0xffffffffu, ok) && lane == 0) {
          s_abort = 1;
          atomicOr(&a.ctrl->flags, FLAG_TIMEOUT);
        }
        if (lane == 0) {
          const double e = s_f[mt - t0] * sqrt_newton(S);
          s_e[mt & 63] = e;
          int stop = 0, degree = 0, fail = 0, nonfin = 0;
          // 10^p times the mean of the window against 1
          if (!bits_finite(abs_bits(e))) {
            nonfin = 1;
            stop = 1;
          } else if (!replay) {
            if (pow10 * (part + e) < (double)(mt - lo + 1)) {
              stop = 1;
              degree = mt;
            } else if (mt >= m_max) {
              stop = 1;
              fail = 1;
            }
          }
          s_stop[m & 1] = stop;
          if (blockIdx.x == 0) {
            Ctrl* c = a.ctrl;
            c->e[mt] = e;
            c->m_last = mt;
            if (nonfin) {
              c->nonfinite = 1;
            } else {
              c->degree = degree;
              c->fail = fail;
              if (stop || m == a.m1) c->err = (part + e) / (double)(mt - lo + 1);
            }
            if (stop) {
              c->done = 1;
              c->stop_m = mt;
            }
          }
        }
      }
    }
    __syncthreads();
    if (s_abort || s_stop[m & 1] || m == a.m1) break;
  }
  // P, and for a continuation the last two vectors and the last partial
  if (work) {
    Tq* qg = q_of<Tq>(a, m);
    Tq* qg1 = q_of<Tq>(a, m - 1);
#pragma unroll
    for (int k = 0; k < KV; ++k)
      if (mask[k] & RS_OWN) {
        const size_t i = (size_t)gv[k] * VEC;
        stP<VEC>(a.P + i, P[k]);
        if (a.keep_q) {
          stv<Tq, VEC>(qg + i, qc[k]);
          Tq q1[VEC];
          ldv<Tq, VEC>(q1, qs + ((size_t)((m - 1) & 1) * nvb + vv[k]) * VEC);
          stv<Tq, VEC>(qg1 + i, q1);
        }
      }
  } else if (sum_warp) {
    publish_norm(m);
  }
}

template <typename Tq, int VEC, int DIM, bool ND>
const void* res_kernel(int kv) {
  if (kv <= 1) return (const void*)k_leja_res<Tq, VEC, DIM, ND, 1>;
  if (kv <= 2) return (const void*)k_leja_res<Tq, VEC, DIM, ND, 2>;
  return (const void*)k_leja_res<Tq, VEC, DIM, ND, kResMaxKV>;
}

const void* res_kernel_of(const erem_ctx* c, int kv) {
  if (c->prec == EREM_FP32_BULK) {
    if (c->dim == 3)
      return c->jl_nodiag ? res_kernel<float, 4, 3, true>(kv) : res_kernel<float, 4, 3, false>(kv);
    return c->jl_nodiag ? res_kernel<float, 4, 2, true>(kv) : res_kernel<float, 4, 2, false>(kv);
  }
  return c->dim == 3 ? res_kernel<double, 2, 3, false>(kv) : res_kernel<double, 2, 2, false>(kv);
}

}  // namespace

namespace {

int res_vec(const erem_ctx* c) { return c->prec == EREM_FP32_BULK ? 4 : 2; }

// Shared memory of a block of `rows` rows: the stored coefficients (FP64:
// without the diagonal) and two Newton vectors.
size_t res_smem(const erem_ctx* c, int rows) {
  const int nc = (c->dim == 3 ? 7 : 5) - (c->jl_nodiag || c->prec == EREM_FP64 ? 1 : 0);
  const size_t esz = c->prec == EREM_FP32_BULK ? sizeof(float) : sizeof(double);
  return (size_t)(nc + 2) * rows * c->px * esz;
}

// The rows of a block, hy x hz: at most one block per SM, the fewest rows in
// the largest block (the slowest CTA decides a term), then the fewest rows
// that other blocks read.
void res_blocks(const erem_ctx* c, int* hy, int* hz) {
  const int sms = c->res_sms;
  const int vrow = c->px / res_vec(c);
  const long long least = std::max(1, kResMinVecs / vrow);
  long long best = -1;
  *hy = *hz = 0;
  for (int z = 1; z <= c->nz; ++z) {
    const int bz = (c->nz + z - 1) / z;
    if (bz > sms) continue;
    const int by = sms / bz;
    const int y = (c->ny + by - 1) / by;
    const long long cost = std::max((long long)y * z, least) * 4096 + y + z;
    if (best < 0 || cost < best) {
      best = cost;
      *hy = y;
      *hz = z;
    }
  }
  // a short row: several to a block, so that its warps are not nearly empty
  if (c->dim == 2) *hy = (int)std::max((long long)*hy, std::min((long long)c->ny, least));
}

}  // namespace

size_t res_msg_bytes(const erem_ctx* c) {
  const size_t esz = c->prec == EREM_FP32_BULK ? sizeof(float) : sizeof(double);
  return 4 * esz * (size_t)c->Np;   // two buffers of twice the data
}
size_t res_part_bytes(const erem_ctx* c) { return sizeof(ulonglong2) * kResRing * (size_t)c->res_sms; }

// Whether the grid takes the resident form: its Leja working set fits on the
// chip and, in FP64, its rows spread well enough.  A block of whole rows is
// the unit of work, and an FP64 term costs about 1.7 us + 4.5 ns per vector
// of the largest block (the FP64 pipe of one SM) against 4.2 us + 0.04 ns per
// vector of the grid for a launch per term, which spreads single vectors: a
// few long rows stay with the launches (2048 x 20: 6.4 against 5.1 us per
// term; 2048 x 64: 6.4 against 7.2; 517 x 389: 4.2 against 9.1).  In
// FP32-bulk the resident form was faster at every shape that fits (3500 x 20:
// 2.9 against 4.3 us).
bool leja_res_fits(erem_ctx* c) {
  if (!c->res_ok) return false;
  if (c->res_hy == 0) res_blocks(c, &c->res_hy, &c->res_hz);
  const int rows = c->res_hy * c->res_hz;
  const long long nv = (long long)rows * (c->px / res_vec(c));
  if (rows <= 0 || nv > (long long)kResMaxKV * kResWork ||
      res_smem(c, rows) > (size_t)(c->smem_optin - kResStatic))
    return false;
  return c->prec == EREM_FP32_BULK || nv <= 384 + c->Np / res_vec(c) / 110;
}

// Terms m0 .. m1 in one launch (see k_leja_res).  With a tape q_m is read from
// and written to its slot up to tape_to (the slots of an interpolation end with
// its table or forced degree); past it, and without a tape, the ping-pong buffer
// of m's parity holds q_{m0-1} and q_{m0-2} and takes the last two vectors when
// keep_q is set.  dd_dev holds ndd entries.  The device refuses a launch whose
// CTAs cannot all run at once (cudaErrorCooperativeLaunchTooLarge).
cudaError_t launch_leja_res(erem_ctx* c, int m0, int m1, int ndd, int keep_q, int tape_to, char* tape,
                            size_t qbytes, double cg, cudaStream_t s) {
  const int rows = c->res_hy * c->res_hz;
  const int kv = (rows * (c->px / res_vec(c)) + kResWork - 1) / kResWork;
  const int nby = (c->ny + c->res_hy - 1) / c->res_hy, nbz = (c->nz + c->res_hz - 1) / c->res_hz;
  ResArgs a{};
  a.jl = c->jl_all;
  a.r0 = c->jl_r0;
  a.q = tape;
  a.qstride = qbytes;
  a.qb[0] = c->q[0];
  a.qb[1] = c->q[1];
  a.tape_to = tape_to;
  a.nxi = c->xi_cap + 1;
  a.ndd = ndd;
  a.P = c->P;
  a.p0 = c->p0;
  a.xi = c->xi_dev;
  a.dd = c->dd_dev;
  a.cg = cg;
  a.px = c->px;
  a.ny = c->ny;
  a.nz = c->nz;
  a.hy = c->res_hy;
  a.hz = c->res_hz;
  a.nby = nby;
  a.m0 = m0;
  a.m1 = m1;
  a.keep_q = keep_q;
  // no message of an earlier launch carries this one's numbers
  if (res_renumbers(c->res_base, m0)) {
    cudaError_t e = cudaMemsetAsync(c->res_msg, 0, res_msg_bytes(c), s);
    if (e == cudaSuccess)
      e = cudaMemsetAsync(c->res_part, 0, res_part_bytes(c), s);
    if (e != cudaSuccess) return e;
    c->res_base = 0;
  }
  a.base = c->res_base;
  c->res_base += (unsigned)m1 + 1u;
  a.msg = (ulonglong2*)c->res_msg;
  a.part = (ulonglong2*)c->res_part;
  a.polls = c->wait_polls >= 0 ? c->wait_polls : kResPolls;
  a.ctrl = c->ctrl;
  const void* kern = res_kernel_of(c, kv);
  const size_t smem = res_smem(c, rows);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       c->smem_optin - kResStatic);
  if (e != cudaSuccess) return e;
  ++c->launches;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel(kern, dim3(nby * nbz), dim3(kResThreads), args, smem, s);
}

}  // namespace erem
