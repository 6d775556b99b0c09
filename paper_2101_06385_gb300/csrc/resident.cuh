// What the resident solves share (csrc/resident.cu on the tensor cores,
// csrc/resident_fp32.cu): the solve's state in shared memory, its control step
// with everything prepared that can be, and the meeting of a gang.
#pragma once

#include "common.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace sp2 {
namespace res {

// The coefficients of the next launch for either branch (index bit 0: sigma <
// 0) and either storage (bit 1: re-centred), and the accelerated layer's new
// bounds, prepared while the layer's products run: FP64 costs 64 cycles a step
// here and would otherwise stand in the chain of every layer.
struct Prepared {
  LayerCoef k[4];
  float ca[4], cb[4];
  double l, h;
  int sign;
  // the loop's decision on (tr Y, ||Y||_F^2): N alpha, N alpha^2, N alpha (1 -
  // alpha), 2 alpha, 1 - 2 alpha, N_occ, sigma eps, the re-centring and 4.5-rule thresholds
  int rule45;
  double na, naa, na1, ta, oa, no, se, rc, r45;
};

struct PreparedCoef {
  const Prepared* p;
  __device__ __forceinline__ void put(Ctl* c, int i, bool final_layer) const {
    set_next(c, p->k[i], p->ca[i], p->cb[i], final_layer);
  }
  __device__ __forceinline__ void branch(Ctl* c, int sigma, bool final_layer) const {
    put(c, (sigma < 0 ? 1 : 0) + (c->recentered ? 2 : 0), final_layer);
  }
  __device__ __forceinline__ int accel(Ctl*, double& l, double& h, LayerCoef&) const {
    l = p->l;
    h = p->h;
    return p->sign;
  }
  __device__ __forceinline__ void next(Ctl* c, const LayerCoef&, bool final_layer) const {
    put(c, c->recentered ? 2 : 0, final_layer);
  }
};

// A solve's control block without its history, the history's last four layers
// and the prepared step, in shared memory.
// With no state or every state occupied S goes to 0 or I and the sums of Y below any
// fixed unit: those solves keep all of them in FP64 (fp64_sums).
__device__ __forceinline__ bool fp64_sums(const Ctl* c) { return c->n_occ == 0 || c->n_occ == c->N; }

struct SolveState {
  int sg[4];
  double ie[4];
  double hot[kCtlHotBytes / 8];
  Prepared prep;
  __device__ __forceinline__ Ctl* ctl() { return reinterpret_cast<Ctl*>(hot); }
  __device__ __forceinline__ const Ctl* ctl() const { return reinterpret_cast<const Ctl*>(hot); }
  // by one warp
  __device__ __forceinline__ void load(const Ctl* gc, int lane) {
    const double* src = reinterpret_cast<const double*>(gc);
    for (int i = lane; i < (int)(kCtlHotBytes / 8); i += 32) hot[i] = __ldcg(src + i);
    __syncwarp();
    const int n = ctl()->n - lane;
    if (lane < 4 && n >= 0) {
      sg[n & 3] = gc->sigma[n];
      ie[n & 3] = gc->iderr[n];
    }
    __syncwarp();
  }
  // the final state for the host (the history was recorded layer by layer)
  __device__ __forceinline__ void store(Ctl* gc, int lane) const {
    double* dst = reinterpret_cast<double*>(gc);
    for (int i = lane; i < (int)(kCtlHotBytes / 8); i += 32) dst[i] = hot[i];
  }
};
static_assert(kCtlHotBytes % 8 == 0, "the hot part is copied in 8-byte words");

// What the next control step can be given beforehand: the candidates (lanes
// 0-3) and the constants of the loop's decision (lane 4).
__device__ __forceinline__ void prepare(SolveState& s, int lane) {
  if (lane == 4) {
    const Ctl* c = s.ctl();
    const double a = c->alpha_next, N = (double)c->N;
    const RingHistory hist{s.sg, s.ie, nullptr};
    const int n1 = c->n + 1;
    s.prep.na = N * a;
    s.prep.naa = N * a * a;
    s.prep.na1 = N * a * (1.0 - a);
    s.prep.ta = 2.0 * a;
    s.prep.oa = 1.0 - 2.0 * a;
    s.prep.no = (double)c->n_occ;
    s.prep.se = (double)hist.sigma(c->n) * c->eps;
    s.prep.rc = kRecenterFrac * N;
    s.prep.rule45 = n1 > 2 && hist.sigma(n1 - 1) != hist.sigma(n1 - 2);
    s.prep.r45 = n1 > 2 ? 4.5 * hist.iderr(n1 - 2) * hist.iderr(n1 - 2) : 0.0;
  }
  if (lane < 4) {
    const Ctl* c = s.ctl();
    const bool rec = (lane & 2) != 0;
    LayerCoef k;
    if (c->accel) {
      double l = c->acc_l, h = c->acc_h, pa, pb, pc;
      const int sg = accel_layer(l, h, pa, pb, pc);
      k = poly_coef(c->alpha_next, pa, pb, pc, rec, c->shift);
      if (lane == 0) {
        s.prep.l = l;
        s.prep.h = h;
        s.prep.sign = sg;
      }
    } else {
      k = branch_coef(c->alpha_next, (lane & 1) ? -1 : 1, rec);
    }
    s.prep.k[lane] = k;
    s.prep.ca[lane] = (float)k.ca;
    s.prep.cb[lane] = (float)k.cb;
  }
  __syncwarp();
}

// The control step of the resident solve: control_step's decision of the loop
// with everything that does not depend on the sums taken from Prepared and the
// comparisons side by side (a chain of seven FP64 operations instead of some
// twenty); the other phases as they are.
__device__ __forceinline__ void resident_step(SolveState& s, double trY, double sqY, Ctl* record) {
  Ctl* c = s.ctl();
  RingHistory hist{s.sg, s.ie, record};
  const Prepared& p = s.prep;
  if (c->phase != PHASE_LOOP || c->stop_pending || c->accel) {
    control_step(c, trY, sqY, hist, PreparedCoef{&p});
    return;
  }
  const int n1 = c->n + 1, max_iter = c->max_iter, rule45 = p.rule45;
  const double tol = c->tol, no = p.no;
  const double NX = fma(p.ta, trY, p.naa) + sqY;             // Tr[S_n^2] = ||S_n||_F^2
  const double NS2 = fma(2.0, trY, 2.0 * p.na - no);         // 2 Tr[S_n] - N_occ
  const double err = fma(p.oa, trY, p.na1) - sqY;            // N_S - N_X
  const double v = fabs(NS2 - NX) - fabs(NX - no) - p.se;
  const bool center = err <= p.rc, low = err <= tol, zero = err <= 0.0, r45 = err > p.r45;
  const int sg = (v >= 0.0) ? 1 : -1;
  const int recentered = (c->recentered || (c->shift && center)) ? 1 : 0;
  int stop = SP2_STOP_NONE;
  if (tol > 0.0 && low)
    stop = SP2_STOP_TOL;
  else if (zero)
    stop = SP2_STOP_IDERR;
  else if (rule45 && r45)
    stop = SP2_STOP_RULE45;
  else if (n1 >= max_iter)
    stop = SP2_STOP_MAXITER;
  c->trY = trY;
  c->sqY = sqY;
  c->alpha = c->alpha_next;
  c->recentered = recentered;
  c->n = n1;
  c->stop_pending = stop;
  if (stop) c->converged_by = stop;
  PreparedCoef{&p}.branch(c, sg, false);
  hist.set(n1, sg, err);
}

__device__ __forceinline__ long long warp_sum_ll(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// A layer's sums over a gang in 64-bit fixed point, exact in any order: tr Y' in
// units of 2^-50, ||Y'||_F^2 as q_hi 2^-25 + q_lo 2^-53 (q_lo of each member in
// [0, 2^28)).  A member with a sum out of range, or no number, adds SQ_BIG to
// q_hi, far above any sum in range (N 2^25): all members then meet once more, with
// their sums in FP64 (meet_fp64).
struct GangSums {
  long long t, q_hi, q_lo;
};
constexpr long long SQ_BIG = 1ll << 42;
constexpr float T_LIMIT = 2.f;            // range of a diagonal element (N of them fill 2^13 / 2^-50 = 63 bits)
constexpr long long T_OUT = 1ll << 62;    // marks a warp's trace that left it
constexpr double T_UNIT = 0x1p-50, Q_HI_UNIT = 0x1p-25, Q_LO_UNIT = 0x1p-53;

__device__ __forceinline__ void to_double(const GangSums& s, double& trY, double& sqY) {
  trY = (double)s.t * T_UNIT;
  sqY = (double)s.q_hi * Q_HI_UNIT + (double)s.q_lo * Q_LO_UNIT;
}

__device__ __forceinline__ bool out_of_range(const GangSums& s) { return s.q_hi >= SQ_BIG / 2; }

// The meeting of a gang after a layer.  Members add their sums and then their
// count into one of eight sectors of the layer's row; a member waits until the
// counts make up the gang.  Three rows serve successive layers: once a member
// has met for layer k every member is done with the row of layer k - 1, so the
// leader empties it then, for layer k + 2.  With a slot per member that everyone
// polled, 144 readers (N = 2048) of 144 slots took 4 us from the last write to
// the last read: calls of the public entry took 10 % longer at N = 2048 with single
// FP16, 5 % at N = 1000 and 30 % in FP32 at N = 512.
constexpr int MEET_GROUPS = 8, MEET_WORDS = 4;  // a sector: t, q_hi, count and q_lo, unused
static_assert(3 * (MEET_GROUPS * MEET_WORDS + 2) == kMeetRows, "three rows, of sums and of arrivals");
constexpr int MEET_SHIFT = 40;                  // the count above q_lo (304 x 2^28 < 2^37)

__device__ __forceinline__ long long* meet_row(long long* rows, int k) {
  return rows + (k % 3) * (MEET_GROUPS * MEET_WORDS);
}

__device__ __forceinline__ void red_add(long long* p, long long v) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ long long ld_word(const long long* p) {
  long long v;
  asm volatile("ld.relaxed.gpu.global.s64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Member `me` joins layer k's meeting with its sums and everything the CTA has
// written before (one thread); sums: whether there are any.
__device__ __forceinline__ void meet_join(long long* rows, int k, int me, const GangSums& s, bool sums = true) {
  long long* p = meet_row(rows, k) + (me % MEET_GROUPS) * MEET_WORDS;
  if (sums) {
    red_add(p, s.t);
    red_add(p + 1, s.q_hi);
  }
  __threadfence();
  red_add(p + 2, (1ll << MEET_SHIFT) + s.q_lo);
}

// Waits (one warp) until all cnt members have joined.  False: abort or time-out.
__device__ __forceinline__ bool meet_wait(long long* rows, int k, int cnt, int lane, const int* err,
                                          const volatile int* abort_flag, unsigned long long limit) {
  const long long* p = meet_row(rows, k) + (lane % MEET_GROUPS) * MEET_WORDS + 2;
  const uint64_t w0 = sp2::tc::globaltimer();
  for (int spin = 0;; ++spin) {
    const int have = lane < MEET_GROUPS ? (int)(ld_word(p) >> MEET_SHIFT) : 0;
    if ((int)__reduce_add_sync(0xffffffffu, have) >= cnt) break;
    if ((spin & 31) == 31) {
      const bool stop = *abort_flag || *(const volatile int*)err != 0 || sp2::tc::globaltimer() - w0 > limit;
      if (__any_sync(0xffffffffu, stop)) return false;
    }
  }
  __threadfence();  // what the gang wrote before it joined
  __syncwarp();
  return true;
}

// The sums of a meeting that is complete (one warp, in every lane).
__device__ __forceinline__ GangSums meet_sums(long long* rows, int k, int lane) {
  const long long* p = meet_row(rows, k) + (lane % MEET_GROUPS) * MEET_WORDS;
  GangSums s{ld_word(p), ld_word(p + 1), ld_word(p + 2) & ((1ll << MEET_SHIFT) - 1)};
#pragma unroll
  for (int o = MEET_GROUPS / 2; o > 0; o >>= 1) {
    s.t += __shfl_xor_sync(0xffffffffu, s.t, o);
    s.q_hi += __shfl_xor_sync(0xffffffffu, s.q_hi, o);
    s.q_lo += __shfl_xor_sync(0xffffffffu, s.q_lo, o);
  }
  return s;
}

// Arrivals: what the next layer's products need of a layer are its planes, not
// its sums.  A member's last epilogue warp counts it in one of four words as
// soon as the member's planes are stored, and each producer polls the four
// itself: a control warp that woke, added up the sums and then polled for both
// let the products start 1.5 us later.
__device__ __forceinline__ unsigned* arrival_row(long long* rows, int k) {
  return reinterpret_cast<unsigned*>(rows + 3 * MEET_GROUPS * MEET_WORDS) + 4 * (k % 3);
}
__device__ __forceinline__ void arrive(long long* rows, int k, int me) {
  __threadfence();
  asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(arrival_row(rows, k) + (me & 3)) : "memory");
}
// How many have; before anything they stored is read: a fence.
__device__ __forceinline__ int arrived(long long* rows, int k) {
  unsigned a, b, c, d;
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(a), "=r"(b), "=r"(c), "=r"(d)
               : "l"(arrival_row(rows, k))
               : "memory");
  return (int)(a + b + c + d);
}

// After the meeting of layer k, by the leader's warp.
__device__ __forceinline__ void meet_empty(long long* rows, int k, int lane) {
  __stcg(meet_row(rows, k + 2) + lane, 0ll);
  if (lane < 4) __stcg(arrival_row(rows, k + 2) + lane, 0u);
  __syncwarp();
}
static_assert(MEET_GROUPS * MEET_WORDS == 32, "one word a lane");

// The gang's sums in FP64 (one warp, in every lane): the members, who all know that a
// sum was out of range, leave theirs in slots and meet on rows of their own, j-th
// time.  The slots are read before the next layer's meeting is joined, so they are
// free when that one says the same again.  False: abort or time-out.
__device__ __forceinline__ bool meet_fp64(long long* rows, int& j, double2* slots, int me, int cnt, int lane,
                                          double& t, double& q, const int* err, const volatile int* abort_flag,
                                          unsigned long long limit) {
  if (lane == 0) {
    __stcg(slots + me, make_double2(t, q));
    meet_join(rows, j, me, GangSums{0, 0, 0}, false);
  }
  if (!meet_wait(rows, j, cnt, lane, err, abort_flag, limit)) return false;
  t = q = 0.0;
  for (int i = lane; i < cnt; i += 32) {
    const double2 v = __ldcg(slots + i);
    t += v.x;
    q += v.y;
  }
  t = warp_sum_d(t);
  q = warp_sum_d(q);
  if (me == 0) meet_empty(rows, j, lane);
  ++j;
  return true;
}

}  // namespace res
}  // namespace sp2
