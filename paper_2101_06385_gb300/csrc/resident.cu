// Resident SP2 solve (sm_103a): every layer of many instances in one launch.
//
// A CTA owns one or two 128 x 128 tiles of the upper super tiles and keeps
// each for all layers of its solve: the FP32 iterate of the tile stays in
// tensor memory next to its accumulator, and only the FP16 operand planes go
// through L2 (with instances of one tile not even those).  The CTAs of one
// instance (its gang) meet after every layer: the next products start when all
// its planes are stored, and each CTA runs the control step of Alg. 1 on the same
// sums meanwhile, so a solve costs no launch per layer and stops at its last one.
//
// What bounds it: for small N the chain of one layer (operand loads, K / 64
// stages of twelve dependent MMAs at 0.47 us each, epilogue, gang meeting);
// for many instances the tensor cores at the 128 x 128 tile's rate (1.8
// PFLOP/s of products with every SM loading, against 2.1 of the CTA pairs'
// 256 x 256 tiles, which leave most of the chip idle at these sizes).
//
// Two slots per CTA hold tiles of the same or of different instances, each
// slot a list that the host planned.  While one slot waits for its gang or
// runs its epilogue the other's MMAs run; the producer takes whichever slot is
// ready.  Every list is in one order of the instances, so the earliest
// unfinished gang has all its tiles at the front of their lists: with at most
// one tile of an instance per slot and all CTAs resident (cooperative launch)
// no wait is circular.  Every wait is bounded all the same.
//
// Tile accumulation order, epilogue arithmetic and the super-tile storage of
// the planes (256 x 256 upper super tiles, K blocks left of the diagonal read
// transposed) are those of the other tensor-core kernels, so D has the same
// bits.
//
// CTA = 20 warps: 0 TMA producer, 1 MMA issuer (and TMEM), 2-17 epilogue
// (one 32 x 32 chunk each), 18 and 19 control of the two slots.
#include <cuda.h>
#include <cuda_fp16.h>

#include "common.cuh"
#include "epilogue.cuh"
#include "kernels.h"
#include "resident.cuh"
#include "resident_tc.cuh"
#include "tc_ptx.cuh"

namespace sp2 {
namespace res {

using namespace sp2::tc;

struct Slot {
  int b, I, J, N;        // instance, tile row and column (128 units), size
  int par, first;        // parity of the operand planes; first layer
  int closed;            // no more work in this slot
  int layer;             // its number
  int cnt, me;           // the gang, and this tile's place in it
  int direct;            // the producer itself watches the gang's arrivals
  int stored;            // epilogue warps that have stored their part of the planes
  float t_limit, sq_limit;  // ranges of a diagonal element and a lane's squares in fixed point; 0: all
  unsigned rn_limit;        //   sums in FP64 (fp64_sums); of a row norm's segment (its bits)
  long long* rows;       // the gang's meeting rows
  SolveState st;
};

struct Shared {
  uint64_t full[STAGES_PLAIN], empty[STAGES_PLAIN];
  uint64_t ready[2];     // control warp -> producer: an instance's first operands, the next ones unless the
                         //   producer watches the gang's arrivals, or the slot's end
  uint64_t coef[2];      // control warp -> epilogue: the layer's coefficients are set
  uint64_t acc_full[2];  // MMA issuer -> epilogue
  uint64_t epi_done[2];  // epilogue warps -> control warp
  uint64_t wq_full[WQ];  // producer -> MMA issuer and epilogue: next slot
  uint64_t drain, never;
  int wq[WQ];
  uint32_t tmem;
  int abort;
  long long red_t[2][EPI_WARPS], red_q[2][EPI_WARPS];  // a layer's sums per warp (fixed point)
  double2 red_d[2][EPI_WARPS];                         // the same in FP64, where a sum is marked out of range
  double red_e[2][EPI_WARPS];                          // Tr[D H] (last layer)
  Slot slot[2];
};

// A layer's sums tr Y' and ||Y'||_F^2 in 64-bit fixed point, exact in any
// order: FP64 adds (64 cycles each, 19 of them a warp on the SM's one pipe)
// would cost a layer's epilogue a microsecond, integer ones half of one
// shuffle.  With a shift alpha in [0, 1] Y' = S' - alpha I has spectral norm <=
// 1, so a lane's FP32 sum of 32 squares is at most 4, a tile's at most 128 and a
// diagonal element at most 1: units of 2^-53 and 2^-50 (trace) lose less than the
// FP64 sums did.  A spectrum of H that lies on one side of zero starts with alpha
// outside [0, 1] and squares it until a branch brings it back, so any magnitude
// can occur: a warp whose sum leaves the range, or is not a number, marks it and
// hands it over in FP64 (so do all of a solve where fp64_sums says so).
constexpr long long SQ_LIMIT = (1ll << 58) + (1ll << 50);  // a 32 x 32 block's 32, with rounding
constexpr float SQ_LANE = 4.f;                             // a lane's sum of 32 squares: elements below T_LIMIT
constexpr unsigned RN_LIMIT = 0x40800000u;                 // a row norm's segment: 4.0
constexpr long long SQ_OUT = -1;                           // marks a warp's sum that is in Shared::red_d (as T_OUT)

__device__ __forceinline__ long long fix_sq(float v) {
  // v = hi 2^-25 + lo 2^-53, both steps exact or rounded once
  const int hi = __float2int_rz(v * 0x1p25f);
  const int lo = __float2int_rn(fmaf(-(float)hi, 0x1p-25f, v) * 0x1p53f);
  return ((long long)hi << 28) + (long long)lo;
}

// Row norm (Y^2)_rr of the layer's input: FP64 ones of the input layer, or the
// sum of the previous layer's segment sums (at most 1 together with a shift in
// [0, 1]; 2^-53 of fixed point is what an FP64 sum near 1 resolves), in FP64 where
// one is above 4 or no number.  The segments were written by other SMs during this
// launch: read through L2.
__device__ __forceinline__ double row_norm(const ResArgs& a, const Slot& s, int r) {
  if (s.first) return a.rn[(long long)s.b * a.ld_rn + r];
  const float* p = a.rnp[s.par ^ 1] + (long long)s.b * a.slot_rnp + r;
  const int nseg = (s.N + 31) >> 5;
  long long acc = 0;
  unsigned top = 0;  // the largest as its bits (no sum of squares is negative; NaN is above every number)
  int g = 0;
  for (; g + 16 <= nseg; g += 16) {
    float v[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) v[u] = __ldcg(p + (long long)(g + u) * a.ld_rnp);
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      acc += fix_sq(v[u]);
      top = max(top, __float_as_uint(v[u]));
    }
  }
  float v[16];
#pragma unroll
  for (int u = 0; u < 16; ++u) v[u] = g + u < nseg ? __ldcg(p + (long long)(g + u) * a.ld_rnp) : 0.f;
#pragma unroll
  for (int u = 0; u < 16; ++u) {
    acc += fix_sq(v[u]);
    top = max(top, __float_as_uint(v[u]));
  }
  if (top > s.rn_limit) {
    auto every8 = [&](int first) {  // epi::row_norm's order
      double sum = 0.0;
#pragma unroll 1
      for (int k = first; k < nseg; k += 8) sum += (double)__ldcg(p + (long long)k * a.ld_rnp);
      return sum;
    };
    double sum = 0.0;
#pragma unroll 1
    for (int h = 0; h < 8; h += 4) sum += (every8(h) + every8(h + 1)) + (every8(h + 2) + every8(h + 3));
    return sum;
  }
  return (double)acc * Q_LO_UNIT;
}

// The warp has stored its part of the layer's planes and row norms and read its
// accumulator; the last of the tile counts it in its gang (Slot::direct: 5 % less
// at N = 1000, 3 % at N = 2048 with single FP16).  With two slots the next products
// are let go by the control warp: a producer that polls for one gang sees the other
// slot late (512 matrices 1 % slower).  A lone tile (LOCAL) starts its own.
template <bool LOCAL>
__device__ __forceinline__ void stored(Shared& sh, int c, int lane) {
  Slot& s = sh.slot[c];
  if (!s.direct) return;
  if (LOCAL) fence_proxy_async_shared();  // the MMAs read the planes next
  tc_fence_before();
  __syncwarp();
  if (lane == 0) {
    __threadfence_block();
    if (atomicAdd(&s.stored, 1) == EPI_WARPS - 1) {
      __threadfence_block();
      s.stored = 0;
      s.par ^= 1;
      s.first = 0;
      const int k = s.layer;
      s.layer = k + 1;
      if (LOCAL)
        mbar_arrive(&sh.ready[c]);
      else
        arrive(s.rows, k, s.me);
    }
  }
}

// One layer of the warp's 32 x 32 chunk of a slot's tile (the lane layouts and
// arithmetic of epi::tile).  False: the accumulator wait failed.
template <bool SPLIT, bool LOCAL>
__device__ __forceinline__ bool epilogue(const ResArgs& a, Shared& sh, int c, uint8_t* area, uint32_t acc_phase,
                                         uint32_t tmem_base, int ew, int q, int lane, float* trb, unsigned long long lim) {
  const Slot& s = sh.slot[c];
  const Ctl* ct = s.st.ctl();
  const int b = s.b, N = s.N, first = s.first;
  const int hc = ew >> 2;
  const int R0 = s.I * TB + q * 32;
  const int nrows = min(32, N - R0);
  const int c0 = s.J * TB + hc * 32;
  const bool mirror = (s.I >> 1) != (s.J >> 1);
  const float unscale = SPLIT ? a.lo_unscale * a.lo_unscale : 1.f;
  const float lo_scale = a.lo_scale;
  const int r4 = lane >> 3, c4 = lane & 7;
  const int ce = c0 + 4 * c4;
  const int rdiag = R0 + 4 * c4 + r4;
  // the one diagonal element a lane holds (chunk c0 == R0 of a diagonal tile,
  // a warp-uniform condition): row = column = rdiag, register 4 c4 + r4
  const bool dchunk = !mirror && c0 == R0;
  const bool dlane = dchunk && rdiag < N;
  const int id = 4 * c4 + r4;
  const bool live = nrows > 0 && c0 < ((N + 63) & ~63);
  const uint32_t tacc = tmem_base + c * SLOT_COLS + ((uint32_t)(q * 32) << 16) + hc * 32;
  const uint32_t ty = tacc + Y_COL;
  const float* H = a.H[b];

  // old values and the diagonal's row norm before the accumulator wait
  float y[32];
  double rn_l = 0.0;
  if (live) {
    if (dlane) rn_l = row_norm(a, s, rdiag);
    if (first) {
      const InputScale in = input_scale(ct->e_min, ct->e_max, a.shift);
      const bool vec_h = (N & 3) == 0 && (reinterpret_cast<uintptr_t>(H) & 15) == 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const bool rok = 4 * i + r4 < nrows;
        const float4 o = rok ? epi::ld4(H + (long long)(R0 + 4 * i + r4) * N + ce, ce, N, vec_h)
                             : make_float4(0.f, 0.f, 0.f, 0.f);
        y[4 * i] = o.x;
        y[4 * i + 1] = o.y;
        y[4 * i + 2] = o.z;
        y[4 * i + 3] = o.w;
      }
      float hd = 0.f;
      if (dchunk) {
#pragma unroll
        for (int k = 0; k < 32; ++k)
          if (k == id) hd = y[k];
      }
#pragma unroll
      for (int k = 0; k < 32; ++k) y[k] = input_offdiag(y[k], in);
      if (dchunk) {
        const float yd0 = input_diag(hd, in);
#pragma unroll
        for (int k = 0; k < 32; ++k)
          if (k == id) y[k] = yd0;
      }
    } else {
      uint32_t w[32];
      __syncwarp();
      tmem_ld32(ty, w);
      tmem_ld_wait();
#pragma unroll
      for (int k = 0; k < 32; ++k) y[k] = __uint_as_float(w[k]);
    }
  }
  // the previous layer's control step runs under this layer's products
  if (!__all_sync(0xffffffffu, mbar_wait(&sh.coef[c], acc_phase, &sh.abort, lim))) return false;
  const LayerParams p = ct->next;
  const bool outD = (p.out_mode == OUT_D);
  // the diagonal needs no product: its square comes from the row norms
  long long tr = 0, sq = 0;
  double yd = 0.0;
  float ydf = 0.f, ydo = 0.f;
  if (dchunk) {
    float yold_d = 0.f;
#pragma unroll
    for (int k = 0; k < 32; ++k)
      if (k == id) yold_d = y[k];
    if (dlane) {
      yd = p.ca_d * (double)yold_d + p.cb_d * rn_l + p.cc_d;
      tr = __double2ll_rn(yd * 0x1p50);
      ydf = (float)yd;
      ydo = outD ? (float)(yd + p.alpha_out) : ydf;
    }
    // (a lone tile's chain runs through here: it looks at the range with its squares)
    if (!LOCAL && __any_sync(0xffffffffu, dlane && !(fabsf(ydf) < s.t_limit))) {
      const double T = warp_sum_d(yd);
      if (lane == 0) sh.red_d[c][ew].x = T;
      tr = T_OUT;
    } else {
      tr = warp_sum_ll(tr);
    }
  }
  if (!__all_sync(0xffffffffu, mbar_wait(&sh.acc_full[c], acc_phase, &sh.abort, lim))) return false;
  tc_fence_after();

  double dtr = 0.0;
  // the warp's sums to the control warp
  auto report = [&]() {
    __syncwarp();
    if (lane == 0) {
      sh.red_t[c][ew] = tr;
      sh.red_q[c][ew] = sq;
      if (outD) sh.red_e[c][ew] = dtr;
      mbar_arrive(&sh.epi_done[c]);
    }
  };
  if (live) {
    const bool full = nrows == 32 && c0 + 32 <= N;
    {
      uint32_t v[32];
      __syncwarp();
      tmem_ld32(tacc, v);
      tmem_ld_wait();
      const float cbu = p.cb * unscale;
      turn(trb, v, lane, [&](int i, const float4& pv) {
        y[4 * i] = fmaf(p.ca, y[4 * i], cbu * pv.x);
        y[4 * i + 1] = fmaf(p.ca, y[4 * i + 1], cbu * pv.y);
        y[4 * i + 2] = fmaf(p.ca, y[4 * i + 2], cbu * pv.z);
        y[4 * i + 3] = fmaf(p.ca, y[4 * i + 3], cbu * pv.w);
      });
    }
    if (!full) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (!(4 * i + r4 < nrows && ce + e < N)) y[4 * i + e] = 0.f;
    }
    if (dchunk) {
#pragma unroll
      for (int k = 0; k < 32; ++k)
        if (dlane && k == id) y[k] = ydf;
    }
    // sums of squares: per row over the 32 columns, per column over the 32
    // rows (the mirror's rows), and the lane's share of ||Y'||_F^2
    float rs[8], cs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      rs[i] = 0.f;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        rs[i] = fmaf(y[4 * i + e], y[4 * i + e], rs[i]);
        cs[e] = fmaf(y[4 * i + e], y[4 * i + e], cs[e]);
      }
    }
    const float sql = ((rs[0] + rs[1]) + (rs[2] + rs[3])) + ((rs[4] + rs[5]) + (rs[6] + rs[7]));
    const bool wild = __any_sync(0xffffffffu, !(sql < s.sq_limit));
    auto sum_squares = [&]() {
      sq = warp_sum_ll(fix_sq(sql));
      if (wild || sq > SQ_LIMIT) {
        const double Q = warp_sum_d((double)sql);
        if (lane == 0) sh.red_d[c][ew].y = Q;
        sq = SQ_OUT;
        if (LOCAL) {
          const double T = warp_sum_d(yd);
          if (lane == 0) sh.red_d[c][ew].x = T;
          tr = T_OUT;
        }
      }
    };
    if (!outD) {
      if (LOCAL) {
        // a lone tile's control step bounds its layer: the sums first, then the
        // planes, which go no further than the operand tiles
        sum_squares();
        report();
        store_planes_shared<SPLIT>(y, area + (hc >> 1) * (SPLIT ? 2 : 1) * HALF_BYTES, q * 32 + r4,
                                   (hc & 1) * 32 + 4 * c4, nrows - r4, lo_scale);
      } else {
        // operand planes of Y' (Eq. 12) first: they are what the gang waits for
        const long long po = (long long)b * a.slot_h + (long long)(R0 + r4) * a.ld_h + ce;
        store_planes<SPLIT>(y, a.p0[s.par ^ 1] + po, SPLIT ? a.p1[s.par ^ 1] + po : nullptr, a.ld_h, nrows - r4,
                            lo_scale);
      }
      // row norms of the next layer
      float* rnp = a.rnp[s.par] + (long long)b * a.slot_rnp;
      const float rsum = epi::lane_sums<8, 0>(rs);
      if (rdiag < N && c0 < N) rnp[(long long)(c0 >> 5) * a.ld_rnp + rdiag] = rsum;
      if (mirror) {
        const float csum = epi::lane_sums<4, 3>(cs);
        const int cm = c0 + 4 * c4 + r4;
        if (cm < N) rnp[(long long)(R0 >> 5) * a.ld_rnp + cm] = csum;
      }
      stored<LOCAL>(sh, c, lane);
      uint32_t w[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) w[k] = __float_as_uint(y[k]);
      __syncwarp();
      tmem_st32(ty, w);
    }
    if (outD || !LOCAL) sum_squares();
    if (!outD && !s.direct) fence_proxy_async();  // the planes are read by the TMA unit next
    if (outD) {
      if (dchunk) {
#pragma unroll
        for (int k = 0; k < 32; ++k)
          if (dlane && k == id) y[k] = ydo;
      }
      float* D = a.D[b];
      const bool vec_n =
          (N & 3) == 0 && ((reinterpret_cast<uintptr_t>(D) | reinterpret_cast<uintptr_t>(H)) & 15) == 0;
      float eo = 0.f;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (4 * i + r4 < nrows) {
          const long long o = (long long)(R0 + 4 * i + r4) * N + ce;
          const float4 hv = epi::ld4(H + o, ce, N, vec_n);
          epi::st4(D + o, make_float4(y[4 * i], y[4 * i + 1], y[4 * i + 2], y[4 * i + 3]), ce, N, vec_n);
          eo = fmaf(y[4 * i], hv.x, eo);
          eo = fmaf(y[4 * i + 1], hv.y, eo);
          eo = fmaf(y[4 * i + 2], hv.z, eo);
          eo = fmaf(y[4 * i + 3], hv.w, eo);
        }
      }
      dtr = warp_sum_d((double)eo);
      if (mirror) {
        dtr *= 2.0;
        // back to lane = row, sixteen rows at a time: the mirror column is
        // contiguous across lanes
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
          for (int i = 4 * h; i < 4 * h + 4; ++i)
            *epi::tr_at(trb, 4 * (i - 4 * h) + r4, c4) = make_float4(y[4 * i], y[4 * i + 1], y[4 * i + 2], y[4 * i + 3]);
          __syncwarp();
          if ((lane >> 4) == h && lane < nrows) {
#pragma unroll
            for (int m = 0; m < 8; ++m) {
              const float4 o = *epi::tr_at(trb, lane & 15, m);
              const float ov[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (c0 + 4 * m + e < N) D[(long long)(c0 + 4 * m + e) * N + R0 + lane] = ov[e];
            }
          }
          __syncwarp();
        }
      }
    }
  } else if (!outD) {
    if (LOCAL) report();
    stored<LOCAL>(sh, c, lane);
  }
  tmem_st_wait();
  tc_fence_before();
  if (outD || !LOCAL) report();
  return true;
}

// Control of one slot: takes the tiles of its list and drives their layers.
template <bool LOCAL>
__device__ __forceinline__ void control(const ResArgs& a, Shared& sh, int c, int lane, unsigned long long idle) {
  Slot& s = sh.slot[c];
  Ctl* hot = s.st.ctl();
  const int sl = c * (int)gridDim.x + (int)blockIdx.x;
  uint32_t done_phase = 0;
  bool ok = true;
  for (int li = a.list_off[sl]; ok && li < a.list_off[sl + 1]; ++li) {
    const int t = a.list[li];
    int b, I, J, h;
    unpack_tile(a.tiles[t], b, I, J, h);
    const Ctl* gc = a.ctl + b;
    s.st.load(gc, lane);  // as the input layer's control step left it
    const int cnt = a.tile_cnt[b], off = a.tile_off[b];
    const bool leader = t == off;
    long long* rows = a.sums + (long long)b * 2 * kMeetRows;
    int wide = 0;  // layers whose sums met in FP64
    const bool twice = (I >> 1) != (J >> 1);  // the mirror's squares
    bool act = hot->next.active != 0;
    unsigned* st = a.stamps + (long long)b * kResStamps;
    uint64_t t0 = 0;
    if (act && leader && lane == 0) t0 = globaltimer();
    if (lane == 0) {
      s.b = b;
      s.I = I;
      s.J = J;
      s.N = hot->N;
      s.par = 0;
      s.first = 1;
      s.closed = 0;
      s.layer = 0;
      s.cnt = cnt;
      s.direct = LOCAL || (cnt > 1 && !a.two_slots);
      s.me = t - off;
      s.stored = 0;
      const bool fp64 = fp64_sums(hot);
      s.t_limit = fp64 ? 0.f : T_LIMIT;
      s.sq_limit = fp64 ? 0.f : SQ_LANE;
      s.rn_limit = fp64 ? 0u : RN_LIMIT;
      s.rows = rows;
      if (act) {
        mbar_arrive(&sh.ready[c]);
        mbar_arrive(&sh.coef[c]);
      }
    }
    __syncwarp();
    for (int k = 0; act; ++k) {
      prepare(s.st, lane);
      if (!__all_sync(0xffffffffu, mbar_wait(&sh.epi_done[c], done_phase, &sh.abort, idle))) {
        ok = false;
        break;
      }
      done_phase ^= 1u;
      // after the layer that writes D the solve is over; any other has a next one
      const bool outD = hot->next.out_mode == OUT_D;
      const bool direct = LOCAL || (cnt > 1 && !a.two_slots);
      if (lane == 0 && !outD && !direct) {
        s.par ^= 1;
        s.first = 0;
        if (cnt == 1) mbar_arrive(&sh.ready[c]);
      }
      // the tile's sums; with one out of range all of them in FP64
      long long rq = lane < EPI_WARPS ? sh.red_q[c][lane] : 0, rt = lane < EPI_WARPS ? sh.red_t[c][lane] : 0;
      const int mul = !LOCAL && twice ? 1 : 0;
      double trY = 0.0, sqY = 0.0;
      const bool out = __any_sync(0xffffffffu, rq == SQ_OUT || rt == T_OUT);
      GangSums G{0, SQ_BIG, 0};
      if (!out) {
        rq = warp_sum_ll(rq);  // at most 2^62 + 2^54: the doubling does not fit into the word
        G = GangSums{warp_sum_ll(rt), rq >> (28 - mul), (rq << mul) & ((1ll << 28) - 1)};
      } else {
        const double2 d = lane < EPI_WARPS ? sh.red_d[c][lane] : make_double2(0.0, 0.0);
        trY = warp_sum_d(rt == T_OUT ? d.x : (double)rt * T_UNIT);
        sqY = warp_sum_d(rq == SQ_OUT ? d.y : (double)rq * Q_LO_UNIT) * (twice ? 2.0 : 1.0);
      }
      double E = 0.0;
      if (outD) E = warp_sum_d(lane < EPI_WARPS ? sh.red_e[c][lane] : 0.0);
      if (cnt > 1) {
        if (lane == 0) {
          if (outD) a.tile_dots[t] = E;
          meet_join(rows, k, t - off, G);
        }
        if (!meet_wait(rows, k, cnt, lane, a.err, &sh.abort, idle)) {
          ok = false;
          break;
        }
        if (lane == 0 && !outD && !direct) mbar_arrive(&sh.ready[c]);
        const GangSums mine = G;
        G = meet_sums(rows, k, lane);
        if (leader) meet_empty(rows, k, lane);
        if (out_of_range(G)) {
          if (!out) to_double(mine, trY, sqY);
          if (!meet_fp64(rows + kMeetRows, wide, a.tile_sums + off, t - off, cnt, lane, trY, sqY, a.err, &sh.abort,
                         idle)) {
            ok = false;
            break;
          }
        }
        if (outD && leader) {
          E = 0.0;
          for (int i = lane; i < cnt; i += 32) E += __ldcg(&a.tile_dots[off + i]);
          E = warp_sum_d(E);
        }
      }
      if (lane == 0) {
        if (!out_of_range(G)) to_double(G, trY, sqY);
        resident_step(s.st, trY, sqY, leader ? a.ctl + b : nullptr);
        if (!outD) mbar_arrive(&sh.coef[c]);
        if (leader) {
          if (outD) a.dots_out[3 * b] = E;
          if (k + 1 < kResStamps) st[k + 1] = (unsigned)(globaltimer() - t0);
        }
      }
      __syncwarp();
      act = hot->next.active != 0;
      if (!act && leader) {
        s.st.store(a.ctl + b, lane);
      }
    }
    __syncwarp();
  }
  if (!ok && lane == 0) {
    give_up(a);
    *(volatile int*)&sh.abort = 1;
  }
  if (lane == 0) {
    s.closed = 1;
    mbar_arrive(&sh.ready[c]);
  }
}

// LOCAL: every instance is one tile, whose planes stay in the operand tiles of its
// slot (N = 128: a layer 5.4 -> 4.6 us, N = 64: 3.7).
template <bool SPLIT, bool LOCAL>
__global__ void __launch_bounds__(THREADS, 1) resident_kernel(const __grid_constant__ ResMaps maps, const ResArgs a) {
  constexpr int STAGES = SPLIT ? STAGES_SPLIT : STAGES_PLAIN;
  constexpr int STAGE_BYTES = SPLIT ? STAGE_SPLIT : STAGE_PLAIN;
  constexpr int PLANES = SPLIT ? 2 : 1;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = smem_raw;
  float* trbuf = reinterpret_cast<float*>(smem + OPERAND_BYTES);
  Shared& sh = *reinterpret_cast<Shared*>(smem + OPERAND_BYTES + TR_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (smem_u32(smem_raw) & 1023u) {  // the swizzled operand tiles need it; the same for every CTA
    if (threadIdx.x == 0) give_up(a, SP2_ERR_UNSUPPORTED);
    return;
  }

  if (threadIdx.x == 0) {
    sh.abort = 0;
    for (int k = 0; k < STAGES; ++k) {
      mbar_init(&sh.full[k], 1);
      mbar_init(&sh.empty[k], 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(&sh.ready[k], 1);
      mbar_init(&sh.coef[k], 1);
      mbar_init(&sh.acc_full[k], 1);
      mbar_init(&sh.epi_done[k], EPI_WARPS);
    }
    for (int k = 0; k < WQ; ++k) mbar_init(&sh.wq_full[k], 1);
    mbar_init(&sh.drain, 1);
    mbar_init(&sh.never, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(&sh.tmem, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = sh.tmem;
  volatile int* abort_flag = &sh.abort;
  const unsigned long long lim = a.wait_ns ? a.wait_ns : kTimeoutNs;
  // waits for work (a gang still forming) last as long as other solves do
  const unsigned long long idle = lim > kTimeoutNs ? lim : kTimeoutNs;

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      uint32_t rphase = 0;  // bit c: phase of ready[c]
      // slot 0's gang and the layer whose planes it waits for (Slot::direct), or none
      long long* rows = nullptr;
      int cnt = 0, layer = 0;
      bool open0 = true, open1 = a.two_slots != 0, ok = true;
      int last = 1, stage = 0;
      uint32_t phase = 0, seq = 0;
      uint32_t armed[STAGES];
#pragma unroll
      for (int k = 0; k < STAGES; ++k) armed[k] = 0;
      for (int k = 0; k < 8; ++k)
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&maps.m[k >> 2][k & 3])) : "memory");
      while (ok && (open0 || open1)) {
        int c = -1;
        const uint64_t w0 = globaltimer();
        bool gang = false;  // slot 0 is ready through its gang's arrivals
        for (int spin = 0; c < 0; ++spin) {
          const int o = last ^ 1;
          if ((o ? open1 : open0) && mbar_test(&sh.ready[o], (rphase >> o) & 1u))
            c = o;
          else if ((last ? open1 : open0) && mbar_test(&sh.ready[last], (rphase >> last) & 1u))
            c = last;
          else if (rows && arrived(rows, layer) >= cnt) {
            __threadfence();  // what the gang stored before it arrived
            gang = true;
            c = 0;
          } else if ((spin & 63) == 63 && (*abort_flag || globaltimer() - w0 > idle))
            break;
        }
        if (c < 0) {
          ok = false;
          break;
        }
        if (!gang) rphase ^= 1u << c;
        last = c;
        const volatile Slot& s = sh.slot[c];
        if (!gang && s.closed) {
          (c ? open1 : open0) = false;
          if (c == 0) rows = nullptr;
          continue;
        }
        const int b = s.b, I = s.I, J = s.J, N = s.N, par = s.par, first = s.first;
        // after this layer's products: its gang's planes, or (the last layer) the
        // control warp
        if (c == 0) {
          rows = s.direct && !LOCAL ? s.rows : nullptr;
          cnt = s.cnt;
          layer = s.layer;
        }
        // a gang's planes come from generic stores and are read by the TMA unit (a
        // proxy fence by each of the storing threads took 0.8 us)
        if (gang) fence_proxy_async();
        sh.wq[seq % WQ] = c;
        mbar_arrive(&sh.wq_full[seq % WQ]);
        ++seq;
        const CUtensorMap* m = maps.m[par];
        const bool same = I == J;  // diagonal tile: one operand serves as both
        const int rowA = I * TB, rowB = J * TB, nk = (N + BK - 1) / BK;
        for (int kb = 0; kb < nk; ++kb) {
          if (!mbar_wait(&sh.empty[stage], phase ^ 1u, abort_flag, lim)) {
            ok = false;
            break;
          }
          // (a lone tile's operands have a place of their own; after the first layer
          // its epilogue has left them there)
          uint8_t* dst = smem + (LOCAL ? (2 * c + kb) * PLANES * HALF_BYTES : stage * STAGE_BYTES);
          ++armed[stage];
          if (LOCAL && !first) {
            mbar_arrive(&sh.full[stage]);
            if (++stage == STAGES) {
              stage = 0;
              phase ^= 1u;
            }
            continue;
          }
          mbar_expect_tx(&sh.full[stage], (same ? 1 : 2) * PLANES * HALF_BYTES);
          const int k0 = kb * BK, ks = k0 / BN;  // super column of this K block
          const bool ta = ks < (I >> 1), tb = ks < (J >> 1);
          load_half(dst, &m[0], &m[2], ta, rowA, k0, b, &sh.full[stage]);
          if (SPLIT) load_half(dst + HALF_BYTES, &m[1], &m[3], ta, rowA, k0, b, &sh.full[stage]);
          if (!same) {
            load_half(dst + PLANES * HALF_BYTES, &m[0], &m[2], tb, rowB, k0, b, &sh.full[stage]);
            if (SPLIT) load_half(dst + 3 * HALF_BYTES, &m[1], &m[3], tb, rowB, k0, b, &sh.full[stage]);
          }
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      sh.wq[seq % WQ] = WQ_END;
      mbar_arrive(&sh.wq_full[seq % WQ]);
      if (!ok || *abort_flag) {
        give_up(a);
        *abort_flag = 1;
        for (int k = 0; k < STAGES; ++k) {  // copies in flight land before the CTA leaves
          if (armed[k] == 0) continue;
          const uint64_t t0 = globaltimer();
          while (!mbar_test(&sh.full[k], (armed[k] - 1u) & 1u) && globaltimer() - t0 < lim) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true, issued = false;
      if (a.stall && !mbar_wait(&sh.never, 0, abort_flag, lim)) ok = false;
      for (uint32_t seq = 0; ok; ++seq) {
        if (!mbar_wait(&sh.wq_full[seq % WQ], (seq / WQ) & 1u, abort_flag, idle)) {
          ok = false;
          break;
        }
        const int c = *(volatile int*)&sh.wq[seq % WQ];
        if (c == WQ_END) break;
        const volatile Slot& s = sh.slot[c];
        const int I = s.I, J = s.J, nk = (s.N + BK - 1) / BK;
        const bool same = I == J;
        tc_fence_after();
        const uint32_t d = tmem_base + c * SLOT_COLS;
        for (int kb = 0; kb < nk; ++kb) {
          if (!mbar_wait(&sh.full[stage], phase, abort_flag, lim)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t st =
              smem_u32(smem + (LOCAL ? (2 * c + kb) * PLANES * HALF_BYTES : stage * STAGE_BYTES));
          const uint32_t sb = same ? st : st + PLANES * HALF_BYTES;
          const int ks = kb * BK / BN;
          const bool ta = ks < (I >> 1), tb = ks < (J >> 1);
          const uint32_t idesc = IDESC_T | (ta ? IDESC_A_MN : 0u) | (tb ? IDESC_B_MN : 0u);
#pragma unroll
          for (int u = 0; u < BK / UMMA_K; ++u) {
            const uint32_t oa = ta ? u * 2048u : u * UMMA_K * 2u, ob = tb ? u * 2048u : u * UMMA_K * 2u;
            const uint64_t a0 = ta ? make_desc_mn128(st + oa) : make_desc_sw128(st + oa);
            const uint64_t b0 = tb ? make_desc_mn128(sb + ob) : make_desc_sw128(sb + ob);
            mma_f16_id(d, a0, b0, idesc, (kb > 0 || u > 0) ? 1u : 0u);  // hp hp (plain: hi hi)
            if (SPLIT) {
              const uint32_t la = st + HALF_BYTES + oa, lb = sb + HALF_BYTES + ob;
              const uint64_t a1 = ta ? make_desc_mn128(la) : make_desc_sw128(la);
              const uint64_t b1 = tb ? make_desc_mn128(lb) : make_desc_sw128(lb);
              mma_f16_id(d, a1, b0, idesc, 1u);  // lo' hp
              mma_f16_id(d, a0, b1, idesc, 1u);  // hp lo'
            }
          }
          mma_commit(&sh.empty[stage]);
          issued = true;
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (ok) mma_commit(&sh.acc_full[c]);
      }
      if (!ok || *abort_flag) {
        give_up(a);
        *abort_flag = 1;
      }
      if (issued) {
        mma_commit(&sh.drain);
        const uint64_t t0 = globaltimer();
        while (!mbar_test(&sh.drain, 0) && globaltimer() - t0 < lim) {
        }
      }
    }
  } else if (warp >= CTL_WARP) {
    const int c = warp - CTL_WARP;
    if (c == 0 || a.two_slots) control<LOCAL>(a, sh, c, lane, idle);
  } else {
    // ------------------------------------------------------------ epilogue
    const int ew = warp - 2, q = warp & 3;
    uint32_t aphase = 0;  // bit c: phase of acc_full[c]
    for (uint32_t seq = 0;; ++seq) {
      if (!__all_sync(0xffffffffu, mbar_wait(&sh.wq_full[seq % WQ], (seq / WQ) & 1u, abort_flag, idle))) break;
      const int c = *(volatile int*)&sh.wq[seq % WQ];
      if (c == WQ_END) break;
      uint8_t* area = smem + 2 * c * PLANES * HALF_BYTES;
      if (!epilogue<SPLIT, LOCAL>(a, sh, c, area, (aphase >> c) & 1u, tmem_base, ew, q, lane, trbuf + ew * (16 * 32), lim)) {
        if (lane == 0) give_up(a);
        *abort_flag = 1;
        break;
      }
      aphase ^= 1u << c;
    }
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

}  // namespace res

// ---------------------------------------------------------------- input layer
// The resident solve's input layer: one warp per row of H forms Y_0 (kept by
// nobody: the first layer's epilogue forms its tile of it again from H), writes
// its operand planes from the row's super tile on, up to the padded row length
// (the only part the operand loads read), and sums the row's squares in FP64
// in the order of rownorm_kernel (vec_norm: its float4 form).  The last block
// of an instance adds the traces and runs the first control step.  HBM-bound:
// H read once, half the planes written.
__global__ void __launch_bounds__(256) resident_input_kernel(const ResArgs a, int vec_norm) {
  const int b = blockIdx.y;
  const int N = a.Ns[b];
  const int nb = (N + 7) / 8;
  if ((int)blockIdx.x >= nb) return;
  Ctl* c = a.ctl + b;
  if (c->phase == PHASE_ERROR) return;
  const InputScale in = input_scale(c->e_min, c->e_max, a.shift);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blockIdx.x * 8 + warp;
  double acc = 0.0, tr = 0.0;
  if (r < N) {
    const float* row = a.H[b] + (long long)r * N;
    __half* p0 = a.p0[0] + (long long)b * a.slot_h + (long long)r * a.ld_h;
    __half* p1 = a.p1[0] ? a.p1[0] + (long long)b * a.slot_h + (long long)r * a.ld_h : nullptr;
    const int cs = r & ~(kTcBN - 1);
    const bool vec_h = (N & 3) == 0 && (reinterpret_cast<uintptr_t>(a.H[b]) & 15) == 0;
    // the diagonal once per row: FP64 per element, even predicated off, would
    // bound the pass (1.97 ms against 0.33 for the bounds' pass over the same
    // 512 matrices)
    const float yd = input_diag(row[r], in);
    tr = lane == 0 ? (double)yd : 0.0;
    auto y0 = [&](float h, int col) { return col == r ? yd : input_offdiag(h, in); };
    acc = res::plane_row(row, N, vec_h, vec_norm, y0, cs, p0, p1, a.lo_scale, lane, [](int, const float (&)[4]) {});
    acc = warp_sum_d(acc);
    if (lane == 0) const_cast<double*>(a.rn)[(long long)b * a.ld_rn + r] = acc;
  }
  __shared__ double s_q[8], s_t[8];
  __shared__ bool s_last;
  if (lane == 0) {
    s_q[warp] = acc;
    s_t[warp] = tr;
  }
  __syncthreads();
  // the gang's meeting rows of the resident launch
  if (blockIdx.x == 0 && threadIdx.x < 2 * kMeetRows) a.sums[(long long)b * 2 * kMeetRows + threadIdx.x] = 0;
  double2* part = a.part + (long long)b * gridDim.x;
  if (threadIdx.x == 0) {
    double q = 0.0, t = 0.0;
    for (int w = 0; w < 8; ++w) {
      q += s_q[w];
      t += s_t[w];
    }
    part[blockIdx.x] = make_double2(t, q);
    __threadfence();
    s_last = atomicAdd(&a.tickets[b], 1u) == (unsigned)nb - 1u;
  }
  __syncthreads();
  if (!s_last || warp != 0) return;
  __threadfence();
  double T = 0.0, Q = 0.0;
  for (int k = lane; k < nb; k += 32) {
    const double2 p = __ldcg(&part[k]);
    T += p.x;
    Q += p.y;
  }
  T = warp_sum_d(T);
  Q = warp_sum_d(Q);
  if (lane == 0) {
    c->alpha_next = a.shift ? c->e_max * (1.0 / (c->e_max - c->e_min)) : 0.0;
    control_step(c, T, Q);
  }
}

cudaError_t launch_resident_input(const ResArgs& a, int vec_norm, int Nmax, int batch, cudaStream_t st) {
  resident_input_kernel<<<dim3((Nmax + 7) / 8, batch), 256, 0, st>>>(a, vec_norm);
  return cudaGetLastError();
}

cudaError_t launch_resident(const ResArgs& a, const ResMaps& maps, bool split, int grid, cudaStream_t st) {
  constexpr int smem = res::OPERAND_BYTES + res::TR_BYTES + (int)sizeof(res::Shared);
  static_assert(smem <= 227 * 1024, "shared memory");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(res::THREADS, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // the gangs wait on one another
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto go = [&](auto kernel) -> cudaError_t {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e == cudaSuccess ? cudaLaunchKernelEx(&cfg, kernel, maps, a) : e;
  };
  if (a.local) return split ? go(res::resident_kernel<true, true>) : go(res::resident_kernel<false, true>);
  return split ? go(res::resident_kernel<true, false>) : go(res::resident_kernel<false, false>);
}

}  // namespace sp2
