// Resident FP32 solve on the CUDA cores: the FFMA comparator's layers in one
// cooperative launch, for matrices too small to fill the chip with the
// 128 x 128 tiles of syrk_simt.cu (N = 512: 10 tiles for 152 SMs, 82 us a
// layer) and to pay two launches per layer, finished or not.
//
// A CTA owns tiles of TS x TS (32 or 64: whichever leaves the busiest CTA less
// to do) of the upper triangle, t = CTA, CTA + grid, ...  Per layer:
//   FFMA warps     products of the tiles (operand rows from L2 by cp.async,
//                  several chunks of 32 k ahead), then, once the layer's
//                  coefficients are known, the update and its mirror;
//   row-norm warps FP64 row norms of the layer's input under the products
//                  (the diagonal of the square and ||Y||_F^2);
//   control warp   two meetings of all CTAs: tiles complete (the next layer's
//                  products may start), then row norms complete (the control
//                  step; the next layer's updates may start).
// Each element accumulates over k in ascending order in one register, and the
// row norms in rownorm_kernel's order, as in the launch-per-layer kernels: the
// same bits.  Measured: N = 512 87 -> 10.3 us a layer (the call 4.33 -> 0.50
// ms), N = 1023 146 -> 40 us.  What is left at N = 512: products 7 us, bound by
// shared-memory loads, the meetings of 136 CTAs and their skew 3 us.
#include "common.cuh"
#include "kernels.h"
#include "resident.cuh"
#include "tc_ptx.cuh"

namespace sp2 {
namespace res32 {

using namespace sp2::tc;
using namespace sp2::res;

constexpr int KC = 32;       // k per staged chunk
constexpr int LDS = KC + 4;  // floats per staged row: eight consecutive rows' float4 cover every bank
constexpr int RN_WARPS = 8;  // row-norm warps

template <int TS>
struct Cfg {
  // four FFMA warps, one a scheduler, of 4 x 2 or 8 x 4 elements (rows x
  // columns) a thread: shared memory hands 32 lanes a value per cycle, so a k
  // of a tile costs (MR + MC) FT / 32 = 24 or 48 cycles there.  Fewer warps of
  // larger pieces (4 x 4 on two: 16 cycles) left two schedulers idle and took
  // 37 a k, more of smaller ones (4 x 4 on eight for side 64: 64 cycles) 70.
  static constexpr int FW = 4;
  static constexpr int FT = 32 * FW;
  static constexpr int MR = TS / 8, MC = TS / 16;
  static constexpr int TX = TS / MC, TY = TS / MR;      // threads along a tile's columns and rows
  static constexpr int THREADS = FT + 32 * RN_WARPS + 32;
  static constexpr int CP = 2 * TS * (KC / 4) / FT;     // 16-byte copies per thread and chunk: 4 or 8
  // chunks in flight or in use: a chunk's products take 0.2 (32) or 0.6 us (64)
  // against about 1 us of L2 latency
  static constexpr int STAGES = TS == 32 ? 8 : 4;
  static constexpr int STAGE_FLOATS = 2 * TS * LDS;     // rows of A, then rows of B
  static constexpr int SMEM = STAGES * STAGE_FLOATS * 4;
};

template <int TS>
struct Shared {
  uint64_t gate, coef, tiles_done, rn_done;
  int abort;
  long long red_t[4];
  double red_d[4];  // the same in FP64, where red_t is marked out of range
  double red_q[RN_WARPS];
  SolveState st;
};

// 16 bytes (the first `bytes` of them, zeros after) from global to shared memory
__device__ __forceinline__ void cp16(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
}

// Row norms of Y's rows first, first + step, ... in rownorm_kernel's order;
// their sum in lane 0.
__device__ __forceinline__ double row_norms(const float* Y, long long ld, int N, double* rn, int first, int step,
                                            int lane) {
  double blk = 0.0;
  for (int i = first; i < N; i += step) {
    const float* row = Y + (long long)i * ld;
    const float4* r4 = reinterpret_cast<const float4*>(row);
    const int n4 = N >> 2;
    double acc = 0.0;
    for (int j0 = 0; j0 < n4; j0 += 32 * 8) {
      float f = 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int j = j0 + u * 32 + lane;
        if (j < n4) {
          const float4 v = __ldcg(r4 + j);
          f = fmaf(v.x, v.x, f);
          f = fmaf(v.y, v.y, f);
          f = fmaf(v.z, v.z, f);
          f = fmaf(v.w, v.w, f);
        }
      }
      acc += (double)f;
    }
    for (int j = (n4 << 2) + lane; j < N; j += 32) acc += (double)__ldcg(row + j) * (double)__ldcg(row + j);
    acc = warp_sum_d(acc);
    if (lane == 0) {
      rn[i] = acc;
      blk += acc;
    }
  }
  return blk;
}

// A CTA's sum of row norms for the meeting (with a shift in [0, 1] they are at most
// 1 each; q < 2^15).
__device__ __forceinline__ GangSums to_fixed(double q) {
  const long long hi = __double2ll_rd(q * 0x1p25);
  return GangSums{0, hi, min((1ll << 28) - 1, __double2ll_rn((q * 0x1p25 - (double)hi) * 0x1p28))};
}

// The control warp: meetings and control steps, layer after layer.  False: abort.
template <int TS>
__device__ __forceinline__ bool control(const Res32Args& a, Shared<TS>& sh, int lane, unsigned long long lim) {
  constexpr int FW = Cfg<TS>::FW;
  const int G = (int)gridDim.x, me = (int)blockIdx.x;
  Ctl* hot = sh.st.ctl();
  const volatile int* ab = &sh.abort;
  sh.st.load(a.ctl, lane);
  if (!hot->next.active) return true;
  const bool exact = fp64_sums(hot);
  long long* fp64_rows = a.sums + 2 * kMeetRows;
  int wide = 0;  // meetings of sums in FP64
  const uint64_t t0 = globaltimer();
  if (lane == 0) {
    mbar_arrive(&sh.gate);
    mbar_arrive(&sh.coef);
  }
  for (int k = 0;; ++k) {
    prepare(sh.st, lane);
    const uint32_t ph = k & 1;
    if (!__all_sync(0xffffffffu, mbar_wait(&sh.tiles_done, ph, &sh.abort, lim))) return false;
    const bool outD = hot->next.out_mode == OUT_D;
    // traces and square norms out of the fixed-point range, or no number, meet once
    // more in FP64, as in csrc/resident.cu
    double trY = 0.0, sqY = 0.0;
    const long long rt = lane < FW ? sh.red_t[lane] : 0;
    const bool out_t = __any_sync(0xffffffffu, rt == T_OUT);
    GangSums S{0, SQ_BIG, 0};
    if (!out_t)
      S = GangSums{warp_sum_ll(rt), 0, 0};
    else
      trY = warp_sum_d(rt == T_OUT ? sh.red_d[lane] : (double)rt * T_UNIT);
    if (lane == 0) meet_join(a.sums, k, me, S);
    if (!meet_wait(a.sums, k, G, lane, a.err, ab, lim)) return false;
    if (lane == 0 && !outD) mbar_arrive(&sh.gate);
    const long long own = S.t;
    S = meet_sums(a.sums, k, lane);
    if (me == 0) meet_empty(a.sums, k, lane);
    if (!out_of_range(S)) {
      trY = (double)S.t * T_UNIT;
    } else {
      if (!out_t) trY = (double)own * T_UNIT;
      if (!meet_fp64(fp64_rows, wide, a.slots, me, G, lane, trY, sqY, a.err, ab, lim)) return false;
    }
    if (!outD) {
      if (!__all_sync(0xffffffffu, mbar_wait(&sh.rn_done, ph, &sh.abort, lim))) return false;
      const double Q = warp_sum_d(lane < RN_WARPS ? sh.red_q[lane] : 0.0);
      long long* norms = a.sums + kMeetRows;
      if (lane == 0) meet_join(norms, k, me, !(Q < 0x1p15) || exact ? GangSums{0, SQ_BIG, 0} : to_fixed(Q));
      if (!meet_wait(norms, k, G, lane, a.err, ab, lim)) return false;
      const GangSums q = meet_sums(norms, k, lane);
      if (me == 0) meet_empty(norms, k, lane);
      double t = 0.0;
      if (!out_of_range(q)) {
        to_double(q, t, sqY);
      } else {
        sqY = Q;
        if (!meet_fp64(fp64_rows, wide, a.slots, me, G, lane, t, sqY, a.err, ab, lim)) return false;
      }
    }
    if (lane == 0) {
      resident_step(sh.st, trY, sqY, me == 0 ? a.ctl : nullptr);
      if (!outD) mbar_arrive(&sh.coef);
      if (me == 0 && k + 1 < kResStamps) a.stamps[k + 1] = (unsigned)(globaltimer() - t0);
    }
    __syncwarp();
    if (outD) {
      if (me == 0) sh.st.store(a.ctl, lane);
      return true;
    }
  }
}

template <int TS>
__global__ void __launch_bounds__(Cfg<TS>::THREADS, 1) resident_fp32_kernel(const Res32Args a) {
  using C = Cfg<TS>;
  __shared__ __align__(16) Shared<TS> sh;
  extern __shared__ __align__(16) float stages[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int N = a.N, G = (int)gridDim.x;
  const long long ld = a.ld_y;
  if (tid == 0) {
    sh.abort = 0;
    mbar_init(&sh.gate, 1);
    mbar_init(&sh.coef, 1);
    mbar_init(&sh.tiles_done, C::FW);
    mbar_init(&sh.rn_done, RN_WARPS);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // a solve that ended in the prologue (bad bounds) leaves at once
  if (!a.ctl->next.active) return;
  const unsigned long long lim = a.wait_ns > kTimeoutNs ? a.wait_ns : kTimeoutNs;
  volatile int* ab = &sh.abort;
  bool ok = true;

  if (warp == C::FW + RN_WARPS) {
    ok = control<TS>(a, sh, lane, lim);
  } else if (warp >= C::FW) {
    // ------------------------------------------------------------ row norms
    const int w = warp - C::FW;
    ok = __all_sync(0xffffffffu, mbar_wait(&sh.gate, 0, ab, lim));
    for (int k = 0; ok; ++k) {
      // layer k writes D: it has no successor; otherwise the gate of layer
      // k + 1 says that the tiles of its input are complete
      ok = __all_sync(0xffffffffu, mbar_wait(&sh.coef, k & 1, ab, lim));
      if (!ok || sh.st.ctl()->next.out_mode == OUT_D) break;
      ok = __all_sync(0xffffffffu, mbar_wait(&sh.gate, (k + 1) & 1, ab, lim));
      if (!ok) break;
      const double q = row_norms(a.Y[(k + 1) & 1], ld, N, a.rn, (int)blockIdx.x * RN_WARPS + w, G * RN_WARPS, lane);
      if (lane == 0) {
        sh.red_q[w] = q;
        mbar_arrive(&sh.rn_done);
      }
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------ products
    const int tx = tid % C::TX, ty = tid / C::TX;
    const int nk = (N + KC - 1) / KC;
    // the named barrier of the FFMA warps; where they have waited, with one
    // answer for all (a warp that gives up leaves none behind in the barrier)
    auto sync = [&]() { asm volatile("barrier.cta.sync 1, %0;" ::"n"(C::FT) : "memory"); };
    auto all = [&](bool mine) {
      int r;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\t"
          "setp.ne.s32 q, %1, 0;\n\t"
          "barrier.cta.red.and.pred p, 1, %2, q;\n\t"
          "selp.s32 %0, 1, 0, p;\n\t}\n"
          : "=r"(r)
          : "r"(mine ? 1 : 0), "n"(C::FT)
          : "memory");
      return r != 0;
    };
    for (int k = 0; ok; ++k) {
      const uint32_t ph = k & 1;
      ok = all(mbar_wait(&sh.gate, ph, ab, lim));
      if (!ok) break;
      const float* Y = a.Y[k & 1];
      float* Yn = a.Y[(k + 1) & 1];
      long long tr = 0;
      bool outD = false, out_t = fp64_sums(sh.st.ctl());
      for (int t = blockIdx.x; t < a.ntiles && ok; t += G) {
        int b, I, J, h;
        unpack_tile(a.tiles[t], b, I, J, h);
        const int r0 = I * TS, c0 = J * TS;
        float acc[C::MR][C::MC];
#pragma unroll
        for (int i = 0; i < C::MR; ++i)
#pragma unroll
          for (int j = 0; j < C::MC; ++j) acc[i][j] = 0.f;
        // chunk kb of both operands' rows into its stage (zeros past N)
        auto fetch = [&](int kb) {
          if (kb < nk) {
            float* st = stages + (kb % C::STAGES) * C::STAGE_FLOATS;
#pragma unroll
            for (int u = 0; u < C::CP; ++u) {
              const int f = tid + u * C::FT, r = f >> 3, kk = kb * KC + (f & 7) * 4;
              const int g = r < TS ? r0 + r : c0 + r - TS;
              const bool in = g < N && kk < N;
              cp16(st + r * LDS + (f & 7) * 4, in ? Y + (long long)g * ld + kk : Y, in ? min(16, 4 * (N - kk)) : 0);
            }
          }
          asm volatile("cp.async.commit_group;" ::: "memory");
        };
#pragma unroll
        for (int u = 0; u < C::STAGES - 1; ++u) fetch(u);
        for (int kb = 0; kb < nk; ++kb) {
          asm volatile("cp.async.wait_group %0;" ::"n"(C::STAGES - 2) : "memory");
          sync();  // the chunk is there for every warp, and the stage refilled below is read by none
          fetch(kb + C::STAGES - 1);
          const float* A = stages + (kb % C::STAGES) * C::STAGE_FLOATS + ty * LDS;
          const float* B = stages + (kb % C::STAGES) * C::STAGE_FLOATS + (TS + tx) * LDS;
          // four k at a time, the next four loaded under the products (one warp a
          // scheduler: nothing else covers the loads)
          float4 av[2][C::MR], bv[2][C::MC];
          auto load = [&](int w, int q) {
#pragma unroll
            for (int i = 0; i < C::MR; ++i) av[w][i] = *reinterpret_cast<const float4*>(A + i * C::TY * LDS + q);
#pragma unroll
            for (int j = 0; j < C::MC; ++j) bv[w][j] = *reinterpret_cast<const float4*>(B + j * C::TX * LDS + q);
          };
          load(0, 0);
#pragma unroll
          for (int q = 0; q < KC; q += 4) {
            const int w = (q >> 2) & 1;
            if (q + 4 < KC) load(w ^ 1, q + 4);
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
              for (int i = 0; i < C::MR; ++i)
#pragma unroll
                for (int j = 0; j < C::MC; ++j)
                  acc[i][j] = fmaf(e == 0 ? av[w][i].x : e == 1 ? av[w][i].y : e == 2 ? av[w][i].z : av[w][i].w,
                                   e == 0 ? bv[w][j].x : e == 1 ? bv[w][j].y : e == 2 ? bv[w][j].z : bv[w][j].w,
                                   acc[i][j]);
          }
        }
        sync();  // the next tile's first chunks go into stages that every warp has read
        // old values (all loads before the first store; the update's elements
        // cannot be told apart by the compiler), then the update, once the coefficients (and the row norms) are there
        float yold[C::MR][C::MC];
#pragma unroll
        for (int i = 0; i < C::MR; ++i)
#pragma unroll
          for (int j = 0; j < C::MC; ++j) {
            const int r = r0 + ty + C::TY * i, c = c0 + tx + C::TX * j;
            yold[i][j] = r < N && c < N ? __ldcg(Y + (long long)r * ld + c) : 0.f;
          }
        ok = all(mbar_wait(&sh.coef, ph, ab, lim));
        if (!ok) break;
        const LayerParams p = sh.st.ctl()->next;
        outD = p.out_mode == OUT_D;
        const bool mirror = I != J;
        float* out = outD ? a.D : Yn;
        const long long lo = outD ? N : ld;
#pragma unroll
        for (int i = 0; i < C::MR; ++i)
#pragma unroll
          for (int j = 0; j < C::MC; ++j) {
            const int r = r0 + ty + C::TY * i, c = c0 + tx + C::TX * j;
            if (r < N && c < N && r != c) {
              const float y = fmaf(p.ca, yold[i][j], p.cb * acc[i][j]);
              out[(long long)r * lo + c] = y;
              if (mirror) out[(long long)c * lo + r] = y;
            }
          }
        // the diagonal in FP64, outside the element loop
        if (!mirror) {
          for (int e = tid; e < TS && r0 + e < N; e += C::FT) {
            const int r = r0 + e;
            const double yd = p.ca_d * (double)__ldcg(Y + (long long)r * ld + r) + p.cb_d * __ldcg(a.rn + r) + p.cc_d;
            tr += __double2ll_rn(yd * 0x1p50);
            out_t = out_t || !(fabsf((float)yd) < T_LIMIT);
            out[(long long)r * lo + r] = outD ? (float)(yd + p.alpha_out) : (float)yd;
          }
        }
      }
      if (!ok) break;
      if (__any_sync(0xffffffffu, out_t)) {
        // the same elements once more, in FP64
        const LayerParams p = sh.st.ctl()->next;
        double trd = 0.0;
#pragma unroll 1
        for (int t = blockIdx.x; t < a.ntiles; t += G) {
          int b, I, J, h;
          unpack_tile(a.tiles[t], b, I, J, h);
          for (int r = I * TS + tid; I == J && r < min(N, (I + 1) * TS); r += C::FT)
            trd += p.ca_d * (double)__ldcg(Y + (long long)r * ld + r) + p.cb_d * __ldcg(a.rn + r) + p.cc_d;
        }
        trd = warp_sum_d(trd);
        if (lane == 0) sh.red_d[warp] = trd;
        tr = T_OUT;
      } else {
        tr = warp_sum_ll(tr);
      }
      __syncwarp();
      if (lane == 0) {
        sh.red_t[warp] = tr;
        mbar_arrive(&sh.tiles_done);
      }
      if (outD) break;
    }
  }
  if (!ok) {
    if (lane == 0) give_up(a);
    *ab = 1;
  }
}

}  // namespace res32

cudaError_t launch_resident_fp32(const Res32Args& a, int tile, int grid, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(tile == 32 ? res32::Cfg<32>::THREADS : res32::Cfg<64>::THREADS, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // the CTAs wait on one another
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto go = [&](auto kernel, int smem) -> cudaError_t {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    cfg.dynamicSmemBytes = smem;
    return cudaLaunchKernelEx(&cfg, kernel, a);
  };
  return tile == 32 ? go(res32::resident_fp32_kernel<32>, res32::Cfg<32>::SMEM)
                    : go(res32::resident_fp32_kernel<64>, res32::Cfg<64>::SMEM);
}

}  // namespace sp2
