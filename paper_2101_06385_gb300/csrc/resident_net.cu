// Resident network layers (sm_103a): the generalised layers of Eq. 16 and their
// adjoint, and the finite-temperature expansion, all layers of a batch in one
// cooperative launch.
//
// As the resident solve (csrc/resident.cu) a CTA keeps one or two 128 x 128
// tiles of the upper super tiles, one per slot, and the tiles of one matrix
// meet after every layer; but what each layer does is a list of operations the
// host wrote (NetOp), with coefficients known beforehand: products P = Y Y, or
// P = Y G + G Y over two K segments; the update of the iterate (or the adjoint
// G) in tensor memory; and per operation what leaves the tile: operand planes
// for the next one, whole matrices (checkpoints, results), the tile's iterate
// for a later operation, dot products.
//
// What bounds it: a small batch, the chain of a layer (5 us at N = 128 against
// 26-46 us of a launch); a large one, the tensor cores at the 128 x 128 tile's
// rate with the two slots taking turns, and neither the iterate nor the
// readout crosses HBM between layers.
//
// Accumulation order and arithmetic per element, and the row norms' and dot
// products' FP32 parts, are those of the launch-per-layer kernels.
#include <cuda.h>
#include <cuda_fp16.h>

#include "common.cuh"
#include "epilogue.cuh"
#include "kernels.h"
#include "resident.cuh"
#include "resident_tc.cuh"
#include "tc_ptx.cuh"

namespace sp2 {
namespace net {

using namespace sp2::tc;
using namespace sp2::res;

struct Slot {
  int b, I, J, t;  // matrix, tile row and column (128 units), tile index
  int closed;      // no more work in this slot
  NetOp op[2];       // operations in progress, by the parity of their number in the slot, and
  LayerParams p[2];  // their coefficients (a layer's first touch of them in global memory would
                     // stand in its chain)
};
static_assert(sizeof(NetOp) % 8 == 0 && sizeof(LayerParams) % 8 == 0, "copied in 8-byte words");

struct Shared {
  uint64_t full[STAGES_PLAIN], empty[STAGES_PLAIN];
  uint64_t ready[2];     // control warp -> producer: operands complete (or slot closed)
  uint64_t acc_full[2];  // MMA issuer -> epilogue
  uint64_t stored[2];    // epilogue warps -> control warp: planes and row norms stored, accumulator read (one slot)
  uint64_t epi_done[2][2];  // [slot][parity] the same: operation finished (a warp without rows may be an
                            //   operation ahead of the others: it must not stand in for them)
  uint64_t wq_full[WQ];  // producer -> MMA issuer and epilogue: next slot
  uint64_t drain, never;
  int wq[WQ];
  uint32_t tmem;
  int abort;
  double red[2][2][EPI_WARPS][3];  // [parity] dot products per warp: tr Yin, <Yin, aux>, <P, aux>
  Slot slot[2];
};

// Sums of FP32 values in 64-bit fixed point with the unit set by the largest
// (2^-53 of its power of two): exact but for terms 2^-29 of it, in any order, and
// without FP64 additions (64 cycles each, 19 a warp on the SM's one pipe).
// e: exponent of the largest, its biased FP32 exponent; fixed_ok(e): in range.
__device__ __forceinline__ bool fixed_ok(int e) { return e > 40 && e < 250; }
__device__ __forceinline__ long long to_fixed(float v, int e) {
  const float s = __int_as_float((279 - e) << 23);       // 2^(25 - (e - 127)): |v s| < 2^26
  const float r = __int_as_float((e - 25) << 23);        // its inverse
  const int hi = __float2int_rz(v * s);
  const int lo = __float2int_rn(fmaf(-(float)hi, r, v) * s * 0x1p28f);
  return ((long long)hi << 28) + (long long)lo;
}
__device__ __forceinline__ double from_fixed(long long v, int e) {
  return (double)v * __longlong_as_double((long long)(e - 127 - 53 + 1023) << 52);
}

// Row norm (Y^2)_rr of the input: FP64 ones, or the sum of the previous
// operation's segment sums (in FP64 where the fixed-point unit would leave its range).
__device__ __forceinline__ double row_norm(const NetArgs& a, const NetOp& o, int b, int r) {
  if (o.rn) return o.rn[(long long)b * a.N + r];
  const float* p = a.rnp[o.rnp ^ 1] + (long long)b * a.slot_rnp + r;
  const int nseg = (a.N + 31) >> 5;
  float top = 0.f;
  for (int s = 0; s < nseg; s += 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = s + u < nseg ? __ldcg(p + (long long)(s + u) * a.ld_rnp) : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) top = (v[u] > top || isnan(v[u])) ? v[u] : top;
  }
  if (top == 0.f) return 0.0;
  const int e = (__float_as_int(top) >> 23) & 255;
  if (!fixed_ok(e)) {
    double acc = 0.0;
    for (int s = 0; s < nseg; ++s) acc += (double)__ldcg(p + (long long)s * a.ld_rnp);
    return acc;
  }
  long long acc = 0;
  for (int s = 0; s < nseg; s += 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = s + u < nseg ? __ldcg(p + (long long)(s + u) * a.ld_rnp) : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) acc += to_fixed(v[u], e);
  }
  return from_fixed(acc, e);
}

// Sums over the warp's lanes of one FP32 value each, two side by side.
__device__ __forceinline__ void lanes_sum(float u, float v, double& su, double& sv) {
  const int eu = __reduce_max_sync(0xffffffffu, (__float_as_int(u) >> 23) & 255);
  const int ev = __reduce_max_sync(0xffffffffu, (__float_as_int(v) >> 23) & 255);
  if (fixed_ok(eu) && fixed_ok(ev)) {
    long long a = to_fixed(u, eu), b = to_fixed(v, ev);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    su = from_fixed(a, eu);
    sv = from_fixed(b, ev);
  } else {
    su = eu ? warp_sum_d((double)u) : 0.0;  // (exponent 0: zeros, and denormals)
    sv = ev ? warp_sum_d((double)v) : 0.0;
  }
}

// The lane's four columns of its eight rows of a matrix of the batch.
__device__ __forceinline__ void load_rows(const float* M, int N, int row, int ce, int rows_left, bool vec,
                                          float (&y)[32]) {
  const float* p = M + (long long)row * N + ce;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 o = 4 * i < rows_left ? epi::ld4(p, ce, N, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    p += 4 * N;
    y[4 * i] = o.x;
    y[4 * i + 1] = o.y;
    y[4 * i + 2] = o.z;
    y[4 * i + 3] = o.w;
  }
}

// Three values summed over the warp in lane 0 (a halving butterfly: six FP64
// additions instead of fifteen).
__device__ __forceinline__ void sum3(double& a, double& b, double& c) {
  const int lane = threadIdx.x & 31;
  // lanes with bit 4 clear take (a, b), the others (c, 0); then bit 3 splits those
  const bool hi = (lane & 16) != 0;
  double x = hi ? c : a, y = hi ? 0.0 : b;
  x += __shfl_xor_sync(0xffffffffu, hi ? a : c, 16);
  const double sb = __shfl_xor_sync(0xffffffffu, b, 16);
  y = hi ? 0.0 : b + sb;
  const bool h2 = (lane & 8) != 0;
  double z = h2 ? y : x;
  z += __shfl_xor_sync(0xffffffffu, h2 ? x : y, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
  a = __shfl_sync(0xffffffffu, z, 0);
  b = __shfl_sync(0xffffffffu, z, 8);
  c = __shfl_sync(0xffffffffu, z, 16);
}

// One operation on the warp's 32 x 32 chunk of a slot's tile (lane layouts of
// epi::tile).  False: the accumulator wait failed.
template <bool SPLIT, bool EARLY>
__device__ __forceinline__ bool epilogue(const NetArgs& a, Shared& sh, int c, uint32_t acc_phase, uint32_t tmem_base,
                                         int ew, int q, int lane, float* trb, unsigned long long lim) {
  const Slot& s = sh.slot[c];
  const uint32_t cur = EARLY ? acc_phase : 0u;  // (both count the slot's operations)
  const NetOp& o = s.op[cur];
  const LayerParams& p = s.p[cur];  // (in shared memory: registers hold the chunk)
  const int b = s.b, N = a.N, I = s.I, J = s.J;
  const bool adj = o.kind != 0;
  const int hc = ew >> 2, R0 = I * TB + q * 32, c0 = J * TB + hc * 32;
  const int nrows = min(32, N - R0);
  const bool mirror = (I >> 1) != (J >> 1);
  const float unscale = SPLIT ? a.lo_unscale * a.lo_unscale : 1.f;
  const int r4 = lane >> 3, c4 = lane & 7, ce = c0 + 4 * c4;
  const int rdiag = R0 + 4 * c4 + r4, id = 4 * c4 + r4;
  const bool dchunk = !mirror && c0 == R0;
  const bool dlane = dchunk && rdiag < N;
  const bool live = nrows > 0 && c0 < ((N + 63) & ~63);
  const uint32_t tacc = tmem_base + c * SLOT_COLS + ((uint32_t)(q * 32) << 16) + hc * 32;
  const uint32_t ty = tacc + Y_COL;
  const long long mat = (long long)b * N * N;
  // the tile's private store of an iterate: 8 float4 per lane, lanes side by side
  const long long priv = ((long long)s.t * EPI_WARPS + ew) * 1024 + lane * 4;

  // The warp has read its accumulator and stored its part of the planes and row
  // norms.  (The planes are read by the TMA units next: a lone tile's by its own;
  // a gang's cross behind the meeting's fence and one proxy fence by each producer.)
  auto stored = [&]() {
    if (!EARLY) return;
    if (live && o.out >= 0 && a.per == 1) fence_proxy_async();
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(&sh.stored[c]);
  };
  // kind 1: Y's four columns of row 4 i + r4
  auto aux4 = [&](int i) {
    if (o.aux) return *reinterpret_cast<const float4*>(o.aux + priv + i * 128);
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (4 * i + r4 < nrows) {
      const float* src = o.aux_x + mat;
      const bool vec = (N & 3) == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0;
      x = epi::ld4(src + (long long)(R0 + 4 * i + r4) * N + ce, ce, N, vec);
      if (dlane && i == c4) {
        const float v = r4 == 0 ? x.x : r4 == 1 ? x.y : r4 == 2 ? x.z : x.w;
        const float w = (float)((double)v + o.aux_add[b]);
        if (r4 == 0) x.x = w;
        if (r4 == 1) x.y = w;
        if (r4 == 2) x.z = w;
        if (r4 == 3) x.w = w;
      }
    }
    return x;
  };

  float y[32];
  float gy = 0.f, py = 0.f, dtr = 0.f;  // this lane's dot products
  double yd = 0.0;
  float yold_d = 0.f, ydf = 0.f;
  if (live) {
    double rn_l = 0.0;
    if (dlane && !adj) rn_l = row_norm(a, o, b, rdiag);
    if (o.from == NET_TMEM) {
      uint32_t w[32];
      __syncwarp();
      tmem_ld32(ty, w);
      tmem_ld_wait();
#pragma unroll
      for (int k = 0; k < 32; ++k) y[k] = __uint_as_float(w[k]);
    } else if (o.from == NET_KEPT) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(o.in + priv + i * 128);
        y[4 * i] = v.x;
        y[4 * i + 1] = v.y;
        y[4 * i + 2] = v.z;
        y[4 * i + 3] = v.w;
      }
    } else {
      const float* in = o.in + mat;
      load_rows(in, N, R0 + r4, ce, nrows - r4, (N & 3) == 0 && (reinterpret_cast<uintptr_t>(in) & 15) == 0, y);
      if (o.from != NET_FULL) {
        // the input layer's scaling of H, or a checkpoint less its shift
        const bool scale = o.from == NET_INPUT;
        const InputScale is = scale ? input_scale(a.ctl[b].e_min, a.ctl[b].e_max, a.shift) : InputScale();
        float hd = 0.f;
        if (dchunk) {
#pragma unroll
          for (int k = 0; k < 32; ++k)
            if (k == id) hd = y[k];
        }
        if (scale) {
#pragma unroll
          for (int k = 0; k < 32; ++k) y[k] = input_offdiag(y[k], is);
        }
        if (dchunk) {
          const float v = scale ? input_diag(hd, is) : (float)((double)hd + o.add[b]);
#pragma unroll
          for (int k = 0; k < 32; ++k)
            if (k == id) y[k] = v;
        }
      }
    }
    if (dchunk) {
#pragma unroll
      for (int k = 0; k < 32; ++k)
        if (k == id) yold_d = y[k];
    }
    if (o.readout == 2) {
      // the input layer's term c_0 X_0 = r_scale Y_0 + r_add I
      const float rd0 = dlane ? (float)((double)a.r_scale * (double)yold_d + a.r_add[b]) : 0.f;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float r_[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) r_[e] = dlane && 4 * i + e == id ? rd0 : a.r_scale * y[4 * i + e];
        *reinterpret_cast<float4*>(a.R + priv + i * 128) = make_float4(r_[0], r_[1], r_[2], r_[3]);
      }
    }
    if (dlane && !adj) {
      yd = p.ca_d * (double)yold_d + p.cb_d * rn_l + p.cc_d;
      ydf = (float)yd;
    }
    if (adj) {
      // <G, Y> on the old values (each lane's 32 products in one FP32 chain)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 x = aux4(i);
        gy = fmaf(y[4 * i], x.x, gy);
        gy = fmaf(y[4 * i + 1], x.y, gy);
        gy = fmaf(y[4 * i + 2], x.z, gy);
        gy = fmaf(y[4 * i + 3], x.w, gy);
      }
      if (dlane) dtr = yold_d;
    }
  }
  float4 x4[4];  // kind 1: Y's rows of a half
  if (live && adj) {
#pragma unroll
    for (int i = 0; i < 4; ++i) x4[i] = aux4(i);
  }
  if (!__all_sync(0xffffffffu, mbar_wait(&sh.acc_full[c], acc_phase, &sh.abort, lim))) return false;
  tc_fence_after();

  if (live) {
    const bool full = nrows == 32 && c0 + 32 <= N;
    const float cbu = p.cb * unscale;
    float p_d = 0.f;
    {
      const float ca = p.ca;
      turn_tmem(trb, tacc, lane, [&](int h) {
        if (adj && h == 1) {
#pragma unroll
          for (int i = 0; i < 4; ++i) x4[i] = aux4(4 + i);
        }
      }, [&](int i, const float4& pv) {
        if (adj) {
          const float4 x = x4[i & 3];
          py = fmaf(pv.x * unscale, x.x, py);
          py = fmaf(pv.y * unscale, x.y, py);
          py = fmaf(pv.z * unscale, x.z, py);
          py = fmaf(pv.w * unscale, x.w, py);
          if (dchunk && i == c4) p_d = (r4 == 0 ? pv.x : r4 == 1 ? pv.y : r4 == 2 ? pv.z : pv.w) * unscale;
        }
        y[4 * i] = fmaf(ca, y[4 * i], cbu * pv.x);
        y[4 * i + 1] = fmaf(ca, y[4 * i + 1], cbu * pv.y);
        y[4 * i + 2] = fmaf(ca, y[4 * i + 2], cbu * pv.z);
        y[4 * i + 3] = fmaf(ca, y[4 * i + 3], cbu * pv.w);
      });
    }
    if (!full) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (!(4 * i + r4 < nrows && ce + e < N)) y[4 * i + e] = 0.f;
    }
    if (dlane && adj) {
      yd = p.ca_d * (double)yold_d + p.cb_d * (double)p_d + p.cc_d;
      ydf = (float)yd;
    }
    if (dchunk) {
#pragma unroll
      for (int k = 0; k < 32; ++k)
        if (dlane && k == id) y[k] = ydf;
    }
    if (o.out >= 0) {
      const long long po = ((long long)o.out * a.batch + b) * a.slot_h + (long long)(R0 + r4) * a.ld_h + ce;
      store_planes<SPLIT>(y, a.p0 + po, SPLIT ? a.p1 + po : nullptr, a.ld_h, nrows - r4, a.lo_scale);
    }
    if (!adj && o.out >= 0) {
      // row norms of Y' for the next operation: per row over the 32 columns, per
      // column over the 32 rows (the mirror's rows)
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
      float* rnp = a.rnp[o.rnp] + (long long)b * a.slot_rnp;
      const float rsum = epi::lane_sums<8, 0>(rs);
      if (rdiag < N && c0 < N) rnp[(long long)(c0 >> 5) * a.ld_rnp + rdiag] = rsum;
      if (mirror) {
        const float csum = epi::lane_sums<4, 3>(cs);
        const int cm = c0 + 4 * c4 + r4;
        if (cm < N) rnp[(long long)(R0 >> 5) * a.ld_rnp + cm] = csum;
      }
    }
    stored();
    if (o.tmem) {
      uint32_t w[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) w[k] = __float_as_uint(y[k]);
      __syncwarp();
      tmem_st32(ty, w);
    }
    if (o.keep) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        *reinterpret_cast<float4*>(o.keep + priv + i * 128) =
            make_float4(y[4 * i], y[4 * i + 1], y[4 * i + 2], y[4 * i + 3]);
    }
    float full_d = ydf;
    if (o.readout) {
      // readout R += rc X' (tile-private), D = I - R in the last operation
      // (in two halves: loads before stores, which the compiler cannot tell apart,
      // within the registers)
      float rold_d = 0.f;
      const bool last = o.full != nullptr;
      const float rc = p.rc;
      float4* rp = reinterpret_cast<float4*>(a.R + priv);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float4 rv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) rv[u] = rp[(4 * h + u) * 32];
        if (dlane && (c4 >> 2) == h) {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (4 * h + u == c4) rold_d = r4 == 0 ? rv[u].x : r4 == 1 ? rv[u].y : r4 == 2 ? rv[u].z : rv[u].w;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = 4 * h + u;
          rv[u].x = fmaf(rc, y[4 * i], rv[u].x);
          rv[u].y = fmaf(rc, y[4 * i + 1], rv[u].y);
          rv[u].z = fmaf(rc, y[4 * i + 2], rv[u].z);
          rv[u].w = fmaf(rc, y[4 * i + 3], rv[u].w);
          if (last) {
            y[4 * i] = -rv[u].x;
            y[4 * i + 1] = -rv[u].y;
            y[4 * i + 2] = -rv[u].z;
            y[4 * i + 3] = -rv[u].w;
          } else {
            rp[i * 32] = rv[u];
          }
        }
      }
      if (dlane) {
        const double rd = (double)rold_d + p.rc_d * (yd + p.alpha_new);
        if (last)
          full_d = (float)(1.0 - rd);
        else
          a.R[priv + c4 * 128 + r4] = (float)rd;
      }
    } else if (dlane && o.full) {
      full_d = o.exact ? (float)(yd + p.alpha_out) : o.full_add ? (float)((double)ydf + o.full_add[b]) : ydf;
    }
    if (o.full) {
      // the whole matrix: this chunk and, off the diagonal super tiles, its mirror
      if (dchunk) {
#pragma unroll
        for (int k = 0; k < 32; ++k)
          if (dlane && k == id) y[k] = full_d;
      }
      float* F = o.full + mat;
      float* F2 = o.full2 ? o.full2 + mat : nullptr;
      const bool vec = (N & 3) == 0 && ((reinterpret_cast<uintptr_t>(F) | reinterpret_cast<uintptr_t>(F2)) & 15) == 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (4 * i + r4 < nrows) {
          const long long at = (long long)(R0 + 4 * i + r4) * N + ce;
          const float4 v = make_float4(y[4 * i], y[4 * i + 1], y[4 * i + 2], y[4 * i + 3]);
          epi::st4(F + at, v, ce, N, vec);
          if (F2) epi::st4(F2 + at, v, ce, N, vec);
        }
      }
      if (mirror) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
          for (int i = 4 * h; i < 4 * h + 4; ++i)
            *epi::tr_at(trb, 4 * (i - 4 * h) + r4, c4) =
                make_float4(y[4 * i], y[4 * i + 1], y[4 * i + 2], y[4 * i + 3]);
          __syncwarp();
          if ((lane >> 4) == h && lane < nrows) {
#pragma unroll
            for (int m = 0; m < 8; ++m) {
              const float4 v = *epi::tr_at(trb, lane & 15, m);
              const float ov[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (c0 + 4 * m + e < N) {
                  const long long at = (long long)(c0 + 4 * m + e) * N + R0 + lane;
                  F[at] = ov[e];
                  if (F2) F2[at] = ov[e];
                }
            }
          }
          __syncwarp();
        }
      }
    }
  }
  if (!live) stored();
  double s0 = 0.0, s1 = 0.0, s2 = 0.0;
  if (adj) {
    const double twice = mirror ? 2.0 : 1.0;
    lanes_sum(gy, py, s1, s2);
    s1 *= twice;
    s2 *= twice;
    double none;
    if (dchunk) lanes_sum(dtr, 0.f, s0, none);
  }
  if (!EARLY && live && o.out >= 0 && a.per == 1) fence_proxy_async();
  tmem_st_wait();
  tc_fence_before();
  __syncwarp();
  if (lane == 0) {
    if (adj) {
      sh.red[cur][c][ew][0] = s0;
      sh.red[cur][c][ew][1] = s1;
      sh.red[cur][c][ew][2] = s2;
    }
    mbar_arrive(&sh.epi_done[c][cur]);
  }
  return true;
}

// Control of one slot: takes the tiles of its list through their operations.
template <bool EARLY>
__device__ __forceinline__ void control(const NetArgs& a, Shared& sh, int c, int lane, unsigned long long idle) {
  Slot& s = sh.slot[c];
  const int sl = c * (int)gridDim.x + (int)blockIdx.x;
  uint32_t done_phase = 0, next = 0;  // parities of the operation to finish, to begin
  uint32_t done_round = 0;            // phase of epi_done[c][done_phase]
  bool ok = true;
  for (int li = a.list_off[sl]; ok && li < a.list_off[sl + 1]; ++li) {
    const int t = a.list[li], cnt = a.per;
    int b, I, J, h;
    unpack_tile(a.tiles[t], b, I, J, h);
    const int off = t - t % cnt;  // every matrix has the same number of tiles
    long long* rows = a.sums + (long long)b * kMeetRows;
    // lane l holds word l of the next operation and of its coefficients
    constexpr int OW = sizeof(NetOp) / 8, PW = sizeof(LayerParams) / 8;
    static_assert(OW <= 32 && PW <= 32, "one word a lane");
    long long wo = 0, wp = 0;
    auto fetch = [&](int k) {
      if (lane < OW) wo = reinterpret_cast<const long long*>(a.ops + k)[lane];
      const int layer = a.ops[k].layer;
      if (lane < PW) wp = reinterpret_cast<const long long*>(a.lp + (long long)layer * a.batch + b)[lane];
    };
    auto begin = [&]() {
      if (lane < OW) reinterpret_cast<long long*>(&s.op[next])[lane] = wo;
      if (lane < PW) reinterpret_cast<long long*>(&s.p[next])[lane] = wp;
      if (EARLY) next ^= 1u;
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.ready[c]);
    };
    fetch(0);
    if (lane == 0) {
      s.b = b;
      s.I = I;
      s.J = J;
      s.t = t;
      s.closed = 0;
    }
    begin();
    for (int k = 0; k < a.nops; ++k) {
      const int kind = __shfl_sync(0xffffffffu, (int)wo, 0);
      if (k + 1 < a.nops) fetch(k + 1);
      // The next operation's products need the gang's planes; the rest of this one's
      // epilogue (readout, whole matrices, dot products) runs beside them: expansion
      // of 8 x 512 220 -> 201 us, network step of 6 x 300 667 -> 634.
      const uint32_t cur = EARLY ? done_phase : 0u;
      auto finished = [&]() {
        return mbar_wait(&sh.epi_done[c][cur], EARLY ? done_round : done_phase, &sh.abort, idle);
      };
      if (!__all_sync(0xffffffffu, EARLY ? mbar_wait(&sh.stored[c], done_phase, &sh.abort, idle) : finished())) {
        ok = false;
        break;
      }
      if (k + 1 < a.nops && cnt > 1) {
        if (lane == 0) meet_join(rows, k, t - off, GangSums{0, 0, 0}, false);
        if (!meet_wait(rows, k, cnt, lane, a.err, &sh.abort, idle)) {
          ok = false;
          break;
        }
        if (t == off) meet_empty(rows, k, lane);
      }
      const int dot = s.op[cur].dot;
      if (k + 1 < a.nops) begin();
      if (EARLY && !__all_sync(0xffffffffu, finished())) {
        ok = false;
        break;
      }
      double d0 = 0.0, d1 = 0.0, d2 = 0.0;
      if (kind != 0 && lane < EPI_WARPS) {
        d0 = sh.red[cur][c][lane][0];
        d1 = sh.red[cur][c][lane][1];
        d2 = sh.red[cur][c][lane][2];
      }
      done_round ^= done_phase;
      done_phase ^= 1u;
      __syncwarp();
      if (kind != 0) {  // under the next operation's products
        sum3(d0, d1, d2);
        if (lane == 0) {
          double* td = a.tile_dots + 3 * ((long long)dot * a.ntiles + t);
          td[0] = d0;
          td[1] = d1;
          td[2] = d2;
        }
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

// EARLY: one slot; the next operation begins when this one's planes are stored
// (with two, where the other slot's products fill the time, its second set of
// operands cost 2 to 4 %).
template <bool SPLIT, bool EARLY>
__global__ void __launch_bounds__(THREADS, 1) resident_net_kernel(const __grid_constant__ NetMaps maps, const NetArgs a) {
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
      mbar_init(&sh.acc_full[k], 1);
      mbar_init(&sh.stored[k], EPI_WARPS);
      mbar_init(&sh.epi_done[k][0], EPI_WARPS);
      mbar_init(&sh.epi_done[k][1], EPI_WARPS);
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
  // waits for work (a gang still forming) last as long as other matrices do
  const unsigned long long idle = lim > kTimeoutNs ? lim : kTimeoutNs;
  const int nk = (a.N + BK - 1) / BK;

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      uint32_t rphase = 0;  // bit c: phase of ready[c]
      bool open0 = true, open1 = a.two_slots != 0, ok = true;
      int last = 1, stage = 0;
      uint32_t phase = 0, seq = 0;
      uint32_t armed[STAGES];
#pragma unroll
      for (int k = 0; k < STAGES; ++k) armed[k] = 0;
      for (int k = 0; k < 4; ++k)
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&maps.m[k])) : "memory");
      while (ok && (open0 || open1)) {
        int c = -1;
        const uint64_t w0 = globaltimer();
        for (int spin = 0; c < 0; ++spin) {
          const int o = last ^ 1;
          if ((o ? open1 : open0) && mbar_test(&sh.ready[o], (rphase >> o) & 1u))
            c = o;
          else if ((last ? open1 : open0) && mbar_test(&sh.ready[last], (rphase >> last) & 1u))
            c = last;
          else if ((spin & 63) == 63 && (*abort_flag || globaltimer() - w0 > idle))
            break;
        }
        if (c < 0) {
          ok = false;
          break;
        }
        rphase ^= 1u << c;
        last = c;
        const volatile Slot& s = sh.slot[c];
        if (s.closed) {
          (c ? open1 : open0) = false;
          continue;
        }
        const int b = s.b, I = s.I, J = s.J;
        const uint32_t cur = EARLY ? ((rphase >> c) & 1u) ^ 1u : 0u;  // (toggled above)
        const bool adj = s.op[cur].kind != 0;
        const int by = s.op[cur].y * a.batch + b, bg = s.op[cur].g * a.batch + b;
        if (a.per > 1) fence_proxy_async();  // the gang's planes, acquired through ready
        sh.wq[seq % WQ] = c;
        mbar_arrive(&sh.wq_full[seq % WQ]);
        ++seq;
        const CUtensorMap* m = maps.m;
        const bool same = I == J && !adj;  // diagonal tile of a square: one operand serves as both
        const int rowA = I * TB, rowB = J * TB, nkt = adj ? 2 * nk : nk;
        for (int kk = 0; kk < nkt; ++kk) {
          if (!mbar_wait(&sh.empty[stage], phase ^ 1u, abort_flag, lim)) {
            ok = false;
            break;
          }
          uint8_t* dst = smem + stage * STAGE_BYTES;
          mbar_expect_tx(&sh.full[stage], (same ? 1 : 2) * PLANES * HALF_BYTES);
          ++armed[stage];
          // Y G, then G Y
          const bool seg2 = kk >= nk;
          const int k0 = (seg2 ? kk - nk : kk) * BK, ks = k0 / BN;  // super column of this K block
          const int ba = seg2 ? bg : by, bb = adj && !seg2 ? bg : by;
          const bool ta = ks < (I >> 1), tb = ks < (J >> 1);
          load_half(dst, &m[0], &m[2], ta, rowA, k0, ba, &sh.full[stage]);
          if (SPLIT) load_half(dst + HALF_BYTES, &m[1], &m[3], ta, rowA, k0, ba, &sh.full[stage]);
          if (!same) {
            load_half(dst + PLANES * HALF_BYTES, &m[0], &m[2], tb, rowB, k0, bb, &sh.full[stage]);
            if (SPLIT) load_half(dst + 3 * HALF_BYTES, &m[1], &m[3], tb, rowB, k0, bb, &sh.full[stage]);
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
      uint32_t ophase = 0;  // bit c: parity of slot c's operation
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
        const int I = s.I, J = s.J;
        const bool adj = s.op[EARLY ? (ophase >> c) & 1u : 0u].kind != 0, same = I == J && !adj;
        ophase ^= 1u << c;
        const int nkt = adj ? 2 * nk : nk;
        tc_fence_after();
        const uint32_t d = tmem_base + c * SLOT_COLS;
        for (int kk = 0; kk < nkt; ++kk) {
          if (!mbar_wait(&sh.full[stage], phase, abort_flag, lim)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t st = smem_u32(smem + stage * STAGE_BYTES);
          const uint32_t sb = same ? st : st + PLANES * HALF_BYTES;
          const int ks = (kk >= nk ? kk - nk : kk) * BK / BN;
          const bool ta = ks < (I >> 1), tb = ks < (J >> 1);
          const uint32_t idesc = IDESC_T | (ta ? IDESC_A_MN : 0u) | (tb ? IDESC_B_MN : 0u);
#pragma unroll
          for (int u = 0; u < BK / UMMA_K; ++u) {
            const uint32_t oa = ta ? u * 2048u : u * UMMA_K * 2u, ob = tb ? u * 2048u : u * UMMA_K * 2u;
            const uint64_t a0 = ta ? make_desc_mn128(st + oa) : make_desc_sw128(st + oa);
            const uint64_t b0 = tb ? make_desc_mn128(sb + ob) : make_desc_sw128(sb + ob);
            mma_f16_id(d, a0, b0, idesc, (kk > 0 || u > 0) ? 1u : 0u);  // hp hp (plain: hi hi)
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
    if (c == 0 || a.two_slots) control<EARLY>(a, sh, c, lane, idle);
  } else {
    // ------------------------------------------------------------ epilogue
    const int ew = warp - 2, q = warp & 3;
    uint32_t aphase = 0;  // bit c: phase of acc_full[c]
    for (uint32_t seq = 0;; ++seq) {
      if (!__all_sync(0xffffffffu, mbar_wait(&sh.wq_full[seq % WQ], (seq / WQ) & 1u, abort_flag, idle))) break;
      const int c = *(volatile int*)&sh.wq[seq % WQ];
      if (c == WQ_END) break;
      if (!epilogue<SPLIT, EARLY>(a, sh, c, (aphase >> c) & 1u, tmem_base, ew, q, lane, trbuf + ew * (16 * 32), lim)) {
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

// Input of the operations, one warp per row: the operand planes of Y_0 = the
// scaled H (x: NET_INPUT), of a checkpoint less its shift (NET_X), or of the
// adjoint (NET_FULL), from the row's super tile on; FP64 row norms; the whole
// X_0 = Y_0 + alpha_0 I as the first checkpoint; for the CTA pairs' layers Y_0
// itself and the expansion's first readout.  One pass for what took the pairs an
// input layer, a checkpoint copy or the readout's start, and the row norms:
// before an expansion of 64 x 2048 1.24 -> 0.48 ms (2.9 GB, 6.0 TB/s).
__global__ void __launch_bounds__(256) net_input_kernel(const NetInput x) {
  const int m = blockIdx.x, b = m % x.batch, N = x.N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blockIdx.y * 8 + warp;
  if (r >= N) return;
  const float* row = x.in + (long long)m * N * N + (long long)r * N;
  const bool scale = x.from == NET_INPUT;
  const InputScale is = scale ? input_scale(x.ctl[b].e_min, x.ctl[b].e_max, x.shift) : InputScale();
  // the diagonal once per row (FP64 per element would bound the pass)
  float yd = row[r];
  if (scale)
    yd = input_diag(yd, is);
  else if (x.from == NET_X)
    yd = (float)((double)yd + x.add[(long long)(m / x.batch) * x.add_stride + b]);
  auto y0 = [&](float h, int col) { return col == r ? yd : scale ? input_offdiag(h, is) : h; };
  float* out = x.x0 ? x.x0 + (long long)m * N * N + (long long)r * N : nullptr;
  const float xd = x.x0 ? (float)((double)yd + x.alpha0[b]) : 0.f;
  const bool vec = (N & 3) == 0 && ((reinterpret_cast<uintptr_t>(x.in) | reinterpret_cast<uintptr_t>(x.x0) |
                                     reinterpret_cast<uintptr_t>(x.y) | reinterpret_cast<uintptr_t>(x.r)) &
                                    15) == 0;
  const int cs = r & ~(kTcBN - 1);
  float* yrow = x.y ? x.y + (long long)m * N * N + (long long)r * N : nullptr;
  float* rrow = x.r ? x.r + (long long)m * N * N + (long long)r * N : nullptr;
  const float rd = x.r ? (float)((double)x.r_scale * (double)yd + x.r_add[b]) : 0.f;
  auto with_diag = [&](int col, const float(&y)[4], float s, float d) {
    float4 v = make_float4(s * y[0], s * y[1], s * y[2], s * y[3]);
    if (r == col) v.x = d;
    if (r == col + 1) v.y = d;
    if (r == col + 2) v.z = d;
    if (r == col + 3) v.w = d;
    return v;
  };
  const long long po = (long long)m * x.slot_h + (long long)r * x.ld_h;
  const double acc =
      plane_row(row, N, vec, x.vec_norm, y0, cs, x.p0 + po, x.p1 ? x.p1 + po : nullptr, x.lo_scale, lane,
                [&](int col, const float(&y)[4]) {
                  if (col >= N) return;
                  if (out) epi::st4(out + col, with_diag(col, y, 1.f, xd), col, N, vec);
                  if (col < cs) return;
                  if (yrow) epi::st4(yrow + col, make_float4(y[0], y[1], y[2], y[3]), col, N, vec);
                  if (rrow) epi::st4(rrow + col, with_diag(col, y, x.r_scale, rd), col, N, vec);
                });
  if (x.rn) {
    const double sum = warp_sum_d(acc);
    if (lane == 0) x.rn[(long long)m * N + r] = sum;
  }
}

// One thread per matrix walks through its layers: X_n = alpha_n I + Y_n with
// alpha_0 = e_max / (e_max - e_min) (0 without the shift) and alpha_{n+1} = a
// alpha^2 + b alpha + c, Y' = (2 a alpha + b) Y + a Y^2.  On the device so that
// no call waits for the bounds before it can enqueue its layers.
__global__ void net_plan_kernel(const NetPlanArgs a) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x, B = a.batch, L = a.L;
  if (b >= B) return;
  const Ctl& c = a.ctl[b];
  const double lo = c.e_min, hi = c.e_max;
  a.status[b] = c.status < 0 ? c.status : 0;
  if (a.bounds) {
    a.bounds[2 * b] = lo;
    a.bounds[2 * b + 1] = hi;
  }
  LayerParams p;
  memset(&p, 0, sizeof(p));
  p.active = 1;
  if (a.expansion) {
    // S_0 = alpha_0 I + Y_0, Y_0 = -H/w; X_0 = I - S_0 = (1 - alpha_0) I - Y_0
    const double* rc = a.coef + 3 * L;
    double al = 1.0 - hi / (hi - lo);
    a.table[b] = rc[0] * al;  // R_0 = c_0 X_0
    for (int n = 0; n < L; ++n) {
      const double t = a.coef[3 * n], u = a.coef[3 * n + 1], v = a.coef[3 * n + 2];
      const double an = t * al * al + u * al + v;
      p.ca_d = (n == 0 ? -1.0 : 1.0) * (2.0 * t * al + u);
      p.cb_d = t;
      p.ca = (float)p.ca_d;
      p.cb = (float)p.cb_d;
      p.rc_d = rc[n + 1];
      p.rc = (float)rc[n + 1];
      p.alpha_new = an;
      a.lp[(long long)n * B + b] = p;
      al = an;
    }
    return;
  }
  double al = a.shift ? hi / (hi - lo) : 0.0;
  double* minus = a.table + (long long)(L + 1) * B;
  for (int n = 0; n <= L; ++n) {
    a.table[(long long)n * B + b] = al;
    if (a.backward) minus[(long long)n * B + b] = -al;
    if (n == L) break;
    const double ca = a.coef[3 * n], cb = a.coef[3 * n + 1], cc = a.coef[3 * n + 2];
    p.ca_d = 2.0 * ca * al + cb;
    p.cb_d = ca;
    p.ca = (float)p.ca_d;
    p.cb = (float)p.cb_d;
    if (a.backward) {
      // G_n = (2 a_n alpha_n + b_n) G + a_n (Y_n G + G Y_n)
      p.cc_d = 0.0;
      a.lp[(long long)(L + n) * B + b] = p;
    }
    const double an = a.shift ? ca * al * al + cb * al + cc : 0.0;
    p.cc_d = a.shift ? 0.0 : cc;
    p.alpha_out = n == L - 1 ? an : 0.0;
    a.lp[(long long)n * B + b] = p;
    p.alpha_out = 0.0;
    al = an;
  }
}

// Dot products of a layer and matrix: the tiles' in their order, by one warp.
__global__ void net_dots_kernel(const double* __restrict__ tile_dots, int ntiles, int per, double* __restrict__ out) {
  const int n = blockIdx.x, b = blockIdx.y, lane = threadIdx.x;
  const double* td = tile_dots + 3 * ((long long)n * ntiles + (long long)b * per);
  double d0 = 0.0, d1 = 0.0, d2 = 0.0;
  for (int k = lane; k < per; k += 32) {
    d0 += td[3 * k];
    d1 += td[3 * k + 1];
    d2 += td[3 * k + 2];
  }
  d0 = warp_sum_d(d0);
  d1 = warp_sum_d(d1);
  d2 = warp_sum_d(d2);
  if (lane == 0) {
    double* o = out + 3 * ((long long)n * gridDim.y + b);
    o[0] = d0;
    o[1] = d1;
    o[2] = d2;
  }
}

}  // namespace net

cudaError_t launch_net_plan(const NetPlanArgs& a, cudaStream_t st) {
  net::net_plan_kernel<<<(a.batch + 31) / 32, 32, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_net_input(const NetInput& x, int count, cudaStream_t st) {
  net::net_input_kernel<<<dim3(count, (x.N + 7) / 8), 256, 0, st>>>(x);
  return cudaGetLastError();
}

cudaError_t launch_net_dots(const double* tile_dots, int ntiles, int per, int L, int B, double* out, cudaStream_t st) {
  net::net_dots_kernel<<<dim3(L, B), 32, 0, st>>>(tile_dots, ntiles, per, out);
  return cudaGetLastError();
}

cudaError_t launch_resident_net(const NetArgs& a, const NetMaps& maps, bool split, int grid, cudaStream_t st) {
  constexpr int smem = res::OPERAND_BYTES + res::TR_BYTES + (int)sizeof(net::Shared);
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
  if (a.two_slots) return split ? go(net::resident_net_kernel<true, false>) : go(net::resident_net_kernel<false, false>);
  return split ? go(net::resident_net_kernel<true, true>) : go(net::resident_net_kernel<false, true>);
}

}  // namespace sp2
