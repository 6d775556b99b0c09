// C ABI of libsp2.so: argument checks, workspace, launch sequences.
//
// A call of sp2_density_matrix enqueues, on the library stream:
//   K1 Gershgorin bounds -> K2 input layer + split, FP64 row norms of Y_0 and
//   the first control step -> all layers in one cooperative launch, which ends
//   with the solve's last one: the resident kernels (csrc/resident.cu, on the
//   CUDA cores csrc/resident_fp32.cu) up to the sizes whose tiles the chip
//   holds, above them a list of layers on the CTA pairs (csrc/syrk_tc2.cu).
//   Control steps run on the device, so there is no host round trip inside the
//   loop; the two layers after its last one are the refinement of Eq. 15, and
//   the last of them writes D_out.
// Networks and expansions go the same two ways (csrc/resident_net.cu, lists).
// A launch a layer remains for batches with a larger matrix, large FP32 solves,
// SP2_SQUARE_KERNEL=single, and where a cooperative launch is refused.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdlib>
#include <cstdio>
#include <cstddef>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "../../include/sp2.h"
#include "common.cuh"
#include "kernels.h"

using namespace sp2;

namespace {

thread_local std::string t_err;

void set_err(const char* fmt, ...) __attribute__((format(printf, 1, 2)));
void set_err(const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  t_err = buf;
}

#define CK(expr)                                                                      \
  do {                                                                                \
    cudaError_t e_ = (expr);                                                          \
    if (e_ != cudaSuccess) {                                                          \
      set_err("%s failed: %s (%s:%d)", #expr, cudaGetErrorString(e_), __FILE__, __LINE__); \
      return e_ == cudaErrorMemoryAllocation ? SP2_ERR_OOM : SP2_ERR_CUDA;            \
    }                                                                                 \
  } while (0)

#define CKS(expr)                   \
  do {                              \
    sp2_status s_ = (expr);         \
    if (s_ != SP2_OK) return s_;    \
  } while (0)

enum BufId {
  B_HI0, B_LO0, B_HI1, B_LO1, B_Y0, B_Y1, B_CTL, B_TILES, B_TOFF, B_TCNT, B_TPART, B_IDONE,
  B_PART, B_TICKET, B_ERR, B_DPTR, B_NS, B_HS, B_TRACES, B_PARAMS, B_BOUNDS, B_RN, B_PART2,
  B_G, B_SEG, B_GH0, B_GL0, B_GH1, B_GL1, B_DOTS, B_TDOTS, B_PARAMS2, B_NALPHA, B_HP0, B_HP1, B_RNP0, B_RNP1,
  B_READOUT, B_RDIAG, B_SEGP, B_WAVE, B_PACK, B_PLANES0, B_PLANES1, B_OPS, B_TSUMS, B_COUNT
};

struct Buf {
  void* p = nullptr;
  size_t bytes = 0;
};

struct State {
  bool init = false;
  int device = 0;
  cudaStream_t stream = nullptr;
  int precision = SP2_PREC_SPLIT_FP16;
  int lo_scale_exp = 11;
  int shift = 1;
  double eps = 0.0;
  int device_sms = 148;
  int num_sms = 148;  // that the library stream can use (stream_sms)
  int max_pairs = 0;  // CTA pairs that the device can run at the same time (0: not known)
  PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  PFN_cuStreamGetGreenCtx_v12040 stream_green = nullptr;
  PFN_cuGreenCtxGetDevResource_v12040 green_resource = nullptr;
  Buf buf[B_COUNT];
  // word in mapped host memory that a kernel sets when a wait of it ran out, for
  // calls that return before their end (its device address too)
  int *late = nullptr, *late_dev = nullptr;
  // pinned staging for small host<->device transfers
  void* stage = nullptr;
  size_t stage_bytes = 0;
  cudaEvent_t stage_done = nullptr;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  cudaEvent_t lev[SP2_MAX_LAYERS + 1] = {};  // around each layer (squaring + row norms)
  cudaEvent_t lsq[SP2_MAX_LAYERS] = {};      // after each squaring launch
  // cached tile list
  int tiles_key_N = -1, tiles_key_B = -1, tiles_key_kind = -1;
  // squaring kernel of the single-matrix solve: CTA pairs with one M = 256
  // MMA per super tile (default) or single CTAs (SP2_SQUARE_KERNEL=single)
  bool pair_kernel = true;
  // the batched solve's launch sequence as an instantiated CUDA graph, and
  // what was baked into it (SP2_GRAPHS=0 enqueues the launches directly)
  bool use_graphs = true;
  cudaGraphExec_t bgraph = nullptr;
  cudaStream_t cap_stream = nullptr;
  // batched schedule: 0 tuned per batch signature, 1 single CTAs, 2 CTA pairs
  int batched_sched = 0;
  std::map<uint64_t, int> batched_choice;
  std::vector<uint64_t> bgraph_key;
  // injected faults (sp2_set_fault / SP2_FAULT): each fires once
  bool fault_alloc = false, fault_nan = false, fault_stall = false;
  size_t alloc_limit = 0;  // injected: larger workspace requests fail (0: none)
  bool fault_no_coop = false;  // injected: cooperative launches are refused
  // side of the square groups of the tile order (SP2_TILE_GROUP, default 8)
  int tile_group = 8;
  // K stages per epoch of the soft pair synchronisation (SP2_WAVE_SYNC, default
  // 16; 0 = off)
  int wave_sync = 16;
  // with the synchronisation: K walked backwards on alternate waves
  // (SP2_SNAKE=1; off by default)
  int snake = 0;
  // wide units for the single solve (SP2_WIDE: 0 off, 1 on, unset: by wave count)
  int wide = -1;
  unsigned long long wait_ns = 0;  // bound of the squaring kernels' waits (0: 4 s)
};

State g;

sp2_status ws(BufId id, size_t bytes, void** out, bool zero = false) {
  if (g.fault_alloc) {
    g.fault_alloc = false;
    set_err("injected allocation failure (fault alloc_fail): the workspace request of %zu bytes was refused",
            bytes);
    return SP2_ERR_OOM;
  }
  Buf& b = g.buf[id];
  if (bytes == 0) bytes = 16;
  if (b.bytes < bytes) {
    if (b.p) {
      CK(cudaStreamSynchronize(g.stream));
      CK(cudaFree(b.p));
      b.p = nullptr;
      b.bytes = 0;
    }
    const cudaError_t e = g.alloc_limit && bytes > g.alloc_limit ? cudaErrorMemoryAllocation : cudaMalloc(&b.p, bytes);
    if (e != cudaSuccess) {
      cudaGetLastError();  // the next launch's check must not find it
      b.p = nullptr;
      set_err("workspace request of %zu bytes failed: %s", bytes, cudaGetErrorString(e));
      return e == cudaErrorMemoryAllocation ? SP2_ERR_OOM : SP2_ERR_CUDA;
    }
    b.bytes = bytes;
    if (id == B_TILES || id == B_TOFF || id == B_TCNT) g.tiles_key_N = -1;
    zero = true;
  }
  if (zero) CK(cudaMemsetAsync(b.p, 0, b.bytes, g.stream));
  *out = b.p;
  return SP2_OK;
}

sp2_status ws_free(BufId id) {
  Buf& b = g.buf[id];
  if (!b.p) return SP2_OK;
  CK(cudaStreamSynchronize(g.stream));
  CK(cudaFree(b.p));
  b = Buf();
  return SP2_OK;
}

sp2_status staging(size_t bytes, void** out) {
  if (g.stage_done) CK(cudaEventSynchronize(g.stage_done));
  if (g.stage_bytes < bytes) {
    if (g.stage) CK(cudaFreeHost(g.stage));
    g.stage = nullptr;
    CK(cudaMallocHost(&g.stage, bytes));
    g.stage_bytes = bytes;
  }
  *out = g.stage;
  return SP2_OK;
}

sp2_status require_init() {
  if (!g.init) {
    set_err("sp2_init has not been called");
    return SP2_ERR_NOT_INITIALIZED;
  }
  CK(cudaSetDevice(g.device));
  return SP2_OK;
}

inline long long round_up(long long x, long long m) { return (x + m - 1) / m * m; }

// Upper-triangle tile list in grouped order: groups of 8 x 8 block tiles
// are visited upper-triangle first, block tiles row-major inside a group, so
// that the CTAs running at the same time share row panels in L2.
// halves: 0 = one tile per block (FFMA kernel), 1 = both 128-row halves of a
// 256 x 256 super tile unless the second lies past N, 2 = both halves always
// (adjacent; the CTA-pair kernel takes them together), 3 = as 2, grouped in
// units of the two super tiles (I, J), (I, J + 1) of a row inside a group
// (the CTA-pair kernel's wide units); a row's odd last tile gets a null
// partner (I = J = 511: rows past any N, nothing is stored for it).
void build_tiles(int N, int B, int tile, int halves, std::vector<uint32_t>& out, int& per_instance) {
  const int T = (N + tile - 1) / tile;
  const int G = g.tile_group;
  std::vector<uint32_t> one;
  for (int gi = 0; gi < T; gi += G)
    for (int gj = gi; gj < T; gj += G)
      for (int I = gi; I < std::min(gi + G, T); ++I)
        for (int J = std::max(I, gj); J < std::min(gj + G, T); ++J) {
          if (halves == 3) {
            const bool pair = J + 1 < std::min(gj + G, T);
            one.push_back(pack_tile(0, I, J, 0));
            one.push_back(pack_tile(0, I, J, 1));
            one.push_back(pair ? pack_tile(0, I, J + 1, 0) : pack_tile(0, 511, 511, 0));
            one.push_back(pair ? pack_tile(0, I, J + 1, 1) : pack_tile(0, 511, 511, 1));
            if (pair) ++J;
          } else if (halves) {
            one.push_back(pack_tile(0, I, J, 0));
            if (halves == 2 || I * tile + tile / 2 < N) one.push_back(pack_tile(0, I, J, 1));
          } else {
            one.push_back(pack_tile(0, I, J, 0));
          }
        }
  per_instance = (int)one.size();
  out.clear();
  out.reserve((size_t)per_instance * B);
  for (int b = 0; b < B; ++b)
    for (uint32_t t : one) out.push_back(t | ((uint32_t)b << 20));
}

// The injected stall, once.
int take_stall() {
  const int s = g.fault_stall ? 1 : 0;
  g.fault_stall = false;
  return s;
}

bool tc_precision(int p) { return p == SP2_PREC_SPLIT_FP16 || p == SP2_PREC_FP16; }

// Uploads a uniform-size tile list (B instances of size N); kind 0 = FFMA
// tiles, 1 = tensor-core halves, 2 = tensor-core super-tile pairs, 3 = the
// pairs' wide units.
sp2_status upload_tiles(int N, int B, int kind, int* ntiles_out) {
  std::vector<uint32_t> tiles;
  int per = 0;
  build_tiles(N, B, kind ? kTcBN : kSimtB, kind, tiles, per);
  const int nt = (int)tiles.size();
  void *dt, *doff, *dcnt, *dpart, *ddone;
  CKS(ws(B_TILES, nt * sizeof(uint32_t), &dt));
  CKS(ws(B_TOFF, B * sizeof(int), &doff));
  CKS(ws(B_TCNT, B * sizeof(int), &dcnt));
  CKS(ws(B_TPART, 2 * nt * sizeof(double2), &dpart));  // two halves: lists of layers
  CKS(ws(B_IDONE, B * sizeof(unsigned), &ddone, true));
  if (!(g.tiles_key_N == N && g.tiles_key_B == B && g.tiles_key_kind == kind)) {
    size_t bytes = nt * sizeof(uint32_t) + 2 * B * sizeof(int);
    void* h;
    CKS(staging(bytes, &h));
    uint8_t* hp = (uint8_t*)h;
    memcpy(hp, tiles.data(), nt * sizeof(uint32_t));
    int* off = (int*)(hp + nt * sizeof(uint32_t));
    int* cnt = off + B;
    for (int b = 0; b < B; ++b) {
      off[b] = b * per;
      cnt[b] = per;
    }
    CK(cudaMemcpyAsync(dt, hp, nt * sizeof(uint32_t), cudaMemcpyHostToDevice, g.stream));
    CK(cudaMemcpyAsync(doff, off, B * sizeof(int), cudaMemcpyHostToDevice, g.stream));
    CK(cudaMemcpyAsync(dcnt, cnt, B * sizeof(int), cudaMemcpyHostToDevice, g.stream));
    CK(cudaEventRecord(g.stage_done, g.stream));
    g.tiles_key_N = N;
    g.tiles_key_B = B;
    g.tiles_key_kind = kind;
  }
  *ntiles_out = nt;
  return SP2_OK;
}

}  // namespace

namespace sp2 {
void set_error_text(const char* s) { t_err = s; }

bool make_tmap_f16(CUtensorMap* out, const void* base, int cols, int rows, int batch, long long ld, long long slot,
                   int box_k, int box_rows) {
  if (!g.encode) return false;
  cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)batch};
  cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)slot * 2};
  cuuint32_t box[3] = {(cuuint32_t)box_k, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = g.encode(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}
}  // namespace sp2

namespace {

// Tensor maps of a plane pair: p0 = hp = 2^s hi and p1 = lo' for the split
// product, p0 = hi (p1 unused, null) for plain FP16.  {p0, p1} with boxes of 64
// columns x 128 rows, then {p0, p1} with 64 x rows2: the 256 B rows of the
// single-CTA kernel, or (kTransBox) the transposed reads of the K blocks left of
// the diagonal by the kernels that keep upper tiles.
constexpr int kTransBox = 64;
sp2_status tmaps4_for(const void* p0, const void* p1, int N, int B, long long ld_h, long long slot_h, CUtensorMap* m,
                      int rows2 = kTcBN) {
  const void* p1_ = p1 ? p1 : p0;
  const bool ok = make_tmap_f16(&m[0], p0, N, N, B, ld_h, slot_h, 64, kTcBM) &&
                  make_tmap_f16(&m[1], p1_, N, N, B, ld_h, slot_h, 64, kTcBM) &&
                  make_tmap_f16(&m[2], p0, N, N, B, ld_h, slot_h, 64, rows2) &&
                  make_tmap_f16(&m[3], p1_, N, N, B, ld_h, slot_h, 64, rows2);
  if (!ok) {
    set_err("cuTensorMapEncodeTiled failed (N=%d, ld=%lld)", N, ld_h);
    return SP2_ERR_CUDA;
  }
  return SP2_OK;
}

// FP16 operand planes of the single-accumulator kernels in buffer set k
// (0, 1): hp and lo' (split) or hi (plain); the others stay null.
sp2_status planes_for(bool split, int k, size_t bytes, void** hi, void** lo, void** hp) {
  *hi = *lo = *hp = nullptr;
  if (split) {
    CKS(ws(k ? B_LO1 : B_LO0, bytes, lo));
    CKS(ws(k ? B_HP1 : B_HP0, bytes, hp));
  } else {
    CKS(ws(k ? B_HI1 : B_HI0, bytes, hi));
  }
  return SP2_OK;
}

// Row-norm segment sums carried between the single-accumulator launches:
// B instances of up to N rows, ceil(N / 32) segments each.
sp2_status rnp_for(int N, int B, SqArgs& A, void** rnp) {
  A.ld_rnp = round_up(N, 32);
  A.slot_rnp = (long long)((N + 31) / 32) * A.ld_rnp;
  CKS(ws(B_RNP0, (size_t)A.slot_rnp * B * sizeof(float), &rnp[0]));
  CKS(ws(B_RNP1, (size_t)A.slot_rnp * B * sizeof(float), &rnp[1]));
  return SP2_OK;
}

// Launch k of a device-driven loop reads the row norms of its input (the
// FP64 ones of the input layer for k = 0) and writes those of its output.
void rnp_step(SqArgs& A, void** rnp, int k) {
  A.rnp_out = (float*)rnp[k & 1];
  A.rnp_in = k > 0 ? (const float*)rnp[(k - 1) & 1] : nullptr;
}

// Epoch counters of the CTA pairs' soft synchronisation for nlaunch layers
// over a tile list of ntiles entries (two per super tile, every tile active)
// whose tiles have nkt K stages: one zeroed slice of *per counters per
// layer, or none when the synchronisation is off (SP2_WAVE_SYNC=0).
sp2_status wave_counters(int ntiles, int grid, int nkt, int nlaunch, unsigned** wave, size_t* per) {
  *wave = nullptr;
  *per = 0;
  if (g.wave_sync <= 0 || grid < 2) return SP2_OK;
  const int ncl = grid / 2, nsuper = ntiles / 2;
  const long long stages = (long long)((nsuper + ncl - 1) / ncl) * nkt;
  *per = (size_t)(stages / g.wave_sync + 2);
  void* wv;
  CKS(ws(B_WAVE, *per * (size_t)nlaunch * sizeof(unsigned), &wv, true));
  *wave = (unsigned*)wv;
  return SP2_OK;
}

// A pool of operand plane pairs, [entries][B] matrices of size N, for the
// CTA-pair kernel.
struct PlanePool {
  __half *p0 = nullptr, *p1 = nullptr;
  long long ld_h = 0, slot_h = 0, entry = 0;
  CUtensorMap m[4];
  sp2_status init(bool split, int entries, int N, int B) {
    ld_h = round_up(N, 64);
    slot_h = ld_h * N;
    entry = slot_h * B;
    void *a, *b = nullptr;
    CKS(ws(split ? B_HP0 : B_HI0, (size_t)entry * entries * 2, &a));
    if (split) CKS(ws(B_LO0, (size_t)entry * entries * 2, &b));
    p0 = (__half*)a;
    p1 = (__half*)b;
    return tmaps4_for(p0, p1, N, B * entries, ld_h, slot_h, m, kTransBox);
  }
  __half* p0_of(int k) const { return p0 + entry * k; }
  __half* p1_of(int k) const { return p1 ? p1 + entry * k : nullptr; }
};

// The SMs that the library stream can use: a stream of a green context has its
// context's alone.  The kernels whose CTAs wait on one another need all of them
// running at once, so their grids (and which sizes they take) go by this.
void stream_sms() {
  g.num_sms = g.device_sms;
  if (!g.stream_green || !g.green_resource || (uintptr_t)g.stream <= 2) return;  // 0 to 2: the default streams
  CUgreenCtx gc = nullptr;
  CUdevResource r;
  if (g.stream_green((CUstream)g.stream, &gc) == CUDA_SUCCESS && gc &&
      g.green_resource(gc, &r, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS && r.sm.smCount > 0)
    g.num_sms = std::min(g.device_sms, (int)r.sm.smCount);
}

// CTAs of a launch of the pair kernel over ntiles half super tiles (or units).
int pair_grid(int ntiles) {
  int n = std::min(ntiles, g.num_sms);
  if (g.max_pairs > 0) n = std::min(n, 2 * g.max_pairs);
  return std::max(2, n & ~1);
}

// A cooperative launch.  What the device (or the share of it that a service gives
// the process) cannot hold at once is refused with an error that leaves the context
// usable; the caller then takes the launch-per-layer way.
constexpr sp2_status kRefused = (sp2_status)2;  // never returned to the user
template <class F>
cudaError_t coop_launch(F f) {
  return g.fault_no_coop ? cudaErrorCooperativeLaunchTooLarge : f();
}
bool refused(cudaError_t e) {
  if (e != cudaErrorCooperativeLaunchTooLarge) return false;
  cudaGetLastError();
  return true;
}

// A list of layers on the CTA pairs: one cooperative launch, or one launch a layer.
cudaError_t launch_pairs(const SqArgs& a, const PairList& l, bool adjoint, const CUtensorMap* m, bool split, int grid) {
  const cudaError_t e = coop_launch([&] { return launch_syrk_tc2(a, l, adjoint, m, split, grid, g.stream); });
  if (!refused(e)) return e;
  SqArgs b = a;
  b.wave_ctr = nullptr;  // pairs that do not run together do not keep in step
  for (int n = 0; n < l.nops; ++n) {
    PairList one = l;
    one.ops = l.ops + n;
    one.nops = 1;
    one.groups = 0;
    one.cooperative = 0;
    if (l.rec) one.rec = l.rec + n;
    if (l.stamps) one.stamps = l.stamps + n;
    cudaError_t s = cudaMemsetAsync(l.done, 0, sizeof(unsigned) * 2 * l.batch, g.stream);
    if (s == cudaSuccess) s = launch_syrk_tc2(b, one, adjoint, m, split, grid, g.stream);
    if (s != cudaSuccess) return s;
    b.stall = 0;
  }
  return cudaSuccess;
}

// Lists of layers for the CTA-pair kernel (one launch each), their flags and
// records in one device buffer, uploaded with one copy.
struct PairLists {
  std::vector<LayerOp> ops;
  std::vector<int> first;  // first layer of each list
  int B = 1;
  uint8_t* dev = nullptr;
  size_t o_rec = 0, o_stamps = 0, o_ops = 0, bytes = 0;

  void begin() { first.push_back((int)ops.size()); }
  // device buffer for the lists as they are; records of control steps for one list
  sp2_status alloc(int B_, bool ctl) {
    B = B_;
    o_rec = round_up(2 * sizeof(unsigned) * B * first.size(), 64);
    o_stamps = o_rec + (ctl ? (ops.size() + 1) * sizeof(LayerParams) : 0);
    o_ops = o_stamps + (ctl ? (ops.size() + 1) * sizeof(unsigned long long) : 0);
    bytes = o_ops + ops.size() * sizeof(LayerOp);
    void* p;
    CKS(ws(B_OPS, bytes, &p));
    dev = (uint8_t*)p;
    return SP2_OK;
  }
  void fill(void* host) const {
    memset(host, 0, o_ops);
    memcpy((uint8_t*)host + o_ops, ops.data(), ops.size() * sizeof(LayerOp));
  }
  // grouped: all layers of a group of instances before the next group, the
  // smallest groups of at least 1.9 units per pair (an instance's next layer
  // then never waits for its last), so that a group's planes and iterates stay
  // in the 129 MB L2 from layer to layer
  PairList list(int i, bool ctl, bool grouped, int per) const {
    PairList l;
    memset(&l, 0, sizeof(l));
    l.ops = (const LayerOp*)(dev + o_ops) + first[i];
    l.nops = (i + 1 < (int)first.size() ? first[i + 1] : (int)ops.size()) - first[i];
    l.batch = B;
    l.per = per;
    l.cooperative = 1;
    if (grouped) {
      const int need = (int)std::ceil(1.9 * (g.num_sms / 2) / per);
      l.groups = std::max(1, B / std::max(1, need));
    }
    l.done = (unsigned*)dev + (size_t)2 * B * i;
    l.step = l.done + B;
    if (ctl) {
      l.rec = (LayerParams*)(dev + o_rec);
      l.stamps = (unsigned long long*)(dev + o_stamps);
    }
    return l;
  }
};

// The input pass of a list of layers (csrc/resident_net.cu) into plane entry
// `entry` of the pool; FP64 row norms as rownorm_kernel's of a matrix at `norm`.
NetInput pair_input(const PlanePool& pool, int from, const float* in, int entry, int N, int B, const void* norm) {
  NetInput x;
  memset(&x, 0, sizeof(x));
  x.N = N;
  x.batch = B;
  x.from = from;
  x.in = in;
  x.p0 = pool.p0_of(entry);
  x.p1 = pool.p1_of(entry);
  x.ld_h = pool.ld_h;
  x.slot_h = pool.slot_h;
  x.vec_norm = (N & 3) == 0 && ((uintptr_t)norm & 15) == 0;
  x.lo_scale = std::ldexp(1.0f, g.lo_scale_exp);
  return x;
}

// One layer, as SqArgs describes it.
PairList one_layer(int B) {
  PairList l;
  memset(&l, 0, sizeof(l));
  l.nops = 1;
  l.batch = B;
  return l;
}

void init_ctl(Ctl* c, int N, int n_occ, double tol, int max_iter) {
  memset(c, 0, sizeof(Ctl));
  c->N = N;
  c->n_occ = n_occ;
  c->max_iter = max_iter;
  c->shift = g.shift;
  c->tol = tol;
  c->eps = g.eps;
  c->phase = PHASE_LOOP;
  c->status = SP2_OK;
  c->next.active = 1;  // lets the first row-norm launch run the first control step
}

void fill_stats(const Ctl& c, sp2_stats* s, double ms, int precision) {
  memset(s, 0, sizeof(*s));
  s->iterations = c.n;
  s->converged_by = c.converged_by;
  s->status_device = c.status;
  s->n_occ = c.n_occ;
  s->e_min = c.e_min;
  s->e_max = c.e_max;
  s->idemp_err = (c.n >= 1 && c.n <= kMaxL) ? c.iderr[c.n] : 0.0;
  s->trace = c.trace_final;
  s->alpha = c.alpha;
  s->time_ms = ms;
  const double N = (double)c.N;
  const double per = (precision == SP2_PREC_SPLIT_FP16 ? 3.0 : 1.0) * N * N * N;
  s->flops_alg = (c.phase == PHASE_DONE && !c.accel ? (c.n + 2) : c.n) * per;
  for (int k = 0; k < kMaxL; ++k) {
    s->sigma[k] = (k + 1 <= c.n) ? (int8_t)c.sigma[k + 1] : 0;
    s->iderr[k] = (k + 1 <= c.n) ? c.iderr[k + 1] : 0.0;
  }
}

// A time-out found in the call's own error word.
sp2_status timed_out() {
  if (g.late) *(volatile int*)g.late = 0;
  set_err("a bounded device wait timed out");
  return SP2_ERR_DEVICE_TIMEOUT;
}

// One left behind by an earlier call that did not wait for its end: reported once.
sp2_status late_error() {
  if (!g.late || *(volatile int*)g.late == 0) return SP2_OK;
  *(volatile int*)g.late = 0;
  set_err("a bounded device wait timed out in an earlier call, whose outputs are not valid");
  return SP2_ERR_DEVICE_TIMEOUT;
}

sp2_status status_of(const Ctl& c, int dev_err) {
  if (dev_err != 0) return timed_out();
  if (c.status < 0) {
    set_err(c.status == SP2_ERR_NONFINITE      ? "non-finite spectral bounds (NaN or Inf in H)"
            : c.status == SP2_ERR_INVALID_ARG  ? "HOMO/LUMO estimates leave no gap inside the spectral bounds"
                                               : "degenerate spectrum: e_max - e_min <= 0 with 0 < N_occ < N");
    return (sp2_status)c.status;
  }
  if (c.phase != PHASE_DONE) {
    set_err("solve did not finish (phase %d)", c.phase);
    return SP2_ERR_CUDA;
  }
  if (c.converged_by == SP2_STOP_MAXITER) return SP2_NOT_CONVERGED;
  return SP2_OK;
}

// The accelerated solves' check of the caller's estimates (instance >= 0: of a batch).
sp2_status check_estimate(const Ctl& c, sp2_status s, int N_occ, int instance) {
  if (s < 0 || std::fabs(c.trace_final - (double)N_occ) <= 0.5) return s;
  char who[32] = "accelerated solve";
  if (instance >= 0) snprintf(who, sizeof who, "instance %d", instance);
  set_err("%s: Tr D = %.3f but N_occ = %d; the HOMO/LUMO estimates do not bracket the gap", who, c.trace_final, N_occ);
  return SP2_ERR_BAD_ESTIMATE;
}

}  // namespace

extern "C" {

sp2_status sp2_set_fault(const char* spec) {
  t_err.clear();
  bool alloc = false, nan = false, stall = false;
  unsigned long long wait_ns = 0;
  size_t alloc_limit = 0;
  bool no_coop = false;
  const std::string sp = spec ? spec : "";
  size_t pos = 0;
  while (pos <= sp.size()) {
    size_t end = sp.find(',', pos);
    if (end == std::string::npos) end = sp.size();
    const std::string item = sp.substr(pos, end - pos);
    if (item.empty() || item == "none") {
    } else if (item == "alloc_fail") {
      alloc = true;
    } else if (item == "nan_input") {
      nan = true;
    } else if (item == "timeout") {
      stall = true;
    } else if (item == "no_cooperative") {
      no_coop = true;
    } else if (item.compare(0, 12, "alloc_limit=") == 0) {
      char* e = nullptr;
      const long v = std::strtol(item.c_str() + 12, &e, 10);
      if (!e || *e != '\0' || e == item.c_str() + 12 || v < 1 || v > 1000000) {
        set_err("sp2_set_fault: alloc_limit must be an integer in [1, 1000000] MiB, got '%s'", item.c_str() + 12);
        return SP2_ERR_INVALID_ARG;
      }
      alloc_limit = (size_t)v << 20;
    } else if (item.compare(0, 8, "wait_ms=") == 0) {
      char* e = nullptr;
      const long v = std::strtol(item.c_str() + 8, &e, 10);
      if (!e || *e != '\0' || e == item.c_str() + 8 || v < 1 || v > 60000) {
        set_err("sp2_set_fault: wait_ms must be an integer in [1, 60000], got '%s'", item.c_str() + 8);
        return SP2_ERR_INVALID_ARG;
      }
      wait_ns = (unsigned long long)v * 1000000ull;
    } else {
      set_err("sp2_set_fault: unknown item '%s' (alloc_fail, alloc_limit=<n>, nan_input, timeout, no_cooperative, "
              "wait_ms=<n>, none)",
              item.c_str());
      return SP2_ERR_INVALID_ARG;
    }
    pos = end + 1;
  }
  g.fault_alloc = alloc;
  g.alloc_limit = alloc_limit;
  g.fault_no_coop = no_coop;
  g.fault_nan = nan;
  g.fault_stall = stall;
  g.wait_ns = wait_ns;
  return SP2_OK;
}

sp2_status sp2_init(const sp2_config* cfg) {
  t_err.clear();
  if (const char* fs = getenv("SP2_FAULT")) CKS(sp2_set_fault(fs));
  sp2_config c;
  c.device = 0;
  c.stream = nullptr;
  c.precision = SP2_PREC_SPLIT_FP16;
  c.lo_scale_exp = 11;
  c.shift_identity = 1;
  c.eps_bias = 0.0;
  if (cfg) c = *cfg;
  if (c.precision < 0 || c.precision > 2 || c.lo_scale_exp < 0 || c.lo_scale_exp > 14 || !std::isfinite(c.eps_bias) ||
      c.device < 0) {
    set_err("invalid sp2_config field");
    return SP2_ERR_INVALID_ARG;
  }
  int ndev = 0;
  CK(cudaGetDeviceCount(&ndev));
  if (c.device >= ndev) {
    set_err("device %d not present (%d devices)", c.device, ndev);
    return SP2_ERR_INVALID_ARG;
  }
  if (g.init && g.device != c.device) sp2_finalize();
  CK(cudaSetDevice(c.device));
  int major = 0, minor = 0;
  CK(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, c.device));
  CK(cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, c.device));
  if (major != 10) {
    set_err("libsp2 is built for sm_103a (compute capability 10.x); device has %d.%d", major, minor);
    return SP2_ERR_UNSUPPORTED;
  }
  CK(cudaDeviceGetAttribute(&g.device_sms, cudaDevAttrMultiProcessorCount, c.device));
  if (!g.encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    CK(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q));
    if (!fn || q != cudaDriverEntryPointSuccess) {
      set_err("cuTensorMapEncodeTiled not available from the driver");
      return SP2_ERR_UNSUPPORTED;
    }
    g.encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    // (absent from older drivers, which have no green contexts)
    auto optional = [&](const char* name) -> void* {
      void* p = nullptr;
      const bool ok = cudaGetDriverEntryPointByVersion(name, &p, 12040, cudaEnableDefault, &q) == cudaSuccess &&
                      q == cudaDriverEntryPointSuccess;
      if (!ok) cudaGetLastError();
      return ok ? p : nullptr;
    };
    g.stream_green = (PFN_cuStreamGetGreenCtx_v12040)optional("cuStreamGetGreenCtx");
    g.green_resource = (PFN_cuGreenCtxGetDevResource_v12040)optional("cuGreenCtxGetDevResource");
  }
  if (g.max_pairs == 0 || !g.init) g.max_pairs = syrk_tc2_max_pairs();
  if (!g.late) {
    CK(cudaHostAlloc(&g.late, sizeof(int), cudaHostAllocMapped));
    *(volatile int*)g.late = 0;
    CK(cudaHostGetDevicePointer(&g.late_dev, g.late, 0));
  }
  if (!g.stage_done) {
    CK(cudaEventCreateWithFlags(&g.stage_done, cudaEventDisableTiming));
    CK(cudaEventCreate(&g.ev0));
    CK(cudaEventCreate(&g.ev1));
    for (int i = 0; i <= SP2_MAX_LAYERS; ++i) CK(cudaEventCreate(&g.lev[i]));
    for (int i = 0; i < SP2_MAX_LAYERS; ++i) CK(cudaEventCreate(&g.lsq[i]));
  }
  {
    const char* kv = getenv("SP2_SQUARE_KERNEL");
    g.pair_kernel = !(kv && strcmp(kv, "single") == 0);
    const char* bk = getenv("SP2_BATCHED_KERNEL");
    g.batched_sched = (bk && strcmp(bk, "single") == 0) ? 1 : (bk && strcmp(bk, "pairs") == 0) ? 2 : 0;
    const char* gv = getenv("SP2_GRAPHS");
    g.use_graphs = !(gv && strcmp(gv, "0") == 0);
    const char* wsy = getenv("SP2_WAVE_SYNC");
    g.wave_sync = wsy ? std::max(0, std::min(4096, atoi(wsy))) : 16;
    const char* sn = getenv("SP2_SNAKE");
    g.snake = (sn && strcmp(sn, "1") == 0) ? 1 : 0;
    const char* wd = getenv("SP2_WIDE");
    g.wide = wd ? (strcmp(wd, "1") == 0 ? 1 : 0) : -1;
    const char* tg = getenv("SP2_TILE_GROUP");
    const int tgv = tg ? atoi(tg) : 8;
    if (tgv != g.tile_group) g.tiles_key_N = -1;
    g.tile_group = (tgv >= 1 && tgv <= 64) ? tgv : 8;
  }
  g.device = c.device;
  g.stream = (cudaStream_t)c.stream;
  stream_sms();
  g.precision = c.precision;
  g.lo_scale_exp = c.lo_scale_exp;
  g.shift = c.shift_identity ? 1 : 0;
  g.eps = c.eps_bias;
  g.init = true;
  return SP2_OK;
}

sp2_status sp2_finalize(void) {
  if (!g.init) return SP2_OK;
  cudaSetDevice(g.device);
  cudaStreamSynchronize(g.stream);
  for (int i = 0; i < B_COUNT; ++i) {
    if (g.buf[i].p) cudaFree(g.buf[i].p);
    g.buf[i] = Buf();
  }
  if (g.late) cudaFreeHost(g.late);
  g.late = g.late_dev = nullptr;
  if (g.stage) cudaFreeHost(g.stage);
  g.stage = nullptr;
  g.stage_bytes = 0;
  if (g.stage_done) cudaEventDestroy(g.stage_done);
  if (g.ev0) cudaEventDestroy(g.ev0);
  if (g.ev1) cudaEventDestroy(g.ev1);
  g.stage_done = g.ev0 = g.ev1 = nullptr;
  for (int i = 0; i <= SP2_MAX_LAYERS; ++i) {
    if (g.lev[i]) cudaEventDestroy(g.lev[i]);
    g.lev[i] = nullptr;
    if (i < SP2_MAX_LAYERS && g.lsq[i]) cudaEventDestroy(g.lsq[i]);
    if (i < SP2_MAX_LAYERS) g.lsq[i] = nullptr;
  }
  if (g.bgraph) cudaGraphExecDestroy(g.bgraph);
  g.bgraph = nullptr;
  if (g.cap_stream) cudaStreamDestroy(g.cap_stream);
  g.cap_stream = nullptr;
  g.bgraph_key.clear();
  g.tiles_key_N = -1;
  g.init = false;
  return SP2_OK;
}

sp2_status sp2_set_stream(void* stream) {
  CKS(require_init());
  g.stream = (cudaStream_t)stream;
  stream_sms();
  return SP2_OK;
}

sp2_status sp2_set_precision(int precision) {
  CKS(require_init());
  if (precision < 0 || precision > 2) {
    set_err("precision must be 0 (split), 1 (fp16) or 2 (fp32)");
    return SP2_ERR_INVALID_ARG;
  }
  g.precision = precision;
  return SP2_OK;
}

const char* sp2_last_error(void) { return t_err.c_str(); }

sp2_status sp2_gershgorin(const float* H, int N, double* bounds_out) {
  t_err.clear();
  CKS(require_init());
  if (!H || !bounds_out || N < 1 || N > 65536) {
    set_err("sp2_gershgorin: invalid argument");
    return SP2_ERR_INVALID_ARG;
  }
  const int grid = (int)std::min<long long>((N + 7) / 8, 4LL * g.num_sms);
  void *part, *tick, *bnd;
  CKS(ws(B_PART, grid * sizeof(double2), &part));
  CKS(ws(B_TICKET, 64 * sizeof(unsigned), &tick, true));
  CKS(ws(B_BOUNDS, 2 * sizeof(double), &bnd));
  CK(launch_gershgorin(H, N, N, (long long)N * N, 1, (double2*)part, (unsigned*)tick, nullptr, (double*)bnd, grid,
                       g.stream));
  CK(cudaMemcpyAsync(bounds_out, bnd, 2 * sizeof(double), cudaMemcpyDeviceToHost, g.stream));
  CK(cudaStreamSynchronize(g.stream));
  return SP2_OK;
}

sp2_status sp2_split(const float* X, int N, int lo_scale_exp, uint16_t* hi, uint16_t* lo) {
  t_err.clear();
  CKS(require_init());
  if (!X || !hi || !lo || N < 1 || N > 65536 || lo_scale_exp < 0 || lo_scale_exp > 14) {
    set_err("sp2_split: invalid argument");
    return SP2_ERR_INVALID_ARG;
  }
  const long long n = (long long)N * N;
  const int grid = (int)std::min<long long>((n + 255) / 256, 8LL * g.num_sms);
  CK(launch_split(X, n, std::ldexp(1.0f, lo_scale_exp), (__half*)hi, (__half*)lo, grid, g.stream));
  return SP2_OK;
}

sp2_status sp2_observable(const float* D, const float* A, int N, double* out) {
  t_err.clear();
  CKS(require_init());
  if (!D || !A || !out || N < 1 || N > 65536) {
    set_err("sp2_observable: invalid argument");
    return SP2_ERR_INVALID_ARG;
  }
  const long long n = (long long)N * N;
  const int grid = (int)std::min<long long>((n + 1023) / 1024, 4LL * g.num_sms);
  void* part;
  CKS(ws(B_PART, grid * sizeof(double2), &part));
  CK(launch_observable(D, A, n, (double*)part, grid, g.stream));
  void* h;
  CKS(staging(grid * sizeof(double), &h));
  CK(cudaMemcpyAsync(h, part, grid * sizeof(double), cudaMemcpyDeviceToHost, g.stream));
  CK(cudaStreamSynchronize(g.stream));
  double s = 0.0;
  for (int i = 0; i < grid; ++i) s += ((double*)h)[i];
  *out = s;
  return SP2_OK;
}

sp2_status sp2_layer(const float* X, int B, int N, float a, float b, float c, float* X_out, double* traces_out) {
  t_err.clear();
  CKS(require_init());
  if (!X || !X_out || X == X_out || B < 1 || N < 1 || N > 65536 || (long long)B * N > (1LL << 31) || B > 4096 ||
      !std::isfinite(a) || !std::isfinite(b) || !std::isfinite(c)) {
    set_err("sp2_layer: invalid argument");
    return SP2_ERR_INVALID_ARG;
  }
  CKS(late_error());
  const bool tc = tc_precision(g.precision);
  const bool split = g.precision == SP2_PREC_SPLIT_FP16;
  int ntiles = 0;
  CKS(upload_tiles(N, B, tc ? 1 : 0, &ntiles));
  void *ns, *params, *traces, *err, *dptr;
  CKS(ws(B_NS, B * sizeof(int), &ns));
  CKS(ws(B_PARAMS, sizeof(LayerParams), &params));
  CKS(ws(B_TRACES, 2 * B * sizeof(double), &traces));
  CKS(ws(B_ERR, sizeof(int), &err, true));
  CKS(ws(B_DPTR, B * sizeof(float*), &dptr));
  void* h;
  CKS(staging(B * sizeof(int) + sizeof(LayerParams), &h));
  int* hn = (int*)h;
  for (int i = 0; i < B; ++i) hn[i] = N;
  LayerParams* hp = (LayerParams*)(hn + B);
  memset(hp, 0, sizeof(*hp));
  hp->ca = b;
  hp->cb = a;
  hp->ca_d = b;
  hp->cb_d = a;
  hp->cc_d = c;
  hp->alpha_out = 0.0;
  hp->active = 1;
  hp->out_mode = OUT_Y;
  CK(cudaMemcpyAsync(ns, hn, B * sizeof(int), cudaMemcpyHostToDevice, g.stream));
  CK(cudaMemcpyAsync(params, hp, sizeof(LayerParams), cudaMemcpyHostToDevice, g.stream));
  CK(cudaEventRecord(g.stage_done, g.stream));

  SqArgs A;
  memset(&A, 0, sizeof(A));
  A.wait_ns = g.wait_ns;
  A.Yin = X;
  A.Yout = X_out;
  A.ld_y = N;
  A.slot_y = (long long)N * N;
  A.Dptr = (float* const*)dptr;
  A.Ns = (const int*)ns;
  A.tiles = (const uint32_t*)g.buf[B_TILES].p;
  A.ntiles = ntiles;
  A.tile_off = (const int*)g.buf[B_TOFF].p;
  A.tile_cnt = (const int*)g.buf[B_TCNT].p;
  A.ctl = nullptr;
  A.lp = (const LayerParams*)params;
  A.lp_per_instance = 0;
  A.tile_part = (double2*)g.buf[B_TPART].p;
  A.inst_done = (unsigned*)g.buf[B_IDONE].p;
  A.traces_out = (double*)traces;
  A.lo_scale = std::ldexp(1.0f, g.lo_scale_exp);
  A.lo_unscale = std::ldexp(1.0f, -g.lo_scale_exp);
  A.err = (int*)err;
  A.late = g.late_dev;
  void* rn;
  CKS(ws(B_RN, (size_t)B * N * sizeof(double), &rn));
  const int rgrid = (int)std::min<long long>((N + 7) / 8, std::max(1, 2 * g.num_sms / B));
  CK(launch_rownorm(X, N, (long long)N * N, (const int*)ns, B, N, (double*)rn, N, nullptr, nullptr, nullptr, rgrid,
                    g.stream));
  A.rn = (const double*)rn;
  A.ld_rn = N;
  if (tc) {
    const long long ld_h = round_up(N, 64), slot_h = ld_h * N;
    void *hi, *lo, *hp;
    CKS(planes_for(split, 0, (size_t)slot_h * B * 2, &hi, &lo, &hp));
    const int grid = (int)std::min<long long>((long long)N * B, 8LL * g.num_sms);
    CK(launch_split_pad(X, N, (long long)N * N, N, B, A.lo_scale, (__half*)hi, (__half*)lo, (__half*)hp, ld_h, slot_h, grid,
                        g.stream));
    CUtensorMap m[4];
    CKS(tmaps4_for(split ? hp : hi, lo, N, B, ld_h, slot_h, m));
    A.hi_out = nullptr;
    A.lo_out = nullptr;
    A.hp_out = nullptr;
    A.ld_h = ld_h;
    A.slot_h = slot_h;
    CK(launch_syrk_tc1(A, m, split, std::min(ntiles, g.num_sms), g.stream));
  } else {
    CK(launch_syrk_simt(A, ntiles, g.stream));
  }
  if (traces_out) {
    void* hb;
    CKS(staging(2 * B * sizeof(double) + sizeof(int), &hb));
    CK(cudaMemcpyAsync(hb, traces, 2 * B * sizeof(double), cudaMemcpyDeviceToHost, g.stream));
    CK(cudaMemcpyAsync((char*)hb + 2 * B * sizeof(double), err, sizeof(int), cudaMemcpyDeviceToHost, g.stream));
    CK(cudaStreamSynchronize(g.stream));
    memcpy(traces_out, hb, 2 * B * sizeof(double));
    if (*(int*)((char*)hb + 2 * B * sizeof(double))) return timed_out();
  }
  return SP2_OK;
}

namespace {

// ---- resident solves (csrc/resident.cu) ----

// Tiles of one instance on the resident kernel: the live 128 x 128 tiles of
// the upper 256 x 256 super tiles, in units of 128.
void resident_tiles(int N, int b, std::vector<uint32_t>* out, int* count) {
  const int T = (N + kTcBN - 1) / kTcBN, L = (N + kResTile - 1) / kResTile;
  int n = 0;
  for (int I = 0; I < T; ++I)
    for (int J = I; J < T; ++J)
      for (int i = 2 * I; i < std::min(2 * I + 2, L); ++i)
        for (int j = 2 * J; j < std::min(2 * J + 2, L); ++j) {
          if (out) out->push_back(pack_tile(b, i, j, 0));
          ++n;
        }
  *count = n;
}

// The resident kernel takes a solve whose largest instance has no more tiles
// than the chip has slots (two per SM; N <= 2944 on 152 SMs): below that the
// CTA pairs' 256 x 256 tiles cannot fill the chip (at N = 2048 there are 36
// for 76 pairs) and every layer pays a launch.
bool resident_fits(int Nmax) {
  if (!tc_precision(g.precision) || !g.pair_kernel || g.snake || g.wide == 1) return false;
  if (Nmax > 32 * kResTile) return false;
  int n = 0;
  resident_tiles(Nmax, 0, nullptr, &n);
  return n <= 2 * g.num_sms;
}

// Plans the slots' tile lists: instance after instance (largest first) onto
// the run of consecutive CTAs of one slot that is free first, by estimated
// solve times, the first slots before the second ones.  Gangs of like size
// then share their CTAs and take turns: while one's products run the other is
// in its epilogue and meeting (N = 1024: 17 us of products per layer and pair
// of tiles; unaligned, a gang also waits for its slowest CTA's other tile,
// 28 us per layer), and a gang finds the CTAs of the one before it free
// together.  More tiles than CTAs: the instance takes both slots.
void resident_plan(const int* order, const int* N, const int* toff, const int* tcnt, int B, int grid, int* loff,
                   int* list) {
  std::vector<double> free_at((size_t)2 * grid, 0.0);
  std::vector<int> at(B), deq(grid);
  std::vector<int> count((size_t)2 * grid, 0);
  for (int k = 0; k < B; ++k) {
    const int b = order[k], t = tcnt[b];
    const double time = 2.0 + 1.06 * ((N[b] + 63) / 64);
    int best = 0;
    double start = 0.0;
    if (t > grid) {
      best = -1;
      for (double f : free_at) start = std::max(start, f);
    } else {
      bool found = false;
      for (int c = 0; c < 2; ++c) {
        const double* f = &free_at[(size_t)c * grid];
        // maxima of the windows of t CTAs
        int head = 0, tail = 0;
        for (int x = 0; x < grid; ++x) {
          while (tail > head && f[deq[tail - 1]] <= f[x]) --tail;
          deq[tail++] = x;
          if (deq[head] <= x - t) ++head;
          if (x >= t - 1 && (!found || f[deq[head]] < start)) {
            found = true;
            start = f[deq[head]];
            best = c * grid + x - t + 1;
          }
        }
      }
    }
    at[b] = best;
    for (int i = 0; i < t; ++i) {
      const int sl = best < 0 ? i : best + i;
      free_at[sl] = start + time;
      ++count[sl];
    }
  }
  loff[0] = 0;
  for (int i = 0; i < 2 * grid; ++i) loff[i + 1] = loff[i] + count[i];
  std::vector<int> pos(loff, loff + 2 * grid);
  for (int k = 0; k < B; ++k) {
    const int b = order[k];
    for (int i = 0; i < tcnt[b]; ++i) list[pos[at[b] < 0 ? i : at[b] + i]++] = toff[b] + i;
  }
}

// Device block of one resident call.  One copy uploads it (the zero-start
// counters with it), and its first part is what the host reads back.
struct ResPack {
  size_t ctl, dots, stamps, err, back_bytes;  // read back
  size_t H, D, tiles, toff, tcnt, ns, tickets, bytes;   // uploaded before the prologue
  size_t loff, list, all;                             // uploaded before the resident launch
  ResPack(int B, int nt, int grid) {
    size_t o = 0;
    auto take = [&](size_t n) {
      const size_t at = o;
      o = (o + n + 15) / 16 * 16;
      return at;
    };
    ctl = take((size_t)B * sizeof(Ctl));
    dots = take((size_t)B * 3 * sizeof(double));
    stamps = take((size_t)B * kResStamps * sizeof(unsigned));
    err = take(sizeof(int));
    back_bytes = o;
    H = take((size_t)B * sizeof(void*));
    D = take((size_t)B * sizeof(void*));
    tiles = take((size_t)nt * sizeof(uint32_t));
    toff = take((size_t)B * sizeof(int));
    tcnt = take((size_t)B * sizeof(int));
    ns = take((size_t)B * sizeof(int));
    tickets = take((size_t)2 * B * sizeof(unsigned));
    bytes = o;
    loff = take((size_t)(2 * grid + 1) * sizeof(int));
    list = take((size_t)nt * sizeof(int));
    all = o;
  }
};

// B instances (largest first in the tile list) through the bounds, input-layer
// and resident kernels, then the read-back and the statistics.  single: the
// single-matrix entry points (their bound kernel and row-norm order).
sp2_status resident_solve(const float* const* H, const int* N, const int* N_occ, int B, int Nmax, double tol,
                          int max_iter, float* const* D_out, sp2_stats* stats, const double* homo, const double* lumo,
                          bool single) {
  const bool accel = homo != nullptr;
  const int nlaunch = accel ? max_iter : max_iter + 2;
  const int prec = g.precision;
  const bool split = prec == SP2_PREC_SPLIT_FP16;
  cudaStream_t st = g.stream;

  std::vector<int> order(B);
  for (int i = 0; i < B; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return N[x] > N[y]; });
  std::vector<uint32_t> tiles;
  std::vector<int> toff(B), tcnt(B);
  for (int b : order) {
    toff[b] = (int)tiles.size();
    resident_tiles(N[b], b, &tiles, &tcnt[b]);
  }
  const int nt = (int)tiles.size();
  const int iblocks = (Nmax + 7) / 8;
  const int ggrid = single ? (int)std::min<long long>((Nmax + 7) / 8, 4LL * g.num_sms)
                           : (int)std::min<long long>((Nmax + 7) / 8,
                                                      std::max((Nmax + 63) / 64, 2 * g.num_sms / B + 1));
  const int grid = std::min(nt, g.num_sms);
  const ResPack P(B, nt, grid);
  void *pack, *part, *sums, *rn, *tdots, *tsums;
  CKS(ws(B_PACK, P.all, &pack));
  CKS(ws(B_PART, (size_t)B * std::max(iblocks, ggrid) * sizeof(double2), &part));
  CKS(ws(B_TPART, (size_t)B * 2 * kMeetRows * sizeof(long long), &sums));
  CKS(ws(B_TDOTS, (size_t)nt * sizeof(double), &tdots));
  CKS(ws(B_TSUMS, (size_t)nt * sizeof(double2), &tsums));
  const long long ld_h = round_up(Nmax, 64), slot_h = ld_h * Nmax;
  void *hi[2], *lo[2], *hp[2];
  CKS(planes_for(split, 0, (size_t)slot_h * B * 2, &hi[0], &lo[0], &hp[0]));
  CKS(planes_for(split, 1, (size_t)slot_h * B * 2, &hi[1], &lo[1], &hp[1]));
  CKS(ws(B_RN, (size_t)B * Nmax * sizeof(double), &rn));
  SqArgs carry;
  void* rnp[2];
  CKS(rnp_for(Nmax, B, carry, rnp));

  void* h;
  CKS(staging(P.all, &h));
  uint8_t* hb = (uint8_t*)h;
  memset(hb + P.dots, 0, P.back_bytes - P.dots);
  memset(hb + P.tickets, 0, P.bytes - P.tickets);
  Ctl* hc = (Ctl*)(hb + P.ctl);
  for (int b = 0; b < B; ++b) {
    init_ctl(hc + b, N[b], N_occ[b], tol, max_iter);
    if (accel) {
      hc[b].accel = 1;
      hc[b].acc_homo = homo[b];
      hc[b].acc_lumo = lumo[b];
      hc[b].tol = tol > 0.0 ? tol : 1e-9;
    }
  }
  memcpy(hb + P.H, H, B * sizeof(void*));
  memcpy(hb + P.D, D_out, B * sizeof(void*));
  memcpy(hb + P.tiles, tiles.data(), nt * sizeof(uint32_t));
  memcpy(hb + P.toff, toff.data(), B * sizeof(int));
  memcpy(hb + P.tcnt, tcnt.data(), B * sizeof(int));
  memcpy(hb + P.ns, N, B * sizeof(int));
  // Few instances are planned at once and uploaded with the records (a second copy
  // would stand between the input pass and the layers: N = 1000 686 -> 672 us, 16
  // solves of up to 400 680 -> 663), many while the prologue runs.
  auto plan = [&]() {
    resident_plan(order.data(), N, toff.data(), tcnt.data(), B, grid, (int*)(hb + P.loff), (int*)(hb + P.list));
  };
  const bool plan_first = B <= 32;
  if (plan_first) plan();
  CK(cudaMemcpyAsync(pack, hb, plan_first ? P.all : P.bytes, cudaMemcpyHostToDevice, st));

  uint8_t* dp = (uint8_t*)pack;
  ResArgs A;
  memset(&A, 0, sizeof(A));
  A.H = (const float* const*)(dp + P.H);
  A.D = (float* const*)(dp + P.D);
  A.Ns = (const int*)(dp + P.ns);
  A.tiles = (const uint32_t*)(dp + P.tiles);
  A.ntiles = nt;
  A.tile_off = (const int*)(dp + P.toff);
  A.tile_cnt = (const int*)(dp + P.tcnt);
  A.ctl = (Ctl*)(dp + P.ctl);
  for (int k = 0; k < 2; ++k) {
    A.p0[k] = (__half*)(split ? hp[k] : hi[k]);
    A.p1[k] = (__half*)lo[k];
    A.rnp[k] = (float*)rnp[k];
  }
  A.ld_h = ld_h;
  A.slot_h = slot_h;
  A.rn = (const double*)rn;
  A.ld_rn = Nmax;
  A.ld_rnp = carry.ld_rnp;
  A.slot_rnp = carry.slot_rnp;
  A.part = (double2*)part;
  A.tile_sums = (double2*)tsums;
  A.tile_dots = (double*)tdots;
  A.dots_out = (double*)(dp + P.dots);
  A.sums = (long long*)sums;
  A.tickets = (unsigned*)(dp + P.tickets) + B;
  unsigned* gtick = (unsigned*)(dp + P.tickets);
  A.list_off = (const int*)(dp + P.loff);
  A.list = (const int*)(dp + P.list);
  A.stamps = (unsigned*)(dp + P.stamps);
  A.lo_scale = std::ldexp(1.0f, g.lo_scale_exp);
  A.lo_unscale = std::ldexp(1.0f, -g.lo_scale_exp);
  A.shift = g.shift;
  A.err = (int*)(dp + P.err);
  A.late = g.late_dev;
  A.wait_ns = g.wait_ns;
  A.two_slots = nt > grid ? 1 : 0;
  A.local = Nmax <= kResTile ? 1 : 0;
  A.stall = take_stall();
  ResMaps maps;
  for (int k = 0; k < 2; ++k) {
    CKS(tmaps4_for(A.p0[k], A.p1[k], Nmax, B, ld_h, slot_h, maps.m[k], kTransBox));
  }

  CK(cudaEventRecord(g.ev0, st));
  if (single) {
    CK(launch_gershgorin(H[0], Nmax, Nmax, (long long)Nmax * Nmax, 1, (double2*)part, gtick, A.ctl, nullptr,
                         ggrid, st, g.fault_nan ? 0 : -1));
    g.fault_nan = false;
  } else {
    CK(launch_gershgorin_batched(A.H, A.Ns, A.ctl, B, (double2*)part, gtick, ggrid, st));
  }
  // the row norms of Y_0 in the order of the kernel that the other paths use
  // (float4 rows: always in the batched layout, by N and D in the single one)
  const int vec_norm = !single || ((Nmax & 3) == 0 && ((uintptr_t)D_out[0] & 15) == 0);
  CK(launch_resident_input(A, vec_norm, Nmax, B, st));
  if (!plan_first) {
    plan();
    CK(cudaMemcpyAsync(dp + P.loff, hb + P.loff, P.all - P.loff, cudaMemcpyHostToDevice, st));
  }
  CK(cudaEventRecord(g.stage_done, st));
  CK(cudaEventRecord(g.lev[0], st));
  const cudaError_t le = coop_launch([&] { return launch_resident(A, maps, split, grid, st); });
  if (refused(le)) return kRefused;
  CK(le);
  CK(cudaEventRecord(g.ev1, st));

  if (!stats) return SP2_OK;
  void* back;
  CKS(staging(P.back_bytes, &back));
  CK(cudaMemcpyAsync(back, pack, P.back_bytes, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  const uint8_t* rb = (const uint8_t*)back;
  float ms = 0.f, pro = 0.f;
  CK(cudaEventElapsedTime(&ms, g.ev0, g.ev1));
  CK(cudaEventElapsedTime(&pro, g.ev0, g.lev[0]));
  const Ctl* cs = (const Ctl*)(rb + P.ctl);
  const int e = *(const int*)(rb + P.err);
  sp2_status worst = SP2_OK;
  for (int b = 0; b < B; ++b) {
    sp2_stats& s = stats[b];
    fill_stats(cs[b], &s, ms, prec);
    s.launches = nlaunch;
    s.energy = ((const double*)(rb + P.dots))[3 * b];
    s.prologue_ms = pro;
    // layer times of this instance (0 past its last layer)
    const unsigned* t = (const unsigned*)(rb + P.stamps) + (size_t)b * kResStamps;
    for (int k = 0; k < nlaunch && t[k + 1] != 0; ++k) s.layer_ms[k] = s.square_ms[k] = (float)(t[k + 1] - t[k]) * 1e-6f;
    sp2_status sb = status_of(cs[b], e);
    if (accel) sb = check_estimate(cs[b], sb, N_occ[b], single ? -1 : b);
    if (sb < 0 && worst >= 0) worst = sb;
    if (sb == SP2_NOT_CONVERGED && worst == SP2_OK) worst = SP2_NOT_CONVERGED;
  }
  if (worst == SP2_OK && !single) t_err.clear();
  return worst;
}

// Upper tiles of side ts of an N x N matrix.
long long upper_tiles(int N, int ts) {
  const long long T = (N + ts - 1) / ts;
  return T * (T + 1) / 2;
}

// Tile side of the resident FP32 solve, or 0 for the launch-per-layer kernels:
// by the measured cost of the busiest CTA, about 30 cycles per k and tile of
// side 32, 70 of side 64, against 240 of a wave of 128 x 128 tiles.
int fp32_tile(int N) {
  if (g.precision != SP2_PREC_FP32 || !g.pair_kernel || N > 2048) return 0;
  const long long c32 = 30 * ((upper_tiles(N, 32) + g.num_sms - 1) / g.num_sms);
  const long long c64 = 70 * ((upper_tiles(N, 64) + g.num_sms - 1) / g.num_sms);
  return std::min(c32, c64) > 240 ? 0 : c32 <= c64 ? 32 : 64;
}

// The single FP32 solve on the resident kernel (csrc/resident_fp32.cu).
sp2_status fp32_solve(const float* H, int N, int N_occ, double tol, int max_iter, float* D_out, sp2_stats* stats,
                      bool accel, double homo, double lumo, int tile) {
  cudaStream_t st = g.stream;
  const int T = (N + tile - 1) / tile, nt = (int)upper_tiles(N, tile), grid = std::min(nt, g.num_sms);
  const int nlaunch = accel ? max_iter : max_iter + 2;
  const int ggrid = (int)std::min<long long>((N + 7) / 8, 4LL * g.num_sms);
  const int igrid = (int)std::min<long long>(N, 8LL * g.num_sms);
  const int rgrid = (int)std::min<long long>((N + 7) / 8, 2LL * g.num_sms);
  // one upload: control block, stamps, error word (read back), then pointers,
  // size, tickets, the meeting rows and the tiles
  const size_t o_st = sizeof(Ctl), o_err = o_st + (kResStamps + 2) / 2 * 8, o_ptr = o_err + 16,
               o_sums = o_ptr + 64, o_tiles = o_sums + 3 * kMeetRows * sizeof(long long), bytes = o_tiles + (size_t)nt * sizeof(uint32_t);
  static_assert(sizeof(Ctl) % 8 == 0, "the offsets after it keep 8-byte alignment");
  void *pack, *part, *rn, *slots, *Y[2];
  CKS(ws(B_PACK, bytes, &pack));
  CKS(ws(B_TSUMS, (size_t)grid * sizeof(double2), &slots));
  CKS(ws(B_PART, std::max(std::max(ggrid, igrid), rgrid) * sizeof(double2), &part));
  CKS(ws(B_RN, (size_t)N * sizeof(double), &rn));
  const long long ld_y = round_up(N, 4), slot_y = ld_y * N;
  CKS(ws(B_Y0, (size_t)slot_y * 4, &Y[0]));
  CKS(ws(B_Y1, (size_t)slot_y * 4, &Y[1]));
  void* h;
  CKS(staging(bytes, &h));
  uint8_t* hb = (uint8_t*)h;
  memset(hb, 0, o_tiles);
  Ctl* hc = (Ctl*)hb;
  init_ctl(hc, N, N_occ, tol, max_iter);
  if (accel) {
    hc->accel = 1;
    hc->acc_homo = homo;
    hc->acc_lumo = lumo;
    hc->tol = tol > 0.0 ? tol : 1e-9;
  }
  memcpy(hb + o_ptr, &H, sizeof(void*));
  memcpy(hb + o_ptr + 8, &N, sizeof(int));
  uint32_t* ht = (uint32_t*)(hb + o_tiles);
  for (int I = 0; I < T; ++I)
    for (int J = I; J < T; ++J) *ht++ = pack_tile(0, I, J, 0);
  uint8_t* dp = (uint8_t*)pack;
  CK(cudaMemcpyAsync(dp, hb, bytes, cudaMemcpyHostToDevice, st));
  CK(cudaEventRecord(g.stage_done, st));
  Res32Args A;
  memset(&A, 0, sizeof(A));
  A.Y[0] = (float*)Y[0];
  A.Y[1] = (float*)Y[1];
  A.ld_y = ld_y;
  A.N = N;
  A.D = D_out;
  A.tiles = (const uint32_t*)(dp + o_tiles);
  A.ntiles = nt;
  A.ctl = (Ctl*)dp;
  A.rn = (double*)rn;
  A.sums = (long long*)(dp + o_sums);
  A.slots = (double2*)slots;
  A.stamps = (unsigned*)(dp + o_st);
  A.err = (int*)(dp + o_err);
  A.late = g.late_dev;
  A.wait_ns = g.wait_ns;
  const float* const* hp = (const float* const*)(dp + o_ptr);
  const int* np = (const int*)(dp + o_ptr + 8);
  unsigned* tick = (unsigned*)(dp + o_ptr + 16);
  CK(cudaEventRecord(g.ev0, st));
  CK(launch_gershgorin(H, N, N, (long long)N * N, 1, (double2*)part, tick, A.ctl, nullptr, ggrid, st,
                       g.fault_nan ? 0 : -1));
  g.fault_nan = false;
  CK(launch_input_layer(hp, np, N, A.Y[0], ld_y, slot_y, nullptr, nullptr, nullptr, 0, 0, N, N, 0.f, A.ctl, nullptr,
                        (double2*)part, tick, g.shift, 1, 1, igrid, st));
  CK(launch_rownorm(A.Y[0], ld_y, slot_y, np, 1, N, A.rn, N, A.ctl, (double2*)part, tick, rgrid, st));
  CK(cudaEventRecord(g.lev[0], st));
  const cudaError_t le = coop_launch([&] { return launch_resident_fp32(A, tile, grid, st); });
  if (refused(le)) return kRefused;
  CK(le);
  CK(cudaEventRecord(g.ev1, st));
  if (!stats) return SP2_OK;
  void* back;
  CKS(staging(o_ptr, &back));
  CK(cudaMemcpyAsync(back, dp, o_ptr, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  float ms = 0.f, pro = 0.f;
  CK(cudaEventElapsedTime(&ms, g.ev0, g.ev1));
  CK(cudaEventElapsedTime(&pro, g.ev0, g.lev[0]));
  const Ctl& c = *(const Ctl*)back;
  fill_stats(c, stats, ms, SP2_PREC_FP32);
  stats->launches = nlaunch;
  stats->prologue_ms = pro;
  const unsigned* t = (const unsigned*)((const uint8_t*)back + o_st);
  for (int k = 0; k < nlaunch && t[k + 1] != 0; ++k)
    stats->layer_ms[k] = stats->square_ms[k] = (float)(t[k + 1] - t[k]) * 1e-6f;
  const sp2_status rs = status_of(c, *(const int*)((const uint8_t*)back + o_err));
  return accel ? check_estimate(c, rs, N_occ, -1) : rs;
}

// The single-matrix solve; accel selects the accelerated layers (bounds from
// the HOMO/LUMO estimates) instead of the trace rule with refinement.
sp2_status density_matrix_impl(const float* H, int N, int N_occ, double tol, int max_iter, float* D_out,
                               sp2_stats* stats, bool accel, double homo, double lumo) {
  sp2_status res = kRefused;
  if (resident_fits(N))
    res = resident_solve(&H, &N, &N_occ, 1, N, tol, max_iter, &D_out, stats, accel ? &homo : nullptr,
                         accel ? &lumo : nullptr, true);
  else if (const int tile = fp32_tile(N))
    res = fp32_solve(H, N, N_occ, tol, max_iter, D_out, stats, accel, homo, lumo, tile);
  if (res != kRefused) return res;
  const int prec = g.precision;
  const bool tc = tc_precision(prec);
  const bool split = prec == SP2_PREC_SPLIT_FP16;
  cudaStream_t st = g.stream;

  // CTA pairs on wide units (two super tiles of a row per pass, a quarter
  // fewer operand bytes) by the waves of 76 pairs, counted in super-tile times
  // (SP2_WIDE=0/1 forces it).  Split products: at large N where it takes no more
  // waves (power bound: N = 16384 358 -> 348 ms; its epilogue no longer overlaps
  // the next unit: 4096 6.57 -> 6.74).  Plain FP16 products are bound by the
  // operand bytes, and a wave of wide units takes 0.82 of two waves of single
  // ones: N = 3000 3.03 -> 2.63 ms, 4096 3.74 -> 3.21, 6500 12.4 -> 12.0, 16384
  // 157 -> 135, but 5000 (3 against 4 waves) 6.15 -> 6.62.
  bool wide = false;
  if (tc && g.pair_kernel && g.wide != 0) {
    const int T = (N + kTcBN - 1) / kTcBN, npairs = std::max(1, g.num_sms / 2);
    const int nsup = T * (T + 1) / 2;
    std::vector<uint32_t> wl;
    int per = 0;
    build_tiles(N, 1, kTcBN, 3, wl, per);
    const int nunits = per / 4;
    const int waves = (nsup + npairs - 1) / npairs, waves_w = 2 * ((nunits + npairs - 1) / npairs);
    wide = g.wide == 1 || (split ? N >= 8192 && waves_w <= waves : 0.82 * waves_w < waves);
  }
  int ntiles = 0;
  CKS(upload_tiles(N, 1, tc ? (g.pair_kernel ? (wide ? 3 : 2) : 1) : 0, &ntiles));
  void *ctl, *ns, *hs, *dptr, *err, *part, *tick;
  CKS(ws(B_CTL, sizeof(Ctl), &ctl));
  CKS(ws(B_NS, sizeof(int), &ns));
  CKS(ws(B_HS, sizeof(float*), &hs));
  CKS(ws(B_DPTR, sizeof(float*), &dptr));
  CKS(ws(B_ERR, sizeof(int), &err, true));
  const int ggrid = (int)std::min<long long>((N + 7) / 8, 4LL * g.num_sms);
  const int igrid = (int)std::min<long long>(N, 8LL * g.num_sms);
  const int rgrid = (int)std::min<long long>((N + 7) / 8, 2LL * g.num_sms);
  CKS(ws(B_PART, std::max(std::max(ggrid, igrid), rgrid) * sizeof(double2), &part));
  CKS(ws(B_TICKET, 64 * sizeof(unsigned), &tick, true));
  void* rn;
  CKS(ws(B_RN, (size_t)N * sizeof(double), &rn));
  // Tr[D H] from the launch that writes D: per-tile partials, then the sum
  void *tdots, *dots;
  CKS(ws(B_TDOTS, (size_t)ntiles * 2 * 3 * sizeof(double), &tdots));
  CKS(ws(B_DOTS, 3 * sizeof(double), &dots, true));
  const bool pairs = tc && g.pair_kernel;
  // launches enqueued (CTA pairs: layers of the list): the loop's layers plus the
  // two of Eq. 15 (the accelerated solve has no refinement layers)
  const int nlaunch = accel ? max_iter : max_iter + 2;
  SqArgs A;
  memset(&A, 0, sizeof(A));
  PlanePool pool;
  PairLists lists;
  void* rnp[2];
  if (tc) CKS(rnp_for(N, 1, A, rnp));
  if (pairs) {
    CKS(pool.init(split, 2, N, 1));
    lists.begin();
    for (int k = 0; k < nlaunch; ++k) {
      LayerOp o;
      memset(&o, 0, sizeof(o));
      o.y = k & 1;
      o.g = -1;
      o.tri_y = 1;  // between layers only the upper triangle of Y' is kept
      o.Yin = o.Yout = D_out;
      o.p0_out = pool.p0_of((k & 1) ^ 1);
      o.p1_out = pool.p1_of((k & 1) ^ 1);
      o.rn = (const double*)rn;
      o.rnp_out = (float*)rnp[k & 1];
      o.rnp_in = k ? (const float*)rnp[(k - 1) & 1] : nullptr;
      o.dots_out = (double*)dots;
      lists.ops.push_back(o);
    }
    CKS(lists.alloc(1, true));
  }

  // small per-call records through pinned staging
  void* h;
  const size_t rec_bytes = round_up(sizeof(Ctl) + 64, 64);
  CKS(staging(rec_bytes + lists.bytes, &h));
  Ctl* hc = (Ctl*)h;
  init_ctl(hc, N, N_occ, tol, max_iter);
  if (accel) {
    hc->accel = 1;
    hc->acc_homo = homo;
    hc->acc_lumo = lumo;
    hc->tol = tol > 0.0 ? tol : 1e-9;
  }
  int* hn = (int*)(hc + 1);
  hn[0] = N;
  const float** hh = (const float**)(hn + 2);
  hh[0] = H;
  float** hd = (float**)(hh + 1);
  hd[0] = D_out;
  CK(cudaMemcpyAsync(ctl, hc, sizeof(Ctl), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(ns, hn, sizeof(int), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(hs, hh, sizeof(float*), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(dptr, hd, sizeof(float*), cudaMemcpyHostToDevice, st));
  if (pairs) {
    lists.fill((uint8_t*)h + rec_bytes);
    CK(cudaMemcpyAsync(lists.dev, (uint8_t*)h + rec_bytes, lists.bytes, cudaMemcpyHostToDevice, st));
  }
  CK(cudaEventRecord(g.stage_done, st));

  A.wait_ns = g.wait_ns;
  A.Dptr = (float* const*)dptr;
  A.Ns = (const int*)ns;
  A.tiles = (const uint32_t*)g.buf[B_TILES].p;
  A.ntiles = ntiles;
  A.tile_off = (const int*)g.buf[B_TOFF].p;
  A.tile_cnt = (const int*)g.buf[B_TCNT].p;
  A.ctl = (Ctl*)ctl;
  A.lp = nullptr;
  A.tile_part = (double2*)g.buf[B_TPART].p;
  A.inst_done = (unsigned*)g.buf[B_IDONE].p;
  A.traces_out = nullptr;
  A.lo_scale = std::ldexp(1.0f, g.lo_scale_exp);
  A.lo_unscale = std::ldexp(1.0f, -g.lo_scale_exp);
  A.err = (int*)err;
  A.late = g.late_dev;
  A.rn = (const double*)rn;
  A.ld_rn = N;
  if (tc) {
    A.Hobs = (const float* const*)hs;
    A.tile_dots = (double*)tdots;
    A.dots_out = (double*)dots;
  }

  CK(cudaEventRecord(g.ev0, st));
  CK(launch_gershgorin(H, N, N, (long long)N * N, 1, (double2*)part, (unsigned*)tick, (Ctl*)ctl, nullptr, ggrid, st,
                       g.fault_nan ? 0 : -1));
  g.fault_nan = false;

  if (tc) {
    const long long ld_h = round_up(N, 64), slot_h = ld_h * N;
    void *hi[2] = {}, *lo[2] = {}, *hp[2] = {};
    CUtensorMap m[2][4];
    if (pairs) {
      (split ? hp[0] : hi[0]) = pool.p0;
      lo[0] = pool.p1;
    } else {
      for (int k = 0; k < 2; ++k) {
        CKS(planes_for(split, k, (size_t)slot_h * 2, &hi[k], &lo[k], &hp[k]));
        CKS(tmaps4_for(split ? hp[k] : hi[k], lo[k], N, 1, ld_h, slot_h, m[k]));
      }
    }
    // K2: Y_0 into D_out, split into buffer 0
    // Buffers hold N rows of ld_h columns; the tensor maps declare N x N, so
    // TMA zero-fills every element outside the matrix.
    CK(launch_input_layer((const float* const*)hs, (const int*)ns, N, D_out, N, (long long)N * N, (__half*)hi[0],
                          (__half*)lo[0], (__half*)hp[0], ld_h, slot_h, N, (int)ld_h, A.lo_scale, (Ctl*)ctl, nullptr,
                          (double2*)part, (unsigned*)tick, g.shift, 1, 1, igrid, st));
    // FP64 row norms of Y_0 and the first control step (sigma_1, IdErr_1)
    CK(launch_rownorm(D_out, N, (long long)N * N, (const int*)ns, 1, N, (double*)rn, N, (Ctl*)ctl, (double2*)part,
                      (unsigned*)tick, rgrid, st));
    A.Yin = D_out;
    A.Yout = D_out;
    A.ld_y = N;
    A.slot_y = (long long)N * N;
    A.ld_h = ld_h;
    A.slot_h = slot_h;
    // the epilogue leaves the row norms of Y' for the next layer and the last
    // tile runs the control step
    A.fused_ctl = 1;
    A.tri_y = 1;  // between layers only the upper triangle of Y' is kept
    CK(cudaEventRecord(g.lev[0], st));
    if (pairs) {
      // All layers in one launch.  With a launch each (N = 4096: 145 us a layer),
      // the 58 launches after convergence took 8.9 us apiece and every layer its
      // launch, fill and control step.
      PairList l = lists.list(0, true, false, 0);
      A.tri_planes = 1;
      A.wide = wide ? 1 : 0;
      A.stall = take_stall();
      const int grid = pair_grid(wide ? ntiles / 2 : ntiles);  // every pair has a unit
      // epoch counters of the soft pair synchronisation, one zeroed slice per
      // layer (per pair: super tiles, or wide units of two)
      // where it pays: split products with operand planes beyond L2 (N = 12000 143.6
      // -> 142.8 ms, 16384 361 -> 348; 5000 11.4 -> 11.7).  Plain FP16 stages are a
      // third as long and lose more in step than they save: 8192 20.3 -> 23.9 ms.
      unsigned* wave = nullptr;
      size_t per = 0;
      if (split && N >= 6144) CKS(wave_counters(ntiles, grid, (N + 63) / 64, nlaunch, &wave, &per));
      A.wave_ctr = wave;
      l.wave_per = (int)per;
      A.sync_stages = g.wave_sync;
      A.snake = g.wave_sync > 0 ? g.snake : 0;
      CK(launch_pairs(A, l, false, pool.m, split, grid));
    } else {
      const int grid = std::min(ntiles, g.num_sms);
      for (int k = 0; k < nlaunch; ++k) {
        const int cur = k & 1;
        A.hi_out = (__half*)hi[cur ^ 1];
        A.lo_out = (__half*)lo[cur ^ 1];
        A.hp_out = (__half*)hp[cur ^ 1];
        rnp_step(A, rnp, k);
        A.stall = take_stall();
        CK(launch_syrk_tc1(A, m[cur], split, grid, st));
        CK(cudaEventRecord(g.lsq[k], st));
        CK(cudaEventRecord(g.lev[k + 1], st));
      }
    }
  } else {
    const long long ld_y = round_up(N, 4), slot_y = ld_y * N;
    void* Y[2];
    CKS(ws(B_Y0, (size_t)slot_y * 4, &Y[0]));
    CKS(ws(B_Y1, (size_t)slot_y * 4, &Y[1]));
    CK(launch_input_layer((const float* const*)hs, (const int*)ns, N, (float*)Y[0], ld_y, slot_y, nullptr, nullptr, nullptr, 0,
                          0, N, N, A.lo_scale, (Ctl*)ctl, nullptr, (double2*)part, (unsigned*)tick, g.shift, 1, 1, igrid,
                          st));
    CK(launch_rownorm((float*)Y[0], ld_y, slot_y, (const int*)ns, 1, N, (double*)rn, N, (Ctl*)ctl, (double2*)part,
                      (unsigned*)tick, rgrid, st));
    A.ld_y = ld_y;
    A.slot_y = slot_y;
    CK(cudaEventRecord(g.lev[0], st));
    for (int k = 0; k < nlaunch; ++k) {
      const int cur = k & 1;
      A.Yin = (float*)Y[cur];
      A.Yout = (float*)Y[cur ^ 1];
      CK(launch_syrk_simt(A, ntiles, st));
      CK(cudaEventRecord(g.lsq[k], st));
      CK(launch_rownorm((float*)Y[cur ^ 1], ld_y, slot_y, (const int*)ns, 1, N, (double*)rn, N, (Ctl*)ctl,
                        (double2*)part, (unsigned*)tick, rgrid, st));
      CK(cudaEventRecord(g.lev[k + 1], st));
    }
  }
  CK(cudaEventRecord(g.ev1, st));

  if (!stats) return SP2_OK;
  void* hb;
  const size_t stamp_bytes = pairs ? (nlaunch + 1) * sizeof(unsigned long long) : 0;
  CKS(staging(rec_bytes + stamp_bytes, &hb));
  CK(cudaMemcpyAsync(hb, ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync((char*)hb + sizeof(Ctl), err, sizeof(int), cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync((char*)hb + sizeof(Ctl) + 16, dots, sizeof(double), cudaMemcpyDeviceToHost, st));
  if (pairs)
    CK(cudaMemcpyAsync((char*)hb + rec_bytes, lists.dev + lists.o_stamps, stamp_bytes, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  float ms = 0.f;
  CK(cudaEventElapsedTime(&ms, g.ev0, g.ev1));
  const Ctl& c = *(const Ctl*)hb;
  const int e = *(const int*)((char*)hb + sizeof(Ctl));
  fill_stats(c, stats, ms, prec);
  stats->launches = nlaunch;
  if (tc) stats->energy = *(const double*)((const char*)hb + sizeof(Ctl) + 16);
  float pm = 0.f;
  CK(cudaEventElapsedTime(&pm, g.ev0, g.lev[0]));
  stats->prologue_ms = pm;
  const unsigned long long* t = (const unsigned long long*)((const char*)hb + rec_bytes);
  for (int k = 0; k < nlaunch; ++k) {
    float lm = 0.f, sm = 0.f;
    if (pairs) {
      if (t[k + 1]) lm = sm = (float)(t[k + 1] - t[k]) * 1e-6f;  // 0 past the last layer
    } else {
      CK(cudaEventElapsedTime(&lm, g.lev[k], g.lev[k + 1]));
      CK(cudaEventElapsedTime(&sm, g.lev[k], g.lsq[k]));
    }
    stats->layer_ms[k] = lm;
    stats->square_ms[k] = sm;
  }
  const sp2_status rs = status_of(c, e);
  return accel ? check_estimate(c, rs, N_occ, -1) : rs;
}

}  // namespace

sp2_status sp2_density_matrix(const float* H, int N, int N_occ, double tol, int max_iter, float* D_out,
                              sp2_stats* stats) {
  t_err.clear();
  CKS(require_init());
  if (!H || !D_out || H == D_out || N < 1 || N > 65536 || N_occ < 0 || N_occ > N || !(tol >= 0.0) ||
      !std::isfinite(tol) || max_iter < 1 || max_iter > SP2_MAX_LAYERS - 3) {
    set_err("sp2_density_matrix: invalid argument");
    return SP2_ERR_INVALID_ARG;
  }
  CKS(late_error());
  return density_matrix_impl(H, N, N_occ, tol, max_iter, D_out, stats, false, 0.0, 0.0);
}

sp2_status sp2_density_matrix_accelerated(const float* H, int N, int N_occ, double homo, double lumo, double tol,
                                          int max_iter, float* D_out, sp2_stats* stats) {
  t_err.clear();
  CKS(require_init());
  if (!H || !D_out || H == D_out || N < 1 || N > 65536 || N_occ < 0 || N_occ > N || !(tol >= 0.0) ||
      !std::isfinite(tol) || max_iter < 1 || max_iter > SP2_MAX_LAYERS - 3 || !std::isfinite(homo) ||
      !std::isfinite(lumo) || !(homo < lumo)) {
    set_err("sp2_density_matrix_accelerated: invalid argument");
    return SP2_ERR_INVALID_ARG;
  }
  CKS(late_error());
  return density_matrix_impl(H, N, N_occ, tol, max_iter, D_out, stats, true, homo, lumo);
}

namespace {

// One batched solve on a fixed schedule (pairs: the CTA-pair squaring kernel
// on super-tile pairs, else single CTAs on 128 x 256 tiles), enqueued on the
// library stream; arguments checked by the caller.
sp2_status batched_once(const float* const* H, const int* N, const int* N_occ, int B, int Nmax, double tol,
                        int max_iter, float* const* D_out, bool pairs, const double* homo, const double* lumo) {
  const bool accel = homo != nullptr;
  // launches per solve: the loop plus the two of Eq. 15 (none after the
  // accelerated layers)
  const int nlaunch = accel ? max_iter : max_iter + 2;
  const int prec = g.precision;
  const bool tc = tc_precision(prec);
  const bool split = prec == SP2_PREC_SPLIT_FP16;
  cudaStream_t st = g.stream;
  pairs = pairs && tc;

  // Tile list: instances by decreasing size (largest work first), the tiles
  // of one instance contiguous (its control step sums them in order).
  std::vector<int> order(B);
  for (int i = 0; i < B; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return N[x] > N[y]; });
  std::vector<uint32_t> tiles;
  std::vector<int> toff(B), tcnt(B);
  const int tile = tc ? kTcBN : kSimtB;
  for (int b : order) {
    std::vector<uint32_t> one;
    int per = 0;
    build_tiles(N[b], 1, tile, tc ? (pairs ? 2 : 1) : 0, one, per);
    toff[b] = (int)tiles.size();
    tcnt[b] = per;
    for (uint32_t t : one) tiles.push_back(t | ((uint32_t)b << 20));
  }
  const int nt = (int)tiles.size();
  g.tiles_key_N = -1;  // the single-size cache no longer matches the device list

  void *dt, *doff, *dcnt, *dpart, *ddone, *ctl, *ns, *hs, *dptr, *err, *part, *tick, *rn;
  CKS(ws(B_TILES, nt * sizeof(uint32_t), &dt));
  CKS(ws(B_TOFF, B * sizeof(int), &doff));
  CKS(ws(B_TCNT, B * sizeof(int), &dcnt));
  CKS(ws(B_TPART, nt * sizeof(double2), &dpart));
  CKS(ws(B_IDONE, B * sizeof(unsigned), &ddone, true));
  CKS(ws(B_CTL, B * sizeof(Ctl), &ctl));
  CKS(ws(B_NS, B * sizeof(int), &ns));
  CKS(ws(B_HS, B * sizeof(float*), &hs));
  CKS(ws(B_DPTR, B * sizeof(float*), &dptr));
  CKS(ws(B_ERR, sizeof(int), &err, true));
  // per-instance grids: at most 16 rows per block for the input layer and 8
  // rows per warp for the row norms and bounds
  const int igrid = (int)std::min<long long>(Nmax, std::max((Nmax + 15) / 16, 8 * g.num_sms / B + 1));
  const int rgrid = (int)std::min<long long>((Nmax + 7) / 8, std::max((Nmax + 63) / 64, 2 * g.num_sms / B + 1));
  const int ggrid = rgrid;
  CKS(ws(B_PART, (size_t)B * std::max(igrid, rgrid) * sizeof(double2), &part));
  CKS(ws(B_TICKET, std::max(64, B) * sizeof(unsigned), &tick, true));
  CKS(ws(B_RN, (size_t)B * Nmax * sizeof(double), &rn));
  void *tdots, *dots;
  CKS(ws(B_TDOTS, (size_t)nt * 3 * sizeof(double), &tdots));
  CKS(ws(B_DOTS, (size_t)B * 3 * sizeof(double), &dots, true));

  // per-call records through pinned staging
  const size_t bytes = (size_t)B * sizeof(Ctl) + nt * sizeof(uint32_t) + 2 * B * sizeof(int) + B * sizeof(int) +
                       2 * B * sizeof(void*) + 64;
  void* h;
  CKS(staging(bytes, &h));
  uint8_t* hbuf = (uint8_t*)h;
  Ctl* hc = (Ctl*)hbuf;
  for (int b = 0; b < B; ++b) {
    init_ctl(hc + b, N[b], N_occ[b], tol, max_iter);
    if (accel) {
      hc[b].accel = 1;
      hc[b].acc_homo = homo[b];
      hc[b].acc_lumo = lumo[b];
      hc[b].tol = tol > 0.0 ? tol : 1e-9;
    }
  }
  const void** hh = (const void**)(hc + B);
  void** hd = (void**)(hh + B);
  uint32_t* ht = (uint32_t*)(hd + B);
  int* hoff = (int*)(ht + nt);
  int* hcnt = hoff + B;
  int* hn = hcnt + B;
  for (int b = 0; b < B; ++b) {
    hh[b] = H[b];
    hd[b] = D_out[b];
    hoff[b] = toff[b];
    hcnt[b] = tcnt[b];
    hn[b] = N[b];
  }
  memcpy(ht, tiles.data(), nt * sizeof(uint32_t));
  CK(cudaMemcpyAsync(ctl, hc, B * sizeof(Ctl), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(hs, hh, B * sizeof(void*), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(dptr, hd, B * sizeof(void*), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(dt, ht, nt * sizeof(uint32_t), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(doff, hoff, B * sizeof(int), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(dcnt, hcnt, B * sizeof(int), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(ns, hn, B * sizeof(int), cudaMemcpyHostToDevice, st));
  CK(cudaEventRecord(g.stage_done, st));

  SqArgs A;
  memset(&A, 0, sizeof(A));
  A.wait_ns = g.wait_ns;
  A.Dptr = (float* const*)dptr;
  A.Ns = (const int*)ns;
  A.tiles = (const uint32_t*)dt;
  A.ntiles = nt;
  A.tile_off = (const int*)doff;
  A.tile_cnt = (const int*)dcnt;
  A.ctl = (Ctl*)ctl;
  A.tile_part = (double2*)dpart;
  A.inst_done = (unsigned*)ddone;
  A.rn = (const double*)rn;
  A.ld_rn = Nmax;
  A.lo_scale = std::ldexp(1.0f, g.lo_scale_exp);
  A.lo_unscale = std::ldexp(1.0f, -g.lo_scale_exp);
  A.err = (int*)err;
  A.late = g.late_dev;
  if (tc) {
    // Tr[D H] per instance from the launch that writes D
    A.Hobs = (const float* const*)hs;
    A.tile_dots = (double*)tdots;
    A.dots_out = (double*)dots;
  }

  // workspace and tensor maps first: the launch sequence below makes only
  // stream operations, so it can be captured into a CUDA graph
  const long long ld_y = round_up(Nmax, 4), slot_y = ld_y * Nmax;
  const long long ld_h = round_up(Nmax, 64), slot_h = ld_h * Nmax;
  void* Y[2] = {nullptr, nullptr};
  void *hi[2] = {nullptr, nullptr}, *lo[2] = {nullptr, nullptr}, *hp[2] = {nullptr, nullptr};
  void* rnp[2] = {nullptr, nullptr};
  CUtensorMap m[2][4];
  CKS(ws(B_Y0, (size_t)slot_y * B * 4, &Y[0]));
  if (tc) {
    CKS(planes_for(split, 0, (size_t)slot_h * B * 2, &hi[0], &lo[0], &hp[0]));
    CKS(planes_for(split, 1, (size_t)slot_h * B * 2, &hi[1], &lo[1], &hp[1]));
    for (int k = 0; k < 2; ++k)
      CKS(tmaps4_for(split ? hp[k] : hi[k], lo[k], Nmax, B, ld_h, slot_h, m[k], pairs ? kTransBox : kTcBN));
    CKS(rnp_for(Nmax, B, A, rnp));
    A.Yin = (float*)Y[0];
    A.Yout = (float*)Y[0];
    A.ld_h = ld_h;
    A.slot_h = slot_h;
    A.fused_ctl = 1;
    A.tri_y = 1;  // between launches only the upper triangle of Y' is kept
    A.tri_planes = pairs ? 1 : 0;  // and of the planes, where the kernel reads them so
  } else {
    CKS(ws(B_Y1, (size_t)slot_y * B * 4, &Y[1]));
  }
  A.ld_y = ld_y;
  A.slot_y = slot_y;

  const int stall = take_stall();
  // event records become graph nodes only with the external flag, which is
  // valid during capture alone
  auto enqueue = [&](cudaStream_t st, bool capturing) -> sp2_status {
    const unsigned evf = capturing ? cudaEventRecordExternal : cudaEventRecordDefault;
    CK(cudaEventRecordWithFlags(g.ev0, st, evf));
    CK(launch_gershgorin_batched((const float* const*)hs, (const int*)ns, (Ctl*)ctl, B, (double2*)part,
                                 (unsigned*)tick, ggrid, st));
    if (tc) {
      // Slots are Nmax x Nmax in the tensor maps: everything outside instance
      // b's N_b x N_b block must read as zero.  The input layer zero-fills
      // buffer 0's slot; the epilogues never write outside N_b x N_b (row
      // tails up to the 32-column chunk are written as zeros), so buffer 1 is
      // cleared here.
      for (void* pl : {hi[1], lo[1], hp[1]})
        if (pl) CK(cudaMemsetAsync(pl, 0, (size_t)slot_h * B * 2, st));
      CK(launch_input_layer((const float* const*)hs, (const int*)ns, 0, (float*)Y[0], ld_y, slot_y, (__half*)hi[0],
                            (__half*)lo[0], (__half*)hp[0], ld_h, slot_h, Nmax, (int)ld_h, A.lo_scale, (Ctl*)ctl,
                            nullptr, (double2*)part, (unsigned*)tick, g.shift, 1, B, igrid, st));
      CK(launch_rownorm((float*)Y[0], ld_y, slot_y, (const int*)ns, B, Nmax, (double*)rn, Nmax, (Ctl*)ctl,
                        (double2*)part, (unsigned*)tick, rgrid, st));
      const int grid = pairs ? pair_grid(nt) : std::min(nt, g.num_sms);
      CK(cudaEventRecordWithFlags(g.lev[0], st, evf));
      for (int k = 0; k < nlaunch; ++k) {
        const int cur = k & 1;
        A.hi_out = (__half*)hi[cur ^ 1];
        A.lo_out = (__half*)lo[cur ^ 1];
        A.hp_out = (__half*)hp[cur ^ 1];
        rnp_step(A, rnp, k);
        A.stall = k == 0 ? stall : 0;
        if (pairs)
          CK(launch_syrk_tc2(A, one_layer(B), false, m[cur], split, grid, st));
        else
          CK(launch_syrk_tc1(A, m[cur], split, grid, st));
        CK(cudaEventRecordWithFlags(g.lsq[k], st, evf));
        CK(cudaEventRecordWithFlags(g.lev[k + 1], st, evf));
      }
    } else {
      CK(launch_input_layer((const float* const*)hs, (const int*)ns, 0, (float*)Y[0], ld_y, slot_y, nullptr, nullptr,
                            nullptr, 0, 0, Nmax, Nmax, A.lo_scale, (Ctl*)ctl, nullptr, (double2*)part,
                            (unsigned*)tick, g.shift, 1, B, igrid, st));
      CK(launch_rownorm((float*)Y[0], ld_y, slot_y, (const int*)ns, B, Nmax, (double*)rn, Nmax, (Ctl*)ctl,
                        (double2*)part, (unsigned*)tick, rgrid, st));
      CK(cudaEventRecordWithFlags(g.lev[0], st, evf));
      for (int k = 0; k < nlaunch; ++k) {
        const int cur = k & 1;
        A.Yin = (float*)Y[cur];
        A.Yout = (float*)Y[cur ^ 1];
        CK(launch_syrk_simt(A, std::min(nt, 65535), st));
        CK(cudaEventRecordWithFlags(g.lsq[k], st, evf));
        CK(launch_rownorm((float*)Y[cur ^ 1], ld_y, slot_y, (const int*)ns, B, Nmax, (double*)rn, Nmax, (Ctl*)ctl,
                          (double2*)part, (unsigned*)tick, rgrid, st));
        CK(cudaEventRecordWithFlags(g.lev[k + 1], st, evf));
      }
    }
    CK(cudaEventRecordWithFlags(g.ev1, st, evf));
    return SP2_OK;
  };

  // The whole sequence replays as one CUDA graph while everything baked into
  // it (sizes, grids, wait bound, workspace addresses, stream) is unchanged; the per-call
  // records (control blocks, pointers, tile list) were uploaded above.
  if (g.use_graphs) {
    const uint64_t key[] = {(uint64_t)B, (uint64_t)Nmax, (uint64_t)nt, (uint64_t)nlaunch, (uint64_t)prec, (uint64_t)pairs,
                            (uint64_t)g.shift, (uint64_t)g.lo_scale_exp, (uint64_t)igrid, (uint64_t)rgrid,
                            (uint64_t)ggrid, (uint64_t)g.num_sms, (uint64_t)g.wait_ns, (uint64_t)stall, (uint64_t)(uintptr_t)st,
                            (uint64_t)(uintptr_t)hs, (uint64_t)(uintptr_t)ns, (uint64_t)(uintptr_t)ctl,
                            (uint64_t)(uintptr_t)dt, (uint64_t)(uintptr_t)doff, (uint64_t)(uintptr_t)dcnt,
                            (uint64_t)(uintptr_t)dpart, (uint64_t)(uintptr_t)ddone, (uint64_t)(uintptr_t)err,
                            (uint64_t)(uintptr_t)part, (uint64_t)(uintptr_t)tick, (uint64_t)(uintptr_t)rn,
                            (uint64_t)(uintptr_t)Y[0], (uint64_t)(uintptr_t)Y[1], (uint64_t)(uintptr_t)hi[0],
                            (uint64_t)(uintptr_t)hi[1], (uint64_t)(uintptr_t)lo[0], (uint64_t)(uintptr_t)lo[1],
                            (uint64_t)(uintptr_t)hp[0], (uint64_t)(uintptr_t)hp[1], (uint64_t)(uintptr_t)rnp[0],
                            (uint64_t)(uintptr_t)rnp[1], (uint64_t)(uintptr_t)tdots, (uint64_t)(uintptr_t)dots};
    std::vector<uint64_t> kv(key, key + sizeof(key) / sizeof(key[0]));
    if (!g.bgraph || g.bgraph_key != kv) {
      if (g.bgraph) {
        CK(cudaGraphExecDestroy(g.bgraph));
        g.bgraph = nullptr;
      }
      // captured on the library's own stream (the legacy default stream
      // cannot capture), launched on the caller's
      if (!g.cap_stream) CK(cudaStreamCreateWithFlags(&g.cap_stream, cudaStreamNonBlocking));
      cudaGraph_t graph = nullptr;
      CK(cudaStreamBeginCapture(g.cap_stream, cudaStreamCaptureModeThreadLocal));
      const sp2_status se = enqueue(g.cap_stream, true);
      const cudaError_t ce = cudaStreamEndCapture(g.cap_stream, &graph);
      if (se != SP2_OK) {
        if (graph) cudaGraphDestroy(graph);
        return se;
      }
      CK(ce);
      const cudaError_t ie = cudaGraphInstantiate(&g.bgraph, graph, 0);
      cudaGraphDestroy(graph);
      CK(ie);
      g.bgraph_key = kv;
    }
    CK(cudaGraphLaunch(g.bgraph, st));
  } else {
    CKS(enqueue(st, false));
  }
  return SP2_OK;
}

// Batch signature for the schedule cache: precision and the sorted sizes.
uint64_t batch_signature(const int* N, int B) {
  std::vector<int> v(N, N + B);
  std::sort(v.begin(), v.end());
  uint64_t h = 1469598103934665603ull ^ (uint64_t)g.precision;
  for (int x : v) h = (h ^ (uint64_t)x) * 1099511628211ull;
  return h ^ ((uint64_t)B << 40);
}

}  // namespace

namespace {

sp2_status batched_impl(const float* const* H, const int* N, const int* N_occ, int batch, double tol, int max_iter,
                        float* const* D_out, sp2_stats* stats, const double* homo, const double* lumo) {
  t_err.clear();
  CKS(require_init());
  const bool accel = homo != nullptr;
  const int nlaunch = accel ? max_iter : max_iter + 2;
  if (!H || !N || !N_occ || !D_out || batch < 1 || batch > 4096 || !(tol >= 0.0) || !std::isfinite(tol) ||
      max_iter < 1 || max_iter > SP2_MAX_LAYERS - 3) {
    set_err("sp2_density_matrix_batched: invalid argument");
    return SP2_ERR_INVALID_ARG;
  }
  int Nmax = 0;
  for (int i = 0; i < batch; ++i) {
    if (!H[i] || !D_out[i] || H[i] == D_out[i] || N[i] < 1 || N[i] > 4096 || N_occ[i] < 0 || N_occ[i] > N[i]) {
      set_err("sp2_density_matrix_batched: invalid argument for instance %d", i);
      return SP2_ERR_INVALID_ARG;
    }
    Nmax = std::max(Nmax, N[i]);
  }
  CKS(late_error());
  const int prec = g.precision;
  const bool tc = tc_precision(prec);
  cudaStream_t st = g.stream;
  const int B = batch;

  if (g.batched_sched == 0 && resident_fits(Nmax)) {
    const sp2_status s = resident_solve(H, N, N_occ, B, Nmax, tol, max_iter, D_out, stats, homo, lumo, false);
    if (s != kRefused) return s;
  }

  // schedule: fixed (SP2_BATCHED_KERNEL=single|pairs) or tuned once per batch
  // signature by timing each candidate on the call itself (every candidate
  // run is a complete solve, so the last one leaves valid results)
  bool pairs = g.batched_sched == 2;
  bool solved = false;
  if (tc && g.batched_sched == 0) {
    const uint64_t sig = batch_signature(N, B);
    auto it = g.batched_choice.find(sig);
    if (it != g.batched_choice.end()) {
      pairs = it->second != 0;
    } else {
      float best = 0.f;
      int pick = 0;
      for (int cand = 0; cand < 2; ++cand) {
        CKS(batched_once(H, N, N_occ, B, Nmax, tol, max_iter, D_out, cand != 0, homo, lumo));
        CK(cudaEventSynchronize(g.ev1));
        float ms = 0.f;
        CK(cudaEventElapsedTime(&ms, g.ev0, g.ev1));
        if (cand == 0 || ms < best) {
          best = ms;
          pick = cand;
        }
      }
      g.batched_choice[sig] = pick;
      pairs = pick != 0;
      // the last candidate's run (pairs) is the result when it won
      solved = pick == 1;
    }
  }
  if (!solved) CKS(batched_once(H, N, N_occ, B, Nmax, tol, max_iter, D_out, pairs, homo, lumo));

  if (!stats) return SP2_OK;
  void* ctl = g.buf[B_CTL].p;
  void* err = g.buf[B_ERR].p;

  void* hb;
  const size_t eoff = (size_t)B * sizeof(Ctl) + 16;
  CKS(staging(eoff + (size_t)B * 3 * sizeof(double), &hb));
  CK(cudaMemcpyAsync(hb, ctl, (size_t)B * sizeof(Ctl), cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync((char*)hb + (size_t)B * sizeof(Ctl), err, sizeof(int), cudaMemcpyDeviceToHost, st));
  if (tc) CK(cudaMemcpyAsync((char*)hb + eoff, g.buf[B_DOTS].p, (size_t)B * 3 * sizeof(double),
                             cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  float ms = 0.f;
  CK(cudaEventElapsedTime(&ms, g.ev0, g.ev1));
  const Ctl* cs = (const Ctl*)hb;
  const int e = *(const int*)((char*)hb + (size_t)B * sizeof(Ctl));
  float pro = 0.f, lms[SP2_MAX_LAYERS], sms[SP2_MAX_LAYERS];
  CK(cudaEventElapsedTime(&pro, g.ev0, g.lev[0]));
  for (int k = 0; k < nlaunch; ++k) {
    CK(cudaEventElapsedTime(&lms[k], g.lev[k], g.lev[k + 1]));
    CK(cudaEventElapsedTime(&sms[k], g.lev[k], g.lsq[k]));
  }
  sp2_status worst = SP2_OK;
  for (int b = 0; b < B; ++b) {
    fill_stats(cs[b], &stats[b], ms, prec);
    stats[b].launches = nlaunch;
    if (tc) stats[b].energy = ((const double*)((const char*)hb + eoff))[3 * b];
    stats[b].prologue_ms = pro;
    for (int k = 0; k < nlaunch; ++k) {
      stats[b].layer_ms[k] = lms[k];
      stats[b].square_ms[k] = sms[k];
    }
    sp2_status sb = status_of(cs[b], e);
    if (accel) sb = check_estimate(cs[b], sb, N_occ[b], b);
    if (sb < 0 && worst >= 0) worst = sb;
    if (sb == SP2_NOT_CONVERGED && worst == SP2_OK) worst = SP2_NOT_CONVERGED;
  }
  if (worst == SP2_OK) t_err.clear();
  return worst;
}

}  // namespace

sp2_status sp2_density_matrix_batched(const float* const* H, const int* N, const int* N_occ, int batch, double tol,
                                      int max_iter, float* const* D_out, sp2_stats* stats) {
  return batched_impl(H, N, N_occ, batch, tol, max_iter, D_out, stats, nullptr, nullptr);
}

sp2_status sp2_density_matrix_batched_accelerated(const float* const* H, const int* N, const int* N_occ,
                                                  const double* homo, const double* lumo, int batch, double tol,
                                                  int max_iter, float* const* D_out, sp2_stats* stats) {
  t_err.clear();
  if (!homo || !lumo || batch < 1 || batch > 4096) {
    set_err("sp2_density_matrix_batched_accelerated: invalid argument");
    return SP2_ERR_INVALID_ARG;
  }
  for (int b = 0; b < batch; ++b)
    if (!std::isfinite(homo[b]) || !std::isfinite(lumo[b]) || !(homo[b] < lumo[b])) {
      set_err("sp2_density_matrix_batched_accelerated: invalid estimates for instance %d", b);
      return SP2_ERR_INVALID_ARG;
    }
  return batched_impl(H, N, N_occ, batch, tol, max_iter, D_out, stats, homo, lumo);
}

// Host-side FP64 shift sequence of the network: X_n = alpha_n I + Y_n with
// alpha_0 = e_max/(e_max - e_min) (shift on) and alpha_{n+1} = a alpha^2 +
// b alpha + c; the layer on Y is Y' = (2 a alpha + b) Y + a Y^2.
namespace {
struct NetPlan {
  std::vector<double> alpha;       // [(L+1) * B]
  std::vector<LayerParams> params; // [L * B]
};

sp2_status network_prologue(const float* H, int B, int N, int L, const float* coef, bool* ok, NetPlan& plan,
                            void** ctl_out, void** ns_out, void** hs_out, void** dptr_out, float* X_out) {
  void *ctl, *ns, *hs, *dptr;
  CKS(ws(B_CTL, (size_t)B * sizeof(Ctl), &ctl));
  CKS(ws(B_NS, B * sizeof(int), &ns));
  CKS(ws(B_HS, B * sizeof(float*), &hs));
  CKS(ws(B_DPTR, B * sizeof(float*), &dptr));
  void* h;
  CKS(staging((size_t)B * sizeof(Ctl) + B * (sizeof(int) + 2 * sizeof(void*)) + 64, &h));
  Ctl* hc = (Ctl*)h;
  for (int b = 0; b < B; ++b) init_ctl(hc + b, N, N / 2, 0.0, 1);
  int* hn = (int*)(hc + B);
  const float** hh = (const float**)(hn + B + (B & 1));
  float** hd = (float**)(hh + B);
  for (int b = 0; b < B; ++b) {
    hn[b] = N;
    hh[b] = H + (size_t)b * N * N;
    hd[b] = X_out + (size_t)b * N * N;
  }
  CK(cudaMemcpyAsync(ctl, hc, (size_t)B * sizeof(Ctl), cudaMemcpyHostToDevice, g.stream));
  CK(cudaMemcpyAsync(ns, hn, B * sizeof(int), cudaMemcpyHostToDevice, g.stream));
  CK(cudaMemcpyAsync(hs, hh, B * sizeof(void*), cudaMemcpyHostToDevice, g.stream));
  CK(cudaMemcpyAsync(dptr, hd, B * sizeof(void*), cudaMemcpyHostToDevice, g.stream));
  CK(cudaEventRecord(g.stage_done, g.stream));
  const int ggrid = (int)std::min<long long>((N + 7) / 8, std::max((N + 63) / 64, 2 * g.num_sms / B + 1));
  void *part, *tick;
  CKS(ws(B_PART, (size_t)B * ggrid * sizeof(double2), &part));
  CKS(ws(B_TICKET, std::max(64, B) * sizeof(unsigned), &tick, true));
  CK(launch_gershgorin_batched((const float* const*)hs, (const int*)ns, (Ctl*)ctl, B, (double2*)part, (unsigned*)tick,
                               ggrid, g.stream));
  // bounds to the host: the FP64 shift sequence is planned there
  void* hb;
  CKS(staging((size_t)B * 2 * sizeof(double) + (size_t)B * sizeof(int), &hb));
  CK(cudaMemcpy2DAsync(hb, 2 * sizeof(double), (char*)ctl + offsetof(Ctl, e_min), sizeof(Ctl), 2 * sizeof(double),
                       B, cudaMemcpyDeviceToHost, g.stream));
  CK(cudaMemcpy2DAsync((char*)hb + (size_t)B * 2 * sizeof(double), sizeof(int), (char*)ctl + offsetof(Ctl, status),
                       sizeof(Ctl), sizeof(int), B, cudaMemcpyDeviceToHost, g.stream));
  CK(cudaStreamSynchronize(g.stream));
  const double* bd = (const double*)hb;
  const int* bs = (const int*)((char*)hb + (size_t)B * 2 * sizeof(double));
  plan.alpha.assign((size_t)(L + 1) * B, 0.0);
  plan.params.assign((size_t)L * B, LayerParams());
  *ok = true;
  for (int b = 0; b < B; ++b) {
    if (bs[b] < 0) {
      set_err("instance %d: %s", b, bs[b] == SP2_ERR_NONFINITE ? "non-finite spectral bounds" : "degenerate spectrum");
      *ok = false;
      return (sp2_status)bs[b];
    }
    const double lo = bd[2 * b], hi = bd[2 * b + 1];
    double a = g.shift ? hi / (hi - lo) : 0.0;
    plan.alpha[b] = a;
    for (int n = 0; n < L; ++n) {
      const double ca = coef[3 * n], cb = coef[3 * n + 1], cc = coef[3 * n + 2];
      LayerParams p;
      memset(&p, 0, sizeof(p));
      p.ca_d = 2.0 * ca * a + cb;  // Y' = (2 a alpha + b) Y + a Y^2
      p.cb_d = ca;
      p.cc_d = g.shift ? 0.0 : cc;
      p.ca = (float)p.ca_d;
      p.cb = (float)p.cb_d;
      p.active = 1;
      const double an = g.shift ? ca * a * a + cb * a + cc : 0.0;
      p.out_mode = (n == L - 1) ? OUT_D : OUT_Y;
      p.alpha_out = (n == L - 1) ? an : 0.0;
      plan.params[(size_t)n * B + b] = p;
      a = an;
      plan.alpha[(size_t)(n + 1) * B + b] = a;
    }
  }
  *ctl_out = ctl;
  *ns_out = ns;
  *hs_out = hs;
  *dptr_out = dptr;
  return SP2_OK;
}
}  // namespace

namespace {

// The resident network kernel takes matrices up to n_many in any number, and
// larger ones while each gang has a window of CTAs and a slot of its own, or a
// single one its tiles.  The CTA pairs cannot fill the chip with few matrices
// (backward, 8 layers: 6 of N = 900 719 against 962 us, 4 of 1280 869 against
// 1079, 2 of 2048 1229 against 1322) and pay for the padding of small ones (64 of
// 512 1.40 against 1.65 ms, 48 of 896 3.34 against 3.51); many large ones are
// faster on their 256 x 256 tiles (5 of 1280 1288 against 1127 us, 3 of 1536 1429
// against 1157, 32 of 1024 3.40 against 2.58 ms).  One matrix from N = 2049 to 2816
// is within 8 % on either.  n_many: 896 (24 of 960: forward 945 against 919 us,
// backward 2.35 against 1.99 ms), 1152 for the expansion, whose epilogue reads and
// writes more on the pairs (20 of 1100 1.29 against 1.65 ms; 12 of 1200 1.07
// against 1.08).
bool net_fits(int B, int N, int n_many) {
  if (!resident_fits(N)) return false;
  int n = 0;
  resident_tiles(N, 0, nullptr, &n);
  return N <= n_many || B <= 2 * (g.num_sms / n) || (B == 1 && n <= 2 * g.num_sms);
}

// A run of the resident network kernel (csrc/resident_net.cu) over B matrices
// of size N: the plan of its tiles, the pool of plane pairs, the operations.
// One upload, the bounds, the coefficients (planned on the device), the inputs,
// the layers: nothing waits for the GPU but the check of the bounds, at the end.
struct NetRun {
  int B, N, L, per = 0, nt = 0, grid = 0, pool = 0, ngrid = 0;
  NetArgs A;
  NetMaps maps;
  NetPlanArgs plan;
  std::vector<NetOp> ops;
  std::vector<double> coef;
  uint8_t* pack = nullptr;  // uploaded: [ops][ctl][H][N][tickets][coef][lists][tiles][err]; then [params][table][status]
  size_t o_ctl = 0, o_hs = 0, o_ns = 0, o_tick = 0, o_coef = 0, o_loff = 0, o_list = 0, o_tiles = 0, o_err = 0, up = 0;
  size_t o_params = 0, o_table = 0, o_status = 0, bytes = 0;
  double2* part = nullptr;

  // nops operations, coef set, ntable FP64 values
  sp2_status init(int B_, int N_, int L_, int pool_, bool split, int nops, size_t nparams, size_t ntable) {
    B = B_;
    N = N_;
    L = L_;
    pool = pool_;
    memset(&A, 0, sizeof(A));
    memset(&plan, 0, sizeof(plan));
    resident_tiles(N, 0, nullptr, &per);
    nt = per * B;
    grid = std::min(nt, g.num_sms);
    ngrid = (int)std::min<long long>((N + 7) / 8, std::max((N + 63) / 64, 2 * g.num_sms / B + 1));
    const long long ld_h = round_up(N, 64), slot_h = ld_h * N;
    void *p0, *p1 = nullptr, *sums, *prt;
    CKS(ws(B_PLANES0, (size_t)slot_h * B * pool * 2, &p0));
    if (split) CKS(ws(B_PLANES1, (size_t)slot_h * B * pool * 2, &p1));
    CKS(ws(B_TPART, (size_t)B * kMeetRows * sizeof(long long), &sums));
    CKS(ws(B_PART, (size_t)B * ngrid * sizeof(double2), &prt));
    part = (double2*)prt;
    SqArgs carry;
    void* rnp[2];
    CKS(rnp_for(N, B, carry, rnp));
    size_t o = 0;
    auto take = [&](size_t n) {
      const size_t at = o;
      o = (o + n + 15) / 16 * 16;
      return at;
    };
    take(nops * sizeof(NetOp));
    o_ctl = take((size_t)B * sizeof(Ctl));
    o_hs = take((size_t)B * sizeof(void*));
    o_ns = take((size_t)B * sizeof(int));
    o_tick = take((size_t)B * sizeof(unsigned));
    o_coef = take(coef.size() * sizeof(double));
    o_loff = take((size_t)(2 * grid + 1) * sizeof(int));
    o_list = take((size_t)nt * sizeof(int));
    o_tiles = take((size_t)nt * sizeof(uint32_t));
    o_err = take(sizeof(int));
    up = o;
    o_params = take(nparams * sizeof(LayerParams));
    o_table = take(ntable * sizeof(double));
    o_status = take((size_t)B * sizeof(int));
    bytes = o;
    void* pk;
    CKS(ws(B_PACK, bytes, &pk));
    pack = (uint8_t*)pk;
    A.N = N;
    A.batch = B;
    A.per = per;
    A.ntiles = nt;
    A.ops = (const NetOp*)pack;
    A.lp = (const LayerParams*)(pack + o_params);
    A.ctl = (const Ctl*)(pack + o_ctl);
    A.p0 = (__half*)p0;
    A.p1 = (__half*)p1;
    A.ld_h = ld_h;
    A.slot_h = slot_h;
    A.rnp[0] = (float*)rnp[0];
    A.rnp[1] = (float*)rnp[1];
    A.ld_rnp = carry.ld_rnp;
    A.slot_rnp = carry.slot_rnp;
    A.tiles = (const uint32_t*)(pack + o_tiles);
    A.list_off = (const int*)(pack + o_loff);
    A.list = (const int*)(pack + o_list);
    A.sums = (long long*)sums;
    A.lo_scale = std::ldexp(1.0f, g.lo_scale_exp);
    A.lo_unscale = std::ldexp(1.0f, -g.lo_scale_exp);
    A.shift = g.shift;
    A.two_slots = nt > grid ? 1 : 0;
    A.err = (int*)(pack + o_err);
    A.late = g.late_dev;
    A.wait_ns = g.wait_ns;
    plan.batch = B;
    plan.L = L;
    plan.shift = g.shift;
    plan.coef = (const double*)(pack + o_coef);
    plan.ctl = A.ctl;
    plan.lp = (LayerParams*)(pack + o_params);
    plan.table = (double*)(pack + o_table);
    plan.status = (int*)(pack + o_status);
    return tmaps4_for(p0, p1, N, B * pool, ld_h, slot_h, maps.m, kTransBox);
  }
  const double* dev(size_t table_index) const { return (const double*)(pack + o_table) + table_index; }

  // The records in one upload, the bounds (of H, or the given window) and the
  // plan; `back` receives the statuses after them (check()).
  sp2_status start(const float* H, const double* window, int** back) {
    cudaStream_t st = g.stream;
    A.nops = (int)ops.size();
    void* h;
    CKS(staging(up + (size_t)B * sizeof(int), &h));
    uint8_t* hb = (uint8_t*)h;
    memcpy(hb, ops.data(), ops.size() * sizeof(NetOp));
    Ctl* hc = (Ctl*)(hb + o_ctl);
    const float** hh = (const float**)(hb + o_hs);
    for (int b = 0; b < B; ++b) {
      init_ctl(hc + b, N, N / 2, 0.0, 1);
      if (window) {
        hc[b].e_min = window[0];
        hc[b].e_max = window[1];
      }
      hh[b] = H + (size_t)b * N * N;
      ((int*)(hb + o_ns))[b] = N;
      ((unsigned*)(hb + o_tick))[b] = 0u;
    }
    memcpy(hb + o_coef, coef.data(), coef.size() * sizeof(double));
    std::vector<int> order(B), Ns(B, N), toff(B), tcnt(B, per);
    std::vector<uint32_t> tiles;
    for (int b = 0; b < B; ++b) {
      order[b] = b;
      toff[b] = b * per;
      int n;
      resident_tiles(N, b, &tiles, &n);
    }
    resident_plan(order.data(), Ns.data(), toff.data(), tcnt.data(), B, grid, (int*)(hb + o_loff), (int*)(hb + o_list));
    memcpy(hb + o_tiles, tiles.data(), nt * sizeof(uint32_t));
    *(int*)(hb + o_err) = 0;
    CK(cudaMemcpyAsync(pack, hb, up, cudaMemcpyHostToDevice, st));
    if (!window)
      CK(launch_gershgorin_batched((const float* const*)(pack + o_hs), (const int*)(pack + o_ns), (Ctl*)(pack + o_ctl),
                                   B, part, (unsigned*)(pack + o_tick), ngrid, st));
    CK(launch_net_plan(plan, st));
    if (back) {
      *back = (int*)(hb + up);
      CK(cudaMemcpyAsync(*back, pack + o_status, (size_t)B * sizeof(int), cudaMemcpyDeviceToHost, st));
    }
    CK(cudaEventRecord(g.stage_done, st));  // also: the statuses are on the host
    CK(cudaMemsetAsync(A.sums, 0, (size_t)B * kMeetRows * sizeof(long long), st));
    return SP2_OK;
  }
  // the statuses of the bounds, once they are on the host
  sp2_status check(const int* status) const {
    for (int b = 0; b < B; ++b) {
      if (status[b] < 0) {
        set_err("instance %d: %s", b,
                status[b] == SP2_ERR_NONFINITE ? "non-finite spectral bounds" : "degenerate spectrum");
        return (sp2_status)status[b];
      }
    }
    return SP2_OK;
  }
  sp2_status wait_and_check(const int* back) const {
    CK(cudaEventSynchronize(g.stage_done));
    return check(back);
  }
  // inputs of one kind into the plane pairs from pool entry `entry` on
  NetInput input(int from, const float* in, int entry) const {
    NetInput x;
    memset(&x, 0, sizeof(x));
    x.N = N;
    x.batch = B;
    x.from = from;
    x.shift = A.shift;
    x.in = in;
    x.ctl = A.ctl;
    x.p0 = A.p0 + (long long)entry * B * A.slot_h;
    x.p1 = A.p1 ? A.p1 + (long long)entry * B * A.slot_h : nullptr;
    x.ld_h = A.ld_h;
    x.slot_h = A.slot_h;
    x.lo_scale = A.lo_scale;
    return x;
  }
};

NetOp net_square(int y, int out, int layer, int rnp) {
  NetOp o;
  memset(&o, 0, sizeof(o));
  o.y = y;
  o.out = out;
  o.layer = layer;
  o.rnp = rnp;
  return o;
}

// The network's forward pass on the resident kernel (net_fits).
sp2_status net_forward_resident(const float* H, int B, int N, int L, const float* coef, int ckpt_every, float* X_out,
                                float* ckpt, double* bounds) {
  const bool split = g.precision == SP2_PREC_SPLIT_FP16;
  const size_t mats = (size_t)B * N * N;
  NetRun R;
  void* rn;
  CKS(ws(B_RN, (size_t)B * N * sizeof(double), &rn));
  R.coef.assign(coef, coef + 3 * L);
  CKS(R.init(B, N, L, 2, split, L, (size_t)L * B, (size_t)(L + 1) * B));
  R.plan.bounds = bounds;
  for (int n = 0; n < L; ++n) {
    const bool last = n == L - 1, kept = ckpt && (n + 1) % ckpt_every == 0;
    NetOp o = net_square(n & 1, last ? -1 : (n & 1) ^ 1, n, n & 1);
    o.from = n == 0 ? NET_INPUT : NET_TMEM;
    o.in = H;
    o.rn = n == 0 ? (const double*)rn : nullptr;
    o.tmem = last ? 0 : 1;
    float* slot = kept ? ckpt + (size_t)((n + 1) / ckpt_every) * mats : nullptr;
    if (last) {
      o.full = X_out;
      o.exact = 1;
      o.full2 = slot;
    } else if (kept) {
      o.full = slot;
      o.full_add = R.dev((size_t)(n + 1) * B);
    }
    R.ops.push_back(o);
  }
  int* back = nullptr;
  CKS(R.start(H, nullptr, &back));
  NetInput x = R.input(NET_INPUT, H, 0);
  x.vec_norm = (N & 3) == 0 && ((uintptr_t)X_out & 15) == 0;
  x.rn = (double*)rn;
  x.x0 = ckpt;
  x.alpha0 = R.dev(0);
  CK(launch_net_input(x, B, g.stream));
  R.A.stall = take_stall();
  const cudaError_t le = coop_launch([&] { return launch_resident_net(R.A, R.maps, split, R.grid, g.stream); });
  if (refused(le)) return kRefused;
  CK(le);
  return R.wait_and_check(back);
}

void coef_gradient(const double* dd, const double* alpha, int L, int B, double* dcoef);

// Whether the adjoint's workspace on the resident kernel is in proportion.  It
// keeps the planes of every segment's first iterate (one input pass makes them
// all) and iterates in whole 128 x 128 tiles: up to 6 GiB, or twice what the CTA
// pairs take, which keep one segment's planes and iterates.  More of it (64 of 896
// take 4.6 GB with a segment a layer, 20 of them; 4096 of N = 1 with 256 layers in
// one segment would take 69 GB, on the pairs 0.3) goes to the pairs.
bool backward_fits(int B, int N, int L, int ce) {
  const bool split = g.precision == SP2_PREC_SPLIT_FP16;
  const double plane = (double)B * N * round_up(N, 64) * (split ? 4.0 : 2.0), mat = 4.0 * B * N * N;
  const int nseg = (L + ce - 1) / ce, kept = std::min(ce, L);
  int per = 0;
  resident_tiles(N, 0, nullptr, &per);
  const double resident = plane * (nseg + kept + 1) + 4.0 * B * per * kResTile * kResTile * std::max(1, kept - 1);
  const double pairs = plane * (ce + 2) + mat * (ce + 1);
  return resident <= std::max(6.0 * 0x1p30, 2.0 * pairs);
}

// The network's adjoint on the resident kernel: per checkpoint segment, from
// the last one, the recomputation of its iterates and the adjoint layers.
sp2_status net_backward_resident(const float* H, int B, int N, int L, const float* coef, int ce, const float* ckpt,
                                 const float* G_out, double* dcoef, float* G_in) {
  const bool split = g.precision == SP2_PREC_SPLIT_FP16;
  cudaStream_t st = g.stream;
  const size_t mats = (size_t)B * N * N, nalpha = (size_t)(L + 1) * B;
  const int nseg = (L + ce - 1) / ce;
  // pool: the segments' first iterates, the others of a segment, G twice
  const int p_rec = nseg, p_g = nseg + std::min(ce, L) - 1;
  NetRun R;
  void *rn, *keep, *tdots, *dots;
  CKS(ws(B_RN, (size_t)nseg * B * N * sizeof(double), &rn));
  R.coef.assign(coef, coef + 3 * L);
  CKS(R.init(B, N, L, p_g + 2, split, 2 * L, (size_t)2 * L * B, 2 * nalpha));
  R.plan.backward = 1;
  const size_t tile_store = (size_t)R.nt * kResTile * kResTile;
  CKS(ws(B_SEG, tile_store * 4 * std::max(1, std::min(ce, L) - 1), &keep));
  CKS(ws(B_TDOTS, (size_t)L * R.nt * 3 * sizeof(double), &tdots));
  CKS(ws(B_DOTS, (size_t)L * B * 3 * sizeof(double) + 16, &dots));
  R.A.tile_dots = (double*)tdots;
  auto minus_alpha = [&](int n) { return R.dev(nalpha + (size_t)n * B); };
  auto store = [&](int k) { return (float*)keep + tile_store * (size_t)(k - 1); };  // iterate n0 + k, k >= 1
  int gcur = 0;
  bool first = true;
  for (int s = nseg - 1; s >= 0; --s) {
    const int n0 = s * ce, n1 = std::min(n0 + ce, L);
    auto planes = [&](int k) { return k == 0 ? s : p_rec + k - 1; };
    const float* X0 = ckpt + (size_t)s * mats;
    for (int n = n0; n + 1 < n1; ++n) {
      const int k = n - n0;
      NetOp o = net_square(planes(k), planes(k + 1), n, k & 1);
      if (k == 0) {
        o.from = NET_X;
        o.in = X0;
        o.add = minus_alpha(n0);
        o.rn = (const double*)rn + (size_t)s * B * N;
      } else {
        o.from = NET_KEPT;
        o.in = store(k);
      }
      o.keep = store(k + 1);
      R.ops.push_back(o);
    }
    for (int n = n1 - 1; n >= n0; --n) {
      const int k = n - n0;
      NetOp o = net_square(planes(k), n == 0 ? -1 : p_g + (gcur ^ 1), L + n, 0);
      o.kind = 1;
      o.g = p_g + gcur;
      o.dot = n;
      o.from = first ? NET_FULL : NET_TMEM;
      o.in = G_out;
      o.tmem = n == 0 ? 0 : 1;
      if (k == 0) {
        o.aux_x = X0;
        o.aux_add = minus_alpha(n0);
      } else {
        o.aux = store(k);
      }
      if (n == 0) o.full = G_in;
      R.ops.push_back(o);
      first = false;
      gcur ^= 1;
    }
  }
  CKS(R.start(H, nullptr, nullptr));
  NetInput x = R.input(NET_X, ckpt, 0);
  x.add = minus_alpha(0);
  x.add_stride = (long long)ce * B;
  x.vec_norm = (N & 3) == 0;
  x.rn = (double*)rn;
  CK(launch_net_input(x, nseg * B, st));
  CK(launch_net_input(R.input(NET_FULL, G_out, p_g), B, st));
  const cudaError_t le = coop_launch([&] { return launch_resident_net(R.A, R.maps, split, R.grid, st); });
  if (refused(le)) return kRefused;
  CK(le);
  CK(launch_net_dots((const double*)tdots, R.nt, R.per, L, B, (double*)dots, st));
  // dot products, shifts, statuses, error word
  const size_t db = (size_t)L * B * 3 * sizeof(double), ab = nalpha * sizeof(double), sb = (size_t)B * sizeof(int);
  void* hd;
  CKS(staging(db + ab + sb + 16, &hd));
  char* hp = (char*)hd;
  CK(cudaMemcpyAsync(hp, dots, db, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(hp + db, R.plan.table, ab, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(hp + db + ab, R.plan.status, sb, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(hp + db + ab + sb, R.A.err, sizeof(int), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  CKS(R.check((const int*)(hp + db + ab)));
  if (*(const int*)(hp + db + ab + sb)) return timed_out();
  CKS(late_error());  // of the forward pass whose checkpoints were read
  coef_gradient((const double*)hp, (const double*)(hp + db), L, B, dcoef);
  return SP2_OK;
}

// dcoef from the dot products [L][B][3] (tr G, <G, Y_n>, <Y_n G + G Y_n, Y_n>):
// dL/da_n = <G, X_n^2> = alpha^2 tr G + 2 alpha <G, Y_n> + <Y_n G + G Y_n, Y_n> / 2
// dL/db_n = <G, X_n>   = alpha tr G + <G, Y_n>;   dL/dc_n = tr G
void coef_gradient(const double* dd, const double* alpha, int L, int B, double* dcoef) {
  for (int n = 0; n < L; ++n) {
    double da = 0.0, db = 0.0, dc = 0.0;
    for (int b = 0; b < B; ++b) {
      const double al = alpha[(size_t)n * B + b];
      const double* v = dd + ((size_t)n * B + b) * 3;
      da += al * al * v[0] + 2.0 * al * v[1] + 0.5 * v[2];
      db += al * v[0] + v[1];
      dc += v[0];
    }
    dcoef[3 * n] = da;
    dcoef[3 * n + 1] = db;
    dcoef[3 * n + 2] = dc;
  }
}

}  // namespace

sp2_status sp2_network_forward(const float* H, int B, int N, int L, const float* coef, int ckpt_every, float* X_out,
                               float* ckpt, double* bounds) {
  t_err.clear();
  CKS(require_init());
  if (!H || !X_out || !coef || H == X_out || B < 1 || B > 4096 || N < 1 || N > 8192 ||
      (long long)B * N * N >= (1LL << 31) || L < 1 || L > 256 || ckpt_every < 1 || ckpt_every > L) {
    set_err("sp2_network_forward: invalid argument");
    return SP2_ERR_INVALID_ARG;
  }
  for (int i = 0; i < 3 * L; ++i)
    if (!std::isfinite(coef[i])) {
      set_err("sp2_network_forward: non-finite coefficient");
      return SP2_ERR_INVALID_ARG;
    }
  CKS(late_error());
  if (net_fits(B, N, 896)) {
    const sp2_status s = net_forward_resident(H, B, N, L, coef, ckpt_every, X_out, ckpt, bounds);
    if (s != kRefused) return s;
  }
  const bool tc = tc_precision(g.precision);
  const bool split = g.precision == SP2_PREC_SPLIT_FP16;
  cudaStream_t st = g.stream;
  bool ok = false;
  NetPlan plan;
  void *ctl, *ns, *hs, *dptr;
  CKS(network_prologue(H, B, N, L, coef, &ok, plan, &ctl, &ns, &hs, &dptr, X_out));
  if (bounds)
    CK(cudaMemcpy2DAsync(bounds, 2 * sizeof(double), (char*)ctl + offsetof(Ctl, e_min), sizeof(Ctl),
                         2 * sizeof(double), B, cudaMemcpyDeviceToDevice, st));
  int ntiles = 0;
  // tensor-core layers on CTA pairs (super-tile pairs sharing B) unless
  // single CTAs are selected, as for the single solve
  const bool pairs = tc && g.pair_kernel;
  CKS(upload_tiles(N, B, tc ? (pairs ? 2 : 1) : 0, &ntiles));
  void *params, *alpha, *rn, *part, *tick, *err;
  CKS(ws(B_PARAMS, plan.params.size() * sizeof(LayerParams), &params));
  CKS(ws(B_BOUNDS, plan.alpha.size() * sizeof(double), &alpha));
  CKS(ws(B_RN, (size_t)B * N * sizeof(double), &rn));
  const int igrid = (int)std::min<long long>(N, std::max(1, 8 * g.num_sms / B + 1));
  CKS(ws(B_PART, (size_t)B * igrid * sizeof(double2), &part));
  CKS(ws(B_TICKET, std::max(64, B) * sizeof(unsigned), &tick, true));
  CKS(ws(B_ERR, sizeof(int), &err, true));
  auto ckpt_slot = [&](int k) { return ckpt + (size_t)k * B * N * N; };
  SqArgs A;
  memset(&A, 0, sizeof(A));
  void* rnp[2] = {nullptr, nullptr};
  if (tc) CKS(rnp_for(N, B, A, rnp));
  PlanePool pool;
  PairLists lists;
  if (pairs) {
    CKS(pool.init(split, 2, N, B));
    lists.begin();
    for (int n = 0; n < L; ++n) {
      LayerOp o;
      memset(&o, 0, sizeof(o));
      o.y = n & 1;
      o.g = -1;
      // only the upper super tiles of Y' are stored; a checkpoint is written
      // whole beside them
      o.tri_y = 1;
      o.Yin = o.Yout = X_out;
      o.p0_out = pool.p0_of((n & 1) ^ 1);
      o.p1_out = pool.p1_of((n & 1) ^ 1);
      o.rn = (const double*)rn;
      o.rnp_out = (float*)rnp[n & 1];
      o.rnp_in = n ? (const float*)rnp[(n - 1) & 1] : nullptr;
      o.lp = (const LayerParams*)params + (size_t)n * B;
      if (ckpt && (n + 1) % ckpt_every == 0 && n < L - 1) {
        o.X = ckpt_slot((n + 1) / ckpt_every);
        o.x_add = (const double*)alpha + (size_t)(n + 1) * B;
      }
      lists.ops.push_back(o);
    }
    CKS(lists.alloc(B, false));
  }
  void* h;
  const size_t plan_bytes = plan.params.size() * sizeof(LayerParams) + plan.alpha.size() * sizeof(double);
  CKS(staging(plan_bytes + lists.bytes, &h));
  memcpy(h, plan.params.data(), plan.params.size() * sizeof(LayerParams));
  memcpy((char*)h + plan.params.size() * sizeof(LayerParams), plan.alpha.data(), plan.alpha.size() * sizeof(double));
  CK(cudaMemcpyAsync(params, h, plan.params.size() * sizeof(LayerParams), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(alpha, (char*)h + plan.params.size() * sizeof(LayerParams), plan.alpha.size() * sizeof(double),
                     cudaMemcpyHostToDevice, st));
  if (pairs) {
    lists.fill((uint8_t*)h + plan_bytes);
    CK(cudaMemcpyAsync(lists.dev, (uint8_t*)h + plan_bytes, lists.bytes, cudaMemcpyHostToDevice, st));
  }
  CK(cudaEventRecord(g.stage_done, st));

  const long long slot = (long long)N * N;
  A.wait_ns = g.wait_ns;
  A.Dptr = (float* const*)dptr;
  A.Ns = (const int*)ns;
  A.tiles = (const uint32_t*)g.buf[B_TILES].p;
  A.ntiles = ntiles;
  A.tile_off = (const int*)g.buf[B_TOFF].p;
  A.tile_cnt = (const int*)g.buf[B_TCNT].p;
  A.ctl = nullptr;
  A.lp_per_instance = 1;
  A.tile_part = (double2*)g.buf[B_TPART].p;
  A.inst_done = (unsigned*)g.buf[B_IDONE].p;
  A.traces_out = nullptr;
  A.rn = (const double*)rn;
  A.ld_rn = N;
  A.lo_scale = std::ldexp(1.0f, g.lo_scale_exp);
  A.lo_unscale = std::ldexp(1.0f, -g.lo_scale_exp);
  A.err = (int*)err;
  A.late = g.late_dev;
  A.ld_y = N;
  A.slot_y = slot;
  const int mgrid = (int)std::min<long long>(N, std::max(1, 4 * g.num_sms / B + 1));
  const int rgrid = (int)std::min<long long>((N + 7) / 8, std::max(1, 2 * g.num_sms / B + 1));

  void* Y[2] = {X_out, nullptr};
  void *hi[2] = {nullptr, nullptr}, *lo[2] = {nullptr, nullptr}, *hp[2] = {nullptr, nullptr};
  long long ld_h = 0, slot_h = 0;
  CUtensorMap m[2][4];
  if (tc) {
    ld_h = round_up(N, 64);
    slot_h = ld_h * N;
    for (int k = 0; k < 2 && !pairs; ++k) {
      CKS(planes_for(split, k, (size_t)slot_h * B * 2, &hi[k], &lo[k], &hp[k]));
      CKS(tmaps4_for(split ? hp[k] : hi[k], lo[k], N, B, ld_h, slot_h, m[k]));
    }
    A.ld_h = ld_h;
    A.slot_h = slot_h;
  } else {
    // FFMA path: Y ping-pongs between two workspace buffers so the last layer
    // (which writes X_out) never reads its own output
    CKS(ws(B_Y0, (size_t)slot * B * 4, &Y[0]));
    CKS(ws(B_Y1, (size_t)slot * B * 4, &Y[1]));
  }
  if (pairs) {
    // X_0 (no control step) and its checkpoint, then every layer in one launch
    // (with one each, and the checkpoints copied by passes of their own, 64 x
    // 2048 x 20 layers took 27 ms)
    NetInput x = pair_input(pool, NET_INPUT, H, 0, N, B, X_out);
    x.shift = g.shift;
    x.ctl = (const Ctl*)ctl;
    x.rn = (double*)rn;
    x.y = X_out;
    x.x0 = ckpt;
    x.alpha0 = (const double*)alpha;
    CK(launch_net_input(x, B, st));
    A.tri_planes = 1;
    A.stall = take_stall();
    CK(launch_pairs(A, lists.list(0, false, true, ntiles / 2 / B), false, pool.m, split, pair_grid(ntiles)));
    if (ckpt && L % ckpt_every == 0)
      CK(cudaMemcpyAsync(ckpt_slot(L / ckpt_every), X_out, (size_t)B * slot * 4, cudaMemcpyDeviceToDevice, st));
    return SP2_OK;
  }
  // input layer X_0 (no control step)
  CK(launch_input_layer((const float* const*)hs, (const int*)ns, N, (float*)Y[0], N, slot, (__half*)hi[0],
                        (__half*)lo[0], (__half*)hp[0],
                        ld_h, slot_h, N, (int)ld_h, A.lo_scale, (Ctl*)ctl, nullptr, (double2*)part, (unsigned*)tick,
                        g.shift, 0, B, igrid, st));
  if (ckpt)
    CK(launch_materialize((float*)Y[0], N, slot, N, B, (const double*)alpha, ckpt_slot(0), N, slot, mgrid, st));
  for (int n = 0; n < L; ++n) {
    const int cur = n & 1;
    float* Yc = (float*)Y[tc ? 0 : cur];
    // tensor-core layers carry the row norms from one launch to the next
    if (!tc || n == 0)
      CK(launch_rownorm(Yc, N, slot, (const int*)ns, B, N, (double*)rn, N, nullptr, nullptr, nullptr, rgrid, st));
    A.lp = (const LayerParams*)params + (size_t)n * B;
    if (tc) {
      A.Yin = X_out;
      A.Yout = X_out;
      // Only the upper super tiles of Y' are stored unless whole rows are read
      // after this launch (a checkpoint; the last layer writes X_L whole anyway)
      const bool to_ckpt = ckpt && (n + 1) % ckpt_every == 0;
      A.tri_y = to_ckpt ? 0 : 1;
      A.hi_out = (__half*)hi[cur ^ 1];
      A.lo_out = (__half*)lo[cur ^ 1];
      A.hp_out = (__half*)hp[cur ^ 1];
      rnp_step(A, rnp, n);
      A.stall = take_stall();
      CK(launch_syrk_tc1(A, m[cur], split, std::min(ntiles, g.num_sms), st));
    } else {
      A.Yin = Yc;
      A.Yout = (float*)Y[cur ^ 1];
      CK(launch_syrk_simt(A, std::min(ntiles, 65535), st));
    }
    if (ckpt && (n + 1) % ckpt_every == 0) {
      const int k = (n + 1) / ckpt_every;
      if (n == L - 1) {
        CK(cudaMemcpyAsync(ckpt_slot(k), X_out, (size_t)B * slot * 4, cudaMemcpyDeviceToDevice, st));
      } else {
        float* Yn = (float*)Y[tc ? 0 : (cur ^ 1)];
        CK(launch_materialize(Yn, N, slot, N, B, (const double*)alpha + (size_t)(n + 1) * B, ckpt_slot(k), N, slot,
                              mgrid, st));
      }
    }
  }
  return SP2_OK;
}

sp2_status sp2_network_backward(const float* H, int B, int N, int L, const float* coef, int ckpt_every,
                                const float* ckpt, const float* G_out, double* dcoef, float* G_in) {
  t_err.clear();
  CKS(require_init());
  if (!H || !ckpt || !G_out || !dcoef || !coef || B < 1 || B > 4096 || N < 1 || N > 8192 ||
      (long long)B * N * N >= (1LL << 31) || L < 1 || L > 256 || ckpt_every < 1 || ckpt_every > L) {
    set_err("sp2_network_backward: invalid argument");
    return SP2_ERR_INVALID_ARG;
  }
  if (!tc_precision(g.precision)) {
    set_err("sp2_network_backward: the adjoint runs on the tensor-core paths (split or fp16)");
    return SP2_ERR_UNSUPPORTED;
  }
  CKS(late_error());
  const bool split = g.precision == SP2_PREC_SPLIT_FP16;
  cudaStream_t st = g.stream;
  const long long slot = (long long)N * N;
  const int ce = ckpt_every;
  if (net_fits(B, N, 896) && backward_fits(B, N, L, ce)) {
    const bool injected = g.fault_alloc;
    const sp2_status s = net_backward_resident(H, B, N, L, coef, ce, ckpt, G_out, dcoef, G_in);
    if (s != kRefused && (s != SP2_ERR_OOM || injected)) return s;
    // the pairs need less; what the attempt holds goes back first
    t_err.clear();
    if (s == SP2_ERR_OOM)
      for (BufId id : {B_PLANES0, B_PLANES1, B_SEG}) CKS(ws_free(id));
  }
  void* G;
  CKS(ws(B_G, (size_t)B * slot * 4, &G));
  bool ok = false;
  NetPlan plan;
  void *ctl, *ns, *hs, *dptr;
  CKS(network_prologue(H, B, N, L, coef, &ok, plan, &ctl, &ns, &hs, &dptr, (float*)G));

  // backward coefficients: G_n = (2 a_n alpha_n + b_n) G + a_n (Y_n G + G Y_n)
  std::vector<LayerParams> bp((size_t)L * B);
  std::vector<double> nalpha(plan.alpha.size());
  for (size_t i = 0; i < nalpha.size(); ++i) nalpha[i] = -plan.alpha[i];
  for (int n = 0; n < L; ++n)
    for (int b = 0; b < B; ++b) {
      const double a = coef[3 * n], bb = coef[3 * n + 1], al = plan.alpha[(size_t)n * B + b];
      LayerParams p;
      memset(&p, 0, sizeof(p));
      p.ca_d = 2.0 * a * al + bb;
      p.cb_d = a;
      p.cc_d = 0.0;
      p.ca = (float)p.ca_d;
      p.cb = (float)p.cb_d;
      p.active = 1;
      p.out_mode = OUT_Y;
      bp[(size_t)n * B + b] = p;
      // forward recomputation never reaches the last layer: keep OUT_Y there
      plan.params[(size_t)n * B + b].out_mode = OUT_Y;
      plan.params[(size_t)n * B + b].alpha_out = 0.0;
    }
  // CTA pairs (M = 256 MMAs) unless the single-CTA kernel was selected; the
  // pair kernel keeps the operand planes as upper super tiles
  const bool pairs = g.pair_kernel;
  int ntiles = 0;
  CKS(upload_tiles(N, B, pairs ? 2 : 1, &ntiles));
  const long long ld_h = round_up(N, 64), slot_h = ld_h * N;
  void *params, *params2, *nal, *rn, *err, *seg, *segp = nullptr, *gh[2] = {}, *gl[2] = {}, *dots, *tdots;
  CKS(ws(B_PARAMS, plan.params.size() * sizeof(LayerParams), &params));
  CKS(ws(B_PARAMS2, bp.size() * sizeof(LayerParams), &params2));
  CKS(ws(B_NALPHA, nalpha.size() * sizeof(double), &nal));
  CKS(ws(B_RN, (size_t)B * N * sizeof(double), &rn));
  CKS(ws(B_ERR, sizeof(int), &err, true));
  CKS(ws(B_SEG, (size_t)ce * B * slot * 4, &seg));
  // operand planes of the ce iterates of a segment, kept from the
  // recomputation for the adjoint layers, and of G (twice): p0 = hp (split) or
  // hi (plain) and p1 = lo' (split only)
  const int nplanes = split ? 2 : 1;
  const size_t plane_bytes = (size_t)slot_h * B * 2;
  PlanePool pool;  // CTA pairs: entries 0 .. ce - 1, G in ce and ce + 1
  if (pairs) {
    CKS(pool.init(split, ce + 2, N, B));
  } else {
    CKS(ws(B_SEGP, plane_bytes * nplanes * ce, &segp));
    CKS(ws(B_GH0, plane_bytes, &gh[0]));
    CKS(ws(B_GH1, plane_bytes, &gh[1]));
    if (split) {
      CKS(ws(B_GL0, plane_bytes, &gl[0]));
      CKS(ws(B_GL1, plane_bytes, &gl[1]));
    }
  }
  CKS(ws(B_DOTS, (size_t)L * B * 3 * sizeof(double), &dots, true));
  CKS(ws(B_TDOTS, (size_t)ntiles * 2 * 3 * sizeof(double), &tdots));
  SqArgs A;
  memset(&A, 0, sizeof(A));
  void* rnp[2];
  CKS(rnp_for(N, B, A, rnp));  // the row-norm carry of the recomputation
  auto segY = [&](int i) { return (float*)seg + (size_t)i * B * slot; };
  // planes of Y_{n0 + k} and of G
  auto segp0 = [&](int k) {
    return pairs ? pool.p0_of(k) : (__half*)((char*)segp + plane_bytes * nplanes * k);
  };
  auto segp1 = [&](int k) {
    return pairs ? pool.p1_of(k) : split ? (__half*)((char*)segp + plane_bytes * (nplanes * k + 1)) : nullptr;
  };
  auto g0 = [&](int k) { return pairs ? pool.p0_of(ce + k) : (__half*)gh[k]; };
  auto g1 = [&](int k) { return pairs ? pool.p1_of(ce + k) : (__half*)gl[k]; };
  const int nseg_layers = (L + ce - 1) / ce;
  PairLists lists;
  if (pairs) {
    int gp = 0;
    for (int sgi = nseg_layers - 1; sgi >= 0; --sgi) {
      const int n0 = sgi * ce, n1 = std::min(n0 + ce, L);
      lists.begin();
      for (int n = n0; n + 1 < n1; ++n) {
        // the recomputed iterates are read only on upper super tiles
        const int k = n - n0;
        LayerOp o;
        memset(&o, 0, sizeof(o));
        o.y = k;
        o.g = -1;
        o.tri_y = 1;
        o.Yin = segY(k);
        o.Yout = segY(k + 1);
        o.p0_out = pool.p0_of(k + 1);
        o.p1_out = pool.p1_of(k + 1);
        o.rn = (const double*)rn;
        o.rnp_out = (float*)rnp[k & 1];
        o.rnp_in = k ? (const float*)rnp[(k - 1) & 1] : nullptr;
        o.lp = (const LayerParams*)params + (size_t)n * B;
        lists.ops.push_back(o);
      }
      for (int n = n1 - 1; n >= n0; --n, gp ^= 1) {
        LayerOp o;
        memset(&o, 0, sizeof(o));
        o.y = n - n0;
        o.g = ce + gp;
        // G is read on upper super tiles only, except after the last adjoint
        // layer (dL/dX_0 is returned whole)
        o.tri_y = n == 0 && G_in ? 0 : 1;
        o.Yin = (float*)G;
        o.Yout = n == 0 && G_in ? G_in : (float*)G;
        o.aux = segY(n - n0);
        o.p0_out = pool.p0_of(ce + (gp ^ 1));
        o.p1_out = pool.p1_of(ce + (gp ^ 1));
        o.lp = (const LayerParams*)params2 + (size_t)n * B;
        o.dots_out = (double*)dots + (size_t)n * B * 3;
        lists.ops.push_back(o);
      }
    }
    CKS(lists.alloc(B, false));
  }
  void* h;
  const size_t pb = plan.params.size() * sizeof(LayerParams), bb2 = bp.size() * sizeof(LayerParams),
               ab = nalpha.size() * sizeof(double);
  CKS(staging(pb + bb2 + ab + lists.bytes, &h));
  memcpy(h, plan.params.data(), pb);
  memcpy((char*)h + pb, bp.data(), bb2);
  memcpy((char*)h + pb + bb2, nalpha.data(), ab);
  CK(cudaMemcpyAsync(params, h, pb, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(params2, (char*)h + pb, bb2, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(nal, (char*)h + pb + bb2, ab, cudaMemcpyHostToDevice, st));
  if (pairs) {
    lists.fill((char*)h + pb + bb2 + ab);
    CK(cudaMemcpyAsync(lists.dev, (char*)h + pb + bb2 + ab, lists.bytes, cudaMemcpyHostToDevice, st));
  }
  CK(cudaEventRecord(g.stage_done, st));

  std::vector<CUtensorMap> mY(pairs ? 0 : (size_t)ce * 4);
  CUtensorMap mG4[2][4];
  if (!pairs) {
    for (int k = 0; k < ce; ++k) CKS(tmaps4_for(segp0(k), segp1(k), N, B, ld_h, slot_h, &mY[(size_t)k * 4]));
    for (int k = 0; k < 2; ++k) CKS(tmaps4_for(gh[k], gl[k], N, B, ld_h, slot_h, mG4[k]));
  }
  const float ls = std::ldexp(1.0f, g.lo_scale_exp);
  A.wait_ns = g.wait_ns;
  A.Dptr = (float* const*)dptr;
  A.Ns = (const int*)ns;
  A.tiles = (const uint32_t*)g.buf[B_TILES].p;
  A.ntiles = ntiles;
  A.tile_off = (const int*)g.buf[B_TOFF].p;
  A.tile_cnt = (const int*)g.buf[B_TCNT].p;
  A.lp_per_instance = 1;
  A.tile_part = (double2*)g.buf[B_TPART].p;
  A.inst_done = (unsigned*)g.buf[B_IDONE].p;
  A.lo_scale = ls;
  A.lo_unscale = std::ldexp(1.0f, -g.lo_scale_exp);
  A.err = (int*)err;
  A.late = g.late_dev;
  A.ld_y = N;
  A.slot_y = slot;
  A.ld_h = ld_h;
  A.slot_h = slot_h;
  const int sgrid = (int)std::min<long long>((long long)N * B, 8LL * g.num_sms);
  const int mgrid = (int)std::min<long long>(N, std::max(1, 4 * g.num_sms / B + 1));
  const int rgrid = (int)std::min<long long>((N + 7) / 8, std::max(1, 2 * g.num_sms / B + 1));
  const int tgrid = pairs ? pair_grid(ntiles) : std::min(ntiles, g.num_sms);
  const SqArgs& R0 = A;

  if (pairs) {
    NetInput x = pair_input(pool, NET_FULL, G_out, ce, N, B, nullptr);
    x.y = (float*)G;
    CK(launch_net_input(x, B, st));
  } else {
    CK(cudaMemcpyAsync(G, G_out, (size_t)B * slot * 4, cudaMemcpyDeviceToDevice, st));
    CK(launch_split_pad((float*)G, N, slot, N, B, ls, split ? nullptr : g0(0), g1(0), split ? g0(0) : nullptr, ld_h,
                        slot_h, sgrid, st));
  }
  int cur = 0;

  for (int sgi = nseg_layers - 1; sgi >= 0; --sgi) {
    const int n0 = sgi * ce, n1 = std::min(n0 + ce, L);
    // Y_{n0} = X_{n0} - alpha_{n0} I from the checkpoint and its planes, then
    // recompute to Y_{n1-1}: each launch also writes the planes of its
    // output and carries the row norms to the next (as in the forward pass)
    if (pairs) {
      NetInput x = pair_input(pool, NET_X, ckpt + (size_t)sgi * B * slot, 0, N, B, segY(0));
      x.add = (const double*)nal + (size_t)n0 * B;
      x.y = segY(0);
      x.rn = n1 - n0 > 1 ? (double*)rn : nullptr;
      CK(launch_net_input(x, B, st));
      // the segment's recomputation and adjoint layers in one launch
      SqArgs P = A;
      P.tri_planes = 1;
      P.tile_dots = (double*)tdots;
      P.rn = (const double*)rn;
      P.ld_rn = N;
      CK(launch_pairs(P, lists.list(nseg_layers - 1 - sgi, false, true, ntiles / 2 / B), true, pool.m, split, tgrid));
      continue;
    }
    CK(launch_materialize(ckpt + (size_t)sgi * B * slot, N, slot, N, B, (const double*)nal + (size_t)n0 * B,
                          segY(0), N, slot, mgrid, st));
    CK(launch_split_pad(segY(0), N, slot, N, B, ls, split ? nullptr : segp0(0), segp1(0), split ? segp0(0) : nullptr,
                        ld_h, slot_h, sgrid, st));
    if (n1 - n0 > 1)
      CK(launch_rownorm(segY(0), N, slot, (const int*)ns, B, N, (double*)rn, N, nullptr, nullptr, nullptr, rgrid, st));
    for (int n = n0; n + 1 < n1; ++n) {
      const int k = n - n0;
      SqArgs F = R0;
      F.Yin = segY(k);
      F.Yout = segY(k + 1);
      F.hi_out = split ? nullptr : segp0(k + 1);
      F.hp_out = split ? segp0(k + 1) : nullptr;
      F.lo_out = segp1(k + 1);
      F.rn = (const double*)rn;
      F.ld_rn = N;
      rnp_step(F, rnp, k);
      F.lp = (const LayerParams*)params + (size_t)n * B;
      F.nseg = 1;
      // the recomputed iterates are read only on upper super tiles (the next
      // layer's old values, the adjoint epilogue's aux)
      F.tri_y = 1;
      CK(launch_syrk_tc1(F, &mY[(size_t)k * 4], split, tgrid, st));
    }
    for (int n = n1 - 1; n >= n0; --n) {
      const int k = n - n0;
      float* Yn = segY(k);
      const CUtensorMap* mYk = &mY[(size_t)k * 4];
      const CUtensorMap* mGk = mG4[cur];
      // segment 1: Y_n rows x G rows (Y G), segment 2: G rows x Y_n rows (G Y)
      const CUtensorMap m8[8] = {mYk[0], mYk[1], mGk[2], mGk[3], mGk[0], mGk[1], mYk[2], mYk[3]};
      SqArgs Bk = A;
      Bk.Yin = (float*)G;
      Bk.Yout = (float*)G;
      Bk.hi_out = split ? nullptr : (__half*)gh[cur ^ 1];
      Bk.hp_out = split ? (__half*)gh[cur ^ 1] : nullptr;
      Bk.lo_out = (__half*)gl[cur ^ 1];
      Bk.rn = nullptr;
      Bk.lp = (const LayerParams*)params2 + (size_t)n * B;
      Bk.nseg = 2;
      Bk.aux = Yn;
      Bk.tile_dots = (double*)tdots;
      Bk.dots_out = (double*)dots + (size_t)n * B * 3;
      // G is read on upper super tiles only, except after the last adjoint
      // layer (dL/dX_0 is returned whole)
      Bk.tri_y = n == 0 ? 0 : 1;
      CK(launch_syrk_tc1(Bk, m8, split, tgrid, st));
      cur ^= 1;
    }
  }
  if (G_in && !pairs) CK(cudaMemcpyAsync(G_in, G, (size_t)B * slot * 4, cudaMemcpyDeviceToDevice, st));
  void* hd;
  CKS(staging((size_t)L * B * 3 * sizeof(double) + 16, &hd));
  CK(cudaMemcpyAsync(hd, dots, (size_t)L * B * 3 * sizeof(double), cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync((char*)hd + (size_t)L * B * 3 * sizeof(double), err, sizeof(int), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  const double* dd = (const double*)hd;
  if (*(const int*)((char*)hd + (size_t)L * B * 3 * sizeof(double))) return timed_out();
  CKS(late_error());  // of the forward pass whose checkpoints were read
  coef_gradient(dd, plan.alpha.data(), L, B, dcoef);
  return SP2_OK;
}

// Finite-temperature expansion (Sec. "Optimized SP2 Finite Temperature
// Fermi-Operator Expansion"): X_0 = (H - e_lo I)/(e_hi - e_lo),
// X_{n+1} = a_n X_n^2 + b_n X_n + c_n I, D = I - sum_i c_i X_i.  The layers
// run on the CTA-pair squaring kernel with the readout accumulated in the
// epilogue; X_0 is the reflection I - S_0 of the SP2 input layer, folded into
// the first layer's coefficients and the readout's start.
sp2_status sp2_fermi_expansion(const float* H, int B, int N, int L, const double* theta, const double* c,
                               double e_lo, double e_hi, float* D_out, double* bounds) {
  t_err.clear();
  CKS(require_init());
  const bool fixed = (e_lo != 0.0 || e_hi != 0.0);
  bool finite = theta && c;
  for (int i = 0; finite && i < 3 * L; ++i) finite = std::isfinite(theta[i]);
  for (int i = 0; finite && i <= L; ++i) finite = std::isfinite(c[i]);
  if (!H || !D_out || H == D_out || B < 1 || B > 4096 || N < 1 || N > 8192 || (long long)B * N * N >= (1LL << 31) ||
      L < 1 || L > SP2_MAX_LAYERS || !finite || (fixed && !(std::isfinite(e_lo) && std::isfinite(e_hi) && e_lo < e_hi))) {
    set_err("sp2_fermi_expansion: invalid argument");
    return SP2_ERR_INVALID_ARG;
  }
  if (!tc_precision(g.precision)) {
    set_err("sp2_fermi_expansion: needs a tensor-core precision (split or fp16)");
    return SP2_ERR_UNSUPPORTED;
  }
  CKS(late_error());
  const bool split = g.precision == SP2_PREC_SPLIT_FP16;
  cudaStream_t st = g.stream;
  const long long slot = (long long)N * N;

  if (net_fits(B, N, 1152)) {
    NetRun run;
    void *rn, *R;
    CKS(ws(B_RN, (size_t)B * N * sizeof(double), &rn));
    run.coef.assign(theta, theta + 3 * L);
    run.coef.insert(run.coef.end(), c, c + L + 1);
    CKS(run.init(B, N, L, 2, split, L, (size_t)L * B, B));
    CKS(ws(B_READOUT, (size_t)run.nt * kResTile * kResTile * sizeof(float), &R));
    run.plan.expansion = 1;
    run.plan.bounds = bounds;
    run.A.shift = 1;
    run.A.R = (float*)R;
    run.A.r_scale = (float)(-c[0]);
    run.A.r_add = run.dev(0);
    for (int n = 0; n < L; ++n) {
      const bool last = n == L - 1;
      NetOp o = net_square(n & 1, last ? -1 : (n & 1) ^ 1, n, n & 1);
      o.from = n == 0 ? NET_INPUT : NET_TMEM;
      o.in = H;
      o.rn = n == 0 ? (const double*)rn : nullptr;
      o.tmem = last ? 0 : 1;
      o.readout = n == 0 ? 2 : 1;
      o.full = last ? D_out : nullptr;
      run.ops.push_back(o);
    }
    const double window[2] = {e_lo, e_hi};
    int* back = nullptr;
    CKS(run.start(H, fixed ? window : nullptr, fixed ? nullptr : &back));
    NetInput x = run.input(NET_INPUT, H, 0);
    x.vec_norm = (N & 3) == 0 && ((uintptr_t)D_out & 15) == 0;
    x.rn = (double*)rn;
    CK(launch_net_input(x, B, st));
    run.A.stall = take_stall();
    const cudaError_t le = coop_launch([&] { return launch_resident_net(run.A, run.maps, split, run.grid, st); });
    if (!refused(le)) {
      CK(le);
      return fixed ? SP2_OK : run.wait_and_check(back);
    }
  }

  // per-instance records; fixed bounds go straight into the control blocks
  void *ctl, *ns, *hs, *dptr;
  CKS(ws(B_CTL, (size_t)B * sizeof(Ctl), &ctl));
  CKS(ws(B_NS, B * sizeof(int), &ns));
  CKS(ws(B_HS, B * sizeof(float*), &hs));
  CKS(ws(B_DPTR, B * sizeof(float*), &dptr));
  const int ggrid = (int)std::min<long long>((N + 7) / 8, std::max((N + 63) / 64, 2 * g.num_sms / B + 1));
  const int igrid = (int)std::min<long long>(N, std::max(1, 8 * g.num_sms / B + 1));
  void *part, *tick, *err;
  CKS(ws(B_PART, (size_t)B * std::max(ggrid, igrid) * sizeof(double2), &part));
  CKS(ws(B_TICKET, std::max(64, B) * sizeof(unsigned), &tick, true));
  CKS(ws(B_ERR, sizeof(int), &err, true));
  {
    void* h;
    CKS(staging((size_t)B * sizeof(Ctl) + B * (sizeof(int) + 2 * sizeof(void*)) + 64, &h));
    Ctl* hc = (Ctl*)h;
    for (int b = 0; b < B; ++b) {
      init_ctl(hc + b, N, N / 2, 0.0, 1);
      if (fixed) {
        hc[b].e_min = e_lo;
        hc[b].e_max = e_hi;
      }
    }
    int* hn = (int*)(hc + B);
    const float** hh = (const float**)(hn + B + (B & 1));
    float** hd = (float**)(hh + B);
    for (int b = 0; b < B; ++b) {
      hn[b] = N;
      hh[b] = H + (size_t)b * slot;
      hd[b] = D_out + (size_t)b * slot;
    }
    CK(cudaMemcpyAsync(ctl, hc, (size_t)B * sizeof(Ctl), cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(ns, hn, B * sizeof(int), cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(hs, hh, B * sizeof(void*), cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(dptr, hd, B * sizeof(void*), cudaMemcpyHostToDevice, st));
    CK(cudaEventRecord(g.stage_done, st));
  }
  std::vector<double> lo_b(B, e_lo), hi_b(B, e_hi);
  if (!fixed) {
    CK(launch_gershgorin_batched((const float* const*)hs, (const int*)ns, (Ctl*)ctl, B, (double2*)part,
                                 (unsigned*)tick, ggrid, st));
    void* hb;
    CKS(staging((size_t)B * 2 * sizeof(double) + (size_t)B * sizeof(int), &hb));
    CK(cudaMemcpy2DAsync(hb, 2 * sizeof(double), (char*)ctl + offsetof(Ctl, e_min), sizeof(Ctl), 2 * sizeof(double),
                         B, cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpy2DAsync((char*)hb + (size_t)B * 2 * sizeof(double), sizeof(int), (char*)ctl + offsetof(Ctl, status),
                         sizeof(Ctl), sizeof(int), B, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    const double* bd = (const double*)hb;
    const int* bs = (const int*)((char*)hb + (size_t)B * 2 * sizeof(double));
    for (int b = 0; b < B; ++b) {
      if (bs[b] < 0) {
        set_err("instance %d: %s", b, bs[b] == SP2_ERR_NONFINITE ? "non-finite spectral bounds" : "degenerate spectrum");
        return (sp2_status)bs[b];
      }
      lo_b[b] = bd[2 * b];
      hi_b[b] = bd[2 * b + 1];
    }
  }
  if (bounds)
    CK(cudaMemcpy2DAsync(bounds, 2 * sizeof(double), (char*)ctl + offsetof(Ctl, e_min), sizeof(Ctl),
                         2 * sizeof(double), B, cudaMemcpyDeviceToDevice, st));

  // FP64 plan on the host: the input layer stores S_0 = alpha_0 I + Y_0 with
  // alpha_0 = e_hi/w and Y_0 = -H/w; X_0 = I - S_0 = (1 - alpha_0) I - Y_0.
  std::vector<LayerParams> params((size_t)L * B);
  std::vector<double> d0(B);
  for (int b = 0; b < B; ++b) {
    const double w = hi_b[b] - lo_b[b];
    double al = 1.0 - hi_b[b] / w;  // identity part of X_0 (= -e_lo/w)
    d0[b] = c[0] * al;               // R_0 = c_0 X_0 = -c_0 Y_0 + c_0 al I
    for (int n = 0; n < L; ++n) {
      const double a = theta[3 * n], bb = theta[3 * n + 1], cp = theta[3 * n + 2];
      const double an = a * al * al + bb * al + cp;
      LayerParams p;
      memset(&p, 0, sizeof(p));
      p.ca_d = (n == 0 ? -1.0 : 1.0) * (2.0 * a * al + bb);  // layer 0 reads Y_0 = -(X_0 - al I)
      p.cb_d = a;
      p.cc_d = 0.0;
      p.ca = (float)p.ca_d;
      p.cb = (float)p.cb_d;
      p.active = 1;
      p.out_mode = (n == L - 1) ? OUT_D : OUT_Y;
      p.rc_d = c[n + 1];
      p.rc = (float)c[n + 1];
      p.alpha_new = an;
      params[(size_t)n * B + b] = p;
      al = an;
    }
  }

  int ntiles = 0;
  CKS(upload_tiles(N, B, 2, &ntiles));
  void *prm, *dd, *R, *rn;
  CKS(ws(B_PARAMS, params.size() * sizeof(LayerParams), &prm));
  CKS(ws(B_RDIAG, (size_t)B * sizeof(double), &dd));
  CKS(ws(B_READOUT, (size_t)B * slot * sizeof(float), &R));
  CKS(ws(B_RN, (size_t)B * N * sizeof(double), &rn));
  SqArgs A;
  memset(&A, 0, sizeof(A));
  void* rnp[2];
  CKS(rnp_for(N, B, A, rnp));
  PlanePool pool;
  CKS(pool.init(split, 2, N, B));
  PairLists lists;
  lists.begin();
  for (int n = 0; n < L; ++n) {
    LayerOp o;
    memset(&o, 0, sizeof(o));
    o.y = n & 1;
    o.g = -1;
    o.tri_y = 1;  // between layers only the upper triangle of Y' is kept
    o.Yin = o.Yout = D_out;
    o.p0_out = pool.p0_of((n & 1) ^ 1);
    o.p1_out = pool.p1_of((n & 1) ^ 1);
    o.rn = (const double*)rn;
    o.rnp_out = (float*)rnp[n & 1];
    o.rnp_in = n ? (const float*)rnp[(n - 1) & 1] : nullptr;
    o.lp = (const LayerParams*)prm + (size_t)n * B;
    lists.ops.push_back(o);
  }
  CKS(lists.alloc(B, false));
  {
    void* h;
    const size_t plan_bytes = params.size() * sizeof(LayerParams) + (size_t)B * sizeof(double);
    CKS(staging(plan_bytes + lists.bytes, &h));
    lists.fill((char*)h + plan_bytes);
    CK(cudaMemcpyAsync(lists.dev, (char*)h + plan_bytes, lists.bytes, cudaMemcpyHostToDevice, st));
    memcpy(h, params.data(), params.size() * sizeof(LayerParams));
    memcpy((char*)h + params.size() * sizeof(LayerParams), d0.data(), (size_t)B * sizeof(double));
    CK(cudaMemcpyAsync(prm, h, params.size() * sizeof(LayerParams), cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(dd, (char*)h + params.size() * sizeof(LayerParams), (size_t)B * sizeof(double),
                       cudaMemcpyHostToDevice, st));
    CK(cudaEventRecord(g.stage_done, st));
  }
  const long long ld_h = round_up(N, 64), slot_h = ld_h * N;
  A.wait_ns = g.wait_ns;
  A.Dptr = (float* const*)dptr;
  A.Ns = (const int*)ns;
  A.tiles = (const uint32_t*)g.buf[B_TILES].p;
  A.ntiles = ntiles;
  A.tile_off = (const int*)g.buf[B_TOFF].p;
  A.tile_cnt = (const int*)g.buf[B_TCNT].p;
  A.lp_per_instance = 1;
  A.tile_part = (double2*)g.buf[B_TPART].p;
  A.inst_done = (unsigned*)g.buf[B_IDONE].p;
  A.rn = (const double*)rn;
  A.ld_rn = N;
  A.lo_scale = std::ldexp(1.0f, g.lo_scale_exp);
  A.lo_unscale = std::ldexp(1.0f, -g.lo_scale_exp);
  A.err = (int*)err;
  A.late = g.late_dev;
  A.Yin = D_out;
  A.Yout = D_out;
  A.ld_y = N;
  A.slot_y = slot;
  A.ld_h = ld_h;
  A.slot_h = slot_h;
  A.R = (float*)R;
  A.tri_planes = 1;  // upper super tiles only

  // S_0 (shifted form) into D_out and its planes, R_0 = c_0 X_0, row norms of Y_0
  NetInput x = pair_input(pool, NET_INPUT, H, 0, N, B, D_out);
  x.shift = 1;
  x.ctl = (const Ctl*)ctl;
  x.rn = (double*)rn;
  x.y = D_out;
  x.r = (float*)R;
  x.r_scale = (float)(-c[0]);
  x.r_add = (const double*)dd;
  CK(launch_net_input(x, B, st));
  A.stall = take_stall();
  CK(launch_pairs(A, lists.list(0, false, true, ntiles / 2 / B), false, pool.m, split, pair_grid(ntiles)));
  return SP2_OK;
}

}  // extern "C"
