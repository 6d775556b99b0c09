// Host-side launch interface of the SP2 kernels (internal to libsp2.so).
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace sp2 {

// Arguments shared by the squaring kernels (FFMA and tcgen05).
//
// Storage of instance b (0 <= b < batch) with size n_b = Ns[b]:
//   Y      FP32 iterate, element (r, c) at Y + b*slot_y + r*ld_y + c
//   planes FP16 planes of Y (tensor-core path: hp = 2^s hi and lo' for the
//          split product, hi for plain FP16), b*slot_h + r*ld_h + c; the
//          region [n_b, ld) of every row and rows >= n_b stay zero
//   Dptr   per-instance final outputs [n_b, n_b] (ld n_b), used by OUT_D
// Tiles: tiles[t] packs (b, I, J, h); the tiles of one instance are
// contiguous, starting at tile_off[b], tile_cnt[b] of them.
struct SqArgs {
  const float* Yin;        // FFMA path: operand and old value (read-only)
  float* Yout;             // updated iterate (may equal Yin on the tensor-core path)
  long long ld_y, slot_y;
  __half* hi_out;          // FP16 planes of the updated iterate, each written when set:
  __half* lo_out;          //   hi = fp16(Y'), lo' = fp16(2^s (Y' - hi)),
  __half* hp_out;          //   hp = 2^s hi (single-accumulator kernels: split writes hp_out
                           //   and lo_out, plain FP16 hi_out and lo_out)
  long long ld_h, slot_h;
  float* const* Dptr;      // [batch] device array of output pointers (OUT_D)
  const int* Ns;           // [batch]
  const uint32_t* tiles;   // [ntiles]
  int ntiles;
  const int* tile_off;     // [batch]
  const int* tile_cnt;     // [batch]
  Ctl* ctl;                // [batch] control blocks, or nullptr
  const LayerParams* lp;   // coefficients when ctl == nullptr
  int lp_per_instance;     // 1: lp[b] per instance, 0: lp[0] shared by the batch
  double2* tile_part;      // [ntiles] per-tile (tr, sq) partials
  unsigned* inst_done;     // [batch] tile-completion counters (zero between launches)
  double* traces_out;      // [batch][2] when ctl == nullptr, or nullptr
  const double* rn;        // [batch][ld_rn] FP64 row norms sum_k Y[r][k]^2 = (Y^2)_rr of the input
  long long ld_rn;
  // Row norms carried between launches (single-accumulator kernels): FP32
  // sums of squares of 32-column segments, rnp[b][seg][row] at
  // b * slot_rnp + seg * ld_rnp + row.  rnp_out receives those of Y' (every
  // (row, segment) once: the direct part of an upper tile or the column sums
  // of its mirror); rnp_in, when set, holds those of the input Y and replaces
  // rn: (Y^2)_rr = sum over segments in FP64.
  float* rnp_out;
  const float* rnp_in;
  long long ld_rnp, slot_rnp;
  int fused_ctl;           // 1: the last tile of an instance runs its control step with
                           //    (tr Y', ||Y'||_F^2) from the tiles (no row-norm launch)
  int nseg;                // 1: P = Y Y (one operand); 2: P = A B^T + B A^T (second map set)
  float* R;                // readout accumulator R = sum_i c_i X_i (layout of Y), or nullptr
  const float* const* Hobs; // [batch] N x N matrices A: the launch that writes D (OUT_D) also
                            // accumulates Tr[D A] per instance into dots_out[3 b] (or nullptr)
  const float* aux;        // adjoint mode: Y_n, same layout as Yin; dots <P, aux>, <Yin, aux>
  double* tile_dots;       // [ntiles][3] per-tile (tr Yin, <Yin, aux>, <P, aux>) in adjoint mode
  double* dots_out;        // [batch][3] per-instance sums of tile_dots
  int tri_planes;          // 1: the operand planes too are kept as upper super tiles (the
                           //    mirror plane stores are skipped); only for the CTA-pair kernel,
                           //    whose operand reads use the upper super tiles alone
  int tri_y;               // 1: Y' is kept as its upper triangle: off-diagonal tiles skip the
                           //    mirror store of Y' (the next launch reads the old values of
                           //    the upper tiles only); the operand planes and the D of the
                           //    final launch are stored whole
  float lo_scale;          // 2^s
  float lo_unscale;        // 2^-s
  int* err;                // device error word (SP2_ERR_DEVICE_TIMEOUT on a timed-out wait)
  int* late;               // the host's word for calls that return before their end, or nullptr
  unsigned long long wait_ns;  // bound of every mbarrier wait of the tcgen05 kernels (0: 4 s)
  int stall;               // fault injection: the MMA issuer first waits on a barrier that
                           // nothing arrives on, so that wait runs out after wait_ns
  // Soft synchronisation of the CTA pairs' K progress (CTA-pair kernel, one
  // instance): every sync_stages K stages a pair publishes the epoch it
  // finished in wave_ctr[epoch] and, before loading further, waits (bounded;
  // it stops waiting for the rest of the layer after one time-out) until
  // every pair has finished the epoch before that one.  Pairs that share an
  // operand panel then read it within a short time of each other, while it
  // is still in L2.  wave_ctr: zeroed counters, PairList::wave_per of each layer;
  // nullptr = off.
  unsigned* wave_ctr;
  int sync_stages;
  int wide;                // CTA-pair kernel: 1 = units of two super tiles (I, J), (I, J + 1) of a
                           //    row (tile list with four entries per unit; a unit without a second
                           //    tile has a null second entry, rows past N), A loaded once per stage
  int snake;               // 1: a pair walks K backwards on its odd-numbered tiles, so that a
                           //    wave starts on the K slices the previous wave left in L2
};

// What differs from layer to layer in a list of layers (PairList); a launch of
// one layer takes it from SqArgs.  Planes are entries of a pool, [entry][batch]
// matrices under one pair of tensor maps.
struct LayerOp {
  int y, g;                // plane entries: P = Y Y, or Y G + G Y (g >= 0, adjoint mode)
  int tri_y;               // as SqArgs::tri_y
  const float* Yin;
  float* Yout;
  const float* aux;        // as in SqArgs
  __half* p0_out;          // planes written: hp and lo' (split) or hi, or nullptr
  __half* p1_out;
  const double* rn;
  const float* rnp_in;
  float* rnp_out;
  const LayerParams* lp;   // [batch]; nullptr: chosen by the control steps
  double* dots_out;
  float* X;                // [batch] matrices X' = Y' + x_add[b] I, stored whole, or nullptr
  const double* x_add;
};

// A list of layers in one cooperative launch of the CTA-pair kernel.  Tiles of
// layer n + 1 of an instance start once all its tiles of layer n are stored.
struct PairList {
  const LayerOp* ops;      // [nops], or nullptr: the one layer that SqArgs describes
  int nops;
  int batch;
  int per;                 // units of an instance (all instances alike), when groups > 0
  int groups;              // 0: layer after layer over all units; else the batch is cut into this many groups
                           //   of instances, all layers of a group before the next.  64 x 2048, 11 layers:
                           //   groups of 5 16.1 ms, of 3 17.6, all 64 18.6 (planes and iterates through DRAM;
                           //   16.2 with the pairs kept in step, SqArgs::wave_ctr, as with a launch a layer);
                           //   all at the 1.4 kW power limit
  unsigned* done;          // [batch] zero: finished tiles over the layers
  unsigned* step;          // [batch] zero: layers whose sums, and control step, are complete
  LayerParams* rec;        // [nops + 1] parameters chosen by the control steps (ctl set: one instance)
  unsigned long long* stamps;  // [nops + 1] ns at the start and after each layer (ctl set), or nullptr
  int wave_per;            // SqArgs::wave_ctr entries of a layer (groups = 0)
  int cooperative;         // more than one layer: the pairs wait on one another
};

// tensor-core tile geometry
constexpr int kTcBM = 128;   // rows per CTA tile (TMEM lanes)
constexpr int kTcBN = 256;   // columns per CTA tile; 256 x 256 "super tiles" hold two CTA tiles
constexpr int kSimtB = 128;  // FFMA tile

// nan_row >= 0 (fault injection): that row of the stacked instances is
// treated as holding a NaN.
cudaError_t launch_gershgorin(const float* H, int N, long long ld, long long slot, int B, double2* partials,
                              unsigned* ticket, Ctl* ctl, double* bounds_out, int grid, cudaStream_t st,
                              long long nan_row = -1);
cudaError_t launch_gershgorin_batched(const float* const* Hs, const int* Ns, Ctl* ctl, int batch, double2* partials,
                                     unsigned* tickets, int grid_x, cudaStream_t st);
cudaError_t launch_input_layer(const float* const* Hs, const int* Ns, long long ld_in, float* Y, long long ld_y,
                               long long slot_y, __half* hi, __half* lo, __half* hp, long long ld_h, long long slot_h,
                               int rows_pad, int cols_pad, float lo_scale, Ctl* ctl, const double* bounds, double2* partials, unsigned* tickets,
                               int shift, int ctl_step, int batch, int grid_x, cudaStream_t st);
cudaError_t launch_split(const float* X, long long n, float lo_scale, __half* hi, __half* lo, int grid,
                         cudaStream_t st);
cudaError_t launch_split_pad(const float* X, long long ld_x, long long slot_x, int N, int B, float lo_scale,
                             __half* hi, __half* lo, __half* hp, long long ld_h, long long slot_h, int grid,
                             cudaStream_t st);
cudaError_t launch_materialize(const float* Y, long long ld_y, long long slot_y, int N, int B, const double* alpha,
                               float* out, long long ld_o, long long slot_o, int grid_x, cudaStream_t st);
cudaError_t launch_observable(const float* D, const float* A, long long n, double* block_out, int grid,
                              cudaStream_t st);

// rn[b][i] = sum_k Y[b][i][k]^2 in FP64 for every row of every instance.
// With ctl: instances whose next launch is inactive are skipped, and the
// last block of an instance runs its control step with (trY_new, sum rn).
cudaError_t launch_rownorm(const float* Y, long long ld_y, long long slot_y, const int* Ns, int batch, int max_rows,
                           double* rn, long long ld_rn, Ctl* ctl, double2* partials, unsigned* tickets, int grid_x,
                           cudaStream_t st);

// Single-accumulator split squaring (tcgen05, double-buffered TMEM): the
// three products hp hp + lo' hp + hp lo' = 2^(2s) (hi hi + lo hi + hi lo)
// go into one FP32 accumulator (hp = 2^s hi, lo' = 2^s lo).  tmaps: {p0(A),
// p1(A), p0(B), p1(B)} with p0 = hp, p1 = lo'; split = false: plain FP16
// with p0 = hi (p1 unused).  The epilogue writes the planes whose output
// pointers are set (hp_out and lo_out for split, hi_out for plain).
cudaError_t launch_syrk_tc1(const SqArgs& a, const CUtensorMap* tmaps, bool split, int grid, cudaStream_t st);
size_t syrk_tc1_smem_bytes(bool split);
// The same product run by CTA pairs (clusters of 2) whose MMAs span both CTAs
// (M = 256 per super tile, each CTA holding 128 rows of A and of B): tiles
// come in (h = 0, h = 1) pairs of one super tile, a.ntiles = 2 x super tiles.
// tmaps: {p0, p1} with 64 x 128 boxes and {p0, p1} with 64 x 64 boxes, through
// which the K blocks left of the diagonal are read transposed from the upper
// tiles.  A list of several layers is a cooperative launch, of at most
// syrk_tc2_max_pairs() pairs; adjoint: it holds adjoint layers.
cudaError_t launch_syrk_tc2(const SqArgs& a, const PairList& l, bool adjoint, const CUtensorMap* tmaps, bool split,
                            int grid, cudaStream_t st);
size_t syrk_tc2_smem_bytes(bool split);
int syrk_tc2_max_pairs();  // pairs of the device that can run at the same time (0: not known)

// Resident solve (csrc/resident.cu): all layers of a batch of instances in one
// cooperative launch on 128 x 128 tiles; the tiles of one instance are
// contiguous, starting at tile_off[b], tile_cnt[b] <= slots (two per CTA).  The
// instances' order is the same in every slot's list.
constexpr int kResTile = 128;
constexpr int kResStamps = kMaxL + 2;
constexpr int kMeetRows = 102;  // words of a gang's meeting rows
struct ResMaps {
  CUtensorMap m[2][4];  // per plane parity: {p0, p1} with 64 x 128 boxes, {p0, p1} with 64 x 64 boxes
};
struct ResArgs {
  const float* const* H;   // [batch] inputs [n_b, n_b]
  float* const* D;         // [batch] outputs
  const int* Ns;           // [batch]
  const uint32_t* tiles;   // [ntiles], rows and columns in units of 128
  int ntiles;
  const int* tile_off;     // [batch]
  const int* tile_cnt;     // [batch]
  Ctl* ctl;                // [batch]
  __half* p0[2];           // operand planes of even / odd layers: hp (split) or hi
  __half* p1[2];           //   lo' (split) or nullptr
  long long ld_h, slot_h;
  const double* rn;        // [batch][ld_rn] FP64 row norms of Y_0
  long long ld_rn;
  float* rnp[2];           // row-norm segment sums, as SqArgs::rnp_out
  long long ld_rnp, slot_rnp;
  double2* part;           // [batch][blocks] block sums of the input layer
  long long* sums;         // [batch][2][kMeetRows] meeting rows (csrc/resident.cuh), zero: of the layers, of FP64 sums
  double2* tile_sums;      // [ntiles] a tile's sums in FP64 (csrc/resident.cuh, meet_fp64)
  double* tile_dots;       // [ntiles] Tr[D H] per tile
  double* dots_out;        // [batch][3], entry 0: Tr[D H]
  unsigned* tickets;       // [batch] zero: finished blocks of the input layer
  const int* list_off;     // [2 grid + 1] slot c of CTA s processes the tiles
  const int* list;         //   list[list_off[c grid + s]] .. in turn
  unsigned* stamps;        // [batch][kResStamps] ns from an instance's start to the end of its k-th layer
  float lo_scale, lo_unscale;
  int shift, two_slots;
  int local;               // every instance is one tile: its planes stay in shared memory
  int stall;               // as SqArgs
  int* err;
  int* late;               // as SqArgs
  unsigned long long wait_ns;
};
cudaError_t launch_resident_input(const ResArgs& a, int vec_norm, int Nmax, int batch, cudaStream_t st);
cudaError_t launch_resident(const ResArgs& a, const ResMaps& maps, bool split, int grid, cudaStream_t st);

// Resident network layers (csrc/resident_net.cu).  One operation of every
// tile; planes are pool entries of [pool][batch] plane pairs.
enum NetFrom : int { NET_TMEM = 0, NET_INPUT = 1, NET_X = 2, NET_FULL = 3, NET_KEPT = 4 };
struct NetOp {
  int kind;                // 0: P = Y Y, 1: P = Y G + G Y (with dot products)
  int y, g;                // pool entries of the planes of Y and G
  int out;                 // pool entry written, or -1
  int layer;               // coefficients lp[layer][batch]
  int dot;                 // kind 1: layer of the dot products
  int from;                // the old value: tensor memory, the input layer of `in`, a matrix `in` with add[b] on
                           //   its diagonal, `in` as it is ([batch][N][N]), or `in` a tile-private store
  int tmem;                // 1: the new value stays in tensor memory
  int rnp;                 // segment sums: written at this parity, read at the other (or rn)
  int exact;               // full's diagonal from the unrounded FP64 one plus the coefficients' alpha_out
  int readout;             // 1: R += rc X', D = I - R into full; 2: R starts here as r_scale Y + r_add[b] I
  const float* in;
  const double* add;
  const double* rn;        // [batch][N] FP64 row norms of the input, or nullptr
  float* keep;             // tile-private store of the new value, or nullptr
  const float* aux;        // kind 1: tile-private store of Y, or nullptr: the matrix aux_x with aux_add[b] on its diagonal
  const float* aux_x;
  const double* aux_add;
  float* full;             // whole result matrices [batch][N][N], or nullptr
  float* full2;            // a second copy
  const double* full_add;  // [batch] added to full's diagonal, or nullptr
};
struct NetMaps {
  CUtensorMap m[4];        // {p0, p1} with 64 x 128 boxes, {p0, p1} with 64 x 64 boxes; pool x batch slots
};
struct NetArgs {
  int N, batch, nops, per, ntiles;  // per: tiles of a matrix
  const NetOp* ops;
  const LayerParams* lp;   // [layers][batch]
  const Ctl* ctl;          // [batch] bounds (NET_INPUT)
  __half* p0;
  __half* p1;              // nullptr: plain FP16
  long long ld_h, slot_h;
  float* rnp[2];
  long long ld_rnp, slot_rnp;
  float* R;                // tile-private readout
  float r_scale;
  const double* r_add;     // [batch]
  double* tile_dots;       // [layers][ntiles][3]
  const uint32_t* tiles;
  const int* list_off;     // as ResArgs
  const int* list;
  long long* sums;         // [batch][kMeetRows] meeting rows, zero
  float lo_scale, lo_unscale;
  int shift, two_slots;
  int stall;               // as SqArgs
  int* err;
  int* late;               // as SqArgs
  unsigned long long wait_ns;
};
struct NetInput {
  int N, batch, from, shift, vec_norm;
  const float* in;         // [count][N][N], matrix m of batch index m mod batch
  const double* add;       // NET_X: add[m / batch * add_stride + m mod batch] on the diagonal
  long long add_stride;
  const Ctl* ctl;
  __half* p0;              // plane pair m
  __half* p1;
  long long ld_h, slot_h;
  double* rn;              // [count][N], or nullptr
  float* x0;               // [count][N][N] Y_0 + alpha0 I, or nullptr
  const double* alpha0;
  float* y;                // [count][N][N] Y_0 from the row's super tile on, or nullptr
  float* r;                // [count][N][N] r_scale Y_0 + r_add[b] I, likewise, or nullptr
  float r_scale;
  const double* r_add;
  float lo_scale;
};
// The layers' coefficients and FP64 shifts from the bounds in ctl, on the device.
struct NetPlanArgs {
  int batch, L, shift;
  int expansion;           // 1: finite-temperature expansion (coef: theta [L][3], then c [L + 1]), table = readout's
                           //   identity part [batch]; 0: network (coef [L][3]), table = alpha_n [L + 1][batch]
  int backward;            // network: also the adjoint's coefficients at lp[L + n], and table + (L + 1) batch = -alpha_n
  const double* coef;
  const Ctl* ctl;
  LayerParams* lp;
  double* table;
  int* status;             // [batch] sp2_status of the bounds
  double* bounds;          // [batch][2] caller's copy, or nullptr
};
cudaError_t launch_net_plan(const NetPlanArgs& a, cudaStream_t st);
cudaError_t launch_net_input(const NetInput& x, int count, cudaStream_t st);
cudaError_t launch_net_dots(const double* tile_dots, int ntiles, int per, int L, int B, double* out, cudaStream_t st);
cudaError_t launch_resident_net(const NetArgs& a, const NetMaps& maps, bool split, int grid, cudaStream_t st);

// Resident FP32 solve (csrc/resident_fp32.cu): one instance, all layers in one
// cooperative launch; Y_0, its row norms and the first control step are there.
struct Res32Args {
  float* Y[2];             // iterates of even / odd layers, leading dimension ld_y (a multiple of 4)
  long long ld_y;
  int N;
  float* D;
  const uint32_t* tiles;   // [ntiles] upper tiles in units of the tile side
  int ntiles;
  Ctl* ctl;
  double* rn;              // [N] row norms of the layer's input
  long long* sums;         // [3][kMeetRows] meeting rows of the traces, of the square norms, of FP64 sums, zero
  double2* slots;          // [grid] each CTA's sum in FP64 (meet_fp64)
  unsigned* stamps;        // as ResArgs
  int* err;
  int* late;               // as SqArgs
  unsigned long long wait_ns;
};
cudaError_t launch_resident_fp32(const Res32Args& a, int tile, int grid, cudaStream_t st);

cudaError_t launch_syrk_simt(const SqArgs& a, int grid, cudaStream_t st);

// Tensor-core squaring.  tmaps: {hi(A box), lo(A box), hi(B box), lo(B box)}
// over the current split buffers, followed (nseg == 2) by the four maps of
// the second K segment.  split = false: plain FP16 (hi only).
cudaError_t launch_syrk_tc(const SqArgs& a, const CUtensorMap* tmaps, bool split, int grid, cudaStream_t st);
size_t syrk_tc_smem_bytes(bool split);

// Encodes a 3D tensor map over FP16 [batch][rows][ld] with box {box_k, box_rows, 1}.
bool make_tmap_f16(CUtensorMap* out, const void* base, int cols, int rows, int batch, long long ld, long long slot,
                   int box_k, int box_rows);

}  // namespace sp2
