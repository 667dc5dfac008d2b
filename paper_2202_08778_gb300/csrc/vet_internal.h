// vet_internal.h -- data shared by the host side and the kernels of libvet.
//
// Geometry is in cell units inside one block: memory-frame coordinates run
// from 0 to B along each axis of the block; the "upwind frame" of a direction
// flips every axis whose direction component is negative, so that backward
// rays always move towards lower upwind-frame coordinates and a block's
// upwind faces sit at upwind-frame coordinate 0.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace vet {

constexpr int kMaxBlock = 32;             // largest block edge B

// The thin-segment cubic: -(1 - e^-x) = y q(y), y = -x log2(e), for x < 1/4
// (q fitted for relative error by Lawson's iteratively reweighted least
// squares: 2.4e-7 in exact arithmetic, 3.4e-7 evaluated in FP32), and the
// threshold on y.
constexpr float kThinQ3 = 8.70478970381660493e-03f, kThinQ2 = 5.53004379372010468e-02f,
                kThinQ1 = 2.40211763951330648e-01f, kThinQ0 = 6.93147011611337405e-01f;
constexpr float kThinY = -0.36067376022224085f;  // x < 1/4
constexpr int kNever = 0x3fff;            // event index of an axis the ray never exits by

// Per-direction ray templates (Sec. 2.2.5 reading: long characteristics in a
// block).  A backward ray from a cell centre crosses the block's cell planes
// at parameters t = (m + 1/2)/|n_a| (m = 0, 1, ...) on axis a, independently
// of which cell it starts from; merging the three sequences gives one event
// list per direction.  A ray from a cell whose upwind-frame coordinate along
// axis a is l_a leaves the block at the event (a, m = l_a), whichever of the
// three comes first in the merged order (ties: lowest axis).  Face-node rays
// start on lattice points and cross planes at t = m/|n_a| (m = 1, 2, ...).
//
// The exit point of a ray leaving through axis a after depth l (cells:
// l + 1/2, nodes: l) has, along another axis b, the upwind-frame coordinate
// l_b + d with d = (1/2 or 0) - depth |n_b|/|n_a|; d depends on the direction
// and l only.  The host evaluates it in FP64 and stores k = floor(d) and the
// interpolation weights (f, 1 - f), f = d - k, so that the device never forms
// a position by cancellation.
//
// One direction's template is a byte blob laid out by TplLayout for the
// block edge B: a TplHead followed by the arrays below (16-byte aligned).
template <typename R>
struct TplHead {
  R n[3];     // direction
  R w;        // quadrature weight 4 pi / N
  int sgn[3]; // +1 if n_a >= 0 (a zero component counts as positive) else -1
  int ext;    // index of this direction in the documented HEALPix order
  int mirror; // 1: this template and its antipode's are exact mirror images
              // and every sign flips (no zero component)
              // (same event lengths, negated offsets, same exit tables)
  // quadrature coefficients w (1, nx, ny, nz, nx nx, ny ny, nz nz, nx ny,
  // nx nz, ny nz) of E, F and P (Eqs. 10-12, c = 1), rounded once from FP64;
  // two unused entries keep the array a multiple of 16 bytes
  alignas(16) R c[12];
  // the same ten coefficients as pairs (c_m, +-c_m) for a cell and its mirror
  // cell: the paired cell pass adds I(c, d) + I(c, -d) into E and P and
  // I(c, d) - I(c, -d) into F, and the mirror cell c' sees -d where c sees d,
  // so its F pair member is negated
  alignas(16) R cp[20];
};

// One event of a ray template: the length of the segment that ends at it,
// scaled by -h log2(e), and the byte offset in the shared-memory tile, from
// the ray's start cell, of the cell that segment crosses (0 for the first
// segment).  Rays are marched downwind, from their last event back to the
// start.
template <typename R>
struct alignas(2 * sizeof(R)) TplEvent {
  R len;
  int off;
};
// FP64 events carry an FP32 copy of the length beside it, from which the
// segment weight (vet_exp64.h) picks its table step: 1024 len.
template <>
struct alignas(16) TplEvent<double> {
  double len;
  int off;
  float lens;
};
inline void set_event(TplEvent<float> &e, double len, int off) { e = {(float)len, off}; }
inline void set_event(TplEvent<double> &e, double len, int off) { e = {len, off, (float)(1024.0 * len)}; }

// The head and the node-ray parts come first, so that the face pass stages
// only [0, node_bytes) of a template.
struct TplLayout {
  int nev;         // TplEvent<R>[3B]  node-ray events
  int npos;        // int16[3][B+1] merged index of node event (a, m); [a][0] = -1
  int nk;          // int16[3][2][B+1] floor(d) of node exits
  int nw;          // R[3][2][B+1][2]  (f, 1-f) of node exits
  int node_bytes;  // head and node-ray parts, a multiple of 16
  int cev;         // TplEvent<R>[3B]  cell-ray events
  int cpos;        // int16[3][B]  merged index of cell event (a, m)
  int ck;          // int16[3][2][B]   floor(d) of cell exits
  int cw;          // R[3][2][B][2]    (f, 1-f) of cell exits
  int bytes;       // total, a multiple of 16
};

__host__ __device__ inline int tpl_align16(int x) { return (x + 15) & ~15; }

template <typename R>
__host__ __device__ inline TplLayout tpl_layout(int B) {
  TplLayout L;
  int o = tpl_align16((int)sizeof(TplHead<R>));
  L.nev = o;  o = tpl_align16(o + 3 * B * (int)sizeof(TplEvent<R>));
  L.npos = o; o = tpl_align16(o + 3 * (B + 1) * 2);
  L.nk = o;   o = tpl_align16(o + 6 * (B + 1) * 2);
  L.nw = o;   o = tpl_align16(o + 6 * (B + 1) * 2 * (int)sizeof(R));
  L.node_bytes = o;
  L.cev = o;  o = tpl_align16(o + 3 * B * (int)sizeof(TplEvent<R>));
  L.cpos = o; o = tpl_align16(o + 3 * B * 2);
  L.ck = o;   o = tpl_align16(o + 6 * B * 2);
  L.cw = o;   o = tpl_align16(o + 6 * B * 2 * (int)sizeof(R));
  L.bytes = o;
  return L;
}

// Fixed sizes of one launch.
struct GridDims {
  int nx, ny, nz;     // cells
  int B;              // block edge
  int nbx, nby, nbz;  // blocks
  int nnode;          // (B+1)^2 face nodes per face
  int fstride;        // elements per stored face: (B+2)^2 rounded up to 16 bytes
  int ndir;           // directions
  long long ncell;    // nx*ny*nz
  int dir_tile;       // directions per cell-pass tile (0: default)
  int paired;         // 1: the cell order lists antipodal pairs (d, -d), see the paired cell pass
  int face_paired;    // 1: face-pass items are mirrored block pairs, see the paired face pass
  const uint32_t *cell_rec;  // ray records, see CellRec and NodeRec
  const uint2 *node_rec;
  const double *exp64;  // FP64 passes: tables of the segment weight (vet_exp64.h)
  int nsm;              // SMs of the device (0: unknown)
  long long beside;     // cells of the grids whose passes run beside this one's (a batch's other members)
};

// Ray records.  Where a ray leaves its block, through which entry of the exit
// tables, and at which node of the incoming faces it starts depend on the
// direction and the cell (or face node) alone, not on the block; a table of
// them, made once per context by ray_records_kernel, replaces the passes' per-ray
// search of the plane events and its index arithmetic.
//   cells: [N][B^3] words (internal direction order; cells in cell_rec_index order)
//   nodes: [N][6][(B+1)^2] words pairs: the nodes of each face axis, then of the
//     three faces merged, each in geom::node_order's order (null: row order)
struct CellRec {
  uint32_t v;  // exit event index 8 bits, row of the weight table 8, face entry (element of the three faces) 16
  __host__ __device__ int last() const { return (int)(v & 255u); }
  __host__ __device__ int row() const { return (int)((v >> 8) & 255u); }
  __host__ __device__ int face() const { return (int)(v >> 16); }
};
struct NodeRec {
  uint2 v;  // x: exit event index + 1, row, face entry as above; y: start cell in the tile 16 bits, stored node 16
  __host__ __device__ int last() const { return (int)(v.x & 255u) - 1; }
  __host__ __device__ int row() const { return (int)((v.x >> 8) & 255u); }
  __host__ __device__ int face() const { return (int)(v.x >> 16); }
  __host__ __device__ int start() const { return (int)(v.y & 65535u); }
  __host__ __device__ int out() const { return (int)(v.y >> 16); }
};
// Place of a block's cell in a direction's records: where the edge is a
// multiple of 4, the 4 x 4 x 2 bricks that the warps of the cell passes take,
// one after another; else row by row.
__host__ __device__ inline int cell_rec_index(int B, int x, int y, int z) {
  if (B % 4) return (z * B + y) * B + x;
  return (((z >> 1) * (B / 4) + (y >> 2)) * (B / 4) + (x >> 2)) * 32 + (z & 1) * 16 + (y & 3) * 4 + (x & 3);
}
inline size_t cell_rec_count(int N, int B) { return (size_t)N * B * B * B; }
inline size_t node_rec_count(int N, int B) { return (size_t)N * 6 * (B + 1) * (B + 1); }

// Shared-memory kappa/S tiles of a block, in entries of 8 bytes (kappa, S) or,
// for the FP32 mirrored passes, 16 bytes (kappa, kappa', S, S').  Face pass:
// cell (x, y, z) at x + (B+1) y + (B+1)^2 z; the three strides are odd, so a
// warp walking a row, column or pillar of a face (and any uniform shift of
// it) touches distinct banks.  Cell pass: where B is a multiple of 4, the y
// stride is the first above B that is 4 mod 8 entries (12 for 8, 20 for 12 and
// 16): a 4 x 4 layer of a warp's 4 x 4 x 2 cell brick is conflict free in 8-byte
// entries, a quarter warp's 4 x 2 cells in 16-byte ones.  Other edges are
// walked row by row and stored without padding.  The last entry is the cell
// pass's identity segment.
struct TileShape {
  int sy, sz, elems;
};
__host__ __device__ inline TileShape node_tile(int B) { return {B + 1, (B + 1) * (B + 1), (B + 1) * (B + 1) * B}; }
__host__ __device__ inline TileShape cell_tile(int B) {
  const int sy = B % 4 ? B : B + 8 - (B + 4) % 8;
  return {sy, sy * B, sy * B * B + 1};
}

// Stored faces: node (ub, uc) of a face, in the upwind frame of the direction
// (the in-plane axes flipped where the direction component is negative), at
// ub * (B + 2) + uc; row and column B + 1 are zero padding.
template <typename R>
__host__ __device__ inline int face_stride_elems(int B) {
  const int per = 16 / (int)sizeof(R);
  return ((B + 2) * (B + 2) + per - 1) / per * per;
}

// One work item of the face pass: a block and a run of directions of one
// octant, all at the same wavefront level.
struct FaceItem {
  int block;
  int dir_begin;     // internal direction index
  int dir_count;
  int mirror_begin;  // paired face pass: internal index of the antipode of dir_begin
  int octant;        // the directions' octant: bit a set where component a is negative
};

// Launchers (vet_kernels.cu).  All return the cudaGetLastError() of the
// launch.  R = float or double.  `bnd` holds the boundary faces materialised
// by launch_fill_boundary; `spin` bounds every device-side wait (polls of an
// mbarrier); a wait that gives up ORs a code into *status and the kernel
// returns early with its outputs incomplete.
//   status bits: 1 face-pass staging, 2 cell-pass staging, 4 cell-pass buffer
//   release or hand-over between two threads, 8 the final wait for copies still in flight.

// Face pass of one wavefront level: nitems items of at most max_dirs
// directions each.
template <typename R>
cudaError_t launch_face_level(const GridDims &g, const R *kappa, const R *S, const unsigned char *tpl,
                              const FaceItem *items, int nitems, int max_dirs, R *faces, const R *bnd,
                              long long spin, int *status, cudaStream_t st);

// Split of the paired cell pass's last partial wave.  With `total` CTAs and
// room for `wave` of them at once (SMs x CTAs per SM) the last wave holds
// r = total mod wave CTAs and leaves the other slots idle for a whole CTA's
// time; the last r CTAs' work is then cut into k shares of their direction
// tiles (k CTAs each), so that the tail takes about ceil(k r / wave) / k of
// a CTA's time.  The shares' partial moments meet in `part`
// ([slot][share][28, or 34 at edges other than 8 and 16][threads] floats) and the last share of a slot to
// finish (counted in `count`, which it resets) adds them in order and writes
// the outputs.
//
// A grid of fewer CTAs than one wave (total < wave) is split whole, every CTA
// into as many shares as fill the wave, so that a small grid's cell pass does
// not take one CTA's time on a part of the SMs.  Its results are the unsplit
// pass's bits (a small grid's closure equals the same grid's in a batch, or
// its blocks' in the learned closure's fallback): the shares store each
// antipodal pair's intensities, and the last share of an item adds
// them in the unsplit order (`ordered`).
struct TailPlan {
  int nfull = 0;          // CTAs that run whole (total - r)
  int k = 1;              // shares per split work item (1: no split)
  int slots = 0;          // r
  size_t part_bytes = 0;  // scratch the moments of the shares need
  bool ordered = false;   // total < wave: per-pair values instead of partial moments
};
TailPlan plan_tail_split(int B, int nblk, int nsm, int ndir, int dir_tile);
// The same for the FP64 cell pass, whose shares always store partial moments
// ([slot][share][14][threads] doubles), also on grids of less than one wave.
TailPlan plan_cell_split64(int B, int nblk, int nsm, int ndir, int dir_tile);
// Largest scratch of an ordered split (beyond: the grid runs unsplit, at edges
// other than 8 and 16 with two threads a pair of cells).
constexpr size_t kOrderedSplitMax = (size_t)128 << 20;

// One grid of a merged launch of the paired FP32 cell pass (the batched
// closure): what a single grid's launch passes as arguments.  M_out null:
// E goes to E_out (the floor rule's input) and only f is written.
struct CellGrid {
  GridDims g;
  const float *kappa, *S;
  const unsigned char *tpl;
  const int *order;
  const float *faces, *bnd;
  float *M_out, *E_out, *f_out;
  void *emax_bits;
  int *status;
};

// The paired FP32 cell pass (moments and f) over the blocks of several grids
// of block edge B (8 or 16) in one launch: items[i] = (grid index, block
// index), both device arrays; with_M: every grid writes M (else none does);
// one direction tile for all (0: untuned).
cudaError_t launch_cell_pass_merged(int B, bool with_M, int dir_tile, const CellGrid *grids, const int2 *items,
                                   int nitems, long long spin, cudaStream_t st);

// What the caller provides for the split: the SM count and the scratch
// (part: part_bytes, count: slots zeroed ints).  part == nullptr: no split
// of the moment passes (the trace needs no scratch).
struct TailSplit {
  int nsm = 0;
  float *part = nullptr;
  size_t part_bytes = 0;
  int *count = nullptr;
  int slots = 0;
};

// mode 0: moments + f (+ E for the floor rule); mode 1: write I_out.  The
// directions are visited in cell_order.  With a block_list (device, nlist
// block indices) only the cells of those blocks are computed.  `split`
// (paired FP32 pass only; null: none) cuts the last partial wave, see
// TailSplit; its part/count must hold the plan's slots.
template <typename R>
cudaError_t launch_cell_pass(const GridDims &g, int mode, const R *kappa, const R *S, const unsigned char *tpl,
                             const int *cell_order, const R *faces, const R *bnd, R *I_out, R *M_out, R *E_out,
                             R *f_out, void *emax_bits, long long spin, int *status, cudaStream_t st,
                             const int *block_list = nullptr, int nlist = 0, const TailSplit *split = nullptr);

// The floor rule on the cells of the listed blocks.
template <typename R>
cudaError_t launch_floor_fix_blocks(const GridDims &g, const int *block_list, int nlist, const R *E,
                                    const void *emax_bits, double floor_rel, R *f_out, cudaStream_t st);

// The ray records of every direction's template (node_order: device, may be
// null).
template <typename R>
cudaError_t launch_ray_records(const GridDims &g, const unsigned char *tpl, const uint16_t *node_order, uint32_t *cell_rec,
                               uint2 *node_rec, cudaStream_t st);

// bnd[face][d] <- constant Ib[face][ext(d)] (or 0 when Ib is NULL).
template <typename R>
cudaError_t launch_fill_boundary(const GridDims &g, const unsigned char *tpl, const R *Ib, R *bnd, void *emax_bits,
                                 cudaStream_t st);

template <typename R>
cudaError_t launch_floor_fix(long long ncell, const R *E, const void *emax_bits, double floor_rel, R *f_out,
                             cudaStream_t st, bool after_cell_pass = false);

// E64 (optional, device): E of every cell summed in FP64, w64 times the sum
// of I over the directions (the weights are all equal to w64).
template <typename R>
cudaError_t launch_moments(long long ncell, int ndir, const R *I, const R *coef, R *M_out, int nsm,
                           cudaStream_t st, double *E64 = nullptr, double w64 = 0.0);

// Dynamic shared memory of an unpaired face-pass CTA staging `dirs` directions.
size_t pass_smem_bytes(int B, int dirs, bool fp64);

// Largest cell-pass direction tile (<= want) whose two buffers fit.
int cell_tile_fit(int B, int want, bool fp64);

// The direction tile the paired FP32 cell pass runs with for a requested
// tile (0: untuned), after its staging ring is fitted to shared memory.
int pair_tile_fit(int B, int want);

// Dynamic shared memory of an unpaired cell-pass CTA with `nslots` staged
// directions.
size_t cell_smem_bytes(int B, int nslots, bool fp64);

// Directions per face-pass item (default; a context may be tuned to 1..8).
constexpr int kFaceGroup = 4;
constexpr int kMaxTune = 8;
// Default of the paired face pass.  An item's rays share its tile and its wait,
// so small blocks take more directions; from 13 on, eight directions' faces leave
// room for one CTA an SM instead of two.  Face pass, 192 directions, 4 and 8 a
// item: edge 4, 64^3 cells, 1.41 and 1.04 ms; 6, 60^3, 0.45 and 0.39; 8, 128^3,
// 1.86 and 1.56; 12, 108x84x60, 0.343 and 0.330; 14, 98^3, 0.580 and 0.596 (7);
// 16, 128^3, 0.757 and 0.834.
constexpr int face_pair_group(int B) { return B <= 12 ? 8 : kFaceGroup; }
// Largest block edge of the mirrored (paired) FP32 passes: their 16-byte tiles
// and staged directions fit a CTA's shared memory.
constexpr int kMaxPairBlock = 16;
// Smallest block edge of the paired cell pass: below, a CTA's few cells do not
// pay for its pairs of staged directions (cell pass, paired against unpaired: edge 4
// 0.42 and 0.38 ms, 5 0.36 and 0.34, 6 0.43 and 0.56, 12 1.6 and 2.7; the paired
// face pass is ahead from 2 on, 0.59 and 0.67 ms).  Those grids fill the SMs; what
// leaves them idle runs in shares (TailPlan) or two threads a pair of cells (HALVES
// in vet_kernels.cu), and is ahead of one ray a thread from one block on.
constexpr int kMinPairBlock = 6;

// Per-device kernel attributes; call with the context's device current.
cudaError_t prepare_kernels();

// Sets the calling thread's message returned by vet_last_error(NULL).
void set_thread_error(const char *msg);

}  // namespace vet
