// GB300 (sm_103a) kernels and C ABI of the compact third-order gas-kinetic
// scheme (Pan & Xu, arXiv:1412.4489).  See include/gks.h for the interface.
//
// One step = four or five launches on the handle's stream, all reading a device-resident
// control block so that the sequence can be captured once in a CUDA graph:
//   k_recon    dt = min(CFL * dt_cfl, dt_max, t_end - t) from the running min
//              (block 0), and the compact reconstruction of every cell (Section 3.2)
//              (FP64 in conservative variables: k_recon_lanes)
//   faces      gas evolution at every x-face and y-face (frame rotated: n = y, t = x; Section 2.2, 3.3, 4):
//              FP64 k_faces or k_faces_split, FP32 Euler k_flux_euler, FP32 Navier-Stokes
//              k_flux<0> and k_flux<1> on two streams
//   k_update   conservative update (Eq. finite) into FP64 averages, or in
//              FP32-bulk mode into double-float (hi + lo FP32) averages, the
//              ghost cells that are images of the updated cells, the next CFL
//              bound (warp-shuffle / block / atomic min) and the physical check
//   k_finish   the update's second and third pass, only for the positivity fallback; advances t and
//              the step counter
// A newly set state's ghost ring is filled as its cells are loaded (k_load_cells, gks_state.cuh); k_ghost refreshes it for
// the unit-level entry points.
// Cell averages and face values are double-buffered; the buffer in use is the
// parity of the device step counter, so a failed step leaves the last good
// state in place.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <string>
#include <type_traits>

#include "../../include/gks.h"
#include "gks_device.cuh"
#include "gks_grid.cuh"
#include "gks_state.cuh"

using namespace gks;

namespace {

constexpr int kProfileParts = 7;  // gks_profile_step's times: the fallback passes' and the end's are one kernel's

// ---------------------------------------------------------------------------
// ghost ring: perimeter of the padded cell array of the current buffer
// ---------------------------------------------------------------------------
template <class R>
__global__ void k_ghost(Geo g, Cells<R> U0, Cells<R> U1, const Ctrl* c, int force) {
  if (!force && c->skip) return;
  const int par = (int)(c->steps & 1);
  ghost_at<R>(g, par ? U1 : U0, blockIdx.x * blockDim.x + threadIdx.x);
}

// ---------------------------------------------------------------------------
// reconstruction; U is the padded cell-average array in the compute type
// ---------------------------------------------------------------------------
// begin = 1: block 0 also opens the step (ctrl_begin); the other blocks then do
// not look at the skip flag it sets (coefficients of a skipped step go unused).
// CHAR: reconstruction in characteristic variables.

// Position k of n along the grid, forwards or backwards.  A step's FP32 kernels go over the grid in alternating
// directions, each starting where the one before ended, and the next step the other way round (back: the step's
// parity): what was written last is still in the L2 cache.  1024^2 Euler 157.7 -> 153.4 us a step, Navier-Stokes 198 ->
// 195; smaller grids fit as a whole, larger ones gain little (2048^2 584.6 -> 582.1).
__device__ __forceinline__ unsigned along(unsigned k, unsigned n, int back) { return back ? n - 1 - k : k; }

// bytes (a multiple of 16, both addresses too) that the warp's lanes wrote to shared memory, to
// global memory in one bulk copy; complete on return.  Every lane of the warp calls it.
__device__ __forceinline__ void bulk_store(void* dst, const void* src, unsigned bytes) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if ((threadIdx.x & 31) == 0) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst),
                 "r"((unsigned)__cvta_generic_to_shared(src)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
}

// block heights (of 32 cells) and resident blocks per SM the reconstruction is compiled for.  FP32
// conservative 8 and 3 (80 registers hold a cell's 13 stencil vectors without spills; 4 blocks at 64 spill: 512^2
// step 49.5 against 48.4 us, 5 blocks 55), FP32 characteristic 8 and 2 (128; 1 and 3 are slower); FP64
// characteristic 1 and 8 (it needs more than 128, and one-warp blocks spread over the SMs evenly)
template <class R> struct ReconRows { static constexpr int value = 8; };
template <> struct ReconRows<double> { static constexpr int value = 1; };
template <class R, bool CHAR> struct ReconBlocks { static constexpr int value = 2; };
template <> struct ReconBlocks<float, false> { static constexpr int value = 3; };
template <> struct ReconBlocks<double, true> { static constexpr int value = 8; };

template <class R, class TW, bool CHAR>
__global__ void __launch_bounds__(32 * ReconRows<R>::value, ReconBlocks<R, CHAR>::value) k_recon(Geo g, const R* U0, const R* U1, const TW* Wx0, const TW* Wx1,
                                               const TW* Wy0, const TW* Wy1, R* __restrict__ rec, R dx, R dy,
                                               R weps, R wC, Ctrl* c, int force, int begin, double cfl,
                                               double dt_max, double t_end) {
  pdl_wait();
  if (begin) {
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0 && threadIdx.y == 0)
      ctrl_begin(c, cfl, dt_max, t_end);
  } else if (!force && c->skip) {
    return;
  }
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int par = (int)(c->steps & 1);
  const int j = (sizeof(R) == 8 ? blockIdx.z * gridDim.y + blockIdx.y : along(blockIdx.y, gridDim.y, par)) * blockDim.y + threadIdx.y;
  if constexpr (sizeof(R) == 8) {
    if (i >= g.nx || j >= g.ny) return;
    recon_cell<R, CHAR>(g, par ? U1 : U0, par ? Wx1 : Wx0, par ? Wy1 : Wy0, rec, i, j, dx, dy, weps, wC);
  } else {
    // FP32: a warp's 32 records are 3,072 contiguous bytes.  Written by its lanes they would go out as 16-byte
    // pieces at a stride of 96; they are laid down in shared memory and leave in one bulk copy
    // (2048^2: 156 -> 139 us).
    __shared__ __align__(16) R stage[ReconRows<R>::value][32 * kRec];
    if (j >= g.ny) return;  // whole warps: a block row is a row of cells
    R* mine = stage[threadIdx.y];
    if (i < g.nx) {
      R r[kRec];
      recon_record<R, CHAR>(g, par ? U1 : U0, par ? Wx1 : Wx0, par ? Wy1 : Wy0, i, j, dx, dy, weps, wC, r);
      Lay<R>::store_rec(mine, threadIdx.x, r);
      ghost_records(g, par ? U1 : U0, rec, i, j);
    }
    const int i0 = blockIdx.x * blockDim.x, count = g.nx - i0 < 32 ? g.nx - i0 : 32;
    bulk_store(rec + rec_at(g, i0, j) * kRec, mine, (unsigned)(count * kRec * sizeof(R)));
  }
  pdl_release();
}

// Warps to a block of the FP64 kernels, whose pipe serves a warp instruction for a quarter of an SM in 64 cycles
// whether its lanes are active or not: as many as spread all warps over the SMs in one block each, at most four, one
// for each quarter (one-warp blocks end up two to a quarter while others idle).
unsigned warps_per_block(unsigned long long warps, int sms) {
  const unsigned long long w = (warps + sms - 1) / sms;
  return w < 1 ? 1 : w > 4 ? 4 : (unsigned)w;
}

// FP64 in conservative variables: four lanes to a cell (recon_cell_lanes), eight cells to a warp,
// numbered through row by row
__global__ void __launch_bounds__(128, 6) k_recon_lanes(Geo g, const double* U0, const double* U1, const double* Wx0,
                                                        const double* Wx1, const double* Wy0, const double* Wy1,
                                                        double* __restrict__ rec, Ctrl* c, int force, int begin,
                                                        double cfl, double dt_max, double t_end) {
  pdl_wait();
  if (begin) {
    if (blockIdx.x == 0 && threadIdx.x == 0) ctrl_begin(c, cfl, dt_max, t_end);
  } else if (!force && c->skip) {
    return;
  }
  const unsigned long long n = (unsigned long long)g.nx * g.ny, k = (unsigned long long)blockIdx.x * (blockDim.x >> 2) + (threadIdx.x >> 2);
  const unsigned long long q = k < n ? k : n - 1;
  const int j = (int)(q / (unsigned)g.nx), i = (int)(q - (unsigned long long)j * g.nx);
  const int par = (int)(c->steps & 1);
  recon_cell_lanes(g, par ? U1 : U0, par ? Wx1 : Wx0, par ? Wy1 : Wy0, rec, i, j, k < n);
  pdl_release();
}

// ---------------------------------------------------------------------------
// face evolution
// ---------------------------------------------------------------------------
// resident 128-thread blocks per SM the FP32 face kernel is compiled for: Euler 5 (96 registers,
// 20 warps per SM; 20 bytes of spill), Navier-Stokes 4 (128 registers; at 96 it spills 100-144 bytes).
// x-faces at 2048^2, 4 / 5 blocks: Euler 222 / 207 us (194 as it is now); Navier-Stokes at 1024^2 79.5 / 80.4 us.  6 blocks (80
// registers) are slower for both, 3 slower for Navier-Stokes.
template <int NS> struct FluxBlocks { static constexpr int value = NS ? 4 : 5; };

// Navier-Stokes faces of one axis (FP32)
template <int AX, class R, class TW>
__global__ void __launch_bounds__(128, FluxBlocks<1>::value) k_flux(Geo g, FaceConst<R> C, const R* __restrict__ rec,
                                                                   TW* Wn0, TW* Wn1, R* __restrict__ F,
                                                                   const Ctrl* c, int force) {
  pdl_enter();
  if (!force && c->skip) return;
  const int par = (int)(c->steps & 1);
  const unsigned by = along(blockIdx.y, gridDim.y, !par);
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int j = by * blockDim.y + threadIdx.y;
  if (AX == 0 && (g.nx & 31) == 0 && blockIdx.x == gridDim.x - 1) {
    // the column of blocks past a row of nx = 32 k x-faces holds only the last face of
    // each row: it takes those faces 128 rows to a block, in whole warps, instead of one
    // busy lane per warp
    i = g.nx;
    j = by * 128 + threadIdx.y * 32 + threadIdx.x;
  }
  const int fx = AX == 0 ? g.nx + 1 : g.nx, fy = AX == 0 ? g.ny : g.ny + 1;
  if (i >= fx || j >= fy) return;
  // new face values go to the other buffer
  flux_face<AX, R, TW, 1>(g, C, rec, par ? Wn0 : Wn1, F, i, j, step_dt<R>(c));
}

template <class R, class TW>
struct FaceArgs {
  FaceConst<R> Cx, Cy;
  const R* rec;
  TW *Wx0, *Wx1, *Wy0, *Wy1;
  R *Fx, *Fy;
  unsigned nbx, first;
};

// FP32 Euler faces of both axes in one launch: blocks [0, nbx) take x-faces, the others y-faces, 32 x 4 to a
// block in tiles (tx tiles to a row); with nx a multiple of 32 the x-tiles' last column as in k_flux.  No second stream to
// fork to and join: 48^2 12.2 -> 10.9 us a step, 512^2 44.6 -> 43.8, from 1024^2 on the same.  (Navier-Stokes faces stay two
// kernels on two streams: mixing the larger bodies costs 2% at 1024^2.)
__global__ void __launch_bounds__(128, FluxBlocks<0>::value) k_flux_euler(Geo g, FaceArgs<float, float> a, const Ctrl* c, int force) {
  pdl_enter();
  if (!force && c->skip) return;
  const int par = (int)(c->steps & 1);
  const float dt = step_dt<float>(c);
  const unsigned b = along(blockIdx.x, gridDim.x, !par) + a.first, tx = (unsigned)(g.nx + 31) / 32, ny4 = (unsigned)(g.ny + 3) / 4;
  if (b < a.nbx) {
    int i, j;
    if (b < tx * ny4) {
      i = (int)(b % tx) * 32 + threadIdx.x;
      j = (int)(b / tx) * 4 + threadIdx.y;
    } else {  // the last faces of 128 rows
      i = g.nx;
      j = (int)(b - tx * ny4) * 128 + threadIdx.y * 32 + threadIdx.x;
    }
    if (i <= g.nx && j < g.ny) flux_face<0, float, float, 0>(g, a.Cx, a.rec, par ? a.Wx0 : a.Wx1, a.Fx, i, j, dt);
  } else {
    const unsigned q = b - a.nbx;
    const int i = (int)(q % tx) * 32 + threadIdx.x, j = (int)(q / tx) * 4 + threadIdx.y;
    if (i < g.nx && j <= g.ny) flux_face<1, float, float, 0>(g, a.Cy, a.rec, par ? a.Wy0 : a.Wy1, a.Fy, i, j, dt);
  }
}

// FP64: every face of the grid in one launch, 32 to a warp, x-faces in warps [0, nbx), y-faces after
// them, numbered through row by row: no idle lanes at the rows' ends, and no second launch with a tail of its own.
// (Instruction fetch, which speaks against mixing the two axes' bodies in FP32, does not matter at the FP64 pipe's
// pace.)  first: the first warp's number (a launch can take one axis alone).
template <int AX>
__device__ __forceinline__ bool face_at(const Geo& g, unsigned block, int lane, int& i, int& j) {
  const unsigned fx = AX == 0 ? g.nx + 1 : g.nx, fy = AX == 0 ? g.ny : g.ny + 1;
  const unsigned long long f = (unsigned long long)block * 32 + lane, n = (unsigned long long)fx * fy;
  const unsigned long long q = f < n ? f : n - 1;
  j = (int)(q / fx);
  i = (int)(q - (unsigned long long)j * fx);
  return f < n;
}

template <class R, class TW, int NS>
__global__ void __launch_bounds__(128, 2) k_faces(Geo g, FaceArgs<R, TW> a, const Ctrl* c, int force) {
  pdl_wait();
  if (!force && c->skip) return;
  const unsigned b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5) + a.first, lane = threadIdx.x & 31;
  const int par = (int)(c->steps & 1);
  const R dt = step_dt<R>(c);
  int i, j;
  if (b < a.nbx) {
    if (face_at<0>(g, b, lane, i, j))
      flux_face<0, R, TW, NS>(g, a.Cx, a.rec, par ? a.Wx0 : a.Wx1, a.Fx, i, j, dt);
  } else if (face_at<1>(g, b - a.nbx, lane, i, j)) {
    flux_face<1, R, TW, NS>(g, a.Cy, a.rec, par ? a.Wy0 : a.Wy1, a.Fy, i, j, dt);
  }
  pdl_release();
}

// The same with three warps to 32 faces (flux_face_split): for grids whose face warps are too few to keep the
// quarters of the SMs busy, where a face's serial time is the kernel's.
template <class R, class TW, int NS>
__global__ void __launch_bounds__(96, 2) k_faces_split(Geo g, FaceArgs<R, TW> a, const Ctrl* c, int force) {
  __shared__ SplitShare<R> sh;
  pdl_wait();
  if (!force && c->skip) return;
  const unsigned b = blockIdx.x + a.first;
  const int par = (int)(c->steps & 1), lane = threadIdx.x & 31;
  const R dt = step_dt<R>(c);
  int i, j;
  if (b < a.nbx) {
    const bool active = face_at<0>(g, b, lane, i, j);
    flux_face_split<0, R, TW, NS>(g, a.Cx, a.rec, par ? a.Wx0 : a.Wx1, a.Fx, i, j, active, dt, sh);
  } else {
    const bool active = face_at<1>(g, b - a.nbx, lane, i, j);
    flux_face_split<1, R, TW, NS>(g, a.Cy, a.rec, par ? a.Wy0 : a.Wy1, a.Fy, i, j, active, dt, sh);
  }
  pdl_release();
}

// Grids of at most kSplitWarps face warps per SM (both axes) take the split launch.  Step times, one warp / three
// warps to 32 faces (us): Euler 32^2 48 / 32, 69^2 (2.0 warps per SM) 49 / 38, 81^2 (2.7) 53 / 51, 96^2
// (3.8) 56 / 57; Navier-Stokes 66 / 38, 67 / 51, 72 / 70, 76 / 89.
constexpr unsigned kSplitWarps = 3;

// ---------------------------------------------------------------------------
// update, CFL bound of the new state, physical check
// ---------------------------------------------------------------------------
// Update pass 1, 2 or 3 (see update_cell): pass 1 marks the cells it leaves
// non-physical; pass 2 runs only if pass 1 marked cells, pass 3 only if pass 2
// still left one; a cell non-physical after pass 3 fails the step.  Each pass
// keeps its own running minimum of the CFL bound.  Blocks walk the grid's tiles
// (32 cells by the block's height) with a stride of the launch grid (update_grid): pass 1
// is a kernel of its own, k_update; passes 2 and 3 (usually no work) run in k_finish.
// Resident blocks per SM the update is compiled for: the rarely taken fallback path
// must not raise the register count of the common one (FP32: 64 registers).
template <class R> struct UpdateBlocks;
template <> struct UpdateBlocks<double> { static constexpr int value = 2; };
template <> struct UpdateBlocks<float> { static constexpr int value = 4; };

template <class R, class TW>
struct UpdateArgs {
  Cells<R> U0, U1;
  const R *Fx, *Fy;
  TW *Wx0, *Wx1, *Wy0, *Wy1;
  unsigned char* bad;
};

template <class R, class TW>
__device__ __forceinline__ void update_pass(const Geo& g, const UpdateArgs<R, TW>& a, Ctrl* c, int pass) {
  const int par = (int)(c->steps & 1);
  R inv_max = R(0);  // over the block's tiles: one block reduction per block
  const unsigned rows = (g.ny + blockDim.y - 1) / blockDim.y;
  for (unsigned q = blockIdx.y; q < rows; q += gridDim.y) {
    const int j0 = along(q, rows, par) * blockDim.y;
    for (int i0 = blockIdx.x * blockDim.x; i0 < g.nx; i0 += gridDim.x * blockDim.x) {
      const int i = i0 + threadIdx.x, j = j0 + threadIdx.y;
      R inv = R(0);
      if (i < g.nx && j < g.ny) {
        bool b;
        inv = update_cell<R, TW>(g, par ? a.U1 : a.U0, par ? a.U0 : a.U1, a.Fx, a.Fy, par ? a.Wx0 : a.Wx1,
                                 par ? a.Wy0 : a.Wy1, a.bad, pass, step_dt<R>(c), i, j, b);
        if (pass == 1) {
          a.bad[(size_t)j * g.nx + i] = b ? 1 : 0;
          if (b) atomicOr(&c->bad_found[0], 1);
        } else if (pass == 2) {
          if (b) atomicOr(&c->bad_found[1], 1);
        } else if (b && atomicCAS(&c->status, GKS_OK, GKS_ENONPHYSICAL) == GKS_OK) {
          c->fail_step = c->steps;
        }
      }
      inv_max = fmax(inv_max, inv);
    }
  }
  block_bound_to<R>(inv_max, &c->dtb[pass - 1]);
}

template <class R, class TW>
__global__ void __launch_bounds__(256, UpdateBlocks<R>::value) k_update(Geo g, UpdateArgs<R, TW> a, Ctrl* c) {
  pdl_enter();
  if (c->skip) return;
  update_pass<R, TW>(g, a, c, 1);
}

// Limit of the fallback's device waits, and the block whose arrival they miss (a test hook; -1: none).
struct Wait {
  unsigned long long limit_ns;
  int skip;
};

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Barrier of all blocks of a cooperative launch; bounded: a block that waits longer than the limit
// fails the step (GKS_ETIMEOUT) and returns false, as do the others.  Only time in which the block runs counts: a
// poll takes about a microsecond, so a longer gap between two of them than a millisecond is time in which this
// context did not have the device (time slices of other processes).
__device__ bool ctrl_barrier(Ctrl* c, Wait w) {
  __syncthreads();
  __shared__ int ok;
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    volatile unsigned* gen = &c->bar_gen;
    volatile int* status = &c->status;
    const unsigned my = *gen;
    __threadfence();
    if ((int)(blockIdx.y * gridDim.x + blockIdx.x) != w.skip && atomicAdd(&c->bar_count, 1u) + 1 == gridDim.x * gridDim.y) {
      c->bar_count = 0;
      __threadfence();
      atomicAdd(&c->bar_gen, 1u);
    }
    unsigned long long last = global_ns(), waited = 0;
    while (*gen == my && *status != GKS_ETIMEOUT) {
      const unsigned long long t = global_ns(), d = t - last;
      waited += d < 1000000ull ? d : 1000000ull;
      last = t;
      if (waited > w.limit_ns) atomicExch(&c->status, GKS_ETIMEOUT);
      __nanosleep(200);
    }
    __threadfence();
    ok = *gen != my;
  }
  __syncthreads();
  return ok;
}

// Passes 2 and 3, when they are needed, and the step's end: one cooperative launch of at most one wave, whose blocks
// meet at a barrier after each pass.  Usually there is no work and the first thread ends the step.  In
// place of three launches (two passes, the end): 64^2 FP32 14.2 -> 12.2 us a step, 512^2 48.2 -> 44.3, 200 x 1
// FP64 39.5 -> 35.6; with programmatic serialisation as well as the cooperative attribute (without:
// 12.8, 47.2, 35.5).
// mirror (optional): page-locked host memory that the first thread leaves the control block in, for a caller that waits
// for this step.
template <class R, class TW>
__global__ void __launch_bounds__(256, UpdateBlocks<R>::value) k_finish(Geo g, UpdateArgs<R, TW> a, Ctrl* c, Ctrl* mirror, Wait w) {
  pdl_enter();
  const bool first = blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0;
  if (!c->skip) {
    bool met = true;
    if (c->bad_found[0]) {
      update_pass<R, TW>(g, a, c, 2);
      met = ctrl_barrier(c, w);
      if (met && *(volatile int*)&c->bad_found[1]) {
        update_pass<R, TW>(g, a, c, 3);
        met = ctrl_barrier(c, w);
      }
    }
    if (first && met) ctrl_end(c);
  }
  if (first && mirror) *mirror = *c;
}

// launch grid of an update in tiles of 32 x rows cells: pass 1 takes one wave of resident
// blocks (blocks_per_sm per SM), each walking ceil(tiles / wave) tiles along y, so
// that the per-block work (control reads, the CFL reduction) is shared by its tiles;
// the fallback passes at most one block per SM (usually no work).  Pass 1 of the FP64 form takes
// warps_per_block rows: its bound is the FP64 pipe too (81^2 in 256-thread blocks keeps 33 of 152 SMs busy).
constexpr int kUpdateRows = 8;

dim3 update_grid(const Geo& g, int pass, int sms, int blocks_per_sm, int rows) {
  unsigned tx = (unsigned)((g.nx + 31) / 32), ty = (unsigned)((g.ny + rows - 1) / rows);
  if (pass == 1) {
    const unsigned wave = (unsigned)sms * (unsigned)(blocks_per_sm * (kUpdateRows / rows));
    const unsigned fit = wave / tx > 0 ? wave / tx : 1;  // block rows that fit in one wave
    const unsigned k = (ty + fit - 1) / fit;             // tiles per block
    ty = (ty + k - 1) / k;
  }
  if (pass > 1) {
    if (tx > 8) tx = 8;
    const unsigned cy = (unsigned)(sms / (int)tx > 0 ? sms / (int)tx : 1);
    if (ty > cy) ty = cy;
  }
  return dim3(tx, ty);
}

// face values = mean of the two adjacent averages (ghosts included)
template <int AX, class TW>
__global__ void k_init_W(Geo g, Cells<TW> U0, Cells<TW> U1, TW* W0, TW* W1, const Ctrl* c) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int fx = AX == 0 ? g.nx + 1 : g.nx, fy = AX == 0 ? g.ny : g.ny + 1;
  if (i >= fx || j >= fy) return;
  const int par = (int)(c->steps & 1);
  const Cells<TW> U = par ? U1 : U0;
  TW* W = par ? W1 : W0;
  const size_t n = (size_t)fx * fy, o = (size_t)j * fx + i;
  for (int v = 0; v < 4; ++v) {
    const double a = U.get(g, v, AX == 0 ? i - 1 : i, AX == 0 ? j : j - 1);
    const double b = U.get(g, v, i, j);
    W[Lay<TW>::w(n, v, 0, o)] = W[Lay<TW>::w(n, v, 1, o)] = TW(0.5 * (a + b));
  }
}

template <class R>
__global__ void k_coef_out(Geo g, Cells<R> U0, Cells<R> U1, const R* rec, double* out, const Ctrl* c) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= g.nx || j >= g.ny) return;
  const Cells<R> U = (c->steps & 1) ? U1 : U0;
  const size_t N = (size_t)g.nx * g.ny, o = (size_t)j * g.nx + i;
  const R* r = rec + rec_at(g, i, j) * kRec;
  for (int v = 0; v < 4; ++v) {
    out[(size_t)(v * 6) * N + o] = U.get(g, v, i, j);
    for (int k = 0; k < 5; ++k) out[(size_t)(v * 6 + k + 1) * N + o] = (double)r[4 + 4 * k + v];
  }
}

// fluxes as planes [4][faces]
template <class R>
__global__ void k_flux_out(const R* F, double* dst, size_t faces) {
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < 4 * faces) dst[k] = (double)F[Lay<R>::f(faces, (int)(k / faces), k % faces)];
}

// opens a step of the partitioned form with the dt the caller reduced over all slabs
__global__ void k_part_begin(Ctrl* c, double dt) {
  c->dt = dt;
  c->dt_f = (float)dt;
  c->skip = (c->status != GKS_OK || !(dt > 0.0)) ? 1 : 0;
  c->dtb[0] = c->dtb[1] = c->dtb[2] = dbits(INFINITY);
  c->bad_found[0] = c->bad_found[1] = 0;
}

__global__ void k_set_dt(Ctrl* c, double dt) {
  c->dt = dt;
  c->dt_f = (float)dt;
  c->skip = 0;
}

}  // namespace

// ===========================================================================
// host side
// ===========================================================================
// steps per graph of gks_advance: a graph's start costs 3 to 5 us beyond its steps (10 steps of a 1024^2 grid
// as 4 + 4 + 1 + 1 graphs instead of ten)
constexpr int kGraphSteps[3] = {16, 4, 1};

// Default limit of the fallback's device waits.  A block waits for the others' shares of a pass, so the limit grows
// with the share: kWaitTileSeconds for each 32 x 8 tile a block walks.  A tile whose 1,024 faces are all evolved
// again takes below 0.2 ms in FP64 (some 1,200 FP64 instructions a thread, four warps to a quarter of an
// SM, 64 cycles each).
constexpr double kWaitSeconds = 2.0, kWaitTileSeconds = 2e-3;

struct gks_handle {
  Geo g;
  int prec;
  cudaStream_t stream;
  bool own_stream;
  cudaStream_t side;              // the y-face evolution runs here, beside the x-faces
  cudaEvent_t fork, join;         // recon -> y-faces, y-faces -> update
  int device;
  int sms;  // multiprocessors of the device
  double* U[2];      // cell averages (Cells<R>: FP64, or FP32 hi / lo planes), 4 * plane doubles each
  void* Wx[2];
  void* Wy[2];
  void* rec;  // reconstruction records (rec_count(g) values of the compute type)
  void* Fx;
  void* Fy;
  unsigned char* bad;  // cells whose first update failed (positivity fallback)
  Ctrl* ctrl;
  Ctrl* hctrl;       // pinned mirror
  double* staging;   // device FP64 scratch for host transfers
  size_t staging_n;
  cudaGraphExec_t graph[3];  // kGraphSteps steps each, captured when first needed
  double graph_cfl, graph_tend;
  double wait_s = kWaitSeconds;  // gks_set_wait_limit
  int wait_skip = -1;
  std::string err;
};

static thread_local std::string g_create_err;

namespace {

size_t n_wx(const Geo& g) { return (size_t)8 * g.ny * (g.nx + 1); }
size_t n_wy(const Geo& g) { return (size_t)8 * (g.ny + 1) * g.nx; }
size_t n_u(const Geo& g) { return (size_t)4 * g.nx * g.ny; }

gks_status fail(gks_handle* h, gks_status s, const std::string& msg) {
  if (h) h->err = msg;
  return s;
}

#define CK(call)                                                                              \
  do {                                                                                        \
    cudaError_t e_ = (call);                                                                  \
    if (e_ != cudaSuccess)                                                                    \
      return fail(h, GKS_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_));          \
  } while (0)

dim3 grid2(int nx, int ny, dim3 b) { return dim3((nx + b.x - 1) / b.x, (ny + b.y - 1) / b.y); }

// launch of a step kernel; pdl: with programmatic stream serialisation (see pdl_enter)
template <typename... KArgs, typename... Args>
cudaError_t launch(bool pdl, void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <class R>
FaceConst<R> fconst(const Geo& g, int axis) {
  return grid_face_const<R>(g, axis);
}

// cell-average buffer b, and the compute-type array of its averages
template <class R> Cells<R> cellbuf(const gks_handle* h, int b) { return Cells<R>{(R*)h->U[b]}; }
template <class R> const R* cells(const gks_handle* h, int b) { return (const R*)h->U[b]; }

template <class R>
void launch_ghost(gks_handle* h, int force) {
  const Geo& g = h->g;
  k_ghost<R><<<(perimeter(g) + 127) / 128, 128, 0, h->stream>>>(g, cellbuf<R>(h, 0), cellbuf<R>(h, 1), h->ctrl, force);
}

template <class R, class TW>
cudaError_t launch_update(bool pdl, cudaStream_t s, const Geo& g, int sms, const UpdateArgs<R, TW>& a, Ctrl* c) {
  const int rows = sizeof(R) == 8 ? (int)warps_per_block((unsigned long long)((g.nx + 31) / 32) * g.ny, sms) : kUpdateRows;
  return launch(pdl, k_update<R, TW>, update_grid(g, 1, sms, UpdateBlocks<R>::value, rows), dim3(32, rows), s, g, a, c);
}

template <class R, class TW>
cudaError_t launch_finish(cudaStream_t s, const Geo& g, int sms, const UpdateArgs<R, TW>& a, Ctrl* c, Ctrl* mirror,
                          double wait_s, int wait_skip, bool pdl = true) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = update_grid(g, 2, sms, 1, kUpdateRows);
  const dim3 tiles = grid2(g.nx, g.ny, dim3(32, kUpdateRows));
  const double per_block = (double)((tiles.x + cfg.gridDim.x - 1) / cfg.gridDim.x) *
                           ((tiles.y + cfg.gridDim.y - 1) / cfg.gridDim.y);
  const Wait w{(unsigned long long)((wait_s + kWaitTileSeconds * per_block) * 1e9), wait_skip};
  cfg.blockDim = dim3(32, kUpdateRows);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k_finish<R, TW>, g, a, c, mirror, w);
}

template <class R, class TW>
cudaError_t launch_recon(bool pdl, cudaStream_t s, const Geo& g, int sms, const R* U0, const R* U1, const TW* Wx0, const TW* Wx1,
                         const TW* Wy0, const TW* Wy1, R* rec, Ctrl* c, int force, int begin, double cfl, double dt_max,
                         double t_end) {
  if constexpr (sizeof(R) == 8) {
    const unsigned long long warps = ((unsigned long long)g.nx * g.ny + 7) / 8;
    const unsigned w = warps_per_block(warps, sms);
    if (!g.characteristic)
      return launch(pdl, k_recon_lanes, dim3((unsigned)((warps + w - 1) / w)), dim3(32 * w), s, g, U0, U1,
                    Wx0, Wx1, Wy0, Wy1, rec, c, force, begin, cfl, dt_max, t_end);
    const dim3 b(32, ReconRows<R>::value);
    // block rows beyond the grid's y limit continue in z
    const unsigned rows = (unsigned)g.ny, gy = rows < 65535u ? rows : 65535u;
    return launch(pdl, k_recon<R, TW, true>, dim3((unsigned)(g.nx + 31) / 32, gy, (rows + gy - 1) / gy), b, s, g, U0, U1, Wx0,
                  Wx1, Wy0, Wy1, rec, R(g.dx), R(g.dy), R(g.weno_eps), R(g.weno_C), c, force, begin, cfl, dt_max, t_end);
  } else {
    const dim3 b(32, ReconRows<R>::value);
    return launch(pdl, g.characteristic ? k_recon<R, TW, true> : k_recon<R, TW, false>, grid2(g.nx, g.ny, b), b, s, g, U0,
                  U1, Wx0, Wx1, Wy0, Wy1, rec, R(g.dx), R(g.dy), R(g.weno_eps), R(g.weno_C), c, force, begin, cfl, dt_max,
                  t_end);
  }
}

template <class R, class TW>
cudaError_t launch_recon(gks_handle* h, int force, int begin = 0, double cfl = 0, double dt_max = 0,
                         double t_end = 0, bool pdl = false) {
  return launch_recon<R, TW>(pdl, h->stream, h->g, h->sms, cells<R>(h, 0), cells<R>(h, 1), (const TW*)h->Wx[0], (const TW*)h->Wx[1],
                             (const TW*)h->Wy[0], (const TW*)h->Wy[1], (R*)h->rec, h->ctrl, force, begin, cfl, dt_max, t_end);
}

// The FP64 face launch over both axes (axes 3) or one of them (1: x, 2: y).
template <class R, class TW>
cudaError_t launch_faces(bool pdl, cudaStream_t s, const Geo& g, int sms, const R* rec, TW* Wx0, TW* Wx1, TW* Wy0, TW* Wy1,
                         R* Fx, R* Fy, const Ctrl* c, int force, int axes = 3) {
  const unsigned nbx = (unsigned)(((unsigned long long)(g.nx + 1) * g.ny + 31) / 32);
  const unsigned nby = (unsigned)(((unsigned long long)g.nx * (g.ny + 1) + 31) / 32);
  const FaceArgs<R, TW> a{fconst<R>(g, 0), fconst<R>(g, 1), rec, Wx0, Wx1, Wy0, Wy1, Fx, Fy, nbx, axes == 2 ? nbx : 0};
  const unsigned n = (axes & 1 ? nbx : 0) + (axes & 2 ? nby : 0);
  const bool ns = g.mu > 0.0, split = (unsigned long long)nbx + nby <= (unsigned long long)kSplitWarps * sms;
  if (split)
    return launch(pdl, ns ? k_faces_split<R, TW, 1> : k_faces_split<R, TW, 0>, dim3(n), dim3(96), s, g, a, c, force);
  const unsigned w = warps_per_block(n, sms);
  return launch(pdl, ns ? k_faces<R, TW, 1> : k_faces<R, TW, 0>, dim3((n + w - 1) / w), dim3(32 * w), s, g, a, c, force);
}

// ev (optional, kProfileParts + 1 events): recorded before each kernel and after the last.
// with_begin_end = false (face evaluation of the current state for gks_debug_flux):
// the ghost ring is refreshed first and the step is neither opened nor closed.
template <class R, class TW>
gks_status launch_step_kernels(gks_handle* h, double cfl, double dt_max, double t_end, bool with_begin_end,
                               bool do_update, int force, cudaEvent_t* ev = nullptr, bool do_recon = true, bool mirror = false) {
  const Geo& g = h->g;
  cudaStream_t s = h->stream;
  auto mark = [&](int k) {
    if (ev) cudaEventRecord(ev[k], s);
  };
  if (!with_begin_end && do_recon) launch_ghost<R>(h, force);
  // programmatic dependent launch between the step's kernels, except when events
  // are recorded between them (per-kernel timing)
  const bool pdl = ev == nullptr;
  cudaError_t le = cudaSuccess;
  auto keep = [&](cudaError_t e) {
    if (le == cudaSuccess) le = e;
  };
  mark(0);
  if (do_recon) keep(launch_recon<R, TW>(h, force, with_begin_end ? 1 : 0, cfl, dt_max, t_end, pdl));
  mark(1);
  const dim3 bf(32, 4);
  bool fork = false;
  if constexpr (sizeof(R) == 8) {
    auto faces = [&](int axes) {
      keep(launch_faces<R, TW>(pdl, s, g, h->sms, (const R*)h->rec, (TW*)h->Wx[0], (TW*)h->Wx[1], (TW*)h->Wy[0],
                               (TW*)h->Wy[1], (R*)h->Fx, (R*)h->Fy, (const Ctrl*)h->ctrl, force, axes));
    };
    if (ev) faces(1);
    mark(2);
    faces(ev ? 2 : 3);
  } else {
    if (g.mu > 0.0) {
      // the x- and y-face evolutions are independent: without per-kernel timing the y-faces run
      // on a side stream (fork after the reconstruction, join before the update), so that each
      // fills the other's tail wave
      fork = ev == nullptr;
      auto yfaces = [&](bool p, cudaStream_t t) {
        keep(launch(p, k_flux<1, R, TW>, grid2(g.nx, g.ny + 1, bf), bf, t, g, fconst<R>(g, 1), (const R*)h->rec,
                    (TW*)h->Wy[0], (TW*)h->Wy[1], (R*)h->Fy, (const Ctrl*)h->ctrl, force));
      };
      if (fork) {
        keep(cudaEventRecord(h->fork, s));
        keep(cudaStreamWaitEvent(h->side, h->fork, 0));
        yfaces(false, h->side);
        keep(cudaEventRecord(h->join, h->side));
      }
      keep(launch(pdl, k_flux<0, R, TW>, grid2(g.nx + 1, g.ny, bf), bf, s, g, fconst<R>(g, 0), (const R*)h->rec,
                  (TW*)h->Wx[0], (TW*)h->Wx[1], (R*)h->Fx, (const Ctrl*)h->ctrl, force));
      mark(2);
      if (fork) keep(cudaStreamWaitEvent(s, h->join, 0));
      else yfaces(pdl, s);
    } else {
      const unsigned tx = (unsigned)(g.nx + 31) / 32, ny4 = (unsigned)(g.ny + 3) / 4;
      const unsigned nbx = tx * ny4 + ((g.nx & 31) ? 0 : (unsigned)(g.ny + 127) / 128);
      const unsigned nby = tx * ((unsigned)g.ny / 4 + 1);
      auto faces = [&](int axes) {
        const FaceArgs<R, TW> a{fconst<R>(g, 0), fconst<R>(g, 1), (const R*)h->rec, (TW*)h->Wx[0], (TW*)h->Wx[1],
                                (TW*)h->Wy[0], (TW*)h->Wy[1], (R*)h->Fx, (R*)h->Fy, nbx, axes == 2 ? nbx : 0};
        keep(launch(pdl, k_flux_euler, dim3((axes & 1 ? nbx : 0) + (axes & 2 ? nby : 0)), bf, s, g, a, (const Ctrl*)h->ctrl,
                    force));
      };
      if (ev) faces(1);
      mark(2);
      faces(ev ? 2 : 3);
    }
  }
  mark(3);
  if (do_update) {
    const UpdateArgs<R, TW> a{cellbuf<R>(h, 0), cellbuf<R>(h, 1), (const R*)h->Fx, (const R*)h->Fy, (TW*)h->Wx[0], (TW*)h->Wx[1],
                              (TW*)h->Wy[0], (TW*)h->Wy[1], h->bad};
    // after the join (two predecessors): an ordinary launch
    keep(launch_update<R, TW>(pdl && !fork, s, g, h->sms, a, h->ctrl));
    mark(4);
    keep(launch_finish<R, TW>(s, g, h->sms, a, h->ctrl, mirror ? h->hctrl : nullptr, h->wait_s, h->wait_skip, pdl));
  } else {
    mark(4);
  }
  mark(5);
  mark(6);
  mark(7);
  CK(le);
  CK(cudaGetLastError());
  return GKS_OK;
}

gks_status launch_step(gks_handle* h, double cfl, double dt_max, double t_end, bool mirror = false) {
  if (h->prec == GKS_FP64) return launch_step_kernels<double, double>(h, cfl, dt_max, t_end, true, true, 0, nullptr, true, mirror);
  return launch_step_kernels<float, float>(h, cfl, dt_max, t_end, true, true, 0, nullptr, true, mirror);
}

// the status that the control block holds, as a call's result
gks_status step_status(gks_handle* h, const char* what) {
  const gks_status st = (gks_status)h->hctrl->status;
  if (st == GKS_OK) return st;
  return fail(h, st, st == GKS_ETIMEOUT ? "a device wait of the positivity fallback ran out; state kept" : what);
}

gks_status read_ctrl(gks_handle* h) {
  CK(cudaMemcpyAsync(h->hctrl, h->ctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return GKS_OK;
}

void destroy_graphs(gks_handle* h) {
  for (cudaGraphExec_t& x : h->graph) {
    if (x) cudaGraphExecDestroy(x);
    x = nullptr;
  }
}

gks_status capture(gks_handle* h, int nsteps, double cfl, double t_end, cudaGraphExec_t* out) {
  cudaGraph_t graph;
  CK(cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
  gks_status st = GKS_OK;
  for (int k = 0; k < nsteps && st == GKS_OK; ++k) st = launch_step(h, cfl, INFINITY, t_end);
  cudaError_t e = cudaStreamEndCapture(h->stream, &graph);
  if (st != GKS_OK) return st;
  if (e != cudaSuccess) return fail(h, GKS_ECUDA, std::string("capture: ") + cudaGetErrorString(e));
  e = cudaGraphInstantiate(out, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) return fail(h, GKS_ECUDA, std::string("instantiate: ") + cudaGetErrorString(e));
  return GKS_OK;
}

// Loads a state.  dU, dWx, dWy: device-accessible arrays, except that one flagged in stage_u / stage_x / stage_y is a
// host array copied through the staging buffer first (in turn: the kernel that reads it comes before the next
// copy in the stream).  dWx / dWy null: mean of the adjacent averages.
template <class TW>
gks_status load_state(gks_handle* h, double t, const double* dU, const double* dWx, const double* dWy, bool stage_u = false,
                      bool stage_x = false, bool stage_y = false) {
  const Geo& g = h->g;
  cudaStream_t s = h->stream;
  const dim3 b2(32, 8);
  const Cells<TW> U0 = cellbuf<TW>(h, 0), U1 = cellbuf<TW>(h, 1);
  TW *Wx0 = (TW*)h->Wx[0], *Wx1 = (TW*)h->Wx[1], *Wy0 = (TW*)h->Wy[0], *Wy1 = (TW*)h->Wy[1];
  const size_t nfx = n_wx(g) / 8, nfy = n_wy(g) / 8;
  auto staged = [&](const double* src, size_t n) {
    const cudaError_t e = cudaMemcpyAsync(h->staging, src, n * sizeof(double), cudaMemcpyHostToDevice, s);
    return e;
  };
  k_state_begin<<<1, 1, 0, s>>>(h->ctrl, t, 1);
  if (stage_u) {
    CK(staged(dU, n_u(g)));
    dU = h->staging;
  }
  k_load_cells<TW><<<blocks_of((size_t)g.nx * g.ny), 256, 0, s>>>(g, dU, U0, U1, h->ctrl);
  for (int axis = 0; axis < 2; ++axis) {
    const double*& src = axis == 0 ? dWx : dWy;
    const size_t n = axis == 0 ? nfx : nfy;
    if (!src) {
      if (axis == 0) k_init_W<0, TW><<<grid2(g.nx + 1, g.ny, b2), b2, 0, s>>>(g, U0, U1, Wx0, Wx1, h->ctrl);
      else k_init_W<1, TW><<<grid2(g.nx, g.ny + 1, b2), b2, 0, s>>>(g, U0, U1, Wy0, Wy1, h->ctrl);
    } else if (axis == 0 ? stage_x : stage_y) {
      CK(staged(src, 8 * n));
      k_face_values<TW, true><<<blocks_of(n), 256, 0, s>>>(axis == 0 ? h->staging : nullptr, axis == 0 ? nullptr : h->staging,
                                                           nfx, nfy, Wx0, Wx1, Wy0, Wy1, h->ctrl);
      src = nullptr;
    }
  }
  if (dWx || dWy)
    k_face_values<TW, true><<<blocks_of((dWx ? nfx : 0) + (dWy ? nfy : 0)), 256, 0, s>>>(
        const_cast<double*>(dWx), const_cast<double*>(dWy), nfx, nfy, Wx0, Wx1, Wy0, Wy1, h->ctrl);
  CK(cudaGetLastError());
  return GKS_OK;
}

template <class TW>
gks_status store_state(gks_handle* h, double* dU, double* dWx, double* dWy) {
  const Geo& g = h->g;
  cudaStream_t s = h->stream;
  const size_t nfx = n_wx(g) / 8, nfy = n_wy(g) / 8;
  if (dU)
    k_store_cells<TW><<<blocks_of((size_t)g.nx * g.ny), 256, 0, s>>>(g, dU, cellbuf<TW>(h, 0), cellbuf<TW>(h, 1), h->ctrl);
  if (dWx || dWy)
    k_face_values<TW, false><<<blocks_of((dWx ? nfx : 0) + (dWy ? nfy : 0)), 256, 0, s>>>(
        dWx, dWy, nfx, nfy, (TW*)h->Wx[0], (TW*)h->Wx[1], (TW*)h->Wy[0], (TW*)h->Wy[1], h->ctrl);
  CK(cudaGetLastError());
  return GKS_OK;
}

void make_geo(Geo& g, int nx, int ny, double Lx, double Ly, double gamma, double Pr, double mu, const gks_bc* bc,
              const gks_options& o) {
  memset(&g, 0, sizeof(g));
  g.nx = nx; g.ny = ny;
  g.dx = Lx / nx; g.dy = Ly / ny;
  g.gamma = gamma; g.mu = mu; g.Pr = Pr;
  g.weno_eps = o.weno_eps; g.weno_C = o.weno_C; g.tau_eps = o.tau_eps; g.tau_C = o.tau_C;
  g.viscous_dt = o.viscous_dt;
  g.characteristic = o.characteristic;
  for (int k = 0; k < 4; ++k) {
    g.bc.kind[k] = bc ? bc[k].kind : GKS_BC_PERIODIC;
    g.bc.uw[k] = bc ? bc[k].u_wall : 0.0;
    g.bc.vw[k] = bc ? bc[k].v_wall : 0.0;
    g.bc.Tw[k] = bc ? bc[k].T_wall : 1.0;
  }
  geo_finish(g);
}

gks_status check_args(int nx, int ny, double Lx, double Ly, double gamma, double Pr, double mu, const gks_bc* bc,
                      const gks_options* o, std::string& why) {
  if (nx < 1 || ny < 1 || (long long)nx * ny > (1LL << 31)) { why = "nx, ny >= 1 and nx * ny <= 2^31 required"; return GKS_EINVAL; }
  // launch grids: the face kernels cover ny + 1 rows with 4-row blocks (grid y <= 65535)
  if (ny > 4 * 65535 - 1) { why = "ny must be < 262140"; return GKS_EINVAL; }
  if (!(Lx > 0) || !(Ly > 0)) { why = "Lx, Ly must be > 0"; return GKS_EINVAL; }
  if (!(gamma > 1.0) || !(gamma < 3.0)) { why = "gamma must lie in (1, 3)"; return GKS_EINVAL; }
  if (!(Pr > 0)) { why = "Pr must be > 0"; return GKS_EINVAL; }
  if (!(mu >= 0)) { why = "mu must be >= 0"; return GKS_EINVAL; }
  if (o->precision != GKS_FP64 && o->precision != GKS_FP32_BULK) { why = "unknown precision"; return GKS_EINVAL; }
  if (o->characteristic != 0 && o->characteristic != 1) { why = "characteristic must be 0 or 1"; return GKS_EINVAL; }
  if (!(o->weno_eps >= 0) || !(o->weno_C > 0) || !(o->tau_eps >= 0) || !(o->tau_C >= 0)) {
    why = "invalid scheme constants"; return GKS_EINVAL;
  }
  if (bc) {
    for (int k = 0; k < 4; ++k) {
      if (bc[k].kind < 0 || bc[k].kind > GKS_BC_EXCHANGE) { why = "unknown boundary kind"; return GKS_EINVAL; }
      if (bc[k].kind == GKS_BC_EXCHANGE && k < 2) { why = "exchange sides are y sides"; return GKS_EINVAL; }
      if (bc[k].kind == GKS_BC_NOSLIP_ISOTHERMAL && !(bc[k].T_wall > 0)) { why = "T_wall must be > 0"; return GKS_EINVAL; }
    }
    if ((bc[0].kind == GKS_BC_PERIODIC) != (bc[1].kind == GKS_BC_PERIODIC) ||
        (bc[2].kind == GKS_BC_PERIODIC) != (bc[3].kind == GKS_BC_PERIODIC)) {
      why = "periodic must be set on both sides of an axis"; return GKS_EINVAL;
    }
    if ((nx == 1 && bc[0].kind != GKS_BC_PERIODIC) ||
        (ny == 1 && bc[2].kind != GKS_BC_PERIODIC && (bc[2].kind != GKS_BC_EXCHANGE || bc[3].kind != GKS_BC_EXCHANGE))) {
      why = "a single cell across needs periodic sides"; return GKS_EINVAL;
    }
  }
  return GKS_OK;
}

}  // namespace

extern "C" {

void gks_default_options(gks_options* o) {
  if (!o) return;
  o->precision = GKS_FP64;
  o->weno_eps = 1e-6;
  o->weno_C = 10.0;
  o->tau_eps = 0.05;
  o->tau_C = 1.0;
  o->viscous_dt = 0;
  o->characteristic = 0;
}

gks_status gks_create(int nx, int ny, double Lx, double Ly, double gamma, double Pr, double mu, const gks_bc* bc,
                      const gks_options* opt, void* cuda_stream, gks_handle** out) {
  if (!out) { g_create_err = "out is NULL"; return GKS_EINVAL; }
  *out = nullptr;
  gks_options o;
  gks_default_options(&o);
  if (opt) o = *opt;
  std::string why;
  if (check_args(nx, ny, Lx, Ly, gamma, Pr, mu, bc, &o, why) != GKS_OK) { g_create_err = why; return GKS_EINVAL; }
  gks_handle* h = new gks_handle();
  Geo& g = h->g;
  make_geo(g, nx, ny, Lx, Ly, gamma, Pr, mu, bc, o);
  h->prec = o.precision;
  const size_t wsz = h->prec == GKS_FP64 ? 8 : 4;
  cudaError_t e = cudaGetDevice(&h->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, h->device);
  if (e == cudaSuccess) {
    if (cuda_stream) { h->stream = (cudaStream_t)cuda_stream; h->own_stream = false; }
    else { e = cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking); h->own_stream = true; }
  }
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&h->side, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->fork, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->join, cudaEventDisableTiming);
  auto alloc = [&](void** p, size_t bytes) {
    if (e == cudaSuccess) e = cudaMalloc(p, bytes);
  };
  for (int b = 0; b < 2; ++b) {
    alloc((void**)&h->U[b], 4 * g.plane * sizeof(double));
    alloc(&h->Wx[b], n_wx(g) * wsz);
    alloc(&h->Wy[b], n_wy(g) * wsz);
  }
  alloc(&h->rec, rec_count(g) * wsz);
  alloc(&h->Fx, (size_t)4 * ny * (nx + 1) * wsz);
  alloc(&h->Fy, (size_t)4 * (ny + 1) * nx * wsz);
  alloc((void**)&h->bad, (size_t)nx * ny);
  alloc((void**)&h->ctrl, sizeof(Ctrl));
  h->staging_n = n_u(g);
  if (n_wx(g) > h->staging_n) h->staging_n = n_wx(g);
  if (n_wy(g) > h->staging_n) h->staging_n = n_wy(g);
  if (h->staging_n < (size_t)24 * nx * ny) h->staging_n = (size_t)24 * nx * ny;
  alloc((void**)&h->staging, h->staging_n * sizeof(double));
  if (e == cudaSuccess) e = cudaMallocHost((void**)&h->hctrl, sizeof(Ctrl));
  if (e == cudaSuccess)
    for (int b = 0; b < 2; ++b) {
      if (e == cudaSuccess) e = cudaMemsetAsync(h->U[b], 0, 4 * g.plane * sizeof(double), h->stream);
      if (e == cudaSuccess) e = cudaMemsetAsync(h->Wx[b], 0, n_wx(g) * wsz, h->stream);
      if (e == cudaSuccess) e = cudaMemsetAsync(h->Wy[b], 0, n_wy(g) * wsz, h->stream);
    }
  if (e != cudaSuccess) {
    g_create_err = std::string("gks_create: ") + cudaGetErrorString(e);
    const gks_status st = e == cudaErrorMemoryAllocation ? GKS_ENOMEM : GKS_ECUDA;
    gks_destroy(h);
    return st;
  }
  k_state_begin<<<1, 1, 0, h->stream>>>(h->ctrl, 0.0, 1);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) {
    g_create_err = std::string("gks_create: ") + cudaGetErrorString(e);
    gks_destroy(h);
    return GKS_ECUDA;
  }
  *out = h;
  return GKS_OK;
}

gks_status gks_set_state_device(gks_handle* h, const double* dU, const double* dWx, const double* dWy, double t) {
  if (!h || !dU) return fail(h, GKS_EINVAL, "gks_set_state: U is required");
  CK(cudaSetDevice(h->device));
  gks_status st = h->prec == GKS_FP64 ? load_state<double>(h, t, dU, dWx, dWy) : load_state<float>(h, t, dU, dWx, dWy);
  if (st != GKS_OK) return st;
  st = read_ctrl(h);
  if (st != GKS_OK) return st;
  if (h->hctrl->status != GKS_OK) return fail(h, GKS_ENONPHYSICAL, "gks_set_state: state has rho <= 0 or p <= 0");
  return GKS_OK;
}

gks_status gks_set_state(gks_handle* h, const double* U, const double* Wx, const double* Wy, double t) {
  if (!h || !U) return fail(h, GKS_EINVAL, "gks_set_state: U is required");
  CK(cudaSetDevice(h->device));
  // page-locked host arrays are read in place by the kernels; the others go through
  // the staging buffer in turn
  const double *dU = mapped_host(U), *dWx = Wx ? mapped_host(Wx) : nullptr, *dWy = Wy ? mapped_host(Wy) : nullptr;
  const bool su = !dU, sx = Wx && !dWx, sy = Wy && !dWy;
  if (su) dU = U;
  if (sx) dWx = Wx;
  if (sy) dWy = Wy;
  gks_status st = h->prec == GKS_FP64 ? load_state<double>(h, t, dU, dWx, dWy, su, sx, sy)
                                      : load_state<float>(h, t, dU, dWx, dWy, su, sx, sy);
  if (st != GKS_OK) return st;
  st = read_ctrl(h);
  if (st != GKS_OK) return st;
  if (h->hctrl->status != GKS_OK) return fail(h, GKS_ENONPHYSICAL, "gks_set_state: state has rho <= 0 or p <= 0");
  return GKS_OK;
}

gks_status gks_step(gks_handle* h, double CFL, double dt_max, double* dt_taken) {
  if (!h) return GKS_EINVAL;
  if (!(CFL > 0) || !(dt_max > 0)) return fail(h, GKS_EINVAL, "gks_step: CFL and dt_max must be > 0");
  CK(cudaSetDevice(h->device));
  gks_status st = launch_step(h, CFL, dt_max, INFINITY, true);
  if (st != GKS_OK) return st;
  CK(cudaStreamSynchronize(h->stream));  // the step left its control block in hctrl
  if (dt_taken) *dt_taken = h->hctrl->skip ? 0.0 : h->hctrl->dt;
  return step_status(h, "step produced a non-physical state; state kept");
}

gks_status gks_advance(gks_handle* h, int nsteps, double CFL, double t_end) {
  if (!h) return GKS_EINVAL;
  if (nsteps < 0 || !(CFL > 0)) return fail(h, GKS_EINVAL, "gks_advance: nsteps >= 0 and CFL > 0 required");
  CK(cudaSetDevice(h->device));
  if (h->graph_cfl != CFL || h->graph_tend != t_end) destroy_graphs(h);
  h->graph_cfl = CFL;
  h->graph_tend = t_end;
  int left = nsteps;
  for (int k = 0; k < 3; ++k) {
    if (left >= kGraphSteps[k] && !h->graph[k]) {
      const gks_status st = capture(h, kGraphSteps[k], CFL, t_end, &h->graph[k]);
      if (st != GKS_OK) { destroy_graphs(h); return st; }
    }
    for (; left >= kGraphSteps[k]; left -= kGraphSteps[k]) CK(cudaGraphLaunch(h->graph[k], h->stream));
  }
  return GKS_OK;
}

gks_status gks_set_wait_limit(gks_handle* h, double seconds, int test_skip_block) {
  if (!h || !(seconds > 0) || !(seconds <= 3600)) return fail(h, GKS_EINVAL, "gks_set_wait_limit: seconds must lie in (0, 3600]");
  CK(cudaSetDevice(h->device));
  destroy_graphs(h);  // they hold the limit
  h->wait_s = seconds;
  h->wait_skip = test_skip_block;
  return GKS_OK;
}

gks_status gks_sync(gks_handle* h, double* t, long long* steps) {
  if (!h) return GKS_EINVAL;
  CK(cudaSetDevice(h->device));
  gks_status st = read_ctrl(h);
  if (st != GKS_OK) return st;
  if (t) *t = h->hctrl->t;
  if (steps) *steps = h->hctrl->steps;
  return step_status(h, "a queued step produced a non-physical state; state kept");
}

gks_status gks_get_state_device(gks_handle* h, double* dU, double* dWx, double* dWy, double* t) {
  if (!h) return GKS_EINVAL;
  CK(cudaSetDevice(h->device));
  gks_status st = h->prec == GKS_FP64 ? store_state<double>(h, dU, dWx, dWy) : store_state<float>(h, dU, dWx, dWy);
  if (st != GKS_OK) return st;
  st = read_ctrl(h);
  if (st != GKS_OK) return st;
  if (t) *t = h->hctrl->t;
  return step_status(h, "a step produced a non-physical state; state kept");
}

gks_status gks_get_state(gks_handle* h, double* U, double* Wx, double* Wy, double* t) {
  if (!h) return GKS_EINVAL;
  CK(cudaSetDevice(h->device));
  const Geo& g = h->g;
  struct { double* host; size_t n; int which; } parts[3] = {{U, n_u(g), 0}, {Wx, n_wx(g), 1}, {Wy, n_wy(g), 2}};
  for (auto& p : parts) {
    if (!p.host) continue;
    // page-locked host arrays are written in place by the kernels; the others through
    // the staging buffer in turn
    double* direct = const_cast<double*>(mapped_host(p.host));
    double* dst = direct ? direct : h->staging;
    gks_status st = h->prec == GKS_FP64
                        ? store_state<double>(h, p.which == 0 ? dst : nullptr, p.which == 1 ? dst : nullptr,
                                              p.which == 2 ? dst : nullptr)
                        : store_state<float>(h, p.which == 0 ? dst : nullptr, p.which == 1 ? dst : nullptr,
                                             p.which == 2 ? dst : nullptr);
    if (st != GKS_OK) return st;
    if (!direct) CK(cudaMemcpyAsync(p.host, h->staging, p.n * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  }
  gks_status st = read_ctrl(h);
  if (st != GKS_OK) return st;
  if (t) *t = h->hctrl->t;
  return step_status(h, "a step produced a non-physical state; state kept");
}

void gks_destroy(gks_handle* h) {
  if (!h) return;
  cudaSetDevice(h->device);
  if (h->stream) cudaStreamSynchronize(h->stream);
  destroy_graphs(h);
  for (int b = 0; b < 2; ++b) {
    cudaFree(h->U[b]);
    cudaFree(h->Wx[b]);
    cudaFree(h->Wy[b]);
  }
  cudaFree(h->rec);
  cudaFree(h->Fx);
  cudaFree(h->Fy);
  cudaFree(h->bad);
  cudaFree(h->ctrl);
  cudaFree(h->staging);
  if (h->hctrl) cudaFreeHost(h->hctrl);
  if (h->side) cudaStreamSynchronize(h->side);
  if (h->fork) cudaEventDestroy(h->fork);
  if (h->join) cudaEventDestroy(h->join);
  if (h->side) cudaStreamDestroy(h->side);
  if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
  delete h;
}

const char* gks_last_error(const gks_handle* h) { return h ? h->err.c_str() : g_create_err.c_str(); }

gks_status gks_profile_step(gks_handle* h, double CFL, float* ms) {
  if (!h || !ms || !(CFL > 0)) return fail(h, GKS_EINVAL, "gks_profile_step: CFL > 0 and ms[7] required");
  CK(cudaSetDevice(h->device));
  cudaEvent_t ev[kProfileParts + 1];
  for (int k = 0; k <= kProfileParts; ++k) CK(cudaEventCreate(&ev[k]));
  gks_status st = h->prec == GKS_FP64 ? launch_step_kernels<double, double>(h, CFL, INFINITY, INFINITY, true, true, 0, ev)
                                      : launch_step_kernels<float, float>(h, CFL, INFINITY, INFINITY, true, true, 0, ev);
  if (st == GKS_OK) {
    cudaError_t e = cudaEventSynchronize(ev[kProfileParts]);
    for (int k = 0; k < kProfileParts && e == cudaSuccess; ++k) e = cudaEventElapsedTime(&ms[k], ev[k], ev[k + 1]);
    if (e != cudaSuccess) st = fail(h, GKS_ECUDA, std::string("gks_profile_step: ") + cudaGetErrorString(e));
  }
  for (int k = 0; k <= kProfileParts; ++k) cudaEventDestroy(ev[k]);
  if (st != GKS_OK) return st;
  st = read_ctrl(h);
  if (st != GKS_OK) return st;
  return step_status(h, "step produced a non-physical state; state kept");
}

int gks_launches_per_step(const gks_handle* h) {
  return h && h->prec == GKS_FP32_BULK && h->g.mu > 0.0 ? 5 : 4;  // reconstruction, faces, update, finish
}

gks_status gks_debug_recon(gks_handle* h, double* coef) {
  if (!h || !coef) return GKS_EINVAL;
  CK(cudaSetDevice(h->device));
  const Geo& g = h->g;
  const dim3 b2(32, 8);
  if (h->prec == GKS_FP64) {
    launch_ghost<double>(h, 1);
    launch_recon<double, double>(h, 1);
    k_coef_out<double><<<grid2(g.nx, g.ny, b2), b2, 0, h->stream>>>(g, cellbuf<double>(h, 0), cellbuf<double>(h, 1),
                                                                     (const double*)h->rec, h->staging, h->ctrl);
  } else {
    launch_ghost<float>(h, 1);
    launch_recon<float, float>(h, 1);
    k_coef_out<float><<<grid2(g.nx, g.ny, b2), b2, 0, h->stream>>>(g, cellbuf<float>(h, 0), cellbuf<float>(h, 1),
                                                                    (const float*)h->rec, h->staging, h->ctrl);
  }
  CK(cudaGetLastError());
  CK(cudaMemcpyAsync(coef, h->staging, (size_t)24 * g.nx * g.ny * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return GKS_OK;
}

gks_status gks_debug_flux(gks_handle* h, double dt, double* Fx, double* Fy, double* Wxn, double* Wyn) {
  if (!h || !(dt > 0)) return fail(h, GKS_EINVAL, "gks_debug_flux: dt > 0 required");
  CK(cudaSetDevice(h->device));
  const Geo& g = h->g;
  k_set_dt<<<1, 1, 0, h->stream>>>(h->ctrl, dt);
  gks_status st = h->prec == GKS_FP64 ? launch_step_kernels<double, double>(h, 0, 0, 0, false, false, 1)
                                      : launch_step_kernels<float, float>(h, 0, 0, 0, false, false, 1);
  if (st != GKS_OK) return st;
  st = read_ctrl(h);
  if (st != GKS_OK) return st;
  // new face values were written to the buffer that is not in use
  const size_t nfx = (size_t)g.ny * (g.nx + 1), nfy = (size_t)(g.ny + 1) * g.nx;
  struct { void *a, *b; double* dst; size_t faces; bool w; } parts[4] = {
      {h->Fx, h->Fx, Fx, nfx, false}, {h->Fy, h->Fy, Fy, nfy, false}, {h->Wx[1], h->Wx[0], Wxn, nfx, true}, {h->Wy[1], h->Wy[0], Wyn, nfy, true}};
  auto values = [&](auto* a, auto* b, size_t faces) {
    using T = std::remove_pointer_t<decltype(a)>;
    k_face_values<T, false><<<blocks_of(faces), 256, 0, h->stream>>>(h->staging, nullptr, faces, 0, a, b, (T*)nullptr, (T*)nullptr, h->ctrl);
  };
  for (auto& p : parts) {
    if (!p.dst) continue;
    const size_t n = (p.w ? 8 : 4) * p.faces;
    const unsigned blocks = (unsigned)((n + 255) / 256);
    if (h->prec == GKS_FP64) {
      if (p.w) values((double*)p.a, (double*)p.b, p.faces);
      else k_flux_out<double><<<blocks, 256, 0, h->stream>>>((const double*)p.a, h->staging, p.faces);
    } else {
      if (p.w) values((float*)p.a, (float*)p.b, p.faces);
      else k_flux_out<float><<<blocks, 256, 0, h->stream>>>((const float*)p.a, h->staging, p.faces);
    }
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(p.dst, h->staging, n * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  }
  CK(cudaStreamSynchronize(h->stream));
  return GKS_OK;
}

// ---- partitioned step (domain decomposition into row slabs) ----

gks_status gks_part_halo_bytes(const gks_handle* h, int what, size_t* bytes) {
  if (!h || !bytes || (what != GKS_PART_STATE && what != GKS_PART_RECORDS)) return GKS_EINVAL;
  const Geo& g = h->g;
  const size_t es = h->prec == GKS_FP64 ? sizeof(double) : sizeof(float);
  // averages: 4 FP64 planes of nx + 2 values, or nx + 2 hi and nx + 2 lo vectors of 4 FP32 values
  *bytes = what == GKS_PART_STATE ? (size_t)8 * sizeof(float) * (g.nx + 2) : (size_t)(g.nx + 2) * kRec * es;
  return GKS_OK;
}

gks_status gks_part_bound(gks_handle* h, double* bound) {
  if (!h || !bound) return GKS_EINVAL;
  CK(cudaSetDevice(h->device));
  gks_status st = read_ctrl(h);
  if (st != GKS_OK) return st;
  memcpy(bound, &h->hctrl->bound, sizeof(double));
  return step_status(h, "the slab's state is not physical");
}

gks_status gks_part_recon(gks_handle* h, double dt) {
  if (!h || !(dt > 0)) return fail(h, GKS_EINVAL, "gks_part_recon: dt > 0 required");
  CK(cudaSetDevice(h->device));
  k_part_begin<<<1, 1, 0, h->stream>>>(h->ctrl, dt);
  CK(cudaGetLastError());
  const cudaError_t e = h->prec == GKS_FP64 ? launch_recon<double, double>(h, 0) : launch_recon<float, float>(h, 0);
  CK(e);
  return GKS_OK;
}

gks_status gks_part_finish(gks_handle* h) {
  if (!h) return GKS_EINVAL;
  CK(cudaSetDevice(h->device));
  gks_status st = h->prec == GKS_FP64
                      ? launch_step_kernels<double, double>(h, 0, 0, 0, true, true, 0, nullptr, false, true)
                      : launch_step_kernels<float, float>(h, 0, 0, 0, true, true, 0, nullptr, false, true);
  if (st != GKS_OK) return st;
  CK(cudaStreamSynchronize(h->stream));
  return step_status(h, "step produced a non-physical state; state kept");
}

namespace {
// one edge or halo row: (device address of its first byte, pitch between planes, planes,
// bytes per plane row); row j of the current buffer
gks_status part_row(gks_handle* h, int side, int what, bool halo, char** p, size_t* pitch, int* rows,
                    size_t* width) {
  if (side != 2 && side != 3) return fail(h, GKS_EINVAL, "side must be 2 (y low) or 3 (y high)");
  if (h->g.bc.kind[side] != GKS_BC_EXCHANGE) return fail(h, GKS_EINVAL, "not an exchange side");
  if (what != GKS_PART_STATE && what != GKS_PART_RECORDS) return fail(h, GKS_EINVAL, "what must be state or records");
  gks_status st = read_ctrl(h);
  if (st != GKS_OK) return st;
  const Geo& g = h->g;
  const int j = halo ? (side == 2 ? -1 : g.ny) : (side == 2 ? 0 : g.ny - 1);
  const size_t es = h->prec == GKS_FP64 ? sizeof(double) : sizeof(float);
  if (what == GKS_PART_STATE) {
    const int par = (int)(h->hctrl->steps & 1);
    // FP64: the row of each of the four planes; FP32: of the hi and of the lo vectors
    const int per = h->prec == GKS_FP64 ? 1 : 4;
    *p = (char*)h->U[par] + ((size_t)(j + 1) * g.pitch) * per * es;
    *pitch = g.plane * per * es;
    *rows = h->prec == GKS_FP64 ? 4 : 2;
    *width = (size_t)(g.nx + 2) * per * es;
  } else {
    *p = (char*)h->rec + rec_at(g, -1, j) * kRec * es;
    *pitch = 0;
    *rows = 1;
    *width = (size_t)(g.nx + 2) * kRec * es;
  }
  return GKS_OK;
}
}  // namespace

gks_status gks_part_get_edge(gks_handle* h, int side, int what, void* dst) {
  if (!h || !dst) return GKS_EINVAL;
  CK(cudaSetDevice(h->device));
  char* p;
  size_t pitch, width;
  int rows;
  gks_status st = part_row(h, side, what, false, &p, &pitch, &rows, &width);
  if (st != GKS_OK) return st;
  CK(cudaMemcpy2DAsync(dst, width, p, rows > 1 ? pitch : width, width, rows, cudaMemcpyDefault, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return GKS_OK;
}

gks_status gks_part_set_halo(gks_handle* h, int side, int what, const void* src) {
  if (!h || !src) return GKS_EINVAL;
  CK(cudaSetDevice(h->device));
  char* p;
  size_t pitch, width;
  int rows;
  gks_status st = part_row(h, side, what, true, &p, &pitch, &rows, &width);
  if (st != GKS_OK) return st;
  CK(cudaMemcpy2DAsync(p, rows > 1 ? pitch : width, src, width, width, rows, cudaMemcpyDefault, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return GKS_OK;
}

}  // extern "C"

// ===========================================================================
// Allocation-free single step (gks_step_noalloc).  For callers that must not
// allocate device memory themselves: code running under another runtime's
// memory manager or a hard memory cap, and latency-critical loops where
// cudaMalloc/cudaFree would synchronise the device.  The scratch of one step
// (the padded cell averages before and after, the reconstruction coefficients,
// the face fluxes and the control block) lives in one file-scope device array
// that every GPU loading this library holds until the process exits.
// ===========================================================================
namespace {

// 60 MiB: any grid of up to 65,536 cells.  The padded cell planes and the ghost ring of
// the reconstruction records make the need largest for a single column (nx = 1, rows
// padded to 4 and 3 records wide): 60,885,248 bytes at 1 x 65,536.
constexpr size_t kNoallocBytes = (size_t)60 << 20;
__device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes];

size_t align256(size_t n) { return (n + 255) & ~(size_t)255; }

// device address of g_noalloc_scratch per device, looked up once with the device current;
// the cache assumes that the device's primary context is never reset (cudaDeviceReset)
void* noalloc_base(int device, std::string& why) {
  static std::atomic<void*> base[64];
  if (device < 0 || device >= 64) { why = "device index out of range"; return nullptr; }
  void* p = base[device].load();
  if (!p) {
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) { why = std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e); return nullptr; }
    base[device].store(p);
  }
  return p;
}

}  // namespace

extern "C" gks_status gks_step_noalloc(int nx, int ny, double Lx, double Ly, double gamma, double Pr, double mu,
                                       const gks_bc* bc, const gks_options* opt, const double* dU,
                                       const double* dWx, const double* dWy, double CFL, double dt_max,
                                       double* dU_out, double* dWx_out, double* dWy_out, double* dt_taken,
                                       void* cuda_stream) {
  gks_options o;
  gks_default_options(&o);
  if (opt) o = *opt;
  std::string why;
  if (check_args(nx, ny, Lx, Ly, gamma, Pr, mu, bc, &o, why) != GKS_OK) { g_create_err = why; return GKS_EINVAL; }
  if (o.precision != GKS_FP64) { g_create_err = "gks_step_noalloc: only GKS_FP64"; return GKS_EINVAL; }
  if (!dU || !dWx || !dWy || !dU_out || !dWx_out || !dWy_out || !(CFL > 0) || !(dt_max > 0)) {
    g_create_err = "gks_step_noalloc: all six state pointers, CFL > 0 and dt_max > 0 are required";
    return GKS_EINVAL;
  }
  {
    // outputs must not overlap inputs or each other: the face kernels write new face values
    // that other faces' reconstruction still reads, and the update reads the old averages
    const size_t nu = (size_t)4 * nx * ny, nwx = (size_t)8 * ny * (nx + 1), nwy = (size_t)8 * (ny + 1) * nx;
    const struct { const double* p; size_t n; } in[3] = {{dU, nu}, {dWx, nwx}, {dWy, nwy}},
                                                 out[3] = {{dU_out, nu}, {dWx_out, nwx}, {dWy_out, nwy}};
    auto overlap = [](const double* a, size_t na, const double* b, size_t nb) { return a < b + nb && b < a + na; };
    for (int k = 0; k < 3; ++k)
      for (int m = 0; m < 3; ++m)
        if (overlap(out[k].p, out[k].n, in[m].p, in[m].n) || (m > k && overlap(out[k].p, out[k].n, out[m].p, out[m].n))) {
          g_create_err = "gks_step_noalloc: the output arrays must not overlap the inputs or each other";
          return GKS_EINVAL;
        }
  }
  Geo g;
  make_geo(g, nx, ny, Lx, Ly, gamma, Pr, mu, bc, o);
  // scratch layout: control block | padded U before | padded U after | reconstruction records | Fx | Fy
  const size_t b_ctrl = align256(sizeof(Ctrl));
  const size_t b_u = align256(4 * g.plane * sizeof(double));
  const size_t b_rec = align256(rec_count(g) * sizeof(double));
  const size_t b_fx = align256((size_t)4 * ny * (nx + 1) * sizeof(double));
  const size_t b_fy = align256((size_t)4 * (ny + 1) * nx * sizeof(double));
  const size_t b_bad = align256((size_t)nx * ny);
  const size_t need = b_ctrl + 2 * b_u + b_rec + b_fx + b_fy + b_bad;
  if ((long long)nx * ny > 65536 || need > kNoallocBytes) {
    g_create_err = "gks_step_noalloc: grid too large for the static scratch (at most 65,536 cells; " +
                   std::to_string(kNoallocBytes >> 20) + " MiB); need " + std::to_string(need) + " bytes";
    return GKS_EINVAL;
  }
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) { g_create_err = std::string("cudaGetDevice: ") + cudaGetErrorString(e); return GKS_ECUDA; }
  int sms = 0;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  if (e != cudaSuccess) { g_create_err = std::string("cudaDeviceGetAttribute: ") + cudaGetErrorString(e); return GKS_ECUDA; }
  unsigned char* base = (unsigned char*)noalloc_base(device, why);
  if (!base) { g_create_err = "gks_step_noalloc: " + why; return GKS_ECUDA; }
  Ctrl* ctrl = (Ctrl*)base;
  double* U0 = (double*)(base + b_ctrl);
  double* U1 = (double*)(base + b_ctrl + b_u);
  double* rec = (double*)(base + b_ctrl + 2 * b_u);
  double* Fx = (double*)(base + b_ctrl + 2 * b_u + b_rec);
  double* Fy = (double*)(base + b_ctrl + 2 * b_u + b_rec + b_fx);
  unsigned char* bad = base + b_ctrl + 2 * b_u + b_rec + b_fx + b_fy;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const Cells<double> C0{U0}, C1{U1};
  // the control block must start from zero state; the rest is fully written before it is read
  k_state_begin<<<1, 1, 0, s>>>(ctrl, 0.0, 1);
  e = launch(true, k_load_cells<double>, dim3(blocks_of((size_t)nx * ny)), dim3(256), s, g, dU, C0, C1, ctrl);
  if (e != cudaSuccess) { g_create_err = std::string("gks_step_noalloc: ") + cudaGetErrorString(e); return GKS_ECUDA; }
  e = launch_recon<double, double>(true, s, g, sms, U0, U1, dWx, dWx_out, dWy, dWy_out, rec, ctrl, 0, 1, CFL, dt_max, INFINITY);
  if (e != cudaSuccess) { g_create_err = std::string("gks_step_noalloc: ") + cudaGetErrorString(e); return GKS_ECUDA; }
  e = launch_faces<double, double>(true, s, g, sms, rec, const_cast<double*>(dWx), dWx_out, const_cast<double*>(dWy),
                                   dWy_out, Fx, Fy, ctrl, 0);
  if (e != cudaSuccess) { g_create_err = std::string("gks_step_noalloc: ") + cudaGetErrorString(e); return GKS_ECUDA; }
  const UpdateArgs<double, double> ua{C0, C1, Fx, Fy, const_cast<double*>(dWx), dWx_out, const_cast<double*>(dWy), dWy_out, bad};
  e = launch_update<double, double>(true, s, g, sms, ua, ctrl);
  if (e == cudaSuccess) e = launch_finish<double, double>(s, g, sms, ua, ctrl, nullptr, kWaitSeconds, -1);
  if (e != cudaSuccess) { g_create_err = std::string("gks_step_noalloc: ") + cudaGetErrorString(e); return GKS_ECUDA; }
  k_store_cells<double><<<blocks_of((size_t)nx * ny), 256, 0, s>>>(g, dU_out, C0, C1, ctrl);
  e = cudaGetLastError();
  Ctrl hc;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hc, ctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) { g_create_err = std::string("gks_step_noalloc: ") + cudaGetErrorString(e); return GKS_ECUDA; }
  if (dt_taken) *dt_taken = hc.skip ? 0.0 : hc.dt;
  if (hc.status != GKS_OK) {
    g_create_err = hc.status == GKS_ETIMEOUT
                       ? "gks_step_noalloc: a device wait of the positivity fallback ran out; outputs are not valid"
                       : "gks_step_noalloc: the step produced a non-physical state; outputs are not valid";
    return (gks_status)hc.status;
  }
  if (hc.skip) { g_create_err = "gks_step_noalloc: dt = 0, no step taken; outputs are not valid"; return GKS_EINVAL; }
  return GKS_OK;
}
