// States in and out of a handle or a batch's grid: between the caller's planes of FP64 values (device memory, or
// page-locked host memory read and written in place) and the padded, per-type layouts, with the ghost
// ring and the CFL bound of a state that goes in.
//
// Each kernel is a straight copy bound by memory (or the host link): one thread per cell or face moves all
// four variables, so that both sides' accesses are contiguous, and the ghost cells and the bound are made
// from the values in registers instead of by further passes.
#pragma once
#include "gks_grid.cuh"

namespace gks {

// control block of a new state at time t; the parity of the step counter stays (first: a new block)
static __global__ void k_state_begin(Ctrl* c, double t, int first) {
  const long long steps = first ? 0 : c->steps;
  *c = Ctrl{};
  c->steps = steps;
  c->t = t;
  c->bound = c->dtb[0] = c->dtb[1] = c->dtb[2] = dbits(INFINITY);
  c->fail_step = -1;
}

// Lower bound on the inverse CFL bound that the state must reach to matter (the running maximum, rounded
// down in FP32), from the slot that holds the running minimum of the bound
__device__ __forceinline__ float inv_floor(const unsigned long long* slot) {
  const float b = (float)bitsd(*(const volatile unsigned long long*)slot);
  return __fdividef(0.9999f, b);  // 0 for an empty slot (infinity)
}

// block maximum of the inverse bounds (bits of non-negative doubles, which order as the doubles do), then the
// atomic minimum of the bound.  Every thread of the block calls it.
__device__ __forceinline__ void block_bound_bits(unsigned long long bits, unsigned long long* slot) {
  __shared__ unsigned long long red[32];
  if (!__syncthreads_or(bits != 0)) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long b = __shfl_xor_sync(0xffffffffu, bits, o);
    bits = b > bits ? b : bits;
  }
  const int t = threadIdx.y * blockDim.x + threadIdx.x, n = (blockDim.x * blockDim.y + 31) >> 5;
  if ((t & 31) == 0) red[t >> 5] = bits;
  __syncthreads();
  if (t == 0) {
    for (int k = 1; k < n; ++k) bits = red[k] > bits ? red[k] : bits;
    if (bits) atomicMin(slot, dbits(1.0 / bitsd(bits)));
  }
}

// cell averages in: planes [4][ny][nx] to the buffer in use, the ghost images of each cell, and the CFL bound of
// the state in FP64 (status: a cell that is not physical).
// FP64 arithmetic costs 64 cycles an instruction here: a cell computes its bound in FP64 only where FP32 does not
// prove it physical and below the maximum so far.
template <class R>
static __global__ void __launch_bounds__(256) k_load_cells(Geo g, const double* __restrict__ src, Cells<R> U0, Cells<R> U1, Ctrl* c) {
  pdl_enter();
  const size_t n = (size_t)g.nx * g.ny, k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const Cells<R> U = (c->steps & 1) ? U1 : U0;
  unsigned long long bits = 0;
  if (k < n) {
    const int j = (int)(k / (unsigned)g.nx), i = (int)(k - (size_t)j * g.nx);
    double w[4];
    CellState<R> S;
#pragma unroll
    for (int v = 0; v < 4; ++v) w[v] = split_value(src[(size_t)v * n + k], S, v);
    store_state(g, U, i, j, S);
    ghosts_of_cell<R>(g, U, i, j);
    if (!surely_below(g, w, inv_floor(&c->bound))) {
      bool ok;
      const double inv = inv_bound<double>(g, w, ok);
      if (!ok || !(inv < INFINITY)) atomicCAS(&c->status, GKS_OK, GKS_ENONPHYSICAL);
      else bits = dbits(inv);
    }
  }
  block_bound_bits(bits, &c->bound);
}

// cell averages out
template <class R>
static __global__ void __launch_bounds__(256) k_store_cells(Geo g, double* __restrict__ dst, Cells<R> U0, Cells<R> U1, const Ctrl* c) {
  const size_t n = (size_t)g.nx * g.ny, k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const Cells<R> U = (c->steps & 1) ? U1 : U0;
  const int j = (int)(k / (unsigned)g.nx), i = (int)(k - (size_t)j * g.nx);
  CellState<R> S;
  load_state(g, U, i, j, S);
#pragma unroll
  for (int v = 0; v < 4; ++v) dst[(size_t)v * n + k] = whole_value(S, v);
}

// face values of both axes between the caller's planes [4][2][faces] (0: that axis is left alone) and the buffer in
// use; nx, ny: faces of each axis
template <class R, bool IN>
static __global__ void __launch_bounds__(256) k_face_values(double* __restrict__ px, double* __restrict__ py, size_t nx, size_t ny,
                                                     R* Wx0, R* Wx1, R* Wy0, R* Wy1, const Ctrl* c) {
  const size_t bx = px ? nx : 0;
  size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int par = (int)(c->steps & 1);
  const bool x = k < bx;
  if (!x) k -= bx;
  double* p = x ? px : py;
  const size_t n = x ? nx : ny;
  if (!p || k >= n) return;
  R* W = x ? (par ? Wx1 : Wx0) : (par ? Wy1 : Wy0);
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    R r[4];
    if (IN) {
#pragma unroll
      for (int v = 0; v < 4; ++v) r[v] = (R)p[(size_t)(2 * v + q) * n + k];
      Lay<R>::store_w(W, n, q, k, r);
    } else {
      Lay<R>::load_w(W, n, q, k, r);
#pragma unroll
      for (int v = 0; v < 4; ++v) p[(size_t)(2 * v + q) * n + k] = (double)r[v];
    }
  }
}

inline unsigned blocks_of(size_t n) { return (unsigned)((n + 255) / 256); }

// The device address of a page-locked host array mapped into the device's address
// space (cudaHostAlloc, cudaHostRegister): kernels then read or write it in place over
// the host link.  nullptr for any other pointer, which goes through the staging buffer: pageable memory, and arrays
// that do not start on a multiple of 8 bytes (a copy takes any address, a kernel's loads do not).
inline const double* mapped_host(const void* p) {
  if ((size_t)p % alignof(double)) return nullptr;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();  // an unknown pointer: clear the error it left
    return nullptr;
  }
  return a.type == cudaMemoryTypeHost && a.devicePointer ? (const double*)a.devicePointer : nullptr;
}

}  // namespace gks
