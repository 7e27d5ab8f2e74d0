// Cloud-in-cell helpers for the deposit and the field gather (Sec. IV-A).
#pragma once

#include "fixpt.h"
#include "sc_internal.cuh"

namespace sc {

// Cell, CIC weights and fractions of a particle: xi = (x - xmin) * inv_hx
// rounded twice (no fused multiply-add, so every platform takes the same
// integer decision), i = floor(xi), fixed-point weight a = rint((xi - i) 2^20)
// (ties to even) and, for FRAC, the float64 fraction fx = xi - i; the
// same for eta.  Inside iff 0 <= xi < nx-1 and 0 <= eta < ny-1; non-finite
// coordinates are outside.  Returns the cell index j*nx+i or -1.  With
// longitudinal slices the particle's slice k = floor((sg - zmin) * inv_dz)
// (same two roundings, 0 <= k < nz) selects the grid and the cell index is
// k*nx*ny + j*nx + i.
//
// locate_exact does the subtract and multiply of each axis on the FP64 pipe
// and decodes floor, fraction and rounding from the bits (cic_split, exact).
template <bool FRAC>
__device__ __noinline__ int locate_exact(const GridGeom& g, double x, double y, double sg, int2& a, double& fx,
                                         double& fy, int& i, int& j, int& k) {
  const double xi = __dmul_rn(__dsub_rn(x, g.xmin), g.inv_hx);
  const double eta = __dmul_rn(__dsub_rn(y, g.ymin), g.inv_hy);
  i = 0;
  j = 0;
  k = 0;
  bool in = cic_split(xi, g.nx - 1, i, a.x, FRAC ? &fx : nullptr);
  in = cic_split(eta, g.ny - 1, j, a.y, FRAC ? &fy : nullptr) && in;
  if (g.nz > 1) in = floor_index(__dmul_rn(__dsub_rn(sg, g.zmin), g.inv_dz), g.nz, k) && in;
  return in ? (k * g.ny + j) * g.nx + i : -1;
}

// The same decision in 64-bit integers (fix_split), without the FP64 pipe (it
// took 4 of its instructions per particle, 6 on sliced grids, 64 clocks each):
// for the one particle in some millions that lies too near a place where the
// decision changes, and on axes the integers do not serve (GridGeom::fix),
// locate_exact decides.  (One turn of 4e6 particles, BF16, 71.4 -> 64.5 ms.)
template <bool FRAC>
__device__ __forceinline__ int locate(const GridGeom& g, double x, double y, double sg, int2& a, double& fx,
                                      double& fy, int& i, int& j, int& k) {
  if (FRAC ? g.fix > 1 : g.fix != 0) {
    uint64_t zx, zy, zz;
    k = 0;
    int in = fix_split(g.ax, x, i, a.x, zx);
    const int iny = fix_split(g.ay, y, j, a.y, zy);
    int und = in | iny;
    in &= iny;
    if (g.nz > 1) {
      int w;
      const int inz = fix_split(g.az, sg, k, w, zz);
      und |= inz;
      in &= inz;
    }
    if (und >= 0) {
      if (FRAC) {
        fx = fix_fraction(g.ax, zx);
        fy = fix_fraction(g.ay, zy);
      }
      return in ? (k * g.ny + j) * g.nx + i : -1;
    }
  }
  int2 b;
  double ex = 0.0, ey = 0.0;
  int ei, ej, ek;
  const int cell = locate_exact<FRAC>(g, x, y, sg, b, ex, ey, ei, ej, ek);
  a = b;
  fx = ex;
  fy = ey;
  i = ei;
  j = ej;
  k = ek;
  return cell;
}

template <bool FRAC>
__device__ __forceinline__ int locate(const GridGeom& g, double x, double y, double sg, int2& a, double& fx,
                                      double& fy, int& k) {
  int i, j;
  return locate<FRAC>(g, x, y, sg, a, fx, fy, i, j, k);
}

template <bool FRAC>
__device__ __forceinline__ int locate(const GridGeom& g, double x, double y, double sg, int2& a, double& fx,
                                      double& fy) {
  int k;
  return locate<FRAC>(g, x, y, sg, a, fx, fy, k);
}

// A block's deposit tile in shared memory: the uint64 bins of its window as a
// plane of low and a plane of high 32-bit words.  Shared memory has native
// 32-bit atomic adds but only a compare-and-swap loop for 64 bits, so a bin is
// added to by its low word, whose old value gives the carry, and its high word
// (the sum is exact whatever the order of the adds).  Words of a plane lie
// next to each other, so a warp's 32 random bins spread over all 32 banks.
// Against 64-bit bins: stand-alone deposit of 1e6 particles on 128^2 15.2 ->
// 11.6 us, a 16-bunch batch's turn 118.5 -> 114.7 ms.
struct Tile {
  uint32_t* lo;
  uint32_t* hi;
};
__device__ __forceinline__ Tile tile_of(void* smem, const GridGeom& g) {
  return Tile{(uint32_t*)smem, (uint32_t*)smem + g.wnx * g.wny};
}

// The four CIC weights in 2^-20 fixed point per axis: a (from locate), b =
// 2^20 - a; the products sum to exactly 2^40 (32 x 32 -> 64-bit multiplies).
// q[0..3] = bx by, ax by, bx ay, ax ay.
__device__ __forceinline__ void weights4(int2 a, unsigned long long (&w)[4]) {
  const unsigned ax = (unsigned)a.x, ay = (unsigned)a.y;
  const unsigned bx = 1048576u - ax, by = 1048576u - ay;
  w[0] = (unsigned long long)bx * by;
  w[1] = (unsigned long long)ax * by;
  w[2] = (unsigned long long)bx * ay;
  w[3] = (unsigned long long)ax * ay;
}
// Added to nodes (cell, cell + 1, cell + nx, cell + nx + 1) of the global
// grid, or of a tile (same [j][i] layout, row length nx).
__device__ __forceinline__ void add4(unsigned long long* Q, int nx, int cell, const unsigned long long (&w)[4]) {
  unsigned long long* q = Q + cell;
  atomicAdd(q, w[0]);
  atomicAdd(q + 1, w[1]);
  atomicAdd(q + nx, w[2]);
  atomicAdd(q + nx + 1, w[3]);
}
// (A tile's high word is 0 for one weight in forty: skipping its add pays in
// the kick/push, 0.7% of a turn, and costs 3% in the stand-alone deposit, whose
// integer slots are the scarce ones: ALWAYS.)
template <bool ALWAYS = false>
__device__ __forceinline__ void add4(const Tile& t, int nx, int cell, const unsigned long long (&w)[4]) {
  const int c[4] = {cell, cell + 1, cell + nx, cell + nx + 1};
  uint32_t old[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) old[k] = atomicAdd(t.lo + c[k], (uint32_t)w[k]);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t l = (uint32_t)w[k];
    const uint32_t h = (uint32_t)(w[k] >> 32) + (old[k] + l < l ? 1u : 0u);
    if (ALWAYS || h) atomicAdd(t.hi + c[k], h);
  }
}
template <class Dst>
__device__ __forceinline__ void deposit4(const Dst& dst, int nx, int cell, int2 a) {
  unsigned long long w[4];
  weights4(a, w);
  add4(dst, nx, cell, w);
}

// Deposit target of a particle in cell (i, j) of slice k (`cell` its global
// index, -1 outside): the block's tile when it holds slice k (the tile takes
// the slice of the first particle that asks, tile_k starting at -1) and the
// tile's window holds the cell's four nodes -- key = the cell's lower-left
// node in the tile -- else the global grid -- key = kGlobalKey | cell.  -1:
// nothing to deposit.
constexpr int kGlobalKey = 1 << 29;

// The tile holds the whole grid of an unsliced deposit: every cell's four
// nodes are in it at their own index (the common case, no key needed).
__device__ __forceinline__ bool tile_is_grid(const GridGeom& g) {
  return g.nz == 1 && g.wnx == g.nx && g.wny == g.ny;
}
__device__ __forceinline__ int deposit_key(bool use_tile, int* tile_k, const GridGeom& g, int cell, int i, int j,
                                           int k) {
  if (cell < 0) return -1;
  if (use_tile) {
    int tk = *(volatile int*)tile_k;
    if (tk < 0) {
      const int prev = atomicCAS(tile_k, -1, k);
      tk = prev < 0 ? k : prev;
    }
    const int li = i - g.wx0, lj = j - g.wy0;
    if (tk == k && (unsigned)li < (unsigned)(g.wnx - 1) && (unsigned)lj < (unsigned)(g.wny - 1))
      return lj * g.wnx + li;
  }
  return kGlobalKey | cell;
}

// The four CIC adds of one particle at its target key (deposit_key; -1: none).
__device__ __forceinline__ void deposit_at(int key, int2 a, const Tile& tile, int wnx, unsigned long long* Q,
                                           int nx) {
  if (key < 0) return;
  if (key & kGlobalKey)
    deposit4(Q, nx, key & (kGlobalKey - 1), a);
  else
    deposit4(tile, wnx, key, a);
}

// One warp's CIC deposits (Sec. IV-A), the lanes of `mask` calling together,
// each with its target key (deposit_key) and fixed-point weights a.  Lanes
// next to each other with the same key form a run (a bunch ordered by cell
// puts a warp's particles in one or two runs); a run's four node sums are
// formed in registers -- over the run, sum bx by = n 2^40 - 2^20 (Sax + Say)
// + Saxay, sum ax by = 2^20 Sax - Saxay, sum bx ay = 2^20 Say - Saxay, sum
// ax ay = Saxay, exact in 64-bit integers -- and its first lane issues the
// four atomic adds.  Integer sums do not depend on their order, so the grid
// gets the same bits as with one atomic per weight.  When no two neighbouring
// lanes share a key each lane adds its own.  (For particles in random order
// the test itself costs more than it saves: callers use deposit_at there.)
__device__ __forceinline__ void deposit_warp(unsigned mask, int key, int2 a, const Tile& tile, int wnx,
                                             unsigned long long* Q, int nx) {
  const int lane = threadIdx.x & 31;
  const int prev = __shfl_up_sync(mask, key, 1);
  const bool head = lane == 0 || !((mask >> (lane - 1)) & 1u) || prev != key;
  const unsigned heads = __ballot_sync(mask, head);
  if (heads == mask) {
    deposit_at(key, a, tile, wnx, Q, nx);
    return;
  }
  // suffix sums over each run by doubling: after the step of offset d, a lane
  // holds the sums of its run's lanes [lane, lane + 2d)
  unsigned sx = (unsigned)a.x, sy = (unsigned)a.y;
  unsigned long long sxy = (unsigned long long)sx * sy;
  const int rid = __popc(heads & ((2u << lane) - 1u));  // runs that start at or below this lane
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned ox = __shfl_down_sync(mask, sx, d);
    const unsigned oy = __shfl_down_sync(mask, sy, d);
    const unsigned long long oxy = __shfl_down_sync(mask, sxy, d);
    const int src = lane + d;
    if (src < 32 && ((mask >> src) & 1u) && __popc(heads & ((2u << src) - 1u)) == rid) {
      sx += ox;
      sy += oy;
      sxy += oxy;
    }
  }
  if (head && key >= 0) {
    // run length: the lanes of the mask from this one up to the next run's head
    const unsigned above = heads & ~((2u << lane) - 1u);
    const unsigned span = above ? ((1u << (__ffs(above) - 1)) - 1u) : 0xffffffffu;
    const unsigned long long n = (unsigned long long)__popc(mask & span & ~((1u << lane) - 1u));
    const unsigned long long one = 1048576ull;
    const unsigned long long w[4] = {(n << 40) - one * ((unsigned long long)sx + sy) + sxy, one * sx - sxy,
                                     one * sy - sxy, sxy};
    if (key & kGlobalKey)
      add4(Q, nx, key & (kGlobalKey - 1), w);
    else
      add4(tile, wnx, key, w);
  }
}

// Cubic Bernstein weights b_m(t) and their derivatives (R = double for the
// float64 form, float for the split form whose potential is float32).
template <typename R>
__device__ __forceinline__ void bernstein3(R t, R (&b)[4], R (&db)[4]) {
  const R u = R(1) - t, uu = u * u, tt = t * t, tu = t * u;
  b[0] = uu * u;
  b[1] = R(3) * tu * u;
  b[2] = R(3) * tu * t;
  b[3] = tt * t;
  db[0] = R(-3) * uu;
  db[1] = fma(R(3), uu, R(-6) * tu);
  db[2] = fma(R(6), tu, R(-3) * tt);
  db[3] = R(3) * tt;
}

// Potential of node (i, j) of one grid, i in -1..nx, j in -1..ny: beyond the
// walls the odd extension (u_{-1} = -u_1, u_n = -u_{n-2}).
template <typename R>
__device__ __forceinline__ R phi_node(const R* __restrict__ phi, int nx, int ny, int i, int j) {
  R sgn = R(1);
  if (i < 0) { i = -i; sgn = -sgn; }
  if (i > nx - 1) { i = 2 * (nx - 1) - i; sgn = -sgn; }
  if (j < 0) { j = -j; sgn = -sgn; }
  if (j > ny - 1) { j = 2 * (ny - 1) - j; sgn = -sgn; }
  return sgn * __ldg(phi + (size_t)j * nx + i);
}

// Bezier surface (Sec. IV-C) of grid phi in cell (i, j) at fractions (fx, fy):
// value u and the derivatives with respect to the cell fractions' span
// parameters (d/dx = gx / (3 hx), d/dy = gy / (3 hy)).
template <typename R, bool VALUE, bool GRAD>
__device__ __forceinline__ void bezier_eval(const R* __restrict__ phi, int nx, int ny, int i, int j, R fx, R fy,
                                            R& u, R& gx, R& gy) {
  R bx[4], dbx[4], by[4], dby[4];
  bernstein3<R>((R(1) + fx) * (R(1) / R(3)), bx, dbx);
  bernstein3<R>((R(1) + fy) * (R(1) / R(3)), by, dby);
  u = gx = gy = R(0);
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    R rv = R(0), rx = R(0);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const R c = phi_node<R>(phi, nx, ny, i + m - 1, j + n - 1);
      rv = fma(c, bx[m], rv);
      if (GRAD) rx = fma(c, dbx[m], rx);
    }
    if (VALUE) u = fma(rv, by[n], u);
    if (GRAD) {
      gx = fma(rx, by[n], gx);
      gy = fma(rv, dby[n], gy);
    }
  }
}

// Zero a shared-memory tile of `cells` bins (whole block; 16-byte stores).
__device__ __forceinline__ void tile_zero(void* tile, int cells) {
  const int quads = cells >> 1;
  for (int c = threadIdx.x; c < quads; c += blockDim.x) ((uint4*)tile)[c] = make_uint4(0u, 0u, 0u, 0u);
  if ((cells & 1) && threadIdx.x == 0) ((unsigned long long*)tile)[cells - 1] = 0ull;
}

// Add the non-zero bins of a block's tile into the global grid Q (one
// slice; whole block; caller synchronises before): bin (li, lj) of the window
// is node (wx0 + li, wy0 + lj).  This is the only cross-block reduction of
// the deposit.
__device__ __forceinline__ void tile_flush(const Tile& t, unsigned long long* Q, const GridGeom& g) {
  const int cells = g.wnx * g.wny;
  if (g.wnx == g.nx && g.wny == g.ny) {  // the tile is the whole slice: same indices
    for (int c = threadIdx.x; c < cells; c += blockDim.x) {
      const unsigned long long v = (unsigned long long)t.hi[c] << 32 | t.lo[c];
      if (v) atomicAdd(Q + c, v);
    }
    return;
  }
  // a window: walk its bins with a running (row, column), no division per bin
  int lj = threadIdx.x / g.wnx, li = threadIdx.x - lj * g.wnx;
  const int step_j = blockDim.x / g.wnx, step_i = blockDim.x - step_j * g.wnx;
  for (int c = threadIdx.x; c < cells; c += blockDim.x) {
    const unsigned long long v = (unsigned long long)t.hi[c] << 32 | t.lo[c];
    if (v) atomicAdd(Q + (size_t)(g.wy0 + lj) * g.nx + g.wx0 + li, v);
    lj += step_j;
    li += step_i;
    if (li >= g.wnx) {
      li -= g.wnx;
      ++lj;
    }
  }
}

// A non-finite coordinate (NaN or infinity), tested on the bits: no FP64 instruction.
__device__ __forceinline__ bool nonfinite(double v) {
  return ((unsigned long long)__double_as_longlong(v) & 0x7ff0000000000000ull) == 0x7ff0000000000000ull;
}

// 1 for a particle whose position (or, on a sliced grid, its sigma) is not
// finite: bit tests only, for particles the deposit found outside grid g; the
// caller sums them in a register like the out-of-grid count (count_out).
__device__ __forceinline__ unsigned int nonfinite_state(const GridGeom& g, double x, double y, double sg) {
  return (unsigned int)(nonfinite(x) | nonfinite(y) | (g.nz > 1 && nonfinite(sg)));
}

// Block-wide sum of per-thread out-of-grid counts into a global counter.
__device__ __forceinline__ void count_out(unsigned int out, unsigned long long* n_out) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) out += __shfl_xor_sync(0xffffffffu, out, o);
  if ((threadIdx.x & 31) == 0 && out && n_out) atomicAdd(n_out, (unsigned long long)out);
}

}  // namespace sc
