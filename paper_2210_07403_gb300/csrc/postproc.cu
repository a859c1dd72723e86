// Solution post-processing: flagging the region enclosed by the immersed boundary (Sec. 5.3.5)
// and the linear interpolation that replaces grid values near Γ (Sec. 5.3.4).
//
// Indicator. χ solves Δχ = −S̃1: the IBDL grid field of the unit density for the plain Laplace
// problem (mean-zero inverse), with the geometry's δ_h, dipole spread and symbol. In the
// continuum χ = 1_enclosed − |enclosed|/|C|; subtracting the value at the box corner leaves ≈ 1
// inside the curves and ≈ 0 outside (≈ −1 inside for inward normals), and the flags are |χ| > ½.
//
// Near-boundary interpolation (2-D). A node x_p of the caller's mask Ω whose nearest boundary
// point lies closer than m1·h takes
//     u(x_p) = u_A |x_B − x_p|/|x_B − x_A| + u_B |x_A − x_p|/|x_B − x_A|,
// with x_A the point of the chord of its two nearest boundary points closest to x_p (if that
// projection leaves the chord: the chord of the two of the three nearest points that lie
// farthest apart, the projection clamped to it), u_A the linear interpolation of U_b along the
// chord, x_B = x_A + m2·h (x_p − x_A)/|x_p − x_A| and u_B the bilinear interpolation of the grid
// values around x_B. Which nodes are replaced and which boundary points are nearest are integer
// decisions: they are taken on FP64 squared minimum-image distances dx·dx + dy·dy, each
// operation rounded on its own (no contraction), equal distances ordered by point index.
//
// Kernels (the interpolation): k_mark flags the nodes within ceil(m1) + 2 cells of some point
// (a superset of the nodes to replace), k_compact lists the row segments of 32 nodes that hold a
// flagged node of Ω, and k_near takes a segment per warp, a node per lane. The points whose cell lies
// within K rows and K + 1 columns of the segment (rows of the geometry's cell-sorted order, an integer
// test of the cell column) are collected in shared memory with their squared y distance, which the
// whole segment shares; every lane then runs through them and keeps its three nearest: three FP64
// instructions per point for 32 nodes. A node whose third distance is not below W = (K − 1)·h is scanned
// again over all M points by the whole warp. The distance comparisons run on the integer pipe
// (non-negative doubles order as their bits), so the FP64 unit only forms the distances. (With a
// warp scanning the points of one node after another, five FP64 instructions per 32 points and node,
// and 16 nodes per warp, some SMs held twice the warps of others: the 1024² circle, 19 000 nodes, took
// 141 µs.)
#include <climits>
#include <cmath>
#include <cstring>

#include "fft.cuh"

namespace ibdl {

namespace {

constexpr int kPPThreads = 256;

__global__ void k_fill(double* __restrict__ p, int64_t n, double v) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    p[i] = v;
}

__global__ void k_indicator_shift(const double* __restrict__ raw, int64_t cells, double* __restrict__ chi,
                                  uint8_t* __restrict__ flags) {
  const double corner = raw[0];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cells; i += (int64_t)gridDim.x * blockDim.x) {
    const double v = raw[i] - corner;
    chi[i] = v;
    flags[i] = fabs(v) > 0.5 ? 1 : 0;
  }
}

__device__ __forceinline__ int wrapn(long long v, int n) {
  long long r = v % n;
  return (int)(r < 0 ? r + n : r);
}

// flag every node within k1 cells (per axis) of a point's first stencil node + 1
__global__ void k_mark(int n, int M, int k1, const int* __restrict__ base, uint8_t* __restrict__ marks) {
  const int w = 2 * k1 + 1;
  const int64_t items = (int64_t)M * w * w;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < items; t += (int64_t)gridDim.x * blockDim.x) {
    const int s = (int)(t / (w * w));
    const int o = (int)(t - (int64_t)s * w * w);
    const int ix = wrapn((long long)base[s] + 1 - k1 + o % w, n);
    const int iy = wrapn((long long)base[M + s] + 1 - k1 + o / w, n);
    marks[(size_t)iy * n + ix] = 1;
  }
}

// nodes of a row segment
__host__ __device__ constexpr int segment_width(int n) { return n < 32 ? n : 32; }

// list the row segments that hold a marked node of Ω (the list order is irrelevant)
__global__ void k_compact(int n, int64_t cells, const uint8_t* __restrict__ marks, const uint8_t* __restrict__ omega,
                          int* __restrict__ list, int* __restrict__ count) {
  const int lane = threadIdx.x & 31, sw = segment_width(n);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) - lane; b < cells; b += stride) {
    const int64_t i = b + lane;
    const unsigned m = __ballot_sync(0xffffffffu, i < cells && marks[i] && omega[i]);
    if (lane % sw == 0 && ((m >> lane) & (0xffffffffu >> (32 - sw)))) list[atomicAdd(count, 1)] = (int)(i / sw);
  }
}

struct NearParams {
  int n, M, c, K;
  double h, L, o0, o1;
  unsigned long long r1key;    // bits of (m1·h)²
  unsigned long long slabkey;  // bits of W², W = (K − 1)·h: a slab result is exact when its third
                               // distance is below W
  unsigned long long halfbits; // bits of L/2
  double halfL;
  double m2h;                  // m2·h
  const double* X;             // [2][M] original order
  const int* base;             // [2][M] first stencil nodes, sorted order
  const int* perm;             // sorted position → original index
  const int* cell_start;       // [n + 1] rows of constant base y
  const double* Ub;            // [c][M]
  const double* u;             // [c][n][n]
  double* out;                 // [c][n][n]
  const uint8_t* marks;
  const uint8_t* omega;
  const int* list;             // segments
  const int* count;
};

// Non-negative doubles order as their bit patterns (as unsigned integers), so distances are
// compared on the integer pipe: the FP64 unit, the bound of this kernel, only forms them.
__device__ __forceinline__ unsigned long long dbits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ unsigned long long absbits(double v) { return dbits(v) & 0x7fffffffffffffffull; }

// minimum-image offset d − L·rint(d/L), each operation rounded on its own
__device__ __forceinline__ double mimg(double d, double L) {
  return __dsub_rn(d, __dmul_rn(L, rint(__ddiv_rn(d, L))));
}

// the same for |d| < L/2 without the division: d/L then rounds to a value of magnitude ≤ ½,
// which rounds to zero (ties to even), and the formula returns d
__device__ __forceinline__ double mimg_fast(double d, const NearParams& p) {
  return absbits(d) < p.halfbits ? d : mimg(d, p.L);
}

__device__ __forceinline__ double sqdist(double dx, double dy) { return __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)); }

__device__ __forceinline__ bool key_less(unsigned long long ka, int ia, unsigned long long kb, int ib) {
  return ka < kb || (ka == kb && ia < ib);
}

constexpr unsigned long long kInfKey = 0x7ff0000000000000ull;  // +∞

// a lane's three nearest, (squared-distance bits, index) ascending
struct Top3 {
  unsigned long long k0, k1, k2;
  int i0, i1, i2;
  __device__ void init() {
    k0 = k1 = k2 = kInfKey;
    i0 = i1 = i2 = INT_MAX;
  }
  __device__ void insert(unsigned long long k, int i) {
    if (!key_less(k, i, k2, i2)) return;
    if (key_less(k, i, k1, i1)) {
      k2 = k1;
      i2 = i1;
      if (key_less(k, i, k0, i0)) {
        k1 = k0;
        i1 = i0;
        k0 = k;
        i0 = i;
      } else {
        k1 = k;
        i1 = i;
      }
    } else {
      k2 = k;
      i2 = i;
    }
  }
};

// lanes scan every point into their own three nearest
__device__ __forceinline__ void scan_all(const NearParams& p, int lane, double px, double py, Top3& t) {
  for (int i = lane; i < p.M; i += 32) {
    const double dx = mimg_fast(__dsub_rn(p.X[i], px), p);
    const double dy = mimg_fast(__dsub_rn(p.X[p.M + i], py), p);
    t.insert(dbits(sqdist(dx, dy)), i);
  }
}

// the warp's three nearest, in every lane: three rounds of a butterfly minimum over the lanes'
// heads; the lane whose head wins pops it
__device__ __forceinline__ void warp_top3(Top3 t, unsigned long long* key, int* idx) {
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    unsigned long long bk = t.k0;
    int bi = t.i0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long ok = __shfl_xor_sync(0xffffffffu, bk, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (key_less(ok, oi, bk, bi)) {
        bk = ok;
        bi = oi;
      }
    }
    key[r] = bk;
    idx[r] = bi;
    if (t.i0 == bi && bi != INT_MAX) {
      t.k0 = t.k1;
      t.i0 = t.i1;
      t.k1 = t.k2;
      t.i1 = t.i2;
      t.k2 = kInfKey;
      t.i2 = INT_MAX;
    }
  }
}

__device__ __forceinline__ double dot2(double ax, double ay, double bx, double by) {
  return __dadd_rn(__dmul_rn(ax, bx), __dmul_rn(ay, by));
}

__device__ __forceinline__ double node_x(const NearParams& p, int i) { return __dadd_rn(p.o0, __dmul_rn(p.h, (double)i)); }
__device__ __forceinline__ double node_y(const NearParams& p, int i) { return __dadd_rn(p.o1, __dmul_rn(p.h, (double)i)); }

// the interpolated value(s) of one node from its three nearest boundary points (original indices)
__device__ void near_tail(const NearParams& p, int node, const int* i3) {
  const int n = p.n;
  const int ix = node % n, iy = node / n;
  const double px = node_x(p, ix), py = node_y(p, iy);
  double dx[3], dy[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    dx[k] = mimg_fast(__dsub_rn(p.X[i3[k]], px), p);
    dy[k] = mimg_fast(__dsub_rn(p.X[p.M + i3[k]], py), p);
  }
  int a = 0, b = 1;
  double sx = __dsub_rn(dx[0], dx[1]), sy = __dsub_rn(dy[0], dy[1]);
  double tt = -__ddiv_rn(dot2(dx[1], dy[1], sx, sy), dot2(sx, sy, sx, sy));
  if (tt < 0.0 || tt > 1.0) {
    // the pair of the three nearest that lies farthest apart (the first of equal ones)
    const double s01 = sqdist(__dsub_rn(dx[0], dx[1]), __dsub_rn(dy[0], dy[1]));
    const double s02 = sqdist(__dsub_rn(dx[0], dx[2]), __dsub_rn(dy[0], dy[2]));
    const double s12 = sqdist(__dsub_rn(dx[1], dx[2]), __dsub_rn(dy[1], dy[2]));
    if (s02 > s01 && s02 >= s12) {
      b = 2;
    } else if (s12 > s01 && s12 > s02) {
      a = 1;
      b = 2;
    }
    sx = __dsub_rn(dx[a], dx[b]);
    sy = __dsub_rn(dy[a], dy[b]);
    tt = -__ddiv_rn(dot2(dx[b], dy[b], sx, sy), dot2(sx, sy, sx, sy));
    tt = fmin(1.0, fmax(0.0, tt));
  }
  const double ax_ = dx[b] + tt * sx, ay_ = dy[b] + tt * sy;  // x_A − x_p
  const double lseg = hypot(sx, sy);
  const double wa1 = hypot(ax_ - dx[b], ay_ - dy[b]) / lseg;  // weight of U_b(x_1)
  const double wa2 = hypot(ax_ - dx[a], ay_ - dy[a]) / lseg;  // weight of U_b(x_2)
  const double rA = hypot(ax_, ay_);
  const int i1 = i3[a], i2 = i3[b];
  const size_t cells = (size_t)n * n;
  if (rA == 0.0) {
    for (int c = 0; c < p.c; ++c)
      p.out[c * cells + node] = p.Ub[(size_t)c * p.M + i1] * wa1 + p.Ub[(size_t)c * p.M + i2] * wa2;
    return;
  }
  const double bx = ax_ - ax_ / rA * p.m2h, by = ay_ - ay_ / rA * p.m2h;  // x_B − x_p
  const double gx = (px + bx - p.o0) / p.h, gy = (py + by - p.o1) / p.h;
  const double fx = floor(gx), fy = floor(gy);
  const double wx = gx - fx, wy = gy - fy;
  const int jx0 = wrapn((long long)fx, n), jy0 = wrapn((long long)fy, n);
  const int jx1 = jx0 + 1 == n ? 0 : jx0 + 1, jy1 = jy0 + 1 == n ? 0 : jy0 + 1;
  const double rB = hypot(bx, by);
  for (int c = 0; c < p.c; ++c) {
    const double* F = p.u + c * cells;
    const double uA = p.Ub[(size_t)c * p.M + i1] * wa1 + p.Ub[(size_t)c * p.M + i2] * wa2;
    const double uB = (1 - wx) * (1 - wy) * F[(size_t)jy0 * n + jx0] + wx * (1 - wy) * F[(size_t)jy0 * n + jx1] +
                      (1 - wx) * wy * F[(size_t)jy1 * n + jx0] + wx * wy * F[(size_t)jy1 * n + jx1];
    p.out[c * cells + node] = (uA * rB + uB * rA) / p.m2h;
  }
}

// One warp per block: the segments (about 1 000 at 1024²) then spread evenly over the SMs.
constexpr int kNearCap = 128;  // points collected before the lanes run through them
__global__ void __launch_bounds__(32) k_near(NearParams p) {
  __shared__ double cx[kNearCap], cy2[kNearCap];
  __shared__ int ci[kNearCap];
  const int lane = threadIdx.x;
  const int count = *p.count;
  const int n = p.n, sw = segment_width(n);
  const bool whole = 2 * p.K + 3 >= n;
  for (int q = blockIdx.x; q < count; q += gridDim.x) {
    const int cell0 = p.list[q] * sw;
    const int iy = cell0 / n, x0 = cell0 - iy * n;
    const bool take = lane < sw && p.marks[cell0 + lane] && p.omega[cell0 + lane];
    const double px = node_x(p, x0 + lane), py = node_y(p, iy);
    Top3 t;
    t.init();
    int cnt = 0;
    auto flush = [&]() {
      __syncwarp();
#pragma unroll 4
      for (int c = 0; c < cnt; ++c) {
        const double dx = mimg_fast(__dsub_rn(cx[c], px), p);
        t.insert(dbits(__dadd_rn(__dmul_rn(dx, dx), cy2[c])), ci[c]);
      }
      __syncwarp();
      cnt = 0;
    };
    // sorted positions [a, b): the points whose cell column is within K + 1 of the segment
    auto collect = [&](int a, int b) {
      for (int s0 = a; s0 < b; s0 += 32) {
        const int s = s0 + lane;
        bool in = s < b;
        if (in && !whole) in = ((p.base[s] + 1 - (x0 - p.K - 1)) & (n - 1)) <= sw + 2 * p.K + 1;
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (in) {
          const int i = p.perm[s], at = cnt + __popc(m & ((1u << lane) - 1u));
          const double dy = mimg_fast(__dsub_rn(p.X[p.M + i], py), p);
          cx[at] = p.X[i];
          cy2[at] = __dmul_rn(dy, dy);
          ci[at] = i;
        }
        cnt += __popc(m);
        if (cnt > kNearCap - 32) flush();
      }
    };
    if (whole) {
      collect(0, p.M);
    } else {
      const int lo = iy - p.K - 2, hi = iy + p.K + 1;  // rows [lo, hi) of base nodes, wrapped
      if (lo < 0) {
        collect(p.cell_start[lo + n], p.cell_start[n]);
        collect(p.cell_start[0], p.cell_start[hi]);
      } else if (hi > n) {
        collect(p.cell_start[lo], p.cell_start[n]);
        collect(p.cell_start[0], p.cell_start[hi - n]);
      } else {
        collect(p.cell_start[lo], p.cell_start[hi]);
      }
    }
    flush();
    // not within m1·h of Γ (a point outside the rows and columns collected is farther still)
    const bool near = take && t.k0 < p.r1key;
    for (unsigned redo = __ballot_sync(0xffffffffu, near && !whole && !(t.k2 < p.slabkey)); redo; redo &= redo - 1) {
      const int k = __ffs(redo) - 1;
      Top3 a;
      a.init();
      scan_all(p, lane, node_x(p, x0 + k), py, a);
      unsigned long long key[3];
      int idx[3];
      warp_top3(a, key, idx);
      if (lane == k) {
        t.i0 = idx[0];
        t.i1 = idx[1];
        t.i2 = idx[2];
      }
    }
    if (near) {
      const int mine[3] = {t.i0, t.i1, t.i2};
      near_tail(p, cell0 + lane, mine);
    }
  }
}

int pp_blocks(int64_t items) {
  const int64_t b = (items + kPPThreads - 1) / kPPThreads;
  return (int)(b < 152 * 16 ? (b > 0 ? b : 1) : 152 * 16);
}

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// scratch: ones [M] | raw field [n^d] | marks [n²] bytes | list [n²] | count
ibdl_status pp_workspace(Geometry* g, double** ones, double** raw, uint8_t** marks, int** list, int** count) {
  size_t cells = (size_t)g->n * g->n;
  if (g->dim == 3) cells *= g->n;
  const size_t b_ones = align256(sizeof(double) * g->M), b_raw = align256(sizeof(double) * cells);
  const size_t b_marks = g->dim == 2 ? align256(cells) : 0, b_list = g->dim == 2 ? align256(sizeof(int) * cells) : 0;
  const size_t need = b_ones + b_raw + b_marks + b_list + 256;
  if (!g->pp_buf) {
    IBDL_CUDA(cudaMalloc(&g->pp_buf, need));
    g->pp_bytes = need;
  }
  char* p = static_cast<char*>(g->pp_buf);
  *ones = reinterpret_cast<double*>(p);
  *raw = reinterpret_cast<double*>(p + b_ones);
  *marks = reinterpret_cast<uint8_t*>(p + b_ones + b_raw);
  *list = reinterpret_cast<int*>(p + b_ones + b_raw + b_marks);
  *count = reinterpret_cast<int*>(p + b_ones + b_raw + b_marks + b_list);
  return IBDL_OK;
}

}  // namespace

ibdl_status indicator_impl(Geometry* g, double* chi, uint8_t* flags, cudaStream_t s) {
  double *ones, *raw;
  uint8_t* marks;
  int *list, *count;
  IBDL_TRY(pp_workspace(g, &ones, &raw, &marks, &list, &count));
  int64_t cells = (int64_t)g->n * g->n;
  if (g->dim == 3) cells *= g->n;
  k_fill<<<pp_blocks(g->M), kPPThreads, 0, s>>>(ones, g->M, 1.0);
  IBDL_CUDA(cudaGetLastError());
  IBDL_TRY(g->dim == 2 ? laplace_field_2d(g, ones, raw, s) : laplace_field_3d(g, ones, raw, s));
  k_indicator_shift<<<pp_blocks(cells), kPPThreads, 0, s>>>(raw, cells, chi, flags);
  g->launches += 2;
  IBDL_CUDA(cudaGetLastError());
  return IBDL_OK;
}

ibdl_status near_boundary_impl(Geometry* g, const double* Ub, const double* u, const uint8_t* omega, double m1,
                               double m2, double* out, cudaStream_t s) {
  double *ones, *raw;
  uint8_t* marks;
  int *list, *count;
  IBDL_TRY(pp_workspace(g, &ones, &raw, &marks, &list, &count));
  const int n = g->n;
  const int64_t cells = (int64_t)n * n;
  IBDL_CUDA(cudaMemcpyAsync(out, u, sizeof(double) * g->ncomp * cells, cudaMemcpyDeviceToDevice, s));
  IBDL_CUDA(cudaMemsetAsync(marks, 0, cells, s));
  IBDL_CUDA(cudaMemsetAsync(count, 0, sizeof(int), s));
  const int k1 = (int)std::ceil(m1) + 2;
  k_mark<<<pp_blocks((int64_t)g->M * (2 * k1 + 1) * (2 * k1 + 1)), kPPThreads, 0, s>>>(n, (int)g->M, k1, g->base,
                                                                                        marks);
  k_compact<<<pp_blocks(cells), kPPThreads, 0, s>>>(n, cells, marks, omega, list, count);
  NearParams p;
  p.n = n;
  p.M = (int)g->M;
  p.c = g->ncomp;
  p.K = (int)std::ceil(m1) + 4;
  p.h = g->h;
  p.L = g->box;
  p.o0 = g->origin[0];
  p.o1 = g->origin[1];
  const double r1 = m1 * g->h;
  const double r1sq = r1 * r1;
  const double slab = (p.K - 1) * g->h;
  const double slabsq = slab * slab;
  p.halfL = 0.5 * g->box;
  std::memcpy(&p.r1key, &r1sq, 8);
  std::memcpy(&p.slabkey, &slabsq, 8);
  std::memcpy(&p.halfbits, &p.halfL, 8);
  p.m2h = m2 * g->h;
  p.X = g->X64;
  p.base = g->base;
  p.perm = g->perm;
  p.cell_start = g->cell_start;
  p.Ub = Ub;
  p.u = u;
  p.out = out;
  p.marks = marks;
  p.omega = omega;
  p.list = list;
  p.count = count;
  k_near<<<152 * 16, 32, 0, s>>>(p);
  g->launches += 3;
  IBDL_CUDA(cudaGetLastError());
  return IBDL_OK;
}

}  // namespace ibdl
