// Surfel attributes on the GPU: the per-point inputs of Alg. 1 in surfel
// mode, computed from the point cloud alone.
//   radius[i]  mean distance to the k_r nearest other points;
//   normal[i]  the smallest principal axis of the k_n nearest points
//              (itself included), turned to agree with a reference normal
//              or away from the bounding-box centre.
//
// Exact k-nearest-neighbour search on a uniform grid: the bounding box
// (reduced on the device) is cut into G^3 cubic cells, the points are
// counting-sorted into cells, and each point searches shells of cells of
// growing Chebyshev radius until its k-th distance is below the distance to
// every unsearched cell.  Neighbours are ordered by (FP32 squared distance,
// index), with the squared distance evaluated in one fixed order, so the
// neighbour sets -- and the radii, which round as FP64 sums from the nearest on
// do -- equal a brute-force search bit for bit.
#include <cstring>

#include "pe_internal.cuh"

namespace {

constexpr int KMAX = 32;
constexpr int kPtThreads = 128;
constexpr int kBoxBlocks = 256;

struct grid_info {
  float lo[3], ctr[3];
  float h, inv_h;
  int G;
};

__global__ void bbox_partial(const float *__restrict__ pos, int64_t n, float *__restrict__ part) {
  __shared__ float red[6][kPtThreads];
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    for (int k = 0; k < 3; ++k) {
      lo[k] = fminf(lo[k], pos[3 * i + k]);
      hi[k] = fmaxf(hi[k], pos[3 * i + k]);
    }
  for (int k = 0; k < 3; ++k) {
    red[k][threadIdx.x] = lo[k];
    red[3 + k][threadIdx.x] = hi[k];
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    float v = red[threadIdx.x][0];
    for (int t = 1; t < kPtThreads; ++t)
      v = threadIdx.x < 3 ? fminf(v, red[threadIdx.x][t]) : fmaxf(v, red[threadIdx.x][t]);
    part[blockIdx.x * 6 + threadIdx.x] = v;
  }
}

// Cubic cells of side h = (largest extent / G) (1 + 2^-10): the farthest
// point falls in cell G - 1.
__global__ void bbox_final(const float *__restrict__ part, int blocks, int G, grid_info *gi) {
  float lo[3], hi[3];
  for (int k = 0; k < 3; ++k) {
    lo[k] = INFINITY;
    hi[k] = -INFINITY;
    for (int b = threadIdx.x; b < blocks; b += 32) {
      lo[k] = fminf(lo[k], part[b * 6 + k]);
      hi[k] = fmaxf(hi[k], part[b * 6 + 3 + k]);
    }
    for (int o = 16; o > 0; o >>= 1) {
      lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
      hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
    }
  }
  if (threadIdx.x != 0) return;
  float ext = fmaxf(fmaxf(hi[0] - lo[0], hi[1] - lo[1]), hi[2] - lo[2]);
  if (!(ext > 0.0f)) ext = 1.0f;
  grid_info g;
  for (int k = 0; k < 3; ++k) {
    g.lo[k] = lo[k];
    g.ctr[k] = 0.5f * (lo[k] + hi[k]);
  }
  g.G = G;
  g.h = ext / (float)G * (1.0f + 1.0f / 1024.0f);
  g.inv_h = 1.0f / g.h;
  *gi = g;
}

__device__ __forceinline__ int cell_1d(const grid_info &g, float x, int k) {
  int c = (int)floorf((x - g.lo[k]) * g.inv_h);
  return c < 0 ? 0 : (c > g.G - 1 ? g.G - 1 : c);
}

__global__ void count_cells(const float *__restrict__ pos, int64_t n, const grid_info *gip,
                            uint32_t *__restrict__ count, uint32_t *__restrict__ cell_of) {
  const grid_info g = *gip;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t c = ((uint32_t)cell_1d(g, pos[3 * i], 0) * g.G + cell_1d(g, pos[3 * i + 1], 1)) * g.G +
                       cell_1d(g, pos[3 * i + 2], 2);
    cell_of[i] = c;
    atomicAdd(count + c, 1u);
  }
}

__global__ void scatter_cells(int64_t n, const uint32_t *__restrict__ cell_of,
                              const uint32_t *__restrict__ offs, uint32_t *__restrict__ cursor,
                              uint32_t *__restrict__ sorted) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t c = cell_of[i];
    sorted[offs[c] + atomicAdd(cursor + c, 1u)] = (uint32_t)i;
  }
}

// The points as 16-byte records {x, y, z, index} in cell order: inside a cell in
// whatever order the atomics give (SORTED = false; the radii do not depend on it),
// or their indices alone, for sort_cells to follow.  count ends at zero.
template <bool SORTED>
__global__ void scatter_points(const float *__restrict__ pos, int64_t n,
                               const uint32_t *__restrict__ cell_of,
                               const uint32_t *__restrict__ offs, uint32_t *__restrict__ count,
                               uint32_t *__restrict__ idx, float4 *__restrict__ pts) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t c = cell_of[i], at = offs[c] + atomicSub(count + c, 1u) - 1u;
    if (SORTED) idx[at] = (uint32_t)i;
    else pts[at] = make_float4(pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], __uint_as_float((uint32_t)i));
  }
}

// The records with the points of a cell by index, so that what is added up in
// this order (the moments of a normal) is the same on every run: a thread per
// point counts the smaller indices of its cell.  A million points, about 36 to a
// cell: 18 us of the 850 for radii and normals.
__global__ void sort_cells(const float *__restrict__ pos, int64_t n,
                           const uint32_t *__restrict__ cell_of, const uint32_t *__restrict__ offs,
                           const uint32_t *__restrict__ idx, float4 *__restrict__ pts) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t i = idx[t], c = cell_of[i], b = offs[c], e = offs[c + 1];
    uint32_t at = b;
    for (uint32_t k = b; k < e; ++k) at += __ldg(idx + k) < i;
    const float *p = pos + 3 * (int64_t)i;
    pts[at] = make_float4(p[0], p[1], p[2], __uint_as_float(i));
  }
}

// FP64 issues at 1/64 of the FP32 rate here, so sums that need more than FP32
// run in pairs of floats (sum s and its error c): an addition's error by Knuth's
// two-sum, a product's by one FMA (the compensated dot product of Ogita, Rump and
// Oishi, as accurate as twice the working precision).
struct pair_sum {
  float s = 0.0f, c = 0.0f;
  __device__ __forceinline__ void add(float v, float e) {  // v + e, |e| small against |v|
    const float t = __fadd_rn(s, v), z = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(v, z)), e));
    s = t;
  }
  // (xh + xl)(yh + yl) without xl yl
  __device__ __forceinline__ void add_product(float xh, float xl, float yh, float yl) {
    const float p = __fmul_rn(xh, yh);
    add(p, fmaf(xh, yl, fmaf(xl, yh, fmaf(xh, yh, -p))));
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};
// a - b = h + l exactly
__device__ __forceinline__ void two_diff(float a, float b, float &h, float &l) {
  h = __fsub_rn(a, b);
  const float z = __fsub_rn(h, a);
  l = __fsub_rn(__fsub_rn(a, __fsub_rn(h, z)), __fadd_rn(b, z));
}
// The range of squared distances in which no product or error term of the pair
// arithmetic that matters leaves the normal floats; outside it FP64 is used.
constexpr float kPairMin = 1e-20f, kPairMax = 1e30f;

// Smallest-eigenvalue unit eigenvector of the symmetric 3x3 matrix
// (a00 a01 a02; a11 a12; a22) by the trigonometric solution of the
// characteristic cubic and the largest cross product of two rows of
// A - lambda I.  (0, 0, 1) when A is a multiple of the identity.
__device__ void smallest_axis(double a00, double a01, double a02, double a11, double a12,
                              double a22, double out[3]) {
  const double p1 = a01 * a01 + a02 * a02 + a12 * a12;
  const double q = (a00 + a11 + a22) / 3.0;
  const double b00 = a00 - q, b11 = a11 - q, b22 = a22 - q;
  const double p2 = b00 * b00 + b11 * b11 + b22 * b22 + 2.0 * p1;
  if (!(p2 > 0.0)) {
    out[0] = 0.0;
    out[1] = 0.0;
    out[2] = 1.0;
    return;
  }
  const double p = sqrt(p2 / 6.0);
  const double ip = 1.0 / p;
  const double c00 = b00 * ip, c11 = b11 * ip, c22 = b22 * ip, c01 = a01 * ip, c02 = a02 * ip,
               c12 = a12 * ip;
  double r = 0.5 * (c00 * (c11 * c22 - c12 * c12) - c01 * (c01 * c22 - c12 * c02) +
                    c02 * (c01 * c12 - c11 * c02));
  r = r < -1.0 ? -1.0 : (r > 1.0 ? 1.0 : r);
  const double phi = acos(r) / 3.0;
  const double lam = q + 2.0 * p * cos(phi + 2.0943951023931957);  // + 2 pi / 3: smallest
  const double r0[3] = {a00 - lam, a01, a02}, r1[3] = {a01, a11 - lam, a12},
               r2[3] = {a02, a12, a22 - lam};
  double best[3] = {0.0, 0.0, 1.0}, bn = 0.0;
  const double *rows[3][2] = {{r0, r1}, {r0, r2}, {r1, r2}};
  for (int k = 0; k < 3; ++k) {
    const double *u = rows[k][0], *v = rows[k][1];
    const double c[3] = {u[1] * v[2] - u[2] * v[1], u[2] * v[0] - u[0] * v[2],
                         u[0] * v[1] - u[1] * v[0]};
    const double nn = c[0] * c[0] + c[1] * c[1] + c[2] * c[2];
    if (nn > bn) {
      bn = nn;
      best[0] = c[0];
      best[1] = c[1];
      best[2] = c[2];
    }
  }
  const double s = bn > 0.0 ? 1.0 / sqrt(bn) : 1.0;
  out[0] = best[0] * s;
  out[1] = best[1] * s;
  out[2] = best[2] * s;
}

// The same axis with FP32 where only a starting value is needed: the matrix is
// scaled by an approximate 1 / p, the cubic's smallest root starts from the FP32
// trigonometric solution (error about 1e-6) and takes two Newton steps in FP64,
// and the length's reciprocal root one; all that is left in FP64 is what the
// result's precision rests on (about 100 operations; the square roots, divisions,
// arc cosine and cosine of the full solution take several times as many).  False
// (and no result) where the two smallest eigenvalues are close, since Newton's
// steps need the cubic's slope, for matrices out of the floats' range, and where
// the squared deviation p^2 from a multiple of the identity, q^2 times the
// identity's, is not above iso q^2.
__device__ bool smallest_axis_newton(double a00, double a01, double a02, double a11, double a12,
                                     double a22, float iso, double out[3]) {
  const double q = (a00 + a11 + a22) * (1.0 / 3.0);
  const double b00 = a00 - q, b11 = a11 - q, b22 = a22 - q;
  float p2;
  {
    const float x = (float)b00, y = (float)b11, z = (float)b22, u = (float)a01, v = (float)a02,
                w = (float)a12;
    p2 = x * x + y * y + z * z + 2.0f * (u * u + v * v + w * w);
  }
  if (!(p2 > 1e-30f && p2 < 1e30f && p2 > iso * ((float)q * (float)q))) return false;
  const double ip = (double)rsqrtf(p2 * (1.0f / 6.0f));
  const double c00 = b00 * ip, c11 = b11 * ip, c22 = b22 * ip, c01 = a01 * ip, c02 = a02 * ip,
               c12 = a12 * ip;
  // det(C - x I) = -(x^3 - k x - d), k = 3 up to the scale's rounding
  const double k = 0.5 * (c00 * c00 + c11 * c11 + c22 * c22) + c01 * c01 + c02 * c02 + c12 * c12;
  const double d = c00 * (c11 * c22 - c12 * c12) - c01 * (c01 * c22 - c12 * c02) +
                   c02 * (c01 * c12 - c11 * c02);
  const float r = fminf(fmaxf(0.5f * (float)d, -1.0f), 1.0f);
  const float x0 = 2.0f * cosf(acosf(r) * (1.0f / 3.0f) + 2.0943951f);  // + 2 pi / 3: smallest
  const float slope = 3.0f * x0 * x0 - (float)k;
  if (!(slope > 0.05f)) return false;
  const double is = (double)__frcp_rn(slope);
  double x = (double)x0;
#pragma unroll
  for (int it = 0; it < 2; ++it) x -= ((x * x - k) * x - d) * is;
  const double e00 = c00 - x, e11 = c11 - x, e22 = c22 - x;
  // the largest cross product of two rows
  double b[3] = {c01 * c12 - c02 * e11, c02 * c01 - e00 * c12, e00 * e11 - c01 * c01};  // 0 x 1
  double bn = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
  const double f[3] = {c01 * e22 - c02 * c12, c02 * c02 - e00 * e22, e00 * c12 - c01 * c02};  // 0 x 2
  const double fn = f[0] * f[0] + f[1] * f[1] + f[2] * f[2];
  const double h[3] = {e11 * e22 - c12 * c12, c12 * c02 - c01 * e22, c01 * c12 - e11 * c02};  // 1 x 2
  const double hn = h[0] * h[0] + h[1] * h[1] + h[2] * h[2];
  if (fn > bn) {
    bn = fn;
    b[0] = f[0];
    b[1] = f[1];
    b[2] = f[2];
  }
  if (hn > bn) {
    bn = hn;
    b[0] = h[0];
    b[1] = h[1];
    b[2] = h[2];
  }
  double s = (double)rsqrtf((float)bn);
  s *= 1.5 - 0.5 * bn * s * s;
  out[0] = b[0] * s;
  out[1] = b[1] * s;
  out[2] = b[2] * s;
  return true;
}

struct knn_args {
  const float4 *pts;  // {x, y, z, index} in cell order
  int64_t n;
  const grid_info *gi;
  const uint32_t *offs;
  int K, k_r, k_n;
  double inv_r, inv_n;  // 1 / k_r, 1 / k_n
  uint32_t err_r;       // bound of the error of k_r roots added in pairs, in 2^-53 of the sum
  const float *ref;
  float *rad, *nrm;
  unsigned int *err;
};

__device__ __forceinline__ float d2_pts(float4 q, float4 p) {
  const float dx = __fsub_rn(p.x, q.x), dy = __fsub_rn(p.y, q.y), dz = __fsub_rn(p.z, q.z);
  return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

// Calls f(begin, end) for the runs of points in the cells at Chebyshev distance
// lo..hi from c: cells are stored with z fastest, so the cells of one (x, y)
// column are one run (two around the part nearer than lo).
template <class F>
__device__ __forceinline__ void for_runs(const uint32_t *__restrict__ offs, int G, const int c[3],
                                         int lo, int hi, F &&f) {
  const int x0 = max(c[0] - hi, 0), x1 = min(c[0] + hi, G - 1);
  const int y0 = max(c[1] - hi, 0), y1 = min(c[1] + hi, G - 1);
  const int z0 = max(c[2] - hi, 0), z1 = min(c[2] + hi, G - 1);
  for (int x = x0; x <= x1; ++x)
    for (int y = y0; y <= y1; ++y) {
      const uint32_t col = ((uint32_t)x * G + y) * G;
      if (lo == 0 || abs(x - c[0]) >= lo || abs(y - c[1]) >= lo) {
        f(__ldg(offs + col + z0), __ldg(offs + col + z1 + 1));
      } else {
        if (z0 <= c[2] - lo) f(__ldg(offs + col + z0), __ldg(offs + col + c[2] - lo + 1));
        if (c[2] + lo <= z1) f(__ldg(offs + col + c[2] + lo), __ldg(offs + col + z1 + 1));
      }
    }
}

// One thread per point, in two scans of its neighbourhood.  The first keeps the
// KT >= K smallest squared distances in registers, sorted: a candidate goes
// through the list by min and max alone (two instructions per entry, no
// indices, no branches beyond one test against the last).  That list alone gives
// the radius: the point itself is one of its zeros, whatever the order of ties.
// The second scan, for the normal, collects the points nearer than the k_n-th
// distance and, of those at it, the smallest indices, into shared memory; their
// moments about the query point are then summed by all lanes together, in pairs
// of floats (within 2^-38 of the sum of the products' sizes, 2^-46 as a rule), and
// the axis found with as little FP64 as its precision needs.  Where the axis is
// badly conditioned (two near eigenvalues, or three), the moments are summed again
// in FP64; elsewhere 2^-46 of them moves the axis by less than 2^-32.
// The points are read as 16-byte records in cell order, a run per (x, y) column
// of cells, and queries follow the same order, so a warp mostly reads the same
// records.  A million points, k_r = 8, k_n = 16: 2.35 ms with lists of (distance,
// index) in local memory, insertion by a data-dependent loop and 27 cells visited
// one by one (13.6 of 32 lanes active); 1.28 ms with both scans as above and
// moments, roots and eigenvectors in FP64, at a 64th of the FP32 rate; 0.70 ms now
// (0.02 of it for radii that round as FP64 does and for points that are NaN).
template <int KT>
__global__ void __launch_bounds__(kPtThreads, KT <= 16 ? 8 : (KT <= 24 ? 7 : 6))
    knn_kernel(const knn_args A) {
  extern __shared__ uint32_t s_list[];  // [k_n][kPtThreads]: positions in pts
  const grid_info g = *A.gi;
  const int G = g.G;
  const int64_t t = (int64_t)blockIdx.x * kPtThreads + threadIdx.x;
  if (t >= A.n) return;
  const float4 q = __ldg(A.pts + t);
  const uint32_t i = __float_as_uint(q.w);
  const int c[3] = {cell_1d(g, q.x, 0), cell_1d(g, q.y, 1), cell_1d(g, q.z, 2)};
  const float qq[3] = {q.x, q.y, q.z};
  const int K = A.K;
  // A NaN coordinate makes NaN of every distance it enters, and a NaN enters no
  // list: such a point has no neighbours and is nobody's.
  if (q.x != q.x || q.y != q.y || q.z != q.z) {
    if (A.rad) A.rad[i] = NAN;
    if (A.nrm)
      for (int k = 0; k < 3; ++k) A.nrm[3 * (int64_t)i + k] = NAN;
    return;
  }
  float bd[KT];
#pragma unroll
  for (int k = 0; k < KT; ++k) bd[k] = INFINITY;
  // the entry at a runtime position (a constant chain of selects)
  auto at = [&](int k) {
    float v = bd[0];
#pragma unroll
    for (int e = 1; e < KT; ++e) v = e == k ? bd[e] : v;
    return v;
  };
  uint32_t seen = 0;
  int s = 1;  // cells within Chebyshev distance s are searched
  for (int lo = 0;; lo = ++s) {
    for_runs(A.offs, G, c, lo, s, [&](uint32_t b, uint32_t e) {
      seen += e - b;
      for (uint32_t m = b; m < e; ++m) {
        const float d2 = d2_pts(q, __ldg(A.pts + m));
        if (d2 < bd[KT - 1]) {
#pragma unroll
          for (int k = KT - 1; k > 0; --k) bd[k] = fmaxf(bd[k - 1], fminf(bd[k], d2));
          bd[0] = fminf(bd[0], d2);
        }
      }
    });
    // stop once the k-th distance is below the distance to every cell
    // outside the searched block (faces at the grid's edge bound nothing)
    float bound = INFINITY;
    for (int k = 0; k < 3; ++k) {
      const float slack = 1e-4f * g.h + 1e-6f * (fabsf(g.lo[k]) + (float)G * g.h);
      if (c[k] - s > 0) bound = fminf(bound, qq[k] - (g.lo[k] + (float)(c[k] - s) * g.h) - slack);
      if (c[k] + s + 1 < G)
        bound = fminf(bound, (g.lo[k] + (float)(c[k] + s + 1) * g.h) - qq[k] - slack);
    }
    if (bound == INFINITY) break;  // every cell searched
    if (seen >= (uint32_t)K && bound > 0.0f && at(K - 1) <= bound * bound) break;
  }
  if (seen < (uint32_t)K) {  // fewer than K points in the cloud: rejected on the host
    pe_raise(A.err, PE_ERR_OVERFLOW);
    return;
  }
  // (an entry that no distance took is infinite, like a distance that overflows)
  bool full = true;
  if (A.rad && !(at(A.k_r) < INFINITY)) {
    uint32_t found = 0;
    for_runs(A.offs, G, c, 0, s, [&](uint32_t b, uint32_t e) {
      for (uint32_t m = b; m < e; ++m) found += d2_pts(q, __ldg(A.pts + m)) >= 0.0f;
    });
    // (an infinite coordinate is at a NaN distance from itself)
    full = found >= (uint32_t)A.k_r + (d2_pts(q, q) == 0.0f);
  }
  if (!full) {
    A.rad[i] = NAN;
  } else if (A.rad) {
    // the first entry is the point's own zero; were it pushed out by more than
    // K coincident points, every entry would be zero
    // (a root of d: its float r and the rest d - r^2, exact in one FMA, over 2 r)
    pair_sum sum;
    bool in_range = true;
#pragma unroll
    for (int e = 1; e < KT; ++e)
      if (e <= A.k_r) {
        if (bd[e] > kPairMin && bd[e] < kPairMax) {
          const float r = __fsqrt_rn(bd[e]);
          sum.add(r, __fdividef(fmaf(-r, r, bd[e]), 2.0f * r));
        } else if (bd[e] != 0.0f) {
          in_range = false;
        }
      }
    // Unless a boundary between two floats lies within the pair's error of the
    // mean, the FP64 mean rounds to the same float; else (for one point in 40000
    // at k_r = 8) FP64 decides.  A float takes 24 of the mean's 53 bits: a
    // boundary is where the other 29 are one half.
    const double mean = sum.value() * A.inv_r;
    float rad = (float)mean;
    const uint32_t rest = (uint32_t)__double2loint(mean) & 0x1fffffffu;
    if (!in_range || rest - 0x10000000u + A.err_r <= 2u * A.err_r) {
      double total = 0.0;
#pragma unroll
      for (int e = 1; e < KT; ++e)
        if (e <= A.k_r) total += sqrt((double)bd[e]);
      rad = (float)(total / (double)A.k_r);
    }
    A.rad[i] = rad;
  }
  if (A.nrm) {
    const int kn = A.k_n;
    const float tau = at(kn - 1);
    int below = 0;  // entries nearer than the k_n-th: the list's points from there on tie
#pragma unroll
    for (int e = 0; e < KT; ++e) below += e < kn && bd[e] < tau;
    uint32_t *list = s_list + threadIdx.x;
    int n_lt = 0, n_eq = below;
    for_runs(A.offs, G, c, 0, s, [&](uint32_t b, uint32_t e) {
      for (uint32_t m = b; m < e; ++m) {
        const float4 p = __ldg(A.pts + m);
        const float d2 = d2_pts(q, p);
        if (!(d2 <= tau)) continue;
        if (d2 < tau) {
          list[n_lt++ * kPtThreads] = m;
        } else if (n_eq < kn) {
          list[n_eq++ * kPtThreads] = m;
        } else {
          // a tie too many: the largest index of the tied goes
          int worst = below;
          uint32_t wi = 0;
          for (int k = below; k < kn; ++k) {
            const uint32_t id = __float_as_uint(__ldg(A.pts + list[k * kPtThreads]).w);
            if (id >= wi) {
              wi = id;
              worst = k;
            }
          }
          if (__float_as_uint(p.w) < wi) list[worst * kPtThreads] = m;
        }
      }
    });
    if (n_lt != below || n_eq != kn) {  // fewer than k_n distances in the whole cloud
      for (int k = 0; k < 3; ++k) A.nrm[3 * (int64_t)i + k] = NAN;
      return;
    }
    // moments about the query point, of exact differences; then about the mean
    double v[3];
    bool have = false;
    if (tau > kPairMin && tau < kPairMax) {
      pair_sum mx, my, mz, xx, xy, xz, yy, yz, zz;
      for (int k = 0; k < kn; ++k) {
        const float4 p = __ldg(A.pts + list[k * kPtThreads]);
        float x, y, z, dx, dy, dz;
        two_diff(p.x, q.x, x, dx);
        two_diff(p.y, q.y, y, dy);
        two_diff(p.z, q.z, z, dz);
        mx.add(x, dx);
        my.add(y, dy);
        mz.add(z, dz);
        xx.add_product(x, dx, x, dx);
        xy.add_product(x, dx, y, dy);
        xz.add_product(x, dx, z, dz);
        yy.add_product(y, dy, y, dy);
        yz.add_product(y, dy, z, dz);
        zz.add_product(z, dz, z, dz);
      }
      const double m0 = mx.value(), m1 = my.value(), m2 = mz.value();
      const double c0 = m0 * A.inv_n, c1 = m1 * A.inv_n, c2 = m2 * A.inv_n;
      have = smallest_axis_newton(xx.value() - m0 * c0, xy.value() - m0 * c1, xz.value() - m0 * c2,
                                  yy.value() - m1 * c1, yz.value() - m1 * c2, zz.value() - m2 * c2,
                                  1e-4f, v);
    }
    if (!have) {
      double m0 = 0, m1 = 0, m2 = 0, a00 = 0, a01 = 0, a02 = 0, a11 = 0, a12 = 0, a22 = 0;
#pragma unroll 1
      for (int k = 0; k < kn; ++k) {
        const float4 p = __ldg(A.pts + list[k * kPtThreads]);
        const double x = (double)p.x - (double)q.x, y = (double)p.y - (double)q.y,
                     z = (double)p.z - (double)q.z;
        m0 += x;
        m1 += y;
        m2 += z;
        a00 += x * x;
        a01 += x * y;
        a02 += x * z;
        a11 += y * y;
        a12 += y * z;
        a22 += z * z;
      }
      const double c0 = m0 * A.inv_n, c1 = m1 * A.inv_n, c2 = m2 * A.inv_n;
      a00 -= m0 * c0;
      a01 -= m0 * c1;
      a02 -= m0 * c2;
      a11 -= m1 * c1;
      a12 -= m1 * c2;
      a22 -= m2 * c2;
      if (!smallest_axis_newton(a00, a01, a02, a11, a12, a22, 0.0f, v))
        smallest_axis(a00, a01, a02, a11, a12, a22, v);
    }
    double w[3];
    if (A.ref) {
      for (int k = 0; k < 3; ++k) w[k] = (double)A.ref[3 * (int64_t)i + k];
    } else {
      for (int k = 0; k < 3; ++k) w[k] = (double)qq[k] - (double)g.ctr[k];
    }
    if (v[0] * w[0] + v[1] * w[1] + v[2] * w[2] < 0.0)
      for (int k = 0; k < 3; ++k) v[k] = -v[k];
    for (int k = 0; k < 3; ++k) A.nrm[3 * (int64_t)i + k] = (float)v[k];
  }
}

template <int KT>
void launch_knn(const knn_args &A, cudaStream_t s) {
  const size_t smem = A.nrm ? sizeof(uint32_t) * kPtThreads * A.k_n : 0;
  knn_kernel<KT><<<(unsigned)((A.n + kPtThreads - 1) / kPtThreads), kPtThreads, smem, s>>>(A);
}

int grid_res(int64_t n) {
  // about (2.5 n^(1/3))^3 cells: a surface sampled by n points puts a few
  // dozen points in each occupied cell
  double g = 2.5 * cbrt((double)n);
  int G = (int)g;
  return G < 4 ? 4 : (G > 255 ? 255 : G);
}

struct pt_ws {
  float *part;
  grid_info *gi;
  uint32_t *count, *offs, *cursor, *tile, *cell_of, *idx;
  float4 *pts;
};

pt_ws carve(pe_carve &c, int64_t n) {
  const int G = grid_res(n);
  const int64_t cells = (int64_t)G * G * G;
  pt_ws w;
  w.part = c.take<float>(kBoxBlocks * 6);
  w.gi = c.take<grid_info>(1);
  w.count = c.take<uint32_t>((size_t)cells);
  w.offs = c.take<uint32_t>((size_t)cells + 1);
  w.cursor = nullptr;
  w.tile = c.take<uint32_t>((size_t)((cells + 4095) / 4096 + 1));
  w.cell_of = c.take<uint32_t>((size_t)n);
  w.idx = c.take<uint32_t>((size_t)n);
  w.pts = c.take<float4>((size_t)n);
  return w;
}

}  // namespace

namespace {

// The processing order of pe_order_points: the same counting sort into a
// 32^3 grid over the bounding box, cells in raster order (a warp's 32 points
// then mostly share a cell of about 1/32 of the target's extent).
constexpr int kOrderGrid = 32;

pt_ws carve_order(pe_carve &c, int64_t n) {
  const int64_t cells = (int64_t)kOrderGrid * kOrderGrid * kOrderGrid;
  pt_ws w;
  w.part = c.take<float>(kBoxBlocks * 6);
  w.gi = c.take<grid_info>(1);
  w.count = c.take<uint32_t>((size_t)cells);
  w.offs = c.take<uint32_t>((size_t)cells + 1);
  w.cursor = c.take<uint32_t>((size_t)cells);
  w.tile = c.take<uint32_t>((size_t)((cells + 4095) / 4096 + 1));
  w.cell_of = c.take<uint32_t>((size_t)n);
  w.idx = nullptr;
  w.pts = nullptr;
  return w;
}

}  // namespace

extern "C" size_t pe_order_points_workspace(int64_t n_points) {
  if (n_points < 1 || n_points >= (int64_t)UINT32_MAX) return 0;
  pe_carve c{nullptr, 0};
  carve_order(c, n_points);
  return c.bytes() + 256;
}

extern "C" pe_status pe_order_points(const float *pos, int64_t n_points, void *ws, size_t ws_bytes,
                                     uint32_t *order, void *stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (!pos || !order || n_points < 1 || n_points >= (int64_t)UINT32_MAX)
    return pe_fail(PE_EINVAL, "pe_order_points: bad arguments");
  const size_t need = pe_order_points_workspace(n_points);
  if (!ws || ws_bytes < need || !pe_aligned(ws, 256))
    return pe_fail(PE_ENOMEM, "pe_order_points: workspace needs %zu bytes", need);
  pe_carve c{static_cast<char *>(ws), 0};
  pt_ws w = carve_order(c, n_points);
  const int64_t cells = (int64_t)kOrderGrid * kOrderGrid * kOrderGrid;
  bbox_partial<<<kBoxBlocks, kPtThreads, 0, s>>>(pos, n_points, w.part);
  PE_TRY_LAUNCH("bbox_partial");
  bbox_final<<<1, 32, 0, s>>>(w.part, kBoxBlocks, kOrderGrid, w.gi);
  PE_TRY_LAUNCH("bbox_final");
  PE_TRY_CUDA(cudaMemsetAsync(w.count, 0, sizeof(uint32_t) * cells, s));
  PE_TRY_CUDA(cudaMemsetAsync(w.cursor, 0, sizeof(uint32_t) * cells, s));
  int64_t b = (n_points + 255) / 256;
  const int blocks = (int)(b < 4096 ? b : 4096);
  count_cells<<<blocks, 256, 0, s>>>(pos, n_points, w.gi, w.count, w.cell_of);
  PE_TRY_LAUNCH("count_cells");
  pe_status st = pe_exclusive_scan_u32(w.count, cells, w.tile, w.offs, s);
  if (st != PE_OK) return st;
  scatter_cells<<<blocks, 256, 0, s>>>(n_points, w.cell_of, w.offs, w.cursor, order);
  PE_TRY_LAUNCH("scatter_cells");
  return PE_OK;
}

extern "C" size_t pe_point_attributes_workspace(int64_t n_points) {
  if (n_points < 1) return 0;
  pe_carve c{nullptr, 0};
  carve(c, n_points);
  return c.bytes() + 256;
}

extern "C" pe_status pe_point_attributes(const float *pos, int64_t n_points, int32_t k_r,
                                         int32_t k_n, const float *ref_nrm, void *ws,
                                         size_t ws_bytes, float *radius, float *normal,
                                         void *stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (!pos || n_points < 1 || n_points >= (int64_t)UINT32_MAX || (!radius && !normal))
    return pe_fail(PE_EINVAL, "pe_point_attributes: bad arguments");
  if ((radius && (k_r < 1 || k_r > KMAX - 1)) || (normal && (k_n < 3 || k_n > KMAX)))
    return pe_fail(PE_EINVAL, "pe_point_attributes: k_r in [1, %d], k_n in [3, %d]", KMAX - 1, KMAX);
  const int K = (radius ? k_r + 1 : 0) > (normal ? k_n : 0) ? k_r + 1 : (normal ? k_n : 0);
  if (n_points < K)
    return pe_fail(PE_EINVAL, "pe_point_attributes: needs at least %d points", K);
  const size_t need = pe_point_attributes_workspace(n_points);
  if (!ws || ws_bytes < need || !pe_aligned(ws, 256))
    return pe_fail(PE_ENOMEM, "pe_point_attributes: workspace needs %zu bytes", need);
  pe_carve c{static_cast<char *>(ws), 0};
  pt_ws w = carve(c, n_points);
  const int G = grid_res(n_points);
  const int64_t cells = (int64_t)G * G * G;
  bbox_partial<<<kBoxBlocks, kPtThreads, 0, s>>>(pos, n_points, w.part);
  PE_TRY_LAUNCH("bbox_partial");
  bbox_final<<<1, 32, 0, s>>>(w.part, kBoxBlocks, G, w.gi);
  PE_TRY_LAUNCH("bbox_final");
  PE_TRY_CUDA(cudaMemsetAsync(w.count, 0, sizeof(uint32_t) * cells, s));
  int64_t b = (n_points + 255) / 256;
  const int blocks = (int)(b < 4096 ? b : 4096);
  count_cells<<<blocks, 256, 0, s>>>(pos, n_points, w.gi, w.count, w.cell_of);
  PE_TRY_LAUNCH("count_cells");
  pe_status st = pe_exclusive_scan_u32(w.count, cells, w.tile, w.offs, s);
  if (st != PE_OK) return st;
  if (normal) {
    scatter_points<true><<<blocks, 256, 0, s>>>(pos, n_points, w.cell_of, w.offs, w.count, w.idx, w.pts);
    PE_TRY_LAUNCH("scatter_points");
    sort_cells<<<blocks, 256, 0, s>>>(pos, n_points, w.cell_of, w.offs, w.idx, w.pts);
    PE_TRY_LAUNCH("sort_cells");
  } else {
    scatter_points<false><<<blocks, 256, 0, s>>>(pos, n_points, w.cell_of, w.offs, w.count, w.idx, w.pts);
    PE_TRY_LAUNCH("scatter_points");
  }
  knn_args A;
  memset(&A, 0, sizeof(A));
  A.pts = w.pts;
  A.n = n_points;
  A.gi = w.gi;
  A.offs = w.offs;
  A.K = K;
  A.k_r = k_r;
  A.k_n = k_n;
  A.inv_r = 1.0 / (double)(k_r > 0 ? k_r : 1);
  A.inv_n = 1.0 / (double)(k_n > 0 ? k_n : 1);
  // k_r corrections, each summed with roundings of at most 3 k_r 2^-48 of the sum;
  // a root's own correction errs by at most 2^-46 of it; 2^-48 = 2^5 2^-53
  A.err_r = (uint32_t)((3 * k_r * k_r + 8) << 5);
  A.ref = ref_nrm;
  A.rad = radius;
  A.nrm = normal;
  A.err = pe_err_word();
  pe_event_before("knn_kernel", s);
  if (K <= 9) launch_knn<9>(A, s);
  else if (K <= 12) launch_knn<12>(A, s);
  else if (K <= 16) launch_knn<16>(A, s);
  else if (K <= 24) launch_knn<24>(A, s);
  else launch_knn<KMAX>(A, s);
  pe_event_after("knn_kernel", s);
  PE_TRY_LAUNCH("knn_kernel");
  return PE_OK;
}
