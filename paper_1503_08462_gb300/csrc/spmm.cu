// Sparse kernels of the solve path: CSR times row-major blocks of vectors.
//
// Layout: every block of vectors is row-major [rows][width], so the `width`
// values of one row are contiguous and a gathered neighbour row is one
// coalesced segment.  A group of G threads (G = width rounded up to a power of
// two, at most 32) owns one matrix row; thread t of the group accumulates the
// columns t, t+G, ... (CPT columns per thread).  Column indices and values of
// the row are loaded once per group (same address across the group).
//
// Steps served (Algorithm 3.1, 0-based levels):
//   defect       r_j = lambda_j M_k u_j - A_k u_j (Eq. Linear_Equation; the
//                AMG call from the initial guess u_j is run in defect form)
//   smoothing    point l1-Jacobi x <- x + D^-1 (b - A x), D = diag(sum_j |a_ij|)
//   transfers    restriction R_l = P_l^T and prolongation P_l (Sec. 2.3)
//   augmentation A_k V and M_k V for the pencil of Algorithm 3.1 step 2
//   recombine    u_j = I_n^k x_j(1:d_n) + V x_j(d_n+1:d_n+q)
#include <algorithm>
#include <cstdio>

#include "common.cuh"
#include "kernels.cuh"
#include "prof.cuh"

namespace amgeig {
namespace {

constexpr int kThreads = 256;

struct Geo {
  int G, rows_per_block, cpt;
};

Geo geo_for(int width) {
  int G = 1;
  while (G < width && G < 32) G <<= 1;
  int cpt = (width + G - 1) / G;
  int c = 1;
  while (c < cpt) c <<= 1;
  return Geo{G, kThreads / G, c};
}

template <typename T>
struct Acc;
template <>
struct Acc<double> {
  using type = double;
};
template <>
struct Acc<float> {
  using type = float;
};

// ------------------------------------------------------------------ defect

template <int CPT, typename TO>
__global__ void __launch_bounds__(kThreads) k_defect(int n, const int* __restrict__ rp, const int* __restrict__ ci,
                                                     const double* __restrict__ a, const double* __restrict__ m,
                                                     const double* __restrict__ U, int q,
                                                     const double* __restrict__ lam, TO* __restrict__ R, int ldr,
                                                     int G, double* __restrict__ partials) {
  extern __shared__ double sred[];  // [rows_per_block][2*G*CPT] when partials != null
  const int rpb = blockDim.x / G;
  const int g = threadIdx.x / G;
  const int lane = threadIdx.x % G;
  const int row = blockIdx.x * rpb + g;
  double aa[CPT], mm[CPT];
#pragma unroll
  for (int t = 0; t < CPT; ++t) aa[t] = mm[t] = 0.0;
  if (row < n) {
    const int p0 = rp[row], p1 = rp[row + 1];
    for (int p = p0; p < p1; ++p) {
      const int j = ci[p];
      const double av = a[p], mv = m[p];
      const double* uj = U + static_cast<long long>(j) * q;
#pragma unroll
      for (int t = 0; t < CPT; ++t) {
        const int c = lane + t * G;
        if (c < q) {
          const double u = uj[c];
          aa[t] = fma(av, u, aa[t]);
          mm[t] = fma(mv, u, mm[t]);
        }
      }
    }
  }
  double rr[CPT];
#pragma unroll
  for (int t = 0; t < CPT; ++t) {
    const int c = lane + t * G;
    rr[t] = 0.0;
    if (row < n && c < q) {
      const double r = fma(lam[c], mm[t], -aa[t]);
      R[static_cast<long long>(row) * ldr + c] = static_cast<TO>(r);
      rr[t] = r;
    }
  }
  if (row < n)
    for (int c = q + lane; c < ldr; c += G) R[static_cast<long long>(row) * ldr + c] = TO(0);
  if (partials == nullptr) return;
  // per-column sums of r^2 and (Mu)^2 over the block's rows, fixed order
  const int W = G * CPT;
#pragma unroll
  for (int t = 0; t < CPT; ++t) {
    sred[g * 2 * W + lane + t * G] = rr[t] * rr[t];
    sred[g * 2 * W + W + lane + t * G] = (row < n) ? mm[t] * mm[t] : 0.0;
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < 2 * q; idx += blockDim.x) {
    const int which = idx / q, c = idx % q;
    double s = 0.0;
    for (int r = 0; r < rpb; ++r) s += sred[r * 2 * W + which * W + c];
    partials[static_cast<long long>(blockIdx.x) * 2 * q + idx] = s;
  }
}

template <typename TO>
void defect_impl(const DevCsr& AM, const double* U, int q, const double* lam, TO* R, int ldr, double* partials,
                 int* nblocks_out, cudaStream_t st) {
  Geo g = geo_for(q);
  const int blocks = ceil_div(AM.rows, g.rows_per_block);
  if (nblocks_out) *nblocks_out = blocks;
  const double N = AM.rows, nnz = AM.nnz;
  ProfScope ps(st, P_DEFECT, 4.0 * (N + 1) + 20.0 * nnz + 8.0 * N * q + sizeof(TO) * N * q, 4.0 * nnz * q);
  const size_t sm = partials ? sizeof(double) * g.rows_per_block * 2 * g.G * g.cpt : 0;
  switch (g.cpt) {
#define AMGEIG_CASE(C)                                                                                        \
  case C:                                                                                                     \
    k_defect<C, TO><<<blocks, kThreads, sm, st>>>(AM.rows, AM.rp, AM.ci, AM.v64, AM.m64, U, q, lam, R, ldr, \
                                                  g.G, partials);                                           \
    break;
    AMGEIG_CASE(1)
    AMGEIG_CASE(2)
    AMGEIG_CASE(4)
    AMGEIG_CASE(8)
#undef AMGEIG_CASE
    default:
      break;
  }
}

// ------------------------------------------------------------------ generic SpMM

template <typename T, int CPT>
__global__ void __launch_bounds__(kThreads) k_spmm(int n, const int* __restrict__ rp, const int* __restrict__ ci,
                                                   const T* __restrict__ v, const T* __restrict__ X, int width,
                                                   T* __restrict__ Y, int G, int accumulate) {
  const int rpb = blockDim.x / G;
  const int lane = threadIdx.x % G;
  const int row = blockIdx.x * rpb + threadIdx.x / G;
  if (row >= n) return;
  T acc[CPT];
#pragma unroll
  for (int t = 0; t < CPT; ++t) acc[t] = T(0);
  const int p0 = rp[row], p1 = rp[row + 1];
  for (int p = p0; p < p1; ++p) {
    const int j = ci[p];
    const T s = v[p];
    const T* xj = X + static_cast<long long>(j) * width;
#pragma unroll
    for (int t = 0; t < CPT; ++t) {
      const int c = lane + t * G;
      if (c < width) acc[t] = fma(s, xj[c], acc[t]);
    }
  }
  T* yr = Y + static_cast<long long>(row) * width;
#pragma unroll
  for (int t = 0; t < CPT; ++t) {
    const int c = lane + t * G;
    if (c < width) yr[c] = accumulate ? yr[c] + acc[t] : acc[t];
  }
}

template <typename T>
void spmm_impl(const DevCsr& S, const T* vals, const T* X, int width, T* Y, bool accumulate, cudaStream_t st,
               int cls = P_TRANSFER) {
  if (S.rows == 0 || width == 0) return;
  Geo g = geo_for(width);
  const int blocks = ceil_div(S.rows, g.rows_per_block);
  const double t = sizeof(T);
  ProfScope ps(st, cls,
               4.0 * (S.rows + 1) + (4.0 + t) * S.nnz + t * S.cols * width + t * S.rows * width * (accumulate ? 2 : 1),
               2.0 * S.nnz * width);
  switch (g.cpt) {
#define AMGEIG_CASE(C)                                                                                     \
  case C:                                                                                                  \
    k_spmm<T, C><<<blocks, kThreads, 0, st>>>(S.rows, S.rp, S.ci, vals, X, width, Y, g.G, accumulate ? 1 : 0); \
    break;
    AMGEIG_CASE(1)
    AMGEIG_CASE(2)
    AMGEIG_CASE(4)
    AMGEIG_CASE(8)
#undef AMGEIG_CASE
    default:
      break;
  }
}

// ------------------------------------------------------------------ smoothing

// mode 0: x = D^-1 b, r = b - A x          (presmooth from zero + residual)
// mode 1: out = x + D^-1 (b - A x)         (one sweep)
// mode 2: r = b - A x                      (residual)
// mode 3: V = U + x + D^-1 (b - A x)       (last sweep on the working level)
template <typename T, int CPT, int MODE>
__global__ void __launch_bounds__(kThreads) k_smooth(int n, const int* __restrict__ rp, const int* __restrict__ ci,
                                                     const T* __restrict__ a, const T* __restrict__ dinv,
                                                     const T* __restrict__ b, const T* __restrict__ x, int width,
                                                     T* __restrict__ out1, T* __restrict__ out2,
                                                     const double* __restrict__ U, double* __restrict__ V, int G) {
  const int rpb = blockDim.x / G;
  const int lane = threadIdx.x % G;
  const int row = blockIdx.x * rpb + threadIdx.x / G;
  if (row >= n) return;
  T acc[CPT];
#pragma unroll
  for (int t = 0; t < CPT; ++t) acc[t] = T(0);
  const int p0 = rp[row], p1 = rp[row + 1];
  for (int p = p0; p < p1; ++p) {
    const int j = ci[p];
    T s = a[p];
    if (MODE == 0) s *= dinv[j];
    const T* xj = (MODE == 0 ? b : x) + static_cast<long long>(j) * width;
#pragma unroll
    for (int t = 0; t < CPT; ++t) {
      const int c = lane + t * G;
      if (c < width) acc[t] = fma(s, xj[c], acc[t]);
    }
  }
  const long long base = static_cast<long long>(row) * width;
  const T di = dinv ? dinv[row] : T(0);
#pragma unroll
  for (int t = 0; t < CPT; ++t) {
    const int c = lane + t * G;
    if (c < width) {
      const T bi = b[base + c];
      const T res = bi - acc[t];
      if (MODE == 0) {
        out1[base + c] = di * bi;
        out2[base + c] = res;
      } else if (MODE == 1) {
        out1[base + c] = fma(di, res, x[base + c]);
      } else if (MODE == 2) {
        out1[base + c] = res;
      } else {
        const T xn = fma(di, res, x[base + c]);
        V[base + c] = U[base + c] + static_cast<double>(xn);
      }
    }
  }
}

template <typename T, int MODE>
void smooth_impl(const DevCsr& A, const T* vals, const T* dinv, const T* b, const T* x, int width, T* out1,
                 T* out2, const double* U, double* V, cudaStream_t st) {
  if (A.rows == 0 || width == 0) return;
  Geo g = geo_for(width);
  const int blocks = ceil_div(A.rows, g.rows_per_block);
  const double t = sizeof(T), N = A.rows;
  // vector traffic per mode: 0 reads b, writes x and r; 1 reads b, x, writes out;
  // 2 reads b, x, writes r; 3 reads b, x, U and writes V (float64)
  const double vec = (MODE == 3) ? (2.0 * t + 16.0) * N * width : 3.0 * t * N * width;
  ProfScope ps(st, P_SMOOTH, 4.0 * (N + 1) + (4.0 + t) * A.nnz + (MODE == 2 ? 0.0 : t * N) + vec,
               2.0 * A.nnz * width);
  switch (g.cpt) {
#define AMGEIG_CASE(C)                                                                                         \
  case C:                                                                                                      \
    k_smooth<T, C, MODE><<<blocks, kThreads, 0, st>>>(A.rows, A.rp, A.ci, vals, dinv, b, x, width, out1, out2, \
                                                      U, V, g.G);                                              \
    break;
    AMGEIG_CASE(1)
    AMGEIG_CASE(2)
    AMGEIG_CASE(4)
    AMGEIG_CASE(8)
#undef AMGEIG_CASE
    default:
      break;
  }
}

// ------------------------------------------------------------------ float32, 16-byte vectors
//
// The float32 V-cycle works on blocks whose row stride is a multiple of 4, so
// rows are moved as float4 (16 bytes).  A row group of G lanes owns a row; lane
// l handles the float4 columns l, l + G, ... (CPT of them, 1..3), so for the
// usual width of 24 floats two lanes take three columns each: per gathered
// row the pair reads 32 contiguous bytes per instruction, the index and value
// of each nonzero are loaded by two lanes instead of eight, and every lane
// keeps three independent 16-byte gathers in flight.

struct F4Geo {
  int G, cpt;
  int S = 1;  // nonzero streams per row: the row's G lanes form S groups of G / S column lanes, group k
              // takes the nonzeros p0 + k, p0 + k + S, ... and the groups' sums are added at the end
  // cpt = 0: one block of G = S * w4 threads per row (k_smooth_row), S streams of w4 lanes
};

// Streams of the block-per-row layout: blocks of 32 (one column lane) to 256 threads.
int row_streams(int w4) { return w4 <= 8 ? 32 : w4 <= 16 ? 16 : 8; }
// Whether a level's rows are long enough for it (see k_smooth_row)
bool row_layout(long long rows, long long nnz) { return nnz >= 96 * rows && rows < 65536; }

// Few lanes per row pay off only while the rows alone keep the GPU full: below
// about four resident waves of row groups the one-column-per-lane layout (more
// threads, shorter chains) is faster on the coarse levels.
F4Geo f4_geo(int w4, long long rows, long long nnz, bool sweep) {
  int G = 1;
  while (G * 3 < w4 && G < 32) G <<= 1;
  int cpt = (w4 + G - 1) / G;
  while (cpt > 3) {
    G <<= 1;
    cpt = (w4 + G - 1) / G;
  }
  if (sweep && w4 <= 32 && row_layout(rows, nnz)) return F4Geo{w4 * row_streams(w4), 0, row_streams(w4)};
  if (rows * G < 4LL * kNumSms * 1024) {
    G = 1;
    while (G < w4 && G < 32) G <<= 1;
    cpt = (w4 + G - 1) / G;
    // Small levels with long rows (the Galerkin coarse operators keep 25-35 nonzeros a
    // row): the chain of dependent gathers along a row, not bandwidth, sets the time, so
    // the row's nonzeros are split over S streams of lanes (a warp per row at most)
    if (nnz >= 12 * rows && rows < 65536 && G < 32) {
      const int S = std::min(4, 32 / G);
      return F4Geo{G * S, cpt, S};
    }
  }
  return F4Geo{G, cpt, 1};
}

// the operator's tuned shape at this width, else the rule (sweep: a smoothing sweep, which has the
// block-per-row layout)
F4Geo geo_of(const DevCsr& S, int w4, bool sweep) {
  if (w4 >= 1 && w4 <= 32 && S.tuned[w4]) {
    const int v = S.tuned[w4];
    // tuned: column lanes per stream (log2, bits 2-4), columns per lane (bits 0-1), streams (log2, bits 5-6);
    // bit 7: the block-per-row layout
    if (v & 128) return F4Geo{w4 * row_streams(w4), 0, row_streams(w4)};
    const int streams = 1 << ((v >> 5) & 3);
    return F4Geo{(1 << ((v >> 2) & 7)) * streams, v & 3, streams};
  }
  return f4_geo(w4, S.rows, S.nnz, sweep);
}

__device__ __forceinline__ void fma4(float s, const float4& x, float4& acc) {
  acc.x = fmaf(s, x.x, acc.x);
  acc.y = fmaf(s, x.y, acc.y);
  acc.z = fmaf(s, x.z, acc.z);
  acc.w = fmaf(s, x.w, acc.w);
}

// MODE 0: x = D^-1 b, r = b - A x (x from 0);  1: x <- x + D^-1 (b - A x);
// 2: r = b - A x;  3: V = U + (x + D^-1 (b - A x)) in float64;  4: the same in
// float-float, plus xadd when given (the sum of the earlier V-cycles).
__device__ __forceinline__ float to_f(float x) { return x; }
__device__ __forceinline__ float to_f(__nv_bfloat16 x) { return __bfloat162float(x); }

// the S streams' partial sums of a row added into stream 0's lanes (the row's
// G = S * (G / S) lanes are consecutive in a warp; every lane of the warp takes part)
template <int CPT>
__device__ __forceinline__ void reduce_streams(float4 (&acc)[CPT], int S, int gs) {
  for (int o = gs; o < gs * S; o <<= 1) {
#pragma unroll
    for (int t = 0; t < CPT; ++t) {
      acc[t].x += __shfl_down_sync(0xffffffffu, acc[t].x, o);
      acc[t].y += __shfl_down_sync(0xffffffffu, acc[t].y, o);
      acc[t].z += __shfl_down_sync(0xffffffffu, acc[t].z, o);
      acc[t].w += __shfl_down_sync(0xffffffffu, acc[t].w, o);
    }
  }
}

// The results of one float4 column c4 of one row from its sum acc = (A x)_row (MODE 0: (A D^-1 b)_row).
template <int MODE>
__device__ __forceinline__ void smooth_store(float4 acc, int row, int c4, int w4, float di,
                                             const float4* __restrict__ b, const float4* __restrict__ x,
                                             float4* __restrict__ out1, float4* __restrict__ out2,
                                             const double* __restrict__ U, double* __restrict__ V, int qv,
                                             const float2* __restrict__ U2, float2* __restrict__ V2,
                                             const float4* __restrict__ xadd) {
  const long long o = static_cast<long long>(row) * w4 + c4;
  const float4 bi = b[o];
  const float4 res = make_float4(bi.x - acc.x, bi.y - acc.y, bi.z - acc.z, bi.w - acc.w);
  if (MODE == 0) {
    out1[o] = make_float4(di * bi.x, di * bi.y, di * bi.z, di * bi.w);
    out2[o] = res;
  } else if (MODE == 2) {
    out1[o] = res;
  } else {
    const float4 xi = x[o];
    const float4 xn = make_float4(fmaf(di, res.x, xi.x), fmaf(di, res.y, xi.y), fmaf(di, res.z, xi.z),
                                  fmaf(di, res.w, xi.w));
    if (MODE == 1) {
      out1[o] = xn;
    } else if (MODE == 3) {
      const long long vb = static_cast<long long>(row) * qv + 4 * c4;
      const float xs[4] = {xn.x, xn.y, xn.z, xn.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (4 * c4 + k < qv) V[vb + k] = U[vb + k] + static_cast<double>(xs[k]);
    } else {
      // MODE 4: float-float V = U + x (+ xadd: the earlier V-cycles' sum)
      const long long vb = static_cast<long long>(row) * qv + 4 * c4;
      float4 xt = xn;
      if (xadd) {
        const float4 e = xadd[o];
        xt = make_float4(xn.x + e.x, xn.y + e.y, xn.z + e.z, xn.w + e.w);
      }
      const float xs[4] = {xt.x, xt.y, xt.z, xt.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (4 * c4 + k < qv) {
          const float2 u = U2[vb + k];
          const df r = df_add(df{u.x, u.y}, df{xs[k], 0.f});
          V2[vb + k] = make_float2(r.hi, r.lo);
        }
    }
  }
}

template <int MODE, int CPT, typename TV>
__global__ void __launch_bounds__(kThreads, 6) k_smooth_f4(int n, const int* __restrict__ rp,
                                                        const int* __restrict__ ci, const TV* __restrict__ a,
                                                        const float* __restrict__ dinv,
                                                        const float4* __restrict__ b, const float4* __restrict__ x,
                                                        int w4, float4* __restrict__ out1, float4* __restrict__ out2,
                                                        const double* __restrict__ U, double* __restrict__ V, int qv,
                                                        int G, const float2* __restrict__ U2 = nullptr,
                                                        float2* __restrict__ V2 = nullptr,
                                                        const float4* __restrict__ xadd = nullptr, int S = 1) {
  const int rpb = blockDim.x / G;
  const int gs = G / S;  // column lanes per stream
  const int lane = threadIdx.x % gs;
  const int sub = (threadIdx.x % G) / gs;
  const int row = blockIdx.x * rpb + threadIdx.x / G;
  if (S == 1 && row >= n) return;
  float4 acc[CPT];
#pragma unroll
  for (int t = 0; t < CPT; ++t) acc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
  const int p0 = row < n ? rp[row] : 0, p1 = row < n ? rp[row + 1] : 0;
  const float4* src = MODE == 0 ? b : x;
#pragma unroll 2
  for (int p = p0 + sub; p < p1; p += S) {
    const int j = ci[p];
    float s = to_f(a[p]);
    if (MODE == 0) s *= dinv[j];
    const float4* sr = src + static_cast<long long>(j) * w4;
#pragma unroll
    for (int t = 0; t < CPT; ++t) {
      const int c4 = lane + t * gs;
      if (c4 < w4) fma4(s, sr[c4], acc[t]);
    }
  }
  if (S > 1) {
    reduce_streams(acc, S, gs);
    if (sub != 0 || row >= n) return;
  }
  const float di = dinv ? dinv[row] : 0.f;
#pragma unroll
  for (int t = 0; t < CPT; ++t) {
    const int c4 = lane + t * gs;
    if (c4 < w4) smooth_store<MODE>(acc[t], row, c4, w4, di, b, x, out1, out2, U, V, qv, U2, V2, xadd);
  }
}

// The same sweep with one block per row, for the coarse levels whose rows are
// long: the Galerkin operators of 3D problems keep 200-600 nonzeros a row at a
// few thousand rows, where a warp per row leaves chains of 50-150 dependent
// gathers and most of the chip idle.  The block's threads are S streams of exactly w4
// column lanes (no idle lanes at widths that are not powers of two), stream k
// takes the nonzeros k, k + S, ..., four gathers in flight per thread, and the
// streams' sums meet in shared memory in a fixed tree.  Bound by the gathers'
// L2 latency and rate.  Cube of 250,047 unknowns, 20 columns (event times, a warp per
// row -> a block per row): 5494 rows of 361 nonzeros 53.5 -> 22.9 us, 2471 x 524 70.9 -> 18.5,
// 1142 x 598 64.1 -> 13.7, 521 x 469 39.9 -> under 12; 12,620 x 214 38.8 -> 33.4; rows
// below ~100 nonzeros gain nothing, which is where the rule's line lies (the tuner times both).
template <int MODE, typename TV>
__global__ void __launch_bounds__(256) k_smooth_row(int n, const int* __restrict__ rp, const int* __restrict__ ci,
                                                    const TV* __restrict__ a, const float* __restrict__ dinv,
                                                    const float4* __restrict__ b, const float4* __restrict__ x, int w4,
                                                    float4* __restrict__ out1, float4* __restrict__ out2,
                                                    const double* __restrict__ U, double* __restrict__ V, int qv,
                                                    int S, const float2* __restrict__ U2, float2* __restrict__ V2,
                                                    const float4* __restrict__ xadd) {
  __shared__ float4 part[256];
  const int row = blockIdx.x;
  const int sub = threadIdx.x / w4, lane = threadIdx.x - sub * w4;
  const int p1 = rp[row + 1];
  const float4* src = (MODE == 0 ? b : x) + lane;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  int p = rp[row] + sub;
  for (; p + 3 * S < p1; p += 4 * S) {
    int j[4];
    float s[4];
    float4 v[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      j[t] = ci[p + t * S];
      s[t] = to_f(a[p + t * S]);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      v[t] = src[static_cast<long long>(j[t]) * w4];
      if (MODE == 0) s[t] *= dinv[j[t]];
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) fma4(s[t], v[t], acc);
  }
  for (; p < p1; p += S) {
    const int j = ci[p];
    float s = to_f(a[p]);
    if (MODE == 0) s *= dinv[j];
    fma4(s, src[static_cast<long long>(j) * w4], acc);
  }
  part[threadIdx.x] = acc;
  __syncthreads();
  for (int o = S >> 1; o > 0; o >>= 1) {
    if (sub < o) {
      const float4 u = part[threadIdx.x + o * w4];
      acc = make_float4(acc.x + u.x, acc.y + u.y, acc.z + u.z, acc.w + u.w);
      part[threadIdx.x] = acc;
    }
    __syncthreads();
  }
  if (sub == 0)
    smooth_store<MODE>(acc, row, lane, w4, dinv ? dinv[row] : 0.f, b, x, out1, out2, U, V, qv, U2, V2, xadd);
}

template <int CPT, typename TV>
__global__ void __launch_bounds__(kThreads, 6) k_spmm_f4(int n, const int* __restrict__ rp, const int* __restrict__ ci,
                                                      const TV* __restrict__ v, const float4* __restrict__ X,
                                                      int w4, float4* __restrict__ Y, int G, int accumulate,
                                                      int S = 1) {
  const int rpb = blockDim.x / G;
  const int gs = G / S;
  const int lane = threadIdx.x % gs;
  const int sub = (threadIdx.x % G) / gs;
  const int row = blockIdx.x * rpb + threadIdx.x / G;
  if (S == 1 && row >= n) return;
  float4 acc[CPT];
#pragma unroll
  for (int t = 0; t < CPT; ++t) acc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
  const int p0 = row < n ? rp[row] : 0, p1 = row < n ? rp[row + 1] : 0;
#pragma unroll 2
  for (int p = p0 + sub; p < p1; p += S) {
    const float s = to_f(v[p]);
    const float4* xr = X + static_cast<long long>(ci[p]) * w4;
#pragma unroll
    for (int t = 0; t < CPT; ++t) {
      const int c4 = lane + t * gs;
      if (c4 < w4) fma4(s, xr[c4], acc[t]);
    }
  }
  if (S > 1) {
    reduce_streams(acc, S, gs);
    if (sub != 0 || row >= n) return;
  }
#pragma unroll
  for (int t = 0; t < CPT; ++t) {
    const int c4 = lane + t * gs;
    if (c4 >= w4) continue;
    const long long o = static_cast<long long>(row) * w4 + c4;
    float4 r = acc[t];
    if (accumulate) {
      const float4 y = Y[o];
      r = make_float4(r.x + y.x, r.y + y.y, r.z + y.z, r.w + y.w);
    }
    Y[o] = r;
  }
}

template <int MODE>
void smooth_f4(const DevCsr& A, const float* dinv, const float* b, const float* x, int w4, float* out1, float* out2,
               const double* U, double* V, int qv, const float2* U2, float2* V2, const float* xadd,
               cudaStream_t st, bool bf16 = false, const F4Geo* force = nullptr) {
  const F4Geo g = force ? *force : geo_of(A, w4, true);
  if (g.cpt == 0) {
#define AMGEIG_SMOOTH_ROW(TV, VALS)                                                                              \
  k_smooth_row<MODE, TV><<<A.rows, g.G, 0, st>>>(                                                                \
      A.rows, A.rp, A.ci, VALS, dinv, reinterpret_cast<const float4*>(b), reinterpret_cast<const float4*>(x), w4, \
      reinterpret_cast<float4*>(out1), reinterpret_cast<float4*>(out2), U, V, qv, g.S, U2, V2,                   \
      reinterpret_cast<const float4*>(xadd))
    if (bf16)
      AMGEIG_SMOOTH_ROW(__nv_bfloat16, A.vbf);
    else
      AMGEIG_SMOOTH_ROW(float, A.v32);
#undef AMGEIG_SMOOTH_ROW
    return;
  }
  const int blocks = ceil_div(A.rows, kThreads / g.G);
#define AMGEIG_SMOOTH_T(C, TV, VALS)                                                                         \
  k_smooth_f4<MODE, C, TV><<<blocks, kThreads, 0, st>>>(                                                       \
      A.rows, A.rp, A.ci, VALS, dinv, reinterpret_cast<const float4*>(b), reinterpret_cast<const float4*>(x), w4, \
      reinterpret_cast<float4*>(out1), reinterpret_cast<float4*>(out2), U, V, qv, g.G, U2, V2,                   \
      reinterpret_cast<const float4*>(xadd), g.S)
#define AMGEIG_SMOOTH(C)                                  \
  if (bf16)                                               \
    AMGEIG_SMOOTH_T(C, __nv_bfloat16, A.vbf);             \
  else                                                    \
    AMGEIG_SMOOTH_T(C, float, A.v32)
  switch (g.cpt) {
    case 1:
      AMGEIG_SMOOTH(1);
      break;
    case 2:
      AMGEIG_SMOOTH(2);
      break;
    default:
      AMGEIG_SMOOTH(3);
      break;
  }
#undef AMGEIG_SMOOTH
#undef AMGEIG_SMOOTH_T
}

// ------------------------------------------------------------------ augmentation

template <int CPT>
__global__ void __launch_bounds__(kThreads) k_dual_spmm(int n, const int* __restrict__ rp, const int* __restrict__ ci,
                                                        const double* __restrict__ a, const double* __restrict__ m,
                                                        const double* __restrict__ V, int q, double* __restrict__ W,
                                                        int G) {
  const int rpb = blockDim.x / G;
  const int lane = threadIdx.x % G;
  const int row = blockIdx.x * rpb + threadIdx.x / G;
  if (row >= n) return;
  double aa[CPT], mm[CPT];
#pragma unroll
  for (int t = 0; t < CPT; ++t) aa[t] = mm[t] = 0.0;
  const int p0 = rp[row], p1 = rp[row + 1];
  for (int p = p0; p < p1; ++p) {
    const int j = ci[p];
    const double av = a[p], mv = m[p];
    const double* vj = V + static_cast<long long>(j) * q;
#pragma unroll
    for (int t = 0; t < CPT; ++t) {
      const int c = lane + t * G;
      if (c < q) {
        const double u = vj[c];
        aa[t] = fma(av, u, aa[t]);
        mm[t] = fma(mv, u, mm[t]);
      }
    }
  }
  double* wr = W + static_cast<long long>(row) * 2 * q;
#pragma unroll
  for (int t = 0; t < CPT; ++t) {
    const int c = lane + t * G;
    if (c < q) {
      wr[c] = aa[t];
      wr[q + c] = mm[t];
    }
  }
}

// ------------------------------------------------------------------ recombination

template <int CPT>
__global__ void __launch_bounds__(kThreads) k_recombine(int n, const double* __restrict__ Xp,
                                                        const double* __restrict__ V, const double* __restrict__ Y,
                                                        int q, double* __restrict__ U, int G) {
  extern __shared__ double ys[];  // q x q
  for (int i = threadIdx.x; i < q * q; i += blockDim.x) ys[i] = Y[i];
  __syncthreads();
  const int rpb = blockDim.x / G;
  const int lane = threadIdx.x % G;
  const int row = blockIdx.x * rpb + threadIdx.x / G;
  if (row >= n) return;
  const long long base = static_cast<long long>(row) * q;
  double acc[CPT];
#pragma unroll
  for (int t = 0; t < CPT; ++t) {
    const int c = lane + t * G;
    acc[t] = (c < q) ? Xp[base + c] : 0.0;
  }
  for (int d = 0; d < q; ++d) {
    const double v = V[base + d];
#pragma unroll
    for (int t = 0; t < CPT; ++t) {
      const int c = lane + t * G;
      if (c < q) acc[t] = fma(v, ys[d * q + c], acc[t]);
    }
  }
#pragma unroll
  for (int t = 0; t < CPT; ++t) {
    const int c = lane + t * G;
    if (c < q) U[base + c] = acc[t];
  }
}

// float-float variant: the block's V rows and Y are staged as float-float
// pairs in shared memory (each converted once), products accumulate with
// compensated float32 arithmetic
template <int CPT>
__global__ void __launch_bounds__(kThreads) k_recombine_df(int n, const double* __restrict__ Xp,
                                                           const double* __restrict__ V,
                                                           const double* __restrict__ Y, int q,
                                                           double* __restrict__ U, int G) {
  extern __shared__ df dsm[];  // Y (q x q) then V rows (rpb x q)
  df* ys = dsm;
  df* vs = dsm + q * q;
  const int rpb = blockDim.x / G;
  for (int i = threadIdx.x; i < q * q; i += blockDim.x) ys[i] = df_from_double(Y[i]);
  const long long row0 = static_cast<long long>(blockIdx.x) * rpb;
  for (int i = threadIdx.x; i < rpb * q; i += blockDim.x) {
    const long long r = row0 + i / q;
    vs[i] = (r < n) ? df_from_double(V[r * q + i % q]) : df{0.f, 0.f};
  }
  __syncthreads();
  const int g = threadIdx.x / G;
  const int lane = threadIdx.x % G;
  const long long row = row0 + g;
  if (row >= n) return;
  const long long base = row * q;
  df_acc acc[CPT];
#pragma unroll
  for (int t = 0; t < CPT; ++t) {
    const int c = lane + t * G;
    acc[t] = acc_zero();
    if (c < q) acc[t].add(df_from_double(Xp[base + c]));
  }
  const df* vr = vs + g * q;
  for (int d = 0; d < q; ++d) {
    const df v = vr[d];
#pragma unroll
    for (int t = 0; t < CPT; ++t) {
      const int c = lane + t * G;
      if (c < q) acc[t].fma(v, ys[d * q + c]);
    }
  }
#pragma unroll
  for (int t = 0; t < CPT; ++t) {
    const int c = lane + t * G;
    if (c < q) U[base + c] = df_to_double(acc[t].value());
  }
}

// ------------------------------------------------------------------ elementwise

template <typename T>
__global__ void k_add_to_v(const double* __restrict__ U, const T* __restrict__ x, long long count,
                           double* __restrict__ V) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < count;
       i += static_cast<long long>(gridDim.x) * blockDim.x)
    V[i] = U[i] + static_cast<double>(x[i]);
}

template <typename T>
__global__ void k_axpy(const T* __restrict__ x, long long count, T* __restrict__ y) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < count;
       i += static_cast<long long>(gridDim.x) * blockDim.x)
    y[i] += x[i];
}

__global__ void k_f64_to_f32(const double* __restrict__ x, long long count, float* __restrict__ y) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < count;
       i += static_cast<long long>(gridDim.x) * blockDim.x)
    y[i] = static_cast<float>(x[i]);
}

// l1-Jacobi inverse diagonal of one level: d_i = 1 / sum_j |a_ij| (the row summed in
// order, float64), also rounded to float32; *zero_row = 1 when a row sum is not positive
__global__ void k_l1_inv_diag(int rows, const int* __restrict__ rp, const double* __restrict__ a,
                              double* __restrict__ d64, float* __restrict__ d32, int* __restrict__ zero_row) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows; i += gridDim.x * blockDim.x) {
    double sa = 0.0;
    for (int p = rp[i]; p < rp[i + 1]; ++p) sa += fabs(a[p]);
    if (!(sa > 0.0)) *zero_row = 1;
    const double d = 1.0 / sa;
    d64[i] = d;
    d32[i] = static_cast<float>(d);
  }
}

__global__ void k_f32_to_f64(const float* __restrict__ x, long long count, double* __restrict__ y) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < count;
       i += static_cast<long long>(gridDim.x) * blockDim.x)
    y[i] = static_cast<double>(x[i]);
}

__global__ void k_add_to_v_strided(const double* __restrict__ U, const float* __restrict__ x, int rows, int q, int ldx,
                                   double* __restrict__ V) {
  const long long total = static_cast<long long>(rows) * q;
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<long long>(gridDim.x) * blockDim.x)
    V[i] = U[i] + static_cast<double>(x[(i / q) * ldx + i % q]);
}

__global__ void k_pad_f64_to_f32(const double* __restrict__ src, int rows, int q, int ld, float* __restrict__ dst) {
  const long long total = static_cast<long long>(rows) * ld;
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long r = i / ld;
    const int c = static_cast<int>(i % ld);
    dst[i] = c < q ? static_cast<float>(src[r * q + c]) : 0.f;
  }
}

__global__ void k_unpad_f32_to_f64(const float* __restrict__ src, int rows, int q, int ld, double* __restrict__ dst) {
  const long long total = static_cast<long long>(rows) * q;
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<long long>(gridDim.x) * blockDim.x)
    dst[i] = static_cast<double>(src[(i / q) * ld + i % q]);
}

int grid_for(long long count) {
  long long b = (count + kThreads - 1) / kThreads;
  if (b > 8LL * kNumSms) b = 8LL * kNumSms;
  return static_cast<int>(b < 1 ? 1 : b);
}

// ---------------------------------------------------------------- Gauss-Seidel
// One colour of a multicolour Gauss-Seidel sweep.  Rows of one colour share no
// nonzero, so they update together from the current x of the other colours:
// x_i <- x_i + (b_i - sum_j a_ij x_j) / a_ii (the j = i term included in the sum).
template <typename T>
__global__ void __launch_bounds__(kThreads) k_gs_colour(int cnt, const int* __restrict__ rows,
                                                        const int* __restrict__ rp, const int* __restrict__ ci,
                                                        const T* __restrict__ a, const T* __restrict__ dinv,
                                                        const T* __restrict__ b, T* x, int ld, int w) {
  const long long total = static_cast<long long>(cnt) * w;
  for (long long it = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; it < total;
       it += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int i = rows[it / w], c = static_cast<int>(it % w);
    const long long o = static_cast<long long>(i) * ld + c;
    T s = b[o];
    const int p1 = rp[i + 1];
    for (int p = rp[i]; p < p1; ++p) s -= a[p] * x[static_cast<long long>(ci[p]) * ld + c];
    x[o] += s * dinv[i];
  }
}

// ---------------------------------------------------------------- composite prolongation
// One level of I_n^k = P_k I_n^{k+1} (a sparse product with d_n columns), one warp
// per row: the row's entries accumulate into a dense d_n-wide float64 row in
// shared memory (flags mark the structural nonzeros), then come out in column
// order.  With out_rp null the pass only counts each row's nonzeros.  Each column
// receives its terms in the order of the row of P_k, as a row-by-row host product
// would add them.
__global__ void __launch_bounds__(kThreads) k_pc_rows(int rows, const int* __restrict__ prp,
                                                      const int* __restrict__ pci, const double* __restrict__ pv,
                                                      const int* __restrict__ nrp, const int* __restrict__ nci,
                                                      const double* __restrict__ nv, int dn,
                                                      const int* __restrict__ out_rp, int* __restrict__ counts,
                                                      int* __restrict__ out_ci, double* __restrict__ out_v) {
  extern __shared__ __align__(16) unsigned char pcs[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  double* acc = reinterpret_cast<double*>(pcs) + static_cast<size_t>(warp) * dn;
  unsigned char* flag = pcs + static_cast<size_t>(wpb) * dn * sizeof(double) + static_cast<size_t>(warp) * dn;
  for (int c = lane; c < dn; c += 32) {
    flag[c] = 0;
    acc[c] = 0.0;
  }
  __syncwarp();
  for (int row = blockIdx.x * wpb + warp; row < rows; row += gridDim.x * wpb) {
    const int p1 = prp[row + 1];
    for (int p = prp[row]; p < p1; ++p) {
      const int t = pci[p];
      const double v = pv[p];
      for (int r = nrp[t] + lane; r < nrp[t + 1]; r += 32) {
        const int c = nci[r];  // distinct within one row of I_n^{k+1}
        flag[c] = 1;
        acc[c] += v * nv[r];
      }
      __syncwarp();
    }
    int base = out_rp ? out_rp[row] : 0;
    for (int c0 = 0; c0 < dn; c0 += 32) {
      const int c = c0 + lane;
      const bool on = c < dn && flag[c];
      const unsigned m = __ballot_sync(0xffffffffu, on);
      if (on && out_rp) {
        const int pos = base + __popc(m & ((1u << lane) - 1u));
        out_ci[pos] = c;
        out_v[pos] = acc[c];
      }
      base += __popc(m);
      if (c < dn) {
        flag[c] = 0;
        acc[c] = 0.0;
      }
    }
    if (!out_rp && lane == 0) counts[row] = base;
    __syncwarp();
  }
}

}  // namespace

void launch_defect_f64(const DevCsr& AM, const double* U, int q, const double* lam, double* R, double* partials,
                       int* nblocks_out, cudaStream_t st) {
  defect_impl<double>(AM, U, q, lam, R, q, partials, nblocks_out, st);
}
void launch_defect_f32out(const DevCsr& AM, const double* U, int q, const double* lam, float* R, int ldr,
                          double* partials, int* nblocks_out, cudaStream_t st) {
  defect_impl<float>(AM, U, q, lam, R, ldr, partials, nblocks_out, st);
}

void launch_spmm_f64(const DevCsr& S, const double* X, int width, double* Y, bool accumulate, cudaStream_t st,
                     int cls) {
  spmm_impl<double>(S, S.v64, X, width, Y, accumulate, st, cls);
}
static void spmm_f4_geo(const DevCsr& S, const float* X, int w4, float* Y, bool accumulate, cudaStream_t st,
                        bool bf16, F4Geo g);

void launch_spmm_f32(const DevCsr& S, const float* X, int width, float* Y, bool accumulate, cudaStream_t st,
                     bool bf16) {
  if (width % 4 != 0 || S.rows == 0) {
    spmm_impl<float>(S, S.v32, X, width, Y, accumulate, st);
    return;
  }
  const int w4 = width / 4;
  const F4Geo g = geo_of(S, w4, false);
  spmm_f4_geo(S, X, w4, Y, accumulate, st, bf16, g);
}

static void spmm_f4_geo(const DevCsr& S, const float* X, int w4, float* Y, bool accumulate, cudaStream_t st,
                        bool bf16, F4Geo g) {
  const int width = 4 * w4;
  const int blocks = ceil_div(S.rows, kThreads / g.G);
  ProfScope ps(st, P_TRANSFER,
               4.0 * (S.rows + 1) + 8.0 * S.nnz + 4.0 * S.cols * width + 4.0 * S.rows * width * (accumulate ? 2 : 1),
               2.0 * S.nnz * width);
  const float4* X4 = reinterpret_cast<const float4*>(X);
  float4* Y4 = reinterpret_cast<float4*>(Y);
  const int acc = accumulate ? 1 : 0;
#define AMGEIG_SPMM(C)                                                                                       \
  if (bf16)                                                                                                  \
    k_spmm_f4<C, __nv_bfloat16><<<blocks, kThreads, 0, st>>>(S.rows, S.rp, S.ci, S.vbf, X4, w4, Y4, g.G, acc, \
                                                             g.S);                                            \
  else                                                                                                       \
    k_spmm_f4<C, float><<<blocks, kThreads, 0, st>>>(S.rows, S.rp, S.ci, S.v32, X4, w4, Y4, g.G, acc, g.S)
  switch (g.cpt) {
    case 1:
      AMGEIG_SPMM(1);
      break;
    case 2:
      AMGEIG_SPMM(2);
      break;
    default:
      AMGEIG_SPMM(3);
      break;
  }
#undef AMGEIG_SPMM
}

void launch_presmooth_residual_f64(const DevCsr& A, const double* dinv, const double* b, int width, double* x,
                                   double* r, cudaStream_t st) {
  smooth_impl<double, 0>(A, A.v64, dinv, b, nullptr, width, x, r, nullptr, nullptr, st);
}
void launch_presmooth_residual_f32(const DevCsr& A, const float* dinv, const float* b, int width, float* x,
                                   float* r, cudaStream_t st, bool bf16) {
  if (width % 4 == 0 && A.rows > 0) {
    const double N = A.rows;
    const double vec = 12.0 * N * width;
    ProfScope ps(st, P_SMOOTH, 4.0 * (N + 1) + 8.0 * A.nnz + 4.0 * N + vec, 2.0 * A.nnz * width);
    smooth_f4<0>(A, dinv, b, nullptr, width / 4, x, r, nullptr, nullptr, 0, nullptr, nullptr, nullptr, st, bf16);
    return;
  }
  smooth_impl<float, 0>(A, A.v32, dinv, b, nullptr, width, x, r, nullptr, nullptr, st);
}
void launch_jacobi_f64(const DevCsr& A, const double* dinv, const double* b, const double* x, int width,
                       double* x_out, cudaStream_t st) {
  smooth_impl<double, 1>(A, A.v64, dinv, b, x, width, x_out, nullptr, nullptr, nullptr, st);
}
void launch_jacobi_f32(const DevCsr& A, const float* dinv, const float* b, const float* x, int width,
                       float* x_out, cudaStream_t st, bool bf16) {
  if (width % 4 == 0 && A.rows > 0) {
    const double N = A.rows;
    const double vec = 12.0 * N * width;
    ProfScope ps(st, P_SMOOTH, 4.0 * (N + 1) + 8.0 * A.nnz + 4.0 * N + vec, 2.0 * A.nnz * width);
    smooth_f4<1>(A, dinv, b, x, width / 4, x_out, nullptr, nullptr, nullptr, 0, nullptr, nullptr, nullptr, st, bf16);
    return;
  }
  smooth_impl<float, 1>(A, A.v32, dinv, b, x, width, x_out, nullptr, nullptr, nullptr, st);
}
void launch_residual_f64(const DevCsr& A, const double* b, const double* x, int width, double* r, cudaStream_t st) {
  smooth_impl<double, 2>(A, A.v64, nullptr, b, x, width, r, nullptr, nullptr, nullptr, st);
}
void launch_residual_f32(const DevCsr& A, const float* b, const float* x, int width, float* r, cudaStream_t st,
                         bool bf16) {
  if (width % 4 == 0 && A.rows > 0) {
    const double N = A.rows;
    const double vec = 12.0 * N * width;
    ProfScope ps(st, P_SMOOTH, 4.0 * (N + 1) + 8.0 * A.nnz + 0.0 + vec, 2.0 * A.nnz * width);
    smooth_f4<2>(A, nullptr, b, x, width / 4, r, nullptr, nullptr, nullptr, 0, nullptr, nullptr, nullptr, st, bf16);
    return;
  }
  smooth_impl<float, 2>(A, A.v32, nullptr, b, x, width, r, nullptr, nullptr, nullptr, st);
}
void launch_jacobi_to_v_f64(const DevCsr& A, const double* dinv, const double* b, const double* x, int width,
                            const double* U, double* V, cudaStream_t st) {
  smooth_impl<double, 3>(A, A.v64, dinv, b, x, width, nullptr, nullptr, U, V, st);
}
void launch_jacobi_to_v_f32(const DevCsr& A, const float* dinv, const float* b, const float* x, int width,
                            const double* U, double* V, cudaStream_t st, int qv) {
  if (width % 4 == 0 && A.rows > 0) {
    const double N = A.rows;
    const double vec = (2.0 * 4 + 16.0) * N * width;
    ProfScope ps(st, P_SMOOTH, 4.0 * (N + 1) + 8.0 * A.nnz + 4.0 * N + vec, 2.0 * A.nnz * width);
    smooth_f4<3>(A, dinv, b, x, width / 4, nullptr, nullptr, U, V, qv, nullptr, nullptr, nullptr, st);
    return;
  }
  smooth_impl<float, 3>(A, A.v32, dinv, b, x, width, nullptr, nullptr, U, V, st);
  (void)qv;
}
void launch_add_to_v_f64(const double* U, const double* x, long long count, double* V, cudaStream_t st) {
  ProfScope ps(st, P_SMOOTH, 24.0 * count, 1.0 * count);
  k_add_to_v<double><<<grid_for(count), kThreads, 0, st>>>(U, x, count, V);
}
void launch_add_to_v_f32(const double* U, const float* x, long long count, double* V, cudaStream_t st) {
  ProfScope ps(st, P_SMOOTH, 20.0 * count, 1.0 * count);
  k_add_to_v<float><<<grid_for(count), kThreads, 0, st>>>(U, x, count, V);
}

void launch_dual_spmm(const DevCsr& AM, const double* V, int q, double* W, cudaStream_t st) {
  Geo g = geo_for(q);
  const int blocks = ceil_div(AM.rows, g.rows_per_block);
  const double N = AM.rows, nnz = AM.nnz;
  ProfScope ps(st, P_AUGMENT, 4.0 * (N + 1) + 20.0 * nnz + 8.0 * N * q + 16.0 * N * q, 4.0 * nnz * q);
  switch (g.cpt) {
#define AMGEIG_CASE(C)                                                                                         \
  case C:                                                                                                      \
    k_dual_spmm<C><<<blocks, kThreads, 0, st>>>(AM.rows, AM.rp, AM.ci, AM.v64, AM.m64, V, q, W, g.G); \
    break;
    AMGEIG_CASE(1)
    AMGEIG_CASE(2)
    AMGEIG_CASE(4)
    AMGEIG_CASE(8)
#undef AMGEIG_CASE
    default:
      break;
  }
}

void launch_recombine(int rows, const double* Xp, const double* V, const double* Y, int q, double* U,
                      cudaStream_t st, bool df_arith) {
  Geo g = geo_for(q);
  const int blocks = ceil_div(rows, g.rows_per_block);
  ProfScope ps(st, P_RECOMBINE, 24.0 * rows * q + 8.0 * q * q, 2.0 * rows * q * q);
  if (df_arith) {
    const size_t sm = sizeof(df) * (static_cast<size_t>(q) * q + static_cast<size_t>(g.rows_per_block) * q);
    switch (g.cpt) {
#define AMGEIG_CASE(C)                                                                            \
  case C:                                                                                         \
    if (sm > 48 * 1024)                                                                           \
      ensure_dynamic_smem(reinterpret_cast<const void*>(k_recombine_df<C>), sm);                    \
    k_recombine_df<C><<<blocks, kThreads, sm, st>>>(rows, Xp, V, Y, q, U, g.G);                     \
    break;
      AMGEIG_CASE(1)
      AMGEIG_CASE(2)
      AMGEIG_CASE(4)
      AMGEIG_CASE(8)
#undef AMGEIG_CASE
      default:
        break;
    }
    return;
  }
  const size_t sm = sizeof(double) * q * q;
  switch (g.cpt) {
#define AMGEIG_CASE(C)                                                                         \
  case C:                                                                                      \
    if (sm > 48 * 1024)                                                                        \
      ensure_dynamic_smem(reinterpret_cast<const void*>(k_recombine<C>), sm);                    \
    k_recombine<C><<<blocks, kThreads, sm, st>>>(rows, Xp, V, Y, q, U, g.G);                     \
    break;
    AMGEIG_CASE(1)
    AMGEIG_CASE(2)
    AMGEIG_CASE(4)
    AMGEIG_CASE(8)
#undef AMGEIG_CASE
    default:
      break;
  }
}

void launch_axpy_f64(const double* x, long long count, double* y, cudaStream_t st) {
  ProfScope ps(st, P_SMOOTH, 24.0 * count, 1.0 * count);
  k_axpy<double><<<grid_for(count), kThreads, 0, st>>>(x, count, y);
}
void launch_axpy_f32(const float* x, long long count, float* y, cudaStream_t st) {
  ProfScope ps(st, P_SMOOTH, 12.0 * count, 1.0 * count);
  k_axpy<float><<<grid_for(count), kThreads, 0, st>>>(x, count, y);
}

void launch_convert_f64_to_f32(const double* x, long long count, float* y, cudaStream_t st) {
  ProfScope ps(st, P_OTHER, 12.0 * count, 0.0);
  k_f64_to_f32<<<grid_for(count), kThreads, 0, st>>>(x, count, y);
}

void launch_l1_inv_diag(const DevCsr& A, double* d64, float* d32, int* zero_row, cudaStream_t st) {
  ProfScope ps(st, P_OTHER, 4.0 * (A.rows + 1) + 8.0 * A.nnz + 12.0 * A.rows, 0.0);
  k_l1_inv_diag<<<grid_for(A.rows), kThreads, 0, st>>>(A.rows, A.rp, A.v64, d64, d32, zero_row);
}

void launch_convert_f32_to_f64(const float* x, long long count, double* y, cudaStream_t st) {
  ProfScope ps(st, P_OTHER, 12.0 * count, 0.0);
  k_f32_to_f64<<<grid_for(count), kThreads, 0, st>>>(x, count, y);
}

void launch_add_to_v_f32_strided(const double* U, const float* x, int rows, int q, int ldx, double* V,
                                 cudaStream_t st) {
  const long long count = static_cast<long long>(rows) * q;
  ProfScope ps(st, P_SMOOTH, 20.0 * count, 1.0 * count);
  k_add_to_v_strided<<<grid_for(count), kThreads, 0, st>>>(U, x, rows, q, ldx, V);
}

void launch_f64_to_f32_pad(const double* src, int rows, int q, int ld, float* dst, cudaStream_t st) {
  const long long count = static_cast<long long>(rows) * ld;
  ProfScope ps(st, P_OTHER, 12.0 * count, 0.0);
  k_pad_f64_to_f32<<<grid_for(count), kThreads, 0, st>>>(src, rows, q, ld, dst);
}

void launch_f32_to_f64_unpad(const float* src, int rows, int q, int ld, double* dst, cudaStream_t st) {
  const long long count = static_cast<long long>(rows) * q;
  ProfScope ps(st, P_OTHER, 12.0 * count, 0.0);
  k_unpad_f32_to_f64<<<grid_for(count), kThreads, 0, st>>>(src, rows, q, ld, dst);
}

void launch_jacobi_to_vdf_f32(const DevCsr& A, const float* dinv, const float* b, const float* x, int width,
                              const float2* U, float2* V, cudaStream_t st, int qv, const float* xadd, bool bf16) {
  if (A.rows == 0) return;
  const double N = A.rows;
  ProfScope ps(st, P_SMOOTH,
               4.0 * (N + 1) + 8.0 * A.nnz + 4.0 * N + ((xadd ? 3.0 : 2.0) * 4 + 16.0) * N * width,
               2.0 * A.nnz * width);
  smooth_f4<4>(A, dinv, b, x, width / 4, nullptr, nullptr, nullptr, nullptr, qv, U, V, xadd, st, bf16);
}

__global__ void k_f32_to_bf16(const float* __restrict__ x, long long count, __nv_bfloat16* __restrict__ y) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < count;
       i += static_cast<long long>(gridDim.x) * blockDim.x)
    y[i] = __float2bfloat16_rn(x[i]);
}

void launch_f32_to_bf16(const float* x, long long count, __nv_bfloat16* y, cudaStream_t st) {
  if (count <= 0) return;
  ProfScope ps(st, P_OTHER, 6.0 * count, 0.0);
  k_f32_to_bf16<<<grid_for(count), kThreads, 0, st>>>(x, count, y);
}

__global__ void k_add_to_vdf(const float2* __restrict__ U, const float* __restrict__ x, int rows, int q, int ldx,
                             float2* __restrict__ V) {
  const long long total = static_cast<long long>(rows) * q;
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    const float2 u = U[i];
    const df r = df_add(df{u.x, u.y}, df{x[(i / q) * ldx + i % q], 0.f});
    V[i] = make_float2(r.hi, r.lo);
  }
}

void launch_add_to_vdf(const float2* U, const float* x, int rows, int q, int ldx, float2* V, cudaStream_t st) {
  const long long count = static_cast<long long>(rows) * q;
  ProfScope ps(st, P_SMOOTH, 20.0 * count, 1.0 * count);
  k_add_to_vdf<<<grid_for(count), kThreads, 0, st>>>(U, x, rows, q, ldx, V);
}

void launch_gs_colour(int cnt, const int* rows, const DevCsr& A, const double* dinv, const double* b, double* x,
                      int ld, int w, double bytes, cudaStream_t st) {
  if (cnt <= 0) return;
  ProfScope ps(st, P_SMOOTH, bytes, 2.0 * w * cnt * (static_cast<double>(A.nnz) / A.rows));
  k_gs_colour<double><<<grid_for(static_cast<long long>(cnt) * w), kThreads, 0, st>>>(cnt, rows, A.rp, A.ci, A.v64,
                                                                                      dinv, b, x, ld, w);
}
void launch_gs_colour(int cnt, const int* rows, const DevCsr& A, const float* dinv, const float* b, float* x, int ld,
                      int w, double bytes, cudaStream_t st) {
  if (cnt <= 0) return;
  ProfScope ps(st, P_SMOOTH, bytes, 2.0 * w * cnt * (static_cast<double>(A.nnz) / A.rows));
  k_gs_colour<float><<<grid_for(static_cast<long long>(cnt) * w), kThreads, 0, st>>>(cnt, rows, A.rp, A.ci, A.v32,
                                                                                     dinv, b, x, ld, w);
}

void launch_composite_rows(const DevCsr& P, const int* nrp, const int* nci, const double* nv, int dn,
                           const int* out_rp, int* counts, int* out_ci, double* out_v, cudaStream_t st) {
  if (P.rows <= 0) return;
  // warps per block: the dense rows (9 bytes per column) within 96 KB of shared memory
  const int wpb = std::max(1, std::min(8, static_cast<int>((96 * 1024) / (9 * static_cast<size_t>(dn)))));
  const size_t sm = static_cast<size_t>(wpb) * dn * 9;
  ensure_dynamic_smem(reinterpret_cast<const void*>(k_pc_rows), sm);
  int blocks = ceil_div(P.rows, wpb);
  if (blocks > 8 * kNumSms) blocks = 8 * kNumSms;
  ProfScope ps(st, P_OTHER, 4.0 * P.rows + 12.0 * P.nnz, 0.0);
  k_pc_rows<<<blocks, 32 * wpb, sm, st>>>(P.rows, P.rp, P.ci, P.v64, nrp, nci, nv, dn, out_rp, counts, out_ci, out_v);
}

TuneResult autotune_f4(DevCsr& S, int kind, int w4, const float* dinv, const float* x, const float* b, float* out,
                       cudaStream_t st) {
  TuneResult r;
  const F4Geo rule = f4_geo(w4, S.rows, S.nnz, kind == 0);
  r.rule_G = rule.G;
  r.rule_cpt = rule.cpt;
  r.S = rule.S;
  if (w4 < 1 || w4 > 32 || S.rows == 0) return r;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    return r;
  }
  auto run = [&](F4Geo g) {
    if (kind == 0)
      smooth_f4<1>(S, dinv, b, x, w4, out, nullptr, nullptr, nullptr, 0, nullptr, nullptr, nullptr, st, false, &g);
    else
      spmm_f4_geo(S, x, w4, out, false, st, false, g);
  };
  auto time_us = [&](F4Geo g) -> float {
    ProfScope ps(st, P_OTHER, 0.0, 0.0, 4);
    run(g);  // warm-up
    float best = 1e30f;
    for (int rep = 0; rep < 3; ++rep) {
      cudaEventRecord(e0, st);
      run(g);
      cudaEventRecord(e1, st);
      float ms = 1e30f;
      if (cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess)
        best = best < ms ? best : ms;
    }
    return best * 1000.f;
  };
  // every power-of-two column-lane count whose share per lane is 1..3 float4s, times 1, 2
  // or 4 nonzero streams per row (at most a warp per row).  The streams change the order
  // in which a row's terms are added, so a tuned shape can round differently from the
  // rule's (a float32 rounding difference); a given shape always gives the same bits.
  float best = 1e30f;
  for (int streams = 1; streams <= 4; streams <<= 1)
    for (int gc = 1; gc * streams <= 32; gc <<= 1) {
      const int cpt = (w4 + gc - 1) / gc;
      if (cpt > 3 || (gc > 1 && gc / 2 >= w4)) continue;
      const float us = time_us(F4Geo{gc * streams, cpt, streams});
      if (us < best) {
        best = us;
        r.G = gc * streams;
        r.cpt = cpt;
        r.S = streams;
      }
    }
  // and, for the smoothing sweeps, the block-per-row layout where a row has a nonzero for every stream
  bool by_row = false;
  if (kind == 0 && S.nnz >= static_cast<long long>(row_streams(w4)) * S.rows) {
    const F4Geo g{w4 * row_streams(w4), 0, row_streams(w4)};
    const float us = time_us(g);
    if (us < best) {
      best = us;
      r.G = g.G;
      r.cpt = g.cpt;
      r.S = g.S;
      by_row = true;
    }
  }
  r.us = best;
  r.rule_us = time_us(rule);
  const bool launched = cudaGetLastError() == cudaSuccess;  // asked once: a refused trial leaves the rule
  if (launched && by_row) {
    S.tuned[w4] = 128;
  } else if (launched && r.G > 0) {
    int lg = 0, ls = 0;
    while ((1 << lg) < r.G / r.S) ++lg;
    while ((1 << ls) < r.S) ++ls;
    S.tuned[w4] = static_cast<unsigned char>((ls << 5) | (lg << 2) | r.cpt);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return r;
}

namespace {
__global__ void k_axpby_f64(const double* __restrict__ x, double alpha, const double* __restrict__ y, long long n,
                            double* __restrict__ z) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<long long>(gridDim.x) * blockDim.x)
    z[i] = fma(alpha, y[i], x[i]);
}
}  // namespace

void launch_axpby_f64(const double* x, double alpha, const double* y, long long count, double* z, cudaStream_t st) {
  ProfScope ps(st, P_OTHER, 24.0 * count, 2.0 * count);
  k_axpby_f64<<<grid_for(count), kThreads, 0, st>>>(x, alpha, y, count, z);
}

}  // namespace amgeig
