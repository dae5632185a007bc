// The dense symmetric eigensolver behind amgeig_sym_eigh and amgeig_sym_eigh_noalloc.
//
// An eigenvector's sign is not determined by the problem: three inverse
// iterations leave the sign of (lambda - shift)^3, and the shift lies within rounding of
// lambda, so the sign follows the last bits of the tridiagonalisation and of the
// shift.  The interface promises no sign, but a vector that turns over between two versions of this
// library is a difference its callers see, so the arithmetic here is kept bit for bit; the
// solve path, whose results have a sign convention of their own, runs the faster form in
// pencil.cu (n = 328, 64 wanted: 4.5 ms here, 1.9 ms there).
//
// Float-float throughout (48-bit significand): Householder tridiagonalisation,
// bisection with Sturm counts for the wanted eigenvalues (float32), each shift refined by
// float-float Sturm multisection, inverse iteration (Gram-Schmidt inside clusters of
// nearly equal shifts), a Rayleigh-Ritz clean-up by parallel cyclic Jacobi on each
// group of close shifts, and back-transformation.  Golub & Van Loan, Matrix Computations,
// 4th ed., 8.3 (tridiagonalisation), 8.4.1 (Sturm bisection), 8.2.2 (inverse iteration),
// 8.5 (Jacobi).
#include <cooperative_groups.h>

#include <algorithm>
#include <map>
#include <mutex>

#include "prof.cuh"
#include "syev.cuh"

namespace amgeig {
namespace {

constexpr int kSyThreads = 1024;

__device__ __forceinline__ int sturm_count(const float* sd, const float* se2, int n, float x, float pivmin) {
  float qv = sd[0] - x;
  int cnt = qv < 0.f;
  for (int i = 1; i < n; ++i) {
    if (fabsf(qv) < pivmin) qv = -pivmin;
    qv = sd[i] - x - __fdividef(se2[i - 1], qv);
    cnt += qv < 0.f;
  }
  return cnt;
}

// The same count in float-float; ee2 holds e_i^2.  The reciprocal of the
// previous pivot replaces the division (one Newton step on the float32 rcp).
__device__ __forceinline__ int sturm_count_df(const df* dd, const df* ee2, int n, df x, float pivmin) {
  df qv = df_sub(dd[0], x);
  int cnt = df_lt0(qv);
  for (int i = 1; i < n; ++i) {
    if (fabsf(qv.hi) < pivmin) qv = df{-pivmin, 0.f};
    qv = df_sub(df_sub(dd[i], x), df_mul(ee2[i - 1], df_recip(qv)));
    cnt += df_lt0(qv);
  }
  return cnt;
}

// The phases of the solver are device functions with two drivers: k_syev_df
// runs all of them in one block (the allocation-free entry point), the split
// path runs the tridiagonalisation in one block (k_syev_tri) and spreads the
// per-eigenvalue phases over many: the shifts one warp each (k_syev_vals),
// inverse iteration and clean-up one block per group of close shifts
// (k_syev_vecs) and the back-transformation one warp per eigenvector
// (k_syev_back).  Each eigenvalue's phases do the same arithmetic on both.

// Householder tridiagonalisation of the symmetric W (n x n, row stride LD,
// full storage) by the whole block.  Four barriers per step: the norm of the
// next column and v^T p are formed from per-warp partial sums written in the
// preceding phase.  On return dd, ee hold the tridiagonal, tau the reflector
// scalars and column k of W below the diagonal the reflector v_k, which is
// also written to hv[k n + i] (i < n - k - 1) when hv is given.  v, p: n df of
// scratch each; red_sig, red_vp: 32 per-warp partial sums each.
__device__ void syev_tridiagonalise(int n, df* W, long long LD, df* v, df* p, df* dd, df* ee, df* tau,
                                    df_acc* red_sig, df_acc* red_vp, df* hv) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  // sigma partials of column 0 (rows 2..n-1)
  {
    df_acc a = acc_zero();
    for (int i = 2 + warp; i < n; i += nw)
      if (lane == 0) a.fma(W[i * LD], W[i * LD]);
    if (lane == 0) red_sig[warp] = a;
  }
  __syncthreads();
  for (int k = 0; k + 2 < n; ++k) {
    const int m = n - k - 1;
    df_acc sa = lane < nw ? red_sig[lane] : acc_zero();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sa.merge(shfl_xor_acc(sa, o));
    const df sigma = sa.value();
    const df x0 = W[(k + 1) * LD + k];
    if (sigma.hi == 0.f) {
      if (tid == 0) {
        tau[k] = df{0.f, 0.f};
        dd[k] = W[k * LD + k];
        ee[k] = x0;
      }
      // partials of the next column, unchanged by this step
      __syncthreads();
      df_acc a = acc_zero();
      for (int i = k + 3 + warp; i < n; i += nw)
        if (lane == 0) a.fma(W[i * LD + k + 1], W[i * LD + k + 1]);
      if (lane == 0) red_sig[warp] = a;
      __syncthreads();
      continue;
    }
    const df nrm = df_sqrt(df_add(df_mul(x0, x0), sigma));
    const df alpha = df_lt0(x0) ? nrm : df_neg(nrm);
    const df v0 = df_sub(x0, alpha);
    const df vtv = df_add(sigma, df_mul(v0, v0));
    const df t = df_div(df{2.f, 0.f}, vtv);
    for (int i = tid; i < m; i += nt) v[i] = (i == 0) ? v0 : W[(k + 1 + i) * LD + k];
    if (tid == 0) {
      tau[k] = t;
      dd[k] = W[k * LD + k];
      ee[k] = alpha;
    }
    __syncthreads();  // (1) v complete
    // p = t * W22 v, and per-warp partials of v^T p; column k keeps v for the back-transformation
    {
      df_acc pv = acc_zero();
      for (int i = warp; i < m; i += nw) {
        df_acc b0 = acc_zero(), b1 = acc_zero();
        const df* row = W + (k + 1 + i) * LD + (k + 1);
        int j = lane;
        for (; j + 32 < m; j += 64) {
          const df r0 = row[j], r1 = row[j + 32];
          const df v0j = v[j], v1j = v[j + 32];
          b0.fma(r0, v0j);
          b1.fma(r1, v1j);
        }
        if (j < m) b0.fma(row[j], v[j]);
        b0.merge(b1);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) b0.merge(shfl_xor_acc(b0, o));
        if (lane == 0) {
          const df pi = df_mul(t, b0.value());
          p[i] = pi;
          pv.fma(v[i], pi);
        }
      }
      if (lane == 0) red_vp[warp] = pv;
      for (int i = tid; i < m; i += nt) W[(k + 1 + i) * LD + k] = v[i];
      if (hv != nullptr)
        for (int i = tid; i < m; i += nt) hv[static_cast<long long>(k) * n + i] = v[i];
    }
    __syncthreads();  // (2) p and v^T p partials complete
    {
      df_acc c = lane < nw ? red_vp[lane] : acc_zero();
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) c.merge(shfl_xor_acc(c, o));
      const df kc = df_mul(df_mul_f(t, 0.5f), c.value());
      for (int i = tid; i < m; i += nt) p[i] = df_sub(p[i], df_mul(kc, v[i]));  // w
    }
    __syncthreads();  // (3) w complete
    // W22 -= v w^T + w v^T over whole rows (coalesced; no mirrored column writes):
    // entry (r, c) takes its two products in the order of (max, min), so both
    // triangles stay bitwise equal.  Lane 0 of each row also accumulates the next
    // column's norm (rows 2.. of the trailing block)
    {
      df_acc sg = acc_zero();
      for (int i = warp; i < m; i += nw) {
        const df vi = v[i], wi = p[i];
        df* rowi = W + (k + 1 + i) * LD + (k + 1);
#pragma unroll 2
        for (int j = lane; j < m; j += 32) {
          df_acc u0 = acc_zero();
          if (j <= i) {
            u0.fma(vi, p[j]);
            u0.fma(wi, v[j]);
          } else {
            u0.fma(v[j], wi);
            u0.fma(p[j], vi);
          }
          const df n0 = df_sub(rowi[j], u0.value());
          rowi[j] = n0;
          if (j == 0 && i >= 2) sg.fma(n0, n0);
        }
      }
      if (lane == 0) red_sig[warp] = sg;
    }
    __syncthreads();  // (4) trailing block and next-column partials complete
  }
  if (tid == 0) {
    if (n >= 2) {
      dd[n - 2] = W[(n - 2) * LD + (n - 2)];
      dd[n - 1] = W[(n - 1) * LD + (n - 1)];
      ee[n - 2] = W[(n - 1) * LD + (n - 2)];
      tau[n - 2] = df{0.f, 0.f};
    } else {
      dd[0] = W[0];
    }
    if (n >= 1) tau[n - 1] = df{0.f, 0.f};
  }
  __syncthreads();
}

// Gershgorin interval of the tridiagonal (float32 diagonal sd, squared
// off-diagonal se2), padded, by one thread: sf = {lower, upper, ||T|| bound,
// pivot floor of the Sturm recurrences}.
__device__ void syev_bounds(const float* sd, const float* se2, int n, float* sf) {
  float gl = 3.0e38f, gu = -3.0e38f, emax2 = 0.f;
  for (int i = 0; i < n; ++i) {
    const float r = (i > 0 ? sqrtf(se2[i - 1]) : 0.f) + (i + 1 < n ? sqrtf(se2[i]) : 0.f);
    gl = fminf(gl, sd[i] - r);
    gu = fmaxf(gu, sd[i] + r);
    if (i + 1 < n) emax2 = fmaxf(emax2, se2[i]);
  }
  const float tn = fmaxf(fabsf(gl), fabsf(gu));
  const float pad = 2.0e-6f * tn + 1.0e-30f;
  sf[0] = gl - pad;
  sf[1] = gu + pad;
  sf[2] = tn;
  sf[3] = fmaxf(1.0e-30f, 1.0e-35f * fmaxf(emax2, 1.f));
}

// float32 bisection for the (j+1)-th smallest eigenvalue, one thread.
__device__ float syev_bisect(int j, const float* sd, const float* se2, int n, float gl, float gu, float pivmin) {
  float lo = gl, hi = gu;
  for (int it = 0; it < 80; ++it) {
    const float mid = 0.5f * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    if (sturm_count(sd, se2, n, mid, pivmin) > j) hi = mid; else lo = mid;
  }
  return 0.5f * (lo + hi);
}

// The same bracket by one warp: 32-point multisection, 33x narrower per round
// (Golub & Van Loan 8.4.1), until the float32 points stop separating.
__device__ float syev_multisect(int j, const float* sd, const float* se2, int n, float gl, float gu, float pivmin) {
  const int lane = threadIdx.x & 31;
  float lo = gl, hi = gu;
  for (int round = 0; round < 40; ++round) {
    const float mid = 0.5f * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    const float x = lo + (hi - lo) * (static_cast<float>(lane + 1) * (1.f / 33.f));
    const unsigned above = __ballot_sync(0xffffffffu, sturm_count(sd, se2, n, x, pivmin) > j);
    const int l1 = above ? __ffs(above) - 1 : 32;  // first point with more than j eigenvalues below
    const float xlo = __shfl_sync(0xffffffffu, x, l1 > 0 ? l1 - 1 : 0);
    const float xhi = __shfl_sync(0xffffffffu, x, l1 < 32 ? l1 : 31);
    if (l1 > 0) lo = fmaxf(lo, xlo);
    if (l1 < 32) hi = fminf(hi, xhi);
  }
  return 0.5f * (lo + hi);
}

// Refine the float32 shift s0 of index j with float-float Sturm counts (one
// warp; ee2 holds e_i^2).  The float32 counts can be off by ~n 2^-24 ||T||,
// far more than the gaps inside a graded spectrum; with float-float shifts the
// inverse iteration separates eigenvalues down to ~1e-9 ||T|| apart on its
// own.  The bracket is first widened until its float-float counts enclose
// index j, then 32-point multisection shrinks it 33x per round.  Returns the
// midpoint of the final bracket (the same on every lane).
__device__ df syev_refine_shift(int j, float s0, const df* dd, const df* ee2, int n, float gl, float gu,
                                float tnorm, float pivmin) {
  const int lane = threadIdx.x & 31;
  float w = 1.0e-4f * tnorm + 1.0e-6f * fabsf(s0) + pivmin;
  df lo = df{s0 - w, 0.f}, hi = df{s0 + w, 0.f};
  for (int attempt = 0; attempt < 12; ++attempt) {
    int c = 0;
    if (lane < 2) c = sturm_count_df(dd, ee2, n, lane == 0 ? lo : hi, pivmin);
    const int clo = __shfl_sync(0xffffffffu, c, 0), chi = __shfl_sync(0xffffffffu, c, 1);
    if (clo <= j && chi > j) break;
    w *= 4.f;
    if (attempt == 11) {
      lo = df{gl, 0.f};
      hi = df{gu, 0.f};
    } else {
      if (clo > j) lo = df{s0 - w, 0.f};
      if (chi <= j) hi = df{s0 + w, 0.f};
    }
  }
  const float tol = 1.0e-14f * tnorm + pivmin;
  for (int round = 0; round < 12; ++round) {
    const df width = df_sub(hi, lo);
    if (!(width.hi > tol)) break;
    const df x = df_add(lo, df_mul_f(width, static_cast<float>(lane + 1) * (1.f / 33.f)));
    const unsigned above = __ballot_sync(0xffffffffu, sturm_count_df(dd, ee2, n, x, pivmin) > j);
    const int l1 = above ? __ffs(above) - 1 : 32;  // first point with more than j eigenvalues below
    const float lhi = __shfl_sync(0xffffffffu, x.hi, l1 > 0 ? l1 - 1 : 0);
    const float llo = __shfl_sync(0xffffffffu, x.lo, l1 > 0 ? l1 - 1 : 0);
    const float hhi = __shfl_sync(0xffffffffu, x.hi, l1 < 32 ? l1 : 31);
    const float hlo = __shfl_sync(0xffffffffu, x.lo, l1 < 32 ? l1 : 31);
    if (l1 > 0) lo = df{lhi, llo};
    if (l1 < 32) hi = df{hhi, hlo};
  }
  return df_mul_f(df_add(lo, hi), 0.5f);
}

// Clusters and clean-up groups of the ascending shifts, by one thread.  Shifts
// closer than 1e-9 ||T|| form clusters, iterated in rounds with Gram-Schmidt
// (cpos[j]: position of j in its cluster, which starts at cstart[j]); runs of
// shifts closer than 1e-4 ||T|| form the groups [gs0[j], gs1[j]) of the
// Rayleigh-Ritz clean-up.  si[0] = the largest cluster position, si[1] = 1 if
// any two shifts are closer than 1e-4 ||T||.
__device__ void syev_groups(const df* shd, int nwant, float tnorm, float pivmin, int* cstart, int* cpos, int* gs0,
                            int* gs1, int* si) {
  const float ctol = 1.0e-9f * tnorm + pivmin, rtol = 1.0e-4f * tnorm;
  int maxpos = 0, close = 0, gstart = 0;
  for (int j = 0; j < nwant; ++j) {
    const float gap = shift_gap(shd, j);
    if (gap <= ctol) {
      cstart[j] = cstart[j - 1];
      cpos[j] = cpos[j - 1] + 1;
    } else {
      cstart[j] = j;
      cpos[j] = 0;
    }
    if (gap <= rtol) {
      close = 1;
    } else if (j > 0) {
      for (int i = gstart; i < j; ++i) gs1[i] = j;
      gstart = j;
    }
    gs0[j] = gstart;
    maxpos = max(maxpos, cpos[j]);
  }
  for (int i = gstart; i < nwant; ++i) gs1[i] = nwant;
  si[0] = maxpos;
  si[1] = close;
}

// A vector alone in its group, one thread: its Rayleigh quotient with T goes
// to *eval and the vector, normalised, to Zn (element i at [i ldn]).  Z holds
// element i at [i ldz].
__device__ void syev_single(const df* Z, long long ldz, const df* dd, const df* ee, int n, df* Zn, long long ldn,
                            double* eval) {
  df_acc sq = acc_zero(), hq = acc_zero();
  for (int i = 0; i < n; ++i) {
    const df z = Z[i * ldz];
    df_acc tz = acc_zero();
    tz.fma(dd[i], z);
    if (i > 0) tz.fma(ee[i - 1], Z[(i - 1) * ldz]);
    if (i + 1 < n) tz.fma(ee[i], Z[(i + 1) * ldz]);
    sq.fma(z, z);
    hq.fma(z, tz.value());
  }
  const df sv = sq.value();
  const df inv = df_div(df{1.f, 0.f}, df_sqrt(sv));
  for (int i = 0; i < n; ++i) Zn[i * ldn] = df_mul(Z[i * ldz], inv);
  *eval = df_to_double(df_div(hq.value(), sv));
}

// ---- one-block driver
//
// Dynamic shared memory: v, p (df, n each), sd, se2 (float, n each), shift
// (float, nwant), cstart, cpos (int, nwant), d, e, tau, e^2 (df, n each),
// shifts (df, nwant), gs0, gs1 (int, nwant), then -- when they fit -- the
// working matrix W (n x ldw df), the inverse-iteration factors (2 x n x nwant
// df) and the tridiagonal eigenvectors Zt (n x nwant df).  `flags` bit 0/1/2
// says which of W / factors / Zt live in shared memory; the others use the
// global workspace (same layout), so one code path serves every size.
constexpr int kSyW = 1, kSyF = 2, kSyZ = 4;

__global__ void __launch_bounds__(kSyThreads) k_syev_df(int n, int nwant, int ldw, int flags,
                                                        const double* __restrict__ H, double* __restrict__ evals,
                                                        double* __restrict__ evecs, df* __restrict__ Wg,
                                                        df* __restrict__ tau_g, df* __restrict__ dd_g,
                                                        df* __restrict__ ee_g, df* __restrict__ facg,
                                                        df* __restrict__ Ztg, df* __restrict__ rrw,
                                                        int* __restrict__ perm, const int* __restrict__ skip) {
  if (skip != nullptr && *skip != 0) return;  // the structured fast path already produced the pairs
  extern __shared__ __align__(16) unsigned char smem_raw[];
  df* v = reinterpret_cast<df*>(smem_raw);
  df* p = v + n;
  float* sd = reinterpret_cast<float*>(p + n);
  float* se2 = sd + n;
  float* shift = se2 + n;
  int* cstart = reinterpret_cast<int*>(shift + nwant);
  int* cpos = cstart + nwant;
  size_t off = (2 * sizeof(df) * n + 2 * sizeof(float) * n + sizeof(float) * nwant + 2 * sizeof(int) * nwant +
                4 * sizeof(df) * n + sizeof(df) * nwant + 2 * sizeof(int) * nwant + 15) &
               ~static_cast<size_t>(15);
  df* W = Wg;
  if (flags & kSyW) {
    W = reinterpret_cast<df*>(smem_raw + off);
    off += sizeof(df) * static_cast<size_t>(n) * ldw;
  }
  df* fac = facg;
  if (flags & kSyF) {
    fac = reinterpret_cast<df*>(smem_raw + off);
    off += sizeof(df) * 2 * static_cast<size_t>(n) * nwant;
  }
  df* Zt = Ztg;
  if (flags & kSyZ) Zt = reinterpret_cast<df*>(smem_raw + off);
  __shared__ df_acc red[32];
  __shared__ float sf[4];
  __shared__ int si[4];

  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const long long N = n, LD = ldw;
  // the tridiagonal (d, e) and the Householder scalars live in shared memory
  df* dd = reinterpret_cast<df*>(cpos + nwant);
  df* ee = dd + n;
  df* tau = ee + n;
  df* ee2 = tau + n;     // e_i^2 in float-float (Sturm counts)
  df* shd = ee2 + n;     // float-float shifts (nwant)
  int* gs0 = reinterpret_cast<int*>(shd + nwant);  // clean-up group [gs0[j], gs1[j]) of index j
  int* gs1 = gs0 + nwant;
  __shared__ df_acc red_sig[32], red_vp[32];

  for (long long i = tid; i < N * N; i += nt) W[(i / N) * LD + (i % N)] = df_from_double(H[i]);
  __syncthreads();
  syev_tridiagonalise(n, W, LD, v, p, dd, ee, tau, red_sig, red_vp, nullptr);

  // ---- bisection (float32) for the nwant smallest eigenvalues, refined in float-float
  for (int i = tid; i < n; i += nt) {
    sd[i] = df_float(dd[i]);
    if (i + 1 < n) {
      const float e = df_float(ee[i]);
      se2[i] = e * e;
    }
  }
  __syncthreads();
  if (tid == 0) syev_bounds(sd, se2, n, sf);
  __syncthreads();
  const float gl = sf[0], gu = sf[1], tnorm = sf[2], pivmin = sf[3];
  for (int j = tid; j < nwant; j += nt) shift[j] = syev_bisect(j, sd, se2, n, gl, gu, pivmin);
  for (int i = tid; i + 1 < n; i += nt) ee2[i] = df_mul(ee[i], ee[i]);
  __syncthreads();
  for (int j = warp; j < nwant; j += nw) {
    const df s = syev_refine_shift(j, shift[j], dd, ee2, n, gl, gu, tnorm, pivmin);
    if (lane == 0) shd[j] = s;
  }
  __syncthreads();
  if (tid == 0) syev_groups(shd, nwant, tnorm, pivmin, cstart, cpos, gs0, gs1, si);
  __syncthreads();
  const int maxpos = si[0];
  const bool cleanup = si[1] != 0;

  // ---- inverse iteration in float-float: T - s I = L D L^T -----------------
  // factor arrays (element i of eigen-index j at [i * nwant + j]):
  //   fac[0 .. n*nwant) = 1/d_i, fac[n*nwant .. 2n*nwant) = l_i
  const long long NW = nwant;
  const df pv = df{fmaxf(3.6e-15f * tnorm, 1.0e-30f), 0.f};
  for (int round = 0; round <= maxpos; ++round) {
    for (int j = tid; j < nwant; j += nt) {
      if (cpos[j] != round) continue;
      syev_inverse_iteration(j, j, cstart[j], shd[j], dd, ee, n, pv, fac, fac + N * NW, Zt, NW);
    }
    __syncthreads();
  }

  df* Zn = fac;
  if (!cleanup) {
    // every gap is above 1e-4 ||T||: the vectors are accurate individually
    // (error ~ 48-bit rounding x ||T|| / gap <= 4e-11); their Rayleigh
    // quotients are the eigenvalues, already in ascending order
    for (long long idx = tid; idx < N * NW; idx += nt) Zn[idx] = Zt[idx];
    for (int j = tid; j < nwant; j += nt) {
      df_acc h = acc_zero();
      for (int i = 0; i < n; ++i) {
        df_acc tz = acc_zero();
        tz.fma(dd[i], Zt[i * NW + j]);
        if (i > 0) tz.fma(ee[i - 1], Zt[(i - 1) * NW + j]);
        if (i + 1 < n) tz.fma(ee[i], Zt[(i + 1) * NW + j]);
        h.fma(Zt[i * NW + j], tz.value());
      }
      evals[j] = df_to_double(h.value());
    }
    __syncthreads();
  } else {
    // single vectors only need their Rayleigh quotient; the groups of two or
    // more run one after another on windows of the workspace
    for (int j = tid; j < nwant; j += nt) {
      if (gs1[j] - gs0[j] != 1) continue;
      syev_single(Zt + j, NW, dd, ee, n, Zn + j, NW, evals + j);
    }
    __syncthreads();
    for (int g0 = 0; g0 < nwant;) {
      const int g1 = gs1[g0], G = g1 - g0;
      if (G >= 2)
        syev_group_rr<2, 2>(G, Zt + g0, NW, dd, ee, n, fac + N * NW + g0, rrw, perm, red, sf, Zn + g0, NW,
                            evals + g0);
      g0 = g1;
    }
  }

  // ---- back-transformation y = H_0 H_1 ... H_{n-3} z ------------------------
  // v_k (column k of W below the diagonal) is staged in shared memory once per
  // step.  Each column of Z is split over S consecutive lanes (S = 1..8 threads
  // per column, as many as the block holds): lane seg takes rows seg, seg + S, ...,
  // the partial products meet in a shuffle tree, and the same lanes apply the
  // update -- row walks stay coalesced across columns and each chain is m / S long.
  int S = 1;
  while (S < 8 && 2 * S * nwant <= nt) S <<= 1;
  for (int k = n - 3; k >= 0; --k) {
    const df t = tau[k];
    if (t.hi == 0.f) continue;
    const int m = n - k - 1;
    for (int i = tid; i < m; i += nt) v[i] = W[(k + 1 + i) * LD + k];
    __syncthreads();
    // for each column c: s_c = v^T z[k+1:, c]; z[k+1:, c] -= t s_c v
    const int total = nwant * S;
    for (int base = warp * 32; base < total; base += nt) {
      const int it = base + lane;
      const bool valid = it < total;
      const int c = valid ? it / S : 0, seg = it % S;
      df* zc = Zn + static_cast<long long>(k + 1) * NW + c;
      df_acc s0 = acc_zero(), s1 = acc_zero(), s2 = acc_zero(), s3 = acc_zero();
      if (valid) {
        int i = seg;
        for (; i + 3 * S < m; i += 4 * S) {
          s0.fma(v[i], zc[i * NW]);
          s1.fma(v[i + S], zc[(i + S) * NW]);
          s2.fma(v[i + 2 * S], zc[(i + 2 * S) * NW]);
          s3.fma(v[i + 3 * S], zc[(i + 3 * S) * NW]);
        }
        for (; i < m; i += S) s0.fma(v[i], zc[i * NW]);
      }
      s0.merge(s1);
      s2.merge(s3);
      s0.merge(s2);
      for (int o = 1; o < S; o <<= 1) s0.merge(shfl_xor_acc(s0, o));
      if (valid) {
        const df f = df_mul(t, s0.value());
        for (int i = seg; i < m; i += S) zc[i * NW] = df_sub(zc[i * NW], df_mul(f, v[i]));
      }
    }
    __syncthreads();
  }
  for (long long idx = tid; idx < N * NW; idx += nt) evecs[idx] = df_to_double(Zn[idx]);
}

// ---- split driver
//
// Global workspace: W (n x ldw df) unless it fits in shared memory, the
// reflectors hv (v_k at hv[k n ..]), dd, ee, tau (df, n each), the shifts shd
// (df, nwant) and their bounds (4 floats), the factors and working vectors of
// groups too wide for shared memory (fac: 3 n nwant df) and the tridiagonal
// eigenvectors Zg (n x nwant df).
constexpr int kSvWarps = 4;  // shifts per block of k_syev_vals
constexpr int kSvecThreads = 512;
constexpr int kSbWarps = 8;  // eigenvectors per block of k_syev_back
constexpr int kSbChunk = 8;  // reflectors staged per barrier in k_syev_back

// Tridiagonalisation, one block: W in shared memory when `inshared`, else the
// global Wg.  Writes dd, ee, tau and the reflectors hv to global memory.
__global__ void __launch_bounds__(kSyThreads) k_syev_tri(int n, int ldw, int inshared, const double* __restrict__ H,
                                                         df* __restrict__ Wg, df* __restrict__ hv,
                                                         df* __restrict__ dd_g, df* __restrict__ ee_g,
                                                         df* __restrict__ tau_g, const int* __restrict__ skip) {
  if (skip != nullptr && *skip != 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  df* v = reinterpret_cast<df*>(smem_raw);
  df* p = v + n;
  df* dd = p + n;
  df* ee = dd + n;
  df* tau = ee + n;
  const size_t off = (5 * sizeof(df) * static_cast<size_t>(n) + 15) & ~static_cast<size_t>(15);
  df* W = inshared ? reinterpret_cast<df*>(smem_raw + off) : Wg;
  __shared__ df_acc red_sig[32], red_vp[32];
  const int tid = threadIdx.x, nt = blockDim.x;
  const long long N = n, LD = ldw;
  for (long long i = tid; i < N * N; i += nt) W[(i / N) * LD + (i % N)] = df_from_double(H[i]);
  __syncthreads();
  syev_tridiagonalise(n, W, LD, v, p, dd, ee, tau, red_sig, red_vp, hv);
  for (int i = tid; i < n; i += nt) {
    dd_g[i] = dd[i];
    tau_g[i] = tau[i];
    if (i + 1 < n) ee_g[i] = ee[i];
  }
}

// The same tridiagonalisation by a thread-block cluster of CS CTAs (2, 4 or 8)
// when W is too large for one block's shared memory: CTA r keeps rows
// r R .. r R + R - 1 of W (full rows, stride ldw) in its own shared memory.
// Per step k the owners of column k's entries below the diagonal write them,
// with their partial sums of squares, into every CTA's copy of v (distributed
// shared memory); after a cluster barrier every CTA forms the same reflector
// from the same partials (merged in rank order), computes p = t W22 v for its
// own rows and sends them, with its partial v^T p, to every CTA; after a
// second barrier each CTA forms w = p - (t/2)(v^T p) v and updates its own rows
// (both triangles in the (max, min) product order, so W stays bitwise
// symmetric).  v, p and the partials are double-buffered by the parity of k:
// a CTA that reaches step k + 1 writes buffers that no CTA still reads.
constexpr int kTriMaxCluster = 8;

__device__ __forceinline__ df_acc block_merge(df_acc a, df_acc* red) {
  // every thread's partial merged: warps by shuffles, then warp 0 over the warps (result in lane 0 of warp 0)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a.merge(shfl_xor_acc(a, o));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane == 0) red[warp] = a;
  __syncthreads();
  df_acc b = acc_zero();
  if (warp == 0) {
    b = lane < nw ? red[lane] : acc_zero();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) b.merge(shfl_xor_acc(b, o));
  }
  __syncthreads();
  return b;
}

__global__ void __launch_bounds__(kSyThreads) k_syev_tri_cl(int n, int ldw, int R, const double* __restrict__ H,
                                                            df* __restrict__ hv, df* __restrict__ dd_g,
                                                            df* __restrict__ ee_g, df* __restrict__ tau_g,
                                                            const int* __restrict__ skip) {
  if (skip != nullptr && *skip != 0) return;  // every CTA of the cluster returns here alike
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int CS = static_cast<int>(cl.num_blocks()), rank = static_cast<int>(cl.block_rank());
  extern __shared__ __align__(16) unsigned char smem_raw[];
  df* W = reinterpret_cast<df*>(smem_raw);  // R x ldw: rows r0 .. r1-1
  df* vb = W + static_cast<long long>(R) * ldw;  // 2 x n
  df* pb = vb + 2 * n;                            // 2 x n
  __shared__ df_acc sigp[2][kTriMaxCluster], vpp[2][kTriMaxCluster], red[32];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int r0 = rank * R, r1 = min(n, r0 + R);
  const long long LD = ldw;
  for (long long idx = tid; idx < static_cast<long long>(r1 - r0) * n; idx += nt) {
    const int i = static_cast<int>(idx / n), j = static_cast<int>(idx % n);
    W[i * LD + j] = df_from_double(H[static_cast<long long>(r0 + i) * n + j]);
  }
  __syncthreads();
  // column c's entries below the diagonal (own rows) into every CTA's v buffer, and
  // the partial sum of squares of rows c + 2 .. into every CTA's partials
  auto send_column = [&](int c) {
    const int buf = c & 1;
    df_acc a = acc_zero();
    for (int i = max(r0, c + 1) + tid; i < r1; i += nt) {
      const df x = W[(i - r0) * LD + c];
      for (int r = 0; r < CS; ++r) cl.map_shared_rank(vb + buf * n, r)[i - c - 1] = x;
      if (i >= c + 2) a.fma(x, x);
    }
    const df_acc s = block_merge(a, red);
    if (tid == 0)
      for (int r = 0; r < CS; ++r) cl.map_shared_rank(&sigp[buf][0], r)[rank] = s;
  };
  cl.sync();  // every CTA has started before its shared memory is written
  send_column(0);
  for (int k = 0; k + 2 < n; ++k) {
    const int buf = k & 1, m = n - k - 1;
    cl.sync();  // (1) column k and its partials are everywhere
    df_acc sa = sigp[buf][0];
    for (int r = 1; r < CS; ++r) sa.merge(sigp[buf][r]);
    const df sigma = sa.value();
    df* v = vb + buf * n;
    df* p = pb + buf * n;
    const df x0 = v[0];
    const bool own_k = k >= r0 && k < r1;
    if (sigma.hi == 0.f) {
      if (own_k) {
        if (tid == 0) {
          tau_g[k] = df{0.f, 0.f};
          dd_g[k] = W[(k - r0) * LD + k];
          ee_g[k] = x0;
        }
      }
      cl.sync();  // (2) the same barrier count as a reflecting step
      send_column(k + 1);
      continue;
    }
    const df nrm = df_sqrt(df_add(df_mul(x0, x0), sigma));
    const df alpha = df_lt0(x0) ? nrm : df_neg(nrm);
    const df v0 = df_sub(x0, alpha);
    const df vtv = df_add(sigma, df_mul(v0, v0));
    const df t = df_div(df{2.f, 0.f}, vtv);
    __syncthreads();  // every thread has read v[0]
    if (tid == 0) {
      v[0] = v0;
      if (own_k) {
        tau_g[k] = t;
        dd_g[k] = W[(k - r0) * LD + k];
        ee_g[k] = alpha;
      }
    }
    __syncthreads();
    if (rank == 0)
      for (int i = tid; i < m; i += nt) hv[static_cast<long long>(k) * n + i] = v[i];
    // p_i = t (W22 v)_i for the own trailing rows, one warp per row; partial v^T p
    {
      df_acc pv = acc_zero();
      for (int i = max(r0, k + 1) + warp; i < r1; i += nw) {
        const df* row = W + (i - r0) * LD + (k + 1);
        df_acc b0 = acc_zero(), b1 = acc_zero();
        int j = lane;
        for (; j + 32 < m; j += 64) {
          b0.fma(row[j], v[j]);
          b1.fma(row[j + 32], v[j + 32]);
        }
        if (j < m) b0.fma(row[j], v[j]);
        b0.merge(b1);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) b0.merge(shfl_xor_acc(b0, o));
        if (lane == 0) {
          const df pi = df_mul(t, b0.value());
          for (int r = 0; r < CS; ++r) cl.map_shared_rank(pb + buf * n, r)[i - k - 1] = pi;
          pv.fma(v[i - k - 1], pi);
        }
      }
      const df_acc s = block_merge(pv, red);
      if (tid == 0)
        for (int r = 0; r < CS; ++r) cl.map_shared_rank(&vpp[buf][0], r)[rank] = s;
    }
    cl.sync();  // (2) every p_i and partial v^T p are everywhere
    {
      df_acc c = vpp[buf][0];
      for (int r = 1; r < CS; ++r) c.merge(vpp[buf][r]);
      const df kc = df_mul(df_mul_f(t, 0.5f), c.value());
      for (int i = tid; i < m; i += nt) p[i] = df_sub(p[i], df_mul(kc, v[i]));  // w
    }
    __syncthreads();
    // own rows: W22 -= v w^T + w v^T, one warp per row, lanes along it (column k keeps
    // the entries of the reduced matrix)
    for (int row = max(r0, k + 1) + warp; row < r1; row += nw) {
      const int i = row - k - 1;  // trailing index of the row
      const df vi = v[i], wi = p[i];
      df* rowp = W + (row - r0) * LD + (k + 1);
#pragma unroll 2
      for (int j = lane; j < m; j += 32) {
        df_acc u0 = acc_zero();
        if (j <= i) {
          u0.fma(vi, p[j]);
          u0.fma(wi, v[j]);
        } else {
          u0.fma(v[j], wi);
          u0.fma(p[j], vi);
        }
        rowp[j] = df_sub(rowp[j], u0.value());
      }
    }
    __syncthreads();
    send_column(k + 1);
  }
  // the last 2 x 2 block
  if (tid == 0) {
    if (n >= 2) {
      if (n - 2 >= r0 && n - 2 < r1) dd_g[n - 2] = W[(n - 2 - r0) * LD + (n - 2)];
      if (n - 1 >= r0 && n - 1 < r1) {
        dd_g[n - 1] = W[(n - 1 - r0) * LD + (n - 1)];
        ee_g[n - 2] = W[(n - 1 - r0) * LD + (n - 2)];
      }
      if (rank == 0) tau_g[n - 2] = df{0.f, 0.f};
    } else if (rank == 0) {
      dd_g[0] = W[0];
    }
    if (rank == 0 && n >= 1) tau_g[n - 1] = df{0.f, 0.f};
  }
  cl.sync();  // no CTA leaves while another may still write into its shared memory
}

// The refined shifts, one warp each (kSvWarps per block): float32 multisection
// then float-float refinement.  Block 0 also writes the bounds.  Shared: dd,
// ee2 (df, n each), sd, se2 (float, n each).
__global__ void __launch_bounds__(32 * kSvWarps) k_syev_vals(int n, int nwant, const df* __restrict__ dd_g,
                                                             const df* __restrict__ ee_g, df* __restrict__ shd,
                                                             float* __restrict__ bounds,
                                                             const int* __restrict__ skip) {
  if (skip != nullptr && *skip != 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  df* dd = reinterpret_cast<df*>(smem_raw);
  df* ee2 = dd + n;
  float* sd = reinterpret_cast<float*>(ee2 + n);
  float* se2 = sd + n;
  __shared__ float sf[4];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < n; i += blockDim.x) {
    const df d = dd_g[i];
    dd[i] = d;
    sd[i] = df_float(d);
    if (i + 1 < n) {
      const df e = ee_g[i];
      const float ef = df_float(e);
      se2[i] = ef * ef;
      ee2[i] = df_mul(e, e);
    }
  }
  __syncthreads();
  if (tid == 0) syev_bounds(sd, se2, n, sf);
  __syncthreads();
  if (blockIdx.x == 0 && tid < 4) bounds[tid] = sf[tid];
  const int j = blockIdx.x * kSvWarps + warp;
  if (j >= nwant) return;  // whole warps: no block barrier below
  const float gl = sf[0], gu = sf[1], tnorm = sf[2], pivmin = sf[3];
  const float s0 = syev_multisect(j, sd, se2, n, gl, gu, pivmin);
  const df s = syev_refine_shift(j, s0, dd, ee2, n, gl, gu, tnorm, pivmin);
  if (lane == 0) shd[j] = s;
}

// Inverse iteration and clean-up, one block per group of close shifts: block b
// takes the group that starts at index b (the others exit at once).  A group's
// clusters lie inside it (1e-9 ||T|| < 1e-4 ||T||), so every block runs alone.
// Writes the tridiagonal eigenvectors Zg (n x nwant) and the eigenvalues.
__global__ void __launch_bounds__(kSvecThreads) k_syev_vecs(int n, int nwant, size_t smem_bytes,
                                                            const df* __restrict__ dd_g, const df* __restrict__ ee_g,
                                                            const df* __restrict__ shd, const float* __restrict__ bounds,
                                                            df* __restrict__ facg, df* __restrict__ rrg,
                                                            df* __restrict__ Zg, double* __restrict__ evals,
                                                            const int* __restrict__ skip) {
  if (skip != nullptr && *skip != 0) return;
  const float tnorm = bounds[2], pivmin = bounds[3];
  const float ctol = 1.0e-9f * tnorm + pivmin, rtol = 1.0e-4f * tnorm;
  const int b = blockIdx.x;
  if (b > 0 && shift_gap(shd, b) <= rtol) return;  // not the first index of a group
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ df_acc red[32];
  __shared__ float sf[4];
  __shared__ int sg[2];
  const int tid = threadIdx.x, nt = blockDim.x;
  if (tid == 0) {
    int g1 = b + 1;
    while (g1 < nwant && shift_gap(shd, g1) <= rtol) ++g1;
    sg[0] = g1 - b;
  }
  __syncthreads();
  const int G = sg[0];
  df* dd = reinterpret_cast<df*>(smem_raw);
  df* ee = dd + n;
  int* cst = reinterpret_cast<int*>(ee + n);  // cluster start, local index
  int* cps = cst + G;                         // position in the cluster
  int* perm = cps + G;
  for (int i = tid; i < n; i += nt) {
    dd[i] = dd_g[i];
    if (i + 1 < n) ee[i] = ee_g[i];
  }
  if (tid == 0) {
    int maxpos = 0;
    for (int jj = 0; jj < G; ++jj) {
      if (jj == 0 || !(shift_gap(shd, b + jj) <= ctol)) {
        cst[jj] = jj;
        cps[jj] = 0;
      } else {
        cst[jj] = cst[jj - 1];
        cps[jj] = cps[jj - 1] + 1;
      }
      maxpos = max(maxpos, cps[jj]);
    }
    sg[1] = maxpos;
  }
  __syncthreads();
  const int maxpos = sg[1];
  const long long N = n, NW = nwant;
  // working storage: shared memory when the group fits, else its columns of the global workspace
  const size_t base = syev_vecs_base(n, G);
  const bool local = base + syev_vecs_work(n, G) <= smem_bytes;
  df *dinv, *lm, *Z, *rrw;
  long long ld;
  if (local) {
    dinv = reinterpret_cast<df*>(smem_raw + base);
    lm = dinv + N * G;
    Z = lm + N * G;
    rrw = Z + N * G;
    ld = G;
  } else {
    dinv = facg + b;
    lm = facg + N * NW + b;
    Z = facg + 2 * N * NW + b;
    rrw = rrg + 4LL * b * NW;  // 4 G^2 <= 4 NW (NW - b): the groups' windows do not overlap
    ld = NW;
  }
  const df pv = df{fmaxf(3.6e-15f * tnorm, 1.0e-30f), 0.f};
  for (int round = 0; round <= maxpos; ++round) {
    for (int jj = tid; jj < G; jj += nt)
      if (cps[jj] == round) syev_inverse_iteration(b + jj, jj, cst[jj], shd[b + jj], dd, ee, n, pv, dinv, lm, Z, ld);
    __syncthreads();
  }
  if (G == 1) {
    if (tid == 0) syev_single(Z, ld, dd, ee, n, Zg + b, NW, evals + b);
  } else {
    syev_group_rr<4, 2>(G, Z, ld, dd, ee, n, dinv, rrw, perm, red, sf, Zg + b, NW, evals + b);
  }
}

// Back-transformation y = H_0 H_1 ... H_{n-3} z, one warp per eigenvector
// (column c of Zg), held in shared memory; the block stages kSbChunk
// reflectors at a time (chunk = reflectors k0, k0 - 1, ...) and each warp then
// applies them to its own column without further barriers.  Writes evecs
// (n x nwant float64).
__global__ void __launch_bounds__(32 * kSbWarps) k_syev_back(int n, int nwant, int chunk, const df* __restrict__ hv,
                                                             const df* __restrict__ tau_g,
                                                             const df* __restrict__ Zg, double* __restrict__ evecs,
                                                             const int* __restrict__ skip) {
  if (skip != nullptr && *skip != 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wpb = blockDim.x >> 5;
  const long long NW = nwant;
  df* zs = reinterpret_cast<df*>(smem_raw);  // wpb x n
  df* vs = zs + static_cast<long long>(wpb) * n;  // chunk x n
  const int c = blockIdx.x * wpb + warp;
  const bool live = c < nwant;
  df* z = zs + static_cast<long long>(warp) * n;
  if (live)
    for (int i = lane; i < n; i += 32) z[i] = Zg[i * NW + c];
  for (int k0 = n - 3; k0 >= 0; k0 -= chunk) {
    const int nk = min(chunk, k0 + 1);
    __syncthreads();  // the previous chunk is no longer read
    for (long long idx = tid; idx < static_cast<long long>(nk) * n; idx += blockDim.x) {
      const int r = static_cast<int>(idx / n), i = static_cast<int>(idx % n);
      const int k = k0 - r, m = n - k - 1;
      vs[idx] = i < m ? hv[static_cast<long long>(k) * n + i] : df{0.f, 0.f};
    }
    __syncthreads();
    if (!live) continue;
    for (int r = 0; r < nk; ++r) {
      const int k = k0 - r;
      const df t = tau_g[k];
      if (t.hi == 0.f) continue;
      const int m = n - k - 1;
      const df* v = vs + static_cast<long long>(r) * n;
      df_acc s = acc_zero();
      for (int i = lane; i < m; i += 32) s.fma(v[i], z[k + 1 + i]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s.merge(shfl_xor_acc(s, o));
      const df f = df_mul(t, s.value());
      for (int i = lane; i < m; i += 32) z[k + 1 + i] = df_sub(z[k + 1 + i], df_mul(f, v[i]));
      __syncwarp();
    }
  }
  if (live)
    for (int i = lane; i < n; i += 32) evecs[i * NW + c] = df_to_double(z[i]);
}

size_t syev_smem_base(int n, int nwant) {
  return (2 * sizeof(df) * n + 2 * sizeof(float) * n + sizeof(float) * nwant + 2 * sizeof(int) * nwant +
          4 * sizeof(df) * n + sizeof(df) * nwant + 2 * sizeof(int) * nwant + 15) &
         ~static_cast<size_t>(15);
}

}  // namespace

// Whether a cluster of c blocks of k_syev_tri_cl with `bytes` of shared memory each can be
// resident on this device (asked once per device and size class; the answer is kept).
static bool cluster_fits(int c, size_t bytes) {
  static std::mutex mu;
  static std::map<std::pair<int, int>, bool> known;  // (device, c * 1024 + KiB)
  int dev = 0;
  cudaGetDevice(&dev);
  const int key = c * 1024 + static_cast<int>((bytes + 1023) / 1024);
  std::lock_guard<std::mutex> lk(mu);
  auto it = known.find({dev, key});
  if (it != known.end()) return it->second;
  const cudaError_t before = cudaPeekAtLastError();
  ensure_dynamic_smem(reinterpret_cast<const void*>(k_syev_tri_cl), bytes);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c);
  cfg.blockDim = dim3(kSyThreads);
  cfg.dynamicSmemBytes = bytes;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = c;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  const bool ok = cudaOccupancyMaxActiveClusters(&clusters, k_syev_tri_cl, &cfg) == cudaSuccess && clusters > 0;
  if (!ok && before == cudaSuccess) cudaGetLastError();  // the answer is no; an earlier launch's error stays
  known[{dev, key}] = ok;
  return ok;
}

void launch_eigh(PencilWork* w, int n, int nwant, const double* H, double* evals, double* evecs,
                    cudaStream_t st) {
  if (n <= 0 || nwant <= 0) return;
  // tridiagonalisation: W in shared memory when it fits beside v, p, d, e, tau
  const int ldw = n | 1;  // odd row stride: column walks of W hit different banks
  const size_t tb = (5 * sizeof(df) * static_cast<size_t>(n) + 15) & ~static_cast<size_t>(15);
  const size_t wb = sizeof(df) * static_cast<size_t>(n) * ldw;
  const int inshared = tb + wb <= kSmemBudget;
  const size_t sm_tri = tb + (inshared ? wb : 0);
  const size_t sm_val = 2 * sizeof(df) * static_cast<size_t>(n) + 2 * sizeof(float) * static_cast<size_t>(n);
  // groups keep their vectors in shared memory up to the budget (the widest possible group: all nwant)
  const size_t sm_vec = std::min(kSmemBudget, syev_vecs_base(n, nwant) + syev_vecs_work(n, nwant));
  // back-transformation: kSbWarps columns and kSbChunk staged reflectors of n df, fewer when n is large
  int wpb = kSbWarps;
  while (wpb > 1 && sizeof(df) * static_cast<size_t>(wpb + 1) * n > kSmemBudget) --wpb;
  const int chunk = static_cast<int>(std::max<size_t>(
      1, std::min<size_t>(kSbChunk, (kSmemBudget - sizeof(df) * static_cast<size_t>(wpb) * n) /
                                        (sizeof(df) * static_cast<size_t>(n)))));
  const size_t sm_back = sizeof(df) * static_cast<size_t>(wpb + chunk) * n;
  ProfScope ps(st, P_PENCIL, 8.0 * n * n + 8.0 * n * nwant, 0.0, 4);
  // W too large for one block: a cluster holding its rows, the largest of 8, 4, 2 blocks that can be scheduled
  // (each block's work per step is its rows times the trailing row length: more blocks, shorter steps)
  int cs = 0, rows_per = 0;
  size_t sm_cl = 0;
  if (!inshared)
    for (int c = kTriMaxCluster; c >= 2 && cs == 0; c /= 2) {
      rows_per = (n + c - 1) / c;
      sm_cl = sizeof(df) * (static_cast<size_t>(rows_per) * ldw + 4 * static_cast<size_t>(n));
      if (sm_cl <= kSmemBudget && cluster_fits(c, sm_cl)) cs = c;
    }
  if (cs > 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(kSyThreads);
    cfg.dynamicSmemBytes = sm_cl;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_syev_tri_cl, n, ldw, rows_per, H, w->hv, w->dd, w->ee, w->tau, nullptr);
  } else {
    ensure_dynamic_smem(reinterpret_cast<const void*>(k_syev_tri), sm_tri);
    k_syev_tri<<<1, kSyThreads, sm_tri, st>>>(n, ldw, inshared, H, w->W, w->hv, w->dd, w->ee, w->tau, nullptr);
  }
  ensure_dynamic_smem(reinterpret_cast<const void*>(k_syev_vals), sm_val);
  k_syev_vals<<<ceil_div(nwant, kSvWarps), 32 * kSvWarps, sm_val, st>>>(n, nwant, w->dd, w->ee, w->shd, w->bounds,
                                                                        nullptr);
  ensure_dynamic_smem(reinterpret_cast<const void*>(k_syev_vecs), sm_vec);
  k_syev_vecs<<<nwant, kSvecThreads, sm_vec, st>>>(n, nwant, sm_vec, w->dd, w->ee, w->shd, w->bounds, w->fac, w->rr,
                                                   w->Zt, evals, nullptr);
  ensure_dynamic_smem(reinterpret_cast<const void*>(k_syev_back), sm_back);
  k_syev_back<<<ceil_div(nwant, wpb), 32 * wpb, sm_back, st>>>(n, nwant, chunk, w->hv, w->tau, w->Zt, evecs, nullptr);
}

void launch_eigh_into(int n, int nwant, const double* H, double* evals, double* evecs, df* W, df* tau, df* dd,
                         df* ee, df* fac, df* Zt, df* rr, int* perm, cudaStream_t st) {
  const int ldw = n | 1;
  size_t sm = syev_smem_base(n, nwant);
  int flags = 0;
  const size_t wb = sizeof(df) * static_cast<size_t>(n) * ldw;
  const size_t fb = sizeof(df) * 2 * static_cast<size_t>(n) * nwant;
  const size_t zb = sizeof(df) * static_cast<size_t>(n) * nwant;
  if (sm + wb <= kSmemBudget) {
    flags |= kSyW;
    sm += wb;
  }
  if (sm + fb <= kSmemBudget) {
    flags |= kSyF;
    sm += fb;
  }
  if (sm + zb <= kSmemBudget) {
    flags |= kSyZ;
    sm += zb;
  }
  ProfScope ps(st, P_PENCIL, 8.0 * n * n + 8.0 * n * nwant, 0.0);
  ensure_dynamic_smem(reinterpret_cast<const void*>(k_syev_df), sm);
  k_syev_df<<<1, kSyThreads, sm, st>>>(n, nwant, ldw, flags, H, evals, evecs, W, tau, dd, ee, fac, Zt, rr, perm,
                                       nullptr);
}

// The one-block tridiagonalisation for the solve path's small and very large matrices.
void launch_syev_tri_block(PencilWork* w, int n, int ldw, const double* H, const int* skip, cudaStream_t st) {
  const size_t tb = (5 * sizeof(df) * static_cast<size_t>(n) + 15) & ~static_cast<size_t>(15);
  const size_t wb = sizeof(df) * static_cast<size_t>(n) * ldw;
  const int inshared = tb + wb <= kSmemBudget;
  const size_t sm = tb + (inshared ? wb : 0);
  ensure_dynamic_smem(reinterpret_cast<const void*>(k_syev_tri), sm);
  k_syev_tri<<<1, kSyThreads, sm, st>>>(n, ldw, inshared, H, w->W, w->hv, w->dd, w->ee, w->tau, skip);
}

}  // namespace amgeig
