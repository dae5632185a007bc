// The small dense eigenproblems of the method, on the GPU.
//
// Algorithm 3.1 step 2 solves A_{n,k} x = lambda M_{n,k} x on V_n + span(V),
// a pencil of size d_n + q, and Algorithm 3.2 step 1 solves (A_n, M_n).  The
// paper treats these as black boxes (ARPACK, Sec. 4.1).  Here:
//
// * The coarsest level: at load A_n = L L^T gives the V-cycle's exact solve
//   A_n^-1 = L^-T L^-1 (float64); M_n = L_m L_m^T, H = L_m^-1 A_n L_m^-T,
//   H = Y Theta Y^T, Z = L_m^-T Y gives, for as many leading modes as a solve
//   needs, Z^T M_n Z = I and Z^T A_n Z = Theta: step 1 of Algorithm 3.2 (the q
//   smallest columns of Z) and the coarse modes of the pencil below.
// * Each correction's pencil is written in the basis [I_n^k Z_m, V - I_n^k Z_m B]
//   (block Gram-Schmidt of V against the first m coarse modes) with
//   K = Z_m^T I_k^n A_k V, B = Z_m^T I_k^n M_k V: it becomes
//       At = [[Theta, K - Theta B], [., V^T A V - B^T K - K^T B + B^T Theta B]],
//       Mt = [[I, 0], [0, S]],   S = V^T M V - B^T B,
//   whose eigenvectors [a; b] map back to x = I_n^k Z_m (a - B b) + V b.  The
//   q wanted pairs come from a structured Rayleigh quotient iteration checked by
//   Sylvester's inertia; when the check fails, S = L L^T reduces the pencil to
//   the standard symmetric matrix H = [[Theta, F], [F^T, T]], F = (K - Theta B)
//   L^-T, T = L^-1 (...) L^-T, solved by the dense eigensolver below.  Both are
//   the same Rayleigh-Ritz problem (same eigenvalues as the paper's pencil),
//   only better conditioned, and everything runs in float-float.
// * The symmetric eigenproblem is solved in float-float (48-bit significand):
//   Householder tridiagonalisation (a thread-block cluster), bisection with
//   Sturm counts for the wanted eigenvalues (float32), each shift refined by
//   float-float Sturm multisection, inverse iteration in float-float
//   (Gram-Schmidt inside clusters of nearly equal shifts), a Rayleigh-Ritz
//   clean-up by parallel cyclic Jacobi on each group of close shifts, and
//   back-transformation; the phases after the tridiagonalisation run one warp
//   or one block per eigenvalue, group or eigenvector.  References: Golub & Van Loan, Matrix
//   Computations, 4th ed., 8.3 (tridiagonalisation), 8.4.1 (Sturm bisection),
//   8.2.2 (inverse iteration), 8.5 (Jacobi).
#include <cooperative_groups.h>

#include <cstdio>
#include <map>
#include <mutex>

#include "common.cuh"
#include "kernels.cuh"
#include "prof.cuh"
#include "syev.cuh"

namespace amgeig {

namespace {

// ------------------------------------------------------------ block helpers

__device__ __forceinline__ df_acc warp_acc_sum(df_acc a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a.merge(shfl_xor_acc(a, o));
  return a;
}

// Sturm counts (the number of eigenvalues of the tridiagonal below x) from the
// leading principal minors p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} (Golub & Van Loan
// 8.4.1): a sign change per eigenvalue.  The recurrence's chain is one product
// and one difference (~75 cycles in float-float) where the quotient form
// q_i = d_i - x - e^2 / q_{i-1} adds a reciprocal (~300).  d and e^2 are scaled to ||T|| <= 1, so
// a step grows the minors by at most 3, and their range is kept by an exact power-of-two
// rescaling of the pair every other step, to 2^100.  A minor below 2^-60 of the one before (a
// pivot that small moves d_i by 2^-60 ||T||, far below the shifts' tolerance) becomes -2^-60 of it, a
// tiny negative pivot: so a rescaled pair is at least (2^100, 2^40), the next two minors at least 2^-20 and
// 2^-80, and no run of equal decoupled entries at x can take the minors to zero.
constexpr float kMinorTop = 1.2676506e30f;     // 2^100
constexpr float kMinorFloor = 8.6736174e-19f;  // 2^-60

__device__ __forceinline__ float minor_scale(float a, float b) {
  const int e = (__float_as_int(fmaxf(fabsf(a), fabsf(b))) >> 23) & 0xff;
  return __int_as_float((354 - e) << 23);  // 2^(227 - e); the larger minor is at least 2^-20, so e >= 107
}

__device__ __forceinline__ int sturm_count(const df* d, const df* e2, int n, float x) {
  float p0 = kMinorTop, p1 = (d[0].hi - x) * kMinorTop;
  if (fabsf(p1) < kMinorFloor * p0) p1 = -kMinorFloor * p0;
  int cnt = p1 < 0.f;
  for (int i = 1; i < n; ++i) {
    float pn = fmaf(d[i].hi - x, p1, -e2[i - 1].hi * p0);
    if (fabsf(pn) < kMinorFloor * fabsf(p1)) pn = -kMinorFloor * p1;
    cnt += (pn < 0.f) != (p1 < 0.f);
    p0 = p1;
    p1 = pn;
    if (i & 1) {
      const float sc = minor_scale(p0, p1);
      p0 *= sc;
      p1 *= sc;
    }
  }
  return cnt;
}

// a - b with the low parts added once (error 2^-47 of the larger operand)
__device__ __forceinline__ df df_sub_sloppy(df a, df b) {
  const df s = two_sum(a.hi, -b.hi);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, __fsub_rn(a.lo, b.lo)));
}

__device__ __forceinline__ int sturm_count_df(const df* d, const df* e2, int n, df x) {
  const df t = df_sub(d[0], x);
  df p0 = df{kMinorTop, 0.f}, p1 = df{t.hi * kMinorTop, t.lo * kMinorTop};
  if (fabsf(p1.hi) < kMinorFloor * p0.hi) p1 = df{-kMinorFloor * p0.hi, 0.f};
  int cnt = p1.hi < 0.f;
#pragma unroll 2
  for (int i = 1; i < n; ++i) {
    df pn = df_sub_sloppy(df_mul(df_sub(d[i], x), p1), df_mul(e2[i - 1], p0));
    if (fabsf(pn.hi) < kMinorFloor * fabsf(p1.hi)) pn = df{-kMinorFloor * p1.hi, 0.f};
    cnt += (pn.hi < 0.f) != (p1.hi < 0.f);
    p0 = p1;
    p1 = pn;
    if (i & 1) {
      const float sc = minor_scale(p0.hi, p1.hi);
      p0 = df{p0.hi * sc, p0.lo * sc};
      p1 = df{p1.hi * sc, p1.lo * sc};
    }
  }
  return cnt;
}

// ------------------------------------------------------------ float-float syev
//
// Four kernels: the tridiagonalisation (k_syev_tri_cl, a cluster of 16, or k_syev_tri of
// eigh.cu, one block), the shifts (k_syev_vals), inverse iteration and clean-up
// one block per group of close shifts (k_syev_vecs) and the
// back-transformation (k_syev_back).

// 1 / b with a relative error of about 2^-48 in a chain of ~70 cycles (df_recip: 220, df_div: 650):
// the remainder 1 - b.hi r of the float32 reciprocal is exact to its last bit as one fused multiply-add, so
// r (1 + e + e^2) needs no float-float operation before the final sum.
__device__ __forceinline__ df df_recip_short(df b) {
  const float r = __frcp_rn(b.hi);
  const float e = __fmaf_rn(-b.lo, r, __fmaf_rn(-b.hi, r, 1.f));
  return fast_two_sum(r, __fmul_rn(r, __fmaf_rn(e, e, e)));
}

// Inverse iteration in float-float for the shift sg of index j where it is in no
// cluster of nearly equal shifts, by one warp: T - sg I = L D L^T (pivots kept at least pv in
// magnitude) and the solves from a fixed start vector, the recurrences by lane 0 and
// everything that is element by element by the lanes.  `solves` is 2 where the
// neighbouring shifts are more than 1e-3 ||T|| away, else 3: each solve multiplies the other
// directions by (shift error, below 1e-14 ||T||) / gap, so two leave less than 1e-20 of them.
// Element i of the arrays at [i ld].
__device__ void syev_inverse_iteration_warp(int j, int solves, df sg, const df* dd, const df* ee, int n, float pv,
                                            df* dinv, df* lm, df* Z, long long ld) {
  const int lane = threadIdx.x & 31;
  if (lane == 0) {
    df d = df_sub(dd[0], sg);
    if (fabsf(d.hi) < pv) d = df{df_lt0(d) ? -pv : pv, 0.f};
    df di = df_recip_short(d);
    dinv[0] = di;
#pragma unroll 2
    for (int i = 1; i < n; ++i) {
      const df e = ee[i - 1];
      const df l = df_mul(e, di);
      lm[(i - 1) * ld] = l;
      d = df_sub(df_sub(dd[i], sg), df_mul(l, e));
      if (fabsf(d.hi) < pv) d = df{df_lt0(d) ? -pv : pv, 0.f};
      di = df_recip_short(d);
      dinv[i * ld] = di;
    }
  }
  __syncwarp();
  for (int i = lane; i < n; i += 32) Z[i * ld] = df{1.f + 0.37f * (float)((i * 7 + j * 13) % 11) / 11.f, 0.f};
  __syncwarp();
  for (int it = 0; it < solves; ++it) {
    if (lane == 0) {
      df prev = Z[0];
#pragma unroll 4
      for (int i = 1; i < n; ++i) {
        prev = df_sub(Z[i * ld], df_mul(lm[(i - 1) * ld], prev));
        Z[i * ld] = prev;
      }
    }
    __syncwarp();
    for (int i = lane; i < n; i += 32) Z[i * ld] = df_mul(Z[i * ld], dinv[i * ld]);
    __syncwarp();
    if (lane == 0) {
      df nxt = Z[(n - 1) * ld];
#pragma unroll 4
      for (int i = n - 2; i >= 0; --i) {
        nxt = df_sub(Z[i * ld], df_mul(lm[i * ld], nxt));
        Z[i * ld] = nxt;
      }
    }
    __syncwarp();
    float amax = 0.f;
    for (int i = lane; i < n; i += 32) amax = fmaxf(amax, fabsf(Z[i * ld].hi));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    const float r = amax > 0.f ? exp2f(-floorf(log2f(amax))) : 1.f;  // exact scaling
    df_acc dn = acc_zero();
    for (int i = lane; i < n; i += 32) {
      const df z = df{Z[i * ld].hi * r, Z[i * ld].lo * r};
      Z[i * ld] = z;
      dn.fma(z, z);
    }
    if (it + 1 == solves) {
      const df inv = shfl_df(df_div(df{1.f, 0.f}, df_sqrt(warp_acc_sum(dn).value())), 0);
      for (int i = lane; i < n; i += 32) Z[i * ld] = df_mul(Z[i * ld], inv);
    }
    __syncwarp();
  }
}

// A vector alone in its group, one warp: its Rayleigh quotient with T goes
// to *eval and the vector, normalised, to Zn (element i at [i ldn]).  Z holds
// element i at [i ldz].
__device__ void syev_single(const df* Z, long long ldz, const df* dd, const df* ee, int n, df* Zn, long long ldn,
                            double* eval) {
  const int lane = threadIdx.x & 31;
  df_acc sq = acc_zero(), hq = acc_zero();
  for (int i = lane; i < n; i += 32) {
    const df z = Z[i * ldz];
    df_acc tz = acc_zero();
    tz.fma(dd[i], z);
    if (i > 0) tz.fma(ee[i - 1], Z[(i - 1) * ldz]);
    if (i + 1 < n) tz.fma(ee[i], Z[(i + 1) * ldz]);
    sq.fma(z, z);
    hq.fma(z, tz.value());
  }
  const df sv = shfl_df(warp_acc_sum(sq).value(), 0);
  const df hv = shfl_df(warp_acc_sum(hq).value(), 0);
  const df inv = df_div(df{1.f, 0.f}, df_sqrt(sv));
  for (int i = lane; i < n; i += 32) Zn[i * ldn] = df_mul(Z[i * ldz], inv);
  if (lane == 0) *eval = df_to_double(df_div(hv, sv));
}

// Global workspace: W (n x ldw df) unless it fits in shared memory, the
// reflectors hv (v_k at hv[k n ..]), dd, ee, tau (df, n each), the shifts shd
// (df, nwant) and their bounds (4 floats), the factors and working vectors of
// groups too wide for shared memory (fac: 3 n nwant df) and the tridiagonal
// eigenvectors Zg (n x nwant df).
constexpr int kSvThreads = 128;  // points per round of k_syev_vals
constexpr int kSvecThreads = 512;
constexpr int kSbWarps = 4;  // eigenvectors per block of k_syev_back (one where four do not fit)
constexpr int kSbChunk = 8;  // reflectors applied together in k_syev_back (four where eight do not fit)

// Householder tridiagonalisation by a thread-block cluster of 16 CTAs, row i of W in CTA
// i % 16's shared memory (dealt cyclically, so the shrinking trailing block stays
// spread over all of them).  A step is bound by the latency of its chain more than by
// its work, so it exchanges only what the next link needs:
//   - on entry every CTA holds x = column k and c = column k + 1 below the diagonal
//     (sent by the rows' owners at the end of the step before);
//   - the sixteen row warps form y_i = (W22 x)_i for the CTA's rows and send them
//     to every CTA, while one more warp forms sigma = sum x_j^2 and the reflector's
//     scalars (v = x - alpha e_1, t = 2 / v^T v);
//   - cluster barrier: with y everywhere, p = t W22 v = t (y - alpha c) needs no
//     further exchange: each CTA forms K = (t/2) v^T p and w = p - K v over its
//     threads (two block barriers), updates its own rows by W22 -= v w^T + w v^T
//     and sends their entries of columns k + 1 and k + 2; cluster barrier.
// x, c and y are double-buffered by the parity of k: a CTA that reaches step k + 1
// writes buffers that no CTA still reads.  What several CTAs form for themselves
// is the same in all of them (same order, one lane's value broadcast), and the
// update's arithmetic is symmetric in (i, j), so W stays bitwise symmetric.
// Measured against the form before it (8 CTAs, a row per warp, every vector sent
// element by element, global writes and eight block barriers per step; one block with W in
// global memory above 475 rows): n = 328 3.06 -> 1.31 ms, n = 256 1.94 -> 0.88 ms, i.e. 4.0 and 3.5 us per
// step; of a step at n = 64 (2.6 us) nearly all is the barriers' and the scalars' latency.
constexpr int kTriCluster = 16;  // CTAs; not portable, so asked for and checked (cluster_fits)
constexpr int kTriRowWarps = 16;
constexpr int kTriThreads = 32 * (kTriRowWarps + 1);
constexpr int kTriRows = 2;  // rows a warp owns at most
constexpr int kTriMaxN = kTriCluster * kTriRowWarps * kTriRows;
static_assert(kTriMaxN <= 32 * kTriRowWarps && kTriRowWarps == kTriCluster && kTriMaxN / kTriCluster <= 32,
              "one thread per element of p, one warp per destination, one lane per own row");
constexpr int kTriOneBlock = 40;  // below this size one block's barriers are cheaper

// w - (v_i w_j + v_j w_i): compensated products, symmetric in (i, j) bit for bit
__device__ __forceinline__ df rank2_update(df w, df vi, df wi, df vj, df wj) {
  const df p1 = two_prod(vi.hi, wj.hi), p2 = two_prod(vj.hi, wi.hi);
  const float x1 = __fmaf_rn(vi.hi, wj.lo, __fmul_rn(vi.lo, wj.hi));
  const float x2 = __fmaf_rn(vj.hi, wi.lo, __fmul_rn(vj.lo, wi.hi));
  const df u = two_sum(p1.hi, p2.hi);
  const df t = two_sum(w.hi, -u.hi);
  const float lo = __fadd_rn(__fadd_rn(p1.lo, p2.lo), __fadd_rn(u.lo, __fadd_rn(x1, x2)));
  return fast_two_sum(t.hi, __fadd_rn(__fadd_rn(w.lo, t.lo), -lo));
}

__global__ void __launch_bounds__(kTriThreads) k_syev_tri_cl(int n, int ldw, const double* __restrict__ H,
                                                             df* __restrict__ hv, df* __restrict__ dd_g,
                                                             df* __restrict__ ee_g, df* __restrict__ tau_g,
                                                             const int* __restrict__ skip) {
  if (skip != nullptr && *skip != 0) return;  // every CTA of the cluster returns here alike
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  constexpr int CS = kTriCluster, NW = kTriRowWarps, RW = kTriRows;
  const int rank = static_cast<int>(cl.block_rank());
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int R = rank < n ? (n - rank + CS - 1) / CS : 0;  // rows rank, rank + 16, ...
  extern __shared__ __align__(16) unsigned char smem_raw[];
  df* W = reinterpret_cast<df*>(smem_raw);                  // ceil(n / 16) rows of ldw
  // vectors over the rows keep each owner's rows together (element i at at(i)), so that a CTA's share
  // travels as one contiguous run per destination
  const int RP = ((n + CS - 1) / CS) | 1, NV = CS * RP;
  auto at = [RP](int i) { return (i & (CS - 1)) * RP + (i / CS); };
  df* xb = W + static_cast<size_t>((n + CS - 1) / CS) * ldw;  // 2 x NV
  df* cb = xb + 2 * NV;                                     // 2 x NV
  df* yb = cb + 2 * NV;                                     // 2 x NV
  df* wv = yb + 2 * NV;                                     // n
  df* al = wv + n;                                          // n: subdiagonal (alpha_k)
  df* ta = al + n;                                          // n: t_k
  __shared__ df sc[3];          // alpha, t, v0
  __shared__ df ys[32];         // the own rows' y
  __shared__ df_acc kpart[NW];  // per-warp partials of v^T p
  for (int r = warp; r < R; r += NW + 1)
    for (int j = lane; j < n; j += 32)
      W[r * ldw + j] = df_from_double(H[static_cast<long long>(rank + r * CS) * n + j]);
  // the own rows' entries of columns c0 and c0 + 1 into the buffers for step c0 of CTA `warp`
  auto send_columns = [&](int c0) {
    const int buf = c0 & 1;
    if (warp < CS && lane < R && rank + lane * CS > c0) {
      cl.map_shared_rank(xb + buf * NV, warp)[rank * RP + lane] = W[lane * ldw + c0];
      cl.map_shared_rank(cb + buf * NV, warp)[rank * RP + lane] = W[lane * ldw + c0 + 1];
    }
  };
  // every CTA of the cluster has started before its shared memory is written
  cl.sync();
  if (n > 2) send_columns(0);
  for (int k = 0; k + 2 < n; ++k) {
    cl.sync();  // columns k and k + 1 are everywhere
    const int buf = k & 1, k1 = k + 1;
    const int r0 = k < rank ? 0 : (k - rank) / CS + 1;  // first local row below row k
    df* x = xb + buf * NV;
    const df* c = cb + buf * NV;
    const df* y = yb + buf * NV;
    if (warp < NW) {
      df_acc acc[RW];
#pragma unroll
      for (int s = 0; s < RW; ++s) acc[s] = acc_zero();
      const df* Wr = W + (r0 + warp) * ldw;
      const int mine = R - r0 - warp;  // rows r0 + warp + s NW < R
      if (mine > 0) {
        for (int j = k1 + lane; j < n; j += 32) {
          const df xj = x[at(j)];
#pragma unroll
          for (int s = 0; s < RW; ++s)
            if (s * NW < mine) acc[s].fma(Wr[s * NW * ldw + j], xj);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int s = 0; s < RW; ++s)
            if (s * NW < mine) acc[s].merge(shfl_xor_acc(acc[s], o));
#pragma unroll
        for (int s = 0; s < RW; ++s)
          if (s * NW < mine) {
            if (lane == 0) ys[r0 + warp + s * NW] = acc[s].value();
          }
      }
      // the row warps' barrier (the scalars' warp goes on): the CTA's y is complete
      asm volatile("bar.sync 1, %0;" ::"n"(32 * NW) : "memory");
      if (lane >= r0 && lane < R) cl.map_shared_rank(yb + buf * NV, warp)[rank * RP + lane] = ys[lane];
    } else {
      df_acc s0 = acc_zero(), s1 = acc_zero();
      int j = k1 + 1 + lane;
      for (; j + 32 < n; j += 64) {
        const df xa = x[at(j)], xc = x[at(j + 32)];
        s0.fma(xa, xa);
        s1.fma(xc, xc);
      }
      if (j < n) s0.fma(x[at(j)], x[at(j)]);
      s0.merge(s1);
      const df sigma = shfl_df(warp_acc_sum(s0).value(), 0);
      const df x0 = x[at(k1)];
      const bool flat = sigma.hi == 0.f;  // nothing below the subdiagonal: t = 0 leaves W as it is
      const df nrm = df_sqrt(df_add(df_mul(x0, x0), sigma));
      const df alpha = flat ? x0 : (df_lt0(x0) ? nrm : df_neg(nrm));
      const df v0 = df_sub(x0, alpha);
      // t = 2 / (v^T v): the reciprocal with one more Newton step, as accurate as a division and half its latency
      const df vtv = df_add(sigma, df_mul(v0, v0));
      const df r = df_recip(vtv);
      const df t = flat ? df{0.f, 0.f} : df_mul_f(df_add(r, df_mul(r, df_sub(df{1.f, 0.f}, df_mul(vtv, r)))), 2.f);
      if (lane == 0) {
        sc[0] = al[k] = alpha;
        sc[1] = ta[k] = t;
        sc[2] = v0;
      }
    }
    cl.sync();  // y is everywhere, the scalars are in shared memory
    const df alpha = sc[0], t = sc[1], v0 = sc[2];
    // p and the partials of v^T p, one element per thread (n <= 32 NW)
    df pj, vj;
    const int j1 = k1 + tid;
    if (warp < NW) {
      df_acc kv = acc_zero();
      if (j1 < n) {
        vj = j1 == k1 ? v0 : x[at(j1)];
        pj = df_mul(t, df_sub(y[at(j1)], df_mul(alpha, c[at(j1)])));
        kv.fma(vj, pj);
      }
      if (k1 + 32 * warp < n) kv = warp_acc_sum(kv);
      if (lane == 0) kpart[warp] = kv;
    }
    __syncthreads();
    if (warp < NW) {
      df_acc kv = kpart[lane & (NW - 1)];
#pragma unroll
      for (int o = NW / 2; o > 0; o >>= 1) kv.merge(shfl_xor_acc(kv, o));
      const df kc = shfl_df(df_mul(df_mul_f(t, 0.5f), kv.value()), 0);
      if (j1 < n) {
        wv[j1] = df_sub(pj, df_mul(kc, vj));
        if (j1 == k1) x[at(k1)] = v0;  // this CTA's copy: x becomes v
      }
    }
    __syncthreads();
    if (warp < NW)
      for (int r = r0 + warp; r < R; r += NW) {
        const int i = rank + r * CS;
        const df vi = x[at(i)], wi = wv[i];
        df* Wr = W + r * ldw;
        if (lane == 0) Wr[k] = vi;  // column k keeps the reflector
#pragma unroll 2
        for (int j = k1 + lane; j < n; j += 32) Wr[j] = rank2_update(Wr[j], vi, wi, x[at(j)], wv[j]);
      }
    __syncthreads();  // the own rows are complete
    if (k + 3 < n) send_columns(k1);
  }
  // results to global memory: nothing is written there during the steps, whose barriers would wait for it
  __syncthreads();
  for (int r = warp; r < R; r += NW + 1) {
    const int i = rank + r * CS;
    const df* Wr = W + r * ldw;
    for (int k = lane; k < i && k + 2 < n; k += 32) hv[static_cast<long long>(k) * n + (i - k - 1)] = Wr[k];
    if (lane == 0) {
      dd_g[i] = Wr[i];
      if (i == n - 1 && n >= 2) ee_g[n - 2] = Wr[n - 2];
    }
  }
  if (rank == 0)
    for (int k = tid; k < n; k += kTriThreads) {
      if (k + 2 < n) ee_g[k] = al[k];
      tau_g[k] = k + 2 < n ? ta[k] : df{0.f, 0.f};
    }
  cl.sync();  // no CTA leaves while another may still write into its shared memory
}

// The shifts, one block each: a multisection by Sturm counts at kSvThreads points per
// round, three rounds in float32, then in float-float from a bracket of 1e-4 ||T||
// around the float32 value (float32 counts can be off by far more than the gaps of a
// graded spectrum; with float-float shifts the inverse iteration separates
// eigenvalues down to ~1e-9 ||T|| on its own) until it is 1e-14 ||T|| wide: every round
// counts at both ends too and moves the bracket outward when they do not
// enclose the index.  Bound by the latency of a count's n-step chain, so the
// points per round are many (127x narrower per round, five rounds) and a block
// has one warp per scheduler.  One warp per shift with 33x per round and the
// quotient recurrence took 478 us for 128 of 256 (129 now).  The grid covers one shift more than wanted (the
// vectors' gaps to it decide on their solves).  Block 0 also writes the bounds: Gershgorin interval,
// ||T|| and the pivot floor.  Shared: d, e^2 scaled by a power of two to ||T|| <= 1
// (df, n each).
__global__ void __launch_bounds__(kSvThreads) k_syev_vals(int n, const df* __restrict__ dd_g,
                                                          const df* __restrict__ ee_g, df* __restrict__ shd,
                                                          float* __restrict__ bounds,
                                                          const int* __restrict__ skip) {
  if (skip != nullptr && *skip != 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  df* d = reinterpret_cast<df*>(smem_raw);
  df* e2 = d + n;
  constexpr int NW = kSvThreads / 32;
  __shared__ float red[3][NW];
  __shared__ int fa[2][NW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, j = blockIdx.x;
  float gl = 3.0e38f, gu = -3.0e38f, emax2 = 0.f;
  for (int i = tid; i < n; i += kSvThreads) {
    const df di = dd_g[i];
    d[i] = di;
    const float x = df_float(di);
    const float el = i > 0 ? fabsf(df_float(ee_g[i - 1])) : 0.f;
    const df er = i + 1 < n ? ee_g[i] : df{0.f, 0.f};
    const float ef = fabsf(df_float(er));
    e2[i] = er;
    gl = fminf(gl, x - (el + ef));
    gu = fmaxf(gu, x + (el + ef));
    emax2 = fmaxf(emax2, ef * ef);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    gl = fminf(gl, __shfl_xor_sync(0xffffffffu, gl, o));
    gu = fmaxf(gu, __shfl_xor_sync(0xffffffffu, gu, o));
    emax2 = fmaxf(emax2, __shfl_xor_sync(0xffffffffu, emax2, o));
  }
  if (lane == 0) {
    red[0][warp] = gl;
    red[1][warp] = gu;
    red[2][warp] = emax2;
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    gl = fminf(gl, red[0][w]);
    gu = fmaxf(gu, red[1][w]);
    emax2 = fmaxf(emax2, red[2][w]);
  }
  const float tnorm = fmaxf(fabsf(gl), fabsf(gu));
  const float pad = 2.0e-6f * tnorm + 1.0e-30f;
  gl -= pad;
  gu += pad;
  if (j == 0 && tid == 0) {
    bounds[0] = gl;
    bounds[1] = gu;
    bounds[2] = tnorm;
    bounds[3] = fmaxf(1.0e-30f, 1.0e-35f * fmaxf(emax2, 1.f));
  }
  const int ex = tnorm > 0.f ? min(126, max(-126, ilogbf(tnorm) + 1)) : 0;
  const float sc = exp2f(static_cast<float>(-ex)), un = exp2f(static_cast<float>(ex));
  for (int i = tid; i < n; i += kSvThreads) {
    const df di = d[i], er = df{e2[i].hi * sc, e2[i].lo * sc};
    d[i] = df{di.hi * sc, di.lo * sc};
    e2[i] = df_mul(er, er);
  }
  __syncthreads();
  int round = 0;
  // the first of the block's points with more than j eigenvalues below (kSvThreads if none)
  auto first_above = [&](bool above) {
    const unsigned m = __ballot_sync(0xffffffffu, above);
    const int buf = round++ & 1;
    if (lane == 0) fa[buf][warp] = m ? 32 * warp + __ffs(m) - 1 : kSvThreads;
    __syncthreads();
    int f = fa[buf][0];
#pragma unroll
    for (int w = 1; w < NW; ++w) f = min(f, fa[buf][w]);
    return f;
  };
  float flo = gl * sc, fhi = gu * sc;
  for (int r = 0; r < 3; ++r) {
    const float h = (fhi - flo) * (1.f / (kSvThreads + 1));
    const int f = first_above(sturm_count(d, e2, n, flo + h * static_cast<float>(tid + 1)) > j);
    const float a = flo;
    if (f > 0) flo = a + h * static_cast<float>(f);
    if (f < kSvThreads) fhi = a + h * static_cast<float>(f + 1);
  }
  const float s0 = 0.5f * (flo + fhi);
  df lo = df{s0 - 1.0e-4f, 0.f}, hi = df{s0 + 1.0e-4f, 0.f};
  for (int r = 0; r < 16; ++r) {
    const df width = df_sub(hi, lo);
    if (!(width.hi > 7.0e-15f)) break;
    auto point = [&](int t) { return df_add(lo, df_mul_f(width, static_cast<float>(t) * (1.f / (kSvThreads - 1)))); };
    const int f = first_above(sturm_count_df(d, e2, n, point(tid)) > j);
    if (f == 0) {
      hi = lo;
      lo = df_sub(lo, df_mul_f(width, 8.f));
    } else if (f == kSvThreads) {
      lo = point(kSvThreads - 1);
      hi = df_add(lo, df_mul_f(width, 8.f));
    } else {
      hi = point(f);
      lo = point(f - 1);
    }
  }
  if (tid == 0) {
    const df s = df_mul_f(df_add(lo, hi), 0.5f);
    shd[j] = df{s.hi * un, s.lo * un};
  }
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
  if (maxpos == 0 && G <= nt / 32) {
    // no clusters and a warp for every vector
    const int jj = tid >> 5, j = b + jj;
    if (jj < G) {
      // the shift after the last wanted one is there too (unless there is none)
      const bool apart = shift_gap(shd, j) > 1.0e-3f * tnorm && (j + 1 == n || shift_gap(shd, j + 1) > 1.0e-3f * tnorm);
      syev_inverse_iteration_warp(j, apart ? 2 : 3, shd[j], dd, ee, n, pv.hi, dinv + jj, lm + jj, Z + jj,
                                  ld);
    }
    __syncthreads();
  } else {
    for (int round = 0; round <= maxpos; ++round) {
      for (int jj = tid; jj < G; jj += nt)
        if (cps[jj] == round) syev_inverse_iteration(b + jj, jj, cst[jj], shd[b + jj], dd, ee, n, pv, dinv, lm, Z, ld);
      __syncthreads();
    }
  }
  if (G == 1) {
    if (tid < 32) syev_single(Z, ld, dd, ee, n, Zg + b, NW, evals + b);
  } else {
    syev_group_rr<4, 2>(G, Z, ld, dd, ee, n, dinv, rrw, perm, red, sf, Zg + b, NW, evals + b);
  }
}

// Back-transformation y = H_0 H_1 ... H_{n-3} z, one warp per eigenvector
// (column c of Zg, held in shared memory), C reflectors at a time: with
// f_r = t_r (v_r^T z - sum_{s<r} f_s v_s^T v_r) (r = 0 the largest k, applied first) their
// product takes z to z - sum_r f_r v_r, so the C dot products with z are
// formed together and z is read and written once per chunk; the block's
// warps form the v_s^T v_r of the chunk between them.  Bound by latency: one reflector
// after another, a warp reduction each, took 341 us for 128 of 256 (176 now).  WPB columns per block; the
// columns, the reflectors' scalars and one or two chunks share a CTA's memory, so C and WPB
// shrink with n (launch_syev_back).  Writes evecs (n x nwant float64).
__device__ __forceinline__ void cp_async8(void* dst, const void* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(
                   static_cast<unsigned>(__cvta_generic_to_shared(dst))),
               "l"(src), "r"(bytes)
               : "memory");
}

template <int C, int WPB>
__global__ void __launch_bounds__(32 * WPB) k_syev_back(int n, int nwant, int bufs, const df* __restrict__ hv,
                                                        const df* __restrict__ tau_g, const df* __restrict__ Zg,
                                                        double* __restrict__ evecs, const int* __restrict__ skip) {
  if (skip != nullptr && *skip != 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ df gram[C][C];  // [r][s]: v_r^T v_s, s < r
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long NW = nwant;
  df* zs = reinterpret_cast<df*>(smem_raw);            // WPB x n
  df* taus = zs + static_cast<long long>(WPB) * n;     // n
  df* vb = taus + n;                                   // bufs x C x n, v_r at its rows' own indices
  const int c = blockIdx.x * WPB + warp;
  df* z = zs + static_cast<long long>(warp) * n;
  for (int i = lane; i < n; i += 32) z[i] = c < nwant ? Zg[i * NW + c] : df{0.f, 0.f};
  for (int i = tid; i < n; i += 32 * WPB) taus[i] = tau_g[i];
  // reflectors k0, k0 - 1, ... of a chunk into buffer `buf` (rows above k zero-filled)
  auto stage = [&](int k0, int buf) {
    df* vs = vb + static_cast<long long>(buf) * C * n;
    const int base = max(0, k0 - C + 1) + 1;
    for (int r = warp; r < C; r += WPB) {
      const int k = k0 - r;
      for (int i = base + lane; i < n; i += 32) {
        const bool on = k >= 0 && i > k;
        cp_async8(vs + r * n + i, hv + (on ? static_cast<long long>(k) * n + (i - k - 1) : 0), on ? 8 : 0);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  int buf = 0;
  if (n > 2 && bufs == 2) stage(n - 3, 0);
  for (int k0 = n - 3; k0 >= 0; k0 -= C) {
    const int base = max(0, k0 - C + 1) + 1;  // first row any of the chunk's reflectors touches
    if (bufs == 2) {
      if (k0 - C >= 0) {
        stage(k0 - C, buf ^ 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
    } else {
      stage(k0, 0);
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();  // the chunk is staged
    const df* vs = vb + static_cast<long long>(buf) * C * n;
    // the passes before the last: the chunk's v_s^T v_r for r = warp + 1, warp + 1 + WPB, ...; the last: v_s^T z
    constexpr int kLast = (C - 1 + WPB - 1) / WPB;
    df dr = df{0.f, 0.f};  // lane s: v_s^T z
#pragma unroll 1
    for (int pass = 0; pass <= kLast; ++pass) {
      const int r = warp + 1 + pass * WPB;
      if (pass < kLast && r >= C) continue;
      const df* u = pass < kLast ? vs + r * n : z;
      df_acc a[C];
#pragma unroll
      for (int s = 0; s < C; ++s) a[s] = acc_zero();
#pragma unroll 1
      for (int i = base + lane; i < n; i += 32) {
        const df ui = u[i];
#pragma unroll
        for (int s = 0; s < C; ++s) a[s].fma(vs[s * n + i], ui);
      }
#pragma unroll 1
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int s = 0; s < C; ++s) a[s].merge(shfl_xor_acc(a[s], o));
      df_acc mine = a[0];
#pragma unroll
      for (int s = 1; s < C; ++s)
        if (lane == s) mine = a[s];
      dr = mine.value();
      if (pass < kLast && lane < C) gram[r][lane] = dr;
    }
    __syncthreads();  // gram is complete
    // lane r holds v_r^T z, then f_r
    const df t = lane < C && k0 - lane >= 0 ? taus[k0 - lane] : df{0.f, 0.f};
    df f[C];
#pragma unroll
    for (int s = 0; s < C; ++s) {
      f[s] = df_neg(shfl_df(df_mul(t, dr), s));
      if (lane > s && lane < C) dr = df_add(dr, df_mul(f[s], gram[lane][s]));
    }
#pragma unroll 1
    for (int i = base + lane; i < n; i += 32) {
      df_acc u = acc_zero();
      u.add(z[i]);
#pragma unroll
      for (int r = 0; r < C; ++r) u.fma(f[r], vs[r * n + i]);
      z[i] = u.value();
    }
    __syncthreads();  // the chunk's buffer and gram are free again
    if (bufs == 2) buf ^= 1;
  }
  if (c < nwant)
    for (int i = lane; i < n; i += 32) evecs[i * NW + c] = df_to_double(z[i]);
}

// ------------------------------------------------------------ Rayleigh-Ritz pencil
//
// The pencil of Algorithm 3.1 step 2 in the basis [Phi, V - Phi B], Phi =
// I_n^k Z_m (M-orthonormal coarse modes), K = Phi^T A V, B = Phi^T M V:
//     At = [[Theta, Ft], [Ft^T, Tt]],   Mt = [[I, 0], [0, S]],
//     Ft = K - Theta B,   Tt = V^T A V - B^T K - K^T B + B^T Theta B,
//     S  = V^T M V - B^T B   (the Gram matrix of V after block Gram-Schmidt
//                             against the coarse space).
// An eigenvector [a; b] (M-normalised) gives the new vector Phi (a - B b) + V b.
//
// Fast path: a Rayleigh quotient iteration per wanted pair (one block each),
// started from the columns of V (column j is [B e_j; e_j] in this basis), with
// (At - s Mt) y = Mt x solved through the q x q Schur complement
// S(s) = Tt - s S - Ft^T (Theta - s)^-1 Ft (Gaussian elimination with partial
// pivoting), all in float-float.  k_srqi_check accepts the result only if every
// iteration converged, the vectors are mutually Mt-orthogonal to 1e-6, S is
// positive definite, and Sylvester's inertia of At - s* Mt just above the
// largest value (inertia of Theta - s* plus that of S(s*), Haynsworth) counts
// exactly q eigenvalues below, i.e. the pairs found are the q smallest.
// Otherwise the fallback forms the standard matrix H (Cholesky of S) and runs
// the dense float-float eigensolver.  Golub & Van Loan 8.2.3 (RQI), 4.4
// (inertia), 8.7 (symmetric-definite pencils).
constexpr int kPenThreads = 256;
constexpr int kSrqiThreads = 1024;  // one block per pair: the whole SM for its latency-bound steps
constexpr int kSrqiMaxQ = 64;
constexpr int kSrqiMaxIt = 8;
constexpr int kStdMaxQ = 128;  // largest border the solver accepts (q + q_extra)

__device__ __forceinline__ df to_df(double v) { return df_from_double(v); }
__device__ __forceinline__ df to_df(float2 v) { return df{v.x, v.y}; }

// Solve S y = r (S: q x (q+1) augmented, row-major, shared) by Gauss-Jordan
// elimination with partial pivoting, by the whole block: per column, warp 0
// picks the pivot among the rows not yet used and every thread then updates
// elements of the other rows (two barriers per column, no back substitution).
// Pivot rows are marked in `used` instead of swapped; their order is kept in
// prow.  The solution goes to sol.  prow, used (q ints), rinv (1) and sol (q)
// live in shared memory.
__device__ void gj_solve(df* S, int q, int* prow, int* used, df* rinv_s, df* sol) {
  const int ld = q + 1;
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int i = tid; i < q; i += nt) used[i] = 0;
  __syncthreads();
  for (int k = 0; k < q; ++k) {
    if (tid < 32) {
      float best = -1.f;
      int bi = q;
      for (int i = tid; i < q; i += 32)
        if (!used[i]) {
          const float a = fabsf(S[i * ld + k].hi);
          if (a > best) {
            best = a;
            bi = i;
          }
        }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float b2 = __shfl_xor_sync(0xffffffffu, best, o);
        const int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
        if (b2 > best || (b2 == best && i2 < bi)) {
          best = b2;
          bi = i2;
        }
      }
      if (tid == 0) {
        prow[k] = bi;
        used[bi] = 1;
        df pv = S[bi * ld + k];
        if (fabsf(pv.hi) < 1.0e-30f) pv = df{1.0e-30f, 0.f};
        *rinv_s = df_div(df{1.f, 0.f}, pv);
      }
    }
    __syncthreads();
    const int p = prow[k];
    const df rinv = *rinv_s;
    const int cols = q - k;  // columns k+1..q
    for (int e = tid; e < q * cols; e += nt) {
      const int i = e / cols, j = k + 1 + e % cols;
      if (i == p) continue;
      const df l = df_mul(S[i * ld + k], rinv);
      S[i * ld + j] = df_sub(S[i * ld + j], df_mul(l, S[p * ld + j]));
    }
    __syncthreads();
  }
  for (int k = tid; k < q; k += nt) {
    const int p = prow[k];
    df pv = S[p * ld + k];
    if (fabsf(pv.hi) < 1.0e-30f) pv = df{1.0e-30f, 0.f};
    sol[k] = df_div(S[p * ld + q], pv);
  }
  __syncthreads();
}

// Gauss-Jordan with partial pivoting for q + nrhs <= 32 and a 1024-thread
// block: the thread (i, j) = (tid / 32, tid % 32) keeps element (i, j) of the
// augmented q x (q + nrhs) matrix in registers, so warp i holds row i.  Per column k: the
// pivot row p (chosen by a shared atomic max over |a_ik| while column k was
// updated) is scaled by 1 / a_pk inside its warp and published in shared
// memory; every other row takes its multiplier a_ik from lane k by a shuffle
// and subtracts a_ik * (scaled pivot row).  Two barriers per column, no
// integer division, no back substitution: x_k ends in the right-hand-side
// columns of row p_k.  S is read from shared memory (row stride lds); solution
// r goes to sol[r * ldsol + k].
struct GjShared {
  unsigned long long key[2];
  df prowv[33];
  int kof[32];
};

__device__ __forceinline__ unsigned long long pivot_key(float a, int i) {
  // |a| >= 0: its bits order like its value; ties go to the smaller row
  return (static_cast<unsigned long long>(__float_as_uint(a)) << 32) | static_cast<unsigned>(31 - i);
}

__device__ void gj_solve_reg(const df* S, int q, int nrhs, int lds, GjShared* g, df* sol, int ldsol) {
  const int tid = threadIdx.x;
  const int i = tid >> 5, j = tid & 31;
  const int ncol = q + nrhs;
  const bool live = i < q && j < ncol;
  df v = live ? S[i * lds + j] : df{0.f, 0.f};
  if (tid == 0) g->key[0] = 0ull;
  __syncthreads();
  if (live && j == 0) atomicMax(&g->key[0], pivot_key(fabsf(v.hi), i));
  unsigned used = 0u;
  __syncthreads();
  for (int k = 0; k < q; ++k) {
    const int p = 31 - static_cast<int>(g->key[k & 1] & 0xffffffffull);
    if (i == p) {
      df pk = shfl_df(v, k);
      if (fabsf(pk.hi) < 1.0e-30f) pk = df{1.0e-30f, 0.f};
      v = (j == k) ? df{1.f, 0.f} : df_mul(v, df_recip(pk));
      if (j < ncol) g->prowv[j] = v;
    }
    if (tid == 0) {
      g->key[(k + 1) & 1] = 0ull;
      g->kof[p] = k;
    }
    used |= 1u << p;
    __syncthreads();
    if (i < q && i != p) {
      const df l = shfl_df(v, k);
      if (j < ncol && j > k) {
        v = df_sub(v, df_mul(l, g->prowv[j]));
        if (j == k + 1 && !((used >> i) & 1u)) atomicMax(&g->key[(k + 1) & 1], pivot_key(fabsf(v.hi), i));
      }
    }
    __syncthreads();
  }
  if (live && j >= q) sol[(j - q) * ldsol + g->kof[i]] = v;
  __syncthreads();
}

// Inertia by symmetric elimination without pivoting (LDL^T) of two q x q
// matrices at once (q <= 31, 1024 threads): thread (i, j) keeps element (i, j)
// of both in registers; per step k warp k scales its row by 1 / d_k and
// publishes it, and rows i > k subtract a_ik times it.  Counts the negative
// (or zero) pivots of A into *negs and flags a non-positive pivot of B in
// *nonpd (both shared, initialised by the caller).
struct LdlShared {
  df ra[32], rb[32];
};

__device__ void ldl_inertia_reg(const df* A, const df* B, int q, LdlShared* g, int* negs, int* nonpd) {
  const int tid = threadIdx.x;
  const int i = tid >> 5, j = tid & 31;
  const bool live = i < q && j < q;
  df a = live ? A[i * q + j] : df{0.f, 0.f};
  df b = live ? B[i * q + j] : df{0.f, 0.f};
  for (int k = 0; k < q; ++k) {
    if (i == k) {
      df da = shfl_df(a, k), db = shfl_df(b, k);
      if (j == 0) {
        if (df_lt0(da) || da.hi == 0.f) ++*negs;
        if (!(db.hi > 0.f)) *nonpd = 1;
      }
      if (da.hi == 0.f) da = df{-1.0e-30f, 0.f};
      if (!(db.hi > 0.f)) db = df{1.f, 0.f};
      if (j < q) {
        g->ra[j] = df_mul(a, df_recip(da));
        g->rb[j] = df_mul(b, df_recip(db));
      }
    }
    __syncthreads();
    if (i > k && i < q) {
      const df la = shfl_df(a, k), lb = shfl_df(b, k);
      if (j > k && j < q) {
        a = df_sub(a, df_mul(la, g->ra[j]));
        b = df_sub(b, df_mul(lb, g->rb[j]));
      }
    }
    __syncthreads();
  }
}

__device__ df block_sum_df(df_acc a, df_acc* red, df* out) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a.merge(shfl_xor_acc(a, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x < 32) {
    df_acc b = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : acc_zero();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) b.merge(shfl_xor_acc(b, o));
    if (threadIdx.x == 0) *out = b.value();
  }
  __syncthreads();
  const df r = *out;
  __syncthreads();
  return r;
}

// KB = Z_m^T C (m x 2q, float-float): K = KB[:, :q], B = KB[:, q:].  One block
// per column of C; the block's four thread groups split the d_n-long sums.
template <typename TC>
__global__ void __launch_bounds__(kPenThreads) k_kb(int dn, int m, int q, const float2* __restrict__ Zdf,
                                                    const TC* __restrict__ C, df* __restrict__ KB) {
  extern __shared__ __align__(16) unsigned char kraw[];
  df* col = reinterpret_cast<df*>(kraw);  // dn
  __shared__ df_acc part[4][64];
  const int c = blockIdx.x, tid = threadIdx.x;
  const int q2 = 2 * q;
  for (int l = tid; l < dn; l += blockDim.x) col[l] = to_df(C[static_cast<long long>(l) * q2 + c]);
  __syncthreads();
  const int il = tid & 63, g = tid >> 6;
  for (int i0 = 0; i0 < m; i0 += 64) {
    const int i = i0 + il;
    df_acc a = acc_zero(), a2 = acc_zero();
    if (i < m) {
      int l = g;
      for (; l + 4 < dn; l += 8) {
        a.fma(to_df(Zdf[static_cast<long long>(l) * dn + i]), col[l]);
        a2.fma(to_df(Zdf[static_cast<long long>(l + 4) * dn + i]), col[l + 4]);
      }
      if (l < dn) a.fma(to_df(Zdf[static_cast<long long>(l) * dn + i]), col[l]);
    }
    a.merge(a2);
    part[g][il] = a;
    __syncthreads();
    if (g == 0 && i < m) {
      df_acc s = part[0][il];
      s.merge(part[1][il]);
      s.merge(part[2][il]);
      s.merge(part[3][il]);
      KB[static_cast<long long>(i) * q2 + c] = s.value();
    }
    __syncthreads();
  }
}

// Ft (m x q), Tt, S (q x q), float-float; block a computes column a of Ft and
// row a of Tt and S.  G = [V^T A V | V^T M V] (q x 2q) is symmetrised.
__global__ void __launch_bounds__(kPenThreads) k_blocks(int m, int q, const df* __restrict__ KB,
                                                        const double* __restrict__ G, const double* __restrict__ th,
                                                        df* __restrict__ Ft, df* __restrict__ Tt, df* __restrict__ St) {
  __shared__ df_acc pt[8][32], ps[8][32];
  const int a = blockIdx.x, tid = threadIdx.x;
  const int q2 = 2 * q;
  for (int i = tid; i < m; i += blockDim.x) {
    const df k = KB[static_cast<long long>(i) * q2 + a], b = KB[static_cast<long long>(i) * q2 + q + a];
    Ft[static_cast<long long>(i) * q + a] = df_sub(k, df_mul(to_df(th[i]), b));
  }
  const int lane = tid & 31, g = tid >> 5;
  for (int b0 = 0; b0 < q; b0 += 32) {
    const int b = b0 + lane;
    df_acc at = acc_zero(), as = acc_zero();
    if (b < q)
      for (int i = g; i < m; i += 8) {
        const long long r = static_cast<long long>(i) * q2;
        const df ka = KB[r + a], ba = KB[r + q + a], kb = KB[r + b], bb = KB[r + q + b];
        const df fb = df_sub(kb, df_mul(to_df(th[i]), bb));  // (K - Theta B)_ib
        at.fma(ba, fb);
        at.fma(ka, bb);
        as.fma(ba, bb);
      }
    pt[g][lane] = at;
    ps[g][lane] = as;
    __syncthreads();
    if (g == 0 && b < q) {
      df_acc t = pt[0][lane], s = ps[0][lane];
      for (int h = 1; h < 8; ++h) {
        t.merge(pt[h][lane]);
        s.merge(ps[h][lane]);
      }
      const double ga = 0.5 * (G[a * static_cast<long long>(q2) + b] + G[b * static_cast<long long>(q2) + a]);
      const double gm =
          0.5 * (G[a * static_cast<long long>(q2) + q + b] + G[b * static_cast<long long>(q2) + q + a]);
      Tt[a * q + b] = df_sub(to_df(ga), t.value());
      St[a * q + b] = df_sub(to_df(gm), s.value());
    }
    __syncthreads();
  }
}

// x^T At x for x = [x1; x2] (m + q)
__device__ df pencil_rq(const df* th, const df* F, const df* T, const df* x, int m, int q, df_acc* red, df* out) {
  const int tid = threadIdx.x, nt = blockDim.x;
  df_acc a = acc_zero();
  for (int i = tid; i < m + q; i += nt) {
    if (i < m) {
      const df fx = dot4(F + i * q, 1, x + m, 1, q).value();
      // x1_i (theta_i x1_i + 2 (Ft x2)_i)
      a.fma(x[i], df_add(df_mul(th[i], x[i]), df_add(fx, fx)));
    } else {
      const int r = i - m;
      a.fma(x[i], dot4(T + r * q, 1, x + m, 1, q).value());
    }
  }
  return block_sum_df(a, red, out);
}

// x = y / ||y||_Mt (y is first scaled by a power of two near 1 / max |y_i|).  sy: q scratch.
__device__ void mt_normalise(const df* S, df* y, df* x, df* sy, int m, int q, df_acc* red, df* out) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const int n = m + q;
  float amax = 0.f;
  for (int i = tid; i < n; i += nt) amax = fmaxf(amax, fabsf(y[i].hi));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  __shared__ float wmax[32];
  if ((tid & 31) == 0) wmax[tid >> 5] = amax;
  __syncthreads();
  float gmax = (tid & 31) < (nt >> 5) ? wmax[tid & 31] : 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) gmax = fmaxf(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
  // power-of-two scale keeps the scaling exact
  const float sc = gmax > 0.f ? exp2f(-floorf(log2f(gmax))) : 1.f;
  for (int i = tid; i < n; i += nt) y[i] = df{y[i].hi * sc, y[i].lo * sc};
  __syncthreads();
  for (int a = tid; a < q; a += nt) sy[a] = dot4(S + a * q, 1, y + m, 1, q).value();
  __syncthreads();
  df_acc acc = acc_zero();
  for (int i = tid; i < n; i += nt) acc.fma(y[i], i < m ? y[i] : sy[i - m]);
  const df nrm = df_sqrt(block_sum_df(acc, red, out));
  const df inv = df_recip(nrm);
  for (int i = tid; i < n; i += nt) x[i] = df_mul(y[i], inv);
  __syncthreads();
}

__global__ void __launch_bounds__(kSrqiThreads) k_srqi(int m, int q, const double* __restrict__ thg,
                                                      const df* __restrict__ KB, const df* __restrict__ Ftg,
                                                      const df* __restrict__ Ttg, const df* __restrict__ Stg,
                                                      double* __restrict__ mu, double* __restrict__ X,
                                                      int* __restrict__ conv) {
  extern __shared__ __align__(16) unsigned char sraw[];
  const int n = m + q;
  df* th = reinterpret_cast<df*>(sraw);
  df* dv = th + m;          // m: 1 / (theta_i - s)
  df* F = dv + m;           // m x q
  df* DF = F + m * q;       // m x q: (Theta - s)^-1 Ft
  df* T = DF + m * q;       // q x q
  df* S = T + q * q;        // q x q
  df* Sc = S + q * q;       // q x (q+1)
  df* x = Sc + q * (q + 1); // n
  df* y = x + n;            // n
  df* sx = y + n;           // q
  __shared__ df_acc red[32];
  __shared__ df outv;
  __shared__ int prow[kSrqiMaxQ], used[kSrqiMaxQ];
  __shared__ df ysol[kSrqiMaxQ], rinv;
  __shared__ GjShared gj;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int j = blockIdx.x;
  const int q2 = 2 * q;
  for (int i = tid; i < m; i += nt) th[i] = to_df(thg[i]);
  for (int idx = tid; idx < m * q; idx += nt) F[idx] = Ftg[idx];
  for (int idx = tid; idx < q * q; idx += nt) {
    T[idx] = Ttg[idx];
    S[idx] = Stg[idx];
  }
  // start: column j of V, i.e. [B e_j; e_j]
  for (int i = tid; i < n; i += nt)
    y[i] = i < m ? KB[static_cast<long long>(i) * q2 + q + j] : df{(i - m) == j ? 1.f : 0.f, 0.f};
  __syncthreads();
  mt_normalise(S, y, x, sx, m, q, red, &outv);
  df sg = pencil_rq(th, F, T, x, m, q, red, &outv);
  const df sg0 = sg;  // reported when the iteration fails: it places the pair for the repair
  int ok = 0;
  for (int it = 0; it < kSrqiMaxIt; ++it) {
    // S x2 for the right-hand side
    for (int a = tid; a < q; a += nt) sx[a] = dot4(S + a * q, 1, x + m, 1, q).value();
    for (int i = tid; i < m; i += nt) {
      df d = df_sub(th[i], sg);
      if (fabsf(d.hi) < 1.0e-30f) d = df{1.0e-30f, 0.f};
      dv[i] = df_recip(d);
    }
    __syncthreads();
    for (int idx = tid; idx < m * q; idx += nt) DF[idx] = df_mul(dv[idx / q], F[idx]);
    __syncthreads();
    // Schur complement S(s) (symmetric: upper triangle, mirrored below) and
    // right-hand side S x2 - Ft^T (Theta - s)^-1 x1
    for (int idx = tid; idx < q * (q + 1); idx += nt) {
      const int a = idx / (q + 1), b = idx % (q + 1);
      if (b < a) continue;
      df_acc acc = acc_zero();
      if (b < q) {
        acc.add(T[a * q + b]);
        acc.fma(df_neg(sg), S[a * q + b]);
        acc.add(df_neg(dot4(F + a, q, DF + b, q, m).value()));
      } else {
        acc.add(sx[a]);
        acc.add(df_neg(dot4(DF + a, q, x, 1, m).value()));
      }
      Sc[idx] = acc.value();
    }
    __syncthreads();
    for (int idx = tid; idx < q * q; idx += nt) {
      const int a = idx / q, b = idx % q;
      if (b < a) Sc[a * (q + 1) + b] = Sc[b * (q + 1) + a];
    }
    __syncthreads();
    if (q <= 31 && nt == 1024)
      gj_solve_reg(Sc, q, 1, q + 1, &gj, ysol, q);
    else
      gj_solve(Sc, q, prow, used, &rinv, ysol);
    // y2 = solution, y1 = (Theta - s)^-1 (x1 - Ft y2)
    for (int i = tid; i < n; i += nt) {
      if (i < m) {
        y[i] = df_mul(dv[i], df_sub(x[i], dot4(F + i * q, 1, ysol, 1, q).value()));
      } else {
        y[i] = ysol[i - m];
      }
    }
    __syncthreads();
    mt_normalise(S, y, x, sx, m, q, red, &outv);
    const df sn = pencil_rq(th, F, T, x, m, q, red, &outv);
    const df dlt = df_abs(df_sub(sn, sg));
    sg = sn;
    // RQI converges cubically: a step that moves the quotient by d (relative)
    // started from a vector with angle error ~sqrt(d), so the vector it
    // produced is accurate to ~d^(3/2): d <= 1e-10 gives working precision
    if (it >= 1 && dlt.hi <= 1.0e-10f * fabsf(sn.hi)) {
      ok = it + 1;
      break;
    }
  }
  for (int i = tid; i < n; i += nt) X[i * static_cast<long long>(q) + j] = df_to_double(x[i]);
  if (tid == 0) {
    mu[j] = df_to_double(ok ? sg : sg0);
    conv[j] = ok;  // iterations taken when converged, 0 otherwise
  }
}

// Accept the fast path (flag[0] = 1) or leave it to the dense solver (flag[0] =
// 0).  Vectors of nearly equal values come out of the iteration only accurate
// to residual / gap, and two iterations may even find the same pair; such
// clusters (chains of sorted neighbours whose Mt-overlap exceeds 1e-9, at most
// kMaxCluster vectors) are repaired by Rayleigh-Ritz on the cluster's span --
// after two steps of block inverse iteration from the starting vectors when
// the cluster holds duplicates.  The result is accepted only if every
// iteration converged, all vectors are Mt-orthogonal to 1e-6 afterwards, S is
// positive definite and the inertia count just above the largest value is q.
// On acceptance writes the ascending values to evals and the vectors [a; b]
// ((m + q) x q) to evecs, made Mt-orthonormal to second order by the first-order
// Lowdin correction X (I - E / 2), E = X^T Mt X - I.
constexpr int kMaxCluster = 4;
constexpr int kRepairRounds = 8;
constexpr float kRepairResidual = 1.0e-12f;  // relative residual of a repaired pair

struct CheckShared {
  int okf, negs, nonpd, theta_cnt, nclus;
  int perm[kSrqiMaxQ];
  int cstart[kSrqiMaxQ + 1];  // clusters: members perm[cstart[c] .. cstart[c+1])
  df muS[kSrqiMaxQ];
  df sstar, shift;
  float res;
  float omax;
  int good[kSrqiMaxQ];  // columns accepted so far (the repaired block is kept Mt-orthogonal to them)
  df Ac[kMaxCluster * kMaxCluster], Mc[kMaxCluster * kMaxCluster], Wc[kMaxCluster * kMaxCluster];
  df evc[kMaxCluster];
  GjShared gj;
  LdlShared lsh;
};

// Mt-overlaps Ov = X^T Mt X - I (upper triangle computed, mirrored); omax = max |Ov| off the diagonal
__device__ void check_overlaps(const df* X, const df* SX, df* Ov, int m, int q, CheckShared* c) {
  const int tid = threadIdx.x, nt = blockDim.x;
  if (tid == 0) c->omax = 0.f;
  __syncthreads();
  for (int idx = tid; idx < q * q; idx += nt) {
    const int a = idx / q, b = idx % q;
    if (b < a) continue;
    df_acc s = dot4(X + a, q, X + b, q, m);
    s.merge(dot4(X + m * q + a, q, SX + b, q, q));
    if (a == b) s.add(df{-1.f, 0.f});
    const df v = s.value();
    Ov[a * q + b] = v;
    Ov[b * q + a] = v;
    const float f = fabsf(df_float(v));
    if (a != b) atomicMax(reinterpret_cast<int*>(&c->omax), __float_as_int(f));  // f >= 0 (NaN sorts above)
  }
  __syncthreads();
}

// SX = S X2 for all columns
__device__ void check_sx(const df* S, const df* X, df* SX, int m, int q) {
  for (int idx = threadIdx.x; idx < q * q; idx += blockDim.x) {
    const int a = idx / q, j = idx % q;
    SX[idx] = dot4(S + a * q, 1, X + m * q + j, q, q).value();
  }
  __syncthreads();
}

// Yb (n x c, column stride 1, row stride kMaxCluster) -> AY = At Yb, MY = Mt Yb
__device__ void pencil_apply(const df* th, const df* F, const df* T, const df* S, const df* Yb, df* AY, df* MY,
                             int m, int q, int c) {
  const int n = m + q;
  constexpr int L = kMaxCluster;
  for (int idx = threadIdx.x; idx < n * c; idx += blockDim.x) {
    const int i = idx / c, r = idx % c;
    if (i < m) {
      const df fy = dot4(F + i * q, 1, Yb + m * L + r, L, q).value();
      AY[i * L + r] = df_add(df_mul(th[i], Yb[i * L + r]), fy);
      MY[i * L + r] = Yb[i * L + r];
    } else {
      const int a = i - m;
      df_acc t = dot4(F + a, q, Yb + r, L, m);
      t.merge(dot4(T + a * q, 1, Yb + m * L + r, L, q));
      AY[i * L + r] = t.value();
      MY[i * L + r] = dot4(S + a * q, 1, Yb + m * L + r, L, q).value();
    }
  }
  __syncthreads();
}

// c x c symmetric-definite Rayleigh-Ritz by one thread: M = L L^T, C = L^-1 A L^-T,
// cyclic Jacobi on C (one exact rotation for c = 2), W <- L^-T W; values ascending.
__device__ void small_rr(df* A, df* M, df* W, df* ev, int c) {
  constexpr int L = kMaxCluster;
  // Cholesky of M in place (lower)
  for (int k = 0; k < c; ++k) {
    df d = M[k * L + k];
    for (int t = 0; t < k; ++t) d = df_sub(d, df_mul(M[k * L + t], M[k * L + t]));
    d = df_sqrt(d.hi > 0.f ? d : df{1.0e-30f, 0.f});
    M[k * L + k] = d;
    const df id = df_recip(d);
    for (int i = k + 1; i < c; ++i) {
      df s = M[i * L + k];
      for (int t = 0; t < k; ++t) s = df_sub(s, df_mul(M[i * L + t], M[k * L + t]));
      M[i * L + k] = df_mul(s, id);
    }
  }
  // C = L^-1 A L^-T (A symmetric; rows then columns)
  for (int j = 0; j < c; ++j)
    for (int i = 0; i < c; ++i) {
      df s = A[i * L + j];
      for (int t = 0; t < i; ++t) s = df_sub(s, df_mul(M[i * L + t], A[t * L + j]));
      A[i * L + j] = df_div(s, M[i * L + i]);
    }
  for (int i = 0; i < c; ++i)
    for (int j = 0; j < c; ++j) {
      df s = A[i * L + j];
      for (int t = 0; t < j; ++t) s = df_sub(s, df_mul(M[j * L + t], A[i * L + t]));
      A[i * L + j] = df_div(s, M[j * L + j]);
    }
  for (int i = 0; i < c; ++i)
    for (int j = 0; j < c; ++j) W[i * L + j] = df{i == j ? 1.f : 0.f, 0.f};
  const int sweeps = c == 2 ? 1 : 6;
  for (int sw = 0; sw < sweeps; ++sw)
    for (int p = 0; p < c; ++p)
      for (int r = p + 1; r < c; ++r) {
        const df apr = df_mul_f(df_add(A[p * L + r], A[r * L + p]), 0.5f);
        const df dif = df_sub(A[r * L + r], A[p * L + p]);
        if (fabsf(apr.hi) <= 1.0e-30f * fabsf(dif.hi) || apr.hi == 0.f) continue;
        // t = sign(th) / (|th| + sqrt(th^2 + 1)), th = (a_rr - a_pp) / (2 a_pr);
        // t = 1 / (2 th) once th^2 would leave the float range
        const df th = df_div(dif, df_add(apr, apr));
        df t;
        if (fabsf(th.hi) > 1.0e15f) {
          t = df_recip(df_add(th, th));
        } else {
          const df rt = df_sqrt(df_add(df_mul(th, th), df{1.f, 0.f}));
          t = df_recip(df_add(df_abs(th), rt));
          if (df_lt0(th)) t = df_neg(t);
        }
        const df cs = df_recip(df_sqrt(df_add(df_mul(t, t), df{1.f, 0.f})));
        const df sn = df_mul(t, cs);
        for (int k = 0; k < c; ++k) {  // columns p, r of A
          const df akp = A[k * L + p], akr = A[k * L + r];
          A[k * L + p] = df_sub(df_mul(cs, akp), df_mul(sn, akr));
          A[k * L + r] = df_add(df_mul(sn, akp), df_mul(cs, akr));
        }
        for (int k = 0; k < c; ++k) {  // rows p, r of A
          const df apk = A[p * L + k], ark = A[r * L + k];
          A[p * L + k] = df_sub(df_mul(cs, apk), df_mul(sn, ark));
          A[r * L + k] = df_add(df_mul(sn, apk), df_mul(cs, ark));
        }
        for (int k = 0; k < c; ++k) {
          const df wkp = W[k * L + p], wkr = W[k * L + r];
          W[k * L + p] = df_sub(df_mul(cs, wkp), df_mul(sn, wkr));
          W[k * L + r] = df_add(df_mul(sn, wkp), df_mul(cs, wkr));
        }
      }
  // W <- L^-T W
  for (int j = 0; j < c; ++j)
    for (int i = c - 1; i >= 0; --i) {
      df s = W[i * L + j];
      for (int t = i + 1; t < c; ++t) s = df_sub(s, df_mul(M[t * L + i], W[t * L + j]));
      W[i * L + j] = df_div(s, M[i * L + i]);
    }
  // ascending order (selection sort of columns)
  for (int i = 0; i < c; ++i) ev[i] = A[i * L + i];
  for (int i = 0; i < c; ++i) {
    int b = i;
    for (int j = i + 1; j < c; ++j)
      if (df_lt0(df_sub(ev[j], ev[b]))) b = j;
    if (b != i) {
      const df e = ev[i];
      ev[i] = ev[b];
      ev[b] = e;
      for (int k = 0; k < c; ++k) {
        const df w = W[k * L + i];
        W[k * L + i] = W[k * L + b];
        W[k * L + b] = w;
      }
    }
  }
}

// columns of Yb (n x c, row stride kMaxCluster) scaled by powers of two to max |.| ~ 1
__device__ void block_scale(df* Yb, int n, int c) {
  constexpr int L = kMaxCluster;
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    for (int r = 0; r < c; ++r) {
      float amax = 0.f;
      for (int i = lane; i < n; i += 32) amax = fmaxf(amax, fabsf(Yb[i * L + r].hi));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
      const float sc = amax > 0.f ? exp2f(-floorf(log2f(amax))) : 1.f;
      for (int i = lane; i < n; i += 32) Yb[i * L + r] = df{Yb[i * L + r].hi * sc, Yb[i * L + r].lo * sc};
    }
  }
  __syncthreads();
}

// Yb <- Yb - X_good (X_good^T Mt Yb), twice (the accepted columns of X are
// Mt-orthonormal to working accuracy).  MY, tmp: n x L scratch; coef: q x L.
__device__ void block_deflate(const df* X, const df* S, df* Yb, df* MY, df* tmp, const int* good, df* coef, int m,
                              int q, int c) {
  constexpr int L = kMaxCluster;
  const int n = m + q, tid = threadIdx.x, nt = blockDim.x;
  for (int pass = 0; pass < 2; ++pass) {
    for (int idx = tid; idx < n * c; idx += nt) {
      const int i = idx / c, r = idx % c;
      MY[i * L + r] = i < m ? Yb[i * L + r] : dot4(S + (i - m) * q, 1, Yb + m * L + r, L, q).value();
    }
    __syncthreads();
    for (int idx = tid; idx < q * c; idx += nt) {
      const int j = idx / c, r = idx % c;
      coef[j * L + r] = good[j] ? dot4(X + j, q, MY + r, L, n).value() : df{0.f, 0.f};
    }
    __syncthreads();
    for (int idx = tid; idx < n * c; idx += nt) {
      const int i = idx / c, r = idx % c;
      // skip the other columns outright: an unconverged one may hold NaN
      df_acc a0 = acc_zero(), a1 = acc_zero();
      int j = 0;
      for (; j + 2 <= q; j += 2) {
        if (good[j]) a0.fma(X[i * q + j], coef[j * L + r]);
        if (good[j + 1]) a1.fma(X[i * q + j + 1], coef[(j + 1) * L + r]);
      }
      if (j < q && good[j]) a0.fma(X[i * q + j], coef[j * L + r]);
      a0.merge(a1);
      tmp[i * L + r] = df_sub(Yb[i * L + r], a0.value());
    }
    __syncthreads();
    for (int idx = tid; idx < n * c; idx += nt) Yb[(idx / c) * L + idx % c] = tmp[(idx / c) * L + idx % c];
    __syncthreads();
  }
}

// Mt-orthonormalise the block: G = Yb^T Mt Yb = L L^T, Yb <- Yb L^-T (Cholesky-QR)
__device__ void block_cholqr(const df* th, const df* F, const df* T, const df* S, df* Yb, df* AY, df* MY,
                             CheckShared* c, int m, int q, int cs) {
  constexpr int L = kMaxCluster;
  const int n = m + q, tid = threadIdx.x, nt = blockDim.x;
  for (int idx = tid; idx < n * cs; idx += nt) {
    const int i = idx / cs, r = idx % cs;
    MY[i * L + r] = i < m ? Yb[i * L + r] : dot4(S + (i - m) * q, 1, Yb + m * L + r, L, q).value();
  }
  __syncthreads();
  for (int idx = tid; idx < cs * cs; idx += nt) {
    const int a = idx / cs, b = idx % cs;
    c->Mc[a * L + b] = dot4(Yb + a, L, MY + b, L, n).value();
  }
  __syncthreads();
  if (tid == 0) {
    for (int k = 0; k < cs; ++k) {  // Cholesky in place (lower); L^-T goes to Wc
      df d = c->Mc[k * L + k];
      for (int t = 0; t < k; ++t) d = df_sub(d, df_mul(c->Mc[k * L + t], c->Mc[k * L + t]));
      d = df_sqrt(d.hi > 0.f ? d : df{1.0e-30f, 0.f});
      c->Mc[k * L + k] = d;
      const df id = df_recip(d);
      for (int i = k + 1; i < cs; ++i) {
        df t2 = c->Mc[i * L + k];
        for (int t = 0; t < k; ++t) t2 = df_sub(t2, df_mul(c->Mc[i * L + t], c->Mc[k * L + t]));
        c->Mc[i * L + k] = df_mul(t2, id);
      }
    }
    for (int j = 0; j < cs; ++j)
      for (int i = cs - 1; i >= 0; --i) {
        df t2 = df{i == j ? 1.f : 0.f, 0.f};
        for (int t = i + 1; t < cs; ++t) t2 = df_sub(t2, df_mul(c->Mc[t * L + i], c->Wc[t * L + j]));
        c->Wc[i * L + j] = df_div(t2, c->Mc[i * L + i]);
      }
  }
  __syncthreads();
  for (int idx = tid; idx < n * cs; idx += nt) {
    const int i = idx / cs, r = idx % cs;
    df_acc t2 = acc_zero();
    for (int t = 0; t <= r; ++t) t2.fma(Yb[i * L + t], c->Wc[t * L + r]);
    AY[i * L + r] = t2.value();
  }
  __syncthreads();
  for (int idx = tid; idx < n * cs; idx += nt) Yb[(idx / cs) * L + idx % cs] = AY[(idx / cs) * L + idx % cs];
  __syncthreads();
}

// Largest relative residual ||At y - mu Mt y|| / (|mu| ||Mt y||) of the Ritz pairs
// (Yb W_r, ev_r), r < cs, from AY = At Yb and MY = Mt Yb; one warp per pair.
// Result in *res (shared).
__device__ void ritz_residual(const df* AY, const df* MY, const df* W, const df* ev, int n, int cs, float* res) {
  constexpr int L = kMaxCluster;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) *res = 0.f;
  __syncthreads();
  if (w < cs) {
    float rr = 0.f, mm = 0.f;
    for (int i = lane; i < n; i += 32) {
      df_acc a = acc_zero(), b = acc_zero();
      for (int t = 0; t < cs; ++t) {
        a.fma(AY[i * L + t], W[t * L + w]);
        b.fma(MY[i * L + t], W[t * L + w]);
      }
      const df my = b.value();
      const float e = df_float(df_sub(a.value(), df_mul(ev[w], my)));
      rr = fmaf(e, e, rr);
      mm = fmaf(my.hi, my.hi, mm);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      rr += __shfl_xor_sync(0xffffffffu, rr, o);
      mm += __shfl_xor_sync(0xffffffffu, mm, o);
    }
    if (lane == 0) {
      const float rel = sqrtf(rr) / (fabsf(ev[w].hi) * sqrtf(mm));
      atomicMax(reinterpret_cast<int*>(res), __float_as_int(rel == rel ? rel : 3.0e38f));
    }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kSrqiThreads) k_srqi_check(int m, int q, const double* __restrict__ thg,
                                                            const df* __restrict__ KB, const df* __restrict__ Ftg,
                                                            const df* __restrict__ Ttg, const df* __restrict__ Stg,
                                                            const double* __restrict__ mu,
                                                            const double* __restrict__ Xg,
                                                            const int* __restrict__ conv,
                                                            double* __restrict__ evals, double* __restrict__ evecs,
                                                            int* __restrict__ flag) {
  extern __shared__ __align__(16) unsigned char craw[];
  constexpr int L = kMaxCluster;
  const int n = m + q;
  df* X = reinterpret_cast<df*>(craw);  // n x q
  df* SX = X + n * q;                   // q x q: S X2
  df* Sc = SX + q * q;                  // q x q: S(s*)
  df* Sl = Sc + q * q;                  // q x q: S
  df* Ov = Sl + q * q;                  // q x q: X^T Mt X - I
  df* T = Ov + q * q;                   // q x q: Tt
  df* dv = T + q * q;                   // m: 1 / (theta_i - shift)
  df* th = dv + m;                      // m
  df* F = th + m;                       // m x q
  df* Sa = F + m * q;                   // q x (q + L): augmented Schur complement of the repair
  df* Yb = Sa + q * (q + L);            // n x L
  df* AY = Yb + n * L;                  // n x L
  df* MY = AY + n * L;                  // n x L
  df* ys = MY + n * L;                  // L x q
  __shared__ CheckShared c;
  const int tid = threadIdx.x, nt = blockDim.x;
  if (tid == 0) {
    c.okf = 1;
    c.negs = 0;
    c.nonpd = 0;
  }
  for (int idx = tid; idx < n * q; idx += nt) X[idx] = to_df(Xg[idx]);
  for (int idx = tid; idx < q * q; idx += nt) {
    Sl[idx] = Stg[idx];
    T[idx] = Ttg[idx];
  }
  for (int idx = tid; idx < m * q; idx += nt) F[idx] = Ftg[idx];
  for (int i = tid; i < m; i += nt) th[i] = to_df(thg[i]);
  for (int j = tid; j < q; j += nt) c.muS[j] = to_df(mu[j]);
  __syncthreads();
  check_sx(Sl, X, SX, m, q);
  check_overlaps(X, SX, Ov, m, q, &c);
  // sort by value (a NaN from a diverged iteration sorts last), then chain
  // sorted neighbours with large overlaps into clusters
  for (int j = tid; j < q; j += nt) {
    const double vj = mu[j] == mu[j] ? mu[j] : HUGE_VAL;
    int r = 0;
    for (int i = 0; i < q; ++i) {
      const double vi = mu[i] == mu[i] ? mu[i] : HUGE_VAL;
      if (vi < vj || (vi == vj && i < j)) ++r;
    }
    c.perm[r] = j;
  }
  __syncthreads();
  if (tid == 0) {
    int nc = 0, bad = 0;
    c.cstart[0] = 0;
    for (int r = 1; r <= q; ++r) {
      // an iteration that did not converge joins its sorted neighbours' cluster
      const bool join = r < q && (fabsf(df_float(Ov[c.perm[r - 1] * q + c.perm[r]])) > 1.0e-9f ||
                                  !conv[c.perm[r - 1]] || !conv[c.perm[r]]);
      if (!join) {
        const int size = r - c.cstart[nc];
        if (size > L || (size > 1 && q + size > 32) || (size == 1 && !conv[c.perm[r - 1]])) bad = 1;
        c.cstart[++nc] = r;
      }
    }
    c.nclus = nc;
    if (bad) c.okf = 0;
  }
  __syncthreads();
  if (!c.okf) {
    if (tid == 0) {
      flag[0] = 0;
      flag[1] = 1;  // a cluster larger than kMaxCluster, or an unconverged singleton
    }
    return;
  }
  bool repaired = false;
  for (int r = tid; r < q; r += nt) c.good[r] = 1;
  __syncthreads();
  if (tid == 0)
    for (int cl = 0; cl < c.nclus; ++cl)
      if (c.cstart[cl + 1] - c.cstart[cl] > 1)
        for (int r = c.cstart[cl]; r < c.cstart[cl + 1]; ++r) c.good[c.perm[r]] = 0;
  __syncthreads();
  for (int cl = 0; cl < c.nclus; ++cl) {
    const int c0 = c.cstart[cl], cs = c.cstart[cl + 1] - c0;
    if (cs < 2) continue;
    repaired = true;
    // duplicates (overlap > 0.5) or an unconverged member: restart from the
    // starting vectors [B e_j; e_j]
    bool dup = false;
    for (int r = 0; r < cs; ++r) {
      if (!conv[c.perm[c0 + r]]) dup = true;
      if (r + 1 < cs && fabsf(df_float(Ov[c.perm[c0 + r] * q + c.perm[c0 + r + 1]])) > 0.5f) dup = true;
    }
    for (int idx = tid; idx < n * cs; idx += nt) {
      const int i = idx / cs, r = idx % cs, j = c.perm[c0 + r];
      Yb[i * L + r] = dup ? (i < m ? KB[static_cast<long long>(i) * 2 * q + q + j]
                                   : df{(i - m) == j ? 1.f : 0.f, 0.f})
                          : X[i * q + j];
    }
    __syncthreads();
    if (dup) {
      // the block only has to find what the accepted vectors do not span:
      // project them out (Mt inner product) and re-normalise
      block_deflate(X, Sl, Yb, MY, AY, c.good, ys, m, q, cs);
      block_cholqr(th, F, T, Sl, Yb, AY, MY, &c, m, q, cs);
      // shift: the mean Rayleigh quotient of the block (inside the cluster)
      pencil_apply(th, F, T, Sl, Yb, AY, MY, m, q, cs);
      for (int idx = tid; idx < 2 * cs; idx += nt) {
        const int which = idx / cs, r = idx % cs;
        (which ? c.Mc : c.Ac)[r] = dot4(Yb + r, L, (which ? MY : AY) + r, L, n).value();
      }
      __syncthreads();
      if (tid == 0) {
        df sum = df{0.f, 0.f};
        for (int r = 0; r < cs; ++r) sum = df_add(sum, df_div(c.Ac[r], c.Mc[r]));
        c.shift = df_div(sum, df{static_cast<float>(cs), 0.f});
      }
      __syncthreads();
    }
    // block inverse iteration, the shift moved to the mean Ritz value after each
    // step, until the Ritz values settle (at most kRepairRounds steps)
    bool settled = false;
    for (int round = 0; dup && round < kRepairRounds; ++round) {
      // (At - s Mt) Y = Mt Yb through the Schur complement at s, all columns at
      // once; s sits 2^-30 (relative) off the mean Ritz value so that a cluster
      // of equal values cannot make the solve exactly singular
      const df sh = df_add(c.shift, df_mul_f(df_abs(c.shift), 9.313225746154785e-10f));
      for (int i = tid; i < m; i += nt) {
        df d = df_sub(th[i], sh);
        if (fabsf(d.hi) < 1.0e-30f) d = df{1.0e-30f, 0.f};
        dv[i] = df_recip(d);
      }
      __syncthreads();
      for (int idx = tid; idx < q * (q + cs); idx += nt) {
        const int a = idx / (q + cs), b = idx % (q + cs);
        df_acc acc = acc_zero();
        if (b < q) {
          acc.add(T[a * q + b]);
          acc.fma(df_neg(sh), Sl[a * q + b]);
          acc.add(df_neg(dot4w(F + a, q, dv, F + b, q, m).value()));
        } else {
          const int r = b - q;
          acc.add(dot4(Sl + a * q, 1, Yb + m * L + r, L, q).value());
          acc.add(df_neg(dot4w(F + a, q, dv, Yb + r, L, m).value()));
        }
        Sa[a * (q + L) + b] = acc.value();
      }
      __syncthreads();
      gj_solve_reg(Sa, q, cs, q + L, &c.gj, ys, q);
      for (int idx = tid; idx < n * cs; idx += nt) {
        const int i = idx / cs, r = idx % cs;
        Yb[i * L + r] = i < m ? df_mul(dv[i], df_sub(Yb[i * L + r], dot4(F + i * q, 1, ys + r * q, 1, q).value()))
                              : ys[r * q + (i - m)];
      }
      __syncthreads();
      block_scale(Yb, n, cs);
      block_deflate(X, Sl, Yb, MY, AY, c.good, ys, m, q, cs);
      block_cholqr(th, F, T, Sl, Yb, AY, MY, &c, m, q, cs);
      pencil_apply(th, F, T, Sl, Yb, AY, MY, m, q, cs);
      for (int idx = tid; idx < 2 * cs * cs; idx += nt) {
        const int which = idx / (cs * cs), e = idx % (cs * cs), a = e / cs, b = e % cs;
        const df v = dot4(Yb + a, L, (which ? MY : AY) + b, L, n).value();
        (which ? c.Mc : c.Ac)[a * L + b] = v;
      }
      __syncthreads();
      if (tid == 0) {
        small_rr(c.Ac, c.Mc, c.Wc, c.evc, cs);
        df sum = df{0.f, 0.f};
        for (int r = 0; r < cs; ++r) sum = df_add(sum, c.evc[r]);
        c.shift = df_div(sum, df{static_cast<float>(cs), 0.f});
      }
      __syncthreads();
      ritz_residual(AY, MY, c.Wc, c.evc, n, cs, &c.res);
      if (c.res <= kRepairResidual) {
        settled = true;
        break;
      }
    }
    // Rayleigh-Ritz on span(Yb); a block that settled in its last round holds
    // it already (Wc, evc and res of this Yb)
    if (!settled) {
      pencil_apply(th, F, T, Sl, Yb, AY, MY, m, q, cs);
      for (int idx = tid; idx < 2 * cs * cs; idx += nt) {
        const int which = idx / (cs * cs), e = idx % (cs * cs), a = e / cs, b = e % cs;
        const df v = dot4(Yb + a, L, (which ? MY : AY) + b, L, n).value();
        (which ? c.Mc : c.Ac)[a * L + b] = v;
      }
      __syncthreads();
      if (tid == 0) small_rr(c.Ac, c.Mc, c.Wc, c.evc, cs);
      __syncthreads();
      ritz_residual(AY, MY, c.Wc, c.evc, n, cs, &c.res);
    }
    // the repaired pairs must be eigenpairs of the pencil to working accuracy
    if (!(c.res <= kRepairResidual)) {
      if (tid == 0) {
        flag[0] = 0;
        flag[1] = 5;  // a cluster repair did not converge
        flag[2] = __float_as_int(c.res);
        flag[3] = cs;
      }
      return;
    }
    // new vectors Yb W into the cluster's columns (in the cluster's sorted order)
    for (int idx = tid; idx < n * cs; idx += nt) {
      const int i = idx / cs, r = idx % cs, j = c.perm[c0 + r];
      df_acc s2 = acc_zero();
      for (int t = 0; t < cs; ++t) s2.fma(Yb[i * L + t], c.Wc[t * L + r]);
      X[i * q + j] = s2.value();
    }
    for (int r = tid; r < cs; r += nt) {
      c.muS[c.perm[c0 + r]] = c.evc[r];
      c.good[c.perm[c0 + r]] = 1;
    }
    __syncthreads();
  }
  if (repaired) {
    check_sx(Sl, X, SX, m, q);
    check_overlaps(X, SX, Ov, m, q, &c);
  }
  if (!(c.omax <= 1.0e-6f)) {  // also rejects NaN
    if (tid == 0) {
      flag[0] = 0;
      flag[1] = 2;  // vectors not orthogonal after the cluster repairs
      int ba = 0, bb = 0;
      float bv = -1.f;
      for (int a = 0; a < q && bv == bv; ++a)
        for (int b = a + 1; b < q; ++b) {
          const float v = fabsf(df_float(Ov[a * q + b]));
          if (!(v <= bv)) {
            bv = v;
            ba = a;
            bb = b;
            if (v != v) break;  // the first NaN
          }
        }
      flag[2] = ba * 64 + bb;  // the worst pair
      flag[3] = __float_as_int(bv);
    }
    return;
  }
  // inertia just above the largest value
  if (tid == 0) {
    df mx = c.muS[0];
    for (int i = 1; i < q; ++i)
      if (df_lt0(df_sub(mx, c.muS[i]))) mx = c.muS[i];
    c.sstar = df_add(mx, df_mul_f(df_abs(mx), 1.0e-9f));
  }
  __syncthreads();
  if (tid < 32) {
    int cnt = 0;
    for (int i = tid; i < m; i += 32) cnt += df_lt0(df_sub(th[i], c.sstar));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if (tid == 0) c.theta_cnt = cnt;
  }
  for (int i = tid; i < m; i += nt) {
    df d = df_sub(th[i], c.sstar);
    if (fabsf(d.hi) < 1.0e-30f) d = df{-1.0e-30f, 0.f};
    dv[i] = df_recip(d);
  }
  __syncthreads();
  for (int idx = tid; idx < q * q; idx += nt) {
    const int a = idx / q, b = idx % q;
    if (b < a) continue;
    df_acc acc = acc_zero();
    acc.add(T[idx]);
    acc.fma(df_neg(c.sstar), Sl[idx]);
    acc.add(df_neg(dot4w(F + a, q, dv, F + b, q, m).value()));
    Sc[idx] = acc.value();
  }
  __syncthreads();
  for (int idx = tid; idx < q * q; idx += nt) {
    const int a = idx / q, b = idx % q;
    if (b < a) Sc[idx] = Sc[b * q + a];
  }
  __syncthreads();
  // LDL^T of S(s*) (negative pivots) and of S (must be positive definite)
  if (q <= 31 && nt == 1024)
    ldl_inertia_reg(Sc, Sl, q, &c.lsh, &c.negs, &c.nonpd);
  else
    for (int k = 0; k < q; ++k) {
      const df pc = Sc[k * q + k], pl = Sl[k * q + k];
      if (tid == 0) {
        if (df_lt0(pc) || pc.hi == 0.f) ++c.negs;
        if (!(pl.hi > 0.f)) c.nonpd = 1;
      }
      const df ic = df_recip((pc.hi == 0.f) ? df{-1.0e-30f, 0.f} : pc);
      const df il = df_recip((pl.hi > 0.f) ? pl : df{1.f, 0.f});
      const int r = q - k - 1;
      __syncthreads();
      for (int idx = tid; idx < 2 * r * r; idx += nt) {
        const int which = idx / (r * r), e = idx % (r * r);
        const int i = k + 1 + e / r, jj = k + 1 + e % r;
        df* Mx = which ? Sl : Sc;
        const df fac = df_mul(Mx[i * q + k], which ? il : ic);
        Mx[i * q + jj] = df_sub(Mx[i * q + jj], df_mul(fac, Mx[k * q + jj]));
      }
      __syncthreads();
    }
  __syncthreads();
  if (c.nonpd || c.theta_cnt + c.negs != q) {
    if (tid == 0) {
      flag[0] = 0;
      flag[1] = c.nonpd ? 3 : 4;  // S not positive definite / not the q smallest
      flag[2] = c.theta_cnt + c.negs;
      flag[3] = q;
    }
    return;
  }
  // final order by the (possibly repaired) values
  for (int j = tid; j < q; j += nt) {
    int r = 0;
    for (int i = 0; i < q; ++i) {
      const df d = df_sub(c.muS[i], c.muS[j]);
      if (df_lt0(d) || (d.hi == 0.f && d.lo == 0.f && i < j)) ++r;
    }
    c.perm[r] = j;  // all values are finite here (the overlap test rejects NaN)
  }
  __syncthreads();
  for (int r = tid; r < q; r += nt) evals[r] = df_to_double(c.muS[c.perm[r]]);
  for (int idx = tid; idx < n * q; idx += nt) {
    const int i = idx / q, r = idx % q, b = c.perm[r];
    const df corr = dot4(X + i * q, 1, Ov + b, q, q).value();
    evecs[idx] = df_to_double(df_sub(X[i * q + b], df{0.5f * corr.hi, 0.5f * corr.lo}));
  }
  if (tid == 0) {
    flag[0] = 1;
    flag[1] = 0;
  }
}

// Column solves of the standard form: one warp per right-hand side, row i = lane + 32 r in slot r of the
// lane's registers (q <= 128: four slots).  Each step's solved entry goes to the warp by a shuffle and every
// remaining row takes its product at once, so a step costs one dependent multiply, shuffle and compensated
// product (~100 cycles) instead of a dot product per row and a division (multiplication by 1 / l_kk instead).
constexpr int kStdSlots = kStdMaxQ / 32;

// x = L^-1 acc, forward; L (row stride ld, shared), dinv = 1 / diag(L)
__device__ __forceinline__ void warp_solve_lower(const df* L, int ld, const df* dinv, int q, df_acc* acc, df* x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 0; s < kStdSlots; ++s) {
    if (32 * s >= q) break;
    const int ke = min(q - 32 * s, 32);
    for (int t = 0; t < ke; ++t) {
      const int k = 32 * s + t;
      const df xk = shfl_df(df_mul(acc[s].value(), dinv[k]), t);
      if (lane == t) x[s] = xk;
      const df nx = df_neg(xk);
#pragma unroll
      for (int r = s; r < kStdSlots; ++r) {
        const int i = lane + 32 * r;
        if (i > k && i < q) acc[r].fma(L[i * ld + k], nx);
      }
    }
  }
}

// x = L^-T acc, backward
__device__ __forceinline__ void warp_solve_upper(const df* L, int ld, const df* dinv, int q, df_acc* acc, df* x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = kStdSlots - 1; s >= 0; --s) {
    if (32 * s >= q) continue;
    for (int t = min(q - 32 * s, 32) - 1; t >= 0; --t) {
      const int k = 32 * s + t;
      const df xk = shfl_df(df_mul(acc[s].value(), dinv[k]), t);
      if (lane == t) x[s] = xk;
      const df nx = df_neg(xk);
#pragma unroll
      for (int r = 0; r <= s; ++r) {
        const int i = lane + 32 * r;
        if (i < k) acc[r].fma(L[k * ld + i], nx);
      }
    }
  }
}

// Fallback: H = [[Theta, Ft L^-T], [L^-1 Ft^T, L^-1 Tt L^-T]] with S = L L^T
// (float-float Cholesky; status = ENOTSPD when S is not positive definite), by
// one cluster.  Every CTA factors S for itself in its own shared memory (square-root
// free, one barrier per column: each thread scales by the reciprocal pivot it
// forms itself; the columns are scaled by 1 / sqrt(d) at the end), which costs
// less than sending the factor around; the m + q columns of L^-1 [Ft^T | Tt] and
// then the q columns of L^-1 (L^-1 Tt)^T are solved one warp each over all the
// CTAs, with a cluster barrier in between.  Bound by the latency of the two chains
// of q steps.  At m = q = 128 the standard form, back-map and Xc took 3.74 ms of the
// pencil's 6.6 ms as one block with one thread per column (2.54 + 0.66 + 2 x 0.27 ms
// of single launches); the pencil is 2.94 ms shorter in this form (0.93 ms at m = 112,
// q = 72).
constexpr int kStdCluster = 8;
constexpr int kStdThreads = 1024;

__global__ void __launch_bounds__(kStdThreads) k_std_form(int m, int q, const double* __restrict__ thg,
                                                          const df* __restrict__ Ft, const df* __restrict__ Tt,
                                                          const df* __restrict__ St, df* __restrict__ L, df* Xs,
                                                          double* H, int* status, const int* skip, int* nfallback) {
  if (skip && *skip) return;  // every CTA of the cluster returns here alike
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = static_cast<int>(cl.block_rank()), CS = static_cast<int>(cl.num_blocks());
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  if (rank == 0 && tid == 0 && nfallback) atomicAdd(nfallback, 1);
  extern __shared__ __align__(16) unsigned char fraw[];
  const int ld = q | 1;                      // odd row stride: column walks hit different banks
  df* A = reinterpret_cast<df*>(fraw);       // q x ld
  df* dinv = A + q * ld;                     // q: 1 / sqrt(d), then 1 / l_kk
  const long long N = m + q;
  for (int idx = tid; idx < q * q; idx += nt) A[(idx / q) * ld + idx % q] = St[idx];
  __syncthreads();
  int bad = 0;
  for (int k = 0; k < q; ++k) {
    df d = A[k * ld + k];
    if (!(d.hi > 0.f)) {
      bad = 1;
      break;  // the same value in every thread of every CTA
    }
    const df rinv = df_recip(d);
    for (int j0 = k + 1; j0 < q; j0 += 32) {
      const int j = j0 + lane;
      const df lj = j < q ? df_mul(A[j * ld + k], rinv) : df{0.f, 0.f};
      for (int i = j0 + warp; i < q; i += nw)
        if (j <= i) A[i * ld + j] = df_sub(A[i * ld + j], df_mul(A[i * ld + k], lj));
    }
    __syncthreads();
  }
  if (bad) {
    if (rank == 0 && tid == 0 && status) status[0] = AMGEIG_ENOTSPD;
    return;
  }
  for (int k = tid; k < q; k += nt) dinv[k] = df_div(df{1.f, 0.f}, df_sqrt(A[k * ld + k]));
  __syncthreads();
  for (int idx = tid; idx < q * q; idx += nt) {
    const int i = idx / q, j = idx % q;
    if (j > i) continue;
    const df l = df_mul(A[i * ld + j], dinv[j]);  // d_j / sqrt(d_j) on the diagonal
    A[i * ld + j] = l;
    if (rank == 0) L[idx] = l;
  }
  __syncthreads();
  for (int k = tid; k < q; k += nt) dinv[k] = df_div(df{1.f, 0.f}, A[k * ld + k]);
  __syncthreads();
  df x[kStdSlots];
  df_acc acc[kStdSlots];
  for (int c = rank * nw + warp; c < m + q; c += CS * nw) {
#pragma unroll
    for (int r = 0; r < kStdSlots; ++r) {
      const int i = lane + 32 * r;
      acc[r] = acc_zero();
      if (i < q) acc[r].add(c < q ? Tt[i * q + c] : Ft[(c - q) * q + i]);
    }
    warp_solve_lower(A, ld, dinv, q, acc, x);
    if (c < q) {
#pragma unroll
      for (int r = 0; r < kStdSlots; ++r)
        if (lane + 32 * r < q) Xs[c * q + lane + 32 * r] = x[r];  // column c of L^-1 Tt
    } else {
      const int row = c - q;
#pragma unroll
      for (int r = 0; r < kStdSlots; ++r) {
        const int i = lane + 32 * r;
        if (i < q) {
          const double v = df_to_double(x[r]);
          H[row * N + m + i] = v;
          H[(m + i) * N + row] = v;
        }
      }
      for (int i = lane; i < m; i += 32) H[row * N + i] = i == row ? thg[row] : 0.0;
    }
  }
  cl.sync();  // L^-1 Tt is complete
  for (int c = rank * nw + warp; c < q; c += CS * nw) {
#pragma unroll
    for (int r = 0; r < kStdSlots; ++r) {
      const int i = lane + 32 * r;
      acc[r] = acc_zero();
      if (i < q) acc[r].add(Xs[i * q + c]);
    }
    warp_solve_lower(A, ld, dinv, q, acc, x);
#pragma unroll
    for (int r = 0; r < kStdSlots; ++r)
      if (lane + 32 * r < q) H[(m + lane + 32 * r) * N + m + c] = df_to_double(x[r]);
  }
  cl.sync();  // the lower right block is complete: symmetrised in place, one thread per pair
  for (int idx = rank * nt + tid; idx < q * q; idx += CS * nt) {
    const int a = idx / q, b = idx % q;
    if (b <= a) continue;
    const double v = 0.5 * (H[(m + a) * N + m + b] + H[(m + b) * N + m + a]);
    H[(m + a) * N + m + b] = v;
    H[(m + b) * N + m + a] = v;
  }
}

// Fallback back-map: b = L^-T b_std in place for the p wanted columns of evecs ((m + q) x p; L is the
// border's q x q factor), one warp per column.
constexpr int kBackWarps = 8;

__global__ void __launch_bounds__(32 * kBackWarps) k_std_back(int m, int q, int p, const df* __restrict__ L,
                                                              double* __restrict__ evecs, const int* skip) {
  if (skip && *skip) return;
  extern __shared__ __align__(16) unsigned char braw[];
  df* Ls = reinterpret_cast<df*>(braw);  // q x q (rows are read along them: no padding needed)
  df* dinv = Ls + q * q;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  for (int idx = tid; idx < q * q; idx += nt)
    if (idx % q <= idx / q) Ls[idx] = L[idx];
  for (int k = tid; k < q; k += nt) dinv[k] = df_div(df{1.f, 0.f}, L[k * q + k]);
  __syncthreads();
  const int c = blockIdx.x * kBackWarps + (tid >> 5);
  if (c >= p) return;
  df x[kStdSlots];
  df_acc acc[kStdSlots];
#pragma unroll
  for (int r = 0; r < kStdSlots; ++r) {
    const int i = lane + 32 * r;
    acc[r] = acc_zero();
    if (i < q) acc[r].add(to_df(evecs[(m + i) * static_cast<long long>(p) + c]));
  }
  warp_solve_upper(Ls, q, dinv, q, acc, x);
#pragma unroll
  for (int r = 0; r < kStdSlots; ++r) {
    const int i = lane + 32 * r;
    if (i < q) evecs[(m + i) * static_cast<long long>(p) + c] = df_to_double(x[r]);
  }
}

// Xc = Z_m (a - B b) (d_n x p, also as float-float pairs in Xc2 when non-null) and Y = b (q x p) from
// evecs = [a; b].  Block (x, y) takes kXcCols columns and the y-th of gridDim.y runs of rows: it stages b, forms
// a - B b in shared memory and then its rows of the product.  Bound by the latency of the loads of B and Z_m,
// so the rows are split over as many blocks as make 128 in all: a - B b is cheap to form again per run, and one block per
// column pair for all rows left narrow borders on one to fourteen SMs.  Launch times on 287 coarse rows at
// 1, 6, 14 and 28 columns, all rows in one run -> split: m = 64 15.5, 23.7, 24.8, 23.8 -> 9.6, 10.8, 12.7, 13.9 us;
// m = 287 49.9, 85.4, 87, 83.5 -> 25.5, 32.4, 39.7, 44.1 us.
// q: the border (columns of V), p: the pairs (columns of evecs, Xc and Y).
constexpr int kXcCols = 2;
constexpr int kXcThreads = 256;
constexpr int kXcBlocks = 128;  // blocks the rows are split for
constexpr int kXcRows = 4;      // rows of a run at least

__global__ void __launch_bounds__(kXcThreads) k_xc(int dn, int m, int q, int p, const float2* __restrict__ Zdf,
                                                   const df* __restrict__ KB, const double* __restrict__ evecs,
                                                   double* __restrict__ Xc, float2* __restrict__ Xc2,
                                                   double* __restrict__ Y) {
  extern __shared__ __align__(16) unsigned char xraw[];
  const int j0 = blockIdx.x * kXcCols, qc = min(kXcCols, p - j0);
  const int rows = (dn + gridDim.y - 1) / gridDim.y, l0 = blockIdx.y * rows, l1 = min(dn, l0 + rows);
  df* bs = reinterpret_cast<df*>(xraw);  // q x kXcCols: b[:, j0:j0+qc]
  df* tmp = bs + q * kXcCols;            // m x kXcCols
  const int tid = threadIdx.x, nt = blockDim.x;
  const int q2 = 2 * q;
  for (int idx = tid; idx < q * qc; idx += nt) {
    const int r = idx / qc, jj = idx % qc;
    const double v = evecs[static_cast<long long>(m + r) * p + j0 + jj];
    bs[r * kXcCols + jj] = to_df(v);
    if (blockIdx.y == 0) Y[r * p + j0 + jj] = v;
  }
  __syncthreads();
  for (int idx = tid; idx < m * qc; idx += nt) {
    const int i = idx / qc, jj = idx % qc;
    const df* Bi = KB + static_cast<long long>(i) * q2 + q;
    // the four-accumulator dot of dot4, unrolled so that the loads of B's row
    // (L2) are in flight together
    df_acc c0 = acc_zero(), c1 = acc_zero(), c2 = acc_zero(), c3 = acc_zero();
    int t = 0;
#pragma unroll 4
    for (; t + 4 <= q; t += 4) {
      c0.fma(Bi[t], bs[t * kXcCols + jj]);
      c1.fma(Bi[t + 1], bs[(t + 1) * kXcCols + jj]);
      c2.fma(Bi[t + 2], bs[(t + 2) * kXcCols + jj]);
      c3.fma(Bi[t + 3], bs[(t + 3) * kXcCols + jj]);
    }
    for (; t < q; ++t) c0.fma(Bi[t], bs[t * kXcCols + jj]);
    c0.merge(c1);
    c2.merge(c3);
    c0.merge(c2);
    tmp[i * kXcCols + jj] = df_sub(to_df(evecs[static_cast<long long>(i) * p + j0 + jj]), c0.value());
  }
  __syncthreads();
  for (int idx = tid; idx < (l1 - l0) * qc; idx += nt) {
    const int l = l0 + idx / qc, jj = idx % qc;
    const float2* zl = Zdf + static_cast<long long>(l) * dn;
    df_acc s0 = acc_zero(), s1 = acc_zero();
    int i = 0;
#pragma unroll 8
    for (; i + 2 <= m; i += 2) {  // unrolled: the row's loads (L2) in flight together
      s0.fma(to_df(zl[i]), tmp[i * kXcCols + jj]);
      s1.fma(to_df(zl[i + 1]), tmp[(i + 1) * kXcCols + jj]);
    }
    if (i < m) s0.fma(to_df(zl[i]), tmp[i * kXcCols + jj]);
    s0.merge(s1);
    const df v = s0.value();
    Xc[static_cast<long long>(l) * p + j0 + jj] = df_to_double(v);
    if (Xc2) Xc2[static_cast<long long>(l) * p + j0 + jj] = make_float2(v.hi, v.lo);
  }
}

// ------------------------------------------------------------ small FP64 kernels

// Float64 Cholesky A = L L^T (row-major, L lower, zero above) of the
// symmetric part of A, right-looking in panels of 32 columns so that the work
// spreads over many blocks (float64 runs at a fraction of the float32 rate):
// per panel the 32 x 32 diagonal block is factored by one block, the rows
// below it solve x L11^T = a one thread each, and the trailing lower triangle
// takes the rank-32 update in 32 x 32 tiles, one block each.  A pivot <= 0
// sets *status = ENOTSPD (and is replaced by 1 so the factorisation finishes).
constexpr int kCb = 32;

__global__ void k_sym_lower(int n, const double* __restrict__ A, double* __restrict__ L) {
  const long long N = n;
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < N * N;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int r = static_cast<int>(i / N), c = static_cast<int>(i % N);
    L[i] = (c <= r) ? 0.5 * (A[r * N + c] + A[c * N + r]) : 0.0;
  }
}

__global__ void __launch_bounds__(1024) k_chol_diag(int n, int j0, int nb, double* __restrict__ L, int* status) {
  __shared__ double T[kCb][kCb + 1];
  __shared__ int bad;
  const int tid = threadIdx.x;
  const long long N = n;
  for (int e = tid; e < nb * nb; e += blockDim.x) {
    const int i = e / nb, j = e % nb;
    T[i][j] = j <= i ? L[(j0 + i) * N + j0 + j] : 0.0;
  }
  if (tid == 0) bad = 0;
  __syncthreads();
  for (int k = 0; k < nb; ++k) {
    if (tid == 0) {
      const double d = T[k][k];
      if (!(d > 0.0)) {
        bad = 1;
        T[k][k] = 1.0;
      } else {
        T[k][k] = sqrt(d);
      }
    }
    __syncthreads();
    if (tid > k && tid < nb) T[tid][k] /= T[k][k];
    __syncthreads();
    const int m = nb - k - 1;
    if (tid < m * m) {
      const int i = k + 1 + tid / m, j = k + 1 + tid % m;
      if (j <= i) T[i][j] -= T[i][k] * T[j][k];
    }
    __syncthreads();
  }
  for (int e = tid; e < nb * nb; e += blockDim.x) {
    const int i = e / nb, j = e % nb;
    if (j <= i) L[(j0 + i) * N + j0 + j] = T[i][j];
  }
  if (tid == 0 && bad && status) status[0] = AMGEIG_ENOTSPD;
}

__global__ void __launch_bounds__(128) k_chol_panel(int n, int j0, int nb, double* __restrict__ L) {
  __shared__ double T[kCb][kCb + 1];
  const long long N = n;
  for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
    const int i = e / nb, j = e % nb;
    T[i][j] = L[(j0 + i) * N + j0 + j];
  }
  __syncthreads();
  const long long r = j0 + nb + blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (r >= n) return;
  double x[kCb];
#pragma unroll
  for (int j = 0; j < kCb; ++j) x[j] = j < nb ? L[r * N + j0 + j] : 0.0;
#pragma unroll
  for (int j = 0; j < kCb; ++j) {
    if (j < nb) {
      double s = x[j];
#pragma unroll
      for (int t = 0; t < j; ++t) s -= x[t] * T[j][t];
      x[j] = s / T[j][j];
    }
  }
#pragma unroll
  for (int j = 0; j < kCb; ++j)
    if (j < nb) L[r * N + j0 + j] = x[j];
}

// lower-triangle tile (ti, tj), tj <= ti, of the trailing block from the block index
__global__ void __launch_bounds__(256) k_chol_syrk(int n, int j0, int nb, double* __restrict__ L) {
  __shared__ double Ai[kCb][kCb + 1], Aj[kCb][kCb + 1];
  int ti = 0;
  while ((ti + 1) * (ti + 2) / 2 <= static_cast<int>(blockIdx.x)) ++ti;
  const int tj = blockIdx.x - ti * (ti + 1) / 2;
  const int base = j0 + nb, i0 = base + ti * kCb, c0 = base + tj * kCb;
  const long long N = n;
  for (int e = threadIdx.x; e < kCb * kCb; e += blockDim.x) {
    const int r = e / kCb, t = e % kCb;
    Ai[r][t] = (i0 + r < n && t < nb) ? L[(i0 + r) * N + j0 + t] : 0.0;
    Aj[r][t] = (c0 + r < n && t < nb) ? L[(c0 + r) * N + j0 + t] : 0.0;
  }
  __syncthreads();
  const int r = threadIdx.x / 8, cb = (threadIdx.x % 8) * 4;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 8
  for (int t = 0; t < kCb; ++t) {
    const double a = Ai[r][t];
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[e] = fma(a, Aj[cb + e][t], acc[e]);
  }
  const int i = i0 + r;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int j = c0 + cb + e;
    if (i < n && j < n && j <= i) L[i * N + j] -= acc[e];
  }
}

void launch_chol_f64(int n, const double* A, double* L, int* status, cudaStream_t st) {
  k_sym_lower<<<ceil_div(static_cast<long long>(n) * n, 256), 256, 0, st>>>(n, A, L);
  for (int j0 = 0; j0 < n; j0 += kCb) {
    const int nb = std::min(kCb, n - j0), rest = n - j0 - nb;
    k_chol_diag<<<1, 1024, 0, st>>>(n, j0, nb, L, status);
    if (rest > 0) {
      k_chol_panel<<<ceil_div(rest, 128), 128, 0, st>>>(n, j0, nb, L);
      const int T = ceil_div(rest, kCb);
      k_chol_syrk<<<T * (T + 1) / 2, 256, 0, st>>>(n, j0, nb, L);
    }
  }
}

int chol_launches(int n) {
  int c = 1;
  for (int j0 = 0; j0 < n; j0 += kCb) c += (n - j0 > kCb) ? 3 : 1;
  return c;
}

// L Y = X in place on ncols columns of the row-major n x ld block X, blocked by 32 rows: rows
// b0 .. b0+31 first take X[b0..] -= L[b0.., 0..b0) X[0..b0) (a float64 product over many blocks), then
// the 32 x 32 diagonal triangle is solved one thread per column (kernel below).
__global__ void __launch_bounds__(128) k_trsm_diag(int n, int b0, int nb, const double* __restrict__ L,
                                                   double* __restrict__ X, int ld, int ncols) {
  __shared__ double T[kCb][kCb + 1];
  const long long N = n, LDX = ld;
  for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
    const int i = e / nb, j = e % nb;
    T[i][j] = j <= i ? L[(b0 + i) * N + b0 + j] : 0.0;
  }
  __syncthreads();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncols) return;
  double x[kCb];
#pragma unroll
  for (int r = 0; r < kCb; ++r) x[r] = r < nb ? X[(b0 + r) * LDX + c] : 0.0;
#pragma unroll
  for (int r = 0; r < kCb; ++r) {
    if (r < nb) {
      double s = x[r];
#pragma unroll
      for (int t = 0; t < r; ++t) s -= T[r][t] * x[t];
      x[r] = s / T[r][r];
    }
  }
#pragma unroll
  for (int r = 0; r < kCb; ++r)
    if (r < nb) X[(b0 + r) * LDX + c] = x[r];
}

void launch_trsm_lower(int n, const double* L, double* X, int ld, int ncols, cudaStream_t st) {
  for (int b0 = 0; b0 < n; b0 += kCb) {
    const int nb = std::min(kCb, n - b0);
    if (b0 > 0)
      launch_gemm_f64(nb, ncols, b0, -1.0, L + static_cast<long long>(b0) * n, n, false, X, ld, false, 1.0,
                      X + static_cast<long long>(b0) * ld, ld, st);
    k_trsm_diag<<<ceil_div(ncols, 128), 128, 0, st>>>(n, b0, nb, L, X, ld, ncols);
  }
}

__global__ void k_transpose_sym(int n, const double* __restrict__ X, double* __restrict__ Y) {
  // Y = 0.5 (X + X^T)
  const long long N = n;
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < N * N;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int r = static_cast<int>(i / N), c = static_cast<int>(i % N);
    Y[i] = 0.5 * (X[r * N + c] + X[c * N + r]);
  }
}

__global__ void k_identity(int n, double* __restrict__ X) {
  const long long N = n;
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < N * N;
       i += static_cast<long long>(gridDim.x) * blockDim.x)
    X[i] = (i / N == i % N) ? 1.0 : 0.0;
}

}  // namespace

// ------------------------------------------------------------ host side

size_t pencil_work_bytes(int dn, int qmax) {
  PencilWork* w = pencil_work_create(dn, qmax, nullptr, true);
  const size_t b = w ? w->bytes : 0;
  pencil_work_destroy(w);
  return b;
}

PencilWork* pencil_work_create(int dn, int qmax, cudaError_t* err, bool dry) {
  auto* w = new PencilWork();
  w->dn = dn;
  w->qmax = qmax;
  w->nmax = dn + qmax;
  w->nwant_max = dn > qmax ? dn : qmax;
  const long long nm = w->nmax;
  const long long nwm = w->nwant_max;
  // two passes over the same list: sizes (256-byte aligned) into one allocation,
  // then the arrays' places in it
  size_t total = 0;
  char* at = nullptr;
  auto alloc = [&](void** p, size_t bytes) {
    const size_t b = ((bytes > 0 ? bytes : 8) + 255) / 256 * 256;
    if (at) {
      *p = at;
      at += b;
    } else {
      total += b;
    }
  };
  for (int pass = 0; pass < 2; ++pass) {
    if (pass == 1) {
      w->bytes = total;
      if (dry) return w;
      cudaError_t e = dev_alloc(&w->base, total);
      if (err) *err = e;
      if (e != cudaSuccess) {
        w->base = nullptr;
        pencil_work_destroy(w);
        return nullptr;
      }
      at = static_cast<char*>(w->base);
    }
    alloc((void**)&w->KB, sizeof(df) * dn * 2 * qmax);
    alloc((void**)&w->Ft, sizeof(df) * dn * qmax);
    alloc((void**)&w->Tt, sizeof(df) * qmax * qmax);
    alloc((void**)&w->St, sizeof(df) * qmax * qmax);
    alloc((void**)&w->Lq, sizeof(df) * qmax * qmax);
    alloc((void**)&w->Xq, sizeof(df) * qmax * qmax);
    alloc((void**)&w->H, sizeof(double) * nm * nm);
    alloc((void**)&w->Yh, sizeof(double) * nm * nwm);
    alloc((void**)&w->W, sizeof(df) * nm * (nm + 1));
    alloc((void**)&w->tau, sizeof(df) * nm);
    alloc((void**)&w->dd, sizeof(df) * nm);
    alloc((void**)&w->ee, sizeof(df) * nm);
    alloc((void**)&w->fac, sizeof(df) * 6 * nm * nwm);
    alloc((void**)&w->Zt, sizeof(df) * nm * nwm);
    alloc((void**)&w->rr, sizeof(df) * 4 * (nwm * nwm > 4 * nwm ? nwm * nwm : 4 * nwm));
    alloc((void**)&w->perm, sizeof(int) * nwm);
    alloc((void**)&w->hv, sizeof(df) * nm * nm);
    alloc((void**)&w->shd, sizeof(df) * (nwm + 1));
    alloc((void**)&w->bounds, sizeof(float) * 4);
    alloc((void**)&w->Lm, sizeof(double) * dn * dn);
    alloc((void**)&w->Hs, sizeof(double) * dn * dn);
    alloc((void**)&w->sr_mu, sizeof(double) * qmax);
    alloc((void**)&w->sr_X, sizeof(double) * nm * qmax);
    alloc((void**)&w->sr_conv, sizeof(int) * qmax);
    alloc((void**)&w->sr_flag, 4 * sizeof(int));
  }
  return w;
}

void pencil_work_destroy(PencilWork* w) {
  if (!w) return;
  if (w->base) dev_release(w->base, w->bytes);  // the caller's work using it has completed
  delete w;
}

cudaLaunchConfig_t tri_config(size_t smem, cudaStream_t st, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kTriCluster);
  cfg.blockDim = dim3(kTriThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kTriCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Whether the tridiagonalisation's cluster with `smem` bytes per CTA can be resident on the current
// device (asked once per device and size class; the answer is kept).
bool cluster_fits(size_t smem) {
  static std::mutex mu;
  static std::map<std::pair<int, int>, bool> known;  // (device, KiB)
  int dev = 0;
  cudaGetDevice(&dev);
  const std::pair<int, int> key = {dev, static_cast<int>((smem + 1023) / 1024)};
  std::lock_guard<std::mutex> lk(mu);
  auto it = known.find(key);
  if (it != known.end()) return it->second;
  const cudaError_t before = cudaPeekAtLastError();
  bool ok = cudaFuncSetAttribute(reinterpret_cast<const void*>(k_syev_tri_cl),
                                 cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  ensure_dynamic_smem(reinterpret_cast<const void*>(k_syev_tri_cl), smem);
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = tri_config(smem, nullptr, attr);
  int clusters = 0;
  ok = ok && cudaOccupancyMaxActiveClusters(&clusters, k_syev_tri_cl, &cfg) == cudaSuccess && clusters > 0;
  if (!ok && before == cudaSuccess) cudaGetLastError();  // the answer is no; an earlier launch's error stays
  known[key] = ok;
  return ok;
}

// Shared memory of k_syev_back: WPB columns, the scalars, `bufs` chunks of C reflectors.
size_t syev_back_smem(int n, int c, int wpb, int bufs) {
  return sizeof(df) * static_cast<size_t>(wpb + 1 + bufs * c) * n;
}

template <int C, int WPB>
void launch_syev_back_as(PencilWork* w, int n, int nwant, int bufs, double* evecs, cudaStream_t st, const int* skip) {
  const size_t sm = syev_back_smem(n, C, WPB, bufs);
  ensure_dynamic_smem(reinterpret_cast<const void*>(k_syev_back<C, WPB>), sm);
  k_syev_back<C, WPB><<<ceil_div(nwant, WPB), 32 * WPB, sm, st>>>(n, nwant, bufs, w->hv, w->tau, w->Zt, evecs, skip);
}

// Eight reflectors and four columns per block while they fit (two chunks in flight up to 1371 rows, one up to
// 2215), then four reflectors, and last one column per block: the largest coarsest level (4096
// rows) with the widest border (128) takes 198 KB.
void launch_syev_back(PencilWork* w, int n, int nwant, double* evecs, cudaStream_t st, const int* skip) {
  const auto fits = [n](int c, int wpb, int bufs) { return syev_back_smem(n, c, wpb, bufs) <= kSmemBudget; };
  if (fits(kSbChunk, kSbWarps, 1))
    launch_syev_back_as<kSbChunk, kSbWarps>(w, n, nwant, fits(kSbChunk, kSbWarps, 2) ? 2 : 1, evecs, st, skip);
  else if (fits(kSbChunk / 2, kSbWarps, 1))
    launch_syev_back_as<kSbChunk / 2, kSbWarps>(w, n, nwant, 1, evecs, st, skip);
  else
    launch_syev_back_as<kSbChunk / 2, 1>(w, n, nwant, 1, evecs, st, skip);
}

void launch_syev_df(PencilWork* w, int n, int nwant, const double* H, double* evals, double* evecs,
                    cudaStream_t st, const int* skip) {
  if (n <= 0 || nwant <= 0) return;
  const int ldw = n | 1;  // odd row stride: column walks of W hit different banks
  const size_t sm_val = 2 * sizeof(df) * static_cast<size_t>(n);
  // groups keep their vectors in shared memory up to the budget (the widest possible group: all nwant)
  const size_t sm_vec = std::min(kSmemBudget, syev_vecs_base(n, nwant) + syev_vecs_work(n, nwant));
  ProfScope ps(st, P_PENCIL, 8.0 * n * n + 8.0 * n * nwant, 0.0, 4);
  // from kTriOneBlock rows a cluster of 16 CTAs, where it can be scheduled
  const size_t tri_rows = ceil_div(n, kTriCluster);
  const size_t sm_cl = sizeof(df) * (tri_rows * ldw + 6 * kTriCluster * (tri_rows | 1) + 3 * static_cast<size_t>(n));
  if (n >= kTriOneBlock && n <= kTriMaxN && cluster_fits(sm_cl)) {
    ensure_dynamic_smem(reinterpret_cast<const void*>(k_syev_tri_cl), sm_cl);
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = tri_config(sm_cl, st, attr);
    cudaLaunchKernelEx(&cfg, k_syev_tri_cl, n, ldw, H, w->hv, w->dd, w->ee, w->tau, skip);
  } else {
    launch_syev_tri_block(w, n, ldw, H, skip, st);
  }
  ensure_dynamic_smem(reinterpret_cast<const void*>(k_syev_vals), sm_val);
  k_syev_vals<<<std::min(nwant + 1, n), kSvThreads, sm_val, st>>>(n, w->dd, w->ee, w->shd, w->bounds, skip);
  ensure_dynamic_smem(reinterpret_cast<const void*>(k_syev_vecs), sm_vec);
  k_syev_vecs<<<nwant, kSvecThreads, sm_vec, st>>>(n, nwant, sm_vec, w->dd, w->ee, w->shd, w->bounds, w->fac, w->rr,
                                                   w->Zt, evals, skip);
  launch_syev_back(w, n, nwant, evecs, st, skip);
}

void launch_pencil_solve(PencilWork* w, int dn, int m, int q, const double* C64, const float2* Cdf,
                         const double* G, const float2* Zdf, const double* theta, double* mu, double* Xc,
                         float2* Xcdf, double* Y, int* status, cudaStream_t st, int* nfallback, int p) {
  if (p <= 0) p = q;  // pairs wanted: the border's width unless a wider border was given
  const int n = m + q;
  auto smem_attr = [](const void* f, size_t bytes) {
    ensure_dynamic_smem(f, bytes);
  };
  const size_t kbs = sizeof(df) * dn;
  const size_t srs = sizeof(df) * (2.0 * m + 2.0 * m * q + 3.0 * q * q + 2.0 * q + 2.0 * n);
  const size_t chs = sizeof(df) * (1.0 * n * q + 5.0 * q * q + 2.0 * m + 1.0 * m * q + 1.0 * q * (q + kMaxCluster) +
                                    3.0 * n * kMaxCluster + 1.0 * kMaxCluster * q);
  const size_t fs = sizeof(df) * (static_cast<size_t>(q) * (q | 1) + q);
  const size_t bks = sizeof(df) * (static_cast<size_t>(q) * q + q);
  const size_t xsc = sizeof(df) * static_cast<size_t>(m + q) * kXcCols;
  // the structured iteration finds one pair per border column: a wider border (p < q) takes the dense path
  const bool fast = p == q && q <= kSrqiMaxQ && srs <= 200 * 1024 && chs <= 220 * 1024;
  // kernels launched here; the dense eigensolver's launcher counts its own
  ProfScope ps(st, P_PENCIL, 8.0 * (2.0 * dn * m + 2.0 * dn * q + 2.0 * m * q + 3.0 * q * q + 1.0 * n * q), 0.0,
               fast ? 7 : 5);
  if (Cdf) {
    smem_attr((const void*)k_kb<float2>, kbs);
    k_kb<float2><<<2 * q, kPenThreads, kbs, st>>>(dn, m, q, Zdf, Cdf, w->KB);
  } else {
    smem_attr((const void*)k_kb<double>, kbs);
    k_kb<double><<<2 * q, kPenThreads, kbs, st>>>(dn, m, q, Zdf, C64, w->KB);
  }
  k_blocks<<<q, kPenThreads, 0, st>>>(m, q, w->KB, G, theta, w->Ft, w->Tt, w->St);
  // structured Rayleigh quotient iteration, checked by inertia; the dense
  // float-float solver runs only when the check rejects it
  const int* skip = nullptr;
  if (fast) {
    smem_attr((const void*)k_srqi, srs);
    smem_attr((const void*)k_srqi_check, chs);
    k_srqi<<<q, kSrqiThreads, srs, st>>>(m, q, theta, w->KB, w->Ft, w->Tt, w->St, w->sr_mu, w->sr_X, w->sr_conv);
    k_srqi_check<<<1, kSrqiThreads, chs, st>>>(m, q, theta, w->KB, w->Ft, w->Tt, w->St, w->sr_mu, w->sr_X,
                                               w->sr_conv, mu, w->Yh, w->sr_flag);
    skip = w->sr_flag;
  }
  smem_attr((const void*)k_std_form, fs);
  {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kStdCluster);
    cfg.blockDim = dim3(kStdThreads);
    cfg.dynamicSmemBytes = fs;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kStdCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_std_form, m, q, theta, static_cast<const df*>(w->Ft), static_cast<const df*>(w->Tt),
                       static_cast<const df*>(w->St), w->Lq, w->Xq, w->H, status, skip, nfallback);
  }
  launch_syev_df(w, n, p, w->H, mu, w->Yh, st, skip);
  smem_attr((const void*)k_std_back, bks);
  k_std_back<<<ceil_div(p, kBackWarps), 32 * kBackWarps, bks, st>>>(m, q, p, w->Lq, w->Yh, skip);
  // Xc = Z_m (a - B b), Y = b
  smem_attr((const void*)k_xc, xsc);
  const int cols = ceil_div(p, kXcCols);
  const int runs = std::max(1, std::min(kXcBlocks / cols, ceil_div(dn, kXcRows)));
  k_xc<<<dim3(cols, runs), kXcThreads, xsc, st>>>(dn, m, q, p, Zdf, w->KB, w->Yh, Xc, Xcdf, Y);
}

void launch_mass_factor(PencilWork* w, int dn, const double* Mn, int* status, cudaStream_t st) {
  ProfScope ps(st, P_PENCIL, 8.0 * dn * dn * 2, dn * static_cast<double>(dn) * dn / 3.0, chol_launches(dn));
  launch_chol_f64(dn, Mn, w->Lm, status, st);
}

void launch_coarse_inverse(int dn, const double* An, double* L, double* Linv, double* Ainv, int* status,
                           cudaStream_t st) {
  // the products count their own launches
  ProfScope ps(st, P_PENCIL, 8.0 * dn * dn * 5, 2.0 * dn * dn * dn, chol_launches(dn) + 1 + ceil_div(dn, kCb));
  // A_n = L L^T; Linv = L^-1 (the identity solved in place); Ainv = Linv^T Linv = L^-T L^-1
  launch_chol_f64(dn, An, L, status, st);
  k_identity<<<ceil_div(static_cast<long long>(dn) * dn, 256), 256, 0, st>>>(dn, Linv);
  launch_trsm_lower(dn, L, Linv, dn, dn, st);
  launch_gemm_f64(dn, dn, dn, 1.0, Linv, dn, true, Linv, dn, false, 0.0, Ainv, dn, st);
}

void launch_coarse_modes(PencilWork* w, int dn, int nwant, const double* An, double* Z, double* theta,
                         cudaStream_t st) {
  // the products and the eigensolver count their own launches
  ProfScope ps(st, P_PENCIL, 8.0 * dn * dn * 6, 4.0 * dn * dn * static_cast<double>(dn), 2 + ceil_div(dn, kCb));
  // Li = L_m^-1 (the identity solved in place, in H); Hs = sym(Li A_n Li^T) by two float64
  // products (scratch: the eigensolver's W, free until the eigensolver runs, and Yh)
  double* Li = w->H;
  double* T = reinterpret_cast<double*>(w->W);
  k_identity<<<ceil_div(static_cast<long long>(dn) * dn, 256), 256, 0, st>>>(dn, Li);
  launch_trsm_lower(dn, w->Lm, Li, dn, dn, st);
  launch_gemm_f64(dn, dn, dn, 1.0, Li, dn, false, An, dn, false, 0.0, T, dn, st);
  launch_gemm_f64(dn, dn, dn, 1.0, T, dn, false, Li, dn, true, 0.0, w->Yh, dn, st);
  k_transpose_sym<<<ceil_div(static_cast<long long>(dn) * dn, 256), 256, 0, st>>>(dn, w->Yh, w->Hs);
  // the nwant lowest eigenpairs of Hs (dn x nwant into Yh); Z's first columns = L_m^-T Y = Li^T Y
  launch_syev_df(w, dn, nwant, w->Hs, theta, w->Yh, st);
  launch_gemm_f64(dn, nwant, dn, 1.0, Li, dn, true, w->Yh, nwant, false, 0.0, Z, dn, st);
}

}  // namespace amgeig
