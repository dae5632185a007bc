// Device code shared by the two forms of the dense symmetric eigensolver: the one
// the solve path runs (pencil.cu) and the one behind the eigensolver entry points
// (eigh.cu), and the workspace both take.
#pragma once

#include "common.cuh"
#include "kernels.cuh"

namespace amgeig {

constexpr size_t kSmemBudget = 225 * 1024;

struct PencilWork {
  int dn = 0, qmax = 0, nmax = 0;
  void* base = nullptr;  // one device allocation holding every array below
  size_t bytes = 0;      // its size
  // Rayleigh-Ritz pencil (float-float)
  df* KB = nullptr;   // dn x 2q   Z_m^T C = [K | B]
  df* Ft = nullptr;   // dn x q    K - Theta B
  df* Tt = nullptr;   // q x q
  df* St = nullptr;   // q x q     Schur complement of the Gram matrix
  df* Lq = nullptr;   // q x q     its Cholesky factor (fallback)
  df* Xq = nullptr;   // q x q     scratch (fallback)
  double* H = nullptr;   // nmax x nmax standard form (fallback)
  double* Yh = nullptr;  // nmax x q eigenvectors [a; b]
  // float-float eigensolver
  df* W = nullptr;     // nmax x nmax
  df* tau = nullptr;   // nmax
  df* dd = nullptr;    // nmax
  df* ee = nullptr;    // nmax
  df* fac = nullptr;   // 6 x nmax x nwant_max
  df* Zt = nullptr;    // nmax x nwant_max
  df* rr = nullptr;    // 4 x nwant_max^2 (Rayleigh-Ritz clean-up)
  int* perm = nullptr; // nwant_max
  df* hv = nullptr;    // nmax x nmax reflectors (split path)
  df* shd = nullptr;   // nwant_max + 1 refined shifts
  float* bounds = nullptr;  // 4: Gershgorin bounds, ||T||, pivot floor (split path)
  int nwant_max = 0;
  // coarse decomposition
  double* Lm = nullptr;  // dn x dn
  double* Hs = nullptr;  // dn x dn
  // structured Rayleigh quotient iteration
  double* sr_mu = nullptr;  // qmax
  double* sr_X = nullptr;   // nmax x qmax
  int* sr_conv = nullptr;   // qmax
  int* sr_flag = nullptr;   // 4: accepted, reason of a rejection, inertia count, q
};

namespace {

__device__ __forceinline__ df shfl_df(df v, int src) {
  return df{__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src)};
}

// sum_i a[i sa] b[i sb] (i < len) in float-float with four interleaved
// accumulators: independent chains keep the float32 pipes busy in these
// latency-bound single-block kernels
__device__ __forceinline__ df_acc dot4(const df* a, int sa, const df* b, int sb, int len) {
  df_acc c0 = acc_zero(), c1 = acc_zero(), c2 = acc_zero(), c3 = acc_zero();
  int i = 0;
  for (; i + 4 <= len; i += 4) {
    c0.fma(a[i * sa], b[i * sb]);
    c1.fma(a[(i + 1) * sa], b[(i + 1) * sb]);
    c2.fma(a[(i + 2) * sa], b[(i + 2) * sb]);
    c3.fma(a[(i + 3) * sa], b[(i + 3) * sb]);
  }
  for (; i < len; ++i) c0.fma(a[i * sa], b[i * sb]);
  c0.merge(c1);
  c2.merge(c3);
  c0.merge(c2);
  return c0;
}

// the same with weights: sum_i a[i sa] w[i] b[i sb]
__device__ __forceinline__ df_acc dot4w(const df* a, int sa, const df* w, const df* b, int sb, int len) {
  df_acc c0 = acc_zero(), c1 = acc_zero(), c2 = acc_zero(), c3 = acc_zero();
  int i = 0;
  for (; i + 4 <= len; i += 4) {
    c0.fma(df_mul(a[i * sa], w[i]), b[i * sb]);
    c1.fma(df_mul(a[(i + 1) * sa], w[i + 1]), b[(i + 1) * sb]);
    c2.fma(df_mul(a[(i + 2) * sa], w[i + 2]), b[(i + 2) * sb]);
    c3.fma(df_mul(a[(i + 3) * sa], w[i + 3]), b[(i + 3) * sb]);
  }
  for (; i < len; ++i) c0.fma(df_mul(a[i * sa], w[i]), b[i * sb]);
  c0.merge(c1);
  c2.merge(c3);
  c0.merge(c2);
  return c0;
}

// Gap between consecutive refined shifts, compared in float32 against the
// cluster and group thresholds below.
__device__ __forceinline__ float shift_gap(const df* shd, int j) {
  return j > 0 ? df_float(df_sub(shd[j], shd[j - 1])) : 3.0e38f;
}

// Inverse iteration in float-float for the shift sg of index j, one thread:
// T - sg I = L D L^T (pivots kept at least pv in magnitude), three solves from
// a fixed start vector, each followed by Gram-Schmidt against the finished
// members c0 .. jj-1 of its cluster and a normalisation.  Element i of the
// vector, of 1/d and of l is at [i ld + jj] of Z, dinv and lm.
__device__ void syev_inverse_iteration(int j, int jj, int c0, df sg, const df* dd, const df* ee, int n, df pv,
                                       df* dinv, df* lm, df* Z, long long ld) {
  df d = df_sub(dd[0], sg);
  if (fabsf(d.hi) < pv.hi) d = df_lt0(d) ? df_neg(pv) : pv;
  df di = df_div(df{1.f, 0.f}, d);
  dinv[jj] = di;
  for (int i = 1; i < n; ++i) {
    const df e = ee[i - 1];
    const df l = df_mul(e, di);
    lm[(i - 1) * ld + jj] = l;
    d = df_sub(df_sub(dd[i], sg), df_mul(l, e));
    if (fabsf(d.hi) < pv.hi) d = df_lt0(d) ? df_neg(pv) : pv;
    di = df_div(df{1.f, 0.f}, d);
    dinv[i * ld + jj] = di;
  }
  // start vector
  for (int i = 0; i < n; ++i) Z[i * ld + jj] = df{1.f + 0.37f * (float)((i * 7 + j * 13) % 11) / 11.f, 0.f};
  for (int it = 0; it < 3; ++it) {
    // L w = x ; z = D^-1 w ; L^T y = z
    df prev = Z[jj];
    for (int i = 1; i < n; ++i) {
      prev = df_sub(Z[i * ld + jj], df_mul(lm[(i - 1) * ld + jj], prev));
      Z[i * ld + jj] = prev;
    }
    df nxt = df_mul(Z[(n - 1) * ld + jj], dinv[(n - 1) * ld + jj]);
    Z[(n - 1) * ld + jj] = nxt;
    for (int i = n - 2; i >= 0; --i) {
      nxt = df_sub(df_mul(Z[i * ld + jj], dinv[i * ld + jj]), df_mul(lm[i * ld + jj], nxt));
      Z[i * ld + jj] = nxt;
    }
    // Gram-Schmidt against finished members of the cluster
    for (int jp = c0; jp < jj; ++jp) {
      df_acc dt = acc_zero();
      for (int i = 0; i < n; ++i) dt.fma(Z[i * ld + jp], Z[i * ld + jj]);
      const df dv = dt.value();
      for (int i = 0; i < n; ++i) Z[i * ld + jj] = df_sub(Z[i * ld + jj], df_mul(dv, Z[i * ld + jp]));
    }
    // normalise (scale first by the largest entry to stay in range)
    float amax = 0.f;
    for (int i = 0; i < n; ++i) amax = fmaxf(amax, fabsf(Z[i * ld + jj].hi));
    const float sc1 = amax > 0.f ? 1.f / amax : 1.f;
    df_acc dn = acc_zero();
    for (int i = 0; i < n; ++i) {
      const df z = df_mul_f(Z[i * ld + jj], sc1);
      Z[i * ld + jj] = z;
      dn.fma(z, z);
    }
    const df inv = df_div(df{1.f, 0.f}, df_sqrt(dn.value()));
    for (int i = 0; i < n; ++i) Z[i * ld + jj] = df_mul(Z[i * ld + jj], inv);
  }
}

// Rayleigh-Ritz clean-up of one group of G >= 2 vectors by the whole block.
// The group's shifts are more than 1e-4 ||T|| from every other group's, so each
// vector's error outside its own group's span is below ~4e-11, and a
// Rayleigh-Ritz step on the span (S = Z_g^T Z_g, Hq = Z_g^T T Z_g) restores
// working accuracy: S = L L^T, C = L^-1 Hq L^-T by parallel cyclic Jacobi,
// vectors Z_g L^-T Q in ascending order.  Column c of the group is at
// Z[i ldz + c] and goes to Zn[i ldn + c], its eigenvalue to evals[c].  rrw:
// 4 G^2 df, perm: G ints, red, sf: block reduction scratch (shared).  TZ: n x G
// df scratch with Z's row stride (T Z, formed once).  TA x TB: the register
// tile of S and Hq per thread.
template <int TA, int TB>
__device__ void syev_group_rr(int G, const df* Z, long long ldz, const df* dd, const df* ee, int n, df* TZ,
                              df* rrw, int* perm, df_acc* red, float* sf, df* Zn, long long ldn, double* evals) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const long long N = n;
  df* S = rrw;
  df* Hq = rrw + G * G;
  df* Qm = rrw + 2 * G * G;
  df* Xm = rrw + 3 * G * G;
  for (int i = warp; i < n; i += nw)
    for (int c = lane; c < G; c += 32) {
      df_acc tz = acc_zero();
      tz.fma(dd[i], Z[i * ldz + c]);
      if (i > 0) tz.fma(ee[i - 1], Z[(i - 1) * ldz + c]);
      if (i + 1 < n) tz.fma(ee[i], Z[(i + 1) * ldz + c]);
      TZ[i * ldz + c] = tz.value();
    }
  __syncthreads();
  // S = Z^T Z and Hq = Z^T (T Z): the upper triangle by TA x TB tiles, one
  // compensated sum per entry over the rows in order; the lower triangle mirrors it
  {
    // tile row ta starts at tile column (ta TA) / TB, the first that reaches the diagonal
    const int na = (G + TA - 1) / TA, nbt = (G + TB - 1) / TB;
    int ntile = 0;
    for (int ta = 0; ta < na; ++ta) ntile += nbt - (ta * TA) / TB;
    for (int tix = tid; tix < ntile; tix += nt) {
      int ta = 0, rem = tix;
      while (rem >= nbt - (ta * TA) / TB) {
        rem -= nbt - (ta * TA) / TB;
        ++ta;
      }
      const int a0 = ta * TA, b0 = ((ta * TA) / TB + rem) * TB;
      df_acc sa[TA][TB], ha[TA][TB];
#pragma unroll
      for (int u = 0; u < TA; ++u)
#pragma unroll
        for (int v = 0; v < TB; ++v) sa[u][v] = ha[u][v] = acc_zero();
      for (int i = 0; i < n; ++i) {
        df za[TA], zb[TB], tb[TB];
#pragma unroll
        for (int u = 0; u < TA; ++u) za[u] = a0 + u < G ? Z[i * ldz + a0 + u] : df{0.f, 0.f};
#pragma unroll
        for (int v = 0; v < TB; ++v) {
          const bool ib = b0 + v < G;
          zb[v] = ib ? Z[i * ldz + b0 + v] : df{0.f, 0.f};
          tb[v] = ib ? TZ[i * ldz + b0 + v] : df{0.f, 0.f};
        }
#pragma unroll
        for (int u = 0; u < TA; ++u)
#pragma unroll
          for (int v = 0; v < TB; ++v) {
            sa[u][v].fma(za[u], zb[v]);
            ha[u][v].fma(za[u], tb[v]);
          }
      }
#pragma unroll
      for (int u = 0; u < TA; ++u)
#pragma unroll
        for (int v = 0; v < TB; ++v) {
          const int a = a0 + u, b = b0 + v;
          if (a <= b && b < G) {
            S[a * G + b] = S[b * G + a] = sa[u][v].value();
            Hq[a * G + b] = Hq[b * G + a] = ha[u][v].value();
          }
        }
    }
  }
  __syncthreads();
  // Cholesky S = L L^T in place (lower), right-looking
  for (int kk = 0; kk < G; ++kk) {
    if (tid == 0) S[kk * G + kk] = df_sqrt(S[kk * G + kk]);
    __syncthreads();
    const df piv = S[kk * G + kk];
    for (int i = kk + 1 + tid; i < G; i += nt) S[i * G + kk] = df_div(S[i * G + kk], piv);
    __syncthreads();
    for (int idx = tid; idx < (G - kk - 1) * (G - kk - 1); idx += nt) {
      const int i = kk + 1 + idx / (G - kk - 1), jj = kk + 1 + idx % (G - kk - 1);
      if (jj <= i) S[i * G + jj] = df_sub(S[i * G + jj], df_mul(S[i * G + kk], S[jj * G + kk]));
    }
    __syncthreads();
  }
  // C = L^-1 Hq L^-T  (two column-parallel forward substitutions; each row's
  // sum over the solved rows in four compensated chains)
  for (int pass = 0; pass < 2; ++pass) {
    df* out = pass == 0 ? Xm : Qm;
    for (int col = tid; col < G; col += nt) {
      for (int i = 0; i < G; ++i) {
        const df rhs = (pass == 0) ? Hq[i * G + col] : Xm[col * G + i];
        const df s = df_sub(rhs, dot4(S + i * G, 1, out + col, G, i).value());
        out[i * G + col] = df_div(s, S[i * G + i]);
      }
    }
    __syncthreads();
  }
  // Qm now holds C (symmetric); move it to Hq and set Qm = I
  for (int idx = tid; idx < G * G; idx += nt) {
    const int a0 = idx / G, b0 = idx % G;
    const df cab = Qm[a0 * G + b0], cba = Qm[b0 * G + a0];
    Hq[idx] = df_mul_f(df_add(cab, cba), 0.5f);
  }
  __syncthreads();
  for (int idx = tid; idx < G * G; idx += nt) Qm[idx] = df{(idx / G == idx % G) ? 1.f : 0.f, 0.f};
  __syncthreads();
  // parallel cyclic Jacobi (round-robin pairing) on C, accumulating Q
  {
    const int np = (G + 1) & ~1;  // even player count; index G is a dummy
    for (int sweep = 0; sweep < 12; ++sweep) {
      // convergence test: largest off-diagonal entry against the largest diagonal one
      float off = 0.f, dia = 0.f;
      for (int idx = tid; idx < G * G; idx += nt) {
        const int a0 = idx / G, b0 = idx % G;
        const float x = fabsf(Hq[idx].hi);
        if (a0 == b0) dia = fmaxf(dia, x); else off = fmaxf(off, x);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        off = fmaxf(off, __shfl_xor_sync(0xffffffffu, off, o));
        dia = fmaxf(dia, __shfl_xor_sync(0xffffffffu, dia, o));
      }
      if (lane == 0) {
        red[warp].s = off;
        red[warp].c = dia;
      }
      __syncthreads();
      if (tid == 0) {
        float o2 = 0.f, d2 = 0.f;
        for (int w2 = 0; w2 < nw; ++w2) {
          o2 = fmaxf(o2, red[w2].s);
          d2 = fmaxf(d2, red[w2].c);
        }
        sf[0] = o2;
        sf[1] = d2;
      }
      __syncthreads();
      const float offmax = sf[0], diamax = sf[1];
      __syncthreads();
      if (!(offmax > 1.0e-15f * fmaxf(diamax, 1.0e-30f))) break;
      for (int r = 0; r < np - 1; ++r) {
        // pair t: players (a, b) of the round-robin schedule
        for (int t = tid; t < np / 2; t += nt) {
          int a0 = (t == 0) ? 0 : 1 + (t - 1 + r) % (np - 1);
          int b0 = 1 + (np - 2 - t + r) % (np - 1);
          if (a0 > b0) {
            const int tmpi = a0;
            a0 = b0;
            b0 = tmpi;
          }
          df cs = df{1.f, 0.f}, sn = df{0.f, 0.f};
          if (b0 < G) {
            const df apq = Hq[a0 * G + b0];
            const df app = Hq[a0 * G + a0], aqq = Hq[b0 * G + b0];
            // skip entries already below the float-float resolution of the diagonal
            const float thr = 1.0e-17f * (sqrtf(fabsf(app.hi)) * sqrtf(fabsf(aqq.hi))) + 1.0e-37f;
            if (fabsf(apq.hi) > thr) {
              // theta = (aqq - app) / (2 apq); t = sign(theta) / (|theta| + sqrt(theta^2 + 1)),
              // and t = 1 / (2 theta) once theta^2 would leave the float range
              const df th = df_div(df_sub(aqq, app), df_mul_f(apq, 2.f));
              df tt;
              if (fabsf(th.hi) > 1.0e12f) {
                tt = df_div(df{0.5f, 0.f}, th);
              } else {
                const df rt = df_sqrt(df_add(df_mul(th, th), df{1.f, 0.f}));
                tt = df_div(df{1.f, 0.f}, df_add(df_abs(th), rt));
                if (df_lt0(th)) tt = df_neg(tt);
              }
              cs = df_div(df{1.f, 0.f}, df_sqrt(df_add(df_mul(tt, tt), df{1.f, 0.f})));
              sn = df_mul(tt, cs);
            }
          }
          // stash rotation in Xm row 0..np/2 (cols 0..3)
          Xm[t * 4 + 0] = cs;
          Xm[t * 4 + 1] = sn;
          reinterpret_cast<int*>(&Xm[t * 4 + 2])[0] = a0;
          reinterpret_cast<int*>(&Xm[t * 4 + 3])[0] = b0;
        }
        __syncthreads();
        // C <- J^T C J by 2 x 2 blocks (pair s, pair t), s <= t, the lower
        // triangle mirrored; the rows of each block turn first, then its columns.
        // The triangle of pair blocks is folded (row s with row P - 1 - s) so
        // that every thread gets the same share.  Q <- Q J alongside.
        {
          const int P = np / 2, half = (P + 1) / 2;
          for (int idx = tid; idx < half * (P + 1); idx += nt) {
            const int fr = idx / (P + 1), cc = idx - fr * (P + 1);
            int ps, pt;
            if (cc < P - fr) {
              ps = fr;
              pt = fr + cc;
            } else {
              ps = P - 1 - fr;
              if (ps == fr) continue;
              pt = ps + (cc - (P - fr));
            }
            const int as = reinterpret_cast<const int*>(&Xm[ps * 4 + 2])[0];
            const int bs = reinterpret_cast<const int*>(&Xm[ps * 4 + 3])[0];
            const int at = reinterpret_cast<const int*>(&Xm[pt * 4 + 2])[0];
            const int bt = reinterpret_cast<const int*>(&Xm[pt * 4 + 3])[0];
            const df css = Xm[ps * 4 + 0], sns = Xm[ps * 4 + 1];
            const df cst = Xm[pt * 4 + 0], snt = Xm[pt * 4 + 1];
            const bool rs = bs < G, rt = bt < G;
            const df zero = df{0.f, 0.f};
            df x00 = Hq[as * G + at], x01 = rt ? Hq[as * G + bt] : zero;
            df x10 = rs ? Hq[bs * G + at] : zero, x11 = (rs && rt) ? Hq[bs * G + bt] : zero;
            if (rs) {
              const df y00 = df_sub(df_mul(css, x00), df_mul(sns, x10));
              const df y10 = df_add(df_mul(sns, x00), df_mul(css, x10));
              const df y01 = df_sub(df_mul(css, x01), df_mul(sns, x11));
              const df y11 = df_add(df_mul(sns, x01), df_mul(css, x11));
              x00 = y00;
              x10 = y10;
              x01 = y01;
              x11 = y11;
            }
            if (rt) {
              const df y00 = df_sub(df_mul(cst, x00), df_mul(snt, x01));
              const df y01 = df_add(df_mul(snt, x00), df_mul(cst, x01));
              const df y10 = df_sub(df_mul(cst, x10), df_mul(snt, x11));
              const df y11 = df_add(df_mul(snt, x10), df_mul(cst, x11));
              x00 = y00;
              x01 = y01;
              x10 = y10;
              x11 = y11;
            }
            if (ps == pt) {
              // diagonal block: (as, bs) and (bs, as) take the same value
              Hq[as * G + as] = x00;
              if (rs) {
                Hq[as * G + bs] = Hq[bs * G + as] = x01;
                Hq[bs * G + bs] = x11;
              }
            } else {
              Hq[as * G + at] = Hq[at * G + as] = x00;
              if (rt) Hq[as * G + bt] = Hq[bt * G + as] = x01;
              if (rs) Hq[bs * G + at] = Hq[at * G + bs] = x10;
              if (rs && rt) Hq[bs * G + bt] = Hq[bt * G + bs] = x11;
            }
          }
          for (int t = warp; t < P; t += nw) {
            const int a0 = reinterpret_cast<const int*>(&Xm[t * 4 + 2])[0];
            const int b0 = reinterpret_cast<const int*>(&Xm[t * 4 + 3])[0];
            if (b0 >= G) continue;
            const df cs = Xm[t * 4 + 0], sn = Xm[t * 4 + 1];
            for (int row = lane; row < G; row += 32) {
              const df x = Qm[row * G + a0], y = Qm[row * G + b0];
              Qm[row * G + a0] = df_sub(df_mul(cs, x), df_mul(sn, y));
              Qm[row * G + b0] = df_add(df_mul(sn, x), df_mul(cs, y));
            }
          }
        }
        __syncthreads();
      }
    }
  }
  // order eigenvalues ascending (selection by rank; ties broken by index); the identity first, so that
  // perm holds valid columns even when a NaN leaves ranks unassigned
  for (int j = tid; j < G; j += nt) perm[j] = j;
  __syncthreads();
  for (int j = tid; j < G; j += nt) {
    const df lj = Hq[j * G + j];
    int rank = 0;
    for (int i = 0; i < G; ++i) {
      const df li = Hq[i * G + i];
      const df dlt = df_sub(li, lj);
      if (df_lt0(dlt) || ((dlt.hi == 0.f && dlt.lo == 0.f) && i < j)) ++rank;
    }
    perm[rank] = j;
  }
  __syncthreads();
  // Xm = L^-T Q  (back substitution per column)
  for (int col = tid; col < G; col += nt) {
    for (int i = G - 1; i >= 0; --i) {
      const df s = df_sub(Qm[i * G + col], dot4(S + (i + 1) * G + i, G, Xm + (i + 1) * G + col, G, G - 1 - i).value());
      Xm[i * G + col] = df_div(s, S[i * G + i]);
    }
  }
  __syncthreads();
  // group eigenvectors Zn[:, c] = Z_g Xm[:, perm[c]] (ascending within the group)
  for (long long idx = tid; idx < N * G; idx += nt) {
    const int i = static_cast<int>(idx / G), c = static_cast<int>(idx % G);
    const int src = perm[c];
    df_acc sa = acc_zero();
    for (int kk = 0; kk < G; ++kk) sa.fma(Z[i * ldz + kk], Xm[kk * G + src]);
    Zn[i * ldn + c] = sa.value();
  }
  for (int c = tid; c < G; c += nt) evals[c] = df_to_double(Hq[perm[c] * G + perm[c]]);
  __syncthreads();
}

// Bytes of shared memory k_syev_vecs keeps for a group of G vectors: d, e
// (2n df), cluster data (2G ints), perm (G ints), and -- in shared memory when
// they fit -- the factors and vectors (3 n G df) and the clean-up matrices (4 G^2 df).
__host__ __device__ inline size_t syev_vecs_base(int n, int G) {
  return (2 * sizeof(df) * static_cast<size_t>(n) + 3 * sizeof(int) * static_cast<size_t>(G) + 15) &
         ~static_cast<size_t>(15);
}
__host__ __device__ inline size_t syev_vecs_work(int n, int G) {
  return sizeof(df) * (3 * static_cast<size_t>(n) * G + 4 * static_cast<size_t>(G) * G);
}

}  // namespace
}  // namespace amgeig
