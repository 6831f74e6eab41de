// Smallest eigenpair of a Hermitian (or real symmetric) n x n matrix, n <= 64,
// by one CTA: the reduction on all of it, the rest on its first warp (the size
// scan and the coprimality test; the deblurring's solves spread every step over
// four warps, cbp_tri_team.cuh, with the helpers of this file).
//
//   1. Householder reduction to a real symmetric tridiagonal T = Q^H G Q
//      (reflectors H_k = I - tau_k v_k v_k^H chosen so that beta_k is real);
//   2. Sturm counts by multisection (each lane counts at its own shift) for
//      the two smallest and the largest eigenvalue of T: single-precision
//      rounds down to the single-precision floor, then double-precision
//      rounds inside the widened brackets;
//   3. inverse iteration on T - sigma I (tridiagonal LU with row interchanges)
//      with sigma inside the bracket of the smallest eigenvalue;
//   4. x = Q y.
//
// All but the first bisection rounds run in double precision: a GPU whose double
// pipe is narrow spends its time on the reduction's rank-2 updates, n^3 / 3
// complex multiply-adds in all.  Sign and exponent tests use the integer pipe;
// reciprocals start from a single-precision seed.
//
// Lane l owns the columns l and l + 32.  The matrix is stored in full with row
// stride n; lane i touches element (j, i) of row j, so every access of a row
// is contiguous across the warp.  Included inside namespace cbp::(anonymous)
// of the solver's translation unit, after its scalar helpers (fma_, to_cd,
// re_, cj_, a2_, Ops).

__device__ __forceinline__ double im_(double) { return 0.0; }
__device__ __forceinline__ float im_(float) { return 0.f; }
template <typename T> __device__ __forceinline__ T im_(cpx<T> x) { return x.im; }
template <typename E, typename R> __device__ __forceinline__ E mk_e(R re, R im);
template <> __device__ __forceinline__ double mk_e<double, double>(double re, double) { return re; }
template <> __device__ __forceinline__ cd mk_e<cd, double>(double re, double im) { return mk(re, im); }
__device__ __forceinline__ double mul_(double a, double b) { return a * b; }
template <typename T> __device__ __forceinline__ cpx<T> mul_(cpx<T> a, cpx<T> b) { return a * b; }
__device__ __forceinline__ double sc_(double s, double a) { return s * a; }
template <typename T> __device__ __forceinline__ cpx<T> sc_(T s, cpx<T> a) { return s * a; }
__device__ __forceinline__ void fma_(cf& acc, cf a, cf b) { cfma(acc, a, b); }
// real scalar type of an element type
template <typename E> struct RealOf { using type = E; };
template <typename T> struct RealOf<cpx<T>> { using type = T; };
// reflector element -> vector element
__device__ __forceinline__ cd to_v(double x, cd) { return mk(x, 0.0); }
__device__ __forceinline__ cd to_v(cd x, cd) { return x; }

// Per-warp work area.
struct TriWs {
  void* A;        // E[n * n]: the matrix; row k then holds reflector v_k (k+1..n-1); 16 (n^2 + n)
                  // bytes: the single-precision path keeps Q (cf [n][n + 1]) behind its reflectors
  void* tau;      // E[n]
  void* w;        // E[n]
  double* d;      // [n] diagonal of T
  double* e;      // [n] off-diagonal of T: e[k] couples rows k and k + 1
  double* e2;     // [n] e^2
  double* u0;     // [n] LU of T - sigma I: diagonal of U
  double* u1;     // [n] first superdiagonal of U
  double* u2;     // [n] second superdiagonal of U (row interchanges)
  double* lm;     // [n] multipliers
  int* piv;       // [n] 1 where rows k and k + 1 were interchanged
  float* df;      // [n] d in single precision
  float* e2f;     // [n] e^2 in single precision
  void* part;     // [8][n] complex: per-warp partial sums of the CTA's reduction
  cd* x;          // [n] the eigenvector of G
  cd* r;          // [n] residual
  cd* z;          // [n] scratch (T coordinates)
  cd* q;          // [n] scratch (T coordinates)
};

// Bytes of one warp's work area; a multiple of 128, so that every warp's area
// (placed back to back) and each of its 16-byte-aligned parts stay aligned.
__host__ __device__ inline size_t tri_ws_bytes(int n) {
  const size_t b = (size_t)16 * ((size_t)n * n + 3 * n) + (size_t)8 * 7 * n + (size_t)4 * 3 * n +
                   (size_t)16 * 4 * n + (size_t)16 * 8 * n + 16 * 20;   // + alignment of the parts
  return (b + 127) & ~size_t(127);
}

__device__ inline TriWs carve_tri(char* p, int n) {
  TriWs W;
  auto take = [&](size_t bytes) {
    char* q = p;
    p += (bytes + 15) & ~size_t(15);
    return q;
  };
  W.A = take((size_t)16 * n * n + (size_t)16 * n);
  W.tau = take((size_t)16 * n);
  W.w = take((size_t)16 * n);
  W.x = (cd*)take((size_t)16 * n);
  W.r = (cd*)take((size_t)16 * n);
  W.z = (cd*)take((size_t)16 * n);
  W.q = (cd*)take((size_t)16 * n);
  W.d = (double*)take((size_t)8 * n);
  W.e = (double*)take((size_t)8 * n);
  W.e2 = (double*)take((size_t)8 * n);
  W.u0 = (double*)take((size_t)8 * n);
  W.u1 = (double*)take((size_t)8 * n);
  W.u2 = (double*)take((size_t)8 * n);
  W.lm = (double*)take((size_t)8 * n);
  W.piv = (int*)take((size_t)4 * n);
  W.df = (float*)take((size_t)4 * n);
  W.e2f = (float*)take((size_t)4 * n);
  W.part = take((size_t)16 * 8 * n);
  return W;
}

// Per-lane work on the columns i = lane and i = lane + 32 of an n-wide row:
// f(ColNo<0>, lane), then f(ColNo<1>, lane + 32) where n reaches it.  The second
// is a loop, i.e. a real branch: a double instruction that is only predicated
// off holds the double unit like any other (measured: 118 cycles for one and
// its select), and `if (lane + 32 < n)` around a few of them compiles to
// predicates -- for n <= 32 that had doubled the solver's double-precision work.
template <int C> struct ColNo { static constexpr int c = C; };
template <class F> __device__ __forceinline__ void cols(int n, const F& f) {
  const int lane = threadIdx.x & 31;
  f(ColNo<0>{}, lane);
  for (int i = lane + 32; i < n; i += 32) f(ColNo<1>{}, i);
}
#define CBP_COLS(n, ...) \
  cols((n), [&](auto col_, const int i) { constexpr int c = decltype(col_)::c; (void)c; __VA_ARGS__ })

// Sign and zero tests of a double on the integer pipe.
__device__ __forceinline__ bool dneg(double x) { return __double_as_longlong(x) < 0; }
__device__ __forceinline__ bool dzero(double x) { return (__double_as_longlong(x) << 1) == 0; }
__device__ __forceinline__ int dexp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// The same reduction by all warps of the CTA (real samples, whose solve has a
// CTA to itself): the lead warp forms each reflector; the matrix-vector
// product and the rank-2 update are split by rows j = w (mod warps), the
// product's per-warp partial sums meeting in part[w][i].
template <typename E>
__device__ void tri_reduce_block(E* A, E* tau, E* w, typename RealOf<E>::type* d,
                                 typename RealOf<E>::type* e, int n, E* part /* [8][n] */) {
  using R = typename RealOf<E>::type;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = min(8, (int)(blockDim.x >> 5));   // warps taking part
  if (warp >= nw) {                                 // the others only keep the barriers
    for (int k = 0; k + 1 < n; ++k) {
      __syncthreads();
      if (!Ops<E>::nz(tau[k])) continue;
      __syncthreads();
      __syncthreads();
      __syncthreads();
    }
    __syncthreads();
    return;
  }
  for (int k = 0; k + 1 < n; ++k) {
    const int k1 = k + 1;
    E* vk = A + (size_t)k * n;
    if (warp == 0) {
      const E alpha = cj_(vk[k1]);
      R xn2 = R(0);
      for (int i = lane; i < n; i += 32)
        if (i > k1) xn2 += a2_(vk[i]);
      xn2 = warp_sum(xn2);
      const R ar = re_(alpha), ai = im_(alpha);
      E tk = Ops<E>::z();
      R beta = ar;
      if (xn2 > R(0) || ai != R(0)) {
        beta = -copysign(sqrt(ar * ar + ai * ai + xn2), ar);
        const R ib = R(1) / beta;
        tk = mk_e<E, R>((beta - ar) * ib, -ai * ib);
        const R dr = ar - beta, dn = R(1) / (dr * dr + ai * ai);
        const E scl = mk_e<E, R>(dr * dn, -ai * dn);
        __syncwarp();
        for (int i = lane; i < n; i += 32) {
          if (i > k1) vk[i] = mul_(cj_(vk[i]), scl);
          else if (i == k1) vk[i] = Ops<E>::o();
        }
      } else {
        __syncwarp();
        for (int i = lane; i < n; i += 32)
          if (i == k1) vk[i] = Ops<E>::o();
      }
      if (lane == 0) {
        d[k] = re_(A[(size_t)k * n + k]);
        e[k] = beta;
        tau[k] = tk;
      }
    }
    __syncthreads();
    const E tk = tau[k];
    if (!Ops<E>::nz(tk)) continue;
    // partial products over this warp's rows
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int i = lane + 32 * c;
      if (i > k && i < n) {
        E acc = Ops<E>::z();
        for (int j = k1 + warp; j < n; j += nw) fma_(acc, cj_(A[(size_t)j * n + i]), vk[j]);
        part[warp * n + i] = acc;
      }
    }
    __syncthreads();
    if (warp == 0) {
      E y[2];
      E dotl = Ops<E>::z();
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int i = lane + 32 * c;
        y[c] = Ops<E>::z();
        if (i > k && i < n) {
          E acc = part[i];
          for (int ww = 1; ww < nw; ++ww) acc = acc + part[ww * n + i];
          y[c] = mul_(tk, acc);
          fma_(dotl, cj_(vk[i]), y[c]);
        }
      }
      const E dot = warp_sum_e(dotl);
      const R hc = R(0.5) * re_(mul_(cj_(tk), dot));
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int i = lane + 32 * c;
        if (i > k && i < n) w[i] = y[c] - sc_(hc, vk[i]);
      }
    }
    __syncthreads();
    // rank-2 update of this warp's rows
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int i = lane + 32 * c;
      if (i > k && i < n) {
        const E cw = cj_(w[i]), cv = cj_(vk[i]);
        for (int j = k1 + warp; j < n; j += nw) {
          E t = mul_(vk[j], cw);
          fma_(t, w[j], cv);
          A[(size_t)j * n + i] = A[(size_t)j * n + i] - t;
        }
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) d[n - 1] = re_(A[(size_t)(n - 1) * n + n - 1]);
  __syncthreads();
}

// Number of eigenvalues of T below sig: sign changes of the leading principal
// minors p_i = det(T_i - sig I) (p_i = (d_i - sig) p_{i-1} - e_{i-1}^2 p_{i-2};
// a zero minor takes the sign opposite to its predecessor's).  The minors
// are rescaled by powers of two when they leave [2^-600, 2^600].
__device__ __forceinline__ int sturm_count(const double* d, const double* e2, int n, double sig) {
  double pm = 1.0, p = d[0] - sig;
  bool negp = dneg(p) || dzero(p);
  int cnt = negp ? 1 : 0;
  for (int i = 1; i < n; ++i) {
    const double pn = fma(d[i] - sig, p, -e2[i - 1] * pm);
    pm = p;
    p = pn;
    const bool neg = dzero(p) ? !negp : dneg(p);
    cnt += neg != negp;
    negp = neg;
    if ((i & 7) == 0) {
      const int ex = max(dexp(p), dexp(pm));
      if (ex > 1023 + 600) {
        p *= 0x1p-600;
        pm *= 0x1p-600;
      } else if (ex < 1023 - 600 && ex > 0) {
        p *= 0x1p600;
        pm *= 0x1p600;
      }
    }
  }
  return cnt;
}

// The same count in single precision, in ratio form q_i = p_i / p_{i-1}
// (a ratio below tiny in magnitude is taken as -tiny).  It is exact for a
// matrix within a few single-precision units of ||T|| of T.
__device__ __forceinline__ int sturm_count_f(const float* d, const float* e2, int n, float sig,
                                             float tiny) {
  float q = d[0] - sig;
  if (fabsf(q) < tiny) q = -tiny;
  int cnt = q < 0.f ? 1 : 0;
  for (int i = 1; i < n; ++i) {
    q = (d[i] - sig) - __fdividef(e2[i - 1], q);
    if (fabsf(q) < tiny) q = -tiny;
    cnt += q < 0.f ? 1 : 0;
  }
  return cnt;
}

// One multisection round for the t-th smallest eigenvalue (t = 0, 1, ...):
// lanes count at 32 interior points of [lo, hi]; the bracket shrinks 33x.
// Brackets of eigenvalues 1 and n - 1 are narrowed from the same counts.
struct Bracket {
  double lo, hi;
};
__device__ __forceinline__ void shrink(Bracket& b, unsigned above, double sig) {
  const int first = above ? __ffs(above) - 1 : 32;
  const double slo = __shfl_sync(0xffffffffu, sig, first > 0 ? first - 1 : 0);
  const double shi = __shfl_sync(0xffffffffu, sig, first < 32 ? first : 31);
  if (first > 0) b.lo = fmax(b.lo, slo);
  if (first < 32) b.hi = fmin(b.hi, shi);
}
// One round on bracket t; the counts narrow all nb brackets (target
// eigenvalue index which[m] each).  SINGLE: counts in single precision at
// shifts rounded to single precision.
template <bool SINGLE>
__device__ void multisect(const TriWs& W, int n, int t, Bracket* br, int nb, const int* which,
                          float tiny_f) {
  const int lane = threadIdx.x & 31;
  const double h = (br[t].hi - br[t].lo) * (1.0 / 33.0);
  double sig = fma(h, (double)(lane + 1), br[t].lo);
  int c;
  if (SINGLE) {
    const float sf = (float)sig;
    sig = (double)sf;
    c = sturm_count_f(W.df, W.e2f, n, sf, tiny_f);
  } else {
    c = sturm_count(W.d, W.e2, n, sig);
  }
  for (int m = 0; m < nb; ++m) {
    const unsigned above = __ballot_sync(0xffffffffu, c > which[m]);
    shrink(br[m], above, sig);
  }
}

// 3. LU of the tridiagonal T - sig I with row interchanges (lane 0 only);
// pivots below tiny = u ||T|| in magnitude become +-tiny.  u0 keeps the
// reciprocals of U's diagonal.
__device__ __forceinline__ double rcp_safe(double x) {
  return fabs(x) > 1e-30 && fabs(x) < 1e30 ? rcp_d(x) : 1.0 / x;
}
__device__ __forceinline__ double rsqrt_safe(double x) {
  return x > 1e-30 && x < 1e30 ? rsqrt_d(x) : 1.0 / sqrt(x);
}
__device__ __forceinline__ double clamp_pivot(double x, double tiny) {
  return fabs(x) >= tiny ? x : (dneg(x) ? -tiny : tiny);
}
__device__ __forceinline__ float clamp_pivot(float x, float tiny) {
  return fabsf(x) >= tiny ? x : (x < 0.f ? -tiny : tiny);
}
template <typename R>
__device__ void tri_lu(const R* d, const R* e, R* u0, R* u1, R* u2, R* lm, int* pv, int n, R sig,
                       R tiny) {
  if ((threadIdx.x & 31) != 0) return;
  for (int i = 0; i < n; ++i) {
    u0[i] = d[i] - sig;
    u1[i] = i + 1 < n ? e[i] : R(0);
    u2[i] = R(0);
  }
  for (int i = 0; i + 1 < n; ++i) {
    const R sub = e[i];   // element (i + 1, i)
    const R piv = u0[i];
    if (fabs(piv) >= fabs(sub)) {
      const R r = rcp_safe(clamp_pivot(piv, tiny));
      const R m = sub * r;
      lm[i] = m;
      pv[i] = 0;
      u0[i] = r;
      u0[i + 1] -= m * u1[i];
    } else {
      const R r = rcp_safe(sub);
      const R m = piv * r;
      const R a1 = u0[i + 1], b1 = u1[i + 1];
      lm[i] = m;
      pv[i] = 1;
      u0[i] = r;
      u0[i + 1] = u1[i] - m * a1;
      u1[i + 1] = -m * b1;
      u1[i] = a1;
      u2[i] = b1;
    }
  }
  u0[n - 1] = rcp_safe(clamp_pivot(u0[n - 1], tiny));
}
__device__ __forceinline__ void tri_lu(const TriWs& W, int n, double sig, double tiny) {
  tri_lu<double>(W.d, W.e, W.u0, W.u1, W.u2, W.lm, W.piv, n, sig, tiny);
}

// Solve (T - sig I) z = b in place from tri_lu's factors (lane 0 only).
template <typename R, typename V>
__device__ void tri_solve(const R* u0, const R* u1, const R* u2, const R* lm, const int* pv, int n,
                          V* b) {
  if ((threadIdx.x & 31) != 0) return;
  for (int i = 0; i + 1 < n; ++i) {
    if (pv[i]) {
      const V t = b[i];
      b[i] = b[i + 1];
      b[i + 1] = t;
    }
    b[i + 1] = b[i + 1] - lm[i] * b[i];
  }
  for (int i = n - 1; i >= 0; --i) {
    V v = b[i];
    if (i + 1 < n) v = v - u1[i] * b[i + 1];
    if (i + 2 < n) v = v - u2[i] * b[i + 2];
    b[i] = u0[i] * v;
  }
}
__device__ __forceinline__ void tri_solve(const TriWs& W, int n, cd* b) {
  tri_solve<double, cd>(W.u0, W.u1, W.u2, W.lm, W.piv, n, b);
}

// Apply Q (back = true: b <- Q b) or Q^H (b <- Q^H b) to b (n, complex V).
template <typename E, typename V>
__device__ void tri_apply_q(const E* A, const E* tau, int n, V* b) {
  using R = typename RealOf<V>::type;
  const int lane = threadIdx.x & 31;
  __syncwarp();
  for (int k = n - 2; k >= 0; --k) {
    const V tk = to_v(tau[k], V());
    if (tk.re == R(0) && tk.im == R(0)) continue;
    const E* vk = A + (size_t)k * n;
    V acc = mk(R(0), R(0));
    for (int i = lane; i < n; i += 32)
      if (i > k) cfmac(acc, to_v(vk[i], V()), b[i]);   // v^H b
    acc = mk(warp_sum(acc.re), warp_sum(acc.im));
    const V f = tk * acc;
    __syncwarp();
    for (int i = lane; i < n; i += 32)
      if (i > k) b[i] = b[i] - f * to_v(vk[i], V());
    __syncwarp();
  }
}

// Real reflectors on a real vector (real samples): half the work of the
// complex form.
__device__ void tri_apply_q_r(const double* A, const double* tau, int n, double* b) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  for (int k = n - 2; k >= 0; --k) {
    const double tk = tau[k];
    if (tk == 0.0) continue;
    const double* vk = A + (size_t)k * n;
    double acc = 0.0;
    for (int i = lane; i < n; i += 32)
      if (i > k) acc = fma(vk[i], b[i], acc);
    const double f = tk * warp_sum(acc);
    __syncwarp();
    for (int i = lane; i < n; i += 32)
      if (i > k) b[i] = fma(-f, vk[i], b[i]);
    __syncwarp();
  }
}
__device__ __forceinline__ double tri_norm2_r(const double* b, int n) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int i = lane; i < n; i += 32) s = fma(b[i], b[i], s);
  return warp_sum(s);
}

__device__ __forceinline__ double tri_norm2(const cd* b, int n) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int i = lane; i < n; i += 32) s += abs2(b[i]);
  return warp_sum(s);
}

struct TriResult {
  double lam_min, lam_2, lam_max;   // eigenvalues of G (T's, scaled back)
  double theta;                     // x^H G x
  int near_degenerate;              // lam_2 - lam_min <= 1e-4 lam_max
};

// Steps 2-4 by one warp, after the CTA's reduction of G 2^-ex (zero: G is the
// zero matrix): the eigenvalue brackets, x; fills res (eigenvalues).
template <typename E>
__device__ void tri_solve_lead(const TriWs& W, int n, bool zero, int ex, TriResult& res) {
  const int lane = threadIdx.x & 31;
  E* A = (E*)W.A;
  E* tau = (E*)W.tau;
  if (zero) {   // every vector is a null vector
    for (int i = lane; i < n; i += 32) W.x[i] = mk(i == 0 ? 1.0 : 0.0, 0.0);
    __syncwarp();
    res.lam_min = res.lam_2 = res.lam_max = 0.0;
    res.near_degenerate = 1;
    return;
  }
  const double gs = ldexp(1.0, ex);
  // Gershgorin interval of T; single-precision copies
  double glo = 1e300, ghi = -1e300;
  for (int i = lane; i < n; i += 32) {
    const double rad = (i > 0 ? fabs(W.e[i - 1]) : 0.0) + (i + 1 < n ? fabs(W.e[i]) : 0.0);
    glo = fmin(glo, W.d[i] - rad);
    ghi = fmax(ghi, W.d[i] + rad);
    const double e2 = i + 1 < n ? W.e[i] * W.e[i] : 0.0;
    W.e2[i] = e2;
    W.df[i] = (float)W.d[i];
    W.e2f[i] = (float)e2;
  }
  glo = -warp_max(-glo);
  ghi = warp_max(ghi);
  const double tnorm = fmax(fabs(glo), fabs(ghi));
  const double eps = 2.220446049250313e-16;
  glo -= 4.0 * eps * tnorm + 1e-300;
  ghi += 4.0 * eps * tnorm + 1e-300;
  __syncwarp();
  // 2. brackets of eigenvalues 0, 1 and n - 1
  const int which[3] = {0, n > 1 ? 1 : 0, n - 1};
  Bracket br[3] = {{glo, ghi}, {glo, ghi}, {glo, ghi}};
  // single-precision rounds while a bracket is wider than its floor
  const double fl = 1e-5 * tnorm;
  const float tiny_f = (float)(1e-30 * fmax(tnorm, 1e-8));
  for (int round = 0; round < 12; ++round) {
    int t = -1;
    for (int m = 2; m >= 0; --m)
      if (br[m].hi - br[m].lo > fl) t = m;
    if (t < 0) break;
    multisect<true>(W, n, t, br, 3, which, tiny_f);
  }
  // widen by the single-precision error bound; check the ends in double
  // precision (a wrong end falls back to the Gershgorin interval)
  for (int m = 0; m < 3; ++m) {
    br[m].lo = fmax(glo, br[m].lo - 4e-6 * tnorm);
    br[m].hi = fmin(ghi, br[m].hi + 4e-6 * tnorm);
  }
  {
    const int m = lane % 3, end = (lane / 3) & 1;
    const double sig = end ? br[m].hi : br[m].lo;
    const int c = lane < 6 ? sturm_count(W.d, W.e2, n, sig) : 0;
    const bool bad = lane < 6 && (end ? c <= which[m] : c > which[m]);
    const unsigned badm = __ballot_sync(0xffffffffu, bad);
    for (int m2 = 0; m2 < 3; ++m2)
      if (badm & (0x9u << m2)) br[m2] = Bracket{glo, ghi};
  }
  const double tol_abs = 8.0 * eps * tnorm;
  for (int round = 0; round < 40; ++round) {
    // isolated well enough: the inverse iteration contracts by 1e-4 per step
    const double w0 = br[0].hi - br[0].lo;
    if (w0 <= tol_abs || (n > 1 && br[1].lo > br[0].hi && w0 <= 1e-4 * (br[1].lo - br[0].hi)))
      break;
    multisect<false>(W, n, 0, br, 3, which, tiny_f);
  }
  if (n > 1) {
    for (int round = 0; round < 40; ++round) {
      const double w1 = br[1].hi - br[1].lo;
      if (w1 <= fmax(tol_abs, 1e-5 * fabs(br[1].hi))) break;
      multisect<false>(W, n, 1, br, 3, which, tiny_f);
    }
  }
  for (int round = 0; round < 40; ++round) {
    const double w2 = br[2].hi - br[2].lo;
    if (w2 <= fmax(tol_abs, 1e-7 * fabs(br[2].hi))) break;
    multisect<false>(W, n, 2, br, 3, which, tiny_f);
  }
  const double lam0 = 0.5 * (br[0].lo + br[0].hi);
  const double lam1 = n > 1 ? 0.5 * (br[1].lo + br[1].hi) : lam0;
  const double lamn = 0.5 * (br[2].lo + br[2].hi);
  // 3. inverse iteration (three steps) from a fixed start vector; 4. x = Q y
  tri_lu(W, n, lam0, eps * tnorm);
  if constexpr (sizeof(E) == sizeof(double)) {   // real: real vectors throughout
    double* y = (double*)W.z;
    for (int i = lane; i < n; i += 32) y[i] = 1.0 + 0.25 * (double)((i * 7) % 5);
    __syncwarp();
    for (int it = 0; it < 3; ++it) {
      tri_solve<double, double>(W.u0, W.u1, W.u2, W.lm, W.piv, n, y);
      __syncwarp();
      const double nz = tri_norm2_r(y, n);
      const double sc = nz > 0.0 ? rsqrt_safe(nz) : 1.0;
      for (int i = lane; i < n; i += 32) y[i] = sc * y[i];
      __syncwarp();
    }
    tri_apply_q_r((const double*)A, (const double*)tau, n, y);
    const double sc = rsqrt_safe(tri_norm2_r(y, n));
    for (int i = lane; i < n; i += 32) W.x[i] = mk(sc * y[i], 0.0);
    __syncwarp();
  } else {
    for (int i = lane; i < n; i += 32) W.z[i] = mk(1.0 + 0.25 * (double)((i * 7) % 5), 0.0);
    __syncwarp();
    for (int it = 0; it < 3; ++it) {
      tri_solve(W, n, W.z);
      __syncwarp();
      const double nz = tri_norm2(W.z, n);
      const double sc = nz > 0.0 ? rsqrt_safe(nz) : 1.0;
      for (int i = lane; i < n; i += 32) W.z[i] = sc * W.z[i];
      __syncwarp();
    }
    for (int i = lane; i < n; i += 32) W.x[i] = W.z[i];
    tri_apply_q<E, cd>(A, tau, n, W.x);
    const double sc = rsqrt_safe(tri_norm2(W.x, n));
    for (int i = lane; i < n; i += 32) W.x[i] = sc * W.x[i];
    __syncwarp();
  }
  res.lam_min = gs * lam0;
  res.lam_2 = gs * lam1;
  res.lam_max = gs * lamn;
  res.near_degenerate = n > 1 && (lam1 - lam0) <= 1e-4 * lamn ? 1 : 0;
}

// ------------------------------------------------------------------------
// Float-float helpers of the real samples' steps 2-5 (mixed path,
// cbp_tri_team.cuh): on this GPU a double-precision instruction holds a
// scheduler's double unit for ~64 cycles, and these steps are chains of them.
// With float-float values (~48 bits) on the single-precision units T's
// eigenvalues come out to ~1e-13 ||T||.

// Sturm count of T - sig I from the leading minors p_i (product form).  Each
// step's coefficients carry the power of two that returns the minors' size to
// about one, found a step earlier so that it stays off the chain (a step
// shrinks the minors by no more than the square of an off-diagonal entry, well
// inside the single-precision range); the chain of a step is one product and
// one sum with a single renormalisation.
__device__ __forceinline__ int sturm_count_x(const fx* d, const fx* e2, int n, fx sig) {
  fx pm = {1.f, 0.f}, p = fx_sub(d[0], sig);
  bool negp = fx_neg_sign(p) || fx_is_zero(p);
  int cnt = negp ? 1 : 0;
  float s = 1.f;
  for (int i = 1; i < n; ++i) {
    const fx a0 = fx_sub(d[i], sig), e = e2[i - 1];
    const fx a = {a0.hi * s, a0.lo * s};
    const fx b = fx_mul({e.hi * s, e.lo * s}, pm);
    const fx pn = fx_neg(fx_fnma(b, a, p));        // a p - b
    const float big = fmaxf(fabsf(p.hi), fabsf(pm.hi)) * s;
    pm = {p.hi * s, p.lo * s};
    const int ex = max(__float_as_int(big) & 0x7f800000, 27 << 23);
    s = __int_as_float(0x7f000000 - ex);
    p = pn;
    const bool neg = fx_is_zero(p) ? !negp : fx_neg_sign(p);
    cnt += neg != negp;
    negp = neg;
  }
  return cnt;
}

__device__ __forceinline__ fx fx_clamp_pivot(fx x, float tiny) {
  return fabsf(x.hi) >= tiny ? x : fx{fx_neg_sign(x) ? -tiny : tiny, 0.f};
}
// sum over the warp, renormalised once: the low parts gather every level's
// rounding term (five levels keep them within a few units of the high part's)
__device__ __forceinline__ fx warp_sum_x(fx v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float h = __shfl_xor_sync(0xffffffffu, v.hi, o), l = __shfl_xor_sync(0xffffffffu, v.lo, o);
    const fx s = fx_two_sum(v.hi, h);
    v = {s.hi, s.lo + (v.lo + l)};
  }
  return fx_norm(v.hi, v.lo);
}
// 1 / ||b|| in single precision (a scale for normalising)
__device__ __forceinline__ float inv_norm_x(const fx* b, int n) {
  const int lane = threadIdx.x & 31;
  float s = 0.f;
  for (int i = lane; i < n; i += 32) s = fmaf(b[i].hi, b[i].hi, s);
  s = warp_sum(s);
  return s > 0.f ? rsqrtf(s) : 1.f;
}

// G: the n x n matrix (row-major, global or shared memory).  Result in W.x
// (unit norm).  Every thread of the CTA calls; the CTA reduces G together, warp
// 0 does the rest and holds the result.
template <typename E>
__device__ TriResult tri_smallest(const TriWs& W, const cd* G, int n) {
  const int lane = threadIdx.x & 31;
  TriResult res = {};
  // the CTA reduces G 2^-ex, its largest diagonal entry in [1/2, 1)
  double gmax = 0.0;
  for (int i = lane; i < n; i += 32) gmax = fmax(gmax, G[(size_t)i * n + i].re);
  gmax = warp_max(gmax);
  const bool zero = !(gmax > 0.0);
  int ex = 0;
  if (!zero) {
    frexp(gmax, &ex);
    const double igs = ldexp(1.0, -ex);
    E* A = (E*)W.A;
    for (int idx = threadIdx.x; idx < n * n; idx += blockDim.x) {
      if constexpr (sizeof(E) == sizeof(double)) A[idx] = mk_e<E, double>(G[idx].re * igs, 0.0);
      else A[idx] = mk_e<E, double>(G[idx].re * igs, G[idx].im * igs);
    }
    __syncthreads();
    tri_reduce_block<E>(A, (E*)W.tau, (E*)W.w, W.d, W.e, n, (E*)W.part);
  }
  if (threadIdx.x >= 32) return res;
  tri_solve_lead<E>(W, n, zero, ex, res);
  // theta = x^H G x
  cd th = mk(0.0, 0.0);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int i = lane + 32 * c;
    if (i < n) {
      cd gx = mk(0.0, 0.0);
      for (int j = 0; j < n; ++j) cfmac(gx, G[(size_t)j * n + i], W.x[j]);   // (G x)_i
      cfmac(th, W.x[i], gx);
    }
  }
  res.theta = warp_sum(th.re);
  return res;
}
