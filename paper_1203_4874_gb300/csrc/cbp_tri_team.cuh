// Smallest eigenpair of a Hermitian (or real symmetric) n x n matrix, n <= 64,
// by a team of four warps -- one per scheduler of the SM: every sample's null
// vector and every pair's scale system.  The method is cbp_tri.cuh's
// (tridiagonal T, Sturm counts, inverse iteration, Newton steps in Olsen's
// form); this file arranges it for latency.
//
// What bounds these solves (measured on the target GPU, cycles of one warp): a
// dependent double FMA or add takes 64, an independent one still holds its
// scheduler for 48-64; a double shuffle and add 108; a double division 570, a
// double square root 612, a double fmax 115; a shared-memory store and load 36;
// a float FMA 5.  So a chain is counted in double instructions on the warp that
// carries it, and the four schedulers' double units are used side by side:
//   - reduction: the three other warps form A x while the lead warp forms the
//     reflector (square root and reciprocals by third-order Newton steps from a
//     single-precision seed), then all four update;
//   - brackets: one warp per wanted eigenvalue; single-precision rounds
//     entirely in single precision;
//   - inverse iteration and the correction equation: T is real, so complex right
//     sides are real ones side by side, one lane each;
//   - single-precision path: Q formed by four lanes per column in registers.
//
// Measured, cycles per solve before (the reduction alone on the CTA, the rest on
// one warp; complex samples on one warp throughout) and after, t1 + t2 = 32,
// M = 17, mixed path: real sample 550k -> 305k, complex sample 300k -> 135k,
// scale system (n = 34) 646k -> 215k; FP64 path, t1 + t2 = 20, M = 11: real 470k
// -> 325k, complex 1130k -> 450k, scale system (n = 22) 776k -> 440k.  Calls:
// kernel estimation of four 720p pairs 0.725 -> 0.443 ms, one 64 x 64 FP64 pair
// 0.66 -> 0.445 ms, 30 480p FP64 pairs 2.80 -> 1.71 ms.
// Included inside namespace cbp::(anonymous) after cbp_tri.cuh.

constexpr int kTeamThreads = 128;

// Barrier of the team (warps 0..3 of the CTA).
__device__ __forceinline__ void team_bar() {
  __syncwarp();
  asm volatile("barrier.sync.aligned 1, 128;" ::: "memory");
}

// Hand-over from the lead warp to the others (barrier 2): the lead warp's
// writes are visible to the others after team_take().
__device__ __forceinline__ void team_give() {
  __threadfence_block();
  __syncwarp();
  asm volatile("barrier.arrive.aligned 2, 128;" ::: "memory");
}
__device__ __forceinline__ void team_take() {
  __syncwarp();
  asm volatile("barrier.sync.aligned 2, 128;" ::: "memory");
}

// x != 0 without a double comparison (113 cycles); NaN counts as nonzero.
__device__ __forceinline__ bool nonzero(double x) { return !dzero(x); }
__device__ __forceinline__ bool nonzero(float x) { return x != 0.f; }
template <typename T> __device__ __forceinline__ bool nonzero(cpx<T> x) { return nonzero(x.re) || nonzero(x.im); }

// Reciprocal and reciprocal square root for 2^-100 < |x| < 2^100 (else the
// library's): the seed's relative error e is below 2^-20, one third-order step
// leaves e^3.
__device__ __forceinline__ bool mid_range(double x) {
  const int ex = dexp(x);
  return ex > 1023 - 100 && ex < 1023 + 100;
}
__device__ __forceinline__ double rcp3_from(double x, float seed) {
  const double y = (double)seed, e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double rsqrt3_from(double x, float seed) {
  const double y = (double)seed, e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}
__device__ __forceinline__ double rcp3(double x) {
  return mid_range(x) ? rcp3_from(x, __fdividef(1.0f, (float)x)) : 1.0 / x;
}
__device__ __forceinline__ double rsqrt3(double x) {
  return mid_range(x) ? rsqrt3_from(x, rsqrtf((float)x)) : 1.0 / sqrt(x);
}

// Sum over the warp's lanes.  Doubles: as 58-bit fixed-point numbers against the
// largest lane's exponent, added exactly by the integer reductions (three 21-bit
// pieces) and converted back -- the error is that of one rounding of the terms
// to 2^-57 of the largest and one of the result (measured over random terms:
// 1.1e-16 of the terms' sum against 2.4e-16 for the tree of double adds), in 240
// cycles against 650 for the tree.  Infinite, NaN and tiny sums take the tree.
struct FixedSum {
  int em;
  __device__ __forceinline__ explicit FixedSum(int ex) : em((int)__reduce_max_sync(0xffffffffu, (unsigned)ex)) {}
  __device__ __forceinline__ bool usable() const { return em != 0x7ff && em >= 64; }
  __device__ __forceinline__ double operator()(double v) const {
    const long long b = __double_as_longlong(v);
    const int ex = dexp(v), sh = min(em - ex, 62);
    long long m = ex ? ((b & 0xfffffffffffffll) | 0x10000000000000ll) << 4 : 0ll;
    m = (m + ((1ll << sh) >> 1)) >> sh;
    if (b < 0) m = -m;
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)(m & 0x1fffff));
    const unsigned mi = __reduce_add_sync(0xffffffffu, (unsigned)((m >> 21) & 0x1fffff));
    const int hi = __reduce_add_sync(0xffffffffu, (int)(m >> 42));
    const long long t = ((long long)hi << 42) + ((long long)mi << 21) + (long long)lo;
    return t ? __longlong_as_double(__double_as_longlong((double)t) + ((long long)(em - 1023 - 56) << 52)) : 0.0;
  }
};
__device__ __forceinline__ double lane_sum(double v) {
  const FixedSum f(dexp(v));
  return f.usable() ? f(v) : warp_sum(v);
}
__device__ __forceinline__ float lane_sum(float v) { return warp_sum(v); }
// two sums at once (doubles: on one exponent each, side by side)
__device__ __forceinline__ void lane_sum2(double& a, double& b) {
  const FixedSum f(dexp(a)), g(dexp(b));
  const double x = f.usable() ? f(a) : warp_sum(a);
  b = g.usable() ? g(b) : warp_sum(b);
  a = x;
}
__device__ __forceinline__ void lane_sum2(float& a, float& b) {
  a = warp_sum(a);
  b = warp_sum(b);
}

// The reflector H = I - tau v v^H, v = (1, x scl), with H^H (alpha, x) = (beta, 0),
// beta real; xn2 = ||x||^2.
// The second reciprocal's seed comes from single-precision copies of the same
// quantities, beside the Newton steps of the square root.
__device__ __forceinline__ void reflector(double alpha, double xn2, double& beta, double& tk, double& scl) {
  const double s2 = fma(alpha, alpha, xn2);
  double rs, nb, dn;
  if (mid_range(s2)) {
    const float sf = (float)s2, rf = rsqrtf(sf), df = __fdividef(1.0f, fmaf(sf, rf, fabsf((float)alpha)));
    rs = rsqrt3_from(s2, rf);
    nb = s2 * rs;
    dn = rcp3_from(fabs(alpha) + nb, df);
  } else {
    nb = sqrt(s2);
    rs = 1.0 / nb;
    dn = 1.0 / (fabs(alpha) + nb);
  }
  beta = -copysign(nb, alpha);
  tk = (fabs(alpha) + nb) * rs;             // (beta - alpha) / beta
  scl = copysign(dn, alpha);                // 1 / (alpha - beta)
}
__device__ __forceinline__ void reflector(cd alpha, double xn2, double& beta, cd& tk, cd& scl) {
  const double ai2 = alpha.im * alpha.im, s2 = fma(alpha.re, alpha.re, ai2 + xn2);
  double rs, nb, dn, dr;
  if (mid_range(s2)) {
    const float sf = (float)s2, rf = rsqrtf(sf), drf = fmaf(sf, rf, fabsf((float)alpha.re)), af = (float)alpha.im;
    const float df = __fdividef(1.0f, fmaf(drf, drf, af * af));
    rs = rsqrt3_from(s2, rf);
    nb = s2 * rs;
    dr = fabs(alpha.re) + nb;
    dn = rcp3_from(fma(dr, dr, ai2), df);
  } else {
    nb = sqrt(s2);
    rs = 1.0 / nb;
    dr = fabs(alpha.re) + nb;
    dn = 1.0 / fma(dr, dr, ai2);
  }
  beta = -copysign(nb, alpha.re);
  const double ib = -copysign(rs, alpha.re), ds = copysign(dr, alpha.re);   // 1 / beta, Re(alpha) - beta
  tk = mk(-ds * ib, -alpha.im * ib);
  scl = mk(ds * dn, -alpha.im * dn);
}
__device__ __forceinline__ void reflector(cf alpha, float xn2, float& beta, cf& tk, cf& scl) {
  beta = -copysignf(sqrtf(alpha.re * alpha.re + alpha.im * alpha.im + xn2), alpha.re);
  const float ib = 1.f / beta, dr = alpha.re - beta, dn = 1.f / (dr * dr + alpha.im * alpha.im);
  tk = mk(-dr * ib, -alpha.im * ib);
  scl = mk(dr * dn, -alpha.im * dn);
}
// acc -= a conj(b), as multiply-adds
__device__ __forceinline__ void fnmac_(double& acc, double a, double b) { acc = fma(-a, b, acc); }
template <typename T> __device__ __forceinline__ void fnmac_(cpx<T>& acc, cpx<T> a, cpx<T> b) {
  acc.re = fma(-a.re, b.re, fma(-a.im, b.im, acc.re));
  acc.im = fma(a.re, b.im, fma(-a.im, b.re, acc.im));
}
// Re(conj(a) b)
__device__ __forceinline__ double redot_(double a, double b) { return a * b; }
template <typename T> __device__ __forceinline__ T redot_(cpx<T> a, cpx<T> b) {
  return fma(a.re, b.re, a.im * b.im);
}

// Householder reduction by the team, results as tri_reduce_block's.  The lead warp
// carries the chain: a column's norm, its reflector, then -- from the others'
// partial products -- w, and at once the next column, whose norm it starts
// while the others (each on its own rows j, owner 1 + j mod 3) update the rest
// and form the next product.  A x is formed from the unscaled column x
// (A v = A e + scl A x).  part: [3][n].
//
// Doubles: rows one at a time (their double instructions are what counts, and
// those of rows past the end would be paid for even if predicated off); singles:
// four rows' loads in flight.
template <typename E>
__device__ __forceinline__ void reduce_rows(E* A, const E* tau, const E* w, int n, E* part) {
  const int own = (threadIdx.x >> 5) - 1;
  constexpr bool DP = sizeof(typename RealOf<E>::type) == sizeof(double);
  for (int k = 0; k + 1 < n; ++k) {
    const int k1 = k + 1;
    const E* vk = A + (size_t)k * n;
    const int j0 = k1 + 1 + (own - (k1 + 1) % 3 + 3) % 3;   // this warp's first row above k1
    team_take();
    CBP_COLS(n, {
      E a[4] = {Ops<E>::z(), Ops<E>::z(), Ops<E>::z(), Ops<E>::z()};
      if (i < n) {
        if constexpr (DP) {
          int j = j0;
          for (; j + 3 < n; j += 6) {
            const E x0 = A[(size_t)j * n + i], x1 = A[(size_t)(j + 3) * n + i];
            fma_(a[0], cj_(x0), cj_(vk[j]));
            fma_(a[1], cj_(x1), cj_(vk[j + 3]));
          }
          for (; j < n; j += 3) fma_(a[0], cj_(A[(size_t)j * n + i]), cj_(vk[j]));
        } else {
          for (int j = j0; j < n; j += 12) {
#pragma unroll
            for (int r = 0; r < 4; ++r)
              if (j + 3 * r < n) fma_(a[r], cj_(A[(size_t)(j + 3 * r) * n + i]), cj_(vk[j + 3 * r]));
          }
          a[0] = a[0] + a[2];
          a[1] = a[1] + a[3];
        }
        part[own * n + i] = a[0] + a[1];
      }
    });
    team_bar();
    team_bar();
    if (!nonzero(tau[k])) continue;
    // A <- A - v w^H - w v^H, rows above k1 (the lead warp takes row k1)
    CBP_COLS(n, {
      if (i > k1 && i < n) {
        const E wi = w[i];
        const E vi = vk[i];
        if constexpr (DP) {
          for (int j = j0; j < n; j += 3) {
            E t = A[(size_t)j * n + i];
            fnmac_(t, vk[j], wi);
            fnmac_(t, w[j], vi);
            A[(size_t)j * n + i] = t;
          }
        } else {
          for (int j = j0; j < n; j += 12) {
            E t[4];
            E vj[4];
            E wj[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              const int jr = min(j + 3 * r, n - 1);
              t[r] = A[(size_t)jr * n + i];
              vj[r] = vk[jr];
              wj[r] = w[jr];
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              fnmac_(t[r], vj[r], wi);
              fnmac_(t[r], wj[r], vi);
              if (j + 3 * r < n) A[(size_t)(j + 3 * r) * n + i] = t[r];
            }
          }
        }
      }
    });
  }
}
template <typename E>
__device__ void tri_reduce_team(E* A, E* tau, E* w, typename RealOf<E>::type* d,
                                typename RealOf<E>::type* e, int n, E* part) {
  using R = typename RealOf<E>::type;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp == 0) {
    if (n > 1) team_give();                    // row 0 is there
    E x[2];                                    // row k, columns lane and lane + 32
#pragma unroll
    for (int c = 0; c < 2; ++c) x[c] = lane + 32 * c < n ? A[lane + 32 * c] : Ops<E>::z();
    for (int k = 0; k + 1 < n; ++k) {
      const int k1 = k + 1;
      E* vk = A + (size_t)k * n;               // row k = conj(column k)
      R xn2 = R(0);
      CBP_COLS(n, {
        if (i > k1) xn2 += a2_(x[c]);
      });
      const E alpha = cj_(vk[k1]);
      xn2 = lane_sum(xn2);
      E tk = Ops<E>::z(), scl = Ops<E>::z();
      R beta = re_(alpha);
      const bool act = nonzero(xn2) || nonzero(im_(alpha));
      E v[2], av[2];
      R t2 = R(0);
      if (act) {
        reflector(alpha, xn2, beta, tk, scl);
        CBP_COLS(n, {
          v[c] = i == k1 ? Ops<E>::o() : Ops<E>::z();
          if (i > k1 && i < n) v[c] = mul_(cj_(x[c]), scl);
        });
        t2 = R(0.5) * a2_(tk);
      }
      team_bar();
      if (act) {
        // w = tau A v - (|tau|^2 / 2) Re(v^H A v) v
        R hp = R(0);
        CBP_COLS(n, {
          av[c] = Ops<E>::z();
          if (i > k && i < n) {
            av[c] = cj_(A[(size_t)k1 * n + i]);
            fma_(av[c], scl, part[i] + part[n + i] + part[2 * n + i]);
            hp += redot_(v[c], av[c]);
            av[c] = mul_(tk, av[c]);
          }
        });
        const R hc = t2 * lane_sum(hp);
        CBP_COLS(n, {
          if (i > k && i < n) {
            av[c] = av[c] - sc_(hc, v[c]);     // w
            w[i] = av[c];
            vk[i] = v[c];
          }
        });
      } else if (lane == 0) {
        vk[k1] = Ops<E>::o();
      }
      if (lane == 0) {
        d[k] = re_(vk[k]);
        e[k] = beta;
        tau[k] = tk;
      }
      team_bar();
      // the next row, updated here
      const E wk = act ? w[k1] : Ops<E>::z(), one = Ops<E>::o();
      CBP_COLS(n, {
        if (i > k && i < n) {
          x[c] = A[(size_t)k1 * n + i];
          if (act) {
            fnmac_(x[c], one, av[c]);
            fnmac_(x[c], wk, v[c]);
            A[(size_t)k1 * n + i] = x[c];
          }
        }
      });
      __syncwarp();
      if (k1 + 1 < n) team_give();
    }
    if (lane == 0) d[n - 1] = re_(A[(size_t)(n - 1) * n + n - 1]);
  } else {
    reduce_rows<E>(A, tau, w, n, part);
  }
  team_bar();
}

// ------------------------------------------------------------- brackets ---
// Single-precision multisection of the bracket [lo, hi] of eigenvalue t by one
// warp, 32 shifts a round, until it is at most fl wide.
__device__ __forceinline__ void bracket_f(const float* df, const float* e2f, int n, int t, float fl,
                                          float tiny, float& lo, float& hi) {
  const int lane = threadIdx.x & 31;
  for (int round = 0; round < 12 && hi - lo > fl; ++round) {
    const float sig = fmaf((hi - lo) * (1.f / 33.f), (float)(lane + 1), lo);
    const unsigned above = __ballot_sync(0xffffffffu, sturm_count_f(df, e2f, n, sig, tiny) > t);
    const int first = above ? __ffs(above) - 1 : 32;
    const float a = __shfl_sync(0xffffffffu, sig, first > 0 ? first - 1 : 0);
    const float b = __shfl_sync(0xffffffffu, sig, first < 32 ? first : 31);
    if (first > 0) lo = a;
    if (first < 32) hi = b;
  }
}

// sturm_count with the rescaling by powers of two on the exponent fields.
__device__ __forceinline__ double scale_exp(double x, int e) {
  return dexp(x) > 0 ? __longlong_as_double(__double_as_longlong(x) + ((long long)e << 52)) : x;
}
__device__ __forceinline__ int sturm_count_d(const double* d, const double* e2, int n, double sig) {
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
      const int sh = ex > 1023 + 400 ? -400 : ex < 1023 - 400 && ex > 0 ? 400 : 0;
      // one far below the other is as good as zero
      p = sh < 0 && dexp(p) <= 400 ? 0.0 : scale_exp(p, sh);
      pm = sh < 0 && dexp(pm) <= 400 ? 0.0 : scale_exp(pm, sh);
    }
  }
  return cnt;
}

// Sturm counts of T in double or float-float.
struct CountD {
  const double *d, *e2;
  int n;
  __device__ __forceinline__ int operator()(double sig) const { return sturm_count_d(d, e2, n, sig); }
};
struct CountX {
  const fx *d, *e2;
  int n;
  __device__ __forceinline__ int operator()(double sig) const { return sturm_count_x(d, e2, n, fx_of(sig)); }
};

// One multisection round of bracket b for eigenvalue t; the counts also narrow
// the bracket b1 of eigenvalue t + 1 from below while it overlaps b (JOINT).
// Loop control in single precision (a double comparison costs as much as a
// double add).
template <bool JOINT, class Cnt>
__device__ __forceinline__ void bracket_round(const Cnt& cnt, int t, Bracket& b, Bracket& b1) {
  const int lane = threadIdx.x & 31;
  const float h = (float)(b.hi - b.lo) * (1.f / 33.f);
  const double sig = b.lo + (double)(h * (float)(lane + 1));
  const int c = cnt(sig);
  const unsigned above = __ballot_sync(0xffffffffu, c > t);
  const int first = above ? __ffs(above) - 1 : 32;
  if (JOINT) {
    const unsigned ab1 = __ballot_sync(0xffffffffu, c > t + 1);
    const int f1 = ab1 ? __ffs(ab1) - 1 : 32;
    const double s = __shfl_sync(0xffffffffu, sig, f1 > 0 ? f1 - 1 : 0);
    const double s2 = __shfl_sync(0xffffffffu, sig, f1 < 32 ? f1 : 31);
    if (f1 > 0 && (float)(s - b1.lo) > 0.f) b1.lo = s;
    if (f1 < 32 && (float)(b1.hi - s2) > 0.f) b1.hi = s2;
  }
  const double lo = __shfl_sync(0xffffffffu, sig, first > 0 ? first - 1 : 0);
  const double hi = __shfl_sync(0xffffffffu, sig, first < 32 ? first : 31);
  if (first > 0) b.lo = lo;
  if (first < 32) b.hi = hi;
}

// Brackets of eigenvalues 0, 1 and n - 1 of T, warps 0..2 one each:
// single-precision rounds to 1e-5 ||T||, widened by their error bound and the
// ends checked by exact counts (a wrong end falls back to the Gershgorin
// interval), then counts `cnt` until eigenvalue 0 is isolated to 1e-4 of its
// gap, eigenvalue 1 known to 1e-5 and the largest to 1e-7 (all no finer than
// tol_abs).  lam[3] (shared): the midpoints.  bs: shared scratch of 6 doubles.
template <class Cnt>
__device__ void tri_brackets_team(const TriWs& W, const Cnt& cnt, int n, double glo, double ghi,
                                  double tnorm, double tol_abs, double* bs, double* lam) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int t = warp == 0 ? 0 : warp == 1 ? (n > 1 ? 1 : 0) : n - 1;
  Bracket b{glo, ghi};
  if (warp < 3) {
    float lo = (float)glo, hi = (float)ghi;
    bracket_f(W.df, W.e2f, n, t, (float)(1e-5 * tnorm), (float)(1e-30 * fmax(tnorm, 1e-8)), lo, hi);
    const double wid = 4e-6 * tnorm;
    b.lo = fmax(glo, (double)lo - wid);
    b.hi = fmin(ghi, (double)hi + wid);
    const int c = lane < 2 ? cnt(lane ? b.hi : b.lo) : 0;
    const bool bad = lane == 0 ? c > t : lane == 1 ? c <= t : false;
    if (__any_sync(0xffffffffu, bad)) b = Bracket{glo, ghi};
    if (lane == 0) {
      bs[2 * warp] = b.lo;
      bs[2 * warp + 1] = b.hi;
    }
  }
  team_bar();
  const float tolf = (float)tol_abs;
  if (warp == 0) {
    Bracket b1{bs[2], bs[3]};
    for (int round = 0; round < 40; ++round) {
      const float w0 = (float)(b.hi - b.lo);
      const float gap = n > 1 ? (float)(b1.lo - b.hi) : 0.f;
      if (!(w0 > tolf) || (gap > 0.f && w0 <= 1e-4f * gap)) break;
      if (gap > 0.f) bracket_round<false>(cnt, t, b, b1);
      else bracket_round<true>(cnt, t, b, b1);
    }
  } else if (warp < 3) {
    Bracket none{0.0, 0.0};
    const float rel = warp == 1 ? 1e-5f : 1e-7f;
    for (int round = 0; round < 40; ++round) {
      if (!((float)(b.hi - b.lo) > fmaxf(tolf, rel * fabsf((float)b.hi)))) break;
      bracket_round<false>(cnt, t, b, none);
    }
  }
  if (warp < 3 && lane == 0) lam[warp] = 0.5 * (b.lo + b.hi);
  team_bar();
}

// ------------------------------------------- tridiagonal LU and solves ---
__device__ __forceinline__ double fnma_(double a, double m, double b) { return fma(-m, b, a); }   // a - m b
__device__ __forceinline__ float fnma_(float a, float m, float b) { return fmaf(-m, b, a); }
__device__ __forceinline__ fx fnma_(fx a, fx m, fx b) { return fx_fnma(a, m, b); }
__device__ __forceinline__ double times_(double a, double b) { return a * b; }
__device__ __forceinline__ float times_(float a, float b) { return a * b; }
__device__ __forceinline__ fx times_(fx a, fx b) { return fx_mul(a, b); }
__device__ __forceinline__ double minus_(double a, double b) { return a - b; }
__device__ __forceinline__ float minus_(float a, float b) { return a - b; }
__device__ __forceinline__ fx minus_(fx a, fx b) { return fx_sub(a, b); }
__device__ __forceinline__ double neg_(double a) { return -a; }
__device__ __forceinline__ float neg_(float a) { return -a; }
__device__ __forceinline__ fx neg_(fx a) { return fx_neg(a); }
__device__ __forceinline__ double recip_(double a) { return rcp3(a); }
__device__ __forceinline__ float recip_(float a) { return 1.0f / a; }
__device__ __forceinline__ fx recip_(fx a) { return fx_div(fx{1.f, 0.f}, a); }
// |a| >= |b| (doubles: on the integer pipe)
__device__ __forceinline__ long long mag_(double a) { return __double_as_longlong(a) & 0x7fffffffffffffffll; }
__device__ __forceinline__ bool mag_ge(double a, double b) { return mag_(a) >= mag_(b); }
__device__ __forceinline__ bool mag_ge(float a, float b) { return fabsf(a) >= fabsf(b); }
__device__ __forceinline__ bool mag_ge(fx a, fx b) { return fabsf(a.hi) >= fabsf(b.hi); }
__device__ __forceinline__ double floor_pivot(double x, double tiny) {
  return mag_ge(x, tiny) ? x : (dneg(x) ? -tiny : tiny);
}
__device__ __forceinline__ float floor_pivot(float x, float tiny) { return clamp_pivot(x, tiny); }
__device__ __forceinline__ fx floor_pivot(fx x, fx tiny) { return fx_clamp_pivot(x, tiny.hi); }
__device__ __forceinline__ void zero_(double& a) { a = 0.0; }
__device__ __forceinline__ void zero_(float& a) { a = 0.f; }
__device__ __forceinline__ void zero_(fx& a) { a = fx{0.f, 0.f}; }

// LU of T - sig I with row interchanges as tri_lu, by lane 0, the running row
// in registers (the next row's entries are loaded ahead of its use).
template <typename R>
__device__ void tri_lu_r(const R* d, const R* e, R* u0, R* u1, R* u2, R* lm, int* pv, int n, R sig, R tiny) {
  if ((threadIdx.x & 31) != 0) return;
  R zero;
  zero_(zero);
  R a = minus_(d[0], sig), b = n > 1 ? e[0] : zero;
  R sub = b, dn = n > 1 ? d[1] : zero, en = n > 2 ? e[1] : zero;
  for (int i = 0; i + 1 < n; ++i) {
    const R dn2 = i + 2 < n ? d[i + 2] : zero, en2 = i + 3 < n ? e[i + 2] : zero;
    const R dr = minus_(dn, sig);
    // operands chosen first: both sides of a branch would be paid for
    const bool keep = mag_ge(a, sub);
    const R r = recip_(keep ? floor_pivot(a, tiny) : sub);
    const R m = times_(keep ? sub : a, r);
    u1[i] = keep ? b : dr;
    u2[i] = keep ? zero : en;
    pv[i] = keep ? 0 : 1;
    a = fnma_(keep ? dr : b, m, keep ? b : dr);
    b = keep ? en : neg_(times_(m, en));
    u0[i] = r;
    lm[i] = m;
    sub = en;
    dn = dn2;
    en = en2;
  }
  u0[n - 1] = recip_(floor_pivot(a, tiny));
}

// Solve (T - sig I) z = b in place for nr right sides, one lane each: entry i of
// side l at b[i * nr + l].  By one warp.
template <typename R>
__device__ void tri_solve_r(const R* u0, const R* u1, const R* u2, const R* lm, const int* pv, int n, R* b,
                            int nr) {
  const int l = threadIdx.x & 31;
  if (l < nr) {
    R cur = b[l];
    R nx = n > 1 ? b[nr + l] : cur, m = lm[0];
    int p = pv[0];
    for (int i = 0; i + 1 < n; ++i) {
      const int in = i + 2 < n ? i + 1 : i;                 // next step's entries, ahead of their use
      const R nx2 = b[(in + 1) * nr + l], m2 = lm[in];
      const int p2 = pv[in];
      const R top = p ? nx : cur, bot = p ? cur : nx;
      b[i * nr + l] = top;
      cur = fnma_(bot, m, top);
      nx = nx2;
      m = m2;
      p = p2;
    }
    R z1, z2;
    zero_(z1);
    zero_(z2);
    R a = cur, r0 = u0[n - 1];
    R r1, r2;
    zero_(r1);
    zero_(r2);
    for (int i = n - 1; i >= 0; --i) {
      const int in = i > 0 ? i - 1 : 0;
      const R an = b[in * nr + l], q0 = u0[in], q1 = u1[in], q2 = u2[in];
      const R z = times_(r0, fnma_(fnma_(a, r2, z2), r1, z1));
      b[i * nr + l] = z;
      z2 = z1;
      z1 = z;
      a = an;
      r0 = q0;
      r1 = q1;
      r2 = q2;
    }
  }
  __syncwarp();
}

// b <- Q b (back) or Q^H b by one warp, b in registers and the
// reflector's product summed by one chain.
__device__ __forceinline__ void mac_conj(cd& acc, cd v, cd b) { cfmac(acc, v, b); }
__device__ __forceinline__ void mac_conj(double& acc, double v, double b) { acc = fma(v, b, acc); }
__device__ __forceinline__ cd sum_all(cd a) {
  lane_sum2(a.re, a.im);
  return a;
}
__device__ __forceinline__ double sum_all(double a) { return lane_sum(a); }
__device__ __forceinline__ void sub_mul(cd& b, cd f, cd v) {
  b.re = fma(-f.re, v.re, fma(f.im, v.im, b.re));
  b.im = fma(-f.re, v.im, fma(-f.im, v.re, b.im));
}
__device__ __forceinline__ void sub_mul(double& b, double f, double v) { b = fma(-f, v, b); }
template <typename E>
__device__ void tri_apply_q_t(const E* A, const E* tau, int n, E* b, bool back) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  E bv[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) bv[c] = lane + 32 * c < n ? b[lane + 32 * c] : Ops<E>::z();
  for (int s = 0; s + 1 < n; ++s) {
    const int k = back ? n - 2 - s : s;
    const E* vk = A + (size_t)k * n;
    E acc = Ops<E>::z(), v[2];
    CBP_COLS(n, {
      v[c] = Ops<E>::z();
      if (i > k && i < n) {
        v[c] = vk[i];
        mac_conj(acc, v[c], bv[c]);            // v^H b
      }
    });
    const E f = mul_(back ? tau[k] : cj_(tau[k]), sum_all(acc));
    CBP_COLS(n, {
      if (i > k && i < n) sub_mul(bv[c], f, v[c]);
    });
  }
#pragma unroll
  for (int c = 0; c < 2; ++c)
    if (lane + 32 * c < n) b[lane + 32 * c] = bv[c];
  __syncwarp();
}
// the same for a real sample's float-float reflectors
__device__ void tri_apply_q_t(const fx* A, const fx* tau, int n, fx* b, bool back) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  fx bv[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) bv[c] = lane + 32 * c < n ? b[lane + 32 * c] : fx{0.f, 0.f};
  for (int s = 0; s + 1 < n; ++s) {
    const int k = back ? n - 2 - s : s;
    const fx* vk = A + (size_t)k * n;
    fx_acc acc;
    fx v[2];
    CBP_COLS(n, {
      v[c] = fx{0.f, 0.f};
      if (i > k && i < n) {
        v[c] = vk[i];
        acc.mac(v[c], bv[c]);
      }
    });
    const fx f = fx_mul(tau[k], warp_sum_x(acc.value()));
    CBP_COLS(n, {
      if (i > k && i < n) bv[c] = fx_fnma(bv[c], f, v[c]);
    });
  }
#pragma unroll
  for (int c = 0; c < 2; ++c)
    if (lane + 32 * c < n) b[lane + 32 * c] = bv[c];
  __syncwarp();
}

__device__ __forceinline__ double norm2_t(const cd* b, int n) {
  double s = 0.0;
  for (int i = threadIdx.x & 31; i < n; i += 32) s += abs2(b[i]);
  return lane_sum(s);
}
// 1 / ||b|| of a warp's vector (n entries), as a double scale.
__device__ __forceinline__ double inv_norm(const double* b, int n) {
  double s = 0.0;
  for (int i = threadIdx.x & 31; i < n; i += 32) s = fma(b[i], b[i], s);
  s = lane_sum(s);
  return s > 0.0 ? rsqrt3(s) : 1.0;
}

// What the team shares besides TriWs.
struct TeamWs {
  double bs[6], lam[3], gs, tnorm, th[4];
  int steps;
};

// Largest diagonal entry of G, by every warp for itself.
__device__ __forceinline__ double diag_max(const cd* G, int n) {
  const int lane = threadIdx.x & 31;
  double g = 0.0;
  for (int i = lane; i < n; i += 32) g = fmax(g, G[(size_t)i * n + i].re);
  return warp_max(g);
}

// Column i of Q = H_0 ... H_{n-2} by four lanes, lane p its rows 4 jj + p in
// registers (NR = n / 4 rounded up); row stride n + 1.
template <int NR>
__device__ __forceinline__ void form_q(const cf* A, const cf* tau, int n, int i, cf* Q) {
  const int p = threadIdx.x & 3;
  cf q[NR];
#pragma unroll
  for (int jj = 0; jj < NR; ++jj) q[jj] = mk(4 * jj + p == i ? 1.f : 0.f, 0.f);
  for (int k = n - 2; k >= 0; --k) {
    const cf* vk = A + (size_t)k * n;
    cf v[NR], s0 = mk(0.f, 0.f), s1 = s0;
#pragma unroll
    for (int jj = 0; jj < NR; ++jj) {
      const int j = 4 * jj + p;
      v[jj] = j > k && j < n ? vk[j] : mk(0.f, 0.f);
      cfmac(jj & 1 ? s1 : s0, v[jj], q[jj]);
    }
    s0 = s0 + s1;
    s0.re += __shfl_xor_sync(0xffffffffu, s0.re, 1);
    s0.im += __shfl_xor_sync(0xffffffffu, s0.im, 1);
    s0.re += __shfl_xor_sync(0xffffffffu, s0.re, 2);
    s0.im += __shfl_xor_sync(0xffffffffu, s0.im, 2);
    const cf f = tau[k] * s0;
#pragma unroll
    for (int jj = 0; jj < NR; ++jj) q[jj] = q[jj] - f * v[jj];
  }
#pragma unroll
  for (int jj = 0; jj < NR; ++jj) {
    const int j = 4 * jj + p;
    if (j < n && i < n) Q[(size_t)j * (n + 1) + i] = q[jj];
  }
}

// The solve in single precision, then Newton steps in Olsen's form against G
// itself, by the team: the residual G x - theta x in double precision, the
// correction equation solved through the single-precision T (contraction
// ~n u ||T|| / gap per step), until the correction stops shrinking or falls
// below 1e-10.  For complex matrices whose two smallest eigenvalues single
// precision separates by more than 3e-5 lambda_max (contraction <~ 0.1 per step,
// at most 12 steps), or separates at all with a gap above 1e-5 lambda_max (at
// most 24 steps, which must bring the correction below 1e-9); returns
// (uniformly) false, having changed nothing but the work area, for the others
// (they take tri_solve_team).  The result is in W.x.
__device__ bool tri_solve_team_sp(const TriWs& W, TeamWs& S, const cd* G, int n, TriResult& res,
                                  long long* tk, const cfx* Gx) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tid = threadIdx.x;
  cf* A = (cf*)W.A;
  cf* tau = (cf*)W.tau;
  float* d = W.df;
  float* e = (float*)W.e;
  const double gmax = diag_max(G, n);
  if (!(gmax > 0.0)) return false;
  int ex;
  frexp(gmax, &ex);
  const double gs = ldexp(1.0, ex), igs = ldexp(1.0, -ex);
  const float igsf = (float)igs;
  for (int idx = tid; idx < n * n; idx += kTeamThreads)
    A[idx] = mk((float)G[idx].re * igsf, (float)G[idx].im * igsf);
  team_bar();
  if (tk && tid == 0) tk[0] = clock64();
  tri_reduce_team<cf>(A, tau, (cf*)W.w, d, e, n, (cf*)W.part);
  if (tk && tid == 0) tk[1] = clock64();
  float glo = 1e30f, ghi = -1e30f;
  for (int i = lane; i < n; i += 32) {
    const float rad = (i > 0 ? fabsf(e[i - 1]) : 0.f) + (i + 1 < n ? fabsf(e[i]) : 0.f);
    glo = fminf(glo, d[i] - rad);
    ghi = fmaxf(ghi, d[i] + rad);
    if (warp == 0) W.e2f[i] = i + 1 < n ? e[i] * e[i] : 0.f;
  }
  glo = -warp_max(-glo);
  ghi = warp_max(ghi);
  const float tn = fmaxf(fabsf(glo), fabsf(ghi)), eb = 4e-6f * tn;
  team_bar();
  if (warp < 3) {
    float lo = glo - eb, hi = ghi + eb;
    bracket_f(d, W.e2f, n, warp == 2 ? n - 1 : warp, 0.25f * eb, 1e-30f * fmaxf(tn, 1e-8f), lo, hi);
    if (lane == 0) {
      S.bs[2 * warp] = (double)lo;
      S.bs[2 * warp + 1] = (double)hi;
    }
  }
  team_bar();
  const double lam0 = 0.5 * (S.bs[0] + S.bs[1]), lam1 = 0.5 * (S.bs[2] + S.bs[3]);
  const double lamn = 0.5 * (S.bs[4] + S.bs[5]);
  const double sep = (S.bs[2] - (double)eb) - (S.bs[1] + (double)eb);
  const bool wide = sep > 3e-5 * lamn;
  if (!wide && !(sep > 0.0 && lam1 - lam0 > 1e-5 * lamn)) return false;
  if (tk && tid == 0) tk[2] = clock64();
  float* u0 = (float*)W.u0;
  float* u1 = (float*)W.u1;
  float* u2 = (float*)W.u2;
  float* lm = (float*)W.lm;
  const float tinyf = 1.2e-7f * tn;
  cf* Q = A + (size_t)n * n;
  const int lq = n + 1;
  float* y = (float*)W.z;
  // warp 0: inverse iteration (three steps) on T; warps 1..3 beside it, then
  // all: Q, eight columns at a time
  if (warp == 0) {
    tri_lu_r<float>(d, e, u0, u1, u2, lm, W.piv, n, (float)lam0, tinyf);
    for (int i = lane; i < n; i += 32) y[i] = 1.0f + 0.25f * (float)((i * 7) % 5);
    __syncwarp();
    for (int it = 0; it < 3; ++it) {
      tri_solve_r<float>(u0, u1, u2, lm, W.piv, n, y, 1);
      float s2 = 0.f;
      for (int i = lane; i < n; i += 32) s2 = fmaf(y[i], y[i], s2);
      s2 = warp_sum(s2);
      const float sc = s2 > 0.f ? rsqrtf(s2) : 1.f;
      for (int i = lane; i < n; i += 32) y[i] *= sc;
      __syncwarp();
    }
  }
  for (int g = warp == 0 ? 3 : warp - 1; 8 * g < n; g += 4) {
    if (n <= 32) form_q<8>(A, tau, n, 8 * g + (lane >> 2), Q);
    else form_q<16>(A, tau, n, 8 * g + (lane >> 2), Q);
  }
  team_bar();
  // x = Q y
  if (warp == 0) {
    float s2 = 0.f;
    cf xv[2];
    CBP_COLS(n, {
      cf acc = mk(0.f, 0.f), acc1 = acc;
      if (i < n) {
        int j = 0;
        for (; j + 1 < n; j += 2) {
          acc = acc + y[j] * Q[(size_t)i * lq + j];
          acc1 = acc1 + y[j + 1] * Q[(size_t)i * lq + j + 1];
        }
        if (j < n) acc = acc + y[j] * Q[(size_t)i * lq + j];
      }
      xv[c] = acc + acc1;
      s2 += abs2(xv[c]);
    });
    const float sc = rsqrtf(warp_sum(s2));
    CBP_COLS(n, {
      if (i < n) W.x[i] = mk((double)(sc * xv[c].re), (double)(sc * xv[c].im));
    });
  }
  team_bar();
  if (tk && tid == 0) tk[3] = clock64();
  // Newton steps against G.  x is kept to a few units of its norm only and
  // normalised at the end: theta is the quotient x^H G x / x^H x.
  cd* gp = (cd*)W.part;          // [4][n] partial G x (or cfx: the same bytes)
  cf* rq = (cf*)W.r;             // r in single precision
  cf* yq = rq + n;               // x in single precision
  float* sv = (float*)W.q;       // [n][4]: u.re, u.im, z.re, z.im
  float* yt = (float*)W.w;       // [n][2]: Q^H x
  cf* dq = (cf*)W.z;             // the correction in T coordinates
  double dprev = 1e300, dn = 1e300;
  const int max_it = wide ? 12 : 24;
  const double stall = wide ? 0.25 : 0.5;
  cfx* xx = (cfx*)(gp + 4 * n);  // x in float-float (float-float residual)
  if (Gx) {
    if (warp == 0)
      for (int i = lane; i < n; i += 32) xx[i] = cfx_of(W.x[i]);
    team_bar();
  }
  for (int it = 0; it < max_it; ++it) {
    // this warp's rows of G x
    CBP_COLS(n, {
      if (i < n) {
        if (Gx) {
          cfx_acc acc;
          for (int j = warp; j < n; j += 4) acc.macc(Gx[(size_t)j * n + i], xx[j]);
          ((cfx*)gp)[warp * n + i] = acc.value();
        } else {
          cd acc = mk(0.0, 0.0);
          for (int j = warp; j < n; j += 4) cfmac(acc, G[(size_t)j * n + i], W.x[j]);
          gp[warp * n + i] = acc;
        }
      }
    });
    team_bar();
    // every warp: theta; warp 0 and 1: r; warp 2: LU
    cd gx[2], xv[2];
    double th = 0.0, xs = 0.0;
    CBP_COLS(n, {
      gx[c] = xv[c] = mk(0.0, 0.0);
      if (i < n) {
        xv[c] = W.x[i];
        if (Gx) {
          const cfx* g = (const cfx*)gp;
          cfx s = g[i];
          for (int w = 1; w < 4; ++w) {
            s.re = fx_add(s.re, g[w * n + i].re);
            s.im = fx_add(s.im, g[w * n + i].im);
          }
          gx[c] = cfx_val(s);
        } else {
          gx[c] = (gp[i] + gp[n + i]) + (gp[2 * n + i] + gp[3 * n + i]);
        }
        th += redot_(xv[c], gx[c]);
        xs += abs2(xv[c]);
      }
    });
    lane_sum2(th, xs);
    const double theta = th * rcp3(xs);
    if (warp == 2) {
      tri_lu_r<float>(d, e, u0, u1, u2, lm, W.piv, n, (float)(theta * igs), tinyf);
    } else if (warp == 0) {
      CBP_COLS(n, {
        if (i < n) {
          rq[i] = mk((float)fma(-theta, xv[c].re, gx[c].re), (float)fma(-theta, xv[c].im, gx[c].im));
          yq[i] = mk((float)xv[c].re, (float)xv[c].im);
        }
      });
    }
    team_bar();
    // r~ = Q^H r (warp 0), y~ = Q^H x (warp 1): lane i column i of Q
    if (warp < 2) {
      const cf* src = warp ? yq : rq;
      for (int i = lane; i < n; i += 32) {
        cf a0 = mk(0.f, 0.f), a1 = a0;
        int j = 0;
        for (; j + 1 < n; j += 2) {
          cfmac(a0, Q[(size_t)j * lq + i], src[j]);
          cfmac(a1, Q[(size_t)(j + 1) * lq + i], src[j + 1]);
        }
        if (j < n) cfmac(a0, Q[(size_t)j * lq + i], src[j]);
        a0 = a0 + a1;
        sv[4 * i + 2 * warp] = a0.re;
        sv[4 * i + 2 * warp + 1] = a0.im;
        if (warp) {
          yt[2 * i] = a0.re;
          yt[2 * i + 1] = a0.im;
        }
      }
    }
    team_bar();
    if (warp == 0) {
      tri_solve_r<float>(u0, u1, u2, lm, W.piv, n, sv, 4);     // u and z
      cf nu = mk(0.f, 0.f), de = nu;
      for (int i = lane; i < n; i += 32) {
        const cf yv = mk(yt[2 * i], yt[2 * i + 1]);
        cfmac(nu, yv, mk(sv[4 * i], sv[4 * i + 1]));
        cfmac(de, yv, mk(sv[4 * i + 2], sv[4 * i + 3]));
      }
      lane_sum2(nu.re, nu.im);
      lane_sum2(de.re, de.im);
      const float dd = abs2(de);
      const cf epsn = dd > 0.f ? (1.0f / dd) * (nu * conj(de)) : mk(0.f, 0.f);
      for (int i = lane; i < n; i += 32)
        dq[i] = igsf * (epsn * mk(sv[4 * i + 2], sv[4 * i + 3]) - mk(sv[4 * i], sv[4 * i + 1]));
    }
    team_bar();
    // x += Q d~
    if (warp == 0) {
      float d2 = 0.f;
      for (int i = lane; i < n; i += 32) {
        cf a0 = mk(0.f, 0.f), a1 = a0;
        int j = 0;
        for (; j + 1 < n; j += 2) {
          cfma(a0, Q[(size_t)i * lq + j], dq[j]);
          cfma(a1, Q[(size_t)i * lq + j + 1], dq[j + 1]);
        }
        if (j < n) cfma(a0, Q[(size_t)i * lq + j], dq[j]);
        a0 = a0 + a1;
        const cd xn = W.x[i] + mk((double)a0.re, (double)a0.im);
        W.x[i] = xn;
        if (Gx) xx[i] = cfx_of(xn);
        d2 += abs2(a0);
      }
      d2 = warp_sum(d2);
      if (lane == 0) S.th[0] = (double)sqrtf(d2);
    }
    team_bar();
    dn = S.th[0];
    if (dn < 1e-10 || dn > stall * dprev) break;
    dprev = dn;
  }
  if (warp == 0) {
    const double sc = rsqrt3(norm2_t(W.x, n));
    for (int i = lane; i < n; i += 32) W.x[i] = sc * W.x[i];
  }
  team_bar();
  if (!wide && !(dn < 1e-9)) return false;
  res.lam_min = gs * lam0;
  res.lam_2 = gs * lam1;
  res.lam_max = gs * lamn;
  res.near_degenerate = (lam1 - lam0) <= 1e-4 * lamn ? 1 : 0;
  S.gs = gs;
  return true;
}

// Gershgorin interval of the double T, its squares and single-precision copies
// (written by warp 0); every warp returns the same interval and norm.
__device__ __forceinline__ void tri_bounds(const TriWs& W, int n, double eps, double& glo, double& ghi,
                                           double& tnorm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  glo = 1e300;
  ghi = -1e300;
  for (int i = lane; i < n; i += 32) {
    const double rad = (i > 0 ? fabs(W.e[i - 1]) : 0.0) + (i + 1 < n ? fabs(W.e[i]) : 0.0);
    glo = fmin(glo, W.d[i] - rad);
    ghi = fmax(ghi, W.d[i] + rad);
    if (warp == 0) {
      const double e2 = i + 1 < n ? W.e[i] * W.e[i] : 0.0;
      W.e2[i] = e2;
      W.df[i] = (float)W.d[i];
      W.e2f[i] = (float)e2;
    }
  }
  glo = -warp_max(-glo);
  ghi = warp_max(ghi);
  tnorm = fmax(fabs(glo), fabs(ghi));
  glo -= eps * tnorm + 1e-300;
  ghi += eps * tnorm + 1e-300;
  team_bar();
}

// Steps 1-4 in double precision (E = cd or double) by the team; FFR (real samples
// of the mixed path, up to kFloatFloatN unknowns): from T on in float-float, the
// reflectors' copies overwriting the double ones in place.  Fills res, S.gs,
// S.tnorm; returns the number of refinement steps to take.
template <typename E, bool FFR>
__device__ int tri_solve_team(const TriWs& W, TeamWs& S, const cd* G, int n, int steps_far,
                              int steps_near, double refine_gap, TriResult& res, long long* tk) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tid = threadIdx.x;
  E* A = (E*)W.A;
  E* tau = (E*)W.tau;
  const double gmax = diag_max(G, n);
  if (!(gmax > 0.0)) {   // zero matrix: every vector is a null vector
    if (warp == 0)
      for (int i = lane; i < n; i += 32) W.x[i] = mk(i == 0 ? 1.0 : 0.0, 0.0);
    res.lam_min = res.lam_2 = res.lam_max = 0.0;
    res.near_degenerate = 1;
    S.gs = 1.0;
    S.tnorm = 0.0;
    team_bar();
    return 0;
  }
  int ex;
  frexp(gmax, &ex);
  const double gs = ldexp(1.0, ex), igs = ldexp(1.0, -ex);
  for (int idx = tid; idx < n * n; idx += kTeamThreads) {
    if constexpr (sizeof(E) == sizeof(double)) A[idx] = G[idx].re * igs;
    else A[idx] = mk(G[idx].re * igs, G[idx].im * igs);
  }
  team_bar();
  if (tk && tid == 0) tk[0] = clock64();
  tri_reduce_team<E>(A, tau, (E*)W.w, W.d, W.e, n, (E*)W.part);
  if (tk && tid == 0) tk[1] = clock64();
  const double eps = 2.220446049250313e-16;
  double glo, ghi, tnorm;
  tri_bounds(W, n, FFR ? 4e-13 : 4.0 * eps, glo, ghi, tnorm);
  fx* dx = (fx*)W.d;
  fx* ex_ = (fx*)W.e;
  fx* e2x = (fx*)W.e2;
  fx* Ax = (fx*)W.A;
  fx* taux = (fx*)W.tau;
  if constexpr (FFR) {
    // T and the reflectors (rows k, entries i > k) in float-float, in place
    if (warp == 0)
      for (int i = lane; i < n; i += 32) {
        const double dv = W.d[i], ev = W.e[i], e2 = W.e2[i], tv = ((const double*)W.tau)[i];
        dx[i] = fx_of(dv);
        ex_[i] = fx_of(ev);
        e2x[i] = fx_of(e2);
        taux[i] = fx_of(tv);
      }
    for (int k = warp; k < n; k += 4)
      for (int i = lane; i < n; i += 32)
        if (i > k) {
          const double v = ((const double*)W.A)[(size_t)k * n + i];
          Ax[(size_t)k * n + i] = fx_of(v);
        }
    team_bar();
    tri_brackets_team(W, CountX{dx, e2x, n}, n, glo, ghi, tnorm, 1e-13 * tnorm, S.bs, S.lam);
  } else {
    tri_brackets_team(W, CountD{W.d, W.e2, n}, n, glo, ghi, tnorm, 8.0 * eps * tnorm, S.bs, S.lam);
  }
  if (tk && tid == 0) tk[2] = clock64();
  const double lam0 = S.lam[0], lam1 = n > 1 ? S.lam[1] : lam0, lamn = S.lam[2];
  // inverse iteration (three steps) from a fixed start vector; x = Q y
  if (warp == 0) {
    if constexpr (FFR) {
      fx* u0 = (fx*)W.u0;
      fx* u1 = (fx*)W.u1;
      fx* u2 = (fx*)W.u2;
      fx* lm = (fx*)W.lm;
      tri_lu_r<fx>(dx, ex_, u0, u1, u2, lm, W.piv, n, fx_of(lam0), fx{(float)(1e-14 * tnorm), 0.f});
      fx* y = (fx*)W.z;
      for (int i = lane; i < n; i += 32) y[i] = fx{1.0f + 0.25f * (float)((i * 7) % 5), 0.f};
      __syncwarp();
      for (int it = 0; it < 3; ++it) {
        tri_solve_r<fx>(u0, u1, u2, lm, W.piv, n, y, 1);
        const float sc = inv_norm_x(y, n);
        for (int i = lane; i < n; i += 32) y[i] = fx_scale(y[i], sc);
        __syncwarp();
      }
      tri_apply_q_t(Ax, taux, n, y, true);
      for (int i = lane; i < n; i += 32) W.x[i] = mk(fx_val(y[i]), 0.0);
      __syncwarp();
      const double sc = rsqrt3(norm2_t(W.x, n));
      for (int i = lane; i < n; i += 32) W.x[i] = sc * W.x[i];
    } else {
      tri_lu_r<double>(W.d, W.e, W.u0, W.u1, W.u2, W.lm, W.piv, n, lam0, eps * tnorm);
      double* y = (double*)W.z;
      for (int i = lane; i < n; i += 32) y[i] = 1.0 + 0.25 * (double)((i * 7) % 5);
      __syncwarp();
      for (int it = 0; it < 3; ++it) {
        tri_solve_r<double>(W.u0, W.u1, W.u2, W.lm, W.piv, n, y, 1);
        const double sc = inv_norm(y, n);
        for (int i = lane; i < n; i += 32) y[i] = sc * y[i];
        __syncwarp();
      }
      E* xe = (E*)W.r;               // y as a vector of E, then Q y
      for (int i = lane; i < n; i += 32) xe[i] = mk_e<E, double>(y[i], 0.0);
      tri_apply_q_t(A, tau, n, xe, true);
      double s2 = 0.0;
      for (int i = lane; i < n; i += 32) s2 += a2_(xe[i]);
      const double sc = rsqrt3(lane_sum(s2));
      for (int i = lane; i < n; i += 32) W.x[i] = sc * to_cd(xe[i]);
    }
  }
  team_bar();
  if (tk && tid == 0) tk[3] = clock64();
  res.lam_min = gs * lam0;
  res.lam_2 = gs * lam1;
  res.lam_max = gs * lamn;
  res.near_degenerate = n > 1 && (lam1 - lam0) <= 1e-4 * lamn ? 1 : 0;
  S.gs = gs;
  S.tnorm = tnorm;
  const bool near = n > 1 && (lam1 - lam0) <= refine_gap * lamn;
  return near ? steps_near : steps_far;
}

// One refinement step by the team after r = (exact operator) x: Olsen's
// correction through T, the two projections and the factorisation on three
// warps at once, all right sides of the two solves side by side.
template <typename E, bool FFR>
__device__ void tri_olsen_team(const TriWs& W, TeamWs& S, int n) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int NR = sizeof(E) == sizeof(double) ? 2 : 4;   // right sides: (u, z) x (re, im)
  const double gs = S.gs, tnorm = S.tnorm, igs = 1.0 / gs;  // powers of two
  double th = 0.0;
  for (int i = lane; i < n; i += 32) th += redot_(W.x[i], W.r[i]);
  const double theta = lane_sum(th);
  if constexpr (FFR) {
    const fx* Ax = (const fx*)W.A;
    const fx* taux = (const fx*)W.tau;
    fx* u0 = (fx*)W.u0;
    fx* u1 = (fx*)W.u1;
    fx* u2 = (fx*)W.u2;
    fx* lm = (fx*)W.lm;
    fx* rt = (fx*)W.w;             // Q^T r
    fx* yt = rt + n;               // Q^T x
    fx* sv = (fx*)W.q;             // [n][2]: u, z
    if (warp == 0) {
      for (int i = lane; i < n; i += 32) rt[i] = fx_of(W.r[i].re - theta * W.x[i].re);
      tri_apply_q_t(Ax, taux, n, rt, false);
      for (int i = lane; i < n; i += 32) sv[2 * i] = rt[i];
    } else if (warp == 1) {
      for (int i = lane; i < n; i += 32) yt[i] = fx_of(W.x[i].re);
      tri_apply_q_t(Ax, taux, n, yt, false);
      for (int i = lane; i < n; i += 32) sv[2 * i + 1] = yt[i];
    } else if (warp == 2) {
      tri_lu_r<fx>((const fx*)W.d, (const fx*)W.e, u0, u1, u2, lm, W.piv, n, fx_of(theta * igs),
                   fx{(float)(1e-14 * tnorm), 0.f});
    }
    team_bar();
    if (warp == 0) {
      tri_solve_r<fx>(u0, u1, u2, lm, W.piv, n, sv, 2);
      fx_acc nu, de;
      for (int i = lane; i < n; i += 32) {
        nu.mac(yt[i], sv[2 * i]);
        de.mac(yt[i], sv[2 * i + 1]);
      }
      const fx nuv = warp_sum_x(nu.value()), dev = warp_sum_x(de.value());
      const fx ep = fx_is_zero(dev) ? fx{0.f, 0.f} : fx_div(nuv, dev);
      fx* zt = (fx*)W.z;
      const float ig = (float)igs;   // a power of two: exact
      for (int i = lane; i < n; i += 32) zt[i] = fx_scale(fx_sub(fx_mul(ep, sv[2 * i + 1]), sv[2 * i]), ig);
      tri_apply_q_t(Ax, taux, n, zt, true);
      for (int i = lane; i < n; i += 32) W.x[i] = mk(W.x[i].re + fx_val(zt[i]), 0.0);
    }
  } else {
    const E* A = (const E*)W.A;
    const E* tau = (const E*)W.tau;
    const double eps = 2.220446049250313e-16;
    E* rt = (E*)W.z;               // Q^H r
    E* yt = (E*)W.w;               // Q^H x
    double* sv = NR == 4 ? (double*)W.part : (double*)W.q;   // [n][NR]: u, z
    if (warp == 0) {
      for (int i = lane; i < n; i += 32)
        rt[i] = mk_e<E, double>(fma(-theta, W.x[i].re, W.r[i].re), fma(-theta, W.x[i].im, W.r[i].im));
      tri_apply_q_t(A, tau, n, rt, false);
      for (int i = lane; i < n; i += 32) {
        sv[NR * i] = re_(rt[i]);
        if (NR == 4) sv[NR * i + 1] = im_(rt[i]);
      }
    } else if (warp == 1) {
      for (int i = lane; i < n; i += 32) yt[i] = mk_e<E, double>(W.x[i].re, W.x[i].im);
      tri_apply_q_t(A, tau, n, yt, false);
      for (int i = lane; i < n; i += 32) {
        sv[NR * i + NR / 2] = re_(yt[i]);
        if (NR == 4) sv[NR * i + 3] = im_(yt[i]);
      }
    } else if (warp == 2) {
      tri_lu_r<double>(W.d, W.e, W.u0, W.u1, W.u2, W.lm, W.piv, n, theta * igs, eps * tnorm);
    }
    team_bar();
    if (warp == 0) {
      tri_solve_r<double>(W.u0, W.u1, W.u2, W.lm, W.piv, n, sv, NR);
      auto side = [&](int i, int h) { return mk_e<E, double>(sv[NR * i + h * (NR / 2)], NR == 4 ? sv[NR * i + h * (NR / 2) + 1] : 0.0); };
      E nu = Ops<E>::z(), de = Ops<E>::z();
      for (int i = lane; i < n; i += 32) {
        mac_conj(nu, yt[i], side(i, 0));
        mac_conj(de, yt[i], side(i, 1));
      }
      nu = sum_all(nu);
      de = sum_all(de);
      const double dd = a2_(de);
      const E ep = dd > 0.0 ? sc_(rcp3(dd), mul_(nu, cj_(de))) : Ops<E>::z();
      // d = (eps z - u) / gs in T coordinates, then back
      E* zt = (E*)W.z;
      for (int i = lane; i < n; i += 32) zt[i] = sc_(igs, mul_(ep, side(i, 1)) - side(i, 0));
      tri_apply_q_t(A, tau, n, zt, true);
      for (int i = lane; i < n; i += 32) W.x[i] = W.x[i] + to_cd(zt[i]);
    }
  }
  if (warp == 0) {
    __syncwarp();
    const double sc = rsqrt3(norm2_t(W.x, n));
    for (int i = lane; i < n; i += 32) W.x[i] = sc * W.x[i];
  }
  team_bar();
}

// The smallest eigenpair by a CTA of at least four warps: warps 0..3 are the
// team, the others take part in apply() only.  The result is valid in warp 0.
// apply(x, out): out = (exact operator) x; its Newton steps: `steps_far` when the
// two smallest eigenvalues are more than refine_gap * lam_max apart, `steps_near`
// otherwise.
// single: complex matrices try the single-precision solve first; ffr: real
// matrices go on in float-float after the double reduction (mixed path).
template <typename E, class Apply>
__device__ TriResult tri_smallest_team(const TriWs& W, const cd* G, int n, int steps_far, int steps_near,
                                       double refine_gap, const Apply& apply, long long* tk = nullptr,
                                       bool single = false, const cfx* Gx = nullptr, bool ffr = false) {
  __shared__ TeamWs S;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool team = warp < 4;
  TriResult res = {};
  if (team) {
    bool done = false;
    int steps = 0;
    if constexpr (sizeof(E) == sizeof(cd)) {
      if (single && n > 2) done = tri_solve_team_sp(W, S, G, n, res, tk, Gx);
      if (!done) steps = tri_solve_team<E, false>(W, S, G, n, steps_far, steps_near, refine_gap, res, tk);
    } else {
      steps = ffr ? tri_solve_team<E, true>(W, S, G, n, steps_far, steps_near, refine_gap, res, tk)
                  : tri_solve_team<E, false>(W, S, G, n, steps_far, steps_near, refine_gap, res, tk);
    }
    if (threadIdx.x == 0) S.steps = steps;
  }
  __syncthreads();
  const int steps = S.steps;
  for (int it = 0; it < steps; ++it) {
    apply(W.x, W.r);
    __syncthreads();
    if (tk && threadIdx.x == 0) tk[6] = clock64();   // end of the last step's apply
    if (team) {
      if constexpr (sizeof(E) == sizeof(double)) {
        if (ffr) tri_olsen_team<E, true>(W, S, n);
        else tri_olsen_team<E, false>(W, S, n);
      } else {
        tri_olsen_team<E, false>(W, S, n);
      }
    }
    __syncthreads();
  }
  if (tk && threadIdx.x == 0) tk[4] = clock64();
  if (team) {
    // theta = x^H G x, the rows split over the team
    double s = 0.0;
    CBP_COLS(n, {
      if (i < n) {
        cd gx = mk(0.0, 0.0);
        for (int j = warp; j < n; j += 4) cfmac(gx, G[(size_t)j * n + i], W.x[j]);   // (G x)_i, part
        s += redot_(W.x[i], gx);
      }
    });
    s = lane_sum(s);
    if (lane == 0) S.th[warp] = s;
    team_bar();
    res.theta = (S.th[0] + S.th[1]) + (S.th[2] + S.th[3]);
  }
  if (tk && threadIdx.x == 0) tk[5] = clock64();
  return res;
}
