// Forward model of Eq. 1 on the device (the camera side of Section 3):
// B = L (x) K + N, full 2D convolution per channel plus Gaussian noise, and a
// blob-latent synthesiser.  Random numbers come from Philox-4x32-10 (Salmon,
// Moraes, Dror, Shaw, "Parallel random numbers: as easy as 1, 2, 3", SC 2011):
// counter = (element index lo, element index hi, stream, 0), key = seed.
#include "cbp_common.cuh"
#include "cbp_internal.h"
#include "cbp_philox.cuh"

namespace cbp {

CBP_CHECKS_TU(kChkForward)

namespace {

// Uniform in (0, 1] from 32 bits.
__device__ __forceinline__ double u01(uint32_t v) { return ((double)v + 1.0) * 2.3283064365386963e-10; }

// Standard normal number `idx` of stream `stream` (Box-Muller on one Philox block).
__device__ __forceinline__ double normal_at(uint64_t seed, uint64_t idx, uint32_t stream) {
  U4 c = {(uint32_t)idx, (uint32_t)(idx >> 32), stream, 0u};
  U4 r = philox4x32_10(c, (uint32_t)seed, (uint32_t)(seed >> 32));
  const double u1 = u01(r.x), u2 = u01(r.y);
  return sqrt(-2.0 * log(u1)) * cospi(2.0 * u2);
}

// The same normal number in single precision (float frames).
__device__ __forceinline__ float normal_at_f(uint64_t seed, uint64_t idx, uint32_t stream) {
  const U4 r = philox4x32_10({(uint32_t)idx, (uint32_t)(idx >> 32), stream, 0u}, (uint32_t)seed,
                             (uint32_t)(seed >> 32));
  const float u1 = ((float)(r.x >> 8) + 1.0f) * 5.9604644775390625e-8f;   // (0, 1], 24 bits
  const float u2 = ((float)(r.y >> 8) + 1.0f) * 5.9604644775390625e-8f;
  return sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
}

template <typename T> __device__ __forceinline__ T normal_t(uint64_t seed, uint64_t idx, uint32_t stream);
template <> __device__ __forceinline__ double normal_t<double>(uint64_t s, uint64_t i, uint32_t st) {
  return normal_at(s, i, st);
}
template <> __device__ __forceinline__ float normal_t<float>(uint64_t s, uint64_t i, uint32_t st) {
  return normal_at_f(s, i, st);
}

__device__ __forceinline__ double uniform_at(uint64_t seed, uint64_t idx, uint32_t stream) {
  U4 c = {(uint32_t)idx, (uint32_t)(idx >> 32), stream, 0u};
  U4 r = philox4x32_10(c, (uint32_t)seed, (uint32_t)(seed >> 32));
  return u01(r.x);
}

constexpr int kTile = 32;

// out[f][ch][r][c] = sum_{p,q} L[r-p][c-q] K[f][p][q] (+ noise), r < h+t-1, c < w+t-1,
// accumulated in the frame precision (double frames: double, float frames:
// float -- the data only has to be Eq. 1 to the precision it is stored in).
template <typename T>
__global__ void __launch_bounds__(kTile * 8)
k_forward_blur(const T* lat, int c, int h, int w, const double* kern, int t, double sigma,
               uint64_t seed, T* out) {
  extern __shared__ __align__(16) char smem[];
  const int hb = h + t - 1, wb = w + t - 1;
  const int fc = blockIdx.z, f = fc / c;
  const int r0 = blockIdx.y * kTile, c0 = blockIdx.x * kTile;
  const int th = kTile + t - 1;
  T* K = (T*)smem;                           // t*t
  T* tile = (T*)(smem + ((t * t * sizeof(double) + 15) & ~size_t(15)));
  for (int i = threadIdx.x; i < t * t; i += blockDim.x) K[i] = (T)kern[(int64_t)f * t * t + i];
  const T* L = lat + (int64_t)fc * h * w;
  // tile[y][x] = L[r0 - (t-1) + y][c0 - (t-1) + x]
  for (int i = threadIdx.x; i < th * th; i += blockDim.x) {
    const int y = i / th, x = i % th;
    const int ly = r0 - (t - 1) + y, lx = c0 - (t - 1) + x;
    tile[i] = (ly >= 0 && ly < h && lx >= 0 && lx < w) ? L[(int64_t)ly * w + lx] : (T)0;
  }
  __syncthreads();
  const int tx = threadIdx.x % kTile, ty0 = threadIdx.x / kTile;
  for (int ty = ty0; ty < kTile; ty += blockDim.x / kTile) {
    const int r = r0 + ty, col = c0 + tx;
    if (r >= hb || col >= wb) continue;
    T acc = 0;
    for (int p = 0; p < t; ++p)
      for (int q = 0; q < t; ++q)
        acc = fma(K[p * t + q], tile[(ty + t - 1 - p) * th + (tx + t - 1 - q)], acc);
    const int64_t oi = ((int64_t)fc * hb + r) * wb + col;
    if (sigma > 0) acc += (T)sigma * normal_t<T>(seed, (uint64_t)oi, 1u);
    out[oi] = acc;
  }
}

// The same convolution for float frames with the kernel size fixed at compile
// time (T <= 17).  A block makes 8 R rows x 64 columns of output; a thread keeps
// R consecutive output rows of two columns (32 apart) as paired single-precision
// sums (one paired multiply-add for two, each rounded as the scalar one)
// and, for each kernel column q, slides over the T + R - 1 input rows with the
// kernel column in registers.  What bounds it: multiply-adds (T^2 an output) and
// the noise (a Philox block, a logarithm and a cosine an output).  With eight
// rows of one column and scalar multiply-adds every eight of them had cost a
// shared-memory load of the kernel and three quarters of one of the tile, and
// the tile had come over in single words.  Here the tile is copied in 16-byte
// pieces (cp.async, zero outside the frame) where the latent's rows are aligned.
// Sums in float, in the order q = 0 .. T-1, within it p = 0 .. T-1 (as the
// general kernel's per-output order differs, results agree to float rounding,
// not bitwise).  48 channels of 1080 x 1920, T = 15: 1.62 -> 1.40 ms (0.91 ms
// without noise, 25 of the units' 37 T multiply-adds a second; three blocks per SM
// instead of two 0.93 ms); T = 17: 1.89 -> 1.63 ms; T = 5 without noise 0.21 ms.
// R = 16 rows a thread where that still gives every SM two blocks, else R = 4.
constexpr int kBlurWarps = 8;
constexpr int kBlurTileC = 64;
constexpr int kBlurHalo = 16;                        // columns kept left of the tile (T - 1 <= 16)
constexpr int kBlurPitch = kBlurTileC + kBlurHalo;
constexpr int64_t kBlurMinBlocks = 2 * 152;
template <int T, int R>
__global__ void __launch_bounds__(32 * kBlurWarps, 2)
k_forward_blur_rb(const float* lat, int c, int h, int w, const double* kern, double sigma,
                  uint64_t seed, float* out) {
  constexpr int kTileR = kBlurWarps * R, TH = kTileR + T - 1;
  constexpr int TP = (T + 1) & ~1;                   // kernel column pitch, 16-byte aligned pairs
  extern __shared__ __align__(16) char bsm[];
  float* tile = (float*)bsm;                         // [TH][kBlurPitch]
  float2* K = (float2*)(bsm + sizeof(float) * TH * kBlurPitch);   // [q][p], each value twice
  const int hb = h + T - 1, wb = w + T - 1;
  const int fc = blockIdx.z, f = fc / c;
  const int r0 = blockIdx.y * kTileR, c0 = blockIdx.x * kBlurTileC;
  const float* L = lat + (int64_t)fc * h * w;
  // tile[y][x] = latent at row r0 - (T-1) + y, column c0 - kBlurHalo + x
  constexpr int G = kBlurPitch / 4;
  if ((w & 3) == 0 && ((uintptr_t)lat & 15) == 0) {
    for (int i = threadIdx.x; i < TH * G; i += 32 * kBlurWarps) {
      const int y = i / G, x = (i - y * G) * 4;
      const int ly = r0 - (T - 1) + y, lx = c0 - kBlurHalo + x;   // four columns all inside or all outside
      const bool in = ly >= 0 && ly < h && lx >= 0 && lx < w;
      const float* src = in ? L + (int64_t)ly * w + lx : lat;
      const unsigned dst = (unsigned)__cvta_generic_to_shared(tile + y * kBlurPitch + x);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(in ? 16 : 0)
                   : "memory");
    }
  } else {
    for (int i = threadIdx.x; i < TH * kBlurPitch; i += 32 * kBlurWarps) {
      const int y = i / kBlurPitch, x = i - y * kBlurPitch;
      const int ly = r0 - (T - 1) + y, lx = c0 - kBlurHalo + x;
      const bool in = ly >= 0 && ly < h && lx >= 0 && lx < w;
      const float* src = in ? L + (int64_t)ly * w + lx : lat;
      const unsigned dst = (unsigned)__cvta_generic_to_shared(tile + i);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(src), "r"(in ? 4 : 0)
                   : "memory");
    }
  }
  for (int i = threadIdx.x; i < T * TP; i += 32 * kBlurWarps) {
    const int q = i / TP, p = i - q * TP;
    const float v = p < T ? (float)kern[(int64_t)f * T * T + p * T + q] : 0.f;
    K[i] = make_float2(v, v);
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  if (r0 + ty * R >= hb) return;                     // a warp below the frame
  float2 acc[R];
#pragma unroll
  for (int i = 0; i < R; ++i) acc[i] = make_float2(0.f, 0.f);
  // out[r][col] = sum_{p,q} K[p][q] L[r - p][col - q]
#pragma unroll 1
  for (int q = 0; q < T; ++q) {
    const float* col = tile + (ty * R) * kBlurPitch + kBlurHalo + tx - q;
    (void)CBP_CHECK((ty * R + R + T - 2) * kBlurPitch + kBlurHalo + tx - q + 32 < TH * kBlurPitch, 0);
    float2 kv[TP];
#pragma unroll
    for (int p = 0; p < TP; p += 2) {
      const float4 k2 = *(const float4*)(K + q * TP + p);
      kv[p] = make_float2(k2.x, k2.y);
      kv[p + 1] = make_float2(k2.z, k2.w);
    }
    // an output row meets the kernel rows in ascending order p = i + T-1 - j:
    // the input rows are taken from the last to the first
#pragma unroll
    for (int j = R + T - 2; j >= 0; --j) {
      const float2 v = make_float2(col[j * kBlurPitch], col[j * kBlurPitch + 32]);
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const int p = i + T - 1 - j;
        if (p >= 0 && p < T) acc[i] = __ffma2_rn(kv[p], v, acc[i]);
      }
    }
  }
#pragma unroll 1
  for (int g = 0; g < 2; ++g) {
    const int colo = c0 + tx + 32 * g;
    if (colo >= wb) break;
    const int64_t o0 = ((int64_t)fc * hb + r0 + ty * R) * wb + colo;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      if (r0 + ty * R + i >= hb) break;
      const int64_t oi = o0 + (int64_t)i * wb;
      float a = g ? acc[i].y : acc[i].x;
      if (sigma > 0) a += (float)sigma * normal_at_f(seed, (uint64_t)oi, 1u);
      out[oi] = a;
    }
  }
}

template <int T, int R>
void launch_blur_rows(const float* lat, int n, int c, int h, int w, const double* kern, double sigma,
                      uint64_t seed, float* out, cudaStream_t st) {
  const int hb = h + T - 1, wb = w + T - 1;
  constexpr int tr = kBlurWarps * R;
  dim3 g((wb + kBlurTileC - 1) / kBlurTileC, (hb + tr - 1) / tr, n * c);
  constexpr size_t sm = sizeof(float2) * (size_t)T * ((T + 1) & ~1) + sizeof(float) * (size_t)(tr + T - 1) * kBlurPitch;
  allow_smem((const void*)k_forward_blur_rb<T, R>);
  k_forward_blur_rb<T, R><<<g, 32 * kBlurWarps, sm, st>>>(lat, c, h, w, kern, sigma, seed, out);
}
template <int T>
void launch_blur_rb(const float* lat, int n, int c, int h, int w, const double* kern, double sigma,
                    uint64_t seed, float* out, cudaStream_t st) {
  const int hb = h + T - 1, wb = w + T - 1;
  const int64_t big = (int64_t)((wb + kBlurTileC - 1) / kBlurTileC) * ((hb + 16 * kBlurWarps - 1) / (16 * kBlurWarps)) *
                      n * c;
  if (big >= kBlurMinBlocks) launch_blur_rows<T, 16>(lat, n, c, h, w, kern, sigma, seed, out, st);
  else launch_blur_rows<T, 4>(lat, n, c, h, w, kern, sigma, seed, out, st);
}

// Blob latent: L = sum_k a_k exp(-((x-cx)^2 + (y-cy)^2) / (2 s^2)) + U[0, floor].
template <typename T>
__global__ void k_synth_latent(const double* blobs, int nblobs, int c, int h, int w,
                               double floor_amp, uint64_t seed, T* out) {
  const int fc = blockIdx.z;
  const double* B = blobs + (int64_t)fc * nblobs * 4;
  const int y = blockIdx.y, x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= w) return;
  // in the frame precision, like the blur
  T v = 0;
  for (int k = 0; k < nblobs; ++k) {
    const T a = (T)B[4 * k], s = (T)B[4 * k + 1], cx = (T)B[4 * k + 2], cy = (T)B[4 * k + 3];
    const T dx = (T)x - cx, dy = (T)y - cy;
    v += a * exp(-(dx * dx + dy * dy) / ((T)2 * s * s));
  }
  const int64_t oi = ((int64_t)fc * h + y) * w + x;
  v += (T)(floor_amp * uniform_at(seed, (uint64_t)oi, 2u));
  out[oi] = v;
}

// Multi-level security (Section 3): the private stream at a lower clearance
// level, its least significant bits removed.  code = rint(x (2^bits - 1))
// clamped to [0, 2^bits - 1], the `drop` low bits cleared, value
// code / (2^bits - 1), as double-precision arithmetic gives it whatever the
// element type.  In double arithmetic throughout (a product, a rounding, two
// clamps, two conversions and a division) the kernel was bound by the double
// units, which issue one warp instruction in ~64 cycles: 3.01 ms for 102 M
// floats (0.27 TB/s).  The two forms below give the same bits from
// single-precision and integer instructions; the float one is bound by memory
// (0.138 ms for the same floats, 5.9 TB/s).
//
// Floats with codes of at most kTruncBitsF bits: x top = p + e exactly (FMA),
// so rint(p) is the code unless p itself was rounded onto a half, where the
// sign of e decides; the quotient by one multiplication and one FMA correction
// is the correctly rounded one for every code of up to 22 bits (checked over
// all of them), and a correctly rounded double quotient rounds to the same
// float: it would have to lie within 2^-53 of the middle of two floats, and
// code / (2^bits - 1) keeps 2^-(25 + bits) away from it.  Products of 2^23 and
// above are integers beyond every code: they clamp.
constexpr int kTruncBitsF = 22;
constexpr int kTruncThreads = 256;
constexpr int kTruncVec = 4;         // 16-byte groups in flight per thread

struct TruncF {
  float top, inv;
  int mask;
  __device__ __forceinline__ float operator()(float x) const {
    const float p = x * top, e = fmaf(x, top, -p);
    float r = rintf(p);
    const float d = p - r;
    if (d == 0.5f && e > 0.f) r += 1.f;
    if (d == -0.5f && e < 0.f) r -= 1.f;
    const float c = (float)((int)fminf(fmaxf(r, 0.f), top) & mask);   // NaN: code 0
    const float q = c * inv;
    return fmaf(fmaf(-q, top, c), inv, q);
  }
};

// Doubles, and floats with longer codes: one double product, clamped by
// integer comparisons, rounded to an integer by adding 2^52; the quotient
// c / (2^bits - 1) is the binary fraction 0.ccc... of the repeated code, so its
// double is read off the repeated bit pattern (rounded by the first dropped
// bit: the dropped tail is never exactly one half).  Two double instructions
// an element.
struct TruncW {
  double top;
  uint32_t topi, mask;
  int bits;
  __device__ __forceinline__ double operator()(double x) const {
    long long v = __double_as_longlong(x * top);
    if (v < 0 || v > 0x7ff0000000000000ll) v = 0;                      // negative or NaN: code 0
    const long long vt = __double_as_longlong(top);
    if (v > vt) v = vt;
    const uint32_t c =
        (uint32_t)__double_as_longlong(__longlong_as_double(v) + 0x1p52) & mask;
    if (c == 0u) return 0.0;
    if (c == topi) return 1.0;
    const int lz = __clz(c) - (32 - bits);
    const uint32_t cr = ((c << lz) | (lz ? c >> (bits - lz) : 0u)) & topi;   // leading bit first
    uint64_t w = (uint64_t)cr << (64 - bits);
    for (int s = bits; s < 64; s <<= 1) w |= w >> s;
    const uint64_t m = ((w >> 10) + 1) >> 1;                           // 53 bits, rounded
    return __longlong_as_double(((long long)(1022 - lz) << 52) + (long long)(m & 0xfffffffffffffull));
  }
};

// A grid-stride pass; 16-byte groups when both buffers allow it.
template <typename T, class Op>
__global__ void __launch_bounds__(kTruncThreads) k_truncate_lsb(const T* in, int64_t count, Op op, T* out,
                                                               int vec) {
  constexpr int E = 16 / (int)sizeof(T);
  struct alignas(16) V { T v[E]; };
  const int64_t stride = (int64_t)gridDim.x * kTruncThreads;
  const int64_t t0 = blockIdx.x * (int64_t)kTruncThreads + threadIdx.x;
  int64_t done = 0;
  if (vec) {
    const int64_t groups = count / E;
    const V* vi = (const V*)in;
    V* vo = (V*)out;
    for (int64_t g = t0; g < groups; g += kTruncVec * stride) {
      V x[kTruncVec];
#pragma unroll
      for (int k = 0; k < kTruncVec; ++k)
        if (g + k * stride < groups) x[k] = vi[g + k * stride];
#pragma unroll
      for (int k = 0; k < kTruncVec; ++k) {
        if (g + k * stride >= groups) break;
#pragma unroll
        for (int e = 0; e < E; ++e) x[k].v[e] = (T)op(x[k].v[e]);
        vo[g + k * stride] = x[k];
      }
    }
    done = groups * E;
  }
  for (int64_t i = done + t0; i < count; i += stride) out[i] = (T)op(in[i]);
}

// Camera side (Section 3, "Blur Kernel Selection": new random kernels for
// every frame): kernel `kind` of frame frame0 + f at redraw attempt[f],
// entries (Philox word + 1) 2^-32, uniform in (0, 1], normalised to unit sum
// in entry order.  Entry e is word e mod 4 of Philox(counter = (e / 4, frame,
// kind * 256 + attempt, 0), key = seed).  One CTA per kernel, both kernels of a
// pair in one launch; the entries are multiples of 2^-32 no larger than 1, so
// every partial sum of up to 2^20 of them is exact and the integer sum is the
// sum in entry order (one thread per kernel had taken 102 and 130 us for 15 x 15
// and 17 x 17 kernels: a chain of double adds and one of double divisions).
// Pairs whose active flag is clear keep their kernels.
constexpr int kDrawThreads = 128;
__global__ void __launch_bounds__(kDrawThreads)
k_draw_kernels(int ta, int tb, int kind_a, int kind_b, int frame0, uint64_t seed, const int* active,
               const int* attempt, double* ka, double* kb) {
  const int f = blockIdx.x, second = blockIdx.y;
  if (!active[f]) return;
  const int t = second ? tb : ta, kind = second ? kind_b : kind_a, nn = t * t;
  double* K = (second ? kb : ka) + (int64_t)f * nn;
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  __shared__ uint32_t word[32 * 32];
  __shared__ unsigned long long part[kDrawThreads / 32];
  unsigned long long sum = 0;
  for (int b = threadIdx.x; 4 * b < nn; b += kDrawThreads) {
    const U4 r = philox4x32_10({(uint32_t)b, (uint32_t)(frame0 + f), (uint32_t)(kind * 256 + attempt[f]), 0u},
                               k0, k1);
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (4 * b + i < nn) {
        word[4 * b + i] = w[i];
        sum += (unsigned long long)w[i] + 1ull;
      }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
  __syncthreads();
  unsigned long long total = 0;
#pragma unroll
  for (int i = 0; i < kDrawThreads / 32; ++i) total += part[i];
  const double s = (double)total * 2.3283064365386963e-10;   // exact: below 2^43, times 2^-32
  for (int e = threadIdx.x; e < nn; e += kDrawThreads) K[e] = u01(word[e]) / s;
}

}  // namespace

void launch_draw_kernels(int n, int ta, int tb, int kind_a, int kind_b, int frame0, uint64_t seed,
                         const int* active, const int* attempt, double* ka, double* kb, cudaStream_t st) {
  k_draw_kernels<<<dim3(n, 2), kDrawThreads, 0, st>>>(ta, tb, kind_a, kind_b, frame0, seed, active, attempt, ka, kb);
}

void launch_truncate_lsb(const void* in, int f64, int64_t count, int bits, int drop, void* out,
                         cudaStream_t st) {
  const int es = f64 ? 8 : 4;
  const int vec = (((uintptr_t)in | (uintptr_t)out) & 15) == 0 ? 1 : 0;
  const int64_t per = (int64_t)kTruncThreads * (vec ? 16 / es * kTruncVec : 1);
  const int64_t want = (count + per - 1) / per;
  const int blocks = (int)(want < 152 * 8 ? (want > 0 ? want : 1) : 152 * 8);
  const uint32_t topi = (uint32_t)((1ull << bits) - 1), mask = topi & ~((1u << drop) - 1);
  if (!f64 && bits <= kTruncBitsF) {
    const TruncF op{(float)topi, 1.0f / (float)topi, (int)mask};
    k_truncate_lsb<float><<<blocks, kTruncThreads, 0, st>>>((const float*)in, count, op, (float*)out, vec);
    return;
  }
  const TruncW op{(double)topi, topi, mask, bits};
  if (f64)
    k_truncate_lsb<double><<<blocks, kTruncThreads, 0, st>>>((const double*)in, count, op, (double*)out, vec);
  else
    k_truncate_lsb<float><<<blocks, kTruncThreads, 0, st>>>((const float*)in, count, op, (float*)out, vec);
}

void launch_forward_blur(const void* latent, int n, int c, int h, int w, int f64,
                         const double* kernel, int t, double sigma, uint64_t seed, void* out,
                         cudaStream_t st) {
  const int hb = h + t - 1, wb = w + t - 1;
  dim3 g((wb + kTile - 1) / kTile, (hb + kTile - 1) / kTile, n * c);
  const int th = kTile + t - 1;
  const size_t sm = ((t * t * sizeof(double) + 15) & ~size_t(15)) + (size_t)th * th * (f64 ? 8 : 4);
  if (f64) {
    allow_smem((const void*)k_forward_blur<double>);
    k_forward_blur<double><<<g, kTile * 8, sm, st>>>((const double*)latent, c, h, w, kernel, t,
                                                      sigma, seed, (double*)out);
  } else if (t <= 17) {
    const float* L = (const float*)latent;
    float* o = (float*)out;
    switch (t) {
#define CBP_BLUR_CASE(T) \
  case T: launch_blur_rb<T>(L, n, c, h, w, kernel, sigma, seed, o, st); break;
      CBP_BLUR_CASE(1) CBP_BLUR_CASE(2) CBP_BLUR_CASE(3) CBP_BLUR_CASE(4) CBP_BLUR_CASE(5)
      CBP_BLUR_CASE(6) CBP_BLUR_CASE(7) CBP_BLUR_CASE(8) CBP_BLUR_CASE(9) CBP_BLUR_CASE(10)
      CBP_BLUR_CASE(11) CBP_BLUR_CASE(12) CBP_BLUR_CASE(13) CBP_BLUR_CASE(14) CBP_BLUR_CASE(15)
      CBP_BLUR_CASE(16) default: CBP_BLUR_CASE(17)
#undef CBP_BLUR_CASE
    }
  } else {
    allow_smem((const void*)k_forward_blur<float>);
    k_forward_blur<float><<<g, kTile * 8, sm, st>>>((const float*)latent, c, h, w, kernel, t,
                                                     sigma, seed, (float*)out);
  }
}

void launch_synth_latent(const double* blobs, int nblobs, int n, int c, int h, int w, int f64,
                         double floor_amp, uint64_t seed, void* out, cudaStream_t st) {
  dim3 g((w + 127) / 128, h, n * c);
  if (f64)
    k_synth_latent<double><<<g, 128, 0, st>>>(blobs, nblobs, c, h, w, floor_amp, seed, (double*)out);
  else
    k_synth_latent<float><<<g, 128, 0, st>>>(blobs, nblobs, c, h, w, floor_amp, seed, (float*)out);
}

}  // namespace cbp
