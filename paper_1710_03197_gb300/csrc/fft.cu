// fft.cu - scaling + zero-padding + oversampled FFT, and inverse FFT + crop +
// rescaling, as pruned line passes over the K^d grid.
//
// Section 2.1.1 (scaling S), Section 2.1.2 (zero-padding and oversampled FFT
// F; the inverse FFT followed by the array copy back), Table 1 rows S, F, F^H,
// S^H.  The paper runs S, a pre-indexed copy and a library FFT as separate
// steps over the whole K^d array.  Here the d-dimensional transform is done
// one axis at a time, and each pass is pruned:
//   forward, axis a: lines whose coordinates on axes < a lie in the padded
//     image's footprint (N_i of the K_i positions), all K on axes > a; only
//     the N_a non-zero inputs of a line are read; all K_a outputs written.
//     The first pass (last axis) reads the image itself and applies S, so
//     the padded array is never materialised.
//   inverse, axis a: lines over the crop footprint on axes < a, all K on
//     axes > a; all K_a inputs read, only the N_a cropped outputs written;
//     the last pass (last axis) applies S^H and writes the image.
// Padded position of image index n along an axis: g = (n - N/2) mod K.
//
// Each line of power-of-two length is transformed by a Stockham auto-sort
// FFT, each thread holding E values per stage in registers: one smaller radix
// if the length asks for it, then radix-E stages, E = 8 or 16.  The first stage
// works on the values as loaded and the last stage's outputs are stored as they
// are; the hand-offs between stages go through two shared-memory buffers used
// in turn (one buffer where there is one hand-off), one barrier per hand-off.
// Twiddles are computed in registers.
// Other line lengths (even, prime factors 2, 3 and 5) run stages of radices 2 to 8
// (k_fft_mixed).
#include <type_traits>

#include "internal.cuh"

namespace nufft {
namespace {

struct FftArgs {
  const float2* src;
  float2* dst;
  const float* s_axis;        // scaling of axis a (image side only)
  const float* s_lead[kMaxDim];
  int a;
  int Na;                     // N_a
  int lead_N[kMaxDim];
  int lead_K[kMaxDim];
  int64_t lead_stride[kMaxDim];
  int64_t nouter;             // prod_{i<a} N_i
  int64_t inner;              // prod_{i>a} K_i (grid stride of axis a)
  int src_image;              // forward first pass: read the image, apply S
  int dst_image;              // inverse last pass: write the image, apply S^H
  int64_t src_bstride;        // batch strides (blockIdx.y selects the batch element)
  int64_t dst_bstride;
  int scale;                  // 0: no S / S^H (plain zero-pad / crop)
  // CG step hooks (see CgHooks): prologue of the first forward pass,
  // epilogue of the last inverse pass
  float2* pro_p;
  const float2* pro_r;
  const double* pro_part;
  int pro_count;
  double* pro_sc;
  int pro_old, pro_new;
  const float2* epi_a;
  double* epi_part;
};

// Sum of v over the CTA (any block size up to 1024) in a fixed order: a
// shuffle tree per warp, then the warps in order.  Every thread must call it;
// every thread gets the sum.  red: 32 doubles of shared scratch.
__device__ __forceinline__ double block_sum_dbl(double v, double* red) {
  const int lane = threadIdx.x & 31;
  const int n = min(32, (int)blockDim.x - (int)(threadIdx.x & ~31u));   // lanes of this warp
  const unsigned mask = n == 32 ? 0xffffffffu : (1u << n) - 1u;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {   // lane 0 ends with the sum of the lanes there are
    const double u = __shfl_xor_sync(mask, v, o);
    v += (lane ^ o) < n ? u : 0.0;
  }
  if (lane == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  const int nw = (blockDim.x + 31) >> 5;
  for (int w = 0; w < nw; ++w) t += red[w];
  __syncthreads();
  return t;
}

// beta of the CG prologue (every CTA computes the same value); CTA 0 stores
// the new <r, r> for the next step.
__device__ __forceinline__ float cg_prologue_beta(const FftArgs& A, double* red) {
  double s = 0.0;
  for (int i = threadIdx.x; i < A.pro_count; i += blockDim.x) s += A.pro_part[i];
  const double rr_new = block_sum_dbl(s, red);
  const double rr_old = A.pro_sc[A.pro_old];
  if (blockIdx.x == 0 && threadIdx.x == 0) A.pro_sc[A.pro_new] = rr_new;
  return (float)(rr_old != 0.0 ? rr_new / rr_old : 0.0);
}

// image element idx of the first forward pass: with the CG prologue,
// p = r + beta p written back in place (read with a plain load: it is written)
__device__ __forceinline__ float2 load_image(const FftArgs& A, const float2* __restrict__ src, int64_t idx,
                                             bool pro, float beta) {
  if (!pro) return __ldg(&src[idx]);
  const float2 pv = A.pro_p[idx], rv = A.pro_r[idx];
  const float2 pn = make_float2(fmaf(beta, pv.x, rv.x), fmaf(beta, pv.y, rv.y));
  A.pro_p[idx] = pn;
  return pn;
}

template <bool INV>
__device__ __forceinline__ float2 rot90(float2 z) {  // z * (-i) forward, z * (+i) inverse
  return INV ? make_float2(-z.y, z.x) : make_float2(z.y, -z.x);
}

template <bool INV>
__device__ __forceinline__ void dft2(float2* v) {
  float2 a = v[0];
  v[0] = cadd(a, v[1]);
  v[1] = csub(a, v[1]);
}

template <bool INV>
__device__ __forceinline__ void dft4(float2& v0, float2& v1, float2& v2, float2& v3) {
  float2 a = cadd(v0, v2), b = csub(v0, v2), c = cadd(v1, v3), e = rot90<INV>(csub(v1, v3));
  v0 = cadd(a, c);
  v1 = cadd(b, e);
  v2 = csub(a, c);
  v3 = csub(b, e);
}

// e + h p, one rounding per component
__device__ __forceinline__ float2 caxpy(float h, float2 p, float2 e) {
  return make_float2(fmaf(h, p.x, e.x), fmaf(h, p.y, e.y));
}

template <bool INV>
__device__ __forceinline__ void dft8(float2* v) {
  const float h = 0.70710678118654752440f;
  float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  float2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4<INV>(e0, e1, e2, e3);
  dft4<INV>(o0, o1, o2, o3);
  // o_k *= W8^k, W8 = exp(-+ 2 pi i / 8): W8 = h (1 -+ i), W8^3 = h (-1 -+ i)
  const float2 p1 = INV ? make_float2(o1.x - o1.y, o1.x + o1.y) : make_float2(o1.x + o1.y, o1.y - o1.x);
  const float2 p3 = INV ? make_float2(-o3.x - o3.y, o3.x - o3.y) : make_float2(o3.y - o3.x, -o3.x - o3.y);
  o2 = rot90<INV>(o2);
  v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
  v[1] = caxpy(h, p1, e1); v[5] = caxpy(-h, p1, e1);
  v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
  v[3] = caxpy(h, p3, e3); v[7] = caxpy(-h, p3, e3);
}

// DFT of 16 points as 4 x 4: DFT-4 over (i, i + 4, i + 8, i + 12), twiddles
// W16^(i j), DFT-4 over i.
template <bool INV>
__device__ __forceinline__ void dft16(float2* v) {
  const float h = 0.70710678118654752440f, c = 0.92387953251128675613f, s = 0.38268343236508977173f;
#pragma unroll
  for (int i = 0; i < 4; ++i) dft4<INV>(v[i], v[i + 4], v[i + 8], v[i + 12]);
  // v[i + 4 j] *= W16^(i j), W16 = exp(-+ 2 pi i / 16) = c -+ i s
  auto mul = [](float2 z, float wr, float wi) { return cmul(z, make_float2(wr, INV ? -wi : wi)); };
  v[5] = mul(v[5], c, -s);
  v[9] = INV ? make_float2(h * (v[9].x - v[9].y), h * (v[9].x + v[9].y))
             : make_float2(h * (v[9].x + v[9].y), h * (v[9].y - v[9].x));
  v[13] = mul(v[13], s, -c);
  v[6] = INV ? make_float2(h * (v[6].x - v[6].y), h * (v[6].x + v[6].y))
             : make_float2(h * (v[6].x + v[6].y), h * (v[6].y - v[6].x));
  v[10] = rot90<INV>(v[10]);
  v[14] = INV ? make_float2(h * (-v[14].x - v[14].y), h * (v[14].x - v[14].y))
              : make_float2(h * (v[14].y - v[14].x), h * (-v[14].x - v[14].y));
  v[7] = mul(v[7], s, -c);
  v[11] = INV ? make_float2(h * (-v[11].x - v[11].y), h * (v[11].x - v[11].y))
              : make_float2(h * (v[11].y - v[11].x), h * (-v[11].x - v[11].y));
  v[15] = mul(v[15], -c, s);
  float2 o[16];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    dft4<INV>(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
#pragma unroll
    for (int q = 0; q < 4; ++q) o[j + 4 * q] = v[4 * j + q];   // output j + 4 q
  }
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = o[k];
}

template <int R, bool INV>
__device__ __forceinline__ void dft(float2* v) {
  if (R == 2) dft2<INV>(v);
  else if (R == 4) dft4<INV>(v[0], v[1], v[2], v[3]);
  else if (R == 8) dft8<INV>(v);
  else dft16<INV>(v);
}

constexpr int ilog2(int x) { return x <= 1 ? 0 : 1 + ilog2(x / 2); }

// Shared-memory position of element p of line b of the CTA's W lines, for the
// hand-off after a stage of radix R and span Ns.  A half-warp's 64-bit accesses
// are free of conflicts when its 16 positions differ mod 16.
// Strided axis: W lines side by side (W consecutive grid columns), a row of W
// values per element: 16 columns fill a half-warp; with fewer, the writers of
// the first hand-off (Ns = 1, row stride R from one thread to the next) need
// the row's low bits mixed with the thread's.
// Contiguous axis: one line after another, one pad word per 16 elements (8 in
// lines of at most 128), and a pitch of 8 mod 16 for lines whose 8 threads
// share a half-warp with the next line's.
template <int L, bool STRIDED>
struct SmemMap {
  static constexpr int kPad = L <= 128 ? 3 : 4;
  static constexpr int kRaw = L + (L >> kPad);
  static constexpr int kLinePitch = L == 128 ? 152 : kRaw;
  template <int R, int NS>
  __device__ __forceinline__ static int at(int wlog, int b, int p) {
    if (!STRIDED) return b * kLinePitch + p + (p >> kPad);
    const int q = NS == 1 && wlog < 4 ? p ^ ((p / R) & ((16 >> wlog) - 1)) : p;
    return (q << wlog) + b;
  }
  __host__ __device__ static size_t words(int w) { return STRIDED ? (size_t)L * w : (size_t)w * kLinePitch; }
};

// Stockham stage of radix R over span Ns on the values a thread holds.
//
// In every stage a thread reads the elements t + k*TPL (k = 0..E-1, TPL = L/E)
// of its line: butterfly q (q < E/R) takes inputs j + r*L/R with j = t + q*TPL,
// which is element t + (q + r*Q)*TPL.  So x[k] holds element t + k*TPL on entry,
// the first stage needs no shared memory, and the outputs of the last stage
// (Ns = L/R, written to j + r*Ns) are again elements t + k*TPL, stored straight
// to global memory.  Only the middle hand-offs go through shared memory.
//
// Twiddles of a radix-E stage, computed: input r of the thread's butterfly gets
// w1^r, w1 = exp(-+ 2 pi i k / (Ns E)), from sincospif (2k / (Ns E) is exact:
// Ns E is a power of two) and products (a few ulp; a table rounded from FP64
// would be 0.5 ulp).  Radix 16 takes w4 from sincospif too, so that no power
// carries more than six single errors.  The passes then issue no twiddle loads
// (the strided 3D passes are bound by issue and the L1/shared pipe, the 2D ones
// by load latency).
//
// Radix 8 states which products are fused: on a smooth image, whose few strong
// frequencies meet few twiddles, that alone moved the error by 3 to 10 %.  The
// inverse squares a root as (1 - 2 s^2, 2 s c): error of an adjoint on a 128^2 to
// 1024^2 grid 0.65 to 0.93 of that with the product, and no slower.  The forward
// passes keep the product: 0.65 to 1 likewise, but 1.3 on a 512^2 grid.
__device__ __forceinline__ float2 cmul_fused(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -__fmul_rn(a.y, b.y)), fmaf(a.y, b.x, __fmul_rn(a.x, b.y)));
}

template <bool INV>
__device__ __forceinline__ void apply_twiddles8(float2 (&x)[8], int k, int Ns) {
  const float inv = 2.0f / (float)(Ns * 8);   // exact
  float sn, cs;
  sincospif((float)k * inv, &sn, &cs);
  const float2 w1 = make_float2(cs, INV ? sn : -sn);
  const float2 w2 = INV ? make_float2(fmaf(-2.0f * w1.y, w1.y, 1.0f), 2.0f * __fmul_rn(w1.x, w1.y))
                        : cmul_fused(w1, w1);
  const float2 w3 = cmul_fused(w2, w1), w4 = cmul_fused(w2, w2);
  const float2 w[8] = {w1, w1, w2, w3, w4, cmul_fused(w4, w1), cmul_fused(w4, w2), cmul_fused(w4, w3)};
#pragma unroll
  for (int r = 1; r < 8; ++r) x[r] = cmul_fused(x[r], w[r]);
}

template <bool INV>
__device__ __forceinline__ void apply_twiddles16(float2 (&x)[16], int k, int Ns) {
  const float inv = 2.0f / (float)(Ns * 16);   // exact
  float sn, cs;
  sincospif((float)k * inv, &sn, &cs);
  const float2 w1 = make_float2(cs, INV ? sn : -sn);
  const float2 w2 = cmul(w1, w1), w3 = cmul(w2, w1);
  sincospif((float)(4 * k) * inv, &sn, &cs);
  const float2 w4 = make_float2(cs, INV ? sn : -sn);
  float2 hi = w4;
  x[1] = cmul(x[1], w1);
  x[2] = cmul(x[2], w2);
  x[3] = cmul(x[3], w3);
#pragma unroll
  for (int r = 4; r < 16; r += 4) {
    x[r] = cmul(x[r], hi);
    x[r + 1] = cmul(x[r + 1], cmul(hi, w1));
    x[r + 2] = cmul(x[r + 2], cmul(hi, w2));
    x[r + 3] = cmul(x[r + 3], cmul(hi, w3));
    if (r + 4 < 16) hi = cmul(hi, w4);
  }
}

template <int E, int R, bool INV>
__device__ __forceinline__ void butterflies(float2 (&x)[E]) {
  constexpr int Q = E / R;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = x[q + r * Q];
    dft<R, INV>(v);
#pragma unroll
    for (int r = 0; r < R; ++r) x[q + r * Q] = v[r];
  }
}

// Hand-off after a stage of radix R and span NS: outputs to their Stockham
// positions, barrier, the thread's next elements.
template <int L, int E, bool STRIDED, int R, int NS>
__device__ __forceinline__ void hand_off(float2* sm, int wlog, int b, int t, float2 (&x)[E]) {
  constexpr int TPL = L / E;
  constexpr int Q = E / R;
  using Map = SmemMap<L, STRIDED>;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int j = t + q * TPL;
    const int k = j & (NS - 1);
    const int base = (j - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) sm[Map::template at<R, NS>(wlog, b, base + r * NS)] = x[q + r * Q];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < E; ++k) x[k] = sm[Map::template at<R, NS>(wlog, b, t + k * TPL)];
}

// Stages of radix E from span NS on; buffer c of the two at sm + c * bufw.
template <int L, int E, bool STRIDED, bool INV, int NS>
__device__ __forceinline__ void radix_e_stages(float2* sm, int cur, int bufw, int wlog, int b, int t, float2 (&x)[E]) {
  if constexpr (NS > 1 && E == 8) apply_twiddles8<INV>(x, t & (NS - 1), NS);
  if constexpr (NS > 1 && E == 16) apply_twiddles16<INV>(x, t & (NS - 1), NS);
  butterflies<E, E, INV>(x);
  if constexpr (NS * E < L) {
    hand_off<L, E, STRIDED, E, NS>(sm + cur * bufw, wlog, b, t, x);
    radix_e_stages<L, E, STRIDED, INV, NS * E>(sm, cur ^ 1, bufw, wlog, b, t, x);
  }
}

constexpr int fft_first_radix(int L, int E) { return 1 << (ilog2(L) % ilog2(E)); }
constexpr int fft_hand_offs(int L, int E) { return (ilog2(L) + ilog2(E) - 1) / ilog2(E) - 1; }

// grid: strided axes (column blocks, outer lines, batch), contiguous axis
// (blocks of W lines, 1, batch); 32-bit indices within a transform (K^d <= 2^30).
// HOOK: the CG step's work (contiguous axis only); a kernel of its own, so that
// the plain pass carries none of its FP64 code.
// WL > 0: log2 of the columns per CTA, fixed, so that the shared-memory addresses
// of a hand-off are one base and immediate offsets; WL = 0: wl_arg.
// Contiguous lines of 1024 points are held to 48 registers (5 CTAs per SM), as many
// as the compiler takes for shorter ones: with the 67 it takes left alone, 8 images
// on a 1024^2 grid 20.3 -> 23.3 us forward.
template <int L, int E, bool STRIDED, bool INV, bool HOOK, int WL>
__global__ void __launch_bounds__(E == 16 ? 256 : (STRIDED ? L : 256), E == 16 ? 4 : (!STRIDED && L == 1024 ? 5 : 1))
k_fft_pass(const FftArgs A, const int wl_arg) {
  constexpr int TPL = L / E;
  const int wlog = WL > 0 ? WL : wl_arg;
  extern __shared__ float2 sm[];
  const int W = 1 << wlog;
  const int bufw = (int)SmemMap<L, STRIDED>::words(W);

  const int tid = threadIdx.x;
  int b, t, o, in;
  if (STRIDED) {
    b = tid & (W - 1);
    t = tid >> wlog;
    o = blockIdx.y;
    in = blockIdx.x * W + b;
  } else {
    b = tid / TPL;
    t = tid % TPL;
    o = blockIdx.x * W + b;
    in = 0;
  }
  const bool live = o < (int)A.nouter;
  const float2* __restrict__ src = A.src + (int64_t)blockIdx.z * A.src_bstride;
  float2* __restrict__ dst = A.dst + (int64_t)blockIdx.z * A.dst_bstride;

  // Outer coordinates: image index on axes < a, mapped to padded grid positions.
  int goff = in;
  float slead = 1.0f;
  if (live) {
    int rem = o;
    for (int i = A.a - 1; i >= 0; --i) {
      int n = rem;
      if (i > 0) {   // the outermost coordinate is what is left
        rem = n / A.lead_N[i];
        n -= rem * A.lead_N[i];
      }
      const int gi = wrapk(n - A.lead_N[i] / 2 + A.lead_K[i], A.lead_K[i]);
      goff += gi * (int)A.lead_stride[i];
      if (A.scale && (A.src_image || A.dst_image)) slead *= A.s_lead[i][n];
    }
  }
  const int half = A.Na >> 1;
  const int stride = STRIDED ? (int)A.inner : 1;
  const bool pro = HOOK && !INV && A.src_image && A.pro_p;
  float beta = 0.f;
  if constexpr (HOOK && !INV) {
    __shared__ double red[32];
    if (pro) beta = cg_prologue_beta(A, red);
  }
  const uint64_t pol = l2_evict_first_policy();   // a pass reads each input element once

  // ---- load the thread's elements t + k*TPL (pruned on the forward side)
  float2 x[E];
#pragma unroll
  for (int k = 0; k < E; ++k) {
    const int p = t + k * TPL;
    float2 v = make_float2(0.f, 0.f);
    if (live) {
      if (!INV) {
        const bool in_image = (p < half) || (p >= L - half);
        if (in_image) {
          if (A.src_image) {
            const int n = p < half ? p + half : p - L + half;
            v = cscale(load_image(A, src, o * A.Na + n, pro, beta), (A.scale ? A.s_axis[n] : 1.0f) * slead);
          } else {
            v = ld_last_use(&src[goff + p * stride], pol);
          }
        }
      } else {
        v = ld_last_use(&src[goff + p * stride], pol);
      }
    }
    x[k] = v;
  }

  // ---- transform: a smaller first radix where the length needs one, then radix E
  constexpr int R0 = fft_first_radix(L, E);
  if constexpr (R0 > 1) {
    butterflies<E, R0, INV>(x);
    hand_off<L, E, STRIDED, R0, 1>(sm, wlog, b, t, x);
    radix_e_stages<L, E, STRIDED, INV, R0>(sm, 1, bufw, wlog, b, t, x);
  } else {
    radix_e_stages<L, E, STRIDED, INV, 1>(sm, 0, bufw, wlog, b, t, x);
  }

  // ---- store the thread's elements t + k*TPL (pruned on the inverse side)
  const bool epi = HOOK && INV && A.dst_image && A.epi_part;
  double dot = 0.0;
  if (live) {
#pragma unroll
    for (int k = 0; k < E; ++k) {
      const int p = t + k * TPL;
      const float2 v = x[k];
      if (!INV) {
        dst[goff + p * stride] = v;
      } else {
        const bool in_image = (p < half) || (p >= L - half);
        if (!in_image) continue;
        if (A.dst_image) {
          const int n = p < half ? p + half : p - L + half;
          const float2 out = cscale(v, (A.scale ? A.s_axis[n] : 1.0f) * slead);
          dst[o * A.Na + n] = out;
          if (epi) {
            const float2 a = A.epi_a[o * A.Na + n];
            dot += (double)a.x * (double)out.x + (double)a.y * (double)out.y;
          }
        } else {
          dst[goff + p * stride] = v;
        }
      }
    }
  }
  if constexpr (HOOK && INV) {
    __shared__ double red[32];
    if (epi) {
      const double tsum = block_sum_dbl(dot, red);
      if (threadIdx.x == 0) A.epi_part[blockIdx.x] = tsum;
    }
  }
}

// CTAs wanted before lines are grouped into wider ones.
constexpr int64_t kTargetBlocks = 2 * 152;

// query: only report the number of CTAs (per batch element) in *nblocks.
// E values per thread.  Lines per CTA: as many as give 256 threads (strided
// axis: at most 16 columns, full 128-byte rows with E = 16, 8 with E = 8), fewer
// when that would leave the GPU with fewer than two CTAs per SM (counting every
// batch element's CTAs).
template <int L, int E, bool STRIDED, bool INV>
cudaError_t launch_LE(const FftArgs& A, int nb, cudaStream_t st, int64_t* nblocks, bool query) {
  constexpr int TPL = L / E;
  constexpr int kBuffers = fft_hand_offs(L, E) > 1 ? 2 : 1;
  int wlog = 0;
  int64_t blocks;
  if (STRIDED) {
    wlog = E == 16 ? std::min(4, ilog2(256 / TPL)) : 3;
    while (wlog > 1 && (A.inner % (1 << wlog) != 0 || A.nouter * (A.inner >> wlog) * nb < kTargetBlocks ||
                        kBuffers * SmemMap<L, STRIDED>::words(1 << wlog) * sizeof(float2) > 96 * 1024))
      --wlog;
    blocks = A.nouter * (A.inner >> wlog);
  } else {
    wlog = TPL >= 256 ? 0 : ilog2(256 / TPL);
    while (wlog > 0 && ((A.nouter + (1 << wlog) - 1) >> wlog) * nb < kTargetBlocks) --wlog;
    blocks = (A.nouter + (1 << wlog) - 1) >> wlog;
  }
  if (nblocks) *nblocks = blocks;
  if (query) return cudaSuccess;
  const size_t smem = kBuffers * SmemMap<L, STRIDED>::words(1 << wlog) * sizeof(float2);
  auto go = [&](auto kern) {
    // always: static shared memory (the CG hooks' scratch) comes on top, so even
    // a 48 KB request needs the opt-in
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess || blocks == 0) return e;
    const dim3 gd = STRIDED ? dim3((unsigned)(A.inner >> wlog), (unsigned)A.nouter, (unsigned)nb)
                            : dim3((unsigned)blocks, 1, (unsigned)nb);
    kern<<<gd, TPL << wlog, smem, st>>>(A, wlog);
    return cudaGetLastError();
  };
  if constexpr (!STRIDED) {
    if (A.pro_p || A.epi_part) return go(k_fft_pass<L, E, STRIDED, INV, true, 0>);
  } else {
    constexpr int kFull = E == 16 && L < 512 ? 4 : 3;
    if (wlog == kFull) return go(k_fft_pass<L, E, STRIDED, INV, false, kFull>);
  }
  return go(k_fft_pass<L, E, STRIDED, INV, false, 0>);
}

// Sixteen values per thread on strided axes of 128 and 256 points that still fill
// the GPU: one hand-off instead of two, fewer twiddles per value, and 128-byte rows
// (with the hand-offs above, a 256^3 grid's transform 105 -> 81 us forward, 104 ->
// 69 us inverse, L2 flushed; the error against 64 bits falls by a fifth).  Lines of
// 512 points need two hand-offs either way and take 64-byte rows: 32 coils of 512^2
// 28.0 -> 26.6 us forward, 26.0 -> 24.3 inverse, but a smooth image's samples are
// 1.22 times further off, so the inverse passes alone have them (their error is that
// of eight values).  The contiguous passes lose more to the registers and the
// scaling's loads, and a small pass is bound by latency: all these take eight, with
// twice the warps.
constexpr int64_t kWideWarps = 8 * 152;

template <int L, bool STRIDED, bool INV>
cudaError_t launch_L(const FftArgs& A, int nb, cudaStream_t st, int64_t* nblocks, bool query) {
  if constexpr (STRIDED && (L == 128 || L == 256 || (L == 512 && INV))) {
    if (A.nouter * A.inner * nb * (L / 16) >= kWideWarps * 32 && A.inner % 16 == 0)
      return launch_LE<L, 16, STRIDED, INV>(A, nb, st, nblocks, query);
  }
  return launch_LE<L, 8, STRIDED, INV>(A, nb, st, nblocks, query);
}

// ---------------------------------------------------------------- other line lengths
// Lines of length L = 2^a 3^b 5^c: a Stockham FFT.  Stage s of radix R and span Ns
// (the product of the earlier radices) takes butterfly j (0 <= j < L/R) from
// elements j + r L/R, multiplies input r by exp(-+ 2 pi i r k / (Ns R)), k = j mod
// Ns, transforms the R values and writes output r to (j - k) R + k + r Ns.  The
// first stage reads global memory and the last one writes it (its outputs are
// j + r Ns), both pruned and scaled as in k_fft_pass; the hand-offs between go
// through two shared-memory buffers used in turn, one barrier each.
// Radices 8 to 2 only: with 9, 10, 12, 15 and 16 too (two or three stages for
// every L) the passes were slower at every size, from a 54^2 grid (136 us for an
// 8-coil CG against 143) to 16 transforms of 384^2 (pair 151 us against 164):
// more registers, fewer threads per line and more code.
constexpr int kMaxStages = 5;
struct MixedRadix {
  int L;
  int nst;
  int radix[kMaxStages];
  int ns[kMaxStages];          // span of the stage
  uint32_t magic[kMaxStages];  // ceil(2^32 / ns): j / ns = umulhi(j, magic) for 1 < ns, j < 2^10
  float step[kMaxStages];      // 2 / (ns radix), the twiddles' angle per k in units of pi,
  float step_lo[kMaxStages];   // and what its rounding left
};

// Fewest stages, then the smallest largest radix; radices in descending order
// (the first stage has no twiddles).
void mixed_search(const int* set, int nset, int rest, int depth, int limit, int* cur, MixedRadix* best) {
  if (rest == 1) {
    if (depth > 0 && (best->nst < 0 || depth < best->nst || (depth == best->nst && cur[0] < best->radix[0]))) {
      best->nst = depth;
      for (int i = 0; i < depth; ++i) best->radix[i] = cur[i];
    }
    return;
  }
  if (depth == kMaxStages) return;
  for (int i = 0; i < nset; ++i) {
    if (set[i] > limit || rest % set[i] != 0) continue;
    cur[depth] = set[i];
    mixed_search(set, nset, rest / set[i], depth + 1, set[i], cur, best);
  }
}

MixedRadix mixed_radix(int L) {
  static const int kRadix[] = {8, 6, 5, 4, 3, 2};
  MixedRadix m;
  memset(&m, 0, sizeof(m));
  m.L = L;
  m.nst = -1;
  int cur[kMaxStages];
  mixed_search(kRadix, 6, L, 0, 8, cur, &m);
  for (int s = 0, ns = 1; s < m.nst; ns *= m.radix[s++]) {
    m.ns[s] = ns;
    m.magic[s] = (uint32_t)((0x100000000ull + ns - 1) / ns);
    const double step = 2.0 / ((double)ns * m.radix[s]);
    m.step[s] = (float)step;
    m.step_lo[s] = (float)(step - (double)m.step[s]);
  }
  return m;
}

// DFT of 3 points: with w = exp(-+ 2 pi i / 3), y1 = v0 + w v1 + w^2 v2 and
// y2 = v0 + w^2 v1 + w v2 split into (v0 - (v1 + v2) / 2) -+ i (sqrt 3 / 2)(v1 - v2).
template <bool INV>
__device__ __forceinline__ void dft3(float2* v) {
  const float h = 0.86602540378443864676f;   // sqrt(3) / 2
  const float2 t1 = cadd(v[1], v[2]);
  const float2 t2 = make_float2(v[0].x - 0.5f * t1.x, v[0].y - 0.5f * t1.y);
  const float2 t3 = rot90<INV>(cscale(csub(v[1], v[2]), h));
  v[0] = cadd(v[0], t1);
  v[1] = cadd(t2, t3);
  v[2] = csub(t2, t3);
}

// DFT of 5 points: with c_k = cos(2 pi k / 5), s_k = sin(2 pi k / 5),
// y1, y4 = v0 + c1 (v1 + v4) + c2 (v2 + v3) -+ i (s1 (v1 - v4) + s2 (v2 - v3)),
// y2, y3 = v0 + c2 (v1 + v4) + c1 (v2 + v3) -+ i (s2 (v1 - v4) - s1 (v2 - v3)).
template <bool INV>
__device__ __forceinline__ void dft5(float2* v) {
  const float c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;
  const float s1 = 0.95105651629515357212f, s2 = 0.58778525229247312917f;
  const float2 t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
  const float2 t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
  const float2 a1 = make_float2(v[0].x + c1 * t1.x + c2 * t2.x, v[0].y + c1 * t1.y + c2 * t2.y);
  const float2 a2 = make_float2(v[0].x + c2 * t1.x + c1 * t2.x, v[0].y + c2 * t1.y + c1 * t2.y);
  const float2 b1 = rot90<INV>(make_float2(s1 * t3.x + s2 * t4.x, s1 * t3.y + s2 * t4.y));
  const float2 b2 = rot90<INV>(make_float2(s2 * t3.x - s1 * t4.x, s2 * t3.y - s1 * t4.y));
  v[0] = make_float2(v[0].x + t1.x + t2.x, v[0].y + t1.y + t2.y);
  v[1] = cadd(a1, b1);
  v[4] = csub(a1, b1);
  v[2] = cadd(a2, b2);
  v[3] = csub(a2, b2);
}

template <int R, bool INV>
__device__ __forceinline__ void dft_any(float2* v);

// DFT of N = N1 N2 points, N1 and N2 coprime, without twiddles (Good and Thomas):
// input (N2 n1 + N1 n2) mod N, output (N2 u1 k1 + N1 u2 k2) mod N with
// u1 = N2^-1 mod N1, u2 = N1^-1 mod N2.
constexpr int inv_mod(int a, int m) {
  for (int x = 1; x < m; ++x)
    if (a * x % m == 1) return x;
  return 0;
}
template <int N1, int N2, bool INV>
__device__ __forceinline__ void dft_coprime(float2* v) {
  constexpr int N = N1 * N2, u1 = inv_mod(N2 % N1, N1) * N2, u2 = inv_mod(N1 % N2, N2) * N1;
  float2 a[N1][N2];
#pragma unroll
  for (int i = 0; i < N1; ++i) {
#pragma unroll
    for (int j = 0; j < N2; ++j) a[i][j] = v[(N2 * i + N1 * j) % N];
    dft_any<N2, INV>(a[i]);
  }
#pragma unroll
  for (int j = 0; j < N2; ++j) {
    float2 c[N1];
#pragma unroll
    for (int i = 0; i < N1; ++i) c[i] = a[i][j];
    dft_any<N1, INV>(c);
#pragma unroll
    for (int i = 0; i < N1; ++i) v[(u1 * i + u2 * j) % N] = c[i];
  }
}

template <int R, bool INV>
__device__ __forceinline__ void dft_any(float2* v) {
  if constexpr (R == 2) dft2<INV>(v);
  else if constexpr (R == 3) dft3<INV>(v);
  else if constexpr (R == 5) dft5<INV>(v);
  else if constexpr (R == 6) dft_coprime<2, 3, INV>(v);
  else dft<R, INV>(v);
}

// exp(-+ i pi k (step + step_lo)): sincospif of the rounded angle, corrected to
// first order for what the rounding left.
template <bool INV>
__device__ __forceinline__ float2 mixed_root(int k, float step, float step_lo) {
  const float kf = (float)k, a = kf * step;
  const float d = 3.14159265358979f * (fmaf(kf, step, -a) + kf * step_lo);
  float sn, cs;
  sincospif(a, &sn, &cs);
  const float c1 = fmaf(-sn, d, cs), s1 = fmaf(cs, d, sn);
  return make_float2(c1, INV ? s1 : -s1);
}

// Input r of a butterfly times w1^r, w1 = exp(-+ i pi k step): w1, for R >= 5 also
// w1^2 (a power multiplies the root's error, and a second root halves the powers),
// and products of depth at most three.
template <int R, bool INV>
__device__ __forceinline__ void mixed_twiddles(float2* v, int k, float step, float step_lo) {
  float2 w[8];
  w[1] = mixed_root<INV>(k, step, step_lo);
  if (R >= 5) w[2] = mixed_root<INV>(2 * k, step, step_lo);
#pragma unroll
  for (int r = 1; r < R; ++r) {
    if (r > 2 || (r == 2 && R < 5)) w[r] = cmul(w[r / 2], w[r - r / 2]);
    v[r] = cmul(v[r], w[r]);
  }
}

// Shared-memory position of element p of line b: strided axis, rows of W columns
// (a skewed row for fewer than 16, so that the threads of a half-warp in
// neighbouring rows differ mod 16); contiguous axis, one pad word per 8.
template <bool STRIDED>
struct MixedMap {
  int wlog, pitch;
  __device__ __forceinline__ MixedMap(int wl, int L) : wlog(wl), pitch(L + (L >> 3) + 1) {}
  __device__ __forceinline__ int at(int b, int p) const {
    return STRIDED ? ((wlog < 4 ? p + (p >> 3) : p) << wlog) + b : b * pitch + p + (p >> 3);
  }
  __host__ __device__ static size_t words(int wlog, int L) { return (size_t)(L + (L >> 3) + 1) << wlog; }
};

// f(integral_constant<int, R>) for a runtime radix R.
template <class F>
__device__ __forceinline__ void for_radix(int R, F f) {
  switch (R) {
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 5: f(std::integral_constant<int, 5>{}); break;
    case 6: f(std::integral_constant<int, 6>{}); break;
    default: f(std::integral_constant<int, 8>{}); break;
  }
}

// grid: as k_fft_pass.  blockDim = TPL << wlog, TPL threads per line.
template <bool STRIDED, bool INV, bool HOOK>
__global__ void __launch_bounds__(512)
k_fft_mixed(const FftArgs A, const int wlog, const __grid_constant__ MixedRadix mr) {
  const int L = mr.L;
  const int TPL = blockDim.x >> wlog;
  const MixedMap<STRIDED> SI(wlog, L);
  extern __shared__ float2 sm[];

  const int tid = threadIdx.x;
  int b, t, o, in;
  if (STRIDED) {
    b = tid & ((1 << wlog) - 1);
    t = tid >> wlog;
    o = blockIdx.y;
    in = (blockIdx.x << wlog) + b;
  } else {
    b = tid / TPL;
    t = tid - b * TPL;
    o = (blockIdx.x << wlog) + b;
    in = 0;
  }
  const bool live = o < (int)A.nouter;
  const float2* __restrict__ src = A.src + (int64_t)blockIdx.z * A.src_bstride;
  float2* __restrict__ dst = A.dst + (int64_t)blockIdx.z * A.dst_bstride;

  int goff = in;
  float slead = 1.0f;
  if (live) {
    int rem = o;
    for (int i = A.a - 1; i >= 0; --i) {
      int n = rem;
      if (i > 0) {
        rem = n / A.lead_N[i];
        n -= rem * A.lead_N[i];
      }
      const int gi = wrapk(n - A.lead_N[i] / 2 + A.lead_K[i], A.lead_K[i]);
      goff += gi * (int)A.lead_stride[i];
      if (A.scale && (A.src_image || A.dst_image)) slead *= A.s_lead[i][n];
    }
  }
  const int half = A.Na >> 1;
  const int stride = STRIDED ? (int)A.inner : 1;
  const bool pro = HOOK && !INV && A.src_image && A.pro_p;
  float beta = 0.f;
  if constexpr (HOOK && !INV) {
    __shared__ double red[32];
    if (pro) beta = cg_prologue_beta(A, red);
  }
  const uint64_t pol = l2_evict_first_policy();   // a pass reads each input element once

  // ---- first stage: global memory (pruned on the forward side) to buffer 0
  auto first = [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    const int nbf = L / R;
    for (int j = t; j < nbf; j += TPL) {
      float2 v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int p = j + r * nbf;
        v[r] = make_float2(0.f, 0.f);
        if (live) {
          if (INV) {
            v[r] = ld_last_use(&src[goff + p * stride], pol);
          } else if ((p < half) || (p >= L - half)) {
            if (A.src_image) {
              const int n = p < half ? p + half : p - L + half;
              v[r] = cscale(load_image(A, src, o * A.Na + n, pro, beta), (A.scale ? A.s_axis[n] : 1.0f) * slead);
            } else {
              v[r] = ld_last_use(&src[goff + p * stride], pol);
            }
          }
        }
      }
      dft_any<R, INV>(v);
#pragma unroll
      for (int r = 0; r < R; ++r) sm[SI.at(b, j * R + r)] = v[r];
    }
  };
  for_radix(mr.radix[0], first);
  __syncthreads();

  // ---- middle stages, from one buffer to the other
  float2* cur = sm;
  float2* nxt = sm + MixedMap<STRIDED>::words(wlog, L);
  for (int s = 1; s + 1 < mr.nst; ++s) {
    const int Ns = mr.ns[s];
    const uint32_t mg = mr.magic[s];
    for_radix(mr.radix[s], [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      const int nbf = L / R;
      for (int j = t; j < nbf; j += TPL) {
        const int k = j - (int)__umulhi((uint32_t)j, mg) * Ns;
        float2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = cur[SI.at(b, j + r * nbf)];
        mixed_twiddles<R, INV>(v, k, mr.step[s], mr.step_lo[s]);
        dft_any<R, INV>(v);
        const int base = (j - k) * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) nxt[SI.at(b, base + r * Ns)] = v[r];
      }
    });
    __syncthreads();
    float2* const tmp = cur;
    cur = nxt;
    nxt = tmp;
  }

  // ---- last stage: to global memory (pruned on the inverse side); Ns = L / R, so
  // k = j and output r is element j + r Ns
  const bool epi = HOOK && INV && A.dst_image && A.epi_part;
  double dot = 0.0;
  auto last = [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    const int nbf = L / R;
    for (int j = t; j < nbf; j += TPL) {
      float2 v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = cur[SI.at(b, j + r * nbf)];
      mixed_twiddles<R, INV>(v, j, mr.step[mr.nst - 1], mr.step_lo[mr.nst - 1]);
      dft_any<R, INV>(v);
      if (!live) continue;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int p = j + r * nbf;
        if (!INV) {
          dst[goff + p * stride] = v[r];
        } else if ((p < half) || (p >= L - half)) {
          if (A.dst_image) {
            const int n = p < half ? p + half : p - L + half;
            const float2 out = cscale(v[r], (A.scale ? A.s_axis[n] : 1.0f) * slead);
            dst[o * A.Na + n] = out;
            if (epi) {
              const float2 a = A.epi_a[o * A.Na + n];
              dot += (double)a.x * (double)out.x + (double)a.y * (double)out.y;
            }
          } else {
            dst[goff + p * stride] = v[r];
          }
        }
      }
    }
  };
  for_radix(mr.radix[mr.nst - 1], last);
  if constexpr (HOOK && INV) {
    __shared__ double red[32];
    if (epi) {
      const double tsum = block_sum_dbl(dot, red);
      if (threadIdx.x == 0) A.epi_part[blockIdx.x] = tsum;
    }
  }
}

// One thread per butterfly of the smallest radix (at most 256 per line), W lines
// per CTA: up to 16 columns on a strided axis (W | inner), as many lines as give
// 256 threads on the contiguous one, and W lowered while the launch would give fewer
// than two CTAs per SM.  At most 512 threads: a strided axis gives up columns for
// that down to 8, rows of 64 bytes, and then lets a thread take several butterflies
// (16 transforms of 360 x 288: 12.3 us with 8 columns of 60 threads, 18.8 with 4 of
// 120).
template <bool STRIDED, bool INV>
cudaError_t launch_mixed(int L, const FftArgs& A, int nb, cudaStream_t st, int64_t* nblocks, bool query) {
  const MixedRadix mr = mixed_radix(L);
  if (mr.nst < 2) return cudaErrorInvalidValue;
  int tpl = std::min(256, L / mr.radix[mr.nst - 1]);
  auto smem = [&](int wlog) {
    return (size_t)std::min(2, mr.nst - 1) * MixedMap<STRIDED>::words(wlog, L) * sizeof(float2);
  };
  int wlog = 0;
  int64_t blocks;
  if (STRIDED) {
    wlog = 4;
    while (wlog > 0 && (A.inner % (1 << wlog) != 0 || A.nouter * (A.inner >> wlog) * nb < kTargetBlocks ||
                        smem(wlog) > 100 * 1024 || (wlog > 3 && (tpl << wlog) > 512)))
      --wlog;
    const int rounds = (tpl + (512 >> wlog) - 1) / (512 >> wlog);
    tpl = (tpl + rounds - 1) / rounds;
    blocks = A.nouter * (A.inner >> wlog);
  } else {
    while ((tpl << (wlog + 1)) <= 256) ++wlog;
    while (wlog > 0 && ((A.nouter + (1 << wlog) - 1) >> wlog) * nb < kTargetBlocks) --wlog;
    blocks = (A.nouter + (1 << wlog) - 1) >> wlog;
  }
  if (nblocks) *nblocks = blocks;
  if (query) return cudaSuccess;
  auto go = [&](auto kern) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem(wlog));
    if (e != cudaSuccess || blocks == 0) return e;
    const dim3 gd = STRIDED ? dim3((unsigned)(A.inner >> wlog), (unsigned)A.nouter, (unsigned)nb)
                            : dim3((unsigned)blocks, 1, (unsigned)nb);
    kern<<<gd, tpl << wlog, smem(wlog), st>>>(A, wlog, mr);
    return cudaGetLastError();
  };
  if constexpr (!STRIDED) {
    if (A.pro_p || A.epi_part) return go(k_fft_mixed<STRIDED, INV, true>);
  }
  return go(k_fft_mixed<STRIDED, INV, false>);
}

template <bool STRIDED, bool INV>
cudaError_t launch_any(int L, const FftArgs& A, int nb, cudaStream_t st, int64_t* nblocks = nullptr,
                       bool query = false) {
  switch (L) {
    case 16: return launch_L<16, STRIDED, INV>(A, nb, st, nblocks, query);
    case 32: return launch_L<32, STRIDED, INV>(A, nb, st, nblocks, query);
    case 64: return launch_L<64, STRIDED, INV>(A, nb, st, nblocks, query);
    case 128: return launch_L<128, STRIDED, INV>(A, nb, st, nblocks, query);
    case 256: return launch_L<256, STRIDED, INV>(A, nb, st, nblocks, query);
    case 512: return launch_L<512, STRIDED, INV>(A, nb, st, nblocks, query);
    case 1024: return launch_L<1024, STRIDED, INV>(A, nb, st, nblocks, query);
    default: return launch_mixed<STRIDED, INV>(L, A, nb, st, nblocks, query);
  }
}

FftArgs make_args(const nufft_plan_t* p, int a) {
  FftArgs A;
  memset(&A, 0, sizeof(A));
  const Geom& g = p->g;
  A.a = a;
  A.Na = g.N[a];
  A.s_axis = p->s + p->s_off[a];
  A.nouter = 1;
  for (int i = 0; i < a; ++i) {
    A.lead_N[i] = g.N[i];
    A.lead_K[i] = g.K[i];
    A.lead_stride[i] = g.Kstride[i];
    A.s_lead[i] = p->s + p->s_off[i];
    A.nouter *= g.N[i];
  }
  A.inner = g.Kstride[a];
  return A;
}

}  // namespace

int launch_fft_forward(nufft_plan_t* p, const float2* x, float2* grid, int nb, bool scale, const CgHooks* h) {
  const int d = p->g.d;
  if (h && nb != 1) return set_error(p, NUFFT_EINVAL, "CG hooks need a single transform");
  for (int a = d - 1; a >= 0; --a) {
    FftArgs A = make_args(p, a);
    A.scale = scale ? 1 : 0;
    A.src_image = (a == d - 1);
    if (h && A.src_image && h->pro_p) {
      A.pro_p = h->pro_p;
      A.pro_r = h->pro_r;
      A.pro_part = h->pro_part;
      A.pro_count = h->pro_count;
      A.pro_sc = h->pro_sc;
      A.pro_old = h->pro_old;
      A.pro_new = h->pro_new;
    }
    A.src = A.src_image ? x : grid;
    A.dst = grid;
    A.src_bstride = A.src_image ? p->Nprod : p->Kprod;
    A.dst_bstride = p->Kprod;
    const bool strided = A.inner > 1;
    cudaError_t e = strided ? launch_any<true, false>(p->g.K[a], A, nb, p->stream)
                            : launch_any<false, false>(p->g.K[a], A, nb, p->stream);
    if (e != cudaSuccess) return cuda_check(p, e, "forward FFT pass");
  }
  return NUFFT_OK;
}

int fft_inverse_last_blocks(nufft_plan_t* p, int64_t* blocks) {
  const int a = p->g.d - 1;
  FftArgs A = make_args(p, a);
  A.dst_image = 1;
  const bool strided = A.inner > 1;
  cudaError_t e = strided ? launch_any<true, true>(p->g.K[a], A, 1, p->stream, blocks, true)
                          : launch_any<false, true>(p->g.K[a], A, 1, p->stream, blocks, true);
  return e == cudaSuccess ? NUFFT_OK : cuda_check(p, e, "inverse FFT pass");
}

int launch_fft_inverse(nufft_plan_t* p, float2* grid, float2* x, int nb, bool scale, const CgHooks* h) {
  const int d = p->g.d;
  if (h && nb != 1) return set_error(p, NUFFT_EINVAL, "CG hooks need a single transform");
  for (int a = 0; a < d; ++a) {
    FftArgs A = make_args(p, a);
    A.scale = scale ? 1 : 0;
    A.dst_image = (a == d - 1);
    A.src = grid;
    A.dst = A.dst_image ? x : grid;
    A.src_bstride = p->Kprod;
    A.dst_bstride = A.dst_image ? p->Nprod : p->Kprod;
    const bool epi = h && A.dst_image && h->epi_part;
    if (epi) {
      A.epi_a = h->epi_a;
      A.epi_part = h->epi_part;
    }
    const bool strided = A.inner > 1;
    int64_t blocks = 0;
    if (epi) {   // the block count first: the partial sums must fit
      cudaError_t e = strided ? launch_any<true, true>(p->g.K[a], A, nb, p->stream, &blocks, true)
                              : launch_any<false, true>(p->g.K[a], A, nb, p->stream, &blocks, true);
      if (e != cudaSuccess) return cuda_check(p, e, "inverse FFT pass");
      if (blocks > h->epi_cap)
        return set_error(p, NUFFT_EINVAL, "CG hooks: %lld partial sums exceed the capacity %d", (long long)blocks,
                         h->epi_cap);
      *h->epi_count = (int)blocks;
    }
    cudaError_t e = strided ? launch_any<true, true>(p->g.K[a], A, nb, p->stream)
                            : launch_any<false, true>(p->g.K[a], A, nb, p->stream);
    if (e != cudaSuccess) return cuda_check(p, e, "inverse FFT pass");
  }
  return NUFFT_OK;
}

}  // namespace nufft
