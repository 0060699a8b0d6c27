// interp.cu - interpolation V (grid -> k-space) and gridding V^H
// (k-space -> grid) with the min-max interpolator.
//
// Section 2.1.3: V maps the oversampled grid to the M non-uniform points, each
// point combining its J^d neighbours; gridding is its conjugate transpose.
// The paper stores V as a CSR matrix and runs a sparse matrix-vector product
// for both directions.  Here each point keeps only its first neighbour per
// dimension and J coefficients per dimension (the d-dimensional weight is their
// product), and points are sorted by grid tile at plan time.
//
// Interpolation: a group of J_last lanes handles one point; lane l owns the
// l-th neighbour along the last (contiguous) axis, so the group reads J_last
// consecutive grid cells per neighbour row, and the partial sums are combined
// with warp shuffles.
//
// Gridding: one CTA per chunk of a tile's points accumulates conj(weight) * y
// into a shared-memory copy of the tile extended by J-1 cells per dimension
// (the "padded tile"), then writes the padded tile to a per-chunk buffer.  A
// second kernel forms every grid cell of a tile as the sum, in a fixed order,
// of the padded tiles that cover it (its own tile's chunks and those of the
// 2^d - 1 lower neighbour tiles).  No global atomics; every grid cell is
// written exactly once.
#include <algorithm>
#include <mutex>

#include "internal.cuh"

namespace nufft {
namespace {

// ---------------------------------------------------------------- interpolation
// Sum of `part` over the lanes base .. base + G - 1 of a lane group, valid in
// lane base; every lane of the warp takes part.  Groups of 6 (J = 6) sum as
// (p0 + p3) + (p1 + p4) + (p2 + p5) with three shuffle steps; other widths add
// the lanes in order.
template <int JF>
__device__ __forceinline__ float2 lane_group_sum(float2 part, int base, int G) {
  if constexpr (JF == 6) {
    float2 a, s;
    a.x = part.x + __shfl_down_sync(0xffffffffu, part.x, 3);
    a.y = part.y + __shfl_down_sync(0xffffffffu, part.y, 3);
    s.x = a.x + __shfl_down_sync(0xffffffffu, a.x, 1);
    s.y = a.y + __shfl_down_sync(0xffffffffu, a.y, 1);
    s.x += __shfl_down_sync(0xffffffffu, a.x, 2);
    s.y += __shfl_down_sync(0xffffffffu, a.y, 2);
    return s;
  } else {
    float2 tot = make_float2(0.f, 0.f);
    for (int r = 0; r < G; ++r) {
      const int src = (base + r) & 31;
      tot.x += __shfl_sync(0xffffffffu, part.x, src);
      tot.y += __shfl_sync(0xffffffffu, part.y, src);
    }
    return tot;
  }
}

// 2D batches with CTAs enough: a thread takes kBatchPer batch elements in turn with
// the point's neighbours and coefficients in registers (JF > 0), so that each element
// costs its J_0 grid loads only.  Fewer CTAs than kBatchPerCtas are bound by the
// chain of a thread's elements and take k_interp, one element per CTA row.  Measured,
// this kernel against k_interp: 1000 points, 4 images 7.4 us against 2.6 (25 CTAs);
// 57,600 points, 2 images 8.2 against 7.7 (1440); 10,000 points, 32 images 17.9
// against 17.5 (2000); 25,000 points, 16 images 18.5 against 20.3 (2500).
constexpr int kBatchPer = 4;
constexpr int64_t kBatchPerCtas = 16 * 152;

template <int JF>
__global__ void __launch_bounds__(256)
k_interp_batch2d(const float2* __restrict__ grid_b, float2* __restrict__ y_b, const Points P, const Geom g, int64_t gbs,
                 int64_t ybs, int nb) {
  const int lane = threadIdx.x & 31;
  constexpr int PW = 32 / JF;
  const int sub = lane / JF;
  const int l = lane - sub * JF;
  const int64_t i = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * PW + sub;
  const bool active = sub < PW && i < P.M;
  float2 c0[JF], cl = make_float2(0.f, 0.f);
  int off[JF], m = 0;
#pragma unroll
  for (int j = 0; j < JF; ++j) {
    c0[j] = make_float2(0.f, 0.f);
    off[j] = 0;
  }
  if (active) {
    const int k0 = P.kf[i];
    const int gl = wrapk(P.kf[P.M + i] + l, g.K[1]);
    m = P.perm[i];
    cl = P.coef[P.coef_off[1] + (int64_t)l * P.M + i];
#pragma unroll
    for (int j = 0; j < JF; ++j) {
      c0[j] = P.coef[P.coef_off[0] + (int64_t)j * P.M + i];
      off[j] = wrapk(k0 + j, g.K[0]) * (int)g.Kstride[0] + gl;
    }
  }
  const int b0 = blockIdx.y * kBatchPer, b1 = min(nb, b0 + kBatchPer);
  const float2* __restrict__ grid = grid_b + b0 * gbs;
  float2* __restrict__ y = y_b + b0 * ybs + m;
  for (int b = b0; b < b1; ++b, grid += gbs, y += ybs) {   // CTA-uniform
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < JF; ++j) acc = cfma(c0[j], __ldg(&grid[off[j]]), acc);
    const float2 tot = lane_group_sum<JF>(cmul(cl, acc), sub * JF, JF);
    if (active && l == 0) *y = tot;
  }
}

template <int D, int JF>
__global__ void __launch_bounds__(256)
k_interp(const float2* __restrict__ grid_b, float2* __restrict__ y_b, const Points P, const Geom g, int64_t gbs,
         int64_t ybs) {
  const float2* __restrict__ grid = grid_b + (int64_t)blockIdx.y * gbs;
  float2* __restrict__ y = y_b + (int64_t)blockIdx.y * ybs;
  const int G = JF > 0 ? JF : g.J[D - 1];
  const int lane = threadIdx.x & 31;
  const int per_warp = 32 / G;
  const int sub = lane / G;
  const int l = lane - sub * G;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t i = warp * per_warp + sub;
  const bool active = (sub < per_warp) && (i < P.M);

  float2 part = make_float2(0.f, 0.f);
  if (active) {
    const int J0 = JF > 0 ? JF : g.J[0];
    const int J1 = JF > 0 ? JF : (D > 1 ? g.J[1] : 1);
    const int kl = P.kf[(int64_t)(D - 1) * P.M + i];
    const int Klast = g.K[D - 1];
    const int gl = wrapk(kl + l, Klast);
    const float2 cl = P.coef[P.coef_off[D - 1] + (int64_t)l * P.M + i];
    if (D == 1) {
      part = cmul(cl, __ldg(&grid[gl]));
    } else if (D == 2) {
      const int k0 = P.kf[i];
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll
      for (int j0 = 0; j0 < (JF > 0 ? JF : kMaxJ); ++j0) {
        if (JF == 0 && j0 >= J0) break;
        const float2 c0 = P.coef[P.coef_off[0] + (int64_t)j0 * P.M + i];
        const int row = wrapk(k0 + j0, g.K[0]) * (int)g.Kstride[0];
        acc = cfma(c0, __ldg(&grid[row + gl]), acc);
      }
      part = cmul(cl, acc);
    } else {
      const int k0 = P.kf[i];
      const int k1 = P.kf[P.M + i];
      float2 c1v[JF > 0 ? JF : kMaxJ];
#pragma unroll
      for (int j1 = 0; j1 < (JF > 0 ? JF : kMaxJ); ++j1) {
        if (JF == 0 && j1 >= J1) break;
        c1v[j1] = P.coef[P.coef_off[1] + (int64_t)j1 * P.M + i];
      }
      // row offsets of the J1 neighbour rows within a plane (32-bit: K^d < 2^31)
      int rowoff[JF > 0 ? JF : kMaxJ];
#pragma unroll
      for (int j1 = 0; j1 < (JF > 0 ? JF : kMaxJ); ++j1) {
        if (JF == 0 && j1 >= J1) break;
        rowoff[j1] = wrapk(k1 + j1, g.K[1]) * (int)g.Kstride[1] + gl;
      }
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll 1
      for (int j0 = 0; j0 < J0; ++j0) {
        const float2 c0 = P.coef[P.coef_off[0] + (int64_t)j0 * P.M + i];
        const float2* plane = grid + wrapk(k0 + j0, g.K[0]) * (int)g.Kstride[0];
        float2 acc1 = make_float2(0.f, 0.f);
#pragma unroll
        for (int j1 = 0; j1 < (JF > 0 ? JF : kMaxJ); ++j1) {
          if (JF == 0 && j1 >= J1) break;
          acc1 = cfma(c1v[j1], __ldg(&plane[rowoff[j1]]), acc1);
        }
        acc = cfma(c0, acc1, acc);
      }
      part = cmul(cl, acc);
    }
  }
  // Sum the G partial values of each lane group (a fixed order).
  const float2 tot = lane_group_sum<JF>(part, sub * G, G);
  if (active && l == 0) y[P.perm[i]] = tot;
}

// ---------------------------------------------------------------- interpolation, per chunk
// One CTA per chunk of a tile's points.  The chunk's padded tile of
// the grid ((T+J-1)^d cells, wrapped at the grid edge) is copied into shared
// memory once, as a plane of real parts and a plane of imaginary parts, and
// every point gathers its J^d neighbours from there instead of from global
// memory.  The plan orders each chunk so that the points sharing a warp
// instruction read disjoint bank windows of these planes (the gridding uses
// the same order for its atomics).  Lane layout, arithmetic and summation
// order are those of k_interp (results agree to rounding: the compiler may
// fuse the multiply-adds differently in the two kernels).

// 3D, any J (k_interp_chunk3d takes equal J from 4 to 7).
__global__ void __launch_bounds__(512, 2)
k_interp_chunk3d_any(const float2* __restrict__ grid, float2* __restrict__ y, const Chunk* __restrict__ chunks,
                     const Points P, const Geom g) {
  extern __shared__ float tile[];
  const int ncell = (int)g.padded_cells;
  const int P1 = g.P[1], P2 = g.P[2];
  float* gre = tile;
  float* gim = tile + ncell;
  const Chunk ch = chunks[blockIdx.x];
  int org[3];
  {
    int rem = ch.bin;
    for (int a = 2; a >= 0; --a) {
      org[a] = (rem % g.nb[a]) * g.T[a];
      rem /= g.nb[a];
    }
  }
  // the padded tile, cell c = (r0, r1, r2) in C order with pitches P
  for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
    const int r2 = c % P2, r1 = (c / P2) % P1, r0 = c / (P2 * P1);
    const float2 v = __ldg(&grid[wrapk(org[0] + r0, g.K[0]) * (int)g.Kstride[0] +
                                 wrapk(org[1] + r1, g.K[1]) * (int)g.Kstride[1] + wrapk(org[2] + r2, g.K[2])]);
    gre[c] = v.x;
    gim[c] = v.y;
  }
  __syncthreads();

  const int G = g.J[2], J0 = g.J[0], J1 = g.J[1];
  const int lane = threadIdx.x & 31;
  const int per_warp = 32 / G;
  const int sub = lane / G;
  const int l = lane - sub * G;
  const int warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  // warp-uniform rounds of per_warp points (the lane-group sum is a full-warp shuffle)
  for (int qb = warp * per_warp; qb < ch.count; qb += nwarps * per_warp) {
    const int q = qb + sub;
    const bool act = (sub < per_warp) && (q < ch.count);
    const int64_t i = (int64_t)ch.start + q;
    float2 part = make_float2(0.f, 0.f);
    if (act) {
      const int ll = P.kf[2 * P.M + i] - org[2] + l;
      const float2 cl = P.coef[P.coef_off[2] + (int64_t)l * P.M + i];
      const int l0 = P.kf[i] - org[0], l1 = P.kf[P.M + i] - org[1];
      float2 acc = make_float2(0.f, 0.f);
      float2 c1v[kMaxJ];
#pragma unroll
      for (int j1 = 0; j1 < kMaxJ; ++j1) {
        if (j1 >= J1) break;
        c1v[j1] = P.coef[P.coef_off[1] + (int64_t)j1 * P.M + i];
      }
#pragma unroll 1
      for (int j0 = 0; j0 < J0; ++j0) {
        const float2 c0 = P.coef[P.coef_off[0] + (int64_t)j0 * P.M + i];
        const int rowbase = ((l0 + j0) * P1 + l1) * P2 + ll;
        float2 acc1 = make_float2(0.f, 0.f);
#pragma unroll
        for (int j1 = 0; j1 < kMaxJ; ++j1) {
          if (j1 >= J1) break;
          const int cell = rowbase + j1 * P2;
          acc1 = cfma(c1v[j1], make_float2(gre[cell], gim[cell]), acc1);
        }
        acc = cfma(c0, acc1, acc);
      }
      part = cmul(cl, acc);
    }
    const float2 tot = lane_group_sum<0>(part, sub * G, G);
    if (act && l == 0) y[P.perm[i]] = tot;
  }
}

// Packed pairs of floats: two FP32 multiply-adds in one instruction (fma.rn.f32x2),
// each rounded as fmaf.  The FP32 pipe takes it at half rate, so it saves issue
// slots, not pipe time: the gathers below issue two loads and two of these per
// complex tap where four fmaf were.
struct f32x2 {
  unsigned long long v;
};
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// 3D with every J = JF (4 to 7): as k_interp_chunk3d_any, and every warp keeps the next
// round's point data in flight while it gathers this one's, with no barrier
// between rounds: lane l of a point loads the l-th coefficient of each axis into
// registers a round ahead; the axis-0 and axis-1 ones reach the point's other
// lanes through a per-warp strip of shared memory.  The J axis-1 taps of a row
// are taken two at a time (fma2 on the pairs (re_j, re_j+1) and (im_j, im_j+1)).
// 128^3 kooshball: 338 us with sub-batches between barriers, 271 us so; bound by
// the shared-memory pipe (86 % busy): two loads per tap.
template <int JF>
struct Chunk3dCfg {
  static constexpr int kThreads = 512;
  static constexpr int kPerWarp = 32 / JF;
  static constexpr int kStrip = 2 * JF * kPerWarp;   // float2 per warp
  // gridding: two words per cell, the samples and the strips, or three words
  static size_t smem_gridding(int64_t cells) {
    return std::max((size_t)cells * 2 * sizeof(int) +
                        ((size_t)kChunkPoints[3] + (kThreads / 32) * kStrip) * sizeof(float2),
                    (size_t)cells * 3 * sizeof(int));
  }
  static size_t smem_interp(int64_t cells) {
    return (size_t)cells * 2 * sizeof(float) + (size_t)(kThreads / 32) * kStrip * sizeof(float2);
  }
};

template <int JF, int TF>
__global__ void __launch_bounds__(Chunk3dCfg<JF>::kThreads, 2)
k_interp_chunk3d(const float2* __restrict__ grid_b, float2* __restrict__ y_b, const Chunk* __restrict__ chunks,
                 const Points P, const Geom g, int64_t gbs, int64_t ybs) {
  constexpr int PF = TF > 0 ? TF + JF - 1 : 0;
  constexpr int PW = Chunk3dCfg<JF>::kPerWarp;
  extern __shared__ float tile[];
  const float2* __restrict__ grid = grid_b + (int64_t)blockIdx.y * gbs;
  float2* __restrict__ y = y_b + (int64_t)blockIdx.y * ybs;
  const int P0 = TF > 0 ? PF : g.P[0];
  const int P1 = TF > 0 ? PF : g.P[1];
  const int P2 = TF > 0 ? PF : g.P[2];
  const int ncell = P0 * P1 * P2;
  float* gre = tile;
  float* gim = tile + ncell;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  // strip: c0 as float2 [JF][PW], then the real and the imaginary parts of c1,
  // [PW][JF] floats each, so that a point's pairs are adjacent
  float2* s_c0 = reinterpret_cast<float2*>(tile + 2 * ncell) + warp * Chunk3dCfg<JF>::kStrip;
  float* s_x1 = reinterpret_cast<float*>(s_c0 + JF * PW);
  float* s_y1 = s_x1 + JF * PW;
  const Chunk ch = chunks[blockIdx.x];
  int org[3];
  {
    int rem = ch.bin;
    for (int a = 2; a >= 0; --a) {
      org[a] = (rem % g.nb[a]) * g.T[a];
      rem /= g.nb[a];
    }
  }
  const int sub = lane / JF;
  const int l = lane - sub * JF;
  constexpr int step = (Chunk3dCfg<JF>::kThreads / 32) * PW;
  const int64_t M = P.M;
  const float2* pc0 = P.coef + P.coef_off[0] + (int64_t)l * M + ch.start;
  const float2* pc1 = P.coef + P.coef_off[1] + (int64_t)l * M + ch.start;
  const float2* pc2 = P.coef + P.coef_off[2] + (int64_t)l * M + ch.start;
  const int32_t* pk = P.kf + ch.start;
  const int32_t* pp = P.perm + ch.start;
  int qb = warp * PW;
  bool act = sub < PW && qb + sub < ch.count;
  float2 n0 = make_float2(0.f, 0.f), n1 = n0, n2 = n0;
  int k0 = 0, k1 = 0, k2 = 0, m = 0;
  if (act) {   // in flight while the tile is copied
    const int q = qb + sub;
    n0 = pc0[q]; n1 = pc1[q]; n2 = pc2[q];
    k0 = pk[q]; k1 = pk[M + q]; k2 = pk[2 * M + q];
    m = pp[q];
  }
  // the padded tile, kBatch cells of a thread in flight at a time (32-bit grid
  // offsets: K^d <= 2^30)
  constexpr int kBatch = 10;
  for (int c0 = threadIdx.x; c0 < ncell; c0 += kBatch * Chunk3dCfg<JF>::kThreads) {
    float2 v[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int c = c0 + k * Chunk3dCfg<JF>::kThreads;
      if (c < ncell) {
        const int r2 = c % P2, r01 = c / P2, r1 = r01 % P1, r0 = r01 / P1;
        const int gi = wrapk(org[0] + r0, g.K[0]) * (int)g.Kstride[0] + wrapk(org[1] + r1, g.K[1]) * (int)g.Kstride[1] +
                       wrapk(org[2] + r2, g.K[2]);
        v[k] = __ldg(&grid[gi]);
      }
    }
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int c = c0 + k * Chunk3dCfg<JF>::kThreads;
      if (c < ncell) {
        gre[c] = v[k].x;
        gim[c] = v[k].y;
      }
    }
  }
  __syncthreads();
  for (; qb < ch.count; qb += step) {   // warp-uniform
    const bool cur = act;
    const float2 cl = n2;
    const int mc = m;
    int base = 0;
    __syncwarp();   // the strip's readers of the previous round are done
    if (cur) {
      s_c0[l * PW + sub] = n0;
      s_x1[sub * JF + l] = n1.x;
      s_y1[sub * JF + l] = n1.y;
      base = ((k0 - org[0]) * P1 + k1 - org[1]) * P2 + k2 - org[2] + l;
    }
    const int qn = qb + step + sub;
    act = sub < PW && qn < ch.count;
    if (act) {
      n0 = pc0[qn]; n1 = pc1[qn]; n2 = pc2[qn];
      k0 = pk[qn]; k1 = pk[M + qn]; k2 = pk[2 * M + qn];
      m = pp[qn];
    }
    __syncwarp();
    float2 part = make_float2(0.f, 0.f);
    if (cur) {
      float x1[JF], y1[JF];
      if (JF & 1) {
#pragma unroll
        for (int j = 0; j < JF; ++j) {
          x1[j] = s_x1[sub * JF + j];
          y1[j] = s_y1[sub * JF + j];
        }
      } else {   // the pairs are 8-byte aligned
#pragma unroll
        for (int j = 0; j + 1 < JF; j += 2) {
          const float2 vx = *reinterpret_cast<const float2*>(&s_x1[sub * JF + j]);
          const float2 vy = *reinterpret_cast<const float2*>(&s_y1[sub * JF + j]);
          x1[j] = vx.x; x1[j + 1] = vx.y;
          y1[j] = vy.x; y1[j + 1] = vy.y;
        }
      }
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll
      for (int j0 = 0; j0 < JF; ++j0) {
        const float* re = gre + base + j0 * P1 * P2;
        const float* im = gim + base + j0 * P1 * P2;
        f32x2 ar = pack2(0.f, 0.f), ai = ar;
#pragma unroll
        for (int j = 0; j + 1 < JF; j += 2) {
          const f32x2 vx = pack2(re[j * P2], re[(j + 1) * P2]), vy = pack2(im[j * P2], im[(j + 1) * P2]);
          const f32x2 cx = pack2(x1[j], x1[j + 1]), cy = pack2(y1[j], y1[j + 1]);
          const f32x2 ny = pack2(-y1[j], -y1[j + 1]);
          ar = fma2(cx, vx, ar);
          ai = fma2(cx, vy, ai);
          ar = fma2(ny, vy, ar);
          ai = fma2(cy, vx, ai);
        }
        const float2 r2 = unpack2(ar), i2 = unpack2(ai);
        float2 t = make_float2(r2.x + r2.y, i2.x + i2.y);
        if (JF & 1) t = cfma(make_float2(x1[JF - 1], y1[JF - 1]), make_float2(re[(JF - 1) * P2], im[(JF - 1) * P2]), t);
        acc = cfma(s_c0[j0 * PW + sub], t, acc);
      }
      part = cmul(cl, acc);
    }
    const float2 tot = lane_group_sum<JF>(part, sub * JF, JF);
    if (cur && l == 0) y[mc] = tot;
  }
}

// ---------------------------------------------------------------- 2D chunks, staged
// Single 2D transforms: the chunk's point data are staged in shared memory too,
// one thread per point (first neighbours, the J0 + J1 coefficients, permutation
// or sample), so a CTA waits for one round of global loads instead of one per
// pass of its warps over the chunk.  Layout: c0[J0][cap] (row by row: the lanes
// of a point read one value), c1[cap][pitch1] (point by point: the lanes of a
// point read consecutive words; an odd pitch keeps the staging threads' stores
// on distinct banks, 2- to 4-way conflicts otherwise, see staged_pitch), k[2][cap]
// (first neighbours relative to the tile origin).
// JF > 0: J0 = J1 = JF; TF > 0: 16^2 tiles, so that the rows of a point's
// neighbours are immediate offsets.
struct Tile2d {
  int org0, org1;   // tile origin on the grid
};
__device__ __forceinline__ Tile2d tile_origin2d(const Geom& g, int bin) {
  const int b0 = bin / g.nb[1];
  return {b0 * g.T[0], (bin - b0 * g.nb[1]) * g.T[1]};
}

struct Staged2d {
  float2* c0;
  float2* c1;
  int* k;
  int pitch1;
  // float2 of shared memory per chunk for the coefficients
  static size_t coefs(int J0, int pitch) { return (size_t)kChunkPoints[2] * (J0 + pitch); }
};

// pitch1 of the staged kernels: J1 | 1, or J1 where the odd pitch would cost a CTA per
// SM (`rest` bytes of shared memory beside the coefficients).  J = 4 to 7 always have
// room.  J = 16: three CTAs per SM, two with the odd pitch; 40,000 points on a
// 360 x 288 grid (432 chunks) 17.7 us against 26.3.
int staged_pitch(int J0, int J1, size_t rest) {
  if (J0 == J1 && J0 >= 4 && J0 <= 7) return J1 | 1;   // fixed in the kernels
  auto ctas = [&](int pitch) {   // 1 KB of each CTA's share is the system's
    return (size_t)(228 * 1024) / (rest + Staged2d::coefs(J0, pitch) * sizeof(float2) + 1024);
  };
  return std::min<size_t>(4, ctas(J1 | 1)) < std::min<size_t>(4, ctas(J1)) ? J1 : J1 | 1;
}

template <int JF>
__device__ __forceinline__ void stage_points2d(const Staged2d& S, const Points& P, const Geom& g, const Chunk& ch,
                                               const Tile2d T) {
  constexpr int cap = kChunkPoints[2];
  const int J0 = JF > 0 ? JF : g.J[0], J1 = JF > 0 ? JF : g.J[1];
  const int q = threadIdx.x;
  if (q >= ch.count) return;
  const int i = ch.start + q;
  S.k[q] = P.kf[i] - T.org0;
  S.k[cap + q] = P.kf[P.M + i] - T.org1;
  const float2* c0 = P.coef + P.coef_off[0] + i;
  const float2* c1 = P.coef + P.coef_off[1] + i;
#pragma unroll
  for (int r = 0; r < (JF > 0 ? JF : kMaxJ); ++r) {
    if (JF == 0 && r >= J0) break;
    S.c0[r * cap + q] = c0[r * P.M];
  }
#pragma unroll
  for (int r = 0; r < (JF > 0 ? JF : kMaxJ); ++r) {
    if (JF == 0 && r >= J1) break;
    S.c1[q * S.pitch1 + r] = c1[r * P.M];
  }
}

// The chunk's padded tile of the grid into planes of real and imaginary parts, one
// row per warp step, the loads of kRows rows in flight at a time (one at a time the
// rows of a tile that is not 16 wide are a chain of round trips: 300 points on a
// 360 x 288 grid 2.97 us, 2.33 us so).  The loops are not unrolled: that costs 14
// registers and two of six CTAs per SM (800,000 points on 1000^2 51 us against 41).
template <int PF>
__device__ __forceinline__ void stage_tile2d(const float2* __restrict__ grid, const Geom& g, const Tile2d T, float* gre,
                                             float* gim) {
  const int P0 = PF > 0 ? PF : g.P[0], P1 = PF > 0 ? PF : g.P[1];
  const int lane = threadIdx.x & 31;
  constexpr int kWarps = kChunkPoints[2] / 32;
  constexpr int kRows = 3;   // 16 + J - 1 <= 24 rows in one step for J <= 9
#pragma unroll 1
  for (int r1 = lane; r1 < P1; r1 += 32) {
    const float2* src = grid + wrapk(T.org1 + r1, g.K[1]);
#pragma unroll 1
    for (int rb = threadIdx.x >> 5; rb < P0; rb += kRows * kWarps) {
      float2 v[kRows];
#pragma unroll
      for (int u = 0; u < kRows; ++u) {
        const int r0 = rb + u * kWarps;
        if (r0 < P0) v[u] = __ldg(&src[wrapk(T.org0 + r0, g.K[0]) * (int)g.Kstride[0]]);
      }
#pragma unroll
      for (int u = 0; u < kRows; ++u) {
        const int r0 = rb + u * kWarps;
        if (r0 < P0) {
          gre[r0 * P1 + r1] = v[u].x;
          gim[r0 * P1 + r1] = v[u].y;
        }
      }
    }
  }
}

// Samples of the chunk's points from the staged tile: store(q, value) in the first
// lane of each point.  Lane layout, arithmetic and summation order of k_interp.
template <int JF, int PF, class Store>
__device__ __forceinline__ void gather_staged2d(const Staged2d& S, const Chunk& ch, const Geom& g, const float* gre,
                                                const float* gim, Store store) {
  constexpr int cap = kChunkPoints[2];
  const int J0 = JF > 0 ? JF : g.J[0], G = JF > 0 ? JF : g.J[1];
  const int P1 = PF > 0 ? PF : g.P[1];
  const int PW = 32 / G;
  const int lane = threadIdx.x & 31;
  const int sub = lane / G;
  const int l = lane - sub * G;
  // warp-uniform rounds of PW points (the lane-group sum is a full-warp shuffle)
  for (int qb = (threadIdx.x >> 5) * PW; qb < ch.count; qb += cap / 32 * PW) {
    const int q = qb + sub;
    const bool act = (sub < PW) && (q < ch.count);
    float2 part = make_float2(0.f, 0.f);
    if (act) {
      const int base = S.k[q] * P1 + S.k[cap + q] + l;
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll
      for (int j0 = 0; j0 < (JF > 0 ? JF : kMaxJ); ++j0) {
        if (JF == 0 && j0 >= J0) break;
        acc = cfma(S.c0[j0 * cap + q], make_float2(gre[base + j0 * P1], gim[base + j0 * P1]), acc);
      }
      part = cmul(S.c1[q * S.pitch1 + l], acc);
    }
    const float2 tot = lane_group_sum<JF>(part, sub * G, G);
    if (act && l == 0) store(q, tot);
  }
}

template <int JF, int TF>
__global__ void __launch_bounds__(256, 4)
k_interp_chunk2d(const float2* __restrict__ grid, float2* __restrict__ y, const Chunk* __restrict__ chunks,
                 const Points P, const Geom g, const int pitch) {
  constexpr int cap = kChunkPoints[2];
  static_assert(cap == 256, "one thread per staged point");
  constexpr int PF = TF > 0 ? TF + JF - 1 : 0;
  extern __shared__ float tile[];
  const int ncell = PF > 0 ? PF * PF : (int)g.padded_cells;
  const int J0 = JF > 0 ? JF : g.J[0];
  Staged2d S;
  S.c0 = reinterpret_cast<float2*>(tile + 2 * ncell);   // 8-byte aligned: 2 * ncell floats
  S.c1 = S.c0 + J0 * cap;
  S.pitch1 = JF > 0 ? JF | 1 : pitch;
  S.k = reinterpret_cast<int*>(S.c1 + S.pitch1 * cap);
  int* s_p = S.k + 2 * cap;
  const Chunk ch = chunks[blockIdx.x];
  const Tile2d T = tile_origin2d(g, ch.bin);
  stage_points2d<JF>(S, P, g, ch, T);
  if (threadIdx.x < ch.count) s_p[threadIdx.x] = P.perm[ch.start + threadIdx.x];
  stage_tile2d<PF>(grid, g, T, tile, tile + ncell);
  __syncthreads();
  gather_staged2d<JF, PF>(S, ch, g, tile, tile + ncell, [&](int q, float2 v) { y[s_p[q]] = v; });
}

// ---------------------------------------------------------------- gridding, per chunk
// Deterministic accumulation.  The points of a chunk add into a shared copy
// of the padded tile in fixed point: every contribution is scaled by a power
// of two S chosen per chunk (and batch element), rounded to an integer and
// added with a 32-bit integer atomic.  Integer addition is exact and
// associative, so the padded tile does not depend on the order in which the
// warps' atomics land, and two runs give bit-identical grids.  S comes from
// a bound on every cell's sum of magnitudes,
//   B = cbound * sum over the chunk's points of (|Re y| + |Im y|),
// cbound = prod_d max |c_d| (a point adds to a cell at most once), taken in a
// fixed order, so S is the same on every run too:
//   1D, 2D (chunks of <= 1024, <= 256 points): one int32 word per component,
//     sums below 2^30 (S = 2^(30 - E), B < 2^E); a contribution's rounding
//     error is at most 2^-31 B;
//   3D (chunks of <= 2048 points): 2^34 of range in three words per cell: the
//     part above 2^20 of both components packed as two 16-bit fields of one
//     word (|sum| <= 2^14 + 1024 each), and the remainders below 2^20 in one
//     word each (|sum| <= 2048 * 2^19); rounding error at most 2^-35 B.
//   3D chunks whose points are spread out use two words instead: the plan keeps
//     W = the largest sum of weight magnitudes over the cells of the chunk's
//     tile (k_chunk_wmax), so a cell's sum is also below B2 = W max|y|, and one
//     int32 word per component holds 2^31 of range (S = 2^(31 - E2),
//     B2 (1 + 2^-9) < 2^E2; the roundings of <= 2048 contributions fit in the
//     margin).  A chunk does so only where its rounding step 2^(E2 - 31) is no
//     larger than the three words' 2^(E - 34), so no result loses precision.
//     A kooshball's outer tiles have B / B2 of 30 to 150 (a few points per
//     cell, hundreds per tile); only its centre and its nearly empty tiles
//     keep three words.  Two words cost two atomics and two conversions per
//     tap where three cost three atomics and the split (about 20 instructions
//     per tap): see k_gridding_chunk.
// A chunk whose bound is not finite (an Inf or NaN sample) writes NaN.
template <int D>
struct Fix {
  static constexpr int kBits = D == 3 ? 34 : 30;   // range of a cell's sum, log2
  static constexpr int kWords = D == 3 ? 3 : 2;    // int32 words per cell
};

// Sum of v over the CTA in a fixed order (shuffle tree, then warps in order);
// every thread gets the sum.  red: 32 floats of shared scratch.
__device__ __forceinline__ float block_sum_fixed(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int nw = blockDim.x >> 5;
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float t = 0.f;
  for (int w = 0; w < nw; ++w) t += red[w];
  __syncthreads();   // red free for reuse
  return t;
}

// Largest v over the CTA (v >= 0; a NaN or Inf shows in the sum taken beside
// it); every thread gets it.  red: 32 floats of shared scratch.
__device__ __forceinline__ float block_max(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int nw = blockDim.x >> 5;
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float t = 0.f;
  for (int w = 0; w < nw; ++w) t = fmaxf(t, red[w]);
  __syncthreads();   // red free for reuse
  return t;
}

struct ChunkScale {
  float S, inv;   // power-of-two scale and its inverse
  bool finite;
  bool two;       // 3D: two words per cell
};

template <int D>
__device__ __forceinline__ ChunkScale chunk_scale(float ysum, const uint32_t* cmax) {
  float cb = 1.f;
#pragma unroll
  for (int a = 0; a < D; ++a) cb *= __uint_as_float(__ldg(&cmax[a]));
  const float B = ysum * cb;
  ChunkScale cs;
  cs.finite = isfinite(B);
  int E = 0;
  frexpf(cs.finite ? B : 0.f, &E);                   // B < 2^E
  E = max(E, Fix<D>::kBits - 126);                   // keep S and 1/S normal floats
  cs.S = ldexpf(1.f, Fix<D>::kBits - E);
  cs.inv = ldexpf(1.f, E - Fix<D>::kBits);
  cs.two = false;
  return cs;
}

// 3D: two words where W max|y| (wmax of the chunk, ymax of its samples) gives
// a rounding step no larger than the three words' (see above).
__device__ __forceinline__ void try_two_words(ChunkScale& cs, float wmax, float ymax, const uint32_t* cmax) {
  const float B2 = wmax * ymax * (1.f + 0x1p-9f);
  if (!cs.finite || !isfinite(B2)) return;
  float cb = ymax * (1.f + 0x1p-9f);   // one contribution stays below 2^30 (round_int)
#pragma unroll
  for (int a = 0; a < 3; ++a) cb *= __uint_as_float(__ldg(&cmax[a]));
  int E1 = 0, E2 = 0;
  frexpf(cb, &E1);
  frexpf(B2, &E2);
  E2 = max(max(E2, E1 + 1), 31 - 126);
  const float inv2 = ldexpf(1.f, E2 - 31);
  if (inv2 > cs.inv) return;
  cs.S = ldexpf(1.f, 31 - E2);
  cs.inv = inv2;
  cs.two = true;
}

// Add one contribution w (already scaled by S) to cell `cell`.
//   two words: acc[0][cell] += rn(Re w), acc[1][cell] += rn(Im w)
//   three: packed high parts in acc[0], remainders in acc[1], acc[2]
template <int WORDS>
__device__ __forceinline__ void fix_add(int* acc, int ncell, int cell, float2 w) {
  if (WORDS == 2) {
    atomicAdd(&acc[cell], __float2int_rn(w.x));
    atomicAdd(&acc[ncell + cell], __float2int_rn(w.y));
  } else {
    // x + 1.5 * 2^23 rounds x to an integer when |x| < 2^22, and the float's
    // bits minus those of 1.5 * 2^23 are that integer (the high parts); the
    // exact remainders are rounded by the conversion unit (the same
    // round-to-nearest-even), one instruction each on an otherwise idle pipe.
    const float magic = 12582912.0f;
    const float hr = fmaf(w.x, 0x1p-20f, magic), hi_ = fmaf(w.y, 0x1p-20f, magic);
    const float lr = fmaf(-(hr - magic), 0x1p20f, w.x);   // remainder (exact)
    const float li = fmaf(-(hi_ - magic), 0x1p20f, w.y);
    const int hre = __float_as_int(hr) - 0x4B400000, him = __float_as_int(hi_) - 0x4B400000;
    atomicAdd(&acc[cell], him * 65536 + hre);
    atomicAdd(&acc[ncell + cell], __float2int_rn(lr));
    atomicAdd(&acc[2 * ncell + cell], __float2int_rn(li));
  }
}

// Value of cell c of the fixed-point tile, unscaled.
template <int D>
__device__ __forceinline__ float2 fix_value(const int* acc, int ncell, int c, const ChunkScale& cs) {
  if (!cs.finite) return make_float2(__int_as_float(0x7fffffff), __int_as_float(0x7fffffff));
  if (D < 3 || cs.two) return make_float2((float)acc[c] * cs.inv, (float)acc[ncell + c] * cs.inv);
  const int w = acc[c];
  const int hre = (int)(short)(w & 0xffff);   // low field, sign-extended
  const int him = (w - hre) / 65536;
  const long long re = (long long)hre * 1048576 + acc[ncell + c];
  const long long im = (long long)him * 1048576 + acc[2 * ncell + c];
  return make_float2((float)re * cs.inv, (float)im * cs.inv);
}

// The accumulator words are held as planes (word k of every cell, then word
// k + 1, ...) so that the J_last lanes of a point hit J_last consecutive banks
// per atomic.
template <int D>
struct GridChunkCfg {
  static constexpr int kThreads = D == 3 ? 512 : 256;
  static constexpr int kMinBlocks = D == 3 ? 2 : 4;
};

// Scatter of one chunk's points into the fixed-point tile (WORDS words per
// cell).  Consecutive points of the chunk share a warp instruction: the plan
// orders each chunk so that every aligned group of per_warp points covers
// disjoint shared-memory bank windows (see the bank-order kernel in plan.cu).
// TF > 0: every tile edge is TF and every J is JF, so the padded-tile pitches
// are compile-time constants and the neighbour loops unroll into fixed
// shared-memory offsets.
template <int D, int JF, int TF, int WORDS>
__device__ __forceinline__ void scatter_chunk(int* acc, const int ncell, const float2* __restrict__ y, const Chunk& ch,
                                              const Points& P, const Geom& g, const int (&org)[kMaxDim], const float S) {
  constexpr int PF = TF > 0 ? TF + JF - 1 : 0;   // padded edge when fixed
  const int G = JF > 0 ? JF : g.J[D - 1];
  const int lane = threadIdx.x & 31;
  const int per_warp = 32 / G;
  const int sub = lane / G;
  const int l = lane - sub * G;
  const int warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  const int P1 = D > 1 ? (TF > 0 ? PF : g.P[1]) : 1;
  const int P2 = D > 2 ? (TF > 0 ? PF : g.P[2]) : 1;
  if (sub >= per_warp) return;
  const int stepq = nwarps * per_warp;
  int q = warp * per_warp + sub;
  // 1D: the dependent load (sample through the permutation) runs one point
  // ahead; 3D has enough work per point to hide it and no registers to spare.
  float2 y_next = make_float2(0.f, 0.f);
  if (D < 3 && q < ch.count) y_next = __ldg(&y[P.perm[(int64_t)ch.start + q]]);
  for (; q < ch.count; q += stepq) {
    const int64_t i = (int64_t)ch.start + q;
    float2 yv;
    if (D < 3) {
      yv = y_next;
      if (q + stepq < ch.count) y_next = __ldg(&y[P.perm[i + stepq]]);
    } else {
      yv = __ldg(&y[P.perm[i]]);
    }
    yv = cscale(yv, S);
    const int ll = P.kf[(int64_t)(D - 1) * P.M + i] - org[D - 1] + l;
    const float2 cl = P.coef[P.coef_off[D - 1] + (int64_t)l * P.M + i];
    const float2 yl = cmulc(cl, yv);  // conj(c_last) * y
    if constexpr (D == 1) {
      fix_add<WORDS>(acc, ncell, ll, yl);
    } else {
      const int l0 = P.kf[i] - org[0];
      const int l1 = P.kf[P.M + i] - org[1];
      const int J0 = JF > 0 ? JF : g.J[0];
      const int J1 = JF > 0 ? JF : g.J[1];
      float2 c1v[JF > 0 ? JF : kMaxJ];
#pragma unroll
      for (int j1 = 0; j1 < (JF > 0 ? JF : kMaxJ); ++j1) {
        if (JF == 0 && j1 >= J1) break;
        c1v[j1] = P.coef[P.coef_off[1] + (int64_t)j1 * P.M + i];
      }
      constexpr int kU0 = TF > 0 ? JF : 1;
#pragma unroll kU0
      for (int j0 = 0; j0 < J0; ++j0) {
        const float2 c0 = P.coef[P.coef_off[0] + (int64_t)j0 * P.M + i];
        const float2 w0 = cmulc(c0, yl);
        const int rowbase = ((l0 + j0) * P1 + l1) * P2 + ll;
#pragma unroll
        for (int j1 = 0; j1 < (JF > 0 ? JF : kMaxJ); ++j1) {
          if (JF == 0 && j1 >= J1) break;
          fix_add<WORDS>(acc, ncell, rowbase + j1 * P2, cmulc(c1v[j1], w0));
        }
      }
    }
  }
}

// rn(x) as an integer for |x| < 1.2e9 on the FP32 and integer pipes: three
// additions and a shift-add, against one F2I, which the conversion unit issues
// at one warp per two cycles and SM.  t holds x rounded to a multiple of 512
// (its ulp), l the remainder plus 1.5 * 2^23, exactly rounded, and the mantissa
// of kT is chosen so that the constant bits of 512 t + l cancel modulo 2^32:
// 512 * 0x5a6000 + 0x4b400000 = 2^32.
__device__ __forceinline__ int round_int(float x) {
  const float kT = __int_as_float(0x4f800000 + 0x5a6000 );   // 2^32 (1 + 0x5a6000 / 2^23): ulp 512
  const float t = __fadd_rn(x, kT);
  const float u = __fsub_rn(t, __fadd_rn(kT, 12582912.0f));   // multiple of 512, less 1.5 * 2^23: exact
  const float l = __fsub_rn(x, u);
  return (__float_as_int(t) << 9) + __float_as_int(l);
}

// 3D chunk pass with every J = JF (4 to 7): as k_gridding_chunk, but a chunk
// that sums in two words keeps its samples in shared memory (they are gathered
// once, for the scale; the third word's space holds them), and every warp keeps
// the next round's coefficients in flight while it scatters this one's: lane l
// of a point loads the l-th coefficient of each axis into registers a round
// ahead, and the axis-0 and axis-1 ones are passed to the point's other lanes
// through a per-warp strip of shared memory.  A chunk that needs three words
// takes scatter_chunk.  128^3 kooshball: 517 us with three words throughout, 324 us
// so, with the shared-memory pipe 78 % and the issue slots 66 % busy.
template <int JF, int TF>
__device__ __forceinline__ void scatter_chunk3d(int* acc, const int ncell, const float2* s_y, float2* strip,
                                                const Chunk& ch, const Points& P, const Geom& g,
                                                const int (&org)[kMaxDim], const float S) {
  constexpr int PF = TF > 0 ? TF + JF - 1 : 0;
  constexpr int PW = Chunk3dCfg<JF>::kPerWarp;
  const int P1 = TF > 0 ? PF : g.P[1];
  const int P2 = TF > 0 ? PF : g.P[2];
  const int lane = threadIdx.x & 31;
  const int sub = lane / JF;
  const int l = lane - sub * JF;
  const int step = (Chunk3dCfg<JF>::kThreads / 32) * PW;
  const int64_t M = P.M;
  const float2* pc0 = P.coef + P.coef_off[0] + (int64_t)l * M + ch.start;
  const float2* pc1 = P.coef + P.coef_off[1] + (int64_t)l * M + ch.start;
  const float2* pc2 = P.coef + P.coef_off[2] + (int64_t)l * M + ch.start;
  const int32_t* pk = P.kf + ch.start;
  int qb = (threadIdx.x >> 5) * PW;
  bool act = sub < PW && qb + sub < ch.count;
  float2 n0 = make_float2(0.f, 0.f), n1 = n0, n2 = n0;
  int k0 = 0, k1 = 0, k2 = 0;
  if (act) {
    const int q = qb + sub;
    n0 = pc0[q]; n1 = pc1[q]; n2 = pc2[q];
    k0 = pk[q]; k1 = pk[M + q]; k2 = pk[2 * M + q];
  }
  for (; qb < ch.count; qb += step) {   // warp-uniform
    const bool cur = act;
    __syncwarp();   // the strip's readers of the previous round are done
    float2 yl = make_float2(0.f, 0.f);
    int base = 0;
    if (cur) {
      strip[l * PW + sub] = n0;
      strip[(JF + l) * PW + sub] = n1;
      yl = cmulc(n2, cscale(s_y[qb + sub], S));   // conj(c_last) * y
      base = ((k0 - org[0]) * P1 + k1 - org[1]) * P2 + k2 - org[2] + l;
    }
    const int qn = qb + step + sub;
    act = sub < PW && qn < ch.count;
    if (act) {
      n0 = pc0[qn]; n1 = pc1[qn]; n2 = pc2[qn];
      k0 = pk[qn]; k1 = pk[M + qn]; k2 = pk[2 * M + qn];
    }
    __syncwarp();
    if (cur) {
      float2 c1v[JF];
#pragma unroll
      for (int j1 = 0; j1 < JF; ++j1) c1v[j1] = strip[(JF + j1) * PW + sub];
#pragma unroll
      for (int j0 = 0; j0 < JF; ++j0) {
        const float2 w0 = cmulc(strip[j0 * PW + sub], yl);
        int* row = acc + base + j0 * P1 * P2;
#pragma unroll
        for (int j1 = 0; j1 < JF; ++j1) {
          const float2 w = cmulc(c1v[j1], w0);
          int* cell = row + j1 * P2;
          // the conversion unit takes the real parts and half of the imaginary
          // ones, the FP32 pipe the rest
          atomicAdd(cell, __float2int_rn(w.x));
          atomicAdd(cell + ncell, (j1 & 1) ? round_int(w.y) : __float2int_rn(w.y));
        }
      }
    }
  }
}

template <int JF, int TF>
__global__ void __launch_bounds__(Chunk3dCfg<JF>::kThreads, 2)
k_gridding_chunk3d(const float2* __restrict__ y_b, float2* __restrict__ tiles_b, const Chunk* __restrict__ chunks,
                   const Points P, const Geom g, int64_t ybs, int64_t tbs) {
  constexpr int PF = TF > 0 ? TF + JF - 1 : 0;
  extern __shared__ int acc[];
  __shared__ float red[32];
  const float2* __restrict__ y = y_b + (int64_t)blockIdx.y * ybs;
  float2* __restrict__ out = tiles_b + (int64_t)blockIdx.y * tbs;
  const int ncell = TF > 0 ? PF * PF * PF : (int)g.padded_cells;
  float2* s_y = reinterpret_cast<float2*>(acc + 2 * ncell);   // 8-byte aligned: 2 * ncell words
  float2* strip = s_y + kChunkPoints[3] + (threadIdx.x >> 5) * Chunk3dCfg<JF>::kStrip;
  const Chunk ch = chunks[blockIdx.x];
  out += (int64_t)ch.slot * g.padded_cells;
  float part = 0.f, ymax = 0.f;
  for (int q = threadIdx.x; q < ch.count; q += blockDim.x) {
    const float2 v = __ldg(&y[P.perm[(int64_t)ch.start + q]]);
    s_y[q] = v;
    const float a = fabsf(v.x), b = fabsf(v.y);
    part += a + b;
    // |v| <= sqrt 2 max(a, b) and <= a + b; either bounds the contributions
    ymax = fmaxf(ymax, fminf(a + b, 1.41421368f * fmaxf(a, b)));
  }
  for (int c = threadIdx.x; c < 2 * ncell; c += blockDim.x) acc[c] = 0;
  // the sums also order the zeroing and s_y before their use
  ChunkScale cs = chunk_scale<3>(block_sum_fixed(part, red), P.cmax);
  try_two_words(cs, __int_as_float(ch.wmax), block_max(ymax, red), P.cmax);
  int org[kMaxDim];
  {
    int rem = ch.bin;
    for (int a = 2; a >= 0; --a) {
      org[a] = (rem % g.nb[a]) * g.T[a];
      rem /= g.nb[a];
    }
  }
  if (cs.two) {   // CTA-uniform
    scatter_chunk3d<JF, TF>(acc, ncell, s_y, strip, ch, P, g, org, cs.S);
  } else if (cs.finite) {
    for (int c = threadIdx.x; c < ncell; c += blockDim.x) acc[2 * ncell + c] = 0;   // over the samples
    __syncthreads();
    scatter_chunk<3, JF, TF, 3>(acc, ncell, y, ch, P, g, org, cs.S);
  }
  __syncthreads();
  for (int c = threadIdx.x; c < ncell; c += blockDim.x) out[c] = fix_value<3>(acc, ncell, c, cs);
}

// 1D chunk pass, and the 3D one for the J that k_gridding_chunk3d does not take
// (2D: k_gridding_chunk_staged).
template <int D, int JF>
__global__ void __launch_bounds__(GridChunkCfg<D>::kThreads, GridChunkCfg<D>::kMinBlocks)
k_gridding_chunk(const float2* __restrict__ y_b, float2* __restrict__ tiles_b, const Chunk* __restrict__ chunks,
                 const Points P, const Geom g, int64_t ybs, int64_t tbs) {
  static_assert(D != 2, "2D has its own kernel");
  extern __shared__ int acc[];
  __shared__ float red[32];
  const float2* __restrict__ y = y_b + (int64_t)blockIdx.y * ybs;
  float2* __restrict__ tiles = tiles_b + (int64_t)blockIdx.y * tbs;
  const int ncell = (int)g.padded_cells;
  const Chunk ch = chunks[blockIdx.x];
  for (int c = threadIdx.x; c < Fix<D>::kWords * ncell; c += blockDim.x) acc[c] = 0;

  // the chunk's scale (the sums also order the zeroing above before the atomics)
  float part = 0.f, ymax = 0.f;
  for (int q = threadIdx.x; q < ch.count; q += blockDim.x) {
    const float2 v = __ldg(&y[P.perm[(int64_t)ch.start + q]]);
    const float a = fabsf(v.x), b = fabsf(v.y);
    part += a + b;
    // |v| <= sqrt 2 max(a, b) and <= a + b; either bounds the contributions
    if (D == 3) ymax = fmaxf(ymax, fminf(a + b, 1.41421368f * fmaxf(a, b)));
  }
  ChunkScale cs = chunk_scale<D>(block_sum_fixed(part, red), P.cmax);
  if (D == 3) try_two_words(cs, __int_as_float(ch.wmax), block_max(ymax, red), P.cmax);

  // tile origin of this chunk's bin
  int org[kMaxDim];
  {
    int rem = ch.bin;
    for (int a = D - 1; a >= 0; --a) {
      org[a] = (rem % g.nb[a]) * g.T[a];
      rem /= g.nb[a];
    }
  }
  if (cs.finite) {   // CTA-uniform
    if (D < 3 || cs.two) scatter_chunk<D, JF, 0, 2>(acc, ncell, y, ch, P, g, org, cs.S);
    else scatter_chunk<D, JF, 0, 3>(acc, ncell, y, ch, P, g, org, cs.S);
  }
  __syncthreads();
  float2* out = tiles + (int64_t)ch.slot * g.padded_cells;
  for (int c = threadIdx.x; c < ncell; c += blockDim.x) out[c] = fix_value<D>(acc, ncell, c, cs);
}

// ---------------------------------------------------------------- gridding, tile reduction
// 1D and 2D (3D: k_gridding_reduce3d; 2D batches: k_gridding_reduce2d).
// One CTA per tile: grid cell c of tile b is the sum over e in {0,1}^d of the
// padded tiles of bin b - e (wrapped per dimension) at local position
// c - origin(b) + e * T, when that position lies inside the padded tile.  Each
// thread owns CPT cells of the tile; their padded-tile offset and the mask of
// neighbours e that reach them are computed once, so every (e, chunk) pair
// costs one predicated load per cell.  The sum runs over e, then over the
// source bin's chunks, in a fixed order.
// The whole CTA reduces grid tile `bin`; `part` is shared scratch of
// blockDim.x * CPT values.
// Entry n (2^D bits at bit 2^D * n) is the set of the e in [0, 2^D) with
// e & ~n == 0: the neighbours whose padded tiles reach a cell that is near the
// low edge of its tile along the axes in n.
template <int D>
__host__ __device__ constexpr uint64_t subset_masks() {
  uint64_t t = 0;
  for (unsigned n = 0; n < (1u << D); ++n)
    for (unsigned e = 0; e < (1u << D); ++e)
      if ((e & ~n) == 0) t |= uint64_t(1) << ((1u << D) * n + e);
  return t;
}

// Per-cell set-up of a tile reduction: the thread's CPT cells are
// tg + k * gsize of tile bc (coordinates in tiles); loc0 is a cell's
// offset in a padded tile, emask the neighbours e whose padded tiles reach it
// (0 beyond cend), goff its grid offset.
template <int D, int CPT, int TF>
__device__ __forceinline__ void reduce_cells(const Geom& g, const int (&bc)[kMaxDim], int tg, int gsize,
                                             int tile_cells, int cend, int (&loc0)[CPT], unsigned (&emask)[CPT],
                                             int (&goff)[CPT]) {
  static_assert(D < 3, "3D has its own kernel");
  const int P1 = D > 1 ? g.P[1] : 1;
  // TF > 0: every tile edge is TF, so the cell decompositions below divide by constants
  const int T1 = D > 1 ? (TF > 0 ? TF : g.T[1]) : 1;
#pragma unroll
  for (int k = 0; k < CPT; ++k) {
    const int c = min(tg + k * gsize, tile_cells - 1);
    const int lc[2] = {c / T1, c % T1};   // 1D: T1 = 1
    loc0[k] = lc[0] * P1 + lc[1];
    // neighbour e reaches the cell iff every axis a with e_a = 1 has the cell
    // within J - 1 of the tile's low edge; with those axes as the bits of
    // `near` (e's bit order), the mask is the set of subsets of near
    unsigned near = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) near |= (lc[a] + g.T[a] < g.P[a] ? 1u : 0u) << (D - 1 - a);
    const unsigned m = (unsigned)(subset_masks<D>() >> ((1 << D) * near)) & ((1u << (1 << D)) - 1u);
    emask[k] = (tg + k * gsize < cend) ? m : 0u;
    int off = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) off += (bc[a] * g.T[a] + lc[a]) * (int)g.Kstride[a];
    goff[k] = off;
  }
}

template <int D, int CPT, int TF>
__device__ __forceinline__ void reduce_tile(const float2* __restrict__ tiles, const int32_t* __restrict__ bin_chunk,
                                            float2* __restrict__ grid, const Geom& g, const int NG, const int bin,
                                            float2* part) {
  // NG thread groups of blockDim/NG threads; group h takes every NG-th (e, chunk)
  // pair, and the groups' sums are added in group order at the end.
  __shared__ int s_q0[1 << kMaxDim], s_q1[1 << kMaxDim], s_delta[1 << kMaxDim];
  int bc[kMaxDim];
  {
    int rem = bin;
#pragma unroll
    for (int a = D - 1; a >= 0; --a) {
      bc[a] = rem % g.nb[a];
      rem /= g.nb[a];
    }
  }
  if (threadIdx.x < (1 << D)) {
    const int e = threadIdx.x;
    int src = 0, delta = 0;
    for (int a = 0; a < D; ++a) {
      const int ea = (e >> (D - 1 - a)) & 1;
      src = src * g.nb[a] + (bc[a] - ea + g.nb[a]) % g.nb[a];
      const int pstride = a == D - 1 ? 1 : g.P[D - 1];
      delta += ea * g.T[a] * pstride;
    }
    s_q0[e] = bin_chunk[src];
    s_q1[e] = bin_chunk[src + 1];
    s_delta[e] = delta;
  }
  __syncthreads();
  int loc0[CPT];
  unsigned emask[CPT];
  int goff[CPT];
  float2 acc[CPT];
  int tile_cells = 1;
  for (int a = 0; a < D; ++a) tile_cells *= TF > 0 ? TF : g.T[a];
  const int gsize = blockDim.x / NG;
  const int h = threadIdx.x / gsize;
  const int tg = threadIdx.x - h * gsize;
  // A tile with few (neighbour, chunk) pairs is summed by group 0 alone; the
  // other groups then skip their set-up (CTA-uniform decision).
  int npairs = 0;
  for (int e = 0; e < (1 << D); ++e) npairs += s_q1[e] - s_q0[e];
  const int NGe = npairs > 2 * (1 << D) ? NG : 1;
  const bool active = h < NGe;
  const int cend = min(tile_cells, gsize * CPT);
#pragma unroll
  for (int k = 0; k < CPT; ++k) acc[k] = make_float2(0.f, 0.f);
  reduce_cells<D, CPT, TF>(g, bc, tg, gsize, tile_cells, cend, loc0, emask, goff);
  const int64_t pc = g.padded_cells;
  if (active) {
    int idx = 0;  // running index over the (e, chunk) pairs
#pragma unroll
    for (int e = 0; e < (1 << D); ++e) {
      const int q0 = s_q0[e], q1 = s_q1[e];
      const int delta = s_delta[e];
      // first pair of this e that belongs to group h
      int q = q0 + ((h - idx) % NGe + NGe) % NGe;
      // DEPTH pairs per step: all their loads are in flight before the adds,
      // which keep the pair order (acc + v(q) + v(q + NGe) + ...).  1D has one tile
      // and a chain of M / 1024 chunks: 200,000 points on 64 cells 20.1 us with two
      // pairs in flight, 13.4 with three, 16.3 with four (1024 cells: 30, 28, 33).
      constexpr int DEPTH = D == 1 ? 3 : 2;
      for (; q + (DEPTH - 1) * NGe < q1; q += DEPTH * NGe) {
        float2 v[DEPTH][CPT];
#pragma unroll
        for (int u = 0; u < DEPTH; ++u) {
          const float2* src = tiles + (int64_t)(q + u * NGe) * pc + delta;
#pragma unroll
          for (int k = 0; k < CPT; ++k) {
            const bool on = (emask[k] >> e) & 1u;
            v[u][k] = on ? __ldg(&src[loc0[k]]) : make_float2(0.f, 0.f);
          }
        }
#pragma unroll
        for (int k = 0; k < CPT; ++k)
          if ((emask[k] >> e) & 1u) {
#pragma unroll
            for (int u = 0; u < DEPTH; ++u) acc[k] = cadd(acc[k], v[u][k]);
          }
      }
      for (; q < q1; q += NGe) {
        const float2* src = tiles + (int64_t)q * pc + delta;
#pragma unroll
        for (int k = 0; k < CPT; ++k)
          if ((emask[k] >> e) & 1u) acc[k] = cadd(acc[k], __ldg(&src[loc0[k]]));
      }
      idx += q1 - q0;
    }
  }
  if (NGe > 1) {
#pragma unroll
    for (int k = 0; k < CPT; ++k) part[h * (CPT * gsize) + k * gsize + tg] = acc[k];
    __syncthreads();
    if (h == 0) {
#pragma unroll
      for (int k = 0; k < CPT; ++k) {
        float2 t = part[k * gsize + tg];
        for (int hh = 1; hh < NGe; ++hh) t = cadd(t, part[hh * (CPT * gsize) + k * gsize + tg]);
        acc[k] = t;
      }
    }
  }
  if (h == 0) {
#pragma unroll
    for (int k = 0; k < CPT; ++k)
      if (tg + k * gsize < cend) grid[goff[k]] = acc[k];
  }
  __syncthreads();   // shared scratch free for the caller
}

// CTA x reduces tile x.
template <int D, int CPT, int TF>
__global__ void __launch_bounds__(1024)
k_gridding_reduce(const float2* __restrict__ tiles_b, const int32_t* __restrict__ bin_chunk,
                  float2* __restrict__ grid_b, const Geom g, const int NG, int64_t tbs, int64_t gbs) {
  extern __shared__ float2 part[];
  reduce_tile<D, CPT, TF>(tiles_b + (int64_t)blockIdx.y * tbs, bin_chunk, grid_b + (int64_t)blockIdx.y * gbs, g,
                          NG, blockIdx.x, part);
}


// One thread group (tg = 0 .. gsize - 1, no barriers) reduces 2D grid tile
// `bin` on its own, in the order of reduce_tile with a single group: neighbour
// e outer, the source bin's chunks in order, so the tile's cells are the same
// bit for bit.  Each thread fetches the four source bins' chunk ranges itself.
template <int CPT, int TF>
__device__ __forceinline__ void reduce_tile_group2d(const float2* __restrict__ tiles,
                                                    const int32_t* __restrict__ bin_chunk, float2* __restrict__ grid,
                                                    const Geom& g, const int bin, const int tg, const int gsize) {
  int bc[kMaxDim] = {bin / g.nb[1], bin % g.nb[1], 0};
  int q0[4], q1[4], delta[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int e0 = e >> 1, e1 = e & 1;
    const int src = ((bc[0] - e0 + g.nb[0]) % g.nb[0]) * g.nb[1] + (bc[1] - e1 + g.nb[1]) % g.nb[1];
    q0[e] = __ldg(&bin_chunk[src]);
    q1[e] = __ldg(&bin_chunk[src + 1]);
    delta[e] = e0 * g.T[0] * g.P[1] + e1 * g.T[1];
  }
  const int tile_cells = TF > 0 ? TF * TF : g.T[0] * g.T[1];
  const int cend = min(tile_cells, gsize * CPT);
  int loc0[CPT];
  unsigned emask[CPT];
  int goff[CPT];
  float2 acc[CPT];
#pragma unroll
  for (int k = 0; k < CPT; ++k) acc[k] = make_float2(0.f, 0.f);
  reduce_cells<2, CPT, TF>(g, bc, tg, gsize, tile_cells, cend, loc0, emask, goff);
  const int64_t pc = g.padded_cells;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    for (int q = q0[e]; q < q1[e]; ++q) {
      const float2* src = tiles + (int64_t)q * pc + delta[e];
#pragma unroll
      for (int k = 0; k < CPT; ++k)
        if ((emask[k] >> e) & 1u) acc[k] = cadd(acc[k], __ldg(&src[loc0[k]]));
    }
  }
#pragma unroll
  for (int k = 0; k < CPT; ++k)
    if (tg + k * gsize < cend) grid[goff[k]] = acc[k];
}

// 2D tile reduction of a single transform over a plan-time work list: item
// {t, -2, -1, -1} is a dense tile (more than 8 (neighbour, chunk) pairs),
// reduced by the whole CTA as in k_gridding_reduce; any other item holds up
// to NG sparse tiles (-1 = none), one per thread group.  Sparse tiles then
// take a quarter of the CTAs they took one per CTA, with every group busy.
template <int CPT, int TF>
__global__ void __launch_bounds__(256, 3)
k_gridding_reduce_packed2d(const float2* __restrict__ tiles, const int32_t* __restrict__ bin_chunk,
                           float2* __restrict__ grid, const int4* __restrict__ work, const Geom g, const int NG) {
  extern __shared__ float2 part[];
  const int4 w = work[blockIdx.x];
  if (w.y == -2) {   // CTA-uniform
    reduce_tile<2, CPT, TF>(tiles, bin_chunk, grid, g, NG, w.x, part);
    return;
  }
  const int gsize = blockDim.x / NG;
  const int h = threadIdx.x / gsize;
  const int t = h == 0 ? w.x : (h == 1 ? w.y : (h == 2 ? w.z : w.w));
  if (t < 0) return;
  reduce_tile_group2d<CPT, TF>(tiles, bin_chunk, grid, g, t, threadIdx.x - h * gsize, gsize);
}


// 2D chunk pass with staged point data (see k_interp_chunk2d for the layout); the
// samples are staged too.  The accumulation follows the lane layout, bank order
// and fixed-point words of k_gridding_chunk; half of the imaginary parts are
// rounded on the FP32 pipe (round_int), as in scatter_chunk3d.
// FUSED (V^H V, the normal operator's grid part): y_b is the oversampled
// spectrum instead of the samples; the chunk's padded tile of it is staged in
// shared memory (two float planes after the point data), and each point's y is
// first gathered from there into shared memory, so the samples never leave the
// CTA and the coefficients are read once for both directions.
template <int JF, int TF, bool FUSED>
__global__ void __launch_bounds__(256, 4)
k_gridding_chunk_staged(const float2* __restrict__ y_b, float2* __restrict__ tiles_b,
                        const Chunk* __restrict__ chunks, const Points P, const Geom g, int64_t ybs, int64_t tbs,
                        const int pitch) {
  constexpr int cap = kChunkPoints[2];
  static_assert(cap == 256, "one thread per staged point");
  constexpr int PF = TF > 0 ? TF + JF - 1 : 0;
  extern __shared__ int acc[];
  __shared__ float red[32];
  const float2* __restrict__ y = y_b + (int64_t)blockIdx.y * ybs;
  float2* __restrict__ tiles = tiles_b + (int64_t)blockIdx.y * tbs;
  const int ncell = PF > 0 ? PF * PF : (int)g.padded_cells;
  const int P1 = PF > 0 ? PF : g.P[1];
  const int J0 = JF > 0 ? JF : g.J[0], J1 = JF > 0 ? JF : g.J[1];
  Staged2d S;
  S.c0 = reinterpret_cast<float2*>(acc + 2 * ncell);   // 8-byte aligned: 2 * ncell words
  S.c1 = S.c0 + J0 * cap;
  S.pitch1 = JF > 0 ? JF | 1 : pitch;
  float2* s_y = S.c1 + S.pitch1 * cap;
  S.k = reinterpret_cast<int*>(s_y + cap);
  const Chunk ch = chunks[blockIdx.x];
  // Loops over the cells take their number from the plan even where it is a constant:
  // unrolled they cost the chunks of a few points more than they save (1024^2 grid,
  // 40,000 points 14.5 us, 12.8 so; 512^2, 200,000 points 10.5, 10.0).
  const int cells = (int)g.padded_cells;
  auto zero = [&] {
    for (int c = threadIdx.x; c < cells; c += blockDim.x) reinterpret_cast<int2*>(acc)[c] = make_int2(0, 0);
  };
  if (!FUSED) zero();   // while the chunk's entry is on its way
  const Tile2d T = tile_origin2d(g, ch.bin);
  const int qs = threadIdx.x;   // the point this thread stages
  int pm = 0;
  if (!FUSED && qs < ch.count) pm = P.perm[ch.start + qs];
  stage_points2d<JF>(S, P, g, ch, T);
  if (FUSED) {
    float* gre = reinterpret_cast<float*>(S.k + 2 * cap);   // the chunk's padded tile of the spectrum
    stage_tile2d<PF>(y, g, T, gre, gre + ncell);
    zero();
  }
  if (!FUSED && qs < ch.count) s_y[qs] = __ldg(&y[pm]);
  __syncthreads();
  if (FUSED) {
    const float* gre = reinterpret_cast<const float*>(S.k + 2 * cap);
    gather_staged2d<JF, PF>(S, ch, g, gre, gre + ncell, [&](int q, float2 v) { s_y[q] = v; });
    __syncthreads();
  }
  // the chunk's scale (also orders the zeroing and staging before the atomics)
  float mag = 0.f;
  if (qs < ch.count) mag = fabsf(s_y[qs].x) + fabsf(s_y[qs].y);
  const ChunkScale cs = chunk_scale<2>(block_sum_fixed(mag, red), P.cmax);
  const int PW = 32 / J1;
  const int lane = threadIdx.x & 31;
  const int sub = lane / J1;
  const int l = lane - sub * J1;
  if (sub < PW && cs.finite) {
    for (int q = (threadIdx.x >> 5) * PW + sub; q < ch.count; q += cap / 32 * PW) {
      const float2 yl = cmulc(S.c1[q * S.pitch1 + l], cscale(s_y[q], cs.S));   // conj(c_last) * y * S
      int* cell = acc + S.k[q] * P1 + S.k[cap + q] + l;
#pragma unroll
      for (int j0 = 0; j0 < (JF > 0 ? JF : kMaxJ); ++j0) {
        if (JF == 0 && j0 >= J0) break;
        const float2 w = cmulc(S.c0[j0 * cap + q], yl);
        atomicAdd(cell + j0 * P1, __float2int_rn(w.x));
        atomicAdd(cell + j0 * P1 + ncell, (j0 & 1) ? round_int(w.y) : __float2int_rn(w.y));
      }
    }
  }
  __syncthreads();
  float2* out = tiles + (int64_t)ch.slot * g.padded_cells;
  for (int c = threadIdx.x; c < cells; c += blockDim.x) out[c] = fix_value<2>(acc, ncell, c, cs);
}

// ---------------------------------------------------------------- 2D chunk passes of a batch
// V and V^H of one chunk of a 2D tile for one batch element, per CTA of two
// warps.  A batch has CTAs enough, and the chunks of a dynamic series' frames are
// small (30 points), so what counts is the instructions spent per CTA: eight
// warps with staged point data (k_gridding_chunk_staged) spend most of theirs on
// set-up, barriers and idle warps.  With fewer CTAs or longer chunks latency is what
// bounds them, and staging everything at once hides it better (one transform on a
// 512^2 grid with 206,336 points: 56 us for the pair, 67 us with these).
// The lane
// layout is that of k_interp (a group of J_1 lanes per point, lane l its l-th
// neighbour along the contiguous axis); every warp loads the next round's point
// data into registers while it works on this one's (no barrier between rounds):
// lane l of a point loads c_0[l] and c_1[l], keeps c_1[l] for its own column and
// passes c_0[l] to the point's other lanes through a per-warp strip of shared
// memory.  JF > 0: J_0 = J_1 = JF; JF = 0: any J, c_0 is loaded in the round.
constexpr int kBatchWarps2d = 2;
// k_gridding_chunk2d runs below this mean chunk and above this many CTAs, batches and
// single transforms alike (one of 300,000 points on 1000^2, 30 per chunk, 31.9 us
// against 41.6 staged).  Measured, k_gridding_chunk2d against k_gridding_chunk_staged: 30 points per
// chunk, 32 coils 76 us against 95; 108 points, 16 images 55 against 46; 105
// points, 8 coils (1968 CTAs) 20 against 14.
constexpr int64_t kBatchMaxMean = 64;
constexpr int64_t kBatchMinCtas = 32 * 152;
template <int JF>
__host__ __device__ inline int strip2d(int J0, int J1) { return (JF > 0 ? JF : J0) * (32 / (JF > 0 ? JF : J1)); }

// Runs body(cur, q, base, c1) for the warp's rounds of points: cur = the lane
// has a point, q = its index in the chunk, base = the padded-tile cell of the
// lane's column in the point's first row, c1 = c_1[l]; c_0[j] of the lane's
// point is strip[j * PW + sub].
template <int JF, class Body>
__device__ __forceinline__ void for_points2d(const Chunk& ch, const Points& P, const Geom& g, const Tile2d T,
                                             float2* strip, Body body) {
  const int J0 = JF > 0 ? JF : g.J[0];
  const int G = JF > 0 ? JF : g.J[1];
  const int PW = 32 / G;
  const int lane = threadIdx.x & 31;
  const int sub = lane / G;
  const int l = lane - sub * G;
  const int step = (blockDim.x >> 5) * PW;
  const int64_t M = P.M;
  const float2* pc0 = P.coef + P.coef_off[0] + ch.start + (JF > 0 ? (int64_t)l * M : 0);
  const float2* pc1 = P.coef + P.coef_off[1] + (int64_t)l * M + ch.start;
  const int32_t* pk = P.kf + ch.start;
  int qb = (threadIdx.x >> 5) * PW;
  bool act = sub < PW && qb + sub < ch.count;
  float2 n0 = make_float2(0.f, 0.f), n1 = n0;
  int k0 = 0, k1 = 0;
  if (act) {
    const int q = qb + sub;
    if (JF > 0) n0 = pc0[q];
    n1 = pc1[q];
    k0 = pk[q];
    k1 = pk[M + q];
  }
  for (; qb < ch.count; qb += step) {   // warp-uniform
    const bool cur = act;
    const int q = qb + sub;
    const float2 c1 = n1;
    int base = 0;
    __syncwarp();   // the strip's readers of the previous round are done
    if (cur) {
      if (JF > 0) {
        strip[l * PW + sub] = n0;
      } else {
        for (int j = l; j < J0; j += G) strip[j * PW + sub] = pc0[(int64_t)j * M + q];
      }
      base = (k0 - T.org0) * g.P[1] + k1 - T.org1 + l;
    }
    const int qn = q + step;
    act = sub < PW && qn < ch.count;
    if (act) {
      if (JF > 0) n0 = pc0[qn];
      n1 = pc1[qn];
      k0 = pk[qn];
      k1 = pk[M + qn];
    }
    __syncwarp();
    body(cur, q, base, c1);
  }
}

// V^H (fixed-point accumulation as in k_gridding_chunk; the samples wait in
// shared memory after the pass that finds the scale).  Shared memory: the two
// accumulator planes, the samples, the strips.
template <int JF>
__global__ void __launch_bounds__(32 * kBatchWarps2d)
k_gridding_chunk2d(const float2* __restrict__ y_b, float2* __restrict__ tiles_b, const Chunk* __restrict__ chunks,
                   const Points P, const Geom g, int64_t ybs, int64_t tbs) {
  extern __shared__ int acc[];
  __shared__ float red[32];
  const float2* __restrict__ y = y_b + (int64_t)blockIdx.y * ybs;
  float2* __restrict__ tiles = tiles_b + (int64_t)blockIdx.y * tbs;
  const int ncell = (int)g.padded_cells;
  float2* s_y = reinterpret_cast<float2*>(acc + 2 * ncell);   // 8-byte aligned: 2 * ncell words
  float2* strip = s_y + kChunkPoints[2] + (threadIdx.x >> 5) * strip2d<JF>(g.J[0], g.J[1]);
  const Chunk ch = chunks[blockIdx.x];
  const Tile2d T = tile_origin2d(g, ch.bin);
  float mag = 0.f;
  for (int q = threadIdx.x; q < ch.count; q += blockDim.x) {
    const float2 v = __ldg(&y[P.perm[ch.start + q]]);
    s_y[q] = v;
    mag += fabsf(v.x) + fabsf(v.y);
  }
  for (int c = threadIdx.x; c < ncell; c += blockDim.x) reinterpret_cast<int2*>(acc)[c] = make_int2(0, 0);
  // the sum also orders the zeroing and s_y before their use
  const ChunkScale cs = chunk_scale<2>(block_sum_fixed(mag, red), P.cmax);
  if (cs.finite) {   // CTA-uniform
    const int J0 = JF > 0 ? JF : g.J[0];
    const int PW = 32 / (JF > 0 ? JF : g.J[1]);
    const int sub = (threadIdx.x & 31) / (JF > 0 ? JF : g.J[1]);
    const int P1 = g.P[1];
    for_points2d<JF>(ch, P, g, T, strip, [&](bool cur, int q, int base, float2 c1) {
      if (!cur) return;
      const float2 yl = cmulc(c1, cscale(s_y[q], cs.S));   // conj(c_last) * y * S
#pragma unroll
      for (int j0 = 0; j0 < (JF > 0 ? JF : kMaxJ); ++j0) {
        if (JF == 0 && j0 >= J0) break;
        const float2 w = cmulc(strip[j0 * PW + sub], yl);
        int* cell = acc + base + j0 * P1;
        atomicAdd(cell, __float2int_rn(w.x));
        atomicAdd(cell + ncell, (j0 & 1) ? round_int(w.y) : __float2int_rn(w.y));   // see scatter_chunk3d
      }
    });
  }
  __syncthreads();
  float2* out = tiles + (int64_t)ch.slot * g.padded_cells;
  for (int c = threadIdx.x; c < ncell; c += blockDim.x) out[c] = fix_value<2>(acc, ncell, c, cs);
}

// 2D, batches: thread (r1, z0) of a tile sums the cells r0 = z0 .. z0 + 7 of its
// column, as k_gridding_reduce3d below does, so a 16^2 tile takes one warp and a
// CTA several tiles.  The same sums in the same order as reduce_tile with one
// group, two partial tiles in flight: a dense tile's list is one chain.  A frame of
// 32 coils on a 512^2 grid (32 x 1024 tiles): 55 us with 64 threads and a neighbour
// mask per cell, 41 us so.  Radial, 200,000 points on a 256^2 grid (111 partial tiles
// in the centre): 2 images 22.4 -> 21.7 us (27.8 with one in flight), 8 images
// 25.2 -> 22.8; on 512^2 2, 8 and 16 images 14.1 -> 12.2, 23.7 -> 19.6, 43 -> 35.
constexpr int kRed2Rows = 8;
constexpr int kRed2Threads = 256;

__global__ void __launch_bounds__(kRed2Threads)
k_gridding_reduce2d(const float2* __restrict__ tiles_b, const int32_t* __restrict__ bin_chunk,
                    float2* __restrict__ grid_b, const Geom g, int64_t tbs, int64_t gbs, int nz) {
  const float2* __restrict__ tiles = tiles_b + (int64_t)blockIdx.y * tbs;
  float2* __restrict__ grid = grid_b + (int64_t)blockIdx.y * gbs;
  const int T0 = g.T[0], T1 = g.T[1], P1 = g.P[1];
  const int item = blockIdx.x * kRed2Threads + threadIdx.x;   // (tile, z, r1)
  const int tz = item / T1, r1 = item - tz * T1;
  const int bin = tz / nz, z0 = (tz - bin * nz) * kRed2Rows;
  if (bin >= (int)g.nbins) return;   // no barriers below
  const int b0 = bin / g.nb[1], b1 = bin - b0 * g.nb[1];
  const int nzc = min(kRed2Rows, T0 - z0);
  float2 acc[kRed2Rows];
#pragma unroll
  for (int k = 0; k < kRed2Rows; ++k) acc[k] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int e = 0; e < 4; ++e) {
    const int e0 = e >> 1, e1 = e & 1;
    const int n = e0 ? min(nzc, g.J[0] - 1 - z0) : nzc;   // the neighbour below reaches r0 < J - 1
    if (n <= 0 || (e1 && r1 >= g.J[1] - 1)) continue;
    const int s0 = e0 ? (b0 > 0 ? b0 : g.nb[0]) - 1 : b0;
    const int s1 = e1 ? (b1 > 0 ? b1 : g.nb[1]) - 1 : b1;
    const int src = s0 * g.nb[1] + s1;
    const int q1 = __ldg(&bin_chunk[src + 1]);
    int q = __ldg(&bin_chunk[src]);
    const float2* ptr = tiles + (int64_t)q * g.padded_cells + (z0 + e0 * T0) * P1 + r1 + e1 * T1;
    for (; q + 2 <= q1; q += 2, ptr += 2 * g.padded_cells) {
      float2 v[2][kRed2Rows];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int k = 0; k < kRed2Rows; ++k)
          v[u][k] = k < n ? __ldg(&ptr[u * g.padded_cells + k * P1]) : make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int k = 0; k < kRed2Rows; ++k)
          if (k < n) acc[k] = cadd(acc[k], v[u][k]);
    }
    for (; q < q1; ++q, ptr += g.padded_cells) {
      float2 v[kRed2Rows];
#pragma unroll
      for (int k = 0; k < kRed2Rows; ++k) v[k] = k < n ? __ldg(&ptr[k * P1]) : make_float2(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < kRed2Rows; ++k)
        if (k < n) acc[k] = cadd(acc[k], v[k]);
    }
  }
  float2* out = grid + ((b0 * T0 + z0) * (int)g.Kstride[0] + b1 * T1 + r1);
#pragma unroll
  for (int k = 0; k < kRed2Rows; ++k)
    if (k < nzc) out[k * (int)g.Kstride[0]] = acc[k];
}

// 3D: thread (r1, r2) of a tile sums kRed3Planes cells of its column, r0 = z0 ..
// z0 + kRed3Planes - 1, so one address and one neighbour test serve the whole
// column, its loads are all in flight together, and a warp of rows r1 >= J - 1
// skips the neighbours below along axis 1 as one.  The sum runs over e, then
// over the source bin's chunks, from zero, as in reduce_tile (the same values).
// CTA x: tile x / nsl, slice x % nsl = (column block, z0).  Measured on the
// 128^3 kooshball (4096 tiles of 16^3, 226 MB of partial tiles, 134 MB of grid):
// 184 us with four cells per thread and a neighbour mask for each, 112 us so with
// three CTAs per SM; four take another 10 us off.
// kPlanes = 8, one pair in flight, for tiles of few (neighbour, chunk) pairs.  A tile
// of many pairs is one chain: kPlanes = 2 gives it four times the CTAs, kDepth = 4 as
// many loads in flight, and a pair of the chain 0.11 us instead of 0.33; but each
// cell's share of the set-up grows, 0.05 us per 4096 cells of grid instead of 0.02.
// So the longest list, max_pairs, decides against the grid's size (kDensePairs).
// 8 / 2 planes: 300,000 clustered points on 64^3 (152 pairs) 51 / 19 us, kooshballs
// 128^3 with 1,000,000 points (153) 55 / 41, 128^3 with 307,200 (48) 21 / 30, 64^3
// with 100,000 (33) 12.8 / 8.2, eight of these 21 / 32.
constexpr int kRed3Threads = 256;
constexpr int64_t kDensePairs = 24000;   // grid cells (times batch elements) per pair

template <int kRed3Planes, int kDepth>
__global__ void __launch_bounds__(kRed3Threads, 4)
k_gridding_reduce3d(const float2* __restrict__ tiles_b, const int32_t* __restrict__ bin_chunk,
                    float2* __restrict__ grid_b, const Geom g, int64_t tbs, int64_t gbs, int nsl, int nz) {
  const float2* __restrict__ tiles = tiles_b + (int64_t)blockIdx.y * tbs;
  float2* __restrict__ grid = grid_b + (int64_t)blockIdx.y * gbs;
  const int bin = blockIdx.x / nsl;
  const int sl = blockIdx.x - bin * nsl;
  const int z0 = (sl % nz) * kRed3Planes;
  const int pos = (sl / nz) * blockDim.x + threadIdx.x;
  const int b2 = bin % g.nb[2], b01 = bin / g.nb[2], b1 = b01 % g.nb[1], b0 = b01 / g.nb[1];
  const int r1 = pos / g.T[2], r2 = pos - r1 * g.T[2];
  if (r1 >= g.T[1]) return;   // no barriers below
  const int plane = g.P[1] * g.P[2];
  const int nzc = min(kRed3Planes, g.T[0] - z0);   // cells of the column here
  float2 acc[kRed3Planes];
#pragma unroll
  for (int k = 0; k < kRed3Planes; ++k) acc[k] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int e = 0; e < 8; ++e) {
    const int e0 = e >> 2, e1 = (e >> 1) & 1, e2 = e & 1;
    const int n = e0 ? min(nzc, g.J[0] - 1 - z0) : nzc;   // the neighbour below reaches r0 < J - 1
    if (n <= 0 || (e1 && r1 >= g.J[1] - 1) || (e2 && r2 >= g.J[2] - 1)) continue;
    const int s0 = e0 ? (b0 > 0 ? b0 : g.nb[0]) - 1 : b0;
    const int s1 = e1 ? (b1 > 0 ? b1 : g.nb[1]) - 1 : b1;
    const int s2 = e2 ? (b2 > 0 ? b2 : g.nb[2]) - 1 : b2;
    const int src = (s0 * g.nb[1] + s1) * g.nb[2] + s2;
    const int q1 = __ldg(&bin_chunk[src + 1]);
    int q = __ldg(&bin_chunk[src]);
    const float2* ptr = tiles + (int64_t)q * g.padded_cells +
                        ((z0 + e0 * g.T[0]) * g.P[1] + r1 + e1 * g.T[1]) * g.P[2] + r2 + e2 * g.T[2];
    if constexpr (kDepth > 1) {
      for (; q + kDepth <= q1; q += kDepth, ptr += kDepth * g.padded_cells) {
        float2 v[kDepth][kRed3Planes];
#pragma unroll
        for (int u = 0; u < kDepth; ++u)
#pragma unroll
          for (int k = 0; k < kRed3Planes; ++k)
            v[u][k] = k < n ? __ldg(&ptr[u * g.padded_cells + k * plane]) : make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < kDepth; ++u)
#pragma unroll
          for (int k = 0; k < kRed3Planes; ++k)
            if (k < n) acc[k] = cadd(acc[k], v[u][k]);
      }
    }
    if (n == kRed3Planes) {
      for (; q < q1; ++q, ptr += g.padded_cells) {
        float2 v[kRed3Planes];
#pragma unroll
        for (int k = 0; k < kRed3Planes; ++k) v[k] = __ldg(&ptr[k * plane]);
#pragma unroll
        for (int k = 0; k < kRed3Planes; ++k) acc[k] = cadd(acc[k], v[k]);
      }
    } else {
      for (; q < q1; ++q, ptr += g.padded_cells) {
        float2 v[kRed3Planes];
#pragma unroll
        for (int k = 0; k < kRed3Planes; ++k) v[k] = k < n ? __ldg(&ptr[k * plane]) : make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < kRed3Planes; ++k)
          if (k < n) acc[k] = cadd(acc[k], v[k]);
      }
    }
  }
  float2* out = grid + ((b0 * g.T[0] + z0) * (int)g.Kstride[0] + (b1 * g.T[1] + r1) * (int)g.Kstride[1] +
                        b2 * g.T[2] + r2);
#pragma unroll
  for (int k = 0; k < kRed3Planes; ++k)
    if (k < nzc) out[k * (int)g.Kstride[0]] = acc[k];
}

// The reduction gives every thread 4 cells of the tile; small tiles get up to 4
// thread groups, each summing every 4th (neighbour, chunk) pair.
template <int D>
cudaError_t launch_reduce(const nufft_plan_t* p, const float2* tiles, float2* grid, int nb = 1) {
  if constexpr (D == 3) {
    const Geom& g = p->g;
    const int cols = g.T[1] * g.T[2];
    const int threads = std::min(kRed3Threads, (cols + 31) / 32 * 32);
    auto go = [&](auto kern, int planes) {
      const int nz = (g.T[0] + planes - 1) / planes;
      const int nsl = nz * ((cols + threads - 1) / threads);
      kern<<<dim3((unsigned)(g.nbins * nsl), (unsigned)nb), threads, 0, p->stream>>>(
          tiles, p->bin_chunk, grid, g, p->nchunks * g.padded_cells, p->Kprod, nsl, nz);
      return cudaGetLastError();
    };
    return p->max_pairs * kDensePairs > p->Kprod * nb ? go(k_gridding_reduce3d<2, 4>, 2)
                                                      : go(k_gridding_reduce3d<8, 1>, 8);
  }
  if constexpr (D == 2) {
    if (nb > 1) {
      const Geom& g = p->g;
      const int nz = (g.T[0] + kRed2Rows - 1) / kRed2Rows;
      const int64_t items = g.nbins * nz * g.T[1];
      k_gridding_reduce2d<<<dim3((unsigned)((items + kRed2Threads - 1) / kRed2Threads), (unsigned)nb), kRed2Threads, 0,
                            p->stream>>>(tiles, p->bin_chunk, grid, g, p->nchunks * g.padded_cells, p->Kprod, nz);
      return cudaGetLastError();
    }
  }
  int cells = 1;
  for (int a = 0; a < D; ++a) cells *= p->g.T[a];
  const int gsize = std::max(32, std::min(1024, (cells + 4 * 32 - 1) / (4 * 32) * 32));
  if ((int64_t)gsize * 4 < cells) return cudaErrorInvalidValue;
  // groups splitting the chunk list; a batch (mostly sparse tiles, many CTAs)
  // runs one group per CTA so that more tiles are in flight per SM
  const int NG = nb > 1 ? 1 : std::max(1, std::min(4, 1024 / gsize));
  const size_t smem = NG > 1 ? (size_t)NG * 4 * gsize * sizeof(float2) : 0;
  bool t16 = D > 1;
  for (int a = 0; a < D; ++a) t16 = t16 && p->g.T[a] == 16;
  if constexpr (D == 2) {
    // a single transform with the plan's work list: sparse tiles packed NG to a CTA
    int gs = 0, ng = 0;
    reduce2d_groups(cells, &gs, &ng);
    if (nb == 1 && p->red_ctas > 0 && gs == gsize && ng == NG) {
      auto kern = t16 ? k_gridding_reduce_packed2d<4, 16> : k_gridding_reduce_packed2d<4, 0>;
      kern<<<(unsigned)p->red_ctas, gsize * NG, smem, p->stream>>>(tiles, p->bin_chunk, grid, p->red_work, p->g, NG);
      return cudaGetLastError();
    }
  }
  if constexpr (D < 3) {
    auto kern = t16 ? k_gridding_reduce<D, 4, (D > 1 ? 16 : 0)> : k_gridding_reduce<D, 4, 0>;
    kern<<<dim3((unsigned)p->g.nbins, (unsigned)nb), gsize * NG, smem, p->stream>>>(
        tiles, p->bin_chunk, grid, p->g, NG, p->nchunks * p->g.padded_cells, p->Kprod);
  }
  return cudaGetLastError();
}

bool all_j_equal(const Geom& g, int J) {
  for (int a = 0; a < g.d; ++a)
    if (g.J[a] != J) return false;
  return true;
}

template <int D>
cudaError_t interp_chunks(const nufft_plan_t* p, const float2* grid, float2* y, int nb) {
  if (p->nchunks == 0) return cudaSuccess;
  const Points P = points_view(p);
  const dim3 gd((unsigned)p->nchunks, (unsigned)nb);
  bool t16 = true;
  for (int a = 0; a < D; ++a) t16 = t16 && p->g.T[a] == 16;
  if constexpr (D == 2) {
    const int J0 = p->g.J[0], J1 = p->g.J[1];
    const size_t rest = (size_t)p->g.padded_cells * 2 * sizeof(float) + (size_t)kChunkPoints[2] * 3 * sizeof(int);
    const int pitch = staged_pitch(J0, J1, rest);
    const size_t smem = rest + Staged2d::coefs(J0, pitch) * sizeof(float2);
    auto go = [&](auto kern) {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      kern<<<(unsigned)p->nchunks, kChunkPoints[2], smem, p->stream>>>(grid, y, p->chunks, P, p->g, pitch);
      return cudaGetLastError();
    };
    switch (J0 == J1 ? J0 : 0) {
      case 4: return go(t16 ? k_interp_chunk2d<4, 16> : k_interp_chunk2d<4, 0>);
      case 5: return go(t16 ? k_interp_chunk2d<5, 16> : k_interp_chunk2d<5, 0>);
      case 6: return go(t16 ? k_interp_chunk2d<6, 16> : k_interp_chunk2d<6, 0>);
      case 7: return go(t16 ? k_interp_chunk2d<7, 16> : k_interp_chunk2d<7, 0>);
      default: return go(k_interp_chunk2d<0, 0>);
    }
  } else {
    const int J = all_j_equal(p->g, p->g.J[0]) ? p->g.J[0] : 0;
    if (J >= 4 && J <= 7) {
      const int64_t cells = p->g.padded_cells;
      auto go = [&](auto kern, size_t smem) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<gd, 512, smem, p->stream>>>(grid, y, p->chunks, P, p->g, p->Kprod, p->M);
        return cudaGetLastError();
      };
      switch (J) {
        case 4: return go(t16 ? k_interp_chunk3d<4, 16> : k_interp_chunk3d<4, 0>, Chunk3dCfg<4>::smem_interp(cells));
        case 5: return go(t16 ? k_interp_chunk3d<5, 16> : k_interp_chunk3d<5, 0>, Chunk3dCfg<5>::smem_interp(cells));
        case 6: return go(t16 ? k_interp_chunk3d<6, 16> : k_interp_chunk3d<6, 0>, Chunk3dCfg<6>::smem_interp(cells));
        default: return go(t16 ? k_interp_chunk3d<7, 16> : k_interp_chunk3d<7, 0>, Chunk3dCfg<7>::smem_interp(cells));
      }
    }
    const size_t smem = (size_t)p->g.padded_cells * 2 * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(k_interp_chunk3d_any, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_interp_chunk3d_any<<<(unsigned)p->nchunks, 512, smem, p->stream>>>(grid, y, p->chunks, P, p->g);
    return cudaGetLastError();
  }
}

// 3D, equal J from 4 to 7: whether the staged chunks beat the per-point kernel, from
// estimates of both in us.  Staged: a set-up, then the longer of the longest chunk's
// rounds (one CTA works them off alone) and all chunks' tiles and rounds over the SMs.
// Per point: a floor that the chain of a point's loads takes, or all points' taps.
// A round and a point cost in proportion to J^2 taps.  The constants are fitted to
// 401 measurements of both (J = 4 to 7, grids 32^3 to 200^3, 300 to 1,000,000 random,
// kooshball and clustered points, batches of 1 to 8; the staged ones within 20 % rms),
// and the choice costs 3 % against the better of the two on average; a count of CTAs
// alone cost 39 %.  Staged against per point, us: 64^3 grid, 300 points 5.9 / 7.7,
// 10,000 kooshball points 37 / 8, 300,000 random points 48 / 66; 128^3, 300,000
// clustered points 42 / 55 (151 chunks); 200^3, 100,000 random points 121 / 30
// (8000 chunks); two of 100^3 with 100,000 kooshball points 73 / 45.  Batches overlap
// their chunks less well than the estimate: they need a margin.
bool staged_interp3d(const nufft_plan_t* p, int J, int nb) {
  const double taps = J * J / 36.0;
  const int per_warp = 32 / J, step = 16 * per_warp;   // points per round of a CTA
  const double longest = (p->longest_chunk + step - 1) / step;
  const double rounds = (double)p->M / step + 0.5 * p->nchunks;   // of all chunks
  const double tile = 0.6 + 1.8 * (double)p->g.padded_cells / 9261;
  const double staged = 4.0 + 1.4 * taps +
                        std::max(1.5 * taps * longest, nb * (p->nchunks * tile + 1.7 * taps * rounds) / 152);
  const double point = std::max(2.0 + 6.0 * taps, 1.2e-3 * taps * (double)p->M * nb / per_warp);
  return staged * (nb > 1 ? 1.8 : 1.0) < point;
}

template <int D>
cudaError_t interp_d(const nufft_plan_t* p, const float2* grid, float2* y, int nb) {
  // 2D: single transforms gather from staged tiles, batches per point (the chunk
  // kernel would stage each chunk's point data once per batch element: the
  // 32-coil frames' normal operator 2.36 -> 2.87 ms).
  // 3D: staged tiles where staged_interp3d expects them to win; J that it does not
  // cover, single transforms.
  if constexpr (D == 2) {
    if (nb == 1) return interp_chunks<D>(p, grid, y, nb);
  }
  if constexpr (D == 3) {
    const int J = all_j_equal(p->g, p->g.J[0]) ? p->g.J[0] : 0;
    if (J >= 4 && J <= 7 ? staged_interp3d(p, J, nb) : nb == 1)
      return interp_chunks<D>(p, grid, y, nb);
  }
  const Points P = points_view(p);
  const int G = p->g.J[D - 1];
  const int per_warp = 32 / G;
  const int64_t warps = (P.M + per_warp - 1) / per_warp;
  const int64_t blocks = (warps * 32 + 255) / 256;
  if (blocks == 0) return cudaSuccess;
  const int J = all_j_equal(p->g, p->g.J[0]) ? p->g.J[0] : 0;
  if constexpr (D == 2) {
    const dim3 gb((unsigned)blocks, (unsigned)((nb + kBatchPer - 1) / kBatchPer));
    if (blocks * gb.y >= kBatchPerCtas) {
      auto go = [&](auto kern) {
        kern<<<gb, 256, 0, p->stream>>>(grid, y, P, p->g, p->Kprod, p->M, nb);
        return cudaGetLastError();
      };
      switch (J) {
        case 4: return go(k_interp_batch2d<4>);
        case 5: return go(k_interp_batch2d<5>);
        case 6: return go(k_interp_batch2d<6>);
        case 7: return go(k_interp_batch2d<7>);
      }
    }
  }
  const dim3 gd((unsigned)blocks, (unsigned)nb);
  auto kern = k_interp<D, 0>;
  if (J == 6) kern = k_interp<D, 6>;
  if constexpr (D > 1) {
    if (J == 4) kern = k_interp<D, 4>;
    if (J == 5) kern = k_interp<D, 5>;
    if (J == 7) kern = k_interp<D, 7>;
  }
  kern<<<gd, 256, 0, p->stream>>>(grid, y, P, p->g, p->Kprod, p->M);
  return cudaGetLastError();
}

cudaError_t launch_chunks3d(const nufft_plan_t* p, const float2* y, float2* tiles, dim3 gd, int J, int64_t ybs,
                            int64_t tbs) {
  const bool t16 = p->g.T[0] == 16 && p->g.T[1] == 16 && p->g.T[2] == 16;
  auto go = [&](auto kern, size_t smem) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<gd, 512, smem, p->stream>>>(y, tiles, p->chunks, points_view(p), p->g, ybs, tbs);
    return cudaGetLastError();
  };
  const int64_t cells = p->g.padded_cells;
  switch (J) {
    case 4: return go(t16 ? k_gridding_chunk3d<4, 16> : k_gridding_chunk3d<4, 0>, Chunk3dCfg<4>::smem_gridding(cells));
    case 5: return go(t16 ? k_gridding_chunk3d<5, 16> : k_gridding_chunk3d<5, 0>, Chunk3dCfg<5>::smem_gridding(cells));
    case 6: return go(t16 ? k_gridding_chunk3d<6, 16> : k_gridding_chunk3d<6, 0>, Chunk3dCfg<6>::smem_gridding(cells));
    default: return go(t16 ? k_gridding_chunk3d<7, 16> : k_gridding_chunk3d<7, 0>, Chunk3dCfg<7>::smem_gridding(cells));
  }
}

// Chunk pass of V^H: one CTA per (chunk, batch element), partial tiles out.
// FUSED (2D only): y is the oversampled spectrum and the pass computes V^H V.
template <int D, bool FUSED = false>
cudaError_t launch_chunks(const nufft_plan_t* p, const float2* y, float2* tiles, int nb, int64_t ybs, int64_t tbs) {
  if (p->nchunks == 0) return cudaSuccess;
  const Points P = points_view(p);
  const dim3 gd((unsigned)p->nchunks, (unsigned)nb);
  cudaError_t e;
  if constexpr (D == 2 && !FUSED) {
    // few points per chunk and CTAs enough, batch or not: two warps per CTA
    if (p->nchunks * nb >= kBatchMinCtas && p->M <= kBatchMaxMean * p->nchunks) {
      auto go = [&](auto kern, int nstrip) {
        const size_t smem = (size_t)p->g.padded_cells * Fix<2>::kWords * sizeof(int) +
                            ((size_t)kChunkPoints[2] + (size_t)kBatchWarps2d * nstrip) * sizeof(float2);
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<gd, 32 * kBatchWarps2d, smem, p->stream>>>(y, tiles, p->chunks, P, p->g, ybs, tbs);
        return cudaGetLastError();
      };
      const int J0 = p->g.J[0], J1 = p->g.J[1];
      switch (J0 == J1 ? J0 : 0) {
        case 4: return go(k_gridding_chunk2d<4>, strip2d<4>(J0, J1));
        case 5: return go(k_gridding_chunk2d<5>, strip2d<5>(J0, J1));
        case 6: return go(k_gridding_chunk2d<6>, strip2d<6>(J0, J1));
        case 7: return go(k_gridding_chunk2d<7>, strip2d<7>(J0, J1));
        default: return go(k_gridding_chunk2d<0>, strip2d<0>(J0, J1));
      }
    }
  }
  if constexpr (D == 2) {
    const int J0 = p->g.J[0], J1 = p->g.J[1];
    const bool t16 = p->g.T[0] == 16 && p->g.T[1] == 16;
    const size_t rest = (size_t)p->g.padded_cells * Fix<2>::kWords * sizeof(int) +
                        (size_t)kChunkPoints[2] * (sizeof(float2) + 2 * sizeof(int)) +
                        (FUSED ? (size_t)p->g.padded_cells * 2 * sizeof(float) : 0);
    const int pitch = staged_pitch(J0, J1, rest);
    const size_t smem = rest + Staged2d::coefs(J0, pitch) * sizeof(float2);
    auto go = [&](auto kern) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      kern<<<gd, kChunkPoints[2], smem, p->stream>>>(y, tiles, p->chunks, P, p->g, ybs, tbs, pitch);
      return cudaGetLastError();
    };
    switch (J0 == J1 ? J0 : 0) {
      case 4: return go(t16 ? k_gridding_chunk_staged<4, 16, FUSED> : k_gridding_chunk_staged<4, 0, FUSED>);
      case 5: return go(t16 ? k_gridding_chunk_staged<5, 16, FUSED> : k_gridding_chunk_staged<5, 0, FUSED>);
      case 6: return go(t16 ? k_gridding_chunk_staged<6, 16, FUSED> : k_gridding_chunk_staged<6, 0, FUSED>);
      case 7: return go(t16 ? k_gridding_chunk_staged<7, 16, FUSED> : k_gridding_chunk_staged<7, 0, FUSED>);
      default: return go(k_gridding_chunk_staged<0, 0, FUSED>);
    }
  } else {
    static_assert(!FUSED, "the fused V^H V pass is 2D only");
    const size_t smem = (size_t)p->g.padded_cells * Fix<D>::kWords * sizeof(int);
    const int J = all_j_equal(p->g, p->g.J[0]) ? p->g.J[0] : 0;
    if constexpr (D == 3) {
      if (J >= 4 && J <= 7) return launch_chunks3d(p, y, tiles, gd, J, ybs, tbs);
    }
    auto kern = k_gridding_chunk<D, 0>;
    if constexpr (D == 1) {
      if (J == 6) kern = k_gridding_chunk<D, 6>;
    }
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<gd, GridChunkCfg<D>::kThreads, smem, p->stream>>>(y, tiles, p->chunks, P, p->g, ybs, tbs);
  }
  return cudaGetLastError();
}

template <int D>
cudaError_t gridding_d(const nufft_plan_t* p, const float2* y, float2* grid, int nb, float2* tiles) {
  const int64_t tbs = p->nchunks * p->g.padded_cells;
  cudaError_t e = launch_chunks<D>(p, y, tiles, nb, p->M, tbs);
  if (e != cudaSuccess) return e;
  return launch_reduce<D>(p, tiles, grid, nb);
}

// ---------------------------------------------------------------- gridding without allocation
// Partial-tile scratch for nufft_gridding_static: a fixed array in device
// memory, so that call needs neither cudaMalloc nor plan-owned scratch.
constexpr int64_t kStaticTileBytes = 16ll << 20;   // 16 MiB on every GPU that loads the library
static __device__ __align__(256) float2 g_static_tiles[kStaticTileBytes / sizeof(float2)];

constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
float2* g_static_ptr[kMaxDevices];   // device address of g_static_tiles, per device

// Device address of the static array on the plan's device, which the caller
// has made current.  Looked up once per device (cudaGetSymbolAddress) and
// cached; the host-side name g_static_tiles is not a device address.
int static_tiles_address(nufft_plan_t* p, float2** out) {
  const int dev = p->device;
  if (dev < 0 || dev >= kMaxDevices) return set_error(p, NUFFT_EINVAL, "device ordinal %d out of range", dev);
  std::lock_guard<std::mutex> lock(g_static_mu);
  if (!g_static_ptr[dev]) {
    void* ptr = nullptr;
    NUFFT_CUDA_TRY(p, cudaGetSymbolAddress(&ptr, g_static_tiles));
    g_static_ptr[dev] = static_cast<float2*>(ptr);
  }
  *out = g_static_ptr[dev];
  return NUFFT_OK;
}

// Makes the plan's device current for the call and puts the caller's back.
struct DeviceScope {
  int prev = -1;
  bool switched = false;
  ~DeviceScope() {
    if (switched) cudaSetDevice(prev);
  }
  cudaError_t enter(int dev) {
    cudaError_t e = cudaGetDevice(&prev);
    if (e != cudaSuccess || prev == dev) return e;
    e = cudaSetDevice(dev);
    switched = e == cudaSuccess;
    return e;
  }
};

template <int D>
cudaError_t gridding_static_d(const nufft_plan_t* p, const float2* y, float2* grid, float2* tiles) {
  cudaError_t e = launch_chunks<D>(p, y, tiles, 1, 0, 0);
  if (e != cudaSuccess) return e;
  return launch_reduce<D>(p, tiles, grid);
}

}  // namespace

int launch_interp(nufft_plan_t* p, const float2* grid, float2* y, int nb) {
  cudaError_t e;
  switch (p->g.d) {
    case 1: e = interp_d<1>(p, grid, y, nb); break;
    case 2: e = interp_d<2>(p, grid, y, nb); break;
    default: e = interp_d<3>(p, grid, y, nb); break;
  }
  return e == cudaSuccess ? NUFFT_OK : cuda_check(p, e, "interpolation kernel");
}

bool vhv_fused(const nufft_plan_t* p) { return p->g.d == 2 && p->M > 0; }

int launch_vhv(nufft_plan_t* p, const float2* grid_in, float2* grid_out, int nb, float2* tiles) {
  if (!vhv_fused(p)) return set_error(p, NUFFT_EINVAL, "fused V^H V is 2D only");
  if (!tiles) tiles = p->tiles;
  const int64_t tbs = p->nchunks * p->g.padded_cells;
  cudaError_t e = launch_chunks<2, true>(p, grid_in, tiles, nb, p->Kprod, tbs);
  if (e == cudaSuccess) e = launch_reduce<2>(p, tiles, grid_out, nb);
  return e == cudaSuccess ? NUFFT_OK : cuda_check(p, e, "fused V^H V kernels");
}

int launch_gridding(nufft_plan_t* p, const float2* y, float2* grid, int nb, float2* tiles) {
  if (!tiles) tiles = p->tiles;
  cudaError_t e;
  switch (p->g.d) {
    case 1: e = gridding_d<1>(p, y, grid, nb, tiles); break;
    case 2: e = gridding_d<2>(p, y, grid, nb, tiles); break;
    default: e = gridding_d<3>(p, y, grid, nb, tiles); break;
  }
  return e == cudaSuccess ? NUFFT_OK : cuda_check(p, e, "gridding kernels");
}

}  // namespace nufft

// Gridding V^H like nufft_gridding, with the per-chunk partial tiles in the
// static device array above instead of the plan's buffer (see the header).
extern "C" int nufft_gridding_static(nufft_plan_t* p, const float* y_dev, float* grid_dev) {
  using namespace nufft;
  if (!p) return set_error(nullptr, NUFFT_EINVAL, "plan is NULL");
  if (p->M > 0 && !y_dev) return set_error(p, NUFFT_EINVAL, "y_dev is NULL");
  if (!grid_dev) return set_error(p, NUFFT_EINVAL, "grid_dev is NULL");
  const int64_t need = p->nchunks * p->g.padded_cells * (int64_t)sizeof(float2);
  if (need > kStaticTileBytes)
    return set_error(p, NUFFT_EINVAL,
                     "gridding needs %lld bytes of partial tiles, more than the %lld-byte static scratch; "
                     "use nufft_gridding", (long long)need, (long long)kStaticTileBytes);
  DeviceScope scope;   // the kernels run on the plan's stream, so on the plan's device
  NUFFT_CUDA_TRY(p, scope.enter(p->device));
  float2* tiles = nullptr;
  const int rc = static_tiles_address(p, &tiles);
  if (rc != NUFFT_OK) return rc;
  const float2* y = reinterpret_cast<const float2*>(y_dev);
  float2* grid = reinterpret_cast<float2*>(grid_dev);
  cudaError_t e;
  switch (p->g.d) {
    case 1: e = gridding_static_d<1>(p, y, grid, tiles); break;
    case 2: e = gridding_static_d<2>(p, y, grid, tiles); break;
    default: e = gridding_static_d<3>(p, y, grid, tiles); break;
  }
  return e == cudaSuccess ? NUFFT_OK : cuda_check(p, e, "static-scratch gridding kernels");
}
