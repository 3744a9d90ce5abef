// Two-colour FP32 sweeps of the refinement's inner pressure solve
// (Sec. 3.4's scheduled relaxation, the library's own schedule).
//
// The cells (point sweeps: colour (i + j + k) & 1; z-line sweeps: columns of
// colour (i + j) & 1) form two colours whose stencils read only the other
// colour, when nx and ny are even.  Sweep m of a cycle relaxes colour m & 1
// alone, in place, with the factor
//   omega_0 = 1,  omega_1 = 1/(1 - sigma^2/2),
//   omega_{m+1} = 1/(1 - sigma^2 omega_m/4),  sigma = 1 - mu_min
// (Chebyshev acceleration on a two-coloured grid; Golub and Varga, Numer.
// Math. 3, 1961).  Because the Jacobi spectrum is symmetric about 1 on such a
// grid, M of these half sweeps reduce the error by the same Chebyshev factor
// 1/T_M as M Jacobi sweeps with the Chebyshev weights: a cycle keeps its
// length, and each sweep touches half the cells.  The factors stay below 2,
// so no partial product amplifies rounding.
//
// Layout: an array of nx ny nz floats holds the two colours one after the
// other, each [nz][ny][nx/2]; cell i of a row is entry i >> 1 of its colour.
// In row (j, k) the cells of colour c are i = 2 m + s, s = (j + zc k + c) & 1
// (zc = 1 for point sweeps, 0 for z lines), their y and z neighbours are
// entry m of the other colour's neighbouring rows, and their x neighbours
// entries m and m - 1 (s = 0) or m + 1 (s = 1) of its row (j, k).
#include <algorithm>

#include "device_util.cuh"
#include "poisson_common.cuh"
#include "stp_internal.cuh"

namespace stp {
namespace {

template <int W>
struct Vec {
  float v[W];
};
template <int W>
__device__ __forceinline__ Vec<W> vld(const float* p) {
  Vec<W> r;
  if constexpr (W == 4) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p));
    r.v[0] = t.x, r.v[1] = t.y, r.v[2] = t.z, r.v[3] = t.w;
  } else if constexpr (W == 2) {
    const float2 t = __ldg(reinterpret_cast<const float2*>(p));
    r.v[0] = t.x, r.v[1] = t.y;
  } else {
    r.v[0] = __ldg(p);
  }
  return r;
}
// values this kernel also writes (the colour being relaxed): plain loads
template <int W>
__device__ __forceinline__ Vec<W> vld_rw(const float* p) {
  Vec<W> r;
  if constexpr (W == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    r.v[0] = t.x, r.v[1] = t.y, r.v[2] = t.z, r.v[3] = t.w;
  } else if constexpr (W == 2) {
    const float2 t = *reinterpret_cast<const float2*>(p);
    r.v[0] = t.x, r.v[1] = t.y;
  } else {
    r.v[0] = *p;
  }
  return r;
}
template <int W>
__device__ __forceinline__ void vst(float* p, const Vec<W>& r) {
  if constexpr (W == 4)
    *reinterpret_cast<float4*>(p) = make_float4(r.v[0], r.v[1], r.v[2], r.v[3]);
  else if constexpr (W == 2)
    *reinterpret_cast<float2*>(p) = make_float2(r.v[0], r.v[1]);
  else
    *p = r.v[0];
}
template <int W>
__device__ __forceinline__ Vec<W> vaxpy(float a, const Vec<W>& x, const Vec<W>& y) {
  Vec<W> r;
#pragma unroll
  for (int e = 0; e < W; e++) r.v[e] = fmaf(a, x.v[e], y.v[e]);
  return r;
}

// One point sweep of one colour: a thread relaxes W cells of a row at KZ
// consecutive levels (the other colour's column of the row rides in
// registers: it serves the x neighbours of its level and the z neighbours
// of the levels around it).  Threads take the row's units, then the rows,
// then the slabs of KZ levels.
template <int W, int KZ>
__global__ void __launch_bounds__(256) k_col_point(Geom<float> g, float* __restrict__ own,
                                                   const float* __restrict__ oth, const float* __restrict__ r,
                                                   float omega, int c) {
  const int ny = g.ny, nz = g.nz, hx = g.nx >> 1, uw = hx / W;
  const unsigned plane = (unsigned)hx * ny;
  const unsigned f = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned pu = (unsigned)uw * ny;
  const unsigned slab = f / pu, rest = f - slab * pu;
  const int j = (int)(rest / (unsigned)uw), x = (int)(rest - (unsigned)j * uw) * W;
  const int k0 = (int)slab * KZ;
  if (k0 >= nz) return;
  const unsigned rc = (unsigned)j * hx + x;
  const unsigned rn = (unsigned)(j == ny - 1 ? 0 : j + 1) * hx + x;
  const unsigned rs = (unsigned)(j == 0 ? ny - 1 : j - 1) * hx + x;
  const unsigned xl = (unsigned)j * hx + (x == 0 ? hx - 1 : x - 1), xr = (unsigned)j * hx + (x + W == hx ? 0 : x + W);
  const float idx2 = g.idx2, idy2 = g.idy2;
  cudaGridDependencySynchronize();
  Vec<W> o[KZ + 2], pc[KZ], yn[KZ], ys[KZ], bb[KZ];
  float ex[KZ];
#pragma unroll
  for (int q = 0; q < KZ + 2; q++) {
    const int k = k0 + q - 1;
    if (k >= 0 && k < nz) o[q] = vld<W>(oth + (unsigned)k * plane + rc);
    else o[q] = Vec<W>{};
  }
#pragma unroll
  for (int q = 0; q < KZ; q++) {
    const int k = k0 + q;
    if (k < nz) {
      const unsigned lev = (unsigned)k * plane;
      ex[q] = __ldg(oth + lev + (((j + k + c) & 1) ? xr : xl));
      yn[q] = vld<W>(oth + lev + rn);
      ys[q] = vld<W>(oth + lev + rs);
      bb[q] = vld<W>(r + lev + rc);
      pc[q] = vld_rw<W>(own + lev + rc);
    }
  }
#pragma unroll
  for (int q = 0; q < KZ; q++) {
    const int k = k0 + q;
    if (k < nz) {
      const bool odd = (j + k + c) & 1;
      // walls: cup (cdn) is zero at the top (bottom) level
      const float cup = __ldg(g.cup + k), cdn = __ldg(g.cdn + k), iS = __ldg(g.iS + k);
      Vec<W> out;
#pragma unroll
      for (int e = 0; e < W; e++) {
        const float prev = e == 0 ? ex[q] : o[q + 1].v[e - 1], next = e == W - 1 ? ex[q] : o[q + 1].v[e + 1];
        out.v[e] = srj_cell_f32(pc[q].v[e], o[q + 1].v[e], odd ? next : prev, yn[q].v[e], ys[q].v[e], o[q + 2].v[e],
                                o[q].v[e], bb[q].v[e], idx2, idy2, cup, cdn, iS, omega);
      }
      vst<W>(own + (unsigned)k * plane + rc, out);
    }
  }
}

// One z-line sweep of one colour of columns: the register-chunked column
// solve of k_line_sweep_chunk (kernels_poisson.cu) on half rows.  A block
// takes 8 units of W columns of a row x NCH level chunks of at most LMAX
// levels; each thread holds its chunk's right-hand side in registers, the
// elimination and substitution recurrences run inside the chunk from zero,
// and the values entering a chunk come from the chunk boundary values in
// shared memory.
template <int W, int NCH, int LMAX, int MINB>
__global__ void __launch_bounds__(8 * NCH, MINB) k_col_line(Geom<float> g, float* __restrict__ own,
                                                            const float* __restrict__ oth,
                                                            const float* __restrict__ r, float omega, int c0l) {
  constexpr int U = 8, H = NCH / 2;
  using V = Vec<W>;
  __shared__ V ZB[NCH][U], WB[NCH][U], XT[U];
  __shared__ float FB[NCH], EB[NCH];
  const int ny = g.ny, nz = g.nz, t = nz >> 1, hx = g.nx >> 1, uw = hx / W;
  const int ntx = (uw + U - 1) / U;
  const int u = threadIdx.x % U, c = threadIdx.x / U;
  const int j = blockIdx.x / ntx, xu = (blockIdx.x % ntx) * U + u;
  const bool act = xu < uw;
  const int x = (act ? xu : uw - 1) * W;
  const unsigned plane = (unsigned)hx * ny;
  const unsigned rc = (unsigned)j * hx + x;
  const unsigned rn = (unsigned)(j == ny - 1 ? 0 : j + 1) * hx + x;
  const unsigned rs = (unsigned)(j == 0 ? ny - 1 : j - 1) * hx + x;
  const bool odd = (j + c0l) & 1;
  const unsigned xe = (unsigned)j * hx + (odd ? (x + W == hx ? 0 : x + W) : (x == 0 ? hx - 1 : x - 1));
  const bool lower = c < H;
  int k0, k1;
  line_chunk_levels<NCH>(c, nz, k0, k1);
  const int L = k1 - k0;
  const bool twist = c == H;
  const float idx2 = g.idx2, idy2 = g.idy2;
  V G[LMAX];
  cudaGridDependencySynchronize();
  {
    V cc = {}, zd = {};
    if (L > 0) {
      cc = vld_rw<W>(own + (unsigned)k0 * plane + rc);
      zd = k0 > 0 ? vld_rw<W>(own + (unsigned)(k0 - 1) * plane + rc) : cc;
    }
#pragma unroll
    for (int q = 0; q < LMAX; q++) {
      if (q < L) {
        const int k = k0 + q;
        const unsigned lev = (unsigned)k * plane;
        const V oc = vld<W>(oth + lev + rc);
        const V yn = vld<W>(oth + lev + rn), ys = vld<W>(oth + lev + rs);
        const V zu = k < nz - 1 ? vld_rw<W>(own + lev + plane + rc) : cc;
        const V bq = vld<W>(r + lev + rc);
        const float ex = __ldg(oth + lev + xe);
        const float4 cf = __ldg(g.lz4 + k);  // cup, cdn (zero at the walls), 1/pivot, elimination ratio
#pragma unroll
        for (int e = 0; e < W; e++) {
          const float pc = cc.v[e];
          const float prev = e == 0 ? ex : oc.v[e - 1], next = e == W - 1 ? ex : oc.v[e + 1];
          // (a fixed sequence of roundings: the widths give the same bits)
          float lap = __fmul_rn(idy2, __fadd_rn(__fsub_rn(yn.v[e], pc), __fsub_rn(ys.v[e], pc)));
          lap = __fmaf_rn(idx2, __fadd_rn(__fsub_rn(oc.v[e], pc), __fsub_rn(odd ? next : prev, pc)), lap);
          lap = __fmaf_rn(cf.x, __fsub_rn(zu.v[e], pc), lap);
          lap = __fmaf_rn(cf.y, __fsub_rn(zd.v[e], pc), lap);
          G[q].v[e] = __fmul_rn(__fsub_rn(bq.v[e], lap), cf.z);
        }
        zd = cc;
        cc = zu;
      }
    }
  }
  // elimination inside the chunk (upward below t, downward above it)
  {
    V z = {};
    float F = 1.f;
    if (lower) {
#pragma unroll
      for (int q = 0; q < LMAX; q++)
        if (q < L) {
          const float f = __ldg(g.lz4 + k0 + q).w;
          z = vaxpy<W>(f, z, G[q]);
          F *= f;
          G[q] = z;
        }
    } else {
#pragma unroll
      for (int q = LMAX - 1; q >= 0; q--)
        if (q < L && (q > 0 || !twist)) {
          const float f = __ldg(g.lz4 + k0 + q).w;
          z = vaxpy<W>(f, z, G[q]);
          F *= f;
          G[q] = z;
        }
    }
    ZB[c][u] = z;
    if (u == 0) FB[c] = F;
  }
  __syncthreads();
  // carries of the elimination from the walls; the twist value
  {
    V carry = {};
    if (lower) {
      for (int cc = 0; cc < c; cc++) carry = vaxpy<W>(FB[cc], carry, ZB[cc][u]);
      float F = 1.f;
#pragma unroll
      for (int q = 0; q < LMAX; q++)
        if (q < L) {
          F *= __ldg(g.lz4 + k0 + q).w;
          G[q] = vaxpy<W>(F, carry, G[q]);
        }
    } else {
      for (int cc = NCH - 1; cc > c; cc--) carry = vaxpy<W>(FB[cc], carry, ZB[cc][u]);
      float F = 1.f;
#pragma unroll
      for (int q = LMAX - 1; q >= 0; q--)
        if (q < L && (q > 0 || !twist)) {
          F *= __ldg(g.lz4 + k0 + q).w;
          G[q] = vaxpy<W>(F, carry, G[q]);
        }
      if (twist) {
        V ylow = {};  // y_{t-1}
        for (int cc = 0; cc < H; cc++) ylow = vaxpy<W>(FB[cc], ylow, ZB[cc][u]);
        const V yup = L >= 2 ? G[1] : carry;  // y_{t+1}
        const float ft = t > 0 ? __ldg(g.lz4 + t).w : 0.f, et = t < nz - 1 ? __ldg(g.tlb + t) : 0.f;
        G[0] = vaxpy<W>(et, yup, vaxpy<W>(ft, ylow, G[0]));
      }
    }
  }
  // substitution inside the chunk (downward below t, upward above it); the
  // twist chunk publishes x_t and its top value
  {
    V w = {};
    float E = 1.f;
    if (lower) {
#pragma unroll
      for (int q = LMAX - 1; q >= 0; q--)
        if (q < L) {
          const float e = __ldg(g.tlb + k0 + q);
          w = vaxpy<W>(e, w, G[q]);
          E *= e;
          G[q] = w;
        }
    } else {
#pragma unroll
      for (int q = 0; q < LMAX; q++)
        if (q < L && (q > 0 || !twist)) {
          const float e = __ldg(g.tlb + k0 + q);
          w = vaxpy<W>(e, w, G[q]);
          E *= e;
          G[q] = w;
        }
      if (twist) {
        w = vaxpy<W>(E, G[0], w);  // x at the chunk's top level, absolute
        E = 0.f;
        XT[u] = G[0];
      }
    }
    WB[c][u] = w;
    if (u == 0) EB[c] = E;
  }
  __syncthreads();
  // carries of the substitution from the twist level; the update (every
  // read of this colour's columns by the block lies before the barriers)
  {
    V carry = twist ? G[0] : XT[u];
    if (lower) {
      for (int cc = H - 1; cc > c; cc--) carry = vaxpy<W>(EB[cc], carry, WB[cc][u]);
      float E = 1.f;
#pragma unroll
      for (int q = LMAX - 1; q >= 0; q--)
        if (q < L) {
          E *= __ldg(g.tlb + k0 + q);
          G[q] = vaxpy<W>(E, carry, G[q]);
        }
    } else {
      for (int cc = H; cc < c; cc++) carry = vaxpy<W>(EB[cc], carry, WB[cc][u]);
      float E = 1.f;
#pragma unroll
      for (int q = 0; q < LMAX; q++)
        if (q < L && (q > 0 || !twist)) {
          E *= __ldg(g.tlb + k0 + q);
          G[q] = vaxpy<W>(E, carry, G[q]);
        }
    }
    if (act) {
#pragma unroll
      for (int q = 0; q < LMAX; q++)
        if (q < L) {
          float* a = own + (unsigned)(k0 + q) * plane + rc;
          vst<W>(a, vaxpy<W>(-omega, G[q], vld_rw<W>(a)));
        }
    }
  }
}

// ||r - L d||_2 in the two-colour layout and the once-per-cycle decision (as
// k_check<float, 1>): a thread takes W entries of both colours of one row.
template <int W>
__global__ void __launch_bounds__(256) k_col_check(Geom<float> g, const float* __restrict__ d,
                                                   const float* __restrict__ r, int zc, SolveCtl* ctl, Red red,
                                                   unsigned nblocks, int graph, cudaGraphConditionalHandle h_loop,
                                                   cudaGraphConditionalHandle h_body) {
  __shared__ double sh[32];
  const int ny = g.ny, nz = g.nz, hx = g.nx >> 1, uw = hx / W;
  const unsigned plane = (unsigned)hx * ny;
  const size_t half = (size_t)plane * nz;
  const unsigned f = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned row = f / (unsigned)uw;
  const int x = (int)(f - row * uw) * W, k = (int)(row / (unsigned)ny), j = (int)(row - (unsigned)k * ny);
  float s2 = 0.f;
  if (k < nz) {
    const unsigned lev = (unsigned)k * plane, rc = lev + (unsigned)j * hx + x;
    const unsigned rn = lev + (unsigned)(j == ny - 1 ? 0 : j + 1) * hx + x;
    const unsigned rs = lev + (unsigned)(j == 0 ? ny - 1 : j - 1) * hx + x;
    const unsigned xl = lev + (unsigned)j * hx + (x == 0 ? hx - 1 : x - 1);
    const unsigned xr = lev + (unsigned)j * hx + (x + W == hx ? 0 : x + W);
    const float idx2 = g.idx2, idy2 = g.idy2, cup = __ldg(g.cup + k), cdn = __ldg(g.cdn + k);
    Vec<W> own = vld<W>(d + rc), oc = vld<W>(d + half + rc);
#pragma unroll
    for (int c = 0; c < 2; c++) {
      const float* oth = d + (c ? 0 : half);
      const float* zn = zc ? oth : d + (c ? half : 0);  // z neighbours: the other colour (point), the same (lines)
      const bool odd = (j + zc * k + c) & 1;
      const Vec<W> yn = vld<W>(oth + rn), ys = vld<W>(oth + rs), bb = vld<W>(r + (c ? half : 0) + rc);
      const Vec<W> zu = k < nz - 1 ? vld<W>(zn + rc + plane) : own, zd = k > 0 ? vld<W>(zn + rc - plane) : own;
      const float ex = __ldg(oth + (odd ? xr : xl));
#pragma unroll
      for (int e = 0; e < W; e++) {
        const float pc = own.v[e];
        const float prev = e == 0 ? ex : oc.v[e - 1], next = e == W - 1 ? ex : oc.v[e + 1];
        float lap = idx2 * ((oc.v[e] - pc) + ((odd ? next : prev) - pc)) +
                    idy2 * ((yn.v[e] - pc) + (ys.v[e] - pc));
        lap += cup * (zu.v[e] - pc);
        lap += cdn * (zd.v[e] - pc);
        const float q = bb.v[e] - lap;
        s2 = fmaf(q, q, s2);
      }
      const Vec<W> t = own;
      own = oc;
      oc = t;
    }
  }
  const double s = block_sum_f32(s2, sh);
  if (publish_partial_tree(red, nblocks, s, 0.0, false)) {
    const double tot = final_sum(red.partial, nblocks, sh);
    if (threadIdx.x == 0) {
      const bool go = cycle_decide<1>(ctl, red, sqrt(tot));
      if (graph) {
        cudaGraphSetConditional(h_loop, go ? 1u : 0u);
        cudaGraphSetConditional(h_body, go ? 1u : 0u);
      }
    }
  }
}

// Refinement residual (as k_outer), r stored in the two-colour layout.
__global__ void __launch_bounds__(kBX* kBY) k_col_outer(Geom<double> g, const double* __restrict__ p,
                                                         const double* __restrict__ b, float* __restrict__ r32, int zc,
                                                         SolveCtl* ctl, Red red, unsigned nblocks, int after_pass,
                                                         int graph, cudaGraphConditionalHandle h_loop) {
  __shared__ double sh[32];
  const int i = blockIdx.x * kBX + threadIdx.x, j = blockIdx.y * kBY + threadIdx.y, k = blockIdx.z;
  const double bmean = __ldcg(red.sc + SC_BMEAN);
  float r2 = 0.f;
  if (i < g.nx && j < g.ny) {
    const float r = (float)(point_residual_sum(g, p, b, i, j, k) - bmean);
    const int hx = g.nx >> 1, c = (i + j + zc * k) & 1;
    r32[((size_t)(c * g.nz + k) * g.ny + j) * hx + (i >> 1)] = r;
    r2 = r * r;
  }
  double s = block_sum_f32(r2, sh);
  if (publish_partial_tree(red, nblocks, s, 0.0, false)) {
    const double tot = final_sum(red.partial, nblocks, sh);
    if (threadIdx.x == 0 && threadIdx.y == 0) {
      const bool go = pass_decide(ctl, red, sqrt(tot), after_pass);
      if (graph) cudaGraphSetConditional(h_loop, go ? 1u : 0u);
    }
  }
}

// p += d, d in the two-colour layout: a thread takes the cells 2 m, 2 m + 1
__global__ void __launch_bounds__(256) k_col_addcorr(double* __restrict__ p, const float* __restrict__ d, int hx,
                                                     int ny, int nz, int zc) {
  const unsigned n = (unsigned)hx * ny * nz;
  for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
    const unsigned row = q / (unsigned)hx, k = row / (unsigned)ny, j = row - k * ny;
    const bool odd = (j + zc * k) & 1;  // colour of cell 2 m
    const float a = __ldg(d + q), b = __ldg(d + n + q);
    double2 v = reinterpret_cast<double2*>(p)[q];
    v.x += (double)(odd ? b : a);
    v.y += (double)(odd ? a : b);
    reinterpret_cast<double2*>(p)[q] = v;
  }
}

template <int W, int KZ>
cudaError_t point_w(const Geom<float>& g, float* own, const float* oth, const float* r, float om, int c,
                    cudaStream_t s) {
  const long long units = (long long)(g.nx / 2 / W) * g.ny * ((g.nz + KZ - 1) / KZ);
  return launch_dep(k_col_point<W, KZ>, (unsigned)((units + 255) / 256), 256, 0, s, g, own, oth, r, om, c);
}

// z-line variants: columns a thread.  The chunks a column are no variant, since
// they round differently and a solve has to repeat bitwise wherever it is timed:
// 16 where their six levels each are enough, else 32 (us a sweep at 16 / 32: 512 x
// 64 x 64 5.8 / 7.0, 256 x 128 x 96 7.3 / 8.1).
constexpr int kLineWidths[] = {4, 2, 1};
constexpr int kLineLevels = 6;  // levels a chunk at most
int line_chunks(int nz) { return nz <= 16 * kLineLevels ? 16 : 32; }

template <int W, int NCH, int MINB>
cudaError_t line_w(const Geom<float>& g, float* own, const float* oth, const float* r, float om, int c,
                   cudaStream_t s) {
  const unsigned blocks = (unsigned)((g.nx / 2 / W + 7) / 8 * g.ny);
  return launch_dep(k_col_line<W, NCH, kLineLevels, MINB>, blocks, 8 * NCH, 0, s, g, own, oth, r, om, c);
}

// Channels of at least this many cells: the size from which two colours lose on
// no grid measured.  ms a solve to 1e-8, Jacobi / two colours, point sweeps: 64^3
// 1.8 / 1.6, 128 x 64 x 64 2.7 / 1.9, 128 x 64 x 128 5.6 / 4.7, 160 x 96 x 128 11.2 /
// 6.3; above the line 192 x 96 x 128 12.4 / 6.5, 240 x 140 x 120 20.6 / 13.2.  z
// lines: 128 x 64 x 64 4.7 / 4.3, 96 x 80 x 128 6.1 / 6.8, 128 x 64 x 128 6.1 / 6.5,
// 128 x 96 x 128 9.0 / 7.8; above it 192 x 96 x 128 11.1 / 10.3, 256 x 128 x 192 36.2 /
// 29.6.  So z lines cross over near 1.5 x 2^20 cells, while point sweeps gain
// down to 2^18 and lose to the cluster below (32^3, three steps: 2.5 / 3.2).
// The two end equally far from the exact solution on every grid (steps of
// 32^3 to 256 x 128 x 192: errors within 2 % of one another).
constexpr long long kColourCells = 1 << 21;

int col_width(int nx) { return nx % 8 == 0 ? 4 : nx % 4 == 0 ? 2 : 1; }

}  // namespace

bool colour_ok(int nx, int ny, int nz, bool line) {
  return nx % 2 == 0 && ny % 2 == 0 && (!line || nz <= 192) && (long long)nx * ny * nz >= kColourCells;
}

int colour_variants(bool line) { return line ? (int)(sizeof(kLineWidths) / sizeof(int)) : 3; }

// point sweeps: 1, 2 or 4 levels a thread; z-line sweeps: kLineWidths
bool colour_variant_ok(int v, int nx, int nz, bool line) {
  if (v < 0 || v >= colour_variants(line)) return false;
  if (!line) return nz >= (1 << v);
  return nx / 2 % kLineWidths[v] == 0;
}

cudaError_t launch_colour_sweep(const Geom<float>& g, float* d, const float* r, float om, int c, int line, int variant,
                                cudaStream_t s) {
  const size_t half = (size_t)(g.nx / 2) * g.ny * g.nz;
  float* own = d + (c ? half : 0);
  const float *oth = d + (c ? 0 : half), *rc = r + (c ? half : 0);
  if (line) {
    const bool few = line_chunks(g.nz) == 16;
    switch (variant) {
      case 0: return few ? line_w<4, 16, 8>(g, own, oth, rc, om, c, s) : line_w<4, 32, 4>(g, own, oth, rc, om, c, s);
      case 1: return few ? line_w<2, 16, 10>(g, own, oth, rc, om, c, s) : line_w<2, 32, 5>(g, own, oth, rc, om, c, s);
      case 2: return few ? line_w<1, 16, 12>(g, own, oth, rc, om, c, s) : line_w<1, 32, 6>(g, own, oth, rc, om, c, s);
      default: return cudaErrorInvalidValue;
    }
  }
  const int w = col_width(g.nx);
#define POINT(W)                                                   \
  switch (variant) {                                               \
    case 1: return point_w<W, 2>(g, own, oth, rc, om, c, s);       \
    case 2: return point_w<W, 4>(g, own, oth, rc, om, c, s);       \
    default: return point_w<W, 1>(g, own, oth, rc, om, c, s);      \
  }
  if (w == 4) POINT(4)
  if (w == 2) POINT(2)
  POINT(1)
#undef POINT
}

cudaError_t launch_colour_check(const Geom<float>& g, const float* d, const float* r, int line, SolveCtl* ctl, Red red,
                                int graph, cudaGraphConditionalHandle h_loop, cudaGraphConditionalHandle h_body,
                                cudaStream_t s) {
  const int w = col_width(g.nx), zc = line ? 0 : 1;
  const unsigned blocks = (unsigned)(((long long)(g.nx / 2 / w) * g.ny * g.nz + 255) / 256);
  if (w == 4) k_col_check<4><<<blocks, 256, 0, s>>>(g, d, r, zc, ctl, red, blocks, graph, h_loop, h_body);
  else if (w == 2) k_col_check<2><<<blocks, 256, 0, s>>>(g, d, r, zc, ctl, red, blocks, graph, h_loop, h_body);
  else k_col_check<1><<<blocks, 256, 0, s>>>(g, d, r, zc, ctl, red, blocks, graph, h_loop, h_body);
  return cudaGetLastError();
}

cudaError_t launch_colour_outer(const Geom<double>& g, const double* p, const double* b, float* r32, int line,
                                SolveCtl* ctl, Red red, int after_pass, int graph, cudaGraphConditionalHandle h_loop,
                                cudaStream_t s) {
  Launch l = plane_launch(g.nx, g.ny, g.nz);
  k_col_outer<<<l.grid, l.block, 0, s>>>(g, p, b, r32, line ? 0 : 1, ctl, red, l.nblocks, after_pass, graph, h_loop);
  return cudaGetLastError();
}

cudaError_t launch_colour_addcorr(const Geom<double>& g, double* p, const float* d, int line, cudaStream_t s) {
  const long long n = (long long)(g.nx / 2) * g.ny * g.nz;
  const unsigned blocks = (unsigned)std::min<long long>((n + 255) / 256, 152 * 16);
  k_col_addcorr<<<blocks, 256, 0, s>>>(p, d, g.nx / 2, g.ny, g.nz, line ? 0 : 1);
  return cudaGetLastError();
}

}  // namespace stp
