// A whole SRJ cycle of FP32 point sweeps in one launch, on one thread-block
// cluster, for channels that fit its shared memory.
//
// A launched sweep of a small channel costs a launch (1.6 us at 32^3, where
// its loads and arithmetic are a tenth of that).  Here the channel is cut
// into slabs of levels or of rows, one a block; the iterate lives in shared
// memory in two buffers, each slab with one ghost slab on either side, and
// the right-hand side in registers.  In a sweep every thread relaxes its
// columns of its block's slabs (from one buffer into the other) and stores
// the boundary slabs also into the neighbours' ghost slabs (distributed
// shared memory); a cluster barrier ends the sweep.  The cell update is the
// one of every FP32 Jacobi sweep (srj_cell_f32), so the result is bitwise
// that of M launched sweeps.
#include <cooperative_groups.h>

#include <algorithm>

#include "device_util.cuh"
#include "poisson_common.cuh"
#include "stp_internal.cuh"

namespace cg = cooperative_groups;

namespace stp {
namespace {

constexpr int kClusterSmem = 227 * 1024;
constexpr int kClusterM = 4096;  // longest cycle stp_init takes

template <int W>
struct F {
  float v[W];
};
template <int W>
__device__ __forceinline__ F<W> ld(const float* p) {
  F<W> r;
  if constexpr (W == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    r.v[0] = t.x, r.v[1] = t.y, r.v[2] = t.z, r.v[3] = t.w;
  } else {
    const float2 t = *reinterpret_cast<const float2*>(p);
    r.v[0] = t.x, r.v[1] = t.y;
  }
  return r;
}
template <int W>
__device__ __forceinline__ void st(float* p, const F<W>& r) {
  if constexpr (W == 4)
    *reinterpret_cast<float4*>(p) = make_float4(r.v[0], r.v[1], r.v[2], r.v[3]);
  else
    *reinterpret_cast<float2*>(p) = make_float2(r.v[0], r.v[1]);
}

// threads a block at most: the right-hand side takes W L NC registers a thread
__host__ __device__ constexpr int cluster_threads(int W, int L, int NC) { return W * L * NC <= 20 ? 1024 : 512; }

// AX 0: slabs of levels (z), rows inside a slab periodic; AX 1: slabs of
// rows (y, periodic), levels inside a slab between the walls.  W cells a
// vector, at most L slabs a block, NC columns (a vector through all the
// block's slabs) a thread.
template <int W, int L, int NC, int AX>
__global__ void __launch_bounds__(cluster_threads(W, L, NC), 1)
    k_cluster_cycle(Geom<float> g, float* __restrict__ d, const float* __restrict__ rhs,
                    const float* __restrict__ omega, int M) {
  extern __shared__ __align__(16) float csm[];
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int nx = g.nx, ny = g.ny, nz = g.nz, uw = nx / W;
  const int S = AX ? ny : nz, N = AX ? nz : ny;  // slabs, rows a slab
  const int s0 = rank * S / C, Lc = (rank + 1) * S / C - s0;
  const int slab = N * nx;  // cells of a slab
  const int cols = N * uw, T = blockDim.x, lane = threadIdx.x & 31;
  // level coefficients and the schedule first: a cluster barrier drops cached
  // global data, so a sweep that read them there would wait for L2
  float4* coef = reinterpret_cast<float4*>(csm);  // [nz] cup, cdn, 1/S
  float* oms = csm + 4 * nz;                      // [M, padded to 4]
  float* buf0 = oms + ((M + 3) & ~3);
  const int bstride = ((S + C - 1) / C + 2) * slab;
  for (int k = threadIdx.x; k < nz; k += T) coef[k] = make_float4(g.cup[k], g.cdn[k], g.iS[k], 0.f);
  for (int m = threadIdx.x; m < M; m += T) oms[m] = omega[m];
  // ghost slabs in the neighbours: mine below their slot 0, above their last + 1
  const int up = rank == C - 1 ? 0 : rank + 1, dn = rank == 0 ? C - 1 : rank - 1;
  const bool has_up = AX || rank < C - 1, has_dn = AX || rank > 0;
  const int dn_slot = (dn + 1) * S / C - dn * S / C + 1;
  // global offset of slab s (0 .. S-1), row q, in cells
  auto goff = [&](int s, int q) -> size_t {
    return AX ? ((size_t)q * ny + s) * nx : ((size_t)s * ny + q) * nx;
  };
  int q_[NC], x_[NC];
  bool act[NC];
  F<W> b[NC][L];
#pragma unroll
  for (int n = 0; n < NC; n++) {
    const int col = threadIdx.x + n * T;
    act[n] = col < cols;
    const int cc = act[n] ? col : cols - 1;
    q_[n] = cc / uw;
    x_[n] = (cc - q_[n] * uw) * W;
#pragma unroll
    for (int l = 0; l < L; l++)
      if (l < Lc) b[n][l] = ld<W>(rhs + goff(s0 + l, q_[n]) + x_[n]);
    if (act[n]) {
      for (int l = 0; l <= Lc + 1; l++) {
        int s = s0 + l - 1;
        if (AX) s = s < 0 ? S - 1 : s >= S ? 0 : s;
        if (s >= 0 && s < S) st<W>(buf0 + l * slab + q_[n] * nx + x_[n], ld<W>(d + goff(s, q_[n]) + x_[n]));
      }
    }
  }
  const float idx2 = g.idx2, idy2 = g.idy2;
  cl.sync();
  for (int m = 0; m < M; m++) {
    const float* src = buf0 + (m & 1 ? bstride : 0);
    float* dst = buf0 + (m & 1 ? 0 : bstride);
    const float om = oms[m];
    float* dst_up = has_up ? cl.map_shared_rank(dst, up) : nullptr;
    float* dst_dn = has_dn ? cl.map_shared_rank(dst, dn) + dn_slot * slab : nullptr;
#pragma unroll
    for (int n = 0; n < NC; n++) {
      const int o = q_[n] * nx + x_[n], q = q_[n];
      const bool rlast = q == N - 1, rfirst = q == 0;
      const int on = rlast ? (AX ? o : o - (N - 1) * nx) : o + nx;  // next row inside the slab
      const int op = rfirst ? (AX ? o : o + (N - 1) * nx) : o - nx;
      const bool xl_out = lane == 0 || x_[n] == 0, xr_out = lane == 31 || x_[n] == nx - W;
      const int xl = q * nx + (x_[n] == 0 ? nx - 1 : x_[n] - 1), xr = q * nx + (x_[n] == nx - W ? 0 : x_[n] + W);
      const bool bottom = !AX && s0 == 0, top = !AX && s0 + Lc == S;
      F<W> cur = ld<W>(src + slab + o);
      F<W> prev = bottom ? cur : ld<W>(src + o);
#pragma unroll
      for (int l = 0; l < L; l++) {
        if (l < Lc) {
          const float* row = src + (l + 1) * slab;
          const int k = AX ? q : s0 + l;
          const float4 cf = coef[k];
          const float cup = cf.x, cdn = cf.y, iS = cf.z;
          const F<W> next = (top && l == Lc - 1) ? cur : ld<W>(row + slab + o);
          const F<W> rn = ld<W>(row + on), rp = ld<W>(row + op);
          float left = __shfl_up_sync(0xffffffffu, cur.v[W - 1], 1);
          float right = __shfl_down_sync(0xffffffffu, cur.v[0], 1);
          if (xl_out) left = row[xl];
          if (xr_out) right = row[xr];
          F<W> out;
#pragma unroll
          for (int e = 0; e < W; e++) {
            const float lv = e == 0 ? left : cur.v[e - 1], rv = e == W - 1 ? right : cur.v[e + 1];
            // AX 0: rows are y, slabs z; AX 1: rows z (at a wall the cell itself), slabs y
            out.v[e] = AX ? srj_cell_f32(cur.v[e], lv, rv, next.v[e], prev.v[e], rn.v[e], rp.v[e], b[n][l].v[e], idx2,
                                         idy2, cup, cdn, iS, om)
                          : srj_cell_f32(cur.v[e], lv, rv, rn.v[e], rp.v[e], next.v[e], prev.v[e], b[n][l].v[e], idx2,
                                         idy2, cup, cdn, iS, om);
          }
          if (act[n]) {
            st<W>(dst + (l + 1) * slab + o, out);
            if (l == 0 && has_dn) st<W>(dst_dn + o, out);
            if (l == Lc - 1 && has_up) st<W>(dst_up + o, out);
          }
          prev = cur;
          cur = next;
        }
      }
    }
    cl.sync();
  }
  const float* fin = buf0 + (M & 1 ? bstride : 0);
#pragma unroll
  for (int n = 0; n < NC; n++)
    if (act[n])
      for (int l = 0; l < Lc; l++)
        st<W>(d + goff(s0 + l, q_[n]) + x_[n], ld<W>(fin + (l + 1) * slab + q_[n] * nx + x_[n]));
}

struct Plan {
  int W, L, NC, threads;
  size_t smem;
};

// how a channel runs on C blocks cut along AX; false if it does not fit
bool plan(int nx, int ny, int nz, int C, int ax, int M, Plan* p) {
  const int S = ax ? ny : nz, N = ax ? nz : ny;
  p->W = nx % 4 == 0 ? 4 : nx % 2 == 0 ? 2 : 0;
  if (p->W == 0 || S < C) return false;
  const int lmax = (S + C - 1) / C;
  p->L = lmax <= 2 ? 2 : lmax <= 4 ? 4 : lmax <= 6 ? 6 : lmax <= 8 ? 8 : 0;
  if (p->L == 0) return false;
  const int cols = N * (nx / p->W);
  p->NC = 1;
  if (cols > cluster_threads(p->W, p->L, 1)) p->NC = 2;
  if (cols > 2 * cluster_threads(p->W, p->L, 2)) return false;
  if (p->W * p->L * p->NC > 48) return false;  // registers
  p->threads = ((cols + p->NC - 1) / p->NC + 31) / 32 * 32;
  p->smem = sizeof(float) * (2 * (size_t)(lmax + 2) * N * nx + 4 * (size_t)nz + ((M + 3) & ~3));
  return p->smem <= (size_t)kClusterSmem;
}

template <int W, int L, int NC, int AX>
cudaError_t go(const Geom<float>& g, float* d, const float* r, const float* omega, int M, int C, const Plan& p,
               cudaStream_t s) {
  auto kern = k_cluster_cycle<W, L, NC, AX>;
  static std::atomic<unsigned> done{0u}, done16{0u};
  cudaError_t e = smem_limit_once(kern, kClusterSmem, done);
  if (e != cudaSuccess) return e;
  {
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    const unsigned bit = 1u << (dev & 31);
    if (!(done16.load(std::memory_order_acquire) & bit)) {
      if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess) return e;
      done16.fetch_or(bit, std::memory_order_acq_rel);
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)C);
  cfg.blockDim = dim3((unsigned)p.threads);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, g, d, r, omega, M);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int W, int L, int NC>
cudaError_t go_ax(const Geom<float>& g, float* d, const float* r, const float* omega, int M, int C, int ax,
                  const Plan& p, cudaStream_t s) {
  return ax ? go<W, L, NC, 1>(g, d, r, omega, M, C, p, s) : go<W, L, NC, 0>(g, d, r, omega, M, C, p, s);
}
template <int W, int L>
cudaError_t go_nc(const Geom<float>& g, float* d, const float* r, const float* omega, int M, int C, int ax,
                  const Plan& p, cudaStream_t s) {
  return p.NC == 1 ? go_ax<W, L, 1>(g, d, r, omega, M, C, ax, p, s) : go_ax<W, L, 2>(g, d, r, omega, M, C, ax, p, s);
}
template <int W>
cudaError_t go_l(const Geom<float>& g, float* d, const float* r, const float* omega, int M, int C, int ax,
                 const Plan& p, cudaStream_t s) {
  switch (p.L) {
    case 2: return go_nc<W, 2>(g, d, r, omega, M, C, ax, p, s);
    case 4: return go_nc<W, 4>(g, d, r, omega, M, C, ax, p, s);
    case 6: return go_nc<W, 6>(g, d, r, omega, M, C, ax, p, s);
    default: return go_ax<W, 8, 1>(g, d, r, omega, M, C, ax, p, s);
  }
}

}  // namespace

// cluster variants: 0 .. 3 = (16 blocks, z slabs), (16, y), (8, z), (8, y)
int cluster_variants() { return 4; }
bool cluster_ok(int v, int nx, int ny, int nz) {
  Plan p;
  if (v < 0 || v >= 4 || !plan(nx, ny, nz, v < 2 ? 16 : 8, v & 1, kClusterM, &p)) return false;
  return p.L < 8 || p.NC == 1;
}
cudaError_t launch_cluster_cycle(const Geom<float>& g, float* d, const float* r, const float* omega, int M, int v,
                                 cudaStream_t s) {
  Plan p;
  const int C = v < 2 ? 16 : 8;
  if (!cluster_ok(v, g.nx, g.ny, g.nz) || !plan(g.nx, g.ny, g.nz, C, v & 1, M, &p) || M > kClusterM) return cudaErrorInvalidValue;
  return p.W == 4 ? go_l<4>(g, d, r, omega, M, C, v & 1, p, s) : go_l<2>(g, d, r, omega, M, C, v & 1, p, s);
}

}  // namespace stp
