// FP64 sweeps of the pressure solve (Sec. 3.4).  GB300 issues two FP64
// operations a clock and SM, a warp's instruction taking 16 clocks whatever
// its active lanes: these kernels are bound by the FP64 operations a cell and
// by lanes that idle, so a thread takes one cell (full warps on any row
// length; loads and index arithmetic hide behind the FP64 pipe) and every
// product of coefficients is formed beforehand.
#include <algorithm>

#include "device_util.cuh"
#include "stp_internal.cuh"

namespace stp {
namespace {

// tab[(m nz + k) 5 ..]: omega_m/S_k times 1/dx^2, 1/dy^2, cup_k, cdn_k, 1
__global__ void k_sweep_table(Geom<double> g, const double* __restrict__ omega, int M, double* __restrict__ tab) {
  const long long n = (long long)M * g.nz;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
    const int m = (int)(q / g.nz), k = (int)(q - (long long)m * g.nz);
    const double w = omega[m] * g.iS[k];
    double* t = tab + 5 * q;
    t[0] = w * g.idx2;
    t[1] = w * g.idy2;
    t[2] = w * g.cup[k];
    t[3] = w * g.cdn[k];
    t[4] = w;
  }
}

// One Jacobi-SOR sweep: p + omega (p^J - p) with p^J = (sum_nb c p_nb - b)/S,
// as (1 - omega) p + sum_nb (omega c/S) p_nb - (omega/S) b: eight FP64
// operations a cell (ten with the coefficients applied one by one).  om1 =
// 1 - omega.  Without a table (TAB false) a thread forms the coefficients; both
// in one kernel would cost their predicated multiplications either way.
// us a sweep, ten operations on double2 units / this: 128 x 64 x 128 19.2 /
// 16.5 (505 Gop/s of the 500-545 the FP64 pipe gives), 112 x 56 x 112 15.4 /
// 11.5, 64^3 6.5 / 5.2, 32 x 16 x 32 2.78 / 1.76 (its rows left half a warp of
// double2 units idle).  Two cells a thread at eight operations: 16.6, 13.2,
// 5.5, 2.25.
template <bool TAB>
__global__ void __launch_bounds__(128) k_sweep_f64(Geom<double> g, const double* __restrict__ p,
                                                    const double* __restrict__ b, double omega,
                                                    double om1, const double* __restrict__ tab,
                                                    double* __restrict__ out) {
  const unsigned nx = g.nx, ny = g.ny, nz = g.nz, plane = nx * ny;
  const unsigned q = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned row = q / nx, i = q - row * nx, k = row / ny, j = row - k * ny;
  const bool act = k < nz;
  double ax = 0, ay = 0, au = 0, ad = 0, ab = 0;
  if (act) {
    if constexpr (TAB) {
      ax = __ldg(tab + 5 * k), ay = __ldg(tab + 5 * k + 1), au = __ldg(tab + 5 * k + 2);
      ad = __ldg(tab + 5 * k + 3), ab = __ldg(tab + 5 * k + 4);
    } else {
      ab = omega * __ldg(g.iS + k);
      ax = ab * g.idx2, ay = ab * g.idy2, au = ab * __ldg(g.cup + k), ad = ab * __ldg(g.cdn + k);
    }
  }
  cudaGridDependencySynchronize();
  if (!act) return;
  const double pc = __ldg(p + q);
  const double e = __ldg(p + (i + 1 == nx ? q + 1 - nx : q + 1)), w = __ldg(p + (i == 0 ? q + nx - 1 : q - 1));
  const double n = __ldg(p + (j + 1 == ny ? q + nx - plane : q + nx)), s = __ldg(p + (j == 0 ? q + plane - nx : q - nx));
  const double u = k + 1 < nz ? __ldg(p + q + plane) : pc, d = k > 0 ? __ldg(p + q - plane) : pc;  // coefficient 0 there
  double t = ax * (e + w);
  t = fma(ay, n + s, t);
  t = fma(au, u, t);
  t = fma(ad, d, t);
  t = fma(-ab, __ldg(b + q), t);
  out[q] = fma(om1, pc, t);
}

// One z-line Jacobi-SOR sweep, p' = p + omega (p^L - p), the columns solved in
// registers in level chunks as in k_line_sweep_chunk (kernels_poisson.cu).  A
// block takes CW columns of a row x NCH chunks of at most LMAX levels.  The right-hand side is that of the line value itself,
//   A p^L = (p_{i+1} + p_{i-1})/dx^2 + (p_{j+1} + p_{j-1})/dy^2 - b,
// six FP64 operations a cell with the pivot (thirteen for A^-1 (b - L p)), and
// the running products of the chunk's coefficients come from tables (pf, pe),
// so that a cell costs twelve FP64 operations in all.  Every chunk a carry
// passes is another multiply-add, so the chunks are long (line_f64_chunks);
// LMAX is the least even bound of their levels, because a predicated
// operation past the chunk's end takes its slot on the FP64 pipe all the same.
template <int CW, int NCH, int LMAX>
__global__ void __launch_bounds__(CW * NCH) k_line_f64(Geom<double> g, const double* __restrict__ p,
                                                       const double* __restrict__ b, double omega,
                                                       double* __restrict__ out) {
  constexpr int H = NCH / 2;
  __shared__ double ZB[NCH][CW], WB[NCH][CW], XT[CW];
  const int nx = g.nx, ny = g.ny, nz = g.nz, t = nz >> 1;
  const int u = threadIdx.x % CW, c = threadIdx.x / CW;
  const int nxb = (nx + CW - 1) / CW, j = blockIdx.x / nxb, i0 = (blockIdx.x % nxb) * CW + u;
  const bool act = i0 < nx;
  const int i = act ? i0 : nx - 1;
  const unsigned plane = (unsigned)nx * ny, rc = (unsigned)j * nx + i;
  const unsigned xe = (unsigned)j * nx + (i + 1 == nx ? 0 : i + 1), xw = (unsigned)j * nx + (i == 0 ? nx - 1 : i - 1);
  const unsigned yn = (unsigned)(j + 1 == ny ? 0 : j + 1) * nx + i, ys = (unsigned)(j == 0 ? ny - 1 : j - 1) * nx + i;
  const bool lower = c < H;
  const int k0 = line_chunk_start(c, NCH, nz), k1 = line_chunk_start(c + 1, NCH, nz), L = k1 - k0;
  const bool twist = c == H;
  // the first level that the elimination and the substitution run over
  const int q0 = twist ? 1 : 0;
  double G[LMAX];
  const double idx2 = g.idx2, idy2 = g.idy2;
  cudaGridDependencySynchronize();
#pragma unroll
  for (int q = 0; q < LMAX; q++)
    if (q < L) {
      const unsigned lev = (unsigned)(k0 + q) * plane;
      double r = idx2 * (__ldg(p + lev + xe) + __ldg(p + lev + xw));
      r = fma(idy2, __ldg(p + lev + yn) + __ldg(p + lev + ys), r) - __ldg(b + lev + rc);
      G[q] = r * __ldg(g.tli + k0 + q);
    }
  // elimination inside the chunk: upward below t, downward above it
  if (lower) {
    double z = 0.0;
#pragma unroll
    for (int q = 0; q < LMAX; q++)
      if (q < L) G[q] = z = fma(__ldg(g.tlf + k0 + q), z, G[q]);
    ZB[c][u] = z;
  } else {
    double z = 0.0;
#pragma unroll
    for (int q = LMAX - 1; q >= 0; q--)
      if (q < L && q >= q0) G[q] = z = fma(__ldg(g.tlf + k0 + q), z, G[q]);
    ZB[c][u] = z;
  }
  __syncthreads();
  // the value entering the chunk, from the walls
  {
    double carry = 0.0;
    if (lower) {
      for (int cc = 0; cc < c; cc++) {
        const int e = line_chunk_start(cc + 1, NCH, nz);
        if (e > line_chunk_start(cc, NCH, nz)) carry = fma(__ldg(g.pf + e - 1), carry, ZB[cc][u]);
      }
    } else {
      for (int cc = NCH - 1; cc > c; cc--) {
        const int e = line_chunk_start(cc, NCH, nz);
        if (e < line_chunk_start(cc + 1, NCH, nz)) carry = fma(__ldg(g.pf + e), carry, ZB[cc][u]);
      }
    }
#pragma unroll
    for (int q = 0; q < LMAX; q++)
      if (q < L && q >= q0) G[q] = fma(__ldg(g.pf + k0 + q), carry, G[q]);
    if (twist) {
      double ylow = 0.0;  // y_{t-1}
      for (int cc = 0; cc < H; cc++) {
        const int e = line_chunk_start(cc + 1, NCH, nz);
        if (e > line_chunk_start(cc, NCH, nz)) ylow = fma(__ldg(g.pf + e - 1), ylow, ZB[cc][u]);
      }
      const double yup = L >= 2 ? G[1] : carry;  // y_{t+1}
      const double ft = t > 0 ? __ldg(g.tlf + t) : 0.0, et = t < nz - 1 ? __ldg(g.tlb + t) : 0.0;
      G[0] = fma(et, yup, fma(ft, ylow, G[0]));
      XT[u] = G[0];
    }
  }
  // substitution inside the chunk: downward below t, upward above it (the
  // twist chunk starts from x_t itself)
  {
    double w = twist ? G[0] : 0.0;
    if (lower) {
#pragma unroll
      for (int q = LMAX - 1; q >= 0; q--)
        if (q < L) G[q] = w = fma(__ldg(g.tlb + k0 + q), w, G[q]);
    } else {
#pragma unroll
      for (int q = 0; q < LMAX; q++)
        if (q < L && q >= q0) G[q] = w = fma(__ldg(g.tlb + k0 + q), w, G[q]);
    }
    WB[c][u] = w;
  }
  __syncthreads();
  {
    double carry = XT[u];
    if (lower) {
      for (int cc = H - 1; cc > c; cc--) {
        const int e = line_chunk_start(cc, NCH, nz);
        if (e < line_chunk_start(cc + 1, NCH, nz)) carry = fma(__ldg(g.pe + e), carry, WB[cc][u]);
      }
    } else if (!twist) {
      carry = WB[H][u];
      for (int cc = H + 1; cc < c; cc++) {
        const int e = line_chunk_start(cc + 1, NCH, nz);
        if (e > line_chunk_start(cc, NCH, nz)) carry = fma(__ldg(g.pe + e - 1), carry, WB[cc][u]);
      }
    }
    if (!twist) {
#pragma unroll
      for (int q = 0; q < LMAX; q++)
        if (q < L) G[q] = fma(__ldg(g.pe + k0 + q), carry, G[q]);
    }
    if (act) {
#pragma unroll
      for (int q = 0; q < LMAX; q++)
        if (q < L) {
          const unsigned a = (unsigned)(k0 + q) * plane + rc;
          const double pv = __ldg(p + a);
          out[a] = fma(omega, G[q] - pv, pv);
        }
    }
  }
}

template <typename... P, typename... A>
cudaError_t launch_dep(void (*kern)(P...), dim3 grid, dim3 block, cudaStream_t s, A... a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, a...);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t launch_sweep_table(const Geom<double>& g, const double* omega, int M, double* tab, cudaStream_t s) {
  k_sweep_table<<<(unsigned)std::min<long long>(((long long)M * g.nz + 255) / 256, 1216), 256, 0, s>>>(g, omega, M, tab);
  return cudaGetLastError();
}

cudaError_t launch_sweep_f64(const Geom<double>& g, const double* p, const double* b, double omega, const double* tab,
                             double* out, cudaStream_t s) {
  const unsigned n = (unsigned)g.nx * g.ny * g.nz;
  const double om1 = 1.0 - omega;
  return launch_dep(tab ? k_sweep_f64<true> : k_sweep_f64<false>, dim3((n + 127) / 128), dim3(128), s, g, p, b, omega,
                    om1, tab, out);
}

namespace {
// Columns a block.  us a sweep at 32 / 16 / 8: 96 x 48 x 64 10.9 / 11.1 / 11.5,
// 64 x 30 x 100 18.8 / 13.8 / 14.1, 112 x 56 x 112 28.6 / 22.5 / 23.5, 32 x 16
// x 32 7.3 / 6.5 / 6.4 (the lock-step shared-memory kernel: 41.2, 35.2, 39.1,
// 21.7): 32 leave SMs without a block or a last wave nearly empty.
constexpr int kLineCols = 16;

template <int NCH>
cudaError_t line_nch(const Geom<double>& g, const double* p, const double* b, double omega, double* out, cudaStream_t s) {
  const dim3 blocks((unsigned)(((g.nx + kLineCols - 1) / kLineCols) * g.ny)), threads(kLineCols * NCH);
  switch ((line_f64_levels(g.nz, NCH) + 1) / 2) {
    case 1: return launch_dep(k_line_f64<kLineCols, NCH, 2>, blocks, threads, s, g, p, b, omega, out);
    case 2: return launch_dep(k_line_f64<kLineCols, NCH, 4>, blocks, threads, s, g, p, b, omega, out);
    case 3: return launch_dep(k_line_f64<kLineCols, NCH, 6>, blocks, threads, s, g, p, b, omega, out);
    case 4: return launch_dep(k_line_f64<kLineCols, NCH, 8>, blocks, threads, s, g, p, b, omega, out);
    case 5: return launch_dep(k_line_f64<kLineCols, NCH, 10>, blocks, threads, s, g, p, b, omega, out);
    case 6: return launch_dep(k_line_f64<kLineCols, NCH, 12>, blocks, threads, s, g, p, b, omega, out);
    default: return cudaErrorInvalidValue;
  }
}
}  // namespace

cudaError_t launch_line_f64(const Geom<double>& g, const double* p, const double* b, double omega, double* out,
                            cudaStream_t s) {
  switch (line_f64_chunks(g.nx, g.ny, g.nz)) {
    case 4: return line_nch<4>(g, p, b, omega, out, s);
    case 8: return line_nch<8>(g, p, b, omega, out, s);
    case 16: return line_nch<16>(g, p, b, omega, out, s);
    case 32: return line_nch<32>(g, p, b, omega, out, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace stp
