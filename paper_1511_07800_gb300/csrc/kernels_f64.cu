// FP64 sweeps of the pressure solve (Sec. 3.4).  GB300 issues two FP64
// operations a clock and SM, a warp's instruction taking 16 clocks whatever
// its active lanes: these kernels are bound by the FP64 operations a cell and
// by lanes that idle, so a thread takes one cell (full warps on any row
// length; loads and index arithmetic hide behind the FP64 pipe) and every
// product of coefficients is formed beforehand.
#include <algorithm>

#include "device_util.cuh"
#include "poisson_common.cuh"
#include "stp_internal.cuh"

namespace stp {
namespace {

// tab[(m nz + k) 6 ..]: omega_m/S_k times 1/dx^2, 1/dy^2, cup_k, cdn_k, 1, and
// 1 - omega_m as 1 less the six neighbours' coefficients as rounded, so that a
// sweep keeps a constant
__global__ void k_sweep_table(Geom<double> g, const double* __restrict__ omega, int M, double* __restrict__ tab) {
  const long long n = (long long)M * g.nz;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
    const int m = (int)(q / g.nz), k = (int)(q - (long long)m * g.nz);
    const double w = omega[m] * g.iS[k];
    double* t = tab + 6 * q;
    t[0] = w * g.idx2;
    t[1] = w * g.idy2;
    t[2] = w * g.cup[k];
    t[3] = w * g.cdn[k];
    t[4] = w;
    double hi = 1.0, lo = 0.0;
    for (int i = 0; i < 4; i++) {
      const double a = i < 2 ? -2.0 * t[i] : -t[i], s = hi + a, z = s - hi;
      lo += (hi - (s - z)) + (a - z);
      hi = s;
    }
    t[5] = hi + lo;
  }
}

// One Jacobi-SOR sweep: p + omega (p^J - p) with p^J = (sum_nb c p_nb - b)/S,
// as (1 - omega) p + sum_nb (omega c/S) p_nb - (omega/S) b: eight FP64
// operations a cell (ten with the coefficients applied one by one).  The
// right-hand side comes first and the z couplings, largest next to stretched
// walls, last: every rounding is of a partial sum, and these stay small the
// longest.  The table's coefficient of p makes the coefficients of p and its
// neighbours sum to one as they are rounded.  Without both, solves stall 1.15
// times higher than with ten operations (1.3 to 1.5 at stretch 3), with them no
// higher.  Without a table (TAB false) a thread forms the coefficients, that of p
// as om1 = 1 - omega; both in one kernel would cost their predicated
// multiplications either way.
// us a sweep, ten operations on double2 units / this: 128 x 64 x 128 19.2 /
// 16.3 (505 Gop/s of the 500-545 the FP64 pipe gives), 112 x 56 x 112 15.4 /
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
  double ax = 0, ay = 0, au = 0, ad = 0, ab = 0, ac = om1;
  if (act) {
    if constexpr (TAB) {
      const double2* c = reinterpret_cast<const double2*>(tab) + 3 * k;
      const double2 c0 = __ldg(c), c1 = __ldg(c + 1), c2 = __ldg(c + 2);
      ax = c0.x, ay = c0.y, au = c1.x, ad = c1.y, ab = c2.x, ac = c2.y;
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
  double t = -ab * __ldg(b + q);
  t = fma(ax, e + w, t);
  t = fma(ay, n + s, t);
  t = fma(au, u, t);
  t = fma(ad, d, t);
  out[q] = fma(ac, pc, t);
}

// r = b - L p in differences of neighbours
__global__ void __launch_bounds__(kBX* kBY) k_residual_f64(Geom<double> g, const double* __restrict__ p,
                                                            const double* __restrict__ b, double* __restrict__ r) {
  const int i = blockIdx.x * kBX + threadIdx.x, j = blockIdx.y * kBY + threadIdx.y, k = blockIdx.z;
  if (i >= g.nx || j >= g.ny) return;
  double pc;
  r[at(g.nx, g.ny, i, j, k)] = point_residual(g, p, b, i, j, k, &pc);
}

// One z-line Jacobi-SOR sweep d' = d + omega (d^L - d) of L d = r, the columns
// solved in registers in level chunks as in k_line_sweep_chunk
// (kernels_poisson.cu).  A block takes CW columns of a row x NCH chunks of at most
// LMAX levels.
//
// The sweeps of a cycle run on the correction d to the pressure the cycle starts
// from, r being its residual: the line value's own equation A d^L = (sum of the
// x and y neighbours) - r takes four operations a cell where A^-1 (r - L d)
// takes ten, and what it rounds is of the size of S d, which vanishes as the solve
// converges: a solve of a smooth field on 64 x 32 x 192 at stretch 2 stalls at
// 4.0e-13 of ||b||; with the same sweeps on the pressure itself, which round with
// S p, at 1.0e-11, in residual form at 4.3e-12.  The cycle's
// first sweep has d = 0 (d null) and its last adds d to the pressure (base:
// written in place of out).
//
// The elimination runs on undivided values (Geom::lf, lb), so that the pivot
// joins omega in one coefficient a level: ten operations a cell (twelve on the
// pressure, fifteen in residual form).  us a sweep, on the pressure with every
// thread walking its own carries / in residual form / this: 32 x 16 x 32 6.3 /
// 5.5 / 4.4, 96 x 48 x 64 11.1 / 11.4 / 8.6, 64 x 30 x 100 13.9 / 11.4 / 9.0, 64 x 32
// x 192 18.1 / 16.9 / 12.5, 112 x 56 x 112 22.4 / 25.1 / 17.7, 128 x 64 x 128 31.6 /
// 38.2 / 27.7 (of which 512 blocks on 152 SMs leave a fifth idle); the lock-step
// kernel took 41.2 at 96 x 48 x 64.  A thread
// counts its levels from the wall's side of the chunk to the twist level's, so
// both sides run the same code.  What enters a chunk is walked chunk by chunk by
// one warp, a lane a column and side (by every thread for itself it took as many
// operations as the columns' own recurrences).  Chunks stay long
// (line_f64_chunks): each is a step of that walk.  LMAX is the most levels a
// chunk has, no more, because an operation past the chunk's end takes its slot
// on the FP64 pipe all the same.
template <int CW, int NCH, int LMAX>
__global__ void __launch_bounds__(CW * NCH) k_line_f64(Geom<double> g, const double* __restrict__ d,
                                                       const double* __restrict__ r, double omega, double om1,
                                                       double* __restrict__ out, double* __restrict__ base) {
  constexpr int H = NCH / 2;
  static_assert(CW == 16 && H % 2 == 0, "a warp holds two chunks of one side");
  extern __shared__ double wt[];  // [nz] omega / pivot
  __shared__ double EB[NCH][CW], CB[NCH][CW], YL[CW], XT[CW], PF[NCH], PE[NCH];
  const int nx = g.nx, ny = g.ny, nz = g.nz, t = nz >> 1;
  const int u = threadIdx.x % CW, c = threadIdx.x / CW, half = threadIdx.x & CW;
  const int nxb = (nx + CW - 1) / CW, j = blockIdx.x / nxb, i0 = (blockIdx.x % nxb) * CW + u;
  const bool act = i0 < nx;
  const int i = act ? i0 : nx - 1;
  const unsigned plane = (unsigned)nx * ny, row = (unsigned)j * nx, rc = row + i;
  const unsigned xe = row + (i + 1 == nx ? 0 : i + 1), xw = row + (i == 0 ? nx - 1 : i - 1);
  const unsigned yn = (unsigned)(j + 1 == ny ? 0 : j + 1) * nx + i, ys = (unsigned)(j == 0 ? ny - 1 : j - 1) * nx + i;
  const bool lower = c < H;
  int k0, k1;
  line_chunk_levels<NCH>(c, nz, k0, k1);
  const int L = k1 - k0;
  const bool twist = c == H;  // holds the twist level t = k0, its last; it has LMAX levels
  const int Le = twist ? LMAX - 1 : L;  // levels the elimination runs over
  auto level = [&](int q) { return lower ? k0 + q : k1 - 1 - q; };
  for (int k = threadIdx.x; k < nz; k += CW * NCH) wt[k] = omega * __ldg(g.tli + k);
  if (u == 0) {
    PF[c] = L > 0 ? __ldg(g.pf + level(L - 1)) : 1.0;
    PE[c] = L > 0 ? __ldg(g.pe + level(0)) : 1.0;
  }
  double C[LMAX], G[LMAX];
  const double idx2 = g.idx2, idy2 = g.idy2;
  cudaGridDependencySynchronize();
  if (d) {
#pragma unroll
    for (int q = 0; q < LMAX; q++)
      if (q < L) {
        const unsigned l = (unsigned)level(q) * plane;
        C[q] = __ldg(d + l + rc);
        double v = fma(idx2, __ldg(d + l + xe) + __ldg(d + l + xw), -__ldg(r + l + rc));
        G[q] = fma(idy2, __ldg(d + l + yn) + __ldg(d + l + ys), v);
      }
  } else {
#pragma unroll
    for (int q = 0; q < LMAX; q++)
      if (q < L) {
        C[q] = 0.0;
        G[q] = -__ldg(r + (unsigned)level(q) * plane + rc);
      }
  }
  // elimination inside the chunk
  {
    double z = 0 < Le ? G[0] : 0.0;
#pragma unroll
    for (int q = 1; q < LMAX; q++)
      if (q < Le) G[q] = z = fma(__ldg(g.lf + level(q)), z, G[q]);
    EB[c][u] = z;
  }
  __syncthreads();
  // the values entering the chunks, from the walls; the last one from below
  // enters the twist level
  if (threadIdx.x < 32) {
    double carry = 0.0;
#pragma unroll
    for (int s = 0; s < H; s++) {
      const int cc = half ? NCH - 1 - s : s;
      CB[cc][u] = carry;
      carry = fma(PF[cc], carry, EB[cc][u]);
    }
    if (!half) YL[u] = carry;
  }
  __syncthreads();
  {
    const double carry = CB[c][u];
#pragma unroll
    for (int q = 0; q < LMAX; q++)
      if (q < Le) G[q] = fma(__ldg(g.pf + level(q)), carry, G[q]);
    if (twist) {
      // lf: from y_{t-1}; lb: from y_{t+1} (zero if t is the top level)
      const double yup = LMAX > 1 ? G[LMAX > 1 ? LMAX - 2 : 0] : carry;
      G[LMAX - 1] = fma(__ldg(g.lb + t), yup, fma(__ldg(g.lf + t), YL[u], G[LMAX - 1]));
      XT[u] = G[LMAX - 1];
    }
  }
  // substitution inside the chunk (the twist chunk starts from X_t itself)
  {
    double w = 0.0;
#pragma unroll
    for (int q = LMAX - 1; q >= 0; q--)
      if (q < L) G[q] = w = q == LMAX - 1 ? G[q] : fma(__ldg(g.lb + level(q)), w, G[q]);
    EB[c][u] = w;
  }
  __syncthreads();
  // the values entering the chunks, from the twist level (above it from the
  // top of the twist chunk, which is complete)
  if (threadIdx.x < 32) {
    double carry = half ? 0.0 : XT[u];
#pragma unroll
    for (int s = 0; s < H; s++) {
      const int cc = half ? H + s : H - 1 - s;
      CB[cc][u] = carry;
      carry = fma(PE[cc], carry, EB[cc][u]);
    }
  }
  __syncthreads();
  const double carry = CB[c][u];
#pragma unroll
  for (int q = 0; q < LMAX; q++)
    if (q < L) {
      if (!twist) G[q] = fma(__ldg(g.pe + level(q)), carry, G[q]);
      G[q] = fma(wt[level(q)], G[q], om1 * C[q]);
    }
  if (!act) return;
  if (base) {
#pragma unroll
    for (int q = 0; q < LMAX; q++)
      if (q < L) base[(unsigned)level(q) * plane + rc] += G[q];
  } else {
#pragma unroll
    for (int q = 0; q < LMAX; q++)
      if (q < L) out[(unsigned)level(q) * plane + rc] = G[q];
  }
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
  return launch_dep(tab ? k_sweep_f64<true> : k_sweep_f64<false>, dim3((n + 127) / 128), dim3(128), 0, s, g, p, b, omega,
                    om1, tab, out);
}

namespace {
// Columns a block.  us a sweep at 32 / 16 / 8 (on the pressure): 96 x 48 x 64 10.9 /
// 11.1 / 11.5, 64 x 30 x 100 18.8 / 13.8 / 14.1, 112 x 56 x 112 28.6 / 22.5 / 23.5,
// 32 x 16 x 32 7.3 / 6.5 / 6.4: 32 leave SMs without a block or a last wave nearly
// empty.
constexpr int kLineCols = 16;

template <int NCH>
cudaError_t line_nch(const Geom<double>& g, const double* d, const double* r, double omega, double* out, double* base,
                     cudaStream_t s) {
  const dim3 blocks((unsigned)(((g.nx + kLineCols - 1) / kLineCols) * g.ny)), threads(kLineCols * NCH);
#define LEVELS(L) \
  case L:                                                                                                      \
    return launch_dep(k_line_f64<kLineCols, NCH, L>, blocks, threads, sizeof(double) * g.nz, s, g, d, r, omega, \
                      1.0 - omega, out, base);
  switch (line_f64_levels(g.nz, NCH)) {
    LEVELS(1) LEVELS(2) LEVELS(3) LEVELS(4) LEVELS(5) LEVELS(6)
    LEVELS(7) LEVELS(8) LEVELS(9) LEVELS(10) LEVELS(11) LEVELS(12)
    default: return cudaErrorInvalidValue;
  }
#undef LEVELS
}
}  // namespace

cudaError_t launch_line_f64(const Geom<double>& g, const double* d, const double* r, double omega, double* out,
                            double* base, cudaStream_t s) {
  switch (line_f64_chunks(g.nx, g.ny, g.nz)) {
    case 4: return line_nch<4>(g, d, r, omega, out, base, s);
    case 8: return line_nch<8>(g, d, r, omega, out, base, s);
    case 16: return line_nch<16>(g, d, r, omega, out, base, s);
    case 32: return line_nch<32>(g, d, r, omega, out, base, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_residual_f64(const Geom<double>& g, const double* p, const double* b, double* r, cudaStream_t s) {
  const Launch l = plane_launch(g.nx, g.ny, g.nz);
  k_residual_f64<<<l.grid, l.block, 0, s>>>(g, p, b, r);
  return cudaGetLastError();
}

}  // namespace stp
