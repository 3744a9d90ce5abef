// Pressure-equation residual norm without any device allocation.
//
// A variant of the solve's residual-check kernel whose scratch memory (the
// z couplings, one partial sum per block, the arrival counter and the
// result) lives in one file-scope device array instead of buffers that
// stp_init allocates.  It serves callers that hold their own device buffers
// for p and b but may not allocate: for example a host program that has
// handed all device memory to its own pool allocator, or a time-critical
// loop that cannot accept the device-wide synchronisation that cudaMalloc
// and cudaFree can cause.
//
// The array is a host-side stand-in in host code: its device address is
// obtained once per device with cudaGetSymbolAddress (the first call on a
// device does this set-up).  With CUDA's lazy module loading (the default
// since CUDA 12.2) that first call can also be what loads this library's
// device code on the device, and with it the array: that one-time load is
// a device allocation made by the CUDA runtime, not by this call.  A caller
// that must not see it at all can load the module eagerly
// (CUDA_MODULE_LOADING=EAGER) or make one call during its set-up.  Every
// call shares the array, which keeps the last call's contents; the arrival
// counter is cleared at the start of each call.  Calls whose work overlaps
// on the GPU (different streams, or several host threads) race on the
// array and must be serialised by the caller.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "device_util.cuh"
#include "stp_internal.cuh"

namespace stp {

// limits of the shared scratch array
constexpr int kNoallocMaxNz = 4096;
constexpr unsigned kNoallocMaxBlocks = 65536;

struct NoallocScratch {
  unsigned counter[2];                // one copy a call brings the counter (0) and
  double coef[2 * kNoallocMaxNz];     // the couplings: cup [nz], cdn [nz]
  double partial[kNoallocMaxBlocks];
  double result[8];
  int flag[8];
};

static __device__ __align__(256) NoallocScratch g_noalloc_scratch;

namespace {

std::mutex g_setup_mutex;
NoallocScratch* g_scratch_addr[256] = {};

// A thread takes W x cells of two rows and walks KZ levels.  The kernel is
// bound by FP64 operations (GB300 gives 500-545 Gop/s), so every difference of
// neighbours is formed once and serves both its cells (x inside the vector, y
// between the two rows, z along the walk), and squares are summed in the
// thread before the block's tree: about eleven operations a cell, where one
// cell a thread took fourteen and six more in the reduction.  256 x 128 x 192:
// 152 us of kernel (eleven operations take 130 us of the FP64 pipe; DRAM 22), a
// call 317 -> 189 us.  Eight levels a thread leave 768 blocks, a sixth of the
// GPU idle in the last wave: 200 us a call.
constexpr int kNoallocLevels = 4;

template <int W>
__global__ void __launch_bounds__(kBX* kBY) k_residual_noalloc(int nx, int ny, int nz, double idx2, double idy2,
                                                                const double* __restrict__ p,
                                                                const double* __restrict__ b,
                                                                double* __restrict__ r_out, NoallocScratch* sc,
                                                                unsigned nblocks) {
  __shared__ double sh[32];
  const int i = (blockIdx.x * kBX + threadIdx.x) * W, j = (blockIdx.y * kBY + threadIdx.y) * 2;
  const int k0 = blockIdx.z * kNoallocLevels, k1 = min(nz, k0 + kNoallocLevels);
  double s = 0.0;
  if (i < nx && j < ny) {
    auto ldv = [](const double* a, double* v) {
      if constexpr (W == 2) {
        const double2 t = *reinterpret_cast<const double2*>(a);
        v[0] = t.x, v[1] = t.y;
      } else {
        v[0] = *a;
      }
    };
    const bool two = j + 1 < ny;  // an odd ny leaves the last row alone
    const size_t plane = (size_t)nx * ny;
    const int jn = j + 2 < ny ? j + 2 : j + 2 - ny, js = j == 0 ? ny - 1 : j - 1;
    const size_t row[2] = {(size_t)j * nx, (size_t)(two ? j + 1 : 0) * nx};
    // the row past the pair: row 1 itself when the pair has one row
    const size_t on = (two ? (size_t)jn * nx : row[1]) + i, os = (size_t)js * nx + i;
    const int il = i == 0 ? nx - 1 : i - 1, ir = i + W == nx ? 0 : i + W;
    double c[2][W], dn[2][W];  // the pair's cells at level k, and p_k - p_{k-1}
#pragma unroll
    for (int y = 0; y < 2; y++) {
      double below[W];
      ldv(p + k0 * plane + row[y] + i, c[y]);
      if (k0 > 0) ldv(p + (k0 - 1) * plane + row[y] + i, below);
#pragma unroll
      for (int e = 0; e < W; e++) dn[y][e] = k0 > 0 ? c[y][e] - below[e] : 0.0;
    }
    for (int k = k0; k < k1; k++) {
      const double* lev = p + k * plane;
      const double cup = sc->coef[k], cdn = sc->coef[nz + k];
      double vn[W], vs[W], dy[3][W];
      ldv(lev + on, vn);
      ldv(lev + os, vs);
      if (!two) ldv(lev + row[1] + i, c[1]);  // the wrapped row after the last
#pragma unroll
      for (int e = 0; e < W; e++) {
        dy[0][e] = c[0][e] - vs[e];
        dy[1][e] = c[1][e] - c[0][e];
        dy[2][e] = two ? vn[e] - c[1][e] : 0.0;
      }
#pragma unroll
      for (int y = 0; y < 2; y++) {
        if (y == 1 && !two) break;
        const double* r = lev + row[y];
        double dx[W + 1], up[W], bv[W], res[W];
        dx[0] = c[y][0] - r[il];
#pragma unroll
        for (int e = 1; e < W; e++) dx[e] = c[y][e] - c[y][e - 1];
        dx[W] = r[ir] - c[y][W - 1];
        if (k < nz - 1) ldv(r + plane + i, up);
        ldv(b + k * plane + row[y] + i, bv);
#pragma unroll
        for (int e = 0; e < W; e++) {
          const double du = k < nz - 1 ? up[e] - c[y][e] : 0.0;
          double t = fma(-idx2, dx[e + 1] - dx[e], bv[e]);
          t = fma(-idy2, dy[y + 1][e] - dy[y][e], t);
          t = fma(-cup, du, t);
          t = fma(cdn, dn[y][e], t);
          res[e] = t;
          s = fma(t, t, s);
          dn[y][e] = du;
          c[y][e] = k < nz - 1 ? up[e] : c[y][e];
        }
        if (r_out) {
          double* o = r_out + k * plane + row[y] + i;
          if constexpr (W == 2)
            *reinterpret_cast<double2*>(o) = make_double2(res[0], res[1]);
          else
            *o = res[0];
        }
      }
    }
  }
  s = block_sum(s, sh);
  Red red{sc->partial, sc->counter, sc->result, sc->flag};
  if (publish_partial(red, nblocks, s, 0.0, false)) {
    const double tot = final_sum(sc->partial, nblocks, sh);
    if (threadIdx.x == 0 && threadIdx.y == 0) {
      sc->result[0] = sqrt(tot);
      sc->counter[0] = 0u;
    }
  }
}

}  // namespace

// defined in api.cu: z couplings of the Poisson operator for a channel, and
// the message stp_last_error(NULL) returns
void poisson_couplings(const stp_config& c, std::vector<double>& cup, std::vector<double>& cdn);
void set_thread_error(const std::string& msg);

namespace {
int noalloc_fail(int code, const std::string& m) {
  set_thread_error(m);
  return code;
}
}  // namespace

}  // namespace stp

using namespace stp;

extern "C" int stp_poisson_residual_noalloc(int nx, int ny, int nz, double Lx, double Ly, double Lz, double stretch,
                                            const double* p, const double* b, double* r_out, double* norm_out,
                                            void* stream) {
  if (!p || !b || !norm_out) return noalloc_fail(STP_EINVAL, "p, b and norm_out are required");
  if (nx < 3 || ny < 3 || nz < 2) return noalloc_fail(STP_EINVAL, "need nx, ny >= 3 and nz >= 2");
  if (!(Lx > 0 && Ly > 0 && Lz > 0) || !(stretch >= 0))
    return noalloc_fail(STP_EINVAL, "box lengths must be positive and stretch >= 0");
  if (nz > kNoallocMaxNz)
    return noalloc_fail(STP_EINVAL, "nz exceeds the scratch limit of " + std::to_string(kNoallocMaxNz));
  const Launch l = plane_launch(nx, ny, nz);
  if ((double)l.grid.x * l.grid.y * l.grid.z > (double)kNoallocMaxBlocks)
    return noalloc_fail(STP_EINVAL, "grid too large for the scratch array: ceil(nx/32)*ceil(ny/8)*nz must be <= " +
                                        std::to_string(kNoallocMaxBlocks));
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return noalloc_fail(STP_ECUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
  if (dev < 0 || dev >= 256) return noalloc_fail(STP_EINVAL, "device ordinal out of range");
  NoallocScratch* sc = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_addr[dev]) {
      void* addr = nullptr;
      e = cudaGetSymbolAddress(&addr, g_noalloc_scratch);
      if (e != cudaSuccess)
        return noalloc_fail(STP_ECUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
      g_scratch_addr[dev] = (NoallocScratch*)addr;
    }
    sc = g_scratch_addr[dev];
  }
  stp_config c;
  stp_config_defaults(&c);
  c.nx = nx;
  c.ny = ny;
  c.nz = nz;
  c.Lx = Lx;
  c.Ly = Ly;
  c.Lz = Lz;
  c.stretch = stretch;
  std::vector<double> cup, cdn;
  poisson_couplings(c, cup, cdn);
  cudaStream_t st = (cudaStream_t)stream;
  // counter (eight zero bytes) and couplings in one copy
  std::vector<double> head(1 + 2 * (size_t)nz);
  head[0] = 0.0;
  std::copy(cup.begin(), cup.end(), head.begin() + 1);
  std::copy(cdn.begin(), cdn.end(), head.begin() + 1 + nz);
  e = cudaMemcpyAsync(sc, head.data(), sizeof(double) * head.size(), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return noalloc_fail(STP_ECUDA, std::string("scratch set-up: ") + cudaGetErrorString(e));
  const double dx = Lx / nx, dy = Ly / ny;
  // pairs of x cells on even rows whose arrays are 16-byte aligned
  const bool vec = nx % 2 == 0 && ((uintptr_t)p | (uintptr_t)b | (uintptr_t)r_out) % 16 == 0;
  const int w = vec ? 2 : 1;
  const dim3 grid((nx + kBX * w - 1) / (kBX * w), (ny + 2 * kBY - 1) / (2 * kBY),
                  (nz + kNoallocLevels - 1) / kNoallocLevels);
  const unsigned nblocks = grid.x * grid.y * grid.z;
  (vec ? k_residual_noalloc<2> : k_residual_noalloc<1>)<<<grid, l.block, 0, st>>>(
      nx, ny, nz, 1.0 / (dx * dx), 1.0 / (dy * dy), p, b, r_out, sc, nblocks);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(norm_out, sc->result, sizeof(double), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return noalloc_fail(STP_ECUDA, std::string("residual kernel: ") + cudaGetErrorString(e));
  return STP_OK;
}
