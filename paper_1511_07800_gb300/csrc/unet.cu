// 3-D U-Net for the learned pressure guess: forward, backward and Adam, all
// in hand-written kernels.  BF16 weights and activations, FP32 accumulation
// on the tensor cores (tcgen05 with TMEM accumulators for the 3x3x3
// convolutions of the larger levels, mma.sync m16n8k16 for the rest), FP32
// master weights, gradients and optimiser state.
//
// Network (channels-last [voxel][channel], voxel = ((n*D + z)*H + y)*W + x):
//   encoder level l = 1..4 (16, 32, 64, 128 channels): two 3x3x3 conv+ReLU,
//     then a 2x2x2 mean pool (not after level 4)
//   decoder level l = 3, 2, 1: input = concat(upsample2(deeper), skip e_l),
//     two 3x3x3 conv+ReLU
//   output: 1x1x1 conv of the 16 channels, linear
// Convolutions are periodic in x and y and zero-padded in z.  The skip of
// level l is written straight into the channel slice of the decoder's
// concat buffer, so no copy is needed.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <string>
#include <vector>

#include "device_util.cuh"
#include "stp_internal.cuh"

namespace stp {
namespace nn {

typedef __nv_bfloat16 bf16;

struct Dims {
  int n, d, h, w;
  __host__ __device__ long long vox() const { return (long long)n * d * h * w; }
};

__device__ __forceinline__ void mma16816(float* c, const unsigned* a, const unsigned* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ unsigned pack2(bf16 lo, bf16 hi) {
  return (unsigned)__bfloat16_as_ushort(lo) | ((unsigned)__bfloat16_as_ushort(hi) << 16);
}

// eight BF16 of a 16-byte vector, as floats and back
__device__ __forceinline__ void unpack8(const uint4& u, float* f) {
  const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; i++) {
    f[2 * i] = __bfloat162float(__ushort_as_bfloat16((unsigned short)(w[i] & 0xFFFFu)));
    f[2 * i + 1] = __bfloat162float(__ushort_as_bfloat16((unsigned short)(w[i] >> 16)));
  }
}
__device__ __forceinline__ uint4 pack8(const float* f) {
  return make_uint4(pack2(__float2bfloat16(f[0]), __float2bfloat16(f[1])),
                    pack2(__float2bfloat16(f[2]), __float2bfloat16(f[3])),
                    pack2(__float2bfloat16(f[4]), __float2bfloat16(f[5])),
                    pack2(__float2bfloat16(f[6]), __float2bfloat16(f[7])));
}
__device__ __forceinline__ uint4 ld16(const bf16* p) { return *reinterpret_cast<const uint4*>(p); }
__device__ __forceinline__ void st16(bf16* p, const uint4& u) { *reinterpret_cast<uint4*>(p) = u; }

// voxel index (below 2^31, checked at creation) as sample and coordinates,
// in 32-bit arithmetic
struct Coord {
  int n, z, y, x;
};
__device__ __forceinline__ Coord coord_of(const Dims& dm, unsigned v) {
  Coord c;
  c.x = (int)(v % (unsigned)dm.w);
  v /= (unsigned)dm.w;
  c.y = (int)(v % (unsigned)dm.h);
  v /= (unsigned)dm.h;
  c.z = (int)(v % (unsigned)dm.d);
  c.n = (int)(v / (unsigned)dm.d);
  return c;
}
__device__ __forceinline__ long long voxel_at(const Dims& dm, int n, int z, int y, int x) {
  return ((long long)(n * dm.d + z) * dm.h + y) * dm.w + x;
}

// ---------------------------------------------------------------------------
// 3x3x3 convolution as an implicit GEMM on the tensor cores (mma.sync):
//   y[v][o] = b[o] + sum_{t, c} wt[t][o][c] x[v + off(t)][c]
// M = voxels, N = output channels, K = 27 taps x input channels, for the levels
// k_conv3_tc does not take.  A block computes 8 x 4 x 2 voxels (a warp two x
// rows of them) x 8 NT channels.  These levels are small, so what they cost
// is latency: the block stages its halo and all 27 taps' weights of its
// channels in shared memory up front (three cp.async groups, the later taps'
// weights landing while the first are multiplied), and a K step is then two
// ldmatrix and NT multiplies.  Each output sees the same sequence of MMAs (taps,
// then channels) at every NT.  128 -> 128 at 16 x 8 x 16 voxels: 26 us, 85 with
// operands loaded step by step from global memory.
// Options: ReLU; multiply by (mask > 0) (the derivative of the ReLU that
// produced this layer's input, used when the kernel runs the backward data
// pass with transposed weights); no bias when bias is NULL.
// ---------------------------------------------------------------------------
constexpr int CS_TX = 8, CS_TY = 4, CS_TZ = 2, CS_HX = CS_TX + 2, CS_HY = CS_TY + 2, CS_HZ = CS_TZ + 2;
constexpr int CS_HVOX = CS_HX * CS_HY * CS_HZ;

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool fill) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(fill ? 16 : 0)
               : "memory");
}
// a coordinate at most one tile outside [0, n), wrapped
__device__ __forceinline__ int wrap1(int a, int n) { return a < 0 ? a + n : a >= n ? (a - n) % n : a; }

// shared memory: the halo, then the weights of `taps` taps, both in chunks of
// 8 input channels (16 bytes a voxel or output channel).  RING: the weights
// stream through a ring of CS_RING taps (several blocks an SM, or channel
// counts whose 27 taps do not fit); else all are resident.
constexpr int CS_RING = 6;
constexpr size_t conv3_smem(int cin, int nt, bool ring) {
  return (size_t)(cin / 8) * 16 * (CS_HVOX + (ring ? CS_RING : 27) * 8 * nt);
}

template <int NT, bool RING>
__global__ void __launch_bounds__(128) k_conv3(Dims dm, const bf16* __restrict__ x, int ldx, int cin,
                                               const bf16* __restrict__ wt, const float* __restrict__ bias, int cout,
                                               bf16* __restrict__ y, int ldy, int relu, const bf16* __restrict__ mask,
                                               int ldm) {
  extern __shared__ __align__(128) uint8_t csm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q = lane & 3;
  const int nch = cin / 8;
  const uint32_t sx = su32(csm), sw = sx + 16 * CS_HVOX * nch;
  const int tx = (dm.w + CS_TX - 1) / CS_TX, ty = (dm.h + CS_TY - 1) / CS_TY, tz = (dm.d + CS_TZ - 1) / CS_TZ;
  int r = blockIdx.x;
  const int x0 = (r % tx) * CS_TX;
  r /= tx;
  const int y0 = (r % ty) * CS_TY;
  r /= ty;
  const int z0 = (r % tz) * CS_TZ, nn = r / tz;
  const int cob = blockIdx.y * NT * 8;
  cudaGridDependencySynchronize();
  for (int i = tid; i < CS_HVOX; i += 128) {
    const int hx = i % CS_HX, hy = (i / CS_HX) % CS_HY, hz = i / (CS_HX * CS_HY);
    const int vz = z0 - 1 + hz;
    const bool in = vz >= 0 && vz < dm.d;
    const bf16* src = x + voxel_at(dm, nn, in ? vz : 0, wrap1(y0 - 1 + hy, dm.h), wrap1(x0 - 1 + hx, dm.w)) * ldx;
    for (int c = 0; c < nch; c++) cp16(sx + 16 * (c * CS_HVOX + i), src + 8 * c, in);
  }
  // weights of taps [ta, tb), one group: a thread keeps its output row and its
  // chunks from tap to tap
  constexpr int TPR = 128 / (8 * NT);  // threads a row
  const int wo = tid / TPR, wc = tid % TPR;
  const bf16* wrow = wt + (long long)(cob + wo) * cin;
  auto load_w = [&](int ta, int tb) {
    for (int t = ta; t < tb; t++) {
      const bf16* src = wrow + (long long)t * cout * cin;
      const uint32_t dst = sw + 16 * ((RING ? t % CS_RING : t) * nch * 8 * NT + wo);
      for (int c = wc; c < nch; c += TPR) cp16(dst + 16 * c * 8 * NT, src + 8 * c, true);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if constexpr (RING) {
    for (int t = 0; t < CS_RING - 1; t++) load_w(t, t + 1);
  } else {
    for (int part = 0; part < 3; part++) load_w(9 * part, 9 * part + 9);
  }
  float acc[NT][4];
#pragma unroll
  for (int n = 0; n < NT; n++) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
  // the warp's voxel rows: y = y0 + 2 (warp & 1) + {0, 1}, z = z0 + warp / 2
  const int wy = 2 * (warp & 1), wz = warp >> 1;
  // A matrices: (rows 0-7, 8-15) x (channels 0-7, 8-15); B: (outputs 0-7 of
  // an 8-channel tile pair) x (channels 0-7, 8-15)
  const int mi = lane >> 3, mr = lane & 7;
  const uint32_t a_lane = sx + 16 * ((mi >> 1) * CS_HVOX + (wz * CS_HY + wy + (mi & 1)) * CS_HX + mr);
  const uint32_t b_lane = sw + 16 * ((mi & 1) * 8 * NT + (mi >> 1) * 8 + mr);
  for (int t = 0; t < 27; t++) {
    if constexpr (RING) {
      // tap t has landed when at most the CS_RING - 2 groups after it are in
      // flight; past the barrier every warp has left tap t - 1, whose slot
      // takes tap t + CS_RING - 1
      asm volatile("cp.async.wait_group %0;" ::"n"(CS_RING - 2) : "memory");
      __syncthreads();
      if (t + CS_RING - 1 < 27)
        load_w(t + CS_RING - 1, t + CS_RING);
      else
        asm volatile("cp.async.commit_group;" ::: "memory");
    } else if (t % 9 == 0) {
      if (t == 0)
        asm volatile("cp.async.wait_group 2;" ::: "memory");
      else if (t == 9)
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      else
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
    }
    const uint32_t at = a_lane + 16 * ((t / 9 * CS_HY + t / 3 % 3) * CS_HX + t % 3);
    const uint32_t bt = b_lane + 16 * (RING ? t % CS_RING : t) * nch * 8 * NT;
#pragma unroll 2
    for (int c = 0; c < nch; c += 2) {
      unsigned a[4];
      asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                   : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                   : "r"(at + 16 * c * CS_HVOX)
                   : "memory");
      const uint32_t bc = bt + 16 * c * 8 * NT;
      if constexpr (NT == 1) {
        unsigned b[2];
        asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
                     : "=r"(b[0]), "=r"(b[1])
                     : "r"(bc)
                     : "memory");
        mma16816(acc[0], a, b);
      } else {
#pragma unroll
        for (int n = 0; n < NT; n += 2) {
          unsigned b[4];
          asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                       : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3])
                       : "r"(bc + 16 * 8 * n)
                       : "memory");
          mma16816(acc[n], a, b);
          mma16816(acc[n + 1], a, b + 2);
        }
      }
    }
  }
  const int vx = x0 + g, vz = z0 + wz;
#pragma unroll
  for (int n = 0; n < NT; n++) {
    const int co = cob + n * 8 + 2 * q;
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int vy = y0 + wy + h;
      if (vx >= dm.w || vy >= dm.h || vz >= dm.d) continue;
      const long long v = voxel_at(dm, nn, vz, vy, vx);
      float v0 = acc[n][2 * h], v1 = acc[n][2 * h + 1];
      if (bias) {
        v0 += bias[co];
        v1 += bias[co + 1];
      }
      if (relu) {
        v0 = fmaxf(v0, 0.f);
        v1 = fmaxf(v1, 0.f);
      }
      if (mask) {
        const bf16* mp = mask + v * ldm + co;
        if (!(__bfloat162float(mp[0]) > 0.f)) v0 = 0.f;
        if (!(__bfloat162float(mp[1]) > 0.f)) v1 = 0.f;
      }
      *reinterpret_cast<unsigned*>(y + v * ldy + co) = pack2(__float2bfloat16(v0), __float2bfloat16(v1));
    }
  }
}

// ---------------------------------------------------------------------------
// The same convolution on the fifth-generation tensor cores (tcgen05, TMEM
// accumulator), for layers whose level has w % 8 == 0 and h % 16 == 0 and
// channel counts that are multiples of 16 (k_conv3_tz below) or whose weights do
// not fit an SM (this kernel: 64 -> 64, 64 -> 128, 128 -> 128, 192 -> 64 and back;
// input channels a multiple of 64).
//
// A tile is zt planes of 128 voxels, 8 (x) x 16 (y) at zt consecutive z, for
// all cout channels: per plane M = 128, N = cout, K = 27 taps x cin, the zt
// accumulators side by side in tensor memory.  The input is staged by groups
// of 64 channels as a halo of 10 x 18 x (zt + 2) voxels (periodic in x
// and y, zeros outside the walls) in the K-major core-matrix layout without
// swizzle: 8-channel chunk j of halo voxel (hx, hy, hz) is 16 bytes at
// j CHUNK + ((hz HY + hy) HX + hx) 16, CHUNK = 16 HX HY (zt + 2).  The A operand
// of tap (dz, dy, dx) for plane p is then the descriptor whose start is the
// halo voxel (1+dx, 1+dy, p+dz): its 8-row core matrices are 8 consecutive x
// (16 bytes apart), the next 8 rows are the next y (SBO = 16 HX bytes), the
// next 8 channels the next chunk (LBO = one chunk of the halo).  So the 27
// taps need no data movement.  The weights come as bulk copies of an image
// kept in shared-memory order, three taps at a time through a ring.
//
// What bounds it: an MMA of M = 128, K = 16 takes 68 clocks whatever the layout
// and N up to 128 when one thread issues them in a loop, 48 when an elected
// thread issues unrolled taps, so a layer cannot take less than
// 27 cin/16 x 48 clocks a 128 voxels.  To keep the MMAs back to back, blocks
// stay for many tiles and their warps take roles: four load halos, one thread
// copies weights, up to two threads issue MMAs, four warps store results (as
// accumulator stages), each waiting on mbarriers for the others.  us, with
// blocks that load, multiply and store one tile after another, several an SM /
// this (both with resident weights where they fit): 16 -> 16 at 128 x 64 x 128 77
// / 49, 48 -> 16 190 / 113, 32 -> 32 at half that size 34 / 20.  With a weight
// stage a tap, handing it over (0.36 us) took as long as its copy: 64 -> 64 at 32
// x 16 x 32 15.5 with one tap a stage, 12.5 with three; 192 -> 64 28.8 / 27.5,
// bound by its weights (660 KB a tile) and three halos in sequence: beside the
// ring there is room for one halo, so a group is loaded when the one before it
// has been multiplied.  Eight loader warps (16 -> 16 62) or a pair of lanes a
// voxel (53) are slower.
//
// Each accumulator sees the same MMAs in the same order (groups, taps,
// 16-channel steps) whatever the plan.  Every wait is bounded; on a time-out
// the role sets *err and the block's failure flag and leaves, the others
// follow, and the block still frees its tensor memory.
// ---------------------------------------------------------------------------
constexpr int TC_TX = 8, TC_TY = 16, TC_HX = 10, TC_HY = 18;
constexpr int TC_PLANE = TC_HX * TC_HY * 16;  // bytes of one halo plane of one 8-channel chunk
constexpr int TC_CG = 64;                     // channels per halo group
constexpr int TC_RING = 8;                    // most weight stages
constexpr int TC_STAPS = 3;                   // taps a weight stage
constexpr int TC_THREADS = 352;               // 4 loader warps, 4 store warps, 2 MMA warps, weights

// shared-memory matrix descriptor: no swizzle, K-major core matrices
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

// instruction descriptor of kind::f16: BF16 A and B, FP32 D, both K-major
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// bounded wait for phase `parity` of an mbarrier (about one second of clock)
__device__ __forceinline__ bool tc_wait(uint32_t mbar, uint32_t parity) {
  long long t0 = 0;
  for (int n = 0;; n++) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (done) return true;
    if (n == 0) t0 = clock64();
    if (clock64() - t0 > 2000000000LL) return false;
    if (n > 16) __nanosleep(40);
  }
}
// the same for a whole warp: one lane polls (the others would take its issue slots)
__device__ __forceinline__ bool tc_wait_warp(uint32_t mbar, uint32_t parity) {
  int ok = 1;
  if ((threadIdx.x & 31) == 0) ok = tc_wait(mbar, parity);
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}
__device__ __forceinline__ void tc_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}
// bytes (a multiple of 16, at most 1 MB) global -> shared, completing on mbar
__device__ __forceinline__ void tc_bulk(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
      "r"(bytes), "r"(mbar)
      : "memory");
}

// one thread of the (converged) warp, chosen in a form the compiler knows to be
// warp-uniform: it then keeps descriptors in uniform registers
__device__ __forceinline__ bool tc_elect() {
  uint32_t e;
  asm volatile("{\n.reg .pred e;\n.reg .b32 t;\nelect.sync t|e, 0xffffffff;\nselp.u32 %0, 1, 0, e;\n}\n" : "=r"(e));
  return e != 0;
}
// descriptors as words: only the low one, which holds the address, changes
__device__ __forceinline__ void tc_mma(uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                       uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\n.reg .b64 da, db;\nmov.b64 da, {%1, %2};\nmov.b64 db, {%3, %4};\nsetp.ne.b32 p, %6, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n}\n" ::"r"(d),
      "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(acc));
}
// the MMAs of one tap of a group of 16 NK channels, NP planes (a_lo: the
// first plane's halo): every offset but the tap's weights is a constant
// (descriptor addresses count 16 bytes); ZT: planes of the halo
template <int NK, int NP, int ZT>
__device__ __forceinline__ void tc_tap(int tap, const uint32_t (&d)[NP], uint32_t a_lo, uint32_t a_hi, uint32_t b_lo,
                                       uint32_t b_hi, uint32_t idesc, bool first) {
  constexpr int CH = TC_PLANE / 16 * (ZT + 2);
  const uint32_t a_tap = a_lo + (uint32_t)(((tap / 9) * TC_HY + (tap / 3) % 3) * TC_HX + tap % 3);
#pragma unroll
  for (int pl = 0; pl < NP; pl++)
#pragma unroll
    for (int kk = 0; kk < NK; kk++)
      tc_mma(d[pl], a_tap + (uint32_t)(pl * (TC_PLANE / 16) + 2 * kk * CH), a_hi, b_lo + 16u * kk, b_hi, idesc,
             kk > 0 || !first ? 1u : 0u);
}

__device__ __forceinline__ void tc_ld16(uint32_t* a, uint32_t col) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(a[8]),
        "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15])
      : "r"(col));
}
// bias (in shared memory, zeros if none), ReLU or mask, BF16 rounding and store
// of 16 channels of a voxel
__device__ __forceinline__ void tc_store16(const uint32_t* a, const float* bias, int relu, const bf16* mask, bf16* y) {
  float v[16];
#pragma unroll
  for (int h = 0; h < 4; h++) {
    const float4 bv = reinterpret_cast<const float4*>(bias)[h];
    v[4 * h] = __uint_as_float(a[4 * h]) + bv.x;
    v[4 * h + 1] = __uint_as_float(a[4 * h + 1]) + bv.y;
    v[4 * h + 2] = __uint_as_float(a[4 * h + 2]) + bv.z;
    v[4 * h + 3] = __uint_as_float(a[4 * h + 3]) + bv.w;
  }
  if (relu)
#pragma unroll
    for (int h = 0; h < 16; h++) v[h] = fmaxf(v[h], 0.f);
  if (mask) {
    float m[16];
    unpack8(ld16(mask), m);
    unpack8(ld16(mask + 8), m + 8);
#pragma unroll
    for (int h = 0; h < 16; h++) v[h] = m[h] > 0.f ? v[h] : 0.f;
  }
  uint32_t o[8];
#pragma unroll
  for (int h = 0; h < 8; h++) o[h] = pack2(__float2bfloat16(v[2 * h]), __float2bfloat16(v[2 * h + 1]));
  // one 32-byte sector (rows and slices are 16 channels)
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(y), "r"(o[0]), "r"(o[1]), "r"(o[2]),
               "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7])
               : "memory");
}
// results of a tile: planes of cout columns from tensor-memory column acc, for
// the voxel v of the first plane, planes vz voxels apart; 32 columns a wait (16
// a wait with scalar reads of the bias and the mask took 0.4 us each)
__device__ __forceinline__ void tc_store(uint32_t acc, long long v, long long vz, int planes, const float* bias,
                                         int cout, bf16* __restrict__ y, int ldy, int relu,
                                         const bf16* __restrict__ mask, int ldm) {
  const int n = planes * cout;
  int c = 0;
  const bf16* mp = mask ? mask + v * ldm : nullptr;
  bf16* yp = y + v * ldy;
  const long long my = vz * ldm, yy = vz * ldy;
  for (int i = 0; i < n; i += 32) {
    uint32_t a[32];
    const bool two = i + 16 < n;
    tc_ld16(a, acc + i);
    if (two) tc_ld16(a + 16, acc + i + 16);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int h = 0; h < 2; h++) {
      if (h == 1 && !two) break;
      tc_store16(a + 16 * h, bias + c, relu, mp ? mp + c : nullptr, yp + c);
      if ((c += 16) == cout) {
        c = 0;
        yp += yy;
        if (mp) mp += my;
      }
    }
  }
}

// how k_conv3_tc runs a layer, one block an SM
struct TcPlan {
  int zt;    // planes a tile
  int ring;  // weight stages
  int as;    // accumulator stages
  int cols;  // tensor-memory columns
  size_t smem;
};

template <int ZT>
__global__ void __launch_bounds__(TC_THREADS) k_conv3_tc(Dims dm, const bf16* __restrict__ x, int ldx, int cin,
                                                         const bf16* __restrict__ wimg, const float* __restrict__ bias,
                                                         int cout, bf16* __restrict__ y, int ldy, int relu,
                                                         const bf16* __restrict__ mask, int ldm, TcPlan P, int* err) {
  extern __shared__ __align__(1024) uint8_t tsm[];
  // mbarriers: halo full and empty, weight full and empty, accumulator full and
  // empty
  __shared__ __align__(8) uint64_t hfull, hempty, wfull[TC_RING], wempty[TC_RING], afull[2], aempty[2], drain[2];
  __shared__ uint32_t tslot;
  __shared__ volatile int sfail;
  __shared__ __align__(16) float sbias[256];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int zt = ZT, hz_n = zt + 2;
  constexpr int NI = ZT > 1 ? 2 : 1, NP = ZT / NI;  // issuing threads, planes each
  const uint32_t stage_bytes = (uint32_t)cout * TC_CG * 2;  // one tap's weights of one group
  constexpr uint32_t chunk = TC_PLANE * hz_n;             // bytes of one 8-channel chunk of the halo
  const uint32_t halo0 = su32(tsm), w0 = halo0 + (TC_CG / 8) * chunk;
  const int ngroups = cin / TC_CG;
  const int nxt = dm.w / TC_TX, nyt = dm.h / TC_TY, nzt = dm.d / zt;
  const int ntiles = nxt * nyt * nzt * dm.n;
  if (tid == 0) {
    auto init = [](uint64_t* m, int count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(m)), "r"(count)); };
    init(&hfull, 128);
    init(&hempty, NI);
    for (int i = 0; i < 2; i++) {
      init(&afull[i], NI);
      init(&aempty[i], 128);
    }
    for (int i = 0; i < TC_RING; i++) {
      init(&wfull[i], 1);
      init(&wempty[i], NI);
    }
    for (int i = 0; i < NI; i++) init(&drain[i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    sfail = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tslot)), "r"(P.cols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  cudaGridDependencySynchronize();
  for (int i = tid; i < cout; i += blockDim.x) sbias[i] = bias ? bias[i] : 0.f;
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tslot;
  struct Tile {
    int x0, y0, z0, n;
  };
  auto tile_at = [&](int t) {
    Tile r;
    r.x0 = t % nxt * TC_TX;
    t /= nxt;
    r.y0 = t % nyt * TC_TY;
    t /= nyt;
    r.z0 = t % nzt * zt;
    r.n = t / nzt;
    return r;
  };
  bool ok = true;
  if (warp < 4) {
    // halos, group by group, tile by tile: a warp takes three rows of ten
    // voxels at a time, a lane a voxel, its chunks inner
    const int hx = lane % TC_HX, hr = lane / TC_HX, rows = TC_HY * hz_n;
    int use = 0;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      const Tile T = tile_at(t);
      int gx = T.x0 - 1 + hx;
      gx = gx < 0 ? gx + dm.w : (gx >= dm.w ? gx - dm.w : gx);
      for (int g = 0; g < ngroups; g++, use++) {
        if (!(ok = tc_wait_warp(su32(&hempty), (use & 1) ^ 1))) break;
        const uint32_t base = halo0 + 16 * hx;
        const bf16* xg = x + (long long)gx * ldx + g * TC_CG;
        for (int row = warp * 3 + hr; row < rows; row += 12) {
          if (hr == 3) break;
          const int hz = row / TC_HY, hy = row - hz * TC_HY;
          int gy = T.y0 - 1 + hy;
          const int gz = T.z0 - 1 + hz;
          gy = gy < 0 ? gy + dm.h : (gy >= dm.h ? gy - dm.h : gy);
          const bool in = gz >= 0 && gz < dm.d;
          const bf16* src = xg + voxel_at(dm, T.n, in ? gz : 0, gy, 0) * ldx;
          const uint32_t dst = base + row * (16 * TC_HX);  // chunk 0; chunk j is `chunk` further
          for (int j = 0; j < TC_CG / 8; j++) cp16(dst + j * chunk, src + 8 * j, in);
        }
        asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_arrive(su32(&hfull));
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  } else if (warp < 8) {
    // results: TMEM lane = output row (a warp reads the lanes of its quarter)
    const int r = (warp - 4) * 32 + lane;
    int it = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, it++) {
      const Tile T = tile_at(t);
      const int st = it % P.as;
      // (the warp stays together: TMEM loads are warp-wide)
      if (!(ok = tc_wait_warp(su32(&afull[st]), (it / P.as) & 1))) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      tc_store(tmem + ((uint32_t)((warp - 4) * 32) << 16) + (uint32_t)(st * zt * cout),
               voxel_at(dm, T.n, T.z0, T.y0 + r / 8, T.x0 + (r % 8)), (long long)dm.h * dm.w, zt, sbias, cout, y, ldy,
               relu, mask, ldm);
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      tc_arrive(su32(&aempty[st]));
    }
  } else if (warp < 8 + NI) {
    // MMAs.  Issued from a loop with runtime counts by one plain lane they cost
    // 300-500 clocks each in descriptor arithmetic, against about 50 this way:
    // an elected thread, every tap unrolled; two threads share a tile's planes
    // (an accumulator belongs to one of them).
    if (tc_elect()) {
      const int mw = warp - 8;
      const uint32_t idesc = tc_idesc(128, cout);
      int hph = 0, ws = 0, wph = 0, as = 0, aph = 0;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        if (!(ok = tc_wait(su32(&aempty[as]), aph ^ 1))) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t d[NP];
#pragma unroll
        for (int pl = 0; pl < NP; pl++) d[pl] = tmem + (uint32_t)((as * ZT + mw * NP + pl) * cout);
        for (int g = 0; g < ngroups && ok; g++) {
          if (!(ok = tc_wait(su32(&hfull), hph))) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          constexpr int NK = TC_CG / 16;
          const uint64_t a_desc = tc_desc(halo0 + mw * NP * TC_PLANE, chunk, TC_HX * 16);
          const uint64_t b_desc = tc_desc(w0, 128, NK * 256);
          const uint32_t a_lo = (uint32_t)a_desc, a_hi = (uint32_t)(a_desc >> 32);
          const uint32_t b_lo = (uint32_t)b_desc, b_hi = (uint32_t)(b_desc >> 32), stage16 = stage_bytes >> 4;
#pragma unroll 3
          for (int row = 0; row < 27 / TC_STAPS; row++) {
            if (!(ok = ok && tc_wait(su32(&wfull[ws]), wph))) continue;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int i = 0; i < TC_STAPS; i++)
              tc_tap<NK, NP, ZT>(row * TC_STAPS + i, d, a_lo, a_hi, b_lo + (ws * TC_STAPS + i) * stage16, b_hi, idesc,
                                 g == 0 && row == 0 && i == 0);
            tc_commit(su32(&wempty[ws]));
            if (++ws == P.ring) ws = 0, wph ^= 1;
          }
          tc_commit(su32(&hempty));
          hph ^= 1;
        }
        tc_commit(su32(&afull[as]));
        if (++as == P.as) as = 0, aph ^= 1;
      }
      // the block may not end with MMAs in flight: the store warps have awaited
      // the last tiles' results; after a time-out they may have left
      if (!ok || sfail) {
        tc_commit(su32(&drain[mw]));
        tc_wait(su32(&drain[mw]), 0);
      }
    }
  } else if (warp == 10 && lane == 0) {
    // weights
    int wuse = 0;
    const uint32_t bytes = TC_STAPS * stage_bytes;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x)
      for (int q = 0; q < ngroups * 27 / TC_STAPS; q++, wuse++) {
        const int ws = wuse % P.ring;
        if (!(ok = tc_wait(su32(&wempty[ws]), ((wuse / P.ring) & 1) ^ 1))) break;
        tc_bulk(w0 + ws * bytes, reinterpret_cast<const uint8_t*>(wimg) + (size_t)q * bytes, bytes, su32(&wfull[ws]));
      }
    // copies still in flight land before the block ends
    for (int r = 0; r < P.ring && r < wuse; r++) {
      const int u = wuse - 1 - r;
      if (!tc_wait(su32(&wfull[u % P.ring]), (u / P.ring) & 1)) ok = false;
    }
  }
  if (!ok) {
    sfail = 1;
    atomicExch(err, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(P.cols));
}

// The same with resident weights, for layers whose weights fit beside two halo
// planes.  The A operand of an MMA is read from shared memory at 128 x 32 bytes,
// about 48 clocks, whatever N up to 128; with N = 16 or 32 output channels the
// multiply itself would take a quarter of that.  So a plane of the input is read
// once for the three output planes it contributes to: accumulators of a tile's
// planes lie side by side in tensor memory, input plane q (from -1) reaches
// output planes q-1, q, q+1 through z taps 2, 1, 0, and the weights of a (y, x)
// tap are stacked in that order, so one MMA of N = 3 cout does all three.  An
// output plane's first product, which must not add, is an MMA of its own.
// Planes q = -1 and q = zt reach one output plane, their neighbours two.  9
// (zt + 2) MMAs of 16 channels a tile of zt planes instead of 27 zt.
//
// The halo is loaded plane by plane (10 x 18 voxels, up to 64 channels) into a
// ring, a loader warp a plane, each with one plane landing while it issues the
// next; no plane is loaded twice in a tile.  Accumulators see the same MMAs in
// the same order (groups, z, y, x taps, 16-channel steps) as in k_conv3_tc.
// us at 128 x 64 x 128, a tap at a time (k_conv3_tc with resident weights) /
// this: 16 -> 16 49 / 38, 48 -> 16 113 / 70; half that size 16 -> 32 20 / 16, 32
// -> 32 21 / 19, 96 -> 32 65 / 46; a quarter 32 -> 64 17 / 9.5.  16 -> 16 takes
// 26 without MMAs and stores, 16 with no loads either, 29 without loads alone:
// the latencies of a block's chain of planes add up.  Not faster: two planes a
// halo stage 40, 16 planes a tile (one accumulator stage) 44, 4 planes 41, three
// blocks an SM (64 registers) 39.
struct TzPlan {
  int zt;      // planes a tile
  int hs;      // halo stages (planes)
  int as;      // accumulator stages
  int cols;    // tensor-memory columns
  int per_sm;  // blocks an SM
  size_t smem;
};
constexpr int TZ_HALO = 8;       // most halo stages
constexpr int TZ_GROUPS = 4;     // most channel groups
constexpr int TZ_THREADS = 320;  // 4 loader warps, 4 store warps, MMA, weights

// the MMAs of one input plane and group of 16 NK channels: d, idesc, b_lo are
// those of all output planes it reaches; with `fresh` the last of them (idesc1,
// at column offset d1 and weight offset b1; the others are idesc0, none if 0)
// starts here
template <int NK>
__device__ __forceinline__ void tz_plane(uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                         uint32_t tap16, uint32_t idesc, bool fresh, uint32_t idesc0, uint32_t idesc1,
                                         uint32_t d1, uint32_t b1) {
  constexpr uint32_t CH = TC_PLANE / 16;
#pragma unroll
  for (int tap = 0; tap < 9; tap++)
#pragma unroll
    for (int kk = 0; kk < NK; kk++) {
      const uint32_t a = a_lo + (uint32_t)(tap / 3 * TC_HX + tap % 3 + 2 * kk * (int)CH);
      const uint32_t b = b_lo + tap * tap16 + 16u * kk;
      if (tap == 0 && kk == 0 && fresh) {
        if (idesc0) tc_mma(d, a, a_hi, b, b_hi, idesc0, 1u);
        tc_mma(d + d1, a, a_hi, b + b1, b_hi, idesc1, 0u);
      } else {
        tc_mma(d, a, a_hi, b, b_hi, idesc, 1u);
      }
    }
}

__global__ void __launch_bounds__(TZ_THREADS) k_conv3_tz(Dims dm, const bf16* __restrict__ x, int ldx, int cin,
                                                         const bf16* __restrict__ wimg, const float* __restrict__ bias,
                                                         int cout, bf16* __restrict__ y, int ldy, int relu,
                                                         const bf16* __restrict__ mask, int ldm, TzPlan P, int* err) {
  extern __shared__ __align__(1024) uint8_t tsm[];
  __shared__ __align__(8) uint64_t hfull[TZ_HALO], hempty[TZ_HALO], wfull[TZ_GROUPS], afull[2], aempty[2], drain;
  __shared__ uint32_t tslot;
  __shared__ volatile int sfail;
  __shared__ __align__(16) float sbias[256];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, zt = P.zt;
  const uint32_t plane_bytes = (uint32_t)(min(cin, TC_CG) / 8) * TC_PLANE;
  const uint32_t halo0 = su32(tsm), w0 = halo0 + P.hs * plane_bytes;
  const int ngroups = (cin + TC_CG - 1) / TC_CG;
  const int nxt = dm.w / TC_TX, nyt = dm.h / TC_TY, nzt = dm.d / zt;
  const int ntiles = nxt * nyt * nzt * dm.n;
  if (tid == 0) {
    auto init = [](uint64_t* m, int count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(m)), "r"(count)); };
    for (int i = 0; i < TZ_HALO; i++) {
      init(&hfull[i], 32);
      init(&hempty[i], 1);
    }
    for (int i = 0; i < TZ_GROUPS; i++) init(&wfull[i], 1);
    for (int i = 0; i < 2; i++) {
      init(&afull[i], 1);
      init(&aempty[i], 128);
    }
    init(&drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    sfail = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tslot)), "r"(P.cols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  cudaGridDependencySynchronize();
  for (int i = tid; i < cout; i += blockDim.x) sbias[i] = bias ? bias[i] : 0.f;
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tslot;
  struct Tile {
    int x0, y0, z0, n;
  };
  auto tile_at = [&](int t) {
    Tile r;
    r.x0 = t % nxt * TC_TX;
    t /= nxt;
    r.y0 = t % nyt * TC_TY;
    t /= nyt;
    r.z0 = t % nzt * zt;
    r.n = t / nzt;
    return r;
  };
  bool ok = true;
  if (warp < 4) {
    // halo planes: unit u (tile by tile, group by group, plane by plane) belongs
    // to warp u mod nl; three rows of ten voxels at a time, a lane a voxel, its
    // chunks inner.  No more warps than stages: a warp that waits for unit u then
    // knows unit u - 2 hs consumed, so the phase it waits for is unambiguous.  A
    // plane is handed over once the warp's next one is issued (`lag`), which needs
    // more stages than warps: the next one's stage must not be waiting for this
    // plane.
    const int hx = lane % TC_HX, hr = lane / TC_HX;
    const int nl = min(4, P.hs);
    const bool lag = P.hs > nl;
    int u = 0, pending = -1;
    auto hand_over = [&]() {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_arrive(su32(&hfull[pending]));
    };
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      const Tile T = tile_at(t);
      int gx = T.x0 - 1 + hx;
      gx = gx < 0 ? gx + dm.w : (gx >= dm.w ? gx - dm.w : gx);
      for (int g = 0; g < ngroups && ok; g++) {
        const int c0 = g * TC_CG, nch = min(TC_CG, cin - c0) / 8;
        const bf16* xg = x + (long long)gx * ldx + c0;
        for (int q = 0; q < zt + 2; q++, u++) {
          if (u % nl != warp) continue;
          const int st = u % P.hs;
          if (!(ok = tc_wait_warp(su32(&hempty[st]), ((u / P.hs) & 1) ^ 1))) break;
          const int gz = T.z0 - 1 + q;
          const bool in = gz >= 0 && gz < dm.d;
          if (hr < 3)
            for (int row = hr; row < TC_HY; row += 3) {
              int gy = T.y0 - 1 + row;
              gy = gy < 0 ? gy + dm.h : (gy >= dm.h ? gy - dm.h : gy);
              const bf16* src = xg + voxel_at(dm, T.n, in ? gz : 0, gy, 0) * ldx;
              const uint32_t dst = halo0 + st * plane_bytes + 16 * (row * TC_HX + hx);
              for (int j = 0; j < nch; j++) cp16(dst + j * TC_PLANE, src + 8 * j, in);
            }
          asm volatile("cp.async.commit_group;" ::: "memory");
          if (lag) {
            if (pending >= 0) {
              asm volatile("cp.async.wait_group 1;" ::: "memory");
              hand_over();
            }
            pending = st;
          } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            pending = st;
            hand_over();
            pending = -1;
          }
        }
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (pending >= 0) hand_over();
  } else if (warp < 8) {
    // results: TMEM lane = output row (a warp reads the lanes of its quarter)
    const int r = (warp - 4) * 32 + lane;
    int it = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, it++) {
      const Tile T = tile_at(t);
      const int st = it % P.as;
      // (the warp stays together: TMEM loads are warp-wide)
      if (!(ok = tc_wait_warp(su32(&afull[st]), (it / P.as) & 1))) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      tc_store(tmem + ((uint32_t)((warp - 4) * 32) << 16) + (uint32_t)(st * zt * cout),
               voxel_at(dm, T.n, T.z0, T.y0 + r / 8, T.x0 + (r % 8)), (long long)dm.h * dm.w, zt, sbias, cout, y, ldy,
               relu, mask, ldm);
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      tc_arrive(su32(&aempty[st]));
    }
  } else if (warp == 8) {
    if (tc_elect()) {
      int hst = 0, hph = 0, as = 0, aph = 0;
      const uint64_t a_desc = tc_desc(halo0, TC_PLANE, TC_HX * 16);
      const uint32_t a_lo0 = (uint32_t)a_desc, a_hi = (uint32_t)(a_desc >> 32);
      const uint32_t idesc1 = tc_idesc(128, cout), istep = tc_idesc(0, cout) - tc_idesc(0, 0);
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        if (!(ok = tc_wait(su32(&aempty[as]), aph ^ 1))) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d_tile = tmem + (uint32_t)(as * zt * cout);
        for (int g = 0; g < ngroups && ok; g++) {
          if (!(ok = tc_wait(su32(&wfull[g]), 0))) break;
          const int nk = min(TC_CG, cin - g * TC_CG) / 16;
          const uint64_t b_desc = tc_desc(w0 + g * (27u * TC_CG * 2) * cout, 128, nk * 256);
          const uint32_t b_hi = (uint32_t)(b_desc >> 32), b_grp = (uint32_t)b_desc;
          const uint32_t blk16 = (uint32_t)(cout * nk * 2), tap16 = 3 * blk16;  // weights of a z tap, of a (y, x) tap
          for (int q = 0; q < zt + 2; q++) {
            if (!(ok = tc_wait(su32(&hfull[hst]), hph))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a_lo = a_lo0 + hst * (plane_bytes >> 4);
            // output planes lo .. hi; plane p through z tap q - p, stacked from tap 2 down
            const int lo = max(0, q - 2), np = min(zt - 1, q) - lo + 1;
            const uint32_t d = d_tile + (uint32_t)(lo * cout), b_lo = b_grp + (q < 2 ? (2 - q) * blk16 : 0u);
            const uint32_t idesc = idesc1 + (np - 1) * istep, idesc0 = np > 1 ? idesc - istep : 0u;
            const bool fresh = g == 0 && q < zt;
            const uint32_t d1 = (uint32_t)((np - 1) * cout), b1 = (uint32_t)(np - 1) * blk16;
            switch (nk) {
              case 1: tz_plane<1>(d, a_lo, a_hi, b_lo, b_hi, tap16, idesc, fresh, idesc0, idesc1, d1, b1); break;
              case 2: tz_plane<2>(d, a_lo, a_hi, b_lo, b_hi, tap16, idesc, fresh, idesc0, idesc1, d1, b1); break;
              case 3: tz_plane<3>(d, a_lo, a_hi, b_lo, b_hi, tap16, idesc, fresh, idesc0, idesc1, d1, b1); break;
              default: tz_plane<4>(d, a_lo, a_hi, b_lo, b_hi, tap16, idesc, fresh, idesc0, idesc1, d1, b1);
            }
            tc_commit(su32(&hempty[hst]));
            if (++hst == P.hs) hst = 0, hph ^= 1;
          }
        }
        tc_commit(su32(&afull[as]));
        if (++as == P.as) as = 0, aph ^= 1;
      }
      // the block may not end with MMAs in flight: the store warps have awaited
      // the last tiles' results; after a time-out they may have left
      if (!ok || sfail) {
        tc_commit(su32(&drain));
        tc_wait(su32(&drain), 0);
      }
    }
  } else if (lane == 0) {
    // weights, a group at a time
    for (int g = 0; g < ngroups; g++) {
      const uint32_t off = g * (27u * TC_CG * 2) * cout;
      tc_bulk(w0 + off, reinterpret_cast<const uint8_t*>(wimg) + off, 27u * 2 * cout * min(TC_CG, cin - g * TC_CG),
              su32(&wfull[g]));
    }
    for (int g = 0; g < ngroups; g++)
      if (!tc_wait(su32(&wfull[g]), 0)) ok = false;
  }
  if (!ok) {
    sfail = 1;
    atomicExch(err, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(P.cols));
}

// First layer: 1 input channel (FP32 input rounded to BF16) -> 16 channels,
// ReLU.  A thread takes four voxels of a row (the width is a multiple of 8):
// a tap's 16 weights are four vector reads of shared memory for 64
// multiply-adds (one scalar read each when a thread took one voxel: 67 us at
// 128 x 64 x 128, FP32 multiply-adds alone 12), and a row's six inputs serve
// its three taps.  The taps are added in order.
__global__ void __launch_bounds__(128) k_conv_in(Dims dm, const float* __restrict__ x, const float* __restrict__ w /*[16][27]*/,
                          const float* __restrict__ bias, bf16* __restrict__ y, int ldy) {
  __shared__ __align__(16) float ws[28][16];
  for (int i = threadIdx.x; i < 16 * 27; i += blockDim.x) ws[i % 27][i / 27] = __bfloat162float(__float2bfloat16(w[i]));
  for (int i = threadIdx.x; i < 16; i += blockDim.x) ws[27][i] = bias[i];
  __syncthreads();
  const bool vec = (reinterpret_cast<uintptr_t>(x) & 15) == 0;  // the caller's array
  const unsigned units = (unsigned)(dm.vox() / 4);
  for (unsigned f = blockIdx.x * blockDim.x + threadIdx.x; f < units; f += gridDim.x * blockDim.x) {
    const Coord c = coord_of(dm, 4 * f);
    float acc[4][16];
#pragma unroll
    for (int o = 0; o < 16; o++)
#pragma unroll
      for (int e = 0; e < 4; e++) acc[e][o] = ws[27][o];
#pragma unroll 1
    for (int r = 0; r < 9; r++) {
      const int z = c.z + r / 3 - 1;
      if (z < 0 || z >= dm.d) continue;  // planes outside the walls add nothing
      int yy = c.y + r % 3 - 1;
      yy = yy < 0 ? yy + dm.h : yy >= dm.h ? yy - dm.h : yy;
      const float* row = x + voxel_at(dm, c.n, z, yy, 0);
      const float* a = row + c.x;
      const float4 m = vec ? __ldg(reinterpret_cast<const float4*>(a)) : make_float4(a[0], a[1], a[2], a[3]);
      float in[6] = {__ldg(row + (c.x == 0 ? dm.w - 1 : c.x - 1)), m.x, m.y, m.z, m.w,
                     __ldg(row + (c.x + 4 == dm.w ? 0 : c.x + 4))};
#pragma unroll
      for (int i = 0; i < 6; i++) in[i] = __bfloat162float(__float2bfloat16(in[i]));
#pragma unroll
      for (int kx = 0; kx < 3; kx++)
#pragma unroll
        for (int o = 0; o < 16; o += 4) {
          const float4 wv = *reinterpret_cast<const float4*>(&ws[3 * r + kx][o]);
#pragma unroll
          for (int e = 0; e < 4; e++) {
            acc[e][o] = fmaf(wv.x, in[e + kx], acc[e][o]);
            acc[e][o + 1] = fmaf(wv.y, in[e + kx], acc[e][o + 1]);
            acc[e][o + 2] = fmaf(wv.z, in[e + kx], acc[e][o + 2]);
            acc[e][o + 3] = fmaf(wv.w, in[e + kx], acc[e][o + 3]);
          }
        }
    }
#pragma unroll
    for (int e = 0; e < 4; e++) {
      unsigned v[8];
#pragma unroll
      for (int o = 0; o < 8; o++)
        v[o] = pack2(__float2bfloat16(fmaxf(acc[e][2 * o], 0.f)), __float2bfloat16(fmaxf(acc[e][2 * o + 1], 0.f)));
      uint4* yp = reinterpret_cast<uint4*>(y + (4LL * f + e) * ldy);
      yp[0] = make_uint4(v[0], v[1], v[2], v[3]);
      yp[1] = make_uint4(v[4], v[5], v[6], v[7]);
    }
  }
}

// Output layer: 1x1x1, 16 channels -> 1, linear, FP32 output.
__global__ void k_conv_out(long long V, const bf16* __restrict__ x, int ldx, const float* __restrict__ w,
                           const float* __restrict__ bias, float* __restrict__ y) {
  cudaGridDependencySynchronize();
  float ws[16];
#pragma unroll
  for (int c = 0; c < 16; c++) ws[c] = __bfloat162float(__float2bfloat16(w[c]));
  const float b = bias[0];
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x) {
    float s = b, e[16];
    unpack8(ld16(x + v * ldx), e);
    unpack8(ld16(x + v * ldx + 8), e + 8);
#pragma unroll
    for (int c = 0; c < 16; c++) s = fmaf(ws[c], e[c], s);
    y[v] = s;
  }
}

// Backward of the output layer: g_d1[v][c] = gy[v] w[c] (d1 > 0);
// dW[c] += sum_v gy[v] d1[v][c], db += sum_v gy[v].
__global__ void k_conv_out_bwd(long long V, const float* __restrict__ gy, const bf16* __restrict__ d1, int ldx,
                               const float* __restrict__ w, bf16* __restrict__ gd, int ldg, float* __restrict__ gw,
                               float* __restrict__ gb) {
  cudaGridDependencySynchronize();
  __shared__ float red[17][33];
  float ws[16], acc[17];
#pragma unroll
  for (int c = 0; c < 16; c++) {
    ws[c] = __bfloat162float(__float2bfloat16(w[c]));
    acc[c] = 0.f;
  }
  acc[16] = 0.f;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x) {
    const float g = gy[v];
    acc[16] += g;
    float a[16], o[16];
    unpack8(ld16(d1 + v * ldx), a);
    unpack8(ld16(d1 + v * ldx + 8), a + 8);
#pragma unroll
    for (int c = 0; c < 16; c++) {
      acc[c] += g * a[c];
      o[c] = a[c] > 0.f ? g * ws[c] : 0.f;
    }
    st16(gd + v * ldg, pack8(o));
    st16(gd + v * ldg + 8, pack8(o + 8));
  }
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < 17; c++) {
    float s = acc[c];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[c][wp] = s;
  }
  __syncthreads();
  if (threadIdx.x < 17) {
    float s = 0.f;
    for (int i = 0; i < (int)(blockDim.x >> 5); i++) s += red[threadIdx.x][i];
    if (threadIdx.x < 16)
      atomicAdd(gw + threadIdx.x, s);
    else
      atomicAdd(gb, s);
  }
}

// ---------------------------------------------------------------------------
// Weight gradient of a 3x3x3 layer on the tensor cores:
//   gw[o][c][t] = sum_v gz[v][o] x[v + off(t)][c],   gb[o] = sum_v gz[v][o]
// GEMMs with M = output channels, N = input channels, K = voxels, one a tap.
// A block takes OT output and CT input channels and all 27 taps over a range
// of spatial tiles of 8 x 8 x 4 voxels: it stages the tile of gz and the tile
// of x with its halo in shared memory once, and the 27 taps read the same
// halo, a tap's operand being the halo rows moved by its offset (ldmatrix
// takes a row address a lane, so no data moves).  Both operands are stored
// voxel by voxel and needed along the voxels: ldmatrix.trans.  Warp w of nine
// keeps the accumulators of the three x taps of row offset (kz, ky) = (w/3,
// w%3) in registers over all its tiles.  Partial sums go to scratch in one
// slice a block range and are added in a fixed order by k_wgrad_sum (no
// atomics: results repeat bitwise); the bias gradient is the product with a
// column of ones, taken by the centre warp of the first input tile.
// Shared memory holds 8-channel chunks, 16 bytes a voxel: eight consecutive x
// are one conflict-free ldmatrix row set.
// A tap at a time from global memory (the kernel this replaces) read both
// operands 27 times in 2-byte loads: 3.8 ms of a 6.2 ms gradient of 4 x 64 x
// 32 x 64, where this takes 0.41 and the sums 0.14.
// ---------------------------------------------------------------------------
constexpr int WG_TX = 8, WG_TY = 8, WG_TZ = 4, WG_VOX = WG_TX * WG_TY * WG_TZ;
constexpr int WG_HX = WG_TX + 2, WG_HY = WG_TY + 2, WG_HZ = WG_TZ + 2, WG_HVOX = WG_HX * WG_HY * WG_HZ;
constexpr int WG_SLOTS = 28;  // taps, then the bias

// smem of a block: gz tile and x halo, in chunks, twice (the next tile lands
// while one is multiplied)
__host__ __device__ constexpr int wg_stage(int OT, int CT) { return 16 * (WG_VOX * OT / 8 + WG_HVOX * CT / 8); }
constexpr int wg_smem(int OT, int CT) { return 2 * wg_stage(OT, CT); }

__device__ __forceinline__ void ldsm4t(unsigned* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

struct WgTiles {
  int nx, ny, nz;  // tiles along x, y, z (z within a sample)
  __host__ __device__ int count(int n) const { return nx * ny * nz * n; }
};
__host__ __device__ inline WgTiles wg_tiles(const Dims& dm) {
  return WgTiles{(dm.w + WG_TX - 1) / WG_TX, (dm.h + WG_TY - 1) / WG_TY, (dm.d + WG_TZ - 1) / WG_TZ};
}
template <int OT, int CT>
__global__ void __launch_bounds__(288) k_wgrad3(Dims dm, const bf16* __restrict__ x, int ldx, int cin,
                                                const bf16* __restrict__ gz, int ldg, int cout,
                                                float* __restrict__ part) {
  extern __shared__ __align__(128) uint8_t wsm[];
  const uint32_t sg = (uint32_t)__cvta_generic_to_shared(wsm), sx = sg + 16 * WG_VOX * (OT / 8);
  constexpr uint32_t STAGE = wg_stage(OT, CT);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q = lane & 3;
  const int cts = cin / CT;
  const int ob = (int)(blockIdx.x / cts) * OT, cb = (int)(blockIdx.x % cts) * CT;
  const WgTiles tl = wg_tiles(dm);
  const int ntiles = tl.count(dm.n);
  const int t0 = (int)((long long)blockIdx.y * ntiles / gridDim.y), t1 = (int)((long long)(blockIdx.y + 1) * ntiles / gridDim.y);
  const bool bias = warp == 4 && cb == 0;
  float acc[3][OT / 16][CT / 8][4], accb[OT / 16][4];
#pragma unroll
  for (int m = 0; m < OT / 16; m++) {
#pragma unroll
    for (int i = 0; i < 4; i++) accb[m][i] = 0.f;
#pragma unroll
    for (int t = 0; t < 3; t++)
#pragma unroll
      for (int n = 0; n < CT / 8; n++) acc[t][m][n][0] = acc[t][m][n][1] = acc[t][m][n][2] = acc[t][m][n][3] = 0.f;
  }
  const unsigned ones[2] = {0x3F803F80u, 0x3F803F80u};  // BF16 1, 1
  // ldmatrix rows: lanes 8 i .. 8 i + 7 address matrix i.  A (gz): matrices
  // (voxels 0-7, 8-15) x (channels 0-7, 8-15) in the order a0 (v0, o0), a1 (v0,
  // o1), a2 (v1, o0), a3 (v1, o1); B (x): b0, b1 of channels 0-7, then of 8-15.
  const int mi = lane >> 3, mr = lane & 7;
  const uint32_t a_lane = sg + 16 * ((mi & 1) * WG_VOX + (mi >> 1) * 8 + mr);
  const uint32_t b_lane = sx + 16 * ((mi >> 1) * WG_HVOX + (mi & 1) * WG_HX + mr);
  const int kz = warp / 3, ky = warp % 3;
  auto load = [&](int tile, uint32_t st) {
    int r = tile;
    const int x0 = (r % tl.nx) * WG_TX;
    r /= tl.nx;
    const int y0 = (r % tl.ny) * WG_TY;
    r /= tl.ny;
    const int z0 = (r % tl.nz) * WG_TZ, nn = r / tl.nz;
    for (int v = tid; v < WG_VOX; v += 288) {
      const int vx = x0 + v % WG_TX, vy = y0 + (v / WG_TX) % WG_TY, vz = z0 + v / (WG_TX * WG_TY);
      const bool in = vx < dm.w && vy < dm.h && vz < dm.d;
      const bf16* src = gz + (in ? voxel_at(dm, nn, vz, vy, vx) : 0) * ldg + ob;
#pragma unroll
      for (int ch = 0; ch < OT / 8; ch++) cp16(sg + st + 16 * (ch * WG_VOX + v), src + 8 * ch, in);
    }
    for (int v = tid; v < WG_HVOX; v += 288) {
      const int hx = v % WG_HX, hy = (v / WG_HX) % WG_HY, hz = v / (WG_HX * WG_HY);
      const int vx = wrap1(x0 - 1 + hx, dm.w), vy = wrap1(y0 - 1 + hy, dm.h), vz = z0 - 1 + hz;
      const bool in = vz >= 0 && vz < dm.d;
      const bf16* src = x + voxel_at(dm, nn, in ? vz : 0, vy, vx) * ldx + cb;
#pragma unroll
      for (int ch = 0; ch < CT / 8; ch++) cp16(sx + st + 16 * (ch * WG_HVOX + v), src + 8 * ch, in);
    }
  };
  cudaGridDependencySynchronize();
  if (t0 < t1) load(t0, 0);
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (int tile = t0; tile < t1; tile++) {
    const uint32_t st = ((tile - t0) & 1) * STAGE;
    if (tile + 1 < t1) load(tile + 1, STAGE - st);
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    // K steps of 16 voxels: two x rows of the tile
#pragma unroll 2
    for (int s = 0; s < WG_VOX / 16; s++) {
      const int vy = (2 * s) % WG_TY, vz = (2 * s) / WG_TY;
      unsigned a[OT / 16][4];
#pragma unroll
      for (int m = 0; m < OT / 16; m++) ldsm4t(a[m], a_lane + st + 16 * (2 * m * WG_VOX + 16 * s));
      const uint32_t br = b_lane + st + 16 * (((vz + kz) * WG_HY + vy + ky) * WG_HX);
#pragma unroll
      for (int t = 0; t < 3; t++)
#pragma unroll
        for (int n = 0; n < CT / 16; n++) {
          unsigned b[4];
          ldsm4t(b, br + 16 * (t + 2 * n * WG_HVOX));
#pragma unroll
          for (int m = 0; m < OT / 16; m++) {
            mma16816(acc[t][m][2 * n], a[m], b);
            mma16816(acc[t][m][2 * n + 1], a[m], b + 2);
          }
        }
      if (bias)
#pragma unroll
        for (int m = 0; m < OT / 16; m++) mma16816(accb[m], a[m], ones);
    }
    __syncthreads();  // every warp has read the tile: its stage takes the one after next
  }
  // slice blockIdx.y of the scratch: [slot][cout][cin]
  float* out = part + (size_t)blockIdx.y * WG_SLOTS * cout * cin;
#pragma unroll
  for (int t = 0; t < 3; t++)
#pragma unroll
    for (int m = 0; m < OT / 16; m++)
#pragma unroll
      for (int n = 0; n < CT / 8; n++) {
        float* o = out + ((size_t)(warp * 3 + t) * cout + ob + 16 * m + g) * cin + cb + 8 * n + 2 * q;
        *reinterpret_cast<float2*>(o) = make_float2(acc[t][m][n][0], acc[t][m][n][1]);
        *reinterpret_cast<float2*>(o + 8 * cin) = make_float2(acc[t][m][n][2], acc[t][m][n][3]);
      }
  if (bias && q == 0)
#pragma unroll
    for (int m = 0; m < OT / 16; m++) {
      out[((size_t)27 * cout + ob + 16 * m + g) * cin] = accb[m][0];
      out[((size_t)27 * cout + ob + 16 * m + g + 8) * cin] = accb[m][2];
    }
}

// gw[o][c][t], gb[o] = sum over the slices: a block takes 32 outputs, its
// eight warps every eighth slice each, added in a fixed order (one thread an
// output walking up to 304 slices waited on memory: 15 us a layer)
__global__ void __launch_bounds__(256) k_wgrad_sum(const float* __restrict__ part, int slices, int cin, int cout,
                                                   float* __restrict__ gw, float* __restrict__ gb) {
  cudaGridDependencySynchronize();
  __shared__ float red[8][32];
  const int n = 27 * cout * cin, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
  const bool in = e < n + cout;
  const size_t off = e < n ? e : (size_t)27 * cout * cin + (size_t)(in ? e - n : 0) * cin;
  const size_t stride = (size_t)WG_SLOTS * cout * cin;
  float s = 0.f;
#pragma unroll 4
  for (int i = warp; i < slices; i += 8) s += part[off + i * stride];
  red[warp][lane] = s;
  __syncthreads();
  if (warp || !in) return;
#pragma unroll
  for (int w = 1; w < 8; w++) s += red[w][lane];
  if (e < n) {
    const int oc = e % (cout * cin), t = e / (cout * cin);
    gw[(size_t)oc * 27 + t] = s;
  } else {
    gb[e - n] = s;
  }
}

// The same for the input layer (one input channel): M = 16 output channels,
// N = 32 columns, the 27 taps' shifted inputs and, as column 27, ones (the
// bias), K = voxels.  The block's eight warps share a tile's K steps; slices
// [32][16] in scratch, one a block.
__global__ void __launch_bounds__(256) k_wgrad_in(Dims dm, const float* __restrict__ x, const bf16* __restrict__ gz,
                                                  int ldg, float* __restrict__ part) {
  cudaGridDependencySynchronize();
  __shared__ __align__(128) uint4 sgz[2 * WG_VOX];
  __shared__ unsigned short sxv[WG_HVOX];
  __shared__ float red[8][16][33];
  const uint32_t sg = (uint32_t)__cvta_generic_to_shared(sgz);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q = lane & 3;
  const WgTiles tl = wg_tiles(dm);
  const int ntiles = tl.count(dm.n);
  const int t0 = (int)((long long)blockIdx.x * ntiles / gridDim.x), t1 = (int)((long long)(blockIdx.x + 1) * ntiles / gridDim.x);
  const int mi = lane >> 3, mr = lane & 7;
  const uint32_t a_lane = sg + 16 * ((mi & 1) * WG_VOX + (mi >> 1) * 8 + mr);
  float acc[4][4];
  int toff[4];  // halo offset of column 8 n + g
#pragma unroll
  for (int n = 0; n < 4; n++) {
    acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
    const int t = 8 * n + g;
    toff[n] = t < 27 ? (t / 9 * WG_HY + t / 3 % 3) * WG_HX + t % 3 : 0;
  }
  for (int tile = t0; tile < t1; tile++) {
    int r = tile;
    const int x0 = (r % tl.nx) * WG_TX;
    r /= tl.nx;
    const int y0 = (r % tl.ny) * WG_TY;
    r /= tl.ny;
    const int z0 = (r % tl.nz) * WG_TZ, nn = r / tl.nz;
    __syncthreads();
    for (int i = tid; i < 2 * WG_VOX; i += 256) {
      const int v = i % WG_VOX, ch = i / WG_VOX;
      const int vx = x0 + v % WG_TX, vy = y0 + (v / WG_TX) % WG_TY, vz = z0 + v / (WG_TX * WG_TY);
      const bool in = vx < dm.w && vy < dm.h && vz < dm.d;
      const long long w = in ? voxel_at(dm, nn, vz, vy, vx) : 0;
      cp16(sg + 16 * i, gz + w * ldg + 8 * ch, in);
    }
    for (int v = tid; v < WG_HVOX; v += 256) {
      const int hx = v % WG_HX, hy = (v / WG_HX) % WG_HY, hz = v / (WG_HX * WG_HY);
      const int vx = wrap1(x0 - 1 + hx, dm.w), vy = wrap1(y0 - 1 + hy, dm.h), vz = z0 - 1 + hz;
      const bool in = vz >= 0 && vz < dm.d;
      sxv[v] = in ? __bfloat16_as_ushort(__float2bfloat16(x[voxel_at(dm, nn, vz, vy, vx)])) : (unsigned short)0;
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int e = 0; e < WG_VOX / 16 / 8; e++) {
      const int s = warp + 8 * e;
      const int vy = (2 * s) % WG_TY, vz = (2 * s) / WG_TY;
      unsigned a[4];
      ldsm4t(a, a_lane + 16 * 16 * s);
      const int base = (vz * WG_HY + vy) * WG_HX + 2 * q;
#pragma unroll
      for (int n = 0; n < 4; n++) {
        unsigned b[2];
        if (n < 3 || g < 3) {
          const unsigned short* c = sxv + base + toff[n];
          b[0] = c[0] | ((unsigned)c[1] << 16);
          b[1] = c[WG_HX] | ((unsigned)c[WG_HX + 1] << 16);
        } else {
          b[0] = b[1] = g == 3 ? 0x3F803F80u : 0u;
        }
        mma16816(acc[n], a, b);
      }
    }
  }
#pragma unroll
  for (int n = 0; n < 4; n++) {
    red[warp][g][8 * n + 2 * q] = acc[n][0];
    red[warp][g][8 * n + 2 * q + 1] = acc[n][1];
    red[warp][g + 8][8 * n + 2 * q] = acc[n][2];
    red[warp][g + 8][8 * n + 2 * q + 1] = acc[n][3];
  }
  __syncthreads();
  for (int e = tid; e < 16 * 32; e += 256) {
    const int o = e / 32, t = e % 32;
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < 8; w++) s += red[w][o][t];
    part[(size_t)blockIdx.x * 512 + t * 16 + o] = s;
  }
}
__global__ void k_wgrad_in_sum(const float* __restrict__ part, int slices, float* __restrict__ gw,
                               float* __restrict__ gb) {
  cudaGridDependencySynchronize();
  // a warp an output (28 x 16 of them): lanes stride the slices
  const int e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (e >= 28 * 16) return;
  const int t = e / 16, o = e % 16;
  float s = 0.f;
  for (int i = lane; i < slices; i += 32) s += part[(size_t)i * 512 + t * 16 + o];
  for (int k = 16; k > 0; k >>= 1) s += __shfl_xor_sync(0xffffffffu, s, k);
  if (lane == 0) (t < 27 ? gw[o * 27 + t] : gb[o]) = s;
}

// ---------------------------------------------------------------------------
// pooling, upsampling and the gradient plumbing between levels
// ---------------------------------------------------------------------------
// Pooling and upsampling move 16-byte channel vectors (c a multiple of 8,
// leading dimensions multiples of 8, so every vector is aligned), in 32-bit
// index arithmetic.  The kernels that reduce 8 fine voxels into a coarse
// one take one 8-channel vector a thread (blockIdx.y); those that write the
// fine level take one voxel a thread, all its channels (whole rows of
// stores).
// out (coarse) = mean of the 2x2x2 fine block (summed in block order); fine dims dm
__global__ void k_pool(Dims dm, const bf16* __restrict__ x, int ldx, int c, bf16* __restrict__ y, int ldy) {
  cudaGridDependencySynchronize();
  const Dims cd{dm.n, dm.d / 2, dm.h / 2, dm.w / 2};
  const unsigned V = (unsigned)cd.vox();
  if ((int)blockIdx.y * 8 >= c) return;
  for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < V; v += gridDim.x * blockDim.x) {
    const Coord q = coord_of(cd, v);
    long long f[8];
#pragma unroll
    for (int k = 0; k < 8; k++)
      f[k] = voxel_at(dm, q.n, 2 * q.z + (k >> 2), 2 * q.y + ((k >> 1) & 1), 2 * q.x + (k & 1));
    const int ch = blockIdx.y * 8;
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, e[8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
      unpack8(ld16(x + f[k] * ldx + ch), e);
#pragma unroll
      for (int i = 0; i < 8; i++) s[i] += e[i];
    }
#pragma unroll
    for (int i = 0; i < 8; i++) s[i] *= 0.125f;
    st16(y + (long long)v * ldy + ch, pack8(s));
  }
}

// fine = coarse value (nearest); coarse dims cd
__global__ void k_upsample(Dims cd, const bf16* __restrict__ x, int ldx, int c, bf16* __restrict__ y, int ldy) {
  cudaGridDependencySynchronize();
  const Dims fd{cd.n, cd.d * 2, cd.h * 2, cd.w * 2};
  const unsigned V = (unsigned)fd.vox();
  for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < V; v += gridDim.x * blockDim.x) {
    const Coord q = coord_of(fd, v);
    const long long cv = voxel_at(cd, q.n, q.z / 2, q.y / 2, q.x / 2);
    for (int ch = 0; ch < c; ch += 8) st16(y + (long long)v * ldy + ch, ld16(x + cv * ldx + ch));
  }
}

// coarse gradient of an upsample = sum over the fine block (in block
// order), times (act > 0)
__global__ void k_upsample_bwd_mask(Dims cd, const bf16* __restrict__ gf, int ldg, int c, const bf16* __restrict__ act,
                                    int lda, bf16* __restrict__ out, int ldo) {
  cudaGridDependencySynchronize();
  const Dims fd{cd.n, cd.d * 2, cd.h * 2, cd.w * 2};
  const unsigned V = (unsigned)cd.vox();
  if ((int)blockIdx.y * 8 >= c) return;
  for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < V; v += gridDim.x * blockDim.x) {
    const Coord q = coord_of(cd, v);
    long long f[8];
#pragma unroll
    for (int k = 0; k < 8; k++)
      f[k] = voxel_at(fd, q.n, 2 * q.z + (k >> 2), 2 * q.y + ((k >> 1) & 1), 2 * q.x + (k & 1));
    const int ch = blockIdx.y * 8;
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, e[8], a[8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
      unpack8(ld16(gf + f[k] * ldg + ch), e);
#pragma unroll
      for (int i = 0; i < 8; i++) s[i] += e[i];
    }
    unpack8(ld16(act + (long long)v * lda + ch), a);
#pragma unroll
    for (int i = 0; i < 8; i++) s[i] = a[i] > 0.f ? s[i] : 0.f;
    st16(out + (long long)v * ldo + ch, pack8(s));
  }
}

// fine gradient of a level's output: pool backward (coarse / 8) plus the skip
// gradient, times (act > 0); fine dims fd
__global__ void k_pool_bwd_add_mask(Dims fd, const bf16* __restrict__ gc, int ldc, const bf16* __restrict__ gskip,
                                    int lds, int c, const bf16* __restrict__ act, int lda, bf16* __restrict__ out,
                                    int ldo) {
  cudaGridDependencySynchronize();
  const Dims cd{fd.n, fd.d / 2, fd.h / 2, fd.w / 2};
  const unsigned V = (unsigned)fd.vox();
  for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < V; v += gridDim.x * blockDim.x) {
    const Coord q = coord_of(fd, v);
    const long long cv = voxel_at(cd, q.n, q.z / 2, q.y / 2, q.x / 2);
    for (int ch = 0; ch < c; ch += 8) {
      float g[8], k[8], a[8], s[8];
      unpack8(ld16(gc + cv * ldc + ch), g);
      unpack8(ld16(gskip + (long long)v * lds + ch), k);
      unpack8(ld16(act + (long long)v * lda + ch), a);
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const float t = 0.125f * g[i] + k[i];
        s[i] = a[i] > 0.f ? t : 0.f;
      }
      st16(out + (long long)v * ldo + ch, pack8(s));
    }
  }
}

// weights: master W[o][c][t] (FP32) -> wt[t][o][c] (BF16) and, for the
// backward data pass, wtt[26-t][c][o] (BF16)
__global__ void k_pack_weights(const float* __restrict__ w, int cout, int cin, bf16* __restrict__ wt,
                               bf16* __restrict__ wtt) {
  const long long total = (long long)cout * cin * 27;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
    const int t = (int)(e % 27);
    const long long oc = e / 27;
    const int c = (int)(oc % cin), o = (int)(oc / cin);
    const bf16 v = __float2bfloat16(w[e]);
    wt[((long long)t * cout + o) * cin + c] = v;
    if (wtt) wtt[((long long)(26 - t) * cin + c) * cout + o] = v;
  }
}

// wt [t][cout][cin] (BF16) -> the weights of the tcgen05 convolutions exactly as
// their shared memory holds them, so that a block loads them with bulk copies:
// 8-channel chunk j of output o, 16 bytes, at (o/8)(nch 128) + (o%8) 16 + j 128
// of its tap (nch: chunks of the group of 64 channels).  k_conv3_tc: group g,
// tap t at (27 g + t) S, S = 2 cout min(cin, 64).  k_conv3_tz (`stacked`): groups
// at 27 x 64 x 2 cout g; a (y, x) tap holds its three z taps, 2 to 0, as 3 cout
// outputs.
__global__ void k_pack_image(const bf16* __restrict__ wt, int cin, int cout, int stacked, bf16* __restrict__ img) {
  const int cg = cin < TC_CG ? cin : TC_CG, ngroups = (cin + TC_CG - 1) / TC_CG;
  const long long S = 2LL * cout * cg;
  const long long total = (long long)ngroups * 27 * cout * (cg / 8);
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(e % (cg / 8));
    long long r = e / (cg / 8);
    const int o = (int)(r % cout);
    r /= cout;
    const int t = (int)(r % 27);
    const int g = (int)(r / 27);
    const int c0 = g * TC_CG, nch = min(TC_CG, cin - c0) / 8;
    if (j >= nch) continue;
    const int row = stacked ? (2 - t / 9) * cout + o : o;
    const long long tap = stacked ? 54LL * cout * TC_CG * g + (t % 9) * (48LL * cout * nch) : (27LL * g + t) * S;
    const long long off = tap + (row / 8) * (nch * 128) + (row % 8) * 16 + j * 128;
    *reinterpret_cast<uint4*>(reinterpret_cast<char*>(img) + off) =
        *reinterpret_cast<const uint4*>(wt + ((long long)t * cout + o) * cin + c0 + 8 * j);
  }
}

// mean((y - t)^2) (block sums, added with one atomic a block) and gy = 2(y - t)/n
__global__ void __launch_bounds__(256) k_mse(long long n, const float* __restrict__ y, const float* __restrict__ t,
                                             float* __restrict__ gy, float* __restrict__ loss) {
  __shared__ float red[8];
  float s = 0.f;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float d = y[i] - t[i];
    s += d * d;
    gy[i] = 2.f * d / (float)n;
  }
  for (int k = 16; k > 0; k >>= 1) s += __shfl_xor_sync(0xffffffffu, s, k);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; w++) s += red[w];
    atomicAdd(loss, s / (float)n);
  }
}

__global__ void k_adam(long long n, float* __restrict__ th, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    th[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// per-sample sums of squares: s2[i] += sum over sample i of r^2 (blockIdx.y = sample)
__global__ void k_sample_sumsq(long long Vs, const float* __restrict__ r, float* __restrict__ s2) {
  const float* rs = r + (long long)blockIdx.y * Vs;
  float s = 0.f;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < Vs; i += (long long)gridDim.x * blockDim.x)
    s += rs[i] * rs[i];
  for (int k = 16; k > 0; k >>= 1) s += __shfl_xor_sync(0xffffffffu, s, k);
  if ((threadIdx.x & 31) == 0) atomicAdd(s2 + blockIdx.y, s);
}

// x = r / s_i and t = dp / s_i with s_i = RMS of sample i's r (0 if r = 0)
__global__ void k_scale_pairs(long long Vs, int nb, const float* __restrict__ r, const float* __restrict__ dp,
                              const float* __restrict__ s2, float kscale, float* __restrict__ x, float* __restrict__ t) {
  const long long total = Vs * nb;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
    const float rms = sqrtf(s2[e / Vs] / (float)Vs);
    const float inv = rms > 0.f ? 1.f / rms : 0.f;
    x[e] = r[e] * inv;
    if (t) t[e] = dp[e] * inv * kscale;
  }
}

// guess in the solver: x = r / s (s = ||r||_2 / sqrt(V), ||r|| read on the device)
__global__ void k_guess_in(long long V, const float* __restrict__ r, const double* __restrict__ norm,
                           float* __restrict__ x) {
  const double s = __ldcg(norm) / sqrt((double)V);
  const float inv = s > 0.0 ? (float)(1.0 / s) : 0.f;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < V; i += (long long)gridDim.x * blockDim.x)
    x[i] = r[i] * inv;
}

// d = s * y / kscale
__global__ void k_guess_out(long long V, const float* __restrict__ y, const double* __restrict__ norm, float kscale,
                            float* __restrict__ d) {
  const float s = (float)(__ldcg(norm) / sqrt((double)V)) / kscale;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < V; i += (long long)gridDim.x * blockDim.x)
    d[i] = s * y[i];
}

// FP32 -> BF16 (round to nearest even) and back, for the single-layer checks
__global__ void k_to_bf16(long long n, const float* __restrict__ a, bf16* __restrict__ b) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = __float2bfloat16_rn(a[i]);
}
__global__ void k_from_bf16(long long n, const bf16* __restrict__ a, float* __restrict__ b) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = __bfloat162float(a[i]);
}

}  // namespace nn
}  // namespace stp

// ===========================================================================
// the network object and its C ABI
// ===========================================================================
using namespace stp;
using namespace stp::nn;

namespace {

const int kCh[4] = {16, 32, 64, 128};

struct Layer {
  int cin, cout, taps;
  long long woff, boff;  // offsets of W and b in the flat parameter vector
  bf16 *wt = nullptr, *wtt = nullptr;
  // wt and wtt in the shared-memory order of the tcgen05 convolutions
  bf16 *img = nullptr, *timg = nullptr;
};

int blocks_for(long long n, int threads = 256) {
  long long b = (n + threads - 1) / threads;
  return (int)std::max<long long>(1, std::min<long long>(b, 152LL * 32));
}

}  // namespace

struct stp_unet {
  Dims dm[4];  // level dims (batch included), level 0 = full resolution
  int nmax;
  cudaStream_t st = nullptr;
  bool own_stream = false;
  std::vector<Layer> L;  // 15 layers in parameter order
  long long np = 0;
  float *theta = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
  long long adam_step = 0;
  // activations (BF16, channels-last)
  bf16 *ha[4] = {}, *e4 = nullptr, *u[3] = {}, *q[3] = {}, *hd[3] = {}, *d[3] = {};
  // gradients of activations
  bf16 *ga[4] = {}, *gb[4] = {}, *gu[3] = {};
  float *y = nullptr, *gy = nullptr, *loss = nullptr;
  float* h_loss = nullptr;  // pinned: loss, then h_err
  int* h_err = nullptr;
  float* wpart = nullptr;                                  // slices of the weight gradients (wgrad_scratch)
  float *xin = nullptr, *tin = nullptr, *snorm = nullptr;  // normalised pairs, per-sample norms
  int guess_kernels = 0;                                   // kernels launched by one guess
  float out_scale = 1.f;                                   // the network predicts out_scale * dp / s
  int* d_err = nullptr;                                    // set by a tensor-core kernel whose wait timed out
  bool use_tc = true;                                      // tcgen05 convolutions where the shapes allow
  int tc_planes = 0;                                       // planes a tcgen05 block computes (0: by layer shape)
  int mma_nt = 0;                                          // mma.sync 8-channel tiles a block (0: by grid size)
  std::vector<void*> allocs;
  std::string err;
};

namespace {

// The network's kernels are launched as programmatic dependents (launch_dep): a
// forward has 21 launches, a gradient 57, with gaps of 2 to 3 us between plain
// ones: 527 us a forward of 128 x 64 x 128 and 1516 a gradient of 4 x 64 x 32 x
// 64, 471 and 1362 this way (some 10 us of each by reading the error flag with the
// results).

int ufail(stp_unet* n, int code, const std::string& m) {
  if (n) n->err = m;
  return code;
}

#define UTRY(n, call)                                                                                  \
  do {                                                                                                 \
    cudaError_t e_ = (call);                                                                           \
    if (e_ != cudaSuccess) return ufail(n, STP_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

// synchronises; did a tensor-core convolution give up waiting?
int check_tc_timeout(stp_unet* n) {
  UTRY(n, cudaMemcpyAsync(n->h_err, n->d_err, sizeof(int), cudaMemcpyDeviceToHost, n->st));
  UTRY(n, cudaStreamSynchronize(n->st));
  if (*n->h_err) return ufail(n, STP_ETIMEOUT, "a tensor-core convolution timed out waiting for its MMAs");
  return STP_OK;
}

template <typename T>
int ualloc(stp_unet* n, T** p, size_t count) {
  cudaError_t e = cudaMalloc((void**)p, sizeof(T) * std::max<size_t>(count, 1));
  if (e != cudaSuccess) return ufail(n, STP_ENOMEM, "cudaMalloc failed in the network");
  n->allocs.push_back(*p);
  return STP_OK;
}

// concat widths: decoder level l (0..2) input = kCh[l+1] + kCh[l]
int cu_width(int l) { return kCh[l + 1] + kCh[l]; }

constexpr size_t kTcSmemMax = 200 * 1024;  // of the mma.sync convolution
constexpr size_t kTcSmemSm = 225 * 1024;   // of an SM's blocks of a tcgen05 convolution

// weights image of k_conv3_tc, elements
size_t tc_image_elems(int cin, int cout) {
  return (size_t)((cin + TC_CG - 1) / TC_CG) * 27 * cout * std::min(cin, TC_CG);
}

// Weights beside two halo planes in an SM's shared memory: k_conv3_tz.
bool tz_takes(int cin, int cout) {
  return cin % 16 == 0 && cout % 16 == 0 && cout <= 256 && cin <= TC_CG * TZ_GROUPS &&
         (size_t)54 * cin * cout + 2 * (size_t)(std::min(cin, TC_CG) / 8) * TC_PLANE <= kTcSmemSm;
}

// How k_conv3_tz runs a layer it takes: planes a tile (8, 4, 2 or 1; an MMA's N
// = 3 cout, or fewer planes', at most 256) and blocks an SM (2 or 1), the pair
// with the fewest plane loads on the busiest SM, a lone block's counted at 6/5
// (one thread issues MMAs at 58 clocks, two blocks' at 49 together).  Two
// accumulator stages where the columns allow.  A forced count of planes
// (STP_UNET_TC_PLANES: 1, 2 or 4) is halved until it fits.
TzPlan tz_plan(const stp_unet* n, const Dims& dm, int cin, int cout) {
  const size_t plane = (size_t)(std::min(cin, TC_CG) / 8) * TC_PLANE, w = (size_t)54 * cin * cout;
  const long long tiles = dm.vox() / (TC_TX * TC_TY);
  const bool forced = n->tc_planes == 1 || n->tc_planes == 2 || n->tc_planes == 4;
  TzPlan best{};
  long long cost = 0;
  for (int zt = forced ? n->tc_planes : 8; zt >= 1; zt /= 2) {
    if (dm.d % zt || std::min(zt, 3) * cout > 256) continue;
    for (int per_sm = 2; per_sm >= 1; per_sm--) {
      const size_t room = per_sm == 2 ? kTcSmemSm / 2 - 2048 : kTcSmemSm;
      TzPlan p;
      p.zt = zt;
      p.per_sm = per_sm;
      if (w + 2 * plane > room || zt * cout > 512 / per_sm) continue;
      p.hs = (int)std::min<size_t>(TZ_HALO, (room - w) / plane);
      p.as = 2 * zt * cout <= 512 / per_sm ? 2 : 1;
      p.cols = 32;
      while (p.cols < p.as * zt * cout) p.cols *= 2;
      p.smem = w + p.hs * plane;
      const long long blocks = 152LL * per_sm, rounds = (tiles / zt + blocks - 1) / blocks;
      const long long c = rounds * (zt + 2 + (p.as == 1 && per_sm == 1 ? zt : 0)) * (per_sm == 2 ? 10 : 6);
      if (best.zt == 0 || c < cost) best = p, cost = c;
    }
    if (forced && best.zt) break;
  }
  return best;
}

// How k_conv3_tc runs a layer; false if it does not take it.  A ring of 96 KB of
// weights, at least two stages of three taps, and one halo stage (a second does
// not fit beside it).  Planes a tile 2 or 1, two if they leave two tiles an SM
// (planes share halo planes: 4 loaded for 2 computed) and the accumulators'
// columns allow; two accumulator stages in 256 columns, else one.  A forced count
// as above.
bool tc_plan(const stp_unet* n, const Dims& dm, int cin, int cout, TcPlan* out) {
  if (cin % TC_CG) return false;
  const size_t stage = (size_t)2 * TC_STAPS * cout * TC_CG;
  const long long tiles = dm.vox() / (TC_TX * TC_TY);
  const bool forced = n->tc_planes == 1 || n->tc_planes == 2 || n->tc_planes == 4;
  for (int zt = 2; zt >= 1; zt--) {
    if (forced ? zt > n->tc_planes : zt > 1 && tiles / zt < 2 * 152) continue;
    if (dm.d % zt || zt * cout > 256) continue;
    TcPlan p;
    p.zt = zt;
    p.ring = (int)std::min<size_t>(TC_RING, std::max<size_t>(2, 96 * 1024 / stage));
    p.as = 2 * zt * cout <= 256 ? 2 : 1;
    p.cols = 32;
    while (p.cols < p.as * zt * cout) p.cols *= 2;
    p.smem = (size_t)(TC_CG / 8) * TC_PLANE * (zt + 2) + p.ring * stage;
    if (p.smem > kTcSmemSm) continue;
    *out = p;
    return true;
  }
  return false;
}

bool conv3_tc_ok(const stp_unet* n, const Dims& dm, int ldx, int cin, int cout, int ldy, int ldm, TcPlan* p) {
  return n->use_tc && dm.w % TC_TX == 0 && dm.h % TC_TY == 0 && cin % 16 == 0 && cout % 16 == 0 && cout <= 256 &&
         ldx % 8 == 0 && ldy % 16 == 0 && ldm % 8 == 0 && (tz_takes(cin, cout) || tc_plan(n, dm, cin, cout, p));
}

// launch a 3x3x3 convolution (forward form): tcgen05 where the shapes allow, else mma.sync
int conv3(stp_unet* n, const Dims& dm, const bf16* x, int ldx, int cin, const bf16* wt, const bf16* wimg,
          const float* bias, int cout, bf16* y, int ldy, int relu, const bf16* mask, int ldm) {
  const long long V = dm.vox();
  TcPlan p;
  if (conv3_tc_ok(n, dm, ldx, cin, cout, ldy, ldm, &p)) {
    if (tz_takes(cin, cout)) {
      static std::atomic<unsigned> donez{0u};
      UTRY(n, smem_limit_once(k_conv3_tz, (int)kTcSmemSm, donez));
      const TzPlan z = tz_plan(n, dm, cin, cout);
      const unsigned tiles = (unsigned)(V / (TC_TX * TC_TY * z.zt));
      UTRY(n, launch_dep(k_conv3_tz, std::min(tiles, 152u * z.per_sm), TZ_THREADS, z.smem, n->st, dm, x, ldx, cin, wimg,
                         bias, cout, y, ldy, relu, mask, ldm, z, n->d_err));
      return STP_OK;
    }
    const unsigned tiles = (unsigned)(V / (TC_TX * TC_TY * p.zt));
    auto go = [&](auto kern, std::atomic<unsigned>& done) -> cudaError_t {
      if (cudaError_t e = smem_limit_once(kern, (int)kTcSmemSm, done)) return e;
      return launch_dep(kern, std::min(tiles, 152u), TC_THREADS, p.smem, n->st, dm, x, ldx, cin, wimg, bias,
                        cout, y, ldy, relu, mask, ldm, p, n->d_err);
    };
    static std::atomic<unsigned> done1{0u}, done2{0u};
    UTRY(n, p.zt == 2 ? go(k_conv3_tc<2>, done2) : go(k_conv3_tc<1>, done1));
    return STP_OK;
  }
  // output channels a block: 32, 16 or 8, the widest that still gives 100
  // blocks; each output sees the same sequence of MMAs whichever width
  // computes it (STP_UNET_MMA_NT = 8, 4, 2 or 1 asks for a width, 8 as 4).
  // Resident weights when they fit and the blocks are one wave of the GPU.
  const long long tiles = (long long)dm.n * ((dm.w + CS_TX - 1) / CS_TX) * ((dm.h + CS_TY - 1) / CS_TY) *
                          ((dm.d + CS_TZ - 1) / CS_TZ);
  const bool forced = n->mma_nt == 8 || n->mma_nt == 4 || n->mma_nt == 2 || n->mma_nt == 1;
  int nt = forced ? std::min(n->mma_nt, 4) : 4;
  while (nt > 1 && (cout % (8 * nt) || (!forced && tiles * (cout / (8 * nt)) < 100))) nt /= 2;
  const long long blocks = tiles * (cout / (8 * nt));
  const bool ring = !(conv3_smem(cin, nt, false) <= kTcSmemMax && (conv3_smem(cin, nt, false) <= 56 * 1024 || blocks <= 152));
  auto go = [&](auto kern, std::atomic<unsigned>& done) -> cudaError_t {
    if (cudaError_t e = smem_limit_once(kern, (int)kTcSmemMax, done)) return e;
    return launch_dep(kern, dim3((unsigned)tiles, (unsigned)(cout / (8 * nt))), 128, conv3_smem(cin, nt, ring), n->st,
                      dm, x, ldx, cin, wt, bias, cout, y, ldy, relu, mask, ldm);
  };
  static std::atomic<unsigned> done[6];
  if (ring)
    UTRY(n, nt == 4 ? go(k_conv3<4, true>, done[0]) : nt == 2 ? go(k_conv3<2, true>, done[1]) : go(k_conv3<1, true>, done[2]));
  else
    UTRY(n, nt == 4 ? go(k_conv3<4, false>, done[3]) : nt == 2 ? go(k_conv3<2, false>, done[4]) : go(k_conv3<1, false>, done[5]));
  return STP_OK;
}

// slices of a layer's weight gradient: enough blocks for two a SM, at most one
// tile each, and at most the scratch
int wgrad_tile(int c) { return c % 32 == 0 ? 32 : 16; }
// input channels a block: with 16 outputs all of 48 (gz is then read once)
int wgrad_ctile(int cin, int cout) { return cin == 48 && wgrad_tile(cout) == 16 ? 48 : wgrad_tile(cin); }
constexpr size_t kWgradScratch = (size_t)6 << 20;  // floats at most
int wgrad_slices(const Dims& dm, int cin, int cout) {
  const long long pairs = (long long)(cin / wgrad_ctile(cin, cout)) * (cout / wgrad_tile(cout));
  const long long tiles = wg_tiles(dm).count(dm.n);
  long long s = std::max<long long>(1, (2 * 152 + pairs - 1) / pairs);
  s = std::min(s, (long long)(kWgradScratch / ((size_t)WG_SLOTS * cin * cout)));
  return (int)std::max<long long>(1, std::min(s, tiles));
}

int wgrad_in_slices(const Dims& dm) { return std::min(wg_tiles(dm).count(dm.n), 4 * 152); }
// floats of the slices of the largest weight gradient of a network (smaller
// batches have no more tiles, so no more slices)
size_t wgrad_scratch(const stp_unet* n) {
  size_t need = (size_t)512 * wgrad_in_slices(n->dm[0]);
  for (int i = 1; i < 14; i++) {
    const Layer& ly = n->L[i];
    const Dims& dm = n->dm[i < 8 ? i / 2 : 2 - (i - 8) / 2];
    need = std::max(need, (size_t)WG_SLOTS * ly.cin * ly.cout * wgrad_slices(dm, ly.cin, ly.cout));
  }
  return need;
}

template <int OT, int CT>
cudaError_t wgrad_launch(const Dims& dm, const bf16* x, int ldx, int cin, const bf16* gz, int ldg, int cout, float* part,
                         int slices, cudaStream_t st) {
  static std::atomic<unsigned> done{0u};
  if (cudaError_t e = smem_limit_once(k_wgrad3<OT, CT>, wg_smem(OT, CT), done)) return e;
  return launch_dep(k_wgrad3<OT, CT>, dim3((unsigned)((cin / CT) * (cout / OT)), (unsigned)slices), 288,
                    wg_smem(OT, CT), st, dm, x, ldx, cin, gz, ldg, cout, part);
}

// weight and bias gradient of a 3x3x3 layer, stored (not added) into n->grad
int wgrad3(stp_unet* n, const Dims& dm, const bf16* x, int ldx, int cin, const bf16* gz, int ldg, int cout,
           const Layer& ly) {
  const int slices = wgrad_slices(dm, cin, cout);
  const int ot = wgrad_tile(cout), ct = wgrad_ctile(cin, cout);
  if (ot == 32)
    UTRY(n, (ct == 32 ? wgrad_launch<32, 32> : wgrad_launch<32, 16>)(dm, x, ldx, cin, gz, ldg, cout, n->wpart, slices, n->st));
  else
    UTRY(n, (ct == 48 ? wgrad_launch<16, 48> : ct == 32 ? wgrad_launch<16, 32> : wgrad_launch<16, 16>)(dm, x, ldx, cin, gz, ldg, cout, n->wpart, slices, n->st));
  const int total = 27 * cin * cout + cout;
  UTRY(n, launch_dep(k_wgrad_sum, (total + 31) / 32, 256, 0, n->st, n->wpart, slices, cin, cout, n->grad + ly.woff,
                     n->grad + ly.boff));
  return STP_OK;
}
int wgrad_in(stp_unet* n, const Dims& dm, const float* x, const bf16* gz, int ldg, const Layer& ly) {
  const int slices = wgrad_in_slices(dm);
  UTRY(n, launch_dep(k_wgrad_in, slices, 256, 0, n->st, dm, x, gz, ldg, n->wpart));
  UTRY(n, launch_dep(k_wgrad_in_sum, (28 * 16 * 32 + 127) / 128, 128, 0, n->st, n->wpart, slices, n->grad + ly.woff,
                     n->grad + ly.boff));
  return STP_OK;
}

int pack_all(stp_unet* n) {
  for (size_t i = 0; i < n->L.size(); i++) {
    Layer& ly = n->L[i];
    if (ly.taps != 27 || ly.cin == 1) continue;
    const long long tot = (long long)ly.cout * ly.cin * 27;
    k_pack_weights<<<blocks_for(tot), 256, 0, n->st>>>(n->theta + ly.woff, ly.cout, ly.cin, ly.wt, ly.wtt);
    UTRY(n, cudaGetLastError());
    k_pack_image<<<blocks_for(tot / 8), 256, 0, n->st>>>(ly.wt, ly.cin, ly.cout, tz_takes(ly.cin, ly.cout), ly.img);
    k_pack_image<<<blocks_for(tot / 8), 256, 0, n->st>>>(ly.wtt, ly.cout, ly.cin, tz_takes(ly.cout, ly.cin), ly.timg);
    UTRY(n, cudaGetLastError());
  }
  return STP_OK;
}

// forward of nb samples; x [nb][D][H][W] FP32 on the device
int forward(stp_unet* n, const float* x, int nb) {
  Dims dm[4];
  for (int l = 0; l < 4; l++) dm[l] = Dims{nb, n->dm[l].d, n->dm[l].h, n->dm[l].w};
  int rc;
  // encoder
  const Layer* P = n->L.data();
  // level 1: input layer, second conv writes e1 into u[0][:, 32:48]
  k_conv_in<<<blocks_for(dm[0].vox() / 4, 128), 128, 0, n->st>>>(dm[0], x, n->theta + P[0].woff, n->theta + P[0].boff, n->ha[0],
                                                         16);
  UTRY(n, cudaGetLastError());
  const bf16* in = nullptr;
  int ldin = 0;
  for (int l = 0; l < 4; l++) {
    const int c = kCh[l];
    const Layer& la = P[2 * l];
    const Layer& lb = P[2 * l + 1];
    if (l > 0) {
      if ((rc = conv3(n, dm[l], in, ldin, la.cin, la.wt, la.img, n->theta + la.boff, c, n->ha[l], c, 1, nullptr, 0))) return rc;
    }
    bf16* e = l < 3 ? n->u[l] + kCh[l + 1] : n->e4;
    const int lde = l < 3 ? cu_width(l) : c;
    if ((rc = conv3(n, dm[l], n->ha[l], c, c, lb.wt, lb.img, n->theta + lb.boff, c, e, lde, 1, nullptr, 0))) return rc;
    if (l < 3) {
      UTRY(n, launch_dep(k_pool, dim3(blocks_for(dm[l + 1].vox()), c / 8), 256, 0, n->st, dm[l], e, lde, c, n->q[l],
                         c));
      in = n->q[l];
      ldin = c;
    }
  }
  // decoder
  const bf16* deeper = n->e4;
  int cdeep = kCh[3];
  for (int l = 2; l >= 0; l--) {
    const int c = kCh[l], cw = cu_width(l);
    UTRY(n, launch_dep(k_upsample, blocks_for(dm[l].vox()), 256, 0, n->st, dm[l + 1], deeper, cdeep, cdeep, n->u[l],
                       cw));
    const Layer& la = P[8 + 2 * (2 - l)];
    const Layer& lb = P[9 + 2 * (2 - l)];
    if ((rc = conv3(n, dm[l], n->u[l], cw, cw, la.wt, la.img, n->theta + la.boff, c, n->hd[l], c, 1, nullptr, 0))) return rc;
    if ((rc = conv3(n, dm[l], n->hd[l], c, c, lb.wt, lb.img, n->theta + lb.boff, c, n->d[l], c, 1, nullptr, 0))) return rc;
    deeper = n->d[l];
    cdeep = c;
  }
  const Layer& lo = P[14];
  UTRY(n, launch_dep(k_conv_out, blocks_for(dm[0].vox()), 256, 0, n->st, dm[0].vox(), n->d[0], 16, n->theta + lo.woff,
                     n->theta + lo.boff, n->y));
  return STP_OK;
}

// backward from gy (FP32 [V0]) into n->grad: the 3x3x3 layers store theirs, the
// output layer's, the last 17 values, is zeroed here and added into
int backward(stp_unet* n, const float* x, int nb) {
  Dims dm[4];
  for (int l = 0; l < 4; l++) dm[l] = Dims{nb, n->dm[l].d, n->dm[l].h, n->dm[l].w};
  const Layer* P = n->L.data();
  int rc;
  // output layer -> gradient of the pre-activation of d1 (ga[0])
  const Layer& lo = P[14];
  UTRY(n, cudaMemsetAsync(n->grad + lo.woff, 0, sizeof(float) * (n->np - lo.woff), n->st));
  UTRY(n, launch_dep(k_conv_out_bwd, blocks_for(dm[0].vox()), 256, 0, n->st, dm[0].vox(), n->gy, n->d[0], 16,
                     n->theta + lo.woff, n->ga[0], 16, n->grad + lo.woff, n->grad + lo.boff));
  // decoder, level 0 up to 2; ga[l] holds the gradient of d_l's pre-activation
  for (int l = 0; l <= 2; l++) {
    const int c = kCh[l], cw = cu_width(l);
    const Layer& la = P[8 + 2 * (2 - l)];
    const Layer& lb = P[9 + 2 * (2 - l)];
    // conv b: input hd[l], gradient ga[l]
    if ((rc = wgrad3(n, dm[l], n->hd[l], c, c, n->ga[l], c, c, lb))) return rc;
    if ((rc = conv3(n, dm[l], n->ga[l], c, c, lb.wtt, lb.timg, nullptr, c, n->gb[l], c, 0, n->hd[l], c))) return rc;
    // conv a: input u[l], gradient gb[l]
    if ((rc = wgrad3(n, dm[l], n->u[l], cw, cw, n->gb[l], c, c, la))) return rc;
    if ((rc = conv3(n, dm[l], n->gb[l], c, c, la.wtt, la.timg, nullptr, cw, n->gu[l], cw, 0, nullptr, 0))) return rc;
    // upsample part -> gradient of the deeper level's output pre-activation
    const int cd = kCh[l + 1];
    const bf16* act = l < 2 ? n->d[l + 1] : n->e4;
    bf16* out = l < 2 ? n->ga[l + 1] : n->ga[3];
    UTRY(n, launch_dep(k_upsample_bwd_mask, dim3(blocks_for(dm[l + 1].vox()), cd / 8), 256, 0, n->st, dm[l + 1],
                       n->gu[l], cw, cd, act, cd, out, cd));
  }
  // encoder, level 3 down to 0.  Buffers at level l: gz (gradient of e_l's
  // pre-activation), gha (of ha_l's), gq (of q_{l-1}, handed to level l-1).
  //   l = 3: gz = ga[3] (from the decoder), gha = gb[3], gq = ga[3]
  //   l < 3: gz = gb[l], gha = ga[l], gq = gb[l]
  // each is overwritten only after its last reader has run.
  const bf16* gq_in = nullptr;
  for (int l = 3; l >= 0; l--) {
    const int c = kCh[l];
    const Layer& la = P[2 * l];
    const Layer& lb = P[2 * l + 1];
    bf16* gz = l == 3 ? n->ga[3] : n->gb[l];
    if (l < 3) {
      // gz = (pool backward of the gradient of q_l + skip gradient) * (e_l > 0)
      const bf16* e = n->u[l] + kCh[l + 1];
      UTRY(n, launch_dep(k_pool_bwd_add_mask, blocks_for(dm[l].vox()), 256, 0, n->st, dm[l], gq_in, c,
                         n->gu[l] + kCh[l + 1], cu_width(l), c, e, cu_width(l), gz, c));
    }
    // conv b: input ha[l]
    if ((rc = wgrad3(n, dm[l], n->ha[l], c, c, gz, c, c, lb))) return rc;
    bf16* gha = l == 3 ? n->gb[3] : n->ga[l];
    if ((rc = conv3(n, dm[l], gz, c, c, lb.wtt, lb.timg, nullptr, c, gha, c, 0, n->ha[l], c))) return rc;
    if (l > 0) {
      // conv a: input q[l-1]
      const int cp = kCh[l - 1];
      if ((rc = wgrad3(n, dm[l], n->q[l - 1], cp, cp, gha, c, c, la))) return rc;
      bf16* gq = l == 3 ? n->ga[3] : n->gb[l];
      if ((rc = conv3(n, dm[l], gha, c, c, la.wtt, la.timg, nullptr, cp, gq, cp, 0, nullptr, 0))) return rc;
      gq_in = gq;
    } else {
      // conv a of level 1: the network input (1 channel)
      if ((rc = wgrad_in(n, dm[0], x, gha, c, la))) return rc;
    }
  }
  return STP_OK;
}

int check_n(stp_unet* n, int nb) {
  if (nb < 1 || nb > n->nmax) return ufail(n, STP_EINVAL, "batch size out of range");
  return STP_OK;
}

}  // namespace

namespace stp {

bool unet_matches(const stp_unet* n, int nz, int ny, int nx) {
  return n && n->dm[0].d == nz && n->dm[0].h == ny && n->dm[0].w == nx;
}

// d = s U(r / s) for one sample on stream st, s = norm / sqrt(V) with the
// norm read on the device; launches only (no synchronisation), so it can be
// captured into a graph.  Returns the number of kernels through *kernels.
int unet_guess(stp_unet* n, const float* r, const double* norm, float* d, cudaStream_t st, int* kernels) {
  cudaStream_t keep = n->st;
  n->st = st;
  const long long V = n->dm[0].vox() / n->nmax;
  int rc = STP_OK;
  k_guess_in<<<blocks_for(V), 256, 0, st>>>(V, r, norm, n->xin);
  if (cudaGetLastError() != cudaSuccess) rc = STP_ECUDA;
  if (rc == STP_OK) rc = forward(n, n->xin, 1);
  if (rc == STP_OK) {
    k_guess_out<<<blocks_for(V), 256, 0, st>>>(V, n->y, norm, n->out_scale, d);
    if (cudaGetLastError() != cudaSuccess) rc = STP_ECUDA;
  }
  n->st = keep;
  // scale in and out + the forward pass: input layer, 7 further encoder
  // convolutions, 3 pools, 3 upsamplings, 6 decoder convolutions, output layer
  if (kernels) *kernels = 2 + 21;
  return rc;
}

}  // namespace stp

extern "C" {

long long stp_unet_param_count(void) {
  long long np = 0;
  int cin = 1;
  for (int l = 0; l < 4; l++) {
    np += 27LL * cin * kCh[l] + kCh[l] + 27LL * kCh[l] * kCh[l] + kCh[l];
    cin = kCh[l];
  }
  for (int l = 2; l >= 0; l--) np += 27LL * cu_width(l) * kCh[l] + kCh[l] + 27LL * kCh[l] * kCh[l] + kCh[l];
  return np + 16 + 1;
}

int stp_unet_create(int nmax, int nz, int ny, int nx, void* stream, stp_unet** out) {
  if (!out) return STP_EINVAL;
  *out = nullptr;
  if (nmax < 1 || nz < 8 || ny < 8 || nx < 8 || nz % 8 || ny % 8 || nx % 8) return STP_EINVAL;
  if ((double)nmax * nz * ny * nx > 2147483647.0) return STP_EINVAL;  // voxel indices are 32-bit
  stp_unet* n = new stp_unet();
  n->nmax = nmax;
  for (int l = 0; l < 4; l++) n->dm[l] = Dims{nmax, nz >> l, ny >> l, nx >> l};
  if (stream) {
    n->st = (cudaStream_t)stream;
  } else {
    if (cudaStreamCreateWithFlags(&n->st, cudaStreamNonBlocking) != cudaSuccess) {
      delete n;
      return STP_ECUDA;
    }
    n->own_stream = true;
  }
  // layers in parameter order
  long long q = 0;
  auto add = [&](int ci, int co, int taps) {
    Layer ly;
    ly.cin = ci;
    ly.cout = co;
    ly.taps = taps;
    ly.woff = q;
    q += (long long)co * ci * taps;
    ly.boff = q;
    q += co;
    n->L.push_back(ly);
  };
  int cin = 1;
  for (int l = 0; l < 4; l++) {
    add(cin, kCh[l], 27);
    add(kCh[l], kCh[l], 27);
    cin = kCh[l];
  }
  for (int l = 2; l >= 0; l--) {
    add(cu_width(l), kCh[l], 27);
    add(kCh[l], kCh[l], 27);
  }
  add(16, 1, 1);
  n->np = q;
  int rc = STP_OK;
  auto A = [&](auto** p, size_t count) {
    if (rc == STP_OK) rc = ualloc(n, p, count);
  };
  A(&n->theta, n->np);
  A(&n->grad, n->np);
  A(&n->m, n->np);
  A(&n->v, n->np);
  for (Layer& ly : n->L) {
    if (ly.taps == 27 && ly.cin > 1) {
      A(&ly.wt, (size_t)ly.cout * ly.cin * 27);
      A(&ly.wtt, (size_t)ly.cout * ly.cin * 27);
      A(&ly.img, tc_image_elems(ly.cin, ly.cout));
      A(&ly.timg, tc_image_elems(ly.cout, ly.cin));
    }
  }
  const long long V[4] = {n->dm[0].vox(), n->dm[1].vox(), n->dm[2].vox(), n->dm[3].vox()};
  for (int l = 0; l < 4; l++) {
    A(&n->ha[l], (size_t)V[l] * kCh[l]);
    A(&n->ga[l], (size_t)V[l] * kCh[l]);
    A(&n->gb[l], (size_t)V[l] * kCh[l]);
  }
  A(&n->e4, (size_t)V[3] * kCh[3]);
  for (int l = 0; l < 3; l++) {
    A(&n->u[l], (size_t)V[l] * cu_width(l));
    A(&n->gu[l], (size_t)V[l] * cu_width(l));
    A(&n->q[l], (size_t)V[l + 1] * kCh[l]);
    A(&n->hd[l], (size_t)V[l] * kCh[l]);
    A(&n->d[l], (size_t)V[l] * kCh[l]);
  }
  A(&n->y, (size_t)V[0]);
  A(&n->xin, (size_t)V[0]);
  A(&n->tin, (size_t)V[0]);
  A(&n->snorm, (size_t)nmax);
  A(&n->gy, (size_t)V[0]);
  A(&n->loss, 1);
  A(&n->wpart, wgrad_scratch(n));
  A(&n->d_err, 1);
  if (const char* e = std::getenv("STP_UNET_TC")) n->use_tc = std::atoi(e) != 0;
  if (const char* e = std::getenv("STP_UNET_TC_PLANES")) n->tc_planes = std::atoi(e);
  if (const char* e = std::getenv("STP_UNET_MMA_NT")) n->mma_nt = std::atoi(e);
  if (rc == STP_OK && cudaMallocHost((void**)&n->h_loss, sizeof(float) + sizeof(int)) != cudaSuccess) rc = STP_ENOMEM;
  if (rc == STP_OK) n->h_err = reinterpret_cast<int*>(n->h_loss + 1);
  if (rc == STP_OK) {
    cudaMemsetAsync(n->theta, 0, sizeof(float) * n->np, n->st);
    cudaMemsetAsync(n->m, 0, sizeof(float) * n->np, n->st);
    cudaMemsetAsync(n->v, 0, sizeof(float) * n->np, n->st);
    cudaMemsetAsync(n->d_err, 0, sizeof(int), n->st);
    if (cudaStreamSynchronize(n->st) != cudaSuccess) rc = STP_ECUDA;
  }
  if (rc != STP_OK) {
    stp_unet_destroy(n);
    return rc;
  }
  *out = n;
  return STP_OK;
}

void stp_unet_destroy(stp_unet* n) {
  if (!n) return;
  if (n->st) cudaStreamSynchronize(n->st);
  for (void* p : n->allocs) cudaFree(p);
  if (n->h_loss) cudaFreeHost(n->h_loss);
  if (n->own_stream && n->st) cudaStreamDestroy(n->st);
  delete n;
}

const char* stp_unet_last_error(const stp_unet* n) { return n ? n->err.c_str() : ""; }

int stp_unet_set_params(stp_unet* n, const float* theta, int where) {
  if (!n || !theta) return STP_EINVAL;
  UTRY(n, cudaMemcpyAsync(n->theta, theta, sizeof(float) * n->np,
                          where == STP_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, n->st));
  UTRY(n, cudaMemsetAsync(n->m, 0, sizeof(float) * n->np, n->st));
  UTRY(n, cudaMemsetAsync(n->v, 0, sizeof(float) * n->np, n->st));
  n->adam_step = 0;
  int rc = pack_all(n);
  if (rc) return rc;
  UTRY(n, cudaStreamSynchronize(n->st));
  return STP_OK;
}

int stp_unet_get_params(stp_unet* n, float* theta, int where) {
  if (!n || !theta) return STP_EINVAL;
  UTRY(n, cudaMemcpyAsync(theta, n->theta, sizeof(float) * n->np,
                          where == STP_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, n->st));
  UTRY(n, cudaStreamSynchronize(n->st));
  return STP_OK;
}

int stp_unet_forward(stp_unet* n, const float* x, float* y, int nb) {
  if (!n || !x || !y) return STP_EINVAL;
  if (int rc = check_n(n, nb)) return rc;
  int rc = forward(n, x, nb);
  if (rc) return rc;
  UTRY(n, cudaMemcpyAsync(y, n->y, sizeof(float) * n->dm[0].vox() / n->nmax * nb, cudaMemcpyDeviceToDevice, n->st));
  return check_tc_timeout(n);
}

int stp_unet_gradient(stp_unet* n, const float* x, const float* target, int nb, float* grad, float* loss) {
  if (!n || !x || !target) return STP_EINVAL;
  if (int rc = check_n(n, nb)) return rc;
  int rc = forward(n, x, nb);
  if (rc) return rc;
  const long long V = n->dm[0].vox() / n->nmax * nb;
  UTRY(n, cudaMemsetAsync(n->loss, 0, sizeof(float), n->st));
  k_mse<<<std::min(blocks_for(V), 4 * 152), 256, 0, n->st>>>(V, n->y, target, n->gy, n->loss);
  UTRY(n, cudaGetLastError());
  if ((rc = backward(n, x, nb))) return rc;
  if (grad) UTRY(n, cudaMemcpyAsync(grad, n->grad, sizeof(float) * n->np, cudaMemcpyDeviceToDevice, n->st));
  UTRY(n, cudaMemcpyAsync(n->h_loss, n->loss, sizeof(float), cudaMemcpyDeviceToHost, n->st));
  rc = check_tc_timeout(n);
  if (loss && (rc == STP_OK || rc == STP_ETIMEOUT)) *loss = *n->h_loss;
  return rc;
}

int stp_unet_train_step(stp_unet* n, const float* x, const float* target, int nb, float lr, float* loss) {
  int rc = stp_unet_gradient(n, x, target, nb, nullptr, loss);
  if (rc) return rc;
  n->adam_step++;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)n->adam_step), c2 = 1.f - std::pow(b2, (float)n->adam_step);
  k_adam<<<blocks_for(n->np), 256, 0, n->st>>>(n->np, n->theta, n->grad, n->m, n->v, lr, b1, b2, 1e-8f, c1, c2);
  UTRY(n, cudaGetLastError());
  if ((rc = pack_all(n))) return rc;
  UTRY(n, cudaStreamSynchronize(n->st));
  return STP_OK;
}

int stp_unet_layer(stp_unet* n, int layer, int mode, const float* a, const float* b, float* out, int nb) {
  if (!n || !a || !out) return STP_EINVAL;
  if (int rc = check_n(n, nb)) return rc;
  if (layer < 0 || layer > 13) return ufail(n, STP_EINVAL, "layer must be 0..13 (the 3x3x3 convolutions)");
  if (mode < 0 || mode > 2 || (mode == 1 && layer == 0)) return ufail(n, STP_EINVAL, "bad mode for this layer");
  if (mode == 2 && !b) return ufail(n, STP_EINVAL, "the weight gradient needs gz");
  const Layer& ly = n->L[layer];
  const int lev = layer < 8 ? layer / 2 : 2 - (layer - 8) / 2;
  const Dims dm{nb, n->dm[lev].d, n->dm[lev].h, n->dm[lev].w};
  const long long V = dm.vox();
  const int ci = ly.cin, co = ly.cout;
  // temporaries: BF16 copies of the inputs and the BF16 output
  bf16 *xa = nullptr, *xb = nullptr, *y = nullptr;
  std::vector<void*> tmp;
  auto talloc = [&](bf16** p, long long count) -> int {
    if (cudaMalloc((void**)p, sizeof(bf16) * std::max<long long>(count, 1)) != cudaSuccess) return STP_ENOMEM;
    tmp.push_back(*p);
    return STP_OK;
  };
  auto done = [&](int rc) {
    cudaStreamSynchronize(n->st);
    for (void* p : tmp) cudaFree(p);
    return rc;
  };
  int rc = STP_OK;
  if (mode == 0) {
    if (layer == 0) {
      if ((rc = talloc(&y, V * co))) return done(ufail(n, rc, "cudaMalloc failed"));
      k_conv_in<<<blocks_for(V / 4, 128), 128, 0, n->st>>>(dm, a, n->theta + ly.woff, n->theta + ly.boff, y, co);
      if (cudaGetLastError() != cudaSuccess) return done(ufail(n, STP_ECUDA, "k_conv_in launch failed"));
    } else {
      if ((rc = talloc(&xa, V * ci)) || (rc = talloc(&y, V * co))) return done(ufail(n, rc, "cudaMalloc failed"));
      k_to_bf16<<<blocks_for(V * ci), 256, 0, n->st>>>(V * ci, a, xa);
      if ((rc = conv3(n, dm, xa, ci, ci, ly.wt, ly.img, n->theta + ly.boff, co, y, co, 1, nullptr, 0)))
        return done(rc);
    }
    k_from_bf16<<<blocks_for(V * co), 256, 0, n->st>>>(V * co, y, out);
  } else if (mode == 1) {
    if ((rc = talloc(&xa, V * co)) || (rc = talloc(&y, V * ci)) || (b && (rc = talloc(&xb, V * ci))))
      return done(ufail(n, rc, "cudaMalloc failed"));
    k_to_bf16<<<blocks_for(V * co), 256, 0, n->st>>>(V * co, a, xa);
    if (b) k_to_bf16<<<blocks_for(V * ci), 256, 0, n->st>>>(V * ci, b, xb);
    if ((rc = conv3(n, dm, xa, co, co, ly.wtt, ly.timg, nullptr, ci, y, ci, 0, xb, xb ? ci : 0))) return done(rc);
    k_from_bf16<<<blocks_for(V * ci), 256, 0, n->st>>>(V * ci, y, out);
  } else {
    UTRY(n, cudaMemsetAsync(n->grad + ly.woff, 0, sizeof(float) * ((long long)co * ci * 27 + co), n->st));
    if ((rc = talloc(&xb, V * co))) return done(ufail(n, rc, "cudaMalloc failed"));
    k_to_bf16<<<blocks_for(V * co), 256, 0, n->st>>>(V * co, b, xb);
    if (layer == 0) {
      if ((rc = wgrad_in(n, dm, a, xb, co, ly))) return done(rc);
    } else {
      if ((rc = talloc(&xa, V * ci))) return done(ufail(n, rc, "cudaMalloc failed"));
      k_to_bf16<<<blocks_for(V * ci), 256, 0, n->st>>>(V * ci, a, xa);
      if ((rc = wgrad3(n, dm, xa, ci, ci, xb, co, co, ly))) return done(rc);
    }
    UTRY(n, cudaMemcpyAsync(out, n->grad + ly.woff, sizeof(float) * ((long long)co * ci * 27 + co),
                            cudaMemcpyDeviceToDevice, n->st));
  }
  if (cudaGetLastError() != cudaSuccess) return done(ufail(n, STP_ECUDA, "a layer-check kernel failed to launch"));
  if (cudaStreamSynchronize(n->st) != cudaSuccess) return done(ufail(n, STP_ECUDA, "layer check failed"));
  return done(check_tc_timeout(n));
}

int stp_unet_set_output_scale(stp_unet* n, float k) {
  if (!n || !(k > 0.f)) return STP_EINVAL;
  n->out_scale = k;
  return STP_OK;
}

int stp_unet_train_pairs(stp_unet* n, const float* r, const float* dp, int nb, float lr, float* loss) {
  if (!n || !r || !dp) return STP_EINVAL;
  if (int rc = check_n(n, nb)) return rc;
  const long long Vs = n->dm[0].vox() / n->nmax;
  UTRY(n, cudaMemsetAsync(n->snorm, 0, sizeof(float) * nb, n->st));
  k_sample_sumsq<<<dim3((unsigned)std::min<long long>(256, (Vs + 255) / 256), nb), 256, 0, n->st>>>(Vs, r, n->snorm);
  UTRY(n, cudaGetLastError());
  k_scale_pairs<<<blocks_for(Vs * nb), 256, 0, n->st>>>(Vs, nb, r, dp, n->snorm, n->out_scale, n->xin, n->tin);
  UTRY(n, cudaGetLastError());
  return stp_unet_train_step(n, n->xin, n->tin, nb, lr, loss);
}

int stp_unet_eval_pairs(stp_unet* n, const float* r, const float* dp, int nb, float* loss) {
  if (!n || !r || !dp) return STP_EINVAL;
  if (int rc = check_n(n, nb)) return rc;
  const long long Vs = n->dm[0].vox() / n->nmax;
  UTRY(n, cudaMemsetAsync(n->snorm, 0, sizeof(float) * nb, n->st));
  k_sample_sumsq<<<dim3((unsigned)std::min<long long>(256, (Vs + 255) / 256), nb), 256, 0, n->st>>>(Vs, r, n->snorm);
  UTRY(n, cudaGetLastError());
  k_scale_pairs<<<blocks_for(Vs * nb), 256, 0, n->st>>>(Vs, nb, r, dp, n->snorm, n->out_scale, n->xin, n->tin);
  UTRY(n, cudaGetLastError());
  int rc = forward(n, n->xin, nb);
  if (rc) return rc;
  UTRY(n, cudaMemsetAsync(n->loss, 0, sizeof(float), n->st));
  k_mse<<<std::min(blocks_for(Vs * nb), 4 * 152), 256, 0, n->st>>>(Vs * nb, n->y, n->tin, n->gy, n->loss);
  UTRY(n, cudaGetLastError());
  UTRY(n, cudaMemcpyAsync(n->h_loss, n->loss, sizeof(float), cudaMemcpyDeviceToHost, n->st));
  rc = check_tc_timeout(n);
  if (loss && (rc == STP_OK || rc == STP_ETIMEOUT)) *loss = *n->h_loss;
  return rc;
}

}  // extern "C"
