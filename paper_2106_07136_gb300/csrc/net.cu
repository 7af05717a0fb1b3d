// net.cu -- the learned coarse proposal: a 6-layer 3x3 convolutional network
// on one pyramid level of the pair (level 4 of the paper's 5 scales, the
// level the learned start runs it on), BF16 weights and activations, FP32
// accumulation, forward and training kernels on the tensor cores. The
// network is fully convolutional: any level size works.
//
// Not part of the paper: the paper's method starts its coarsest level from 0
// (Sec. 2.1); this network proposes a start instead, and BDIS refines it.
//
// Architecture (all 3x3, zero padding, dilations 1, 2, 4, 4, 2, 1 so the
// receptive field spans +-14 pixels of its level):
//   x0 = [(L - 128) / 64, (R - 128) / 64]           2 channels (padded to 16)
//   a1..a5 = relu(conv(a_{i-1}) + b_i)              32 channels
//   d = conv(a5) + b6                               1 channel (padded to 16), one per pixel
// Activations are NHWC bf16 (channels innermost).
//
// Every convolution is an implicit GEMM (bf16 in, f32 accumulate): rows =
// pixels, columns = output channels, K = 9 taps x input channels. The forward
// convolutions run on the 5th-generation tensor cores (tcgen05, below) by
// default, or on mma.sync.m16n8k16. The data-gradient of a layer is the same
// kernel run on the output gradient with transposed, tap-flipped weights and
// the previous layer's ReLU mask fused into the store; the weight-gradient is a
// GEMM with rows = output channels, columns = (tap, input channel), K = pixels,
// whose blocks write partial sums that a second kernel adds in a fixed order.
#include <cuda_bf16.h>
#include <limits.h>
#include <stdint.h>

#include <algorithm>
#include <new>
#include <vector>

#include "bdis_internal.cuh"

namespace {

constexpr int kLayers = 6;
constexpr int kDil[kLayers] = {1, 2, 4, 4, 2, 1};
constexpr int kCin[kLayers] = {2, 32, 32, 32, 32, 32};    // real channels
constexpr int kCout[kLayers] = {32, 32, 32, 32, 32, 1};
constexpr int kCinP[kLayers] = {16, 32, 32, 32, 32, 32};  // padded (multiples of 16)
constexpr int kCoutP[kLayers] = {32, 32, 32, 32, 32, 16};

constexpr int master_w_offset(int l) {
  int off = 0;
  for (int i = 0; i < l; ++i) off += kCout[i] * 9 * kCin[i] + kCout[i];
  return off;
}
constexpr int kMasterCount = master_w_offset(kLayers);

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}

// D (16x8 f32) += A (16x16 bf16, row) * B (16x8 bf16, col)
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// ------------------------------------------------------------ input pack

// x0[p][0] = (L - 128)/64, x0[p][1] = (R - 128)/64, channels 2..15 zero.
__global__ void pack_input_kernel(const float *__restrict__ L, const float *__restrict__ R,
                                  int r_stride, long long total, __nv_bfloat16 *__restrict__ x0) {
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= total) return;
  uint4 *dst = reinterpret_cast<uint4 *>(x0 + p * 16);
  const float l = (__ldg(L + p) - 128.f) * (1.f / 64.f);
  const float r = (__ldg(R + p * r_stride) - 128.f) * (1.f / 64.f);
  uint4 v0 = make_uint4(pack_bf16(l, r), 0u, 0u, 0u);
  dst[0] = v0;
  dst[1] = make_uint4(0u, 0u, 0u, 0u);
}

// ------------------------------------------------------------ conv (mma)

enum ConvMode { kFwdRelu = 0, kFwdLinearF32 = 1, kBwdDataMasked = 2 };

// One warp computes MT x 16 consecutive pixels x COUT channels (MT m-tiles
// share every weight fragment it loads); a block of 4 warps covers 64 MT
// pixels per tile and loops over tiles (persistent), so the weights (COUT x 9
// x CIN bf16) are staged in shared memory once per block.
template <int CIN, int COUT, int MODE, int MT = 4>
__global__ void __launch_bounds__(128) conv_mma_kernel(
    const __nv_bfloat16 *__restrict__ in, const __nv_bfloat16 *__restrict__ wt,
    const float *__restrict__ bias, int dil, int H, int W, long long total,
    const __nv_bfloat16 *__restrict__ mask, void *__restrict__ out) {
  static_assert(CIN % 16 == 0 && COUT % 8 == 0, "tile");
  constexpr int NT = COUT / 8;
  __shared__ __align__(16) __nv_bfloat16 ws[COUT * 9 * CIN];
  for (int i = threadIdx.x * 8; i < COUT * 9 * CIN; i += blockDim.x * 8)
    *reinterpret_cast<uint4 *>(ws + i) = *reinterpret_cast<const uint4 *>(wt + i);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, q = lane & 3;
  const long long plane = (long long)H * W;
  const long long per_tile = 64LL * MT;
  for (long long tile = blockIdx.x; tile * per_tile < total; tile += gridDim.x) {
    const long long p0 = tile * per_tile + (long long)warp * 16 * MT;
    // pixel rows of this thread: m-tile m feeds rows p0 + 16 m + g and + 8
    long long pr[MT][2];
    int pb[MT][2], py[MT][2], px[MT][2];
    bool pv[MT][2];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        pr[m][i] = p0 + 16 * m + g + 8 * i;
        pv[m][i] = pr[m][i] < total;
        const long long pp = pv[m][i] ? pr[m][i] : 0;
        pb[m][i] = (int)(pp / plane);
        const int rem = (int)(pp - (long long)pb[m][i] * plane);
        py[m][i] = rem / W;
        px[m][i] = rem - py[m][i] * W;
      }
    float acc[MT][NT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int n = 0; n < NT; ++n) acc[m][n][0] = acc[m][n][1] = acc[m][n][2] = acc[m][n][3] = 0.f;
#pragma unroll 1
    for (int tap = 0; tap < 9; ++tap) {
      const int dy = (tap / 3 - 1) * dil, dx = (tap % 3 - 1) * dil;
      const __nv_bfloat16 *src[MT][2];
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int yy = py[m][i] + dy, xx = px[m][i] + dx;
          const bool ok = pv[m][i] && yy >= 0 && yy < H && xx >= 0 && xx < W;
          src[m][i] = ok ? in + (((long long)pb[m][i] * H + yy) * W + xx) * CIN : nullptr;
        }
#pragma unroll
      for (int kb = 0; kb < CIN / 16; ++kb) {
        const int c0 = kb * 16 + q * 2;
        uint32_t b[NT][2];
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const __nv_bfloat16 *wr = ws + ((n * 8 + g) * 9 + tap) * CIN + c0;
          b[n][0] = *reinterpret_cast<const uint32_t *>(wr);
          b[n][1] = *reinterpret_cast<const uint32_t *>(wr + 8);
        }
#pragma unroll
        for (int m = 0; m < MT; ++m) {
          uint32_t a[4];
          a[0] = src[m][0] ? *reinterpret_cast<const uint32_t *>(src[m][0] + c0) : 0u;
          a[1] = src[m][1] ? *reinterpret_cast<const uint32_t *>(src[m][1] + c0) : 0u;
          a[2] = src[m][0] ? *reinterpret_cast<const uint32_t *>(src[m][0] + c0 + 8) : 0u;
          a[3] = src[m][1] ? *reinterpret_cast<const uint32_t *>(src[m][1] + c0 + 8) : 0u;
#pragma unroll
          for (int n = 0; n < NT; ++n) mma_bf16(acc[m][n], a, b[n]);
        }
      }
    }
    // epilogue: acc[m][n][0..1] -> row 16m + g, channels 8n + 2q + {0,1}; [2..3] -> row + 8
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (!pv[m][i]) continue;
        const long long p = pr[m][i];
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const int c = n * 8 + q * 2;
          float v0 = acc[m][n][2 * i], v1 = acc[m][n][2 * i + 1];
          if (MODE == kFwdRelu) {
            v0 = fmaxf(v0 + bias[c], 0.f);
            v1 = fmaxf(v1 + bias[c + 1], 0.f);
            *reinterpret_cast<uint32_t *>(reinterpret_cast<__nv_bfloat16 *>(out) + p * COUT + c) =
                pack_bf16(v0, v1);
          } else if (MODE == kFwdLinearF32) {
            float *o = reinterpret_cast<float *>(out) + p * COUT + c;
            o[0] = v0 + bias[c];
            o[1] = v1 + bias[c + 1];
          } else {  // data gradient times the previous layer's ReLU derivative
            const __nv_bfloat162 mk =
                *reinterpret_cast<const __nv_bfloat162 *>(mask + p * COUT + c);
            v0 = __bfloat162float(mk.x) > 0.f ? v0 : 0.f;
            v1 = __bfloat162float(mk.y) > 0.f ? v1 : 0.f;
            *reinterpret_cast<uint32_t *>(reinterpret_cast<__nv_bfloat16 *>(out) + p * COUT + c) =
                pack_bf16(v0, v1);
          }
        }
      }
  }
}

// ------------------------------------------------------- conv (tcgen05)

// The same forward convolutions on the 5th-generation tensor cores, as an
// implicit GEMM without an im2col copy. Pixels are numbered in a padded frame:
// each image becomes (H + 2 dil) x (W + 2 dil) with zero borders, so a tap
// (dy, dx) is the constant shift dy dil (W + 2 dil) + dx dil of that
// numbering. A block (one warpgroup, 128 threads) owns a tile of 128
// consecutive padded positions and stages, once, the slab of padded positions
// [tile - s, tile + 127 + s] (s = the largest shift) in shared memory: for each
// group of 8 channels a plane of slab rows, 16 bytes per row. In the
// no-swizzle K-major layout that is a run of core matrices (8 rows x 16 bytes,
// 128 B apart along M), so the A operand of tap t is the slab window starting
// s + shift(t) rows in (a descriptor start 16 B per row), and the two channel
// groups of one MMA (K = 16) are one plane apart (the leading offset). B (the
// COUT x 9 CIN weights) is staged once per block. One thread issues the
// 9 CIN / 16 MMAs (M 128, N COUT, K 16) into a tensor-memory accumulator and
// commits them to an mbarrier; every thread then reads its row of D (warp w
// owns tensor-memory lanes 32 w .. 32 w + 31) and, if its position is a real
// pixel, writes the layer output. Waits are bounded by the global timer: on a
// timeout the block writes NaN, sets the network's fault word (read by
// bdis_net_status), frees its tensor memory and returns.

__device__ __forceinline__ uint64_t umma_smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);  // no swizzle
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// wait until the mbarrier's phase `parity` has completed, at most ~200 ms
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
  const uint64_t t0 = global_ns();
  while (true) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (done) return true;
    if (global_ns() - t0 > 200000000ull) return false;
  }
}

// slab rows of a tile: 128 positions plus the largest shift on either side
__host__ __device__ __forceinline__ int tc_slab_rows(int dil, int W) {
  return 128 + 2 * (dil * (W + 2 * dil) + dil);
}

template <int CIN, int COUT>
int tc_smem_bytes(int dil, int W) {  // the slab and the weights
  return (CIN / 8) * tc_slab_rows(dil, W) * 16 + (9 * CIN / 8) * (COUT / 8) * 128;
}

template <int CIN, int COUT, int MODE>
__global__ void __launch_bounds__(128) conv_tc_kernel(
    const __nv_bfloat16 *__restrict__ in, const __nv_bfloat16 *__restrict__ wt,
    const float *__restrict__ bias, int dil, int H, int W, int count,
    void *__restrict__ out, int *__restrict__ fault) {
  static_assert(CIN % 16 == 0 && (COUT == 16 || COUT == 32), "tile");
  static_assert(MODE == kFwdRelu || MODE == kFwdLinearF32, "forward only");
  constexpr int KG = 9 * CIN / 8;  // 8-element k-groups of the weights
  constexpr int NG = COUT / 8;
  constexpr int CG = CIN / 8;      // channel groups (slab planes)
  extern __shared__ __align__(128) uint8_t tc_smem[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_slot;
  const int Wp = W + 2 * dil, Hp = H + 2 * dil;
  const int NS = tc_slab_rows(dil, W), soff = dil * Wp + dil;
  const long long planep = (long long)Hp * Wp, totalp = planep * count;
  uint8_t *Ss = tc_smem, *Bs = tc_smem + CG * NS * 16;  // slab, weights
  const int tid = threadIdx.x, warp = tid >> 5;
  // B: weight row co (K = 9 CIN contiguous) -> core (kg, co / 8), row co % 8
  for (int i = tid; i < COUT * KG; i += 128) {
    const int co = i / KG, kg = i - co * KG;
    const uint4 v = *reinterpret_cast<const uint4 *>(wt + (size_t)co * 9 * CIN + kg * 8);
    *reinterpret_cast<uint4 *>(Bs + ((kg * NG + co / 8) * 8 + co % 8) * 16) = v;
  }
  const uint32_t mbar_a = (uint32_t)__cvta_generic_to_shared(&mbar);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(mbar_a));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    const uint32_t slot = (uint32_t)__cvta_generic_to_shared(&tmem_slot);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 32;\n" ::"r"(slot));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = tmem_slot;
  const uint32_t s_base = (uint32_t)__cvta_generic_to_shared(Ss);
  const uint32_t b_base = (uint32_t)__cvta_generic_to_shared(Bs);
  constexpr uint32_t idesc = (1u << 4)                    // D: f32
                             | (1u << 7) | (1u << 10)     // A, B: bf16, both K-major
                             | ((uint32_t)(COUT >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
  // a padded position -> its real pixel index, or -1 on a border or past the end
  auto real_pixel = [&](long long q) -> long long {
    if (q < 0 || q >= totalp) return -1;
    const int b = (int)(q / planep);
    const int rem = (int)(q - (long long)b * planep);
    const int y = rem / Wp - dil, x = rem - (rem / Wp) * Wp - dil;
    if (y < 0 || y >= H || x < 0 || x >= W) return -1;
    return ((long long)b * H + y) * W + x;
  };
  uint32_t parity = 0;
  bool ok = true;
  for (long long tile = blockIdx.x; tile * 128 < totalp && ok; tile += gridDim.x) {
    const long long q0 = tile * 128 - soff;  // padded position of slab row 0
    for (int i = tid; i < NS; i += 128) {
      const long long pix = real_pixel(q0 + i);
      const __nv_bfloat16 *src = pix >= 0 ? in + pix * CIN : in;
#pragma unroll
      for (int cg = 0; cg < CG; ++cg)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(
                         s_base + (cg * NS + i) * 16),
                     "l"(src + cg * 8), "r"(pix >= 0 ? 16 : 0));
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    const uint32_t sb = s_base;
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // visible to the tensor cores
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (tid == 0) {
#pragma unroll 1
      for (int tap = 0; tap < 9; ++tap) {
        const int row0 = soff + (tap / 3 - 1) * dil * Wp + (tap % 3 - 1) * dil;
#pragma unroll
        for (int kk = 0; kk < CIN / 16; ++kk) {
          const uint64_t ad =
              umma_smem_desc(sb + (2 * kk * NS + row0) * 16, (uint32_t)NS * 16, 128);
          const uint64_t bd =
              umma_smem_desc(b_base + (tap * CG + 2 * kk) * NG * 128, NG * 128, 128);
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
              "l"(ad), "l"(bd), "r"(idesc), "r"(tap | kk));
        }
      }
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
              mbar_a));
    }
    // every thread of the block takes the same branch below (the loads are
    // warp-collective and the loop has block barriers)
    ok = __syncthreads_and(mbar_wait(mbar_a, parity)) != 0;
    if (!ok && tid == 0) atomicOr(fault, 1);  // reported by bdis_net_status
    parity ^= 1u;
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    float d[COUT];
    if (ok) {
      const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16);
      if constexpr (COUT == 32) {
        uint32_t r[32];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
            "%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
              "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
              "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
              "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
              "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
              "=r"(r[31])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
        for (int c = 0; c < COUT; ++c) d[c] = __uint_as_float(r[c]);
      } else {
        uint32_t r[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
            "%13,%14,%15}, [%16];\n"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
              "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
              "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
        for (int c = 0; c < COUT; ++c) d[c] = __uint_as_float(r[c]);
      }
    } else {
#pragma unroll
      for (int c = 0; c < COUT; ++c) d[c] = __int_as_float(0x7fc00000);
    }
    const long long p = real_pixel(tile * 128 + tid);
    if (p >= 0) {
      if constexpr (MODE == kFwdRelu) {
        uint32_t pk[COUT / 2];
#pragma unroll
        for (int c = 0; c < COUT; c += 2)
          pk[c / 2] = pack_bf16(fmaxf(d[c] + bias[c], 0.f), fmaxf(d[c + 1] + bias[c + 1], 0.f));
        uint4 *o = reinterpret_cast<uint4 *>(reinterpret_cast<__nv_bfloat16 *>(out) + p * COUT);
#pragma unroll
        for (int v = 0; v < COUT / 8; ++v)
          o[v] = make_uint4(pk[4 * v], pk[4 * v + 1], pk[4 * v + 2], pk[4 * v + 3]);
      } else {
        float *o = reinterpret_cast<float *>(out) + p * COUT;
#pragma unroll
        for (int c = 0; c < COUT; ++c) o[c] = d[c] + bias[c];
      }
    }
    // every thread has read D and the MMAs are done: the slab and D may be rewritten
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");  // none left in flight (timeout exit)
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 32;\n" ::"r"(tmem));
}

// ------------------------------------------------------ conv (tcgen05, banded)

// Forward passes, and training, keep every activation in a padded planar
// layout in global memory: each image is framed by kPad zero rows and
// columns (kPad = the largest dilation, so every tap of a real pixel lands
// inside its own frame), frames are numbered back to back, and each group of
// 8 channels is its own plane of 16-byte rows, with zero guard rows before
// and after. A 3x3 tap is then a constant shift of the position numbering, a
// plane's rows are exactly the 8-row x 16-byte core matrices of the tensor
// cores' no-swizzle K-major operand layout, and the rows any band of
// positions reads form one contiguous range per plane: one bulk copy each.
//
// A whole forward pass is one cooperative launch, one block per SM: the
// input is packed, then the six layers run in turn with a grid barrier
// between steps (a band's halo was written by other blocks). Within a layer
// the block is warp-specialised, three stages in flight:
//   - warps 8-11 (one lane each) issue each unit's MMAs (9 taps x CIN / 16
//     per 128-position tile; M 128, N = COUT, K 16; every 4th tile each)
//     into one of two tensor-memory accumulators, one COUT-column slice per
//     tile; warp 8 also stages the units (a band of BH image rows of one
//     image, all padded columns, with its halo of up to dil rows + dil
//     columns either side) by bulk copies into two slab buffers;
//   - warps 0-7 (warp w reads tensor-memory lanes 32 (w % 4) .. + 31, of
//     every other tile) take each finished accumulator, add the bias, apply
//     the ReLU, pack to bf16 and write the real pixels, then hand the
//     accumulator back; two warps per lane quarter hide each other's latency.
// So unit k's MMAs run while unit k + 1's copy travels and unit k - 1's
// epilogue drains. The MMAs bound it: measured on GB300, an M 128 x K 16
// MMA whose A operand (4 KB) is read afresh from no-swizzle shared memory
// takes about 68 cycles whether N is 32 or 64, so with 32 output channels
// the tensor pipe runs at about a quarter of its dense rate.
// Every wait is bounded by the global timer (200 ms on an mbarrier, 1 s at a
// grid barrier): on a timeout the block records it in the network's fault
// word, waits (bounded) for its own copies and MMAs in flight, writes NaN
// over its bands of the map, frees its tensor memory and returns; the other
// blocks then time out at the next grid barrier, if there is one, and do
// the same. In training the word is the call's own, which its last kernel reads:
// a call with a failed wait in any of its kernels gives a loss and a gradient of
// NaN, and takes no Adam step.
constexpr int kPad = 4;                // frame border = the largest dilation
constexpr int kBandCols = 256;         // tensor-memory columns per accumulator (two)
constexpr int kBandSmem = 224 * 1024;  // dynamic shared memory per block (one per SM)
constexpr int kBandEpiWarps = 8;       // two per tensor-memory lane quarter
constexpr int kBandMmaWarps = 4;       // MMA issue: one lane of each takes every 4th tile
constexpr int kBandThreads = 32 * (kBandEpiWarps + kBandMmaWarps);

__host__ __device__ __forceinline__ long long pp_guard(int W) {
  return (long long)kPad * (W + 2 * kPad) + kPad + 128;
}

// elements (bf16) between two channel planes of a padded planar buffer
__host__ __device__ __forceinline__ long long pp_plane(int H, int W, int count) {
  return ((long long)count * (H + 2 * kPad) * (W + 2 * kPad) + 2 * pp_guard(W)) * 8;
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes,
                                          uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(mbar)
      : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mbar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(mbar), "r"(count));
}

__device__ __forceinline__ void *band_smem_base() {
  extern __shared__ __align__(128) uint8_t band_smem[];
  return band_smem;
}

// One layer of the fused kernel below.
struct BandLayer {
  const __nv_bfloat16 *in, *wt;
  const float *bias;
  void *out;      // kFwdLinearF32: dense float map; else padded planar bf16
  const __nv_bfloat16 *mask;  // kBwdDataMasked: the ReLU outputs (padded planar)
  int dil, BH, nsb;  // dilation, band rows, slab rows per channel plane
};
struct BandNet {
  BandLayer layer[6];
  const float *L, *R;  // forward: the level planes (R with element stride r_stride)
  const float *map, *label;  // backward: the forward map and its labels (NaN = none)
  float *loss;               // backward: the loss, zero at launch
  int r_stride, H, W, count;
  int slab_bytes;      // per slab buffer (the largest layer's), two buffers
  unsigned *sync;      // grid barrier counter, zero at launch
  int *fault;          // set when a bounded wait ran out
};

// Shared state of the fused kernel's block.
struct BandShared {
  uint32_t s_base, b_base, tmem;
  uint32_t full_a[2], mma_a[2], free_a[2];
};

// Grid-wide barrier of the cooperative launch (all blocks are resident): the
// block's writes are published, one thread counts the block in and waits,
// bounded, for every block of the grid. `target` = barriers passed so far x
// gridDim.x. Returns false (on every thread) if the wait ran out.
__device__ __forceinline__ bool grid_barrier(unsigned *count, unsigned target) {
  __threadfence();
  __syncthreads();
  int ok = 1;
  if (threadIdx.x == 0) {
    atomicAdd(count, 1u);
    const uint64_t t0 = global_ns();
    while (true) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(count) : "memory");
      if (v >= target) break;
      if (global_ns() - t0 > 1000000000ull) {  // 1 s
        ok = 0;
        break;
      }
      __nanosleep(64);
    }
  }
  return __syncthreads_and(ok) != 0;
}

// One layer: the roles of the module comment over the layer's units. kg counts
// the block's units over all layers (buffer = kg & 1, barrier phase = (kg >> 1)
// & 1); on return every unit of the layer is written and its accumulators are
// handed back. MODE kFwdRelu, kBwdDataMasked: out is a padded planar bf16 buffer
// of COUT channels (the latter zero where the layer's mask is not positive, no
// bias); kFwdLinearF32: out is the dense float map of channel 0.
template <int CIN, int COUT, int MODE>
__device__ bool band_layer(const BandNet &net, const BandLayer &ly, const BandShared &sh,
                           float *sbias, long long &kg) {
  static_assert(CIN % 16 == 0 && (COUT == 16 || COUT == 32), "tile");
  constexpr int KG = 9 * CIN / 8, NG = COUT / 8, CG = CIN / 8;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int H = net.H, W = net.W, count = net.count, dil = ly.dil, BH = ly.BH;
  const int nsb_max = ly.nsb, slab_bytes = net.slab_bytes;
  const int Wp = W + 2 * kPad, Hp = H + 2 * kPad;
  const long long F = (long long)Hp * Wp;
  const long long plane_in = pp_plane(H, W, count), guard = pp_guard(W);
  const int soff = dil * Wp + dil;
  const int nb = (H + BH - 1) / BH;
  const long long units = (long long)count * nb;
  // the layer's weights and bias (the previous layer's MMAs are all done)
  uint8_t *Bs = reinterpret_cast<uint8_t *>(band_smem_base()) + 2 * slab_bytes;
  for (int i = tid; i < COUT * KG; i += kBandThreads) {
    const int kgr = i / COUT, co = i - kgr * COUT;  // consecutive threads: consecutive rows
    const uint4 v = *reinterpret_cast<const uint4 *>(ly.wt + (size_t)co * 9 * CIN + kgr * 8);
    *reinterpret_cast<uint4 *>(Bs + ((kgr * NG + co / 8) * 8 + co % 8) * 16) = v;
  }
  if (MODE != kBwdDataMasked && tid < COUT) sbias[tid] = ly.bias[tid];
  // weights: generic-proxy writes read by the tensor cores; the input: written
  // by other blocks before the grid barrier, read by this block's bulk copies
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  asm volatile("fence.proxy.async.global;\n" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  auto band = [&](long long u, long long &q_s, int &cnt, int &tiles) {
    const int b = (int)(u / nb), j = (int)(u - (long long)b * nb);
    const int rows = min(BH, H - j * BH);
    q_s = (long long)b * F + (long long)(kPad + j * BH) * Wp;
    cnt = rows * Wp;
    tiles = (cnt + 127) >> 7;
  };
  const long long nk = units > blockIdx.x ? (units - 1 - blockIdx.x) / gridDim.x + 1 : 0;
  bool ok = true;
  if (warp >= kBandEpiWarps) {
    // ---- copies (issuer 0) and MMAs (one lane of each issuer warp)
    const int issuer = warp - kBandEpiWarps;
    if (lane == 0 && nk > 0) {
      constexpr uint32_t idesc = (1u << 4)                 // D: f32
                                 | (1u << 7) | (1u << 10)  // A, B: bf16, both K-major
                                 | ((uint32_t)(COUT >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      auto issue_load = [&](long long k) {
        long long q_s;
        int cnt, tiles;
        band(blockIdx.x + k * gridDim.x, q_s, cnt, tiles);
        const int s = (int)((kg + k) & 1), nsb = tiles * 128 + 2 * soff;
        mbar_expect_tx(sh.full_a[s], (uint32_t)(CG * nsb * 16));
        for (int cg = 0; cg < CG; ++cg)
          bulk_load(sh.s_base + (uint32_t)(s * slab_bytes + cg * nsb_max * 16),
                    ly.in + ((long long)cg * plane_in / 8 + guard + q_s - soff) * 8,
                    (uint32_t)(nsb * 16), sh.full_a[s]);
      };
      // the last unit whose copy / MMAs went to each buffer (-1: none), for the timeout path
      long long last_load[2] = {-1, -1}, last_mma[2] = {-1, -1};
      if (issuer == 0) {
        issue_load(0);
        last_load[kg & 1] = kg;
      }
      for (long long k = 0; k < nk && ok; ++k) {
        const long long g = kg + k;
        const int s = (int)(g & 1);
        const uint32_t ph = (uint32_t)((g >> 1) & 1);
        ok = mbar_wait(sh.full_a[s], ph);  // unit k's slab has landed
        if (ok && g >= 2) ok = mbar_wait(sh.free_a[s], ph ^ 1u);  // unit g - 2's epilogue is done
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        long long q_s;
        int cnt, tiles;
        band(blockIdx.x + k * gridDim.x, q_s, cnt, tiles);
        // descriptors advance in 16-byte units of their start-address field
        // (shared memory is far below the field's 256 KB reach, so no carry)
        const uint64_t a0 = umma_smem_desc(sh.s_base + (uint32_t)(s * slab_bytes),
                                           (uint32_t)nsb_max * 16, 128);
        const uint64_t b0 = umma_smem_desc(sh.b_base, NG * 128, 128);
        const uint32_t t0 = sh.tmem + (uint32_t)(s * kBandCols);
#pragma unroll 1
        for (int i = issuer; i < tiles; i += kBandMmaWarps) {
          const uint32_t d_tmem = t0 + (uint32_t)(i * COUT);
          const int rowi = soff + i * 128;
#pragma unroll
          for (int tap = 0; tap < 9; ++tap) {
            const int row0 = rowi + (tap / 3 - 1) * dil * Wp + (tap % 3 - 1) * dil;
#pragma unroll
            for (int kk = 0; kk < CIN / 16; ++kk) {
              const uint64_t ad = a0 + (uint64_t)(row0 + 2 * kk * nsb_max);
              const uint64_t bd = b0 + (uint64_t)((tap * CG + 2 * kk) * NG * 8);
              asm volatile(
                  "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                  " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
                  "l"(ad), "l"(bd), "r"(idesc), "r"(tap | kk));
            }
          }
        }
        asm volatile(
            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                sh.mma_a[s]));
        last_mma[s] = g;
        // the next unit's copy goes to the other slab once unit g - 1's MMAs
        // (queued ahead of unit g's) have read it
        if (issuer == 0 && k + 1 < nk) {
          if (k >= 1) ok = mbar_wait(sh.mma_a[s ^ 1], (uint32_t)(((g - 1) >> 1) & 1));
          if (!ok) break;
          issue_load(k + 1);
          last_load[s ^ 1] = g + 1;
        }
      }
      if (!ok) {
        atomicOr(net.fault, 1);  // reported by bdis_net_status
        // let the copies and MMAs this block issued land before its memory is released
        for (int b2 = 0; b2 < 2; ++b2) {
          if (last_load[b2] >= 0) mbar_wait(sh.full_a[b2], (uint32_t)((last_load[b2] >> 1) & 1));
          if (last_mma[b2] >= 0) mbar_wait(sh.mma_a[b2], (uint32_t)((last_mma[b2] >> 1) & 1));
        }
      }
    }
  } else {
    // ---- epilogue (warps 0 .. kBandEpiWarps - 1)
    const int quarter = warp & 3, parity = warp >> 2;
    const float *bs = sbias;
    for (long long k = 0; k < nk; ++k) {
      const long long g = kg + k;
      const int s = (int)(g & 1);
      long long q_s;
      int cnt, tiles;
      band(blockIdx.x + k * gridDim.x, q_s, cnt, tiles);
      ok = mbar_wait(sh.mma_a[s], (uint32_t)((g >> 1) & 1));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const int b = (int)(q_s / F);
      for (int i = parity; i < tiles; i += kBandEpiWarps / 4) {
        const uint32_t taddr = sh.tmem + ((uint32_t)(quarter * 32) << 16) +
                               (uint32_t)(s * kBandCols + i * COUT);
        float d[COUT];
        if constexpr (COUT == 32) {
          uint32_t r[32];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
              "%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
              : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]),
                "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
                "=r"(r[30]), "=r"(r[31])
              : "r"(taddr));
          asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
          for (int c = 0; c < COUT; ++c) d[c] = __uint_as_float(r[c]);
        } else {
          uint32_t r[16];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
              "%13,%14,%15}, [%16];\n"
              : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
              : "r"(taddr));
          asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
          for (int c = 0; c < COUT; ++c) d[c] = __uint_as_float(r[c]);
        }
        const int m = i * 128 + quarter * 32 + lane;  // position within the band
        const int xp = m % Wp, x = xp - kPad;
        if (m < cnt && x >= 0 && x < W) {
          const long long q = q_s + m;
          if constexpr (MODE != kFwdLinearF32) {
            uint32_t pk[COUT / 2];
            const long long plane_out = pp_plane(H, W, count) / 8;  // in 16-byte rows
            if constexpr (MODE == kFwdRelu) {
#pragma unroll
              for (int c = 0; c < COUT; c += 2)
                pk[c / 2] = pack_bf16(fmaxf(d[c] + bs[c], 0.f), fmaxf(d[c + 1] + bs[c + 1], 0.f));
            } else {
              const uint4 *mp = reinterpret_cast<const uint4 *>(ly.mask) + guard + q;
#pragma unroll
              for (int v = 0; v < COUT / 8; ++v) {
                const uint4 m4 = __ldg(mp + v * plane_out);
                const uint32_t mw[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const __nv_bfloat162 m = *reinterpret_cast<const __nv_bfloat162 *>(&mw[e]);
                  const int c = 8 * v + 2 * e;
                  pk[c / 2] = pack_bf16(__bfloat162float(m.x) > 0.f ? d[c] : 0.f,
                                        __bfloat162float(m.y) > 0.f ? d[c + 1] : 0.f);
                }
              }
            }
            uint4 *o = reinterpret_cast<uint4 *>(ly.out) + guard + q;
#pragma unroll
            for (int v = 0; v < COUT / 8; ++v)
              o[v * plane_out] =
                  make_uint4(pk[4 * v], pk[4 * v + 1], pk[4 * v + 2], pk[4 * v + 3]);
          } else {
            const int y = (int)((q - (long long)b * F) / Wp) - kPad;
            reinterpret_cast<float *>(ly.out)[((long long)b * H + y) * W + x] = d[0] + bs[0];
          }
        }
      }
      // this accumulator is read: the unit two later may overwrite it
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      mbar_arrive(sh.free_a[s]);
    }
  }
  kg += nk;
  return __syncthreads_and(ok ? 1 : 0) != 0;
}

// Huber (delta 1) loss of one pixel against its label (NaN = no label) over
// the mean's 1 / n, and its gradient.
__device__ __forceinline__ float huber_at(float z, float label, float inv_n, float &grad) {
  grad = 0.f;
  if (!isfinite(label)) return 0.f;
  const float e = z - label, ae = fabsf(e);
  grad = (ae <= 1.f ? e : copysignf(1.f, e)) * inv_n;
  return ae <= 1.f ? 0.5f * e * e : ae - 0.5f;
}

// The whole forward pass (or, BACK, the loss and all data gradients) in one
// cooperative launch (one block per SM): the input planes are packed into x0
// (the loss gradient into the last layer's), then the layers run in turn, a
// grid barrier between steps (a layer reads the bands around its own, which
// other blocks wrote). Weights and bias are restaged per layer; the slabs,
// barriers and tensor memory carry over. BACK's layers are in their order of
// execution, the last layer's data gradient first.
template <bool BACK>
__global__ void __launch_bounds__(kBandThreads, 1) net_chain_kernel(const BandNet net) {
  __shared__ __align__(8) uint64_t mb_full[2], mb_mma[2], mb_free[2];
  __shared__ uint32_t tmem_slot;
  __shared__ float sbias[32];
  const int tid = threadIdx.x, warp = tid >> 5;
  BandShared sh;
  for (int i = 0; i < 2; ++i) {
    sh.full_a[i] = (uint32_t)__cvta_generic_to_shared(&mb_full[i]);
    sh.mma_a[i] = (uint32_t)__cvta_generic_to_shared(&mb_mma[i]);
    sh.free_a[i] = (uint32_t)__cvta_generic_to_shared(&mb_free[i]);
  }
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(sh.full_a[i], 1);
      mbar_init(sh.mma_a[i], kBandMmaWarps);
      mbar_init(sh.free_a[i], 32 * kBandEpiWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    const uint32_t slot = (uint32_t)__cvta_generic_to_shared(&tmem_slot);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(slot),
                 "n"(2 * kBandCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  // x0: plane 0 = [(L - 128) / 64, (R - 128) / 64, 0 x 6] (BACK: the loss
  // gradient, 0 x 7) at every real pixel (plane 1 and the borders stay zero)
  {
    const int H = net.H, W = net.W, Wp = W + 2 * kPad, Hp = H + 2 * kPad;
    const long long plane = (long long)H * W, total = plane * net.count;
    uint4 *x0 = reinterpret_cast<uint4 *>(const_cast<__nv_bfloat16 *>(net.layer[0].in));
    const float inv_n = 1.f / (float)total;
    float loss = 0.f;
    for (long long p = (long long)blockIdx.x * kBandThreads + tid; p < total;
         p += (long long)gridDim.x * kBandThreads) {
      const int b = (int)(p / plane);
      const int rem = (int)(p - (long long)b * plane);
      const int y = rem / W, x = rem - (rem / W) * W;
      const long long q = ((long long)b * Hp + y + kPad) * Wp + x + kPad;
      if constexpr (BACK) {
        float g;
        loss += huber_at(__ldg(net.map + p), __ldg(net.label + p), inv_n, g);
        x0[pp_guard(W) + q] = make_uint4(pack_bf16(g, 0.f), 0u, 0u, 0u);
      } else {
        const float l = (__ldg(net.L + p) - 128.f) * (1.f / 64.f);
        const float r = (__ldg(net.R + p * net.r_stride) - 128.f) * (1.f / 64.f);
        x0[pp_guard(W) + q] = make_uint4(pack_bf16(l, r), 0u, 0u, 0u);
      }
    }
    if constexpr (BACK) {
      for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
      if ((tid & 31) == 0) atomicAdd(net.loss, loss * inv_n);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  sh.tmem = tmem_slot;
  sh.s_base = (uint32_t)__cvta_generic_to_shared(band_smem_base());
  sh.b_base = sh.s_base + 2u * (uint32_t)net.slab_bytes;
  long long kg = 0;
  unsigned passed = 0;
  bool ok = grid_barrier(net.sync, ++passed * gridDim.x);
  constexpr int kMid = BACK ? kBwdDataMasked : kFwdRelu;
  if (ok) ok = band_layer<16, 32, kMid>(net, net.layer[0], sh, sbias, kg);
  for (int l = 1; l < 5 && ok; ++l) {
    ok = grid_barrier(net.sync, ++passed * gridDim.x);
    if (ok) ok = band_layer<32, 32, kMid>(net, net.layer[l], sh, sbias, kg);
  }
  if constexpr (!BACK) {
    if (ok) ok = grid_barrier(net.sync, ++passed * gridDim.x);
    if (ok) ok = band_layer<32, 16, kFwdLinearF32>(net, net.layer[5], sh, sbias, kg);
  }
  if (!ok) {
    // a wait ran out (ok is uniform over the block): record it, and mark this
    // block's bands of the map as missing (NaN), whatever was written there
    if (tid == 0) atomicOr(net.fault, 1);
    if constexpr (!BACK) {
      const BandLayer &ly = net.layer[5];
      const int H = net.H, W = net.W, nb = (H + ly.BH - 1) / ly.BH;
      const long long units = (long long)net.count * nb;
      for (long long u = blockIdx.x; u < units; u += gridDim.x) {
        const int b = (int)(u / nb), j = (int)(u - (long long)b * nb);
        const int n = min(ly.BH, H - j * ly.BH) * W;
        float *o = reinterpret_cast<float *>(ly.out) + ((long long)b * H + j * ly.BH) * W;
        for (int i = tid; i < n; i += kBandThreads) o[i] = __int_as_float(0x7fc00000);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(sh.tmem),
                 "n"(2 * kBandCols));
}

// ------------------------------------------------------- weight gradient

// dW[co][tap][ci] = sum_p G[p][co] X[p shifted by tap][ci]; db[co] = sum_p
// G[p][co], for all six layers in one launch, on mma.sync (M = co, N = (tap,
// ci), K = pixels: 32 rows at most, which tcgen05's M of 64 or 128 would leave
// half empty, and both operands pixel-major).
//
// Pixels are numbered so that a tap is a constant shift: for activations in the
// banded kernel's padded planar layout (PLANAR) by their positions there, the
// padded rows of an image after one another; for NHWC ones (images too wide for
// the banded kernel) in frames of (H + dil) x (W + dil) positions, zero past the
// image. A block takes tiles of 128 positions of one layer. Per tile it stages
// G once and X as three segments of 128 + 2 dil positions (one per kernel row,
// whatever the image width), a plane of 16-byte rows per 8 channels, two tiles
// in flight: from the planar layout by one bulk copy per plane and segment.
// ldmatrix.trans turns the pixel-major rows into both operands' fragments (eight
// rows are 128 consecutive bytes: no bank conflicts). A warp owns 8 input
// channels (the first layer, with 2, is split over the warps by pixels instead)
// and all nine taps; a block writes its totals to a partial buffer of its own,
// which reduce_grad_kernel adds in a fixed order: no atomics, the same gradient
// every time.
constexpr int kWgTile = 128;
constexpr int kWgRows = kWgTile + 2 * 4;  // rows of a segment at the largest dilation
constexpr int kWgX = 3 * kWgRows * 16, kWgG = kWgTile * 16;  // bytes of a staged plane
constexpr int kWgStage = 4 * (kWgX + kWgG);  // bytes of one staged tile (X, then G)
constexpr int kWgSmem = 2 * kWgStage, kWgPerSm = 3;  // 3 x 67 KB per SM
constexpr int kPart = 32 * 9 * 32 + 32;  // floats of one block's partial: dW, then db

struct WgradLayer {
  const __nv_bfloat16 *X, *G;
  int dil, first, blocks;  // blocks first .. first + blocks - 1 take the layer
};
struct WgradArgs {
  WgradLayer layer[kLayers];
  int H, W, count;
  float *part;
  int *fault;
};

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

// One layer's tiles t = rank, rank + ranks, ... XS, GS: channels stored per
// pixel (NHWC); XC, GC: planes of 8 channels used. False if a bounded wait for
// the copies ran out.
template <bool PLANAR, int XS, int XC, int GS, int GC>
__device__ __forceinline__ bool wgrad_layer(const WgradArgs &args, const WgradLayer &ly,
                                            uint8_t *smem, uint32_t mbar, float *part) {
  constexpr int MT = (GC + 1) / 2;       // 16-channel m-tiles
  constexpr bool SPLIT = XC < 4;         // warps share the pixels, not the channels
  static_assert(XC == 1 || XC == 4, "one warp per 8 input channels, or one group");
  constexpr int CIW = XC * 8;            // input channels of the partial
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int H = args.H, W = args.W, dil = ly.dil;
  const int Wp = W + (PLANAR ? 2 * kPad : dil), Hp = H + (PLANAR ? 2 * kPad : dil);
  const long long frame = (long long)Hp * Wp;
  // PLANAR: tiles of each image's rows (H Wp positions); else of all positions
  const int per_image = (H * Wp + kWgTile - 1) / kWgTile;
  const long long total = frame * args.count;
  const long long tiles = PLANAR ? (long long)per_image * args.count : (total + kWgTile - 1) / kWgTile;
  const long long plane = PLANAR ? pp_plane(H, W, args.count) / 8 : 0, guard = pp_guard(W);
  const int seg = kWgTile + 2 * dil, rank = (int)blockIdx.x - ly.first;
  const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(smem);
  constexpr uint32_t goff = XC * kWgX;
  auto pixel = [&](long long q) -> long long {
    if (q < 0 || q >= total) return -1;
    int b, rem;
    if (total < (1ll << 31)) {
      b = (int)((unsigned)q / (unsigned)frame);
      rem = (int)((unsigned)q - (unsigned)b * (unsigned)frame);
    } else {
      b = (int)(q / frame);
      rem = (int)(q - (long long)b * frame);
    }
    const int y = rem / Wp, x = rem - y * Wp;
    return y < H && x < W ? ((long long)b * H + y) * W + x : -1;
  };
  auto stage = [&](long long tile, int buf) {
    const uint32_t base = s0 + buf * kWgStage;
    if constexpr (PLANAR) {
      const int b = (int)(tile / per_image), i = (int)(tile - (long long)b * per_image) * kWgTile;
      const int n = min(kWgTile, H * Wp - i);  // positions of the tile; G past them is zero
      const long long q = guard + b * frame + (long long)kPad * Wp + i;
      if (n < kWgTile && warp != 0)
        for (int r = n + tid - 32; r < kWgTile; r += 96)
#pragma unroll
          for (int c = 0; c < GC; ++c)
            *reinterpret_cast<uint4 *>(smem + buf * kWgStage + goff + c * kWgG + r * 16) =
                make_uint4(0u, 0u, 0u, 0u);
      if (tid == 0) {
        // the buffer's last reads (ldmatrix) come before these writes
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        mbar_expect_tx(mbar + 8 * buf, (uint32_t)(XC * 3 * seg + GC * n) * 16u);
        for (int c = 0; c < XC; ++c)
          for (int ty = 0; ty < 3; ++ty)
            bulk_load(base + c * kWgX + ty * seg * 16,
                      ly.X + (c * plane + q + (long long)(ty - 1) * dil * Wp - dil) * 8,
                      (uint32_t)seg * 16u, mbar + 8 * buf);
        for (int c = 0; c < GC; ++c)
          bulk_load(base + goff + c * kWgG, ly.G + (c * plane + q) * 8, (uint32_t)n * 16u,
                    mbar + 8 * buf);
      }
    } else {
      for (int i = tid; i < 3 * seg + kWgTile; i += 128) {
        const bool isx = i < 3 * seg;
        const int ty = i / seg, row = isx ? i - ty * seg : i - 3 * seg;
        const long long q = tile * kWgTile + (isx ? (long long)(ty - 1) * dil * Wp - dil : 0) + row;
        const long long p = pixel(q);
        const int ok = p >= 0 ? 16 : 0;
        if (isx) {
#pragma unroll
          for (int c = 0; c < XC; ++c)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(
                             base + c * kWgX + i * 16),
                         "l"(ly.X + (p >= 0 ? p * XS + c * 8 : 0)), "r"(ok));
        } else {
#pragma unroll
          for (int c = 0; c < GC; ++c)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(
                             base + goff + c * kWgG + row * 16),
                         "l"(ly.G + (p >= 0 ? p * GS + c * 8 : 0)), "r"(ok));
        }
      }
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
  };
  // the lane's ldmatrix rows: X rows of tap t for pixels 0 .. 31 of the tile, G
  // rows for pixels 0 .. 15
  uint32_t xo[9], go[MT];
#pragma unroll
  for (int t = 0; t < 9; ++t)
    xo[t] = (SPLIT ? 0 : warp) * kWgX + ((t / 3) * seg + (t % 3) * dil + lane) * 16;
#pragma unroll
  for (int m = 0; m < MT; ++m) {
    const int mat = lane >> 3, c = GC == 1 ? 0 : m * 2 + (mat & 1);
    go[m] = goff + c * kWgG + ((mat >> 1) * 8 + (lane & 7)) * 16;
  }
  float acc[MT][9][4], adb[MT][4];
#pragma unroll
  for (int m = 0; m < MT; ++m) {
    adb[m][0] = adb[m][1] = adb[m][2] = adb[m][3] = 0.f;
#pragma unroll
    for (int t = 0; t < 9; ++t) acc[m][t][0] = acc[m][t][1] = acc[m][t][2] = acc[m][t][3] = 0.f;
  }
  const uint32_t ones[2] = {0x3f803f80u, 0x3f803f80u};
  if (rank < tiles) stage(rank, 0);
  int buf = 0;
  uint32_t phases = 0u;  // bit b: the parity that buffer b's copies complete next
  for (long long tile = rank; tile < tiles; tile += ly.blocks, buf ^= 1) {
    bool ok = true;
    if constexpr (PLANAR) {
      ok = mbar_wait(mbar + 8 * buf, (phases >> buf) & 1u);
    } else {
      asm volatile("cp.async.wait_all;\n" ::: "memory");
    }
    // tile staged; the other buffer is read no more (and, after a wait that ran
    // out, no copy but this one is in flight: give it one more wait)
    if (!__syncthreads_and(ok)) {
      mbar_wait(mbar + 8 * buf, (phases >> buf) & 1u);
      return false;
    }
    phases ^= 1u << buf;
    if (tile + ly.blocks < tiles) stage(tile + ly.blocks, buf ^ 1);
    const uint32_t base = s0 + buf * kWgStage;
#pragma unroll 1
    for (int k32 = SPLIT ? warp : 0; k32 < kWgTile / 32; k32 += SPLIT ? 4 : 1) {
      uint32_t ga[MT][2][4];
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
          ldsm4t(ga[m][ks], base + go[m] + (k32 * 32 + ks * 16) * 16);
          if (GC == 1) ga[m][ks][1] = ga[m][ks][3] = 0u;  // channels 8 .. 15 do not exist
        }
      // a kernel row's three taps at a time: 3 MT independent MMAs before the
      // accumulators come round again
#pragma unroll
      for (int ty = 0; ty < 3; ++ty) {
        uint32_t xb[3][4];
#pragma unroll
        for (int tx = 0; tx < 3; ++tx)
          ldsm4t(xb[tx], base + xo[ty * 3 + tx] + k32 * 32 * 16);
#pragma unroll
        for (int ks = 0; ks < 2; ++ks)
#pragma unroll
          for (int tx = 0; tx < 3; ++tx) {
            const uint32_t bb[2] = {xb[tx][2 * ks], xb[tx][2 * ks + 1]};
#pragma unroll
            for (int m = 0; m < MT; ++m) mma_bf16(acc[m][ty * 3 + tx], ga[m][ks], bb);
          }
      }
      if (SPLIT || warp == 0)
#pragma unroll
        for (int ks = 0; ks < 2; ++ks)
#pragma unroll
          for (int m = 0; m < MT; ++m) mma_bf16(adb[m], ga[m][ks], ones);
    }
  }
  // acc[m][t][0..1] -> channel 16 m + g, inputs 2q, 2q + 1; [2..3] -> channel + 8
  const int g = lane >> 2, q = lane & 3;
  float *dst = part;
  if (SPLIT) {  // the warps' sums meet in shared memory, one warp after the other
    dst = reinterpret_cast<float *>(smem);
    __syncthreads();
  }
  for (int turn = 0; turn < (SPLIT ? 4 : 1); ++turn) {
    if (!SPLIT || turn == warp)
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int co = m * 16 + h * 8 + g;
          if (co >= GC * 8) continue;
#pragma unroll
          for (int t = 0; t < 9; ++t) {
            float2 *o = reinterpret_cast<float2 *>(dst + (co * 9 + t) * CIW +
                                                   (SPLIT ? 0 : warp * 8) + 2 * q);
            const float2 old = SPLIT && turn ? *o : make_float2(0.f, 0.f);
            *o = make_float2(old.x + acc[m][t][2 * h], old.y + acc[m][t][2 * h + 1]);
          }
          if (q == 0 && (SPLIT || warp == 0)) {
            float *o = dst + kPart - 32 + co;
            *o = (SPLIT && turn ? *o : 0.f) + adb[m][2 * h];
          }
        }
    if (SPLIT) __syncthreads();
  }
  if (SPLIT) {
    for (int i = tid; i < GC * 8 * 9 * CIW; i += 128) part[i] = dst[i];
    if (tid < GC * 8) part[kPart - 32 + tid] = dst[kPart - 32 + tid];
  }
  return true;
}

template <bool PLANAR>
__global__ void __launch_bounds__(128, kWgPerSm) conv_wgrad_kernel(const WgradArgs args) {
  extern __shared__ __align__(128) uint8_t wg_smem[];
  __shared__ __align__(8) uint64_t mbars[2];
  const uint32_t mbar = (uint32_t)__cvta_generic_to_shared(mbars);
  if (threadIdx.x == 0) {
    mbar_init(mbar, 1);
    mbar_init(mbar + 8, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  bdis::pdl_enter();
  // the activations, written by other kernels' plain stores, are read by copies
  asm volatile("fence.proxy.async.global;\n" ::: "memory");
  int l = 0;
  while (l + 1 < kLayers && (int)blockIdx.x >= args.layer[l + 1].first) ++l;
  float *part = args.part + (long long)blockIdx.x * kPart;
  bool ok;
  if (l == 0)
    ok = wgrad_layer<PLANAR, 16, 1, 32, 4>(args, args.layer[0], wg_smem, mbar, part);
  else if (l == 5)
    ok = wgrad_layer<PLANAR, 32, 4, 16, 1>(args, args.layer[5], wg_smem, mbar, part);
  else
    ok = wgrad_layer<PLANAR, 32, 4, 32, 4>(args, args.layer[l], wg_smem, mbar, part);
  if (!ok && threadIdx.x == 0) atomicOr(args.fault, 1);  // the sum below is then not a number
}

struct LayerBlocks {
  int first[kLayers], blocks[kLayers];
};

// Layer and position of master element i: weight (co, tap, ci), or bias (tap = 9).
struct MasterAt {
  int l, co, tap, ci;
};
__device__ __forceinline__ MasterAt master_at(int i) {
  constexpr int first = master_w_offset(1), mid = master_w_offset(2) - first;
  const int l = i < first ? 0 : 1 + (i - first) / mid;
  const int cin = l == 0 ? 2 : 32, cout = l == 5 ? 1 : 32;
  const int r = l == 0 ? i : i - first - (l - 1) * mid;
  if (r >= cout * 9 * cin) return {l, r - cout * 9 * cin, 9, 0};
  const int co = r / (9 * cin), m = r - co * 9 * cin;
  return {l, co, m / cin, m % cin};
}

// The blocks' partial sums in master order: a block takes 32 elements, warp s
// the partials s, s + 8, ..., and the eight sums are added in order. Where a wait
// of the call's kernels ran out (`failed`), what they left is partly that of an
// earlier call: the loss and the gradient become NaN, and the network's fault
// word is set, for bdis_net_status.
__global__ void __launch_bounds__(256) reduce_grad_kernel(const float *__restrict__ part,
                                                          const LayerBlocks lb,
                                                          float *__restrict__ grad,
                                                          const int *__restrict__ failed,
                                                          float *__restrict__ loss,
                                                          int *__restrict__ fault) {
  __shared__ float slice[8][32];
  bdis::pdl_enter();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
  float sum = 0.f;
  if (i < kMasterCount) {
    const MasterAt m = master_at(i);
    const int ciw = m.l == 0 ? 8 : 32;
    const float *p = part + (long long)lb.first[m.l] * kPart +
                     (m.tap == 9 ? kPart - 32 + m.co : (m.co * 9 + m.tap) * ciw + m.ci);
#pragma unroll 8
    for (int b = warp; b < lb.blocks[m.l]; b += 8) sum += __ldg(p + (long long)b * kPart);
  }
  slice[warp][lane] = sum;
  __syncthreads();
  if (warp == 0 && i < kMasterCount) {
    for (int s = 1; s < 8; ++s) sum += slice[s][lane];
    const bool bad = __ldcg(failed) != 0;
    grad[i] = bad ? __int_as_float(0x7fc00000) : sum;
    if (bad && i == 0) {
      *loss = __int_as_float(0x7fc00000);
      atomicOr(fault, 1);
    }
  }
}

// ------------------------------------------------------ loss, weights, adam

// Huber (delta 1) loss of channel 0 of z6 (p x 16 f32) against label
// (NaN = no label), averaged over all pixels; its gradient into g6 (p x 16 bf16).
__global__ void loss_kernel(const float *__restrict__ z6, const float *__restrict__ label,
                            long long total, float inv_n, __nv_bfloat16 *__restrict__ g6,
                            float *__restrict__ loss_sum) {
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  float l = 0.f, gr = 0.f;
  if (p < total) {
    l = huber_at(z6[p * 16], label[p], inv_n, gr);
    uint4 *dst = reinterpret_cast<uint4 *>(g6 + p * 16);
    dst[0] = make_uint4(pack_bf16(gr, 0.f), 0u, 0u, 0u);
    dst[1] = make_uint4(0u, 0u, 0u, 0u);
  }
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if ((threadIdx.x & 31) == 0 && loss_sum) atomicAdd(loss_sum, l * inv_n);
}

// Master weights (f32, real channels) -> padded bf16 forward weights
// [coutP][9][cinP] and, for layers > 0, the transposed tap-flipped copies the
// data gradient uses: [cinP][9][coutP] with wt_t[ci][t][co] = w[co][8-t][ci].
__global__ void pack_weights_kernel(const float *__restrict__ master, __nv_bfloat16 *fwd,
                                    __nv_bfloat16 *bwd, int layer_offset, int cin, int cout,
                                    int cinP, int coutP) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int n = coutP * 9 * cinP;
  if (i >= n) return;
  const int co = i / (9 * cinP), rem = i - co * 9 * cinP, t = rem / cinP, ci = rem - t * cinP;
  float v = 0.f;
  if (co < cout && ci < cin) v = master[layer_offset + (co * 9 + t) * cin + ci];
  fwd[i] = __float2bfloat16_rn(v);
  if (bwd) bwd[(ci * 9 + (8 - t)) * coutP + co] = __float2bfloat16_rn(v);
}

__global__ void bias_pad_kernel(const float *__restrict__ master, float *bias, int off, int cout,
                                int coutP) {
  const int c = threadIdx.x;
  if (c < coutP) bias[c] = c < cout ? master[off + c] : 0.f;
}

// Adam on the master weights; none of it where the gradient's call failed.
__global__ void adam_kernel(float *__restrict__ w, float *__restrict__ m, float *__restrict__ v,
                            const float *__restrict__ grad, int n, float lr, float b1, float b2,
                            float eps, float c1, float c2, const int *__restrict__ failed) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || __ldcg(failed) != 0) return;
  const float gr = grad[i];
  const float mi = b1 * m[i] + (1.f - b1) * gr;
  const float vi = b2 * v[i] + (1.f - b2) * gr * gr;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Level-3 net output (channel 0 of z6) -> plain map.
__global__ void take_channel0_kernel(const float *__restrict__ z6, long long total, float *out) {
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < total) out[p] = z6[p * 16];
}

inline unsigned nblocks(long long n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// A layer's packed weights: its own, the transposed copy, the bias. Every block of
// a launch reads a layer's at the same time, so where they lie in L2 counts: a
// forward pass of 8 images of 40x30 takes 34.7 us with the layers 57,344 B apart,
// 36.2 end to end (37,376 B), and 35.2 to 36.7 at nine other distances (40,960 to
// 131,072); four images of 135x240 72.1, 74.0 and 72.1 to 74.2.
constexpr size_t kLayerBytes = 2 * 32 * 9 * 32, kLayerPitch = 57344;

struct bdis_net {
  int device = 0;
  // master weights and Adam state (f32, real channels, master order)
  float *w = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr;
  // per-layer padded bf16 weights, transposed copies, padded biases, in `packed`
  char *packed = nullptr;
  __nv_bfloat16 *wf[kLayers] = {}, *wb[kLayers] = {};
  float *bias[kLayers] = {};
  // the loss, and the word that a wait of a gradient's kernels sets when it runs
  // out; both cleared when a gradient begins
  float *loss = nullptr;
  int *failed = nullptr;
  bool inject = false;  // the next gradient begins as failed (for tests)
  long long step = 0;
  // activations for `cap` pixels
  long long cap = 0;
  // (gact: gradients of the layers' outputs, one each, or two for all layers in
  // turn; the last layer's is g6)
  __nv_bfloat16 *x0 = nullptr, *a[5] = {}, *gact[5] = {}, *g6 = nullptr;
  __nv_bfloat16 *gact_of(int l) const { return gact[2] ? gact[l] : gact[l & 1]; }
  float *z6 = nullptr;
  float *part = nullptr;  // partial weight gradients, one per block of conv_wgrad_kernel
  int part_blocks = 0;
  // device word for bdis_net_status: a bounded wait of a forward pass or of a
  // gradient's kernels ran out
  int *fault = nullptr;
  // activations in the padded planar layout for count h x w images: of
  // inference, and of training (with the gradients of the layers' outputs)
  struct Planar {
    __nv_bfloat16 *x0 = nullptr, *a[5] = {}, *g[5] = {}, *g6 = nullptr;
    float *map = nullptr;  // training: the forward map
    // grid barrier counter of the launches on these buffers (its own, so that a
    // forward pass and a gradient on two streams share nothing they write)
    unsigned *sync = nullptr;
    int h = 0, w = 0, count = 0;
    size_t plane_cap = 0, map_cap = 0;  // bytes allocated per plane, and of the map
    bool captured = false;  // a captured graph refers to them
    bool holds(int hh, int ww, int cc) const { return h == hh && w == ww && count == cc; }
  } infer, train;
  // those a captured graph refers to (and at most one more each) while other
  // shapes run
  std::vector<Planar> kept_infer, kept_train;
};

namespace {

void net_free_acts(bdis_net *n) {
  cudaFree(n->x0);
  for (auto &p : n->a) cudaFree(p);
  for (auto &p : n->gact) cudaFree(p);
  cudaFree(n->g6);
  cudaFree(n->z6);
  n->x0 = nullptr;
  for (auto &p : n->a) p = nullptr;
  for (auto &p : n->gact) p = nullptr;
  n->g6 = nullptr;
  n->z6 = nullptr;
  n->cap = 0;
}

void net_free_planar(bdis_net::Planar &p) {
  cudaFree(p.x0);
  for (auto &q : p.a) cudaFree(q);
  for (auto &q : p.g) cudaFree(q);
  cudaFree(p.g6);
  cudaFree(p.map);
  p = bdis_net::Planar();
}

// Padded planar activations for count h x w images (with `train`, also the
// gradients), zeroed (borders and guards stay zero: only real pixels are ever
// written). Another shape that fits is zeroed anew in the same memory, once the
// device has finished with the one before: a
// gradient of 64 and of 48 images of 40x30 in turn takes 247 us where reallocating
// took 1115, a forward pass 78 where it took 535. Under capture nothing may be
// waited for, and the buffers are allocated anew. Buffers that a captured graph
// refers to serve their shape only (its launches rely on the borders) and go
// aside, to `kept`, while another shape runs.
bdis_status net_reserve_planar(bdis_net::Planar &p, std::vector<bdis_net::Planar> &kept, int h,
                               int w, int count, bool train, cudaStream_t st) {
  auto mark = [&]() {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (!p.captured && cudaStreamIsCapturing(st, &cap) == cudaSuccess &&
        cap != cudaStreamCaptureStatusNone)
      p.captured = true;
  };
  if (!p.holds(h, w, count))
    for (auto &q : kept)
      if (q.holds(h, w, count)) {
        std::swap(p, q);
        break;
      }
  if (p.holds(h, w, count)) {
    mark();
    return BDIS_OK;
  }
  if (p.captured) {
    auto q = std::find_if(kept.begin(), kept.end(), [](auto &k) { return !k.captured; });
    if (q != kept.end()) {
      std::swap(p, *q);
    } else {
      kept.push_back(p);
      p = bdis_net::Planar();
    }
  }
  const size_t plane = (size_t)pp_plane(h, w, count) * sizeof(__nv_bfloat16);
  const size_t map = train ? sizeof(float) * (size_t)h * w * count : 0;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(st, &cap);
  const bool fits = plane <= p.plane_cap && map <= p.map_cap && cap == cudaStreamCaptureStatusNone;
  if (e == cudaSuccess && fits)
    e = cudaDeviceSynchronize();
  else
    net_free_planar(p);
  p.h = p.w = p.count = 0;
  auto take = [&](__nv_bfloat16 *&q, int planes, size_t extra = 0) {
    if (e == cudaSuccess && !fits) e = bdis::device_alloc((void **)&q, planes * plane + extra);
    if (e == cudaSuccess) e = cudaMemsetAsync(q, 0, planes * plane, st);
  };
  take(p.x0, 2, sizeof(unsigned));  // the counter behind the planes
  if (e == cudaSuccess && !fits)
    p.sync = reinterpret_cast<unsigned *>(reinterpret_cast<char *>(p.x0) + 2 * plane);
  for (auto &q : p.a) take(q, 4);
  if (train) {
    for (auto &q : p.g) take(q, 4);
    take(p.g6, 2);
    if (e == cudaSuccess && !fits) e = bdis::device_alloc((void **)&p.map, map);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    net_free_planar(p);
    return e == cudaErrorMemoryAllocation ? BDIS_E_NOMEM : bdis::record_cuda(e);
  }
  if (!fits) {
    p.plane_cap = plane;
    p.map_cap = map;
  }
  p.h = h;
  p.w = w;
  p.count = count;
  mark();
  return BDIS_OK;
}

// The weight gradient's partial sums.
bdis_status net_reserve_part(bdis_net *n) {
  if (n->part) return BDIS_OK;
  n->part_blocks = kWgPerSm * bdis::device_sms() + kLayers;
  if (bdis::device_alloc((void **)&n->part, sizeof(float) * kPart * n->part_blocks) != cudaSuccess) {
    cudaGetLastError();
    n->part = nullptr;
    return BDIS_E_NOMEM;
  }
  return BDIS_OK;
}

// NHWC activations for `pixels` pixels; with `train`, also the gradients of
// every layer's output (768 B per pixel in all). Where those cannot be had, two
// gradient buffers that the layers take in turn (576 B), with the planar training
// buffers given back.
bdis_status net_reserve(bdis_net *n, long long pixels, bool train) {
  if (pixels <= n->cap && (!train || n->gact[0])) return BDIS_OK;
  pixels = std::max(pixels, n->cap);
  cudaError_t e = cudaErrorMemoryAllocation;
  for (int grads = train ? 5 : 0; e != cudaSuccess; grads = 2) {
    net_free_acts(n);
    e = cudaSuccess;
    auto alloc = [&](void **p, size_t bytes) {
      if (e == cudaSuccess) e = bdis::device_alloc(p, bytes);
    };
    alloc((void **)&n->x0, pixels * 16 * 2);
    for (auto &p : n->a) alloc((void **)&p, pixels * 32 * 2);
    for (int i = 0; i < grads; ++i) alloc((void **)&n->gact[i], pixels * 32 * 2);
    alloc((void **)&n->g6, pixels * 16 * 2);
    alloc((void **)&n->z6, pixels * 16 * 4);
    if (e == cudaSuccess) break;
    cudaGetLastError();
    if (grads != 5) {
      net_free_acts(n);
      return BDIS_E_NOMEM;
    }
    if (!n->train.captured) net_free_planar(n->train);
  }
  n->cap = pixels;
  return BDIS_OK;
}

cudaError_t pack_all(bdis_net *n, cudaStream_t st) {
  for (int l = 0; l < kLayers; ++l) {
    const int cnt = kCoutP[l] * 9 * kCinP[l];
    pack_weights_kernel<<<nblocks(cnt, 256), 256, 0, st>>>(n->w, n->wf[l], l > 0 ? n->wb[l] : nullptr,
                                                           master_w_offset(l), kCin[l], kCout[l],
                                                           kCinP[l], kCoutP[l]);
    bias_pad_kernel<<<1, 32, 0, st>>>(n->w, n->bias[l],
                                      master_w_offset(l) + kCout[l] * 9 * kCin[l], kCout[l],
                                      kCoutP[l]);
  }
  return cudaGetLastError();
}

int g_sms = 0;
// convolutions: 1 = banded tcgen05 kernel for forward passes and data gradients
// (default; what it does not take runs as under 2), 2 = forward passes per tile on
// tcgen05, data gradients on mma.sync, 0 = all on mma.sync
int g_net_tc = 1;

// Dynamic shared memory of the tcgen05 kernel is exactly its slab and the
// weights (19 to 72 KB for 80-pixel-wide inputs), so up to four
// blocks share an SM: some stage their slab while others multiply. (Double-
// buffering the slab within a block measured slower: it halves the blocks per
// SM.) Images too wide for one slab (over ~200 KB) take the mma.sync kernel.
constexpr int kTcSmemMax = 200 * 1024;

template <int CIN, int COUT, int MODE>
bool conv_tc(const __nv_bfloat16 *in, const __nv_bfloat16 *wt, const float *bias, int dil,
             int H, int W, long long total, void *out, int *fault, cudaStream_t st) {
  const int smem = tc_smem_bytes<CIN, COUT>(dil, W);
  if (smem > kTcSmemMax) return false;
  // the shared-memory limit is a per-device attribute of the kernel
  static uint64_t attr_set = 0;  // bit d: set on device d
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 64 || !(attr_set >> dev & 1u)) {
    if (cudaFuncSetAttribute(conv_tc_kernel<CIN, COUT, MODE>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kTcSmemMax) != cudaSuccess) {
      cudaGetLastError();  // not sticky: clear it, the mma.sync kernel runs instead
      return false;
    }
    if (dev < 64) attr_set |= 1ull << dev;
  }
  const int count = (int)(total / ((long long)H * W));
  const long long totalp = (long long)(H + 2 * dil) * (W + 2 * dil) * count;
  const long long tiles = (totalp + 127) / 128;
  const int per_sm = std::max(1, std::min(4, (227 * 1024) / (smem + 1024)));
  const unsigned grid = (unsigned)std::min<long long>(tiles, (long long)per_sm * g_sms);
  conv_tc_kernel<CIN, COUT, MODE><<<grid, 128, smem, st>>>(in, wt, bias, dil, H, W, count, out,
                                                             fault);
  return true;
}

void init_sms() {
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
  if (g_sms <= 0) g_sms = 152;
}

template <int CIN, int COUT, int MODE>
void conv(const __nv_bfloat16 *in, const __nv_bfloat16 *wt, const float *bias, int dil, int H,
          int W, long long total, const __nv_bfloat16 *mask, void *out, int *fault,
          cudaStream_t st) {
  if (!g_sms) init_sms();
  if constexpr (MODE == kFwdRelu || MODE == kFwdLinearF32) {
    if (g_net_tc && conv_tc<CIN, COUT, MODE>(in, wt, bias, dil, H, W, total, out, fault, st))
      return;
  }
  const long long tiles = (total + 255) / 256;  // 64 pixels x 4 m-tiles per block tile
  const unsigned grid = (unsigned)std::min<long long>(tiles, (long long)g_sms * 3);
  conv_mma_kernel<CIN, COUT, MODE><<<grid, 128, 0, st>>>(in, wt, bias, dil, H, W, total, mask,
                                                         out);
}

// Band height of one layer of the fused kernel: the tallest band whose two
// slabs fit the shared memory beside the largest layer's weights and whose
// tiles fit one accumulator's tensor-memory columns; 0 if none does (images
// too wide: the per-tile kernels run instead).
constexpr int kBandWeightsMax = 36 * 4 * 128;  // 32 -> 32 channels, 9 taps

template <int CIN, int COUT>
int band_rows(int dil, int H, int W, int *nsb_out) {
  const int Wp = W + 2 * kPad, soff = dil * Wp + dil;
  for (int bh = H; bh >= 1; --bh) {
    const int tiles = (bh * Wp + 127) / 128;
    if (tiles * COUT > kBandCols) continue;
    const int nsb = tiles * 128 + 2 * soff;
    if (2 * (CIN / 8) * nsb * 16 + kBandWeightsMax <= kBandSmem) {
      *nsb_out = nsb;
      return bh;
    }
  }
  return 0;
}

// Whether images of this size fit the banded kernel (its slabs, every layer).
bool band_fits(int H, int W) {
  int nsb = 0;
  return band_rows<32, 32>(4, H, W, &nsb) && band_rows<16, 32>(1, H, W, &nsb) &&
         band_rows<32, 16>(1, H, W, &nsb);
}

// Band height of a layer of at most `limit` rows a band: of the numbers of equal
// bands per image, that whose rounds over the SMs cost least, a round being a band's
// tiles and two more for its fill and drain; at the same cost more bands only where
// they spare an eighth of the tiles. Bands of fewer rows spread a small batch over
// the SMs, but a last round that few blocks have work in costs as much as a full
// one: 64 images of 40x30 in 3 bands each were 192 bands on 152 SMs (59 us a forward
// pass by host clock), in 2 they are 128 (51); 32 in 5 bands 52, in 4 40; 100 in 2
// bands 74, in 3 61. With one tile for fill and drain, 160 images of 80x64 took 292
// us, with two 281; 512 of 32x24 181 and 175; with two and no more bands at the same
// cost, 56 of 60x34 66 where more take 62. A result does not depend on the band
// height: each position's MMAs and epilogue are the same. Only the least number of
// bands of each height is looked at (a call spends 2 us on this, not 20, where
// images are 240 rows high).
int band_height(int H, int Wp, int count, int limit) {
  int best = 0;
  long long cost = 0, work = 0;
  for (int nb = (H + limit - 1) / limit;;) {
    const int rows = (H + nb - 1) / nb, tiles = (rows * Wp + 127) / 128;
    const long long rounds = ((long long)count * ((H + rows - 1) / rows) + g_sms - 1) / g_sms;
    const long long c = rounds * (tiles + 2), w = rounds * tiles;
    if (!best || c < cost || (c == cost && 8 * w <= 7 * work)) {
      best = rows;
      cost = c;
      work = w;
    }
    if (rows == 1) return best;
    nb = (H + rows - 2) / (rows - 1);
    if ((long long)count * (nb - 1) >= 8LL * g_sms) return best;  // more rounds only add fills
  }
}

// One cooperative launch of net_chain_kernel<BACK> over `layers` layers with
// their buffers filled in (dilation included): picks the band heights. Returns
// false, having launched nothing, when the images are too wide for it or the
// device cannot run the grid cooperatively.
template <bool BACK>
bool launch_chain(bdis_net *n, BandNet &net, int H, int W, int count, cudaStream_t st) {
  const int layers = BACK ? 5 : 6;
  int nsb[6] = {}, bh[6] = {};
  for (int l = 0; l < layers; ++l)
    bh[l] = l == 0   ? band_rows<16, 32>(net.layer[l].dil, H, W, &nsb[l])
            : l == 5 ? band_rows<32, 16>(net.layer[l].dil, H, W, &nsb[l])
                     : band_rows<32, 32>(net.layer[l].dil, H, W, &nsb[l]);
  int limit[6];
  std::copy(bh, bh + 6, limit);
  int slab = 0;
  // one block per SM, or one per band where a layer has fewer bands (a
  // single image): fewer blocks meet at each grid barrier and restage the
  // weights
  long long units = 1;
  for (int l = 0; l < layers; ++l) {
    if (!bh[l]) return false;
    const int Wp = W + 2 * kPad, soff = net.layer[l].dil * Wp + net.layer[l].dil;
    int m = 0;
    while (limit[m] != bh[l]) ++m;  // the choice depends on the limit alone
    const int best = m < l ? net.layer[m].BH : band_height(H, Wp, count, bh[l]);
    if (best < bh[l]) {  // the limits still hold
      bh[l] = best;
      nsb[l] = (best * Wp + 127) / 128 * 128 + 2 * soff;
    }
    net.layer[l].BH = bh[l];
    net.layer[l].nsb = nsb[l];
    slab = std::max(slab, (l == 0 ? 2 : 4) * nsb[l] * 16);
    units = std::max(units, (long long)count * ((H + bh[l] - 1) / bh[l]));
  }
  const int smem = 2 * slab + kBandWeightsMax;
  static uint64_t attr_set = 0;  // bit d: the shared-memory limit is set on device d
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 64 || !(attr_set >> dev & 1u)) {
    if (cudaFuncSetAttribute(net_chain_kernel<BACK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kBandSmem) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    if (dev < 64) attr_set |= 1ull << dev;
  }
  net.H = H;
  net.W = W;
  net.count = count;
  net.slab_bytes = slab;
  if (cudaMemsetAsync(net.sync, 0, sizeof(unsigned), st) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const unsigned grid = (unsigned)std::min<long long>(g_sms, units);
  void *args[] = {&net};
  if (cudaLaunchCooperativeKernel((const void *)net_chain_kernel<BACK>, dim3(grid),
                                  dim3(kBandThreads), args, (size_t)smem, st) != cudaSuccess) {
    cudaGetLastError();  // not sticky: the per-tile kernels run instead
    return false;
  }
  return true;
}

// The forward pass as one cooperative launch: level planes in, the proposal
// (channel 0 of the last layer) written straight to `out`. `fault`: the word that
// a wait which ran out sets.
bool forward_planar(bdis_net *n, const bdis_net::Planar &p, const float *L3, const float *R3,
                    int r_stride, int H, int W, int count, float *out, int *fault,
                    cudaStream_t st) {
  BandNet net{};
  for (int l = 0; l < 6; ++l) {
    net.layer[l].in = l ? p.a[l - 1] : p.x0;
    net.layer[l].wt = n->wf[l];
    net.layer[l].bias = n->bias[l];
    net.layer[l].out = l < 5 ? (void *)p.a[l] : (void *)out;
    net.layer[l].dil = kDil[l];
  }
  net.L = L3;
  net.R = R3;
  net.r_stride = r_stride;
  net.sync = p.sync;
  net.fault = fault;
  return launch_chain<false>(n, net, H, W, count, st);
}

// The loss and every layer's data gradient as one cooperative launch, on the
// activations that forward_planar left.
bool backward_planar(bdis_net *n, const bdis_net::Planar &p, const float *label, int H, int W,
                     int count, cudaStream_t st) {
  BandNet net{};
  for (int i = 0; i < 5; ++i) {  // the gradient of layer l's output becomes that of its input
    const int l = 5 - i;
    net.layer[i].in = l == 5 ? p.g6 : p.g[l];
    net.layer[i].wt = n->wb[l];
    net.layer[i].mask = p.a[l - 1];
    net.layer[i].out = p.g[l - 1];
    net.layer[i].dil = kDil[l];
  }
  net.map = p.map;
  net.label = label;
  net.loss = n->loss;
  net.sync = p.sync;
  net.fault = n->failed;
  return launch_chain<true>(n, net, H, W, count, st);
}

cudaError_t forward(bdis_net *n, const float *L3, const float *R3, int r_stride, int H, int W,
                    long long total, int *fault, cudaStream_t st) {
  pack_input_kernel<<<nblocks(total, 256), 256, 0, st>>>(L3, R3, r_stride, total, n->x0);
  conv<16, 32, kFwdRelu>(n->x0, n->wf[0], n->bias[0], kDil[0], H, W, total, nullptr, n->a[0],
                         fault, st);
  for (int l = 1; l < 5; ++l)
    conv<32, 32, kFwdRelu>(n->a[l - 1], n->wf[l], n->bias[l], kDil[l], H, W, total, nullptr,
                           n->a[l], fault, st);
  conv<32, 16, kFwdLinearF32>(n->a[4], n->wf[5], n->bias[5], kDil[5], H, W, total, nullptr,
                              n->z6, fault, st);
  return cudaGetLastError();
}

// The weight gradients' blocks and arguments, on planar activations or (p null)
// NHWC ones.
void plan_weight_gradients(bdis_net *n, const bdis_net::Planar *p, int H, int W, int count,
                           WgradArgs &wa, LayerBlocks &lb) {
  // Blocks per layer: as many in all as run at once, in proportion to the
  // layers' work (a tile of the first or last layer is a fraction of a middle
  // one's)
  static const double kCost[kLayers] = {0.4, 1, 1, 1, 1, 0.6};
  long long tiles[kLayers];
  double work = 0;
  for (int l = 0; l < kLayers; ++l) {
    tiles[l] = p ? (long long)((H * (W + 2 * kPad) + kWgTile - 1) / kWgTile) * count
                 : ((long long)(H + kDil[l]) * (W + kDil[l]) * count + kWgTile - 1) / kWgTile;
    work += tiles[l] * kCost[l];
  }
  int blocks = 0;
  for (int l = 0; l < kLayers; ++l) {
    const double share = (n->part_blocks - kLayers) * tiles[l] * kCost[l] / work;
    lb.first[l] = blocks;
    lb.blocks[l] = (int)std::max(1ll, std::min(tiles[l], (long long)share));
    blocks += lb.blocks[l];
    wa.layer[l] = {p ? (l ? p->a[l - 1] : p->x0) : (l ? n->a[l - 1] : n->x0),
                   p ? (l < 5 ? p->g[l] : p->g6) : (l < 5 ? n->gact_of(l) : n->g6), kDil[l],
                   lb.first[l], lb.blocks[l]};
  }
  wa.H = H;
  wa.W = W;
  wa.count = count;
  wa.part = n->part;
  wa.fault = n->failed;
}

// Every layer's weight gradient in one launch, or (only >= 0) that layer's.
cudaError_t launch_weight_gradients(WgradArgs wa, const LayerBlocks &lb, bool planar, int only,
                                    cudaStream_t st) {
  int blocks = lb.first[kLayers - 1] + lb.blocks[kLayers - 1];
  if (only >= 0) {  // the same blocks, numbered from 0
    blocks = lb.blocks[only];
    wa.part += (long long)lb.first[only] * kPart;
    for (int l = 0; l < kLayers; ++l) wa.layer[l].first = l <= only ? 0 : INT_MAX;
  }
  auto kernel = planar ? conv_wgrad_kernel<true> : conv_wgrad_kernel<false>;
  cudaError_t e =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmem);
  if (e == cudaSuccess)
    e = bdis::launch_maybe_overlapped(kernel, dim3((unsigned)blocks), dim3(128), (size_t)kWgSmem,
                                      st, wa);
  return e;
}

// The sum of the weight gradients' partials.
cudaError_t sum_weight_gradients(bdis_net *n, const LayerBlocks &lb, cudaStream_t st) {
  return bdis::launch_maybe_overlapped(reduce_grad_kernel, dim3(nblocks(kMasterCount, 32)),
                                       dim3(256), 0, st, (const float *)n->part, lb, n->grad,
                                       (const int *)n->failed, n->loss, n->fault);
}

// Begins a gradient: its loss and its word for failed waits.
cudaError_t begin_gradient(bdis_net *n, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(n->loss, 0, sizeof(float) + sizeof(int), st);
  if (e == cudaSuccess && n->inject) e = cudaMemsetAsync(n->failed, 1, sizeof(int), st);
  return e;
}

// The gradients of NHWC activations: the data gradients layer by layer, then all
// weight gradients; each layer's weight gradient before its output's gradient is
// overwritten, where two buffers hold those (the same blocks, so the same sums).
cudaError_t gradients(bdis_net *n, int H, int W, int count, cudaStream_t st) {
  const long long total = (long long)H * W * count;
  const bool in_turn = !n->gact[2];
  WgradArgs wa{};
  LayerBlocks lb{};
  plan_weight_gradients(n, nullptr, H, W, count, wa, lb);
  cudaError_t e = cudaSuccess;
  for (int l = 5; l >= 0 && e == cudaSuccess; --l) {
    if (in_turn) e = launch_weight_gradients(wa, lb, false, l, st);
    if (e != cudaSuccess || l == 0) break;
    // g[l - 1] = (W^T g[l]) * relu'(a[l - 1])
    if (l == 5)
      conv<16, 32, kBwdDataMasked>(n->g6, n->wb[5], nullptr, kDil[5], H, W, total, n->a[4],
                                   n->gact_of(4), n->failed, st);
    else
      conv<32, 32, kBwdDataMasked>(n->gact_of(l), n->wb[l], nullptr, kDil[l], H, W, total,
                                   n->a[l - 1], n->gact_of(l - 1), n->failed, st);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && !in_turn) e = launch_weight_gradients(wa, lb, false, -1, st);
  if (e == cudaSuccess) e = sum_weight_gradients(n, lb, st);
  return e;
}

void net_release(bdis_net *n) {
  if (!n) return;
  net_free_acts(n);
  net_free_planar(n->infer);
  net_free_planar(n->train);
  for (auto &p : n->kept_infer) net_free_planar(p);
  for (auto &p : n->kept_train) net_free_planar(p);
  cudaFree(n->part);
  cudaFree(n->w);
  cudaFree(n->m);
  cudaFree(n->v);
  cudaFree(n->grad);
  cudaFree(n->loss);
  cudaFree(n->fault);
  cudaFree(n->packed);
  delete n;
}

// Whether a gradient takes the padded planar layout, for images that fit it. Its
// launches have 60 us less to set up, but a band is one image's and works in tiles
// of 128 positions of its padded rows, which large batches of images of a few
// pixels hardly fill. By the time per image, measured over 17 sizes (1x1 to 15x20)
// x 100 to 200,000 pixels (us, planar and per layer): 0.10 and 0.09 per tile, against
// 0.0018 per pixel and 0.00066 per position of the dilation-4 weight gradient's
// frame. 5555 images of 3x3: 1155 planar, 394 per layer; 111: 138 and 189; 462 of
// 9x12: 273 and 295.
bool planar_gradient(int H, int W, int count) {
  const double planar = 0.10 + 0.09 * (((long long)H * (W + 2 * kPad) + kWgTile - 1) / kWgTile);
  const double layers = 0.0018 * H * W + 0.00066 * (H + 4) * (W + 4);
  return count * (planar - layers) <= 60.0;
}

}  // namespace

namespace bdis {

bdis_status net_forward_on(bdis_net *n, const float *L, const float *R, int r_stride, int w,
                           int h, int count, float *out, cudaStream_t st) {
  const long long total = (long long)w * h * count;
  if (!g_sms) init_sms();
  if (g_net_tc == 1 && band_fits(h, w)) {
    bdis_status s = net_reserve_planar(n->infer, n->kept_infer, h, w, count, false, st);
    if (s != BDIS_OK) return s;
    if (forward_planar(n, n->infer, L, R, r_stride, h, w, count, out, n->fault, st))
      return record_cuda(cudaGetLastError());
  }
  bdis_status s = net_reserve(n, total, false);
  if (s != BDIS_OK) return s;
  cudaError_t e = forward(n, L, R, r_stride, h, w, total, n->fault, st);
  if (e == cudaSuccess) {
    take_channel0_kernel<<<nblocks(total, 256), 256, 0, st>>>(n->z6, total, out);
    e = cudaGetLastError();
  }
  return record_cuda(e);
}

}  // namespace bdis

extern "C" {

int bdis_net_weight_count(void) { return kMasterCount; }

void bdis_set_net_variant(int tensor_path) {
  g_net_tc = tensor_path < 0 ? 0 : (tensor_path > 2 ? 1 : tensor_path);
}

int bdis_get_net_variant(void) { return g_net_tc; }

bdis_status bdis_net_create(int device, const float *weights, bdis_net **out) {
  if (!out || !weights) return BDIS_E_INVALID_ARG;
  *out = nullptr;
  cudaError_t e = cudaSetDevice(device);
  if (e != cudaSuccess) return bdis::record_cuda(e);
  bdis_net *n = new (std::nothrow) bdis_net();
  if (!n) return BDIS_E_NOMEM;
  n->device = device;
  auto alloc = [&](void **p, size_t bytes) {
    if (e == cudaSuccess) e = bdis::device_alloc(p, bytes);
  };
  const size_t wb = sizeof(float) * kMasterCount;
  alloc((void **)&n->w, wb);
  alloc((void **)&n->m, wb);
  alloc((void **)&n->v, wb);
  alloc((void **)&n->grad, wb);
  alloc((void **)&n->loss, sizeof(float) + sizeof(int));
  n->failed = reinterpret_cast<int *>(n->loss + 1);
  alloc((void **)&n->fault, sizeof(int));
  alloc((void **)&n->packed, kLayers * kLayerPitch);
  for (int l = 0; l < kLayers; ++l) {
    char *p = n->packed + l * kLayerPitch;
    n->wf[l] = reinterpret_cast<__nv_bfloat16 *>(p);
    n->wb[l] = l > 0 ? reinterpret_cast<__nv_bfloat16 *>(p + kLayerBytes) : nullptr;
    n->bias[l] = reinterpret_cast<float *>(p + 2 * kLayerBytes);
  }
  if (e == cudaSuccess) e = cudaMemcpy(n->w, weights, wb, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(n->m, 0, wb);
  if (e == cudaSuccess) e = cudaMemset(n->v, 0, wb);
  if (e == cudaSuccess) e = cudaMemset(n->fault, 0, sizeof(int));
  if (e == cudaSuccess) e = pack_all(n, nullptr);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    cudaGetLastError();
    net_release(n);
    return e == cudaErrorMemoryAllocation ? BDIS_E_NOMEM : bdis::record_cuda(e);
  }
  *out = n;
  return BDIS_OK;
}

bdis_status bdis_net_forward(bdis_net *n, const float *L3, const float *R3, int r_stride,
                             int width, int height, int count, float *disparity, void *stream) {
  if (!n || !L3 || !R3 || !disparity || width < 1 || height < 1 || count < 1 ||
      (r_stride != 1 && r_stride != 2))
    return BDIS_E_INVALID_ARG;
  return bdis::net_forward_on(n, L3, R3, r_stride, width, height, count, disparity,
                              static_cast<cudaStream_t>(stream));
}

bdis_status bdis_net_gradient(bdis_net *n, const float *L3, const float *R3, int r_stride,
                              int width, int height, int count, const float *label,
                              float *loss_out, float *grad_out, void *stream) {
  if (!n || !L3 || !R3 || !label || width < 1 || height < 1 || count < 1 ||
      (r_stride != 1 && r_stride != 2))
    return BDIS_E_INVALID_ARG;
  const long long total = (long long)width * height * count;
  bdis_status s = net_reserve_part(n);
  if (s != BDIS_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaSuccess;
  if (!g_sms) init_sms();
  // Images that fit the banded kernel train in its layout: the forward pass,
  // the loss with the data gradients, and the weight gradients are one launch
  // each (64 images of 40x30: 310 us by per-layer launches, 211 now). Its
  // padded planes take 704 B per position where the NHWC ones take 768 B per
  // pixel (576 at least); a batch beyond 32 GB of them, or for which they cannot be
  // had, keeps the NHWC form, and so does a large batch of images of a few pixels.
  bool done = false;
  const double planar_bytes = 704.0 * (height + 2 * kPad) * (width + 2 * kPad) * (double)count;
  if (g_net_tc == 1 && planar_bytes <= 32e9 && planar_gradient(height, width, count) &&
      band_fits(height, width)) {
    bdis_net::Planar &p = n->train;
    s = net_reserve_planar(p, n->kept_train, height, width, count, true, st);
    if (s != BDIS_OK && s != BDIS_E_NOMEM) return s;
    done = s == BDIS_OK && begin_gradient(n, st) == cudaSuccess &&
           forward_planar(n, p, L3, R3, r_stride, height, width, count, p.map, n->failed, st) &&
           backward_planar(n, p, label, height, width, count, st);
    if (done) {
      WgradArgs wa{};
      LayerBlocks lb{};
      plan_weight_gradients(n, &p, height, width, count, wa, lb);
      e = launch_weight_gradients(wa, lb, true, -1, st);
      if (e == cudaSuccess) e = sum_weight_gradients(n, lb, st);
    }
  }
  if (!done) {
    s = net_reserve(n, total, true);
    if (s != BDIS_OK) return s;
    e = begin_gradient(n, st);
    if (e == cudaSuccess)
      e = forward(n, L3, R3, r_stride, height, width, total, n->failed, st);
    if (e == cudaSuccess) {
      loss_kernel<<<nblocks(total, 256), 256, 0, st>>>(n->z6, label, total, 1.f / (float)total,
                                                       n->g6, n->loss);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = gradients(n, height, width, count, st);
  }
  n->inject = false;
  if (e == cudaSuccess && loss_out)
    e = cudaMemcpyAsync(loss_out, n->loss, sizeof(float), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && grad_out)
    e = cudaMemcpyAsync(grad_out, n->grad, sizeof(float) * kMasterCount, cudaMemcpyDeviceToHost,
                        st);
  if (e == cudaSuccess && (loss_out || grad_out)) e = cudaStreamSynchronize(st);
  return bdis::record_cuda(e);
}

bdis_status bdis_net_train_step(bdis_net *n, const float *L3, const float *R3, int r_stride,
                                int width, int height, int count, const float *label, float lr,
                                float *loss_out, void *stream) {
  bdis_status s = bdis_net_gradient(n, L3, R3, r_stride, width, height, count, label, nullptr,
                                    nullptr, stream);
  if (s != BDIS_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  n->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)n->step), c2 = 1.f - powf(b2, (float)n->step);
  adam_kernel<<<nblocks(kMasterCount, 256), 256, 0, st>>>(n->w, n->m, n->v, n->grad, kMasterCount,
                                                          lr, b1, b2, 1e-8f, c1, c2, n->failed);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = pack_all(n, st);
  if (e == cudaSuccess && loss_out) {
    e = cudaMemcpyAsync(loss_out, n->loss, sizeof(float), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  return bdis::record_cuda(e);
}

bdis_status bdis_net_get_weights(bdis_net *n, float *weights_out) {
  if (!n || !weights_out) return BDIS_E_INVALID_ARG;
  cudaError_t e = cudaSetDevice(n->device);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e == cudaSuccess)
    e = cudaMemcpy(weights_out, n->w, sizeof(float) * kMasterCount, cudaMemcpyDeviceToHost);
  return bdis::record_cuda(e);
}

bdis_status bdis_net_status(bdis_net *n, void *stream) {
  if (!n) return BDIS_E_INVALID_ARG;
  int cur = -1;
  cudaError_t e = cudaGetDevice(&cur);
  if (e == cudaSuccess && cur != n->device) e = cudaSetDevice(n->device);
  if (e == cudaSuccess) e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
  int fault = 0;
  if (e == cudaSuccess) e = cudaMemcpy(&fault, n->fault, sizeof(int), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && fault) e = cudaMemset(n->fault, 0, sizeof(int));
  n->inject = false;
  if (e != cudaSuccess) return bdis::record_cuda(e);
  if (fault) {
    bdis::set_last_error("proposal network: a bounded wait of a forward pass (its tile was "
                         "written as NaN) or of a gradient (its loss and gradient are NaN) ran out");
    return BDIS_E_TIMEOUT;
  }
  return BDIS_OK;
}

bdis_status bdis_net_inject_timeout(bdis_net *n) {
  if (!n) return BDIS_E_INVALID_ARG;
  const int one = 1;
  cudaError_t e = cudaSetDevice(n->device);
  if (e == cudaSuccess) e = cudaMemcpy(n->fault, &one, sizeof(int), cudaMemcpyHostToDevice);
  n->inject = true;
  return bdis::record_cuda(e);
}

void bdis_net_destroy(bdis_net *n) {
  if (!n) return;
  cudaSetDevice(n->device);
  cudaDeviceSynchronize();
  net_release(n);
}

}  // extern "C"
