// Channel mixing of the learned charge/dipole network on the fifth-generation tensor cores:
// Y[M][NOUT] (+)= X[M][K] W, with X float32 activations and W a bfloat16 weight matrix.
//
// The network's linear layers (the "self-interaction" products of a Cartesian-tensor message-
// passing layer and the readout's hidden layer, Sections 2.1-2.2) mix channels at every ion:
// M = ions (x 3 Cartesian components for vector features, x 2 when a tangent is carried), K
// and NOUT are 16..64. These are the only dense contractions of the learned model.
//
// Design (sm_103a, tcgen05):
//   * one CTA of 128 threads per 128-row tile; the tile of X is read with coalesced float4
//     loads and split into two bfloat16 parts, X = X_hi + X_lo (X_hi = bf16(X),
//     X_lo = bf16(X - X_hi)), so the products keep about 16 significant bits of the float32
//     activations while the tensor cores only ever see bfloat16 operands (the weights are
//     stored in bfloat16) and accumulate in float32;
//   * both operands are staged in shared memory in the canonical K-major layout without
//     swizzle (8-row x 16-byte core matrices; core matrices adjacent along K are 128 bytes
//     apart, 8-row groups K/8 x 128 bytes apart), described by tcgen05 shared-memory
//     descriptors;
//   * one elected thread issues 2 x K/16 tcgen05.mma.kind::f16 instructions (M = 128,
//     N = NOUT, K = 16 each: first the X_hi products, then the X_lo products accumulated on
//     top) into a float32 accumulator in tensor memory (TMEM), and commits them to an
//     mbarrier;
//   * every warp waits on the mbarrier (bounded: after kSpinLimit polls it records
//     kNetFlagTimeout in the error word and skips the read-back), then reads its 32 rows of
//     the accumulator with tcgen05.ld (row = TMEM lane) and writes (or adds) them to Y by way
//     of shared memory, in whole lines;
//   * the TMEM columns are freed by the warp that allocated them before the CTA exits.
#include <cuda_bf16.h>

#include <cstdint>

#include "net.cuh"

namespace gbnet {

namespace {

constexpr int kTile = 128;
constexpr long kSpinLimit = 1L << 24;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// (x, y) rounded to bfloat16 (nearest even), x in the low half; and the halves' values
__device__ __forceinline__ uint32_t bf16_pair(float x, float y) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(x, y);
  return uint32_t(__bfloat16_as_ushort(p.x)) | (uint32_t(__bfloat16_as_ushort(p.y)) << 16);
}
__device__ __forceinline__ float bf16_lo(uint32_t p) { return __uint_as_float(p << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t p) { return __uint_as_float(p & 0xFFFF0000u); }

// Shared-memory matrix descriptor (tcgen05): start address, leading-dimension byte offset
// (between core matrices adjacent along K), stride-dimension byte offset (between 8-row
// groups), descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return uint64_t((addr & 0x3FFFFu) >> 4) | (uint64_t((lbo >> 4) & 0x3FFFu) << 16) |
         (uint64_t((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: float32 accumulator, bfloat16 A and B, both K-major,
// M = 128, N = n.
__host__ __device__ constexpr uint32_t instr_desc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(n >> 3) << 17) | (uint32_t(kTile >> 4) << 24);
}

// byte offset of element (row, k) of a K-major no-swizzle tile with K columns
__device__ __forceinline__ uint32_t kmajor_off(int row, int k, int K) {
  return uint32_t((row >> 3) * (K >> 3) * 128 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

template <int N>
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[N], int c0) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr + uint32_t(c0)));
#pragma unroll
  for (int j = 0; j < 16; ++j) v[c0 + j] = __uint_as_float(r[j]);
}

// Shared memory of a tile: X_hi, X_lo and W while the products run, the warps' result rows after
// (row stride NOUT + 4 floats, so that neither the row-wise writes nor the coalesced reads
// conflict on the banks).
template <int K, int NOUT>
struct MixSmem {
  static constexpr int operands = 2 * kTile * K * 2 + NOUT * K * 2, rows = NOUT > 0 ? kTile * (NOUT + 4) * 4 : 0;
  static constexpr int bytes = operands > rows ? operands : rows;
};

template <int K, int NOUT>
__device__ __forceinline__ void mix_tile(const MixJob& J, int tile, int* err, unsigned char* smem, uint64_t& mbar,
                                         uint32_t& tmem_slot) {
  static_assert(K % 16 == 0 && K >= 16 && K <= 64, "K: 16..64, multiple of 16");
  static_assert(NOUT % 16 == 0 && NOUT >= 16 && NOUT <= 64, "NOUT: 16..64, multiple of 16");
  constexpr int kCols = NOUT <= 32 ? 32 : 64;            // TMEM columns (power of two >= 32)
  constexpr uint32_t kBytesA = kTile * K * 2;
  unsigned char* sA_hi = smem;
  unsigned char* sA_lo = smem + kBytesA;
  unsigned char* sB = smem + 2 * kBytesA;
  const float* X = J.X;
  const int M = J.M;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long row0 = long(tile) * kTile;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(smem_u32(&tmem_slot)), "r"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&mbar)));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }

  // X tile -> (X_hi, X_lo) bfloat16 in the K-major layout; the tile is contiguous in memory
  const float4* X4 = reinterpret_cast<const float4*>(X + row0 * K);
  const long rows_left = long(M) - row0;
  float4 xv[K / 4];   // all of a thread's loads in flight
#pragma unroll
  for (int u = 0; u < K / 4; ++u) {
    const int e = tid + u * kTile;
    xv[u] = (e * 4) / K < rows_left ? X4[e] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
#pragma unroll
  for (int u = 0; u < K / 4; ++u) {
    const int e = tid + u * kTile, row = (e * 4) / K, k = (e * 4) % K;
    const float4 x = xv[u];
    const uint32_t h0 = bf16_pair(x.x, x.y), h1 = bf16_pair(x.z, x.w);
    const uint32_t l0 = bf16_pair(x.x - bf16_lo(h0), x.y - bf16_hi(h0));
    const uint32_t l1 = bf16_pair(x.z - bf16_lo(h1), x.w - bf16_hi(h1));
    const uint32_t off = kmajor_off(row, k, K);
    *reinterpret_cast<uint2*>(sA_hi + off) = make_uint2(h0, h1);
    *reinterpret_cast<uint2*>(sA_lo + off) = make_uint2(l0, l1);
  }
  // W^T [NOUT][K] bfloat16 -> K-major layout
  const uint2* W2 = reinterpret_cast<const uint2*>(J.Wt);
  for (int e = tid; e < NOUT * K / 4; e += kTile) {
    const int n = (e * 4) / K, k = (e * 4) % K;
    *reinterpret_cast<uint2*>(sB + kmajor_off(n, k, K)) = W2[e];
  }
  // make the generic-proxy shared-memory writes visible to the tensor cores (async proxy)
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;

  if (tid == 0) {
    constexpr uint32_t idesc = instr_desc(NOUT);
    constexpr uint32_t sbo = (K / 8) * 128;
    const uint32_t a_hi = smem_u32(sA_hi), a_lo = smem_u32(sA_lo), b = smem_u32(sB);
#pragma unroll
    for (int part = 0; part < 2; ++part) {
#pragma unroll
      for (int s = 0; s < K / 16; ++s) {
        const uint64_t ad = smem_desc((part ? a_lo : a_hi) + s * 256, 128, sbo);
        const uint64_t bd = smem_desc(b + s * 256, 128, sbo);
        const uint32_t acc = (part | s) ? 1u : 0u;
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
            :: "r"(tmem), "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
      }
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 :: "r"(smem_u32(&mbar)) : "memory");
  }

  // bounded wait for the products (phase 0 of the mbarrier)
  uint32_t done = 0;
  for (long it = 0; it < kSpinLimit && !done; ++it) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(smem_u32(&mbar)), "r"(0u) : "memory");
  }
  done = __all_sync(0xffffffffu, done);   // tcgen05.ld below is warp-collective
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!done) {
    if (lane == 0) atomicOr(err, kNetFlagTimeout);
  } else {
    float v[NOUT];
    const uint32_t taddr = tmem + (uint32_t(warp * 32) << 16);
#pragma unroll
    for (int c = 0; c < NOUT; c += 16) tmem_ld16<NOUT>(taddr, v, c);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    // the warp's 32 rows through shared memory (the operands are dead: every warp's products are
    // committed), so that Y is written in whole lines
    constexpr int kStride = NOUT + 4;
    float* srow = reinterpret_cast<float*>(smem) + warp * 32 * kStride;
#pragma unroll
    for (int c = 0; c < NOUT / 4; ++c)
      *reinterpret_cast<float4*>(srow + lane * kStride + 4 * c) =
          make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
    __syncwarp();
    const long base = row0 + warp * 32;
    float4* y = reinterpret_cast<float4*>(J.Y + base * NOUT);
#pragma unroll
    for (int u = 0; u < NOUT / 4; ++u) {
      const int e = lane + 32 * u, row = e / (NOUT / 4), c = e % (NOUT / 4);
      if (base + row < M) {
        float4 o = *reinterpret_cast<const float4*>(srow + row * kStride + 4 * c);
        if (J.accumulate) {
          const float4 p = y[e];
          o.x += p.x; o.y += p.y; o.z += p.z; o.w += p.w;
        }
        y[e] = o;
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(kCols));
  }
}

// One product, or two of one stage (K2 > 0: the scalar and the vector channels') in one launch:
// blocks [0, blocks_a) take a's tiles, the rest b's. A single product of a 32-frame step fills
// two to five blocks per SM and is bound by their latency (loads, products and write-back in a
// row), so pairs cost little more than the larger of the two. With the loads of a tile in flight
// together, conversions two at a time and Y written in whole lines, the gradient over 32 frames of
// 512 ions (31 products, now 19 launches) went from 1367 to 1220 us.
template <int K1, int N1, int K2, int N2>
__global__ void __launch_bounds__(kTile) k_mix(MixJob a, MixJob b, int blocks_a, int* err) {
  const int bx = gbpme::pdl_begin_block();
  constexpr int kBytes1 = MixSmem<K1, N1>::bytes, kBytes2 = MixSmem<K2, N2>::bytes;
  __shared__ __align__(1024) unsigned char smem[kBytes1 > kBytes2 ? kBytes1 : kBytes2];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_slot;
  if constexpr (K2 > 0) {
    if (bx >= blocks_a) {
      mix_tile<K2, N2>(b, bx - blocks_a, err, smem, mbar, tmem_slot);
      return;
    }
  }
  mix_tile<K1, N1>(a, bx, err, smem, mbar, tmem_slot);
}

template <int K1, int N1, int K2, int N2>
int launch_mix_kn(cudaStream_t s, const MixJob& a, const MixJob& b, int* err) {
  const int ba = a.M > 0 ? (a.M + kTile - 1) / kTile : 0, bb = K2 > 0 && b.M > 0 ? (b.M + kTile - 1) / kTile : 0;
  if (ba + bb == 0) return 0;
  gbpme::pdl_launch(k_mix<K1, N1, K2, N2>, ba + bb, kTile, 0, s, a, b, ba, err);
  gbpme::count_launch();
  return cudaGetLastError() == cudaSuccess ? 0 : PME_ERR_CUDA;
}

}  // namespace

int launch_mix(cudaStream_t s, int K, int NOUT, const MixJob& a, int* err) {
#define GBNET_MIX_CASE(k, n) \
  if (K == k && NOUT == n) return launch_mix_kn<k, n, 0, 0>(s, a, MixJob{}, err);
  GBNET_MIX_CASE(32, 48)   // A = h^s WA
  GBNET_MIX_CASE(16, 32)   // B = h^v WB; input gradient of WY
  GBNET_MIX_CASE(48, 48)   // U = m^s WU and its input gradient
  GBNET_MIX_CASE(32, 16)   // Y = m^v WY; input gradient of WB
  GBNET_MIX_CASE(32, 64)   // H = h^s Wh
  GBNET_MIX_CASE(48, 32)   // input gradient of WA
  GBNET_MIX_CASE(64, 32)   // input gradient of Wh
#undef GBNET_MIX_CASE
  return PME_ERR_UNSUPPORTED;
}

int launch_mix_pair(cudaStream_t s, int K1, int N1, const MixJob& a, int K2, int N2, const MixJob& b, int* err) {
#define GBNET_MIX_CASE(k, n, l, m) \
  if (K1 == k && N1 == n && K2 == l && N2 == m) return launch_mix_kn<k, n, l, m>(s, a, b, err);
  GBNET_MIX_CASE(32, 48, 16, 32)   // A and B
  GBNET_MIX_CASE(48, 48, 32, 16)   // U and Y
  GBNET_MIX_CASE(48, 48, 16, 32)   // input gradients of WU and WY
  GBNET_MIX_CASE(48, 32, 32, 16)   // input gradients of WA and WB
#undef GBNET_MIX_CASE
  return PME_ERR_UNSUPPORTED;
}

}  // namespace gbnet
