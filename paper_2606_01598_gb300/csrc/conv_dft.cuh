// What the hand-written mesh transforms (conv.cu, conv_two.cu) share: small DFTs in registers,
// compensated sums, the argument block and the block-to-plane map. The multiply-adds of the
// DFTs are written out: conv_two.cu is compiled with -fmad=false, so that its kernels with and
// without the virial sums round the spectra the same way.
#pragma once

#include "kernels.h"

namespace gbpme {

struct ConvArgs {
  FrameDesc one;
  FrameMaps maps;
  const int2* planes;   // batched pass A / C: block -> (frame, plane index of the frame)
  const float2* tw;     // twiddle tables
  float* mesh;          // pass A: rho base (input); pass C: Phi base (output)
  float2* spec;
  int tangent;
  int cap;              // complex entries of each plane buffer (pass A / C)
  const float* dconv;
  float inv4a2;
  double* partials;
  double* vparts;
  const float* gtab;
  const int* keep;      // tangent passes: *keep == 0 skips rho / Phi (the forward's stay)
};

// conv_two.cu: the passes of plans whose every axis splits into two register steps
int launch_two_plane(pme_plan_t p, cudaStream_t s, const ConvArgs& a, int grid, bool inverse);
int launch_two_x(pme_plan_t p, cudaStream_t s, const ConvArgs& a, int grid);
// conv_line.cu: the z and y passes of meshes whose planes do not fit in shared memory
int launch_line(pme_plan_t p, cudaStream_t s, const ConvArgs& a, bool inverse);

namespace {

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(__fmaf_rn(a.x, b.x, -(a.y * b.y)), __fmaf_rn(a.x, b.y, a.y * b.x));
}
// The odd radices' sums in packed instructions (f32x2: both parts in one issue slot, each rounded
// as alone), and a + i s b crosswise as scalar multiply-adds (a pair with its halves exchanged would
// have to be moved first). The two-step kernels issue more than they wait: forward + backward of
// the uneven batch of 256 frames 1069.5 -> 1064.2 us.
// Power-of-two DFTs stay scalar: packed too, 128^3 lost what the batch gained (258 -> 260.5 us).
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 psub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 pfma(float s, float2 a, float2 b) { return __ffma2_rn(make_float2(s, s), a, b); }
__device__ __forceinline__ float2 pmul(float s, float2 a) { return __fmul2_rn(make_float2(s, s), a); }
__device__ __forceinline__ float2 add_is(float2 a, float s, float2 b) {
  return make_float2(__fmaf_rn(-s, b.y, a.x), __fmaf_rn(s, b.x, a.y));
}
// times -i (forward transform) or +i (inverse)
template <bool INV>
__device__ __forceinline__ float2 rot(float2 a) {
  return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// R-point DFTs in place, X_k = sum_n v_n e^(-+2 pi i n k / R) (minus: forward).
template <bool INV>
__device__ __forceinline__ void dft4(float2& v0, float2& v1, float2& v2, float2& v3) {
  const float2 t0 = cadd(v0, v2), t1 = csub(v0, v2), t2 = cadd(v1, v3), t3 = rot<INV>(csub(v1, v3));
  v0 = cadd(t0, t2);
  v2 = csub(t0, t2);
  v1 = cadd(t1, t3);
  v3 = csub(t1, t3);
}

template <int A, int B, bool INV>
__device__ __forceinline__ void dft_coprime(float2* v);
template <bool INV>
__device__ __forceinline__ void dft9(float2* v);
template <bool INV>
__device__ __forceinline__ void dft16(float2* v);

template <int R, bool INV>
__device__ __forceinline__ void dft(float2* v) {
  if constexpr (R == 1) {
  } else if constexpr (R == 2) {
    const float2 a = v[0];
    v[0] = cadd(a, v[1]);
    v[1] = csub(a, v[1]);
  } else if constexpr (R == 4) {
    dft4<INV>(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 8) {
    // radix-2 split: even and odd 4-point DFTs, odd outputs times w8^k
    float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    float2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<INV>(e0, e1, e2, e3);
    dft4<INV>(o0, o1, o2, o3);
    const float h = 0.70710678118654752f;   // cos(pi / 4)
    o1 = INV ? make_float2(h * (o1.x - o1.y), h * (o1.x + o1.y)) : make_float2(h * (o1.x + o1.y), h * (o1.y - o1.x));
    o2 = rot<INV>(o2);
    o3 = INV ? make_float2(-h * (o3.x + o3.y), h * (o3.x - o3.y)) : make_float2(h * (o3.y - o3.x), -h * (o3.x + o3.y));
    v[0] = cadd(e0, o0);
    v[4] = csub(e0, o0);
    v[1] = cadd(e1, o1);
    v[5] = csub(e1, o1);
    v[2] = cadd(e2, o2);
    v[6] = csub(e2, o2);
    v[3] = cadd(e3, o3);
    v[7] = csub(e3, o3);
  } else if constexpr (R == 3) {
    const float c = -0.5f, s = 0.86602540378443865f;   // cos, sin of 2 pi / 3
    const float2 a = v[0], sm = padd(v[1], v[2]), d = psub(v[1], v[2]);
    const float2 m = pfma(c, sm, a);
    v[0] = padd(a, sm);
    v[1] = add_is(m, INV ? s : -s, d);
    v[2] = add_is(m, INV ? -s : s, d);
  } else if constexpr (R == 5) {
    const float c1 = 0.30901699437494742f, c2 = -0.80901699437494742f;   // cos 2pi/5, cos 4pi/5
    const float s1 = 0.95105651629515357f, s2 = 0.58778525229247313f;    // sin 2pi/5, sin 4pi/5
    const float2 a = v[0];
    const float2 s14 = padd(v[1], v[4]), d14 = psub(v[1], v[4]);
    const float2 s23 = padd(v[2], v[3]), d23 = psub(v[2], v[3]);
    const float2 m1 = pfma(c2, s23, pfma(c1, s14, a));
    const float2 m2 = pfma(c1, s23, pfma(c2, s14, a));
    const float2 n1 = pfma(s1, d14, pmul(s2, d23));
    const float2 n2 = pfma(s2, d14, pmul(-s1, d23));
    v[0] = padd(a, padd(s14, s23));
    v[1] = add_is(m1, INV ? 1.f : -1.f, n1);
    v[4] = add_is(m1, INV ? -1.f : 1.f, n1);
    v[2] = add_is(m2, INV ? 1.f : -1.f, n2);
    v[3] = add_is(m2, INV ? -1.f : 1.f, n2);
  } else if constexpr (R == 6) {
    dft_coprime<2, 3, INV>(v);
  } else if constexpr (R == 9) {
    dft9<INV>(v);
  } else if constexpr (R == 10) {
    dft_coprime<2, 5, INV>(v);
  } else if constexpr (R == 12) {
    dft_coprime<4, 3, INV>(v);
  } else if constexpr (R == 15) {
    dft_coprime<3, 5, INV>(v);
  } else {
    static_assert(R == 16, "radix");
    dft16<INV>(v);
  }
}

// Length A B with A and B coprime, without twiddles (Good 1958, Thomas 1963): the inputs
// n = (B n1 + A n2) mod A B go through B DFTs of A points and A DFTs of B points, and output
// (k1, k2) is X_k with k = k1 mod A, k = k2 mod B.
__host__ __device__ constexpr int inverse_mod(int a, int m) {
  for (int x = 1; x < m; ++x)
    if (a * x % m == 1) return x;
  return 1;
}
template <int A, int B, bool INV>
__device__ __forceinline__ void dft_coprime(float2* v) {
  constexpr int KA = B * inverse_mod(B, A), KB = A * inverse_mod(A, B);   // 1 mod A, 0 mod B; and the reverse
  float2 t[A][B];
#pragma unroll
  for (int n2 = 0; n2 < B; ++n2) {
    float2 u[A];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) u[n1] = v[(B * n1 + A * n2) % (A * B)];
    dft<A, INV>(u);
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) t[k1][n2] = u[k1];
  }
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    dft<B, INV>(t[k1]);
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) v[(KA * k1 + KB * k2) % (A * B)] = t[k1][k2];
  }
}

// Nine points as 3 x 3 with the twiddles w9^(n2 k1) between the two steps.
template <bool INV>
__device__ __forceinline__ void dft9(float2* v) {
  const float c1 = 0.76604444311897804f, s1 = 0.64278760968653933f;    // cos, sin of 2 pi / 9
  const float c2 = 0.17364817766693035f, s2 = 0.98480775301220806f;    // 4 pi / 9
  const float c4 = -0.93969262078590838f, s4 = 0.34202014332566873f;   // 8 pi / 9
  const float sg = INV ? 1.f : -1.f;
  float2 t[3][3];   // [k1][n2]
#pragma unroll
  for (int n2 = 0; n2 < 3; ++n2) {
    float2 u[3] = {v[n2], v[n2 + 3], v[n2 + 6]};
    dft<3, INV>(u);
    t[0][n2] = u[0];
    t[1][n2] = u[1];
    t[2][n2] = u[2];
  }
  t[1][1] = cmul(t[1][1], make_float2(c1, sg * s1));
  t[1][2] = cmul(t[1][2], make_float2(c2, sg * s2));
  t[2][1] = cmul(t[2][1], make_float2(c2, sg * s2));
  t[2][2] = cmul(t[2][2], make_float2(c4, sg * s4));
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    dft<3, INV>(t[k1]);
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = t[k1][k2];
  }
}

// 16-point DFT in registers: 4 x 4 with the twiddles w16^(n1 k1) between the two radix-4
// steps; output in natural order.
template <bool INV>
__device__ __forceinline__ void dft16(float2* v) {
  const float c1 = 0.92387953251128674f, s1 = 0.38268343236508978f, h = 0.70710678118654752f;
  float2 t[4][4];
#pragma unroll
  for (int n1 = 0; n1 < 4; ++n1) {
    float2 a0 = v[n1], a1 = v[n1 + 4], a2 = v[n1 + 8], a3 = v[n1 + 12];
    dft4<INV>(a0, a1, a2, a3);
    t[n1][0] = a0;
    t[n1][1] = a1;
    t[n1][2] = a2;
    t[n1][3] = a3;
  }
  // forward twiddles w16^j = (cos, -sin)(2 pi j / 16); the inverse takes their conjugates
  const float sg = INV ? -1.f : 1.f;
  auto tw = [&](float2 a, float wr, float wi) {   // a (wr + i sg wi)
    const float wj = sg * wi;
    return make_float2(__fmaf_rn(a.x, wr, -(a.y * wj)), __fmaf_rn(a.x, wj, a.y * wr));
  };
  t[1][1] = tw(t[1][1], c1, -s1);   // j = 1
  t[1][2] = tw(t[1][2], h, -h);     // j = 2
  t[1][3] = tw(t[1][3], s1, -c1);   // j = 3
  t[2][1] = tw(t[2][1], h, -h);     // j = 2
  t[2][2] = rot<INV>(t[2][2]);      // j = 4
  t[2][3] = tw(t[2][3], -h, -h);    // j = 6
  t[3][1] = tw(t[3][1], s1, -c1);   // j = 3
  t[3][2] = tw(t[3][2], -h, -h);    // j = 6
  t[3][3] = tw(t[3][3], -c1, s1);   // j = 9
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    float2 b0 = t[0][k1], b1 = t[1][k1], b2 = t[2][k1], b3 = t[3][k1];
    dft4<INV>(b0, b1, b2, b3);
    v[k1] = b0;
    v[k1 + 4] = b1;
    v[k1 + 8] = b2;
    v[k1 + 12] = b3;
  }
}

__device__ __forceinline__ void comp_add(float& s, float& c, float v) {
  const float t = s + v;
  c += fabsf(s) >= fabsf(v) ? (s - t) + v : (v - t) + s;
  s = t;
}

// Block sum of per-thread compensated pairs: float within a warp, float64 across warps;
// thread 0 gets the total.
__device__ double block_comp_sum(float v, float c, double* wsum) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float v2 = __shfl_xor_sync(0xffffffffu, v, o);
    const float c2 = __shfl_xor_sync(0xffffffffu, c, o);
    c += c2;
    comp_add(v, c, v2);
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = double(v) + double(c);
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < int(blockDim.x >> 5); ++w) t += wsum[w];
  return t;
}

// element t of a tile with c columns: row t / c, column t mod c. The float quotient is off
// by at most one for t < 2^20, which the correction absorbs.
__device__ __forceinline__ void split_rc(int t, int c, float rc, int& row, int& col) {
  row = int((float(t) + 0.5f) * rc);
  col = t - row * c;
  if (col < 0) {
    --row;
    col += c;
  } else if (col >= c) {
    ++row;
    col -= c;
  }
}

// Pass A / C block: frame, mesh copy (0: rho / Phi, 1: the tangent one), first plane x0 and
// plane count pc (F.conv_pp consecutive x-planes per block, fewer in the last one).
template <bool BATCH>
__device__ __forceinline__ const FrameDesc& plane_block(const ConvArgs& a, int& copy, int& x0, int& pc) {
  int f = 0, local = blockIdx.x;
  if (BATCH) {
    const int2 m = a.planes[blockIdx.x];
    f = m.x;
    local = m.y;
  }
  const FrameDesc& F = frame_at<BATCH>(a.one, a.maps, f);
  const int Nx = F.g.N[0], P = F.conv_pp;
  const int per_copy = (Nx + P - 1) / P;
  copy = local >= per_copy ? 1 : 0;
  x0 = (local - copy * per_copy) * P;
  pc = min(P, Nx - x0);
  return F;
}

// The first launch of a kernel on a device raises its dynamic shared-memory limit to the
// device's opt-in maximum (one call per kernel and device; the launch's own size decides the
// occupancy). The plan checked its sizes against that maximum when it was made.
template <typename K>
int set_smem(pme_plan_t p, K kernel, unsigned& done_mask) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 32 && (done_mask & (1u << dev))) return PME_OK;
  int optin = 0;
  int st = check_cuda(p, cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev),
                      "cudaDeviceGetAttribute");
  if (st) return st;
  st = check_cuda(p, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 1024),
                  "cudaFuncSetAttribute");
  if (!st && dev < 32) done_mask |= 1u << dev;
  return st;
}

}  // namespace

}  // namespace gbpme
