// The learned charge/dipole network and its force-matching training step (gbnet.h).
//
// Sections 2.1-2.2 of the paper: latent charges from the scalar features (Eq. charge_pred),
// dipoles from the vector features (Eq. dipole_pred) and site energies (Eq. site_energy) of a
// Cartesian-tensor message-passing net; Section 2.4: the model energy E_sr + E_PME, forces
// by differentiation through every path (Eq. forces) and the loss of Eq. loss, whose
// parameter gradient needs the derivative of the forces (a second derivative of E).
//
// Differentiation. Every kernel is written once over a scalar type T: float for a plain
// pass, Dual (value + tangent) for a pass that also carries the directional derivative
// along a position tangent r' (forward mode). Running the reverse pass (the backward
// kernels) in Dual arithmetic gives d/de [dE/dtheta (r + e r')], i.e. forward-over-reverse.
// The gradient of the force term of Eq. loss is exactly that with r' = -w,
// w = 2 lambda_f / (3 sum N) (F - F_ref); seeding the energy cotangent as 1 + e c_b,
// c_b = 2 lambda_e (E_b - E_ref,b) / (F N_b^2), adds the energy term, so the tangent part of
// one Dual backward is dL/dtheta. The PME's part of that tangent is its Hessian-vector
// product, which pme_batch_backward evaluates.
//
// Layout: every activation buffer holds two planes, [value][rows][C] then [tangent][rows][C];
// a Dual pass reads and writes both, a plain pass the first. The tensor-core products
// (net_mix.cu) treat the two planes as one matrix of 2 rows x C rows, since the tangent of
// X W is X' W. Per-ion work is one warp per ion with lane = channel; edges come from
// per-ion neighbour lists (symmetric, so the reverse-mode scatter onto senders is done as a
// gather over the receiver's own list); parameter gradients are reduced over fixed
// per-block partials (deterministic, no atomics).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "dual.cuh"
#include "net.cuh"

namespace gbnet {

using gbpme::Dual;
using gbpme::pdl_launch;
using gbpme::rcpT;
using gbpme::sqrtT;
using gbpme::sincosT;
using gbpme::sigmoidT;
using gbpme::siluT;
using gbpme::dsiluT;
using gbpme::shfl_xor;
using gbpme::warp_sum;

namespace {

constexpr int S = GBNET_SCALARS, V = GBNET_VECTORS, NR = GBNET_RADIAL;
constexpr int kMaxNbr = GBNET_MAX_NEIGHBOURS;
constexpr float kRc = float(GBNET_CUTOFF);
constexpr float kInvAvg = 1.0f / 16.0f;    // message normalisation: mean neighbour count
constexpr int kWarps = 8;                  // warps per block of the per-ion kernels
constexpr int NCOL = S + 3 * V;            // radial weight columns: ss 32, sv 16, vs 16, vv 16

// parameter offsets (floats) of the layout documented in gbnet.h
constexpr int kLayerSize = S * (S + V) + V * 2 * V + NR * NCOL + (S + V) * (S + V) + 2 * V * V;
constexpr int oEmb = 0;
constexpr int oLayer0 = 2 * S;
constexpr int oWA = 0, oWB = oWA + S * (S + V), oWR = oWB + V * 2 * V, oWU = oWR + NR * NCOL,
              oWY = oWU + (S + V) * (S + V);
constexpr int oWh = oLayer0 + 2 * kLayerSize;
constexpr int oBh = oWh + S * 2 * S;
constexpr int oWq = oBh + 2 * S;
constexpr int oBq = oWq + S;
constexpr int oWE = oBq + 1;
constexpr int oBE = oWE + S;
constexpr int oWmu = oBE + 1;
constexpr int kParams = oWmu + V;
static_assert(kParams == GBNET_NUM_PARAMS, "parameter layout");
constexpr int kReadoutW = S + S + 2 * S + 1 + 1 + V;   // wq, wE, bh, bq, bE, wmu partials

// the nine channel-mixing matrices (param offset, K = fan-in, N = fan-out)
struct MixW {
  int off, K, N;
};
constexpr int kNumMix = 9;
__host__ __device__ constexpr MixW mix_w(int w) {
  return w == 8 ? MixW{oWh, S, 2 * S}
                : (w % 4 == 0 ? MixW{oLayer0 + (w / 4) * kLayerSize + oWA, S, S + V}
                   : w % 4 == 1 ? MixW{oLayer0 + (w / 4) * kLayerSize + oWB, V, 2 * V}
                   : w % 4 == 2 ? MixW{oLayer0 + (w / 4) * kLayerSize + oWU, S + V, S + V}
                                : MixW{oLayer0 + (w / 4) * kLayerSize + oWY, 2 * V, V});
}

template <typename T> __device__ __forceinline__ T mk(float v, float d);
template <> __device__ __forceinline__ float mk<float>(float v, float) { return v; }
template <> __device__ __forceinline__ Dual mk<Dual>(float v, float d) { return Dual(v, d); }
__device__ __forceinline__ float val(float x) { return x; }
__device__ __forceinline__ float val(Dual x) { return x.v; }
__device__ __forceinline__ float tan_(float) { return 0.f; }
__device__ __forceinline__ float tan_(Dual x) { return x.d; }
// the plane a pass's parameter gradients come from: the value of a float pass, the tangent of
// a Dual one
__device__ __forceinline__ float plane_of(float x) { return x; }
__device__ __forceinline__ float plane_of(Dual x) { return x.d; }

// two-plane loads and stores: plane = floats per plane
__device__ __forceinline__ void ldv(const float* p, size_t i, size_t, float& o) { o = p[i]; }
__device__ __forceinline__ void ldv(const float* p, size_t i, size_t pl, Dual& o) { o = Dual(p[i], p[i + pl]); }
template <typename T> __device__ __forceinline__ T ldT(const float* p, size_t i, size_t pl) {
  T x;
  ldv(p, i, pl, x);
  return x;
}
__device__ __forceinline__ void stT(float* p, size_t i, size_t, float v) { p[i] = v; }
__device__ __forceinline__ void stT(float* p, size_t i, size_t pl, Dual v) { p[i] = v.v; p[i + pl] = v.d; }
// positions: value array and (Dual) tangent array
__device__ __forceinline__ void ldpos(const float* p, const float*, size_t i, float& o) { o = p[i]; }
__device__ __forceinline__ void ldpos(const float* p, const float* dp, size_t i, Dual& o) { o = Dual(p[i], dp[i]); }

template <typename T> struct Vec3 { T x, y, z; };
template <typename T> __device__ __forceinline__ T dot3(const Vec3<T>& a, const Vec3<T>& b) {
  return a.x * b.x + a.y * b.y + a.z * b.z;
}

// ---------------------------------------------------------------------------------------
// frames and neighbour lists
// ---------------------------------------------------------------------------------------
struct NetFrame {
  int off, n;
  float C[9];     // rows = lattice vectors
  float Ci[9];    // C^{-1}
  int ortho;      // orthorhombic box: the rounded fractional difference is the nearest image
};

struct Nbr {
  const int* cnt;     // [n]
  const int* j;       // [n][kMaxNbr]
  const float4* sh;   // [n][kMaxNbr]: lattice shift of the image (d = r_j - r_i + sh)
};

// One warp per ion: every other ion of the frame within r_c (nearest image), compacted in
// increasing j order.
__global__ void k_nbr(const NetFrame* __restrict__ frames, const int* frame_of,
                      const float* pos, int n, int* cnt, int* nj, float4* nsh, int* flags) {
  const int bx = gbpme::pdl_begin_block();
  const int i = bx * kWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;
  const NetFrame F = frames[frame_of[i]];
  const float xi = pos[3 * i], yi = pos[3 * i + 1], zi = pos[3 * i + 2];
  if (!(isfinite(xi) && isfinite(yi) && isfinite(zi)) && lane == 0) atomicOr(flags, kNetFlagNonFinite);
  const float rc2 = kRc * kRc;
  int c = 0;
  for (int j0 = F.off; j0 < F.off + F.n; j0 += 32) {
    const int j = j0 + lane;
    bool hit = false;
    float sx = 0.f, sy = 0.f, sz = 0.f;
    if (j < F.off + F.n && j != i) {
      const float dx = pos[3 * j] - xi, dy = pos[3 * j + 1] - yi, dz = pos[3 * j + 2] - zi;
      // fractional difference, wrapped to the nearest cell
      const float fa = rintf(dx * F.Ci[0] + dy * F.Ci[3] + dz * F.Ci[6]);
      const float fb = rintf(dx * F.Ci[1] + dy * F.Ci[4] + dz * F.Ci[7]);
      const float fc = rintf(dx * F.Ci[2] + dy * F.Ci[5] + dz * F.Ci[8]);
      const int rng = F.ortho ? 0 : 1;
      for (int a = -rng; a <= rng && !hit; ++a)
        for (int b = -rng; b <= rng && !hit; ++b)
          for (int cc = -rng; cc <= rng && !hit; ++cc) {
            const float na = -fa + a, nb = -fb + b, nc = -fc + cc;
            const float tx = na * F.C[0] + nb * F.C[3] + nc * F.C[6];
            const float ty = na * F.C[1] + nb * F.C[4] + nc * F.C[7];
            const float tz = na * F.C[2] + nb * F.C[5] + nc * F.C[8];
            const float ex = dx + tx, ey = dy + ty, ez = dz + tz;
            const float r2 = ex * ex + ey * ey + ez * ez;
            if (r2 < rc2 && r2 > 0.f) {
              hit = true;
              sx = tx; sy = ty; sz = tz;
            }
          }
    }
    const unsigned m = __ballot_sync(0xffffffffu, hit);
    const int slot = c + __popc(m & ((1u << lane) - 1u));
    if (hit && slot < kMaxNbr) {
      nj[size_t(i) * kMaxNbr + slot] = j;
      nsh[size_t(i) * kMaxNbr + slot] = make_float4(sx, sy, sz, 0.f);
    }
    c += __popc(m);
  }
  if (lane == 0) {
    if (c > kMaxNbr) atomicOr(flags, kNetFlagNbrFull);
    cnt[i] = min(c, kMaxNbr);
  }
}

// Edge geometry along one neighbour: d, r, d^, the basis e_k and de_k/dr (k = 1..8).
template <typename T>
__device__ __forceinline__ void edge_basis(const Vec3<T>& d, T& r, Vec3<T>& dh, T (&e)[NR], T (&de)[NR]) {
  const T r2 = dot3(d, d);
  r = sqrtT(r2);
  const T ri = rcpT(r);
  dh = Vec3<T>{d.x * ri, d.y * ri, d.z * ri};
  const float w = float(gbpme::kPi) / kRc;
  T s1, c1;
  sincosT(r * w, s1, c1);
  // envelope u(x) = 1 - 21 x^5 + 35 x^6 - 15 x^7 and u'(x)
  const T x = r * (1.f / kRc);
  const T x2 = x * x, x4 = x2 * x2;
  const T u = 1.f + x4 * x * (-21.f + x * (35.f - 15.f * x));
  const T du = x4 * (-105.f + x * (210.f - 105.f * x)) * (1.f / kRc);
  const float nrm = sqrtf(2.f / kRc);
  // sin(k w r) and cos(k w r) by the angle-addition recurrence
  T sk = s1, ck = c1;
#pragma unroll
  for (int k = 0; k < NR; ++k) {
    const float kw = float(k + 1) * w;
    const T a = nrm * sk * ri;                               // sqrt(2/rc) sin(k w r) / r
    const T da = nrm * (kw * ck * ri - sk * ri * ri);        // its r-derivative
    e[k] = a * u;
    de[k] = da * u + a * du;
    const T sn = sk * c1 + ck * s1, cn = ck * c1 - sk * s1;
    sk = sn;
    ck = cn;
  }
}

struct MsgArgs {
  const NetFrame* frames;
  const int* frame_of;
  Nbr nb;
  const float* pos;    // [n][3]
  const float* dpos;   // [n][3] tangent (Dual passes)
  const float* WR;     // [8][80] of this layer (float32 master)
  int n;
  size_t plS, plV;     // plane sizes: n * 48 (scalar-shaped 48) and n * 96 (vector-shaped 3 x 32)
};

// Edge records of the message kernels. The basis and geometry of an edge depend on the edge
// alone, not on the channel, so one lane forms them for one edge (a warp's 32 lanes for up to
// 32 edges of its ion at once) and stores them in shared memory, where the channel loop reads
// them back as broadcast 16-byte loads:
//   [0..1] e_1..e_8, [2] (d^, 1/r), then (DE) [3..4] de_k/dr, or (Dual) [3..4] the tangents
//   of e_k and [5] of d^.
// Formed in every lane for every edge, they were most of the kernels' instructions. With the
// weights in registers and only the outputs that a pass reads afterwards, the four message
// kernels of a gradient over 32 frames of 512 ions (265 k edges) went from 1.88 ms to about
// 0.5 ms, and the gradient from 2.87 to 1.51 ms. They wait on their neighbours' rows, so warps in
// flight count for more than the 20 to 70 bytes that a few spill: held to 64 to 128 registers, two
// to four blocks of eight warps per SM instead of one to three, the gradient went from 1489 to
// 1401 us.
template <typename T, bool DE>
struct EdgeRec {
  static constexpr bool kDual = sizeof(T) > sizeof(float);
  static_assert(!(kDual && DE), "no Dual pass uses the r-derivatives");
  static constexpr int kVec = kDual ? 6 : (DE ? 5 : 3);   // float4 per record
};

template <typename T, bool DE>
__device__ __forceinline__ void edge_store(const MsgArgs& a, const Vec3<T>& ri, int j, const float4& sh,
                                           float4* rec) {
  Vec3<T> rj;
  ldpos(a.pos, a.dpos, 3 * j, rj.x);
  ldpos(a.pos, a.dpos, 3 * j + 1, rj.y);
  ldpos(a.pos, a.dpos, 3 * j + 2, rj.z);
  const Vec3<T> d{rj.x - ri.x + sh.x, rj.y - ri.y + sh.y, rj.z - ri.z + sh.z};
  T r, e[NR], de[NR];
  Vec3<T> dh;
  edge_basis(d, r, dh, e, de);
  rec[0] = make_float4(val(e[0]), val(e[1]), val(e[2]), val(e[3]));
  rec[1] = make_float4(val(e[4]), val(e[5]), val(e[6]), val(e[7]));
  rec[2] = make_float4(val(dh.x), val(dh.y), val(dh.z), 1.f / val(r));
  if constexpr (DE) {
    rec[3] = make_float4(val(de[0]), val(de[1]), val(de[2]), val(de[3]));
    rec[4] = make_float4(val(de[4]), val(de[5]), val(de[6]), val(de[7]));
  } else if constexpr (EdgeRec<T, DE>::kDual) {
    rec[3] = make_float4(tan_(e[0]), tan_(e[1]), tan_(e[2]), tan_(e[3]));
    rec[4] = make_float4(tan_(e[4]), tan_(e[5]), tan_(e[6]), tan_(e[7]));
    rec[5] = make_float4(tan_(dh.x), tan_(dh.y), tan_(dh.z), 0.f);
  }
}

__device__ __forceinline__ void unpack8(const float4& p, const float4& q, float (&e)[NR]) {
  e[0] = p.x; e[1] = p.y; e[2] = p.z; e[3] = p.w;
  e[4] = q.x; e[5] = q.y; e[6] = q.z; e[7] = q.w;
}
__device__ __forceinline__ void edge_load(const float4* rec, float (&e)[NR], Vec3<float>& dh) {
  unpack8(rec[0], rec[1], e);
  const float4 g = rec[2];
  dh = Vec3<float>{g.x, g.y, g.z};
}
__device__ __forceinline__ void edge_load(const float4* rec, Dual (&e)[NR], Vec3<Dual>& dh) {
  float v[NR], t[NR];
  unpack8(rec[0], rec[1], v);
  unpack8(rec[3], rec[4], t);
#pragma unroll
  for (int k = 0; k < NR; ++k) e[k] = Dual(v[k], t[k]);
  const float4 g = rec[2], h = rec[5];
  dh = Vec3<Dual>{Dual(g.x, h.x), Dual(g.y, h.y), Dual(g.z, h.z)};
}

// The radial weights of this lane's channels, kept in registers: w0 ss, w1 sv (lanes of the
// first 16 channels, lo) or vv (the others), w2 vs (lo).
__device__ __forceinline__ void lane_weights(const float* __restrict__ WR, int c, bool lo, float (&w0)[NR],
                                             float (&w1)[NR], float (&w2)[NR]) {
#pragma unroll
  for (int k = 0; k < NR; ++k) {
    const float* row = WR + k * NCOL;
    w0[k] = __ldg(row + c);
    w1[k] = __ldg(row + (lo ? S + c : S + V + c));   // hi: S + 2 V + (c - V)
    w2[k] = lo ? __ldg(row + S + V + c) : 0.f;
  }
}

template <typename T>
__device__ __forceinline__ T radial(const T (&e)[NR], const float (&w)[NR]) {
  T r = e[0] * w[0];
#pragma unroll
  for (int k = 1; k < NR; ++k) r += e[k] * w[k];
  return r;
}

template <typename T>
__device__ __forceinline__ Vec3<T> ldrow3(const float* p, int j, int c, size_t pl) {
  const size_t o = size_t(j) * 3 * 2 * V + c;
  return Vec3<T>{ldT<T>(p, o, pl), ldT<T>(p, o + 2 * V, pl), ldT<T>(p, o + 4 * V, pl)};
}

// Messages of one layer: ms [n][48], mv [n][3][32] from A [n][48], B [n][3][32]. One warp per
// ion, lane = channel. FIRST: the first layer, whose vector features are zero, so B (= h^v WB)
// is too and is neither formed nor read.
template <typename T, bool FIRST>
__global__ void __launch_bounds__(32 * kWarps, sizeof(T) > 4 ? 3 : 4)
k_msg_fwd(MsgArgs a, const float* A, const float* B, float* ms, float* mv) {
  const int bx = gbpme::pdl_begin_block();
  constexpr int VEC = EdgeRec<T, false>::kVec;
  __shared__ float4 srec[kWarps][32 * VEC];
  __shared__ int sj[kWarps][32];
  const int w = threadIdx.x >> 5, c = threadIdx.x & 31;
  const int i = bx * kWarps + w;
  if (i >= a.n) return;
  const bool lo = c < V;
  float w0[NR], w1[NR], w2[NR];
  lane_weights(a.WR, c, lo, w0, w1, w2);
  Vec3<T> ri;
  ldpos(a.pos, a.dpos, 3 * i, ri.x);
  ldpos(a.pos, a.dpos, 3 * i + 1, ri.y);
  ldpos(a.pos, a.dpos, 3 * i + 2, ri.z);
  T acc_s = 0.f, acc_s2 = 0.f;
  Vec3<T> acc_v{T(0.f), T(0.f), T(0.f)};
  const int ne = a.nb.cnt[i];
  for (int q0 = 0; q0 < ne; q0 += 32) {
    const int nq = min(32, ne - q0);
    __syncwarp();
    if (c < nq) {
      const int j = a.nb.j[size_t(i) * kMaxNbr + q0 + c];
      sj[w][c] = j;
      edge_store<T, false>(a, ri, j, a.nb.sh[size_t(i) * kMaxNbr + q0 + c], &srec[w][c * VEC]);
    }
    __syncwarp();
#pragma unroll 2
    for (int q = 0; q < nq; ++q) {
      const int j = sj[w][q];
      T e[NR];
      Vec3<T> dh;
      edge_load(&srec[w][q * VEC], e, dh);
      acc_s += radial(e, w0) * ldT<T>(A, size_t(j) * (S + V) + c, a.plS);
      Vec3<T> Bj;
      if (!FIRST) Bj = ldrow3<T>(B, j, c, a.plV);
      if (lo) {
        if (!FIRST) acc_s2 += radial(e, w1) * dot3(dh, Bj);
        const T t = radial(e, w2) * ldT<T>(A, size_t(j) * (S + V) + S + c, a.plS);
        acc_v.x += t * dh.x;
        acc_v.y += t * dh.y;
        acc_v.z += t * dh.z;
      } else if (!FIRST) {
        const T R1 = radial(e, w1);
        acc_v.x += R1 * Bj.x;
        acc_v.y += R1 * Bj.y;
        acc_v.z += R1 * Bj.z;
      }
    }
  }
  stT(ms, size_t(i) * (S + V) + c, a.plS, acc_s * kInvAvg);
  if (lo) stT(ms, size_t(i) * (S + V) + S + c, a.plS, acc_s2 * kInvAvg);
  stT(mv, (size_t(i) * 3 + 0) * 2 * V + c, a.plV, acc_v.x * kInvAvg);
  stT(mv, (size_t(i) * 3 + 1) * 2 * V + c, a.plV, acc_v.y * kInvAvg);
  stT(mv, (size_t(i) * 3 + 2) * 2 * V + c, a.plV, acc_v.z * kInvAvg);
}

// Reverse pass of the messages. Inputs: the layer's A, B and the cotangents g_ms [n][48],
// g_mv [n][3][32] of its messages. POS: the position gradient g_pos [n][3] (added). GRAD: the
// cotangents g_A [n][48] and (not FIRST) g_B [n][3][32], written, and per-block partials of
// dL/dWR [8][80] (the pass's plane). A pass asks only for what is read after it: the loss's
// float pass needs the positions (and the cotangents of the second layer, GA), its Dual pass
// the parameters. FIRST: B is zero and its cotangent unused, as in k_msg_fwd.
template <typename T, bool POS, bool GA, bool GRAD, bool FIRST>
__global__ void __launch_bounds__(32 * kWarps, sizeof(T) > 4 || GRAD ? 2 : 3)
k_msg_bwd(MsgArgs a, const float* A, const float* B, const float* gms,
          const float* gmv, float* gA_out, float* gB_out, float* gpos, float* wr_part) {
  const int bx = gbpme::pdl_begin_block();
  constexpr int VEC = EdgeRec<T, POS>::kVec;
  constexpr int kRecFloats = kWarps * 32 * VEC * 4, kPartFloats = kWarps * NR * NCOL;
  // the edge records; after the edge loop the warps' partials of dL/dWR in the same place
  __shared__ __align__(16) float smem[GRAD ? (kRecFloats > kPartFloats ? kRecFloats : kPartFloats) : kRecFloats];
  __shared__ int sj[kWarps][32];
  const int w = threadIdx.x >> 5, c = threadIdx.x & 31;
  const int i = bx * kWarps + w;
  const bool lo = c < V;
  float4* srec = reinterpret_cast<float4*>(smem) + w * 32 * VEC;
  // per-lane partials of dL/dWR for this lane's columns: cols c, and (lo) S + c, S + V + c,
  // (hi) S + V + c (= S + 2 V + c - V)
  float gw0[NR], gw1[NR], gw2[NR];
#pragma unroll
  for (int k = 0; k < NR; ++k) gw0[k] = gw1[k] = gw2[k] = 0.f;
  if (i < a.n) {
    float w0[NR], w1[NR], w2[NR];
    lane_weights(a.WR, c, lo, w0, w1, w2);
    Vec3<T> ri;
    ldpos(a.pos, a.dpos, 3 * i, ri.x);
    ldpos(a.pos, a.dpos, 3 * i + 1, ri.y);
    ldpos(a.pos, a.dpos, 3 * i + 2, ri.z);
    const size_t iS = size_t(i) * (S + V);
    const Vec3<T> zero{T(0.f), T(0.f), T(0.f)};
    const T Gs_i = ldT<T>(gms, iS + c, a.plS) * kInvAvg;
    const T Gs2_i = lo && !FIRST ? ldT<T>(gms, iS + S + c, a.plS) * kInvAvg : T(0.f);
    Vec3<T> Gv_i = ldrow3<T>(gmv, i, c, a.plV);
    Gv_i = Vec3<T>{Gv_i.x * kInvAvg, Gv_i.y * kInvAvg, Gv_i.z * kInvAvg};
    T A_i = 0.f, A2_i = 0.f;
    Vec3<T> B_i = zero;
    if (POS) {
      A_i = ldT<T>(A, iS + c, a.plS);
      if (lo) A2_i = ldT<T>(A, iS + S + c, a.plS);
      if (!FIRST) B_i = ldrow3<T>(B, i, c, a.plV);
    }
    T gA = 0.f, gA2 = 0.f;
    Vec3<T> gBv = zero, gp = zero;
    const int ne = a.nb.cnt[i];
    for (int q0 = 0; q0 < ne; q0 += 32) {
      const int nq = min(32, ne - q0);
      __syncwarp();
      if (c < nq) {
        const int j = a.nb.j[size_t(i) * kMaxNbr + q0 + c];
        sj[w][c] = j;
        edge_store<T, POS>(a, ri, j, a.nb.sh[size_t(i) * kMaxNbr + q0 + c], srec + c * VEC);
      }
      __syncwarp();
      for (int q = 0; q < nq; ++q) {
        const int j = sj[w][q];
        const float4* rec = srec + q * VEC;
        T e[NR];
        Vec3<T> dh;
        edge_load(rec, e, dh);
        // neighbour's data
        const size_t jS = size_t(j) * (S + V);
        const T Gs_j = ldT<T>(gms, jS + c, a.plS) * kInvAvg;
        Vec3<T> Gv_j = ldrow3<T>(gmv, j, c, a.plV);
        Gv_j = Vec3<T>{Gv_j.x * kInvAvg, Gv_j.y * kInvAvg, Gv_j.z * kInvAvg};
        const T Gs2_j = lo && !FIRST ? ldT<T>(gms, jS + S + c, a.plS) * kInvAvg : T(0.f);
        T A_j = 0.f, A2_j = 0.f;
        Vec3<T> B_j = zero;
        if (POS || GRAD) {
          A_j = ldT<T>(A, jS + c, a.plS);
          if (lo) A2_j = ldT<T>(A, jS + S + c, a.plS);
          if (!FIRST) B_j = ldrow3<T>(B, j, c, a.plV);
        }
        // the contractions of both directions: s0, p1, p2 (or s1) of receiver i and sender j
        // (d^), t0, m1, m2 (or u1) of receiver j and sender i (d^' = -d^)
        const T s0 = Gs_i * A_j;
        T p1 = 0.f, p2 = 0.f;
        if (POS || GRAD) {
          if (lo) {
            if (!FIRST) p1 = Gs2_i * dot3(dh, B_j);
            p2 = A2_j * dot3(dh, Gv_i);
          } else if (!FIRST) {
            p1 = dot3(Gv_i, B_j);
          }
        }
        if constexpr (GRAD) {
#pragma unroll
          for (int k = 0; k < NR; ++k) {
            gw0[k] += plane_of(e[k] * s0);
            if (!FIRST) gw1[k] += plane_of(e[k] * p1);
            gw2[k] += plane_of(e[k] * p2);   // zero in the hi lanes
          }
        }
        const T dGv = dot3(dh, Gv_j);
        T R1 = 0.f, R2 = 0.f;
        if (GA || POS) {
          if (!FIRST || GA) R1 = radial(e, w1);
          R2 = radial(e, w2);
        }
        if constexpr (GA) {
          gA += radial(e, w0) * Gs_j;
          if (lo) {
            // g_A_i[32+c] += R_vs (d^' . Gv_j),  g_B_i[:,c] += R_sv d^' Gs_j[32+c]
            gA2 -= R2 * dGv;
            if (!FIRST) {
              const T f = R1 * Gs2_j;
              gBv.x -= f * dh.x;
              gBv.y -= f * dh.y;
              gBv.z -= f * dh.z;
            }
          } else if (!FIRST) {
            gBv.x += R1 * Gv_j.x;
            gBv.y += R1 * Gv_j.y;
            gBv.z += R1 * Gv_j.z;
          }
        }
        if constexpr (POS) {
          // scalar-type terms: Phi += R s, dPhi/dd = R' s d^; vector-type terms: Phi += R (d^.t),
          // dPhi/dd = R' (d^.t) d^ + R (t - (d^.t) d^) / r. With both directions (the reverse one
          // has d^' = -d^ and adds to g_pos_i with the opposite sign):
          //   g_pos_i -= radial d^ + tv
          float de[NR];
          unpack8(rec[3], rec[4], de);
          const float rinv = rec[2].w;
          T rad = radial(de, w0) * (s0 + Gs_j * A_i);
          Vec3<T> tv = zero;
          const T dR1 = FIRST ? T(0.f) : radial(de, w1);
          if (lo) {
            const T dR2 = radial(de, w2);
            const T f1 = R1 * rinv, f2 = R2 * rinv;
            // t of receiver i: Gs2_i B_j + A2_j Gv_i; of receiver j (sign flipped): Gs2_j B_i + A2_i Gv_j
            const T q1 = FIRST ? T(0.f) : p1 - Gs2_j * dot3(dh, B_i);
            const T q2 = p2 - A2_i * dGv;
            rad += dR1 * q1 + dR2 * q2 - (f1 * q1 + f2 * q2);
            tv.x = f2 * (A2_j * Gv_i.x - A2_i * Gv_j.x);
            tv.y = f2 * (A2_j * Gv_i.y - A2_i * Gv_j.y);
            tv.z = f2 * (A2_j * Gv_i.z - A2_i * Gv_j.z);
            if (!FIRST) {
              tv.x += f1 * (Gs2_i * B_j.x - Gs2_j * B_i.x);
              tv.y += f1 * (Gs2_i * B_j.y - Gs2_j * B_i.y);
              tv.z += f1 * (Gs2_i * B_j.z - Gs2_j * B_i.z);
            }
          } else if (!FIRST) {
            rad += dR1 * (p1 + dot3(Gv_j, B_i));
          }
          gp.x -= rad * dh.x + tv.x;
          gp.y -= rad * dh.y + tv.y;
          gp.z -= rad * dh.z + tv.z;
        }
      }
    }
    if constexpr (GA) {
      stT(gA_out, iS + c, a.plS, gA);
      if (lo) stT(gA_out, iS + S + c, a.plS, gA2);
      if (!FIRST) {
        stT(gB_out, (size_t(i) * 3 + 0) * 2 * V + c, a.plV, gBv.x);
        stT(gB_out, (size_t(i) * 3 + 1) * 2 * V + c, a.plV, gBv.y);
        stT(gB_out, (size_t(i) * 3 + 2) * 2 * V + c, a.plV, gBv.z);
      }
    }
    if constexpr (POS) {
      gp.x = warp_sum(gp.x);
      gp.y = warp_sum(gp.y);
      gp.z = warp_sum(gp.z);
      if (c == 0) {
        gpos[3 * size_t(i)] += val(gp.x);
        gpos[3 * size_t(i) + 1] += val(gp.y);
        gpos[3 * size_t(i) + 2] += val(gp.z);
      }
    }
  }
  if constexpr (GRAD) {
    // block partials of dL/dWR [block][NR][NCOL]: the pass's plane (value, or tangent for Dual)
    __syncthreads();
    float* sG = smem + w * NR * NCOL;
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      sG[k * NCOL + c] = gw0[k];
      sG[k * NCOL + (lo ? S + c : S + V + c)] = gw1[k];
      if (lo) sG[k * NCOL + S + V + c] = gw2[k];
    }
    __syncthreads();
    for (int k = threadIdx.x; k < NR * NCOL; k += blockDim.x) {
      float acc = 0.f;
      for (int ww = 0; ww < kWarps; ++ww) acc += smem[ww * NR * NCOL + k];
      wr_part[size_t(bx) * NR * NCOL + k] = acc;
    }
  }
}

// ---------------------------------------------------------------------------------------
// per-ion elementwise stages
// ---------------------------------------------------------------------------------------

// h^s = emb[species] (both planes: the embedding has no position tangent); h^v = 0 is not
// stored (the first layer's kernels take it as zero)
__global__ void k_embed(const float* __restrict__ P, const int* __restrict__ species, int n, float* hs, size_t plS,
                        int planes) {
  const int bx = gbpme::pdl_begin_block();
  const size_t t = size_t(bx) * blockDim.x + threadIdx.x;
  if (t >= size_t(n) * S) return;
  const int i = int(t / S), c = int(t % S);
  hs[t] = P[oEmb + species[i] * S + c];
  if (planes > 1) hs[t + plS] = 0.f;
}

// h^s_out = h^s_in + SiLU(U[:, :32]);  h^v_out = h^v_in + sigmoid(U[:, 32:]) * Y.
// One thread per (ion, scalar channel); the first 16 also do the vector channel. hv_in null:
// zero (the first layer).
template <typename T>
__global__ void k_update_fwd(int n, const float* U, const float* Y,
                             const float* hs_in, const float* hv_in, float* hs_out,
                             float* hv_out, size_t plU, size_t plY, size_t plS, size_t plV) {
  const int bx = gbpme::pdl_begin_block();
  const size_t t = size_t(bx) * blockDim.x + threadIdx.x;
  if (t >= size_t(n) * S) return;
  const size_t i = t / S;
  const int c = int(t % S);
  // (every load before the first store: the compiler cannot move them past one)
  const T h = ldT<T>(hs_in, t, plS), u = ldT<T>(U, i * (S + V) + c, plU);
  T ug = 0.f, y[3], v[3];
  if (c < V) {
    ug = ldT<T>(U, i * (S + V) + S + c, plU);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      y[a] = ldT<T>(Y, (i * 3 + a) * V + c, plY);
      if (hv_in) v[a] = ldT<T>(hv_in, (i * 3 + a) * V + c, plV);
    }
  }
  stT(hs_out, t, plS, h + siluT(u));
  if (c < V) {
    const T g = sigmoidT(ug);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const T gy = g * y[a];
      stT(hv_out, (i * 3 + a) * V + c, plV, hv_in ? v[a] + gy : gy);
    }
  }
}

// Reverse of k_update_fwd: g_U [n][48], g_Y [n][3][16] from the output cotangents g_hs, g_hv
// (which also pass unchanged to the layer input through the residual).
template <typename T>
__global__ void k_update_bwd(int n, const float* U, const float* Y,
                             const float* ghs, const float* ghv, float* gU, float* gY,
                             size_t plU, size_t plY, size_t plS, size_t plV) {
  const int bx = gbpme::pdl_begin_block();
  const size_t t = size_t(bx) * blockDim.x + threadIdx.x;
  if (t >= size_t(n) * S) return;
  const size_t i = t / S;
  const int c = int(t % S);
  const T gs = ldT<T>(ghs, t, plS), u = ldT<T>(U, i * (S + V) + c, plU);
  T ug = 0.f, gh[3], y[3];   // every load before the first store, as in k_update_fwd
  if (c < V) {
    ug = ldT<T>(U, i * (S + V) + S + c, plU);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      gh[a] = ldT<T>(ghv, (i * 3 + a) * V + c, plV);
      y[a] = ldT<T>(Y, (i * 3 + a) * V + c, plY);
    }
  }
  stT(gU, i * (S + V) + c, plU, gs * dsiluT(u));
  if (c < V) {
    const T g = sigmoidT(ug);
    T acc = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      acc += gh[a] * y[a];
      stT(gY, (i * 3 + a) * V + c, plY, gh[a] * g);
    }
    stT(gU, i * (S + V) + S + c, plU, acc * (g * (1.f - g)));
  }
}

// Readouts of one warp per ion: q~ (before neutralisation), site energy, dipole.
template <typename T>
__global__ void k_readout_fwd(int n, const float* __restrict__ P, const float* H,
                              const float* hv, float* qt, float* ei, float* mu, size_t plH,
                              size_t plV, size_t pln) {
  const int bx = gbpme::pdl_begin_block();
  const int i = bx * kWarps + (threadIdx.x >> 5), c = threadIdx.x & 31;
  if (i >= n) return;
  const T hq = ldT<T>(H, size_t(i) * 2 * S + c, plH) + P[oBh + c];
  const T he = ldT<T>(H, size_t(i) * 2 * S + S + c, plH) + P[oBh + S + c];
  T sq = P[oWq + c] * siluT(hq);
  T se = P[oWE + c] * siluT(he);
  T m[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) m[a] = c < V ? ldT<T>(hv, (size_t(i) * 3 + a) * V + c, plV) * P[oWmu + c] : T(0.f);
  sq = warp_sum(sq);
  se = warp_sum(se);
#pragma unroll
  for (int a = 0; a < 3; ++a) m[a] = warp_sum(m[a]);
  if (c == 0) {
    stT(qt, i, pln, sq + P[oBq]);
    stT(ei, i, pln, se + P[oBE]);
#pragma unroll
    for (int a = 0; a < 3; ++a) stT(mu, 3 * size_t(i) + a, 3 * pln, m[a]);
  }
}

// One block per frame: q = q~ - mean(q~) (both planes for Dual) and E_sr = sum of site
// energies (float64, value only).
template <typename T>
__global__ void k_frame_fwd(const NetFrame* __restrict__ frames, const float* qt,
                            const float* ei, float* q, double* esr, size_t pln) {
  const int bx = gbpme::pdl_begin_block();
  const NetFrame F = frames[bx];
  double sq = 0.0, sqd = 0.0, se = 0.0;
  for (int i = F.off + threadIdx.x; i < F.off + F.n; i += blockDim.x) {
    const T x = ldT<T>(qt, i, pln);
    sq += double(val(x));
    sqd += double(tan_(x));
    se += double(val(ldT<T>(ei, i, pln)));
  }
  __shared__ double red[3][32];
  sq = gbpme::warp_sum_d(sq);
  sqd = gbpme::warp_sum_d(sqd);
  se = gbpme::warp_sum_d(se);
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = sq;
    red[1][threadIdx.x >> 5] = sqd;
    red[2][threadIdx.x >> 5] = se;
  }
  __syncthreads();
  __shared__ float mean[2];
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0, e = 0.0;
    for (int w = 0; w < int(blockDim.x >> 5); ++w) {
      a += red[0][w];
      b += red[1][w];
      e += red[2][w];
    }
    mean[0] = F.n ? float(a / F.n) : 0.f;
    mean[1] = F.n ? float(b / F.n) : 0.f;
    if (esr) esr[bx] = e;
  }
  __syncthreads();
  for (int i = F.off + threadIdx.x; i < F.off + F.n; i += blockDim.x) {
    q[i] = qt[i] - mean[0];
    if (sizeof(T) > sizeof(float)) q[i + pln] = qt[i + pln] - mean[1];
  }
}

// Per-frame mean of the charge cotangent (both planes): the reverse of the neutralisation.
template <typename T>
__global__ void k_frame_mean(const NetFrame* __restrict__ frames, const float* g, float* mean,
                             size_t pln) {
  const int bx = gbpme::pdl_begin_block();
  const NetFrame F = frames[bx];
  double a = 0.0, b = 0.0;
  for (int i = F.off + threadIdx.x; i < F.off + F.n; i += blockDim.x) {
    const T x = ldT<T>(g, i, pln);
    a += double(val(x));
    b += double(tan_(x));
  }
  a = gbpme::block_sum_d(a);
  __syncthreads();
  b = gbpme::block_sum_d(b);
  if (threadIdx.x == 0) {
    mean[2 * bx] = F.n ? float(a / F.n) : 0.f;
    mean[2 * bx + 1] = F.n ? float(b / F.n) : 0.f;
  }
}

struct ReadoutBwdArgs {
  const float* P;
  const int* frame_of;
  const float* H;       // [n][64] (before the bias)
  const float* hv;      // [n][3][16] final vector features
  const float* gq;      // [n] cotangent of q (may be null)
  const float* gq_mean; // [F][2]
  const float* gmu;     // [n][3] (may be null)
  const float* gesr;    // [F] value and tangent: gesr[2 f], gesr[2 f + 1] (may be null)
  float* gH;            // [n][64]
  float* ghv;           // [n][3][16] (written)
  float* part;          // [block][kReadoutW], the pass's plane (null: no parameter gradients)
  int n;
  size_t pln, plH, plV;
};

template <typename T>
__global__ void __launch_bounds__(32 * kWarps) k_readout_bwd(ReadoutBwdArgs a) {
  const int bx = gbpme::pdl_begin_block();
  __shared__ float sp[kWarps][kReadoutW];
  const int w = threadIdx.x >> 5, c = threadIdx.x & 31;
  const int i = bx * kWarps + w;
  for (int k = c; k < kReadoutW; k += 32) sp[w][k] = 0.f;
  __syncwarp();
  if (i < a.n) {
    const int f = a.frame_of[i];
    T gqt = 0.f;
    if (a.gq) gqt = ldT<T>(a.gq, i, a.pln) - mk<T>(a.gq_mean[2 * f], a.gq_mean[2 * f + 1]);
    const T ge = a.gesr ? mk<T>(a.gesr[2 * f], a.gesr[2 * f + 1]) : T(0.f);
    const T hq = ldT<T>(a.H, size_t(i) * 2 * S + c, a.plH) + a.P[oBh + c];
    const T he = ldT<T>(a.H, size_t(i) * 2 * S + S + c, a.plH) + a.P[oBh + S + c];
    const T gHq = gqt * a.P[oWq + c] * dsiluT(hq);
    const T gHe = ge * a.P[oWE + c] * dsiluT(he);
    stT(a.gH, size_t(i) * 2 * S + c, a.plH, gHq);
    stT(a.gH, size_t(i) * 2 * S + S + c, a.plH, gHe);
    const T pwq = gqt * siluT(hq), pwe = ge * siluT(he);
    sp[w][c] = plane_of(pwq);
    sp[w][S + c] = plane_of(pwe);
    sp[w][2 * S + c] = plane_of(gHq);
    sp[w][3 * S + c] = plane_of(gHe);
    if (c == 0) {
      sp[w][4 * S] = plane_of(gqt);
      sp[w][4 * S + 1] = plane_of(ge);
    }
    if (c < V) {
      T gw = 0.f;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const T gm = a.gmu ? ldT<T>(a.gmu, 3 * size_t(i) + d, 3 * a.pln) : T(0.f);
        const size_t k = (size_t(i) * 3 + d) * V + c;
        stT(a.ghv, k, a.plV, gm * a.P[oWmu + c]);
        gw += gm * ldT<T>(a.hv, k, a.plV);
      }
      sp[w][4 * S + 2 + c] = plane_of(gw);
    }
  }
  if (!a.part) return;
  __syncthreads();
  for (int k = threadIdx.x; k < kReadoutW; k += blockDim.x) {
    float acc = 0.f;
    for (int ww = 0; ww < kWarps; ++ww) acc += sp[ww][k];
    a.part[size_t(bx) * kReadoutW + k] = acc;
  }
}

// ---------------------------------------------------------------------------------------
// parameter gradients
//
// Every parameter gradient of a backward pass is a sum over ions, formed in two launches at
// the end of the pass: k_wgrad (all channel-mixing matrices and the embedding, one block per
// matrix and chunk of rows) writes per-block partials next to those the readout and message
// kernels left, and k_reduce adds the partials of every parameter in a fixed order (float64).
// A pass wants one plane only -- the value plane of a float pass, the tangent plane of a Dual
// one -- so only that plane is formed. Bound: k_wgrad shared-memory reads and FMAs (520 M FMA
// for 32 frames of 512 ions), k_reduce the latency of the partials' loads. One thread per
// parameter walking up to 2048 partials in a row, in one to three blocks per matrix, took
// 1.83 ms of that step's 4.31 ms, and nine separate weight-gradient launches 0.28 ms; with
// thirty-two threads per parameter and one launch for all of them the step takes 2.87 ms.
// ---------------------------------------------------------------------------------------
constexpr int kWgThreads = 256;
constexpr int kWgSub = 32;       // rows staged at a time
constexpr int kWgRows = 128;     // rows per block of the scalar-channel products and the embedding
constexpr int kWgRowsV = 256;    // rows per block of the vector-channel products (3 rows per ion)

enum WgKind { kWgU, kWgY, kWgA, kWgB, kWgH, kWgEmb };

struct WgJob {
  const float* X;      // [rows][K] (embedding: unused)
  const float* G;      // [rows][N]
  size_t plX, plG;     // tangent plane offsets
  float* part;         // [blocks][K N]
  int rows, kind, first;   // first: the job's first block of the launch
};
constexpr int kWgMaxJobs = 10;
struct WgJobs {
  WgJob job[kWgMaxJobs];
  int n;
  const int* species;
};

// Staged column k, row r of a [K][kWgSub] tile: 16-byte groups of four rows permuted by a
// function of k that is distinct over eight consecutive columns (the products' reads) and over
// eight columns four apart (the transposing stores), so neither conflicts on the banks.
__device__ __forceinline__ int wg_group(int k, int g) { return k * kWgSub + 4 * (g ^ (((k >> 2) + 2 * (k & 3)) & 7)); }

template <int C>
__device__ __forceinline__ void wg_stage(const float* src, int r0, int rows, float* dst) {
  for (int e = threadIdx.x; e < kWgSub * C / 4; e += kWgThreads) {
    const int r = e / (C / 4), k = 4 * (e % (C / 4));
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r0 + r < rows) v = *reinterpret_cast<const float4*>(src + size_t(r0 + r) * C + k);
    const int g = r >> 2, o = r & 3;
    dst[wg_group(k, g) + o] = v.x;
    dst[wg_group(k + 1, g) + o] = v.y;
    dst[wg_group(k + 2, g) + o] = v.z;
    dst[wg_group(k + 3, g) + o] = v.w;
  }
}

__device__ __forceinline__ float dot4(const float4& a, const float4& b, float acc) {
  acc = fmaf(a.x, b.x, acc);
  acc = fmaf(a.y, b.y, acc);
  acc = fmaf(a.z, b.z, acc);
  return fmaf(a.w, b.w, acc);
}

// One block of a weight gradient: part[k][n] = sum over its ROWS rows of X[r][k] G[r][n]
// (PL = 1), or of X'[r][k] G[r][n] + X[r][k] G'[r][n] (PL = 2). Each thread owns TK x TN
// outputs; where those are fewer than the threads, RG groups of threads share the rows.
template <int PL, int K, int N, int TK, int TN, int ROWS>
__device__ __forceinline__ void wgrad_block(const WgJob& J, int blk, float* sm) {
  constexpr int NN = N / TN, NK = K / TK, NTH = NN * NK, RG = kWgThreads / NTH;
  static_assert(NTH * RG == kWgThreads && PL * (K + N) * kWgSub >= (RG - 1) * K * N, "thread split");
  float* sX = sm;
  float* sG = sm + PL * K * kWgSub;
  const int t = threadIdx.x % NTH, rg = threadIdx.x / NTH;
  const int n0 = t % NN, k0 = t / NN;
  float acc[TK][TN];
#pragma unroll
  for (int i = 0; i < TK; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
  const int end = min(J.rows, (blk + 1) * ROWS);
  for (int r0 = blk * ROWS; r0 < end; r0 += kWgSub) {
    __syncthreads();
    wg_stage<K>(J.X, r0, end, sX);
    wg_stage<N>(J.G, r0, end, sG);
    if (PL > 1) {
      wg_stage<K>(J.X + J.plX, r0, end, sX + K * kWgSub);
      wg_stage<N>(J.G + J.plG, r0, end, sG + N * kWgSub);
    }
    __syncthreads();
#pragma unroll 2
    for (int g = rg; g < kWgSub / 4; g += RG) {
      float4 x[PL][TK], y[PL][TN];
#pragma unroll
      for (int p = 0; p < PL; ++p) {
#pragma unroll
        for (int i = 0; i < TK; ++i)
          x[p][i] = *reinterpret_cast<const float4*>(sX + p * K * kWgSub + wg_group(k0 + NK * i, g));
#pragma unroll
        for (int j = 0; j < TN; ++j)
          y[p][j] = *reinterpret_cast<const float4*>(sG + p * N * kWgSub + wg_group(n0 + NN * j, g));
      }
#pragma unroll
      for (int i = 0; i < TK; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          if (PL > 1) acc[i][j] = dot4(x[0][i], y[PL - 1][j], dot4(x[PL - 1][i], y[0][j], acc[i][j]));
          else acc[i][j] = dot4(x[0][i], y[0][j], acc[i][j]);
        }
    }
  }
  if (RG > 1) {
    __syncthreads();
    if (rg > 0) {
#pragma unroll
      for (int i = 0; i < TK; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) sm[(rg - 1) * K * N + (k0 + NK * i) * N + n0 + NN * j] = acc[i][j];
    }
    __syncthreads();
  }
  if (rg == 0) {
    float* out = J.part + size_t(blk) * K * N;
#pragma unroll
    for (int i = 0; i < TK; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int o = (k0 + NK * i) * N + n0 + NN * j;
        float v = acc[i][j];
        for (int q = 1; q < RG; ++q) v += sm[(q - 1) * K * N + o];
        out[o] = v;
      }
  }
}

// dL/d emb [2][32] over kWgRows ions: the layer-0 input cotangent added per species.
__device__ __forceinline__ void emb_block(const WgJob& J, const int* __restrict__ species, int blk, size_t pl,
                                          float* sm) {
  const int slot = threadIdx.x >> 5, c = threadIdx.x & 31;
  float a0 = 0.f, a1 = 0.f;
#pragma unroll 4
  for (int i = blk * kWgRows + slot; i < min(J.rows, (blk + 1) * kWgRows); i += kWgThreads / 32) {
    const float g = J.G[size_t(i) * S + c + pl];
    if (species[i] == 0) a0 += g;
    else a1 += g;
  }
  sm[slot * 2 * S + c] = a0;
  sm[slot * 2 * S + S + c] = a1;
  __syncthreads();
  if (threadIdx.x < 2 * S) {
    float v = 0.f;
    for (int q = 0; q < kWgThreads / 32; ++q) v += sm[q * 2 * S + threadIdx.x];
    J.part[size_t(blk) * 2 * S + threadIdx.x] = v;
  }
}

__host__ __device__ constexpr int wg_rows(int kind) { return kind == kWgY || kind == kWgB ? kWgRowsV : kWgRows; }

template <int PL>
__global__ void __launch_bounds__(kWgThreads) k_wgrad(WgJobs jobs) {
  const int bx = gbpme::pdl_begin_block();
  __shared__ __align__(16) float sm[PL * 96 * kWgSub];
  int u = 0;
  while (u + 1 < jobs.n && bx >= jobs.job[u + 1].first) ++u;
  const WgJob& J = jobs.job[u];
  const int blk = bx - J.first;
  switch (J.kind) {
    case kWgU: wgrad_block<PL, S + V, S + V, 3, 3, kWgRows>(J, blk, sm); break;
    case kWgA: wgrad_block<PL, S, S + V, 2, 3, kWgRows>(J, blk, sm); break;
    case kWgH: wgrad_block<PL, S, 2 * S, 2, 4, kWgRows>(J, blk, sm); break;
    case kWgY: wgrad_block<PL, 2 * V, V, 2, 2, kWgRowsV>(J, blk, sm); break;
    case kWgB: wgrad_block<PL, V, 2 * V, 2, 2, kWgRowsV>(J, blk, sm); break;
    default: emb_block(J, jobs.species, blk, PL > 1 ? J.plG : 0, sm); break;
  }
}

// Parameter index of readout partial k (wq, wE, bh, bq, bE, wmu).
__device__ __forceinline__ int readout_param(int k) {
  if (k < S) return oWq + k;
  if (k < 2 * S) return oWE + (k - S);
  if (k < 4 * S) return oBh + (k - 2 * S);
  if (k == 4 * S) return oBq;
  if (k == 4 * S + 1) return oBE;
  return oWmu + (k - 4 * S - 2);
}

struct RedJob {
  const float* part;   // [nblk][width]
  int nblk, width;
  int out;             // parameter offset; -1: the readout's (readout_param)
  int first;           // first block of the launch
};
constexpr int kRedMaxJobs = 14;
struct RedJobs {
  RedJob job[kRedMaxJobs];
  int n;
};

// grad[w] (+)= sum over b of part[b][w]: 32 consecutive parameters per block, one per lane;
// warp s adds the partials b = s, s + 32, ... in float64, then the 32 sums are added in order.
// (A float32 sum with its rounding errors by two-sum is 44 us faster over 32 frames of 512 ions, but
// holds fewer bits and makes NaN of an infinite partial.)
__global__ void __launch_bounds__(1024) k_reduce(RedJobs jobs, float* grad, int accumulate) {
  const int bx = gbpme::pdl_begin_block();
  __shared__ double sum[32][33];
  int u = 0;
  while (u + 1 < jobs.n && bx >= jobs.job[u + 1].first) ++u;
  const RedJob& J = jobs.job[u];
  const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
  const int k = (bx - J.first) * 32 + lane;
  double acc = 0.0;
  if (k < J.width) {
    const float* p = J.part + k;
    for (int b0 = slice; b0 < J.nblk; b0 += 8 * 32) {   // eight loads in flight
      float v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = b0 + 32 * q < J.nblk ? p[size_t(b0 + 32 * q) * J.width] : 0.f;
#pragma unroll
      for (int q = 0; q < 8; ++q) acc += double(v[q]);
    }
  }
  sum[slice][lane] = acc;
  __syncthreads();
  if (slice == 0 && k < J.width) {
    double t = 0.0;
#pragma unroll 8
    for (int q = 0; q < 32; ++q) t += sum[q][lane];
    const int o = J.out < 0 ? readout_param(k) : J.out + k;
    grad[o] = accumulate ? grad[o] + float(t) : float(t);
  }
}

// ---------------------------------------------------------------------------------------
// loss, optimiser, weights
// ---------------------------------------------------------------------------------------

// Per frame (one block each): E_b = E_pme,b + E_sr,b; energy cotangent c_b; per ion: the
// model force F = F_pme - g_pos(net), the force residual and the position tangent r' = -w.
// part[f] = (L_E, L_F) contributions of frame f (float64).
__global__ void k_loss(const NetFrame* __restrict__ frames, int nframes, int ntot, const double* e_pme,
                       const double* e_sr, const double* e_ref,
                       const float* f_pme, const float* gpos_net,
                       const float* f_ref, double lambda_e, double lambda_f, double* cvec,
                       float* force, float* dpos, float* wneg, double* part) {
  const int bx = gbpme::pdl_begin_block();
  const NetFrame F = frames[bx];
  const double wf = 2.0 * lambda_f / (3.0 * double(ntot));
  double lf = 0.0;
  for (int t = threadIdx.x; t < 3 * F.n; t += blockDim.x) {
    const size_t k = 3 * size_t(F.off) + t;
    const float Fm = f_pme[k] - gpos_net[k];
    const float res = Fm - f_ref[k];
    if (force) force[k] = Fm;
    lf += double(res) * double(res);
    const float wv = float(wf * double(res));
    dpos[k] = -wv;
    wneg[k] = wv;     // g_force of the PME Hessian-vector product: -r' = w
  }
  lf = gbpme::block_sum_d(lf);
  if (threadIdx.x == 0) {
    const double E = e_pme[bx] + e_sr[bx];
    const double dE = (E - e_ref[bx]) / double(max(F.n, 1));
    cvec[bx] = F.n ? 2.0 * lambda_e * dE / (double(nframes) * double(F.n)) : 0.0;
    part[2 * bx] = lambda_e * dE * dE / double(nframes);
    part[2 * bx + 1] = lambda_f * lf / (3.0 * double(ntot));
  }
}

__global__ void k_loss_total(const double* part, int nframes, double* loss) {
  const int bx = gbpme::pdl_begin_block();
  double le = 0.0, lf = 0.0;   // one block
  for (int f = bx + int(threadIdx.x); f < nframes; f += blockDim.x) {
    le += part[2 * f];
    lf += part[2 * f + 1];
  }
  le = gbpme::block_sum_d(le);
  __syncthreads();
  lf = gbpme::block_sum_d(lf);
  if (threadIdx.x == 0) {
    loss[0] = le + lf;
    loss[1] = le;
    loss[2] = lf;
  }
}

// energy cotangent seeds of the Dual backward: gesr[2 f] = 1, gesr[2 f + 1] = c_f
__global__ void k_seed_esr(int nframes, const double* cvec, float* gesr, int with_tangent) {
  const int bx = gbpme::pdl_begin_block();
  const int f = bx * blockDim.x + threadIdx.x;
  if (f >= nframes) return;
  gesr[2 * f] = 1.f;
  gesr[2 * f + 1] = with_tangent ? float(cvec[f]) : 0.f;
}

// dst[k] = s * src[k] (and optionally a second array into the tangent plane of dst)
__global__ void k_scale(size_t m, const float* src, float s, float* dst) {
  const int bx = gbpme::pdl_begin_block();
  const size_t t = size_t(bx) * blockDim.x + threadIdx.x;
  if (t < m) dst[t] = s * src[t];
}

// bfloat16 copies of the channel-mixing matrices: W [K][N] and W^T [N][K]
__global__ void k_cast_weights(const float* P, uint16_t* wbf, const int* __restrict__ offs) {
  const int bx = gbpme::pdl_begin_block();
  const int w = blockIdx.y;
  const MixW m = mix_w(w);
  uint16_t* dW = wbf + offs[2 * w];
  uint16_t* dWt = wbf + offs[2 * w + 1];
  for (int t = bx * blockDim.x + threadIdx.x; t < m.K * m.N; t += gridDim.x * blockDim.x) {
    const int k = t / m.N, nn = t % m.N;
    const uint32_t u = __float_as_uint(P[m.off + t]);
    const uint16_t b = uint16_t((u + 0x7FFFu + ((u >> 16) & 1u)) >> 16);
    dW[t] = b;
    dWt[nn * m.K + k] = b;
  }
}

__global__ void k_adam(int np, float* P, float* m, float* v,
                       const float* g, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int bx = gbpme::pdl_begin_block();
  const int t = bx * blockDim.x + threadIdx.x;
  if (t >= np) return;
  const float gt = g[t];
  const float mt = b1 * m[t] + (1.f - b1) * gt;
  const float vt = b2 * v[t] + (1.f - b2) * gt * gt;
  m[t] = mt;
  v[t] = vt;
  P[t] -= lr * (mt * c1) / (sqrtf(vt * c2) + eps);
}

}  // namespace
}  // namespace gbnet

// =========================================================================================
// host side
// =========================================================================================
using gbpme::Dual;
using gbnet::NetFrame;

struct gbnet_s {
  int max_ions = 0, max_frames = 0, n = 0, nframes = 0, dev = 0;
  std::string err;
  long long launches = 0;
  int adam_step = 0;
  // parameters, optimiser state, gradients
  float *P = nullptr, *am = nullptr, *av = nullptr, *grad = nullptr, *gscratch = nullptr;
  uint16_t* wbf = nullptr;
  int* wbf_offs_d = nullptr;
  int wbf_offs[2 * gbnet::kNumMix] = {};
  int* flags = nullptr;
  // frames and neighbours
  NetFrame* frames_d = nullptr;
  std::vector<int> offsets_h;
  int* frame_of = nullptr;
  int* species = nullptr;
  int *nbr_cnt = nullptr, *nbr_j = nullptr;
  float4* nbr_sh = nullptr;
  // activations (two planes each)
  float *hs[3] = {}, *hv[3] = {}, *A[2] = {}, *B[2] = {}, *ms[2] = {}, *mv[2] = {}, *U[2] = {}, *Y[2] = {};
  float *H = nullptr, *qt = nullptr, *ei = nullptr, *q = nullptr, *mu = nullptr;
  // backward scratch
  // (the products' cotangents of both layers stay until the pass's weight gradients are formed)
  float *gA[2] = {}, *gB[2] = {}, *gU[2] = {}, *gY[2] = {};
  float *ghs = nullptr, *ghv = nullptr, *gms = nullptr, *gmv = nullptr, *gH = nullptr, *gpos = nullptr,
        *gq = nullptr, *gmu = nullptr,
        *gq_mean = nullptr, *gesr = nullptr, *part = nullptr;
  size_t part_cap = 0;
  // loss scratch
  double *e_sr = nullptr, *e_pme = nullptr, *cvec = nullptr, *lpart = nullptr;
  float *q_plain = nullptr, *mu_plain = nullptr, *f_pme = nullptr, *field = nullptr, *dpos = nullptr,
        *wneg = nullptr, *mut_neg = nullptr, *gp_scratch = nullptr, *pos_saved = nullptr;
  std::vector<void*> owned;
};

namespace gbnet {
namespace {

int fail(gbnet_t net, int st, const std::string& msg) {
  if (net) net->err = msg;
  return st;
}

int cuda_ok(gbnet_t net, cudaError_t e, const char* what) {
  if (e == cudaSuccess) return PME_OK;
  return fail(net, PME_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// A loss gradient is about eighty launches of 3 to 100 us on one stream, each waiting for the one
// before: launched with pdl_launch they are scheduled while that one drains (32 frames of 512 ions,
// 1220 -> 1124 us).
#define NET_LAUNCHED(net)                                                          \
  do {                                                                             \
    gbpme::count_launch();                                                         \
    ++(net)->launches;                                                             \
    const cudaError_t e_ = cudaGetLastError();                                     \
    if (e_ != cudaSuccess) return cuda_ok((net), e_, "kernel launch");             \
  } while (0)

inline unsigned blocks_for(size_t m, int t) { return unsigned((m + t - 1) / t); }

// One channel mixing: Y [M][N] (+)= X [M][K] with matrix w (or its transpose, the input gradient).
struct Mix {
  int M, K, N;
  const float* X;
  int w;
  bool transposed_weights;
  float* Y;
  bool acc;
};

int mix(gbnet_t net, cudaStream_t s, const Mix& m, const Mix* second = nullptr) {
  auto job = [&](const Mix& x) {
    return MixJob{x.X, net->wbf + net->wbf_offs[2 * x.w + (x.transposed_weights ? 1 : 0)], x.Y, x.M, x.acc ? 1 : 0};
  };
  const int st = second ? launch_mix_pair(s, m.K, m.N, job(m), second->K, second->N, job(*second), net->flags)
                        : launch_mix(s, m.K, m.N, job(m), net->flags);
  ++net->launches;
  return st ? fail(net, st, "channel mixing") : PME_OK;
}

template <typename T>
MsgArgs msg_args(gbnet_t net, int layer, const float* pos, const float* dpos) {
  MsgArgs a;
  a.frames = net->frames_d;
  a.frame_of = net->frame_of;
  a.nb = Nbr{net->nbr_cnt, net->nbr_j, net->nbr_sh};
  a.pos = pos;
  a.dpos = dpos;
  a.WR = net->P + oLayer0 + layer * kLayerSize + oWR;
  a.n = net->n;
  a.plS = size_t(net->n) * (S + V);
  a.plV = size_t(net->n) * 3 * 2 * V;
  return a;
}

// The message kernels, which read their neighbours' rows at random behind the products' tiles: from
// two waves on with their own L1 split (loss gradient over 32 frames of 512 ions, 2048 blocks of
// which 304 to 608 are resident: 1115 -> 1100 us).
template <auto K, typename... Args>
static void launch_l1(unsigned grid, int threads, cudaStream_t s, Args... args) {
  gbpme::launch_with(true, gbpme::own_split<K>(grid, threads, 2), K, grid, threads, 0, s, args...);
}

// forward pass; dpos is the position tangent (Dual passes only)
template <typename T>
int forward_pass(gbnet_t net, cudaStream_t s, const float* pos, const float* dpos) {
  constexpr int planes = sizeof(T) / sizeof(float);
  const int n = net->n;
  const size_t plS = size_t(n) * S, plV = size_t(n) * 3 * V, pl48 = size_t(n) * (S + V),
               pl96 = size_t(n) * 3 * 2 * V, pl64 = size_t(n) * 2 * S;
  int st;
  if (n == 0) return PME_OK;
  pdl_launch(k_embed, blocks_for(size_t(n) * S, 256), 256, 0, s,
             net->P, net->species, n, net->hs[0], plS, planes);
  NET_LAUNCHED(net);
  for (int t = 0; t < 2; ++t) {
    const Mix mA{planes * n, S, S + V, net->hs[t], 4 * t + 0, true, net->A[t], false};
    const Mix mB{planes * 3 * n, V, 2 * V, net->hv[t], 4 * t + 1, true, net->B[t], false};
    if ((st = mix(net, s, mA, t > 0 ? &mB : nullptr))) return st;   // (h^v = 0 below the first layer)
    const MsgArgs a = msg_args<T>(net, t, pos, dpos);
    if (t == 0)
      launch_l1<&k_msg_fwd<T, true>>(blocks_for(n, kWarps), 32 * kWarps, s, a, net->A[t], nullptr, net->ms[t],
                                     net->mv[t]);
    else
      launch_l1<&k_msg_fwd<T, false>>(blocks_for(n, kWarps), 32 * kWarps, s, a, net->A[t], net->B[t], net->ms[t],
                                      net->mv[t]);
    NET_LAUNCHED(net);
    const Mix mU{planes * n, S + V, S + V, net->ms[t], 4 * t + 2, true, net->U[t], false};
    const Mix mY{planes * 3 * n, 2 * V, V, net->mv[t], 4 * t + 3, true, net->Y[t], false};
    if ((st = mix(net, s, mU, &mY))) return st;
    pdl_launch(k_update_fwd<T>, blocks_for(size_t(n) * S, 256), 256, 0, s, n,
               net->U[t], net->Y[t], net->hs[t], net->hv[t], net->hs[t + 1], net->hv[t + 1], pl48, plV, plS, plV);
    NET_LAUNCHED(net);
  }
  if ((st = mix(net, s, Mix{planes * n, S, 2 * S, net->hs[2], 8, true, net->H, false}))) return st;
  pdl_launch(k_readout_fwd<T>, blocks_for(n, kWarps), 32 * kWarps, 0, s, n,
             net->P, net->H, net->hv[2], net->qt, net->ei, net->mu, pl64, plV, size_t(n));
  NET_LAUNCHED(net);
  pdl_launch(k_frame_fwd<T>, net->nframes, 256, 0, s, net->frames_d, net->qt, net->ei, net->q, net->e_sr,
             size_t(n));
  NET_LAUNCHED(net);
  (void)pl96;
  return PME_OK;
}

// Offsets (floats) of the partial sums of one backward pass over n ions.
struct PartLayout {
  size_t readout, wr[2], u[2], y[2], a[2], b[2], h, emb, total;
};
PartLayout part_layout(int n) {
  const size_t ion = blocks_for(size_t(n), kWarps), row = blocks_for(size_t(n), kWgRows),
               rowv = blocks_for(3 * size_t(n), kWgRowsV);
  PartLayout L;
  size_t o = 0;
  auto take = [&](size_t blocks, size_t width) {
    const size_t at = o;
    o += blocks * width;
    return at;
  };
  L.readout = take(ion, kReadoutW);
  for (int t = 0; t < 2; ++t) {
    L.wr[t] = take(ion, NR * NCOL);
    L.u[t] = take(row, (S + V) * (S + V));
    L.y[t] = take(rowv, 2 * V * V);
    L.a[t] = take(row, S * (S + V));
    L.b[t] = take(rowv, V * 2 * V);
  }
  L.h = take(row, S * 2 * S);
  L.emb = take(row, 2 * S);
  L.total = o;
  return L;
}

// The parameter gradients of a backward pass whose cotangents are in place: grad (+)= ...
template <typename T>
int param_grads(gbnet_t net, cudaStream_t s, float* grad, bool acc) {
  constexpr int planes = sizeof(T) / sizeof(float);
  const int n = net->n;
  const PartLayout L = part_layout(n);
  float* P = net->part;
  WgJobs wj{};
  RedJobs rj{};
  int wblocks = 0, rblocks = 0;
  auto red = [&](const float* part, int nblk, int width, int out) {
    rj.job[rj.n++] = RedJob{part, nblk, width, out, rblocks};
    rblocks += int(blocks_for(size_t(width), 32));
  };
  auto wg = [&](int kind, int rows, const float* X, int K, const float* G, int N, size_t off, int out) {
    const int nblk = int(blocks_for(size_t(rows), wg_rows(kind)));
    wj.job[wj.n++] = WgJob{X, G, size_t(rows) * K, size_t(rows) * N, P + off, rows, kind, wblocks};
    wblocks += nblk;
    red(P + off, nblk, K * N, out);
  };
  for (int t = 1; t >= 0; --t) {
    const int base = oLayer0 + t * kLayerSize;
    wg(kWgU, n, net->ms[t], S + V, net->gU[t], S + V, L.u[t], base + oWU);
    wg(kWgA, n, net->hs[t], S, net->gA[t], S + V, L.a[t], base + oWA);
    wg(kWgY, 3 * n, net->mv[t], 2 * V, net->gY[t], V, L.y[t], base + oWY);
    if (t > 0) wg(kWgB, 3 * n, net->hv[t], V, net->gB[t], 2 * V, L.b[t], base + oWB);
    else red(P + L.b[t], 0, V * 2 * V, base + oWB);   // h^v = 0: a zero gradient, no partials
    red(P + L.wr[t], int(blocks_for(size_t(n), kWarps)), NR * NCOL, base + oWR);
  }
  wg(kWgH, n, net->hs[2], S, net->gH, 2 * S, L.h, oWh);
  wg(kWgEmb, n, nullptr, 2, net->ghs, S, L.emb, oEmb);
  rj.job[rj.n - 1].width = 2 * S;   // two species rows of S channels
  red(P + L.readout, int(blocks_for(size_t(n), kWarps)), kReadoutW, -1);
  wj.species = net->species;
  pdl_launch(k_wgrad<planes>, wblocks, kWgThreads, 0, s, wj);
  NET_LAUNCHED(net);
  pdl_launch(k_reduce, rblocks, 1024, 0, s, rj, grad, acc ? 1 : 0);
  NET_LAUNCHED(net);
  return PME_OK;
}

// Backward pass of the last forward_pass<T>. Seeds: gq [planes][n], gmu [planes][n][3] (each
// may be null), gesr_f [F][2] float (value, tangent). Outputs: gpos [planes][n][3] (net->gpos,
// written; a Dual pass forms only its parameter gradients) and, unless grad is null, the parameter gradients: the value plane of a float pass,
// the tangent plane of a Dual one (written, or added when acc).
template <typename T>
int backward_pass(gbnet_t net, cudaStream_t s, const float* pos, const float* dpos, const float* gq,
                  const float* gmu, const float* gesr_f, float* grad, bool acc) {
  constexpr int planes = sizeof(T) / sizeof(float);
  const int n = net->n;
  const size_t plS = size_t(n) * S, plV = size_t(n) * 3 * V, pl48 = size_t(n) * (S + V),
               pl96 = size_t(n) * 3 * 2 * V, pl64 = size_t(n) * 2 * S;
  const PartLayout L = part_layout(n);
  int st;
  if ((st = cuda_ok(net, cudaMemsetAsync(net->gpos, 0, sizeof(float) * planes * 3 * size_t(n), s), "memset")))
    return st;
  if (n == 0) return PME_OK;
  if (gq) {
    pdl_launch(k_frame_mean<T>, net->nframes, 256, 0, s, net->frames_d, gq, net->gq_mean, size_t(n));
    NET_LAUNCHED(net);
  }
  ReadoutBwdArgs ra;
  ra.P = net->P;
  ra.frame_of = net->frame_of;
  ra.H = net->H;
  ra.hv = net->hv[2];
  ra.gq = gq;
  ra.gq_mean = net->gq_mean;
  ra.gmu = gmu;
  ra.gesr = gesr_f;
  ra.gH = net->gH;
  ra.ghv = net->ghv;
  ra.part = grad ? net->part + L.readout : nullptr;
  ra.n = n;
  ra.pln = size_t(n);
  ra.plH = pl64;
  ra.plV = plV;
  const int nb_ion = int(blocks_for(n, kWarps));
  pdl_launch(k_readout_bwd<T>, nb_ion, 32 * kWarps, 0, s, ra);
  NET_LAUNCHED(net);
  if ((st = mix(net, s, Mix{planes * n, 2 * S, S, net->gH, 8, false, net->ghs, false}))) return st;
  for (int t = 1; t >= 0; --t) {
    pdl_launch(k_update_bwd<T>, blocks_for(size_t(n) * S, 256), 256, 0, s, n,
               net->U[t], net->Y[t], net->ghs, net->ghv, net->gU[t], net->gY[t], pl48, plV, plS, plV);
    NET_LAUNCHED(net);
    const Mix mU{planes * n, S + V, S + V, net->gU[t], 4 * t + 2, false, net->gms, false};
    const Mix mY{planes * 3 * n, V, 2 * V, net->gY[t], 4 * t + 3, false, net->gmv, false};
    if ((st = mix(net, s, mU, &mY))) return st;
    const MsgArgs a = msg_args<T>(net, t, pos, dpos);
    float* wr = grad ? net->part + L.wr[t] : nullptr;
#define GB_MSG_BWD(POS, GA, GRAD, FIRST)                                                                          \
  launch_l1<&k_msg_bwd<T, POS, GA, GRAD, FIRST>>(nb_ion, 32 * kWarps, s, a,                                     \
             net->A[t], net->B[t], net->gms, net->gmv, net->gA[t], net->gB[t], net->gpos, wr)
    if constexpr (planes > 1) {   // the Dual pass: parameters only
      if (t == 0) GB_MSG_BWD(false, true, true, true);
      else GB_MSG_BWD(false, true, true, false);
    } else if (grad) {
      if (t == 0) GB_MSG_BWD(true, true, true, true);
      else GB_MSG_BWD(true, true, true, false);
    } else {
      if (t == 0) GB_MSG_BWD(true, false, false, true);
      else GB_MSG_BWD(true, true, false, false);
    }
#undef GB_MSG_BWD
    NET_LAUNCHED(net);
    // below the first layer lie only the embedding (a parameter) and h^v = 0
    if (t == 0 && !grad) break;
    const Mix mA{planes * n, S + V, S, net->gA[t], 4 * t + 0, false, net->ghs, true};
    const Mix mB{planes * 3 * n, 2 * V, V, net->gB[t], 4 * t + 1, false, net->ghv, true};
    if ((st = mix(net, s, mA, t > 0 ? &mB : nullptr))) return st;
  }
  if (grad && (st = param_grads<T>(net, s, grad, acc))) return st;
  (void)pl96;
  return PME_OK;
}

int build_neighbours(gbnet_t net, cudaStream_t s, const float* pos) {
  if (net->n == 0) return PME_OK;
  pdl_launch(k_nbr, blocks_for(net->n, kWarps), 32 * kWarps, 0, s, net->frames_d, net->frame_of, pos, net->n,
             net->nbr_cnt, net->nbr_j, net->nbr_sh, net->flags);
  NET_LAUNCHED(net);
  return PME_OK;
}

__global__ void k_gesr_from(int nframes, const double* g, float* out) {
  const int bx = gbpme::pdl_begin_block();
  const int f = bx * blockDim.x + threadIdx.x;
  if (f >= nframes) return;
  out[2 * f] = g ? float(g[f]) : 0.f;
  out[2 * f + 1] = 0.f;
}

__global__ void k_frame_of(const int* __restrict__ offs, int nframes, int* frame_of) {
  const int f = blockIdx.x;
  for (int i = offs[f] + threadIdx.x; i < offs[f + 1]; i += blockDim.x) frame_of[i] = f;
}

bool invert3(const double* a, double* inv) {
  const double det = a[0] * (a[4] * a[8] - a[5] * a[7]) - a[1] * (a[3] * a[8] - a[5] * a[6]) +
                     a[2] * (a[3] * a[7] - a[4] * a[6]);
  if (!std::isfinite(det) || std::fabs(det) < 1e-300) return false;
  const double id = 1.0 / det;
  inv[0] = (a[4] * a[8] - a[5] * a[7]) * id;
  inv[1] = (a[2] * a[7] - a[1] * a[8]) * id;
  inv[2] = (a[1] * a[5] - a[2] * a[4]) * id;
  inv[3] = (a[5] * a[6] - a[3] * a[8]) * id;
  inv[4] = (a[0] * a[8] - a[2] * a[6]) * id;
  inv[5] = (a[2] * a[3] - a[0] * a[5]) * id;
  inv[6] = (a[3] * a[7] - a[4] * a[6]) * id;
  inv[7] = (a[1] * a[6] - a[0] * a[7]) * id;
  inv[8] = (a[0] * a[4] - a[1] * a[3]) * id;
  return true;
}

}  // namespace
}  // namespace gbnet

using namespace gbnet;

extern "C" {

int gbnet_create(gbnet_t* out, int max_ions, int max_frames) {
  if (!out || max_ions < 0 || max_frames < 1 || max_ions > (1 << 24)) return PME_ERR_ARG;
  *out = nullptr;
  gbnet_t net = new (std::nothrow) gbnet_s;
  if (!net) return PME_ERR_NOMEM;
  net->max_ions = max_ions;
  net->max_frames = max_frames;
  cudaGetDevice(&net->dev);
  const size_t N = size_t(std::max(max_ions, 1));
  bool ok = true;
  auto A = [&](auto** p, size_t bytes) {
    void* q = nullptr;
    if (ok && cudaMalloc(&q, std::max<size_t>(bytes, 16)) == cudaSuccess) {
      net->owned.push_back(q);
      *p = static_cast<std::remove_pointer_t<decltype(p)>>(q);
    } else {
      ok = false;
    }
  };
  const size_t f = sizeof(float);
  A(&net->P, f * kParams);
  A(&net->am, f * kParams);
  A(&net->av, f * kParams);
  A(&net->grad, f * kParams);
  A(&net->gscratch, f * kParams);
  int woff = 0;
  for (int w = 0; w < kNumMix; ++w) {
    const MixW m = mix_w(w);
    net->wbf_offs[2 * w] = woff;
    woff += m.K * m.N;
    net->wbf_offs[2 * w + 1] = woff;
    woff += m.K * m.N;
  }
  A(&net->wbf, sizeof(uint16_t) * woff);
  A(&net->wbf_offs_d, sizeof(int) * 2 * kNumMix);
  A(&net->flags, sizeof(int));
  A(&net->frames_d, sizeof(NetFrame) * max_frames);
  A(&net->frame_of, sizeof(int) * N);
  A(&net->species, sizeof(int) * N);
  A(&net->nbr_cnt, sizeof(int) * N);
  A(&net->nbr_j, sizeof(int) * N * kMaxNbr);
  A(&net->nbr_sh, sizeof(float4) * N * kMaxNbr);
  for (int t = 0; t < 3; ++t) {
    A(&net->hs[t], 2 * f * N * S);
    if (t > 0) A(&net->hv[t], 2 * f * N * 3 * V);   // hv[0] = 0 is not stored
  }
  for (int t = 0; t < 2; ++t) {
    A(&net->A[t], 2 * f * N * (S + V));
    A(&net->B[t], 2 * f * N * 3 * 2 * V);
    A(&net->ms[t], 2 * f * N * (S + V));
    A(&net->mv[t], 2 * f * N * 3 * 2 * V);
    A(&net->U[t], 2 * f * N * (S + V));
    A(&net->Y[t], 2 * f * N * 3 * V);
  }
  A(&net->H, 2 * f * N * 2 * S);
  A(&net->qt, 2 * f * N);
  A(&net->ei, 2 * f * N);
  A(&net->q, 2 * f * N);
  A(&net->mu, 2 * f * N * 3);
  A(&net->ghs, 2 * f * N * S);
  A(&net->ghv, 2 * f * N * 3 * V);
  for (int t = 0; t < 2; ++t) {
    A(&net->gA[t], 2 * f * N * (S + V));
    A(&net->gB[t], 2 * f * N * 3 * 2 * V);
    A(&net->gU[t], 2 * f * N * (S + V));
    A(&net->gY[t], 2 * f * N * 3 * V);
  }
  A(&net->gms, 2 * f * N * (S + V));
  A(&net->gmv, 2 * f * N * 3 * 2 * V);
  A(&net->gH, 2 * f * N * 2 * S);
  A(&net->gpos, 2 * f * N * 3);
  A(&net->gq, 2 * f * N);
  A(&net->gmu, 2 * f * N * 3);
  A(&net->gq_mean, 2 * f * max_frames);
  A(&net->gesr, 2 * f * max_frames);
  // partial sums of every parameter gradient of one pass, side by side
  net->part_cap = part_layout(int(N)).total;
  A(&net->part, f * net->part_cap);
  A(&net->e_sr, sizeof(double) * max_frames);
  A(&net->e_pme, sizeof(double) * max_frames);
  A(&net->cvec, sizeof(double) * max_frames);
  A(&net->lpart, sizeof(double) * 2 * max_frames);
  A(&net->q_plain, f * N);
  A(&net->mu_plain, f * N * 3);
  A(&net->f_pme, f * N * 3);
  A(&net->field, f * N * 3);
  A(&net->dpos, f * N * 3);
  A(&net->wneg, f * N * 3);
  A(&net->mut_neg, f * N * 3);
  A(&net->gp_scratch, f * N * 3);
  A(&net->pos_saved, f * N * 3);
  if (!ok) {
    gbnet_destroy(net);
    return PME_ERR_NOMEM;
  }
  if (cudaMemcpy(net->wbf_offs_d, net->wbf_offs, sizeof(int) * 2 * kNumMix, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemset(net->P, 0, f * kParams) != cudaSuccess || cudaMemset(net->flags, 0, sizeof(int)) != cudaSuccess ||
      cudaMemset(net->wbf, 0, sizeof(uint16_t) * woff) != cudaSuccess) {
    gbnet_destroy(net);
    return PME_ERR_CUDA;
  }
  *out = net;
  return PME_OK;
}

int gbnet_destroy(gbnet_t net) {
  if (!net) return PME_ERR_ARG;
  for (void* p : net->owned) cudaFree(p);
  delete net;
  return PME_OK;
}

const char* gbnet_last_error(gbnet_t net) { return net ? net->err.c_str() : "null handle"; }

int gbnet_set_frames(gbnet_t net, void* stream, int nframes, const int* offsets, const double* boxes,
                     const int* species) {
  if (!net || !offsets || !boxes || nframes < 1 || nframes > net->max_frames) return PME_ERR_ARG;
  if (offsets[0] != 0) return fail(net, PME_ERR_ARG, "offsets[0] must be 0");
  for (int f = 0; f < nframes; ++f)
    if (offsets[f + 1] < offsets[f]) return fail(net, PME_ERR_ARG, "offsets must not decrease");
  const int n = offsets[nframes];
  if (n > net->max_ions) return fail(net, PME_ERR_ARG, "more ions than max_ions");
  if (n > 0 && !species) return fail(net, PME_ERR_ARG, "species is NULL");
  std::vector<NetFrame> fr(nframes);
  for (int f = 0; f < nframes; ++f) {
    const double* C = boxes + 9 * f;
    double Ci[9];
    if (!invert3(C, Ci)) return fail(net, PME_ERR_ARG, "singular box");
    const double vol = std::fabs(C[0] * (C[4] * C[8] - C[5] * C[7]) - C[1] * (C[3] * C[8] - C[5] * C[6]) +
                                 C[2] * (C[3] * C[7] - C[4] * C[6]));
    for (int a = 0; a < 3; ++a) {
      const double* u = C + 3 * ((a + 1) % 3);
      const double* v = C + 3 * ((a + 2) % 3);
      const double cx = u[1] * v[2] - u[2] * v[1], cy = u[2] * v[0] - u[0] * v[2], cz = u[0] * v[1] - u[1] * v[0];
      const double width = vol / std::sqrt(cx * cx + cy * cy + cz * cz);
      if (width < 2.0 * GBNET_CUTOFF) return fail(net, PME_ERR_ARG, "box narrower than twice the cutoff");
    }
    fr[f].off = offsets[f];
    fr[f].n = offsets[f + 1] - offsets[f];
    for (int k = 0; k < 9; ++k) {
      fr[f].C[k] = float(C[k]);
      fr[f].Ci[k] = float(Ci[k]);
    }
    fr[f].ortho = (C[1] == 0 && C[2] == 0 && C[3] == 0 && C[5] == 0 && C[6] == 0 && C[7] == 0) ? 1 : 0;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  net->offsets_h.assign(offsets, offsets + nframes + 1);
  net->n = n;
  net->nframes = nframes;
  int st;
  if ((st = cuda_ok(net, cudaMemcpyAsync(net->frames_d, fr.data(), sizeof(NetFrame) * nframes,
                                         cudaMemcpyHostToDevice, s), "copy frames")))
    return st;
  // frame_of from the offsets (staged through the tail of the loss scratch)
  int* offs_d = reinterpret_cast<int*>(net->lpart);
  if (size_t(nframes + 1) * sizeof(int) > sizeof(double) * 2 * size_t(net->max_frames))
    return fail(net, PME_ERR_ARG, "too many frames");
  if ((st = cuda_ok(net, cudaMemcpyAsync(offs_d, offsets, sizeof(int) * (nframes + 1), cudaMemcpyHostToDevice, s),
                    "copy offsets")))
    return st;
  k_frame_of<<<nframes, 256, 0, s>>>(offs_d, nframes, net->frame_of);
  NET_LAUNCHED(net);
  if (n > 0 &&
      (st = cuda_ok(net, cudaMemcpyAsync(net->species, species, sizeof(int) * n, cudaMemcpyDeviceToDevice, s),
                    "copy species")))
    return st;
  // the offsets copy above must finish before the host array can go away
  return cuda_ok(net, cudaStreamSynchronize(s), "set frames");
}

int gbnet_set_params(gbnet_t net, void* stream, const float* params) {
  if (!net || !params) return PME_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int st;
  if ((st = cuda_ok(net, cudaMemcpyAsync(net->P, params, sizeof(float) * kParams, cudaMemcpyDeviceToDevice, s),
                    "copy params")))
    return st;
  if ((st = cuda_ok(net, cudaMemsetAsync(net->am, 0, sizeof(float) * kParams, s), "memset")) ||
      (st = cuda_ok(net, cudaMemsetAsync(net->av, 0, sizeof(float) * kParams, s), "memset")))
    return st;
  net->adam_step = 0;
  pdl_launch(k_cast_weights, dim3(8, kNumMix), 256, 0, s, net->P, net->wbf, net->wbf_offs_d);
  NET_LAUNCHED(net);
  return PME_OK;
}

int gbnet_get_params(gbnet_t net, void* stream, float* params) {
  if (!net || !params) return PME_ERR_ARG;
  return cuda_ok(net, cudaMemcpyAsync(params, net->P, sizeof(float) * kParams, cudaMemcpyDeviceToDevice,
                                      static_cast<cudaStream_t>(stream)),
                 "copy params");
}

int gbnet_forward(gbnet_t net, void* stream, const float* pos, float* q, float* mu, double* e_sr) {
  if (!net || (net->n > 0 && !pos)) return PME_ERR_ARG;
  if (net->nframes == 0) return fail(net, PME_ERR_ARG, "no frames set");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t n = size_t(net->n);
  int st;
  // the positions are kept for gbnet_backward (the edge geometry is recomputed there)
  if (n && (st = cuda_ok(net, cudaMemcpyAsync(net->pos_saved, pos, sizeof(float) * 3 * n, cudaMemcpyDeviceToDevice, s),
                         "copy positions")))
    return st;
  if ((st = build_neighbours(net, s, net->pos_saved))) return st;
  if ((st = forward_pass<float>(net, s, net->pos_saved, nullptr))) return st;
  if (q && n && (st = cuda_ok(net, cudaMemcpyAsync(q, net->q, sizeof(float) * n, cudaMemcpyDeviceToDevice, s), "copy")))
    return st;
  if (mu && n &&
      (st = cuda_ok(net, cudaMemcpyAsync(mu, net->mu, sizeof(float) * 3 * n, cudaMemcpyDeviceToDevice, s), "copy")))
    return st;
  if (e_sr &&
      (st = cuda_ok(net, cudaMemcpyAsync(e_sr, net->e_sr, sizeof(double) * net->nframes, cudaMemcpyDeviceToDevice, s),
                    "copy")))
    return st;
  return PME_OK;
}

int gbnet_backward(gbnet_t net, void* stream, const float* g_q, const float* g_mu, const double* g_esr,
                   float* g_pos, float* g_params) {
  if (!net) return PME_ERR_ARG;
  if (net->nframes == 0) return fail(net, PME_ERR_ARG, "no frames set");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  pdl_launch(k_gesr_from, blocks_for(net->nframes, 128), 128, 0, s, net->nframes, g_esr, net->gesr);
  NET_LAUNCHED(net);
  int st;
  if ((st = backward_pass<float>(net, s, net->pos_saved, nullptr, g_q, g_mu, net->gesr, g_params, false)))
    return st;
  if (g_pos && net->n &&
      (st = cuda_ok(net, cudaMemcpyAsync(g_pos, net->gpos, sizeof(float) * 3 * size_t(net->n),
                                         cudaMemcpyDeviceToDevice, s), "copy")))
    return st;
  return PME_OK;
}

static int loss_grad(gbnet_t net, pme_plan_t pme, cudaStream_t s, const float* pos, const double* e_ref,
                     const float* f_ref, double lambda_e, double lambda_f, double* loss, float* force, float* grad,
                     bool acc) {
  const int n = net->n, F = net->nframes;
  const size_t nn = size_t(n);
  int st;
  if (pme_batch_frames(pme) != F) return fail(net, PME_ERR_ARG, "the PME plan's frames differ from the network's");
  net->launches = 0;
  if (n && (st = cuda_ok(net, cudaMemcpyAsync(net->pos_saved, pos, sizeof(float) * 3 * nn, cudaMemcpyDeviceToDevice, s),
                         "copy positions")))
    return st;
  // 1. plain forward of the network and of the PME on its charges and dipoles
  if ((st = build_neighbours(net, s, net->pos_saved))) return st;
  if ((st = forward_pass<float>(net, s, net->pos_saved, nullptr))) return st;
  if (n && ((st = cuda_ok(net, cudaMemcpyAsync(net->q_plain, net->q, sizeof(float) * nn, cudaMemcpyDeviceToDevice, s),
                          "copy")) ||
            (st = cuda_ok(net, cudaMemcpyAsync(net->mu_plain, net->mu, sizeof(float) * 3 * nn,
                                               cudaMemcpyDeviceToDevice, s), "copy"))))
    return st;
  // phi goes straight into the value plane of the charge cotangent
  if ((st = pme_batch_forward(pme, s, net->pos_saved, net->q_plain, net->mu_plain, net->e_pme, net->f_pme, net->gq,
                              net->field, nullptr)))
    return fail(net, st, std::string("pme_batch_forward: ") + pme_last_error(pme));
  // 2. plain backward of the network with seeds (phi, dE/dmu = -field, 1): the net's part of dE/dr
  if (n) {
    pdl_launch(k_scale, blocks_for(3 * nn, 256), 256, 0, s, 3 * nn, net->field, -1.f, net->gmu);
    NET_LAUNCHED(net);
  }
  pdl_launch(k_seed_esr, blocks_for(F, 128), 128, 0, s, F, net->cvec, net->gesr, 0);
  NET_LAUNCHED(net);
  if ((st = backward_pass<float>(net, s, net->pos_saved, nullptr, net->gq, net->gmu, net->gesr, nullptr, false)))
    return st;
  // 3. loss, energy cotangents c_b, position tangent r' = -w
  pdl_launch(k_loss, F, 256, 0, s, net->frames_d, F, n, net->e_pme, net->e_sr, e_ref, net->f_pme, net->gpos, f_ref,
             lambda_e, lambda_f, net->cvec, force, net->dpos, net->wneg, net->lpart);
  NET_LAUNCHED(net);
  pdl_launch(k_loss_total, 1, 256, 0, s, net->lpart, F, loss);
  NET_LAUNCHED(net);
  // 4. forward of the network carrying the tangent r'
  if ((st = forward_pass<Dual>(net, s, net->pos_saved, net->dpos))) return st;
  // 5. PME Hessian-vector product along (r', q', mu') plus c_b times the gradient: the tangents
  //    of (dE/dq, dE/dmu) land in the tangent planes of the cotangents
  if (n) {
    pdl_launch(k_scale, blocks_for(3 * nn, 256), 256, 0, s, 3 * nn, net->mu + 3 * nn, -1.f, net->mut_neg);
    NET_LAUNCHED(net);
  }
  if ((st = pme_batch_backward(pme, s, net->pos_saved, net->q_plain, net->mu_plain, net->cvec, net->wneg, net->q + nn,
                               net->mut_neg, net->gp_scratch, net->gq + nn, net->gmu + 3 * nn)))
    return fail(net, st, std::string("pme_batch_backward: ") + pme_last_error(pme));
  // 6. Dual backward of the network with energy seeds 1 + e c_b: its tangent plane is dL/dtheta
  pdl_launch(k_seed_esr, blocks_for(F, 128), 128, 0, s, F, net->cvec, net->gesr, 1);
  NET_LAUNCHED(net);
  if ((st = backward_pass<Dual>(net, s, net->pos_saved, net->dpos, net->gq, net->gmu, net->gesr, grad, acc)))
    return st;
  return PME_OK;
}

int gbnet_loss_grad(gbnet_t net, pme_plan_t pme, void* stream, const float* pos, const double* e_ref,
                    const float* f_ref, double lambda_e, double lambda_f, double* loss, float* force, float* grad,
                    int accumulate) {
  if (!net || !pme || !e_ref || !loss || !grad || (net->n > 0 && (!pos || !f_ref))) return PME_ERR_ARG;
  if (net->nframes == 0) return fail(net, PME_ERR_ARG, "no frames set");
  return loss_grad(net, pme, static_cast<cudaStream_t>(stream), pos, e_ref, f_ref, lambda_e, lambda_f, loss, force,
                   grad, accumulate != 0);
}

int gbnet_adam(gbnet_t net, void* stream, const float* grad, double lr, double beta1, double beta2, double eps) {
  if (!net || !grad) return PME_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  ++net->adam_step;
  const double c1 = 1.0 / (1.0 - std::pow(beta1, net->adam_step));
  const double c2 = 1.0 / (1.0 - std::pow(beta2, net->adam_step));
  pdl_launch(k_adam, blocks_for(kParams, 256), 256, 0, s, kParams,
             net->P, net->am, net->av, grad, float(lr), float(beta1), float(beta2), float(eps), float(c1), float(c2));
  NET_LAUNCHED(net);
  pdl_launch(k_cast_weights, dim3(8, kNumMix), 256, 0, s, net->P, net->wbf, net->wbf_offs_d);
  NET_LAUNCHED(net);
  return PME_OK;
}

int gbnet_train_step(gbnet_t net, pme_plan_t pme, void* stream, const float* pos, const double* e_ref,
                     const float* f_ref, double lambda_e, double lambda_f, double lr, double* loss) {
  if (!net || !pme || !e_ref || !loss || (net->n > 0 && (!pos || !f_ref))) return PME_ERR_ARG;
  if (net->nframes == 0) return fail(net, PME_ERR_ARG, "no frames set");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int st = loss_grad(net, pme, s, pos, e_ref, f_ref, lambda_e, lambda_f, loss, nullptr, net->grad, false);
  if (st) return st;
  const long long l = net->launches;
  st = gbnet_adam(net, stream, net->grad, lr, 0.9, 0.999, 1e-8);
  net->launches += l;
  return st;
}

int gbnet_mix(void* stream, int M, int k, int nout, const float* X, const unsigned short* wt, float* Y,
              int accumulate, int* err) {
  if (M < 0 || (M > 0 && (!X || !wt || !Y))) return PME_ERR_ARG;
  if ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) & 15) return PME_ERR_ARG;
  static int* dummy = nullptr;
  if (!err) {
    if (!dummy && cudaMalloc(&dummy, sizeof(int)) != cudaSuccess) return PME_ERR_NOMEM;
    err = dummy;
  }
  return launch_mix(static_cast<cudaStream_t>(stream), k, nout, MixJob{X, wt, Y, M, accumulate != 0}, err);
}

int gbnet_sync_status(gbnet_t net, void* stream) {
  if (!net) return PME_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int flags = 0;
  int st;
  if ((st = cuda_ok(net, cudaStreamSynchronize(s), "synchronise"))) return st;
  if ((st = cuda_ok(net, cudaMemcpy(&flags, net->flags, sizeof(int), cudaMemcpyDeviceToHost), "read flags"))) return st;
  if ((st = cuda_ok(net, cudaMemset(net->flags, 0, sizeof(int)), "clear flags"))) return st;
  if (flags & kNetFlagTimeout) return fail(net, PME_ERR_TIMEOUT, "a tensor-core wait gave up");
  if (flags & kNetFlagNbrFull) return fail(net, PME_ERR_ARG, "an ion had more than GBNET_MAX_NEIGHBOURS neighbours");
  if (flags & kNetFlagNonFinite) return fail(net, PME_ERR_NONFINITE, "non-finite position");
  return PME_OK;
}

long long gbnet_last_launches(gbnet_t net) { return net ? net->launches : -1; }

}  // extern "C"
