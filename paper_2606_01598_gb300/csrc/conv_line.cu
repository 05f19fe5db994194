// Mesh convolution for meshes of 64, 128 or 256 points per axis whose planes do not fit in shared
// memory (256 x 256 above all): the z and y transforms, which conv.cu and conv_two.cu do together
// on one x-plane, as separate passes over lines, the x pass as in conv_two.cu:
//   k_line_r2c  blocks of row pairs: each pair of real rows is one complex row, transformed
//               along z, separated into the two half spectra and stored;
//   k_line_y    blocks of columns of one plane, transformed along y in place (both directions);
//   k_line_c2r  the reverse of k_line_r2c.
// Every 1D transform is two register steps with one exchange (see conv_two.cu), lengths and
// strides compile-time.
//
// Bound: memory. Five passes read and write a mesh or a spectrum each (134 MB at 256^3, against
// 129 MB of L2). cuFFT with the influence pass takes seven, and in a backward on the forward's
// inputs transforms rho again, which these passes skip. Forward + backward of 262144 ions on
// 256^3: 1.97 -> 1.82 ms.
#include "conv_dft.cuh"

namespace gbpme {

namespace {

template <int L>
struct Split {
  static constexpr int P = L == 64 ? 8 : 16, Q = L / P;
};

// DFT of step 1 and its twiddles w_L^(t k)
template <int P, bool INV>
__device__ __forceinline__ void line_step1(float2 (&v)[P], int t, const float2* __restrict__ tw) {
  dft<P, INV>(v);
#pragma unroll
  for (int k = 1; k < P; ++k) {
    float2 w = __ldg(tw + t * k);
    if (INV) w.y = -w.y;
    v[k] = cmul(v[k], w);
  }
}

constexpr int kLineThreads = 256;
template <int NZ>
__host__ __device__ constexpr int line_pairs() { return kLineThreads / Split<NZ>::P; }   // row pairs per block
template <int NZ>
__host__ __device__ constexpr int line_row_stride() { return Split<NZ>::P * (Split<NZ>::Q | 1) + 1; }   // odd
template <int NZ>
constexpr int line_row_smem() { return line_pairs<NZ>() * line_row_stride<NZ>() * int(sizeof(float2)); }

// mesh copy of this block: 0 rho / Phi, 1 the tangent one; false: nothing to do (the forward's
// rho spectrum and Phi stay)
__device__ __forceinline__ bool line_copy(const ConvArgs& a, int blocks_per_copy, int& copy, int& blk) {
  copy = int(blockIdx.x) >= blocks_per_copy ? 1 : 0;
  blk = int(blockIdx.x) - copy * blocks_per_copy;
  return !(copy == 0 && a.keep && *a.keep == 0);
}

template <int NZ>
__global__ void __launch_bounds__(kLineThreads) k_line_r2c(ConvArgs a, int blocks_per_copy) {
  pdl_begin();
  constexpr int P = Split<NZ>::P, Q = Split<NZ>::Q, QO = Q | 1, RP = line_pairs<NZ>(), NZH = NZ / 2 + 1;
  constexpr int RS = line_row_stride<NZ>();
  static_assert(RS >= NZ, "the natural-order row fits in the exchange row");
  extern __shared__ __align__(16) float2 csm[];
  int copy, blk;
  if (!line_copy(a, blocks_per_copy, copy, blk)) return;
  const FrameDesc& F = a.one;
  const float* src = a.mesh + (copy ? F.tmesh_off : F.mesh_off) + size_t(blk) * RP * 2 * NZ;
  float2* dst = a.spec + (copy ? F.tspec_off : F.spec_off) + size_t(blk) * RP * 2 * NZH;
  const float2* tz = a.tw + F.tw_off[2];
  const int tid = threadIdx.x;
  if (tid < RP * Q) {
    const int pr = tid / Q, t = tid % Q;
    const float* r0 = src + pr * 2 * NZ + t;
    float2 v[P];
#pragma unroll
    for (int m = 0; m < P; ++m) v[m] = make_float2(r0[Q * m], r0[NZ + Q * m]);
    line_step1<P, false>(v, t, tz);
#pragma unroll
    for (int k = 0; k < P; ++k) csm[pr * RS + k * QO + t] = v[k];
  }
  __syncthreads();
  const int pr = tid / P, k1 = tid % P;
  float2 u[Q];
#pragma unroll
  for (int t = 0; t < Q; ++t) u[t] = csm[pr * RS + k1 * QO + t];
  dft<Q, false>(u);
  __syncthreads();
#pragma unroll
  for (int k2 = 0; k2 < Q; ++k2) csm[pr * RS + k1 + P * k2] = u[k2];
  __syncthreads();
  // row 2 pr is (Z_k + conj Z_{N-k}) / 2, row 2 pr + 1 is (Z_k - conj Z_{N-k}) / 2i
  for (int it = tid; it < RP * NZH; it += kLineThreads) {
    const int p = it / NZH, k = it - p * NZH;
    const float2 zk = csm[p * RS + k], zm = csm[p * RS + ((NZ - k) & (NZ - 1))];
    float2* d = dst + p * 2 * NZH + k;
    d[0] = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
    d[NZH] = make_float2(0.5f * (zk.y + zm.y), 0.5f * (zm.x - zk.x));
  }
}

template <int NZ>
__global__ void __launch_bounds__(kLineThreads) k_line_c2r(ConvArgs a, int blocks_per_copy) {
  pdl_begin();
  constexpr int P = Split<NZ>::P, Q = Split<NZ>::Q, QO = Q | 1, RP = line_pairs<NZ>(), NZH = NZ / 2 + 1;
  constexpr int RS = line_row_stride<NZ>();
  extern __shared__ __align__(16) float2 csm[];
  int copy, blk;
  if (!line_copy(a, blocks_per_copy, copy, blk)) return;
  const FrameDesc& F = a.one;
  const float2* src = a.spec + (copy ? F.tspec_off : F.spec_off) + size_t(blk) * RP * 2 * NZH;
  float* dst = a.mesh + (copy ? F.tmesh_off : F.mesh_off) + size_t(blk) * RP * 2 * NZ;
  const float2* tz = a.tw + F.tw_off[2];
  const int tid = threadIdx.x;
  if (tid < RP * Q) {
    // complex row = (half row 2 pr) + i (half row 2 pr + 1), extended by Hermitian symmetry (the
    // n_z = 0 and Nyquist entries of a real row's spectrum are real)
    const int pr = tid / Q, t = tid % Q;
    const float2* ra = src + pr * 2 * NZH;
    float2 v[P];
#pragma unroll
    for (int m = 0; m < P; ++m) {
      const int k = t + Q * m;
      const bool up = k < NZH;
      const int kk = up ? k : NZ - k;
      float2 A = ra[kk], B = ra[NZH + kk];
      if (!up) {
        A.y = -A.y;
        B.y = -B.y;
      } else if (k == 0 || 2 * k == NZ) {
        A.y = 0.f;
        B.y = 0.f;
      }
      v[m] = make_float2(A.x - B.y, A.y + B.x);
    }
    line_step1<P, true>(v, t, tz);
#pragma unroll
    for (int k = 0; k < P; ++k) csm[pr * RS + k * QO + t] = v[k];
  }
  __syncthreads();
  const int pr = tid / P, k1 = tid % P;
  float2 u[Q];
#pragma unroll
  for (int t = 0; t < Q; ++t) u[t] = csm[pr * RS + k1 * QO + t];
  dft<Q, true>(u);
  float* r0 = dst + pr * 2 * NZ + k1;
#pragma unroll
  for (int k2 = 0; k2 < Q; ++k2) {
    r0[P * k2] = u[k2].x;
    r0[NZ + P * k2] = u[k2].y;
  }
}

// Columns of a k_line_y tile: 22 divides 65 and 129 columns with little left over, and its
// NY / 16 x 22 first-step items fill eleven warps at 256 points.
constexpr int kLineCols = 22;
constexpr int kLineYThreads = 352;

template <int NY, bool INV>
__global__ void __launch_bounds__(kLineYThreads, 3) k_line_y(ConvArgs a, int blocks_per_copy, int tiles) {
  pdl_begin();
  constexpr int P = Split<NY>::P, Q = Split<NY>::Q;
  extern __shared__ __align__(16) float2 csm[];
  int copy, blk;
  if (!line_copy(a, blocks_per_copy, copy, blk)) return;
  const FrameDesc& F = a.one;
  const int Nzh = F.g.N[2] / 2 + 1;
  const int x = blk / tiles, tile = blk - x * tiles;
  const int c0 = tile * kLineCols, nc = min(kLineCols, Nzh - c0);
  float2* base = a.spec + (copy ? F.tspec_off : F.spec_off) + size_t(x) * NY * Nzh + c0;
  const float2* ty = a.tw + F.tw_off[1];
  for (int it = threadIdx.x; it < Q * kLineCols; it += kLineYThreads) {
    const int t = it / kLineCols, c = it - t * kLineCols;
    if (c >= nc) continue;
    const float2* s = base + t * Nzh + c;
    float2 v[P];
#pragma unroll
    for (int m = 0; m < P; ++m) v[m] = s[Q * m * Nzh];
    line_step1<P, INV>(v, t, ty);
#pragma unroll
    for (int k = 0; k < P; ++k) csm[(t + Q * k) * kLineCols + c] = v[k];
  }
  __syncthreads();
  for (int it = threadIdx.x; it < P * kLineCols; it += kLineYThreads) {
    const int k1 = it / kLineCols, c = it - k1 * kLineCols;
    if (c >= nc) continue;
    float2 u[Q];
#pragma unroll
    for (int t = 0; t < Q; ++t) u[t] = csm[(t + Q * k1) * kLineCols + c];
    dft<Q, INV>(u);
    float2* d = base + k1 * Nzh + c;
#pragma unroll
    for (int k2 = 0; k2 < Q; ++k2) d[P * k2 * Nzh] = u[k2];
  }
}

template <int NZ>
int launch_rows(pme_plan_t p, cudaStream_t s, const ConvArgs& a, int copies, bool inverse) {
  const int* N = p->frames_h[0].g.N;
  const int blocks = N[0] * N[1] / 2 / line_pairs<NZ>();
  int st;
  if (inverse) {
    static unsigned done = 0;
    if ((st = set_smem(p, k_line_c2r<NZ>, done))) return st;
    pdl_launch(k_line_c2r<NZ>, copies * blocks, kLineThreads, line_row_smem<NZ>(), s, a, blocks);
  } else {
    static unsigned done = 0;
    if ((st = set_smem(p, k_line_r2c<NZ>, done))) return st;
    pdl_launch(k_line_r2c<NZ>, copies * blocks, kLineThreads, line_row_smem<NZ>(), s, a, blocks);
  }
  count_launch();
  return check_launch(p, "k_line_z");
}

template <int NY>
int launch_columns(pme_plan_t p, cudaStream_t s, const ConvArgs& a, int copies, bool inverse) {
  const int* N = p->frames_h[0].g.N;
  const int tiles = (N[2] / 2 + 1 + kLineCols - 1) / kLineCols, blocks = N[0] * tiles;
  const size_t smem = size_t(NY) * kLineCols * sizeof(float2);
  int st;
  if (inverse) {
    static unsigned done = 0;
    if ((st = set_smem(p, k_line_y<NY, true>, done))) return st;
    pdl_launch(k_line_y<NY, true>, copies * blocks, kLineYThreads, smem, s, a, blocks, tiles);
  } else {
    static unsigned done = 0;
    if ((st = set_smem(p, k_line_y<NY, false>, done))) return st;
    pdl_launch(k_line_y<NY, false>, copies * blocks, kLineYThreads, smem, s, a, blocks, tiles);
  }
  count_launch();
  return check_launch(p, "k_line_y");
}

}  // namespace

bool line_axes_ok(const int N[3]) {
  for (int a = 0; a < 3; ++a)
    if (N[a] != 64 && N[a] != 128 && N[a] != 256) return false;
  return true;
}

// The z and y transforms of rho (and, tangent, of d rho): forward z then y, inverse y then z.
int launch_line(pme_plan_t p, cudaStream_t s, const ConvArgs& a, bool inverse) {
  const int* N = p->frames_h[0].g.N;
  const int copies = a.tangent ? 2 : 1;
  int st = PME_OK;
  for (int half = 0; half < 2 && !st; ++half) {
    if ((half == 0) != inverse) {
      if (N[2] == 256) st = launch_rows<256>(p, s, a, copies, inverse);
      else if (N[2] == 128) st = launch_rows<128>(p, s, a, copies, inverse);
      else st = launch_rows<64>(p, s, a, copies, inverse);
    } else {
      if (N[1] == 256) st = launch_columns<256>(p, s, a, copies, inverse);
      else if (N[1] == 128) st = launch_columns<128>(p, s, a, copies, inverse);
      else st = launch_columns<64>(p, s, a, copies, inverse);
    }
  }
  return st;
}

}  // namespace gbpme
