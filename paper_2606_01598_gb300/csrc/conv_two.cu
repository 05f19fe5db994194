// Mesh convolution for 2,3,5-smooth meshes (Sections 2.3.3-2.3.4, Eqs. potential_k,
// energy_recip): the three passes of conv.cu (same layouts, same energy and virial partials)
// with every 1D transform of length L = P Q in two register steps and one shared-memory
// exchange (the four-step split of Bailey, J. Supercomputing 4, 1990):
//   step 1, for each t < Q: the P-point DFT over m of x[t + Q m], times w_L^(t k);
//   step 2, for each k1 < P: the Q-point DFT over t, which is X[k1 + P k2].
// P and Q are at most 16 (two_step_factors), chosen per axis when the plan is made; a step
// switches on its radix once per block, so one launch serves frames of any mix of shapes.
// Global loads feed the first step of a pass and its last step stores to global memory; the
// real-pair separation rides in the y loads of the R2C and the Hermitian extension in the z
// loads of the C2R. The x pass keeps the influence multiply and both DFTs around it in
// registers: the thread that forms X[k1 + P k2] for one k1 holds exactly the inputs of one
// Q-point DFT of the inverse transform split as Q P, so the tile crosses shared memory twice,
// in place, with two barriers.
//
// Bound: instruction issue and the barriers between steps; the data stay in L2 between the
// passes. Against the Stockham kernels (four to six shared-memory stages per axis): the uneven
// batch of 256 frames, forward + backward, 1.43 -> 1.27 ms; single frames leave cuFFT (sizes at
// conv_wanted): forward of 512 ions on 32^3 0.123 -> 0.102 ms, of 9999 ions on 80x81x90 with the
// virial 0.132 -> 0.114 ms, forward + backward of 1999 ions on 48x50x54 0.245 -> 0.219 ms.
#include <type_traits>

#include "conv_dft.cuh"

namespace gbpme {

namespace {

constexpr int kTwoMaxThreads = 512;   // pass A / C
constexpr int kTwoXThreads = 256;     // pass B

// MAXR: 10 where no factor of the plan's axes exceeds 10 (kSmallRadix; every axis up to 64
// points and some up to 100), else 16. Without the 12- to 16-point DFTs the kernels hold 64
// registers (76 to 80 with them, or spills), a third more warps per SM, and less code: forward +
// backward of the uneven batch of 256 frames 1203 -> 1113 us (1148 with the large ones held to 64
// registers), forward of 512 ions on 32^3 53.7 -> 51.7 us.
constexpr int kSmallRadix = 10;
template <int MAXR, class F>
__device__ __forceinline__ void with_radix(int r, F&& f) {
  if constexpr (MAXR <= kSmallRadix) {
    switch (r) {
      case 1: f(std::integral_constant<int, 1>{}); break;
      case 2: f(std::integral_constant<int, 2>{}); break;
      case 3: f(std::integral_constant<int, 3>{}); break;
      case 4: f(std::integral_constant<int, 4>{}); break;
      case 5: f(std::integral_constant<int, 5>{}); break;
      case 6: f(std::integral_constant<int, 6>{}); break;
      case 8: f(std::integral_constant<int, 8>{}); break;
      case 9: f(std::integral_constant<int, 9>{}); break;
      default: f(std::integral_constant<int, 10>{}); break;
    }
    return;
  }
  switch (r) {
    case 1: f(std::integral_constant<int, 1>{}); break;
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 5: f(std::integral_constant<int, 5>{}); break;
    case 6: f(std::integral_constant<int, 6>{}); break;
    case 8: f(std::integral_constant<int, 8>{}); break;
    case 9: f(std::integral_constant<int, 9>{}); break;
    case 10: f(std::integral_constant<int, 10>{}); break;
    case 12: f(std::integral_constant<int, 12>{}); break;
    case 15: f(std::integral_constant<int, 15>{}); break;
    default: f(std::integral_constant<int, 16>{}); break;
  }
}

// DFT of step 1 and its twiddles w_L^(t k) (tw: the forward table of length L)
template <int P, bool INV>
__device__ __forceinline__ void step1(float2 (&v)[P], int t, const float2* __restrict__ tw) {
  dft<P, INV>(v);
#pragma unroll
  for (int k = 1; k < P; ++k) {
    float2 w = __ldg(tw + t * k);
    if (INV) w.y = -w.y;
    v[k] = cmul(v[k], w);
  }
}

// The block's planes: shapes, factors and the two shared-memory buffers.
//   Z  complex rows after z step 1: slot (k1, t) of row pr at (pr P + k1) (Q | 1) + t
//   Z2 complex rows in natural order, row stride Nz | 1 (pass A)
//   S  half spectra, entry (y, kz) of plane pl at y Sw + pl Nzh + kz; pass C's second copy
// Z and S share the first buffer (one is dead when the other is written), Z2 and pass C's S2
// the second.
struct TwoPlane {
  int Ny, Nz, Nzh, np, rows, Sw, Pz, Qz, Py, Qy, Qo, Zs;
  float rQz, rPz, rnp, rSw, rnzh;
  float2 *b0, *b1;
};

__device__ __forceinline__ TwoPlane two_plane(const FrameDesc& F, int pc, float2* sm) {
  TwoPlane T;
  T.Ny = F.g.N[1];
  T.Nz = F.g.N[2];
  T.Nzh = T.Nz / 2 + 1;
  T.np = (T.Ny + 1) >> 1;
  T.rows = pc * T.np;
  T.Sw = pc * T.Nzh;
  T.Py = F.conv_p[1];
  T.Qy = F.conv_q[1];
  T.Pz = F.conv_p[2];
  T.Qz = F.conv_q[2];
  T.Qo = T.Qz | 1;
  T.Zs = T.Nz | 1;
  T.rQz = 1.f / float(T.Qz);
  T.rPz = 1.f / float(T.Pz);
  T.rnp = 1.f / float(T.np);
  T.rSw = 1.f / float(T.Sw);
  T.rnzh = 1.f / float(T.Nzh);
  T.b0 = sm;
  T.b1 = sm + max(T.rows * T.Pz * T.Qo, T.Ny * T.Sw);
  return T;
}

template <bool BATCH, int MAXR>
__global__ void __launch_bounds__(kTwoMaxThreads, MAXR <= kSmallRadix ? 2 : 0) k_two_r2c(ConvArgs a) {
  pdl_begin();
  extern __shared__ __align__(16) float2 csm[];
  int copy, x0, pc;
  const FrameDesc& F = plane_block<BATCH>(a, copy, x0, pc);
  if (copy == 0 && a.keep && *a.keep == 0) return;   // rho's spectrum is not needed again
  const TwoPlane T = two_plane(F, pc, csm);
  const float* src = a.mesh + (copy ? F.tmesh_off : F.mesh_off) + size_t(x0) * T.Ny * T.Nz;
  float2* dst = a.spec + (copy ? F.tspec_off : F.spec_off) + size_t(x0) * T.Ny * T.Nzh;
  const float2* tz = a.tw + F.tw_off[2];
  const float2* ty = a.tw + F.tw_off[1];
  float2* Z = T.b0;
  float2* Z2 = T.b1;
  float2* S = T.b0;
  const int tid = threadIdx.x, NT = blockDim.x;
  // z step 1: complex row pr = real rows 2 pp (real part) and 2 pp + 1 (imaginary part)
  with_radix<MAXR>(T.Pz, [&](auto rc) {
    constexpr int P = decltype(rc)::value;
    for (int it = tid; it < T.rows * T.Qz; it += NT) {
      int pr, t, pl = 0, pp;
      split_rc(it, T.Qz, T.rQz, pr, t);
      if (pc > 1) split_rc(pr, T.np, T.rnp, pl, pp);
      else pp = pr;
      const float* r0 = src + (pl * T.Ny + 2 * pp) * T.Nz + t;
      const float* r1 = 2 * pp + 1 < T.Ny ? r0 + T.Nz : nullptr;   // an odd last row has no partner
      float2 v[P];
#pragma unroll
      for (int m = 0; m < P; ++m) v[m] = make_float2(r0[T.Qz * m], r1 ? r1[T.Qz * m] : 0.f);
      step1<P, false>(v, t, tz);
#pragma unroll
      for (int k = 0; k < P; ++k) Z[(pr * P + k) * T.Qo + t] = v[k];
    }
  });
  __syncthreads();
  with_radix<MAXR>(T.Qz, [&](auto rc) {
    constexpr int Q = decltype(rc)::value;
    for (int it = tid; it < T.rows * T.Pz; it += NT) {
      int pr, k1;
      split_rc(it, T.Pz, T.rPz, pr, k1);
      float2 u[Q];
#pragma unroll
      for (int t = 0; t < Q; ++t) u[t] = Z[it * (Q | 1) + t];
      dft<Q, false>(u);
#pragma unroll
      for (int k2 = 0; k2 < Q; ++k2) Z2[pr * T.Zs + k1 + T.Pz * k2] = u[k2];
    }
  });
  __syncthreads();
  // y step 1 on the real rows' half spectra: row 2 pp is (Z_k + conj Z_{N-k}) / 2, row 2 pp + 1
  // is (Z_k - conj Z_{N-k}) / 2i, with Z the spectrum of complex row pp
  with_radix<MAXR>(T.Py, [&](auto rc) {
    constexpr int P = decltype(rc)::value;
    for (int it = tid; it < T.Qy * T.Sw; it += NT) {
      int t, col, pl = 0, kz;
      split_rc(it, T.Sw, T.rSw, t, col);
      if (pc > 1) split_rc(col, T.Nzh, T.rnzh, pl, kz);
      else kz = col;
      const float2* zr = Z2 + pl * T.np * T.Zs;
      const int km = kz == 0 ? 0 : T.Nz - kz;
      float2 v[P];
#pragma unroll
      for (int m = 0; m < P; ++m) {
        const int y = t + T.Qy * m;
        const float2 zk = zr[(y >> 1) * T.Zs + kz], zm = zr[(y >> 1) * T.Zs + km];
        v[m] = (y & 1) ? make_float2(0.5f * (zk.y + zm.y), 0.5f * (zm.x - zk.x))
                       : make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
      }
      step1<P, false>(v, t, ty);
#pragma unroll
      for (int k = 0; k < P; ++k) S[(t + T.Qy * k) * T.Sw + col] = v[k];
    }
  });
  __syncthreads();
  // y step 2, straight to the planes' [ky][kz] blocks of the spectrum
  with_radix<MAXR>(T.Qy, [&](auto rc) {
    constexpr int Q = decltype(rc)::value;
    for (int it = tid; it < T.Py * T.Sw; it += NT) {
      int k1, col, pl = 0, kz;
      split_rc(it, T.Sw, T.rSw, k1, col);
      if (pc > 1) split_rc(col, T.Nzh, T.rnzh, pl, kz);
      else kz = col;
      float2 u[Q];
#pragma unroll
      for (int t = 0; t < Q; ++t) u[t] = S[(t + Q * k1) * T.Sw + col];
      dft<Q, false>(u);
      float2* d = dst + (pl * T.Ny + k1) * T.Nzh + kz;
#pragma unroll
      for (int k2 = 0; k2 < Q; ++k2) d[T.Py * k2 * T.Nzh] = u[k2];
    }
  });
}

template <bool BATCH, int MAXR>
__global__ void __launch_bounds__(kTwoMaxThreads, MAXR <= kSmallRadix ? 2 : 0) k_two_c2r(ConvArgs a) {
  pdl_begin();
  extern __shared__ __align__(16) float2 csm[];
  int copy, x0, pc;
  const FrameDesc& F = plane_block<BATCH>(a, copy, x0, pc);
  if (copy == 0 && a.keep && *a.keep == 0) return;   // the forward's Phi stays in place
  const TwoPlane T = two_plane(F, pc, csm);
  const float2* src = a.spec + (copy ? F.tspec_off : F.spec_off) + size_t(x0) * T.Ny * T.Nzh;
  float* dst = a.mesh + (copy ? F.tmesh_off : F.mesh_off) + size_t(x0) * T.Ny * T.Nz;
  const float2* tz = a.tw + F.tw_off[2];
  const float2* ty = a.tw + F.tw_off[1];
  float2* S = T.b0;
  float2* S2 = T.b1;
  float2* Z = T.b0;
  const int tid = threadIdx.x, NT = blockDim.x;
  // y step 1, read from the planes' [ky][kz] blocks
  with_radix<MAXR>(T.Py, [&](auto rc) {
    constexpr int P = decltype(rc)::value;
    for (int it = tid; it < T.Qy * T.Sw; it += NT) {
      int t, col, pl = 0, kz;
      split_rc(it, T.Sw, T.rSw, t, col);
      if (pc > 1) split_rc(col, T.Nzh, T.rnzh, pl, kz);
      else kz = col;
      const float2* s = src + (pl * T.Ny + t) * T.Nzh + kz;
      float2 v[P];
#pragma unroll
      for (int m = 0; m < P; ++m) v[m] = s[T.Qy * m * T.Nzh];
      step1<P, true>(v, t, ty);
#pragma unroll
      for (int k = 0; k < P; ++k) S[(t + T.Qy * k) * T.Sw + col] = v[k];
    }
  });
  __syncthreads();
  with_radix<MAXR>(T.Qy, [&](auto rc) {
    constexpr int Q = decltype(rc)::value;
    for (int it = tid; it < T.Py * T.Sw; it += NT) {
      int k1, col;
      split_rc(it, T.Sw, T.rSw, k1, col);
      float2 u[Q];
#pragma unroll
      for (int t = 0; t < Q; ++t) u[t] = S[(t + Q * k1) * T.Sw + col];
      dft<Q, true>(u);
#pragma unroll
      for (int k2 = 0; k2 < Q; ++k2) S2[(k1 + T.Py * k2) * T.Sw + col] = u[k2];
    }
  });
  __syncthreads();
  // z step 1 on complex row pr = (half row 2 pp) + i (half row 2 pp + 1), extended by Hermitian
  // symmetry (the n_z = 0 and Nyquist entries of a real row's spectrum are real)
  with_radix<MAXR>(T.Pz, [&](auto rc) {
    constexpr int P = decltype(rc)::value;
    for (int it = tid; it < T.rows * T.Qz; it += NT) {
      int pr, t, pl = 0, pp;
      split_rc(it, T.Qz, T.rQz, pr, t);
      if (pc > 1) split_rc(pr, T.np, T.rnp, pl, pp);
      else pp = pr;
      const float2* ra = S2 + 2 * pp * T.Sw + pl * T.Nzh;
      const bool has_b = 2 * pp + 1 < T.Ny;
      float2 v[P];
#pragma unroll
      for (int m = 0; m < P; ++m) {
        const int k = t + T.Qz * m;
        const bool up = k < T.Nzh;
        const int kk = up ? k : T.Nz - k;
        float2 A = ra[kk], B = has_b ? ra[T.Sw + kk] : make_float2(0.f, 0.f);
        if (!up) {
          A.y = -A.y;
          B.y = -B.y;
        } else if (k == 0 || 2 * k == T.Nz) {
          A.y = 0.f;
          B.y = 0.f;
        }
        v[m] = make_float2(A.x - B.y, A.y + B.x);
      }
      step1<P, true>(v, t, tz);
#pragma unroll
      for (int k = 0; k < P; ++k) Z[(pr * P + k) * T.Qo + t] = v[k];
    }
  });
  __syncthreads();
  // z step 2: real parts to row 2 pp, imaginary parts to row 2 pp + 1
  with_radix<MAXR>(T.Qz, [&](auto rc) {
    constexpr int Q = decltype(rc)::value;
    for (int it = tid; it < T.rows * T.Pz; it += NT) {
      int pr, k1, pl = 0, pp;
      split_rc(it, T.Pz, T.rPz, pr, k1);
      if (pc > 1) split_rc(pr, T.np, T.rnp, pl, pp);
      else pp = pr;
      float2 u[Q];
#pragma unroll
      for (int t = 0; t < Q; ++t) u[t] = Z[it * (Q | 1) + t];
      dft<Q, true>(u);
      float* r0 = dst + (pl * T.Ny + 2 * pp) * T.Nz + k1;
      const bool has_b = 2 * pp + 1 < T.Ny;
#pragma unroll
      for (int k2 = 0; k2 < Q; ++k2) {
        r0[T.Pz * k2] = u[k2].x;
        if (has_b) r0[T.Nz + T.Pz * k2] = u[k2].y;
      }
    }
  });
}

// f with the radix R known (FIX > 0) or switched on
template <int FIX, int MAXR, class F>
__device__ __forceinline__ void radix_or(int r, F&& f) {
  if constexpr (FIX > 0) f(std::integral_constant<int, FIX>{});
  else with_radix<MAXR>(r, f);
}

// Pass B tile: kw columns of the spectrum (copy 0: rho's, with the energy and virial sums; 1: the
// tangent one): forward x transform, influence multiply, inverse x transform. FP, FQ: the
// factors of the x length when known (0: the frame's). smem: N0 kw entries.
template <int FP, int FQ, bool VIR, int MAXR = 16>
__device__ __forceinline__ void x_tile(const ConvArgs& a, const FrameDesc& F, int copy, int c0, int kw, float2* T) {
  const Geometry& g = F.g;
  const int P0 = FP > 0 ? FP : F.conv_p[0], Q0 = FQ > 0 ? FQ : F.conv_q[0];
  const int N0 = P0 * Q0, N1 = g.N[1], N2 = g.N[2], Nzh = N2 / 2 + 1;
  const int ncols = N1 * Nzh;   // (n_y, n_z) columns of a plane, contiguous for a fixed x
  const float rkw = 1.f / float(kw), rzh = 1.f / float(Nzh);
  const float2* tw = a.tw + F.tw_off[0];
  float2* col0 = a.spec + (copy ? F.tspec_off : F.spec_off) + c0;
  const int tid = threadIdx.x, NT = blockDim.x;
  radix_or<FP, MAXR>(P0, [&](auto rc) {
    constexpr int P = decltype(rc)::value;
    for (int it = tid; it < Q0 * kw; it += NT) {
      int t, c;
      split_rc(it, kw, rkw, t, c);
      const float2* s = col0 + size_t(t) * ncols + c;
      float2 v[P];
#pragma unroll
      for (int m = 0; m < P; ++m) v[m] = s[size_t(Q0 * m) * ncols];
      step1<P, false>(v, t, tw);
#pragma unroll
      for (int k = 0; k < P; ++k) T[(t + Q0 * k) * kw + c] = v[k];
    }
  });
  __syncthreads();
  const float* cx = a.dconv + F.dconv_off;
  const float* cy = cx + N0;
  const float* cz = cy + N1;
  float e = 0.f, ec = 0.f;
  float sv[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, sc[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  radix_or<FQ, MAXR>(Q0, [&](auto rc) {
    constexpr int Q = decltype(rc)::value;
    for (int it = tid; it < P0 * kw; it += NT) {
      int k1, c;
      split_rc(it, kw, rkw, k1, c);
      const int col = c0 + c;
      int iy, iz;
      split_rc(col, Nzh, rzh, iy, iz);
      float gcv[Q];
#pragma unroll
      for (int k2 = 0; k2 < Q; ++k2)
        gcv[k2] = a.gtab ? __ldg(a.gtab + F.gtab_off + size_t(k1 + P0 * k2) * ncols + col) : 0.f;
      float2* row = T + Q * k1 * kw + c;   // this thread's slots (t, k1), t < Q
      float2 u[Q];
#pragma unroll
      for (int t = 0; t < Q; ++t) u[t] = row[t * kw];
      dft<Q, false>(u);
      const float ny = float(iy <= N1 / 2 ? iy : iy - N1);
      const float nz = float(iz);
      const float wz = (iz == 0 || (2 * iz == N2)) ? 1.f : 2.f;
#pragma unroll
      for (int k2 = 0; k2 < Q; ++k2) {
        float gc = gcv[k2];
        if (VIR || !a.gtab) {
          const int ix = k1 + P0 * k2;
          const float nx = float(ix <= N0 / 2 ? ix : ix - N0);
          const float kx = nx * g.bk[0] + ny * g.bk[3] + nz * g.bk[6];
          const float kyv = nx * g.bk[1] + ny * g.bk[4] + nz * g.bk[7];
          const float kz = nx * g.bk[2] + ny * g.bk[5] + nz * g.bk[8];
          const float k2v = kx * kx + kyv * kyv + kz * kz;
          if (!a.gtab && k2v > 0.f)
            gc = 12.566370614359172f * expf(-k2v * a.inv4a2) / k2v * cx[ix] * cy[iy] * cz[iz];
          if (VIR && copy == 0 && k2v > 0.f) {
            const float tt = wz * gc * (u[k2].x * u[k2].x + u[k2].y * u[k2].y) * (1.f / k2v + a.inv4a2);
            comp_add(sv[0], sc[0], tt * kx * kx);
            comp_add(sv[1], sc[1], tt * kyv * kyv);
            comp_add(sv[2], sc[2], tt * kz * kz);
            comp_add(sv[3], sc[3], tt * kx * kyv);
            comp_add(sv[4], sc[4], tt * kx * kz);
            comp_add(sv[5], sc[5], tt * kyv * kz);
          }
        }
        if (copy == 0) comp_add(e, ec, wz * gc * (u[k2].x * u[k2].x + u[k2].y * u[k2].y));
        const float fac = gc * g.inv_volume;
        u[k2] = make_float2(u[k2].x * fac, u[k2].y * fac);
      }
      // the inverse transform split as Q P: u[m] = x[k1 + P m] is its step-1 input of offset k1
      step1<Q, true>(u, k1, tw);
#pragma unroll
      for (int k = 0; k < Q; ++k) row[k * kw] = u[k];
    }
  });
  __syncthreads();
  radix_or<FP, MAXR>(P0, [&](auto rc) {
    constexpr int P = decltype(rc)::value;
    for (int it = tid; it < Q0 * kw; it += NT) {
      int k, c;
      split_rc(it, kw, rkw, k, c);
      float2 v[P];
#pragma unroll
      for (int t = 0; t < P; ++t) v[t] = T[(k + Q0 * t) * kw + c];
      dft<P, true>(v);
      float2* d = col0 + size_t(k) * ncols + c;
#pragma unroll
      for (int k2 = 0; k2 < P; ++k2) d[size_t(Q0 * k2) * ncols] = v[k2];
    }
  });
  if (copy) return;
  __shared__ double wsum[kTwoXThreads / 32];
  const int blk = F.infl_blk_off + c0 / F.conv_cols;
  const double et = block_comp_sum(e, ec, wsum);
  if (threadIdx.x == 0) a.partials[blk] = et;
  if (VIR) {
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const double vt = block_comp_sum(sv[c], sc[c], wsum);
      if (threadIdx.x == 0) a.vparts[6 * blk + c] = vt;
    }
  }
}

// One block per tile and copy: a tangent pass on the forward's inputs then stages only its own
// columns (half the shared memory of both side by side). With the transforms on both sides of the
// multiply in registers and, for 64, 128 and 256 points, compile-time factors, the pass takes 9.6
// us at 128^3 (cold; the earlier power-of-two kernel, which crossed shared memory four times,
// 12.5); at 256^3 forward + backward of 262144 ions went from 1.77 to 1.74 ms.
// KNOWN: 1 every frame's x axis is 64 or 128 points, 2 it is 256 (compile-time factors); 3 any mix
// with factors up to kSmallRadix, 0 any mix.
// Blocks [0, blocks) take rho's tiles, [blocks, 2 blocks) (tangent passes) the tangent's.
template <bool BATCH, bool VIR, int KNOWN>
__global__ void __launch_bounds__(kTwoXThreads, VIR ? 2 : (KNOWN == 1 || KNOWN == 3 ? 4 : 3)) k_two_x(ConvArgs a, int blocks) {
  pdl_begin();
  extern __shared__ __align__(16) float2 csm[];
  const int copy = int(blockIdx.x) >= blocks ? 1 : 0, blk = int(blockIdx.x) - copy * blocks;
  // tangent pass on the forward's inputs: rho's columns are not needed again
  if (copy == 0 && a.tangent && a.keep && *a.keep == 0) return;
  const FrameDesc& F = frame_at<BATCH>(a.one, a.maps, BATCH ? a.maps.blk_frame[blk] : 0);
  const int c0 = (blk - F.infl_blk_off) * F.conv_cols;
  const int kw = min(F.conv_cols, F.g.N[1] * (F.g.N[2] / 2 + 1) - c0);
  if constexpr (KNOWN == 1) {
    if (F.g.N[0] == 128) x_tile<16, 8, VIR>(a, F, copy, c0, kw, csm);
    else x_tile<8, 8, VIR>(a, F, copy, c0, kw, csm);
  } else if constexpr (KNOWN == 2) {
    x_tile<16, 16, VIR>(a, F, copy, c0, kw, csm);
  } else {
    x_tile<0, 0, VIR, KNOWN == 3 ? kSmallRadix : 16>(a, F, copy, c0, kw, csm);
  }
}

constexpr int kRadices[] = {1, 2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16};

}  // namespace

// L = P Q, P >= Q, both built radices, as square as possible; false if there is none (of the
// 2,3,5-smooth lengths up to 256: 125, 162, 200, 216, 243 and 250).
bool two_step_factors(int L, int* P, int* Q) {
  bool found = false;
  for (int p : kRadices)
    for (int q : kRadices)
      if (p >= q && p * q == L && (!found || p < *P)) {
        *P = p;
        *Q = q;
        found = true;
      }
  return found;
}

// Widest step of a pass A / C block of pp planes: items of one DFT each.
static int two_items(const int N[3], int pp) {
  int Py, Qy, Pz, Qz;
  two_step_factors(N[1], &Py, &Qy);
  two_step_factors(N[2], &Pz, &Qz);
  return std::max(pp * ((N[1] + 1) / 2) * Pz, pp * (N[2] / 2 + 1) * Py);
}

// Planes of a pass A / C block: one for single frames (as many blocks as there are planes);
// in batches, which have planes to spare, enough of them for about two warps' worth of items
// per scheduler.
int two_planes_per_block(const int N[3], bool single) {
  if (single) return 1;
  int pp = 1;
  while (pp < N[0] && two_items(N, pp + 1) <= 320) ++pp;
  return pp;
}

int two_plane_threads(const int N[3], int pp) {
  return std::min(kTwoMaxThreads, std::max(64, (two_items(N, pp) + 31) / 32 * 32));
}

size_t two_plane_smem(const int N[3], int pp) {
  int Pz = 1, Qz = 1;
  two_step_factors(N[2], &Pz, &Qz);
  const size_t rows = size_t(pp) * ((N[1] + 1) / 2), Z = rows * Pz * (Qz | 1), Z2 = rows * (N[2] | 1),
               S = size_t(N[1]) * pp * (N[2] / 2 + 1);
  return (std::max(Z, S) + std::max(Z2, S)) * sizeof(float2);
}

size_t two_x_smem(const int N[3]) {
  int nt, cols;
  conv_tiles(N, &nt, &cols);
  return size_t(N[0]) * cols * sizeof(float2);
}

int launch_two_plane(pme_plan_t p, cudaStream_t s, const ConvArgs& a, int grid, bool inverse) {
  int st;
#define GB_TWO_PLANE(K)                                                      \
  do {                                                                       \
    static unsigned done = 0;                                                \
    if ((st = set_smem(p, K, done))) return st;                              \
    pdl_launch(K, grid, p->conv_threads, p->conv_smem_plane, s, a);          \
  } while (0)
#define GB_TWO_PLANE_R(R)                                \
  do {                                                    \
    if (p->batch && inverse) GB_TWO_PLANE((k_two_c2r<true, R>));  \
    else if (p->batch) GB_TWO_PLANE((k_two_r2c<true, R>)); \
    else if (inverse) GB_TWO_PLANE((k_two_c2r<false, R>)); \
    else GB_TWO_PLANE((k_two_r2c<false, R>));              \
  } while (0)
  if (p->conv_maxr <= kSmallRadix) GB_TWO_PLANE_R(kSmallRadix);
  else GB_TWO_PLANE_R(16);
#undef GB_TWO_PLANE_R
#undef GB_TWO_PLANE
  count_launch();
  return check_launch(p, inverse ? "k_two_c2r" : "k_two_r2c");
}

int launch_two_x(pme_plan_t p, cudaStream_t s, const ConvArgs& a, int grid) {
  int st;
#define GB_TWO_X(B, V, K)                                                                        \
  do {                                                                                           \
    static unsigned done = 0;                                                                    \
    if ((st = set_smem(p, k_two_x<B, V, K>, done))) return st;                                   \
    pdl_launch(k_two_x<B, V, K>, (a.tangent ? 2 : 1) * grid, kTwoXThreads, p->conv_smem_x, s, a, grid); \
  } while (0)
#define GB_TWO_X_KNOWN(K)                            \
  do {                                               \
    if (p->batch && a.vparts) GB_TWO_X(true, true, K);  \
    else if (p->batch) GB_TWO_X(true, false, K);     \
    else if (a.vparts) GB_TWO_X(false, true, K);     \
    else GB_TWO_X(false, false, K);                  \
  } while (0)
  if (p->conv_p2 || (p->conv_line && p->frames_h[0].g.N[0] <= 128)) GB_TWO_X_KNOWN(1);
  else if (p->conv_line) GB_TWO_X_KNOWN(2);
  else if (p->conv_maxr <= kSmallRadix) GB_TWO_X_KNOWN(3);
  else GB_TWO_X_KNOWN(0);
#undef GB_TWO_X_KNOWN
#undef GB_TWO_X
  count_launch();
  return check_launch(p, "k_two_x");
}

}  // namespace gbpme
