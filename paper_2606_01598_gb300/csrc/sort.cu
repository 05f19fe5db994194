// Sorting ions into mesh bricks and pair cells.
//
// Every ion gets two keys in one pass: the brick holding its first stencil point m0
// (Section 2.3.2, Eq. w3d) and the pair cell holding its position, both offset by its
// frame's first global key, so that one counting sort orders every frame of a batch and the
// ions of a frame stay contiguous. k_bin counts (one integer atomic per ion and key, never
// per stencil point), forms each ion's records and adds up each frame's charges (and tangent
// charges) in a fixed order for the background term; k_scan turns the counts into segment
// starts;
// k_scatter places ions in arrival order, and k_rank_records re-ranks each segment by caller
// index, which makes the order -- and hence every later sum -- deterministic, while writing
// the per-ion records both orders need. (The allocation-free spread, which needs no charge
// sums, skips them.) A backward whose inputs are bit for bit those of the plan's last forward
// (checked on the device first) keeps that forward's order and records and only adds the
// charge sums and the tangent records.
#include <algorithm>

#include "kernels.h"

namespace gbpme {

namespace {

constexpr int kSortThreads = kRedItem;   // binning: one block per reduction item
constexpr int kRankMaxSegment = 2048;   // longer segments keep arrival order

// Segments of a count array: one block each, kScanThreads threads on a whole number of int4s
// (both arrays are allocated padded to a multiple of 4 entries past n + 1). A block finds its
// own first start by adding up every count before its segment, so the blocks do not wait for
// one another; at most kScanMaxSegs segments keep that re-reading small (91125 pair cells: 22
// blocks reading 180 KB each on average, from L2).
constexpr int kScanThreads = 1024;
constexpr int kScanSeg = 4 * kScanThreads;
constexpr int kScanMaxSegs = 64;
__host__ __device__ __forceinline__ int scan_segment(int n) {
  const int whole = (n + kScanSeg - 1) / kScanSeg;
  return kScanSeg * max(1, (whole + kScanMaxSegs - 1) / kScanMaxSegs);
}

__device__ __forceinline__ int warp_inclusive(int v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  return v;
}

// start[k] for the counts of segment seg (length len, starting at entry seg len); the last
// segment also writes start[n] = total. The counts stay in place (k_scatter clears them).
__device__ void scan_one_segment(const int* count, int* start, int n, int seg, int len) {
  __shared__ int part[32];
  __shared__ int carry;
  const int lo = seg * len, hi = min(n, lo + len);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int before = 0;
#pragma unroll 4
  for (int k = 4 * threadIdx.x; k < lo; k += kScanSeg) {
    const int4 c = __ldcg(reinterpret_cast<const int4*>(count + k));
    before += (c.x + c.y) + (c.z + c.w);
  }
  before = __reduce_add_sync(0xffffffffu, before);
  if (lane == 0) part[wid] = before;
  __syncthreads();
  if (wid == 0) {
    const int t = __reduce_add_sync(0xffffffffu, part[lane]);
    if (lane == 0) carry = t;
  }
  __syncthreads();
  int run0 = carry;
  for (int k0 = lo; k0 < hi; k0 += kScanSeg) {
    const int k = k0 + 4 * threadIdx.x;
    int4 c = k < hi ? __ldcg(reinterpret_cast<const int4*>(count + k)) : make_int4(0, 0, 0, 0);
    if (k + 1 >= hi) c.y = 0;
    if (k + 2 >= hi) c.z = 0;
    if (k + 3 >= hi) c.w = 0;
    const int local = (c.x + c.y) + (c.z + c.w);
    const int v = warp_inclusive(local, lane);
    __syncthreads();   // part is read below in the round before
    if (lane == 31) part[wid] = v;
    __syncthreads();
    const int w = warp_inclusive(part[lane], lane);   // every warp: inclusive prefix over the warps
    const int total = __shfl_sync(0xffffffffu, w, 31);
    const int warps_before = __shfl_sync(0xffffffffu, w, max(wid - 1, 0));
    if (k < hi) {
      int4 o;
      o.x = run0 + v - local + (wid > 0 ? warps_before : 0);
      o.y = o.x + c.x;
      o.z = o.y + c.y;
      o.w = o.z + c.z;
      *reinterpret_cast<int4*>(start + k) = o;
    }
    run0 += total;
  }
  __syncthreads();   // the write of start[n] follows the padding entries of the last int4
  if (hi == n && threadIdx.x == 0) start[n] = run0;
}

// Mesh and cell coordinates of an ion in compensated float32 (GB300's float64 rate is a small
// fraction of its float32 rate); positions beyond the float path's range, or not finite, take
// the float64 path.
__device__ __forceinline__ void ion_origins(const Geometry& g, float rx, float ry, float rz, int (&m0)[3],
                                            float (&fb)[3], int (&c)[3], float (&fc)[3]) {
  bool fast = true;
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    fast = fast && stencil_origin_f(g, rx, ry, rz, b, m0[b], fb[b]);
    fast = fast && cell_origin_f(g, rx, ry, rz, b, c[b], fc[b]);
  }
  if (fast) return;
  double s[3];
  frac_coords(g, rx, ry, rz, s);
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    stencil_origin(s[b], g.N[b], g.order, m0[b], fb[b]);
    cell_origin(s[b], g.ncell[b], c[b], fc[b]);
  }
}

// Charge and dipole of ion i (non-finite values as zero) and, tangent, its (dq, dr, d' = dmu + q dr).
struct IonSources {
  float q, mu[3], dq, dr[3], dp[3];
};
__device__ __forceinline__ IonSources ion_sources(const IonInputs& in, int i, int tangent) {
  IonSources S;
  S.q = in.q ? in.q[i] : 0.f;
  if (!isfinite(S.q)) S.q = 0.f;
  float dmu[3] = {0.f, 0.f, 0.f};
  S.dq = tangent && in.gphi ? in.gphi[i] : 0.f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    S.mu[a] = in.mu ? in.mu[3 * i + a] : 0.f;
    if (!isfinite(S.mu[a])) S.mu[a] = 0.f;
    S.dr[a] = tangent && in.gforce ? -in.gforce[3 * i + a] : 0.f;
    if (tangent && in.gfield) dmu[a] = -in.gfield[3 * i + a];
    S.dp[a] = dmu[a] + S.q * S.dr[a];
  }
  return S;
}
__device__ __forceinline__ void to_mesh(const Geometry& g, const float (&v)[3], float (&o)[3]) {
#pragma unroll
  for (int b = 0; b < 3; ++b) o[b] = v[0] * g.D[0 * 3 + b] + v[1] * g.D[1 * 3 + b] + v[2] * g.D[2 * 3 + b];
}
__device__ __forceinline__ void store_mesh_tangent(const Geometry& g, const MeshRecords& mr, int dest,
                                                   const IonSources& S) {
  float pd[3], pt[3];
  to_mesh(g, S.dp, pd);
  to_mesh(g, S.dr, pt);
  mr.tq[dest] = make_float4(S.dq, pd[0], pd[1], pd[2]);
  mr.tt[dest] = make_float4(pt[0], pt[1], pt[2], 0.f);
}
__device__ __forceinline__ void store_pair_tangent(const PairRecords& pr, int dest, const IonSources& S) {
  pr.tq[dest] = make_float4(S.dq, S.dp[0], S.dp[1], S.dp[2]);
  pr.dr[dest] = make_float4(S.dr[0], S.dr[1], S.dr[2], 0.f);
}

// One block per reduction item (kRedItem = kSortThreads ions of one frame, one per thread):
// the ion's brick key and pair-cell key with one counting atomic each, its records in caller
// order, and the item's charge sums (k_scan adds a frame's items in order).
template <bool BATCH>
__global__ void __launch_bounds__(kSortThreads)
k_bin(FrameDesc one, FrameMaps maps, IonInputs in, const PassIO* io, SortBuffers sb, int tangent, int* flags,
      const int* reuse, float* save, int ld, int* saved_n) {
  pdl_begin();
  if (io) in = io->in;
  static_assert(kRedItem == kSortThreads, "one ion per thread");
  const int item = blockIdx.x;
  const int f = BATCH ? maps.item_frame[item] : 0;
  const FrameDesc& F = frame_at<BATCH>(one, maps, f);
  int lo, hi;
  item_range(F, item, lo, hi);
  const int i = lo + int(threadIdx.x);
  // reuse: the inputs are those of the forward whose sort is still in place; only the charge
  // sums are formed
  const bool re = reuse && *reuse == 0;
  if (!re && saved_n && item == 0 && threadIdx.x == 0) *saved_n = save ? in.n : 0;
  float qa = 0.f, qb = 0.f;
  if (re && i < hi) {
    const float qi = in.q ? in.q[i] : 0.f;
    qa = isfinite(qi) ? qi : 0.f;
    qb = (tangent && in.gphi) ? in.gphi[i] : 0.f;
  } else if (i < hi) {
    const Geometry& g = F.g;
    const float rx = in.pos[3 * i], ry = in.pos[3 * i + 1], rz = in.pos[3 * i + 2];
    const float qi = in.q ? in.q[i] : 0.f;
    if (save) {
      // the forward's inputs, bit for bit, for the comparison a later backward makes
      save[3 * i] = rx;
      save[3 * i + 1] = ry;
      save[3 * i + 2] = rz;
      save[3 * ld + i] = qi;
#pragma unroll
      for (int a = 0; a < 3; ++a) save[4 * ld + 3 * i + a] = in.mu ? in.mu[3 * i + a] : 0.f;
    }
    bool ok = isfinite(rx) && isfinite(ry) && isfinite(rz) && isfinite(qi);
    if (in.mu) ok = ok && isfinite(in.mu[3 * i]) && isfinite(in.mu[3 * i + 1]) && isfinite(in.mu[3 * i + 2]);
    if (in.theta) {
#pragma unroll
      for (int a = 0; a < 6; ++a) ok = ok && isfinite(in.theta[6 * i + a]);
    }
    if (!ok) atomicOr(flags, kFlagNonFinite);
    int m0[3], c[3];
    float fb[3], fc[3];
    ion_origins(g, rx, ry, rz, m0, fb, c, fc);
    const int kb = F.brick_off + ((m0[0] / g.brick[0]) * g.nb[1] + m0[1] / g.brick[1]) * g.nb[2] +
                   m0[2] / g.brick[2];
    const int kc = F.cell_off + (c[0] * g.ncell[1] + c[1]) * g.ncell[2] + c[2];
    sb.key_b[i] = kb;
    sb.key_c[i] = kc;
    sb.slot_b[i] = atomicAdd(&sb.count_b[kb], 1);
    sb.slot_c[i] = atomicAdd(&sb.count_c[kc], 1);
    if (sb.t_bidx) {
      // the primal records of both orders, in caller order (the rank pass moves them)
      const float qs = isfinite(qi) ? qi : 0.f;
      float mu[3] = {0.f, 0.f, 0.f};
      if (in.mu) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          mu[a] = in.mu[3 * i + a];
          if (!isfinite(mu[a])) mu[a] = 0.f;
        }
      }
      float pm[3];
#pragma unroll
      for (int b = 0; b < 3; ++b) pm[b] = mu[0] * g.D[0 * 3 + b] + mu[1] * g.D[1 * 3 + b] + mu[2] * g.D[2 * 3 + b];
      sb.t_bidx[i] = make_int4(m0[0], m0[1], m0[2], i);
      sb.t_bfq[i] = make_float4(fb[0], fb[1], fb[2], qs);
      sb.t_bdm[i] = make_float4(pm[0], pm[1], pm[2], 0.f);
      sb.t_cidx[i] = make_int4(c[0], c[1], c[2], i);
      sb.t_cfq[i] = make_float4(fc[0], fc[1], fc[2], __int_as_float(c[2]));
      sb.t_cmu[i] = make_float4(mu[0], mu[1], mu[2], qs);
    }
    qa = isfinite(qi) ? qi : 0.f;
    qb = (tangent && in.gphi) ? in.gphi[i] : 0.f;
  }
  if (sb.qpart) {
    double A, B;
    block_sum2_f(qa, qb, A, B);
    if (threadIdx.x == 0) {
      sb.qpart[2 * item] = A;
      sb.qpart[2 * item + 1] = B;
    }
  }
}

// Segment starts from the final counts (skipped on reuse) and the frames' charge sums from
// their items' partials: blocks [0, nb) scan the brick counts, [nb, nb + nc) the cell counts, the
// rest add the items of 32 frames each, one warp per frame. One 1024-thread block per array took
// 50 us at 262144 ions (91125 cells) and 22 us for 256 uneven frames; the charge sums were the
// binning pass's last block, alone on its SM for 2.8 us of every sort. Forward of 32768 ions 142.6 ->
// 137.5 us, forward + backward of 262144 ions 1.82 -> 1.78 ms, 256 uneven frames 1.25 -> 1.23 ms.
template <bool BATCH>
__global__ void __launch_bounds__(kScanThreads)
k_scan(FrameDesc one, FrameMaps maps, int nframes, SortBuffers sb, int nbricks, int ncells, int nb, int nc,
       const int* reuse) {
  pdl_begin();
  const int b = blockIdx.x;
  if (b < nb + nc) {
    if (reuse && *reuse == 0) return;
    if (b < nb) scan_one_segment(sb.count_b, sb.start_b, nbricks, b, scan_segment(nbricks));
    else scan_one_segment(sb.count_c, sb.start_c, ncells, b - nb, scan_segment(ncells));
    return;
  }
  const int f = (b - nb - nc) * (kScanThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (f >= nframes) return;
  const FrameDesc& F = frame_at<BATCH>(one, maps, f);
  const double2* part = reinterpret_cast<const double2*>(sb.qpart) + F.item_off;
  double qa = 0.0, qb = 0.0;
#pragma unroll 4
  for (int k = lane; k < F.nitems; k += 32) {
    const double2 v = __ldcg(part + k);
    qa += v.x;
    qb += v.y;
  }
  qa = warp_sum_d(qa);
  qb = warp_sum_d(qb);
  if (lane == 0) {
    sb.qsum[2 * f] = qa;
    sb.qsum[2 * f + 1] = qb;
  }
}

__global__ void __launch_bounds__(kSortThreads)
k_scatter(int n, SortBuffers sb, int nbricks, int ncells, int need_mesh, int need_pair, const int* reuse) {
  pdl_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (reuse && *reuse == 0) return;
  // the counts are dead once scanned: leave them zero for the next sort
  for (int k = 4 * i; k < nbricks; k += 4 * gridDim.x * blockDim.x)
    *reinterpret_cast<int4*>(sb.count_b + k) = make_int4(0, 0, 0, 0);
  for (int k = 4 * i; k < ncells; k += 4 * gridDim.x * blockDim.x)
    *reinterpret_cast<int4*>(sb.count_c + k) = make_int4(0, 0, 0, 0);
  if (i >= n) return;
  if (need_mesh) {
    const int d = sb.start_b[sb.key_b[i]] + sb.slot_b[i];
    if (index_ok(d, n)) sb.perm_b[d] = i;
  }
  if (need_pair) {
    const int d = sb.start_c[sb.key_c[i]] + sb.slot_c[i];
    if (index_ok(d, n)) sb.perm_c[d] = i;
  }
}

__device__ __forceinline__ int stable_rank(const int* perm, int seg_lo, int seg_hi, int self,
                                           int fallback) {
  if (seg_hi - seg_lo > kRankMaxSegment) return fallback;
  int r = 0;
#pragma unroll 8
  for (int u = seg_lo; u < seg_hi; ++u) r += (perm[u] < self) ? 1 : 0;   // eight loads in flight
  return seg_lo + r;
}

template <bool BATCH>
__global__ void __launch_bounds__(kSortThreads)
k_rank_records(FrameDesc one, FrameMaps maps, IonInputs in, const PassIO* io, SortBuffers sb, MeshRecords mr,
               PairRecords pr, int tangent, int need_mesh, int need_pair, const int* reuse) {
  pdl_begin();
  if (io) in = io->in;
  const int n = in.n;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  const bool mesh_side = t < n;
  if (!mesh_side) t -= n;
  if (t >= n) return;
  if (mesh_side && !need_mesh) return;
  if (!mesh_side && !need_pair) return;
  // reuse: the forward's records stay; only the tangent records are written, at the sorted
  // slot the forward gave each ion
  const bool re = reuse && *reuse == 0;
  int i, dest;
  if (re) {
    dest = t;
    i = mesh_side ? mr.idx[t].w : pr.idx[t].w;
  } else if (mesh_side) {
    i = sb.perm_b[t];
    const int k = sb.key_b[i];
    dest = stable_rank(sb.perm_b, sb.start_b[k], sb.start_b[k + 1], i, t);
  } else {
    i = sb.perm_c[t];
    const int k = sb.key_c[i];
    dest = stable_rank(sb.perm_c, sb.start_c[k], sb.start_c[k + 1], i, t);
  }
  if (!index_ok(i, n) || !index_ok(dest, n)) return;
  const int f = BATCH ? maps.ion_frame[i] : 0;
  const FrameDesc& F = frame_at<BATCH>(one, maps, f);
  const Geometry& g = F.g;
  const float rx = in.pos[3 * i], ry = in.pos[3 * i + 1], rz = in.pos[3 * i + 2];
  const IonSources S = ion_sources(in, i, tangent);
  if (tangent) {
    if (mesh_side) store_mesh_tangent(g, mr, dest, S);
    else store_pair_tangent(pr, dest, S);
  }
  if (re) return;
  if (sb.t_bidx) {
    // primal records from the binning pass
    if (mesh_side) {
      mr.idx[dest] = sb.t_bidx[i];
      mr.fq[dest] = sb.t_bfq[i];
      mr.dm[dest] = sb.t_bdm[i];
    } else {
      pr.idx[dest] = sb.t_cidx[i];
      pr.fq[dest] = sb.t_cfq[i];
      pr.mu[dest] = sb.t_cmu[i];
    }
    return;
  }
  // the binning pass's coordinates: compensated float32, float64 where that does not apply
  double s[3];
  bool fast = true;
  int m0[3], cc[3];
  float fm[3], fcl[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    if (mesh_side) fast = fast && stencil_origin_f(g, rx, ry, rz, b, m0[b], fm[b]);
    else fast = fast && cell_origin_f(g, rx, ry, rz, b, cc[b], fcl[b]);
  }
  if (!fast) frac_coords(g, rx, ry, rz, s);
  if (mesh_side) {
    float fr[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      if (fast) fr[b] = fm[b];
      else stencil_origin(s[b], g.N[b], g.order, m0[b], fr[b]);
    }
    float pm[3];
    to_mesh(g, S.mu, pm);
    mr.idx[dest] = make_int4(m0[0], m0[1], m0[2], i);
    mr.fq[dest] = make_float4(fr[0], fr[1], fr[2], S.q);
    mr.dm[dest] = make_float4(pm[0], pm[1], pm[2], 0.f);
  } else {
    int c[3];
    float fr[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      if (fast) {
        c[b] = cc[b];
        fr[b] = fcl[b];
      } else {
        cell_origin(s[b], g.ncell[b], c[b], fr[b]);
      }
    }
    pr.idx[dest] = make_int4(c[0], c[1], c[2], i);
    pr.fq[dest] = make_float4(fr[0], fr[1], fr[2], __int_as_float(c[2]));
    pr.mu[dest] = make_float4(S.mu[0], S.mu[1], S.mu[2], S.q);
  }
}

// ---- small systems: the whole sort in one block ------------------------------------------
// A few hundred ions keep four (with the input check, five) kernels of one to sixteen blocks
// busy for about 2 us each, most of it launch and memory latency. One block does the same
// in one kernel, a thread per ion, with the counts, the starts and both orders in shared memory;
// keys, records, order and outputs are those of the kernels above. Taken for single frames of up
// to kSmallIons ions whose keys fit; beyond, one SM's own work outlasts the launches it saves.
// Forward pass with this sort and with the kernels above, us: 64 ions 39.0 and 42.1, 200: 41.8
// and 45.9, 300: 44.3 and 47.7, 400: 48.1 and 49.5, 512: 47.3 and 46.8, 1200: 57.5 and 49.9;
// forward + backward of 64: 69.1 and 74.3, 300: 80.6 and 84.9, 400: 86.1 and 88.1.
constexpr int kSmallIons = 384;
constexpr int kSmallKeys = 8192;

// saved / in_diff / cache_bad / list_cnt: as k_input_check (in_diff null: no check); save, saved_n: as k_bin.
__global__ void __launch_bounds__(kSmallIons)
k_sort_small(FrameDesc one, IonInputs in, const PassIO* io, SortBuffers sb, MeshRecords mr, PairRecords pr,
             int tangent, int need_mesh, int need_pair, int* flags, int nbricks, int ncells, float* save, int ld,
             const float* saved, const int* list_cnt, int* in_diff, int* cache_bad, int* saved_n) {
  pdl_begin();
  if (io) in = io->in;
  extern __shared__ __align__(16) int keys[];   // [nbricks + ncells] counts, then starts
  const int n = in.n, T = blockDim.x, tid = threadIdx.x, nk = nbricks + ncells;
  unsigned short* order_b = reinterpret_cast<unsigned short*>(keys + nk);
  unsigned short* order_c = order_b + kSmallIons;
  const Geometry& g = one.g;
  bool re = false;
  if (in_diff) {
    bool same = *saved_n == n, lists = true;
    for (int k = tid; k < 3 * n; k += T) {
      same = same && __float_as_int(in.pos[k]) == __float_as_int(saved[k]);
      same = same && __float_as_int(in.mu ? in.mu[k] : 0.f) == __float_as_int(saved[4 * ld + k]);
    }
    for (int k = tid; k < n; k += T) {
      same = same && __float_as_int(in.q ? in.q[k] : 0.f) == __float_as_int(saved[3 * ld + k]);
      if (list_cnt) lists = lists && list_cnt[k] >= 0;
    }
    const bool diff = __syncthreads_or(!same), bad = __syncthreads_or(!lists);
    if (tid == 0) {
      *in_diff = diff;
      *cache_bad = diff || bad;
    }
    re = !diff;
  }
  if (!re)
    for (int k = tid; k < nk; k += T) keys[k] = 0;
  __syncthreads();
  if (!re && saved_n && tid == 0) *saved_n = save ? n : 0;
  // keys and arrival slots of this thread's ion (n <= T)
  const int i = tid;
  int kb = 0, kc = 0, slot_b = 0, slot_c = 0, m0[3], c[3];
  float fb[3], fc[3];
  double qa = 0.0, qb = 0.0;
  if (i < n) {
    const float qi = in.q ? in.q[i] : 0.f;
    qa += isfinite(qi) ? double(qi) : 0.0;
    if (tangent && in.gphi) qb += double(in.gphi[i]);
    if (!re) {
      const float rx = in.pos[3 * i], ry = in.pos[3 * i + 1], rz = in.pos[3 * i + 2];
      bool ok = isfinite(rx) && isfinite(ry) && isfinite(rz) && isfinite(qi);
      if (save) {
        save[3 * i] = rx;
        save[3 * i + 1] = ry;
        save[3 * i + 2] = rz;
        save[3 * ld + i] = qi;
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float m = in.mu ? in.mu[3 * i + a] : 0.f;
        ok = ok && isfinite(m);
        if (save) save[4 * ld + 3 * i + a] = m;
      }
      if (in.theta) {
#pragma unroll
        for (int a = 0; a < 6; ++a) ok = ok && isfinite(in.theta[6 * i + a]);
      }
      if (!ok) atomicOr(flags, kFlagNonFinite);
      ion_origins(g, rx, ry, rz, m0, fb, c, fc);
      kb = ((m0[0] / g.brick[0]) * g.nb[1] + m0[1] / g.brick[1]) * g.nb[2] + m0[2] / g.brick[2];
      kc = nbricks + (c[0] * g.ncell[1] + c[1]) * g.ncell[2] + c[2];
      slot_b = atomicAdd(&keys[kb], 1);
      slot_c = atomicAdd(&keys[kc], 1);
    }
  }
  block_sum2_d(qa, qb);   // (its barriers also end the counting)
  if (tid == 0) {
    sb.qsum[0] = qa;
    sb.qsum[1] = qb;
  }
  if (re) {
    if (!tangent) return;
    for (int t = tid; t < 2 * n; t += T) {
      const bool mesh_side = t < n;
      const int dest = mesh_side ? t : t - n;
      if (mesh_side ? !need_mesh : !need_pair) continue;
      const int ion = mesh_side ? mr.idx[dest].w : pr.idx[dest].w;
      if (!index_ok(ion, n)) continue;
      const IonSources S = ion_sources(in, ion, tangent);
      if (mesh_side) store_mesh_tangent(g, mr, dest, S);
      else store_pair_tangent(pr, dest, S);
    }
    return;
  }
  // exclusive scan of the bricks' and the cells' counts laid end to end, in place: the bricks hold
  // all n ions, so a cell's start is its prefix less n
  __syncthreads();
  {
    __shared__ int part[32];
    const int lane = tid & 31, wid = tid >> 5, nw = T >> 5;
    const int chunk = ((nk + T - 1) / T) | 1,   // odd: a warp's chunks start in different banks
               lo = min(nk, tid * chunk), hi = min(nk, lo + chunk);
    int local = 0;
    for (int k = lo; k < hi; ++k) local += keys[k];
    const int v = warp_inclusive(local, lane);
    if (lane == 31) part[wid] = v;
    __syncthreads();
    const int w = warp_inclusive(lane < nw ? part[lane] : 0, lane);
    int run = v - local + __shfl_sync(0xffffffffu, w, max(wid - 1, 0)) * (wid > 0 ? 1 : 0);
    for (int k = lo; k < hi; ++k) {
      const int cnt = keys[k], start = k < nbricks ? run : run - n;
      keys[k] = start;
      if (k < nbricks) sb.start_b[k] = start;
      else sb.start_c[k - nbricks] = start;
      run += cnt;
    }
    if (tid == 0) {
      sb.start_b[nbricks] = n;
      sb.start_c[ncells] = n;
    }
  }
  __syncthreads();
  if (i < n) {
    order_b[keys[kb] + slot_b] = (unsigned short)i;
    order_c[keys[kc] + slot_c] = (unsigned short)i;
  }
  __syncthreads();
  if (i < n) {
    // rank by caller index within the brick and within the cell
    const int b0 = keys[kb], b1 = kb + 1 < nbricks ? keys[kb + 1] : n;
    const int c0 = keys[kc], c1 = kc + 1 < nk ? keys[kc + 1] : n;
    int db = b0, dc = c0;
    for (int k = b0; k < b1; ++k) db += order_b[k] < i ? 1 : 0;
    for (int k = c0; k < c1; ++k) dc += order_c[k] < i ? 1 : 0;
    const IonSources S = ion_sources(in, i, tangent);
    if (need_mesh && index_ok(db, n)) {
      float pm[3];
      to_mesh(g, S.mu, pm);
      mr.idx[db] = make_int4(m0[0], m0[1], m0[2], i);
      mr.fq[db] = make_float4(fb[0], fb[1], fb[2], S.q);
      mr.dm[db] = make_float4(pm[0], pm[1], pm[2], 0.f);
      if (tangent) store_mesh_tangent(g, mr, db, S);
    }
    if (need_pair && index_ok(dc, n)) {
      pr.idx[dc] = make_int4(c[0], c[1], c[2], i);
      pr.fq[dc] = make_float4(fc[0], fc[1], fc[2], __int_as_float(c[2]));
      pr.mu[dc] = make_float4(S.mu[0], S.mu[1], S.mu[2], S.q);
      if (tangent) store_pair_tangent(pr, dc, S);
    }
  }
}

// Bitwise comparison of the backward's inputs with the saved forward inputs (which count only while
// that forward's state is in place: *saved_n == n).
__global__ void __launch_bounds__(256)
k_input_check(int n, IonInputs in, const PassIO* io, const float* saved, int ld, const int* list_cnt, int* in_diff,
              int* cache_bad, const int* saved_n) {
  pdl_begin();
  if (io) in = io->in;
  bool same = *saved_n == n, lists = true;
  const int stride = gridDim.x * blockDim.x;
  const int t0 = blockIdx.x * blockDim.x + threadIdx.x;
  for (int k = t0; k < 3 * n; k += stride) {
    same = same && __float_as_int(in.pos[k]) == __float_as_int(saved[k]);
    const float m = in.mu ? in.mu[k] : 0.f;
    same = same && __float_as_int(m) == __float_as_int(saved[4 * ld + k]);
  }
  for (int k = t0; k < n; k += stride) {
    const float q = in.q ? in.q[k] : 0.f;
    same = same && __float_as_int(q) == __float_as_int(saved[3 * ld + k]);
    if (list_cnt) lists = lists && list_cnt[k] >= 0;
  }
  const bool diff = __any_sync(0xffffffffu, !same);
  const bool bad = __any_sync(0xffffffffu, !lists);
  if ((threadIdx.x & 31) == 0) {
    if (diff) *in_diff = 1;
    if (diff || bad) *cache_bad = 1;
  }
}

bool sort_is_small(pme_plan_t p, int n) {
  return !p->batch && p->nframes == 1 && p->sb.qsum && n > 0 && n <= kSmallIons && p->sb.qpart &&
         p->total_bricks + p->total_cells <= kSmallKeys;
}

int launch_input_check(pme_plan_t p, cudaStream_t s, const IonInputs& in, bool with_lists) {
  // (a recorded pass's first node clears the flags)
  int st = p->io_live ? PME_OK : check_cuda(p, cudaMemsetAsync(p->in_flags, 0, 2 * sizeof(int), s), "memset");
  if (st || in.n == 0) return st;
  const int grid = std::min(4 * device_sm_count(), (3 * in.n + 255) / 256);
  pdl_launch(k_input_check, grid, 256, 0, s, in.n, in, live_io(p), p->in_saved, p->max_ions, with_lists ? p->plist_cnt : nullptr,
                                      p->in_diff, p->cache_bad, p->saved_n);
  count_launch();
  return check_launch(p, "k_input_check");
}

template <bool BATCH>
int launch_sort_t(pme_plan_t p, cudaStream_t s, const IonInputs& in, bool tangent, bool need_mesh,
                  bool need_pair, const int* reuse, float* save, bool check_lists) {
  const int n = in.n;
  const int nblk = (n + kSortThreads - 1) / kSortThreads;
  FrameDesc one = p->frames_h[0];
  if (!BATCH) {
    one.n = n;
    one.item_off = 0;
    one.nitems = std::max(1, (n + kRedItem - 1) / kRedItem);
  }
  int st = PME_OK;
  if (!BATCH && sort_is_small(p, n)) {
    const int nk = p->total_bricks + p->total_cells;
    const int threads = std::max(128, (n + 31) / 32 * 32);
    const bool check = reuse != nullptr;
    pdl_launch(k_sort_small, 1, threads, sizeof(int) * nk + 2 * sizeof(unsigned short) * kSmallIons, s, one, in,
               live_io(p), p->sb, p->mr, p->pr, tangent ? 1 : 0, need_mesh ? 1 : 0, need_pair ? 1 : 0, p->flags,
               p->total_bricks, p->total_cells, save, p->max_ions, check ? p->in_saved : nullptr,
               check && check_lists ? p->plist_cnt : nullptr, check ? p->in_diff : nullptr,
               check ? p->cache_bad : nullptr, p->saved_n);
    count_launch();
    return check_launch(p, "k_sort_small");
  }
  if (reuse && (st = launch_input_check(p, s, in, check_lists))) return st;
  if (!p->counts_clean) {
    st = check_cuda(p, cudaMemsetAsync(p->sb.count_b, 0, sizeof(int) * (p->total_bricks + 1), s),
                    "memset brick counts");
    if (st) return st;
    st = check_cuda(p, cudaMemsetAsync(p->sb.count_c, 0, sizeof(int) * (p->total_cells + 1), s),
                    "memset cell counts");
    if (st) return st;
  }
  p->counts_clean = false;   // until k_scatter, which clears them, is launched
  {
    const int items = BATCH ? p->total_items : one.nitems;
    pdl_launch(k_bin<BATCH>, items, kSortThreads, 0, s, one, p->maps, in, live_io(p), p->sb, tangent ? 1 : 0, p->flags,
                                                reuse, save, p->max_ions, p->saved_n);
    count_launch();
    if ((st = check_launch(p, "k_bin"))) return st;
    const int nb = (p->total_bricks + scan_segment(p->total_bricks) - 1) / scan_segment(p->total_bricks);
    const int nc = (p->total_cells + scan_segment(p->total_cells) - 1) / scan_segment(p->total_cells);
    const int nq = p->sb.qpart ? (p->nframes + kScanThreads / 32 - 1) / (kScanThreads / 32) : 0;
    pdl_launch(k_scan<BATCH>, nb + nc + nq, kScanThreads, 0, s, one, p->maps, p->nframes, p->sb, p->total_bricks,
               p->total_cells, nb, nc, reuse);
    count_launch();
    if ((st = check_launch(p, "k_scan"))) return st;
  }
  if (nblk > 0) {
    const int clear = (std::max(p->total_bricks, p->total_cells) / 4 + kSortThreads - 1) / kSortThreads;
    pdl_launch(k_scatter, std::max(nblk, std::min(clear, 4 * device_sm_count())), kSortThreads, 0, s, n, p->sb,
               p->total_bricks, p->total_cells, need_mesh ? 1 : 0, need_pair ? 1 : 0, reuse);
    count_launch();
    if ((st = check_launch(p, "k_scatter"))) return st;
    const int nblk2 = (2 * n + kSortThreads - 1) / kSortThreads;
    pdl_launch(k_rank_records<BATCH>, nblk2, kSortThreads, 0, s, one, p->maps, in, live_io(p), p->sb, p->mr, p->pr,
                                                         tangent ? 1 : 0, need_mesh ? 1 : 0,
                                                         need_pair ? 1 : 0, reuse);
    count_launch();
    if ((st = check_launch(p, "k_rank_records"))) return st;
  }
  p->counts_clean = true;
  return PME_OK;
}

}  // namespace

int launch_sort(pme_plan_t p, cudaStream_t s, const IonInputs& in, bool tangent, bool need_mesh,
                bool need_pair, const int* reuse, float* save, bool check_lists) {
  if (!reuse) p->fwd_n = -1;   // the sorted records no longer belong to the saved inputs
  return p->batch ? launch_sort_t<true>(p, s, in, tangent, need_mesh, need_pair, reuse, save, check_lists)
                  : launch_sort_t<false>(p, s, in, tangent, need_mesh, need_pair, reuse, save, check_lists);
}

GBPME_BOUNDS_READER(bounds_hit_sort)

}  // namespace gbpme
