// The star path's finishing kernels (star.cuh): the hull of the single-read
// front's raw survivors, and the whole hull of a small input in one launch.
//
// k_cand   tests K1's raw survivors against the polygon of the angular
//          candidates (about 60k of 20M points of a disk come in, 3k go on)
//          and appends the rest to a list;
// k_star   one block sorts the list by angle and finds the hull in shared
//          memory.  It is a kernel of its own, not k_cand's last block, so
//          that k_cand's blocks need little shared memory and fit beside
//          another lane's K1, which leaves two SMs free for this one.
// k_small  one block: frame, sample polygon, one pass over the points, then
//          the same on the points left.
//
// Both are bound by latency (barriers and dependent loads), so the design
// counts those: what the bucket sort and the chain merges did in eight
// launches over the same few thousand points is one block's shared memory
// here (k_star 22-27 us for 20M points under the profiler, 14-17 for 100k,
// against 115-130 us of kernels before).  An input on one line or on one point
// is decided here too.  A list beyond kStarCap, a crowded bin or an input
// without a polygon for another reason sets ERR_RETRY: the call goes on with
// the sectors (k_sector.cu) or the bucket sort.
#include "hull_internal.cuh"
#include "kernels.h"
#include "star.cuh"

namespace gbh {

namespace {

constexpr int KS_BLOCK = 1024;
constexpr int KS_CAP = (int)kStarCap;
// Up to this many points k_small takes them all into its list: below it the
// sample polygon costs more than it saves (1,000 points 38-41 us a call
// without; at the line 49-53 without, 40-49 with it at 4,097, where the
// sample of 4,096 points is as long as the list).
constexpr u32 KS_DIRECT = 4096;
constexpr u32 KS_SLABS = 2048;
constexpr int KS_SAMPLES = 4;         // samples per thread of k_small's polygon

typedef star::ListSmem<KS_BLOCK, KS_CAP, kStarBins> List;
typedef star::CandTab<kStarBins> Cands;

struct SmallSmem {
  List list;
  union {
    struct {
      u64 key[kStarBins];
      Cands cands;
    };
    u32 tab[KS_SLABS];
  };
  star::FrameSmem<KS_BLOCK> frame;
  star::PolySmem poly;
  u64 best[kPolyDirs];
  u32 count, error;
};

// No polygon: a degenerate input (1; k_star tries the line); too many raw
// survivors for one block (2).
__device__ __forceinline__ int not_here(const PolyTab* T, u32 q, u32 n) {
  return !T->head.ok ? 1 : q > many_raw(n) ? 2 : 0;
}

constexpr int KC_BLOCK = 512;

__global__ void __launch_bounds__(KC_BLOCK)
k_cand(const int2* __restrict__ P, u32 n, PolyTab* T, const int2* rxy, const u32* ridx, int2* lxy, u32* lidx) {
  __shared__ Cands S;
  const int lane = threadIdx.x & 31, t = threadIdx.x;
  if (t < kStarBins / 32) S.occ[t] = 0u;
  pdl_wait();
  // Everything that hangs on nothing else is under way at once: the keys, the
  // head and this thread's first survivor (its slot exists, whatever it holds).
  constexpr int PER = kStarBins / KC_BLOCK;
  u64 k[PER];
  int2 p[PER];
  #pragma unroll
  for (int j = 0; j < PER; ++j) k[j] = __ldcg(&T->key[t + j * KC_BLOCK]);
  u32 i = blockIdx.x * (u32)KC_BLOCK + t;
  int2 w = i < n ? rxy[i] : make_int2(0, 0);
  u32 id = i < n ? ridx[i] : 0u;
  const u32 q = min(T->raw_count, n);
  const StarFrame F = T->frame;
  if (not_here(T, q, n) || blockIdx.x * (u32)KC_BLOCK >= q) return;
  __syncthreads();
  #pragma unroll
  for (int j = 0; j < PER; ++j) p[j] = k[j] ? P[min(~(u32)k[j], n - 1u)] : make_int2(0, 0);
  #pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int b = t + j * KC_BLOCK;
    if (k[j]) {
      S.cand[b] = p[j];
      S.cid[b] = ~(u32)k[j];
      atomicOr(&S.occ[b >> 5], 1u << (b & 31));
    }
  }
  __syncthreads();
  const u32 step = gridDim.x * (u32)KC_BLOCK;
  for (u32 i0 = blockIdx.x * (u32)KC_BLOCK; i0 < q; i0 += step, i += step) {
    const int2 w1 = i + step < q ? rxy[i + step] : make_int2(0, 0);
    const u32 id1 = i + step < q ? ridx[i + step] : 0u;
    bool keep = false;
    if (i < q) {
      float u, v;
      star::to_uv(F, w.x - F.cx, w.y - F.cy, u, v);
      keep = !star::dropped_by_cands<kStarBins>(S, F, star::bin_of<kStarBins>(u, v), w.x, w.y, id);
    }
    const u32 bal = __ballot_sync(0xFFFFFFFFu, keep);
    u32 base = 0;
    if (lane == 0 && bal) base = atomicAdd(&T->list_count, (u32)__popc(bal));
    base = __shfl_sync(0xFFFFFFFFu, base, 0) + __popc(bal & ((1u << lane) - 1u));
    if (keep && base < kStarCap) { lxy[base] = w; lidx[base] = id; }
    w = w1;
    id = id1;
  }
}

__global__ void __launch_bounds__(KS_BLOCK)
k_star(u32 n, PolyTab* T, const int2* rxy, const u32* ridx, const int2* lxy, const u32* lidx, Plan* plan, int* out,
       long long cap) {
  extern __shared__ __align__(16) unsigned char ks_smem[];
  List& S = *reinterpret_cast<List*>(ks_smem);
  const int t = threadIdx.x;
  pdl_wait();
  const int2 p0 = lxy[t];             // the first entries with the sizes (the slots exist)
  const u32 id0 = lidx[t];
  const u32 q = min(T->raw_count, n), err = T->error;
  const int why = not_here(T, q, n);
  u32 m = T->list_count;
  int h = -1;
  if (why) {
    // One line or one point, if the raw survivors say so; else s = 1 tells the
    // degenerate case from too many points.
    if (why == 1 && q >= 1u && q <= kStarCap && !(err & ERR_RANGE))
      h = star::rest_of_list<KS_BLOCK>(S, rxy, ridx, q, out, cap);
    m = why == 1 ? 1u : 0u;
  } else if (m <= kStarCap && !(err & ERR_RANGE)) {
    for (u32 i = t; i < m; i += KS_BLOCK) {
      S.p[i] = i < (u32)KS_BLOCK ? p0 : lxy[i];
      S.id[i] = i < (u32)KS_BLOCK ? id0 : lidx[i];
      S.ta[i] = (unsigned short)i;
    }
    const StarFrame F = T->frame;
    __syncthreads();
    h = star::list_hull<KS_BLOCK, KS_CAP, kStarBins>(S, m, F, out, cap);
  }
  if (t == 0) star_summary(plan, n, q, m, h, cap, err);
  // Decided: the table is left clear for the next call.
  if (h >= 0) {
    static_assert(kPolyClearBytes % sizeof(u64) == 0, "whole words");
    u64* w = reinterpret_cast<u64*>(T);
    for (u32 i = t; i < (u32)(kPolyClearBytes / sizeof(u64)); i += KS_BLOCK) w[i] = 0ull;
  }
}

__global__ void __launch_bounds__(KS_BLOCK)
k_small(const int2* __restrict__ P, u32 n, Plan* plan, int* out, long long cap) {
  extern __shared__ __align__(16) unsigned char ks_smem[];
  SmallSmem& S = *reinterpret_cast<SmallSmem*>(ks_smem);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, t = threadIdx.x;
  if (t == 0) { S.count = 0u; S.error = 0u; }
  if (t < kPolyDirs) S.best[t] = 0ull;
  StarFrame F;
  u32 m0 = n;
  bool bad = false, flat = false, dirs = false;
  if (n <= KS_DIRECT) {
    static_assert(KS_DIRECT <= KS_SAMPLES * KS_BLOCK, "the points in registers");
    int2 p[KS_SAMPLES];
    #pragma unroll
    for (int r = 0; r < KS_SAMPLES; ++r) p[r] = r * KS_BLOCK + t < n ? P[r * KS_BLOCK + t] : make_int2(0, 0);
    F = star::make_frame<KS_BLOCK>(P, n, S.frame);
    #pragma unroll
    for (int r = 0; r < KS_SAMPLES; ++r) {
      const u32 i = r * KS_BLOCK + t;
      if (i < n) {
        S.list.p[i] = p[r];
        S.list.id[i] = i;
        bad = bad || star::out_of_range(p[r].x, p[r].y);
      }
    }
  } else {
    // The sample, in runs of four points, also gives the frame.
    constexpr u32 NS = KS_SAMPLES * KS_BLOCK;
    static_assert(NS <= KS_DIRECT && KS_SAMPLES % 4 == 0, "whole runs, a stride of at least their length");
    const u32 stride = n / (NS / 4u);
    int2 p[KS_SAMPLES];
    #pragma unroll
    for (int r = 0; r < KS_SAMPLES; ++r) p[r] = P[star::sample_at(r * KS_BLOCK + t, stride)];
    F = star::frame_of<KS_BLOCK>(p, P[0], S.frame);
    #pragma unroll
    for (int r = 0; r < KS_SAMPLES; ++r) star::offer_sample(F, p[r], r * KS_BLOCK + t, S.best);
    __syncthreads();
    if (t < kPolyDirs) {
      const u32 i = ~(u32)S.best[t];
      S.poly.p[t] = i < NS ? P[star::sample_at(i, stride)] : make_int2(0, 0);
      const u32 h = __ballot_sync(0xFFFFFFFFu, i < NS);
      if (lane == 0) S.poly.has[wid] = h;
    }
    __syncthreads();
    const PolyHead H = star::build_poly<KS_BLOCK>(S.poly, F, S.tab, KS_SLABS);
    dirs = H.ok != 0;
    if (dirs) star::bin_normals<KS_BLOCK, kStarBins>(S.poly, F, S.list.dirs());
    __syncthreads();
    star::ListSink<decltype(S.list)> sink{&S.list, &S.count, (u32)KS_CAP, false};
    star::stream_points<4>(P, n, 0u, (u32)wid, (u32)(KS_BLOCK / 32), H, S.tab, sink, [] {});
    bad = sink.bad;
    flat = !H.ok;
    __syncthreads();
    m0 = S.count;
  }
  if (bad) S.error = ERR_RANGE;
  __syncthreads();
  const u32 err = S.error;
  int h = -1;
  u32 m = m0;
  if (m0 <= (u32)KS_CAP && !err) {
    m = star::filter_list<KS_BLOCK, KS_CAP, kStarBins>(S.list, m0, F, S.key, S.cands, dirs ? S.list.dirs() : nullptr);
    h = star::list_hull<KS_BLOCK, KS_CAP, kStarBins>(S.list, m, F, out, cap);
  }
  if (h < 0 && !err && (flat || m0 <= (u32)KS_CAP)) {
    h = star::rest_hull<KS_BLOCK>(S.list, P, nullptr, n, out, cap);
    m = 0u;                           // not undecided for being too many
  }
  if (t == 0) star_summary(plan, n, 0, m, h, cap, err);
}

}  // namespace

cudaError_t star_configure() {
  cudaError_t e = cudaFuncSetAttribute(k_star, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(List));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallSmem));
  return e;
}

cudaError_t launch_star(const int* xy, u32 n, PolyTab* T, const int2* rxy, const u32* ridx, int2* lxy, u32* lidx,
                        Plan* plan, int* out, long long cap, int num_sms, cudaStream_t st) {
  // A block per 32,768 input points, half the SMs at most: every block
  // gathers all candidates, and two points a thread hide that as well.
  const u32 want = n / (64u * KC_BLOCK) + 1u, most = ((u32)num_sms + 1u) / 2u;
  const cudaError_t e = launch_after(k_cand, dim3(want < most ? want : most), dim3(KC_BLOCK), 0, st,
                                     reinterpret_cast<const int2*>(xy), n, T, rxy, ridx, lxy, lidx);
  if (e != cudaSuccess) return e;
  return launch_after(k_star, dim3(1), dim3(KS_BLOCK), sizeof(List), st, n, T, rxy, ridx, lxy, lidx, plan, out, cap);
}

cudaError_t launch_small(const int* xy, u32 n, Plan* plan, int* out, long long cap, cudaStream_t st) {
  k_small<<<1, KS_BLOCK, sizeof(SmallSmem), st>>>(reinterpret_cast<const int2*>(xy), n, plan, out, cap);
  return cudaGetLastError();
}

}  // namespace gbh
