// The star path (star.cuh) over a batch of instances.
//
// Small instances (up to BS_SMALL points): one block does the whole hull,
// several blocks per SM (kb_small).  Large ones: a block per instance builds
// its frame and sample polygon (kb_poly), one flat pass streams all their
// points, every block an equal share of the tiles (kb_stream), and a block
// per instance finishes its raw survivors (kb_finish).  Every point is read
// once; what the two-pass segmented path and the one-block pipeline spent
// went into reading the points twice, the witness tables and the sorts of
// some 1-4 % of them.  Instances that the star path does not decide are
// listed for the general path (k_batch and the segmented passes).
#include "hull_internal.cuh"
#include "kernels.h"
#include "star.cuh"

namespace gbh {

namespace {

constexpr int BF_NB = 512;            // angular bins of an instance
constexpr int BF_CAP = 2048;          // most points that a block finishes
constexpr u32 BF_SLABS = 1024;
constexpr u32 BF_TILE = 16384;        // points per tile of the flat pass

struct BRec {
  StarFrame frame;
  PolyHead head;
  PolyLine line;
  u32 raw_count, pad;
  u64 key[BF_NB];
  u32 tab[BF_SLABS];
  float2 nrm[BF_NB];
};

// More raw survivors than this: not for one block.
__device__ __forceinline__ u32 many(u32 n) { return max(16384u, n / 4u); }

// ---- small instances
constexpr int BS_BLOCK = 256;
constexpr u32 BS_SLABS = 512;
constexpr u32 BS_DIRECT = 1024;       // up to this many points go to the list whole
constexpr int BS_SAMPLES = 4;         // samples per thread

struct SmallSmem {
  star::ListSmem<BS_BLOCK, BF_CAP, BF_NB> list;
  union {
    struct {
      u64 key[BF_NB];
      star::CandTab<BF_NB> cands;
    };
    u32 tab[BS_SLABS];
  };
  star::FrameSmem<BS_BLOCK> frame;
  star::PolySmem poly;
  u64 best[kPolyDirs];
  u32 count, bad;
  int inst;
};

// One instance's outcome (one thread).
__device__ __forceinline__ void put_result(const BatchStar& a, int inst, int h, bool bad) {
  a.hcount[inst] = h > 0 ? (u32)h : 0u;
  if (bad) atomicOr(a.error, ERR_RANGE);
  else if (h < 0) a.redo[atomicAdd(a.nredo, 1u)] = inst;
}

__global__ void __launch_bounds__(BS_BLOCK, 4)
kb_small(BatchStar a) {
  extern __shared__ __align__(16) unsigned char bs_smem[];
  SmallSmem& S = *reinterpret_cast<SmallSmem*>(bs_smem);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, t = threadIdx.x;
  for (;;) {
    if (t == 0) {
      const u32 q = atomicAdd(a.queue, 1u);
      S.inst = q < (u32)a.ns ? a.order[a.nh + q] : -1;
      S.count = 0u; S.bad = 0u;
    }
    if (t < kPolyDirs) S.best[t] = 0ull;
    __syncthreads();
    const int inst = S.inst;
    if (inst < 0) break;
    const long long off = a.offsets[inst];
    const u32 n = (u32)(a.offsets[inst + 1] - off);
    const int2* P = reinterpret_cast<const int2*>(a.xy) + off;
    int* out = a.out_tmp + a.slot0[inst];
    if (n == 0) {
      if (t == 0) put_result(a, inst, 0, false);
      __syncthreads();
      continue;
    }
    StarFrame F;
    u32 m0 = n;
    bool bad = false, flat = false, dirs = false;
    if (n <= BS_DIRECT) {
      static_assert(BS_DIRECT <= BS_SAMPLES * BS_BLOCK, "the points in registers");
      int2 p[BS_SAMPLES];
      #pragma unroll
      for (int r = 0; r < BS_SAMPLES; ++r) p[r] = r * BS_BLOCK + t < n ? P[r * BS_BLOCK + t] : make_int2(0, 0);
      F = star::make_frame<BS_BLOCK>(P, n, S.frame);
      #pragma unroll
      for (int r = 0; r < BS_SAMPLES; ++r) {
        const u32 i = r * BS_BLOCK + t;
        if (i < n) {
          S.list.p[i] = p[r];
          S.list.id[i] = i;
          bad = bad || star::out_of_range(p[r].x, p[r].y);
        }
      }
    } else {
      // The sample, in runs of four points, also gives the frame.
      constexpr u32 NS = BS_SAMPLES * BS_BLOCK;
      static_assert(NS <= BS_DIRECT && BS_SAMPLES % 4 == 0, "whole runs, a stride of at least their length");
      const u32 stride = n / (NS / 4u);
      int2 p[BS_SAMPLES];
      #pragma unroll
      for (int r = 0; r < BS_SAMPLES; ++r) p[r] = P[star::sample_at(r * BS_BLOCK + t, stride)];
      F = star::frame_of<BS_BLOCK>(p, P[0], S.frame);
      #pragma unroll
      for (int r = 0; r < BS_SAMPLES; ++r) star::offer_sample(F, p[r], r * BS_BLOCK + t, S.best);
      __syncthreads();
      if (t < kPolyDirs) {
        const u32 i = ~(u32)S.best[t];
        S.poly.p[t] = i < NS ? P[star::sample_at(i, stride)] : make_int2(0, 0);
        const u32 h = __ballot_sync(0xFFFFFFFFu, i < NS);
        if (lane == 0) S.poly.has[wid] = h;
      }
      __syncthreads();
      const PolyHead H = star::build_poly<BS_BLOCK>(S.poly, F, S.tab, BS_SLABS);
      dirs = H.ok != 0;
      if (dirs) star::bin_normals<BS_BLOCK, BF_NB>(S.poly, F, S.list.dirs());
      __syncthreads();
      star::ListSink<decltype(S.list)> sink{&S.list, &S.count, (u32)BF_CAP, false};
      star::stream_points<4>(P, n, 0u, (u32)wid, (u32)(BS_BLOCK / 32), H, S.tab, sink, [] {});
      bad = sink.bad;
      flat = !H.ok;
      __syncthreads();
      m0 = S.count;
    }
    if (bad) S.bad = 1u;
    __syncthreads();
    const bool err = S.bad != 0u;
    int h = -1;
    if (m0 <= (u32)BF_CAP && !err) {
      const u32 m = star::filter_list<BS_BLOCK, BF_CAP, BF_NB>(S.list, m0, F, S.key, S.cands, dirs ? S.list.dirs() : nullptr);
      h = star::list_hull<BS_BLOCK, BF_CAP, BF_NB>(S.list, m, F, out, n);
    }
    if (h < 0 && !err && (flat || m0 <= (u32)BF_CAP)) h = star::rest_hull<BS_BLOCK>(S.list, P, nullptr, n, out, n);
    if (t == 0) put_result(a, inst, err ? 0 : h, err);
    __syncthreads();
  }
}

// ---- large instances
constexpr int BP_BLOCK = 512;
constexpr int BP_ITEMS = 2;           // samples per thread loaded together

struct PolyBlockSmem {
  star::FrameSmem<BP_BLOCK> frame;
  star::PolySmem poly;
  u64 best[kPolyDirs];
};

// Sample: n / 32 points (1,024 to 16,384) in runs of four: 6 % of the
// input's DRAM granules, and 1-2 % of a disk's points left outside the
// polygon.
__global__ void __launch_bounds__(BP_BLOCK)
kb_poly(BatchStar a) {
  __shared__ PolyBlockSmem S;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, t = threadIdx.x;
  const int inst = a.order[blockIdx.x];
  BRec& R = reinterpret_cast<BRec*>(a.rec)[blockIdx.x];
  const long long off = a.offsets[inst];
  const u32 n = (u32)(a.offsets[inst + 1] - off);
  const int2* P = reinterpret_cast<const int2*>(a.xy) + off;
  for (int b = t; b < BF_NB; b += BP_BLOCK) R.key[b] = 0ull;
  if (t == 0) R.raw_count = 0u;
  if (t < kPolyDirs) S.best[t] = 0ull;
  const u32 ns = min(max(n / 32u, 1024u), 16384u) & ~3u, stride = n / (ns / 4u);
  // The first round's points also give the frame (points past the sample
  // repeat its last one).
  int2 p[BP_ITEMS];
  #pragma unroll
  for (int r = 0; r < BP_ITEMS; ++r) p[r] = P[star::sample_at(min(t + r * BP_BLOCK, ns - 1u), stride)];
  const StarFrame F = star::frame_of<BP_BLOCK>(p, P[0], S.frame);
  for (u32 i0 = t; i0 < ns; i0 += BP_ITEMS * BP_BLOCK) {
    int2 q[BP_ITEMS];
    #pragma unroll
    for (int r = 0; r < BP_ITEMS; ++r) {
      const u32 i = i0 + (BP_ITEMS + r) * BP_BLOCK;
      q[r] = i < ns ? P[star::sample_at(i, stride)] : make_int2(0, 0);
    }
    #pragma unroll
    for (int r = 0; r < BP_ITEMS; ++r) {
      if (i0 + r * BP_BLOCK < ns) star::offer_sample(F, p[r], i0 + r * BP_BLOCK, S.best);
      p[r] = q[r];
    }
  }
  __syncthreads();
  if (t < kPolyDirs) {
    const u32 i = ~(u32)S.best[t];
    S.poly.p[t] = i < ns ? P[star::sample_at(i, stride)] : make_int2(0, 0);
    const u32 h = __ballot_sync(0xFFFFFFFFu, i < ns);
    if (lane == 0) S.poly.has[wid] = h;
  }
  __syncthreads();
  const PolyHead H = star::build_poly<BP_BLOCK>(S.poly, F, R.tab, BF_SLABS);
  if (H.ok) star::bin_normals<BP_BLOCK, BF_NB>(S.poly, F, R.nrm);
  if (t == 0) { R.frame = F; R.head = H; R.line = S.poly.line; }
}

constexpr int BT_BLOCK = 128;
constexpr int BT_WARPS = BT_BLOCK / 32;
constexpr int BT_SLICE = 256;         // staged points per warp: at least a chunk
constexpr int BT_CH = 256;            // points per chunk
constexpr int BT_STAGES = 4;          // chunks in flight per warp

struct StreamSmem {
  int4 ring[BT_WARPS][BT_STAGES][BT_CH / 2];
  u64 bar[BT_WARPS][BT_STAGES];
  int2 sxy[BT_WARPS][BT_SLICE];
  u32 sidx[BT_WARPS][BT_SLICE];
  u32 tab[BF_SLABS];
};

// Four warps a block, each with its ring, four blocks an SM: the reads of an
// instance's record at the start of a run overlap the other blocks' streams
// (one block of sixteen warps took 75 us instead of 44 for 1,024 instances of
// 19,531 points, where a run has five chunks a warp).  With a ballot per
// point slot the pass over 232M points of 2,095 instances took 485 us, with
// the survivors pushed lane by lane 359 (5.2 TB/s).
// Block b of G streams its share of the T tiles, [b T / G, (b + 1) T / G), in
// runs of one instance each, raw survivors to the instance's second key / index scratch.
__global__ void __launch_bounds__(BT_BLOCK, 4)
kb_stream(BatchStar a) {
  extern __shared__ __align__(128) unsigned char bt_smem[];
  StreamSmem& S = *reinterpret_cast<StreamSmem*>(bt_smem);
  const int wid = threadIdx.x >> 5;
  const int t1 = (int)(((long long)(blockIdx.x + 1) * a.ntiles) / gridDim.x);
  int t = (int)(((long long)blockIdx.x * a.ntiles) / gridDim.x);
  star::Ring<BT_STAGES, BT_CH> ring{&S.ring[wid][0][0], S.bar[wid], 0u, true};
  ring.init();
  int lo = 0, hi = a.nh - 1;          // the last instance whose first tile is at most t
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a.tfirst[mid] <= t) lo = mid; else hi = mid - 1;
  }
  for (; t < t1; ++lo) {
    const int tf = a.tfirst[lo], te = min(t1, a.tfirst[lo + 1]);
    const int inst = a.order[lo];
    const long long off = a.offsets[inst];
    const u32 n = (u32)(a.offsets[inst + 1] - off);
    const long long sl = a.slot0[inst];
    BRec& R = reinterpret_cast<BRec*>(a.rec)[lo];
    const u32 p0 = (u32)(t - tf) * BF_TILE, p1 = min(n, (u32)(te - tf) * BF_TILE);
    PolyHead H;
    star::RawSink<BF_NB, BT_SLICE> sink{S.sxy[wid], S.sidx[wid], 0u, &R.frame, &R.raw_count, a.error, R.key, R.nrm,
                                        reinterpret_cast<int2*>(a.kb + sl), a.ib + sl, n, many(n), 0u,
                                        reinterpret_cast<const int2*>(a.xy) + off};
    star::stream_ring(ring, reinterpret_cast<const int2*>(a.xy) + off + p0, p1 - p0, p0, (u32)wid, (u32)BT_WARPS, H,
                      &R.line, S.tab, sink, a.error, a.spin_limit, [&] {
      H = R.head;
      for (u32 q = threadIdx.x; q < H.nslab; q += BT_BLOCK) S.tab[q] = R.tab[q];
      __syncthreads();
    }, [] {});                        // kb_finish takes such an instance whole
    if (sink.fill) sink.flush();
    __syncthreads();                  // the table is replaced by the next run's
    t = te;
  }
}

constexpr int BE_BLOCK = 256;

// An instance whose sample lies on the line L, from its points (the whole
// block; out of line, so that kb_finish keeps its registers): 1 or 2 vertices
// when every point lies on it, -1 when one does not, -2 for a coordinate out
// of range.  One block reads it: 100,000 points in about 10 us, where the
// general path took 2,800 us for 64 such instances.  (Done by kb_stream's warps
// it cost that kernel registers and the batch of 4,096 instances 1.5 %.)
__device__ __noinline__ int line_instance(const PolyLine* line, const int2* __restrict__ P, u32 n, int* out) {
  __shared__ u64 s_lo, s_hi;
  __shared__ u32 s_il, s_ih;
  const int t = threadIdx.x;
  const PolyLine L = *line;
  if (t == 0) { s_lo = ~0ull; s_hi = 0ull; s_il = s_ih = 0xFFFFFFFFu; }
  __syncthreads();
  u64 lo = ~0ull, hi = 0ull;
  u32 il = 0xFFFFFFFFu, ih = 0xFFFFFFFFu;         // a thread's indices increase: the first of equal points
  bool off = false, bad = false;
  constexpr u32 V = 4;
  for (u32 i0 = t; i0 < n; i0 += V * BE_BLOCK) {
    int2 p[V];
    #pragma unroll
    for (u32 r = 0; r < V; ++r) p[r] = P[min(i0 + r * BE_BLOCK, n - 1u)];
    #pragma unroll
    for (u32 r = 0; r < V; ++r) {
      const u32 i = min(i0 + r * BE_BLOCK, n - 1u);
      const u64 v = star::lex_key(p[r]);
      bad = bad || star::out_of_range(p[r].x, p[r].y);
      off = off || !star::on_line(L, p[r]);
      if (v < lo) { lo = v; il = i; }
      if (ih == 0xFFFFFFFFu || v > hi) { hi = v; ih = i; }
    }
  }
  if (il != 0xFFFFFFFFu) { atomicMin(&s_lo, lo); atomicMax(&s_hi, hi); }
  const bool any_bad = __syncthreads_or(bad), any_off = __syncthreads_or(off);
  if (any_bad || any_off) return any_bad ? -2 : -1;
  if (il != 0xFFFFFFFFu && lo == s_lo) atomicMin(&s_il, il);
  if (ih != 0xFFFFFFFFu && hi == s_hi) atomicMin(&s_ih, ih);
  __syncthreads();
  const int h = s_lo == s_hi ? 1 : 2;
  if (t == 0) { out[0] = (int)s_il; if (h == 2) out[1] = (int)s_ih; }
  return h;
}

struct FinishSmem {
  star::ListSmem<BE_BLOCK, BF_CAP, BF_NB> list;
  star::CandTab<BF_NB> cands;
  u32 count;
};

__global__ void __launch_bounds__(BE_BLOCK, 4)
kb_finish(BatchStar a) {
  extern __shared__ __align__(16) unsigned char be_smem[];
  FinishSmem& S = *reinterpret_cast<FinishSmem*>(be_smem);
  const int lane = threadIdx.x & 31, t = threadIdx.x;
  const int inst = a.order[blockIdx.x];
  const BRec& R = reinterpret_cast<const BRec*>(a.rec)[blockIdx.x];
  const long long off = a.offsets[inst];
  const u32 n = (u32)(a.offsets[inst + 1] - off);
  const long long sl = a.slot0[inst];
  const int2* P = reinterpret_cast<const int2*>(a.xy) + off;
  const int2* rxy = reinterpret_cast<const int2*>(a.kb + sl);
  const u32* ridx = a.ib + sl;
  const u32 q = min(R.raw_count, n);
  if (!R.head.ok && R.line.ok) {
    const int h = line_instance(&R.line, P, n, a.out_tmp + sl);
    if (t == 0) put_result(a, inst, h == -2 ? 0 : h, h == -2);
    return;
  }
  // Most points next to the hull: not for one block.
  if (q > many(n) || q == 0u) {
    if (t == 0) put_result(a, inst, -1, false);
    return;
  }
  if (t < BF_NB / 32) S.cands.occ[t] = 0u;
  if (t == 0) S.count = 0u;
  __syncthreads();
  for (int b = t; b < BF_NB; b += BE_BLOCK) {
    const u64 k = R.key[b];
    if (k) {
      const u32 id = min(~(u32)k, n - 1u);
      S.cands.cand[b] = P[id];
      S.cands.cid[b] = id;
      atomicOr(&S.cands.occ[b >> 5], 1u << (b & 31));
    }
  }
  const StarFrame F = R.frame;
  __syncthreads();
  constexpr int V = 4;                // points per thread loaded together
  for (u32 i0 = 0; i0 < q; i0 += V * BE_BLOCK) {
    int2 p[V];
    u32 id[V];
    #pragma unroll
    for (int r = 0; r < V; ++r) {
      const u32 i = i0 + r * BE_BLOCK + t;
      p[r] = i < q ? rxy[i] : make_int2(0, 0);
      id[r] = i < q ? ridx[i] : 0u;
    }
    #pragma unroll
    for (int r = 0; r < V; ++r) {
      bool keep = false;
      if (i0 + r * BE_BLOCK + t < q) {
        float u, v;
        star::to_uv(F, p[r].x - F.cx, p[r].y - F.cy, u, v);
        keep = !star::dropped_by_cands<BF_NB>(S.cands, F, star::bin_of<BF_NB>(u, v), p[r].x, p[r].y, id[r]);
      }
      const u32 bal = __ballot_sync(0xFFFFFFFFu, keep);
      if (bal) {
        u32 base = 0;
        if (lane == 0) base = atomicAdd(&S.count, (u32)__popc(bal));
        base = __shfl_sync(0xFFFFFFFFu, base, 0) + __popc(bal & ((1u << lane) - 1u));
        if (keep && base < (u32)BF_CAP) {
          S.list.p[base] = p[r];
          S.list.id[base] = id[r];
          S.list.ta[base] = (unsigned short)base;
        }
      }
    }
  }
  __syncthreads();
  const u32 m = S.count;
  int h = -1;
  if (m <= (u32)BF_CAP) h = star::list_hull<BE_BLOCK, BF_CAP, BF_NB>(S.list, m, F, a.out_tmp + sl, n);
  if (t == 0) put_result(a, inst, h, false);
}

}  // namespace

int batch_star_tile() { return (int)BF_TILE; }
size_t batch_star_rec_bytes() { return sizeof(BRec); }

cudaError_t batch_star_configure() {
  cudaError_t e = cudaFuncSetAttribute(kb_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallSmem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kb_stream, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(StreamSmem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kb_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FinishSmem));
  return e;
}

cudaError_t launch_batch_star_small(const BatchStar& a, int num_sms, cudaStream_t st) {
  if (a.ns <= 0) return cudaSuccess;
  const int cap = num_sms * 4;
  kb_small<<<a.ns < cap ? a.ns : cap, BS_BLOCK, sizeof(SmallSmem), st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_batch_star_large(const BatchStar& a, int num_sms, cudaStream_t st) {
  if (a.nh <= 0) return cudaSuccess;
  kb_poly<<<a.nh, BP_BLOCK, 0, st>>>(a);
  const int cap = num_sms * (512 / BT_BLOCK);
  kb_stream<<<a.ntiles < cap ? a.ntiles : cap, BT_BLOCK, sizeof(StreamSmem), st>>>(a);
  kb_finish<<<a.nh, BE_BLOCK, sizeof(FinishSmem), st>>>(a);
  return cudaGetLastError();
}

}  // namespace gbh
