// The star path for inputs with many points next to the hull (a ring: half
// of its points are raw survivors, one in twenty a vertex): list_hull's
// steps over sectors of the angle, one block each.
//
//   ks_hist, ks_scan, ks_scatter   the raw survivors counted, placed by fine
//            angular bin; consecutive bins form sectors of about SB_T points;
//   ks_sectors   a block per sector: the order inside the bins, then rounds
//            of drops with the sector's two ends kept;
//   ks_rounds    twice: the points left, in cyclic order, cut into chunks of
//            SB_CAP that straddle the previous cuts, the same rounds;
//   ks_verify, ks_out   every consecutive triple of what is left must be a
//            strict left turn about c; then it is the hull (star.cuh), written
//            from its lexicographic minimum on.  Otherwise (a crowded bin,
//            or drops that needed more than three cuts) ERR_RETRY.
// It replaces the bucket sort, second round and chain merges there (0.41 +
// 0.49 of 1.19 ms of a 4M ring).  Every kernel reads its sizes from the
// device, the grids are bounds, and no block waits for another.
#include "hull_internal.cuh"
#include "kernels.h"
#include "star.cuh"

namespace gbh {

namespace {

constexpr int SB_BLOCK = 512;
constexpr int SB_CAP = 2048;             // points of a sector or chunk
constexpr u32 SB_T = SB_CAP - star::kBinMax;   // a sector starts at the first bin at or past every multiple of it
constexpr int SB_BIN_BITS = 16;
constexpr int SB_BINS = 1 << SB_BIN_BITS;
constexpr int SB_MAX = 3584;             // most sectors
constexpr int SB_VBLOCKS = 512;          // most blocks of ks_verify

struct SectorTab {
  // cleared per call
  u32 error;                             // ks_scan's: a crowded bin, too many sectors
  u32 bad;                               // ks_verify's
  u32 pad[2];
  u32 start[SB_BINS];                    // the bins' counts
  // written before read
  u32 pos[SB_BINS], cur[SB_BINS];        // first positions, next positions of the placement
  u32 first[SB_MAX + 2];                 // first position of every sector, then the number of points
  u32 cnt[3][SB_MAX];                    // points left per sector / chunk after each pass
  u64 pmin[SB_VBLOCKS];                  // ks_verify's blocks: lexicographic minimum and its place
  u32 pidx[SB_VBLOCKS];
};
constexpr size_t kSectorClear = offsetof(SectorTab, pos);

struct PassSmem {
  int2 p[SB_CAP];
  u32 id[SB_CAP];
  unsigned short ta[SB_CAP], tb[SB_CAP];
  u32 ws[2][SB_BLOCK / 32];
};

__device__ __forceinline__ u32 fine_bin(const StarFrame& F, int2 p) {
  float u, v;
  star::to_uv(F, p.x - F.cx, p.y - F.cy, u, v);
  return star::bin_of<SB_BINS>(u, v);
}

// Sectors (and bound of the later passes' chunks) for q points.
__device__ __forceinline__ u32 sectors(u32 q) { return q / SB_T + 1u; }

constexpr int SB_V = 4;                  // points per thread loaded together

__global__ void __launch_bounds__(SB_BLOCK)
ks_hist(const PolyTab* __restrict__ T, const int2* __restrict__ rxy, u32 n, SectorTab* D) {
  const u32 q = min(T->raw_count, n);
  const StarFrame F = T->frame;
  const u32 step = gridDim.x * SB_BLOCK;
  for (u32 i0 = blockIdx.x * SB_BLOCK + threadIdx.x; i0 < q; i0 += SB_V * step) {
    int2 p[SB_V];
    #pragma unroll
    for (int r = 0; r < SB_V; ++r) p[r] = i0 + r * step < q ? rxy[i0 + r * step] : make_int2(0, 0);
    #pragma unroll
    for (int r = 0; r < SB_V; ++r)
      if (i0 + r * step < q) atomicAdd(&D->start[fine_bin(F, p[r])], 1u);
  }
}

constexpr int SC_BLOCK = 1024;
constexpr int SC_GRID = SB_BINS / SC_BLOCK;

// Block b turns the counts of bins [b SC_BLOCK, (b + 1) SC_BLOCK) into first
// positions; it sums the bins before them itself (at most 256 KB from L2), so
// no block waits for another.  (One block scanning all bins took 42 us.)
__global__ void __launch_bounds__(SC_BLOCK)
ks_scan(const PolyTab* __restrict__ T, u32 n, SectorTab* D) {
  __shared__ u32 ws[2][SC_BLOCK / 32];
  const u32 q = min(T->raw_count, n);
  const u32 b = blockIdx.x * (u32)SC_BLOCK + threadIdx.x;
  u32 sum = 0, before, at, tot;
  const uint4* c4 = reinterpret_cast<const uint4*>(D->start);
  #pragma unroll 4
  for (u32 j = threadIdx.x; j < blockIdx.x * (u32)(SC_BLOCK / 4); j += SC_BLOCK) {
    const uint4 v = c4[j];
    sum += v.x + v.y + v.z + v.w;
  }
  star::block_scan<SC_BLOCK>(sum, ws[0], before);
  const u32 c = D->start[b];
  if (c > star::kBinMax || (b == 0 && sectors(q) > (u32)SB_MAX)) atomicOr(&D->error, ERR_RETRY);
  at = before + star::block_scan<SC_BLOCK>(c, ws[1], tot);
  // The next sector starts at the end of the bin that crosses its multiple.
  const u32 e = at + c;
  if (e / SB_T != at / SB_T && e / SB_T <= (u32)SB_MAX) D->first[e / SB_T] = e;
  D->pos[b] = at;
  D->cur[b] = at;
  if (b == 0) {
    D->first[0] = 0u;
    if (sectors(q) <= (u32)SB_MAX) D->first[sectors(q)] = q;
  }
}

__global__ void __launch_bounds__(SB_BLOCK)
ks_scatter(const PolyTab* __restrict__ T, const int2* __restrict__ rxy, const u32* __restrict__ ridx, u32 n,
           SectorTab* D, int2* __restrict__ oxy, u32* __restrict__ oidx) {
  if (D->error) return;
  const u32 q = min(T->raw_count, n);
  const StarFrame F = T->frame;
  const u32 step = gridDim.x * SB_BLOCK;
  for (u32 i0 = blockIdx.x * SB_BLOCK + threadIdx.x; i0 < q; i0 += SB_V * step) {
    int2 p[SB_V];
    u32 id[SB_V], pos[SB_V];
    #pragma unroll
    for (int r = 0; r < SB_V; ++r) {
      const u32 i = i0 + r * step;
      p[r] = i < q ? rxy[i] : make_int2(0, 0);
      id[r] = i < q ? ridx[i] : 0u;
    }
    #pragma unroll
    for (int r = 0; r < SB_V; ++r) pos[r] = i0 + r * step < q ? atomicAdd(&D->cur[fine_bin(F, p[r])], 1u) : q;
    #pragma unroll
    for (int r = 0; r < SB_V; ++r)
      if (pos[r] < q) { oxy[pos[r]] = p[r]; oidx[pos[r]] = id[r]; }
  }
}

// The entries cur[0, m) of S to (oxy, oidx)[0, m).
__device__ __forceinline__ void write_left(const PassSmem& S, const unsigned short* cur, u32 m, int2* oxy, u32* oidx) {
  for (u32 i = threadIdx.x; i < m; i += SB_BLOCK) {
    const u32 k = cur[i];
    oxy[i] = S.p[k];
    oidx[i] = S.id[k];
  }
}

// In place: a sector's points come back at its first position.
__global__ void __launch_bounds__(SB_BLOCK, 3)
ks_sectors(const PolyTab* __restrict__ T, u32 n, SectorTab* D, int2* xy, u32* idx) {
  __shared__ PassSmem S;
  if (D->error) return;
  const u32 q = min(T->raw_count, n);
  const u32 s = blockIdx.x;
  if (s >= sectors(q)) return;
  const u32 base = D->first[s], end = D->first[s + 1];
  const u32 m = min(end - base, (u32)SB_CAP);
  const StarFrame F = T->frame;
  for (u32 i = threadIdx.x; i < m; i += SB_BLOCK) {
    S.p[i] = xy[base + i];
    S.id[i] = idx[base + i];
    S.ta[i] = S.tb[i] = (unsigned short)i;
  }
  __syncthreads();
  for (u32 i = threadIdx.x; i < m; i += SB_BLOCK) {
    const u32 b = fine_bin(F, S.p[i]);
    const u32 s0 = max(D->pos[b], base) - base;
    const u32 e0 = min(min(b + 1u < (u32)SB_BINS ? D->pos[b + 1u] : q, end) - base, m);
    bool dead;
    const u32 r = star::bin_rank(S.p, S.id, S.tb, s0, e0, i, F, dead);
    S.ta[min(s0 + r, m - 1u)] = (unsigned short)(i | (dead ? 0x8000u : 0u));
  }
  __syncthreads();
  unsigned short* cur = S.ta;
  star::mend_order<SB_BLOCK, true>(S, m, F, cur);
  bool done;
  const u32 left = star::drop_rounds<SB_BLOCK, true>(S, m, F, S.tb, cur, true, done);
  __syncthreads();
  write_left(S, cur, left, xy + base, idx + base);
  if (threadIdx.x == 0) D->cnt[0][s] = left;
}

// Exclusive prefix of cnt[0, ns) in pre[0, ns], the total returned.
__device__ __forceinline__ u32 prefix_counts(const u32* cnt, u32 ns, u32* pre, u32* ws) {
  constexpr int PER = SB_MAX / SB_BLOCK;
  u32 c[PER], sum = 0, tot;
  #pragma unroll
  for (int j = 0; j < PER; ++j) {
    const u32 s = threadIdx.x * PER + j;
    c[j] = s < ns ? cnt[s] : 0u;
    sum += c[j];
  }
  u32 at = star::block_scan<SB_BLOCK>(sum, ws, tot);
  #pragma unroll
  for (int j = 0; j < PER; ++j) {
    const u32 s = threadIdx.x * PER + j;
    if (s < ns) pre[s] = at;
    at += c[j];
  }
  if (threadIdx.x == 0) pre[ns] = tot;
  __syncthreads();
  return tot;
}

// The part (sector or chunk) of the g-th point: the last one whose prefix is at most g.
__device__ __forceinline__ u32 part_of(const u32* pre, u32 ns, u32 g) {
  u32 lo = 0, hi = ns - 1u;
  while (lo < hi) {
    const u32 mid = (lo + hi + 1u) >> 1;
    if (pre[mid] <= g) lo = mid; else hi = mid - 1u;
  }
  return lo;
}

// One pass over the points left by pass `pass` (0: the sectors; later ones:
// chunks of SB_CAP slots), in cyclic order from point SB_CAP / 2 on, chunk c
// to slots c SB_CAP ...
__global__ void __launch_bounds__(SB_BLOCK, 3)
ks_rounds(const PolyTab* __restrict__ T, u32 n, SectorTab* D, int pass, const int2* __restrict__ xy,
          const u32* __restrict__ idx, int2* __restrict__ oxy, u32* __restrict__ oidx) {
  __shared__ PassSmem S;
  __shared__ u32 pre[SB_MAX + 1];
  if (D->error) return;
  const u32 ns = sectors(min(T->raw_count, n));
  if (blockIdx.x >= ns) return;
  const u32 M = prefix_counts(D->cnt[pass], ns, pre, S.ws[0]);
  const u32 c0 = blockIdx.x * (u32)SB_CAP;
  if (c0 >= M) {
    if (threadIdx.x == 0) D->cnt[pass + 1][blockIdx.x] = 0u;
    return;
  }
  const u32 m = min((u32)SB_CAP, M - c0);
  const StarFrame F = T->frame;
  for (u32 i = threadIdx.x; i < m; i += SB_BLOCK) {
    const u32 g = (c0 + i + (u32)SB_CAP / 2u) % M;
    const u32 s = part_of(pre, ns, g);
    const u32 src = (pass == 0 ? D->first[s] : s * (u32)SB_CAP) + (g - pre[s]);
    S.p[i] = xy[src];
    S.id[i] = idx[src];
    S.ta[i] = (unsigned short)i;
  }
  __syncthreads();
  unsigned short* cur = S.ta;
  star::mend_order<SB_BLOCK, true>(S, m, F, cur);
  bool done;
  const u32 left = star::drop_rounds<SB_BLOCK, true>(S, m, F, S.tb, cur, false, done);
  __syncthreads();
  write_left(S, cur, left, oxy + c0, oidx + c0);
  if (threadIdx.x == 0) D->cnt[pass + 1][blockIdx.x] = left;
}

// The points left by the last pass: every triple a strict left turn with c
// strictly left of the edges; each block's lexicographic minimum.
__global__ void __launch_bounds__(SB_BLOCK)
ks_verify(const PolyTab* __restrict__ T, u32 n, SectorTab* D, const int2* __restrict__ xy) {
  __shared__ u32 pre[SB_MAX + 1];
  __shared__ u32 ws[SB_BLOCK / 32];
  __shared__ u64 s_min;
  __shared__ u32 s_idx;
  if (D->error) return;
  const u32 ns = sectors(min(T->raw_count, n));
  if (threadIdx.x == 0) { s_min = ~0ull; s_idx = 0u; }
  const u32 M = prefix_counts(D->cnt[2], ns, pre, ws);
  const StarFrame F = T->frame;
  auto at = [&](u32 g) {
    const u32 s = part_of(pre, ns, g);
    return xy[s * (u32)SB_CAP + (g - pre[s])];
  };
  u64 mn = ~0ull;
  u32 mi = 0;
  bool bad = M < 3u;
  for (u32 g = blockIdx.x * SB_BLOCK + threadIdx.x; g < M; g += gridDim.x * SB_BLOCK) {
    const int2 Q = at(g), A = at(g > 0u ? g - 1u : M - 1u), B = at(g + 1u < M ? g + 1u : 0u);
    const int2 q = make_int2(Q.x - F.cx, Q.y - F.cy), a = make_int2(A.x - F.cx, A.y - F.cy),
               b = make_int2(B.x - F.cx, B.y - F.cy);
    const long long aq = cross2(a.x, a.y, q.x, q.y), qb = cross2(q.x, q.y, b.x, b.y);
    const long long o = cross2(a.x, a.y, b.x, b.y) - aq - qb;
    bad = bad || !(aq > 0 && qb > 0 && o < 0);
    const u64 v = ((u64)((u32)Q.x ^ 0x80000000u) << 32) | (u64)((u32)Q.y ^ 0x80000000u);
    if (v < mn) { mn = v; mi = g; }
  }
  if (mn != ~0ull) atomicMin(&s_min, mn);
  const bool any = __syncthreads_or(bad);
  if (mn != ~0ull && mn == s_min) s_idx = mi;      // one point: they are distinct, or the check fails
  __syncthreads();
  if (threadIdx.x == 0) {
    if (any) D->bad = 1u;
    D->pmin[blockIdx.x] = s_min;
    D->pidx[blockIdx.x] = s_idx;
  }
}

__global__ void __launch_bounds__(SB_BLOCK)
ks_out(const PolyTab* __restrict__ T, u32 n, SectorTab* D, int vblocks, const u32* __restrict__ idx, Plan* plan,
       int* __restrict__ out, long long cap) {
  __shared__ u32 pre[SB_MAX + 1];
  __shared__ u32 ws[SB_BLOCK / 32];
  __shared__ u64 s_min;
  __shared__ u32 s_idx;
  const u32 q = min(T->raw_count, n);
  const bool ok = D->error == 0u && D->bad == 0u;
  u32 M = 0;
  if (ok) {
    if (threadIdx.x == 0) s_min = ~0ull;
    M = prefix_counts(D->cnt[2], sectors(q), pre, ws);
    u64 mn = ~0ull;
    u32 mi = 0;
    for (int v = threadIdx.x; v < vblocks; v += SB_BLOCK)
      if (D->pmin[v] < mn) { mn = D->pmin[v]; mi = D->pidx[v]; }
    if (mn != ~0ull) atomicMin(&s_min, mn);
    __syncthreads();
    if (mn != ~0ull && mn == s_min) s_idx = mi;
    __syncthreads();
    if ((long long)M <= cap) {
      const u32 ns = sectors(q), st = s_idx;
      for (u32 g = blockIdx.x * SB_BLOCK + threadIdx.x; g < M; g += gridDim.x * SB_BLOCK) {
        const u32 s = part_of(pre, ns, g);
        out[g >= st ? g - st : g + M - st] = (int)idx[s * (u32)SB_CAP + (g - pre[s])];
      }
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) star_summary(plan, n, q, M, ok ? (int)M : -1, cap, T->error);
}

}  // namespace

size_t sector_bytes() { return sizeof(SectorTab); }
u32 sector_max_points() { return (u32)(SB_MAX - 1) * SB_T; }

cudaError_t launch_sectors(u32 n, u32 bound, PolyTab* T, void* tab, int2* axy, u32* aidx, int2* bxy, u32* bidx,
                           Plan* plan, int* out, long long cap, int num_sms, cudaStream_t st) {
  SectorTab* D = reinterpret_cast<SectorTab*>(tab);
  const u32 ns = bound / SB_T + 1u;
  const u32 want = (bound + SB_BLOCK * SB_V - 1) / (SB_BLOCK * SB_V), most = (u32)num_sms * 4u;
  const u32 flat = want < 1u ? 1u : (want < most ? want : most);
  u32 vb = (bound + SB_BLOCK - 1) / SB_BLOCK;
  vb = vb < 1u ? 1u : (vb < (u32)num_sms ? vb : (u32)num_sms);
  if (vb > (u32)SB_VBLOCKS) vb = (u32)SB_VBLOCKS;
  cudaError_t e = cudaMemsetAsync(D, 0, kSectorClear, st);
  if (e != cudaSuccess) return e;
  ks_hist<<<flat, SB_BLOCK, 0, st>>>(T, axy, n, D);
  ks_scan<<<SC_GRID, SC_BLOCK, 0, st>>>(T, n, D);
  ks_scatter<<<flat, SB_BLOCK, 0, st>>>(T, axy, aidx, n, D, bxy, bidx);
  ks_sectors<<<ns, SB_BLOCK, 0, st>>>(T, n, D, bxy, bidx);
  ks_rounds<<<ns, SB_BLOCK, 0, st>>>(T, n, D, 0, bxy, bidx, axy, aidx);
  ks_rounds<<<ns, SB_BLOCK, 0, st>>>(T, n, D, 1, axy, aidx, bxy, bidx);
  ks_verify<<<vb, SB_BLOCK, 0, st>>>(T, n, D, bxy);
  ks_out<<<vb, SB_BLOCK, 0, st>>>(T, n, D, (int)vb, bidx, plan, out, cap);
  return cudaGetLastError();
}

}  // namespace gbh
