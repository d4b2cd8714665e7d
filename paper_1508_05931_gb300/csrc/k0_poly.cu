// K0 of the single-read front: the frame and the sample polygon.
//
// Per angular sector of the whitened plane the sample point of the largest
// radius is a candidate.  The candidates are input points, so the convex
// polygon that they reduce to is spanned by input points: a point strictly
// inside it is strictly inside the hull of the input and is no vertex of it
// (the argument of Section 2.2.2 for any filter polygon whose corners are
// input points).  The float sectors and radii only choose the corners; the
// polygon and the table built from it are exact.  The last block builds both
// (star::build_poly).
//
// Sample: about n / 128 points (at least 4,096) in runs of four, one per
// thread and round: a 20M disk keeps 0.3 % of its points against 0.64 % for
// 32 directions of n / 1,024 points (the area outside a regular 32-gon
// alone), for 2.5 MB read.
#include "hull_internal.cuh"
#include "kernels.h"
#include "star.cuh"

namespace gbh {

namespace {

constexpr int K0_BLOCK = 512;

struct K0Smem {
  star::FrameSmem<K0_BLOCK> frame;
  u64 best[kPolyDirs];
  star::PolySmem poly;
  u32 tab[kPolySlabs + kPolySlabs / 32];
  bool last;
};

__global__ void __launch_bounds__(K0_BLOCK)
k0_poly(const int2* __restrict__ P, u32 n, u32 ns, u32 slabs, PolyTab* __restrict__ T) {
  __shared__ K0Smem S;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, t = threadIdx.x;
  const u32 stride = n / (ns / 4u), step = gridDim.x * K0_BLOCK;
  u32 i = blockIdx.x * K0_BLOCK + t;
  int2 p = i < ns ? P[star::sample_at(i, stride)] : make_int2(0, 0);
  if (t < kPolyDirs) S.best[t] = 0ull;
  const StarFrame F = star::make_frame<K0_BLOCK>(P, n, S.frame);    // its barriers publish S.best
  while (i < ns) {
    const u32 i1 = i + step;
    const int2 p1 = i1 < ns ? P[star::sample_at(i1, stride)] : make_int2(0, 0);
    star::offer_sample(F, p, i, S.best);
    p = p1;
    i = i1;
  }
  pdl_launch();
  __syncthreads();
  // The threads that update T->best order their updates before the block's
  // arrival; those of the last block order the arrivals before their reads.
  if (t < kPolyDirs) {
    if (S.best[t]) atomicMax(&T->best[t], S.best[t]);
    __threadfence();
  }
  __syncthreads();
  if (t == 0) S.last = atomicAdd(&T->done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!S.last) return;
  if (t < kPolyDirs) {
    __threadfence();
    const u64 v = *reinterpret_cast<volatile u64*>(&T->best[t]);
    S.poly.p[t] = v ? P[star::sample_at(~(u32)v, stride)] : make_int2(0, 0);
    const u32 h = __ballot_sync(0xFFFFFFFFu, v != 0ull);
    if (lane == 0) S.poly.has[wid] = h;
  }
  __syncthreads();
  // The table through shared memory: written by runs straight to T, every
  // store of a warp touched 32 sectors (11,000 cycles for 8,192 slabs).
  const PolyHead H = star::build_poly<K0_BLOCK, true>(S.poly, F, S.tab, slabs);
  if (H.ok) star::bin_normals<K0_BLOCK, kStarBins>(S.poly, F, T->nrm);
  __syncthreads();
  for (u32 s = t; s < H.nslab; s += K0_BLOCK) T->tab[s] = S.tab[star::pad_slab(s)];
  if (t == 0) {
    T->frame = F;
    T->head = H;
    T->line = S.poly.line;
  }
}

}  // namespace

cudaError_t launch_poly(const int* xy, u32 n, PolyTab* T, int num_sms, cudaStream_t st) {
  u32 ns = n / 128u;
  if (ns < 4096u) ns = 4096u;
  if (ns > n) ns = n;
  ns &= ~3u;                          // whole runs; n is above 4,096
  u32 grid = (ns + K0_BLOCK - 1) / K0_BLOCK;
  if (grid > (u32)num_sms) grid = (u32)num_sms;
  // Slabs: the staircase left outside takes about one slab's width of every
  // column, so a large input wants narrow slabs, while every K1 block of a
  // small one reads the whole table for a few points.
  const u32 slabs = n < (1u << 21) ? 2048u : (u32)kPolySlabs;
  k0_poly<<<grid, K0_BLOCK, 0, st>>>(reinterpret_cast<const int2*>(xy), n, ns, slabs, T);
  return cudaGetLastError();
}

}  // namespace gbh
