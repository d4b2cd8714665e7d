// The star path: the hull of the points that survive a sample polygon,
// found in angular order around an interior point c (Section 2.1
// steps 3-8 with the pivot moved inside: distance and angle about c, the
// sort by angle, and the scan that pops non-left turns, run as rounds in
// which every point looks at its neighbours).
//
// A frame holds c and a linear map that whitens the sample's covariance, so
// that elongated sets spread evenly over the angular bins.  The map, the
// bins and the choice of candidates are float and only steer; every
// decision to drop a point is exact in 64-bit integers:
//   a point q inside the closed triangle (c, a, b) of three input points
//   with cross(a - c, b - c) > 0, not on the side a b, is no hull vertex; on
//   the open segment a b neither; equal to a or b it is the duplicate with
//   the larger index.  (This takes c strictly inside the hull, which the
//   verification below proves before any result is used.)
// The drops of a round may use points that the same round drops: those are
// input points too.  The rounds end with a closed list that is verified: every
// consecutive cross product about c positive and every turn strictly left.
// That makes it a convex polygon of input points with c strictly inside, in
// which every other input point was shown to lie, because the list goes round
// c once.  The two local tests alone do not say so (a pentagram passes them);
// the order does: the bins are one sweep of the whitened angle, whose error is
// far below a right angle (frame_of bounds the map), inside a bin points stand
// in exact order, and mend_order exchanges neighbours only.  Each step is
// positive and below a half turn, and the angles follow one sweep, so the
// steps add up to one turn.  A change of the order has to keep that.  Anything
// else (a degenerate set, a crowded bin, too many points or rounds) returns
// failure and the caller takes the general path.
#pragma once

#include "hull_internal.cuh"

namespace gbh {
namespace star {

__device__ __forceinline__ void to_uv(const StarFrame& F, int dx, int dy, float& u, float& v) {
  const float fx = (float)dx, fy = (float)dy;
  u = __fmul_rn(fx, F.m00);
  v = __fmaf_rn(fy, F.m11, __fmul_rn(fx, F.m10));
}

// Angular bin of (u, v): the diamond angle t in [0, 4), monotone in the
// polar angle (up to rounding, which the exact tests absorb).
template <int NB>
__device__ __forceinline__ u32 bin_of(float u, float v) {
  const float t = __fdividef(v, fabsf(u) + fabsf(v));
  const float a = u >= 0.0f ? (v >= 0.0f ? t : 4.0f + t) : 2.0f - t;
  const int b = (int)(a * (float)(NB / 4));      // NaN (the point c itself) converts to 0
  return (u32)min(max(b, 0), NB - 1);
}

// Candidate key of a point: how far it reaches along the bin's direction w,
// then the smaller index (all duplicates of a point share its bin and reach).
// Without a polygon w is the point itself (its radius); with one, the outward
// normal of the polygon's edge that the bin looks at: along a flat side the
// largest radius is at the bin's far end, not nearest the side (a 20M square
// left 5,600 points of 17k that way).
__device__ __forceinline__ u64 cand_key(float2 w, float u, float v, u32 idx) {
  const float r = fmaxf(__fmaf_rn(w.x, u, __fmul_rn(w.y, v)), 0.0f);
  return ((u64)__float_as_uint(r) << 32) | (u64)(~idx);
}

__device__ __forceinline__ bool out_of_range(int x, int y) {
  return (u32)x + (u32)kCoordLimit > 2u * (u32)kCoordLimit || (u32)y + (u32)kCoordLimit > 2u * (u32)kCoordLimit;
}

// (x, y) as one word that orders points lexicographically, and back.
__device__ __forceinline__ u64 lex_key(int2 p) {
  return ((u64)((u32)p.x ^ 0x80000000u) << 32) | (u64)((u32)p.y ^ 0x80000000u);
}
__device__ __forceinline__ int2 lex_point(u64 v) {
  return make_int2((int)((u32)(v >> 32) ^ 0x80000000u), (int)((u32)v ^ 0x80000000u));
}

// p in range and on the line through the extremes of L (their one point when they are equal).
__device__ __forceinline__ bool on_line(const PolyLine& L, int2 p) {
  if (out_of_range(p.x, p.y)) return false;
  if (L.ax == L.bx && L.ay == L.by) return p.x == L.ax && p.y == L.ay;
  return orient(L.ax, L.ay, L.bx, L.by, p.x, p.y) == 0;
}

// q dropped by the triangle (c, a, b); a, b, q relative to c.
// orient(a, b, q) = cross(a, b) - cross(a, q) - cross(q, b): three products
// (each below 2^61, the sum below 2^63).
__device__ __forceinline__ bool dropped_by(int2 a, int2 b, int2 q) {
  const long long ab = cross2(a.x, a.y, b.x, b.y);
  const long long aq = cross2(a.x, a.y, q.x, q.y), qb = cross2(q.x, q.y, b.x, b.y);
  const long long o = ab - aq - qb;
  return ab > 0 && aq >= 0 && qb >= 0 && (o > 0 || (o == 0 && aq > 0 && qb > 0));
}

// Exclusive block scan; `ws` holds BLOCK / 32 words that no warp still reads
// (callers alternate two areas, so one barrier per scan suffices).
template <int BLOCK>
__device__ __forceinline__ u32 block_scan(u32 v, u32* ws, u32& total) {
  constexpr int W = BLOCK / 32;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  u32 inc = v;
  #pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u32 t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) ws[wid] = inc;
  __syncthreads();
  u32 x = lane < W ? ws[lane] : 0u;
  #pragma unroll
  for (int o = 1; o < W; o <<= 1) {
    const u32 t = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += t;
  }
  total = __shfl_sync(0xFFFFFFFFu, x, W - 1);
  const u32 before = __shfl_sync(0xFFFFFFFFu, x, wid > 0 ? wid - 1 : 0);
  return (wid > 0 ? before : 0u) + inc - v;
}

// ---------------------------------------------------------------- frame
// From strided points (V of every thread, relative to one point o of the
// input): c, their mean rounded to integers, and the whitening map of their
// covariance (the inverse Cholesky factor, determinant > 0).  Every block that calls it with the same P and n gets
// the same frame.  Nothing is assumed of c: a polygon of input points that
// verifies about it proves that it lies inside.  The map is bounded whatever
// the sums lost to rounding (o far from a tight rest): |l21| <= sqrt(d) and
// l22 >= 1e-4 sqrt(d) keep |m10| <= 1e4 m00, so a point's v is known to 3e4 x
// 2^-24 |u| (two conversions and a product) and its angle to about 2^-9: a bin
// spans far less than a half turn (bin_rank's order is total) and the bins are
// one sweep of the angle.
template <int BLOCK>
struct FrameSmem {
  float sum[BLOCK / 32][5];
};

template <int BLOCK, int V>
__device__ __forceinline__ StarFrame frame_of(const int2 (&p)[V], int2 o, FrameSmem<BLOCK>& S) {
  constexpr int W = BLOCK / 32;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  float s[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  #pragma unroll
  for (int r = 0; r < V; ++r) {
    const float fx = (float)p[r].x - (float)o.x, fy = (float)p[r].y - (float)o.y;
    s[0] += fx; s[1] += fy; s[2] += fx * fx; s[3] += fx * fy; s[4] += fy * fy;
  }
  #pragma unroll
  for (int k = 0; k < 5; ++k) {
    #pragma unroll
    for (int d = 16; d > 0; d >>= 1) s[k] += __shfl_xor_sync(0xFFFFFFFFu, s[k], d);
    if (lane == 0) S.sum[wid][k] = s[k];
  }
  __syncthreads();
  #pragma unroll
  for (int k = 0; k < 5; ++k) {
    s[k] = lane < W ? S.sum[lane][k] : 0.0f;
    #pragma unroll
    for (int d = 16; d > 0; d >>= 1) s[k] += __shfl_xor_sync(0xFFFFFFFFu, s[k], d);
    s[k] *= 1.0f / (float)(BLOCK * V);
  }
  const float mx = s[0], my = s[1];
  const float a = fmaxf(s[2] - mx * mx, 1.0f), d = fmaxf(s[4] - my * my, 1.0f), b = s[3] - mx * my;
  const float l11 = sqrtf(a), sd = sqrtf(d), l21 = fminf(fmaxf(b / l11, -sd), sd);
  const float l22 = sqrtf(fmaxf(d - l21 * l21, 1.0e-8f * d));
  StarFrame F;
  F.m00 = 1.0f / l11;
  F.m11 = 1.0f / l22;
  F.m10 = -(l21 / l11) / l22;
  // Inside the coordinate range whatever the points hold.
  const float L = (float)kCoordLimit;
  F.cx = (int)rintf(fminf(fmaxf((float)o.x + mx, -L), L));
  F.cy = (int)rintf(fminf(fmaxf((float)o.y + my, -L), L));
  return F;
}

template <int BLOCK>
__device__ __forceinline__ StarFrame make_frame(const int2* __restrict__ P, u32 n, FrameSmem<BLOCK>& S) {
  const int2 p[1] = {P[(u32)(((u64)threadIdx.x * n) / BLOCK)]};
  return frame_of<BLOCK>(p, P[0], S);
}

// ---------------------------------------------------------------- sample polygon
// The sample's candidates: per angular sector (kPolyDirs of them) the point
// of the largest whitened radius (cand_key of the sample's position).  One
// sector per sample: projecting every sample on every direction found the
// same polygon at 30 times the instructions (8,500 cycles of a 1,024-thread
// block for 2,048 samples).
// Sample i of n / stride4 runs of four consecutive points (a run is one
// 32-byte sector: four samples for the traffic of one).
__device__ __forceinline__ size_t sample_at(u32 i, u32 stride4) { return (size_t)(i >> 2) * stride4 + (i & 3u); }

__device__ __forceinline__ void offer_sample(const StarFrame& F, int2 p, u32 pos, u64* best) {
  float u, v;
  to_uv(F, p.x - F.cx, p.y - F.cy, u, v);
  const u64 k = cand_key(make_float2(u, v), u, v, pos);
  u64* slot = &best[bin_of<kPolyDirs>(u, v)];
  if (k > *(volatile u64*)slot) atomicMax(slot, k);
}

struct PolySmem {
  int2 p[kPolyDirs];                    // candidates by sector
  u32 has[2];                           // sectors with one
  int hx[kPolyDirs + 2], hy[kPolyDirs + 2];
  float slope[kPolyDirs + 2];
  int k, ir, ymin, ymax;
  u64 alive;                            // sectors of the polygon's corners
  PolyLine line;
};

// The polygon of the candidates (in angular order about c) and the table of
// its x slabs (see PolyHead).  Whole block; S.p and S.has are written and
// visible; `tab` (shared or global) gets at most `slabs` words.
//
// Warp 0 reduces the candidates to a convex polygon by rounds (the rule of
// list_hull, the alive sectors in one 64-bit mask) and verifies it; a set
// that does not verify gets no polygon (nothing is dropped but, when all
// candidates lie on one line, what lies between points of that line: S.line).
//
// Lower chain: corners 0 .. ir, x non-decreasing; upper chain: corners
// ir .. k (corner k = corner 0), x non-increasing.  The lower chain is
// convex and the upper one concave, so over a slab's columns their extreme
// values lie at its ends; a slab of several columns takes the first column of
// the next one as its end.  An edge's height over its start, p = slope (x -
// x_e), carries at most 6 x 2^-24 of relative error (two conversions and the
// division of the slope, one conversion, two roundings), so with e = |p|
// 2^-21 the chain lies below y_e + floor(p + e) + 1 and above y_e + ceil(p -
// e) - 1: integer heights strictly between floor(p + e) of the lower edge
// and ceil(p - e) of the upper one are strictly inside.  For small
// coordinates that is the exact test.  The heights are stored in 16 bits, in
// units of 2^shy rounded inwards.
// PAD: word s goes to tab[s + s / 32] (a thread's run of slabs then spreads
// over the shared-memory banks).
__device__ __forceinline__ u32 pad_slab(u32 s) { return s + (s >> 5); }

// The line that all candidates lie on, if there is one (warp 0).
static __device__ __noinline__ void line_of_sample(PolySmem& S) {
  const int lane = threadIdx.x & 31;
  const u64 has = ((u64)S.has[1] << 32) | S.has[0];
  u64 mn = ~0ull, mx = 0ull;
  #pragma unroll
  for (int w = 0; w < 2; ++w)
    if ((has >> (lane + 32 * w)) & 1ull) {
      const u64 v = lex_key(S.p[lane + 32 * w]);
      mn = v < mn ? v : mn; mx = v > mx ? v : mx;
    }
  #pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const u64 a = __shfl_xor_sync(0xFFFFFFFFu, mn, o), b = __shfl_xor_sync(0xFFFFFFFFu, mx, o);
    mn = a < mn ? a : mn; mx = b > mx ? b : mx;
  }
  const int2 A = lex_point(mn), B = lex_point(mx);
  PolyLine L{1, A.x, A.y, B.x, B.y};
  bool on = has != 0ull && !out_of_range(A.x, A.y) && !out_of_range(B.x, B.y);
  #pragma unroll
  for (int w = 0; w < 2; ++w)
    if ((has >> (lane + 32 * w)) & 1ull) on = on && on_line(L, S.p[lane + 32 * w]);
  L.ok = __all_sync(0xFFFFFFFFu, on);
  __syncwarp();
  if (lane == 0) S.line = L;
}

template <int BLOCK, bool PAD = false>
__device__ PolyHead build_poly(PolySmem& S, const StarFrame& F, u32* tab, u32 slabs) {
  static_assert(kPolyDirs == 64, "two candidates per lane of a warp, one mask word");
  const int lane = threadIdx.x & 31, t = threadIdx.x;
  PolyHead H;
  H.ok = 0; H.x1 = 0; H.xw = 0; H.sh = 0; H.y0 = 0; H.shy = 0; H.nslab = 0;
  if (t < 32) {
    u64 alive = ((u64)S.has[1] << 32) | S.has[0];
    auto rel = [&](int j) { const int2 p = S.p[j]; return make_int2(p.x - F.cx, p.y - F.cy); };
    bool ok = false;
    for (int round = 0; round < 64 && __popcll(alive) >= 3; ++round) {
      u32 drop[2], bad = 0;
      #pragma unroll
      for (int w = 0; w < 2; ++w) {
        const int j = lane + 32 * w;
        bool d = false;
        if ((alive >> j) & 1ull) {
          const u64 below = alive & ((1ull << j) - 1ull), above = j < 63 ? alive >> (j + 1) << (j + 1) : 0ull;
          const int pj = 63 - __clzll((long long)(below ? below : above));
          const int nj = __ffsll((long long)(above ? above : below)) - 1;
          const int2 a = rel(pj), b = rel(nj), q = rel(j);
          const long long ab = cross2(a.x, a.y, b.x, b.y);
          const long long aq = cross2(a.x, a.y, q.x, q.y), qb = cross2(q.x, q.y, b.x, b.y);
          const long long o = ab - aq - qb;
          d = ab > 0 && aq >= 0 && qb >= 0 && (o > 0 || (o == 0 && aq > 0 && qb > 0));
          bad |= !(aq > 0 && qb > 0 && o < 0) || out_of_range(S.p[j].x, S.p[j].y);
        }
        drop[w] = __ballot_sync(0xFFFFFFFFu, d);
      }
      if (!(drop[0] | drop[1])) {
        ok = !__any_sync(0xFFFFFFFFu, bad != 0u);
        break;
      }
      alive &= ~(((u64)drop[1] << 32) | drop[0]);
    }
    // Corners from the lexicographic minimum on.
    const int k = ok ? __popcll(alive) : 0;
    if (ok) {
      auto lex = [&](int j) { return lex_key(S.p[j]); };
      u64 mn = ~0ull, mx = 0ull;
      int ylo = 0x7FFFFFFF, yhi = (int)0x80000000;
      #pragma unroll
      for (int w = 0; w < 2; ++w) {
        const int j = lane + 32 * w;
        if ((alive >> j) & 1ull) {
          const u64 v = lex(j);
          mn = v < mn ? v : mn; mx = v > mx ? v : mx;
          ylo = min(ylo, S.p[j].y); yhi = max(yhi, S.p[j].y);
        }
      }
      #pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const u64 a = __shfl_xor_sync(0xFFFFFFFFu, mn, o), b = __shfl_xor_sync(0xFFFFFFFFu, mx, o);
        mn = a < mn ? a : mn; mx = b > mx ? b : mx;
      }
      ylo = __reduce_min_sync(0xFFFFFFFFu, ylo);
      yhi = __reduce_max_sync(0xFFFFFFFFu, yhi);
      int r0 = -1, r1 = -1;
      #pragma unroll
      for (int w = 0; w < 2; ++w) {
        const int j = lane + 32 * w;
        if ((alive >> j) & 1ull) {
          const int r = __popcll(alive & ((1ull << j) - 1ull));
          if (lex(j) == mn) r0 = r;
          if (lex(j) == mx) r1 = r;
        }
      }
      r0 = __reduce_max_sync(0xFFFFFFFFu, r0);
      r1 = __reduce_max_sync(0xFFFFFFFFu, r1);
      #pragma unroll
      for (int w = 0; w < 2; ++w) {
        const int j = lane + 32 * w;
        if ((alive >> j) & 1ull) {
          const int r = __popcll(alive & ((1ull << j) - 1ull)) - r0, q = r < 0 ? r + k : r;
          S.hx[q] = S.p[j].x; S.hy[q] = S.p[j].y;
        }
      }
      __syncwarp();
      for (int e = lane; e < k; e += 32) {
        const int en = e + 1 < k ? e + 1 : 0;
        const int dx = S.hx[en] - S.hx[e];
        S.slope[e] = dx != 0 ? (float)(S.hy[en] - S.hy[e]) / (float)dx : 0.0f;    // vertical edges are never active
      }
      if (lane == 0) { S.ir = r1 >= r0 ? r1 - r0 : r1 - r0 + k; S.ymin = ylo; S.ymax = yhi; S.hx[k] = S.hx[0]; }
    }
    if (lane == 0) { S.k = k; S.alive = alive; S.line.ok = 0; }
    if (!ok) line_of_sample(S);
  }
  __syncthreads();
  const int k = S.k;
  if (k < 3) return H;
  const int ir = S.ir, xl = S.hx[0], xr = S.hx[ir], ymin = S.ymin, ymax = S.ymax;
  if (xr - xl < 2 || ymax - ymin < 2) return H;
  H.x1 = xl + 1;
  H.xw = (u32)(xr - xl - 1);          // interior columns x1 .. x1 + xw - 1
  while ((H.xw - 1u) >> H.sh >= slabs) ++H.sh;
  H.nslab = ((H.xw - 1u) >> H.sh) + 1u;
  H.y0 = ymin;
  while ((u32)(ymax - ymin) >> H.shy > 65534u) ++H.shy;
  H.ok = 1;
  // A thread takes a run of slabs: along it the active lower edge le (x(le)
  // < x <= x(le + 1)) only moves forward and the active upper edge ue (x(ue)
  // > x >= x(ue + 1)) only backward.
  const u32 per = (H.nslab + BLOCK - 1) / BLOCK;
  const u32 s0 = t * per, s1 = min(H.nslab, s0 + per);
  if (s0 >= s1) return H;
  auto column = [&](u32 s) { return H.x1 + (int)min(H.xw - 1u, s << H.sh); };
  int le = 0, ue = ir;
  {
    const int x = column(s0);
    for (int hi = ir - 1; le < hi;) {
      const int mid = (le + hi) >> 1;
      if (S.hx[mid + 1] < x) le = mid + 1; else hi = mid;
    }
    for (int hi = k - 1; ue < hi;) {
      const int mid = (ue + hi + 1) >> 1;
      if (S.hx[mid] > x) ue = mid; else hi = mid - 1;
    }
  }
  int lx = S.hx[le], lend = S.hx[le + 1], ly = S.hy[le];
  int ux = S.hx[ue], uy = S.hy[ue];
  float ls = S.slope[le], us = S.slope[ue];
  auto heights = [&](int x, int& lo, int& hi) {
    while (le < ir - 1 && lend < x) { ++le; lx = lend; lend = S.hx[le + 1]; ly = S.hy[le]; ls = S.slope[le]; }
    while (ue > ir && ux <= x) { --ue; ux = S.hx[ue]; uy = S.hy[ue]; us = S.slope[ue]; }
    const float p = __fmul_rn((float)(x - lx), ls), q = __fmul_rn((float)(x - ux), us);
    lo = ly + (int)floorf(fmaf(fabsf(p), 4.76837158e-7f, p));
    hi = uy + (int)ceilf(fmaf(fabsf(q), -4.76837158e-7f, q));
  };
  int lo0, hi0;
  heights(column(s0), lo0, hi0);
  for (u32 s = s0; s < s1; ++s) {
    int lo1 = lo0, hi1 = hi0;
    if (H.sh) heights(column(s + 1), lo1, hi1);      // past the last slab: its own last column
    const int ylo = max(max(lo0, lo1), ymin), yhi = min(min(hi0, hi1), ymax);
    u32 w = 0;
    if (ylo < yhi) {
      const u32 A = ((u32)(ylo - ymin) >> H.shy) + 1u, B = (u32)(yhi - ymin) >> H.shy;
      if (B > A) w = A | ((B - A) << 16);
    }
    tab[PAD ? pad_slab(s) : s] = w;
    if (!H.sh && s + 1 < s1) heights(column(s + 1), lo1, hi1);
    lo0 = lo1; hi0 = hi1;
  }
  return H;
}

// The directions of the bins' candidates (cand_key): the outward normals, in
// the whitened plane, of the edges that the bins' middles look at.  After a
// build_poly that gave a polygon, the whole block.
template <int BLOCK, int NB>
__device__ __forceinline__ void bin_normals(const PolySmem& S, const StarFrame& F, float2* nrm) {
  const u64 alive = S.alive;
  auto before = [&](int j) {            // the last corner's sector below j, cyclically
    const u64 m = alive & ((1ull << j) - 1ull);
    return 63 - __clzll((long long)(m ? m : alive));
  };
  for (int b = threadIdx.x; b < NB; b += BLOCK) {
    const int j = b / (NB / kPolyDirs);
    int ja = j;
    if ((alive >> j) & 1ull) {
      const int2 p = S.p[j];
      float u, v;
      to_uv(F, p.x - F.cx, p.y - F.cy, u, v);
      if ((int)bin_of<NB>(u, v) > b) ja = before(j);
    } else {
      ja = before(j);
    }
    const u64 above = ja < 63 ? alive >> (ja + 1) << (ja + 1) : 0ull;
    const int jb = __ffsll((long long)(above ? above : alive)) - 1;
    const int2 A = S.p[ja], B = S.p[jb];
    float ua, va, ub, vb;
    to_uv(F, A.x - F.cx, A.y - F.cy, ua, va);
    to_uv(F, B.x - F.cx, B.y - F.cy, ub, vb);
    nrm[b] = make_float2(vb - va, ua - ub);
  }
}

// Strictly inside the sample polygon (its table): word w holds the first
// inside height unit (low half) and their number (high half).
__device__ __forceinline__ bool inside_poly(const PolyHead& H, const u32* tab, int x, int y) {
  const u32 xo = (u32)(x - H.x1);
  u32 w = 0;
  if (xo < H.xw) w = tab[xo >> H.sh];
  return ((u32)(y - H.y0) >> H.shy) - (w & 0xFFFFu) < (w >> 16);
}

// ---------------------------------------------------------------- the stream
// Flag in a lane's mask of survivors (which has at most 16 bits): its chunk
// did not come in time.
constexpr u32 kLate = 0x80000000u;

// Where a warp puts the points on or outside the polygon: its slice of
// SLICE staged points, flushed with one atomic reservation into (rxy, ridx),
// in no particular order; every flushed point is offered as the candidate of
// its angular bin.
template <int NB, int SLICE>
struct RawSink {
  int2* sxy;
  u32* sidx;
  u32 fill;                 // uniform over the warp
  const StarFrame* frame;
  u32* raw_count;
  u32* error;
  u64* key;
  const float2* nrm;
  int2* rxy;
  u32* ridx;
  u32 bound;                // capacity of (rxy, ridx)
  u32 many;                 // past this many raw survivors nobody reads the candidates

  u32 last;                 // the raw survivors' number at this warp's last flush
  const int2* pts;          // the input (point of index id)

  // A duplicate of its bin's candidate with a larger index goes no further
  // (4M points of 40 distinct ones would leave a million); any other point
  // is one more load away from it only when it reaches exactly as far.
  __device__ __forceinline__ void flush() {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    u32 keep = 0;
    static_assert(SLICE <= 1024, "a mask bit per round");
    const bool cands = last <= many;
    const StarFrame F = *frame;
    for (u32 r = 0; r * 32u < fill; ++r) {
      const u32 q = lane + 32u * r;
      if (q >= fill) break;
      const int2 p = sxy[q];
      const u32 id = sidx[q];
      bool dup = false;
      if (out_of_range(p.x, p.y)) atomicOr(error, ERR_RANGE);
      if (cands) {
        float u, v;
        to_uv(F, p.x - F.cx, p.y - F.cy, u, v);
        const u32 b = bin_of<NB>(u, v);
        const u64 k = cand_key(__ldcg(&nrm[b]), u, v, id), c = __ldcg(&key[b]);
        if (k > c) {
          atomicMax(&key[b], k);
        } else if ((u32)(k >> 32) == (u32)(c >> 32)) {
          const u32 cid = ~(u32)c;
          const int2 w = pts[cid];
          dup = w.x == p.x && w.y == p.y && id > cid;
        }
      }
      if (!dup) keep |= 1u << r;
    }
    __syncwarp();
    u32 tot = 0;
    for (u32 r = 0; r * 32u < fill; ++r) tot += __popc(__ballot_sync(0xFFFFFFFFu, (keep >> r) & 1u));
    u32 at = 0;
    if (lane == 0) at = atomicAdd(raw_count, tot);
    last = at = __shfl_sync(0xFFFFFFFFu, at, 0);
    for (u32 r = 0; r * 32u < fill; ++r) {
      const u32 bal = __ballot_sync(0xFFFFFFFFu, (keep >> r) & 1u);
      if ((keep >> r) & 1u) {
        const u32 o = at + __popc(bal & ((1u << lane) - 1u));
        if (o < bound) { rxy[o] = sxy[lane + 32u * r]; ridx[o] = sidx[lane + 32u * r]; }
      }
      at += __popc(bal);
    }
    __syncwarp();
    fill = 0;
  }
  // Bit 2 u + v of m: the lane's point at[64 u + v] survives (index id + 64 u
  // + v); the whole warp calls it, at most SLICE points in all.  A scan over
  // the lanes and a loop over each one's few points: a ballot per slot cost
  // as much as the tests themselves where one point in fifty survives.  A lane
  // with kLate set in m: nothing is pushed and all lanes get false (its vote
  // rides on the scan: a vote of its own took 1 % of the batched pass).
  __device__ __forceinline__ bool push_lanes(u32 m, const int2* at, u32 id) {
    const int lane = threadIdx.x & 31;
    const u32 c = __popc(m & ~kLate) + (m >> 31 << 16);
    u32 inc = c;
    #pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u32 t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += t;
    }
    const u32 tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
    if (tot >> 16) return false;
    if (fill + tot > (u32)SLICE) flush();
    u32 q = fill + inc - c;
    while (m) {
      const u32 e = __ffs(m) - 1u;
      m &= m - 1u;
      const u32 k = 64u * (e >> 1) + (e & 1u);
      sxy[q] = at[k];
      sidx[q] = id + k;
      ++q;
    }
    fill += tot;
    return true;
  }
  // One point per lane (the whole warp calls it; out: the point survives).
  __device__ __forceinline__ void push(bool out, int x, int y, u32 id) {
    const u32 bal = __ballot_sync(0xFFFFFFFFu, out);
    if (bal) {
      if (fill + __popc(bal) > (u32)SLICE) flush();
      if (out) {
        const u32 q = fill + __popc(bal & ((1u << (threadIdx.x & 31)) - 1u));
        sxy[q] = make_int2(x, y);
        sidx[q] = id;
      }
      fill += __popc(bal);
    }
  }
};

// N pairs of points per lane (pair u has indices id + 64 u and the next): all
// tested first (independent lookups in flight together), one vote for the
// warp, then the survivors pushed slot by slot.
template <int N, class Sink>
__device__ __forceinline__ void take_pairs(const PolyHead& H, const u32* tab, const int4* w, u32 id, Sink& sink) {
  u32 m = 0;
  #pragma unroll
  for (int u = 0; u < N; ++u) {
    m |= inside_poly(H, tab, w[u].x, w[u].y) ? 0u : 1u << (2 * u);
    m |= inside_poly(H, tab, w[u].z, w[u].w) ? 0u : 2u << (2 * u);
  }
  if (__any_sync(0xFFFFFFFFu, m != 0u)) {
    #pragma unroll
    for (int u = 0; u < N; ++u) {
      sink.push((m >> (2 * u)) & 1u, w[u].x, w[u].y, id + 64u * u);
      sink.push((m >> (2 * u + 1)) & 1u, w[u].z, w[u].w, id + 64u * u + 1u);
    }
  }
}

// The same through a ring of bulk copies into shared memory, one ring per
// warp (STAGES chunks of CH points; no block barrier, no registers held by
// loads in flight: 64 registers a thread for the register double buffer kept
// every other kernel off the SM).  The warp takes chunks first + k step.
// Waits are bounded by the call's spin limit; one that runs out sets
// ERR_TIMEOUT and ends the warp's stream.
template <int STAGES, int CH>
struct Ring {
  int4* buf;                // [STAGES][CH / 2], this warp's
  u64* bar;                 // [STAGES]
  u32 it;                   // chunks consumed so far
  bool ok;                  // no wait has run out

  // Whole warp, once; `buf` and `bar` are this warp's alone.
  __device__ __forceinline__ void init() {
    it = 0;
    ok = true;
    if ((threadIdx.x & 31) == 0) {
      for (int k = 0; k < STAGES; ++k) mbar_init(&bar[k], 1u);
      mbar_fence_init();
    }
    __syncwarp();
  }
  // Lane 0: chunk number `at` of the ring's sequence from src.
  __device__ __forceinline__ void load(u32 at, const int4* src, u64 pol) {
    const u32 st = at % STAGES;
    mbar_arrive_expect_tx(&bar[st], CH * 8u);
    bulk_load_hint(buf + st * (CH / 2), src, CH * 8u, &bar[st], pol);
  }
};

// The points of a set whose sample lies on the line L: of those on it only
// each warp's lexicographic extremes survive (what lies between two of them
// is no vertex, an equal point with a larger index neither), every other
// point does.  As raw survivors all points of a line went on to the bucket sort
// (20M points 1,943 us a call, 115 this way).  Out of line, with a sink of
// its own that it empties: the ring's loop keeps its registers.
template <class Sink>
__device__ __noinline__ void stream_line(const int2* Q, u32 cnt, u32 id0, u32 first, u32 step, const PolyLine* line,
                                         Sink sink) {
  const PolyLine L = *line;
  constexpr u32 V = 4, R = 32u * V;
  const int lane = threadIdx.x & 31;
  u64 lo = ~0ull, hi = 0ull;
  u32 ilo = 0xFFFFFFFFu, ihi = 0xFFFFFFFFu;       // a lane's indices increase: the first of equal points
  for (u32 b = first; b < (cnt + R - 1u) / R; b += step) {
    int2 p[V];
    #pragma unroll
    for (u32 r = 0; r < V; ++r) p[r] = b * R + 32u * r + lane < cnt ? Q[b * R + 32u * r + lane] : make_int2(0, 0);
    #pragma unroll
    for (u32 r = 0; r < V; ++r) {
      const u32 i = b * R + 32u * r + lane;
      const bool in = i < cnt, on = in && on_line(L, p[r]);
      if (on) {
        const u64 v = lex_key(p[r]);
        if (v < lo) { lo = v; ilo = id0 + i; }
        if (ihi == 0xFFFFFFFFu || v > hi) { hi = v; ihi = id0 + i; }
      }
      sink.push(in && !on, p[r].x, p[r].y, id0 + i);
    }
  }
  #pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const u64 a = __shfl_xor_sync(0xFFFFFFFFu, lo, o), c = __shfl_xor_sync(0xFFFFFFFFu, hi, o);
    const u32 ia = __shfl_xor_sync(0xFFFFFFFFu, ilo, o), ic = __shfl_xor_sync(0xFFFFFFFFu, ihi, o);
    if (a < lo || (a == lo && ia < ilo)) { lo = a; ilo = ia; }
    if (c > hi || (c == hi && ic < ihi)) { hi = c; ihi = ic; }
  }
  const bool any = ilo != 0xFFFFFFFFu;
  const int2 w = lex_point(lane == 0 ? lo : hi);
  sink.push(any && (lane == 0 || (lane == 1 && lo != hi)), w.x, w.y, lane == 0 ? ilo : ihi);
  if (sink.fill) sink.flush();
}

// flat(): called by the warp instead of the stream when the sample lies on
// one line (its copies have landed).
template <int STAGES, int CH, class Sink, class Prep, class Flat>
__device__ __forceinline__ void stream_ring(Ring<STAGES, CH>& ring, const int2* __restrict__ Q, u32 cnt, u32 id0,
                                            u32 first, u32 step, const PolyHead& H, const PolyLine* line,
                                            const u32* tab, Sink& sink, u32* error, u32 spin, Prep prep, Flat flat) {
  static_assert(CH % 64 == 0 && CH <= 512, "whole pairs per lane, a mask bit per point below kLate");
  constexpr u32 R = CH / 2;                       // pairs per chunk
  const int lane = threadIdx.x & 31;
  const u32 head = (reinterpret_cast<uintptr_t>(Q) & 15u) && cnt ? 1u : 0u;
  const int4* p4 = reinterpret_cast<const int4*>(Q + head);
  const u32 npair = (cnt - head) >> 1;
  const u32 nfull = npair / R;
  const u32 mine = ring.ok && first < nfull ? (nfull - 1u - first) / step + 1u : 0u;
  const u64 pol = policy_evict_first();
  if (lane == 0)
    for (u32 k = 0; k < min(mine, (u32)STAGES); ++k) ring.load(ring.it + k, p4 + (size_t)(first + k * step) * R, pol);
  prep();
  if (!H.ok && line->ok) {            // the chunks under way are not needed
    const u32 out = min(mine, (u32)STAGES);
    bool got = true;
    for (u32 j = 0; j < out; ++j)
      got = mbar_wait(&ring.bar[(ring.it + j) % STAGES], ((ring.it + j) / STAGES) & 1u) && got;
    ring.it += out;
    if (!__all_sync(0xFFFFFFFFu, got)) {
      if (lane == 0) atomicOr(error, ERR_TIMEOUT);
      ring.ok = false;
    }
    flat();
    return;
  }
  for (u32 k = 0; k < mine; ++k, ++ring.it) {
    const u32 st = ring.it % STAGES;
    // A limit of one gives up on what is not there at once (a try suspends for
    // as long as the hardware likes).
    const u32 par = (ring.it / STAGES) & 1u;
    const bool got = spin > 1u ? mbar_wait(&ring.bar[st], par, spin) : mbar_test_wait(&ring.bar[st], par);
    const int4* b = ring.buf + st * R + lane;
    const u32 id = id0 + head + 2u * ((first + k * step) * R + lane);
    u32 m = got ? 0u : kLate;         // the lane's points outside, pair u's at bits 2 u and 2 u + 1
    #pragma unroll
    for (int u = 0; u < (int)R / 32; ++u) {
      const int4 w = b[32 * u];
      m |= inside_poly(H, tab, w.x, w.y) ? 0u : 1u << (2 * u);
      m |= inside_poly(H, tab, w.z, w.w) ? 0u : 2u << (2 * u);
    }
    if (__any_sync(0xFFFFFFFFu, m != 0u) && !sink.push_lanes(m, reinterpret_cast<const int2*>(b), id)) {
      // The whole warp gives up, whichever lane's wait ran out.
      if (lane == 0) atomicOr(error, ERR_TIMEOUT);
      ring.ok = false;                // no further copy; those in flight, this one too, get their time
      for (u32 j = 0; j < (u32)STAGES && k + j < mine; ++j)
        mbar_wait(&ring.bar[(ring.it + j) % STAGES], ((ring.it + j) / STAGES) & 1u);
      __syncwarp();
      break;
    }
    __syncwarp();
    if (lane == 0 && k + STAGES < mine) ring.load(ring.it + STAGES, p4 + (size_t)(first + (k + STAGES) * step) * R, pol);
  }
  // The pairs past the last full chunk, and the points outside the pairs: one warp.
  if (first == nfull % step) {
    for (u32 b = nfull * R; b < npair; b += 32u) {
      const u32 j = b + lane;
      const bool in = j < npair;
      const int4 w = in ? p4[j] : make_int4(0, 0, 0, 0);
      const u32 id = id0 + head + 2u * j;
      sink.push(in && !inside_poly(H, tab, w.x, w.y), w.x, w.y, id);
      sink.push(in && !inside_poly(H, tab, w.z, w.w), w.z, w.w, id + 1u);
    }
    const u32 rest = (cnt - head) & 1u;
    const bool in = lane < 2 && (lane == 0 ? head : rest) != 0u;
    const u32 j = lane == 0 ? 0u : cnt - 1u;
    const int2 p = in ? Q[j] : make_int2(0, 0);
    sink.push(in && !inside_poly(H, tab, p.x, p.y), p.x, p.y, id0 + j);
  }
}

// The stream's sink of a block that finishes its points itself: its list.
template <class L>
struct ListSink {
  L* list;
  u32* count;
  u32 cap;
  bool bad;                 // a coordinate out of range
  __device__ __forceinline__ void push(bool out, int x, int y, u32 id) {
    const u32 bal = __ballot_sync(0xFFFFFFFFu, out);
    if (bal) {
      const int lane = threadIdx.x & 31;
      u32 base = 0;
      if (lane == 0) base = atomicAdd(count, (u32)__popc(bal));
      base = __shfl_sync(0xFFFFFFFFu, base, 0) + __popc(bal & ((1u << lane) - 1u));
      if (out) {
        if (base < cap) { list->p[base] = make_int2(x, y); list->id[base] = id; }
        bad = bad || out_of_range(x, y);
      }
    }
  }
};

// Streams the points Q[0, cnt) (indices id0 ..) through the polygon's test:
// this warp takes the rounds of 32 V pairs that start at pair 32 V (first +
// k step).  The next round's loads go out before a round is tested; prep()
// runs after the first loads are issued (it fills `tab` and has the block's
// barrier).  Q starts on any row: the point before its 16-byte boundary and
// the odd last one go to warp 0's lanes.
template <int V, class Sink, class Prep>
__device__ __forceinline__ void stream_points(const int2* __restrict__ Q, u32 cnt, u32 id0, u32 first, u32 step,
                                              const PolyHead& H, const u32* tab, Sink& sink, Prep prep) {
  const int lane = threadIdx.x & 31;
  const u32 head = (reinterpret_cast<uintptr_t>(Q) & 15u) && cnt ? 1u : 0u;
  const int4* p4 = reinterpret_cast<const int4*>(Q + head);
  const u32 npair = (cnt - head) >> 1;
  constexpr u32 R = 32u * V;
  u32 w0 = first * R;                             // the warp's first pair of the round
  int4 cur[V];
  if (w0 + R <= npair) {
    #pragma unroll
    for (int u = 0; u < V; ++u) cur[u] = p4[w0 + lane + 32u * u];
  }
  prep();
  while (w0 + R <= npair) {
    const u32 w1 = w0 + step * R;
    int4 nxt[V];
    if (w1 + R <= npair) {
      #pragma unroll
      for (int u = 0; u < V; ++u) nxt[u] = p4[w1 + lane + 32u * u];
    }
    take_pairs<V>(H, tab, cur, id0 + head + 2u * (w0 + lane), sink);
    #pragma unroll
    for (int u = 0; u < V; ++u) cur[u] = nxt[u];
    w0 = w1;
  }
  // The last, partial round (one warp has it).
  for (u32 b = w0; b < min(npair, w0 + R); b += 32u) {
    const u32 j = b + lane;
    const bool in = j < npair;
    const int4 w = in ? p4[j] : make_int4(0, 0, 0, 0);
    const u32 id = id0 + head + 2u * j;
    sink.push(in && !inside_poly(H, tab, w.x, w.y), w.x, w.y, id);
    sink.push(in && !inside_poly(H, tab, w.z, w.w), w.z, w.w, id + 1u);
  }
  if (first == 0) {
    const u32 rest = (cnt - head) & 1u;
    const bool in = lane < 2 && (lane == 0 ? head : rest) != 0u;
    const u32 j = lane == 0 ? 0u : cnt - 1u;
    const int2 p = in ? Q[j] : make_int2(0, 0);
    sink.push(in && !inside_poly(H, tab, p.x, p.y), p.x, p.y, id0 + j);
  }
}

// ---------------------------------------------------------------- candidates
// Candidate points of the angular bins: cand / cid with the occupancy bits.
template <int NB>
struct CandTab {
  int2 cand[NB];
  u32 cid[NB];
  u32 occ[NB / 32];
};
// Nearest occupied bin after / before b, cyclically (b itself last); some
// bin is occupied.
template <int NB>
__device__ __forceinline__ u32 next_bin(const u32* occ, u32 b) {
  constexpr u32 NW = NB / 32;
  u32 w = b >> 5;
  u32 m = (b & 31u) == 31u ? 0u : occ[w] & (0xFFFFFFFFu << ((b & 31u) + 1u));
  for (u32 it = 0; it < NW && m == 0u; ++it) { w = (w + 1u) & (NW - 1u); m = occ[w]; }
  return m ? (w << 5) + (u32)__ffs(m) - 1u : b;
}
template <int NB>
__device__ __forceinline__ u32 prev_bin(const u32* occ, u32 b) {
  constexpr u32 NW = NB / 32;
  u32 w = b >> 5;
  u32 m = occ[w] & ((1u << (b & 31u)) - 1u);
  for (u32 it = 0; it < NW && m == 0u; ++it) { w = (w + NW - 1u) & (NW - 1u); m = occ[w]; }
  return m ? (w << 5) + 31u - (u32)__clz(m) : b;
}

// Point (x, y) with index id in bin b: dropped by its wedge of the candidate
// polygon?
template <int NB>
__device__ __forceinline__ bool dropped_by_cands(const CandTab<NB>& C, const StarFrame& F, u32 b, int x, int y,
                                                 u32 id) {
  const int2 q = make_int2(x - F.cx, y - F.cy);
  u32 ba, bb;
  if ((C.occ[b >> 5] >> (b & 31u)) & 1u) {
    const int2 p = C.cand[b];
    const bool after = cross2(p.x - F.cx, p.y - F.cy, q.x, q.y) >= 0;
    ba = after ? b : prev_bin<NB>(C.occ, b);
    bb = after ? next_bin<NB>(C.occ, b) : b;
  } else {
    ba = prev_bin<NB>(C.occ, b);
    bb = next_bin<NB>(C.occ, b);
  }
  const int2 A = C.cand[ba], B = C.cand[bb];
  if ((x == A.x && y == A.y && id > C.cid[ba]) || (x == B.x && y == B.y && id > C.cid[bb])) return true;
  return dropped_by(make_int2(A.x - F.cx, A.y - F.cy), make_int2(B.x - F.cx, B.y - F.cy), q);
}

// ---------------------------------------------------------------- hull of a list
constexpr u32 kBinMax = 192;       // most points of one bin ordered by counting
constexpr int kRounds = 48;        // most rounds

// p, id: the points (any order) and their input indices, [0, CAP).  ta holds
// the positions of the m points to start from.
template <int BLOCK, int CAP, int NB>
struct ListSmem {
  int2 p[CAP];
  u32 id[CAP];
  unsigned short bn[CAP];
  unsigned short ta[CAP], tb[CAP];
  __align__(8) u32 cnt[NB];
  u32 cur[NB];
  u32 ws[2][BLOCK / 32];
  u64 first;
  u32 flag;
  // The bins' directions for filter_list, in the place of the counts that list_hull needs later.
  __device__ float2* dirs() { return reinterpret_cast<float2*>(cnt); }
};

// The rank of entry i of the bin's entries at[s, e) (positions in p) in the
// order: counter-clockwise about c, along a ray the farther first, equal
// points by index.  dead: not the first of its ray (a nearer point of a ray
// is no vertex), or c itself.
__device__ __forceinline__ u32 bin_rank(const int2* p, const u32* id, const unsigned short* at, u32 s, u32 e, u32 i,
                                        const StarFrame& F, bool& dead) {
  const u32 k = at[i];
  const int2 w = p[k];
  const int2 q = make_int2(w.x - F.cx, w.y - F.cy);
  const u32 qr = (u32)abs(q.x) + (u32)abs(q.y), qi = id[k];
  u32 r = 0;
  dead = q.x == 0 && q.y == 0;
  for (u32 j = s; j < e; ++j) {
    if (j == i) continue;
    const u32 kj = at[j];
    const int2 v = p[kj];
    const int2 d = make_int2(v.x - F.cx, v.y - F.cy);
    const long long c = cross2(d.x, d.y, q.x, q.y);
    if (c > 0) { ++r; continue; }
    if (c < 0) continue;
    const u32 dr = (u32)abs(d.x) + (u32)abs(d.y);
    if (dr > qr || (dr == qr && id[kj] < qi)) { ++r; dead = true; }
  }
  return r;
}

// Neighbours in cur[0, m) that stand in the wrong order about c change
// places, twice over the even and the odd pairs: points of adjacent bins
// whose angles are closer than the float bins tell them apart (elongated
// sets lose digits to the whitening).  OPEN: the ends are no neighbours.
// Ends with a barrier.
template <int BLOCK, bool OPEN, class L>
__device__ __forceinline__ void mend_order(const L& S, u32 m, const StarFrame& F, unsigned short* cur) {
  #pragma unroll
  for (int k = 0; k < 4; ++k) {
    for (u32 i = 2u * threadIdx.x + (k & 1u); i < m; i += 2u * BLOCK) {
      const u32 j = i + 1u < m ? i + 1u : 0u;
      if (j == 0u && (OPEN || (i & 1u) == 0u)) continue;   // (no wrapping pair of an odd number of entries)
      const unsigned short a = cur[i], b = cur[j];
      const int2 p = S.p[a & 0x7FFFu], q = S.p[b & 0x7FFFu];
      const int ax = p.x - F.cx, ay = p.y - F.cy, bx = q.x - F.cx, by = q.y - F.cy;
      if (cross2(ax, ay, bx, by) < 0 && (long long)ax * bx + (long long)ay * by > 0) { cur[i] = b; cur[j] = a; }
    }
    __syncthreads();
  }
}

// The rounds over the entries cur[0, m) (positions in S.p in angular order,
// bit 15: marked for removal when `marked`): thread t owns a run of
// consecutive entries and drops those that the wedge of their neighbours
// covers.  OPEN: the entries are a run of a longer cyclic list and its two
// ends stay; otherwise they are the whole cyclic list and `done` reports
// that the last round dropped nothing and every entry is a vertex of a
// convex polygon about c.  `cur` and `nxt` may be exchanged; returns the
// number of entries left in cur.
template <int BLOCK, bool OPEN, class L>
__device__ u32 drop_rounds(L& S, u32 m, const StarFrame& F, unsigned short* nxt, unsigned short*& cur, bool marked,
                           bool& done) {
  const int t = threadIdx.x;
  auto rel = [&](u32 k) { const int2 p = S.p[k]; return make_int2(p.x - F.cx, p.y - F.cy); };
  u32 par = 1;
  done = false;
  for (int round = marked ? 0 : 1; round <= kRounds; ++round) {
    const u32 per = (m + BLOCK - 1) / BLOCK;
    const u32 i0 = min(m, t * per), i1 = min(m, i0 + per);
    u32 kept = 0, mask = 0;                 // at most 32 entries a thread (the lists' assertions)
    bool bad = false;
    for (u32 i = i0; i < i1; ++i) {
      const u32 k = cur[i];
      bool keep;
      if (round == 0) {
        keep = !(k & 0x8000u);
      } else if (OPEN && (i == 0 || i == m - 1)) {
        keep = true;
      } else {
        const int2 q = rel(k);
        const int2 a = rel(cur[i > 0 ? i - 1 : m - 1]), b = rel(cur[i + 1 < m ? i + 1 : 0]);
        const long long ab = cross2(a.x, a.y, b.x, b.y);
        const long long aq = cross2(a.x, a.y, q.x, q.y), qb = cross2(q.x, q.y, b.x, b.y);
        const long long o = ab - aq - qb;
        keep = !(ab > 0 && aq >= 0 && qb >= 0 && (o > 0 || (o == 0 && aq > 0 && qb > 0)));
        // A vertex of the verified polygon: c strictly left of both its
        // edges, a strict left turn (o < 0).
        bad = bad || !(aq > 0 && qb > 0 && o < 0);
        if (keep && round <= 3 && m > 8 && (!OPEN || (i >= 2 && i + 2 < m))) {
          // A wider wedge drops runs of points in fewer rounds.
          const int2 a2 = rel(cur[i >= 2 ? i - 2 : i + m - 2]), b2 = rel(cur[i + 2 < m ? i + 2 : i + 2 - m]);
          keep = !dropped_by(a2, b2, q);
        }
      }
      if (keep) { mask |= 1u << (i - i0); ++kept; }
    }
    u32 tot;
    u32 pos = block_scan<BLOCK>(kept, S.ws[par], tot);
    par ^= 1u;
    if (round > 0 && tot == m) {         // uniform: nothing dropped
      done = OPEN || !__syncthreads_or(bad);
      break;
    }
    for (u32 i = i0; i < i1; ++i)
      if ((mask >> (i - i0)) & 1u) nxt[pos++] = cur[i];
    __syncthreads();
    unsigned short* w = cur; cur = nxt; nxt = w;
    m = tot;
    if (m < 3) break;
  }
  return m;
}

// The hull of the m points named by S.ta (the whole block; S.p, S.id, S.ta
// written and visible).  Returns its number of vertices, written as input
// indices counter-clockwise from the lexicographic minimum into out[0, cap)
// (nothing when it exceeds cap), or -1: not decided here.
template <int BLOCK, int CAP, int NB>
__device__ int list_hull(ListSmem<BLOCK, CAP, NB>& S, u32 m, const StarFrame& F, int* out, long long cap) {
  static_assert(NB % BLOCK == 0 || BLOCK % NB == 0, "whole bins per thread");
  static_assert(CAP <= 32768 && CAP / BLOCK <= 32, "a position and a flag in 16 bits, one mask bit per owned entry");
  constexpr int PER = NB / BLOCK > 0 ? NB / BLOCK : 1;
  const int t = threadIdx.x;
  if (m < 3 || m > (u32)CAP) return -1;
  for (int b = t; b < NB; b += BLOCK) S.cnt[b] = 0u;
  if (t == 0) { S.flag = 0u; S.first = ~0ull; }
  __syncthreads();
  for (u32 i = t; i < m; i += BLOCK) {
    const u32 k = S.ta[i];
    const int2 p = S.p[k];
    float u, v;
    to_uv(F, p.x - F.cx, p.y - F.cy, u, v);
    const u32 b = bin_of<NB>(u, v);
    S.bn[k] = (unsigned short)b;
    if (atomicAdd(&S.cnt[b], 1u) >= kBinMax) S.flag = 1u;
  }
  __syncthreads();
  if (S.flag) return -1;
  {
    u32 c[PER], sum = 0, tot;
    #pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int b = t * PER + j;
      c[j] = b < NB ? S.cnt[b] : 0u;
      sum += c[j];
    }
    u32 ex = block_scan<BLOCK>(sum, S.ws[0], tot);
    #pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int b = t * PER + j;
      if (b < NB) S.cur[b] = ex;
      ex += c[j];
    }
  }
  __syncthreads();
  for (u32 i = t; i < m; i += BLOCK) {
    const unsigned short k = S.ta[i];
    S.tb[atomicAdd(&S.cur[S.bn[k]], 1u)] = k;       // cur[b] ends at the bin's end
  }
  __syncthreads();
  // Order inside the bins by counting, the removals marked (bit 15).
  for (u32 i = t; i < m; i += BLOCK) {
    const u32 k = S.tb[i], b = S.bn[k];
    const u32 e = S.cur[b], s = e - S.cnt[b];
    bool dead;
    const u32 r = bin_rank(S.p, S.id, S.tb, s, e, i, F, dead);
    S.ta[min(s + r, m - 1u)] = (unsigned short)(k | (dead ? 0x8000u : 0u));
  }
  __syncthreads();
  unsigned short* cur = S.ta;
  mend_order<BLOCK, false>(S, m, F, cur);
  bool done = false;
  m = drop_rounds<BLOCK, false>(S, m, F, S.tb, cur, true, done);
  if (!done) return -1;
  // The lexicographic minimum starts the output.
  auto lex = [&](u32 i) { return lex_key(S.p[cur[i]]); };
  u64 mn = ~0ull;
  for (u32 i = t; i < m; i += BLOCK) { const u64 v = lex(i); mn = v < mn ? v : mn; }
  {
    const u32 hi = __reduce_min_sync(0xFFFFFFFFu, (u32)(mn >> 32));
    const u32 lo = __reduce_min_sync(0xFFFFFFFFu, (u32)(mn >> 32) == hi ? (u32)mn : 0xFFFFFFFFu);
    if ((t & 31) == 0 && (t & ~31) < (int)m) atomicMin(&S.first, ((u64)hi << 32) | lo);
  }
  __syncthreads();
  const u64 f = S.first;
  for (u32 i = t; i < m; i += BLOCK)
    if (lex(i) == f) S.flag = i;              // one vertex: they are distinct
  __syncthreads();
  const u32 st = S.flag;
  if ((long long)m <= cap)
    for (u32 i = t; i < m; i += BLOCK) {
      const u32 j = st + i;
      out[i] = (int)S.id[cur[j < m ? j : j - m]];
    }
  return (int)m;
}

// The candidates of the list S.p[0, m0) and the points that they do not
// drop: their positions to S.ta, their number returned (the whole block;
// key: NB words of scratch; nrm: the bins' directions, null without a polygon).
template <int BLOCK, int CAP, int NB>
__device__ u32 filter_list(ListSmem<BLOCK, CAP, NB>& S, u32 m0, const StarFrame& F, u64* key, CandTab<NB>& C,
                           const float2* nrm) {
  const int t = threadIdx.x;
  for (int b = t; b < NB; b += BLOCK) key[b] = 0ull;
  for (int b = t; b < NB / 32; b += BLOCK) C.occ[b] = 0u;
  if (t == 0) S.flag = 0u;
  __syncthreads();
  for (u32 i = t; i < m0; i += BLOCK) {
    const int2 p = S.p[i];
    float u, v;
    to_uv(F, p.x - F.cx, p.y - F.cy, u, v);
    const u32 b = bin_of<NB>(u, v);
    const u64 k = cand_key(nrm ? nrm[b] : make_float2(u, v), u, v, S.id[i]);
    S.bn[i] = (unsigned short)b;
    if (k > *(volatile u64*)&key[b]) atomicMax(&key[b], k);
  }
  __syncthreads();
  for (u32 i = t; i < m0; i += BLOCK) {
    const u32 b = S.bn[i], id = S.id[i];
    if ((u32)key[b] == ~id) {
      C.cand[b] = S.p[i];
      C.cid[b] = id;
      atomicOr(&C.occ[b >> 5], 1u << (b & 31u));
    }
  }
  __syncthreads();
  const int lane = t & 31;
  for (u32 i0 = 0; i0 < m0; i0 += BLOCK) {
    const u32 i = i0 + t;
    bool keep = false;
    if (i < m0) {
      const int2 p = S.p[i];
      keep = !dropped_by_cands<NB>(C, F, S.bn[i], p.x, p.y, S.id[i]);
    }
    const u32 bal = __ballot_sync(0xFFFFFFFFu, keep);
    u32 base = 0;
    if (lane == 0 && bal) base = atomicAdd(&S.flag, (u32)__popc(bal));
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    if (keep) S.ta[base + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)i;
  }
  __syncthreads();
  const u32 m = S.flag;
  __syncthreads();
  return m;
}

// A degenerate or tiny set that the rounds did not decide (n >= 1 points in
// range with input indices ids, null: their positions; the whole block): all
// points equal or on one line, found from the lexicographic extremes; up to 64
// points by Andrew's chain in one thread.  The number of vertices (in out when
// they fit) or -1.  Out of line: a rare call that shall not cost its callers
// registers (inlined, kb_small took 112 us of a batch instead of 108).
template <int BLOCK, class L>
__device__ __noinline__ int rest_hull(L& S, const int2* P, const u32* ids, u32 n, int* out, long long cap) {
  __shared__ u64 s_lo, s_hi;
  __shared__ u32 s_il, s_ih;
  const int t = threadIdx.x;
  auto id = [&](u32 i) { return ids ? ids[i] : i; };
  __syncthreads();
  if (t == 0) { s_lo = ~0ull; s_hi = 0ull; s_il = s_ih = 0xFFFFFFFFu; }
  __syncthreads();
  u64 lo = ~0ull, hi = 0ull;
  for (u32 i = t; i < n; i += BLOCK) {
    const u64 v = lex_key(P[i]);
    lo = v < lo ? v : lo; hi = v > hi ? v : hi;
  }
  #pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    const u64 a = __shfl_xor_sync(0xFFFFFFFFu, lo, d), b = __shfl_xor_sync(0xFFFFFFFFu, hi, d);
    lo = a < lo ? a : lo; hi = b > hi ? b : hi;
  }
  if ((t & 31) == 0) { atomicMin(&s_lo, lo); atomicMax(&s_hi, hi); }
  __syncthreads();
  lo = s_lo; hi = s_hi;
  const int2 A = lex_point(lo), B = lex_point(hi);
  bool off = false;
  for (u32 i = t; i < n; i += BLOCK) {
    const int2 p = P[i];
    const u64 v = lex_key(p);
    if (v == lo) atomicMin(&s_il, id(i));
    if (v == hi) atomicMin(&s_ih, id(i));
    off = off || orient(A.x, A.y, B.x, B.y, p.x, p.y) != 0;
  }
  if (!__syncthreads_or(off)) {
    const int h = lo == hi ? 1 : 2;
    if (t == 0 && h <= cap) { out[0] = (int)s_il; if (h == 2) out[1] = (int)s_ih; }
    return h;
  }
  if (n > 64u) return -1;
  // Sorted by (x, y), the smallest index of equal points only.
  __shared__ u32 s_keep[2];
  const u64 v = t < (int)n ? lex_key(P[t]) : 0ull;
  bool keep = t < (int)n;
  for (u32 j = 0; j < n && keep; ++j) keep = lex_key(P[j]) != v || id(j) >= id(t);
  const u32 km = __ballot_sync(0xFFFFFFFFu, keep);
  if (t < 64 && (t & 31) == 0) s_keep[t >> 5] = km;
  __syncthreads();
  u32 r = 0;
  if (keep)
    for (u32 j = 0; j < n; ++j) r += ((s_keep[j >> 5] >> (j & 31u)) & 1u) && lex_key(P[j]) < v ? 1u : 0u;
  if (keep) S.ta[r] = (unsigned short)t;
  const int m = __syncthreads_count(keep);
  if (t == 0) {
    int k = 0;
    auto chain = [&](int i, int base) {
      const int2 p = P[S.ta[i]];
      while (k >= base + 2) {
        const int2 a = P[S.tb[k - 2]], b = P[S.tb[k - 1]];
        if (orient(a.x, a.y, b.x, b.y, p.x, p.y) > 0) break;
        --k;
      }
      S.tb[k++] = S.ta[i];
    };
    for (int i = 0; i < m; ++i) chain(i, 0);
    const int base = k - 1;
    for (int i = m - 2; i >= 0; --i) chain(i, base);
    --k;                                 // the first point again
    S.flag = (u32)k;
    if (k <= cap)
      for (int i = 0; i < k; ++i) out[i] = (int)id(S.tb[i]);
  }
  __syncthreads();
  return (int)S.flag;
}

// rest_hull of the q points of a list in global memory, out of line too.
template <int BLOCK, class L>
__device__ __noinline__ int rest_of_list(L& S, const int2* xy, const u32* idx, u32 q, int* out, long long cap) {
  for (u32 i = threadIdx.x; i < q; i += BLOCK) { S.p[i] = xy[i]; S.id[i] = idx[i]; }
  __syncthreads();
  return rest_hull<BLOCK>(S, S.p, S.id, q, out, cap);
}

}  // namespace star

// The call's summary (one thread).  h < 0: not decided.
__device__ __forceinline__ void star_summary(Plan* plan, u32 n, u32 raw, u32 s, int h, long long cap, u32 error) {
  plan->n = n;
  u32 e = error;
  if (!(e & ERR_RANGE)) {
    if (h < 0) e |= ERR_RETRY;
    else if ((long long)h > cap) e |= ERR_CAPACITY;
  }
  plan->error = e;
  plan->s = s; plan->s_quad = 0; plan->s_raw = raw; plan->r_lo = s; plan->r_up = 0;
  plan->h = h > 0 ? (u32)h : 0u; plan->h_lo = 0; plan->h_up = 0;
  plan->ncorner = 0; plan->learned_used = 0; plan->npasses = 0;
  plan->sorted_in_b = 1; plan->ngroups = 1;
}

}  // namespace gbh
