// Learned filter proposal (the project's addition beside the paper's
// quadrilateral of Section 2.1 step 2 / Section 3.1):
//
//   K6  features of a strided sample of the input: its centre, a 32-bin
//       angular histogram (fraction of points, maximum radius normalised by
//       the largest) = 64 features, and the sample's extreme point in each
//       of 32 directions u_j = (cos 2 pi j / 32, sin 2 pi j / 32);
//   K8  inference of an MLP 64 -> 128 -> 128 -> 32 (ReLU, FP16 weights,
//       FP32 accumulation); the 8 highest scores pick 8 directions, and the
//       filter polygon becomes the exact (int64) convex hull of the four
//       quadrilateral corners and those 8 extremes (at most 12 corners).  It
//       contains the quadrilateral, so it never discards less; points are
//       discarded only when strictly inside a polygon spanned by input
//       points, so the hull stays exact whatever the weights;
//   K10 labels for training: for every direction j the discard fraction of
//       hull(quad corners + e_j) minus the quadrilateral's, counted exactly;
//   training: batched forward / backward of the MLP (FP32 FFMA, on the
//       FP16-rounded weights used at inference), mean squared error on the
//       labels, Adam on FP32 master weights.
#include <cmath>

#include "hull_internal.cuh"
#include "kernels.h"
#include "learned_common.cuh"

namespace gbh {

using namespace learned;

namespace {

constexpr int F_SAMPLE = 16384;
constexpr int F_BLOCK = 512;

__device__ __forceinline__ float fp16r(float w) { return __half2float(__float2half_rn(w)); }

// K6: features and extremes of the sample of one input (one block).
__global__ void __launch_bounds__(F_BLOCK)
k6_features(const int* __restrict__ xy, u32 n, float* __restrict__ feat, int* __restrict__ ext,
            int* __restrict__ ext_xy) {
  __shared__ FeatSmem sm;
  __shared__ float s_x[D0];
  const u32 S = n < (u32)F_SAMPLE ? n : (u32)F_SAMPLE;
  block_features<F_BLOCK>(reinterpret_cast<const int2*>(xy), n, S, sm, s_x, ext_xy, ext);
  if (threadIdx.x < D0) feat[threadIdx.x] = s_x[threadIdx.x];
}

// K8: inference on one feature vector and the filter polygon (one block).
__global__ void __launch_bounds__(128)
k8_infer(const float* __restrict__ feat, const __half* __restrict__ w16, const int* __restrict__ ext_xy,
         Plan* plan) {
  __shared__ MlpSmem sm;
  if (plan->error & ERR_RANGE) return;
  if (threadIdx.x < D0) sm.x[threadIdx.x] = feat[threadIdx.x];
  __syncthreads();
  block_mlp(w16, sm);
  if (threadIdx.x != 0) return;
  int qx[4], qy[4], ox[kMaxCorners], oy[kMaxCorners];
  const int nq = plan->ncorner < 4 ? plan->ncorner : 4;
  for (int j = 0; j < nq; ++j) { qx[j] = plan->cx[j]; qy[j] = plan->cy[j]; }
  const int k = learned_polygon(sm.z, ext_xy, qx, qy, nq, ox, oy);
  if (k > 0) {
    plan->ncorner = k;
    for (int j = 0; j < k; ++j) { plan->cx[j] = ox[j]; plan->cy[j] = oy[j]; }
    plan->learned_used = 1;
  }
}

// K6 + K8 in one launch behind a gate (the pipeline's path): the
// quadrilateral's discard on PG_SAMPLE strided points i_k = floor(k n / G)
// first; when it discards PG_DISCARD of them or more, there is too little
// left for a larger polygon to discard and the quadrilateral stays (no
// features, no inference: the call costs this one short launch).
// Otherwise the features, the MLP and the polygon exactly as K6 and K8.
constexpr int PG_SAMPLE = F_BLOCK;
constexpr float PG_DISCARD = 0.95f;

__global__ void __launch_bounds__(F_BLOCK)
k6_propose(const int* __restrict__ xy, u32 n, const __half* __restrict__ w16, float* __restrict__ feat,
           int* __restrict__ ext, int* __restrict__ ext_xy, Plan* plan) {
  __shared__ FeatSmem sm;
  __shared__ MlpSmem msm;
  __shared__ u32 s_in;
  if (plan->error & ERR_RANGE) return;
  const int2* P = reinterpret_cast<const int2*>(xy);
  const int k = plan->ncorner < 4 ? plan->ncorner : 4;
  if (threadIdx.x == 0) s_in = 0;
  __syncthreads();
  const u32 G = n < (u32)PG_SAMPLE ? n : (u32)PG_SAMPLE;
  if (threadIdx.x < G && k >= 3) {
    const int2 p = P[(u32)(((unsigned long long)threadIdx.x * n) / G)];
    bool in = true;
    for (int j = 0; j < k && in; ++j) {
      const int jn = j + 1 < k ? j + 1 : 0;
      in = orient(plan->cx[j], plan->cy[j], plan->cx[jn], plan->cy[jn], p.x, p.y) > 0;
    }
    if (in) atomicAdd(&s_in, 1u);
  }
  __syncthreads();
  if ((float)s_in >= PG_DISCARD * (float)G) return;
  const u32 S = n < (u32)F_SAMPLE ? n : (u32)F_SAMPLE;
  block_features<F_BLOCK>(P, n, S, sm, msm.x, ext_xy, ext);
  if (threadIdx.x < D0) feat[threadIdx.x] = msm.x[threadIdx.x];
  __syncthreads();
  block_mlp(w16, msm);
  if (threadIdx.x != 0) return;
  int qx[4], qy[4], ox[kMaxCorners], oy[kMaxCorners];
  for (int j = 0; j < k; ++j) { qx[j] = plan->cx[j]; qy[j] = plan->cy[j]; }
  const int kk = learned_polygon(msm.z, ext_xy, qx, qy, k, ox, oy);
  if (kk > 0) {
    plan->ncorner = kk;
    for (int j = 0; j < kk; ++j) { plan->cx[j] = ox[j]; plan->cy[j] = oy[j]; }
    plan->learned_used = 1;
  }
}

// K10: exact counts of points strictly inside the quadrilateral (slot 32)
// and inside hull(quad corners + e_j) (slot j), for one instance.
__global__ void __launch_bounds__(256)
k10_labels(const int* __restrict__ xy, u32 n, const int* __restrict__ quad, int nq,
           const int* __restrict__ ext_xy, unsigned long long* __restrict__ counts) {
  __shared__ int s_px[NB + 1][8], s_py[NB + 1][8], s_k[NB + 1];
  __shared__ u32 s_c[NB + 1];
  if (threadIdx.x <= NB) {
    const int j = threadIdx.x;
    int px[8], py[8], m = 0;
    for (int q = 0; q < nq; ++q) { px[m] = quad[2 * q]; py[m] = quad[2 * q + 1]; ++m; }
    if (j < NB) { px[m] = ext_xy[2 * j]; py[m] = ext_xy[2 * j + 1]; ++m; }
    int hx[16], hy[16];
    const int k = small_hull(px, py, m, hx, hy);
    s_k[j] = k;
    for (int q = 0; q < k && q < 8; ++q) { s_px[j][q] = hx[q]; s_py[j][q] = hy[q]; }
    s_c[j] = 0;
  }
  __syncthreads();
  const int2* p2 = reinterpret_cast<const int2*>(xy);
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int2 p = p2[i];
    for (int j = 0; j <= NB; ++j) {
      const int k = s_k[j];
      bool in = k >= 3;
      for (int q = 0; q < k && in; ++q) {
        const int q2 = q + 1 == k ? 0 : q + 1;
        in = orient64(s_px[j][q], s_py[j][q], s_px[j][q2], s_py[j][q2], p.x, p.y) > 0;
      }
      const u32 bal = __ballot_sync(__activemask(), in);
      if ((threadIdx.x & 31) == (__ffs(__activemask()) - 1) && bal) atomicAdd(&s_c[j], __popc(bal));
    }
  }
  __syncthreads();
  if (threadIdx.x <= NB && s_c[threadIdx.x]) atomicAdd(&counts[threadIdx.x], (unsigned long long)s_c[threadIdx.x]);
}

// ---------------------------------------------------------------- training
// C[M x N] (row-major) = A (M x K) B^T (B stored N x K) + bias (ReLU), the
// weights and biases rounded to FP16.
__global__ void __launch_bounds__(256)
k_gemm(const float* __restrict__ A, const float* __restrict__ Bm, float* __restrict__ C, int M, int N, int K,
       const float* __restrict__ bias, int relu) {
  __shared__ float sa[16][17], sb[16][17];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int row = blockIdx.y * 16 + ty, col = blockIdx.x * 16 + tx;
  float acc = 0.f;
  for (int k0 = 0; k0 < K; k0 += 16) {
    const int ka = k0 + tx, kb = k0 + ty;
    float av = 0.f, bv = 0.f;
    if (row < M && ka < K) av = A[(size_t)row * K + ka];
    if (col < N && kb < K) bv = fp16r(Bm[(size_t)col * K + kb]);
    sa[ty][tx] = av;
    sb[ty][tx] = bv;
    __syncthreads();
    #pragma unroll
    for (int q = 0; q < 16; ++q) acc = fmaf(sa[ty][q], sb[q][tx], acc);
    __syncthreads();
  }
  if (row < M && col < N) {
    acc += fp16r(bias[col]);
    if (relu) acc = fmaxf(acc, 0.f);
    C[(size_t)row * N + col] = acc;
  }
}

// The forward pass and the backward pass down to the layers' pre-activation
// gradients, in one launch: everything but the parameter gradients is local
// to a row.  A block takes MR_ROWS rows and all weights (rounded to FP16, 57
// KB of shared memory, odd word pitches); a thread owns one unit of every
// layer for two rows, its sums in increasing order of the inputs, as the tile
// kernel's.  Bound by latency: 14 launches of 3-7 us each (tiles, column sums
// of one block, masks) took 70 us of device time for 64 rows.
constexpr int MR_ROWS = 4;
constexpr int MR_BLOCK = 256;

struct RowSmem {
  __half w1[D1][D0 + 2], w2[D2][D1 + 2], w3[D3][D2 + 2];
  float b1[D1], b2[D2], b3[D3];
  float x[MR_ROWS][D0], h1[MR_ROWS][D1], h2[MR_ROWS][D2], dz[MR_ROWS][D3], d2[MR_ROWS][D2];
  float loss[MR_ROWS];
};

// sum over k of in[k] w[k], then + bias, in the tile kernel's order.
template <int K>
__device__ __forceinline__ float unit(const float* in, const __half* w, float bias) {
  float acc = 0.f;
  #pragma unroll 8
  for (int k = 0; k < K; k += 2) {
    const float2 v = __half22float2(*reinterpret_cast<const __half2*>(w + k));
    acc = fmaf(in[k], v.x, acc);
    acc = fmaf(in[k + 1], v.y, acc);
  }
  return acc + bias;
}

template <int K, int N>
__device__ __forceinline__ void load_weights(const float* __restrict__ W, __half (&w)[N][K + 2]) {
  #pragma unroll 4
  for (int q = threadIdx.x; q < N * K / 4; q += MR_BLOCK) {
    const float4 v = reinterpret_cast<const float4*>(W)[q];
    __half2* d = reinterpret_cast<__half2*>(&w[4 * q / K][4 * q % K]);
    d[0] = __floats2half2_rn(v.x, v.y);
    d[1] = __floats2half2_rn(v.z, v.w);
  }
}

__global__ void __launch_bounds__(MR_BLOCK)
k_mlp_rows(const float* __restrict__ W, const float* __restrict__ X, const float* __restrict__ Y, int B, float scale,
           float* __restrict__ H1, float* __restrict__ H2, float* __restrict__ dZ, float* __restrict__ dH2,
           float* __restrict__ dH1, float* __restrict__ lossp) {
  extern __shared__ __align__(16) unsigned char mr_smem[];
  RowSmem& S = *reinterpret_cast<RowSmem*>(mr_smem);
  const int t = threadIdx.x, r0 = blockIdx.x * MR_ROWS, nr = min(MR_ROWS, B - r0);
  static_assert((OFF_W1 % 4) == 0 && (OFF_W2 % 4) == 0 && (OFF_W3 % 4) == 0, "16-byte rows of the weights");
  load_weights<D0, D1>(W + OFF_W1, S.w1);
  load_weights<D1, D2>(W + OFF_W2, S.w2);
  load_weights<D2, D3>(W + OFF_W3, S.w3);
  if (t < D1) { S.b1[t] = fp16r(W[OFF_B1 + t]); S.b2[t] = fp16r(W[OFF_B2 + t]); }
  if (t < D3) S.b3[t] = fp16r(W[OFF_B3 + t]);
  static_assert(MR_ROWS * D0 == MR_BLOCK && D1 == 128 && D2 == 128 && MR_BLOCK == 2 * D1, "thread layout");
  S.x[t / D0][t % D0] = t / D0 < nr ? X[(size_t)r0 * D0 + t] : 0.f;
  __syncthreads();
  const int j = t & (D1 - 1), p = t / D1 * 2;          // unit j of rows p, p + 1
  #pragma unroll
  for (int r = p; r < p + 2; ++r) {
    const float v = fmaxf(unit<D0>(S.x[r], S.w1[j], S.b1[j]), 0.f);
    S.h1[r][j] = v;
    if (r < nr) H1[(size_t)(r0 + r) * D1 + j] = v;
  }
  __syncthreads();
  #pragma unroll
  for (int r = p; r < p + 2; ++r) {
    const float v = fmaxf(unit<D1>(S.h1[r], S.w2[j], S.b2[j]), 0.f);
    S.h2[r][j] = v;
    if (r < nr) H2[(size_t)(r0 + r) * D2 + j] = v;
  }
  __syncthreads();
  if (t < MR_ROWS * D3) {                              // a warp per row
    const int r = t / D3, q = t % D3;
    float d = 0.f;
    if (r < nr) d = unit<D2>(S.h2[r], S.w3[q], S.b3[q]) - Y[(size_t)(r0 + r) * D3 + q];
    const float g = 2.f * d * scale;
    S.dz[r][q] = g;
    if (r < nr) dZ[(size_t)(r0 + r) * D3 + q] = g;
    float l = d * d;
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xFFFFFFFFu, l, o);
    if (q == 0) S.loss[r] = l * scale;
  }
  __syncthreads();
  if (t == 0) {
    float l = 0.f;
    for (int r = 0; r < MR_ROWS; ++r) l += S.loss[r];
    lossp[blockIdx.x] = l;
  }
  #pragma unroll
  for (int r = p; r < p + 2; ++r) {
    float acc = 0.f;
    #pragma unroll 8
    for (int k = 0; k < D3; ++k) acc = fmaf(S.dz[r][k], __half2float(S.w3[k][j]), acc);
    if (!(S.h2[r][j] > 0.f)) acc = 0.f;
    S.d2[r][j] = acc;
    if (r < nr) dH2[(size_t)(r0 + r) * D2 + j] = acc;
  }
  __syncthreads();
  #pragma unroll
  for (int r = p; r < p + 2; ++r) {
    float acc = 0.f;
    #pragma unroll 8
    for (int k = 0; k < D2; ++k) acc = fmaf(S.d2[r][k], __half2float(S.w2[k][j]), acc);
    if (!(S.h1[r][j] > 0.f)) acc = 0.f;
    if (r < nr) dH1[(size_t)(r0 + r) * D1 + j] = acc;
  }
}

// The parameter gradients, one 16 x 16 tile a block over all three layers:
// dW = D^T A summed over the rows in increasing order, with D the layer's
// pre-activation gradient and A its input; the tiles of the first columns
// also sum db, the first block the loss.
constexpr int MG_ROWS = 64;            // rows staged at a time
constexpr int MG_T3 = (D3 / 16) * (D2 / 16), MG_T2 = (D2 / 16) * (D1 / 16), MG_T1 = (D1 / 16) * (D0 / 16);

__global__ void __launch_bounds__(256)
k_mlp_grad(const float* __restrict__ X, const float* __restrict__ H1, const float* __restrict__ H2,
           const float* __restrict__ dZ, const float* __restrict__ dH2, const float* __restrict__ dH1, int B,
           const float* __restrict__ lossp, int nloss, float* __restrict__ grad, float* __restrict__ loss) {
  __shared__ float sa[MG_ROWS][17], sb[MG_ROWS][17];
  int b = blockIdx.x;
  if (b == 0 && threadIdx.x < 32) {
    float l = 0.f;
    for (int q = threadIdx.x; q < nloss; q += 32) l += lossp[q];
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xFFFFFFFFu, l, o);
    if (threadIdx.x == 0) *loss = l;
  }
  const float *D, *A;
  float *g, *gb;
  int M, N;
  if (b < MG_T3) { D = dZ; A = H2; g = grad + OFF_W3; gb = grad + OFF_B3; M = D3; N = D2; }
  else if (b < MG_T3 + MG_T2) { b -= MG_T3; D = dH2; A = H1; g = grad + OFF_W2; gb = grad + OFF_B2; M = D2; N = D1; }
  else { b -= MG_T3 + MG_T2; D = dH1; A = X; g = grad + OFF_W1; gb = grad + OFF_B1; M = D1; N = D0; }
  const int m0 = b / (N / 16) * 16, n0 = b % (N / 16) * 16;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float acc = 0.f, sum = 0.f;
  for (int k0 = 0; k0 < B; k0 += MG_ROWS) {
    const int kn = min(MG_ROWS, B - k0);
    #pragma unroll
    for (int q = ty; q < MG_ROWS; q += 16) {
      sa[q][tx] = q < kn ? D[(size_t)(k0 + q) * M + m0 + tx] : 0.f;
      sb[q][tx] = q < kn ? A[(size_t)(k0 + q) * N + n0 + tx] : 0.f;
    }
    __syncthreads();
    #pragma unroll 16
    for (int q = 0; q < MG_ROWS; ++q) acc = fmaf(sa[q][ty], sb[q][tx], acc);
    if (n0 == 0 && ty == 0)
      for (int q = 0; q < kn; ++q) sum += sa[q][tx];
    __syncthreads();
  }
  g[(size_t)(m0 + ty) * N + n0 + tx] = acc;
  if (n0 == 0 && ty == 0) gb[m0 + tx] = sum;
}

__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int count, float lr, float b1, float b2, float eps,
                       float c1, float c2, __half* __restrict__ w16) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi; v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    w16[i] = __float2half_rn(wi);
  }
}

__global__ void k_to_half(const float* __restrict__ w, __half* __restrict__ w16, int count) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
    w16[i] = __float2half_rn(w[i]);
}

void gemm(const float* A, const float* Bm, float* C, int M, int N, int K, const float* bias, int relu,
          cudaStream_t st) {
  dim3 grid((N + 15) / 16, (M + 15) / 16);
  k_gemm<<<grid, 256, 0, st>>>(A, Bm, C, M, N, K, bias, relu);
}

}  // namespace

int mlp_num_params() { return N_PARAMS; }

cudaError_t launch_features(const int* xy, u32 n, float* feat, int* ext, int* ext_xy, cudaStream_t st) {
  k6_features<<<1, F_BLOCK, 0, st>>>(xy, n, feat, ext, ext_xy);
  return cudaGetLastError();
}

cudaError_t launch_propose(const int* xy, u32 n, const void* w16, float* feat, int* ext, int* ext_xy, Plan* plan,
                           cudaStream_t st) {
  k6_propose<<<1, F_BLOCK, 0, st>>>(xy, n, reinterpret_cast<const __half*>(w16), feat, ext, ext_xy, plan);
  return cudaGetLastError();
}

cudaError_t launch_infer(const float* feat, const void* w16, const int* ext_xy, Plan* plan,
                         cudaStream_t st) {
  k8_infer<<<1, 128, 0, st>>>(feat, reinterpret_cast<const __half*>(w16), ext_xy, plan);
  return cudaGetLastError();
}

cudaError_t launch_labels(const int* xy, u32 n, const int* quad, int nq, const int* ext_xy,
                          unsigned long long* counts, int grid, cudaStream_t st) {
  k10_labels<<<grid, 256, 0, st>>>(xy, n, quad, nq, ext_xy, counts);
  return cudaGetLastError();
}

cudaError_t launch_to_half(const float* w, void* w16, int count, cudaStream_t st) {
  k_to_half<<<64, 256, 0, st>>>(w, reinterpret_cast<__half*>(w16), count);
  return cudaGetLastError();
}

// Forward pass for B feature rows; activations in act = [H1 (B x 128) |
// H2 (B x 128) | Z (B x 32)].
cudaError_t mlp_forward(const float* W, const float* X, int B, float* act, cudaStream_t st) {
  float* H1 = act;
  float* H2 = H1 + (size_t)B * D1;
  float* Z = H2 + (size_t)B * D2;
  gemm(X, W + OFF_W1, H1, B, D1, D0, W + OFF_B1, 1, st);
  gemm(H1, W + OFF_W2, H2, B, D2, D1, W + OFF_B2, 1, st);
  gemm(H2, W + OFF_W3, Z, B, D3, D2, W + OFF_B3, 0, st);
  return cudaGetLastError();
}

// Forward pass and gradient of the mean squared error (over B x 32 entries)
// with respect to the parameters (evaluated at the FP16-rounded weights);
// grad and loss are overwritten.  act holds B * 256 floats, scratch
// mlp_scratch_floats(B).
size_t mlp_scratch_floats(int B) { return (size_t)B * (D3 + D2 + D1) + (size_t)(B + MR_ROWS - 1) / MR_ROWS; }

cudaError_t mlp_configure() {
  return cudaFuncSetAttribute(k_mlp_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RowSmem));
}

cudaError_t mlp_gradient(const float* W, const float* X, const float* Y, int B, float* act, float* grad, float* loss,
                         float* scratch, cudaStream_t st) {
  float* H1 = act;
  float* H2 = H1 + (size_t)B * D1;
  float* dZ = scratch;
  float* dH2 = dZ + (size_t)B * D3;
  float* dH1 = dH2 + (size_t)B * D2;
  float* lossp = dH1 + (size_t)B * D1;
  const int blocks = (B + MR_ROWS - 1) / MR_ROWS;
  k_mlp_rows<<<blocks, MR_BLOCK, sizeof(RowSmem), st>>>(W, X, Y, B, 1.f / (float)(B * D3), H1, H2, dZ, dH2, dH1, lossp);
  k_mlp_grad<<<MG_T3 + MG_T2 + MG_T1, 256, 0, st>>>(X, H1, H2, dZ, dH2, dH1, B, lossp, blocks, grad, loss);
  return cudaGetLastError();
}

cudaError_t mlp_adam(float* W, const float* grad, float* m, float* v, int step, float lr,
                     void* w16, cudaStream_t st) {
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  k_adam<<<64, 256, 0, st>>>(W, grad, m, v, N_PARAMS, lr, b1, b2, eps, c1, c2,
                             reinterpret_cast<__half*>(w16));
  return cudaGetLastError();
}

}  // namespace gbh
