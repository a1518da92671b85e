// The key projection of the SA step (paper Sec. 3.1: S = (P W_Q)(X W_K)^T /
// sqrt(d), sketch A X; App. G.3: K = X W_K) folded into the prototypes.
//
// With keys k_i = x_i W_K and values x_i, the scores are
//     S[j,i] = q_j . (x_i W_K) = (q_j W_K^T) . x_i,
// so the sketching step runs unchanged on K = V = X with prototypes
// Q' = Q W_K^T: no K is materialised, X is the only per-token input, and the
// projection costs P d^2 per head instead of L d^2 per token range.  The
// backward maps the step's gradients (dK', dV, dQ' with respect to K = X, V = X
// and Q') back to the caller's parameters:
//     dX  = dV + dK'                 (X enters as the keys and as the values)
//     dQ  = dQ' W_K,   dW_K = dQ'^T Q   (chain rule through Q' = Q W_K^T)
// dX is summed in the tensor-core backward's own epilogue (Args::sum_dx), in
// fp32 and stored once; after the CUDA-core backward a pass adds dK' to dV.
// The prototype-sized products run on one tiled CUDA-core kernel (fp32
// accumulation): a block owns 32 x 32 outputs and stages 32-deep operand tiles
// in shared memory.  P = 512, d = 128, H = 8 is 134 MFLOP per product, a few
// microseconds of FMA; one thread per output reading its operands from global
// memory took 265 us (Q') and 171 us (dQ and dW_K together).
// The step of 12 users (256K tokens, P = 512, d = 128): 3.76 ms with those and
// the separate dX pass (538 us), 2.40 ms without (2.09 ms with the present backward).
#include "sa_kernels.cuh"

namespace sa {

constexpr int kTileMN = 32, kTileK = 32;

// out[m, n] = sum_k A(m, k) B(k, n) for the block's 32 x 32 tile, k in order.
// A_T / B_T: the operand is stored with k as its row index (A[k][m], B[k][n]);
// otherwise with k as its column (A[m][k], B[n][k]).  256 threads: thread (r, c)
// = (tid / 32, tid % 32) computes rows r, r + 8, r + 16, r + 24 of column c.
template <bool A_T, bool B_T, typename TA, typename TB, typename TO>
__device__ __forceinline__ void tile_product(const TA* __restrict__ A, int lda, const TB* __restrict__ B, int ldb,
                                             int M, int N, int K, int m0, int n0, TO* __restrict__ out, int ldo) {
  __shared__ float as[kTileK][kTileMN + 1], bs[kTileK][kTileMN + 1];
  const int c = threadIdx.x & 31, r = threadIdx.x >> 5;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int k0 = 0; k0 < K; k0 += kTileK) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int x = r + 8 * q;  // the slow index of the load; c runs along a row of the source
      if (A_T)
        as[x][c] = (k0 + x < K && m0 + c < M) ? ld_f32(A + int64_t(k0 + x) * lda + m0 + c) : 0.f;
      else
        as[c][x] = (m0 + x < M && k0 + c < K) ? ld_f32(A + int64_t(m0 + x) * lda + k0 + c) : 0.f;
      if (B_T)
        bs[x][c] = (k0 + x < K && n0 + c < N) ? ld_f32(B + int64_t(k0 + x) * ldb + n0 + c) : 0.f;
      else
        bs[c][x] = (n0 + x < N && k0 + c < K) ? ld_f32(B + int64_t(n0 + x) * ldb + k0 + c) : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kTileK; ++k) {
      const float b = bs[k][c];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = fmaf(as[k][r + 8 * q], b, acc[q]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (m0 + r + 8 * q < M && n0 + c < N) st_from_f32(out + int64_t(m0 + r + 8 * q) * ldo + n0 + c, acc[q]);
}

// Q'[h] = Q[h] Wk[h]^T: grid (ceil(P / 32), ceil(d / 32), H).
template <typename T>
__global__ void __launch_bounds__(256) fold_wk_kernel(const T* __restrict__ Q, const T* __restrict__ Wk, int P,
                                                      int d, T* __restrict__ Qf) {
  const int64_t h = blockIdx.z;
  tile_product<false, false>(Q + h * P * d, d, Wk + h * d * d, d, P, d, d, blockIdx.x * kTileMN,
                             blockIdx.y * kTileMN, Qf + h * P * d, d);
}

// dX += dK' elementwise (both of type T).
template <typename T>
__global__ void add_into_kernel(T* __restrict__ dX, const T* __restrict__ dKf, int64_t n) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    st_from_f32(dX + i, ld_f32(dX + i) + ld_f32(dKf + i));
}

// dst = -src elementwise (exact in bf16 and fp32).
template <typename T>
__global__ void negate_kernel(const T* __restrict__ src, T* __restrict__ dst, int64_t n) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    dst[i] = -src[i];
}

// dQ[h] = dQ'[h] Wk[h]  (P x d),  dWk[h] = dQ'[h]^T Q[h]  (d x d); fp32 outputs.
// grid (ceil(P / 32) + ceil(d / 32), ceil(d / 32), H): the first blocks of x take
// dWk's rows (their sums are the longer ones), the others dQ's.
template <typename T>
__global__ void __launch_bounds__(256) wk_grads_kernel(const float* __restrict__ dQf, const T* __restrict__ Q,
                                                       const T* __restrict__ Wk, int P, int d,
                                                       float* __restrict__ dQ, float* __restrict__ dWk) {
  const int64_t h = blockIdx.z;
  const int nw = (d + kTileMN - 1) / kTileMN, n0 = blockIdx.y * kTileMN;
  const float* G = dQf + h * P * d;
  if (int(blockIdx.x) < nw)
    tile_product<true, true>(G, d, Q + h * P * d, d, d, d, P, blockIdx.x * kTileMN, n0, dWk + h * d * d, d);
  else
    tile_product<false, true>(G, d, Wk + h * d * d, d, P, d, d, (blockIdx.x - nw) * kTileMN, n0, dQ + h * P * d, d);
}

cudaError_t launch_fold_wk(const void* Q, const void* Wk, int H, int P, int d, sa_dtype dt, void* Qf,
                           cudaStream_t st) {
  const dim3 grid((P + kTileMN - 1) / kTileMN, (d + kTileMN - 1) / kTileMN, H);
  if (dt == SA_BF16)
    fold_wk_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(static_cast<const __nv_bfloat16*>(Q),
                                                        static_cast<const __nv_bfloat16*>(Wk), P, d,
                                                        static_cast<__nv_bfloat16*>(Qf));
  else
    fold_wk_kernel<float><<<grid, 256, 0, st>>>(static_cast<const float*>(Q), static_cast<const float*>(Wk), P, d,
                                                static_cast<float*>(Qf));
  return cudaGetLastError();
}

cudaError_t launch_add_into(void* dX, const void* dKf, int64_t n, sa_dtype dt, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  if (dt == SA_BF16)
    add_into_kernel<__nv_bfloat16><<<2048, 256, 0, st>>>(static_cast<__nv_bfloat16*>(dX),
                                                         static_cast<const __nv_bfloat16*>(dKf), n);
  else
    add_into_kernel<float><<<2048, 256, 0, st>>>(static_cast<float*>(dX), static_cast<const float*>(dKf), n);
  return cudaGetLastError();
}

cudaError_t launch_negate(const void* src, void* dst, int64_t n, sa_dtype dt, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const int blocks = int((n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024);
  if (dt == SA_BF16)
    negate_kernel<__nv_bfloat16><<<blocks, 256, 0, st>>>(static_cast<const __nv_bfloat16*>(src),
                                                         static_cast<__nv_bfloat16*>(dst), n);
  else
    negate_kernel<float><<<blocks, 256, 0, st>>>(static_cast<const float*>(src), static_cast<float*>(dst), n);
  return cudaGetLastError();
}

cudaError_t launch_wk_grads(const float* dQf, const void* Q, const void* Wk, int H, int P, int d, sa_dtype dt,
                            float* dQ, float* dWk, cudaStream_t st) {
  const int nw = (d + kTileMN - 1) / kTileMN;
  const dim3 grid((P + kTileMN - 1) / kTileMN + nw, nw, H);
  if (dt == SA_BF16)
    wk_grads_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(dQf, static_cast<const __nv_bfloat16*>(Q),
                                                         static_cast<const __nv_bfloat16*>(Wk), P, d, dQ, dWk);
  else
    wk_grads_kernel<float><<<grid, 256, 0, st>>>(dQf, static_cast<const float*>(Q), static_cast<const float*>(Wk),
                                                 P, d, dQ, dWk);
  return cudaGetLastError();
}

}  // namespace sa
