// CUDA-core kernels of the SA sketching step: the ragged planner and a
// fp32-arithmetic path used for fp32 inputs and for shapes the tensor-core
// kernels do not cover.
//
// Forward (paper Sec. 3.1): per token the log-sum-exp over the P prototypes is
// computed first (simt_lse_kernel), then blocks of 64 prototypes accumulate
// A[j,i] V_i with A[j,i] = exp(S[j,i] - lse_i) over a worker's tile range.
// Backward (chain rule of Sec. 3.1): per token tile dV and D_i = dV_i . v_i,
// then dK; dQ is accumulated per worker and head and reduced in a fixed order.
#include <type_traits>

#include "sa_kernels.cuh"
#include "sa_simt_util.cuh"

namespace sa {

constexpr int ST = 32;    // tokens per tile on this path
constexpr int SPB = 64;   // prototypes per block
constexpr int SNT = 128;  // threads per block

// ------------------------------------------------------------------ planner
// One block: validates cu_seqlens and writes the per-head tile prefix.
__global__ void __launch_bounds__(1024) plan_kernel(const int32_t* __restrict__ cu, int B,
                                                    int64_t N, int T, void* ws,
                                                    int64_t* __restrict__ prefix, uint64_t wait_ns) {
  __shared__ int64_t warp_tot[32];
  __shared__ int64_t carry;
  __shared__ int bad;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) {
    carry = 0;
    bad = (cu[0] != 0) || (int64_t(cu[B]) != N);
    ws_header(ws)->timeout_site = 0;
    ws_header(ws)->wait_limit_ns = wait_ns;
  }
  __syncthreads();
  for (int base = 0; base < B; base += 1024) {
    const int b = base + tid;
    int64_t n = 0;
    if (b < B) {
      const int64_t L = int64_t(cu[b + 1]) - int64_t(cu[b]);
      if (L < 0) bad = 1;
      n = L > 0 ? (L + T - 1) / T : 0;
    }
    int64_t x = n;  // inclusive warp scan
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[wid] = x;
    __syncthreads();
    if (wid == 0) {
      int64_t s = warp_tot[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
      }
      warp_tot[lane] = s;  // inclusive over warps
    }
    __syncthreads();
    const int64_t before = carry + (wid > 0 ? warp_tot[wid - 1] : 0) + (x - n);
    if (b < B) prefix[b] = before;
    __syncthreads();
    if (tid == 0) carry += warp_tot[31];
    __syncthreads();
  }
  if (tid == 0) {
    prefix[B] = carry;
    ws_header(ws)->tiles_per_head = carry;
    ws_header(ws)->err = bad ? uint32_t(SA_ERR_BAD_SEQLENS) : 0u;
  }
}

// ------------------------------------------------------------- block products
// Blocks of 128 threads work on 32 tokens x 64 prototypes.  What bounds these
// kernels is how many FMAs each shared-memory wavefront feeds, so every thread
// owns a 4 x 4 (scores) or 4 x 4..16 (sums) register tile and reads its operands
// as 16-byte vectors: the scores take 8 vector loads per 64 FMAs, the sums 2 to 5
// per 16 to 64.  Row strides are 4 (rows read along d), 8 or 4 (weights) modulo
// the 32 banks, which keeps every access of a warp free of conflicts.  DM is d
// rounded up to 32, 64 or 128.  With one thread per row or column of one value at
// a time the fp32 step of 8 users (10.6K tokens, H = 4, P = 200, d = 64) took
// 1.89 ms, the lse 0.49 ms of it with Q read from global memory by every warp;
// now 0.53 ms.  The forward of one 4096-token user (P = d = 64) went from 65.6 to
// 41.0 us.
template <int DM> struct Ld { static constexpr int v = DM + 4; };
constexpr int kLdPT = 40;  // weights [64 prototypes][tokens]
constexpr int kLdTP = 68;  // weights [32 tokens][prototypes]
constexpr int kTok = 4, kPro = 4;  // scores per thread: kTok tokens x kPro prototypes

// tokens of this thread: tok_of(i) = 8 i + lane % 8; prototypes: pro_of(j)
__device__ __forceinline__ int tok_of(int i) { return 8 * i + int(threadIdx.x & 7); }
__device__ __forceinline__ int pro_of(int j) { return int(threadIdx.x >> 5) * 16 + 4 * j + int((threadIdx.x & 31) >> 3); }

// rows [0, n) of a [*, src_ld] source to [rmax][DM + 4] fp32, zero rows past n
template <typename T, int DM>
__device__ __forceinline__ void stage(float* dst, const T* src, int64_t src_ld, int n, int rmax, int d) {
  constexpr int VN = Vec<T>::n, LD = Ld<DM>::v;
  const int per = d / VN;
  for (int e = threadIdx.x; e < rmax * per; e += SNT) {
    const int r = e / per, c = (e - r * per) * VN;
    float v[VN];
    if (r < n) {
      Vec<T>::load(src + int64_t(r) * src_ld + c, v);
    } else {
#pragma unroll
      for (int k = 0; k < VN; ++k) v[k] = 0.f;
    }
#pragma unroll
    for (int k = 0; k < VN; k += 4)
      *reinterpret_cast<float4*>(dst + r * LD + c + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
  }
}
// the same from fp32 rows whose base may be any 4-byte address (dsketch)
template <int DM>
__device__ __forceinline__ void stage_f32(float* dst, const float* src, int n, int rmax, int d) {
  if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
    stage<float, DM>(dst, src, d, n, rmax, d);
    return;
  }
  for (int e = threadIdx.x; e < rmax * d; e += SNT) {
    const int r = e / d, c = e - r * d;
    dst[r * Ld<DM>::v + c] = r < n ? src[int64_t(r) * d + c] : 0.f;
  }
}

// s[i][j] = X[tok_of(i)] . Y[pro_of(j)], the sum over d in order
template <int DM>
__device__ __forceinline__ void dots(const float* X, const float* Y, int d, float (&s)[kTok][kPro]) {
  constexpr int LD = Ld<DM>::v;
#pragma unroll
  for (int i = 0; i < kTok; ++i)
#pragma unroll
    for (int j = 0; j < kPro; ++j) s[i][j] = 0.f;
  const float* x0 = X + tok_of(0) * LD;
  const float* y0 = Y + pro_of(0) * LD;
#pragma unroll 2
  for (int c = 0; c < d; c += 4) {
    float4 x[kTok], y[kPro];
#pragma unroll
    for (int i = 0; i < kTok; ++i) x[i] = *reinterpret_cast<const float4*>(x0 + 8 * i * LD + c);
#pragma unroll
    for (int j = 0; j < kPro; ++j) y[j] = *reinterpret_cast<const float4*>(y0 + 4 * j * LD + c);
#pragma unroll
    for (int i = 0; i < kTok; ++i)
#pragma unroll
      for (int j = 0; j < kPro; ++j) {
        s[i][j] = fmaf(x[i].x, y[j].x, s[i][j]);
        s[i][j] = fmaf(x[i].y, y[j].y, s[i][j]);
        s[i][j] = fmaf(x[i].z, y[j].z, s[i][j]);
        s[i][j] = fmaf(x[i].w, y[j].w, s[i][j]);
      }
  }
}

// acc[r][..] += sum over k < n of Wt[k][4 rows of this thread] * Z[k][its columns],
// k in order.  NCG column groups share the columns: thread cg owns columns 4 cg + 4
// NCG m (two columns per group when DM / NCG = 2).
template <int DM, int NCG, int LDW>
__device__ __forceinline__ void outer(const float* Wt, int row4, const float* Z, int cg, int n,
                                      float (&acc)[4][DM / NCG]) {
  constexpr int LD = Ld<DM>::v, CP = DM / NCG;
#pragma unroll 4
  for (int k = 0; k < n; ++k) {
    const float4 w = *reinterpret_cast<const float4*>(Wt + k * LDW + row4);
    float z[CP];
    if (CP == 2) {
      const float2 v = *reinterpret_cast<const float2*>(Z + k * LD + 2 * cg);
      z[0] = v.x;
      z[CP - 1] = v.y;
    } else {
#pragma unroll
      for (int m = 0; m < CP / 4; ++m) {
        const float4 v = *reinterpret_cast<const float4*>(Z + k * LD + 4 * cg + 4 * NCG * m);
        z[4 * m] = v.x;
        z[4 * m + 1] = v.y;
        z[4 * m + 2] = v.z;
        z[4 * m + 3] = v.w;
      }
    }
#pragma unroll
    for (int m = 0; m < CP; ++m) {
      acc[0][m] = fmaf(w.x, z[m], acc[0][m]);
      acc[1][m] = fmaf(w.y, z[m], acc[1][m]);
      acc[2][m] = fmaf(w.z, z[m], acc[2][m]);
      acc[3][m] = fmaf(w.w, z[m], acc[3][m]);
    }
  }
}
// the column of acc[.][m] in the layout above
template <int DM, int NCG>
__device__ __forceinline__ int col_of(int cg, int m) {
  constexpr int CP = DM / NCG;
  return CP == 2 ? 2 * cg + m : 4 * cg + 4 * NCG * (m >> 2) + (m & 3);
}

// Row statistics of the scores seen so far, per token of this thread (its share of
// the prototypes): maximum m and sum of exp(s - shift(m)).  An infinite maximum is no
// shift: of -inf alone the sum is 0, and an overflowed score makes it, and the lse, +inf,
// so that the other prototypes' weights are exact zeros; a NaN reaches the sum either way.
struct RowStat {
  float m[kTok], z[kTok];
};
__device__ __forceinline__ float shift(float m) { return fabsf(m) == INFINITY ? 0.f : m; }

// (max, sum) of every token over all threads that share it, to red[2][32]
__device__ __forceinline__ void reduce_stat(RowStat& r, float (*red)[2][32]) {
  const int warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < kTok; ++i) {
#pragma unroll
    for (int o = 8; o < 32; o <<= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, r.m[i], o), z2 = __shfl_xor_sync(0xffffffffu, r.z[i], o);
      const float mm = fmaxf(r.m[i], m2);
      const float za = r.z[i] == 0.f ? 0.f : r.z[i] * expf(r.m[i] - shift(mm));
      const float zb = z2 == 0.f ? 0.f : z2 * expf(m2 - shift(mm));
      r.m[i] = mm;
      r.z[i] = za + zb;
    }
    if ((threadIdx.x & 31) < 8) {
      red[warp][0][tok_of(i)] = r.m[i];
      red[warp][1][tok_of(i)] = r.z[i];
    }
  }
}

// ----------------------------------------------------------- lse (forward)
// lse[t, h] = log sum_j exp(scale q_j . k_t): one block per tile of 32 tokens and
// head, the prototypes in chunks of 64 with a running maximum.
template <typename T, int DM>
__global__ void __launch_bounds__(SNT) simt_lse_kernel(Args a, float* __restrict__ lse) {
  extern __shared__ __align__(16) float smem[];
  __shared__ float red[SNT / 32][2][32];
  if (ws_failed(a.ws)) return;
  constexpr int LD = Ld<DM>::v;
  float* Ks = smem;
  float* Qs = Ks + ST * LD;
  const int64_t tph = reinterpret_cast<const WsHeader*>(a.ws)->tiles_per_head;
  const int64_t t = blockIdx.x;
  if (t >= tph * a.H) return;
  const int d = a.d, P = a.P, H = a.H;
  const TileRef r = locate_tile(t, tph, a.prefix, a.cu, a.B, ST);
  const T* Q = static_cast<const T*>(a.Q) + int64_t(q_row(a, r.b, r.h)) * P * d;
  stage<T, DM>(Ks, static_cast<const T*>(a.K) + (r.tok0 * H + r.h) * int64_t(d), int64_t(H) * d, r.n, ST, d);
  RowStat rs;
#pragma unroll
  for (int i = 0; i < kTok; ++i) {
    rs.m[i] = -INFINITY;
    rs.z[i] = 0.f;
  }
  for (int p0 = 0; p0 < P; p0 += SPB) {
    const int np = min(SPB, P - p0);
    __syncthreads();
    stage<T, DM>(Qs, Q + int64_t(p0) * d, d, np, SPB, d);
    __syncthreads();
    float s[kTok][kPro];
    dots<DM>(Ks, Qs, d, s);
#pragma unroll
    for (int i = 0; i < kTok; ++i) {
      float m = rs.m[i];
#pragma unroll
      for (int j = 0; j < kPro; ++j) {
        s[i][j] = pro_of(j) < np ? s[i][j] * a.scale : -INFINITY;
        m = fmaxf(m, s[i][j]);
      }
      const float sh = shift(m);
      float z = rs.z[i] * expf(rs.m[i] - sh);
#pragma unroll
      for (int j = 0; j < kPro; ++j) z += expf(s[i][j] - sh);
      rs.m[i] = m;
      rs.z[i] = z;
    }
  }
  reduce_stat(rs, red);
  __syncthreads();
  const int tid = threadIdx.x;
  if (tid < r.n) {
    float m = red[0][0][tid];
#pragma unroll
    for (int w = 1; w < SNT / 32; ++w) m = fmaxf(m, red[w][0][tid]);
    float z = 0.f;
#pragma unroll
    for (int w = 0; w < SNT / 32; ++w)
      if (red[w][1][tid] != 0.f) z += red[w][1][tid] * expf(red[w][0][tid] - shift(m));
    lse[(r.tok0 + tid) * H + r.h] = m + logf(z);
  }
}

// --------------------------------------------------- aggregation (forward)
// grid = (W workers, ceil(P/64) prototype blocks).  Each block walks its worker's
// tile range and accumulates sketch rows p0..p0+63 in registers (thread: prototypes
// 4 pg .. 4 pg + 3, columns col_of).
template <typename T, int DM>
__global__ void __launch_bounds__(SNT) simt_fwd_agg_kernel(Args a, const float* __restrict__ lse,
                                                           float* __restrict__ sketch) {
  extern __shared__ __align__(16) float smem[];
  if (ws_failed(a.ws)) return;
  constexpr int LD = Ld<DM>::v, NCG = 8, CP = DM / NCG;
  const int d = a.d, P = a.P, H = a.H;
  float* Qs = smem;              // [64][LD]
  float* Ks = Qs + SPB * LD;     // [32][LD]
  float* Vs = Ks + ST * LD;      // [32][LD]
  float* At = Vs + ST * LD;      // [32][68]
  float* ls = At + ST * kLdTP;   // [32]
  const int64_t tph = reinterpret_cast<const WsHeader*>(a.ws)->tiles_per_head;
  const int64_t total = tph * H;
  const int W = gridDim.x, w = blockIdx.x;
  const int p0 = blockIdx.y * SPB, np = min(SPB, P - p0);
  const int64_t tb = range_begin(total, W, w), te = range_begin(total, W, w + 1);
  if (tb >= te) return;
  const T* K = static_cast<const T*>(a.K);
  const T* V = static_cast<const T*>(a.V);
  const T* Q = static_cast<const T*>(a.Q);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int pg = (lane & 7) + 8 * (warp & 1), cg = (lane >> 3) + 4 * (warp >> 1);
  float acc[4][CP];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int m = 0; m < CP; ++m) acc[r][m] = 0.f;
  int cur_q = -1;
  for (int64_t t = tb; t < te; ++t) {
    const TileRef r = locate_tile(t, tph, a.prefix, a.cu, a.B, ST);
    __syncthreads();
    const int qr = q_row(a, r.b, r.h);
    if (qr != cur_q) {
      stage<T, DM>(Qs, Q + (int64_t(qr) * P + p0) * d, d, np, SPB, d);
      cur_q = qr;
    }
    stage<T, DM>(Ks, K + (r.tok0 * H + r.h) * int64_t(d), int64_t(H) * d, r.n, ST, d);
    stage<T, DM>(Vs, V + (r.tok0 * H + r.h) * int64_t(d), int64_t(H) * d, r.n, ST, d);
    if (tid < ST) ls[tid] = tid < r.n ? lse[(r.tok0 + tid) * H + r.h] : 0.f;
    __syncthreads();
    float s[kTok][kPro];
    dots<DM>(Ks, Qs, d, s);
#pragma unroll
    for (int i = 0; i < kTok; ++i) {
      const int tk = tok_of(i);
      const float l = ls[tk];
#pragma unroll
      for (int j = 0; j < kPro; ++j)
        At[tk * kLdTP + pro_of(j)] = (tk < r.n && pro_of(j) < np) ? expf(s[i][j] * a.scale - l) : 0.f;
    }
    __syncthreads();
    outer<DM, NCG, kLdTP>(At, 4 * pg, Vs, cg, r.n, acc);
    if (t + 1 == te || t + 1 == r.seg1) {
      float* dst;
      if (r.seg0 >= tb && r.seg1 <= te) {
        dst = sketch + ((int64_t(r.b) * H + r.h) * P + p0) * d;
      } else {
        const int slot = partial_slot(total, W, w, r.seg0);
        dst = a.partial + ((int64_t(w) * 2 + slot) * P + p0) * d;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int m = 0; m < CP; ++m) {
          const int c = col_of<DM, NCG>(cg, m);
          if (c < d && 4 * pg + k < np) dst[int64_t(4 * pg + k) * d + c] = acc[k][m];
          acc[k][m] = 0.f;
        }
    }
  }
}

// ----------------------------------------------------- backward per token
// One block per (head, user, tile of 32 tokens): dV, D_i = dV_i . v_i, dK.
// Thread: tokens 4 tg .. 4 tg + 3 and columns col_of of both sums.
template <typename T, int DM>
__global__ void __launch_bounds__(SNT) simt_bwd_tokens_kernel(Args a, const float* __restrict__ dsk,
                                                              const float* __restrict__ lse,
                                                              T* __restrict__ dK, T* __restrict__ dV,
                                                              float* __restrict__ Dco) {
  extern __shared__ __align__(16) float smem[];
  __shared__ float red[SNT / 32][ST];
  if (ws_failed(a.ws)) return;
  constexpr int LD = Ld<DM>::v, NCG = 16, CP = DM / NCG;
  const int d = a.d, P = a.P, H = a.H;
  const int64_t tph = reinterpret_cast<const WsHeader*>(a.ws)->tiles_per_head;
  const int64_t t = blockIdx.x;
  if (t >= tph * H) return;
  float* Ks = smem;              // [32][LD]
  float* Vs = Ks + ST * LD;      // [32][LD]
  float* Qs = Vs + ST * LD;      // [64][LD]
  float* Gs = Qs + SPB * LD;     // [64][LD]
  float* As = Gs + SPB * LD;     // [64][40]
  float* ls = As + SPB * kLdPT;  // [32]
  float* Ds = ls + ST;           // [32]
  const TileRef r = locate_tile(t, tph, a.prefix, a.cu, a.B, ST);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tg = lane & 7, cg = (lane >> 3) + 4 * warp;
  stage<T, DM>(Ks, static_cast<const T*>(a.K) + (r.tok0 * H + r.h) * int64_t(d), int64_t(H) * d, r.n, ST, d);
  stage<T, DM>(Vs, static_cast<const T*>(a.V) + (r.tok0 * H + r.h) * int64_t(d), int64_t(H) * d, r.n, ST, d);
  if (tid < ST) ls[tid] = tid < r.n ? lse[(r.tok0 + tid) * H + r.h] : 0.f;
  const T* Q = static_cast<const T*>(a.Q) + int64_t(q_row(a, r.b, r.h)) * P * d;
  const float* G = dsk + (int64_t(r.b) * H + r.h) * int64_t(P) * d;
  float acc[4][CP];
  auto clear = [&]() {
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int m = 0; m < CP; ++m) acc[k][m] = 0.f;
  };
  auto put = [&](T* out, float mul) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (4 * tg + k >= r.n) continue;
      T* row = out + ((r.tok0 + 4 * tg + k) * H + r.h) * int64_t(d);
#pragma unroll
      for (int m = 0; m < CP; ++m) {
        const int c = col_of<DM, NCG>(cg, m);
        if (c < d) st_from_f32(row + c, acc[k][m] * mul);
      }
    }
  };
  clear();
  // pass 1: dV_i = sum_j A[j,i] G_j
  for (int pc = 0; pc < P; pc += SPB) {
    const int np = min(SPB, P - pc);
    __syncthreads();
    stage<T, DM>(Qs, Q + int64_t(pc) * d, d, np, SPB, d);
    stage_f32<DM>(Gs, G + int64_t(pc) * d, np, SPB, d);
    __syncthreads();
    float s[kTok][kPro];
    dots<DM>(Ks, Qs, d, s);
#pragma unroll
    for (int i = 0; i < kTok; ++i) {
      const int tk = tok_of(i);
#pragma unroll
      for (int j = 0; j < kPro; ++j)
        As[pro_of(j) * kLdPT + tk] = (tk < r.n && pro_of(j) < np) ? expf(s[i][j] * a.scale - ls[tk]) : 0.f;
    }
    __syncthreads();
    outer<DM, NCG, kLdPT>(As, 4 * tg, Gs, cg, np, acc);
  }
  {
    float part[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      part[k] = 0.f;
#pragma unroll
      for (int m = 0; m < CP; ++m) {
        const int c = col_of<DM, NCG>(cg, m);
        if (c < d) part[k] = fmaf(acc[k][m], Vs[(4 * tg + k) * LD + c], part[k]);
      }
      part[k] += __shfl_xor_sync(0xffffffffu, part[k], 8);
      part[k] += __shfl_xor_sync(0xffffffffu, part[k], 16);
      if (lane < 8) red[warp][4 * tg + k] = part[k];
    }
    put(dV, 1.f);
    __syncthreads();
    if (tid < ST) {
      const float D = (red[0][tid] + red[1][tid]) + (red[2][tid] + red[3][tid]);
      Ds[tid] = D;
      if (tid < r.n) Dco[(r.tok0 + tid) * H + r.h] = D;
    }
  }
  clear();
  // pass 2: dS = A o (G V^T - D), dK_i = scale sum_j dS[j,i] Q_j
  for (int pc = 0; pc < P; pc += SPB) {
    const int np = min(SPB, P - pc);
    __syncthreads();
    if (P > SPB) {  // a single chunk is still there
      stage<T, DM>(Qs, Q + int64_t(pc) * d, d, np, SPB, d);
      stage_f32<DM>(Gs, G + int64_t(pc) * d, np, SPB, d);
      __syncthreads();
    }
    float s[kTok][kPro], g[kTok][kPro];
    dots<DM>(Ks, Qs, d, s);
    dots<DM>(Vs, Gs, d, g);
#pragma unroll
    for (int i = 0; i < kTok; ++i) {
      const int tk = tok_of(i);
#pragma unroll
      for (int j = 0; j < kPro; ++j) {
        const float A = expf(s[i][j] * a.scale - ls[tk]);
        As[pro_of(j) * kLdPT + tk] = (tk < r.n && pro_of(j) < np) ? A * (g[i][j] - Ds[tk]) : 0.f;
      }
    }
    __syncthreads();
    outer<DM, NCG, kLdPT>(As, 4 * tg, Qs, cg, np, acc);
  }
  put(dK, a.scale);
}

// ------------------------------------------------------------ backward dQ
// grid = (W workers, ceil(P/64)); per worker and head one fp32 partial of
// dQ[h] = scale sum_i dS[:, i] K_i, summed over the workers later.
template <typename T, int DM>
__global__ void __launch_bounds__(SNT) simt_bwd_dq_kernel(Args a, const float* __restrict__ dsk,
                                                          const float* __restrict__ lse,
                                                          const float* __restrict__ Dco) {
  extern __shared__ __align__(16) float smem[];
  if (ws_failed(a.ws)) return;
  constexpr int LD = Ld<DM>::v, NCG = 8, CP = DM / NCG;
  const int d = a.d, P = a.P, H = a.H;
  float* Qs = smem;              // [64][LD]
  float* Gs = Qs + SPB * LD;     // [64][LD]
  float* Ks = Gs + SPB * LD;     // [32][LD]
  float* Vs = Ks + ST * LD;      // [32][LD]
  float* At = Vs + ST * LD;      // [32][68]
  float* ls = At + ST * kLdTP;   // [32]
  float* Ds = ls + ST;           // [32]
  const int64_t tph = reinterpret_cast<const WsHeader*>(a.ws)->tiles_per_head;
  const int64_t total = tph * H;
  const int W = gridDim.x, w = blockIdx.x;
  const int p0 = blockIdx.y * SPB, np = min(SPB, P - p0);
  const int64_t tb = range_begin(total, W, w), te = range_begin(total, W, w + 1);
  if (tb >= te) return;
  const T* K = static_cast<const T*>(a.K);
  const T* V = static_cast<const T*>(a.V);
  const T* Q = static_cast<const T*>(a.Q);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int pg = (lane & 7) + 8 * (warp & 1), cg = (lane >> 3) + 4 * (warp >> 1);
  float acc[4][CP];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int m = 0; m < CP; ++m) acc[k][m] = 0.f;
  int cur_h = -1, cur_b = -1, cur_q = -1;
  for (int64_t t = tb; t < te; ++t) {
    const TileRef r = locate_tile(t, tph, a.prefix, a.cu, a.B, ST);
    __syncthreads();
    const int qr = q_row(a, r.b, r.h);
    if (qr != cur_q) stage<T, DM>(Qs, Q + (int64_t(qr) * P + p0) * d, d, np, SPB, d);
    cur_q = qr;
    if (r.h != cur_h || r.b != cur_b)
      stage_f32<DM>(Gs, dsk + ((int64_t(r.b) * H + r.h) * P + p0) * d, np, SPB, d);
    cur_h = r.h;
    cur_b = r.b;
    stage<T, DM>(Ks, K + (r.tok0 * H + r.h) * int64_t(d), int64_t(H) * d, r.n, ST, d);
    stage<T, DM>(Vs, V + (r.tok0 * H + r.h) * int64_t(d), int64_t(H) * d, r.n, ST, d);
    if (tid < ST) {
      ls[tid] = tid < r.n ? lse[(r.tok0 + tid) * H + r.h] : 0.f;
      Ds[tid] = tid < r.n ? Dco[(r.tok0 + tid) * H + r.h] : 0.f;
    }
    __syncthreads();
    float s[kTok][kPro], g[kTok][kPro];
    dots<DM>(Ks, Qs, d, s);
    dots<DM>(Vs, Gs, d, g);
#pragma unroll
    for (int i = 0; i < kTok; ++i) {
      const int tk = tok_of(i);
      const float l = ls[tk], D = Ds[tk];
#pragma unroll
      for (int j = 0; j < kPro; ++j) {
        const float A = expf(s[i][j] * a.scale - l);
        At[tk * kLdTP + pro_of(j)] = (tk < r.n && pro_of(j) < np) ? A * (g[i][j] - D) : 0.f;
      }
    }
    __syncthreads();
    outer<DM, NCG, kLdTP>(At, 4 * pg, Ks, cg, r.n, acc);
    // flush where the row of Q changes: at a head's end (shared queries: the
    // worker's partial of head h) or at a user segment's end (per-user queries:
    // dQ[b, h] when this worker holds the whole segment, else its partial slot)
    const bool flush = a.uq ? (t + 1 == te || t + 1 == r.seg1) : (t + 1 == te || (t + 1) / tph != t / tph);
    if (flush) {
      float* dst;
      if (!a.uq) {
        dst = a.dq_partial + ((int64_t(w) * H + r.h) * P + p0) * d;
      } else if (r.seg0 >= tb && r.seg1 <= te) {
        dst = a.dq_user + ((int64_t(r.b) * H + r.h) * P + p0) * d;
      } else {
        dst = a.partial + ((int64_t(w) * 2 + partial_slot(total, W, w, r.seg0)) * P + p0) * d;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int m = 0; m < CP; ++m) {
          const int c = col_of<DM, NCG>(cg, m);
          if (c < d && 4 * pg + k < np) dst[int64_t(4 * pg + k) * d + c] = acc[k][m] * a.scale;
          acc[k][m] = 0.f;
        }
    }
  }
}

// ------------------------------------------------------------------ launchers
cudaError_t launch_plan(const Args& a, int T, cudaStream_t st) {
  plan_kernel<<<1, 1024, 0, st>>>(a.cu, a.B, a.N, T, a.ws, a.prefix, wait_limit_ns());
  return cudaGetLastError();
}

// f(element type, DM) for the call's dtype and width
template <class F>
static cudaError_t with_types(const Args& a, F&& f) {
  auto width = [&](auto t) {
    if (a.d <= 32) return f(t, std::integral_constant<int, 32>());
    if (a.d <= 64) return f(t, std::integral_constant<int, 64>());
    return f(t, std::integral_constant<int, 128>());
  };
  return a.dt == SA_BF16 ? width(__nv_bfloat16()) : width(float());
}

template <class Fn, class... Xs>
static cudaError_t run(Fn* fn, dim3 grid, size_t floats, cudaStream_t st, Xs... xs) {
  const size_t sm = sizeof(float) * floats;
  const cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void*>(fn),
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm));
  if (e != cudaSuccess) return e;
  fn<<<grid, SNT, sm, st>>>(xs...);
  return cudaGetLastError();
}

// one block per tile: H x ceil(L_b / 32) summed over the users, of whom at most N have
// tokens, is at most this
static unsigned max_tiles(const Args& a) {
  const int64_t users = a.N < a.B ? a.N : a.B;
  return unsigned(int64_t(a.H) * ((a.N + (ST - 1) * users) / ST));
}

cudaError_t launch_simt_lse(const Args& a, float* lse, cudaStream_t st) {
  if (a.N == 0) return cudaSuccess;
  return with_types(a, [&](auto t, auto dm) {
    using T = decltype(t);
    constexpr int DM = decltype(dm)::value;
    return run(&simt_lse_kernel<T, DM>, dim3(max_tiles(a)), size_t(ST + SPB) * Ld<DM>::v, st, a, lse);
  });
}

cudaError_t launch_simt_fwd(const Args& a, int W, const float* lse, float* sketch, cudaStream_t st) {
  return with_types(a, [&](auto t, auto dm) {
    using T = decltype(t);
    constexpr int DM = decltype(dm)::value;
    return run(&simt_fwd_agg_kernel<T, DM>, dim3(W, (a.P + SPB - 1) / SPB),
               size_t(SPB + 2 * ST) * Ld<DM>::v + ST * kLdTP + ST, st, a, lse, sketch);
  });
}

cudaError_t launch_simt_bwd_tokens(const Args& a, const float* dsk, const float* lse, void* dK, void* dV,
                                   float* Dco, cudaStream_t st) {
  if (a.N == 0) return cudaSuccess;
  return with_types(a, [&](auto t, auto dm) {
    using T = decltype(t);
    constexpr int DM = decltype(dm)::value;
    return run(&simt_bwd_tokens_kernel<T, DM>, dim3(max_tiles(a)),
               size_t(2 * ST + 2 * SPB) * Ld<DM>::v + SPB * kLdPT + 2 * ST, st, a, dsk, lse, static_cast<T*>(dK),
               static_cast<T*>(dV), Dco);
  });
}

cudaError_t launch_simt_bwd_dq(const Args& a, int W, const float* dsk, const float* lse, const float* Dco,
                               cudaStream_t st) {
  return with_types(a, [&](auto t, auto dm) {
    using T = decltype(t);
    constexpr int DM = decltype(dm)::value;
    return run(&simt_bwd_dq_kernel<T, DM>, dim3(W, (a.P + SPB - 1) / SPB),
               size_t(2 * ST + 2 * SPB) * Ld<DM>::v + ST * kLdTP + 2 * ST, st, a, dsk, lse, Dco);
  });
}

int simt_tile_tokens() { return ST; }
int simt_workers(int num_sms, int P) {
  const int nb = (P + SPB - 1) / SPB;
  int w = (3 * num_sms + nb - 1) / nb;
  return w < 1 ? 1 : w > kMaxWorkers ? kMaxWorkers : w;
}

}  // namespace sa
