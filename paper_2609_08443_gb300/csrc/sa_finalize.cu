// Sums of the pieces that workers leave behind: the sketch (or per-user dQ) of
// every (user, head) segment cut by a worker boundary, the per-worker dQ of
// every head, and the token-wise variant's (sum, shift, weight) pieces.
//
// What bounds it: the bytes of the pieces are few (a 16-user batch of 100K
// tokens at P = 512, d = 128 leaves 58 MB), so the time is latency.  One block
// per (user, head), each thread adding its element's pieces one after the
// other, took 82 us for one user of 1531 tokens (8 blocks, 19 pieces each) and
// 282 us for one fp32 user (1 block, 128 pieces), more than the forward itself.
// Here every block first lists the cut segments, one thread per worker boundary
// (each segment at the first boundary inside it, so all blocks hold the same
// list), and the list's (segment, column range) items are dealt to all blocks.  Segments of up to
// kFewPieces pieces (a long batch) give each thread one column and its pieces
// in order; longer chains (a short batch) are split over the block's eight
// warps, whose sums are added in warp order.  Token-wise lse and sketches feed the backward's
// differences, where another order of the sums shows as flipped bf16 roundings: their
// pieces are always added in order, relative to the largest shift, one thread per column
// (a narrow shape, P = 1 and d = 8 say, leaves the whole chain to two threads, as the
// kernel before this did).  All orders depend
// only on the plan, so the result stays bitwise reproducible.  Measured, the
// calls with the old and with this kernel and nothing else changed: one user of 1531
// tokens 69.6 and 32.0 us, one fp32 user of 4096 tokens 226 and 65.6 us, the token-wise
// step of 12 users (P = 512, d = 128, 215K tokens) 2.99 and 2.05 ms, of which the sum
// itself 971 us before.
#include "sa_kernels.cuh"
#include "sa_tc_common.cuh"

namespace sa {

namespace {

constexpr int kFinThreads = 256;
constexpr int kFinWarps = kFinThreads / 32;
// Up to four pieces in order, more split.  Forwards at d = 64, P = 256 (at d = 128,
// P = 512), us, in order and split: two or three pieces a segment 68.5 and 81.6 (92 and
// 119), five 49.7 and 55.7 (89 and 102), ten 48.4 and 51.1, nineteen 33.4 and 33.4.  The
// split pays for chains of a hundred (one fp32 user: 226 and 65.6 us with the whole
// kernel).  The line could lie at 16; it is left at 4, where every sum keeps its order.
constexpr int kFewPieces = 4;

enum Kind { kSketch = 0, kHeadDq = 1, kTokenwise = 2 };

struct FinArgs {
  const void* ws;
  const int64_t* prefix;
  int B, H, P, d, W;
  const float* src;        // pieces: [W][2][P][d] per cut segment, [W][H][P][d] per head
  const float2* stat;      // token-wise: [W][2][P] (shift, weight sum) of each piece
  float* out;              // [B][H][P][d] (dQ per head: [H][P][d])
  float* lse;              // token-wise: [B][H][P]
};

template <int V> struct Col;
template <> struct Col<4> {
  float x[4];
  __device__ __forceinline__ void load(const float* p) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
  }
  __device__ __forceinline__ void store(float* p) const {
    *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
  }
};
template <> struct Col<1> {
  float x[1];
  __device__ __forceinline__ void load(const float* p) { x[0] = *p; }
  __device__ __forceinline__ void store(float* p) const { *p = x[0]; }
};

// a cut segment (or a head): its row in `out`, its first tile and the workers
// that hold a piece; items before its own in the item list
struct Seg {
  int64_t seg0;
  int row, g0, g1, item0;
};

// Largest g with rb[g] <= t (rb[0] = 0 <= t < rb[W]): the worker that holds tile t.
__device__ __forceinline__ int holder(const int64_t* rb, int W, int64_t t) {
  int lo = 0, hi = W - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (rb[mid] <= t) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Sum of pieces.  Token-wise pieces carry a shift m and a weight sum l (l < 0: no
// piece); the sum is relative to M, the largest shift of the segment.
template <int V, int KIND>
struct Acc {
  Col<V> s;
  float M, L;
  __device__ __forceinline__ Acc() : M(-INFINITY), L(0.f) {
#pragma unroll
    for (int k = 0; k < V; ++k) s.x[k] = 0.f;
  }
  __device__ __forceinline__ void add(const Col<V>& v, float m, float l) {
    if (KIND != kTokenwise) {
#pragma unroll
      for (int k = 0; k < V; ++k) s.x[k] += v.x[k];
      return;
    }
    if (l < 0.f) return;
    const float f = expf(m - M);
    L = fmaf(l, f, L);
#pragma unroll
    for (int k = 0; k < V; ++k) s.x[k] = fmaf(v.x[k], f, s.x[k]);
  }
};

// Users without tokens get zero rows (token-wise: lse = -inf).  Each is cut into slices, a
// head's worth or less but a store of every thread at least, so that a few users with much
// to clear still take the whole chip; the threads of a block look at its next 256 (user,
// slice) items at once.  A forward
// call of one such user with 64 heads, P = 2048, d = 128 (67 MB): 1022 us when one block
// cleared it, 18.9 us this way.
template <int V, int KIND>
__device__ __forceinline__ void zero_empty_users(const FinArgs& a) {
  __shared__ uint32_t empty_s[kFinWarps];
  const int tid = threadIdx.x, grid = int(gridDim.x);
  const int64_t len = int64_t(a.H) * a.P * a.d;
  const int slices = int(min(int64_t(max(a.H, (grid + a.B - 1) / a.B)), max(int64_t(1), len / (kFinThreads * V))));
  const int64_t per = ((len + slices - 1) / slices + 3) & ~int64_t(3), items = int64_t(a.B) * slices;
  for (int64_t base = blockIdx.x; base < items; base += int64_t(grid) * kFinThreads) {
    const int64_t mine = base + int64_t(tid) * grid;
    const int64_t b = mine / slices;
    const bool empty = mine < items && a.prefix[b] == a.prefix[b + 1];
    const uint32_t m = __ballot_sync(0xffffffffu, empty);
    if ((tid & 31) == 0) empty_s[tid >> 5] = m;
    if (!__syncthreads_or(empty)) continue;
    for (int w = 0; w < kFinWarps; ++w)
      for (uint32_t left = empty_s[w]; left != 0u; left &= left - 1u) {
        const int64_t it = base + int64_t(32 * w + __ffs(left) - 1) * grid;
        const int64_t user = it / slices;
        const int s = int(it - user * slices);
        Col<V> zero;
#pragma unroll
        for (int k = 0; k < V; ++k) zero.x[k] = 0.f;
        float* out = a.out + user * len;
        for (int64_t e = s * per + int64_t(tid) * V; e < min(len, (s + 1) * per); e += kFinThreads * V)
          zero.store(out + e);
        if (KIND == kTokenwise)
          for (int j = s * kFinThreads + tid; j < a.H * a.P; j += slices * kFinThreads)
            a.lse[user * a.H * a.P + j] = -INFINITY;
      }
    __syncthreads();
  }
}

template <int V, int KIND>
__global__ void __launch_bounds__(kFinThreads) finalize_kernel(FinArgs a) {
  __shared__ int64_t rb[kMaxWorkers + 1];
  __shared__ Seg segs[kMaxWorkers];
  __shared__ int nitems_s;
  __shared__ float red[kFinWarps][32][V];
  if (ws_failed(a.ws)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t tph = reinterpret_cast<const WsHeader*>(a.ws)->tiles_per_head;
  const int64_t total = tph * a.H;
  const int64_t PD = int64_t(a.P) * a.d;
  const int W = a.W;
  if (KIND == kHeadDq) {
    if (total == 0) {
      for (int64_t e = blockIdx.x * int64_t(kFinThreads) + tid; e < a.H * PD; e += int64_t(gridDim.x) * kFinThreads)
        a.out[e] = 0.f;
      return;
    }
  } else {
    zero_empty_users<V, KIND>(a);
    if (total == 0) return;
  }
  for (int w = tid; w <= W; w += kFinThreads) rb[w] = range_begin(total, W, w);
  __syncthreads();
  if (KIND == kHeadDq) {
    for (int h = tid; h < a.H; h += kFinThreads)
      segs[h] = Seg{int64_t(h) * tph, h, holder(rb, W, int64_t(h) * tph), holder(rb, W, int64_t(h + 1) * tph - 1), 0};
  } else {
    // boundary w opens the cut of a segment if its tile lies inside the segment
    // and the boundary before it does not
    for (int w = tid; w < W; w += kFinThreads) {
      segs[w].row = -1;
      const int64_t t = rb[w];
      if (w == 0 || t >= total || t == rb[w + 1]) continue;
      const int64_t h = t / tph, r = t - h * tph;
      const int b = find_user(a.prefix, a.B, r);
      const int64_t s0 = h * tph + a.prefix[b], s1 = h * tph + a.prefix[b + 1];
      if (t == s0) continue;
      int p = w - 1;
      while (p > 0 && rb[p] == t) --p;
      if (rb[p] > s0) continue;
      segs[w] = Seg{s0, b * a.H + int(h), p, holder(rb, W, s1 - 1), 0};
    }
  }
  __syncthreads();
  const int nseg = KIND == kHeadDq ? a.H : W;
  auto in_order = [](const Seg& g) { return KIND == kTokenwise || g.g1 - g.g0 < kFewPieces; };
  const int cols = int(PD / V);
  if (warp == 0) {  // exclusive scan of the items per segment
    int carry = 0;
    for (int s = 0; s < nseg; s += 32) {
      int n = 0;
      if (s + lane < nseg && segs[s + lane].row >= 0) {
        const int per = in_order(segs[s + lane]) ? kFinThreads : 32;
        n = (cols + per - 1) / per;
      }
      int x = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (s + lane < nseg) segs[s + lane].item0 = carry + x - n;
      carry += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) nitems_s = carry;
  }
  __syncthreads();
  const int nitems = nitems_s;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    int lo = 0, hi = nseg - 1;  // last entry with item0 <= it (entries without items share the next one's)
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (segs[mid].item0 <= it) lo = mid; else hi = mid - 1;
    }
    const Seg sg = segs[lo];
    const bool few = in_order(sg);
    const int col = (it - sg.item0) * (few ? kFinThreads : 32) + (few ? tid : lane);
    const bool in = col < cols;
    const int64_t e = int64_t(col) * V;
    const int j = in && KIND == kTokenwise ? int(e / a.d) : 0;
    // index of worker g's piece, in units of one [P][d] block
    auto piece = [&](int g) {
      return KIND == kHeadDq ? int64_t(g) * a.H + sg.row : int64_t(g) * 2 + (rb[g] >= sg.seg0 ? 0 : 1);
    };
    Acc<V, KIND> acc;
    if (KIND == kTokenwise && in) {
#pragma unroll 8
      for (int g = sg.g0; g <= sg.g1; ++g)
        if (rb[g] != rb[g + 1]) acc.M = fmaxf(acc.M, a.stat[piece(g) * a.P + j].x);
    }
    constexpr int U = KIND == kTokenwise ? 8 : 4;
    auto run = [&](int ga, int gb) {  // pieces [ga, gb), U loads in flight
      for (int g = ga; g < gb; g += U) {
        Col<V> v[U];
        float2 st[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
          const bool have = in && g + k < gb && rb[g + k] != rb[g + k + 1];
#pragma unroll
          for (int q = 0; q < V; ++q) v[k].x[q] = 0.f;
          st[k] = make_float2(0.f, -1.f);
          if (have) {
            const int64_t pc = piece(g + k);
            v[k].load(a.src + pc * PD + e);
            if (KIND == kTokenwise) st[k] = a.stat[pc * a.P + j];
          }
        }
#pragma unroll
        for (int k = 0; k < U; ++k) acc.add(v[k], st[k].x, st[k].y);
      }
    };
    auto write = [&]() {
      if (!in) return;
      if (KIND == kTokenwise) {
#pragma unroll
        for (int k = 0; k < V; ++k) acc.s.x[k] = acc.s.x[k] / acc.L;
        if (e == int64_t(j) * a.d) a.lse[int64_t(sg.row) * a.P + j] = acc.M + logf(acc.L);
      }
      acc.s.store(a.out + int64_t(sg.row) * PD + e);
    };
    if (few) {
      run(sg.g0, sg.g1 + 1);
      write();
      continue;
    }
    const int per = (sg.g1 - sg.g0 + kFinWarps) / kFinWarps;  // ceil of (g1 - g0 + 1) / warps
    const int ga = sg.g0 + warp * per;
    run(ga, min(ga + per, sg.g1 + 1));
#pragma unroll
    for (int k = 0; k < V; ++k) red[warp][lane][k] = acc.s.x[k];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
      for (int w = 1; w < kFinWarps; ++w) {
        Col<V> v;
#pragma unroll
        for (int k = 0; k < V; ++k) v.x[k] = red[w][lane][k];
        acc.add(v, 0.f, 0.f);
      }
      write();
    }
    __syncthreads();
  }
}

template <int KIND>
cudaError_t launch_finalize(const FinArgs& f, cudaStream_t st) {
  const int blocks = 4 * tcc::device_sm_count();
  const bool vec = (f.d & 3) == 0 && ((reinterpret_cast<uintptr_t>(f.src) | reinterpret_cast<uintptr_t>(f.out)) & 15) == 0;
  if (vec) finalize_kernel<4, KIND><<<blocks, kFinThreads, 0, st>>>(f);
  else finalize_kernel<1, KIND><<<blocks, kFinThreads, 0, st>>>(f);
  return cudaGetLastError();
}

FinArgs fin_args(const Args& a, int W, const float* src, float* out) {
  return FinArgs{a.ws, a.prefix, a.B, a.H, a.P, a.d, W, src, nullptr, out, nullptr};
}

}  // namespace

cudaError_t launch_finalize_sketch(const Args& a, int W, float* sketch, cudaStream_t st) {
  return launch_finalize<kSketch>(fin_args(a, W, a.partial, sketch), st);
}

cudaError_t launch_finalize_dq(const Args& a, int W, float* dQ, cudaStream_t st) {
  return launch_finalize<kHeadDq>(fin_args(a, W, a.dq_partial, dQ), st);
}

cudaError_t launch_tw_finalize(const Args& a, int W, const float2* stat_part, float* sketch, float* lse_tok,
                               cudaStream_t st) {
  FinArgs f = fin_args(a, W, a.partial, sketch);
  f.stat = stat_part;
  f.lse = lse_tok;
  return launch_finalize<kTokenwise>(f, st);
}

}  // namespace sa
