// Pieces shared by the tensor-core kernels: the tile walker every warp role
// uses to follow its worker's range, TMA tensor maps, TMEM sizing and the
// epilogue that stores a sketch block from TMEM.
#pragma once
#include <cuda.h>

#include "sa_kernels.cuh"
#include "sa_ptx.cuh"

namespace sa {
namespace tcc {

constexpr int T = 128;           // tokens per tile = UMMA M
constexpr int kThreads = 384;    // 12 warps
constexpr int kSoftWarp0 = 4;    // warps 4..11: softmax / epilogue
constexpr int kSoftWarps = 8;

__host__ __device__ constexpr int tmem_cols_for(int c) {
  return c <= 32 ? 32 : c <= 64 ? 64 : c <= 128 ? 128 : c <= 256 ? 256 : 512;
}

// Follows worker tiles [tb, te) in (head, user, tile) order; all warp roles
// construct their own walker and see the same sequence.
struct TileWalker {
  const int64_t* prefix;
  const int32_t* cu;
  int B, Tt, H, uq;
  int64_t tph, t, tb, te;
  int h, b;
  int qk;  // row of Q this tile reads: h (shared queries) or b*H + h (per user)
  int64_t k, nk, tok0, seg0, seg1;
  int64_t cub, Lb;  // cu[b] and L_b of the current user, read once per segment
  int n;
  bool seg_first, seg_last;

  __device__ TileWalker(const Args& a, int64_t tb_, int64_t te_, int T_)
      : prefix(a.prefix), cu(a.cu), B(a.B), Tt(T_), H(a.H), uq(a.uq), t(tb_), tb(tb_), te(te_) {
    tph = reinterpret_cast<const WsHeader*>(a.ws)->tiles_per_head;
    if (t < te) relocate();
  }
  __device__ void relocate() { set(locate_tile(t, tph, prefix, cu, B, Tt)); }
  __device__ void set(const TileRef& r) {
    h = r.h;
    b = r.b;
    qk = uq ? b * H + h : h;
    seg0 = r.seg0;
    seg1 = r.seg1;
    nk = seg1 - seg0;
    k = t - seg0;
    cub = r.tok0 - k * Tt;
    Lb = r.L;
    fields();
  }
  __device__ void fields() {
    tok0 = cub + k * Tt;
    const int64_t left = Lb - k * Tt;
    n = int(left < Tt ? left : Tt);
    seg_first = (k == 0) || (t == tb);
    seg_last = (k == nk - 1) || (t == te - 1);
  }
  // First token, size and head of the tile after this one (n = 0 past the range).
  __device__ void peek_next(int64_t& tok0_n, int& n_n, int& h_n) const {
    int qk_n;
    peek_next(tok0_n, n_n, h_n, qk_n);
  }
  // ... and the row of Q it reads (qk_n = qk past the range)
  __device__ void peek_next(int64_t& tok0_n, int& n_n, int& h_n, int& qk_n) const {
    if (t + 1 >= te) {
      tok0_n = 0;
      n_n = 0;
      h_n = h;
      qk_n = qk;
      return;
    }
    if (k + 1 < nk) {
      tok0_n = tok0 + Tt;
      const int64_t left = Lb - (k + 1) * Tt;
      n_n = int(left < Tt ? left : Tt);
      h_n = h;
      qk_n = qk;
    } else {
      const TileRef r = locate_next_segment(t + 1, h, b, tph, prefix, cu, B, Tt);
      tok0_n = r.tok0;
      n_n = r.n;
      h_n = r.h;
      qk_n = uq ? r.b * H + r.h : r.h;
    }
  }
  __device__ void next() {
    ++t;
    if (t >= te) return;
    if (k + 1 < nk) {
      ++k;
      fields();
    } else {
      set(locate_next_segment(t, h, b, tph, prefix, cu, B, Tt));
    }
  }
};

// The same walk with the binary search at every segment end instead of the
// forward scan.  The token-wise forward uses it: with the scan inlined in its
// roles' per-tile loops ptxas spilled more of its registers, and the 100K-token
// workload's token-wise forward ran 14 % slower; its segments are long there.
struct TileWalkerSearch : TileWalker {
  using TileWalker::TileWalker;
  __device__ void next() {
    ++t;
    if (t >= te) return;
    if (k + 1 < nk) {
      ++k;
      fields();
    } else {
      relocate();
    }
  }
};

// Whether this CTA leaves before any set-up: the call has failed, or the base is not on
// the 1024 bytes that the 128-byte swizzle atoms need (recorded under `site`).  Another CTA
// of the same launch may set the error word, when a wait gives up, between two threads'
// reads of it, so the CTA votes: all of its threads leave or none, and no warp runs on
// without the barriers and the tensor memory that another one was to set up.
__device__ __forceinline__ bool cta_leaves(void* ws, uint32_t smem_base, uint32_t site) {
  const bool misaligned = (smem_base & 1023u) != 0u;
  if (misaligned && threadIdx.x == 0) ws_set_error(ws, SA_ERR_CUDA, site);
  return __syncthreads_or(misaligned || ws_failed(ws)) != 0;
}

// The lse of one (token, head).  Volatile: it may lie where the token side writes the pair
// (lse log2 e, D) of the same token later, so it is read exactly once, before.
__device__ __forceinline__ float load_token_lse(const float* lse, const Args& a, int64_t tok, int h) {
  float x;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(x) : "l"(lse + tok * a.lse_ts + h * a.lse_hs));
  return x;
}

// Where a worker's dQ block of prototypes [p0, p0 + PS) for the tiles ending
// at walker position w goes.  Shared queries: the worker's partial of head h
// ([W][H][P][d], summed over workers afterwards).  Per-user queries: dQ[b, h]
// itself when the worker holds the whole (user, head) segment, else the
// worker's partial slot of that segment ([W][2][P][d], summed like the sketch).
__device__ __forceinline__ float* dq_block_dst(const Args& a, int wk, int W, int64_t total, const TileWalker& w,
                                               int p0, int D) {
  if (!a.uq) return a.dq_partial + ((int64_t(wk) * a.H + w.h) * a.P + p0) * D;
  if (w.seg0 >= w.tb && w.seg1 <= w.te) return a.dq_user + ((int64_t(w.b) * a.H + w.h) * a.P + p0) * D;
  return a.partial + ((int64_t(wk) * 2 + partial_slot(total, W, wk, w.seg0)) * a.P + p0) * D;
}

__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
  if (ptx::mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = ptx::globaltimer();
  while (!ptx::mbar_try_wait(bar, parity))
    if (ptx::globaltimer() - t0 > limit_ns) return false;
  return true;
}

// 32 consecutive floats of one row, which may start on any 4 bytes (the caller's sketch).
// The 32 threads of a warp write 32 different rows, so an instruction touches 32 lines
// whatever its width: 32-byte stores, which need their alignment, take half as many as
// 16-byte ones.  Forward kernel, 1024 short users
// and one of 1M tokens (P = 256, d = 64): 1.93 ms with 16-byte stores, 1.72 ms with these.
__device__ __forceinline__ void store_row32(float* dst, const float* v) {
  if ((reinterpret_cast<uintptr_t>(dst) & 31) == 0) {
#pragma unroll
    for (int k = 0; k < 32; k += 8)
      asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + k), "f"(v[k]), "f"(v[k + 1]),
                   "f"(v[k + 2]), "f"(v[k + 3]), "f"(v[k + 4]), "f"(v[k + 5]), "f"(v[k + 6]), "f"(v[k + 7])
                   : "memory");
  } else if ((reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
#pragma unroll
    for (int k = 0; k < 32; k += 4)
      *reinterpret_cast<float4*>(dst + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
  } else {
#pragma unroll
    for (int k = 0; k < 32; ++k) dst[k] = v[k];
  }
}

// Sketch block (PS prototypes x D) from TMEM to global memory.
//  TRANS (D = 128): TMEM holds O^T: lane = feature d, column = prototype.
//  else (D = 64):   TMEM holds O in PS/128 blocks: lane = prototype, column = d.
template <int D, int PS, bool TRANS, int O_COL>
__device__ __forceinline__ void store_sketch(uint32_t tmem, uint32_t lane_off, int sw, int q, int lane, float* dst) {
  float v[32];
  if (TRANS) {
    const int d = 32 * q + lane;
#pragma unroll 1
    for (int c = 0; c < PS / 2 / 32; ++c) {
      const int pbase = sw * (PS / 2) + 32 * c;
      ptx::tmem_ld32(tmem + lane_off + O_COL + pbase, v);
      ptx::tmem_ld_wait();
      float* col = dst + int64_t(pbase) * D + d;  // prototype pbase, feature d; the next prototype is D floats on
#pragma unroll
      for (int k = 0; k < 32; ++k) col[k * D] = v[k];
    }
  } else {
    constexpr int NB = PS / 128;
    const int blk = NB == 2 ? sw : 0;
    const int p = 128 * blk + 32 * q + lane;
    const int c0 = NB == 2 ? 0 : 32 * sw;
    const int c1 = NB == 2 ? D : c0 + 32;
#pragma unroll 1
    for (int c = c0; c < c1; c += 32) {
      ptx::tmem_ld32(tmem + lane_off + O_COL + blk * D + c, v);
      ptx::tmem_ld_wait();
      store_row32(dst + int64_t(p) * D + c, v);
    }
  }
}

// Prototype-major accumulator ([PS/128 blocks] lanes = prototype, columns = d)
// times `mul` to global rows [PS][D] (used for dQ partials).
template <int D, int PS, int O_COL>
__device__ __forceinline__ void store_sketch_scaled(uint32_t tmem, uint32_t lane_off, int sw, int q, int lane,
                                                    float* dst, float mul) {
  float v[32];
  constexpr int NB = PS / 128;
  const int blk = NB == 2 ? sw : 0;
  const int p = 128 * blk + 32 * q + lane;
  const int c0 = NB == 2 ? 0 : (D / 2) * sw;
  const int c1 = NB == 2 ? D : c0 + D / 2;
#pragma unroll 1
  for (int c = c0; c < c1; c += 32) {
    ptx::tmem_ld32(tmem + lane_off + O_COL + blk * D + c, v);
    ptx::tmem_ld_wait();
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] *= mul;
    store_row32(dst + int64_t(p) * D + c, v);
  }
}

// ------------------------------------------------------------- host helpers
bool make_kv_map(CUtensorMap* m, const void* base, int64_t N, int H, int D);
bool make_q_map(CUtensorMap* m, const void* Q, int H, int P, int D, int box_rows);
bool device_is_sm103();
int device_sm_count();

}  // namespace tcc

bool tc_path_enabled();

}  // namespace sa
