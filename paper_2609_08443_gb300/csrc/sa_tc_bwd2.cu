// Two-sweep tensor-core backward of the SA sketching step (sm_103a), for up to
// 512 prototypes: token side (dV, dK, D) and, where TMEM holds it, dQ as well.
//
// Chain rule of Sec. 3.1 with upstream G = dL/dsketch[b, h] and the forward's
// per-token log-sum-exp (FlashSA's softmax statistic, Sec. 4.4).  Per tile of 128
// tokens, over chunks c of 128 prototypes:
//   sweep 1:  S_c = K Q_c^T,  A_c = exp(scale S_c - lse),  dV += A_c G_c
//   between:  D_i = dV_i . v_i                       (= sum_j A[j,i] dA[j,i])
//   sweep 2:  dA_c = V G_c^T,  dS_c = A_c o (dA_c - D),  dK += dS_c Q_c
//             and, fused (FUSE), dQ_c += dS_c^T K
// What makes it fast: every weight stays in TMEM.  A_c is written there as bf16
// pairs, the A operand of dV += A_c G_c (TS form), and stays until sweep 2 reads
// it back and overwrites it with dS_c, the A operand of dK += dS_c Q_c.  So A and
// dS never pass through shared memory, S is formed once, and no product exists
// only to get D (a one-sweep kernel needs qbar = A Q for dK = u - D qbar): 8 P d
// executed per token-head for dV and dK, against 10 P d.
// TMEM (512 columns): S/dA 128, A/dS P/2, dV and dK D columns each (shared when
// there is no room for both: dK_0 follows dV's read-out anyway), dQ (P/128) D.
// Shared memory: G of the user stays resident ([chunk][d/64][128][64]); Q stays
// resident too except at P = 512, d = 128, where its 16 KB blocks stream through
// a two-slot ring in the order S and dK consume them.
// One S/dA buffer: the next product into it is issued once the softmax warps hold
// its values in registers, so it runs while they form A or dS.
//
// SUM: K = V = X (the key projection): dX = dV + dK.  dS carries the scale and dK
// accumulates on top of dV in TMEM, so one read-out stores the sum.
//
// Warp roles: 0 tile sequence + K, V (and resident Q) loads; 1 issues S and dA, 2
// (also TMEM) issues dV, dK and dQ; 3 converts dsketch (FUSE) or loads G and streams
// Q; 4-11 softmax and epilogue.  A shared-memory round trip takes 250-450 cycles
// beside running products, so the two issuers wait independently and poll all that a
// product needs at once, the softmax warps keep a tile's info in registers, and the
// rows of dV and dK go straight to global memory, dV's only after the first dS has
// been handed over: staging them for TMA stores put three more round trips on the
// chain.  The issuers' chunk loops stay rolled (unrolled, the kernel is 160 KB of code
// for 99, and slower).  Every wait is bounded (sa_ptx.cuh).
// Measured, kernel alone: 64 users (1.5M tokens, H = 8, P = 256, d = 64) 3.19 ms with
// the one-sweep kernel that kept A and dS in shared memory, 2.14 ms now; 16 users of
// 100K tokens at P = 512, d = 128 6.82 and 6.15 ms; 12 users of 137K tokens with their
// own queries 0.61 and 0.56 ms.
#include <cuda.h>

#include "sa_handoff.cuh"
#include "sa_ptx.cuh"
#include "sa_tc.cuh"
#include "sa_tc_common.cuh"

namespace sa {
namespace tcs {

using namespace ptx;
using namespace tcc;

constexpr uint32_t kRegsCtl = 152, kRegsSoft = 176;
static_assert(128 * kRegsCtl + 256 * kRegsSoft == 384 * 168, "register split = launch allocation");
constexpr float kLog2e = 1.4426950408889634f;

// What every role needs to know of a tile, written once by warp 0 into a ring.
struct TileInfo {
  int64_t tok0;   // first token row
  float* dq_dst;  // FUSE, last tile of a run: where the run's dQ goes
  int h, n, b;
  uint32_t flags;
};
// A run is a sequence of tiles that read one row of Q: a head, or with per-user
// queries one (user, head) segment.
enum : uint32_t { kRunFirst = 1u, kRunLast = 2u, kSegFirst = 4u, kSegLast = 8u };

template <int D, int P, bool FUSE, bool SUM>
struct SCfg {
  static constexpr int NC = 128, NCH = P / NC, ND = D / 64;
  static constexpr int BLK = 128 * 128;  // 128 rows x 64 bf16, 128-byte swizzle
  static constexpr int TILE = ND * BLK;  // K, V, and a chunk of Q or G
  static constexpr bool Q_RES = !(D == 128 && P == 512);
  static constexpr int NQ = Q_RES ? NCH * ND : 2;  // Q blocks in shared memory
  // Q barriers: one, or when streamed two slots whose blocks announce themselves on
  // eight barriers in turn (sa_handoff.cuh)
  static constexpr int NQF = Q_RES ? 1 : 8, NQE = Q_RES ? 1 : 2;
  static_assert(Q_RES || (NCH == 4 && ND == 2), "streamed blocks of one issuer are at most eight apart");
  static constexpr int NG = FUSE && D == 64 ? 2 : 1;  // G buffers (the next user's is converted meanwhile)
  static constexpr int NGB = FUSE ? NG : NCH;      // G barriers: per buffer, or per chunk
  static constexpr int NK = (D == 64 || FUSE) ? 2 : 1;  // fused: K(i) is read until dQ(i), after S(i+1)
  static constexpr int NV = D == 64 ? 2 : 1;
  static constexpr int NI = 4;  // tile infos
  static constexpr int OFF_G = 0;
  static constexpr int OFF_Q = OFF_G + NG * NCH * TILE;
  static constexpr int OFF_K = OFF_Q + NQ * BLK;
  static constexpr int OFF_V = OFF_K + NK * TILE;
  static constexpr int OFF_DS = OFF_V + NV * TILE;  // FUSE: dS [P/64][128 tokens][64], A operand of dQ
  static constexpr int OFF_STATS = OFF_DS + (FUSE ? NCH * 2 * BLK : 0);
  static constexpr bool SPLIT_D = D == 128;  // D_i from two half dots, exchanged between the warpgroups
  static constexpr int OFF_INFO = OFF_STATS + (SPLIT_D ? 2 * 2 * T * 4 : 0);
  static constexpr int OFF_BAR = OFF_INFO + NI * int(sizeof(TileInfo));
  static constexpr int NCB = handoff::chunk_bars(NCH);
  static constexpr int NBAR = 2 * NK + 2 * NV + NQF + NQE + 2 * NGB + 2 * NI + NCH + 2 * NCB + 8;
  static constexpr int OFF_MISC = OFF_BAR + NBAR * 8;
  static constexpr int SMEM = OFF_MISC + 16;
  static constexpr int SD_COL = 0, A_COL = NC, DV_COL = A_COL + P / 2;
  static constexpr int DQ_COLS = FUSE ? NCH * D : 0;
  static constexpr bool SHARED_ACC = SUM || DV_COL + 2 * D + DQ_COLS > 512;
  static constexpr int DK_COL = SHARED_ACC ? DV_COL : DV_COL + D;
  static constexpr int DQ_COL = DK_COL + D;
  static constexpr int TMEM_COLS = tmem_cols_for(DQ_COL + DQ_COLS);
  static_assert(DQ_COL + DQ_COLS <= 512 && SMEM <= 232448, "budget");
  static_assert(OFF_INFO % 16 == 0 && OFF_BAR % 8 == 0, "alignment");
};

// 64 (or 32) bf16 values, 32 packed words at most, to a 16-byte aligned row (the
// entry points refuse others): 32-byte stores where the row allows them (whole
// sectors per thread).
template <int NW>
__device__ __forceinline__ void store_packed(__nv_bfloat16* dst, const uint32_t* pk, bool by32) {
  if (by32) {
#pragma unroll
    for (int k = 0; k < NW; k += 8)
      asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + 2 * k), "r"(pk[k]),
                   "r"(pk[k + 1]), "r"(pk[k + 2]), "r"(pk[k + 3]), "r"(pk[k + 4]), "r"(pk[k + 5]), "r"(pk[k + 6]),
                   "r"(pk[k + 7])
                   : "memory");
  } else {
#pragma unroll
    for (int k = 0; k < NW; k += 4)
      *reinterpret_cast<uint4*>(dst + 2 * k) = make_uint4(pk[k], pk[k + 1], pk[k + 2], pk[k + 3]);
  }
}

__device__ __forceinline__ float lo16(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi16(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// sum of v[8k .. 8k+7] times the eight bf16 values of w
__device__ __forceinline__ float dot8(const float* v, uint4 w, float s) {
  s = fmaf(v[0], lo16(w.x), s);
  s = fmaf(v[1], hi16(w.x), s);
  s = fmaf(v[2], lo16(w.y), s);
  s = fmaf(v[3], hi16(w.y), s);
  s = fmaf(v[4], lo16(w.z), s);
  s = fmaf(v[5], hi16(w.z), s);
  s = fmaf(v[6], lo16(w.w), s);
  return fmaf(v[7], hi16(w.w), s);
}

template <int D, int P, bool FUSE, bool SUM>
__global__ void __launch_bounds__(kThreads, 1)
    tc_bwd2_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                   const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmG,
                   Args a, const float* __restrict__ dsk, const float* lse, float* Dco,
                   __nv_bfloat16* __restrict__ dK, __nv_bfloat16* __restrict__ dV) {
  using C = SCfg<D, P, FUSE, SUM>;
  constexpr int NCH = C::NCH, ND = C::ND, BLK = C::BLK;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (cta_leaves(a.ws, smem_u32(smem), 0xB41u)) return;
  const uint32_t sbase = smem_u32(smem);
  const uint32_t sG = sbase + C::OFF_G, sQ = sbase + C::OFF_Q, sK = sbase + C::OFF_K, sV = sbase + C::OFF_V,
                 sDS = sbase + C::OFF_DS;
  uint32_t nb = sbase + C::OFF_BAR;
  auto take = [&](int n) {
    const uint32_t r = nb;
    nb += 8u * uint32_t(n);
    return r;
  };
  const uint32_t k_full = take(C::NK), k_empty = take(C::NK), v_full = take(C::NV), v_empty = take(C::NV),
                 q_full = take(C::NQF), q_empty = take(C::NQE), g_full = take(C::NGB), g_empty = take(C::NGB),
                 i_full = take(C::NI), i_empty = take(C::NI), dk_done = take(NCH), sd_full = take(1),
                 sd_free = take(1), a_full = take(C::NCB), dv_full = take(1), ds_full = take(C::NCB), acc_free = take(1),
                 dq_free = take(1), st_ready = take(1), drain = take(2);
  TileInfo* infos = reinterpret_cast<TileInfo*>(smem + C::OFF_INFO);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::OFF_MISC + 4);

  const int64_t tph = reinterpret_cast<const WsHeader*>(a.ws)->tiles_per_head;
  const int64_t total = tph * a.H;
  const int W = int(gridDim.x), wk = int(blockIdx.x);
  const int64_t tb = range_begin(total, W, wk), te = range_begin(total, W, wk + 1);
  const int ntiles = int(te - tb);

  if (threadIdx.x == 0) {
    auto init = [&](uint32_t bar, int n, uint32_t count) {
      for (int k = 0; k < n; ++k) mbar_init(bar + 8u * k, count);
    };
    init(k_full, C::NK, 1);
    init(k_empty, C::NK, FUSE ? 2 : 1);  // the last S, and dQ
    init(v_full, C::NV, 1);
    init(v_empty, C::NV, 1 + kSoftWarps);  // the last dA, and the warps' reads for D
    init(q_full, C::NQF, 1);
    init(q_empty, C::NQE, C::Q_RES ? 2 : 1);  // resident: the run's last S and last dK
    init(g_full, C::NGB, 1);
    init(g_empty, C::NGB, 2);  // dV and dA
    init(i_full, C::NI, 1);
    init(i_empty, C::NI, 2 + kSoftWarps + (FUSE ? 0 : 1));
    init(dk_done, NCH, 1);
    init(sd_full, 1, 1);
    init(sd_free, 1, kSoftWarps);
    init(a_full, C::NCB, kSoftWarps);
    init(dv_full, 1, 1);
    init(ds_full, C::NCB, kSoftWarps);
    init(acc_free, 1, kSoftWarps);
    init(dq_free, 1, kSoftWarps);
    init(st_ready, 1, kSoftWarps);
    init(drain, 2, 1);
    wait_ctl_init(abort_flag, a.ws);
    fence_mbar_init();
  }
  if (warp == 2) tmem_alloc(smem_u32(tmem_slot), C::TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  auto i_slot = [](int li) { return li % C::NI; };
  auto i_par = [](int li) { return uint32_t(li / C::NI) & 1u; };
  auto chunk_bar = [](int li, int c) { return 8u * uint32_t(handoff::chunk_bar(li, c, NCH)); };
  auto chunk_par = [](int li, int c) { return handoff::chunk_parity(li, c, NCH); };

  if (ntiles > 0 && warp < kSoftWarp0) {
    setmaxnreg_dec<kRegsCtl>();
    if (warp == 0 && lane == 0) {
      // ------------------------------------------- tile sequence, K, V (, Q)
      tma_prefetch_desc(&tmK);
      tma_prefetch_desc(&tmV);
      tma_prefetch_desc(&tmQ);
      TileWalker w(a, tb, te, T);  // the tile whose info was written last
      int prev_q = -1, hc = 0, loaded_k = 0, loaded_v = 0;
      bool ok = true;
      uint32_t fl = 0;
      auto put_info = [&](int li) {
        if (li >= C::NI) ok = mbar_wait(i_empty + 8u * i_slot(li), i_par(li) ^ 1u, abort_flag, a.ws, 0xC11);
        if (!ok) return;
        int64_t t0n;
        int nn, hn, qkn;
        w.peek_next(t0n, nn, hn, qkn);
        const bool last = li + 1 >= ntiles || qkn != w.qk;
        fl = (w.qk != prev_q ? kRunFirst : 0u) | (last ? kRunLast : 0u) | (w.seg_first ? kSegFirst : 0u) |
             (w.seg_last ? kSegLast : 0u);
        prev_q = w.qk;
        TileInfo& o = infos[i_slot(li)];
        o.tok0 = w.tok0;
        o.dq_dst = FUSE && last ? dq_block_dst(a, wk, W, total, w, 0, D) : nullptr;
        o.h = w.h;
        o.n = w.n;
        o.b = w.b;
        o.flags = fl;
        mbar_arrive(i_full + 8u * i_slot(li));
      };
      put_info(0);
      for (int li = 0; li < ntiles && ok; ++li) {
        const int h = w.h, qk = w.qk, t0 = int(w.tok0);
        const bool run_first = (fl & kRunFirst) != 0;
        if (li + 1 < ntiles) {
          w.next();
          put_info(li + 1);
          if (!ok) break;
#pragma unroll
          for (int dh = 0; dh < ND; ++dh) {  // the next tile into L2
            tma_prefetch_l2_3d(&tmK, 64 * dh, w.h, int(w.tok0));
            tma_prefetch_l2_3d(&tmV, 64 * dh, w.h, int(w.tok0));
          }
        }
        const int ks = li % C::NK, ku = li / C::NK;
        if (ku > 0) ok = mbar_wait(k_empty + 8u * ks, uint32_t(ku - 1) & 1u, abort_flag, a.ws, 0xC12);
        if (!ok) break;
        mbar_arrive_expect_tx(k_full + 8u * ks, C::TILE);
#pragma unroll
        for (int dh = 0; dh < ND; ++dh) tma_load_3d(sK + ks * C::TILE + dh * BLK, &tmK, k_full + 8u * ks, 64 * dh, h, t0);
        loaded_k = li + 1;
        if (C::Q_RES && run_first) {
          if (hc > 0) ok = mbar_wait(q_empty, uint32_t(hc - 1) & 1u, abort_flag, a.ws, 0xC13);
          if (!ok) break;
          mbar_arrive_expect_tx(q_full, NCH * C::TILE);
#pragma unroll
          for (int c = 0; c < NCH; ++c)
#pragma unroll
            for (int dh = 0; dh < ND; ++dh)
              tma_load_3d(sQ + (c * ND + dh) * BLK, &tmQ, q_full, 64 * dh, c * C::NC, qk);
          ++hc;
        }
        const int vs = li % C::NV, vu = li / C::NV;
        if (vu > 0) ok = mbar_wait(v_empty + 8u * vs, uint32_t(vu - 1) & 1u, abort_flag, a.ws, 0xC14);
        if (!ok) break;
        mbar_arrive_expect_tx(v_full + 8u * vs, C::TILE);
#pragma unroll
        for (int dh = 0; dh < ND; ++dh) tma_load_3d(sV + vs * C::TILE + dh * BLK, &tmV, v_full + 8u * vs, 64 * dh, h, t0);
        loaded_v = li + 1;
      }
      if (!ok) {  // the copies in flight land before the CTA may exit
        for (int li = (loaded_k > C::NK ? loaded_k - C::NK : 0); li < loaded_k; ++li)
          mbar_wait_bounded(k_full + 8u * (li % C::NK), uint32_t(li / C::NK) & 1u, 200000000ull);
        for (int li = (loaded_v > C::NV ? loaded_v - C::NV : 0); li < loaded_v; ++li)
          mbar_wait_bounded(v_full + 8u * (li % C::NV), uint32_t(li / C::NV) & 1u, 200000000ull);
        if (hc > 0) mbar_wait_bounded(q_full, uint32_t(hc - 1) & 1u, 200000000ull);
      }
    } else if (warp == 1 || warp == 2) {
      // -------------------------------------------------------- UMMA issuers
      // warp 1: S_0(0), then per tile S_1 .., dA_0 .., S_0 of the next tile, each as
      // soon as the S/dA columns are free; warp 2: per tile dV_0 .., dK_0 .. (dQ)
      bool ok = true;
      uint32_t gseg = 0, gmask = 0;  // segments so far, G chunks of this one waited for
      auto wt = [&](uint32_t bar, uint32_t par, uint32_t site) {
        return ok = ok && mbar_wait_warp(bar, par, abort_flag, a.ws, site);
      };
      auto info_flags = [&](int li) -> uint32_t {
        wt(i_full + 8u * i_slot(li), i_par(li), 0xD11);
        return ok ? infos[i_slot(li)].flags : 0u;
      };
      auto kstep = [](int k) { return uint32_t((k >> 2) * BLK + (k & 3) * 32); };
      // the wait for chunk c of this segment's G, once per segment, else `x`
      auto g_phase = [&](int c, BarPhase x) {
        const int bit = FUSE ? 0 : c;
        if ((gmask >> bit) & 1u) return x;
        gmask |= 1u << bit;
        return FUSE ? BarPhase{g_full + 8u * (gseg % C::NG), (gseg / C::NG) & 1u} : BarPhase{g_full + 8u * c, gseg & 1u};
      };
      auto g_ofs = [&](int c) { return uint32_t((FUSE ? int(gseg % C::NG) * NCH : 0) + c) * uint32_t(C::TILE); };
      auto g_bar = [&](int c) { return g_empty + 8u * (FUSE ? int(gseg % C::NG) : c); };
      auto qb_S = [&](int li, int c) { return handoff::q_block_of_S(li, c, NCH, ND); };
      auto qb_dK = [&](int li, int c) { return handoff::q_block_of_dK(li, c, li + 1 >= ntiles, NCH, ND); };
      auto q_phase = [&](uint32_t x) {
        return BarPhase{q_full + 8u * handoff::q_block_bar(x), handoff::q_block_parity(x)};
      };
      if (warp == 1) {
        constexpr uint32_t idS = idesc_bf16(128, C::NC, 0, 0);  // [tok x chunk], K = d
        const uint64_t dKk = sdesc(sK, 16, 1024), dVk = sdesc(sV, 16, 1024), dQk = sdesc(sQ, 16, 1024),
                       dGk = sdesc(sG, 16, 1024);
        uint32_t u = 0;
        int hc = 0;
        // the S/dA columns are free, once the warps hold the last product
        auto sd_phase = [&](BarPhase x) {
          const BarPhase r = u > 0 ? BarPhase{sd_free, (u - 1) & 1u} : x;
          ++u;
          return r;
        };
        auto issue_S = [&](int li, int c, uint32_t fl) {
          const int ks = li % C::NK;
          const BarPhase kf{k_full + 8u * ks, uint32_t(li / C::NK) & 1u};  // also waited for when c > 0: complete then
          const uint64_t dK_ = sdesc_add(dKk, uint32_t(ks) * C::TILE);
          if (C::Q_RES) {
            const bool run = c == 0 && (fl & kRunFirst);
            const BarPhase b[3] = {kf, sd_phase(kf), run ? BarPhase{q_full, uint32_t(hc) & 1u} : kf};
            ok = ok && mbar_wait_warp_all(b, abort_flag, a.ws, 0xD15);
            hc += run ? 1 : 0;
            if (!ok) return;
            tc_fence_after();
            if (elect_one()) {
              const uint64_t dQ_ = sdesc_add(dQk, uint32_t(c) * C::TILE);
#pragma unroll
              for (int k = 0; k < D / 16; ++k)
                umma_ss(tmem + C::SD_COL, sdesc_add(dK_, kstep(k)), sdesc_add(dQ_, kstep(k)), idS, k > 0 ? 1u : 0u);
            }
          } else {
            const uint32_t qb = qb_S(li, c);
            const BarPhase b[3] = {kf, sd_phase(kf), q_phase(qb)};
            ok = ok && mbar_wait_warp_all(b, abort_flag, a.ws, 0xD15);
#pragma unroll
            for (int dh = 0; dh < ND; ++dh) {
              const uint32_t x = qb + uint32_t(dh), s = x & 1u;
              if (dh > 0) wt(q_phase(x).bar, q_phase(x).parity, 0xD16);
              if (!ok) return;
              tc_fence_after();
              if (elect_one()) {
                const uint64_t dQ_ = sdesc_add(dQk, s * BLK), dKh = sdesc_add(dK_, uint32_t(dh) * BLK);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                  umma_ss(tmem + C::SD_COL, sdesc_add(dKh, 32u * k), sdesc_add(dQ_, 32u * k), idS,
                          (dh > 0 || k > 0) ? 1u : 0u);
                umma_commit(q_empty + 8u * s);
              }
            }
          }
          if (elect_one()) {
            umma_commit(sd_full);
            if (c == NCH - 1) {
              umma_commit(k_empty + 8u * ks);
              if (C::Q_RES && (fl & kRunLast)) umma_commit(q_empty);
            }
          }
        };
        auto issue_dA = [&](int li, int c, uint32_t fl) {
          const int vs = li % C::NV;
          const BarPhase vf{v_full + 8u * vs, uint32_t(li / C::NV) & 1u};
          const BarPhase b[3] = {vf, sd_phase(vf), g_phase(c, vf)};
          ok = ok && mbar_wait_warp_all(b, abort_flag, a.ws, 0xD18);
          if (!ok) return;
          tc_fence_after();
          if (elect_one()) {
            const uint64_t dV_ = sdesc_add(dVk, uint32_t(vs) * C::TILE), dG_ = sdesc_add(dGk, g_ofs(c));
#pragma unroll
            for (int k = 0; k < D / 16; ++k)
              umma_ss(tmem + C::SD_COL, sdesc_add(dV_, kstep(k)), sdesc_add(dG_, kstep(k)), idS, k > 0 ? 1u : 0u);
            umma_commit(sd_full);
            if (c == NCH - 1) umma_commit(v_empty + 8u * vs);
            if ((fl & kSegLast) && (!FUSE || c == NCH - 1)) umma_commit(g_bar(c));
          }
        };
        uint32_t fl = info_flags(0);
        if (ok) issue_S(0, 0, fl);
        for (int li = 0; li < ntiles && ok; ++li) {
          const bool more = li + 1 < ntiles;
          if (fl & kSegFirst) gmask = 0;
#pragma unroll 1
          for (int c = 1; c < NCH; ++c)
            if (ok) issue_S(li, c, fl);
#pragma unroll 1
          for (int c = 0; c + 1 < NCH; ++c)
            if (ok) issue_dA(li, c, fl);
          const uint32_t fn = more && ok ? info_flags(li + 1) : 0u;  // its wait runs beside these products
          if (ok) issue_dA(li, NCH - 1, fl);
          if (more && ok) issue_S(li + 1, 0, fn);
          if (fl & kSegLast) ++gseg;
          if (elect_one()) mbar_arrive(i_empty + 8u * i_slot(li));
          fl = fn;
        }
        if (elect_one()) umma_commit(drain);  // no UMMA may still run when TMEM is released
        mbar_wait_bounded(drain, 0, 200000000ull);
      } else {
        constexpr uint32_t idT = idesc_bf16(128, C::Q_RES ? D : 64, 0, 1);  // [tok x d], K = chunk, A from TMEM
        constexpr uint32_t idV = idesc_bf16(128, D, 0, 1);
        constexpr uint32_t idQ = idesc_bf16(128, D, 1, 1);  // [proto x d], K = tokens
        const uint64_t dKm = sdesc(sK, BLK, 1024), dQm = sdesc(sQ, BLK, 1024), dGm = sdesc(sG, BLK, 1024),
                       dDm = sdesc(sDS, BLK, 1024);
        int hc = 0, hp = 0;
        auto issue_dV = [&](int li, int c, uint32_t fl) {
          const BarPhase af{a_full + chunk_bar(li, c), chunk_par(li, c)};
          const BarPhase b[3] = {af, C::SHARED_ACC && c == 0 && li > 0 ? BarPhase{acc_free, uint32_t(li - 1) & 1u} : af,
                                 g_phase(c, af)};
          ok = ok && mbar_wait_warp_all(b, abort_flag, a.ws, 0xD19);
          if (!ok) return;
          tc_fence_after();
          if (elect_one()) {
            const uint64_t dG_ = sdesc_add(dGm, g_ofs(c));
#pragma unroll
            for (int k = 0; k < C::NC / 16; ++k)
              umma_ts(tmem + C::DV_COL, tmem + C::A_COL + c * (C::NC / 2) + 8 * k, sdesc_add(dG_, 2048u * k), idV,
                      (c > 0 || k > 0) ? 1u : 0u);
            if (c == NCH - 1) umma_commit(dv_full);
            if ((fl & kSegLast) && (!FUSE || c == NCH - 1)) umma_commit(g_bar(c));
          }
        };
        auto issue_dK = [&](int li, int c, uint32_t fl) {
          const int ks = li % C::NK;
          const bool run = C::Q_RES && c == 0 && (fl & kRunFirst);
          const BarPhase df{ds_full + chunk_bar(li, c), chunk_par(li, c)};
          const BarPhase af = !C::SHARED_ACC && c == 0 && li > 0 ? BarPhase{acc_free, uint32_t(li - 1) & 1u} : df;
          const uint32_t ta = tmem + C::A_COL + c * (C::NC / 2);
          if (C::Q_RES) {
            const BarPhase b[4] = {df, af, run ? BarPhase{q_full, uint32_t(hc) & 1u} : df,
                                   FUSE && run && hp > 0 ? BarPhase{dq_free, uint32_t(hp - 1) & 1u} : df};
            ok = ok && mbar_wait_warp_all(b, abort_flag, a.ws, 0xD1B);
            hc += run ? 1 : 0;
            if (!ok) return;
            tc_fence_after();
            if (elect_one()) {
              const uint64_t dQ_ = sdesc_add(dQm, uint32_t(c) * C::TILE);
#pragma unroll
              for (int k = 0; k < C::NC / 16; ++k)
                umma_ts(tmem + C::DK_COL, ta + 8 * k, sdesc_add(dQ_, 2048u * k), idT,
                        (SUM || c > 0 || k > 0) ? 1u : 0u);
            }
          } else {
            const uint32_t qb = qb_dK(li, c);
            const BarPhase b[3] = {df, af, q_phase(qb)};
            ok = ok && mbar_wait_warp_all(b, abort_flag, a.ws, 0xD1B);
#pragma unroll
            for (int dh = 0; dh < ND; ++dh) {
              const uint32_t x = qb + uint32_t(dh), s = x & 1u;
              if (dh > 0) wt(q_phase(x).bar, q_phase(x).parity, 0xD1E);
              if (!ok) return;
              tc_fence_after();
              if (elect_one()) {
                const uint64_t dQ_ = sdesc_add(dQm, s * BLK);
#pragma unroll
                for (int k = 0; k < C::NC / 16; ++k)
                  umma_ts(tmem + C::DK_COL + 64 * dh, ta + 8 * k, sdesc_add(dQ_, 2048u * k), idT,
                          (SUM || c > 0 || k > 0) ? 1u : 0u);
                umma_commit(q_empty + 8u * s);
              }
            }
          }
          if (elect_one()) {
            if (FUSE) {
              const uint64_t dD_ = sdesc_add(dDm, uint32_t(c) * 2 * BLK), dK_ = sdesc_add(dKm, uint32_t(ks) * C::TILE);
#pragma unroll
              for (int k = 0; k < T / 16; ++k)
                umma_ss(tmem + C::DQ_COL + c * D, sdesc_add(dD_, 2048u * k), sdesc_add(dK_, 2048u * k), idQ,
                        ((fl & kRunFirst) && k == 0) ? 0u : 1u);
            }
            umma_commit(dk_done + 8u * c);
            if (c == NCH - 1) {
              if (FUSE) umma_commit(k_empty + 8u * ks);
              if (C::Q_RES && (fl & kRunLast)) umma_commit(q_empty);
            }
          }
          if (c == NCH - 1 && (fl & kRunLast)) ++hp;
        };
        uint32_t fl = info_flags(0);
        for (int li = 0; li < ntiles && ok; ++li) {
          if (fl & kSegFirst) gmask = 0;
          uint32_t fn = 0u;
          {  // the next tile's info and (FUSE) this one's K, read by dQ
            const int ln = li + 1 < ntiles ? li + 1 : li;
            const BarPhase nf{i_full + 8u * i_slot(ln), i_par(ln)};
            const BarPhase b[2] = {nf, FUSE ? BarPhase{k_full + 8u * (li % C::NK), uint32_t(li / C::NK) & 1u} : nf};
            ok = mbar_wait_warp_all(b, abort_flag, a.ws, 0xD20);
            if (!ok) break;
            if (li + 1 < ntiles) fn = infos[i_slot(li + 1)].flags;
          }
#pragma unroll 1
          for (int c = 0; c < NCH; ++c)
            if (ok) issue_dV(li, c, fl);
#pragma unroll 1
          for (int c = 0; c < NCH; ++c)
            if (ok) issue_dK(li, c, fl);
          if (fl & kSegLast) ++gseg;
          if (elect_one()) mbar_arrive(i_empty + 8u * i_slot(li));
          fl = fn;
        }
        if (elect_one()) umma_commit(drain + 8u);
        mbar_wait_bounded(drain + 8u, 0, 200000000ull);
      }
    } else if (FUSE && warp == 3) {
      // ---------------- dsketch rows -> bf16, swizzled [chunk][d/64][128][64]
      TileWalker cur(a, tb, te, T);
      int gc = 0;
      bool ok = true;
      for (int li = 0; li < ntiles && ok; ++li) {
        if (cur.seg_first) {
          const int gb = gc % C::NG;
          if (gc >= C::NG)
            ok = mbar_wait_warp(g_empty + 8u * gb, uint32_t((gc / C::NG) - 1) & 1u, abort_flag, a.ws, 0xE11);
          if (!ok) break;
          const float* src = dsk + (int64_t(cur.b) * a.H + cur.h) * a.P * D;
          if (cur.seg1 < te && lane == 0) {  // the next segment's dsketch into L2 (short users: one tile each)
            const TileRef nx = locate_next_segment(cur.seg1, cur.h, cur.b, tph, a.prefix, a.cu, a.B, T);
            bulk_prefetch_l2(dsk + (int64_t(nx.b) * a.H + nx.h) * a.P * D, P * D * 4);
          }
          __syncwarp();
          uint8_t* gdst = smem + C::OFF_G + gb * NCH * C::TILE;
#pragma unroll 16
          for (int e = lane; e < P * D / 8; e += 32) {
            const int p = e / (D / 8), dd = (e % (D / 8)) * 8;
            const float4 x = *reinterpret_cast<const float4*>(src + int64_t(p) * D + dd);
            const float4 y = *reinterpret_cast<const float4*>(src + int64_t(p) * D + dd + 4);
            *reinterpret_cast<uint4*>(gdst + (p >> 7) * C::TILE + (dd >> 6) * BLK + (p & 127) * 128 +
                                      ((((dd & 63) >> 3) ^ (p & 7)) << 4)) =
                make_uint4(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w), pack_bf16(y.x, y.y), pack_bf16(y.z, y.w));
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(g_full + 8u * gb);
          ++gc;
        }
        cur.next();
      }
    } else if (!FUSE && warp == 3 && lane == 0) {
      // ----------------------------- G chunks of a new segment, streamed Q blocks
      tma_prefetch_desc(&tmG);
      uint32_t qb = 0;
      int gc = 0, loaded_g = 0;
      bool ok = true;
      // chunk c of segment gc, once dV_c and dA_c of the last segment have read it
      auto load_G = [&](int row) {
#pragma unroll 1
        for (int c = 0; c < NCH; ++c) {
          if (gc > 0) ok = ok && mbar_wait(g_empty + 8u * c, uint32_t(gc - 1) & 1u, abort_flag, a.ws, 0xE13);
          if (!ok) return;
          mbar_arrive_expect_tx(g_full + 8u * c, C::TILE);
#pragma unroll
          for (int dh = 0; dh < ND; ++dh)
            tma_load_3d(sG + c * C::TILE + dh * BLK, &tmG, g_full + 8u * c, 64 * dh, c * C::NC, row);
          loaded_g = c + 1;
        }
        ++gc;
        loaded_g = 0;
      };
      auto load_Q = [&](int c, int qk) {
#pragma unroll
        for (int dh = 0; dh < ND; ++dh, ++qb) {
          const uint32_t s = qb & 1u;
          if (qb >= 2u) ok = ok && mbar_wait(q_empty + 8u * s, ((qb >> 1) + 1) & 1u, abort_flag, a.ws, 0xE14);
          if (!ok) return;
          const uint32_t full = q_full + 8u * handoff::q_block_bar(qb);
          mbar_arrive_expect_tx(full, BLK);
          tma_load_3d(sQ + s * BLK, &tmQ, full, 64 * dh, c * C::NC, qk);
        }
      };
      int qk = 0, row = 0;
      uint32_t fl = 0;
      auto read_info = [&](int li) {
        ok = ok && mbar_wait(i_full + 8u * i_slot(li), i_par(li), abort_flag, a.ws, 0xE15);
        if (!ok) return;
        const TileInfo& o = infos[i_slot(li)];
        row = o.b * a.H + o.h;
        qk = a.uq ? row : o.h;
        fl = o.flags;
      };
      read_info(0);
      if constexpr (!C::Q_RES) {
        if (ok) load_Q(0, qk);
      }
      for (int li = 0; li < ntiles && ok; ++li) {
        const int qc = qk;
        if (fl & kSegFirst) load_G(row);
        if constexpr (!C::Q_RES) {
          for (int c = 1; c < NCH && ok; ++c) load_Q(c, qc);
          for (int c = 0; c + 1 < NCH && ok; ++c) load_Q(c, qc);
        }
        if (li + 1 < ntiles && ok) {
          read_info(li + 1);
          if constexpr (!C::Q_RES) {
            if (ok) load_Q(0, qk);
          }
        }
        if constexpr (!C::Q_RES) {
          if (ok) load_Q(NCH - 1, qc);
        }
        mbar_arrive(i_empty + 8u * i_slot(li));
      }
      if (!ok) {  // the copies in flight land before the CTA may exit
        for (uint32_t k = qb > 2u ? qb - 2u : 0u; k < qb; ++k)
          mbar_wait_bounded(q_full + 8u * handoff::q_block_bar(k), handoff::q_block_parity(k), 200000000ull);
        for (int c = 0; c < NCH; ++c) {
          const int n = gc + (c < loaded_g ? 1 : 0);  // loads of chunk c so far
          if (n > 0) mbar_wait_bounded(g_full + 8u * c, uint32_t(n - 1) & 1u, 200000000ull);
        }
      }
    }
  } else if (ntiles > 0) {
    setmaxnreg_inc<kRegsSoft>();
    // ------------------------------------------------ softmax + epilogue
    const int sw = (warp - kSoftWarp0) >> 2, q = warp & 3, row = 32 * q + lane;
    const uint32_t lane_off = uint32_t(32 * q) << 16;
    const uint32_t t_sd = tmem + lane_off + C::SD_COL + 64 * sw, t_a = tmem + lane_off + C::A_COL + 32 * sw;
    const float c2 = a.scale * kLog2e;
    float* stats = reinterpret_cast<float*>(smem + C::OFF_STATS);
    const bool by32 = ((reinterpret_cast<uintptr_t>(dK) | reinterpret_cast<uintptr_t>(dV)) & 31) == 0;
    bool ok = true;
    auto wwait = [&](uint32_t bar, uint32_t par, uint32_t site) {
      return mbar_wait_warp(bar, par, abort_flag, a.ws, site);
    };
    // 64 packed columns of this warpgroup to the chunk's TMEM operand
    auto put_operand = [&](int c, const uint32_t* pk) {
      tmem_st16(t_a + c * (C::NC / 2), pk);
      tmem_st16(t_a + c * (C::NC / 2) + 16, pk + 16);
      tmem_st_wait();
      tc_fence_before();
    };
    // a tile's info, copied to registers a sweep before it is needed
    struct Tile {
      int64_t tok0;
      int h, n;
      uint32_t flags;
    };
    auto read_tile = [&](int li) {
      const TileInfo& o = infos[i_slot(li)];
      return Tile{o.tok0, o.h, o.n, o.flags};
    };
    // this thread's D/2 columns of an output row
    auto put_row = [&](__nv_bfloat16* out, const Tile& o, const uint32_t* pk) {
      if (row < o.n)
        store_packed<D / 4>(out + ((o.tok0 + row) * a.H + o.h) * int64_t(D) + sw * (D / 2), pk, by32);
    };
    // dK (or dV + dK) rows of tile li and, at the end of a run, its dQ
    auto finish = [&](int li, const Tile& o, bool waited) -> bool {
      if (!waited && !wwait(dk_done + 8u * (NCH - 1), uint32_t(li) & 1u, 0xF11)) return false;
      tc_fence_after();
      {
        float v[D / 2];
        uint32_t pk[D / 4];
#pragma unroll
        for (int k = 0; k < D / 2; k += 32) tmem_ld32(tmem + lane_off + C::DK_COL + sw * (D / 2) + k, v + k);
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_free);
        const float mul = SUM ? 1.f : a.scale;
#pragma unroll
        for (int k = 0; k < D / 4; ++k) pk[k] = pack_bf16(v[2 * k] * mul, v[2 * k + 1] * mul);
        put_row(SUM ? dV : dK, o, pk);
      }
      if constexpr (FUSE) {
        if (o.flags & kRunLast) {
          store_sketch_scaled<D, P, C::DQ_COL>(tmem, lane_off, sw, q, lane, infos[i_slot(li)].dq_dst, SUM ? 1.f : a.scale);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(dq_free);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(i_empty + 8u * i_slot(li));
      return true;
    };
    // which chunk of sweep 1 the last tile's outputs follow: the first where dV needs
    // their accumulator, else the second, whose wait covers theirs
    constexpr int kFin = C::SHARED_ACC || NCH == 1 ? 0 : 1;
    auto load_lse = [&](const Tile& o) {
      if (row >= o.n) return float(INFINITY);
      return FUSE ? __ldg(lse + (o.tok0 + row) * a.H + o.h) : load_token_lse(lse, a, o.tok0 + row, o.h);
    };
    ok = wwait(i_full, 0, 0xF12);
    Tile cur{}, prev{};
    if (ok) cur = read_tile(0);
    float lse_cur = ok ? load_lse(cur) : 0.f;
    for (int li = 0; li < ntiles && ok; ++li) {
      const Tile o = cur;
      const int th = o.h;
      const int64_t tok = o.tok0 + row;
      const bool valid = row < o.n;
      const float L2 = lse_cur * kLog2e;  // +inf past the tile's tokens: their weights are exact zeros
      const uint32_t u0 = uint32_t(li) * 2u * NCH;
      // ---- sweep 1: A_c
#pragma unroll 1
      for (int c = 0; c < NCH; ++c) {
        {  // with S_0: dK_0 (and dQ_0) of the last tile have read dS_0; with S_kFin: all of them
          const BarPhase sf{sd_full, (u0 + c) & 1u};
          const BarPhase b[3] = {sf, c == 0 && li > 0 ? BarPhase{dk_done, uint32_t(li - 1) & 1u} : sf,
                                 kFin == 1 && c == 1 && li > 0 ? BarPhase{dk_done + 8u * (NCH - 1), uint32_t(li - 1) & 1u}
                                                               : sf};
          ok = mbar_wait_warp_all(b, abort_flag, a.ws, 0xF13);
        }
        if (!ok) break;
        tc_fence_after();
        float v[64];
        tmem_ld32(t_sd, v);
        tmem_ld32(t_sd + 32, v + 32);
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(sd_free);
        exp2_shift<64>(v, c2, L2);
        uint32_t pk[32];
#pragma unroll
        for (int k = 0; k < 32; ++k) pk[k] = pack_bf16(v[2 * k], v[2 * k + 1]);
        put_operand(c, pk);
        __syncwarp();
        if (lane == 0) mbar_arrive(a_full + chunk_bar(li, c));
        if (c == kFin && li > 0) {
          ok = finish(li - 1, prev, kFin == 1);
          if (!ok) break;
        }
      }
      if (!ok) break;
      // ---- dV and D_i = dV_i . v_i; the next tile's info and lse, a sweep ahead of their use
      float Dv = 0.f, lse_nxt = 0.f;
      {
        const int ln = li + 1 < ntiles ? li + 1 : li;
        const BarPhase b[3] = {{dv_full, uint32_t(li) & 1u},
                               {v_full + 8u * (li % C::NV), uint32_t(li / C::NV) & 1u},
                               {i_full + 8u * i_slot(ln), i_par(ln)}};
        ok = mbar_wait_warp_all(b, abort_flag, a.ws, 0xF16);
        if (!ok) break;
        prev = o;
        if (li + 1 < ntiles) {
          cur = read_tile(li + 1);
          lse_nxt = load_lse(cur);
        }
      }
      tc_fence_after();
      uint32_t dvp[D / 4];  // this thread's dV columns, stored after the first dS
      const int vs = li % C::NV;
      const uint8_t* vrow = smem + C::OFF_V + vs * C::TILE + row * 128;
      if constexpr (C::SPLIT_D) {  // this warpgroup's 64 columns: d block sw
        float v[64];
        tmem_ld32(tmem + lane_off + C::DV_COL + 64 * sw, v);
        tmem_ld32(tmem + lane_off + C::DV_COL + 64 * sw + 32, v + 32);
        tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 8; ++k)
          Dv = dot8(v + 8 * k, *reinterpret_cast<const uint4*>(vrow + sw * BLK + ((k ^ (row & 7)) << 4)), Dv);
        float* st = stats + (li & 1) * 2 * T;
        st[sw * T + row] = Dv;
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(st_ready);
          mbar_arrive(v_empty + 8u * vs);
        }
        if (!SUM) {
#pragma unroll
          for (int k = 0; k < 32; ++k) dvp[k] = pack_bf16(v[2 * k], v[2 * k + 1]);
        }
        ok = wwait(st_ready, uint32_t(li) & 1u, 0xF18);
        if (!ok) break;
        Dv = st[row] + st[T + row];
      } else {  // all 64 columns in both warpgroups, no exchange
        float v[64];
        tmem_ld32(tmem + lane_off + C::DV_COL, v);
        tmem_ld32(tmem + lane_off + C::DV_COL + 32, v + 32);
        tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 8; ++k)
          Dv = dot8(v + 8 * k, *reinterpret_cast<const uint4*>(vrow + ((k ^ (row & 7)) << 4)), Dv);
        __syncwarp();
        if (lane == 0) mbar_arrive(v_empty + 8u * vs);
        if (!SUM) {
#pragma unroll
          for (int k = 0; k < 16; ++k)
            dvp[k] = sw ? pack_bf16(v[32 + 2 * k], v[33 + 2 * k]) : pack_bf16(v[2 * k], v[2 * k + 1]);
        }
      }
      if (!FUSE && sw == 0 && valid) reinterpret_cast<float2*>(Dco)[int64_t(th) * a.N + tok] = make_float2(L2, Dv);
      // ---- sweep 2: dS_c = A_c o (dA_c - D)
      const float mul = SUM ? a.scale : 1.f;
#pragma unroll 1
      for (int c = 0; c < NCH; ++c) {
        ok = wwait(sd_full, (u0 + NCH + c) & 1u, 0xF19);
        if (!ok) break;
        tc_fence_after();
        float v[64];
        uint32_t pk[32];
        tmem_ld32(t_sd, v);
        tmem_ld32(t_sd + 32, v + 32);
        tmem_ld32(t_a + c * (C::NC / 2), reinterpret_cast<float*>(pk));
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(sd_free);
#pragma unroll
        for (int k = 0; k < 32; ++k) {
          float x = lo16(pk[k]) * (v[2 * k] - Dv), y = hi16(pk[k]) * (v[2 * k + 1] - Dv);
          if (SUM) x *= mul, y *= mul;
          pk[k] = pack_bf16(x, y);
        }
        if (FUSE) {
          uint8_t* drow = smem + C::OFF_DS + (2 * c + sw) * BLK + row * 128;
#pragma unroll
          for (int k = 0; k < 8; ++k)
            *reinterpret_cast<uint4*>(drow + ((k ^ (row & 7)) << 4)) =
                make_uint4(pk[4 * k], pk[4 * k + 1], pk[4 * k + 2], pk[4 * k + 3]);
          fence_proxy_async_smem();
        }
        put_operand(c, pk);
        __syncwarp();
        if (lane == 0) mbar_arrive(ds_full + chunk_bar(li, c));
        if (c == 0 && !SUM) put_row(dV, o, dvp);
      }
      lse_cur = lse_nxt;
    }
    if (ok) finish(ntiles - 1, prev, false);
  }
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem, C::TMEM_COLS);
  }
}

template <int D, int P, bool FUSE, bool SUM>
static cudaError_t launch_t(const Args& a, int W, const float* dsk, const __nv_bfloat16* gbf, const float* lse,
                            float* Dco, void* dK, void* dV, cudaStream_t st) {
  using C = SCfg<D, P, FUSE, SUM>;
  CUtensorMap tk, tv, tq, tg;
  if (!make_kv_map(&tk, a.K, a.N, a.H, D) || !make_kv_map(&tv, a.V, a.N, a.H, D) ||
      !make_q_map(&tq, a.Q, a.uq ? a.B * a.H : a.H, a.P, D, C::NC))
    return cudaErrorInvalidValue;
  if (FUSE) tg = tq;  // unused: dsketch is converted in the kernel
  else if (!make_q_map(&tg, gbf, a.B * a.H, a.P, D, C::NC)) return cudaErrorInvalidValue;
  auto fn = &tc_bwd2_kernel<D, P, FUSE, SUM>;
  const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  fn<<<W, kThreads, C::SMEM, st>>>(tk, tv, tq, tg, a, dsk, lse, Dco, static_cast<__nv_bfloat16*>(dK),
                                   static_cast<__nv_bfloat16*>(dV));
  return cudaGetLastError();
}

template <int D, int P, bool FUSE>
static cudaError_t launch_sum_t(const Args& a, int W, const float* dsk, const __nv_bfloat16* gbf, const float* lse,
                                float* Dco, void* dK, void* dV, cudaStream_t st) {
  return a.sum_dx ? launch_t<D, P, FUSE, true>(a, W, dsk, gbf, lse, Dco, dK, dV, st)
                  : launch_t<D, P, FUSE, false>(a, W, dsk, gbf, lse, Dco, dK, dV, st);
}

}  // namespace tcs

cudaError_t launch_tc_bwd2_fused(const Args& a, int W, const float* dsk, const float* lse, void* dK, void* dV,
                                 cudaStream_t st) {
  if (a.N == 0) return cudaSuccess;
  if (a.d == 64 && a.P == 256) return tcs::launch_sum_t<64, 256, true>(a, W, dsk, nullptr, lse, nullptr, dK, dV, st);
  if (a.d == 64 && a.P == 128) return tcs::launch_sum_t<64, 128, true>(a, W, dsk, nullptr, lse, nullptr, dK, dV, st);
  if (a.d == 128 && a.P == 128) return tcs::launch_sum_t<128, 128, true>(a, W, dsk, nullptr, lse, nullptr, dK, dV, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_tc_bwd2_tok(const Args& a, int W, const __nv_bfloat16* gbf, const float* lse, float* Dco, void* dK,
                               void* dV, cudaStream_t st) {
  if (a.N == 0) return cudaSuccess;
  if (a.d == 128 && a.P == 512) return tcs::launch_sum_t<128, 512, false>(a, W, nullptr, gbf, lse, Dco, dK, dV, st);
  if (a.d == 128 && a.P == 256) return tcs::launch_sum_t<128, 256, false>(a, W, nullptr, gbf, lse, Dco, dK, dV, st);
  if (a.d == 64 && a.P == 512) return tcs::launch_sum_t<64, 512, false>(a, W, nullptr, gbf, lse, Dco, dK, dV, st);
  return cudaErrorInvalidValue;
}

}  // namespace sa
