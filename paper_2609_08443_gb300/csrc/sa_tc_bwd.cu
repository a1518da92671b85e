// tcgen05 / TMEM / TMA backward of the SA sketching step (sm_103a): the choice of
// kernels, and the token side for shapes whose weights do not stay in TMEM.
//
// Chain rule of Sec. 3.1 with upstream G = dL/dsketch[b, h] and the forward's
// per-token log-sum-exp (FlashSA's softmax statistic, Sec. 4.4), so the weights are
// recomputed as A = exp(S - lse) without any reduction.  Up to 512 prototypes run on
// the two-sweep kernel (sa_tc_bwd2.cu), with dQ in the same kernel where TMEM holds
// it; above that, and for the token-wise normalisation, tc_bwd_tok_kernel below
// computes dV, dK and D_i in one sweep.  dQ comes from prototype slices
// (sa_tc_bwd_dq.cu) wherever it is not fused.  Every wait is bounded.
#include <cuda.h>

#include "sa_ptx.cuh"
#include "sa_tc.cuh"
#include "sa_tc_common.cuh"

namespace sa {
namespace tcb {

using namespace ptx;
using namespace tcc;

// one token row of dV or dK (fp32 from TMEM) -> bf16 global row, columns
// [c0, c0 + NCOL) of this warpgroup's half
template <int NCOL>
__device__ __forceinline__ void store_row_bf16(uint32_t taddr, __nv_bfloat16* dst, float mul, bool valid) {
  float v[32];
#pragma unroll
  for (int c = 0; c < NCOL; c += 32) {
    tmem_ld32(taddr + c, v);
    tmem_ld_wait();
    if (valid) {
      uint4* o = reinterpret_cast<uint4*>(dst + c);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint4 pk;
        pk.x = pack_bf16(v[8 * k + 0] * mul, v[8 * k + 1] * mul);
        pk.y = pack_bf16(v[8 * k + 2] * mul, v[8 * k + 3] * mul);
        pk.z = pack_bf16(v[8 * k + 4] * mul, v[8 * k + 5] * mul);
        pk.w = pack_bf16(v[8 * k + 6] * mul, v[8 * k + 7] * mul);
        o[k] = pk;
      }
    }
  }
}

__device__ __forceinline__ float bf16lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

}  // namespace tcb

bool tc_bwd_supported(int P, int d, sa_dtype dt) {
  if (dt != SA_BF16 || !tcc::device_is_sm103() || !tc_path_enabled()) return false;
  return ((d == 64 || d == 128) && (P == 128 || P == 256 || P == 512 || P == 1024 || P == 2048));
}

const char* tc_bwd_name(int P, int d) {
  if (P == 2048) return d == 64 ? "tc_bwd_tok_kernel<64,2048>" : "tc_bwd_tok_kernel<128,2048>";
  if (P == 1024) return d == 64 ? "tc_bwd_tok_kernel<64,1024>" : "tc_bwd_tok_kernel<128,1024>";
  if (P == 512) return d == 64 ? "tc_bwd2_kernel<64,512>" : "tc_bwd2_kernel<128,512>";
  if (P == 256) return d == 64 ? "tc_bwd2_kernel<64,256,dq>" : "tc_bwd2_kernel<128,256>";
  return d == 64 ? "tc_bwd2_kernel<64,128,dq>" : "tc_bwd2_kernel<128,128,dq>";
}

int tc_bwd_workers(int num_sms, int, int) { return num_sms; }

}  // namespace sa

// ===================================================================== tokens
// Token side of the backward where the weights of a tile do not stay in TMEM
// (P > 512; token-wise): all P prototypes pass through the CTA in chunks of
// NC = 128 (Q and a bf16 copy of dsketch streamed by TMA), in one pass:
//   dV_i   = sum_j A[j,i] G_j                   (UMMA, accumulates over chunks)
//   u_i    = sum_j A[j,i] dA[j,i] Q_j            (UMMA on E = A o dA)
//   qbar_i = sum_j A[j,i] Q_j                    (UMMA)
//   D_i    = sum_j A[j,i] dA[j,i]                (registers)
//   dK_i   = scale (u_i - D_i qbar_i)            (= scale sum_j dS[j,i] Q_j)
// and D_i is written out for the prototype-side dQ slices.
namespace sa {
namespace tcb {

template <int D, int P>
struct TokCfg {
  static constexpr int NC = 128;
  static constexpr int NCH = P / NC;
  static constexpr int SLOT = T * D * 2;  // one K, V, Q-chunk or G-chunk tile (NC == T)
  static constexpr int NSLOT = 6;         // three pairs: (K, V) of a tile or (G, Q) of a chunk
  static constexpr int OFF_SLOTS = 0;
  static constexpr int OFF_AB = NSLOT * SLOT;  // A, then E = A o dA, of one chunk; epilogue staging
  static constexpr int OFF_STATS = OFF_AB + T * NC * 2;
  static constexpr int OFF_BAR = OFF_STATS + 2 * T * 4;
  static constexpr int NBAR = 2 * NSLOT + 20;
  static constexpr int OFF_MISC = OFF_BAR + NBAR * 8;
  static constexpr int SMEM = OFF_MISC + 16;
  // dV and qbar side by side: one N = 2D MMA against the adjacent G, Q chunks
  static constexpr int SD_COL = 0, DV_COL = NC, QB_COL = NC + D, U_COL = NC + 2 * D;
  static constexpr int TMEM_COLS = tmem_cols_for(NC + 3 * D);
  static constexpr int HALF = NC / 2;
  static_assert(NC == T && TMEM_COLS <= 512 && SMEM <= 232448, "budget");
};

// Where dA lands: with prototype-wise weights S and dA share SD_COL (TMEM is
// full); token-wise needs no qbar, so dA takes QB_COL and the two do not wait
// for each other.
template <int D, int P, bool TW>
__host__ __device__ constexpr int tok_da_col() {
  return TW ? TokCfg<D, P>::QB_COL : TokCfg<D, P>::SD_COL;
}

// Pair 0 holds the tile's K and V; the next tile's K loads into it once the
// tile's last S has read K, its V once the last dA has read V, and both tiles
// are pulled into L2 a tile ahead.  Chunks alternate between pairs 1 and 2
// (the chunk count per tile is even).  A chunk pair holds G in its first slot
// and Q in the second, so the four 64-column blocks of G and Q sit at one
// stride and [G | Q] is a single N = 2D operand.
__device__ __forceinline__ int tok_kv_pair(int) { return 0; }
__device__ __forceinline__ int tok_qg_pair(int, int c) { return 1 + (c & 1); }

// TW = false: prototype-wise weights (Sec. 3.1), lse per token and head; Dco is
// written here, float2 [H][N] (lse log2 e, D_i).  TW = true: token-wise weights (Sec. 5.1), lse and Dco
// per prototype [B][H][P] (both read), so dS = A o (dA - D_j) goes to shared
// memory in place of E and dK = scale dS Q needs no qbar.
// SUM: K = V = X, and dV's buffer takes dV + dK (Args::sum_dx; not token-wise).
template <int D, int P, bool TW, bool SUM>
__device__ __forceinline__ void bwd_tok_body(const CUtensorMap& tmK, const CUtensorMap& tmV, const CUtensorMap& tmQ,
                                             const CUtensorMap& tmG, const CUtensorMap& tmDK,
                                             const CUtensorMap& tmDV, const Args& a, const float* lse,
                                             float* Dco, __nv_bfloat16* __restrict__ dK,
                                             __nv_bfloat16* __restrict__ dV) {
  using C = TokCfg<D, P>;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (cta_leaves(a.ws, smem_u32(smem), 0xB21u)) return;
  const uint32_t sbase = smem_u32(smem);
  const uint32_t sSlots = sbase + C::OFF_SLOTS, sAB = sbase + C::OFF_AB;
  auto slot_addr = [&](int s) { return sSlots + uint32_t(s) * C::SLOT; };
  const uint32_t bar0 = sbase + C::OFF_BAR;
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (C::NSLOT + s); };
  const uint32_t b1 = bar0 + 8u * (2 * C::NSLOT);
  const uint32_t s_full = b1, sd_free_s = b1 + 8, da_full = b1 + 16, sd_free_da = b1 + 24, a_full = b1 + 32,
                 ab_free_a = b1 + 40, e_full = b1 + 48, ab_free_e = b1 + 56, acc_full = b1 + 64,
                 acc_empty = b1 + 72, st_ready = b1 + 80, st_used = b1 + 88, epi_ready = b1 + 96, epi_free = b1 + 104,
                 drain = b1 + 112;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::OFF_MISC + 4);
  const int64_t tph = reinterpret_cast<const WsHeader*>(a.ws)->tiles_per_head;
  const int64_t total = tph * a.H;
  const int W = gridDim.x, wk = blockIdx.x;
  const int64_t tb = range_begin(total, W, wk), te = range_begin(total, W, wk + 1);
  const int ntiles = int(te - tb);
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::NSLOT; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(s_full, 1);
    mbar_init(sd_free_s, kSoftWarps);
    mbar_init(da_full, 1);
    mbar_init(sd_free_da, kSoftWarps);
    mbar_init(a_full, kSoftWarps);
    mbar_init(ab_free_a, 1);
    mbar_init(e_full, kSoftWarps);
    mbar_init(ab_free_e, 1);
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, kSoftWarps);
    mbar_init(st_ready, kSoftWarps);
    mbar_init(st_used, kSoftWarps);
    mbar_init(epi_ready, kSoftWarps);
    mbar_init(epi_free, 1);
    mbar_init(drain, 1);
    wait_ctl_init(abort_flag, a.ws);
    fence_mbar_init();
  }
  if (warp == 2) tmem_alloc(smem_u32(tmem_slot), C::TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // Registers: the control warpgroup (warps 0-3) hands registers to the two
  // softmax warpgroups (128 x 152 + 256 x 176 = 384 x 168, the launch allocation).
  if (ntiles > 0 && warp < kSoftWarp0) {
    setmaxnreg_dec<152>();
    if (warp == 0 && lane == 0) {
      // ---------------------------------------------------------- TMA producer
      tma_prefetch_desc(&tmK);
      tma_prefetch_desc(&tmV);
      tma_prefetch_desc(&tmQ);
      tma_prefetch_desc(&tmG);
      TileWalker it(a, tb, te, T), nx(a, tb, te, T);
      nx.next();
      static_assert(C::NCH % 2 == 0, "chunks alternate between two pairs");
      // per slot, as bits (registers, not an indexed array): loaded before, and
      // the parity of the wait for its next release
      uint32_t used = 0u, par = 0u;
      bool ok = true;
      // box origin (64*dh, c1, c2): K / V maps are (d, head, token); Q / G maps
      // are (d, prototype, head) and (d, prototype, user*H + head)
      auto load = [&](int s, const CUtensorMap* map, int c1, int c2) {
        if ((used >> s) & 1u) {
          ok = ok && mbar_wait(empty_bar(s), (par >> s) & 1u, abort_flag, a.ws, 0x801);
          if (!ok) return;  // par stays that of the slot's last load, which the drain below waits for
          par ^= 1u << s;
        }
        if (!ok) return;
        used |= 1u << s;
        mbar_arrive_expect_tx(full_bar(s), C::SLOT);
#pragma unroll
        for (int dh = 0; dh < D / 64; ++dh) tma_load_3d(slot_addr(s) + dh * T * 128, map, full_bar(s), 64 * dh, c1, c2);
      };
      auto prefetch_kv = [&](const TileWalker& w) {
#pragma unroll
        for (int dh = 0; dh < D / 64; ++dh) {
          tma_prefetch_l2_3d(&tmK, 64 * dh, w.h, int(w.tok0));
          tma_prefetch_l2_3d(&tmV, 64 * dh, w.h, int(w.tok0));
        }
      };
      // Order of loads: ..., Q/G(li, last), K(li+1), Q/G(li+1, 0), V(li+1), ...:
      // K(li+1) waits for S(li, last), V(li+1) for dA(li, last).
      load(0, &tmK, it.h, int(it.tok0));
      load(1, &tmV, it.h, int(it.tok0));
      if (ntiles > 1) prefetch_kv(nx);
      for (int li = 0; li < ntiles && ok; ++li) {
        for (int c = 0; c < C::NCH && ok; ++c) {
          const int pr = tok_qg_pair(li, c);
          load(2 * pr + 1, &tmQ, c * C::NC, it.qk);
          load(2 * pr, &tmG, c * C::NC, int(it.b) * a.H + it.h);
          if (c == 0 && li > 0) load(1, &tmV, it.h, int(it.tok0));
          if (c == C::NCH - 1 && li + 1 < ntiles) load(0, &tmK, nx.h, int(nx.tok0));
        }
        it.next();
        nx.next();
        if (li + 2 < ntiles) prefetch_kv(nx);
      }
      if (!ok) {
        for (int s = 0; s < C::NSLOT; ++s)
          if ((used >> s) & 1u) mbar_wait_bounded(full_bar(s), (par >> s) & 1u, 200000000ull);
      }
    } else if (warp == 1) {
      // ---------------------------------------------------------- UMMA issuer
      // Per chunk g: dA_g, [dV | qbar]_g, S_{g+1}, u_g.  Shared-memory
      // descriptors are built once per operand and stepped by constant offsets,
      // so the issue loop carries no address arithmetic.
      constexpr uint32_t idS = idesc_bf16(128, C::NC, 0, 0);    // [tok x chunk], K = d
      constexpr uint32_t idGQ = idesc_bf16(128, TW ? D : 2 * D, 0, 1);  // [tok x (d | d)] (TW: d), K = chunk
      constexpr uint32_t idU = idesc_bf16(128, D, 0, 1);        // [tok x d], K = chunk prototypes
      bool ok = true;
      uint32_t fpar = 0u;  // per slot, as bits: parity of the next "full" phase
      auto wt = [&](uint32_t bar, uint32_t parity, uint32_t site) {
        return ok = ok && mbar_wait_warp(bar, parity, abort_flag, a.ws, site);
      };
      auto wfull = [&](int s, uint32_t site) {
        wt(full_bar(s), (fpar >> s) & 1u, site);
        fpar ^= 1u << s;
      };
      // K-major [128 rows x D] operand: K step k at +(k / 4) * 128 rows + (k % 4) * 32 B
      auto kmaj = [](uint32_t addr) { return sdesc(addr, 16, 1024); };
      auto kstep = [](int k) { return uint32_t((k >> 2) * (T * 128) + (k & 3) * 32); };
      const uint64_t dAB = kmaj(sAB);
      const uint32_t nchunks = uint32_t(ntiles) * C::NCH;
      auto issue_S = [&](uint32_t g) {
        const int li = int(g / C::NCH), c = int(g % C::NCH);
        const uint64_t dK = kmaj(slot_addr(2 * tok_kv_pair(li))), dQ = kmaj(slot_addr(2 * tok_qg_pair(li, c) + 1));
#pragma unroll
        for (int k = 0; k < D / 16; ++k)
          umma_ss(tmem + C::SD_COL, sdesc_add(dK, kstep(k)), sdesc_add(dQ, kstep(k)), idS, k > 0 ? 1u : 0u);
        umma_commit(s_full);
        if (c == C::NCH - 1) umma_commit(empty_bar(2 * tok_kv_pair(li)));  // last S: K free
      };
      wfull(2 * tok_kv_pair(0), 0x901);
      wfull(2 * tok_qg_pair(0, 0) + 1, 0x902);
      if (ok) {
        tc_fence_after();
        if (elect_one()) issue_S(0);
      }
      for (uint32_t g = 0; g < nchunks && ok; ++g) {
        const int li = int(g / C::NCH), c = int(g % C::NCH);
        const int kvp = tok_kv_pair(li), qgp = tok_qg_pair(li, c);
        const uint32_t aG = slot_addr(2 * qgp), aQ = slot_addr(2 * qgp + 1);
        // ---- dA_g = V G_g^T (into S's columns once S_g is read, or, token-wise,
        // into its own columns once dA_{g-1} is read)
        {
          const BarPhase gf{full_bar(2 * qgp), (fpar >> (2 * qgp)) & 1u};
          const BarPhase three[3] = {gf, c == 0 ? BarPhase{full_bar(2 * kvp + 1), (fpar >> (2 * kvp + 1)) & 1u} : gf,
                                     !TW ? BarPhase{sd_free_s, g & 1u} : g > 0 ? BarPhase{sd_free_da, (g - 1) & 1u} : gf};
          ok = ok && mbar_wait_warp_all(three, abort_flag, a.ws, 0x904);
          fpar ^= (1u << (2 * qgp)) | (c == 0 ? 1u << (2 * kvp + 1) : 0u);
        }
        if (!ok) break;
        tc_fence_after();
        if (elect_one()) {
          const uint64_t dV = kmaj(slot_addr(2 * kvp + 1)), dG = kmaj(aG);
#pragma unroll
          for (int k = 0; k < D / 16; ++k)
            umma_ss(tmem + tok_da_col<D, P, TW>(), sdesc_add(dV, kstep(k)), sdesc_add(dG, kstep(k)), idS,
                    k > 0 ? 1u : 0u);
          umma_commit(da_full);
          if (c == C::NCH - 1) umma_commit(empty_bar(2 * kvp + 1));  // last dA: V free
        }
        // ---- [dV | qbar] += A [G_g | Q_g]
        {
          const BarPhase af{a_full, g & 1u};
          const BarPhase both[2] = {af, c == 0 && li > 0 ? BarPhase{acc_empty, uint32_t(li - 1) & 1u} : af};
          ok = ok && mbar_wait_warp_all(both, abort_flag, a.ws, 0x906);
        }
        if (!ok) break;
        tc_fence_after();
        if (elect_one()) {
          const uint64_t dGQ = sdesc(aG, C::NC * 128, 1024);  // MN-major, 64-column blocks 16 KB apart
#pragma unroll
          for (int k = 0; k < C::NC / 16; ++k)
            umma_ss(tmem + C::DV_COL, sdesc_add(dAB, kstep(k)), sdesc_add(dGQ, k * 2048), idGQ,
                    (c == 0 && k == 0) ? 0u : 1u);
          umma_commit(ab_free_a);
          umma_commit(empty_bar(2 * qgp));  // G chunk free
        }
        // ---- S_{g+1}
        if (g + 1 < nchunks) {
          const uint32_t gn = g + 1;
          const int lin = int(gn / C::NCH), cn = int(gn % C::NCH);
          const int sk = 2 * tok_kv_pair(lin), sq = 2 * tok_qg_pair(lin, cn) + 1;
          const BarPhase qf{full_bar(sq), (fpar >> sq) & 1u};
          const BarPhase three[3] = {qf, cn == 0 ? BarPhase{full_bar(sk), (fpar >> sk) & 1u} : qf,
                                     {TW ? sd_free_s : sd_free_da, g & 1u}};  // S's columns read
          ok = ok && mbar_wait_warp_all(three, abort_flag, a.ws, 0x909);
          fpar ^= (1u << sq) | (cn == 0 ? 1u << sk : 0u);
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) issue_S(gn);
        }
        // ---- u += E Q_g
        wt(e_full, g & 1, 0x90B);
        if (!ok) break;
        tc_fence_after();
        if (elect_one()) {
          const uint64_t dQm = sdesc(aQ, C::NC * 128, 1024);
#pragma unroll
          for (int k = 0; k < C::NC / 16; ++k)
            umma_ss(tmem + C::U_COL, sdesc_add(dAB, kstep(k)), sdesc_add(dQm, k * 2048), idU,
                    (c == 0 && k == 0) ? 0u : 1u);
          umma_commit(ab_free_e);
          umma_commit(empty_bar(2 * qgp + 1));  // Q chunk free
          if (c == C::NCH - 1) umma_commit(acc_full);
        }
      }
      if (elect_one()) umma_commit(drain);
      mbar_wait_bounded(drain, 0, 200000000ull);
    }
  } else if (ntiles > 0) {
    setmaxnreg_inc<176>();
    {
      // ------------------------------------------------ softmax + epilogue
      const int sw = (warp - kSoftWarp0) >> 2, q = warp & 3, row = 32 * q + lane;
      const uint32_t lane_off = uint32_t(32 * q) << 16;
      const float c2 = a.scale * 1.4426950408889634f;
      float* stats = reinterpret_cast<float*>(smem + C::OFF_STATS);
      TileWalker cur(a, tb, te, T);
      bool ok = true;
      auto wwait = [&](uint32_t bar, uint32_t par, uint32_t site) {
        return __all_sync(0xffffffffu, mbar_wait(bar, par, abort_flag, a.ws, site));
      };
      uint32_t g = 0;
      int epi = 0;  // staged epilogue stores so far
      auto put_tile = [&](const uint32_t* pk) {
        uint8_t* rowp = smem + C::OFF_AB + row * 128;
#pragma unroll
        for (int k = 0; k < C::HALF / 8; ++k) {
          const int p = sw * C::HALF + 8 * k;
          const int blk = p >> 6, chunk = (p & 63) >> 3;
          *reinterpret_cast<uint4*>(rowp + blk * (T * 128) + ((chunk ^ (row & 7)) << 4)) =
              make_uint4(pk[4 * k], pk[4 * k + 1], pk[4 * k + 2], pk[4 * k + 3]);
        }
      };
      // one staged [128 tokens][D] bf16 tile in AB -> global through TMA
      auto stage_and_store = [&](const CUtensorMap* map, const TileWalker& w) -> bool {
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(epi_ready);
        if (warp == kSoftWarp0 && lane == 0) {
          if (mbar_wait(epi_ready, epi & 1, abort_flag, a.ws, 0xA08)) {
#pragma unroll
            for (int dh = 0; dh < D / 64; ++dh) tma_store_3d(map, sAB + dh * T * 128, 64 * dh, w.h, int(w.tok0));
            bulk_commit_group();
            bulk_wait_read_all();
          }
          mbar_arrive(epi_free);
        }
        const bool r = wwait(epi_free, epi & 1, 0xA09);
        ++epi;
        return r;
      };
      float lse_cur = (!TW && row < cur.n) ? load_token_lse(lse, a, cur.tok0 + row, cur.h) : 0.f;
      for (int li = 0; li < ntiles && ok; ++li) {
        const bool valid = row < cur.n;
        const int64_t tok = cur.tok0 + row;
        const float L2 = lse_cur * 1.4426950408889634f;
        if (!TW) {
          int64_t t0n;
          int nn, hn;
          cur.peek_next(t0n, nn, hn);
          lse_cur = row < nn ? load_token_lse(lse, a, t0n + row, hn) : 0.f;
        }
        // token-wise: this segment's per-prototype lse and D_j (the same for
        // every thread: broadcast loads)
        const int64_t seg_row = (int64_t(cur.b) * a.H + cur.h) * a.P;
        float Dp = 0.f;
        for (int c = 0; c < C::NCH && ok; ++c, ++g) {
          uint32_t apk[C::HALF / 2];
          float v[C::HALF];  // this warpgroup's columns of S, then of dA (both loads before one wait)
          const int j0 = c * C::NC + sw * C::HALF;  // first prototype of this warpgroup's columns
          ok = wwait(s_full, g & 1, 0xA01);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int cc = 0; cc < C::HALF / 32; ++cc) tmem_ld32(tmem + lane_off + C::SD_COL + sw * C::HALF + 32 * cc, v + 32 * cc);
          tmem_ld_wait();
          // S is in registers: its columns may take dA_g (or S_{g+1}) while the weights are formed
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(sd_free_s);
#pragma unroll
          for (int cc = 0; cc < C::HALF / 32; ++cc) {
            if (TW) {
              const float4* l4 = reinterpret_cast<const float4*>(lse + seg_row + j0 + 32 * cc);
#pragma unroll
              for (int j4 = 0; j4 < 8; ++j4) {
                const float4 l = __ldg(l4 + j4);
                const float x0 = valid ? ex2(fmaf(v[32 * cc + 4 * j4 + 0], c2, -l.x * 1.4426950408889634f)) : 0.f;
                const float x1 = valid ? ex2(fmaf(v[32 * cc + 4 * j4 + 1], c2, -l.y * 1.4426950408889634f)) : 0.f;
                const float x2 = valid ? ex2(fmaf(v[32 * cc + 4 * j4 + 2], c2, -l.z * 1.4426950408889634f)) : 0.f;
                const float x3 = valid ? ex2(fmaf(v[32 * cc + 4 * j4 + 3], c2, -l.w * 1.4426950408889634f)) : 0.f;
                apk[16 * cc + 2 * j4] = pack_bf16(x0, x1);
                apk[16 * cc + 2 * j4 + 1] = pack_bf16(x2, x3);
              }
            } else {
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const float x0 = valid ? ex2(fmaf(v[32 * cc + 2 * j], c2, -L2)) : 0.f;
                const float x1 = valid ? ex2(fmaf(v[32 * cc + 2 * j + 1], c2, -L2)) : 0.f;
                apk[16 * cc + j] = pack_bf16(x0, x1);
              }
            }
          }
          if (g > 0) {
            ok = wwait(ab_free_e, (g - 1) & 1, 0xA02);  // u of the previous chunk has read E
            if (!ok) break;
          }
          put_tile(apk);
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(a_full);
          // E = A o dA (token-wise: dS = A o (dA - D_j))
          ok = wwait(da_full, g & 1, 0xA03);
          if (!ok) break;
          tc_fence_after();
          uint32_t epk[C::HALF / 2];
#pragma unroll
          for (int cc = 0; cc < C::HALF / 32; ++cc)
            tmem_ld32(tmem + lane_off + tok_da_col<D, P, TW>() + sw * C::HALF + 32 * cc, v + 32 * cc);
          tmem_ld_wait();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(sd_free_da);
#pragma unroll
          for (int cc = 0; cc < C::HALF / 32; ++cc) {
            if (TW) {
              const float4* d4 = reinterpret_cast<const float4*>(Dco + seg_row + j0 + 32 * cc);
#pragma unroll
              for (int j4 = 0; j4 < 8; ++j4) {
                const float4 dd = __ldg(d4 + j4);
                const uint32_t w0 = apk[16 * cc + 2 * j4], w1 = apk[16 * cc + 2 * j4 + 1];
                epk[16 * cc + 2 * j4] = pack_bf16(bf16lo(w0) * (v[32 * cc + 4 * j4 + 0] - dd.x),
                                                  bf16hi(w0) * (v[32 * cc + 4 * j4 + 1] - dd.y));
                epk[16 * cc + 2 * j4 + 1] = pack_bf16(bf16lo(w1) * (v[32 * cc + 4 * j4 + 2] - dd.z),
                                                      bf16hi(w1) * (v[32 * cc + 4 * j4 + 3] - dd.w));
              }
            } else {
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const uint32_t w = apk[16 * cc + j];
                const float e0 = bf16lo(w) * v[32 * cc + 2 * j], e1 = bf16hi(w) * v[32 * cc + 2 * j + 1];
                Dp += e0 + e1;
                epk[16 * cc + j] = pack_bf16(e0, e1);
              }
            }
          }
          ok = wwait(ab_free_a, g & 1, 0xA04);  // dV and qbar have read A
          if (!ok) break;
          put_tile(epk);
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(e_full);
        }
        if (!ok) break;
        // D_i = (half from warpgroup 0) + (half from warpgroup 1), same order in
        // both; token-wise: u already is sum_j dS[j,i] Q_j, so D_i = 0 below
        float Dv = 0.f;
        if (!TW) {
          if (li > 0) {
            ok = wwait(st_used, (li - 1) & 1, 0xA05);
            if (!ok) break;
          }
          stats[sw * T + row] = Dp;
          __syncwarp();
          if (lane == 0) mbar_arrive(st_ready);
          ok = wwait(st_ready, li & 1, 0xA06);
          if (!ok) break;
          Dv = stats[row] + stats[T + row];
          __syncwarp();
          if (lane == 0) mbar_arrive(st_used);
          if (sw == 0 && valid) reinterpret_cast<float2*>(Dco)[int64_t(cur.h) * a.N + tok] = make_float2(L2, Dv);
        }
        // epilogue: dV and dK = scale (u - D qbar); this warpgroup owns columns [sw*D/2, +D/2)
        ok = wwait(acc_full, li & 1, 0xA07);
        if (!ok) break;
        tc_fence_after();
        const bool whole = cur.n == T;  // a full tile is stored by TMA; a ragged tail row by row
        uint8_t* rowp = smem + C::OFF_AB + row * 128;
        auto put_half = [&](const float* x, int cc) {  // 32 columns [sw*D/2 + cc, +32) of this row
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int col = sw * (D / 2) + cc + 8 * k;
            const int dh = col >> 6, chunk = (col & 63) >> 3;
            *reinterpret_cast<uint4*>(rowp + dh * (T * 128) + ((chunk ^ (row & 7)) << 4)) =
                make_uint4(pack_bf16(x[8 * k], x[8 * k + 1]), pack_bf16(x[8 * k + 2], x[8 * k + 3]),
                           pack_bf16(x[8 * k + 4], x[8 * k + 5]), pack_bf16(x[8 * k + 6], x[8 * k + 7]));
          }
        };
        // with K = V = X (SUM) one tile dV + dK, summed in fp32, goes to dV's buffer
        if (whole) {
          float x[32];
          if (!SUM) {
#pragma unroll
            for (int cc = 0; cc < D / 2; cc += 32) {
              tmem_ld32(tmem + lane_off + C::DV_COL + sw * (D / 2) + cc, x);
              tmem_ld_wait();
              put_half(x, cc);
            }
            ok = stage_and_store(&tmDV, cur);
            if (!ok) break;
          }
          float uu[32], qb[32];
#pragma unroll
          for (int cc = 0; cc < D / 2; cc += 32) {
            tmem_ld32(tmem + lane_off + C::U_COL + sw * (D / 2) + cc, uu);
            if (!TW) tmem_ld32(tmem + lane_off + C::QB_COL + sw * (D / 2) + cc, qb);
            if (SUM) tmem_ld32(tmem + lane_off + C::DV_COL + sw * (D / 2) + cc, x);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              uu[j] = TW ? a.scale * uu[j] : a.scale * fmaf(-Dv, qb[j], uu[j]);
              if (SUM) uu[j] += x[j];
            }
            put_half(uu, cc);
          }
          ok = stage_and_store(SUM ? &tmDV : &tmDK, cur);
          if (!ok) break;
        } else {
          __nv_bfloat16* dvr = dV + (tok * a.H + cur.h) * int64_t(D) + sw * (D / 2);
          if (!SUM) store_row_bf16<D / 2>(tmem + lane_off + C::DV_COL + sw * (D / 2), dvr, 1.f, valid);
          __nv_bfloat16* dkr =
              SUM ? dvr : dK + (tok * a.H + cur.h) * int64_t(D) + sw * (D / 2);
          float uu[32], qb[32];
#pragma unroll
          for (int cc = 0; cc < D / 2; cc += 32) {
            tmem_ld32(tmem + lane_off + C::U_COL + sw * (D / 2) + cc, uu);
            if (!TW) tmem_ld32(tmem + lane_off + C::QB_COL + sw * (D / 2) + cc, qb);
            float dv[32];
            if (SUM) tmem_ld32(tmem + lane_off + C::DV_COL + sw * (D / 2) + cc, dv);
            tmem_ld_wait();
            if (valid) {
              uint4* o = reinterpret_cast<uint4*>(dkr + cc);
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                float x[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  x[j] = TW ? a.scale * uu[8 * k + j] : a.scale * fmaf(-Dv, qb[8 * k + j], uu[8 * k + j]);
                  if (SUM) x[j] += dv[8 * k + j];
                }
                o[k] = make_uint4(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]), pack_bf16(x[4], x[5]),
                                  pack_bf16(x[6], x[7]));
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty);
        cur.next();
      }
      if (warp == kSoftWarp0 && lane == 0) bulk_wait_all();  // stores complete before exit
    }
  }
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem, C::TMEM_COLS);
  }
}

template <int D, int P, bool SUM>
__global__ void __launch_bounds__(kThreads, 1)
    tc_bwd_tok_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                      const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmG,
                      const __grid_constant__ CUtensorMap tmDK, const __grid_constant__ CUtensorMap tmDV, Args a,
                      const float* lse, float* Dco, __nv_bfloat16* __restrict__ dK,
                      __nv_bfloat16* __restrict__ dV) {
  bwd_tok_body<D, P, false, SUM>(tmK, tmV, tmQ, tmG, tmDK, tmDV, a, lse, Dco, dK, dV);
}

template <int D, int P>
__global__ void __launch_bounds__(kThreads, 1)
    tc_tw_bwd_tok_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                         const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmG,
                         const __grid_constant__ CUtensorMap tmDK, const __grid_constant__ CUtensorMap tmDV, Args a,
                         const float* __restrict__ lse_tok, float* __restrict__ Dtw, __nv_bfloat16* __restrict__ dK,
                         __nv_bfloat16* __restrict__ dV) {
  bwd_tok_body<D, P, true, false>(tmK, tmV, tmQ, tmG, tmDK, tmDV, a, lse_tok, Dtw, dK, dV);
}

// dsketch fp32 -> bf16 copy in the workspace, the layout TMA streams ([B*H][P][D])
__global__ void to_bf16_kernel(const float* __restrict__ src, __nv_bfloat16* __restrict__ dst, int64_t n8,
                               const void* ws) {
  if (ws_failed(ws)) return;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n8; i += int64_t(gridDim.x) * blockDim.x) {
    const float4 x = reinterpret_cast<const float4*>(src)[2 * i];
    const float4 y = reinterpret_cast<const float4*>(src)[2 * i + 1];
    reinterpret_cast<uint4*>(dst)[i] =
        make_uint4(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w), pack_bf16(y.x, y.y), pack_bf16(y.z, y.w));
  }
}

template <int D, int P, bool TW = false>
static cudaError_t launch_tok_t(const Args& a, int W, const __nv_bfloat16* gbf, const float* lse, float* Dco,
                                void* dK, void* dV, cudaStream_t st) {
  using C = TokCfg<D, P>;
  CUtensorMap tk, tv, tq, tg, tdk, tdv;
  if (!make_kv_map(&tk, a.K, a.N, a.H, D) || !make_kv_map(&tv, a.V, a.N, a.H, D) ||
      !make_q_map(&tq, a.Q, a.uq ? a.B * a.H : a.H, a.P, D, C::NC) || !make_q_map(&tg, gbf, a.B * a.H, a.P, D, C::NC) ||
      !make_kv_map(&tdk, dK, a.N, a.H, D) || !make_kv_map(&tdv, dV, a.N, a.H, D))
    return cudaErrorInvalidValue;
  auto fn = [&] {
    if constexpr (TW) return &tc_tw_bwd_tok_kernel<D, P>;
    else return a.sum_dx ? &tc_bwd_tok_kernel<D, P, true> : &tc_bwd_tok_kernel<D, P, false>;
  }();
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  fn<<<W, kThreads, C::SMEM, st>>>(tk, tv, tq, tg, tdk, tdv, a, lse, Dco, static_cast<__nv_bfloat16*>(dK),
                                   static_cast<__nv_bfloat16*>(dV));
  return cudaGetLastError();
}

}  // namespace tcb

bool tc_bwd_split(int P, int d) {
  return (d == 128 && (P == 256 || P == 512 || P == 1024 || P == 2048)) ||
         (d == 64 && (P == 512 || P == 1024 || P == 2048));
}

cudaError_t launch_tc_g_bf16(const Args& a, const float* dsk, __nv_bfloat16* gbf, cudaStream_t st) {
  const int64_t n8 = int64_t(a.B) * a.H * a.P * a.d / 8;
  tcb::to_bf16_kernel<<<1024, 256, 0, st>>>(dsk, gbf, n8, a.ws);
  return cudaGetLastError();
}

cudaError_t launch_tc_bwd_tok(const Args& a, int W, const __nv_bfloat16* gbf, const float* lse, float* Dco, void* dK,
                              void* dV, cudaStream_t st) {
  if (a.N == 0) return cudaSuccess;
  if (a.P <= 512) return launch_tc_bwd2_tok(a, W, gbf, lse, Dco, dK, dV, st);
  if (a.d == 64)
    return a.P == 2048 ? tcb::launch_tok_t<64, 2048>(a, W, gbf, lse, Dco, dK, dV, st)
                       : tcb::launch_tok_t<64, 1024>(a, W, gbf, lse, Dco, dK, dV, st);
  return a.P == 2048 ? tcb::launch_tok_t<128, 2048>(a, W, gbf, lse, Dco, dK, dV, st)
                     : tcb::launch_tok_t<128, 1024>(a, W, gbf, lse, Dco, dK, dV, st);
}

int tc_bwd_dq_workers(int num_sms, int P) {
  const int w = num_sms / (P / 128);
  return w < 1 ? 1 : w;
}

}  // namespace sa

namespace sa {
// Token-wise normalisation (Sec. 5.1): the same two kernels with per-prototype
// lse_tok and D_j = G_j . O_j ([B][H][P]); d = 128 and P in {256, ..., 2048}.
bool tc_tw_bwd_supported(int P, int d, sa_dtype dt) {
  return dt == SA_BF16 && d == 128 && (P == 256 || P == 512 || P == 1024 || P == 2048) && tcc::device_is_sm103() &&
         tc_path_enabled();
}

cudaError_t launch_tc_tw_bwd_tok(const Args& a, int W, const __nv_bfloat16* gbf, const float* lse_tok,
                                 const float* Dtw, void* dK, void* dV, cudaStream_t st) {
  if (a.N == 0) return cudaSuccess;
  float* Dp = const_cast<float*>(Dtw);  // read only in token-wise mode
  if (a.P == 2048) return tcb::launch_tok_t<128, 2048, true>(a, W, gbf, lse_tok, Dp, dK, dV, st);
  if (a.P == 1024) return tcb::launch_tok_t<128, 1024, true>(a, W, gbf, lse_tok, Dp, dK, dV, st);
  if (a.P == 512) return tcb::launch_tok_t<128, 512, true>(a, W, gbf, lse_tok, Dp, dK, dV, st);
  return tcb::launch_tok_t<128, 256, true>(a, W, gbf, lse_tok, Dp, dK, dV, st);
}

}  // namespace sa
