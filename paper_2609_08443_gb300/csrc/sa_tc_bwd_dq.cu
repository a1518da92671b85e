// Prototype side of the backward (sm_103a): dQ of one slice of 128 prototypes per
// CTA, prototypes on TMEM lanes, tokens on columns:
//   S^T = Q_r K^T,  dA^T = G_r V^T             (UMMA, [128 x tokens])
//   dS  = exp(scale S - lse_t) o (dA - D_t)    (registers)
//   dQ_r += dS K                               (UMMA)
// D_t comes from the token-side kernel, with lse_t beside it: float2 [H][N] (lse
// log2 e, D), so a tile's 128 tokens are one bulk copy that travels with its K.
//
// What bounds it: a 128 x 128 x 16 UMMA with both operands in shared memory reads 8
// KB in its 64 cycles, all of the SM's 128 B/cycle; while such a group runs, every
// other shared-memory access (barrier polls above all) takes hundreds of cycles, and
// with one S/dA buffer those waits lie on the chain S -> dS -> dQ.
// So all three products take their A operand from TMEM: Q_r and G_r are written
// there as bf16 pairs when a run or segment starts, dS where its S was, which
// leaves B alone in shared memory (half the bandwidth).  And each tile runs as two
// independent halves of 64 tokens, one per softmax warpgroup, each with its own S
// and dA columns: while one half's dS is formed the other half's products run.
// lse_t and D_t are per-column values, read as broadcasts of four from shared memory
// (32 vector loads per thread and half, 1024 cycles of the load path per tile, issued
// ahead of the waits for the products).  Adding them in the products instead (ones
// times their three bf16 terms as one more K step) is 13% faster, but rounds the
// exponent in the accumulator at the size of lse / scale: enough bf16 weights flip
// that dQ differs by 3e-5 from the order of operations used here (2e-6 with it).
// The issuers wait for all that a tile needs in one round of polls and read the next
// tile's flags a tile ahead: seven waits in turn, 250-450 cycles each although
// satisfied, had cost 2100 cycles per tile.
// Measured: 16 users of 100K tokens (H = 8, P = 512, d = 128) 4.37 ms before, 3.58 ms
// now; 12 users, 215K tokens, token-wise 678 and 452 us; P = 1024, 141K tokens, 797
// and 622 us.  With lse and D as two arrays of their own, copied one by one, the first
// took 3.92 ms; with lse in natural units, scaled when it is laid out, 3.72.
// TMEM: per half S 64 (dS over its first 32) and dA 64, G D/2, Q D/2, dQ D columns.
//
// Warp roles: 0 tile sequence, loads; 1 issues S and dA, 2 (also TMEM) issues dQ; 3
// lays out the per-token values; 4-7 and 8-11 the two halves.
#include <cuda.h>

#include "sa_ptx.cuh"
#include "sa_tc.cuh"
#include "sa_tc_common.cuh"

namespace sa {
namespace tcd {

using namespace ptx;
using namespace tcc;

constexpr uint32_t kRegsCtl = 136, kRegsSoft = 184;
static_assert(128 * kRegsCtl + 256 * kRegsSoft == 384 * 168, "register split = launch allocation");
constexpr float kLog2e = 1.4426950408889634f;

// What the other roles need of a tile, written by warp 0 into a ring.  A run is a
// sequence of tiles that read one row of Q: a head, or with per-user queries one
// (user, head) segment.
struct TileInfo {
  int64_t tok0;
  float* dq_dst;  // last tile of a run: where the run's dQ slice goes
  int h, n, b;
  uint32_t flags;
};
enum : uint32_t { kRunFirst = 1u, kRunLast = 2u, kSegFirst = 4u, kSegLast = 8u };

template <int D>
struct DCfg {
  static constexpr int PS = 128, HT = T / 2;  // prototypes per slice, tokens per half
  static constexpr int ND = D / 64, BLK = T * 128, TILE = ND * BLK;
  // K(i) is read by S(i) and, a tile later, by dQ(i); V(i) only by dA(i)
  static constexpr int NK = 3, NV = 2, NI = 4;
  static constexpr int OFF_K = 0, OFF_V = NK * TILE;
  // per-token values of two tiles: [2 bufs][lse log2 e, D][128 tokens]
  static constexpr int OFF_COL = OFF_V + NV * TILE, COL = 2 * T * 4;
  // raw (lse log2 e, D) of the tile in each K slot: the copy starts at an even index
  static constexpr int RAW = (T + 2) * 8;
  static constexpr int OFF_RAW = OFF_COL + 2 * COL;
  static constexpr int OFF_INFO = OFF_RAW + NK * RAW;
  static constexpr int OFF_BAR = OFF_INFO + NI * int(sizeof(TileInfo));
  static constexpr int NBAR = 2 * NK + 2 * NV + 2 * NI + 20;
  static constexpr int OFF_MISC = OFF_BAR + NBAR * 8;
  static constexpr int SMEM = OFF_MISC + 16;
  static constexpr int S_COL = 0, DA_COL = HT, HALF_COLS = 2 * HT;  // half h at h * HALF_COLS
  static constexpr int G_COL = 2 * HALF_COLS, Q_COL = G_COL + D / 2, DQ_COL = Q_COL + D / 2;
  static constexpr int TMEM_COLS = tmem_cols_for(DQ_COL + D);
  static_assert(DQ_COL + D <= 512 && SMEM <= 232448, "budget");
};

// TW = false: prototype-wise weights, lse and D per token.  TW = true: token-wise
// weights (Sec. 5.1), lse and D per prototype [B][H][P]: per-row (per-thread)
// values, and columns past the tile's tokens are masked here.
template <int D, bool TW>
__device__ __forceinline__ void bwd_dq_body(const CUtensorMap& tmK, const CUtensorMap& tmV, const Args& a,
                                            const float* __restrict__ dsk, const float* __restrict__ lse,
                                            const float* __restrict__ Dco) {
  using C = DCfg<D>;
  constexpr int ND = C::ND, BLK = C::BLK, HT = C::HT;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (cta_leaves(a.ws, smem_u32(smem), 0xB31u)) return;
  const uint32_t sbase = smem_u32(smem);
  const uint32_t sK = sbase + C::OFF_K, sV = sbase + C::OFF_V, sRaw = sbase + C::OFF_RAW;
  const float2* tokv = reinterpret_cast<const float2*>(Dco);  // prototype-wise: [H][N]
  uint32_t nb = sbase + C::OFF_BAR;
  auto take = [&](int n) {
    const uint32_t r = nb;
    nb += 8u * uint32_t(n);
    return r;
  };
  // s_full, da_full, ds_full, buf_free: one per half
  const uint32_t k_full = take(C::NK), k_empty = take(C::NK), v_full = take(C::NV), v_empty = take(C::NV),
                 i_full = take(C::NI), i_empty = take(C::NI), s_full = take(2), da_full = take(2), ds_full = take(2),
                 buf_free = take(2), col_full = take(2), col_empty = take(2), q_full = take(1), q_empty = take(1),
                 g_full = take(1), g_empty = take(1), dq_full = take(1), dq_empty = take(1), drain = take(2);
  TileInfo* infos = reinterpret_cast<TileInfo*>(smem + C::OFF_INFO);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::OFF_MISC + 4);
  const int64_t tph = reinterpret_cast<const WsHeader*>(a.ws)->tiles_per_head;
  const int64_t total = tph * a.H;
  const int W = gridDim.x, wk = blockIdx.x;
  const int p0 = int(blockIdx.y) * C::PS;
  const int64_t tb = range_begin(total, W, wk), te = range_begin(total, W, wk + 1);
  const int ntiles = __shfl_sync(0xffffffffu, int(te - tb), 0);
  if (threadIdx.x == 0) {
    auto init = [&](uint32_t bar, int n, uint32_t count) {
      for (int k = 0; k < n; ++k) mbar_init(bar + 8u * k, count);
    };
    init(k_full, C::NK, 1);
    init(k_empty, C::NK, TW ? 1 : 2);  // dQ, and the per-token values read
    init(v_full, C::NV, 1);
    init(v_empty, C::NV, 1);
    init(i_full, C::NI, 1);
    init(i_empty, C::NI, 2 + kSoftWarps + (TW ? 0 : 1));
    init(s_full, 2, 1);
    init(da_full, 2, 1);
    init(ds_full, 2, 4);
    init(buf_free, 2, 1);
    init(col_full, 2, 1);
    init(col_empty, 2, kSoftWarps);
    init(q_full, 1, kSoftWarps);
    init(q_empty, 1, 1);
    init(g_full, 1, kSoftWarps);
    init(g_empty, 1, 1);
    init(dq_full, 1, 1);
    init(dq_empty, 1, kSoftWarps);
    init(drain, 2, 1);
    wait_ctl_init(abort_flag, a.ws);
    fence_mbar_init();
  }
  if (warp == 2) tmem_alloc(smem_u32(tmem_slot), C::TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  auto i_slot = [](int li) { return li % C::NI; };
  auto i_par = [](int li) { return uint32_t(li / C::NI) & 1u; };

  if (ntiles > 0 && warp < kSoftWarp0) {
    setmaxnreg_dec<kRegsCtl>();
    bool ok = true;
    auto wt = [&](uint32_t bar, uint32_t par, uint32_t site) {
      return ok = ok && mbar_wait_warp(bar, par, abort_flag, a.ws, site);
    };
    auto info_flags = [&](int li) -> uint32_t {
      wt(i_full + 8u * i_slot(li), i_par(li), 0xD01);
      return ok ? infos[i_slot(li)].flags : 0u;
    };
    if (warp == 0 && lane == 0) {
      // ------------------------------------------------- tile sequence, K, V
      tma_prefetch_desc(&tmK);
      tma_prefetch_desc(&tmV);
      TileWalker w(a, tb, te, T);
      int prev_q = -1, loaded_k = 0, loaded_v = 0;
      for (int li = 0; li < ntiles && ok; ++li) {
        if (li >= C::NI) ok = mbar_wait(i_empty + 8u * i_slot(li), i_par(li) ^ 1u, abort_flag, a.ws, 0xC01);
        if (!ok) break;
        int64_t t0n;
        int nn, hn, qkn;
        w.peek_next(t0n, nn, hn, qkn);
        const bool last = li + 1 >= ntiles || qkn != w.qk;
        TileInfo& o = infos[i_slot(li)];
        o.tok0 = w.tok0;
        o.dq_dst = last ? dq_block_dst(a, wk, W, total, w, p0, D) : nullptr;
        o.h = w.h;
        o.n = w.n;
        o.b = w.b;
        o.flags = (w.qk != prev_q ? kRunFirst : 0u) | (last ? kRunLast : 0u) | (w.seg_first ? kSegFirst : 0u) |
                  (w.seg_last ? kSegLast : 0u);
        prev_q = w.qk;
        mbar_arrive(i_full + 8u * i_slot(li));
        const int ks = li % C::NK, vs = li % C::NV;
        if (li >= C::NK) ok = mbar_wait(k_empty + 8u * ks, uint32_t(li / C::NK - 1) & 1u, abort_flag, a.ws, 0xC02);
        if (!ok) break;
        mbar_arrive_expect_tx(k_full + 8u * ks, C::TILE + (TW ? 0 : C::RAW));
        if (!TW)  // 16-byte aligned: from the even index at or before the tile's first token
          bulk_load(sRaw + ks * C::RAW, tokv + ((int64_t(w.h) * a.N + w.tok0) & ~int64_t(1)), C::RAW, k_full + 8u * ks);
#pragma unroll
        for (int dh = 0; dh < ND; ++dh)
          tma_load_3d(sK + ks * C::TILE + dh * BLK, &tmK, k_full + 8u * ks, 64 * dh, w.h, int(w.tok0));
        loaded_k = li + 1;
        if (li >= C::NV) ok = mbar_wait(v_empty + 8u * vs, uint32_t(li / C::NV - 1) & 1u, abort_flag, a.ws, 0xC03);
        if (!ok) break;
        mbar_arrive_expect_tx(v_full + 8u * vs, C::TILE);
#pragma unroll
        for (int dh = 0; dh < ND; ++dh)
          tma_load_3d(sV + vs * C::TILE + dh * BLK, &tmV, v_full + 8u * vs, 64 * dh, w.h, int(w.tok0));
        loaded_v = li + 1;
        w.next();
      }
      if (!ok) {  // let the copies in flight land before the CTA exits
#pragma unroll 1
        for (int li = (loaded_k > C::NK ? loaded_k - C::NK : 0); li < loaded_k; ++li)
          mbar_wait_bounded(k_full + 8u * (li % C::NK), uint32_t(li / C::NK) & 1u, 200000000ull);
#pragma unroll 1
        for (int li = (loaded_v > C::NV ? loaded_v - C::NV : 0); li < loaded_v; ++li)
          mbar_wait_bounded(v_full + 8u * (li % C::NV), uint32_t(li / C::NV) & 1u, 200000000ull);
      }
    } else if (warp == 1) {
      // ------------------------------------------------------- S and dA issuer
      constexpr uint32_t idPT = idesc_bf16(128, HT, 0, 0);  // [proto x 64 tokens], K = d, A from TMEM
      const uint64_t dKk = sdesc(sK, 16, 1024), dVk = sdesc(sV, 16, 1024);
      auto kstep = [](int k) { return uint32_t((k >> 2) * BLK + (k & 3) * 32); };
      int rc = 0, gc = 0;
      uint32_t fl = info_flags(0);
      for (int li = 0; li < ntiles && ok; ++li) {
        const int ks = li % C::NK, vs = li % C::NV;
        if (fl & kRunFirst) wt(q_full, uint32_t(rc++) & 1u, 0xD02);
        if (fl & kSegFirst) wt(g_full, uint32_t(gc++) & 1u, 0xD05);
        // everything the first half needs, and the next tile's info, in one round trip
        {
          const uint32_t pp = uint32_t(li - 1) & 1u;  // before the first tile: the phase that counts as done
          const int ln = li + 1 < ntiles ? li + 1 : li;
          const BarPhase b[4] = {{k_full + 8u * ks, uint32_t(li / C::NK) & 1u},
                                 {v_full + 8u * vs, uint32_t(li / C::NV) & 1u},
                                 {buf_free, pp},
                                 {i_full + 8u * i_slot(ln), i_par(ln)}};
          ok = ok && mbar_wait_warp_all(b, abort_flag, a.ws, 0xD03);
        }
        if (!ok) break;
        const uint32_t fn = li + 1 < ntiles ? infos[i_slot(li + 1)].flags : 0u;  // used a tile later
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          if (hf == 1) {
            wt(buf_free + 8u, uint32_t(li - 1) & 1u, 0xD04);
            if (!ok) break;
          }
          tc_fence_after();
          const uint32_t col = tmem + uint32_t(hf * C::HALF_COLS);
          if (elect_one()) {
            const uint64_t dK_ = sdesc_add(dKk, uint32_t(ks) * C::TILE + uint32_t(hf) * (HT * 128));
            const uint64_t dV_ = sdesc_add(dVk, uint32_t(vs) * C::TILE + uint32_t(hf) * (HT * 128));
#pragma unroll
            for (int k = 0; k < D / 16; ++k)
              umma_ts(col + C::S_COL, tmem + C::Q_COL + 8 * k, sdesc_add(dK_, kstep(k)), idPT,
                      k > 0 ? 1u : 0u);
            umma_commit(s_full + 8u * hf);
#pragma unroll
            for (int k = 0; k < D / 16; ++k)
              umma_ts(col + C::DA_COL, tmem + C::G_COL + 8 * k, sdesc_add(dV_, kstep(k)), idPT,
                      k > 0 ? 1u : 0u);
            umma_commit(da_full + 8u * hf);
            if (hf == 1) {
              umma_commit(v_empty + 8u * vs);
              if (fl & kRunLast) umma_commit(q_empty);  // last S of this row of Q
              if (fl & kSegLast) umma_commit(g_empty);  // last dA of this segment
              mbar_arrive(i_empty + 8u * i_slot(li));
            }
          }
        }
        fl = fn;
      }
      if (elect_one()) umma_commit(drain);
      mbar_wait_bounded(drain, 0, 200000000ull);
    } else if (warp == 2) {
      // ------------------------------------------------------------ dQ issuer
      constexpr uint32_t idQ = idesc_bf16(128, D, 0, 1);  // [proto x d], K = tokens, A from TMEM
      const uint64_t dKm = sdesc(sK, BLK, 1024);          // MN-major: d blocks 16 KB apart
      int hp = 0;
      uint32_t fl = info_flags(0);
      for (int li = 0; li < ntiles && ok; ++li) {
        const int ks = li % C::NK;
        if ((fl & kRunFirst) && hp > 0) wt(dq_empty, uint32_t(hp - 1) & 1u, 0xD08);
        {
          const int ln = li + 1 < ntiles ? li + 1 : li;
          const BarPhase b[3] = {{k_full + 8u * ks, uint32_t(li / C::NK) & 1u},
                                 {ds_full, uint32_t(li) & 1u},
                                 {i_full + 8u * i_slot(ln), i_par(ln)}};
          ok = ok && mbar_wait_warp_all(b, abort_flag, a.ws, 0xD07);
        }
        if (!ok) break;
        const uint32_t fn = li + 1 < ntiles ? infos[i_slot(li + 1)].flags : 0u;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          if (hf == 1) wt(ds_full + 8u, uint32_t(li) & 1u, 0xD09);
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            const uint64_t dK_ = sdesc_add(dKm, uint32_t(ks) * C::TILE + uint32_t(hf) * (HT * 128));
            const uint32_t ds = tmem + uint32_t(hf * C::HALF_COLS) + C::S_COL;
#pragma unroll
            for (int k = 0; k < HT / 16; ++k)
              umma_ts(tmem + C::DQ_COL, ds + 8 * k, sdesc_add(dK_, 2048u * k), idQ,
                      ((fl & kRunFirst) && hf == 0 && k == 0) ? 0u : 1u);
            umma_commit(buf_free + 8u * hf);
            if (hf == 1) {
              umma_commit(k_empty + 8u * ks);
              if (fl & kRunLast) umma_commit(dq_full);
              mbar_arrive(i_empty + 8u * i_slot(li));
            }
          }
        }
        if (fl & kRunLast) ++hp;
        fl = fn;
      }
      if (elect_one()) umma_commit(drain + 8u);
      mbar_wait_bounded(drain + 8u, 0, 200000000ull);
    } else if (warp == 3 && !TW) {
      // ------------------------------------------------ per-token values
      for (int li = 0; li < ntiles && ok; ++li) {
        const int buf = li & 1, ks = li % C::NK;
        wt(i_full + 8u * i_slot(li), i_par(li), 0xE01);
        wt(k_full + 8u * ks, uint32_t(li / C::NK) & 1u, 0xE03);
        if (!ok) break;
        const TileInfo& o = infos[i_slot(li)];
        const int n = o.n;
        const float2* raw = reinterpret_cast<const float2*>(smem + C::OFF_RAW + ks * C::RAW) +
                            int((int64_t(o.h) * a.N + o.tok0) & 1);
        float2 x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          x[k] = raw[lane + 32 * k];
          if (lane + 32 * k >= n) x[k] = make_float2(INFINITY, 0.f);  // exp2(-inf) = 0 for padding
        }
        if (li >= 2) wt(col_empty + 8u * buf, uint32_t((li >> 1) - 1) & 1u, 0xE02);
        if (!ok) break;
        float* cl = reinterpret_cast<float*>(smem + C::OFF_COL + buf * C::COL);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          cl[lane + 32 * k] = x[k].x;
          cl[T + lane + 32 * k] = x[k].y;
        }
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(col_full + 8u * buf);
          mbar_arrive(k_empty + 8u * ks);  // the raw values go with the K slot
          mbar_arrive(i_empty + 8u * i_slot(li));
        }
      }
    }
  } else if (ntiles > 0) {
    setmaxnreg_inc<kRegsSoft>();
    // ------------------------------------------------ dS of one half, dQ out
    const int hf = (warp - kSoftWarp0) >> 2, q = warp & 3;
    const uint32_t lane_off = uint32_t(32 * q) << 16;
    const uint32_t t_half = tmem + lane_off + uint32_t(hf * C::HALF_COLS);
    const float c2 = a.scale * kLog2e;
    bool ok = true;
    int gc = 0, rc = 0;
    auto wwait = [&](uint32_t bar, uint32_t par, uint32_t site) {
      return mbar_wait_warp(bar, par, abort_flag, a.ws, site);
    };
    // A operands of the products, bf16 pairs: this thread's prototype row, this
    // warpgroup's half of the d columns.  Written once the last product that read
    // the previous one is done.
    auto put_g = [&](int b, int h) -> bool {
      const float4* src = reinterpret_cast<const float4*>(
          dsk + ((int64_t(b) * a.H + h) * a.P + p0 + 32 * q + lane) * D + (D / 2) * hf);
      uint32_t pk[D / 4];
#pragma unroll
      for (int j = 0; j < D / 8; ++j) {
        const float4 x = src[j];
        pk[2 * j] = pack_bf16(x.x, x.y);
        pk[2 * j + 1] = pack_bf16(x.z, x.w);
      }
      if (gc > 0 && !wwait(g_empty, uint32_t(gc - 1) & 1u, 0xF06)) return false;
      tc_fence_after();
#pragma unroll
      for (int k = 0; k < D / 4; k += 16) tmem_st16(tmem + lane_off + C::G_COL + (D / 4) * hf + k, pk + k);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(g_full);
      ++gc;
      return true;
    };
    auto put_q = [&](int b, int h) -> bool {
      const int64_t qk = a.uq ? int64_t(b) * a.H + h : h;
      const uint4* src = reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(a.Q) +
                                                        (qk * a.P + p0 + 32 * q + lane) * D + (D / 2) * hf);
      uint32_t pk[D / 4];
#pragma unroll
      for (int j = 0; j < D / 16; ++j) {
        const uint4 x = src[j];
        pk[4 * j] = x.x;
        pk[4 * j + 1] = x.y;
        pk[4 * j + 2] = x.z;
        pk[4 * j + 3] = x.w;
      }
      if (rc > 0 && !wwait(q_empty, uint32_t(rc - 1) & 1u, 0xF07)) return false;
      tc_fence_after();
#pragma unroll
      for (int k = 0; k < D / 4; k += 16) tmem_st16(tmem + lane_off + C::Q_COL + (D / 4) * hf + k, pk + k);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(q_full);
      ++rc;
      return true;
    };
    ok = wwait(i_full, 0, 0xF01);
    if (ok) ok = put_q(infos[0].b, infos[0].h);
    if (ok) ok = put_g(infos[0].b, infos[0].h);
    float l2r = 0.f, dr = 0.f;  // token-wise: this row's lse (log2 units) and D, per segment
    for (int li = 0; li < ntiles && ok; ++li) {
      const TileInfo& o = infos[i_slot(li)];  // waited for a tile ahead, released below
      if (TW && (o.flags & kSegFirst)) {
        const int64_t r = (int64_t(o.b) * a.H + o.h) * a.P + p0 + 32 * q + lane;
        l2r = lse[r] * kLog2e;
        dr = Dco[r];
      }
      const int left = o.n - HT * hf;  // tokens of this half
      // the values of 4 tokens a load, ahead of the waits that they would prolong
      const float4* cl = reinterpret_cast<const float4*>(smem + C::OFF_COL + (li & 1) * C::COL) + (HT / 4) * hf;
      float4 l4[TW ? 1 : HT / 4];
      if (!TW) {
        ok = wwait(col_full + 8u * (li & 1), uint32_t(li >> 1) & 1u, 0xF02);
        if (!ok) break;
#pragma unroll
        for (int j = 0; j < HT / 4; ++j) l4[TW ? 0 : j] = cl[j];
      }
      ok = wwait(s_full + 8u * hf, uint32_t(li) & 1u, 0xF03);
      if (!ok) break;
      tc_fence_after();
      float sv[HT];
      tmem_ld32(t_half + C::S_COL, sv);
      tmem_ld32(t_half + C::S_COL + 32, sv + 32);
      tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < HT; j += 4) {
        if (TW) {
#pragma unroll
          for (int i = 0; i < 4; ++i) sv[j + i] = j + i < left ? ex2(fmaf(sv[j + i], c2, -l2r)) : 0.f;
        } else {
          const float4 l = l4[TW ? 0 : j / 4];
          sv[j] = ex2(fmaf(sv[j], c2, -l.x));
          sv[j + 1] = ex2(fmaf(sv[j + 1], c2, -l.y));
          sv[j + 2] = ex2(fmaf(sv[j + 2], c2, -l.z));
          sv[j + 3] = ex2(fmaf(sv[j + 3], c2, -l.w));
        }
      }
      float4 d4[TW ? 1 : HT / 4];
      if (!TW) {
#pragma unroll
        for (int j = 0; j < HT / 4; ++j) d4[TW ? 0 : j] = cl[T / 4 + j];
      }
      ok = wwait(da_full + 8u * hf, uint32_t(li) & 1u, 0xF04);
      if (!ok) break;
      tc_fence_after();
      uint32_t pk[HT / 2];
#pragma unroll
      for (int c = 0; c < HT; c += 32) {
        float dv[32];
        tmem_ld32(t_half + C::DA_COL + c, dv);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          const float4 d = TW ? make_float4(dr, dr, dr, dr) : d4[TW ? 0 : (c + j) / 4];
          pk[(c + j) / 2] = pack_bf16(sv[c + j] * (dv[j] - d.x), sv[c + j + 1] * (dv[j + 1] - d.y));
          pk[(c + j) / 2 + 1] = pack_bf16(sv[c + j + 2] * (dv[j + 2] - d.z), sv[c + j + 3] * (dv[j + 3] - d.w));
        }
      }
      if (!TW) {
        __syncwarp();
        if (lane == 0) mbar_arrive(col_empty + 8u * (li & 1));
      }
      tmem_st16(t_half + C::S_COL, pk);
      tmem_st16(t_half + C::S_COL + 16, pk + 16);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(ds_full + 8u * hf);
      }
      const uint32_t fl = o.flags;
      float* const dst = o.dq_dst;
      __syncwarp();
      if (lane == 0) mbar_arrive(i_empty + 8u * i_slot(li));
      if (li + 1 < ntiles) {
        ok = wwait(i_full + 8u * i_slot(li + 1), i_par(li + 1), 0xF05);
        if (!ok) break;
        const TileInfo& x = infos[i_slot(li + 1)];
        if (x.flags & kRunFirst) ok = put_q(x.b, x.h);
        if (ok && (x.flags & kSegFirst)) ok = put_g(x.b, x.h);
        if (!ok) break;
      }
      if (fl & kRunLast) {  // dQ of the run
        ok = wwait(dq_full, uint32_t(rc - 1 - (li + 1 < ntiles ? 1 : 0)) & 1u, 0xF08);
        if (!ok) break;
        tc_fence_after();
        store_sketch_scaled<D, C::PS, C::DQ_COL>(tmem, lane_off, hf, q, lane, dst, a.scale);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(dq_empty);
      }
    }
  }
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem, C::TMEM_COLS);
  }
}

template <int D, int PS>
__global__ void __launch_bounds__(kThreads, 1)
    tc_bwd_dq_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, Args a,
                     const float* __restrict__ dsk, const float* __restrict__ lse, const float* __restrict__ Dco) {
  bwd_dq_body<D, false>(tmK, tmV, a, dsk, lse, Dco);
}

template <int D, int PS>
__global__ void __launch_bounds__(kThreads, 1)
    tc_tw_bwd_dq_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, Args a,
                        const float* __restrict__ dsk, const float* __restrict__ lse_tok,
                        const float* __restrict__ Dtw) {
  bwd_dq_body<D, true>(tmK, tmV, a, dsk, lse_tok, Dtw);
}

template <int D, bool TW>
static cudaError_t launch_dq_t(const Args& a, int W, const float* dsk, const float* lse, const float* Dco,
                               cudaStream_t st) {
  using C = DCfg<D>;
  CUtensorMap tk, tv;
  if (!make_kv_map(&tk, a.K, a.N, a.H, D) || !make_kv_map(&tv, a.V, a.N, a.H, D)) return cudaErrorInvalidValue;
  auto fn = [] {
    if constexpr (TW) return &tc_tw_bwd_dq_kernel<D, C::PS>;
    else return &tc_bwd_dq_kernel<D, C::PS>;
  }();
  const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  const dim3 grid(W, a.P / C::PS);
  fn<<<grid, kThreads, C::SMEM, st>>>(tk, tv, a, dsk, lse, Dco);
  return cudaGetLastError();
}

}  // namespace tcd

cudaError_t launch_tc_bwd_dq(const Args& a, int W, const float* dsk, const float* lse, const float* Dco,
                             cudaStream_t st) {
  if (a.N == 0) return cudaSuccess;
  return a.d == 64 ? tcd::launch_dq_t<64, false>(a, W, dsk, lse, Dco, st)
                   : tcd::launch_dq_t<128, false>(a, W, dsk, lse, Dco, st);
}

cudaError_t launch_tc_tw_bwd_dq(const Args& a, int W, const float* dsk, const float* lse_tok, const float* Dtw,
                                cudaStream_t st) {
  if (a.N == 0) return cudaSuccess;
  return tcd::launch_dq_t<128, true>(a, W, dsk, lse_tok, Dtw, st);
}

}  // namespace sa
