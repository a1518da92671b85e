// Hand-off rules of the two-sweep backward (sa_tc_bwd2.cu): which barrier, in which
// phase, a chunk's weights and a streamed block of Q are announced on.  Plain functions
// without CUDA types, so that the host can check them as well.
#pragma once
#include <cstdint>

#if defined(__CUDACC__)
#define SA_HANDOFF __host__ __device__ constexpr
#else
#define SA_HANDOFF constexpr
#endif

namespace sa {
namespace handoff {

// A_c and dS_c: one barrier per chunk, one phase per tile.  A parity tells one completed
// phase from none, not from two, so what completes the next phase has to lie behind the
// wait for this one, whoever is late.  The next tile's A_c is announced only after dv_full
// of this tile, which the issuer of dV commits past its waits for every A_c; the next
// tile's dS_c only after this tile's last dk_done, which it commits past its waits for
// every dS_c.  (Two barriers in turn, the chunk's number as the phase, are not enough at
// four chunks: nothing but S, K and Q holds the softmax warps in sweep 1, so with G late
// A_1 and A_3 both completed the same barrier before the issuer, still at dV_0, had seen
// the first.)
SA_HANDOFF int chunk_bars(int nch) { return nch; }
SA_HANDOFF int chunk_bar(int, int c, int) { return c; }
SA_HANDOFF uint32_t chunk_parity(int tile, int, int) { return uint32_t(tile) & 1u; }

// Q streamed through two slots: blocks x of 128 prototypes x 64 features, in the order in
// which S and dK consume them: S_0(0); per tile S_1 .., dK_0 .. dK_(last-1), S_0 of the next
// tile, dK_last.  A slot's next load waits for its last reader, so block x + 8 comes after
// x has been read.  Eight barriers in turn: each issuer waits only for its own blocks, at
// most eight apart, so the phase before the one it waits for is always complete.  (dK_0(0)
// alone has no block of its issuer before it: dV_0(0), issued before, waited for A_0(0), which
// needs the block whose barrier it shares.)
SA_HANDOFF uint32_t q_block_of_S(int tile, int c, int nch, int nd) {
  if (c > 0) return uint32_t(nd + tile * 2 * nch * nd + (c - 1) * nd);
  return tile > 0 ? uint32_t(nd + (tile - 1) * 2 * nch * nd + 2 * (nch - 1) * nd) : 0u;
}
SA_HANDOFF uint32_t q_block_of_dK(int tile, int c, bool last_tile, int nch, int nd) {
  const int base = nd + tile * 2 * nch * nd;
  if (c + 1 < nch) return uint32_t(base + (nch - 1 + c) * nd);
  return uint32_t(base + 2 * (nch - 1) * nd + (last_tile ? 0 : nd));
}
SA_HANDOFF uint32_t q_block_bar(uint32_t x) { return x & 7u; }
SA_HANDOFF uint32_t q_block_parity(uint32_t x) { return (x >> 3) & 1u; }

}  // namespace handoff
}  // namespace sa
