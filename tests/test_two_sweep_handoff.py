"""The hand-offs of the two-sweep backward (csrc/sa_tc_bwd2.cu), on the host: the
kernel's roles as they wait and arrive, over mbarriers that know only a phase's
parity, with every copy, product and warp arbitrarily late.  The barrier and the
parity of a chunk and of a streamed Q block are the kernel's own (csrc/sa_handoff.cuh,
compiled here for the host).

A run is wrong if no role can move while work is left (a phase went by unseen), or if
a wait passes before the phase it stands for is complete.
"""
import ctypes
import random
import shutil
import subprocess
from collections import deque

import pytest

from paper_2609_08443_gb300 import build

SOFT = 3  # softmax warps in the model (eight in the kernel)
WRAP = r"""
#include "sa_handoff.cuh"
extern "C" {
int bars(int nch) { return sa::handoff::chunk_bars(nch); }
int bar(int tile, int c, int nch) { return sa::handoff::chunk_bar(tile, c, nch); }
int par(int tile, int c, int nch) { return int(sa::handoff::chunk_parity(tile, c, nch)); }
int q_s(int tile, int c, int nch, int nd) { return int(sa::handoff::q_block_of_S(tile, c, nch, nd)); }
int q_dk(int tile, int c, int last, int nch, int nd) {
  return int(sa::handoff::q_block_of_dK(tile, c, last != 0, nch, nd));
}
int q_bar(int x) { return int(sa::handoff::q_block_bar(unsigned(x))); }
int q_par(int x) { return int(sa::handoff::q_block_parity(unsigned(x))); }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("handoff")
    (d / "w.cpp").write_text(WRAP)
    cc = shutil.which("g++") or shutil.which("c++")
    subprocess.run([cc, "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, str(d / "w.cpp"), "-o", str(d / "w.so")],
                   check=True)
    return ctypes.CDLL(str(d / "w.so"))


class Bar:
    def __init__(self, count):
        self.count, self.left, self.done = count, count, 0

    def arrive(self):
        self.left -= 1
        if self.left == 0:
            self.done, self.left = self.done + 1, self.count

    def passes(self, parity):
        return (self.done & 1) != parity


class Model:
    """One CTA walking `tiles`, a list of (run_first, run_last, seg_first, seg_last)."""

    def __init__(self, rule, P, d, fuse, summed, tiles, rng, late):
        self.r, self.rng, self.late = rule, rng, late
        self.tiles, self.fuse, self.d = tiles, fuse, d
        self.NCH, self.ND = P // 128, d // 64
        self.res = not (d == 128 and P == 512)
        dv = 128 + P // 2
        self.shared = summed or dv + 2 * d + (self.NCH * d if fuse else 0) > 512
        self.NK, self.NV, self.NI = (2 if d == 64 or fuse else 1), (2 if d == 64 else 1), 4
        self.NG = 2 if fuse and d == 64 else 1
        ngb = self.NG if fuse else self.NCH
        mk = lambda n, c: [Bar(c) for _ in range(n)]
        self.k_full, self.k_empty = mk(self.NK, 1), mk(self.NK, 2 if fuse else 1)
        self.v_full, self.v_empty = mk(self.NV, 1), mk(self.NV, 1 + SOFT)
        self.q_full, self.q_empty = mk(1 if self.res else 8, 1), mk(1 if self.res else 2, 2 if self.res else 1)
        self.g_full, self.g_empty = mk(ngb, 1), mk(ngb, 2)
        self.i_full, self.i_empty = mk(self.NI, 1), mk(self.NI, 2 + SOFT + (0 if fuse else 1))
        self.dk_done = mk(self.NCH, 1)
        self.sd_full, self.sd_free, self.dv_full = Bar(1), Bar(SOFT), Bar(1)
        nb = rule.bars(self.NCH)
        self.a_full, self.ds_full = mk(nb, SOFT), mk(nb, SOFT)
        self.acc_free, self.dq_free, self.st_ready = Bar(SOFT), Bar(SOFT), Bar(SOFT)
        self.queues = {}  # copies and products in flight, each queue in its own order

    # ------------------------------------------------------------ primitives
    def post(self, queue, bar):
        self.queues.setdefault(queue, deque()).append(bar)

    @staticmethod
    def w(bar, n):  # wait for completed phase n of a barrier used once per n
        return (bar, n & 1, n + 1)

    def chunk(self, bars, li, c):
        return (bars[self.r.bar(li, c, self.NCH)], self.r.par(li, c, self.NCH), None)

    def q_block(self, x):
        return (self.q_full[self.r.q_bar(x)], self.r.q_par(x), x // 8 + 1)

    # ----------------------------------------------------------------- roles
    def loader(self):
        T, n = self.tiles, len(self.tiles)

        def info(li):
            if li >= self.NI:
                yield [self.w(self.i_empty[li % self.NI], li // self.NI - 1)]
            self.i_full[li % self.NI].arrive()

        runs = 0
        yield from info(0)
        for li in range(n):
            if li + 1 < n:
                yield from info(li + 1)
            ks, ku = li % self.NK, li // self.NK
            if ku:
                yield [self.w(self.k_empty[ks], ku - 1)]
            self.post("K", self.k_full[ks])
            if self.res and T[li][0]:
                if runs:
                    yield [self.w(self.q_empty[0], runs - 1)]
                self.post("Q", self.q_full[0])
                runs += 1
            vs, vu = li % self.NV, li // self.NV
            if vu:
                yield [self.w(self.v_empty[vs], vu - 1)]
            self.post("V", self.v_full[vs])

    def g_wait(self, st, c):
        bit = 0 if self.fuse else c
        if bit in st["seen"]:
            return []
        st["seen"].add(bit)
        b = self.g_full[st["seg"] % self.NG if self.fuse else c]
        return [self.w(b, st["seg"] // self.NG if self.fuse else st["seg"])]

    def g_release(self, st, c, queue):
        self.post(queue, self.g_empty[st["seg"] % self.NG if self.fuse else c])

    def issuer1(self):
        T, n, N = self.tiles, len(self.tiles), self.NCH
        st, q = dict(seg=0, seen=set(), u=0, runs=0), "mma1"

        def sd():
            r = [self.w(self.sd_free, st["u"] - 1)] if st["u"] else []
            st["u"] += 1
            return r

        def S(li, c):
            kf = self.w(self.k_full[li % self.NK], li // self.NK)
            if self.res:
                run = c == 0 and T[li][0]
                yield [kf] + sd() + ([self.w(self.q_full[0], st["runs"])] if run else [])
                st["runs"] += run
            else:
                x = self.r.q_s(li, c, N, self.ND)
                yield [kf] + sd() + [self.q_block(x)]
                for dh in range(self.ND):
                    if dh:
                        yield [self.q_block(x + dh)]
                    self.post(q, self.q_empty[(x + dh) & 1])
            self.post(q, self.sd_full)
            if c == N - 1:
                self.post(q, self.k_empty[li % self.NK])
                if self.res and T[li][1]:
                    self.post(q, self.q_empty[0])

        def dA(li, c):
            yield [self.w(self.v_full[li % self.NV], li // self.NV)] + sd() + self.g_wait(st, c)
            self.post(q, self.sd_full)
            if c == N - 1:
                self.post(q, self.v_empty[li % self.NV])
            if T[li][3] and (not self.fuse or c == N - 1):
                self.g_release(st, c, q)

        yield [self.w(self.i_full[0], 0)]
        yield from S(0, 0)
        for li in range(n):
            if T[li][2]:
                st["seen"] = set()
            for c in range(1, N):
                yield from S(li, c)
            for c in range(N - 1):
                yield from dA(li, c)
            if li + 1 < n:
                yield [self.w(self.i_full[(li + 1) % self.NI], (li + 1) // self.NI)]
            yield from dA(li, N - 1)
            if li + 1 < n:
                yield from S(li + 1, 0)
            st["seg"] += T[li][3]
            self.i_empty[li % self.NI].arrive()

    def issuer2(self):
        T, n, N, q = self.tiles, len(self.tiles), self.NCH, "mma2"
        st, runs, hp = dict(seg=0, seen=set()), 0, 0
        yield [self.w(self.i_full[0], 0)]
        for li in range(n):
            if T[li][2]:
                st["seen"] = set()
            ln = min(li + 1, n - 1)
            kf = [self.w(self.k_full[li % self.NK], li // self.NK)] if self.fuse else []
            yield [self.w(self.i_full[ln % self.NI], ln // self.NI)] + kf
            for c in range(N):
                acc = [self.w(self.acc_free, li - 1)] if self.shared and c == 0 and li else []
                yield [self.chunk(self.a_full, li, c)] + acc + self.g_wait(st, c)
                if c == N - 1:
                    self.post(q, self.dv_full)
                if T[li][3] and (not self.fuse or c == N - 1):
                    self.g_release(st, c, q)
            for c in range(N):
                df = [self.chunk(self.ds_full, li, c)]
                df += [self.w(self.acc_free, li - 1)] if not self.shared and c == 0 and li else []
                if self.res:
                    run = c == 0 and T[li][0]
                    yield (df + ([self.w(self.q_full[0], runs)] if run else []) +
                           ([self.w(self.dq_free, hp - 1)] if self.fuse and run and hp else []))
                    runs += run
                else:
                    x = self.r.q_dk(li, c, int(li + 1 >= n), N, self.ND)
                    yield df + [self.q_block(x)]
                    for dh in range(self.ND):
                        if dh:
                            yield [self.q_block(x + dh)]
                        self.post(q, self.q_empty[(x + dh) & 1])
                self.post(q, self.dk_done[c])
                if c == N - 1:
                    if self.fuse:
                        self.post(q, self.k_empty[li % self.NK])
                    if self.res and T[li][1]:
                        self.post(q, self.q_empty[0])
                    hp += T[li][1]
            st["seg"] += T[li][3]
            self.i_empty[li % self.NI].arrive()

    def converter(self):  # fused: dsketch into shared memory
        g = 0
        for li in range(len(self.tiles)):
            if self.tiles[li][2]:
                if g >= self.NG:
                    yield [self.w(self.g_empty[g % self.NG], g // self.NG - 1)]
                yield []
                self.g_full[g % self.NG].arrive()
                g += 1

    def streamer(self):  # split: chunks of G, blocks of Q
        T, n, N, g, x = self.tiles, len(self.tiles), self.NCH, 0, 0
        order = []  # the chunk of Q each block belongs to, as the loader brings them

        def load_q(c, li, dk):
            nonlocal x
            want = (self.r.q_dk(li, c, int(li + 1 >= n), N, self.ND) if dk else self.r.q_s(li, c, N, self.ND))
            assert x == want, "the issuer's block number is the loader's"
            for _ in range(self.ND):
                if x >= 2:
                    yield [self.w(self.q_empty[x & 1], x // 2 - 1)]
                self.post("Q", self.q_full[self.r.q_bar(x)])
                order.append(c)
                x += 1

        yield [self.w(self.i_full[0], 0)]
        if not self.res:
            yield from load_q(0, 0, False)
        for li in range(n):
            if T[li][2]:
                for c in range(N):
                    if g:
                        yield [self.w(self.g_empty[c], g - 1)]
                    self.post("G", self.g_full[c])
                g += 1
            if not self.res:
                for c in range(1, N):
                    yield from load_q(c, li, False)
                for c in range(N - 1):
                    yield from load_q(c, li, True)
            if li + 1 < n:
                yield [self.w(self.i_full[(li + 1) % self.NI], (li + 1) // self.NI)]
                if not self.res:
                    yield from load_q(0, li + 1, False)
            if not self.res:
                yield from load_q(N - 1, li, True)
            self.i_empty[li % self.NI].arrive()

    def softmax(self):
        T, n, N = self.tiles, len(self.tiles), self.NCH
        fin = 0 if self.shared or N == 1 else 1

        def finish(li, waited):
            if not waited:
                yield [self.w(self.dk_done[N - 1], li)]
            self.acc_free.arrive()
            if self.fuse and T[li][1]:
                self.dq_free.arrive()
            self.i_empty[li % self.NI].arrive()

        yield [self.w(self.i_full[0], 0)]
        for li in range(n):
            u0 = 2 * N * li
            for c in range(N):
                b = [self.w(self.sd_full, u0 + c)]
                if c == 0 and li:
                    b.append(self.w(self.dk_done[0], li - 1))
                if fin == 1 and c == 1 and li:
                    b.append(self.w(self.dk_done[N - 1], li - 1))
                yield b
                self.sd_free.arrive()
                yield []
                self.a_full[self.r.bar(li, c, N)].arrive()
                if c == fin and li:
                    yield from finish(li - 1, fin == 1)
            ln = min(li + 1, n - 1)
            yield [self.w(self.dv_full, li), self.w(self.v_full[li % self.NV], li // self.NV),
                   self.w(self.i_full[ln % self.NI], ln // self.NI)]
            if self.d == 128:
                self.st_ready.arrive()
                self.v_empty[li % self.NV].arrive()
                yield [self.w(self.st_ready, li)]
            else:
                self.v_empty[li % self.NV].arrive()
            for c in range(N):
                yield [self.w(self.sd_full, u0 + N + c)]
                self.sd_free.arrive()
                yield []
                self.ds_full[self.r.bar(li, c, N)].arrive()
        yield from finish(n - 1, False)

    # ------------------------------------------------------------- scheduler
    def run(self):
        roles = {"loader": self.loader(), "issuer1": self.issuer1(), "issuer2": self.issuer2(),
                 "side": self.converter() if self.fuse else self.streamer()}
        roles.update({f"softmax{k}": self.softmax() for k in range(SOFT)})
        # what a role waits for, and how far it has come: None while it has not polled all
        # at once yet, then the index of the barrier it polls in turn
        wait = {name: [[], None] for name in roles}

        def poll(name):
            b, at = wait[name]
            if at is None:
                if not all(x[0].passes(x[1]) for x in b):
                    wait[name][1] = 0
                    return poll(name) or True  # the first round of polls itself is a step
            else:
                if not b[at][0].passes(b[at][1]):
                    return False
                wait[name][1] = at + 1
                if at + 1 < len(b):
                    return True
            for x in b:
                assert x[2] is None or x[0].done >= x[2], f"{name} went past a phase that is not complete"
            try:
                wait[name] = [next(roles[name]), None]
            except StopIteration:
                del roles[name], wait[name]
            return True

        for _ in range(200000):
            if not roles:
                return
            moves = [("role", k) for k in roles] + [("copy", k) for k, v in self.queues.items() if v]
            self.rng.shuffle(moves)
            moves.sort(key=lambda m: m[1] in self.late)  # what is late moves when nothing else can
            for kind, k in moves:
                if kind == "copy":
                    self.queues[k].popleft().arrive()
                    break
                if poll(k):
                    break
            else:
                raise AssertionError(f"no role can move: {sorted(roles)} are left")
        raise AssertionError("no end")


def sequence(rng, n, per_user):
    """n tiles: segments of one to four tiles; a run is a head or, per user, a segment."""
    segs = []
    while sum(segs) < n:
        segs.append(min(rng.choice([1, 1, 2, 4]), n - sum(segs)))
    out = []
    for s, k in enumerate(segs):
        head = per_user or s % 3 == 0
        last = per_user or s % 3 == 2 or s + 1 == len(segs)
        out += [(int(head and i == 0), int(last and i == k - 1), int(i == 0), int(i == k - 1)) for i in range(k)]
    return out


LATE = [(), ("G",), ("Q",), ("K",), ("V",), ("mma1",), ("mma2",), ("issuer1",), ("issuer2",), ("side",), ("loader",),
        ("softmax0",), ("softmax0", "softmax1"), ("G", "Q"), ("G", "issuer2"), ("Q", "issuer2"), ("mma2", "issuer2")]


@pytest.mark.parametrize("late", LATE, ids=lambda x: "+".join(x) or "nothing")
@pytest.mark.parametrize("P,d,fuse", [(128, 64, True), (256, 64, True), (128, 128, True), (256, 128, False),
                                      (512, 64, False), (512, 128, False)], ids=lambda x: str(x))
def test_every_role_moves_on(rule, P, d, fuse, late):
    for seed in range(8):
        rng = random.Random(1000 * P + d + seed)
        Model(rule, P, d, fuse, seed % 2 == 1, sequence(rng, rng.choice([1, 2, 7, 13]), seed % 4 >= 2), rng, late).run()
