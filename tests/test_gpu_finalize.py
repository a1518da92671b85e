"""Reassembly of segments cut across workers (csrc/sa_finalize.cu) against the
fp64 oracle: short chains of pieces (one thread per column), long ones (split
over a block's warps), chains with empty workers between them, a width that
fills no whole block, and an output that rules out 16-byte accesses.

Tolerance: the suite's 1e-4 (fp32) and 2e-2 (bf16) of max|oracle|.
"""
import pytest
import torch

import harness
from paper_2609_08443_gb300 import binding, workloads as wl

pytestmark = pytest.mark.gpu

# (lengths, H, P, d, dtype): the tiles of one user over 152 or more workers leave
# from one piece per segment to more than a hundred
CASES = [
    ([4096], 1, 64, 64, wl.F32),            # 128 pieces
    ([160, 33], 2, 5, 12, wl.F32),          # more workers than tiles, 60 floats per row block
    ([900, 0, 5000, 1], 2, 200, 36, wl.F32),
    ([1531], 8, 256, 64, wl.BF16),          # 19 pieces per segment
    ([40000, 300], 2, 128, 64, wl.BF16),    # 76 pieces
    ([3000] * 24, 2, 256, 64, wl.BF16),     # two or three pieces
    ([2000, 0, 700], 2, 512, 128, wl.BF16),
]


@pytest.mark.parametrize("lens,H,P,d,dt", CASES, ids=lambda x: str(x).replace(" ", "")[:20])
def test_cut_segments(cuda_lib, lens, H, P, d, dt):
    spec = wl.custom(lens, H=H, P=P, d=d, dtype=dt, seed=P + d + len(lens))
    harness.check_spec(spec, bwd=True)


def test_cut_segments_per_user_queries(cuda_lib):
    spec = wl.custom([6000, 0, 129], H=2, P=256, d=64, dtype=wl.BF16, seed=9)
    harness.check_spec(spec, bwd=True, per_user_q=True)


def test_output_off_16_bytes(cuda_lib):
    spec = wl.custom([3000, 17], H=1, P=40, d=16, dtype=wl.F32, seed=4)
    t = wl.host_to_torch(spec, wl.make_host(spec), torch.device("cuda"))
    want = binding.sa_sketch_fwd(t["K"], t["V"], t["cu_seqlens"], t["Q"], spec.scale)
    flat = torch.empty(want.numel() + 1, dtype=torch.float32, device="cuda")[1:]
    got = binding.sa_sketch_fwd(t["K"], t["V"], t["cu_seqlens"], t["Q"], spec.scale, out=flat.view(want.shape))
    assert got.data_ptr() % 16 == 4
    assert torch.equal(got, want)
