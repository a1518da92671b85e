"""Users without tokens: their rows are cleared whatever the buffer held, wherever they
stand, and by the whole chip however few they are (one user of 64 heads is as many bytes
as 64 users of one).
"""
import numpy as np
import pytest
import torch

from paper_2609_08443_gb300 import binding, workloads as wl

pytestmark = pytest.mark.gpu


def batch(lens, H, P, d, dtype=wl.BF16):
    spec = wl.custom(lens, H=H, P=P, d=d, dtype=dtype, seed=len(lens) + P)
    return spec, wl.host_to_torch(spec, wl.make_host(spec), torch.device("cuda"))


@pytest.mark.parametrize("H,P,d,dt", [(2, 256, 64, wl.BF16), (3, 512, 128, wl.BF16), (2, 7, 12, wl.F32),
                                      (1, 1, 4, wl.F32)], ids=str)
@pytest.mark.parametrize("lens", [[0], [0, 0, 5], [300, 0, 0, 1, 0], [0, 1] * 400, [0] * 1500 + [2000] + [0] * 700],
                         ids=lambda x: f"B{len(x)}")
def test_rows_are_cleared(cuda_lib, lens, H, P, d, dt):
    spec, t = batch(lens, H, P, d, dt)
    B = len(lens)
    empty = torch.tensor([n == 0 for n in lens], device="cuda")
    a = (t["K"], t["V"], t["cu_seqlens"], t["Q"])
    want = binding.sa_sketch_fwd(*a, spec.scale)
    for shift in (0, 1):  # 16-byte stores and single ones
        out = torch.full((B * H * P * d + 1,), float("nan"), device="cuda")[shift:][:B * H * P * d].view(B, H, P, d)
        binding.sa_sketch_fwd(*a, spec.scale, out=out)
        assert not out[empty].any() and torch.equal(out, want)
    sketch, lse = binding.sa_sketch_fwd_tokenwise(*a, spec.scale, want_lse=True)
    assert not sketch[empty].any()
    assert bool((lse[empty] == -np.inf).all()) and bool(torch.isfinite(lse[~empty]).all())


def test_few_users_take_the_whole_chip(cuda_lib):
    P, d = 2048, 128

    def time(B, H):
        _, t = batch([0] * B, H, P, d)
        out = torch.empty(B, H, P, d, device="cuda")
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        for k in range(13):
            if k == 3:
                ev[0].record()
            binding.sa_sketch_fwd(t["K"], t["V"], t["cu_seqlens"], t["Q"], 0.1, out=out)
        ev[1].record()
        torch.cuda.synchronize()
        return ev[0].elapsed_time(ev[1])

    one, many = time(1, 64), time(64, 1)
    assert one <= 3 * many, (one, many)
