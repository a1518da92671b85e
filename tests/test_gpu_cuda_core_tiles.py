"""The CUDA-core kernels (csrc/sa_simt.cu) at the edges of their 32-token x
64-prototype tiles and of their three width classes (d <= 32, 64, 128), both
dtypes, against the fp64 oracle; the backward with and without the saved lse, and
a dsketch that rules out 16-byte loads.

Tolerance: the suite's 1e-4 (fp32) and 2e-2 (bf16) of max|oracle|.
"""
import pytest
import torch

import harness
from paper_2609_08443_gb300 import binding, workloads as wl

pytestmark = pytest.mark.gpu

LENS = [1, 31, 32, 33, 0, 65, 700]


@pytest.mark.parametrize("P,d,dt,H", [
    (1, 4, wl.F32, 1), (63, 32, wl.F32, 2), (64, 36, wl.F32, 1), (65, 64, wl.F32, 2), (129, 68, wl.F32, 1),
    (300, 128, wl.F32, 2), (2048, 16, wl.F32, 1),
    (2, 8, wl.BF16, 1), (64, 64, wl.BF16, 2), (130, 32, wl.BF16, 1), (200, 96, wl.BF16, 2), (257, 128, wl.BF16, 1),
], ids=lambda x: str(x))
@pytest.mark.parametrize("pass_lse", [True, False])
def test_tile_edges(cuda_lib, P, d, dt, H, pass_lse):
    assert binding.sa_main_kernel_name(P, d, binding.SA_F32 if dt == wl.F32 else binding.SA_BF16,
                                       True).startswith("simt")
    spec = wl.custom(LENS, H=H, P=P, d=d, dtype=dt, seed=P + d)
    harness.check_spec(spec, bwd=True, pass_lse=pass_lse)


def test_per_user_queries(cuda_lib):
    spec = wl.custom(LENS, H=2, P=70, d=40, dtype=wl.F32, seed=8)
    harness.check_spec(spec, bwd=True, per_user_q=True)


def test_dsketch_off_16_bytes(cuda_lib):
    spec = wl.custom(LENS, H=1, P=66, d=20, dtype=wl.F32, seed=3)
    t = wl.host_to_torch(spec, wl.make_host(spec), torch.device("cuda"))
    args = (t["K"], t["V"], t["cu_seqlens"], t["Q"])
    want = binding.sa_sketch_bwd(*args, t["dsketch"], spec.scale)
    g = torch.empty(t["dsketch"].numel() + 1, dtype=torch.float32, device="cuda")[1:].view(t["dsketch"].shape)
    g.copy_(t["dsketch"])
    assert g.data_ptr() % 16 == 4
    for a, b in zip(binding.sa_sketch_bwd(*args, g, spec.scale), want):
        assert torch.equal(a, b)
