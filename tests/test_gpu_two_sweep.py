"""The two-sweep backward (csrc/sa_tc_bwd2.cu): every shape it serves, with shared and
per-user queries (the resident Q and the dQ accumulators change hands at each run),
users of one token to several tiles, one-tile segments in a row (the dsketch buffers
alternate), and outputs on a 16-byte but not 32-byte boundary.

Tolerance: the suite's 2e-2 of max|oracle|; the boundary changes no value.
"""
import pytest
import torch

import harness
from paper_2609_08443_gb300 import binding, workloads as wl

pytestmark = pytest.mark.gpu

LENS = [1, 128, 127, 0, 5, 64, 300, 129, 2, 0, 0, 77, 1500, 256]
SHAPES = [(128, 64, 3), (256, 64, 2), (512, 64, 2), (128, 128, 2), (256, 128, 2), (512, 128, 3)]


@pytest.mark.parametrize("per_user_q", [False, True])
@pytest.mark.parametrize("P,d,H", SHAPES, ids=lambda x: str(x))
def test_shapes(cuda_lib, P, d, H, per_user_q):
    assert binding.sa_main_kernel_name(P, d, binding.SA_BF16, True).startswith("tc_bwd2")
    spec = wl.custom(LENS, H=H, P=P, d=d, dtype=wl.BF16, seed=P + d)
    harness.check_spec(spec, bwd=True, per_user_q=per_user_q)


@pytest.mark.parametrize("P,d,H", SHAPES, ids=lambda x: str(x))
def test_outputs_on_16_bytes(cuda_lib, P, d, H):
    spec = wl.custom([300, 33], H=H, P=P, d=d, dtype=wl.BF16, seed=5)
    t = wl.host_to_torch(spec, wl.make_host(spec), torch.device("cuda"))
    args = (t["K"], t["V"], t["cu_seqlens"], t["Q"], t["dsketch"], spec.scale)
    want = binding.sa_sketch_bwd(*args)
    off = [torch.empty(t["K"].numel() + 8, dtype=torch.bfloat16, device="cuda")[8:].view(t["K"].shape)
           for _ in range(2)]
    got = binding.sa_sketch_bwd(*args, outs=(*off, torch.empty_like(want[2])))
    assert off[0].data_ptr() % 32 == 16
    for g, w in zip(got, want):
        assert torch.equal(g, w)
    with pytest.raises(binding.SketchError):  # rows on no 16-byte boundary are refused
        bad = torch.empty(t["K"].numel() + 1, dtype=torch.bfloat16, device="cuda")[1:].view(t["K"].shape)
        binding.sa_sketch_bwd(*args, outs=(bad, off[1], torch.empty_like(want[2])))
