"""Sketch rows leave the tensor-core forward in 32-byte stores where the buffer allows
it and in 16-byte ones elsewhere: both give the same bits, for whole segments (written
straight to the output) and for users split between workers (written as partials)."""
import pytest
import torch

from paper_2609_08443_gb300 import binding, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,d", [(128, 64), (256, 64), (512, 128), (1024, 64)])
def test_sketch_on_16_bytes(cuda_lib, P, d):
    spec = wl.custom([300, 0, 1, 128, 40000, 33], H=2, P=P, d=d, dtype=wl.BF16, seed=P)
    t = wl.host_to_torch(spec, wl.make_host(spec), torch.device("cuda"))
    args = (t["K"], t["V"], t["cu_seqlens"], t["Q"], spec.scale)
    want = binding.sa_sketch_fwd(*args)
    want = want[0] if isinstance(want, tuple) else want
    out = torch.empty(want.numel() + 4, device="cuda")[4:].view(want.shape)
    assert out.data_ptr() % 32 == 16
    binding.sa_sketch_fwd(*args, out=out)
    assert torch.equal(out, want)
