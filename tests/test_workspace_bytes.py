"""What sa_workspace_size asks for, section by section, and that a call runs in exactly
that: callers keep buffers of these sizes."""
import pytest

import harness
from paper_2609_08443_gb300 import binding, build, workloads as wl


def align(x):
    return (x + 255) // 256 * 256


def simt_bytes(B, N, H, P, d, W, bwd):
    b = 256
    b = align(b + 8 * (B + 1))                     # tile prefix
    b = align(b + 4 * W * 2 * P * d)               # pieces of cut segments
    if bwd:
        b = align(b + 4 * W * H * P * d)           # dQ pieces
    b = align(b + 4 * N * H)                       # lse
    if bwd:
        b = align(b + 4 * N * H)                   # D
        if (d == 128 and P > 128) or (d == 64 and P > 256):
            b = align(b + 2 * B * H * P * d)       # bf16 copy of dsketch
    if P >= 1024:
        b = align(b + 8 * N * H * ((P + 511) // 512))
    return align(b + 4 * H * P * d)                # negated prototypes


@pytest.mark.parametrize("bwd", [0, 1])
@pytest.mark.parametrize("dt,P,d", [(0, 64, 64), (0, 200, 36), (1, 256, 64), (1, 128, 128), (1, 512, 128), (1, 1024, 64)],
                         ids=str)
def test_sections(dt, P, d, bwd):
    build.build()
    for B, N, H in ((1, 0, 1), (3, 1001, 2), (64, 100000, 8)):
        got = binding.sa_workspace_size(B, N, H, P, d, dt, bwd)
        # the workers depend on the device: one SM and up where there is none
        assert any(got == simt_bytes(B, N, H, P, d, W, bwd) for W in range(1, 1025)), (B, N, H)


# odd token counts put the tiles of the later heads on every offset modulo 16 bytes
@pytest.mark.gpu
@pytest.mark.parametrize("pass_lse", [True, False])
@pytest.mark.parametrize("P,d,H", [(256, 64, 3), (256, 128, 3), (512, 64, 3), (512, 128, 5), (1024, 64, 3),
                                   (1024, 128, 3), (2048, 128, 2), (1024, 128, 1), (200, 32, 2)], ids=str)
def test_runs_in_exactly_that(cuda_lib, P, d, H, pass_lse):
    import torch

    spec = wl.custom([1, 63, 0, 130, 700, 3], H=H, P=P, d=d, dtype=wl.BF16, seed=P + d + H)
    host = wl.make_host(spec)
    t = wl.host_to_torch(spec, host, torch.device("cuda"))
    a = (t["K"], t["V"], t["cu_seqlens"], t["Q"])
    need = binding.sa_workspace_size(6, 897, H, P, d, binding.SA_BF16, 1)
    guard = torch.full((need + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    lse = binding.sa_sketch_fwd(*a, spec.scale, want_lse=True)[1]
    dK, dV, dQ = binding.sa_sketch_bwd(*a, t["dsketch"], spec.scale, lse=lse if pass_lse else None, ws=guard[:need])
    assert binding.sa_get_device_error(guard) == 0
    assert bool((guard[need:] == 0xA5).all())
    ref = harness.oracle_outputs(spec, host)
    for name, x in (("dK", dK), ("dV", dV), ("dQ", dQ)):
        harness.assert_close(name, wl.torch_as_f64(x), ref[name], harness.TOL[wl.BF16])
