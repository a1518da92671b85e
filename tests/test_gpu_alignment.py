"""Buffers off the boundaries that the tensor-core kernels need: refused with
SA_ERR_INVALID_ARG before anything is enqueued, on every entry point; outputs that
need none give the same bits wherever they start."""
import pytest
import torch

from paper_2609_08443_gb300 import binding, workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(256, 64), (128, 128), (512, 64), (512, 128), (1024, 128)]


def inputs(P, d, per_user_q=False, lens=(300, 33)):
    spec = wl.custom(list(lens), H=2, P=P, d=d, dtype=wl.BF16, seed=5)
    return spec, wl.host_to_torch(spec, wl.make_host(spec, per_user_q=per_user_q), torch.device("cuda"))


def off(t):
    """A buffer like t one element past a 16-byte boundary, with its values."""
    x = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)[1:].view(t.shape)
    return x.copy_(t)


def refused(call):
    n = binding.sa_launch_count()
    with pytest.raises(binding.SketchError) as e:
        call()
    assert e.value.status == 1
    assert binding.sa_launch_count() == n


def raw(entry, *args):
    binding._check(entry(*(a.data_ptr() if isinstance(a, torch.Tensor) else a for a in args)), "entry")


def stream():
    return torch.cuda.current_stream().cuda_stream


@pytest.mark.parametrize("which", [0, 1], ids=["dK", "dV"])
@pytest.mark.parametrize("P,d", SHAPES, ids=lambda x: str(x))
def test_gradient_rows(cuda_lib, P, d, which):
    spec, t = inputs(P, d)
    outs = [torch.empty_like(t["K"]), torch.empty_like(t["K"]), torch.empty(t["Q"].shape, device="cuda")]
    outs[which] = off(outs[which])
    a = (t["K"], t["V"], t["cu_seqlens"], t["Q"], t["dsketch"], spec.scale)
    refused(lambda: binding.sa_sketch_bwd(*a, outs=outs))


@pytest.mark.parametrize("P,d", SHAPES, ids=lambda x: str(x))
def test_dx(cuda_lib, P, d):
    spec, t = inputs(P, d)
    lib, H = binding.load(), 2
    Wk = torch.zeros(H, d, d, dtype=torch.bfloat16, device="cuda")
    N, B = t["K"].shape[0], 2
    ws = torch.empty(lib.sa_workspace_size_x(B, N, H, P, d, 1, 1), dtype=torch.uint8, device="cuda")
    dQ, dWk = torch.empty(H, P, d, device="cuda"), torch.empty(H, d, d, device="cuda")
    refused(lambda: raw(lib.sa_sketch_bwd_x, t["K"], t["cu_seqlens"], B, N, t["Q"], Wk, H, P, d, spec.scale, 1,
                        t["dsketch"], None, off(t["K"]), dQ, dWk, ws, ws.numel(), stream()))


@pytest.mark.parametrize("which", [0, 1], ids=["dK", "dV"])
def test_tokenwise_gradient_rows(cuda_lib, which):
    P, d, H = 512, 128, 2
    spec, t = inputs(P, d)
    lib, N, B = binding.load(), t["K"].shape[0], 2
    ws = torch.empty(lib.sa_workspace_size_tokenwise(B, N, H, P, d, 1, 1), dtype=torch.uint8, device="cuda")
    outs = [torch.empty_like(t["K"]), torch.empty_like(t["K"])]
    outs[which] = off(outs[which])
    dQ = torch.empty(H, P, d, device="cuda")
    refused(lambda: raw(lib.sa_sketch_bwd_tokenwise, t["K"], t["V"], t["cu_seqlens"], B, N, t["Q"], H, P, d,
                        spec.scale, 1, None, None, t["dsketch"], *outs, dQ, ws, ws.numel(), stream()))


@pytest.mark.parametrize("P,d", SHAPES, ids=lambda x: str(x))
def test_dsketch(cuda_lib, P, d):
    spec, t = inputs(P, d)
    a = (t["K"], t["V"], t["cu_seqlens"], t["Q"])
    refused(lambda: binding.sa_sketch_bwd(*a, off(t["dsketch"]), spec.scale))
    Wk = torch.zeros(2, d, d, dtype=torch.bfloat16, device="cuda")
    refused(lambda: binding.sa_sketch_bwd_x(t["K"], t["cu_seqlens"], t["Q"], Wk, off(t["dsketch"]), spec.scale))


@pytest.mark.parametrize("per_user_q", [False, True])
@pytest.mark.parametrize("P,d", SHAPES, ids=lambda x: str(x))
def test_dq_may_start_anywhere(cuda_lib, P, d, per_user_q):
    spec, t = inputs(P, d, per_user_q=per_user_q)
    a = (t["K"], t["V"], t["cu_seqlens"], t["Q"], t["dsketch"], spec.scale)
    want = binding.sa_sketch_bwd(*a)
    got = binding.sa_sketch_bwd(*a, outs=(torch.empty_like(t["K"]), torch.empty_like(t["K"]), off(want[2])))
    assert all(torch.equal(x, y) for x, y in zip(got, want))


# users of one tile, which one worker writes whole, and one cut across workers
LENS = [60] * 300 + [3000]


@pytest.mark.parametrize("P,d", [(128, 64), (256, 64), (512, 64), (1024, 64), (128, 128), (512, 128)],
                         ids=lambda x: str(x))
def test_sketch_may_start_anywhere(cuda_lib, P, d):
    spec, t = inputs(P, d, lens=LENS)
    a = (t["K"], t["V"], t["cu_seqlens"], t["Q"], spec.scale)
    want = binding.sa_sketch_fwd(*a)
    assert torch.equal(binding.sa_sketch_fwd(*a, out=off(want)), want)


@pytest.mark.parametrize("P,d", [(256, 64), (384, 64), (512, 128)], ids=lambda x: str(x))
def test_tokenwise_sketch_may_start_anywhere(cuda_lib, P, d):
    spec, t = inputs(P, d, lens=LENS)
    lib, N, B, H = binding.load(), t["K"].shape[0], len(LENS), 2
    want = binding.sa_sketch_fwd_tokenwise(t["K"], t["V"], t["cu_seqlens"], t["Q"], spec.scale)
    ws = torch.empty(lib.sa_workspace_size_tokenwise(B, N, H, P, d, 1, 0), dtype=torch.uint8, device="cuda")
    sketch = off(want)
    raw(lib.sa_sketch_fwd_tokenwise, t["K"], t["V"], t["cu_seqlens"], B, N, t["Q"], H, P, d, spec.scale, 1, sketch,
        None, ws, ws.numel(), stream())
    assert torch.equal(sketch, want)


@pytest.mark.parametrize("P,d", [(256, 64), (512, 128)], ids=lambda x: str(x))
def test_gradient_of_a_cat(cuda_lib, P, d):
    """autograd hands a sketch inside a cat a view of the cat's gradient."""
    spec, t = inputs(P, d)
    grads = []
    for pad in (0, 1):
        leaves = [t[k].clone().requires_grad_(True) for k in ("K", "V", "Q")]
        s = binding.sa_sketch(leaves[0], leaves[1], t["cu_seqlens"], leaves[2], spec.scale)
        row = torch.cat([torch.zeros(pad, device="cuda"), s.flatten()])
        row.backward(torch.cat([torch.zeros(pad, device="cuda"), t["dsketch"].flatten()]))
        grads.append([x.grad for x in leaves])
    assert all(torch.equal(x, y) for x, y in zip(*grads))
