"""The binding's cached workspaces: one per device and stream, held by one call at a time
while it is enqueued, bounded, and no part of a captured graph.

The cache itself is tested on the CPU, with torch's stream handle faked; on the GPU, calls
of other shapes on two streams, in two threads and in a replayed graph give the bits that
the same calls give one after the other."""
import threading

import pytest
import torch

from paper_2609_08443_gb300 import binding, workloads as wl

CPU = torch.device("cpu")


@pytest.fixture
def fake(monkeypatch):
    state = dict(stream=7, capturing=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda index: state["stream"], raising=False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "init", lambda: None)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: state["capturing"])
    monkeypatch.setattr(binding, "_ws_cache", {})
    return state


def test_one_per_stream(fake):
    a = binding.workspace(1000, CPU)
    assert binding.workspace(500, CPU) is a and a.numel() >= 1000
    fake["stream"] = 8
    b = binding.workspace(1000, CPU)
    assert b.data_ptr() != a.data_ptr()
    fake["stream"] = 7
    assert binding.workspace(1000, CPU) is a
    assert binding.workspace(5000, CPU).numel() >= 5000


def test_bounded(fake):
    for s in range(100):
        fake["stream"] = s
        binding.workspace(64, CPU)
    assert len(binding._ws_cache) <= 16


def test_none_kept_of_a_capture(fake):
    a = binding.workspace(1000, CPU)
    fake["capturing"] = True
    b = binding.workspace(1000, CPU)
    assert b.data_ptr() != a.data_ptr() and binding.workspace(1000, CPU).data_ptr() != b.data_ptr()
    fake["capturing"] = False
    assert binding.workspace(1000, CPU) is a


def test_a_call_holds_its_workspace(fake):
    """Another thread's call on the stream waits until this one is enqueued."""
    _, _, lock = binding._workspace(1000, CPU)
    entered = threading.Event()

    def other():
        _, _, mine = binding._workspace(1000, CPU)
        with mine:
            entered.set()

    with lock:
        t = threading.Thread(target=other)
        t.start()
        assert not entered.wait(0.2)
    t.join(5)
    assert entered.is_set()


# ------------------------------------------------------------------- on the GPU
SPECS = [dict(lens=[3000, 0, 129, 40], H=2, P=256, d=64, dtype=wl.BF16, seed=1),
         dict(lens=[700, 5000], H=3, P=512, d=128, dtype=wl.BF16, seed=2),
         dict(lens=[33, 900, 1], H=1, P=200, d=36, dtype=wl.F32, seed=3)]


def step(spec, t):
    a = (t["K"], t["V"], t["cu_seqlens"], t["Q"])
    sketch, lse = binding.sa_sketch_fwd(*a, spec.scale, want_lse=True)
    return [sketch, lse, *binding.sa_sketch_bwd(*a, t["dsketch"], spec.scale, lse=lse)]


def made():
    for s in SPECS:
        spec = wl.custom(s["lens"], H=s["H"], P=s["P"], d=s["d"], dtype=s["dtype"], seed=s["seed"])
        t = wl.host_to_torch(spec, wl.make_host(spec), torch.device("cuda"))
        yield spec, t, step(spec, t)
    torch.cuda.synchronize()


def same(got, want):
    return all(torch.equal(x, y) for x, y in zip(got, want))


@pytest.mark.gpu
def test_two_streams(cuda_lib):
    cases = list(made())
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    out = []
    for i in range(30):
        spec, t, want = cases[i % 3]
        with torch.cuda.stream(streams[i % 2]):
            out.append((step(spec, t), want))
    torch.cuda.synchronize()
    assert all(same(g, w) for g, w in out)


@pytest.mark.gpu
def test_two_threads_on_one_stream(cuda_lib):
    cases = list(made())
    out = [[], []]

    def work(k):
        for i in range(30):
            spec, t, want = cases[(i + k) % 3]
            out[k].append((step(spec, t), want))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert all(len(o) == 30 and all(same(g, w) for g, w in o) for o in out)


@pytest.mark.gpu
def test_graph_beside_eager_calls(cuda_lib):
    """A graph's calls keep their workspace when eager ones outgrow theirs."""
    spec, t, want = next(made())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = step(spec, t)
    for spec2, t2, want2 in list(made())[1:]:
        graph.replay()
        assert same(step(spec2, t2), want2)
        torch.cuda.synchronize()
        assert same(out, want)
