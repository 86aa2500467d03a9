"""The first kernel of a step may be launched while the work before it on the
stream is still finishing; it waits for that work before it reads anything.
The work before it: a copy, a memset and a kernel of the caller's; the last
kernel of the step before, the one kernel that lets the next start early; work
of another stream.  Eagerly and captured in a graph."""
import pytest
import torch

from paper_2607_01455_gb300.ember import Ember

pytestmark = pytest.mark.gpu

V_SMALL, D_SMALL = 512, 64       # one cluster launch
V_MID, D_MID, N = 20000, 512, 600


def setup(kind, device):
    V, D = (V_SMALL, D_SMALL) if kind == "cluster" else (V_MID, D_MID)
    emb = Ember(V, D, wdtype="f32", variant="row" if kind == "row" else "full", max_sparse_N=6000, device=device)
    g = torch.Generator(device=device).manual_seed(3)
    W = torch.randn(V, D, generator=g, device=device)
    src = torch.randn(6000 if "sparse" in kind else V, D, generator=g, device=device) * 1e-3
    ids = torch.randint(0, V, (6000,), generator=g, device=device)
    return emb, W, src, ids


@pytest.mark.parametrize("kind", ["cluster", "dense", "row", "sparse_small", "sparse"])
@pytest.mark.parametrize("captured", [False, True])
def test_step_waits_for_the_work_before_it(cuda_device, kind, captured):
    emb, W, src, ids = setup(kind, cuda_device)
    n = {"sparse_small": N, "sparse": 6000}.get(kind)
    buf, ibuf = torch.zeros_like(src), torch.zeros_like(ids)

    def work(e, w, t, stream):
        buf.zero_()
        buf.copy_(src)       # a copy of the gradient, then a kernel on it
        buf.mul_(1.0 + t)
        ibuf.copy_(ids)
        if n:
            e.step_sparse(w, ibuf[:n], buf[:n], 1e-3, t, stream=stream)
        else:
            e.step_dense(w, buf, 1e-3, t, stream=stream)

    # the reference: every part waited for
    ref, Wr, _, _ = setup(kind, cuda_device)
    for t in (1, 2, 3):
        work(ref, Wr, t, None)
        torch.cuda.synchronize()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        if captured:
            graphs = []
            for t in (1, 2, 3):
                graphs.append(torch.cuda.CUDAGraph())
                with torch.cuda.graph(graphs[-1], stream=s):
                    work(emb, W, t, s)
            for g in graphs:
                g.replay()
        else:
            for t in (1, 2, 3):
                work(emb, W, t, s)
    torch.cuda.synchronize()
    assert torch.equal(W, Wr)
    assert torch.equal(emb.state, ref.state)


KINDS = ["cluster", "dense", "row", "sparse_early", "sparse_small", "sparse", "mixed"]


def make_steps(kind, device, n=6):
    """A function that runs step t of a sequence on inputs made beforehand."""
    V, D = (V_SMALL, D_SMALL) if kind == "cluster" else (V_MID, D_MID)
    g = torch.Generator(device=device).manual_seed(5)
    ids = [torch.randint(0, V, (6000,), generator=g, device=device) for _ in range(n)]
    Gs = [torch.randn(6000 if "sparse" in kind else V, D, generator=g, device=device) * 1e-3 for _ in range(n)]
    W0 = torch.randn(V, D, generator=g, device=device)
    count = {"sparse_early": 100, "sparse_small": N, "sparse": 6000}.get(kind)

    def fresh():
        emb = Ember(V, D, wdtype="f32", variant="row" if kind == "row" else "full", max_sparse_N=6000, device=device)
        return emb, W0.clone()

    def step(emb, W, t, stream=None):
        k = t - 1
        if kind == "mixed" and t % 2 == 0:  # dense, the dedup alone and sparse batches of every form in turn
            m = (100, 600, 6000)[t // 2 % 3]
            emb.step_sparse(W, ids[k][:m], Gs[k][:m], 1e-3, t, stream=stream)
        elif count:
            emb.step_sparse(W, ids[k][:count], Gs[k][:count], 1e-3, t, stream=stream)
        else:
            emb.step_dense(W, Gs[k], 1e-3, t, stream=stream)

    return fresh, step, n


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("captured", [False, True])
def test_steps_right_after_each_other(cuda_device, kind, captured):
    """Nothing between the steps: the kernels of the next are launched while the
    update of the one before still reads the sums that they write anew."""
    fresh, step, n = make_steps(kind, cuda_device)
    ref, Wr = fresh()
    for t in range(1, n + 1):
        step(ref, Wr, t)
        torch.cuda.synchronize()
    s = torch.cuda.Stream()
    for _ in range(3):
        emb, W = fresh()
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=s):
                    for t in range(1, n + 1):
                        step(emb, W, t, s)
                graph.replay()
            else:
                for t in range(1, n + 1):
                    step(emb, W, t, s)
        torch.cuda.synchronize()
        assert torch.equal(W, Wr) and torch.equal(emb.state, ref.state)


@pytest.mark.parametrize("kind", ["cluster", "dense", "row", "sparse_early", "sparse_small", "sparse"])
@pytest.mark.parametrize("captured", [False, True])
def test_step_waits_for_another_stream(cuda_device, kind, captured):
    """The gradient is made on another stream, by kernels that take a while; the
    step's stream waits for its event, runs the step, and that stream waits
    for the step before it makes the next gradient."""
    emb, W, src, ids = setup(kind.replace("_early", "_small"), cuda_device)
    ref, Wr, _, _ = setup(kind.replace("_early", "_small"), cuda_device)
    n = {"sparse_early": 100, "sparse_small": N, "sparse": 6000}.get(kind)
    buf = torch.empty_like(src)
    scratch = torch.randn(2048, 2048, device=cuda_device)

    def make(t):
        x = scratch
        for _ in range(8):
            x = x @ scratch * 1e-2
        torch.mul(src, 1.0 + t + 0.0 * x[0, 0].nan_to_num(0.0, 0.0, 0.0), out=buf)

    def step(e, w, t, stream=None):
        if n:
            e.step_sparse(w, ids[:n], buf[:n], 1e-3, t, stream=stream)
        else:
            e.step_dense(w, buf, 1e-3, t, stream=stream)

    for t in (1, 2, 3):
        make(t)
        torch.cuda.synchronize()
        step(ref, Wr, t)
        torch.cuda.synchronize()
    s, other = torch.cuda.Stream(), torch.cuda.Stream()

    def run():  # on s, with `other` forked from it and joined again
        for t in (1, 2, 3):
            other.wait_stream(s)
            with torch.cuda.stream(other):
                make(t)
            s.wait_stream(other)
            step(emb, W, t, s)

    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=s):
                run()
            graph.replay()
        else:
            run()
    torch.cuda.synchronize()
    assert torch.equal(W, Wr) and torch.equal(emb.state, ref.state)
