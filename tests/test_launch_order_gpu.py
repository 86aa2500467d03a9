"""The first kernel of a step may be launched while the work before it on the
stream is still finishing; it waits for that work before it reads anything.
Here a copy, a memset and a kernel of the caller's come right before the step,
eagerly and captured in a graph."""
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
