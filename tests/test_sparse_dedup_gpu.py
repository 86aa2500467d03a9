"""Edges of the sparse step's dedup, both of its forms (one launch up to 3072
occurrences, a counting sort above): runs as long as a thread orders (128) and
longer, occurrences on both sides of a bitmap window (65536), and tables that
fill one id range, its neighbours and more than one scan tile."""
import pytest
import torch

from paper_2607_01455_gb300 import ember
from paper_2607_01455_gb300.ember import Ember
from parity import Opt
from test_sparse_gpu import check_dedup, gated_sparse_step

pytestmark = pytest.mark.gpu


def ids_of(V, counts, N, device, seed):
    """N shuffled ids: exactly counts[i] times id i * (V - 1) / len, the rest
    uniform over the other ids."""
    g = torch.Generator(device=device).manual_seed(seed)
    k = len(counts)
    at = [i * (V - 1) // max(1, k - 1) for i in range(k)]
    parts = [torch.full((c,), i, device=device, dtype=torch.int64) for i, c in zip(at, counts)]
    others = torch.ones(V, dtype=torch.bool, device=device)
    others[at] = False
    others = others.nonzero().flatten()
    if N > sum(counts):
        parts.append(others[torch.randint(0, others.numel(), (N - sum(counts),), generator=g, device=device)])
    ids = torch.cat(parts)
    return ids[torch.randperm(N, generator=g, device=device)]


@pytest.mark.parametrize("V,N,counts", [
    (300, 1100, (127, 128, 129)), (256, 129, (129,)), (257, 600, (300, 130)), (77824, 3000, (130, 1, 2)),
    (77825, 5000, (1000, 1000, 1000)), (400000, 2000, (129, 500)),
    (1000, 65536, (65536,)), (1000, 65537, (65537,)), (50000, 270000, (140000, 300, 90000)),
    # either side of the line between the two forms, and of the longest run a
    # thread of the counting form orders
    (1000, 3072, (127, 128, 129)), (1000, 3073, (127, 128, 129)), (70000, 3500, (129,)), (70000, 3500, (128,)),
    (9000, 9000, (128, 129) * 20), (60000, 140000, (129, 128, 127, 70000)),
])
@pytest.mark.parametrize("idtype", [torch.int64, torch.int32])
def test_dedup_edges(cuda_device, V, N, counts, idtype):
    D = 8
    emb = Ember(V, D, wdtype="bf16", max_sparse_N=N, device=cuda_device)
    ids = ids_of(V, counts, N, cuda_device, V + N).to(idtype)
    check_dedup(emb, ids)
    W = torch.zeros(V, D, device=cuda_device, dtype=torch.bfloat16)
    for t in (1, 2):
        rows = torch.randn(N, D, device=cuda_device, generator=torch.Generator(device=cuda_device).manual_seed(t)) * 1e-4
        gated_sparse_step(emb, W, ids, rows, 1e-3, t, Opt())


@pytest.mark.parametrize("V,N,counts", [
    (5000, 900, (127, 128, 129)), (5000, 3072, (5, 300)), (5000, 3073, (5, 300)), (70000, 9000, (128, 129) * 20),
    (5000, 40000, (127, 128, 129, 20000)), (5000, 140000, (128, 129, 70000)), (3, 5000, (1700, 1700, 1600)),
])
def test_runs_are_summed_in_increasing_occurrence(cuda_device, V, N, counts):
    """The bits of a batch are those of the same batch sorted by id beforehand
    (stably): every run is added in increasing occurrence.  The values span
    eight decades, so that another order shows: of 64 columns, swapping two of
    2, 3, 5 or 129 occurrences changes 1, 8, 7 or 20 compensated sums."""
    D = 64
    ids = ids_of(V, counts, N, cuda_device, N)
    g = torch.Generator(device=cuda_device).manual_seed(N)
    rows = torch.randn(N, D, generator=g, device=cuda_device) * 1e-4
    rows *= 10 ** (torch.rand(N, D, generator=g, device=cuda_device) * 8 - 4)
    order = torch.sort(ids, stable=True).indices
    outs = []
    for i, x in ((ids, rows), (ids[order], rows[order].contiguous())):
        emb = Ember(V, D, wdtype="f32", max_sparse_N=N, device=cuda_device)
        W = torch.zeros(V, D, device=cuda_device)
        for t in (1, 2):
            emb.step_sparse(W, i, x, 1e-3, t)
        outs.append((W, emb.state))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])


def test_order_within_runs_is_deterministic(cuda_device):
    """Occurrences arrive in any order; the sums are those of increasing
    occurrence, so repeated steps give the same bits."""
    V, D, N = 5000, 64, 200000
    ids = ids_of(V, (120000, 400, 129, 128), N, cuda_device, 1)
    rows = torch.randn(N, D, device=cuda_device) * 1e-4
    outs = []
    for _ in range(4):
        emb = Ember(V, D, wdtype="f32", max_sparse_N=N, device=cuda_device)
        W = torch.zeros(V, D, device=cuda_device)
        emb.step_sparse(W, ids, rows, 1e-3, 1)
        outs.append((W, emb.state))
    for W, st in outs[1:]:
        assert torch.equal(W.view(torch.int32), outs[0][0].view(torch.int32))
        assert torch.equal(st.view(torch.int32), outs[0][1].view(torch.int32))


@pytest.mark.parametrize("lead,length", [(0, 5000), (17, 4095), (32, 4096), (5, 70001), (65530, 9000)])
def test_stretches_of_one_id(cuda_device, lead, length):
    """Stretches of one id (a padded batch): whole words of the bitmap, partial
    ones at both ends, one window and several, other ids of the run around."""
    V, D = 3000, 64
    g = torch.Generator(device=cuda_device).manual_seed(length)
    noise = torch.randint(0, V, (lead + 3000,), generator=g, device=cuda_device)
    pad = torch.full((length,), 5, device=cuda_device)
    mixed = torch.where(torch.rand(2000, generator=g, device=cuda_device) < 0.9, 5, 6)
    ids = torch.cat([noise[:lead], pad, noise[lead:], mixed, pad])
    N = ids.numel()
    emb = Ember(V, D, wdtype="f32", max_sparse_N=N, device=cuda_device)
    W = torch.randn(V, D, generator=g, device=cuda_device)
    rows = torch.rand(N, D, generator=g, device=cuda_device) * 1e-4
    gated_sparse_step(emb, W, ids, rows, 1e-3, 1, Opt())
    # in increasing occurrence: the same bits as the batch sorted by id beforehand
    order = torch.sort(ids, stable=True).indices
    ref = Ember(V, D, wdtype="f32", max_sparse_N=N, device=cuda_device)
    emb.state.zero_()
    W1, W2 = W.clone(), W.clone()
    emb.step_sparse(W1, ids, rows, 1e-3, 1)
    ref.step_sparse(W2, ids[order], rows[order].contiguous(), 1e-3, 1)
    assert torch.equal(W1, W2) and torch.equal(emb.state, ref.state)


@pytest.mark.parametrize("V", [311296, 311297, 304 * 8192, 304 * 8192 + 5, 5000001, (1 << 23) + 3])
@pytest.mark.parametrize("N", [9, 3500])
def test_tall_tables(cuda_device, V, N):
    """Ranges of one tile, of one and a bit, of a whole batch of tiles, of more;
    mostly empty ones, ids in the first and last rows; r on a 16-byte boundary
    and off it give the same bits, and the dedup clears its map each time."""
    D = 4
    g = torch.Generator(device=cuda_device).manual_seed(V + N)
    ids = torch.randint(0, V, (N,), generator=g, device=cuda_device)
    ids[:6] = torch.tensor([0, V - 1, V - 1, 1024, 8191, 8192], device=cuda_device)
    ids[N // 2:] = ids[N // 2:] % 3000 + V // 2
    emb = Ember(V, D, wdtype="f32", max_sparse_N=N, device=cuda_device)
    check_dedup(emb, ids)
    check_dedup(emb, ids.flip(0))
    W = torch.randn(V, D, generator=g, device=cuda_device)
    W0 = W.clone()
    emb.state.copy_(torch.rand(V + D, generator=g, device=cuda_device) * 1e-6)
    st0 = emb.state.clone()
    rows = torch.randn(N, D, generator=g, device=cuda_device) * 1e-3
    gated_sparse_step(emb, W, ids, rows, 1e-3, 3, Opt())
    buf = torch.empty(V + D + 3, device=cuda_device)
    for off in (1, 2, 3):
        st = buf[off:off + V + D]
        st.copy_(st0)
        W1 = W0.clone()
        ember.ember_step_sparse(emb.handle, W1, ids, ember.EMBER_I64, N, rows, st, 1e-3, 3)
        assert torch.equal(st, emb.state) and torch.equal(W1, W)
