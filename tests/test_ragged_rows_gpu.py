"""Widths that no 16-byte access divides: the update of aligned arrays takes
shifted 16-byte accesses where the rows are long enough for them, that of
arrays which start off a 16-byte boundary 4-byte ones.  The update is
elementwise, so both give the same bits."""
import pytest
import torch

from paper_2607_01455_gb300.ember import Ember

pytestmark = pytest.mark.gpu


def shifted(x, by):
    """A copy of x that starts `by` elements after an aligned address, between canaries."""
    buf = torch.full((x.numel() + by + 64,), 7.0, dtype=x.dtype, device=x.device)
    view = buf[by:by + x.numel()].view_as(x)
    view.copy_(x)
    return buf, view


@pytest.mark.parametrize("V,D", [(5, 1), (9, 2), (300, 3), (700, 5), (305, 31), (306, 33), (1000, 61), (257, 127),
                                 (999, 130), (777, 253),
                                 # both sides of the widths from which shifted accesses are taken
                                 (500, 7), (500, 9), (400, 63), (400, 65), (400, 129), (300, 255), (300, 257), (100, 511), (100, 513),
                                 (60, 1027), (33, 2047), (310, 509), (305, 1021), (306, 1025), (40, 2047),
                                 (33, 2049), (21, 3001)])
@pytest.mark.parametrize("wdtype", ["bf16", "f32"])
@pytest.mark.parametrize("variant", ["full", "col"])
def test_shifted_accesses_match_scalar_ones(cuda_device, V, D, wdtype, variant):
    wt = torch.bfloat16 if wdtype == "bf16" else torch.float32
    g = torch.Generator(device=cuda_device).manual_seed(V * D)
    W0 = (torch.randn(V, D, generator=g, device=cuda_device) * 0.02).to(wt)
    outs = []
    for by in (0, 1, 3):
        emb = Ember(V, D, wdtype=wdtype, variant=variant, device=cuda_device)
        buf, W = shifted(W0, by)
        gg = torch.Generator(device=cuda_device).manual_seed(1)
        for t in (1, 2):
            G0 = torch.randn(V, D, generator=gg, device=cuda_device) * 1e-3
            emb.step_dense(W, shifted(G0, by)[1], 1e-3, t)
        torch.cuda.synchronize()
        assert bool((buf[:by] == 7).all()) and bool((buf[by + V * D:] == 7).all())
        outs.append((W.clone(), emb.state.clone()))
    for W, st in outs[1:]:
        assert torch.equal(W, outs[0][0])
        assert torch.equal(st, outs[0][1])
