"""A solve that the caller captures in a CUDA graph of its own: a replay is no
flgf_solve, so what the reads report must be the replay's (potentials, and the
device error flag)."""
import pytest
import torch

from paper_1911_10228_gb300 import flgf as F
from paper_1911_10228_gb300.inputs import box_coords, refine_mesh, torus

pytestmark = pytest.mark.gpu


def _graph(ctx, fn):
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=ctx.stream):
        fn()
    return g


def _replay(ctx, g):
    with torch.cuda.stream(ctx.stream):
        g.replay()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_flag_of_a_replayed_solve(precision):
    p = refine_mesh(lambda x: torus(x, (0.5, 0.5, 0.5), 0.22, 0.05), box_coords(4), 8, 1.0 / 32, 2, 0.3)
    ctx = F.Context(N=8, n_interp=6, precision=precision)
    bs = F.BlockSet(ctx, [p.coords], [p.h0])
    f = [torch.as_tensor(x).cuda() for x in p.f]
    for l, x in enumerate(f):
        bs.load_source(0, l, x)
    bs.solve()
    ref = bs.potential(0, 1).clone()
    g = _graph(ctx, bs.solve)
    for l, x in enumerate(f):
        bs.load_source(0, l, 2 * x)
    _replay(ctx, g)
    assert torch.equal(bs.potential(0, 1), 2 * ref)   # doubling is exact
    # one coarse-fine entry marked absent: the next replay raises the flag
    bs.set_option(F.OPT_FAULT_HALO, 1)
    _replay(ctx, g)
    with pytest.raises(F.FLGFError) as ei:
        bs.potential(0, 1)
    assert ei.value.code == F.FLGF_EDEVICE
    # and a solve outside the graph its own
    bs.solve()
    with pytest.raises(F.FLGFError):
        bs.potential(0, 0)
    bs.close()
    ctx.close()


def test_flag_of_a_replayed_adjoint():
    p = refine_mesh(lambda x: torus(x, (0.5, 0.5, 0.5), 0.22, 0.05), box_coords(4), 8, 1.0 / 32, 2, 0.3)
    ctx = F.Context(N=8, n_interp=6, precision="fp64")
    bs = F.BlockSet(ctx, [p.coords], [p.h0])
    for l, x in enumerate(p.f):
        bs.load_source(0, l, torch.as_tensor(x).cuda())
        bs.load_adjoint(0, l, torch.as_tensor(x).cuda())
    bs.solve_adjoint()
    bs.gradient(0, 0)
    g = _graph(ctx, bs.solve_adjoint)
    bs.set_option(F.OPT_FAULT_HALO, 1)
    bs.solve()
    with pytest.raises(F.FLGFError):
        bs.potential(0, 1)
    _replay(ctx, g)          # the adjoint's own lists are whole: its flag is clear
    bs.gradient(0, 0)
    bs.close()
    ctx.close()
