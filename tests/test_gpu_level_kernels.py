"""The whole-level kernels at the sizes and alignments where they can go wrong:
the 7-point Laplacian against the oracle (both block sides and precisions, a
field at an unaligned address, missing neighbours), and the refinement step on
coordinates whose keys vary in all 63 bits, on one to several tiles of the radix
sort, and with a block given twice."""
import numpy as np
import pytest
import torch

from oracle.meshgen import refine_level as oracle_refine
from oracle.multires import Level, laplacian_on_level
from paper_1911_10228_gb300 import flgf as F
from paper_1911_10228_gb300.inputs import box_coords

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [8, 16])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("offset", [0, 1])
def test_laplacian(N, precision, offset):
    ctx = F.Context(N=N, n_interp=4, precision=precision)
    rng = np.random.default_rng(N)
    allc = box_coords(4, 3, 5, origin=(-2, 0, 1))
    coords = allc[rng.random(len(allc)) < 0.7]
    bs = F.BlockSet(ctx, [[coords]], [0.25])
    n = len(coords) * N ** 3
    u = torch.empty(n + offset, dtype=ctx.dtype, device="cuda")[offset:].view(len(coords), N, N, N)
    u.copy_(torch.as_tensor(rng.standard_normal(u.shape)))
    got = bs.laplacian(0, 0, u).double().cpu().numpy()
    ref, mask = laplacian_on_level(Level(coords, N), u.double().cpu().numpy(), 0.25)
    # a sum of 7 terms of up to 6 |u| / h^2, each rounded: 12 units of round-off of 12 max|u| / h^2
    eps = 2.0 ** (-53 if precision == "fp64" else -24)
    assert np.max(np.abs(got - ref)) < 12 * eps * 12 * float(u.abs().max()) * 16
    assert np.all(got[~mask] == 0.0)
    bs.close()
    ctx.close()


@pytest.mark.parametrize("n,spread", [(2, 1), (33, 1 << 18), (4096, 12), (4097, 400), (9000, 1 << 18)])
def test_refinement_step(n, spread):
    ctx = F.Context(N=8, n_interp=4, precision="fp32")
    rng = np.random.default_rng(n)
    coords = np.unique(rng.integers(-spread, spread + 1, size=(n, 3)), axis=0)
    rng.shuffle(coords)
    f = rng.standard_normal((len(coords), 8, 8, 8)).astype(np.float32) * rng.uniform(0, 2, (len(coords), 1, 1, 1)) ** 3
    f = f.astype(np.float32)
    flags, ch, buf = ctx.refine_level(torch.as_tensor(f), coords, 0.3)
    of, och, obuf = oracle_refine(coords, f.astype(np.float64), 0.3)
    assert np.array_equal(flags.cpu().numpy(), of)
    assert np.array_equal(ch.cpu().numpy(), och)
    assert np.array_equal(buf.cpu().numpy(), obuf)
    # the first block once more: the lists hold every coordinate once
    f2 = np.concatenate([f, f[:1]])
    _, ch2, buf2 = ctx.refine_level(torch.as_tensor(f2), np.concatenate([coords, coords[:1]]), 0.3)
    assert torch.equal(ch2, ch) and torch.equal(buf2, buf)
    ctx.close()
