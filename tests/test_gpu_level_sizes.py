"""Sizes and shapes that no other test reaches: refinement steps whose missing
neighbours sort in tiles of 4096 keys (more than 2^18 of them), and the
allocation-free convolution on boxes with parents that are absent, or have
neighbours along every axis and few children."""
import numpy as np
import pytest
import torch

from oracle.conv import hockney
from oracle.flgf import blocks_to_dense, dense_to_blocks
from oracle.meshgen import refine_level as oracle_refine
from paper_1911_10228_gb300 import flgf as F
from paper_1911_10228_gb300.inputs import box_coords

pytestmark = pytest.mark.gpu


# blocks far apart (26 missing neighbours each, all key bits vary), and at a tenth of a box (neighbours shared)
@pytest.mark.parametrize("spread", [1 << 18, 24])
def test_refinement_with_more_than_2_18_missing_neighbours(spread):
    rng = np.random.default_rng(spread)
    coords = np.unique(rng.integers(-spread, spread + 1, size=(13000, 3)), axis=0)
    rng.shuffle(coords)
    f = rng.uniform(0.5, 1.0, (len(coords), 8, 8, 8)).astype(np.float32)
    f[:: len(coords) // 50] = 0.0     # a few blocks are not refined
    ctx = F.Context(N=8, n_interp=4, precision="fp32")
    flags, ch, buf = ctx.refine_level(torch.as_tensor(f), coords, 0.25)
    ctx.close()
    of, och, obuf = oracle_refine(coords, f.astype(np.float64), 0.25)
    level = {tuple(c) for c in coords.tolist()}
    near = [d for d in np.ndindex(3, 3, 3) if d != (1, 1, 1)]
    missing = sum(tuple(np.add(c, d) - 1) not in level for c in coords[of][:200].tolist() for d in near) / 200
    assert missing * of.sum() > 1.05 * (1 << 18)
    assert np.array_equal(flags.cpu().numpy(), of)
    assert np.array_equal(ch.cpu().numpy(), och)
    assert np.array_equal(buf.cpu().numpy(), obuf)


def _random_part(n):
    box = box_coords(4, 4, 4, origin=(-4, 2, 0))
    c = box[np.random.default_rng(n).permutation(64)[:n]]
    return c


STATIC = {
    "one": lambda: np.array([[5, -3, 2]]),
    "box_3x3x3": lambda: box_coords(3, 3, 3),
    "box_2x2x4": lambda: box_coords(2, 2, 4, origin=(0, -2, 2)),
    "odd_column": lambda: box_coords(1, 1, 3, origin=(1, 3, -3)),
    "two_opposite_parents": lambda: np.array([[0, 0, 0], [3, 3, 3]]),
    "absent_parents": lambda: np.array([[0, 1, 0], [1, 0, 3], [2, 2, 1], [3, 3, 0], [2, 3, 1]]),
    "random_5": lambda: _random_part(5),
    "random_13": lambda: _random_part(13),
    "random_32": lambda: _random_part(32),
}


@pytest.mark.parametrize("shape", list(STATIC))
@pytest.mark.parametrize("N", [8, 16])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("fp32", 1e-5)])  # the repository's bounds
def test_static_convolution_of_part_filled_boxes(G, shape, N, precision, tol):
    coords, h = STATIC[shape](), 0.5
    f = np.random.default_rng(len(coords)).standard_normal((len(coords), N, N, N))
    dense, origin = blocks_to_dense(coords, f, N)
    ref = dense_to_blocks(hockney(G, dense, h), origin, coords, N)
    ctx = F.Context(N=N, n_interp=4, precision=precision)
    got = ctx.convolve_static(coords, torch.as_tensor(f, device="cuda"), h=h).double().cpu().numpy()
    ctx.close()
    assert np.max(np.abs(got - ref)) < tol * np.max(np.abs(ref))
