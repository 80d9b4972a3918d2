"""Device memory of a block set: the fields, and spectra of no more than every
block of the largest phase and as many sums, in the levels between parents too."""
import numpy as np
import pytest
import torch

from paper_1911_10228_gb300 import flgf as F
from paper_1911_10228_gb300.inputs import box_coords, random_sparse_problem

pytestmark = pytest.mark.gpu


def _octree_blocks(coords):
    """Blocks of the octree over a level's blocks, up to a level of at most 2^3 parents."""
    c = np.asarray(coords)
    n = len(c)
    while np.any(np.ptp(c >> 1, axis=0) > 1):
        c = np.unique(c >> 1, axis=0)
        n += len(c)
    return n


MESHES = {"box": [[box_coords(12)]], "batch": [random_sparse_problem(s, N=8).coords for s in range(4)]}


@pytest.mark.parametrize("mesh", list(MESHES))
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_device_memory_of_a_block_set(mesh, precision):
    problems, N = MESHES[mesh], 16
    ctx = F.Context(N=N, n_interp=6, precision=precision)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    bs = F.BlockSet(ctx, problems, [1.0] * len(problems))
    used = free - torch.cuda.mem_get_info()[0]
    bs.close()
    ctx.close()
    rs = 4 if precision == "fp32" else 8
    levels = max(len(p) for p in problems)
    # a refinement level runs once, and once more from its leaf sources where it has refined blocks
    octree = [sum(_octree_blocks(p[l]) * (1 if l + 1 == len(p) else 2) for p in problems if l < len(p))
              for l in range(levels)]
    blocks = sum(len(c) for p in problems for c in p)
    widest = max(len(c) for p in problems for c in p)
    fields = rs * N ** 3 * (2 * sum(octree) + 3 * blocks + 2 * widest)
    spectra = 2 * 2 * rs * (2 * N) * (2 * N) * (N + 1) * max(octree)
    # 64 MB: launch lists, and allocations rounded up
    assert used <= fields + spectra + (64 << 20), (used, fields, spectra)


def test_passes_match_single_problems():
    """Parents in several passes (the batch's largest phase in FP64): every
    problem as in a block set of its own, whose parents share one pass, to the
    repository's bound for FP64 solves."""
    probs = [random_sparse_problem(s, N=8) for s in range(4)]
    rng = np.random.default_rng(3)
    ctx = F.Context(N=16, n_interp=6, precision="fp64")
    f = [[torch.as_tensor(rng.standard_normal((len(c), 16, 16, 16))).cuda() for c in p.coords] for p in probs]

    def solve(ids):
        bs = F.BlockSet(ctx, [probs[i].coords for i in ids], [probs[i].h0 for i in ids])
        for j, i in enumerate(ids):
            for l, x in enumerate(f[i]):
                bs.load_source(j, l, x)
                bs.load_adjoint(j, l, x)
        bs.solve()
        bs.solve_adjoint()
        out = [[(bs.potential(j, l), bs.gradient(j, l)) for l in range(len(f[i]))] for j, i in enumerate(ids)]
        bs.close()
        return out

    together = solve(range(4))
    for i in range(4):
        for a, b in zip(together[i], solve([i])[0]):
            for x, y in zip(a, b):
                assert float((x - y).abs().max()) < 1e-10 * float(y.abs().max())
    ctx.close()
