"""Neighbour search at the edges of its fast path (GPU only): lists that
overflow, radii that admit too few, searches past the 27 cells, wrapped and
unwrapped atoms, long cells; each atom against the oracle's brute force."""
import numpy as np
import pytest

import oracle as O
from paper_1603_05143_gb300 import inputs as I
from parity import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ptm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_05143_gb300 import PTM
    p = PTM(0)
    yield p
    p.close()


def _frame(kind, rng):
    """Positions and cell of an awkward arrangement."""
    c = I.crystal("fcc", I.A_FCC_CU, (5, 4, 4), sigma=0.08, seed=3, rotation=I.random_rotation(rng))
    L = 4 * I.A_FCC_CU
    if kind == "crystal":
        return c.positions, c.cell
    if kind == "clump":                  # 45 atoms inside one first shell: every radius admits too many or too few
        clump = c.positions[7] + rng.normal(0, 0.25, (45, 3))
        return np.vstack([c.positions, clump]), c.cell
    if kind == "hole":                   # a void: its rim reaches past the 27 cells
        d = np.linalg.norm(c.positions - c.positions.mean(0), axis=1)
        return c.positions[d > 5.5], c.cell
    if kind == "dilute":                 # fewer atoms than neighbours wanted in most cells
        return rng.random((60, 3)) * 3 * L, np.eye(3) * 3 * L
    if kind == "handful":                # fewer than 15 atoms in the whole box
        return rng.random((9, 3)) * L + 1.0, np.eye(3) * 2 * L
    if kind == "long":                   # one long side: large shifts and coordinates
        p = c.positions + np.array([0.0, 0.0, 0.0])
        cell = np.diag([4000.0, L, L])
        q = I.crystal("fcc", I.A_FCC_CU, (6, 4, 4), sigma=0.05, seed=4).positions
        q[:, 0] = np.mod(q[:, 0] - 3 * I.A_FCC_CU, 4000.0)
        return q, cell
    raise ValueError(kind)


@pytest.mark.parametrize("kind", ["crystal", "clump", "hole", "dilute", "handful", "long"])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("pbc", [(True, True, True), (True, False, True), (False, False, False)])
@pytest.mark.parametrize("wrap", ["inside", "unwrapped"])
def test_neighbours_at_the_edges(ptm, kind, dtype, pbc, wrap):
    import torch
    rng = I.rng_for(41)
    pos, cell = _frame(kind, rng)
    if wrap == "unwrapped":              # integer images along the periodic sides
        pos = pos + (rng.integers(-2, 3, (len(pos), 3)) * np.array(pbc)) @ cell
    f = I.Frame(np.ascontiguousarray(pos, dtype), cell, pbc, None, kind)
    for ordering in ("euclidean", "topological"):
        out = ptm.classify(torch.from_numpy(f.positions).cuda(), f.cell, f.pbc, ordering=ordering)
        torch.cuda.synchronize()
        ref = O.Frame(f.positions, f.cell, f.pbc).classify(None, ordering=ordering)
        compare({k: v.cpu().numpy() for k, v in out.items()}, ref)
        assert ptm.stats()["internal"] == 0
