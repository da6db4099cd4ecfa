"""Atoms whose best candidates tie (GPU only): the selection in FP64, which a warp
does together, gives what the FP64 form selects one atom per thread, with one or
several lanes of a warp tied and in launches that give a warp few atoms."""
import numpy as np
import pytest

from paper_1603_05143_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [4, 9, 22])
@pytest.mark.parametrize("every", [1, 3, 40])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_tied_candidates(side, every, dtype):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_05143_gb300 import PTM
    # a hexagon, a triangle below it and one above it halfway between the fcc and the
    # hcp position: the triangle's three-fold symmetry makes both covariances equal, so the
    # two templates tie but for the positions' rounding; the other clusters are noisy
    rng = I.rng_for(side)
    ring = lambda a, z, r: [[r * np.cos(a + t), r * np.sin(a + t), z] for t in 2 * np.pi * np.arange(3) / 3]  # noqa: E731
    r, h = 1 / np.sqrt(3), np.sqrt(2 / 3)
    sym = 2.55 * np.array([[0, 0, 0]] + ring(0, 0, 1) + ring(np.pi / 3, 0, 1) + ring(np.pi / 6, -h, r) + ring(0, h, r))
    cells = np.array([[x, y, z] for x in range(side) for y in range(side) for z in range(side)], float) * 12.0 + 6.0
    pos = []
    for i, c in enumerate(cells):
        pos.append(c + (sym if i % every == 0 else sym + rng.normal(0, 0.1, sym.shape)))
    pos = torch.from_numpy(np.ascontiguousarray(np.vstack(pos), dtype)).cuda()
    cell, pbc = np.eye(3) * 12.0 * side, (True, True, True)
    fast, slow = PTM(0), PTM(0, precision="fp64")
    a, b = fast.classify(pos, cell, pbc), slow.classify(pos, cell, pbc)
    torch.cuda.synchronize()
    for k in ("structure", "alloy", "correspondence"):
        assert torch.equal(a[k], b[k]), k
    assert fast.stats()["tie_fp64"] >= (side ** 3 + every - 1) // every
    fast.close()
    slow.close()
