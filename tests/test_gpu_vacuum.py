"""A cluster in a box of vacuum (GPU only): the cell list is sized by the box, so that a few
cells hold everything.  Each of the atoms taken against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1603_05143_gb300 import inputs as I
from parity import compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [40, 700, 1500, 2500])
@pytest.mark.parametrize("vacuum", [3, 10])                # box over diameter
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("pbc", [(False, False, False), (True, True, True)])
@pytest.mark.parametrize("ordering", ["euclidean", "topological"])
def test_cluster_in_vacuum(n, vacuum, dtype, pbc, ordering):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_05143_gb300 import PTM
    f = I.crystal("fcc", I.A_FCC_CU, 12, sigma=0.1, seed=n, rotation=I.random_rotation(I.rng_for(n)), wrap=False)
    pos = f.positions - f.positions.mean(0)
    pos = pos[np.argsort((pos ** 2).sum(1))[:n]]
    side = 2 * vacuum * np.sqrt((pos ** 2).sum(1).max())
    # around a corner of a periodic box (in unwrapped coordinates), or in its middle
    pos = np.ascontiguousarray(pos + side * (0.0 if pbc[0] else 0.5), dtype)
    ptm = PTM(0)
    out = ptm.classify(torch.from_numpy(pos).cuda(), np.eye(3) * side, pbc, ordering=ordering)
    torch.cuda.synchronize()
    assert ptm.stats()["internal"] == 0
    atoms = np.arange(0, n, max(1, n // 300))
    ref = O.Frame(pos, np.eye(3) * side, pbc).classify(atoms, ordering=ordering)
    compare({k: v.cpu().numpy() for k, v in out.items()}, ref, atoms)
    ptm.close()


@pytest.mark.parametrize("n,vacuum", [(8000, 4), (8000, 8), (24576, 10), (26000, 10), (60000, 9)])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("ordering", ["euclidean", "topological"])
def test_crowded_cells(n, vacuum, dtype, ordering):
    """The sizes where the search of such a frame changes hands, unwrapped at a corner: against
    the same atoms in a box that fits them, whose cells are ordinary."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_05143_gb300 import PTM
    f = I.crystal("fcc", I.A_FCC_CU, 32, sigma=0.1, seed=n, rotation=I.random_rotation(I.rng_for(n)), wrap=False)
    pos = f.positions - f.positions.mean(0)
    pos = np.ascontiguousarray(pos[np.argsort((pos ** 2).sum(1))[:n]], dtype)
    diameter = 2 * np.sqrt((pos.astype(np.float64) ** 2).sum(1).max())
    ptm = PTM(0)
    dev = torch.from_numpy(pos).cuda()
    wide = ptm.classify(dev, np.eye(3) * diameter * vacuum, (True, True, True), ordering=ordering)
    torch.cuda.synchronize()
    assert ptm.stats()["internal"] == 0 and ptm.stats()["knn_fail"] == 0
    near = ptm.classify(dev, np.eye(3) * diameter * 1.5, (True, True, True), ordering=ordering)
    torch.cuda.synchronize()
    assert ptm.stats()["knn_fail"] == 0
    for k in wide:
        assert torch.equal(wide[k], near[k]), k
    ptm.close()
