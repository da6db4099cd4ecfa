"""The thread-per-atom neighbour search at its edges (GPU only).  A single frame of up to
1,536 atoms is searched by a warp per atom; a batch takes the thread-per-atom kernel at
every size, so the arrangements and near-ties that this kernel has to decide run here as
batches of one frame, each atom against the oracle's brute force."""
import numpy as np
import pytest

import oracle as O
from paper_1603_05143_gb300 import inputs as I
from parity import compare
from test_gpu_knn import _frame

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


def _check(ptm, pos, cell, pbc, ordering):
    import torch
    b = ptm.batch([{"positions": torch.from_numpy(pos).cuda(), "cell": cell, "pbc": pbc, "ordering": ordering}])
    b.run()
    torch.cuda.synchronize()
    ref = O.Frame(pos, cell, pbc).classify(None, ordering=ordering)
    compare({k: v.cpu().numpy() for k, v in b.outputs[0].items()}, ref)
    s = b.stats()
    assert s["internal"] == 0
    b.close()
    return s


@pytest.mark.parametrize("kind", ["crystal", "clump", "hole", "dilute", "handful", "long"])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("pbc", [(True, True, True), (True, False, True), (False, False, False)])
@pytest.mark.parametrize("wrap", ["inside", "unwrapped"])
def test_neighbours_at_the_edges(ptm, kind, dtype, pbc, wrap):
    rng = I.rng_for(41)
    pos, cell = _frame(kind, rng)
    if wrap == "unwrapped":
        pos = pos + (rng.integers(-2, 3, (len(pos), 3)) * np.array(pbc)) @ cell
    for ordering in ("euclidean", "topological"):
        _check(ptm, np.ascontiguousarray(pos, dtype), cell, pbc, ordering)


@pytest.mark.parametrize("kind,a,reps", [("fcc", I.A_FCC_CU, 3), ("fcc", I.A_FCC_CU, 6), ("bcc", I.A_BCC_FE, 5),
                                         ("hcp", I.A_HCP, (5, 3, 3)), ("sc", I.A_SC, 5)])
@pytest.mark.parametrize("sigma", [0.0, 1e-6])
@pytest.mark.parametrize("wrap", ["inside", "unwrapped"])
def test_near_ties_follow_fp64(ptm, kind, a, reps, sigma, wrap):
    """Mirror-image neighbours whose float32 distances do not give the FP64 order."""
    f = I.crystal(kind, a, reps, sigma=sigma, seed=4, rotation=I.random_rotation(I.rng_for(31)))
    pos = f.positions
    if wrap == "unwrapped":
        pos = pos + I.rng_for(9).integers(-2, 3, (f.n, 3)) @ f.cell
    s = _check(ptm, np.ascontiguousarray(pos, np.float32), f.cell, f.pbc, "euclidean")
    assert s["knn_fp64"] > f.n // 4


@pytest.mark.parametrize("sigma", [0.0, 1e-7])
def test_near_ties_across_a_long_periodic_side(ptm, sigma):
    """As above, for neighbours reached through an image 1,000 Angstrom away."""
    c = I.crystal("fcc", I.A_FCC_CU, (8, 4, 4), sigma=sigma, seed=6)
    cell = np.diag([1000.0, 4 * I.A_FCC_CU, 4 * I.A_FCC_CU])
    pos = c.positions.copy()
    pos[:, 0] = np.mod(pos[:, 0] - 4 * I.A_FCC_CU, 1000.0)
    s = _check(ptm, np.ascontiguousarray(pos, np.float32), cell, (True, True, True), "euclidean")
    assert s["knn_fp64"] > 0


@pytest.mark.parametrize("kind,a,reps", [("fcc", I.A_FCC_CU, 29), ("bcc", I.A_BCC_FE, 36)])
def test_a_full_shell_inside_the_widest_radius_is_enough(ptm, kind, a, reps):
    """The 18 nearest of an fcc atom are its first two shells, and the third lies outside
    the radius that 27 cells cover: no reason for the warp search, which counts every
    atom it takes in FP64."""
    import torch
    f = I.crystal(kind, a, reps, sigma=0.01, seed=1, dtype=np.float32)
    out = ptm.classify(torch.from_numpy(f.positions).cuda(), f.cell, f.pbc, ordering="topological")
    torch.cuda.synchronize()
    s = ptm.stats()
    assert s["internal"] == 0 and s["knn_fp64"] < f.n // 8
    atoms = I.rng_for(5).permutation(f.n)[:24]
    ref = O.Frame(f.positions, f.cell, f.pbc).classify(atoms, ordering="topological")
    compare({k: v.cpu().numpy() for k, v in out.items()}, ref, atoms)
