"""Doubled atoms (GPU only): two atoms on one point, as a bad restart file or a
joined pair of frames leaves them, against the oracle in both neighbour orders.  The
copy at distance zero has no bisector plane: its face has no area."""
import numpy as np
import pytest

import oracle as O
from paper_1603_05143_gb300 import inputs as I
from parity import compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reps", [6, 8])                  # 867 and 2,051 atoms: either side of the small frames' search
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("ordering", ["euclidean", "topological"])
@pytest.mark.parametrize("path", ["frame", "batch"])
def test_doubled_atoms(reps, dtype, ordering, path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_05143_gb300 import PTM
    f = I.crystal("fcc", I.A_FCC_CU, reps, sigma=0.08, seed=reps, dtype=dtype)
    side = reps * I.A_FCC_CU

    def apart(x):                                          # minimum-image distance of every atom from x
        d = f.positions.astype(np.float64) - x
        return np.linalg.norm(d - side * np.round(d / side), axis=1)

    sites = [0]                                            # three atoms that are not among each other's neighbours
    while len(sites) < 3:
        sites.append(int(np.argmax(np.min([apart(f.positions[s]) for s in sites], axis=0))))
    pos = np.vstack([f.positions, f.positions[sites]])
    copies = np.array(sites + [f.n, f.n + 1, f.n + 2])
    atoms = np.arange(len(pos))
    if ordering == "topological":
        # an atom with both copies among its 18 nearest has two faces in one plane,
        # divided by rounding alone: no reference for those
        near = np.min([apart(f.positions[s]) for s in sites], axis=0) < 1.7 * I.A_FCC_CU
        near[sites] = False
        atoms = np.concatenate([np.nonzero(~near)[0], copies[3:]])
    ptm = PTM(0)
    dev = torch.from_numpy(np.ascontiguousarray(pos)).cuda()
    if path == "frame":
        out = ptm.classify(dev, f.cell, f.pbc, ordering=ordering)
        torch.cuda.synchronize()
        assert ptm.stats()["internal"] == 0
    else:
        b = ptm.batch([{"positions": dev, "cell": f.cell, "pbc": f.pbc, "ordering": ordering}])
        b.run()
        torch.cuda.synchronize()
        assert b.stats()["internal"] == 0
        out = b.outputs[0]
    got = {k: v.cpu().numpy() for k, v in out.items()}
    ref = O.Frame(pos, f.cell, f.pbc).classify(atoms, ordering=ordering)
    # a nearest neighbour on the atom itself leaves no hull around the centre in the
    # Euclidean order; by face area the twelve real neighbours come first
    assert np.all(ref["structure"][np.isin(atoms, copies)] == (2 if ordering == "topological" else 0))
    compare(got, ref, atoms)
    if path == "batch":
        b.close()
    ptm.close()


@pytest.mark.parametrize("e,block", [(1e-7, 4), (1e-7, 6), (1e-8, 0), (1e-8, 2)])
def test_neighbours_almost_on_one_point(e, block):
    """Clusters with one second-shell neighbour doubled at a distance e: FP32 cannot place the
    line between the two faces, so it must not choose what the FP64 areas are cut by.  In
    these sets 2 or 3 of the 4,000 centres took a wrong structure when it did."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_05143_gb300 import PTM
    rng = np.random.default_rng([block, 2 if e == 1e-7 else 3])
    grid = np.array([[a, b, c] for a in range(-2, 3) for b in range(-2, 3) for c in range(-2, 3)
                     if (a or b or c) and (a + b + c) % 2 == 0], float)

    def cluster():
        p = 1.8 * grid + rng.uniform(0.02, 0.12) * rng.normal(size=grid.shape)
        p = p[np.argsort((p ** 2).sum(1))]
        w = rng.integers(12, 18)
        return np.vstack([np.zeros((1, 3)), p, p[w:w + 1] + e * rng.normal(size=(1, 3))])

    side, n = 16, 4000
    clusters = [cluster() for _ in range(n)]
    at = np.array([[x, y, z] for x in range(side) for y in range(side) for z in range(side)], float)[:n] * 30.0 + 15.0
    clusters = [c + x for c, x in zip(clusters, at)]
    cell = np.eye(3) * 30.0 * side
    ptm = PTM(0)
    out = ptm.classify(torch.from_numpy(np.vstack(clusters)).cuda(), cell, (True, True, True), ordering="topological")
    got = out["structure"].cpu().numpy()[::len(clusters[0])]
    want = np.array([O.Frame(c, cell).classify(np.array([0]), ordering="topological")["structure"][0] for c in clusters])
    assert np.array_equal(got, want), np.nonzero(got != want)[0]
    ptm.close()
