"""Clusters in boxes of vacuum inside a batch (GPU only): their cells are read by a thread per
atom, in one pass that keeps the nearest.  Against the same atoms in boxes that fit them,
and against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1603_05143_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _ptm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_05143_gb300 import PTM
    return PTM(0)


def _cluster(kind, a, n, sigma, seed):
    f = I.crystal(kind, a, 20, sigma=sigma, seed=seed, rotation=I.random_rotation(I.rng_for(seed)), wrap=False)
    pos = f.positions - f.positions.mean(0)
    return pos[np.argsort((pos ** 2).sum(1), kind="stable")[:n]]


def _same_match(got, ref, atoms):
    """Structure and correspondence, atom ids in their order: what the neighbour lists decide.  (The
    FP32 strain of a perfect surface's chance matches, flat to rounding, is not compared.)"""
    assert np.array_equal(got["structure"].cpu().numpy()[atoms], ref["structure"])
    assert np.array_equal(got["correspondence"].cpu().numpy()[atoms], ref["corr"])


def _run(ptm, clusters, boxes, pbc, ordering):
    import torch
    b = ptm.batch([{"positions": torch.from_numpy(c).cuda(), "cell": np.eye(3) * s, "pbc": pbc, "ordering": ordering}
                   for c, s in zip(clusters, boxes)])
    b.run()
    torch.cuda.synchronize()
    s = b.stats()
    assert s["internal"] == 0 and s["knn_fail"] == 0
    outputs = [{k: v.clone() for k, v in o.items()} for o in b.outputs]
    b.close()
    return outputs


@pytest.mark.parametrize("n,frames", [(300, 40), (700, 16), (1100, 10), (3000, 4), (8000, 2)])
@pytest.mark.parametrize("vacuum", [2, 3, 10])             # box over diameter
@pytest.mark.parametrize("sigma", [0.0, 0.1])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("ordering", ["euclidean", "topological"])
def test_clusters_in_a_batch(n, frames, vacuum, sigma, dtype, ordering):
    import torch
    ptm = _ptm()
    kinds = [("fcc", I.A_FCC_CU), ("bcc", I.A_BCC_FE), ("hcp", I.A_HCP), ("sc", I.A_SC)]
    clusters, wide, near = [], [], []
    for i in range(frames):
        c = _cluster(*kinds[i % 4], n, sigma, 10 * n + i)
        clusters.append(np.ascontiguousarray(c, dtype))    # around a corner: in unwrapped coordinates
        d = 2 * np.sqrt((c ** 2).sum(1).max())
        wide.append(vacuum * d)
        near.append(1.5 * d)
    a = _run(ptm, clusters, wide, (True, True, True), ordering)
    b = _run(ptm, clusters, near, (True, True, True), ordering)
    for x, y in zip(a, b):
        for k in x:
            assert torch.equal(x[k], y[k]), k
    atoms = np.arange(0, n, max(1, n // 20))
    for i in (0, 1):
        ref = O.Frame(clusters[i], np.eye(3) * wide[i], (True, True, True)).classify(atoms, ordering=ordering)
        _same_match(a[i], ref, atoms)
    ptm.close()


@pytest.mark.parametrize("points", [10, 13, 40, 70, 100])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("ordering", ["euclidean", "topological"])
def test_many_atoms_at_one_distance(points, dtype, ordering):
    """A centre, a first shell of 12, and then more atoms at almost one distance than a list
    holds, amid crystals that crowd the cells: no radius parts them."""
    ptm = _ptm()
    rng = I.rng_for(points)
    shell = rng.normal(size=(points, 3))
    shell *= 4.0 / np.linalg.norm(shell, axis=1, keepdims=True)
    first = _cluster("fcc", I.A_FCC_CU, 13, 0.0, 3)
    ball = _cluster("fcc", I.A_FCC_CU, 1300, 0.08, 4)
    r = np.sqrt((ball ** 2).sum(1).max())
    pos = np.vstack([first - first[0], shell, ball + [r + 9.0, 0.0, 0.0]])
    side = 60.0 * r
    frames = [np.ascontiguousarray(pos + side / 2 + rng.normal(size=3), dtype) for _ in range(8)]
    out = _run(ptm, frames, [side] * 8, (False, False, False), ordering)
    atoms = np.arange(0, 13 + points)
    if ordering == "topological":
        atoms = atoms[:1]        # atoms of the random shell may touch: faces divided by rounding alone
    for f, o in zip(frames, out):
        ref = O.Frame(f, np.eye(3) * side, (False, False, False)).classify(atoms, ordering=ordering)
        _same_match(o, ref, atoms)
    ptm.close()
