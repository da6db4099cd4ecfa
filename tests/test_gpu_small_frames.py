"""Frames around the sizes where launches change shape (GPU only): one warp per
neighbour search, one block for the cell list, fewer atoms per warp.  Every size
equals the same atoms classified inside a batch, which takes none of these."""
import numpy as np
import pytest

from paper_1603_05143_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [15, 31, 33, 607, 609, 1217, 1536, 1537, 2047, 2048, 2049, 4097])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_launch_shapes_agree(n, dtype):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_05143_gb300 import PTM
    side = int(np.ceil((n / 2) ** (1 / 3)))
    f = I.crystal("b2", I.A_BCC_FE, side, sigma=0.15, seed=n, rotation=I.random_rotation(I.rng_for(n)))
    keep = np.sort(I.rng_for(n + 1).permutation(f.n)[:n])                  # a few vacancies
    pos = torch.from_numpy(np.ascontiguousarray(f.positions[keep], dtype)).cuda()
    if n > 600:
        pos[5] = float("nan")                                             # excluded, nobody's neighbour
    sp = torch.from_numpy(f.species[keep]).cuda()
    ptm = PTM(0)
    one = ptm.classify(pos, f.cell, f.pbc, species=sp)
    b = ptm.batch([{"positions": pos, "species": sp, "cell": f.cell, "pbc": f.pbc}])
    b.run()
    torch.cuda.synchronize()
    for k, v in one.items():
        assert torch.equal(v, b.outputs[0][k]), k
    s1, s2 = ptm.stats(), b.stats()
    for k in ("atoms", "matched", "excluded", "internal", "candidates", "candidate_points", "sos"):
        assert s1[k] == s2[k], k
    assert s1["excluded"] == (1 if n > 600 else 0)
    b.close()
    ptm.close()
