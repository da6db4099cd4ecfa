"""``knn_fp64`` (GPU only): the atoms with two candidates within the FP32 error bound,
whichever kernel searched.  A small frame, whose atoms each have a warp, counts what the
same frame counts inside a batch."""
import numpy as np
import pytest

from paper_1603_05143_gb300 import inputs as I
from test_gpu_knn import _frame

pytestmark = pytest.mark.gpu


def _case(kind):
    rng = I.rng_for(17)
    if kind in ("clump", "hole", "dilute", "long", "handful"):
        return _frame(kind, rng)
    sigma = {"perfect": 0.0, "cold": 1e-6, "warm": 0.1, "unwrapped": 0.1}[kind]
    f = I.crystal("fcc", I.A_FCC_CU, 6, sigma=sigma, seed=2, rotation=I.random_rotation(rng))
    pos = f.positions
    if kind == "unwrapped":
        pos = pos + rng.integers(-2, 3, (f.n, 3)) @ f.cell
    return pos, f.cell


@pytest.mark.parametrize("kind", ["perfect", "cold", "warm", "unwrapped", "clump", "hole", "dilute", "long", "handful"])
@pytest.mark.parametrize("ordering", ["euclidean", "topological"])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_small_frame_counts_what_its_batch_counts(kind, ordering, dtype):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_05143_gb300 import PTM
    pos, cell = _case(kind)
    pos = torch.from_numpy(np.ascontiguousarray(pos, dtype)).cuda()
    pbc = (True, True, True)
    ptm = PTM(0)
    one = ptm.classify(pos, cell, pbc, ordering=ordering)
    b = ptm.batch([{"positions": pos, "cell": cell, "pbc": pbc, "ordering": ordering}])
    b.run()
    torch.cuda.synchronize()
    for k, v in one.items():
        assert torch.equal(v, b.outputs[0][k]), k
    s, t = ptm.stats()["knn_fp64"], b.stats()["knn_fp64"]
    assert s == t
    if dtype == np.float64:
        assert s == 0
    elif kind == "perfect":
        assert s > len(pos) // 2
    elif kind == "warm":
        assert s < len(pos) // 10
    b.close()
    ptm.close()
