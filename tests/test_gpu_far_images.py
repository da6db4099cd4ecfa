"""Coordinates many periods outside the cell (GPU only): up to 100 are accepted, so
two neighbours may stand 200 images apart.  Against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1603_05143_gb300 import inputs as I
from parity import compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reps", [4, 8])                  # 256 and 2,048 atoms
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("ordering", ["euclidean", "topological"])
@pytest.mark.parametrize("path", ["frame", "batch"])
@pytest.mark.parametrize("pbc", [(True, True, True), (True, False, True)])
def test_atoms_many_periods_apart(reps, dtype, ordering, path, pbc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_05143_gb300 import PTM
    f = I.crystal("fcc", I.A_FCC_CU, reps, sigma=0.08, seed=reps)
    n = I.rng_for(reps).integers(-98, 99, (f.n, 3)) * np.array(pbc)
    pos = np.ascontiguousarray(f.positions + n @ f.cell, dtype)
    ptm = PTM(0)
    dev = torch.from_numpy(pos).cuda()
    if path == "frame":
        out = ptm.classify(dev, f.cell, pbc, ordering=ordering)
    else:
        b = ptm.batch([{"positions": dev, "cell": f.cell, "pbc": pbc, "ordering": ordering}])
        b.run()
        out = b.outputs[0]
    torch.cuda.synchronize()
    s = ptm.stats() if path == "frame" else b.stats()
    assert s["internal"] == 0 and s["excluded"] == 0
    got = {k: v.cpu().numpy() for k, v in out.items()}
    atoms = np.arange(0, f.n, max(1, f.n // 400))
    compare(got, O.Frame(pos, f.cell, pbc).classify(atoms, ordering=ordering), atoms)
    if path == "batch":
        b.close()
    ptm.close()
