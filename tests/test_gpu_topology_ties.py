"""Faces of perfect lattices (GPU only): corners of a face lie on further planes, which
rounding may put on either side.  The FP32 pass decides such faces itself, and the order
is still the oracle's."""
import numpy as np
import pytest

import oracle as O
from paper_1603_05143_gb300 import inputs as I
from parity import compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,a,reps", [("sc", I.A_SC, 45), ("fcc", I.A_FCC_CU, 29), ("hcp", I.A_HCP, (30, 20, 18))])
@pytest.mark.parametrize("sigma", [0.0, 1e-6])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("rotate", [False, True])
def test_perfect_faces_stay_in_fp32(kind, a, reps, sigma, dtype, rotate):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_05143_gb300 import PTM
    f = I.crystal(kind, a, reps, sigma=sigma, seed=1, rotation=I.random_rotation(I.rng_for(3)) if rotate else None,
                  dtype=dtype)
    ptm = PTM(0)
    out = ptm.classify(torch.from_numpy(f.positions).cuda(), f.cell, f.pbc, ordering="topological")
    torch.cuda.synchronize()
    s = ptm.stats()
    assert s["topo_fp64"] == 0 and s["internal"] == 0
    atoms = I.rng_for(5).permutation(f.n)[:24]
    ref = O.Frame(f.positions, f.cell, f.pbc).classify(atoms, ordering="topological")
    compare({k: v.cpu().numpy() for k, v in out.items()}, ref, atoms)
    ptm.close()
