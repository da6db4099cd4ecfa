"""An area gap at the edge of the equal-area band beside three faces (GPU only): two of them
differ by less than FP32 resolves, so FP32 cannot tell which one the gap belongs to.  Against
the oracle, with a mask that leaves the match to the first six neighbours in the order."""
import numpy as np
import pytest

import oracle as O
from paper_1603_05143_gb300 import inputs as I
from parity import compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_faces_that_may_change_places_beside_a_gap(dtype):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_05143_gb300 import PTM
    f = I.crystal("bcc", I.A_BCC_FE, 80, sigma=0.01, seed=2, rotation=I.random_rotation(I.rng_for(3)), dtype=np.float32)
    # the neighbourhoods of one such atom and of some others, cut out of the crystal
    for atom in (713175, 1000, 500000):
        d = np.linalg.norm(f.positions.astype(np.float64) - f.positions[atom], axis=1)
        near = np.nonzero(d < 9.0)[0]
        pos = np.ascontiguousarray(f.positions[near], dtype)
        at = np.nonzero(near == atom)[0]
        ptm = PTM(0)
        out = ptm.classify(torch.from_numpy(pos).cuda(), f.cell, (False, False, False), mask=1, ordering="topological")
        torch.cuda.synchronize()
        got = {k: v.cpu().numpy() for k, v in out.items()}
        ref = O.Frame(pos, f.cell, (False, False, False)).classify(at, mask=1, ordering="topological")
        compare(got, ref, at)
        ptm.close()
