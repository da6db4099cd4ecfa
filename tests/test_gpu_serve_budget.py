"""What a server's budget admits (GPU only): a float32 frame is charged 359 bytes an atom, 416
in the topological order, and a frame that fits is served."""
import numpy as np
import pytest

from paper_1603_05143_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ordering,per_atom", [("euclidean", 359), ("topological", 420)])
@pytest.mark.parametrize("wrap", [True, False])
def test_frame_at_the_budget(ordering, per_atom, wrap):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_05143_gb300 import PTM, PTMError, Server
    f = I.crystal("fcc", I.A_FCC_CU, 24, sigma=0.05, seed=1, dtype=np.float32)     # 55,296 atoms
    pos = f.positions if wrap else (f.positions + I.rng_for(3).integers(-2, 3, (f.n, 3)) @ f.cell).astype(np.float32)
    ptm = PTM(0)
    budget = per_atom * f.n + 80 * 1024                 # descriptors, tables and their alignment
    srv = Server(ptm, hbm_budget_bytes=budget)
    out = srv.wait(srv.submit(pos, f.cell, f.pbc, ordering=ordering), 60000)
    want = ptm.classify(torch.from_numpy(pos).cuda(), f.cell, f.pbc, ordering=ordering)
    torch.cuda.synchronize()
    for k, v in want.items():
        assert np.array_equal(out[k], v.cpu().numpy()), k
    srv.close()
    srv = Server(ptm, hbm_budget_bytes=budget - 8 * f.n)
    with pytest.raises(PTMError):
        srv.wait(srv.submit(pos, f.cell, f.pbc, ordering=ordering), 60000)
    srv.close()
    ptm.close()
