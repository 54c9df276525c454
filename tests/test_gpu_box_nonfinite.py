"""A Dirichlet box with charges exactly on boundary nodes, whose boundary values are
infinite: mixed contexts answer as FP64 ones do (status, residual, sweeps, which results
are finite), and the engine stays usable.
"""
import numpy as np
import pytest

from paper_1503_08509_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_08509_gb300 import api as a, build
    build.build()
    return a


# the charges put on nodes (element coordinates; 8 elements, L = 1: exact), and their values
@pytest.mark.parametrize("at", [[((0, 0, 0), 1.0)], [((8, 3, 2), -1.0)], [((0, 0, 0), 1.0), ((1, 0, 0), -1.0)],
                                [((0, 4, 4), 1.0), ((0, 4, 5), 1.0), ((0, 5, 4), -2.0)], [((3, 3, 8), 0.0)]])
def test_infinite_boundary_value(api, at):
    import torch
    pos, Q = workloads.box_charges(40, L=1.0, seed=11)
    bad, Qb = pos.copy(), Q.copy()
    for i, (x, q) in enumerate(at):
        bad[i], Qb[i] = np.array(x) / 8.0, q
    got = {}
    for precision in ("fp64", "mixed"):
        eng = api.FEP3M(1.0, 8, precision=precision, dirichlet=True)
        eng.set_particles(torch.tensor(bad, device="cuda"), torch.tensor(Qb, device="cuda"))
        out = eng.compute(forces=False, allow_noconv=True)
        st = eng.stats()
        got[precision] = (out["status"], repr(st["mg_rel_residual"]), st["refine_steps"],
                          torch.isfinite(out["phi"]).cpu().tolist(), np.isfinite(eng.mesh()["phi_mesh"]).tolist())
        eng.set_particles(torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda"))
        assert np.isfinite(eng.compute(forces=False)["phi"].cpu().numpy()).all()
        eng.close()
    assert got["mixed"] == got["fp64"], [g[:3] + (sum(g[3]), sum(g[4])) for g in got.values()]
