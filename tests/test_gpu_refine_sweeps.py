"""The refinement of the boxes and of the order-q mesh: its cap on the sweeps is the
caller's (also past the residual norms kept on the device).
"""
import pytest

from paper_1503_08509_gb300 import workloads

pytestmark = pytest.mark.gpu

KINDS = [dict(dirichlet=True), dict(neumann=True), dict(q=2)]


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_08509_gb300 import api as a, build
    build.build()
    return a


def engine(api, precision, kind, n_el=8, **kw):
    import torch
    pos, Q = workloads.uniform_pm(60, seed=1) if "q" in kind else workloads.box_charges(60, L=1.0, seed=1)
    eng = api.FEP3M(1.0, n_el, precision=precision, **kind, **kw)
    eng.set_particles(torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda"))
    return eng


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("cap", [1, 31, 32, 45])
def test_cap_on_the_sweeps(api, precision, kind, cap):
    """A tolerance out of reach: as many sweeps as the caller allows, the second time too."""
    eng = engine(api, precision, kind, mg_rtol=1e-30, mg_max_cycles=cap)
    for _ in range(2):
        out = eng.compute(forces=False, allow_noconv=True)
        st = eng.stats()
        assert out["status"] != 0 and st["refine_steps"] == cap
        assert 0.0 < st["mg_rel_residual"] < (1e-3 if cap == 1 else 1e-11)
    eng.close()
