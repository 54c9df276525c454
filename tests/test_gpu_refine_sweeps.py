"""The refinement of the boxes and of the order-q mesh: its cap on the sweeps is the
caller's (also past the residual norms kept on the device), a tight tolerance is met, and a solution does not depend
on what the engine solved before (the sweeps queued before the norms are read follow the
last solve).
"""
import numpy as np
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


@pytest.mark.parametrize("n_el", [8, 20])
@pytest.mark.parametrize("kind", KINDS)
def test_tight_tolerance(api, kind, n_el):
    """Mixed contexts: residuals that FP64 arithmetic reaches (2e-15 to 2e-14 at 8^3, growing with
    the mesh) and float pairs do not (1e-13 and more)."""
    eng = engine(api, "mixed", kind, n_el, mg_rtol=5e-15 * (n_el / 8))
    out = eng.compute(forces=False)
    assert out["status"] == 0 and eng.stats()["mg_rel_residual"] <= 5e-14 * (n_el / 8)
    eng.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("kind", KINDS)
def test_no_memory_of_earlier_solves(api, precision, kind):
    """An easy right-hand side (alternating: the largest eigenvalues, no level to remove) after a
    harder one and on a fresh engine, and the harder one after the easy one: the same bits."""
    import torch

    def easy(eng):
        m = round(eng.nodes ** (1 / 3))
        s = (-1.0) ** np.arange(m)
        b = torch.tensor((s[:, None, None] * s[:, None] * s).ravel(), device="cuda")
        b += 0.1 * torch.randn(eng.nodes, dtype=torch.float64, device="cuda",
                               generator=torch.Generator("cuda").manual_seed(2))
        phi, st = eng.solve_mesh(b), eng.stats()
        return phi, st["refine_steps"], st["mg_rel_residual"]

    def hard(eng):
        phi, st = eng.compute(forces=False)["phi"].clone(), eng.stats()
        return phi, st["refine_steps"], st["mg_rel_residual"]

    for first, second in ((easy, hard), (hard, easy)):
        eng = engine(api, precision, kind)
        want = second(eng)
        eng.close()
        eng = engine(api, precision, kind)
        first(eng)
        got = second(eng)
        eng.close()
        assert torch.equal(got[0], want[0]) and got[1:] == want[1:], (got[1:], want[1:])
