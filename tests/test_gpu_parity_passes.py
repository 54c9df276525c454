"""The transform passes by parity (periodic meshes of 160 nodes per axis and more): the
mesh solve alone, and one step with its paired right-hand sides, on the smallest such
mesh, odd node counts (a middle node without a partner), counts that leave partial tiles
and chunks, and rows that are and are not whole vectors, against the multigrid inner
solver and against one right-hand side at a time.

Tolerances: the residual the refinement reaches (mixed 1e-10, FP64 1e-13), with the
solves' agreement at ten times it and more for the conditioning (relative 1e-8, 1e-11).
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


@pytest.mark.parametrize("n_el", [54, 55, 57, 64, 86])
def test_mesh_solve(api, n_el):
    import torch
    b = torch.randn((3 * n_el) ** 3, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n_el))
    b -= b.mean()
    ref = api.FEP3M(1.0, n_el, precision="fp64", solver="multigrid")
    want = ref.solve_mesh(b)
    assert ref.stats()["mg_rel_residual"] <= 1e-13
    ref.close()
    for precision, tol, rtol in (("fp64", 1e-11, 1e-13), ("mixed", 1e-8, 1e-10)):
        eng = api.FEP3M(1.0, n_el, precision=precision)
        for _ in range(2):   # the checked solve, then its replay
            phi = eng.solve_mesh(b)
            assert eng.stats()["mg_rel_residual"] <= rtol
            assert float((phi - want).abs().max()) < tol * float(want.abs().max())
        eng.close()


@pytest.mark.parametrize("n_el", [55, 56])
def test_paired_step(api, n_el):
    """Phi and forces of a step (both right-hand sides in each pass) against the FP64
    path's, and Phi against the same step without forces (one right-hand side)."""
    import torch
    pos, Q = workloads.uniform_pm(3000, seed=41)
    p, q = torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda")
    out = {}
    for precision in ("fp64", "mixed"):
        eng = api.FEP3M(1.0, n_el, precision=precision)
        eng.set_particles(p, q)
        out[precision] = eng.compute(forces=True)
        one = eng.compute(forces=False)["phi"]
        assert float((out[precision]["phi"] - one).abs().max()) < 1e-9 * float(one.abs().max())
        eng.close()
    for key, tol in (("phi", 1e-6), ("forces", 1e-5)):
        a, b = out["mixed"][key], out["fp64"][key]
        assert float((a - b).norm()) < tol * float(b.norm())


def test_many_steps_agree(api):
    """Persistent CTAs, their barriers' phases over many jobs: the same step ten times."""
    import torch
    pos, Q = workloads.uniform_pm(5000, seed=42)
    eng = api.FEP3M(1.0, 60, precision="mixed")
    p, q = torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda")
    first = None
    for _ in range(10):
        eng.set_particles(p, q)
        o = eng.compute(forces=True)
        got = np.concatenate([o["phi"].cpu().numpy(), o["forces"].cpu().numpy().ravel()])
        if first is None:
            first = got
        assert np.array_equal(first, got) or np.abs(first - got).max() < 1e-9 * np.abs(first).max()
    eng.close()
