"""fep3m_vjp after a forward without forces reuses that forward's mesh solution: the
gradients agree with those after a forward with forces (which evaluated the charges'
fields itself) and with those of a vjp that had no forward at all, whatever was asked of
the context in between, and a second one repeats the first bit by bit.

Tolerances: the two forwards' mesh solutions agree to the refinement's residual, 1e-10
(mixed) and 1e-13 (FP64); the gradients to a hundred times that.
"""
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


@pytest.mark.parametrize("precision,tol", [("mixed", 1e-8), ("fp64", 1e-11)])
@pytest.mark.parametrize("n_el,n_sr,N,kw", [(7, 3, 60, {}), (12, 2, 900, {}), (12, 3, 900, dict(solver="multigrid")),
                                            (54, 3, 4000, {})])
def test_vjp_reuses_the_forward(api, precision, tol, n_el, n_sr, N, kw):
    import torch
    pos, Q = workloads.uniform_pm(N, seed=n_el)
    p, q = torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda")
    g = torch.randn(N, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    eng = api.FEP3M(1.0, n_el, n_sr=n_sr, precision=precision, **kw)

    def after(prepare):
        eng.set_particles(p, q)
        prepare()
        return [t.clone() for t in eng.vjp(0.7, g)]

    def between():
        eng.compute(forces=False)
        eng.solve_mesh(torch.linspace(-1, 1, (3 * n_el) ** 3, dtype=torch.float64, device="cuda"))
        eng.binning()
        eng.mesh()
        eng.stats()

    want = after(lambda: eng.compute(forces=True))
    for prepare in (lambda: eng.compute(forces=False), lambda: None, between):
        for _ in range(2):
            got = after(prepare)
            for a, b in zip(got, want):
                assert float((a - b).norm()) < tol * float(b.norm())
        again = eng.vjp(0.7, g)
        assert all(torch.equal(a, b) for a, b in zip(again, got))
    # other charges: nothing of the earlier forward is used
    q2 = -q
    eng.set_particles(p, q2)
    eng.compute(forces=False)
    dpos, dQ = eng.vjp(0.7, g)
    eng.set_particles(p, q2)
    ref = eng.vjp(0.7, g)
    for a, b in zip((dpos, dQ), ref):
        assert float((a - b).norm()) < tol * float(b.norm())
    eng.close()
