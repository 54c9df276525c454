"""FP64 contexts: fep3m_vjp is linear in (gU, gphi) over a wide range of units, and the
forces are quadratic in the charges' unit over the admitted range, although the screen
adjoint's sums run in float pairs.

Powers of two, so that nothing but the range could tell the results apart.  Tolerance:
2^-48, the pairs' rounding, for the sums whose exponents differ (the mesh solve scales its
residuals by powers of two itself).
"""
import pytest

from paper_1503_08509_gb300 import workloads

pytestmark = pytest.mark.gpu

TOL = 2.0 ** -48


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_08509_gb300 import api as a, build
    build.build()
    return a


def setup(api, n_el, n_sr, N):
    import torch
    pos, Q = workloads.uniform_pm(N, seed=3)
    eng = api.FEP3M(1.0, n_el, n_sr=n_sr, precision="fp64")
    return eng, torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda")


@pytest.mark.parametrize("n_el,n_sr,N", [(9, 2, 400), (10, 4, 300), (41, 3, 1500)])
@pytest.mark.parametrize("gU,gphi", [(0.7, True), (0.0, True), (0.7, False)])
def test_vjp_is_linear(api, n_el, n_sr, N, gU, gphi):
    import torch
    eng, p, q = setup(api, n_el, n_sr, N)
    eng.set_particles(p, q)
    eng.compute(forces=True)
    g = torch.randn(N, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1)) if gphi else None
    want = [t.clone() for t in eng.vjp(gU, g)]
    for k in (-180, -130, -100, -60, 60, 100, 130, 180):
        s = 2.0 ** k
        got = eng.vjp(gU * s, g * s if gphi else None)
        for a, b in zip(got, want):
            assert float((a / s - b).norm()) <= TOL * float(b.norm()), k
    if gphi:   # no weights at all, and one charge's alone
        assert all(float(t.abs().max()) == 0.0 for t in eng.vjp(0.0, torch.zeros_like(g)))
        one = torch.zeros_like(g)
        one[N // 2] = 1.0
        want = [t.clone() for t in eng.vjp(0.0, one)]
        for a, b in zip(eng.vjp(0.0, one * 2.0 ** -170), want):
            assert float((a * 2.0 ** 170 - b).norm()) <= TOL * float(b.norm())
    eng.close()


@pytest.mark.parametrize("gU", [0.0, 1e-300, 5e-324])
def test_vanishing_weights_on_a_fresh_engine(api, gU):
    """Weights of zero, and ones that the scale's exponent cannot take to its target: finite."""
    import torch
    eng, p, q = setup(api, 9, 2, 400)
    eng.set_particles(p, q)
    for t in eng.vjp(gU, None):
        assert bool(torch.isfinite(t).all()) and (gU > 0.0 or float(t.abs().max()) == 0.0)
    eng.close()


@pytest.mark.parametrize("n_el,n_sr,N", [(9, 2, 400), (10, 4, 300)])
def test_forces_scale_with_the_charges(api, n_el, n_sr, N):
    eng, p, q = setup(api, n_el, n_sr, N)
    eng.set_particles(p, q)
    want = eng.compute(forces=True)["forces"].clone()
    for k in (-100, -90, -40, 40, 90, 100):
        eng.set_particles(p, q * 2.0 ** k)
        got = eng.compute(forces=True)["forces"] / 4.0 ** k
        assert float((got - want).norm()) <= TOL * float(want.norm()), k
    eng.close()
