"""The screen adjoint's gather, with eight threads per vertex (below 40 elements per axis)
and with one: forces against the energy's central difference along a random direction, on
meshes with whole and partial last CTAs, most elements empty, every block half-width.

Tolerances: the difference quotient's truncation is (step / nearest distance)^2 < 1e-6 and
its rounding below 1e-6 of the slope (1e-5 allowed); the mixed path's forces have its
32-bit accuracy (2e-5 of the largest).
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


@pytest.mark.parametrize("n_sr", [1, 2, 3, 4])
@pytest.mark.parametrize("n_el", [39, 40, 41])
def test_forces_are_the_energys_slope(api, n_el, n_sr):
    import torch
    pos, Q = workloads.uniform_pm(300, seed=n_el + n_sr)
    p, q = torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda")
    h = 1.0 / n_el
    # away from the element faces, where the discrete energy has kinks: the elements stay the same
    p = ((p / h).floor() + 0.01 + 0.98 * ((p / h) % 1.0)) * h
    t = torch.randn(p.shape, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n_sr))
    step = 1e-4 * h / float(t.abs().max())
    eng = api.FEP3M(1.0, n_el, n_sr=n_sr, precision="fp64")

    def energy(x):
        eng.set_particles(x, q)
        return eng.compute(forces=False)["U"]
    slope = (energy(p + step * t) - energy(p - step * t)) / (2 * step)
    eng.set_particles(p, q)
    F = eng.compute(forces=True)["forces"]
    eng.close()
    assert abs(float((F * t).sum()) + slope) < 1e-5 * float((F * t).norm())
    eng = api.FEP3M(1.0, n_el, n_sr=n_sr, precision="mixed")
    eng.set_particles(p, q)
    Fm = eng.compute(forces=True)["forces"]
    eng.close()
    assert float((Fm - F).abs().max()) < 2e-5 * float(F.abs().max())
