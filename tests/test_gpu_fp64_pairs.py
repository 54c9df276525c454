"""The FP64 path's kernels in float pairs (screen contraction and screen adjoint by
parity, singular sums) and the element deposit where their sizes and ranges differ:
every block half-width, meshes that are not whole bricks or whole tiles of 32
elements, one charge, crowded elements, nearly coincident charges, extreme units.

Tolerances: FP64 max|d| / max|ref| 1e-11 for potentials and 1e-10 for gradients (those
of the FP64 path); powers of two of the charges scale the results to rounding.
"""
import numpy as np
import pytest

from oracle import fep3m as ofe
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


def run(api, pos, Q, n_el, n_sr, precision="fp64"):
    import torch
    eng = api.FEP3M(1.0, n_el, n_sr=n_sr, precision=precision, neutralize=True)
    eng.set_particles(torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda"))
    out = eng.compute(forces=True)
    phi, F, U = out["phi"].cpu().numpy(), out["forces"].cpu().numpy(), out["U"]
    eng.close()
    return phi, F, U


def maxrel(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


def charges(kind, N):
    pos, Q = workloads.uniform_pm(N, seed=31)
    if kind == "crowded":       # most charges in a few elements
        pos[: 3 * N // 4] = 0.3 + 0.02 * pos[: 3 * N // 4]
    return pos, Q


@pytest.mark.parametrize("n_el,n_sr,kind,N", [
    (3, 1, "uniform", 1), (5, 2, "uniform", 70), (9, 4, "uniform", 120), (7, 3, "crowded", 300), (10, 3, "uniform", 33)])
def test_matches_oracle(api, n_el, n_sr, kind, N):
    pos, Q = charges(kind, N)
    ref = ofe.forward(pos, Q, 1.0, n_el, n_sr=n_sr, want_grad=True)
    dx, _, _ = ofe.vjp(ref, Q, n_sr=n_sr)
    phi, F, U = run(api, pos, Q, n_el, n_sr)
    assert maxrel(phi, ref["phi"]) < 1e-11
    assert abs(U - ref["U"]) <= 1e-11 * abs(ref["U"])
    assert np.abs(F + dx).max() <= 1e-10 * np.abs(dx).max() + 1e-13


@pytest.mark.parametrize("d", [1e-6, 1e-9, 1e-12])
def test_nearly_coincident_charges(api, d):
    """A pair a distance d apart, inside and outside the pairs' range.  The charges' local
    coordinates (element units, below 1) are rounded to 2^-53, twice each: the pair's own
    term may be off by 8 2^-53 n_el / d of itself, everything else as usual."""
    n_el = 7
    pos, Q = charges("uniform", 40)
    pos[1] = pos[0] + [d, 0.0, 0.0]
    ref = ofe.forward(pos, Q, 1.0, n_el)["phi"]
    phi, _, _ = run(api, pos, Q, n_el, 3)
    own = 8 * 2.0 ** -53 / (d * n_el)
    assert np.all(np.abs(phi[:2] - ref[:2]) < (own + 1e-11) * np.abs(ref[:2]))
    assert maxrel(phi[2:], ref[2:]) < 1e-11


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n_el,kind,N", [(9, "uniform", 50), (7, "crowded", 900)])
def test_deposit_matches_oracle(api, precision, n_el, kind, N):
    """The adjoint's deposit over tiles of 32 elements, their charges held 32 at a time."""
    pos, Q = charges(kind, N)
    ref = ofe.forward(pos, Q, 1.0, n_el, want_grad=True)
    dx, _, _ = ofe.vjp(ref, Q)
    _, F, _ = run(api, pos, Q, n_el, 3, precision)
    assert np.linalg.norm(F + dx) < (1e-10 if precision == "fp64" else 1e-5) * np.linalg.norm(dx)


@pytest.mark.parametrize("unit", [2.0 ** -80, 2.0 ** 80])
def test_units(api, unit):
    pos, Q = charges("uniform", 200)
    a = run(api, pos, Q, 8, 3)
    b = run(api, pos, unit * Q, 8, 3)
    assert maxrel(b[0] / unit, a[0]) < 1e-12
    assert maxrel(b[1] / unit ** 2, a[1]) < 1e-11
