"""The box's boundary sums (Dirichlet boundary values, Neumann face loads) where
their staging and their range can go wrong: every block half-width, blocks with
fewer charges than one staged chunk and with several, a partial last chunk,
charges of extreme units, charges on the faces, and a charge on a boundary node.

Tolerances: those of the box path (FP64 max|d| / max|ref| 1e-11, mixed relative
RMS 1e-6); the results scale with the charges and the data to rounding.
"""
import numpy as np
import pytest

from oracle import dirichlet, neumann
from paper_1503_08509_gb300 import workloads

pytestmark = pytest.mark.gpu

L = 1.1


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_08509_gb300 import api as a, build
    build.build()
    return a


def g(x):
    return 0.4 + 0.3 * x[:, 0] - 0.2 * x[:, 1] ** 2 + 0.1 * x[:, 2]


def gn(x, nr):
    return np.einsum('mk,mk->m', np.stack([0.3 + 0 * x[:, 0], -0.4 * x[:, 1], 0.2 + 0 * x[:, 2]], axis=1), nr)


def charges(N, dense):
    pos, Q = workloads.box_charges(N, L=L, seed=11)
    if dense:   # most of them in one corner: several staged chunks per block, the last one partial
        pos[6:] = pos[6:] * 0.4
    return pos, Q


def solve(api, kind, n_el, n_sr, precision, pos, Q, unit=1.0):
    import torch
    eng = api.FEP3M(L, n_el, n_sr=n_sr, precision=precision, **{kind: True})
    data = g(eng.node_points()) if kind == "dirichlet" else gn(*eng.face_points())
    eng.set_boundary(unit * data)
    eng.set_particles(torch.tensor(pos, device="cuda"), torch.tensor(unit * Q, device="cuda"))
    phi = eng.compute(forces=False)["phi"].cpu().numpy()
    eng.close()
    return phi / unit


@pytest.mark.parametrize("kind", ["dirichlet", "neumann"])
@pytest.mark.parametrize("n_el,n_sr,N,dense", [(5, 1, 7, False), (5, 2, 430, True), (9, 4, 61, False), (7, 3, 330, True)])
def test_boundary_sums(api, kind, n_el, n_sr, N, dense):
    pos, Q = charges(N, dense)
    ref = (dirichlet.forward(pos, Q, L, n_el, g, n_sr=n_sr) if kind == "dirichlet"
           else neumann.forward(pos, Q, L, n_el, gn, n_sr=n_sr))["phi"]
    for precision in ("fp64", "mixed"):
        phi = solve(api, kind, n_el, n_sr, precision, pos, Q)
        if precision == "fp64":
            assert np.abs(phi - ref).max() < 1e-11 * np.abs(ref).max()
        else:
            assert np.linalg.norm(phi - ref) < 1e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("kind", ["dirichlet", "neumann"])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 1e-5)])
@pytest.mark.parametrize("unit", [2.0 ** -80, 2.0 ** 80])
def test_units(api, kind, precision, tol, unit):
    """Charges and data times a power of two: the same potentials times it."""
    pos, Q = charges(150, False)
    a = solve(api, kind, 7, 3, precision, pos, Q)
    b = solve(api, kind, 7, 3, precision, pos, Q, unit=unit)
    assert np.abs(a - b).max() < tol * np.abs(a).max()


@pytest.mark.parametrize("Lb,n_el", [(L, 7), (1.0, 8)])   # beside the node by a rounding, and exactly on it
def test_charge_on_a_boundary_node(api, Lb, n_el):
    """Its boundary value is infinite or nearly so; the call returns and the engine stays usable."""
    import torch
    pos, Q = charges(40, False)
    pos = pos * (Lb / L)
    bad = pos.copy()
    bad[0] = 0.0
    eng = api.FEP3M(Lb, n_el, n_sr=3, precision="fp64", dirichlet=True)
    eng.set_boundary(g(eng.node_points()))
    eng.set_particles(torch.tensor(bad, device="cuda"), torch.tensor(Q, device="cuda"))
    eng.compute(forces=False, allow_noconv=True)
    eng.set_particles(torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda"))
    phi = eng.compute(forces=False)["phi"].cpu().numpy()
    ref = dirichlet.forward(pos, Q, Lb, n_el, g, n_sr=3)["phi"]
    assert np.abs(phi - ref).max() < 1e-11 * np.abs(ref).max()
