"""The order-q screen contraction by parity where its sizes differ: even and odd
numbers of screen nodes and of mesh nodes per axis (q = 2, 3, 4), the smallest and
the widest block, tiles and pieces of elements with remainders (q = 3 on 11^3
elements takes more than one piece), empty elements, and extreme units.

Tolerances: those of the order-q path (FP64 max|d| / max|ref| 1e-11, mixed relative
RMS 1e-6); powers of two of the charges scale the potentials to rounding.
"""
import numpy as np
import pytest

from oracle import highorder
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


def run(api, q, n_el, n_sr, support, precision, pos, Q):
    import torch
    eng = api.FEP3M(1.0, n_el, n_sr=n_sr, precision=precision, q=q, one_element=support == "element")
    eng.set_particles(torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda"))
    phi = eng.compute(forces=False)["phi"].cpu().numpy()
    eng.close()
    return phi


@pytest.mark.parametrize("q,n_el,n_sr,N,support", [
    (2, 3, 1, 4, "patch"), (2, 9, 4, 90, "patch"), (3, 5, 1, 60, "element"), (3, 11, 3, 200, "patch"),
    (4, 5, 2, 50, "patch")])
def test_matches_oracle(api, q, n_el, n_sr, N, support):
    pos, Q = workloads.uniform_pm(N, seed=21)
    ref = highorder.forward(pos, Q, 1.0, n_el, q, n_sr=n_sr, half_width=n_sr + 3, ngl=8, support=support)["phi"]
    phi = run(api, q, n_el, n_sr, support, "fp64", pos, Q)
    assert np.abs(phi - ref).max() < 1e-11 * np.abs(ref).max()
    phi = run(api, q, n_el, n_sr, support, "mixed", pos, Q)
    assert np.linalg.norm(phi - ref) < 1e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("unit", [2.0 ** -80, 2.0 ** 80])
def test_units(api, unit):
    pos, Q = workloads.uniform_pm(200, seed=22)
    a = run(api, 2, 7, 3, "patch", "fp64", pos, Q)
    b = run(api, 2, 7, 3, "patch", "fp64", pos, unit * Q) / unit
    assert np.abs(a - b).max() < 1e-12 * np.abs(a).max()
