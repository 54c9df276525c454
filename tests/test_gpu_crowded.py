"""Crowded elements: the adjoint's deposit on a small mesh (rows of 32 elements dealt to a CTA
each, the last one a partial one), and on a larger one with rows that hold just as many
charges as their warp takes in series, one more, and many more (dealt to the CTA's warps).

Tolerances: those of the steps, FP64 forces 1e-10 of the largest, mixed relative RMS 1e-5,
against the oracle.
"""
import numpy as np
import pytest

from oracle import fep3m as ofe

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_08509_gb300 import api as a, build
    build.build()
    return a


def charges(n_el, groups, seed):
    """groups: (first element, number of elements, charges) triples; neutral."""
    rng = np.random.default_rng(seed)
    e = np.concatenate([first + rng.integers(0, k, count) for first, k, count in groups])
    c = np.stack([e % n_el, (e // n_el) % n_el, e // n_el ** 2], 1)
    Q = np.where(np.arange(len(e)) % 2 == 0, 1.0, -1.0) * rng.uniform(0.5, 1.5, len(e))
    return (c + rng.uniform(0.02, 0.98, c.shape)) / n_el, Q - Q.mean()


def check(api, n_el, pos, Q):
    import torch
    ref = ofe.forward(pos, Q, 1.0, n_el, want_grad=True)
    want = -ofe.vjp(ref, Q)[0]
    for precision in ("fp64", "mixed"):
        eng = api.FEP3M(1.0, n_el, precision=precision)
        eng.set_particles(torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda"))
        F = eng.compute(forces=True)["forces"].cpu().numpy()
        eng.close()
        if precision == "fp64":
            assert np.abs(F - want).max() < 1e-10 * np.abs(want).max()
        else:
            assert np.linalg.norm(F - want) < 1e-5 * np.linalg.norm(want)


# 7^3 = 343 elements: ten whole rows of 32 and one of 23
@pytest.mark.parametrize("groups", [
    [(64, 32, 64), (0, 343, 6)], [(64, 1, 70), (100, 3, 200)], [(320, 23, 100), (0, 320, 40)],
    [(0, 343, 700)]])
def test_deposit_on_a_small_mesh(api, groups):
    check(api, 7, *charges(7, groups, len(groups) + groups[0][2]))


# 22^3 = 10648 elements: 332 whole rows and one of 24, in CTAs of eight rows but the last, of five
@pytest.mark.parametrize("groups", [
    [(64, 32, 160)], [(64, 32, 161)], [(10624, 24, 200), (0, 10624, 100)], [(96, 64, 330), (5000, 1, 40)],
    [(250, 12, 300)]])
def test_deposit_of_crowded_rows(api, groups):
    check(api, 22, *charges(22, groups, len(groups) + groups[0][2]))
