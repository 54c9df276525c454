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


@pytest.mark.parametrize("forces", [False, True])
@pytest.mark.parametrize("counts", [(1600,), (1537, 1545), (1700, 5, 11, 12, 13)])
def test_singular_sums_from_global_memory(api, counts, forces):
    """An element over the staging area: its bricks' blocks are read from global memory, element
    by element, eight (potentials: twelve) charges at a time.  Against the FP64 path, whose
    singular sums have a kernel of their own.

    Tolerance, per charge: the FP32 coordinates' rounding, 2^-24 of an element along each axis of
    a difference, through 1 / r (and 1 / r^2); 64 roundings of the sum of the terms' sizes, for
    their arithmetic and the sums; and the mixed path's 1e-6 (forces 1e-5) of the RMS.  A charge
    left out or taken twice is a hundred times that."""
    import torch
    elements, n = [73, 74, 0, 511, 200], 8   # neighbours, the corners (rows that wrap)
    groups = [(elements[i], 1, c) for i, c in enumerate(counts)] + [(0, 512, 60)]
    pos, Q = charges(n, groups, len(counts))
    p, q = torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda")
    out = {}
    for precision in ("fp64", "mixed"):
        eng = api.FEP3M(1.0, n, precision=precision)
        eng.set_particles(p, q)
        assert eng.stats()["max_per_element"] > 1536
        out[precision] = eng.compute(forces=forces)
        eng.close()
    r = p[:, None] - p
    r = (r - r.round()).norm(dim=2)
    r.fill_diagonal_(float("inf"))
    eps, shift = 2.0 ** -24, 3 ** 0.5 * 2.0 ** -24 / n
    terms = [(q.abs() / r ** k).sum(1) for k in (1, 2, 3)]
    ref = out["fp64"]["phi"]
    tol = shift * terms[1] + 64 * eps * terms[0] + 1e-6 * ref.square().mean().sqrt()
    assert bool(((out["mixed"]["phi"] - ref).abs() < tol).all())
    if forces:
        ref = out["fp64"]["forces"]
        tol = q.abs() * (2 * shift * terms[2] + 64 * eps * terms[1]) + 1e-5 * ref.square().mean().sqrt()
        assert bool(((out["mixed"]["forces"] - ref).abs() < tol[:, None]).all())
