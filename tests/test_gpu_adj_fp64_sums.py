"""FP64 contexts: the screen adjoint's sums over a block keep FP64's accuracy where the
weights are of one sign, so that up to (2 n_sr)^3 terms add up to many times each of them
(both kernels' splits: one thread per vertex from 40 elements on, eight below).

The gradient is linear in the weights: those of one sign, 1.5 plus signed ones, against
the sum of their two parts' gradients, of which the signed part's sums stay small and the
constant part's, the same at every charge of a lattice, differ from them in rounding.
Tolerance: the sum of |w| / r over a block, over h^2 (its gradient's scale before the
corners of an element cancel), times 2^-48, the rounding of a single term, times 8 for
their number and the shape functions' slopes.
"""
import itertools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_08509_gb300 import api as a, build
    build.build()
    return a


@pytest.mark.parametrize("n_el,n_sr", [(10, 4), (12, 3), (40, 4), (40, 3), (40, 1)])
def test_weights_of_one_sign(api, n_el, n_sr):
    import torch
    i = np.arange(n_el ** 3)
    c = np.stack([i % n_el, (i // n_el) % n_el, i // n_el ** 2], 1)
    pos, Q = (c + np.array([0.3, 0.45, 0.6])) / n_el, np.where(c.sum(1) % 2 == 0, 1.0, -1.0)
    r = torch.rand(n_el ** 3, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(5)) - 0.5
    flat = torch.full_like(r, 1.5)
    eng = api.FEP3M(1.0, n_el, n_sr=n_sr, precision="fp64", mg_rtol=1e-15)
    eng.set_particles(torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda"))
    eng.compute(forces=False, allow_noconv=True)
    got = [[t.clone() for t in eng.vjp(0.0, g)] for g in (flat + r, flat, r)]
    eng.close()
    block = sum(1.0 / np.sqrt(x * x + y * y + z * z)
                for x, y, z in itertools.product(range(-n_sr, n_sr + 1), repeat=3) if (x, y, z) != (0, 0, 0))
    tol = 8 * 2.0 ** -48 * 2.0 * block * n_el ** 2
    worst = float((got[0][0] - got[1][0] - got[2][0]).abs().max())
    assert worst < tol, (worst, tol)
