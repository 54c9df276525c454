"""FP64 contexts: a large level of the field over an element (charges of one sign) does not
enter the forces' rounding.

A lattice of equal charges at the element centres, neutralised: every force is zero by
symmetry, and what is computed is rounding.  The screens of a block add up to a level of
sum 1 / r over the block's elements (element units) in each nodal value; the nodal values
are held relative to one of them, so the slopes of the shape functions (up to 5.5, ten per
node row) act on the variation alone.  Tolerance: twice the level's own rounding, 2^-53.
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


@pytest.mark.parametrize("n_el", [8, 16])
def test_forces_of_a_lattice_of_one_sign(api, n_el):
    import torch
    i = np.arange(n_el ** 3)
    pos = (np.stack([i % n_el, (i // n_el) % n_el, i // n_el ** 2], 1) + 0.5) / n_el
    eng = api.FEP3M(1.0, n_el, n_sr=3, precision="fp64", neutralize=True)
    eng.set_particles(torch.tensor(pos, device="cuda"), torch.ones(n_el ** 3, dtype=torch.float64, device="cuda"))
    out = eng.compute(forces=True, allow_noconv=True)   # (the load is zero to rounding: no residual to reduce)
    eng.close()
    level = sum(1.0 / np.sqrt(x * x + y * y + z * z) for x, y, z in itertools.product(range(-3, 4), repeat=3) if (x, y, z) != (0, 0, 0))
    worst = float(out["forces"].abs().max()) / n_el ** 2
    assert worst < 2 * 2.0 ** -53 * level, worst
