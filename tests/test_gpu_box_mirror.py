"""FP64 boxes: what a charge's screens add at the boundary is the field that is subtracted at
the charges, one table, symmetric under reflection.

A single charge and its mirror image (coordinates exact in binary): the Dirichlet box's
boundary values are the same terms in another order.  Those on the planes between elements
are left out, as a node there belongs to the block of one of the two.  Tolerance: the terms'
sum (1 / r, below 4, and the screens', less) times 2^-52.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N_EL = 8   # h = 1/8: exact


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_08509_gb300 import api as a, build
    build.build()
    return a


def images(x):
    yield x, None
    for a in range(3):
        y = x.copy()
        y[:, a] = 1.0 - y[:, a]
        yield y, a


@pytest.mark.parametrize("at", [(1.3125, 2.25, 3.6875), (0.375, 0.5, 4.0625), (7.625, 6.75, 2.5)])
def test_dirichlet_values_of_a_mirrored_charge(api, at):
    import torch
    m = 3 * N_EL + 1
    k = np.arange(m)
    face, plane = ((k == 0) | (k == m - 1)).astype(int), (k % 3 == 0).astype(int)

    def count(f):
        return f[:, None, None] + f[:, None] + f

    inner = (count(face) == 1) & (count(plane) == 1)
    want = None
    for x, a in images(np.array([at]) / N_EL):
        eng = api.FEP3M(1.0, N_EL, n_sr=3, precision="fp64", dirichlet=True)
        eng.set_particles(torch.tensor(x, device="cuda"), torch.ones(1, dtype=torch.float64, device="cuda"))
        eng.compute(forces=False)
        v = eng.mesh()["phi_mesh"].reshape(m, m, m) / N_EL   # element units, [z, y, x]
        eng.close()
        if a is None:
            want = v[inner]
        else:
            worst = np.abs(np.flip(v, 2 - a)[inner] - want).max()
            assert worst <= 8 * 2.0 ** -52, worst
