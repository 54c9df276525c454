"""The replayed mixed solve's last residual from the correction alone (two sweeps, a
tolerance of 1e-11 and more): the residual reported against the returned solution's,
computed in FP64, and a step's numbers against those of a tolerance that forms the
residual of the new iterate (the same two sweeps, so the same bits).

The reported residual differs from the solution's by the FP32 rounding of K e, at most of
the size of what the FP32 inner solve leaves of the residual and independent of it: within
a factor sqrt(2), 1.5 allowed.
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


def axis_matrices(n):
    """Periodic order-3 mass and stiffness matrices of n elements on [0, 1]."""
    import torch
    N = 3 * n
    Me = torch.tensor([[128, 99, -36, 19], [99, 648, -81, -36], [-36, -81, 648, 99], [19, -36, 99, 128]],
                      dtype=torch.float64) / 1680 / n
    Ke = torch.tensor([[148, -189, 54, -13], [-189, 432, -297, 54], [54, -297, 432, -189], [-13, 54, -189, 148]],
                      dtype=torch.float64) / 40 * n
    M, K = torch.zeros(N, N, dtype=torch.float64), torch.zeros(N, N, dtype=torch.float64)
    for e in range(n):
        ix = torch.tensor([(3 * e + i) % N for i in range(4)])
        M[ix[:, None], ix[None]] += Me
        K[ix[:, None], ix[None]] += Ke
    return M.cuda(), K.cuda()


def stiffness(M, K, x):
    import torch

    def along(A, t, d):
        return torch.movedim(torch.tensordot(A, t, dims=([1], [d])), 0, d)
    mx, kx = along(M, x, 2), along(K, x, 2)
    return along(M, along(M, kx, 1) + along(K, mx, 1), 0) + along(K, along(M, mx, 1), 0)


@pytest.mark.parametrize("n_el", [7, 8, 17, 33, 54, 55])
def test_reported_residual(api, n_el):
    import torch
    N = 3 * n_el
    b = torch.randn((N, N, N), dtype=torch.float64, device="cuda",
                    generator=torch.Generator("cuda").manual_seed(n_el))
    w = torch.where(torch.arange(N, device="cuda") % 3 == 0, 0.25, 0.375).double()
    w3 = w[:, None, None] * w[None, :, None] * w[None, None, :]
    b -= b.sum() / w3.sum() * w3     # no constant component: the solver removes it along w3
    eng = api.FEP3M(1.0, n_el, precision="mixed")
    for _ in range(2):   # the checked solve, then its replay
        phi = eng.solve_mesh(b.reshape(-1)).reshape(N, N, N)
    st = eng.stats()
    eng.close()
    M, K = axis_matrices(n_el)
    true = float((b - stiffness(M, K, phi)).norm() / b.norm())
    assert st["refine_steps"] == 2
    assert true / 1.5 < st["mg_rel_residual"] < true * 1.5


@pytest.mark.parametrize("n_el", [7, 8, 17])
def test_step_is_unchanged(api, n_el):
    import torch
    pos, Q = workloads.uniform_pm(40 * n_el, seed=n_el)
    p, q = torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda")
    got = []
    for rtol in (1e-10, 9e-12):
        eng = api.FEP3M(1.0, n_el, precision="mixed", mg_rtol=rtol)
        for _ in range(2):
            eng.set_particles(p, q)
            out = eng.compute(forces=True)
        st = eng.stats()
        eng.close()
        assert st["refine_steps"] == 2
        got.append((out["phi"], out["forces"], st))
    (a, b) = got
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    for key in ("mg_rel_residual", "adj_rel_residual"):
        assert b[2][key] / 1.5 < a[2][key] < b[2][key] * 1.5
