"""The screen adjoint's persistent row GEMM (meshes of 54 elements per axis and more): forces
and their adjoint against the FP64 path, over the block half-widths (64 to 1000 offsets: a
part of a column tile, whole ones, a partial last one) and meshes with whole and partial
last row tiles.  Tolerance: the mixed path's 32-bit accuracy, 2e-5 of the largest.
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


@pytest.mark.parametrize("n_el,n_sr", [(54, 1), (55, 2), (56, 3), (57, 3), (55, 4)])
def test_forces_and_adjoint(api, n_el, n_sr):
    import torch
    pos, Q = workloads.uniform_pm(20000, seed=n_el + n_sr)
    p, q = torch.tensor(pos, device="cuda"), torch.tensor(Q, device="cuda")
    g = torch.randn(20000, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    got = []
    for precision in ("fp64", "mixed"):
        eng = api.FEP3M(1.0, n_el, n_sr=n_sr, precision=precision)
        eng.set_particles(p, q)
        F = eng.compute(forces=True)["forces"]
        got.append([F] + [t.clone() for t in eng.vjp(0.5, g)])
        eng.close()
    for a, b in zip(*got):
        assert float((a - b).abs().max()) < 2e-5 * float(a.abs().max())
