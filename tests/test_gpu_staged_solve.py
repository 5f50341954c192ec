"""Solves with every in-iteration hop forced to a staged launch shape (links and neighbours
of a 4D site shared by its n5 threads): the norm-reducing hop and the fused update over
several systems, 4D sites that straddle blocks, a partial last block, FP32 and FP16, and
domain wall. The hop's bits are those of the plain shape, and so is the grouping of the
partial sums (128 sites per block), so the solve is the same to the last bit."""
import numpy as np
import pytest

from oracle import dwf, wilson
from synthetic import gauge_field, gaussian_spinor
from tests.test_gpu_tune import _force

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BC = (1.0, 1.0, 1.0, -1.0)


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1512_03487_gb300 as L
    from paper_1512_03487_gb300 import fields
    L.fields = fields
    yield L
    L.lqcd_tune_clear()
    L.lqcd_release_caches()


def _solves(L, tmp_path, dims, n5, op, sloppy, seed, graph):
    F, lat = L.fields, L.lattice(dims, n5=n5, bc=BC)
    U, b = gauge_field(dims, "haar", seed), gaussian_spinor(dims, seed + 1, lead=(n5,))
    g64, gs = F.gauge_to_device(U, lat, 0, 18), F.gauge_to_device(U, lat, sloppy, 12)
    bd = F.spinor_to_device(b, lat, 0, L.LQCD_FULL)
    prm = L.solver_params(tol=1e-10, maxiter=2000, sloppy_prec=sloppy, sloppy_recon=12, delta=1e-3 if sloppy == 1 else 1e-4,
                          delta_mid=0.01 if sloppy == 2 else 0.0, use_graph=graph)
    ws = F.empty(L.lqcd_eo_solve_workspace_bytes(lat, op, prm))
    seen = {}
    for shape in (0, 4, 5, 9):
        _force(L, tmp_path, dims, n5, shape)
        L.lqcd_release_caches()  # graphs captured under another shape
        x = torch.zeros(L.lqcd_spinor_bytes(lat, 0, L.LQCD_FULL), dtype=torch.uint8, device="cuda")
        info = L.lqcd_eo_solve(x, bd, g64, gs, lat, op, prm, ws)
        seen[shape] = (info.iterations, info.reliable_updates, info.residual_replacements, x)
    for shape in (4, 5, 9):
        assert seen[shape][:3] == seen[0][:3], shape
        assert torch.equal(seen[shape][3], seen[0][3]), shape
    return U, b, F.spinor_to_host(seen[4][3], lat, 0, L.LQCD_FULL)


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("sloppy", [1, 2])
@pytest.mark.parametrize("n5,dims", [(4, (4, 4, 4, 4)), (5, (6, 2, 6, 10)), (12, (6, 2, 2, 10))])
def test_staged_shapes_give_the_plain_multi_rhs_solve(L, tmp_path, n5, dims, sloppy, graph):
    m = 0.1
    U, b, x = _solves(L, tmp_path, dims, n5, L.operator(mass=m), sloppy, 2701, graph)
    for k in range(n5):
        r = b[k:k + 1] - wilson.dirac(U, x[k:k + 1], m, BC)
        assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(b[k]), k


@pytest.mark.parametrize("sloppy", [1, 2])
@pytest.mark.parametrize("Ls,dims", [(4, (4, 2, 6, 10)), (8, (2, 4, 6, 2)), (6, (4, 2, 2, 6))])
def test_staged_shapes_give_the_plain_domain_wall_solve(L, tmp_path, Ls, dims, sloppy):
    M5, mf = 1.8, 0.05
    op = L.operator(kind=L.LQCD_DWF, M5=M5, mf=mf)
    U, b, x = _solves(L, tmp_path, dims, Ls, op, sloppy, 2711, 1)
    r = b - dwf.dirac(U, x, M5, mf, BC)
    assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(b)
