"""The hop with links and neighbours staged per 4D site, scalar and packed: slices that
divide a block, straddle blocks, the most an operator takes, and the smallest number that is staged;
every one bit-identical to the plain shape."""
import numpy as np
import pytest

from oracle import wilson
from synthetic import gauge_field, gaussian_spinor
from tests.layout import rel_l2
from tests.test_gpu_tune import _force

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BC = (-1.0, 1.0, 1.0, -1.0)
TOL = {1: 1e-5, 2: 3e-3}  # the hop's bars: rounding of FP32, of FP16 storage


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1512_03487_gb300 as L
    from paper_1512_03487_gb300 import fields
    L.fields = fields
    yield L
    L.lqcd_tune_clear()


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("recon", [12, 18])
@pytest.mark.parametrize("n5,dims", [(4, (2, 2, 2, 2)), (5, (6, 2, 2, 10)), (16, (4, 2, 4, 2)), (31, (2, 4, 2, 2)),
                                     (63, (2, 2, 2, 4)), (64, (2, 2, 4, 2))])
def test_staged_shapes_give_the_plain_hop(L, tmp_path, prec, recon, n5, dims):
    U, psi = gauge_field(dims, "haar", 2401), gaussian_spinor(dims, 2402, lead=(n5,))
    lat = L.lattice(dims, n5=n5, bc=BC)
    op = L.operator(mass=0.1, prec=prec, recon=recon)
    F = L.fields
    g = F.gauge_to_device(U, lat, prec, recon)
    fin = F.spinor_to_device(psi, lat, prec, L.LQCD_FULL)
    for dag in (0, 1):
        got = {}
        for shape in (0, 3, 4, 5):
            _force(L, tmp_path, dims, n5, shape)
            out = torch.zeros(L.lqcd_spinor_bytes(lat, prec, L.LQCD_FULL), dtype=torch.uint8, device="cuda")
            L.lqcd_dslash(out, fin, g, lat, op, L.LQCD_FULL, dag)
            got[shape] = out
        assert all(torch.equal(got[s], got[0]) for s in (3, 4, 5))
        assert rel_l2(F.spinor_to_host(got[4], lat, prec, L.LQCD_FULL), wilson.hop(U, psi, BC, dag)) <= TOL[prec]
