"""Packing and unpacking at the edges: values outside the normal range of the stored
type, ties, zeros, infinities and NaN round as numpy rounds them; host-layout
buffers that are only 8-byte aligned; ragged and tiny lattices; several slices."""
import numpy as np
import pytest

from synthetic import gauge_field, gaussian_spinor, make_rng
from tests.layout import to_cb

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
NP = {0: np.float64, 1: np.float32, 2: np.float16}


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1512_03487_gb300 as L
    from paper_1512_03487_gb300 import fields
    L.fields = fields
    return L


def _edge_values(n):
    """Values around the limits of float and half, ties of either, and ordinary ones."""
    v = [0.0, -0.0, 1.0, -1.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, 1e-45, 7e-46, 1.17549435e-38, 1.1754943e-38,
         2.0 ** -126, 2.0 ** -127, 3.4028234e38, 3.4028235677973366e38, 3.5e38, 1e300, 65504.0, 65519.99, 65520.0, 7e4,
         6.1e-5, 2.0 ** -14, 2.0 ** -15, 2.0 ** -24, 2.0 ** -25, 2.0 ** -26, 1e-8]
    for e in (-20, -3, 0, 5, 12):  # ties and their neighbours for 23 and 10 mantissa bits
        for k in (23, 10):
            for odd in (0, 1):
                x = 2.0 ** e * (1.0 + (odd + 0.5) * 2.0 ** -k)
                v += [x, np.nextafter(x, 0.0), np.nextafter(x, 1e9), -x]
        v += [2.0 ** e * (2.0 - 2.0 ** -24), 2.0 ** e * (2.0 - 2.0 ** -12)]
    v = np.array(v)
    return np.where(np.arange(n) % 3 < 2, np.resize(v, n), make_rng(1901).standard_normal(n))


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("offset", [0, 1])
def test_links_round_as_numpy(L, prec, recon, offset):
    dims = (4, 2, 6, 2)
    lat = L.lattice(dims)
    n = 4 * int(np.prod(dims)) * 18
    vals = _edge_values(n)
    src = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    src[offset:offset + n] = torch.from_numpy(vals).cuda()
    dst = torch.full((L.lqcd_gauge_bytes(lat, prec, recon),), 0xff, dtype=torch.uint8, device="cuda")
    L.lqcd_gauge_pack(dst, prec, recon, src[offset:], lat)
    back = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    L.lqcd_gauge_unpack(back[offset:], dst, prec, recon, lat)
    with np.errstate(over="ignore"):
        expect = vals.astype(NP[prec]).astype(np.float64).reshape(-1, 18)
    got = back[offset:offset + n].cpu().numpy().reshape(-1, 18)[:, :recon]  # the third row is rebuilt from the others
    expect = expect[:, :recon]
    np.testing.assert_array_equal(got, expect)
    np.testing.assert_array_equal(np.signbit(got[~np.isnan(got)]), np.signbit(expect[~np.isnan(expect)]))


@pytest.mark.parametrize("subset", [0, 1, 2])
@pytest.mark.parametrize("n5,dims", [(1, (4, 2, 6, 2)), (3, (2, 2, 2, 6)), (7, (6, 2, 2, 2)), (40, (2, 2, 4, 2))])
@pytest.mark.parametrize("offset", [0, 1])
def test_spinors_round_as_numpy(L, subset, n5, dims, offset):
    lat = L.lattice(dims, n5=n5)
    shape = L.fields.host_spinor_shape(lat, subset)
    n = 2 * int(np.prod(shape))
    vals = _edge_values(n)
    for prec in (0, 1):
        src = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
        src[offset:offset + n] = torch.from_numpy(vals).cuda()
        dst = torch.full((L.lqcd_spinor_bytes(lat, prec, subset),), 0xff, dtype=torch.uint8, device="cuda")
        L.lqcd_spinor_pack(dst, prec, subset, src[offset:], lat)
        back = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
        L.lqcd_spinor_unpack(back[offset:], dst, prec, subset, lat)
        with np.errstate(over="ignore"):
            expect = vals.astype(NP[prec]).astype(np.float64)
        np.testing.assert_array_equal(back[offset:offset + n].cpu().numpy(), expect)
    # FP16: site norm times halves, 2^-11 of the largest component of the site
    psi = gaussian_spinor(dims, 1902, lead=(n5,))
    psi = psi if subset == 2 else to_cb(psi, subset)
    back = L.fields.spinor_to_host(L.fields.spinor_to_device(psi, lat, 2, subset), lat, 2, subset)
    psi = psi.reshape(back.shape)
    top = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(axis=(-1, -2), keepdims=True)
    assert np.max(np.maximum(np.abs((back - psi).real), np.abs((back - psi).imag)) / top) <= 2.0 ** -11


@pytest.mark.parametrize("n5,recon", [(1, 18), (3, 18), (12, 12)])
def test_double_float_hop_with_several_slices(L, n5, recon):
    """The double-float hop's shared-memory columns with 4D sites straddling blocks:
    1e-12 of the oracle, as for one slice."""
    from oracle import wilson
    from tests.layout import rel_l2
    bc = (1.0, 1.0, 1.0, -1.0)
    dims = (6, 2, 6, 10)
    U, psi = gauge_field(dims, "haar", 1911), gaussian_spinor(dims, 1912, lead=(n5,))
    lat = L.lattice(dims, n5=n5, bc=bc)
    g = L.fields.gauge_to_device(U, lat, 0, recon)
    fin = L.fields.spinor_to_device(psi, lat, 0, 2)
    for dag in (0, 1):
        out = L.fields.empty(L.lqcd_spinor_bytes(lat, 0, 2))
        L.lqcd_dslash(out, fin, g, lat, L.operator(prec=L.LQCD_F64_DF, recon=recon), 2, dag)
        assert rel_l2(L.fields.spinor_to_host(out, lat, 0, 2), wilson.hop(U, psi, bc, dag)) <= 1e-12
