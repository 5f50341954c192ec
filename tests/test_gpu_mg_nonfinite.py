"""Values that are not finite, and sums beyond FP32's range, in the FP32 restriction and
coarse operator: what the same FP32 terms summed in FP64 and rounded once give."""
import numpy as np
import pytest

from oracle import mg
from synthetic import gaussian_spinor, make_rng

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1512_03487_gb300 as L
    from paper_1512_03487_gb300 import fields
    L.fields = fields
    return L


def _f32(a):
    return a.astype(np.complex64).astype(np.complex128)


def _same(got, re, im):
    """The kinds (finite, +inf, -inf, NaN) agree, and finite values to 2e-6 of the largest."""
    for g, e in ((got.real, re), (got.imag, im)):
        np.testing.assert_array_equal(np.isnan(g), np.isnan(e))
        np.testing.assert_array_equal(np.isposinf(g), np.isposinf(e))
        np.testing.assert_array_equal(np.isneginf(g), np.isneginf(e))
        f = np.isfinite(e)
        assert np.abs(g[f] - e[f]).max() <= 2e-6 * np.abs(e[f]).max()


@pytest.mark.parametrize("b,dims", [(2, (4, 2, 2, 4)), (4, (8, 4, 4, 4))])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_restrict_carries_values_that_are_not_finite(L, b, dims, value):
    """One such number in one aggregate and chirality; every other coarse value stays as it was."""
    nv, lat = 5, L.lattice(dims)
    P, psi = _f32(gaussian_spinor(dims, 2501, lead=(nv,))), _f32(gaussian_spinor(dims, 2502))
    psi.reshape(-1, 4, 3)[3, 1, 2] = value + 0.5j
    c = torch.zeros(int(np.prod(mg.coarse_dims(dims, b))) * 2 * nv, dtype=torch.complex64, device="cuda")
    dev = [L.fields.spinor_to_device(f, lat, 1, 2) for f in (psi, *P)]
    L.lqcd_mg_restrict(c, dev[0], torch.cat(dev[1:]), nv, b, 1, lat)

    def part(p, s):  # of real fields, so that no 0 times infinity arises that the kernel does not form
        return mg.restrict(p, s, b).real.reshape(-1)

    _same(c.cpu().numpy(), part(P.real, psi.real) + part(P.imag, psi.imag),
          part(P.real, psi.imag) - part(P.imag, psi.real))


@pytest.mark.parametrize("b", [2, 4])
@pytest.mark.parametrize("axis", [0, 1, 2, 3])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_restrict_partial_sums_beyond_the_range(L, b, axis, sign):
    """Terms +3e38 on half of an aggregate's sites and -3e38 on the others, and one
    of them 1e37 larger: the sum is finite, its parts are not in FP32."""
    dims, lat = (b,) * 4, L.lattice((b,) * 4)
    P, psi = np.zeros((1,) + dims + (4, 3), complex), np.zeros(dims + (4, 3), complex)
    upper = np.indices(dims)[axis] < b // 2
    big, more = float(np.float32(3e38)), float(np.float32(1e37))
    P[0, ..., 0, 0], psi[..., 0, 0] = 1.0, sign * np.where(upper, big, -big)
    P[0, 0, 0, 0, 0, 1, 1], psi[0, 0, 0, 0, 1, 1] = 1.0, sign * more
    c = torch.zeros(2, dtype=torch.complex64, device="cuda")
    L.lqcd_mg_restrict(c, L.fields.spinor_to_device(psi, lat, 1, 2), L.fields.spinor_to_device(P[0], lat, 1, 2), 1, b,
                       1, lat)
    got = c.cpu().numpy()
    # the one term is rounded to FP32 in the kernel; everything else is exact
    assert got[0].real == np.float32(sign * (float(np.float32(big + more)) - big))
    assert got[0].imag == 0 and got[1] == 0


@pytest.mark.parametrize("nv,dims", [(1, (8, 4, 2, 4)), (2, (8, 4, 2, 4)), (12, (8, 4, 2, 4)),  # a warp per row
                                     (3, (16, 16, 8, 8)), (4, (16, 16, 8, 8)), (12, (8, 8, 8, 6)), (28, (8, 8, 8, 4))])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_coarse_apply_carries_values_that_are_not_finite(L, nv, dims, value):
    lat, cd, rng = L.lattice(dims), tuple(d // 2 for d in dims), make_rng(2511 + nv)
    Y = _f32(rng.standard_normal((9,) + cd[::-1] + (2 * nv, 2 * nv, 2)) @ np.array([1.0, 1j]))
    c = _f32(rng.standard_normal(cd[::-1] + (2 * nv, 2)) @ np.array([1.0, 1j]))
    c.reshape(-1)[2 * nv + 1] = value - 0.25j
    out = torch.zeros(c.size, dtype=torch.complex64, device="cuda")
    dev = [torch.from_numpy(a.astype(np.complex64)).cuda() for a in (c, Y)]
    L.lqcd_mg_coarse_apply(out, dev[0], dev[1], nv, 2, 1, 0, lat)

    def part(y, v):
        return mg.coarse_apply(y, v).reshape(-1)

    with np.errstate(invalid="ignore"):
        _same(out.cpu().numpy(), part(Y.real, c.real) - part(Y.imag, c.imag),
              part(Y.real, c.imag) + part(Y.imag, c.real))


@pytest.mark.parametrize("nv,dims", [(1, (2, 2, 2, 2)), (3, (16, 16, 8, 8))])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_coarse_apply_sums_beyond_the_range(L, nv, dims, sign):
    """Nine blocks of products 5e37 each: the sum leaves FP32's range, with its sign."""
    lat, sites, nc = L.lattice(dims), int(np.prod(dims)) // 16, 2 * nv
    c = torch.full((sites * nc,), sign * 5e37, dtype=torch.complex64, device="cuda")
    Y = torch.ones(9 * sites * nc * nc, dtype=torch.complex64, device="cuda")
    out = torch.zeros(sites * nc, dtype=torch.complex64, device="cuda")
    L.lqcd_mg_coarse_apply(out, c, Y, nv, 2, 1, 0, lat)
    assert (out.cpu().numpy().real == sign * np.inf).all()
