"""Restriction and coarse operator over the numbers of vectors and lattice sizes where
their work split changes: groups of four vectors, rows of 1 to 8 16-byte pieces per
lane and other lengths, aggregates that fill no block. The tolerances are those of
the full-size pieces: 1e-12 (FP64) and 2e-6 (FP32) of the largest element."""
import numpy as np
import pytest

from oracle import mg
from synthetic import gaussian_spinor, make_rng

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
TOL = {0: 1e-12, 1: 2e-6}
CT = {0: np.complex128, 1: np.complex64}


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1512_03487_gb300 as L
    from paper_1512_03487_gb300 import fields
    L.fields = fields
    return L


def _rel(a, b):
    return float(np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max())


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("b,dims", [(2, (4, 4, 4, 4)), (2, (6, 2, 4, 6)), (4, (4, 4, 4, 4)), (4, (12, 4, 4, 8))])
@pytest.mark.parametrize("nv", [1, 3, 4, 5, 9])
def test_restrict(L, prec, b, dims, nv):
    lat = L.lattice(dims)
    P = gaussian_spinor(dims, 2201, lead=(nv,))
    psi = gaussian_spinor(dims, 2202)
    Pd = torch.cat([L.fields.spinor_to_device(v, lat, prec, 2) for v in P])
    if prec == 1:
        P, psi = (f.astype(np.complex64).astype(np.complex128) for f in (P, psi))
    n = int(np.prod(mg.coarse_dims(dims, b))) * 2 * nv
    c = torch.full((n,), np.nan, dtype=torch.complex128 if prec == 0 else torch.complex64, device="cuda")
    L.lqcd_mg_restrict(c, L.fields.spinor_to_device(psi, lat, prec, 2), Pd, nv, b, prec, lat)
    assert _rel(c.cpu().numpy(), mg.restrict(P, psi, b).reshape(-1)) <= TOL[prec]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 2, 4)])
@pytest.mark.parametrize("nv", [1, 2, 3, 4, 5, 8, 12, 16, 20, 24, 31, 32])
@pytest.mark.parametrize("dagger", [0, 1])
def test_coarse_apply(L, prec, dims, nv, dagger):
    lat = L.lattice(dims)
    cd = tuple(d // 2 for d in dims)
    rng = make_rng(2211 + nv)
    Y = (rng.standard_normal((9,) + cd[::-1] + (2 * nv, 2 * nv, 2)) @ np.array([1.0, 1j])).astype(CT[prec])
    c = (rng.standard_normal(cd[::-1] + (2 * nv, 2)) @ np.array([1.0, 1j])).astype(CT[prec])
    out = torch.full((c.size,), np.nan, dtype=torch.complex128 if prec == 0 else torch.complex64, device="cuda")
    L.lqcd_mg_coarse_apply(out, torch.from_numpy(c).cuda(), torch.from_numpy(Y).cuda(), nv, 2, prec, dagger, lat)
    expect = mg.coarse_apply(Y.astype(np.complex128), c.astype(np.complex128), bool(dagger))
    assert _rel(out.cpu().numpy(), expect.reshape(-1)) <= TOL[prec]
