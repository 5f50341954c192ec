"""Gauge force, fermion force, plaquette and link update at the edges of their work split: lattices
that fill a fraction of a block, one block and a ragged last block, momenta on
either side of the exponential's degree and scaling thresholds, and matrices
that are not Hermitian."""
import numpy as np
import pytest

from oracle import force as oforce
from oracle import gauge as og
from synthetic import gauge_field, gaussian_spinor, make_rng, random_su3_algebra
from tests.layout import rel_l2

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


def _rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


# sums of at most some hundred products of entries below 1: 1e-13 is about 500 roundings
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 2, 2, 4), (4, 2, 2, 6), (6, 2, 10, 2)])
def test_gauge_force_and_plaquette_on_ragged_blocks(L, dims):
    F = L.fields
    lat = L.lattice(dims)
    U = gauge_field(dims, "haar", 1801)
    U *= 1.0 + 0.1 * make_rng(1802).standard_normal(U.shape)  # the formulas hold for any matrices
    Ud = F.gauge_to_device(U, lat, 0, 18)
    out = torch.full((L.lqcd_gauge_bytes(lat, 0, 18),), 0xff, dtype=torch.uint8, device="cuda")
    L.lqcd_gauge_force(out, Ud, lat, 5.6)
    assert _rel(F.gauge_to_host(out, lat, 0, 18), og.force(U, 5.6)) <= 1e-13
    ws = F.empty(L.lqcd_reduce_workspace_bytes(lat))
    assert L.lqcd_plaquette(Ud, lat, ws) == pytest.approx(og.mean_plaquette(U), rel=1e-13, abs=1e-14)


# |A|_F against the thresholds 1/4 (degree 13 or 20) and 1 (halvings); at 6 there
# are three squarings, each doubling some tens of roundings: below 1e-13
@pytest.mark.parametrize("norm", [0.0, 0.2499, 0.2501, 0.9999, 1.0001, 6.0])
@pytest.mark.parametrize("hermitian", [True, False])
def test_link_update_around_its_thresholds(L, norm, hermitian):
    from scipy.linalg import expm
    F = L.fields
    dims = (4, 2, 2, 2)
    lat = L.lattice(dims)
    U = gauge_field(dims, "haar", 1811)
    n = U.size // 9
    rng = make_rng(1812)
    P = random_su3_algebra(rng, n) if hermitian else rng.standard_normal((n, 3, 3)) + 1j * rng.standard_normal((n, 3, 3))
    P *= (norm / 0.5 / np.linalg.norm(P, axis=(1, 2)))[:, None, None]
    expect = np.einsum("nij,njk->nik", np.stack([expm(0.5j * p) for p in P]), U.reshape(n, 3, 3)).reshape(U.shape)
    Ud = F.gauge_to_device(U, lat, 0, 18)
    L.lqcd_gauge_exp_update(Ud, F.gauge_to_device(P.reshape(U.shape), lat, 0, 18), 0.5, lat)
    assert _rel(F.gauge_to_host(Ud, lat, 0, 18), expect) <= 1e-13


# Links side by side with a Hermitian P (one triangle used), one that is so only up to its
# last bits and any matrix: the same tolerance as above for each. A NaN or an asymmetry that
# stands in the lower triangle alone counts.
@pytest.mark.parametrize("norm", [0.2, 0.9, 3.0])
def test_link_update_of_hermitian_and_general_momenta_side_by_side(L, norm):
    from scipy.linalg import expm
    F = L.fields
    dims = (2, 4, 2, 6)
    lat = L.lattice(dims)
    U = gauge_field(dims, "haar", 1821)
    n = U.size // 9
    rng = make_rng(1822)
    P = rng.standard_normal((n, 3, 3)) + 1j * rng.standard_normal((n, 3, 3))
    P *= (norm / 0.5 / np.linalg.norm(P, axis=(1, 2)))[:, None, None]
    kind = rng.integers(0, 3, n)
    herm = 0.5 * (P + P.conj().transpose(0, 2, 1))
    P = np.where((kind < 2)[:, None, None], herm, P)
    P[kind == 1, 2, 0] *= 1.0 + 4e-16
    expect = np.einsum("nij,njk->nik", np.stack([expm(0.5j * p) for p in P]), U.reshape(n, 3, 3))
    bad = np.flatnonzero(kind == 0)[:2]
    P[bad[0], 2, 1] = np.nan
    P[bad[1], 1, 1] += 1e-3j
    expect[bad[1]] = expm(0.5j * P[bad[1]]) @ U.reshape(n, 3, 3)[bad[1]]
    Ud = F.gauge_to_device(U, lat, 0, 18)
    L.lqcd_gauge_exp_update(Ud, F.gauge_to_device(P.reshape(U.shape), lat, 0, 18), 0.5, lat)
    got = F.gauge_to_host(Ud, lat, 0, 18).reshape(n, 3, 3)
    assert np.isnan(got[bad[0]]).all()
    keep = np.arange(n) != bad[0]
    assert _rel(got[keep], expect[keep]) <= 1e-13


# sums of at most a hundred products, as in the oracle: 1e-12 as for the full lattices
@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 2, 2, 2), (2, 6, 2, 6)])
def test_fermion_force_on_ragged_blocks(L, dims, recon):
    F = L.fields
    bc = (1.0, -1.0, 1.0, -1.0)
    U, X, Y = gauge_field(dims, "haar", 1821), gaussian_spinor(dims, 1822), gaussian_spinor(dims, 1823)
    lat = L.lattice(dims, bc=bc)
    op = L.operator(mass=0.05, recon=recon)
    g = F.gauge_to_device(U, lat, 0, recon)
    Xd, Yd = (F.spinor_to_device(f[None], lat, 0, 2) for f in (X, Y))
    grad, ta = oforce.force_terms(U, X, Y, bc)
    for kind, ref in ((L.LQCD_FORCE_TA, ta), (L.LQCD_FORCE_GRAD, grad)):
        out = torch.full((L.lqcd_gauge_bytes(lat, 0, 18),), 0xff, dtype=torch.uint8, device="cuda")
        L.lqcd_force(out, g, Xd, Yd, lat, op, kind)
        assert rel_l2(F.gauge_to_host(out, lat, 0, 18), ref) <= 1e-12
