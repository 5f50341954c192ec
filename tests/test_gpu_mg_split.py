"""Restriction and coarse operator on both sides of the sizes where their work is split
otherwise: all vectors of an aggregate in a block, or some; four lanes or a warp per coarse
row. The tolerances are those of the full-size pieces: 1e-12 (FP64) and 2e-6 (FP32) of the
largest element."""
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


def _device(prec):
    return torch.complex128 if prec == 0 else torch.complex64


# 192 blocks of aggregates (all vectors in a block), 81 and 16 (a few), 1 (one each)
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("b,dims,nv", [(4, (16, 16, 16, 12), 3), (4, (16, 16, 16, 12), 9), (2, (16, 16, 16, 12), 5),
                                       (4, (12, 12, 12, 12), 9), (4, (8, 8, 8, 8), 24), (2, (8, 8, 8, 8), 13),
                                       (2, (4, 4, 4, 4), 24)])
def test_restrict(L, prec, b, dims, nv):
    lat = L.lattice(dims)
    P, psi = gaussian_spinor(dims, 3001, lead=(nv,)), gaussian_spinor(dims, 3002)
    Pd = torch.cat([L.fields.spinor_to_device(v, lat, prec, 2) for v in P])
    if prec == 1:
        P, psi = (f.astype(np.complex64).astype(np.complex128) for f in (P, psi))
    n = int(np.prod(mg.coarse_dims(dims, b))) * 2 * nv
    c = torch.full((n,), np.nan, dtype=_device(prec), device="cuda")
    L.lqcd_mg_restrict(c, L.fields.spinor_to_device(psi, lat, prec, 2), Pd, nv, b, prec, lat)
    assert _rel(c.cpu().numpy(), mg.restrict(P, psi, b).reshape(-1)) <= TOL[prec]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nv", [1, 2, 3, 4, 5, 7, 8, 9, 12, 15, 16, 20, 24, 31, 32])
def test_coarse_apply(L, prec, nv):
    """4,096 rows and more; fewer are in the other tests."""
    dims = (16, 16, 8, 8) if nv < 16 else (8, 8, 8, 4)
    lat, cd, rng = L.lattice(dims), tuple(d // 2 for d in dims), make_rng(3011 + nv)
    Y = (rng.standard_normal((9,) + cd[::-1] + (2 * nv, 2 * nv, 2)) @ np.array([1.0, 1j])).astype(CT[prec])
    c = (rng.standard_normal(cd[::-1] + (2 * nv, 2)) @ np.array([1.0, 1j])).astype(CT[prec])
    out = torch.full((c.size,), np.nan, dtype=_device(prec), device="cuda")
    L.lqcd_mg_coarse_apply(out, torch.from_numpy(c).cuda(), torch.from_numpy(Y).cuda(), nv, 2, prec, 0, lat)
    expect = mg.coarse_apply(Y.astype(np.complex128), c.astype(np.complex128))
    assert _rel(out.cpu().numpy(), expect.reshape(-1)) <= TOL[prec]


def test_small_set_ups_are_spread_over_the_chip(L):
    """24 FP64 vectors on 16 aggregates of 4^4: with all vectors of an aggregate in one block the restriction
    took 18 times as long as that of one vector, and the coarse operator on 16 sites 3 times as long as its
    adjoint, which has a warp per row."""
    dims, nv, lat = (8, 8, 8, 8), 24, L.lattice((8, 8, 8, 8))
    vecs = torch.zeros(nv * L.lqcd_spinor_bytes(lat, 0, 2), dtype=torch.uint8, device="cuda")
    psi = torch.zeros(L.lqcd_spinor_bytes(lat, 0, 2), dtype=torch.uint8, device="cuda")
    c, d = (torch.zeros(16 * 2 * nv, dtype=torch.complex128, device="cuda") for _ in range(2))
    Y = torch.zeros(9 * 16 * 4 * nv * nv, dtype=torch.complex128, device="cuda")

    def us(f):
        f()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for _ in range(20):
                f()
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = 1e9
        for _ in range(6):
            start.record()
            graph.replay()
            end.record()
            end.synchronize()
            best = min(best, start.elapsed_time(end))
        return best * 50

    one = us(lambda: L.lqcd_mg_restrict(c, psi, vecs, 1, 4, 0, lat))
    assert us(lambda: L.lqcd_mg_restrict(c, psi, vecs, nv, 4, 0, lat)) <= 6 * one
    dag = us(lambda: L.lqcd_mg_coarse_apply(d, c, Y, nv, 4, 0, 1, lat))
    assert us(lambda: L.lqcd_mg_coarse_apply(d, c, Y, nv, 4, 0, 0, lat)) <= 1.5 * dag
