"""How many iterations a body of the solver's graph holds: launches that return at once
behind a requested update stay few, whatever the distance between updates and the size.
One iteration per body (check_interval 1) launches none of them."""
import pytest

from synthetic import gauge_field, gaussian_spinor

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
    return L


def _launches(L, lat, op, b, g64, gs, check, **kw):
    prm = L.solver_params(tol=1e-10, maxiter=500, sloppy_recon=12, check_interval=check, **kw)
    ws = L.fields.empty(L.lqcd_eo_solve_workspace_bytes(lat, op, prm))
    x = torch.zeros_like(b)
    L.lqcd_eo_solve(x, b, g64, gs, lat, op, prm, ws)  # launch shapes are timed here
    before = L.lqcd_launch_count()
    info = L.lqcd_eo_solve(x, b, g64, gs, lat, op, prm, ws)
    return L.lqcd_launch_count() - before, info


@pytest.mark.parametrize("sloppy,delta,mid", [(1, 0.9, 0.0), (1, 0.5, 0.0), (1, 0.3, 0.0), (1, 0.1, 0.0), (2, 0.1, 0.0),
                                              (2, 1e-5, 0.1), (1, 0.01, 0.0), (2, 1e-5, 0.01), (1, 1e-5, 0.0)])
def test_frequent_updates_launch_few_skipped_iterations(L, sloppy, delta, mid):
    """At most a third more launches than with one iteration per body; the API's defaults are delta 0.1 and
    check_interval 16."""
    F, dims = L.fields, (4, 4, 4, 8)
    lat, op = L.lattice(dims, bc=BC), L.operator(mass=0.05)
    U = gauge_field(dims, "haar", 2601)
    b = F.spinor_to_device(gaussian_spinor(dims, 2602, lead=(1,)), lat, 0, L.LQCD_FULL)
    g64, gs = F.gauge_to_device(U, lat, 0, 18), F.gauge_to_device(U, lat, sloppy, 12)
    kw = dict(sloppy_prec=sloppy, delta=delta, delta_mid=mid)
    one, i1 = _launches(L, lat, op, b, g64, gs, 1, **kw)
    many, i16 = _launches(L, lat, op, b, g64, gs, 16, **kw)
    assert (i1.iterations, i1.reliable_updates, i1.residual_replacements) == \
        (i16.iterations, i16.reliable_updates, i16.residual_replacements)
    assert many <= one * 4 / 3


def test_large_solves_skip_no_iteration(L):
    """8,192 blocks per hop: one iteration per body, so only the launches of the chunks' starts differ."""
    F, dims, n5 = L.fields, (16, 16, 16, 16), 32
    lat, op = L.lattice(dims, n5=n5, bc=BC), L.operator(mass=0.05)
    U = gauge_field(dims, "haar", 2611)
    g64, gs = F.gauge_to_device(U, lat, 0, 18), F.gauge_to_device(U, lat, 1, 12)
    b = torch.zeros(L.lqcd_spinor_bytes(lat, 0, L.LQCD_FULL), dtype=torch.uint8, device="cuda")
    host = torch.randn((n5, 16, 16, 16, 16, 4, 3, 2), dtype=torch.float64, device="cuda",
                       generator=torch.Generator(device="cuda").manual_seed(2612))
    L.lqcd_spinor_pack(b, 0, L.LQCD_FULL, host, lat)
    kw = dict(sloppy_prec=1, delta=0.1, update_prec=L.LQCD_F64_DF)
    one, i1 = _launches(L, lat, op, b, g64, gs, 1, **kw)
    many, i64 = _launches(L, lat, op, b, g64, gs, 64, **kw)
    assert i1.iterations == i64.iterations and i1.reliable_updates == i64.reliable_updates
    assert many == one - (i1.iterations - 1)
