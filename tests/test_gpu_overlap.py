"""Launches that start while their predecessor runs, and several iterations per body of
the solver's graph: chains without host synchronisation give the bits of the same
chain synchronised after every call, and a solve's iterations, updates and solution
do not depend on how many iterations a graph body holds."""
import numpy as np
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


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (8, 8, 8, 16)])
@pytest.mark.parametrize("prec,recon", [(0, 18), (1, 12), (2, 12), (3, 18)])
@pytest.mark.parametrize("stream", [False, True])
def test_chained_operators_without_synchronisation(L, dims, prec, recon, stream):
    """Links packed (an ordinary launch), then 24 operators each reading its
    predecessor's output through buffers that are reused every other call, links
    replaced half way; on the default and on another stream."""
    F = L.fields
    lat = L.lattice(dims, bc=BC)
    op = L.operator(mass=0.1, prec=prec, recon=recon)
    store = 0 if prec == 3 else prec
    U = [torch.view_as_real(torch.from_numpy(gauge_field(dims, "haar", 2301 + k)).cuda()) for k in (0, 1)]
    psi = F.spinor_to_device(gaussian_spinor(dims, 2303, lead=(1,)), lat, store, L.LQCD_FULL)
    links = F.empty(L.lqcd_gauge_bytes(lat, store, recon))
    warm = torch.zeros_like(psi)
    L.lqcd_gauge_pack(links, store, recon, U[0], lat)
    L.lqcd_M(warm, psi, links, lat, op, L.LQCD_FULL, 0, None)  # launch shapes are timed here, not below
    L.lqcd_M(warm, psi, links, lat, op, L.LQCD_FULL, 1, None)
    torch.cuda.synchronize()

    def chain(sync):
        bufs = [psi.clone(), torch.zeros_like(psi), torch.zeros_like(psi)]
        s = torch.cuda.Stream() if stream else torch.cuda.current_stream()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            for k in range(24):
                if k % 12 == 0:
                    L.lqcd_gauge_pack(links, store, recon, U[k // 12], lat)
                src, dst = bufs[0 if k == 0 else 1 + (k - 1) % 2], bufs[1 + k % 2]
                L.lqcd_M(dst, src, links, lat, op, L.LQCD_FULL, k % 2, None)
                if sync:
                    torch.cuda.synchronize()
            out = bufs[2].clone()
        torch.cuda.synchronize()
        return out

    expect = chain(True)
    for _ in range(5):
        assert torch.equal(chain(False), expect)


@pytest.mark.parametrize("sloppy,mid", [(0, 0.0), (1, 0.0), (2, 0.01)])
def test_solve_does_not_depend_on_the_iterations_per_graph_body(L, sloppy, mid):
    F = L.fields
    dims, m = (4, 4, 4, 8), 0.05
    lat = L.lattice(dims, bc=BC)
    op = L.operator(mass=m)
    U, b = gauge_field(dims, "haar", 2311), gaussian_spinor(dims, 2312, lead=(1,))
    g64 = F.gauge_to_device(U, lat, 0, 18)
    gs = F.gauge_to_device(U, lat, sloppy, 12) if sloppy else g64
    bd = F.spinor_to_device(b, lat, 0, L.LQCD_FULL)
    seen = []
    for check in (1, 2, 3, 7, 8, 11, 12, 64):  # 1, 2, 3, 7, 8, 1, 6, 8 iterations per body
        prm = L.solver_params(tol=1e-10, maxiter=500, sloppy_prec=sloppy, sloppy_recon=12, delta=1e-3, delta_mid=mid,
                              check_interval=check)
        ws = F.empty(L.lqcd_eo_solve_workspace_bytes(lat, op, prm))
        x = F.empty(L.lqcd_spinor_bytes(lat, 0, L.LQCD_FULL))
        i = L.lqcd_eo_solve(x, bd, g64, gs, lat, op, prm, ws)
        seen.append((i.iterations, i.reliable_updates, i.residual_replacements, x.clone()))
    for s in seen[1:]:
        assert s[:3] == seen[0][:3]
        assert torch.equal(s[3], seen[0][3])


@pytest.mark.parametrize("maxiter", [1, 5, 8, 9])
def test_iteration_cap_inside_a_body(L, maxiter):
    """The cap ends the solve at exactly maxiter iterations, with the FP64 residual known."""
    F = L.fields
    dims = (4, 4, 4, 8)
    lat = L.lattice(dims, bc=BC)
    op = L.operator(mass=0.05)
    U, b = gauge_field(dims, "haar", 2321), gaussian_spinor(dims, 2322, lead=(1,))
    g64, g32 = F.gauge_to_device(U, lat, 0, 18), F.gauge_to_device(U, lat, 1, 12)
    bd = F.spinor_to_device(b, lat, 0, L.LQCD_FULL)
    x = F.empty(L.lqcd_spinor_bytes(lat, 0, L.LQCD_FULL))
    res = []
    for check, graph in ((64, 1), (1, 1), (1, 0)):
        prm = L.solver_params(tol=1e-12, maxiter=maxiter, sloppy_prec=1, sloppy_recon=12, delta=0.0,
                              check_interval=check, use_graph=graph)
        ws = F.empty(L.lqcd_eo_solve_workspace_bytes(lat, op, prm))
        i = L.lqcd_eo_solve(x, bd, g64, g32, lat, op, prm, ws, raise_on_error=False)
        assert i.iterations == maxiter and i.status != 0
        res.append(i.true_rel_residual)
    assert np.isfinite(res).all() and res[0] == res[1]
    assert res[0] == pytest.approx(res[2], rel=1e-6)  # the host-driven path: the same kernels
