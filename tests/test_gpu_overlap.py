"""Launches that start while their predecessor runs: chains without host
synchronisation give the bits of the same chain synchronised after every call."""
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
