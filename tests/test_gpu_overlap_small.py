"""Overlapping launches of hops that fill the SMs about once cost no more than ordinary
ones: the blocks of a hop must not be placed while its predecessor holds most of the SMs."""
import pytest

from synthetic import gauge_field

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _us(f):
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = 1e9
    for r in range(8):  # the first one warms up
        start.record()
        for _ in range(10):
            f()
        end.record()
        end.synchronize()
        best = min(best, start.elapsed_time(end) * 100 if r else best)
    return best


@pytest.mark.parametrize("dims,n5,full,gparity", [((8, 8, 8, 8), 4, True, 0), ((12, 12, 12, 24), 1, False, 0),
                                                  ((10, 6, 14, 18), 1, True, 0), ((10, 6, 14, 18), 2, False, 5)])
def test_direct_calls_cost_no_more_than_captured_ones(dims, n5, full, gparity):
    """FP64 M^dag M back to back, directly and as a replayed graph (whose launches are ordinary): at
    most 15 % more; with blocks placed early it took 1.4 to 2.2 times as long."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1512_03487_gb300 as L
    from paper_1512_03487_gb300 import fields as F
    lat, subset = L.lattice(dims, n5=n5, bc=(1.0, 1.0, 1.0, -1.0)), L.LQCD_FULL if full else L.LQCD_EVEN
    op = L.operator(mass=0.1, prec=0, recon=12, gparity=gparity)
    links = F.gauge_to_device(gauge_field(dims, "haar", 2801), L.lattice(dims), 0, 12)
    src = torch.zeros(L.lqcd_spinor_bytes(lat, 0, subset), dtype=torch.uint8, device="cuda")
    out = torch.zeros_like(src)
    tmp = torch.zeros(L.lqcd_operator_workspace_bytes(lat, op, subset), dtype=torch.uint8, device="cuda")

    def call():
        L.lqcd_MdagM(out, src, links, lat, op, subset, tmp)

    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    assert _us(call) <= 1.15 * _us(graph.replay)
