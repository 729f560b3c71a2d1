"""The ray-mesh projection through copied planes against the same call from the fields, which a captured stream takes."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hrt():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_12913_gb300 import hrt as h
    return h


# mesh side, box, observer, half shell, (iota, p_min, mu, m_pix): half a mesh cell per ray-mesh cell, many boxes wide and in
# more than one slab; 0.9 of a mesh cell, towards and beside the observer; one slab with fewer planes than a block copies;
# more planes than one block copies
CASES = [(64, 64.0, (32.0, 32.0, 0.0), (1000.0, 1060.0), (0.5, 256.0, 1e-4, 500)),
         (60, 120.0, (3.0, 118.0, 7.0), (970.0, 900.0), (0.9, 256.0, 1e-4, 500)),
         (96, 96.0, (48.0, 48.0, 0.0), (500.0, 510.0), (0.5, 256.0, 1e-4, 300)),
         (64, 64.0, (1.0, 60.0, 0.0), (400.0, 433.0), (0.5, 256.0, 1e-4, 300))]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_planes_match_the_fields(hrt, case):
    n, box, obs, chi, cfg = CASES[case]
    g = torch.Generator(device="cuda").manual_seed(case)
    fields = torch.randn(2, n, n, n, device="cuda", generator=g)
    geom = hrt.make_geom(n, box, obs, 1.0)
    rm = hrt.RayMesh(hrt.make_raymesh_config(*cfg))
    _, _, n2d = hrt.hrt_raymesh_geometry(rm.cfg, chi[0], chi[1], box / n)
    assert n2d * n2d * abs(chi[1] - chi[0]) * n / box > 1 << 23  # large enough for the planes
    planes = rm.hrt_raymesh_kick(fields[0], fields[1], geom, *chi)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        direct = rm.hrt_raymesh_kick(fields[0], fields[1], geom, *chi)
    graph.replay()
    torch.cuda.synchronize()
    # the same weights and values; sums of a few hundred terms at most, each within 2^-24, so that both are within
    # 1e-5 of the largest value
    assert (planes - direct).abs().max() <= 1e-5 * direct.abs().max()
    assert direct.abs().max() > 0
    rm.close()
