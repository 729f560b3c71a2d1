"""The library's count of its own kernel launches, against what the calls' routes launch."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hrt():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_12913_gb300 import hrt as h
    return h


def _count(hrt, fn):
    before = hrt.hrt_kernel_launches()
    fn()
    return hrt.hrt_kernel_launches() - before


@pytest.mark.parametrize("n,kernels", [(60, 1), (64, 5), (256, 5)])  # the k-space kernel; five FFT passes
def test_a_solve(hrt, n, kernels):
    pm = hrt.PM(n, float(n))
    rho, grad = torch.ones(n, n, n, device="cuda"), torch.empty(3, n, n, n, device="cuda")
    assert _count(hrt, lambda: pm.solve(rho, 0.45, hrt.make_filter(), grad)) == kernels
    pm.close()


@pytest.mark.parametrize("r,nodes,kernels", [(16383, 512, 1), (16384, 256, 3), (65536, 62, 1), (65536, 64, 3)])
def test_a_ray_step(hrt, r, nodes, kernels):
    # bounds, planes and the step from 2^14 rays and 2^22 ray-nodes on, else the step alone
    fields = torch.zeros(2, 64, 64, 64, device="cuda")
    geom = hrt.make_geom(64, 64.0, (32.0, 32.0, 0.0))
    rays = hrt.RayState(r)
    hrt.hrt_rays_init(rays, torch.zeros(r, 2, dtype=torch.float64, device="cuda"))
    chi = (1000.0, 1000.0 + nodes)
    assert sum(hrt.hrt_ray_step_coefficients(geom, *chi, 0.0, 0.3)[:2]) == nodes
    assert _count(hrt, lambda: hrt.hrt_ray_step(rays, fields[0], fields[1], geom, *chi, 0.0, 0.3)) == kernels


@pytest.mark.parametrize("planes,kernels", [(8, 2), (64, 3)])
def test_a_ray_mesh_kick(hrt, planes, kernels):
    # 512^2 nodes: projection and filter; above 2^23 node-planes the copy of the planes too (one slab)
    n = 128
    fields = torch.zeros(2, n, n, n, device="cuda")
    geom = hrt.make_geom(n, float(n), (64.0, 64.0, 0.0), 1.0)
    rm = hrt.RayMesh(hrt.make_raymesh_config(0.5, 128.0, 1e-4, 200))
    assert hrt.hrt_raymesh_geometry(rm.cfg, 1000.0, 1000.0 + planes, 1.0)[2] == 512
    assert _count(hrt, lambda: rm.hrt_raymesh_kick(fields[0], fields[1], geom, 1000.0, 1000.0 + planes)) == kernels
    rm.close()
