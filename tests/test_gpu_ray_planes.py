"""The ray step on node planes against the same step from the fields, which smaller bundles of rays take."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hrt():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_12913_gb300 import hrt as h
    return h


def _step(hrt, fields, geom, theta, eta, chi, part):
    """One step of the bundle in parts of `part` rays: theta, eta, A, B of all."""
    out = []
    for lo in range(0, theta.shape[0], part):
        rays = hrt.RayState(min(part, theta.shape[0] - lo))
        hrt.hrt_rays_init(rays, theta[lo:lo + part].contiguous())
        rays.eta.copy_(eta[lo:lo + part])
        hrt.hrt_ray_step(rays, fields[0], fields[1], geom, chi[0], chi[1], 0.0, 0.3)
        out.append([rays.theta, rays.eta, rays.A, rays.B])
    return [torch.cat(x) for x in zip(*out)]


# mesh side, box, observer, half width of the bundle (rad), shell, spread of eta: a bundle within the box; one wider than
# the box, off the origin; a shell towards the observer, with fewer samples than cells; rays that leave the first
# half shell's cells in the second
CASES = [(64, 100.0, (50.0, 50.0, 0.0), 0.02, (900.0, 1000.0), 0.0, 1.0),
         (60, 60.0, (3.0, 61.0, 7.0), 0.05, (900.0, 950.0), 0.0, 1.0),
         (96, 200.0, (100.0, 20.0, 0.0), 0.01, (700.0, 560.0), 0.0, 0.4),
         (64, 100.0, (50.0, 50.0, 0.0), 0.005, (500.0, 700.0), 200.0, 2.0)]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_planes_match_the_fields(hrt, case):
    n, box, obs, width, chi, spread, samples = CASES[case]
    g = torch.Generator(device="cuda").manual_seed(case)
    fields = torch.randn(2, n, n, n, device="cuda", generator=g)
    r = 200 * 300  # above the planes' smallest bundle; no image
    theta = (2.0 * torch.rand(r, 2, device="cuda", generator=g, dtype=torch.float64) - 1.0) * width
    eta = spread * torch.randn(r, 2, device="cuda", generator=g)
    geom = hrt.make_geom(n, box, obs, samples)
    whole = _step(hrt, fields, geom, theta, eta, chi, r)
    parts = _step(hrt, fields, geom, theta, eta, chi, 10000)
    # the same cells and numbers, the position's fraction rounded from 2^-32 cells instead of FP64: a ray whose node lies
    # within 2^-24 of a cell face may take the other cell's derivative, which A and B then carry
    for a, b, exact in zip(whole, parts, (True, True, False, False)):
        scale = b.abs().max()
        off = (a - b).abs().amax(dim=1) / scale
        assert off.median() <= 1e-6
        if exact:
            assert off.max() <= 1e-5
        else:
            assert (off > 1e-4).float().mean() <= 1e-3
    assert not torch.equal(whole[3], torch.zeros_like(whole[3]))


def test_an_angle_that_is_not_finite_stays_its_own(hrt):
    n = 64
    g = torch.Generator(device="cuda").manual_seed(9)
    fields = torch.randn(2, n, n, n, device="cuda", generator=g)
    theta = 0.01 * (2.0 * torch.rand(60000, 2, device="cuda", generator=g, dtype=torch.float64) - 1.0)
    geom = hrt.make_geom(n, 100.0, (50.0, 50.0, 0.0))
    eta = torch.zeros(60000, 2, device="cuda")
    want = _step(hrt, fields, geom, theta, eta, (900.0, 1000.0), 60000)
    eta[7] = float("inf")  # its angle of the second half shell
    got = _step(hrt, fields, geom, theta, eta, (900.0, 1000.0), 60000)
    keep = torch.ones(60000, dtype=torch.bool, device="cuda")
    keep[7] = False
    for a, b in zip(got, want):
        assert torch.equal(a[keep], b[keep])
