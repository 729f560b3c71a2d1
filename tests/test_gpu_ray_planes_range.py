"""Node planes of the ray step at the ends of their range: bundles that do reach the planes, against the fields that their
parts gather from."""
import pytest
import torch

pytestmark = pytest.mark.gpu

PLANE_WORK = 1 << 22  # rays times nodes from which a bundle's step goes through the planes


@pytest.fixture(scope="module")
def hrt():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_12913_gb300 import hrt as h
    return h


def _nodes(hrt, geom, chi):
    n1, n2 = hrt.hrt_ray_step_coefficients(geom, *chi, 0.0, 0.3)[:2]
    return n1, n2


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


def _bundle(n, r, width, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    fields = torch.randn(2, n, n, n, device="cuda", generator=g)
    theta = (2.0 * torch.rand(r, 2, device="cuda", generator=g, dtype=torch.float64) - 1.0) * width
    return fields, theta


@pytest.mark.parametrize("value", [3e38, -3e38, float("inf"), float("nan")])
@pytest.mark.parametrize("obs", [(50.0, 50.0, 0.0), (-50.0, 1.0, 0.0)])
def test_a_far_angle_in_a_half_shell_of_one_node(hrt, value, obs):
    # The deflection of one ray takes its angle of the second half shell to about 1e33 (or beyond all numbers): the
    # half shell's only node has no offset along the line of sight, so that the cell alone says that it is far out.
    n, r, chi = 64, 1 << 21, (900.0, 901.0)
    fields, theta = _bundle(n, r, 0.01, 1)
    geom = hrt.make_geom(n, 100.0, obs)
    assert _nodes(hrt, geom, chi) == (1, 1) and 2 * r >= PLANE_WORK
    eta = torch.zeros(r, 2, device="cuda")
    want = _step(hrt, fields, geom, theta, eta, chi, r)
    eta[7, 0] = value
    eta[11] = value
    got = _step(hrt, fields, geom, theta, eta, chi, r)
    keep = torch.ones(r, dtype=torch.bool, device="cuda")
    keep[7] = keep[11] = False
    for a, b in zip(got, want):
        assert torch.equal(a[keep], b[keep])
    # The far rays gather from the fields there, as in a bundle of their own.  Their first half shell's kicks are of
    # fields up to about 5 with weights 0.3 (eta) and 170 (B), in a few FP32 operations: 2^-24 * 8 * 5 of the weight.
    far = torch.tensor([7, 11], device="cuda")
    alone = _step(hrt, fields, geom, theta[far], eta[far], chi, 2)
    for a, b, atol in zip(got, alone, (1e-6, 1e-6, 1e-6, 1e-3)):
        assert torch.allclose(a[far], b, rtol=1e-5, atol=atol, equal_nan=True)
