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


def _compare(whole, parts):
    """Same cells and numbers, other rounding of the position: a ray whose node lies within about 2^-24 of a cell face may
    take the other cell's derivative, which A and B then carry."""
    for a, b, exact in zip(whole, parts, (True, True, False, False)):
        off = (a - b).abs().amax(dim=1) / b.abs().max()
        assert off.median() <= 1e-6
        if exact:
            assert off.max() <= 1e-5
        else:
            assert (off > 1e-4).float().mean() <= 1e-3


# half width of the bundle (rad), rays, whether there are planes: 0.95 and 1.08 cells per ray, 0.97 and 1.03 of 384 bytes per
# ray, 0.95 and 1.03 of 512 MB
@pytest.mark.parametrize("width,r,planes", [(0.11, 64000, True), (0.117, 64000, False), (0.194, 400000, True),
                                            (0.2, 400000, False), (0.36, 1500000, True), (0.375, 1500000, False)])
def test_planes_end_where_they_no_longer_pay(hrt, width, r, planes):
    n, chi = 64, (1000.0, 1100.0)
    fields, theta = _bundle(n, r, width, r)
    geom = hrt.make_geom(n, float(n), (32.0, 32.0, 0.0))
    nodes = sum(_nodes(hrt, geom, chi))
    side = int(2.0 * width * (chi[1] - 0.5)) + 6
    assert r * nodes >= PLANE_WORK
    limit = min(r, min(max(384 * r, 96 << 20), 512 << 20) // 8 // nodes)
    assert (side - 4) ** 2 < side ** 2 <= limit if planes else (side - 4) ** 2 > limit
    eta = torch.zeros(r, 2, device="cuda")
    whole = _step(hrt, fields, geom, theta, eta, chi, r)
    parts = _step(hrt, fields, geom, theta, eta, chi, 40000)
    assert 40000 * nodes < PLANE_WORK
    _compare(whole, parts)
    # the planes' arithmetic is packed, so that of so many rays some round otherwise; the fields' is the parts'
    assert torch.equal(whole[1], parts[1]) != planes


# mesh side, box, observer, half width of the bundle (rad), shell, spread of eta, samples per cell: a bundle within the box; one
# wider than the box, off the origin; a shell towards the observer, with fewer samples than cells; rays that leave the
# first half shell's cells in the second
CASES = [(64, 100.0, (50.0, 50.0, 0.0), 0.02, (900.0, 1000.0), 0.0, 1.0),
         (60, 60.0, (3.0, 61.0, 7.0), 0.05, (900.0, 950.0), 0.0, 1.0),
         (96, 200.0, (100.0, 20.0, 0.0), 0.01, (700.0, 560.0), 0.0, 0.4),
         (64, 100.0, (50.0, 50.0, 0.0), 0.005, (500.0, 700.0), 200.0, 2.0)]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_bundles_that_reach_the_planes_match_the_fields(hrt, case):
    n, box, obs, width, chi, spread, samples = CASES[case]
    geom = hrt.make_geom(n, box, obs, samples)
    nodes = sum(_nodes(hrt, geom, chi))
    r = PLANE_WORK // nodes + 1
    part = PLANE_WORK // nodes // 2
    fields, theta = _bundle(n, r, width, case)
    eta = spread * torch.randn(r, 2, device="cuda", generator=torch.Generator(device="cuda").manual_seed(case + 10))
    whole = _step(hrt, fields, geom, theta, eta, chi, r)
    parts = _step(hrt, fields, geom, theta, eta, chi, part)
    _compare(whole, parts)
    assert not torch.equal(whole[3], parts[3])  # the planes' packed arithmetic rounds some of so many rays otherwise
    assert parts[3].abs().max() > 0


@pytest.mark.parametrize("value", [float("inf"), float("nan"), 1e30])
def test_an_angle_out_of_range_stays_its_own(hrt, value):
    # in half shells of many nodes, of a bundle on the planes
    n, chi, r = 64, (900.0, 1000.0), 70000
    geom = hrt.make_geom(n, 100.0, (50.0, 50.0, 0.0))
    assert r * sum(_nodes(hrt, geom, chi)) >= PLANE_WORK
    fields, theta = _bundle(n, r, 0.01, 9)
    eta = torch.zeros(r, 2, device="cuda")
    want = _step(hrt, fields, geom, theta, eta, chi, r)
    eta[7] = value  # its angle of the second half shell
    got = _step(hrt, fields, geom, theta, eta, chi, r)
    keep = torch.ones(r, dtype=torch.bool, device="cuda")
    keep[7] = False
    for a, b in zip(got, want):
        assert torch.equal(a[keep], b[keep])
    parts = _step(hrt, fields, geom, theta, eta, chi, r // 2)
    assert not torch.equal(got[3][keep], parts[3][keep])  # the whole bundle's came from the planes


def test_an_angle_that_is_not_finite_at_the_start_leaves_all_to_the_fields(hrt):
    # the box of the rays is no sensible number of cells then
    n, chi, r = 64, (900.0, 1000.0), 70000
    geom = hrt.make_geom(n, 100.0, (50.0, 50.0, 0.0))
    fields, theta = _bundle(n, r, 0.01, 9)
    eta = torch.zeros(r, 2, device="cuda")
    for value in (float("nan"), float("inf"), 1e12):
        theta[5, 1] = value
        whole = _step(hrt, fields, geom, theta, eta, chi, r)
        parts = _step(hrt, fields, geom, theta, eta, chi, r // 2)
        keep = torch.ones(r, dtype=torch.bool, device="cuda")
        keep[5] = False
        for a, b in zip(whole, parts):
            assert torch.equal(a[keep], b[keep])
