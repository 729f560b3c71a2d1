"""The ray-step adjoint's field cotangents, summed over a warp's rays of one cell: an image, whose warps hold long runs of a
cell, against the same rays in random order, and cotangents on 16-byte boundaries against others."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hrt():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_12913_gb300 import hrt as h
    return h


def _adjoint(hrt, fields, theta, bars, chi, n, box, offset, width):
    r = theta.shape[0]
    rays, bar = hrt.RayState(r), hrt.RayState(r)
    hrt.hrt_rays_init(rays, theta)
    for x, y in zip((bar.theta, bar.eta, bar.A, bar.B), bars):
        x.copy_(y)
    out = [torch.zeros(n ** 3 + offset, device="cuda")[offset:].view(n, n, n) for _ in range(2)]
    node = torch.zeros(3, hrt.MAX_RAY_NODES, dtype=torch.float64, device="cuda")
    drift = torch.zeros(1, dtype=torch.float64, device="cuda")
    geom = hrt.make_geom(n, box, (0.5 * box, 0.4 * box, 0.0), 1.0, image_width=width)
    hrt.hrt_ray_step_adjoint(rays, fields[0], fields[1], geom, chi[0], chi[1], 0.0, 0.3, bar, out[0], out[1], node, drift)
    return torch.stack(out), node, [bar.theta, bar.eta, bar.A, bar.B]


# mesh side (a multiple of 4; of 2), image side and field of view: runs of about 10 rays, of 2, of less than 1, and one that
# fills no whole warp of the last tile row
@pytest.mark.parametrize("n,m,fov", [(64, 48, 0.01), (62, 48, 0.01), (64, 48, 0.05), (64, 64, 0.3), (30, 16, 0.004), (64, 33, 0.02)])
def test_order_and_alignment_do_not_matter(hrt, n, m, fov):
    box, chi = float(n), (500.0, 500.0 + 0.6 * n)
    g = torch.Generator(device="cuda").manual_seed(n + m)
    fields = torch.randn(2, n, n, n, device="cuda", generator=g)
    c = (torch.arange(m, dtype=torch.float64, device="cuda") + 0.5 - 0.5 * m) * (fov / m)
    ty, tx = torch.meshgrid(c, c, indexing="ij")
    theta = torch.stack([tx.reshape(-1), ty.reshape(-1)], 1).contiguous()
    bars = [torch.randn(m * m, k, device="cuda", generator=g).reshape(s).to(t) for k, s, t in
            ((2, (m * m, 2), torch.float64), (2, (m * m, 2), torch.float32), (4, (m * m, 4), torch.float32), (4, (m * m, 4), torch.float32))]
    shapes = [x.shape for x in (lambda b: (b.theta, b.eta, b.A, b.B))(hrt.RayState(m * m))]
    bars = [b.reshape(s) for b, s in zip(bars, shapes)]
    image = _adjoint(hrt, fields, theta, bars, chi, n, box, 0, m)
    order = torch.randperm(m * m, device="cuda", generator=g)
    other = _adjoint(hrt, fields, theta[order].contiguous(), [b[order] for b in bars], chi, n, box, 1, 0)
    # sums of up to m^2 float terms of either sign in different orders: 2^-24 sqrt(terms) each, over what cancels
    assert (image[0] - other[0]).abs().max() <= 1e-5 * image[0].abs().max()
    assert (image[1] - other[1]).abs().max() <= 1e-5 * image[1].abs().max()
    for a, b in zip(image[2], other[2]):
        assert torch.equal(a[order], b)  # a ray's own cotangents do not depend on its neighbours
