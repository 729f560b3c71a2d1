"""The ray mesh's lower edge: rays between -1 and 0 of its first node are inside, however close to -1."""
from fractions import Fraction

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hrt():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_12913_gb300 import hrt as h
    return h


@pytest.mark.parametrize("axis", [0, 1])
def test_a_ray_just_above_minus_one_is_inside(hrt, axis):
    n, chi = 64, (100.0, 102.0)
    g = torch.Generator(device="cuda").manual_seed(axis)
    fields = torch.randn(2, n, n, n, device="cuda", generator=g)
    geom = hrt.make_geom(n, float(n), (32.0, 32.0, 0.0), 1.0, window=(0.0, 101.0))  # the first half shell's plane only
    rm = hrt.RayMesh(hrt.make_raymesh_config(1.0, 3.0, 1e-4, 1))
    _, x2d, n2d = hrt.hrt_raymesh_geometry(rm.cfg, 100.0, 101.0, 1.0)
    inv, half = 1.0 / x2d, Fraction(n2d, 2)
    # positions as the step sees them, theta / x2d + n2d / 2, exact: -1 + (2^-52, 2^-48), -1 + 2^-30 and below -1
    t, close = -(n2d / 2 + 1) / inv, None
    for k in range(-64, 64):
        c = t * (1.0 + k * 2.0 ** -52)
        if Fraction(1, 2 ** 52) < Fraction(c) * Fraction(inv) + half + 1 < Fraction(1, 2 ** 48):
            close = c
    assert close is not None
    theta = torch.zeros(3, 2, dtype=torch.float64, device="cuda")
    theta[:, axis] = torch.tensor([close, (-(n2d / 2 + 1) + 2.0 ** -30) / inv, (-(n2d / 2 + 1) - 2.0 ** -30) / inv],
                                  dtype=torch.float64)
    theta[:, 1 - axis] = 0.3 * x2d
    rays = hrt.RayState(3)
    hrt.hrt_rays_init(rays, theta)
    rm.hrt_raymesh_ray_step(rays, fields[0], fields[1], geom, chi[0], chi[1], 0.0, 0.3)
    # the derivative of the interpolant does not depend on the place along the axis: it is the same for the first two
    # (to a few roundings, and 2^-30 of a cell in the other derivative), and 0 outside
    B = rays.B.double()
    scale = B[1].abs().max()
    assert scale > 0.0
    assert (B[0] - B[1]).abs().max() <= 1e-6 * scale
    assert B[2].abs().max() == 0.0
    rm.close()
