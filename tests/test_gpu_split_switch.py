"""The switch between the FFT passes and the 3D plans: there and back at every side of the passes."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SIDES = [64, 96, 128, 192, 256, 384, 512, 768, 1024]


@pytest.fixture(scope="module")
def hrt():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_12913_gb300 import hrt as h
    return h


@pytest.mark.parametrize("n", SIDES)
def test_back_to_the_passes(hrt, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    rho = torch.randn(n, n, n, device="cuda", generator=g)
    f = hrt.make_filter(4.0, 1.0)
    pm = hrt.PM(n, float(n))
    out = []
    for path in (None, False, True):
        if path is not None:
            pm.set_split(path)
        grad = torch.empty(3, n, n, n, device="cuda")
        pm.solve(rho.clone(), 0.45, f, grad)
        out.append(grad)
    assert torch.equal(out[0], out[2])  # the default is the passes, and they are deterministic
    # the 3D path: rounding of 2 log2(n^3) FP32 butterfly levels in each, as against a 64-bit solve
    assert (out[0] - out[1]).norm() <= 6e-6 * out[1].norm()
    pm.close()


def test_other_sides_have_no_passes(hrt):
    pm = hrt.PM(60, 60.0)
    pm.set_split(False)
    with pytest.raises(hrt.HRTError) as e:
        pm.set_split(True)
    assert e.value.status == 1
    pm.close()
