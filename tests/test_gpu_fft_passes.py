"""The FFT passes of the Poisson solve against a plain 64-bit torch FFT solve of the same density."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hrt():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_12913_gb300 import hrt as h
    return h


def _solve64(rho, box, pref, deconv, smooth, comps, table=None, k_max=0.0):
    n = rho.shape[0]
    kf = 2.0 * math.pi / box
    k = torch.fft.fftfreq(n, 1.0 / n, device="cuda").double().round() * kf
    axes = [k[:, None, None], k[None, :, None], k[: n // 2 + 1].abs()[None, None, :]]
    k2 = sum(a * a for a in axes)
    m = torch.where(k2 > 0, -pref / torch.where(k2 > 0, k2, 1.0), 0.0) * torch.exp(-0.5 * k2 * smooth * smooth)
    for a in axes:
        m = m * torch.special.sinc(a * (box / n / (2.0 * math.pi))) ** -deconv
    if table is not None:
        t = torch.sqrt(k2) * ((table.numel() - 1) / k_max)
        j = t.long().clamp(max=table.numel() - 2)
        g = table.double()
        m = m * torch.where(t < table.numel() - 1, g[j] + (g[j + 1] - g[j]) * (t - j), 1.0)
    f = torch.fft.rfftn(rho.double()) * m
    out = []
    for c in range(comps):
        d = axes[c].clone().reshape(-1)
        d[n // 2] = 0.0
        out.append(torch.fft.irfftn(f * (1j * d.reshape(axes[c].shape)), s=(n, n, n)))
    return out


@pytest.mark.parametrize("n,rays", [(64, True), (96, True), (128, False), (192, True), (256, False), (256, True), (384, True),
                                    (512, True), (768, True), (1024, False)])
def test_solve_matches_a_64_bit_solve(hrt, n, rays):
    # zero-mean white noise: every mode, the Nyquist planes included, carries the same power.  Rounding of 2 log2(n^3)
    # FP32 butterfly levels plus the multiplier's few factors, each 2^-24 relative to the signal's rms and independent:
    # sqrt(60) 2^-24 + 8 2^-24 is below 1e-6 of the rms in the 2-norm; the bound leaves a factor of three.
    box, pref = 1.1 * n, 0.45
    g = torch.Generator(device="cuda").manual_seed(n)
    rho = torch.randn(n, n, n, device="cuda", generator=g)
    f = hrt.make_filter(4.0, box / n)
    pm = hrt.PM(n, box, 2 if rays else 0)
    grad = torch.empty(3, n, n, n, device="cuda")
    want = _solve64(rho, box, pref, 4.0, box / n, 3)
    table = (1.5 - torch.linspace(0.0, 1.0, 301, device="cuda") ** 2).float()
    k_max = 2.0 * math.pi * n / box / 3.0  # ends inside the mesh's |k|: 1 beyond
    if rays:
        ray = torch.empty(2, n, n, n, device="cuda")
        fr = hrt.make_filter(2.0, 0.5 * box / n, table, k_max)
        pm.solve(rho.clone(), pref, f, grad, fr, ray)
        want += _solve64(rho, box, pref, 2.0, 0.5 * box / n, 2, table, k_max)
        got = [*grad, *ray]
    else:
        pm.solve(rho.clone(), pref, f, grad)
        got = list(grad)
    for x, y in zip(got, want):
        assert (x - y).norm() <= 3e-6 * y.norm()
    pm.close()


def test_ray_fields_of_a_plan_may_be_left_out(hrt):
    n, box = 256, 256.0
    g = torch.Generator(device="cuda").manual_seed(3)
    rho = torch.randn(n, n, n, device="cuda", generator=g)
    f = hrt.make_filter(4.0, box / n)
    out = []
    for rays in (0, 2):
        pm = hrt.PM(n, box, rays)
        grad = torch.empty(3, n, n, n, device="cuda")
        pm.solve(rho.clone(), 0.45, f, grad)
        out.append(grad)
        pm.close()
    assert torch.equal(*out)


@pytest.mark.parametrize("n", [64, 96, 128, 192, 384, 768])
def test_density_spectrum_after_a_solve(hrt, n):
    # sides whose solve always offered the density's 3D spectrum still do, with and without ray fields
    box = float(n)
    g = torch.Generator(device="cuda").manual_seed(n)
    rho = torch.randn(n, n, n, device="cuda", generator=g)
    want = torch.fft.rfftn(rho.double())
    f = hrt.make_filter(4.0, 1.0)
    for rays in (0, 2):
        pm = hrt.PM(n, box, rays)
        grad = torch.empty(3, n, n, n, device="cuda")
        ray = torch.empty(2, n, n, n, device="cuda") if rays else None
        pm.solve(rho.clone(), 0.45, f, grad, f if rays else None, ray)
        out = torch.empty(n, n, n // 2 + 1, dtype=torch.complex64, device="cuda")
        pm.density_spectrum(out)
        assert (out - want).norm() <= 1e-6 * want.norm()  # log2(n^3) butterfly levels of 2^-24
        pm.close()


@pytest.mark.parametrize("n,learned", [(64, False), (96, True), (128, False), (192, False), (256, True), (256, False), (384, False),
                                       (512, False), (768, False)])
def test_adjoint_matches_a_64_bit_transpose(hrt, n, learned):
    # rho_bar = sum_j C2R(conj(H_j) R2C(g_j)) with H_j the solve's factors; the rounding bound of the solve
    box, pref = 0.9 * n, 0.45
    g = torch.Generator(device="cuda").manual_seed(n)
    bar = torch.randn(3, n, n, n, device="cuda", generator=g)
    table = (1.5 - torch.linspace(0.0, 1.0, 301, device="cuda") ** 2).float() if learned else None
    k_max = 2.0 * math.pi * n / box / 3.0
    f = hrt.make_filter(4.0, box / n, table, k_max) if learned else hrt.make_filter(4.0, box / n)
    want = 0.0
    for c in range(3):  # -d_c of the solve of each component: the transpose of an odd real operator
        want = want - _solve64(bar[c], box, pref, 4.0, box / n, 3, table, k_max)[c]
    pm = hrt.PM(n, box)
    out = torch.empty(n, n, n, device="cuda")
    pm.solve_adjoint(bar, pref, f, out)
    assert (out - want).norm() <= 3e-6 * want.norm()
    pm.close()
