"""Rounding of the power-spectrum bins alone: a map of four pixels a quarter of its side apart, whose float32 spectrum is
known to the bit (twiddles 1, i, -1 and -i)."""
import math

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


@pytest.mark.parametrize("seed", [1, 4])
def test_bins_round_as_FP64_sums(hrt, seed):
    # 256 columns and 129 rows: a bin's sums are at most 129 numbers of a warp each, added in FP64.  Those additions and the
    # three or four operations around them, each within 2^-53 and mostly of either sign: 0.3 sqrt(133) 2^-53 = 3.8e-16 for a
    # bin that every row reaches, less for the others; the bound is on the mean over the bins.
    m, nbins, dth = 256, 20, 3e-4
    a, b, c, d = np.random.default_rng(seed).normal(size=4).astype(np.float32)
    kappa = torch.zeros(m, m, device="cuda")
    kappa[:: m // 4, 0] = torch.tensor([a, b, c, d], device="cuda")
    re, im = np.array([(a + c) + (b + d), a - c, (a + c) - (b + d), a - c]), np.array([0, d - b, 0, b - d])
    square = re.astype(np.longdouble) ** 2 + im.astype(np.longdouble) ** 2  # by kx mod 4
    base = 2.0 * math.pi / (m * dth)
    ell, p, count = hrt.hrt_kappa_power(kappa.reshape(-1), m, dth, nbins, base, base * m / 2)
    nx, nz = np.fft.fftfreq(m, 1.0 / m).round().astype(np.int64), np.arange(m // 2 + 1)
    n2 = nx[:, None] ** 2 + nz[None] ** 2
    modes = np.broadcast_to(np.where((nz == 0) | (nz == m // 2), 1, 2), n2.shape)
    n = np.sqrt(n2.astype(np.longdouble))
    with np.errstate(divide="ignore"):
        bins = np.floor(nbins * np.log(n.astype(float)) / math.log(m / 2) + 1e-9)
    power = np.broadcast_to(square[nx % 4][:, None], n2.shape) * (np.longdouble(dth) ** 4 / (m * np.longdouble(dth)) ** 2)
    off_p, off_ell = [], []
    for k in range(nbins):
        s = (bins == k) & (n2 > 0)
        assert count[k] == modes[s].sum()
        if count[k] == 0:
            continue
        want = (n[s] * modes[s]).sum() / modes[s].sum() * (2 * np.pi / np.longdouble(m * dth))
        off_ell.append(abs(float(ell[k] / want - 1)))
        off_p.append(abs(float(p[k] / ((power[s] * modes[s]).sum() / modes[s].sum()) - 1)))
    assert len(off_p) > 10
    assert np.mean(off_ell) <= 4e-16 and np.mean(off_p) <= 4e-16, (off_ell, off_p)
