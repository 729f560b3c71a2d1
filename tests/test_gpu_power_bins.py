"""Power-spectrum bins by integer |n|^2 against the oracle's rule: counts equal, ell and P to rounding."""
import math

import numpy as np
import pytest
import torch

import synthetic
from oracle import power as opow

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hrt():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_12913_gb300 import hrt as h
    return h


# map side, bins, ell range in units of the fundamental: one column, more bins than modes, columns of a warp's last
# segment only, a first bin above the lowest modes, an end below the highest, edges on exact |n|^2
@pytest.mark.parametrize("m,nbins,lo,hi", [(2, 1, 0.5, 2.0), (60, 256, 1.0, 30.0), (510, 20, 1.0, 255.0),
                                           (514, 20, 3.7, 301.0), (66, 7, 1.0, 128.0), (2050, 33, 2.0, 64.0)])
def test_bins_match_the_rule(hrt, m, nbins, lo, hi):
    dth = 3e-4
    base = 2.0 * math.pi / (m * dth)
    kap = synthetic.gaussian_field(m, (m, m), 0.02).astype(np.float32)
    ell, p, cnt = hrt.hrt_kappa_power(torch.tensor(kap, device="cuda").reshape(-1), m, dth, nbins, lo * base, hi * base)
    ell_w, p_w, cnt_w = opow.kappa_power(kap.astype(np.float64), dth, nbins, lo * base, hi * base)
    assert np.array_equal(cnt, cnt_w)
    ok = cnt_w > 0
    assert np.allclose(ell[ok], ell_w[ok], rtol=1e-12)
    # FP32 FFT: a mode is off by at most log2(m^2) 2^-24 of the map's rms power times the few butterflies' factor
    assert np.allclose(p[ok], p_w[ok], rtol=2e-5)


def test_scale_of_the_map(hrt):
    # the squares are formed in FP64: a map of 1e-25 has the spectrum of the same map, scaled
    m, dth = 128, 3e-4
    kap = torch.tensor(synthetic.gaussian_field(5, (m, m), 1.0), dtype=torch.float32, device="cuda").reshape(-1)
    lo, hi = 2.0 * math.pi / (m * dth), math.pi / dth
    p1 = hrt.hrt_kappa_power(kap, m, dth, 8, lo, hi)[1]
    p2 = hrt.hrt_kappa_power(kap * 2.0 ** -80, m, dth, 8, lo, hi)[1]
    assert np.allclose(p2, p1 * 2.0 ** -160, rtol=1e-12)
