"""Initial conditions allocate what their transforms need and nothing of a Poisson solve."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hrt():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_12913_gb300 import hrt as h
    yield h
    h.hrt_inject_alloc_failure(0)


# at most the FFT work area, the noise's spectrum, the three fields' spectra and the transfer table; 2LPT: and its six fields
@pytest.mark.parametrize("call,most", [("hrt_ic_zeldovich", 4), ("hrt_ic_2lpt", 5)])
@pytest.mark.parametrize("n", [60, 64])  # without and with FFT passes of its side
def test_allocations_of_initial_conditions(hrt, call, most, n):
    noise = torch.randn(n ** 3, device="cuda")
    disp = torch.empty(3, n ** 3, device="cuda")
    mom = torch.empty_like(disp)
    run = lambda: getattr(hrt, call)(noise, n, 100.0, 0.3, 0.7, 0.96, 0.8, 0.02, disp, mom)  # noqa: E731
    hrt.hrt_inject_alloc_failure(1)
    with pytest.raises(hrt.HRTError) as e:
        run()
    assert e.value.status == 2
    hrt.hrt_inject_alloc_failure(most + 1)  # the allocation after the last that it may make
    run()
    hrt.hrt_inject_alloc_failure(0)
