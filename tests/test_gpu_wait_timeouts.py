"""A solve on the FFT passes whose wait for a copy timed out is reported, once, and what comes after is sound (the error
word is set from the host)."""
import pytest
import torch

import synthetic

pytestmark = pytest.mark.gpu

STATE, TIMEOUT = 4, 6


@pytest.fixture
def hrt():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_12913_gb300 import hrt as h
    yield h
    h.hrt_inject_wait_timeout(0)


def _raises(hrt, status, fn):
    with pytest.raises(hrt.HRTError) as e:
        fn()
    assert e.value.status == status, e.value


@pytest.mark.parametrize("adjoint", [False, True])
@pytest.mark.parametrize("n", [64, 256])
def test_a_solve_reports(hrt, n, adjoint):
    g = torch.Generator(device="cuda").manual_seed(n)
    pm, f = hrt.PM(n, float(n)), hrt.make_filter(4.0, 1.0)
    src = torch.randn((3, n, n, n) if adjoint else (n, n, n), device="cuda", generator=g)
    out = torch.empty((n, n, n) if adjoint else (3, n, n, n), device="cuda")

    def solve():
        (pm.solve_adjoint if adjoint else pm.solve)(src.clone(), 0.45, f, out)
        return out.clone()

    want = solve()
    pm.status()
    hrt.hrt_inject_wait_timeout(2)  # the second from here
    solve()
    pm.status()
    solve()
    _raises(hrt, TIMEOUT, pm.status)
    pm.status()  # reported once
    hrt.hrt_inject_wait_timeout(1)
    solve()
    _raises(hrt, TIMEOUT, solve)  # in place of the next solve
    assert torch.equal(solve(), want)
    pm.status()
    pm.close()


def test_sides_without_passes_have_nothing_to_report(hrt):
    pm = hrt.PM(60, 60.0)
    grad = torch.empty(3, 60, 60, 60, device="cuda")
    hrt.hrt_inject_wait_timeout(1)
    pm.solve(torch.ones(60, 60, 60, device="cuda"), 0.45, hrt.make_filter(), grad)
    pm.status()
    pm.close()


def test_objects_have_error_words_of_their_own(hrt):
    # more objects than the library's page has words, some given back in between
    f, rho = hrt.make_filter(4.0, 1.0), torch.ones(64, 64, 64, device="cuda")
    grad = torch.empty(3, 64, 64, 64, device="cuda")
    pms = [hrt.PM(64, 64.0) for _ in range(1030)]
    for i in range(0, 1030, 2):
        pms[i].close()
    for i in range(0, 1030, 2):
        pms[i] = hrt.PM(64, 64.0)
    for i in (0, 1, 514, 1029):
        hrt.hrt_inject_wait_timeout(1)
        pms[i].solve(rho, 0.45, f, grad)
    for i, pm in enumerate(pms):
        if i in (0, 1, 514, 1029):
            _raises(hrt, TIMEOUT, pm.status)
        pm.status()
        pm.close()


def _context(hrt):
    ctx = hrt.Context(hrt.make_config(64, 64.0, 32, observer=(32.0, 32.0, 0.0), n_sources=1))
    g = torch.Generator(device="cuda").manual_seed(2)
    disp = 0.3 * torch.randn(3, 32 ** 3, device="cuda", generator=g)
    mom = 0.1 * torch.randn(3, 32 ** 3, device="cuda", generator=g)
    theta = torch.tensor(synthetic.pixel_grid(32, 0.05), device="cuda")

    def start():
        ctx.hrt_init_particles(disp, mom, 1.0)
        ctx.hrt_init_rays(theta)

    return ctx, start


@pytest.mark.parametrize("call", ["hrt_step", "hrt_read_rays", "hrt_save_state", "hrt_ctx_kappa_power", "hrt_read_wait"])
def test_a_context_reports(hrt, call):
    ctx, start = _context(hrt)
    start()
    ctx.hrt_step(0.97, 0)
    want = ctx.hrt_read_rays()[0].clone()
    start()
    ctx.hrt_read_rays_async(torch.empty(32 * 32, 2, dtype=torch.float64).pin_memory())  # so that there is a copy to wait for
    hrt.hrt_inject_wait_timeout(1)
    ctx.hrt_step(0.97, 0)
    args = {"hrt_step": (0.95,), "hrt_ctx_kappa_power": (0, 32, 0.05 / 32, 4, 2.0, 60.0)}.get(call, ())
    _raises(hrt, TIMEOUT, lambda: getattr(ctx, call)(*args))
    _raises(hrt, STATE, lambda: ctx.hrt_step(0.95))  # no sound force
    start()  # the same context goes on from new particles
    ctx.hrt_step(0.97, 0)
    assert torch.allclose(ctx.hrt_read_rays()[0], want, rtol=0, atol=1e-6 * float(want.abs().max()))
    ctx.hrt_step(0.95)
    ctx.close()


def test_the_checks_report_and_clear(hrt):
    ctx, start = _context(hrt)
    ctx.hrt_set_nonfinite_check(True)
    start()
    hrt.hrt_inject_wait_timeout(1)
    _raises(hrt, TIMEOUT, lambda: ctx.hrt_step(0.97, 0))
    start()
    ctx.hrt_step(0.97, 0)
    ctx.close()


def test_the_adjoint_of_a_run_reports(hrt):
    ctx = hrt.Context(hrt.make_config(64, 64.0, 32, observer=(32.0, 32.0, 0.0), n_sources=1))
    ctx.hrt_set_checkpointing(1)
    noise = torch.randn(32 ** 3, device="cuda", generator=torch.Generator(device="cuda").manual_seed(4))

    def run():
        ctx.hrt_init_particles_zeldovich(noise, 0.9)
        ctx.hrt_step(1.0)
        ctx.hrt_sync_particles()
        ctx.hrt_init_rays(torch.tensor(synthetic.pixel_grid(32, 0.05), device="cuda"))
        ctx.hrt_step(0.97, 0)
        torch.cuda.synchronize()

    kbar = torch.ones(1, 32 * 32, device="cuda")
    run()
    want = ctx.hrt_adjoint(kbar)[0].clone()
    run()
    hrt.hrt_inject_wait_timeout(1)  # the first solve of the backward pass, recomputed or transposed
    _raises(hrt, TIMEOUT, lambda: ctx.hrt_adjoint(kbar))
    run()
    got = ctx.hrt_adjoint(kbar)[0]
    assert torch.allclose(got, want, rtol=0, atol=1e-4 * float(want.abs().max()))
    ctx.close()
