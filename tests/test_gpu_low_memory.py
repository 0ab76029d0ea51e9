"""Plans on a nearly full device: what a plan needs comes first, the fixed-point forms of its factors and
tables only where they leave room, and without them the binary64 kernels give the same results."""
import contextlib

import numpy as np
import pytest

from oracle import rexi_coeffs as rc
from paper_1812_03431_gb300 import inputs

pytestmark = pytest.mark.gpu
ORDER = 1e-13  # the same sums in another order
MB = 1 << 20


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_1812_03431_gb300 import rexi
    rexi.load()
    return torch, rexi


@contextlib.contextmanager
def only(torch, nbytes):
    """Leaves `nbytes` of the device free."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    if free < nbytes + 64 * MB:
        pytest.skip("the device has no such memory free")
    hold = torch.empty(free - nbytes, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        torch.cuda.synchronize()
        del hold
        torch.cuda.empty_cache()


def fieldwise(a, b):
    return max(np.linalg.norm(a[:, f] - b[:, f]) / max(np.linalg.norm(b[:, f]), 1e-300) for f in range(3))


def test_a_plan_that_fits_without_the_fixed_point_factors_is_created(env):
    """60 MB less than the plan takes with its digits, which are 100 MB of it."""
    torch, rexi = env
    N, B = 63, 64
    al, be, _ = rc.rexi_coefficients(128, 0.2)
    make = lambda: rexi.Plan(N, 96, 192, tau=1800.0, max_batch=B, layout="spectral", alpha=al, beta=be)  # noqa: E731
    x = torch.from_numpy(inputs.random_spectral(N, B, 3)).cuda()
    full = make()
    want, info = full.step(x).cpu().numpy(), full.info()
    full.close()
    assert info["fixed_factors"] == 2
    out = torch.empty_like(x)
    with only(torch, info["device_bytes"] - 60 * MB):
        plan = make()
        assert plan.info()["fixed_factors"] == 0
        got = plan.step(x, out=out).cpu().numpy()
        plan.close()
    assert fieldwise(got, want) < ORDER


def test_transforms_and_steps_without_any_fixed_point_form(env):
    """40 MB less than the plan takes with its Legendre digits (twice the 101 MB of the tables they replace)
    and its solve's factors (some 150): 210 MB beside what it needs, a third of which holds neither."""
    torch, rexi = env
    N, nlat, nlon, B = 255, 384, 768, 2
    al, be, _ = rc.rexi_coefficients(32, 0.2)
    k = al.size // 2
    make = lambda: rexi.Plan(N, nlat, nlon, tau=600.0, max_batch=B, alpha=al[k - 2:k + 3], beta=be[k - 2:k + 3])  # noqa: E731
    S = torch.from_numpy(inputs.random_spectral(N, B, 5)).cuda()
    g = torch.from_numpy(inputs.random_grid(B, nlat, nlon, 4)).cuda()
    run = lambda p: [v.cpu().numpy() for v in (p.analyze(g), p.synthesize(S), p.step(g), p.step_adjoint(g))]  # noqa: E731
    full = make()
    info, want = full.info(), run(full)
    full.close()
    assert info["fixed_factors"] == 1
    tables = (N + 1) * (N + 2) // 2 * (nlat // 2) * 16  # Pbar and H in binary64; as digits twice that
    with only(torch, info["device_bytes"] - 40 * MB):
        plan = make()
        low = plan.info()
        got = run(plan)
        plan.close()
    assert low["fixed_factors"] == 0 and low["device_bytes"] < info["device_bytes"] - tables
    for a, b in zip(got, want):  # sums of up to 192 terms and two transforms: as against the oracle elsewhere
        assert fieldwise(a, b) < 1e-11


@pytest.mark.parametrize("B", [8, 2])
def test_the_adjoint_takes_no_more_than_its_share(env, B):
    """Room for the adjoint's binary64 factors and as much as its fixed-point ones take: more than a third."""
    torch, rexi = env
    N, P = 127, 151
    al, be, _ = rc.rexi_coefficients(64, 0.2)
    k = (al.size - P) // 2
    make = lambda: rexi.Plan(N, 192, 384, tau=1200.0, max_batch=B, layout="spectral", alpha=al[k:k + P], beta=be[k:k + P])  # noqa: E731
    g = torch.from_numpy(inputs.random_spectral(N, B, 6)).cuda()
    full = make()
    want = full.step_adjoint(g).cpu().numpy()
    with_both = full.info()["device_bytes"]
    full.close()
    plan = make()
    before = plan.info()["device_bytes"]
    binary64 = 9 * 16 * P * ((N + 1) * (N + 2) // 2 - 1)
    fixed = with_both - before - binary64
    assert fixed > 40 * MB
    out = torch.empty_like(g)
    with only(torch, binary64 + fixed + 32 * MB):
        got = plan.step_adjoint(g, out=out).cpu().numpy()
        assert plan.info()["device_bytes"] - before < binary64 + 2 * MB
    assert fieldwise(got, want) < ORDER
    plan.close()
