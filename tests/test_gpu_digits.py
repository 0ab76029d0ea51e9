"""The fixed-point solves (both contractions of the shifted solves exactly: on the tensor cores
above five states, in integer limbs up to five) against the pole-slot solve, the oracle and its own linearity."""
import numpy as np
import pytest

from oracle import rexi_coeffs as rc
from oracle import step as ostep
from oracle.swe import Consts
from paper_1812_03431_gb300 import inputs

pytestmark = pytest.mark.gpu
TOL = 1e-10    # against the oracle, as for every binary64 path
ORDER = 1e-13  # against the pole-slot solve: the same sums in another order
C = Consts()


def fieldwise(a, b):
    return max(np.linalg.norm(a[:, f] - b[:, f]) / max(np.linalg.norm(b[:, f]), 1e-300) for f in range(3))


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_1812_03431_gb300 import rexi
    rexi.load()
    return torch, rexi


def poles(P):
    """The middle P poles of a longer set (any P runs)."""
    al, be, _ = rc.rexi_coefficients(64, 0.2)
    k = (al.size - P) // 2
    return al[k:k + P], be[k:k + P]


def spectral_plan(rexi, N, B, al, be, tau=1800.0, **k):
    nlon = next(n for n in (12, 24, 48, 72, 96, 144, 192) if n >= 3 * N + 3)
    return rexi.Plan(N, nlon // 2, nlon, tau=tau, max_batch=B, layout="spectral", alpha=al, beta=be, **k)


# truncations down to one row per system; pole counts around a window of eight (above five
# states) and around 32 and 64 (up to five); batches around a tile of eight states
@pytest.mark.parametrize("N,P,B", [(1, 1, 5), (1, 1, 6), (1, 9, 8), (2, 7, 9), (3, 8, 5), (3, 8, 6), (8, 16, 16), (13, 17, 7), (21, 31, 17),
                                   (42, 57, 8), (63, 149, 6),
                                   (1, 1, 1), (2, 31, 1), (8, 32, 1), (13, 33, 1), (21, 64, 1), (42, 65, 1), (63, 149, 1),
                                   (3, 15, 2), (13, 17, 2), (21, 33, 2), (31, 100, 2), (5, 8, 3), (21, 9, 3), (31, 57, 4),
                                   (42, 149, 4)])
def test_matches_slot_solve(env, N, P, B):
    torch, rexi = env
    al, be = poles(P)
    x = torch.from_numpy(inputs.random_spectral(N, B, 7)).cuda()
    plan = spectral_plan(rexi, N, B, al, be)
    got, adj = plan.step(x).cpu().numpy(), plan.step_adjoint(x).cpu().numpy()  # the default
    for slots in (1, 2, 0, 1000):
        assert plan.set_pole_slots(B, slots, 5) >= 1
        y = plan.step(x).cpu().numpy()
        np.testing.assert_array_equal(y, plan.step(x).cpu().numpy())  # a fixed order
        assert fieldwise(y, got) < ORDER
        assert fieldwise(plan.step_adjoint(x).cpu().numpy(), adj) < ORDER
    plan.set_pole_slots(B, 1, 0)
    assert fieldwise(got, plan.step(x).cpu().numpy()) < ORDER
    assert fieldwise(adj, plan.step_adjoint(x).cpu().numpy()) < ORDER
    plan.close()


@pytest.mark.parametrize("B", [1, 2, 4, 8])
@pytest.mark.parametrize("field", [0, 1, 2])
def test_single_inputs_keep_the_rounding_of_binary64(env, B, field):
    """White noise in one input field, all poles of a set (their weights differ by 2^5): each output
    next to the pole-slot solve's.  A rounding of binary64 is 4e-17 rms; either side takes some eight
    of them (right-hand side, two recurrences, sum, row scale), together 1.6e-16; here four times that."""
    torch, rexi = env
    N = 42
    al, be, _ = rc.rexi_coefficients(64, 0.2)
    x = torch.zeros((B, 3, (N + 1) * (N + 2) // 2), dtype=torch.complex128)
    x[:, field] = torch.from_numpy(np.random.default_rng(field).standard_normal((2, B, x.shape[2]))[0] * (10.0, 1e-5, 1e-5)[field])
    x = x.cuda()
    plan, slots = spectral_plan(rexi, N, B, al, be), spectral_plan(rexi, N, B, al, be, pole_slots=8)
    assert fieldwise(plan.step(x).cpu().numpy(), slots.step(x).cpu().numpy()) < 3 * 2.0**-52
    plan.close()
    slots.close()


@pytest.mark.parametrize("N,M,B,tau", [(15, 32, 5, 3600.0), (31, 48, 10, 1200.0), (15, 32, 1, 3600.0), (31, 48, 3, 1200.0)])
def test_matches_oracle(env, N, M, B, tau):
    torch, rexi = env
    al, be, _ = rc.rexi_coefficients(M, 0.2)
    S = inputs.random_spectral(N, B, 5)
    plan = spectral_plan(rexi, N, B, al, be, tau)
    ref = ostep.rexi_step_spectral(S, N, al, be, tau, C)
    assert fieldwise(plan.step(torch.from_numpy(S).cuda()).cpu().numpy(), ref) < TOL
    plan.close()


@pytest.mark.parametrize("B", [11, 4])
def test_states_keep_their_own_scale(env, B):
    """Every group's fixed-point scale is a power of two of its own, so a state times a power of
    two gives that power times the result, bit for bit, whatever the other states hold."""
    torch, rexi = env
    N = 21
    al, be = poles(45)
    S = inputs.random_spectral(N, B, 9)
    scale = 2.0 ** np.array([0, 300, -300, 0, 60, -60, 500, 1, -1, 0, -450])[:B]
    T = S * scale[:, None, None]
    T[3] = 0.0
    plan = spectral_plan(rexi, N, B, al, be)
    a = plan.step(torch.from_numpy(S).cuda()).cpu().numpy() * scale[:, None, None]
    a[3] = 0.0
    np.testing.assert_array_equal(plan.step(torch.from_numpy(T).cuda()).cpu().numpy(), a)
    # fields of one state far apart in scale: no worse than the slot solve against the oracle
    S[:, 1:] *= 1e-9
    plan2 = spectral_plan(rexi, N, B, al, be, pole_slots=4)
    x = torch.from_numpy(S).cuda()
    assert fieldwise(plan.step(x).cpu().numpy(), plan2.step(x).cpu().numpy()) < ORDER
    plan.close()
    plan2.close()


@pytest.mark.parametrize("value,B,s", [(np.nan, 9, 4), (np.inf, 9, 8), (-np.inf, 9, 0), (np.nan, 1, 0), (np.inf, 2, 1),
                                       (-np.inf, 3, 2)])
def test_values_that_are_not_finite_stay_in_their_state_and_order(env, value, B, s):
    torch, rexi = env
    N = 21
    al, be = poles(45)
    S = inputs.random_spectral(N, B, 11)
    plan = spectral_plan(rexi, N, B, al, be)
    clean = plan.step(torch.from_numpy(S).cuda()).cpu().numpy()
    bad = S.copy()
    bad[s, 2, (N + 1) + 6] = value  # delta at m = 1, n = 7
    x = torch.from_numpy(bad).cuda()
    got = plan.step(x).cpu().numpy()
    plan.set_pole_slots(B, 4, 0)
    ref = plan.step(x).cpu().numpy()
    np.testing.assert_array_equal(np.isfinite(got), np.isfinite(ref))
    keep = np.arange(B) != s
    np.testing.assert_array_equal(got[keep], clean[keep])
    fine = np.isfinite(got[s])
    np.testing.assert_array_equal(got[s][fine], clean[s][fine])
    plan.close()


# rows around chunks of three, poles around windows of 32, one to five states
@pytest.mark.parametrize("N,P,B", [(1, 1, 1), (2, 32, 1), (3, 33, 1), (5, 64, 1), (7, 65, 1), (13, 100, 1), (63, 149, 1),
                                   (5, 16, 2), (13, 33, 2), (5, 9, 3), (21, 31, 4), (31, 57, 3), (8, 40, 5)])
def test_windows_shared_by_a_block(env, N, P, B):
    """Packing 3 (a block's warps share a window's rows) does the arithmetic of packing 1 in its order."""
    torch, rexi = env
    al, be = poles(P)
    plan = spectral_plan(rexi, N, B, al, be)
    x = torch.from_numpy(inputs.random_spectral(N, B, 11)).cuda()
    for slots in (1, 2):
        out = []
        for packing in (1, 3):
            assert plan.set_pole_slots(B, 65536 * packing + slots, 5) >> 16 == packing
            out.append((plan.step(x).cpu().numpy(), plan.step_adjoint(x).cpu().numpy()))
        np.testing.assert_array_equal(out[0][0], out[1][0])
        np.testing.assert_array_equal(out[0][1], out[1][1])
    plan.close()


@pytest.mark.parametrize("B", [8, 2])
def test_poles_of_unlike_scale_keep_the_other_solves(env, B):
    """Couplings of one pole that differ by more than eight bits from the middle pole's stay with
    the binary64 kernels, by default and on request."""
    torch, rexi = env
    N = 13
    al = np.array([-1e-3 + 0j, -1e3 + 1j, -1.0 + 2j])
    be = np.array([1e-3 + 0j, 1.0 + 1j, 0.5 - 1j])
    x = torch.from_numpy(inputs.random_spectral(N, B, 3)).cuda()
    plan, slots = spectral_plan(rexi, N, B, al, be), spectral_plan(rexi, N, B, al, be, pole_slots=1)
    assert fieldwise(plan.step(x).cpu().numpy(), slots.step(x).cpu().numpy()) < ORDER
    with pytest.raises(rexi.RexiError):
        plan.set_pole_slots(B, 0, 5)
    plan.close()
    slots.close()


@pytest.mark.parametrize("B", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("N,M", [(42, 64), (63, 128)])
def test_small_batches_of_a_larger_plan(env, N, M, B):
    """Batches below the tile of eight, on both sides of the rule's line, against the pole-slot solve."""
    torch, rexi = env
    al, be, _ = rc.rexi_coefficients(M, 0.2)
    x = torch.from_numpy(inputs.random_spectral(N, B, 13)).cuda()
    plan, slots = spectral_plan(rexi, N, 6, al, be), spectral_plan(rexi, N, 6, al, be, pole_slots=8)
    assert fieldwise(plan.step(x).cpu().numpy(), slots.step(x).cpu().numpy()) < ORDER
    assert fieldwise(plan.step_adjoint(x).cpu().numpy(), slots.step_adjoint(x).cpu().numpy()) < ORDER
    plan.close()
    slots.close()


@pytest.mark.parametrize("B,slots", [(8, 65536), (8, 2 * 65536 + 3), (2, 4 * 65536), (2, 7 * 65536 + 1)])
def test_packings_that_a_plan_does_not_have_are_refused(env, B, slots):
    """Packings are the limbs' (1 to 3); the layout in use stays."""
    torch, rexi = env
    al, be = poles(45)
    plan = spectral_plan(rexi, 13, B, al, be)
    x = torch.from_numpy(inputs.random_spectral(13, B, 3)).cuda()
    used = plan.set_pole_slots(B, 2, 5)
    y = plan.step(x).cpu().numpy()
    with pytest.raises(rexi.RexiError) as e:
        plan.set_pole_slots(B, slots, 5)
    assert e.value.status == rexi.REXI_EINVAL
    np.testing.assert_array_equal(plan.step(x).cpu().numpy(), y)
    assert plan.set_pole_slots(B, used, 5) == used  # what the call returned is taken back
    plan.close()


def test_the_adjoints_factors_wait_for_a_batch_that_they_serve(env):
    """One state in a plan for eight takes the binary64 factors only; eight states, or a call that
    chooses the fixed-point solve for one, the others as well; results as the slot solve's throughout."""
    torch, rexi = env
    N, P, B = 42, 149, 8
    al, be = poles(P)
    x = torch.from_numpy(inputs.random_spectral(N, B, 17)).cuda()
    slots = spectral_plan(rexi, N, B, al, be, pole_slots=4)
    want = slots.step_adjoint(x).cpu().numpy()
    binary64 = 9 * 16 * P * ((N + 1) * (N + 2) // 2 - 1)
    for choose in (False, True):
        plan = spectral_plan(rexi, N, B, al, be)
        start = plan.info()["device_bytes"]
        assert fieldwise(plan.step_adjoint(x[:1]).cpu().numpy(), want[:1]) < ORDER
        assert plan.info()["device_bytes"] == start + binary64
        if choose:
            plan.set_pole_slots(1, 0, 5)
        else:
            assert fieldwise(plan.step_adjoint(x).cpu().numpy(), want) < ORDER
        assert plan.info()["device_bytes"] > start + 2 * binary64
        assert fieldwise(plan.step_adjoint(x[:1]).cpu().numpy(), want[:1]) < ORDER
        plan.close()
    slots.close()


@pytest.mark.parametrize("N,P,B", [(1, 1, 1), (3, 26, 1), (8, 45, 2), (21, 31, 3), (31, 149, 4), (42, 65, 5)])
def test_small_batches_are_stepped_in_the_callers_layout(env, N, P, B):
    """No transposes around the limb solve, and the bits of the step that has them (rexi_integrate)."""
    torch, rexi = env
    al, be = poles(P)
    plan = spectral_plan(rexi, N, B, al, be)
    x = torch.from_numpy(inputs.random_spectral(N, B, 19)).cuda()
    plan.profile_enable(1)
    y = plan.step(x).cpu().numpy()
    st, _ = plan.profile_read()
    assert st["transpose_in"] == 0.0 and st["transpose_out"] == 0.0
    np.testing.assert_array_equal(y, plan.integrate(x, 1).cpu().numpy())
    plan.close()


@pytest.mark.parametrize("N", [4, 5, 8, 9])
@pytest.mark.parametrize("B", [1, 2, 4, 5])
def test_grid_steps_of_few_rows(env, N, B):
    """On both sides of the lines below which grid plans keep the fused solve."""
    torch, rexi = env
    al, be = poles(45)
    make = lambda **k: rexi.Plan(N, 12, 24, tau=1800.0, max_batch=B, alpha=al, beta=be, **k)  # noqa: E731
    plan, slots = make(), make(pole_slots=2)
    x = torch.from_numpy(inputs.random_grid(B, 12, 24, 3)).cuda()
    for f, g in ((plan.step, slots.step), (plan.step_adjoint, slots.step_adjoint)):
        assert fieldwise(f(x).cpu().numpy(), g(x).cpu().numpy()) < ORDER
    plan.close()
    slots.close()


@pytest.mark.parametrize("layout", ["spectral", "grid"])
def test_every_kernel_of_a_limb_step_has_its_stage(env, layout):
    """Up to five states the default is the limb solve, whose slots a second kernel sums."""
    torch, rexi = env
    N, B = 31, 4
    plan = rexi.Plan(N, 48, 96, M=32, max_batch=B, layout=layout)
    assert plan.info()["fixed_factors"] == 1
    S = torch.from_numpy(inputs.random_spectral(N, B, 9)).cuda()
    x = S if layout == "spectral" else plan.synthesize(S)
    plan.profile_enable(1)
    plan.step(x)
    st, n = plan.profile_read()
    ran = {"spectral": {"solve", "sums"}, "grid": {"fft_fwd", "leg_ana", "solve", "sums", "leg_syn", "fft_inv"}}[layout]
    assert n == 1 and {k for k, v in st.items() if v > 0} == ran
    plan.close()
