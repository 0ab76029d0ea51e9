"""The FP64 form's transforms (Legendre sums as exact fixed-point products on the tensor cores)
against the oracle's, at the edges of their tiles: 16 degrees or latitudes, groups of 64 terms,
four states."""
import numpy as np
import pytest

from oracle import sphere
from paper_1812_03431_gb300 import inputs

pytestmark = pytest.mark.gpu
A, G = inputs.EARTH["radius"], inputs.EARTH["gravity"]
TOL = 1e-11  # sums of up to 130 terms with weights up to 1 / (1 - mu^2) ~ 3e3: 130 x 3e3 x 2^-53 = 4e-11 at worst


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_1812_03431_gb300 import rexi
    rexi.load()
    return torch, rexi


def oracle_analysis(g, x):
    cos = g.coslat[:, None]
    zeta, delta = g.uv_to_vortdiv(x[:, 1] * cos, x[:, 2] * cos, A)
    return np.stack([G * g.analysis(x[:, 0]), zeta, delta], axis=1)


def oracle_synthesis(g, S):
    u, v = g.vortdiv_to_uv(S[:, 1], S[:, 2], A)
    return np.stack([g.synthesis(S[:, 0]) / G, u / g.coslat[:, None], v / g.coslat[:, None]], axis=1)


# (N, nlat, nlon, states): one to 66 degrees per class, 2 to 65 latitude pairs
@pytest.mark.parametrize("N,nlat,nlon,B", [(1, 4, 8, 1), (2, 6, 12, 2), (15, 32, 48, 4), (16, 34, 48, 5), (30, 64, 96, 3),
                                           (31, 66, 96, 8), (33, 128, 108, 9), (63, 130, 192, 1), (64, 96, 200, 2),
                                           (130, 132, 400, 1)])
def test_transforms_match_oracle(env, N, nlat, nlon, B):
    torch, rexi = env
    plan = rexi.Plan(N, nlat, nlon, M=8, max_batch=B)
    g = sphere.Grid(N, nlat, nlon)
    x = inputs.random_grid(B, nlat, nlon, 3)  # white noise: every latitude counts
    got = plan.analyze(torch.from_numpy(x).cuda()).cpu().numpy()
    ref = oracle_analysis(g, x)
    ref[:, 1:, 0] = got[:, 1:, 0]  # zeta_0^0 and delta_0^0 are not state
    S = inputs.random_spectral(N, B, 5, slope=0.0)  # white spectrum: every degree counts
    grid = plan.synthesize(torch.from_numpy(S).cuda()).cpu().numpy()
    want = oracle_synthesis(g, S)
    for f in range(3):
        assert np.linalg.norm(got[:, f] - ref[:, f]) < TOL * np.linalg.norm(ref[:, f])
        assert np.linalg.norm(grid[:, f] - want[:, f]) < TOL * np.linalg.norm(want[:, f])
    plan.close()


@pytest.mark.parametrize("N,nlat,nlon", [(1, 2, 4), (2, 4, 8), (15, 32, 48), (16, 36, 48), (31, 64, 96), (33, 128, 108),
                                         (66, 132, 200), (127, 192, 384)])
def test_one_state_alone_as_in_a_batch(env, N, nlat, nlon):
    """A single state's fields share a column tile; each product is exact up to 2^-59 of its group and
    is rounded as in a batch, the sums over groups in another order (up to four of them)."""
    torch, rexi = env
    plan = rexi.Plan(N, nlat, nlon, M=8, max_batch=2)
    x = torch.from_numpy(inputs.random_grid(2, nlat, nlon, 7)).cuda()
    S = torch.from_numpy(inputs.random_spectral(N, 2, 8, slope=0.0)).cuda()
    for f, v in ((plan.analyze, x), (plan.synthesize, S)):
        one, two = f(v[1:].contiguous()).cpu().numpy()[0], f(v).cpu().numpy()[1]
        for k in range(3):
            assert np.linalg.norm(one[k] - two[k]) <= 4 * 2.0**-52 * np.linalg.norm(two[k])
    plan.close()


def test_scales_and_values_that_are_not_finite_stay_in_their_state(env):
    """Groups are scaled per state and order by powers of two: a power of two times a state gives
    that power times its result, bit for bit, and a NaN reaches no other state."""
    torch, rexi = env
    N, nlat, nlon, B = 20, 40, 64, 6
    plan = rexi.Plan(N, nlat, nlon, M=8, max_batch=B)
    x = inputs.random_grid(B, nlat, nlon, 3)
    S = inputs.random_spectral(N, B, 5)
    scale = 2.0 ** np.array([0, 200, -200, 3, 0, -1])
    run = lambda a: plan.analyze(torch.from_numpy(a).cuda()).cpu().numpy()  # noqa: E731
    syn = lambda a: plan.synthesize(torch.from_numpy(a).cuda()).cpu().numpy()  # noqa: E731
    a, s = run(x), syn(S)
    np.testing.assert_array_equal(run(x * scale[:, None, None, None]), a * scale[:, None, None])
    np.testing.assert_array_equal(syn(S * scale[:, None, None]), s * scale[:, None, None, None])
    x[3, 0, 7, 9] = np.nan
    S[3, 1, 30] = np.inf
    b, t = run(x), syn(S)
    keep = np.arange(B) != 3
    np.testing.assert_array_equal(b[keep], a[keep])
    np.testing.assert_array_equal(t[keep], s[keep])
    assert not np.isfinite(b[3, 0]).any() and np.isfinite(b[3, 1:]).all()  # h' reaches Phi only
    assert not np.isfinite(t[3, 1]).all() and np.isfinite(t[3, 0]).all()   # zeta reaches the wind only
    plan.close()


@pytest.mark.parametrize("nlon", [8, 10, 16, 18, 24, 30, 64, 90, 100, 250, 486, 1024, 2000])
def test_longitude_transforms(env, nlon):
    """Every radix and row length against the oracle, for rows that a common scale suits least: one
    point among zeros, one field 1e-9 of the others, a constant row."""
    torch, rexi = env
    N, nlat, B = min(3, nlon // 2 - 1), 6, 3
    plan = rexi.Plan(N, nlat, nlon, M=8, max_batch=B)
    g = sphere.Grid(N, nlat, nlon)
    x = inputs.random_grid(B, nlat, nlon, 8)
    x[0] = 0.0
    x[0, :, 2, nlon // 3] = 1.0
    x[1, 0] *= 1e-9
    x[2, 1] = 7.0
    got = plan.analyze(torch.from_numpy(x).cuda()).cpu().numpy()
    ref = oracle_analysis(g, x)
    ref[:, 1:, 0] = got[:, 1:, 0]
    S = got.copy()
    grid = plan.synthesize(torch.from_numpy(S).cuda()).cpu().numpy()
    want = oracle_synthesis(g, S)
    for b in range(B):
        assert np.linalg.norm(got[b, 0] - ref[b, 0]) < TOL * np.linalg.norm(ref[b, 0])
        assert np.linalg.norm(got[b, 1:] - ref[b, 1:]) < TOL * np.linalg.norm(ref[b, 1:])
        assert np.linalg.norm(grid[b, 0] - want[b, 0]) < TOL * np.linalg.norm(want[b, 0])
        assert np.linalg.norm(grid[b, 1:] - want[b, 1:]) < TOL * np.linalg.norm(want[b, 1:])
    plan.close()


@pytest.mark.parametrize("N,nlat,nlon", [(42, 64, 128), (63, 96, 192)])
@pytest.mark.parametrize("B", [1, 2])
def test_a_smooth_flow_among_small_coefficients(env, N, nlat, nlon, B):
    """One zonal coefficient, alone and with noise of 1e-4 of it in every degree: the winds are those of
    either alone, within three roundings (the synthesis' groups hold low and high degrees)."""
    torch, rexi = env
    plan = rexi.Plan(N, nlat, nlon, M=8, max_batch=B)
    small = inputs.random_spectral(N, B, 9) * 1e-4
    big = np.zeros_like(small)
    big[:, 1, 1] = 10 * np.abs(inputs.random_spectral(N, B, 9)[:, 1]).max()
    wind = lambda s: plan.synthesize(torch.from_numpy(s).cuda()).cpu().numpy()[:, 1:]
    both, alone = wind(big + small), wind(big)
    assert np.linalg.norm(both - wind(small) - alone) < 3 * 2.0**-52 * np.linalg.norm(alone)
    plan.close()


# batches whose CTAs of one state fill two (304, analysis) or four (608, synthesis) places per SM or just do
# not, and the same states fewer at a time
@pytest.mark.parametrize("N,nlat,nlon,B,few", [(1, 2, 4, 153, 152), (2, 4, 8, 103, 7), (15, 32, 48, 20, 3), (16, 36, 48, 18, 17),
                                               (31, 64, 96, 10, 9), (33, 128, 108, 9, 4), (37, 76, 120, 9, 8),
                                               (66, 132, 200, 5, 2), (127, 192, 384, 3, 2), (130, 132, 400, 3, 2),
                                               (15, 32, 48, 39, 38), (16, 36, 48, 36, 35), (31, 64, 96, 20, 19), (33, 128, 108, 18, 5),
                                               (66, 132, 200, 10, 9), (127, 192, 384, 5, 4)])
def test_one_and_four_states_per_block(env, N, nlat, nlon, B, few):
    """Each product is exact up to 2^-59 of its group and rounded alike in both forms, the sums over the
    groups are in another order (up to four of them)."""
    torch, rexi = env
    plan = rexi.Plan(N, nlat, nlon, M=8, max_batch=B)
    x = torch.from_numpy(inputs.random_grid(B, nlat, nlon, 11)).cuda()
    S = torch.from_numpy(inputs.random_spectral(N, B, 12, slope=0.0)).cuda()
    for f, v in ((plan.analyze, x), (plan.synthesize, S)):
        four = f(v).cpu().numpy()
        one = np.concatenate([f(v[i:i + few].contiguous()).cpu().numpy() for i in range(0, B, few)])
        for b in range(B):
            for k in range(3):
                assert np.linalg.norm(one[b, k] - four[b, k]) <= 4 * 2.0**-52 * np.linalg.norm(four[b, k])
    plan.close()
