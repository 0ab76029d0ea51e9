"""The spectral step's error against long double arithmetic: the fixed-point solves' next to that of the
binary64 slot solve, which reads the same factors."""
import numpy as np
import pytest

from extended_util import CL, step_order
from oracle import rexi_coeffs as rc
from oracle.sphere import idx
from oracle.swe import Consts

pytestmark = pytest.mark.gpu
C = Consts()
# Either solve's own roundings (right-hand side, two recurrences, sum, row scale), some eight of 4e-17 rms
# binary64 roundings, add in quadrature to the error of the shared factors; four times their 1.6e-16 here.
OWN = 3 * 2.0**-52


@pytest.mark.parametrize("M", [64, 512])  # 151 and 1047 poles: |alpha| up to 15 and 105
@pytest.mark.parametrize("field", [0, 1, 2])
def test_fixed_point_steps_are_as_close_to_extended_precision(M, field):
    import torch
    from paper_1812_03431_gb300 import rexi
    N, B, tau = 42, 8, 1800.0
    al, be, _ = rc.rexi_coefficients(M, 0.2)
    n = (N + 1) * (N + 2) // 2
    g = np.random.default_rng(100 * M + field)
    S = np.zeros((B, 3, n), dtype=np.complex128)
    S[:, field] = (g.standard_normal((B, n)) + 1j * g.standard_normal((B, n))) * (10.0, 1e-5, 1e-5)[field]
    S[..., :N + 1].imag = 0.0
    S[:, 1:, 0] = 0.0
    ref = np.zeros(S.shape, dtype=CL)
    for m in range(N + 1):
        ref[..., idx(m, m, N):idx(m, N, N) + 1] = step_order(S, m, N, al, be, tau, C)
    x = torch.from_numpy(S).cuda()

    def errors(max_batch, **k):
        plan = rexi.Plan(N, 64, 128, tau=tau, max_batch=max_batch, layout="spectral", alpha=al, beta=be, **k)
        kind = plan.info()["fixed_factors"]
        y = np.concatenate([plan.step(x[i:i + max_batch].contiguous()).cpu().numpy() for i in range(0, B, max_batch)])
        plan.close()
        return kind, [float(np.linalg.norm(y[:, f] - ref[:, f]) / np.linalg.norm(ref[:, f])) for f in range(3)]

    _, slots = errors(B, pole_slots=8)
    assert max(slots) < 1e-13
    for max_batch, kind in ((1, 1), (4, 1), (B, 2)):
        k, fixed = errors(max_batch)
        assert k == kind
        for a, b in zip(fixed, slots):
            assert a * a <= b * b + OWN * OWN
