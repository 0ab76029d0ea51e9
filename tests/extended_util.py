"""The spectral step for single zonal orders in numpy's long double (80 bits on x86, 113 on Arm)."""
import numpy as np

from oracle.sphere import idx

L, CL = np.longdouble, np.clongdouble


def step_order(S, m, N, alpha, beta, tau, c):
    """sum_k beta_k (alpha_k + tau L_m)^-1 of states S [B, 3, nspec] at zonal order m: [B, 3, N - m + 1].
    Phi and zeta eliminated, one tridiagonal system in delta per parity and pole."""
    al, be, tau = np.asarray(alpha, dtype=CL), np.asarray(beta, dtype=CL), L(tau)
    lo = max(m, 1)
    e = lambda n: np.sqrt(L(n * n - m * m) / L(4 * n * n - 1)) if n > m else L(0)  # noqa: E731
    two = 2 * L(c.omega)
    C = {n: two * e(n) * L(n + 1) / L(n) if n - 1 >= lo else L(0) for n in range(lo, N + 2)}
    D = {n: two * e(n + 1) * L(n) / L(n + 1) if lo <= n < N else L(0) for n in range(lo - 1, N + 1)}
    G = {n: L(n * (n + 1)) / L(c.radius) ** 2 for n in range(lo, N + 1)}
    s = {n: al + 1j * tau * two * L(m) / L(n * (n + 1)) for n in range(lo, N + 1)}
    pb = L(c.gravity) * L(c.mean_depth)
    x = S[..., idx(m, m, N):idx(m, N, N) + 1].astype(CL)
    f0, z0, d0 = ({n: x[:, f, n - m][:, None] for n in range(lo, N + 1)} for f in range(3))
    delta = {}
    for first in (lo, lo + 1):
        rows = list(range(first, N + 1, 2))
        diag, up, y = {}, {}, {}
        for n in rows:
            a, r = s[n] + tau * tau * pb * G[n] / al, d0[n] - tau * G[n] * f0[n] / al
            low, up[n] = 0, 0
            if n - 1 >= lo:
                a, r = a + tau * tau * C[n] * D[n - 1] / s[n - 1], r - tau * C[n] * z0[n - 1] / s[n - 1]
                low = tau * tau * C[n] * C.get(n - 1, L(0)) / s[n - 1]
            if n + 1 <= N:
                a, r = a + tau * tau * D[n] * C[n + 1] / s[n + 1], r - tau * D[n] * z0[n + 1] / s[n + 1]
                up[n] = tau * tau * D[n] * D[n + 1] / s[n + 1]
            if n > first:
                w = low / diag[n - 2]
                a, r = a - w * up[n - 2], r - w * y[n - 2]
            diag[n], y[n] = a, r
        for n in reversed(rows):
            delta[n] = (y[n] - (up[n] * delta[n + 2] if n + 2 in delta else 0)) / diag[n]
    out = np.zeros(x.shape, dtype=CL)
    for n in range(lo, N + 1):
        z = z0[n] + tau * (C[n] * delta[n - 1] if n - 1 >= lo else 0) + tau * (D[n] * delta[n + 1] if n + 1 <= N else 0)
        out[:, 0, n - m] = ((f0[n] + tau * pb * delta[n]) / al * be).sum(-1)
        out[:, 1, n - m] = (z / s[n] * be).sum(-1)
        out[:, 2, n - m] = (delta[n] * be).sum(-1)
    if m == 0:
        out[:, 0, 0] = x[:, 0, 0] * (be / al).sum()  # n = 0: Phi only
        out = out.real.astype(CL)
    return out
