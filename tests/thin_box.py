"""One right-hand side of a rectilinear box in extended precision (numpy
longdouble), for elements much wider than high, with the sizes that bound the
rounding of any evaluation: the tests of the FP64 kernels on thin elements."""
import numpy as np

from .helpers import lobatto_derivative

LD = np.longdouble


def _derivative(N):
    D = lobatto_derivative(N)
    return np.array([[LD(float(v)) + LD(float(v - type(v)(float(v)))) for v in row] for row in D])


def thin_flow(m, cfg):
    """Smooth flow of 20 m/s with W ~ U dz/dx and a pressure perturbation of some
    100 Pa, a different phase in every variable."""
    L = cfg["L"]
    x, y, z = (m.coords()[d] / L[d] for d in range(3))
    rho0, th0 = m.ref()[:2]
    q = np.empty((5, m.Ng))
    wave = lambda a, b, c, p: np.sin(2.1 * a * x + p) * np.cos(1.7 * b * y - p) * np.cos(1.9 * c * z + 0.3 * p)  # noqa: E731
    q[0] = 1e-3 * rho0 * wave(1, 1, 1, 0.4)
    q[1] = 20.0 * rho0 * wave(1, 1, 1, 0.9)
    q[2] = 15.0 * rho0 * wave(1, 1, 1, 1.7)
    q[3] = 20.0 * L[2] / L[0] * rho0 * wave(1, 1, 1, 2.3)
    q[4] = 1e-3 * th0 * wave(1, 1, 1, 3.1)
    return q


def thin_rhs(m, cfg, q, dtype=LD):
    """R [5][Ng] of a walled box of straight elements, and per variable
    S = max sum_c K_c |D| |F_c|, K_c = 2 / h_c: what a sum of products is rounded
    relative to."""
    N, ne, L = cfg["N"], cfg["ne"], cfg["L"]
    D = _derivative(N).astype(dtype)
    n = [ne[d] * N + 1 for d in range(3)]
    f = lambda a: np.asarray(a, dtype=dtype).reshape(n[2], n[1], n[0])  # noqa: E731
    rho0, th0, p0 = (f(v) for v in m.ref()[:3])
    rp, U, tp = f(q[0]), [f(q[1 + c]) for c in range(3)], f(q[4])
    rho, gam = rho0 + rp, dtype(cfg["cp"]) / dtype(cfg["cv"])
    u, theta = [Uc / rho for Uc in U], (th0 + tp) / rho
    pp = p0 * np.expm1(gam * np.log1p(tp / th0))

    def deriv(F, c, A):
        F = np.moveaxis(F, 2 - c, 0)
        out, cnt = np.zeros_like(F), np.zeros(n[c], dtype=dtype)
        for e in range(ne[c]):
            s = slice(e * N, (e + 1) * N + 1)
            out[s] += np.tensordot(A, F[s], axes=(1, 0))
            cnt[s] += 1
        out = out / cnt[:, None, None] * (dtype(2 * ne[c]) / dtype(L[c]))
        return np.moveaxis(out, 0, 2 - c)

    R, S = np.zeros((5,) + rho.shape, dtype=dtype), np.zeros(5)
    for v in range(5):
        F = U if v == 0 else [theta * Uc for Uc in U] if v == 4 else [U[c] * u[v - 1] + (pp if c == v - 1 else 0) for c in range(3)]
        t = [deriv(F[c], c, D) for c in range(3)]
        R[v] = -(t[0] + t[1] + t[2])
        S[v] = float(sum(deriv(np.abs(F[c]), c, np.abs(D)) for c in range(3)).max())
    R[3] -= rp * dtype(cfg["g"])
    for c in range(3):  # walls: no normal momentum tendency
        w = np.moveaxis(R[1 + c], 2 - c, 0)
        w[0] = w[-1] = 0
    return R.reshape(5, -1), S
