"""Singular values inside and outside the bounds of the SVD-free targets
(proj3.cuh strain_of), and the rule itself in FP64."""
import numpy as np

E = 1e-3     # distance from a bound


def root(s):
    """mu of d_i (d_i - s_i) = mu, prod d_i = 1, every d_i the larger root; None where there is none."""
    s = np.abs(np.asarray(s, np.float64))
    f = lambda mu: np.prod(0.5 * (s + np.sqrt(np.maximum(s * s + 4 * mu, 0.0)))) - 1.0     # noqa: E731
    lo, hi = -0.25 * s.min() ** 2, 4.0
    if f(lo) >= 0:
        return None
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if f(mid) < 0 else (lo, mid)
    return 0.5 * (lo + hi)


def accepted(s):
    """What the path takes: J > 0, J^2 < 3.6, lambda_1 <= 4.5 lambda_3, lambda_3 >= 1/4, lambda_1 lambda_3 >= 0.14 and
    mu >= -0.24 lambda_3."""
    s, l1, l3 = np.asarray(s, np.float64), np.abs(s).max() ** 2, np.abs(s).min() ** 2
    if np.prod(s) <= 0 or np.prod(s) ** 2 >= 3.6 or l3 < 0.25 or l1 * l3 < 0.14 or l1 > 4.5 * l3:
        return False
    mu = root(s)
    return mu is not None and mu >= -0.24 * l3


def cases():
    J = np.sqrt(3.6)
    out = [(1, 1, 1), (1.2, 0.9, 0.9), (1.1, 1.1, 0.8), (0.7, 0.7, 0.7), (1.3, 1.0, 0.7), (0.98, 1.01, 1.0)]
    for f in (1 - E, 1 + E):
        out += [(J * f, 1, 1), (J ** (1 / 3) * f, J ** (1 / 3), J ** (1 / 3)), (1.5 * f, 1.3, J / 1.95)]     # J
        out += [(1.5, 1.5, 0.84 * f), (1.6 * f, 1.2, 0.98)]                                                  # J about 1.89
        out += [(np.sqrt(6) * 0.6 * f, 0.8, 0.6), (np.sqrt(6) * 0.3 * f, 0.4, 0.3)]                          # beyond the
        out += [(0.4, 0.3, 0.2 * f), (0.2 * f, 0.2 * f, 0.2 * f)]                                            # bounds
        out += [(np.sqrt(4.5) * 0.65 * f, 0.8, 0.65), (np.sqrt(4.5) * 0.6 * f, 0.6, 0.6)]                        # the ratio
        out += [(np.sqrt(4.5) * 0.7 * f, np.sqrt(4.5) * 0.695, 0.7)]
        out += [(1.0, 0.7, 0.5 * f), (0.9, 0.5 * f, 0.5 * f)]                                                # lambda_3
        out += [(0.68 * f, 0.6, np.sqrt(0.14) / 0.68), (0.14 ** 0.25 * f, 0.14 ** 0.25 * f, 0.14 ** 0.25 * f)]   # both
        out += [(1.1, 0.9, -0.5 * f)]                                                                        # det F
        # the floor of mu at J = 1.85: s_3 where mu = -0.24 lambda_3 along (1.85 / (1.5 t), 1.5, t), and a clear miss
        t = FLOOR_T * (1 + 5 * (f - 1))
        out += [(1.85 / (1.5 * t), 1.5, t), (1.7, 1.6, 0.695 * f)]
    return np.asarray(out, np.float64)


def _floor_t():
    lo, hi = 0.70, 0.80     # mu / lambda_3 rises through -0.24 between them
    g = lambda t: root((1.85 / (1.5 * t), 1.5, t)) / t ** 2 + 0.24     # noqa: E731
    assert g(lo) < 0 < g(hi)
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if g(mid) < 0 else (lo, mid)
    return 0.5 * (lo + hi)


FLOOR_T = _floor_t()


def rotations(rng, n):
    q, r = np.linalg.qr(rng.standard_normal((n, 3, 3)))
    q *= np.sign(np.einsum("nii->ni", r))[:, None, :]
    q[np.linalg.det(q) < 0, :, 0] *= -1
    return q


def gradients(rng, s, n):
    """n deformation gradients with singular values s, float32."""
    return np.einsum("nij,j,nkj->nik", rotations(rng, n), s, rotations(rng, n)).astype(np.float32)
