"""Projections at the edges of the SVD-free path (det F > 0, J < 1.9,
lambda_1 <= 6 lambda_3, lambda_3 >= 0.04): elements just inside and just
outside each bound, coincident singular values and the rest state, through
pd_project (which mixes both paths within a warp) against the FP64 oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


def _cases():
    e = 1e-3
    sig = [(1, 1, 1), (1.2, 0.9, 0.9), (1.1, 1.1, 0.8), (1.3, 1.3, 1.3), (0.7, 0.7, 0.7)]
    for f in (1 - e, 1 + e):
        sig += [(1.9 * f, 1, 1), (1.24 * f, 1.24, 1.2357)]                       # J about 1.9
        sig += [(np.sqrt(6) * 0.6 * f, 0.8, 0.6), (np.sqrt(6) * 0.3 * f, 0.4, 0.3)]   # lambda_1 about 6 lambda_3
        sig += [(0.4, 0.3, 0.2 * f)]                                             # lambda_3 about 0.04
        sig += [(1.1, 0.9, -0.5 * f)]                                            # inverted
    return np.asarray(sig, np.float64)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 1000])
def test_targets_at_the_path_edges(n):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from oracle.projections import project_both
    from paper_2405_12484_gb300.sim import project
    rng = np.random.default_rng(n)
    sig = _cases()
    s = sig[rng.integers(0, len(sig), n)]

    def rot():
        q, r = np.linalg.qr(rng.standard_normal((n, 3, 3)))
        q *= np.sign(np.einsum("nii->ni", r))[:, None, :]
        q[np.linalg.det(q) < 0, :, 0] *= -1
        return q

    F = np.einsum("nij,nj,nkj->nik", rot(), s, rot()).astype(np.float32)
    R, V, sg = (a.cpu().numpy().astype(np.float64) for a in project(torch.as_tensor(F).cuda()))
    for k in range(n):
        Ro, Vo = project_both(F[k].astype(np.float64))[:2]
        so = np.linalg.svd(F[k].astype(np.float64))[1]
        kappa2 = (so[0] / so[2]) ** 2
        # F^T F carries the squared condition number; some 30 operations of half a unit each.  The volume
        # target's smallest factor moves 1 / rho_3 <= 10 times as fast as the data on these cases.
        tol = 30 * EPS * max(kappa2, 1.0)
        assert np.abs(R[k] - Ro).max() <= tol
        assert np.abs(V[k] - Vo).max() <= 10 * tol
        assert np.abs(np.abs(sg[k]) - so).max() <= tol * so[0]
