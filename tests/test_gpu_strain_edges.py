"""Accuracy of the SVD-free targets up to their bounds (J^2 = 3.6,
lambda_1 = 4.5 lambda_3, lambda_3 = 1/4, lambda_1 lambda_3 = 0.14), through
pd_project against the FP64 oracle: root-mean-square errors over many orientations, u = 2^-24.

R = F C^-1/2: the entries of C carry u s_1^2 each, which F h(C) turns into
s_1 (1/2) s_3^-3 sqrt(6) u s_1^2 = 1.2 u kappa^3; the eigenvalues' own errors and
the ten roundings of the evaluation are of the same size: 4 u kappa^3 in all.
V = F h(C), where a change of lambda_3 moves the target by up to 1 + s_3 / r_3
(r_3 = sqrt(lambda_3 + 4 mu)) times as much, and the product of the targets is
one to 3e-7 = 5 u only.  sigma: u l_1 sqrt(6) / (2 s_3) = 1.2 u kappa s_1 and as
much again from the eigenvalues: 4 u kappa s_1."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from strain_cases import accepted, cases, gradients, root  # noqa: E402

U = 2.0 ** -24


@pytest.mark.parametrize("k", [k for k, s in enumerate(cases()) if accepted(s)])
def test_rms_error_up_to_the_bounds(k):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from oracle.projections import project_both
    from paper_2405_12484_gb300.sim import project
    s = cases()[k]
    F = gradients(np.random.default_rng(k), s, 2000)
    R, V, sg = (a.cpu().numpy().astype(np.float64) for a in project(torch.as_tensor(F).cuda()))
    Ro, Vo = project_both(F.astype(np.float64))[:2]
    so = np.linalg.svd(F.astype(np.float64))[1]
    kappa, l3, mu = s.max() / s.min(), s.min() ** 2, root(s)
    grow, d1 = 1.0 + s.min() / np.sqrt(l3 + 4 * mu), 0.5 * (s.max() + np.sqrt(s.max() ** 2 + 4 * mu))
    rms = lambda a: np.sqrt(np.mean(a ** 2, axis=0)).max()     # noqa: E731
    assert rms(R - Ro) <= 4 * U * kappa ** 3
    assert rms(V - Vo) <= grow * 4 * U * kappa ** 3 + 5 * U * d1
    assert rms(sg - so) <= 4 * U * kappa * s.max()
