"""Block inverse and products of the prefactorisation at the edges of their
64-wide blocks (one pivot, one more column, two and three pivots; one domain,
and two with an interface), with mild and with seven decades of element
stiffness, through pd_solve against the dense FP64 inverse of the oracle's
matrix."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_helpers import make_pair  # noqa: E402

from workloads.meshes import slab_workload  # noqa: E402


@pytest.mark.parametrize("decades", [1.0, 7.0])
@pytest.mark.parametrize("nx,domains", [(1, 1), (14, 1), (15, 1), (16, 1), (31, 1), (32, 1), (63, 2), (65, 3)])
def test_inverse_at_block_edges(nx, domains, decades):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    w = slab_workload(nx, 1, 1, 0.01, 6, (domains, 1), seed=3, n_iter=1, pin_edge=False)
    rng = np.random.default_rng(nx)
    w.gamma_s = 10.0 ** rng.uniform(0.0, decades, w.n_t)
    w.gamma_v = 10.0 * w.gamma_s
    m, o = make_pair(w)
    r = rng.standard_normal((w.n_v, 3)).astype(np.float32)
    x = m.solve(torch.as_tensor(r)).cpu().numpy().astype(np.float64)
    m.close()
    inv = np.linalg.inv(o.K_ff.toarray())
    # FP32 entries and FP32 sums over n terms, n the order of the matrix; each further level (boundary
    # modes, interface) repeats them on vectors bounded by the same |K^-1| |r|
    bound = (1 if domains == 1 else 4) * (w.n_v + 4) * 2.0 ** -24 * (np.abs(inv) @ np.abs(r))
    assert np.all(np.abs(x - inv @ r) <= bound)
