"""Launch paths chosen by size or by use: long stages and narrow tiles of the
per-domain products (few blocks, a tile longer than the ring), and the solve
and the CG iterations replayed as graphs after a few calls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_helpers import f32, make_pair, rel  # noqa: E402

from workloads.meshes import slab_workload  # noqa: E402


def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("precision,refine", [("fp32", 0), ("tf32", 2), ("bf16", 2)])
@pytest.mark.parametrize("nx,ny,nz,domains", [(21, 19, 4, (2, 1)), (9, 40, 2, (1, 3)), (12, 12, 1, (4, 4))])
def test_solve_with_few_blocks(nx, ny, nz, domains, precision, refine):
    """Tiles of up to about 1,000 rows in a ring that holds fewer; FP32-level accuracy (1e-5, as the subspace solve's
    other tests: FP32 entries and sums, or two FP64-residual refinements)."""
    _need_gpu()
    w = slab_workload(nx, ny, nz, 0.01, 6, domains, seed=5, n_iter=1)
    m, o = make_pair(w, precision=precision, refine=refine)
    r = np.random.default_rng(nx).standard_normal((w.n_v, 3)).astype(np.float32)
    r[o.pin_ids] = 0.0
    x = m.solve(torch.as_tensor(r)).cpu().numpy()
    m.close()
    assert rel(x[o.free], o.chol.solve(r.astype(np.float64)[o.free])) < 1e-5


def test_solve_graph_repeats_and_follows_new_materials():
    _need_gpu()
    w = slab_workload(8, 8, 2, 0.01, 6, (2, 2), seed=2, n_iter=1)
    m, o = make_pair(w)
    rs = [torch.as_tensor(np.random.default_rng(k).standard_normal((w.n_v, 3)).astype(np.float32)) for k in range(2)]
    first = [m.solve(r).cpu() for r in rs]
    for _ in range(4):      # plain launches, then the graph
        for r, x in zip(rs, first):
            assert torch.equal(m.solve(r).cpu(), x)
    m.set_materials(3.0 * w.gamma_s, 3.0 * w.gamma_v)
    m.prefactor(w.dt)
    o.set_materials(f32(3.0 * w.gamma_s), f32(3.0 * w.gamma_v))
    for _ in range(6):
        x = m.solve(rs[0]).cpu().numpy()
        assert rel(x[o.free], o.chol.solve(rs[0].numpy().astype(np.float64)[o.free])) < 1e-5
    m.close()


@pytest.mark.parametrize("cg_iters", [1, 2, 3, 8, 9])
def test_cg_graph_repeats_bitwise(cg_iters):
    """Equilibrium steps whose linear solves run as plain launches, then from the graph: the same state bitwise."""
    _need_gpu()
    from paper_2405_12484_gb300.sim import Adjoint
    w = slab_workload(8, 8, 2, 0.01, 5, (2, 2), seed=4, n_iter=1)
    m, _ = make_pair(w, factor_oracle=False)
    a = Adjoint(m, cg_iters)
    x0 = torch.as_tensor(w.rest).cuda()
    states = []
    for k in range(6):
        if k == 3:      # a new factorisation drops the graphs
            m.prefactor(w.dt)
        a.set_state64(x0, torch.zeros_like(x0))
        a.equilibrium_step(torch.as_tensor(w.pin_targets(0), dtype=torch.float32), w.gravity, 5, 2)
        states.append(a.get_state64()[0].cpu())
    for s in states[1:]:
        assert torch.equal(s, states[0])
    a.close()
    m.close()
