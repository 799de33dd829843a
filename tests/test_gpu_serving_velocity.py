"""Velocities of served frames.  The batch takes the SVD-free targets where the
stepper's FP32 frames take the SVD: two roundings of the same local step, so
against the FP64 oracle a served frame may be off by at most twice what the
stepper's frame is (positions and velocities), on a coarse one-layer shell and
a long thin slab, where the rounding of the targets moves the velocities most."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from workloads.meshes import slab_workload, sweater_shell  # noqa: E402

FRAMES, N_ITER = 5, 20


def _workloads():
    return {"shell": sweater_shell(seed=22, n_theta=24, n_z=7, n_r=1, dom_theta=2, dom_z=1),
            "slab": slab_workload(100, 6, 1, 0.01, 6, (2, 1), seed=5, n_iter=N_ITER)}


@pytest.mark.parametrize("name", ["shell", "slab"])
def test_served_velocities_are_as_exact_as_the_steppers(name):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from gpu_helpers import make_pair, rel
    from paper_2405_12484_gb300.sim import Server
    w = _workloads()[name]
    m, o = make_pair(w)
    x, v = w.rest.copy(), np.zeros_like(w.rest)
    for _ in range(FRAMES):
        x, v = o.step(x, v, None, w.gravity, N_ITER)
        m.step(None, w.gravity, N_ITER)
    m.sync()
    xs, vs = (a.cpu().numpy().astype(np.float64) for a in m.get_state())
    m.close()
    srv = Server(1 << 32, max_slots=4, n_iter=N_ITER)
    ids = [srv.submit(w, n) for n in (FRAMES - 1, FRAMES)]
    srv.run()
    before, after = (srv.fetch(i)[0].astype(np.float64) for i in ids)
    srv.close()
    assert rel(after, x) <= 2 * rel(xs, x)
    assert rel((after - before) / w.dt, v) <= 2 * rel(vs, v)
