"""FP64 lattices at rest (GPU): a density of zero, alone or around a start confined to a part of
the lattice, is stepped in about the time of any other (its sites take neither form of the
collision), and stays exactly zero."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_03540_gb300 import build

    build.build()
    import paper_1711_03540_gb300 as lb

    return lb


def _time(lb, Q, Ns, r0, **kw):
    k = len(Ns)
    h = lb.lb_ks_batch_init(Q, Ns, Ns * 0.1, np.full(k, 1e-4), np.full(k, 2.0), r0, lb.lb_ks_default_opts(**kw))
    try:
        times = []
        for _ in range(7):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda.synchronize()
            a.record()
            lb.lb_ks_step(h, 64)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        out = np.empty(r0.size)
        lb.lb_ks_rho(h, out)
    finally:
        lb.lb_ks_free(h)
    return float(np.median(times[2:])), out


@pytest.mark.parametrize("Q", [5, 7])
@pytest.mark.parametrize("kernel", [0, 1])
def test_rest_costs_no_more_than_motion(lb, Q, kernel):
    """Both forms of the collision at a site take three times as long as one."""
    rng = np.random.default_rng(5)
    Ns = np.full(600, 1500, dtype=np.int64)
    moving = 0.05 * rng.standard_normal(Ns.sum())
    part = moving.copy()
    part.reshape(600, 1500)[:, 400:] = 0.0
    t, _ = _time(lb, Q, Ns, moving, kernel=kernel)
    t0, out = _time(lb, Q, Ns, np.zeros(Ns.sum()), kernel=kernel)
    t1, _ = _time(lb, Q, Ns, part, kernel=kernel)
    assert not out.any()
    assert t0 <= 1.5 * t, (t0, t)
    assert t1 <= 1.5 * t, (t1, t)
