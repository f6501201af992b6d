"""The autotuner (GPU): a tuned handle starts from its initial state, cleared of the trials', and
its run gives the untuned handle's bits."""
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


def _state(lb, h):
    buf = np.zeros(lb.lb_ks_state_bytes(h), dtype=np.uint8)
    lb.lb_ks_save(h, buf)
    return buf


@pytest.mark.parametrize("prec,kernel,recentre", [(0, 0, 0), (0, 0, 70), (1, 0, 70), (0, 4, 0), (1, 4, 70)])
def test_tuned_equals_untuned(lb, prec, kernel, recentre):
    rng = np.random.default_rng(29)
    Ns = np.array([61, 300, 1500, 4096, 6000], dtype=np.int64)
    r0 = np.concatenate([0.02 * rng.standard_normal(n) for n in Ns])
    dx, dt, tau = (0.2, 5e-5, 1.0) if kernel == 4 else (0.1, 1e-4, 2.0)
    runs = []
    for tune in (0, 1):
        h = lb.lb_ks_batch_init(7, Ns, Ns * dx, np.full(5, dt), np.full(5, tau), r0, lb.lb_ks_default_opts(
            precision=prec, kernel=kernel, recentre_every=recentre, autotune=tune))
        try:
            assert lb.lb_ks_steps_done(h) == 0
            state = [_state(lb, h)]
            lb.lb_ks_step(h, 201)
            state.append(_state(lb, h))
        finally:
            lb.lb_ks_free(h)
        runs.append(state)
    for a, b in zip(*runs):
        np.testing.assert_array_equal(a, b)
