"""FP64 storage where its fixed-point collision hands over to FP64 arithmetic (GPU):
lattices with stretches of zeros, tiny, ordinary and large densities side by side, so that
neighbouring sites take either path.  Every kernel family takes the same path at a site, so
they agree bitwise; against the oracle the method's FP64 bar holds (1e-12 of the largest
density)."""
import numpy as np
import pytest

from oracle import lbks as ora

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


@pytest.mark.parametrize("Q", [5, 7])
@pytest.mark.parametrize("level", [0.0, 1e-290, 1e-30, 1.0, 40.0, 300.0])
def test_sites_on_either_path(lb, Q, level):
    Ns = np.array([Q, 61, 300, 1025], dtype=np.int64)
    rng = np.random.default_rng(17)
    parts = []
    for n in Ns:
        r = level * rng.standard_normal(n)
        r[n // 3: n // 2] = 0.0
        r[: n // 8] *= 1e-20
        parts.append(r)
    r0 = np.concatenate(parts)
    dx, dt, tau, n = np.full(4, 0.3), np.full(4, 2e-4), np.array([1.0, 1.3, 2.0, 3.0]), 12
    ref, _ = ora.run_batch(Q, Ns, dx, dt, tau, r0, n)
    outs = []
    for kw in (dict(kernel=1), dict(kernel=2), dict(kernel=3), dict(kernel=3, sites_per_thread=4, threads_per_block=64),
               dict(kernel=3, sites_per_thread=8, threads_per_block=256)):
        h = lb.lb_ks_batch_init(Q, Ns, Ns * dx, dt, tau, r0, lb.lb_ks_default_opts(**kw))
        try:
            lb.lb_ks_step(h, n)
            out = np.empty(r0.size)
            lb.lb_ks_rho(h, out)
        finally:
            lb.lb_ks_free(h)
        outs.append(out)
    assert np.max(np.abs(outs[0] - ref)) <= 1e-12 * np.abs(ref).max()
    for out in outs[1:]:
        np.testing.assert_array_equal(outs[0], out)
