"""A density whose square overflows FP32 (GPU): reported by the guard at its next step, whether
the kernel leaves out the terms whose weight is zero (D1Q7's default weights) or has them (the
full-inverse weights)."""
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


@pytest.mark.parametrize("variant", [0, 2])
@pytest.mark.parametrize("opts", [dict(sites_per_thread=20, threads_per_block=256), dict(),
                                  dict(kernel=4, sites_per_thread=32, threads_per_block=256), dict(kernel=4)])
def test_overflow_is_reported_at_the_next_guard(lb, variant, opts):
    rng = np.random.default_rng(31)
    Ns = np.array([300, 4096, 6000], dtype=np.int64)
    r0 = np.concatenate([0.02 * rng.standard_normal(n) for n in Ns])
    r0[1000] = 3e19
    dx, dt, tau = (0.2, 5e-5, 1.0) if opts.get("kernel") == 4 else (0.1, 1e-4, 2.0)
    h = lb.lb_ks_batch_init(7, Ns, Ns * dx, np.full(3, dt), np.full(3, tau), r0, lb.lb_ks_default_opts(
        precision=lb.F32, recentre_every=1, dm_variant=variant, **opts))
    try:
        lb.lb_ks_step(h, 1)
        out = np.empty(r0.size)
        with pytest.raises(lb.LbKsError) as e:
            lb.lb_ks_rho(h, out)
        assert e.value.code == -4
    finally:
        lb.lb_ks_free(h)
