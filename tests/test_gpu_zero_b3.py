"""The resident and collapse kernels' instances for lattices whose c = +-3 planes carry no
rho^2 term (D1Q7's first-moment weights are zero there) against the general ones: with the
default and the full-inverse weights they equal the one-step-per-launch kernels bitwise,
and a checkpoint whose constants have the term, loaded into a handle planned without it,
continues as the handle that saved it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NS = np.array([700, 3000, 5000, 9000], dtype=np.int64)


@pytest.fixture(scope="module")
def lb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_03540_gb300 import build

    build.build()
    import paper_1711_03540_gb300 as lb

    return lb


def _make(lb, collapse, **kw):
    rng = np.random.default_rng(23)
    r0 = np.concatenate([0.05 * rng.standard_normal(n) for n in NS])
    k = len(NS)
    dx, dt, tau = (0.2, 5e-5, np.ones(k)) if collapse else (0.1, 1e-4, np.linspace(1.5, 3.0, k))
    return lb.lb_ks_batch_init(7, NS, NS * dx, np.full(k, dt), tau, r0, lb.lb_ks_default_opts(recentre_every=40, **kw))


def _step_rho(lb, h, n):
    lb.lb_ks_step(h, n)
    out = np.empty(int(NS.sum()))
    lb.lb_ks_rho(h, out)
    return out


@pytest.mark.parametrize("collapse,prec,S,NT", [(False, 1, 20, 256), (False, 1, 16, 256), (False, 1, 8, 512),
                                                (False, 2, 18, 256), (True, 1, 32, 256), (True, 0, 16, 256)])
def test_both_instances_and_a_checkpoint_between_them(lb, collapse, prec, S, NT):
    tiling = dict(precision=prec, sites_per_thread=S, threads_per_block=NT, kernel=lb.KERNEL_COLLAPSE if collapse else 3)
    hs = {v: _make(lb, collapse, dm_variant=v, **tiling) for v in (0, lb.WEIGHTS_FULL_INVERSE)}
    other = _make(lb, collapse, dm_variant=0, **tiling)
    try:
        for v, h in hs.items():
            got = _step_rho(lb, h, 50)
            if prec != 2:  # (scaled FP16: one step per launch rounds every step)
                one = dict(kernel=lb.KERNEL_COLLAPSE, steps_per_launch=1) if collapse else dict(kernel=1)
                p = _make(lb, collapse, dm_variant=v, precision=prec, **one)
                np.testing.assert_array_equal(got, _step_rho(lb, p, 50))
                lb.lb_ks_free(p)
        lb.lb_ks_step(other, 10)
        lb.lb_ks_step(other, 10)  # (a captured sequence, of the other instance)
        src = hs[lb.WEIGHTS_FULL_INVERSE]
        buf = np.zeros(lb.lb_ks_state_bytes(src), dtype=np.uint8)
        lb.lb_ks_save(src, buf)
        lb.lb_ks_load(other, buf)
        np.testing.assert_array_equal(_step_rho(lb, src, 30), _step_rho(lb, other, 30))
    finally:
        for h in (*hs.values(), other):
            lb.lb_ks_free(h)
