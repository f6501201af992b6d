"""The tau = 1 collapse's register-resident tiling chosen by size (choose_collapse in
csrc/lbks_plan.h): bitwise the results of 32 sites x 256 threads, for batches that take each of
the tilings, with lattices shorter than S (S - 1) among them (held as copies)."""
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


def _run(lb, Q, Ns, r0, **kw):
    k = len(Ns)
    h = lb.lb_ks_batch_init(Q, Ns, Ns * 0.2, np.full(k, 5e-5), np.full(k, 1.0), r0,
                            lb.lb_ks_default_opts(precision=lb.F32, kernel=lb.KERNEL_COLLAPSE, recentre_every=60, **kw))
    try:
        for n in (1, 53, 76):
            lb.lb_ks_step(h, n)
        out = np.empty(r0.size)
        lb.lb_ks_rho(h, out)
    finally:
        lb.lb_ks_free(h)
    return out


@pytest.mark.parametrize("Q", [5, 7])
@pytest.mark.parametrize("nruns,nmin,nmax", [(984, 194, 447), (101, 1504, 3031), (156, 650, 3790), (200, 16, 4000),
                                             (2223, 119, 3922), (700, 256, 8192), (758, 824, 1481), (764, 24, 65)])
def test_tiling_chosen_by_size_equals_the_fixed_one(lb, Q, nruns, nmin, nmax):
    rng = np.random.default_rng(73)
    Ns = np.round(np.exp(rng.uniform(np.log(nmin), np.log(nmax), nruns))).astype(np.int64)
    r0 = np.concatenate([0.02 * rng.standard_normal(n) for n in Ns])
    np.testing.assert_array_equal(_run(lb, Q, Ns, r0), _run(lb, Q, Ns, r0, sites_per_thread=32, threads_per_block=256))
