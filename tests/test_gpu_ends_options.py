"""Lattices with fixed-value ends (GPU): the options that ask for one step per launch are
honoured, and the many-steps form (one block, stretches, clusters) gives the same bits."""
import numpy as np
import pytest

from oracle import front

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


def _run(lb, Q, alphas, taus, beta, n, **opts):
    Ns = np.array([front.nodes(a).size for a in alphas], dtype=np.int64)
    r0 = np.concatenate([front.rho_exact(front.nodes(a), 0.0) for a in alphas])
    k = len(alphas)
    h = lb.lb_ks_batch_init_reservoir(Q, Ns, np.full(k, 60.0), np.full(k, beta), taus, r0, np.full(k, front.RHO_LEFT),
                                      np.full(k, front.RHO_RIGHT), lb.lb_ks_default_opts(**opts))
    try:
        d, lanes = lb.lb_ks_describe(h), lb.lb_ks_describe_lanes(h)
        before = lb.lb_ks_launches(h)
        for m in (1, n - 4, 3):
            lb.lb_ks_step(h, m)
        launches = lb.lb_ks_launches(h) - before
        out = np.empty(r0.size)
        lb.lb_ks_rho(h, out)
    finally:
        lb.lb_ks_free(h)
    return out, d, lanes, launches


BATCHES = {"one block": [0.4, 0.3], "stretches": [0.05], "clusters": [0.2] * 61 + [0.1] * 61}


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("Q", [5, 7])
@pytest.mark.parametrize("which", sorted(BATCHES))
def test_options_of_lattices_with_ends(lb, prec, Q, which):
    alphas, n, beta = BATCHES[which], 60, 2e-5
    taus = np.linspace(1.5, 2.4, len(alphas))
    many, d, lanes, launches = _run(lb, Q, alphas, taus, beta, n, precision=prec)
    assert d["sites_per_thread"] == 1 and d["steps_per_launch"] > 1 and len(lanes) == 1
    assert launches < n
    if prec == 0:
        assert (d["cluster_size"] > 1) == (which == "clusters")
    for opts in (dict(kernel=lb.KERNEL_PLAIN), dict(steps_per_launch=1)):
        one, d, lanes, launches = _run(lb, Q, alphas, taus, beta, n, precision=prec, **opts)
        assert d["sites_per_thread"] == 0 and len(lanes) == 0
        assert launches == n
        np.testing.assert_array_equal(one, many)


@pytest.mark.parametrize("Q", [5, 7])
def test_collapse_with_ends_reports_its_plan(lb, Q):
    """The tau = 1 collapse with ends likewise."""
    alphas, taus = [0.4, 0.1], np.ones(2)
    many, d, lanes, launches = _run(lb, Q, alphas, taus, 2e-6, 60, kernel=lb.KERNEL_COLLAPSE)
    assert d["sites_per_thread"] == 1 and len(lanes) == 1 and launches < 60
    one, d, lanes, launches = _run(lb, Q, alphas, taus, 2e-6, 60, kernel=lb.KERNEL_COLLAPSE, steps_per_launch=1)
    assert d["sites_per_thread"] == 0 and len(lanes) == 0 and launches == 60
    np.testing.assert_array_equal(one, many)
