"""The one-site-per-thread kernel over the blocks of a cluster (FP64 batches with lattices
longer than a block, csrc/lbks_kernels_blocked.cu): bitwise equal to the plain kernel, and
with reservoir ends within 1e-12 of the oracle, on batches whose lattices end at, before and
after block edges, over calls that end inside a launch."""
import numpy as np
import pytest

from oracle import front, lbks as ora

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


def _run(lb, Q, Ns, r0, calls, **kw):
    k = len(Ns)
    h = lb.lb_ks_batch_init(Q, Ns, Ns * 0.1, np.full(k, 1e-4), np.linspace(1.5, 3.0, k), r0,
                            lb.lb_ks_default_opts(precision=lb.F64, **kw))
    try:
        for n in calls:
            lb.lb_ks_step(h, n)
        out = np.empty(r0.size)
        lb.lb_ks_rho(h, out)
        desc = lb.lb_ks_describe(h)
    finally:
        lb.lb_ks_free(h)
    return out, desc


@pytest.mark.parametrize("Q", [5, 7])
@pytest.mark.parametrize("nruns,nmin,nmax", [(100, 200, 960), (200, 5, 600), (400, 400, 600), (100, 300, 1480),
                                             (1000, 500, 600)])
@pytest.mark.parametrize("recentre", [0, 60])
def test_cluster_equals_plain_bitwise(lb, Q, nruns, nmin, nmax, recentre):
    rng = np.random.default_rng(17)
    Ns = rng.integers(max(nmin, Q), nmax + 1, nruns).astype(np.int64)
    Ns[:6] = np.minimum(nmax, [255, 256, 257, 511, 512, 513])
    r0 = np.concatenate([0.05 * rng.standard_normal(n) for n in Ns])
    a, d = _run(lb, Q, Ns, r0, (1, 53, 100), recentre_every=recentre)
    b, _ = _run(lb, Q, Ns, r0, (154,), recentre_every=recentre, kernel=lb.KERNEL_PLAIN)
    assert d["sites_per_thread"] == 1
    if nruns in (100, 200) and nmax < 1000:  # (elsewhere whichever form is estimated faster)
        assert d["cluster_size"] in (4, 8) or Q == 5
    np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("Q", [5, 7])
def test_reservoir_ends_match_oracle(lb, Q):
    alphas = [0.2] * 61 + [0.1] * 61
    taus = np.concatenate([np.linspace(1.5, 2.4, 61)] * 2)
    Ns = np.array([front.nodes(a).size for a in alphas], dtype=np.int64)
    r0 = np.concatenate([front.rho_exact(front.nodes(a), 0.0) for a in alphas])
    k, n, beta = len(alphas), 151, 1e-4
    h = lb.lb_ks_batch_init_reservoir(Q, Ns, np.full(k, 60.0), np.full(k, beta), taus, r0,
                                      np.full(k, front.RHO_LEFT), np.full(k, front.RHO_RIGHT))
    try:
        for m in (1, 2, 100, n - 103):
            lb.lb_ks_step(h, m)
        out = np.empty(r0.size)
        lb.lb_ks_rho(h, out)
    finally:
        lb.lb_ks_free(h)
    at = np.concatenate([[0], np.cumsum(Ns)])
    for r in (0, 1, 30, 60, 61, 90, 121):
        ref = ora.run(Q, r0[at[r]:at[r + 1]], alphas[r], beta, taus[r], n, boundary="reservoir",
                      rho_left=front.RHO_LEFT, rho_right=front.RHO_RIGHT)
        assert np.max(np.abs(out[at[r]:at[r + 1]] - ref)) <= 1e-12 * np.abs(ref).max()
