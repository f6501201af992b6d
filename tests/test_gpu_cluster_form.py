"""The form of the FP64 kernel that spreads lattices over thread block clusters is the one that
runs, for both schemes, on batches of lattices somewhat longer than a block (GPU), and gives the
plain kernel's bits there."""
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


@pytest.mark.parametrize("Q", [5, 7])
@pytest.mark.parametrize("nruns,nmin,nmax", [(100, 200, 960), (200, 7, 600)])
def test_clusters_run(lb, Q, nruns, nmin, nmax):
    rng = np.random.default_rng(23)
    Ns = rng.integers(nmin, nmax + 1, nruns).astype(np.int64)
    r0 = np.concatenate([0.05 * rng.standard_normal(n) for n in Ns])
    outs = []
    for kernel in (lb.KERNEL_AUTO, lb.KERNEL_PLAIN):
        h = lb.lb_ks_batch_init(Q, Ns, Ns * 0.1, np.full(nruns, 1e-4), np.linspace(1.5, 3.0, nruns), r0,
                                lb.lb_ks_default_opts(kernel=kernel))
        try:
            if kernel == lb.KERNEL_AUTO:
                assert lb.lb_ks_describe(h)["cluster_size"] > 1
                assert lb.lb_ks_describe_lanes(h)[0]["blocks_per_group"] > 1
            lb.lb_ks_step(h, 97)
            out = np.empty(r0.size)
            lb.lb_ks_rho(h, out)
        finally:
            lb.lb_ks_free(h)
        outs.append(out)
    np.testing.assert_array_equal(outs[0], outs[1])
