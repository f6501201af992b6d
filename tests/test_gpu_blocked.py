"""The one-site-per-thread kernel (csrc/lbks_kernels_blocked.cu), the default for FP64 storage
and for FP32 batches too small for the register-resident kernel: bitwise equal to the plain
kernel (one step per launch), and with reservoir ends within 1e-12 of the oracle, on
lattices from the minimum length over the edges of its blocks to many stretches, alone,
packed many to a block and mixed, over step counts that end inside a launch."""
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
                            lb.lb_ks_default_opts(**kw))
    try:
        for n in calls:
            lb.lb_ks_step(h, n)
        out = np.empty(r0.size)
        lb.lb_ks_rho(h, out)
        desc = lb.lb_ks_describe(h)
    finally:
        lb.lb_ks_free(h)
    return out, desc


def _batch(which, Q):
    rng = np.random.default_rng(61)
    if which == "packed":  # 7 .. 40 sites, up to 16 a block
        Ns = rng.integers(Q, 41, 2500)
    elif which == "mixed":
        Ns = np.concatenate([rng.integers(Q, 700, 300), [1024, 4097, 5000]])
    else:
        Ns = np.array([which])
    Ns = Ns.astype(np.int64)
    return Ns, np.concatenate([0.05 * rng.standard_normal(n) for n in Ns])


SIZES = ["Q", 32, 63, 64, 65, 383, 384, 385, 512, 513, 4096, 100001, "packed", "mixed"]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("Q", [5, 7])
@pytest.mark.parametrize("which", SIZES)
def test_blocked_equals_plain_bitwise(lb, prec, Q, which):
    Ns, r0 = _batch(Q if which == "Q" else which, Q)
    kw = dict(precision=prec, recentre_every=70 if prec else 0)
    a, da = _run(lb, Q, Ns, r0, (1, 53, 100), **kw)
    b, _ = _run(lb, Q, Ns, r0, (154,), kernel=1, **kw)
    assert da["kernel"] == lb.KERNEL_RESIDENT
    if prec == 0 or len(Ns) == 1:  # (FP32 batches: whichever tiling is estimated faster)
        assert da["sites_per_thread"] == 1
    np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("Q", [5, 7])
@pytest.mark.parametrize("runs", [1, 40])
def test_reservoir_ends_match_oracle(lb, Q, runs):
    """Lattices of one block and of several stretches (the fixed ends inside the outer ones)."""
    alphas = [0.4, 0.12, 0.05] if runs == 1 else [0.4, 0.2, 0.15] * 13 + [0.1]
    Ns = np.array([front.nodes(a).size for a in alphas], dtype=np.int64)
    r0 = np.concatenate([front.rho_exact(front.nodes(a), 0.0) for a in alphas])
    k, n, beta, tau = len(alphas), 301, 1e-6, 1.3
    ref = np.concatenate([ora.run(Q, front.rho_exact(front.nodes(a), 0.0), a, beta, tau, n, boundary="reservoir",
                                  rho_left=front.RHO_LEFT, rho_right=front.RHO_RIGHT) for a in alphas])
    outs = []
    for calls in ((n,), (100, 2, n - 102)):
        h = lb.lb_ks_batch_init_reservoir(Q, Ns, np.full(k, 60.0), np.full(k, beta), np.full(k, tau), r0,
                                          np.full(k, front.RHO_LEFT), np.full(k, front.RHO_RIGHT))
        try:
            for m in calls:
                lb.lb_ks_step(h, m)
            out = np.empty(r0.size)
            lb.lb_ks_rho(h, out)
        finally:
            lb.lb_ks_free(h)
        outs.append(out)
    assert np.max(np.abs(outs[0] - ref)) <= 1e-12 * np.abs(ref).max()
    np.testing.assert_array_equal(outs[0], outs[1])


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("nruns,nmin,nmax", [(1, 1000, 1000), (4, 500, 2700), (24, 256, 8192), (60, 100, 600),
                                             (238, 164, 549), (354, 548, 1770), (1024, 64, 256), (2500, 100, 700),
                                             (1024, 220, 4000), (3, 9000, 11000), (1187, 18, 6303), (1187, 16, 3000)])
def test_tiling_chosen_by_size_equals_the_fixed_one(lb, prec, nruns, nmin, nmax):
    """FP32 and scaled FP16 (rounded at launch edges, which the choice must not move): the
    default plan's results are those of 20 sites x 256 threads, bitwise."""
    rng = np.random.default_rng(71)
    Ns = np.round(np.exp(rng.uniform(np.log(nmin), np.log(nmax), nruns))).astype(np.int64)
    r0 = np.concatenate([0.02 * rng.standard_normal(n) for n in Ns])
    kw = dict(precision=prec, recentre_every=60)
    a, _ = _run(lb, 7, Ns, r0, (130,), **kw)
    b, d = _run(lb, 7, Ns, r0, (130,), sites_per_thread=20, threads_per_block=256, **kw)
    assert d["sites_per_thread"] == 20
    np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("Q", [5, 7])
@pytest.mark.parametrize("which", SIZES)
def test_blocked_collapse_equals_streaming_bitwise(lb, prec, Q, which):
    """The tau = 1 collapse, one value per thread, against one step per launch."""
    Ns, r0 = _batch(Q if which == "Q" else which, Q)
    k, outs = len(Ns), []
    for spl, calls in ((0, (1, 53, 100)), (1, (154,))):
        h = lb.lb_ks_batch_init(Q, Ns, Ns * 0.2, np.full(k, 5e-5), np.ones(k), r0, lb.lb_ks_default_opts(
            kernel=lb.KERNEL_COLLAPSE, precision=prec, recentre_every=70 if prec else 0, steps_per_launch=spl))
        try:
            for n in calls:
                lb.lb_ks_step(h, n)
            out = np.empty(r0.size)
            lb.lb_ks_rho(h, out)
            spt = lb.lb_ks_describe(h)["sites_per_thread"]
        finally:
            lb.lb_ks_free(h)
        assert spt == (0 if spl else 1)
        outs.append(out)
    np.testing.assert_array_equal(outs[0], outs[1])


@pytest.mark.parametrize("Q", [5, 7])
@pytest.mark.parametrize("prec", [0, 1])
def test_blocked_collapse_reservoir_ends(lb, Q, prec):
    """Reservoir ends on the collapse: many steps per launch against one."""
    alphas = [0.4, 0.2, 0.1]
    Ns = np.array([front.nodes(a).size for a in alphas], dtype=np.int64)
    r0 = np.concatenate([front.rho_exact(front.nodes(a), 0.0) for a in alphas])
    outs = []
    for spl in (0, 1):
        h = lb.lb_ks_batch_init_reservoir(Q, Ns, np.full(3, 60.0), np.full(3, 2e-6), np.ones(3), r0,
                                          np.full(3, front.RHO_LEFT), np.full(3, front.RHO_RIGHT), lb.lb_ks_default_opts(
                                              kernel=lb.KERNEL_COLLAPSE, precision=prec, steps_per_launch=spl))
        try:
            for n in (2, 131):
                lb.lb_ks_step(h, n)
            out = np.empty(r0.size)
            lb.lb_ks_rho(h, out)
        finally:
            lb.lb_ks_free(h)
        outs.append(out)
    np.testing.assert_array_equal(outs[0], outs[1])
