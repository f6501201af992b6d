"""Source check of the autotuner (no GPU needed): its trials must do the work of a run, which
cannot be seen from outside.  Each timed trial starts from the handle's own initial
populations, not from cleared arenas, whose sites an FP64 step leaves alone."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
API = os.path.join(ROOT, "paper_1711_03540_gb300", "csrc", "lbks_api.cu")


def _tuner():
    with open(API) as f:
        src = f.read()
    a = src.index("int autotune_resident(lb_ks* h) {")
    return src[a:src.index("\n}\n", a)]


def test_trials_start_from_the_initial_state():
    body = _tuner()
    trial = body[re.search(r"for \(int rep = 0;", body).start():]
    init, timed, steps = (trial.index(t) for t in ("init_populations(h)", "cudaEventRecord(e0", "issue_steps(h"))
    assert init < timed < steps
