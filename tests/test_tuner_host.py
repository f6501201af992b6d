"""Source check of the autotuner (no GPU needed): its trials must do the work of a run, which
cannot be seen from outside.  Each timed trial starts from the handle's own initial
populations, not from cleared arenas, whose sites an FP64 step leaves alone, and all run the same
number of steps, which the plan made before tuning does not decide (it may be one of few
steps per launch, at which launch edges would weigh more than in a run)."""
import os
import re
import shutil
import subprocess

import pytest

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


def test_trials_do_not_take_their_length_from_the_plan_before_tuning():
    body = _tuner()
    before = body[:body.index("for (const Cand& c : cands)")]
    assert re.search(r"trial = tuner_steps\(kring, std::min\(kseg, kring\)\);", before)
    assert "h->kmax" not in body and "h->kseg" not in body


def test_trial_length(tmp_path):
    cuda = "/usr/local/cuda/include"
    if shutil.which("g++") is None or not os.path.exists(os.path.join(cuda, "vector_types.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    src = tmp_path / "t.cpp"
    src.write_text("""
#include "lbks_plan.h"
using namespace lbks::plan;
int main() {
  const int kseg = segment_steps(8, 256, 3);  // 34
  return kseg == 34 && segment_steps(4, 32, 3) == 2 && segment_steps(1, 32, 3) == 1 && tuner_steps(1000, kseg) == 500 &&
                 tuner_steps(70, kseg) == 70 && tuner_steps(20, 20) == 40 && tuner_steps(1000, 273) == 546
             ? 0 : 1;
}
""")
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-I" + os.path.dirname(API), "-I" + cuda, str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0
