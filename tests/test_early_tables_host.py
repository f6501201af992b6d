"""Source check of what the one-site-per-thread kernels read before they wait for the previous grid
(no GPU needed).  They are launched with programmatic stream serialisation, like the kernels of
test_early_launch_host.py, but look up their piece in two tables first, `bundles` and `pieces`, to
have the addresses of the populations at hand when the wait ends.  That is safe because no grid
writes these tables: they come to the device once, when the plan is made, by a copy that is
complete before the first launch.  So the body up to the wait names no other global memory, the
tables are const to every kernel, and the host writes them in one place."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1711_03540_gb300", "csrc")
KERNELS = ("blocked_step_kernel", "blocked_collapse_kernel")


def _read(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def _kernel(src, name):
    m = re.search(r"__global__[^;{]*?\b" + name + r"\s*\(([^{]*)\)\s*\{", src, re.S)
    return m.group(1), src[m.end():]


def test_only_the_tables_are_read_before_the_wait():
    src = _read("lbks_kernels_blocked.cu")
    for name in KERNELS:
        params, body = _kernel(src, name)
        assert re.search(r"const\s+Piece\s*\*\s*__restrict__\s+pieces", params)
        assert re.search(r"const\s+int2\s*\*\s*__restrict__\s+bundles", params)
        head = body[:body.index("wait_prior_grid();")]
        assert "pieces[" in head  # (else this test has nothing to guard)
        for other in ("runs[", "src.", "dst.", "runs->", "*runs", "src,"):
            assert other not in head, (name, other)


def test_a_read_of_the_run_table_before_the_wait_is_caught():
    src = _read("lbks_kernels_blocked.cu").replace("  wait_prior_grid();\n  const RunDesc& d = runs[pc.run];",
                                                   "  const RunDesc& d = runs[pc.run];\n  wait_prior_grid();")
    body = _kernel(src, KERNELS[0])[1]
    assert "runs[" in body[:body.index("wait_prior_grid();")]


def test_the_tables_are_written_once_when_the_plan_is_made():
    api = _read("lbks_api.cu")
    writes = re.findall(r"cudaMem(?:cpy|set)\w*\(\s*[\w.>-]*d_(?:pieces|bundles)\b", api)
    assert len(writes) == 2
    a = api.index("int upload_lane(")
    body = api[a:api.index("\n}\n", a)]
    assert len(re.findall(r"cudaMemcpy\(L->d_(?:pieces|bundles)\b", body)) == 2  # (blocking copies)
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            assert not re.search(r"(?<!const )\bPiece\s*\*\s*(?:__restrict__\s*)?pieces\b", _read(name)), name
