"""Source check of the order of copies and kernels on different streams (no GPU needed, and none
should be used: what it guards against is a race).  Tables are copied from pageable memory with
cudaMemcpy, on the default stream, which may return before the copy has reached the device; the
handle's and the capture stream need not wait for the default stream.  So a kernel on one of them
that reads such a table comes after a synchronisation of the default stream, or the copy goes on
the kernel's stream."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WAIT = "cudaStreamSynchronize(cudaStreamLegacy)"


def _function(name):
    with open(os.path.join(ROOT, "paper_1711_03540_gb300", "csrc", "lbks_api.cu")) as f:
        src = f.read()
    a = src.index(name)
    return src[a:src.index("\n}\n" if "\n}\n" in src[a:] else "\n}", a)]


def test_checkpoint_load():
    with open(os.path.join(ROOT, "paper_1711_03540_gb300", "csrc", "lbks_api.cu")) as f:
        src = f.read()
    a = src.index("int lb_ks_load(")
    body = src[a:src.index("} catch (...)", a)]
    copy, kernel = body.index("cudaMemcpy(h->d_runs"), body.index("launch_fix_coef(")
    assert WAIT in body[copy:kernel]
    last = max(body.rindex("cudaMemcpy("), body.rindex("cudaMemset("))
    assert WAIT in body[last:]


def test_creation():
    """Here the copies go on the stream of the kernel that reads the tables."""
    body = _function("int create_body(")
    up = body[body.index("auto up = "):]
    assert re.match(r"auto up = \[&\][^{]*\{\s*return cudaMemcpyAsync\([^;]*, is\);", up)
    kernel = body[body.index("launch_init_stats("):]
    assert re.match(r"launch_init_stats\([^;]*?,\s*is\)\)", kernel)
    assert body.index("CopyWait tables;") > body.index("std::vector<Tile> st;")  # (waits before they go)
