"""Source check (no GPU needed; a test that filled the device's memory would be no neighbour): a
batch whose arenas fit the device but whose one-site-per-thread tables do not keeps the kernel it
had before, as every upload of those tables hands an allocation failure on as "not this plan"."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_tables_that_do_not_fit_are_no_error():
    with open(os.path.join(ROOT, "paper_1711_03540_gb300", "csrc", "lbks_api.cu")) as f:
        src = f.read()
    a = src.index("int setup_blocked(lb_ks* h, int sms, double than) {")
    body = src[a:src.index("\n}\n", a)]
    uploads = re.findall(r"upload_lane\([^;]*;", body)
    assert len(uploads) == 2 and all("return no_room(rc)" in u for u in uploads)
    guard = body[body.index("const auto no_room"):]
    guard = guard[:guard.index("};")]
    assert "rc != LB_KS_ENOMEM" in guard and "release_lanes(h)" in guard and "return 1" in guard
