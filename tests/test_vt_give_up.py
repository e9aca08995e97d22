"""Every wait of the V^T kernel that gives up reaches the host's error flag (CPU: the kernel's source).
A wait reports through the CTA's fail flag, which is copied to the error flag at the kernel's end, or,
where the CTA returns before that end (the product of a stopped attempt), writes the error
flag itself.  Making such a wait run out on the GPU would leave a bulk copy in flight."""
import os
import re

from test_host_tables import ROOT


def _kernel():
    src = open(os.path.join(ROOT, "paper_2110_12165_gb300", "csrc", "hbi_hmvm.cu")).read()
    body = src[src.index("vt_stream_kernel(\n"):]
    return body[:body.index("\n}\n")]


def test_the_stopped_path_reports_its_own_waits():
    body = _kernel()
    stopped = body[body.index("if (stopped && lane == 0) {"):body.index("if (stopped) return;")]
    waits = re.findall(r"thread_wait\([^;]*;", stopped)
    assert waits
    for w in waits:
        assert "raise_error(err)" in w, w


def test_nothing_returns_between_a_reported_wait_and_the_end():
    body = _kernel()
    # the returns of a stopped product: before any wait that reports through the fail flag
    returns = [m.start() for m in re.finditer(r"\breturn;", body)]
    assert len(returns) == 2
    waits = [m.start() for m in re.finditer(r"(warp_wait\([^;]*fail\)|\*fail = 1;)", body)]
    consumers = body.index("// ---- consumers")
    assert returns[0] < min(waits) and all(w > returns[1] for w in waits if w > consumers)
    assert re.search(r"__syncthreads\(\);\s*if \(tid == 0 && s_fail\) raise_error\(err\);\s*$", body)
