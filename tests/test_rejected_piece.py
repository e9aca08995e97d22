"""A piece record that the bounds-checked build rejects is left out as a whole: its rows are not
computed, and no stage runs for the elements of its unchecked range (CPU; needs nvcc).  The record's
element range is formed in one place, which knows whether the record passed: the host harness runs
that function, and the kernel forms the range nowhere else."""
import os
import re
import subprocess

import pytest

from test_host_tables import ROOT, _nvcc


def test_a_rejected_record_has_no_elements(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "host_rejected_piece")
    r = subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-o", exe,
                        os.path.join(ROOT, "tests", "host_rejected_piece.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split("\n")
    recs = [tuple(int(v) for v in line.split()) for line in out if line.strip()]
    assert len(recs) == 12
    for rows, off, nout, ok, e0, ne in recs:
        if ok and off >= 0:
            assert (e0, ne) == (off // nout, rows // nout)
        if not ok:
            assert ne == 0


def test_the_kernel_takes_every_stage_range_from_that_function():
    src = open(os.path.join(ROOT, "paper_2110_12165_gb300", "csrc", "hbi_hmvm.cu")).read()
    body = src[src.index("uy_gemv_kernel("):]
    body = body[:body.index("\n}\n")]
    assert not re.search(r"(tk\.rows|tk\.out_off)\s*/\s*ode\.nout", body)
    calls = re.findall(r"piece_elems\(([^)]*)\)", body)
    assert len(calls) == 2 and all(c.split(",")[-1].strip() == "task_ok" for c in calls)
