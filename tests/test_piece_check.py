"""The packer checks the UY pieces that the kernel is given, not only the units they are cut from (CPU;
needs nvcc): the cutter's pieces pass, and a piece with wrong rows, offsets, columns, gather list or
model, a missing or a surplus one is reported."""
import os
import subprocess

import pytest

from test_host_tables import ROOT, _nvcc


def test_corrupted_pieces_are_reported(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "host_piece_check")
    r = subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-o", exe,
                        os.path.join(ROOT, "tests", "host_piece_check.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split("\n")
    res = dict((line.split()[0], int(line.split()[1])) for line in out if line.strip())
    assert res.pop("pieces") > res.pop("units")
    assert res.pop("valid") == 0 and res.pop("valid_reversed") == 0
    assert len(res) == 14
    for name, bad in res.items():
        assert bad >= 1, name


def test_the_packer_checks_the_pieces_it_uploads():
    src = open(os.path.join(ROOT, "paper_2110_12165_gb300", "csrc", "hbi_hmvm.cu")).read()
    check, up = src.index("check_uy_pieces(units, t2, nout, &first)"), src.index("upload(&h->d_tasks2, t2)")
    assert check < up and "t2 =" not in src[check:up] and "sort(t2" not in src[check:up]
