"""The step kernel's work plans (plan_steps in csrc/host_prep.cpp) replayed on
the CPU: every entry in exactly one slot, every row with exactly one epilogue,
every index inside its array, and in the bulk plan the row sums of the per-pass
kernel bit for bit (step_plan_check.cpp)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import lpgen

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    out = str(tmp_path_factory.mktemp("plan") / "step_plan_check")
    subprocess.run([gxx, "-O1", "-std=c++17", "-pthread", os.path.join(ROOT, "tests", "step_plan_check.cpp"),
                    os.path.join(ROOT, "paper_2511_13894_gb300", "csrc", "host_prep.cpp"), "-o", out], check=True)
    return out


def _rows(lens, n, seed):
    r = np.random.default_rng(seed)
    cols = [np.sort(r.choice(n, size=min(k, n), replace=False)) for k in lens]
    rp = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int64)
    return dict(m=len(lens), n=n, row_ptr=rp, col_idx=np.concatenate(cols).astype(np.int32) if rp[-1] else
                np.zeros(0, np.int32), val=r.standard_normal(int(rp[-1])))


LPS = {
    "empty": lambda: _rows([0, 0, 0], 5, 1),
    "one_entry": lambda: _rows([1], 1, 2),
    "31_32_33_rows": lambda: _rows([1 + i % 3 for i in range(33)], 31, 3),
    "slice_widths": lambda: _rows([1, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257] * 3, 400, 4),
    "long_rows": lambda: _rows([4095, 4096, 4097, 9000, 300, 0, 7], 9000, 5),
    "power_law": lambda: lpgen.power_law_lp(1500, 6000, 80, 1, kmax=500),
    "transport": lambda: lpgen.transportation_lp(40, 300, 2),
}


@pytest.mark.parametrize("name", list(LPS))
def test_plan_covers_every_entry_once(exe, name, tmp_path):
    lp = LPS[name]()
    path = str(tmp_path / "lp.bin")
    with open(path, "wb") as f:
        np.array([lp["m"], lp["n"], len(lp["col_idx"])], dtype=np.int64).tofile(f)
        np.asarray(lp["row_ptr"], dtype=np.int64).tofile(f)
        np.asarray(lp["col_idx"], dtype=np.int32).tofile(f)
        np.asarray(lp["val"], dtype=np.float64).tofile(f)
    p = subprocess.run([exe, path], stdout=subprocess.PIPE, text=True)
    assert p.returncode == 0 and p.stdout.strip() == "ok", p.stdout
