"""Barriers of the row loop for short streams (gen_rows_brief), checked on the
CPU as those of the other row loops are."""
import os
import re
import shutil
import subprocess

import pytest

from test_row_barriers import CSRC, MAIN, SHIM, _function

LOOP = "static uint32_t min(uint32_t a, uint32_t b) { return a < b ? a : b; }\n"


def _races(tmp_path, K, n, pos, drop=-1):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    fn = _function(open(os.path.join(CSRC, "mtgp_brief.cu")).read(), "gen_rows_brief")
    if drop >= 0:
        at = [m.start() for m in re.finditer(r"__syncwarp\(\);", fn)][drop]
        fn = fn[:at] + fn[at + len("__syncwarp();"):]
    cpp, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    cpp.write_text(SHIM + LOOP + fn + MAIN % {
        "n": n, "pos": pos, "rows": "gen_rows_brief<%d, 0>(S, ow, P, lane, g_tb, (1u + run) * P.n);" % K,
        "part": "gen_rows_brief<%d, 0>(S, ow, P, lane, g_tb, P.n / 2u);" % K})
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-w", "-o", str(exe), str(cpp)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout)
    return int(re.search(r"races (\d+)", r.stdout).group(1)), r.stdout


@pytest.mark.parametrize("K,n,pos", [(4, 351, 223), (4, 351, 1), (4, 352, 96), (4, 726, 598), (4, 1391, 1263),
                                     (4, 129, 1), (2, 101, 37), (2, 133, 69), (2, 128, 64), (2, 65, 1)])
def test_no_word_is_read_and_written_between_two_barriers(tmp_path, K, n, pos):
    n_races, log = _races(tmp_path, K, n, pos)
    assert n_races == 0, log


@pytest.mark.parametrize("K,n,pos,drop", [(4, 351, 95, 0), (4, 351, 95, 1), (2, 101, 37, 0), (2, 101, 37, 1)])
def test_the_check_sees_a_missing_barrier(tmp_path, K, n, pos, drop):
    assert _races(tmp_path, K, n, pos, drop)[0] > 0
