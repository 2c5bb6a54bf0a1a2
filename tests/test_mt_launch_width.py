"""CTAs of a comparison-generator launch (mt_ctas), on the CPU.

The rule's own source text is compiled as host code and asked for many
launches on 152 SMs of four-warp CTAs.
"""
import os
import re
import shutil
import subprocess

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1501_07701_gb300", "csrc",
                   "mt_gen.cu")
SMS, WARPS = 152, 4


@pytest.fixture(scope="module")
def ctas(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    text = open(SRC).read()
    fn = re.search(r"static long long mt_ctas\(.*?\n}\n", text, re.S)
    assert fn, "mt_ctas"
    assert "kWarpsPerCta = %d;" % WARPS in text
    d = tmp_path_factory.mktemp("mt")
    (d / "m.cpp").write_text("#include <algorithm>\n#include <cstdint>\n#include <cstdio>\n"
                             "constexpr int kWarpsPerCta = %d;\n%s\nint main()\n{\n    unsigned n;\n"
                             "    unsigned long long t, m;\n    while (scanf(\"%%u %%llu %%llu\", &n, &t, &m) == 3)\n"
                             "        printf(\"%%lld\\n\", mt_ctas(n, t, m, %d));\n}\n" % (WARPS, fn.group(0), SMS))
    subprocess.run([cxx, "-std=c++17", "-O1", "-o", str(d / "m"), str(d / "m.cpp")], check=True)

    def run(launches):
        r = subprocess.run([str(d / "m")], input="\n".join("%d %d %d" % x for x in launches), capture_output=True,
                           text=True, check=True)
        return [int(v) for v in r.stdout.split()]
    return run


def test_equal_streams_have_a_warp_each(ctas):
    ns = list(range(1, 5000))
    for n, c in zip(ns, ctas([(n, n << 16, 1 << 16) for n in ns])):
        assert c == (n + WARPS - 1) // WARPS, n   # residency caps it at launch


def test_streams_of_about_one_length_have_a_warp_each(ctas):
    """n - 1 streams a little shorter than the longest: pace is below n, and
    no launch gets fewer warps than that."""
    ns = list(range(600, 3000))
    for n, c in zip(ns, ctas([(n, 60000 * (n - 1) + 65536, 65536) for n in ns])):
        pace = (60000 * (n - 1) + 65536 + 65535) // 65536
        assert c * WARPS >= max(min(n, SMS * WARPS), pace), n


def test_uneven_launches_fill_whole_numbers_of_ctas_per_sm(ctas):
    # 10 000 streams; a pace of 1224 warps is 306 CTAs, two more than two per SM
    assert ctas([(10000, 1224 << 22, 1 << 22)]) == [2 * SMS]
    assert ctas([(10000, 1216 << 22, 1 << 22), (10000, 100 << 22, 1 << 22), (300, 100 << 22, 1 << 22)]) == [
        2 * SMS, SMS, 75]
    assert ctas([(10000, (4 * (SMS + SMS // 8)) << 22, 1 << 22), (10000, (4 * (SMS + SMS // 8 + 1)) << 22, 1 << 22)]) == [
        SMS, SMS + SMS // 8 + 1]
