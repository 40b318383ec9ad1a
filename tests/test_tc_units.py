"""Host logic of the tensor-core far field: the size of the work units (tc_unit in csrc/tc_lists.h), compiled
with the host compiler.  No GPU."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1812_10722_gb300", "csrc")
MAIN = """
#include <cstdio>
#include <cstdlib>
#include "tc_lists.h"
int main(int, char **v) {
    const int64_t total = std::atoll(v[1]);
    const int sms = std::atoi(v[2]), lo = std::atoi(v[3]), hi = std::atoi(v[4]);
    const int seg = lspr::tc_unit(total, sms, lo, hi);
    std::vector<lspr::TcItem> units{{0, 0, (int)total, 0}};
    if (total > 0) lspr::tc_cut_m2p(seg, units);
    std::printf("%d %d\\n", seg, (int)units.size());
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("tc_units")
    src = d / "main.cpp"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(d / "main")], check=True)
    return str(d / "main")


# at the limits, either side of them, and where no SM count is known
@pytest.mark.parametrize("total,sms,lo,hi", [
    (0, 152, 32, 112), (1, 152, 32, 112), (12160, 152, 32, 112), (12540, 152, 32, 112), (23979, 152, 32, 112),
    (42560, 152, 32, 112), (42940, 152, 32, 112), (1 << 30, 152, 1024, 4096), (500, 0, 32, 64)])
def test_units_per_block(exe, total, sms, lo, hi):
    seg, units = map(int, subprocess.run([exe, str(total), str(sms), str(lo), str(hi)], check=True,
                                         capture_output=True, text=True).stdout.split())
    assert lo <= seg <= hi
    assert units == max(1, -(-total // seg))
    if seg > lo:   # longer units only where at least 2.5 of them per block remain
        assert total >= 2.5 * sms * seg
    if seg < hi:   # and as long as that allows
        assert total < 2.5 * max(1, sms) * (seg + 1)
