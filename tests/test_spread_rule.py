"""Shared memory that spreads a small grid over the SMs (no GPU needed): the rule compiled as plain C++
against the documented allocation (an SM's 228 KB, 1 KB per block for the system, a block's total rounded
up to 128 bytes, 227 KB per block at most)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_07294_gb300", "csrc")

MAIN = """
#include <cstdio>
#include <initializer_list>
#include "launch_rules.h"
int main() {
    for (int st : {%s})
        for (int sms : {1, 148, 152})
            for (int res = 1; res <= 32; ++res)
                for (int blocks = 1; blocks <= res * sms; blocks += blocks < 40 ? 1 : 37)
                    for (int beside = 0; beside < 2; ++beside)
                        std::printf("%%d %%d %%d %%d %%d %%zu\\n", beside, st, sms, res, blocks,
                                    wd::spread_bytes(blocks, sms, res, st, beside));
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no C++ compiler")
def test_as_many_blocks_fit_as_the_grid_needs(tmp_path):
    (tmp_path / "m.cpp").write_text(MAIN % "0, 2048, 3000, 6144")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(tmp_path / "m.cpp"), "-o", str(tmp_path / "m")], check=True)
    out = subprocess.run([str(tmp_path / "m")], check=True, capture_output=True, text=True).stdout
    rows = [tuple(map(int, l.split())) for l in out.splitlines()]
    assert len(rows) > 1000
    for beside, static, sms, resident, blocks, dyn in rows:
        need = -(-blocks // sms)
        if need >= resident or (beside and 2 * need < resident):   # fills the device, or leaves it to others
            assert dyn == 0
            continue
        total = -(-(static + dyn + 1024) // 128) * 128
        assert static + dyn <= 227 * 1024
        # (seven blocks: six fit, measured the same alone and better beside other streams)
        assert (228 * 1024) // total == (6 if need == 7 else need), (static, sms, resident, blocks, dyn)
        assert (228 * 1024) // (total - 128) > (6 if need == 7 else need)   # no more than that takes
