"""The lines between launch shapes of the transforms, on the host: they follow the SM count they are given."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_03024_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "launch_rules.h"
using namespace fhe;
int main(int argc, char** argv) {
    long v[5] = {0};
    for (int i = 1; i < argc; i++) v[i - 1] = std::atol(argv[i]);
    if (v[0] == 0) std::printf("%d\n", (int)rules::few_rows((int)v[1], (int)v[2], (size_t)v[3]));
    else if (v[0] == 2) std::printf("%d\n", (int)rules::single_pass((int)v[1], (int)v[2], v[3] & 1, v[3] & 2, (size_t)v[4]));
    else std::printf("%d\n", rules::rows_per_cta((int)v[1], (int)v[2], (size_t)v[3], (size_t)v[4]));
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", f"-I{CSRC}", str(d / "main.cpp"), "-o", str(d / "rules")], check=True)
    return lambda *a: int(subprocess.run([str(d / "rules"), *map(str, a)], capture_output=True, text=True, check=True).stdout)


@pytest.mark.parametrize("sms", [1, 76, 132, 152])
@pytest.mark.parametrize("log_n", [12, 13, 14, 15, 16])
def test_few_rows_is_sixteen_warps_per_sm(rule, sms, log_n):
    line = -(-sms * 512 * 16 // (1 << log_n))        # first count with 512 threads of 16 residues on every SM
    assert rule(0, sms, log_n, line - 1) == 1 and rule(0, sms, log_n, line) == 0


@pytest.mark.parametrize("sms,ctas", [(76, 3), (152, 3), (152, 8)])
def test_row_pass_keeps_eight_waves(rule, sms, ctas):
    wave8 = sms * ctas * 8
    for rows, tiles, want in ((wave8 // 16, 16, 1), (wave8 // 8, 16, 2), (wave8 // 4, 16, 4), (wave8 * 10, 16, 4), (1, 16, 1)):
        assert rule(1, sms, ctas, rows, tiles) == want


@pytest.mark.parametrize("sms", [76, 152])
def test_one_or_two_passes(rule, sms):
    for kind in range(4):                            # bit 0: fused passes, bit 1: inverse
        for rows in (1, sms, 100 * sms):
            assert [rule(2, sms, n, kind, rows) for n in (9, 11, 13, 16)] == [1, 1, 0, 0]
    few, many = sms // 3, 4 * sms
    for rows, plain_fwd, plain_inv in ((1, 0, 0), (few, 0, 0), (few + 1, 1, 1), (many, 1, 1), (many + 1, 0, 1)):
        assert [rule(2, sms, 12, kind, rows) for kind in range(4)] == [plain_fwd, 1, plain_inv, 1]
