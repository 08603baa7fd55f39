"""The SM shares of the FP64 factorisation's two streams (host code), on GPUs and partitions of any size."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_06936_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include <initializer_list>
#include "shares.cuh"
int main() {
  const long long rows[] = {128, 640, 3200, 11776, 40000, 89600};
  for (int sms = 2; sms <= 160; ++sms)
    for (long long m : rows) std::printf("%d %lld %d\n", sms, m, exa::side_share(m, 512, sms));
  for (int sms = 2; sms <= 160; ++sms)
    for (int wanted : {0, 1, 2, 3, 20, 64, 104, 128}) std::printf("g %d %d %d\n", sms, wanted, exa::diag_grid(wanted, sms));
}
"""


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("shares")
    (d / "shares.cpp").write_text(SOURCE)
    subprocess.check_call([cxx, "-std=c++17", "-Wall", "-Werror", "-I" + CSRC, "-o", str(d / "shares"), str(d / "shares.cpp")])
    return subprocess.check_output([str(d / "shares")], text=True).splitlines()


def test_both_streams_get_an_sm(lines):
    shares = [tuple(map(int, l.split())) for l in lines if l[0] != "g"]
    assert len(shares) == 159 * 6
    for sms, _, share in shares:
        assert 2 <= share <= 104 and (share < sms or sms < 3), (sms, share)
    # the whole GPU: a block in the update's shadow gets few SMs, one that sets the pace all that help
    whole = {m: s for sms, m, s in shares if sms == 152}
    assert whole[128] == 104 and whole[89600] == 16


def test_a_diagonal_block_fits_the_gpu(lines):
    for line in lines:
        if line[0] == "g":
            sms, wanted, grid = map(int, line.split()[1:])
            assert 2 <= grid <= sms and grid <= 104
            if 2 <= wanted <= min(sms, 104):
                assert grid == wanted
