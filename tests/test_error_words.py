"""The statuses that the bits of the device error word become: the input's faults first, an exhausted wait always as an
internal error.  Compiled and run on the host."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_09713_b200", "csrc")

PROGRAM = """
#include "errors.h"
#include <cstdio>
using namespace spsyrk;
int main() {
    for (uint32_t e = 0; e < 32; ++e) std::printf("%u %d %d\\n", e, (int)status_of(e), (int)status_of(e, SPSYRK_ERR_INVALID_ARG));
}
"""


@pytest.fixture(scope="module")
def table(tmp_path_factory):
    d = tmp_path_factory.mktemp("errors")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, "-o", str(d / "t"), str(d / "t.cpp")])
    return [tuple(map(int, line.split())) for line in subprocess.check_output([str(d / "t")], text=True).splitlines()]


def test_statuses(table):
    ok, invalid_arg, bad_csr, internal = 0, 1, 2, 7
    rowptr, col, unsorted, gave_up, upper = 1, 2, 4, 8, 16
    for e, status, status_of_map in table:
        if e & (rowptr | unsorted | upper):
            assert status == status_of_map == bad_csr
        elif e & col:
            assert (status, status_of_map) == (bad_csr, invalid_arg)
        else:
            assert status == status_of_map == (internal if e & gave_up else ok)


def test_no_call_reads_the_word_another_way():
    """Where a call reads the error word back, its status comes from status_of."""
    for name in os.listdir(CSRC):
        text = open(os.path.join(CSRC, name)).read()
        if name != "errors.h":
            assert "return SPSYRK_ERR_BAD_CSR" not in text, name
