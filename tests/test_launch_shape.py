"""The launch shape of a run that nobody chose one for, from the library's own host
code (no GPU: a device without SMs, for which no run is a short one)."""
import subprocess

import pytest

from host_program import build_program

PROGRAM = r"""
#include "perch_host.cuh"
#include <cstdio>
using namespace perch_host;
static void print(const char* what, const perch::ScoreConfig& c)
{
    printf("%s %d %d %d %d\n", what, c.threads, c.zcap_words, c.bin_cap, (int)c.fixed);
}
int main()
{
    perch_ctx c;
    perch::ScoreConfig cfg = c.cfg;
    default_shape(&c, 100000, 1026, &cfg);
    print("long", cfg);
}
"""


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    exe = build_program(tmp_path_factory.mktemp("shape"), PROGRAM)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    return {line.split()[0]: tuple(int(x) for x in line.split()[1:]) for line in out.splitlines()}


def test_long_runs_take_the_base_shape(shapes):
    """Whatever the size of the image: a smaller z-buffer for small images walks the
    mesh twice when the object fills more of the image than it holds."""
    assert shapes["long"] == (256, 7064, 0, 0)
