"""The launch shape of a run that nobody chose one for, and which calls choose one, from
the library's own host code (a run of 100,000 hypotheses is no short one anywhere)."""
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
    perch_set_raster_bins(&c, 0);
    print("no_bins", c.cfg);
    perch_set_raster_bins(&c, 1024);
    print("bins", c.cfg);
    adopt_tuned(&c, perch::ScoreConfig{128, 4096, 0, 4096}, short_run(&c, 100000));
    print("tuned", c.cfg);
    perch_set_launch_config(&c, 128, 2048, 0);
    print("chosen", c.cfg);
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


def test_what_counts_as_chosen_for_short_runs(shapes):
    """A shape that the caller set does; tile bins are not a shape, and a shape tuned on
    a long batch was not timed on short runs."""
    assert shapes["no_bins"] == (256, 7064, 0, 0) and shapes["bins"] == (256, 7064, 1024, 0)
    assert shapes["tuned"] == (128, 4096, 4096, 0)
    assert shapes["chosen"] == (128, 2048, 4096, 1)
