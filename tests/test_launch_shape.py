"""CTAs of a single-source launch (host arithmetic, CPU only): the default, explicit
settings, and the two that the autotuner times, which have to be two launches."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS, RESIDENT = 152, 304
DO, TD, BU, RANDOM = 0, 1, 2, 3


@pytest.fixture(scope="module")
def shape(tmp_path_factory):
    d = tmp_path_factory.mktemp("launch_shape")
    prog = d / "shape.cpp"
    prog.write_text("""
#include <cstdio>
#include <cstdlib>
#include "launch_shape.h"
int main(int, char** a) {
  const long long n = atoll(a[1]);
  const int mode = atoi(a[2]), per_sm = atoi(a[3]), sms = atoi(a[4]), resident = atoi(a[5]);
  int t[2];
  bfsrt::tuner_ctas(n, mode, sms, resident, t);
  printf("%d %d %d\\n", bfsrt::search_grid(n, mode, per_sm, sms, resident), t[0], t[1]);
}
""")
    exe = str(d / "shape")
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1705_04590_gb300", "csrc"), str(prog),
                           "-o", exe])

    def call(n, mode=DO, per_sm=0, sms=SMS, resident=RESIDENT):
        return [int(x) for x in subprocess.check_output([exe] + [str(v) for v in (n, mode, per_sm, sms, resident)]).split()]
    return call


@pytest.mark.parametrize("mode", [DO, BU, RANDOM, TD])
@pytest.mark.parametrize("n", [1, 1 << 18, (1 << 18) + 1, 1 << 26])
def test_default_and_explicit_settings(shape, n, mode):
    assert shape(n, mode)[0] == (SMS if n <= 1 << 18 and mode != TD else RESIDENT)
    for per_sm, grid in ((1, SMS), (2, RESIDENT), (7, RESIDENT)):
        assert shape(n, mode, per_sm)[0] == grid
    # a server's executor with fewer CTAs than SMs keeps them
    assert shape(n, mode, 0, SMS, 38)[0] == 38 and shape(n, mode, 1, SMS, 38)[0] == 38


@pytest.mark.parametrize("resident", [304, 456])
@pytest.mark.parametrize("n", [1, 4096, 1 << 18, (1 << 18) + 1, 1 << 26])
def test_the_autotuner_times_two_launches(shape, n, resident):
    settings = shape(n, resident=resident)[1:]
    assert [shape(n, DO, s, resident=resident)[0] for s in settings] == [SMS, resident]
    assert settings[0] == 1 and (n <= 1 << 18 or settings[1] == 0)
