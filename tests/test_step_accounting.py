"""The host loop of lbm_step (csrc/lbm_steps.h) with launches that fail, faked on
the host: the steps launched before the failure count, so that the context's step
counter and the parity of its layout stay those of the state on the device."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2112_08479_gb300", "csrc")

# argv: odd, nsteps, steps a chain takes (0: none), launches that succeed.  Prints
# the error, the steps counted, and the (parity, steps) of the launches made.
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "lbm_steps.h"
int main(int, char** a) {
    const int odd = atoi(a[1]), n = atoi(a[2]), sweep = atoi(a[3]);
    int left = atoi(a[4]), got = -1;
    char log[4096]; int at = 0; log[0] = 0;
    auto launch = [&](bool o, int s) {
        if (left-- <= 0) return 7;
        at += snprintf(log + at, sizeof log - at, " %d:%d", (int)o, s);
        return 0;
    };
    const int e = lbmgpu::enqueue_steps(odd != 0, n, got,
        [&](bool o, int m, int& done) {
            done = sweep ? m - m % sweep : 0;
            return done ? launch(o, done) : 0;
        },
        [&](bool o) { return launch(o, 1); });
    printf("%d %d%s\n", e, got, log);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("steps")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++20", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t")], check=True)

    def call(*args):
        out = subprocess.run([str(d / "t"), *map(str, args)], check=True, capture_output=True,
                             text=True).stdout.split()
        return int(out[0]), int(out[1]), [tuple(map(int, w.split(":"))) for w in out[2:]]
    return call


@pytest.mark.parametrize("odd", [0, 1])
@pytest.mark.parametrize("nsteps,sweep", [(0, 0), (1, 3), (5, 0), (3, 3), (8, 3), (10, 1), (4, 4)])
@pytest.mark.parametrize("succeed", range(6))
def test_steps_before_a_failed_launch_count(run, odd, nsteps, sweep, succeed):
    whole = nsteps - nsteps % sweep if sweep and nsteps >= 2 else 0
    sizes = ([whole] if whole else []) + [1] * (nsteps - whole)
    err, counted, made = run(odd, nsteps, sweep, succeed)
    assert [s for _, s in made] == sizes[:succeed]
    assert counted == sum(sizes[:succeed])
    assert err == (0 if succeed >= len(sizes) else 7)
    at = 0
    for o, s in made:                       # each launch starts on the parity of its first step
        assert o == (odd + at) % 2
        at += s
