"""A sampling call's helper threads run on the CPUs of the calling thread, also where an
earlier call from a thread held to other CPUs has started them."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import os, sys
sys.path[:0] = ["tests"]
import aeb_inputs as ai, paper_2604_27193_gb300 as aeb
aeb.build()
every = os.sched_getaffinity(0)
one = {min(every)}
m, sc = ai.single_model(), ai.single_scenario(1)

def masks(first, then):
    old = set(os.listdir("/proc/self/task"))
    os.sched_setaffinity(0, first)
    aeb.aeb_sample_params(m, sc, 0, 20_000, n_threads=3)
    os.sched_setaffinity(0, then)
    aeb.aeb_sample_params(m, sc, 0, 1_500_000, n_threads=3)  # ~90 ms: the helpers join in
    new = set(os.listdir("/proc/self/task")) - old
    os.sched_setaffinity(0, every)
    return [os.sched_getaffinity(int(t)) for t in new]

got = masks(*[eval(a) for a in sys.argv[1:]])
print(len(got), all(g == eval(sys.argv[2]) for g in got))
"""


@pytest.mark.skipif(len(os.sched_getaffinity(0)) < 2, reason="one CPU")
@pytest.mark.parametrize("first,then", [("one", "every"), ("every", "one")])
def test_helpers_run_where_the_call_may(first, then):
    r = subprocess.run([sys.executable, "-c", CODE, first, then], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.split() == ["2", "True"], (r.stdout, r.stderr)
