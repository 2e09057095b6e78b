"""The library stays mapped after a dlclose: its idle sampling threads (up to a second
after a call) must not return into unmapped code.  Stated in the file itself
(DF_1_NODELETE), not left to what the compiler happens to put in it."""
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def path():
    from paper_2604_27193_gb300 import _build
    return _build.build()


def test_marked_to_stay(path):
    out = subprocess.run(["readelf", "-dW", path], capture_output=True, text=True, check=True)
    assert re.search(r"FLAGS_1.*NODELETE", out.stdout), out.stdout


def test_closed_with_idle_helpers(path):
    code = f"""
import _ctypes, ctypes, os, time
import aeb_inputs as ai, paper_2604_27193_gb300 as aeb
L = aeb.lib()
aeb.aeb_sample_params(ai.single_model(), ai.single_scenario(1), 0, 20_000, n_threads=3)
_ctypes.dlclose(L._handle)
assert "libaeb.so" in open("/proc/self/maps").read()
time.sleep(1.5)  # the helpers end
again = ctypes.CDLL({path!r})
assert again.aeb_abi_version() == aeb.ABI_VERSION
print("ok")
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", (r.returncode, r.stdout, r.stderr)
