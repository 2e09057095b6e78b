"""The launch configuration that a fresh process reports is the one its launches use:
tickets of 32 samples in both precisions.  So a caller who reads it, changes the
resident blocks and writes it back does not change the tile."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_default_tile_is_the_one_in_use():
    code = ("import paper_2604_27193_gb300 as m\n"
            "m.build()\n"
            "for p in (m.FP64_PLAIN, m.FP32_COMP):\n"
            "    c = m.aeb_get_launch_config(p)\n"
            "    m.aeb_set_launch_config(p, c.tile, 4)\n"
            "    d = m.aeb_get_launch_config(p)\n"
            "    print(c.tile, c.blocks_per_sm, d.tile, d.blocks_per_sm)\n")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True,
                       check=True, timeout=300)
    assert r.stdout.split("\n")[:2] == ["32 0 32 4"] * 2, r.stdout
