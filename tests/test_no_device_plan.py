"""Where the device cannot be asked (how many SMs, how many resident blocks),
a long stream is planned in the one-wave form, which needs no such number,
never as a persistent launch of zero blocks.  Run in a process that sees no
device, so that every query fails.
"""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import paper_2011_13579_gb300 as vd
from paper_2011_13579_gb300 import synth
vd.build()
for K, gens, f, v, lanes in ((7, synth.K7_GENS, 256, 42, (1, 2)), (9, synth.K9_GENS, 512, 64, (4, 8))):
    code = vd.Code(K, gens)
    for n in (50_000, 1 << 24, 1 << 27):
        named = []
        for l in lanes:
            t = vd.VdTune()
            t.lanes, t.form = l, 2
            named.append(vd.vd_scratch_bytes(code.handle, n, f, v, 2, t))
        got = vd.vd_scratch_bytes(code.handle, n, f, v)
        assert got > 0 and got in named, (K, n, got, named)
print("ok")
"""


def test_long_streams_without_device_queries_take_the_one_wave_form():
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
