"""vd_decode_shape: what vd_decode runs, and its errors (no device work)."""
import os
import subprocess
import sys

import pytest

import paper_2011_13579_gb300 as vd
from paper_2011_13579_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def codes():
    vd.build()
    return {7: vd.Code(7, synth.K7_GENS), 9: vd.Code(9, synth.K9_GENS)}


def named(lanes, form=0):
    t = vd.VdTune()
    t.lanes, t.form = lanes, form
    return t


@pytest.mark.parametrize("K,lanes", [(7, 1), (7, 2), (7, 4), (9, 4), (9, 8)])
@pytest.mark.parametrize("radix", [2, 4])
def test_a_named_shape_is_what_runs(codes, K, lanes, radix):
    s = vd.vd_decode_shape(codes[K].handle, vd.VD_LLR_S8, 100_000, 256, 42, radix, 0, named(lanes, 2))
    n_pairs = (vd.vd_num_frames(100_000, 256) + 1) // 2
    assert (s.form, s.radix, s.lanes, s.warp_pairs, s.cluster) == (vd.VD_FORM_ONE_WAVE, radix, lanes, 32 // lanes, 1)
    assert s.blocks == -(-n_pairs * lanes // 128)


def test_errors_are_those_of_vd_decode(codes):
    h = codes[7].handle
    for args in ((vd.VD_LLR_S8, 100, 0, 42), (vd.VD_LLR_S8, 100, 64, -1), (vd.VD_LLR_S8, 100, 48, 42), (9, 100, 64, 42),
                 (vd.VD_LLR_S8, 0, 64, 42), (vd.VD_LLR_S8, -1, 64, 42)):
        with pytest.raises(vd.VdError) as e:
            vd.vd_decode_shape(h, *args)
        assert e.value.status == vd.VD_EINVAL
    with pytest.raises(vd.VdError) as e:
        vd.vd_decode_shape(h, vd.VD_LLR_S8, 100, 64, 42, 2, 0, named(8))
    assert e.value.status == vd.VD_EUNSUPPORTED
    punctured = vd.Code(7, synth.K7_GENS, puncture=synth.PUNCT_R34.tolist())
    with pytest.raises(vd.VdError) as e:
        vd.vd_decode_shape(punctured.handle, vd.VD_LLR_F16, 100, 64, 42)
    assert e.value.status == vd.VD_EUNSUPPORTED


def test_without_a_device_the_one_wave_form_is_reported():
    child = ("import paper_2011_13579_gb300 as vd\nfrom paper_2011_13579_gb300 import synth\n"
             "c = vd.Code(7, synth.K7_GENS)\nfor n in (100, 1 << 24, 1 << 27):\n"
             "    s = vd.vd_decode_shape(c.handle, vd.VD_LLR_S8, n, 256, 42, 4)\n"
             "    assert s.form == vd.VD_FORM_ONE_WAVE and s.blocks > 0 and s.radix == 2, (n, s.form, s.blocks, s.radix)\n")
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", child], cwd=ROOT, env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr
