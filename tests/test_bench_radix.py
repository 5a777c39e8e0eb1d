"""bench.py reports the radix that it was asked for, so its vd_decode calls have
to run it: the shape of each call, as the library reports it."""
import pytest

import bench
import paper_2011_13579_gb300 as vd
from paper_2011_13579_gb300 import synth


@pytest.mark.parametrize("K,gens,f,v,lanes", [(7, synth.K7_GENS, 256, 42, (0, 1, 2, 4)), (9, synth.K9_GENS, 512, 64, (0, 4, 8))])
@pytest.mark.parametrize("radix", [2, 4])
def test_stream_calls_run_the_radix_asked_for(K, gens, f, v, lanes, radix):
    vd.build()
    code = vd.Code(K, gens)
    for l in lanes:
        s = vd.vd_decode_shape(code.handle, vd.VD_LLR_S8, 1 << 24, f, v, radix, 0, bench.named_tune(vd, radix, l, K))
        assert s.radix == radix and (not l or s.lanes == l)
