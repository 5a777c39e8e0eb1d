"""A plan's first launch may be a chained one, also when the caller names the
kernel shape (so that no tuning launch ran before): the task counters start at
zero whatever the memory held.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2011_13579_gb300 as vd  # noqa: E402
from paper_2011_13579_gb300 import synth  # noqa: E402


def test_first_launch_chained_with_named_shape():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vd.build()
    n = 200_000
    code = vd.Code(7, synth.K7_GENS)
    llr = torch.from_numpy(synth.segmented_stream(3.0, n_info=n).s8().view(np.uint8)).cuda()
    want = vd.decode(code, llr, n, 256, 42)
    tune = vd.VdTune()
    tune.radix, tune.lanes = 2, 1
    pk = {"n_info": np.array([n]), "llr_offset": np.array([0]), "out_word_offset": np.array([0]),
          "f": np.array([256]), "v": np.array([42])}
    for _ in range(4):
        # memory given back to the device with every bit set: the plan's small allocations may land in it
        dirty = [torch.full((1 << 18,), -1, dtype=torch.int32, device="cuda") for _ in range(64)]
        torch.cuda.synchronize()
        del dirty
        torch.cuda.empty_cache()
        plan = vd.BatchPlan([code], pk, tune=tune)
        out = torch.zeros_like(want)
        plan.launch(llr, out, chained=True)
        torch.cuda.synchronize()
        plan.status()
        assert torch.equal(out, want)
        plan.close()
