"""Each form of vd_decode that a stream's length can lead to, by name of the
form (vd_decode_shape), against the CPU oracle: bits and canonical final
metrics, equal or wrong.

* few frames over many lanes (wide): frames of ordinary length beyond the
  segmented form's limit of frames, with a warp's pairs full, one more, two
  more and one less, and frames so long that a warp takes one pair;
* radix 4, which runs only where the caller names lanes or a form (K=7).
"""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2011_13579_gb300 as vd  # noqa: E402
from paper_2011_13579_gb300 import synth  # noqa: E402

GENS = {7: synth.K7_GENS, 9: synth.K9_GENS}
THREADS = max(1, len(os.sched_getaffinity(0)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vd.build()
    yield


def compare(K, n, f, v, term, unknown, seed, radix=2, tune=None, erase=0.0):
    rng = np.random.Generator(np.random.PCG64(seed))
    code, beta = vd.Code(K, GENS[K]), len(GENS[K])
    q = synth.make_stream(rng, K, GENS[K], n, 2.0, term).s8()
    q[rng.random(q.size) < erase] = 0
    out = torch.full(((n + 31) // 32,), -1, dtype=torch.int32, device="cuda")
    pm = torch.full((vd.vd_num_frames(n, f), 1 << (K - 1)), -1, dtype=torch.int32, device="cuda")
    flags = (vd.VD_TERMINATED if term else 0) | (vd.VD_START_UNKNOWN if unknown else 0)
    vd.vd_decode(code.handle, torch.from_numpy(q.view(np.uint8)).cuda(), vd.VD_LLR_S8, n, f, v, radix, flags, out, pm, tune)
    vd.vd_sync()
    ow, opm = oracle.decode(oracle.Code(K, GENS[K]), q.reshape(-1, beta).astype(np.int32), n, f, v, terminated=term,
                            start_unknown=unknown, threads=THREADS, want_pm=True)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), ow), (n, f, v)
    assert np.array_equal(pm.cpu().numpy().astype(np.int64), opm), (n, f, v)   # every frame has K-1 stages or more
    return vd.vd_decode_shape(code.handle, vd.VD_LLR_S8, n, f, v, radix, flags, tune)


# K, f, v, the segmented form's frames per SM at that length, pairs per warp
WIDE = [(7, 256, 42, 2, 4), (7, 512, 42, 3, 4), (7, 2560, 42, 3, 1), (7, 8192, 42, 3, 1), (9, 512, 64, 3, 1), (9, 96, 64, 1, 1)]


@pytest.mark.parametrize("term,unknown", [(True, False), (False, True)])
@pytest.mark.parametrize("K,f,v,frames_per_sm,warp_pairs", WIDE)
def test_wide_form_beyond_the_segmented_one(K, f, v, frames_per_sm, warp_pairs, term, unknown):
    limit = frames_per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    first = -(-(limit + 1) // 8) * 8           # frames of a whole number of warps
    for extra in (0, 1, 2, 7) if f <= 512 else (1,):
        n = (first + extra - 1) * f + 45       # the last frame is a short one
        s = compare(K, n, f, v, term, unknown, seed=n + K + term, erase=0.3 if extra == 2 else 0.0)
        assert (s.form, s.warp_pairs) == (vd.VD_FORM_FEW_FRAMES, warp_pairs), (n, s.form, s.warp_pairs)


def test_forms_around_the_segmented_limit():
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    code = vd.Code(7, GENS[7])
    forms = [vd.vd_decode_shape(code.handle, vd.VD_LLR_S8, frames * 256, 256, 42).form for frames in (1, 2 * sm, 2 * sm + 1)]
    assert forms == [vd.VD_FORM_SEGMENTS, vd.VD_FORM_SEGMENTS, vd.VD_FORM_FEW_FRAMES]


@pytest.mark.parametrize("K,f,v,per_sm,few", [(7, 32, 6, 37, True), (7, 32, 6, 42, False), (7, 64, 30, 37, True),
                                              (7, 64, 30, 46, False), (7, 32, 6, 80, False), (9, 32, 6, 23, True),
                                              (9, 32, 6, 60, False), (9, 64, 30, 40, False)])
def test_short_frames_leave_the_wide_form_by_blocks_per_sm(K, f, v, per_sm, few):
    """per_sm: blocks of the wide form (four pairs for K=7, one for K=9) per SM."""
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count * (8 if K == 7 else 2) * f
    s = compare(K, n, f, v, True, False, seed=n)
    assert (s.form == vd.VD_FORM_FEW_FRAMES) == few, s.form


@pytest.mark.parametrize("K,n", [(7, 3_000_000), (9, 600_000)])
def test_short_frames_can_be_captured_without_scratch(K, n):
    """A first call for short frames inside a stream capture, where nothing may be allocated."""
    f, v = 32, 6
    code = vd.Code(K, GENS[K])
    q = synth.make_stream(np.random.Generator(np.random.PCG64(n)), K, GENS[K], n, 2.0, False).s8()
    llr = torch.from_numpy(q.view(np.uint8)).cuda()
    want = vd.decode(code, llr, n, f, v)
    vd.vd_sync()
    assert vd.vd_decode_shape(code.handle, vd.VD_LLR_S8, n, f, v).form != vd.VD_FORM_FEW_FRAMES
    out = torch.full_like(want, -1)
    torch.cuda.synchronize()
    vd.vd_release_scratch()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        vd.decode(code, llr, n, f, v, out=out)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)


@pytest.mark.parametrize("radix", [2, 4])
@pytest.mark.parametrize("K,lanes,pairs_per_block", [(7, 1, 128), (9, 4, 32)])
def test_one_wave_keeps_three_blocks_per_sm_beyond_the_deep_ring(K, lanes, pairs_per_block, radix):
    """As many blocks as the deep traceback ring leaves resident (two per SM for
    these shapes, three for K=7 radix 4), and one more, which has to take the form of three."""
    t = vd.VdTune()
    t.lanes, t.form = lanes, vd.VD_FORM_ONE_WAVE
    code, f, v = vd.Code(K, GENS[K]), 32, 8
    sm = torch.cuda.get_device_properties(0).multi_processor_count

    def blocks_per_sm(blocks):
        n = blocks * pairs_per_block * 2 * f
        return n, vd.vd_decode_shape(code.handle, vd.VD_LLR_S8, n, f, v, radix, 0, t).blocks_per_sm

    deep = 3 if (K, radix) == (7, 4) else 2
    assert blocks_per_sm(deep * sm)[1] == deep
    n, after = blocks_per_sm(deep * sm + 1)
    assert after == 3
    s = compare(K, n - 45, f, v, True, False, seed=n, radix=radix, tune=t)
    assert s.blocks == deep * sm + 1


@pytest.mark.parametrize("form", [vd.VD_FORM_PERSISTENT, vd.VD_FORM_ONE_WAVE])
@pytest.mark.parametrize("K,lanes", [(7, 1), (7, 2), (7, 4), (9, 4), (9, 8)])
def test_radix_4_in_both_named_forms(K, lanes, form):
    t = vd.VdTune()
    t.lanes, t.form = lanes, form
    f, v = (256, 42) if K == 7 else (512, 64)
    s = compare(K, 150_777, f, v, True, False, seed=600 + K + lanes, radix=4, tune=t)
    assert (s.form, s.radix, s.lanes) == (form, 4, lanes)


def test_radix_4_persistent_with_several_tasks_a_warp():
    t = vd.VdTune()
    t.lanes, t.form = 1, vd.VD_FORM_PERSISTENT
    n, f = (1 << 22) + 77, 32                  # 2049 tasks of 32 pairs
    s = compare(7, n, f, 8, False, False, seed=66, radix=4, tune=t)
    assert s.radix == 4 and (vd.vd_num_frames(n, f) + 63) // 64 > s.blocks * 4
