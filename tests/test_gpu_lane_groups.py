"""Several lanes per frame pair, with the lane groups of one warp out of step:
frames of a batch that begin in different chunks, from the reset state or not,
and streams whose last warp has groups without a pair.  Against the CPU
oracle, bit for bit (integer arithmetic: no tolerance).
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
SHAPES = [(7, 2), (7, 4), (9, 4), (9, 8)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vd.build()
    yield


@pytest.mark.parametrize("radix", [2, 4])
@pytest.mark.parametrize("K,lanes", SHAPES)
def test_groups_that_begin_in_different_chunks(K, lanes, radix):
    rng = np.random.Generator(np.random.PCG64(4100 + 10 * K + lanes + radix))
    n = 83                                   # no whole number of pairs or of a warp's groups
    n_info = rng.integers(1, 500, n).astype(np.int64)
    term = rng.random(n) < 0.5
    unknown = rng.random(n) < 0.4
    f = np.where(rng.random(n) < 0.5, np.maximum(n_info, 1), 64).astype(np.int32)
    v = np.where(f == 64, 40, K - 1).astype(np.int32)
    beta = len(GENS[K])
    T = n_info + np.where(term, K - 1, 0)
    streams = [synth.make_stream(rng, K, GENS[K], int(n_info[i]), 2.0, bool(term[i])).s8() for i in range(n)]
    off = np.concatenate([[0], np.cumsum(beta * T)[:-1]]).astype(np.int64)
    words = (n_info + 31) // 32
    word_off = np.concatenate([[0], np.cumsum(words)[:-1]]).astype(np.int64)
    arena = np.concatenate(streams)
    pk = {"n_info": n_info, "llr_offset": off, "out_word_offset": word_off, "f": f, "v": v,
          "flags": (np.where(term, vd.VD_TERMINATED, 0) | np.where(unknown, vd.VD_START_UNKNOWN, 0)).astype(np.uint32)}
    tune = vd.VdTune()
    tune.radix, tune.lanes = radix, lanes
    plan = vd.BatchPlan([vd.Code(K, GENS[K])], pk, tune=tune)
    out = torch.full((int(words.sum()),), -1, dtype=torch.int32, device="cuda")
    plan.launch(torch.from_numpy(arena.view(np.uint8)).cuda(), out)
    plan.status()
    want = oracle.decode_packets([oracle.Code(K, GENS[K])], np.zeros(n), off, n_info, f, v, term, unknown, word_off, arena,
                                 int(words.sum()), threads=THREADS)
    got = out.cpu().numpy().view(np.uint32)
    bad = [i for i in range(n) if not np.array_equal(got[word_off[i]:word_off[i] + words[i]],
                                                     want[word_off[i]:word_off[i] + words[i]])]
    assert not bad, (bad[:5], [(int(n_info[i]), int(f[i]), bool(term[i]), bool(unknown[i])) for i in bad[:5]])
    plan.close()


@pytest.mark.parametrize("form", [1, 2])
@pytest.mark.parametrize("K,lanes", SHAPES)
def test_streams_with_idle_groups(K, lanes, form):
    code, oc, beta = vd.Code(K, GENS[K]), oracle.Code(K, GENS[K]), len(GENS[K])
    tune = vd.VdTune()
    tune.lanes, tune.form = lanes, form
    for n, f, v in ((33, 32, 5), (64 * 5, 64, 200), (64 * 21 + 1, 64, 30), (32 * 67, 32, 9)):
        for unknown in (False, True):
            rng = np.random.Generator(np.random.PCG64(n + K + lanes))
            q = synth.make_stream(rng, K, GENS[K], n, 1.5, True).s8()
            out = torch.full(((n + 31) // 32,), -1, dtype=torch.int32, device="cuda")
            flags = vd.VD_TERMINATED | (vd.VD_START_UNKNOWN if unknown else 0)
            vd.vd_decode(code.handle, torch.from_numpy(q.view(np.uint8)).cuda(), vd.VD_LLR_S8, n, f, v, 2, flags, out, None, tune)
            vd.vd_sync()
            want = oracle.decode(oc, q.reshape(-1, beta).astype(np.int32), n, f, v, terminated=True, start_unknown=unknown)
            assert np.array_equal(out.cpu().numpy().view(np.uint32), want), (n, f, v, unknown)
