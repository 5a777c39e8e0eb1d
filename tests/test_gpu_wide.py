"""The forms of vd_decode for few frames (a pair over many lanes with its
survivors in shared memory; long frames in segments) against the CPU oracle: decoded bits and canonical final metrics, element by element.

Sizes sit at the form's edges: streams shorter than the K-1 memory, one pair,
a pair with one frame, a warp's four pairs (K=7) and one more, frames long
enough for one pair per warp, frames whose first stage falls at every place of
a chunk of K-1 stages, several frames that begin at stage 0 (v >= f), values at any byte offset.  Integer
arithmetic: equal or wrong, no tolerance.
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
SHAPES = ([(1, 32, 8), (31, 32, 0), (33, 64, 6), (70, 64, 100), (256, 256, 42), (513, 256, 42), (2048, 256, 42), (2049, 256, 42),
           (2999, 3000, 8), (9001, 128, 30)] + [(200 + i, 4096, 8) for i in range(8)] + [(300, 64, v) for v in range(8, 16)])
# frames decoded in segments: one block's worth, a chunk more than a whole number of segments, clusters of 2 to 8 blocks,
# several long frames, frames too long for one block's shared memory
LONG = {7: [(400, 400, 6), (1151, 1151, 6), (4096, 4096, 6), (4601, 4601, 0), (20011, 20011, 6), (9000, 2048, 42), (3000, 640, 700)],
        9: [(520, 520, 8), (1031, 1031, 8), (4096, 4096, 8), (9001, 9001, 8), (6000, 2048, 64)]}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vd.build()
    yield


def values(K, n, T, kind, rng):
    beta = len(GENS[K])
    if kind == "noisy":
        return synth.make_stream(rng, K, GENS[K], n, 1.0, T > n).s8()
    if kind == "zeros":
        return np.zeros(beta * T, np.int8)
    if kind == "faint":      # no codeword and hardly any information: survivors take long to meet, segments run again
        return rng.integers(-1, 2, beta * T).astype(np.int8) * (rng.random(beta * T) < 0.15)
    if kind == "saturated":
        return (127 * (1 - 2 * rng.integers(0, 2, beta * T))).astype(np.int8)
    q = rng.integers(-127, 128, beta * T).astype(np.int8)
    q[rng.random(beta * T) < 0.6] = 0
    return q


@pytest.mark.parametrize("kind", ["noisy", "zeros", "saturated", "erasures"])
@pytest.mark.parametrize("term,unknown", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("K", [7, 9])
def test_wide_matches_oracle(K, term, unknown, kind):
    rng = np.random.Generator(np.random.PCG64(700 + K + 2 * term + unknown))
    code, oc, beta = vd.Code(K, GENS[K]), oracle.Code(K, GENS[K]), len(GENS[K])
    check(K, code, oc, beta, SHAPES, term, unknown, kind, rng)


@pytest.mark.parametrize("kind", ["noisy", "zeros", "erasures", "faint"])
@pytest.mark.parametrize("term,unknown", [(True, False), (False, True)])
@pytest.mark.parametrize("K", [7, 9])
def test_segmented_frames_match_oracle(K, term, unknown, kind):
    rng = np.random.Generator(np.random.PCG64(900 + K + 2 * term + unknown))
    check(K, vd.Code(K, GENS[K]), oracle.Code(K, GENS[K]), len(GENS[K]), LONG[K], term, unknown, kind, rng)


def check(K, code, oc, beta, shapes, term, unknown, kind, rng):
    for i, (n, f, v) in enumerate(shapes):
        T = n + (K - 1 if term else 0)
        q = values(K, n, T, kind, rng)
        buf = torch.zeros(q.size + 16, dtype=torch.uint8, device="cuda")
        off = i % 4
        buf[off:off + q.size] = torch.from_numpy(q.view(np.uint8)).cuda()
        out, pm = vd.decode(code, buf[off:off + q.size], n, f, v, terminated=term, start_unknown=unknown, want_pm=True)
        ow, opm = oracle.decode(oc, q.reshape(T, beta).astype(np.int32), n, f, v, terminated=term, start_unknown=unknown,
                                threads=max(1, len(os.sched_getaffinity(0))), want_pm=True)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), ow), (n, f, v)
        whole = [min(T, (s + 1) * f + v) - max(0, s * f - v) >= K - 1 for s in range(pm.shape[0])]
        assert np.array_equal(pm.cpu().numpy()[whole].astype(np.int64), opm[whole]), (n, f, v)


@pytest.mark.parametrize("K,lanes,sizes", [(7, 1, (3_000_001, 9_000_000, 16_000_007, 21_000_000)),
                                           (9, 4, (1_500_001, 3_000_000, 9_000_000, 12_000_001, 21_000_000))])
def test_every_choice_of_form_gives_the_same_bits(K, lanes, sizes):
    """Streams on each side of the lines between the forms: what the library
    chooses, for either radix, against the one-wave kernel with the lanes named."""
    rng = np.random.Generator(np.random.PCG64(950 + K))
    code, beta = vd.Code(K, GENS[K]), len(GENS[K])
    f, v = (256, 42) if K == 7 else (512, 64)
    q = torch.from_numpy(synth.make_stream(rng, K, GENS[K], 1 << 20, 2.0, False).s8().view(np.uint8)).cuda()
    q = q.repeat(sizes[-1] // (1 << 20) + 1)      # one received stretch over and over: a codeword but at the seams
    tune = vd.VdTune()
    tune.lanes, tune.form = lanes, 2
    for n in sizes:
        outs = [torch.full(((n + 31) // 32,), -1, dtype=torch.int32, device="cuda") for _ in range(3)]
        vd.vd_decode(code.handle, q[:beta * n], vd.VD_LLR_S8, n, f, v, 2, vd.VD_START_UNKNOWN, outs[0], None, tune)
        for radix, out in ((2, outs[1]), (4, outs[2])):
            vd.vd_decode(code.handle, q[:beta * n], vd.VD_LLR_S8, n, f, v, radix, vd.VD_START_UNKNOWN, out)
        vd.vd_sync()
        assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2]), n
