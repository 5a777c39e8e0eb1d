"""The input pre-pass (erased positions, 4-bit values, hard decisions) at the
edges of its output words: every period from 1 to 8, sources at any byte
offset, lengths whose last word is partial.  A stream decoded from its kept values
equals the stream decoded from the same values expanded by numpy (erased positions 0); single
streams and a batch of packets.  Whole numbers: equal or wrong.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2011_13579_gb300 as vd  # noqa: E402
from paper_2011_13579_gb300 import synth  # noqa: E402

GENS = {7: synth.K7_GENS, 9: synth.K9_GENS}
TYPES = {"s8": vd.VD_LLR_S8, "s4": vd.VD_LLR_S4, "hard": vd.VD_LLR_HARD}


def packed(q, kind):
    return q.view(np.uint8) if kind == "s8" else synth.pack_s4(q) if kind == "s4" else synth.pack_hard((q < 0).astype(np.uint8))


@pytest.mark.parametrize("kind", ["s8", "s4", "hard"])
@pytest.mark.parametrize("K", [7, 9])
def test_prepass_equals_expansion(K, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vd.build()
    rng = np.random.Generator(np.random.PCG64(1000 + K))
    beta, f, v = len(GENS[K]), 64, 20
    full = vd.Code(K, GENS[K])
    for period in range(1, 9):
        pattern = rng.integers(0, 2, (beta, period))
        pattern[rng.integers(0, beta), pattern.sum(axis=0) == 0] = 1
        code = vd.Code(K, GENS[K], puncture=pattern.tolist())
        packets, wants, raws, offset = [], [], [], 0
        for n in (1, 2, 3, 7, 8, 61, 1000, 4099):
            T = n + K - 1
            mask = np.tile(pattern.T.astype(bool), (-(-T // period), 1))[:T]
            q = rng.integers(-7, 8, int(mask.sum())).astype(np.int8)
            if kind == "hard":
                q = np.where(q < 0, -1, 1).astype(np.int8)
            whole = np.zeros((T, beta), np.int8)
            whole[mask] = q
            want = vd.decode(full, torch.from_numpy(whole.reshape(-1).view(np.uint8)).cuda(), n, f, v, terminated=True)
            raw = packed(q, kind)
            off = int(rng.integers(0, 4))
            buf = torch.full((raw.size + 8,), 0xFF, dtype=torch.uint8, device="cuda")
            buf[off:off + raw.size] = torch.from_numpy(raw).cuda()
            got = vd.decode(code, buf[off:off + raw.size], n, f, v, terminated=True, llr_type=TYPES[kind])
            assert torch.equal(got, want), (period, n)
            packets.append(n)
            wants.append(want)
            raws.append((raw, offset))
            offset += raw.size + int(rng.integers(0, 3))
        arena = np.full(offset + 8, 0xFF, np.uint8)
        for raw, o in raws:
            arena[o:o + raw.size] = raw
        words = np.array([(n + 31) // 32 for n in packets])
        outs = np.concatenate([[0], np.cumsum(words)[:-1]])
        per = {"s8": 1, "s4": 2, "hard": 8}[kind]
        pk = {"n_info": np.array(packets), "llr_offset": per * np.array([o for _, o in raws]), "out_word_offset": outs,
              "llr_type": np.full(len(packets), TYPES[kind]), "flags": np.full(len(packets), vd.VD_TERMINATED),
              "f": np.full(len(packets), f), "v": np.full(len(packets), v)}
        out = torch.zeros(int(words.sum()), dtype=torch.int32, device="cuda")
        plan = vd.BatchPlan([code], pk)
        plan.launch(torch.from_numpy(arena).cuda(), out)
        torch.cuda.synchronize()
        for want, o in zip(wants, outs):
            assert torch.equal(out[o:o + want.numel()], want), period
