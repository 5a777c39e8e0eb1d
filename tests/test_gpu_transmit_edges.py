"""vd_transmit at the edges of its single-precision path (values a rounding
border leaves open come from the double-precision transform): stream ends
inside a thread's eight values, output at any alignment, noise from none to far
beyond the clip, against the oracle's double-precision samples.  Quantised
values are equal or wrong; the only exception is a sample within 1e-9 of a
quantiser border (relative 1e-10 for half precision), where the two sides'
double-precision libraries may differ.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2011_13579_gb300 as vd  # noqa: E402
from paper_2011_13579_gb300 import synth  # noqa: E402
from test_gpu_transmit import TYPES, _near_boundary, _unpack  # noqa: E402


@pytest.mark.parametrize("kind", ["s8", "s4", "f16", "hard"])
@pytest.mark.parametrize("sigma", [0.0, 1e-3, 0.5, 30.0, 1e6])
def test_transmit_edges(kind, sigma):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if kind == "f16" and sigma == 0.0:
        pytest.skip("half-precision values need noise")
    vd.build()
    rng = np.random.Generator(np.random.PCG64(820))
    # one kept value per stage, one per period of two; whole, partial and single groups of eight
    patterns = (None, [[1, 1], [1, 0]], [[1, 0], [0, 1]], [[1], [0]])
    for i, n in enumerate((1, 2, 3, 5, 8, 13, 4096, 65537)):
        for pat in patterns:
            pattern = None if pat is None else np.array(pat, np.uint8)
            code = vd.Code(7, synth.K7_GENS, puncture=pat)
            oc = oracle.Code(7, synth.K7_GENS, puncture=pattern)
            bits = synth.random_bits(rng, n)
            d_bits = torch.from_numpy(oracle.pack_bits(bits).view(np.int32)).cuda()
            nb = vd.vd_transmit_bytes(code.handle, n, vd.VD_TERMINATED, TYPES[kind])
            off = 2 * (i % 8) if kind == "f16" else i % 8
            buf = torch.full((nb + 32,), 0xA5, dtype=torch.uint8, device="cuda")
            vd.vd_transmit(code.handle, d_bits, n, vd.VD_TERMINATED, sigma, 7, 5 + n, TYPES[kind], buf[off:off + nb])
            raw = buf.cpu().numpy()
            assert np.all(raw[:off] == 0xA5) and np.all(raw[off + nb:] == 0xA5)
            y = oracle.transmit(oc, bits, n, True, sigma, 7, 5 + n)
            got, want = _unpack(raw[off:off + nb].copy(), kind, y.size), oracle.quantise(y, kind, sigma)
            if kind == "f16":
                got, want = got.view(np.uint16), want.view(np.uint16)
            assert not np.any((got != want) & ~_near_boundary(y, kind, sigma)), (n, pat)
