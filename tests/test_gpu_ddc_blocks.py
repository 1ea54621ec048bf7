"""The down-converter's tap blocks (16, 8 and single taps), plane layouts and
output packing at the sizes where they can go wrong, against the FP64 oracle:
filters of every remainder, the shortest chunks (all history), outputs that
are not a multiple of a thread's 16 or of a CTA's, and streams whose packed
output does not start on a 4-byte boundary."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2303_09886_gb300 import synth
from tests.fe_harness import streams
from tests.test_gpu_narrowband import _cuda, _run  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,Th,L", [(2, 1, 1 << 12), (2, 5, 16 * 131), (4, 3, 16 * 77), (8, 1, 48), (8, 7, 16 * 301),
                                    (8, 12, 1 << 15), (16, 9, 32 * 300), (16, 12, 1 << 16), (32, 5, 64 * 77),
                                    (32, 64, 1 << 15)])
def test_every_block_and_remainder(D, Th, L):
    fc, g, n_chunks = 0.213, 1.1, 2
    s = streams(synth.SEED_BASE + 950 + D + Th, 1, n_chunks * L, 40.0, tones=[(fc + 0.2 / D, 120.0, 0.2)])
    h = O.ddc_weights(D, Th)
    Lo = 2 * L // D
    for c, (packed, yf) in enumerate(_run(s, D, Th, L, fc, g, n_chunks)):
        for p in range(2):
            y_o, q_o = O.ddc(s[0, p].astype(np.int32), 0, D, h, fc, g, c * Lo, Lo)
            rel = np.sqrt(np.sum((yf[0, p].astype(np.float64) - y_o) ** 2) / np.sum(y_o ** 2))
            assert rel <= 1e-5, f"chunk {c} pol {p}: relative RMS {rel:.3g}"
            q = O.unpack10(packed[0, p], Lo)
            np.testing.assert_array_equal(q, [O.quantise10(v) for v in yf[0, p]])
            assert np.abs(q - q_o).max() <= 1
