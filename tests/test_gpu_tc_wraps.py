"""The tensor-core first stage with resident operand blocks (below 16384 channels)
where a pass at another delay than the columns' own has some of a CTA's columns
wrap into the row before or after: one of them, all of them, delays further apart
than the columns, both signs, one and two columns per output column, against the
FP64 oracle. Bars: those of the reduced-precision forms."""
import pytest

from paper_2303_09886_gb300 import fengine, synth
from tests.fe_harness import REL_RMS_REDUCED, Seg, compare_call, run_gpu, streams
from tests.test_gpu_narrowband import _cuda  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [  # (channels, taps, spectra, delay, rate)
    (64, 4, 300, 20.3, 3e-4), (1024, 8, 150, 3.4, 2e-5), (1024, 2, 40, 900.2, -2e-3), (4096, 4, 130, 50.4, 4e-6),
    (8192, 2, 140, 40.3, -2e-6), (8192, 4, 20, 100.1, 2e-4), (8192, 1, 30, 1600.4, -2e-4),
]


@pytest.mark.parametrize("precision", [fengine.TC_FP16, fengine.TC_BF16])
@pytest.mark.parametrize("n,T,M,d,rate", CASES)
def test_wrapping_columns(n, T, M, d, rate, precision):
    L = 2 * n * M
    s = streams(synth.SEED_BASE + 3 * n + 5 * T + M, 1, L, 40.0, tones=[(0.21, 70.0, 0.3)])
    delays = [[[Seg(delay=d + 0.37 * p, rate=rate * (1 - 0.3 * p), phase=0.2)] for p in range(2)]]
    gains = [[synth.random_gains(9 * n + p, 1, n)[0] for p in range(2)]]
    res, M_, S_ = run_gpu(s, n, T, L, 1, delays, gains, S=min(M, 7), D=4096, precision=precision, taps=False)
    compare_call(s, res[0], M_, S_, n, T, delays, gains, rel_rms=REL_RMS_REDUCED)
