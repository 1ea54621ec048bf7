"""The streamed tensor-core first stage over many delay steps, against the FP64
oracle: runs that leave most of a tile out (a run's samples alone are copied),
columns that wrap into the row before or after beside columns that do not, in
one stage, tiles whose runs take several accumulators in turn, and more runs
than accumulators. Bars: those of the reduced-precision forms."""
import pytest

from paper_2303_09886_gb300 import fengine, synth
from tests.fe_harness import REL_RMS_REDUCED, Seg, compare_call, run_gpu, streams
from tests.test_gpu_narrowband import _cuda  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [  # (channels, taps, antennas, spectra, delay, rate)
    (16384, 4, 1, 140, 33.4, 4e-6), (16384, 2, 1, 20, 700.2, -3e-5), (16384, 1, 2, 12, 0.6, 6e-5),
    (32768, 2, 1, 40, 2.2, 4e-6), (32768, 4, 2, 9, 1100.4, -4e-5), (32768, 1, 1, 30, 1500.4, 1.6e-5),
]


@pytest.mark.parametrize("precision", [fengine.TC_FP16, fengine.TC_BF16])
@pytest.mark.parametrize("n,T,ants,M,d,rate", CASES)
def test_many_runs(n, T, ants, M, d, rate, precision):
    L = 2 * n * M
    s = streams(synth.SEED_BASE + n + 5 * T + M, ants, L, 40.0, tones=[(0.21, 70.0, 0.3)])
    delays = [[[Seg(delay=d + 0.37 * p + 11 * a, rate=rate * (1 - 0.3 * p), phase=0.2)] for p in range(2)]
              for a in range(ants)]
    gains = [[synth.random_gains(9 * n + 2 * a + p, 1, n)[0] for p in range(2)] for a in range(ants)]
    res, M_, S_ = run_gpu(s, n, T, L, 1, delays, gains, S=min(M, 7), D=2048, precision=precision, taps=False)
    compare_call(s, res[0], M_, S_, n, T, delays, gains, rel_rms=REL_RMS_REDUCED)
