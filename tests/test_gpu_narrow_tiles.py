"""Phase-1 tiles of fewer than 512 columns (16 to 128 channels), whose CTAs have a
thread per pair of columns: every tap count against the FP64 oracle, over more
than one tile and block, with delay steps, odd spectra and a second call whose
first rows lie in the history."""
import pytest

from paper_2303_09886_gb300 import synth
from tests.fe_harness import REL_RMS_FP32, Seg, compare_call, run_gpu, streams
from tests.test_gpu_narrowband import _cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 2, 4, 8, 16, 32])
@pytest.mark.parametrize("n,M,rate", [(16, 333, 0.0), (32, 161, 2e-4), (64, 97, 0.0), (128, 65, 1e-4)])
def test_every_tap_count(n, M, rate, T):
    L = 2 * n * M
    s = streams(synth.SEED_BASE + 40 * n + T, 1, 2 * L, 30.0, tones=[(0.13, 60.0, 0.4)])
    delays = [[[Seg(delay=21.3 + 7.7 * p, rate=rate, phase=0.2)] for p in range(2)]]
    gains = [[synth.random_gains(3 * n + p, 1, n)[0] for p in range(2)]]
    res, M_, S_ = run_gpu(s, n, T, L, 2, delays, gains, S=17, D=64, taps=False)
    for r in res:
        compare_call(s, r, M_, S_, n, T, delays, gains, rel_rms=REL_RMS_FP32)
