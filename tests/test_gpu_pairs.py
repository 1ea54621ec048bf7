"""Phase 1's spans, sweeps and spectrum pairs and the packed second stage at
the sizes where they can go wrong, against the FP64 oracle: calls of one, few
and odd numbers of spectra (a pair with one spectrum, CTAs of 8 to 128 rows),
windows that begin in the history at every alignment of it, chunks that are
not 16-byte aligned, 32 taps (two sweeps), delay steps at block edges, heaps
whose rows are 4, 8 and 16-byte aligned, and gain sets that change inside a
work item."""
import numpy as np
import pytest

from paper_2303_09886_gb300 import fengine, synth
from tests.fe_harness import Seg, compare_call, run_gpu, streams

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_09886_gb300 import build
    build.build()
    fengine.load()


CASES = [  # (channels, taps, spectra per call, spectra per heap, calls, delay, rate, bytes into a buffer)
    (16, 16, 70, 7, 2, 3.2, 0.0, 0), (32, 8, 45, 0, 2, 11.4, 0.0, 4), (64, 32, 131, 5, 2, 5.5, 0.0, 0),
    (128, 4, 37, 3, 2, 17.7, 0.0, 8), (256, 32, 65, 4, 2, 50.3, 0.0, 0), (1024, 16, 1, 1, 18, 7.3, 0.0, 0),
    (1024, 32, 129, 6, 1, 30.1, 0.0, 12), (1024, 2, 33, 0, 1, 0.0, 0.0, 0), (1024, 1, 40, 8, 1, 9.5, 0.0, 0),
    (4096, 16, 3, 3, 7, 120.6, 0.0, 0), (4096, 8, 35, 5, 2, 2.0, 0.0, 4), (4096, 4, 66, 6, 1, 77.2, 2e-6, 0),
    (8192, 16, 34, 34, 1, 600.4, 1e-6, 0), (8192, 32, 9, 2, 1, 44.9, 0.0, 0), (16384, 16, 10, 10, 1, 90.2, 0.0, 0),
    (32768, 32, 5, 4, 1, 33.3, 0.0, 4),
]


@pytest.mark.parametrize("n,T,M,S,calls,d,rate,off", CASES)
def test_pairs_spans_and_sweeps(n, T, M, S, calls, d, rate, off):
    L = 2 * n * M
    s = streams(synth.SEED_BASE + n + T + M, 1, calls * L, 30.0, tones=[(0.13, 60.0, 0.4)])
    gains = [[synth.random_gains(5 * n + p, 1, n)[0] for p in range(2)]]
    delays = [[[Seg(delay=d + 0.3 * p, rate=rate, phase=0.2)] for p in range(2)]]
    res, M_, S_ = run_gpu(s, n, T, L, calls, delays, gains, S=S, D=int(d) + 64, taps=False, in_offset=off)
    for r in res:
        compare_call(s, r, M_, S_, n, T, delays, gains)


def test_gain_sets_change_inside_a_work_item():
    """A set applied two spectra into a group of four, at another spectrum in
    the other polarisation, with and without the spectra before quantisation:
    the 8-bit output is the same bytes."""
    n, T, M = 4096, 8, 24
    L = 2 * n * M
    s = streams(synth.SEED_BASE + 77, 1, L, 30.0, tones=[(0.2, 50.0, 0.1)])
    g = synth.random_gains(9, 4, n)
    gains = [[[(-(2 ** 62), g[0]), (2 * n * 6, g[1])], [(-(2 ** 62), g[2]), (2 * n * 9, g[3])]]]
    delays = [[[Seg(delay=4.4)], [Seg(delay=8.1)]]]
    a, M_, S_ = run_gpu(s, n, T, L, 1, delays, gains, D=32, taps=False)
    compare_call(s, a[0], M_, S_, n, T, delays, gains)
    b, _, _ = run_gpu(s, n, T, L, 1, delays, gains, D=32, taps=False, prequant=False)
    np.testing.assert_array_equal(a[0]["out"], b[0]["out"])


@pytest.mark.parametrize("n,T,M,off", [(1024, 16, 33, 0), (4096, 8, 9, 4), (2048, 32, 70, 0), (8192, 4, 2, 12)])
def test_shared_64_point_transforms(n, T, M, off):
    """First radix 64 (two threads per transform) behind every second stage, with one to many row pairs per
    block, windows that begin in the history, and chunks that are not 16-byte aligned (copies word by word)."""
    L = 2 * n * M
    s = streams(synth.SEED_BASE + 31 * n + M, 1, 2 * L, 30.0, tones=[(0.31, 60.0, 0.4)])
    gains = [[synth.random_gains(3 * n + p, 1, n)[0] for p in range(2)]]
    delays = [[[Seg(delay=20.2 + 5.5 * p, rate=1e-6, phase=0.4)] for p in range(2)]]
    res, M_, S_ = run_gpu(s, n, T, L, 2, delays, gains, D=64, taps=False, fft_n1=64, in_offset=off)
    for r in res:
        compare_call(s, r, M_, S_, n, T, delays, gains)
