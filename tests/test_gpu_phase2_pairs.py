"""The second stage on pairs of spectra (256 and 512 points): a call large enough
for it gives the bytes (and the spectra before quantisation) of small calls,
which the other kernel does, in every form of the intermediate; and the sizes
where it can go wrong against the FP64 oracle: odd numbers of spectra, heaps
whose rows are 4, 8 and 16-byte aligned or end inside a group of four, gain sets
that change inside a pair, first radices with many classes."""
import numpy as np
import pytest

from paper_2303_09886_gb300 import fengine, synth
from tests.fe_harness import REL_RMS_FP32, REL_RMS_REDUCED, Seg, compare_call, run_gpu, streams

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_09886_gb300 import build
    build.build()
    fengine.load()


@pytest.mark.parametrize("precision", [fengine.FP32, fengine.TC_FP16, fengine.TC_BF16])
@pytest.mark.parametrize("prequant", [False, True])
def test_large_and_small_calls_agree(precision, prequant):
    n, T, M, parts = 1024, 4, 1956, 12          # 5 x 245 CTAs in one call, 5 x 21 in each of the parts
    L = 2 * n * M
    s = streams(synth.SEED_BASE + 411, 1, L, 30.0, tones=[(0.17, 60.0, 0.4)])
    g = synth.random_gains(3, 4, n)
    gains = [[[(-(2 ** 62), g[0]), (2 * n * 1001, g[1])], [(-(2 ** 62), g[2]), (2 * n * 318, g[3])]]]
    delays = [[[Seg(delay=14.4, rate=1e-7, phase=0.3)], [Seg(delay=38.1)]]]
    kw = dict(S=M // parts, D=64, taps=False, prequant=prequant, precision=precision)
    one, _, _ = run_gpu(s, n, T, L, 1, delays, gains, **kw)
    few, _, _ = run_gpu(s, n, T, L // parts, parts, delays, gains, **kw)
    np.testing.assert_array_equal(one[0]["out"], np.concatenate([r["out"] for r in few]))
    if prequant:
        np.testing.assert_array_equal(one[0]["pre"], np.concatenate([r["pre"] for r in few], axis=2))


CASES = [  # (channels, taps, spectra, spectra per heap, first radix, delay, bytes into a buffer)
    (2048, 4, 1, 1, 0, 3.2), (2048, 16, 37, 5, 0, 20.7), (2048, 8, 66, 6, 0, 9.9), (2048, 2, 40, 8, 0, 0.0),
    (4096, 4, 19, 19, 16, 5.1), (8192, 2, 7, 2, 32, 61.3), (16384, 4, 6, 6, 64, 17.7), (2048, 1, 15, 15, 0, 2.5),
]


@pytest.mark.parametrize("n,T,M,S,n1,d", CASES)
def test_512_points_match_oracle(n, T, M, S, n1, d):
    L = 2 * n * M
    s = streams(synth.SEED_BASE + 7 * n + M, 1, L, 30.0, tones=[(0.13, 60.0, 0.4)])
    g = synth.random_gains(11, 3, n)
    gains = [[[(-(2 ** 62), g[0]), (2 * n * (M // 2 | 1), g[1])], g[2]]]
    delays = [[[Seg(delay=d + 0.3 * p, phase=0.2)] for p in range(2)]]
    res, M_, S_ = run_gpu(s, n, T, L, 1, delays, gains, S=S, D=int(d) + 64, taps=False, fft_n1=n1)
    compare_call(s, res[0], M_, S_, n, T, delays, gains, rel_rms=REL_RMS_FP32)


@pytest.mark.parametrize("precision", [fengine.TC_FP16, fengine.TC_BF16])
def test_512_points_behind_the_tensor_cores(precision):
    n, T, M = 2048, 8, 133
    L = 2 * n * M
    s = streams(synth.SEED_BASE + 92, 1, L, 40.0, tones=[(0.21, 70.0, 0.3)])
    gains = [[synth.random_gains(17 + p, 1, n)[0] for p in range(2)]]
    delays = [[[Seg(delay=40.3 + p, phase=0.2)] for p in range(2)]]
    res, M_, S_ = run_gpu(s, n, T, L, 1, delays, gains, S=7, D=128, taps=False, precision=precision)
    compare_call(s, res[0], M_, S_, n, T, delays, gains, rel_rms=REL_RMS_REDUCED)
