"""The tensor-core first stage with streamed operand blocks (16384 channels and
more) at the sizes where it can go wrong, against the FP64 oracle: one to a few
tiles and items per unit (units with idle accumulators), odd numbers of spectra
(a pair with one spectrum), slabs whose last tile is partial, delay steps inside
a pair and a tile (one round over the blocks per run, pairs written by two
rounds), window taps, every contraction length from the padded single tap to
32 taps, and heaps whose rows are not 4-byte multiples. Bars: those of the
reduced-precision forms."""
import pytest

from paper_2303_09886_gb300 import fengine, synth
from tests.fe_harness import REL_RMS_REDUCED, Seg, compare_call, run_gpu, streams

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_09886_gb300 import build
    build.build()
    fengine.load()


CASES = [  # (channels, taps, spectra per call, spectra per heap, calls, slab, delay, rate, taps out)
    (16384, 1, 7, 7, 1, 0, 3.2, 0.0, True), (16384, 16, 1, 1, 3, 0, 600.4, 0.0, True),
    (16384, 8, 130, 5, 1, 128, 70.1, 0.0, False), (16384, 4, 9, 3, 1, 0, 200.3, 2e-5, True),
    (32768, 2, 5, 5, 2, 0, 90.7, 1e-5, True), (32768, 32, 3, 3, 1, 0, 44.4, 0.0, False),
    (32768, 4, 34, 17, 1, 32, 130.6, -2e-5, False),
]


@pytest.mark.parametrize("precision", [fengine.TC_FP16, fengine.TC_BF16])
@pytest.mark.parametrize("n,T,M,S,calls,slab,d,rate,taps", CASES)
def test_streamed_blocks(n, T, M, S, calls, slab, d, rate, taps, precision):
    L = 2 * n * M
    s = streams(synth.SEED_BASE + n + 3 * T + M, 1, calls * L, 40.0, tones=[(0.21, 70.0, 0.3)])
    gains = [[synth.random_gains(7 * n + p, 1, n)[0] for p in range(2)]]
    delays = [[[Seg(delay=d + 0.3 * p, rate=rate, phase=0.2)] for p in range(2)]]
    res, M_, S_ = run_gpu(s, n, T, L, calls, delays, gains, S=S, D=int(d) + 64, precision=precision, slab_spectra=slab,
                          taps=taps)
    for r in res:
        compare_call(s, r, M_, S_, n, T, delays, gains, rel_rms=REL_RMS_REDUCED)
