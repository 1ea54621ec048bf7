"""The two second-stage kernels of 256 points give the same bits: a call with
enough CTAs for the one on pairs against its parts, which are far too small for
it. The sizes follow the device's SM count, on which the choice rests."""
import numpy as np
import pytest

from paper_2303_09886_gb300 import fengine, synth
from tests.fe_harness import Seg, run_gpu, streams
from tests.test_gpu_narrowband import _cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [fengine.FP32, fengine.TC_FP16, fengine.TC_BF16])
def test_both_sides_of_the_line_agree(precision):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n, T, parts, classes = 1024, 4, 12, 5
    each = -(-9 * sms // (classes * parts)) * 8 - 3          # spectra of a part
    M = parts * each
    assert classes * -(-M // 8) >= 8 * sms > 4 * classes * -(-each // 8)
    L = 2 * n * M
    s = streams(synth.SEED_BASE + 413, 1, L, 30.0, tones=[(0.17, 60.0, 0.4)])
    g = synth.random_gains(5, 4, n)
    gains = [[[(-(2 ** 62), g[0]), (2 * n * 1001, g[1])], [(-(2 ** 62), g[2]), (2 * n * 318, g[3])]]]
    delays = [[[Seg(delay=14.4, rate=1e-7, phase=0.3)], [Seg(delay=38.1)]]]
    kw = dict(S=each, D=64, taps=False, prequant=True, precision=precision)
    one, _, _ = run_gpu(s, n, T, L, 1, delays, gains, **kw)
    few, _, _ = run_gpu(s, n, T, L // parts, parts, delays, gains, **kw)
    np.testing.assert_array_equal(one[0]["out"], np.concatenate([r["out"] for r in few]))
    np.testing.assert_array_equal(one[0]["pre"], np.concatenate([r["pre"] for r in few], axis=2))
