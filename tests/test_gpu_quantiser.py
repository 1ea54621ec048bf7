"""The requantiser of every second-stage kernel on chosen values. With a filter
that is 1 at its first tap and 0 elsewhere, and a unit impulse at the start of
each spectrum, every product and sum of the transform is exact, so that a
channel's spectrum is its gain: exact ties, their neighbours, values beyond the
8-bit range up to the largest float. The bytes are those of fengine_quantise, in
both epilogues (with and without the spectra before quantisation)."""
import numpy as np
import pytest

from paper_2303_09886_gb300 import fengine, synth
from tests.test_gpu_narrowband import _cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _values(n):
    """complex64 [n]: every tie in [-130, 130] with its neighbours, extremes, and random values; at most n."""
    h = np.arange(-260, 261).astype(np.float32) / 2
    up = np.nextafter(h, np.float32(np.inf))
    down = np.nextafter(h, np.float32(-np.inf))
    big = np.array([127.25, 127.499, 127.5, 128.4, 255.5, 1e4, 2.2e9, 4.3e9, 1e30, np.finfo(np.float32).max, 1e-30,
                    0.49999997, 0.0], np.float32)
    v = np.concatenate([big, -big, h, up, down])
    rng = np.random.default_rng(20230317)
    v = np.concatenate([v, rng.uniform(-140, 140, max(0, 2 * n - v.size)).astype(np.float32)])
    v = v[:2 * n] if 2 * n < v.size else v
    return rng.permutation(v)[:2 * n].view(np.complex64)


KERNELS = [  # (channels, spectra, precision); spectra 0: enough for the kernel that large calls take
    (16, 9, fengine.FP32), (64, 5, fengine.FP32), (1024, 3, fengine.FP32), (1024, 0, fengine.FP32),
    (2048, 5, fengine.FP32), (8192, 7, fengine.FP32), (32768, 3, fengine.FP32),
    (64, 5, fengine.TC_FP16), (2048, 5, fengine.TC_FP16), (8192, 7, fengine.TC_FP16), (32768, 3, fengine.TC_FP16),
    (2048, 5, fengine.TC_BF16), (8192, 7, fengine.TC_BF16), (32768, 3, fengine.TC_BF16),
]


@pytest.mark.parametrize("n,M,precision", KERNELS)
def test_bytes_are_the_rule_s(n, M, precision):
    import torch
    if M == 0:
        M = 8 * (-(-8 * torch.cuda.get_device_properties(0).multi_processor_count // 5)) + 1
    N = 2 * n
    w = np.zeros(N, np.float32)
    w[0] = 1.0
    gains = [_values(n), np.ascontiguousarray(_values(n)[::-1])]
    plan = fengine.Plan(1, n, 1, N * M, spectra_per_heap=M, weights=w, precision=precision)
    s = np.zeros(N * M, np.int16)
    s[::N] = 1
    packed = torch.from_numpy(np.stack([synth.pack10(s)] * 2)[None]).cuda()
    for p in range(2):
        plan.set_gains(0, p, gains[p])
    for call, want_pre in enumerate([True, False]):
        out = torch.empty(plan.info.out_bytes, dtype=torch.int8, device="cuda")
        pre = torch.empty((2, M, n, 2), device="cuda") if want_pre else None
        plan.process(packed, call * N * M, out, pre)
        torch.cuda.synchronize()
        got = out.cpu().numpy().reshape(n, M, 2, 2)
        for p in range(2):
            g = gains[p].view(np.float32).reshape(n, 2)
            if want_pre:
                np.testing.assert_array_equal(pre[p].cpu().numpy(), np.broadcast_to(g, (M, n, 2)))
            want = np.array([fengine.quantise(float(x)) for x in g.ravel()], np.int8).reshape(n, 1, 2)
            np.testing.assert_array_equal(got[:, :, p], np.broadcast_to(want, (n, M, 2)))
    plan.device_status()
    plan.close()
