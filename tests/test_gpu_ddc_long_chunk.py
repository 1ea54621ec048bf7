"""The down-converter on chunks whose stream is more than 2^32 words of packed
samples: the history it keeps for the next call is that of a down-converter fed
the chunk's last samples as a chunk of their own, bit for bit; and
the last outputs of chunks with more than 2^32 outputs."""
import pytest

from paper_2303_09886_gb300 import fengine
from tests.test_gpu_narrowband import _cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [16, 32])
def test_history_of_a_long_chunk(D):
    import torch
    Th, short = 8, 1 << 16
    L = (1 << 34) * 4 // 5 + (1 << 20)           # 5 L / 16 words of 32 bits: just over 2^32
    L -= L % (4 * D)
    assert 5 * L // 16 > 1 << 32 and L <= 1 << 34
    if torch.cuda.mem_get_info()[0] < 60e9:
        pytest.skip("needs 60 GB of device memory")
    g = torch.Generator(device="cuda")
    g.manual_seed(20230317 + D)
    nb = short * 5 // 4
    ends = torch.randint(0, 256, (2, 1, 2, nb), dtype=torch.uint8, device="cuda", generator=g)   # first, last samples
    x = torch.zeros((1, 2, L * 5 // 4), dtype=torch.uint8, device="cuda")
    x[..., :nb], x[..., -nb:] = ends[0], ends[1]

    def second_call(ddc, first, second, t):
        out = torch.empty((1, 2, ddc.out_samples * 5 // 4), dtype=torch.uint8, device="cuda")
        ddc.process(first, t, out)
        ddc.process(second, t + ddc.chunk_samples, out)
        torch.cuda.synchronize()
        ddc.close()
        return out

    want = second_call(fengine.DDC(1, D, Th, short, 0.213), ends[1], ends[0], L - short)
    got = second_call(fengine.DDC(1, D, Th, L, 0.213), x, x, 0)
    assert torch.equal(got[..., :want.shape[-1]], want)
    del x, got
    torch.cuda.empty_cache()


def test_outputs_beyond_32_bits():
    import torch
    D, Th, short, L = 2, 4, 1 << 16, (1 << 32) + (1 << 20)
    if torch.cuda.mem_get_info()[0] < 40e9:
        pytest.skip("needs 40 GB of device memory")
    g = torch.Generator(device="cuda")
    g.manual_seed(20230318)
    nb = short * 5 // 4
    last = torch.randint(0, 256, (2, 1, 2, nb), dtype=torch.uint8, device="cuda", generator=g)
    x = torch.zeros((1, 2, L * 5 // 4), dtype=torch.uint8, device="cuda")
    x[..., -2 * nb:-nb], x[..., -nb:] = last[0], last[1]
    ddc = fengine.DDC(1, D, Th, short, 0.213)
    want = torch.empty((1, 2, ddc.out_samples * 5 // 4), dtype=torch.uint8, device="cuda")
    for i in range(2):
        ddc.process(last[i], L - (2 - i) * short, want)
    torch.cuda.synchronize()
    ddc.close()
    ddc = fengine.DDC(1, D, Th, L, 0.213)
    got = torch.zeros((1, 2, ddc.out_samples * 5 // 4), dtype=torch.uint8, device="cuda")
    ddc.process(x, 0, got)
    torch.cuda.synchronize()
    ddc.close()
    assert torch.equal(got[..., -want.shape[-1]:], want)
    del x, got
    torch.cuda.empty_cache()
