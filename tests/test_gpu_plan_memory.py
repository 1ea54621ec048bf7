"""The memory a plan takes: one that fits with slabs of 256 MiB is made, however
little the device has left beside it (the built-in slab gives way, the rest of
the plan does not)."""
import pytest

from paper_2303_09886_gb300 import fengine
from tests.test_gpu_narrowband import _cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def test_plan_next_to_little_free_memory():
    import torch
    n, ants, M = 1024, 12, 1 << 17
    if torch.cuda.mem_get_info()[0] < 60e9:
        pytest.skip("needs 60 GB of device memory")
    shape = dict(n_antennas=ants, n_channels=n, n_taps=4, chunk_samples=2 * n * M, precision=fengine.TC_BF16)
    per_spectrum = 2 * ants * 5 * 256 * 8                  # of the intermediate, FP32 pairs of 5 classes x 256
    slab = (256 << 20) // per_spectrum // 32 * 32
    plan = fengine.Plan(**shape, slab_spectra=slab)
    need = int(plan.info.device_bytes)
    assert need > 20e9                                     # mostly the column sequences
    plan.close()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - need - (256 << 20), dtype=torch.uint8, device="cuda")
    try:
        plan = fengine.Plan(**shape)
        assert plan.info.slab_spectra >= slab
        plan.close()
    finally:
        del fill
        torch.cuda.empty_cache()
