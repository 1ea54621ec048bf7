"""The memory a plan takes: one that fits with slabs of 256 MiB is made, however
little the device has left beside it (the built-in slab gives way, the rest of
the plan does not), and the slabs of a call that takes several are even."""
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


@pytest.mark.parametrize("precision", [fengine.FP32, fengine.TC_FP16])
def test_slabs_are_even(precision):
    n, ants = 8192, 8
    per_spectrum = 2 * ants * 9 * 1024 * (8 if precision == fengine.FP32 else 4)
    M = (3 << 30) // per_spectrum + 40                     # a little more than 3 GiB of intermediate
    plan = fengine.Plan(ants, n, 4, 2 * n * M, precision=precision)
    k, slab = int(plan.info.slabs_per_chunk), int(plan.info.slab_spectra)
    bytes_ = int(plan.info.scratch_bytes)
    plan.close()
    assert k >= 2 and slab % 32 == 0 and k * slab < M + 32 * k
    if precision == fengine.FP32:
        assert bytes_ < 2 * slab * per_spectrum + (1 << 20)
