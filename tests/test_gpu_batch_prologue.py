"""The members' prologues as one grid: more members than one grid holds (two
grids, of 64 and of the rest), with received-heap flags, delay and gain updates
of some members between calls, give the bytes of each plan's own calls."""
import numpy as np
import pytest

from paper_2303_09886_gb300 import fengine, synth

pytestmark = pytest.mark.gpu


def test_more_members_than_one_grid():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_09886_gb300 import build
    build.build()
    fengine.load()
    members, calls = 67, 2
    g = torch.Generator(device="cuda")
    g.manual_seed(synth.SEED_BASE + 5)
    spec = [(256, 4, 8 * (2 + i % 3)) if i % 2 else (1024, 8, 4 + 2 * (i % 3)) for i in range(members)]
    chunks = [[torch.randint(0, 256, (1, 2, 2 * n * m * 5 // 4), dtype=torch.uint8, device="cuda", generator=g)
               for _ in range(calls)] for n, _, m in spec]
    res = []
    for batched in (True, False):
        plans = [fengine.Plan(1, n, T, 2 * n * m, max_delay_samples=200) for n, T, m in spec]
        batch, outs = fengine.Batch(4), []
        for c in range(calls):
            todo = []
            for i, pl in enumerate(plans):
                n, _, m = spec[i]
                if c == 0 or i % 5 == 0:
                    for p in range(2):
                        pl.set_delay(0, p, 20.5 + i + c, 1e-9, 0.1 * i, 0.0, t_apply=c * pl.chunk_samples)
                        pl.set_gains(0, p, synth.random_gains(100 * i + 10 * c + p, 1, n)[0], c * pl.chunk_samples)
                heaps = pl.chunk_samples // fengine.HEAP_SAMPLES
                valid = torch.ones((1, 2, heaps), dtype=torch.uint8, device="cuda")
                valid[0, i % 2, heaps // 2] = i % 3 != 0
                out = torch.empty(pl.info.out_bytes, dtype=torch.int8, device="cuda")
                flags = torch.full((1, pl.heaps), 7, dtype=torch.uint8, device="cuda")
                todo.append((pl, chunks[i][c], c * pl.chunk_samples, out, valid, flags))
            if batched:
                batch.process(todo)
            else:
                for pl, x, t, out, valid, flags in todo:
                    pl.process(x, t, out, valid=valid, heap_flags=flags)
            torch.cuda.synchronize()
            outs += [(o.cpu().numpy(), f.cpu().numpy()) for _, _, _, o, _, f in todo]
        for pl in plans:
            pl.device_status()
            pl.close()
        batch.close()
        res.append(outs)
    for (o, f), (o2, f2) in zip(*res):
        np.testing.assert_array_equal(o, o2)
        np.testing.assert_array_equal(f, f2)
    assert {0, 1} == set(np.unique(np.concatenate([f.ravel() for _, f in res[0]])))
