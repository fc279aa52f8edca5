"""A batch whose time budget runs out: every model that did not transport all of its packages
reports it, also those no warp had turned to yet. The packages of a launch are shared out by
number, so a model of 100 beside one of 1e7 has to wait for the large one."""
import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_small", [3, 40, 300])
def test_unfinished_models_report_the_budget(n_small):
    n = [10 ** 7] + [100] * n_small
    large = w.disk_model(n_base=32, max_level=1, n_bins=50)
    small = w.sphere_model(n_base=4, n_bins=50)
    grids = [rt.Grid(large)] + [rt.Grid(small) for _ in range(n_small)]
    for g, k in zip(grids, n):
        g.emit_star(k)
    b = rt.Batch(grids, n, seed=0, budget_s=0.001)
    b.run()
    torch.cuda.synchronize()
    silent = []
    for i, (g, k) in enumerate(zip(grids, n)):
        sed = torch.zeros((2, g.n_dir, g.B), dtype=torch.int64, device="cuda")
        g.sed(out=sed)                       # a device read does not look at the status
        done = int(sed[0].sum())
        try:
            assert g.counters()["emitted"] == k == done
        except rt.RTError as e:
            assert e.code == 4               # RT_ERR_TIMEOUT
        except AssertionError:
            silent.append((i, done))
    assert not silent
    # the same plan without a limit finishes every model
    again = rt.Batch(grids, [20_000] + n[1:], seed=0)
    again.run()
    for g, k in zip(grids, [20_000] + n[1:]):
        assert g.counters()["emitted"] == k
    assert np.isfinite(again.temperatures(n_small)).all()
    b.close()
    again.close()
    for g in grids:
        g.close()
