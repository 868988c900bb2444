"""The separable kernels' failure path: a wait of the thread that issues a CTA's matrix operations
that runs out is reported, nothing is written from operands or accumulators that were not ready,
and the device stays usable (the plans have subgrids of one and of several tiles, batches and periods)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1909_07226_gb300 import idg
from paper_1909_07226_gb300 import synthetic as syn
from tests.gpu_util import dev, parity, workload_to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1909_07226_gb300 import build
    build.build()
    idg.load()


@pytest.mark.parametrize("L", [32, 24, 16])
@pytest.mark.parametrize("n_chan,n_t", [(1, 3), (9, 114)])
def test_an_issuing_thread_that_gives_up_is_reported_and_writes_nothing(L, n_chan, n_t):
    import torch
    wl = syn.make_small(seed=400 + n_t, n_st=3, n_t=n_t, n_chan=n_chan, L=L, N=8 * L, max_t=n_t, n_slots=1,
                        diameter_m=100.0, cell=2.0e-4, df=0.2e6, dt=1.0)
    p = idg.plan_from_workload(wl)
    op = O.plan(wl)
    assert p.stats.separable == 1
    d = workload_to_device(wl)
    G = syn.random_grid(np.random.default_rng(44), p.n_w_layers, wl.grid_size)
    model = dev(G)
    mark = complex(3.0, -7.0)
    g = torch.full(G.shape, mark, dtype=torch.complex64, device="cuda")
    v = torch.full(wl.vis.shape, mark, dtype=torch.complex64, device="cuda")
    idg.device_errors()
    idg.selftest_issue_timeout(p, d["vis"], model, d["aterms"], g, v)
    with pytest.raises(idg.IDGError) as ei:
        idg.device_errors()
    assert ei.value.status == 4
    idg.device_errors()                                 # the words were cleared
    assert torch.all(g == mark).item() and torch.all(v == mark).item()
    # the kernels run as before
    g.zero_()
    idg.grid(p, d["vis"], None, d["aterms"], d["taper"], g)
    idg.degrid(p, model, None, d["aterms"], d["taper"], v)
    idg.device_errors()
    parity(g.cpu().numpy(), O.grid(wl, op), f"grid after the self-test L={L}")
    parity(v.cpu().numpy(), O.degrid(wl, op, G), f"degrid after the self-test L={L}")
