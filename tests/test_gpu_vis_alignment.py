"""Degridding into a complex64 buffer that starts at a multiple of 8 but not of 16 bytes (a slice of
a larger one), in every kind of degridder: separable, direct on the tensor cores, packed FP32, scalar,
recurrence, and the batches' persistent kernels.  And gridding into such a grid on the fused
separable path, which adds 8 bytes at a time."""
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


def _sliced(shape):
    import torch
    n = int(np.prod(shape))
    t = torch.zeros(n + 1, dtype=torch.complex64, device="cuda")[1:].view(shape)
    assert t.data_ptr() % 16 == 8
    return t


NARROW = dict(diameter_m=100.0, cell=2.0e-4, df=0.2e6, dt=1.0)
CASES = {
    "direct_L8": (dict(L=8, N=64, n_t=20, n_chan=5, max_t=20), {}),
    "direct_L48": (dict(L=48, N=192, n_t=20, n_chan=5, max_t=20), {}),
    "tensor_core_L32": (dict(L=32, N=512, cell=1e-3, diameter_m=800.0, n_t=80, n_chan=8, max_t=80), {}),
    "short_L32": (dict(L=32, N=512, cell=1e-3, diameter_m=800.0, n_t=12, n_chan=1, max_t=3), {}),
    "recurrence_L32": (dict(L=32, N=256, n_t=40, n_chan=9, max_t=40, **NARROW), dict(precision_mode=idg.PHASOR_RECURRENCE)),
    "separable_L32": (dict(L=32, N=256, n_t=40, n_chan=9, max_t=40, **NARROW), {}),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_degrid_into_a_buffer_of_8_byte_alignment(case):
    kw, opts = CASES[case]
    wl = syn.make_small(seed=500, n_st=4, n_slots=1, flag_p=0.1, **kw)
    p = idg.plan_from_workload(wl, **opts)
    op = O.plan(wl)
    d = workload_to_device(wl)
    G = syn.random_grid(np.random.default_rng(45), p.n_w_layers, wl.grid_size)
    v = _sliced(wl.vis.shape)
    # (a range takes every subgrid whole: the direct kernels where one is past the remainder bound)
    idg.degrid_range(p, 0, p.n_subgrids, dev(G), d["flags"], d["aterms"], d["taper"], v)
    idg.device_errors()
    parity(v.cpu().numpy(), O.degrid(wl, op, G), f"degrid {case}, 8-byte aligned")


def test_batch_degrid_into_a_buffer_of_8_byte_alignment():
    wl = syn.make_small(seed=501, n_st=4, n_t=20, n_chan=5, L=8, N=64, max_t=20, n_slots=1, flag_p=0.1)
    p = idg.plan_from_workload(wl)
    op = O.plan(wl)
    d = workload_to_device(wl)
    G = syn.random_grid(np.random.default_rng(46), p.n_w_layers, wl.grid_size)
    v = _sliced(wl.vis.shape)
    b = idg.Batch([p], [dict(vis_out=v, flags=d["flags"], aterms=d["aterms"], taper=d["taper"], grid=dev(G))])
    b.degrid()
    idg.device_errors()
    parity(v.cpu().numpy(), O.degrid(wl, op, G), "batch degrid, 8-byte aligned")


@pytest.mark.parametrize("L", [32, 24, 16])
def test_grid_into_a_grid_of_8_byte_alignment(L):
    wl = syn.make_small(seed=502, n_st=4, n_t=40, n_chan=9, L=L, N=8 * L, max_t=40, n_slots=1, flag_p=0.1, **NARROW)
    p = idg.plan_from_workload(wl)
    op = O.plan(wl)
    assert p.stats.separable == 1
    d = workload_to_device(wl)
    g = _sliced((p.n_w_layers, wl.grid_size, wl.grid_size, 4))
    idg.grid(p, d["vis"], d["flags"], d["aterms"], d["taper"], g)
    idg.device_errors()
    parity(g.cpu().numpy(), O.grid(wl, op), f"grid L={L}, 8-byte aligned")
