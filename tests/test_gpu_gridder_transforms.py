"""Gridding with the sorted or the compensated adder at L = 32: where the plan's gridder is the
separable one and its transform the FP32 one, gridder and transform run in one launch (no launch of
the transform in the profile); every other choice launches it separately.  Both against the FP64
oracle (tests.gpu_util.parity), at subgrid sizes around the gridder's groups, batches and periods."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1909_07226_gb300 import idg
from paper_1909_07226_gb300 import synthetic as syn
from tests.gpu_util import parity, workload_to_device

pytestmark = pytest.mark.gpu

SORTED, COMP = idg.ADDER_SORTED, idg.ADDER_COMPENSATED


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1909_07226_gb300 import build
    build.build()
    idg.load()


def _grid(L, n_chan, n_t, variant=0, **opts):
    import torch
    wl = syn.make_small(seed=600 + n_t, n_st=3, n_t=n_t, n_chan=n_chan, L=L, N=8 * L, max_t=n_t, n_slots=1, flag_p=0.1,
                        diameter_m=100.0, cell=2.0e-4, df=0.2e6, dt=1.0)
    p = idg.plan_from_workload(wl, **opts)
    idg.plan_set_kernel_variant(p, "gridder", variant)
    op = O.plan(wl)
    assert p.stats.separable == 1 and set(op.desc[:, O.D_KP].tolist()) == {n_chan * n_t}
    d = workload_to_device(wl)
    g = torch.zeros((p.n_w_layers, wl.grid_size, wl.grid_size, 4), dtype=torch.complex64, device="cuda")
    idg.profile_enable(True)
    try:
        idg.profile_read(reset=True)
        idg.grid(p, d["vis"], d["flags"], d["aterms"], d["taper"], g)
        launches = {k: r["launches"] for k, r in idg.profile_read(reset=True).items() if r["launches"]}
    finally:
        idg.profile_enable(False)
    idg.device_errors()
    parity(g.cpu().numpy(), O.grid(wl, op), f"grid L={L} K={n_chan * n_t} {opts}")
    return launches


# 1, 17, 255, 257, 513, 1026 visibilities
@pytest.mark.parametrize("n_chan,n_t", [(1, 1), (1, 17), (15, 17), (1, 257), (9, 57), (9, 114)])
@pytest.mark.parametrize("adder", [SORTED, COMP])
def test_one_launch_for_gridder_and_transform(adder, n_chan, n_t):
    assert _grid(32, n_chan, n_t, adder_mode=adder) == {"gridder": 1, "adder": 1}


@pytest.mark.parametrize("L,variant,opts", [
    (32, 0, dict(adder_mode=SORTED, fft_mode=idg.FFT_TC_SPLIT)),
    (32, 0, dict(adder_mode=SORTED, precision_mode=idg.PHASOR_RECURRENCE)),
    (32, 2, dict(adder_mode=COMP)),
    (24, 0, dict(adder_mode=SORTED)),
    (16, 0, dict(adder_mode=COMP)),
])
def test_a_separate_transform_otherwise(L, variant, opts):
    assert _grid(L, 9, 57, variant, **opts) == {"gridder": 1, "fft": 1, "adder": 1}
