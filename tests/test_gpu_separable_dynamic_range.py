"""Weak visibilities beside strong ones in the separable gridder.  Each subgrid holds 2048
visibilities, with the identity as A-terms, so that the polarisations stay apart.  Polarisation 0
sets the subgrid's scale: by one visibility `ratio` times the others, or by being `1 / cross` times
polarisations 1 and 2 throughout (parallel hands beside cross hands).  The other polarisations'
grids must stay as accurate as without it.

Bound: the two phasors of a product have FP32 phases of at most 35 rad (rms rounding of phase and
coefficient 5e-7 each), sine and cosine 2e-7, and the tensor cores' accumulation over 512
visibilities adds about as much: 1e-6 together, 3e-6 with room.  The hi/lo products of values kept
to 22 bits of their own, or to 2^-13 of a quantum of 1/128 of their polarisation's mean, add 2e-7; a
quantum fixed below the subgrid's largest value, on the other hand, 3e-5 at a ratio of 300 or a cross
of 0.01 and 3e-4 at a ratio of 10^4."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1909_07226_gb300 import idg
from paper_1909_07226_gb300 import synthetic as syn
from tests.gpu_util import parity, workload_to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1909_07226_gb300 import build
    build.build()
    idg.load()


@pytest.mark.parametrize("ratio,cross", [(1.0, 1.0), (300.0, 1.0), (1e4, 1.0), (1.0, 0.01)])
@pytest.mark.parametrize("L", [32, 24, 16])
def test_weak_visibilities_beside_strong_ones(L, ratio, cross):
    import torch
    wl = syn.make_small(seed=300, n_st=4, n_t=128, n_chan=16, L=L, N=8 * L, max_t=128, n_slots=1, flag_p=0.0,
                        aterms="identity", diameter_m=100.0, cell=2.0e-4, df=0.2e6, dt=1.0)
    wl.vis = syn.gaussian_noise(np.random.default_rng(301), wl.vis.shape, 1.0)
    wl.vis[:, 37, 5, 0] *= np.float32(ratio)
    wl.vis[..., 1:3] *= np.float32(cross)
    p = idg.plan_from_workload(wl)
    op = O.plan(wl)
    assert p.stats.separable == 1 and op.desc[:, O.D_KP].min() >= 2048
    d = workload_to_device(wl)
    g = torch.zeros((p.n_w_layers, wl.grid_size, wl.grid_size, 4), dtype=torch.complex64, device="cuda")
    idg.grid(p, d["vis"], d["flags"], d["aterms"], d["taper"], g)
    idg.device_errors()
    got, ref = g.cpu().numpy(), O.grid(wl, op)
    for pol in (1, 2, 3):
        parity(got[..., pol], ref[..., pol], f"pol {pol} L={L} ratio={ratio:g} cross={cross:g}", tol=3e-6)
