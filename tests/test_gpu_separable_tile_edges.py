"""GPU parity of the separable tensor-core kernels where a subgrid's visibilities end in the
middle of the kernels' units: groups of 8 visibilities and stages of two groups, staged batches
of 256 and accumulation periods of 512 (gridder), tiles of 128 and lane quarters of 32
(degridder).  A plan has, per baseline, one subgrid of the size under test and one long one in a
second A-term slot, so that both directions run fused.  Against the FP64 oracle, relative RMS <=
1e-5 (tests.gpu_util.parity): the FP16 hi/lo products keep 22 bits and the first-order w
remainder of a separable plan is at most 2^-20, both well under the bound."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1909_07226_gb300 import idg
from paper_1909_07226_gb300 import synthetic as syn
from tests.gpu_util import dev, parity, workload_to_device

pytestmark = pytest.mark.gpu

# (channels, timesteps): 1, 7, 8, 9, 16, 17 | 33, 96, 128, 129 | 255, 256, 257 | 510, 513, 1026
SIZES = [(1, 1), (7, 1), (8, 1), (3, 3), (4, 4), (1, 17), (11, 3), (3, 32), (4, 32), (3, 43), (15, 17), (4, 64),
         (1, 257), (15, 34), (9, 57), (9, 114)]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1909_07226_gb300 import build
    build.build()
    idg.load()


@pytest.mark.parametrize("L", [32, 24, 16])
@pytest.mark.parametrize("n_chan,n_t", SIZES)
def test_sizes_around_the_kernels_units(L, n_chan, n_t):
    import torch
    long_t = -(-600 // n_chan)
    total = n_t + long_t
    wl = syn.make_small(seed=200 + n_t, n_st=3, n_t=total, n_chan=n_chan, L=L, N=8 * L, max_t=total, n_slots=2,
                        flag_p=0.1, diameter_m=100.0, cell=2.0e-4, df=0.2e6, dt=1.0)
    wl.aterm_offsets = np.array([0, n_t, total], dtype=np.int32)
    p = idg.plan_from_workload(wl)
    op = O.plan(wl)
    assert np.array_equal(p.export(), op.desc) and p.stats.separable == 1
    sizes = set(op.desc[:, O.D_KP].tolist())
    assert sizes == {n_chan * n_t, n_chan * long_t}
    d = workload_to_device(wl)
    g = torch.zeros((p.n_w_layers, wl.grid_size, wl.grid_size, 4), dtype=torch.complex64, device="cuda")
    v = torch.full(wl.vis.shape, complex(3.0, -7.0), dtype=torch.complex64, device="cuda")
    G = syn.random_grid(np.random.default_rng(41), p.n_w_layers, wl.grid_size)
    idg.profile_enable(True)
    try:
        idg.profile_read(reset=True)
        idg.grid(p, d["vis"], d["flags"], d["aterms"], d["taper"], g)
        idg.degrid(p, dev(G), d["flags"], d["aterms"], d["taper"], v)
        launches = {k: r["launches"] for k, r in idg.profile_read(reset=True).items() if r["launches"]}
    finally:
        idg.profile_enable(False)
    idg.device_errors()
    assert launches == {"gridder": 1, "degridder": 1}        # fused, the separable kernels
    parity(g.cpu().numpy(), O.grid(wl, op), f"grid L={L} K={n_chan * n_t}")
    parity(v.cpu().numpy(), O.degrid(wl, op, G), f"degrid L={L} K={n_chan * n_t}")


@pytest.mark.parametrize("L", [32, 24, 16])
def test_degrid_into_an_8_byte_aligned_buffer(L):
    # the fused separable degridder writes two polarisations at a time; a complex64 buffer
    # may start at any multiple of 8 bytes
    import torch
    wl = syn.make_small(seed=260, n_st=3, n_t=40, n_chan=5, L=L, N=8 * L, max_t=40, n_slots=1, flag_p=0.1,
                        diameter_m=100.0, cell=2.0e-4, df=0.2e6, dt=1.0)
    p = idg.plan_from_workload(wl)
    op = O.plan(wl)
    assert p.stats.separable == 1 and p.stats.n_vis_dropped == 0 and op.desc[:, O.D_KP].min() >= 64
    d = workload_to_device(wl)
    G = syn.random_grid(np.random.default_rng(43), p.n_w_layers, wl.grid_size)
    v = torch.full((wl.n_vis * 4 + 1,), complex(3.0, -7.0), dtype=torch.complex64, device="cuda")[1:].view(wl.vis.shape)
    assert v.data_ptr() % 16 == 8
    idg.degrid(p, dev(G), d["flags"], d["aterms"], d["taper"], v)
    idg.device_errors()
    parity(v.cpu().numpy(), O.degrid(wl, op, G), f"degrid L={L} into an 8-byte aligned buffer")
