"""Device buffers that the kernels could not address are refused on the host, before any launch:
gridding reads visibilities and A-terms, and degridding the grid, 16 bytes at a time; visibilities
that a call writes may start at any multiple of 8.  The addresses here are made up and never used:
without a CUDA device an aligned call goes on to the refusal of a host-only plan."""
import ctypes

import pytest

from paper_1909_07226_gb300 import build as B
from paper_1909_07226_gb300 import idg
from paper_1909_07226_gb300 import synthetic as syn

OK16, OK8, OFF8, OFF4 = 0x1000, 0x1008, 0x1008, 0x1004
P = ctypes.c_void_p


@pytest.fixture(scope="module")
def lib():
    import torch
    if torch.cuda.is_available():
        pytest.skip("made-up addresses: only where no kernel can run")
    B.build()
    return idg.load()


@pytest.fixture(scope="module")
def plan(lib):
    wl = syn.make_small(seed=1, n_st=4, n_t=8, n_chan=2, L=16, N=64, with_vis=False, aterms="identity")
    p = idg.plan_from_workload(wl)
    assert p.n_subgrids > 1
    return p


# entry point -> call with its buffers {name: address}, and each buffer's alignment
CALLS = {
    "idg_grid": (lambda L, h, b: L.idg_grid(h, b["d_vis"], None, b["d_aterms"], None, b["d_grid"], None),
                 dict(d_vis=16, d_aterms=16)),
    "idg_degrid": (lambda L, h, b: L.idg_degrid(h, b["d_grid"], None, b["d_aterms"], None, b["d_vis_out"], None),
                   dict(d_grid=16, d_aterms=16, d_vis_out=8)),
    "idg_grid_range": (lambda L, h, b: L.idg_grid_range(h, 0, 1, b["d_vis"], None, b["d_aterms"], None, b["d_grid"], None),
                       dict(d_vis=16, d_aterms=16)),
    "idg_degrid_range": (lambda L, h, b: L.idg_degrid_range(h, 0, 1, b["d_grid"], None, b["d_aterms"], None,
                                                            b["d_vis_out"], None),
                         dict(d_grid=16, d_aterms=16, d_vis_out=8)),
    "idg_aterm_gradient": (lambda L, h, b: L.idg_aterm_gradient(h, b["d_grid"], b["d_vis"], None, b["d_aterms"], None,
                                                                b["d_residual"], b["d_gradient"], None, None),
                           dict(d_grid=16, d_vis=16, d_aterms=16, d_residual=16, d_gradient=16)),
    "idg_grid_no_alloc": (lambda L, h, b: L.idg_grid_no_alloc(h, b["d_vis"], None, b["d_aterms"], P(OK16), b["d_grid"], None),
                          dict(d_vis=16, d_aterms=16, d_grid=16)),
    "idg_classical_grid": (lambda L, h, b: L.idg_classical_grid(h, 8, 8, 0.0, b["d_vis"], None, b["d_aterms"], None,
                                                                b["d_grid"], None),
                           dict(d_vis=16, d_aterms=8, d_grid=16)),
    "idg_grid_subgrids": (lambda L, h, b: L.idg_grid_subgrids(h, 0, 1, b["d_vis"], None, b["d_aterms"], None,
                                                              b["d_subgrids"], None),
                          dict(d_vis=16, d_aterms=16, d_subgrids=16)),
    "idg_fft_subgrids": (lambda L, h, b: L.idg_fft_subgrids(h, 1, 1, b["d_subgrids"], None), dict(d_subgrids=16)),
    "idg_add_subgrids": (lambda L, h, b: L.idg_add_subgrids(h, 0, 1, b["d_subgrids"], b["d_grid"], None),
                         dict(d_subgrids=16, d_grid=16)),
    "idg_split_subgrids": (lambda L, h, b: L.idg_split_subgrids(h, 0, 1, b["d_grid"], b["d_subgrids"], None),
                           dict(d_grid=16, d_subgrids=16)),
    "idg_degrid_subgrids": (lambda L, h, b: L.idg_degrid_subgrids(h, 0, 1, b["d_subgrids"], None, b["d_aterms"], None,
                                                                  b["d_vis_out"], None),
                            dict(d_subgrids=16, d_aterms=16, d_vis_out=8)),
    "idg_image_from_grid": (lambda L, h, b: L.idg_image_from_grid(h, b["d_grid"], None, b["d_image"], None),
                            dict(d_grid=16, d_image=16)),
    "idg_grid_from_image": (lambda L, h, b: L.idg_grid_from_image(h, b["d_image"], None, b["d_grid"], None),
                            dict(d_image=16, d_grid=16)),
}
NAMES = ["d_vis", "d_aterms", "d_grid", "d_vis_out", "d_residual", "d_gradient", "d_subgrids", "d_image"]


def _refused_for(lib, name):
    return name.encode() + b" must start at a multiple of" in lib.idg_last_error()


@pytest.mark.parametrize("entry", sorted(CALLS))
def test_misaligned_buffers_are_refused(lib, plan, entry):
    call, need = CALLS[entry]
    for name, bytes_ in need.items():
        for off in ([OFF8, OFF4] if bytes_ == 16 else [OFF4]):
            bufs = {k: P(OK16) for k in NAMES}
            bufs[name] = P(off)
            assert call(lib, plan.handle, bufs) == 1
            assert _refused_for(lib, name), (entry, name, off, lib.idg_last_error())


@pytest.mark.parametrize("entry", sorted(CALLS))
def test_aligned_buffers_are_not(lib, plan, entry):
    call, need = CALLS[entry]
    bufs = {k: P(OK8 if need.get(k) == 8 else OK16) for k in NAMES}
    assert call(lib, plan.handle, bufs) != 0                       # (no device)
    assert b"must start at a multiple" not in lib.idg_last_error()


def test_a_call_that_touches_no_buffer_is_not_refused_for_one(lib, plan):
    st = lib.idg_grid_range(plan.handle, 0, 0, P(OFF8), None, None, None, P(OFF8), None)
    assert st == 1 and b"without a CUDA device" in lib.idg_last_error()
