"""The hand-over of staged visibility batches in the separable gridder (csrc/staging.h): every
interleaving of one loader and several readers, with barriers that know only the parity of
their phase (as mbarriers do), over the header's own buffer, barrier and parity rules.  In no
reachable state may a reader meet another batch than its own, may the loader fill a buffer that
a reader still uses, or may every side wait for ever."""
import ctypes
import os
import subprocess

import pytest

from paper_1909_07226_gb300 import build as B

SHIM = """
#include "staging.h"
extern "C" {
int buffers() { return idg::kStagingBuffers; }
int barriers() { return idg::kStagingBarriers; }
int buffer_of(int b) { return idg::staging_buffer(b); }
int barrier_of(int b) { return idg::staging_barrier(b); }
unsigned full_parity(int b) { return idg::staging_full_parity(b); }
unsigned free_parity(int b) { return idg::staging_free_parity(b); }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("staging")
    src, lib = os.path.join(d, "shim.cpp"), os.path.join(d, "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", B.CSRC, src, "-o", lib], check=True)
    return ctypes.CDLL(lib)


def _passes(phase, parity):
    # a parity wait passes when the phase of that parity was the last to complete
    return (phase & 1) != parity


def _explore(r, n_batches, n_readers):
    """Breadth-first over (loader step, reader steps, barrier phases, arrivals pending on the free
    barriers, batch in each buffer); returns the number of states, raises on a violation.  A loader
    step is (batch, 0 wait | 1 fill | 2 arrive), a reader's (batch, 0 wait | 1 read | 2 arrive)."""
    nb, nu = r.barriers(), r.buffers()
    start = ((1, 0), ((0, 1),) * n_readers, (0,) * nb, (0,) * nb, (0,) * nb, (0,) + (-1,) * (nu - 1))
    seen, todo = {start}, [start]
    while todo:
        loader, readers, full, free, pending, held = state = todo.pop()
        out = []
        b, step = loader
        if b < n_batches:
            k, bar = r.buffer_of(b), r.barrier_of(b)
            if step == 0:
                if b < nu or _passes(free[bar], r.free_parity(b)):
                    out.append(((b, 1), readers, full, free, pending, held))
            elif step == 1:
                inside = [rb for rb, rs in readers if rb < b and r.buffer_of(rb) == k]
                assert not inside, f"batch {b} is filled while a reader is at batch {inside[0]}"
                out.append(((b, 2), readers, full, free, pending, held[:k] + (b,) + held[k + 1:]))
            else:
                out.append(((b + 1, 0), readers, full[:bar] + (full[bar] + 1,) + full[bar + 1:], free, pending, held))
        for i, (b, step) in enumerate(readers):
            if b >= n_batches:
                continue
            k, bar = r.buffer_of(b), r.barrier_of(b)
            move = lambda to, fr=free, pe=pending: (loader, readers[:i] + (to,) + readers[i + 1:], full, fr, pe, held)
            if step == 0:
                if _passes(full[bar], r.full_parity(b)):
                    out.append(move((b, 1)))
            elif step == 1:
                assert held[k] == b, f"a reader of batch {b} meets batch {held[k]}"
                out.append(move((b, 2)))
            else:
                n = pending[bar] + 1
                done = n == n_readers
                out.append(move((b + 1, 0), free[:bar] + (free[bar] + done,) + free[bar + 1:],
                                pending[:bar] + (0 if done else n,) + pending[bar + 1:]))
        ended = loader[0] >= n_batches and all(b >= n_batches for b, _ in readers)
        assert out or ended, f"every side waits: loader {loader}, readers {readers}, full {full}, free {free}"
        for s in out:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return len(seen)


@pytest.mark.parametrize("n_batches,n_readers", [(1, 2), (2, 2), (3, 2), (7, 1), (9, 2), (7, 3)])
def test_every_interleaving_ends_with_the_right_batches(rules, n_batches, n_readers):
    assert _explore(rules, n_batches, n_readers) > 0
