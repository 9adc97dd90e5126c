"""Allocation-free counts of two grids in flight at once, from two threads on
two streams: each call returns its own bond count (the static scratch that the
calls share holds no more than the overflow flag)."""
import ctypes
import threading

import pytest
import torch

import pd_workloads as W

pytestmark = pytest.mark.gpu


def test_overlapping_counts_are_their_own(built_lib):
    pd = built_lib
    grids = [W.Grid(140, 40, 40, 1e-3, 3.01), W.Grid(60, 40, 40, 1e-3, 3.01, 1, 60, 20)]
    want = [pd.build_neighbours(g)[1].numel() for g in grids]
    rows = [torch.empty(g.n_nodes + 1, dtype=torch.int32, device="cuda") for g in grids]
    streams = [torch.cuda.Stream() for _ in grids]
    torch.cuda.synchronize()
    got = [[], []]
    start = threading.Barrier(2)

    def count(k):
        G, nb = pd.grid_struct(grids[k]), ctypes.c_int64(0)
        start.wait(timeout=60)
        for _ in range(300):
            rc = pd.lib().pd_build_neighbours_noalloc(ctypes.byref(G), pd._ptr(rows[k]), None, 0, ctypes.byref(nb),
                                                      pd._stream(streams[k]))
            got[k].append((rc, nb.value))

    threads = [threading.Thread(target=count, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=120)
    for k in range(2):
        assert got[k] == [(pd.PD_OK, want[k])] * 300
