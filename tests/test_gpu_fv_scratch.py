"""Memory of the two-launch step: a grid holds its fields only while a call
runs, whatever the number of grids, streams and threads; a call captured into
a graph has fields of its own, and gives the bits of a plain one."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KW = dict(tau=0.3, tau_g=0.25, dt=0.05, beta=1e-2, grav=1.0, T0=1.0, T_bot=1.3, T_top=0.8, u0=0.02, amp=0.01)
GIB = 1 << 30


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_grids_hold_no_fields_between_calls(lbgpu):
    """Ten FP64 thermal grids of 1024 x 512 need 216 MiB of fields each while
    they step.  Afterwards the library keeps at most 1 GiB of it, and nothing
    once the grids are gone."""
    lb = lbgpu
    lb.Grid(8, 8, store="f64").init(kind=lb.LB_INIT_TGV, **KW).step_fv(1).close()
    free0 = _free()
    grids = [lb.Grid(1024, 512, thermal=True, store="f64").init(kind=lb.LB_INIT_TGV, **KW) for _ in range(10)]
    free1 = _free()
    for g in grids:
        assert g.fv_schedule() == (lb.LB_FV_TILE, 2)
        g.step_fv(2)  # all ten in flight at once
    assert free1 - _free() <= GIB + (64 << 20)
    assert np.isfinite(grids[-1].conservation()).all()
    for g in grids:
        g.close()
    assert free0 - _free() <= 64 << 20


def test_streams_and_threads_borrow_apart(lbgpu):
    """Grids on streams of their own, stepped from threads of their own at the
    same time, in many short calls: the bits of a grid stepped alone."""
    import torch
    lb = lbgpu

    def grid(k, stream=None):
        return lb.Grid(70 + 8 * k, 61, bcy=1, thermal=True, store="f64", stream=stream).init(kind=lb.LB_INIT_TGV, **KW)

    want = []
    for k in range(4):
        g = grid(k)
        want.append(g.step_fv(60).get_pops())
        g.close()
    streams = [torch.cuda.Stream() for _ in range(4)]
    grids = [grid(k, streams[k].cuda_stream) for k in range(4)]
    torch.cuda.synchronize()
    bad = []

    def run(k):
        try:
            for n in (1, 2, 3, 4) * 6:
                grids[k].step_fv(n)
        except Exception as e:  # noqa: BLE001
            bad.append(e)

    threads = [threading.Thread(target=run, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    for g, w in zip(grids, want):
        for a, b in zip(g.get_pops(), w):
            assert np.array_equal(a, b)
        g.close()


@pytest.mark.parametrize("store", ["f64", "f32"])
def test_captured_call(lbgpu, store):
    """The first call of a grid, captured: the same launches and, replayed, the same bits as a plain call."""
    import torch
    lb = lbgpu
    stream = torch.cuda.Stream()
    outs = []
    for captured in (False, True):
        g = lb.Grid(96, 50, bcy=1, thermal=True, store=store, stream=stream.cuda_stream)
        g.init(kind=lb.LB_INIT_TGV, **KW)
        g.sync()
        l0 = lb.lb_kernel_launches()
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                g.step_fv(8)
            with torch.cuda.stream(stream):
                graph.replay()
        else:
            g.step_fv(8)
        assert lb.lb_kernel_launches() - l0 == 17
        outs.append(g.get_pops())
        if captured:
            del graph
        g.close()
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
