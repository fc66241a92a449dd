"""The kernels of a call overlap the end of the one before them (programmatic launches):
repeated calls back to back, calls on two streams and a captured call give the same bits."""
import numpy as np
import pytest
import torch

import grkv_inputs as gi
from paper_2605_31105_gb300 import binding as b
from tests import gpu_cases as G

pytestmark = pytest.mark.gpu

WL = {
    "m128": gi.Workload("chain128", 6, 4, 1500, 128, 32, 300, 7, 1e-2, "bf16", "lowrank", 91),
    "m256": gi.Workload("chain256", 3, 4, 1500, 128, 64, 300, 7, 1e-1, "bf16", "spans", 92),
    "f32": gi.Workload("chainf32", 2, 2, 900, 128, 16, 150, 7, 1e-2, "f32", "lowrank", 93),
}


class Call:
    def __init__(self, wl, ragged):
        self.c = G.Case(wl)
        self.p = G.lib_params(wl, wl.units)
        self.p.flags = b.GRKV_DETERMINISTIC
        self.budgets = [wl.budget - 40 * u for u in range(wl.units)] if ragged else None
        size = b.grkv_compress_ragged_workspace_size(self.p, self.budgets) if ragged \
            else b.grkv_workspace_size(self.p)
        rows = sum(self.budgets) if ragged else wl.units * wl.budget
        dt = torch.float32 if wl.dtype == "f32" else torch.bfloat16
        self.ws = torch.full((size,), 0xFF, dtype=torch.uint8, device="cuda")
        self.idx = torch.empty((rows,), dtype=torch.int32, device="cuda")
        self.ko = torch.empty((rows, 128), dtype=dt, device="cuda")
        self.vo = torch.empty_like(self.ko)

    def run(self):
        c = self.c
        if self.budgets:
            b.grkv_compress_ragged(self.p, self.budgets, c.dq, c.dk, c.dv, self.ko, self.vo,
                                   self.idx, self.ws)
        else:
            b.grkv_compress(self.p, c.dq, c.dk, c.dv, self.ko, self.vo, self.idx, self.ws)

    def out(self):
        torch.cuda.synchronize()
        return [t.clone() for t in (self.idx, self.ko, self.vo)]

    def wipe(self):
        for t in (self.idx, self.ko, self.vo, self.ws):
            t.view(torch.uint8).fill_(0xFF)


def _same(got, want):
    for g, w in zip(got, want):
        np.testing.assert_array_equal(g.view(torch.uint8).cpu().numpy(),
                                      w.view(torch.uint8).cpu().numpy())


@pytest.mark.parametrize("ragged", [False, True], ids=["compress", "ragged"])
@pytest.mark.parametrize("name", list(WL))
def test_chained_calls(grkv_lib, name, ragged):
    call, other = Call(WL[name], ragged), Call(WL[name], ragged)
    call.run()
    want = call.out()
    for _ in range(20):     # back to back, each over the last one's workspace
        call.run()
    _same(call.out(), want)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for x in (call, other):
        x.wipe()
    torch.cuda.synchronize()
    for _ in range(10):
        for st, x in zip(streams, (call, other)):
            with torch.cuda.stream(st):
                x.run()
    _same(call.out(), want)
    _same(other.out(), want)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call.run()
    call.wipe()
    for _ in range(3):
        graph.replay()
    _same(call.out(), want)
