"""The calls that do not synchronise work under stream capture: the no-alloc step
and a run of steps with a device read, each replayed from a graph with the bits of
the direct call, also where the capture begins with a memset or a copy."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1701_07452_gb300 import binding
    binding.lib()
    return binding


class Capture:
    """A graph of what the body enqueues on stream (thread-local capture)."""

    def __init__(self, lib, stream):
        self.lib, self.s = lib, ctypes.c_void_p(stream.cuda_stream)
        self.graph, self.exe = ctypes.c_void_p(), ctypes.c_void_p()

    def __enter__(self):
        assert self.lib.cudaStreamBeginCapture(self.s, 1) == 0
        return self

    def __exit__(self, *exc):
        rc = self.lib.cudaStreamEndCapture(self.s, ctypes.byref(self.graph))
        if exc[0] is None:
            assert rc == 0

    def kernels(self):
        n = ctypes.c_size_t(0)
        assert self.lib.cudaGraphGetNodes(self.graph, None, ctypes.byref(n)) == 0
        nodes = (ctypes.c_void_p * n.value)()
        assert self.lib.cudaGraphGetNodes(self.graph, nodes, ctypes.byref(n)) == 0
        kind, count = ctypes.c_int(0), 0
        for v in nodes:
            assert self.lib.cudaGraphNodeGetType(ctypes.c_void_p(v), ctypes.byref(kind)) == 0
            count += kind.value == 0  # cudaGraphNodeTypeKernel
        return count

    def replay(self):
        if not self.exe:
            assert self.lib.cudaGraphInstantiate(ctypes.byref(self.exe), self.graph, ctypes.c_ulonglong(0)) == 0
        assert self.lib.cudaGraphLaunch(self.exe, self.s) == 0

    def __del__(self):
        if self.exe:
            self.lib.cudaGraphExecDestroy(self.exe)
        if self.graph:
            self.lib.cudaGraphDestroy(self.graph)


@pytest.mark.parametrize("bc", [(0, 0, 0), (1, 0, 1)])
@pytest.mark.parametrize("lead", ["nothing", "memset", "copy"])
def test_noalloc_step_captured(wb, bc, lead):
    import torch
    from paper_1701_07452_gb300.initial_conditions import random_box
    n = (12, 10, 9)
    stream = torch.cuda.Stream()
    inputs = []
    for seed in (5, 6):
        st = random_box(n, seed=seed)
        g = wb.Grid(n, length=st["length"], bc=bc, stream=stream)
        g.load_state(st)
        inputs.append([t.clone() for t in g.read(on_device=True)[:4]])
        stream.synchronize()
    d = wb.make_desc(n, length=st["length"], bc=bc)
    held = [torch.empty_like(t) for t in inputs[0]]
    outs = [torch.empty_like(t) for t in inputs[0]]
    dt = torch.zeros(1, dtype=torch.float64, device="cuda")
    with torch.cuda.stream(stream):
        wb.step_noalloc(d, *inputs[0], *outs, dt, stream=stream)  # module loading stays outside the capture
        stream.synchronize()
        cap = Capture(wb.lib(), stream)
        with cap:
            if lead == "memset":
                assert wb.lib().cudaMemsetAsync(ctypes.c_void_p(dt.data_ptr()), 0, ctypes.c_size_t(8), cap.s) == 0
            if lead == "copy":
                assert wb.lib().cudaMemcpyAsync(ctypes.c_void_p(outs[0].data_ptr()), ctypes.c_void_p(held[0].data_ptr()),
                                                ctypes.c_size_t(8), 3, cap.s) == 0
            wb.step_noalloc(d, *held, *outs, dt, stream=stream)
        for src in inputs:
            want, wdt = [torch.empty_like(t) for t in src], torch.zeros_like(dt)
            wb.step_noalloc(d, *src, *want, wdt, stream=stream)
            for h, s in zip(held, src):
                h.copy_(s)
            cap.replay()
            stream.synchronize()
            assert torch.equal(dt, wdt) and float(dt) > 0
            for a, b in zip(outs, want):
                assert torch.equal(a, b)


@pytest.mark.parametrize("n,kw", [((20, 16, 12), {}), ((20, 16, 12), {"bc": (1, 0, 0)}), ((24, 20, 1), {}),
                                  ((24, 24, 24), {"patches": (2, 2, 2)}),
                                  ((32, 32, 24), {"patches": (2, 2, 2), "batch_patches": 4}),
                                  ((24, 24, 24), {"patches": (2, 2, 2), "batch_patches": 3})])
def test_steps_and_device_read_captured(wb, n, kw):
    """Three steps a replay; the kernels of a step are those that the bench counts."""
    import torch

    import bench
    from paper_1701_07452_gb300.initial_conditions import random_box
    st = random_box(n, seed=9)
    stream = torch.cuda.Stream()
    runs = []
    for captured in (False, True):
        g = wb.Grid(n, length=st["length"], stream=stream, **kw)
        g.load_state(st)
        out = g.read(on_device=True)
        if captured:
            counts = []
            for steps in (2, 3):
                cap = Capture(wb.lib(), stream)
                with cap:
                    g.advance(steps, sync=False)
                counts.append(cap.kernels())
            assert counts[1] - counts[0] == bench.step_launches(g.desc)
            cap = Capture(wb.lib(), stream)
            with cap:
                g.advance(3, sync=False)
                g._check(wb.lib().wb_read_state(g._h, *[ctypes.c_void_p(t.data_ptr()) for t in out], 1))
            cap.replay()
            cap.replay()
        else:
            g.advance(6)
            g._check(wb.lib().wb_read_state(g._h, *[ctypes.c_void_p(t.data_ptr()) for t in out], 1))
        stream.synchronize()
        runs.append([t.cpu().numpy() for t in out] + [np.float64(g.counters()["t"])])
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
