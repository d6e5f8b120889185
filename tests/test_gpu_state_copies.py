"""State in and out by device arrays.  FP32 bulk takes arrays of this device
straight to its float planes and back; anything else (managed memory, pointers
that are not 8-byte aligned, ranges that leave their allocation) takes the copies.
Both ways and host arrays give the same bits."""
import ctypes
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2508_13705_gb300 import cgks, inputs  # noqa: E402

NAMES = ("W", "Wx", "Wy", "Wx_line", "Wy_line")
FORMS = [(dim, precision) for dim in (1, 2) for precision in (cgks.FP64, cgks.FP32_BULK)]


def new(dim, precision, **kw):
    """A solver of 37 cells or 13 x 7 and a state for it (None: no such field)."""
    if dim == 1:
        return cgks.Solver(1, 9, 37, precision=precision, **kw), list(inputs.shu_osher_1d(37)[:2]) + [None] * 3
    ext = (0.0, 1.3, 0.0, 0.7)
    prim = lambda x, y: (1 + 0.2 * np.sin(5 * x) * np.cos(4 * y), 0.3 + 0.1 * y, 0.1 - 0.2 * x, 1 + 0.1 * np.cos(3 * x))
    st = inputs.cell_state_2d(prim, 13, 7, ext, 5)
    return cgks.Solver(2, 5, 13, 7, extent=ext, precision=precision, **kw), list(st)


def cuda(a):
    return None if a is None else torch.from_numpy(np.array(a, np.float64, order="C")).cuda()


def assert_same(a, b):
    assert set(a) == set(b)
    for n in a:
        assert np.array_equal(a[n], b[n]), n


@pytest.mark.parametrize("dim,precision", FORMS)
def test_device_and_host_arrays_mix(dim, precision):
    h, st = new(dim, precision)
    d, _ = new(dim, precision)
    h.set_state(*st)
    d.set_state_device(*[cuda(a) for a in st])
    for _ in range(2):  # as set, and after a step
        want = h.get_state()
        assert_same(d.get_state(), want)
        out = {n: torch.full(a.shape, float("nan"), dtype=torch.float64, device="cuda") for n, a in want.items()}
        h.get_state_device(out)
        torch.cuda.synchronize()
        assert_same({n: a.cpu().numpy() for n, a in out.items()}, want)
        dt = h.compute_dt()
        h.step(dt)
        d.step(dt)
        h.sync()
        d.sync()


@pytest.mark.parametrize("dim,precision", FORMS)
def test_fields_are_read_alone(dim, precision):
    s, st = new(dim, precision)
    s.set_state_device(*[cuda(a) for a in st])
    s.step(s.compute_dt())
    want = s.get_state()
    for n in want:
        out = torch.full(want[n].shape, float("nan"), dtype=torch.float64, device="cuda")
        s.get_state_device({n: out})
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want[n]), n


class Managed:
    """Managed memory of n doubles."""

    def __init__(self, n):
        self.p = ctypes.c_void_p()
        assert cgks.lib().cudaMallocManaged(ctypes.byref(self.p), ctypes.c_size_t(8 * n), 1) == 0
        self.a = np.ctypeslib.as_array(ctypes.cast(self.p, ctypes.POINTER(ctypes.c_double)), (n,))

    def close(self):
        torch.cuda.synchronize()
        del self.a
        assert cgks.lib().cudaFree(self.p) == 0


class Unaligned:
    """Device memory of n doubles from the middle of one on."""

    def __init__(self, n):
        self.t = torch.empty(8 * n + 8, dtype=torch.uint8, device="cuda")[4:8 * n + 4]
        self.p = ctypes.c_void_p(self.t.data_ptr())

    @property
    def a(self):
        return np.frombuffer(self.t.cpu().numpy().tobytes(), np.float64)

    def fill(self, x):
        self.t.copy_(torch.from_numpy(np.frombuffer(x.tobytes(), np.uint8).copy()))

    def close(self):
        pass


@pytest.mark.parametrize("memory", [Managed, Unaligned])
@pytest.mark.parametrize("dim,precision", FORMS)
def test_other_memory_takes_the_copies(dim, precision, memory):
    h, st = new(dim, precision)
    d, _ = new(dim, precision)
    h.set_state(*st)
    bufs = [None if a is None else memory(np.size(a)) for a in st]
    for b, a in zip(bufs, st):
        if b is not None:
            b.fill(np.ascontiguousarray(a)) if memory is Unaligned else np.copyto(b.a, np.ravel(a))
    torch.cuda.synchronize()
    ptrs = [None if b is None else b.p for b in bufs]
    assert cgks.lib().cgks_set_state_device(d.h, *ptrs, None, None) == 0
    d.sync()
    assert_same(d.get_state(), h.get_state())
    h.step(1e-4)
    d.step(1e-4)
    h.sync()
    assert cgks.lib().cgks_get_state_device(d.h, *ptrs, None, None) == 0
    d.sync()
    torch.cuda.synchronize()
    want = h.get_state()
    for n, b in zip(NAMES, bufs):
        if b is not None:
            assert np.array_equal(b.a, np.ravel(want[n])), n
            b.close()


def test_range_beyond_its_allocation_is_not_taken_by_the_kernel():
    """Shown without running anything: the call is captured and the graph's nodes
    are counted.  W alone in an allocation of one double fewer than it needs."""
    L = cgks.lib()
    stream = torch.cuda.Stream()

    def kernels(short):
        s, st = new(2, cgks.FP32_BULK, stream=stream.cuda_stream)
        t = [cuda(a) for a in st]
        sig = [torch.zeros(7 * 14, dtype=torch.float64, device="cuda"), torch.zeros(8 * 13, dtype=torch.float64, device="cuda")]
        whole = ctypes.c_void_p()
        assert L.cudaMalloc(ctypes.byref(whole), ctypes.c_size_t(8 * t[0].numel())) == 0
        p = [ctypes.c_void_p(x.data_ptr()) for x in t + sig]
        p[0] = ctypes.c_void_p(whole.value + (8 if short else 0))
        torch.cuda.synchronize()
        assert L.cudaStreamBeginCapture(ctypes.c_void_p(stream.cuda_stream), 2) == 0
        code = L.cgks_set_state_device(s.h, *p)
        graph = ctypes.c_void_p()
        end = L.cudaStreamEndCapture(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(graph))
        count = None
        if end == 0 and code == 0:
            n = ctypes.c_size_t()
            assert L.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
            nodes = (ctypes.c_void_p * n.value)()
            assert L.cudaGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
            kind = ctypes.c_int()
            kinds = []
            for x in nodes:
                assert L.cudaGraphNodeGetType(ctypes.c_void_p(x), ctypes.byref(kind)) == 0
                kinds.append(kind.value)
            count = kinds.count(1)  # memory copies (0: kernels)
        if graph.value:
            L.cudaGraphDestroy(graph)
        L.cudaGetLastError()
        s.close()
        assert L.cudaFree(whole) == 0
        return code, count

    code, direct = kernels(False)
    assert code == 0
    code, copies = kernels(True)
    # five state arrays by copies, unless the copy of W was refused outright
    assert code != 0 or copies == direct + 5


@pytest.mark.parametrize("mode,other_thread", [("relaxed", False), ("thread_local", True)])
def test_first_compute_dt_beside_a_capture(mode, other_thread):
    """It allocates its host memory and waits for its own stream; the capture of
    another stream goes on, where its mode lets this thread make such calls."""
    a, st = new(2, cgks.FP32_BULK)
    b, _ = new(2, cgks.FP32_BULK)
    a.set_state(*st)
    b.set_state(*st)
    want = a.compute_dt()
    x = torch.ones(1000, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with ThreadPoolExecutor(1) as ex, torch.cuda.graph(g, capture_error_mode=mode):
        y = 2 * x
        dt = ex.submit(b.compute_dt).result() if other_thread else b.compute_dt()
        y = y + 1
    g.replay()
    torch.cuda.synchronize()
    assert dt == want
    assert float(y.sum()) == 3000.0
