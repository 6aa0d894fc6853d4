"""What still reads a spectrum holds its memory: releases with work in
flight, on other streams than the one that builds the next spectrum.  The
results compared are the same kernels' on the same values, so they are equal
bit for bit."""

import ctypes
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1907_02891_gb300 import lp  # noqa: E402

DEV = "cuda:0"
SIDE = 2250                      # of the spectra under test: 20 MB complex


@pytest.fixture()
def ctx():
    c = lp.lp_create(0)
    yield c
    lp.lp_destroy(c)


def _psf(seed, side=31):
    """Not point-symmetric: a complex spectrum."""
    return torch.from_numpy(np.random.default_rng(seed).uniform(0.1, 1.0, (side, side))).to(DEV)


def _copy_buffer():
    return torch.full((SIDE // 2 + 1, SIDE, 2), float("nan"), device=DEV)


class _Busy:
    """Keeps a stream busy for tens of milliseconds: maps of a spectrum of its own."""

    def __init__(self, ctx, stream):
        self.ctx, self.stream = ctx, stream
        self.spec = lp.lp_kernel_spectrum(ctx, _psf(100), pad_ny=8192, pad_nx=8192)
        self.L = torch.ones(8000, 8000, device=DEV)
        self.out = torch.empty_like(self.L)
        lp.lp_sync_status(ctx)
        lp.lp_map(ctx, self.L, [self.spec], [self.out], stream=stream)   # the stream's workspace
        lp.lp_sync_status(ctx, stream=stream)

    def start(self):
        for _ in range(100):
            lp.lp_map(self.ctx, self.L, [self.spec], [self.out], stream=self.stream)

    def running(self):
        return lp.lp_sync_status_code(self.ctx, stream=self.stream, timeout_ms=0) == lp.LP_ERR_TIMEOUT


@pytest.mark.parametrize("symmetric,prec", [(False, lp.LP_PREC_FP32), (True, lp.LP_PREC_FP32),
                                            (False, lp.LP_PREC_SPLIT_BF16)])
def test_release_with_a_copy_in_flight(ctx, symmetric, prec):
    """A copy queued behind other work, the spectrum released, and another
    PSF's spectrum of the same size built on another stream: the memory is
    still held, and the copy has the first spectrum's values."""
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    busy = _Busy(ctx, a)
    side = next(n for n in lp.supported_sizes() if n >= SIDE and (prec == lp.LP_PREC_FP32 or lp.lp_split_supported(n)))

    def build(seed, stream=None):
        K = _psf(seed)
        if symmetric:
            K = K + K.flip(0, 1)
        torch.cuda.synchronize()
        return lp.lp_kernel_spectrum(ctx, K, pad_ny=side, pad_nx=side, prec=prec, stream=stream)

    spec = build(1)
    want, got = (torch.full((side // 2 + 1, side, 1 if symmetric else 2), float("nan"), device=DEV) for _ in range(2))
    lp.lp_spectrum_copy(spec, want)
    lp.lp_sync_status(ctx)
    K2 = _psf(2)
    if symmetric:
        K2 = K2 + K2.flip(0, 1)
    torch.cuda.synchronize()
    held = lp.lp_bytes_in_use(ctx)
    busy.start()
    lp.lp_spectrum_copy(spec, got, stream=a)
    lp.lp_spectrum_release(ctx, spec)
    after_release = lp.lp_bytes_in_use(ctx)
    other = lp.lp_kernel_spectrum(ctx, K2, pad_ny=side, pad_nx=side, prec=prec, stream=b)
    after_build = lp.lp_bytes_in_use(ctx)
    assert busy.running(), "the stream drained before the release could be told from a wait"
    lp.lp_sync_status(ctx, stream=b)
    lp.lp_sync_status(ctx, stream=a)
    assert after_release == held
    assert after_build > held
    assert torch.equal(got, want)
    lp.lp_sync_status(ctx)
    assert lp.lp_bytes_in_use(ctx) == held       # the first went, the second of its size came
    lp.lp_spectrum_release(ctx, other)


def test_copy_waits_for_a_build_on_another_stream(ctx):
    s_build, s_copy = torch.cuda.Stream(), torch.cuda.Stream()
    got, want = (torch.full((8820 // 2 + 1, 8820, 2), float("nan"), device=DEV) for _ in range(2))
    K = _psf(3, 601)
    torch.cuda.synchronize()
    spec = lp.lp_kernel_spectrum(ctx, K, pad_ny=8820, pad_nx=8820, stream=s_build)
    lp.lp_spectrum_copy(spec, got, stream=s_copy)
    torch.cuda.synchronize()
    lp.lp_spectrum_copy(spec, want)
    lp.lp_sync_status(ctx)
    assert torch.equal(got, want)
    lp.lp_spectrum_release(ctx, spec)


class _Capture:
    """Capture of a stream into a graph of its own, by the driver's calls
    (torch's synchronises the device first)."""

    def __init__(self, stream):
        self.cuda, self.stream = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(stream.cuda_stream)

    def __enter__(self):
        assert self.cuda.cuStreamBeginCapture_v2(self.stream, 2) == 0       # relaxed
        return self

    def __exit__(self, *exc):
        self.graph = ctypes.c_void_p()
        assert self.cuda.cuStreamEndCapture(self.stream, ctypes.byref(self.graph)) == 0

    def node_types(self):
        n = ctypes.c_size_t()
        assert self.cuda.cuGraphGetNodes(self.graph, None, ctypes.byref(n)) == 0
        nodes, kind, kinds = (ctypes.c_void_p * n.value)(), ctypes.c_int(), []
        assert self.cuda.cuGraphGetNodes(self.graph, nodes, ctypes.byref(n)) == 0
        for node in nodes:
            assert self.cuda.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
            kinds.append(kind.value)
        return kinds

    def destroy(self):
        assert self.cuda.cuGraphDestroy(self.graph) == 0


@pytest.mark.parametrize("entry", ["map", "multiclass", "copy"])
def test_capture_leaves_earlier_uses_alone(ctx, entry):
    """A call captured on a stream does not hide the stream's queued work with
    the same spectrum from the release."""
    a = torch.cuda.Stream()
    busy = _Busy(ctx, a)
    spec = lp.lp_kernel_spectrum(ctx, _psf(6), pad_ny=SIDE, pad_nx=SIDE)
    L = torch.ones(2200, 2200, device=DEV)
    out = torch.empty_like(L)
    want, got = _copy_buffer(), _copy_buffer()
    lp.lp_spectrum_copy(spec, want)
    lp.lp_map_multiclass(ctx, [L], [spec], out, stream=a)       # workspace
    torch.cuda.synchronize()
    held = lp.lp_bytes_in_use(ctx)
    busy.start()
    lp.lp_spectrum_copy(spec, got, stream=a)
    with _Capture(a) as c:
        if entry == "map":
            lp.lp_map(ctx, L, [spec], [out], stream=a)
        elif entry == "multiclass":
            lp.lp_map_multiclass(ctx, [L], [spec], out, stream=a)
        else:
            lp.lp_spectrum_copy(spec, got, stream=a)
    assert 0 in c.node_types()                                  # kernels
    c.destroy()
    lp.lp_spectrum_release(ctx, spec)
    after_release = lp.lp_bytes_in_use(ctx)
    assert busy.running()
    lp.lp_sync_status(ctx, stream=a)
    assert after_release == held
    assert lp.lp_bytes_in_use(ctx) < held
    assert torch.equal(got, want)


def test_uses_go_by_stream_not_by_handle(ctx):
    """cudaStreamPerThread (handle 2) is another stream in every thread: a
    finished use in one thread says nothing about another's."""
    worker = ThreadPoolExecutor(1)              # one thread, its per-thread stream

    def there(f, *a, **k):
        return worker.submit(f, *a, **k).result()

    busy = there(_Busy, ctx, 2)
    spec = lp.lp_kernel_spectrum(ctx, _psf(4), pad_ny=SIDE, pad_nx=SIDE)
    want, got, here = (_copy_buffer() for _ in range(3))
    lp.lp_spectrum_copy(spec, want)
    lp.lp_sync_status(ctx)
    held = lp.lp_bytes_in_use(ctx)
    there(busy.start)
    there(lp.lp_spectrum_copy, spec, got, stream=2)
    lp.lp_spectrum_copy(spec, here, stream=2)
    torch.cuda.ExternalStream(2).synchronize()  # this thread's
    lp.lp_spectrum_release(ctx, spec)
    after_release = lp.lp_bytes_in_use(ctx)
    assert there(busy.running)
    there(lp.lp_sync_status, ctx, stream=2)
    assert after_release == held
    assert lp.lp_bytes_in_use(ctx) < held
    assert torch.equal(got, want) and torch.equal(here, want)
    worker.shutdown()


def test_release_after_uses_on_many_streams(ctx):
    """More streams than a spectrum keeps use events for, one after the other."""
    spec = lp.lp_kernel_spectrum(ctx, _psf(5), pad_ny=SIDE, pad_nx=SIDE)
    dst = _copy_buffer()
    torch.cuda.synchronize()
    held = lp.lp_bytes_in_use(ctx)
    for _ in range(12):
        s = torch.cuda.Stream()
        lp.lp_spectrum_copy(spec, dst, stream=s)
        s.synchronize()
    lp.lp_spectrum_release(ctx, spec)
    assert lp.lp_bytes_in_use(ctx) < held


@pytest.mark.parametrize("entry", ["map", "tiled", "multiclass", "host", "serve"])
def test_a_call_that_fails_half_way_holds_its_spectra(ctx, entry):
    """The column pass is enqueued (behind other work, where the call runs on
    the caller's stream) when the call fails: its spectrum stays until that
    pass is done, and not longer."""
    a = torch.cuda.Stream()
    busy = _Busy(ctx, a)
    spec = lp.lp_kernel_spectrum(ctx, _psf(7), pad_ny=SIDE, pad_nx=SIDE)
    L = torch.ones(2200, 2200, device=DEV)
    out = torch.empty_like(L)
    hL, hout = (torch.ones(2200, 2200).pin_memory() for _ in range(2))
    if entry == "serve":
        lp.lp_serve_start(ctx, 1)

    def call():
        if entry == "map":
            lp.lp_map(ctx, L, [spec], [out], stream=a)
        elif entry == "tiled":
            lp.lp_map_tiled(ctx, L, [spec], [out], stream=a)
        elif entry == "multiclass":
            lp.lp_map_multiclass(ctx, [L], [spec], out, stream=a)
        elif entry == "host":
            lp.lp_map_host(ctx, hL, [spec], [hout], stream=a)
        else:
            lp.lp_serve_poll(ctx, lp.lp_serve_submit(ctx, L, [spec], [out]), timeout_ms=60000)

    call()                                                      # workspaces
    torch.cuda.synchronize()
    held = lp.lp_bytes_in_use(ctx)
    if entry in ("map", "tiled", "multiclass"):                 # (the others run on streams of their own)
        busy.start()
    lp.lp_set_test_hook(ctx, lp.LP_TEST_ROWS_FAIL)
    with pytest.raises(lp.LpError) as e:
        call()
    assert e.value.status == lp.LP_ERR_CUDA
    lp.lp_spectrum_release(ctx, spec)
    if entry in ("map", "tiled", "multiclass"):
        after_release = lp.lp_bytes_in_use(ctx)
        assert busy.running()
        assert after_release == held
    torch.cuda.synchronize()
    lp.lp_sync_status(ctx)
    assert lp.lp_bytes_in_use(ctx) < held
    if entry == "serve":
        lp.lp_serve_stop(ctx)


@pytest.mark.parametrize("by", ["workspace", "build"])
def test_failed_allocation_gives_kept_memory_back(ctx, by):
    """An allocation that fails (on the host, by LP_TEST_OOM) right after a
    spectrum has been released gets its memory: most of the 155 MB that the
    context would have kept for the next build are the device's again (all but
    the pool's blocks that hold a live spectrum beside it)."""
    small = lp.lp_kernel_spectrum(ctx, _psf(8), pad_ny=128, pad_nx=128)
    K = _psf(9)
    K = K + K.flip(0, 1)
    L, out = torch.ones(90, 90, device=DEV), torch.empty(90, 90, device=DEV)
    big = lp.lp_kernel_spectrum(ctx, K, pad_ny=8820, pad_nx=8820)
    torch.cuda.synchronize()
    size = 4 * 4411 * 8820
    free = torch.cuda.mem_get_info()[0]
    lp.lp_spectrum_release(ctx, big)
    lp.lp_set_test_hook(ctx, lp.LP_TEST_OOM)
    if by == "workspace":
        lp.lp_map(ctx, L, [small], [out])
    else:
        K2 = _psf(10)
        lp.lp_kernel_spectrum(ctx, K2, pad_ny=128, pad_nx=128)
    assert torch.cuda.mem_get_info()[0] >= free + size // 2
    torch.cuda.synchronize()
    lp.lp_sync_status(ctx)


@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("where", ["pinned", "pinned+4", "device+4"])
def test_copy_writes_any_addressable_destination_itself(ctx, symmetric, where):
    """Pinned host memory and 4-byte aligned addresses: the same values as an
    aligned device destination, nothing beside them, and a captured copy is
    kernels alone (a buffer in between would be an allocation in the graph)."""
    K = _psf(11)
    if symmetric:
        K = K + K.flip(0, 1)
    spec = lp.lp_kernel_spectrum(ctx, K, pad_ny=210, pad_nx=96)
    n = 49 * 210 * (1 if symmetric else 2)
    want = torch.empty(n, device=DEV)
    lp.lp_spectrum_copy(spec, want)
    lp.lp_sync_status(ctx)
    buf = torch.full((n + 4,), -7.0)
    buf = buf.pin_memory() if where.startswith("pinned") else buf.to(DEV)
    off = 1 if where.endswith("+4") else 0
    torch.cuda.synchronize()
    a = torch.cuda.Stream()
    with _Capture(a) as c:
        lp.lp_spectrum_copy(spec, buf[off:off + n], stream=a)
    kinds = c.node_types()
    c.destroy()
    assert kinds and set(kinds) == {0}
    assert (buf == -7).all()
    lp.lp_spectrum_copy(spec, buf[off:off + n], stream=a)
    lp.lp_sync_status(ctx, stream=a)
    assert torch.equal(buf[off:off + n].to(DEV), want)
    assert (buf[:off] == -7).all() and (buf[off + n:] == -7).all()
