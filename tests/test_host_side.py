"""The host side of libdgagg on a CUDA runtime without a GPU (fake_cudart.cpp): in what order it waits, frees and
launches, on which device, and what is left behind when an allocation or a launch fails."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2104_06700_b200 import binding, build

HERE = os.path.dirname(os.path.abspath(__file__))


class Fake:
    """libdgagg linked with the fake runtime."""

    def __init__(self, path):
        self.lib = ctypes.CDLL(path)
        self.lib.fake_event.restype = ctypes.c_char_p
        self.lib.dg_last_error.restype = ctypes.c_char_p
        self.lib.fake_alloc_limit.argtypes = self.lib.fake_reserved.argtypes = [ctypes.c_size_t]
        self.lib.dg_graph_set_param.argtypes = [ctypes.c_void_p, ctypes.c_char_p, ctypes.c_int64]
        self.lib.dg_graph_get_param.argtypes = [ctypes.c_void_p, ctypes.c_char_p, ctypes.c_void_p]
        self.keep = []

    def reset(self):
        self.on_sync(None)
        self.lib.fake_alloc_limit(ctypes.c_size_t(-1).value)
        self.lib.fake_reserved(0)
        self.lib.fake_failing_kernel(b"")
        self.lib.fake_plan_totals(0, 0)
        self.lib.cudaSetDevice(0)

    def on_sync(self, f):
        """f() runs in the middle of every wait for the device: what another thread does meanwhile."""
        self.callback = ctypes.CFUNCTYPE(None)(f) if f else None
        self.lib.fake_on_sync(self.callback)

    def events(self):
        """(what, current device, pointer) since the last call."""
        got = []
        for i in range(self.lib.fake_events()):
            device, pointer, size = ctypes.c_int(), ctypes.c_void_p(), ctypes.c_size_t()
            what = self.lib.fake_event(i, ctypes.byref(device), ctypes.byref(pointer), ctypes.byref(size))
            got.append((what.decode(), device.value, pointer.value))
        self.lib.fake_clear()
        return got

    def call(self, name, *args):
        """A call with integers as int32, bytes as strings and None as NULL."""
        given = [ctypes.c_int32(a) if isinstance(a, int) else a for a in args]
        return getattr(self.lib, name)(*given, None)

    def transposed(self, n, nnz):
        g = self.graph(n, nnz)
        storage, scratch = ctypes.c_size_t(), ctypes.c_size_t()
        self.lib.dg_graph_transpose_workspace(g, ctypes.byref(storage), ctypes.byref(scratch))
        buffers = []
        for size in (storage.value, scratch.value):
            address = self.array(size + 256, dtype=np.uint8).value
            buffers += [ctypes.c_void_p((address + 255) // 256 * 256), ctypes.c_size_t(size)]
        assert self.lib.dg_graph_transpose(g, *buffers, None) == binding.DG_OK
        return g

    def array(self, *shape, dtype=np.float32):
        a = np.zeros(shape, dtype)
        self.keep.append(a)
        return ctypes.c_void_p(a.ctypes.data)

    def graph(self, n=64, nnz=256):
        h = ctypes.c_void_p()
        st = self.lib.dg_graph_create(ctypes.c_int64(n), ctypes.c_int64(nnz), self.array(n + 1, dtype=np.int64),
                                      self.array(nnz, dtype=np.int32), None, ctypes.byref(h))
        assert st == binding.DG_OK, self.lib.dg_last_error()
        return h


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    build.build()
    objects = [os.path.join(build.BUILD_DIR, s[:-3] + ".o") for s in build.SOURCES]
    if not all(os.path.exists(o) for o in objects):  # the library came without them
        build.build(force=True)
    path = str(tmp_path_factory.mktemp("fake") / "libdgagg_host.so")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-Wl,-Bsymbolic", "-I", cuda, "-o", path,
                    os.path.join(HERE, "fake_cudart.cpp"), *objects], check=True)
    return Fake(path)


@pytest.fixture
def fake(library):
    library.reset()
    library.events()
    yield library
    library.reset()


def test_a_handle_destroyed_during_the_wait_keeps_its_memory(fake):
    """While dg_graph_create waits for the device another thread queues work on its own handle and destroys it:
    that wait does not cover the work, so the memory is freed after a later wait."""
    old = fake.graph()
    events = fake.events()
    blocks = {p for what, _, p in events if what == "alloc"}
    word = [p for what, _, p in events if what == "copy"]
    waits = []

    def other_thread():
        if not waits:
            fake.lib.dg_graph_destroy(old)
        waits.append(1)

    fake.on_sync(other_thread)
    new = fake.graph()
    fake.on_sync(None)
    events = fake.events()
    assert waits and not blocks & {p for what, _, p in events if what == "free"}
    assert not set(word) & {p for what, _, p in events if what == "copy"}  # nor are its counters written again
    third = fake.graph()
    events = fake.events()
    order = [what for what, _, _ in events]
    freed = [i for i, (what, _, p) in enumerate(events) if what == "free" and p in blocks]
    assert len(freed) == len(blocks) and min(freed) > order.index("sync")
    for h in (new, third):
        fake.lib.dg_graph_destroy(h)


@pytest.mark.parametrize("n,nnz,what", [(64, 256, "the list stays short"), (700000, 45000000, "the list is full")])
def test_a_handle_is_destroyed_on_its_own_device(fake, n, nnz, what):
    """Whatever device is current when a handle goes, or has a knob set: waits and frees act on the handle's, and the
    current device is the caller's again afterwards."""
    handle = fake.graph(n, nnz)
    fake.lib.cudaSetDevice(1)
    assert fake.lib.dg_graph_set_param(handle, b"rows_per_block", 64) == binding.DG_OK
    fake.lib.fake_reserved(1 << 30)  # the pool has grown: the last handle gives memory back
    fake.lib.dg_graph_destroy(handle)
    device = ctypes.c_int()
    fake.lib.cudaGetDevice(ctypes.byref(device))
    assert device.value == 1
    events = [e for e in fake.events() if e[0] in ("sync", "free", "free host", "trim")]
    assert {"sync", "free", "trim"} <= {e[0] for e in events}
    # the events up to here are the creation's, on device 0 too
    assert {e[1] for e in events} == {0}


@pytest.mark.parametrize("failure", ["memory", "launch"])
def test_a_knob_that_cannot_be_set_leaves_the_handle_as_it_was(fake, failure):
    handle = fake.graph(2000, 1 << 20)
    blocks = {p for what, _, p in fake.events() if what == "alloc"}

    def knob(name):
        value = ctypes.c_int64()
        assert fake.lib.dg_graph_get_param(handle, name, ctypes.byref(value)) == binding.DG_OK
        return value.value

    before = knob(b"heavy_threshold"), knob(b"rows_per_block")
    if failure == "memory":
        fake.lib.fake_alloc_limit(1000)
    else:
        fake.lib.fake_failing_kernel(b"plan_kernel")
    assert fake.lib.dg_graph_set_param(handle, b"heavy_threshold", 4096) == binding.DG_ERR_CUDA
    assert fake.lib.dg_graph_set_param(handle, b"rows_per_block", 64) == binding.DG_ERR_CUDA
    assert before == (knob(b"heavy_threshold"), knob(b"rows_per_block"))
    fake.reset()
    other = fake.graph()  # waits for the device and frees what is not in use any more
    assert not blocks & {p for what, _, p in fake.events() if what == "free"}
    assert fake.lib.dg_graph_set_param(handle, b"rows_per_block", 64) == binding.DG_OK
    assert knob(b"rows_per_block") == 64
    for h in (handle, other):
        fake.lib.dg_graph_destroy(h)


def aggregation_calls(fake, n, nnz, F):
    """(name, call) of every call that gathers a matrix, on a graph of n vertices and nnz edges."""
    g = fake.transposed(n, nnz)
    X, Y, dV, arg = (fake.array(n, F) for _ in range(4))
    fE, dE = fake.array(nnz), fake.array(nnz)
    max_, sum_, copy, mul, div = (binding.DG_RED_MAX, binding.DG_RED_SUM, binding.DG_BIN_COPY_LHS, binding.DG_BIN_MUL,
                                  binding.DG_BIN_DIV)
    calls = [("fwd", lambda: fake.call("dg_aggregate_fwd", g, X, F, binding.DG_OP_SUM, Y)),
             ("bwd mean", lambda: fake.call("dg_aggregate_bwd", g, X, F, binding.DG_OP_MEAN, Y)),
             ("max", lambda: fake.call("dg_ap_fwd", g, X, None, 1, F, copy, max_, Y, arg)),
             ("dV of div", lambda: fake.call("dg_ap_bwd", g, X, Y, fE, 1, F, div, sum_, None, dV, None)),
             ("edge grad", lambda: fake.call("dg_aggregate_edge_grad", g, X, Y, F, binding.DG_OP_SUM, dE))]
    return g, calls


def test_a_padded_copy_that_does_not_launch_is_an_error(fake):
    g, calls = aggregation_calls(fake, 5000, 200000, 101)
    for name, call in calls:
        assert call() == binding.DG_OK, name
        fake.lib.fake_failing_kernel(b"pad_rows_kernel")
        assert call() == binding.DG_ERR_CUDA, name
        fake.lib.fake_failing_kernel(b"")
    fake.lib.dg_graph_destroy(g)


def test_misaligned_statistics_of_the_loss_are_refused(fake):
    """The kernels read and write them 8 bytes at a time."""
    g = fake.graph(8, 16)
    logits, grads, index, labels = fake.array(8, 4), fake.array(8, 4), fake.array(4, dtype=np.int64), fake.array(8, dtype=np.int64)
    stats, result = fake.array(12), fake.array(2)
    for shift, want in ((0, binding.DG_OK), (4, binding.DG_ERR_INVALID_ARG)):
        at = ctypes.c_void_p((stats.value + 7) // 8 * 8 + shift)
        assert fake.lib.dg_cross_entropy_fwd(g, logits, 4, index, ctypes.c_int64(4), labels, at, result, None) == want
        assert fake.lib.dg_cross_entropy_bwd(g, logits, 4, index, ctypes.c_int64(4), labels, at, result, result, grads,
                                             None) == want
    fake.lib.dg_graph_destroy(g)


@pytest.mark.parametrize("how", ["no memory", "scratch_mb"])
def test_calls_do_without_scratch(fake, how):
    """No call needs memory of its own: the parts of cut rows, padded copies, the mask of max / min, partial sums."""
    fake.lib.fake_plan_totals(3, 1)
    n, nnz, F = 5000, 200000, 101
    g, calls = aggregation_calls(fake, n, nnz, F)
    X, Y, dV, arg, fE = fake.array(n, F), fake.array(n, F), fake.array(n, F), fake.array(n, F), fake.array(nnz, F)
    index, labels, row = fake.array(n, dtype=np.int64), fake.array(n, dtype=np.int64), fake.array(2 * n + 2)
    row = ctypes.c_void_p((row.value + 7) // 8 * 8)
    calls += [
        ("mul", lambda: fake.call("dg_ap_fwd", g, X, fE, F, F, binding.DG_BIN_MUL, binding.DG_RED_SUM, Y, None)),
        ("dV of max", lambda: fake.call("dg_ap_bwd", g, X, Y, None, 1, F, binding.DG_BIN_COPY_LHS, binding.DG_RED_MAX, arg,
                                        dV, None))]
    cut = {name for name, _ in calls} - {"edge grad"}
    calls += [("layer", lambda: fake.call("dg_layer_bwd", g, X, Y, F, row, dV, Y)),
              ("loss", lambda: fake.lib.dg_cross_entropy_fwd(g, X, F, index, ctypes.c_int64(n), labels, row, Y, None))]
    fake.events()
    if how == "no memory":
        fake.lib.fake_alloc_limit(0)
    else:
        assert fake.lib.dg_graph_set_param(g, b"scratch_mb", 0) == binding.DG_OK
    for name, call in calls:
        assert call() == binding.DG_OK, (name, fake.lib.dg_last_error())
        done = [what for what, _, _ in fake.events()]
        assert "alloc" not in done and done, name
        assert any("pieces_kernel" in what for what in done) == (name in cut), name
    fake.lib.dg_graph_destroy(g)
