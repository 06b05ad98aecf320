"""The library's host code on the CPU: its own objects linked with a CUDA
runtime that has no device (``fake_cudart.cpp``), so that the order, streams,
buffers and failures of a call's device operations can be looked at.  Kernels
do not run; nothing here says anything about results."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HOOK = ctypes.CFUNCTYPE(None, ctypes.c_char_p, ctypes.c_void_p, ctypes.c_size_t)
STREAM = 0x5150


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2609_38599_gb300 import build as b
    srcs = [os.path.join(b.CSRC, f) for f in os.listdir(b.CSRC)] + [os.path.join(ROOT, "include", "jarq.h")]
    objs = [os.path.join(b.BUILD, f[:-3] + ".o") for f in os.listdir(b.CSRC) if f.endswith(".cu")]
    newest = max(os.path.getmtime(f) for f in srcs)
    if not all(os.path.exists(o) and os.path.getmtime(o) >= newest for o in objs):
        b.build()
    out = str(tmp_path_factory.mktemp("fake") / "libjarq_host.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(b.nvcc())), "include")
    subprocess.run(["g++", "-O1", "-fPIC", "-shared", "-std=c++17", "-Wl,-Bsymbolic", "-I" + cuda,
                    os.path.join(ROOT, "tests", "fake_cudart.cpp"), *objs, "-o", out, "-pthread"], check=True)
    lib = ctypes.CDLL(out)
    lib.fake_log.restype = ctypes.c_char_p
    lib.fake_live.restype = ctypes.c_size_t
    lib.fake_hook.argtypes = [HOOK]
    return lib


class Device:
    """Buffers, handles and the log of one test."""

    def __init__(self, lib):
        self.lib, self.hooks, self.bufs, self.handles = lib, [], [], []
        lib.fake_reset()

    def buf(self, nbytes):
        p = ctypes.c_void_p()
        assert self.lib.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(nbytes)) == 0
        self.bufs.append(p)
        return p

    def prepare(self, din, g, stream=STREAM):
        h = ctypes.c_void_p()
        rc = self.lib.jarq_prepare_hessian(self.buf(4 * din * din), din, g, ctypes.c_float(0), ctypes.byref(h),
                                           ctypes.c_void_p(stream))
        if rc == 0:
            self.handles.append(h)
        return rc, h

    def layer(self, din, dout, g):
        G = din // g
        return self.buf(4 * din * dout), self.buf(4 * dout * G), self.buf(din * dout), self.buf(4 * dout * G)

    def refine(self, h, lay, dout, bits=3, stream=STREAM):
        return self.lib.jarq_refine_layer(h, *lay, dout, bits, None, None, ctypes.c_void_p(stream))

    def refine_mu(self, h, lay, dout, K, XX, bits=3, stream=STREAM):
        return self.lib.jarq_refine_layer_mu(h, *lay, dout, bits, K, XX, ctypes.c_float(0.5), ctypes.c_float(0),
                                             None, None, ctypes.c_void_p(stream))

    def hook(self, fn):
        """`fn(what, pointer, bytes)` inside every operation from now on."""
        h = HOOK(lambda what, p, n: fn(what.decode(), p, n))
        self.hooks.append(h)
        self.lib.fake_hook(h)

    def log(self):
        """Operations so far: (what, stream, rest)."""
        return [tuple(x.split(" ", 2)) for x in self.lib.fake_log().decode().splitlines()]

    def close(self):
        self.lib.fake_reset()
        for h in self.handles:
            self.lib.jarq_hessian_destroy(h)
        for p in self.bufs:
            self.lib.cudaFree(p)


@pytest.fixture
def dev(lib):
    d = Device(lib)
    yield d
    d.close()


def _overlapped(dev, call):
    """Runs `call(stream)` and, while it waits for its stream, a second one;
    the addresses of the status words that the two clear."""
    cleared = {}
    state = {"inside": False}

    def note(what, p, n):
        who = "second" if state["inside"] else "first"
        if what == "memset" and n == 4:
            cleared[who] = p
        if what == "sync" and not state["inside"] and "second" not in cleared:
            state["inside"] = True
            assert call(STREAM + 1) == 0
            state["inside"] = False

    dev.hook(note)
    assert call(STREAM) == 0
    assert set(cleared) == {"first", "second"}
    return cleared


def test_overlapping_writeback_calls_have_a_status_word_each(dev):
    """The write-back kernels write only while their call's status word is
    clear: a call on another stream must not set or clear that word."""
    lib = dev.lib
    S, Q, Z, out = dev.buf(4 * 8 * 2), dev.buf(8 * 128), dev.buf(4 * 8 * 2), dev.buf(4 * 8 * 128)
    calls = {
        "canonicalize": lambda s: lib.jarq_canonicalize(S, Q, Z, 8, 128, 64, 3, ctypes.c_void_p(s)),
        "dequantize": lambda s: lib.jarq_dequantize(S, Q, Z, 8, 128, 64, 3, 1, out, ctypes.c_void_p(s)),
        "pack": lambda s: lib.jarq_pack_codes(Q, 8, 128, 3, out, ctypes.c_void_p(s)),
    }
    for name, call in calls.items():
        words = _overlapped(dev, call)
        assert words["first"] != words["second"], name


def test_overlapping_hessian_calls_have_a_status_word_each(dev):
    """A call that starts while another one runs must not clear the word in
    which that one's kernel reports a wait that gave up."""
    X, H = dev.buf(2 * 64 * 64), dev.buf(4 * 64 * 64)
    words = _overlapped(dev, lambda s: dev.lib.jarq_accumulate_hessian(X, 64, 64, ctypes.c_float(1), H,
                                                                       ctypes.c_void_p(s)))
    assert words["first"] != words["second"]


def _mu_handle(dev, din=192, dout=40, g=64):
    """A handle whose padding (din no multiple of 128) has to be zeroed, a
    layer, K and XX."""
    rc, h = dev.prepare(din, g)
    assert rc == 0
    return h, dev.layer(din, dout, g), dout, dev.buf(4 * din * din), dev.buf(4 * din * din)


def test_a_call_works_on_its_own_stream_only(dev):
    """Every call of a handle, from its first on: each copy, fill and launch on
    the caller's stream.  One on the default stream is not ordered with a
    non-blocking stream's."""
    h, lay, dout, K, XX = _mu_handle(dev)
    st, F = ctypes.c_void_p(STREAM), dev.buf(8 * dout)
    assert dev.refine(h, lay, dout) == 0 and dev.refine_mu(h, lay, dout, K, XX) == 0
    assert dev.lib.jarq_objective(h, *lay, dout, 3, F, st) == 0
    assert dev.lib.jarq_multicode_probe(h, *lay, dout, 3, 1, None, None, None, None, None, st) == 0
    for method in range(3):
        assert dev.lib.jarq_fit_scales(h, *lay, dout, 3, method, 2, F, F, st) == 0
    others = [op for op in dev.log() if op[0] != "attribute" and op[1] != str(STREAM)]
    assert not others


def test_a_corrected_target_call_after_a_failed_allocation(dev):
    """Each allocation of a handle's first corrected-target call fails once;
    the call says so, and the next one has all buffers and tensor maps."""
    lib, n = dev.lib, 1
    while True:
        h, lay, dout, K, XX = _mu_handle(dev)
        K1 = ctypes.c_void_p(dev.buf(4 * 192 * 192 + 16).value + 4)     # misaligned: staged
        lib.fake_fail_malloc(n)
        rc = dev.refine_mu(h, lay, dout, K1, XX)
        lib.fake_fail_malloc(0)
        if rc == 0:
            break
        assert rc == 6, n                           # out of memory
        lib.fake_watch(b"12slice_kernel", 1)        # the block exponents
        lib.fake_watch(b"tc_proj_kernel", 1)        # the base of the digits' tensor map
        start = len(dev.log())
        assert dev.refine_mu(h, lay, dout, K1, XX) == 0
        seen = [op[2].split("arg=")[1] for op in dev.log()[start:] if op[0] == "launch" and "arg=" in op[2]]
        assert len(seen) == 5 and "0" not in seen, (n, seen)       # two slicings, three projections
        n += 1
    assert n > 3


@pytest.mark.parametrize("call", ["prepare", "independent fit", "probe"])
def test_the_other_group_size_at_the_same_time(dev, call):
    """A kernel's limit of dynamic shared memory belongs to the process: a call
    with groups of 64 that runs while one with 128 is on its way must not lower
    it under a launch that needs more."""
    lib, dout, state = dev.lib, 40, {"busy": False}
    handle = {g: dev.prepare(256, g)[1] for g in (64, 128)}
    layer = {g: dev.layer(256, dout, g) for g in (64, 128)}

    def run(g, stream):
        st = ctypes.c_void_p(stream)
        if call == "prepare":
            return dev.prepare(256, g, stream)[0]
        if call == "probe":
            return lib.jarq_multicode_probe(handle[g], *layer[g], dout, 3, 1, None, None, None, None, None, st)
        return lib.jarq_fit_scales(handle[g], *layer[g], dout, 3, 1, 1, None, None, st)

    def note(what, p, n):
        if what == "attribute" and not state["busy"]:
            state["busy"] = True
            assert run(64, STREAM + 1) == 0
            state["busy"] = False

    assert run(128, STREAM) == 0        # limits that are set once are set
    dev.hook(note)
    assert run(128, STREAM) == 0


@pytest.mark.parametrize("kernel,part", [
    (b"target", "tc_target_kernel"), (b"gram", "tc_gram_kernel"), (b"proj", "tc_proj_kernel"),
    (b"ptilde", "tc_fold_kernel"), (b"hr_full", "tc_hr_kernel"), (b"syrk", "tc_syrk_kernel")])
def test_stalled_kernel_selftest_launches_the_kernel_named(dev, kernel, part):
    live = dev.lib.fake_live()
    assert dev.lib.jarq_selftest_stalled_kernel(kernel, ctypes.c_void_p(STREAM)) == 0
    launches = [op[2] for op in dev.log() if op[0] == "launch"]
    assert part in launches[-1] and dev.lib.fake_live() == live
    assert dev.lib.jarq_selftest_stalled_kernel(b"no such kernel", ctypes.c_void_p(STREAM)) == 1


@pytest.mark.parametrize("g", [64, 128])
def test_band_holds_what_the_sweep_reads(dev, g):
    """The blocks of Ht beside the diagonal that a group's changes act on: the
    other groups of a block of 256 columns, no more."""
    rc, _ = dev.prepare(512, g)
    assert rc == 0
    grid = [op[2].split("grid=")[1] for op in dev.log() if op[0] == "launch" and "band_kernel" in op[2]]
    assert grid == [f"{(g // 32) ** 2},{512 // g},{256 // g - 1}"]


def test_profile_names_of_a_refinement(dev):
    """The sweep's kernels are recorded once per block of 256 columns, and read
    under the names that they had when a launch covered one group as well."""
    lib, n, ms = dev.lib, ctypes.c_longlong(), ctypes.c_double()
    _, h = dev.prepare(640, 128)
    lay = dev.layer(640, 40, 128)

    def read(name):
        assert lib.jarq_profile_read(name, ctypes.byref(n), ctypes.byref(ms)) == 0, name
        return n.value

    lib.jarq_profile_reset()
    lib.jarq_profile_enable(1)
    assert dev.refine(h, lay, 40) == 0                  # three iterations
    assert lib.jarq_multicode_probe(h, *lay, 40, 3, 1, None, None, None, None, None, ctypes.c_void_p(STREAM)) == 0
    lib.jarq_profile_enable(0)
    assert [read(k) for k in (b"sweep_product", b"target")] == [3 * 3 + 1] * 2      # and the probe's
    assert [read(k) for k in (b"sweep_babai", b"babai")] == [3 * 3] * 2
    assert read(b"gram") == 3 and read(b"phase_hr") == 0
    assert lib.jarq_profile_read(b"no such kernel", ctypes.byref(n), ctypes.byref(ms)) == -1


def test_launch_count_of_overlapping_calls(dev):
    """Calls that may overlap on several host threads all count."""
    import threading
    lib = dev.lib
    lib.jarq_launch_count.restype = ctypes.c_longlong
    bufs = [(dev.buf(128), dev.buf(128)) for _ in range(8)]
    n0, calls = lib.jarq_launch_count(), 6000
    call = ctypes.CDLL(lib._name).jarq_pack_codes

    def run(q, out):
        for _ in range(calls):
            call(q, 1, 128, 3, out, None)

    threads = [threading.Thread(target=run, args=b) for b in bufs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert lib.jarq_launch_count() - n0 == 2 * calls * len(bufs)
