"""The host side of the step's two entry points without a device: api.cu compiled for the CPU against stand-ins for the CUDA
runtime and the launchers (`host_fake.cpp`) that log every call and can fail on demand."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

from paper_2408_15562_b200 import binding

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2408_15562_b200", "csrc")
STREAM = 0x77


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("host_side") / "libhostside.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic",
                           "-DatomicCAS(p,a,b)=((void)(p),(void)(a),(void)(b))",
                           "-I" + os.path.join(ROOT, "include"), "-I" + CSRC, "-I/usr/local/cuda/include",
                           "-x", "c++", os.path.join(CSRC, "api.cu"), os.path.join(HERE, "host_fake.cpp"), "-o", out])
    lib = ctypes.CDLL(out)
    vp, ci = ctypes.c_void_p, ctypes.c_int
    lib.fspad_create.argtypes = [ctypes.POINTER(binding.FspadConfig), ctypes.POINTER(vp)]
    lib.fspad_destroy.argtypes = [vp]
    lib.fspad_destroy.restype = None
    lib.fspad_verify_step.argtypes = [vp, vp, ci] + [vp] * 10 + [ci, ci] + [vp] * 6
    lib.fspad_verify_step_host.argtypes = [vp] * 12 + [ci, ci] + [vp] * 6
    lib.fspad_tree_accept.argtypes = [vp] * 7 + [ci, ci] + [vp] * 4
    lib.fake_log.restype = ctypes.c_char_p
    lib.fake_fail.argtypes = [ctypes.c_char_p, ci]
    lib.fake_pin.argtypes = [vp, ctypes.c_size_t]
    lib.fake_device.argtypes = [vp]
    return lib


class Step:
    """One context and one set of (never read) buffers for both entry points."""

    def __init__(self, lib, hq=32, hkv=8, nodes=60, batch=1, vocab=4096, max_len=2176, sampling=True, layers=1):
        self.lib, self.n, self.batch, self.vocab, self.sampling = lib, nodes, batch, vocab, sampling
        cfg = binding.FspadConfig(hq, hkv, 128, nodes, vocab, layers, max_len, batch, 0.0)
        self.ctx = ctypes.c_void_p()
        assert lib.fspad_create(ctypes.byref(cfg), ctypes.byref(self.ctx)) == 0
        raw = np.zeros(batch * nodes * vocab + 8, np.float32)
        skip = (-raw.ctypes.data // 4) % 4
        self.draft = raw[skip:skip + batch * nodes * vocab]              # 16-byte aligned
        self.small = np.zeros(batch * (max(nodes, 64) + 1) + 8, np.int32)
        self.parent = np.zeros((batch, nodes), np.int32)                 # stars; the one array that the host entry looks at
        lib.fake_reset()

    def __del__(self):
        self.lib.fspad_destroy(self.ctx)

    def host(self, parent=None):
        big = 0x1000                                     # never dereferenced by the stand-ins
        p, parent = self.small.ctypes.data, parent or self.parent.ctypes.data
        draft, unif = (self.draft.ctypes.data, p) if self.sampling else (None, None)
        rc = self.lib.fspad_verify_step_host(self.ctx, big, big, big, big, parent, big, big, draft, big, big, unif, self.n, self.batch,
                                             big, p, p, p, p, STREAM)
        return rc, self.lib.fake_log().decode().splitlines()

    def device(self, tree=None):
        big = 0x1000
        draft, unif = (big, big) if self.sampling else (None, None)
        rc = self.lib.fspad_verify_step(self.ctx, big, 0, big, tree, tree, big, big, big, draft, big, big, unif, self.n, self.batch, big,
                                        big, big, big, big, STREAM)
        return rc, self.lib.fake_log().decode().splitlines()


    def accept(self):
        big = 0x1000
        draft, unif = (big, big) if self.sampling else (None, None)
        rc = self.lib.fspad_tree_accept(self.ctx, big, draft, big, big, big, unif, self.n, self.batch, big, big, big, STREAM)
        return rc, self.lib.fake_log().decode().splitlines()


def _field(log, name, key):
    line = next(x for x in log if x.startswith(name + " "))
    return re.search(key + r"=(\S+)", line).group(1)


@pytest.mark.parametrize("sampling", [True, False])
@pytest.mark.parametrize("hq,hkv,nodes,batch,max_len", [(32, 8, 60, 1, 2176), (52, 52, 60, 1, 4224), (64, 8, 60, 1, 8320),
                                                        (32, 32, 26, 1, 320), (32, 8, 24, 3, 384), (28, 4, 8, 2, 512)])
def test_host_entry_cuts_the_attention_as_the_device_entry_does(lib, hq, hkv, nodes, batch, max_len, sampling):
    """The number of key ranges decides which probabilities are rounded against which reference: the two entry points give the
    same bits only if they let the attention fill the same number of SMs."""
    step = Step(lib, hq, hkv, nodes, batch, max_len=max_len, sampling=sampling)
    rc, log = step.device()
    want = _field(log, "attention", "sms")
    lib.fake_reset()
    rc_h, log_h = step.host()
    assert rc == 0 and rc_h == 0
    assert _field(log_h, "attention", "sms") == want


@pytest.mark.parametrize("sampling,vocab,hkv,layers,max_len,by_walk", [
    (True, 32000, 32, 1, 320, True), (True, 32000, 32, 4, 320, True), (True, 32000, 43, 3, 320, False),       # one stream: 64, 256, 258 slices
    (True, 4000, 32, 1, 320, True), (True, 4000, 33, 1, 320, False),         # a single CTA walks: 64, 66
    (True, 8192, 32, 2, 320, True), (True, 8192, 33, 2, 320, False),         # a cluster of four: 128, 132
    (True, 128256, 8, 4, 2176, True), (True, 128256, 8, 5, 2176, False),     # one stream, the attention a short one: 64, 80
    (False, 4000, 32, 1, 320, True), (False, 4000, 33, 1, 320, False),       # greedy, one stream
])
def test_who_compacts(lib, sampling, vocab, hkv, layers, max_len, by_walk):
    """The walk moves the cache rows where a warp of its CTAs gets two slices at most (64 slices in any case), else the kernel does."""
    step = Step(lib, 4 * hkv if hkv == 8 else hkv, hkv, 60 if hkv == 8 else 8, 1, vocab, max_len, sampling, layers)
    rc, log = step.device(0x1000)
    assert rc == 0 and _field(log, "walk", "compacts") == str(int(by_walk))
    assert any(x.startswith("compact ") for x in log) != by_walk


@pytest.mark.parametrize("sampling,hq,hkv,nodes,batch,max_len,called,captured", [
    (True, 32, 8, 60, 1, 2176, "fork", "fork"),          # several ranges of three chunks
    (True, 52, 52, 60, 1, 4224, "one", "fork"),          # two ranges of 17 chunks
    (True, 32, 8, 60, 1, 16384, "one", "fork"),          # eight ranges of 16
    (True, 32, 32, 60, 4, 320, "one", "one"),            # 128 CTAs, more than the walk leaves room for
    (True, 32, 32, 60, 16, 4224, "fork", "fork"),        # walks on more than half of the SMs
    (False, 32, 32, 26, 1, 320, "one", "fork"),          # short greedy step
    (False, 32, 32, 26, 1, 1024, "one", "fork"),         # the same with two ranges
    (False, 32, 32, 26, 1, 8320, "fork", "fork"),        # long greedy step
])
def test_capture_decides_on_the_order_and_not_on_the_cut(lib, sampling, hq, hkv, nodes, batch, max_len, called, captured):
    """One stream: scan, walk, attention beside the walk, no event.  Fork: the attention on the second stream between two events.
    The SMs the attention is cut for, and with them the results' bits, are the same either way."""
    sms = set()
    for on, want in ((0, called), (1, captured)):
        step = Step(lib, hq, hkv, nodes, batch, 32768 if sampling else 4096, max_len, sampling)
        lib.fake_capture(on)
        try:
            rc, log = step.device()
        finally:
            lib.fake_capture(0)
        assert rc == 0
        sms.add(_field(log, "attention", "sms"))
        events = [x for x in log if x.startswith("event_record ") or x.startswith("stream_wait ")]
        if want == "one":
            assert not events and _field(log, "attention", "early") == "1" and _field(log, "attention", "stream") == "%x" % STREAM
            assert [x.split()[0] for x in log][:3] == ["scan", "walk", "attention"]
        else:
            assert len(events) == 4 and _field(log, "attention", "early") == "0" and _field(log, "attention", "stream") != "%x" % STREAM
    assert len(sms) == 1


@pytest.mark.parametrize("hq,hkv,nodes,batch,max_len,vocab,called,captured", [
    (32, 8, 60, 1, 2176, 128256, "one", "scan first"),       # 16 CTAs to a range, nine ranges: 144 of 148 SMs
    (64, 8, 24, 1, 2176, 128256, "one", "scan first"),       # few rows of a large vocabulary
    (32, 8, 40, 2, 2176, 50257, "one", "scan first"),
    (52, 52, 60, 1, 1100, 50257, "one", "one"),              # 104 SMs, the scan does not go first
    (32, 8, 60, 1, 2176, 32768, "fork", "fork"),             # below the line
    (32, 8, 24, 9, 1024, 128256, "fork", "fork"),            # walks (clusters of ten) on more than half of the SMs
    (32, 8, 12, 5, 2176, 50257, "fork", "fork"),             # small trees: below their line
])
def test_order_behind_larger_scans(lib, hq, hkv, nodes, batch, max_len, vocab, called, captured):
    """A sampled step with a short attention: one stream from a number of logits on, captured only where the scan would not go first
    of two streams; the scan goes by the trees or not by a line of its own.  The attention's cut is the same either way."""
    sms = set()
    for on, want in ((0, called), (1, captured)):
        step = Step(lib, hq, hkv, nodes, batch, vocab, max_len, True)
        lib.fake_capture(on)
        try:
            rc, log = step.device(0x1000)
        finally:
            lib.fake_capture(0)
        assert rc == 0
        sms.add(_field(log, "attention", "sms"))
        order = [x.split()[0] for x in log]
        events = [x for x in order if x in ("event_record", "stream_wait")]
        if want == "one":
            assert not events and order[:3] == ["scan", "walk", "attention"] and _field(log, "attention", "early") == "1"
        else:
            assert len(events) == 4 and _field(log, "attention", "early") == "0"
            if want == "scan first":
                assert order[:3] == ["scan", "event_record", "stream_wait"] and order[3] == "walk"
    assert len(sms) == 1


@pytest.mark.parametrize("pins,in_place", [(((0, 1.0),), True), ((), False), (((0, 0.5),), False), (((0, 0.999),), False),
                                           (((0.5, 0.5),), False), (((0, 0.25), (0.75, 0.25)), False), (((0, 0.5), (0.5, 0.5)), False)])
def test_draft_rows_are_read_in_place_only_where_all_of_them_are_pinned(lib, pins, in_place):
    """(first byte, length) of the registered parts, as shares of the draft rows."""
    step = Step(lib)
    n = step.draft.nbytes
    for at, share in pins:
        lib.fake_pin(step.draft.ctypes.data + int(at * n), int(share * n))
    rc, log = step.host()
    assert rc == 0
    copied = any(x.startswith("h2d host=%x " % step.draft.ctypes.data) for x in log)
    assert copied != in_place and _field(log, "walk", "far") == str(int(in_place))
    if in_place:
        assert int(_field(log, "walk", "draft"), 16) == step.draft.ctypes.data


@pytest.mark.parametrize("share,nodes,batch,vocab,in_place", [(1.0, 60, 1, 4096, True), (1.0, 200, 2, 33, True), (0.99, 60, 1, 4096, False), (0, 60, 1, 4096, False),
                                                              (1.0, 256, 33, 8, False)])        # 8448 rows: more than the scan by the trees takes
def test_logits_stay_where_all_of_them_are_pinned(lib, share, nodes, batch, vocab, in_place):
    step = Step(lib, nodes=nodes, batch=batch, vocab=vocab, sampling=False)
    bytes_ = batch * nodes * vocab * 4
    if share:
        lib.fake_pin(0x1000, int(share * bytes_))
    rc, log = step.host()
    copied = any(x.startswith("h2d host=1000 bytes=%d " % bytes_) for x in log)
    assert rc == 0 and copied != in_place and any(x.startswith("scan ") for x in log)


@pytest.mark.parametrize("nodes,batch,vocab,chains,in_place", [
    (60, 1, 128256, 0, True), (60, 1, 128256, 1, False), (60, 2, 32000, 2, False), (60, 2, 32000, 1, True), (8, 1, 128256, 1, True),
    (8, 1, 8000, 1, True), (60, 1, 2000, 1, False), (256, 32, 333, 32, False), (1, 1, 32000, 1, True)])
def test_logits_of_chains_are_copied(lib, nodes, batch, vocab, chains, in_place):
    """Page-locked logits: read in place unless most rows would be, where a copy is the faster way.  Parents that no tree has count as
    the root, as they do on the device, and none is looked at outside of the array."""
    for bad in (False, True):
        step = Step(lib, nodes=nodes, batch=batch, vocab=vocab, sampling=False)
        step.parent[:chains] = np.arange(-1, nodes - 1)
        if bad:
            step.parent[step.parent == 0] = 1 << 30
            step.parent[:, 0] = 77
        bytes_ = batch * nodes * vocab * 4
        lib.fake_pin(0x1000, bytes_)
        rc, log = step.host()
        copied = any(x.startswith("h2d host=1000 bytes=%d " % bytes_) for x in log)
        assert rc == 0 and copied != in_place and _field(log, "scan", "staged") == str(int(in_place))


def test_a_device_array_for_the_trees_is_left_to_the_copy(lib):
    """The host entry looks at the trees only where the host can: a device array given for them is the copy's error, as it was."""
    step = Step(lib, nodes=60, vocab=128256, sampling=False)
    lib.fake_pin(0x1000, 60 * 128256 * 4)
    lib.fake_device(0x5000)
    lib.fake_fail(b"h2d", 2)                             # (what the runtime says to it)
    rc, log = step.host(parent=0x5000)
    assert rc == -6 and any(x.startswith("h2d host=5000 ") for x in log)


# just below and on the line from which the scan goes by the trees: alone, in a step
@pytest.mark.parametrize("sampling,nodes,batch,vocab,alone,step", [
    (True, 9, 1, 8192, False, False), (True, 9, 1, 8193, True, True), (False, 3, 3, 32000, True, True), (False, 5, 2, 32000, False, False),
    (True, 40, 2, 31000, False, False), (True, 40, 2, 32000, False, True), (True, 24, 6, 32000, True, True), (True, 24, 5, 32000, False, False),
    (True, 16, 8, 46000, False, True), (True, 16, 8, 47000, True, True), (True, 8, 20, 49000, False, False), (True, 8, 20, 50000, True, True),
    (True, 24, 1, 62000, False, False), (True, 24, 1, 64000, False, True), (True, 24, 1, 84000, False, True), (True, 32, 1, 128256, True, True),            # one wave of pieces
    (False, 40, 2, 31000, False, False), (False, 40, 2, 32000, False, True), (False, 40, 4, 32000, True, True),
    (False, 40, 2, 32001, False, False), (False, 40, 2, 50257, False, True), (False, 40, 4, 59001, False, True), (False, 40, 4, 60001, True, True),
    (False, 24, 7, 32000, False, False), (False, 24, 8, 32000, False, True), (False, 24, 8, 32001, False, False), (False, 24, 9, 45000, True, True),
    (False, 8, 16, 128256, False, True), (False, 8, 25, 128256, True, True), (False, 24, 1, 128256, False, False), (False, 32, 1, 128256, False, True)])
def test_when_the_scan_goes_by_the_trees(lib, sampling, nodes, batch, vocab, alone, step):
    step_ = Step(lib, nodes=nodes, batch=batch, vocab=vocab, sampling=sampling, max_len=2176)
    rc, log = step_.accept()
    assert rc == 0 and _field(log, "scan", "trees") == str(int(alone))
    lib.fake_reset()
    rc, log = step_.device(0x1000)
    assert rc == 0 and _field(log, "scan", "trees") == str(int(step)) and _field(log, "scan", "staged") == "0"
    lib.fake_reset()
    rc, log = step_.host()                       # pageable logits: as the step
    assert rc == 0 and _field(log, "scan", "trees") == str(int(step)) and _field(log, "scan", "staged") == "0"
    lib.fake_reset()
    lib.fake_pin(0x1000, batch * nodes * vocab * 4)
    rc, log = step_.host()                       # pinned ones: brought to the device by a scan by the trees
    assert rc == 0 and _field(log, "scan", "trees") == "1" and _field(log, "scan", "staged") == "1"


FAILING = [("h2d", k) for k in range(1, 10)] + [("d2h", k) for k in range(1, 7)] + \
    [(name, 1) for name in ("scatter", "attention", "scan", "walk", "compact", "sync")] + \
    [("event_record", k) for k in (1, 2)] + [("stream_wait", k) for k in (1, 2)]


@pytest.mark.parametrize("name,nth", FAILING)
def test_host_entry_returns_an_error_only_when_nothing_is_under_way(lib, name, nth):
    """Copies and the walk use the caller's memory: whatever call fails, both streams have been waited for after the last thing queued."""
    step = Step(lib)
    lib.fake_fail(name.encode(), nth)
    rc, log = step.host()
    assert rc == -6                                                  # FSPAD_ERR_CUDA
    side = next((re.search(r"stream=(\S+)", x).group(1) for x in log if x.startswith("attention ")), None)
    for stream in {"%x" % STREAM, side} - {None}:
        mine = [k for k, x in enumerate(log) if x.endswith("stream=" + stream) and not x.startswith("sync ")]
        waits = [k for k, x in enumerate(log) if x == "sync stream=" + stream]
        assert not mine or (waits and max(waits) > max(mine)), (stream, log)
