"""The host side of the library (csrc/mixaq.cu, csrc/merge_static.cu) against a stand-in for the CUDA runtime and the kernel launchers
(host_path/): which calls are recorded as graphs and replayed, and what happens when a call fails."""
import ctypes as C
import os
import subprocess
import threading

import numpy as np
import pytest

from paper_2507_19131_b200 import binding as mq
from paper_2507_19131_b200 import build as mq_build

HERE = os.path.dirname(os.path.abspath(__file__))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


class Counts(C.Structure):
    _fields_ = [(n, C.c_long) for n in ("captures", "instantiated", "live_graphs", "graph_launches", "direct", "captured",
                                        "side_launches", "copies", "guard_launches", "violations")]


class SelectArgs(C.Structure):
    _fields_ = [(n, C.c_void_p) for n in ("energy", "score", "order", "cls", "rowsrc_hi", "rowsrc_lo", "rowsrc_pr", "win_hi", "win_lo")] + \
               [(n, C.c_int) for n in ("B", "H", "W", "shift", "nwx", "nW", "n_hi", "n_lo", "n_pr", "reverse")] + [("narrow", C.c_bool)]


class Range(C.Structure):
    _fields_ = [("at", C.c_void_p), ("bytes", C.c_size_t), ("code_bits", C.c_int)]


class Copy(C.Structure):
    _fields_ = [("dst", C.c_void_p), ("src", C.c_void_p), ("bytes", C.c_size_t)]


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")
    out = str(tmp_path_factory.mktemp("host_path") / "libhost.so")
    flags = [f for f in mq_build.NVCC_FLAGS if f not in ("-O3", "-lineinfo")]
    fake = os.path.join(HERE, "host_path")
    subprocess.check_call([NVCC] + flags + ["-cudart", "none", "-Xlinker", "-Bsymbolic", "-o", out, os.path.join(mq_build.CSRC, "mixaq.cu"), os.path.join(mq_build.CSRC, "merge_static.cu"),
                                            os.path.join(fake, "fake_launch.cu"), os.path.join(fake, "fake_runtime.cpp"), "-ldl"])
    lib = C.CDLL(out)
    lib.mixaq_last_error.restype = C.c_char_p
    for n in ("mixaq_block_workspace_bytes", "mixaq_backbone_workspace_bytes", "mixaq_calibrate_block_workspace_bytes",
              "mixaq_calibrate_merge_workspace_bytes"):
        getattr(lib, n).restype = C.c_size_t
    return lib


class Host:
    """A context of the library over the stand-in, with parameters at made-up addresses."""
    OWN = C.c_void_p(0x10)                        # a stream of the caller's
    DEFAULT = C.c_void_p(None)

    def __init__(self, L):
        self.L, self.h, self.next = L, C.c_void_p(), 0x7000_0000_0000
        for flag in ("fail_capture", "fail_instantiate", "fail_graph_launch", "fake_device_word", "written_count"):
            self.set(flag, 0)
        L.fake_reset()
        assert L.mixaq_create(C.byref(self.h), 0) == 0
        self.keep = []

    def set(self, flag, value):
        C.c_int.in_dll(self.L, flag).value = value

    @property
    def counts(self):
        return Counts.in_dll(self.L, "counts")

    def addr(self, offset=0):
        self.next += 1 << 24
        return self.next + offset

    def linear(self, o, i):
        return mq.LinearS(self.addr(), self.addr(), o, i, 8)

    def block(self, dim=32, shift=0):
        s = mq.BlockS()
        s.dim, s.heads, s.window, s.shift, s.hidden = dim, dim // 32, 7, shift, 4 * dim
        s.qkv, s.proj, s.fc1, s.fc2 = self.linear(3 * dim, dim), self.linear(dim, dim), self.linear(4 * dim, dim), self.linear(dim, 4 * dim)
        s.relpos_table, s.prepared, s.score_inv_scale = self.addr(), self.addr(), 20.0
        for br, bits in ((s.hi, 8), (s.lo, 4)):
            for n in ("ln1_g", "ln1_b", "ln2_g", "ln2_b", "b_qkv", "b_proj", "b_fc1", "b_fc2"):
                setattr(br, n, self.addr())
            for n in ("qkv_in", "q", "k", "v", "proj_in", "fc1_in", "fc2_in"):
                setattr(br, n, mq.AQ(bits, 0.1, 10.0, 3))
            br.bits = bits
        return s

    def backbone(self, norms=False):
        blocks = (mq.BlockS * 2)(self.block(), self.block(shift=3))
        depths = (C.c_int * 1)(2)
        s = mq.BackboneS(1, depths, blocks, None, None, None, None)
        if norms:
            s.out_norm_g = (C.c_void_p * 1)(self.addr())
            s.out_norm_b = (C.c_void_p * 1)(self.addr())
        ws = self.L.mixaq_backbone_workspace_bytes(C.byref(s), 1, 14, 14)
        return dict(s=s, ws=C.c_void_p(self.addr()), ws_bytes=C.c_size_t(ws), out=(C.c_void_p * 1)(self.addr()))

    def run_backbone(self, b, x, stream=None, low=0.5):
        return self.L.mixaq_backbone_forward(self.h, C.byref(b["s"]), C.c_void_p(x), b["out"], 1, 14, 14, (C.c_float * 1)(low), None,
                                             b["ws"], b["ws_bytes"], stream if stream is not None else self.DEFAULT)

    def run_block(self, s, x, y, ws, stream=None, sel=None, energy=None, taps=None):
        n = C.c_size_t(self.L.mixaq_block_workspace_bytes(C.byref(s), 1, 14, 14))
        return self.L.mixaq_block_forward(self.h, C.byref(s), C.c_void_p(x), C.c_void_p(y), 1, 14, 14, C.c_float(0.5), C.c_float(0.25),
                                          C.byref(mq.SelectOpts(energy, 0)), C.byref(sel) if sel is not None else None,
                                          C.c_void_p(ws), n, C.byref(taps) if taps is not None else None, stream if stream is not None else self.DEFAULT)

    def close(self):
        assert self.L.mixaq_destroy(self.h) == 0


@pytest.fixture
def host(L):
    h = Host(L)
    yield h
    assert h.counts.violations == 0
    h.close()
    assert h.counts.live_graphs == 0


@pytest.mark.parametrize("stream", [Host.DEFAULT, Host.OWN])
def test_backbone_calls_are_recorded_at_the_second_call_and_then_replayed(host, stream):
    b, xs = host.backbone(), [host.addr() for _ in range(16)]
    for step in range(4):
        for x in xs:
            assert host.run_backbone(b, x, stream) == 0
        assert host.counts.captures == host.counts.instantiated == (0 if step == 0 else 16)
        assert host.counts.graph_launches == 16 * step
    assert host.L.mixaq_last_launch_count(host.h) > 10


@pytest.mark.parametrize("stream", [Host.DEFAULT, Host.OWN])
def test_backbone_calls_that_never_repeat_soon_are_never_recorded(host, stream):
    """More input buffers in rotation than graphs are kept, and new ratios on every call."""
    b, xs = host.backbone(), [host.addr() for _ in range(32)]
    for i in range(4 * 32):
        assert host.run_backbone(b, xs[i % 32], stream) == 0
    for i in range(64):
        assert host.run_backbone(b, xs[0], stream, low=i / 64) == 0
    assert host.counts.captures == 0 and host.counts.graph_launches == 0


def calls_in_pairs(host, kind, n):
    """Runs n calls of distinct arguments, each twice in a row."""
    b, s, ws = host.backbone(), host.block(), host.addr()
    for _ in range(n):
        x, y = host.addr(), host.addr()
        for _ in range(2):
            assert (host.run_backbone(b, x) if kind == "backbone" else host.run_block(s, x, y, ws)) == 0


@pytest.mark.parametrize("kind,budget", [("backbone", 16), ("block", 8)])
def test_recordings_that_are_not_replayed_stop_and_a_steady_caller_still_gets_its_graph(host, kind, budget):
    calls_in_pairs(host, kind, 5 * budget)
    assert host.counts.captures == budget and host.counts.live_graphs == budget
    b, s, ws, x, y = host.backbone(), host.block(), host.addr(), host.addr(), host.addr()
    for i in range(40):
        assert (host.run_backbone(b, x) if kind == "backbone" else host.run_block(s, x, y, ws)) == 0
    assert host.counts.captures == budget + 1 and host.counts.live_graphs == budget
    assert host.counts.graph_launches == budget + 40 - 31          # the pairs' second calls; recorded at the 32nd call
    # replays earn further recordings, one for every 32
    for i in range(64):
        assert (host.run_backbone(b, x) if kind == "backbone" else host.run_block(s, x, y, ws)) == 0
    calls_in_pairs(host, kind, 1)
    assert host.counts.captures == budget + 2


@pytest.mark.parametrize("off_cls,off_order,off_score", [(0, 0, 0), (1, 0, 4), (3, 2, 0), (1, 1, 1), (0, 4, 8)])
def test_selection_outputs_at_any_address(host, off_cls, off_order, off_score):
    """The kernels only get buffers that whole elements can be written to; the others are filled by copies."""
    s, x, y, ws = host.block(), host.addr(), host.addr(), host.addr()
    sel = mq.Selection(host.addr(off_cls), host.addr(off_order), host.addr(off_score), host.addr(), host.addr(), host.addr())
    assert host.run_block(s, x, y, ws, sel=sel) == 0
    args, copies = SelectArgs.in_dll(host.L, "last_select"), (Copy * 16).in_dll(host.L, "last_copies")
    late = {c.dst: (c.src, c.bytes) for c in copies[:host.counts.copies]}
    assert args.cls == sel.cls
    for name, size in (("order", 4), ("score", 8)):
        want, got = getattr(sel, name), getattr(args, name)
        assert got % size == 0
        assert got == want if want % size == 0 else late.pop(want) == (got, 4 * size)      # 4 windows of a 14 x 14 map
    assert not late


def test_only_scores_of_the_librarys_own_energies_are_ranked_in_32_bits(host):
    """A caller's energies may be of any size, wherever their map lies (the library's own is the first buffer of the workspace)."""
    x, y, ws = host.addr(), host.addr(), host.addr()
    narrow = []
    for energy in (None, host.addr(), ws):
        assert host.run_block(host.block(), x, y, ws, energy=energy) == 0
        narrow.append(SelectArgs.in_dll(host.L, "last_select").narrow)
    assert narrow == [True, False, False]


def test_misaligned_arrays_are_refused_before_a_launch(host):
    x, y, ws = host.addr(), host.addr(), host.addr()
    sel = lambda **kw: mq.Selection(**{n: host.addr() for n in ("cls", "order", "score", "idx_hi", "idx_lo", "idx_pr")} | kw)  # noqa: E731
    for name in ("idx_hi", "idx_lo", "idx_pr"):
        assert host.run_block(host.block(), x, y, ws, sel=sel(**{name: host.addr(2)})) == -1
    assert host.run_block(host.block(), x, y, ws, energy=host.addr(1)) == -1
    for setter in (lambda s: setattr(s.qkv, "scale", host.addr(2)), lambda s: setattr(s.lo, "b_fc1", host.addr(1)),
                   lambda s: setattr(s, "relpos_table", host.addr(3))):
        s = host.block()
        setter(s)
        assert host.run_block(s, x, y, ws) == -1
    assert b"aligned" in host.L.mixaq_last_error(host.h)
    assert host.counts.direct == 0


def test_patch_merging_refuses_misaligned_buffers_with_and_without_a_workspace(host):
    def merge(**off):
        at = lambda n: host.addr(off.get(n, 0))                                              # noqa: E731
        m = mq.MergeS(at("ln_g"), at("ln_b"), mq.AQ(8, 0.1, 10.0, 3), host.linear(64, 128), at("prepared"))
        m.reduction.codes = at("codes")
        x, y = C.c_void_p(at("x")), C.c_void_p(at("y"))
        return (host.L.mixaq_merge_forward(host.h, C.byref(m), x, y, 1, 8, 8, C.c_void_p(host.addr()), C.c_size_t(1 << 20), None),
                host.L.mixaq_merge_forward_static(host.h, C.byref(m), x, y, 1, 8, 8, None))
    for off in (dict(x=4), dict(y=8), dict(codes=1), dict(ln_g=4), dict(ln_b=4), dict(prepared=16)):
        assert merge(**off) == (-1, -1), off
    assert host.counts.direct == 0
    assert merge() == (0, 0) and host.counts.direct == 4


@pytest.mark.parametrize("kind", ["backbone", "block"])
@pytest.mark.parametrize("stream", [Host.DEFAULT, Host.OWN])
@pytest.mark.parametrize("flag", ["fail_capture", "fail_instantiate", "fail_graph_launch"])
def test_a_call_that_cannot_be_recorded_is_issued(host, kind, stream, flag):
    """No memory for a graph, or a stream that cannot be captured just now: the call does its work, and is recorded later."""
    b, s, x, y, ws = host.backbone(norms=True), host.block(), host.addr(), host.addr(), host.addr()
    call = lambda: host.run_backbone(b, x, stream) if kind == "backbone" else host.run_block(s, x, y, ws, stream)   # noqa: E731
    assert call() == 0
    launches = host.counts.direct
    host.set(flag, 1)
    for i in range(2, 5):
        assert call() == 0
        assert host.counts.direct == i * launches and host.L.mixaq_last_launch_count(host.h) == launches
    assert host.counts.graph_launches == 0 and host.counts.live_graphs == 0
    host.set(flag, 0)
    for _ in range(3):
        assert call() == 0
    assert host.counts.live_graphs == 1 and host.counts.graph_launches > 0


@pytest.mark.parametrize("kind", ["backbone", "block"])
@pytest.mark.parametrize("stream", [Host.DEFAULT, Host.OWN])
def test_guard_zones_and_ranges_apply_to_calls_that_were_recorded_before(host, kind, stream):
    b, s, x, y, ws = host.backbone(), host.block(), host.addr(), host.addr(), host.addr()
    call = lambda: host.run_backbone(b, x, stream) if kind == "backbone" else host.run_block(s, x, y, ws, stream)   # noqa: E731
    for _ in range(3):
        assert call() == 0
    replayed, launches = host.counts.graph_launches, host.L.mixaq_last_launch_count(host.h)
    blocks = 2 if kind == "backbone" else 1
    host.L.mixaq_set_workspace_guards(host.h, 1)
    assert call() == 0 and host.counts.guard_launches == 2 * blocks                 # filled, compared
    host.L.mixaq_set_workspace_guards(host.h, 0)
    host.L.mixaq_set_nvtx(host.h, 1)
    direct = host.counts.direct
    assert call() == 0 and host.counts.direct == direct + launches
    host.L.mixaq_set_nvtx(host.h, 0)
    assert host.counts.graph_launches == replayed
    assert call() == 0 and host.counts.graph_launches == replayed + 1


def test_two_threads_share_a_context(host):
    """Two threads, blocks and backbones on a stream of their own and on the default stream, new keys and old ones mixed:
    recordings do not meet (the stand-in counts launches into another thread's capture and captures of a busy stream)."""
    failed = []

    def work(t):
        h, b, s = host, made[t][0], made[t][1]
        try:
            for i in range(60):
                stream = (Host.DEFAULT, C.c_void_p(0x20 + 0x10 * t))[i % 3 == 0]
                assert h.run_backbone(b, xs[t][i // 4 % 5], stream) == 0
                assert h.run_block(s, xs[t][5], xs[t][6 + i // 4 % 5], ws[t], stream) == 0
        except BaseException as e:                                                               # noqa: BLE001
            failed.append(e)
    made = [(host.backbone(norms=True), host.block()) for _ in range(2)]
    xs = [[host.addr() for _ in range(11)] for _ in range(2)]
    ws = [host.addr() for _ in range(2)]
    threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    assert host.counts.violations == 0 and host.counts.graph_launches > 0 and host.counts.side_launches > 0


def test_recording_leaves_the_callers_stream_alone(host):
    """A stream being captured refuses what other threads put on it, and a blocking one their work on the default stream
    too: calls are recorded on a stream of the context's own."""
    b, s, ws = host.backbone(norms=True), host.block(), host.addr()
    for _ in range(3):
        assert host.run_backbone(b, 0x7000_0000, Host.OWN) == 0
        assert host.run_block(s, 0x7100_0000, 0x7200_0000, ws, Host.OWN) == 0
    assert host.counts.captures == 2
    origins = (C.c_void_p * 16).in_dll(host.L, "capture_origins")
    assert all(o != Host.OWN.value for o in origins[:2])


@pytest.mark.parametrize("stream", [Host.DEFAULT, Host.OWN])
def test_output_norms_run_beside_the_chain_also_after_eviction(host, stream):
    """Every recording of an image backbone puts its norms on the side stream, also when earlier graphs have left."""
    b = host.backbone(norms=True)
    xs = [host.addr() for _ in range(17)]
    for x in xs[:16] + [xs[0]] * 40:                           # replays that earn a further recording
        for _ in range(2):
            assert host.run_backbone(b, x, stream) == 0
    for _ in range(2):
        assert host.run_backbone(b, xs[16], stream) == 0       # displaces xs[1], the least recently used
    assert (host.counts.captures, host.counts.live_graphs, host.counts.side_launches) == (17, 16, 17)
    replayed = host.counts.graph_launches
    assert host.run_backbone(b, xs[0], stream) == 0 and host.counts.graph_launches == replayed + 1
    assert host.run_backbone(b, xs[1], stream) == 0 and host.counts.graph_launches == replayed + 1


def test_a_calibration_whose_waits_ran_out_says_so(host):
    """The status word that the product's kernels raise comes back with the ranges; the host's own copy of it is not stale."""
    s, r = host.block(), mq.BlockRangesS()
    m, rm = mq.MergeS(host.addr(), host.addr(), mq.AQ(8, 0.1, 10.0, 3), host.linear(64, 128), host.addr()), mq.RangeS()
    x, y, ws = (C.c_void_p(host.addr()) for _ in range(3))
    n = C.c_size_t(host.L.mixaq_calibrate_block_workspace_bytes(C.byref(s), 1, 14, 14))
    nm = C.c_size_t(host.L.mixaq_calibrate_merge_workspace_bytes(C.byref(m), 1, 8, 8))
    calls = (lambda: host.L.mixaq_calibrate_block(host.h, C.byref(s), 0, x, y, 1, 14, 14, C.byref(r), ws, n, None),
             lambda: host.L.mixaq_calibrate_merge(host.h, C.byref(m), x, y, 1, 8, 8, C.byref(rm), ws, nm, None))
    for call in calls:
        for word in (0, 1, 0):
            host.set("fake_device_word", word)
            assert call() == (-5 if word else 0)                 # MIXAQ_DEVICE_TIMEOUT


@pytest.mark.parametrize("taps", [False, True])
@pytest.mark.parametrize("bits,mult", [((8, 4), 4), ((4, 2), 4), ((2, 2), 4), ((2, 2), 64)])
def test_guard_zones_lie_around_the_buffers_that_calls_use(host, bits, mult, taps):
    """One code per byte inside the packed workspace, unless taps ask for packed codes or the hidden layer is too wide: with the
    zones on as without, each buffer followed by its own zone."""
    s, x, y, ws = host.block(dim=64, shift=3), host.addr(), host.addr(), host.addr()
    s.hidden = s.fc1.out_features = s.fc2.in_features = 64 * mult
    for br, b in ((s.hi, bits[0]), (s.lo, bits[1])):
        br.bits = b
        for n in ("qkv_in", "q", "k", "v", "proj_in", "fc1_in", "fc2_in"):
            setattr(br, n, mq.AQ(b, 0.1, 10.0, 1))
    found = []
    for guards in (1, 0):
        host.L.mixaq_set_workspace_guards(host.h, guards)
        host.set("written_count", 0)
        assert host.run_block(s, x, y, ws, taps=mq.Taps() if taps else None) == 0
        n = C.c_int.in_dll(host.L, "written_count").value
        found.append([(r.at, r.bytes, r.code_bits) for r in (Range * 256).in_dll(host.L, "written")[:n]])
    assert found[0] == found[1] and len(found[0]) == 2 * 6
    packed = taps or mult == 64
    assert [r[2] for r in found[0] if r[2]] == 5 * (list(bits) if packed else [8, 8])
    zones = (C.c_void_p * 64).in_dll(host.L, "guard_zones")[:C.c_int.in_dll(host.L, "guard_count").value]
    end = ws + host.L.mixaq_block_workspace_bytes(C.byref(s), 1, 14, 14)
    for z in zones:
        assert ws < z <= end - 256
        assert all(z + 256 <= at or at + size <= z for at, size, _ in found[0])
    # what lies side by side or overlaps (both branches' rows, buffers that take turns) has one zone behind it
    groups = []
    for at, size, _ in sorted(found[0]):
        if groups and at <= groups[-1][1]:
            groups[-1][1] = max(groups[-1][1], at + size)
        else:
            groups.append([at, at + size])
    assert len(groups) == (12 if packed else 4)
    for (_, last), following in zip(groups, [g[0] for g in groups[1:]] + [end]):
        assert sum(last <= z < following for z in zones) == 1


@pytest.mark.parametrize("mult", [1, 4, 16])
def test_calibration_workspace_shares_memory_of_what_is_dead(host, mult):
    """fc2's byte planes lie over what no product behind fc1 reads; nothing else overlaps."""
    dim, s = 96, host.block(dim=96)
    s.hidden = s.fc1.out_features = s.fc2.in_features = dim * mult
    ws, x, y, r = host.addr(), C.c_void_p(host.addr()), C.c_void_p(host.addr()), mq.BlockRangesS()
    M = 2 * 9 * 49                                                        # 2 maps of 17 x 20: 9 windows each
    bytes_ = host.L.mixaq_calibrate_block_workspace_bytes(C.byref(s), 2, 17, 20)
    assert host.L.mixaq_calibrate_block(host.h, C.byref(s), 0, x, y, 2, 17, 20, C.byref(r), C.c_void_p(ws), C.c_size_t(bytes_), None) == 0
    names = ("obs", "rowsrc", "expo", "x1", "h", "ln", "qkv", "o", "slices", "slices_fc2")
    size = dict(obs=4 * 17, rowsrc=4 * M, expo=4 * M, x1=4 * M * dim, h=4 * M * s.hidden, ln=4 * M * dim, qkv=12 * M * dim, o=4 * M * dim,
                slices=7 * M * dim, slices_fc2=7 * M * s.hidden)
    at = dict(zip(names, (C.c_void_p * 10).in_dll(host.L, "last_calibration")))
    over = {"ln", "qkv", "o", "slices"}                                   # what slices_fc2 may overlap
    for a in names:
        assert ws <= at[a] and at[a] + size[a] <= ws + bytes_ and at[a] % 256 == 0
        for b in names:
            if a < b and not ({a, b} - over == {"slices_fc2"}):
                assert at[a] + size[a] <= at[b] or at[b] + size[b] <= at[a], (a, b)
    if mult == 4:
        assert bytes_ <= M * (48 * dim + 8) + 10 * 512
