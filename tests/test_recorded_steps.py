"""TrainStep.run issues recorded calls from native code.  Here, without a GPU, every run is compared with the walk over the
layers on the same object: the same entry points, with the same arguments, on the same streams, in the same order.  The
library's launching entry points are replaced by a log; lpdt_run_calls is decoded into it by the layout that the header
states."""
import contextlib
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2111_09389_b200 import _lib, api
from paper_2111_09389_b200 import workloads as wlmod
from paper_2111_09389_b200.step import TrainStep

# host arrays of an entry point: argument -> (element type, index of the argument that counts them, elements more than that)
HOST = {"lpdt_quantize_batch": {i: (C.c_int64, 3, 0) for i in (4, 5, 6)},
        "lpdt_range_evonorm_bwd_params_batch": {3: (C.c_int32, 2, 0), 4: (C.c_uint64, 2, 0), 5: (C.c_int64, 2, 0)},
        "lpdt_dequantize_acc_batch": {3: (C.c_int64, 2, 0), 4: (C.c_int64, 2, 0), 5: (C.c_int64, 2, 0),
                                      6: (C.c_uint64, 2, 0), 7: (C.c_uint64, 2, 0)},
        "lpdt_gossip_mix": {8: (C.c_int64, 7, 1), 9: (C.c_int64, 7, 0)},
        "lpdt_gossip_mix_q8": {8: (C.c_int64, 7, 1), 9: (C.c_int64, 7, 0)}}
FLOAT_BITS = lambda v: C.c_uint32.from_buffer(C.c_float(v)).value


class Stream:
    made = 0

    def __init__(self, device=None):
        Stream.made += 1
        self.cuda_stream, self.device_index = 1000 + Stream.made, 0

    def wait_stream(self, other):
        Log.calls.append(("wait", self.cuda_stream, other.cuda_stream))


class Event:
    made = 0

    def __init__(self, *a, **kw):
        Event.made += 1
        self.cuda_event = 5000 + Event.made

    def record(self, *a):
        pass


class Log:
    calls, native, stack = [], 0, []


def entry(name, args):
    """A call as a comparable tuple: floats by their bits, descriptors and host arrays by their contents."""
    if name in ("lpdt_quantize", "lpdt_quantize_with_range") and args[5] == 0:
        args = (*args[:6], 0, *args[7:])                   # the seed of a call that draws nothing
    out = [name, int(args[-1] or 0)]
    for i, (kind, a) in enumerate(zip(_lib.SIGNATURES[name][1][:-1], args)):
        if kind is C.c_float:
            out.append(FLOAT_BITS(a))
        elif kind is C.POINTER(_lib.ConvDesc):
            d = a._obj if hasattr(a, "_obj") else _lib.ConvDesc.from_address(a)
            out.append(tuple(getattr(d, f) for f, _ in d._fields_))
        elif i in HOST.get(name, {}):
            t, count, more = HOST[name][i]
            out.append(tuple((t * (args[count] + more)).from_address(a)))
        else:
            out.append(int(a or 0))
    return tuple(out)


class Library:
    def __init__(self, real):
        self.real, self.ids = real, {}
        for name in _lib.SIGNATURES:
            i = real.lpdt_call_id(name.encode())
            if i >= 0:
                self.ids[i] = name

    def __getattr__(self, name):
        if name not in api.LAUNCHING and name != "lpdt_fill_zero":
            return getattr(self.real, name)

        def call(*args):
            assert len(args) == len(_lib.SIGNATURES[name][1])
            Log.calls.append(entry(name, args))
            return 0
        return call

    def lpdt_run_calls(self, code, n_words, streams, n_streams, failed):
        Log.native += 1
        w = list((C.c_uint64 * n_words).from_address(code))
        handles = list((C.c_uint64 * n_streams).from_address(streams))
        i = 0
        while i < n_words:
            if w[i] == api.CALL_WAIT:
                assert w[i + 3]
                Log.calls.append(("wait", handles[w[i + 1]], handles[w[i + 2]]))
                i += 4
                continue
            name = self.ids[w[i]]
            kinds = _lib.SIGNATURES[name][1][:-1]
            args = [C.c_float.from_buffer(C.c_uint32(v)).value if k is C.c_float else
                    C.c_int64(v).value if k in (C.c_int32, C.c_int64) else v for k, v in zip(kinds, w[i + 2:])]
            Log.calls.append(entry(name, args + [handles[w[i + 1]]]))
            i += 2 + len(kinds)
        return 0


@pytest.fixture(autouse=True)
def no_gpu(monkeypatch):
    library = Library(_lib.lib())
    Log.calls, Log.native, Log.stack = [], 0, [Stream()]

    @contextlib.contextmanager
    def on(stream):
        Log.stack.append(stream)
        yield
        Log.stack.pop()
    for name, value in dict(is_available=lambda: True, Stream=Stream, Event=Event, stream=on, synchronize=lambda: None,
                            current_stream=lambda *a: Log.stack[-1], is_current_stream_capturing=lambda: False).items():
        monkeypatch.setattr(torch.cuda, name, value)
    monkeypatch.setattr(api, "_load", lambda: library)
    monkeypatch.setattr(api, "_ptr", lambda t: None if t is None else t.data_ptr())


def make(name="conv16", cls=TrainStep, **kw):
    if name == "conv16":
        wl = wlmod.make_workload("conv16")
    else:
        wl = wlmod.make_workload("resnet20_topk", nodes=4, batch=2)
    st = cls.from_workload(wl, device="cpu", **kw)
    st.Wmix.copy_(torch.from_numpy(wl["Wmix"]))
    return st


def issued(fn):
    Log.calls = []
    fn()
    return Log.calls


def same(st, what=""):
    """One run issues what a walk over the layers issues; True if it was issued natively."""
    before = Log.native
    got = issued(st.run)
    native = Log.native - before
    state = (st.out, st.input_grad_out, [(b.get("x"), b.get("addend")) for g in (st, *st.groups) for b in g.buf])
    want = issued(st._run)
    assert got == want, what
    after = (st.out, st.input_grad_out, [(b.get("x"), b.get("addend")) for g in (st, *st.groups) for b in g.buf])
    assert state[0] is after[0] and state[1] is after[1] and all(a is b for p, q in zip(state[2], after[2]) for a, b in zip(p, q)), what
    return bool(native)


def settles(st):
    """Runs are issued natively again once nothing changes any more."""
    return any([same(st) for _ in range(70)][-3:])


def recorded(*a, **kw):
    st = make(*a, **kw)
    for _ in range(3):
        same(st)
    assert same(st)                                        # issued natively by now
    return st


# ---- the walk's own code ------------------------------------------------------------------------
def clipping(st):
    """An update with arithmetic of its own between the library calls; returns the list of its executions."""
    done = []

    def update():
        done.append(1)
        st.grads.clamp_(-1, 1)
        api.lpdt_sgd_update(st.N * st.d, st.params, st.grads, 0.5, st.x_half)     # a rate of its own
        api.lpdt_gossip_mix(st.N, st.d, st.x_half, st.x_hat, st.x_out, st.Wmix, 0.25, st.seg_offsets, st.seg_k, st.ws)
    return update, done


@pytest.mark.parametrize("where", ["subclass", "instance", "class", "late", "entry point"])
def test_replaced_parts_of_the_step_run_every_time(where, monkeypatch):
    if where == "subclass":
        class Mine(TrainStep):
            def update(self):
                clipping(self)[0]()
                done.append(1)
        done, st = [], make(cls=Mine)
    else:
        st = make()
        update, done = clipping(st)
        if where == "instance":
            st.update = update
        elif where == "class":
            monkeypatch.setattr(TrainStep, "update", lambda self: update())
        elif where == "late":
            for _ in range(4):
                same(st)
            st.update = update
        else:
            st.gamma = 0.125

            def mix(*a, **kw):
                done.append(1)
            monkeypatch.setattr(api, "lpdt_sgd_gossip_mix", mix)
    for i in range(5):
        del done[:]
        got = issued(st.run)
        assert len(done) == 1, i
        assert got == issued(st._run)
        if where != "entry point":
            rates = [c[5] for c in got if c[0] == "lpdt_sgd_update"]
            assert rates == [FLOAT_BITS(0.5)]
            assert [c[8] for c in got if c[0] == "lpdt_gossip_mix"] == [FLOAT_BITS(0.25)]


def test_an_overridden_run_is_logged_and_captured(monkeypatch):
    class Mine(TrainStep):
        def run(self):
            super().run()
            done.append(torch.cuda.is_current_stream_capturing())
            api.lpdt_sgd_update(self.N * self.d, self.params, self.grads, 0.5, self.x_half)

    capturing = []

    @contextlib.contextmanager
    def graph(g):
        capturing.append(g)
        yield
        capturing.pop()
    monkeypatch.setattr(torch.cuda, "CUDAGraph", object)
    monkeypatch.setattr(torch.cuda, "graph", graph)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: bool(capturing))
    done, st = [], make(cls=Mine)
    log = st.record()
    assert done == [False] and [r[0] for r in log][-1] == "lpdt_sgd_update"
    for _ in range(4):
        st.run()
    native = Log.native
    del done[:]
    got = issued(st.capture)
    assert done == [False, True]                           # the warm-up, and the captured one
    assert [c[0] for c in got].count("lpdt_sgd_update") == 2
    assert Log.native == native + 1                        # nothing native is captured but the warm-up's


# ---- everything else a walk reads ---------------------------------------------------------------
OPTIONS = [("conv16", {}), ("conv16", dict(grad_rounding=1, message_bits=8)), ("resnet20", dict(node_groups=2)),
           ("resnet20", dict(quantize_wgrad=True, recompute_norm_input=True)),
           ("resnet20", dict(fuse_requantize=True, message_bits=8, node_groups=3))]


def replaying_or_not(st):
    st._unused = st._rest = 0
    return [same(st) for _ in range(4)]


def replaying(st):
    st._unused = st._rest = 0
    while not same(st):
        pass


@pytest.mark.parametrize("name,kw", OPTIONS)
def test_any_replaced_tensor_is_used_by_the_next_run(name, kw):
    """Every tensor of the step and of its node groups, and those of some layers, replaced by a copy between two runs that
    are issued natively."""
    st = recorded(name, **kw)
    native = 0
    for who in (st, *st.groups):
        for n in [n for n, t in who.__dict__.items() if isinstance(t, torch.Tensor) and n not in ("out", "input_grad_out")]:
            setattr(who, n, getattr(who, n).clone())
            native += same(st, n)
            replaying(st)
    assert native > 0                                      # those that share no memory with others do not even walk
    for who in (st, *st.groups):
        for li, b in list(enumerate(who.buf))[:4] + list(enumerate(who.buf))[-2:]:
            for n in [n for n, t in b.items() if isinstance(t, torch.Tensor) and n not in ("x", "addend")]:
                b[n] = b[n].clone()
                same(st, (li, n))
                replaying(st)


@pytest.mark.parametrize("name,kw", OPTIONS)
def test_any_changed_setting_counts_for_the_next_run(name, kw):
    st = recorded(name, **kw)
    for who in (st, *st.groups):
        for n, v in (("eps", 1e-4), ("lr", 0.25), ("gamma", 0.75), ("seed", 99), ("lr", torch.tensor(0.125)), ("side", Stream()),
                     ("stream", Stream()), ("labels", None), ("quantize_wgrad", False), ("input_grad", False), ("out", None)):
            if n == "stream" and who is st:
                continue
            old = getattr(who, n)
            setattr(who, n, v)
            same(st, n)
            same(st, n)
            setattr(who, n, old)
            for _ in range(4):
                same(st, n)
    st.lr = torch.tensor(0.125)
    same(st)
    st.lr.mul_(0.5)
    same(st)


@pytest.mark.parametrize("kw", [dict(), dict(node_groups=2)])
def test_layer_entries_lists_and_streams_count_too(kw):
    st = recorded("resnet20", **kw)
    again = lambda what: [same(st, what) for _ in range(4)]
    for who in (st, *st.groups):
        conv = next(b for b in who.buf if "desc" in b)
        d = conv["desc"]
        conv["desc"] = api.conv_desc(d.nodes, d.B, d.H, d.W, d.Cin, d.Cout, 1, 1, 1, 0)
        again("descriptor")
        conv["desc"].pad = 7
        again("descriptor in place")
        conv["desc"] = d
        again("descriptor back")
        who.buf = [dict(b) for b in who.buf]
        again("layers")
        who.buf[0] = dict(who.buf[0])
        who.buf[0]["out"] = who.buf[0]["out"].clone()
        again("layer")
    st.seg_k[0] -= 1
    again("kept")
    st.w_dst[-1] += 256
    again("weights")
    st.ops[-1]["b_off"] -= 1
    again("layer list")
    st.seg_k, st.seg_offsets = [5, 6], [0, 100, st.d]
    st.msg_scale = torch.zeros(st.N, 2)
    again("segments")
    st.message_bits = 8
    again("messages")
    for kept, offsets in (((5, 6), (0, 100, st.d)), (np.array([5, 7]), np.array([0, 100, st.d])), ([5, 6], [0, 100, st.d])):
        st.seg_k, st.seg_offsets = kept, offsets           # any sequence will do
        replaying_or_not(st)
    st.ws = torch.zeros(st.ws.numel() + 512, dtype=torch.uint8)
    again("workspace")
    first = st.ws
    for view in (first[256:], first[:-256], first):
        st.ws = view
        again("workspace in place")
    st.x.data = torch.zeros_like(st.x)
    again("storage")
    with torch.cuda.stream(Stream()):
        assert same(st, "stream")
        with torch.cuda.stream(st.side):                   # the walk's two streams become one
            again("side")
    again("stream")
    st.params = torch.zeros(st.N, 2 * st.d)[:, ::2]
    again("strides")
    b = next(b for b in (st.groups or [st])[-1].buf if "amin" in b)
    for missing in (dict(amin=None), {}):
        amin = b.pop("amin")
        b.update(missing)
        if missing:
            again("missing")
        else:
            for _ in range(3):
                with pytest.raises(KeyError):
                    st.run()
        b["amin"] = amin
        again("there again")
    assert settles(st)


def test_swapped_and_new_buffers_do_not_walk():
    for kw in ({}, dict(node_groups=2)):
        st = recorded("resnet20", **kw)
        for _ in range(5):
            st.x_hat, st.x_half = st.x_half, st.x_hat
            if not kw:
                st.params, st.x_out = st.x_out, st.params
                st.x = torch.zeros_like(st.x)
                st.labels = torch.zeros_like(st.labels)
            assert same(st)


def off_boundary(t):
    """A copy of a tensor, four bytes off a 16-byte boundary."""
    flat = torch.zeros(t.numel() + 4, dtype=t.dtype)
    at = next(i for i in range(4) if flat[i:].data_ptr() % 16 == 4)
    return flat[at:at + t.numel()].view(t.shape).copy_(t)


def pooled_step(**kw):
    """A norm layer with pooling behind it at either end of the step."""
    ren = lambda H, at: dict(op="ren", H=H, W=H, C=16, groups=2, p_off=at)
    pool = lambda H: dict(op="maxpool", H=H, W=H, C=16)
    ops = [ren(8, 0), pool(8), dict(op="conv", H=4, W=4, cin=16, cout=16, R=3, S=3, stride=1, pad=1, w_off=48), ren(4, 2352), pool(4)]
    return TrainStep(ops, 2400, 4, 3, (8, 8, 16), has_labels=False, input_grad=True, device="cpu", **kw)


@pytest.mark.parametrize("kw", [{}, dict(node_groups=2)])
def test_pooling_takes_a_launch_of_its_own_where_four_values_cannot_be_read(kw):
    """Whatever lies off a 16-byte boundary, in the walk and between recorded runs: that layer and its pooling are two calls."""
    st = pooled_step(**kw)
    groups = st.groups or [st]

    def counts():
        got = [c[0] for c in issued(st.run)]
        return [got.count("lpdt_range_evonorm_" + n) // len(groups) for n in ("pool_fwd", "pool_bwd")] + [
            got.count("lpdt_maxpool2x2" + n) // len(groups) for n in ("", "_bwd")]
    for _ in range(4):
        same(st)
    assert same(st) and counts() == [2, 2, 0, 0]
    for who in (st, *st.groups):                           # nothing is kept that the one launch does not write
        assert [("out" in b, "dx" in b) for b in who.buf] == [(False, True), (True, False), (True, True), (False, True), (True, False)]
    for name, want in (("x", [1, 1, 1, 1]), ("dy", [2, 1, 0, 1]), (("out", 2), [1, 1, 1, 1]), (("dx", 0), [2, 1, 0, 1]),
                       (("out", 4), [1, 2, 1, 0])):
        who = groups[0]
        entry, key = (who.__dict__, name) if isinstance(name, str) else (who.buf[name[1]], name[0])
        old = entry[key]
        entry[key] = off_boundary(old)
        for _ in range(3):
            same(st, name)
        if not kw:
            assert counts() == want, name
        entry[key] = old
        for _ in range(3):
            same(st, name)
        assert counts() == [2, 2, 0, 0]
    if not kw:
        replaying(st)
        st.loss = off_boundary(st.loss)                    # not one of theirs
        assert same(st)


@pytest.mark.parametrize("kw", [{}, dict(node_groups=2)])
def test_no_sums_are_kept_for_weight_gradients_of_one_launch(kw):
    conv = lambda c, at: dict(op="conv", H=2, W=2, cin=c, cout=c, R=3, S=3, stride=1, pad=1, w_off=at)
    size = lambda c: 9 * c * c
    ops = [conv(256, 0), conv(256, size(256))]
    st = TrainStep(ops, 2 * size(256), 8, 4, (2, 2, 256), has_labels=False, device="cpu", **kw)
    assert all(b["direct"] and "gacc" not in b for who in (st, *st.groups) for b in who.buf) and st.g_acc.numel() == 64
    calls = [c for c in issued(st.run) if c[0].startswith(("lpdt_qconv_bwd_weight", "lpdt_dequantize_acc"))]
    assert len(calls) == 2 * max(len(st.groups), 1)
    few = TrainStep([conv(16, 0), conv(32, size(16))], size(16) + size(32), 8, 4, (2, 2, 16), has_labels=False, device="cpu", **kw)
    sums = [b for b in few.buf if not b["direct"]]
    assert few.g_acc.numel() == max(64, sum(8 * b["wn"] for b in sums)) and all(b["gacc"].shape == (8, b["wn"]) for b in sums)


def test_recordings_that_are_never_replayed_become_rare():
    st = make()
    noted = 0
    for i in range(200):
        st.eps = 1e-5 * (1 + i)                            # something else in every run
        assert not same(st)
        noted += st._calls is not None
    assert noted <= 8
    assert settles(st)


def test_a_property_in_the_place_of_a_buffer():
    class Mine(TrainStep):
        @property
        def x(self):
            return self.__dict__["_x"]

        @x.setter
        def x(self, v):
            self.__dict__["_x"] = v
    st = make(cls=Mine)
    for _ in range(5):
        same(st)
        st.x = st.x.clone()
    assert same(st)
