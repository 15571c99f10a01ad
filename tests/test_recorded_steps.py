"""TrainStep.run issues recorded calls from native code.  Here, without a GPU, every run is compared with the walk over the
layers on the same object: the same entry points, with the same arguments, on the same streams, in the same order.  The
library's launching entry points are replaced by a log; lpdt_run_calls is decoded into it by the layout that the header
states."""
import contextlib
import ctypes as C

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
