"""The hot calls marshalled in C (_kvdcall) hand the library what ctypes hands it, and leave every argument that is not
plain to ctypes: same values, same exceptions (no GPU: callbacks stand in for the library)."""
import ctypes
import os
import subprocess
import sys
import sysconfig

import numpy as np
import pytest
import torch

from paper_2603_19664_b200 import binding as B

LIB = B.load()
SEEN = []


def _bytes(address, count, struct):
    return None if not address else ctypes.string_at(address, count * ctypes.sizeof(struct))


# (arguments, {index of an array: (index of its length, element)})
ARRAYS = {
    "kvd_recompute_kv_step": {2: (3, B.kvd_store_range)},
    "kvd_decode_step_kv": {2: (3, B.kvd_store_range), 8: (7, ctypes.c_int32)},
    "kvd_decode_attention": {4: (2, ctypes.c_int32), 5: (lambda a: a[2] * a[6], B.kvd_kv_segment)},
    "kvd_prefill_attention": {5: (6, B.kvd_kv_segment)},
}


@pytest.fixture
def fake(monkeypatch):
    """A context whose library calls are recorded, by ctypes and by _kvdcall alike; they answer 0."""
    keep, fns = [], {}
    for name in B._CALLS:
        real = getattr(LIB, name)
        types = [ctypes.c_void_p if t not in (ctypes.c_int, ctypes.c_int64, ctypes.c_float) else t for t in real.argtypes]

        def record(*a, name=name):
            a = list(a)
            for i, (count, struct) in ARRAYS.get(name, {}).items():
                a[i] = _bytes(a[i], count(a) if callable(count) else a[count], struct)
            SEEN.append((name, a))
            return 0

        keep.append(ctypes.CFUNCTYPE(ctypes.c_int, *types)(record))
        fns[name] = ctypes.cast(keep[-1], ctypes.c_void_p).value
        B._calls.bind(name, fns[name])

    class Lib:
        pass

    lib = Lib()
    for name in B._CALLS:
        f = ctypes.CFUNCTYPE(ctypes.c_int, *getattr(LIB, name).argtypes)(fns[name])
        setattr(lib, name, f)
    c = B.Kvd.__new__(B.Kvd)
    c._lib, c._h, c._addr, c._keep = lib, ctypes.c_void_p(0x1000), 0x1000, []
    monkeypatch.setattr(B, "_stream", lambda s: 77 if s is None else int(s))
    del SEEN[:]
    yield c
    c._h = None
    for name in B._CALLS:
        B._calls.bind(name, ctypes.cast(getattr(LIB, name), ctypes.c_void_p).value)


T = torch.zeros((8, 64))


class Slow:
    """Calls of these names are answered -1, as for an argument that is not plain."""

    def __getattr__(self, name):
        return lambda *a: -1


def _both(fake, monkeypatch, call):
    call(fake)
    plain = list(SEEN)
    del SEEN[:]
    with monkeypatch.context() as m:
        m.setattr(B, "_calls", Slow())
        call(fake)
    slow = list(SEEN)
    del SEEN[:]
    assert plain == slow and len(plain) == 1
    return plain[0]


RANGES = [(i, 3 + i, 10, T[1], T[2]) for i in range(3)]
SEGS = [[(T[0], T[1], 192, 0, 5), (T[2], T[3], 1 << 33, 5, 1)], [], ((T[4], T[5], 64, 9, 2),)]
CALLS = [
    lambda c: c.kvd_reset_sequence(3),
    lambda c: c.kvd_checkpoint_residual(1, 2, T, T[1], 7),
    lambda c: c.kvd_checkpoint_residual(1, 2, None, None, 7, stream=5),
    lambda c: c.kvd_recompute_kv(0, T, T[1], 5, T[2], T[3], 1 << 35, seq=4, first_row=9),
    lambda c: c.kvd_recompute_kv(0, None, None, 5, T[2], T[3], 64),
    lambda c: c.kvd_recompute_kv_step(0, RANGES, T, T[1], 1, T[2], T[3], 64),
    lambda c: c.kvd_recompute_kv_step(0, tuple(RANGES), None, None, 0, None, None, 64),
    lambda c: c.kvd_decode_step_kv(0, RANGES[:1], 64, T, T[1], 2, [5, 6], T[2], T[3], 128),
    lambda c: c.kvd_decode_step_kv(0, [], 64, T, T[1], 2, None, T[2], T[3], 128),
    lambda c: c.kvd_decode_attention(0, 3, T, [7, 8, 9], SEGS, 0.25, T[6]),
    lambda c: c.kvd_decode_attention(0, 64, T, list(range(64)), [SEGS[0]] * 64, 0.0, T[6], stream=3),
    lambda c: c.kvd_prefill_attention(0, 5, T, T[1], SEGS[0], 0.0, T[6]),
    lambda c: c.kvd_prefill_attention(0, 5, T, T[1], [], 0.5, T[6]),
    # not plain: marshalled by ctypes, in both runs
    lambda c: c.kvd_reset_sequence(np.int32(3).item()),
    lambda c: c.kvd_decode_attention(0, 1, T, np.array([4]), [SEGS[0]], 0.0, T[6]),
    lambda c: c.kvd_decode_attention(0, 1, T, [4], [[(1 << 20, 256, 64, 0, 5)]], 1, T[6]),
    lambda c: c.kvd_decode_attention(0, 1, T, [4], [[(T, None, 64, (1 << 33) + 2, 5)]], 0.0, T[6]),
    lambda c: c.kvd_recompute_kv_step(0, [(0, (1 << 32) + 1, 2, T[1], T[2])], None, None, 0, None, None, 64),
    lambda c: c.kvd_decode_step_kv(0, [], 64, T, T[1], 2, (np.int64(1), 2), T[2], T[3], 128),
]


@pytest.mark.parametrize("i", range(len(CALLS)))
def test_the_library_sees_the_same_call(fake, monkeypatch, i):
    _both(fake, monkeypatch, CALLS[i])


def test_values_arrive(fake):
    CALLS[9](fake)
    name, a = SEEN[0]
    assert name == "kvd_decode_attention" and a[:3] == [0x1000, 0, 3] and a[3] == T.data_ptr() and a[6] == 2 and a[7] == 0.25 and a[9] == 77
    assert list((ctypes.c_int32 * 3).from_buffer_copy(a[4])) == [7, 8, 9]
    e = (B.kvd_kv_segment * 6).from_buffer_copy(a[5])
    assert (e[0].k, e[1].v, e[1].row_stride, e[1].first_pos, e[1].len) == (T.data_ptr(), T[3].data_ptr(), 1 << 33, 5, 1)
    assert (e[2].k, e[2].len, e[3].k, e[4].k, e[4].first_pos, e[5].len) == (None, 0, None, T[4].data_ptr(), 9, 0)


@pytest.mark.parametrize("call,error", [
    (lambda c: c.kvd_checkpoint_residual(1, 2, 123, T, 7), AttributeError),
    (lambda c: c.kvd_checkpoint_residual(1, "2", T, T, 7), ctypes.ArgumentError),
    (lambda c: c.kvd_recompute_kv_step(0, [(0, 0, 1, T)], None, None, 0, None, None, 64), ValueError),
    (lambda c: c.kvd_decode_attention(0, 2, T, [1], [SEGS[0]], 0.0, T), IndexError),
    (lambda c: c.kvd_decode_attention(0, 1, T, [1], [[(T, T, 64, 0)]], 0.0, T), ValueError),
    (lambda c: c.kvd_prefill_attention(0, 1, T, T, 5, 0.0, T), TypeError),
])
def test_what_was_refused_is_refused(fake, monkeypatch, call, error):
    for slow in (False, True):
        with monkeypatch.context() as m:
            if slow:
                m.setattr(B, "_calls", Slow())
            with pytest.raises(error):
                call(fake)
    assert not SEEN


def test_an_interrupt_inside_an_argument_is_not_swallowed(fake):
    class Interrupted:
        calls = 0

        def data_ptr(self):
            self.calls += 1
            if self.calls == 1:
                raise KeyboardInterrupt
            return 0

    for call in (lambda c, t: c.kvd_checkpoint_residual(1, 2, t, T, 7), lambda c, t: c.kvd_decode_attention(0, 1, T, [4], [[(t, T, 64, 0, 5)]], 0.0, T)):
        with pytest.raises(KeyboardInterrupt):
            call(fake, Interrupted())
    assert not SEEN


def test_a_failing_call_and_a_closed_context_raise():
    c = B.Kvd.__new__(B.Kvd)
    c._lib, c._h, c._addr, c._keep = LIB, None, None, []
    with pytest.raises(B.KvdError):
        c.kvd_checkpoint_residual(0, 0, T, T, 1, stream=0)
    with pytest.raises(B.KvdError):
        c.kvd_decode_attention(0, 1, T, [0], [SEGS[0]], 0.0, T, stream=0)


def test_the_module_is_named_for_its_interpreter():
    """It is not built against the limited API: another interpreter in the same tree must not load it."""
    here = os.path.dirname(B.__file__)
    assert os.path.basename(B._calls.__file__) == "_kvdcall" + sysconfig.get_config_var("EXT_SUFFIX")
    assert not os.path.exists(os.path.join(here, "_kvdcall.so"))


def test_the_binding_works_without_the_module(fake, monkeypatch):
    """No C compiler or no Python headers: the library loads, and its calls are marshalled by ctypes."""
    code = ("import sys; sys.modules['paper_2603_19664_b200._kvdcall'] = None\n"
            "import paper_2603_19664_b200.binding as B\n"
            "lib = B.load(); c = B.Kvd.__new__(B.Kvd); c._lib, c._h, c._addr, c._keep = lib, None, None, []\n"
            "try: c.kvd_reset_sequence(0)\n"
            "except B.KvdError: print('refused by the library')\n")
    out = subprocess.run([sys.executable, "-c", code], cwd=os.path.dirname(os.path.dirname(B.__file__)), capture_output=True, text=True, check=True)
    assert "refused by the library" in out.stdout
    for call in CALLS:
        with monkeypatch.context() as m:
            m.setattr(B, "_calls", B._NoCalls())
            call(fake)
    assert len(SEEN) == len(CALLS)


def test_a_build_without_a_compiler_goes_on(monkeypatch, tmp_path, capsys):
    from paper_2603_19664_b200 import build as build_module

    monkeypatch.setattr(build_module, "CALLS", str(tmp_path / "_kvdcall.so"))
    monkeypatch.setenv("CC", str(tmp_path / "no-such-compiler"))
    assert os.path.exists(build_module.build())
    assert "ctypes" in capsys.readouterr().err
