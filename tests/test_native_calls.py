"""The binding's native calls (csrc/py_calls.cpp): what an entry point receives is what it receives through ctypes, for every entry point
that is called natively and every form of an argument; refusals are the ones of Python and ctypes."""
import ctypes
import gc
import sys
import threading

import numpy as np
import pytest
import torch

from paper_2609_33503_b200 import binding as B

NATIVE = B._native()
KINDS = {n: a.replace(" ", "") for n, (_, a) in B._SIGNATURES.items()}


def _recorder(name):
    """A C function of the entry point's type that notes its arguments, and its two callers: bound and through ctypes."""
    seen = []
    types = [B._CTYPE[c] for c in KINDS[name]]

    def note(*args):
        seen.append(tuple(a or 0 if c == "p" else a for c, a in zip(KINDS[name], args)))
        return 5

    proto = ctypes.CFUNCTYPE(ctypes.c_int32, *types)
    callback = proto(note)
    address = ctypes.cast(callback, ctypes.c_void_p).value
    plain = proto(address)
    return seen, NATIVE.bind(name, address, plain), plain, callback


NAMES = [n for n in B.ENTRY_POINTS if NATIVE.bind(n, 0, None) is not None]         # the rest goes through ctypes alone


def test_the_calls_of_a_pass_are_native():
    assert {"relaxkv_select_topk", "relaxkv_build_active_sets", "relaxkv_sparse_ctx_attention", "relaxkv_scatter_kv"} <= set(NAMES)


@pytest.mark.parametrize("name", NAMES)
def test_an_entry_point_receives_the_same(name):
    seen, bound, plain, keep = _recorder(name)
    value = {"p": 0x7f0012345670, "i": 70000, "l": 1 << 40, "z": (1 << 33) + 5, "f": 0.15625, "d": 0.1}
    rows = [[value[c] for c in KINDS[name]], [None if c == "p" else 1 if c in "fd" else -3 if c in "il" else 0 for c in KINDS[name]],
            [(1 << 40) + 7 if c in "pilz" else float("inf") for c in KINDS[name]], [True if c in "il" else value[c] for c in KINDS[name]]]
    for row in rows:
        assert bound(*row) == plain(*row) == 5
        assert seen[-1] == seen[-2]
    for bad in ([], rows[0][:-1], [object()] + rows[0][1:], [1.5] + rows[0][1:]):
        with pytest.raises((TypeError, ctypes.ArgumentError)) as by_ctypes:
            plain(*bad)
        with pytest.raises(by_ctypes.type):
            bound(*bad)
    i = ctypes.c_int32(9)                                        # a reference goes through ctypes
    if KINDS[name][0] == "p":
        assert bound(ctypes.byref(i), *rows[0][1:]) == 5 and seen[-1][0] == ctypes.addressof(i)


@pytest.mark.parametrize("xs", [[], [7], [1, -2, 2**31 - 1, -2**31], (3, 4), np.arange(5), np.array([3], dtype=np.int64), torch.tensor([5, 6]),
                                [np.int32(4), torch.tensor(9), True, "12", 3.7], range(40), list(range(65)), list(range(300)), [2**32 + 5]])
def test_host_integers_are_the_array_ctypes_makes(xs):
    got, = NATIVE.marshal("h", xs)
    assert got == bytes(B._i32(xs))
    held, = NATIVE.marshal("h", xs)
    assert ctypes.string_at(ctypes.c_char_p(held), len(held)) == got if b"\0" not in got else len(held) == 4 * len(xs)


def test_arguments_by_code():
    t, s = torch.zeros(8), B.Shape(8, 2, 128, [64])
    assert NATIVE.marshal("ps.hp.", t, s.c, 3, [2], None, 1.5) == (t.data_ptr(), ctypes.addressof(s.c), 3, b"\2\0\0\0", None, 1.5)
    assert NATIVE.marshal("h", None) == (None,)
    off = B.Offsets(t, 2)
    assert NATIVE.marshal("p", off) == (t.data_ptr() + 8,)
    for codes, args, error in (("p", (5,), AttributeError), ("p", (2.5,), AttributeError), ("h", (5,), TypeError), ("h", (["x"],), ValueError),
                               ("h", ([None],), TypeError), ("h", (iter([1]),), TypeError), ("s", (None,), TypeError), ("s", (7,), TypeError),
                               ("pp", (t,), TypeError), ("", (t,), TypeError), ("q", (t,), TypeError)):
        with pytest.raises(error):
            NATIVE.marshal(codes, *args)
    with pytest.raises(TypeError):
        NATIVE.marshal()


def test_a_list_that_shrinks_while_it_is_read_is_refused():
    xs = [1, None, 3, 4]

    class Shrinks:
        def __int__(self):
            del xs[1:]
            return 2
    xs[1] = Shrinks()
    with pytest.raises(RuntimeError, match="size"):
        NATIVE.marshal("h", xs)


def test_references_and_threads():
    """No argument is kept or lost over many calls, and calls of several threads do not disturb each other (the lock is free meanwhile)."""
    seen, bound, plain, keep = _recorder("relaxkv_select_topk")
    t, s, k = torch.zeros(8), B.Shape(8, 2, 128, [64]), [1 << 20]
    before = [sys.getrefcount(x) for x in (t, s.c, k, None, plain)]

    def work():
        for _ in range(2000):
            assert bound(*NATIVE.marshal("s.hppp.", s.c, 1, k, t, None, t, 0)) == 5
    threads = [threading.Thread(target=work) for _ in range(4)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert len(seen) == 8000 and {(r[0], r[1], r[3], r[4], r[5]) for r in seen} == {(ctypes.addressof(s.c), 1, t.data_ptr(), 0, t.data_ptr())}
    del threads
    gc.collect()
    after = [sys.getrefcount(x) for x in (t, s.c, k, None, plain)]
    assert before[:3] == after[:3] and abs(after[4] - before[4]) <= 1
    entry_refs = sys.getrefcount(plain)
    del bound
    assert sys.getrefcount(plain) == entry_refs - 1


def test_the_calls_name_nothing_newer_than_python_3_10():
    """The member descriptors go by the names of structmember.h (their Py_ forms came with 3.12), and nothing else of the C API that came with
    3.11 to 3.14 is named."""
    import os
    import re
    from paper_2609_33503_b200 import build
    with open(os.path.join(build.CSRC, "py_calls.cpp")) as f:
        words = set(re.findall(r"\w+", re.sub(r"//.*", "", f.read())))
    newer = {w for w in words if re.fullmatch(r"Py_(T_\w+|READONLY|RELATIVE_OFFSET|AUDIT_READ|mod_gil|MOD_GIL_\w+|tp_vectorcall)", w)}
    newer |= words & {"PyType_GetName", "PyType_GetQualName", "PyType_FromMetaclass", "PyErr_GetRaisedException", "PyErr_SetRaisedException", "PyObject_GetOptionalAttr",
                      "PyLong_AsInt", "PyLong_AsNativeBytes", "PyList_GetItemRef", "PyDict_GetItemRef", "PyUnicode_EqualToUTF8", "PyBuffer_ReleaseBuffer",
                      "Py_HashPointer", "PyWeakref_GetRef", "PyUnstable_Long_IsCompact", "PyImport_AddModuleRef"}
    assert not newer and "structmember" in words
