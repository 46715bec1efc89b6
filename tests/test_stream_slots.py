"""The streams' scratch slots (stream_slots.h), compiled with the host compiler.
CPU only."""
import ctypes
import os
import subprocess
import threading

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2510_08230_gb300", "csrc")


def test_first_streams_keep_a_slot_each(tmp_path):
    src, so = str(tmp_path / "slots.cpp"), str(tmp_path / "slots.so")
    with open(src, "w") as f:
        f.write('#include "stream_slots.h"\n'
                'extern "C" void* slots() { return new gk::StreamSlots; }\n'
                'extern "C" int of(void* s, unsigned long long id) '
                '{ return static_cast<gk::StreamSlots*>(s)->of(id); }\n')
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + CSRC, src, "-o", so],
                   check=True, capture_output=True, text=True)
    lib = ctypes.CDLL(so)
    lib.slots.restype = ctypes.c_void_p
    lib.of.argtypes = [ctypes.c_void_p, ctypes.c_ulonglong]
    s = lib.slots()
    ids = [0, 7, 2 ** 63, 3, 4, 5]  # 0 is an id like any other
    got = [lib.of(s, i) for i in ids]
    assert got == [0, 1, 2, 3, -1, -1]
    assert [lib.of(s, i) for i in ids] == got  # kept
    for _ in range(50):  # streams that ask at once never share one
        s, out = lib.slots(), {}
        go = threading.Barrier(8)

        def ask(i):
            go.wait()
            out[i] = [lib.of(s, i) for _ in range(3)]

        ts = [threading.Thread(target=ask, args=(i,)) for i in range(8)]
        [t.start() for t in ts]
        [t.join() for t in ts]
        assert all(len(set(v)) == 1 for v in out.values())
        assert sorted(v[0] for v in out.values()) == [-1] * 4 + [0, 1, 2, 3]
