"""Host-side rules of the persistent grid solvers, compiled from their plain
C++ headers with the host compiler.  CPU only."""
import ctypes
import os
import subprocess
import threading
import time

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2510_08230_gb300", "csrc")


def _compile(tmp_path_factory, name, body):
    d = tmp_path_factory.mktemp(name)
    src, so = str(d / (name + ".cpp")), str(d / (name + ".so"))
    with open(src, "w") as f:
        f.write(body)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-pthread", "-I" + CSRC, src,
                    "-o", so], check=True, capture_output=True, text=True)
    return ctypes.CDLL(so)


@pytest.fixture(scope="module")
def limits(tmp_path_factory):
    lib = _compile(tmp_path_factory, "limits", '#include "grid_limits.h"\n'
                   'extern "C" int fits(long long k, long long s, long long v) '
                   '{ return gk::grid_offsets_fit(k, s, v); }\n')
    lib.fits.argtypes = [ctypes.c_longlong] * 3
    return lib.fits


@pytest.mark.parametrize("value_bytes", [8, 4, 2])
def test_offsets_of_values_and_columns_fit_32_bits(limits, value_bytes):
    """The byte offset of entry (K + 8) stride, one past the last that is
    formed, in the values and in the 4-byte columns: both sides of the limit,
    at the smallest and largest strides, and the 16-bit matrices whose values
    fit but whose columns do not."""
    entry = max(value_bytes, 4)
    for stride in (32, 64, 96, 1 << 12, 1 << 21, 4 << 20, (1 << 28) - 32):
        last = (2 ** 32 - 1) // (entry * stride)  # entries a row, 8 more among them
        for k in (last - 9, last - 8, last - 7, last):
            if k < 1:
                continue
            end = (k + 8) * stride * entry
            assert limits(k, stride, value_bytes) == (end < 2 ** 32), (k, stride)
    assert not limits(601, 1 << 21, value_bytes)  # 609 * 2^21 * 2 < 2^32 < 601 * 2^21 * 4
    assert not limits(270, 4 << 20, value_bytes)
    assert limits(7, 1 << 21, value_bytes)


@pytest.fixture(scope="module")
def seats(tmp_path_factory):
    lib = _compile(tmp_path_factory, "seats", '#include "grid_seats.h"\n'
                   'static gk::SeatPools pools;\n'
                   'extern "C" float take(int d, int n, int cap) { return pools.of(d).take(n, cap); }\n'
                   'extern "C" void give(int d, int n) { pools.of(d).give(n); }\n')
    lib.take.restype = ctypes.c_float
    return lib


def test_seats_are_a_device_s_own(seats):
    """A device whose seats are all taken does not keep another one's solves
    waiting."""
    assert seats.take(0, 304, 304) == 0.0
    done = threading.Event()
    t = threading.Thread(target=lambda: (seats.take(1, 304, 304), seats.take(2, 100, 264),
                                         done.set()), daemon=True)
    t.start()
    assert done.wait(5)
    for d, n in ((0, 304), (1, 304), (2, 100)):
        seats.give(d, n)


def test_seats_in_order_of_arrival(seats):
    """On one device a large request is not overtaken by later small ones,
    and the wait it reports is the time it queued."""
    assert seats.take(3, 200, 304) == 0.0
    order, waited = [], {}

    def ask(name, n):
        waited[name] = seats.take(3, n, 304)
        order.append(name)
        seats.give(3, n)

    ts = []
    for name, n in (("large", 304), ("small", 50)):
        ts.append(threading.Thread(target=ask, args=(name, n), daemon=True))
        ts[-1].start()
        time.sleep(0.2)
    assert order == []
    seats.give(3, 200)
    for t in ts:
        t.join(5)
    assert order == ["large", "small"]
    assert waited["large"] >= 300 and waited["small"] >= 150
