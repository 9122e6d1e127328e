"""The tagged doubles the blocks of the FP64 tridiagonalisation exchange (csrc/tri_packet.h), compiled
for the host: the value comes back with all its bits, whatever the tag."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2303_00689_gb300 import build

SOURCE = """
#include "tri_packet.h"
extern "C" void through(long n, const unsigned long long* x, unsigned long long tag, unsigned long long* packet,
                        unsigned long long* y) {
  for (long i = 0; i < n; ++i) {
    packet[i] = kx::packet_encode(x[i], tag ? kx::kPacketTag : 0);
    y[i] = kx::packet_decode(packet[i]);
  }
}
"""


@pytest.fixture(scope="module")
def through(tmp_path_factory):
    d = tmp_path_factory.mktemp("packet")
    (d / "packet.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I", build.SRC, str(d / "packet.cpp"), "-o",
                    str(d / "packet.so")], check=True)
    fn = ctypes.CDLL(os.path.join(str(d), "packet.so")).through

    def call(x, tag):
        x = np.ascontiguousarray(x, dtype=np.float64)
        packet, y = np.empty(x.shape, np.uint64), np.empty_like(x)
        fn(ctypes.c_long(x.size), x.ctypes.data_as(ctypes.c_void_p), ctypes.c_ulonglong(tag),
           packet.ctypes.data_as(ctypes.c_void_p), y.ctypes.data_as(ctypes.c_void_p))
        return packet, y
    return call


@pytest.mark.parametrize("tag", [0, 1])
def test_every_bit_of_a_sum_comes_back(through, tag):
    rng = np.random.default_rng(0)
    e = np.concatenate([rng.integers(-766, 257, 20000), [-766, -766, 256, 256, 0]])
    x = np.ldexp(1.0 + rng.integers(0, 2 ** 52, e.size) * 2.0 ** -52, e) * rng.choice([-1.0, 1.0], e.size)
    packet, y = through(x, tag)
    assert np.array_equal(x.view(np.uint64), y.view(np.uint64))
    assert ((packet >> np.uint64(62) & np.uint64(1)) == tag).all()


@pytest.mark.parametrize("tag", [0, 1])
def test_values_outside_the_range_of_sums(through, tag):
    exact = np.array([0.0, -0.0, np.inf, -np.inf, 2.0 ** 257, -(2.0 ** 1023), 2.0 ** -767, 2.0 ** -1022])
    packet, y = through(exact, tag)
    assert np.array_equal(exact.view(np.uint64), y.view(np.uint64))
    assert ((packet >> np.uint64(62) & np.uint64(1)) == tag).all()
    assert np.isnan(through(np.array([np.nan]), tag)[1]).all()
    rng = np.random.default_rng(1)
    x = np.ldexp(1.0 + rng.random(20000), np.concatenate([rng.integers(257, 1023, 10000), rng.integers(-1022, -766, 10000)]))
    assert (np.abs(through(x, tag)[1] / x - 1.0) <= 2.0 ** -41).all()
