"""Rules that the kernels and the host entry share with plain C++ (headers under csrc/), compiled here for the CPU."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_21135_b200", "csrc")


def _compile(tmp_path_factory, name, source):
    d = tmp_path_factory.mktemp(name)
    src, lib = str(d / "shim.cpp"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(source)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, "-o", lib, src])
    return ctypes.CDLL(lib)


@pytest.fixture(scope="module")
def topk(tmp_path_factory):
    """The rounds of the device's selection over the keys of one token."""
    lib = _compile(tmp_path_factory, "topk", """
        #include "topk_rule.h"
        extern "C" void select(const float* l, int E, int k, int* idx) {
            uint32_t key[256];
            for (int e = 0; e < E; ++e) key[e] = dyn::topk_key(l[e]);
            for (int j = 0; j < k; ++j) {
                int b = 0;
                for (int e = 1; e < E; ++e) if (key[e] > key[b]) b = e;
                idx[j] = b;
                key[b] = dyn::TOPK_TAKEN;
            }
        }
        extern "C" uint32_t key(float v) { return dyn::topk_key(v); }
        extern "C" float value(uint32_t k) { return dyn::topk_value(k); }
        """)
    lib.key.restype, lib.key.argtypes = ctypes.c_uint32, [ctypes.c_float]
    lib.value.restype, lib.value.argtypes = ctypes.c_float, [ctypes.c_uint32]

    def select(logits, k):
        lg = np.ascontiguousarray(logits, np.float32)
        idx = np.empty((lg.shape[0], k), np.int32)
        for t in range(lg.shape[0]):
            row = np.ascontiguousarray(lg[t])
            lib.select(row.ctypes.data_as(ctypes.c_void_p), lg.shape[1], k, idx[t].ctypes.data_as(ctypes.c_void_p))
        return idx

    return lib, select


def test_keys_order_the_logits(topk):
    lib, _ = topk
    v = np.array([-np.inf, -3e38, -1.5, -1e-45, 0.0, 1e-45, 2.0, 3e38, np.inf], np.float32)
    keys = [lib.key(x) for x in v]
    assert keys == sorted(set(keys))
    assert lib.key(-0.0) == lib.key(0.0)
    assert [lib.value(k) for k in keys] == v.tolist()
    for bits in (0x7fc00000, 0xffc00000, 0x7f800001, 0xffffffff):
        nan = np.array([bits], np.uint32).view(np.float32)[0]
        assert 0 < lib.key(nan) < keys[0] and np.isnan(lib.value(lib.key(nan)))


@pytest.mark.parametrize("E,k", [(1, 1), (8, 2), (8, 8), (40, 3), (64, 6), (256, 8)])
def test_selection_follows_the_oracle_and_stays_in_range(topk, E, k):
    _, select = topk
    rng = np.random.default_rng(E * 10 + k)
    lg = rng.standard_normal((40, E)).astype(np.float32)
    lg[5:10] = np.round(lg[5:10])                       # ties
    lg[10:20][rng.random((10, E)) < 0.7] = -np.inf      # masked experts, fewer left than k among them
    lg[20] = -np.inf
    lg[21] = 0.0
    lg[21, ::2] = -0.0
    assert np.array_equal(select(lg, k), oracle.route(lg, k)[0])
    nan = lg.copy()
    nan[22:30][rng.random((8, E)) < 0.7] = np.nan
    nan[30] = np.nan
    nan[10:20][rng.random((10, E)) < 0.3] = np.nan
    got = select(nan, k)
    assert got.min() >= 0 and got.max() < E
    assert all(len(set(row)) == k for row in got.tolist())
    for t in range(40):                                 # numbers first, among them the order of the numbers alone
        n = min(k, int(np.isfinite(nan[t]).sum()))
        assert np.array_equal(got[t, :n], oracle.route(np.where(np.isnan(nan[t]), -np.inf, nan[t])[None], k)[0][0, :n])


@pytest.fixture(scope="module")
def covers(tmp_path_factory):
    lib = _compile(tmp_path_factory, "covers", """
        #include "host_range.h"
        extern "C" bool covers(uint64_t start, uint64_t size, uint64_t p, uint64_t bytes) {
            return dyn::range_covers(start, size, p, bytes);
        }
        """)
    lib.covers.restype, lib.covers.argtypes = ctypes.c_bool, [ctypes.c_uint64] * 4
    return lib.covers


def test_a_buffer_has_to_lie_within_one_registration(covers):
    page = 4096
    first, second = (16 * page, 2 * page), (24 * page, 2 * page)      # pages 18 .. 23 between them are not registered
    assert covers(*first, 16 * page, 2 * page) and covers(*first, 17 * page, page) and covers(*first, 18 * page - 16, 16)
    assert not covers(*first, 18 * page - 16, 17)
    assert not covers(*first, 17 * page, second[0] + second[1] - 17 * page)   # both ends registered, the middle not
    assert not covers(*second, 17 * page, second[0] + second[1] - 17 * page)
    assert not covers(*first, 15 * page, 3 * page)
    assert not covers(0, 0, 16 * page, 1) and not covers(*first, 16 * page, 2 ** 64 - 1)
    top = 2 ** 64 - page
    assert covers(top, page - 1, top, page - 1) and not covers(top, page - 1, top + 8, page)


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    lib = _compile(tmp_path_factory, "layout", """
        #define __host__
        #define __device__
        #include "layout.cuh"
        extern "C" int scale_exp(int bits, int k) { return dyn::x_scale_exp(bits, k); }
        extern "C" int parts(int bits, int k) { return dyn::code_parts(bits, k); }
        extern "C" void loc(int bits, int r, int k, int part, int* out) {
            const dyn::CodeLoc l = dyn::code_loc(bits, r, k, part);
            out[0] = l.byte_off; out[1] = l.shift; out[2] = l.width; out[3] = l.lo;
        }
        """)

    def loc(bits, r, k, part):
        out = (ctypes.c_int * 4)()
        lib.loc(bits, r, k, part, out)
        return list(out)

    return lib, loc


@pytest.mark.parametrize("bits,bias,offsets", [(2, 4, [0, 2, 4, 6, 8, 0, 2, 4]), (3, 3, [0, 2, 4, 6] * 2), (4, 2, [0, 4] * 4),
                                               (6, 2, [0, 4] * 4), (8, 0, [0] * 8)])
def test_codes_lie_at_the_offsets_that_the_sums_are_exact_for(layout, bits, bias, offsets):
    """The activation of a code at bit offset o carries 2^(bias - o), and the tensor cores align their sums by the operands'
    exponents: the offsets decide the last bits of a result and how exact it is (3-bit codes at 0, 3 and 6: twice the error)."""
    lib, _ = layout
    for k in range(256):
        phi = 2 * (k >> 4 & 3) + (k >> 1 & 1)
        assert lib.scale_exp(bits, k) == bias - offsets[phi]


@pytest.mark.parametrize("bits", [2, 3, 4, 6, 8])
def test_every_bit_of_an_atom_belongs_to_one_code(layout, bits):
    lib, loc = layout
    taken = np.zeros(256 * bits * 8, np.int32)
    for r in range(16):
        for k in range(128):
            code = 0
            for part in range(lib.parts(bits, k)):
                off, shift, width, lo = loc(bits, r, k, part)
                assert off % 4 == 0 and 0 <= shift and shift + width <= 32
                taken[off * 8 + shift: off * 8 + shift + width] += 1
                assert code & (((1 << width) - 1) << lo) == 0
                code |= ((1 << width) - 1) << lo
            assert code == (1 << bits) - 1
    assert np.all(taken == 1)
