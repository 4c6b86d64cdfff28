"""The FP64 path's fixed-point arithmetic (su2_fixed.cuh), compiled for the
host: conversion of links and its range checks, sums of products, and the
elementary functions of a draw, against rational or extended arithmetic."""
import ctypes as C
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1010_4834_gb300", "csrc")
UNIT = Fraction(1, 1 << 58)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fixed") / "fixed_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fwrapv", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "fixed_host.cpp"), "-o", so], check=True)
    L = C.CDLL(so)
    p64 = C.POINTER(C.c_int64)
    dp = C.POINTER(C.c_double)
    L.fixed_link.argtypes = [dp, C.c_int, p64]
    L.fixed_any_link.argtypes = L.fixed_link.argtypes
    L.fixed_any.argtypes, L.fixed_any.restype = [C.c_double], C.c_int64
    L.fixed_triples.argtypes = [dp, dp, dp, C.c_int, p64]
    L.fixed_neg_log.argtypes, L.fixed_neg_log.restype = [C.c_uint32], C.c_int64
    L.fixed_cos2.argtypes, L.fixed_cos2.restype = [C.c_uint32], C.c_uint64
    L.fixed_sincos.argtypes = [C.c_uint32, p64]
    assert L.fixed_frac() == 58
    return L


def _link(lib, v, conj=0):
    a, out = np.array(v, np.float64), np.zeros(4, np.int64)
    ok = lib.fixed_link(a.ctypes.data_as(C.POINTER(C.c_double)), conj, out.ctypes.data_as(C.POINTER(C.c_int64)))
    return ok, out


def _units(rng, n):
    q = rng.standard_normal((n, 4))
    return q / np.linalg.norm(q, axis=1, keepdims=True)


def test_links_convert_within_one_unit(lib):
    rng = np.random.default_rng(1)
    q = _units(rng, 2000)
    q[:400] *= 1 + 0.05 * rng.uniform(-1, 1, (400, 1))
    # components down to the smallest the conversion takes, and exact powers
    # of two, whose significand is zero
    q[400:800, 1] = rng.choice([-1, 1], 400) * np.exp2(rng.uniform(-30.99, -8, 400))
    q[800:832, 2] = -np.exp2(-np.arange(1, 33.0).clip(1, 31))
    q[400:832] /= np.linalg.norm(q[400:832], axis=1, keepdims=True)
    q[832] = [0.5, -0.5, 0.5, -0.5]
    q[833] = [-1.0, 2.0 ** -31, -2.0 ** -31, 2.0 ** -30]
    q[834] = [np.nextafter(1.0, 2.0), -2.0 ** -20, 2.0 ** -20, 2.0 ** -20]
    for v in q:
        for conj in (0, 1):
            ok, got = _link(lib, v, conj)
            if np.abs(v).min() < 2.0 ** -31:
                continue
            assert ok, v
            sign = [1] + [-1 if conj else 1] * 3
            for c in range(4):
                assert abs(int(got[c]) * UNIT - sign[c] * Fraction(float(v[c]))) <= UNIT


@pytest.mark.parametrize("v", [[1.0, 0.0, 0.0, 0.0], [2.0, 0.1, 0.1, 0.1], [-4.0, 0.1, 0.1, 0.1], [0.4, 0.4, 0.4, 0.4],
                               [0.6, 0.6, 0.6, 0.6], [1e300, 0.5, 0.5, 0.5], [np.inf, 0.5, 0.5, 0.5],
                               [np.nan, 0.5, 0.5, 0.5], [0.9, 2.0 ** -32, 0.3, 0.3], [1e-310, 0.5, 0.5, 0.7],
                               [1.07, 0.01, 0.01, 0.01], [0.92, 0.01, 0.01, 0.01], [-1.9, 1.9, 1.9, -1.9],
                               [0.0, 0.0, 0.0, 0.0], [-np.inf, 1.0, 1.0, 1.0], [2.0 ** 32, 0.5, 0.5, 0.5]])
def test_links_out_of_range_are_flagged(lib, v):
    for k in range(4):
        assert not _link(lib, np.roll(v, k))[0]
        assert not _link(lib, -np.roll(v, k), 1)[0]


def test_links_with_components_of_any_size_convert(lib):
    # zeros, tiny and subnormal components: refused by the first conversion, taken
    # by the second, within one unit of 2^-58
    rng = np.random.default_rng(5)
    q = _units(rng, 500)
    q[:, 1] = rng.choice([-1, 1], 500) * np.exp2(rng.uniform(-80, -32, 500))
    q[::5, 2] = rng.choice([0.0, -0.0, 5e-324], 100)
    q[:400] /= np.linalg.norm(q[:400], axis=1, keepdims=True)
    axes = np.concatenate([np.eye(4), -np.eye(4)])
    dp, ip = C.POINTER(C.c_double), C.POINTER(C.c_int64)
    for v in np.concatenate([q, axes]):
        for conj in (0, 1):
            out = np.zeros(4, np.int64)
            inside = abs(np.sum(v * v) - 1) < 0.124
            assert not _link(lib, v, conj)[0]
            assert lib.fixed_any_link(v.ctypes.data_as(dp), conj, out.ctypes.data_as(ip)) or not inside
            for c in range(4):
                assert abs(int(out[c]) * UNIT - (-1 if conj and c else 1) * Fraction(float(v[c]))) <= UNIT
    for v in ([2.0, 0.0, 0.0, 0.0], [np.inf, 0, 0, 0], [np.nan, 0, 0, 0], [0.0] * 4, [0.9, 0, 0, 0], [1.07, 0, 0, 0], [1e300, 0, 0, 0]):
        for k in range(4):
            v_ = np.roll(np.array(v, np.float64), k)
            assert not lib.fixed_any_link(v_.ctypes.data_as(dp), 0, out.ctypes.data_as(ip))


def test_any_component_converts_within_one_unit(lib):
    rng = np.random.default_rng(2)
    v = rng.choice([-1, 1], 4000) * np.exp2(rng.uniform(-70, 0.99, 4000))
    for x in np.concatenate([v, [0.0, -0.0, 1.0, -1.0, 5e-324, 2.0 ** -58, -2.0 ** -59, 1.9999999999999998]]):
        assert abs(lib.fixed_any(float(x)) * UNIT - Fraction(float(x))) <= UNIT


def test_sums_of_products_are_closer_than_fp64(lib):
    # six products of three links, as a staple sum adds them: random links, and
    # links that all but align (the largest sums)
    rng = np.random.default_rng(3)

    def mul(a, b):
        return [a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3], a[0] * b[1] + a[1] * b[0] - a[2] * b[3] + a[3] * b[2],
                a[0] * b[2] + a[2] * b[0] - a[3] * b[1] + a[1] * b[3], a[0] * b[3] + a[3] * b[0] - a[1] * b[2] + a[2] * b[1]]

    dp = C.POINTER(C.c_double)
    worst, off, off64 = 0.0, [], []
    for trial in range(300):
        q = _units(rng, 18)
        if trial % 3 == 1:
            q = np.array([1, 1e-3, 1e-3, 1e-3]) + 1e-3 * rng.standard_normal((18, 4))
            q *= 1.0606 / np.linalg.norm(q, axis=1, keepdims=True)     # the largest norm taken
            q *= rng.choice([-1, 1])
        elif trial % 3 == 2:
            q = np.full((18, 4), 0.53) * rng.choice([-1, 1], (18, 4))
        a, b, c = (np.ascontiguousarray(q[i::3]) for i in range(3))
        out = np.zeros(4, np.int64)
        assert lib.fixed_triples(a.ctypes.data_as(dp), b.ctypes.data_as(dp), c.ctypes.data_as(dp), 6,
                                 out.ctypes.data_as(C.POINTER(C.c_int64)))
        ref = [Fraction(0)] * 4
        f64 = np.zeros(4)
        for i in range(6):
            fa, fb, fc = ([Fraction(float(x)) for x in v[i]] for v in (a, b, c))
            ref = [s + t for s, t in zip(ref, mul(mul(fa, fb), fc))]
            f64 += mul(mul(a[i], b[i]), c[i])
        e = max(abs(int(out[k]) * UNIT - ref[k]) for k in range(4))
        worst = max(worst, float(e))
        off += [float(int(out[k]) * UNIT - ref[k]) for k in range(4)]
        off64 += [float(Fraction(float(f64[k])) - ref[k]) for k in range(4)]
    # a product of two links: 4 n (conversions) + 4 (low limbs left out) + 4 (rounding)
    # units of 2^-58, n = 1.0607; times a third link 2 n times that, + 2 n^2 + 2; six
    # terms and the sum's rounding
    n = 1.0607
    assert worst < (6 * (2 * n * (4 * n + 8) + 2 * n * n + 2) + 4) * float(UNIT)
    assert np.sqrt(np.mean(np.square(off))) < 0.25 * np.sqrt(np.mean(np.square(off64)))


def test_log_table_entries_are_aligned_for_their_16_byte_load(lib):
    # the device reads an entry (two 8-byte words) by one 16-byte load
    assert lib.fixed_log_entry_size() == 16
    assert lib.fixed_log_entry_alignment() == 16


def _draws():
    rng = np.random.default_rng(4)
    edge = [0, 1, 2, 3, (1 << 32) - 1, (1 << 32) - 2, (1 << 31) - 1, 1 << 31, (1 << 30) - 1, 1 << 30, 3 << 30, (3 << 30) - 1,
            1 << 29, (1 << 29) - 1]
    near = [((1 << 32) // 128 * i + d) & 0xFFFFFFFF for i in range(128) for d in (-1, 0, 1)]
    return [int(x) for x in np.concatenate([edge, near, rng.integers(0, 1 << 32, 20000), 1 << rng.integers(0, 32, 64)])]


def test_logarithm_and_angles_of_a_draw(lib):
    ld = np.longdouble
    if np.finfo(ld).nmant < 63:
        pytest.skip("long double has no more bits than double here")
    pi = ld("3.14159265358979323846264338327950288")
    x = np.array(_draws(), np.int64)
    u = (x.astype(ld) * 2 + 1) / ld(2) ** 33
    sc = np.zeros(2, np.int64)
    log, cos2, sn, cs = [], [], [], []
    for v in x:
        log.append(lib.fixed_neg_log(int(v)))
        cos2.append(lib.fixed_cos2(int(v)))
        lib.fixed_sincos(int(v), sc.ctypes.data_as(C.POINTER(C.c_int64)))
        sn.append(int(sc[0]))
        cs.append(int(sc[1]))
    log = np.array(log, np.int64).astype(ld) / ld(2) ** 58
    cos2 = np.array(cos2, np.uint64).astype(ld) / ld(2) ** 63
    sn, cs = (np.array(v, np.int64).astype(ld) / ld(2) ** 62 for v in (sn, cs))
    # absolute errors; the reference's own, from 64 bits or more, is below 2^-59
    # for the logarithm (values to 23) and 2^-61 for the angles
    # ln 2 rounded to 2^-58 counts up to 33 times: half a unit for each factor 2
    assert (np.abs(log + np.log(u)) / (1 - np.log(u))).max() < 2.0 ** -57
    q = np.floor(u * 4)
    a = (u * 4 - q - ld(0.5)) * (pi / 2)          # angle from the quadrant's middle, exact reduction
    m = (q + ld(0.5)) * (pi / 2)
    c, s = np.cos(m) * np.cos(a) - np.sin(m) * np.sin(a), np.sin(m) * np.cos(a) + np.cos(m) * np.sin(a)
    assert np.abs(cs - c).max() < 2.0 ** -59
    assert np.abs(sn - s).max() < 2.0 ** -59
    assert np.abs(cos2 - c * c).max() < 2.0 ** -59
