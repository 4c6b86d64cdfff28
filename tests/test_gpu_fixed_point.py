"""The FP64 kernels in fixed point, and their FP64 path for links outside the
fixed-point range; the small-lattice substep at the edges of its range; the
temporal-gauge Wilson kernel on time extents of every remainder.  FP64 against
the oracle at 1e-12 (values up to 6 and about a hundred operations of 2^-53
each leave 1e-14; loops up to W = |U|^64 on scaled links are compared relative to
their size)."""
import ctypes as C
import os
import subprocess
import time

import numpy as np
import pytest

import oracle
from paper_1010_4834_gb300 import Batch, Lattice, inputs
from paper_1010_4834_gb300.build import ARCH, CSRC, INCLUDE, nvcc_path
from test_gpu_parity import MTOL, as_stored, substep_compare

pytestmark = pytest.mark.gpu

DIMS = (4, 6, 8, 4)


def _field(kind, dims=DIMS, seed=3):
    """Links in and out of the fixed-point range (components 0 or below 2^-31,
    norms off one), everywhere or on some links only."""
    U = inputs.random_field(dims, seed)
    rng = np.random.default_rng(seed)
    some = rng.random(U.shape[:2]) < 0.1
    if kind == "abelian":
        return inputs.abelian_field(inputs.abelian_angles(dims, seed))
    if kind == "cold":
        return np.broadcast_to(np.array([1.0, 0.0, 0.0, 0.0]), U.shape).copy()
    if kind == "tiny":                    # one component below the range, of either sign
        U[some, 1] = rng.choice([-1, 1], some.sum()) * np.exp2(rng.uniform(-60, -30, some.sum()))
        return U / np.linalg.norm(U, axis=-1, keepdims=True)
    if kind == "edge":                    # norms at the edge of the range
        return U * (1 + 0.06 * rng.uniform(-1, 1, U.shape[:2]))[..., None]
    if kind == "scaled":
        U[some] *= 1.3
    return U


KINDS = ["random", "abelian", "cold", "tiny", "edge", "scaled"]


@pytest.mark.parametrize("kind", KINDS)
def test_fp64_substep_on_any_links(kind):
    U = _field(kind)
    for mu, p in ((0, 0), (1, 1), (2, 0), (3, 1)):
        lat = Lattice(DIMS, 2.3, seed=7, prec="f64")
        lat.set_links(U)
        lat.substep(mu, p, 5)
        ref = U.copy()
        oracle.substep(list(DIMS), ref, oracle.chain(2.3, seed=7), 5, mu, p)
        assert (ref != U).any()
        np.testing.assert_allclose(lat.get_links(), ref, atol=1e-12, rtol=0)


@pytest.mark.parametrize("beta,sampler,tries", [(0.02, "kp", 64), (0.3, "kp", 64), (0.08, "kp", 2), (0.3, "creutz", 64),
                                                (2.4, "creutz", 3), (2.4, "kp", 1), (40.0, "kp", 64), (300.0, "kp", 3)])
def test_fp64_draws_over_couplings(beta, sampler, tries):
    # small beta: alpha on both sides of the value below which a trial runs in FP64
    substep_compare(DIMS, "f64", beta, _field("random"), 1, 0, sweep=2, sampler=sampler, max_tries=tries)


@pytest.mark.parametrize("kind", KINDS)
def test_fp64_overrelaxation_smearing_and_measurements_on_any_links(kind):
    U = _field(kind)
    d = list(DIMS)
    lat = Lattice(DIMS, 2.0, prec="f64")
    lat.set_links(U)
    np.testing.assert_allclose(lat.plaquette(), oracle.plaquette(d, U), atol=2e-12, rtol=0)
    assert abs(lat.polyakov() - oracle.polyakov(d, U)) < 2e-12
    np.testing.assert_allclose(lat.wilson_loops(4, 4), oracle.wilson_loops(d, U, 4, 4), atol=2e-12, rtol=1e-11)
    lat.ape_smear(0.6, 2)
    S = oracle.ape_smear(d, U.copy(), 0.6, 2)
    np.testing.assert_allclose(lat.wilson_loops(4, 4, smeared=True), oracle.wilson_loops(d, S, 4, 4), atol=2e-12, rtol=1e-11)
    lat.overrelax(1)
    for mu in range(4):
        for p in range(2):
            oracle.overrelax_substep(d, U, mu, p)
    # U' = W U^+ W keeps |U|; a staple sum that all but vanishes has no direction
    np.testing.assert_allclose(lat.get_links(), U, atol=1e-11, rtol=0)


@pytest.mark.parametrize("prec,dims", [("f64", (32, 16, 38, 4)), ("f64", (34, 16, 38, 4)), ("f64", (2, 2, 2, 2)),
                                       ("f64", (6, 2, 2, 10)), ("f64", (8, 8, 8, 18)), ("f64", (8, 8, 8, 20)),
                                       ("f64", (16, 16, 8, 18)), ("f64", (16, 16, 16, 10)), ("f32", (32, 32, 38, 4)), ("f32", (34, 32, 38, 4)),
                                       ("f32", (2, 2, 2, 2)), ("f32", (6, 10, 2, 14)), ("f16q", (32, 32, 38, 4)),
                                       ("f16q", (10, 6, 2, 4))])
@pytest.mark.parametrize("sampler,tries,nor", [("kp", 64, 0), ("creutz", 64, 1), ("kp", 2, 2)])
def test_small_lattice_substeps_leave_the_other_kernels_links(prec, dims, sampler, tries, nor):
    # at and just past the largest lattice of the small kernel (152 SMs) and of
    # its FP64 forms with eight and two lanes a link, and at volumes that do not
    # fill a block or a warp: direct launches, replayed graphs and measured
    # sweeps, against the batched kernel or (below FP64, where batches and
    # single lattices may round products differently) the fused parity pair
    a = Lattice(dims, 2.2, seed=9, start="hot", prec=prec)
    m = Lattice(dims, 2.2, seed=9, start="hot", prec=prec)
    if prec == "f64":
        b = Batch([dims], [2.2], seed=9, start="hot", prec=prec)
    else:
        b = Lattice(dims, 2.2, seed=9, start="hot", prec=prec)
        b.set_schedule("pair")
    for x in (a, m, b):
        x.set_options(tries, sampler)
        x.set_overrelax(nor)
    a.sweep(3)
    a.sweep(16)
    m.sweep_measure(2)
    hist = m.sweep_measure(17)
    b.sweep(19)
    got = a.get_links()
    assert np.array_equal(got, b.get_links(0) if prec == "f64" else b.get_links())
    assert np.array_equal(got, m.get_links())
    np.testing.assert_allclose(hist[-1, :3], a.plaquette(), atol=MTOL[prec], rtol=0)
    assert abs(hist[-1, 3] - a.polyakov()) < 1e-12
    if prec == "f64":
        np.testing.assert_allclose(b.plaquette()[0], a.plaquette(), atol=1e-13, rtol=0)
        np.testing.assert_allclose(b.polyakov()[0], a.polyakov(), atol=1e-13, rtol=0)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("nt", [2, 4, 6, 10, 12, 14, 18, 20, 24, 28, 36, 40, 46, 56, 62])
def test_wilson_loops_on_every_remainder_of_the_time_extent(nt, prec):
    dims = (6, 4, 6, nt)
    U = inputs.random_field(dims, 31)
    ref = oracle.wilson_loops(list(dims), as_stored(U, prec), 4, min(nt, 16))
    lat = Lattice(dims, 2.0, prec=prec)
    lat.set_links(U)
    for rmax, tmax in ((4, min(nt, 16)), (3, min(nt, 5)), (1, 1)):
        np.testing.assert_allclose(lat.wilson_loops(rmax, tmax), ref[:rmax, :tmax], atol=MTOL[prec] * 5, rtol=0)


@pytest.mark.parametrize("prec", ["f32", "f16q"])
@pytest.mark.parametrize("nt", [4, 8, 10, 20, 24, 40])
def test_wilson_loops_on_both_sides_of_the_time_outer_kernels_range(nt, prec):
    # planes just wider than 32 columns: the kernel changes with R and T
    dims = (34, 6, 6, nt)
    U = inputs.random_field(dims, 32)
    ref = oracle.wilson_loops(list(dims), as_stored(U, prec), 6, min(nt, 6))
    lat = Lattice(dims, 2.0, prec=prec)
    lat.set_links(U)
    for rmax in (1, 2, 3, 4, 5, 6):
        for tmax in range(1, min(nt, 6) + 1):
            np.testing.assert_allclose(lat.wilson_loops(rmax, tmax), ref[:rmax, :tmax], atol=MTOL[prec] * 5, rtol=0)


def _off_unit(nt, off, where, dims=(6, 4, 6)):
    """Ordered links (large loops) whose norms differ by up to off from one, link
    by link, up and down in the two halves of the lattice, or all alike: a loop
    carries its own links' norms."""
    dims = (*dims, nt)
    rng = np.random.default_rng(nt)
    U = np.array([1.0, 0.0, 0.0, 0.0]) + 0.3 * inputs.random_field(dims, 5)
    U /= np.linalg.norm(U, axis=-1, keepdims=True)
    w = {"links": rng.uniform(-1, 1, U.shape[:2]), "halves": np.sign(np.arange(U.shape[0]) - U.shape[0] // 2 + 0.5)[:, None],
         "all": np.ones((1, 1))}[where]
    return dims, U * (1 + off * w)[..., None]


@pytest.mark.parametrize("nt", [12, 16, 24])
@pytest.mark.parametrize("off", [1e-6, 1e-5, 1e-2])
@pytest.mark.parametrize("where", ["links", "halves", "all"])
def test_fp32_wilson_loops_on_links_off_unit_norm(nt, off, where):
    # below 2^-18 in |U|^2 the norms of a loop's 2 T time links are dropped: 24 x 1e-6
    # where all links are off alike, in the mean over loops much less where they
    # differ; 5e-6 for FP32's own rounding
    atol = 5e-6 + (24 * off if where == "all" and off < 1.9e-6 else 0.0)
    dims, U = _off_unit(nt, off, where)
    lat = Lattice(dims, 2.0, prec="f32")
    lat.set_links(U)
    ref = oracle.wilson_loops(list(dims), as_stored(U, "f32"), 4, 12)
    for _ in range(2):
        np.testing.assert_allclose(lat.wilson_loops(4, 12), ref, atol=atol, rtol=0)


@pytest.mark.parametrize("nt", [12, 16, 24])
@pytest.mark.parametrize("off", [1e-15, 1e-13, 1e-11, 1e-9, 1e-7, 1e-4])
@pytest.mark.parametrize("where", ["links", "halves", "all"])
def test_fp64_wilson_loops_on_links_off_unit_norm(nt, off, where):
    # 32 links of a loop, four products each of 2^-53
    dims, U = _off_unit(nt, off, where)
    lat = Lattice(dims, 2.0, prec="f64")
    lat.set_links(U)
    ref = oracle.wilson_loops(list(dims), U, 4, 12)
    for _ in range(2):
        np.testing.assert_allclose(lat.wilson_loops(4, 12), ref, atol=1e-14, rtol=0)


def _seconds(call, n=10):
    times = []
    for _ in range(n):
        t0 = time.perf_counter()
        call()
        times.append(time.perf_counter() - t0)
    return min(times)


def test_fp64_wilson_loops_of_a_store_rounded_to_fp32_stay_in_temporal_gauge():
    # 2.5 times a chain's links' time; 17 times where the loops are multiplied out
    dims = (16, 16, 16, 16)
    lat = Lattice(dims, 2.4, seed=1, start="hot", prec="f64")
    unit = _seconds(lambda: lat.wilson_loops(8, 8))
    lat.set_links(as_stored(lat.get_links(), "f32"))
    assert _seconds(lambda: lat.wilson_loops(8, 8)) < 6 * unit


def test_fp64_wilson_loops_at_64_time_slices_fit_the_temporal_gauge_kernel():
    # planes of 24 columns with lines to 16 fill shared memory; nine times the time
    # where they do not fit
    short, full = (Lattice((24, 16, 16, nt), 2.4, seed=1, start="hot", prec="f64") for nt in (56, 64))
    assert _seconds(lambda: full.wilson_loops(16, 16)) < 3 * _seconds(lambda: short.wilson_loops(16, 16))


def test_batched_measurements_of_uneven_lattices():
    dims = [(4, 4, 4, 4), (16, 8, 12, 6), (2, 2, 2, 2), (6, 10, 4, 14), (8, 8, 8, 8)]
    for prec in ("f64", "f32", "f16q"):
        b = Batch(dims, [2.0] * len(dims), seed=1, start="cold", prec=prec)
        fields = [inputs.random_field(d, 50 + i) for i, d in enumerate(dims)]
        for i, U in enumerate(fields):
            b.set_links(i, U)
        for _ in range(2):                # the second call finds the counters at zero
            plaq, poly = b.plaquette(), b.polyakov()
            for i, (d, U) in enumerate(zip(dims, fields)):
                ref = as_stored(U, prec)
                np.testing.assert_allclose(plaq[i], oracle.plaquette(list(d), ref), atol=MTOL[prec], rtol=0)
                assert abs(poly[i] - oracle.polyakov(list(d), ref)) < MTOL[prec]


@pytest.mark.parametrize("prec", ["f64", "f32", "f16q"])
def test_batched_polyakov_loops_of_long_time_extents(prec):
    # lines in one, two, four and eight segments, the last of a length that is no
    # multiple of the loads' eight; a lattice of fewer lines than a block has threads
    dims = [(4, 2, 2, 14), (2, 2, 2, 16), (4, 4, 2, 40), (2, 4, 2, 72), (6, 6, 6, 136)]
    b = Batch(dims, [2.0] * len(dims), seed=1, start="cold", prec=prec)
    fields = [inputs.random_field(d, 70 + i) for i, d in enumerate(dims)]
    for i, U in enumerate(fields):
        b.set_links(i, U)
    for _ in range(2):
        poly, plaq = b.polyakov(), b.plaquette()
        for i, (d, U) in enumerate(zip(dims, fields)):
            ref = as_stored(U, prec)
            assert abs(poly[i] - oracle.polyakov(list(d), ref)) < MTOL[prec]
            np.testing.assert_allclose(plaq[i], oracle.plaquette(list(d), ref), atol=MTOL[prec], rtol=0)


def test_a_batch_measures_long_time_extents_like_a_lattice():
    # one thread a line took three times a single lattice's time
    dims = (8, 8, 8, 512)
    lat, b = Lattice(dims, 2.4, prec="f64"), Batch([dims], [2.4], prec="f64")
    assert _seconds(b.polyakov) < 2 * _seconds(lat.polyakov)


def test_roots_and_reciprocal_within_a_unit_in_the_last_place(tmp_path):
    # against numpy's extended arithmetic: every exponent that a staple's square or
    # an alpha can have and far beyond, both parities of it, significands near 1 and 2
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("long double has no more bits than double here")
    so = str(tmp_path / "roots.so")
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.run([nvcc_path(), *ARCH, "-O3", "-std=c++17", "-ftz=true", "-shared", "-Xcompiler", "-fPIC", "-I", INCLUDE,
                    "-I", CSRC, os.path.join(here, "roots_device.cu"), "-o", so], check=True)
    rng = np.random.default_rng(6)
    v = np.exp2(rng.uniform(-40, 70, 300000))
    v = np.concatenate([v, np.exp2(np.arange(-900, 901.0)), np.nextafter(np.exp2(np.arange(-900, 901.0)), 0),
                        np.nextafter(np.exp2(np.arange(-900, 901.0)), np.inf), np.exp2(rng.uniform(-900, 900, 20000))])
    out = np.zeros((3, v.size))
    dp = C.POINTER(C.c_double)
    assert C.CDLL(so).roots(v.ctypes.data_as(dp), C.c_int(v.size), out.ctypes.data_as(dp)) == 0
    x = v.astype(np.longdouble)
    for got, ref in zip(out, (1 / np.sqrt(x), np.sqrt(x), 0.5 / x)):
        ulp = np.spacing(ref.astype(np.float64))
        assert (np.abs(got.astype(np.longdouble) - ref) / ulp).max() < 1
    # zero, negative and subnormal under the root; an infinite alpha
    edge = np.array([0.0, -0.0, -1.0, 5e-324, np.inf, 1e300 * 1e8])
    out = np.zeros((3, edge.size))
    assert C.CDLL(so).roots(edge.ctypes.data_as(dp), C.c_int(edge.size), out.ctypes.data_as(dp)) == 0
    assert (out[1, :4] == 0).all() and (out[2, 4:] == 0).all()
