"""Long rows packed into slices of 32 rows, on the host: the words reproduce the rows they came from for
every period and remainder, and one row much longer than the others costs its own slice, not the lattice."""
import ctypes
import os
import resource
import subprocess
import sys
import time

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("slices") / "slices.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_1310_6143_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "_slices_host.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.slices_hash.restype = ctypes.c_uint64
    return lib


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _pack(lib, rp, col, bid, zero):
    n = len(rp) - 1
    sizes, h = np.zeros(4, np.int64), ctypes.c_void_p()
    if lib.slices_pack(ctypes.c_int64(n), _p(rp), _p(col), _p(bid), zero, ctypes.byref(h), _p(sizes)):
        raise MemoryError
    sl, off, words = np.zeros((sizes[1], 2), np.int32), np.zeros(sizes[2] + 1, np.int64), np.zeros(sizes[3], np.uint32)
    lib.slices_copy(h, _p(sl), _p(off), _p(words))
    lib.slices_free(h)
    return int(sizes[0]), sl, off, words


def _positions(lib, n, period):
    pos = np.zeros(n, np.int64)
    lib.slices_positions(ctypes.c_int64(n), period, _p(pos))
    return pos


def _rows(n, cells, basis, seed):
    """Rows like those of a lattice of `basis` sites a cell, the cells on a ring, with some bonds missing."""
    rng = np.random.default_rng(seed)
    cols, rp = [], [0]
    for i in range(n):
        c, b = divmod(i, basis)
        j = [(c + d) * basis + q for d in range(-cells, cells + 1) for q in range(basis)]
        j = [x % n for x in j if x % n != i]
        j = [x for x in j if rng.random() > 0.1 * (i % 7 == 0)]
        cols += j
        rp.append(len(cols))
    bid = np.array([(x * 31) % 5 for x in cols], np.uint8)
    return np.array(rp, np.int32), np.array(cols, np.int32), bid


@pytest.mark.parametrize("n,basis", [(1, 1), (31, 1), (33, 2), (64, 2), (130, 4), (131, 4), (515, 4), (1027, 6), (1029, 8)])
def test_words_give_the_rows_back(host, n, basis):
    rp, col, bid = _rows(n, 3, basis, n)
    period, sl, off, words = _pack(host, rp, col, bid, 5)
    pos = _positions(host, n, period)
    seen = np.zeros(n, bool)
    for s, (form, row0) in enumerate(sl):
        w = words[off[form]:off[form + 1]].reshape(-1, 32)
        for lane in range(32):
            i = row0 + lane * period
            at, jd = (32 * s + (w[:, lane] >> 8)) & 0xFFFFFF, w[:, lane] & 255
            ln = rp[i + 1] - rp[i] if i < n else 0
            assert np.all(jd[ln:] == 5) and np.all(at[ln:] == 32 * s + lane)  # padding: itself with J = 0
            if i < n:
                assert not seen[i] and pos[i] == 32 * s + lane
                seen[i] = True
                np.testing.assert_array_equal(at[:ln], pos[col[rp[i]:rp[i + 1]]])
                np.testing.assert_array_equal(jd[:ln], bid[rp[i]:rp[i + 1]])
    assert seen.all()


@pytest.mark.parametrize("vacancies", [0, 1, 2, 3])
def test_lattice_sizes_off_the_period(host, vacancies):
    # the lattices that tests/test_gpu_uneven_rows.py steps: period 4, classes of 225 and 224 rows
    from test_gpu_uneven_rows import fcc_with_vacancies

    lat = fcc_with_vacancies(vacancies)
    period, sl, off, words = _pack(host, lat.row_ptr.astype(np.int32), lat.col.astype(np.int32),
                                   np.zeros(lat.nnz, np.uint8), 1)
    assert period == 4 and lat.n == 900 - vacancies and len(sl) == 32 - vacancies


@pytest.mark.parametrize("period", [1, 2, 3, 4, 6, 8])
def test_positions_are_distinct_and_in_range(host, period):
    for n in list(range(period, 300)) + [4093, 4096, 4099]:
        pos = _positions(host, n, period)
        per_class = [-(-len(range(b, n, period)) // 32) for b in range(period)]
        assert len(np.unique(pos)) == n and pos.min() == 0 and pos.max() < 32 * sum(per_class)


def test_one_long_row_among_short_ones(host):
    # 200,000 rows of 16 bonds and one of 100,000: 26 MB of words.  With the longest row's width
    # for every slice it would be 80 GB; 4 GB more than the process already has are allowed.
    n, hub = 200_000, 100_000
    i = np.arange(n)
    col = ((i[:, None] + np.r_[-8:0, 1:9]) % n).astype(np.int32)
    rows = np.concatenate([col[:1].ravel(), np.arange(100, 100 + hub), col[1:].ravel()]).astype(np.int32)
    rp = np.concatenate([[0], np.cumsum(np.full(n, 16) + hub * (i == 0))]).astype(np.int32)
    used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
    soft, hard = resource.getrlimit(resource.RLIMIT_AS)
    resource.setrlimit(resource.RLIMIT_AS, (used + (4 << 30), hard))
    try:
        period, sl, off, words = _pack(host, rp, rows, np.zeros(len(rows), np.uint8), 1)
    finally:
        resource.setrlimit(resource.RLIMIT_AS, (soft, hard))
    assert len(words) <= 32 * (n // 32 + 8) * 16 + 32 * (hub + 16)


def test_every_word_counts_in_the_hash(host):
    # slices alike but for a few bonds must not share a hash: each would be compared with all of them
    rng = np.random.default_rng(1)
    words = rng.integers(0, 1 << 32, 32 * 17, dtype=np.uint32)

    def h(w):
        return host.slices_hash(_p(w), ctypes.c_int64(len(w)))

    seen = {h(words)}
    for q in range(len(words)):  # one altered bond, in each place; then two neighbouring ones, and three in a row
        w = words.copy()
        w[q] += 256
        seen.add(h(w))
    for d in ((1, -1), (1, -2, 1)):
        for q in range(len(words) - 2):
            w = words.copy()
            w[q:q + len(d)] += np.array(d, np.int64).astype(np.uint32)
            seen.add(h(w))
    assert len(seen) == 1 + len(words) + 2 * (len(words) - 2)


def test_dilute_impurities_pack_in_linear_time(host):
    # 48,000 slices, each with altered bonds of its own: a second's work, most of a minute's
    # when every slice is compared with all before it
    n = 32 * 48_000
    i = np.arange(n)
    col = ((i[:, None] + np.r_[-10:0, 1:11]) % n).astype(np.int32)
    bid = np.zeros((n, 20), np.uint8)
    for b in range(16):  # the slice's number in bonds 17 to 19 of its rows
        bid[np.arange(48_000) * 32 + 3 + b // 3, 17 + b % 3] = (np.arange(48_000) >> b) & 1
    rp = (20 * np.arange(n + 1)).astype(np.int32)
    t0 = time.perf_counter()
    period, sl, off, words = _pack(host, rp, col.ravel(), bid.ravel(), 2)
    assert time.perf_counter() - t0 < 10.0
    assert len(off) - 1 > 40_000


def _dictionary(lib, J):
    d, zero, bid = np.zeros(256, np.float32), ctypes.c_int(), np.zeros(len(J), np.uint8)
    k = lib.slices_dictionary(_p(J), ctypes.c_int64(len(J)), _p(d), ctypes.byref(zero), _p(bid))
    return (None if k < 0 else d[:k]), zero.value, bid


@pytest.mark.parametrize("values,with_zero", [(1, False), (1, True), (254, True), (255, False), (255, True), (256, False)])
def test_dictionary_of_bond_values(host, values, with_zero):
    rng = np.random.default_rng(values)
    v = np.concatenate([1e-3 * np.arange(1, values + 1), [0.0] * with_zero]).astype(np.float32)
    J = np.concatenate([v, rng.choice(v, 5000)])
    d, zero, bid = _dictionary(host, J)
    if values > 255:
        assert d is None
        return
    assert len(d) == values + 1 and d[zero] == 0.0
    np.testing.assert_array_equal(d[bid], J)


def test_dictionary_of_many_values_in_linear_time(host):
    # 200 values in no order, as disordered exchange has them: 20 M bonds at a few ns each
    J = np.random.default_rng(3).integers(1, 201, 20_000_000).astype(np.float32)
    t0 = time.perf_counter()
    d, zero, bid = _dictionary(host, J)
    assert time.perf_counter() - t0 < 1.0
    assert len(d) == 201


def test_create_reports_host_memory_that_runs_out():
    # the table of 2^31 - 1 systems does not fit 1 GB: an error code, not the end of the process
    code = ("import ctypes, resource\n"
            "from paper_1310_6143_gb300 import _binding as B\n"
            "lib = B.load()\n"
            "used = int(open('/proc/self/statm').read().split()[0]) * resource.getpagesize()\n"
            "resource.setrlimit(resource.RLIMIT_AS, (used + (1 << 30), resource.RLIM_INFINITY))\n"
            "p, h = B.SSParams(), ctypes.c_void_p()\n"
            "assert lib.spin_batch_create(ctypes.byref(p), 2**31 - 1, ctypes.byref(h)) == 3  # SS_ERR_OOM\n"
            "assert not h\n")
    from paper_1310_6143_gb300 import build

    build.build()
    subprocess.run([sys.executable, "-c", code], cwd=ROOT, check=True, timeout=300)
