"""Rows of very different length, and lattices whose size is no multiple of the period of the packed slices:
a warp per slice gives exactly what a thread per row gives, in single steps and in runs."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1310_6143_gb300 import lattice as L

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _ring(n, reach, hub):
    """Spins on a ring bonded up to `reach` apart; spin 0 with every spin up to `hub` away as well."""
    nb = [[(i + d) % n for d in range(-reach, reach + 1) if d] for i in range(n)]
    for j in range(reach + 1, hub + 1):
        nb[0].append(j)
        nb[j].append(0)
    row_ptr = np.concatenate([[0], np.cumsum([len(r) for r in nb])]).astype(np.int64)
    col = np.array([j for r in nb for j in r], dtype=np.int32)
    mu, ku, ax = L._homogeneous(n, 1.5 * L.MU_B, 1e-24, (0, 0.6, 0.8))
    return L.SpinLattice(row_ptr, col, np.full(len(col), 2e-22), mu, ku, ax, None, None)


def drop_last(lat, k):
    """The lattice without its last k spins (vacancies at one corner)."""
    n = lat.n - k
    keep = np.repeat(np.arange(lat.n) < n, np.diff(lat.row_ptr)) & (lat.col < n)
    rows = np.add.reduceat(keep, lat.row_ptr[:-1])[:n]
    row_ptr = np.concatenate([[0], np.cumsum(rows)]).astype(np.int64)
    return L.SpinLattice(row_ptr, lat.col[keep], lat.J[keep], lat.mu_s[:n], lat.k_u[:n], lat.easy_axis[:n], None, None)


def fcc_with_vacancies(k):
    """225 cells of four sites, the period of their slices: without k spins, k of the four classes are
    a spin shorter, 224, and take a slice less."""
    return drop_last(L.fcc_long_range(5, 5, 9, r_cut=2.0), k)


def _run(lat, precision, mode, runs):
    from paper_1310_6143_gb300.system import SpinSystem

    with SpinSystem(lat, alpha=0.1, dt=1e-16, T=300.0, H=(0.3, 0.0, 0.1), seed=3, precision=precision,
                    init_random=True, check_symmetry=True) as s:
        s.set_exchange_rows(mode)
        s.set_exec("kernels")
        for k in runs:
            s.step(k)
        return s.spins(), s.record(0, sum(runs))


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_one_long_row_among_short_ones(precision):
    lat = _ring(3001, 12, 2900)
    ref = _run(lat, precision, "thread", [1] * 6)
    for runs in ([1] * 6, [6]):
        got = _run(lat, precision, "warp", runs)
        np.testing.assert_array_equal(got[0], ref[0])
        np.testing.assert_array_equal(got[1], ref[1])


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("vacancies", [0, 1, 2, 3])
def test_sizes_that_are_no_multiple_of_the_period(vacancies, precision):
    lat = fcc_with_vacancies(vacancies)
    ref = _run(lat, precision, "thread", [1] * 6)
    for runs in ([1] * 6, [6], [2, 4]):
        got = _run(lat, precision, "warp", runs)
        np.testing.assert_array_equal(got[0], ref[0])
        np.testing.assert_array_equal(got[1], ref[1])


def test_row_passes_switched_off_and_on_between_runs():
    # runs without row passes write the float4 spins in another order: the padding between the
    # classes, gathered with J = 0, must come back finite
    from paper_1310_6143_gb300.system import SpinSystem

    lats = [fcc_with_vacancies(3), fcc_with_vacancies(1), _ring(331, 12, 12)]  # a batch of 2,127: no multiple of 4
    out = []
    for modes in (["thread"] * 5, ["warp", "thread", "warp", "thread", "warp"], ["thread", "warp", "warp", "thread", "warp"]):
        with SpinSystem(lats, alpha=0.1, dt=1e-16, T=300.0, seed=3, precision="fp32", init_random=True) as s:
            s.set_exec("kernels")
            for m in modes:
                s.set_exchange_rows(m)
                s.step(5)
                s.semi_implicit_step(1)
            out.append((s.spins(), s.record(0, 30)))
    for o in out[1:]:
        np.testing.assert_array_equal(o[0], out[0][0])
        np.testing.assert_array_equal(o[1], out[0][1])


@pytest.mark.parametrize("every", [1, 3, 5, 100])
def test_float4_runs_with_demagnetising_field_and_cubic_anisotropy(every):
    from paper_1310_6143_gb300.system import SpinSystem

    a = 3e-10
    lat = L.simple_cubic(9, 8, 7, periodic=(False, False, False), J=6e-21, k_u=1e-23, a=a, with_pos=True)
    lat.k_c = np.where(np.arange(lat.n) % 3 == 0, 2e-23, 0.0)
    out = []
    for runs in ([1] * 23, [23], [4, 6, 13]):
        with SpinSystem(lat, alpha=0.1, dt=1e-16, T=300.0, H=(0.3, 0.0, 0.1), seed=3, precision="fp32",
                        init_random=True) as s:
            s.set_exec("kernels")
            s.set_demag(2 * a, a ** 3, every=every)
            for k in runs:
                s.step(k)
            out.append((s.spins(), s.record(0, 23), [v.cpu().numpy() for v in s.state_device(1)]))
    for o in out[1:]:
        np.testing.assert_array_equal(o[0], out[0][0])
        np.testing.assert_array_equal(o[1], out[0][1])
        for x, y in zip(o[2], out[0][2]):
            np.testing.assert_array_equal(x, y)


def _walk(path):
    """Every kind of step on rows of uneven length, for the checked build (see below)."""
    from paper_1310_6143_gb300.system import SpinSystem

    res = {}
    for name, lat in (("columns", L.core_shell_sphere(diameter=4e-9, r_core=1.6e-9)), ("vacancies", fcc_with_vacancies(3)),
                      ("hub", _ring(3001, 12, 2900)), ("long", drop_last(L.fcc_long_range(9, 9, 9, r_cut=3.0), 5))):
        for precision in ("fp32", "fp64"):
            with SpinSystem(lat, alpha=0.1, dt=1e-16, T=300.0, seed=3, precision=precision, init_random=True) as s:
                s.set_exec("kernels")
                s.step(2)
                s.step(6)
                s.midpoint_step(1, iterations=2)
                s.semi_implicit_step(1)
                s.mc_step(2)
                res[f"{name}_{precision}"] = s.spins()
                res[f"{name}_{precision}_record"] = s.record(0, 12)
    np.savez(path, **res)


def test_checked_build_gathers_in_bounds(tmp_path):
    # the bounds-checked build reports an index out of range as an error instead of using it
    from paper_1310_6143_gb300 import build

    out = []
    for lib in (build.build(checked=True), build.build()):
        path = str(tmp_path / f"{len(out)}.npz")
        subprocess.run([sys.executable, "-c", f"import test_gpu_uneven_rows as t; t._walk({path!r})"], check=True, timeout=900,
                       env=dict(os.environ, SPINSYS_LIB=lib, PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")])))
        out.append(np.load(path))
    assert sorted(out[0].files) == sorted(out[1].files)
    for k in out[0].files:
        np.testing.assert_array_equal(out[0][k], out[1][k])
