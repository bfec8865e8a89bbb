"""Rows of very different length, and lattices whose size is no multiple of the period of the packed slices:
a warp per slice gives exactly what a thread per row gives, in single steps and in runs."""
import numpy as np
import pytest

from paper_1310_6143_gb300 import lattice as L

pytestmark = pytest.mark.gpu


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
