"""Rows without row forms stored in columns of packed bonds give exactly the CSR results (the same
terms in the same order, padding adds exact zeros), for every step kind; and runs of steps over
float4 spins give exactly the results of single steps, whatever the launch shape."""
import numpy as np
import pytest

from paper_1310_6143_gb300 import lattice as L

pytestmark = pytest.mark.gpu


def _graph(n, most, values, seed):
    """A random symmetric neighbour graph of at most `most` bonds per spin: as many row forms as spins."""
    rng = np.random.default_rng(seed)
    nb = [dict() for _ in range(n)]
    for i, j, v in zip(rng.integers(0, n, most * n), rng.integers(0, n, most * n), rng.integers(0, len(values), most * n)):
        if i != j and j not in nb[i] and len(nb[i]) < most and len(nb[j]) < most:
            nb[i][int(j)] = nb[j][int(i)] = values[v]
    nb[0].clear()  # an isolated spin: a row of padding only
    for d in nb[1:]:
        d.pop(0, None)
    row_ptr = np.concatenate([[0], np.cumsum([len(d) for d in nb])]).astype(np.int64)
    col = np.array([j for d in nb for j in d], dtype=np.int32)
    J = np.array([v for d in nb for v in d.values()])
    mu, ku, ax = L._homogeneous(n, 1.5 * L.MU_B, 1e-24, (0, 0.6, 0.8))
    return L.SpinLattice(row_ptr, col, J, mu, ku, ax, None, None)


def _run(lat, precision, columns, steps):
    from paper_1310_6143_gb300.system import SpinSystem

    out = []
    with SpinSystem(lat, alpha=0.1, dt=1e-16, T=300.0, H=(0.3, 0.0, 0.1), seed=3, precision=precision,
                    init_random=True, check_symmetry=True) as s:
        s.set_row_patterns(columns)
        s.set_exec("kernels")
        for k in steps:
            s.step(k)
        out += [s.spins(), s.record(0, sum(steps)), s.magnetisation(), s.energy()]
        s.mc_step(2)
        s.semi_implicit_step(1)
        out.append(s.spins())
    return out


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,most,nvalues", [(33, 6, 1), (1001, 6, 3), (2560, 12, 3), (3001, 12, 254), (3001, 12, 400)])
def test_columns_equal_the_csr(n, most, nvalues, precision):
    # 255 values fill the dictionary, 400 do not fit it: the CSR is read
    values = [1e-21 * (1 + 0.01 * k) for k in range(nvalues)]
    lat = _graph(n, most, values, 11)
    a, b = _run(lat, precision, True, [6]), _run(lat, precision, False, [6])
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("lats", ["film", "sphere", "batch", "long", "tensor"])
def test_runs_over_float4_spins_equal_single_steps(lats):
    from paper_1310_6143_gb300.system import SpinSystem

    systems = {"film": lambda: L.film(13, 11, 17), "sphere": lambda: L.core_shell_sphere(diameter=4e-9, r_core=1.6e-9),
               "batch": lambda: [L.simple_cubic(3, 3, 115), L.simple_cubic(11, 31, 3), L.dimer()],
               "long": lambda: L.fcc_long_range(6, 5, 7, r_cut=2.0),
               "tensor": lambda: L.with_dm(L.fcc(5, 4, 6, with_pos=True), D=1e-21)}[lats]()
    ref = None
    for block, slots, runs in ((256, 1, [1] * 9), (256, 1, [9]), (256, 3, [4, 5]), (512, 1, [3, 6]), (128, 5, [1, 8])):
        with SpinSystem(systems, alpha=0.1, dt=1e-16, T=500.0, seed=8, precision="fp32", init_random=True) as s:
            s.set_exec("kernels")
            s.set_launch(block, block * slots)
            for k in runs:
                s.step(k)
            S, P = s.spins(), [v.cpu().numpy() for v in s.state_device(1)]
        if ref is None:
            ref = S, P
        np.testing.assert_array_equal(S, ref[0])
        for x, y in zip(P, ref[1]):  # the predictor spins of the last step as well
            np.testing.assert_array_equal(x, y)
