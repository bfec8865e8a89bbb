"""Monte Carlo steps whose record and step counter ride in the last colour pass: classes of few trials
(64-thread blocks) and of many, one, some and many systems, one and two classes; the record of every
step equals the state it was taken from, and captured steps equal plain ones bit for bit.

The record's sums run over at most 6e4 terms of float pairs (exact to 2^-48) or FP64 in an order of
their own: within 6e4 x 2^-48 < 3e-10 of the largest sum's scale, held to 1e-9.
"""
import numpy as np
import pytest

from paper_1310_6143_gb300 import lattice as L

pytestmark = pytest.mark.gpu

SYSTEMS = {"small": lambda: L.simple_cubic(6, 7, 9, periodic=(False, False, False)),
           "large": lambda: L.film(66, 64, 19), "free": lambda: L.single_spin(),
           "two": lambda: [L.simple_cubic(4, 6, 8), L.dimer()],
           "many": lambda: [L.simple_cubic(4, 4, 4 + 2 * (k % 3)) for k in range(11)]}


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("name", sorted(SYSTEMS))
def test_record_and_counter(name, precision):
    from paper_1310_6143_gb300.system import SpinSystem

    lats = SYSTEMS[name]()
    kw = dict(T=250.0, H=(0.2, 0.0, -0.4), seed=17, precision=precision, init_random=True)
    out = []
    for mode, runs in (("kernels", [1] * 3 + [63]), ("auto", [66])):
        with SpinSystem(lats, **kw) as s:
            s.set_exec(mode)
            for k in runs:
                before = [np.concatenate([s.energy(q), s.magnetisation(q)[:3]]) for q in range(s.num_systems)]
                first = s.step_index
                s.mc_step(k)
                assert s.step_index == first + k
                rec = s.record(first, 1)[0]
                for q, b in enumerate(before):
                    scale = max(np.abs(rec[q, 4:7]).max(), 1e-30)
                    assert np.all(np.abs(rec[q, [7, 4, 5, 6]] - b[:4]) <= 1e-9 * 3 * scale + 4e-7 * scale * (precision == "fp32"))
                    assert np.all(np.abs(rec[q, :3] / rec[q, 3] - b[4:]) <= 1e-9)
            out.append((s.spins(), s.record(0, 66), [s.mc_stats(q) for q in range(s.num_systems)]))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]
