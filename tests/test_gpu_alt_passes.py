"""The alternative integrators' passes: tiles cut into parts, row forms against the CSR.

Spins do not depend on the tile shape or on how rows are stored (the same terms in the same
order), so they are compared bit for bit.  The record's sums are FP64 (FP32-mixed: float pairs
exact to 2^-48) in an order that depends on the tiles: n < 2^14 terms of one sign scale differ by
at most n 2^-48 < 6e-11 of the largest sum, held to 1e-10.
"""
import numpy as np
import pytest

from paper_1310_6143_gb300 import lattice as L

pytestmark = pytest.mark.gpu


def _run(lats, method, precision, tile, forms):
    from paper_1310_6143_gb300.system import SpinSystem

    with SpinSystem(lats, alpha=0.1, dt=1e-16, T=300.0, H=(0.3, 0.0, -0.2), seed=5, precision=precision,
                    init_random=True) as s:
        s.set_launch(256, tile)
        s.set_row_patterns(forms)
        if method == "sib":
            s.semi_implicit_step(3)
        else:
            s.midpoint_step(3, iterations=method)
        return s.spins(), s.record(0, 3)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("method", ["sib", 1, 2, 3])
@pytest.mark.parametrize("lats", ["film", "batch", "sphere"])
def test_tile_parts_and_row_forms(lats, method, precision):
    systems = {"film": lambda: L.film(24, 20, 17), "sphere": lambda: L.core_shell_sphere(diameter=4e-9, r_core=1.6e-9),
               # ragged: a system of one tile part and a bit, one spin short of a part, a tiny one
               "batch": lambda: [L.simple_cubic(3, 3, 114), L.simple_cubic(11, 31, 3), L.dimer()]}[lats]()
    S0, r0 = _run(systems, method, precision, 256, False)   # a part per tile, the CSR
    for tile, forms in ((256, True), (512, True), (1024, False), (4096, True), (2816, True)):
        S, r = _run(systems, method, precision, tile, forms)
        np.testing.assert_array_equal(S, S0)
        scale = np.abs(r0).max(axis=0, keepdims=True)
        scale[..., :4] = scale[..., 3:4]
        scale[..., 4:] = scale[..., 4:].max(axis=-1, keepdims=True)
        assert np.all(np.abs(r - r0) <= 1e-10 * scale)
