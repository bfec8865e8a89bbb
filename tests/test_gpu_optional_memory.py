"""The buffers a handle can do without -- the float4 spins of FP32-mixed runs, the columns of packed
bonds -- are held only by handles that use them, are done without when the memory is short, and
are given back to calls that need it; the results are the same, bit for bit."""
import numpy as np
import pytest

from paper_1310_6143_gb300 import lattice as L

pytestmark = pytest.mark.gpu

KW = dict(alpha=0.1, dt=1e-16, T=300.0, H=(0.3, 0.0, 0.1), seed=3, precision="fp32", init_random=True)


@pytest.fixture()
def env():
    from paper_1310_6143_gb300 import _binding as B
    from paper_1310_6143_gb300.system import SpinSystem

    lib = B.load()
    yield lib, SpinSystem
    lib.ss_debug_limit_bytes(-1)


def _film():
    return L.film(300, 300, 15)  # 1.35 M spins: 76 MB of float4 spins, allocated by the first run of 8 steps


def _sphere():
    return L.core_shell_sphere(diameter=4e-9, r_core=1.6e-9)


def test_held_by_runs_only(env):
    lib, SS = env
    with SS(_film(), **KW) as s:
        s.set_exec("kernels")
        s.mc_step(2)
        held = s.info()["device_bytes"]
        s.mc_step(2)
        s.semi_implicit_step(5)
        s.midpoint_step(4)
        s.step(7)
        s.set_exec("persistent")
        s.step(8)
        s.set_exec("kernels")
        s.set_row_patterns(False)
        s.step(8)
        s.set_row_patterns(True)
        assert s.info()["device_bytes"] == held
        s.step(8)
        assert s.info()["device_bytes"] == held + 56 * s.n
        s.step(8)
        assert s.info()["device_bytes"] == held + 56 * s.n


def test_small_handles_hold_it_from_the_start(env):
    lib, SS = env
    out, whole = [], 0
    base = lib.ss_debug_live_bytes()
    for short in (False, True):
        if short:
            lib.ss_debug_limit_bytes(base + whole - 16)  # done without
        with SS(L.film(24, 20, 17), **KW) as s:
            lib.ss_debug_limit_bytes(-1)
            held = lib.ss_debug_live_bytes() - base
            whole = whole or held
            assert (held <= whole - 56 * s.n) == short
            s.set_exec("kernels")
            s.step(12)
            assert lib.ss_debug_live_bytes() - base == held
            s.set_exec("graph")
            s.step(130)
            out.append((s.spins(), s.record(0, 142)))
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)


def test_small_handles_of_the_cluster_do_not(env):
    lib, SS = env
    with SS(L.film(13, 10, 12), **KW) as s:  # 1,560 spins
        s.step(40)
        s.set_exec("kernels")
        s.step(11)
        held = s.info()["device_bytes"]
        s.step(12)
        assert s.info()["device_bytes"] == held + 56 * s.n


@pytest.mark.parametrize("mode,runs", [("kernels", [14, 15]), ("graph", [2, 70]), ("auto", [3, 130])])
def test_runs_without_the_memory(env, mode, runs):
    lib, SS = env
    out = []
    for short in (False, True):
        with SS(_film(), **KW) as s:
            s.set_exec(mode)
            if short:
                lib.ss_debug_limit_bytes(lib.ss_debug_live_bytes())
            for k in runs:
                s.step(k)
            lib.ss_debug_limit_bytes(-1)
            s.step(runs[-1])  # (not tried again)
            out.append((s.spins(), s.record(0, runs[0] + 2 * runs[1])))
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("lat", [_film, _sphere])
@pytest.mark.parametrize("mode", ["kernels", "graph"])
def test_given_back_to_a_call_that_needs_it(env, lat, mode):
    lib, SS = env
    out = []
    for short in (False, True):
        with SS(lat(), **KW) as s:
            s.set_exec(mode)
            s.step(66)
            held = s.info()["device_bytes"]
            if short:
                lib.ss_debug_limit_bytes(lib.ss_debug_live_bytes())
            s.mc_step(3)  # allocates its order and tiles
            assert (s.info()["device_bytes"] < held) == short
            lib.ss_debug_limit_bytes(-1)
            s.step(70)  # the launches captured before named the buffers
            s.semi_implicit_step(2)
            out.append((s.spins(), s.record(0, 141), s.energy()))
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)


def test_columns_given_back_while_a_handle_is_made(env):
    lib, SS = env
    base = lib.ss_debug_live_bytes()
    with SS(_sphere(), **KW) as s:
        whole = lib.ss_debug_live_bytes() - base
        s.step(6)
        ref = s.spins()
    lib.ss_debug_limit_bytes(base + whole - 16)
    with SS(_sphere(), **KW) as s:
        lib.ss_debug_limit_bytes(-1)
        assert lib.ss_debug_live_bytes() - base < whole - 24 * s.n  # rows of 12 take 48 bytes a spin
        s.step(6)
        np.testing.assert_array_equal(s.spins(), ref)


def test_first_run_inside_a_callers_capture(env):
    import torch

    lib, SS = env
    with SS(_film(), **KW) as s:
        s.step(30)  # (loads the kernels, too)
        ref = s.spins(), s.record(0, 30)
    stream = torch.cuda.Stream()
    with SS(_film(), **KW) as s:
        s.set_stream(stream)
        s.set_exec("kernels")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            s.step(15)
        with torch.cuda.stream(stream):
            for _ in range(2):
                graph.replay()
        held = s.info()["device_bytes"]
        assert held >= 56 * s.n
        np.testing.assert_array_equal(s.spins(), ref[0])
        np.testing.assert_array_equal(s.record(0, 30), ref[1])
        # memory that runs out later: the caller's graph names the buffer, so it stays
        lib.ss_debug_limit_bytes(lib.ss_debug_live_bytes())
        from paper_1310_6143_gb300._binding import SpinSysError

        with pytest.raises(SpinSysError, match="OOM"):
            s.mc_step(1)
        lib.ss_debug_limit_bytes(-1)
        assert s.info()["device_bytes"] == held
        torch.cuda.synchronize()


@pytest.mark.parametrize("lats", ["film", "batch", "tensor", "wide"])
def test_longer_runs_equal_single_steps(env, lats):
    # the lengths from which float4 spins are taken: 12 steps below 10,000 spins, 32 above
    lib, SS = env
    systems = {"film": lambda: L.film(13, 11, 17), "wide": lambda: L.film(41, 30, 9),
               "batch": lambda: [L.simple_cubic(3, 3, 115), L.simple_cubic(11, 31, 3), L.dimer(), L.film(9, 8, 7)],
               "tensor": lambda: L.with_dm(L.fcc(5, 4, 6, with_pos=True), D=1e-21)}[lats]()
    steps = 34 if lats == "wide" else 14
    ref = None
    for block, slots, runs in ((256, 1, [1] * steps), (256, 1, [steps]), (256, 3, [1, steps - 1]), (512, 1, [steps - 2, 2]),
                               (128, 5, [steps])):
        with SS(systems, **KW) as s:
            s.set_exec("kernels")
            s.set_launch(block, block * slots)
            for k in runs:
                s.step(k)
            out = [s.spins()] + [v.cpu().numpy() for v in s.state_device(1)]
        ref = ref or out
        for x, y in zip(out, ref):
            np.testing.assert_array_equal(x, y)
