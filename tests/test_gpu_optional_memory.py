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
    return L.film(24, 20, 17)


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
        s.step(3)
        s.set_exec("system_blocks")
        s.step(5)
        s.set_exec("persistent")
        s.step(5)
        assert s.info()["device_bytes"] == held
        s.set_exec("kernels")
        s.step(4)
        assert s.info()["device_bytes"] == held + 56 * s.n
        s.step(8)
        assert s.info()["device_bytes"] == held + 56 * s.n


@pytest.mark.parametrize("mode,runs", [("kernels", [5, 6]), ("graph", [2, 70]), ("auto", [3, 130])])
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
        s.step(20)  # (loads the kernels, too)
        ref = s.spins(), s.record(0, 20)
    stream = torch.cuda.Stream()
    with SS(_film(), **KW) as s:
        s.set_stream(stream)
        s.set_exec("kernels")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            s.step(5)
        with torch.cuda.stream(stream):
            for _ in range(4):
                graph.replay()
        held = s.info()["device_bytes"]
        np.testing.assert_array_equal(s.spins(), ref[0])
        np.testing.assert_array_equal(s.record(0, 20), ref[1])
        # memory that runs out later: the caller's graph names the buffer, so it stays
        lib.ss_debug_limit_bytes(lib.ss_debug_live_bytes())
        from paper_1310_6143_gb300._binding import SpinSysError

        with pytest.raises(SpinSysError, match="OOM"):
            s.mc_step(1)
        lib.ss_debug_limit_bytes(-1)
        assert s.info()["device_bytes"] == held
        torch.cuda.synchronize()
