"""What the autotuner stores and times: an entry is taken only for the same storage of the rows and the
same version of the kernels."""
import pytest

from paper_1310_6143_gb300 import lattice as L

pytestmark = pytest.mark.gpu

KW = dict(alpha=0.1, dt=1e-16, T=300.0, seed=4, precision="fp32", init_random=True)


@pytest.fixture()
def cache(tmp_path, monkeypatch):
    path = tmp_path / "tune.txt"
    monkeypatch.setenv("SPINSYS_AUTOTUNE_CACHE", str(path))
    return path


@pytest.mark.parametrize("lat", [lambda: L.film(24, 20, 17), lambda: L.core_shell_sphere(diameter=4e-9, r_core=1.6e-9)])
def test_storage_of_the_rows_is_in_the_key(cache, lat):
    from paper_1310_6143_gb300.system import SpinSystem

    for on, lines in ((True, 1), (False, 2), (True, 2), (False, 2)):
        with SpinSystem(lat(), **KW) as s:
            s.set_row_patterns(on)
            s.autotune(4)
        assert len(cache.read_text().splitlines()) == lines


def test_entries_of_older_kernels_are_not_taken(cache):
    from paper_1310_6143_gb300.system import SpinSystem

    lat = L.film(24, 20, 17)
    with SpinSystem(lat, **KW) as s:
        s.autotune(4)
    key = cache.read_text().split("\t")[0]
    fields = key.split("|")
    # the entry that the array kernels' version wrote for this workload, with a shape no trial tries
    cache.write_text("|".join(["v2"] + fields[1:9]) + "\t1 512 8192 3 0\n")
    with SpinSystem(lat, **KW) as s:
        info = s.autotune(4)
    assert (info["block"], info["tile"]) != (512, 8192)
    assert len(cache.read_text().splitlines()) == 2


def test_trials_launch_what_runs_launch():
    # however few steps are asked for: the trials run over the float4 spins that runs take
    from paper_1310_6143_gb300.system import SpinSystem

    with SpinSystem(L.film(300, 300, 15), **KW) as s:
        held, ref = s.info()["device_bytes"], s.spins()
        s.autotune(1)
        assert (s.spins() == ref).all() and s.step_index == 0
        s.set_gaussian_pass(0)
        s.set_launch(256, 256)
        now = s.info()["device_bytes"]
        s.set_exec("kernels")
        s.step(8)
        assert s.info()["device_bytes"] == now > held + 56 * s.n
