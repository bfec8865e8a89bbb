"""Launch shapes picked from sizes, on the host: tiles are counted within the systems of a batch, so that
the busiest SM has little more than its share."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS = 152


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("shape") / "shape.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_1310_6143_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "_slices_host.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.shape_mc_tile.restype = lib.shape_busiest_sm.restype = ctypes.c_int64
    return lib


def _mc_tile(lib, mixed, sizes):
    c = [np.array([(n + 1 - k) // 2 for n in sizes], np.int64) for k in (0, 1)]
    return lib.shape_mc_tile(int(mixed), SMS, int(len(sizes) <= 2), len(sizes),
                             *(a.ctypes.data_as(ctypes.c_void_p) for a in c)), c[0]


def _share(tile, trials):
    """Trials of the busiest SM's tiles, against an even share of the class."""
    tiles = np.sum(-(-trials // tile))
    return -(-tiles // SMS) * tile / (trials.sum() / SMS)


BATCHES = [[20 ** 3] * 40, [30 ** 3] * 40, [40 ** 3] * 9, [40 ** 3] * 8, [12 ** 3] * 100, [8 ** 3] * 400, [80 ** 3], [100 ** 3],
           [512 * 512 * 16], [64 ** 3], [48 ** 3, 48 ** 3, 2000]]


@pytest.mark.parametrize("mixed", [True, False])
@pytest.mark.parametrize("sizes", BATCHES, ids=lambda s: f"{len(s)}x{s[0]}")
def test_monte_carlo_tiles_of_batches(host, sizes, mixed):
    tile, trials = _mc_tile(host, mixed, sizes)
    assert tile == 64 or (tile % 256 == 0 and 256 <= tile <= 2560)
    assert _share(tile, trials) < 1.3


@pytest.mark.parametrize("mixed", [True, False])
def test_monte_carlo_tiles_of_drawn_batches(host, mixed):
    rng = np.random.default_rng(7)
    for _ in range(300):
        sizes = rng.integers(2000, 200_000, rng.integers(1, 60)).tolist()
        tile, trials = _mc_tile(host, mixed, sizes)
        if trials.sum() < 256 * SMS:
            assert tile == 64
        else:
            # a ragged tile per system and a last round per SM in tiles of 256, and 0.3 for the
            # reductions that longer tiles save
            assert _share(tile, trials) < 1.3 + 256 * (SMS + len(sizes)) / trials.sum()


@pytest.mark.parametrize("sizes,worst", [([128 ** 3], 2304), ([120 ** 3], 2048)])
def test_monte_carlo_tiles_that_leave_half_a_wave_over(host, sizes, worst):
    # 456 tiles of 2,304 and 422 of 2,048 are three and 2.8 for each of 152 SMs, but four on some
    # of them: two blocks are resident, and of the 152 or 118 that take a second tile some share an SM
    tile, _ = _mc_tile(host, False, sizes)
    assert tile != worst


def test_tiles_of_the_busiest_sm(host):
    def busiest(tiles, resident):
        return host.shape_busiest_sm(ctypes.c_int64(tiles), SMS, resident)

    for resident in (1, 2, 3, 4):
        for tiles in range(1, 5000, 7):
            k, mean = busiest(tiles, resident), tiles / SMS
            assert mean <= k < mean + 1 + resident
            assert k == -(-tiles // SMS) or tiles > resident * SMS
    assert [busiest(t, 2) for t in (152, 303, 304, 304 + 117, 304 + 118, 456, 608)] == [1, 2, 2, 3, 4, 4, 4]


@pytest.mark.parametrize("mixed", [True, False])
def test_record_blocks_stay_in_the_last_round(host, mixed):
    def blocks(nsys, grid, rounds):
        return host.shape_record_blocks(int(mixed), ctypes.c_int64(nsys), min(nsys, 64), ctypes.c_int64(grid),
                                        ctypes.c_int64(rounds), SMS)

    for nsys in (1, 2, 5, 40, 64, 300, 1200):
        for grid in list(range(1, 460)) + [608, 1216]:
            for rounds in (1, 9):
                k, most, room = blocks(nsys, grid, rounds), min(nsys, 64), -grid % SMS
                if room < most and nsys <= room * max(8, (1 if mixed else 4) * rounds * -(-grid // SMS)):
                    assert k == room  # the launch takes the rounds that its own blocks take
                else:
                    assert k == most  # room for all, or for too few
    assert blocks(40, 440, 10) == 16 and blocks(60, 299, 9) == 5 and blocks(60, 275, 10) == 29
    assert blocks(100, 300, 11) == (64 if mixed else 4)


# us per step of FP32-mixed runs of 1024 x 1024 films by layers and spins per thread (512-thread blocks, GB300)
FILMS = {8: {6: 298, 7: 301, 8: 299, 9: 290, 10: 314, 11: 294, 12: 315}, 10: {6: 371, 7: 375, 8: 384, 9: 376, 10: 365, 11: 364, 12: 380},
         13: {6: 485, 7: 486, 8: 472, 9: 473, 10: 475, 11: 463, 12: 460}, 14: {6: 518, 7: 513, 8: 511, 9: 512, 10: 523, 11: 516, 12: 504},
         15: {6: 545, 7: 559, 8: 553, 9: 536, 10: 529, 11: 535, 12: 559}, 16: {6: 585, 7: 595, 8: 585, 9: 570, 10: 576, 11: 573, 12: 571}}


@pytest.mark.parametrize("layers", sorted(FILMS))
def test_spins_per_thread_of_large_films(host, layers):
    n = np.array([1024 * 1024 * layers], np.int64)
    slots = host.shape_heun_slots(1, 512, SMS, 1, n.ctypes.data_as(ctypes.c_void_p))
    assert FILMS[layers][slots] <= 1.025 * min(FILMS[layers].values())
