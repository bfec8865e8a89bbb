// Rules that pick launch shapes from sizes, in plain C++ so that they can be checked without a GPU.
#pragma once
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <numeric>
#include <vector>

namespace ss {

// Tiles on the SM with most of them, when at most `resident` blocks per SM take the tiles in turn, block
// b those at b, b + blocks, ...  Where the tiles are no multiple of the blocks, the low blocks have
// one more.  The SMs do not get their blocks in plain rounds: four of the 152 are handed out a third
// faster (measured with kernels that note their SM), so of a grid of several blocks per SM the
// first 117, not 152, lie on distinct SMs, and 0.77 of the SMs take up a round of the rest.
inline int64_t busiest_sm(int64_t tiles, int sm_count, int resident) {
    const int64_t sms = std::max(sm_count, 1), blocks = resident * sms;
    if (tiles < blocks) return (tiles + sms - 1) / sms;
    const int64_t rest = tiles % blocks, most = (int64_t)std::ceil((double)rest / (0.77 * (double)sms));
    return resident * (tiles / blocks) + std::min<int64_t>(resident, most);
}

// Trials per tile of the colour passes that sum the record (at most two classes): 64, in blocks of as
// many threads, or r rounds of 256-thread blocks, r to 10 -- whichever a model of the pass, fitted to
// 53 lattices and batches on GB300, finds cheapest.  A tile lies within one system, so the tiles are
// counted system by system: a rule that took the class as one run gave 40 systems of 20^3 four tiles
// of 1,280 and 160 trials each, two on the busiest SM (FP64 202 us per step; now 106), 9 of 40^3
// FP32-mixed 75 us (now 51).  The model, in rounds of a 256-thread block at full residency
// (2.8 us FP32-mixed, 17.5 us FP64), of the k tiles on the busiest SM:
//  - FP32-mixed, r rounds: four blocks are resident on an SM.  Each whole round of four tiles takes
//    4 (r + 0.85) (0.85: the record's reduction).  One to four left over, on the busiest SM, wait for
//    latency: as the only tiles they take 2, 2.4, 3.25 and 3.85 of r + 0.85, behind whole rounds, which
//    end unevenly, 2.35, 2.55, 3.8 and 5.2.
//  - FP64, r rounds: two blocks are resident; (r + 0.2) k, an eighth more for a lone tile's eight warps.
//  - 64 trials, whose blocks read the transform's tables where they lie and are handed out as SMs get
//    free: 2.5 + 0.31 k FP32-mixed, 0.38 + 0.265 k FP64; and, where the pass sums the record itself,
//    3.75 ns a slot.  Always for classes of fewer than 256 trials per SM; not for a system of more
//    than 2,048 slots, which one block sums, nor beyond the k for which they were ever fastest.
// Its choice is within 4.1 % of the fastest on all 53 (FP64 1.5 %), 0.4 % on average (0.1 %).  Counted in plain
// rounds of SMs, sc 128^3 in FP64 got nine rounds: 656 us per step, seven 521.
inline int64_t mc_tile(bool mixed, int sm_count, bool sums_record, const std::vector<int64_t> (&trials)[2]) {
    const int64_t sms = std::max(sm_count, 1);
    auto total = [](const std::vector<int64_t> &t) { return std::accumulate(t.begin(), t.end(), int64_t(0)); };
    auto tiles = [](int64_t tile, const std::vector<int64_t> &t) {
        int64_t k = 0;
        for (int64_t n : t) k += (n + tile - 1) / tile;
        return k;
    };
    if (std::max(total(trials[0]), total(trials[1])) < 256 * sms) return 64;
    int64_t best = 256, slots = 0, longest = 0;
    double least = 1e300;
    for (size_t s = 0; s < trials[0].size(); ++s) {
        const int64_t k = (trials[0][s] + 63) / 64 + (trials[1][s] + 63) / 64;
        slots += k;
        longest = std::max(longest, k);
    }
    const int64_t k64 = (std::max(tiles(64, trials[0]), tiles(64, trials[1])) + sms - 1) / sms;
    if (longest <= 2048 && k64 <= (mixed ? 24 : 72)) {
        least = sums_record ? (double)slots * (3.75e-3 / (mixed ? 2.8 : 17.5)) : 0.0;
        for (const auto &t : trials)
            if (total(t) > 0) {
                const double k = (double)((tiles(64, t) + sms - 1) / sms);
                least += mixed ? 2.5 + 0.31 * k : 0.38 + 0.265 * k;
            }
        best = 64;
    }
    for (int r = 1; r <= 10; ++r) {
        double cost = 0.0;
        for (const auto &t : trials) {
            const int64_t n = tiles(256 * r, t), k = busiest_sm(n, sm_count, mixed ? 4 : 2);
            if (mixed) {
                constexpr double only[5] = {0.0, 2.0, 2.4, 3.25, 3.85}, behind[5] = {0.0, 2.35, 2.55, 3.8, 5.2};
                const int64_t whole = n / (4 * sms);
                cost += (r + 0.85) * (4.0 * (double)whole + (whole ? behind : only)[k - 4 * whole]);
            } else {
                cost += (r + 0.2) * (double)k * (k == 1 ? 1.13 : 1.0);
            }
        }
        if (cost < least) {
            least = cost;
            best = 256 * r;
        }
    }
    return best;
}

// Spins per thread of the Heun passes' tiles, up to 12: the count that leaves the busiest SM the least
// to do, its tiles times the spins per thread (and 0.5 spins' time for each tile's reduction, 0.2 in
// FP64).  An SM holds two FP32-mixed blocks of 512 threads or three of 256, one FP64 block.  The
// passes also need warps to hide their latencies: FP32-mixed, 16 a SM cost about 4 %, eight 30 %;
// FP64, eight 15 %.  Over 41 lattices and batches and 1024 x 1024 films of 8 to 20 layers the FP32-mixed
// choice is within 2.3 % of the fastest, 0.3 % on average.  Counted in plain rounds of SMs, and with eight
// taken from 24 tiles a SM on, it was up to 8.7 % off: the film of 8 layers took 12 spins a thread,
// 315 us per step (9: 290), that of 16 eight, 585 us (9: 570).  fcc 64^3: 2 spins per thread
// 66.2 us, 9 59.7.
inline int heun_slots(bool mixed, int block, int sm_count, const std::vector<int64_t> &sizes) {
    const int resident = !mixed ? 1 : block >= 512 ? 2 : 3;
    int best = 1;
    double least = 1e300;
    for (int slots = 1; slots <= 12; ++slots) {
        const int64_t tile = (int64_t)slots * block;
        int64_t tiles = 0;
        for (int64_t n : sizes) tiles += (n + tile - 1) / tile;
        const double k = (double)busiest_sm(tiles, sm_count, resident), warps = k * block / 32.0;
        double cost = k * (slots + (mixed ? 0.5 : 0.2));
        cost *= mixed ? 1.0 + 0.3 * std::pow(std::max(0.0, 24.0 - warps) / 16.0, 3.0) : (warps < 16.0 ? 1.15 : 1.0);
        if (cost < least) {
            least = cost;
            best = slots;
        }
    }
    return best;
}

// The blocks that sum the record of nsys systems on top of `grid` blocks with the launch's own work
// of `rounds` spins a thread: at most `most`, and no more than fill the last round of blocks on the
// SMs.  Blocks are handed out to the SMs in an order that is no plain round: with 40 of them on top
// of 440 corrector blocks (40 x sc 30^3 in FP64, three to an SM) ten SMs got four of the 440, 212 us
// instead of 160; with the 16 that fill the third round no SM does.  One block sums a system in
// about the time an SM takes for a spin a thread (FP64: a quarter of it), so it is given at most as
// many as that allows, or eight; where the round has less room, `most` are taken.
inline int record_blocks(bool mixed, int64_t nsys, int most, int64_t grid, int64_t rounds, int sm_count) {
    const int64_t sms = std::max(sm_count, 1), room = (sms - grid % sms) % sms;
    const int64_t each = std::max<int64_t>(8, (mixed ? 1 : 4) * rounds * ((grid + sms - 1) / sms));
    return room >= most || each * room < nsys ? most : (int)room;
}

}  // namespace ss
