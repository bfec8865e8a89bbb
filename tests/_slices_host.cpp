// Host code of the library that needs no GPU, as plain C functions for tests/test_slices_host.py and
// tests/test_shape_host.py.
#include "ss_shape.h"
#include "ss_slices.h"

#include <new>

using namespace ss;

extern "C" {

// Packs the rows; sizes[] = (period, slices, distinct slices, words), nothing is copied out.
// Returns 0, or 1 when the host memory does not suffice.
int slices_pack(int64_t n, const int32_t *rp, const int32_t *col, const uint8_t *bid, int zero, Slices **out,
                int64_t sizes[4]) {
    *out = nullptr;
    Slices *s = new Slices;
    try {
        pack_slices(n, rp, col, bid, zero, *s);
    } catch (const std::bad_alloc &) {
        delete s;
        return 1;
    }
    sizes[0] = s->period;
    sizes[1] = (int64_t)s->slice.size();
    sizes[2] = (int64_t)s->off.size() - 1;
    sizes[3] = (int64_t)s->words.size();
    *out = s;
    return 0;
}

void slices_copy(const Slices *s, int32_t *slice, int64_t *off, uint32_t *words) {
    std::memcpy(slice, s->slice.data(), s->slice.size() * sizeof(SliceRef));
    std::memcpy(off, s->off.data(), s->off.size() * sizeof(int64_t));
    std::memcpy(words, s->words.data(), s->words.size() * sizeof(uint32_t));
}

void slices_free(Slices *s) { delete s; }

void slices_positions(int64_t n, int period, int64_t *pos) {
    const Classes c = Classes::of(n, period);
    for (int64_t i = 0; i < n; ++i) pos[i] = c.pos(i);
}

uint64_t slices_hash(const uint32_t *words, int64_t count) {
    return slice_hash(std::vector<uint32_t>(words, words + count));
}

// Entries of the dictionary, or -1 with too many; zero and each bond's entry.
int slices_dictionary(const float *J, int64_t nnz, float *dict, int *zero, uint8_t *bid) {
    std::vector<float> d;
    std::vector<uint8_t> b;
    if (!bond_dictionary<float>(std::vector<float>(J, J + nnz), nnz, d, *zero, bid ? &b : nullptr)) return -1;
    std::memcpy(dict, d.data(), d.size() * sizeof(float));
    if (bid) std::memcpy(bid, b.data(), b.size());
    return (int)d.size();
}

int64_t shape_mc_tile(int mixed, int sms, int sums_record, int nsys, const int64_t *class0, const int64_t *class1) {
    const std::vector<int64_t> t[2] = {std::vector<int64_t>(class0, class0 + nsys), std::vector<int64_t>(class1, class1 + nsys)};
    return mc_tile(mixed != 0, sms, sums_record != 0, t);
}

int shape_record_blocks(int mixed, int64_t nsys, int most, int64_t grid, int64_t rounds, int sms) {
    return record_blocks(mixed != 0, nsys, most, grid, rounds, sms);
}

int64_t shape_busiest_sm(int64_t tiles, int sms, int resident) { return busiest_sm(tiles, sms, resident); }

int shape_heun_slots(int mixed, int block, int sms, int nsys, const int64_t *sizes) {
    return heun_slots(mixed != 0, block, sms, std::vector<int64_t>(sizes, sizes + nsys));
}
}
