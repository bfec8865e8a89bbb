// Long rows as packed bonds in slices of 32 rows (the sliced pass, k_rows_sell): where a spin lies
// in that pass's copy of the spins, and the host code that builds the slices.  Plain C++ but for
// the mark below, so that the layout can be built and checked without a GPU.
#pragma once
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <type_traits>
#include <unordered_map>
#include <vector>

#ifdef __CUDACC__
#define SS_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define SS_HOST_DEVICE inline
#endif

namespace ss {

// The classes of a period: spins i = b, b + period, ... of each b, one class after the other, each
// padded to whole slices.  The first `rest` classes have hi slices, the others lo.  Fewer than 2^24
// positions.
struct Classes {
    int32_t period, rest, hi, lo;
    static Classes of(int64_t n, int period) {
        return Classes{period, (int32_t)(n % period), (int32_t)((n / period + 1 + 31) / 32),
                       (int32_t)((n / period + 31) / 32)};
    }
    // First slice of class b (b = period: their number).
    SS_HOST_DEVICE int32_t first(int32_t b) const {
        const int32_t over = b - rest;
        return over <= 0 ? b * hi : rest * hi + over * lo;
    }
    int64_t slices() const { return first(period); }
    // Position of spin i.
    SS_HOST_DEVICE int64_t pos(int64_t i) const {
        if (period == 1) return i;
        const uint32_t c = (uint32_t)i / (uint32_t)period, b = (uint32_t)i - c * (uint32_t)period;
        return 32 * (int64_t)first((int32_t)b) + c;
    }
};

// A slice: the distinct slice that holds its words, and its first row.
struct alignas(8) SliceRef {
    int32_t form, row;
};

// The distinct J_ij / mu_s,i of the bonds (at most 255 beside 0, which is always there, for padding),
// the entry of 0, and each bond's entry (if asked for).  False with more.
template <typename R>
bool bond_dictionary(const std::vector<R> &J, int64_t nnz, std::vector<R> &dict, int &zero, std::vector<uint8_t> *bid) {
    using Bits = typename std::conditional<sizeof(R) == 8, uint64_t, uint32_t>::type;
    constexpr int kSlots = 1024;
    std::vector<Bits> key(kSlots);
    std::vector<int> id(kSlots, -1);
    Bits last = 0;
    dict.clear();
    if (bid) bid->resize((size_t)nnz);
    zero = -1;
    for (int64_t k = 0; k < nnz; ++k) {
        Bits b;
        std::memcpy(&b, &J[k], sizeof(R));
        if (k > 0 && b == last) {  // (bonds of a row mostly repeat)
            if (bid) (*bid)[(size_t)k] = (*bid)[(size_t)k - 1];
            continue;
        }
        last = b;
        uint32_t hsh = (uint32_t)(((uint64_t)b * 0x9E3779B97F4A7C15ull) >> 54);  // 10 bits
        while (id[hsh] >= 0 && key[hsh] != b) hsh = (hsh + 1) & (kSlots - 1);
        if (id[hsh] < 0) {
            if (b != 0 && dict.size() - (zero >= 0 ? 1 : 0) == 255) return false;
            key[hsh] = b;
            id[hsh] = (int)dict.size();
            if (b == 0) zero = id[hsh];
            dict.push_back(J[k]);
        }
        if (bid) (*bid)[(size_t)k] = (uint8_t)id[hsh];
    }
    if (zero < 0) {
        zero = (int)dict.size();
        dict.push_back((R)0);
    }
    return true;
}

// The hash by which equal slices are found (their contents are compared as well).  Of every word: with
// a sample of them, slices that differ in a few bonds elsewhere (dilute impurities) all share a hash and
// each is compared with all the others (48,000 slices of 640 words: 41 s to pack, now 0.5 s).  Four lanes of
// two words, so that the products overlap: fcc 32^3 to 4a, 139 M bonds, is hashed in 0.07 s.
inline uint64_t slice_hash(const std::vector<uint32_t> &words) {
    constexpr uint64_t k = 0x9E3779B97F4A7C15ull;
    uint64_t lane[4] = {words.size(), 1, 2, 3};
    for (size_t q = 0; q + 8 <= words.size(); q += 8) {  // (a slice is a multiple of 32 words)
        uint64_t v[4];
        std::memcpy(v, words.data() + q, sizeof(v));
        for (int l = 0; l < 4; ++l) {
            const uint64_t m = (lane[l] ^ v[l]) * k;
            lane[l] = (m << 31) | (m >> 33);
        }
    }
    uint64_t hsh = 0;
    for (uint64_t l : lane) hsh = (hsh ^ l ^ (l >> 32)) * k;
    return hsh ^ (hsh >> 31);
}

// The slices of k_rows_sell.  Row l of a slice is its first row + l * period; bond k of row l is word
// 32 k + l: (position of the neighbour - that of the slice's first row, modulo 2^24) << 8 | the bond's
// dictionary entry, rows padded to the slice's longest with J = 0 bonds to themselves.  Slices with
// the same words share them: those of distinct slice f lie at words[off[f]] to words[off[f + 1]].
struct Slices {
    int period = 1;
    std::vector<SliceRef> slice;
    std::vector<int64_t> off;
    std::vector<uint32_t> words;  // (one unused word when no row has a bond)
};

// The period is the one of a few whose slices' bonds touch the fewest 128-byte lines of the spins'
// copy (a sample of the rows; a larger one has to be a tenth better), as long as the positions fit
// a bond word.  rp [n + 1], col and bid (dictionary entries) are the rows, zero the entry of J = 0.
inline int slice_period(int64_t n, const int32_t *rp, const int32_t *col) {
    int period = 1;
    int64_t least = INT64_MAX;
    for (int p : {1, 2, 3, 4, 6, 8}) {
        const Classes c = Classes::of(n, p);
        if (32 * c.slices() >= (int64_t(1) << 24) || p > n) continue;
        int64_t lines = 0;
        std::vector<int64_t> seen;
        for (int q = 0; q < 8; ++q) {  // slices spread over the rows, some of their bonds
            const int64_t i0 = (n - 1) * q / 8;
            int32_t len = INT32_MAX;
            for (int l = 0; l < 32 && i0 + (int64_t)l * p < n; ++l) len = std::min(len, rp[i0 + (int64_t)l * p + 1] - rp[i0 + (int64_t)l * p]);
            for (int32_t k = 0; k < len; k += 1 + len / 16) {
                seen.clear();
                for (int l = 0; l < 32 && i0 + (int64_t)l * p < n; ++l) seen.push_back(c.pos(col[rp[i0 + (int64_t)l * p] + k]) >> 3);
                std::sort(seen.begin(), seen.end());
                lines += std::unique(seen.begin(), seen.end()) - seen.begin();
            }
        }
        if (lines < least - least / 10) {
            least = lines;
            period = p;
        }
    }
    return period;
}

inline void pack_slices(int64_t n, const int32_t *rp, const int32_t *col, const uint8_t *bid, int zero, Slices &out) {
    const int period = slice_period(n, rp, col);
    const Classes c = Classes::of(n, period);
    const int64_t nsl = c.slices();
    std::vector<int32_t> pos((size_t)n);
    for (int32_t b = 0; b < period; ++b) {
        int32_t at = 32 * c.first(b);
        for (int64_t i = b; i < n; i += period) pos[(size_t)i] = at++;
    }
    out.period = period;
    out.slice.resize((size_t)nsl);
    out.off.assign(1, 0);
    std::vector<uint32_t> words, &sell = out.words;
    // Each slice's longest row, and the words if no two slices are alike (of the pages reserved for
    // them only those written are touched).
    std::vector<int32_t> longest((size_t)nsl, 0);
    size_t most = 0;
    for (int32_t b = 0; b < period; ++b)
        for (int64_t i = b, at = 32 * (int64_t)c.first(b); i < n; i += period, ++at)
            longest[(size_t)(at / 32)] = std::max(longest[(size_t)(at / 32)], rp[i + 1] - rp[i]);
    for (int32_t w : longest) most += 32 * (size_t)w;
    sell.reserve(most);
    std::unordered_multimap<uint64_t, int32_t> form_of;  // hash of a slice's words -> form (contents compared)
    for (int32_t b = 0; b < period; ++b) {
        for (int64_t s = c.first(b); s < c.first(b + 1); ++s) {
            const int64_t row0 = b + (int64_t)period * 32 * (s - c.first(b));
            const int32_t w = longest[(size_t)s];
            words.resize(32 * (size_t)w);
            const int32_t base = (int32_t)(32 * s);
            for (int l = 0; l < 32; ++l) {
                const int64_t i = row0 + (int64_t)l * period;
                const int32_t len = i < n ? rp[i + 1] - rp[i] : 0;
                const uint32_t pad = ((uint32_t)l << 8) | (uint32_t)zero;
                uint32_t *to = words.data() + l;
                const int32_t *cj = i < n ? col + rp[i] : nullptr;
                const uint8_t *bj = i < n ? bid + rp[i] : nullptr;
                for (int32_t k = 0; k < len; ++k) to[32 * (size_t)k] = ((uint32_t)(pos[(size_t)cj[k]] - base) << 8) | bj[k];
                for (int32_t k = len; k < w; ++k) to[32 * (size_t)k] = pad;
            }
            const uint64_t hsh = slice_hash(words);
            int32_t form = -1;
            const auto range = form_of.equal_range(hsh);
            for (auto it = range.first; it != range.second && form < 0; ++it) {
                const int64_t o = out.off[(size_t)it->second], len = out.off[(size_t)it->second + 1] - o;
                if (len == (int64_t)words.size() && std::equal(words.begin(), words.end(), sell.begin() + o)) form = it->second;
            }
            if (form < 0) {
                form = (int32_t)out.off.size() - 1;
                form_of.emplace(hsh, form);
                sell.insert(sell.end(), words.begin(), words.end());
                out.off.push_back((int64_t)sell.size());
            }
            out.slice[(size_t)s] = SliceRef{form, (int32_t)row0};
        }
    }
    if (sell.empty()) sell.push_back(0);
}

}  // namespace ss
