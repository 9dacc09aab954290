// The 3-gram counts behind the edit-distance filters: letter classes and
// buckets.  Plain C++ where no CUDA compiler reads it, so that the bound can be
// checked on the CPU with the functions that the kernels use.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define GTS_HD __host__ __device__ __forceinline__
#else
#define GTS_HD inline
#endif

namespace gts {

// A lower bound for edit distance from the counts of the strings' 3-grams
// (Ukkonen 1992, q-gram distance): a substitution changes at most 3 of a
// string's 3-grams and an insertion or deletion at most 2 old and 3 new ones,
// so the L1 distance between the two 3-gram count vectors is at most 6 times
// the edit distance.  Counting the 3-grams of letter classes instead of letters
// (64 buckets, sums of the exact counts) and capping a count can only lower that
// L1 distance, so L1(buckets) > 6 t proves d > t, whatever the classes are.
constexpr int kQgBuckets = 64;
constexpr int kQgCap = 255;

// The classes only decide how sharp the bound is: four classes of letters that
// occur about equally often spread the 3-grams over all 64 buckets.  The letters,
// most frequent first, go one by one to the class with the fewest occurrences so
// far: A, C, G and T get a class each, 0 and 1 two of them.  (Fixed classes by two
// bits of the letter put 0 and 1 into one, so that their strings differed in
// nothing but length; a multiplicative hash of the three bytes left a third of
// the buckets empty on DNA.  Pairs of 9,000 x 120 strings of 70 letters that limit 42
// keeps, these classes / two bits / hash, 18,000 of them related: digits 18,927 /
// 21,335 / 18,074, ACGT 18,401 / 18,401 / 52,534, a-z 18,614 / 18,303 / 18,046.  2,000
// digit strings against 200,000: two bits 0.78 ms, these 0.70.)  Letters that were not counted keep those two bits.
// order: the letters by falling count.
GTS_HD void letter_classes(const uint32_t *count, const uint8_t *order, uint8_t *cls) {
    uint64_t load[4] = {0, 0, 0, 0};
    for (int i = 0; i < 256; ++i) {
        const int c = order[i];
        if (count[c] == 0) {
            cls[c] = (uint8_t)((c >> 1) & 3);
            continue;
        }
        int best = 0;
        for (int k = 1; k < 4; ++k)
            if (load[k] < load[best]) best = k;
        load[best] += count[c];
        cls[c] = (uint8_t)best;
    }
}

// the bucket of the 3-gram that ends with a letter of class c, from the bucket
// of the one before
GTS_HD uint32_t next_bucket(uint32_t bucket, uint32_t c) { return ((bucket << 2) | c) & (kQgBuckets - 1); }

// the counts (saturating) of a string's 3-grams; h zeroed by the caller
GTS_HD void qgram_counts(const uint8_t *s, int64_t len, const uint8_t *cls, uint8_t *h) {
    uint32_t b = 0;
    for (int64_t j = 0; j < len; ++j) {
        b = next_bucket(b, cls[s[j]]);
        if (j >= 2 && h[b] < kQgCap) ++h[b];
    }
}

// The tensor-core filter's code: levels 1 .. of each bucket's count, 249 places
constexpr int kQgPlaces = 249;
GTS_HD constexpr int code_levels(int bucket) { return 3 * kQgBuckets + bucket < kQgPlaces ? 4 : 3; }

}  // namespace gts
