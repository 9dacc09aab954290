// Edit-distance filtering tiles (3-gram count bound): declarations for the
// search driver.
#pragma once

#include "gts_impl.cuh"
#include "tile_tc.cuh"

namespace gts {

struct StrQuery {
    const uint8_t *qg = nullptr;    // the tree rows' 3-gram bucket counts [n, 64]
    const uint8_t *qgq = nullptr;   // the batch's queries' [nq, 64]
    int64_t nq = 0;                 // queries of the batch
    int any_deleted = 1;
    int queries = 64;               // queries per tile chunk: 32 or 64
};

// Both sides at most 32 characters: the tiles also run the edit distance itself
// (one 32-bit word per column) on the pairs the bound keeps.
constexpr int kShortStr = 32;

struct ShortQuery {
    const uint8_t *S = nullptr;     // the tree rows' bytes and offsets
    const int64_t *Soff = nullptr;
    int max_len = 0;                // the longest row
    const uint8_t *QS = nullptr;    // the queries'
    const int64_t *QSoff = nullptr;
};

// The tiles run the items [i0, i1) of a regrouping and return the number of pairs
// written; more than `most`: their number, nothing usable is written.

// over a regrouping of short strings: the (query, row, distance) triples within
// the records' thresholds
int64_t short_run(const Tree &t, const StrQuery &sq, const ShortQuery &hq, const TcRegroup &rg, int64_t i0, int64_t i1,
                  DBuf<int32_t> &out_q, DBuf<int32_t> &out_row, DBuf<float> &out_d, int64_t cap_hint, int64_t most,
                  int *launches, cudaStream_t st);

// the (query, row) pairs that the bound keeps (the records carry each query's
// threshold)
int64_t qgram_run(const Tree &t, const StrQuery &sq, const TcRegroup &rg, int64_t i0, int64_t i1, DBuf<int32_t> &out_q,
                  DBuf<int32_t> &out_row, int64_t cap_hint, int64_t most, int *launches, cudaStream_t st);

// The same bound on the tensor cores (tile_qtc.cu), with the counts capped at
// 4: keeps every pair that qgram_run keeps and a few more.  256-byte codes of the
// rows and of the batch's queries (thr: their thresholds; rows: null).
constexpr int64_t kQtcRows = 1 << 24;    // rows whose codes are kept with the index (4 GiB)
constexpr int64_t kQtcPairs = 32 << 20;  // least (entry, row) pairs
bool qtc_pays(const Tree &t, int64_t nq, const TcRegroup &rg);
void qtc_codes(const uint8_t *qg, int64_t n, const float *thr, uint8_t *code, cudaStream_t st);
int64_t qtc_run(const Tree &t, const StrQuery &sq, const TcRegroup &rg, int64_t i0, int64_t i1, int64_t nq,
                const uint8_t *xcode, const uint8_t *qcode, DBuf<int32_t> &out_q, DBuf<int32_t> &out_row,
                int64_t cap_hint, int64_t most, int *launches, cudaStream_t st);

}  // namespace gts
