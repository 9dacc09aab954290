// L2 verification tiles in FP32 on the CUDA cores: declarations for the
// search driver.
#pragma once

#include "gts_impl.cuh"
#include "tile_tc.cuh"

namespace gts {

struct L2fQuery {
    const float *Q = nullptr;     // the batch's queries [nq, dim]
    float absf = 0.f;             // absolute slack of every FP32 distance bound
    int any_deleted = 1;
};

// every FP32 vector set under L2 (dimension and alignment only choose the copy width)
bool l2f_tiles_supported(const Tree &t);
// run the tiles of a regrouping's items [i0, i1); returns the number of (query,
// row) pairs written: a superset of the pairs within the records' thresholds.
// More than `most`: their number, nothing usable is written.
int64_t l2f_run(const Tree &t, const L2fQuery &lq, int64_t nq, const TcRegroup &rg, int64_t i0, int64_t i1,
                DBuf<int32_t> &out_q, DBuf<int32_t> &out_row, int64_t cap_hint, int64_t most, int *launches,
                cudaStream_t st);

}  // namespace gts
