// Edit-distance filtering tiles on the tensor cores: the 3-gram count bound of
// tile_str.cu for ranges whose (node rows x queries) blocks are well filled (kNN's
// first thresholds exclude little, and every pair kept is looked up).
//
// The L1 distance of two strings' bucket counts, each capped at 4, is the
// Hamming distance of their thermometer codes (bucket b, level l: one if the
// count is at least l), and that is |A| + |B| - 2 A.B for the codes' numbers of
// ones and their dot product: a contraction.  Capping only lowers the L1
// distance, so the bound (L1 <= 6 d) stays one, and nearly as sharp (random
// reads of 108, limit 48: 4.3e-5 of the pairs pass, 1.9e-5 uncapped); the pairs
// kept go on to the uncapped bound and the exact DP as before.
//
// A string's code takes 256 bytes of e4m3: 249 levels (the fourth level of the
// last seven buckets is left out, which lowers the distance only) and seven
// places that fold the test into the product: digits of |A| against -1/2, -4,
// -32, and the digits of 6 t - |B| against 1/2, 4, 32, and 1/4, so that
//     D = A.B - |A| / 2 + (6 t - |B|) / 2 + 1/4
// is at least 1/4 for a pair that the bound keeps and at most -1/4 otherwise:
// its sign bit decides.  Every product is a multiple of 1/4 and every partial sum
// lies below 2^10, so the FP32 accumulation is exact in any order.
//
// What bounds it: 10^6 reads of 108 x 20,000 queries, 2 * 10^10 pairs of 256
// places, 3.9 ms = 2.6 PFLOP/s (the byte-wise sums of tile_str.cu: 31.4 ms, at
// the rate of the integer units).  With the two accumulators' epilogues on the
// same eight warps, 32 columns at a time, they held the MMAs back: 5.0 ms.
// Layout: a unit of work is two 128-row blocks of nodes (A, by TMA) against the
// windows of 256 consecutive queries that either node has an entry in (B, by
// TMA, two buffers; loaded once for both blocks, since reading B from L2 once
// per block would take longer than the MMAs).  One thread issues per window and
// block eight 128 x 256 x 32 MMAs from shared memory into the block's TMEM
// accumulator; while the other block's run, the block's own eight epilogue warps
// read it and look for a clear sign bit (one logic operation per two pairs).  The few pairs
// found wait in a queue per warp until 32 of them look up their entry's record
// (leaf mask, sequence number) together.
#include <cuda_fp8.h>

#include "gts_impl.cuh"
#include "qgram.cuh"
#include "tc.cuh"
#include "tile_str.cuh"

namespace gts {

namespace {

constexpr int kRowsQ = 128;      // rows of a block (MMA M)
constexpr int kWinQ = 256;       // queries of a window (MMA N)
constexpr int kCode = 256;       // bytes of a string's code: two panels of 128
constexpr int kPlaces = kQgPlaces;   // of them levels; then |A|'s digits, the constants
constexpr int kEpiQ = 8;         // epilogue warps of each block
constexpr int kThreadsQ = (4 + 2 * kEpiQ) * 32;   // warp 0 producer, 1 MMA, 2 TMEM, 4.. epilogue
constexpr int kABytes = kRowsQ * kCode, kBBytes = kWinQ * kCode;
constexpr int kDescs = 4;        // window descriptors: the epilogue is at most two windows behind
constexpr int kQueue = 64;
constexpr int kMaxLim = 512;     // limits at or above |A| + |B| keep every pair

struct Window {
    int32_t stop, new_unit, last, w;
};
struct Block {
    int32_t row0, nrow, rb, node, size;
};

struct QtcArgs {
    int F, any_deleted;
    const int32_t *npos, *nsize;
    int64_t lvl_last, nq, nw, nwin;
    const int64_t *row_del;
    const uint32_t *wany;        // [nodes, ceil(nwin / 32)]: the node's non-empty windows
    const uint32_t *bits;        // node x query bitmap
    const int32_t *wpre;
    const int64_t *noff;
    const TileRec *grec;
    const int4 *items;
    int64_t n_items;
    int split;                   // parts of a pair of items' windows
    int *work_counter;
    int32_t *out_q, *out_row;
    int64_t cap;
    unsigned long long *out_count;
    int *status;
};

__device__ __forceinline__ uint8_t e4m3(float v) { return __nv_cvt_float_to_fp8(v, __NV_SATFINITE, __NV_E4M3); }

// The codes, a warp per string; thr (queries): the thresholds t, null for rows.
__global__ void k_codes(const uint8_t *__restrict__ qg, int64_t n, const float *__restrict__ thr,
                        uint8_t *__restrict__ code) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const uint8_t one = e4m3(1.f);
    for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < n; i += nwarps) {
        const int c0 = qg[i * 64 + lane], c1 = qg[i * 64 + 32 + lane];
        uint8_t *o = code + i * kCode;
        const bool fourth = code_levels(32 + lane) == 4;   // this lane's second bucket has its fourth level
        const int ones = __reduce_add_sync(0xffffffffu, min(c0, 4) + min(c1, fourth ? 4 : 3));
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            o[l * 64 + lane] = c0 > l ? one : 0;
            if (l < 3 || fourth) o[l * 64 + 32 + lane] = c1 > l ? one : 0;
        }
        if (!fourth) {
            const int p = 3 * 64 + 32 + lane - kPlaces;   // 0 .. 6
            const float w = p % 3 == 0 ? 0.5f : p % 3 == 1 ? 4.f : 32.f;
            float v;
            if (p == 6) {
                v = 0.5f;
            } else if (thr) {
                const float t = thr[i];
                const int lim = t < (float)kMaxLim ? max((int)(6.f * t), -8) : kMaxLim;
                const int s = min(lim, kMaxLim) - ones, a = abs(s);
                const int dg = p == 3 ? a & 7 : p == 4 ? (a >> 3) & 7 : a >> 6;
                v = p < 3 ? -w : (float)(s < 0 ? -dg : dg);
            } else {
                const int dg = p == 0 ? ones & 7 : p == 1 ? (ones >> 3) & 7 : ones >> 6;
                v = p < 3 ? (float)dg : w;
            }
            o[kPlaces + p] = e4m3(v);
        }
    }
}

// the nodes' non-empty windows as bits: a thread per (node, 32 windows)
__global__ void k_windows_any(const uint32_t *__restrict__ bits, int64_t nn, int64_t nw, int64_t nwin,
                              uint32_t *__restrict__ wany) {
    const int64_t per = (nwin + 31) / 32;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nn * per; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t node = i / per, c0 = (i % per) * 32;
        uint32_t m = 0;
        for (int c = 0; c < 32; ++c)
            for (int j = 0; j < kWinQ / 32; ++j) {
                const int64_t w = (c0 + c) * (kWinQ / 32) + j;
                if (w < nw && bits[node * nw + w]) m |= 1u << c;
            }
        wany[i] = m;
    }
}

__device__ __forceinline__ void mma_e4m3(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__global__ void __launch_bounds__(kThreadsQ, 1)
    k_tile_qgram_tc(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_q, QtcArgs a) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sA = smem;                       // two blocks
    uint8_t *sB = smem + 2 * kABytes;         // two windows
    __shared__ __align__(8) uint64_t b_full[2], b_empty[2], acc_full[2], acc_empty[2], d_full[kDescs], a_full, a_empty;
    __shared__ Window s_win[kDescs];
    __shared__ Block s_blk[kDescs][2];
    __shared__ int4 s_queue[2 * kEpiQ][kQueue];   // query, row, node, leaf bit
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 2) tc::tmem_alloc(&s_tmem, 512);
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&b_full[i], 1);
            tc::mbar_init(&b_empty[i], 1);
            tc::mbar_init(&acc_full[i], 1);
            tc::mbar_init(&acc_empty[i], kEpiQ);
        }
        for (int i = 0; i < kDescs; ++i) tc::mbar_init(&d_full[i], 1);
        tc::mbar_init(&a_full, 1);
        tc::mbar_init(&a_empty, 1);
        tc::mbar_fence_init();
        s_abort = 0;
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = s_tmem;
    auto fail = [&](int code) {
        s_abort = 1;
        atomicExch(a.status, code);
    };

    if (warp == 0) {
        // ================================================= producer
        if (lane == 0) {
            const int64_t units = (a.n_items + 1) / 2 * a.split;
            const int64_t per = (a.nwin + 31) / 32;
            uint32_t k = 0, unit = 0;   // windows and units handed on
            bool ok = true;
            // window w (or the end) into the next buffer
            auto emit = [&](const Window &win) -> bool {
                const int b = k & 1;
                if (k >= 2 && !tc::mbar_wait(&b_empty[b], ((k - 2) >> 1) & 1)) {
                    fail(1);
                    return false;
                }
                s_win[k % kDescs] = win;
                if (win.stop) {
                    tc::mbar_arrive(&b_full[b]);
                } else {
                    tc::mbar_expect_tx(&b_full[b], kBBytes);
                    tc::tma_load_3d(sB + b * kBBytes, &map_q, 0, win.w * kWinQ, 0, &b_full[b]);
                }
                tc::mbar_arrive(&d_full[k % kDescs]);
                ++k;
                return true;
            };
            while (ok && !s_abort) {
                const int64_t u = atomicAdd(a.work_counter, 1);
                if (u >= units) break;
                const int64_t i0 = u / a.split * 2;
                const int part = (int)(u % a.split);
                const int64_t w0 = a.nwin * part / a.split, w1 = a.nwin * (part + 1) / a.split;
                Block blk[2];
                for (int b = 0; b < 2; ++b) {
                    const bool has = i0 + b < a.n_items;   // (an odd last item: its block twice, the second without rows)
                    const int4 it = a.items[has ? i0 + b : i0];
                    blk[b].node = it.x;
                    blk[b].size = a.nsize[a.lvl_last + it.x];
                    blk[b].rb = it.w * kRowsQ;
                    blk[b].row0 = a.npos[a.lvl_last + it.x] + blk[b].rb;
                    blk[b].nrow = has ? min(kRowsQ, blk[b].size - blk[b].rb) : 0;
                }
                bool first = true;
                // (the unit's data before its first window's descriptor; four
                // slots: the epilogue has finished window k - 4)
                auto hand_on = [&](int64_t w, bool last) -> bool {
                    if (first) {
                        s_blk[unit % kDescs][0] = blk[0];
                        s_blk[unit % kDescs][1] = blk[1];
                    }
                    if (!emit({0, first ? 1 : 0, last ? 1 : 0, (int32_t)w})) return false;
                    if (first) {
                        if (unit > 0 && !tc::mbar_wait(&a_empty, (unit - 1) & 1)) {
                            fail(2);
                            return false;
                        }
                        tc::mbar_expect_tx(&a_full, 2 * kABytes);
                        tc::tma_load_3d(sA, &map_x, 0, blk[0].row0, 0, &a_full);
                        tc::tma_load_3d(sA + kABytes, &map_x, 0, blk[1].row0, 0, &a_full);
                        ++unit;
                    }
                    first = false;
                    return true;
                };
                int64_t pend = -1;   // a window found and not handed on yet
                for (int64_t c = w0 / 32; ok && c * 32 < w1; ++c) {
                    uint32_t m = a.wany[blk[0].node * per + c] | a.wany[blk[1].node * per + c];
                    while (ok && m) {
                        const int64_t w = c * 32 + __ffs(m) - 1;
                        m &= m - 1;
                        if (w < w0 || w >= w1) continue;
                        if (pend >= 0) ok = hand_on(pend, false);
                        pend = w;
                    }
                }
                if (ok && pend >= 0) ok = hand_on(pend, true);
            }
            const uint32_t loaded = k;
            if (ok) emit({1, 0, 0, 0});
            if (s_abort) {   // copies in flight land before the kernel ends
                for (uint32_t j = loaded > 2 ? loaded - 2 : 0; j < loaded; ++j)
                    tc::mbar_wait(&b_full[j & 1], (j >> 1) & 1);
                if (unit > 0) tc::mbar_wait(&a_full, (unit - 1) & 1);
            }
        }
    } else if (warp == 1) {
        // ================================================= MMA issuer
        if (lane == 0) {
            const uint32_t idesc = (1u << 4) | ((uint32_t)(kWinQ >> 3) << 17) | ((uint32_t)(kRowsQ >> 4) << 24);
            const uint64_t da = tc::sdesc_k_sw128(tc::smem_u32(sA)), db = tc::sdesc_k_sw128(tc::smem_u32(sB));
            uint32_t unit = 0, k = 0;
            int64_t last[2] = {-1, -1};   // the last window issued for each block
            for (;; ++k) {
                const int b = k & 1;
                if (!tc::mbar_wait(&b_full[b], (k >> 1) & 1)) {
                    fail(3);
                    break;
                }
                const Window win = s_win[k % kDescs];
                if (win.stop || s_abort) break;
                if (win.new_unit) {
                    if (!tc::mbar_wait(&a_full, unit & 1)) {
                        fail(4);
                        break;
                    }
                    ++unit;
                }
                bool ok = true;
                for (int blk = 0; blk < 2; ++blk) {
                    if (k > 0 && !tc::mbar_wait(&acc_empty[blk], (k - 1) & 1)) {
                        fail(5);
                        ok = false;
                        break;
                    }
                    tc::tc_fence_after();
#pragma unroll
                    for (int s = 0; s < kCode / 32; ++s) {
                        // panel s / 4, 32-byte step s % 4 within its 128-byte rows
                        const uint64_t ao = (uint64_t)((blk * kABytes + (s >> 2) * kRowsQ * 128 + (s & 3) * 32) >> 4);
                        const uint64_t bo = (uint64_t)((b * kBBytes + (s >> 2) * kWinQ * 128 + (s & 3) * 32) >> 4);
                        mma_e4m3(tmem + (uint32_t)(blk * kWinQ), da + ao, db + bo, idesc, s > 0);
                    }
                    tc::mma_commit(&acc_full[blk]);
                    last[blk] = k;
                }
                if (!ok) break;
                tc::mma_commit(&b_empty[b]);
                if (win.last) tc::mma_commit(&a_empty);
            }
            // issued MMAs end before TMEM is released
            if (s_abort)
                for (int blk = 0; blk < 2; ++blk)
                    if (last[blk] >= 0) tc::mbar_wait(&acc_full[blk], (uint32_t)(last[blk] & 1));
        }
    } else if (warp >= 4) {
        // ================================================= epilogue
        const int quad = warp & 3, half = ((warp - 4) >> 2) & 1, blk = (warp - 4) / kEpiQ;
        const int r = quad * 32 + lane;                     // row of the block
        int4 *queue = s_queue[warp - 4];
        int queued = 0;                                     // warp-uniform
        uint32_t unit = 0;
        bool valid = false;
        int32_t row = 0, node = 0, leaf = 0;
        // the first n queued pairs: entry, leaf, visibility
        auto flush = [&](int n) {
            __syncwarp();
            bool keep = false;
            int4 e = make_int4(0, 0, 0, 0);
            if (lane < n) {
                e = queue[lane];
                const int64_t wi = (int64_t)e.z * a.nw + (e.x >> 5);
                const uint32_t word = a.bits[wi], bit = 1u << (e.x & 31);
                if (word & bit) {
                    const TileRec rc = a.grec[a.noff[e.z] + a.wpre[wi] + __popc(word & (bit - 1u))];
                    keep = ((rc.mask >> e.w) & 1ull) && !(a.any_deleted && a.row_del[e.y] <= rc.seq);
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            if (m) {
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(a.out_count, (unsigned long long)__popc(m));
                base = __shfl_sync(0xffffffffu, base, 0) + __popc(m & ((1u << lane) - 1u));
                if (keep && (int64_t)base < a.cap) {
                    a.out_q[base] = e.x;
                    a.out_row[base] = e.y;
                }
            }
            __syncwarp();
        };
        for (uint32_t k = 0;; ++k) {
            if (!tc::mbar_wait(&d_full[k % kDescs], (k / kDescs) & 1)) {
                fail(6);
                break;
            }
            const Window win = s_win[k % kDescs];
            if (win.stop || s_abort) break;
            if (win.new_unit) {
                const Block bl = s_blk[unit % kDescs][blk];
                valid = r < bl.nrow;
                row = bl.row0 + r;
                node = bl.node;
                const int32_t avg = bl.size / a.F;
                leaf = min(avg > 0 ? (bl.rb + r) / avg : a.F - 1, a.F - 1);
                ++unit;
            }
            if (!tc::mbar_wait(&acc_full[blk], k & 1)) {
                fail(7);
                break;
            }
            tc::tc_fence_after();
            const uint32_t acc = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(blk * kWinQ + half * (kWinQ / 2));
            // 64 columns at a time
            for (int g = 0; g < kWinQ / 128; ++g) {
                uint32_t v[2][32];
                tc::tmem_ld32(acc + 64 * g, v[0]);
                tc::tmem_ld32(acc + 64 * g + 32, v[1]);
                tc::tmem_ld_wait();
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int64_t q0 = (int64_t)win.w * kWinQ + half * (kWinQ / 2) + 64 * g + 32 * u;
                    uint32_t all = v[u][0];
#pragma unroll
                    for (int i = 1; i < 32; ++i) all &= v[u][i];
                    if (!__any_sync(0xffffffffu, valid && !(all >> 31)) || q0 >= a.nq) continue;
                    uint32_t pass = 0;
#pragma unroll
                    for (int i = 0; i < 32; ++i) pass |= (~v[u][i] >> 31) << i;
                    if (q0 + 32 > a.nq) pass &= (1u << (a.nq - q0)) - 1u;   // (no queries past the batch)
                    if (!valid) pass = 0;
                    for (unsigned act = __ballot_sync(0xffffffffu, pass != 0); act;
                         act = __ballot_sync(0xffffffffu, pass != 0)) {
                        if (pass) {
                            const int i = __ffs(pass) - 1;
                            pass &= pass - 1;
                            queue[queued + __popc(act & ((1u << lane) - 1u))] =
                                make_int4((int32_t)q0 + i, row, node, leaf);
                        }
                        queued += __popc(act);
                        if (queued >= 32) {
                            flush(32);
                            const int4 e = lane < queued - 32 ? queue[32 + lane] : make_int4(0, 0, 0, 0);
                            __syncwarp();
                            queue[lane] = e;
                            queued -= 32;
                            __syncwarp();
                        }
                    }
                }
            }
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&acc_empty[blk]);
        }
        if (queued > 0) flush(queued);
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == 2) tc::tmem_dealloc(tmem, 512);
}

}  // namespace

bool qtc_pays(const Tree &t, int64_t nq, const TcRegroup &rg) {
    if (rg.nw == 0 || rg.n_items == 0 || t.n > kQtcRows) return false;
    const int64_t win = (nq + kWinQ - 1) / kWinQ;
    // the integer units take 1.6 ps a pair, the tensor cores 0.25 ps a place of the
    // windows
    return rg.n_pairs >= kQtcPairs && rg.n_pairs * 6 >= std::min(t.n, rg.n_items * kRowsQ) * win * kWinQ;
}

void qtc_codes(const uint8_t *qg, int64_t n, const float *thr, uint8_t *code, cudaStream_t st) {
    k_codes<<<(unsigned)std::min<int64_t>((n + 7) / 8, 1 << 16), 256, 0, st>>>(qg, n, thr, code);
    check_launch("3-gram codes");
}

int64_t qtc_run(const Tree &t, const StrQuery &sq, const TcRegroup &rg, int64_t i0, int64_t i1, int64_t nq,
                const uint8_t *xcode, const uint8_t *qcode, DBuf<int32_t> &out_q, DBuf<int32_t> &out_row,
                int64_t cap_hint, int64_t most, int *launches, cudaStream_t st) {
    *launches = 0;
    const int64_t n_items = i1 - i0;
    if (n_items <= 0) return 0;
    int dev = 0, sms = 0;
    GTS_CUDA(cudaGetDevice(&dev));
    GTS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    constexpr int smem = 2 * kABytes + 2 * kBBytes + 1024;
    GTS_CUDA(cudaFuncSetAttribute(k_tile_qgram_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    const int64_t nwin = (nq + kWinQ - 1) / kWinQ, pairs = (n_items + 1) / 2;
    // at least four units per SM where the windows allow it
    const int split = (int)std::max<int64_t>(1, std::min<int64_t>(nwin, (4 * sms + pairs - 1) / pairs));
    const int64_t nodes = t.lvl_off[rg.h] - t.lvl_off[rg.h - 1];
    const int64_t per = (nwin + 31) / 32;
    DBuf<uint32_t> wany(nodes * per, st);
    k_windows_any<<<(unsigned)std::min<int64_t>((nodes * per + 255) / 256, 1 << 16), 256, 0, st>>>(
        rg.bits.get(), nodes, rg.nw, nwin, wany.get());
    ++*launches;
    const CUtensorMap map_x = tc_byte_map(xcode, t.n, kRowsQ), map_q = tc_byte_map(qcode, nq, kWinQ);
    DBuf<int> counter(2, st);   // work counter, status
    DBuf<unsigned long long> count(1, st);
    int64_t cap = cap_hint > 0 ? cap_hint : 1 << 20;
    for (int attempt = 0; attempt < 2; ++attempt) {
        out_q.alloc(cap, st);
        out_row.alloc(cap, st);
        GTS_CUDA(cudaMemsetAsync(counter.get(), 0, 8, st));
        GTS_CUDA(cudaMemsetAsync(count.get(), 0, 8, st));
        QtcArgs a;
        a.F = t.F;
        a.any_deleted = sq.any_deleted;
        a.npos = t.npos.get();
        a.nsize = t.nsize.get();
        a.lvl_last = t.lvl_off[rg.h - 1];
        a.nq = nq;
        a.nw = rg.nw;
        a.nwin = nwin;
        a.row_del = t.row_del.get();
        a.wany = wany.get();
        a.bits = rg.bits.get();
        a.wpre = rg.wpre.get();
        a.noff = rg.noff.get();
        a.grec = rg.grec.get();
        a.items = rg.items.get() + i0;
        a.n_items = n_items;
        a.split = split;
        a.work_counter = counter.get();
        a.out_q = out_q.get();
        a.out_row = out_row.get();
        a.cap = cap;
        a.out_count = count.get();
        a.status = counter.get() + 1;
        k_tile_qgram_tc<<<(unsigned)std::min<int64_t>(pairs * split, sms), kThreadsQ, smem, st>>>(map_x, map_q, a);
        ++*launches;
        check_launch("3-gram tensor-core tile");
        unsigned long long hcount = 0;
        int hstatus = 0;
        GTS_CUDA(cudaMemcpyAsync(&hcount, count.get(), 8, cudaMemcpyDeviceToHost, st));
        GTS_CUDA(cudaMemcpyAsync(&hstatus, a.status, 4, cudaMemcpyDeviceToHost, st));
        GTS_CUDA(cudaStreamSynchronize(st));
        GTS_REQUIRE(hstatus == 0, GTS_ETIMEOUT,
                    "3-gram tensor-core tile: a bounded mbarrier wait ran out (status " + std::to_string(hstatus) + ")");
        if ((int64_t)hcount <= cap || (int64_t)hcount > most) return (int64_t)hcount;
        cap = (int64_t)hcount;   // rerun with room for every pair
    }
    GTS_REQUIRE(false, GTS_ECUDA, "3-gram tensor-core tile: output count changed between identical runs");
    return 0;
}

}  // namespace gts
