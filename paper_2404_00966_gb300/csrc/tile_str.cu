// Edit-distance filtering tiles: the 3-gram count bound over (node rows x
// queries) blocks.
//
// For strings the lower bounds of Lemma 1 / 2 prune little when the distances
// concentrate (random-like sequences), and most (query, row) pairs of the
// surviving leaves reach verification.  Before the bit-parallel DP, each pair
// is tested against the 3-gram count bound: the L1 distance between the
// strings' 3-gram bucket counts (qgram.cuh) is at most 6 times the edit distance
// (a substitution changes at most 3 of a string's 3-grams, an insertion or a
// deletion at most 2 old and 3 new ones; summing counts into buckets and
// capping them at 255 can only lower the L1 distance), so L1 > 6 t proves
// d > t.  The surviving (query, node) entries are regrouped by node; one CTA
// takes a block of up to 128 node rows (a lane holds four rows' 64-byte bucket
// vectors in registers) and the node's queries in chunks of 32 or 64 (their
// vectors in shared memory); a pair is kept if the row's leaf survived for the
// query, the row is visible at the query's sequence number and the bound does
// not exclude it.  Ranges that fill the blocks take tile_qtc.cu instead.  The
// kept pairs go on to the exact DP.
#include "gts_impl.cuh"
#include "metric.cuh"
#include "tile_str.cuh"

namespace gts {

namespace {

constexpr int kRowsS = 128;     // rows of one node block (the regrouping's block size)
constexpr int kThreadsS = 256;
constexpr int kWords = 16;      // 64 one-byte buckets as 16 words
constexpr int kGroups = kThreadsS / 32;   // query groups of a chunk, one per warp
constexpr int kRPL = kRowsS / 32;         // rows per lane: lane + 32 h

struct StrArgs {
    int F;
    const int32_t *npos, *nsize;
    int64_t lvl_last;
    const int64_t *row_del;
    int any_deleted;
    const uint8_t *qg;          // rows' bucket counts [n, 64]
    const uint8_t *qgq;         // queries' bucket counts [nq, 64]
    const TileRec *grec;
    const int32_t *gq;          // the records' queries
    const int4 *items;
    int64_t units;              // work units: item u / split, its query chunks u % split, + split, ...
    int split;
    int *work_counter;
    int32_t *out_q, *out_row;
    int64_t cap;
    unsigned long long *out_count;
};

__device__ __forceinline__ void cpa16s(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// l[h] += the L1 distances of the lane's first NH rows' counts and the query's
template <int NH>
__device__ __forceinline__ void add_l1(uint32_t (&l)[kRPL], const uint32_t (&rw)[kRPL][kWords], const uint4 *qv) {
#pragma unroll
    for (int v = 0; v < kWords / 4; ++v) {
        const uint4 x = qv[v];
#pragma unroll
        for (int h = 0; h < NH; ++h) l[h] = __vsadu4(rw[h][4 * v], x.x) + l[h];
#pragma unroll
        for (int h = 0; h < NH; ++h) l[h] = __vsadu4(rw[h][4 * v + 1], x.y) + l[h];
#pragma unroll
        for (int h = 0; h < NH; ++h) l[h] = __vsadu4(rw[h][4 * v + 2], x.z) + l[h];
#pragma unroll
        for (int h = 0; h < NH; ++h) l[h] = __vsadu4(rw[h][4 * v + 3], x.w) + l[h];
    }
}

// NQS: queries per chunk (32 or 64; a tuning parameter), NQS / 8 per warp.
// The ALU pipe bounds it: 16 four-byte sums of absolute differences per pair
// (19 T a second on the device, 60 of 64 lanes per SM and cycle: 1.9 * 10^10
// pairs cannot take less than 16 ms).  A warp therefore holds the whole block,
// four rows a lane: a query's 64 bytes are four 16-byte broadcast loads, each
// of which takes the shared-memory port four cycles to write back, and with
// two rows a lane (31.9 ms; now 31.4) or one (53.0) they held the kernel back.
// The sums
// start at -(limit + 1), so that the test is their sign bit, shifted into the
// pass masks; a block of at most 32 or 64 rows (small nodes) skips the lanes' empty
// rows (110 M pairs in nodes of 15 rows: 1.5 ms; a row a thread took 2.3); a
// chunk's records and vectors are copied while the one before is
// computed (the query ids they need are read two chunks ahead); and the leaf
// and visibility tests run on the few pairs that pass.
template <int NQS>
__global__ void __launch_bounds__(kThreadsS, 2) k_tile_qgram(StrArgs a) {
    constexpr int kPer = NQS / kGroups;
    __shared__ uint4 sQ[2][NQS][kWords / 4];
    __shared__ __align__(16) TileRec sRec[2][NQS];
    __shared__ int s_item;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cj = tid / 4, cw = tid & 3;   // the vector piece this thread copies (tid < 4 NQS)
    for (;;) {
        if (tid == 0) s_item = atomicAdd(a.work_counter, 1);
        __syncthreads();
        const int64_t unit = s_item;
        if (unit >= a.units) break;
        const int4 it = a.items[unit / a.split];
        const int part = (int)(unit % a.split);
        const int64_t g = a.lvl_last + it.x;
        const int first = it.y, total = it.z;
        // the unit's chunks: c = 0, 1, ..  is the node's chunk part + c split
        const int nchunk = ((total + NQS - 1) / NQS - part + a.split - 1) / a.split;
        if (nchunk <= 0) {
            __syncthreads();   // s_item is read by everyone
            continue;
        }
        auto begin = [&](int c) { return (part + c * a.split) * NQS; };
        // chunk c into buffer c & 1; qid: the query of this thread's piece
        auto query_of = [&](int c) -> int32_t {
            const int j = begin(c) + cj;
            return c < nchunk && cj < NQS && j < total ? a.gq[first + j] : -1;
        };
        auto stage = [&](int c, int32_t qid) {
            const int cnt = min(NQS, total - begin(c));
            if (qid >= 0)
                cpa16s(&sQ[c & 1][cj][cw], reinterpret_cast<const uint4 *>(a.qgq + (int64_t)qid * 64) + cw);
            if (tid < 2 * cnt)
                cpa16s(reinterpret_cast<uint4 *>(&sRec[c & 1][0]) + tid,
                       reinterpret_cast<const uint4 *>(a.grec + first + begin(c)) + tid);
        };
        const int32_t qid0 = query_of(0);
        int32_t qnext = query_of(1);
        const int rb = it.w * kRowsS;
        const int32_t pos = a.npos[g], size = a.nsize[g];
        const int nrow = min(kRowsS, size - rb);
        const int32_t avg = size / a.F;
        stage(0, qid0);
        // this lane's rows: bucket counts, leaf bits, delete marks
        uint32_t rw[kRPL][kWords];
        uint64_t rowbit[kRPL], any = 0;
#pragma unroll
        for (int h = 0; h < kRPL; ++h) {
            const int r = lane + 32 * h;
            const bool valid = r < nrow;
            const int64_t row = (int64_t)pos + (valid ? rb + r : 0);
            int32_t jl = avg > 0 ? (rb + r) / avg : a.F - 1;
            if (jl > a.F - 1) jl = a.F - 1;
            rowbit[h] = valid ? (1ull << jl) : 0ull;
            any |= rowbit[h];
            const uint4 *src = reinterpret_cast<const uint4 *>(a.qg + row * 64);
#pragma unroll
            for (int v = 0; v < kWords / 4; ++v) {
                const uint4 x = src[v];
                rw[h][4 * v] = x.x;
                rw[h][4 * v + 1] = x.y;
                rw[h][4 * v + 2] = x.z;
                rw[h][4 * v + 3] = x.w;
            }
        }
        // the leaves of the block's rows: a query that kept none of them is passed over
        const uint64_t wmask = (uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)any) |
                               ((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(any >> 32)) << 32);
        for (int c = 0; c < nchunk; ++c) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();   // chunk c has landed; the other buffer is no longer read
            if (c + 1 < nchunk) {
                stage(c + 1, qnext);
                qnext = query_of(c + 2);
            }
            const int cnt = min(NQS, total - begin(c));
            const TileRec *rec = sRec[c & 1];
            const int j0 = warp * kPer;
            const int nj = max(0, min(kPer, cnt - j0));
            // lane i < nj: query j0 + i's limit (keep iff L1 <= 6 t, whole
            // numbers; an unbounded t keeps all) and whether the warp's rows
            // hold a leaf it kept
            int start = 0;
            bool live = false;
            if (lane < nj) {
                const float t = rec[j0 + lane].thr;
                start = -1 - (t < 1e8f ? (int)(6.f * t) : 1 << 30);
                live = (rec[j0 + lane].mask & wmask) != 0;
            }
            const unsigned lives = __ballot_sync(0xffffffffu, live);
            uint32_t pass = 0;   // bit 8 h + nj - 1 - i: row lane + 32 h passes query j0 + i
            for (int i = 0; i < nj; ++i) {
                uint32_t l[kRPL] = {0u, 0u, 0u, 0u};
                if ((lives >> i) & 1u) {   // warp-uniform
                    const uint32_t s0 = (uint32_t)__shfl_sync(0xffffffffu, start, i);
                    const uint4 *qv = sQ[c & 1][j0 + i];
                    l[0] = s0;
                    if (nrow > 64) {
                        l[1] = l[2] = l[3] = s0;
                        add_l1<4>(l, rw, qv);
                    } else if (nrow > 32) {
                        l[1] = s0;
                        add_l1<2>(l, rw, qv);
                    } else {
                        add_l1<1>(l, rw, qv);
                    }
                }
                // (nj <= 8: a row's bits stay inside its byte)
                pass = (pass << 1) | (l[0] >> 31) | ((l[1] >> 31) << 8) | ((l[2] >> 31) << 16) | ((l[3] >> 31) << 24);
            }
            if (__any_sync(0xffffffffu, pass != 0)) {
                for (uint32_t left = pass; left; left &= left - 1) {   // leaf and visibility of the passing pairs
                    const int b = __ffs(left) - 1, h = b >> 3;
                    const TileRec &rc = rec[j0 + nj - 1 - (b & 7)];
                    const uint64_t rbit = h == 0 ? rowbit[0] : h == 1 ? rowbit[1] : h == 2 ? rowbit[2] : rowbit[3];
                    if (!(rc.mask & rbit) || (a.any_deleted && a.row_del[(int64_t)pos + rb + lane + 32 * h] <= rc.seq))
                        pass &= ~(1u << b);
                }
                const int np = __popc(pass);
                int incl = np;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += v;
                }
                const int wtot = __shfl_sync(0xffffffffu, incl, 31);
                if (wtot > 0) {
                    unsigned long long base = 0;
                    if (lane == 31) base = atomicAdd(a.out_count, (unsigned long long)wtot);
                    base = __shfl_sync(0xffffffffu, base, 31);
                    unsigned long long o = base + (unsigned long long)(incl - np);
                    while (pass) {
                        const int b = __ffs(pass) - 1;
                        pass &= pass - 1;
                        if ((int64_t)o < a.cap) {
                            a.out_q[o] = rec[j0 + nj - 1 - (b & 7)].q;
                            a.out_row[o] = pos + rb + lane + 32 * (b >> 3);
                        }
                        ++o;
                    }
                }
            }
        }
    }
}

// ---- short strings: filter and distance in one tile
//
// For words the 3-gram bound excludes little (two words of ten letters differ
// in at most 16 3-grams, 6 t passes that at t = 3), and nearly every pair went
// through a candidate list, a sort by query and a verification pass: 3.3 ms
// for 50 M pairs, of which the distances themselves need 0.4 ms.  Here a
// thread holds one row of the block, its text (eight words) and its 3-gram
// counts, the chunk's queries have their match masks in shared memory (one word
// per character and query), and a pair costs 13 operations per character of
// its row; only pairs within the threshold are written, with their distance.
// The integer / logic pipe bounds it.
constexpr int kNQD = 32;        // queries per chunk
struct ShortArgs {
    StrArgs s;
    const uint8_t *S, *QS;
    const int64_t *Soff, *QSoff;
    int max_len;
    float *out_d;
};

__global__ void __launch_bounds__(kThreadsS, 3) k_tile_short(ShortArgs A) {
    const StrArgs &a = A.s;
    constexpr int kPer = kNQD / 2;
    __shared__ __align__(16) uint32_t sPeq[kNQD][256];
    __shared__ uint4 sQ[kNQD][kWords / 4];
    __shared__ TileRec sRec[kNQD];
    __shared__ int sLen[kNQD];
    __shared__ int s_item;
    const int tid = threadIdx.x, lane = tid & 31;
    const int r = tid % kRowsS, half = tid / kRowsS;
    for (;;) {
        if (tid == 0) s_item = atomicAdd(a.work_counter, 1);
        __syncthreads();
        const int64_t unit = s_item;
        if (unit >= a.units) break;
        const int4 it = a.items[unit / a.split];
        const int part = (int)(unit % a.split);
        const int64_t g = a.lvl_last + it.x;
        const int first = it.y, total = it.z;
        const int rb = it.w * kRowsS;
        const int32_t pos = a.npos[g], size = a.nsize[g];
        const bool valid = rb + r < size;
        const int64_t row = (int64_t)pos + (valid ? rb + r : 0);
        const int32_t avg = size / a.F;
        int32_t jl = avg > 0 ? (rb + r) / avg : a.F - 1;
        if (jl > a.F - 1) jl = a.F - 1;
        const uint64_t rowbit = valid ? (1ull << jl) : 0ull;
        const int64_t rdel = (valid && a.any_deleted) ? a.row_del[row] : kNever;
        const int len = (int)(A.Soff[row + 1] - A.Soff[row]);
        const int wlen = __reduce_max_sync(0xffffffffu, len);   // the warp's longest row
        uint32_t tw[kShortStr / 4], rw[kWords];
        {
            TextWords tr(A.S + A.Soff[row], len);
#pragma unroll
            for (int i = 0; i < kShortStr / 4; ++i) tw[i] = 4 * i < len ? tr.next4() : 0u;
            const uint4 *src = reinterpret_cast<const uint4 *>(a.qg + row * 64);
#pragma unroll
            for (int v = 0; v < kWords / 4; ++v) {
                const uint4 x = src[v];
                rw[4 * v] = x.x;
                rw[4 * v + 1] = x.y;
                rw[4 * v + 2] = x.z;
                rw[4 * v + 3] = x.w;
            }
        }
        for (int c0 = part * kNQD; c0 < total; c0 += a.split * kNQD) {
            const int cnt = min(kNQD, total - c0);
            __syncthreads();   // the previous chunk's shared data is no longer read
            for (int i = tid; i < kNQD * 64; i += kThreadsS)
                reinterpret_cast<uint4 *>(&sPeq[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
            const int qj = tid >> 3;   // eight threads a query
            int32_t q = -1;
            int m = 0;
            if (qj < cnt) {
                q = a.gq[first + c0 + qj];
                m = (int)(A.QSoff[q + 1] - A.QSoff[q]);
                if ((tid & 7) == 0) {
                    sRec[qj] = a.grec[first + c0 + qj];
                    sLen[qj] = m;
                }
                if ((tid & 7) >= 4)
                    sQ[qj][tid & 3] = reinterpret_cast<const uint4 *>(a.qgq + (int64_t)q * 64)[tid & 3];
            }
            __syncthreads();
            if (q >= 0) {
                const uint8_t *p = A.QS + A.QSoff[q];
                for (int i = tid & 7; i < m; i += 8) atomicOr(&sPeq[qj][p[i]], 1u << i);
            }
            __syncthreads();
            const int j0 = half * kPer, j1 = min(j0 + kPer, cnt);
            for (int j = j0; j < j1; ++j) {
                const TileRec &rc = sRec[j];
                const int mq = sLen[j];
                const int lim = rc.thr < 1e8f ? (int)rc.thr : 1 << 24;
                bool on = (rc.mask & rowbit) && rdel > rc.seq && abs(mq - len) <= lim;
                // the 3-gram bound, where it can exclude anything
                if (6 * (int64_t)lim < mq + A.max_len - 4) {
                    uint32_t l1 = 0;
#pragma unroll
                    for (int v = 0; v < kWords / 4; ++v) {
                        const uint4 x = sQ[j][v];
                        l1 = __vsadu4(rw[4 * v], x.x) + l1;
                        l1 = __vsadu4(rw[4 * v + 1], x.y) + l1;
                        l1 = __vsadu4(rw[4 * v + 2], x.z) + l1;
                        l1 = __vsadu4(rw[4 * v + 3], x.w) + l1;
                    }
                    on = on && l1 <= 6u * (uint32_t)lim;
                }
                int d = 1 << 25;
                if (on) {
                    uint32_t Pv = ~0u, Mv = 0u;
                    const uint32_t *peq = sPeq[j];
#pragma unroll
                    for (int v = 0; v < kShortStr / 4; ++v) {
                        if (4 * v >= wlen) break;
#pragma unroll
                        for (int i = 4 * v; i < 4 * v + 4; ++i) {
                            if (i < len) {
                                const uint32_t Eq = peq[(tw[v] >> (8 * (i % 4))) & 255u];
                                const uint32_t Xh = (((Eq & Pv) + Pv) ^ Pv) | Eq;
                                const uint32_t Ph = ((Mv | ~(Xh | Pv)) << 1) | 1u;
                                const uint32_t Mh = (Pv & Xh) << 1;
                                const uint32_t Xv = Eq | Mv;
                                Pv = Mh | ~(Xv | Ph);
                                Mv = Ph & Xv;
                            }
                        }
                    }
                    const uint32_t rows = mq >= 32 ? ~0u : (1u << mq) - 1u;
                    d = len + __popc(Pv & rows) - __popc(Mv & rows);
                }
                const unsigned b = __ballot_sync(0xffffffffu, d <= lim);
                if (b) {
                    unsigned long long base = 0;
                    if (lane == 0) base = atomicAdd(a.out_count, (unsigned long long)__popc(b));
                    base = __shfl_sync(0xffffffffu, base, 0);
                    const unsigned long long o = base + __popc(b & ((1u << lane) - 1u));
                    if (((b >> lane) & 1u) && (int64_t)o < a.cap) {
                        a.out_q[o] = rc.q;
                        a.out_row[o] = (int32_t)row;
                        A.out_d[o] = (float)d;
                    }
                }
            }
        }
        __syncthreads();
    }
}

// parts of an item's query chunks: more than one while there are fewer than four
// units per resident CTA (5,000 words in 20 nodes, 2,000 queries: 40 blocks of rows)
int chunk_parts(int64_t items, int64_t resident, int64_t nq, int chunk) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((nq + chunk - 1) / chunk, (4 * resident + items - 1) / items));
}

StrArgs str_args(const Tree &t, const StrQuery &sq, const TcRegroup &rg, int64_t i0, int64_t i1, int split) {
    StrArgs a;
    a.F = t.F;
    a.npos = t.npos.get();
    a.nsize = t.nsize.get();
    a.lvl_last = t.lvl_off[rg.h - 1];
    a.row_del = t.row_del.get();
    a.any_deleted = sq.any_deleted;
    a.qg = sq.qg;
    a.qgq = sq.qgq;
    a.grec = rg.grec.get();
    a.gq = rg.gq.get();
    a.items = rg.items.get() + i0;
    a.units = (i1 - i0) * split;
    a.split = split;
    return a;
}

}  // namespace

int64_t short_run(const Tree &t, const StrQuery &sq, const ShortQuery &hq, const TcRegroup &rg, int64_t i0, int64_t i1,
                  DBuf<int32_t> &out_q, DBuf<int32_t> &out_row, DBuf<float> &out_d, int64_t cap_hint, int64_t most,
                  int *launches, cudaStream_t st) {
    *launches = 0;
    if (i1 <= i0) return 0;
    int dev = 0, sms = 0, per_sm = 0;
    GTS_CUDA(cudaGetDevice(&dev));
    GTS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    GTS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tile_short, kThreadsS, 0));
    if (per_sm < 1) per_sm = 1;
    const int64_t resident = (int64_t)sms * per_sm;
    const int split = chunk_parts(i1 - i0, resident, sq.nq, kNQD);
    const int64_t grid = std::min<int64_t>((i1 - i0) * split, resident);
    DBuf<int> counter(1, st);
    DBuf<unsigned long long> count(1, st);
    int64_t cap = cap_hint > 0 ? cap_hint : 1 << 20;
    for (int attempt = 0; attempt < 2; ++attempt) {
        out_q.alloc(cap, st);
        out_row.alloc(cap, st);
        out_d.alloc(cap, st);
        GTS_CUDA(cudaMemsetAsync(counter.get(), 0, 4, st));
        GTS_CUDA(cudaMemsetAsync(count.get(), 0, 8, st));
        ShortArgs A;
        A.s = str_args(t, sq, rg, i0, i1, split);
        A.s.work_counter = counter.get();
        A.s.out_q = out_q.get();
        A.s.out_row = out_row.get();
        A.s.cap = cap;
        A.s.out_count = count.get();
        A.S = hq.S;
        A.Soff = hq.Soff;
        A.max_len = hq.max_len;
        A.QS = hq.QS;
        A.QSoff = hq.QSoff;
        A.out_d = out_d.get();
        k_tile_short<<<(unsigned)grid, kThreadsS, 0, st>>>(A);
        ++*launches;
        check_launch("short-string tile");
        unsigned long long hcount = 0;
        GTS_CUDA(cudaMemcpyAsync(&hcount, count.get(), 8, cudaMemcpyDeviceToHost, st));
        GTS_CUDA(cudaStreamSynchronize(st));
        if ((int64_t)hcount <= cap || (int64_t)hcount > most) return (int64_t)hcount;
        cap = (int64_t)hcount;   // rerun with room for every pair
    }
    GTS_REQUIRE(false, GTS_ECUDA, "short-string tile: output count changed between identical runs");
    return 0;
}

int64_t qgram_run(const Tree &t, const StrQuery &sq, const TcRegroup &rg, int64_t i0, int64_t i1, DBuf<int32_t> &out_q,
                  DBuf<int32_t> &out_row, int64_t cap_hint, int64_t most, int *launches, cudaStream_t st) {
    *launches = 0;
    if (i1 <= i0) return 0;
    int dev = 0, sms = 0;
    GTS_CUDA(cudaGetDevice(&dev));
    GTS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    int per_sm = 0;
    if (sq.queries == 32)
        GTS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tile_qgram<32>, kThreadsS, 0));
    else
        GTS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tile_qgram<64>, kThreadsS, 0));
    if (per_sm < 1) per_sm = 1;
    const int64_t resident = (int64_t)sms * per_sm;
    const int split = chunk_parts(i1 - i0, resident, sq.nq, sq.queries == 32 ? 32 : 64);
    const int64_t grid = std::min<int64_t>((i1 - i0) * split, resident);
    DBuf<int> counter(1, st);
    DBuf<unsigned long long> count(1, st);
    int64_t cap = cap_hint > 0 ? cap_hint : 1 << 20;
    for (int attempt = 0; attempt < 2; ++attempt) {
        out_q.alloc(cap, st);
        out_row.alloc(cap, st);
        GTS_CUDA(cudaMemsetAsync(counter.get(), 0, 4, st));
        GTS_CUDA(cudaMemsetAsync(count.get(), 0, 8, st));
        StrArgs a = str_args(t, sq, rg, i0, i1, split);
        a.work_counter = counter.get();
        a.out_q = out_q.get();
        a.out_row = out_row.get();
        a.cap = cap;
        a.out_count = count.get();
        if (sq.queries == 32)
            k_tile_qgram<32><<<(unsigned)grid, kThreadsS, 0, st>>>(a);
        else
            k_tile_qgram<64><<<(unsigned)grid, kThreadsS, 0, st>>>(a);
        ++*launches;
        check_launch("3-gram tile");
        unsigned long long hcount = 0;
        GTS_CUDA(cudaMemcpyAsync(&hcount, count.get(), 8, cudaMemcpyDeviceToHost, st));
        GTS_CUDA(cudaStreamSynchronize(st));
        if ((int64_t)hcount <= cap || (int64_t)hcount > most) return (int64_t)hcount;
        cap = (int64_t)hcount;   // rerun with room for every pair
    }
    GTS_REQUIRE(false, GTS_ECUDA, "3-gram tile: output count changed between identical runs");
    return 0;
}

}  // namespace gts
