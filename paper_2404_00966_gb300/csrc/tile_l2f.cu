// L2 verification tiles in FP32 on the CUDA cores (GTS_PREC_FP32).
//
// The surviving (query, last-level node) entries are regrouped by node, as for
// the tensor-core and L1 tiles, and one CTA computes the product form
//     d~^2 = |q|^2 + |x|^2 - 2 q.x
// of up to 128 node rows against up to 128 of the node's queries at once, all
// in FP32.  A pair is kept only if the row's leaf survived for the query, the
// row is visible and a proven lower bound of its distance is within the
// query's threshold; the kept pairs then take the same FP32 distance (sum of
// squared differences) and FP64 recheck as every candidate of the plain path,
// so the answers and their distances are the plain path's, bit for bit.
//
// What bounds it: the FP32 pipe, one fused multiply-add per coordinate of a
// pair (the difference form needs two operations), 152 SMs x 128 lanes.  A
// candidate at a time (a warp per pair, k_verify_vec) every pair reads its
// object row from L2 again: 10^6 x 128, 2,000 queries, k = 10: 58.4 ms for
// the two table scans and the verification of 390 M candidates.
// Layout: thread (lane, warp) holds the sums of rows lane + 32 i (i < 4) for
// queries warp * QPT + j; a chunk of at most 32, 64 or 128 queries takes QPT =
// 4, 8 or 16, so that a short chunk keeps all eight warps busy.  Both operands
// stream through shared memory in slices of 32 coordinates (asynchronous
// copies, double-buffered): per 4 coordinates a warp issues 4 + QPT 16-byte
// shared loads for 16 QPT fused multiply-adds.
//
// Error bound, u = 2^-24: the FP32 sum s of D products (fused multiply-adds,
// any order) and the norms lie within gamma_D = D u / (1 - D u) relative to
// |q||x|, |q|^2 and |x|^2 (Higham, 2nd ed., 3.1), so
//     |d~^2 - d^2| <= 2 gamma_D (|q|^2 + |x|^2)
// (2 |q||x| <= |q|^2 + |x|^2), and the test's own few operations add at most
// 12 u (|q|^2 + |x|^2) plus a relative 4 u of the threshold's square.  With
// c = 2.2 (D + 16) u a pair may be dropped if
//     (1 - c)(|q|^2 + |x|^2) - 2 s > t^2,
// t the threshold with its absolute slack, enlarged by 1e-6.  Norms above
// 1e36 (whose squares or sums could overflow) drop nothing.
#include "gts_impl.cuh"
#include "metric.cuh"
#include "tile_l2f.cuh"

namespace gts {

namespace {

constexpr int kRowsF = 128;     // rows of one node block (the regrouping's block size)
constexpr int kNQF = 128;       // queries of one chunk, at most
constexpr int kThreadsF = 256;
constexpr int kRPTF = 4;        // rows per thread: lane + 32 i
constexpr int kKCF = 32;        // coordinates per pipeline stage
constexpr int kLdF = kKCF + 4;  // padded shared-memory row stride (floats): conflict-free 16-byte loads

struct L2fArgs {
    int dim, F;
    const float *X;             // rows in leaf order [n, dim]
    const float *Q;             // queries [nq, dim]
    const float *qn2;           // their squared norms
    const int64_t *row_del;
    const int32_t *npos, *nsize;
    int64_t lvl_last;
    const TileRec *grec;
    const int4 *items;
    int64_t units;              // work units: item u / split, its chunks u % split, + split, ...
    int split;
    int *work_counter;
    int32_t *out_q, *out_row;
    int64_t cap;
    unsigned long long *out_count;
    float c, absf;              // the bound's coefficient, the thresholds' absolute slack
    int any_deleted;
};

__device__ __forceinline__ uint32_t saddr_f(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// asynchronous copies of 16 and of 4 bytes; with valid == false nothing is
// read and the destination is filled with zeros
__device__ __forceinline__ void cpa16(void *dst, const void *src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(saddr_f(dst)), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cpa4(void *dst, const void *src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(saddr_f(dst)), "l"(src), "r"(valid ? 4 : 0)
                 : "memory");
}

// Copy coordinates [k0, k0 + 32) of the block's rows and of the chunk's
// queries (NQ = 8 QPT of them); coordinates past dim and rows / queries past
// the block are zeros.  V16: rows start on 16-byte boundaries.
template <int NQ, bool V16>
__device__ __forceinline__ void stage_f(const L2fArgs &a, int64_t row0, int nrow, const int32_t *sq, int cnt, int k0,
                                        float *sX, float *sQ) {
    const int tid = threadIdx.x;
    if (V16) {
#pragma unroll
        for (int c = tid; c < kRowsF * (kKCF / 4); c += kThreadsF) {
            const int r = c >> 3, ch = c & 7, k = k0 + ch * 4;
            const bool v = r < nrow && k < a.dim;
            cpa16(sX + r * kLdF + ch * 4, v ? a.X + (row0 + r) * a.dim + k : a.X, v);
        }
#pragma unroll
        for (int c = tid; c < NQ * (kKCF / 4); c += kThreadsF) {
            const int j = c >> 3, ch = c & 7, k = k0 + ch * 4;
            const bool v = j < cnt && k < a.dim;
            cpa16(sQ + j * kLdF + ch * 4, v ? a.Q + (int64_t)sq[j] * a.dim + k : a.Q, v);
        }
    } else {
#pragma unroll 4
        for (int c = tid; c < kRowsF * kKCF; c += kThreadsF) {
            const int r = c >> 5, ch = c & 31, k = k0 + ch;
            const bool v = r < nrow && k < a.dim;
            cpa4(sX + r * kLdF + ch, v ? a.X + (row0 + r) * a.dim + k : a.X, v);
        }
#pragma unroll 4
        for (int c = tid; c < NQ * kKCF; c += kThreadsF) {
            const int j = c >> 5, ch = c & 31, k = k0 + ch;
            const bool v = j < cnt && k < a.dim;
            cpa4(sQ + j * kLdF + ch, v ? a.Q + (int64_t)sq[j] * a.dim + k : a.Q, v);
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// The stage's products for M of the block's four 32-row groups (group idx[i]
// of each at rows + 32 idx[i]) and the warp's QPT queries.
template <int QPT, int M>
__device__ __forceinline__ void stage_products(float (&acc)[kRPTF][QPT], const float *xs, const float *qs,
                                               const int (&idx)[kRPTF]) {
#pragma unroll 1
    for (int kk = 0; kk < kKCF; kk += 4) {
        float4 xv[M];
#pragma unroll
        for (int i = 0; i < M; ++i) xv[i] = *reinterpret_cast<const float4 *>(xs + idx[i] * (32 * kLdF) + kk);
#pragma unroll
        for (int j = 0; j < QPT; ++j) {
            const float4 qv = *reinterpret_cast<const float4 *>(qs + j * kLdF + kk);
#pragma unroll
            for (int i = 0; i < M; ++i) {
                acc[i][j] = fmaf(xv[i].x, qv.x, acc[i][j]);
                acc[i][j] = fmaf(xv[i].y, qv.y, acc[i][j]);
                acc[i][j] = fmaf(xv[i].z, qv.z, acc[i][j]);
                acc[i][j] = fmaf(xv[i].w, qv.w, acc[i][j]);
            }
        }
    }
}

struct BlockF {          // one node block
    int64_t row0;
    int nrow;
    bool norms;          // the rows' norms are still to be formed (the block's first chunk)
};

// One chunk of cnt <= 8 QPT queries (records sRec[0 .. cnt), limits sLim).
template <int QPT, bool V16>
__device__ __forceinline__ void chunk_f(const L2fArgs &a, const BlockF &blk, int cnt, float *sX, float *sQ,
                                        const TileRec *sRec, const float *sLim, const int32_t *sQid,
                                        const uint64_t *sRowBit, const int64_t *sRowDel, float *sAx) {
    constexpr int NQ = 8 * QPT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nstage = (a.dim + kKCF - 1) / kKCF;
    // (10^6 x 128, 2,000 queries: 10.6 -> 8.8 ms a call, this kernel 5.0)
    // the 32-row groups that hold a leaf some query of the warp kept (queries
    // come in the order of their region, so a warp's queries keep much the
    // same leaves), compacted to the first m places of idx: warp-uniform
    int idx[kRPTF] = {0, 0, 0, 0}, m = 0;
    {
        const int mine = min(QPT, cnt - warp * QPT);
        const uint64_t mk = lane < mine ? sRec[warp * QPT + lane].mask : 0ull;
        const uint64_t kept = (uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)mk) |
                              ((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(mk >> 32)) << 32);
#pragma unroll
        for (int g = 0; g < kRPTF; ++g) {
            if (__any_sync(0xffffffffu, (sRowBit[lane + 32 * g] & kept) != 0)) {
#pragma unroll
                for (int i = 0; i < kRPTF; ++i)
                    if (i == m) idx[i] = g;
                ++m;
            }
        }
    }
    const bool active = m > 0;
    float acc[kRPTF][QPT];
#pragma unroll
    for (int i = 0; i < kRPTF; ++i)
#pragma unroll
        for (int j = 0; j < QPT; ++j) acc[i][j] = 0.f;
    float rn = 0.f;   // the norm of half of row tid / 2's coordinates
    stage_f<NQ, V16>(a, blk.row0, blk.nrow, sQid, cnt, 0, sX, sQ);
    for (int s = 0; s < nstage; ++s) {
        const int b = s & 1;
        if (s + 1 < nstage) {
            stage_f<NQ, V16>(a, blk.row0, blk.nrow, sQid, cnt, (s + 1) * kKCF, sX + (b ^ 1) * kRowsF * kLdF,
                             sQ + (b ^ 1) * kNQF * kLdF);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        if (blk.norms) {
            const float *xr = sX + b * kRowsF * kLdF + (tid >> 1) * kLdF + (tid & 1) * (kKCF / 2);
#pragma unroll
            for (int k = 0; k < kKCF / 2; k += 4) {
                const float4 v = *reinterpret_cast<const float4 *>(xr + k);
                rn = fmaf(v.x, v.x, rn);
                rn = fmaf(v.y, v.y, rn);
                rn = fmaf(v.z, v.z, rn);
                rn = fmaf(v.w, v.w, rn);
            }
        }
        if (active) {
            const float *xs = sX + b * kRowsF * kLdF + lane * kLdF;
            const float *qs = sQ + b * kNQF * kLdF + warp * QPT * kLdF;
            if (m == 4) stage_products<QPT, 4>(acc, xs, qs, idx);
            else if (m == 3) stage_products<QPT, 3>(acc, xs, qs, idx);
            else if (m == 2) stage_products<QPT, 2>(acc, xs, qs, idx);
            else stage_products<QPT, 1>(acc, xs, qs, idx);
        }
        __syncthreads();   // the buffer is refilled next stage
    }
    if (blk.norms) {   // (1 - c) |x|^2; a norm near overflow drops nothing
        rn += __shfl_xor_sync(0xffffffffu, rn, 1);
        if ((tid & 1) == 0) sAx[tid >> 1] = rn <= 1e36f ? (1.f - a.c) * rn : __int_as_float(0xff800000);
        __syncthreads();
    }
    // ---- epilogue: distance bound, leaf and visibility tests; emit kept pairs
    uint64_t pass = 0;
    if (active) {
        float ax[kRPTF];
#pragma unroll
        for (int i = 0; i < kRPTF; ++i) ax[i] = sAx[lane + 32 * idx[i]];
#pragma unroll
        for (int j = 0; j < QPT; ++j) {
            const int jj = warp * QPT + j;
            if (jj >= cnt) break;
            const float lim = sLim[jj];
#pragma unroll
            for (int i = 0; i < kRPTF; ++i)
                if (i < m && !(fmaf(-2.f, acc[i][j], ax[i]) > lim)) pass |= 1ull << (i * QPT + j);   // (a NaN is kept)
        }
        if (pass) {
            uint64_t left = pass;
            while (left) {
                const int b = __ffsll((long long)left) - 1;
                left &= left - 1;
                const int gi = b / QPT;
                const int r = lane + 32 * (gi == 0 ? idx[0] : gi == 1 ? idx[1] : gi == 2 ? idx[2] : idx[3]);
                const TileRec &rc = sRec[warp * QPT + b % QPT];
                if (!(rc.mask & sRowBit[r]) || sRowDel[r] <= rc.seq) pass &= ~(1ull << b);
            }
        }
    }
    const int np = __popcll(pass);
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
            const int b = __ffsll((long long)pass) - 1;
            pass &= pass - 1;
            if ((int64_t)o < a.cap) {
                const int gi = b / QPT;
                a.out_q[o] = sQid[warp * QPT + b % QPT];
                a.out_row[o] = (int32_t)(blk.row0 + lane +
                                         32 * (gi == 0 ? idx[0] : gi == 1 ? idx[1] : gi == 2 ? idx[2] : idx[3]));
            }
            ++o;
        }
    }
}

template <bool V16>
__global__ void __launch_bounds__(kThreadsF, 2) k_tile_l2f(L2fArgs a) {
    extern __shared__ __align__(16) float smem_f[];
    float *sX = smem_f;                                  // 2 x [128][kLdF]
    float *sQ = sX + 2 * kRowsF * kLdF;                  // 2 x [128][kLdF]
    TileRec *sRec = reinterpret_cast<TileRec *>(sQ + 2 * kNQF * kLdF);   // [128]
    float *sLim = reinterpret_cast<float *>(sRec + kNQF);                 // [128]
    int32_t *sQid = reinterpret_cast<int32_t *>(sLim + kNQF);            // [128]
    __shared__ uint64_t sRowBit[kRowsF];
    __shared__ int64_t sRowDel[kRowsF];
    __shared__ float sAx[kRowsF];
    __shared__ int s_unit;
    const int tid = threadIdx.x;
    for (;;) {
        if (tid == 0) s_unit = atomicAdd(a.work_counter, 1);
        __syncthreads();
        const int64_t unit = s_unit;
        if (unit >= a.units) break;
        const int4 it = a.items[unit / a.split];
        const int part = (int)(unit % a.split);
        const int64_t g = a.lvl_last + it.x;
        const int first = it.y, total = it.z;
        const int rb = it.w * kRowsF;
        const int32_t pos = a.npos[g], size = a.nsize[g];
        BlockF blk;
        blk.nrow = min(kRowsF, size - rb);
        blk.row0 = (int64_t)pos + rb;
        blk.norms = true;
        // per-row constants: leaf bit within the node (even split, remainder
        // in the last child) and delete mark
        if (tid < kRowsF) {
            const int32_t avg = size / a.F;
            int32_t jl = avg > 0 ? (rb + tid) / avg : a.F - 1;
            if (jl > a.F - 1) jl = a.F - 1;
            sRowBit[tid] = tid < blk.nrow ? (1ull << jl) : 0ull;
            sRowDel[tid] = (tid < blk.nrow && a.any_deleted) ? a.row_del[blk.row0 + tid] : kNever;
        }
        for (int c0 = part * kNQF; c0 < total; c0 += a.split * kNQF) {
            const int cnt = min(kNQF, total - c0);
            for (int j = tid; j < cnt; j += kThreadsF) {
                const TileRec rc = a.grec[first + c0 + j];
                sRec[j] = rc;
                sQid[j] = rc.q;
                const float q2 = a.qn2[rc.q];
                const float t = (rc.thr + a.absf) * (1.f + 1e-6f);
                // (an overflowing limit keeps every pair)
                sLim[j] = q2 <= 1e36f && t <= 1e18f ? t * t * (1.f + 1e-6f) - (1.f - a.c) * q2 + 1e-30f
                                                    : __int_as_float(0x7f800000);
            }
            __syncthreads();
            if (cnt <= 32)
                chunk_f<4, V16>(a, blk, cnt, sX, sQ, sRec, sLim, sQid, sRowBit, sRowDel, sAx);
            else if (cnt <= 64)
                chunk_f<8, V16>(a, blk, cnt, sX, sQ, sRec, sLim, sQid, sRowBit, sRowDel, sAx);
            else
                chunk_f<16, V16>(a, blk, cnt, sX, sQ, sRec, sLim, sQid, sRowBit, sRowDel, sAx);
            blk.norms = false;
            __syncthreads();   // sRec / sQid are rewritten by the next chunk
        }
        __syncthreads();       // s_unit is read by everyone (a unit may hold no chunk)
    }
}

// squared norms of the queries, a warp each
__global__ void k_query_norms(const float *__restrict__ Q, int64_t nq, int dim, float *__restrict__ n2) {
    const int lane = threadIdx.x & 31;
    const int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (q >= nq) return;
    float s = 0.f;
    for (int i = lane; i < dim; i += 32) s = fmaf(Q[q * dim + i], Q[q * dim + i], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) n2[q] = s;
}

size_t l2f_smem_bytes() {
    return (size_t)(2 * kRowsF * kLdF + 2 * kNQF * kLdF) * 4 + (size_t)kNQF * (sizeof(TileRec) + 4 + 4);
}

}  // namespace

bool l2f_tiles_supported(const Tree &t) {
    return t.metric == GTS_L2 && t.dim > 0 && t.n > 0 && t.n < ((int64_t)1 << 31);
}

int64_t l2f_run(const Tree &t, const L2fQuery &lq, int64_t nq, const TcRegroup &rg, int64_t i0, int64_t i1,
                DBuf<int32_t> &out_q, DBuf<int32_t> &out_row, int64_t cap_hint, int64_t most, int *launches,
                cudaStream_t st) {
    *launches = 0;
    const int64_t n_items = i1 - i0;
    if (n_items <= 0) return 0;
    int dev = 0, sms = 0;
    GTS_CUDA(cudaGetDevice(&dev));
    GTS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const size_t smem = l2f_smem_bytes();
    const bool v16 = (t.dim & 3) == 0 && (((uintptr_t)lq.Q | (uintptr_t)t.X.get()) & 15) == 0;
    void (*kern)(L2fArgs) = v16 ? k_tile_l2f<true> : k_tile_l2f<false>;
    GTS_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    GTS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreadsF, smem));
    if (per_sm < 1) per_sm = 1;
    // a block's chunks are split over several units while there are fewer
    // than four units per resident CTA (a small tree, a large batch)
    const int64_t resident = (int64_t)(sms > 0 ? sms : 1) * per_sm;
    const int64_t max_chunks = (nq + kNQF - 1) / kNQF;
    const int64_t split =
        std::max<int64_t>(1, std::min<int64_t>(max_chunks, (4 * resident + n_items - 1) / n_items));
    const int64_t units = n_items * split;
    GTS_REQUIRE(units < ((int64_t)1 << 31) - resident, GTS_EINVAL, "too many FP32 tiles");
    const int64_t grid = std::min<int64_t>(units, resident);
    DBuf<float> qn2(nq > 0 ? nq : 1, st);
    k_query_norms<<<(unsigned)((nq * 32 + 255) / 256), 256, 0, st>>>(lq.Q, nq, t.dim, qn2.get());
    ++*launches;
    DBuf<int> counter(1, st);
    DBuf<unsigned long long> count(1, st);
    int64_t cap = cap_hint > 0 ? cap_hint : 1 << 20;
    for (int attempt = 0; attempt < 2; ++attempt) {
        out_q.alloc(cap, st);
        out_row.alloc(cap, st);
        GTS_CUDA(cudaMemsetAsync(counter.get(), 0, 4, st));
        GTS_CUDA(cudaMemsetAsync(count.get(), 0, 8, st));
        L2fArgs a;
        a.dim = t.dim;
        a.F = t.F;
        a.X = t.X.get();
        a.Q = lq.Q;
        a.qn2 = qn2.get();
        a.row_del = t.row_del.get();
        a.npos = t.npos.get();
        a.nsize = t.nsize.get();
        a.lvl_last = t.lvl_off[t.h - 1];
        a.grec = rg.grec.get();
        a.items = rg.items.get() + i0;
        a.units = units;
        a.split = (int)split;
        a.work_counter = counter.get();
        a.out_q = out_q.get();
        a.out_row = out_row.get();
        a.cap = cap;
        a.out_count = count.get();
        a.c = 2.2f * (float)(t.dim + 16) * 5.9604645e-8f;
        a.absf = lq.absf;
        a.any_deleted = lq.any_deleted;
        kern<<<(unsigned)grid, kThreadsF, smem, st>>>(a);
        ++*launches;
        check_launch("FP32 L2 tile");
        unsigned long long hcount = 0;
        GTS_CUDA(cudaMemcpyAsync(&hcount, count.get(), 8, cudaMemcpyDeviceToHost, st));
        GTS_CUDA(cudaStreamSynchronize(st));
        if ((int64_t)hcount <= cap || (int64_t)hcount > most) return (int64_t)hcount;
        cap = (int64_t)hcount;   // rerun with room for every pair
    }
    GTS_REQUIRE(false, GTS_ECUDA, "FP32 L2 tile: output count changed between identical runs");
    return 0;
}

}  // namespace gts
