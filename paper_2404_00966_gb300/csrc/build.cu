// Index construction on the GPU (Section 4.3, Algorithms 1-3).
//
// All nodes of one level are processed together (the paper's level-parallel
// construction).  Per pivot level l = 0 .. h-1:
//   1. pivot choice (Algorithm 2, FFT): one block per node picks the object
//      whose smallest distance to the pivots of its ancestors is largest
//      (ties to the smallest id); the root pivot is given.
//   2. mapping (Algorithm 2): every object's distance to its node's pivot,
//      computed exactly (FP64 in the reference operation order for L1/L2,
//      bit-parallel integer DP for edit distance), stored as float32.
//   3. partitioning (Algorithm 3): one global radix sort of 64-bit keys
//      (node index << 32 | distance bits) over objects listed in id order;
//      the sort is stable, so ties fall to the smaller id.  This plays the
//      role of the paper's encoded key i + dis / (max + 1) without its
//      floating-point collisions at large node indices.
//   4. even split of each node into fanout children by count, the last child
//      taking the remainder; a child's [lo, hi] is its first and last distance.
// Objects stay in input order while the levels are built (per-object columns);
// at the end they are gathered once into leaf order.
#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_scan.cuh>

#include "gts_impl.cuh"
#include "metric.cuh"

namespace gts {

uint64_t splitmix64(uint64_t x) {
    // SplitMix64 (Steele, Lea, Flood 2014): one output for state x.
    uint64_t z = x + 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

int tree_height(int64_t n, int F, int n_pivots) {
    if (n_pivots > 0) return n_pivots < kMaxHeight ? n_pivots : kMaxHeight;
    // ceil(log_F(n + 1)) - 1 (Algorithm 1), in integers; at least one pivot level
    int t = 0;
    long double p = 1;
    while (p < (long double)n + 1) {
        p *= F;
        ++t;
    }
    // at least one pivot level; at most kMaxHeight (small fanouts over large sets)
    const int h = t - 1 < 1 ? 1 : t - 1;
    return h < kMaxHeight ? h : kMaxHeight;
}

// thread per node of the pivot levels
__global__ static void k_order_children(const int32_t *__restrict__ nsize, const float *__restrict__ nlo,
                                        const float *__restrict__ nhi, int64_t nodes, int F, int8_t *__restrict__ nord) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= nodes) return;
    // (Eq. 1 over all levels in one array: the children of node g are nodes g F + 1 ..)
    const int64_t c0 = g * F + 1;
    int j0 = -1;
    bool ok = true;
    float lo = 0.f, hi = 0.f;
    for (int j = 0; j < F; ++j) {
        const bool ne = nsize[c0 + j] > 0;
        if (!ne) {
            if (j0 >= 0) ok = false;
            continue;
        }
        const float l = nlo[c0 + j], h = nhi[c0 + j];
        if (!(l >= lo && h >= hi && h >= l)) ok = false;   // (from 0 on: distances)
        lo = l;
        hi = h;
        if (j0 < 0) j0 = j;
    }
    nord[g] = ok ? (int8_t)j0 : (int8_t)-1;
}

void order_children(Tree &t, cudaStream_t st) {
    const int64_t nodes = t.lvl_off[t.h];
    t.nord = reinterpret_cast<int8_t *>(t.npiv.get() + t.lvl_off[t.h + 1]);
    if (nodes > 0)
        k_order_children<<<(unsigned)((nodes + 255) / 256), 256, 0, st>>>(t.nsize.get(), t.nlo.get(), t.nhi.get(), nodes,
                                                                         t.F, t.nord);
    check_launch("order of the children");
}

size_t Tree::device_bytes() const {
    return X.bytes() + Xr.bytes() + S.bytes() + Soff.bytes() + row_id.bytes() + table.bytes() + row_del.bytes() +
           npos.bytes() + nsize.bytes() + npiv.bytes() + nlo.bytes() + nhi.bytes() +
           // built on first use
           tc.Xh.bytes() + tc.Xl.bytes() + tc.xn2.bytes() + tc.xr.bytes() + tc.Ph.bytes() + tc.Pl.bytes() +
           tc.pn2.bytes() + xrn2.bytes() + qg.bytes() + qcode.bytes();
}

namespace {

constexpr int kThreads = 256;

inline unsigned blocks_for(int64_t n, int per = kThreads) {
    int64_t b = (n + per - 1) / per;
    if (b < 1) b = 1;
    if (b > 0x7fffffff) b = 0x7fffffff;
    return (unsigned)b;
}

__global__ void k_iota_i32(int32_t *a, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        a[i] = (int32_t)i;
}

__global__ void k_fill_i32(int32_t *a, int64_t n, int32_t v) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        a[i] = v;
}

__global__ void k_fill_i64(int64_t *a, int64_t n, int64_t v) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        a[i] = v;
}

// FFT pivot of every node of level l >= 1.  Key = (score bits << 32) |
// (0x7fffffff - object index): the maximum has the largest score, then the
// smallest index (objects are listed in increasing id order).
__global__ void k_fft_pivot(const int32_t *__restrict__ perm, const float *__restrict__ T, int64_t n, int l,
                            const int32_t *__restrict__ lpos, const int32_t *__restrict__ lsize,
                            int32_t *__restrict__ piv_obj) {
    const int node = blockIdx.x;
    const int32_t s = lpos[node], c = lsize[node];
    if (c == 0) {
        if (threadIdx.x == 0) piv_obj[node] = -1;
        return;
    }
    unsigned long long best = 0ull;
    for (int32_t r = threadIdx.x; r < c; r += blockDim.x) {
        const int32_t o = perm[s + r];
        float sc = T[o];
        for (int a = 1; a < l; ++a) sc = fminf(sc, T[(int64_t)a * n + o]);
        const unsigned long long key =
            ((unsigned long long)__float_as_uint(sc) << 32) | (unsigned long long)(0x7fffffffu - (uint32_t)o);
        best = key > best ? key : best;
    }
    __shared__ unsigned long long red[kThreads / 32];
    for (int off = 16; off > 0; off >>= 1) {
        unsigned long long o2 = __shfl_xor_sync(0xffffffffu, best, off);
        best = o2 > best ? o2 : best;
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long b = red[0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) b = red[w] > b ? red[w] : b;
        piv_obj[node] = (int32_t)(0x7fffffffu - (uint32_t)(b & 0xffffffffull));
    }
}

// Mapping for vectors: one thread per table position, FP64 in the reference
// order, rounded once to float32.  Also records each object's node.
template <bool L2>
__global__ void k_map_vec(const float *__restrict__ X, int dim, const int32_t *__restrict__ perm,
                          const int32_t *__restrict__ pos_node, const int32_t *__restrict__ piv_obj, int64_t n,
                          float *__restrict__ Tl, int32_t *__restrict__ node_of) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t o = perm[p];
        const int32_t node = pos_node[p];
        const int32_t pv = piv_obj[node];
        const float *a = X + (int64_t)o * dim;
        const float *b = X + (int64_t)pv * dim;
        // (l2sq_fp64_seq / l1_fp64_seq without their unrolling, which long rows need: a
        // level of 10^6 rows of 2 coordinates, us: L2 54.9 with, 44.6 without; L1 32.4, 26.3)
        double d = 0.0;
        for (int i = 0; i < dim; ++i) {
            const double t = __dsub_rn((double)a[i], (double)b[i]);
            d = __dadd_rn(d, L2 ? __dmul_rn(t, t) : fabs(t));
        }
        if (L2) d = __dsqrt_rn(d);
        Tl[o] = __double2float_rn(d);
        node_of[o] = node;
    }
}

// ---- mapping of vectors in double-single arithmetic
//
// The table holds RN32(d) of the FP64 distance summed in the reference order,
// and GB300 has 2 FP64 lanes per SM and cycle: three FP64 operations per
// coordinate of 10^6 x 128 take 0.61 ms per level (1.21 ms measured, a thread
// per row; this form 0.18 ms), eight times the pass over the rows.  Here eight
// lanes sum a row: every difference (exact, Knuth's two-sum), square (Dekker's
// product by a fused multiply-add) and partial sum is an unevaluated FP32 pair.
// Then one warp of the block takes its 32 rows, a lane each: the pair's proven
// error decides whether the FP32 rounding of the distance is certain; if it is
// not (a few rows in ten thousand), the lane sums the row in FP64 in the
// reference order.  The values are those of k_map_vec bit for bit.
// (The test is some 19 FP64 instructions: by the lanes that had the sums, four
// rows a warp, it took more FP64 time than the distances of up to 40 coordinates.)
//
// Error of a lane's pair over n <= dim / 8 + 4 terms, u = 2^-24, S the sum: lo is
// folded into hi every four terms, so |lo| <= u S after that and at most 8 u S
// before the next (each term's part of lo is below u S + 3 u p_i, p_i its square);
// a term's two roundings of lo then add u^2 (10 S + 3 p_i), the products' dropped
// and rounded parts 4 u^2 p_i, the three merges 60 u^2 S: below (10 n + 70) u^2 S
// in all.  `del` is more than twice that, which also covers the FP64 reference's own
// (dim + 4) 2^-53.  (Without the folding the error grows with the square of the
// terms, and from 3,000 dimensions on many rows took FP64.)  Results outside [1e-18,
// 1e30], where FP32 squares could lose their low parts or overflow, take FP64.
constexpr int kMapLanes = 8;
// Up to these dimensions a thread sums a row in FP64, which is then as fast (L1
// has one FP64 operation less per coordinate).  Builds of 10^6 rows, a thread a row / this form, us:
// L2, 8 dimensions 2149 / 2084, 9: 2215 / 2048, 24: 2793 / 2200; L1, 9: 2083 / 2178,
// 16: 2285 / 2272, 17: 2362 / 2224.  (Of 20,000 rows both take 0.52 ms up to 24.)
constexpr int kMapSingleL2 = 8, kMapSingleL1 = 16;
constexpr int kMapRows = kThreads / kMapLanes;   // rows of a block: one per lane of the warp that decides
static_assert(kMapRows == 32, "one row per lane of the deciding warp");

inline double map_error(int dim) { return (10.0 * (dim / 8 + 4) + 80.0) / 140737488355328.0; }   // 2^-47

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float bp = __fsub_rn(s, a), ap = __fsub_rn(s, bp);
    e = __fadd_rn(__fsub_rn(a, ap), __fsub_rn(b, bp));
}

template <bool L2>
__device__ __forceinline__ void ds_add_term(float a, float b, float &hi, float &lo, float &big) {
    float s, e;
    two_sum(a, -b, s, e);
    big = fmaxf(big, fabsf(s));
    float p, q;
    if (L2) {
        p = __fmul_rn(s, s);
        q = __fmaf_rn(__fadd_rn(s, s), e, __fmaf_rn(s, s, -p));
    } else {
        p = fabsf(s);
        q = s < 0.f ? -e : e;
    }
    float t, r;
    two_sum(hi, p, t, r);
    hi = t;
    lo = __fadd_rn(lo, __fadd_rn(r, q));
}
// lo into hi (|lo| <= hi: the short form of the two-sum is exact)
__device__ __forceinline__ void ds_fold(float &hi, float &lo) {
    const float t = __fadd_rn(hi, lo);
    lo = __fsub_rn(lo, __fsub_rn(t, hi));
    hi = t;
}

// RN32 of the distance whose (L2: squared) value lies within a relative del
// of hi + lo, or -1 if two FP32 values are possible (or the first guess, one
// Newton step from the root of hi, is not the nearest)
template <bool L2>
__device__ __forceinline__ float ds_round(float hi_s, float lo_s, double S, double del) {
    float r;
    if (L2) {
        const float r0 = __fsqrt_rn(hi_s);
        r = __fadd_rn(r0, __fdividef(__fadd_rn(__fmaf_rn(-r0, r0, hi_s), lo_s), r0 + r0));
    } else {
        r = __fadd_rn(hi_s, lo_s);
    }
    const double below = 0.5 * ((double)r + (double)__uint_as_float(__float_as_uint(r) - 1u));
    const double above = 0.5 * ((double)r + (double)__uint_as_float(__float_as_uint(r) + 1u));
    // (25-bit midpoints: their squares are exact in FP64)
    const double lo = L2 ? below * below : below, hi = L2 ? above * above : above;
    return lo < S * (1.0 - del) && S * (1.0 + del) < hi ? r : -1.f;
}

// block b: the rows at positions [32 b, 32 b + 32)
template <bool L2, bool V4>
__global__ void __launch_bounds__(kThreads) k_map_vec_ds(const float *__restrict__ X, int dim,
                                                         const int32_t *__restrict__ perm,
                                                         const int32_t *__restrict__ pos_node,
                                                         const int32_t *__restrict__ piv_obj, int64_t n, double del,
                                                         float *__restrict__ Tl, int32_t *__restrict__ node_of) {
    __shared__ float s_hi[kMapRows], s_lo[kMapRows];   // hi < 0: every difference was 0
    const int sub = threadIdx.x & (kMapLanes - 1);
    const int64_t p0 = (int64_t)blockIdx.x * kMapRows;
    {
        const int64_t p = p0 + threadIdx.x / kMapLanes;
        float hi = 0.f, lo = 0.f, big = 0.f;
        if (p < n) {
            const float *a = X + (int64_t)perm[p] * dim, *b = X + (int64_t)piv_obj[pos_node[p]] * dim;
            if (V4) {
                const float4 *a4 = reinterpret_cast<const float4 *>(a), *b4 = reinterpret_cast<const float4 *>(b);
#pragma unroll 4
                for (int i = sub; i < dim / 4; i += kMapLanes) {
                    const float4 x = a4[i], y = b4[i];
                    ds_add_term<L2>(x.x, y.x, hi, lo, big);
                    ds_add_term<L2>(x.y, y.y, hi, lo, big);
                    ds_add_term<L2>(x.z, y.z, hi, lo, big);
                    ds_add_term<L2>(x.w, y.w, hi, lo, big);
                    ds_fold(hi, lo);
                }
            } else {
#pragma unroll 4
                for (int i = sub; i < dim; i += kMapLanes) {
                    ds_add_term<L2>(a[i], b[i], hi, lo, big);
                    if ((i & (3 * kMapLanes)) == 3 * kMapLanes) ds_fold(hi, lo);   // every fourth of the lane's terms
                }
            }
        }
#pragma unroll
        for (int off = 1; off < kMapLanes; off <<= 1) {
            const float h2 = __shfl_xor_sync(0xffffffffu, hi, off), l2 = __shfl_xor_sync(0xffffffffu, lo, off);
            float t, r;
            two_sum(hi, h2, t, r);
            hi = t;
            lo = __fadd_rn(__fadd_rn(lo, l2), r);
            big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, off));
        }
        if (sub == 0) {
            s_hi[threadIdx.x / kMapLanes] = big == 0.f ? -1.f : fmaxf(hi, 0.f);
            s_lo[threadIdx.x / kMapLanes] = lo;
        }
    }
    __syncthreads();
    const int64_t p = p0 + threadIdx.x;
    if (threadIdx.x >= kMapRows || p >= n) return;
    const float hi = s_hi[threadIdx.x], lo = s_lo[threadIdx.x];
    const int32_t o = perm[p], node = pos_node[p];
    const double S = (double)hi + (double)lo;
    float r = -1.f;
    if (hi < 0.f) r = 0.f;   // (a NaN cannot occur: builds reject non-finite coordinates)
    else if (S >= 1e-18 && S <= 1e30) r = ds_round<L2>(hi, lo, S, del);
    if (r < 0.f) {
        const float *a = X + (int64_t)o * dim, *b = X + (int64_t)piv_obj[node] * dim;
        double d = L2 ? l2sq_fp64_seq(a, b, dim) : l1_fp64_seq(a, b, dim);
        if (L2) d = __dsqrt_rn(d);
        r = __double2float_rn(d);
    }
    Tl[o] = r;
    node_of[o] = node;
}

// Mapping for strings: a block takes a run of table positions; for every node
// in the run it loads the node pivot's match masks into shared memory and each
// thread computes one object's distance to the pivot (pattern = pivot).
template <int B>
__global__ void k_map_str(const uint8_t *__restrict__ S, const int64_t *__restrict__ Soff,
                          const int32_t *__restrict__ perm, const int32_t *__restrict__ pos_node,
                          const int32_t *__restrict__ piv_obj, const int32_t *__restrict__ lpos,
                          const int32_t *__restrict__ lsize, int64_t n, int chunk, float *__restrict__ Tl,
                          int32_t *__restrict__ node_of) {
    __shared__ __align__(16) uint32_t Peq[256 * B];
    const int64_t p0 = (int64_t)blockIdx.x * chunk;
    const int64_t p1 = p0 + chunk < n ? p0 + chunk : n;
    int64_t s = p0;
    while (s < p1) {
        const int32_t node = pos_node[s];
        int64_t e = (int64_t)lpos[node] + lsize[node];
        if (e > p1) e = p1;
        const int32_t pv = piv_obj[node];
        const int m = (int)(Soff[pv + 1] - Soff[pv]);
        if (m > 0) build_peq<B>(Peq, S + Soff[pv], m);
        for (int64_t p = s + threadIdx.x; p < e; p += blockDim.x) {
            const int32_t o = perm[p];
            const int len = (int)(Soff[o + 1] - Soff[o]);
            const int d = m > 0 ? edit_bits<B, TextBytes>(Peq, m, S + Soff[o], len) : len;
            Tl[o] = (float)d;
            node_of[o] = node;
        }
        __syncthreads();
        s = e;
    }
}

__global__ void k_keys(const int32_t *__restrict__ node_of, const float *__restrict__ Tl, int64_t n,
                       uint64_t *__restrict__ keys, int32_t *__restrict__ vals) {
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < n; o += (int64_t)gridDim.x * blockDim.x) {
        keys[o] = ((uint64_t)(uint32_t)node_of[o] << 32) | (uint64_t)__float_as_uint(Tl[o]);
        vals[o] = (int32_t)o;
    }
}

// Children of every node of level l: even split by count (Algorithm 3).  The
// rows rise with the distance, so the non-empty children rise from the first on;
// nord (this level's): that child, or -1.  (A launch and a buffer of its own for
// nord made builds of up to 50,000 rows 1 % longer: 20,000 x 2, 512 against 506 us.)
__global__ void k_children(const int32_t *__restrict__ lpos, const int32_t *__restrict__ lsize, int64_t nn, int F,
                           const int32_t *__restrict__ perm, const float *__restrict__ Tl,
                           int32_t *__restrict__ cpos, int32_t *__restrict__ csize, float *__restrict__ clo,
                           float *__restrict__ chi, int8_t *__restrict__ nord) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nn * F; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / F;
        const int j = (int)(t - i * F);
        const int32_t s = lpos[i], c = lsize[i];
        const int32_t avg = c / F;
        const int32_t cs = s + j * avg;
        const int32_t cc = j < F - 1 ? avg : c - avg * (F - 1);
        if (j == 0) nord[i] = c == 0 ? (int8_t)-1 : avg > 0 ? (int8_t)0 : (int8_t)(F - 1);
        cpos[t] = cs;
        csize[t] = cc;
        if (cc > 0) {
            clo[t] = Tl[perm[cs]];
            chi[t] = Tl[perm[cs + cc - 1]];
        } else {
            clo[t] = __int_as_float(0x7f800000);   // +inf
            chi[t] = __int_as_float(0xff800000);   // -inf
        }
    }
}

__global__ void k_next_pos_node(int32_t *__restrict__ pos_node, int64_t n, const int32_t *__restrict__ lpos,
                                const int32_t *__restrict__ lsize, int F) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t node = pos_node[p];
        const int32_t s = lpos[node], c = lsize[node];
        const int32_t avg = c / F;
        int32_t j = avg > 0 ? (int32_t)((p - s) / avg) : F - 1;
        if (j > F - 1) j = F - 1;
        pos_node[p] = node * F + j;
    }
}

// rows into leaf order: 16 bytes a thread where the rows allow it (10^6 x 128:
// 0.20 ms; one float and a 64-bit division a thread took 0.70 ms)
template <class V>
__global__ void k_gather_rows(const V *__restrict__ X, int per_row, const int32_t *__restrict__ perm, int64_t n,
                              V *__restrict__ Xl) {
    const int64_t total = n * (int64_t)per_row;
    if (total < ((int64_t)1 << 31)) {   // 32-bit division
        const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x, pr = (uint32_t)per_row;
        if (t >= total) return;
        const uint32_t p = t / pr;
        Xl[t] = X[(int64_t)perm[p] * pr + (t - p * pr)];
        return;
    }
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = t / per_row;
        Xl[t] = X[(int64_t)perm[p] * per_row + (t - p * per_row)];
    }
}

__global__ void k_gather_meta(const int32_t *__restrict__ perm, int64_t n, int h, const float *__restrict__ T,
                              const int64_t *__restrict__ ids_in, float *__restrict__ table,
                              int64_t *__restrict__ row_id, int32_t *__restrict__ inv) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t o = perm[p];
        for (int l = 0; l < h; ++l) table[(int64_t)l * n + p] = T[(int64_t)l * n + o];
        row_id[p] = ids_in ? ids_in[o] : (int64_t)o;
        inv[o] = (int32_t)p;
    }
}

__global__ void k_str_lengths(const int64_t *__restrict__ Soff, const int32_t *__restrict__ perm, int64_t n,
                              int64_t *__restrict__ len) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t o = perm[p];
        len[p] = Soff[o + 1] - Soff[o];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) len[n] = 0;
}

__global__ void k_gather_str(const uint8_t *__restrict__ S, const int64_t *__restrict__ Soff,
                             const int32_t *__restrict__ perm, int64_t n, const int64_t *__restrict__ Loff,
                             uint8_t *__restrict__ SL) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t p = warp; p < n; p += nw) {
        const int32_t o = perm[p];
        const int64_t a = Soff[o], len = Soff[o + 1] - a, d = Loff[p];
        for (int64_t i = lane; i < len; i += 32) SL[d + i] = S[a + i];
    }
}

__global__ void k_piv_rows(int32_t *__restrict__ piv, int64_t cnt, const int32_t *__restrict__ inv) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x)
        if (piv[i] >= 0) piv[i] = inv[piv[i]];
}

template <int B>
void launch_map_str(const Objects &o, const int32_t *perm, const int32_t *pos_node, const int32_t *piv,
                    const int32_t *lpos, const int32_t *lsize, int64_t n, float *Tl, int32_t *node_of,
                    cudaStream_t st) {
    const int chunk = 256;
    k_map_str<B><<<blocks_for(n, chunk), 128, 0, st>>>(o.S, o.Soff, perm, pos_node, piv, lpos, lsize, n, chunk, Tl,
                                                       node_of);
}

void gather_rows(const float *X, int dim, const int32_t *perm, int64_t n, float *out, cudaStream_t st) {
    if (dim % 4 == 0 && (((uintptr_t)X | (uintptr_t)out) & 15) == 0)
        k_gather_rows<float4><<<blocks_for(n * (dim / 4)), kThreads, 0, st>>>(
            reinterpret_cast<const float4 *>(X), dim / 4, perm, n, reinterpret_cast<float4 *>(out));
    else
        k_gather_rows<float><<<blocks_for(n * (int64_t)dim), kThreads, 0, st>>>(X, dim, perm, n, out);
}

}  // namespace

void build_tree(Tree &t, const Objects &objs, const int64_t *d_ids, int metric, int F, int h, int64_t root,
                cudaStream_t st, const float *raw_rows) {
    const int64_t n = objs.n;
    t.metric = metric;
    t.cosine = raw_rows != nullptr;
    t.dim = objs.dim;
    t.F = F;
    t.h = h;
    t.n = n;
    t.lvl_off.assign(h + 2, 0);
    int64_t cnt = 1;
    for (int l = 0; l <= h; ++l) {
        t.lvl_off[l + 1] = t.lvl_off[l] + cnt;
        if (l < h) {
            cnt *= F;
            GTS_REQUIRE(t.lvl_off[l + 1] + cnt <= (int64_t)1 << 28, GTS_EINVAL,
                        "fanout^height too large: more than 2^28 tree nodes");
        }
    }
    const int64_t total_nodes = t.lvl_off[h + 1];
    t.npos.alloc(total_nodes, st);
    t.nsize.alloc(total_nodes, st);
    t.npiv.alloc(total_nodes + nord_spare(t), st);
    t.nord = reinterpret_cast<int8_t *>(t.npiv.get() + total_nodes);
    t.nlo.alloc(total_nodes, st);
    t.nhi.alloc(total_nodes, st);
    k_fill_i32<<<blocks_for(total_nodes), kThreads, 0, st>>>(t.npiv.get(), total_nodes, -1);
    {
        int32_t zero = 0, nn32 = (int32_t)n;
        float ninf = -INFINITY, pinf = INFINITY;
        GTS_CUDA(cudaMemcpyAsync(t.npos.get(), &zero, 4, cudaMemcpyHostToDevice, st));
        GTS_CUDA(cudaMemcpyAsync(t.nsize.get(), &nn32, 4, cudaMemcpyHostToDevice, st));
        GTS_CUDA(cudaMemcpyAsync(t.nlo.get(), &ninf, 4, cudaMemcpyHostToDevice, st));
        GTS_CUDA(cudaMemcpyAsync(t.nhi.get(), &pinf, 4, cudaMemcpyHostToDevice, st));
        GTS_CUDA(cudaStreamSynchronize(st));
    }
    t.row_del.alloc(n, st);
    t.row_id.alloc(n, st);
    t.table.alloc((size_t)h * n, st);
    if (n == 0) {
        if (objs.dim == 0) {
            t.Soff.alloc(1, st);
            GTS_CUDA(cudaMemsetAsync(t.Soff.get(), 0, 8, st));
        }
        GTS_CUDA(cudaStreamSynchronize(st));
        return;
    }
    t.max_len = objs.dim == 0 ? objs.max_len : 0;
    DBuf<int32_t> perm(n, st), perm2(n, st), pos_node(n, st), node_of(n, st), inv(n, st);
    DBuf<float> T((size_t)h * n, st);
    DBuf<uint64_t> keys(n, st), keys2(n, st);
    k_iota_i32<<<blocks_for(n), kThreads, 0, st>>>(perm.get(), n);
    k_fill_i32<<<blocks_for(n), kThreads, 0, st>>>(pos_node.get(), n, 0);
    {
        int32_t r32 = (int32_t)root;
        GTS_CUDA(cudaMemcpyAsync(t.npiv.get(), &r32, 4, cudaMemcpyHostToDevice, st));
        GTS_CUDA(cudaStreamSynchronize(st));
    }
    size_t sort_tmp_bytes = 0;
    cub::DeviceRadixSort::SortPairs(nullptr, sort_tmp_bytes, keys.get(), keys2.get(), perm.get(), perm2.get(), n, 0,
                                    64, st);
    DBuf<uint8_t> sort_tmp(sort_tmp_bytes, st);
    for (int l = 0; l < h; ++l) {
        const int64_t nn = t.lvl_off[l + 1] - t.lvl_off[l];
        int32_t *lpos = t.npos.get() + t.lvl_off[l];
        int32_t *lsize = t.nsize.get() + t.lvl_off[l];
        int32_t *lpiv = t.npiv.get() + t.lvl_off[l];
        float *Tl = T.get() + (int64_t)l * n;
        if (l > 0) k_fft_pivot<<<(unsigned)nn, kThreads, 0, st>>>(perm.get(), T.get(), n, l, lpos, lsize, lpiv);
        check_launch("fft pivot");
        if (objs.dim > 0) {
            if (objs.dim > (metric == GTS_L2 ? kMapSingleL2 : kMapSingleL1)) {
                const bool v4 = objs.dim % 4 == 0 && ((uintptr_t)objs.X & 15) == 0;
                const double del = map_error(objs.dim);
                const unsigned grid = blocks_for(n, kMapRows);
#define GTS_MAP(L2V, V4V)                                                                                            \
    k_map_vec_ds<L2V, V4V><<<grid, kThreads, 0, st>>>(objs.X, objs.dim, perm.get(), pos_node.get(), lpiv, n, del, Tl, \
                                                      node_of.get())
                if (metric == GTS_L2) {
                    if (v4) GTS_MAP(true, true);
                    else GTS_MAP(true, false);
                } else {
                    if (v4) GTS_MAP(false, true);
                    else GTS_MAP(false, false);
                }
#undef GTS_MAP
            } else if (metric == GTS_L2) {
                k_map_vec<true><<<blocks_for(n), kThreads, 0, st>>>(objs.X, objs.dim, perm.get(), pos_node.get(), lpiv,
                                                                    n, Tl, node_of.get());
            } else {
                k_map_vec<false><<<blocks_for(n), kThreads, 0, st>>>(objs.X, objs.dim, perm.get(), pos_node.get(), lpiv,
                                                                     n, Tl, node_of.get());
            }
        } else {
            const int W = (t.max_len + 31) / 32;   // 32-bit words of the longest pattern
#define GTS_MAP_STR(BB) \
    launch_map_str<BB>(objs, perm.get(), pos_node.get(), lpiv, lpos, lsize, n, Tl, node_of.get(), st)
            if (W <= 1) GTS_MAP_STR(1);
            else if (W <= 2) GTS_MAP_STR(2);
            else if (W <= 4) GTS_MAP_STR(4);
            else if (W <= 8) GTS_MAP_STR(8);
            else if (W <= 16) GTS_MAP_STR(16);
            else GTS_MAP_STR(32);
#undef GTS_MAP_STR
        }
        check_launch("mapping");
        k_keys<<<blocks_for(n), kThreads, 0, st>>>(node_of.get(), Tl, n, keys.get(), perm2.get());
        int node_bits = 0;
        while (((int64_t)1 << node_bits) < nn) ++node_bits;
        size_t tb = sort_tmp_bytes;
        GTS_CUDA(cub::DeviceRadixSort::SortPairs(sort_tmp.get(), tb, keys.get(), keys2.get(), perm2.get(), perm.get(),
                                                 n, 0, 32 + node_bits, st));
        k_children<<<blocks_for(nn * F), kThreads, 0, st>>>(lpos, lsize, nn, F, perm.get(), Tl,
                                                           t.npos.get() + t.lvl_off[l + 1],
                                                           t.nsize.get() + t.lvl_off[l + 1],
                                                           t.nlo.get() + t.lvl_off[l + 1], t.nhi.get() + t.lvl_off[l + 1],
                                                           t.nord + t.lvl_off[l]);
        k_next_pos_node<<<blocks_for(n), kThreads, 0, st>>>(pos_node.get(), n, lpos, lsize, F);
        check_launch("partitioning");
    }
    // final gather into leaf order
    k_gather_meta<<<blocks_for(n), kThreads, 0, st>>>(perm.get(), n, h, T.get(), d_ids, t.table.get(),
                                                      t.row_id.get(), inv.get());
    k_piv_rows<<<blocks_for(t.lvl_off[h]), kThreads, 0, st>>>(t.npiv.get(), t.lvl_off[h], inv.get());
    k_fill_i64<<<blocks_for(n), kThreads, 0, st>>>(t.row_del.get(), n, kNever);
    if (objs.dim > 0) {
        t.X.alloc((size_t)n * objs.dim, st);
        gather_rows(objs.X, objs.dim, perm.get(), n, t.X.get(), st);
        if (raw_rows) {   // angular distance: the raw rows in the same (leaf) order
            t.Xr.alloc((size_t)(n > 0 ? n : 1) * objs.dim, st);
            gather_rows(raw_rows, objs.dim, perm.get(), n, t.Xr.get(), st);
        }
    } else {
        DBuf<int64_t> len(n + 1, st);
        t.Soff.alloc(n + 1, st);
        k_str_lengths<<<blocks_for(n), kThreads, 0, st>>>(objs.Soff, perm.get(), n, len.get());
        size_t tb = 0;
        cub::DeviceScan::ExclusiveSum(nullptr, tb, len.get(), t.Soff.get(), n + 1, st);
        DBuf<uint8_t> tmp(tb, st);
        GTS_CUDA(cub::DeviceScan::ExclusiveSum(tmp.get(), tb, len.get(), t.Soff.get(), n + 1, st));
        int64_t total = 0;
        GTS_CUDA(cudaMemcpyAsync(&total, t.Soff.get() + n, 8, cudaMemcpyDeviceToHost, st));
        GTS_CUDA(cudaStreamSynchronize(st));
        t.S.alloc(total + kTextPad, st);
        k_gather_str<<<blocks_for(n * 32), kThreads, 0, st>>>(objs.S, objs.Soff, perm.get(), n, t.Soff.get(),
                                                            t.S.get());
    }
    check_launch("gather");
    GTS_CUDA(cudaStreamSynchronize(st));
    t.persist();
}

}  // namespace gts
