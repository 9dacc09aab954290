// Device-side distance functions (Section 3: edit distance, L1, L2).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gts {

// ---------------------------------------------------------------- FP32 vectors

// Partial sum over the lanes of a warp; every lane returns the full sum.
// L2 returns the squared distance.  Each lane adds about dim / 32 terms in
// sequence, then five shuffle levels add the lane sums (a binary tree).
template <bool L2>
__device__ __forceinline__ float warp_vec_dist(const float *__restrict__ q, const float *__restrict__ x,
                                               int dim, int lane) {
    float s = 0.f;
    if ((dim & 3) == 0 && ((((uintptr_t)q) | ((uintptr_t)x)) & 15) == 0) {
        const float4 *q4 = reinterpret_cast<const float4 *>(q);
        const float4 *x4 = reinterpret_cast<const float4 *>(x);
        for (int i = lane; i < (dim >> 2); i += 32) {
            float4 a = q4[i], b = __ldg(x4 + i);
            float d0 = a.x - b.x, d1 = a.y - b.y, d2 = a.z - b.z, d3 = a.w - b.w;
            if (L2) s += d0 * d0 + d1 * d1 + d2 * d2 + d3 * d3;
            else s += fabsf(d0) + fabsf(d1) + fabsf(d2) + fabsf(d3);
        }
    } else {
        for (int i = lane; i < dim; i += 32) {
            float d = q[i] - __ldg(x + i);
            s += L2 ? d * d : fabsf(d);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// Same sum with the query already in registers as float4 chunks (NV = dim /
// 128 per lane); NV = 0 falls back to warp_vec_dist.
template <bool L2, int NV>
__device__ __forceinline__ float row_dist_regs(const float4 (&qr)[NV > 0 ? NV : 1], const float *xv, const float *qv,
                                               int dim, int lane) {
    if (NV > 0) {
        const float4 *x4 = reinterpret_cast<const float4 *>(xv);
        float s = 0.f;
#pragma unroll
        for (int v = 0; v < (NV > 0 ? NV : 1); ++v) {
            const float4 b = __ldg(x4 + v * 32 + lane);
            const float4 a = qr[v];
            const float d0 = a.x - b.x, d1 = a.y - b.y, d2 = a.z - b.z, d3 = a.w - b.w;
            if (L2) s += d0 * d0 + d1 * d1 + d2 * d2 + d3 * d3;
            else s += fabsf(d0) + fabsf(d1) + fabsf(d2) + fabsf(d3);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return s;
    }
    return warp_vec_dist<L2>(qv, xv, dim, lane);
}

// Proven relative error bound of the FP32 distance above against the exact
// distance: with u = 2^-24, any summation order of `dim` non-negative terms,
// each with up to three roundings, stays within gamma_{dim+2}; the square
// root halves it and adds u.  (dim + 8) u covers both with room to spare and
// also covers the FP64 reference's own error (<= (dim + 1) 2^-53).
__host__ __device__ __forceinline__ float fp32_rel_bound(int dim) { return (float)(dim + 8) * 5.9604645e-8f; }
// Absolute floor for results that underflow FP32 (squares below FLT_MIN).
constexpr float kAbsFloor = 1e-17f;

// ---------------------------------------------------------------- FP64 recheck

// The exact operation order of the CPU reference: increasing i, every
// subtraction, product and sum rounded on its own (no fused multiply-add).
// Rows on 16-byte boundaries are read 32 coordinates at a time (eight 16-byte
// loads of each in flight; with a coordinate's loads at a time the sums waited
// for memory: 130,000 keys of 128 coordinates 0.229 -> 0.193 ms), the sums keep
// their order.  WIDE = false: a coordinate at a time, for kernels that form few
// keys beside other work or rows of up to 16 coordinates -- the wide form takes
// 12 to 20 registers more (k_verify_vec 48 -> 64, and the range batches that it
// decides 5 to 9 % longer).
template <bool WIDE, class Term>
__device__ __forceinline__ void fp64_terms(const float *q, const float *x, int dim, Term term) {
    int i = 0;
    if (WIDE && (dim & 3) == 0 && ((((uintptr_t)q) | ((uintptr_t)x)) & 15) == 0) {
        const float4 *q4 = reinterpret_cast<const float4 *>(q), *x4 = reinterpret_cast<const float4 *>(x);
        for (; i + 32 <= dim; i += 32) {
            float4 a[8], b[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                a[u] = __ldg(q4 + (i >> 2) + u);
                b[u] = __ldg(x4 + (i >> 2) + u);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                term(a[u].x, b[u].x);
                term(a[u].y, b[u].y);
                term(a[u].z, b[u].z);
                term(a[u].w, b[u].w);
            }
        }
    }
#pragma unroll 4
    for (; i < dim; ++i) term(q[i], x[i]);
}

template <bool WIDE = true>
__device__ __forceinline__ double l2sq_fp64_seq(const float *q, const float *x, int dim) {
    double s = 0.0;
    fp64_terms<WIDE>(q, x, dim, [&](float a, float b) {
        const double t = __dsub_rn((double)a, (double)b);
        s = __dadd_rn(s, __dmul_rn(t, t));
    });
    return s;
}

// The angular distance's key, 1 - cos: the three sums q.x, |q|^2, |x|^2 in
// increasing i, every product and sum rounded on its own, c = dot /
// (sqrt(|q|^2) sqrt(|x|^2)) clamped to [-1, 1] -- the reference operation
// order.
__device__ __forceinline__ double cos_key_fp64(double dot, double nq, double nx) {
    double c = __ddiv_rn(dot, __dmul_rn(__dsqrt_rn(nq), __dsqrt_rn(nx)));
    c = c > 1.0 ? 1.0 : (c < -1.0 ? -1.0 : c);
    return __dsub_rn(1.0, c);
}
template <bool WIDE = true>
__device__ __forceinline__ double dot_fp64_seq(const float *q, const float *x, int dim) {
    double dot = 0.0;
    fp64_terms<WIDE>(q, x, dim, [&](float a, float b) { dot = __dadd_rn(dot, __dmul_rn((double)a, (double)b)); });
    return dot;
}
template <bool WIDE = true>
__device__ __forceinline__ double cos_key_fp64_seq(const float *q, const float *x, int dim) {
    double dot = 0.0, nq = 0.0, nx = 0.0;
    fp64_terms<WIDE>(q, x, dim, [&](float fa, float fb) {
        const double a = (double)fa, b = (double)fb;
        dot = __dadd_rn(dot, __dmul_rn(a, b));
        nq = __dadd_rn(nq, __dmul_rn(a, a));
        nx = __dadd_rn(nx, __dmul_rn(b, b));
    });
    return cos_key_fp64(dot, nq, nx);
}

template <bool WIDE = true>
__device__ __forceinline__ double l1_fp64_seq(const float *q, const float *x, int dim) {
    double s = 0.0;
    fp64_terms<WIDE>(q, x, dim,
               [&](float a, float b) { s = __dadd_rn(s, fabs(__dsub_rn((double)a, (double)b))); });
    return s;
}

// ---------------------------------------------------------------- edit distance

// Reads a string four bytes at a time from aligned 32-bit words.  Only words
// that hold at least one of its bytes are read; the buffers that hold texts
// start on a 4-byte boundary and end with kTextPad spare bytes, so every such
// word lies inside them.
constexpr int kTextPad = 4;

struct TextWords {
    const uint32_t *w;
    uint32_t cur;
    int mis, end, k;   // byte offset of the string in its first word, end of its bytes, next word
    __host__ __device__ __forceinline__ TextWords(const uint8_t *text, int n) {
        mis = (int)((uintptr_t)text & 3);
        w = reinterpret_cast<const uint32_t *>((uintptr_t)text - (uintptr_t)mis);
        end = mis + n;
        k = 1;
        cur = n > 0 ? w[0] : 0u;
    }
    // the next four characters, the first in the low byte (garbage past the end)
    __host__ __device__ __forceinline__ uint32_t next4() {
        const uint32_t nxt = 4 * k < end ? w[k] : 0u;
        ++k;
        const uint64_t both = ((uint64_t)nxt << 32) | cur;
        cur = nxt;
        return (uint32_t)(both >> (8 * mis));
    }
};
// The same, byte by byte, for a caller's buffer (no spare bytes).
struct TextBytes {
    const uint8_t *p;
    int n, j;
    __host__ __device__ __forceinline__ TextBytes(const uint8_t *text, int len) : p(text), n(len), j(0) {}
    __host__ __device__ __forceinline__ uint32_t next4() {
        uint32_t v = 0;
        for (int i = 0; i < 4; ++i)
            if (j + i < n) v |= (uint32_t)p[j + i] << (8 * i);
        j += 4;
        return v;
    }
};

// s = x + y over B 32-bit words (little-endian), one carry chain per eight words
template <int B>
__device__ __forceinline__ void add_words(uint32_t (&s)[B], const uint32_t (&x)[B], const uint32_t (&y)[B]) {
    if constexpr (B == 1) {
        s[0] = x[0] + y[0];
    } else if constexpr (B == 2) {
        asm("add.cc.u32 %0, %2, %4;\n\taddc.u32 %1, %3, %5;" : "=&r"(s[0]), "=r"(s[1]) : "r"(x[0]), "r"(x[1]), "r"(y[0]), "r"(y[1]));
    } else if constexpr (B == 4) {
        asm("add.cc.u32 %0, %4, %8;\n\taddc.cc.u32 %1, %5, %9;\n\taddc.cc.u32 %2, %6, %10;\n\taddc.u32 %3, %7, %11;"
            : "=&r"(s[0]), "=&r"(s[1]), "=&r"(s[2]), "=r"(s[3])
            : "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]));
    } else {
        static_assert(B % 8 == 0, "1, 2, 4 or a multiple of 8 words");
        uint32_t carry = 0;
#pragma unroll
        for (int b = 0; b < B; b += 8) {
            uint32_t t[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) t[i] = x[b + i];
            asm("{\n\t.reg .u32 z;\n\tadd.cc.u32 z, %8, 0xffffffff;\n\t"
                "addc.cc.u32 %0, %0, %9;\n\taddc.cc.u32 %1, %1, %10;\n\taddc.cc.u32 %2, %2, %11;\n\t"
                "addc.cc.u32 %3, %3, %12;\n\taddc.cc.u32 %4, %4, %13;\n\taddc.cc.u32 %5, %5, %14;\n\t"
                "addc.cc.u32 %6, %6, %15;\n\taddc.cc.u32 %7, %7, %16;\n\taddc.u32 %8, 0, 0;\n\t}"
                : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "+r"(t[6]), "+r"(t[7]),
                  "+r"(carry)
                : "r"(y[b]), "r"(y[b + 1]), "r"(y[b + 2]), "r"(y[b + 3]), "r"(y[b + 4]), "r"(y[b + 5]), "r"(y[b + 6]),
                  "r"(y[b + 7]));
#pragma unroll
            for (int i = 0; i < 8; ++i) s[b + i] = t[i];
        }
    }
}

// Bit-parallel Levenshtein distance (Myers 1999) between a pattern of length
// m, 1 <= m <= 32 B, given as match masks Peq[c * B + b] (bit i of word b set
// iff pattern[32 b + i] == c), and a text of n characters.  The state is the
// column of vertical deltas of the DP matrix in the bit vectors Pv (+1) and Mv
// (-1); every text symbol updates the whole column as one B-word integer: the
// addition's carry chain and the funnel shifts cross the words, so no
// horizontal delta is handed from block to block.  The top boundary row of
// global edit distance has horizontal delta +1, shifted into the lowest bit.
// The distance is D[m][n] = D[0][n] + the column's deltas = n + |Pv| - |Mv|
// over the pattern's m rows, counted once at the end.  Exact.
// The integer / logic pipe bounds it: 10 operations per word and symbol.  160 M
// pivot distances of 108 x 108 symbols take 40.6 ms; a block form with explicit
// horizontal deltas, a running score and one-byte text loads took 61.9 ms.
template <int B, class Text>
__device__ __forceinline__ int edit_bits(const uint32_t *__restrict__ Peq, int m, const uint8_t *__restrict__ text,
                                         int n) {
    uint32_t Pv[B], Mv[B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
        Pv[b] = ~0u;
        Mv[b] = 0u;
    }
    auto step = [&](uint32_t c) {
        uint32_t Eq[B], x[B], sum[B], Ph[B];
        const uint32_t *row = Peq + c * B;
        if constexpr (B % 4 == 0) {
#pragma unroll
            for (int b = 0; b < B; b += 4) {
                const uint4 v = *reinterpret_cast<const uint4 *>(row + b);
                Eq[b] = v.x;
                Eq[b + 1] = v.y;
                Eq[b + 2] = v.z;
                Eq[b + 3] = v.w;
            }
        } else if constexpr (B == 2) {
            const uint2 v = *reinterpret_cast<const uint2 *>(row);
            Eq[0] = v.x;
            Eq[1] = v.y;
        } else {
            Eq[0] = row[0];
        }
#pragma unroll
        for (int b = 0; b < B; ++b) x[b] = Eq[b] & Pv[b];
        add_words<B>(sum, x, Pv);
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const uint32_t Xh = (sum[b] ^ Pv[b]) | Eq[b];
            Ph[b] = Mv[b] | ~(Xh | Pv[b]);
            x[b] = Pv[b] & Xh;   // Mh
        }
#pragma unroll
        for (int b = B - 1; b >= 0; --b) {
            const uint32_t p = b > 0 ? __funnelshift_l(Ph[b > 0 ? b - 1 : 0], Ph[b], 1) : ((Ph[0] << 1) | 1u);
            const uint32_t h = b > 0 ? __funnelshift_l(x[b > 0 ? b - 1 : 0], x[b], 1) : (x[0] << 1);
            const uint32_t Xv = Eq[b] | Mv[b];
            Pv[b] = h | ~(Xv | p);
            Mv[b] = p & Xv;
        }
    };
    Text tr(text, n);
    int j = 0;
    for (; j + 4 <= n; j += 4) {
        const uint32_t c4 = tr.next4();
        step(c4 & 255u);
        step((c4 >> 8) & 255u);
        step((c4 >> 16) & 255u);
        step(c4 >> 24);
    }
    if (j < n) {
        uint32_t c4 = tr.next4();
        for (; j < n; ++j) {
            step(c4 & 255u);
            c4 >>= 8;
        }
    }
    int d = n;
#pragma unroll
    for (int b = 0; b < B; ++b) {
        const int left = m - 32 * b;
        const uint32_t valid = left >= 32 ? ~0u : left > 0 ? (1u << left) - 1u : 0u;
        d += __popc(Pv[b] & valid) - __popc(Mv[b] & valid);
    }
    return d;
}

// The same distance when it is at most t, or some value above t (Hyyro 2003,
// the diagonal band).  T: a 32-bit window for t <= 15, a 64-bit one for t <=
// 31 (2 t + 2 bits at least).  Bit b of column j stands for row j + b - t, so
// the window moves down one row per column and D0 is shifted right where the
// full form shifts the horizontal deltas left.  Rows above the first have no
// matches and no vertical deltas, which gives the top row its horizontal
// deltas of +1; the row entering at the bottom has D0 = 0, an upper bound of
// a cell outside the band that no path of cost <= t uses.  The score follows
// the diagonal that ends in D[m][n]: it never falls, so the text is left as
// soon as it passes t -- after some 20 symbols for unrelated reads and t = 8.
// Peq: rows of kBandRow words per character, the pattern's bits from bit 32 on
// (build_band_peq).
template <int B>
constexpr int kBandRow = B + 3;   // 32 zero bits, the pattern, zero words for the window's end (odd: no bank conflicts)

template <int B, class T>
__host__ __device__ __forceinline__ int edit_band(const uint32_t *__restrict__ Peq, int m,
                                                  const uint8_t *__restrict__ text, int n, int t) {
    if (m - n > t || n - m > t) return t + 1;
    T VP = (T)~(T)0 << t, VN = 0;
    const int diag = t + (m - n);   // the bit of the diagonal ending in (m, n), 0 .. 2 t
    int score = m > n ? m - n : 0;
    auto step = [&](uint32_t c, int j0) {
        const int pos = 32 + j0 - t, w = pos >> 5, sh = pos & 31;
        const uint32_t *row = Peq + c * kBandRow<B> + w;
        T Eq;
        if constexpr (sizeof(T) == 4) {
            Eq = (T)((((uint64_t)row[1] << 32) | row[0]) >> sh);
        } else {
            const uint32_t lo = (uint32_t)((((uint64_t)row[1] << 32) | row[0]) >> sh);
            const uint32_t hi = (uint32_t)((((uint64_t)row[2] << 32) | row[1]) >> sh);
            Eq = ((T)hi << 32) | lo;
        }
        const T D0 = ((((Eq & VP) + VP) ^ VP) | Eq) | VN;
        const T HP = VN | ~(D0 | VP);
        const T HN = D0 & VP;
        score += 1 - (int)((D0 >> diag) & 1);
        VP = HN | ~((D0 >> 1) | HP);
        VN = (D0 >> 1) & HP;
    };
    TextWords tr(text, n);
    int j = 0;
    for (; j + 4 <= n; j += 4) {
        const uint32_t c4 = tr.next4();
        step(c4 & 255u, j);
        step((c4 >> 8) & 255u, j + 1);
        step((c4 >> 16) & 255u, j + 2);
        step(c4 >> 24, j + 3);
        if (score > t) return score;
    }
    if (j < n) {
        uint32_t c4 = tr.next4();
        for (; j < n; ++j) {
            step(c4 & 255u, j);
            c4 >>= 8;
        }
    }
    return score;
}

// Fill the match masks of `pat` (length m, 1 <= m <= 32 B) into shared memory
// `Peq` (256 * B words).  Call with the whole block; ends with __syncthreads().
template <int B>
__device__ __forceinline__ void build_peq(uint32_t *Peq, const uint8_t *pat, int m) {
    for (int i = threadIdx.x; i < 256 * B; i += blockDim.x) Peq[i] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += blockDim.x) atomicOr(&Peq[(int)pat[i] * B + (i >> 5)], 1u << (i & 31));
    __syncthreads();
}
// The same in edit_band's layout (256 * kBandRow<B> words).
template <int B>
__device__ __forceinline__ void build_band_peq(uint32_t *Peq, const uint8_t *pat, int m) {
    for (int i = threadIdx.x; i < 256 * kBandRow<B>; i += blockDim.x) Peq[i] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += blockDim.x)
        atomicOr(&Peq[(int)pat[i] * kBandRow<B> + 1 + (i >> 5)], 1u << (i & 31));
    __syncthreads();
}

}  // namespace gts
