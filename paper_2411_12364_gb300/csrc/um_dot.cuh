// um_dot.cuh -- the tiled contraction of the CUDA-core path (fp32 storage, and
// bf16 layers whose rows TMA cannot read): C[m][n] = sum_k A[m][k] B[n][k]
// over a slice of k, with each thread's sums taken in increasing k.
//
// fp32 storage sums by Dot2 (um_internal.cuh), ten fp32 operations a product,
// so the kernels are bound by the fp32 pipe: packed instructions take two
// outputs' operations each, which leaves half of the issue slots for the
// staging.  128 threads a CTA; the next 32 k of both operands are on their
// way into registers while the current ones are used from shared memory.
#pragma once

#include "um_internal.cuh"

namespace um {
namespace dot {

constexpr int kThreads = 128;
constexpr int kK = 32;   // k staged at once

// One pair of outputs' Dot2 sums (Dot2's steps, packed).  add takes the A
// value in both halves as it is and negated: with np = -(a b) rounded, every
// step of Dot2 is one packed instruction, and each half rounds as there.
// Products go into multiply-adds only: the compiler fuses a packed product
// with a packed sum that takes it, although both round on their own.
struct Dot2x2 {
    using Elem = float4;   // an A value as it is staged: (a, a, -a, -a)
    static __device__ __forceinline__ Elem stage(float a) { return make_float4(a, a, -a, -a); }
    f2 s, c;
    __device__ __forceinline__ Dot2x2() : s(0ull), c(0ull) {}
    __device__ __forceinline__ void add(f2 a, f2 na, f2 b) {
        const f2 m1 = 0xbf800000bf800000ull;               // (-1, -1)
        const f2 np = mul2(na, b);
        const f2 pe = fma2(a, b, np);                      // a b - p, exact
        const f2 t = fma2(np, m1, s);                      // s + p
        const f2 zn = fma2(t, m1, s);                      // -z = s - t
        const f2 v = fma2(add2(t, zn), m1, s);             // s - (t - z)
        const f2 w = fma2(np, m1, zn);                     // p - z
        s = t;
        c = add2(c, add2(v, w));
        c = add2(c, pe);
    }
    __device__ __forceinline__ float2 value() const { return unpack2(add2(s, c)); }
};
struct Plain2 {   // plain fp32 sums
    using Elem = float2;
    static __device__ __forceinline__ Elem stage(float a) { return make_float2(a, a); }
    f2 s;
    __device__ __forceinline__ Plain2() : s(0ull) {}
    __device__ __forceinline__ void add(f2 a, f2, f2 b) { s = fma2(a, b, s); }
    __device__ __forceinline__ float2 value() const { return unpack2(s); }
};

// The thread grid of a tile: TY threads along m (TPT rows each), TX along n
// (NP pairs of outputs each).
template <int TPT, int NP> struct Shape {
    static constexpr int TX = NP == 1 ? 32 : 16, TY = kThreads / TX;
    static constexpr int TM = TY * TPT, TN = TX * 2 * NP;   // 4, 16 or 32 x 64
};

template <class Acc, int TPT, int NP> struct Stage {
    using S = Shape<TPT, NP>;
    __align__(16) typename Acc::Elem a[kK][S::TM];
    __align__(16) float b[kK][S::TN];   // quads of columns swizzled, see quad_at
};

// Where row k of the staged B holds its quad (4 columns): swizzled, so that
// both the stores (8 quads of k of one column quad a warp) and the reads
// (neighbouring quads of a row) touch every bank once.
__device__ __forceinline__ int quad_at(int k, int quad) { return quad ^ ((k >> 2) & 7); }

// The operands: A rows of TA, B rows of TB (BK: B is [n][k], else [k][n]).
// vec: A's (and, with BK, B's) rows and k0 allow 16-byte reads of 4 values;
// vecb the same for B's rows along n (not BK).
template <typename TA, typename TB> struct Operands {
    const TA *A;
    const TB *B;
    int64_t lda, ldb;
    int M, N;      // rows of A and of the result's columns
    int kb, ke;    // the slice of k
    bool veca, vecb;
};

template <typename T> __device__ __forceinline__ void load4(const T *p, float (&v)[4], bool vec) {
    if constexpr (std::is_same<T, float>::value) {
        if (vec) {
            const float4 x = *reinterpret_cast<const float4 *>(p);
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
            return;
        }
    } else {
        if (vec) {
            const uint2 x = *reinterpret_cast<const uint2 *>(p);
            v[0] = __uint_as_float(x.x << 16);
            v[1] = __uint_as_float(x.x & 0xffff0000u);
            v[2] = __uint_as_float(x.y << 16);
            v[3] = __uint_as_float(x.y & 0xffff0000u);
            return;
        }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = to_f(p[e]);
}

// The tile's sums for rows m0 .. and columns n0 ..: acc[i][j] of this thread
// is row m0 + TPT ty + i, columns n0 + 2 (NP tx + j) and the next.  after(k):
// called once the terms below k are in (every kK of them, and at the end).
template <class Acc, int TPT, int NP, bool BK, typename TA, typename TB, class After>
__device__ __forceinline__ void tile(const Operands<TA, TB> &o, int m0, int n0,
                                     Stage<Acc, TPT, NP> &st, Acc (&acc)[TPT][NP], After after) {
    using S = Shape<TPT, NP>;
    constexpr int QA = S::TM * kK / 4, QB = S::TN * kK / 4;   // groups of 4 values
    constexpr int RA = (QA + kThreads - 1) / kThreads, RB = QB / kThreads;
    const int t = threadIdx.x, tx = t % S::TX, ty = t / S::TX;
    float va[RA][4], vb[RB][4];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < RA; ++i) {
            // neighbouring threads take neighbouring rows (conflict-free stores)
            const int e = t + i * kThreads, m = m0 + e % S::TM, k = k0 + 4 * (e / S::TM);
#pragma unroll
            for (int j = 0; j < 4; ++j) va[i][j] = 0.f;
            if (e < QA && m < o.M) {
                const TA *src = o.A + m * o.lda + k;
                if (k + 4 <= o.ke) load4(src, va[i], o.veca);
                else
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (k + j < o.ke) va[i][j] = to_f(src[j]);
            }
        }
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int e = t + i * kThreads;
#pragma unroll
            for (int j = 0; j < 4; ++j) vb[i][j] = 0.f;
            if (BK) {
                const int n = n0 + e / (kK / 4), k = k0 + 4 * (e % (kK / 4));
                if (n < o.N) {
                    const TB *src = o.B + n * o.ldb + k;
                    if (k + 4 <= o.ke) load4(src, vb[i], o.vecb);
                    else
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (k + j < o.ke) vb[i][j] = to_f(src[j]);
                }
            } else {
                const int k = k0 + e / (S::TN / 4), n = n0 + 4 * (e % (S::TN / 4));
                if (k < o.ke) {
                    const TB *src = o.B + k * o.ldb + n;
                    if (n + 4 <= o.N) load4(src, vb[i], o.vecb);
                    else
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (n + j < o.N) vb[i][j] = to_f(src[j]);
                }
            }
        }
    };
    fetch(o.kb);
    for (int k0 = o.kb; k0 < o.ke; k0 += kK) {
        __syncthreads();   // the previous 32 k have been used
#pragma unroll
        for (int i = 0; i < RA; ++i) {
            const int e = t + i * kThreads;
            if (e < QA)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    st.a[4 * (e / S::TM) + j][e % S::TM] = Acc::stage(va[i][j]);
        }
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int e = t + i * kThreads;
            if (BK) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    st.b[4 * (e % (kK / 4)) + j]
                        [4 * quad_at(4 * (e % (kK / 4)), e / (kK / 4) / 4) + e / (kK / 4) % 4] =
                            vb[i][j];
            } else {
                const int k = e / (S::TN / 4);
                *reinterpret_cast<float4 *>(&st.b[k][4 * quad_at(k, e % (S::TN / 4))]) =
                    make_float4(vb[i][0], vb[i][1], vb[i][2], vb[i][3]);
            }
        }
        __syncthreads();
        if (k0 + kK < o.ke) fetch(k0 + kK);
        // 8 k at a time (past ke: zeros, which leave the sums as they are)
        const int kn = min(kK, o.ke - k0);
#pragma unroll 1
        for (int k8 = 0; k8 < kn; k8 += 8)
#pragma unroll
        for (int kj = 0; kj < 8; ++kj) {
            const int kk = k8 + kj;
            f2 b[NP];
            if constexpr (NP == 2) {
                const ulonglong2 v =
                    *reinterpret_cast<const ulonglong2 *>(&st.b[kk][4 * quad_at(kk, tx)]);
                b[0] = v.x;
                b[1] = v.y;
            } else {
                b[0] = *reinterpret_cast<const f2 *>(
                    &st.b[kk][4 * quad_at(kk, tx >> 1) + 2 * (tx & 1)]);
            }
            if constexpr (sizeof(typename Acc::Elem) == 16) {
#pragma unroll
                for (int i = 0; i < TPT; ++i) {
                    const ulonglong2 a =
                        *reinterpret_cast<const ulonglong2 *>(&st.a[kk][TPT * ty + i]);
#pragma unroll
                    for (int j = 0; j < NP; ++j) acc[i][j].add(a.x, a.y, b[j]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < TPT; ++i) {
                    const f2 a = *reinterpret_cast<const f2 *>(&st.a[kk][TPT * ty + i]);
#pragma unroll
                    for (int j = 0; j < NP; ++j) acc[i][j].add(a, 0ull, b[j]);
                }
            }
        }
        after(min(k0 + kK, o.ke));
    }
}

// put(row, column, value) for the outputs of this thread.
template <class Acc, int TPT, int NP, class Put>
__device__ __forceinline__ void each(const Acc (&acc)[TPT][NP], Put put) {
    using S = Shape<TPT, NP>;
    const int tx = threadIdx.x % S::TX, ty = threadIdx.x / S::TX;
#pragma unroll
    for (int i = 0; i < TPT; ++i)
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            const float2 v = acc[i][j].value();
            put(TPT * ty + i, 2 * (NP * tx + j), v.x);
            put(TPT * ty + i, 2 * (NP * tx + j) + 1, v.y);
        }
}

// Whether a contraction takes 4-token tiles (an output pair a thread) instead
// of 16-token ones: `ctas` of the latter, four times as many of the former;
// each SM works through its share one after another, and the small tiles'
// shared-memory reads cost about a quarter more per product.
inline bool small_tiles(int64_t ctas) {
    const int64_t sms = device_sm_count();
    return 5 * ((4 * ctas + sms - 1) / sms) < 4 * 4 * ((ctas + sms - 1) / sms);
}

template <typename T>
using AccFor = typename std::conditional<std::is_same<T, float>::value, Dot2x2, Plain2>::type;

}  // namespace dot
}  // namespace um
