// um_score.cu -- query projection (S1) and row/column scores (S2-S3, Eq. 4
// and 6) on CUDA cores in fp32: the path of fp32 storage, and of bf16 layers
// whose rows TMA cannot read.  The query projection is split over D_i so that
// enough CTAs stream W_q; the split CTAs of a tile are a cluster, which adds
// their partial sums through distributed shared memory: in fp32 for the score
// kernel and, with fp32 storage, in fp64 for the selection (which computes the
// weights from it).  With fp32 storage each partial is a compensated dot
// product (Dot2); the scores here only decide which keys survive, and the
// selection recomputes the survivors' exactly.
// Measured on GB300 (decode_1m in fp32, 77 tokens; kernel spans in the call),
// with 32 x 64 tiles loaded element by element between barriers, the partials
// summed again by every score CTA and a full launch between the kernels ->
// this: query 19.8 -> 15.1 us, score 29.5 -> 11.5, projection 55.5 -> 32.5 (its
// fp32 pipe floor is 21), gather 15.5 -> 5.7, a forward 151.5 -> 83.2; tiny_fp32
// with 16 tokens 50.5 -> 28.7.
#include "um_dot.cuh"
#include "um_tc.cuh"

namespace um {
namespace {

using dot::kThreads;

// The value of a shared-memory location of CTA `rank` of the cluster.
__device__ __forceinline__ float ld_peer(const float *p, uint32_t rank) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];"
                 : "=f"(v)
                 : "r"(tc::mapa_shared(tc::smem_u32(p), rank))
                 : "memory");
    return v;
}

// One D_i slice of q = W_q x, a tile of tokens x outputs.  TX: the token
// rows' type (T, or fp32 for the convolved input x~ of Trick 4, which the
// caller then passes as p.x).  With `reduce` the splits of a tile are one
// cluster: q_part's split 0 gets their sum in fp32 and, with fp32 storage and
// several splits, split 1 the sum in fp64 rounded once; else (the query
// LayerNorm adds them itself) the partials are stored.
template <typename T, typename TX, int TPT, int NP>
__global__ void __launch_bounds__(kThreads) query_kernel(Dims d, Ptrs p, int reduce) {
    using Acc = dot::AccFor<T>;
    using S = dot::Shape<TPT, NP>;
    __shared__ dot::Stage<Acc, TPT, NP> st;
    static_assert(sizeof(st) >= sizeof(float) * S::TM * S::TN, "the partial tile fits the stage");
    pdl_wait();
    stamp_begin(p.stamp);
    pdl_trigger();
    const int a = blockIdx.z / d.q_splits, split = blockIdx.z % d.q_splits;
    const int HD = d.H * d.d_k, o_tiles = (HD + S::TN - 1) / S::TN;
    const int o0 = blockIdx.x % o_tiles * S::TN, b0 = blockIdx.x / o_tiles * S::TM;
    const int chunk = (d.d_in + d.q_splits - 1) / d.q_splits;
    dot::Operands<TX, T> o;
    o.A = static_cast<const TX *>(p.x);
    o.B = static_cast<const T *>(a == 0 ? p.w_q : p.w_q_col);
    o.lda = o.ldb = d.d_in;
    o.M = d.B;
    o.N = HD;
    o.kb = min(d.d_in, split * chunk);
    o.ke = min(d.d_in, o.kb + chunk);
    const bool quads = ((d.d_in | chunk) & 3) == 0;
    o.veca = quads && ((uintptr_t)o.A & (4 * sizeof(TX) - 1)) == 0;
    o.vecb = quads && ((uintptr_t)o.B & (4 * sizeof(T) - 1)) == 0;
    Acc acc[TPT][NP];
    dot::tile<Acc, TPT, NP, true>(o, b0, o0, st, acc, [](int) {});
    const int64_t plane = (int64_t)d.A * d.B * HD;
    float *q = p.q_part + (int64_t)a * d.B * HD;
    if (!reduce || d.q_splits == 1) {
        dot::each<Acc, TPT, NP>(acc, [&](int i, int j, float v) {
            if (b0 + i < d.B && o0 + j < HD)
                q[split * plane + (int64_t)(b0 + i) * HD + o0 + j] = v;
        });
    } else {
        float *part = reinterpret_cast<float *>(&st);   // [TM][TN]
        __syncthreads();
        dot::each<Acc, TPT, NP>(acc, [&](int i, int j, float v) { part[i * S::TN + j] = v; });
        tc::cluster_sync();
        for (int e = split * kThreads + threadIdx.x; e < S::TM * S::TN;
             e += d.q_splits * kThreads) {
            const int b = b0 + e / S::TN, c = o0 + e % S::TN;
            if (b >= d.B || c >= HD) continue;
            float v[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) v[r] = r < d.q_splits ? ld_peer(part + e, r) : 0.f;
            float sum = 0.f;
            double sum_d = 0.0;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                if (r < d.q_splits) {
                    sum += v[r];
                    sum_d += (double)v[r];
                }
            }
            q[(int64_t)b * HD + c] = sum;
            if (std::is_same<T, float>::value) q[plane + (int64_t)b * HD + c] = (float)sum_d;
        }
        tc::cluster_sync();   // the peers have read this CTA's tile
    }
    stamp_end(p.stamp);
}

// For each rank chunk alpha, S_alpha[b][i] = sum_{c < dk} key[h][i][alpha*dk + c]
// * q[b][h][alpha*dk + c] (Eq. 4 with the r x K x (D_k/r) reshape); the chunk
// scores are folded into the rank-1 score a = sum_alpha coef[alpha] S_alpha
// (coef = u for row keys, t for column keys, Eq. 6-7) and its
// order-preserving key is stored: akey[b][h][axis][i].
// Tile: 32 tokens x 64 keys; each thread owns 4 tokens x 4 keys.
template <typename T>
__global__ void __launch_bounds__(kThreads) score_kernel(Dims d, Ptrs p) {
    constexpr int TPT = 4, NP = 2;
    using Acc = dot::Plain2;
    using S = dot::Shape<TPT, NP>;
    __shared__ dot::Stage<Acc, TPT, NP> st;
    pdl_wait();
    stamp_begin(p.stamp);
    pdl_trigger();
    const int h = blockIdx.z >> 1, axis = blockIdx.z & 1;
    const int aq = (axis == 1 && d.A == 2) ? 1 : 0;
    const float *coef = (axis == 0 ? p.u : p.t) + (int64_t)h * d.r;
    const int i0 = blockIdx.x * S::TN, b0 = blockIdx.y * S::TM;
    const int HD = d.H * d.d_k;
    dot::Operands<float, T> o;
    o.A = p.q_part + (int64_t)aq * d.B * HD + h * d.d_k;
    o.B = static_cast<const T *>(axis == 0 ? p.k_row : p.k_col) + (int64_t)h * d.K * d.d_k;
    o.lda = HD;
    o.ldb = d.d_k;
    o.M = d.B;
    o.N = d.K;
    const bool quads = ((d.d_k | d.dk) & 3) == 0;
    o.veca = quads;   // q_part is the library's, HD and h D_k multiples of 4
    o.vecb = quads && ((uintptr_t)o.B & (4 * sizeof(T) - 1)) == 0;
    Acc acc[TPT][NP];
    f2 folded[TPT][NP];
    int al = 0;
    // the terms of chunk al are in: fold them in and start the next chunk
    auto fold = [&]() {
        const f2 cf = pack2(coef[al], coef[al]);
#pragma unroll
        for (int i = 0; i < TPT; ++i)
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                folded[i][j] = al == 0 ? mul2(cf, acc[i][j].s) : fma2(cf, acc[i][j].s, folded[i][j]);
                acc[i][j] = Acc();
            }
        ++al;
    };
    if (d.dk % dot::kK == 0) {   // whole stages a chunk: one pass over D_k
        o.kb = 0;
        o.ke = d.d_k;
        dot::tile<Acc, TPT, NP, true>(o, b0, i0, st, acc, [&](int k) {
            if (k == (al + 1) * d.dk) fold();
        });
    } else {
        while (al < d.r) {
            o.kb = al * d.dk;
            o.ke = o.kb + d.dk;
            dot::tile<Acc, TPT, NP, true>(o, b0, i0, st, acc, [](int) {});
            fold();
        }
    }
    const int tx = threadIdx.x % S::TX, ty = threadIdx.x / S::TX;
    const int i = i0 + 4 * tx;
#pragma unroll
    for (int t = 0; t < TPT; ++t) {
        const int b = b0 + TPT * ty + t;
        if (b >= d.B) continue;
        const float2 x = unpack2(folded[t][0]), y = unpack2(folded[t][1]);
        uint32_t *dst = p.akey + (((int64_t)b * d.H + h) * 2 + axis) * d.K + i;
        if ((d.K & 3) == 0) {
            if (i < d.K)
                *reinterpret_cast<uint4 *>(dst) = make_uint4(f2ord(x.x), f2ord(x.y), f2ord(y.x),
                                                             f2ord(y.y));
        } else {
            const uint32_t v[4] = {f2ord(x.x), f2ord(x.y), f2ord(y.x), f2ord(y.y)};
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (i + e < d.K) dst[e] = v[e];
        }
    }
    stamp_end(p.stamp);
}

template <typename T, typename TX, int TPT, int NP>
cudaError_t launch_query_t(const Dims &d, const Ptrs &p, bool reduce, cudaStream_t st) {
    using S = dot::Shape<TPT, NP>;
    const int HD = d.H * d.d_k;
    // tiles along x, outputs first (2^20 tokens are more tiles than y takes)
    dim3 grid(((HD + S::TN - 1) / S::TN) * ((d.B + S::TM - 1) / S::TM), 1, d.A * d.q_splits);
    const unsigned cl = reduce && d.q_splits > 1 ? (unsigned)d.q_splits : 1u;
    constexpr auto k = query_kernel<T, TX, TPT, NP>;
    const size_t sm = d.pdl ? spread_smem(0, static_smem_of<k>(), ctas_of(grid)) : 0;
    return launch_kernel(d.pdl, cl, k, grid, kThreads, sm, st, d, p, (int)reduce);
}
template <typename T, typename TX>
cudaError_t launch_query_x(const Dims &d, const Ptrs &p, bool reduce, cudaStream_t st) {
    const int64_t ctas = (int64_t)((d.H * d.d_k + 63) / 64) * ((d.B + 15) / 16) * d.A * d.q_splits;
    return dot::small_tiles(ctas) ? launch_query_t<T, TX, 1, 1>(d, p, reduce, st)
                                  : launch_query_t<T, TX, 2, 2>(d, p, reduce, st);
}

}  // namespace

cudaError_t launch_query(const Dims &d, const Ptrs &p, bool x_f32, bool reduce, cudaStream_t st) {
    if (d.q_splits > 8) return cudaErrorInvalidValue;   // one portable cluster
    if (d.dtype == ULTRAMEM_BF16)
        return x_f32 ? launch_query_x<__nv_bfloat16, float>(d, p, reduce, st)
                     : launch_query_x<__nv_bfloat16, __nv_bfloat16>(d, p, reduce, st);
    return launch_query_x<float, float>(d, p, reduce, st);
}

template <auto K> static cudaError_t allow_padded() {
    return cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(kSmemPerCta - static_smem_of<K>()));
}
template <typename T, typename TX> static cudaError_t allow_query() {
    cudaError_t e = allow_padded<query_kernel<T, TX, 2, 2>>();
    return e == cudaSuccess ? allow_padded<query_kernel<T, TX, 1, 1>>() : e;
}
cudaError_t configure_cuda_core() {
    cudaError_t e = allow_query<float, float>();
    if (e == cudaSuccess) e = allow_query<__nv_bfloat16, float>();
    if (e == cudaSuccess) e = allow_query<__nv_bfloat16, __nv_bfloat16>();
    if (e == cudaSuccess) e = allow_padded<score_kernel<float>>();
    if (e == cudaSuccess) e = allow_padded<score_kernel<__nv_bfloat16>>();
    return e;
}

cudaError_t launch_score(const Dims &d, const Ptrs &p, cudaStream_t st) {
    dim3 grid((d.K + 63) / 64, (d.B + 31) / 32, d.H * 2);
    // dependent launches of a few CTAs per SM are spread over the SMs (see
    // spread_smem)
    auto go = [&](auto kernel, size_t fixed) {
        return launch_kernel(d.pdl, kernel, grid, kThreads, spread_smem(0, fixed, ctas_of(grid)),
                             st, d, p);
    };
    return d.dtype == ULTRAMEM_BF16
               ? go(score_kernel<__nv_bfloat16>, static_smem_of<score_kernel<__nv_bfloat16>>())
               : go(score_kernel<float>, static_smem_of<score_kernel<float>>());
}

}  // namespace um
