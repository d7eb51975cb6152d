// um_gather.cu -- S8 (weighted gather-sum grouped by virtual block, Eq. 15's
// inner V^T s^_p) and S9 on CUDA cores (the IVE projection o = sum_p W_p^T
// acc_p, used for fp32 storage; there with compensated sums, Dot2).
//
// Gather, one CTA per token.  Random 512-byte rows of a multi-GB table reach
// the HBM copy rate only with many rows in flight per SM (measured on GB300:
// about 6.8 TB/s from 32 warps per SM with 8 rows each), so the main kernel
// keeps few registers per thread:
//   * the token's H*m slots are bucketed by virtual block p with a stable
//     counting sort in shared memory (ballots per block, a scan over warps);
//   * each warp serves one block, so a lane owns 16 bytes of every row and
//     8 fp32 accumulators, and issues 8 row loads before using any;
//   * 16 warps per CTA, two CTAs per SM; the warps of a block are summed in a
//     fixed order at the end (deterministic).
// Wider rows or more slots take the per-lane multi-block kernels below.  Row
// loads bypass L1 (read-only path).
//
// fp32 storage accumulates with compensated sums (Dot2; the general kernels in
// fp64): the fp32 mode's outputs carry the working precision element by
// element (see Dot2 in um_internal.cuh), and its projection reads fp32 pooled
// rows that are rounded once.
//
// Multi-Core Scoring (Eq. 17): a slot has nc weights and weight i scales
// columns [i*D_v/nc, (i+1)*D_v/nc) of the row.  Slices are whole 16-byte
// vectors (D_v/nc is a multiple of 8), so a lane's vector lies in one slice
// and the lane picks that slice's weight.
#include "um_dot.cuh"
#include "um_internal.cuh"

namespace um {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kUnroll = 8;   // rows in flight per warp

__device__ __forceinline__ uint4 ld_stream(const void *ptr) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(ptr));
    return v;
}

// The accumulator type of a gather: fp64 for fp32 storage, else fp32.
template <typename T>
using AccOf = typename std::conditional<std::is_same<T, float>::value, double, float>::type;

__device__ __forceinline__ float mul_add(float w, float v, float acc) { return fmaf(w, v, acc); }
__device__ __forceinline__ double mul_add(float w, float v, double acc) {
    return fma((double)w, (double)v, acc);
}

// add w * (8 bf16 or 4 fp32 packed in 16 bytes) into dst
template <typename A>
__device__ __forceinline__ void fma_vec(A *dst, uint4 v, float w, __nv_bfloat16) {
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float lo = __uint_as_float(u[q] << 16), hi = __uint_as_float(u[q] & 0xffff0000u);
        dst[2 * q] = mul_add(w, lo, dst[2 * q]);
        dst[2 * q + 1] = mul_add(w, hi, dst[2 * q + 1]);
    }
}
template <typename A>
__device__ __forceinline__ void fma_vec(A *dst, uint4 v, float w, float) {
    dst[0] = mul_add(w, __uint_as_float(v.x), dst[0]);
    dst[1] = mul_add(w, __uint_as_float(v.y), dst[1]);
    dst[2] = mul_add(w, __uint_as_float(v.z), dst[2]);
    dst[3] = mul_add(w, __uint_as_float(v.w), dst[3]);
}

template <typename T>
__device__ __forceinline__ void unpack(uint4 v, float (&f)[16 / sizeof(T)]);
template <>
__device__ __forceinline__ void unpack<__nv_bfloat16>(uint4 v, float (&f)[8]) {
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        f[2 * q] = __uint_as_float(u[q] << 16);
        f[2 * q + 1] = __uint_as_float(u[q] & 0xffff0000u);
    }
}
template <>
__device__ __forceinline__ void unpack<float>(uint4 v, float (&f)[4]) {
    f[0] = __uint_as_float(v.x);
    f[1] = __uint_as_float(v.y);
    f[2] = __uint_as_float(v.z);
    f[3] = __uint_as_float(v.w);
}

// Register-accumulating gather for E <= EMAX blocks and rows of at most
// 32 vectors (one 16-byte vector per lane).  Each warp takes a contiguous
// run of the token's H*m slots; their (row, block, weight) are loaded once,
// one slot per lane, and broadcast by shuffle; 8 value loads per warp are
// in flight together.
template <typename T, int EMAX>
__global__ void __launch_bounds__(kThreads) gather_reg_kernel(Dims d, Ptrs p) {
    using A = AccOf<T>;
    extern __shared__ __align__(16) unsigned char red_raw[];
    A *red = reinterpret_cast<A *>(red_raw);   // [kWarps][E][D_v]
    constexpr int EPV = 16 / sizeof(T);
    const int b = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int EDv = d.E * d.d_v;
    const int VPR = d.d_v / EPV;          // vectors per row, <= 32 here
    const bool active = lane < VPR;
    const int hm = d.H * d.m;
    const int64_t base = (int64_t)b * hm;
    const T *V = static_cast<const T *>(p.values) + lane * EPV;
    const int per_warp = (hm + kWarps - 1) / kWarps;
    const int e_begin = min(hm, warp * per_warp), e_end = min(hm, e_begin + per_warp);
    pdl_wait();
    stamp_begin(p.stamp);
    pdl_trigger();
    A acc[EMAX][EPV];
#pragma unroll
    for (int q = 0; q < EMAX; ++q)
#pragma unroll
        for (int c = 0; c < EPV; ++c) acc[q][c] = 0;

    for (int c0 = e_begin; c0 < e_end; c0 += 32) {
        const int n = min(32, e_end - c0);
        int row_l = 0, blk_l = -1;
        float w_l = 0.f;
        if (lane < n) {
            row_l = p.sel_row[base + c0 + lane];
            blk_l = p.sel_p[base + c0 + lane];
            w_l = p.sel_w[base + c0 + lane];
        }
        for (int j0 = 0; j0 < n; j0 += kUnroll) {
            uint4 val[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const int j = j0 + u;
                const int row = __shfl_sync(0xffffffffu, row_l, j & 31);
                val[u] = (j < n && active) ? ld_stream(V + (int64_t)row * d.d_v)
                                           : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const int j = j0 + u;
                const int blk = __shfl_sync(0xffffffffu, blk_l, j & 31);
                const float w = j < n ? __shfl_sync(0xffffffffu, w_l, j & 31) : 0.f;
                float f[EPV];
                unpack<T>(val[u], f);
#pragma unroll
                for (int q = 0; q < EMAX; ++q) {
                    const float wq = blk == q ? w : 0.f;   // branch-free block select
#pragma unroll
                    for (int c = 0; c < EPV; ++c) acc[q][c] = mul_add(wq, f[c], acc[q][c]);
                }
            }
        }
    }
    // sum the warps' partial accumulators
    if (active)
#pragma unroll
        for (int q = 0; q < EMAX; ++q)
            if (q < d.E)
#pragma unroll
                for (int c = 0; c < EPV; ++c)
                    red[(size_t)warp * EDv + q * d.d_v + lane * EPV + c] = acc[q][c];
    __syncthreads();
    for (int i = threadIdx.x; i < EDv; i += kThreads) {
        A s = 0;
#pragma unroll
        for (int wv = 0; wv < kWarps; ++wv) s += red[(size_t)wv * EDv + i];
        store_pooled<T>(d, p, b, i, (float)s);
    }
    stamp_end(p.stamp);
}

constexpr int kBMaxE = 16;
constexpr int kMaxCores = 8;   // MCS component cores per head

// bytes of one accumulator of the layer's gather (fp32 storage: fp64, or the
// two halves of a Dot2)
size_t acc_bytes(const Dims &d) { return d.dtype == ULTRAMEM_F32 ? 8 : 4; }

size_t bucket_smem_bytes(const Dims &d, int warps) {
    const int hm = d.H * d.m;
    return acc_bytes(d) * (size_t)warps * d.d_v + sizeof(int) * (size_t)hm +
           sizeof(float) * (size_t)hm * d.nc;
}

// The bucketed gathers' slots: a stable counting sort of token b's slots by
// block (slot order kept within a block) into row_s and w_s, block q's at
// start[q] .. start[q] + tot[q].  ADDR: the slots come as given addresses and
// weights (p.idx_in, p.w_in) instead of the selection's sel_row / sel_p /
// sel_w, and each thread works its slot out itself: the slots kernel before
// the gather, its launch and the round trip of 12 bytes a slot through memory
// go.  Whole block; ends with a barrier.
template <int THREADS, bool ADDR>
__device__ __forceinline__ void bucket_slots(const Dims &d, const Ptrs &p, int64_t base, int hm,
                                             int (*wcnt)[kBMaxE], int *tot, int *start,
                                             int *row_s, float *w_s) {
    constexpr int kBWarps = THREADS / 32;
    const int E = d.E, nc = d.nc;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    int row = 0, blk = -1;
    float w[kMaxCores];   // the slot's weight, or its nc slice weights (MCS)
#pragma unroll
    for (int ci = 0; ci < kMaxCores; ++ci) w[ci] = 0.f;
    if (t < hm) {
        if constexpr (ADDR) {   // an invalid address weighs 0
            const bool ok = slot_of_address(d, p, p.idx_in[base + t], row, blk);
#pragma unroll
            for (int ci = 0; ci < kMaxCores; ++ci)
                if (ci < nc) w[ci] = ok ? p.w_in[(base + t) * nc + ci] : 0.f;
        } else {
            row = p.sel_row[base + t];
            blk = p.sel_p[base + t];
#pragma unroll
            for (int ci = 0; ci < kMaxCores; ++ci)
                if (ci < nc) w[ci] = p.sel_w[(base + t) * nc + ci];
        }
        if (blk < 0 || blk >= E) blk = -1;   // not a slot of this layer: skipped
    }
    int rank = 0;
    for (int q = 0; q < E; ++q) {
        const unsigned m = __ballot_sync(0xffffffffu, blk == q);
        if (blk == q) rank = __popc(m & ((1u << lane) - 1u));
        if (lane == 0) wcnt[warp][q] = __popc(m);
    }
    __syncthreads();
    if (t < E) {
        int run = 0;
        for (int wv = 0; wv < kBWarps; ++wv) {
            const int c = wcnt[wv][t];
            wcnt[wv][t] = run;
            run += c;
        }
        tot[t] = run;
    }
    __syncthreads();
    if (t == 0) {
        int run = 0;
        for (int q = 0; q < E; ++q) {
            start[q] = run;
            run += tot[q];
        }
    }
    __syncthreads();
    if (blk >= 0) {
        const int pos = start[blk] + wcnt[warp][blk] + rank;
        row_s[pos] = row;
#pragma unroll
        for (int ci = 0; ci < kMaxCores; ++ci)
            if (ci < nc) w_s[pos * nc + ci] = w[ci];
    }
    __syncthreads();
}

// The bucketed gather of bf16 rows (a 16-byte vector a lane).
// THREADS = 512 (2 CTAs per SM) for batches up to about two CTAs per SM,
// where each token's latency matters; 256 (4 CTAs per SM) for longer
// grids, where CTAs in their bucketing or reduction phase overlap others'
// loads (measured: 6.5 TB/s over 2.15 GB at 16384 tokens, against 5.4 with
// 512).  fp32 rows have a kernel of their own below: as one template with
// theirs this one's code came out slower, 3.2 -> 3.7 us at decode_1m with 64
// tokens, 4.6 -> 5.2 at mid_4m with 32.
template <int THREADS, bool ADDR>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) gather_bucket_kernel(Dims d, Ptrs p) {
    using T = __nv_bfloat16;
    constexpr int kBThreads = THREADS, kBWarps = THREADS / 32;
    extern __shared__ __align__(16) unsigned char gsm[];
    __shared__ int wcnt[kBWarps][kBMaxE];   // per warp and block: count, then offset
    __shared__ int tot[kBMaxE], start[kBMaxE];
    constexpr int EPV = 16 / sizeof(T);
    const int b = blockIdx.x, E = d.E, hm = d.H * d.m, Dv = d.d_v;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int64_t base = (int64_t)b * hm;
    float *red = reinterpret_cast<float *>(gsm);                 // [kBWarps][D_v]
    int *row_s = reinterpret_cast<int *>(red + kBWarps * Dv);    // [hm] bucketed rows
    float *w_s = reinterpret_cast<float *>(row_s + hm);          // [hm][nc] their weights
    const int nc = d.nc;
    pdl_wait();
    stamp_begin(p.stamp);
    pdl_trigger();
    bucket_slots<THREADS, ADDR>(d, p, base, hm, wcnt, tot, start, row_s, w_s);

    // warps [q*wpb, (q+1)*wpb) serve block q, each a contiguous share
    const int wpb = kBWarps / E;
    const int q = warp / wpb, sub = warp - q * wpb;
    const bool active = lane * EPV < Dv;
    const int wsel = nc == 1 || !active ? 0 : (lane * EPV) / (Dv / nc);   // this lane's slice
    const T *V = static_cast<const T *>(p.values) + lane * EPV;
    float acc[EPV];
#pragma unroll
    for (int c = 0; c < EPV; ++c) acc[c] = 0.f;
    if (q < E) {
        const int n = tot[q], per = (n + wpb - 1) / wpb;
        const int lo = start[q] + min(n, sub * per), hi = start[q] + min(n, (sub + 1) * per);
        for (int j0 = lo; j0 < hi; j0 += kUnroll) {
            uint4 val[kUnroll];
            float wu[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const int j = j0 + u;
                const bool ok = j < hi;
                wu[u] = ok ? w_s[j * nc + wsel] : 0.f;
                val[u] = (ok && active) ? ld_stream(V + (int64_t)row_s[j] * Dv)
                                        : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                float f[EPV];
                unpack<T>(val[u], f);
#pragma unroll
                for (int c = 0; c < EPV; ++c) acc[c] = mul_add(wu[u], f[c], acc[c]);
            }
        }
        if (active)
#pragma unroll
            for (int c = 0; c < EPV; ++c) red[warp * Dv + lane * EPV + c] = acc[c];
    }
    __syncthreads();
    const int EDv = E * Dv;
    for (int i = t; i < EDv; i += kBThreads) {
        const int qq = i / Dv, c = i - qq * Dv;
        float sum = 0.f;
        for (int sb = 0; sb < wpb; ++sb) sum += red[(qq * wpb + sb) * Dv + c];
        store_pooled<T>(d, p, b, i, sum);
    }
    stamp_end(p.stamp);
}

// The same for fp32 rows, with compensated sums (Dot2).  VPL: 16-byte vectors
// of a row that a lane owns (2: rows of up to 256 values; half as many rows in
// flight).  A sum and its error term take twice the registers of a plain sum,
// so half as many CTAs per SM.  Dot2 has fp32's range: a sum that is not finite
// (it may have passed FLT_MAX on the way) or so small that its products' error
// terms may have underflowed is taken again in fp64.
constexpr float kDot2Min = 0x1p-96f;   // products that lose error terms are below 2^-101
template <int THREADS, int VPL>
__global__ void __launch_bounds__(THREADS, 512 / THREADS) gather_bucket_exact(Dims d, Ptrs p) {
    using T = float;
    constexpr int kBThreads = THREADS, kBWarps = THREADS / 32, kRows = kUnroll / VPL;
    extern __shared__ __align__(16) unsigned char gsm[];
    __shared__ int wcnt[kBWarps][kBMaxE];   // per warp and block: count, then offset
    __shared__ int tot[kBMaxE], start[kBMaxE];
    constexpr int EPV = 16 / sizeof(T);
    const int b = blockIdx.x, E = d.E, hm = d.H * d.m, Dv = d.d_v;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int64_t base = (int64_t)b * hm;
    float2 *red = reinterpret_cast<float2 *>(gsm);   // the warps' s and c of Dot2 [kBWarps][D_v]
    int *row_s = reinterpret_cast<int *>(red + kBWarps * Dv);    // [hm] bucketed rows
    float *w_s = reinterpret_cast<float *>(row_s + hm);          // [hm][nc] their weights
    const int nc = d.nc;
    pdl_wait();
    stamp_begin(p.stamp);
    pdl_trigger();
    bucket_slots<THREADS, false>(d, p, base, hm, wcnt, tot, start, row_s, w_s);

    // warps [q*wpb, (q+1)*wpb) serve block q, each a contiguous share
    const int wpb = kBWarps / E;
    const int q = warp / wpb, sub = warp - q * wpb;
    bool active[VPL];
    int wsel[VPL];   // the slice that a vector lies in
#pragma unroll
    for (int x = 0; x < VPL; ++x) {
        const int c0 = (lane + 32 * x) * EPV;
        active[x] = c0 < Dv;
        wsel[x] = nc == 1 || !active[x] ? 0 : c0 / (Dv / nc);
    }
    const T *V = static_cast<const T *>(p.values) + lane * EPV;
    dot::Dot2x2 ex[VPL][EPV / 2];   // pairs of columns
    if (q < E) {
        const int n = tot[q], per = (n + wpb - 1) / wpb;
        const int lo = start[q] + min(n, sub * per), hi = start[q] + min(n, (sub + 1) * per);
        for (int j0 = lo; j0 < hi; j0 += kRows) {
            uint4 val[kRows][VPL];
            float wu[kRows][VPL];
#pragma unroll
            for (int u = 0; u < kRows; ++u) {
                const int j = j0 + u;
                const bool ok = j < hi;
#pragma unroll
                for (int x = 0; x < VPL; ++x) {
                    wu[u][x] = ok ? w_s[j * nc + wsel[x]] : 0.f;
                    val[u][x] = (ok && active[x])
                                    ? ld_stream(V + (int64_t)row_s[j] * Dv + 32 * x * EPV)
                                    : make_uint4(0, 0, 0, 0);
                }
            }
#pragma unroll
            for (int u = 0; u < kRows; ++u)
#pragma unroll
                for (int x = 0; x < VPL; ++x) {
                    float f[EPV];
                    unpack<T>(val[u][x], f);
                    const f2 w2 = pack2(wu[u][x], wu[u][x]), n2 = pack2(-wu[u][x], -wu[u][x]);
#pragma unroll
                    for (int c = 0; c < EPV; c += 2) ex[x][c / 2].add(w2, n2, pack2(f[c], f[c + 1]));
                }
        }
#pragma unroll
        for (int x = 0; x < VPL; ++x)
            if (active[x])
#pragma unroll
                for (int c = 0; c < EPV; ++c) {
                    const float2 sv = unpack2(ex[x][c / 2].s), cv = unpack2(ex[x][c / 2].c);
                    red[warp * Dv + (lane + 32 * x) * EPV + c] =
                        c & 1 ? make_float2(sv.y, cv.y) : make_float2(sv.x, cv.x);
                }
    }
    __syncthreads();
    const int EDv = E * Dv;
    for (int i = t; i < EDv; i += kBThreads) {
        const int qq = i / Dv, c = i - qq * Dv;
        Dot2 all;
        for (int sb = 0; sb < wpb; ++sb) {
            const float2 v = red[(qq * wpb + sb) * Dv + c];
            Dot2 o;
            o.s = v.x;
            o.c = v.y;
            all.merge(o);
        }
        float sum = all.value_any();
        if (!(fabsf(sum) >= kDot2Min && fabsf(sum) < INFINITY)) {
            const float *col = static_cast<const float *>(p.values) + c;
            const int ws = nc == 1 ? 0 : c / (Dv / nc);
            double s = 0.0;
            for (int j = start[qq]; j < start[qq] + tot[qq]; ++j)
                s += (double)w_s[j * nc + ws] * (double)col[(int64_t)row_s[j] * Dv];
            sum = (float)s;
        }
        store_pooled<T>(d, p, b, i, sum);
    }
    stamp_end(p.stamp);
}

// Long batches with a virtual expansion (bf16): one warp per (token, block),
// four to a CTA, nothing shared between them.  A warp reads its token's slots,
// keeps those of its block (ballots; slot order) in its own list, and sums
// their rows, 8 in flight, a lane owning 16 bytes of each, so that the pooled
// entries leave as 16-byte stores.  Against a CTA per token that sorts its
// slots by block together: no barriers, no sums of several warps, and the SM
// refills a warp at a time.  Bound: HBM.  Measured on GB300 (a call): decode_1m
// with 2000 tokens and the query extras 157.0 -> 149.4 us (its gather 23 -> 16),
// a lookup of 2048 tokens at mid_4m 84.0 -> 79.1, prefill_16k 1902 -> 1888
// (376 us for 2.2 GB, 5.9 TB/s); with component cores, whose weights are
// another dependent read, it is slower (180 -> 186 us at mid_4m with 1000).
// HALVES (E = 4): the block's rows as two sums, of the first and the second
// half, which are the sums of the bucketed gather's two warps a block, bit for
// bit.  Else (E = 9, 16, which took the general kernel's eight partial sums
// before) 8 rows at a time by a tree: at most n / 8 + 5 roundings on the way to
// a sum of n rows, no more than the n / 8 + 8 there.
constexpr int kGWarps = 4;
constexpr int kGSlots = 256;   // slots a token
template <bool ADDR, bool HALVES>
__global__ void __launch_bounds__(32 * kGWarps, 32 / kGWarps) gather_warp_kernel(Dims d, Ptrs p) {
    extern __shared__ __align__(16) unsigned char gsm[];
    constexpr int EPV = 8;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int hm = d.H * d.m, Dv = d.d_v;
    const int64_t gw = (int64_t)blockIdx.x * kGWarps + warp;
    const int64_t b = gw / d.E;
    const int q = (int)(gw - b * d.E);
    float4 *first_s = reinterpret_cast<float4 *>(gsm) + warp * 64;   // the first half's sums
    int *row_s = reinterpret_cast<int *>(gsm + kGWarps * 1024) + warp * 2 * hm;   // its list
    float *w_s = reinterpret_cast<float *>(row_s + hm);
    pdl_wait();
    stamp_begin(p.stamp);
    pdl_trigger();
    if (b < d.B) {   // warp-uniform
        const int64_t base = b * hm;
        int n = 0;
        for (int j0 = 0; j0 < hm; j0 += 128) {   // 4 slots a lane: their loads together
            int row[4], blk[4];
            float w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = j0 + 32 * u + lane;
                blk[u] = -1;
                row[u] = 0;
                w[u] = 0.f;
                if (j < hm) {
                    if constexpr (ADDR) {   // an invalid address weighs 0
                        w[u] = p.w_in[base + j];
                        if (!slot_of_address(d, p, p.idx_in[base + j], row[u], blk[u])) w[u] = 0.f;
                    } else {
                        row[u] = p.sel_row[base + j];
                        blk[u] = p.sel_p[base + j];
                        w[u] = p.sel_w[base + j];
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned mine = __ballot_sync(0xffffffffu, blk[u] == q);
                if (blk[u] == q) {
                    const int at = n + __popc(mine & ((1u << lane) - 1u));
                    row_s[at] = row[u];
                    w_s[at] = w[u];
                }
                n += __popc(mine);
            }
        }
        __syncwarp();
        const bool active = lane * EPV < Dv;
        const __nv_bfloat16 *V = static_cast<const __nv_bfloat16 *>(p.values) + lane * EPV;
        float acc[EPV];
        const int half = HALVES ? (n + 1) / 2 : 0;
#pragma unroll 1
        for (int part = HALVES ? 0 : 1; part < 2; ++part) {
            const int lo = part ? half : 0, hi = part ? n : half;
#pragma unroll
            for (int c = 0; c < EPV; ++c) acc[c] = 0.f;
#pragma unroll 1
            for (int j0 = lo; j0 < hi; j0 += kUnroll) {
                uint4 val[kUnroll];
                float wu[kUnroll];
#pragma unroll
                for (int u = 0; u < kUnroll; ++u) {
                    const int j = j0 + u;
                    const bool ok = j < hi;
                    wu[u] = ok ? w_s[j] : 0.f;
                    val[u] = (ok && active) ? ld_stream(V + (int64_t)row_s[j] * Dv)
                                            : make_uint4(0, 0, 0, 0);
                }
                if constexpr (HALVES) {
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u) {
                        float f[EPV];
                        unpack<__nv_bfloat16>(val[u], f);
#pragma unroll
                        for (int c = 0; c < EPV; ++c) acc[c] = fmaf(wu[u], f[c], acc[c]);
                    }
                } else {   // the 8 rows by a tree
                    static_assert(kUnroll == 8, "pairs, fours, eight");
                    float four[EPV];
#pragma unroll
                    for (int u = 0; u < kUnroll; u += 4) {
                        float f0[EPV], f1[EPV], two[EPV];
                        unpack<__nv_bfloat16>(val[u], f0);
                        unpack<__nv_bfloat16>(val[u + 1], f1);
#pragma unroll
                        for (int c = 0; c < EPV; ++c)
                            two[c] = fmaf(wu[u + 1], f1[c], wu[u] * f0[c]);
                        unpack<__nv_bfloat16>(val[u + 2], f0);
                        unpack<__nv_bfloat16>(val[u + 3], f1);
#pragma unroll
                        for (int c = 0; c < EPV; ++c) {
                            const float s4 =
                                two[c] + fmaf(wu[u + 3], f1[c], wu[u + 2] * f0[c]);
                            if (u == 0) four[c] = s4;
                            else acc[c] += four[c] + s4;
                        }
                    }
                }
            }
            if (HALVES && !part) {
                first_s[lane] = make_float4(acc[0], acc[1], acc[2], acc[3]);
                first_s[32 + lane] = make_float4(acc[4], acc[5], acc[6], acc[7]);
            }
        }
        if (HALVES) {
            const float4 x = first_s[lane], y = first_s[32 + lane];
            const float h[EPV] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
            for (int c = 0; c < EPV; ++c) acc[c] = h[c] + acc[c];
        }
        if (active) store_pooled8(d, p, b, q * Dv + lane * EPV, acc);
    }
    stamp_end(p.stamp);
}

// Shared-memory-accumulating gather for any E and row width (A: the
// accumulator, fp64 for fp32 storage while [kWarps][E][D_v] of it fits).
template <typename T, typename A>
__global__ void __launch_bounds__(kThreads) gather_kernel(Dims d, Ptrs p) {
    extern __shared__ __align__(16) unsigned char acc_raw[];
    A *acc_w = reinterpret_cast<A *>(acc_raw);   // [kWarps][E][D_v]
    const int b = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int EDv = d.E * d.d_v;
    pdl_wait();
    stamp_begin(p.stamp);
    pdl_trigger();
    A *mine = acc_w + (size_t)warp * EDv;
    for (int i = lane; i < EDv; i += 32) mine[i] = 0;
    __syncwarp();

    constexpr int EPV = 16 / sizeof(T);   // elements per 16-byte vector
    const int VPR = d.d_v / EPV;          // vectors per row
    const int hm = d.H * d.m;
    const int64_t base = (int64_t)b * hm;
    const T *V = static_cast<const T *>(p.values);
    for (int e0 = warp * kUnroll; e0 < hm; e0 += kWarps * kUnroll) {
        int row[kUnroll], blk[kUnroll];
        float w[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            int e = e0 + u;
            bool ok = e < hm;
            row[u] = ok ? p.sel_row[base + e] : 0;
            blk[u] = ok ? p.sel_p[base + e] : 0;
            w[u] = ok && d.nc == 1 ? p.sel_w[base + e] : 0.f;
        }
        for (int vv = lane; vv < VPR; vv += 32) {
            uint4 val[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u)
                val[u] = (e0 + u < hm) ? ld_stream(V + (int64_t)row[u] * d.d_v + vv * EPV)
                                       : make_uint4(0, 0, 0, 0);
            if (d.nc > 1) {   // MCS: the weight of this vector's value slice
                const int ws = (vv * EPV) / (d.d_v / d.nc);
#pragma unroll
                for (int u = 0; u < kUnroll; ++u)
                    if (e0 + u < hm) w[u] = p.sel_w[(base + e0 + u) * d.nc + ws];
            }
#pragma unroll
            for (int u = 0; u < kUnroll; ++u)
                if (e0 + u < hm) fma_vec(mine + blk[u] * d.d_v + vv * EPV, val[u], w[u], T());
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < EDv; i += kThreads) {
        A s = 0;
#pragma unroll
        for (int wv = 0; wv < kWarps; ++wv) s += acc_w[(size_t)wv * EDv + i];
        store_pooled<T>(d, p, b, i, (float)s);
    }
    stamp_end(p.stamp);
}

// proj_part[split][b][o] = sum over this split's slice of E*D_v of acc[b][c] W[c][o]
// (W = the E projectors stacked: [E*D_v][D'_v]); fp32 storage: compensated
// sums (Dot2), each partial to the working precision.
template <typename T, int TPT, int NP>
__global__ void __launch_bounds__(dot::kThreads) proj_kernel(Dims d, Ptrs p) {
    using Acc = dot::AccFor<T>;
    using S = dot::Shape<TPT, NP>;
    __shared__ dot::Stage<Acc, TPT, NP> st;
    const int Kd = d.E * d.d_v, split = blockIdx.z;
    const int chunk = (Kd + d.p_splits - 1) / d.p_splits;
    const int o_tiles = (d.d_out + S::TN - 1) / S::TN;
    const int o0 = blockIdx.x % o_tiles * S::TN, b0 = blockIdx.x / o_tiles * S::TM;
    pdl_wait();
    stamp_begin(p.stamp);
    pdl_trigger();
    dot::Operands<float, T> o;
    o.A = p.acc;
    o.B = static_cast<const T *>(p.w_proj);
    o.lda = Kd;
    o.ldb = d.d_out;
    o.M = d.B;
    o.N = d.d_out;
    o.kb = min(Kd, split * chunk);
    o.ke = min(Kd, o.kb + chunk);
    o.veca = ((Kd | chunk) & 3) == 0;   // acc is the library's, 16-byte aligned
    o.vecb = (d.d_out & 3) == 0 && ((uintptr_t)o.B & (4 * sizeof(T) - 1)) == 0;
    Acc acc[TPT][NP];
    dot::tile<Acc, TPT, NP, false>(o, b0, o0, st, acc, [](int) {});
    dot::each<Acc, TPT, NP>(acc, [&](int i, int j, float v) {
        if (b0 + i < d.B && o0 + j < d.d_out)
            p.proj_part[((int64_t)split * d.B + b0 + i) * d.d_out + o0 + j] = v;
    });
    stamp_end(p.stamp);
}

// out = the sum of the split-K partials (fp32 storage: compensated, one
// rounding of the output)
template <typename T>
__global__ void proj_reduce_kernel(Dims d, Ptrs p) {
    pdl_wait();
    stamp_begin(p.stamp);
    pdl_trigger();
    const int64_t total = (int64_t)d.B * d.d_out;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        float v[8], out;
#pragma unroll
        for (int sp = 0; sp < 8; ++sp)
            v[sp] = sp < d.p_splits ? p.proj_part[(int64_t)sp * total + i] : 0.f;
        if constexpr (std::is_same<T, float>::value) {
            Dot2 sum;
#pragma unroll
            for (int sp = 0; sp < 8; ++sp) sum.two_sum_into(v[sp]);
            out = sum.value_any();
            if (!(fabsf(out) < INFINITY)) {   // beyond fp32's range on the way, perhaps
                double s = 0.0;
#pragma unroll
                for (int sp = 0; sp < 8; ++sp) s += (double)v[sp];
                out = (float)s;
            }
        } else {
            out = 0.f;
#pragma unroll
            for (int sp = 0; sp < 8; ++sp)
                if (sp < d.p_splits) out += v[sp];
        }
        static_cast<T *>(p.out)[i] = from_f<T>(out);
    }
    stamp_end(p.stamp);
}

}  // namespace

size_t gather_smem_bytes(const Dims &d) { return acc_bytes(d) * kWarps * d.E * d.d_v; }

template <typename K> static cudaError_t allow(K kern, size_t bytes) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
// the per-CTA maximum of dynamic shared memory next to the kernel's static share
template <auto K> static cudaError_t allow_padded() {
    return allow(K, kSmemPerCta - static_smem_of<K>());
}

// Every gather kernel may use up to the per-CTA maximum of dynamic shared
// memory: a kernel's limit is a process-wide attribute, so it is only ever
// raised (set once to the maximum), never set to one layer's need, which
// would fail a later launch for a larger layer created earlier.
cudaError_t configure_gather(const Dims &) {
    cudaError_t e = allow_padded<gather_kernel<float, double>>();
    if (e == cudaSuccess) e = allow_padded<gather_kernel<float, float>>();
    if (e == cudaSuccess) e = allow_padded<gather_kernel<__nv_bfloat16, float>>();
    if (e == cudaSuccess) e = allow_padded<gather_reg_kernel<float, 1>>();
    if (e == cudaSuccess) e = allow_padded<gather_reg_kernel<float, 4>>();
    if (e == cudaSuccess) e = allow_padded<gather_reg_kernel<__nv_bfloat16, 1>>();
    if (e == cudaSuccess) e = allow_padded<gather_reg_kernel<__nv_bfloat16, 4>>();
    // the bucketed kernels may also be padded up to a whole SM's share (spread_smem)
    if (e == cudaSuccess) e = allow_padded<gather_bucket_kernel<512, false>>();
    if (e == cudaSuccess) e = allow_padded<gather_bucket_kernel<256, false>>();
    if (e == cudaSuccess) e = allow_padded<gather_bucket_kernel<512, true>>();
    if (e == cudaSuccess) e = allow_padded<gather_bucket_kernel<256, true>>();
    if (e == cudaSuccess) e = allow_padded<gather_bucket_exact<512, 1>>();
    if (e == cudaSuccess) e = allow_padded<gather_bucket_exact<256, 1>>();
    if (e == cudaSuccess) e = allow_padded<gather_bucket_exact<512, 2>>();
    if (e == cudaSuccess) e = allow_padded<gather_bucket_exact<256, 2>>();
    if (e == cudaSuccess) e = allow_padded<proj_kernel<float, 2, 2>>();
    if (e == cudaSuccess) e = allow_padded<proj_kernel<float, 1, 1>>();
    if (e == cudaSuccess) e = allow_padded<proj_kernel<__nv_bfloat16, 2, 2>>();
    if (e == cudaSuccess) e = allow_padded<proj_kernel<__nv_bfloat16, 1, 1>>();
    return e;
}

// The bucketed gather, where it serves the layer's shape (*taken).  fp32 rows
// of 33 to 64 vectors (D_v to 256) take two vectors a lane.
template <auto K512, auto K256>
static cudaError_t launch_bucket_k(const Dims &d, const Ptrs &p, bool *taken, cudaStream_t st) {
    *taken = true;
    // spread over the SMs (see spread_smem)
    if (d.B <= 2 * 152 && d.H * d.m <= 512)
        return launch_kernel(d.pdl, K512, d.B, 512,
                             spread_smem(bucket_smem_bytes(d, 16), static_smem_of<K512>(), d.B),
                             st, d, p);
    if (d.H * d.m <= 256 && d.E <= 8)
        return launch_kernel(d.pdl, K256, d.B, 256,
                             spread_smem(bucket_smem_bytes(d, 8), static_smem_of<K256>(), d.B), st,
                             d, p);
    *taken = false;
    return cudaSuccess;
}
template <typename T, bool ADDR>
static cudaError_t launch_bucket(const Dims &d, const Ptrs &p, bool *taken, cudaStream_t st) {
    constexpr int epv = 16 / (int)sizeof(T);
    *taken = false;
    if (d.d_v % epv || d.E > kBMaxE) return cudaSuccess;
    if constexpr (!std::is_same<T, float>::value) {
        // from 305 tokens on (the 512-thread CTAs' limit), blocks to spread over
        if (d.B > 2 * 152 && d.E > 1 && d.nc == 1 && d.H * d.m <= kGSlots &&
            d.d_v / epv <= 32) {
            *taken = true;
            const int64_t warps = (int64_t)d.B * d.E;
            const int grid = (int)((warps + kGWarps - 1) / kGWarps);
            const size_t smem = (size_t)kGWarps * (1024 + 8 * (size_t)d.H * d.m);
            return d.E == 4 ? launch_kernel(d.pdl, gather_warp_kernel<ADDR, true>, grid,
                                            32 * kGWarps, smem, st, d, p)
                            : launch_kernel(d.pdl, gather_warp_kernel<ADDR, false>, grid,
                                            32 * kGWarps, smem, st, d, p);
        }
    }
    if constexpr (std::is_same<T, float>::value) {
        if (d.d_v / epv <= 32)
            return launch_bucket_k<gather_bucket_exact<512, 1>, gather_bucket_exact<256, 1>>(
                d, p, taken, st);
        if (d.d_v / epv <= 64)
            return launch_bucket_k<gather_bucket_exact<512, 2>, gather_bucket_exact<256, 2>>(
                d, p, taken, st);
    } else if (d.d_v / epv <= 32) {
        return launch_bucket_k<gather_bucket_kernel<512, ADDR>, gather_bucket_kernel<256, ADDR>>(
            d, p, taken, st);
    }
    return cudaSuccess;
}

cudaError_t launch_gather_addresses(const Dims &d, const Ptrs &p, bool *taken, cudaStream_t st) {
    *taken = false;
    if (d.dtype != ULTRAMEM_BF16) return cudaSuccess;
    return launch_bucket<__nv_bfloat16, true>(d, p, taken, st);
}

template <typename T>
static cudaError_t launch_gather_t(const Dims &d, const Ptrs &p, cudaStream_t st) {
    const size_t bytes = gather_smem_bytes(d);
    const bool fits_lanes = d.d_v / (16 / (int)sizeof(T)) <= 32;
    bool taken;
    const cudaError_t be = launch_bucket<T, false>(d, p, &taken, st);
    if (taken) return be;
    // the shared-memory-accumulating kernel: fp64 accumulators (fp32 storage)
    // while they fit, else fp32 ones
    auto general = [&]() {
        if (std::is_same<T, float>::value && bytes <= kSmemPerCta)
            return launch_kernel(d.pdl, gather_kernel<T, AccOf<T>>, d.B, kThreads, bytes, st, d,
                                 p);
        return launch_kernel(d.pdl, gather_kernel<T, float>, d.B, kThreads,
                             sizeof(float) * kWarps * d.E * d.d_v, st, d, p);
    };
    if (d.nc > 1)   // MCS beyond the bucketed kernel's range
        return general();
    if (fits_lanes && d.E == 1)
        return launch_kernel(d.pdl, gather_reg_kernel<T, 1>, d.B, kThreads, bytes, st, d, p);
    if (fits_lanes && d.E <= 4)
        return launch_kernel(d.pdl, gather_reg_kernel<T, 4>, d.B, kThreads, bytes, st, d, p);
    return general();
}

cudaError_t launch_gather(const Dims &d, const Ptrs &p, cudaStream_t st) {
    if (d.dtype == ULTRAMEM_BF16) return launch_gather_t<__nv_bfloat16>(d, p, st);
    return launch_gather_t<float>(d, p, st);
}

template <typename T, int TPT, int NP>
static cudaError_t launch_proj_t(const Dims &d, const Ptrs &p, cudaStream_t st) {
    using S = dot::Shape<TPT, NP>;
    // tiles along x, outputs first (2^20 tokens are more tiles than y takes)
    const int64_t tiles = (int64_t)((d.d_out + S::TN - 1) / S::TN) * ((d.B + S::TM - 1) / S::TM);
    if (tiles > 0x7fffffff) return cudaErrorInvalidValue;
    dim3 grid((unsigned)tiles, 1, d.p_splits);
    // a dependent launch is spread over the SMs (see spread_smem)
    constexpr auto k = proj_kernel<T, TPT, NP>;
    const size_t sm = d.pdl ? spread_smem(0, static_smem_of<k>(), ctas_of(grid)) : 0;
    cudaError_t e = launch_kernel(d.pdl, k, grid, dot::kThreads, sm, st, d, p);
    if (e != cudaSuccess) return e;
    const int64_t total = (int64_t)d.B * d.d_out;
    const int64_t blocks = (total + 255) / 256;
    return launch_kernel(d.pdl, proj_reduce_kernel<T>, (unsigned)(blocks < 4096 ? blocks : 4096),
                         256, 0, st, d, p);
}

cudaError_t launch_proj(const Dims &d, const Ptrs &p, cudaStream_t st) {
    const bool small = dot::small_tiles((int64_t)((d.d_out + 63) / 64) * ((d.B + 15) / 16) *
                                        d.p_splits);
    if (d.dtype == ULTRAMEM_BF16)
        return small ? launch_proj_t<__nv_bfloat16, 1, 1>(d, p, st)
                     : launch_proj_t<__nv_bfloat16, 2, 2>(d, p, st);
    return small ? launch_proj_t<float, 1, 1>(d, p, st) : launch_proj_t<float, 2, 2>(d, p, st);
}

}  // namespace um
