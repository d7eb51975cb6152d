// um_exact.cu -- Eq. 5 (or Eq. 2 with product keys) by brute force: the
// exact top-m of the whole K x K grid of each (token, head).  It is not on
// the forward path; it measures the recall of the approximate search of
// Eq. 6-10 (which the forward runs) against the exact one.
//
// One CTA of 512 threads per (token, head), or per share of its rows (below):
//   1. the head's chunk scores (Eq. 4) of the CTA's row keys and all column
//      keys, from its query and the key rows, kept in shared memory as
//      R[i] = S_row[:,i]^T C and S_col[:,j] (product keys: s_row[i] and
//      s_col[j]), so that g(i,j) = R[i] . S_col[j] (or the sum) with the
//      forward's own arithmetic;
//   2. rows that cannot hold a winner are dropped: a score is at most
//      |R[i]| |S_col[j]|, so from a bound tau0 <= the m-th largest score, taken
//      by steps 3 and 4 over the 64 or so longest rows alone, every row with
//      |R[i]| max_j |S_col[j]| < tau0 goes (a Gaussian grid of 2048 rows keeps
//      some tens of them);
//   3. one pass over the rows left: a thread holds four columns' S_col in
//      registers, streams the rows (broadcast from shared memory, two rows a
//      packed fp32 instruction) and keeps the largest score of each of 8
//      shares of its pairs, so the grid falls into 4096 groups;
//   4. tau, at most the m-th largest of the group maxima (m distinct groups
//      reach it, so the top m is >= tau); only the groups whose maximum
//      reaches tau are scored again, a warp per group, and their scores >=
//      tau, as (key, ~v) composites, go to a list;
//   5. ranks by (score desc, address asc).
// Measured on GB300, decode_1m's 64 tokens x 2 heads: 9146 us with the radix
// select below for every grid (9 passes over the pairs, a histogram atomic per
// pair and pass), 179 us with steps 3 to 5 over every row (the pass alone is
// 27 us of fp32 work) and a warp per 16 keys in step 1, 84 us now.
//
// When the list overflows (heavy ties) or a chunk score is not finite (its
// score may be a NaN, which the maxima would not see), the CTA takes an
// exact radix select of the m-th largest key over its pairs instead, 8 bits
// a pass, and, when several slots share that key, of the largest address
// among the tied ones that is still taken (ties go to the smaller address).
//
// Fewer (token, head) pairs than half the SMs are split into shares of rows,
// a CTA each, so that about one CTA per SM runs: each leaves the exact top m
// of its share, and a second kernel ranks the shares' winners.
// Shared memory is 8 (K r + D_k) bytes plus 9 to 18 KB (K r <= 25600 fits) and,
// where there is room for it, step 1's stage: 40 KB (bf16) or 72 KB (fp32).
#include "um_internal.cuh"

namespace um {
namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxM = 1024;
constexpr int kMaxR = 8;
constexpr unsigned kFull = 0xffffffffu;

typedef unsigned long long u64;

constexpr int kCols = 4;          // columns a thread holds
constexpr int kParts = 8;         // groups a thread keeps the maximum of
constexpr int kListMax = 2048;    // listed candidates (at least kMaxM)
constexpr int kBoundBits = 20;    // leading key bits that tau is searched in
constexpr int kMaxShares = 16;

struct ExactShared {
    int hist[256];        // the radix select's; before it, the bound searches' counts
    int scan[kWarps];
    uint32_t smax;        // the largest |S_col|^2 (product keys: key of S_col)
    int count;            // listed candidates (may exceed the list)
    uint32_t prefix;      // key bits fixed so far
    int need;             // how many of the remaining keys are still to take
    int ties;             // slots whose key equals the threshold
    uint32_t vcut;        // largest tied address taken
    int general;          // a chunk score that is not finite: radix select
};

constexpr size_t kStatic = (sizeof(ExactShared) + 15) & ~size_t(15);

// Dynamic shared memory: the candidate list (the core in it while the chunk
// scores are computed), R [r][rows] and S_col [r][K] by rank (rows and K
// padded to 16 bytes), the query [2][D_k].
// With room for it, a stage: 32 keys x 32 elements a warp for step 1, then the
// seed rows and the kept rows' numbers of step 2.
__host__ __device__ inline int pad4(int x) { return (x + 3) & ~3; }
constexpr int kSeedRows = 64, kSeedMax = 128;
template <typename T> __host__ __device__ constexpr int stage_pitch() {
    return 32 * (int)sizeof(T) + 16;   // bytes a key: its 16-byte reads miss no bank twice
}
inline size_t stage_bytes_of(const Dims &d, int rows) {
    const size_t keys = (size_t)kWarps * 32 *
                        (d.dtype == ULTRAMEM_F32 ? stage_pitch<float>() : stage_pitch<uint16_t>());
    const size_t prune = 4 * (size_t)kSeedMax * d.r + ((2 * (size_t)rows + 15) & ~size_t(15));
    return keys > prune ? keys : prune;
}
inline size_t exact_smem(const Dims &d, int rows, int list) {
    return 8 * (size_t)list + sizeof(float) * ((size_t)d.r * (pad4(rows) + pad4(d.K)) + 2 * d.d_k);
}
// The list's length: as long as fits, at most kListMax, at least kMaxM.
inline int list_len(const Dims &d, int rows, size_t stage) {
    int n = kListMax;
    while (n > kMaxM && exact_smem(d, rows, n) + stage + kStatic > kSmemPerCta) n -= 128;
    return n;
}
// Shares of rows per (token, head): about one CTA per SM, at most K / m (so
// that a share's row or rows of K pairs hold m, and the shares' m winners fit
// the rank-1 keys' space [2][K]) and at most 1024 winners to merge.
inline int row_shares(const Dims &d) {
    int64_t n = (int64_t)device_sm_count() / ((int64_t)d.B * d.H);
    n = n < kMaxShares ? n : kMaxShares;
    if (n > d.K / d.m) n = d.K / d.m;
    if (n > kMaxM / d.m) n = kMaxM / d.m;
    if (n < 1) n = 1;
    const int per = (int)((d.K + n - 1) / n);
    return (d.K + per - 1) / per;   // none empty
}

template <typename T>
__device__ __forceinline__ float elem(const T *p, int i) { return to_f(p[i]); }

// The grid score of (row i of the CTA's share, column j) from the chunk
// scores in shared memory.
struct Grid {
    const float *R, *S;   // [r][Rp], [r][Sp]
    int Rp, Sp, r, pkm;
    __device__ __forceinline__ float score(int i, int j) const {
        if (pkm) return R[i] + S[j];
        if (r == 2) return fmaf(R[Rp + i], S[Sp + j], R[i] * S[j]);
        float g = 0.f;
        for (int be = 0; be < r; ++be) g = fmaf(R[be * Rp + i], S[be * Sp + j], g);
        return g;
    }
};

// Adds one count for `bin` (0..255; 256 = none) with one atomic per distinct
// bin of the warp.
__device__ __forceinline__ void warp_hist(int *hist, int bin) {
    const unsigned peers = __match_any_sync(kFull, bin);
    const int lane = threadIdx.x & 31;
    if (bin < 256 && lane == __ffs(peers) - 1) atomicAdd(&hist[bin], __popc(peers));
}

// The bin, counted from the top, that holds the need-th largest entry;
// updates need to the rank within that bin.  One warp; returns the bin.
__device__ int pick_bin_from_top(const int *hist, int &need) {
    const int lane = threadIdx.x & 31;
    // lane l owns bins 255 - 8 l .. 248 - 8 l (descending)
    int c[8], s = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        c[q] = hist[255 - 8 * lane - q];
        s += c[q];
    }
    int incl = s;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, off);
        if (lane >= off) incl += y;
    }
    const int excl = incl - s;
    const unsigned hit = __ballot_sync(kFull, excl < need && incl >= need);
    const int owner = __ffs(hit) - 1;
    int bin = 0, above = 0;
    if (lane == owner) {
        int run = excl;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (run + c[q] >= need) {
                bin = 255 - 8 * lane - q;
                above = run;
                break;
            }
            run += c[q];
        }
    }
    bin = __shfl_sync(kFull, bin, owner);
    above = __shfl_sync(kFull, above, owner);
    need -= above;
    return bin;
}

// The same from the bottom (the need-th smallest).
__device__ int pick_bin_from_bottom(const int *hist, int &need) {
    const int lane = threadIdx.x & 31;
    int c[8], s = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        c[q] = hist[8 * lane + q];
        s += c[q];
    }
    int incl = s;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, off);
        if (lane >= off) incl += y;
    }
    const int excl = incl - s;
    const unsigned hit = __ballot_sync(kFull, excl < need && incl >= need);
    const int owner = __ffs(hit) - 1;
    int bin = 0, below = 0;
    if (lane == owner) {
        int run = excl;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (run + c[q] >= need) {
                bin = 8 * lane + q;
                below = run;
                break;
            }
            run += c[q];
        }
    }
    bin = __shfl_sync(kFull, bin, owner);
    below = __shfl_sync(kFull, below, owner);
    need -= below;
    return bin;
}

// The exact top m of the share's pairs into list (sh.count entries: m, or
// fewer than the share holds never) by a radix select of the m-th largest
// key over the scores, recomputed each pass, with one shared atomic per
// distinct bin and warp.  `fixed` leading key bits (0 or 16) are known: no key
// is above those of `prefix`, and m keys share them.  Whole block; ends with a
// barrier.
__device__ __noinline__ void radix_top_m(Grid gd, u64 *list, const uint16_t *map, int i0, int nr,
                                         int K, int m, uint32_t prefix, int fixed,
                                         ExactShared &sh) {
    // the address of (row i, column j); map: the numbers of the rows kept, or null
    auto addr = [&](int i, int j) {
        return (uint32_t)(i0 + (map ? (int)map[i] : i)) * (uint32_t)K + (uint32_t)j;
    };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t total = (int64_t)nr * K;
    const int64_t iters = (total + kThreads - 1) / kThreads;
    // slot c = it * kThreads + tid, as (i, j) stepped without division
    const int di = kThreads / K, dj = kThreads % K;
    if (threadIdx.x == 0) {
        sh.count = 0;
        sh.prefix = prefix;
        sh.need = m;
    }
    __syncthreads();
    // the m-th largest key, 8 bits a pass
    for (int shift = 24 - fixed; shift >= 0; shift -= 8) {
        for (int e = threadIdx.x; e < 256; e += kThreads) sh.hist[e] = 0;
        __syncthreads();
        const uint32_t pre = sh.prefix;
        const uint32_t hi_mask = shift == 24 ? 0u : ~0u << (shift + 8);
        int i = threadIdx.x / K, j = threadIdx.x % K;
        for (int64_t it = 0; it < iters; ++it) {
            int bin = 256;
            if (i < nr) {
                const uint32_t key = f2ord(gd.score(i, j));
                if ((key & hi_mask) == (pre & hi_mask)) bin = (key >> shift) & 255;
            }
            warp_hist(sh.hist, bin);
            i += di;
            j += dj;
            if (j >= K) { j -= K; ++i; }
        }
        __syncthreads();
        if (warp == 0) {
            int need = sh.need;
            const int bin = pick_bin_from_top(sh.hist, need);
            if (lane == 0) {
                sh.prefix = pre | ((uint32_t)bin << shift);
                sh.need = need;
                sh.ties = sh.hist[bin];
            }
        }
        __syncthreads();
    }
    const uint32_t thr = sh.prefix;   // the m-th largest key
    // ties at the threshold: the need-th smallest address among them
    uint32_t vcut = ~0u;
    if (sh.ties > sh.need) {
        if (threadIdx.x == 0) sh.vcut = 0;
        for (int shift = 24; shift >= 0; shift -= 8) {
            for (int e = threadIdx.x; e < 256; e += kThreads) sh.hist[e] = 0;
            __syncthreads();
            const uint32_t pre = sh.vcut;
            const uint32_t hi_mask = shift == 24 ? 0u : ~0u << (shift + 8);
            int i = threadIdx.x / K, j = threadIdx.x % K;
            for (int64_t it = 0; it < iters; ++it) {
                int bin = 256;
                if (i < nr && f2ord(gd.score(i, j)) == thr) {
                    const uint32_t v = addr(i, j);
                    if ((v & hi_mask) == (pre & hi_mask)) bin = (v >> shift) & 255;
                }
                warp_hist(sh.hist, bin);
                i += di;
                j += dj;
                if (j >= K) { j -= K; ++i; }
            }
            __syncthreads();
            if (warp == 0) {
                int need = sh.need;
                const int bin = pick_bin_from_bottom(sh.hist, need);
                if (lane == 0) {
                    sh.vcut = pre | ((uint32_t)bin << shift);
                    sh.need = need;
                }
            }
            __syncthreads();
        }
        vcut = sh.vcut;
    }

    // the winners: keys above the threshold, and the tied ones up to vcut
    {
        int i = threadIdx.x / K, j = threadIdx.x % K;
        for (int64_t it = 0; it < iters; ++it) {
            bool take = false;
            uint32_t key = 0, v = 0;
            if (i < nr) {
                key = f2ord(gd.score(i, j));
                v = addr(i, j);
                take = key > thr || (key == thr && v <= vcut);
            }
            const unsigned bal = __ballot_sync(kFull, take);
            if (bal) {
                int base = 0;
                if (lane == 0) base = atomicAdd(&sh.count, __popc(bal));
                base = __shfl_sync(kFull, base, 0);
                const int pos = base + __popc(bal & ((1u << lane) - 1u));
                if (take && pos < m) list[pos] = comp_of(key, v);
            }
            i += di;
            j += dj;
            if (j >= K) { j -= K; ++i; }
        }
    }
    __syncthreads();
}

// The chunk scores of `n` keys (rows of D values at `rows`) against q, a warp
// per 32 / RP keys: lane l sums the products of the elements l, l + 32, ...
// of each rank chunk, and the 32 lanes' sums of the warp's 32 (key, chunk)
// values are added by recursive halving (31 shuffles; the tree of a value is
// that of a butterfly over the lanes), which leaves value l in lane l.  Then
// put(key, lane's chunk, its sum v, the first lane of the key's chunks).
// dk % 32 == 0.  The key rows are read once per (token, head), 2-byte loads:
// 4 requests a key at D_k = 128.
template <typename T, int RP, class Put>
__device__ __forceinline__ void chunk_scores(const T *rows, int n, const float *q, int D, int dk,
                                             int r, Put put) {
    constexpr int KB = 32 / RP;   // keys a warp takes at once
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int k0 = warp * KB; k0 < n; k0 += kWarps * KB) {
        float v[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] = 0.f;
#pragma unroll
        for (int al = 0; al < RP; ++al) {
            if (al < r) {
                for (int c = al * dk + lane; c < (al + 1) * dk; c += 32) {
                    const float qc = q[c];
                    float x[KB];
#pragma unroll
                    for (int kk = 0; kk < KB; ++kk)
                        x[kk] = elem(rows + (int64_t)min(k0 + kk, n - 1) * D, c);
#pragma unroll
                    for (int kk = 0; kk < KB; ++kk)
                        v[kk * RP + al] = __fadd_rn(v[kk * RP + al], __fmul_rn(x[kk], qc));
                }
            }
        }
#pragma unroll
        for (int half = 16; half > 0; half >>= 1) {
            const bool up = (lane & half) != 0;
#pragma unroll
            for (int e = 0; e < half; ++e) {
                const float keep = up ? v[e + half] : v[e], send = up ? v[e] : v[e + half];
                v[e] = __fadd_rn(keep, __shfl_xor_sync(kFull, send, half));
            }
        }
        put(k0 + lane / RP, lane % RP, v[0], lane - lane % RP);
    }
}

// The chunk scores of `n` keys against q, a lane per key: a warp's 32 rows come
// in 32 elements at a time through its stage (16-byte loads of whole sectors,
// the next ones on their way meanwhile), and a lane adds up its key's
// products by the same tree as chunk_scores' 32 lanes: 32 partial sums over
// the elements l, l + 32, ... of a chunk, packed in pairs, then halves.
// put(key, s): the lane's chunk sums.  dk % 32 == 0, rows 16-byte aligned.
template <typename T, int RP, class Put>
__device__ __forceinline__ void chunk_scores_staged(const T *rows, int n, const float *q, int D,
                                                    int dk, int r, unsigned char *stage, Put put) {
    constexpr int VB = 32 * (int)sizeof(T) / 16, PITCH = stage_pitch<T>();
    constexpr int EPV = 16 / (int)sizeof(T);
    constexpr f2 kMinus1 = 0xbf800000bf800000ull;   // (-1, -1)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *mine = stage + warp * 32 * PITCH;
    const int steps = D / 32;
    for (int k0 = warp * 32; k0 < n; k0 += kWarps * 32) {
        uint4 buf[VB];
        auto fetch = [&](int st) {
#pragma unroll
            for (int i = 0; i < VB; ++i) {
                const int e = i * 32 + lane, key = min(k0 + e / VB, n - 1);
                buf[i] = *reinterpret_cast<const uint4 *>(rows + (int64_t)key * D + 32 * st +
                                                          e % VB * EPV);
            }
        };
        float s[RP];
#pragma unroll
        for (int a = 0; a < RP; ++a) s[a] = 0.f;
        f2 v[16];
        int al = 0, left = dk / 32;   // the chunk, and its steps to go
        fetch(0);
#pragma unroll 1
        for (int st = 0; st < steps; ++st) {
            __syncwarp();   // the previous elements have been read
#pragma unroll
            for (int i = 0; i < VB; ++i) {
                const int e = i * 32 + lane;
                *reinterpret_cast<uint4 *>(mine + e / VB * PITCH + e % VB * 16) = buf[i];
            }
            __syncwarp();
            if (st + 1 < steps) fetch(st + 1);
            if (left == dk / 32)   // uniform: a chunk starts
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = 0ull;
#pragma unroll
            for (int i = 0; i < VB; ++i) {
                const uint4 x = *reinterpret_cast<const uint4 *>(mine + lane * PITCH + i * 16);
                const ulonglong2 *qq =
                    reinterpret_cast<const ulonglong2 *>(q + 32 * st + i * EPV);
                const uint32_t w[4] = {x.x, x.y, x.z, x.w};
                f2 xe[EPV / 2];
#pragma unroll
                for (int c = 0; c < EPV / 2; ++c) {
                    if constexpr (sizeof(T) == 2)
                        xe[c] = pack2(__uint_as_float(w[c] << 16),
                                      __uint_as_float(w[c] & 0xffff0000u));
                    else
                        xe[c] = pack2(__uint_as_float(w[2 * c]), __uint_as_float(w[2 * c + 1]));
                }
#pragma unroll
                for (int c = 0; c < EPV / 2; c += 2) {
                    const ulonglong2 q2 = qq[c / 2];
                    const int at = i * (EPV / 2) + c;
                    // v holds the negated sums: a product of -1 keeps the
                    // compiler from fusing the product into the sum
                    v[at] = fma2(mul2(xe[c], q2.x), kMinus1, v[at]);
                    v[at + 1] = fma2(mul2(xe[c + 1], q2.y), kMinus1, v[at + 1]);
                }
            }
            if (--left == 0) {
#pragma unroll
                for (int half = 8; half > 0; half >>= 1)
#pragma unroll
                    for (int j = 0; j < half; ++j) v[j] = add2(v[j], v[j + half]);
                const float2 x = unpack2(v[0]);
                const float sum = -__fadd_rn(x.x, x.y);
#pragma unroll
                for (int a = 0; a < RP; ++a)
                    if (a == al) s[a] = sum;
                ++al;
                left = dk / 32;
            }
        }
        if (k0 + lane < n) put(k0 + lane, s);
    }
}

// The largest value with zero low bits (`bits` leading ones of 32 decided)
// that at least `need` of the block's keys reach; each(f) calls f(key) for the
// thread's keys.  cnt: `bits` counters, zero.  Whole block.
template <class Each>
__device__ __forceinline__ uint32_t block_bound(int need, int bits, int *cnt, Each each) {
    uint32_t T = 0u;
#pragma unroll 1
    for (int st = 0; st < bits; ++st) {
        const uint32_t c = T | (0x80000000u >> st);
        int n = 0;
        each([&](uint32_t key) { n += key >= c; });
        n = __reduce_add_sync(kFull, n);
        if ((threadIdx.x & 31) == 0 && n) atomicAdd(&cnt[st], n);
        __syncthreads();
        if (cnt[st] >= need) T = c;
    }
    return T;
}

// Exclusive prefix sum of one int per thread over the block, and the total.
__device__ __forceinline__ int block_scan(int v, ExactShared &sh, int *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, off);
        if (lane >= off) incl += y;
    }
    __syncthreads();   // the previous scan's sums have been read
    if (lane == 31) sh.scan[warp] = incl;
    __syncthreads();
    int before = 0, all = 0;
    for (int w = 0; w < kWarps; ++w) {
        const int x = sh.scan[w];
        before += w < warp ? x : 0;
        all += x;
    }
    *total = all;
    return before + incl - v;
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float m;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(a), "f"(b), "f"(c));
    return m;
}

// A thread's part of a pass: column group cg of a block of columns takes kCols
// consecutive ones; when the columns are fewer than the threads hold, rs_n
// threads share a column group and take every rs_n-th quad of rows.  Part q
// of a thread is the q-th eighth of its `mine` quads.
struct PassShape {
    int rs_n, rs, cg, mine;
    bool busy;
    __device__ __forceinline__ PassShape(int nr, int K) {
        const int cgs = min(kThreads, (K + kCols - 1) / kCols);
        rs_n = kThreads / cgs;
        rs = threadIdx.x / cgs;
        cg = threadIdx.x - rs * cgs;
        busy = rs < rs_n;
        const int quads = pad4(nr) >> 2;
        mine = busy && quads > rs ? (quads - rs + rs_n - 1) / rs_n : 0;
    }
    __device__ __forceinline__ int lo(int q) const { return mine * q / kParts; }
};

// The largest score of each of the thread's parts, as keys (0: an empty part),
// over the rows R [r][Rp] (the last quad padded by repeats) and all columns.
template <int RP, bool PKM>
__device__ __forceinline__ void group_maxima(const float *R, int Rp, const float *S, int Sp, int r,
                                             int K, const PassShape &ps, uint32_t (&gk)[kParts]) {
    float gm[kParts];
#pragma unroll
    for (int q = 0; q < kParts; ++q) gm[q] = -INFINITY;
    for (int j0 = kCols * ps.cg; ps.busy && j0 < K; j0 += kCols * kThreads) {
        // the columns' S, each in both halves; a missing column repeats the
        // thread's first (which changes no maximum)
        f2 sc[RP][kCols];
#pragma unroll
        for (int be = 0; be < RP; ++be)
#pragma unroll
            for (int c = 0; c < kCols; ++c) {
                const float v = be < r ? S[be * Sp + (j0 + c < K ? j0 + c : j0)] : 0.f;
                sc[be][c] = pack2(v, v);
            }
#pragma unroll
        for (int q = 0; q < kParts; ++q) {
            const int hi = ps.lo(q + 1);
            float mx0 = gm[q], mx1 = -INFINITY;
#pragma unroll 2
            for (int t = ps.lo(q); t < hi; ++t) {
                const int i = 4 * (ps.rs + t * ps.rs_n);
                f2 ra[RP][2];   // rows i, i + 1 and i + 2, i + 3
#pragma unroll
                for (int be = 0; be < RP; ++be) {
                    ulonglong2 v = make_ulonglong2(0ull, 0ull);
                    if (be < r) v = *reinterpret_cast<const ulonglong2 *>(R + be * Rp + i);
                    ra[be][0] = v.x;
                    ra[be][1] = v.y;
                }
#pragma unroll
                for (int c = 0; c < kCols; ++c) {
                    f2 g[2];
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        if (PKM) {
                            g[u] = add2(ra[0][u], sc[0][c]);
                        } else {
                            g[u] = mul2(ra[0][u], sc[0][c]);
#pragma unroll
                            for (int be = 1; be < RP; ++be)
                                g[u] = fma2(ra[be][u], sc[be][c], g[u]);
                        }
                    }
                    const float2 x = unpack2(g[0]), y = unpack2(g[1]);
                    mx0 = max3(mx0, x.x, x.y);
                    mx1 = max3(mx1, y.x, y.y);
                }
            }
            gm[q] = fmaxf(mx0, mx1);
        }
    }
#pragma unroll
    for (int q = 0; q < kParts; ++q)
        gk[q] = ps.lo(q + 1) > ps.lo(q) && kCols * ps.cg < K ? f2ord(gm[q]) : 0u;
}

// RP: the rank rounded up to 1, 2, 4 or 8 (missing chunks are zeros, which
// leave the sums as they are).
template <typename T, int RP, bool PKM>
__global__ void __launch_bounds__(kThreads, 1)
    exact_kernel(Dims d, Ptrs p, int shares, int list_n, int staged, int64_t *idx_out,
                 float *w_out) {
    extern __shared__ __align__(16) unsigned char exact_raw[];
    __shared__ ExactShared sh;
    const int pair = blockIdx.x / shares, share = blockIdx.x - pair * shares;
    const int b = pair / d.H, h = pair % d.H;
    const int K = d.K, r = d.r, D = d.d_k, dk = d.dk, m = d.m;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // rows [i0, i0 + nr) of the grid; every share's space is the first one's
    const int per = (K + shares - 1) / shares;
    const int i0 = share * per;
    int nr = min(per, K - i0);
    const int Rp = pad4(per), Sp = pad4(K);
    u64 *list = reinterpret_cast<u64 *>(exact_raw);
    float *core = reinterpret_cast<float *>(list);
    float *R = reinterpret_cast<float *>(list + list_n), *S = R + (size_t)r * Rp,
          *qv = S + (size_t)r * Sp;
    unsigned char *stage = reinterpret_cast<unsigned char *>(qv + 2 * pad4(D));
    pdl_wait();
    pdl_trigger();

    const int HD = d.H * D;
    for (int e = threadIdx.x; e < 2 * D; e += kThreads) {
        const int axis = e / D, c = e - axis * D;
        const int a = (axis == 1 && d.A == 2) ? 1 : 0;
        qv[e] = p.q_part[((int64_t)a * d.B + b) * HD + h * D + c];
    }
    if (threadIdx.x < r * r) core[threadIdx.x] = p.core[(int64_t)h * r * r + threadIdx.x];
    if (threadIdx.x < 256) sh.hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        sh.count = 0;
        sh.prefix = 0;
        sh.need = m;
        sh.general = 0;
        sh.smax = 0u;
    }
    __syncthreads();

    // 1. chunk scores (Eq. 4): R = S_row^T C of the share's rows, S_col
    const T *krow = static_cast<const T *>(p.k_row) + ((int64_t)h * K + i0) * D;
    const T *kcol = static_cast<const T *>(p.k_col) + (int64_t)h * K * D;
    bool odd = false;   // a chunk score that is not finite
    auto put_r = [&](int i, int be, float acc) {
        if (i < nr && be < r) R[be * Rp + i] = acc;
        if (i < nr && be < r && !(fabsf(acc) < INFINITY)) odd = true;
    };
    auto put_s = [&](int j, int be, float v) {
        if (j < K && be < r) S[be * Sp + j] = v;
        if (j < K && be < r && !(fabsf(v) < INFINITY)) odd = true;
    };
    if (staged && dk % 32 == 0) {
        chunk_scores_staged<T, RP>(krow, nr, qv, D, dk, r, stage, [&](int i, const float (&v)[RP]) {
#pragma unroll
            for (int be = 0; be < RP; ++be) {
                float acc = 0.f;
#pragma unroll
                for (int a = 0; a < RP; ++a)
                    if (a < r && be < r) acc = fmaf(v[a], core[a * r + be], acc);
                put_r(i, be, acc);
            }
        });
        chunk_scores_staged<T, RP>(kcol, K, qv + D, D, dk, r, stage,
                                   [&](int j, const float (&v)[RP]) {
#pragma unroll
                                       for (int be = 0; be < RP; ++be) put_s(j, be, v[be]);
                                   });
    } else if (dk % 32 == 0) {
        chunk_scores<T, RP>(krow, nr, qv, D, dk, r, [&](int i, int be, float v, int l0) {
            float acc = 0.f;
#pragma unroll
            for (int a = 0; a < RP; ++a) {
                const float sa = __shfl_sync(kFull, v, l0 + a);
                if (a < r) acc = fmaf(sa, be < r ? core[a * r + be] : 0.f, acc);
            }
            put_r(i, be, acc);
        });
        chunk_scores<T, RP>(kcol, K, qv + D, D, dk, r,
                            [&](int j, int be, float v, int) { put_s(j, be, v); });
    } else {
        for (int key = warp; key < nr + K; key += kWarps) {   // a warp per key
            const int axis = key >= nr, i = axis ? key - nr : key;
            const T *row = (axis ? kcol : krow) + (int64_t)i * D;
            const float *q = qv + axis * D;
            float s[kMaxR];
#pragma unroll
            for (int a = 0; a < kMaxR; ++a) s[a] = 0.f;
            for (int c = lane; c < D; c += 32) {
                const float pr = elem(row, c) * q[c];
                const int al = c / dk;
#pragma unroll
                for (int a = 0; a < kMaxR; ++a) s[a] += a == al ? pr : 0.f;
            }
#pragma unroll
            for (int a = 0; a < kMaxR; ++a) {
                if (a < r)
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1)
                        s[a] += __shfl_xor_sync(kFull, s[a], off);
            }
            if (lane == 0) {
                for (int be = 0; be < r; ++be) {
                    if (axis == 0) {   // R = S_row^T C
                        float acc = 0.f;
                        for (int a = 0; a < r; ++a) acc = fmaf(s[a], core[a * r + be], acc);
                        put_r(i, be, acc);
                    } else {
                        put_s(i, be, s[be]);
                    }
                }
            }
        }
    }
    if (odd) sh.general = 1;
    __syncthreads();
    // the rows padding the last quad repeat the last row (their scores change
    // no maximum); ends with a barrier
    auto pad_rows = [&](float *rows, int pitch, int n) {
        if (threadIdx.x < 4 * r) {
            const int be = threadIdx.x >> 2, i = n + (threadIdx.x & 3);
            if (i < pad4(n)) rows[be * pitch + i] = rows[be * pitch + n - 1];
        }
        __syncthreads();
    };
    pad_rows(R, Rp, nr);

    bool general = sh.general != 0;   // uniform
    const uint16_t *map = nullptr;    // the kept rows' numbers
    if (!general && staged && nr >= 4 * kSeedMax) {
        // 2. |R[i]|^2 (product keys: R[i]) as a key; pads keep underflowed
        // squares from pruning
        constexpr float kPad = 1e-36f;
        auto row_key = [&](int i) {
            if (PKM) return f2ord(R[i]);
            float n2 = kPad;
            for (int be = 0; be < r; ++be) n2 = fmaf(R[be * Rp + i], R[be * Rp + i], n2);
            return f2ord(n2);
        };
        auto my_rows = [&](auto f) {
            for (int i = threadIdx.x; i < nr; i += kThreads) f(row_key(i));
        };
        uint32_t sm = 0u;
        for (int j = threadIdx.x; j < K; j += kThreads) {
            float n2 = kPad;
            if (!PKM)
                for (int be = 0; be < r; ++be) n2 = fmaf(S[be * Sp + j], S[be * Sp + j], n2);
            sm = max(sm, f2ord(PKM ? S[j] : n2));
        }
        sm = __reduce_max_sync(kFull, sm);
        if (lane == 0) atomicMax(&sh.smax, sm);
        const uint32_t long_row = block_bound(kSeedRows, 16, sh.hist + 32, my_rows);
        // the seeds: the first kSeedMax rows that reach it
        float *seed = reinterpret_cast<float *>(stage);   // [r][kSeedMax]
        int got = 0;
        for (int i = threadIdx.x; i < nr; i += kThreads) got += row_key(i) >= long_row;
        int seeds;
        int at = block_scan(got, sh, &seeds);
        for (int i = threadIdx.x; i < nr; i += kThreads)
            if (row_key(i) >= long_row) {
                if (at < kSeedMax)
                    for (int be = 0; be < r; ++be) seed[be * kSeedMax + at] = R[be * Rp + i];
                ++at;
            }
        seeds = min(seeds, kSeedMax);
        __syncthreads();
        pad_rows(seed, kSeedMax, seeds);
        const PassShape ps(seeds, K);
        uint32_t gk[kParts];
        group_maxima<RP, PKM>(seed, kSeedMax, S, Sp, r, K, ps, gk);
        const uint32_t tau0 = block_bound(m, kBoundBits, sh.hist + 64, [&](auto f) {
#pragma unroll
            for (int q = 0; q < kParts; ++q) f(gk[q]);
        });
        const float t0 = ord2f(tau0), smax = ord2f(sh.smax);
        // (tau0 = 0: fewer than m groups.)  The scores' rounding, at most a few
        // ulps of |R| |S|, is far inside the margin 2^-12.
        if (tau0 != 0u && (PKM || (t0 > 1e-12f && t0 < 1e18f))) {
            auto keep = [&](int i) {
                const uint32_t key = row_key(i);
                if (PKM) return f2ord(ord2f(key) + smax) >= tau0;
                return !(ord2f(key) * smax * (1.f + 1.f / 4096.f) < t0 * t0);
            };
            const int per_t = (nr + kThreads - 1) / kThreads;
            const int lo = min(nr, (int)threadIdx.x * per_t), hi = min(nr, lo + per_t);
            int mine = 0, kept;
            for (int i = lo; i < hi; ++i) mine += keep(i);
            int to = block_scan(mine, sh, &kept);
            uint16_t *rows = reinterpret_cast<uint16_t *>(stage + 4 * kSeedMax * r);
            for (int i = lo; i < hi; ++i)
                if (keep(i)) rows[to++] = (uint16_t)i;
            __syncthreads();
            // rows[i] >= i: whole batches move down without overwriting a later one
            for (int base = 0; base < kept; base += kThreads) {
                const int i = base + threadIdx.x;
                float v[RP];
#pragma unroll
                for (int be = 0; be < RP; ++be)
                    if (i < kept && be < r) v[be] = R[be * Rp + rows[i]];
                __syncthreads();
#pragma unroll
                for (int be = 0; be < RP; ++be)
                    if (i < kept && be < r) R[be * Rp + i] = v[be];
                __syncthreads();
            }
            map = rows;
            nr = kept;   // at least one: the rows that reach tau0
            pad_rows(R, Rp, nr);
        }
    }
    const Grid gd{R, S, Rp, Sp, r, d.pkm};
    uint32_t prefix = 0u;   // see radix_top_m
    int fixed = 0;
    if (!general) {
        // 3. group maxima, and tau
        const PassShape ps(nr, K);
        uint32_t gk[kParts];
        group_maxima<RP, PKM>(R, Rp, S, Sp, r, K, ps, gk);
        const uint32_t tau = block_bound(m, kBoundBits, sh.hist, [&](auto f) {
#pragma unroll
            for (int q = 0; q < kParts; ++q) f(gk[q]);
        });
        // 4. the groups that reach tau, a warp each: the pairs >= tau to the
        // list (tau = 0, fewer than m groups: every pair)
#pragma unroll
        for (int q = 0; q < kParts; ++q) {
            unsigned todo = __ballot_sync(kFull, gk[q] != 0u && gk[q] >= tau);
            const int lo = ps.lo(q), hi = ps.lo(q + 1);
            while (todo) {
                const int src = __ffs(todo) - 1;
                todo &= todo - 1u;
                const int glo = __shfl_sync(kFull, lo, src), ghi = __shfl_sync(kFull, hi, src);
                const int grs = __shfl_sync(kFull, ps.rs, src);
                const int gcg = __shfl_sync(kFull, ps.cg, src);
                // an overflow is certain: stop early
                if (__any_sync(kFull, *(volatile int *)&sh.count > list_n)) break;
                for (int e = lane; e < 4 * (ghi - glo); e += 32) {
                    const int i = 4 * (grs + (glo + (e >> 2)) * ps.rs_n) + (e & 3);
                    if (i >= nr) continue;
                    const uint32_t row = (uint32_t)(i0 + (map ? (int)map[i] : i)) * (uint32_t)K;
                    for (int j0 = kCols * gcg; j0 < K; j0 += kCols * kThreads)
                        for (int j = j0; j < min(j0 + kCols, K); ++j) {
                            const uint32_t key = f2ord(gd.score(i, j));
                            if (key >= tau) {
                                const int at = atomicAdd(&sh.count, 1);
                                if (at < list_n) list[at] = comp_of(key, row + (uint32_t)j);
                            }
                        }
                }
                __syncwarp();
            }
        }
        __syncthreads();
        general = sh.count > list_n || sh.count < m;   // (fewer: never expected)
        // tied scores: when no group's maximum is above tau in its leading 16
        // bits, those are the m-th largest key's as well
        bool above = tau == 0u;
#pragma unroll
        for (int q = 0; q < kParts; ++q) above = above || gk[q] >> 16 > tau >> 16;
        if (!__syncthreads_or(above)) {
            prefix = tau & 0xffff0000u;
            fixed = 16;
        }
    }
    if (general) radix_top_m(gd, list, map, i0, nr, K, m, prefix, fixed, sh);
    const int n = min(sh.count, list_n);
    if (sh.count < m && threadIdx.x == 0) atomicOr(p.err, kErrInternal);   // never expected

    // 5. ranks by (key desc, v asc): the number of composites above each
    const int64_t base = (int64_t)pair * m;
    u64 *part = reinterpret_cast<u64 *>(p.akey) + ((int64_t)pair * shares + share) * m;
    for (int e = threadIdx.x; e < n; e += kThreads) {
        const u64 x = list[e];
        int rank = 0;
        for (int f = 0; f < n; ++f) rank += list[f] > x;
        if (rank >= m) continue;
        if (shares > 1) {
            part[rank] = x;
        } else {
            idx_out[base + rank] = (int64_t)pos_of(x);
            if (w_out) w_out[base + rank] = ord2f(key_of(x));
        }
    }
}

// The top m of the shares' winners ([shares * m] composites, distinct) of
// one (token, head) per CTA.
__global__ void __launch_bounds__(kThreads) exact_merge_kernel(Dims d, Ptrs p, int shares,
                                                               int64_t *idx_out, float *w_out) {
    __shared__ u64 c[kMaxM];
    pdl_wait();
    pdl_trigger();
    const int n = shares * d.m;   // <= kMaxM
    const u64 *part = reinterpret_cast<const u64 *>(p.akey) + (int64_t)blockIdx.x * n;
    for (int e = threadIdx.x; e < n; e += kThreads) c[e] = part[e];
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * d.m;
    for (int e = threadIdx.x; e < n; e += kThreads) {
        const u64 x = c[e];
        int rank = 0;
        for (int f = 0; f < n; ++f) rank += c[f] > x;
        if (rank >= d.m) continue;
        idx_out[base + rank] = (int64_t)pos_of(x);
        if (w_out) w_out[base + rank] = ord2f(key_of(x));
    }
}

}  // namespace

bool exact_fits(const Dims &d) {
    return d.m <= kMaxM && d.r <= kMaxR &&
           exact_smem(d, d.K, kMaxM) + kStatic <= kSmemPerCta;
}

// kernel(std::integral_constant RP, PKM) for the layer's rank
template <class F> static cudaError_t by_rank(const Dims &d, F f) {
    if (d.pkm) return f(std::integral_constant<int, 1>(), std::true_type());
    if (d.r == 1) return f(std::integral_constant<int, 1>(), std::false_type());
    if (d.r == 2) return f(std::integral_constant<int, 2>(), std::false_type());
    if (d.r <= 4) return f(std::integral_constant<int, 4>(), std::false_type());
    return f(std::integral_constant<int, 8>(), std::false_type());
}

// The limit of dynamic shared memory is a process-wide attribute of the
// kernel: it is set to the maximum, never to one layer's need.
cudaError_t configure_exact(const Dims &d) {
    return by_rank(d, [](auto rp, auto pkm) {
        const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
        constexpr auto kf = exact_kernel<float, rp(), pkm()>;
        constexpr auto kb = exact_kernel<__nv_bfloat16, rp(), pkm()>;
        cudaError_t e = cudaFuncSetAttribute(kf, a, (int)(kSmemPerCta - static_smem_of<kf>()));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kb, a, (int)(kSmemPerCta - static_smem_of<kb>()));
        return e;
    });
}

cudaError_t launch_exact(const Dims &d, const Ptrs &p, int64_t *idx_out, float *w_out,
                         int *launches, cudaStream_t st) {
    const int shares = row_shares(d), rows = (d.K + shares - 1) / shares;
    // a stage where it fits beside a list of kMaxM, and the key rows allow
    // 16-byte reads (dk % 32 == 0 makes their length do)
    const size_t stage = stage_bytes_of(d, rows);
    const int staged = d.dk % 32 == 0 && rows <= 65536 &&
                       (((uintptr_t)p.k_row | (uintptr_t)p.k_col) & 15) == 0 &&
                       exact_smem(d, rows, kMaxM) + stage + kStatic <= kSmemPerCta;
    const int list = list_len(d, rows, staged ? stage : 0);
    const size_t smem = exact_smem(d, rows, list) + (staged ? stage : 0);
    const int grid = d.B * d.H * shares;
    cudaError_t e = by_rank(d, [&](auto rp, auto pkm) {
        return d.dtype == ULTRAMEM_BF16
                   ? launch_kernel(d.pdl, exact_kernel<__nv_bfloat16, rp(), pkm()>, grid,
                                   kThreads, smem, st, d, p, shares, list, staged, idx_out, w_out)
                   : launch_kernel(d.pdl, exact_kernel<float, rp(), pkm()>, grid, kThreads, smem,
                                   st, d, p, shares, list, staged, idx_out, w_out);
    });
    *launches = shares > 1 ? 2 : 1;
    if (e == cudaSuccess && shares > 1)
        e = launch_kernel(d.pdl, exact_merge_kernel, d.B * d.H, kThreads, 0, st, d, p, shares,
                          idx_out, w_out);
    return e;
}

}  // namespace um
