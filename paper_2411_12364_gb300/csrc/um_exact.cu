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
//   2. one pass over the grid: a thread holds four columns' S_col in
//      registers, streams the rows (broadcast from shared memory, two rows a
//      packed fp32 instruction) and keeps the largest score of each of 8
//      shares of its pairs, so the grid falls into 4096 groups;
//   3. tau, at most the m-th largest of the group maxima (m distinct groups
//      reach it, so the top m is >= tau); only the groups whose maximum
//      reaches tau (about m of 4096) are scored again, a warp per group, and
//      their scores >= tau, as (key, ~v) composites, go to a list;
//   4. ranks by (score desc, address asc).
// The one full pass is bound by the fp32 pipe: two operations a pair at rank
// 2, 27 us for decode_1m's 64 tokens x 2 heads x 2048^2 pairs at 152 SMs x
// 128 lanes x 2.07 GHz.  Measured there: 9146 us with the radix select below
// for every grid (9 passes over the pairs, a histogram atomic per pair and
// pass, a warp per key in step 1) -> 179 us.
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
// Shared memory is 8 (K r + D_k) bytes plus 9 to 18 KB (K r <= 25600 fits).
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
    int hist[256];        // the radix select's; before it, entry st counts the group
                          // maxima at or above the trial bound of step st
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
__host__ __device__ inline int pad4(int x) { return (x + 3) & ~3; }
inline size_t exact_smem(const Dims &d, int rows, int list) {
    return 8 * (size_t)list + sizeof(float) * ((size_t)d.r * (pad4(rows) + pad4(d.K)) + 2 * d.d_k);
}
// The list's length: as long as fits, at most kListMax, at least kMaxM.
inline int list_len(const Dims &d, int rows) {
    int n = kListMax;
    while (n > kMaxM && exact_smem(d, rows, n) + kStatic > kSmemPerCta) n -= 128;
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
// distinct bin and warp.  Whole block; ends with a barrier.
__device__ __noinline__ void radix_top_m(Grid gd, u64 *list, int i0, int nr, int K, int m,
                                         ExactShared &sh) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t total = (int64_t)nr * K;
    const int64_t iters = (total + kThreads - 1) / kThreads;
    // slot c = it * kThreads + tid, as (i, j) stepped without division
    const int di = kThreads / K, dj = kThreads % K;
    if (threadIdx.x == 0) {
        sh.count = 0;
        sh.prefix = 0;
        sh.need = m;
    }
    __syncthreads();
    // the m-th largest key, 8 bits a pass
    for (int shift = 24; shift >= 0; shift -= 8) {
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
                    const uint32_t v = (uint32_t)(i0 + i) * (uint32_t)K + (uint32_t)j;
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
                v = (uint32_t)(i0 + i) * (uint32_t)K + (uint32_t)j;
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

// RP: the rank rounded up to 1, 2, 4 or 8 (missing chunks are zeros, which
// leave the sums as they are).
template <typename T, int RP, bool PKM>
__global__ void __launch_bounds__(kThreads, 1)
    exact_kernel(Dims d, Ptrs p, int shares, int list_n, int64_t *idx_out, float *w_out) {
    extern __shared__ __align__(16) unsigned char exact_raw[];
    __shared__ ExactShared sh;
    const int pair = blockIdx.x / shares, share = blockIdx.x - pair * shares;
    const int b = pair / d.H, h = pair % d.H;
    const int K = d.K, r = d.r, D = d.d_k, dk = d.dk, m = d.m;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // rows [i0, i0 + nr) of the grid; every share's space is the first one's
    const int per = (K + shares - 1) / shares;
    const int i0 = share * per, nr = min(per, K - i0);
    const int Rp = pad4(per), Sp = pad4(K);
    u64 *list = reinterpret_cast<u64 *>(exact_raw);
    float *core = reinterpret_cast<float *>(list);
    float *R = reinterpret_cast<float *>(list + list_n), *S = R + (size_t)r * Rp,
          *qv = S + (size_t)r * Sp;
    pdl_wait();
    pdl_trigger();

    const int HD = d.H * D;
    const int64_t split_stride = (int64_t)d.A * d.B * HD;
    for (int e = threadIdx.x; e < 2 * D; e += kThreads) {   // summed over the D_i splits
        const int axis = e / D, c = e - axis * D;
        const int a = (axis == 1 && d.A == 2) ? 1 : 0;
        const float *src = p.q_part + ((int64_t)a * d.B + b) * HD + h * D + c;
        float q = 0.f;
        for (int sp = 0; sp < d.q_splits; ++sp) q += src[sp * split_stride];
        qv[e] = q;
    }
    if (threadIdx.x < r * r) core[threadIdx.x] = p.core[(int64_t)h * r * r + threadIdx.x];
    if (threadIdx.x < kBoundBits) sh.hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        sh.count = 0;
        sh.prefix = 0;
        sh.need = m;
        sh.general = 0;
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
    if (dk % 32 == 0) {
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
    // no maximum)
    if (threadIdx.x < 4 * r) {
        const int be = threadIdx.x >> 2, i = nr + (threadIdx.x & 3);
        if (i < pad4(nr)) R[be * Rp + i] = R[be * Rp + nr - 1];
    }
    __syncthreads();

    const Grid gd{R, S, Rp, Sp, r, d.pkm};
    bool general = sh.general != 0;   // uniform
    if (!general) {
        // 2. group maxima.  Column group cg of a block of columns takes 4
        // consecutive ones; when the columns are fewer than the threads
        // hold, `rs_n` threads share a column group and take every rs_n-th
        // quad of rows.  Part q of a thread is the q-th eighth of its quads.
        const int cgs = min(kThreads, (K + kCols - 1) / kCols);
        const int rs_n = kThreads / cgs;
        const int rs = threadIdx.x / cgs, cg = threadIdx.x - rs * cgs;
        const bool busy = rs < rs_n;
        const int quads = pad4(nr) >> 2, mine = busy && quads > rs ? (quads - rs + rs_n - 1) / rs_n : 0;
        float gm[kParts];
#pragma unroll
        for (int q = 0; q < kParts; ++q) gm[q] = -INFINITY;
        for (int j0 = kCols * cg; busy && j0 < K; j0 += kCols * kThreads) {
            // the columns' S, each in both halves; a missing column repeats
            // the thread's first (which changes no maximum)
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
                const int lo = mine * q / kParts, hi = mine * (q + 1) / kParts;
                float mx0 = gm[q], mx1 = -INFINITY;
#pragma unroll 2
                for (int t = lo; t < hi; ++t) {
                    const int i = 4 * (rs + t * rs_n);
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
                        mx0 = fmaxf(mx0, fmaxf(x.x, x.y));
                        mx1 = fmaxf(mx1, fmaxf(y.x, y.y));
                    }
                }
                gm[q] = fmaxf(mx0, mx1);
            }
        }
        // 3. tau: the largest value with zero low bits that m group maxima
        // reach (the leading kBoundBits of the key, from the top)
        uint32_t gk[kParts];
#pragma unroll
        for (int q = 0; q < kParts; ++q)
            gk[q] = mine * (q + 1) / kParts > mine * q / kParts && kCols * cg < K ? f2ord(gm[q])
                                                                                  : 0u;
        uint32_t tau = 0u;
#pragma unroll 1
        for (int st = 0; st < kBoundBits; ++st) {
            const uint32_t c = tau | (0x80000000u >> st);
            int n = 0;
#pragma unroll
            for (int q = 0; q < kParts; ++q) n += gk[q] >= c;
            n = __reduce_add_sync(kFull, n);
            if (lane == 0 && n) atomicAdd(&sh.hist[st], n);
            __syncthreads();
            if (sh.hist[st] >= m) tau = c;
        }
        // the groups that reach tau, a warp each: the pairs >= tau to the
        // list (tau = 0, fewer than m groups: every pair)
#pragma unroll
        for (int q = 0; q < kParts; ++q) {
            unsigned todo = __ballot_sync(kFull, gk[q] != 0u && gk[q] >= tau);
            const int lo = mine * q / kParts, hi = mine * (q + 1) / kParts;
            while (todo) {
                const int src = __ffs(todo) - 1;
                todo &= todo - 1u;
                const int glo = __shfl_sync(kFull, lo, src), ghi = __shfl_sync(kFull, hi, src);
                const int grs = __shfl_sync(kFull, rs, src), gcg = __shfl_sync(kFull, cg, src);
                // an overflow is certain: stop early
                if (__any_sync(kFull, *(volatile int *)&sh.count > list_n)) break;
                for (int e = lane; e < 4 * (ghi - glo); e += 32) {
                    const int i = 4 * (grs + (glo + (e >> 2)) * rs_n) + (e & 3);
                    if (i >= nr) continue;
                    for (int j0 = kCols * gcg; j0 < K; j0 += kCols * kThreads)
                        for (int j = j0; j < min(j0 + kCols, K); ++j) {
                            const uint32_t key = f2ord(gd.score(i, j));
                            if (key >= tau) {
                                const uint32_t v = (uint32_t)(i0 + i) * (uint32_t)K + (uint32_t)j;
                                const int at = atomicAdd(&sh.count, 1);
                                if (at < list_n) list[at] = comp_of(key, v);
                            }
                        }
                }
                __syncwarp();
            }
        }
        __syncthreads();
        general = sh.count > list_n || sh.count < m;   // (fewer: never expected)
        __syncthreads();
    }
    if (general) radix_top_m(gd, list, i0, nr, K, m, sh);
    const int n = min(sh.count, list_n);
    if (sh.count < m && threadIdx.x == 0) atomicOr(p.err, kErrInternal);   // never expected

    // 4. ranks by (key desc, v asc): the number of composites above each
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
    const int list = list_len(d, rows);
    const size_t smem = exact_smem(d, rows, list);
    const int grid = d.B * d.H * shares;
    cudaError_t e = by_rank(d, [&](auto rp, auto pkm) {
        return d.dtype == ULTRAMEM_BF16
                   ? launch_kernel(d.pdl, exact_kernel<__nv_bfloat16, rp(), pkm()>, grid,
                                   kThreads, smem, st, d, p, shares, list, idx_out, w_out)
                   : launch_kernel(d.pdl, exact_kernel<float, rp(), pkm()>, grid, kThreads, smem,
                                   st, d, p, shares, list, idx_out, w_out);
    });
    *launches = shares > 1 ? 2 : 1;
    if (e == cudaSuccess && shares > 1)
        e = launch_kernel(d.pdl, exact_merge_kernel, d.B * d.H, kThreads, 0, st, d, p, shares,
                          idx_out, w_out);
    return e;
}

}  // namespace um
