// um_select.cu -- S4..S7 for one (token, head) per CTA (on long grids one per
// warp, select_warp_kernel below, with the same results):
//   top-k of each axis on the rank-1 score keys         (Eq. 8-9)
//   exact chunk scores S_alpha of the 2k survivors      (Eq. 4)
//   exact Tucker score g on the k*k survivor pairs      (Eq. 10; with product
//                                                         keys s_row + s_col, Eq. 2)
//   top-m of g, ordered by (score desc, v asc)          (Eq. 10)
//   weights (raw scores, or PKM's softmax), shuffle     (Trick 1, Eq. 3, Eq. 14)
//   with h component cores (MCS), the h individual scores of each winner
//                                                        (Eq. 16-17)
// No K*K grid is ever formed.  The scoring kernel leaves, per key, the
// order-preserving 32-bit key of its fp32 rank-1 score; the exact chunk
// scores of the k survivors of each axis are recomputed here from q and the
// key rows.  Ties go to the smaller index.
//
// Top-k of n keys in a CTA, in two stages.  Candidates: each thread keeps the two
// largest of its share of the keys; each warp takes the j-th largest of its
// lanes' 64 values (j = ceil(k / 8): j rounds of a warp max that removes one
// instance) and tau is the smallest of the 8 warp values.  Every warp owns at
// least j keys >= tau, so at least k keys are >= tau whatever the input:
// every key of the top k is >= tau.  The keys >= tau are appended to one
// flat list per selection (a hit mask per lane, a warp scan, one shared
// atomic per warp).  When the list is long the same bound is taken again over
// it; when it overflows (heavy ties) an exact radix select replaces it.
// Order: the candidates are 64-bit composites (key, ~position) whose
// descending order is key descending then position ascending; the rank of
// each is the number of candidates above it (counted by a group of lanes per
// candidate, or by binary searches in sorted warp runs on long grids), and the
// ones ranked below k are the winners, in rank order.
#include "um_internal.cuh"

namespace um {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kCap = 1024;                 // candidates per selection
constexpr int kPerThread = kCap / kThreads;
constexpr int kMaxK = 128;
constexpr int kMaxM = 1024;
static_assert(kMaxM <= kCap, "the final winners reuse a candidate list");
constexpr int kMaxR = 8;
constexpr int kRankSort = 256;             // longer lists are tightened first
constexpr uint32_t kPairMix = 421;         // prime > kMaxK: the order of the Tucker pairs
static_assert(kWarps == 8, "the Tucker pairs' assignment spreads rows over 8 warps");
static_assert(kPairMix > kMaxK, "kPairMix must be coprime with every k^2");
// value rows of a batch beyond this are not prefetched into L2 by the
// selection: they would be evicted before the gather reads them
constexpr uint64_t kPrefetchMaxBytes = 64ull << 20;
constexpr unsigned kFull = 0xffffffffu;

// counter slots of SelShared::cnt
constexpr int kCntAxis = 0;      // +s: first pass of axis s
constexpr int kCntAxisT = 2;     // +s: tightened axis s
constexpr int kCntTop = 4;       // final top-m
constexpr int kCntTopT = 5;      // tightened final top-m

typedef unsigned long long u64;

struct SelShared {
    __align__(16) u64 cand[2][kCap];   // flat candidate lists, one per selection; the
                                       // final winners by rank reuse list 1
    __align__(16) u64 win[2][kMaxK];   // axis winners by rank
    float core[kMaxR * kMaxR];         // C of this head
    int cnt[8];                        // list lengths (may exceed kCap: overflow)
    uint32_t vt[2][kWarps];
    __align__(16) u64 runs[kThreads];  // sorted warp runs of rank_sorted
    int hist[256];
    int warp_tot[kWarps];
    int digit, remaining;
    float scalar;
    double dscalar;   // fp32 storage: the softmax denominator in fp64
    unsigned long long xbar;   // paired selection: the row CTA's exchange mbarrier
};

template <typename T>
__device__ __forceinline__ void unpack16(uint4 v, float (&f)[16 / sizeof(T)]);
template <>
__device__ __forceinline__ void unpack16<__nv_bfloat16>(uint4 v, float (&f)[8]) {
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        f[2 * q] = __uint_as_float(u[q] << 16);
        f[2 * q + 1] = __uint_as_float(u[q] & 0xffff0000u);
    }
}
template <>
__device__ __forceinline__ void unpack16<float>(uint4 v, float (&f)[4]) {
    f[0] = __uint_as_float(v.x);
    f[1] = __uint_as_float(v.y);
    f[2] = __uint_as_float(v.z);
    f[3] = __uint_as_float(v.w);
}

// Inserts v into a lane's two largest values m1 >= m2.
__device__ __forceinline__ void top2(uint32_t v, uint32_t &m1, uint32_t &m2) {
    m2 = max(m2, min(v, m1));
    m1 = max(m1, v);
}

// The j-th largest (1 <= j <= 32) of the warp's 64 values {m1, m2}: j rounds
// of a warp maximum, each removing one instance (the lowest lane holding it).
__device__ __forceinline__ uint32_t warp_jth_top2(uint32_t m1, uint32_t m2, int j) {
    const int lane = threadIdx.x & 31;
    uint32_t t = 0u;
#pragma unroll 1
    for (int r = 0; r < j; ++r) {
        t = __reduce_max_sync(kFull, m1);
        const unsigned bal = __ballot_sync(kFull, m1 == t);
        if (lane == __ffs(bal) - 1) {
            m1 = m2;
            m2 = 0u;
        }
    }
    return t;
}

// Each warp's bound for a top-kk selection into sh.vt[s][warp] from its
// lanes' two largest keys (a0 >= a1 of selection 0, b0 >= b1 of selection 1).
// No barrier.
__device__ __forceinline__ void warp_bounds(uint32_t a0, uint32_t a1, uint32_t b0, uint32_t b1,
                                            int ns, int kk, SelShared &sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int j = (kk + kWarps - 1) / kWarps;
    const uint32_t t0 = j <= 32 ? warp_jth_top2(a0, a1, j) : 0u;
    const uint32_t t1 = ns > 1 && j <= 32 ? warp_jth_top2(b0, b1, j) : 0u;
    if (lane == 0) {
        sh.vt[0][warp] = t0;
        sh.vt[1][warp] = t1;
    }
}

__device__ __forceinline__ uint32_t block_bound(int s, const SelShared &sh) {
    uint32_t tau = sh.vt[s][0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) tau = min(tau, sh.vt[s][w]);
    return tau;
}

// Exclusive prefix sum of one int per thread over the block; also syncs.
__device__ int block_exclusive_scan(int v, SelShared &sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        int y = __shfl_up_sync(kFull, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) sh.warp_tot[warp] = incl;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += sh.warp_tot[w];
    __syncthreads();
    return before + incl - v;
}

// One digit of a radix select: given the histogram of the current digit
// over the entries that match the digits chosen so far, warp 0 finds the
// digit that holds the `remaining`-th largest entry and leaves it, and the
// rank still to go within it, in sh.digit and sh.remaining.
__device__ __forceinline__ void radix_digit(int remaining, SelShared &sh) {
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int cnt[8], s = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            cnt[j] = sh.hist[255 - 8 * lane - j];
            s += cnt[j];
        }
        int incl = s;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            int y = __shfl_up_sync(kFull, incl, off);
            if (lane >= off) incl += y;
        }
        int before = incl - s;
        if (before < remaining && remaining <= incl) {
            int acc = before;
            for (int j = 0; j < 8; ++j) {
                if (acc + cnt[j] >= remaining) {
                    sh.digit = 255 - 8 * lane - j;
                    sh.remaining = remaining - acc;
                    break;
                }
                acc += cnt[j];
            }
        }
    }
}

// Radix select (8-bit digits, most significant first) of the kk-th largest
// key among key[0..n).  Returns that key T; *need_eq = how many keys equal to
// T belong to the top kk (count(key > T) = kk - *need_eq).
__device__ uint32_t select_kth_largest(const uint32_t *key, int n, int kk, SelShared &sh,
                                       int *need_eq) {
    uint32_t prefix = 0, mask = 0;
    int remaining = kk;
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int i = threadIdx.x; i < 256; i += kThreads) sh.hist[i] = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += kThreads) {
            uint32_t v = key[i];
            if ((v & mask) == prefix) atomicAdd(&sh.hist[(v >> shift) & 255u], 1);
        }
        __syncthreads();
        radix_digit(remaining, sh);
        __syncthreads();
        prefix |= (uint32_t)sh.digit << shift;
        mask |= 255u << shift;
        remaining = sh.remaining;
        __syncthreads();
    }
    *need_eq = remaining;
    return prefix;
}

// Exact replacement of an overflowed list: exactly kk candidates (every key
// > T, then the first ties at T in position order) into cand[s], length in
// cnt[slot].  Out of line: it only runs on heavy ties.
__device__ __noinline__ void radix_fallback(const uint32_t *key, int n, int kk, int s, int slot,
                                            SelShared &sh) {
    int need_eq;
    const uint32_t T = select_kth_largest(key, n, kk, sh, &need_eq);
    const int n_gt = kk - need_eq;
    const int per = (n + kThreads - 1) / kThreads;
    const int beg = min(n, (int)threadIdx.x * per), end = min(n, beg + per);
    int gt = 0, eq = 0;
    for (int i = beg; i < end; ++i) {
        gt += key[i] > T;
        eq += key[i] == T;
    }
    int o = block_exclusive_scan(gt, sh);
    int e = block_exclusive_scan(eq, sh);
    for (int i = beg; i < end; ++i) {
        const uint32_t v = key[i];
        if (v > T) sh.cand[s][o++] = comp_of(v, (uint32_t)i);
        else if (v == T && e < need_eq) sh.cand[s][n_gt + e++] = comp_of(v, (uint32_t)i);
        else if (v == T) ++e;
    }
    if (threadIdx.x == 0) sh.cnt[slot] = kk;
    __syncthreads();
}

// Appends the lanes' composites with pr set to list (length counter *cnt):
// one shared atomic per warp.  Entries past kCap are dropped (the counter
// still counts them, which marks the overflow).
__device__ __forceinline__ void warp_append(bool pr, u64 comp, u64 *list, int *cnt) {
    const int lane = threadIdx.x & 31;
    const unsigned bal = __ballot_sync(kFull, pr);
    if (bal == 0u) return;
    int base = 0;
    if (lane == 0) base = atomicAdd(cnt, __popc(bal));
    base = __shfl_sync(kFull, base, 0);
    const int slot = base + __popc(bal & ((1u << lane) - 1u));
    if (pr && slot < kCap) list[slot] = comp;
}

// The scoring's candidate list of axis s (Dims::cand): every key of the
// axis' top k is in it, with the keys above a bound, as composites.  The
// list is G segments of 64 entries (one per 64 keys); segment g holds its
// keys' candidates, in position order, in its first cnt[g] entries.  Up to
// kCap entries are gathered into cand[s] (placed by a block scan of the
// threads' counts); a longer list (heavy ties) is replaced by its exact top
// kk, a radix select over the 64-bit composites (distinct: exactly kk are >=
// the kk-th largest).  Length in cnt[slot].  Whole block; ends with a barrier.
constexpr int kSeg = 64;               // keys and entries of a list segment
constexpr int kMaxSegPerThread = 1;   // G <= 256 segments
__device__ __noinline__ void cand_fallback(const u64 *seg, const uint32_t *cnt, int G, int kk,
                                           int s, int slot, SelShared &sh) {
    const int n = kSeg * G;
    auto entry = [&](int i) -> u64 {   // 0 for an empty slot (below every composite kept)
        return i % kSeg < (int)min(cnt[i / kSeg], (uint32_t)kSeg) ? seg[i] : 0ull;
    };
    u64 prefix = 0, mask = 0;
    int remaining = kk;
    for (int shift = 56; shift >= 0; shift -= 8) {
        for (int i = threadIdx.x; i < 256; i += kThreads) sh.hist[i] = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += kThreads) {
            const u64 v = entry(i);
            if (v && (v & mask) == prefix) atomicAdd(&sh.hist[(int)((v >> shift) & 255u)], 1);
        }
        __syncthreads();
        radix_digit(remaining, sh);
        __syncthreads();
        prefix |= (u64)sh.digit << shift;
        mask |= (u64)255 << shift;
        remaining = sh.remaining;
        __syncthreads();
    }
    if (threadIdx.x == 0) sh.cnt[slot] = 0;
    __syncthreads();
    for (int i0 = 0; i0 < n; i0 += kThreads) {   // uniform trip count
        const int i = i0 + threadIdx.x;
        const u64 v = i < n ? entry(i) : 0ull;
        warp_append(v && v >= prefix, v, sh.cand[s], &sh.cnt[slot]);
    }
    __syncthreads();
}

// Both axes' lists of one (token, head) (lists `list0` and `list0 + 1`)
// into cand[0] and cand[1], lengths in cnt[kCntAxis + s].  One block scan
// places both (the two axes' counts packed in the low and high 16 bits:
// each total is at most 64 G <= 16384), and each thread loads the first
// entry of all its segments before it stores any, so that the copies cost
// one round trip to memory, not one per segment.  Whole block; ends with a
// barrier.
__device__ void load_lists(const Ptrs &p, int64_t list0, int G, int kk, SelShared &sh) {
    const uint32_t *cnt[2] = {p.gstat + list0 * G, p.gstat + (list0 + 1) * G};
    const u64 *seg[2] = {p.cand + list0 * (int64_t)G * kSeg, p.cand + (list0 + 1) * (int64_t)G * kSeg};
    int mine[2][kMaxSegPerThread], tot = 0;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
#pragma unroll
        for (int q = 0; q < kMaxSegPerThread; ++q) {
            const int g = threadIdx.x + q * kThreads;
            mine[s][q] = g < G ? (int)min(cnt[s][g], (uint32_t)kSeg) : 0;
            tot += mine[s][q] << (16 * s);
        }
    }
    const int o = block_exclusive_scan(tot, sh);
    if (threadIdx.x == kThreads - 1) {
        sh.cnt[kCntAxis] = (o + tot) & 0xffff;
        sh.cnt[kCntAxis + 1] = (o + tot) >> 16;
    }
    __syncthreads();
    const int c[2] = {sh.cnt[kCntAxis], sh.cnt[kCntAxis + 1]};
    // the first entry of every segment of this thread, then the rest
    u64 first[2][kMaxSegPerThread];
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int q = 0; q < kMaxSegPerThread; ++q)
            first[s][q] = mine[s][q] > 0 && c[s] <= kCap
                              ? seg[s][(int64_t)(threadIdx.x + q * kThreads) * kSeg]
                              : 0ull;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        if (c[s] > kCap) continue;   // uniform: the radix select below replaces it
        int at = (o >> (16 * s)) & 0xffff;
#pragma unroll
        for (int q = 0; q < kMaxSegPerThread; ++q) {
            if (mine[s][q] == 0) continue;
            const u64 *sg = seg[s] + (int64_t)(threadIdx.x + q * kThreads) * kSeg;
            sh.cand[s][at++] = first[s][q];
            for (int e = 1; e < mine[s][q]; ++e) sh.cand[s][at++] = sg[e];
        }
        // fewer than kk is impossible (the bound guarantees kk); should it
        // happen, positions past K mark the missing entries (recorded)
        for (int f = c[s] + threadIdx.x; f < kk; f += kThreads)
            sh.cand[s][f] = comp_of(0u, 0xffffffffu - (uint32_t)f);
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        if (c[s] > kCap) {
            cand_fallback(seg[s], cnt[s], G, kk, s, kCntAxis + s, sh);
        } else if (c[s] < kk) {
            if (threadIdx.x == 0) {
                sh.cnt[kCntAxis + s] = kk;
                atomicOr(p.err, kErrInternal);
            }
        }
    }
    __syncthreads();
}

// Appends key[i] >= tau_s (i < n) of NS selections to their lists.  A round
// covers 4 kThreads 16-byte groups of keys; lane l of warp w reads groups
// (q kWarps + w) 32 + l, q < 4, so that a warp's loads are contiguous, and
// marks its hits in a 16-bit mask.  A warp scan of the lanes' hit counts
// places them, one shared atomic per warp and selection reserves the room,
// and each lane writes its hits by walking its mask (re-reading a hit's key).
// The last group may extend past n (up to the 16-byte end of the array's
// section); its extra entries are masked.
template <int NS>
__device__ void compact(const uint32_t *key0, const uint32_t *key1, int n, uint32_t tau0,
                        uint32_t tau1, SelShared &sh, int slot0, int slot1) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n4 = (n + 3) >> 2;
#pragma unroll 1
    for (int r0 = 0; r0 < n4; r0 += 4 * kThreads) {
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const uint32_t *key = s ? key1 : key0;
            const uint4 *k4 = reinterpret_cast<const uint4 *>(key);
            const uint32_t tau = s ? tau1 : tau0;
            uint32_t mask = 0u;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int g = r0 + (q * kWarps + warp) * 32 + lane;
                if (g < n4) {
                    const uint4 v = k4[g];
                    uint32_t m4 = (uint32_t)(v.x >= tau) | (uint32_t)(v.y >= tau) << 1 |
                                  (uint32_t)(v.z >= tau) << 2 | (uint32_t)(v.w >= tau) << 3;
                    const int valid = n - 4 * g;   // >= 1
                    if (valid < 4) m4 &= (1u << valid) - 1u;
                    mask |= m4 << (4 * q);
                }
            }
            const int cnt = __popc(mask);
            int incl = cnt;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(kFull, incl, off);
                if (lane >= off) incl += y;
            }
            const int tot = __shfl_sync(kFull, incl, 31);
            if (tot == 0) continue;   // warp-uniform
            int base = 0;
            if (lane == 31) base = atomicAdd(&sh.cnt[s ? slot1 : slot0], tot);
            int slot = __shfl_sync(kFull, base, 31) + incl - cnt;
            u64 *list = sh.cand[s];
            while (mask) {
                const int b = __ffs(mask) - 1;
                mask &= mask - 1u;
                const int i = 4 * (r0 + ((b >> 2) * kWarps + warp) * 32 + lane) + (b & 3);
                if (slot < kCap) list[slot] = comp_of(key[i], (uint32_t)i);
                ++slot;
            }
        }
    }
}

// The same bound taken again over list s (c entries, c <= kCap); the
// survivors replace the list, length in cnt[slot_out].  Whole block; ends
// with a barrier.
__device__ void tighten(int s, int c, int kk, int slot_out, SelShared &sh) {
    u64 mine[kPerThread];
    uint32_t m1 = 0u, m2 = 0u;
#pragma unroll
    for (int q = 0; q < kPerThread; ++q) {
        const int f = threadIdx.x + q * kThreads;
        mine[q] = f < c ? sh.cand[s][f] : 0ull;
        top2(key_of(mine[q]), m1, m2);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int j = (kk + kWarps - 1) / kWarps;
    const uint32_t tw = j <= 32 ? warp_jth_top2(m1, m2, j) : 0u;
    if (lane == 0) sh.vt[s][warp] = tw;
    __syncthreads();   // also: every list entry has been read
    const uint32_t tau = block_bound(s, sh);
#pragma unroll
    for (int q = 0; q < kPerThread; ++q) {
        const bool pr = threadIdx.x + q * kThreads < c && key_of(mine[q]) >= tau;
        warp_append(pr, mine[q], sh.cand[s], &sh.cnt[slot_out]);
    }
    __syncthreads();
}

// Length of list s once it can be ranked: the radix select replaces an
// overflowed list, a long one is tightened.  Uniform; may sync.
__device__ int settle(int s, const uint32_t *key, int n, int kk, int slot, int slot_t,
                      SelShared &sh) {
    const int c = sh.cnt[slot];
    if (c > kCap) {
        radix_fallback(key, n, kk, s, slot, sh);
        return kk;
    }
    if (c > kRankSort && c > 2 * kk) {
        tighten(s, c, kk, slot_t, sh);
        return sh.cnt[slot_t];
    }
    return c;
}

// Ranks of the c entries of list (threads [0, nt) of the selection, nt a
// power of two, tid the thread's index among them): a group of G lanes per
// entry counts the entries above it; entries of rank < kk go to win[rank].
__device__ __forceinline__ void rank_list(const u64 *list, int c, int kk, u64 *win, int tid,
                                          int nt) {
    int G = 1;
    while (G < 32 && 2 * G * c <= nt) G <<= 1;
    const int sub = tid & (G - 1), slots = nt / G;
    const int span = (((c + G - 1) / G) + 7) & ~7;
    const int lo = min(c, sub * span), hi = min(c, lo + span);
    const ulonglong2 *l2 = reinterpret_cast<const ulonglong2 *>(list);
#pragma unroll 1
    for (int f0 = 0; f0 < c; f0 += slots) {
        const int f = f0 + tid / G;
        const u64 me = f < c ? list[f] : ~0ull;
        int before = 0, g = lo;
#pragma unroll 1
        for (; g + 8 <= hi; g += 8) {
            const ulonglong2 a = l2[g / 2], b = l2[g / 2 + 1], x = l2[g / 2 + 2],
                             y = l2[g / 2 + 3];
            before += (a.x > me) + (a.y > me) + (b.x > me) + (b.y > me) + (x.x > me) +
                      (x.y > me) + (y.x > me) + (y.y > me);
        }
        for (; g < hi; ++g) before += list[g] > me;
        for (int off = G >> 1; off > 0; off >>= 1) before += __shfl_xor_sync(kFull, before, off);
        if (sub == 0 && f < c && before < kk) win[before] = me;
    }
}

// Prefetch of [ptr, ptr + bytes) into L2, one 128-byte line per request.
__device__ __forceinline__ void prefetch_l2(const void *ptr, uint32_t bytes) {
    const char *c = static_cast<const char *>(ptr);
    for (uint32_t o = 0; o < bytes; o += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(c + o));
}

template <int ID>
__device__ __forceinline__ void named_barrier(int nthreads) {
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "r"(nthreads) : "memory");
}

// Exact ranks of the c <= nt entries of list (distinct composites) for
// threads [0, nt) of the selection (tid the thread's index among them, nt a
// multiple of 32): each warp sorts its run of 32 in registers (descending
// bitonic network), the runs go to runs[nt], and an entry's rank is its place
// in its own run plus, per other run, the number of entries above it (a
// 5-step binary search).  Entries of rank < kk go to win[rank].  BAR: the
// named barrier of these nt threads.
template <int BAR, int NT>
__device__ void rank_sorted(const u64 *list, int c, int kk, u64 *win, u64 *runs, int tid) {
    constexpr int nt = NT, nw = NT / 32;
    const int lane = tid & 31, w = tid >> 5;
    u64 x = tid < c ? list[tid] : 0ull;   // padding sorts below every entry
#pragma unroll
    for (int blk = 2; blk <= 32; blk <<= 1)
#pragma unroll
        for (int st = blk >> 1; st > 0; st >>= 1) {
            const u64 o = __shfl_xor_sync(kFull, x, st);
            const bool keep_max = ((lane & st) == 0) == ((lane & blk) == 0);
            x = keep_max ? (x > o ? x : o) : (x < o ? x : o);
        }
    runs[w * 32 + lane] = x;
    named_barrier<BAR>(nt);
    const int cw = min(32, max(0, c - 32 * w));   // real entries of this run
    if (lane < cw) {
        // the searches of the other runs are independent: interleaved steps
        int pos[nw];
#pragma unroll
        for (int v = 0; v < nw; ++v) pos[v] = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
#pragma unroll
            for (int v = 0; v < nw; ++v)
                if (runs[v * 32 + pos[v] + step - 1] > x) pos[v] += step;
        int rank = lane;
#pragma unroll
        for (int v = 0; v < nw; ++v) {
            // entries of the descending run above x: 0 .. 32 (the steps reach 31)
            const int cnt = pos[v] + (runs[v * 32 + pos[v]] > x);
            rank += v == w ? 0 : cnt;
        }
        if (rank < kk) win[rank] = x;
    }
}

struct SelLayout {
    float *qv;          // [2][D_k] row and column query of this (token, head)
    uint32_t *key0;     // [max(K, k*k)] axis-0 keys, then the g keys
    uint32_t *key1;     // [K] axis-1 keys (free once the axis winners are ranked)
    int *sel_i, *sel_j; // [k] surviving rows / columns in increasing index
    float *R, *scol;    // [k][r] R = S_row^T C and S_col of the survivors
    float *srow;        // MCS, fp32: [k][r] S_row of the row survivors } in key1's
    float *cparts;      // MCS: [nc][r][r] component cores of this head } space
};

// Dynamic shared memory layout; every section starts on 16 bytes.
struct SelOffsets {
    size_t qv, key0, key1, sel_i, sel_j, R, scol, srow, cparts, total;
};
__host__ __device__ inline SelOffsets sel_offsets(const Dims &d) {
    auto up = [](size_t x) { return (x + 15) & ~size_t(15); };
    SelOffsets o;
    size_t off = 0;
    o.qv = off;    off = up(off + sizeof(float) * 2 * d.d_k);
    // streamed keys: the axes' keys stay in L2 (read twice), not in shared
    // memory; candidate lists: the selection reads no keys
    const int Ka = d.stream_keys || d.cand ? 0 : d.K;
    o.key0 = off;  off = up(off + sizeof(uint32_t) * (Ka > d.k * d.k ? Ka : d.k * d.k));
    // with MCS (and with fp32 storage), key1's space later holds S_row of the
    // row survivors and the component cores (so that the block's shared
    // memory does not grow)
    const bool mcs = d.nc > 1;
    const bool keep_srow = mcs || d.dtype == ULTRAMEM_F32;
    const int mcs_floats = keep_srow ? d.k * d.r + (mcs ? d.nc * d.r * d.r : 0) : 0;
    o.key1 = off;  off = up(off + sizeof(uint32_t) * (Ka > mcs_floats ? Ka : mcs_floats));
    o.srow = o.key1;
    o.cparts = o.key1 + sizeof(float) * d.k * d.r;
    o.sel_i = off; off = up(off + sizeof(int) * d.k);
    o.sel_j = off; off = up(off + sizeof(int) * d.k);
    o.R = off;     off = up(off + sizeof(float) * d.k * d.r);
    o.scol = off;  off = up(off + sizeof(float) * d.k * d.r);
    o.total = off;
    return o;
}

__device__ SelLayout carve(const Dims &d, unsigned char *base) {
    const SelOffsets o = sel_offsets(d);
    SelLayout L;
    L.qv = reinterpret_cast<float *>(base + o.qv);
    L.key0 = reinterpret_cast<uint32_t *>(base + o.key0);
    L.key1 = reinterpret_cast<uint32_t *>(base + o.key1);
    L.sel_i = reinterpret_cast<int *>(base + o.sel_i);
    L.sel_j = reinterpret_cast<int *>(base + o.sel_j);
    L.R = reinterpret_cast<float *>(base + o.R);
    L.scol = reinterpret_cast<float *>(base + o.scol);
    L.srow = reinterpret_cast<float *>(base + o.srow);
    L.cparts = reinterpret_cast<float *>(base + o.cparts);
    return L;
}

// Loads the rank-1 score keys of both axes (Eq. 6-7, written by the scoring
// kernel) into shared memory and returns this thread's two largest of each
// axis (padding reads as 0, below every key); all loads of a round are
// issued before any store.  Each key is read once: the loads are streaming
// (L2 evict-first), so that a long batch's keys do not push the key rows,
// which every (token, head) reads again, out of L2.  With `stream` the keys
// are not stored (the compaction reads them again from L2) and are loaded
// with the L2 caching kept.
__device__ __forceinline__ uint4 ld_key4(const uint4 *p, bool stream) {
    return stream ? __ldcg(p) : __ldcs(p);
}
__device__ __forceinline__ uint32_t ld_key(const uint32_t *p, bool stream) {
    return stream ? __ldcg(p) : __ldcs(p);
}
template <int NS = 2>   // axes loaded: both, or (NS = 1) the one in A0
__device__ __forceinline__ void load_keys(const uint32_t *A0, const uint32_t *A1, int K,
                                          const SelLayout &L, uint32_t (&top)[2][2],
                                          bool stream) {
    uint32_t a1 = 0u, a2 = 0u, b1 = 0u, b2 = 0u;
    if ((K & 3) == 0) {
        const uint4 *V0 = reinterpret_cast<const uint4 *>(A0);
        const uint4 *V1 = reinterpret_cast<const uint4 *>(A1);
        uint4 *S0 = reinterpret_cast<uint4 *>(L.key0), *S1 = reinterpret_cast<uint4 *>(L.key1);
        const int nv = K >> 2;
#pragma unroll 1
        for (int v0 = threadIdx.x; v0 < nv; v0 += 4 * kThreads) {
            uint4 a[4], c[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = v0 + q * kThreads;
                a[q] = i < nv ? ld_key4(V0 + i, stream) : make_uint4(0, 0, 0, 0);
                c[q] = NS > 1 && i < nv ? ld_key4(V1 + i, stream) : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = v0 + q * kThreads;
                if (i < nv && !stream) {
                    S0[i] = a[q];
                    if (NS > 1) S1[i] = c[q];
                }
                top2(a[q].x, a1, a2);
                top2(a[q].y, a1, a2);
                top2(a[q].z, a1, a2);
                top2(a[q].w, a1, a2);
                top2(c[q].x, b1, b2);
                top2(c[q].y, b1, b2);
                top2(c[q].z, b1, b2);
                top2(c[q].w, b1, b2);
            }
        }
    } else {
#pragma unroll 1
        for (int i0 = threadIdx.x; i0 < K; i0 += 4 * kThreads) {
            uint32_t a[4], c[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = i0 + q * kThreads;
                a[q] = i < K ? ld_key(A0 + i, stream) : 0u;
                c[q] = NS > 1 && i < K ? ld_key(A1 + i, stream) : 0u;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = i0 + q * kThreads;
                if (i < K && !stream) {
                    L.key0[i] = a[q];
                    if (NS > 1) L.key1[i] = c[q];
                }
                top2(a[q], a1, a2);
                top2(c[q], b1, b2);
            }
        }
    }
    top[0][0] = a1;
    top[0][1] = a2;
    top[1][0] = b1;
    top[1][1] = b2;
}

// A 16-byte load of a key row with the L2 evict-last policy: the rows are
// read again by the other (token, head) pairs of the batch.
__device__ __forceinline__ uint64_t key_row_policy() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ uint4 ld_key_row(const uint4 *ptr, uint64_t pol) {
    uint4 v;
    asm volatile("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(ptr), "l"(pol));
    return v;
}
__device__ __forceinline__ uint4 ld_key_row(const uint4 *ptr) {
    return ld_key_row(ptr, key_row_policy());
}
// The same into v when `go`, without a branch (which would keep the work
// around it from interleaving).
__device__ __forceinline__ void ld_key_row_if(uint4 &v, const uint4 *ptr, uint64_t pol, bool go) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "@p ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;\n\t}"
        : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w)
        : "l"(ptr), "l"(pol), "r"((int)go));
}

// The paired decode selection's cluster barrier (arrive, then wait).
__device__ __forceinline__ void cl_arrive_relaxed() {
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The exchange mbarrier of the paired selection (in the row CTA): one
// arrival, which also expects the column CTA's survivors' bytes; the init is
// published to the pair by a release fence and the pair's first cluster
// barrier.
__device__ __forceinline__ void xbar_init(unsigned long long *bar, uint32_t bytes) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(bar);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(a) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(a), "r"(bytes)
                 : "memory");
}
// A 32-bit store into the same shared-memory location of CTA `rank`, which
// completes 4 bytes of that CTA's mbarrier at the same offset as `bar`.
__device__ __forceinline__ void st_async_u32(const void *local, uint32_t rank, uint32_t v,
                                             const unsigned long long *bar) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(local);
    const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar);
    uint32_t ra, rb;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(b), "r"(rank));
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(ra),
                 "r"(v), "r"(rb)
                 : "memory");
}
// Bounded wait (about a second of SM cycles) for phase 0 of the exchange
// mbarrier, with cluster-scope acquire: the column CTA's stores are then
// visible.  Returns false when it gave up.
__device__ __forceinline__ bool xbar_wait(unsigned long long *bar) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(bar);
    const long long start = clock64();
    for (;;) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(a)
            : "memory");
        if (ok) return true;
        if (clock64() - start > (1ll << 31)) return false;
    }
}

// The 2k axis survivors, one group of G lanes each: the survivor's place in
// increasing key index (so that enumerating I x J row-major is increasing
// v = i*K + j), and its exact chunk scores S_alpha (Eq. 4) from 16-byte
// loads of its key row split over the group.  Row survivors store
// R[i][b] = sum_a S_row[a,i] C[a,b], column survivors S_col[j][b].
// RM >= r bounds the rank at compile time (2 for the common ranks, else 8).
// gax < 0: both axes (winners of axis s in win[s]); gax = 0 or 1 (the
// paired decode selection): only axis gax, whose winners are in win[0].
template <typename T, int RM>
__device__ void axis_survivors(const Dims &d, const Ptrs &p, int h, const SelLayout &L,
                               const SelShared &sh, int gax = -1) {
    constexpr int EPV = 16 / sizeof(T);
    const int k = d.k, r = d.r, dk = d.dk, D = d.d_k;
    const int nl = gax < 0 ? 2 : 1;   // lists
    // G = 2^lg lanes per survivor, sized for two lists in either case: the
    // lanes' partial sums (and so the scores' roundings) are then the same
    // whether one CTA takes both axes or a pair one each
    int lg = 0;
    while (lg < 5 && 2 * k * (2 << lg) <= kThreads) ++lg;
    const int G = 1 << lg;
    const int lane = threadIdx.x & 31, sub = lane & (G - 1);
    const int sv = threadIdx.x >> lg;   // 2k G <= kThreads: one pass
    const bool active = sv < nl * k;
    const int ls = active && sv >= k ? 1 : 0;   // the list
    const int s = gax < 0 ? ls : gax;           // its axis
    const int qi = active ? sv - ls * k : 0;
    uint32_t pos = active ? pos_of(sh.win[ls][qi]) : 0u;
    if (active && pos >= (uint32_t)d.K) {   // never expected: record and skip
        if (sub == 0) atomicOr(p.err, kErrInternal);
        pos = 0u;
    }

    const T *row = static_cast<const T *>(s ? p.k_col : p.k_row) + ((int64_t)h * d.K + pos) * D;
    const float *q = L.qv + s * D;
    const bool vec = D % EPV == 0 && dk % EPV == 0 && ((uintptr_t)row & 15) == 0;
    const uint4 *rv = reinterpret_cast<const uint4 *>(row);
    const int nvec = vec ? D / EPV : 0;
    // the first batch of the row's 16-byte loads is issued before the order
    // scan below, which reads shared memory only
    uint4 buf[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int iv = sub + u * G;
        buf[u] = active && iv < nvec ? ld_key_row(rv + iv) : make_uint4(0, 0, 0, 0);
    }

    int ord = 0;
    if (active) {
        int g = sub;
        for (; g + 3 * G < k; g += 4 * G) {
            const uint32_t a = pos_of(sh.win[ls][g]), b = pos_of(sh.win[ls][g + G]),
                           c = pos_of(sh.win[ls][g + 2 * G]), e = pos_of(sh.win[ls][g + 3 * G]);
            ord += (a < pos) + (b < pos) + (c < pos) + (e < pos);
        }
        for (; g < k; g += G) ord += pos_of(sh.win[ls][g]) < pos;
    }
    for (int off = G >> 1; off > 0; off >>= 1) ord += __shfl_xor_sync(kFull, ord, off);

    float S[RM];
#pragma unroll
    for (int a = 0; a < RM; ++a) S[a] = 0.f;
    // fp32 storage: each chunk score as a compensated dot product (Dot2),
    // so that the weights carry the working precision (see Dot2)
    constexpr bool kExact = std::is_same<T, float>::value;
    Dot2 SX[kExact ? RM : 1];
    if (vec) {
        // 16-byte group iv of the row belongs to chunk iv / cpv
        const int cpv = dk / EPV;
        // (rank > 2) chunk of element x = floor(x / dk), as floor((x + 1/2) /
        // dk) in fp32: exact while x, dk < 2^20 (the error stays below 1/(2 dk))
        const float inv_dk = 1.f / (float)dk;
#pragma unroll 1
        for (int u0 = sub; u0 < nvec; u0 += 8 * G) {
            if (u0 != sub) {
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int iv = u0 + u * G;
                    buf[u] = active && iv < nvec ? ld_key_row(rv + iv) : make_uint4(0, 0, 0, 0);
                }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int iv = u0 + u * G;
                if (iv < nvec) {
                    float f[EPV];
                    unpack16<T>(buf[u], f);
                    // q + iv*EPV is 16-byte aligned: qv is, and D % EPV == 0
                    const float4 *qq = reinterpret_cast<const float4 *>(q + iv * EPV);
                    if constexpr (kExact) {
                        // the vector lies in one chunk: add its products there
                        const int al = RM == 2 ? (iv >= cpv ? RM - 1 : 0)
                                               : (int)(((float)(iv * EPV) + 0.5f) * inv_dk);
#pragma unroll
                        for (int a = 0; a < RM; ++a) {
                            if (a == al) {
#pragma unroll
                                for (int e4 = 0; e4 < EPV / 4; ++e4) {
                                    const float4 q4 = qq[e4];
                                    SX[a].add(f[4 * e4], q4.x);
                                    SX[a].add(f[4 * e4 + 1], q4.y);
                                    SX[a].add(f[4 * e4 + 2], q4.z);
                                    SX[a].add(f[4 * e4 + 3], q4.w);
                                }
                            }
                        }
                        continue;
                    }
                    float pv = 0.f;
#pragma unroll
                    for (int e4 = 0; e4 < EPV / 4; ++e4) {
                        const float4 q4 = qq[e4];
                        pv = fmaf(f[4 * e4], q4.x, pv);
                        pv = fmaf(f[4 * e4 + 1], q4.y, pv);
                        pv = fmaf(f[4 * e4 + 2], q4.z, pv);
                        pv = fmaf(f[4 * e4 + 3], q4.w, pv);
                    }
                    if (RM == 2) {   // rank 1 or 2: the second chunk starts at cpv
                        const bool hi = iv >= cpv;
                        S[0] += hi ? 0.f : pv;
                        S[RM - 1] += hi ? pv : 0.f;
                    } else {
                        const int al = (int)(((float)(iv * EPV) + 0.5f) * inv_dk);
#pragma unroll
                        for (int a = 0; a < RM; ++a)
                            if (a < r) S[a] += a == al ? pv : 0.f;   // r is uniform
                    }
                }
            }
        }
    } else {
#pragma unroll
        for (int a = 0; a < RM; ++a) {
            if (a < r && active) {
                float acc = 0.f;
                for (int c = a * dk + sub; c < (a + 1) * dk; c += G) {
                    if constexpr (kExact) SX[a].add(to_f(row[c]), q[c]);
                    else acc = fmaf(to_f(row[c]), q[c], acc);
                }
                S[a] = acc;
            }
        }
    }
    if constexpr (kExact) {
        // the group's partial sums merged with their error terms
#pragma unroll
        for (int a = 0; a < RM; ++a) {
            if (a < r) {
                for (int off = G >> 1; off > 0; off >>= 1) {
                    Dot2 o;
                    o.s = __shfl_xor_sync(kFull, SX[a].s, off);
                    o.c = __shfl_xor_sync(kFull, SX[a].c, off);
                    SX[a].merge(o);
                }
                S[a] = SX[a].value();
            }
        }
    } else {
#pragma unroll
        for (int a = 0; a < RM; ++a) {
            if (a < r)
                for (int off = G >> 1; off > 0; off >>= 1) S[a] += __shfl_xor_sync(kFull, S[a], off);
        }
    }
    if (active && sub == 0) {
        if (s == 0) {
            L.sel_i[ord] = (int)pos;
            // MCS (the individual scores) and fp32 storage (the weights in
            // fp64) need S_row itself
            if (d.nc > 1 || kExact)
#pragma unroll
                for (int a = 0; a < RM; ++a)
                    if (a < r) L.srow[ord * r + a] = S[a];
#pragma unroll
            for (int b = 0; b < RM; ++b) {
                if (b < r) {
                    float acc = 0.f;
#pragma unroll
                    for (int a = 0; a < RM; ++a)
                        if (a < r) acc = fmaf(S[a], sh.core[a * r + b], acc);
                    L.R[ord * r + b] = acc;
                }
            }
        } else {
            L.sel_j[ord] = (int)pos;
#pragma unroll
            for (int b = 0; b < RM; ++b)
                if (b < r) L.scol[ord * r + b] = S[b];
        }
    }
}

// MINB: resident CTAs per SM the registers are sized for (3: about 80
// registers, for grids of up to about three CTAs per SM, where a CTA's
// latency matters; 4: 64 registers, for long grids, where occupancy does).
// RM >= r: the rank bound of the survivor phase (2, or 8 for larger ranks),
// one per kernel so that each carries a single copy of it.
// PAIR (decode grids of at most one (token, head) per SM): a cluster of two
// CTAs per (token, head), blockIdx.z = its axis.  Each takes one axis through
// the key load, bound, compaction, rank and survivors (half the work a warp
// does in those phases); the column CTA then sends its survivors (indices
// and S_col) into the row CTA's shared memory with asynchronous stores that
// complete bytes of the row CTA's exchange mbarrier, and the row CTA, once
// that barrier completes, goes on alone (Tucker scores, top-m, outputs).
// FIRST: the body of a kernel, with its dependency wait and stamps; else a
// (token, head) that the warp-wise selection below left to its block.
template <typename T, int MINB, int RM, bool PAIR, bool FIRST>
__device__ __forceinline__ void select_block(const Dims &d, const Ptrs &p, int bh,
                                             unsigned char *smem_raw, SelShared &sh) {
    const int b = bh / d.H, h = bh % d.H;
    const int ax = PAIR ? (int)blockIdx.z : 0;   // the cluster's rank (cluster 1 x 1 x 2)
    const SelLayout L = carve(d, smem_raw);
    const int r = d.r, K = d.K, k = d.k, m = d.m;
    const uint32_t *A0 = p.akey + (((int64_t)b * d.H + h) * 2 + ax) * (int64_t)K;
    const uint32_t *A1 = A0 + K;   // (not read when PAIR)

    if (threadIdx.x < 8) sh.cnt[threadIdx.x] = 0;
    if constexpr (PAIR) {
        // the row CTA's exchange barrier, expecting the column CTA's
        // survivors (k indices and k r scores); the pair's cluster barrier
        // arrival publishes it, its wait comes just before the exchange
        if (ax == 0 && threadIdx.x == 0) xbar_init(&sh.xbar, (uint32_t)(d.k + d.k * d.r) * 4u);
        cl_arrive_relaxed();
    }
    // C of this head (a weight: read before the dependency wait) and the
    // row/column query of this (token, head): loaded before the keys, stored
    // after them
    const float core_e = threadIdx.x < r * r ? p.core[(int64_t)h * r * r + threadIdx.x] : 0.f;
    // MCS component cores (nc r^2 <= 2 kThreads), stored once key1 is free
    const int ncrr = d.nc > 1 ? d.nc * r * r : 0;
    const float *cp = p.cores + (int64_t)h * ncrr;
    const float cp0 = threadIdx.x < ncrr ? cp[threadIdx.x] : 0.f;
    const float cp1 = threadIdx.x + kThreads < ncrr ? cp[threadIdx.x + kThreads] : 0.f;
    if constexpr (FIRST) {
        pdl_wait();
        stamp_begin(p.stamp);
        pdl_trigger();
    }
    const int HD = d.H * d.d_k;
    const int64_t split_stride = (int64_t)d.A * d.B * HD;
    auto q_src = [&](int e) {
        const int axis = e / d.d_k, c = e - axis * d.d_k;
        const int a = (axis == 1 && d.A == 2) ? 1 : 0;
        return p.q_part + ((int64_t)a * d.B + b) * HD + h * d.d_k + c;
    };
    // (the query kernel has added up the D_i splits: one round of these loops.
    // Without them the warp-wise kernels, which end in this code, came out
    // slower: retrievals with lists 85.9 -> 87.5 us at K = 16000 with 256 tokens,
    // 67.4 -> 68.3 at K = 9000 with 520.)
    auto q_of = [&](int e) {
        const float *src = q_src(e);
        if constexpr (std::is_same<T, float>::value) {
            double q = 0.0;
            for (int s = 0; s < d.q_splits; ++s) q += (double)src[s * split_stride];
            return (float)q;
        } else {
            float q = 0.f;
            for (int s = 0; s < d.q_splits; ++s) q += src[s * split_stride];
            return q;
        }
    };
    const bool one_split = d.q_splits == 1;
    // the query elements this CTA needs: both axes', or its own axis'
    const int e0 = PAIR ? ax * d.d_k : 0, ne = PAIR ? d.d_k : 2 * d.d_k;
    float q0 = 0.f;
    if (threadIdx.x < ne) q0 = one_split ? *q_src(e0 + threadIdx.x) : q_of(e0 + threadIdx.x);
    uint32_t top[2][2];
    const bool stream = d.stream_keys != 0;   // uniform
    // candidate lists: only the long-grid instantiation reads them (the
    // launch picks it whenever they are on)
    const bool lists = MINB >= 4 && d.cand;
    if constexpr (PAIR) load_keys<1>(A0, A1, K, L, top, stream);
    else if (!lists) load_keys(A0, A1, K, L, top, stream);
    // the axes' keys: in shared memory, or (streamed) in L2, where the
    // compaction reads them a second time
    const uint32_t *KA = stream ? A0 : L.key0, *KB = stream ? A1 : L.key1;
    if (threadIdx.x < r * r) sh.core[threadIdx.x] = core_e;
    if (threadIdx.x < ne) L.qv[e0 + threadIdx.x] = q0;
    for (int e = threadIdx.x + kThreads; e < ne; e += kThreads) L.qv[e0 + e] = q_of(e0 + e);

    // Eq. 8-9: top-k of both axes
    if constexpr (PAIR) {   // this CTA's axis as list 0
        warp_bounds(top[0][0], top[0][1], 0u, 0u, 1, k, sh);
        __syncthreads();
        compact<1>(KA, nullptr, K, block_bound(0, sh), 0u, sh, kCntAxis, kCntAxis);
        __syncthreads();
    } else if (lists) {   // the scoring left each axis' candidates
        __syncthreads();
        load_lists(p, ((int64_t)b * d.H + h) * 2, d.n_segs, k, sh);
    } else {
        warp_bounds(top[0][0], top[0][1], top[1][0], top[1][1], 2, k, sh);
        __syncthreads();
        compact<2>(KA, KB, K, block_bound(0, sh), block_bound(1, sh), sh, kCntAxis,
                   kCntAxis + 1);
        __syncthreads();
    }
    const int c0 = settle(0, KA, K, k, kCntAxis, kCntAxisT, sh);
    const int c1 = PAIR ? 0 : settle(1, KB, K, k, kCntAxis + 1, kCntAxisT + 1, sh);
    if constexpr (PAIR) {
        rank_list(sh.cand[0], c0, k, sh.win[0], threadIdx.x, kThreads);
    } else {
        const int s = threadIdx.x >= kThreads / 2, cs = s ? c1 : c0;
        const int tid = threadIdx.x & (kThreads / 2 - 1);
        // long grids (issue-bound) rank by sorted runs, which execute fewer
        // instructions; decode grids (latency-bound) by counting, which
        // has the shorter dependency chain
        if (MINB >= 4 && c0 <= kThreads / 2 && c1 <= kThreads / 2) {   // uniform
            if (s)   // warp-uniform: each half of the block has its own barrier
                rank_sorted<2, kThreads / 2>(sh.cand[1], cs, k, sh.win[1], sh.runs + kThreads / 2,
                                             tid);
            else
                rank_sorted<1, kThreads / 2>(sh.cand[0], cs, k, sh.win[0], sh.runs, tid);
        } else
            rank_list(sh.cand[s], cs, k, sh.win[s], tid, kThreads / 2);
    }
    __syncthreads();
    if (threadIdx.x < ncrr) L.cparts[threadIdx.x] = cp0;   // key1 is free now
    if (threadIdx.x + kThreads < ncrr) L.cparts[threadIdx.x + kThreads] = cp1;
    // survivors in increasing index with their exact chunk scores (Eq. 4)
    axis_survivors<T, RM>(d, p, h, L, sh, PAIR ? ax : -1);
    __syncthreads();
    if constexpr (PAIR) {
        // the column CTA sends its survivors into the row CTA with
        // asynchronous stores that complete bytes of the row CTA's exchange
        // mbarrier, and is done; the row CTA waits on that barrier
        cl_wait();   // the exchange barrier is initialised
        if (ax == 1) {
            for (int i = threadIdx.x; i < k; i += kThreads)
                st_async_u32(L.sel_j + i, 0u, (uint32_t)L.sel_j[i], &sh.xbar);
            for (int i = threadIdx.x; i < k * r; i += kThreads)
                st_async_u32(L.scol + i, 0u, __float_as_uint(L.scol[i]), &sh.xbar);
            stamp_end(p.stamp);
            return;
        }
        if (!xbar_wait(&sh.xbar) && threadIdx.x == 0) atomicOr(p.err, kErrTimeout);
    }

    u64 *const fwin = sh.cand[1];   // final winners by rank (list 1 is free now)

    // Eq. 10: g(i,j) = sum_b R[i][b] S_col[b,j] on I x J, R = S_row^T C.
    // Which thread computes which pair decides how tight the bound below is:
    // it is the smallest of the 8 warps' values, so every warp should hold a
    // spread sample of rows and columns.  In index order (pair c to thread
    // c mod 256) a warp holds a few rows and half of the columns, and about
    // twice as many candidates pass (final list at decode_1m, median over
    // CTAs: 126 of 1024 for m = 32; 49 with a spread assignment).
    const int k2 = k * k;
    uint32_t g1 = 0u, g2 = 0u;
    if (!d.pkm && r == 2 && (k & 31) == 0) {   // uniform
        // lane l of warp w owns columns l + 32 h (h < k/32; S_col in
        // registers) and, of each, the rows ((w + l) mod 8) + 8 i (i < k/8):
        // a warp holds every row and every column (8 warps, kThreads = 256)
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        const int i0 = (w + lane) & 7;
        for (int jj = lane; jj < k; jj += 32) {
            const float2 b2 = *reinterpret_cast<const float2 *>(L.scol + jj * 2);
            for (int ii = i0; ii < k; ii += 8) {
                const float2 a2 = *reinterpret_cast<const float2 *>(L.R + ii * 2);
                const uint32_t kg = f2ord(fmaf(a2.y, b2.y, a2.x * b2.x));
                L.key0[ii * k + jj] = kg;
                top2(kg, g1, g2);
            }
        }
    } else {
        // any shape: thread t visits the pairs p = t, t + kThreads, ... as
        // pair index pp = p kPairMix mod k^2 (a bijection: kPairMix is a
        // prime above kMaxK)
        const uint32_t uk2 = (uint32_t)k2;
        const uint32_t step = (uint32_t)(((uint64_t)kThreads * kPairMix) % uk2);
        uint32_t pp = (uint32_t)(((uint64_t)threadIdx.x * kPairMix) % uk2);
        // ii = pp / k as floor((pp + 1/2) / k) in fp32: pp < 2^14 and k <= 128,
        // so the rounding error (< 2^-16) stays below the 1/(2k) margin
        const float inv_k = 1.f / (float)k;
        for (int c = threadIdx.x; c < k2; c += kThreads) {
            const int ii = (int)(((float)pp + 0.5f) * inv_k);
            const int jj = (int)pp - ii * k;
            float g;
            if (d.pkm) {    // product keys (Eq. 2): s_row[i] + s_col[j]
                g = L.R[ii] + L.scol[jj];
            } else if (r == 2) {   // the common rank, without the loop
                const float2 a2 = *reinterpret_cast<const float2 *>(L.R + ii * 2);
                const float2 b2 = *reinterpret_cast<const float2 *>(L.scol + jj * 2);
                g = fmaf(a2.y, b2.y, a2.x * b2.x);
            } else {
                g = 0.f;
                for (int be = 0; be < r; ++be) g = fmaf(L.R[ii * r + be], L.scol[jj * r + be], g);
            }
            const uint32_t kg = f2ord(g);
            L.key0[pp] = kg;
            top2(kg, g1, g2);
            pp += step;
            if (pp >= uk2) pp -= uk2;
        }
    }
    warp_bounds(g1, g2, 0u, 0u, 1, m, sh);
    __syncthreads();
    compact<1>(L.key0, nullptr, k2, block_bound(0, sh), 0u, sh, kCntTop, kCntTop);
    __syncthreads();
    const int cf = settle(0, L.key0, k2, m, kCntTop, kCntTopT, sh);
    if (MINB >= 4 && cf <= kThreads)
        rank_sorted<3, kThreads>(sh.cand[0], cf, m, fwin, sh.runs, threadIdx.x);
    else rank_list(sh.cand[0], cf, m, fwin, threadIdx.x, kThreads);
    __syncthreads();

    // fp32 storage: the weights are the winners' scores recomputed in fp64
    // from the exact chunk scores (S_row, S_col) and the core, rounded once;
    // the fp32 scores above only decided the order
    constexpr bool kExact = std::is_same<T, float>::value;
    auto exact_g = [&](int ii, int jj, const float *Cm) -> double {
        if (d.pkm) return (double)L.srow[ii] + (double)L.scol[jj];   // Eq. 2: r = 1
        double g = 0.0;
        for (int a = 0; a < r; ++a) {
            double cs = 0.0;
            for (int be = 0; be < r; ++be)
                cs += (double)Cm[a * r + be] * (double)L.scol[jj * r + be];
            g += (double)L.srow[ii * r + a] * cs;
        }
        return g;
    };
    auto pair_of = [&](u64 wc, int &ii, int &jj) {
        int c = (int)pos_of(wc);
        if ((uint32_t)c >= (uint32_t)k2) c = 0;   // recorded below
        ii = c / k;
        jj = c - ii * k;
    };
    double gmax_d = 0.0;
    if constexpr (kExact) {
        if (d.act == ULTRAMEM_ACT_SOFTMAX) {
            int i0, j0;
            pair_of(fwin[0], i0, j0);
            gmax_d = exact_g(i0, j0, sh.core);
            if (threadIdx.x < 32) {
                double z = 0.0;
                for (int e = threadIdx.x; e < m; e += 32) {
                    int ii, jj;
                    pair_of(fwin[e], ii, jj);
                    z += exp(exact_g(ii, jj, sh.core) - gmax_d);
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) z += __shfl_xor_sync(kFull, z, off);
                if (threadIdx.x == 0) sh.dscalar = z;
            }
            __syncthreads();
        }
    }

    // PKM's softmax over the m selected scores (Eq. 3); Trick 1 skips it
    const float gmax = ord2f(key_of(fwin[0]));
    if (!kExact && d.act == ULTRAMEM_ACT_SOFTMAX) {
        if (threadIdx.x < 32) {
            float z = 0.f;
            for (int e = threadIdx.x; e < m; e += 32) z += __expf(ord2f(key_of(fwin[e])) - gmax);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) z += __shfl_xor_sync(kFull, z, off);
            if (threadIdx.x == 0) sh.scalar = z;
        }
        __syncthreads();
    }
    const int64_t base = ((int64_t)b * d.H + h) * m;
    const uint32_t N = (uint32_t)d.N;
    const uint32_t row_bytes = (uint32_t)d.d_v * (d.dtype == ULTRAMEM_BF16 ? 2u : 4u);
    const bool prefetch = (uint64_t)d.B * d.H * m * row_bytes <= kPrefetchMaxBytes;
    for (int e = threadIdx.x; e < m; e += kThreads) {
        const u64 wc = fwin[e];
        int c = (int)pos_of(wc);
        if ((uint32_t)c >= (uint32_t)k2) {   // never expected: record and skip
            atomicOr(p.err, kErrInternal);
            c = 0;
        }
        const int ii = c / k, jj = c - ii * k;
        const uint64_t v = (uint64_t)L.sel_i[ii] * (uint64_t)K + (uint64_t)L.sel_j[jj];
        const float g = ord2f(key_of(wc));
        float w;
        if constexpr (kExact) {
            const double gd = exact_g(ii, jj, sh.core);
            w = (float)(d.act == ULTRAMEM_ACT_SOFTMAX ? exp(gd - gmax_d) / sh.dscalar : gd);
        } else {
            w = d.act == ULTRAMEM_ACT_SOFTMAX ? __expf(g - gmax) / sh.scalar : g;
        }
        const uint32_t vs = (uint32_t)shuffle_address(d, p.perm, v);   // Eq. 14, < M < 2^32
        const uint32_t pb = vs / N;
        const uint32_t prow = vs - pb * N;
        p.sel_row[base + e] = (int32_t)prow;
        p.sel_p[base + e] = (int32_t)pb;
        if (p.idx_out) p.idx_out[base + e] = (int64_t)v;
        if (d.nc == 1) {
            p.sel_w[base + e] = w;
            if (p.w_out) p.w_out[base + e] = w;
        } else {
            // MCS (Eq. 16-17): the individual scores S_row^T C^(i) S_col of
            // this slot, one per value slice (the softmax is not allowed here)
            float sr[RM], sc[RM];
#pragma unroll
            for (int a = 0; a < RM; ++a) {
                sr[a] = a < r ? L.srow[ii * r + a] : 0.f;
                sc[a] = a < r ? L.scol[jj * r + a] : 0.f;
            }
            for (int ci = 0; ci < d.nc; ++ci) {
                const float *Cc = L.cparts + ci * r * r;
                if constexpr (kExact) {   // fp32 storage: in fp64, rounded once
                    const float gx = (float)exact_g(ii, jj, Cc);
                    p.sel_w[(base + e) * d.nc + ci] = gx;
                    if (p.w_out) p.w_out[(base + e) * d.nc + ci] = gx;
                    continue;
                }
                float gi = 0.f;
#pragma unroll
                for (int a = 0; a < RM; ++a) {
                    if (a < r) {
                        float cs = 0.f;
#pragma unroll
                        for (int be = 0; be < RM; ++be)
                            if (be < r) cs = fmaf(Cc[a * r + be], sc[be], cs);
                        gi = fmaf(sr[a], cs, gi);
                    }
                }
                p.sel_w[(base + e) * d.nc + ci] = gi;
                if (p.w_out) p.w_out[(base + e) * d.nc + ci] = gi;
            }
        }
    }
    // The gather will read the winners' value rows: start moving them into
    // L2 (unless the batch's rows would not stay there until then).  Winner
    // e's row is fetched by a thread of the warps after those that stored
    // the slots (for m <= 128), which works out the slot again: a prefetch
    // holds its warp for about 1300 cycles (the row's address translation,
    // measured at decode), and this way the stores above do not wait behind
    // it.
    if (prefetch) {
        const int sw = (m + 31) / 32;   // warps that stored slots
        const int shift = 2 * sw * 32 <= kThreads ? 32 * sw : 32;
        for (int e = (threadIdx.x + kThreads - shift) % kThreads; e < m; e += kThreads) {
            int c = (int)pos_of(fwin[e]);
            if ((uint32_t)c >= (uint32_t)k2) c = 0;   // recorded above
            const int ii = c / k, jj = c - ii * k;
            const uint64_t v = (uint64_t)L.sel_i[ii] * (uint64_t)K + (uint64_t)L.sel_j[jj];
            const uint32_t vs = (uint32_t)shuffle_address(d, p.perm, v);
            const uint32_t prow = vs - (vs / N) * N;
            prefetch_l2(static_cast<const unsigned char *>(p.values) + (size_t)prow * row_bytes,
                        row_bytes);
        }
    }
    if constexpr (FIRST) stamp_end(p.stamp);
}

template <typename T, int MINB, int RM, bool PAIR = false>
__global__ void __launch_bounds__(kThreads, MINB) select_kernel(Dims d, Ptrs p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ SelShared sh;
    select_block<T, MINB, RM, PAIR, true>(d, p, (int)blockIdx.x, smem_raw, sh);
}

// ---- long grids: one warp per (token, head) ---------------------------------
// A block per (token, head) spends most of its instructions on what a block
// needs to work on one selection: barriers, block scans, bounds per warp,
// and sorts of runs of 32 that are merged by searches (21.6 thousand warp
// instructions a selection at prefill_16k, issue-bound at 2.7 a cycle).  Here
// each of a CTA's 8 warps selects for its own (token, head), without a
// barrier:
//   * an axis' top k: from the candidate lists (loaded in position order), or
//     from every key (read twice, 16 bytes a lane, with the bound taken from
//     256 group maxima); the k-th largest key is found bit by bit over the
//     candidates' keys in registers, from the first bit in which they differ
//     until exactly k are at or above it;
//   * the survivors' chunk scores, 16 (k = 64) to 8 (k = 32) rows at a time,
//     each by the same lanes in the same order as the block does;
//   * the k x k Tucker scores twice: a lane holds two columns and streams the
//     rows, two at a time (packed fp32), first for 8 group maxima a lane, of
//     which the m-th largest is the bound, then for a mask of the pairs at or
//     above it.  Nothing of the k x k grid is stored;
//   * the top m of those (about 120 at k = m = 64) by the same bit search,
//     then one bitonic sort of 64 in registers.
// The scores, the order and so the selection are those of select_block, bit
// for bit.  What a warp cannot hold (longer lists than kWCap or kWTop, scores
// that are not finite, a list shorter than k) it leaves to select_block: its
// CTA takes those (token, head)s one by one after its warps are done (12 to 30 us
// for a single one, n = 3000 with 384 tokens), but for zero queries.
// About 6200 warp instructions a selection at prefill_16k.  Measured on GB300:
// the selection of prefill_16k 1660 -> 650 us (a pass 2930 -> 1902), at mid_4m with
// 1000 tokens and two cores 118 -> 64 us, at decode_1m with 2000 tokens (every
// key) 105 -> 59 us.  Bound by latency: 8 warps a scheduler (64 registers),
// chains of shared-memory reads, shuffles and warp reductions.
constexpr int kWCap = 192;    // candidates of an axis
constexpr int kWTop = 384;    // candidates of the final top m
constexpr int kWParts = 8;    // group maxima a lane
constexpr int kWMaxK = 64;
constexpr int kWMaxD = 256;   // D_k

// The kk-th largest of the warp's keys (key[q] of the valid entries; 0 where
// there is none, below every key), or any value between it and the next
// smaller one; *cnt = how many keys are at or above it (kk unless keys tie
// with it).  1 <= kk <= c, the number of valid entries.  With a slack the
// search stops at a value that kk to kk + slack keys reach.
template <int NQ>
__device__ __forceinline__ uint32_t warp_kth(const uint32_t (&key)[NQ], int c, int kk, int *cnt,
                                             int slack = 0) {
    uint32_t mx = 0u, mn = 0xffffffffu;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        mx = max(mx, key[q]);
        mn = min(mn, key[q] - 1u);   // an empty entry wraps to the largest value
    }
    mx = __reduce_max_sync(kFull, mx);
    mn = __reduce_min_sync(kFull, mn) + 1u;
    *cnt = c;
    if (c <= kk + slack || mx == mn) return mn;
    int bit = 31 - __clz(mx ^ mn);
    uint32_t T = mx & ~((2u << bit) - 1u);
    for (; bit >= 0; --bit) {
        const uint32_t t = T | (1u << bit);
        int n = 0;
#pragma unroll
        for (int q = 0; q < NQ; ++q) n += key[q] >= t;
        n = __reduce_add_sync(kFull, n);
        if (n >= kk) {
            T = t;
            *cnt = n;
            if (n <= kk + slack) break;
        }
    }
    return T;
}

// put(i, entry) for the kk largest of the c <= 32 NQ composites of list
// (distinct), i counting them in list order.
template <int NQ, class Put>
__device__ __forceinline__ void warp_top(const u64 *list, int c, int kk, Put put) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t key[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) key[q] = lane + 32 * q < c ? key_of(list[lane + 32 * q]) : 0u;
    int cnt;
    const uint32_t T = warp_kth<NQ>(key, c, kk, &cnt);
    unsigned win = 0u;   // bit q: this lane's entry q is taken
#pragma unroll
    for (int q = 0; q < NQ; ++q) win |= (uint32_t)(key[q] >= T && key[q]) << q;
    if (cnt > kk) {   // keys tie with the kk-th: the smaller positions go first
        unsigned tie = 0u;
#pragma unroll
        for (int q = 0; q < NQ; ++q) tie |= (uint32_t)(key[q] == T && key[q]) << q;
        win &= ~tie;
        int need = kk - (int)__reduce_add_sync(kFull, __popc(win));
        while (need > 0) {
            uint32_t best = 0u;   // the largest ~position of this lane's ties
            int bq = 0;
#pragma unroll 1
            for (unsigned t = tie; t; t &= t - 1u) {
                const int q = __ffs(t) - 1;
                const uint32_t lo = (uint32_t)list[lane + 32 * q];
                if (lo >= best) {
                    best = lo;
                    bq = q;
                }
            }
            const uint32_t all = __reduce_max_sync(kFull, tie ? best : 0u);
            const unsigned bal = __ballot_sync(kFull, tie && best == all);
            if (bal == 0u) break;   // (positions are distinct: never expected)
            if (lane == __ffs(bal) - 1) {
                win |= 1u << bq;
                tie &= ~(1u << bq);
            }
            --need;
        }
    }
    int base = 0;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const unsigned bal = __ballot_sync(kFull, (win >> q) & 1u);
        if ((win >> q) & 1u) put(base + __popc(bal & lt), list[lane + 32 * q]);
        base += __popc(bal);
    }
}

// Inclusive scan over the warp.
__device__ __forceinline__ int warp_scan(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(kFull, v, off);
        if (lane >= off) v += y;
    }
    return v;
}

// Both axes' candidate lists (see load_lists; counts cnt and segments seg of
// axis 0, then of axis 1) into list0 and list1, in position order; returns
// whether both fit kWCap, their lengths in c.  Two rounds of 32 segments, a
// lane each, of both axes are taken together, with the loads of their counts
// and then of their first four entries in flight at once.
__device__ __forceinline__ bool warp_load_lists(const uint32_t *cnt, const u64 *seg, int G,
                                                u64 *list0, u64 *list1, int (&c)[2]) {
    const int lane = threadIdx.x & 31;
    int total = 0;   // both lists' lengths, 16 bits each
    for (int g0 = 0; g0 < G; g0 += 64) {
        uint32_t n[2][2];
        ulonglong2 e01[2][2], e23[2][2];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int g = g0 + 32 * u + lane;
                n[u][s] = g < G ? min(__ldcs(cnt + s * G + g), (uint32_t)kSeg) : 0u;
            }
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const ulonglong2 *src = reinterpret_cast<const ulonglong2 *>(
                    seg + (int64_t)(s * G + g0 + 32 * u + lane) * kSeg);
                if (n[u][s] > 0) e01[u][s] = __ldcs(src);
                if (n[u][s] > 2) e23[u][s] = __ldcs(src + 1);
            }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int both = (int)(n[u][0] | n[u][1] << 16);
            const int incl = warp_scan(both);
            const int before = total + incl - both;
            total += __shfl_sync(kFull, incl, 31);
            if ((total & 0xffff) > kWCap || (total >> 16) > kWCap) return false;   // uniform
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                u64 *dst = (s ? list1 : list0) + (s ? before >> 16 : before & 0xffff);
                const uint32_t m = n[u][s];
                if (m > 0) dst[0] = e01[u][s].x;
                if (m > 1) dst[1] = e01[u][s].y;
                if (m > 2) dst[2] = e23[u][s].x;
                if (m > 3) dst[3] = e23[u][s].y;
                const u64 *src = seg + (int64_t)(s * G + g0 + 32 * u + lane) * kSeg;
                for (uint32_t f = 4; f < m; ++f) dst[f] = __ldcs(src + f);
            }
        }
    }
    c[0] = total & 0xffff;
    c[1] = total >> 16;
    return true;
}

// One axis' candidates from every key (K % 4 == 0): those at or above a
// bound that at least kk keys reach, into list (in no order); returns their
// number, or -1 when it is larger than kWCap.
__device__ __forceinline__ int warp_scan_keys(const uint32_t *A, int K, int kk, u64 *list) {
    const int lane = threadIdx.x & 31;
    const uint4 *A4 = reinterpret_cast<const uint4 *>(A);
    const int nv = K >> 2, its = (nv + 31) >> 5;
    uint32_t gm[kWParts];
#pragma unroll
    for (int q = 0; q < kWParts; ++q) {
        uint32_t mx = 0u;
        const int hi = its * (q + 1) / kWParts;
#pragma unroll 4
        for (int t = its * q / kWParts; t < hi; ++t) {
            const int i = t * 32 + lane;
            const uint4 v = i < nv ? __ldcg(A4 + i) : make_uint4(0u, 0u, 0u, 0u);
            mx = max(mx, max(max(v.x, v.y), max(v.z, v.w)));
        }
        gm[q] = mx;
    }
    int groups = 0;
#pragma unroll
    for (int q = 0; q < kWParts; ++q) groups += gm[q] != 0u;
    groups = (int)__reduce_add_sync(kFull, groups);
    int cnt;
    if (groups < kk) return -1;
    const uint32_t tau = warp_kth<kWParts>(gm, groups, kk, &cnt);
    int total = 0;
    for (int t0 = 0; t0 < its; t0 += 32) {   // 4096 keys: four masks of 8 rounds
        uint32_t hit[4];
        int mine = 0;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            uint32_t m = 0u;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = (t0 + 8 * w + u) * 32 + lane;
                if (i < nv) {
                    const uint4 v = __ldcg(A4 + i);
                    m |= (uint32_t)(v.x >= tau) << (4 * u) | (uint32_t)(v.y >= tau) << (4 * u + 1) |
                         (uint32_t)(v.z >= tau) << (4 * u + 2) |
                         (uint32_t)(v.w >= tau) << (4 * u + 3);
                }
            }
            hit[w] = m;
            mine += __popc(m);
        }
        const int incl = warp_scan(mine);
        int at = total + incl - mine;
        total += __shfl_sync(kFull, incl, 31);
        if (total > kWCap) return -1;   // uniform
#pragma unroll
        for (int w = 0; w < 4; ++w)
            for (uint32_t m = hit[w]; m; m &= m - 1u) {
                const int bt = __ffs(m) - 1;
                const int i = 4 * ((t0 + 8 * w + (bt >> 2)) * 32 + lane) + (bt & 3);
                list[at++] = comp_of(A[i], (uint32_t)i);
            }
    }
    return total;
}

// The k <= 64 positions of sel in increasing order.
__device__ __forceinline__ void warp_sort_positions(int *sel, int k) {
    const int lane = threadIdx.x & 31;
    uint32_t x0 = 2 * lane < k ? (uint32_t)sel[2 * lane] : 0xffffffffu;
    uint32_t x1 = 2 * lane + 1 < k ? (uint32_t)sel[2 * lane + 1] : 0xffffffffu;
#pragma unroll
    for (int blk = 2; blk <= 64; blk <<= 1)
#pragma unroll
        for (int st = blk >> 1; st > 0; st >>= 1) {
            const bool up = ((2 * lane) & blk) == 0;   // ascending block
            if (st == 1) {
                const uint32_t a = min(x0, x1), b = max(x0, x1);
                x0 = up ? a : b;
                x1 = up ? b : a;
            } else {
                const uint32_t o0 = __shfl_xor_sync(kFull, x0, st >> 1);
                const uint32_t o1 = __shfl_xor_sync(kFull, x1, st >> 1);
                const bool lo = (((2 * lane) & st) == 0) == up;
                x0 = lo ? min(x0, o0) : max(x0, o0);
                x1 = lo ? min(x1, o1) : max(x1, o1);
            }
        }
    __syncwarp();   // every position has been read
    if (2 * lane < k) sel[2 * lane] = (int)x0;
    if (2 * lane + 1 < k) sel[2 * lane + 1] = (int)x1;
    __syncwarp();
}

// A warp's shared memory.  R: row pairs, [k / 2][RM][2] (row 2 t + e's entry
// b at t 2 RM + 2 b + e); srow and scol [k][RM], S_row and S_col; entries past
// the rank are 0.
struct WarpSel {
    u64 *list[2];   // [kWCap] each; the final candidates (kWTop) use both
    u64 *top;       // [kWMaxK] the top m; before it, the final candidates' places
    float *q;       // [2][D_k]
    int *sel[2];    // [kWMaxK] survivors by increasing position
    float *R, *srow, *scol;   // scol right behind srow
};
static_assert(kWTop <= 2 * kWCap, "the final candidates fit the axes' lists");

constexpr int kWTopWords = kWMaxK > kWTop / 4 ? kWMaxK : kWTop / 4;   // of 8 bytes
__host__ __device__ inline size_t warp_sel_bytes(const Dims &d, int rm) {
    return 8 * (2 * kWCap + kWTopWords) + 4 * (2 * (size_t)d.d_k + 2 * kWMaxK) +
           4 * (size_t)kWMaxK * rm * 3;
}
__device__ __forceinline__ WarpSel carve_warp(const Dims &d, int rm, unsigned char *base) {
    WarpSel W;
    W.list[0] = reinterpret_cast<u64 *>(base);
    W.list[1] = W.list[0] + kWCap;
    W.top = W.list[1] + kWCap;
    W.R = reinterpret_cast<float *>(W.top + kWTopWords);
    W.srow = W.R + kWMaxK * rm;
    W.scol = W.srow + kWMaxK * rm;
    W.q = W.scol + kWMaxK * rm;
    W.sel[0] = reinterpret_cast<int *>(W.q + 2 * d.d_k);
    W.sel[1] = W.sel[0] + kWMaxK;
    return W;
}

// Lanes per survivor (2^lg), as in axis_survivors.
__device__ __forceinline__ int survivor_lanes_log2(int k) {
    int lg = 0;
    while (lg < 5 && 2 * k * (2 << lg) <= kThreads) ++lg;
    return lg;
}

// The row of survivor sv (rows 0 .. k - 1, then columns) in the key tables.
__device__ __forceinline__ const uint4 *warp_row(const Dims &d, const Ptrs &p, int h, int sv,
                                                 int *sel) {
    const int s = sv >= d.k;
    uint32_t pos = 0u;
    if (sv < 2 * d.k) {
        int *at = sel + (s ? kWMaxK + sv - d.k : sv);
        pos = (uint32_t)*at;
        if (pos >= (uint32_t)d.K) {   // never expected: record and skip
            atomicOr(p.err, kErrInternal);
            pos = 0u;
            *at = 0;
        }
    }
    const __nv_bfloat16 *keys = static_cast<const __nv_bfloat16 *>(s ? p.k_col : p.k_row);
    return reinterpret_cast<const uint4 *>(keys + ((int64_t)h * d.K + pos) * d.d_k);
}

// R = S_row^T C of the row survivors, from the chunk scores (rows' in scol's
// and srow's place beside it, see WarpSel); returns whether R and S_col are
// finite.  Row pairs past the last one, up to a multiple of kWParts, repeat
// it, and so does the missing second row of an odd k.
template <int RM>
__device__ __forceinline__ bool warp_fold_rows(const Dims &d, const float *core, const WarpSel &W) {
    const int lane = threadIdx.x & 31, k = d.k, r = d.r;
    const int np = (k + 1) >> 1, npad = (np + kWParts - 1) / kWParts * kWParts;
    bool fin = true;
    for (int i = lane; i < 2 * npad; i += 32) {
        const int sv = min(i < 2 * np ? i : 2 * np - 2 + (i & 1), k - 1);
        float S[RM];
#pragma unroll
        for (int a = 0; a < RM; ++a) {
            S[a] = W.srow[sv * RM + a];
            if (i < k) fin = fin && fabsf(W.scol[i * RM + a]) < INFINITY;
        }
#pragma unroll
        for (int b = 0; b < RM; ++b) {
            float v = 0.f;
            if (b < r)
#pragma unroll
                for (int a = 0; a < RM; ++a)
                    if (a < r) v = fmaf(S[a], core[a * r + b], v);
            W.R[((i >> 1) * RM + b) * 2 + (i & 1)] = v;
            fin = fin && fabsf(v) < INFINITY;
        }
    }
    return __all_sync(kFull, fin);
}

// The query's place in W.q for the chunk scores below: vectors u and u + 1
// (u even) of a lane interleaved, so that a 16-byte read gives two elements
// of each.
__device__ __forceinline__ int paired_q(int c, int lg) {
    const int iv = c >> 3, u = iv >> lg, sub = iv & ((1 << lg) - 1);
    return ((((u >> 1) << lg) + sub) << 4) + 2 * (c & 7) + (u & 1);
}

// The 2k survivors' chunk scores (bf16 rows of whole 16-byte vectors): G
// lanes per survivor and the order of the sums as in axis_survivors.  A lane
// takes NV vectors of its row, NV / CH of each of the CH chunks, two at a
// time (packed fp32; the sums of the two stay apart), and asks for the next
// survivor's vector as soon as it has used one, so that NV loads a lane stay
// in flight.  The scores go to srow [2 kWMaxK][RM] (scol is its second
// half), zeros past the rank.
template <int RM, int NV, int lg, int CH>
__device__ __forceinline__ void warp_survivors(const Dims &d, const Ptrs &p, int h,
                                               const WarpSel &W) {
    constexpr int G = 1 << lg, per = 32 >> lg;
    const int lane = threadIdx.x & 31, sub = lane & (G - 1);
    const int n = 2 * d.k;
    int sv = lane >> lg;
    const uint4 *row = warp_row(d, p, h, sv, W.sel[0]) + sub;
    const uint64_t pol = key_row_policy();
    uint4 buf[NV];
#pragma unroll
    for (int u = 0; u < NV; ++u) buf[u] = ld_key_row(row + (u << lg), pol);
#pragma unroll 1
    for (int s0 = 0; s0 < n; s0 += per, sv += per) {
        const bool more = s0 + per < n;   // uniform
        row = warp_row(d, p, h, sv + per, W.sel[0]) + sub;   // (its first row past the last)
        const float *q = W.q + (sv >= d.k && sv < n ? d.d_k : 0) + (sub << 4);
        float S[RM];
#pragma unroll
        for (int a = 0; a < RM; ++a) S[a] = 0.f;
        // NC vector pairs at a time: their chains of sums interleave
        constexpr int NC = NV >= 4 ? 2 : 1;
#pragma unroll
        for (int u0 = 0; u0 < NV; u0 += 2 * NC) {
            u64 pv[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) pv[c] = 0ull;   // (0, 0)
#pragma unroll
            for (int w = 0; w < 4; ++w)   // elements 2 w and 2 w + 1 of the vectors
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const int u = u0 + 2 * c;
                    const uint32_t x = (&buf[u].x)[w], y = (&buf[u + 1].x)[w];
                    const ulonglong2 q2 = *reinterpret_cast<const ulonglong2 *>(
                        q + ((u >> 1) << (lg + 4)) + 4 * w);
                    pv[c] = fma2(pack2(__uint_as_float(x << 16), __uint_as_float(y << 16)), q2.x,
                                 pv[c]);
                    pv[c] = fma2(pack2(__uint_as_float(x & 0xffff0000u),
                                       __uint_as_float(y & 0xffff0000u)),
                                 q2.y, pv[c]);
                }
#pragma unroll
            for (int u = u0; u < u0 + 2 * NC; ++u) ld_key_row_if(buf[u], row + (u << lg), pol, more);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int u = u0 + 2 * c;
                const float2 v = unpack2(pv[c]);
                S[u * CH / NV] += v.x;
                S[(u + 1) * CH / NV] += v.y;
            }
        }
#pragma unroll
        for (int a = 0; a < CH; ++a)
            for (int off = G >> 1; off > 0; off >>= 1) S[a] += __shfl_xor_sync(kFull, S[a], off);
        if (sub == 0 && sv < n) {
            float *dst = W.srow + (sv < d.k ? sv : kWMaxK + sv - d.k) * RM;
#pragma unroll
            for (int a = 0; a < RM; ++a) dst[a] = S[a];
        }
    }
}

// The same for any number of vectors and chunks (the query in plain order).
template <int RM>
__device__ __noinline__ void warp_survivors_any(const Dims &d, const Ptrs &p, int h, int lg,
                                                const WarpSel &W) {
    const int lane = threadIdx.x & 31, G = 1 << lg, sub = lane & (G - 1), per = 32 >> lg;
    const int n = 2 * d.k, nvec = d.d_k >> 3;
    const float inv_dk = 1.f / (float)d.dk;   // see axis_survivors
#pragma unroll 1
    for (int s0 = 0; s0 < n; s0 += per) {
        const int sv = s0 + (lane >> lg);
        const uint4 *row = warp_row(d, p, h, sv, W.sel[0]);
        const float *q = W.q + (sv >= d.k && sv < n ? d.d_k : 0);
        float S[RM];
#pragma unroll
        for (int a = 0; a < RM; ++a) S[a] = 0.f;
#pragma unroll 2
        for (int iv = sub; iv < nvec; iv += G) {
            float f[8];
            unpack16<__nv_bfloat16>(ld_key_row(row + iv), f);
            float pv = 0.f;
#pragma unroll
            for (int e = 0; e < 8; ++e) pv = fmaf(f[e], q[iv * 8 + e], pv);
            const int al = (int)(((float)(iv * 8) + 0.5f) * inv_dk);
#pragma unroll
            for (int a = 0; a < RM; ++a) S[a] += a == al ? pv : 0.f;
        }
#pragma unroll
        for (int a = 0; a < RM; ++a)
            for (int off = G >> 1; off > 0; off >>= 1) S[a] += __shfl_xor_sync(kFull, S[a], off);
        if (sub == 0 && sv < n) {
            float *dst = W.srow + (sv < d.k ? sv : kWMaxK + sv - d.k) * RM;
#pragma unroll
            for (int a = 0; a < RM; ++a) dst[a] = S[a];
        }
    }
}

// RM >= r: 2 or 4 (PKM: 2).  Returns false when the (token, head) is left to
// select_block.
template <int RM, bool PKM, bool LISTS>
__device__ __forceinline__ bool select_warp(const Dims &d, const Ptrs &p, int bh,
                                            const WarpSel &W) {
    const int lane = threadIdx.x & 31;
    const int b = bh / d.H, h = bh - b * d.H;
    const int k = d.k, m = d.m, K = d.K, D = d.d_k;
    // the vectors a lane takes of a survivor's row, when they split evenly
    // over the G lanes and the chunks (else 0)
    constexpr int CH = PKM ? 1 : RM;
    const int lg = survivor_lanes_log2(k);
    int nv = D >> (3 + lg);
    if (nv << (3 + lg) != D || d.r != CH || nv % CH || (nv & 1)) nv = 0;
    const bool paired = (nv == 8 && lg == 1) || (nv == 4 && (lg == 1 || lg == 2)) ||
                        (nv == 2 && CH <= 2 && (lg == 2 || lg == 3));
    // the row and column query of this (token, head)
    const int HD = d.H * D;
    for (int e = 4 * lane; e < 2 * D; e += 128) {
        const int axis = e >= D, c = e - axis * D;
        const int a = (axis == 1 && d.A == 2) ? 1 : 0;
        const float4 v = *reinterpret_cast<const float4 *>(
            p.q_part + ((int64_t)a * d.B + b) * HD + h * D + c);
        if (paired) {
            float *dst = W.q + axis * D + paired_q(c, lg);
            dst[0] = v.x;
            dst[2] = v.y;
            dst[4] = v.z;
            dst[6] = v.w;
        } else {
            *reinterpret_cast<float4 *>(W.q + e) = v;
        }
    }
    // Eq. 8-9: the top k of each axis
    int c[2];
    const int64_t li = (int64_t)bh * 2;
    if (LISTS) {
        if (!warp_load_lists(p.gstat + li * d.n_segs, p.cand + li * d.n_segs * kSeg, d.n_segs,
                             W.list[0], W.list[1], c))
            return false;
    } else {
        for (int s = 0; s < 2; ++s)
            c[s] = warp_scan_keys(p.akey + (li + s) * K, K, k, W.list[s]);
    }
    if (c[0] < k || c[1] < k) return false;   // uniform
    __syncwarp();
#pragma unroll 1
    for (int s = 0; s < 2; ++s) {
        int *sel = W.sel[0] + s * kWMaxK;
        const u64 *list = W.list[0] + s * kWCap;
        auto put = [&](int i, u64 x) { sel[i] = (int)pos_of(x); };
        const int n = s ? c[1] : c[0];
        if (n <= 96) warp_top<3>(list, n, k, put);
        else warp_top<kWCap / 32>(list, n, k, put);
        __syncwarp();
        if (!LISTS) warp_sort_positions(sel, k);
    }
    // the survivors' chunk scores (Eq. 4)
    const float *core = p.core + (int64_t)h * d.r * d.r;
    // (NV, lg) at compile time, so that the loads' offsets are immediates
    if (paired && nv == 8) warp_survivors<RM, 8, 1, CH>(d, p, h, W);
    else if (paired && nv == 4 && lg == 2) warp_survivors<RM, 4, 2, CH>(d, p, h, W);
    else if (paired && nv == 4 && lg == 1) warp_survivors<RM, 4, 1, CH>(d, p, h, W);
    else if (paired)   // 8 or 4 lanes, RM = 2
        lg == 3 ? warp_survivors<RM, 2, 3, (CH <= 2 ? CH : 1)>(d, p, h, W)
                : warp_survivors<RM, 2, 2, (CH <= 2 ? CH : 1)>(d, p, h, W);
    else warp_survivors_any<RM>(d, p, h, lg, W);
    __syncwarp();
    if (!warp_fold_rows<RM>(d, core, W)) return false;
    __syncwarp();

    // Eq. 10 on the k x k pairs, twice.  Lane l holds columns l and l + 32
    // (a missing second column repeats the first, which changes no maximum).
    const bool col0 = lane < k, col1 = lane + 32 < k;
    const bool wide = k > 32;   // uniform
    u64 sc[RM][2];
#pragma unroll
    for (int be = 0; be < RM; ++be) {
        const float v0 = W.scol[(col0 ? lane : 0) * RM + be];
        const float v1 = col1 ? W.scol[(lane + 32) * RM + be] : v0;
        sc[be][0] = pack2(v0, v0);
        sc[be][1] = pack2(v1, v1);
    }
    auto scores = [&](int t, u64 (&g)[2]) {   // rows 2 t, 2 t + 1 of both columns
        u64 ra[RM];
#pragma unroll
        for (int be = 0; be < RM; be += 2) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(W.R + (t * RM + be) * 2);
            ra[be] = v.x;
            ra[be + 1] = v.y;
        }
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
            if (PKM) {
                g[cc] = add2(ra[0], sc[0][cc]);
            } else {
                g[cc] = mul2(ra[0], sc[0][cc]);
#pragma unroll
                for (int be = 1; be < RM; ++be) g[cc] = fma2(ra[be], sc[be][cc], g[cc]);
            }
        }
    };
    // Part q of a lane is the row pairs [q tp, (q + 1) tp), tp <= 4 (past the
    // last one, repeats of it: they count in the last real part only).
    const int np = (k + 1) >> 1, tp = (np + kWParts - 1) / kWParts;
    uint32_t gk[kWParts];
    bool fin = true;
    {
        float gm[kWParts];
#pragma unroll
        for (int q = 0; q < kWParts; ++q) gm[q] = -INFINITY;
#pragma unroll 1
        for (int j = 0; j < tp; ++j) {
#pragma unroll
            for (int q = 0; q < kWParts; ++q) {
                u64 g[2];
                scores(q * tp + j, g);
                const float2 x = unpack2(g[0]), y = unpack2(g[1]);
                gm[q] = fmaxf(gm[q], fmaxf(x.x, x.y));
                if (wide) gm[q] = fmaxf(gm[q], fmaxf(y.x, y.y));
            }
        }
#pragma unroll
        for (int q = 0; q < kWParts; ++q) {
            const bool real = col0 && q * tp < np;
            fin = fin && fabsf(gm[q]) < INFINITY;
            gk[q] = real ? f2ord(gm[q]) : 0u;
        }
    }
    if (!__all_sync(kFull, fin)) return false;   // an overflowed product
    const int groups = min(k, 32) * ((np + tp - 1) / tp);
    int cnt;
    const bool all = groups < m;   // (small k) every pair is a candidate
    const float tau = all ? 0.f : ord2f(warp_kth<kWParts>(gk, groups, m, &cnt, m >> 3));
    // masks of the pairs >= tau: a score below it leaves a sign bit in
    // g - tau (0 - tau turns a zero bound positive, so that -0 and +0 tie).
    // Part q's mask holds tp row pairs of 4 pairs (rows 2 t, 2 t + 1 of
    // column 0, then of column 1), the last one pushed in the low bits.
    const u64 nt = pack2(0.f - tau, 0.f - tau);
    uint32_t below[kWParts];
#pragma unroll
    for (int q = 0; q < kWParts; ++q) below[q] = 0u;
#pragma unroll 1
    for (int j = 0; j < tp; ++j) {
#pragma unroll
        for (int q = 0; q < kWParts; ++q) {
            u64 g[2];
            scores(q * tp + j, g);
            const float2 x = unpack2(add2(g[0], nt)), y = unpack2(add2(g[1], nt));
            uint32_t m4 = below[q];
            m4 = __funnelshift_l(__float_as_uint(x.x), m4, 1);
            m4 = __funnelshift_l(__float_as_uint(x.y), m4, 1);
            m4 = __funnelshift_l(__float_as_uint(y.x), m4, 1);
            below[q] = __funnelshift_l(__float_as_uint(y.y), m4, 1);
        }
    }
    const int nb = 4 * tp;   // bits a part, <= 16
    const uint32_t cols = !col0 ? 0u : col1 ? 0xffffu : 0xccccu;   // bits 4 x + 3, + 2: column 0
    uint32_t hit[kWParts / 2];   // parts 2 w (high half) and 2 w + 1
    int mine = 0;
#pragma unroll
    for (int w = 0; w < kWParts / 2; ++w) {
        hit[w] = 0u;
#pragma unroll
        for (int z = 0; z < 2; ++z) {
            const int q = 2 * w + z, miss = max(0, min(tp, (q + 1) * tp - np));   // repeats
            uint32_t m4 = all ? 0xffffu : ~below[q];
            m4 &= cols & ((1u << nb) - 1u) & ~((1u << 4 * miss) - 1u);
            // the repeated row of an odd k: its pair's second row
            if ((k & 1) && q * tp < np && (q + 1) * tp >= np) m4 &= ~(5u << 4 * miss);
            hit[w] = hit[w] << 16 | m4;
        }
        mine += __popc(hit[w]);
    }
    const int incl = warp_scan(mine);
    const int nc = __shfl_sync(kFull, incl, 31);
    if (nc > kWTop || nc < m) return false;   // uniform
    u64 *const list = W.list[0];
    // the hits' places (lane and bit), packed, then a hit a lane: a hot column
    // has many, and its lane would work them out alone
    uint16_t *const code = reinterpret_cast<uint16_t *>(W.top);   // [kWTop]
    int at = incl - mine;
#pragma unroll
    for (int w = 0; w < kWParts / 2; ++w)
        for (uint32_t mk = hit[w]; mk; mk &= mk - 1u)
            code[at++] = (uint16_t)(lane << 7 | w << 5 | (__ffs(mk) - 1));
    __syncwarp();
#pragma unroll 1
    for (int i = lane; i < nc; i += 32) {
        const int cd = code[i], bt = cd & 31;
        // bit 4 x + 3 - e of a part: row pair tp - 1 - x, e = 2 column + row
        const int q = 2 * (cd >> 5 & 3) + (bt < 16), x = bt & 15, e = 3 - (x & 3);
        const int t = q * tp + tp - 1 - (x >> 2), z = e & 1, jj = (cd >> 7) + 32 * (e >> 1);
        const float *Rt = W.R + t * 2 * RM + z, *Sj = W.scol + jj * RM;
        float g = PKM ? Rt[0] + Sj[0] : Rt[0] * Sj[0];
        if (!PKM) {
#pragma unroll
            for (int be = 1; be < RM; ++be) g = fmaf(Rt[2 * be], Sj[be], g);
        }
        list[i] = comp_of(f2ord(g), (uint32_t)((2 * t + z) * k + jj));
    }
    __syncwarp();
    // the top m, sorted (lane l ends with ranks 2 l and 2 l + 1)
    u64 *const top = W.top;
    {
        auto put = [&](int i, u64 x) { top[i] = x; };
        if (nc <= 128) warp_top<4>(list, nc, m, put);
        else if (nc <= 224) warp_top<7>(list, nc, m, put);
        else warp_top<kWTop / 32>(list, nc, m, put);
    }
    __syncwarp();
    u64 x0 = 2 * lane < m ? top[2 * lane] : 0ull, x1 = 2 * lane + 1 < m ? top[2 * lane + 1] : 0ull;
#pragma unroll
    for (int blk = 2; blk <= 64; blk <<= 1)
#pragma unroll
        for (int st = blk >> 1; st > 0; st >>= 1) {
            const bool down = ((2 * lane) & blk) == 0;   // descending block
            if (st == 1) {
                const bool sw = (x0 < x1) == down;
                const u64 a = sw ? x1 : x0, z = sw ? x0 : x1;
                x0 = a;
                x1 = z;
            } else {
                const u64 o0 = __shfl_xor_sync(kFull, x0, st >> 1);
                const u64 o1 = __shfl_xor_sync(kFull, x1, st >> 1);
                const bool big = (((2 * lane) & st) == 0) == down;
                x0 = (x0 > o0) == big ? x0 : o0;
                x1 = (x1 > o1) == big ? x1 : o1;
            }
        }

    // weights (raw scores, or PKM's softmax), shuffle, outputs
    float gmax = 0.f, z = 0.f;
    if (d.act == ULTRAMEM_ACT_SOFTMAX) {
        gmax = ord2f(key_of(__shfl_sync(kFull, x0, 0)));
        __syncwarp();   // top has been read
        if (2 * lane < m) top[2 * lane] = x0;
        if (2 * lane + 1 < m) top[2 * lane + 1] = x1;
        __syncwarp();
        for (int e = lane; e < m; e += 32) z += __expf(ord2f(key_of(top[e])) - gmax);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) z += __shfl_xor_sync(kFull, z, off);
    }
    const int64_t base = (int64_t)bh * m;
    const uint32_t N = (uint32_t)d.N;
    const uint32_t row_bytes = (uint32_t)d.d_v * 2u;
    const bool prefetch = (uint64_t)d.B * d.H * m * row_bytes <= kPrefetchMaxBytes;
    const float inv_k = 1.f / (float)k;   // c / k as in select_block's pairs
    // a lane's two winners together: ranks e and e + 1
    const int e = 2 * lane;
    if (e >= m) return true;
    const bool two = e + 1 < m;
    int ii[2], jj[2], prow[2], pb[2];
    int64_t v[2];
    float w[2];
#pragma unroll
    for (int z2 = 0; z2 < 2; ++z2) {
        const u64 x = z2 && two ? x1 : x0;
        const int cc = (int)pos_of(x);
        ii[z2] = (int)(((float)cc + 0.5f) * inv_k);
        jj[z2] = cc - ii[z2] * k;
        v[z2] = (int64_t)W.sel[0][ii[z2]] * K + W.sel[1][jj[z2]];
        const float g = ord2f(key_of(x));
        w[z2] = d.act == ULTRAMEM_ACT_SOFTMAX ? __expf(g - gmax) / z : g;
        const uint32_t vs = (uint32_t)shuffle_address(d, p.perm, (uint64_t)v[z2]);   // Eq. 14
        pb[z2] = (int)(vs / N);
        prow[z2] = (int)(vs - (uint32_t)pb[z2] * N);
    }
    const int64_t at0 = base + e;
    // 8-byte stores when every (token, head) starts on 8 bytes
    const bool even = two && (m & 1) == 0;
    auto put2 = [&](auto *dst, auto y0, auto y1, bool vec) {
        using Y = decltype(y0);
        struct alignas(2 * sizeof(Y)) Two {
            Y a, b;
        };
        if (vec) {
            *reinterpret_cast<Two *>(dst + at0) = Two{y0, y1};
        } else {
            dst[at0] = y0;
            if (two) dst[at0 + 1] = y1;
        }
    };
    put2(p.sel_row, prow[0], prow[1], even);
    put2(p.sel_p, pb[0], pb[1], even);
    if (p.idx_out)
        put2(p.idx_out, v[0], v[1], even && ((uintptr_t)p.idx_out & 15) == 0);
    if (d.nc == 1) {
        put2(p.sel_w, w[0], w[1], even);
        if (p.w_out) put2(p.w_out, w[0], w[1], even && ((uintptr_t)p.w_out & 7) == 0);
    } else {
        const int r = d.r;
#pragma unroll
        for (int z2 = 0; z2 < 2; ++z2) {
            if (z2 && !two) break;
            for (int ci = 0; ci < d.nc; ++ci) {   // Eq. 16-17, as in select_block
                const float *Cc = p.cores + ((int64_t)h * d.nc + ci) * r * r;
                float gi = 0.f;
#pragma unroll
                for (int a = 0; a < RM; ++a) {
                    if (a < r) {
                        float cs = 0.f;
#pragma unroll
                        for (int be = 0; be < RM; ++be)
                            if (be < r) cs = fmaf(Cc[a * r + be], W.scol[jj[z2] * RM + be], cs);
                        gi = fmaf(W.srow[ii[z2] * RM + a], cs, gi);
                    }
                }
                p.sel_w[(at0 + z2) * d.nc + ci] = gi;
                if (p.w_out) p.w_out[(at0 + z2) * d.nc + ci] = gi;
            }
        }
    }
    if (prefetch) {   // the gather reads these rows next
        const unsigned char *V = static_cast<const unsigned char *>(p.values);
        prefetch_l2(V + (size_t)prow[0] * row_bytes, row_bytes);
        if (two) prefetch_l2(V + (size_t)prow[1] * row_bytes, row_bytes);
    }
    return true;
}

// A (token, head) whose query is zero (a padding token: all its scores tie, which
// overflows a warp's lists).  Every score that is a number is then zero, so by
// address the slots are the first row with the first m <= k columns (of the axes'
// candidates, or of all keys when each scores zero); false, nothing written,
// where a factor that is not finite may make other ones.  One warp.  Retrievals
// of zero tokens, a block per (token, head) -> the block's search for a CTA's
// eight one by one -> this: decode_1m with 800 tokens 337 -> 619 -> 43 us, mid_4m
// with 512 270 -> 615 -> 72, with 4096 4153 -> 5776 -> 1723 (the list passes, which
// write every key).
template <bool LISTS>
__device__ __noinline__ bool select_zero_query(const Dims &d, const Ptrs &p, int bh, int *sel) {
    const int lane = threadIdx.x & 31, m = d.m, K = d.K, G = d.n_segs;
    const int b = bh / d.H, h = bh - b * d.H, HD = d.H * d.d_k;
    bool nz = false;
    for (int e = lane; e < 2 * d.d_k; e += 32) {
        const int axis = e >= d.d_k, a = axis && d.A == 2;
        nz = nz || p.q_part[((int64_t)a * d.B + b) * HD + h * d.d_k + e - axis * d.d_k] != 0.f;
    }
    if (__any_sync(kFull, nz)) return false;
    const uint32_t zero = f2ord(0.f);
    bool ok = true;
    const int rr = d.r * d.r, ncrr = d.nc > 1 ? d.nc * rr : 0;
    for (int e = lane; e < rr; e += 32) ok = ok && fabsf(p.core[(int64_t)h * rr + e]) < INFINITY;
    for (int e = lane; e < ncrr; e += 32)
        ok = ok && fabsf(p.cores[(int64_t)h * ncrr + e]) < INFINITY;
    if (!__all_sync(kFull, ok)) return false;
    for (int s = 0; s < 2; ++s) {
        const int64_t li = (int64_t)bh * 2 + s;
        const int need = s ? m : 1;   // positions of the axis that are used
        int *at = sel + s * kWMaxK;
        if constexpr (LISTS) {
            const uint32_t *cnt = p.gstat + li * G;
            const u64 *seg = p.cand + li * G * kSeg;
            int c = 0;
            for (int g = lane; g < G; g += 32) c += (int)min(__ldcg(cnt + g), (uint32_t)kSeg);
            if ((int)__reduce_add_sync(kFull, c) < d.k) return false;
            for (int g = 0, got = 0; got < need; ++g) {   // (ends: k >= need are listed)
                const int n = (int)min(__ldcg(cnt + g), (uint32_t)kSeg);
                for (int e = lane; e < n && got + e < need; e += 32) {
                    const u64 x = __ldcg(seg + (int64_t)g * kSeg + e);
                    at[got + e] = (int)pos_of(x);
                    ok = ok && key_of(x) == zero;
                }
                got += n;
            }
        } else {
            const uint4 *A = reinterpret_cast<const uint4 *>(p.akey + li * K);
#pragma unroll 4
            for (int i = lane; i < K >> 2; i += 32) {
                const uint4 v = __ldcg(A + i);
                ok = ok && v.x == zero && v.y == zero && v.z == zero && v.w == zero;
            }
            for (int e = lane; e < need; e += 32) at[e] = e;
        }
    }
    if (!__all_sync(kFull, ok)) return false;
    __syncwarp();
    const uint32_t N = (uint32_t)d.N;
    const float w = d.act == ULTRAMEM_ACT_SOFTMAX ? 1.f / (float)m : 0.f;
    for (int e = lane; e < m; e += 32) {
        const int64_t o = (int64_t)bh * m + e, v = (int64_t)sel[0] * K + sel[kWMaxK + e];
        const uint32_t vs = (uint32_t)shuffle_address(d, p.perm, (uint64_t)v);   // Eq. 14
        p.sel_p[o] = (int)(vs / N);
        p.sel_row[o] = (int)(vs % N);
        if (p.idx_out) p.idx_out[o] = v;
        for (int ci = 0; ci < d.nc; ++ci) {
            p.sel_w[o * d.nc + ci] = w;
            if (p.w_out) p.w_out[o * d.nc + ci] = w;
        }
    }
    return true;
}

// A (token, head) that its warp left to the block.
template <int RM>
__device__ __noinline__ void select_left(const Dims &d, const Ptrs &p, int bh,
                                         unsigned char *smem) {
    SelShared &sh = *reinterpret_cast<SelShared *>(smem);
    select_block<__nv_bfloat16, 4, (RM > 2 ? kMaxR : 2), false, false>(
        d, p, bh, smem + sizeof(SelShared), sh);
}

// The CTA's warps in `left`, without those of zero queries, which they settle.
// Whole block.  (Out of line, and before the loop over the rest: the kernel's own
// code then stays as fast; with the call inside the loop, or the loop inside it,
// retrievals with lists took 1 to 2 % longer.)
template <int RM, bool LISTS>
__device__ __noinline__ unsigned select_zeros(const Dims &d, const Ptrs &p, unsigned left,
                                              unsigned char *smem) {
    __shared__ unsigned again;
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) again = 0u;
    __syncthreads();
    if ((left >> warp & 1u) &&
        !select_zero_query<LISTS>(d, p, (int)blockIdx.x * kWarps + warp,
                                  reinterpret_cast<int *>(smem) + warp * 2 * kWMaxK) &&
        (threadIdx.x & 31) == 0)
        atomicOr(&again, 1u << warp);
    __syncthreads();
    return again;
}

template <int RM, bool PKM, bool LISTS>
__global__ void __launch_bounds__(kThreads, 4) select_warp_kernel(Dims d, Ptrs p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned left;
    const int warp = threadIdx.x >> 5;
    const int bh = (int)blockIdx.x * kWarps + warp;
    if (threadIdx.x == 0) left = 0u;
    __syncthreads();
    pdl_wait();
    stamp_begin(p.stamp);
    pdl_trigger();
    if (bh < d.B * d.H) {   // warp-uniform
        const WarpSel W = carve_warp(d, RM, smem_raw + warp * warp_sel_bytes(d, RM));
        if (!select_warp<RM, PKM, LISTS>(d, p, bh, W) && (threadIdx.x & 31) == 0)
            atomicOr(&left, 1u << warp);
    }
    __syncthreads();
    for (unsigned t = left ? select_zeros<RM, LISTS>(d, p, left, smem_raw) : 0u; t;
         t &= t - 1u) {   // uniform
        select_left<RM>(d, p, (int)blockIdx.x * kWarps + __ffs(t) - 1, smem_raw);
        __syncthreads();
    }
    stamp_end(p.stamp);
}


// Candidate lists (Dims::cand), between the two scoring passes: the bound of
// one (token, head, axis) per warp.  tau is the largest T whose low 16 bits
// are zero with at least k of the axis' G group maxima (groups of 16 keys)
// >= T, found bit by bit from the top: k distinct groups hold a key >= tau,
// so the axis' top k is among the keys >= tau.  tau is at most the k-th
// largest group maximum and agrees with it in the sign, the exponent and
// the first 7 mantissa bits of the score; the low bits would tighten the
// lists by a few keys for twice the rounds.
constexpr int kBoundWarps = 8;
constexpr int kMaxGroupsPerLane = 32;   // G <= 1024 groups (K <= 16384 keys)
static_assert(32 * kMaxGroupsPerLane == 4 * kMaxSegPerThread * kThreads, "one limit on K");
template <int NQ>   // group maxima a lane holds, 32 NQ >= G
__global__ void __launch_bounds__(32 * kBoundWarps) cand_bound_kernel(Dims d, Ptrs p) {
    pdl_wait();
    stamp_begin(p.stamp);
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const int64_t w = (int64_t)blockIdx.x * kBoundWarps + (threadIdx.x >> 5);
    if (w < (int64_t)d.B * d.H * 2) {   // warp-uniform
        const int G = d.n_groups;
        const uint32_t *g = p.gstat + w * G;
        uint32_t v[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int e = lane + 32 * q;
            v[q] = e < G ? g[e] : 0u;   // 0: below every score's key
        }
        uint32_t T = 0u;
#pragma unroll 4
        for (int bit = 31; bit >= 16; --bit) {
            const uint32_t c = T | (1u << bit);
            int n = 0;
#pragma unroll
            for (int q = 0; q < NQ; ++q) n += v[q] >= c;
            if (__reduce_add_sync(kFull, n) >= d.k) T = c;
        }
        if (lane == 0) p.tau[w] = T;
    }
    stamp_end(p.stamp);
}

// lookup_reduce input: given virtual addresses and weights -> (row, p, w).
// An address outside [0, E*N) is recorded in the error word and skipped
// (weights 0, row 0).  With MCS each slot has nc weights.
__global__ void slots_kernel(Dims d, Ptrs p) {
    const int64_t total = (int64_t)d.B * d.H * d.m;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        int row, blk;
        const bool ok = slot_of_address(d, p, p.idx_in[e], row, blk);
        for (int ci = 0; ci < d.nc; ++ci)
            p.sel_w[e * d.nc + ci] = ok ? p.w_in[e * d.nc + ci] : 0.f;
        p.sel_row[e] = row;
        p.sel_p[e] = blk;
    }
}

}  // namespace

size_t select_smem_bytes(const Dims &d) { return sel_offsets(d).total; }

// One warp per (token, head): bf16 rows of whole 16-byte vectors and chunks,
// rank up to 4, k up to 64 and m <= k (the group maxima then bound the top m
// well), the candidate lists or at least 1024 keys an axis, and enough
// (token, head)s: a warp alone takes about 30 us for one whatever the grid
// (35 with every key), the blocks longer grids.  Measured on GB300, a
// retrieval, blocks -> warps: with the lists 64.5 -> 69.9 us at 800 (mid_4m,
// 200 tokens), 62.4 -> 65.8 and 80.7 -> 77.4 at 1024 (K = 4096 and 5000),
// 103.0 -> 100.4 at 1600 (the lists forced there; where the scoring takes them by
// itself just over 1000 (1024, 1040 at K = 9000), K = 8600, 9000, 16000 and 16000 with 4, 2, 4 and 2 heads,
// 79.8 -> 70.7, 74.3 -> 66.4, 91.5 -> 84.7 and 89.8 -> 82.5); with every key (K =
// 2048) 42.4 -> 49.2 at 1000, 82.0 -> 69.2 at 2000.
constexpr int64_t kWarpGridLists = 1000, kWarpGridKeys = 1500;
static bool warp_select_fits(const Dims &d, const Ptrs &p) {
    return d.dtype == ULTRAMEM_BF16 && d.r <= 4 && d.k <= kWMaxK && d.m <= d.k &&
           d.d_k <= kWMaxD && d.dk % 8 == 0 &&
           (((uintptr_t)p.k_row | (uintptr_t)p.k_col) & 15) == 0 &&
           (d.cand || (d.K % 4 == 0 && d.K >= 1024)) &&
           (int64_t)d.B * d.H > (d.cand ? kWarpGridLists : kWarpGridKeys);
}
template <int RM, bool PKM, bool LISTS>
static cudaError_t launch_select_warp(Dims d, const Ptrs &p, cudaStream_t st) {
    // what is left to the block reads its keys from L2 (16-byte loads)
    if (!LISTS) d.stream_keys = 1;
    const size_t block = sizeof(SelShared) + select_smem_bytes(d);
    const size_t warps = kWarps * warp_sel_bytes(d, RM);
    const int grid = (int)(((int64_t)d.B * d.H + kWarps - 1) / kWarps);
    constexpr auto k = select_warp_kernel<RM, PKM, LISTS>;
    // spread over the SMs (see spread_smem): the CTAs are placed while the
    // scoring's hold most of them
    const size_t sm =
        spread_smem(block > warps ? block : warps, static_smem_of<k>(), grid);
    return launch_kernel(d.pdl, k, grid, kThreads, sm, st, d, p);
}
template <bool LISTS>
static cudaError_t launch_select_warps(const Dims &d, const Ptrs &p, cudaStream_t st) {
    if (d.pkm) return launch_select_warp<2, true, LISTS>(d, p, st);
    return d.r <= 2 ? launch_select_warp<2, false, LISTS>(d, p, st)
                    : launch_select_warp<4, false, LISTS>(d, p, st);
}

template <typename T, int RM>
static cudaError_t launch_select_t(const Dims &d, const Ptrs &p, size_t smem, cudaStream_t st) {
    if (d.B * d.H > 3 * 152 || d.cand)
        return launch_kernel(d.pdl, select_kernel<T, 4, RM>, d.B * d.H, kThreads, smem, st, d, p);
    if (d.B * d.H <= device_sm_count()) {
        // at most one (token, head) per SM: a CTA pair per (token, head), the
        // pairs spread over the SMs
        const size_t sm =
            spread_smem(smem, static_smem_of<select_kernel<T, 3, RM, true>>(), 2 * d.B * d.H);
        return launch_kernel(d.pdl, 2u, select_kernel<T, 3, RM, true>, dim3(d.B * d.H, 1, 2),
                             kThreads, sm, st, d, p);
    }
    // decode grids: spread over the SMs (see spread_smem)
    const size_t sm = spread_smem(smem, static_smem_of<select_kernel<T, 3, RM>>(), d.B * d.H);
    return launch_kernel(d.pdl, select_kernel<T, 3, RM>, d.B * d.H, kThreads, sm, st, d, p);
}

cudaError_t launch_select(const Dims &d, const Ptrs &p, cudaStream_t st) {
    if (warp_select_fits(d, p))
        return d.cand ? launch_select_warps<true>(d, p, st) : launch_select_warps<false>(d, p, st);
    const size_t smem = select_smem_bytes(d);
    if (d.dtype == ULTRAMEM_BF16)
        return d.r <= 2 ? launch_select_t<__nv_bfloat16, 2>(d, p, smem, st)
                        : launch_select_t<__nv_bfloat16, kMaxR>(d, p, smem, st);
    return d.r <= 2 ? launch_select_t<float, 2>(d, p, smem, st)
                    : launch_select_t<float, kMaxR>(d, p, smem, st);
}

cudaError_t launch_cand_bound(const Dims &d, const Ptrs &p, cudaStream_t st) {
    if (d.n_groups < d.k || d.n_groups > 32 * kMaxGroupsPerLane) return cudaErrorInvalidValue;
    const int64_t warps = (int64_t)d.B * d.H * 2;
    const int blocks = (int)((warps + kBoundWarps - 1) / kBoundWarps);
    const int nq = (d.n_groups + 31) / 32;
    auto go = [&](auto kernel) {
        return launch_kernel(d.pdl, kernel, blocks, 32 * kBoundWarps, 0, st, d, p);
    };
    if (nq <= 1) return go(cand_bound_kernel<1>);
    if (nq <= 2) return go(cand_bound_kernel<2>);
    if (nq <= 4) return go(cand_bound_kernel<4>);
    if (nq <= 8) return go(cand_bound_kernel<8>);
    if (nq <= 16) return go(cand_bound_kernel<16>);
    return go(cand_bound_kernel<kMaxGroupsPerLane>);
}

cudaError_t launch_slots_from_addresses(const Dims &d, const Ptrs &p, cudaStream_t st) {
    int64_t total = (int64_t)d.B * d.H * d.m;
    int blocks = (int)((total + 255) / 256);
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    slots_kernel<<<blocks, 256, 0, st>>>(d, p);
    return cudaGetLastError();
}

// Each selection kernel may use up to the per-CTA maximum of dynamic shared
// memory (the decode-grid one is padded to spread its CTAs; see
// spread_smem).  The limit is a process-wide attribute of the kernel, so it
// is set once to the maximum, never lowered to one layer's need.
template <typename T, int RM> static cudaError_t allow_select() {
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(
        select_kernel<T, 3, RM>, a, (int)(kSmemPerCta - static_smem_of<select_kernel<T, 3, RM>>()));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(
            select_kernel<T, 3, RM, true>, a,
            (int)(kSmemPerCta - static_smem_of<select_kernel<T, 3, RM, true>>()));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(select_kernel<T, 4, RM>, a,
                                 (int)(kSmemPerCta - static_smem_of<select_kernel<T, 4, RM>>()));
    return e;
}
template <int RM, bool PKM, bool LISTS> static cudaError_t allow_select_warp() {
    constexpr auto k = select_warp_kernel<RM, PKM, LISTS>;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(kSmemPerCta - static_smem_of<k>()));
}

cudaError_t configure_select(const Dims &) {
    cudaError_t e = allow_select<float, 2>();
    if (e == cudaSuccess) e = allow_select<float, kMaxR>();
    if (e == cudaSuccess) e = allow_select<__nv_bfloat16, 2>();
    if (e == cudaSuccess) e = allow_select<__nv_bfloat16, kMaxR>();
    if (e == cudaSuccess) e = allow_select_warp<2, true, true>();
    if (e == cudaSuccess) e = allow_select_warp<2, true, false>();
    if (e == cudaSuccess) e = allow_select_warp<2, false, true>();
    if (e == cudaSuccess) e = allow_select_warp<2, false, false>();
    if (e == cudaSuccess) e = allow_select_warp<4, false, true>();
    if (e == cudaSuccess) e = allow_select_warp<4, false, false>();
    return e;
}

}  // namespace um
