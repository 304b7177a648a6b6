// Reduced-precision list scan on the tensor cores, then an exact FP32
// re-rank (the precision pattern of the hot path; the paper scans FP32
// only).
//
// Lists keep a BF16 or an FP8 E4M3 copy of every payload row (per-list
// scale for FP8).  One persistent CTA per SM takes (list, tile of up to TN
// queries, slab chunk) items from a work counter.  The list's slabs stream
// through shared memory as 128-row A tiles (TMA 2-D loads, 128-byte
// swizzle); the query tile, rounded to the same format, is the B operand;
// tcgen05.mma accumulates the 128 x TN dot products in FP32 in tensor
// memory (all 512 columns: 8 or 16 accumulators, so the next tiles' MMAs
// overlap the epilogue of this one, and the first tiles of an item can be
// looked at for a bound before anything is appended).  The epilogue forms
// the expanded distance ||q||^2 + ||x||^2 - 2 s q.x (FP32 norms of the
// unrounded vectors, s the dequantisation scale), and every query keeps its
// best K' (= 4k) (distance, slot) candidates.  A per-query shared bound (the K'-th
// distance any item has found) prunes the rest.  A final pass recomputes
// the K' survivors' distances exactly in FP32 from the FP32 payload and
// keeps the best k by (distance, id).
//
// Roles inside the CTA, all running one item ahead of the epilogue:
//   warp 2  item contexts: takes the next item, stages its queries' norms,
//           scales and bounds, its slab ids and validity bitmaps, and
//           prefetches the first slabs into L2 (two contexts in flight);
//   warp 3  builds the rounded, swizzled query tile (two B buffers);
//   warp 0  (one lane) TMA loads of the A tiles, plus L2 prefetches of
//           the payload rows and their ||x||^2 further ahead in the list;
//   warp 1  (one lane) issues the MMAs; warp 2 also owns the TMEM;
//   warps 4.. the epilogue: three warps per TMEM lane quarter, 16 query
//           columns each (where TN has fewer blocks of columns, the quarter's
//           warps share the tiles); each thread reads its row's ||x||^2 from
//           global memory (L2) before it waits for the accumulator.
// A tile's passing rows are appended to their query's buffer, each lane its
// own, at a position taken by a shared atomic; a buffer is reduced to little
// more than its best K' (left unsorted) only after a tile that leaves it too
// full for the next one, so most tiles end on a single barrier.  Each item writes its rows' candidates unsorted with their
// count; a per-query merge makes the exact selection of the best K' of all
// its items.  Every wait is bounded, and a wait that gives up stops every
// role.
#include <cudaTypedefs.h>
#include <math.h>

#include "device_utils.cuh"
#include "kernels.cuh"
#include "tc.cuh"

namespace sivf {

constexpr int TC_M = 128;       // rows per A tile (MMA M)
constexpr int TC_NCOL = 16;     // query columns per epilogue warp
constexpr int TC_META = 256;    // slabs of one sub-item (ids and bitmaps staged together)
constexpr int TC_CTX = 2;       // item contexts in flight
constexpr int TC_MAXST = 4;     // most A-tile stages
constexpr int TC_HIST = 256;    // radix-select bins per epilogue warp
constexpr int TC_PF_BYTES = 192 * 1024;  // L2 prefetch distance per CTA

// Query tiles: 48 queries for K' <= 64 (small enough candidate buffers for
// three A stages), 32 for K' <= 128, 16 (and candidate buffers up to
// K' = 512) for deeper re-ranks.
template <int TN> struct TcShape {
    static constexpr int N = TN;                        // queries per tile (MMA N)
    // epilogue warps: three per TMEM lane quarter, also where TN has fewer
    // blocks of 16 columns (they then share the tiles); FW of them fold
    static constexpr int EW = 12;
    static constexpr int FW = 4 * (TN / TC_NCOL);
    static constexpr int EPI = EW * 32;                 // epilogue threads
    static constexpr int NT = 128 + EPI;                // + TMA, MMA, context, B warps
    static constexpr int KMAX = TN == 48 ? 64 : TN == 32 ? 128 : 512;  // deepest K'
    // TMEM columns per accumulator buffer (power of two, >= 32), and buffers:
    // all 512 columns, so that a list of 1,024 rows is looked at twice
    static constexpr int TB = TN <= 32 ? 32 : 64;
    static constexpr int NACC = 512 / TB;
};

struct TcArgs {
    const float *q;
    int64_t nq;
    int P, K, M;
    const int32_t *qlist, *loff, *lcnt, *nch;
    const int32_t *prun;  // first output run of each pair (-1: not scanned)
    const int2 *items;
    const float *qn, *qsc;
    const unsigned char *qcast;  // [nq, d] queries in the scan format (BF16), or
                                 // [nq * P, d] residuals q - c_l of each pair (E4M3)
    int per_pair;                // qn, qsc, qcast are per (query, probe) pair (FP8)
    float *part_d;
    int64_t *part_i;  // global slot (slab * C + slot) of each candidate
    int32_t *part_n;  // candidates in each run (at most RK)
    int RK;           // run length: K' plus room an approximate reduction may keep
    float *thr;
    const float *xnorm;
    const uint32_t *bits;
    const int32_t *nslabs, *dir;
    const float *inv_scale8;
    const unsigned char *pay;  // the scanned copy (BF16 or E4M3 rows)
    int64_t n_slabs, dir_cap;
    int L, d, C, KC;  // KC = 128-byte K chunks per row
    int nst;          // A-tile stages
    int pf_tiles;     // A tiles prefetched into L2 ahead of the loads
    uint64_t wait_ns; // time after which a wait of the scan gives up
    int seed_slabs;   // > 0: seed launch: the first seed_slabs slabs of each
                      // item, bounds published, no runs written
    int tile_box;     // the 128-row map is valid: a tile of consecutive slabs
                      // is one TMA box
    Ctl *ctl;
    uint32_t *err;
};

// One item context: a header, the tile's queries, the sub-item's slabs.
//   int32 hdr[16]: list, m, first slab, slabs, A tiles, row stride ME,
//                  -, chunk, flags (1 first, 2 last, 4 stop), inv scale
//   int32 qpair[TN]; float qn[TN], qsc[TN], kd0[TN]; int32 qi[TN];
//   int32 sl[TC_META]; uint32 bits[TC_META][4]
enum : int { CF_FIRST = 1, CF_LAST = 2, CF_STOP = 4 };
__host__ __device__ constexpr size_t tc_ctx_bytes(int TN)
{
    return 64 + (size_t)20 * TN + (size_t)4 * TC_META + (size_t)16 * TC_META;
}

struct TcSmem {
    size_t a, b, xn, bd, bs, ctx, hist, bars, total;
};
template <int TN>
__host__ __device__ inline TcSmem tc_smem(int KC, int M, int nst)
{
    using S = TcShape<TN>;
    TcSmem s;
    s.a = 0;                                             // nst x KC x 16 KB
    s.b = s.a + (size_t)nst * KC * TC_M * 128;           // 2 x KC x TN rows x 128 B
    s.xn = s.b + (size_t)2 * KC * TN * 128;              // (no norm ring)
    s.bd = s.xn;
    s.bs = s.bd + (size_t)TN * M * 4;
    s.ctx = s.bs + (size_t)TN * M * 4;
    s.hist = s.ctx + (size_t)TC_CTX * tc_ctx_bytes(TN);
    s.bars = s.hist + (size_t)S::FW * TC_HIST * 4;
    s.total = s.bars + 64 * 8 + 1024;                    // + base alignment slack
    return s;
}

// (distance, slot) order with pads (+inf, INT_MAX) last
__device__ __forceinline__ bool ds_less(float a, int32_t sa, float b, int32_t sb)
{
    return a < b || (a == b && sa < sb);
}

// 64-bit key with the (distance, slot) order
__device__ __forceinline__ uint64_t ds_key(float d, int32_t s)
{
    return ((uint64_t)fkey(d) << 32) | (uint32_t)s;
}

// Ascending bitonic sort of 32*E (distance, slot) pairs held E per lane.
template <int E>
__device__ __forceinline__ void warp_sort32(float (&v)[E], int32_t (&s)[E], int lane)
{
    constexpr int N = 32 * E;
#pragma unroll
    for (int size = 2; size <= N; size <<= 1)
#pragma unroll
        for (int st = size >> 1; st > 0; st >>= 1)
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int i = lane + 32 * e;
                const bool up = (i & size) == 0;
                if (st >= 32) {
                    const int pe = e ^ (st >> 5);
                    if (pe > e) {
                        const bool sw = up ? ds_less(v[pe], s[pe], v[e], s[e])
                                           : ds_less(v[e], s[e], v[pe], s[pe]);
                        if (sw) {
                            const float tv = v[e];
                            v[e] = v[pe];
                            v[pe] = tv;
                            const int32_t ts = s[e];
                            s[e] = s[pe];
                            s[pe] = ts;
                        }
                    }
                } else {
                    const float ov = __shfl_xor_sync(0xffffffffu, v[e], st);
                    const int32_t os = __shfl_xor_sync(0xffffffffu, s[e], st);
                    const bool lower = (lane & st) == 0;
                    const bool take = (lower == up) ? ds_less(ov, os, v[e], s[e])
                                                    : ds_less(v[e], s[e], ov, os);
                    if (take) {
                        v[e] = ov;
                        s[e] = os;
                    }
                }
            }
}

// Radix select over n distinct 64-bit keys key(i), i < n: returns the
// (prefix, mask) for which exactly the K smallest keys satisfy
// (key & mask) <= prefix.  Keys equal to ~0 are padding: they never count
// among the K smallest, and at least K keys are not padding.  8 bits per
// pass, starting at the highest bit where the keys differ and stopping at
// the first pass whose chosen bin is taken whole.
template <class KeyF>
__device__ __forceinline__ void warp_radix_kth(KeyF key, int n, int K, uint32_t *hist, int lane,
                                               uint64_t &prefix_out, uint64_t &mask_out)
{
    uint64_t kmin = ~0ull, kmax = 0ull;
    for (int i = lane; i < n; i += 32) {
        const uint64_t k = key(i);
        if (k != ~0ull) {
            kmin = min(kmin, k);
            kmax = max(kmax, k);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        kmin = min(kmin, (uint64_t)__shfl_xor_sync(0xffffffffu, (unsigned long long)kmin, o));
        kmax = max(kmax, (uint64_t)__shfl_xor_sync(0xffffffffu, (unsigned long long)kmax, o));
    }
    const uint64_t diff = kmin ^ kmax;
    const int top = diff ? 63 - __clzll((long long)diff) : 0;
    uint64_t mask = top >= 63 ? 0ull : ~((2ull << top) - 1ull);
    uint64_t prefix = kmin & mask;
    uint32_t need = (uint32_t)K;
    for (int hi = top; hi >= 0; hi -= 8) {
        const int shift = max(hi - 7, 0);
        const uint32_t bmask = (1u << (hi - shift + 1)) - 1u;
#pragma unroll
        for (int b = 0; b < 8; ++b) hist[lane * 8 + b] = 0u;
        __syncwarp();
        for (int i = lane; i < n; i += 32) {
            const uint64_t k = key(i);
            if (k != ~0ull && (k & mask) == prefix)
                atomicAdd(&hist[(uint32_t)(k >> shift) & bmask], 1u);
        }
        __syncwarp();
        uint32_t loc[8], sum = 0;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            loc[b] = hist[lane * 8 + b];
            sum += loc[b];
        }
        uint32_t incl = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const uint32_t excl = incl - sum;
        const bool mine = excl < need && incl >= need;
        uint32_t bin = 0, below = 0, cnt = 0;
        if (mine) {
            uint32_t cum = excl;
            for (int b = 0; b < 8; ++b) {
                if (cum + loc[b] >= need) {
                    bin = (uint32_t)(lane * 8 + b);
                    below = cum;
                    cnt = loc[b];
                    break;
                }
                cum += loc[b];
            }
        }
        const uint32_t who = __ballot_sync(0xffffffffu, mine);
        const int src = who ? __ffs(who) - 1 : 0;
        bin = __shfl_sync(0xffffffffu, bin, src);
        below = __shfl_sync(0xffffffffu, below, src);
        cnt = __shfl_sync(0xffffffffu, cnt, src);
        prefix |= (uint64_t)bin << shift;
        mask |= (uint64_t)bmask << shift;
        need -= below;
        __syncwarp();
        if (cnt == need) break;
    }
    prefix_out = prefix;
    mask_out = mask;
}

// Keep in bd/bs[0, K) the K smallest (distance, slot) entries of the two
// unsorted runs [0, nb) and [PB, PB + nc) (PB >= K), with nb + nc > K; the kept
// entries stay unsorted (a slot appears once per buffer, so the keys are
// distinct).  Returns the largest kept distance.
__device__ float warp_select_keep(float *bd, int32_t *bs, int K, int PB, int nb, int nc,
                                  uint32_t *hist, int lane)
{
    auto at = [&](int i) { return i < nb ? i : PB + (i - nb); };
    uint64_t prefix, mask;
    warp_radix_kth([&](int i) { return ds_key(bd[at(i)], bs[at(i)]); }, nb + nc, K, hist, lane,
                   prefix, mask);
    // stable compaction in place (every write index <= its read index)
    int w = 0;
    float dmax = -INFINITY;
    for (int i0 = 0; i0 < nb; i0 += 32) {
        const int i = i0 + lane;
        float dv = 0.f;
        int32_t sv = 0;
        bool take = false;
        if (i < nb) {
            dv = bd[i];
            sv = bs[i];
            take = (ds_key(dv, sv) & mask) <= prefix;
        }
        const uint32_t mk = __ballot_sync(0xffffffffu, take);
        __syncwarp();
        if (take) {
            const int p = w + __popc(mk & lanemask_lt());
            bd[p] = dv;
            bs[p] = sv;
            dmax = fmaxf(dmax, dv);
        }
        w += __popc(mk);
        __syncwarp();
    }
    for (int i0 = 0; i0 < nc; i0 += 32) {
        const int i = PB + i0 + lane;
        float dv = 0.f;
        int32_t sv = 0;
        bool take = false;
        if (i0 + lane < nc) {
            dv = bd[i];
            sv = bs[i];
            take = (ds_key(dv, sv) & mask) <= prefix;
        }
        const uint32_t mk = __ballot_sync(0xffffffffu, take);
        if (take) {
            const int p = w + __popc(mk & lanemask_lt());
            if (p < K) {
                bd[p] = dv;
                bs[p] = sv;
            }
            dmax = fmaxf(dmax, dv);
        }
        w += __popc(mk);
    }
    __syncwarp();
    for (int o = 16; o > 0; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    return dmax;
}

// Reduce the two unsorted runs [0, nb) and [PB, PB + nc) of one row
// (nb + nc <= 32 * EK, more than Kw entries) to between K and Kw of their
// smallest (distance, slot) entries, written unsorted to [0, kept); returns
// the largest kept distance, a bound on the row's K-th smallest.  The
// 32-bit distance keys and the slots live in registers; a bisection on the
// key value with ballot counts stops at the first value with between K and
// Kw keys at or below it, which takes a few rounds where the exact K-th
// needs one per key bit.  Only when ties at the K-th key span past Kw is
// the cut made exact (K kept, ties to the lower slots).
template <int EK>
__device__ float warp_select_window(float *bd, int32_t *bs, int K, int Kw, int PB, int nb,
                                    int nc, int lane, int &kept)
{
    const int n = nb + nc;
    uint32_t key[EK];
    int32_t slt[EK];
#pragma unroll
    for (int e = 0; e < EK; ++e) {
        const int i = lane + 32 * e;
        const int ai = i < nb ? i : PB + (i - nb);
        key[e] = i < n ? fkey(bd[ai]) : 0xffffffffu;
        slt[e] = i < n ? bs[ai] : 0x7fffffff;
    }
    uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll
    for (int e = 0; e < EK; ++e)
        if (key[e] != 0xffffffffu) {
            kmin = min(kmin, key[e]);
            kmax = max(kmax, key[e]);
        }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    // invariant: #(key <= hi) >= K; stop at any value with K..Kw keys below
    uint32_t lo = kmin, hi = kmax, cnt = 0;
    bool found = false;
    while (lo < hi) {
        const uint32_t mid = lo + ((hi - lo) >> 1);
        uint32_t c = 0;
#pragma unroll
        for (int e = 0; e < EK; ++e) c += __popc(__ballot_sync(0xffffffffu, key[e] <= mid));
        if (c >= (uint32_t)K && c <= (uint32_t)Kw) {
            lo = mid;
            cnt = c;
            found = true;
            break;
        }
        if (c > (uint32_t)Kw) hi = mid;
        else lo = mid + 1;
    }
    const uint32_t v = lo;  // found: K..Kw keys <= v; else v is the K-th key
    if (!found) {
        uint32_t c = 0;
#pragma unroll
        for (int e = 0; e < EK; ++e) c += __popc(__ballot_sync(0xffffffffu, key[e] <= v));
        cnt = c;
    }
    int32_t cut = 0x7fffffff;  // entries equal to v kept: slot <= cut
    if (cnt > (uint32_t)Kw) {  // ties at v span past Kw: keep exactly K
        uint32_t clt = 0;
#pragma unroll
        for (int e = 0; e < EK; ++e) clt += __popc(__ballot_sync(0xffffffffu, key[e] < v));
        const uint32_t need = (uint32_t)K - clt;
        int32_t slo = 0, shi = 0x7fffffff;
        while (slo < shi) {
            const int32_t mid = slo + ((shi - slo) >> 1);
            uint32_t c = 0;
#pragma unroll
            for (int e = 0; e < EK; ++e)
                c += __popc(__ballot_sync(0xffffffffu, key[e] == v && slt[e] <= mid));
            if (c >= need) shi = mid;
            else slo = mid + 1;
        }
        cut = slo;
    }
    __syncwarp();  // every lane has read its entries before any is written
    int w = 0;
    uint32_t kk = 0u;
#pragma unroll
    for (int e = 0; e < EK; ++e) {
        const bool take = key[e] < v || (key[e] == v && slt[e] <= cut);
        const uint32_t mk = __ballot_sync(0xffffffffu, take);
        if (take) {
            const int p = w + __popc(mk & lanemask_lt());
            bd[p] = fkey_inv(key[e]);
            bs[p] = slt[e];
            kk = max(kk, key[e]);
        }
        w += __popc(mk);
    }
    __syncwarp();
    kept = w;
    return fkey_inv(__reduce_max_sync(0xffffffffu, kk));
}

// Fold the nc pending candidates of one row (at [PB, PB + nc)) into its
// held set [0, nb): when the union holds more than Kw entries it is reduced
// to between K and Kw of its smallest (exactly K for long buffers, by the
// radix select), else the pending entries move down whole.  Returns a bound
// on the row's K-th smallest distance (+inf while fewer than K are held).
__device__ __forceinline__ float fold_row(float *bd, int32_t *bs, int K, int Kw, int PB, int &nb,
                                          int nc, uint32_t *hist, int lane)
{
    const int n = nb + nc;
    if (n > Kw) {
        int kept = K;
        const float kd = n <= 64    ? warp_select_window<2>(bd, bs, K, Kw, PB, nb, nc, lane, kept)
                         : n <= 128 ? warp_select_window<4>(bd, bs, K, Kw, PB, nb, nc, lane, kept)
                         : n <= 192 ? warp_select_window<6>(bd, bs, K, Kw, PB, nb, nc, lane, kept)
                         : n <= 320 ? warp_select_window<10>(bd, bs, K, Kw, PB, nb, nc, lane, kept)
                                    : warp_select_keep(bd, bs, K, PB, nb, nc, hist, lane);
        nb = kept;
        return kd;
    }
    for (int i = lane; i < nc; i += 32) {  // write index < PB <= read index
        const float dv = bd[PB + i];
        const int32_t sv = bs[PB + i];
        bd[nb + i] = dv;
        bs[nb + i] = sv;
    }
    nb += nc;
    __syncwarp();
    if (nb < K) return INFINITY;
    float dmax = -INFINITY;
    for (int i = lane; i < nb; i += 32) dmax = fmaxf(dmax, bd[i]);
    for (int o = 16; o > 0; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    return dmax;
}

// As kth_bound (device_utils.cuh) for more values than registers hold, by
// histograms of TC_HIST equal steps of the value range: of all values, then
// of the step the K-th falls into, until little more than K lie within.
// 2,304 values: about 5 passes over them where the bisection took 18.
template <class V>
__device__ float kth_bound_hist(V val, int n, int K, uint32_t *hist, int lane)
{
    const int Kw = K + (K >> 5) + 1;
    float lo = INFINITY, hi = -INFINITY;
    int fin = 0;
#pragma unroll 8
    for (int i = lane; i < n; i += 32) {
        const float v = val(i);
        if (v < INFINITY) {
            lo = fminf(lo, v);
            hi = fmaxf(hi, v);
            ++fin;
        }
    }
    if (__reduce_add_sync(0xffffffffu, fin) < K) return INFINITY;
    int below = 0;  // values under lo
    for (int round = 0; round < 4; ++round) {
        for (int o = 16; o > 0; o >>= 1) {
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        const float scale = (float)TC_HIST / (hi - lo);
        if (!(scale < INFINITY) || !(hi > lo)) break;
        // the same rounding in every pass: monotone in v
        auto bin = [&](float v) { return min(TC_HIST - 1, (int)__fmul_rn(__fsub_rn(v, lo), scale)); };
#pragma unroll
        for (int b = 0; b < TC_HIST / 32; ++b) hist[lane * (TC_HIST / 32) + b] = 0u;
        __syncwarp();
#pragma unroll 8
        for (int i = lane; i < n; i += 32) {
            const float v = val(i);
            if (v >= lo && v <= hi) atomicAdd(&hist[bin(v)], 1u);
        }
        __syncwarp();
        uint32_t loc[TC_HIST / 32], sum = 0;
#pragma unroll
        for (int b = 0; b < TC_HIST / 32; ++b) {
            loc[b] = hist[lane * (TC_HIST / 32) + b];
            sum += loc[b];
        }
        uint32_t incl = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const uint32_t need = (uint32_t)(K - below);
        uint32_t cum = incl - sum;
        const bool mine = cum < need && incl >= need;
        int at = 0;
        uint32_t under = 0, upto = 0;
        if (mine)
            for (int b = 0; b < TC_HIST / 32; ++b) {
                if (cum + loc[b] >= need) {
                    at = lane * (TC_HIST / 32) + b;
                    under = cum;
                    upto = cum + loc[b];
                    break;
                }
                cum += loc[b];
            }
        const uint32_t who = __ballot_sync(0xffffffffu, mine);
        const int src = who ? __ffs(who) - 1 : 0;
        at = __shfl_sync(0xffffffffu, at, src);
        under = __shfl_sync(0xffffffffu, under, src);
        upto = __shfl_sync(0xffffffffu, upto, src);
        __syncwarp();
        // the step's own range; its largest value bounds the K-th
        float l2 = INFINITY, h2 = -INFINITY;
#pragma unroll 8
        for (int i = lane; i < n; i += 32) {
            const float v = val(i);
            if (v >= lo && v <= hi && bin(v) == at) {
                l2 = fminf(l2, v);
                h2 = fmaxf(h2, v);
            }
        }
        lo = l2;
        hi = h2;
        if (below + (int)upto <= Kw) break;
        below += (int)under;
    }
    for (int o = 16; o > 0; o >>= 1) hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    return hi;
}

// 16-byte asynchronous copy global -> shared; bytes past `src_bytes` (0 or
// 16) are zero-filled
__device__ __forceinline__ void cp_async16(void *dst, const void *src, uint32_t src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(src_bytes)
                 : "memory");
}

__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.commit_group;\n cp.async.wait_group 0;\n" ::: "memory");
}

__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(p), "r"(bytes) : "memory");
}

template <int DT, int TN>  // DT: 0 = BF16, 1 = FP8 E4M3; TN: queries per tile
__global__ __launch_bounds__(TcShape<TN>::NT, 1) void k_scan_tc(
    const __grid_constant__ CUtensorMap tmap, const __grid_constant__ CUtensorMap tmap_t,
    TcArgs a)
{
    pdl_begin();
    using S = TcShape<TN>;
    constexpr int EW = S::EW, FW = S::FW, EPI = S::EPI, TB = S::TB, NACC = S::NACC;
    constexpr int ESZ = DT == 0 ? 2 : 1;
    constexpr int EPC = 128 / ESZ;  // elements per 128-byte chunk
    extern __shared__ unsigned char smem_raw[];
    // 1024-byte alignment for the swizzled operand tiles
    unsigned char *smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    const int KC = a.KC, M = a.M, K = a.K, C = a.C, d = a.d, NST = a.nst;
    const TcSmem L = tc_smem<TN>(KC, M, NST);
    unsigned char *A = smem + L.a;
    unsigned char *B = smem + L.b;
    float *BD = reinterpret_cast<float *>(smem + L.bd);
    int32_t *BS = reinterpret_cast<int32_t *>(smem + L.bs);
    unsigned char *CTX = smem + L.ctx;
    uint32_t *Hist = reinterpret_cast<uint32_t *>(smem + L.hist);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L.bars);
    static_assert(TC_MAXST <= 4 && NACC <= 16 && TC_CTX == 2, "barrier layout");
    uint64_t *full = bars, *empty = bars + 4, *tfull = bars + 8, *tempty = bars + 24,
             *cfull = bars + 40, *cempty = bars + 42,
             *bfull = bars + 44, *bfree = bars + 46;
    uint32_t *tmem_base = reinterpret_cast<uint32_t *>(bars + 48);
    volatile int *s_abort = reinterpret_cast<volatile int *>(bars + 49);
    __shared__ int32_t s_cnt[TN], s_nb[TN];  // pending candidates, held best
    __shared__ float s_kd[TN];
    __shared__ __align__(16) float s_t[TN];   // kd - ||q||^2 of each row
    __shared__ __align__(16) float s_sc[TN];  // 2 x dequantisation scale of each row

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int SPB = TC_M / C;  // slabs per A tile
    const uint32_t idesc = DT == 0 ? mma_idesc(1, 1, TC_M, TN) : mma_idesc(0, 0, TC_M, TN);
    constexpr size_t CTXB = tc_ctx_bytes(TN);
    auto hdr = [&](int j) { return reinterpret_cast<int32_t *>(CTX + j * CTXB); };
    auto c_qpair = [&](int j) { return reinterpret_cast<int32_t *>(CTX + j * CTXB + 64); };
    auto c_qn = [&](int j) { return reinterpret_cast<float *>(CTX + j * CTXB + 64 + 4 * TN); };
    auto c_qsc = [&](int j) { return reinterpret_cast<float *>(CTX + j * CTXB + 64 + 8 * TN); };
    auto c_kd0 = [&](int j) { return reinterpret_cast<float *>(CTX + j * CTXB + 64 + 12 * TN); };
    auto c_qi = [&](int j) { return reinterpret_cast<int32_t *>(CTX + j * CTXB + 64 + 16 * TN); };
    auto c_sl = [&](int j) { return reinterpret_cast<int32_t *>(CTX + j * CTXB + 64 + 20 * TN); };
    auto c_bits = [&](int j) {
        return reinterpret_cast<uint32_t *>(CTX + j * CTXB + 64 + 20 * TN + 4 * TC_META);
    };

    if (tid == 0) {
        for (int i = 0; i < NST; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < NACC; ++i) {
            mbar_init(&tfull[i], 1);
            mbar_init(&tempty[i], EW);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bfull[i], 32);
            mbar_init(&bfree[i], 1);
        }
        for (int i = 0; i < TC_CTX; ++i) {
            mbar_init(&cfull[i], 32);
            mbar_init(&cempty[i], EW);
        }
        fence_mbar_init();
        *s_abort = 0;
    }
    if (warp == 2) tmem_alloc(tmem_base, NACC * TB);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = *tmem_base;

    if (warp == 2) {
        // ---- item contexts
        int sub = 0, nsub = 0, l = 0, m = 0, s0 = 0, ns = 0, chunk = 0, qb = 0;
        float inv_l = 1.f;
        for (int it = 0;; ++it) {
            const int j = it % TC_CTX;
            const uint32_t cu = (uint32_t)(it / TC_CTX);
            bool ok = cu == 0 || mbar_wait_ab(&cempty[j], (cu - 1) & 1, a.err, s_abort, a.wait_ns);
            if (!__all_sync(0xffffffffu, ok)) break;
            int32_t *h = hdr(j);
            bool stop = false;
            if (sub == nsub) {
                int nx = 0, go = 0;
                if (lane == 0) {
                    nx = atomicAdd(&a.ctl->next_item, 1);
                    go = nx < a.ctl->nitems && !*s_abort;
                }
                nx = __shfl_sync(0xffffffffu, nx, 0);
                if (!__shfl_sync(0xffffffffu, go, 0)) {
                    stop = true;
                } else {
                    const int2 itv = a.items[nx];
                    l = itv.x;
                    const int nc_l = a.nch[l];
                    const int tile = itv.y >> 8;
                    chunk = itv.y & 255;
                    const int r0 = tile * TN;
                    m = min(TN, a.lcnt[l] - r0);
                    int ns_total = a.nslabs[l];
                    if (ns_total > a.dir_cap) {
                        if (lane == 0) atomicOr(a.err, ERR_DIR_BOUND);
                        ns_total = (int)a.dir_cap;
                    }
                    s0 = (int)((int64_t)ns_total * chunk / nc_l);
                    ns = (int)((int64_t)ns_total * (chunk + 1) / nc_l) - s0;
                    if (a.seed_slabs > 0) ns = chunk == 0 ? min(ns, a.seed_slabs) : 0;
                    nsub = max(1, (ns + TC_META - 1) / TC_META);
                    sub = 0;
                    qb = a.loff[l] + r0;
                    inv_l = DT == 1 ? a.inv_scale8[l] : 1.f;
                }
            }
            __syncwarp();
            if (stop) {
                if (lane == 0) h[8] = CF_STOP;
                __syncwarp();
                mbar_arrive(&cfull[j]);
                break;
            }
            const int ss0 = s0 + sub * TC_META;
            const int sns = max(0, min(TC_META, ns - sub * TC_META));
            const int nblk = (sns + SPB - 1) / SPB;
            if (lane == 0) {
                h[0] = l;
                h[1] = m;
                h[2] = ss0;
                h[3] = sns;
                h[4] = nblk;
                h[5] = max(M, ((TN * M) / max(m, 1)) & ~7);  // rows of a thin tile get longer buffers
                h[7] = chunk;
                h[8] = (sub == 0 ? CF_FIRST : 0) | (sub + 1 == nsub ? CF_LAST : 0);
                h[9] = __float_as_int(inv_l);
            }
            int32_t *qp = c_qpair(j), *cqi = c_qi(j);
            float *cqn = c_qn(j), *cqsc = c_qsc(j), *ckd = c_kd0(j);
            for (int r = lane; r < TN; r += 32) {
                const int pr = r < m ? a.qlist[qb + r] : -1;
                const int qi = pr >= 0 ? pr / a.P : 0;
                const int qrow = a.per_pair ? (pr >= 0 ? pr : 0) : qi;  // row of qn, qsc, qcast
                qp[r] = pr;
                cqi[r] = qrow;
                cqn[r] = pr >= 0 ? a.qn[qrow] : 0.f;
                cqsc[r] = pr >= 0 ? a.qsc[qrow] : 1.f;
                ckd[r] = pr >= 0 ? __ldcg(a.thr + qi) : INFINITY;
            }
            int32_t *sl = c_sl(j);
            uint32_t *bt = c_bits(j);
            const int32_t *dirl = a.dir + (size_t)l * a.dir_cap + ss0;
            const int W = C / 32;
            const uint32_t pay_bytes = (uint32_t)(C * d * ESZ);
            for (int i = lane; i < sns; i += 32) {
                const int s = dirl[i];
                const bool okk = s >= 0 && s < a.n_slabs;
                if (!okk) atomicOr(a.err, ERR_BAD_SLAB);
                sl[i] = okk ? s : -1;
                for (int w = 0; w < W; ++w) bt[i * 4 + w] = okk ? __ldg(a.bits + (size_t)s * W + w) : 0u;
                if (okk && i < a.pf_tiles * SPB) {
                    prefetch_l2(a.pay + (size_t)s * pay_bytes, pay_bytes);
                    prefetch_l2(a.xnorm + (size_t)s * C, (uint32_t)(C * 4));
                }
            }
            __syncwarp();
            mbar_arrive(&cfull[j]);
            ++sub;
        }
    } else if (warp == 3) {
        // ---- query tiles (B operand), rounded and swizzled
        for (int it = 0;; ++it) {
            const int j = it % TC_CTX, bb = it & 1;
            bool ok = mbar_wait_ab(&cfull[j], (uint32_t)(it / TC_CTX) & 1, a.err, s_abort, a.wait_ns);
            if (!__all_sync(0xffffffffu, ok)) break;
            if (hdr(j)[8] & CF_STOP) break;
            ok = it < 2 || mbar_wait_ab(&bfree[bb], (uint32_t)((it >> 1) - 1) & 1, a.err, s_abort, a.wait_ns);
            if (!__all_sync(0xffffffffu, ok)) break;
            const int32_t *cqi = c_qi(j);
            const int m = hdr(j)[1];
            unsigned char *Bb = B + (size_t)bb * KC * TN * 128;
            // 16-byte asynchronous copies of the rounded query rows straight
            // into the swizzled tile (no registers, every copy in flight at
            // once); chunks past the row (d * ESZ < KC * 128) are zero-filled
            const int rowc = d * ESZ / 16, CPR = KC * 8;
            for (int e = lane; e < m * CPR; e += 32) {
                const int r = (CPR & (CPR - 1)) == 0 ? e >> (__ffs(CPR) - 1) : e / CPR;
                const int c = e - r * CPR, kc = c >> 3, cc = c & 7;
                const bool in = c < rowc;
                const unsigned char *src = a.qcast + (in ? ((size_t)cqi[r] * d * ESZ + (size_t)c * 16) : 0);
                cp_async16(Bb + (size_t)kc * TN * 128 + (size_t)(r >> 3) * 1024 + (r & 7) * 128 +
                               ((cc ^ (r & 7)) << 4),
                           src, in ? 16u : 0u);
            }
            cp_async_wait_all();
            fence_proxy_async_smem();  // B is read by the tensor cores (async proxy)
            mbar_arrive(&bfull[bb]);
        }
    } else if (warp == 0) {
        // ---- TMA producer
        if (lane == 0) {
            uint32_t g = 0;
            const uint32_t pay_bytes = (uint32_t)(C * d * ESZ);
            for (int it = 0;; ++it) {
                const int j = it % TC_CTX;
                if (!mbar_wait_ab(&cfull[j], (uint32_t)(it / TC_CTX) & 1, a.err, s_abort, a.wait_ns)) break;
                const int32_t *h = hdr(j);
                if (h[8] & CF_STOP) break;
                const int sns = h[3], nblk = h[4];
                const int32_t *sl = c_sl(j);
                bool ab = false;
                for (int b = 0; b < nblk; ++b, ++g) {
                    const uint32_t st = g % NST, u = g / NST;
                    if (u >= 1 && !mbar_wait_ab(&empty[st], (u - 1) & 1, a.err, s_abort, a.wait_ns)) {
                        ab = true;
                        break;
                    }
                    const int nsl = min(SPB, sns - b * SPB);
                    int okc = 0;
                    for (int jj = 0; jj < nsl; ++jj) okc += sl[b * SPB + jj] >= 0;
                    mbar_arrive_expect_tx(&full[st], (uint32_t)(okc * KC * C * 128));
                    // a whole tile of consecutive slabs s0 .. s0 + SPB - 1 is one
                    // 128-row box (the same bytes, the same swizzled layout)
                    auto consecutive = [&](int bb, int ns) {
                        const int s0 = sl[bb * SPB];
                        bool r = a.tile_box && ns == SPB && s0 >= 0;
                        for (int jj = 1; jj < ns && r; ++jj) r = sl[bb * SPB + jj] == s0 + jj;
                        return r;
                    };
                    if (consecutive(b, nsl)) {
                        const int s0 = sl[b * SPB];
                        for (int kc = 0; kc < KC; ++kc)
                            tma_load_2d(A + (size_t)st * KC * TC_M * 128 + (size_t)kc * TC_M * 128,
                                        &tmap_t, kc * EPC, s0 * C, &full[st]);
                    } else {
                        for (int jj = 0; jj < nsl; ++jj) {
                            const int s = sl[b * SPB + jj];
                            if (s < 0) continue;
                            for (int kc = 0; kc < KC; ++kc)
                                tma_load_2d(A + (size_t)st * KC * TC_M * 128 +
                                                (size_t)kc * TC_M * 128 + (size_t)jj * C * 128,
                                            &tmap, kc * EPC, s * C, &full[st]);
                        }
                    }
                    const int bp = b + a.pf_tiles;  // keep the L2 prefetch ahead
                    if (bp < nblk) {
                        const int nsp = min(SPB, sns - bp * SPB);
                        if (consecutive(bp, nsp)) {
                            const int s0 = sl[bp * SPB];
                            prefetch_l2(a.pay + (size_t)s0 * pay_bytes, (uint32_t)(SPB * pay_bytes));
                            prefetch_l2(a.xnorm + (size_t)s0 * C, (uint32_t)(SPB * C * 4));
                        } else {
                            for (int jj = 0; jj < nsp; ++jj) {
                                const int s = sl[bp * SPB + jj];
                                if (s < 0) continue;
                                prefetch_l2(a.pay + (size_t)s * pay_bytes, pay_bytes);
                                prefetch_l2(a.xnorm + (size_t)s * C, (uint32_t)(C * 4));
                            }
                        }
                    }
                }
                if (ab) break;
            }
            // the copies of the last tiles issued have landed before exit
            for (uint32_t t = g > (uint32_t)NST ? g - NST : 0; t < g; ++t)
                mbar_wait_bounded(&full[t % NST], (t / NST) & 1, a.err);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---- MMA issuer
        if (lane == 0) {
            uint32_t g = 0;
            for (int it = 0;; ++it) {
                const int j = it % TC_CTX, bb = it & 1;
                if (!mbar_wait_ab(&cfull[j], (uint32_t)(it / TC_CTX) & 1, a.err, s_abort, a.wait_ns)) break;
                if (hdr(j)[8] & CF_STOP) break;
                const int nblk = hdr(j)[4];
                if (!mbar_wait_ab(&bfull[bb], (uint32_t)(it >> 1) & 1, a.err, s_abort, a.wait_ns)) break;
                const uint32_t bbase = smem_u32(B + (size_t)bb * KC * TN * 128);
                bool ab = false;
                for (int b = 0; b < nblk; ++b, ++g) {
                    const uint32_t st = g % NST, u = g / NST, buf = g % NACC, ub = g / NACC;
                    if (!mbar_wait_ab(&full[st], u & 1, a.err, s_abort, a.wait_ns)) {
                        ab = true;
                        break;
                    }
                    if (ub >= 1 && !mbar_wait_ab(&tempty[buf], (ub - 1) & 1, a.err, s_abort, a.wait_ns)) {
                        ab = true;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t abase = smem_u32(A + (size_t)st * KC * TC_M * 128);
                    for (int kc = 0; kc < KC; ++kc)
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) {
                            const uint64_t ad = smem_desc_sw128(abase + kc * TC_M * 128 + ks * 32, 1024);
                            const uint64_t bd = smem_desc_sw128(bbase + kc * TN * 128 + ks * 32, 1024);
                            const uint32_t acc = (kc | ks) != 0;
                            if (DT == 0) mma_bf16(tbase + buf * TB, ad, bd, idesc, acc);
                            else mma_fp8(tbase + buf * TB, ad, bd, idesc, acc);
                        }
                    mma_commit(&tfull[buf]);
                    mma_commit(&empty[st]);
                }
                if (ab) break;
                mma_commit(&bfree[bb]);
            }
            // the last accumulator is written before TMEM is released
            if (g > 0) mbar_wait_bounded(&tfull[(g - 1) % NACC], ((g - 1) / NACC) & 1, a.err);
        }
        __syncwarp();
    } else if (warp >= 4) {
        // ---- epilogue
        // An item of at most 16 live columns per warp block leaves the other
        // blocks' warps without columns: TP sets of warps then take every
        // TP-th tile instead.  A group is the NACC tiles whose accumulators
        // TMEM holds.  When some row has no bound yet, the item's first group
        // is looked at twice: first each thread keeps the smallest distance
        // of its rows per column (in `nbank` banks of tiles), and the K'-th
        // smallest of those minima is a bound of the row's K'-th distance at
        // least as many rows lie within; little more than K' rows pass it
        // (128 minima of 8 rows: 45 for K' = 40).  Without it the first rows
        // all pass and are reduced by folds that hold up every warp: 186 us
        // against 118 for 10,000 queries' nearest of 1,024 lists.
        const int ew = warp - 4;             // epilogue warp
        const int qt = ew & 3;               // its TMEM lane quarter (warp % 4)
        const int et = ew * 32 + lane;       // epilogue thread
        const int v = qt * 32 + lane;        // A row = vector of the tile
        const uint32_t tlane = (uint32_t)(qt * 32) << 16;
        uint32_t *hist = Hist + min(ew, FW - 1) * TC_HIST;
        float *smin = BD;                    // the minima, while no candidate is held
        uint32_t g = 0;
        for (int it = 0;; ++it) {
            const int j = it % TC_CTX;
            const bool ok = mbar_wait_ab(&cfull[j], (uint32_t)(it / TC_CTX) & 1, a.err, s_abort, a.wait_ns);
            if (!named_bar_and(1, EPI, ok && !*s_abort)) break;
            const int32_t *h = hdr(j);
            const int flags = h[8];
            if (flags & CF_STOP) break;
            const int m = h[1], sns = h[3], nblk = h[4], ME = h[5], chunk = h[7];
            const float inv_l = __int_as_float(h[9]);
            // columns and tiles of this warp
            // (no more sets than a row's buffer has room for, twice over where a
            // fold is dear)
            const int ncb = (m + TC_NCOL - 1) / TC_NCOL;
            const int TP = max(1, min((EW / 4) / ncb, (ME - a.RK) / (K > 128 ? 2 * TC_M : TC_M)));
            const int set = (ew >> 2) / ncb, c0 = ((ew >> 2) % ncb) * TC_NCOL;
            const bool act = set < TP;
            // a row holds [0, nb) (at most RK) and appends at RK; its pending
            // candidates are folded once a step leaves more than FT of them:
            // FT plus one step always fits.  A step is a round of TP tiles, or,
            // where a thin item's long buffers have room for it, a whole group:
            // its warps then meet no barrier from tile to tile.  A fold keeps
            // K' .. Kw.  For K' <= 128, more than 96 pending before a step cost
            // more in a fold than the extra folds that a lower trigger brings
            // (measured at K' = 40); deeper sets fold only when the room is
            // full (the held K' dominate a fold's cost)
            const int RK = a.RK, Kw = K + ((RK - K) >> 1);
            const bool freely = ME - RK >= NACC * TC_M + 96;
            const int step = freely ? NACC * TC_M : TP * TC_M;
            const int FT = K > 128 ? ME - RK - step : min(ME - RK - step, 96);
            const int32_t *qp = c_qpair(j);
            const float *cqn = c_qn(j), *cqsc = c_qsc(j), *ckd = c_kd0(j);
            const int32_t *sl = c_sl(j);
            const uint32_t *bt = c_bits(j);
            bool unbound = false;
            if (flags & CF_FIRST) {
                for (int r = et; r < TN; r += EPI) {
                    const bool on = r < m;
                    s_cnt[r] = 0;
                    s_nb[r] = 0;
                    s_kd[r] = on ? ckd[r] : INFINITY;
                    s_t[r] = on ? ckd[r] - cqn[r] : -INFINITY;
                    s_sc[r] = DT == 0 ? 2.f : 2.f / (inv_l * cqsc[r]);
                    unbound |= on && ckd[r] > 1e38f;
                }
            }
            // the tiles of one column are worth a second look from two on
            const bool look = named_bar_or(1, EPI, unbound && nblk > 1);
            bool run = true;
            // the slab of this thread's row in A tile b (-1: none), its slot
            const int slot = v % C, jr = v / C;
            auto row_slab = [&](int b) {
                return jr < min(SPB, sns - b * SPB) ? sl[b * SPB + jr] : -1;
            };
            auto row_live = [&](int b, int sv) {
                return sv >= 0 && ((bt[(b * SPB + jr) * 4 + (slot >> 5)] >> (slot & 31)) & 1u);
            };
            auto row_norm = [&](int sv) {
                return sv >= 0 ? __ldg(a.xnorm + (size_t)sv * C + slot) : 0.f;
            };
            auto tile_wait = [&](int i) {  // accumulator of the group's tile i
                const bool w = mbar_wait_ab(&tfull[(g + i) % NACC], ((g + i) / NACC) & 1, a.err, s_abort,
                                            a.wait_ns);
                return __all_sync(0xffffffffu, w);  // tcgen05.ld is warp-aligned
            };
            auto tile_load = [&](int i, float (&dv)[TC_NCOL]) {
                tmem_ld16(tbase + ((g + i) % NACC) * TB + c0 + tlane, dv);
                tmem_ld_wait(dv);
            };
            auto scales = [&](int i4, float (&sc)[4]) {
                sc[0] = sc[1] = sc[2] = sc[3] = 2.f;
                if (DT == 1) {
                    const float4 sv = reinterpret_cast<const float4 *>(s_sc + c0)[i4];
                    sc[0] = sv.x;
                    sc[1] = sv.y;
                    sc[2] = sv.z;
                    sc[3] = sv.w;
                }
            };
            for (int gb = 0; gb < nblk && run; gb += NACC) {
                const int ng = min(NACC, nblk - gb);
                if (look && gb == 0) {
                    // banks of a set: 2.5 K' minima per column at least; a bank per
                    // tile for deep sets where they fit (every row its own minimum:
                    // 412 of K' = 400's bound pass, else a quarter more than fit a run)
                    const int tset = (ng + TP - 1) / TP;
                    int nbs = max(1, ((5 * K + 255) / 256 + TP - 1) / TP);
                    if (K > 128) nbs = max(nbs, min(tset, (TN * M * 8) / (TP * m * TC_M * 4)));
                    const int per = (tset + nbs - 1) / nbs;                       // tiles of a bank
                    bool wok = true;
                    tc_fence_after();
                    if (act) {
                        float mn[TC_NCOL];
                        int b = set;
                        int s_next = b < ng ? row_slab(b) : -1;
                        float x_next = row_norm(s_next);
                        for (int bk = 0; bk < nbs; ++bk) {
#pragma unroll
                            for (int i = 0; i < TC_NCOL; ++i) mn[i] = INFINITY;
                            for (int k = 0; k < per && b < ng; ++k, b += TP) {
                                const bool live = row_live(b, s_next);
                                const float xn = x_next;
                                s_next = b + TP < ng ? row_slab(b + TP) : -1;
                                x_next = row_norm(s_next);
                                wok = wok && tile_wait(b);
                                tc_fence_after();
                                float dv[TC_NCOL];
                                if (wok) {
                                    tile_load(b, dv);
#pragma unroll
                                    for (int i4 = 0; i4 < TC_NCOL / 4; ++i4) {
                                        float sc[4];
                                        scales(i4, sc);
#pragma unroll
                                        for (int c = 0; c < 4; ++c) {
                                            const int i = 4 * i4 + c;
                                            const float part = fmaf(-sc[c], dv[i], xn);
                                            if (live) mn[i] = fminf(mn[i], part);
                                        }
                                    }
                                }
                            }
                            float *o = smin + (size_t)((set * nbs + bk) * m + c0) * TC_M + v;
#pragma unroll
                            for (int i = 0; i < TC_NCOL; ++i)
                                if (c0 + i < m) o[i * TC_M] = mn[i];
                        }
                    }
                    tc_fence_before();
                    run = named_bar_and(1, EPI, wok && !*s_abort);
                    if (!run) break;
                    const int nv = TP * nbs * TC_M;  // minima per column
                    const bool many = nv > 32 * 12;  // past a warp's registers
                    for (int n = many && ew >= FW ? m : ew; n < m; n += many ? FW : EW) {
                        auto val = [&](int i) {
                            return smin[((size_t)(i >> 7) * m + n) * TC_M + (i & 127)];
                        };
                        const float b = many ? kth_bound_hist(val, nv, K, hist, lane)
                                             : kth_bound<12>(val, nv, K, lane);
                        if (lane == 0 && b < INFINITY) {
                            // room for the roundings of ||q||^2 + ||x||^2 - 2 s q.x, formed
                            // in another order for the distances that are kept
                            const float t = __fadd_ru(b, __fmul_ru(fabsf(b) + cqn[n], 4.8e-7f));
                            const float kd = __fadd_ru(t, cqn[n]);
                            if (t < s_t[n]) s_t[n] = t;
                            if (kd < s_kd[n]) {
                                s_kd[n] = kd;
                                if (kd >= 0.f)
                                    atomicMin(reinterpret_cast<int *>(a.thr) + qp[n] / a.P,
                                              __float_as_int(kd));
                            }
                        }
                    }
                    named_bar_sync(1, EPI);
                } else if (gb > 0) {
                    // bounds other items of the queries have left meanwhile
                    if (et < m) {
                        const float kd = __ldcg(a.thr + qp[et] / a.P);
                        if (kd < s_kd[et]) {
                            s_kd[et] = kd;
                            s_t[et] = fminf(s_t[et], kd - cqn[et]);
                        }
                    }
                    named_bar_sync(1, EPI);
                }
                int s_next = act && set < ng ? row_slab(gb + set) : -1;
                float x_next = row_norm(s_next);
                bool need = false, wok = true;
                for (int b0 = 0; b0 < ng; b0 += TP) {
                    const int b = b0 + set;  // this warp's tile of the round
                    const bool mine = act && b < ng;
                    const int sv = s_next;
                    const float xn = x_next;
                    float dv[TC_NCOL];
                    if (mine) {
                        s_next = b + TP < ng ? row_slab(gb + b + TP) : -1;
                        x_next = row_norm(s_next);
                        wok = wok && tile_wait(b);
                        tc_fence_after();
                        if (wok) tile_load(b, dv);
                        tc_fence_before();
                    }
                    __syncwarp();
                    if (lane == 0)
                        for (int t = b0; t < min(ng, b0 + TP); ++t) mbar_arrive(&tempty[(g + t) % NACC]);

                    // the row passes for query n when -s q.x + ||x||^2 <= kd_n -
                    // ||q_n||^2: one bit per column, then each lane takes its
                    // passing columns one after the other (one lane in three has
                    // any where a bound holds), a place in the column's buffer
                    // by a shared atomic each
                    if (wok && mine) {
                        uint32_t pm = 0u;
                        const float4 *t4 = reinterpret_cast<const float4 *>(s_t + c0);
#pragma unroll
                        for (int i4 = 0; i4 < TC_NCOL / 4; ++i4) {
                            const float4 tv = t4[i4];
                            const float tt[4] = {tv.x, tv.y, tv.z, tv.w};
                            float sc[4];
                            scales(i4, sc);
#pragma unroll
                            for (int c = 0; c < 4; ++c)
                                if (fmaf(-sc[c], dv[4 * i4 + c], xn) <= tt[c]) pm |= 1u << (4 * i4 + c);
                        }
                        // columns past m hold what an earlier item left there
                        if (m - c0 < TC_NCOL) pm &= (1u << (m - c0)) - 1u;
                        if (!row_live(gb + b, sv)) pm = 0u;
                        const int32_t gslot = sv * C + slot;
                        while (pm) {
                            const int i = __ffs(pm) - 1, n = c0 + i;
                            pm &= pm - 1;
                            float x8[8], x4[4];
#pragma unroll
                            for (int k = 0; k < 8; ++k) x8[k] = i & 8 ? dv[k + 8] : dv[k];
#pragma unroll
                            for (int k = 0; k < 4; ++k) x4[k] = i & 4 ? x8[k + 4] : x8[k];
                            const float xa = i & 2 ? x4[2] : x4[0], xb = i & 2 ? x4[3] : x4[1];
                            const int p = atomicAdd(&s_cnt[n], 1);
                            BD[n * ME + RK + p] = fmaf(-s_sc[n], i & 1 ? xb : xa, cqn[n] + xn);
                            BS[n * ME + RK + p] = gslot;
                            need |= p >= FT;
                        }
                        __syncwarp();
                    }
                    if (freely && b0 + TP < ng) continue;
                    if (named_bar_or(1, EPI, need || !wok || *s_abort)) {
                        run = named_bar_and(1, EPI, wok && !*s_abort);
                        if (!run) break;
                        need = false;
                        // fold the rows with pending candidates of about this
                        // many together: one row's fold holds every warp up, so
                        // rows that would follow in the next tiles go with it
                        for (int n = ew < FW ? ew : m; n < m; n += FW) {
                            const int cc = s_cnt[n];
                            if (cc <= (K > 128 ? FT : FT >> 2)) continue;
                            int nb = s_nb[n];
                            const float kd = fold_row(BD + (size_t)n * ME, BS + (size_t)n * ME, K, Kw,
                                                      RK, nb, cc, hist, lane);
                            if (lane == 0) {
                                s_nb[n] = nb;
                                s_cnt[n] = 0;
                                if (kd < s_kd[n]) {
                                    s_kd[n] = kd;
                                    s_t[n] = fminf(s_t[n], kd - cqn[n]);
                                    // items over other chunks of the list read it
                                    if (kd >= 0.f)
                                        atomicMin(reinterpret_cast<int *>(a.thr) + qp[n] / a.P,
                                                  __float_as_int(kd));
                                }
                            }
                            __syncwarp();
                        }
                        named_bar_sync(1, EPI);
                    }
                }
                g += ng;
            }
            if (!run) {
                if (et == 0) *s_abort = 1;
                break;
            }
            if (flags & CF_LAST) {
                // each row's run: between K' and RK of its smallest
                // candidates (all of them when fewer), unsorted, with their
                // count (the per-query merge selects and sorts the best K');
                // a bound on its K'-th distance becomes a bound of the query
                // for the items that follow
                named_bar_sync(1, EPI);
                for (int n = ew < FW ? ew : m; n < m; n += FW) {
                    const int cc = s_cnt[n];
                    int nb = s_nb[n];
                    float *bd = BD + (size_t)n * ME;
                    int32_t *bs = BS + (size_t)n * ME;
                    float kd = s_kd[n];
                    if (cc > 0) kd = fminf(kd, fold_row(bd, bs, K, RK, RK, nb, cc, hist, lane));
                    const int run = a.seed_slabs > 0 ? -1 : a.prun[qp[n]];
                    const int64_t base = ((int64_t)run + chunk) * RK;
                    for (int i = lane; i < nb && run >= 0; i += 32) {
                        a.part_d[base + i] = bd[i];
                        a.part_i[base + i] = (int64_t)bs[i];
                    }
                    if (lane == 0 && run >= 0) a.part_n[run + chunk] = nb;
                    if (lane == 0 && kd >= 0.f && kd < INFINITY)
                        atomicMin(reinterpret_cast<int *>(a.thr) + qp[n] / a.P, __float_as_int(kd));
                    __syncwarp();
                }
            }
            named_bar_sync(1, EPI);
            if (lane == 0) mbar_arrive(&cempty[j]);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 2) tmem_dealloc(tbase, NACC * TB);
}

// ------------------------------------------------------- per-query merge
// One warp per query: the best K' (distance, slot) of the query's item
// outputs (runs of RK entries of which the first part_n[run] are valid,
// unsorted; the runs of one scan phase are contiguous, qrun[phase][q] =
// (first run, runs)) by a radix select over the 64-bit (distance, slot)
// keys of the valid entries, then sorted ascending, padded with (+inf, -1).
constexpr int MT_NT = 128;
// The K smallest (distance, slot) entries of the warp's buffer sd / ss (n > K
// distinct ones), in place and unsorted (every write index <= its read
// index); returns the largest distance kept.
__device__ __noinline__ float merge_reduce(float *sd, int32_t *ss, int n, int K, uint32_t *hist,
                                           int lane)
{
    __syncwarp();
    uint64_t prefix, mask;
    warp_radix_kth([&](int i) { return ds_key(sd[i], ss[i]); }, n, K, hist, lane, prefix, mask);
    int w = 0;
    float top = -INFINITY;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        const float dv = i < n ? sd[i] : INFINITY;
        const int32_t sv = i < n ? ss[i] : 0;
        const bool take = i < n && (ds_key(dv, sv) & mask) <= prefix;
        const uint32_t mk = __ballot_sync(0xffffffffu, take);
        __syncwarp();
        if (take) {
            const int p = w + __popc(mk & lanemask_lt());
            sd[p] = dv;
            ss[p] = sv;
            top = fmaxf(top, dv);
        }
        w += __popc(mk);
        __syncwarp();
    }
    for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
    return top;
}

// entries of the selection's shared buffer per warp (8 bytes each)
__host__ __device__ constexpr int merge_cap(int E) { return 64 * E > 512 ? 64 * E : 512; }
// The selection of one query (one warp): its best K' valid entries, unsorted,
// into sd / ss (merge_cap(E) entries of the warp's shared memory); returns
// their number, min(valid entries, K').  hist: TC_HIST words of shared memory.
// `bound` is the query's shared bound after the scan: at least K' entries
// lie at or below it, so only those are gathered, four runs' entries in
// flight at once.  A list cut into many chunks leaves a loose bound (a K'-th
// distance within one chunk), under which thousands of entries may lie:
// whenever the buffer is nearly full it is reduced to its K' smallest (a
// radix select on the 64-bit (distance, slot) keys) and the bound to the
// largest of them.
template <int E>
__device__ int merge_select(const int2 *__restrict__ qrun, int64_t nq, int64_t q, int nphase,
                            int K, int RK, float bound, const int32_t *__restrict__ part_n,
                            const float *__restrict__ part_d, const int64_t *__restrict__ part_i,
                            uint32_t *hist, float *sd, int32_t *ss, int lane)
{
    constexpr int CAP = merge_cap(E);
    const int2 r0 = qrun[q];
    const int2 r1 = nphase > 1 ? qrun[nq + q] : make_int2(0, 0);
    const int NR = r0.y + r1.y;
    auto run_of = [&](int t) -> int64_t { return t < r0.y ? r0.x + t : r1.x + (t - r0.y); };
    int have = 0;
    for (int t0 = 0; t0 < NR; t0 += 32) {
        const int cl = t0 + lane < NR ? min(part_n[run_of(t0 + lane)], RK) : 0;
        for (int u = 0; u < 32 && t0 + u < NR; u += 4) {
            int c[4], cm = 0;
            int64_t rb[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                c[r] = __shfl_sync(0xffffffffu, cl, u + r);
                rb[r] = c[r] > 0 ? run_of(t0 + u + r) * RK + lane : 0;
                cm = max(cm, c[r]);
            }
            for (int j0 = 0; j0 < cm; j0 += 64) {
                if (have > CAP - 256) {  // warp-uniform; K <= CAP - 256
                    bound = fminf(bound, merge_reduce(sd, ss, have, K, hist, lane));
                    have = K;
                }
                float dv[8];
                int32_t sv[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int r = e >> 1, j = j0 + 32 * (e & 1);
                    const bool ok = j + lane < c[r];
                    dv[e] = ok ? part_d[rb[r] + j] : INFINITY;
                    sv[e] = ok ? (int32_t)part_i[rb[r] + j] : -1;
                }
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const bool in = sv[e] >= 0 && dv[e] <= bound;
                    const uint32_t mk = __ballot_sync(0xffffffffu, in);
                    if (in) {
                        const int p = have + __popc(mk & lanemask_lt());
                        sd[p] = dv[e];
                        ss[p] = sv[e];
                    }
                    have += __popc(mk);
                }
            }
        }
    }
    if (have <= K) {
        __syncwarp();
        return have;
    }
    merge_reduce(sd, ss, have, K, hist, lane);
    return K;
}

template <int E>
__global__ __launch_bounds__(MT_NT) void k_merge_tc(const int2 *__restrict__ qrun, int64_t nq,
                                                    int nphase, int K, int RK,
                                                    const float *__restrict__ thr,
                                                    const int32_t *__restrict__ part_n,
                                                    const float *__restrict__ part_d,
                                                    const int64_t *__restrict__ part_i,
                                                    float *__restrict__ out_d,
                                                    int64_t *__restrict__ out_s)
{
    pdl_begin();
    constexpr int NW = MT_NT / 32;
    __shared__ uint32_t hist_s[NW][TC_HIST];
    __shared__ float sd[NW][merge_cap(E)];
    __shared__ int32_t ss[NW][merge_cap(E)];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t q = (blockIdx.x * (int64_t)MT_NT + threadIdx.x) >> 5;
    if (q >= nq) return;  // whole warps
    uint32_t *hist = hist_s[warp];
    const int nk = merge_select<E>(qrun, nq, q, nphase, K, RK, thr[q], part_n, part_d, part_i, hist,
                                   sd[warp], ss[warp], lane);
    float v[E];
    int32_t sv[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = lane + 32 * e;
        v[e] = i < nk ? sd[warp][i] : INFINITY;
        sv[e] = i < nk ? ss[warp][i] : 0x7fffffff;
    }
    warp_sort32<E>(v, sv, lane);
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = lane + 32 * e;
        if (i < K) {
            out_d[q * K + i] = i < nk ? v[e] : INFINITY;
            out_s[q * K + i] = i < nk ? (int64_t)sv[e] : -1;
        }
    }
}

void merge_tc(sivf_index *ix, int64_t nq, int nphase, const SearchScratch &s, int Kc, int RK,
              float *out_d, int64_t *out_s, cudaStream_t st)
{
    const unsigned blocks = (unsigned)((nq * 32 + MT_NT - 1) / MT_NT);
    const int tok = prof_begin(ix, PROF_MERGE, 1, st);
#define SIVF_MTC(E_)                                                                               \
    launch_pdl(k_merge_tc<E_>, blocks, MT_NT, 0, st, s.qrun, nq, nphase, Kc, RK, s.thr, s.part_n,  \
               s.part_d, s.part_i, out_d, out_s)
    if (Kc <= 32) SIVF_MTC(1);
    else if (Kc <= 64) SIVF_MTC(2);
    else if (Kc <= 128) SIVF_MTC(4);
    else if (Kc <= 256) SIVF_MTC(8);
    else SIVF_MTC(16);
#undef SIVF_MTC
    prof_end(ix, tok, st);
}

// ---------------------------------------------------------------- re-rank
// The per-query merge and the re-rank in one warp per query (K' <= 128):
// merge_select leaves the query's best K' (distance, slot) entries in shared
// memory, and the warp computes those slots' FP32 direct-form distances (eight
// lanes per candidate row, RK_UNR rounds of four, the query in registers),
// so the candidate lists never go through global memory and nothing sorts
// them by approximate distance.
// rounds of four candidate rows per warp batch of the re-ranks that run with
// more resident warps (fused merge + re-rank, wide re-rank)
constexpr int RR_UNR = 2;
// d <= 128: nine blocks of four warps per SM (at most 56 registers, no
// spills), 5,472 resident warps, so 10,000 queries take two waves instead of
// the three of eight blocks (0.062 -> 0.052 ms, same results)
template <int E, int NQ>
__global__ __launch_bounds__(MT_NT, NQ <= 4 ? 9 : 2) void k_merge_rerank(
    const int2 *__restrict__ qrun, int64_t nq, int nphase, int K, int RK,
    const float *__restrict__ thr, const int32_t *__restrict__ part_n,
    const float *__restrict__ part_d, const int64_t *__restrict__ part_i,
    const float *__restrict__ q, int d,
    const float *__restrict__ x32, const int64_t *__restrict__ ids, int k,
    float *__restrict__ dist, int64_t *__restrict__ labels)
{
    pdl_begin();
    constexpr int NW = MT_NT / 32;
    __shared__ uint32_t hist_s[NW][TC_HIST];
    // the selection's buffer; once 32 E are left, their ids and sort keys behind
    __shared__ __align__(16) float sd[NW][160 * E > merge_cap(E) ? 160 * E : merge_cap(E)];
    __shared__ int32_t ss[NW][merge_cap(E)];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 3, t = lane & 7;
    const int64_t qi = (blockIdx.x * (int64_t)MT_NT + threadIdx.x) >> 5;
    if (qi >= nq) return;  // whole warps
    const int nk = merge_select<E>(qrun, nq, qi, nphase, K, RK, thr[qi], part_n, part_d, part_i,
                                   hist_s[warp], sd[warp], ss[warp], lane);
    // the ids of the candidates, read now and used by the sort
    int64_t *sid = reinterpret_cast<int64_t *>(sd[warp] + 32 * E);
    for (int c = lane; c < nk; c += 32) sid[c] = __ldg(ids + ss[warp][c]);
    const int n4 = d >> 2;
    const float4 *q4 = reinterpret_cast<const float4 *>(q + (size_t)qi * d);
    float4 qv[NQ];
#pragma unroll
    for (int u = 0; u < NQ; ++u)
        qv[u] = t + 8 * u < n4 ? __ldg(q4 + t + 8 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 *x4 = reinterpret_cast<const float4 *>(x32);
    for (int c0 = 0; c0 < nk; c0 += 4 * RR_UNR) {
        float4 xv[RR_UNR][NQ];
        int64_t gs[RR_UNR];
#pragma unroll
        for (int r = 0; r < RR_UNR; ++r) {
            const int c = c0 + 4 * r + g;
            gs[r] = c < nk ? (int64_t)ss[warp][c] : -1;
#pragma unroll
            for (int u = 0; u < NQ; ++u)
                xv[r][u] = gs[r] >= 0 && t + 8 * u < n4 ? __ldg(x4 + gs[r] * n4 + t + 8 * u)
                                                       : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int r = 0; r < RR_UNR; ++r) {
            float acc = 0.f;
#pragma unroll
            for (int u = 0; u < NQ; ++u) {
                float dd = qv[u].x - xv[r][u].x;
                acc = fmaf(dd, dd, acc);
                dd = qv[u].y - xv[r][u].y;
                acc = fmaf(dd, dd, acc);
                dd = qv[u].z - xv[r][u].z;
                acc = fmaf(dd, dd, acc);
                dd = qv[u].w - xv[r][u].w;
                acc = fmaf(dd, dd, acc);
            }
            acc += __shfl_xor_sync(0xffffffffu, acc, 4);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            const int c = c0 + 4 * r + g;
            __syncwarp();
            if (t == 0 && c < nk) sd[warp][c] = acc;  // the approximate distance is no longer needed
        }
    }
    __syncwarp();
    warp_order<E>(
        nk, [&](int c) { return sd[warp][c]; }, [&](int c) { return sid[c]; },
        [&](int i, float v, int64_t id) {
            if (i >= k) return;
            dist[qi * k + i] = v;
            labels[qi * k + i] = id;
        },
        reinterpret_cast<uint64_t *>(sid + 32 * E), lane);
    for (int i = nk + lane; i < k; i += 32) {
        dist[qi * k + i] = INFINITY;
        labels[qi * k + i] = -1;
    }
}

// Merge and re-rank with one block per query (K' <= 512; deep sets, and few
// queries).  The entries of the query's runs at or below its bound are
// gathered into shared memory (four runs at a time or more) and reduced to the best K' by a block-wide radix
// select on the 64-bit (distance, slot) keys, also whenever the buffer could
// overflow; then the block's warps compute the candidates' exact FP32
// direct-form distances (eight lanes per candidate row with 16-byte loads,
// RR_UNR rounds of four rows per warp loaded before they are reduced, the
// query in registers), and the block sorts them by (distance, id) with a
// bitonic network and writes the best k.  Two rounds per batch keep the
// registers low enough for four blocks per SM: the gather is bound by loads
// in flight, i.e. by resident warps.  A warp per query for the merge, its
// sorted candidates through global memory, took 301 + 582 us for 10,000
// queries at K' = 400; fused 571 us (the rows alone: 230 us of HBM).
constexpr int RR_NT = 256;
constexpr int RR_MAX = 512;
constexpr int RR_CAP = 2048;  // gathered entries: at most 4 RR_NT more than K' at once

// the K smallest of the n > K entries sd / ss, in place and unsorted (whole
// block; n <= RR_CAP); returns the largest distance kept
__device__ float block_reduce_k(float *sd, int32_t *ss, int n, int K, uint32_t *hist)
{
    constexpr int PT = RR_CAP / RR_NT;
    __shared__ unsigned long long s_min, s_max, s_prefix;
    __shared__ uint32_t s_need, s_cnt;
    __shared__ int s_n, s_top;
    const int tid = threadIdx.x, lane = tid & 31;
    uint64_t key[PT];
    uint64_t kmin = ~0ull, kmax = 0ull;
#pragma unroll
    for (int e = 0; e < PT; ++e) {
        const int i = tid + e * RR_NT;
        key[e] = i < n ? ds_key(sd[i], ss[i]) : ~0ull;
        if (i < n) {
            kmin = min(kmin, key[e]);
            kmax = max(kmax, key[e]);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        kmin = min(kmin, (uint64_t)__shfl_xor_sync(0xffffffffu, (unsigned long long)kmin, o));
        kmax = max(kmax, (uint64_t)__shfl_xor_sync(0xffffffffu, (unsigned long long)kmax, o));
    }
    if (tid == 0) {
        s_min = ~0ull;
        s_max = 0ull;
        s_n = 0;
        s_top = 0;
    }
    __syncthreads();
    if (lane == 0) {
        atomicMin(&s_min, (unsigned long long)kmin);
        atomicMax(&s_max, (unsigned long long)kmax);
    }
    __syncthreads();
    const uint64_t diff = s_min ^ s_max;
    const int top = diff ? 63 - __clzll((long long)diff) : 0;
    uint64_t mask = top >= 63 ? 0ull : ~((2ull << top) - 1ull), prefix = s_min & mask;
    uint32_t need = (uint32_t)K;
    for (int hi = top; hi >= 0; hi -= 8) {
        const int shift = max(hi - 7, 0);
        const uint32_t bmask = (1u << (hi - shift + 1)) - 1u;
        hist[tid] = 0u;  // RR_NT bins
        __syncthreads();
#pragma unroll
        for (int e = 0; e < PT; ++e)
            if (tid + e * RR_NT < n && (key[e] & mask) == prefix)
                atomicAdd(&hist[(uint32_t)(key[e] >> shift) & bmask], 1u);
        __syncthreads();
        if (tid < 32) {
            uint32_t loc[8], sum = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                loc[k] = hist[lane * 8 + k];
                sum += loc[k];
            }
            uint32_t incl = sum;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            uint32_t cum = incl - sum;
            if (cum < need && incl >= need)
                for (int k = 0; k < 8; ++k) {
                    if (cum + loc[k] >= need) {
                        s_prefix = prefix | ((uint64_t)(lane * 8 + k) << shift);
                        s_need = need - cum;
                        s_cnt = loc[k];
                        break;
                    }
                    cum += loc[k];
                }
        }
        __syncthreads();
        prefix = s_prefix;
        need = s_need;
        mask |= (uint64_t)bmask << shift;
        if (s_cnt == need) break;
    }
    // every entry is in registers: the kept ones go back to the front
    uint32_t kk = 0u;
#pragma unroll
    for (int e = 0; e < PT; ++e) {
        const bool take = tid + e * RR_NT < n && (key[e] & mask) <= prefix;
        const uint32_t mk = __ballot_sync(0xffffffffu, take);
        int base = 0;
        if (lane == 0 && mk) base = atomicAdd(&s_n, __popc(mk));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (take) {
            const int p = base + __popc(mk & lanemask_lt());
            sd[p] = fkey_inv((uint32_t)(key[e] >> 32));
            ss[p] = (int32_t)(uint32_t)key[e];
            kk = max(kk, (uint32_t)(key[e] >> 32));
        }
    }
    kk = __reduce_max_sync(0xffffffffu, kk);
    if (lane == 0) atomicMax(reinterpret_cast<uint32_t *>(&s_top), kk);
    __syncthreads();
    return fkey_inv((uint32_t)s_top);
}

template <int NQ>  // 16-byte chunks of the row per lane (d <= 32 NQ)
__global__ __launch_bounds__(RR_NT, NQ <= 4 ? 4 : 1) void k_merge_rerank_wide(
    const int2 *__restrict__ qrun, int64_t nq, int nphase, int K, int RK, int tpr,
    const float *__restrict__ thr, const int32_t *__restrict__ part_n,
    const float *__restrict__ part_d, const int64_t *__restrict__ part_i,
    const float *__restrict__ q, int d, const float *__restrict__ x32,
    const int64_t *__restrict__ ids, int k, float *__restrict__ dist, int64_t *__restrict__ labels)
{
    pdl_begin();
    __shared__ __align__(16) float sd[RR_CAP];
    __shared__ int32_t ss[RR_CAP];
    __shared__ int64_t si[RR_MAX];
    __shared__ uint32_t hist[RR_NT];
    __shared__ int s_have;
    const int64_t qi = blockIdx.x;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 3, t = lane & 7;
    const int64_t PAD = 0x7fffffffffffffffLL;  // pads sort after every id
    const int n4 = d >> 2;
    const float4 *q4 = reinterpret_cast<const float4 *>(q + (size_t)qi * d);
    const float4 *x4 = reinterpret_cast<const float4 *>(x32);
    const int2 r0 = qrun[qi];
    const int2 r1 = nphase > 1 ? qrun[nq + qi] : make_int2(0, 0);
    const int NR = r0.y + r1.y;
    auto run_of = [&](int r) -> int64_t { return r < r0.y ? r0.x + r : r1.x + (r - r0.y); };
    float bound = thr[qi];
    if (tid == 0) s_have = 0;
    __syncthreads();
    int have = 0;  // uniform over the block
    // tpr threads read a run, 4 RR_NT / tpr runs at a time; the next ones'
    // counts are read meanwhile
    const int rw = RR_NT / tpr, j = tid % tpr, rj = tid / tpr;
    int cn[4];
    auto counts = [&](int rb) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
            cn[r] = rb + r * rw + rj < NR ? min(part_n[run_of(rb + r * rw + rj)], RK) : 0;
    };
    counts(0);
    for (int rb = 0; rb < NR; rb += 4 * rw) {
        int c[4];
        int64_t base[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            c[r] = cn[r];
            base[r] = c[r] > 0 ? run_of(rb + r * rw + rj) * RK : 0;
        }
        counts(rb + 4 * rw);
        for (int j0 = 0; j0 < RK; j0 += tpr) {
            if (have > RR_CAP - 4 * RR_NT) {
                bound = fminf(bound, block_reduce_k(sd, ss, have, K, hist));
                have = K;
                if (tid == 0) s_have = K;
                __syncthreads();
            }
            float dv[4];
            int32_t sv[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const bool ok = j0 + j < c[r];
                dv[r] = ok ? part_d[base[r] + j0 + j] : INFINITY;
                sv[r] = ok ? (int32_t)part_i[base[r] + j0 + j] : -1;
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const bool in = sv[r] >= 0 && dv[r] <= bound;
                const uint32_t mk = __ballot_sync(0xffffffffu, in);
                int b = 0;
                if (lane == 0 && mk) b = atomicAdd(&s_have, __popc(mk));
                b = __shfl_sync(0xffffffffu, b, 0);
                if (in) {
                    const int p = b + __popc(mk & lanemask_lt());
                    sd[p] = dv[r];
                    ss[p] = sv[r];
                }
            }
            __syncthreads();
            have = s_have;
            __syncthreads();  // every thread has read it before it grows again
        }
    }
    if (have > K) {
        block_reduce_k(sd, ss, have, K, hist);
        have = K;
    }
    float4 qv[NQ];
#pragma unroll
    for (int u = 0; u < NQ; ++u)
        qv[u] = t + 8 * u < n4 ? __ldg(q4 + t + 8 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
    int N = 32;
    while (N < have) N <<= 1;  // <= RR_MAX
    constexpr int CPW = 4 * RR_UNR;  // candidates per warp and batch
    for (int c0 = warp * CPW; c0 < N; c0 += (RR_NT / 32) * CPW) {
        float4 xv[RR_UNR][NQ];
        int64_t gs[RR_UNR];
#pragma unroll
        for (int r = 0; r < RR_UNR; ++r) {
            const int c = c0 + 4 * r + g;
            gs[r] = c < have ? (int64_t)ss[c] : -1;
#pragma unroll
            for (int u = 0; u < NQ; ++u)
                xv[r][u] = gs[r] >= 0 && t + 8 * u < n4 ? __ldg(x4 + gs[r] * n4 + t + 8 * u)
                                                       : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int r = 0; r < RR_UNR; ++r) {
            float acc = 0.f;
#pragma unroll
            for (int u = 0; u < NQ; ++u) {
                float dd = qv[u].x - xv[r][u].x;
                acc = fmaf(dd, dd, acc);
                dd = qv[u].y - xv[r][u].y;
                acc = fmaf(dd, dd, acc);
                dd = qv[u].z - xv[r][u].z;
                acc = fmaf(dd, dd, acc);
                dd = qv[u].w - xv[r][u].w;
                acc = fmaf(dd, dd, acc);
            }
            acc += __shfl_xor_sync(0xffffffffu, acc, 4);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            const int c = c0 + 4 * r + g;
            if (t == 0 && c < N) {
                sd[c] = gs[r] >= 0 ? acc : INFINITY;  // the approximate one is no longer needed
                si[c] = gs[r] >= 0 ? __ldg(ids + gs[r]) : PAD;
            }
        }
    }
    __syncthreads();
    // sort by exact distance: 64-bit keys (distance, place), two per thread,
    // exchanged by shuffles within a warp and through shared memory beyond
    // (every stage through shared memory with the ids took as long as the rows'
    // gather); equal distances are ranked by id below
    uint64_t ky[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int i = tid + e * RR_NT;
        ky[e] = i < N && si[i] != PAD ? ((uint64_t)fkey(sd[i]) << 32) | (uint32_t)i : ~0ull;
    }
    __syncthreads();
    uint64_t *xk = reinterpret_cast<uint64_t *>(sd);  // RR_MAX keys
    for (int size = 2; size <= N; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride == RR_NT) {  // size = 512: ascending
                const uint64_t a = min(ky[0], ky[1]), b = max(ky[0], ky[1]);
                ky[0] = a;
                ky[1] = b;
                continue;
            }
            uint64_t o[2];
            if (stride >= 32) {
#pragma unroll
                for (int e = 0; e < 2; ++e) xk[tid + e * RR_NT] = ky[e];
                __syncthreads();
#pragma unroll
                for (int e = 0; e < 2; ++e) o[e] = xk[(tid ^ stride) + e * RR_NT];
                __syncthreads();
            } else {
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    o[e] = __shfl_xor_sync(0xffffffffu, (unsigned long long)ky[e], stride);
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const bool up = ((tid + e * RR_NT) & size) == 0, lower = (tid & stride) == 0;
                ky[e] = lower == up ? min(ky[e], o[e]) : max(ky[e], o[e]);
            }
        }
#pragma unroll
    for (int e = 0; e < 2; ++e) xk[tid + e * RR_NT] = ky[e];
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int i = tid + e * RR_NT;
        if (i >= N) continue;
        const uint64_t me = ky[e];
        if (me == ~0ull) {
            if (i < k) {
                dist[qi * k + i] = INFINITY;
                labels[qi * k + i] = -1;
            }
            continue;
        }
        const uint32_t dk = (uint32_t)(me >> 32);
        const int64_t id = si[(uint32_t)me];
        int pos = i;  // among equal distances: by id
        for (int j = i - 1; j >= 0 && (uint32_t)(xk[j] >> 32) == dk; --j)
            pos -= si[(uint32_t)xk[j]] > id;
        for (int j = i + 1; j < N && (uint32_t)(xk[j] >> 32) == dk && xk[j] != ~0ull; ++j)
            pos += si[(uint32_t)xk[j]] < id;
        if (pos < k) {
            dist[qi * k + pos] = fkey_inv(dk);
            labels[qi * k + pos] = id;
        }
    }
    for (int i = N + tid; i < k; i += RR_NT) {  // fewer candidates than k
        dist[qi * k + i] = INFINITY;
        labels[qi * k + i] = -1;
    }
}

// per query (BF16 form): FP32 ||q||^2, unit scale, and the row rounded to
// BF16 (round to nearest even).  The FP8 form codes each (query, probe)
// pair instead (k_pair_prep).
__global__ void k_query_prep(const float *__restrict__ q, int64_t nq, int d,
                             float *__restrict__ qn, float *__restrict__ qsc,
                             unsigned char *__restrict__ qcast)
{
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (i >= nq) return;
    const float *qr = q + (size_t)i * d;
    float ss = 0.f;
    __nv_bfloat16 *o = reinterpret_cast<__nv_bfloat16 *>(qcast) + (size_t)i * d;
    for (int j = lane; j < d; j += 32) {
        const float v = qr[j];
        ss = fmaf(v, v, ss);
        o[j] = __float2bfloat16_rn(v);
    }
    ss = warp_sum(ss);
    if (lane == 0) {
        qn[i] = ss;
        qsc[i] = 1.f;
    }
}

void query_prep(sivf_index *ix, const float *q, int64_t nq, float *qn, float *qsc,
                unsigned char *qcast, cudaStream_t st)
{
    ix->launches += 1;
    launch_pdl(k_query_prep, (unsigned)((nq * 32 + 255) / 256), 256, 0, st, q, nq, ix->d, qn, qsc,
               qcast);
}

// FP8 residual scan: per (query, probe) pair e = q * P + p with list l =
// probes[e]: the residual r = fl32(q - c_l), ||r||^2 (FP32), its inverse
// scale 448 / (2 max_j |r_j|) (1 when r = 0) and the row E4M3(fl32(r_j *
// scale)) (round to nearest even, saturated).  One warp per pair; pairs with
// no list are left untouched (they are never scanned).
constexpr int PP_V4 = 2;  // float4 of the residual per lane (d <= 256)
__global__ void k_pair_prep(const float *__restrict__ q, int64_t npairs, int P, int p1, int d, int L,
                            const int32_t *__restrict__ probes, const float *__restrict__ cent,
                            float *__restrict__ qn, float *__restrict__ qsc,
                            unsigned char *__restrict__ qcast)
{
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (t >= npairs) return;
    const int64_t e = (t / p1) * P + t % p1;
    const int l = probes[e];
    if (l < 0 || l >= L) return;
    const float *qr = q + (size_t)(e / P) * d;
    const float *cl = cent + (size_t)l * d;
    unsigned char *o = qcast + (size_t)e * d;
    float ss = 0.f, mx = 0.f;
    if ((d & 3) == 0 && d <= 32 * 4 * PP_V4) {
        // the residual held in registers, one float4 per lane and round
        const int n4 = d >> 2;
        float4 r4[PP_V4];
#pragma unroll
        for (int u = 0; u < PP_V4; ++u) {
            const int j4 = lane + 32 * u;
            r4[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j4 < n4) {
                const float4 a = __ldg(reinterpret_cast<const float4 *>(qr) + j4);
                const float4 b = __ldg(reinterpret_cast<const float4 *>(cl) + j4);
                r4[u] = make_float4(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y),
                                    __fsub_rn(a.z, b.z), __fsub_rn(a.w, b.w));
            }
            ss = fmaf(r4[u].x, r4[u].x, ss);
            ss = fmaf(r4[u].y, r4[u].y, ss);
            ss = fmaf(r4[u].z, r4[u].z, ss);
            ss = fmaf(r4[u].w, r4[u].w, ss);
            mx = fmaxf(mx, fmaxf(fmaxf(fabsf(r4[u].x), fabsf(r4[u].y)),
                                 fmaxf(fabsf(r4[u].z), fabsf(r4[u].w))));
        }
        ss = warp_sum(ss);
        for (int o2 = 16; o2 > 0; o2 >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o2));
        const float sc = mx > 0.f ? 448.f / (2.f * mx) : 1.f;
        if (lane == 0) {
            qn[e] = ss;
            qsc[e] = sc;
        }
#pragma unroll
        for (int u = 0; u < PP_V4; ++u) {
            const int j4 = lane + 32 * u;
            if (j4 >= n4) break;
            const uint32_t lo = __nv_cvt_float2_to_fp8x2(
                make_float2(__fmul_rn(r4[u].x, sc), __fmul_rn(r4[u].y, sc)), __NV_SATFINITE, __NV_E4M3);
            const uint32_t hi = __nv_cvt_float2_to_fp8x2(
                make_float2(__fmul_rn(r4[u].z, sc), __fmul_rn(r4[u].w, sc)), __NV_SATFINITE, __NV_E4M3);
            reinterpret_cast<uint32_t *>(o)[j4] = (lo & 0xffffu) | (hi << 16);
        }
        return;
    }
    for (int j = lane; j < d; j += 32) {
        const float r = __fsub_rn(qr[j], cl[j]);
        ss = fmaf(r, r, ss);
        mx = fmaxf(mx, fabsf(r));
    }
    ss = warp_sum(ss);
    for (int o2 = 16; o2 > 0; o2 >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o2));
    const float sc = mx > 0.f ? 448.f / (2.f * mx) : 1.f;
    if (lane == 0) {
        qn[e] = ss;
        qsc[e] = sc;
    }
    for (int j = 2 * lane; j < d; j += 64) {
        const float2 p = make_float2(__fmul_rn(__fsub_rn(qr[j], cl[j]), sc),
                                     __fmul_rn(__fsub_rn(qr[j + 1], cl[j + 1]), sc));
        const uint32_t two = __nv_cvt_float2_to_fp8x2(p, __NV_SATFINITE, __NV_E4M3);
        o[j] = (unsigned char)(two & 0xffu);
        o[j + 1] = (unsigned char)(two >> 8);
    }
}

void pair_prep(sivf_index *ix, const float *q, int64_t nq, int P, int p1, const int32_t *probes,
               float *qn, float *qsc, unsigned char *qcast, cudaStream_t st)
{
    ix->launches += 1;
    const int64_t np = nq * p1;
    launch_pdl(k_pair_prep, (unsigned)((np * 32 + 255) / 256), 256, 0, st, q, np, P, p1, ix->d,
               ix->nlist, probes, ix->cent, qn, qsc, qcast);
}

// global slots -> labels (padding stays -1)
__global__ void k_slots_to_ids(int64_t *v, int64_t n, const int64_t *__restrict__ ids)
{
    pdl_begin();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        if (v[i] >= 0) v[i] = ids[v[i]];
}

void slots_to_ids(sivf_index *ix, int64_t *v, int64_t n, cudaStream_t st)
{
    ix->launches += 1;
    launch_pdl(k_slots_to_ids, (unsigned)std::min<int64_t>((n + 255) / 256, 152 * 8), 256, 0,
               st, v, n, ix->ids);
}

// --------------------------------------------------------------- host side
PFN_cuTensorMapEncodeTiled_v12000 tmap_encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        cudaDriverEntryPointQueryResult q;
        void *p = nullptr;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

bool tc_make_maps(sivf_index *ix)
{
    auto enc = tmap_encode_fn();
    if (!enc) return false;
    const cuuint64_t rows = (cuuint64_t)ix->n_slabs * ix->C;
    if (ix->xb16) {
        cuuint64_t dims[2] = {(cuuint64_t)ix->d, rows};
        cuuint64_t strides[1] = {(cuuint64_t)ix->d * 2};
        cuuint32_t box[2] = {64, (cuuint32_t)ix->C};
        cuuint32_t es[2] = {1, 1};
        if (enc(reinterpret_cast<CUtensorMap *>(ix->tmap_bf16), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                ix->xb16, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    if (ix->x8) {
        cuuint64_t dims[2] = {(cuuint64_t)ix->d, rows};
        cuuint64_t strides[1] = {(cuuint64_t)ix->d};
        cuuint32_t box[2] = {128, (cuuint32_t)ix->C};
        cuuint32_t es[2] = {1, 1};
        if (enc(reinterpret_cast<CUtensorMap *>(ix->tmap_fp8), CU_TENSOR_MAP_DATA_TYPE_UINT8, 2,
                ix->x8, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    // 128-row boxes for tiles whose slabs are consecutive in the pool
    ix->tmap_tile_ok = false;
    if (ix->C < TC_M && TC_M % ix->C == 0) {
        bool ok = true;
        if (ix->xb16) {
            cuuint64_t dims[2] = {(cuuint64_t)ix->d, rows};
            cuuint64_t strides[1] = {(cuuint64_t)ix->d * 2};
            cuuint32_t box[2] = {64, (cuuint32_t)TC_M};
            cuuint32_t es[2] = {1, 1};
            ok = ok && enc(reinterpret_cast<CUtensorMap *>(ix->tmap_bf16_t),
                           CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ix->xb16, dims, strides, box, es,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        }
        if (ix->x8) {
            cuuint64_t dims[2] = {(cuuint64_t)ix->d, rows};
            cuuint64_t strides[1] = {(cuuint64_t)ix->d};
            cuuint32_t box[2] = {128, (cuuint32_t)TC_M};
            cuuint32_t es[2] = {1, 1};
            ok = ok && enc(reinterpret_cast<CUtensorMap *>(ix->tmap_fp8_t),
                           CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, ix->x8, dims, strides, box, es,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        }
        ix->tmap_tile_ok = ok;
    }
    return qt_make_maps(ix, enc);
}

// a row's run and held set: K' plus the room an approximate reduction may
// keep beyond it (a quarter of K', at least 32), a multiple of 8
int tc_run_len(int K) { return (K + max(32, K / 4) + 7) / 8 * 8; }

// a row's candidate buffer: its held set plus room for `tiles` tiles of
// candidates (TC_M each)
static int tc_buf_len(int K, int tiles) { return tc_run_len(K) + tiles * TC_M; }

// queries per tile of the reduced-precision scan for K' candidates
int tc_tile_queries(int Kc)
{
    return Kc <= TcShape<48>::KMAX ? 48 : Kc <= TcShape<32>::KMAX ? 32 : 16;
}

// dynamic shared memory one CTA may take (the kernel's static arrays aside)
constexpr size_t kTcSmemMax = 227 * 1024 - 4096;

template <int TN>
static int tc_stages(int KC, int M)
{
    int nst = TC_MAXST;
    while (nst > 2 && tc_smem<TN>(KC, M, nst).total > kTcSmemMax) --nst;
    return nst;
}

static size_t tc_total(int tn, int KC, int M, int nst)
{
    switch (tn) {
    case 48: return tc_smem<48>(KC, M, nst).total;
    case 32: return tc_smem<32>(KC, M, nst).total;
    default: return tc_smem<16>(KC, M, nst).total;
    }
}

// Entries of a row's candidate buffer.  A row folds its pending candidates
// into its best K' once more than FT = room - step of them wait (for K' <= 128
// at most 96), a step being what is appended between two checks: a round of TP
// tiles, or a whole group of accumulators where an item runs without checks.
// With room for one step any candidate at all costs a fold; the default takes
// room for three tiles (K' > 128) or two where three A stages still fit beside
// it, else one.  sel > 0 asks for sel tiles of room.
int tc_buf_entries(const sivf_index *ix, int dtype, int Kc, int sel)
{
    if (sel > 0) return tc_buf_len(Kc, sel);
    const int esz = dtype == SIVF_BF16 ? 2 : 1;
    const int KC = (ix->d * esz + 127) / 128;
    const int tn = tc_tile_queries(Kc);
    // K' > 128: three tiles of room where they fit, so a fold (dominated by
    // the held K') comes every third tile while no bound prunes
    if (Kc > 128 && tc_total(tn, KC, tc_buf_len(Kc, 3), 3) <= kTcSmemMax)
        return tc_buf_len(Kc, 3);
    if (tc_total(tn, KC, tc_buf_len(Kc, 2), 3) <= kTcSmemMax) return tc_buf_len(Kc, 2);
    return tc_buf_len(Kc, 1);
}

// a buffer of M entries fits beside two A stages
bool tc_buf_fits(const sivf_index *ix, int dtype, int Kc, int M)
{
    const int esz = dtype == SIVF_BF16 ? 2 : 1;
    const int KC = (ix->d * esz + 127) / 128;
    const int tn = tc_tile_queries(Kc);
    return (tn != 16 || Kc <= TcShape<16>::KMAX) && tc_total(tn, KC, M, 2) <= kTcSmemMax;
}

int tc_wide_entries(const sivf_index *ix, int dtype, int Kc)
{
    if (Kc <= TcShape<32>::KMAX || Kc > TcShape<16>::KMAX) return 0;
    const int esz = dtype == SIVF_BF16 ? 2 : 1;
    const int KC = (ix->d * esz + 127) / 128;
    const int M = tc_buf_len(Kc, 1);
    return tc_smem<32>(KC, M, 2).total <= kTcSmemMax ? M : 0;
}

bool tc_fits(const sivf_index *ix, int Kc)
{
    const int esz = 2;  // the larger of the two formats
    const int KC = (ix->d * esz + 127) / 128;
    const int M = tc_buf_len(Kc, 1);
    switch (tc_tile_queries(Kc)) {
    case 48: return tc_smem<48>(KC, M, 2).total <= kTcSmemMax;
    case 32: return tc_smem<32>(KC, M, 2).total <= kTcSmemMax;
    default: return Kc <= TcShape<16>::KMAX && tc_smem<16>(KC, M, 2).total <= kTcSmemMax;
    }
}

template <int DT, int TN>
static void launch_tc(const unsigned char *tmap, const unsigned char *tmap_t, TcArgs a,
                      cudaStream_t st)
{
    a.nst = tc_stages<TN>(a.KC, a.M);
    const size_t smem = tc_smem<TN>(a.KC, a.M, a.nst).total;
    static KernelSetup su;
    opt_in_smem(su, k_scan_tc<DT, TN>, smem);
    launch_pdl(k_scan_tc<DT, TN>, 152, TcShape<TN>::NT, smem, st,
               *reinterpret_cast<const CUtensorMap *>(tmap),
               *reinterpret_cast<const CUtensorMap *>(tmap_t), a);
}

void scan_lists_tc(sivf_index *ix, int dtype, const float *q, int64_t nq, int P, int Kc,
                   const SearchPlan &pl, const SearchScratch &s, cudaStream_t st, int seed_slabs)
{
    TcArgs a;
    a.q = q;
    a.nq = nq;
    a.P = P;
    a.K = Kc;
    a.M = pl.M;
    a.prun = s.prun;
    a.qlist = s.qlist;
    a.loff = s.loff;
    a.lcnt = s.lcnt;
    a.nch = s.nch;
    a.part_d = s.part_d;
    a.part_i = s.part_i;
    a.part_n = s.part_n;
    a.RK = pl.RK;
    a.thr = s.thr;
    a.items = s.items;
    a.per_pair = dtype == SIVF_FP8E4M3;
    a.qn = a.per_pair ? s.pqn : s.qn;
    a.qsc = a.per_pair ? s.pqsc : s.qsc;
    a.qcast = s.qcast;
    a.xnorm = a.per_pair ? ix->rnorm : ix->xnorm;
    a.bits = ix->bits;
    a.nslabs = ix->nslabs;
    a.dir = ix->dir;
    a.inv_scale8 = ix->inv_scale8;
    a.n_slabs = ix->n_slabs;
    a.dir_cap = ix->dir_cap;
    a.L = ix->nlist;
    a.d = ix->d;
    a.C = ix->C;
    const int esz = dtype == SIVF_BF16 ? 2 : 1;
    a.pay = dtype == SIVF_BF16 ? reinterpret_cast<const unsigned char *>(ix->xb16) : ix->x8;
    a.KC = (ix->d * esz + 127) / 128;
    a.nst = 2;
    a.pf_tiles = std::max(2, TC_PF_BYTES / (TC_M * ix->d * esz));
    a.tile_box = ix->tmap_tile_ok ? 1 : 0;
    a.ctl = ix->ctl;
    a.err = ix->err;
    a.seed_slabs = seed_slabs;
    a.wait_ns = ix->wait_ns;
    const int tn = pl.tq;  // the plan's tile: 48 / 32 / 16 (tc_tile_queries), 32 wide
    const int tok = prof_begin(ix, PROF_SCAN, 1, st);
    if (dtype == SIVF_BF16) {
        if (tn == 48) launch_tc<0, 48>(ix->tmap_bf16, ix->tmap_bf16_t, a, st);
        else if (tn == 32) launch_tc<0, 32>(ix->tmap_bf16, ix->tmap_bf16_t, a, st);
        else launch_tc<0, 16>(ix->tmap_bf16, ix->tmap_bf16_t, a, st);
    } else {
        if (tn == 48) launch_tc<1, 48>(ix->tmap_fp8, ix->tmap_fp8_t, a, st);
        else if (tn == 32) launch_tc<1, 32>(ix->tmap_fp8, ix->tmap_fp8_t, a, st);
        else launch_tc<1, 16>(ix->tmap_fp8, ix->tmap_fp8_t, a, st);
    }
    prof_end(ix, tok, st);
}

// merge and re-rank of a search: a block per query for K' > 128 and for few
// queries (one wave of blocks: a warp's chain of loads over the chunked lists'
// runs takes 40 us however few the queries are, a block's 24; 1,000 queries
// 41 against 46 us), else a warp each
void merge_rerank(sivf_index *ix, const float *q, int64_t nq, int nphase,
                  const SearchScratch &s, int Kc, int RK, int k, float *dist, int64_t *labels,
                  cudaStream_t st)
{
    if (Kc > 128 || nq <= 4 * 152) {
        const int tok = prof_begin(ix, PROF_RERANK, 1, st);
        const int tpr = RK <= 64 ? 64 : RK <= 128 ? 128 : RR_NT;
        auto go = [&](auto kern) {
            launch_pdl(kern, (unsigned)nq, RR_NT, 0, st, s.qrun, nq, nphase, Kc, RK, tpr, s.thr, s.part_n,
                       s.part_d, s.part_i, q, ix->d, ix->x32, ix->ids, k, dist, labels);
        };
        if (ix->d > 128) go(&k_merge_rerank_wide<8>);
        else go(&k_merge_rerank_wide<4>);
        prof_end(ix, tok, st);
        return;
    }
    const unsigned blocks = (unsigned)((nq * 32 + MT_NT - 1) / MT_NT);
    const int tok = prof_begin(ix, PROF_RERANK, 1, st);
#define SIVF_MRR(E_, NQ_)                                                                          \
    launch_pdl(k_merge_rerank<E_, NQ_>, blocks, MT_NT, 0, st, s.qrun, nq, nphase, Kc, RK, s.thr,   \
               s.part_n, s.part_d, s.part_i, q, ix->d, ix->x32, ix->ids, k, dist,                  \
               labels)
    const bool wide = ix->d > 128;
    if (Kc <= 32) {
        if (wide) SIVF_MRR(1, 8);
        else SIVF_MRR(1, 4);
    } else if (Kc <= 64) {
        if (wide) SIVF_MRR(2, 8);
        else SIVF_MRR(2, 4);
    } else {
        if (wide) SIVF_MRR(4, 8);
        else SIVF_MRR(4, 4);
    }
#undef SIVF_MRR
    prof_end(ix, tok, st);
}

}  // namespace sivf
