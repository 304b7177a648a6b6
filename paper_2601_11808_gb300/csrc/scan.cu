// List scan and top-k of the search (Algorithm 3, redone list-centrically).
//
// Algorithm 3 gives one warp to one query and walks each probed list's slab
// chain.  Here the (query, list) pairs of a whole batch are first grouped by
// list, and one CTA scans one list for a tile of up to TQ queries: every slab
// of the list is read from HBM once per tile instead of once per query, and
// the list's slabs come from its directory, so the next slabs are fetched
// (whole, by one bulk copy each, into shared memory) while the current one
// is being scored.  Distances are the direct form sum_j (q_j - x_j)^2 in
// FP32 (the paper's metric, squared L2).  A slot is read only when its
// validity bit is set (Theorem 2).  Each (query, list tile) keeps its best K
// (distance, id) pairs; a final merge per query keeps the best k of all
// probed lists, ties to the lower id, padded with (+inf, -1).
//
// A search of enough pairs scans each query's nearest list first and then
// only those of its other lists that may hold a vector within the distance
// the nearest left (the pair pruning below, also of the reduced-precision
// scans).
#include <math.h>

#include <cmath>

#include "device_utils.cuh"
#include "kernels.cuh"
#include "tc.cuh"

namespace sivf {

// ------------------------------------------------------ grouping by list
// pairs (q, p) with p in [p0, p1): rank of each pair inside its list group
__global__ void k_srch_hist(const int32_t *__restrict__ probes, int64_t nq, int P, int p0,
                            int p1, int L, bool dedupe, bool flagged,
                            int32_t *__restrict__ lcnt, int32_t *__restrict__ prank)
{
    pdl_begin();
    const int np = p1 - p0;
    const int64_t n = nq * np;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = (t / np) * P + p0 + t % np;
        const int l = probes[e];
        bool ok = l >= 0 && l < L && !(flagged && prank[e] < 0);
        if (ok && dedupe) {
            const int64_t q0 = (e / P) * P;
            for (int64_t f = q0; f < e; ++f)
                if (probes[f] == l) {
                    ok = false;
                    break;
                }
        }
        prank[e] = ok ? atomicAdd(&lcnt[l], 1) : -1;
    }
}

// inclusive scans of two values over the 1,024 threads of a block; `sh` is
// 64 ints of shared memory; *ta, *tb receive the totals
__device__ __forceinline__ void block_scan2(int32_t &a, int32_t &b, int32_t *sh, int32_t *ta,
                                            int32_t *tb)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t va = __shfl_up_sync(0xffffffffu, a, o), vb = __shfl_up_sync(0xffffffffu, b, o);
        if (lane >= o) {
            a += va;
            b += vb;
        }
    }
    __syncthreads();  // sh may still be read from an earlier scan
    if (lane == 31) {
        sh[w] = a;
        sh[32 + w] = b;
    }
    __syncthreads();
    if (w == 0) {
        int32_t sa = sh[lane], sb = sh[32 + lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t va = __shfl_up_sync(0xffffffffu, sa, o),
                          vb = __shfl_up_sync(0xffffffffu, sb, o);
            if (lane >= o) {
                sa += va;
                sb += vb;
            }
        }
        sh[lane] = sa;
        sh[32 + lane] = sb;
    }
    __syncthreads();
    if (w > 0) {
        a += sh[w - 1];
        b += sh[32 + w - 1];
    }
    *ta = sh[31];
    *tb = sh[63];
}

// the launch's whole work, summed over a block of 1,024 threads
__device__ __forceinline__ unsigned long long block_work(unsigned long long w,
                                                         unsigned long long *sw)
{
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = w;
    __syncthreads();
    unsigned long long W = 0;
    for (int i = 0; i < 32; ++i) W += sw[i];
    return W;
}

// Slabs a chunk has at least.  A list is cut into slab chunks so that no
// work item is longer than 1 / (ips * 152) of the launch's whole work W
// (query tiles x slabs summed over the probed lists) and no chunk is shorter
// than `spc` slabs, at most `chmax` chunks per list; a heavy list (a skewed
// distribution puts most vectors in a few lists) is spread over many SMs
// instead of holding one SM for the length of the launch.  With
// target = max(spc, ceil(W / (ips * 152))) the chunks beyond the first of
// every list add at most ips * 152 items, and at most tq * ips * 152 output
// runs, to one tile per pair: the scratch is sized from that bound.
__device__ __forceinline__ int chunk_target(unsigned long long W, int spc, int ips)
{
    const unsigned long long slots = (unsigned long long)ips * 152;
    return (int)min(max((unsigned long long)spc, (W + slots - 1) / slots), 1ull << 30);
}

// pairs scored and slab bytes streamed (per tile, and once per list)
struct ScanCount {
    unsigned long long pairs = 0, bytes = 0, ubytes = 0;
    __device__ void list(int m, int nt, int ns, int live, int64_t slab_bytes)
    {
        pairs += (unsigned long long)m * (unsigned long long)max(live, 0);
        bytes += (unsigned long long)nt * ns * slab_bytes;
        ubytes += (unsigned long long)ns * slab_bytes;
    }
    __device__ void add_to(int64_t *stat) const  // whole warps
    {
        unsigned long long v[3] = {pairs, bytes, ubytes};
        for (int i = 0; i < 3; ++i) {
            for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
            if ((threadIdx.x & 31) == 0 && v[i])
                atomicAdd(reinterpret_cast<unsigned long long *>(stat + 1 + i), v[i]);
        }
    }
};

// One block: the lists' chunks (chunk_target), then exclusive scans over the
// lists of the pair counts and of the work items.  Thread t takes the lists
// t, t + 1024, ... (their order in the groups and items is of no account), so
// that its loads are coalesced and independent: contiguous lists per thread
// took 50 us at 16,384 lists, a chain of strided loads.
constexpr int PLAN_BIG = 256;  // heavy lists taken by the block
__global__ __launch_bounds__(1024) void k_srch_plan(const int32_t *__restrict__ lcnt,
                                                    const int32_t *__restrict__ nslabs,
                                                    const int32_t *__restrict__ list_live,
                                                    int L, int tq, int chmax, int spc, int ips,
                                                    int64_t item_cap, int64_t slab_bytes,
                                                    int32_t *__restrict__ loff,
                                                    int32_t *__restrict__ nch,
                                                    int2 *__restrict__ items, Ctl *ctl,
                                                    int64_t *stat, uint32_t *err)
{
    pdl_begin();
    __shared__ int32_t sh[64];
    __shared__ unsigned long long sw[32];
    const int tid = threadIdx.x;
    unsigned long long wsum = 0;
#pragma unroll 8
    for (int l = tid; l < L; l += 1024) {
        const int m = lcnt[l], ns = nslabs[l];
        if (m > 0 && ns > 0) wsum += (unsigned long long)((m + tq - 1) / tq) * ns;
    }
    const int target = chunk_target(block_work(wsum, sw), spc, ips);
    int32_t ca = 0, cb = 0;
    ScanCount cnt;
#pragma unroll 4
    for (int l = tid; l < L; l += 1024) {
        const int m = lcnt[l], ns = nslabs[l], live = list_live[l];
        const int nt = (m + tq - 1) / tq;
        const int c = (m > 0 && ns > 0) ? min(min(chmax, max(1, (ns + target - 1) / target)), ns) : 0;
        nch[l] = c;
        ca += m;
        cb += nt * c;
        if (c) cnt.list(m, nt, ns, live, slab_bytes);
    }
    if (stat) cnt.add_to(stat);
    int32_t ea = ca, eb = cb, ta, tb;
    block_scan2(ea, eb, sh, &ta, &tb);
    ea -= ca;
    eb -= cb;
    // work items of list l: (list, tile << 8 | chunk); a heavy list's are
    // written by the whole block (one thread took 35 us for 1,750)
    __shared__ int s_big;
    __shared__ int4 big[PLAN_BIG];
    if (tid == 0) s_big = 0;
    __syncthreads();
#pragma unroll 4
    for (int l = tid; l < L; l += 1024) {
        const int m = lcnt[l], c = nch[l], nt = (m + tq - 1) / tq;
        loff[l] = ea;
        const int slot = nt * c > 16 ? atomicAdd(&s_big, 1) : PLAN_BIG;
        if (slot < PLAN_BIG) {
            big[slot] = make_int4(l, c, nt * c, eb);
        } else {
            for (int t = 0; t < nt * c; ++t)
                if (eb + t < item_cap) items[eb + t] = make_int2(l, ((t / c) << 8) | (t % c));
        }
        ea += m;
        eb += nt * c;
    }
    __syncthreads();
    for (int b = tid >> 5; b < min(s_big, PLAN_BIG); b += 32) {
        const int4 w = big[b];
        for (int t = tid & 31; t < w.z; t += 32)
            if (w.w + t < item_cap) items[w.w + t] = make_int2(w.x, ((t / w.y) << 8) | (t % w.y));
    }
    if (tid == 0) {
        if (tb > item_cap) atomicOr(err, ERR_PLAN);
        ctl->nitems = (int32_t)min((int64_t)tb, item_cap);
        ctl->nscan = ta;
        ctl->next_item = 0;
    }
}

// The whole grouping of a small launch (at most SH_PAIRS pairs, two per
// thread) in one block: count the pairs of each touched list, cut the lists
// into chunks, lay out the groups, the items and the output runs.  Pairs are
// taken in query order, so that a scan over them gives every query one
// contiguous block of runs; the lists' counts stand in a hash table in shared
// memory, so that the chain of global round trips is the probes, the slab
// counts and the stores.  It replaces a memset and three launches and looks
// only at the lists the pairs touch: 9 to 15 us for 8 to 2,000 pairs.  More
// pairs per thread are the slower way: 34 us for 7,000, the three kernels 20.
constexpr int SH_PER = 2;
constexpr int SH_PAIRS = 1024 * SH_PER;
constexpr int SH_SLOTS = 2 * SH_PAIRS;  // a power of two, at most half full
constexpr size_t SH_SMEM = (size_t)SH_SLOTS * 16 + SH_PAIRS * 8;
__global__ __launch_bounds__(1024) void k_srch_hash(
    const int32_t *__restrict__ probes, int64_t nq, int P, int p0, int p1, int L, bool dedupe,
    const int32_t *__restrict__ flags, const int32_t *__restrict__ nslabs,
    const int32_t *__restrict__ list_live, int tq, int chmax, int spc, int ips, int64_t item_cap,
    int64_t slab_bytes, int32_t *lcnt, int32_t *loff, int32_t *nch, int2 *items, int32_t *qlist,
    int32_t *prun, int2 *qrun, Ctl *ctl, int64_t run_cap, int64_t *stat, uint32_t *err)
{
    pdl_begin();
    extern __shared__ int32_t shm[];
    int32_t *key = shm, *cnt = key + SH_SLOTS, *off = cnt + SH_SLOTS, *chk = off + SH_SLOTS;
    int32_t *touched = chk + SH_SLOTS, *first = touched + SH_PAIRS;
    __shared__ int32_t sh[64];
    __shared__ unsigned long long sw[32];
    __shared__ int s_nt, s_base;
    const int tid = threadIdx.x, np = p1 - p0, n = (int)nq * np;
    const int per = (n + 1023) / 1024;  // <= SH_PER
    int ev[SH_PER], lv[SH_PER], rk[SH_PER], sl[SH_PER];
#pragma unroll
    for (int i = 0; i < SH_PER; ++i) {
        const int t = tid * per + i;
        ev[i] = i < per && t < n ? (t / np) * P + p0 + t % np : -1;
        lv[i] = ev[i] >= 0 ? probes[ev[i]] : -1;
        if (lv[i] >= L || (flags && ev[i] >= 0 && flags[ev[i]] < 0)) lv[i] = -1;
    }
    for (int i = tid; i < SH_SLOTS; i += 1024) {
        key[i] = -1;
        cnt[i] = 0;
    }
    if (tid == 0) s_nt = 0;
    if (dedupe)
#pragma unroll
        for (int i = 0; i < SH_PER; ++i) {
            if (lv[i] < 0) continue;
            for (int f = (ev[i] / P) * P; f < ev[i]; ++f)
                if (probes[f] == lv[i]) {
                    lv[i] = -1;
                    break;
                }
        }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < SH_PER; ++i) {
        rk[i] = sl[i] = 0;
        if (lv[i] < 0) continue;
        int h = (int)(((uint32_t)lv[i] * 2654435761u) >> 16) & (SH_SLOTS - 1);
        for (;;) {  // at most SH_PAIRS of the SH_SLOTS slots are taken
            const int was = atomicCAS(&key[h], -1, lv[i]);
            if (was == -1) touched[atomicAdd(&s_nt, 1)] = h;
            if (was == -1 || was == lv[i]) break;
            h = (h + 1) & (SH_SLOTS - 1);
        }
        sl[i] = h;
        rk[i] = atomicAdd(&cnt[h], 1);
    }
    __syncthreads();
    const int nt = s_nt;
    // the touched lists: chunks, groups, items
    int hj[SH_PER], ns[SH_PER], lj[SH_PER], live[SH_PER];
    unsigned long long wsum = 0;
#pragma unroll
    for (int i = 0; i < SH_PER; ++i) {
        const int j = tid + 1024 * i;
        hj[i] = j < nt ? touched[j] : -1;
        lj[i] = hj[i] >= 0 ? key[hj[i]] : 0;
        ns[i] = hj[i] >= 0 ? nslabs[lj[i]] : 0;
        live[i] = hj[i] >= 0 ? list_live[lj[i]] : 0;
    }
#pragma unroll
    for (int i = 0; i < SH_PER; ++i)
        if (hj[i] >= 0 && ns[i] > 0) wsum += (unsigned long long)((cnt[hj[i]] + tq - 1) / tq) * ns[i];
    const int target = chunk_target(block_work(wsum, sw), spc, ips);
    int32_t ca = 0, cb = 0;
    ScanCount sc;
#pragma unroll
    for (int i = 0; i < SH_PER; ++i) {
        if (hj[i] < 0) continue;
        const int m = cnt[hj[i]], k = (m + tq - 1) / tq;
        const int c = ns[i] > 0 ? min(min(chmax, max(1, (ns[i] + target - 1) / target)), ns[i]) : 0;
        chk[hj[i]] = c;
        ca += m;
        cb += k * c;
        if (c) sc.list(m, k, ns[i], live[i], slab_bytes);
    }
    if (stat) sc.add_to(stat);
    int32_t ea = ca, eb = cb, ta, tb;
    block_scan2(ea, eb, sh, &ta, &tb);
    ea -= ca;
    eb -= cb;
#pragma unroll
    for (int i = 0; i < SH_PER; ++i) {
        if (hj[i] < 0) continue;
        const int l = lj[i], m = cnt[hj[i]], c = chk[hj[i]], k = (m + tq - 1) / tq;
        lcnt[l] = m;
        loff[l] = ea;
        nch[l] = c;
        off[hj[i]] = ea;
        for (int t = 0; t < k * c; ++t)
            if (eb + t < item_cap) items[eb + t] = make_int2(l, ((t / c) << 8) | (t % c));
        ea += m;
        eb += k * c;
    }
    if (tid == 0) {
        if (tb > item_cap) atomicOr(err, ERR_PLAN);
        ctl->nitems = (int32_t)min((int64_t)tb, item_cap);
        ctl->nscan = ta;
        ctl->next_item = 0;
    }
    __syncthreads();
    // the pairs: their place in the list's group, their output runs
    int cv[SH_PER], mine = 0;
#pragma unroll
    for (int i = 0; i < SH_PER; ++i) {
        cv[i] = 0;
        if (lv[i] < 0) continue;
        qlist[off[sl[i]] + rk[i]] = ev[i];
        cv[i] = chk[sl[i]];
        mine += cv[i];
    }
    int32_t run = mine, dummy = 0, total, td;
    block_scan2(run, dummy, sh, &total, &td);
    if (tid == 0) s_base = atomicAdd(&ctl->nruns, total);
    __syncthreads();
    const int base = s_base;
    const bool fits = base >= 0 && (int64_t)base + total <= run_cap;
    if (!fits && tid == 0) atomicOr(err, ERR_PLAN);
    run += base - mine;
    const int start = run;
#pragma unroll
    for (int i = 0; i < SH_PER; ++i) {
        if (ev[i] < 0) continue;
        prun[ev[i]] = cv[i] > 0 && fits ? run : -1;
        if (ev[i] % P == p0) first[ev[i] / P] = run;
        run += cv[i];
    }
    __syncthreads();  // every query's first run is written
    int2 *qr = qrun + (p0 > 0 ? nq : 0);
    run = start;
#pragma unroll
    for (int i = 0; i < SH_PER; ++i) {
        if (ev[i] < 0) continue;
        run += cv[i];
        if (ev[i] % P == p1 - 1) {
            const int q = ev[i] / P;
            qr[q] = fits ? make_int2(first[q], run - first[q]) : make_int2(0, 0);
        }
    }
}

// ------------------------------------------------------- pair pruning
// Which of a query's farther lists (p >= 1) may hold a vector within the
// bound t its nearest list left.  Every member x of list l lies within R_l
// of the centroid, so ||q - x|| >= ||q - c_l|| - R_l (triangle inequality);
// when the scan's own distance of every x is then provably above t, the pair
// takes no part: none of its vectors could have been kept, so the results
// are the same.  Where cells overlap (a query's neighbours in one cluster)
// nothing is pruned and the kernel costs a read of each pair's centroid;
// between separate clusters it removes the pair's whole scan: the 63 farther
// lists of a Deep-like search (10,000 queries, 4,096 lists) took 2.4 of 5.4
// ms.  Lower bounds of the scan's distance D, rq = ||q - c_l||, rounded
// towards keeping the pair:
//   FP32: D >= (rq - R)^2 up to the direct form's rounding;
//   BF16: D >= (rq - R)^2 - 2 e ||q|| (||c|| + R), e the error of the BF16
//     products (first_stage_rel, doubled), and the norms' roundings;
//   FP8: D = rq^2 + rx^2 - 2 s q^.x^ with ||q^|| <= rq + eq and ||x^|| <= rx +
//     ex (E4M3 rounds to 2^-4 relative, 2^-10 of a code unit below the
//     smallest normal; saturation only shortens x^), least at rx = R.
// Sums of squares below FP32's range lose up to 2^-150 a term, 2e-43 in all (R
// grows and the bound sinks by what covers it), and one beyond the range says
// nothing of D: the pair stays.
// One warp takes PR consecutive pairs of one query (8, or 4 for d > 128),
// their centroid rows in flight together, and works out the bounds one pair
// per lane (every lane for every pair: 324 against 82 us for 630,000 pairs);
// a FP8 pair that stays gets its residual codes here.
__host__ __device__ constexpr int prune_per(int NV) { return NV == 1 ? 8 : 4; }
struct PruneArgs {
    const float *q;
    int64_t nq;
    int P, d, L;
    const int32_t *probes;
    bool dedupe;
    const float *cent, *cnrm_up, *lrad2, *thr, *inv_scale8, *qn;
    float e_bf16;
    float *pqn, *pqsc;
    unsigned char *qcast;
    int32_t *prank;
};

template <int DT, int NV>  // sivf_scan_dtype; float4 of a row per lane (d <= 128 NV)
__global__ __launch_bounds__(256) void k_pair_prune(PruneArgs a)
{
    pdl_begin();
    constexpr int PR_P = prune_per(NV);
    const int lane = threadIdx.x & 31, d = a.d, n4 = d >> 2;
    const int np = a.P - 1, ng = (np + PR_P - 1) / PR_P;
    const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (t >= a.nq * ng) return;  // whole warps
    const int64_t qi = t / ng;
    const int pb = 1 + (int)(t % ng) * PR_P;
    const float *qr = a.q + (size_t)qi * d;
    int lv[PR_P];
    float4 r[PR_P][NV];
#pragma unroll
    for (int k = 0; k < PR_P; ++k) {
        const int64_t e = qi * a.P + pb + k;
        lv[k] = pb + k < a.P ? a.probes[e] : -1;
        if (lv[k] >= a.L) lv[k] = -1;
    }
#pragma unroll
    for (int k = 0; k < PR_P; ++k)
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int j4 = lane + 32 * u;
            r[k][u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (lv[k] >= 0 && j4 < n4)
                r[k][u] = __ldg(reinterpret_cast<const float4 *>(a.cent + (size_t)lv[k] * d) + j4);
        }
    float ss[PR_P], mx[PR_P];
#pragma unroll
    for (int k = 0; k < PR_P; ++k) ss[k] = mx[k] = 0.f;
#pragma unroll
    for (int u = 0; u < NV; ++u) {
        const int j4 = lane + 32 * u;
        if (j4 >= n4) break;
        const float4 v = __ldg(reinterpret_cast<const float4 *>(qr) + j4);
#pragma unroll
        for (int k = 0; k < PR_P; ++k) {
            const float4 c = r[k][u];
            r[k][u] = make_float4(__fsub_rn(v.x, c.x), __fsub_rn(v.y, c.y), __fsub_rn(v.z, c.z),
                                  __fsub_rn(v.w, c.w));
            ss[k] = fmaf(r[k][u].x, r[k][u].x, ss[k]);
            ss[k] = fmaf(r[k][u].y, r[k][u].y, ss[k]);
            ss[k] = fmaf(r[k][u].z, r[k][u].z, ss[k]);
            ss[k] = fmaf(r[k][u].w, r[k][u].w, ss[k]);
            if (DT == SIVF_FP8E4M3)
                mx[k] = fmaxf(mx[k], fmaxf(fmaxf(fabsf(r[k][u].x), fabsf(r[k][u].y)),
                                           fmaxf(fabsf(r[k][u].z), fabsf(r[k][u].w))));
        }
    }
#pragma unroll
    for (int k = 0; k < PR_P; ++k) ss[k] = warp_sum(ss[k]);
    if (DT == SIVF_FP8E4M3)
#pragma unroll
        for (int k = 0; k < PR_P; ++k)
            for (int o = 16; o > 0; o >>= 1) mx[k] = fmaxf(mx[k], __shfl_xor_sync(0xffffffffu, mx[k], o));
    // lane k takes pair pb + k
    const int np_here = min(PR_P, a.P - pb);
    int l = -1;
    float s2 = 0.f, mxl = 0.f;
#pragma unroll
    for (int k = 0; k < PR_P; ++k)
        if (lane == k) {
            l = lv[k];
            s2 = ss[k];
            mxl = mx[k];
        }
    bool keep = lane < np_here && l >= 0;
    if (a.dedupe)
        for (int k = 0; k < np_here; ++k) {
            const int lk = __shfl_sync(0xffffffffu, l, k);
            bool dup = false;
            for (int f = lane; f < pb + k; f += 32) dup |= a.probes[qi * a.P + f] == lk;
            dup = __any_sync(0xffffffffu, dup);
            if (lane == k) keep &= !dup;
        }
    const float sc = mxl > 0.f ? 448.f / (2.f * mxl) : 1.f;
    if (keep) {
        const float u32 = 5.9604645e-08f;  // 2^-24
        const float up = 1.f + (2.f * d + 32.f) * u32, dn = 1.f - (2.f * d + 32.f) * u32;
        const float bound = __ldcg(a.thr + qi);
        const float R = __fadd_ru(__fsqrt_ru(__ldg(a.lrad2 + l)), 2e-21f);
        const float rlo = __fsqrt_rd(__fmul_rd(s2, dn)), rhi = __fsqrt_ru(__fmul_ru(s2, up));
        const float gap = __fsub_rd(rlo, R);
        float lo = -INFINITY;  // lower bound of the scan's distances
        if (gap > 0.f && rlo < INFINITY) {
            if (DT == SIVF_FP32) {
                lo = __fmul_rd(__fmul_rd(gap, gap), dn);
            } else if (DT == SIVF_BF16) {
                const float qn = __fsqrt_ru(__fmul_ru(__ldg(a.qn + qi), up));
                const float xn = __fadd_ru(__ldg(a.cnrm_up + l), R);
                const float n2 = __fadd_ru(__fmul_ru(qn, qn), __fmul_ru(xn, xn));
                const float err = __fadd_ru(__fmul_ru(__fmul_ru(a.e_bf16, qn), __fmul_ru(2.f, xn)),
                                            __fmul_ru(n2, (2.f * d + 64.f) * u32));
                lo = __fsub_rd(__fmul_rd(gap, gap), err);
            } else {
                const float sq = sqrtf((float)d) * 1.01f * 9.765625e-04f;  // 2^-10
                const float A = __fadd_ru(__fmul_ru(rhi, 1.0626f), __fdiv_ru(sq, sc));
                const float X = __fadd_ru(__fmul_ru(R, 1.0626f),
                                          __fdiv_ru(sq, __ldg(a.inv_scale8 + l)));
                // products' accumulation (4 d u) and the norms' roundings
                const float err = __fmul_ru(__fadd_ru(__fmul_ru(rhi, rhi), __fmul_ru(A, X)),
                                            (16.f * d + 64.f) * u32);
                lo = __fsub_rd(__fsub_rd(__fadd_rd(__fmul_rd(rlo, rlo), __fmul_rd(__fmul_rd(R, R), dn)),
                                         __fmul_ru(2.f, __fmul_ru(A, X))),
                               err);
            }
        }
        keep = !(__fsub_rd(lo, 1e-42f) > bound);
    }
    if (lane < np_here) {
        const int64_t e = qi * a.P + pb + lane;
        a.prank[e] = keep ? 0 : -1;
        if (DT == SIVF_FP8E4M3 && keep) {
            a.pqn[e] = s2;
            a.pqsc[e] = sc;
        }
    }
    const uint32_t stay = __ballot_sync(0xffffffffu, keep);
    if (DT == SIVF_FP8E4M3 && stay) {
#pragma unroll
        for (int k = 0; k < PR_P; ++k) {
            if (!((stay >> k) & 1u)) continue;  // warp-uniform
            const int64_t e = qi * a.P + pb + k;
            const float sk = __shfl_sync(0xffffffffu, sc, k);
#pragma unroll
            for (int u = 0; u < NV; ++u) {
                const int j4 = lane + 32 * u;
                if (j4 >= n4) break;
                const uint32_t lo8 = __nv_cvt_float2_to_fp8x2(
                    make_float2(__fmul_rn(r[k][u].x, sk), __fmul_rn(r[k][u].y, sk)), __NV_SATFINITE, __NV_E4M3);
                const uint32_t hi8 = __nv_cvt_float2_to_fp8x2(
                    make_float2(__fmul_rn(r[k][u].z, sk), __fmul_rn(r[k][u].w, sk)), __NV_SATFINITE, __NV_E4M3);
                reinterpret_cast<uint32_t *>(a.qcast + (size_t)e * d)[j4] = (lo8 & 0xffffu) | (hi8 << 16);
            }
        }
    }
}

void prune_pairs(sivf_index *ix, int dtype, const float *q, int64_t nq, int P,
                 const int32_t *probes, bool dedupe, const SearchScratch &s, cudaStream_t st)
{
    PruneArgs a;
    a.q = q;
    a.nq = nq;
    a.P = P;
    a.d = ix->d;
    a.L = ix->nlist;
    a.probes = probes;
    a.dedupe = dedupe;
    a.cent = ix->cent;
    a.cnrm_up = ix->cnrm_up;
    a.lrad2 = ix->lrad2;
    a.thr = s.thr;
    a.inv_scale8 = ix->inv_scale8;
    a.qn = s.qn;
    a.e_bf16 = (float)(2.0 * first_stage_rel(ix->d, 1) * (1.0 + 1e-6));
    a.pqn = s.pqn;
    a.pqsc = s.pqsc;
    a.qcast = s.qcast;
    a.prank = s.prank;
    const int NV = ix->d <= 128 ? 1 : 2, per = prune_per(NV);
    const int64_t warps = nq * ((P - 1 + per - 1) / per);
    const unsigned blocks = (unsigned)((warps * 32 + 255) / 256);
    const int tg = prof_begin(ix, PROF_GROUP, 1, st);
    auto go = [&](auto one, auto two) { launch_pdl(NV == 1 ? one : two, blocks, 256, 0, st, a); };
    if (dtype == SIVF_FP32) go(&k_pair_prune<SIVF_FP32, 1>, &k_pair_prune<SIVF_FP32, 2>);
    else if (dtype == SIVF_BF16) go(&k_pair_prune<SIVF_BF16, 1>, &k_pair_prune<SIVF_BF16, 2>);
    else go(&k_pair_prune<SIVF_FP8E4M3, 1>, &k_pair_prune<SIVF_FP8E4M3, 2>);
    prof_end(ix, tg, st);
}

// Phase 1's plan: a chunk of the nearest list leaves a bound only when it
// holds K vectors, so it gets twice that many slots
SearchPlan bound_plan(const sivf_index *ix, SearchPlan pl)
{
    pl.slabs_per_chunk = std::max(pl.slabs_per_chunk, (2 * pl.K + ix->C - 1) / ix->C);
    return pl;
}

// A launch of the nearest lists alone pays where the others have work to
// save: its four extra launches cost about 12 us, a scan of 2,048 pairs more
// than that; a handful of pairs is scanned at once
bool fp32_two_phase(int64_t nq, int P) { return P > 1 && nq * P >= 2048; }

// One thread per query, whole warps together: each pair goes to its list's
// group (qlist), and the query's pairs of this phase reserve consecutive
// output runs (one per slab chunk of the pair's list; one atomic per warp).
__global__ void k_srch_scatter_t(const int32_t *__restrict__ probes, int64_t nq, int P, int p0,
                                 int p1, const int32_t *__restrict__ prank,
                                 const int32_t *__restrict__ loff, const int32_t *__restrict__ nch,
                                 int32_t *__restrict__ qlist, int32_t *__restrict__ prun,
                                 int2 *__restrict__ qrun, Ctl *ctl, int64_t run_cap,
                                 uint32_t *err)
{
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); q0 < nq;
         q0 += stride) {
        const int64_t q = q0 + lane;
        int cnt = 0;
        if (q < nq)
            for (int p = p0; p < p1; ++p) {
                const int64_t e = q * P + p;
                const int r = prank[e];
                int c = 0;
                if (r >= 0) {
                    const int l = probes[e];
                    qlist[loff[l] + r] = (int32_t)e;
                    c = nch[l];
                }
                prun[e] = c;
                cnt += c;
            }
        int incl = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        int base = 0;
        if (lane == 31) base = atomicAdd(&ctl->nruns, incl);
        base = __shfl_sync(0xffffffffu, base, 31) + incl - cnt;
        if (q < nq) {
            const bool fits = base >= 0 && (int64_t)base + cnt <= run_cap;
            if (!fits) atomicOr(err, ERR_PLAN);
            int run = base;
            for (int p = p0; p < p1; ++p) {
                const int64_t e = q * P + p;
                const int c = prun[e];
                prun[e] = (c > 0 && fits) ? run : -1;
                run += c;
            }
            qrun[(p0 > 0 ? nq : 0) + q] = fits ? make_int2(base, cnt) : make_int2(0, 0);
        }
    }
}

// The same with one warp per query, SC_Q queries per block, for phases of
// many probes: the warp's lanes take the probes p0 + lane + 32 j, runs are
// assigned in probe order (one atomic per block).
// prun = the pair's first run (-1: not scanned); qrun[phase][q] = (first
// run, runs) of the query.  A reservation past run_cap (the plan's bound
// makes this impossible) sets ERR_PLAN and leaves the query's runs out.
constexpr int SC_Q = 8;
__global__ __launch_bounds__(SC_Q * 32) void k_srch_scatter(
    const int32_t *__restrict__ probes, int64_t nq, int P, int p0, int p1,
    const int32_t *__restrict__ prank, const int32_t *__restrict__ loff,
    const int32_t *__restrict__ nch, int32_t *__restrict__ qlist, int32_t *__restrict__ prun,
    int2 *__restrict__ qrun, Ctl *ctl, int64_t run_cap, uint32_t *err)
{
    pdl_begin();
    __shared__ int s_cnt[SC_Q];
    __shared__ int s_base;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int64_t qb = (int64_t)blockIdx.x * SC_Q; qb < nq; qb += (int64_t)gridDim.x * SC_Q) {
        const int64_t q = qb + w;
        int cnt = 0;
        if (q < nq)
            for (int p = p0 + lane; p < p1; p += 32) {
                const int64_t e = q * P + p;
                const int r = prank[e];
                int c = 0;
                if (r >= 0) {
                    const int l = probes[e];
                    qlist[loff[l] + r] = (int32_t)e;
                    c = nch[l];
                }
                prun[e] = c;
                cnt += c;
            }
        for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        if (lane == 0) s_cnt[w] = cnt;
        __syncthreads();
        if (threadIdx.x == 0) {
            int tot = 0;
            for (int k = 0; k < SC_Q; ++k) tot += s_cnt[k];
            s_base = atomicAdd(&ctl->nruns, tot);
        }
        __syncthreads();
        int base = s_base;
        for (int k = 0; k < w; ++k) base += s_cnt[k];
        if (q < nq) {
            const bool fits = base >= 0 && (int64_t)base + cnt <= run_cap;
            if (!fits && lane == 0) atomicOr(err, ERR_PLAN);
            int run = base;
            for (int pb = p0; pb < p1; pb += 32) {  // warp-uniform
                const int p = pb + lane;
                const int64_t e = q * P + p;
                const int c = p < p1 ? prun[e] : 0;  // this lane's own count from above
                int incl = c;
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += v;
                }
                if (p < p1) prun[e] = (c > 0 && fits) ? run + incl - c : -1;
                run += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) qrun[(p0 > 0 ? nq : 0) + q] = fits ? make_int2(base, cnt) : make_int2(0, 0);
        }
        __syncthreads();  // s_cnt and s_base are reused by the next queries
    }
}

// ------------------------------------------------------------ the scan
constexpr int SCAN_NT = 256;
constexpr int NST = 2;  // slab stages in flight

struct ScanArgs {
    const float *q;
    int64_t nq;
    int P, K, M;
    int nbs;              // slabs of a block (scan_block)
    const int32_t *qlist, *loff, *lcnt, *nch;
    const int32_t *prun;  // first output run of each pair
    const int2 *items;
    float *part_d;
    int64_t *part_i;
    float *thr;          // [nq] shared upper bound of each query's k-th distance
    // index
    const float *x32;
    const int64_t *ids;
    const uint32_t *bits;
    const SlabMeta *meta;
    const int32_t *nslabs, *dir;
    int64_t n_slabs, dir_cap;
    int L, d;
    Ctl *ctl;
    uint32_t *err;
};

__host__ __device__ constexpr int scan_next_pow2(int v)
{
    int p = 1;
    while (p < v) p <<= 1;
    return p;
}

// Entries per row of the best-K + candidate buffer: the best K, then room
// for 64 candidates (merged by rank, at most 256 entries); for larger K a
// power of two that the bitonic fallback can sort.
__host__ __device__ constexpr int scan_buf_len(int K, int C)
{
    return K + 64 <= 256 ? ((K + 64 + 15) & ~15) : scan_next_pow2(K + C);
}

// shared memory of one CTA: at most this, and half of the SM where a block
// of at least SCAN_BMIN rows' distances leaves room for two CTAs
constexpr size_t SCAN_SMEM = 222 * 1024;
constexpr size_t SCAN_HALF = 110 * 1024;
constexpr int SCAN_BMIN = 256;
// rows of a block at most: the few warps with a row of an 8-query tile keep 512
// distances in registers for the selection, more they read again and again
__host__ __device__ constexpr int scan_bmax(int TQ) { return TQ <= 8 ? 512 : 1024; }

// shared memory carve-up, identical on host and device; nbs: slabs of a
// block, whose distances the rows keep until they are selected from
struct ScanSmem {
    size_t xs, qs, bd, bi, dm, misc, total;
};
__host__ __device__ inline ScanSmem scan_smem_at(int TQ, int C, int d, int M, int nbs)
{
    ScanSmem s;
    const size_t DP = d + 4;
    s.xs = 0;  // swizzled slabs: 1024-byte aligned (C d 4 is a multiple then)
    s.qs = s.xs + (size_t)NST * C * d * 4;
    s.bd = s.qs + (size_t)TQ * DP * 4;
    s.bi = s.bd + (size_t)TQ * M * 4;
    s.bi = (s.bi + 15) & ~(size_t)15;
    s.dm = s.bi + (size_t)TQ * M * 8;
    s.misc = s.dm + (size_t)TQ * (nbs * C + 4) * 4;
    s.misc = (s.misc + 15) & ~(size_t)15;
    s.total = s.misc + 64 + (size_t)nbs * 4;
    return s;
}
// slabs of a block: the most rows up to scan_bmax, two CTAs per SM for the
// tiles of at most 16 queries where SCAN_BMIN rows fit then
__host__ __device__ inline int scan_block(int TQ, int C, int d, int M)
{
    const int most = scan_bmax(TQ) / C;
    if (TQ <= 16)
        for (int n = most; n * C >= SCAN_BMIN; --n)
            if (scan_smem_at(TQ, C, d, M, n).total <= SCAN_HALF) return n;
    int n = most;
    while (n > 1 && scan_smem_at(TQ, C, d, M, n).total > SCAN_SMEM) --n;
    return n;
}
__host__ __device__ inline ScanSmem scan_smem(int TQ, int C, int d, int M)
{
    return scan_smem_at(TQ, C, d, M, scan_block(TQ, C, d, M));
}

// Merge one query's candidates into its best list (one warp).  Every
// element of the union finds its rank by counting the elements that precede
// it in (distance, id) order -- candidates by a broadcast scan, best entries
// by binary search -- and then all elements land at once.  best[0, nb) is
// sorted, cand[K, K + nc) is not; ids are distinct, so ranks are too.
template <int EPL>
__device__ __forceinline__ void warp_rank_merge(float *bd, int64_t *bi, int K, int nb, int nc,
                                                int lane)
{
    const int n = nb + nc;
    float vd[EPL];
    int64_t vi[EPL];
    int pos[EPL];
#pragma unroll
    for (int t = 0; t < EPL; ++t) {
        const int e = lane + 32 * t;
        pos[t] = K;
        if (e >= n) continue;
        const int src = e < nb ? e : K + (e - nb);
        const float dv = bd[src];
        const int64_t iv = bi[src];
        vd[t] = dv;
        vi[t] = iv;
        int r = 0;
        for (int j = 0; j < nc; ++j) r += dk_less(bd[K + j], bi[K + j], dv, iv);
        if (e < nb) {
            r += e;
        } else {
            int lo = 0, hi = nb;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (dk_less(bd[mid], bi[mid], dv, iv)) lo = mid + 1;
                else hi = mid;
            }
            r += lo;
        }
        pos[t] = r;
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < EPL; ++t)
        if (pos[t] < K) {
            bd[pos[t]] = vd[t];
            bi[pos[t]] = vi[t];
        }
    __syncwarp();
}

// Fallback for large buffers: bitonic sort of all M entries (pads first).
__device__ void warp_bitonic_merge(float *bd, int64_t *bi, int K, int nb, int nc, int M,
                                   int lane)
{
    for (int e = nb + lane; e < K; e += 32) {
        bd[e] = INFINITY;
        bi[e] = -1;
    }
    for (int e = K + nc + lane; e < M; e += 32) {
        bd[e] = INFINITY;
        bi[e] = -1;
    }
    __syncwarp();
    for (int size = 2; size <= M; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = lane; t < M / 2; t += 32) {
                const int pos = 2 * t - (t & (stride - 1));
                const int par = pos + stride;
                const bool up = (pos & size) == 0;
                const float d0 = bd[pos], d1 = bd[par];
                const int64_t i0 = bi[pos], i1 = bi[par];
                // pads (id -1) sort after every real entry
                const bool lt = (i1 >= 0 && i0 < 0) ||
                                (i1 >= 0 && i0 >= 0 && dk_less(d1, i1, d0, i0));
                if (lt == up) {
                    bd[pos] = d1;
                    bd[par] = d0;
                    bi[pos] = i1;
                    bi[par] = i0;
                }
            }
            __syncwarp();
        }
}

// Direct-form distances of the first RQA row groups of a thread's tile:
// acc[i][r] = sum_j (q_{i}[j] - x_{r}[j])^2, FP32, j in steps of 4.
// SW: the slab lies in segments of 32 floats per row with the 128-byte
// swizzle (16-byte chunk c of row r at c ^ (r & 7)).  A warp reads four rows
// at a time; rows of d % 32 == 0 floats side by side start on the same bank,
// and the unswizzled reads took four passes each, more than the arithmetic.
template <int RQA, bool SW, int C, int RQ, int RX>
__device__ __forceinline__ void dist_tile(float (&acc)[RQ][RX], const float *__restrict__ qrow,
                                          const float *__restrict__ xs, int row0, int d, int DP)
{
#pragma unroll
    for (int i = 0; i < RQA; ++i)
#pragma unroll
        for (int r = 0; r < RX; ++r) acc[i][r] = 0.f;
    auto step = [&](const float4 (&qv)[RQA], const float4 (&xv)[RX]) {
#pragma unroll
        for (int i = 0; i < RQA; ++i)
#pragma unroll
            for (int r = 0; r < RX; ++r) {
                const float t0 = qv[i].x - xv[r].x, t1 = qv[i].y - xv[r].y;
                const float t2 = qv[i].z - xv[r].z, t3 = qv[i].w - xv[r].w;
                float v = acc[i][r];
                v = fmaf(t0, t0, v);
                v = fmaf(t1, t1, v);
                v = fmaf(t2, t2, v);
                v = fmaf(t3, t3, v);
                acc[i][r] = v;
            }
    };
    if (SW) {
        for (int g = 0; g < d; g += 32) {
            const float *xg = xs + (size_t)g * C + row0 * 32;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                float4 qv[RQA], xv[RX];
#pragma unroll
                for (int i = 0; i < RQA; ++i)
                    qv[i] = *reinterpret_cast<const float4 *>(qrow + (size_t)i * 8 * DP + g + 4 * c);
#pragma unroll
                for (int r = 0; r < RX; ++r)
                    xv[r] = *reinterpret_cast<const float4 *>(xg + r * 128 +
                                                              ((c ^ ((row0 + 4 * r) & 7)) << 2));
                step(qv, xv);
            }
        }
        return;
    }
#pragma unroll 4
    for (int j = 0; j < d; j += 4) {
        float4 qv[RQA], xv[RX];
#pragma unroll
        for (int i = 0; i < RQA; ++i)
            qv[i] = *reinterpret_cast<const float4 *>(qrow + (size_t)i * 8 * DP + j);
#pragma unroll
        for (int r = 0; r < RX; ++r)
            xv[r] = *reinterpret_cast<const float4 *>(xs + (size_t)(row0 + 4 * r) * d + j);
        step(qv, xv);
    }
}

// ONE: shared memory leaves room for one CTA per SM, so that a thread may have
// all the registers (at the 128 of two CTAs the small tiles spill: 12 queries of
// 25 lists of 13,400 vectors, d = 192, 1,119 us, 785 so)
template <int TQ, int C, bool XS, bool ONE>
__global__ __launch_bounds__(SCAN_NT, ONE ? 1 : 2) void k_scan(
    const __grid_constant__ CUtensorMap tmap, ScanArgs a)
{
    pdl_begin();
    constexpr int QW = TQ >= 32 ? TQ / 32 : 1;
    constexpr int SW = 8 / QW;
    constexpr int RQ = TQ / (8 * QW);
    constexpr int RX = C / (4 * SW);
    constexpr int W = C / 32;
    static_assert(RQ >= 1 && RX >= 1, "tile shape");

    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *smem = XS ? smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023) : smem_raw;
    const int d = a.d, DP = d + 4, M = a.M, K = a.K;
    const int CB = M - K;  // candidate buffer capacity (>= 32)
    const int NBS = a.nbs, DS = NBS * C + 4;  // slabs of a block, row stride of its distances
    const ScanSmem L = scan_smem_at(TQ, C, d, M, NBS);
    float *Qs = reinterpret_cast<float *>(smem + L.qs);
    float *Xs = reinterpret_cast<float *>(smem + L.xs);
    float *BD = reinterpret_cast<float *>(smem + L.bd);
    int64_t *BI = reinterpret_cast<int64_t *>(smem + L.bi);
    float *DM = reinterpret_cast<float *>(smem + L.dm);
    unsigned char *misc = smem + L.misc;
    uint64_t *mbar = reinterpret_cast<uint64_t *>(misc);  // [NST]
    int *s_item = reinterpret_cast<int *>(misc + 8 * NST);
    int *s_abort = s_item + 1;
    int *stage_slab = s_item + 2;                         // [NST]
    int *block_slab = stage_slab + NST;                   // [NBS] slabs of the block
    __shared__ int32_t s_qpair[TQ];   // (query, probe) pair of each row
    __shared__ int s_cc[TQ];          // candidates waiting per row
    __shared__ int s_nb[TQ];          // valid best entries per row
    __shared__ float s_kd[TQ];        // admission threshold per row
    __shared__ int64_t s_ki[TQ];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wq = warp % QW, ws = warp / QW;
    const int qy = lane & 7, sx = lane >> 3;
    const int64_t NOID = 0x7fffffffffffffffLL;

    if (tid == 0) {
        for (int s = 0; s < NST; ++s) mbar_init(&mbar[s], 1);
        fence_mbar_init();
        *s_abort = 0;
    }
    __syncthreads();

    const uint32_t slab_bytes = (uint32_t)(C * d * 4);
    uint32_t g_cons = 0, g_issue = 0;  // slabs consumed / issued by this CTA

    auto issue = [&](int stage, int s) {
        // called by thread 0 only
        bool ok = s >= 0 && s < a.n_slabs;
        if (!ok) atomicOr(a.err, ERR_BAD_SLAB);
        stage_slab[stage] = ok ? s : -1;
        if (ok) {
            mbar_arrive_expect_tx(&mbar[stage], slab_bytes);
            if (XS) {
                for (int g = 0; g < d; g += 32)
                    tma_load_2d(Xs + (size_t)stage * C * d + (size_t)g * C, &tmap, g, s * C,
                                &mbar[stage]);
            } else {
                bulk_g2s(Xs + (size_t)stage * C * d, a.x32 + (size_t)s * C * d, slab_bytes,
                         &mbar[stage]);
            }
        } else {
            mbar_arrive(&mbar[stage]);
        }
    };

    // merge the waiting candidates of row qr (one warp), then refresh the
    // row's threshold from its own K-th entry and the query's shared bound
    auto merge_row = [&](int qr) {
        float *bd = BD + (size_t)qr * M;
        int64_t *bi = BI + (size_t)qr * M;
        const int nb = s_nb[qr], nc = s_cc[qr];
        if (nc > 0) {
            if (nb + nc <= 32) warp_rank_merge<1>(bd, bi, K, nb, nc, lane);
            else if (nb + nc <= 64) warp_rank_merge<2>(bd, bi, K, nb, nc, lane);
            else if (nb + nc <= 128) warp_rank_merge<4>(bd, bi, K, nb, nc, lane);
            else if (nb + nc <= 256) warp_rank_merge<8>(bd, bi, K, nb, nc, lane);
            else warp_bitonic_merge(bd, bi, K, nb, nc, M, lane);
        }
        const int nb2 = min(K, nb + nc);
        if (lane == 0) {
            s_nb[qr] = nb2;
            s_cc[qr] = 0;
            float kd = s_kd[qr];
            int64_t ki = s_ki[qr];
            const int q = s_qpair[qr] / a.P;
            if (nb2 == K && dk_less(bd[K - 1], bi[K - 1], kd, ki)) {
                kd = bd[K - 1];
                ki = bi[K - 1];
                atomicMin(reinterpret_cast<int *>(a.thr) + q, __float_as_int(kd));
            }
            const float g = __ldcg(a.thr + q);
            if (g < kd) {
                kd = g;
                ki = NOID;
            }
            s_kd[qr] = kd;
            s_ki[qr] = ki;
        }
        __syncwarp();
    };

    // Select from the n distances of the block for row qr (one warp): the row's
    // K-th or the query's bound is the bar; while the row holds fewer than K and
    // many lie within that, a value K of them lie at or below (kth_bound; always
    // sought, it cost 780 queries of 11 lists among overlapping cells a quarter of
    // their time: 1,354 us, 1,055 so); what is within it (ties included) goes to the
    // candidates, slots first, and is merged with its ids
    auto select_row = [&](int qr, int n, bool last) {
        const float *dr = DM + (size_t)qr * DS;
        float *bd = BD + (size_t)qr * M + K;
        int64_t *bi = BI + (size_t)qr * M + K;
        float bar = s_kd[qr];
        bool many = s_nb[qr] < K;  // more within the bar than a merge takes cheaply
        if (many && bar < 1e38f) {
            int c = 0;
#pragma unroll 8
            for (int i = lane; i < n; i += 32) c += dr[i] <= bar;
            many = __reduce_add_sync(0xffffffffu, c) > K + 16;
        }
        if (many)
            bar = fminf(bar, kth_bound<16>([&](int i) { return i < n ? dr[i] : INFINITY; },
                                           (n + 31) & ~31, K, lane));
        int cc = M > 256 ? s_cc[qr] : 0;  // those of earlier blocks have their ids
        auto merge = [&](bool now) {
            __syncwarp();
            for (int e = lane; e < cc; e += 32) {
                const int i = ~(int)bi[e];
                if (i >= 0) bi[e] = __ldg(a.ids + (size_t)block_slab[i / C] * C + i % C);
            }
            if (lane == 0) s_cc[qr] = cc;
            __syncwarp();
            if (now) merge_row(qr);
        };
        for (int i0 = 0; i0 < n; i0 += 32) {
            const float v = dr[i0 + lane];  // n is a multiple of 32
            const bool in = v <= bar && v < INFINITY;
            const uint32_t mk = __ballot_sync(0xffffffffu, in);
            if (mk == 0u) continue;
            if (cc + __popc(mk) > CB) {
                merge(true);
                bar = fminf(bar, s_kd[qr]);
                cc = 0;
            }
            if (in) {
                const int p = cc + __popc(mk & lanemask_lt());
                bd[p] = v;
                bi[p] = ~(int64_t)(i0 + lane);  // its place in the block, negative
            }
            cc += __popc(mk);
        }
        // more than 256 entries are sorted as a whole, whatever is new among them:
        // they wait for a full buffer or the item's end (large K leaves room for
        // blocks of one slab: K = 500, 1,000 queries of 16 of 90 skewed lists of a
        // million vectors, 37.9 ms with a sort per block, 7.6 so)
        merge(M <= 256 || last || s_nb[qr] + cc <= 256);
    };

    for (;;) {
        if (tid == 0) *s_item = atomicAdd(&a.ctl->next_item, 1);
        __syncthreads();
        const int item = *s_item;
        if (item >= a.ctl->nitems || *s_abort) break;

        // item -> list, query tile, slab chunk
        const int2 it = a.items[item];
        const int l = it.x;
        const int nc_l = a.nch[l];
        const int tile = it.y >> 8, chunk = it.y & 255;
        const int mcount = a.lcnt[l];
        const int r0 = tile * TQ;                     // tiles filled from the front;
        const int m = min(TQ, mcount - r0);           // the last one skips empty groups
        int ns_total = a.nslabs[l];
        if (ns_total > a.dir_cap) {
            if (tid == 0) atomicOr(a.err, ERR_DIR_BOUND);
            ns_total = (int)a.dir_cap;
        }
        const int s0 = (int)((int64_t)ns_total * chunk / nc_l);
        const int s1 = (int)((int64_t)ns_total * (chunk + 1) / nc_l);
        const int ns = s1 - s0;
        const int32_t *dirl = a.dir + (size_t)l * a.dir_cap;

        // stage the first slabs while the query tile is gathered
        if (tid == 0) {
            for (int t = 0; t < NST && t < ns; ++t) {
                issue((g_issue % NST), dirl[s0 + t]);
                ++g_issue;
            }
        }
        const int qb = a.loff[l] + r0;
        for (int r = tid; r < TQ; r += SCAN_NT) {
            const int pr = r < m ? a.qlist[qb + r] : -1;
            s_qpair[r] = pr;
            s_cc[r] = 0;
            s_nb[r] = 0;
            s_kd[r] = pr >= 0 ? __ldcg(a.thr + pr / a.P) : INFINITY;
            s_ki[r] = NOID;
        }
        __syncthreads();
        for (int e = tid; e < TQ * (d / 4); e += SCAN_NT) {
            const int r = e / (d / 4), j4 = e % (d / 4);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            const int pr = s_qpair[r];
            if (pr >= 0)
                v = *reinterpret_cast<const float4 *>(a.q + (size_t)(pr / a.P) * d + 4 * j4);
            *reinterpret_cast<float4 *>(Qs + (size_t)r * DP + 4 * j4) = v;
        }
        __syncthreads();

        const bool warp_active = wq * 8 * RQ < m;  // some row of this warp is real
        for (int idx = 0; idx < ns; ++idx) {
            const int stage = g_cons % NST;
            const uint32_t parity = (g_cons / NST) & 1u;
            if (!mbar_wait_bounded(&mbar[stage], parity, a.err)) *s_abort = 1;
            ++g_cons;
            const int s = stage_slab[stage];
            if (s >= 0 && warp_active && !*s_abort) {
                const float *xs = Xs + (size_t)stage * C * d;
                float acc[RQ][RX];
                const float *qrow = Qs + (size_t)(wq * 8 * RQ + qy) * DP;
                const int row0 = ws * 4 * RX + sx;
                // only the row groups that hold queries are computed
                const int nact = min(RQ, (m - wq * 8 * RQ + 7) / 8);
                if (nact >= RQ) dist_tile<RQ, XS, C>(acc, qrow, xs, row0, d, DP);
                else if (nact == 1) dist_tile<1, XS, C>(acc, qrow, xs, row0, d, DP);
                else if (nact == 2) dist_tile<(RQ >= 2 ? 2 : 1), XS, C>(acc, qrow, xs, row0, d, DP);
                else dist_tile<(RQ >= 3 ? 3 : 1), XS, C>(acc, qrow, xs, row0, d, DP);
                uint32_t bw[W];
#pragma unroll
                for (int w = 0; w < W; ++w) bw[w] = __ldg(a.bits + (size_t)s * W + w);
                float *dm = DM + (idx % NBS) * C;
#pragma unroll
                for (int i = 0; i < RQ; ++i) {
                    const int qr = wq * 8 * RQ + qy + 8 * i;
                    if (i >= nact) continue;
#pragma unroll
                    for (int r = 0; r < RX; ++r) {
                        const int slot = ws * 4 * RX + sx + 4 * r;
                        const bool live = (bw[slot >> 5] >> (slot & 31)) & 1u;
                        dm[(size_t)qr * DS + slot] = live ? acc[i][r] : INFINITY;
                    }
                }
            } else if (warp_active) {  // a skipped slab has no distances
#pragma unroll
                for (int i = 0; i < RQ; ++i)
#pragma unroll
                    for (int r = 0; r < RX; ++r)
                        DM[(size_t)(wq * 8 * RQ + qy + 8 * i) * DS + (idx % NBS) * C + ws * 4 * RX + sx +
                           4 * r] = INFINITY;
            }
            if (tid == 0) block_slab[idx % NBS] = max(s, 0);
            __syncthreads();
            // the stage is free: fetch the slab NST ahead into it
            if (tid == 0 && idx + NST < ns && !*s_abort) {
                fence_proxy_async_smem();
                issue(g_issue % NST, dirl[s0 + idx + NST]);
                ++g_issue;
            }
            if (idx % NBS == NBS - 1 || idx + 1 == ns) {
                for (int qr = warp; qr < m; qr += SCAN_NT / 32)
                    select_row(qr, (idx % NBS + 1) * C, idx + 1 == ns);
                __syncthreads();
            }
        }

        // the best K of each row of the tile (padded with (+inf, -1))
        for (int e = tid; e < m * K; e += SCAN_NT) {
            const int r = e / K, j = e % K;
            const int run = a.prun[s_qpair[r]];
            if (run < 0) continue;
            const int64_t base = ((int64_t)run + chunk) * K;
            const bool ok = j < s_nb[r];
            a.part_d[base + j] = ok ? BD[(size_t)r * M + j] : INFINITY;
            a.part_i[base + j] = ok ? BI[(size_t)r * M + j] : -1;
        }
        __syncthreads();
    }
    // after an abort, give copies still in flight a bounded chance to land
    // before the CTA (and its shared memory) goes away
    if (tid == 0)
        while (g_cons < g_issue) {
            mbar_wait_bounded(&mbar[g_cons % NST], (g_cons / NST) & 1u, a.err, 100000u);
            ++g_cons;
        }
}

// ------------------------------------------------------- per-query merge
// threads of a block: two warps' tables of 1,024 entries take 40 KB
__host__ __device__ constexpr int merge_nt(int E) { return E <= 16 ? 128 : 64; }
constexpr int MERGE_RUNS_PER_LANE = 64;  // both phases' runs: at most 2,048 per query
constexpr int MERGE_LONG = 32;           // entries of a run that a lane takes alone

// One warp per query.  A query's runs of one scan phase (K entries each,
// sorted, padded with (+inf, -1)) are contiguous, and at least k entries lie
// at or below its shared bound after the scan: the warp gathers those (usually
// little more than k) and sorts them in registers.  The bound is loose where
// long lists were scanned in many chunks at once (few queries): a full table is
// cut down to a value k of its entries lie at or below (kth_bound), which is the
// bound from then on.  Short runs are streamed; of long ones a lane takes each
// and leaves it at its first entry past the bound (14 queries, k = 100, 90
// skewed lists: 137 us by streaming and then a cursor per run, 77 by cursors
// alone).  Only where cutting leaves no room (ties, or k > 960) does it walk
// all runs, a cursor per run, one result after the other.
template <int E>
__global__ __launch_bounds__(merge_nt(E)) void k_merge(const int2 *__restrict__ qrun, int64_t nq,
                                                    int nphase, int K, int k,
                                                    const float *__restrict__ thr,
                                                    const float *__restrict__ part_d,
                                                    const int64_t *__restrict__ part_i,
                                                    float *__restrict__ dist,
                                                    int64_t *__restrict__ labels)
{
    pdl_begin();
    constexpr int MU = 8;  // loads in flight per lane
    constexpr int NT = merge_nt(E);
    __shared__ float sd[NT / 32][32 * E];
    __shared__ int64_t si[NT / 32][32 * E];
    __shared__ uint64_t sk[NT / 32][32 * E];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t q = (blockIdx.x * (int64_t)NT + threadIdx.x) >> 5;
    if (q >= nq) return;  // whole warps
    const int2 r0 = qrun[q];
    const int2 r1 = nphase > 1 ? qrun[nq + q] : make_int2(0, 0);
    float bound = thr[q];
    int have = 0;
    bool room = k + k / 32 + 33 <= 32 * E;  // an append fits after a cut (kth_bound)
    // the warp's entries v within the bound, at `e` of the runs
    auto gather = [&](float v, int64_t e) {
        uint32_t mk = __ballot_sync(0xffffffffu, v <= bound);  // pads are +inf
        if (have + __popc(mk) > 32 * E) {
            room = have >= k;
            if (!room) return;
            __syncwarp();
            bound = fminf(bound, kth_bound<E>([&](int i) { return i < have ? sd[w][i] : INFINITY; },
                                              32 * E, k, lane));
            int n2 = 0;
            for (int i0 = 0; i0 < have; i0 += 32) {
                const int i = i0 + lane;
                const float u = i < have ? sd[w][i] : INFINITY;
                const int64_t id = i < have ? si[w][i] : -1;
                const uint32_t keep = __ballot_sync(0xffffffffu, u <= bound);
                if (u <= bound) {  // at or before i
                    const int p = n2 + __popc(keep & lanemask_lt());
                    sd[w][p] = u;
                    si[w][p] = id;
                }
                n2 += __popc(keep);
                __syncwarp();
            }
            have = n2;
            mk = __ballot_sync(0xffffffffu, v <= bound);
            room = have + __popc(mk) <= 32 * E;
            if (!room) return;
        }
        if (v <= bound) {
            const int p = have + __popc(mk & lanemask_lt());
            sd[w][p] = v;
            si[w][p] = part_i[e];
        }
        have += __popc(mk);
    };
    for (int ph = 0; ph < 2 && room; ++ph) {
        const int64_t b = (int64_t)(ph ? r1.x : r0.x) * K;
        const int64_t n = (int64_t)(ph ? r1.y : r0.y) * K;
        if (K >= MERGE_LONG) {
            for (int64_t g = 0; g < n && room; g += 32 * (int64_t)K) {
                const int64_t e0 = g + (int64_t)lane * K;
                bool on = e0 < n;
                for (int j0 = 0; j0 < K && room && __any_sync(0xffffffffu, on); j0 += MU) {
                    float v[MU];
#pragma unroll
                    for (int u = 0; u < MU; ++u)
                        v[u] = on && j0 + u < K ? part_d[b + e0 + j0 + u] : INFINITY;
#pragma unroll
                    for (int u = 0; u < MU; ++u)
                        if (room) gather(v[u], b + e0 + j0 + u);
                    on &= v[MU - 1] <= bound;  // +inf past the run's end
                }
            }
            continue;
        }
        for (int64_t i0 = lane; i0 - lane < n && room; i0 += 32 * MU) {
            float v[MU];
#pragma unroll
            for (int u = 0; u < MU; ++u)
                v[u] = i0 + 32 * u < n ? part_d[b + i0 + 32 * u] : INFINITY;
#pragma unroll
            for (int u = 0; u < MU; ++u)
                if (room) gather(v[u], b + i0 + 32 * u);
        }
    }
    __syncwarp();
    if (room) {
        warp_order<E>(
            have, [&](int i) { return sd[w][i]; }, [&](int i) { return si[w][i]; },
            [&](int i, float v, int64_t id) {
                if (i >= k) return;
                dist[q * k + i] = v;
                labels[q * k + i] = id;
            },
            sk[w], lane);
        for (int i = have + lane; i < k; i += 32) {
            dist[q * k + i] = INFINITY;
            labels[q * k + i] = -1;
        }
        return;
    }
    // cursors: run r = lane + 32 j of both phases' runs
    const int NR = r0.y + r1.y;
    int cur[MERGE_RUNS_PER_LANE];
    int nrun = 0;
    for (int r = lane; r < NR && nrun < MERGE_RUNS_PER_LANE; r += 32) cur[nrun++] = 0;
    auto head = [&](int j, float &hd, int64_t &hi) {
        int r = lane + 32 * j;
        if (cur[j] >= K) {
            hd = INFINITY;
            hi = -1;
            return;
        }
        const int64_t e = (int64_t)(r < r0.y ? r0.x + r : r1.x + (r - r0.y)) * K + cur[j];
        hd = part_d[e];
        hi = part_i[e];
        if (hi < 0) hd = INFINITY;
    };
    float bd = INFINITY;
    int64_t bi = -1;
    int bj = -1;
    auto rescan = [&]() {
        bd = INFINITY;
        bi = -1;
        bj = -1;
        for (int j = 0; j < nrun; ++j) {
            float hd;
            int64_t hi;
            head(j, hd, hi);
            if (hi >= 0 && (bj < 0 || dk_less(hd, hi, bd, bi))) {
                bd = hd;
                bi = hi;
                bj = j;
            }
        }
    };
    rescan();
    for (int o = 0; o < k; ++o) {
        float wd = bd;
        int64_t wi = bi;
        int wl = bj >= 0 ? lane : 32;
        for (int s = 16; s > 0; s >>= 1) {
            float od = __shfl_xor_sync(0xffffffffu, wd, s);
            int64_t oi = __shfl_xor_sync(0xffffffffu, wi, s);
            int ol = __shfl_xor_sync(0xffffffffu, wl, s);
            bool take = ol < 32 && (wl >= 32 || dk_less(od, oi, wd, wi));
            if (take) {
                wd = od;
                wi = oi;
                wl = ol;
            }
        }
        if (lane == 0) {
            dist[q * k + o] = wl < 32 ? wd : INFINITY;
            labels[q * k + o] = wl < 32 ? wi : -1;
        }
        if (wl == lane) {
            ++cur[bj];
            rescan();
        }
    }
}

// --------------------------------------------------------------- drivers
template <int TQ, int C, bool SW, bool ONE>
static void launch_scan(sivf_index *ix, const ScanArgs &a, size_t smem, int grid,
                        cudaStream_t st)
{
    if (SW) smem += 1024;  // base alignment slack
    static KernelSetup su;
    opt_in_smem(su, k_scan<TQ, C, SW, ONE>, smem);
    // as many CTAs per SM as fit: the small tiles' shared memory leaves room
    // for two or more, which hide each other's barriers and load latency
    int dev = 0;
    cudaGetDevice(&dev);
    const int occ = su.resident(dev, smem, [&] {
        int n = 1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_scan<TQ, C, SW, ONE>, SCAN_NT, smem) !=
            cudaSuccess)
            n = 1;
        return std::max(1, n);
    });
    const int tok = prof_begin(ix, PROF_SCAN, 1, st);
    launch_pdl(k_scan<TQ, C, SW, ONE>, grid * occ, SCAN_NT, smem, st,
               *reinterpret_cast<const CUtensorMap *>(ix->tmap_x32), a);
    prof_end(ix, tok, st);
}

// TMA descriptor of the FP32 payload in boxes of 32 floats x one slab, with
// the 128-byte swizzle: d % 32 == 0 (other rows start on other banks as they
// are, and a box past the row would only add bytes)
bool scan_make_map(sivf_index *ix)
{
    if (ix->d % 32) return false;
    auto enc = tmap_encode_fn();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)ix->d, (cuuint64_t)ix->n_slabs * ix->C};
    cuuint64_t strides[1] = {(cuuint64_t)ix->d * 4};
    cuuint32_t box[2] = {32, (cuuint32_t)ix->C};
    cuuint32_t es[2] = {1, 1};
    return enc(reinterpret_cast<CUtensorMap *>(ix->tmap_x32), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
               ix->x32, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int tune_bucket(const sivf_index *ix, int64_t nq, int P)
{
    const double r = std::max((double)nq * P / ix->nlist, 1.0 / 256);
    const int b = (int)std::floor(std::log2(r)) + 8;
    return std::min(std::max(b, 0), kTuneB - 1);
}

int tune_kbucket(int K) { return K <= 16 ? 0 : K <= 64 ? 1 : K <= 256 ? 2 : 3; }

// What an FP32 tile may ask for: its queries, two slabs with their ids and
// the rows' best K with room for two slabs of candidates (or the tile's) in
// 220 KB.  The scan keeps a block's distances instead of the ids; a tile
// that leaves no room for them is narrowed when the plan is made.
static bool fp32_fits(int TQ, int C, int d, int K, int slabs)
{
    const int v = K + (slabs ? slabs : 2) * C;
    const int M = v <= 256 ? ((v + 15) & ~15) : scan_next_pow2(slabs ? v : K + C);
    const size_t rows = ((size_t)TQ * (d + 4 + M) + (size_t)NST * C * (d + 2)) * 4;
    return ((rows + 15) & ~(size_t)15) + (size_t)TQ * M * 8 + 256 <= 220 * 1024;
}

// k-select buffer of the FP32 scan: the best K plus `slabs` slabs of
// candidates, beyond 256 entries a power of two (bitonic fallback);
// slabs = 0 is the built-in width
static int fp32_width(int K, int C, int slabs)
{
    if (slabs == 0) return scan_buf_len(K, C);
    const int v = K + slabs * C;
    return v <= 256 ? ((v + 15) & ~15) : scan_next_pow2(v);
}

sivf_tile default_tile(const sivf_index *ix, int dtype, int64_t nq, int P, int K)
{
    sivf_tile t;
    if (dtype == SIVF_FP32) {
        const double ppl = (double)nq * P / ix->nlist;
        // 16 from eight pairs per list on: 390 against 437 us at 9.8 of d = 128,
        // 315 against 285 at 7.1 of d = 192
        t.queries_per_tile = ppl >= 48 ? 64 : ppl >= 24 ? 32 : ppl >= 8 ? 16 : 8;
        while (t.queries_per_tile > 8 &&
               scan_smem(t.queries_per_tile, ix->C, ix->d, scan_buf_len(K, ix->C)).total > SCAN_SMEM)
            t.queries_per_tile >>= 1;
        t.slabs_per_chunk = 2;
        t.items_per_sm = 4;
        t.select_slabs = 0;
        t.nearest_first = 0;
    } else {
        // the vector-row scan (the query-row scan, 128, is a tile option)
        t.queries_per_tile = 64;
        t.slabs_per_chunk = 4;
        t.items_per_sm = 4;
        t.select_slabs = 0;
        t.nearest_first = 1;
    }
    return t;
}

bool tile_valid(const sivf_index *ix, int dtype, const sivf_tile &t, int K)
{
    if (t.slabs_per_chunk < 1 || t.slabs_per_chunk > 16 || t.items_per_sm < 1 ||
        t.items_per_sm > 16)
        return false;
    if (dtype == SIVF_FP32) {
        const int tq = t.queries_per_tile;
        if (!(tq == 8 || tq == 16 || tq == 32 || tq == 64)) return false;
        if (t.select_slabs < 0 || t.select_slabs > 8) return false;
        return fp32_fits(tq, ix->C, ix->d, K, t.select_slabs);
    }
    if (t.nearest_first < 0 || t.nearest_first > 2) return false;
    if (t.queries_per_tile == 128)
        return t.select_slabs >= 0 && t.select_slabs <= 3 && qt_shape(ix, dtype, K).ok;
    if (t.queries_per_tile != 64) return false;
    if (t.select_slabs < 0 || t.select_slabs > 3) return false;
    return tc_buf_fits(ix, dtype, K, tc_buf_entries(ix, dtype, K, t.select_slabs));
}

sivf_tile current_tile(const sivf_index *ix, int dtype, int64_t nq, int P, int K)
{
    const TileChoice &c = ix->tune[dtype][tune_bucket(ix, nq, P)][tune_kbucket(K)];
    if (c.set && tile_valid(ix, dtype, c.t, K)) return c.t;
    return default_tile(ix, dtype, nq, P, K);
}

SearchPlan plan_from_tile(const sivf_index *ix, int dtype, int64_t nq, int P, int K,
                          const sivf_tile &t)
{
    SearchPlan pl;
    const bool fp32 = dtype == SIVF_FP32;
    pl.qt = !fp32 && t.queries_per_tile == 128;
    pl.tq = fp32 ? t.queries_per_tile : pl.qt ? 128 : tc_tile_queries(K);
    pl.K = K;
    pl.M = fp32  ? fp32_width(K, ix->C, t.select_slabs)
           : pl.qt ? qt_shape(ix, dtype, K).ME
                   : tc_buf_entries(ix, dtype, K, t.select_slabs);
    while (fp32 && pl.tq > 8 && scan_smem(pl.tq, ix->C, ix->d, pl.M).total > SCAN_SMEM) {
        if (pl.M > scan_buf_len(K, ix->C)) pl.M = scan_buf_len(K, ix->C);
        else pl.tq >>= 1;
    }
    if (fp32 && scan_smem(pl.tq, ix->C, ix->d, pl.M).total > SCAN_SMEM) pl.M = scan_buf_len(K, ix->C);
    pl.split = fp32 ? 0 : t.nearest_first;
    pl.sel = t.select_slabs;
    pl.RK = (fp32 || pl.qt) ? K : tc_run_len(K);
    // slab chunks: a list is split when its items would be long against the
    // launch's work per SM (decided on the device from the grouped pairs);
    // at most 2048 runs per query reach the merge
    pl.ch = std::max(1, std::min(kMaxChunks, 2048 / std::max(P, 1)));
    pl.slabs_per_chunk = t.slabs_per_chunk;
    pl.ips = t.items_per_sm;
    // the other lists of split 1 run under the bounds of the nearest, so few
    // rows reach a buffer: K' > 128 takes 32-query tiles with one tile of
    // room there (half the tiles of 16)
    pl.tq2 = pl.tq;
    pl.M2 = pl.M;
    if (!fp32 && !pl.qt && pl.split == 1 && P > 1) {
        const int m2 = tc_wide_entries(ix, dtype, K);
        if (m2 > 0) {
            pl.tq2 = 32;
            pl.M2 = m2;
        }
    }
    pl.run_cap = plan_run_cap(nq, P, std::max(pl.tq, pl.tq2), pl.ips);
    pl.item_cap = plan_item_cap(nq, P, ix->nlist, pl.ips);
    return pl;
}

int64_t plan_run_cap(int64_t nq, int P, int tq, int ips)
{
    // a run per scanned pair, plus per scan phase (at most two) the chunks
    // past the first: at most tq * ips * 152
    return nq * P + 2 * (int64_t)tq * ips * 152;
}

int64_t plan_item_cap(int64_t nq, int P, int L, int ips)
{
    // a tile per (list, up to tq pairs), plus at most ips * 152 extra chunks
    return nq * P + L + (int64_t)ips * 152;
}

SearchPlan plan_search(const sivf_index *ix, int64_t nq, int P, int K)
{
    return plan_from_tile(ix, SIVF_FP32, nq, P, K, current_tile(ix, SIVF_FP32, nq, P, K));
}

bool scan_fits(const sivf_index *ix, int K)
{
    return fp32_fits(8, ix->C, ix->d, K, 0);
}

void group_pairs(sivf_index *ix, int64_t nq, int P, int p0, int p1, const int32_t *probes,
                 bool dedupe, const SearchPlan &pl, const SearchScratch &s, int64_t slab_bytes,
                 cudaStream_t st, bool stats, bool flagged)
{
    const int L = ix->nlist;
    const int64_t n = nq * (p1 - p0);
    if (n <= SH_PAIRS) {
        static KernelSetup su;
        opt_in_smem(su, k_srch_hash, SH_SMEM);
        const int tg = prof_begin(ix, PROF_GROUP, 1, st);
        launch_pdl(k_srch_hash, 1, 1024, SH_SMEM, st, probes, nq, P, p0, p1, L, dedupe,
                   flagged ? s.prank : nullptr, ix->nslabs, ix->list_live, pl.tq, pl.ch,
                   pl.slabs_per_chunk, pl.ips, pl.item_cap, slab_bytes, s.lcnt, s.loff, s.nch,
                   s.items, s.qlist, s.prun, s.qrun, ix->ctl, pl.run_cap,
                   stats ? ix->stat : nullptr, ix->err);
        prof_end(ix, tg, st);
        return;
    }
    cudaMemsetAsync(s.lcnt, 0, sizeof(int32_t) * L, st);
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16));
    const int tg = prof_begin(ix, PROF_GROUP, 3, st);
    launch_pdl(k_srch_hist, g, 256, 0, st, probes, nq, P, p0, p1, L, dedupe, flagged, s.lcnt, s.prank);
    launch_pdl(k_srch_plan, 1, 1024, 0, st, s.lcnt, ix->nslabs, ix->list_live, L, pl.tq, pl.ch,
               pl.slabs_per_chunk, pl.ips, pl.item_cap, slab_bytes, s.loff, s.nch, s.items,
               ix->ctl, stats ? ix->stat : nullptr, ix->err);
    if (p1 - p0 >= 8) {
        const int gs = (int)std::max<int64_t>(1, std::min<int64_t>((nq + SC_Q - 1) / SC_Q, 152 * 16));
        launch_pdl(k_srch_scatter, gs, SC_Q * 32, 0, st, probes, nq, P, p0, p1, s.prank, s.loff,
                   s.nch, s.qlist, s.prun, s.qrun, ix->ctl, pl.run_cap, ix->err);
    } else {
        const int gq = (int)std::max<int64_t>(1, std::min<int64_t>((nq + 255) / 256, 152 * 16));
        launch_pdl(k_srch_scatter_t, gq, 256, 0, st, probes, nq, P, p0, p1, s.prank, s.loff, s.nch,
                   s.qlist, s.prun, s.qrun, ix->ctl, pl.run_cap, ix->err);
    }
    prof_end(ix, tg, st);
}

static void scan_launch(sivf_index *ix, int tq, ScanArgs a, cudaStream_t st)
{
    a.nbs = scan_block(tq, ix->C, ix->d, a.M);
    const size_t smem = scan_smem_at(tq, ix->C, ix->d, a.M, a.nbs).total;
    const int grid = 152;  // persistent: one CTA per SM
    const bool one = smem > SCAN_HALF;
#define SIVF_SCAN_CASE(TQ_, C_)                                                                        \
    if (tq == TQ_ && ix->C == C_) {                                                                    \
        if (one || TQ_ > 16)                                                                           \
            return ix->tmap_x32_ok ? launch_scan<TQ_, C_, true, true>(ix, a, smem, grid, st)           \
                                   : launch_scan<TQ_, C_, false, true>(ix, a, smem, grid, st);         \
        return ix->tmap_x32_ok ? launch_scan<TQ_, C_, true, (TQ_ > 16)>(ix, a, smem, grid, st)         \
                               : launch_scan<TQ_, C_, false, (TQ_ > 16)>(ix, a, smem, grid, st);       \
    }
    SIVF_SCAN_CASE(8, 32) SIVF_SCAN_CASE(16, 32) SIVF_SCAN_CASE(32, 32) SIVF_SCAN_CASE(64, 32)
    SIVF_SCAN_CASE(8, 64) SIVF_SCAN_CASE(16, 64) SIVF_SCAN_CASE(32, 64) SIVF_SCAN_CASE(64, 64)
    SIVF_SCAN_CASE(8, 128) SIVF_SCAN_CASE(16, 128) SIVF_SCAN_CASE(32, 128)
    SIVF_SCAN_CASE(64, 128)
#undef SIVF_SCAN_CASE
}

void scan_lists(sivf_index *ix, const float *q, int64_t nq, int P, const int32_t *probes,
                bool dedupe, const SearchPlan &pl, const SearchScratch &s, cudaStream_t st)
{
    const int L = ix->nlist;
    cudaMemsetAsync(s.thr, 0x7f, sizeof(float) * nq, st);  // 3.4e38: no bound yet
    const int64_t sb = (int64_t)ix->C * (ix->d * 4 + 8) + ix->C / 8;

    ScanArgs a;
    a.q = q;
    a.nq = nq;
    a.P = P;
    a.K = pl.K;
    a.M = pl.M;
    a.prun = s.prun;
    a.qlist = s.qlist;
    a.loff = s.loff;
    a.lcnt = s.lcnt;
    a.nch = s.nch;
    a.part_d = s.part_d;
    a.part_i = s.part_i;
    a.thr = s.thr;
    a.items = s.items;
    a.x32 = ix->x32;
    a.ids = ix->ids;
    a.bits = ix->bits;
    a.meta = ix->meta;
    a.nslabs = ix->nslabs;
    a.dir = ix->dir;
    a.n_slabs = ix->n_slabs;
    a.dir_cap = ix->dir_cap;
    a.L = L;
    a.d = ix->d;
    a.ctl = ix->ctl;
    a.err = ix->err;
    // the nearest lists first: the others then meet a tight bound, which most
    // of their vectors do not pass and whole lists may not (prune_pairs)
    const int split = fp32_two_phase(nq, P) ? 1 : P;
    SearchPlan pl1 = pl;
    if (split < P) {
        // one pair per query: a list gets nq / nlist of them, so the tile of
        // the whole batch would stay mostly empty (64-query tiles for the 10
        // of 10,000 queries over 1,024 lists: half the warps without a row)
        pl1 = bound_plan(ix, pl);
        pl1.tq = std::min(pl.tq, current_tile(ix, SIVF_FP32, nq, 1, pl.K).queries_per_tile);
    }
    group_pairs(ix, nq, P, 0, split, probes, dedupe, pl1, s, sb, st);
    scan_launch(ix, pl1.tq, a, st);
    if (split < P) {
        prune_pairs(ix, SIVF_FP32, q, nq, P, probes, dedupe, s, st);
        group_pairs(ix, nq, P, split, P, probes, false, pl, s, sb, st, true, true);
        scan_launch(ix, pl.tq, a, st);
    }
}

void merge_topk(sivf_index *ix, int64_t nq, int P, const SearchPlan &pl,
                const SearchScratch &s, int k, float *dist, int64_t *labels, cudaStream_t st)
{
    const int nphase = fp32_two_phase(nq, P) ? 2 : 1;
    const int tok = prof_begin(ix, PROF_MERGE, 1, st);
#define SIVF_MERGE(E_)                                                                            \
    launch_pdl(k_merge<E_>, (unsigned)((nq * 32 + merge_nt(E_) - 1) / merge_nt(E_)), merge_nt(E_), 0, st, \
               s.qrun, nq, nphase, pl.K, k, s.thr, s.part_d, s.part_i, dist, labels)
    if (k <= 24) SIVF_MERGE(2);
    else if (k <= 72) SIVF_MERGE(4);
    else if (k <= 160) SIVF_MERGE(8);
    else if (k <= 448) SIVF_MERGE(16);
    else SIVF_MERGE(32);
#undef SIVF_MERGE
    prof_end(ix, tok, st);
}

}  // namespace sivf
