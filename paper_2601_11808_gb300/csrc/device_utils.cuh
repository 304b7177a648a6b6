// Device helpers: bulk async copies into shared memory completed on an
// mbarrier, mbarrier waits bounded by an iteration limit (a wait that runs
// out records ERR_TIMEOUT and returns false instead of spinning forever),
// warp reductions and order-preserving keys for floats.
#pragma once

#include <stdint.h>

#include "sivf_internal.cuh"

namespace sivf {

// -------------------------------------------------------------- mbarrier
__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)),
                 "r"(count));
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile(
        "{\n .reg .b64 st;\n"
        " mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(
            smem_u32(bar)),
        "r"(bytes)
        : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile(
        "{\n .reg .b64 st;\n"
        " mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n"
        " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// nanoseconds of the GPU's global timer
__device__ __forceinline__ uint64_t gtimer_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}


// Wait for phase `parity` of `bar`, giving up once `limit_ns` of global
// time has passed since the first unsuccessful poll (each try_wait itself
// suspends for a hardware-defined time; a poll count of 2^30 is a second
// limit in case the timer stalls).  Returns false and sets ERR_TIMEOUT
// when a limit is hit.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity,
                                                  uint32_t *err,
                                                  uint64_t limit_ns = kWaitNs)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = gtimer_ns();
    for (uint32_t it = 1; it < (1u << 30); ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (gtimer_ns() - t0 > limit_ns) break;
    }
    atomicOr(err, ERR_TIMEOUT);
    return false;
}

// mbarrier wait bounded in time (the index's wait limit) that also gives
// up as soon as another role of the CTA has stopped (abort flag in shared
// memory); a wait that runs out sets ERR_TIMEOUT and the abort flag.
// Copies already in flight are drained by the producer with the default
// limit before the CTA exits.
__device__ __forceinline__ bool mbar_wait_ab(uint64_t *bar, uint32_t parity, uint32_t *err,
                                             volatile int *abort_flag, uint64_t limit_ns)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = gtimer_ns();
    for (uint32_t it = 1; it < (1u << 30); ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63u) == 0u && *abort_flag) return false;
        if (gtimer_ns() - t0 > limit_ns) break;
    }
    atomicOr(err, ERR_TIMEOUT);
    *abort_flag = 1;
    return false;
}

// One bulk copy global -> shared of `bytes` (multiple of 16, both addresses
// 16-byte aligned) that completes transaction bytes on `bar`.
__device__ __forceinline__ void bulk_g2s(void *dst_smem, const void *src_gmem,
                                         uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1], %2, [%3];\n" ::"r"(smem_u32(dst_smem)),
        "l"(src_gmem), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// ---------------------------------------------------------------- warps
__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ uint32_t lanemask_lt()
{
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// (distance, id) lexicographic order used by every top-k
__device__ __forceinline__ bool dk_less(float a, int64_t ia, float b, int64_t ib)
{
    return a < b || (a == b && ia < ib);
}

// float -> uint32 key with the same order (for radix selection)
__device__ __forceinline__ uint32_t fkey(float f)
{
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float fkey_inv(uint32_t k)
{
    uint32_t u = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
    return __uint_as_float(u);
}

// A value at least K of the n values val(i) (n a multiple of 32, +inf for
// none) lie at or below, by a bisection on the order-preserving keys that
// stops at about K + K / 8 of them; +inf when fewer than K are finite.
template <int R, class V>  // R: values per lane held in registers (n <= 32 R)
__device__ __forceinline__ float kth_bound(V val, int n, int K, int lane)
{
    uint32_t key[R];
    const bool regs = n <= 32 * R;
    uint32_t kmin = 0xffffffffu, kmax = 0u;
    int fin = 0;
    const uint32_t kinf = fkey(INFINITY);
    auto see = [&](uint32_t k) {
        kmin = min(kmin, k);
        if (k < kinf) {
            kmax = max(kmax, k);
            ++fin;
        }
    };
    if (regs) {
#pragma unroll
        for (int e = 0; e < R; ++e) {
            key[e] = 32 * e < n ? fkey(val(32 * e + lane)) : 0xffffffffu;
            see(key[e]);
        }
    } else {
        for (int i = lane; i < n; i += 32) see(fkey(val(i)));
    }
    if (__reduce_add_sync(0xffffffffu, fin) < K) return INFINITY;
    uint32_t lo = __reduce_min_sync(0xffffffffu, kmin), hi = __reduce_max_sync(0xffffffffu, kmax);
    const int Kw = K + (K > 128 ? K >> 5 : K >> 3) + 1;
    for (int t = 0; lo < hi; ++t) {  // invariant: #(key <= hi) >= K
        // halves of the value range first (about ten, where the keys' range
        // spends its halvings on the exponents around zero), then of the keys
        uint32_t mid = lo + ((hi - lo) >> 1);
        if (t < 12) mid = min(max(fkey(0.5f * fkey_inv(lo) + 0.5f * fkey_inv(hi)), lo), hi - 1u);
        int c = 0;
        if (regs) {
#pragma unroll
            for (int e = 0; e < R; ++e) c += key[e] <= mid;
        } else {
            for (int i = lane; i < n; i += 32) c += fkey(val(i)) <= mid;
        }
        c = __reduce_add_sync(0xffffffffu, c);
        if (c >= K) hi = mid;
        else lo = mid + 1;
        if (c >= K && c <= Kw) break;
    }
    return fkey_inv(hi);
}

// Ascending bitonic sort of 32*E keys held E per lane (element i = lane + 32 e)
template <int E>
__device__ __forceinline__ void warp_sort_keys(uint64_t (&v)[E], int lane)
{
    constexpr int N = 32 * E;
#pragma unroll
    for (int size = 2; size <= N; size <<= 1)
#pragma unroll
        for (int st = size >> 1; st > 0; st >>= 1)
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const bool up = ((lane + 32 * e) & size) == 0;
                if (st >= 32) {
                    const int pe = e ^ (st >> 5);
                    if (pe > e) {
                        const uint64_t a = min(v[e], v[pe]), b = max(v[e], v[pe]);
                        v[e] = up ? a : b;
                        v[pe] = up ? b : a;
                    }
                } else {
                    const uint64_t o = __shfl_xor_sync(0xffffffffu, (unsigned long long)v[e], st);
                    v[e] = ((lane & st) == 0) == up ? min(v[e], o) : max(v[e], o);
                }
            }
}

// The n <= 32 E entries of a warp in ascending (distance, id) order: `put(place,
// distance, id)` is called once per entry.  Distances and places are sorted
// as 64-bit keys in registers; only entries of equal distance look at ids.
// (Sorting distances and 64-bit ids took three shuffles and a two-word
// comparison per stage: a third of a query's merge and re-rank.)  sk: 32 E
// keys of the warp's shared memory.
template <int E, class D, class I, class P>
__device__ __forceinline__ void warp_order(int n, D dist, I id, P put, uint64_t *sk, int lane)
{
    uint64_t ky[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = lane + 32 * e;
        ky[e] = i < n ? ((uint64_t)fkey(dist(i)) << 32) | (uint32_t)i : ~0ull;
    }
    warp_sort_keys<E>(ky, lane);
#pragma unroll
    for (int e = 0; e < E; ++e) sk[lane + 32 * e] = ky[e];
    __syncwarp();
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = lane + 32 * e;
        if (i >= n) continue;
        const uint32_t dk = (uint32_t)(ky[e] >> 32);
        const int64_t me = id((int)(uint32_t)ky[e]);
        int pos = i;
        for (int j = i - 1; j >= 0 && (uint32_t)(sk[j] >> 32) == dk; --j)
            pos -= id((int)(uint32_t)sk[j]) > me;
        for (int j = i + 1; j < n && (uint32_t)(sk[j] >> 32) == dk; ++j)
            pos += id((int)(uint32_t)sk[j]) < me;
        put(pos, fkey_inv(dk), me);
    }
}

}  // namespace sivf
