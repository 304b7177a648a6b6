// Coarse quantizer of the index (Sec. 3.3, "the coarse lists returned by
// the quantizer"): nearest centroid for insert (A1) and the nprobe nearest
// centroids for search (A4).
//
// The result must equal the FP64 definition  argmin_c sum_j (x_j - c_j)^2
// (ties to the lowest index) bit for bit.  The fast part is an FP32 GEMM
//     Dt[i][c] = fl(||c||^2 - 2 x_i.c)
// which differs from the exact  Q = ||c||^2 - 2 x.c  (= D - ||x||^2) by at
// most
//     E = 2 * ( u (fl||c||^2 + |Dt|) + 2 gamma_d ||x|| ||c|| )
// (u = 2^-24, gamma_d = d u / (1 - d u); the dot product error of any
// summation order is gamma_d sum_j |x_j c_j| <= gamma_d ||x|| ||c||; the
// factor 2 covers the roundings of the bound arithmetic itself).  The
// selection then works on intervals [Dt - E, Dt + E]:
//   T  = the P-th smallest upper bound,
//   S  = { c : lower bound <= T }         (contains the whole top-P set),
//   c in S is *sure* when UB_c <= T and fewer than P others have a lower
//   bound <= UB_c; the remaining places go to the best of the other members
//   of S by their FP64 distance, computed in the same order and with the
//   same roundings as the definition (no fused multiply-add).
// Only near-ties ever reach the FP64 step.
//
// With d % 16 == 0 the distances of the first stage come from the tensor
// cores instead (tcgen05.mma, FP32 accumulation; the BF16 product, or the
// three products of the split x = hi + lo): the same selection then runs
// twice.  With the bound of that stage (rounding of x and c plus the
// accumulation) it keeps the lists S_b that can still be among the top P;
// their distances are recomputed in FP32 and the selection above runs on S_b
// with the FP32 bound.  Lists outside S_b have exact distances above the
// P-th smallest, so the result is the same set.
//
// The forms (d % 16 == 0 and d <= 128 in the first three):
//   P = 1, 16 <= L     k_coarse_fused, k_coarse_finish: no distance matrix;
//     <= 4096            few rows: k_coarse_dist, k_coarse_near
//   2 <= P <= 128 of   k_coarse_dist, k_coarse_pick: the matrix with group
//   at least 32 P        minima, of which a row reads a few groups (P <= 8
//                        only where L d >= 32,768)
//   P <= 8, L <= 4096  k_coarse_tc (k_coarse_gemm where d % 16), then
//                        k_coarse_select_w
//   else               k_coarse_gemm (FP32), k_coarse_select
#include <float.h>
#include <math.h>

#include <cmath>

#include "device_utils.cuh"
#include "kernels.cuh"
#include "tc.cuh"

namespace sivf {

// ------------------------------------------------------------ centroid prep
// One warp per centroid, lanes over the coordinates (one thread per centroid
// walked its row with dependent FP64 additions: 63 us for 1,024 x 128).
__global__ void k_centroid_norms(const float *__restrict__ cent, int L, int d,
                                 float *__restrict__ cn, float *__restrict__ cnrm_up,
                                 float *__restrict__ cmax, uint16_t *__restrict__ cb,
                                 uint16_t *__restrict__ clo)
{
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (c >= L) return;
    const float *v = cent + (size_t)c * d;
    double s = 0.0;
    for (int j = lane; j < d; j += 32) {
        const float f = v[j];
        const double t = (double)f;
        s = __dadd_rn(s, __dmul_rn(t, t));
        if (cb) {
            const __nv_bfloat16 h = __float2bfloat16_rn(f);
            cb[(size_t)c * d + j] = *reinterpret_cast<const uint16_t *>(&h);
            if (clo) {
                const __nv_bfloat16 l = __float2bfloat16_rn(f - __bfloat162float(h));
                clo[(size_t)c * d + j] = *reinterpret_cast<const uint16_t *>(&l);
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
        const float n2 = __double2float_rn(s), nu = __double2float_ru(sqrt(s) * (1.0 + 1e-12));
        cn[c] = n2;
        cnrm_up[c] = nu;
        // the largest of each (not negative, so their bits order as integers).
        // A NaN's would be above all: its list is never chosen and counts for no
        // bound, which a NaN would make undecidable for every other list
        if (n2 == n2) {
            atomicMax(reinterpret_cast<int *>(cmax), __float_as_int(n2));
            atomicMax(reinterpret_cast<int *>(cmax) + 1, __float_as_int(nu));
        }
    }
}

// ----------------------------------------------------- FP32 tile GEMM (SIMT)
// out[i][c] = fl(cn[c] - 2 * sum_j x[i][j] * cent[c][j]) for i < m, c < L.
// 128 x 128 tiles, 256 threads, 8 x 8 outputs per thread, k-tiles of 16.
constexpr int GBM = 128, GBN = 128, GBK = 16;

__global__ __launch_bounds__(256) void k_coarse_gemm(const float *__restrict__ x, int m,
                                                     int d, const float *__restrict__ cent,
                                                     const float *__restrict__ cn, int L,
                                                     float *__restrict__ out)
{
    pdl_begin();
    __shared__ __align__(16) float As[GBK][GBM];
    __shared__ __align__(16) float Bs[GBK][GBN];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int row0 = blockIdx.y * GBM, col0 = blockIdx.x * GBN;
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;

    for (int k0 = 0; k0 < d; k0 += GBK) {
        for (int e = tid; e < GBM * GBK / 4; e += 256) {
            int r = e / (GBK / 4), c4 = e % (GBK / 4);
            int gk = k0 + c4 * 4;
            int gr = row0 + r;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (gr < m && gk < d) v = *reinterpret_cast<const float4 *>(x + (size_t)gr * d + gk);
            As[c4 * 4 + 0][r] = v.x;
            As[c4 * 4 + 1][r] = v.y;
            As[c4 * 4 + 2][r] = v.z;
            As[c4 * 4 + 3][r] = v.w;
            int gc = col0 + r;
            float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
            if (gc < L && gk < d) w = *reinterpret_cast<const float4 *>(cent + (size_t)gc * d + gk);
            Bs[c4 * 4 + 0][r] = w.x;
            Bs[c4 * 4 + 1][r] = w.y;
            Bs[c4 * 4 + 2][r] = w.z;
            Bs[c4 * 4 + 3][r] = w.w;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GBK; ++kk) {
            float4 a0 = *reinterpret_cast<const float4 *>(&As[kk][ty * 4]);
            float4 a1 = *reinterpret_cast<const float4 *>(&As[kk][64 + ty * 4]);
            float4 b0 = *reinterpret_cast<const float4 *>(&Bs[kk][tx * 4]);
            float4 b1 = *reinterpret_cast<const float4 *>(&Bs[kk][64 + tx * 4]);
            float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        int r = row0 + (i < 4 ? ty * 4 + i : 64 + ty * 4 + i - 4);
        if (r >= m) continue;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            int c = col0 + (j < 4 ? tx * 4 + j : 64 + tx * 4 + j - 4);
            if (c < L) out[(size_t)r * L + c] = fmaf(-2.f, acc[i][j], cn[c]);
        }
    }
}

// ------------------------------------------------------- exact selection
constexpr int SEL_NT = 256;
constexpr int SEL_SCAP = 1024;   // candidate capacity before the slow path

struct SelArgs {
    const float *D;        // [m, L] approximate distances (row stride L)
    int m, L, P, d;
    const float *x;        // [m, d] rows being assigned / queries
    const float *cent;     // [L, d]
    const float *cn;       // [L]
    const float *cnrm_up;  // [L]
    float gamma2;          // 2 * gamma_d
    float gamma2_first;    // the same factor for the first-stage distances D
    float gamma2_re;       // and for FP32 dot products summed across a warp (re_ops) or, by
    float gamma2_w;        // the pick, eight lanes of it (pk_ops); gamma2_w: across a warp
    int two_level;         // D is the BF16 tensor-core stage: recheck S in FP32
    const int *nhard;      // k_coarse_finish: how many records (on the device), and the
    const int32_t *S;      // records [row, n, lists...] of the rows the fused first stage
    int s_cap;             // left undecided (room for s_cap)
    float *Dw;             // refine_rows: the same distances, to be rewritten
    float *gmin;           // [m, groups of 16 lists] the distances' group minima
    const float *cmaxes;   // the largest ||c||^2 and ||c||
    int32_t *out;          // [m, P]
    uint32_t *err;
};

// FP64 distance in the order and with the roundings of the definition
__device__ __forceinline__ double exact_dist(const float *__restrict__ a,
                                             const float *__restrict__ b, int d)
{
    double acc = 0.0;
    for (int j = 0; j < d; ++j) {
        double t = __dsub_rn((double)a[j], (double)b[j]);
        acc = __dadd_rn(acc, __dmul_rn(t, t));
    }
    return acc;
}

// The same of rows whose start and length are multiples of 16 bytes (d % 4 ==
// 0): sixteen values of each loaded ahead of the additions that wait for one
// another.
__device__ __forceinline__ double exact_dist4(const float4 *a, const float4 *__restrict__ b, int d)
{
    double acc = 0.0;
    auto add = [&](float x, float y) {
        const double t = __dsub_rn((double)x, (double)y);
        acc = __dadd_rn(acc, __dmul_rn(t, t));
    };
    const int n4 = d >> 2;
    for (int j = 0; j < n4; j += 4) {
        float4 va[4], vb[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (j + u < n4) {
                va[u] = a[j + u];
                vb[u] = __ldg(b + j + u);
            }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (j + u < n4) {
                add(va[u].x, vb[u].x);
                add(va[u].y, vb[u].y);
                add(va[u].z, vb[u].z);
                add(va[u].w, vb[u].w);
            }
    }
    return acc;
}

// The same of n <= EX_FEW lists by a warp (d <= 128), the m-th list's in lane m:
// each lane squares the differences of four coordinates of every list, then the
// lanes 0 .. n-1 add up a list each, in the definition's order.  An FP64
// instruction of a warp takes the same time for one lane as for 32: a list per
// lane issues 640 of them at d = 128, this 176, which counts where several warps
// of an SM are at it; the chain of additions (about 300 cycles each) is the same.
constexpr int EX_FEW = 4;
template <class Idx>
__device__ __forceinline__ double exact_four(const float4 *x4, const float *__restrict__ cent,
                                             Idx list, int n, int d, int lane)
{
    const int n4 = d >> 2;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 xv = lane < n4 ? x4[lane] : zero;
    const double x[4] = {(double)xv.x, (double)xv.y, (double)xv.z, (double)xv.w};
    double v[4][4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const float4 cv = m < n && lane < n4
                              ? __ldg(reinterpret_cast<const float4 *>(cent + (size_t)list(m) * d) + lane)
                              : zero;
        const float c[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[m][k] = 0.0;
            if (m < n) {
                const double t = __dsub_rn(x[k], (double)c[k]);
                v[m][k] = __dmul_rn(t, t);
            }
        }
    }
    double acc = 0.0;
    for (int l = 0; l < n4; ++l)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            double t = __shfl_sync(0xffffffffu, v[0][k], l);
#pragma unroll
            for (int m = 1; m < 4; ++m)
                if (m < n) {
                    const double u = __shfl_sync(0xffffffffu, v[m][k], l);
                    if (lane == m) t = u;
                }
            acc = __dadd_rn(acc, t);
        }
    return acc;
}

// Bound E of |Dt - Q|.  Written with explicit-rounding intrinsics so that
// every evaluation for the same inputs gives the same bits (no contraction).
__device__ __forceinline__ float bound_of(float Dt, float cnc, float cnrm, float xn,
                                          float gamma2)
{
    const float u = 5.9604645e-08f;  // 2^-24
    float t1 = __fmul_rn(u, __fadd_rn(cnc, fabsf(Dt)));
    float t2 = __fmul_rn(__fmul_rn(gamma2, xn), cnrm);
    return __fadd_rn(__fmul_rn(2.f, __fadd_rn(t1, t2)), 1e-30f);
}
__device__ __forceinline__ float upper_of(float Dt, float E) { return __fadd_rn(Dt, E); }
__device__ __forceinline__ float lower_of(float Dt, float E) { return __fsub_rn(Dt, E); }

// Upper bound of ||x|| from an FP32 sum of squares of d values (any order:
// relative error <= d u).  An FP64 sum and root here held the FP64 pipe for
// most of a selection's time (rows of 128: 11 ns per row over the chip).
__device__ __forceinline__ float norm_up(float ss, int d)
{
    return __fsqrt_ru(__fmul_ru(ss, 1.f + 4.f * (float)d * 5.9604645e-08f));
}

// the smallest of a block of NT threads
template <int NT>
__device__ float block_min(float v, float *red)
{
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
        v = l < NT / 32 ? red[l] : INFINITY;
        for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (l == 0) red[0] = v;
    }
    __syncthreads();
    float r = red[0];
    __syncthreads();
    return r;
}

// the tables of one row's selection
struct SelTab {
    double dx[SEL_SCAP];
    float LB[SEL_SCAP], UB[SEL_SCAP], red[32];
    int idx[SEL_SCAP], sel[kMaxK];
    uint32_t hist[256], prefix, rank;
    int ns, nsel;
    unsigned char sure[SEL_SCAP];
};

// One row, by a block.  FRESH: the distances were written by this kernel (other
// blocks of it, too), so they are read from L2.
template <int NT, bool FRESH>
__device__ void select_row(const SelArgs &a, int row, SelTab &tab)
{
    auto ld = [](const float *p) { return FRESH ? __ldcg(p) : *p; };
    const int tid = threadIdx.x;
    const float *Dr = a.D + (size_t)row * a.L;
    const float *xr = a.x + (size_t)row * a.d;

    float *red = tab.red, *sLB = tab.LB, *sUB = tab.UB;
    uint32_t *hist = tab.hist, &s_prefix = tab.prefix, &s_rank = tab.rank;
    int &s_ns = tab.ns, &s_nsel = tab.nsel, *sIdx = tab.idx, *sSel = tab.sel;
    unsigned char *sSure = tab.sure;
    double *sDx = tab.dx;

    // every warp sums the row's squares for itself
    float part = 0.f;
    for (int j = tid & 31; j < a.d; j += 32) part = fmaf(xr[j], xr[j], part);
    const float xn = norm_up(warp_sum(part), a.d);
    const float gamma2 = a.two_level ? a.gamma2_first : a.gamma2;  // of the distances D
    __syncthreads();  // shared memory may still be read for the block's last row

    // T = P-th smallest upper bound
    float T;
    if (a.P == 1) {
        float v = INFINITY;
        for (int c = tid; c < a.L; c += NT) {
            float Dt = ld(Dr + c);
            v = fminf(v, upper_of(Dt, bound_of(Dt, a.cn[c], a.cnrm_up[c], xn, gamma2)));
        }
        T = block_min<NT>(v, red);
    } else {
        if (tid == 0) {
            s_prefix = 0;
            s_rank = (uint32_t)a.P;
        }
        uint32_t mask = 0;
        for (int pass = 0; pass < 4; ++pass) {
            const int shift = 24 - 8 * pass;
            for (int h = tid; h < 256; h += NT) hist[h] = 0;
            __syncthreads();
            const uint32_t prefix = s_prefix;
            for (int c = tid; c < a.L; c += NT) {
                float Dt = ld(Dr + c);
                uint32_t k = fkey(upper_of(Dt, bound_of(Dt, a.cn[c], a.cnrm_up[c], xn, gamma2)));
                if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & 255u], 1u);
            }
            __syncthreads();
            if (tid < 32) {
                // lane l owns bins 8l .. 8l+7
                uint32_t loc[8], s = 0;
                for (int b = 0; b < 8; ++b) {
                    loc[b] = hist[tid * 8 + b];
                    s += loc[b];
                }
                uint32_t incl = s;
                for (int o = 1; o < 32; o <<= 1) {
                    uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (tid >= o) incl += t;
                }
                uint32_t excl = incl - s, need = s_rank;
                bool mine = excl < need && incl >= need;
                if (mine) {
                    uint32_t cum = excl;
                    for (int b = 0; b < 8; ++b) {
                        if (cum + loc[b] >= need) {
                            s_prefix = prefix | ((uint32_t)(tid * 8 + b) << shift);
                            s_rank = need - cum;
                            break;
                        }
                        cum += loc[b];
                    }
                }
            }
            mask |= 255u << shift;
            __syncthreads();
        }
        T = fkey_inv(s_prefix);
    }

    // candidate set S
    if (tid == 0) {
        s_ns = 0;
        s_nsel = 0;
    }
    __syncthreads();
    for (int c = tid; c < a.L; c += NT) {
        float Dt = ld(Dr + c);
        float E = bound_of(Dt, a.cn[c], a.cnrm_up[c], xn, gamma2);
        if (lower_of(Dt, E) <= T) {
            int p = atomicAdd(&s_ns, 1);
            if (p < SEL_SCAP) {
                sLB[p] = lower_of(Dt, E);
                sUB[p] = upper_of(Dt, E);
                sIdx[p] = c;
            }
        }
    }
    __syncthreads();
    const int ns = s_ns;
    int32_t *outr = a.out + (size_t)row * a.P;

    if (ns <= SEL_SCAP) {
        // sure members
        for (int p = tid; p < ns; p += NT) {
            float ub = sUB[p];
            int cnt = 0;
            for (int q = 0; q < ns; ++q) cnt += (q != p && sLB[q] <= ub);
            bool sure = ub <= T && cnt < a.P;
            sSure[p] = sure;
            if (sure) {
                int s = atomicAdd(&s_nsel, 1);
                if (s < kMaxK) sSel[s] = sIdx[p];
            }
        }
        __syncthreads();
        const int nsure = s_nsel;
        const int r = a.P - nsure;
        if (r > 0) {
            // boundary members: exact FP64 distances, then rank among them
            const int nb = ns - nsure;
            if (nb > r) {
                for (int p = tid; p < ns; p += NT)
                    if (!sSure[p]) sDx[p] = exact_dist(xr, a.cent + (size_t)sIdx[p] * a.d, a.d);
                __syncthreads();
            }
            for (int p = tid; p < ns; p += NT) {
                if (sSure[p]) continue;
                bool take = true;
                if (nb > r) {
                    const double Dc = sDx[p];
                    const int c = sIdx[p];
                    int rank = 0;
                    for (int q = 0; q < ns; ++q) {
                        if (q == p || sSure[q]) continue;
                        rank += (sDx[q] < Dc || (sDx[q] == Dc && sIdx[q] < c));
                    }
                    take = rank < r;
                }
                if (take) {
                    int s = atomicAdd(&s_nsel, 1);
                    if (s < kMaxK) sSel[s] = sIdx[p];
                }
            }
        }
        __syncthreads();
    } else if (tid == 0) {
        // pathological: more than SEL_SCAP candidates (e.g. many identical
        // centroids).  Exact FP64 selection by insertion into a sorted
        // array of P (distance, index) pairs, scanning lists in index order.
        double *hd = sDx;  // P <= SEL_SCAP entries
        int n = 0;
        for (int c = 0; c < a.L; ++c) {
            float Dt = ld(Dr + c);
            float E = bound_of(Dt, a.cn[c], a.cnrm_up[c], xn, gamma2);
            if (lower_of(Dt, E) > T) continue;
            double Dc = exact_dist(xr, a.cent + (size_t)c * a.d, a.d);
            if (n == a.P && !(Dc < hd[n - 1])) continue;  // index order keeps ties
            int pos = n < a.P ? n : a.P - 1;
            while (pos > 0 && Dc < hd[pos - 1]) {
                hd[pos] = hd[pos - 1];
                sSel[pos] = sSel[pos - 1];
                --pos;
            }
            hd[pos] = Dc;
            sSel[pos] = c;
            if (n < a.P) ++n;
        }
        s_nsel = n;
    }
    __syncthreads();

    // write the selected set nearest first: ascending approximate distance,
    // ties to the lower list index (the set itself is the exact one)
    const int nsel = min(s_nsel, a.P);
    if (s_nsel != a.P && tid == 0) atomicOr(a.err, ERR_SELECT);
    for (int s = tid; s < nsel; s += NT) {  // their FP32 distances (P <= SEL_SCAP)
        const int c = sSel[s];
        float dc = ld(Dr + c);
        if (a.two_level) {
            float dot = 0.f;
            for (int j = 0; j < a.d; ++j) dot = fmaf(xr[j], __ldg(a.cent + (size_t)c * a.d + j), dot);
            dc = fmaf(-2.f, dot, a.cn[c]);
        }
        sLB[s] = dc;
    }
    __syncthreads();
    for (int s = tid; s < a.P; s += NT) {
        if (s >= nsel) {
            outr[s] = -1;
            continue;
        }
        const int c = sSel[s];
        const float dc = sLB[s];
        int pos = 0;
        for (int q = 0; q < nsel; ++q) {
            const int c2 = sSel[q];
            const float d2 = sLB[q];
            pos += d2 < dc || (d2 == dc && c2 < c);
        }
        outr[pos] = c;
    }
}

__global__ __launch_bounds__(SEL_NT) void k_coarse_select(SelArgs a)
{
    pdl_begin();
    __shared__ SelTab tab;
    for (int row = blockIdx.x; row < a.m; row += gridDim.x) select_row<SEL_NT, false>(a, row, tab);
}

// ------------------------------------------ BF16 tensor-core first stage
// out[i][c] = fl(cn[c] - 2 * acc[i][c]) with, accumulated in FP32 by
// tcgen05.mma,
//   SPLIT = 1:  acc = sum_j bf16(x_ij) bf16(c_cj)
//   SPLIT = 3:  acc = sum_j xh xh' ... the three leading products of
//               x = xh + xl, c = ch + cl (xh = bf16(x), xl = bf16(x - xh),
//               likewise c): xh ch + xh cl + xl ch.
// One CTA: 128 rows of x (rounded, split and swizzled by its threads)
// against 256 centroids (BF16 rows copied with cp.async), K = d (d % 16 ==
// 0), accumulator in 256 TMEM columns; four warps read their TMEM lane
// quarter back.
constexpr int CT_M = 128, CT_N = 256;
constexpr int CT_NT = 256;  // threads: 8 warps, two per TMEM lane quarter in the epilogue
constexpr int CT_AU = 4;    // A chunks each thread loads before converting

__host__ __device__ inline size_t coarse_tc_smem(int d, int split)
{
    const int KC = (d * 2 + 127) / 128;
    return (size_t)(split == 3 ? 2 : 1) * KC * (CT_M + CT_N) * 128 + 1024;
}

__device__ __forceinline__ void cp_async16_c(void *dst, const void *src, uint32_t src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(src_bytes)
                 : "memory");
}

template <int SPLIT>
__global__ __launch_bounds__(CT_NT, 1) void k_coarse_tc(const float *__restrict__ x, int m, int d,
                                                        const uint16_t *__restrict__ cb,
                                                        const uint16_t *__restrict__ clo,
                                                        const float *__restrict__ cn, int L,
                                                        float *__restrict__ out, uint32_t *err)
{
    pdl_begin();
    constexpr int NP = SPLIT == 3 ? 2 : 1;  // hi (and lo) parts
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    __shared__ uint64_t bar;
    __shared__ uint32_t tmem_base;
    const int KC = (d * 2 + 127) / 128;
    unsigned char *A = smem;                                // NP x KC x 128 rows x 128 B
    unsigned char *B = smem + (size_t)NP * KC * CT_M * 128;  // NP x KC x 256 rows x 128 B
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int row0 = blockIdx.x * CT_M, col0 = blockIdx.y * CT_N;
    const int ncol = min(CT_N, L - col0);
    if (tid == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    if (warp == 0) tmem_alloc(&tmem_base, CT_N);
    // B: BF16 centroid rows; chunks past L or d are zero
    for (int pp = 0; pp < NP; ++pp) {
        const uint16_t *src0 = pp ? clo : cb;
        unsigned char *Bp = B + (size_t)pp * KC * CT_N * 128;
        for (int e = tid; e < CT_N * KC * 8; e += CT_NT) {
            const int r = e / (KC * 8), kc = (e >> 3) % KC, c = e & 7;
            const int k0 = kc * 64 + c * 8;  // first element of the 16-byte chunk
            const bool in = col0 + r < L && k0 < d;
            cp_async16_c(Bp + (size_t)kc * CT_N * 128 + (size_t)(r >> 3) * 1024 + (r & 7) * 128 +
                             ((c ^ (r & 7)) << 4),
                         in ? (const void *)(src0 + (size_t)(col0 + r) * d + k0) : (const void *)src0,
                         in ? 16u : 0u);
        }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    // A: rows of x rounded to BF16 (round to nearest even); zero past m or d.
    // Each thread loads CT_AU chunks before converting any (loads in flight)
    const int nA = CT_M * KC * 8;
    for (int e0 = tid; e0 < nA; e0 += CT_NT * CT_AU) {
        float4 f0[CT_AU], f1[CT_AU];
#pragma unroll
        for (int u = 0; u < CT_AU; ++u) {
            const int e = e0 + u * CT_NT;
            const int r = e / (KC * 8), kc = (e >> 3) % KC, c = e & 7;
            const int k0 = kc * 64 + c * 8;
            f0[u] = f1[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (e < nA && row0 + r < m && k0 < d) {
                const float4 *xr = reinterpret_cast<const float4 *>(x + (size_t)(row0 + r) * d + k0);
                f0[u] = __ldg(xr);
                f1[u] = __ldg(xr + 1);
            }
        }
#pragma unroll
        for (int u = 0; u < CT_AU; ++u) {
            const int e = e0 + u * CT_NT;
            if (e >= nA) break;
            const int r = e / (KC * 8), kc = (e >> 3) % KC, c = e & 7;
            const float f[8] = {f0[u].x, f0[u].y, f0[u].z, f0[u].w,
                                f1[u].x, f1[u].y, f1[u].z, f1[u].w};
            uint32_t w[4], wl[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * t], f[2 * t + 1]);
                w[t] = *reinterpret_cast<uint32_t *>(&h);
                if (NP == 2) {
                    __nv_bfloat162 l = __floats2bfloat162_rn(f[2 * t] - __low2float(h),
                                                             f[2 * t + 1] - __high2float(h));
                    wl[t] = *reinterpret_cast<uint32_t *>(&l);
                }
            }
            const size_t off = (size_t)kc * CT_M * 128 + (size_t)(r >> 3) * 1024 + (r & 7) * 128 +
                               ((c ^ (r & 7)) << 4);
            *reinterpret_cast<uint4 *>(A + off) = make_uint4(w[0], w[1], w[2], w[3]);
            if (NP == 2)
                *reinterpret_cast<uint4 *>(A + (size_t)KC * CT_M * 128 + off) =
                    make_uint4(wl[0], wl[1], wl[2], wl[3]);
        }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = tmem_base;
    if (tid == 0) {
        const uint32_t idesc = mma_idesc(1, 1, CT_M, CT_N);
        // products: (x hi, c hi), then for the split (x hi, c lo), (x lo, c hi)
        constexpr int NPROD = SPLIT == 3 ? 3 : 1;
        for (int pr = 0; pr < NPROD; ++pr) {
            const int pa = pr == 2 ? 1 : 0, pb = pr == 1 ? 1 : 0;
            const uint32_t abase = smem_u32(A + (size_t)pa * KC * CT_M * 128);
            const uint32_t bbase = smem_u32(B + (size_t)pb * KC * CT_N * 128);
            for (int kc = 0; kc < KC; ++kc)
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    mma_bf16(tbase, smem_desc_sw128(abase + kc * CT_M * 128 + ks * 32, 1024),
                             smem_desc_sw128(bbase + kc * CT_N * 128 + ks * 32, 1024), idesc,
                             (pr | kc | ks) != 0);
        }
        mma_commit(&bar);
    }
    __syncwarp();
    const bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(&bar, 0, err));
    tc_fence_after();
    // epilogue: warp w reads TMEM lanes 32 (w mod 4) .. +31 (its lane
    // quarter) and every other group of 16 columns, starting at w div 4
    const int q = warp & 3, half = warp >> 2;
    const int r = row0 + q * 32 + lane;
    const bool vec = (L & 3) == 0;
    for (int c16 = half; c16 * 16 < ncol; c16 += CT_NT / 128) {  // warp-uniform
        float v[16];
        if (ok) {
            tmem_ld16(tbase + c16 * 16 + ((uint32_t)(q * 32) << 16), v);
            tmem_ld_wait();
        }
        if (!ok || r >= m) continue;
        const int cb0 = col0 + c16 * 16;
        float *o = out + (size_t)r * L + cb0;
        if (vec && c16 * 16 + 16 <= ncol) {
#pragma unroll
            for (int i4 = 0; i4 < 4; ++i4) {
                const float4 cv = __ldg(reinterpret_cast<const float4 *>(cn + cb0) + i4);
                reinterpret_cast<float4 *>(o)[i4] =
                    make_float4(fmaf(-2.f, v[4 * i4], cv.x), fmaf(-2.f, v[4 * i4 + 1], cv.y),
                                fmaf(-2.f, v[4 * i4 + 2], cv.z), fmaf(-2.f, v[4 * i4 + 3], cv.w));
            }
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (c16 * 16 + i < ncol) o[i] = fmaf(-2.f, v[i], __ldg(cn + cb0 + i));
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tbase, CT_N);
}

// ------------------------------- fused BF16 first stage for assignment
// P = 1 against ALL centroids, without writing the distance matrix.  One
// persistent CTA per SM takes tiles of 128 rows of x; the BF16 centroids
// pass once per tile in chunks of 128 (TMA boxes of 64 columns x 128 rows,
// 128-byte swizzle), one tcgen05.mma group per chunk into one of four
// 128-column TMEM buffers.  PARTS = 1: the single product, four chunk
// buffers; PARTS = 2: the split (x hi c hi + x hi c lo + x lo c hi), two.
// Warp 17 issues the copies and warp 16 the MMAs, so that a chunk is asked
// for as soon as the MMAs have read the buffer it goes into (one thread for
// both asks only when the next MMAs can be issued: 350 against 266 us for
// the split over 200,000 rows and 2,048 lists).  Warps 0-15 (four threads per row, one
// TMEM lane quarter and every fourth group of 16 columns each) hold the next
// tile's rows in registers while they work on this one, and store them
// (rounded, swizzled) as soon as the last chunk's MMAs have read the tile:
// the next tile's first MMAs run under this tile's last epilogue.
//
// Per group of 16 lists a thread takes the smallest and second smallest Dt,
// the list's place in the group carried in the key's low four mantissa bits
// (a relative change below 2^-19 of Dt), and keeps the best three groups and
// the fourth's minimum.  With Amax >= |Dt| (max ||c||^2 + 2.04 ||x|| max ||c||:
// the parts' roundings included), Ebig >= E_c for every c (the bound of the
// selection evaluated at max ||c||^2, Amax and max ||c||, rounded up) and delta
// >= the key error, T = min key + delta + Ebig is >= the smallest upper bound
// Dt_c + E_c, and a list can belong to the selection's set S only if its key is
// at most thr = T + Ebig + delta plus one unit in the last place of T (rounded
// up).  A row whose second smallest key is above thr has its argmin as the
// answer.  Any other row gets a record of the lists that can qualify (a group's
// 16 lists when its second is within thr) for k_coarse_finish, or, when they are
// more than CF_CAP, a thread's fourth group is within thr or the records are
// full, a place on its CTA's list of rows for the second pass.
// ||x|| is bounded from the FP32 sum of squares s of the tile's rows
// (relative error <= d u) as RU(sqrt(RU(s (1 + 4 d u)))).
//
// Second pass.  Several lists in one cluster are closer together than the
// products' error, so that many lists in many groups can qualify: most rows of
// the single product there, a tenth of the split's.  When its tiles are done,
// the CTA gathers those rows into tiles of their own and lets the centroids
// pass twice more, in the split form whichever form the first pass took: once
// for the smallest Dt of each row, once for a bit per list within thr, which
// k_coarse_finish decides from, however many they are.
//
// What bounds it: the epilogue's min/max and selects (4.3 half-rate
// operations per list and row); a chunk's MMAs and its copy from L2 run
// under it.  1,000,000 rows, 1,024 lists, d = 128: 526 us, 1,190 in launches
// of one tile per CTA and two passes over the centroids; the split stage,
// 200,000 rows: 141 us + 36 us to finish the undecided rows, 1,580 us when
// the matrix of distances was written and read back.  With the second pass,
// 200,000 rows of 512 trained lists in 16 clusters: 0.70 ms, 10.3 when the rows
// without a record were recomputed from every list, 2.3 by the matrix.
constexpr int CF_CAP = 32;                  // lists of one undecided row's record
constexpr int CF_SUB = 4;                   // threads per row
constexpr int CF_STRIDE = CF_CAP + 2;       // ints per record: row, n, lists
constexpr int CF_EPI = 128 * CF_SUB;        // epilogue threads
constexpr int CF_NT = CF_EPI + 64;          // + the MMA warp and the copy warp
constexpr int CF_HDR = 8;                   // ints (32 bytes) before the rows: how many records, how
                                            // many rows with bits
constexpr int CF_CN = 128;                  // centroids of a chunk (and of a TMA box)
constexpr int CF_TB = 4;                    // TMEM buffers
constexpr int CF_LMIN = 16;                 // fewer lists take the matrix form

constexpr int CW_LMAX = 4096;  // most lists of the fused stage and of one warp per row

__host__ __device__ constexpr int cf_buffers(int parts) { return parts == 1 ? 4 : 2; }
__host__ __device__ inline size_t coarse_fused_smem(int KC)
{
    // both parts of A, two chunk buffers of both parts (or four of one), ||c||^2
    return (size_t)KC * 2 * (CT_M + cf_buffers(2) * CF_CN) * 128 + CW_LMAX * 4 + 1024;
}

// Amax and Ebig: a bound of every |Dt| (the parts' roundings included), and
// of every list's bound_of, evaluated at the maxima with every step rounded
// up, times 1 + 2^-10 (covers the roundings of the bound itself)
__device__ __forceinline__ float abs_max(float cnmax, float xn, float cmax)
{
    return __fadd_ru(cnmax, __fmul_ru(__fmul_ru(2.04f, xn), cmax));
}
__device__ __forceinline__ float bound_max(float cnmax, float ab, float xn, float cmax, float g1)
{
    const float t1 = __fmul_ru(5.9604645e-08f, __fadd_ru(cnmax, ab));
    const float t2 = __fmul_ru(__fmul_ru(g1, xn), cmax);
    return __fadd_ru(__fmul_ru(__fmul_ru(2.f, __fadd_ru(t1, t2)), 1.f + 1.f / 1024.f), 1e-30f);
}

__device__ __forceinline__ float min3f(float a, float b, float c)
{
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// The largest split distance a list of the P nearest can have, from a value b
// that P lists lie at or below: Dt - E <= T with T = b + Ebig needs Dt <= T +
// Ebig + its roundings
__device__ __forceinline__ float pick_limit(float b, float eb)
{
    const float T0 = __fadd_ru(b, eb);
    return __fadd_ru(__fadd_ru(T0, eb), __fadd_ru(__fmul_ru(fabsf(T0), 1.2e-7f), 1e-30f));
}

// A tile of 128 rows held in registers by CF_EPI threads: fetched as FP32
// (zero past m or d), stored rounded to BF16 (and its low parts, abytes
// further) in the swizzled operand layout; sxn receives the norms' bounds.
template <int KC, int PARTS>
struct RowTile {
    static constexpr int W = KC * 8;              // 16-byte chunks of a row
    static constexpr int AU = CT_M * W / CF_EPI;  // chunks per thread: 2 KC
    float4 f0[AU], f1[AU];
    // row_of(r): the row of x in the tile's place r, -1 for none
    template <class R>
    __device__ __forceinline__ void fetch(const float *__restrict__ x, R row_of, int d, int tid)
    {
#pragma unroll
        for (int u = 0; u < AU; ++u) {
            const int e = tid + u * CF_EPI, row = row_of(e / W), k0 = (e & (W - 1)) * 8;
            f0[u] = f1[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row >= 0 && k0 < d) {
                const float4 *xr = reinterpret_cast<const float4 *>(x + (size_t)row * d + k0);
                f0[u] = __ldg(xr);
                f1[u] = __ldg(xr + 1);
            }
        }
    }
    __device__ __forceinline__ void store(unsigned char *A, uint32_t abytes, int d, int tid, float *sxn)
    {
        const float fx = 1.f + 4.f * (float)d * 5.9604645e-08f;
#pragma unroll
        for (int u = 0; u < AU; ++u) {
            const int e = tid + u * CF_EPI, r = e / W, kc = (e >> 3) % KC, c = e & 7;
            const float f[8] = {f0[u].x, f0[u].y, f0[u].z, f0[u].w,
                                f1[u].x, f1[u].y, f1[u].z, f1[u].w};
            uint32_t w[4], wl[4];
            float sq = 0.f;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * t], f[2 * t + 1]);
                w[t] = *reinterpret_cast<uint32_t *>(&h);
                if (PARTS == 2) {
                    __nv_bfloat162 l = __floats2bfloat162_rn(f[2 * t] - __low2float(h),
                                                             f[2 * t + 1] - __high2float(h));
                    wl[t] = *reinterpret_cast<uint32_t *>(&l);
                }
                sq = fmaf(f[2 * t], f[2 * t], sq);
                sq = fmaf(f[2 * t + 1], f[2 * t + 1], sq);
            }
            unsigned char *o = A + (size_t)kc * CT_M * 128 + (size_t)(r >> 3) * 1024 + (r & 7) * 128 +
                               ((c ^ (r & 7)) << 4);
            *reinterpret_cast<uint4 *>(o) = make_uint4(w[0], w[1], w[2], w[3]);
            if (PARTS == 2)
                *reinterpret_cast<uint4 *>(o + abytes) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
            // the W chunks of a row sit in consecutive lanes
#pragma unroll
            for (int t = W >> 1; t > 0; t >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, t);
            if ((tid & (W - 1)) == 0) sxn[r] = __fsqrt_ru(__fmul_ru(sq, fx));
        }
    }
};

// The nearest of a row's candidate lists (one warp; d <= 128: one float4 of the
// row per lane).  The FP32 distances of up to ND_WIN lists at a time (ND_RG in
// flight); those whose lower bound is at most the smallest upper bound so far
// stay for the next window, and of the last that stay, when they are several,
// the FP64 distances decide (ties to the lower index).  fill(at, w0) writes the
// candidates' numbers from the w0-th on to tab[at, ND_WIN) and returns how many
// there are in all.  tab, lbs: ND_WIN entries of the warp's shared memory.  -1
// when no list qualifies.
constexpr int ND_WIN = 64;
constexpr int ND_RG = 8;
struct NearArgs {
    const float *cent, *cn, *cnrm_up;
    float gamma_re;      // bound_of's factor of FP32 dot products summed across a warp
};
template <class Fill>
__device__ __forceinline__ int decide_nearest(const NearArgs &a, Fill fill, int d, const float *xr,
                                              float xn, int *tab, float *lbs, int lane)
{
    const int n4 = d >> 2;
    const float4 *x4 = reinterpret_cast<const float4 *>(xr);
    const float4 xv = lane < n4 ? __ldg(x4 + lane) : make_float4(0.f, 0.f, 0.f, 0.f);
    double bd = INFINITY;  // the best by FP64 distance and index
    int bc = 0x7fffffff;
    bool exact = false;    // some were decided by FP64 distance
    // the FP64 distances of the k lists in the table, next to each other: a pass
    // costs the same for one as for 32
    auto decide = [&](int k) {
        auto take = [&](double D, int c) {
            if (D < bd || (D == bd && c < bc)) {
                bd = D;
                bc = c;
            }
        };
        if (k <= EX_FEW) {
            const double D = exact_four(x4, a.cent, [&](int m) { return tab[m]; }, k, d, lane);
            if (lane < k) take(D, tab[lane]);
        } else {
            for (int p = lane; p < k; p += 32)
                take(exact_dist4(x4, reinterpret_cast<const float4 *>(a.cent + (size_t)tab[p] * d), d),
                     tab[p]);
        }
        exact = true;
        __syncwarp();
    };
    int total = fill(0, 0), k = 0;  // k: lists that stay
    if (total == 0) return -1;
    if (total == 1) return tab[0];
    float T = INFINITY;
    for (int w0 = 0; w0 < total;) {
        const int n = k + min(total - w0, ND_WIN - k);
        if (w0 > 0) fill(k, w0);
        w0 += n - k;
        for (int p0 = k; p0 < n; p0 += ND_RG) {
            float s[ND_RG];
#pragma unroll
            for (int t = 0; t < ND_RG; ++t) {
                const float4 *c4 = reinterpret_cast<const float4 *>(a.cent + (size_t)tab[min(p0 + t, n - 1)] * d);
                const float4 cv = lane < n4 ? __ldg(c4 + lane) : make_float4(0.f, 0.f, 0.f, 0.f);
                s[t] = fmaf(xv.w, cv.w, fmaf(xv.z, cv.z, fmaf(xv.y, cv.y, xv.x * cv.x)));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int t = 0; t < ND_RG; ++t) s[t] += __shfl_xor_sync(0xffffffffu, s[t], o);
            float dot = s[0];
#pragma unroll
            for (int t = 1; t < ND_RG; ++t)
                if (lane == t) dot = s[t];
            if (lane < ND_RG && p0 + lane < n) {
                const int c = tab[p0 + lane];
                const float cnc = __ldg(a.cn + c), Dt = fmaf(-2.f, dot, cnc);
                const float E = bound_of(Dt, cnc, __ldg(a.cnrm_up + c), xn, a.gamma_re);
                lbs[p0 + lane] = lower_of(Dt, E);
                T = fminf(T, upper_of(Dt, E));
            }
        }
        for (int o = 16; o > 0; o >>= 1) T = fminf(T, __shfl_xor_sync(0xffffffffu, T, o));
        __syncwarp();
        k = 0;
        for (int p0 = 0; p0 < n; p0 += 32) {  // every place is at most the one it is read from
            const bool in = p0 + lane < n && lbs[p0 + lane] <= T;
            const int c = in ? tab[p0 + lane] : 0;
            const float lb = in ? lbs[p0 + lane] : 0.f;
            const uint32_t mk = __ballot_sync(0xffffffffu, in);
            __syncwarp();
            if (in) {
                tab[k + __popc(mk & lanemask_lt())] = c;
                lbs[k + __popc(mk & lanemask_lt())] = lb;
            }
            k += __popc(mk);
            __syncwarp();
        }
        if (k > ND_WIN / 2 && w0 < total) {  // room for the next window
            decide(k);
            k = 0;
        }
    }
    if (!exact && k <= 1) return k == 1 ? tab[0] : -1;
    if (k > 0) decide(k);
    for (int o = 16; o > 0; o >>= 1) {
        const double od = __shfl_xor_sync(0xffffffffu, bd, o);
        const int oc = __shfl_xor_sync(0xffffffffu, bc, o);
        if (od < bd || (od == bd && oc < bc)) {
            bd = od;
            bc = oc;
        }
    }
    return bc;
}

// Second pass of the fused stage: arguments, barriers, the pass itself.
struct SecondArgs {
    int32_t *rows;       // [m] the rows of each CTA's list (second_place)
    int32_t *list;       // [m] the places of those whose bits are written, and
    int *n;              // how many
    uint16_t *bits;      // [m / 128][groups of 16 lists][stride] lists within thr, by place
    int stride;          // rows of a tile: 128, or all there are
    float gamma;         // the split products' factor in bound_of
};
// where a CTA keeps the p-th row of its list: as far down its own tiles
__device__ __forceinline__ int second_place(int p)
{
    return (int)(blockIdx.x + (uint32_t)(p >> 7) * gridDim.x) * CT_M + (p & 127);
}
struct SecondBars {
    uint64_t fullb[2], freeb[2], mmab[CF_TB], tempty[CF_TB], afull;
    __device__ void init()
    {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&fullb[i], 1);
            mbar_init(&freeb[i], 1);
        }
        for (int i = 0; i < CF_TB; ++i) {
            mbar_init(&mmab[i], 1);
            mbar_init(&tempty[i], CF_EPI / 32);
        }
        mbar_init(&afull, CF_EPI / 32);
    }
};

template <int KC>
__device__ __noinline__ void second_pass(const CUtensorMap &tmB, const CUtensorMap &tmBlo,
                                         const float *__restrict__ x, int d, int L, int n,
                                         const SecondArgs &a, int32_t *__restrict__ out1,
                                         unsigned char *A, unsigned char *B, const float *scn,
                                         const float *cmaxes, uint32_t tbase, SecondBars &bar,
                                         volatile int *s_abort, float *sxn, float (*sMin)[CT_M],
                                         int *srow, uint32_t *err)
{
    constexpr int CN = CF_CN, NB = 2, TB = CF_TB;
    constexpr uint32_t PBYTES = KC * CN * 128, BBYTES = 2 * PBYTES, ABYTES = KC * CT_M * 128;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nch = (L + CN - 1) / CN, ntiles = (n + CT_M - 1) / CT_M, G = (L + 15) / 16;
    const uint32_t steps = (uint32_t)ntiles * 2u * (uint32_t)nch;
    if (warp == CF_EPI / 32 + 1) {
        // ---- copies (one lane)
        if (lane == 0) {
            uint32_t g = 0;
            for (; g < steps; ++g) {
                const uint32_t b = g % NB, u = g / NB;
                if (u >= 1 && !mbar_wait_ab(&bar.freeb[b], (u - 1) & 1, err, s_abort, kWaitNs)) break;
                const int j = (int)(g % (uint32_t)nch);
                mbar_arrive_expect_tx(&bar.fullb[b], BBYTES);
#pragma unroll
                for (int pp = 0; pp < 2; ++pp)
#pragma unroll
                    for (int kc = 0; kc < KC; ++kc)
                        tma_load_2d(B + b * BBYTES + pp * PBYTES + (size_t)kc * CN * 128,
                                    pp ? &tmBlo : &tmB, kc * 64, j * CN, &bar.fullb[b]);
            }
            for (uint32_t t = g > NB ? g - NB : 0; t < g; ++t)  // landed before exit
                mbar_wait_bounded(&bar.fullb[t % NB], (t / NB) & 1, err);
        }
        __syncwarp();
    } else if (warp == CF_EPI / 32) {
        // ---- MMAs (one lane)
        if (lane == 0) {
            const uint32_t idesc = mma_idesc(1, 1, CT_M, CN), abase = smem_u32(A);
            uint32_t g = 0;
            for (; g < steps; ++g) {
                const uint32_t b = g % NB, tb = g % TB, ut = g / TB;
                bool ok = mbar_wait_ab(&bar.fullb[b], (g / NB) & 1, err, s_abort, kWaitNs);
                if (ok && g % (2u * (uint32_t)nch) == 0)  // the tile's rows are stored
                    ok = mbar_wait_ab(&bar.afull, (g / (2u * (uint32_t)nch)) & 1, err, s_abort, kWaitNs);
                if (ok && ut >= 1) ok = mbar_wait_ab(&bar.tempty[tb], (ut - 1) & 1, err, s_abort, kWaitNs);
                if (!ok) break;
                tc_fence_after();
                const uint32_t bbase = smem_u32(B + b * BBYTES);
#pragma unroll
                for (int pr = 0; pr < 3; ++pr) {  // (x hi, c hi), (x hi, c lo), (x lo, c hi)
                    const uint32_t ap = abase + (pr == 2 ? ABYTES : 0u);
                    const uint32_t bp = bbase + (pr == 1 ? PBYTES : 0u);
#pragma unroll
                    for (int kc = 0; kc < KC; ++kc)
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            mma_bf16(tbase + tb * CN,
                                     smem_desc_sw128(ap + kc * CT_M * 128 + ks * 32, 1024),
                                     smem_desc_sw128(bp + kc * CN * 128 + ks * 32, 1024), idesc,
                                     (pr | kc | ks) != 0);
                }
                mma_commit(&bar.freeb[b]);
                mma_commit(&bar.mmab[tb]);
            }
            if (g > 0) mbar_wait_bounded(&bar.mmab[(g - 1) % TB], ((g - 1) / TB) & 1, err);
        }
        __syncwarp();
    } else {
        // ---- rows in, epilogue
        const int q = warp & 3, sub = warp >> 2, rloc = q * 32 + lane;
        const float cnmax = __ldg(cmaxes), cmax = __ldg(cmaxes + 1);
        uint32_t g = 0;
        bool ok = true;
        RowTile<KC, 2> rows;
        for (int t = 0; t < ntiles; ++t) {
            const int nrow = min(CT_M, n - t * CT_M), place = second_place(t * CT_M);
            uint16_t *bits = a.bits + (size_t)(place >> 7) * G * a.stride;
            if (tid < CT_M) srow[tid] = tid < nrow ? a.rows[second_place(t * CT_M + tid)] : -1;
            named_bar_sync(1, CF_EPI);
            rows.fetch(x, [&](int r) { return srow[r]; }, d, tid);
            rows.store(A, ABYTES, d, tid, sxn);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar.afull);
            float mn = INFINITY, thr = 0.f;
            for (int pass = 0; pass < 2; ++pass) {
                for (int j = 0; j < nch; ++j, ++g) {
                    const uint32_t tb = g % TB;
                    ok = __all_sync(0xffffffffu, ok && mbar_wait_ab(&bar.mmab[tb], (g / TB) & 1, err,
                                                                    s_abort, kWaitNs));
                    tc_fence_after();
                    if (ok) {
                        const uint32_t tad = tbase + tb * CN + sub * 16 + ((uint32_t)(q * 32) << 16);
#pragma unroll
                        for (int k = 0; k < CN / 64; ++k) {
                            const int grp = j * (CN / 16) + sub + 4 * k;
                            const float4 *cv4 = reinterpret_cast<const float4 *>(scn + grp * 16);
                            float v[16];
                            tmem_ld16(tad + k * 64, v);
                            tmem_ld_wait(v);
                            uint32_t within = 0u;
#pragma unroll
                            for (int i4 = 0; i4 < 4; ++i4) {
                                const float4 cv = cv4[i4];
                                const float c4[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    const float Dt = fmaf(-2.f, v[4 * i4 + i], c4[i]);
                                    if (pass == 0) mn = fminf(mn, Dt);
                                    else if (Dt <= thr) within |= 1u << (4 * i4 + i);
                                }
                            }
                            if (pass == 1 && grp < G && rloc < nrow) {
                                if (L - grp * 16 < 16) within &= (1u << (L - grp * 16)) - 1u;
                                bits[(size_t)grp * a.stride + rloc] = (uint16_t)within;
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar.tempty[tb]);
                }
                if (pass == 0) {
                    sMin[sub][rloc] = mn;
                    ok = named_bar_and(1, CF_EPI, ok && !*s_abort);
                    if (!ok) break;
                    mn = fminf(fminf(sMin[0][rloc], sMin[1][rloc]), fminf(sMin[2][rloc], sMin[3][rloc]));
                    const float xn = sxn[rloc];
                    const float eb = bound_max(cnmax, abs_max(cnmax, xn, cmax), xn, cmax, a.gamma);
                    thr = pick_limit(mn, eb);
                }
            }
            if (ok) ok = named_bar_and(1, CF_EPI, ok && !*s_abort);
            if (!ok) {
                // a wait ran out (the sticky error word is set): list 0 for the rows left
                for (int p = t * CT_M + tid; p < n; p += CF_EPI) out1[a.rows[second_place(p)]] = 0;
                break;
            }
            if (tid < nrow) a.list[atomicAdd(a.n, 1)] = place + tid;
            named_bar_sync(1, CF_EPI);  // srow, sxn and sMin are reused
        }
    }
}

template <int KC, int PARTS>
__global__ __launch_bounds__(CF_NT, 1) void k_coarse_fused(
    const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmBlo,
    const float *__restrict__ x, int m, int d, const float *__restrict__ cn,
    const float *__restrict__ cmaxes, int L, float g1, int32_t *__restrict__ out1,
    int32_t *__restrict__ outS, int cap, int *nhard, const __grid_constant__ SecondArgs sp,
    uint32_t *err)
{
    pdl_begin();
    constexpr int CN = CF_CN, NB = cf_buffers(PARTS), TB = CF_TB;
    constexpr uint32_t PBYTES = KC * CN * 128;    // one part of a chunk
    constexpr uint32_t BBYTES = PARTS * PBYTES;
    constexpr uint32_t ABYTES = KC * CT_M * 128;  // one part of the row tile
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    unsigned char *A = smem;                               // 2 x KC x 128 rows x 128 B
    unsigned char *B = smem + 2 * ABYTES;                  // NB x PARTS x KC x CN rows x 128 B
    float *scn = reinterpret_cast<float *>(B + NB * BBYTES);
    // chunk copied, chunk read (both per chunk buffer), products ready,
    // products read (per TMEM buffer), row tile stored
    __shared__ uint64_t fullb[NB], freeb[NB], mmab[TB], tempty[TB], afull;
    __shared__ SecondBars bars2;
    __shared__ uint32_t tmem_base;
    __shared__ int s_abort_, s_second;  // s_second: rows left to the second pass
    volatile int *s_abort = &s_abort_;
    // by tile parity: the row's norm, and each thread's best key, its list,
    // the best key of its other lists, and its candidate count
    __shared__ float sxn[2][CT_M], sMin[2][CF_SUB][CT_M], sSec[2][CF_SUB][CT_M];
    __shared__ int sArg[2][CF_SUB][CT_M], sn[CF_SUB][CT_M];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < NB; ++i) {
            mbar_init(&fullb[i], 1);
            mbar_init(&freeb[i], 1);
        }
        for (int i = 0; i < TB; ++i) {
            mbar_init(&mmab[i], 1);
            mbar_init(&tempty[i], CF_EPI / 32);
        }
        mbar_init(&afull, CF_EPI / 32);
        bars2.init();
        fence_mbar_init();
        s_abort_ = 0;
        s_second = 0;
    }
    if (warp == CF_EPI / 32) tmem_alloc(&tmem_base, TB * CN);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = tmem_base;
    const int nch = (L + CN - 1) / CN, ntiles = (m + CT_M - 1) / CT_M;
    const uint32_t mine = (ntiles - 1 - blockIdx.x) / gridDim.x + 1;  // gridDim.x <= ntiles

    if (warp == CF_EPI / 32 + 1) {
        // ---- copies (one lane)
        if (lane == 0) {
            const uint32_t steps = mine * (uint32_t)nch;
            uint32_t g = 0;
            for (; g < steps; ++g) {
                const uint32_t b = g % NB, u = g / NB;
                if (u >= 1 && !mbar_wait_ab(&freeb[b], (u - 1) & 1, err, s_abort, kWaitNs)) break;
                const int j = (int)(g % (uint32_t)nch);
                mbar_arrive_expect_tx(&fullb[b], BBYTES);
#pragma unroll
                for (int pp = 0; pp < PARTS; ++pp)
#pragma unroll
                    for (int kc = 0; kc < KC; ++kc)
                        tma_load_2d(B + b * BBYTES + pp * PBYTES + (size_t)kc * CN * 128,
                                    pp ? &tmBlo : &tmB, kc * 64, j * CN, &fullb[b]);
            }
            // the copies issued last have landed before exit
            for (uint32_t t = g > NB ? g - NB : 0; t < g; ++t)
                mbar_wait_bounded(&fullb[t % NB], (t / NB) & 1, err);
        }
        __syncwarp();
    } else if (warp == CF_EPI / 32) {
        // ---- MMAs (one lane)
        if (lane == 0) {
            const uint32_t steps = mine * (uint32_t)nch;
            const uint32_t idesc = mma_idesc(1, 1, CT_M, CN);
            const uint32_t abase = smem_u32(A);
            uint32_t g = 0;
            for (; g < steps; ++g) {
                const uint32_t b = g % NB, tb = g % TB, ut = g / TB;
                bool ok = mbar_wait_ab(&fullb[b], (g / NB) & 1, err, s_abort, kWaitNs);
                if (ok && g % (uint32_t)nch == 0)  // the tile's rows are stored
                    ok = mbar_wait_ab(&afull, (g / (uint32_t)nch) & 1, err, s_abort, kWaitNs);
                if (ok && ut >= 1)  // this TMEM buffer has been read
                    ok = mbar_wait_ab(&tempty[tb], (ut - 1) & 1, err, s_abort, kWaitNs);
                if (!ok) break;
                tc_fence_after();
                const uint32_t bbase = smem_u32(B + b * BBYTES);
                // products: (x hi, c hi), then for the split (x hi, c lo), (x lo, c hi)
#pragma unroll
                for (int pr = 0; pr < (PARTS == 2 ? 3 : 1); ++pr) {
                    const uint32_t ap = abase + (pr == 2 ? ABYTES : 0u);
                    const uint32_t bp = bbase + (pr == 1 ? PBYTES : 0u);
#pragma unroll
                    for (int kc = 0; kc < KC; ++kc)
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            mma_bf16(tbase + tb * CN,
                                     smem_desc_sw128(ap + kc * CT_M * 128 + ks * 32, 1024),
                                     smem_desc_sw128(bp + kc * CN * 128 + ks * 32, 1024), idesc,
                                     (pr | kc | ks) != 0);
                }
                mma_commit(&freeb[b]);
                mma_commit(&mmab[tb]);
            }
            // the last products are written before TMEM is released
            if (g > 0) mbar_wait_bounded(&mmab[(g - 1) % TB], ((g - 1) / TB) & 1, err);
        }
        __syncwarp();
    } else {
        // ---- rows in, epilogue
        const int q = warp & 3, sub = warp >> 2, rloc = q * 32 + lane;
        RowTile<KC, PARTS> rows;
        auto fetch = [&](int tile) {
            rows.fetch(x, [&](int r) { return tile * CT_M + r < m ? tile * CT_M + r : -1; }, d, tid);
        };
        auto store = [&](int par) {
            rows.store(A, ABYTES, d, tid, sxn[par]);
            fence_proxy_async_smem();  // A (generic stores) is read by the MMAs
            __syncwarp();
            if (lane == 0) mbar_arrive(&afull);
        };
        fetch((int)blockIdx.x);
        store(0);
        // ||c||^2, lists past L far away
        for (int c = tid; c < nch * CN; c += CF_EPI) scn[c] = c < L ? __ldg(cn + c) : 3.0e38f;
        named_bar_sync(1, CF_EPI);
        const float cnmax = __ldg(cmaxes), cmax = __ldg(cmaxes + 1);
        uint32_t g = 0;
        bool ok = true;
        for (uint32_t t = 0; t < mine; ++t) {
            const int tile = (int)(blockIdx.x + t * gridDim.x), row = tile * CT_M + rloc;
            const int par = (int)(t & 1);
            const bool more = t + 1 < mine;
            if (more) fetch(tile + (int)gridDim.x);
            // the best three groups (key, second key in it, group) and the
            // best key of the others
            float dg[3], sg[3], d4 = 3.3e38f;
            int gi[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                dg[i] = sg[i] = 3.3e38f;
                gi[i] = 0;
            }
            for (int j = 0; j < nch; ++j, ++g) {
                const uint32_t b = g % TB;
                ok = __all_sync(0xffffffffu, ok && mbar_wait_ab(&mmab[b], (g / TB) & 1, err, s_abort,
                                                                kWaitNs));
                tc_fence_after();
                if (j == nch - 1 && more && ok) store(par ^ 1);  // this tile's MMAs are done
                if (ok) {
                    const uint32_t tad = tbase + b * CN + sub * 16 + ((uint32_t)(q * 32) << 16);
#pragma unroll
                    for (int k = 0; k < CN / 64; ++k) {
                        const int grp = j * (CN / 16) + sub + 4 * k;
                        const float4 *cv4 = reinterpret_cast<const float4 *>(scn + grp * 16);
                        float v[16];
                        tmem_ld16(tad + k * 64, v);
                        tmem_ld_wait(v);
                        // the smallest key of the group and its second: any other key
                        // is in another row or another column of the 4 x 4 square, so
                        // the second is the smaller second of the rows' and of the
                        // columns' minima (30 operations, 37 by a tree of pairs)
                        float key[16];
#pragma unroll
                        for (int i4 = 0; i4 < 4; ++i4) {
                            const float4 cv = cv4[i4];
                            const float c4[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const float Dt = fmaf(-2.f, v[4 * i4 + i], c4[i]);
                                key[4 * i4 + i] = __uint_as_float((__float_as_uint(Dt) & ~15u) |
                                                                  (uint32_t)(4 * i4 + i));
                            }
                        }
                        float rw[4], cl[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            rw[i] = min3f(key[4 * i], key[4 * i + 1], fminf(key[4 * i + 2], key[4 * i + 3]));
                            cl[i] = min3f(key[i], key[4 + i], fminf(key[8 + i], key[12 + i]));
                        }
                        const float ra = fminf(rw[0], rw[1]), rb = fminf(rw[2], rw[3]);
                        const float ca = fminf(cl[0], cl[1]), cb = fminf(cl[2], cl[3]);
                        const float r2 = min3f(fmaxf(rw[0], rw[1]), fmaxf(rw[2], rw[3]), fmaxf(ra, rb));
                        const float c2 = min3f(fmaxf(cl[0], cl[1]), fmaxf(cl[2], cl[3]), fmaxf(ca, cb));
                        // insert the group into the sorted three
                        float mv = fminf(ra, rb), ms = fminf(r2, c2);
                        int mg = grp;
#pragma unroll
                        for (int i = 0; i < 3; ++i) {
                            const bool lt = mv < dg[i];
                            const float td = dg[i], ts = sg[i];
                            const int tg = gi[i];
                            dg[i] = lt ? mv : td;
                            sg[i] = lt ? ms : ts;
                            gi[i] = lt ? mg : tg;
                            mv = lt ? td : mv;
                            ms = lt ? ts : ms;
                            mg = lt ? tg : mg;
                        }
                        d4 = fminf(d4, mv);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty[b]);
            }
            const int c1 = gi[0] * 16 + (int)(__float_as_uint(dg[0]) & 15u);
            sMin[par][sub][rloc] = dg[0];
            sSec[par][sub][rloc] = fminf(sg[0], dg[1]);
            sArg[par][sub][rloc] = c1;
            ok = named_bar_and(1, CF_EPI, ok && !*s_abort);
            if (!ok) {
                // a wait ran out (the sticky error word is set): the rows left
                // get list 0, so that nothing downstream reads garbage
                for (uint32_t t2 = t; t2 < mine; ++t2) {
                    const int r = (int)(blockIdx.x + t2 * gridDim.x) * CT_M + rloc;
                    if (sub == 0 && r < m) out1[r] = 0;
                }
                break;
            }
            int kmin = 0;
            float mn = sMin[par][0][rloc];
#pragma unroll
            for (int k = 1; k < CF_SUB; ++k) {
                const float v = sMin[par][k][rloc];
                if (v < mn) kmin = k;
                mn = fminf(mn, v);
            }
            float second = sSec[par][kmin][rloc];
#pragma unroll
            for (int k = 0; k < CF_SUB; ++k)
                if (k != kmin) second = fminf(second, sMin[par][k][rloc]);
            const float xn = sxn[par][rloc];
            const float ab = abs_max(cnmax, xn, cmax), eb = bound_max(cnmax, ab, xn, cmax, g1);
            const float delta = __fadd_ru(__fmul_ru(ab, 1.9073486e-06f), 1e-36f);  // 2^-19
            const float T = __fadd_ru(__fadd_ru(mn, delta), eb);
            // RN(Dt - E) <= T needs Dt < T + E + ulp(T) <= thr - delta
            const float thr = __fadd_ru(__fadd_ru(__fadd_ru(T, eb), delta),
                                        __fadd_ru(__fmul_ru(fabsf(T), 1.2e-7f), 1e-30f));
            const bool decided = !(second <= thr) && mn <= thr;
            if (decided && sub == 0 && row < m) out1[row] = sArg[par][kmin][rloc];
            if (!named_bar_or(1, CF_EPI, !decided && row < m)) continue;
            // undecided rows: each thread's lists that can qualify (a whole group
            // may reach past L, whose lists never qualify)
            int nl[3], nmine = 0;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                nl[i] = !(dg[i] <= thr) ? 0 : sg[i] <= thr ? max(0, min(16, L - gi[i] * 16)) : 1;
                nmine += nl[i];
            }
            sn[sub][rloc] = d4 <= thr ? -1 : nmine;
            named_bar_sync(1, CF_EPI);
            int h = -1, before = 0, total = 0;
            if (!decided && row < m) {
                bool redo = false;
#pragma unroll
                for (int k = 0; k < CF_SUB; ++k) {
                    const int nk = sn[k][rloc];
                    redo |= nk < 0;
                    before += k < sub ? nk : 0;
                    total += nk;
                }
                if (sub == 0) {
                    redo |= total > CF_CAP;
                    if (!redo) {
                        h = atomicAdd(nhard, 1);
                        redo = h >= cap;
                        if (redo) h = -1;
                    }
                    if (redo) {
                        sp.rows[second_place(atomicAdd(&s_second, 1))] = row;
                    } else {
                        outS[(size_t)h * CF_STRIDE] = row;
                        outS[(size_t)h * CF_STRIDE + 1] = total;
                    }
                }
            }
            if (sub == 0) sArg[par][0][rloc] = h;  // the row's record, for its other threads
            named_bar_sync(1, CF_EPI);
            if (!decided && row < m) {
                h = sArg[par][0][rloc];
                if (h >= 0) {
                    int32_t *o = outS + (size_t)h * CF_STRIDE + 2 + before;
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        const bool whole = sg[i] <= thr;
                        const int first = gi[i] * 16 + (whole ? 0 : (int)(__float_as_uint(dg[i]) & 15u));
                        for (int k = 0; k < nl[i]; ++k) *o++ = min(first + k, L - 1);
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const int nsecond = s_second;
    if (nsecond > 0 && !s_abort_) {
        second_pass<KC>(tmB, tmBlo, x, d, L, nsecond, sp, out1, A, B, scn, cmaxes, tbase, bars2,
                        s_abort, sxn[0], sMin[0], &sn[0][0], err);
    } else if (nsecond > 0 && tid < CF_EPI) {  // a wait ran out: list 0, as above
        for (int p = tid; p < nsecond; p += CF_EPI) out1[sp.rows[second_place(p)]] = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == CF_EPI / 32) tmem_dealloc(tbase, TB * CN);
}

// ------------------------------------ split first stage for probe selection
// Dt of tiles of 128 rows against the centroids' chunks, in the split BF16
// form, written to out[row][list], and the smallest Dt of each group of 16
// lists to gmin[row][group].  Roles and buffers as in k_coarse_fused.  The
// (tile, chunk) steps are dealt out evenly, a contiguous range per CTA, so
// that a few rows over many lists fill the chip as well as many over few.
// Bound by its stores: a thread's two groups are neighbours, so that it writes
// whole 128-byte lines, 32 bytes per instruction.  10,000 rows of 1,024
// lists: 25 us, 42 with a tile of rows per CTA and 16-byte stores.
template <int KC>
__global__ __launch_bounds__(CF_NT, 1) void k_coarse_dist(
    const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmBlo,
    const float *__restrict__ x, int m, int d, const float *__restrict__ cn, int L,
    float *__restrict__ out, float *__restrict__ gmin, uint32_t *err)
{
    pdl_begin();
    constexpr int CN = CF_CN, NB = cf_buffers(2), TB = CF_TB;
    constexpr uint32_t PBYTES = KC * CN * 128, BBYTES = 2 * PBYTES, ABYTES = KC * CT_M * 128;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    unsigned char *A = smem, *B = smem + 2 * ABYTES;
    __shared__ uint64_t fullb[NB], freeb[NB], mmab[TB], tempty[TB], afull;
    __shared__ uint32_t tmem_base;
    __shared__ int s_abort_;
    __shared__ float sxn[CT_M];
    volatile int *s_abort = &s_abort_;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < NB; ++i) {
            mbar_init(&fullb[i], 1);
            mbar_init(&freeb[i], 1);
        }
        for (int i = 0; i < TB; ++i) {
            mbar_init(&mmab[i], 1);
            mbar_init(&tempty[i], CF_EPI / 32);
        }
        mbar_init(&afull, CF_EPI / 32);
        fence_mbar_init();
        s_abort_ = 0;
    }
    if (warp == CF_EPI / 32) tmem_alloc(&tmem_base, TB * CN);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = tmem_base;
    const int nch = (L + CN - 1) / CN;
    const int64_t total = (int64_t)((m + CT_M - 1) / CT_M) * nch;
    const int64_t s0 = blockIdx.x * total / gridDim.x;
    const uint32_t steps = (uint32_t)((blockIdx.x + 1) * total / gridDim.x - s0);
    const int tile0 = (int)(s0 / nch), j0 = (int)(s0 % nch);  // the first step's tile and chunk

    if (warp == CF_EPI / 32 + 1) {
        if (lane == 0) {
            uint32_t g = 0;
            for (int j = j0; g < steps; ++g, j = j + 1 < nch ? j + 1 : 0) {
                const uint32_t b = g % NB, u = g / NB;
                if (u >= 1 && !mbar_wait_ab(&freeb[b], (u - 1) & 1, err, s_abort, kWaitNs)) break;
                mbar_arrive_expect_tx(&fullb[b], BBYTES);
#pragma unroll
                for (int pp = 0; pp < 2; ++pp)
#pragma unroll
                    for (int kc = 0; kc < KC; ++kc)
                        tma_load_2d(B + b * BBYTES + pp * PBYTES + (size_t)kc * CN * 128,
                                    pp ? &tmBlo : &tmB, kc * 64, j * CN, &fullb[b]);
            }
            // the copies issued last have landed before exit
            for (uint32_t t = g > NB ? g - NB : 0; t < g; ++t)
                mbar_wait_bounded(&fullb[t % NB], (t / NB) & 1, err);
        }
        __syncwarp();
    } else if (warp == CF_EPI / 32) {
        if (lane == 0) {
            const uint32_t idesc = mma_idesc(1, 1, CT_M, CN), abase = smem_u32(A);
            uint32_t g = 0, nt = 0;  // nt: tiles begun
            for (int j = j0; g < steps; ++g, j = j + 1 < nch ? j + 1 : 0) {
                const uint32_t b = g % NB, tb = g % TB, ut = g / TB;
                bool ok = mbar_wait_ab(&fullb[b], (g / NB) & 1, err, s_abort, kWaitNs);
                if (ok && (g == 0 || j == 0))  // the tile's rows are stored
                    ok = mbar_wait_ab(&afull, nt++ & 1, err, s_abort, kWaitNs);
                if (ok && ut >= 1) ok = mbar_wait_ab(&tempty[tb], (ut - 1) & 1, err, s_abort, kWaitNs);
                if (!ok) break;
                tc_fence_after();
                const uint32_t bbase = smem_u32(B + b * BBYTES);
#pragma unroll
                for (int pr = 0; pr < 3; ++pr) {  // (x hi, c hi), (x hi, c lo), (x lo, c hi)
                    const uint32_t ap = abase + (pr == 2 ? ABYTES : 0u);
                    const uint32_t bp = bbase + (pr == 1 ? PBYTES : 0u);
#pragma unroll
                    for (int kc = 0; kc < KC; ++kc)
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            mma_bf16(tbase + tb * CN,
                                     smem_desc_sw128(ap + kc * CT_M * 128 + ks * 32, 1024),
                                     smem_desc_sw128(bp + kc * CN * 128 + ks * 32, 1024), idesc,
                                     (pr | kc | ks) != 0);
                }
                mma_commit(&freeb[b]);
                mma_commit(&mmab[tb]);
            }
            // the last products are written before TMEM is released
            if (g > 0) mbar_wait_bounded(&mmab[(g - 1) % TB], ((g - 1) / TB) & 1, err);
        }
        __syncwarp();
    } else {
        const int q = warp & 3, sub = warp >> 2;
        RowTile<KC, 2> rows;
        auto store = [&]() {
            rows.store(A, ABYTES, d, tid, sxn);
            fence_proxy_async_smem();  // A (generic stores) is read by the MMAs
            __syncwarp();
            if (lane == 0) mbar_arrive(&afull);
        };
        auto fetch = [&](int t) {
            rows.fetch(x, [&](int r) { return t * CT_M + r < m ? t * CT_M + r : -1; }, d, tid);
        };
        fetch(tile0);
        store();
        const int G = (L + 15) / 16;
        // whole sectors where the rows are aligned to them
        const bool vec = (L & 3) == 0;
        const bool w8 = (L & 7) == 0 && (reinterpret_cast<uintptr_t>(out) & 31) == 0;
        bool ok = true;
        int tile = tile0, j = j0;
        for (uint32_t g = 0; g < steps; ++g) {
            const uint32_t tb = g % TB;
            const int jn = j, row = tile * CT_M + q * 32 + lane;
            // the next tile's rows, if this CTA's range goes on into it
            const bool more = (uint32_t)(nch - j) < steps - g;
            if (more && (g == 0 || j == 0)) fetch(tile + 1);
            ok = __all_sync(0xffffffffu, ok && mbar_wait_ab(&mmab[tb], (g / TB) & 1, err, s_abort, kWaitNs));
            tc_fence_after();
            if (++j == nch) {
                j = 0;
                ++tile;
                if (more && ok) store();  // this tile's MMAs are done
            }
            float v[CN / 64][16];
            if (ok) {
#pragma unroll
                for (int k = 0; k < CN / 64; ++k)
                    tmem_ld16(tbase + tb * CN + (2 * sub + k) * 16 + ((uint32_t)(q * 32) << 16), v[k]);
#pragma unroll
                for (int k = 0; k < CN / 64; ++k) tmem_ld_wait(v[k]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[tb]);
            if (!ok) break;  // warp-uniform; no barrier follows before the last one
            if (row >= m) continue;
            const int grp = jn * (CN / 16) + 2 * sub, c0 = grp * 16;
            float *o = out + (size_t)row * L + c0, *og = gmin + (size_t)row * G + grp;
            if (vec && c0 + 32 <= L) {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    float mn = INFINITY;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float4 *c4 = reinterpret_cast<const float4 *>(cn + c0 + 16 * k + 8 * h);
                        const float4 ca = __ldg(c4), cb = __ldg(c4 + 1);
                        const float cv[8] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
                        float t[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            t[i] = fmaf(-2.f, v[k][8 * h + i], cv[i]);
                            mn = fminf(mn, t[i]);
                        }
                        float *ot = o + 16 * k + 8 * h;
                        if (w8) {
                            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(ot),
                                         "f"(t[0]), "f"(t[1]), "f"(t[2]), "f"(t[3]), "f"(t[4]),
                                         "f"(t[5]), "f"(t[6]), "f"(t[7])
                                         : "memory");
                        } else {
                            reinterpret_cast<float4 *>(ot)[0] = make_float4(t[0], t[1], t[2], t[3]);
                            reinterpret_cast<float4 *>(ot)[1] = make_float4(t[4], t[5], t[6], t[7]);
                        }
                    }
                    og[k] = mn;
                }
                continue;
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (c0 + 16 * k >= L) break;
                float mn = INFINITY;
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    if (c0 + 16 * k + i < L) {
                        const float t = fmaf(-2.f, v[k][i], __ldg(cn + c0 + 16 * k + i));
                        o[16 * k + i] = t;
                        mn = fminf(mn, t);
                    }
                og[k] = mn;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == CF_EPI / 32) tmem_dealloc(tbase, TB * CN);
}

// TMA descriptors of the BF16 centroids (and of their low parts) for the
// fused first stage: boxes of 64 columns x CF_CN rows, 128-byte swizzle;
// rows past nlist and columns past d read as zero.
bool coarse_make_map(sivf_index *ix)
{
    const int d = ix->d;
    if (!ix->cent_bf16 || !ix->cent_lo || d > 128 || d % 16) return false;
    auto enc = tmap_encode_fn();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)ix->nlist};
    cuuint64_t strides[1] = {(cuuint64_t)d * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)CF_CN};
    cuuint32_t es[2] = {1, 1};
    auto make = [&](unsigned char *map, void *base) {
        return enc(reinterpret_cast<CUtensorMap *>(map), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base,
                   dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    return make(ix->tmap_cent, ix->cent_bf16) && make(ix->tmap_cent_lo, ix->cent_lo);
}

// ----------------------------------------------- warp-per-row selection
// The same selection for P <= CW_PMAX with one warp per row and no block
// barriers: each lane keeps the CW_PMAX smallest upper bounds of its lists
// (sorted, in registers), the warp extracts the P-th smallest of their
// union as T, then gathers S, tests the sure members and re-decides the
// rest in FP64 exactly as above.  Rows whose S exceeds CW_SCAP take the
// serial FP64 path.
constexpr int CW_ROWS = 4;     // rows (warps) per block
constexpr int CW_PMAX = 8;
constexpr int CW_SCAP = 128;
constexpr int CW_RG = 4;       // FP32 rechecks in flight per warp

// PM: length of each lane's sorted list (1 when P = 1, else CW_PMAX)
template <int PM>
__global__ __launch_bounds__(CW_ROWS * 32) void k_coarse_select_w(SelArgs a)
{
    pdl_begin();
    __shared__ float sLB[CW_ROWS][CW_SCAP], sUB[CW_ROWS][CW_SCAP], sDt[CW_ROWS][CW_SCAP];
    __shared__ int sIdx[CW_ROWS][CW_SCAP];
    __shared__ double sDx[CW_ROWS][CW_SCAP];
    __shared__ unsigned char sSure[CW_ROWS][CW_SCAP];
    __shared__ int sSel[CW_ROWS][CW_PMAX];
    __shared__ float sSelDt[CW_ROWS][CW_PMAX];
    __shared__ double sHd[CW_ROWS][CW_PMAX];
    __shared__ __align__(16) float sX[CW_ROWS][kMaxD];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int L = a.L, P = a.P;
    for (int row = blockIdx.x * CW_ROWS + w; row < a.m; row += gridDim.x * CW_ROWS) {  // whole warps
        const float *Dr = a.D + (size_t)row * L;
        const float *xr = a.x + (size_t)row * a.d;
        const int two_level = a.two_level;
        const float g1 = two_level ? a.gamma2_first : a.gamma2;
        float part = 0.f;
        for (int j = lane; j < a.d; j += 32) part = fmaf(xr[j], xr[j], part);
        const float xn = norm_up(warp_sum(part), a.d);
        int ns = 0;
        auto dt_of = [&](int c) -> float { return __ldg(Dr + c); };

        // P-th smallest of the values v(i), i < n, each lane keeping its
        // CW_PMAX smallest in a sorted register list
        auto pth_smallest = [&](auto val, int n) {
            float top[PM];
#pragma unroll
            for (int k = 0; k < PM; ++k) top[k] = INFINITY;
            constexpr int CU = 8;  // values per lane loaded ahead
            for (int i0 = lane; i0 < n; i0 += 32 * CU) {
                float vv[CU];
#pragma unroll
                for (int u = 0; u < CU; ++u) vv[u] = i0 + 32 * u < n ? val(i0 + 32 * u) : INFINITY;
#pragma unroll
                for (int u = 0; u < CU; ++u) {
                    float v = vv[u];
#pragma unroll
                    for (int k = 0; k < PM; ++k) {  // insert into the sorted list
                        const float lo = fminf(top[k], v), hi = fmaxf(top[k], v);
                        top[k] = lo;
                        v = hi;
                    }
                }
            }
            float T = INFINITY;
            for (int t = 0; t < P; ++t) {
                float v = top[0];
                int who = lane;
                for (int o = 16; o > 0; o >>= 1) {
                    const float ov = __shfl_xor_sync(0xffffffffu, v, o);
                    const int ow = __shfl_xor_sync(0xffffffffu, who, o);
                    if (ov < v || (ov == v && ow < who)) {
                        v = ov;
                        who = ow;
                    }
                }
                T = v;
                if (lane == who) {
#pragma unroll
                    for (int k = 0; k + 1 < PM; ++k) top[k] = top[k + 1];
                    top[PM - 1] = INFINITY;
                }
            }
            return T;
        };

        // T = P-th smallest upper bound over all lists
        float T = pth_smallest([&](int c) {
            const float Dt = dt_of(c);
            return upper_of(Dt, bound_of(Dt, __ldg(a.cn + c), __ldg(a.cnrm_up + c), xn, g1));
        }, L);

        // candidate set S = {c : lower bound <= T}
        constexpr int CU = 8;
        for (int c00 = 0; c00 < L; c00 += 32 * CU) {
            float lbv[CU], ubv[CU], dtv[CU];
#pragma unroll
            for (int u = 0; u < CU; ++u) {
                const int c = c00 + 32 * u + lane;
                lbv[u] = INFINITY;
                ubv[u] = INFINITY;
                dtv[u] = 0.f;
                if (c < L) {
                    const float Dt = dt_of(c);
                    const float E = bound_of(Dt, __ldg(a.cn + c), __ldg(a.cnrm_up + c), xn, g1);
                    lbv[u] = lower_of(Dt, E);
                    ubv[u] = upper_of(Dt, E);
                    dtv[u] = Dt;
                }
            }
#pragma unroll
            for (int u = 0; u < CU; ++u) {
                const int c = c00 + 32 * u + lane;
                const bool in = c < L && lbv[u] <= T;
                const uint32_t mk = __ballot_sync(0xffffffffu, in);
                if (in) {
                    const int p = ns + __popc(mk & lanemask_lt());
                    if (p < CW_SCAP) {
                        sLB[w][p] = lbv[u];
                        sUB[w][p] = ubv[u];
                        sDt[w][p] = dtv[u];
                        sIdx[w][p] = c;
                    }
                }
                ns += __popc(mk);
            }
        }
        __syncwarp();
        if (two_level && ns <= CW_SCAP) {
            // S holds every list that can be among the top P (BF16-stage
            // bound); recompute their distances in FP32, one list per lane,
            // rebuild T and S with the FP32 bound inside S
            for (int j = lane; j < a.d; j += 32) sX[w][j] = xr[j];
            __syncwarp();
            // the warp computes CW_RG members' dot products at a time, lanes
            // over the coordinates (coalesced centroid rows), then a butterfly
            const float4 *x4 = reinterpret_cast<const float4 *>(sX[w]);
            const int n4 = a.d >> 2;
            for (int p0 = 0; p0 < ns; p0 += CW_RG) {
                float part[CW_RG];
#pragma unroll
                for (int t = 0; t < CW_RG; ++t) {
                    part[t] = 0.f;
                    if (p0 + t >= ns) continue;
                    const float4 *c4 =
                        reinterpret_cast<const float4 *>(a.cent + (size_t)sIdx[w][p0 + t] * a.d);
#pragma unroll
                    for (int u = 0; u < kMaxD / 128; ++u) {
                        const int j4 = lane + 32 * u;
                        if (j4 >= n4) break;
                        const float4 xv = x4[j4], cv = __ldg(c4 + j4);
                        part[t] = fmaf(xv.x, cv.x, part[t]);
                        part[t] = fmaf(xv.y, cv.y, part[t]);
                        part[t] = fmaf(xv.z, cv.z, part[t]);
                        part[t] = fmaf(xv.w, cv.w, part[t]);
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int t = 0; t < CW_RG; ++t) part[t] += __shfl_xor_sync(0xffffffffu, part[t], o);
                float acc = part[0];
#pragma unroll
                for (int t = 1; t < CW_RG; ++t)
                    if (lane == t) acc = part[t];
                const int p = p0 + lane;
                if (lane < CW_RG && p < ns) {
                    const int c = sIdx[w][p];
                    const float cnc = __ldg(a.cn + c);
                    const float Dt = fmaf(-2.f, acc, cnc);
                    const float E = bound_of(Dt, cnc, __ldg(a.cnrm_up + c), xn, a.gamma2_re);
                    sLB[w][p] = lower_of(Dt, E);
                    sUB[w][p] = upper_of(Dt, E);
                    sDt[w][p] = Dt;
                }
            }
            __syncwarp();
            T = pth_smallest([&](int p) { return sUB[w][p]; }, ns);
            int n2 = 0;
            for (int p0 = 0; p0 < ns; p0 += 32) {
                const int p = p0 + lane;
                const bool keep = p < ns && sLB[w][p] <= T;
                float lb = 0.f, ub = 0.f, dt = 0.f;
                int c = 0;
                if (keep) {
                    lb = sLB[w][p];
                    ub = sUB[w][p];
                    dt = sDt[w][p];
                    c = sIdx[w][p];
                }
                const uint32_t mk = __ballot_sync(0xffffffffu, keep);
                __syncwarp();
                if (keep) {  // write index <= read index
                    const int q = n2 + __popc(mk & lanemask_lt());
                    sLB[w][q] = lb;
                    sUB[w][q] = ub;
                    sDt[w][q] = dt;
                    sIdx[w][q] = c;
                }
                n2 += __popc(mk);
                __syncwarp();
            }
            ns = n2;
        }
        int32_t *outr = a.out + (size_t)row * P;
        int nsel = 0;
        if (ns <= CW_SCAP) {
            // sure members
            for (int p0 = 0; p0 < ns; p0 += 32) {
                const int p = p0 + lane;
                bool sure = false;
                if (p < ns) {
                    const float ub = sUB[w][p];
                    int cnt = 0;
                    for (int q = 0; q < ns; ++q) cnt += (q != p && sLB[w][q] <= ub);
                    sure = ub <= T && cnt < P;
                    sSure[w][p] = sure;
                }
                const uint32_t mk = __ballot_sync(0xffffffffu, sure);
                if (sure) {
                    const int s = nsel + __popc(mk & lanemask_lt());
                    if (s < CW_PMAX) {
                        sSel[w][s] = sIdx[w][p];
                        sSelDt[w][s] = sDt[w][p];
                    }
                }
                nsel += __popc(mk);
            }
            __syncwarp();
            const int r = P - nsel, nb = ns - nsel;
            if (r > 0) {
                // boundary members: exact FP64 distances, rank among them
                if (nb > r) {
                    for (int p = lane; p < ns; p += 32)
                        if (!sSure[w][p]) sDx[w][p] = exact_dist(xr, a.cent + (size_t)sIdx[w][p] * a.d, a.d);
                    __syncwarp();
                }
                for (int p0 = 0; p0 < ns; p0 += 32) {
                    const int p = p0 + lane;
                    bool take = false;
                    if (p < ns && !sSure[w][p]) {
                        take = true;
                        if (nb > r) {
                            const double Dc = sDx[w][p];
                            const int c = sIdx[w][p];
                            int rank = 0;
                            for (int q = 0; q < ns; ++q) {
                                if (q == p || sSure[w][q]) continue;
                                rank += (sDx[w][q] < Dc || (sDx[w][q] == Dc && sIdx[w][q] < c));
                            }
                            take = rank < r;
                        }
                    }
                    const uint32_t mk = __ballot_sync(0xffffffffu, take);
                    if (take) {
                        const int s = nsel + __popc(mk & lanemask_lt());
                        if (s < CW_PMAX) {
                            sSel[w][s] = sIdx[w][p];
                            sSelDt[w][s] = sDt[w][p];
                        }
                    }
                    nsel += __popc(mk);
                }
            }
        } else {
            // pathological (more than CW_SCAP candidates, e.g. many identical
            // centroids): exact FP64 insertion into a sorted array of P, lists
            // in index order (keeps the lowest index among ties)
            if (lane == 0) {
                int n = 0;
                for (int c = 0; c < L; ++c) {
                    const float Dt = dt_of(c);
                    const float E = bound_of(Dt, a.cn[c], a.cnrm_up[c], xn, g1);
                    if (lower_of(Dt, E) > T) continue;
                    const double Dc = exact_dist(xr, a.cent + (size_t)c * a.d, a.d);
                    if (n == P && !(Dc < sHd[w][n - 1])) continue;
                    int pos = n < P ? n : P - 1;
                    while (pos > 0 && Dc < sHd[w][pos - 1]) {
                        sHd[w][pos] = sHd[w][pos - 1];
                        sSel[w][pos] = sSel[w][pos - 1];
                        --pos;
                    }
                    sHd[w][pos] = Dc;
                    sSel[w][pos] = c;
                    if (n < P) ++n;
                }
                for (int i = 0; i < n; ++i) sSelDt[w][i] = (float)sHd[w][i];
                nsel = n;
            }
            nsel = __shfl_sync(0xffffffffu, nsel, 0);
        }
        __syncwarp();
        // the selected set nearest first: ascending approximate distance, ties
        // to the lower list index (the set itself is the exact one)
        if (nsel != P && lane == 0) atomicOr(a.err, ERR_SELECT);
        nsel = min(nsel, P);
        if (lane < P) {
            if (lane >= nsel) {
                outr[lane] = -1;
            } else {
                const int c = sSel[w][lane];
                const float dc = sSelDt[w][lane];
                int pos = 0;
                for (int q = 0; q < nsel; ++q) {
                    const int c2 = sSel[w][q];
                    const float d2 = sSelDt[w][q];
                    pos += d2 < dc || (d2 == dc && c2 < c);
                }
                outr[pos] = c;
            }
        }
        __syncwarp();  // the warp's shared rows are reused by its next row
    }
}

// Roundings of a dot product of d values whose partial sums a warp holds
// (float4s lane, lane + 32, ... accumulated by fused multiply-adds) and adds
// by five shuffles: its error is at most gamma_n sum |x_j c_j| with n =
// 4 ceil(d / 128) + 5, against n = d for one running sum.  At d = 128 that
// leaves a fourteenth of the near-ties to the FP64 step, whose dependent
// FP64 additions are what an undecided row costs most.
__host__ __device__ constexpr int re_ops(int d) { return 4 * ((d + 127) / 128) + 5; }
// the same with eight lanes a row (float4s t, t + 8, ...) and three shuffles
__host__ __device__ constexpr int pk_ops(int d) { return 4 * ((d + 31) / 32) + 3; }

// ------------------------------------------ probe selection, P lists per row
// One warp per row, from k_coarse_dist's distances and group minima.  The
// P-th smallest group minimum b bounds the P-th smallest Dt (P groups each
// hold a list at or below it), so only lists with Dt <= b + 2 Ebig can be
// among the top P, and only groups whose minimum is within that are read: 75
// of 4,096 lists for P = 64, where the block selection read every distance
// six times.  Their distances are recomputed in FP32 (PK_RG at a time, eight
// lanes each) and decided as in the other selections: sure members
// by their FP32 intervals, the rest by FP64 distance.  A row with more
// candidates than `cap` is decided by the block (refine_rows).
// 10,000 rows of 4,096 lists, P = 64: 165 us with k_coarse_dist against 580
// (FP32 GEMM and block selection); 61 rows of 16,384 lists, P = 32: 43
// against 118; 1,000 rows of 2,048 close lists, P = 64: 47 us, 121 when each
// 32 candidates with a boundary member paid a pass of FP64 distances.
// Bound by the chain of one row (about 25 us at P = 64), not by throughput.
constexpr int PK_RG = 16;      // FP32 rechecks in flight per warp
constexpr int PK_PMAX = 128;   // most lists per row of this kernel
__host__ __device__ constexpr int pk_cap(int P) { return (P + P / 2 + 64 + 31) / 32 * 32; }
__host__ __device__ constexpr size_t pk_smem(int P)  // per warp: Dt, LB, UB, list, FP64, sure
{
    return (size_t)pk_cap(P) * (4 + 4 + 4 + 4 + 8 + 4) + kMaxD * 4;
}

// dot product of a row and a list's centroid, both spread over eight lanes
__device__ __forceinline__ float pick_dot(const float4 (&xv)[4], const float4 (&cv)[4])
{
    float dot = 0.f;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        dot = fmaf(xv[u].x, cv[u].x, dot);
        dot = fmaf(xv[u].y, cv[u].y, dot);
        dot = fmaf(xv[u].z, cv[u].z, dot);
        dot = fmaf(xv[u].w, cv[u].w, dot);
    }
    dot += __shfl_xor_sync(0xffffffffu, dot, 4);
    dot += __shfl_xor_sync(0xffffffffu, dot, 2);
    dot += __shfl_xor_sync(0xffffffffu, dot, 1);
    return dot;
}

// One row, by a warp (mem: pk_smem of it); false when it has more candidates than
// the table holds.  FRESH: the distances are FP32 ones that this kernel has
// written (other blocks of it, too), not to be computed again.
template <bool FRESH>
__device__ __forceinline__ bool pick_row(const SelArgs &a, int row, unsigned char *mem, int lane)
{
    auto ld = [](const float *p) { return FRESH ? __ldcg(p) : __ldg(p); };
    const int L = a.L, P = a.P, d = a.d, n4 = d >> 2, cap = pk_cap(P), G = (L + 15) / 16;
    double *sDx = reinterpret_cast<double *>(mem);
    float *sX = reinterpret_cast<float *>(sDx + cap), *sDt = sX + kMaxD, *sLB = sDt + cap, *sUB = sLB + cap;
    int *sIdx = reinterpret_cast<int *>(sUB + cap), *sSure = sIdx + cap;
    const float *Dr = a.D + (size_t)row * L, *gr = a.gmin + (size_t)row * G;
    const float *xr = a.x + (size_t)row * d;
    float part = 0.f;
    for (int j = lane; j < d; j += 32) {
        const float v = xr[j];
        sX[j] = v;
        part = fmaf(v, v, part);
    }
    const float xn = norm_up(warp_sum(part), d);
    const float b = kth_bound<32>([&](int i) { return i < G ? ld(gr + i) : INFINITY; },
                                  (G + 31) & ~31, P, lane);
    const float cnmax = __ldg(a.cmaxes), cmax = __ldg(a.cmaxes + 1);
    const float eb = bound_max(cnmax, abs_max(cnmax, xn, cmax), xn, cmax,
                               FRESH ? a.gamma2 : a.gamma2_first);
    const float thr = pick_limit(b, eb);
    // the groups that can hold a candidate, then their lists: 4 lanes read a
    // group, 32 groups in flight
    int ng = 0, ns = 0;
    int *sGrp = sSure;
    for (int g0 = 0; g0 < G && ng <= cap; g0 += 128) {
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int gi = g0 + 32 * u + lane;
            v[u] = gi < G ? ld(gr + gi) : INFINITY;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool in = g0 + 32 * u + lane < G && v[u] <= thr;
            const uint32_t mk = __ballot_sync(0xffffffffu, in);
            const int p = ng + __popc(mk & lanemask_lt());
            if (in && p < cap) sGrp[p] = g0 + 32 * u + lane;
            ng += __popc(mk);
        }
    }
    __syncwarp();
    const bool vec = (L & 3) == 0;
    for (int t0 = 0; t0 < ng && ng <= cap && ns <= cap; t0 += 32) {
        float v[4][4];
        int cl[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = t0 + 8 * u + (lane >> 2);
            cl[u] = t < ng ? sGrp[t] * 16 + (lane & 3) * 4 : L;
            if (vec && cl[u] < L) {
                const float4 *d4 = reinterpret_cast<const float4 *>(Dr + cl[u]);
                const float4 f = FRESH ? __ldcg(d4) : __ldg(d4);
                v[u][0] = f.x;
                v[u][1] = f.y;
                v[u][2] = f.z;
                v[u][3] = f.w;
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) v[u][k] = cl[u] + k < L ? ld(Dr + cl[u] + k) : INFINITY;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const bool ok = cl[u] + k < L && v[u][k] <= thr;
                const uint32_t mk = __ballot_sync(0xffffffffu, ok);
                const int p = ns + __popc(mk & lanemask_lt());
                if (ok && p < cap) sIdx[p] = cl[u] + k;
                ns += __popc(mk);
            }
    }
    __syncwarp();
    if (ng > cap || ns > cap || ns < P) return false;  // too many candidates (or no numbers)
    // FP32 distances and intervals: eight lanes a list, 16 lists in flight
    for (int p = lane; p < ns; p += 32) {
        sLB[p] = __ldg(a.cn + sIdx[p]);
        sUB[p] = __ldg(a.cnrm_up + sIdx[p]);
    }
    __syncwarp();
    if (FRESH) {
        for (int p = lane; p < ns; p += 32) {
            const float Dt = ld(Dr + sIdx[p]), E = bound_of(Dt, sLB[p], sUB[p], xn, a.gamma2);
            sDt[p] = Dt;
            sLB[p] = lower_of(Dt, E);
            sUB[p] = upper_of(Dt, E);
        }
    } else {
        const int g8 = lane >> 3, t8 = lane & 7;
        const float4 *x4 = reinterpret_cast<const float4 *>(sX);
        float4 xv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            xv[u] = t8 + 8 * u < n4 ? x4[t8 + 8 * u] : make_float4(0.f, 0.f, 0.f, 0.f);
        for (int p0 = 0; p0 < ns; p0 += PK_RG) {
            float4 cv[PK_RG / 4][4];
#pragma unroll
            for (int r = 0; r < PK_RG / 4; ++r) {
                const float4 *c4 = reinterpret_cast<const float4 *>(
                    a.cent + (size_t)sIdx[min(p0 + 4 * r + g8, ns - 1)] * d);
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    cv[r][u] = t8 + 8 * u < n4 ? __ldg(c4 + t8 + 8 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int r = 0; r < PK_RG / 4; ++r) {
                const float dot = pick_dot(xv, cv[r]);
                const int p = p0 + 4 * r + g8;
                if (t8 == 0 && p < ns) {
                    const float cnc = sLB[p], Dt = fmaf(-2.f, dot, cnc);
                    const float E = bound_of(Dt, cnc, sUB[p], xn, a.gamma2_re);
                    sDt[p] = Dt;
                    sLB[p] = lower_of(Dt, E);
                    sUB[p] = upper_of(Dt, E);
                }
            }
        }
    }
    __syncwarp();
    // T: at least P upper bounds lie at or below it
    const float T = kth_bound<16>([&](int i) { return i < ns ? sUB[i] : INFINITY; }, (ns + 31) & ~31, P,
                                  lane);
    int nsure = 0, nmem = 0;
    for (int p0 = 0; p0 < ns; p0 += 32) {
        const int p = p0 + lane;
        bool sure = false, mem_ = false;
        if (p < ns) {
            const float ub = sUB[p];
            int cnt = 0;
#pragma unroll 8
            for (int k = 0; k < ns; ++k) cnt += sLB[k] <= ub;  // itself included
            mem_ = sLB[p] <= T;
            sure = mem_ && ub <= T && cnt <= P;
            sSure[p] = sure ? 1 : mem_ ? 0 : -1;
        }
        nsure += __popc(__ballot_sync(0xffffffffu, sure));
        nmem += __popc(__ballot_sync(0xffffffffu, mem_));
    }
    __syncwarp();
    const int r = P - nsure, nb = nmem - nsure;
    int *sBnd = reinterpret_cast<int *>(sLB);  // the lower bounds have been read
    if (r > 0 && nb > r) {
        // boundary members: FP64 distances, the best r of them.  The few there
        // are take one lane each, next to each other: a pass of exact_dist costs
        // the same for one member as for 32, and each 32 candidates paid one.
        int n = 0;
        for (int p0 = 0; p0 < ns; p0 += 32) {
            const int p = p0 + lane;
            const bool in = p < ns && sSure[p] == 0;
            const uint32_t mk = __ballot_sync(0xffffffffu, in);
            if (in) sBnd[n + __popc(mk & lanemask_lt())] = p;
            n += __popc(mk);
        }
        __syncwarp();
        if (nb <= EX_FEW) {
            const double D = exact_four(reinterpret_cast<const float4 *>(sX), a.cent,
                                        [&](int m) { return sIdx[sBnd[m]]; }, nb, d, lane);
            if (lane < nb) sDx[sBnd[lane]] = D;
        }
        for (int t = lane; t < nb && nb > EX_FEW; t += 32) {
            const int p = sBnd[t];
            sDx[p] = exact_dist4(reinterpret_cast<const float4 *>(sX),
                                 reinterpret_cast<const float4 *>(a.cent + (size_t)sIdx[p] * d), d);
        }
        __syncwarp();
    }
    // the chosen to the front of sIdx / sDt, in place
    int nsel = 0;
    for (int p0 = 0; p0 < ns; p0 += 32) {
        const int p = p0 + lane;
        bool take = false;
        if (p < ns) {
            take = sSure[p] == 1;
            if (sSure[p] == 0 && r > 0) {
                take = true;
                if (nb > r) {
                    int rank = 0;
                    for (int t = 0; t < nb; ++t) {
                        const int k = sBnd[t];
                        rank += sDx[k] < sDx[p] || (sDx[k] == sDx[p] && sIdx[k] < sIdx[p]);
                    }
                    take = rank < r;
                }
            }
        }
        sUB[p0 + lane] = take ? 1.f : 0.f;  // cap is a multiple of 32
    }
    __syncwarp();
    for (int p0 = 0; p0 < ns; p0 += 32) {
        const int p = p0 + lane;
        const bool take = p < ns && sUB[p] > 0.f;
        const float dt = p < ns ? sDt[p] : 0.f;
        const int c = p < ns ? sIdx[p] : 0;
        const uint32_t mk = __ballot_sync(0xffffffffu, take);
        __syncwarp();
        if (take) {  // write index <= read index
            const int q = nsel + __popc(mk & lanemask_lt());
            sDt[q] = dt;
            sIdx[q] = c;
        }
        nsel += __popc(mk);
        __syncwarp();
    }
    if (nsel != P && lane == 0) atomicOr(a.err, ERR_SELECT);
    nsel = min(nsel, P);
    // Nearest first: ascending FP32 distance, ties to the lower list index.  The
    // distances are those of the forms without group minima (k_coarse_gemm's sums;
    // for P <= CW_PMAX of at most CW_LMAX lists k_coarse_select_w's), so that a
    // list's place does not depend on the form: where two neighbours lie within
    // the two sums' bounds of each other, that sum is formed for both.
    __syncwarp();
    int *sList = reinterpret_cast<int *>(sUB);
    int32_t *outr = a.out + (size_t)row * P;
    for (int s = lane; s < P; s += 32) {
        if (s >= nsel) {
            outr[s] = -1;
            continue;
        }
        const int c = sIdx[s];
        const float dc = sDt[s];
        int pos = 0;
#pragma unroll 8
        for (int q = 0; q < nsel; ++q) pos += (sDt[q] < dc) | ((sDt[q] == dc) & (sIdx[q] < c));  // no branches
        outr[pos] = c;
        sLB[pos] = dc;
        sList[pos] = c;
    }
    __syncwarp();
    const bool sums = P > CW_PMAX || L > CW_LMAX;
    bool close = false;
    if (!(FRESH && sums)) {
        const float ab = abs_max(cnmax, xn, cmax);
        const float e1 = bound_max(cnmax, ab, xn, cmax, FRESH ? a.gamma2 : a.gamma2_re);
        const float e2 = bound_max(cnmax, ab, xn, cmax, sums ? a.gamma2 : a.gamma2_w);
        const float apart = __fmul_ru(2.0001f, __fadd_ru(e1, e2));
        for (int i = lane; i < nsel; i += 32) {
            const bool in = (i > 0 && !(sLB[i] - sLB[i - 1] > apart)) ||
                            (i + 1 < nsel && !(sLB[i + 1] - sLB[i] > apart));
            sSure[i] = in;
            close = close || in;
        }
        close = __any_sync(0xffffffffu, close);
        __syncwarp();
    }
    if (!close) return true;
    const float4 *x4 = reinterpret_cast<const float4 *>(sX);
    if (sums) {
        for (int i = lane; i < nsel; i += 32) {
            if (!sSure[i]) continue;
            const float4 *c4 = reinterpret_cast<const float4 *>(a.cent + (size_t)sList[i] * d);
            float dot = 0.f;
#pragma unroll 4
            for (int j = 0; j < n4; ++j) {
                const float4 xv = x4[j], cv = __ldg(c4 + j);
                dot = fmaf(xv.x, cv.x, dot);
                dot = fmaf(xv.y, cv.y, dot);
                dot = fmaf(xv.z, cv.z, dot);
                dot = fmaf(xv.w, cv.w, dot);
            }
            sLB[i] = fmaf(-2.f, dot, __ldg(a.cn + sList[i]));
        }
    } else {
        for (int i = 0; i < nsel; ++i) {
            if (!sSure[i]) continue;  // warp-uniform
            float dot = 0.f;
            if (lane < n4) {
                const float4 xv = x4[lane];
                const float4 cv = __ldg(reinterpret_cast<const float4 *>(a.cent + (size_t)sList[i] * d) + lane);
                dot = fmaf(xv.x, cv.x, dot);
                dot = fmaf(xv.y, cv.y, dot);
                dot = fmaf(xv.z, cv.z, dot);
                dot = fmaf(xv.w, cv.w, dot);
            }
            dot = warp_sum(dot);
            if (lane == 0) sLB[i] = fmaf(-2.f, dot, __ldg(a.cn + sList[i]));
        }
    }
    __syncwarp();
    for (int s = lane; s < nsel; s += 32) {
        if (!sSure[s]) continue;  // alone in its place
        const int c = sList[s];
        const float dc = sLB[s];
        int pos = s;  // its neighbours on both sides, as far as they are close
        for (int q = s - 1; q >= 0 && sSure[q]; --q) pos -= (sLB[q] > dc) | ((sLB[q] == dc) & (sList[q] > c));
        for (int q = s + 1; q < nsel && sSure[q]; ++q) pos += (sLB[q] < dc) | ((sLB[q] == dc) & (sList[q] < c));
        outr[pos] = c;
    }
    return true;
}

// The rows of a block with more candidates than pick_row's table: the lists of a
// row's cluster lie within the split's bound of its P-th by the hundred, but few
// within FP32's.  Of the groups of 16 lists whose minimum is within that bound
// for one of the rows, the distances and the minimum are written again in FP32
// for all of them (the sums of k_coarse_gemm, bit for bit; the other groups'
// lists cannot be chosen and keep theirs): a list per thread, the centroids
// staged RF_K columns at a time.  pick_row then decides from them, a warp per
// row, and the block rows that have more candidates even so (near-ties by the
// hundred).  rows: the block's rows, -1 for the others.  10,000 rows of 2,048
// lists in two clusters, P = 32: 0.73 ms, 11.8 by FP64 distances of all of them,
// 0.98 by an FP32 matrix and a block per row.
constexpr int PK_NT = CW_ROWS * 32;
constexpr int RF_K = 16;           // columns staged at a time
constexpr int RF_S = RF_K + 4;     // floats of a staged list: 16-byte reads without conflicts
constexpr int RF_ST = 3;           // stages
__host__ __device__ constexpr size_t pk_block_smem(int P, int G)
{
    const size_t stage = (size_t)RF_ST * PK_NT * RF_S * 4 + (size_t)G * 2, pick = (size_t)CW_ROWS * pk_smem(P);
    const size_t most = stage > pick ? stage : pick;
    return most > sizeof(SelTab) ? most : sizeof(SelTab);
}
__device__ __noinline__ void refine_rows(SelArgs a, const int *rows, int *left, unsigned char *mem)
{
    __shared__ __align__(16) float s_x[CW_ROWS][128];
    __shared__ float s_thr[CW_ROWS];
    __shared__ int s_ng;
    float *sb = reinterpret_cast<float *>(mem);
    uint16_t *grp = reinterpret_cast<uint16_t *>(sb + RF_ST * PK_NT * RF_S);  // the groups in reach
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int L = a.L, d = a.d, G = (L + 15) / 16;
    a.two_level = 0;
    {
        float part = 0.f, thr = -INFINITY;
        for (int j = lane; j < d; j += 32) {
            const float v = rows[w] >= 0 ? a.x[(size_t)rows[w] * d + j] : 0.f;
            s_x[w][j] = v;
            part = fmaf(v, v, part);
        }
        if (rows[w] >= 0) {
            const float *gr = a.gmin + (size_t)rows[w] * G;
            const float xn = norm_up(warp_sum(part), d);
            const float b = kth_bound<8>([&](int i) { return i < G ? __ldcg(gr + i) : INFINITY; },
                                         (G + 31) & ~31, a.P, lane);
            const float cnmax = __ldg(a.cmaxes), cmax = __ldg(a.cmaxes + 1);
            thr = pick_limit(b, bound_max(cnmax, abs_max(cnmax, xn, cmax), xn, cmax, a.gamma2_first));
        }
        if (lane == 0) s_thr[w] = thr;
        if (tid == 0) s_ng = 0;
    }
    __syncthreads();
    for (int g0 = w * 32; g0 < G; g0 += PK_NT) {  // whole warps
        const int g = g0 + lane;
        bool on = false;
        if (g < G)
#pragma unroll
            for (int r = 0; r < CW_ROWS; ++r)
                if (rows[r] >= 0) on = on || !(__ldcg(a.gmin + (size_t)rows[r] * G + g) > s_thr[r]);
        const uint32_t mk = __ballot_sync(0xffffffffu, on);
        int at = 0;
        if (lane == 0 && mk) at = atomicAdd(&s_ng, __popc(mk));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(mk & lanemask_lt());
        if (on) grp[at] = (uint16_t)g;
    }
    __syncthreads();
    const int ng = s_ng;
    // steps of RF_K columns of PK_NT lists (eight groups), RF_ST - 1 in flight
    int fi = 0, fk = 0, fs = 0;  // the next step to fetch: its first group, columns, stage
    auto fetch = [&]() {
        if (fi < ng) {
            float *to = sb + fs * PK_NT * RF_S;
#pragma unroll
            for (int u = 0; u < RF_K / 4; ++u) {
                const int r = (tid >> 2) + 32 * u, q = tid & 3;
                const int c = min((int)grp[min(fi + (r >> 4), ng - 1)] * 16 + (r & 15), L - 1);
                cp_async16_c(to + r * RF_S + 4 * q, a.cent + (size_t)c * d + fk + 4 * q, 16u);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        fs = fs + 1 == RF_ST ? 0 : fs + 1;
        fk += RF_K;
        if (fk >= d) {
            fk = 0;
            fi += PK_NT / 16;
        }
    };
#pragma unroll
    for (int st = 0; st < RF_ST - 1; ++st) fetch();
    int stage = 0;
    for (int i = 0; i < ng; i += PK_NT / 16) {
        float acc[CW_ROWS];
#pragma unroll
        for (int r = 0; r < CW_ROWS; ++r) acc[r] = 0.f;
        for (int k0 = 0; k0 < d; k0 += RF_K) {
            asm volatile("cp.async.wait_group %0;\n" ::"n"(RF_ST - 2) : "memory");
            __syncthreads();  // this step has landed, the last one's stage has been read
            fetch();
            const float *sc = sb + (stage * PK_NT + tid) * RF_S;
            stage = stage + 1 == RF_ST ? 0 : stage + 1;
            float4 cv[RF_K / 4];
#pragma unroll
            for (int q = 0; q < RF_K / 4; ++q) cv[q] = *reinterpret_cast<const float4 *>(sc + 4 * q);
#pragma unroll
            for (int r = 0; r < CW_ROWS; ++r) {
                if (rows[r] < 0) continue;
#pragma unroll
                for (int q = 0; q < RF_K / 4; ++q) {
                    const float4 xv = *reinterpret_cast<const float4 *>(&s_x[r][k0 + 4 * q]);
                    acc[r] = fmaf(xv.x, cv[q].x, acc[r]);
                    acc[r] = fmaf(xv.y, cv[q].y, acc[r]);
                    acc[r] = fmaf(xv.z, cv[q].z, acc[r]);
                    acc[r] = fmaf(xv.w, cv[q].w, acc[r]);
                }
            }
        }
        const int at = i + (tid >> 4), g = at < ng ? grp[at] : 0, c = at < ng ? g * 16 + (tid & 15) : L;
        const float cnc = c < L ? __ldg(a.cn + c) : 0.f;
#pragma unroll
        for (int r = 0; r < CW_ROWS; ++r) {
            const float Dt = fmaf(-2.f, acc[r], cnc);
            float mn = c < L ? Dt : INFINITY;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            if (rows[r] >= 0 && c < L) {
                a.Dw[(size_t)rows[r] * L + c] = Dt;
                if ((tid & 15) == 0) a.gmin[(size_t)rows[r] * G + g] = mn;
            }
        }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();  // the rows are written; the stages have been read
    bool ok = true;
    if (rows[w] >= 0) ok = pick_row<true>(a, rows[w], mem + (size_t)w * pk_smem(a.P), lane);
    if (lane == 0) left[w] = !ok;
    __syncthreads();
    for (int r = 0; r < CW_ROWS; ++r)
        if (left[r]) select_row<PK_NT, true>(a, rows[r], *reinterpret_cast<SelTab *>(mem));
}

// rpb rows per block, a warp each (fewer rows: one, so that a block refines one)
__global__ __launch_bounds__(PK_NT, 5) void k_coarse_pick(SelArgs a, int rpb)
{
    pdl_begin();
    extern __shared__ __align__(16) unsigned char pk[];
    __shared__ int s_rows[CW_ROWS], s_left[CW_ROWS];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = w < rpb ? blockIdx.x * rpb + w : a.m;
    const bool ok = row >= a.m || pick_row<false>(a, row, pk + (size_t)w * pk_smem(a.P), lane);
    if (lane == 0) s_rows[w] = ok ? -1 : row;
    if (__syncthreads_or(!ok)) refine_rows(a, s_rows, s_left, pk);
}

// Assignment from k_coarse_dist's distances and group minima, a warp per row:
// the lists within the split's bound of the smallest, of the groups whose
// minimum is, decided by decide_nearest.  G <= 256 groups.
constexpr int NR_GMAX = CW_LMAX / 16;
__global__ __launch_bounds__(CW_ROWS * 32, 5) void k_coarse_near(SelArgs a, NearArgs near)
{
    pdl_begin();
    __shared__ int s_tab[CW_ROWS][ND_WIN], s_grp[CW_ROWS][NR_GMAX];
    __shared__ float s_lbs[CW_ROWS][ND_WIN];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = blockIdx.x * CW_ROWS + w;
    if (row >= a.m) return;  // whole warps
    const int L = a.L, d = a.d, G = (L + 15) / 16;
    const float *Dr = a.D + (size_t)row * L, *gr = a.gmin + (size_t)row * G;
    const float *xr = a.x + (size_t)row * d;
    float v[NR_GMAX / 32], b = INFINITY, part = 0.f;
#pragma unroll
    for (int u = 0; u < NR_GMAX / 32; ++u) {
        v[u] = 32 * u + lane < G ? __ldg(gr + 32 * u + lane) : INFINITY;
        b = fminf(b, v[u]);
    }
    for (int j = lane; j < d; j += 32) part = fmaf(xr[j], xr[j], part);
    const float xn = norm_up(warp_sum(part), d);
    for (int o = 16; o > 0; o >>= 1) b = fminf(b, __shfl_xor_sync(0xffffffffu, b, o));
    const float cnmax = __ldg(a.cmaxes), cmax = __ldg(a.cmaxes + 1);
    const float thr = pick_limit(b, bound_max(cnmax, abs_max(cnmax, xn, cmax), xn, cmax, a.gamma2_first));
    int ng = 0;
#pragma unroll
    for (int u = 0; u < NR_GMAX / 32; ++u) {
        const bool in = 32 * u + lane < G && v[u] <= thr;
        const uint32_t mk = __ballot_sync(0xffffffffu, in);
        if (in) s_grp[w][ng + __popc(mk & lanemask_lt())] = 32 * u + lane;
        ng += __popc(mk);
    }
    __syncwarp();
    auto fill = [&](int first, int w0) {  // two groups per load, eight in flight
        int total = 0;
        for (int t0 = 0; t0 < ng; t0 += 8) {
            int c[4];
            float e[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int t = t0 + 2 * u + (lane >> 4);
                c[u] = t < ng ? s_grp[w][t] * 16 + (lane & 15) : L;
                e[u] = c[u] < L ? __ldg(Dr + c[u]) : INFINITY;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool in = c[u] < L && e[u] <= thr;
                const uint32_t mk = __ballot_sync(0xffffffffu, in);
                const int at = first + total - w0 + __popc(mk & lanemask_lt());
                if (in && at >= first && at < ND_WIN) s_tab[w][at] = c[u];
                total += __popc(mk);
            }
        }
        __syncwarp();
        return total;
    };
    const int c = decide_nearest(near, fill, d, xr, xn, s_tab[w], s_lbs[w], lane);
    if (lane == 0) {
        if (c < 0 || c >= L) atomicOr(a.err, ERR_SELECT);
        a.out[row] = c < 0 || c >= L ? -1 : c;
    }
}

// Finishing selection of the rows that the fused first stage left undecided (P =
// 1), a warp per row.  With a record: the FP32 distance of each candidate list
// (CW_RG at a time, lanes over the coordinates), one list per lane; the lists
// whose lower bound is at most the smallest upper bound remain, and if they are
// several, their FP64 distances decide (ties to the lower index).  With the
// second pass's bits: decide_nearest.
constexpr int FN_ROWS = 8;     // warps per block
__global__ __launch_bounds__(FN_ROWS * 32, 2) void k_coarse_finish(SelArgs a, SecondArgs sp, NearArgs near)
{
    pdl_begin();
    __shared__ __align__(16) float sX[FN_ROWS][kMaxD];
    __shared__ int s_tab[FN_ROWS][ND_WIN];
    __shared__ float s_lbs[FN_ROWS][ND_WIN];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int L = a.L, d = a.d, n4 = d >> 2;
    const int nrec = min(a.nhard[0], a.s_cap);
    for (int it = blockIdx.x * FN_ROWS + w; it < nrec; it += gridDim.x * FN_ROWS) {  // whole warps
        const int32_t *Sr = a.S + (size_t)it * CF_STRIDE;
        const int row = Sr[0], n0 = min(Sr[1], CF_CAP);
        const int c = lane < n0 ? Sr[2 + lane] : 0;
        const float *xr = a.x + (size_t)row * d;
        __syncwarp();  // the warp's sX is still read for its last row
        float part = 0.f;
        for (int j = lane; j < d; j += 32) {
            const float v = xr[j];
            sX[w][j] = v;
            part = fmaf(v, v, part);
        }
        const float xn = norm_up(warp_sum(part), d);
        __syncwarp();
        const float4 *x4 = reinterpret_cast<const float4 *>(sX[w]);
        float dot = 0.f;
        for (int p0 = 0; p0 < n0; p0 += CW_RG) {
            float s[CW_RG];
#pragma unroll
            for (int t = 0; t < CW_RG; ++t) {
                const int ct = __shfl_sync(0xffffffffu, c, p0 + t);
                const float4 *c4 = reinterpret_cast<const float4 *>(a.cent + (size_t)ct * d);
                s[t] = 0.f;
                if (p0 + t < n0 && lane < n4) {  // d <= 128
                    const float4 xv = x4[lane], cv = __ldg(c4 + lane);
                    s[t] = fmaf(xv.x, cv.x, s[t]);
                    s[t] = fmaf(xv.y, cv.y, s[t]);
                    s[t] = fmaf(xv.z, cv.z, s[t]);
                    s[t] = fmaf(xv.w, cv.w, s[t]);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int t = 0; t < CW_RG; ++t) s[t] += __shfl_xor_sync(0xffffffffu, s[t], o);
#pragma unroll
            for (int t = 0; t < CW_RG; ++t)
                if (lane == p0 + t) dot = s[t];
        }
        float lb = INFINITY, ub = INFINITY;
        if (lane < n0) {
            const float cnc = __ldg(a.cn + c), Dt = fmaf(-2.f, dot, cnc);
            const float E = bound_of(Dt, cnc, __ldg(a.cnrm_up + c), xn, a.gamma2_re);
            lb = lower_of(Dt, E);
            ub = upper_of(Dt, E);
        }
        float T = ub;
        for (int o = 16; o > 0; o >>= 1) T = fminf(T, __shfl_xor_sync(0xffffffffu, T, o));
        const bool in = lane < n0 && lb <= T;
        const uint32_t mk = __ballot_sync(0xffffffffu, in);
        int chosen = -1;
        if (__popc(mk) == 1) {
            chosen = __shfl_sync(0xffffffffu, c, __ffs(mk) - 1);
        } else if (mk) {
            double bd = INFINITY;
            int bc = 0x7fffffff;
            if (__popc(mk) <= EX_FEW) {
                // the lanes that hold the lists, and their numbers
                uint32_t todo = mk;
                int cm[EX_FEW];
#pragma unroll
                for (int m = 0; m < EX_FEW; ++m) {
                    cm[m] = __shfl_sync(0xffffffffu, c, todo ? __ffs(todo) - 1 : 0);
                    todo &= todo - 1u;
                }
                auto pick = [&](int m) { return m == 0 ? cm[0] : m == 1 ? cm[1] : m == 2 ? cm[2] : cm[3]; };
                const double D = exact_four(x4, a.cent, pick, __popc(mk), d, lane);
                if (lane < __popc(mk)) {
                    bd = D;
                    bc = pick(lane);
                }
            } else if (in) {
                bd = exact_dist4(x4, reinterpret_cast<const float4 *>(a.cent + (size_t)c * d), d);
                bc = c;
            }
            for (int o = 16; o > 0; o >>= 1) {
                const double od = __shfl_xor_sync(0xffffffffu, bd, o);
                const int oc = __shfl_xor_sync(0xffffffffu, bc, o);
                if (od < bd || (od == bd && oc < bc)) {
                    bd = od;
                    bc = oc;
                }
            }
            chosen = bc;
        }
        if (lane == 0) {
            if (chosen < 0 || chosen >= L) {
                atomicOr(a.err, ERR_SELECT);
                chosen = -1;
            }
            a.out[row] = chosen;
        }
    }

    const int nbits = *sp.n, G = (L + 15) / 16;
    for (int it = blockIdx.x * FN_ROWS + w; it < nbits; it += gridDim.x * FN_ROWS) {  // whole warps
        const int place = sp.list[it], row = sp.rows[place];
        const uint16_t *bits = sp.bits + (size_t)(place >> 7) * G * sp.stride + (place & 127);
        const float *xr = a.x + (size_t)row * d;
        float part = 0.f;
        for (int j = lane; j < d; j += 32) part = fmaf(xr[j], xr[j], part);
        const float xn = norm_up(warp_sum(part), d);
        auto fill = [&](int first, int w0) {
            int total = 0;
            for (int g0 = 0; g0 < G; g0 += 32) {
                uint32_t mk = g0 + lane < G ? bits[(size_t)(g0 + lane) * sp.stride] : 0u;
                const int k = __popc(mk);
                int at = k;
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(0xffffffffu, at, o);
                    if (lane >= o) at += v;
                }
                const int all = __shfl_sync(0xffffffffu, at, 31);
                at += first + total - k - w0;
                for (; mk; mk &= mk - 1, ++at)
                    if (at >= first && at < ND_WIN) s_tab[w][at] = (g0 + lane) * 16 + __ffs(mk) - 1;
                total += all;
            }
            __syncwarp();
            return total;
        };
        const int c = decide_nearest(near, fill, d, xr, xn, s_tab[w], s_lbs[w], lane);
        if (lane == 0) {
            if (c < 0 || c >= L) atomicOr(a.err, ERR_SELECT);
            a.out[row] = c < 0 || c >= L ? -1 : c;
        }
        __syncwarp();  // the warp's tables are reused
    }
}

// FP8 inverse scale of each list for its residual codes x - c_l: 448 / R_l
// with R_l the distance from c_l to its nearest other centroid (FP64, the
// squared distance summed in index order, no fused multiply-add); with a
// single list or a duplicated centroid (R_l = 0) the raw-magnitude rule
// 448 / (2 max_j |c_lj|) (1 for a zero centroid).  One warp per list, its
// lanes striding over the other centroids.
__global__ void k_fp8_scales(const float *__restrict__ cent, int L, int d,
                             float *__restrict__ inv_scale8)
{
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const int l = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (l >= L) return;
    const float *cl = cent + (size_t)l * d;
    double best = INFINITY;
    for (int o = lane; o < L; o += 32) {
        if (o == l) continue;
        const float *co = cent + (size_t)o * d;
        double s = 0.0;
        for (int j = 0; j < d; ++j) {
            const double t = __dsub_rn((double)cl[j], (double)co[j]);
            s = __dadd_rn(s, __dmul_rn(t, t));
        }
        best = fmin(best, s);
    }
    for (int o = 16; o > 0; o >>= 1) best = fmin(best, __shfl_xor_sync(0xffffffffu, best, o));
    if (lane == 0) {
        float inv;
        if (best > 0.0 && best < INFINITY) {
            inv = __double2float_rn(448.0 / sqrt(best));
        } else {
            double mx = 0.0;
            for (int j = 0; j < d; ++j) mx = fmax(mx, fabs((double)cl[j]));
            inv = mx > 0.0 ? __double2float_rn(448.0 / (2.0 * mx)) : 1.0f;
        }
        inv_scale8[l] = inv;
    }
}

// ------------------------------------------------------------ host drivers
void centroid_prep(sivf_index *ix, cudaStream_t st)
{
    ix->launches += 1;
    cudaMemsetAsync(ix->cmax, 0, 2 * sizeof(float), st);
    launch_pdl(k_centroid_norms, (ix->nlist * 32 + 127) / 128, 128, 0, st, ix->cent, ix->nlist, ix->d,
               ix->cnorm, ix->cnrm_up, ix->cmax, ix->cent_bf16, ix->cent_lo);
    if (ix->x8) {
        ix->launches += 1;
        launch_pdl(k_fp8_scales, (ix->nlist * 32 + 127) / 128, 128, 0, st, ix->cent, ix->nlist,
                   ix->d, ix->inv_scale8);
    }
}

// Squared distance from each centroid to its nearest other centroid, FP32
// (a statistic that picks the first stage, never a result).  A block takes
// GAP_N centroids against every GAP_N-row tile of a share of the others,
// both in shared memory (rows padded by one float4 against bank conflicts),
// each thread 2 x 2 pairs; the shares meet by atomicMin (distances are not
// negative, so their bits order as integers).  At L = 1,024, d = 128 the
// arithmetic is 10 us; with one warp per centroid, every lane walking a row
// of its own, the uncoalesced reads took 555 us.
constexpr int GAP_N = 32;
constexpr int GAP_NT = GAP_N * GAP_N / 4;
__global__ __launch_bounds__(GAP_NT) void k_cent_gap(const float *__restrict__ cent, int L, int d,
                                                     int *__restrict__ gap2)
{
    pdl_begin();
    extern __shared__ __align__(16) float4 gsm[];
    const int n4 = d >> 2, DP = n4 + 1, tid = threadIdx.x;
    float4 *sa = gsm, *sb = gsm + GAP_N * DP;
    const int a0 = blockIdx.x * GAP_N, ta = tid / (GAP_N / 2), tb = tid % (GAP_N / 2);
    const float4 *c4 = reinterpret_cast<const float4 *>(cent);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    auto stage = [&](float4 *to, int r0) {
        for (int e = tid; e < GAP_N * n4; e += GAP_NT) {
            const int r = e / n4, j = e % n4;
            to[r * DP + j] = r0 + r < L ? __ldg(c4 + (size_t)(r0 + r) * n4 + j) : zero;
        }
    };
    stage(sa, a0);
    float best[2] = {INFINITY, INFINITY};
    for (int b0 = blockIdx.y * GAP_N; b0 < L; b0 += gridDim.y * GAP_N) {
        __syncthreads();
        stage(sb, b0);
        __syncthreads();
        float s[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
        for (int j = 0; j < n4; ++j) {
            const float4 u[2] = {sa[ta * DP + j], sa[(ta + GAP_N / 2) * DP + j]};
            const float4 v[2] = {sb[tb * DP + j], sb[(tb + GAP_N / 2) * DP + j]};
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    float t = u[i].x - v[k].x;
                    s[i][k] = fmaf(t, t, s[i][k]);
                    t = u[i].y - v[k].y;
                    s[i][k] = fmaf(t, t, s[i][k]);
                    t = u[i].z - v[k].z;
                    s[i][k] = fmaf(t, t, s[i][k]);
                    t = u[i].w - v[k].w;
                    s[i][k] = fmaf(t, t, s[i][k]);
                }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int a = a0 + ta + i * (GAP_N / 2), b = b0 + tb + k * (GAP_N / 2);
                if (b < L && b != a) best[i] = fminf(best[i], s[i][k]);
            }
    }
    // the 16 threads of a row sit in one half warp
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        for (int o = 8; o > 0; o >>= 1) best[i] = fminf(best[i], __shfl_xor_sync(0xffffffffu, best[i], o));
        const int a = a0 + ta + i * (GAP_N / 2);
        if (tb == 0 && a < L) atomicMin(gap2 + a, __float_as_int(best[i]));
    }
}

// relative error of the BF16 first stage's dot products, |acc - x.c| /
// (||x|| ||c||): unit roundoff of BF16 ub = 2^-8; the FP32 accumulation of
// the exact BF16 products is taken as up to two ulps per addition, over d
// (single) or 3 d (split) terms.  Single: 2 ub + ub^2 (both roundings) plus
// the accumulation; split: the dropped products xl cl, and the roundings of
// xl and cl (each ub^2 relative), 3.1 ub^2 in all, plus the accumulation.
double first_stage_rel(int d, int split)
{
    const double ub = 1.0 / 256.0;
    const double gacc = (split == 3 ? 3.0 * d : (double)d) * std::ldexp(1.0, -22);
    return split == 3 ? 3.1 * ub * ub + gacc * (1 + 2 * ub)
                      : (2 * ub + ub * ub) + gacc * (1 + ub) * (1 + ub);
}

// Which first stage nearest-list assignment takes.  The single BF16 product
// decides a row on its own when the row's second-nearest list is farther
// than its nearest by more than twice the bound the fused stage uses,
// E = 2 gamma ||x|| max ||c|| (gamma = 2 first_stage_rel, the bound on one
// distance, doubled for safety); otherwise the row's candidates are
// recorded and re-decided, and a row with more candidates than its records
// hold is redone from every list.  For a point near its centroid that gap
// is about the squared distance R^2 from the centroid to its nearest
// neighbour, so when 2 E (taken at ||x|| = max ||c||) exceeds the median
// R^2, most rows would be undecided and the split first stage (bound about
// 60x tighter) is taken instead.  Both give the same assignment.
// Synchronizes `st`.
cudaError_t assign_stage_choose(sivf_index *ix, cudaStream_t st)
{
    ix->assign_split = false;
    const int L = ix->nlist, d = ix->d;
    if (!ix->cent_bf16 || !ix->cent_lo || L < 2 || L > CW_LMAX || d % 16 || d > 128)
        return cudaSuccess;
    float *gap2 = nullptr;
    cudaError_t e = cudaMallocAsync(reinterpret_cast<void **>(&gap2), sizeof(float) * L, st);
    if (e != cudaSuccess) return e;
    ix->launches += 1;
    // 0x7f7f7f7f: 3.4e38, no other centroid seen yet
    cudaMemsetAsync(gap2, 0x7f, sizeof(float) * L, st);
    const int na = (L + GAP_N - 1) / GAP_N;
    const size_t gsmem = (size_t)2 * GAP_N * (d / 4 + 1) * 16;  // 33.8 KB at d = 128
    launch_pdl(k_cent_gap, dim3(na, std::min(na, std::max(1, 152 * 4 / na))), GAP_NT, gsmem, st,
               ix->cent, L, d, reinterpret_cast<int *>(gap2));
    std::vector<float> g((size_t)L), cn((size_t)L);
    e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(g.data(), gap2, sizeof(float) * L, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(cn.data(), ix->cnorm, sizeof(float) * L, cudaMemcpyDeviceToHost, st);
    cudaFreeAsync(gap2, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    std::nth_element(g.begin(), g.begin() + L / 2, g.end());
    const double med = g[(size_t)L / 2];
    const double c2 = *std::max_element(cn.begin(), cn.end());
    const double e_max = 4.0 * first_stage_rel(d, 1) * c2;  // E at ||x|| = max ||c||
    ix->assign_split = std::isfinite(med) && 2.0 * e_max > med;
    return cudaSuccess;
}

// First stage of the selection of P lists: 1 the single BF16 product, 3
// the split BF16 products, 0 FP32.  The single product is within a few
// percent of ||x|| ||c||: tight enough to isolate the nearest centroid
// (assignment, P = 1) unless the centroids are close together against
// their norms (assign_stage_choose), but not to separate the P-th from the
// (P+1)-th of a dense shell of far centroids; probe selection takes the
// split form (three products, ~1e-4 of ||x|| ||c||), which needs twice the
// shared memory (d <= 128).  One warp per row suits up to a few thousand
// lists; beyond, the block kernel (256 threads per row) selects, from the
// FP32 first stage.
int first_stage_split(const sivf_index *ix, int P)
{
    const int d = ix->d;
    if (P > CW_PMAX || ix->nlist > CW_LMAX || d % 16) return 0;
    const bool single = P == 1 && !ix->assign_split;
    if (single) return ix->cent_bf16 && d <= kMaxD ? 1 : 0;
    return ix->cent_lo && d <= 128 ? 3 : 0;
}

// Probe selection by k_coarse_dist and k_coarse_pick: P lists need twice as
// many groups of 16 for the group minima to bound them well (L >= 32 P); the
// warp's candidate table holds P <= 128.  Few short rows to select from are read
// whole as fast (10,000 rows of 512 lists, d = 32, P = 2: 51 us, 60 by the pick).
bool coarse_picks(const sivf_index *ix, int P)
{
    if (P < 2 || P > PK_PMAX || !ix->tmap_cent_ok || (int64_t)ix->nlist < 32 * (int64_t)P) return false;
    return P > CW_PMAX || (int64_t)ix->nlist * ix->d >= 32768;
}

// Assignment of few rows: the fused stage gives 128 of them to a CTA, which
// passes over every list, and over every list twice more for the rows that
// need the second pass; k_coarse_dist deals its (tile, chunk) steps to all SMs.
// Up to 40 tiles of close centroids, 20 of others: 301 rows of 2,048 trained
// lists in 64 clusters take 34 us (host time included), 103 by the fused stage;
// 5,000 rows 53 and 129, 10,000 rows 139 and 100.  2,500 rows of 527 lists in 32
// clusters by the single product: 42 and 82; lists apart: the same to 2,500 rows,
// then the fused stage (10,000 rows of 1,024 lists: 38 us, 53).
static bool assign_near(const sivf_index *ix, int64_t m)
{
    const int L = ix->nlist;
    if (!ix->tmap_cent_ok || L < CF_LMIN || L > CW_LMAX) return false;
    return m <= (ix->assign_split ? 40 : 20) * CT_M;
}

// rows [0, m) of x -> out[m, P]; `Dbuf` holds at least `room` floats, L of
// them at least.
void coarse_topP(sivf_index *ix, const float *x, int64_t m, int P, int32_t *out,
                 float *Dbuf, int64_t room, cudaStream_t st)
{
    const int L = ix->nlist, d = ix->d;
    const double u = 5.9604644775390625e-08;
    const double gd = d * u / (1.0 - d * u);
    const bool warp_rows = P <= CW_PMAX && L <= CW_LMAX;
    // distances and group minima of at least one row
    const int64_t pick_row = L + (L + 15) / 16;
    const bool near = P == 1 && assign_near(ix, m) && room >= CF_HDR + std::min<int64_t>(m, 8 * CT_M) * pick_row;
    const bool pick = near || (coarse_picks(ix, P) && room >= CF_HDR + pick_row);
    const int split = pick ? 3 : first_stage_split(ix, P);
    const bool two = split != 0;
    const float gamma2_first = (float)(2.0 * first_stage_rel(d, split) * (1.0 + 1e-6));
    const int ro = pick && !near ? pk_ops(d) : re_ops(d);
    auto gamma_sum = [&](int ops) { return (float)(2.0 * (ops * u / (1.0 - ops * u)) * (1.0 + 1e-6)); };
    const float gamma2_re = gamma_sum(ro);
    // assignment (d <= 128) takes the fused first stage, which keeps only the
    // undecided rows and their candidate lists.  It needs far less room than
    // the matrix: a launch takes as many rows as leave records for half of
    // them beside the second pass's rows and bits (349,000 where the matrix of
    // L = 1024 lists takes 16,384); among close centroids about a third are
    // undecided
    const bool fused = P == 1 && two && !pick && ix->tmap_cent_ok && L >= CF_LMIN;
    const NearArgs na{ix->cent, ix->cnorm, ix->cnrm_up, gamma2_re};
    int nsm = 0;
    if (fused || pick) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        nsm = std::max(nsm, 1);
    }
    // ints of the second pass's rows, their list and bits for r rows in one launch
    const int64_t G = (L + 15) / 16;
    auto second_ints = [&](int64_t r) {
        return 2 * r + ((r + CT_M - 1) / CT_M * G * std::min<int64_t>(r, CT_M) + 1) / 2;
    };
    int64_t rows = std::min<int64_t>(std::max<int64_t>(room / L, 1), m);
    if (fused) {
        // with records for half of the rows, or what a tile can have
        const int64_t most = room - CF_HDR, rec = CF_STRIDE / 2, row = 2 + (G + 1) / 2;
        const int64_t many = (most - G * CT_M / 2) / (row + rec);
        const int64_t tile = std::min<int64_t>(CT_M, most / (row + 4));
        rows = std::min<int64_t>(std::max<int64_t>({many, tile, 1}), m);
    } else if (pick) {
        rows = std::min<int64_t>((room - CF_HDR) / pick_row, m);
    }
    for (int64_t r0 = 0; r0 < m; r0 += rows) {
        int mc = (int)std::min<int64_t>(rows, m - r0);
        const int64_t sec = fused ? second_ints(mc) : 0;
        SecondArgs sa{};
        const int cap = fused ? (int)std::max<int64_t>(0, std::min<int64_t>((room - CF_HDR - sec) / CF_STRIDE, mc)) : 0;
        const int tok = prof_begin(ix, PROF_COARSE, 2, st);
        // the distance buffer of the fused stage: the numbers of records and of
        // rows with bits, the second pass's rows, their list and bits, the
        // records; of the pick: the distances and the group minima
        int32_t *nh = reinterpret_cast<int32_t *>(Dbuf), *rec = nh + CF_HDR + sec;
        float *Dm = pick ? Dbuf + CF_HDR : Dbuf, *gm = Dm + (size_t)mc * L;
        if (pick) {
            const int KC = d <= 64 ? 1 : 2;
            const size_t smem = coarse_fused_smem(KC);
            const int nt = (mc + CT_M - 1) / CT_M, nch = (L + CF_CN - 1) / CF_CN;
            const CUtensorMap &tm = *reinterpret_cast<const CUtensorMap *>(ix->tmap_cent);
            const CUtensorMap &tl = *reinterpret_cast<const CUtensorMap *>(ix->tmap_cent_lo);
            static KernelSetup su[2];
            auto go = [&](auto kern, int i) {
                opt_in_smem(su[i], kern, smem);
                launch_pdl(kern, (unsigned)std::min<int64_t>((int64_t)nt * nch, nsm), CF_NT, smem, st,
                           tm, tl, x + r0 * d, mc, d, ix->cnorm, L, Dm, gm, ix->err);
            };
            if (KC == 1) go(k_coarse_dist<1>, 0);
            else go(k_coarse_dist<2>, 1);
        } else if (fused) {
            const int KC = d <= 64 ? 1 : 2, parts = split == 3 ? 2 : 1;
            const size_t smem = coarse_fused_smem(KC);
            sa.n = nh + 1;
            sa.rows = nh + CF_HDR;
            sa.list = sa.rows + mc;
            sa.bits = reinterpret_cast<uint16_t *>(sa.list + mc);
            sa.stride = std::min(mc, CT_M);
            sa.gamma = (float)(2.0 * first_stage_rel(d, 3) * (1.0 + 1e-6));
            cudaMemsetAsync(nh, 0, 2 * sizeof(int32_t), st);
            const int nt = (mc + CT_M - 1) / CT_M;
            const CUtensorMap &tm = *reinterpret_cast<const CUtensorMap *>(ix->tmap_cent);
            const CUtensorMap &tl = *reinterpret_cast<const CUtensorMap *>(ix->tmap_cent_lo);
            static KernelSetup su[4];
            auto go = [&](auto kern, int i) {
                opt_in_smem(su[i], kern, smem);
                launch_pdl(kern, std::min(nt, nsm), CF_NT, smem, st, tm, tl, x + r0 * d, mc, d,
                           ix->cnorm, ix->cmax, L, gamma2_first, out + r0, rec, cap, nh, sa, ix->err);
            };
            if (parts == 1) {
                if (KC == 1) go(k_coarse_fused<1, 1>, 0);
                else go(k_coarse_fused<2, 1>, 1);
            } else {
                if (KC == 1) go(k_coarse_fused<1, 2>, 2);
                else go(k_coarse_fused<2, 2>, 3);
            }
        } else if (two) {
            const size_t smem = coarse_tc_smem(d, split);
            dim3 g((mc + CT_M - 1) / CT_M, (L + CT_N - 1) / CT_N);
            if (split == 1) {
                static KernelSetup su;
                opt_in_smem(su, k_coarse_tc<1>, smem);
                launch_pdl(k_coarse_tc<1>, g, CT_NT, smem, st, x + r0 * d, mc, d, ix->cent_bf16,
                           nullptr, ix->cnorm, L, Dbuf, ix->err);
            } else {
                static KernelSetup su;
                opt_in_smem(su, k_coarse_tc<3>, smem);
                launch_pdl(k_coarse_tc<3>, g, CT_NT, smem, st, x + r0 * d, mc, d, ix->cent_bf16,
                           ix->cent_lo, ix->cnorm, L, Dbuf, ix->err);
            }
        } else {
            dim3 g((L + GBN - 1) / GBN, (mc + GBM - 1) / GBM);
            launch_pdl(k_coarse_gemm, g, 256, 0, st, x + r0 * d, mc, d, ix->cent, ix->cnorm, L,
                       Dbuf);
        }
        SelArgs a;
        a.D = fused ? nullptr : Dm;
        a.nhard = nh;
        a.S = rec;
        a.s_cap = cap;
        a.m = mc;
        a.L = L;
        a.P = P;
        a.d = d;
        a.x = x + r0 * d;
        a.cent = ix->cent;
        a.cn = ix->cnorm;
        a.cnrm_up = ix->cnrm_up;
        a.gamma2 = (float)(2.0 * gd * (1.0 + 1e-6));
        a.gamma2_first = gamma2_first;
        a.gamma2_re = gamma2_re;
        a.gamma2_w = gamma_sum(re_ops(d));
        a.two_level = two;
        a.Dw = pick ? Dm : nullptr;
        a.gmin = pick ? gm : nullptr;
        a.cmaxes = ix->cmax;
        a.out = out + r0 * P;
        a.err = ix->err;
        if (near) {
            launch_pdl(k_coarse_near, (unsigned)((mc + CW_ROWS - 1) / CW_ROWS), CW_ROWS * 32, 0, st, a, na);
        } else if (pick) {
            const int rpb = mc <= 4 * nsm ? 1 : CW_ROWS;
            launch_pdl(k_coarse_pick, (unsigned)((mc + rpb - 1) / rpb), PK_NT,
                       pk_block_smem(P, (L + 15) / 16), st, a, rpb);
        } else if (warp_rows) {
            const unsigned gw = (unsigned)((mc + CW_ROWS - 1) / CW_ROWS);
            if (fused)  // loops over the records
                launch_pdl(k_coarse_finish,
                           std::min<unsigned>((unsigned)((mc + FN_ROWS - 1) / FN_ROWS), 5u * (unsigned)nsm),
                           FN_ROWS * 32, 0, st, a, sa, na);
            else if (P == 1) launch_pdl(k_coarse_select_w<1>, gw, CW_ROWS * 32, 0, st, a);
            else launch_pdl(k_coarse_select_w<CW_PMAX>, gw, CW_ROWS * 32, 0, st, a);
        } else {
            launch_pdl(k_coarse_select, mc, SEL_NT, 0, st, a);
        }
        prof_end(ix, tok, st);
    }
}

}  // namespace sivf
