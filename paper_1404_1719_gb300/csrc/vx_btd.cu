// vx_btd.cu -- batched block-tridiagonal solve of the per-ray Newton systems (include/vx_btd.h).
//
// A ray's zones are a sequential chain. With many rays each belongs to one CTA, with fewer to two that eliminate from
// both ends, and with few a CTA takes a segment of a ray (each chosen by vx_btd_solve). k_btd_validate
// first checks that the ray offsets partition the zones (else every kernel returns at once):
//  * k_btd_convert: the caller's FP64 blocks to FP32, with the zero patterns of the couplings' rows.
//  * k_btd_factor: block elimination along the ray in FP32, one or two CTAs per ray. Per zone:
//    D_k = B_k - A_k G_{k-1} on the tensor cores, D_k inverted in place by Gauss-Jordan elimination with
//    partial pivoting in panels of eight columns (one warp eliminates within a panel, the others apply its
//    rank-8 transform on the tensor cores), G_k = D_k^{-1} C_k on the tensor cores. D_k^{-1} and G_k
//    replace B_k and C_k in the workspace.
//  * k_btd_segment, k_btd_join: the same for segments of rays, which leaves the system of their last zones to
//    k_btd_factor (or to k_btd_segment again); k_btd_again restores the blocks of a ray that could not be done so.
//  * k_btd_sweep, k_btd_seg_sweep: solve M delta = rhs with those: forward
//    y_k = D_k^{-1} (rhs_k - A_k y_{k-1}), backward delta_k = y_k - G_k delta_{k+1}, a chain of
//    matrix-vector products. The first sweep writes x = delta, later ones add delta to x in FP64.
//  * k_btd_resid: the FP64 residual r = d - M x from the caller's FP64 blocks, eight rows per warp, four
//    lanes per row (coalesced), zero groups of the couplings left out, FMA accumulation and a fixed two-step
//    shuffle reduction per row.
//  * k_btd_fp64: rays with a block whose inverse in FP32 says too little, in FP64.
// The host runs validate, convert, [segment, join, once or twice], factor, sweep, then n_refine times (resid,
// sweep), once or twice more for the rays with ill-conditioned blocks, and fp64, all on the caller's stream; with
// segments the factor kernel and the sweeps run once for the segments' system and once for the rays that have to be
// done as a whole (3 us each when there are none).
// With the inverse instead of the elimination's multipliers (which the sweeps replayed, a shuffle per
// unknown), GB300, m = 84, 400 zones a ray: one ray (one CTA) factor 24.3 -> 10.0 ms, a sweep 3.0 -> 1.3 ms; 304 rays
// 29.7 -> 14.0 ms (which included the conversion, now 5.9 ms apart) and 3.1 -> 1.7 ms (10.3 GB, 6.1 TB/s).
// The solution's error without refinement and with one sweep is 0.2 to 0.8 of what it was (m = 34 to 128).
#include "../../include/vx_btd.h"

#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <cstdint>
#include <new>

namespace vx {
vx_status set_error(vx_status s, const char *msg);  // the library's last-error text (vx_rates.cu)
}

namespace {

constexpr int kFactorThreads = 256;
constexpr int kResidThreads = 256;

vx_status bfail(vx_status s, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    return vx::set_error(s, buf);
}

// Device memory of the current device (or managed memory) with the given alignment; a host or
// unregistered pointer is rejected before anything is launched.
vx_status device_array(const void *p, size_t align, const char *name) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return bfail(VX_ERR_INVALID_ARG, "%s: not a CUDA pointer", name);
    }
    if (a.type != cudaMemoryTypeDevice && a.type != cudaMemoryTypeManaged)
        return bfail(VX_ERR_INVALID_ARG, "%s must be device memory", name);
    if ((uintptr_t)p % align) return bfail(VX_ERR_INVALID_ARG, "%s must be %zu-byte aligned", name, align);
    return VX_OK;
}

#define BTD_CU(call)                                                                          \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess)                                                                \
            return bfail(e_ == cudaErrorMemoryAllocation ? VX_ERR_OOM : VX_ERR_CUDA, "%s: %s (%s:%d)", \
                         #call, cudaGetErrorString(e_), __FILE__, __LINE__);                  \
    } while (0)

struct BtdArgs {
    int m, ld, mp, nbuf, nring, halves, n_rays;  // ld: row stride of the FP32 blocks; mp: m rounded up to 8;
                                                // halves: CTAs per ray (1 or 2)
    long long n_zones;
    const int *off;
    const double *A, *B, *C, *d, *rhs;
    double *x, *r;
    float *Di, *Gt, *At, *y;  // per zone B_k, then D_k^{-1}; C_k, then G_k; A_k in FP32, row-major [m][ld]; y_k [m]
    unsigned short *nz;       // [Z][C, A][mp] zero patterns of the rows
    // zbad, zmid: at a ray's first zone, whether a pivot failed, and the zone its eliminations meet at, from there;
    // before the elimination, zmid says of every zone which ends of its ray it is (kFirst, kLast)
    int *zbad, *zmid, *flag;
    int *zill;    // at a ray's first zone: how ill-conditioned its blocks are (pivot_level, the highest)
    int min_ill;  // only the rays of that level or more
    // Of such rays, at 2 (the first zone): max|residual| after their last sweep and max|d|, as bits; norm: k_btd_resid
    // raises them
    unsigned *znorm;
    bool norm;
    const int *inval;  // set by k_btd_validate when the offsets are not a partition of the zones
    // Rays in segments (k_btd_segment): parts > 0: this is the system of the segments' last zones, ray r's from r parts
    // on (above > 0: of segments of such a system, of `above` parts a ray); parts = 0 and pbad: only the rays
    // that pbad marks, whose elimination by segments failed
    int parts, above;
    int *pbad;
};

constexpr int kFirst = 1, kLast = 2;

// The segments of a ray of n zones: at most `parts`, of four zones or more.
__host__ __device__ __forceinline__ int seg_count(long long n, int parts) {
    const long long s = n / 4 < parts ? n / 4 : parts;
    return n < 1 ? 0 : s < 1 ? 1 : (int)s;
}

// The zone range of a ray; false (nothing to do) when the offsets failed validation.
__device__ __forceinline__ bool ray_range(const BtdArgs &a, int ray, long long &z0, long long &z1) {
    if (*a.inval) return false;
    z0 = a.off[ray];
    z1 = a.off[ray + 1];
    if (a.pbad && (a.parts > 0) == (a.pbad[ray] != 0)) return false;
    if (a.min_ill > 0 && (z1 == z0 || a.zill[z0] < a.min_ill)) return false;
    if (a.parts > 0) {
        const int s = seg_count(a.above > 0 ? seg_count(z1 - z0, a.above) : z1 - z0, a.parts);
        z0 = (long long)ray * a.parts;
        z1 = z0 + s;
    }
    return true;
}

// The zone at which a ray's two eliminations meet: its last with one CTA per ray, or few zones.
__device__ __forceinline__ long long ray_mid(const BtdArgs &a, long long z0, long long z1) {
    return a.halves == 2 && z1 - z0 >= 4 ? z0 + (z1 - z0) / 2 : z1 - 1;
}

// offsets[0] = 0, offsets[n_rays] = n_zones and non-decreasing; any violation marks the whole call
// invalid (so no two rays can share zones) and raises the numeric flag.
__global__ void k_btd_validate(const int *off, int n_rays, long long n_zones, int *inval, int *flag, int *zbad, int *zill,
                               unsigned *znorm, int *ends, int *pbad) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i > n_rays) return;
    if (pbad && i < n_rays) pbad[i] = 0;
    const long long v = off[i];
    bool bad = v < 0 || v > n_zones || (i == 0 && v != 0) || (i == n_rays && v != n_zones);
    const long long e = i < n_rays ? off[i + 1] : v;
    if (e < v) bad = true;
    if (bad) {
        atomicOr(inval, 1);
        atomicOr(flag, 1);
    } else if (v < e && e <= n_zones) {
        zbad[v] = 0;  // the factor kernel's arrival count
        zill[v] = 0;
        znorm[2 * v] = znorm[2 * v + 1] = 0u;
        ends[v] = v == e - 1 ? kFirst | kLast : kFirst;  // (zero before)
        if (v < e - 1) ends[e - 1] = kLast;
    }
}

__device__ __forceinline__ void btd_mma(float (&d)[4], const unsigned (&a)[4], const unsigned (&b)[2]) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// v = hi + lo, hi the nearest TF32 value (half an ulp of TF32 added to the magnitude bits, the last 13
// cleared), lo the exact remainder cut to TF32: a whole number of at most 2^12 ulps of v, of which TF32 holds all or all
// but the last bit, so cutting and rounding are off by the same, an ulp of v at most (2^-23 |v|).
__device__ __forceinline__ void btd_split(float v, unsigned &hi, unsigned &lo) {
    hi = (__float_as_uint(v) + 0x1000u) & 0xffffe000u;
    lo = __float_as_uint(__fsub_rn(v, __uint_as_float(hi))) & 0xffffe000u;
}
// A product at FP32 accuracy takes three of them: low x high, high x low, high x high (the dropped low x low is
// 2^-22 of a product, near FP32's rounding).

// Products of two m x m matrices U V in shared memory (row stride ld): eight warps (wm, wn) = 2 x 4 compute
// NT x NT tiles of 16 x 8 each, rows 16 (wm NT + x), columns 8 (wn NT + y). Fragment layout of m16n8k8:
// lane = 4 g + q holds U's rows g and g + 8 at columns q and q + 4 of a step of eight, V's rows q and q + 4
// at column g, and the result's rows g, g + 8 at columns 2q, 2q + 1. The radial couplings A_k and C_k
// are mostly zeros, so a row tile of A (a column tile of C) takes only the steps that nz marks: those whose
// 16 x 8 (8 x 8) block holds anything else.
//
// One row tile: d[y] = rows r0, r1 of U (offsets) times the NT column tiles of V.
template <int NT>
__device__ __forceinline__ void product_row(const float *U, int r0, int r1, const float *V, int ld, int m, int wn,
                                            int lane, unsigned nz, float (&d)[NT][4]) {
    const int g = lane >> 2, q = lane & 3;
#pragma unroll
    for (int y = 0; y < NT; ++y) d[y][0] = d[y][1] = d[y][2] = d[y][3] = 0.f;
#pragma unroll 1
    for (; nz; nz &= nz - 1) {
        const int k0 = 8 * (__ffs(nz) - 1);
        const bool ia = k0 + q < m, ib = k0 + q + 4 < m;
        const int ka = ia ? k0 + q : 0, kb = ib ? k0 + q + 4 : 0;
        float u[4], v[NT][2];
        u[0] = U[r0 + ka]; u[1] = U[r1 + ka]; u[2] = U[r0 + kb]; u[3] = U[r1 + kb];
#pragma unroll
        for (int y = 0; y < NT; ++y) {
            const int c = 8 * (wn * NT + y) + g;
            v[y][0] = c < m ? V[ka * ld + c] : 0.f;
            v[y][1] = c < m ? V[kb * ld + c] : 0.f;
        }
        unsigned ah[4], al[4], bh[NT][2], bl[NT][2];
        btd_split(ia ? u[0] : 0.f, ah[0], al[0]);
        btd_split(ia ? u[1] : 0.f, ah[1], al[1]);
        btd_split(ib ? u[2] : 0.f, ah[2], al[2]);
        btd_split(ib ? u[3] : 0.f, ah[3], al[3]);
#pragma unroll
        for (int y = 0; y < NT; ++y) {
            btd_split(ia ? v[y][0] : 0.f, bh[y][0], bl[y][0]);
            btd_split(ib ? v[y][1] : 0.f, bh[y][1], bl[y][1]);
        }
#pragma unroll
        for (int y = 0; y < NT; ++y) btd_mma(d[y], al, bh[y]);
#pragma unroll
        for (int y = 0; y < NT; ++y) btd_mma(d[y], ah, bl[y]);
#pragma unroll
        for (int y = 0; y < NT; ++y) btd_mma(d[y], ah, bh[y]);
    }
}
// One column tile: d[x] = the NT row tiles of U (row offsets ur) times column tile c0 / 8 of V, whose rows are
// taken in the order vrow.
template <int NT>
__device__ __forceinline__ void product_col(const float *U, const int (&ur)[NT][2], const float *V, const int *vrow,
                                            int ld, int m, int c0, int lane, unsigned nz, float (&d)[NT][4]) {
    const int g = lane >> 2, q = lane & 3;
    const bool ic = c0 + g < m;
#pragma unroll
    for (int x = 0; x < NT; ++x) d[x][0] = d[x][1] = d[x][2] = d[x][3] = 0.f;
#pragma unroll 1
    for (; nz; nz &= nz - 1) {
        const int k0 = 8 * (__ffs(nz) - 1);
        const bool ia = k0 + q < m, ib = k0 + q + 4 < m;
        const int ka = ia ? k0 + q : 0, kb = ib ? k0 + q + 4 : 0;
        float u[NT][4];
#pragma unroll
        for (int x = 0; x < NT; ++x) {
            u[x][0] = U[ur[x][0] + ka]; u[x][1] = U[ur[x][1] + ka];
            u[x][2] = U[ur[x][0] + kb]; u[x][3] = U[ur[x][1] + kb];
        }
        const float v0 = ic ? V[vrow[ka] * ld + c0 + g] : 0.f, v1 = ic ? V[vrow[kb] * ld + c0 + g] : 0.f;
        unsigned ah[NT][4], al[NT][4], bh[2], bl[2];
        btd_split(ia ? v0 : 0.f, bh[0], bl[0]);
        btd_split(ib ? v1 : 0.f, bh[1], bl[1]);
#pragma unroll
        for (int x = 0; x < NT; ++x) {
            btd_split(ia ? u[x][0] : 0.f, ah[x][0], al[x][0]);
            btd_split(ia ? u[x][1] : 0.f, ah[x][1], al[x][1]);
            btd_split(ib ? u[x][2] : 0.f, ah[x][2], al[x][2]);
            btd_split(ib ? u[x][3] : 0.f, ah[x][3], al[x][3]);
        }
#pragma unroll
        for (int x = 0; x < NT; ++x) btd_mma(d[x], al[x], bh);
#pragma unroll
        for (int x = 0; x < NT; ++x) btd_mma(d[x], ah[x], bl);
#pragma unroll
        for (int x = 0; x < NT; ++x) btd_mma(d[x], ah[x], bh);
    }
}

// Shared-memory stores under a predicate (no branch around them).
__device__ __forceinline__ void st4_if(bool p, unsigned a, float x, float y, float z, float w) {
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %0, 0;\n @p st.shared.v4.f32 [%1], {%2, %3, %4, %5};\n}" ::"r"((unsigned)p),
                 "r"(a), "f"(x), "f"(y), "f"(z), "f"(w)
                 : "memory");
}
__device__ __forceinline__ void st2_if(bool p, unsigned a, float x, float y) {
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %0, 0;\n @p st.shared.v2.f32 [%1], {%2, %3};\n}" ::"r"((unsigned)p), "r"(a),
                 "f"(x), "f"(y)
                 : "memory");
}
// The lane whose key won publishes its row (eight values at a) and the row's number (at b).
__device__ __forceinline__ void st_row_if(unsigned key, unsigned best, unsigned a, const float (&v)[8], unsigned b, int row) {
    asm volatile("{\n .reg .pred p;\n setp.eq.u32 p, %0, %1;\n @p st.shared.v4.f32 [%2], {%3, %4, %5, %6};\n"
                 " @p st.shared.v4.f32 [%2 + 16], {%7, %8, %9, %10};\n @p st.shared.u32 [%11], %12;\n}" ::"r"(key), "r"(best),
                 "r"(a), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "r"(b), "r"(row)
                 : "memory");
}
__device__ __forceinline__ void st1_if(bool p, unsigned a, unsigned x) {
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %0, 0;\n @p st.shared.u32 [%1], %2;\n}" ::"r"((unsigned)p), "r"(a), "r"(x)
                 : "memory");
}

// (float)x in integer operations: the conversion instruction runs on the FP64 pipe, at 2 per clock and SM on GB300
// (measured); this form is about ten integer operations. Nearly half an ulp is added (ties to even) and the
// exponent rebiased by 896. For zeros and for magnitudes from 2^-126 to below 2^127, which is what
// btd_plain says; the rest (FP32 subnormals, the last binade, infinities and NaN) goes by the instruction. The
// bits come by a move, so that the compiler does not turn the tests on them into FP64 comparisons.
__device__ __forceinline__ unsigned long long btd_bits(double x) {
    unsigned long long u;
    asm("mov.b64 %0, %1;" : "=l"(u) : "d"(x));
    return u;
}
__device__ __forceinline__ bool btd_plain(unsigned long long u) {
    const unsigned e = (unsigned)(u >> 32) & 0x7fffffffu;
    return e - (897u << 20) < 253u << 20 || e == 0u;
}
__device__ __forceinline__ float btd_plain_f32(unsigned long long u) {
    const unsigned long long b = u + 0x0fffffffull + ((u >> 29) & 1ull);
    const unsigned hi = (unsigned)(b >> 32), e = hi & 0x7fffffffu;
    return __uint_as_float((e < 1u << 20 ? 0u : __funnelshift_l((unsigned)b, e - (896u << 20), 3)) | (hi & 0x80000000u));
}

// The blocks in FP32, row-major with row stride ld, for the factor kernel and the sweeps: A_k to At, B_k to Di
// and C_k to Gt (the factor kernel puts D_k^{-1} and G_k in the places of B_k and C_k, which it has read by
// then), and per row of C and A a bit per eight columns that hold anything but zeros (nz[k][C, A][mp]; decided on
// the FP64 entries, so that the residual can go by it as well). A CTA takes a matrix at a time, a warp
// kConvRows of its rows, all their loads in flight together. Bound by HBM (8 m^2 bytes read and 4 m^2 written
// per block); apart from the factor kernel because the loads' registers, and the conversions' instructions,
// cost that kernel more than the extra pass. A of a ray's first zone and C of its last are left out: the caller's
// blocks there are not read, and nothing later reads theirs here.
constexpr int kConvThreads = 256, kConvRows = 4, kConvGrid = 8;  // kConvGrid: CTAs per SM
template <int NT>
__global__ void __launch_bounds__(kConvThreads) k_btd_convert(const BtdArgs a) {
    if (*a.inval) return;
    const int m = a.m, ld = a.ld, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = kConvThreads / 32;
    int ends = a.zmid[blockIdx.x / 3];
    for (long long q = blockIdx.x; q < 3 * a.n_zones; q += gridDim.x) {
        const long long k = q / 3;
        const int w = (int)(q - 3 * k);
        const bool skip = (w == 0 && (ends & kFirst)) || (w == 2 && (ends & kLast));
        if (q + gridDim.x < 3 * a.n_zones) ends = a.zmid[(q + gridDim.x) / 3];  // on its way while this one is done
        if (skip) continue;
        const double *src = (w == 0 ? a.A : w == 1 ? a.B : a.C) + (size_t)k * m * m + lane;
        float *dst = (w == 0 ? a.At : w == 1 ? a.Di : a.Gt) + (size_t)k * m * ld + lane;
        unsigned short *nz = a.nz + ((size_t)k * 2 + (w == 0)) * a.mp;
        for (int i0 = warp; i0 < m; i0 += kConvRows * nw) {
            double v[kConvRows][NT];
#pragma unroll
            for (int r = 0; r < kConvRows; ++r)
#pragma unroll
                for (int t = 0; t < NT; ++t)
                    v[r][t] = i0 + r * nw < m && (t < NT - 1 || lane + 32 * t < m) ? __ldcs(src + (i0 + r * nw) * m + 32 * t) : 0.0;
#pragma unroll
            for (int r = 0; r < kConvRows; ++r) {
                const int i = i0 + r * nw;
                if (i >= m) break;
                unsigned bits = 0u;
                bool plain = true;
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    const unsigned long long u = btd_bits(v[r][t]);
                    plain = plain && btd_plain(u);
                    if (t < NT - 1 || lane + 32 * t < m) dst[i * ld + 32 * t] = btd_plain_f32(u);
                    bits |= u << 1 != 0ull ? 1u << (4 * t) : 0u;
                }
                if (!plain) {
#pragma unroll 1
                    for (int t = lane; t < m; t += 32) dst[i * ld + t - lane] = (float)src[i * m + t - lane];
                }
                if (w == 1) continue;
                bits = __reduce_or_sync(0xffffffffu, bits << (lane >> 3));
                if (lane == 0) nz[i] = (unsigned short)bits;
            }
        }
    }
}

// Asynchronous 16-byte copies of n floats (a multiple of 4) by the whole CTA.
__device__ __forceinline__ void copy_async(float *dst, const float *src, int n, int tid, int nthreads) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst) + 16u * (unsigned)tid;
#pragma unroll 4
    for (int e = 4 * tid, i = 0; e < n; e += 4 * nthreads, ++i)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16u * (unsigned)(i * nthreads)), "l"(src + e) : "memory");
}
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.commit_group;\n cp.async.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ float btd_rcp(float p) {  // p and 1/p normal numbers
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(p));
    return fmaf(y, fmaf(-p, y, 1.f), y);  // a Newton step: the approximation's ulp would stay in the pivot row
}

// D^{-1} applied to a vector, unlike the elimination done over on it, carries the inverse's own error: where the product
// is much smaller than its terms, as with ill-conditioned blocks, the solution is further off (random blocks without a
// dominant diagonal, coupled by 0.3 of their size: 2 to 4 times in the median, 30 times in one ray of ten). A ray
// whose largest pivot in some zone exceeds the smallest kPivots1 or kPivots2 times is therefore refined once or twice
// more than asked, and not cut into segments. If a residual of more than kSlowest^(n_refine + 2) of d is left then (of
// 1e-10 of it with many sweeps, which end at the FP64 residual's rounding), a block's inverse in FP32 says too little,
// and the ray is solved in FP64 (k_btd_fp64). (The pivots are at hand; max|D| max|D^{-1}| says the same, and looking for
// it cost 2 to 4 %.) Blocks with dominant diagonals have a ratio of 1 to 2, Newton systems 10 to 13, those random
// blocks 15 to 1e4. A limit on the pivots instead of the residual (4096) also took rays that converge: random blocks
// coupled by 0.03 of their size, m = 84, 304 rays of 100 zones: 100 ms against 15.
constexpr float kPivots1 = 24.f, kPivots2 = 256.f, kSlowest = 0.03f;

// The panel warp's state: lane x holds rows x + 32 t of the panel's eight columns.
template <int NT>
struct Panel {
    float v[NT][8];
    unsigned cand[NT];  // magnitude mask of a row that can still be a pivot, 0 once it has been one
    unsigned piv;       // bit t: the row is one of this panel's pivots
    unsigned kmin, kmax;

    __device__ __forceinline__ void start(int m, int lane) {
#pragma unroll
        for (int t = 0; t < NT; ++t) cand[t] = lane + 32 * t < m ? 0x7fffff80u : 0u;
        kmin = 0xffffffffu;
        kmax = 0u;
    }
    // Rows lane + 32 t of columns c0 .. c0 + 7 of X.
    __device__ __forceinline__ static void fetch(float (&u)[NT][8], const float *X, int ld, int m, int c0, int lane) {
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const int i = lane + 32 * t;
            const float4 *s = reinterpret_cast<const float4 *>(X + (i < m ? i : 0) * ld + c0);
            const float4 a = s[0], b = s[1];
            u[t][0] = a.x; u[t][1] = a.y; u[t][2] = a.z; u[t][3] = a.w;
            u[t][4] = b.x; u[t][5] = b.y; u[t][6] = b.z; u[t][7] = b.w;
        }
    }
    // Zeros past the m-th row and column.
    __device__ __forceinline__ void trim(int m, int c0, int lane) {
        if (lane + 32 * (NT - 1) >= m) {
#pragma unroll
            for (int c = 0; c < 8; ++c) v[NT - 1][c] = 0.f;
        }
        if (c0 + 8 > m) {
#pragma unroll
            for (int t = 0; t < NT; ++t)
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (c0 + c >= m) v[t][c] = 0.f;
        }
    }
    __device__ __forceinline__ void store(float *X, int ld, int m, int c0, int lane) const {
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const int i = lane + 32 * t;
            const unsigned d = (unsigned)__cvta_generic_to_shared(X + (i < m ? i : 0) * ld + c0);
            if (c0 + 8 <= m) {
                st4_if(i < m, d, v[t][0], v[t][1], v[t][2], v[t][3]);
                st4_if(i < m, d + 16, v[t][4], v[t][5], v[t][6], v[t][7]);
            } else {
#pragma unroll
                for (int c = 0; c < 8; ++c) st1_if(i < m && c0 + c < m, d + 4 * c, __float_as_uint(v[t][c]));
            }
        }
    }
    // Goes on to the panel of columns c0 .. c0 + 7: they take the transform W this warp has just found (its
    // registers; pivot rows pr[0..7]): new = (X with the pivot rows zeroed) + W X_R.
    __device__ __forceinline__ void advance(const float *X, int ld, int m, int c0, const int *pr, int lane) {
        const int4 p0 = reinterpret_cast<const int4 *>(pr)[0], p1 = reinterpret_cast<const int4 *>(pr)[1];
        const int pk[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
        float u[NT][8];
        fetch(u, X, ld, m, c0, lane);
        float2 w[NT][4];
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int c = 0; c < 4; ++c)
                w[t][c] = (piv >> t) & 1u ? make_float2(0.f, 0.f) : make_float2(u[t][2 * c], u[t][2 * c + 1]);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float4 *s = reinterpret_cast<const float4 *>(X + pk[k] * ld + c0);
            const float4 a = s[0], b = s[1];
            const float2 y[4] = {make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(b.x, b.y), make_float2(b.z, b.w)};
#pragma unroll
            for (int t = 0; t < NT; ++t)
#pragma unroll
                for (int c = 0; c < 4; ++c) w[t][c] = __ffma2_rn(make_float2(v[t][k], v[t][k]), y[c], w[t][c]);
        }
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                v[t][2 * c] = w[t][c].x;
                v[t][2 * c + 1] = w[t][c].y;
            }
        trim(m, c0, lane);
    }
    // Gauss-Jordan steps of columns c0 .. c0 + nv - 1 within the panel, in place: after step j the column
    // holds what the elimination so far makes of the unit vector of its pivot row. The columns shift by one
    // register per step (free: each update writes the register before), so that the loop is not unrolled
    // and its instructions stay in the nearest cache. One warp reduction finds a pivot: the key holds the
    // magnitude's leading bits and, below them, 127 - row, so that keys differ and the lowest row wins among
    // magnitudes equal to 2^-16 (partial pivoting up to that factor). A second one broadcasts its value
    // while the pivot row goes through shared memory (rowbuf, two buffers of eight). The next column is
    // updated first and its pivot search started before the rest. The pivot rows are scaled by their
    // reciprocal pivots at the end.
    __device__ __forceinline__ void factor(int m, int c0, int nv, int *cur, float *rowbuf, int lane) {
        const unsigned rb = (unsigned)__cvta_generic_to_shared(rowbuf), cb = (unsigned)__cvta_generic_to_shared(cur + c0);
        float sc[NT];
        unsigned kt[NT], best = 0u;
        piv = 0u;
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            sc[t] = 1.f;
            kt[t] = (__float_as_uint(v[t][0]) & cand[t]) | (unsigned)(127 - lane - 32 * t);
            best = max(best, kt[t]);
        }
#pragma unroll 1
        for (int j = 0; j < nv; ++j) {
            best = __reduce_max_sync(0xffffffffu, best);
            kmin = min(kmin, best);
            kmax = max(kmax, best);
            const unsigned rj = rb + 32u * (unsigned)(j & 1);
            unsigned mine = 0u;
            bool own[NT];
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                own[t] = kt[t] == best;
                mine |= own[t] ? __float_as_uint(v[t][0]) : 0u;
            }
            const float p = __uint_as_float(__reduce_or_sync(0xffffffffu, mine));
#pragma unroll
            for (int t = 0; t < NT; ++t)  // a row past m - 1 wins only where no pivot is left
                st_row_if(kt[t], best, rj, v[t], cb + 4u * (unsigned)j, min(lane + 32 * t, m - 1));
            const float rp = best - 0x00800000u < 0x7d800000u ? btd_rcp(p) : 1.f / p;  // |p| in [2^-126, 2^125)
            __syncwarp();
            const float4 *rr = reinterpret_cast<const float4 *>(rowbuf + 8 * (j & 1));
            const float4 ya = rr[0], yb = rr[1];
            const float y[8] = {ya.x, ya.y, ya.z, ya.w, yb.x, yb.y, yb.z, yb.w};
            float l[NT];
            best = 0u;
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                l[t] = own[t] ? 0.f : -v[t][0] * rp;
                cand[t] = own[t] ? 0u : cand[t];
                sc[t] = own[t] ? rp : sc[t];
                piv |= own[t] ? 1u << t : 0u;
                v[t][0] = fmaf(l[t], y[1], v[t][1]);
                kt[t] = (__float_as_uint(v[t][0]) & cand[t]) | (unsigned)(127 - lane - 32 * t);
                best = max(best, kt[t]);
            }
#pragma unroll
            for (int t = 0; t < NT; ++t) {
#pragma unroll
                for (int c = 2; c < 8; ++c) v[t][c - 1] = fmaf(l[t], y[c], v[t][c]);
                v[t][7] = own[t] ? 1.f : l[t];
            }
        }
#pragma unroll 1
        for (int j = nv; j < 8; ++j) {  // a panel of fewer columns: zeros, shifted back into place
            st1_if(lane == 0, cb + 4u * (unsigned)j, 0u);
#pragma unroll
            for (int t = 0; t < NT; ++t) {
#pragma unroll
                for (int c = 1; c < 8; ++c) v[t][c - 1] = v[t][c];
                v[t][7] = 0.f;
            }
        }
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int c = 0; c < 8; ++c) v[t][c] *= sc[t];
        __syncwarp();
    }
    // -1: a column had no pivot (all candidates zero) or one that is not finite; else how ill-conditioned the block is.
    __device__ __forceinline__ int level() const {
        if (kmin < 128u || kmax >= 0x7f800000u) return -1;
        const float lo = __uint_as_float(kmin & 0x7fffff80u), hi = __uint_as_float(kmax & 0x7fffff80u);
        return (hi > kPivots1 * lo) + (hi > kPivots2 * lo);
    }
};

// Applies panel p's transform to one or two other 8-column tiles of X (t1 < 0: one), on the tensor cores:
// X = (X with the panel's pivot rows zeroed) + W X_R, a rank-8 product: one m16n8k8 step per 16 x 8 tile.
// A warp owns all rows of its tiles, so the pivot rows X_R are read, and zeroed, before it goes through the
// rows, NT tiles of 16 at a time so that their chains overlap. Rows past the m-th are computed from
// whatever follows in shared memory and not stored.
template <int NT>
__device__ __forceinline__ void tile_update(float *X, int ld, int m, int p, int t0, int t1, const int *cur, int lane) {
    const int g = lane >> 2, q = lane & 3;
    const bool ia = 8 * p + q < m, ib = 8 * p + q + 4 < m;  // the last panel may hold fewer than 8 columns
    const int ra = cur[8 * p + q] * ld, rb = cur[8 * p + q + 4] * ld;
    unsigned bh[2][2], bl[2][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int t = h ? t1 : t0;
        if (t >= 0) {
            const int c = 8 * t + g;
            btd_split(ia && c < m ? X[ra + c] : 0.f, bh[h][0], bl[h][0]);
            btd_split(ib && c < m ? X[rb + c] : 0.f, bh[h][1], bl[h][1]);
        }
    }
    __syncwarp();
    const unsigned xs = (unsigned)__cvta_generic_to_shared(X);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int t = h ? t1 : t0;
        if (t >= 0) {
            const int c = 8 * t + g;
            st1_if(ia && c < m, xs + 4u * (unsigned)(ra + c), 0u);
            st1_if(ib && c < m, xs + 4u * (unsigned)(rb + c), 0u);
        }
    }
    __syncwarp();
    const float *W = X + g * ld + 8 * p + q;
    const int c0 = g * ld + 8 * t0 + 2 * q, c1 = g * ld + 8 * (t1 < 0 ? t0 : t1) + 2 * q;
#pragma unroll 1
    for (int i0 = 0; i0 < m; i0 += 16 * NT) {
        unsigned ah[NT][4], al[NT][4];
#pragma unroll
        for (int x = 0; x < NT; ++x) {
            const float *w = W + (i0 + 16 * x) * ld;
            btd_split(w[0], ah[x][0], al[x][0]);
            btd_split(w[8 * ld], ah[x][1], al[x][1]);
            btd_split(w[4], ah[x][2], al[x][2]);
            btd_split(w[8 * ld + 4], ah[x][3], al[x][3]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int t = h ? t1 : t0;
            if (t < 0) break;
            float *y = X + i0 * ld + (h ? c1 : c0);
            float d[NT][4];
            float2 e[NT][2];
#pragma unroll
            for (int x = 0; x < NT; ++x) {
                d[x][0] = d[x][1] = d[x][2] = d[x][3] = 0.f;
                e[x][0] = *reinterpret_cast<const float2 *>(y + 16 * x * ld);
                e[x][1] = *reinterpret_cast<const float2 *>(y + (16 * x + 8) * ld);
            }
#pragma unroll
            for (int x = 0; x < NT; ++x) btd_mma(d[x], al[x], bh[h]);
#pragma unroll
            for (int x = 0; x < NT; ++x) btd_mma(d[x], ah[x], bl[h]);
#pragma unroll
            for (int x = 0; x < NT; ++x) btd_mma(d[x], ah[x], bh[h]);
            // added in FP32, rounded to nearest: the tensor core's own accumulation cuts the sum's last bits
#pragma unroll
            for (int x = 0; x < NT; ++x) {
                d[x][0] += e[x][0].x; d[x][1] += e[x][0].y;
                d[x][2] += e[x][1].x; d[x][3] += e[x][1].y;
            }
            if (8 * t + 8 <= m) {
#pragma unroll
                for (int x = 0; x < NT; ++x) {
                    const unsigned ys = xs + 4u * (unsigned)(y - X) + 64u * (unsigned)(x * ld);
                    st2_if(i0 + 16 * x + g < m, ys, d[x][0], d[x][1]);
                    st2_if(i0 + 16 * x + g + 8 < m, ys + 32u * (unsigned)ld, d[x][2], d[x][3]);
                }
            } else {
                const bool j0 = 8 * t + 2 * q < m, j1 = 8 * t + 2 * q + 1 < m;
#pragma unroll
                for (int x = 0; x < NT; ++x) {
                    const bool r0 = i0 + 16 * x + g < m, r1 = i0 + 16 * x + g + 8 < m;
                    const unsigned ys = xs + 4u * (unsigned)(y - X) + 64u * (unsigned)(x * ld);
                    st1_if(r0 && j0, ys, __float_as_uint(d[x][0]));
                    st1_if(r0 && j1, ys + 4u, __float_as_uint(d[x][1]));
                    st1_if(r1 && j0, ys + 32u * (unsigned)ld, __float_as_uint(d[x][2]));
                    st1_if(r1 && j1, ys + 32u * (unsigned)ld + 4u, __float_as_uint(d[x][3]));
                }
            }
        }
    }
}

// Shared memory of the factor and segment kernels: nbuf buffers of m x ld floats (16 floats of slack each: the last
// tiles read past the end of a row), the zero patterns of C_k's and A_{k+1}'s rows, two rows
// of a panel, the pivot rows and their inverse.
__host__ __device__ constexpr int factor_buf(int m, int ld) { return (m * ld + 16 + 3) & ~3; }
__host__ __device__ constexpr size_t factor_smem(int m, int ld, int nbuf) {
    return (size_t)nbuf * factor_buf(m, ld) * sizeof(float) + (size_t)(16 + 3 * ((m + 7) & ~7)) * sizeof(int) +
           (size_t)m * sizeof(int);
}

// Row stride of the blocks: 4 mod 8 floats, so that the MMA fragments of the left operand (eight rows, four columns) fall
// in distinct banks, and a matrix is copied in whole 16-byte pieces.
__host__ __device__ constexpr int row_stride(int m) { return m + (12 - m % 8) % 8; }

// tile_update reads whole groups of 16 NT rows, so up to 31 rows past the end of X, and eight columns of the last panel.
// X is the first buffer, or the second of four or more: what it reads there has to be memory of the CTA.
constexpr bool reads_stay_inside() {
    for (int m = 1; m <= VX_BTD_MAX_M; ++m) {
        const int nt = (m + 31) / 32, ld = row_stride(m), rows = (m + 16 * nt - 1) / (16 * nt) * 16 * nt;
        for (int nbuf = 3; nbuf <= 5; ++nbuf) {
            const size_t x = nbuf > 3 ? factor_buf(m, ld) : 0, end = x + (size_t)(rows - 1) * ld + 8 * ((m + 7) / 8);
            if (end * sizeof(float) > factor_smem(m, ld, nbuf)) return false;
        }
    }
    return true;
}
static_assert(reads_stay_inside(), "tile_update reads past the shared memory");

// X -= U V, all in shared memory; the rows of U hold something only in the groups that nz marks.
template <int NT>
__device__ __forceinline__ void subtract_product(float *X, const float *U, const float *V, const unsigned short *nz, int ld,
                                                 int m, int wm, int wn, int lane) {
    const int g = lane >> 2, q = lane & 3;
#pragma unroll 1
    for (int x = 0; x < NT; ++x) {
        const int i0 = 16 * (wm * NT + x), i = i0 + (lane & 15);
        const unsigned todo = __reduce_or_sync(0xffffffffu, i < m ? (unsigned)nz[i] : 0u);
        float d[NT][4];
        const int r0 = i0 + g < m ? i0 + g : m - 1, r1 = i0 + g + 8 < m ? i0 + g + 8 : m - 1;
        product_row<NT>(U, r0 * ld, r1 * ld, V, ld, m, wn, lane, todo, d);
        const bool i0m = i0 + g < m, i1m = i0 + g + 8 < m;
#pragma unroll
        for (int y = 0; y < NT; ++y) {
            const int c = 8 * (wn * NT + y) + 2 * q;
            float *x0 = X + r0 * ld + c, *x1 = X + r1 * ld + c;
            if (c + 1 < m) {
                const float2 e0 = *reinterpret_cast<float2 *>(x0), e1 = *reinterpret_cast<float2 *>(x1);
                if (i0m) *reinterpret_cast<float2 *>(x0) = make_float2(e0.x - d[y][0], e0.y - d[y][1]);
                if (i1m) *reinterpret_cast<float2 *>(x1) = make_float2(e1.x - d[y][2], e1.y - d[y][3]);
            } else if (c < m) {
                if (i0m) *x0 -= d[y][0];
                if (i1m) *x1 -= d[y][2];
            }
        }
    }
}

// Inverts X in place up to the order of its rows and columns: eliminates panel after panel, one CTA barrier each;
// in step it, warp 0 eliminates within panel it, the others apply panel it - 1. Pivot j's row is cur[j], pos its
// inverse: X^{-1}[j][cur[q]] = X[cur[j]][q]. Returns Panel::level in warp 0, else 0. No barrier at its end.
template <int NT>
__device__ __forceinline__ int invert(float *X, int ld, int m, int *cur, int *pos, float *rowbuf, int tid) {
    const int lane = tid & 31, warp = tid >> 5, nw = kFactorThreads / 32, P = (m + 7) >> 3;
    Panel<NT> pn;
    if (warp == 0) pn.start(m, lane);
    for (int it = 0; it <= P; ++it) {  // step P: the last panel's transform, by all warps
        const int nu = it < P ? nw - 1 : nw, u = warp - (nw - nu);  // the warps that update, and this one's number
        if (u < 0) {
            if (it == 0) {
                Panel<NT>::fetch(pn.v, X, ld, m, 0, lane);
                pn.trim(m, 0, lane);
            } else {
                pn.advance(X, ld, m, 8 * it, cur + 8 * (it - 1), lane);
            }
            pn.factor(m, 8 * it, m - 8 * it < 8 ? m - 8 * it : 8, cur, rowbuf, lane);
            pn.store(X, ld, m, 8 * it, lane);
        } else {
            if (it > 0) {  // every tile but it - 1 (the transform itself) and it
                const int t0 = u, t1 = u + nu, nt = it < P ? P - 2 : P - 1;
                if (t0 < nt)
                    tile_update<NT>(X, ld, m, it - 1, t0 < it - 1 ? t0 : t0 + 2, t1 < nt ? (t1 < it - 1 ? t1 : t1 + 2) : -1,
                                    cur, lane);
            }
            if (it == P && tid < m) pos[cur[tid]] = tid;
        }
        if (it < P) __syncthreads();
    }
    return warp == 0 ? pn.level() : 0;
}

// The inverse of X (as invert leaves it), row by row, to Di.
template <int NT>
__device__ __forceinline__ void store_inverse(float *Di, const float *X, int ld, int m, const int *cur, const int *pos, int tid) {
    const int lane = tid & 31, warp = tid >> 5, nw = kFactorThreads / 32;
    int pc[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) pc[t] = lane + 32 * t < m ? pos[lane + 32 * t] : 0;
    for (int j = warp; j < m; j += nw) {
        const float *row = X + cur[j] * ld;
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const int c = lane + 32 * t;
            if (c < m) Di[j * ld + c] = row[pc[t]];
        }
    }
}

// acc[column tile][row tile] = X^{-1} V, X as invert leaves it; V's rows hold something only in the groups that
// nzr marks (all: in every group).
template <int NT>
__device__ __forceinline__ void inverse_times(float (&acc)[NT][NT][4], const float *X, const float *V, const unsigned short *nzr,
                                              const int *cur, int ld, int m, int wm, int wn, int lane) {
    const int g = lane >> 2;
    int ur[NT][2];
    unsigned nz[NT];
#pragma unroll
    for (int x = 0; x < NT; ++x) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = 16 * (wm * NT + x) + g + 8 * h;
            ur[x][h] = cur[i < m ? i : m - 1] * ld;
        }
        nz[x] = 0u;
    }
#pragma unroll
    for (int t = 0; t < NT; ++t) {  // row lane + 32 t in pivot order belongs to step (lane >> 3) + 4 t
        const int j = lane + 32 * t;
        const unsigned f = j < m ? (nzr ? (unsigned)nzr[cur[j]] : 0xffffu) >> (wn * NT) : 0u;
#pragma unroll
        for (int x = 0; x < NT; ++x) nz[x] |= ((f >> x) & 1u) << ((lane >> 3) + 4 * t);
    }
#pragma unroll
    for (int y = 0; y < NT; ++y) {
        const unsigned todo = __reduce_or_sync(0xffffffffu, nz[y]);
        product_col<NT>(X, ur, V, cur, ld, m, 8 * (wn * NT + y), lane, todo, acc[y]);
    }
}

// acc, times sign, to row-major matrices in shared (S) and global (D) memory; raises big to its largest magnitude and
// clears finite if an entry is not.
template <int NT>
__device__ __forceinline__ void store_tiles(float *S, float *D, const float (&acc)[NT][NT][4], float sign, int ld, int m, int wm,
                                            int wn, int lane, float &big, bool &finite) {
    const int g = lane >> 2, q = lane & 3;
#pragma unroll
    for (int x = 0; x < NT; ++x)
#pragma unroll
        for (int y = 0; y < NT; ++y)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = 16 * (wm * NT + x) + g + 8 * h, c = 8 * (wn * NT + y) + 2 * q;
                if (i < m && c < m) {
                    const float e0 = sign * acc[y][x][2 * h], e1 = sign * acc[y][x][2 * h + 1];
                    if (!(fabsf(e0) < INFINITY && fabsf(e1) < INFINITY)) finite = false;
                    big = fmaxf(big, fmaxf(fabsf(e0), fabsf(e1)));
                    if (c + 1 < m) {
                        if (S) *reinterpret_cast<float2 *>(S + i * ld + c) = make_float2(e0, e1);
                        if (D) *reinterpret_cast<float2 *>(D + i * ld + c) = make_float2(e0, e1);
                    } else {
                        if (S) S[i * ld + c] = e0;
                        if (D) D[i * ld + c] = e0;
                    }
                }
            }
}

// The factor kernel: CTAs of eight warps, one per ray, or two where one would leave SMs without work
// (a.halves): then one eliminates from the ray's first zone outwards and one from its last zone inwards, D_k =
// B_k - C_k H_{k+1} with H_k = D_k^{-1} A_k, and whichever comes second to the zone between them (mid) takes
// that one too, D = B - A G_{mid-1} - C H_{mid+1}: the same arithmetic in half the time. Elimination from
// the last zone needs what elimination from the first does not (a B of the last zone that can be
// inverted, say), so if the inner-going half meets a failed pivot, or |H| above kMaxGrowth, the ray goes on from mid
// to its last zone as if by one CTA, from blocks converted again. One CTA: mid is the last zone.
// Per zone k, in either direction (below for the outward one):
//  - D_k = B_k - A_k G_{k-1} on the tensor cores (all three in shared memory);
//  - D_k is inverted in place by Gauss-Jordan elimination with partial pivoting, eight columns (a panel) at
//    a time: warp 0 eliminates within a panel in registers, with no barrier between its eight pivots;
//    the other warps apply the panel's rank-8 transform to the remaining column tiles on the tensor
//    cores while warp 0 brings the next panel up to date and eliminates in it. One CTA barrier per
//    panel. Rows are never moved: pivot j's row is cur[j], and D_k^{-1}[j][cur[q]] = X[cur[j]][q];
//  - meanwhile C_k, A_{k+1} and (with a fourth buffer) B_{k+1} arrive in shared memory (cp.async);
//  - G_k = D_k^{-1} C_k on the tensor cores.
// D_k^{-1} replaces B_k in the workspace and G_k replaces C_k (H_k replaces A_k); the FP32 copy of the other
// coupling stays, for the sweeps. The chain of pivots (a warp
// reduction, a shuffle and a reciprocal each) bounds a zone; the warps beside it do everything else.
// GB300, m = 84, 400 zones: one ray 10.1 -> 5.1 ms with two CTAs.
// Largest entry of G, H, L, R and L' with which a ray is left in halves or segments. Above it the errors of the local
// eliminations multiply: random 150-zone rays without a dominant diagonal (FP32, two levels of segments), the
// error before refinement against plain elimination from the first zone: entries up to 4, 1500 rays, median 1.0,
// worst 33 (the other way 60) and 3e-13 after two sweeps (plain 5e-14); entries up to 64, worst 400, and 2e-4
// after two sweeps where plain has 4e-13. Systems with dominant diagonals have entries below 1, Newton systems
// about their largest flux number (2.9 with 3).
constexpr float kMaxGrowth = 4.f;
template <int NT>
__global__ void __launch_bounds__(kFactorThreads, NT > 3 ? 1 : 2) k_btd_factor(const BtdArgs a) {
    extern __shared__ __align__(16) float sm[];
    __shared__ int s_bad, s_grow, s_all, s_ill;
    const int m = a.m, ld = a.ld, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int bs = factor_buf(m, ld), P = (m + 7) >> 3;
    const bool four = a.nbuf == 4;
    // D_k and the next zone's B come first: tile_update reads past the end of D_k (reads_stay_inside)
    // (offsets, not pointers, are exchanged from zone to zone: the compiler then knows the address space)
    int xo = 0, bo = four ? bs : 0;
    float *const sG = sm + bo + bs, *const sA = sG + bs;
    unsigned short *nzr = reinterpret_cast<unsigned short *>(sm + a.nbuf * bs);  // [next coupling, previous coupling][mp]
    float *rowbuf = sm + a.nbuf * bs + a.mp;  // [2][8]
    int *cur = reinterpret_cast<int *>(rowbuf + 16);
    int *pos = cur + 8 * P;
    long long z0, z1;
    const int half = a.halves == 2 ? (int)(blockIdx.x & 1) : 0;
    if (!ray_range(a, blockIdx.x / a.halves, z0, z1) || z1 == z0) return;
    long long mid = ray_mid(a, z0, z1);
    if (half == 1 && mid == z1 - 1) return;
    if (tid == 0) s_bad = s_grow = s_ill = 0;
    int *const ill = a.zill + a.off[blockIdx.x / a.halves];
    if (tid < m) pos[tid] = tid;  // in range also where a failed pivot leaves an entry unset
    const int mw = m * ld;
    const int wm = warp & 1, wn = warp >> 1;
    // zeros behind every buffer: the last panel's transform, if it has fewer than eight columns, is read that far
    // (and multiplied by zeros, so it must be finite)
    for (int i = tid; i < a.nbuf * (bs - mw); i += kFactorThreads) sm[i / (bs - mw) * bs + mw + i % (bs - mw)] = 0.f;
    auto load = [&](float *dst, const float *src) { copy_async(dst, src, mw, tid, kFactorThreads); };
    auto load_nz = [&](int to, long long k, int which) {  // the zero pattern of C_k (which 0) or A_k (1)
        copy_async(reinterpret_cast<float *>(nzr + to * a.mp), reinterpret_cast<const float *>(a.nz + ((size_t)k * 2 + which) * a.mp),
                   a.mp / 2, tid, kFactorThreads);
    };
    auto at = [&](float *w, long long k) { return w + (size_t)k * mw; };
    auto schur = [&](float *X) {  // X -= (coupling in sA) (matrix in sG)
        subtract_product<NT>(X, sA, sG, nzr + a.mp, ld, m, wm, wn, lane);
        __syncthreads();
    };
    // this CTA's chain: left zones from k on in direction dir, their couplings to the next zone in nx and to
    // the one before in pv; passes: products to subtract from the zone at hand
    int dir = half ? -1 : 1, left = (int)(half ? z1 - 1 - mid : mid - z0), passes = 0;
    long long k = half ? z1 - 1 : z0;
    float *nx = half ? a.At : a.Gt, *pv = half ? a.Gt : a.At;
    bool joined = a.halves == 1 || mid == z1 - 1;  // no other half to wait for
    if (left > 0) {
        load(sm, at(a.Di, k));
        copy_wait();
        __syncthreads();
    }
    for (;;) {
        const bool at_mid = left == 0;
        float *const X = sm + xo, *const sB = sm + bo;
        if (at_mid) {
            __syncthreads();
            if (!joined) {
                // the second half to arrive goes on: + 1 each, + 16 for a failed outward half, + 256 inward
                if (tid == 0) {
                    if (a.parts > 0) s_bad |= s_ill;
                    else if (s_ill) atomicMax(ill, s_ill);
                    const int add = 1 + (half ? ((s_bad | s_grow) ? 256 : 0) : (s_bad ? 16 : 0));
                    __threadfence();
                    s_all = atomicAdd(a.zbad + z0, add) + add;
                    __threadfence();
                }
                __syncthreads();
                const int all = s_all;
                if ((all & 3) < 2) return;
                joined = true;
                if (tid == 0) {
                    s_bad = (all & 16) != 0 || ((all & 256) && !a.A);
                    s_grow = 0;
                }
                if ((all & 256) && !(all & 16) && a.A) {  // on from mid to the last zone, outwards
                    for (long long e = (long long)mid * m * m + tid; e < z1 * m * m; e += kFactorThreads) {
                        const long long row = e / m;
                        const int c = (int)(e - row * m);
                        a.At[(size_t)row * ld + c] = (float)a.A[e];
                        a.Di[(size_t)row * ld + c] = (float)a.B[e];
                    }
                    __threadfence();
                    __syncthreads();
                    k = mid;
                    left = (int)(z1 - 1 - mid);
                    passes = mid > z0;
                    mid = z1 - 1;
                    dir = 1;
                    nx = a.Gt;
                    pv = a.At;
                    load(X, at(a.Di, k));
                    if (passes) {
                        load(sA, at(a.At, k));
                        load(sG, at(a.Gt, k - 1));
                        load_nz(1, k, 1);
                    }
                    copy_wait();
                    __syncthreads();
                    if (left > 0) continue;
                }
            }
            k = mid;
            load(X, at(a.Di, k));
            if (mid > z0) {
                load(sA, at(a.At, k));
                load(sG, at(a.Gt, k - 1));
                load_nz(1, k, 1);
                copy_wait();
                __syncthreads();
                schur(X);
            }
            if (mid < z1 - 1) {
                load(sA, at(a.Gt, k));
                load(sG, at(a.At, k + 1));
                load_nz(1, k, 0);
                copy_wait();
                __syncthreads();
                schur(X);
            }
            copy_wait();
            __syncthreads();
        } else {
            if (passes) schur(X);
            load(sG, at(nx, k));
            load_nz(0, k, dir > 0 ? 0 : 1);
            if (left > 1) {
                load(sA, at(pv, k + dir));
                load_nz(1, k + dir, dir > 0 ? 1 : 0);
                if (four) load(sB, at(a.Di, k + dir));
            }
        }
        const int level = invert<NT>(X, ld, m, cur, pos, rowbuf, tid);
        if (tid == 0) {
            if (level < 0) s_bad = 1;
            else s_ill = max(s_ill, level);
        }
        copy_wait();
        __syncthreads();
        store_inverse<NT>(at(a.Di, k), X, ld, m, cur, pos, tid);
        if (at_mid) break;
        float acc[NT][NT][4], big = 0.f;
        bool finite = true;
        inverse_times<NT>(acc, X, sG, nzr, cur, ld, m, wm, wn, lane);
        __syncthreads();  // the next coupling and D_k^{-1} have been read
        store_tiles<NT>(sG, at(nx, k), acc, 1.f, ld, m, wm, wn, lane, big, finite);
        if (!finite) s_bad = 1;
        if (big > kMaxGrowth) s_grow = 1;
        --left;
        k += dir;
        passes = 1;
        if (left > 0) {
            if (four) {
                const int t = xo;
                xo = bo;
                bo = t;
            } else {
                load(X, at(a.Di, k));
                copy_wait();
            }
        }
        __syncthreads();
    }
    __syncthreads();
    if (tid == 0) {
        if (a.parts > 0) s_bad |= s_ill;
        else if (s_ill) atomicMax(ill, s_ill);
        a.zbad[z0] = s_bad;
        a.zmid[z0] = (int)(mid - z0);
        if (s_bad) {
            if (a.parts > 0) a.pbad[blockIdx.x / a.halves] = 1;
            else atomicOr(a.flag, 2);
        }
    }
}

// Rays in segments, where there are so few that most SMs would have none: a ray of n zones is cut into S segments, all
// eliminated at the same time by a CTA each. The segment's last zone e stays; the others, a .. e - 1, are
// eliminated outwards, with a second right-hand side for their coupling to the zone p = a - 1 before the segment,
//   x_k = y_k - G_k x_{k+1} - L_k x_p,  L_a = D_a^{-1} A_a,  L_k = -D_k^{-1} A_k L_{k-1},
// and then once more inwards for the segment's first zone, x_a = y' - R x_e - L' x_p (R_k = -G_k R_{k+1},
// L'_k = L_k - G_k L'_{k+1}). That leaves a block-tridiagonal system of the segments' last zones,
//   Ar_e = -A_e L_{e-1},  Br_e = B_e - A_e G_{e-1} - C_e L'_{next a},  Cr_e = -C_e R_{next a},
// for k_btd_factor, or of enough rows to be cut into segments once more. A ray in which a pivot fails, a block is
// ill-conditioned (kPivots1), or an entry of G, L, R or L' is above kMaxGrowth, is done again as a whole by k_btd_factor
// (pbad). The time is that of n / S + S / 2 zones, not n / 2.
// GB300, m = 84, 400 zones, one ray: 5.11 ms by two CTAs -> 0.27 ms for 69 segments, 0.29 for 14 of
// their last zones and 0.29 for those segments' last zones (0.58 and 0.66 with 34 segments and one level).
struct SegArgs {
    BtdArgs a;
    int parts, above, nbuf;     // above: parts of the level whose last zones these segments are made of, or 0
    float *Lt;                  // L_k, per zone
    float *Dr, *Cr, *Ar, *Er;   // [n_rays][parts] Br_e without its last term, Cr_e, Ar_e, that term
    unsigned short *nzr;        // zero patterns of Cr, Ar: none
    int *zbadr, *pbad;
    double *rr, *xr;            // [n_rays][parts][m] the right-hand sides and the solution of that system
};

// Segment s of ray r: its zones za .. ze (the one that stays), its row in the system of those.
struct Seg {
    long long za, ze, row;
    bool first, last;
    __device__ __forceinline__ bool find(const SegArgs &p, int block, bool good) {
        const int ray = block / p.parts, i = block % p.parts;
        if (*p.a.inval || (good && p.pbad[ray])) return false;
        long long z0 = p.a.off[ray], n = p.a.off[ray + 1] - z0;
        if (p.above > 0) {
            n = seg_count(n, p.above);
            z0 = (long long)ray * p.above;
        }
        const int S = seg_count(n, p.parts);
        if (i >= S) return false;
        za = z0 + n * i / S;
        ze = z0 + n * (i + 1) / S - 1;
        row = (long long)ray * p.parts + i;
        first = i == 0;
        last = i == S - 1;
        return true;
    }
};

template <int NT>
__global__ void __launch_bounds__(kFactorThreads, 1) k_btd_segment(const SegArgs p) {
    extern __shared__ __align__(16) float sm[];
    __shared__ int s_bad, s_go;
    const BtdArgs &a = p.a;
    Seg sg;
    // Whether the ray is still good is asked once for the whole CTA: another segment of the ray may mark it (pbad, at
    // the end of this kernel) while this one starts, and threads that read the mark each for themselves
    // would not agree on going on. Which answer a CTA gets does not matter, since a marked ray's results are not used.
    if (threadIdx.x == 0) {
        s_go = sg.find(p, blockIdx.x, p.above > 0);
        s_bad = 0;
    }
    __syncthreads();
    if (!s_go) return;
    sg.find(p, blockIdx.x, false);
    const int m = a.m, ld = a.ld, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wm = warp & 1, wn = warp >> 1;
    const int bs = factor_buf(m, ld), P = (m + 7) >> 3, mw = m * ld;
    const bool five = p.nbuf == 5;  // a buffer for the next zone's B
    int xo = 0, bo = five ? bs : 0;
    float *const sG = sm + bo + bs, *const sA = sG + bs, *const sL = sA + bs;
    unsigned short *nzr = reinterpret_cast<unsigned short *>(sm + p.nbuf * bs);  // [C_k, A_k][mp]
    float *rowbuf = sm + p.nbuf * bs + a.mp;                                      // [2][8]
    int *cur = reinterpret_cast<int *>(rowbuf + 16);
    int *pos = cur + 8 * P;
    if (tid < m) pos[tid] = tid;
    for (int i = tid; i < p.nbuf * (bs - mw); i += kFactorThreads) sm[i / (bs - mw) * bs + mw + i % (bs - mw)] = 0.f;
    auto load = [&](float *dst, const float *src) { copy_async(dst, src, mw, tid, kFactorThreads); };
    auto load_nz = [&](int to, long long k, int which) {  // the zero pattern of C_k (which 0) or A_k (1)
        copy_async(reinterpret_cast<float *>(nzr + to * a.mp), reinterpret_cast<const float *>(a.nz + ((size_t)k * 2 + which) * a.mp),
                   a.mp / 2, tid, kFactorThreads);
    };
    auto at = [&](float *w, long long k) { return w + (size_t)k * mw; };
    // acc = U V, U's zero pattern in nz (null: none)
    auto rows_times = [&](float (&acc)[NT][NT][4], const float *U, const float *V, const unsigned short *nz) {
#pragma unroll
        for (int x = 0; x < NT; ++x) {
            const int i0 = 16 * (wm * NT + x), i = i0 + (lane & 15), g = lane >> 2;
            const unsigned todo = nz ? __reduce_or_sync(0xffffffffu, i < m ? (unsigned)nz[i] : 0u) : (1u << P) - 1u;
            const int r0 = i0 + g < m ? i0 + g : m - 1, r1 = i0 + g + 8 < m ? i0 + g + 8 : m - 1;
            float d[NT][4];
            product_row<NT>(U, r0 * ld, r1 * ld, V, ld, m, wn, lane, todo, d);
#pragma unroll
            for (int y = 0; y < NT; ++y)
#pragma unroll
                for (int h = 0; h < 4; ++h) acc[y][x][h] = d[y][h];
        }
    };
    float big = 0.f, any = 0.f;  // the largest magnitude of G, L, R and L'; of products with a coupling
    bool finite = true;
    float acc[NT][NT][4];
    load(sm, at(a.Di, sg.za));
    copy_wait();
    __syncthreads();
    for (long long k = sg.za;; ++k) {
        float *const X = sm + xo, *const sB = sm + bo;
        if (k > sg.za) {
            subtract_product<NT>(X, sA, sG, nzr + a.mp, ld, m, wm, wn, lane);
            if (!sg.first) {
                rows_times(acc, sA, sL, nzr + a.mp);
                __syncthreads();
                if (k < sg.ze) store_tiles<NT>(sL, nullptr, acc, -1.f, ld, m, wm, wn, lane, any, finite);
                else store_tiles<NT>(nullptr, at(p.Ar, sg.row), acc, -1.f, ld, m, wm, wn, lane, any, finite);
            }
            __syncthreads();
        }
        if (k == sg.ze) {
            for (int i = 4 * tid; i < mw; i += 4 * kFactorThreads)
                *reinterpret_cast<float4 *>(at(p.Dr, sg.row) + i) = *reinterpret_cast<const float4 *>(X + i);
            break;
        }
        load(sG, at(a.Gt, k));
        load_nz(0, k, 0);
        if (k == sg.za && !sg.first) load(sL, at(a.At, k));
        load(sA, at(a.At, k + 1));
        load_nz(1, k + 1, 1);
        if (five) load(sB, at(a.Di, k + 1));
        if (invert<NT>(X, ld, m, cur, pos, rowbuf, tid) && lane == 0) s_bad = 1;  // (failed, or ill-conditioned)
        copy_wait();
        __syncthreads();
        store_inverse<NT>(at(a.Di, k), X, ld, m, cur, pos, tid);
        inverse_times<NT>(acc, X, sG, nzr, cur, ld, m, wm, wn, lane);
        __syncthreads();
        store_tiles<NT>(sG, at(a.Gt, k), acc, 1.f, ld, m, wm, wn, lane, big, finite);
        if (!sg.first) {
            inverse_times<NT>(acc, X, sL, nullptr, cur, ld, m, wm, wn, lane);
            __syncthreads();
            store_tiles<NT>(sL, at(p.Lt, k), acc, 1.f, ld, m, wm, wn, lane, big, finite);
        }
        if (five) {
            const int t = xo;
            xo = bo;
            bo = t;
        } else {
            load(X, at(a.Di, k + 1));
            copy_wait();
        }
        __syncthreads();
    }
    if (!sg.first) {
        // R and L' back to the segment's first zone, in sG and sL
        for (long long k = sg.ze - 2; k >= sg.za; --k) {
            __syncthreads();
            load(sA, at(a.Gt, k));
            copy_wait();
            __syncthreads();
            rows_times(acc, sA, sG, nullptr);
            __syncthreads();
            store_tiles<NT>(sG, nullptr, acc, -1.f, ld, m, wm, wn, lane, big, finite);
            rows_times(acc, sA, sL, nullptr);
            const int g = lane >> 2, q = lane & 3;
            const float *L = at(p.Lt, k);
#pragma unroll
            for (int x = 0; x < NT; ++x)
#pragma unroll
                for (int y = 0; y < NT; ++y)
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const int i = 16 * (wm * NT + x) + g + 8 * (h >> 1), c = 8 * (wn * NT + y) + 2 * q + (h & 1);
                        if (i < m && c < m) acc[y][x][h] -= L[i * ld + c];
                    }
            __syncthreads();
            store_tiles<NT>(sL, nullptr, acc, -1.f, ld, m, wm, wn, lane, big, finite);
        }
        // the terms of the zone before the segment
        __syncthreads();
        load(sA, at(a.Gt, sg.za - 1));
        load_nz(0, sg.za - 1, 0);
        copy_wait();
        __syncthreads();
        rows_times(acc, sA, sG, nzr);
        store_tiles<NT>(nullptr, at(p.Cr, sg.row - 1), acc, -1.f, ld, m, wm, wn, lane, any, finite);
        rows_times(acc, sA, sL, nzr);
        store_tiles<NT>(nullptr, at(p.Er, sg.row - 1), acc, 1.f, ld, m, wm, wn, lane, any, finite);
    }
    if (!finite || big > kMaxGrowth) s_bad = 1;
    __syncthreads();
    if (tid == 0 && s_bad) atomicOr(p.pbad + blockIdx.x / p.parts, 1);
}

// Br_e's last term, and what k_btd_factor wants of the segments' system besides: zero patterns and arrival counts.
__global__ void __launch_bounds__(256) k_btd_join(const SegArgs p) {
    Seg sg;
    if (!sg.find(p, blockIdx.x, true)) return;
    const BtdArgs &a = p.a;
    const int mw = a.m * a.ld;
    if (!sg.last)
        for (int i = 4 * (256 * blockIdx.y + threadIdx.x); i < mw; i += 4 * 256 * gridDim.y) {  // (the padding is zero in both)
            float4 *d = reinterpret_cast<float4 *>(p.Dr + (size_t)sg.row * mw + i);
            const float4 u = *d, v = *reinterpret_cast<const float4 *>(p.Er + (size_t)sg.row * mw + i);
            *d = make_float4(u.x - v.x, u.y - v.y, u.z - v.z, u.w - v.w);
        }
    if (blockIdx.y) return;
    for (int i = threadIdx.x; i < 2 * a.mp; i += 256) p.nzr[(size_t)sg.row * 2 * a.mp + i] = (unsigned short)((1u << (a.mp / 8)) - 1u);
    if (threadIdx.x == 0) p.zbadr[sg.row] = 0;
}

// The blocks that k_btd_segment has overwritten, again, for the rays that it could not do.
__global__ void __launch_bounds__(256) k_btd_again(const BtdArgs a) {
    long long z0, z1;
    if (!ray_range(a, blockIdx.x, z0, z1)) return;
    const long long mm = (long long)a.m * a.m;
    for (long long e = z0 * mm + blockIdx.y * 256 + threadIdx.x; e < z1 * mm; e += 256 * gridDim.y) {
        const long long row = e / a.m, at = row * a.ld + (e - row * a.m);
        a.Di[at] = (float)a.B[e];
        if (e < (z1 - 1) * mm) a.Gt[at] = (float)a.C[e];
    }
}

// The solve sweep, one CTA of eight warps per ray, or a cluster of two (a.halves) that go along with the two
// halves of the elimination: outwards y_k = D_k^{-1} (rhs_k - A_k y_{k-1}), inwards
// y_k = D_k^{-1} (rhs_k - C_k y_{k+1}), the zone between from both, delta = D^{-1} (rhs - A y - C y), and back
// delta_k = y_k - G_k delta_{k+1} and y_k - H_k delta_{k-1}; x += delta in FP64 (FIRST: x = delta). The halves
// exchange y and delta at the middle through distributed shared memory. Every step is one
// matrix-vector product with an m x m FP32 matrix that is used once, so the matrices of the whole
// sweep run through a ring of nring shared-memory buffers (16-byte cp.async by all threads), and each
// step costs one CTA barrier: eight lanes take a row (128 consecutive bytes per load; rows
// 4 warp + lane / 8 + 32 u, u < NT = ceil(m / 32)), three shuffles finish it, and the row's first lane
// holds its vector entries. What a step needs from the vectors in memory is loaded kAhead zones ahead.
// GB300, m = 84, 400 zones: one ray 1.25 -> 0.55 ms with two CTAs.
constexpr int kSweepThreads = 256;
constexpr int kAhead = 2;
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Stores to the same shared-memory variable of the cluster's CTA `rank`.
__device__ __forceinline__ void store_remote(float *p, int rank, float v) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(r), "f"(v) : "memory");
}
template <bool FIRST, bool LAST, int NT>
__global__ void __launch_bounds__(kSweepThreads, 2) k_btd_sweep(const BtdArgs a) {
    extern __shared__ __align__(16) float sbuf[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gl = lane & 7;
    long long z0, z1;
    const int half = a.halves == 2 ? (int)(blockIdx.x & 1) : 0;  // the rank in the cluster
    if (!ray_range(a, blockIdx.x / a.halves, z0, z1) || z1 == z0) return;
    const int m = a.m, lw = a.ld, nb = a.nring, mw = m * lw;
    float *vin = sbuf + nb * mw;               // [2][VX_BTD_MAX_M] the vector of a step and of the next
    float *vx = vin + 2 * VX_BTD_MAX_M;        // [VX_BTD_MAX_M] from the other half
    if (a.zbad[z0]) {
        if (LAST && half == 0)
            for (long long e = z0 * m + tid; e < z1 * m; e += kSweepThreads) a.x[e] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    const long long mid = z0 + a.zmid[z0];
    const bool both = mid < z1 - 1;  // the ray has an inward half
    if (half == 1 && !both) return;  // (its pair does not wait for it either)
    for (int i = tid; i < 3 * VX_BTD_MAX_M; i += kSweepThreads) vin[i] = 0.f;
    // this half's chain: n zones from kf on in direction dir, then (outward half) the middle zone, then back
    const int dir = half ? -1 : 1, n = (int)(half ? z1 - 1 - mid : mid - z0);
    const long long kf = half ? z1 - 1 : z0;
    const float *pv = half ? a.Gt : a.At, *nx = half ? a.At : a.Gt;  // couplings to the zone before; G or H
    // steps: D^{-1} of the first zone, then coupling and D^{-1} of the later ones; at the middle zone its couplings
    // to either side and D^{-1}; then G (H) from the last zone back
    const int nf = n > 0 ? 2 * n - 1 : 0, nm = half ? 0 : (n > 0) + both + 1, total = nf + nm + n;
    const unsigned sb = (unsigned)__cvta_generic_to_shared(sbuf) + 16u * (unsigned)tid;
    int si = 0, bi = 0;  // the next step to bring in and its buffer
    auto issue = [&]() {
        if (si < total) {
            const float *src;
            if (si < nf) {
                src = ((si & 1) ? pv : a.Di) + (size_t)(kf + dir * ((si + 1) / 2)) * mw;
            } else if (si < nf + nm) {
                const int c = si - nf + (n > 0 ? 0 : 1);  // 0: A, 1: C or D^{-1}, 2: D^{-1}
                src = (c == 0 ? a.At : c == 1 && both ? a.Gt : a.Di) + (size_t)mid * mw;
            } else {
                src = nx + (size_t)(kf + dir * (n - 1 - (si - nf - nm))) * mw;
            }
            src += 4 * tid;
            const unsigned dst = sb + 4u * (unsigned)(bi * mw);
#pragma unroll
            for (int i = 0; i <= NT * NT; ++i)  // 1024 (NT^2 + 1) >= m lw
                if (4 * (tid + kSweepThreads * i) < mw)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * (unsigned)(kSweepThreads * i)),
                                 "l"(src + 4 * kSweepThreads * i)
                                 : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        ++si;
        bi = bi + 1 == nb ? 0 : bi + 1;
    };
    for (int s = 0; s < nb - 1; ++s) issue();
    bool own[NT];  // this lane keeps the row's vector entries
    int row[NT];
#pragma unroll
    for (int u = 0; u < NT; ++u) {
        row[u] = 4 * warp + 32 * u + (lane >> 3);
        own[u] = gl == 0 && row[u] < m;
    }
    double rn[kAhead][NT];  // right-hand sides (on the way to the middle) or x (back) of the next zones
    float yn[kAhead][NT];
    // right-hand side of the chain's i-th zone, the middle one (outward half) the n-th
    const int nr = half ? n : n + 1;
    auto rhs_at = [&](int i, int u) { return own[u] && i < nr ? a.rhs[(kf + (long long)dir * i) * m + row[u]] : 0.0; };
    float t[NT];
#pragma unroll
    for (int u = 0; u < NT; ++u) {
        t[u] = (float)rhs_at(0, u);
#pragma unroll
        for (int h = 0; h < kAhead; ++h) {
            rn[h][u] = rhs_at(h + 1, u);
            yn[h][u] = 0.f;
        }
    }
    if (both) cluster_sync();  // the other CTA has started and cleared its vectors
    __syncthreads();
#pragma unroll
    for (int u = 0; u < NT; ++u)
        if (own[u]) vin[row[u]] = t[u];
    int bs = 0, par = 0;  // the step's buffer and vector
    float p[NT];
    auto step = [&]() {  // p = (the step's matrix) (its vector), in every lane of a row's group
        // all but the newest nb - 2 groups have landed: the step's matrix is in its buffer
        if (nb == 4) asm volatile("cp.async.wait_group 2;" ::: "memory");
        else if (nb == 3) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // ... for every thread; the step before is done with its buffer and its vector
        issue();
        const float *M = sbuf + bs * mw + 4 * gl, *v = vin + VX_BTD_MAX_M * par + 4 * gl;
        float4 x[NT];
#pragma unroll
        for (int c = 0; c < NT; ++c) x[c] = *reinterpret_cast<const float4 *>(v + 32 * c);
#pragma unroll
        for (int u = 0; u < NT; ++u) {
            const float *r = M + min(row[u], m - 1) * lw;
            float e0 = 0.f, e1 = 0.f;
#pragma unroll
            for (int c = 0; c < NT; ++c) {
                float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
                if (c < NT - 1 || 32 * c + 4 * gl < lw) w = *reinterpret_cast<const float4 *>(r + 32 * c);
                e0 = fmaf(w.x, x[c].x, e0);
                e1 = fmaf(w.y, x[c].y, e1);
                e0 = fmaf(w.z, x[c].z, e0);
                e1 = fmaf(w.w, x[c].w, e1);
            }
            p[u] = e0 + e1;
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
#pragma unroll
            for (int u = 0; u < NT; ++u) p[u] += __shfl_xor_sync(0xffffffffu, p[u], o);
        bs = bs + 1 == nb ? 0 : bs + 1;
        par ^= 1;
    };
    auto give = [&](const float (&v)[NT]) {  // the next step's vector
#pragma unroll
        for (int u = 0; u < NT; ++u)
            if (own[u]) vin[VX_BTD_MAX_M * par + row[u]] = v[u];
    };
    static_assert(kAhead == 2, "the vectors' shifts are written out");
    for (int i = 0; i < n; ++i) {  // to the middle
        step();  // p = y_k
        give(p);
        if (i + 1 < n) {
#pragma unroll
            for (int u = 0; u < NT; ++u)
                if (own[u]) a.y[(kf + (long long)dir * i) * m + row[u]] = p[u];
            step();  // p = (coupling) y_k
#pragma unroll
            for (int u = 0; u < NT; ++u) {
                t[u] = (float)rn[0][u] - p[u];
                rn[0][u] = rn[1][u];
                rn[1][u] = rhs_at(i + 3, u);
            }
            give(t);
        }
    }
    float yl[NT];  // y of the chain's last zone
#pragma unroll
    for (int u = 0; u < NT; ++u) {
        yl[u] = p[u];
        if (n > 0) t[u] = (float)rn[0][u];
    }
    if (half == 0) {
        if (n > 0) {
            step();  // A y
#pragma unroll
            for (int u = 0; u < NT; ++u) t[u] -= p[u];
        }
        if (both) {
            cluster_sync();  // the inward half's y has arrived
#pragma unroll
            for (int u = 0; u < NT; ++u) p[u] = own[u] ? vx[row[u]] : 0.f;
            give(p);
            step();  // C y
#pragma unroll
            for (int u = 0; u < NT; ++u) t[u] -= p[u];
        }
        give(t);
        step();  // p = delta of the middle zone
        give(p);
#pragma unroll
        for (int u = 0; u < NT; ++u)
            if (own[u]) {
                if (both) store_remote(vx + row[u], 1, p[u]);
                double *x = a.x + mid * m + row[u];
                *x = FIRST ? (double)p[u] : *x + (double)p[u];
            }
        if (both) cluster_sync();
    } else {
#pragma unroll
        for (int u = 0; u < NT; ++u)
            if (own[u]) store_remote(vx + row[u], 0, yl[u]);
        cluster_sync();
        cluster_sync();  // the middle zone's delta has arrived
#pragma unroll
        for (int u = 0; u < NT; ++u) p[u] = own[u] ? vx[row[u]] : 0.f;
        give(p);
    }
#pragma unroll
    for (int u = 0; u < NT; ++u)
        if (own[u]) {
            yn[0][u] = yl[u];
            yn[1][u] = n > 1 ? a.y[(kf + (long long)dir * (n - 2)) * m + row[u]] : 0.f;
#pragma unroll
            for (int h = 0; h < kAhead; ++h)
                if (!FIRST) rn[h][u] = n > h ? a.x[(kf + (long long)dir * (n - 1 - h)) * m + row[u]] : 0.0;
        }
    for (int i = n - 1; i >= 0; --i) {  // back
        step();  // p = G_k delta_{k+1}
        const long long k = kf + (long long)dir * i;
#pragma unroll
        for (int u = 0; u < NT; ++u)
            if (own[u]) {
                const float dl = yn[0][u] - p[u];
                vin[VX_BTD_MAX_M * par + row[u]] = dl;
                a.x[k * m + row[u]] = FIRST ? (double)dl : rn[0][u] + (double)dl;
                yn[0][u] = yn[1][u];
                yn[1][u] = i > 1 ? a.y[(k - 2 * dir) * m + row[u]] : 0.f;
                if (!FIRST) {
                    rn[0][u] = rn[1][u];
                    rn[1][u] = i > 1 ? a.x[(k - 2 * dir) * m + row[u]] : 0.0;
                }
            }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// The sweeps of rays in segments, a CTA per segment, with the steps and the ring of k_btd_sweep.
// BACK false: y_k outwards, and the right-hand sides of the segments' system (zero before):
// rr_e += rhs_e - A_e y_{e-1}, rr_p -= C_p y'_a, y' = y_k - G_k y'_{k+1} (two terms: their order doesn't matter).
// BACK true: from that system's solution, x_k = y_k - G_k x_{k+1} - L_k x_p inwards; x += (FIRST: =).
// GB300, m = 84, 400 zones, one ray: 0.55 ms by two CTAs -> 0.016 outwards
// and 0.016 inwards for 69 segments, 0.013 + 0.013 for 14 of their last zones, 0.025 for those' last zones.
template <bool BACK, bool FIRST, int NT>
__global__ void __launch_bounds__(kSweepThreads, 1) k_btd_seg_sweep(const SegArgs pa) {
    extern __shared__ __align__(16) float sbuf[];
    const BtdArgs &a = pa.a;
    Seg sg;
    if (!sg.find(pa, blockIdx.x, true)) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gl = lane & 7;
    const int m = a.m, lw = a.ld, nb = a.nring, mw = m * lw;
    float *vin = sbuf + nb * mw;         // [2][VX_BTD_MAX_M] the vector of a step and of the next
    float *vx = vin + 2 * VX_BTD_MAX_M;  // [VX_BTD_MAX_M] x_p
    for (int i = tid; i < 3 * VX_BTD_MAX_M; i += kSweepThreads) vin[i] = 0.f;
    const int n = (int)(sg.ze - sg.za), nf = 2 * n - 1, ns = sg.first ? 1 : 2;
    const int total = n == 0 ? 0 : BACK ? ns * n : nf + 1 + (sg.first ? 0 : n);
    const unsigned sb = (unsigned)__cvta_generic_to_shared(sbuf) + 16u * (unsigned)tid;
    int si = 0, bi = 0;  // the next step to bring in and its buffer
    auto issue = [&]() {
        if (si < total) {
            const float *src;
            if (BACK) src = (ns == 1 || (si & 1) ? a.Gt : pa.Lt) + (size_t)(sg.ze - 1 - si / ns) * mw;
            else if (si <= nf) src = ((si & 1) ? a.At : a.Di) + (size_t)(sg.za + (si + 1) / 2) * mw;  // si = nf: A_e
            else src = a.Gt + (size_t)(sg.ze - 1 - (si - nf)) * mw;                                   // last: C_p
            src += 4 * tid;
            const unsigned dst = sb + 4u * (unsigned)(bi * mw);
#pragma unroll
            for (int i = 0; i <= NT * NT; ++i)  // 1024 (NT^2 + 1) >= m lw
                if (4 * (tid + kSweepThreads * i) < mw)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * (unsigned)(kSweepThreads * i)),
                                 "l"(src + 4 * kSweepThreads * i)
                                 : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        ++si;
        bi = bi + 1 == nb ? 0 : bi + 1;
    };
    for (int s = 0; s < nb - 1; ++s) issue();
    bool own[NT];  // this lane keeps the row's vector entries
    int row[NT];
#pragma unroll
    for (int u = 0; u < NT; ++u) {
        row[u] = 4 * warp + 32 * u + (lane >> 3);
        own[u] = gl == 0 && row[u] < m;
    }
    int bs = 0, par = 0;  // the step's buffer and vector
    float p[NT], q[NT];
    auto step = [&](float (&p)[NT], const float *v) {  // p = (the step's matrix) v, in every lane of a row's group
        if (nb == 4) asm volatile("cp.async.wait_group 2;" ::: "memory");
        else if (nb == 3) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // ... for every thread; the step before is done with its buffer and its vector
        issue();
        const float *M = sbuf + bs * mw + 4 * gl;
        float4 x[NT];
#pragma unroll
        for (int c = 0; c < NT; ++c) x[c] = *reinterpret_cast<const float4 *>(v + 4 * gl + 32 * c);
#pragma unroll
        for (int u = 0; u < NT; ++u) {
            const float *r = M + min(row[u], m - 1) * lw;
            float e0 = 0.f, e1 = 0.f;
#pragma unroll
            for (int c = 0; c < NT; ++c) {
                float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
                if (c < NT - 1 || 32 * c + 4 * gl < lw) w = *reinterpret_cast<const float4 *>(r + 32 * c);
                e0 = fmaf(w.x, x[c].x, e0);
                e1 = fmaf(w.y, x[c].y, e1);
                e0 = fmaf(w.z, x[c].z, e0);
                e1 = fmaf(w.w, x[c].w, e1);
            }
            p[u] = e0 + e1;
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
#pragma unroll
            for (int u = 0; u < NT; ++u) p[u] += __shfl_xor_sync(0xffffffffu, p[u], o);
        bs = bs + 1 == nb ? 0 : bs + 1;
    };
    // the vector of the next step; that step's barrier publishes it, and the one before it has read the other half
    auto give = [&](const float (&v)[NT]) {
        par ^= 1;
#pragma unroll
        for (int u = 0; u < NT; ++u)
            if (own[u]) vin[VX_BTD_MAX_M * par + row[u]] = v[u];
    };
    auto given = [&]() { return (const float *)(vin + VX_BTD_MAX_M * par); };
    double dn[kAhead][NT];  // right-hand sides (BACK: x) of the next zones
    float yn[kAhead][NT], t[NT];
    auto y_at = [&](long long k, int u) { return own[u] && k >= sg.za ? a.y[k * m + row[u]] : 0.f; };
    if (!BACK) {
        auto rhs_at = [&](long long k, int u) { return own[u] && k <= sg.ze ? a.rhs[k * m + row[u]] : 0.0; };
#pragma unroll
        for (int u = 0; u < NT; ++u) {
            t[u] = (float)rhs_at(sg.za, u);
#pragma unroll
            for (int h = 0; h < kAhead; ++h) dn[h][u] = rhs_at(sg.za + 1 + h, u);
        }
        if (n == 0) {
#pragma unroll
            for (int u = 0; u < NT; ++u)
                if (own[u]) atomicAdd(pa.rr + sg.row * m + row[u], (double)t[u]);
            return;
        }
        __syncthreads();
        give(t);
        for (long long k = sg.za; k < sg.ze; ++k) {
            step(p, given());  // y_k
            give(p);
#pragma unroll
            for (int u = 0; u < NT; ++u)
                if (own[u]) a.y[k * m + row[u]] = p[u];
            step(q, given());  // A_{k+1} y_k
#pragma unroll
            for (int u = 0; u < NT; ++u) {
                t[u] = (float)dn[0][u] - q[u];
                dn[0][u] = dn[1][u];
                dn[1][u] = rhs_at(k + 3, u);
            }
            if (k + 1 < sg.ze) give(t);
        }
#pragma unroll
        for (int u = 0; u < NT; ++u)
            if (own[u]) atomicAdd(pa.rr + sg.row * m + row[u], (double)t[u]);
        if (sg.first) return;
#pragma unroll
        for (int u = 0; u < NT; ++u)
#pragma unroll
            for (int h = 0; h < kAhead; ++h) yn[h][u] = y_at(sg.ze - 2 - h, u);
        give(p);
        for (long long k = sg.ze - 2; k >= sg.za; --k) {
            step(q, given());  // G_k y'_{k+1}
#pragma unroll
            for (int u = 0; u < NT; ++u) {
                t[u] = yn[0][u] - q[u];
                yn[0][u] = yn[1][u];
                yn[1][u] = y_at(k - 2, u);
            }
            give(t);
        }
        step(q, given());  // C_p y'_a
#pragma unroll
        for (int u = 0; u < NT; ++u)
            if (own[u]) atomicAdd(pa.rr + (sg.row - 1) * m + row[u], (double)-q[u]);
    } else {
        auto x_at = [&](long long k, int u) { return !FIRST && own[u] && k >= sg.za ? a.x[k * m + row[u]] : 0.0; };
        __syncthreads();
#pragma unroll
        for (int u = 0; u < NT; ++u) {
            const double xe = own[u] ? pa.xr[sg.row * m + row[u]] : 0.0;
            t[u] = (float)xe;
            if (own[u]) {
                if (!sg.first) vx[row[u]] = (float)pa.xr[(sg.row - 1) * m + row[u]];
                double *x = a.x + sg.ze * m + row[u];
                *x = FIRST ? xe : *x + xe;
            }
#pragma unroll
            for (int h = 0; h < kAhead; ++h) {
                yn[h][u] = y_at(sg.ze - 1 - h, u);
                dn[h][u] = x_at(sg.ze - 1 - h, u);
            }
        }
        give(t);
        for (long long k = sg.ze - 1; k >= sg.za; --k) {
#pragma unroll
            for (int u = 0; u < NT; ++u) q[u] = 0.f;
            if (!sg.first) step(q, vx);  // L_k x_p
            step(p, given());            // G_k x_{k+1}
#pragma unroll
            for (int u = 0; u < NT; ++u) {
                t[u] = yn[0][u] - q[u] - p[u];
                if (own[u]) a.x[k * m + row[u]] = FIRST ? (double)t[u] : dn[0][u] + (double)t[u];
                yn[0][u] = yn[1][u];
                dn[0][u] = dn[1][u];
                yn[1][u] = y_at(k - 2, u);
                dn[1][u] = x_at(k - 2, u);
            }
            give(t);
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// The FP64 residual, a ray's zones split over blockIdx.y CTAs, a warp per eight rows of a zone. Every matrix
// element costs one FP64 FMA, at two per clock and SM of GB300 at most (less than HBM can feed), so the layout
// minimises FP64 instructions beyond those FMAs and leaves out what is known to be zero: groups of eight
// columns that are zero in a row of A_k or C_k (nz) are neither read nor multiplied. Lane 4 r + c
// takes row i0 + r and the columns c, c + 4, ... (four lanes read 32 contiguous bytes of a row, eight rows
// per load instruction; in A and C each row goes through its own groups), accumulates with FMAs only, and two
// shuffle-add steps finish the row.
// GB300, m = 84, 304 rays x 400 zones: one coupling per row 5.3 -> 2.2 ms, dense couplings 5.3 -> 5.1 ms (FP64
// pipe: 4.1 at that rate); one ray 0.88 -> 0.02 ms (was four CTAs).
constexpr int kResidB = 7;  // quads of B in flight
constexpr int kResidG = 3;  // column groups of A or C (two loads a lane each) in flight
__device__ __forceinline__ double resid_groups(const double *M, const double *x, unsigned todo, int cc, int m) {
    double s = 0.0;
    while (__any_sync(0xffffffffu, todo)) {
        int j[kResidG];
        double v[kResidG][2];
#pragma unroll
        for (int u = 0; u < kResidG; ++u) {
            j[u] = todo ? 8 * (__ffs(todo) - 1) + cc : m;  // m: none left
            todo &= todo - 1;                              // 0 stays 0
#pragma unroll
            for (int h = 0; h < 2; ++h) v[u][h] = j[u] + 4 * h < m ? M[j[u] + 4 * h] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kResidG; ++u) {
            if (!__any_sync(0xffffffffu, j[u] < m)) break;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (j[u] + 4 * h < m) s = fma(v[u][h], x[j[u] + 4 * h], s);
        }
    }
    return s;
}
__global__ void __launch_bounds__(kResidThreads) k_btd_resid(const BtdArgs a) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = kResidThreads / 32;
    const int rr = lane >> 2, cc = lane & 3;
    long long z0, z1;
    if (!ray_range(a, blockIdx.x, z0, z1) || z1 == z0 || a.zbad[z0]) return;
    const int m = a.m, np = (m + 7) >> 3;
    const long long units = (z1 - z0) * np;
    float big = 0.f, size = 0.f;  // max|r|, max|d| of this lane's rows
    for (long long q = units * blockIdx.y / gridDim.y + warp, qe = units * (blockIdx.y + 1) / gridDim.y; q < qe; q += nw) {
        const long long k = z0 + q / np;
        const int i0 = 8 * (int)(q % np);
        const int i = i0 + rr < m ? i0 + rr : m - 1;  // rows past the end repeat the last one
        const size_t ro = ((size_t)k * m + i) * m;
        const unsigned nc = k + 1 < z1 ? a.nz[(size_t)k * 2 * a.mp + i] : 0u, na = k > z0 ? a.nz[((size_t)k * 2 + 1) * a.mp + i] : 0u;
        const double *B = a.B + ro, *x0 = a.x + k * m;
        double s = 0.0;
        for (int j0 = cc; j0 < m; j0 += 4 * kResidB) {
            double v[kResidB];
#pragma unroll
            for (int u = 0; u < kResidB; ++u) v[u] = j0 + 4 * u < m ? B[j0 + 4 * u] : 0.0;
#pragma unroll
            for (int u = 0; u < kResidB; ++u)
                if (j0 + 4 * u < m) s = fma(v[u], x0[j0 + 4 * u], s);
        }
        s += resid_groups(a.A + ro, x0 - m, na, cc, m);
        s += resid_groups(a.C + ro, x0 + m, nc, cc, m);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (cc == 0 && i0 + rr < m) {
            const double d = a.d[k * m + i];
            a.r[k * m + i] = d - s;
            if (a.norm) {
                big = fmaxf(big, fabs(d - s) <= 1e300 ? (float)fabs(d - s) : INFINITY);  // (NaN counts as infinite)
                size = fmaxf(size, (float)fabs(d));
            }
        }
    }
    if (a.norm) {
        atomicMax(a.znorm + 2 * z0, __float_as_uint(big));
        atomicMax(a.znorm + 2 * z0 + 1, __float_as_uint(size));
    }
}

// Rays with ill-conditioned blocks that the sweeps do not settle (kSlowest), all in FP64: a CTA of eight warps per ray,
// block elimination from the first zone on. D_k is eliminated in shared memory by Gauss-Jordan steps with partial
// pivoting, its columns replaced by the multipliers; these are then done over on [C_k, d_k - A_k y_{k-1}], `cols`
// columns at a time, which leaves G_k and y_k (an inverse would square the block's condition number in the error; so
// would the multipliers in FP32, 0.5 ms a zone, in some rays). G_k is kept as the two words of its doubles in the places
// of G_k and A_k, y_k in x. Bound by the FP64 pipe and the steps' barriers (2.5 m^3 FMAs a zone; 0.85 ms at m = 84):
// for the few rays that need it.
constexpr int kExactThreads = 256;
constexpr size_t exact_smem(int m, int cols) {
    return ((size_t)m * m + (size_t)m * cols + m) * sizeof(double) + (size_t)m * sizeof(int);
}
__global__ void __launch_bounds__(kExactThreads) k_btd_fp64(const BtdArgs a, int cols, float enough) {
    extern __shared__ __align__(16) double W[];  // [m][m]; V: [m][cols]; t: [m]; the pivots' rows
    __shared__ double s_best[kExactThreads / 32];
    __shared__ int s_row[kExactThreads / 32], s_bad;
    long long z0, z1;
    if (!ray_range(a, blockIdx.x, z0, z1) || a.zbad[z0]) return;
    if (__uint_as_float(a.znorm[2 * z0]) <= enough * __uint_as_float(a.znorm[2 * z0 + 1])) return;
    const int m = a.m, ld = a.ld, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double *V = W + m * m, *t = V + m * cols;
    int *cur = reinterpret_cast<int *>(t + m);
    int *const G1 = reinterpret_cast<int *>(a.Gt), *const G0 = reinterpret_cast<int *>(a.At);  // high and low words
    auto G = [&](long long k, int i, int j) {
        const size_t e = ((size_t)k * m + i) * ld + j;
        return __hiloint2double(G1[e], G0[e]);
    };
    if (tid == 0) s_bad = 0;
    for (long long k = z0; k < z1; ++k) {
        const double *A = a.A + (size_t)k * m * m, *B = a.B + (size_t)k * m * m, *C = a.C + (size_t)k * m * m;
        for (int e = tid; e < m * m; e += kExactThreads) {
            const int i = e / m, j = e - i * m;
            double v = B[e];
            if (k > z0)
                for (int q = 0; q < m; ++q) v = fma(-A[i * m + q], G(k - 1, q, j), v);
            W[e] = v;
        }
        for (int i = tid; i < m; i += kExactThreads) {
            double v = a.d[k * m + i];
            if (k > z0)
                for (int q = 0; q < m; ++q) v = fma(-A[i * m + q], a.x[(k - 1) * m + q], v);
            t[i] = v;
        }
        bool used = false;  // row tid has been a pivot
        for (int j = 0; j < m; ++j) {
            __syncthreads();
            double best = tid < m && !used ? fabs(W[tid * m + j]) : -1.0;  // (m <= kExactThreads)
            int row = tid;
            for (int o = 16; o > 0; o >>= 1) {
                const double b = __shfl_down_sync(0xffffffffu, best, o);
                const int r = __shfl_down_sync(0xffffffffu, row, o);
                if (b > best) {
                    best = b;
                    row = r;
                }
            }
            if (lane == 0) {
                s_best[warp] = best;
                s_row[warp] = row;
            }
            __syncthreads();
            best = s_best[0];
            row = s_row[0];
            for (int w = 1; w < kExactThreads / 32; ++w)
                if (s_best[w] > best) {
                    best = s_best[w];
                    row = s_row[w];
                }
            row = row < m ? row : m - 1;
            const double p = W[row * m + j];
            if (tid == 0) {
                cur[j] = row;
                if (!(fabs(p) > 0.0 && fabs(p) < INFINITY)) s_bad = 1;
            }
            if (tid == row) used = true;
            __syncthreads();  // (everyone has the pivot)
            if (tid < m && tid != row) W[tid * m + j] = -W[tid * m + j] / p;
            __syncthreads();
            const int n = m - 1 - j;
            for (int e = tid; e < m * n; e += kExactThreads) {
                const int i = e / n, c = j + 1 + e - i * n;
                if (i != row) W[i * m + c] = fma(W[i * m + j], W[row * m + c], W[i * m + c]);
            }
        }
        __syncthreads();
        for (int c0 = k + 1 < z1 ? 0 : m; c0 <= m; c0 += cols) {  // columns of [C, t]
            const int n = min(cols, m + 1 - c0);
            for (int e = tid; e < m * n; e += kExactThreads) {
                const int i = e / n, c = e - i * n;
                V[e] = c0 + c < m ? C[i * m + c0 + c] : t[i];
            }
            for (int j = 0; j < m; ++j) {
                __syncthreads();
                const int row = cur[j];
                for (int e = tid; e < m * n; e += kExactThreads) {
                    const int i = e / n, c = e - i * n;
                    if (i != row) V[e] = fma(W[i * m + j], V[row * n + c], V[e]);
                }
            }
            __syncthreads();
            for (int e = tid; e < m * n; e += kExactThreads) {
                const int j = e / n, c = e - j * n;
                const double v = V[cur[j] * n + c] / W[cur[j] * m + j];
                if (c0 + c < m) {
                    const size_t g = ((size_t)k * m + j) * ld + c0 + c;
                    G1[g] = __double2hiint(v);
                    G0[g] = __double2loint(v);
                } else {
                    a.x[k * m + j] = v;
                }
            }
            __syncthreads();
        }
    }
    for (long long k = z1 - 2; k >= z0; --k) {
        for (int j = warp; j < m; j += kExactThreads / 32) {
            double v = 0.0;
            for (int q = lane; q < m; q += 32) v = fma(G(k, j, q), a.x[(k + 1) * m + q], v);
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) a.x[k * m + j] -= v;
        }
        __syncthreads();
    }
    if (!s_bad) return;
    for (long long e = z0 * m + tid; e < z1 * m; e += kExactThreads) a.x[e] = __longlong_as_double(0x7ff8000000000000ll);
    if (tid == 0) atomicOr(a.flag, 2);
}

}  // namespace

// The factor kernel for NT = ceil(m / 32) row slots per lane.
static const void *factor_kernel(int m) {
    if (m <= 32) return (const void *)k_btd_factor<1>;
    if (m <= 64) return (const void *)k_btd_factor<2>;
    if (m <= 96) return (const void *)k_btd_factor<3>;
    return (const void *)k_btd_factor<4>;
}
static void launch_factor(int m, int grid, size_t smem, cudaStream_t s, const BtdArgs &a) {
    if (m <= 32) k_btd_factor<1><<<grid, kFactorThreads, smem, s>>>(a);
    else if (m <= 64) k_btd_factor<2><<<grid, kFactorThreads, smem, s>>>(a);
    else if (m <= 96) k_btd_factor<3><<<grid, kFactorThreads, smem, s>>>(a);
    else k_btd_factor<4><<<grid, kFactorThreads, smem, s>>>(a);
}
static void launch_convert(int m, long long zones, int sms, cudaStream_t s, const BtdArgs &a) {
    const int grid = (int)(3 * zones < kConvGrid * sms ? 3 * zones : kConvGrid * sms);
    if (m <= 32) k_btd_convert<1><<<grid, kConvThreads, 0, s>>>(a);
    else if (m <= 64) k_btd_convert<2><<<grid, kConvThreads, 0, s>>>(a);
    else if (m <= 96) k_btd_convert<3><<<grid, kConvThreads, 0, s>>>(a);
    else k_btd_convert<4><<<grid, kConvThreads, 0, s>>>(a);
}
template <bool F, bool L>
static const void *sweep_kernel(int m) {
    if (m <= 32) return (const void *)k_btd_sweep<F, L, 1>;
    if (m <= 64) return (const void *)k_btd_sweep<F, L, 2>;
    if (m <= 96) return (const void *)k_btd_sweep<F, L, 3>;
    return (const void *)k_btd_sweep<F, L, 4>;
}
template <bool F, bool L>
static cudaError_t launch_sweep(int m, int grid, size_t smem, cudaStream_t s, const BtdArgs &a) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kSweepThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)a.halves;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (m <= 32) return cudaLaunchKernelEx(&cfg, k_btd_sweep<F, L, 1>, a);
    if (m <= 64) return cudaLaunchKernelEx(&cfg, k_btd_sweep<F, L, 2>, a);
    if (m <= 96) return cudaLaunchKernelEx(&cfg, k_btd_sweep<F, L, 3>, a);
    return cudaLaunchKernelEx(&cfg, k_btd_sweep<F, L, 4>, a);
}

template <bool BACK, bool FIRST>
static const void *seg_sweep_kernel(int m) {
    if (m <= 32) return (const void *)k_btd_seg_sweep<BACK, FIRST, 1>;
    if (m <= 64) return (const void *)k_btd_seg_sweep<BACK, FIRST, 2>;
    if (m <= 96) return (const void *)k_btd_seg_sweep<BACK, FIRST, 3>;
    return (const void *)k_btd_seg_sweep<BACK, FIRST, 4>;
}
static const void *segment_kernel(int m) {
    if (m <= 32) return (const void *)k_btd_segment<1>;
    if (m <= 64) return (const void *)k_btd_segment<2>;
    if (m <= 96) return (const void *)k_btd_segment<3>;
    return (const void *)k_btd_segment<4>;
}
static cudaError_t launch_seg(const void *kernel, int grid, size_t smem, cudaStream_t s, SegArgs &p) {
    void *args[1] = {&p};
    return cudaLaunchKernel(kernel, dim3((unsigned)grid), dim3(kFactorThreads), args, smem, s);
}

// Shared memory that lets two CTAs share an SM (228 KB, 1 KB of it reserved per CTA), and one CTA's limit.
constexpr size_t kSmemHalf = 113 * 1024 - 64, kSmemFull = 226 * 1024;

// Zones from which on segments are laid out, and for which they have room.
constexpr long long kSegMinZones = 40, kSegMaxZones = 16384, kSegTwoLevels = 150;
constexpr int kSegMinParts = 5;  // fewest segments of a ray

struct vx_btd {
    int m = 0, ld = 0, mp = 0, nbuf = 3, nring = 2, n_refine = 0;
    long long max_zones = 0;
    size_t smem = 0, smem_sweep = 0;
    // Room for blocks * m * ld floats: a call lays B, C and A of its zones there, one array after the other, and
    // then L, if it cuts rays into segments and a quarter of the room holds its zones. A handle of 21,845 zones or more
    // has that for the 16,384 zones that segments go to at most; for smaller ones the room is larger by up to a third.
    float *blk = nullptr, *y = nullptr;
    size_t blocks = 0;
    unsigned short *nz = nullptr;
    int slots = 0;  // factor CTAs the device holds at once
    unsigned *znorm = nullptr;
    int *zbad = nullptr, *zmid = nullptr, *zill = nullptr, *flag = nullptr;  // flag[0]: numeric flag, flag[1]: offsets invalid
    double *r = nullptr;
    // segments: most zones of a call that is cut into them (0: none), and their system's arrays (a row per SM)
    int sms = 1, seg_nbuf = 0;
    long long seg_zones = 0;
    size_t smem_seg = 0;
    float *Sr = nullptr;  // per level, the system's four blocks per row; then L of its rows, then the levels' y
    unsigned short *nzr = nullptr;       // per level
    int *zr = nullptr;                   // per level zbad, zmid of that system; pbad
    double *vr = nullptr;                // right-hand sides of both levels' systems, then the solutions
};

static void btd_free(vx_btd *h) {
    if (!h) return;
    cudaFree(h->blk);
    cudaFree(h->nz);
    cudaFree(h->y);
    cudaFree(h->zbad);
    cudaFree(h->zmid);
    cudaFree(h->zill);
    cudaFree(h->znorm);
    cudaFree(h->Sr);
    cudaFree(h->nzr);
    cudaFree(h->zr);
    cudaFree(h->vr);
    cudaFree(h->flag);
    cudaFree(h->r);
    delete h;
}

extern "C" vx_status vx_btd_create(int m, long long max_zones, int n_refine, vx_btd **out) {
    return vx_btd_create_rays(m, max_zones, n_refine, 1, out);
}

extern "C" vx_status vx_btd_create_rays(int m, long long max_zones, int n_refine, int min_rays, vx_btd **out) {
    if (!out) return bfail(VX_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (m < 1 || m > VX_BTD_MAX_M) return bfail(VX_ERR_INVALID_ARG, "m = %d outside 1..%d", m, VX_BTD_MAX_M);
    if (max_zones < 0) return bfail(VX_ERR_INVALID_ARG, "max_zones = %lld < 0", max_zones);
    if (n_refine < 0 || n_refine > VX_BTD_MAX_REFINE)
        return bfail(VX_ERR_INVALID_ARG, "n_refine = %d outside 0..%d", n_refine, VX_BTD_MAX_REFINE);
    if (min_rays < 1) return bfail(VX_ERR_INVALID_ARG, "min_rays = %d < 1", min_rays);
    vx_btd *h = new (std::nothrow) vx_btd;
    if (!h) return bfail(VX_ERR_OOM, "host allocation failed");
    h->m = m;
    h->ld = row_stride(m);
    h->mp = (m + 7) & ~7;
    h->n_refine = n_refine;
    h->max_zones = max_zones;
    // a fourth buffer (the next zone's B) where it costs no second CTA per SM: m <= 84, and from 97 on
    // where one CTA fills an SM with three as well
    const size_t s3 = factor_smem(m, h->ld, 3), s4 = factor_smem(m, h->ld, 4);
    h->nbuf = s4 <= kSmemHalf || (s3 > kSmemHalf && s4 <= kSmemFull) ? 4 : 3;
    h->smem = h->nbuf == 4 ? s4 : s3;
    const size_t mw = (size_t)m * h->ld;
    auto ring = [&](int nb) { return (nb * mw + 3 * VX_BTD_MAX_M) * sizeof(float); };
    h->nring = ring(4) <= kSmemHalf ? 4 : ring(3) <= kSmemFull ? 3 : 2;
    h->smem_sweep = ring(h->nring);
    const size_t zc = (size_t)(max_zones > 0 ? max_zones : 1);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, dev);
    // segments where their four or five buffers fit; without the memory for them, rays go as a whole
    h->seg_nbuf = factor_smem(m, h->ld, 5) <= kSmemFull ? 5 : factor_smem(m, h->ld, 4) <= kSmemFull ? 4 : 0;
    bool seg = h->seg_nbuf && max_zones >= kSegMinZones && min_rays <= h->sms / kSegMinParts;
    h->blocks = 3 * zc;
    if (e == cudaSuccess && seg) {
        const size_t rows = (size_t)h->sms;
        h->seg_zones = max_zones < kSegMaxZones ? max_zones : kSegMaxZones;
        h->smem_seg = factor_smem(m, h->ld, h->seg_nbuf);
        if (4 * (size_t)h->seg_zones > h->blocks) h->blocks = 4 * (size_t)h->seg_zones;
        cudaError_t q = cudaMalloc(&h->blk, h->blocks * mw * sizeof(float));
        if (q == cudaSuccess) q = cudaMalloc(&h->Sr, rows * (9 * mw + 2 * m) * sizeof(float));
        if (q == cudaSuccess) q = cudaMalloc(&h->nzr, 2 * rows * 2 * h->mp * sizeof(unsigned short));
        if (q == cudaSuccess) q = cudaMalloc(&h->zr, 5 * rows * sizeof(int));
        if (q == cudaSuccess) q = cudaMalloc(&h->vr, 4 * rows * m * sizeof(double));
        if (q == cudaSuccess) {
            if (h->ld != m) e = cudaMemset(h->Sr, 0, rows * (9 * mw + 2 * m) * sizeof(float));
            const void *ks[4] = {segment_kernel(m), seg_sweep_kernel<false, true>(m), seg_sweep_kernel<true, true>(m),
                                 seg_sweep_kernel<true, false>(m)};
            for (int i = 0; i < 4 && e == cudaSuccess; ++i)
                e = cudaFuncSetAttribute(ks[i], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemFull);
        } else {
            h->seg_zones = 0;
            if (q == cudaErrorMemoryAllocation) (void)cudaGetLastError();
            else e = q;
            if (h->blocks > 3 * zc) {
                cudaFree(h->blk);
                h->blk = nullptr;
                h->blocks = 3 * zc;
            }
        }
    }
    if (e == cudaSuccess && !h->blk) e = cudaMalloc(&h->blk, h->blocks * mw * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&h->nz, zc * 2 * h->mp * sizeof(unsigned short));
    if (e == cudaSuccess) e = cudaMalloc(&h->y, zc * m * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&h->zbad, zc * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&h->zmid, zc * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&h->zill, zc * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&h->znorm, zc * 2 * sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMalloc(&h->r, zc * m * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&h->flag, 2 * sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(h->flag, 0, 2 * sizeof(int));
    h->slots = h->sms * (h->smem <= kSmemHalf && m <= 96 ? 2 : 1);
    if (h->ld != m && e == cudaSuccess)  // the columns that pad a row are read by the sweeps and never written
        e = cudaMemset(h->blk, 0, h->blocks * mw * sizeof(float));
    // the kernels' limit, not this handle's size: handles of several m share them
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(factor_kernel(m), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemFull);
    const void *sweeps[4] = {sweep_kernel<true, true>(m), sweep_kernel<true, false>(m), sweep_kernel<false, true>(m),
                             sweep_kernel<false, false>(m)};
    for (int i = 0; i < 4 && e == cudaSuccess; ++i)
        e = cudaFuncSetAttribute(sweeps[i], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemFull);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void *)k_btd_fp64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemFull);
    if (e != cudaSuccess) {
        btd_free(h);
        return bfail(e == cudaErrorMemoryAllocation ? VX_ERR_OOM : VX_ERR_CUDA, "vx_btd_create: %s",
                     cudaGetErrorString(e));
    }
    *out = h;
    return VX_OK;
}

extern "C" vx_status vx_btd_solve(vx_btd *h, int n_rays, long long n_zones, const int *ray_offsets, const double *A,
                                  const double *B, const double *C, const double *d, double *x, vx_stream stream) {
    if (!h) return bfail(VX_ERR_INVALID_ARG, "handle is NULL");
    if (n_rays < 0) return bfail(VX_ERR_INVALID_ARG, "n_rays = %d < 0", n_rays);
    if (n_zones < 0 || n_zones > h->max_zones)
        return bfail(VX_ERR_INVALID_ARG, "n_zones = %lld outside 0..%lld", n_zones, h->max_zones);
    if (n_zones > 0 && n_rays == 0) return bfail(VX_ERR_INVALID_ARG, "n_zones > 0 with no rays");
    if (n_zones == 0) return VX_OK;
    if (!ray_offsets || !A || !B || !C || !d || !x) return bfail(VX_ERR_INVALID_ARG, "NULL array");
    {
        vx_status st;
        const void *arr[6] = {ray_offsets, A, B, C, d, x};
        const char *nm[6] = {"ray_offsets", "A", "B", "C", "d", "x"};
        for (int k = 0; k < 6; ++k)
            if ((st = device_array(arr[k], k ? 8 : 4, nm[k])) != VX_OK) return st;
    }
    const size_t vec = (size_t)n_zones * h->m * sizeof(double), blk = vec * h->m;
    auto overlap = [](const void *p, size_t np, const void *q, size_t nq) {
        const char *a = (const char *)p, *b = (const char *)q;
        return a < b + nq && b < a + np;
    };
    if (overlap(x, vec, d, vec) || overlap(x, vec, A, blk) || overlap(x, vec, B, blk) || overlap(x, vec, C, blk))
        return bfail(VX_ERR_INVALID_ARG, "x overlaps an input");
    cudaStream_t s = (cudaStream_t)stream;
    BtdArgs a;
    a.m = h->m;
    a.ld = h->ld;
    a.mp = h->mp;
    a.nbuf = h->nbuf;
    a.nring = h->nring;
    a.n_rays = n_rays;
    a.n_zones = n_zones;
    a.off = ray_offsets;
    a.A = A;
    a.B = B;
    a.C = C;
    a.d = d;
    a.rhs = d;
    a.x = x;
    a.r = h->r;
    const size_t arr = (size_t)n_zones * h->m * h->ld;
    a.Di = h->blk;
    a.Gt = a.Di + arr;
    a.At = a.Gt + arr;
    a.nz = h->nz;
    a.y = h->y;
    a.zbad = h->zbad;
    a.zmid = h->zmid;
    a.zill = h->zill;
    a.min_ill = 0;
    a.znorm = h->znorm;
    a.norm = false;
    // Two CTAs per ray while they all find room at once, and with rays of 16 zones or more where the last wave of
    // one CTA per ray would be less than 5/8 full. GB300, one -> two, 100 zones: m = 84, 20 rays 3.60 -> 1.98 ms,
    // 152 4.76 -> 3.73, 160 5.91 -> 5.32, 330 10.58 -> 9.02, 480 13.25 -> 12.54, but 240 6.67 -> 6.70 and
    // 304 (all slots) 7.33 -> 7.41; m = 120 (40 zones), 200 rays 8.50 -> 7.12, 110 4.40 -> 4.46; rays of
    // 4 to 8 zones, 2000 of them, 3.04 -> 3.18.
    const int rest = n_rays % h->slots;
    a.halves = 2 * n_rays <= h->slots ||
                       (n_rays < 4 * h->slots && n_zones >= 16ll * n_rays && rest > 0 && 8 * rest <= 5 * h->slots)
                   ? 2
                   : 1;
    a.flag = h->flag;
    a.inval = h->flag + 1;
    a.parts = a.above = 0;
    a.pbad = nullptr;
    // Segments per ray: one per SM at most, and S^2 <= 3 n, about as many as make n / S zones with their extra
    // products and S / 2 zones of the segments' system take least (S^2 = 2 n and 5 n: 4 to 12 % slower at 100
    // zones). GB300, m = 84, by halves -> in segments: 1 ray of 400 zones 6.65 -> 1.61 ms, 8 rays 7.12 ->
    // 2.24, 30 rays (5 segments) 8.03 -> 6.66, 38 rays (4 segments) 8.18 -> 8.12; of 100 zones, 1 ray
    // 1.74 -> 0.82, 30 rays 2.09 -> 1.83, 38 rays 2.13 -> 2.19; of 32 zones, 8 rays 0.63 -> 0.54 but 30 rays
    // 0.74 -> 0.76 and with m = 16 0.18 -> 0.19; of 24 zones 0.50 -> 0.49.
    const long long mean = n_zones / n_rays;
    const int most_parts = n_rays < h->sms ? h->sms / n_rays : 0;
    int parts = most_parts, top = 0;
    while (parts > kSegMinParts && (long long)parts * parts > 3 * mean) --parts;
    const bool seg = parts >= kSegMinParts && mean >= kSegMinZones && n_zones <= h->seg_zones;
    // Two levels where there is room for more: S^1.5 <= 1.45 n segments of the ray, and 1.75 S^0.5 of their system
    // (at 48, 58 and 38 us a zone of either level and of the last system, that takes least).
    // GB300, m = 84, one level -> two: 1 ray of 100 zones 0.82 -> 0.82 ms, 150 1.03 -> 0.86, 400 1.61 -> 1.16, 1000
    // 2.60 -> 1.64; 4 rays of 150 1.10 -> 0.95, 400 1.78 -> 1.52; m = 8, 100 zones 0.22 -> 0.23, 400 0.32 -> 0.28.
    if (seg && mean >= kSegTwoLevels && most_parts >= 32) {
        parts = most_parts;
        while (4.0 * parts * parts * parts > 8.4 * (double)mean * (double)mean) --parts;
        top = parts;
        while (16ll * top * top > 49ll * parts) --top;
    }
    const int levels = top > 0 ? 2 : 1;
    SegArgs p[2];   // the segments
    BtdArgs b;      // the last level's system
    BtdArgs f = a;  // the rays whose elimination by segments failed
    if (seg) {
        const size_t rows = (size_t)h->sms, mw = (size_t)h->m * h->ld, vec32 = rows * h->m;
        f.pbad = h->zr + 4 * rows;
        b = f;
        b.A = b.B = b.C = nullptr;
        b.halves = 2;
        for (int l = 0; l < levels; ++l) {
            SegArgs &q = p[l];
            q.a = l ? b : a;
            q.parts = l ? top : parts;
            q.above = l ? parts : 0;
            q.nbuf = h->seg_nbuf;
            q.Lt = l ? h->Sr + rows * 8 * mw : a.At + arr;
            q.Dr = h->Sr + l * rows * 4 * mw;
            q.Cr = q.Dr + rows * mw;
            q.Ar = q.Cr + rows * mw;
            q.Er = q.Ar + rows * mw;
            q.nzr = h->nzr + l * rows * 2 * h->mp;
            q.zbadr = h->zr + l * 2 * rows;
            q.pbad = f.pbad;
            q.rr = h->vr + l * vec32;
            q.xr = h->vr + (2 + l) * vec32;
            b.parts = q.parts;
            b.above = q.above;
            b.Di = q.Dr;
            b.Gt = q.Cr;
            b.At = q.Ar;
            b.y = h->Sr + rows * 9 * mw + l * vec32;
            b.nz = q.nzr;
            b.zbad = q.zbadr;
            b.zmid = q.zbadr + rows;
            b.rhs = q.rr;
            b.x = q.xr;
        }
    }
    BTD_CU(cudaMemsetAsync(h->flag + 1, 0, sizeof(int), s));
    BTD_CU(cudaMemsetAsync(h->zmid, 0, (size_t)n_zones * sizeof(int), s));
    k_btd_validate<<<(unsigned)((n_rays + 256) / 256), 256, 0, s>>>(ray_offsets, n_rays, n_zones, h->flag + 1, h->flag, h->zbad,
                                                                   h->zill, h->znorm, h->zmid, f.pbad);
    BTD_CU(cudaGetLastError());
    launch_convert(h->m, n_zones, h->sms, s, a);
    BTD_CU(cudaGetLastError());
    if (seg) {
        for (int l = 0; l < levels; ++l) {
            BTD_CU(launch_seg(segment_kernel(h->m), n_rays * p[l].parts, h->smem_seg, s, p[l]));
            k_btd_join<<<dim3(n_rays * p[l].parts, 4), 256, 0, s>>>(p[l]);
            BTD_CU(cudaGetLastError());
        }
        launch_factor(h->m, 2 * n_rays, h->smem, s, b);
        BTD_CU(cudaGetLastError());
        k_btd_again<<<dim3(n_rays, 32), 256, 0, s>>>(f);
        BTD_CU(cudaGetLastError());
    }
    const int ctas = a.halves * n_rays;
    launch_factor(h->m, ctas, h->smem, s, f);
    BTD_CU(cudaGetLastError());
    // CTAs per ray of the residual: enough to fill the chip with few rays, at most one per eight units (row octets)
    const long long units = n_zones * ((h->m + 7) / 8);
    long long split = (8ll * h->sms + n_rays - 1) / n_rays, most = (units + 8 * n_rays - 1) / (8 * (long long)n_rays);
    split = split > most ? most : split;
    split = split < 16 ? 16 : split;
    for (int it = 0; it <= h->n_refine; ++it) {
        if (it > 0) {
            k_btd_resid<<<dim3(n_rays, (unsigned)split), kResidThreads, 0, s>>>(a);
            BTD_CU(cudaGetLastError());
            f.rhs = p[0].a.rhs = h->r;
        }
        const bool last = it == h->n_refine;
        if (seg) {
            BTD_CU(cudaMemsetAsync(h->vr, 0, (size_t)levels * h->sms * h->m * sizeof(double), s));
            for (int l = 0; l < levels; ++l)
                BTD_CU(launch_seg(seg_sweep_kernel<false, true>(h->m), n_rays * p[l].parts, h->smem_sweep, s, p[l]));
            BTD_CU((launch_sweep<true, false>(h->m, 2 * n_rays, h->smem_sweep, s, b)));
            for (int l = levels - 1; l >= 0; --l)
                BTD_CU(launch_seg(l || it == 0 ? seg_sweep_kernel<true, true>(h->m) : seg_sweep_kernel<true, false>(h->m),
                                  n_rays * p[l].parts, h->smem_sweep, s, p[l]));
        }
        BTD_CU((it == 0 ? (last ? launch_sweep<true, true> : launch_sweep<true, false>)
                        : (last ? launch_sweep<false, true> : launch_sweep<false, false>))(h->m, ctas, h->smem_sweep, s, f));
    }
    f.rhs = h->r;
    for (int level = 1; level <= 2; ++level) {  // rays with ill-conditioned blocks (never those in segments)
        a.min_ill = f.min_ill = level;
        k_btd_resid<<<dim3(n_rays, (unsigned)split), kResidThreads, 0, s>>>(a);
        BTD_CU(cudaGetLastError());
        BTD_CU((launch_sweep<false, false>(h->m, ctas, h->smem_sweep, s, f)));
    }
    a.min_ill = 1;
    a.norm = true;
    k_btd_resid<<<dim3(n_rays, (unsigned)split), kResidThreads, 0, s>>>(a);
    BTD_CU(cudaGetLastError());
    int cols = h->m + 1;
    while (exact_smem(h->m, cols) > kSmemFull) --cols;
    k_btd_fp64<<<n_rays, kExactThreads, exact_smem(h->m, cols), s>>>(
        a, cols, fmaxf(powf(kSlowest, (float)h->n_refine + 2.f), 1e-10f));
    BTD_CU(cudaGetLastError());
    return VX_OK;
}

extern "C" vx_status vx_btd_check(vx_btd *h, vx_stream stream) {
    if (!h) return bfail(VX_ERR_INVALID_ARG, "handle is NULL");
    BTD_CU(cudaStreamSynchronize((cudaStream_t)stream));
    int f = 0;
    BTD_CU(cudaMemcpy(&f, h->flag, sizeof(int), cudaMemcpyDeviceToHost));
    if (f) {
        BTD_CU(cudaMemset(h->flag, 0, sizeof(int)));
        return bfail(VX_ERR_NUMERIC, "block-tridiagonal solve: %s%s", (f & 2) ? "zero or non-finite pivot" : "",
                     (f & 1) ? ((f & 2) ? "; invalid ray offsets" : "invalid ray offsets") : "");
    }
    return VX_OK;
}

extern "C" void vx_btd_destroy(vx_btd *h) { btd_free(h); }
