// vx_fp64.cu -- FP64 form of the pair-process kernel (forward only).
//
// The same discrete rule as the mixed form and the same exact rewrite of the azimuth-averaged matrix
// element into three non-negative moments, at FP64 accuracy throughout. Production is e^{-eps_i/T} e^{-eps_j/T}
// times annihilation, as FP64 products that underflow where the definition itself underflows.
//
// Bound by the FP64 pipe, two lanes wide on an SM of GB300 (a probe of FMAs gets 1.68 per clock, this kernel 1.85) against
// 128 FP32 or 64 integer ones, so the node loop is written for the fewest FP64 operations and leaves the rest to the
// other pipes. With d = h/T (h = |q|/2) a mirror pair of nodes tau, -tau has
//   e1(+-tau) = c1 2^-+t,  e2(+-tau) = c2 2^+-t,  t = d tau log2 e,
//   c1 = e^{eta - q0/2T},  c2 = e^{-eta - q0/2T},  (1 + e1)(1 + e2) = 1 + e^{-q0/T} + e1 + e2,
// so one reduced argument serves both nodes and both leptons, and one reciprocal (of the product of the two
// denominators: MUFU start and one cubic Newton step, half an ulp and a little) both blocking factors. 2^+-t come
// from a table of 2^{j/4096} and a polynomial in the remainder r/4096, |r| <= 1/2: its linear term in FP64, the
// quadratic one (up to 3.6e-9) from a 32-bit integer square in units of 2^-59, the rest (up to 2e-13, so that
// FP32's rounding of it is below 1e-20) in FP32, added in the same units. 2^t is within 2.2e-16 (the table's rounding and
// the last one), rms 6.7e-17; with the quadratic term in FP32 it was 6.5e-16, rms 1.1e-16. 23 FP64 operations
// per mirror pair against 84 with two library exponentials and a division per node. The arguments' rounding errors
// (of 1/T, and of d) are carried along as small corrections, so e1 and e2 are good to a few units in the last
// place at any |t|, where a rounded argument loses |t| of them. Zones so cold that 2^+-t would leave
// the FP64 range (q0/2T + |eta| above 690) take the plain node loop.
// GB300, 2 rays x 400 zones, 21 bins, 32 x 64: 37.7 -> 8.1 ms. Against the same rule in 80 bits, over seven grids and
// quadratures, T from 1 to 30 MeV and eta_e from -5 to 60, the mean zone's kernel and rates (2-norm) are
// 1.4e-16 to 1.2e-15 off, 0.54 to 1.14 of what library exponentials and divisions gave (mostly below 1).
#include "vx_internal.h"

namespace vx {

constexpr int kExpBits = 12, kExpTab = 1 << kExpBits;  // 2^{j / 4096}
constexpr int kTpb64 = VX_TPB_FP64;

__host__ __device__ inline size_t smem_fp64_bytes(int N, int S) {
    return (2 * (size_t)N * N + 4 * (size_t)S * N + 2 * (size_t)N + 4 * VX_MAX_NE + kExpTab + 8 * (size_t)kTpb64) * sizeof(double);
}
size_t smem_fp64(const Common &c) { return smem_fp64_bytes(c.N, c.S); }

struct Zone64 {
    double T, eta, iT, iTl;  // 1/T and its remainder
    double ep, em;           // e^eta, e^-eta
    int bad, fast;
};

// FP64 to FP32 by integer operations (the conversion instruction runs on the FP64 pipe), rounded to nearest; numbers
// below the FP32 normal range to 0.
__device__ __forceinline__ float to_f32(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) + 0x10000000ull;
    const unsigned hi = (unsigned)(b >> 32), e = hi & 0x7fffffffu;
    const float f = __uint_as_float((__funnelshift_l((unsigned)b, e - (896u << 20), 3) & 0x7fffffffu) | (hi & 0x80000000u));
    return e < (897u << 20) ? 0.f : f;
}
// |x| 2^32 for |x| <= 1/2, cut, by integer operations as well.
__device__ __forceinline__ unsigned fixed32(double x) {
    const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu;
    const unsigned w = __funnelshift_r((unsigned)__double2loint(x), (hi & 0xfffffu) | 0x100000u, 21);  // |x| = w 2^{e - 1054}
    return __funnelshift_rc(w, 0u, 1022u - (hi >> 20));
}
// Moments of the blocking factor of one (pair, omega) unit over the electron-energy nodes.
struct Mom64 {
    double p, m, z;
};

// nodes: {tau, w(1+tau)^2, w(1-tau)^2, w(1-tau^2)} of the nodes tau >= 0; mid: the first is tau = 0.
__device__ __forceinline__ void nodes_fast(const double *__restrict__ nodes, const double *__restrict__ tab, int n, bool mid,
                                           double Bs, float Bl, double c1, double c2, double oneQ, Mom64 &M) {
    const double magic = 6755399441055744.0;  // 1.5 2^52: adding it rounds to an integer in the low word
    // 2^{n + r/4096} = 2^{n - kShift/4096} (1 + b) (1 + y) with 1 + b = 2^{kShift/4096}: of (1 + b)(1 + y) - 1, which lies
    // around b = 0.0116, the low word counts units of 2^-59 and no term can carry out of the binade.
    constexpr int kShift = 68;
    const double L1 = 0.0001692253858788929, b1 = 1.01157379021457800244;  // ln 2 / 4096, 1 + b
    const long long bBits = 0x3f87b3ffd3b2f2e4ll;                          // b
    const double unit = 576460752303423488.0;                              // 2^59
    const double Lb = L1 * b1;
    const unsigned L2u = (unsigned)(L1 * L1 / 2.0 * b1 * unit / 2.0 + 0.5);  // of r^2 2^33, times 2^-32
    const float L3f = (float)(L1 * L1 * L1 / 6.0 * b1 * unit), L1f = (float)(L1 * b1 * unit);
    M.p = M.m = M.z = 0.0;
    int k = 0;
    if (mid) {
        const double r = 1.0 / (oneQ + (c1 + c2));
        M.p = nodes[1] * r;
        M.m = nodes[2] * r;
        M.z = nodes[3] * r;
        k = 1;
    }
#pragma unroll 2
    for (; k < n; ++k) {
        const double tau = nodes[4 * k], wp = nodes[4 * k + 1], wm = nodes[4 * k + 2], wz = nodes[4 * k + 3];
        const double u = fma(Bs, tau, magic), un = u - magic, r = fma(Bs, tau, -un);  // t 4096 = un + r, |r| <= 1/2
        const int q = __double2loint(u) - kShift, qm = -q - 2 * kShift;
        const float rf = to_f32(r), tf = to_f32(tau);
        const unsigned ri = fixed32(r);
        const long long ev = bBits + __umulhi(2u * __umulhi(ri, ri), L2u);
        const int od = __float2int_rn(fmaf(L3f * rf * rf, rf, L1f * Bl * tf));  // the cubic term, and d's remainder
        const double yp = fma(Lb, r, __longlong_as_double(ev + od)), ym = fma(-Lb, r, __longlong_as_double(ev - od));
        double tp = tab[q & (kExpTab - 1)], tm = tab[qm & (kExpTab - 1)];
        tp = __hiloint2double(__double2hiint(tp) + ((q >> kExpBits) << 20), __double2loint(tp));
        tm = __hiloint2double(__double2hiint(tm) + ((qm >> kExpBits) << 20), __double2loint(tm));
        const double P = fma(tp, yp, tp), Mi = fma(tm, ym, tm);  // 2^t, 2^-t
        const double Da = fma(c1, Mi, fma(c2, P, oneQ)), Db = fma(c1, P, fma(c2, Mi, oneQ));
        const double D = Da * Db;
        double y;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(D));
        const double e = fma(-D, y, 1.0), R = fma(y, fma(e, e, e), y);
        const double Oa = R * Db, Ob = R * Da;
        M.p = fma(wp, Oa, fma(wm, Ob, M.p));
        M.m = fma(wm, Oa, fma(wp, Ob, M.m));
        M.z = fma(wz, Oa, fma(wz, Ob, M.z));
    }
}

// The plain loop, exponentials node by node.
__device__ __noinline__ void nodes_plain(const double *__restrict__ nodes, int n, bool mid, double h, double Em, double iT,
                                         double eta, Mom64 &M) {
    const double B = h * iT, Pe = fma(Em, iT, -eta), Pp = fma(Em, iT, eta);
    M.p = M.m = M.z = 0.0;
    for (int k = 0; k < n; ++k) {
        const double t = nodes[4 * k];
        for (int s = 0; s < (mid && k == 0 ? 1 : 2); ++s) {
            const double u = s ? 1.0 - t : 1.0 + t, v = s ? 1.0 + t : 1.0 - t;
            const double r = 1.0 / ((1.0 + exp(-fma(B, u, Pe))) * (1.0 + exp(-fma(B, v, Pp))));
            M.p = fma(nodes[4 * k + (s ? 2 : 1)], r, M.p);
            M.m = fma(nodes[4 * k + (s ? 1 : 2)], r, M.m);
            M.z = fma(nodes[4 * k + 3], r, M.z);
        }
    }
}

// e^{x + xl} for a small correction xl.
__device__ __forceinline__ double exp_pair(double x, double xl) {
    const double e = exp(x);
    return fma(e, xl, e);
}

// CTA = zone, or one of L.parts shares of it. A zone's bin pairs go in up to eight parts, always the same ones, so that
// its results do not depend on how many CTAs take them; a part's (pair, omega) units in equal contiguous
// ranges, one per thread, and partial sums of pairs that two threads share added in thread order. Shares meet in
// global memory (L.phi_part): whichever ends last reads the others' kernel matrices and contracts; none waits.
__global__ void __launch_bounds__(kTpb64) k_pair_fp64(const __grid_constant__ Launch64 L) {
    extern __shared__ __align__(16) double smd[];
    __shared__ Zone64 zs;
    __shared__ long long s_zone;
    const Common &C = L.c;
    __shared__ int s_last;
    const int N = C.N, S = C.S, N2 = N * N, nmu = C.n_mu, parts = L.parts;
    double *A0 = smd, *A1 = smd + N2, *vec = smd + 2 * N2, *em = vec + 4 * S * N, *hx = em + N;
    double *nodes = hx + N, *tab = nodes + 4 * VX_MAX_NE, *part = tab + kExpTab;  // part[slot][4][threads]
    const int tid = threadIdx.x, TB = blockDim.x;
    const int nh = (C.n_e + 1) / 2;
    const bool mid = C.n_e & 1;
    for (int k = tid; k < nh; k += TB) {
        const int q = C.n_e / 2 + k;
        nodes[4 * k] = L.n64.tau[q];
        nodes[4 * k + 1] = L.n64.cp[q];
        nodes[4 * k + 2] = L.n64.cm[q];
        nodes[4 * k + 3] = L.n64.c0[q];
    }
    for (int k = tid; k < kExpTab; k += TB) tab[k] = L.exptab[k];
    validate_offsets(L.off, L.n_rays, L.Z, L.flag);

    for (;;) {
        if (tid == 0) s_zone = (long long)atomicAdd(L.counter, 1ull);
        __syncthreads();
        const long long z = s_zone / parts;
        if (z >= L.Z) break;
        const int share = (int)(s_zone - z * parts), K = L.count;
        auto first_pair = [&](int k) { return min(C.npair, L.group * (L.groups * k / K)); };  // of part k
        if (tid == 0) {
            const double T = L.state[4 * z + 0], eta = L.state[4 * z + 1], iT = 1.0 / T;
            zs.T = T;
            zs.eta = eta;
            zs.bad = !(T > 0.0) || !isfinite(T) || !isfinite(eta) || fabs(eta) > VX_ETA_MAX;
            zs.iT = iT;
            zs.iTl = fma(-T, iT, 1.0) * iT;
            zs.ep = exp(eta);
            zs.em = exp(-eta);
            zs.fast = C.q0h_max * iT + fabs(eta) < 690.0;
        }
        __syncthreads();
        const double T = zs.T, iT = zs.iT, iTl = zs.iTl;
        if (zs.bad) {
            const double nan = __longlong_as_double(0x7ff8000000000000ll);
            for (int e = tid; share == 0 && e < S * N; e += TB) {
                size_t o = (size_t)z * S * N + e;
                L.j0[o] = nan; L.chi0[o] = nan; L.j1[o] = nan; L.chi1[o] = nan;
            }
            if (L.phi && share == 0)
                for (int e = tid; e < 4 * N2; e += TB) L.phi[(size_t)z * 4 * N2 + e] = nan;
            if (tid == 0) atomicOr(L.flag, VX_FLAG_BAD_STATE);
            __syncthreads();
            continue;
        }
        for (int e = tid; e < 4 * S * N; e += TB) {
            int o = e / (S * N), s = (e / N) % S, j = e % N;
            size_t a = ((size_t)z * S + C.partner[s]) * N + j;
            double v;
            if (o == 0) v = C.w[j] * (1.0 - L.J[a]);
            else if (o == 1) v = C.w[j] * L.J[a];
            else v = C.w[j] * L.H[a];
            vec[e] = v;
        }
        for (int i = tid; i < N; i += TB) {
            em[i] = exp(-C.eps[i] / T);
            const double f = 0.5 * C.eps[i], x = f * iT;  // e^{-eps/2T}
            hx[i] = exp_pair(-x, -fma(f, iT, -x) - f * iTl);
        }
        __syncthreads();

        // log2(e) 4096 / T as a value and its remainder
        const double LG = 5909.278887481194, LGl = 8.337520124285351e-14;  // 4096 log2(e)
        const double gT = LG * iT, gTl = fma(LG, iT, -gT) + fma(LG, iTl, LGl * iT);
        for (int k = K * share / parts; k < K * (share + 1) / parts; ++k) {
            const int q0 = first_pair(k), q1 = first_pair(k + 1), U = (q1 - q0) * nmu;
            const int u0 = q0 * nmu + (int)((long long)tid * U / TB), u1 = q0 * nmu + (int)((long long)(tid + 1) * U / TB);
            double a0 = 0, b0 = 0, a1 = 0, b1 = 0;  // l = 0 terms I, II; l = 1
            int p = u0 / nmu, m = u0 - (u0 / nmu) * nmu, mb = m, slot = 0;
            for (int u = u0; u < u1; ++u) {
                const double *rec = L.tab64 + (size_t)u * 5;
                const double h = rec[0], Em = rec[1], kp = rec[2], km = rec[3], k0 = rec[4];
                Mom64 M;
                if (zs.fast) {
                    const double Q0 = hx[C.pij[p] >> 8] * hx[C.pij[p] & 0xff];
                    const double Bs = h * gT;
                    const float Bl = to_f32(fma(h, gT, -Bs) + h * gTl);
                    nodes_fast(nodes, tab, nh, mid, Bs, Bl, zs.ep * Q0, zs.em * Q0, fma(Q0, Q0, 1.0), M);
                } else {
                    nodes_plain(nodes, nh, mid, h, Em, iT, zs.eta, M);
                }
                const double t = C.t64[m], KI = fma(kp, M.p, fma(km, M.m, k0 * M.z)), KII = fma(km, M.p, fma(kp, M.m, k0 * M.z));
                a0 += KI;
                b0 += KII;
                a1 = fma(t, KI, a1);
                b1 = fma(t, KII, b1);
                ++m;
                if (m == nmu || u + 1 == u1) {
                    if (mb == 0 && m == nmu) {
                        const int pi = C.pij[p] >> 8, pj = C.pij[p] & 0xff;
                        A0[pi * N + pj] = a0; A1[pi * N + pj] = a1;
                        if (pi != pj) { A0[pj * N + pi] = b0; A1[pj * N + pi] = b1; }
                    } else {
                        double *q = part + slot * 4 * TB + tid;
                        q[0] = a0; q[TB] = b0; q[2 * TB] = a1; q[3 * TB] = b1;
                    }
                    a0 = b0 = a1 = b1 = 0.0;
                    slot = 1;
                    ++p;
                    m = mb = 0;
                }
            }
            __syncthreads();
            // pairs split between threads: owner of unit v is thread ceil((v + 1) TB / U) - 1
            for (int q = q0 + tid; q < q1; q += TB) {
                const long long ua = (long long)(q - q0) * nmu, ub = ua + nmu - 1;
                const int ta = (int)(((ua + 1) * TB + U - 1) / U) - 1, tb = (int)(((ub + 1) * TB + U - 1) / U) - 1;
                if (ta == tb) continue;
                double s[4] = {0, 0, 0, 0};
                for (int t = ta; t <= tb; ++t) {
                    if (U < TB && t * U / TB == (t + 1) * U / TB) continue;  // fewer units than threads: an empty range
                    const int sl = t == ta && ua > (long long)t * U / TB ? 1 : 0;
                    for (int c = 0; c < 4; ++c) s[c] += part[(sl * 4 + c) * TB + t];
                }
                const int pi = C.pij[q] >> 8, pj = C.pij[q] & 0xff;
                A0[pi * N + pj] = s[0]; A1[pi * N + pj] = s[2];
                if (pi != pj) { A0[pj * N + pi] = s[1]; A1[pj * N + pi] = s[3]; }
            }
            __syncthreads();
        }
        if (parts > 1) {
            double *F = L.phi_part + (size_t)z * 2 * N2;
            const int qb = first_pair(K * share / parts), qe = first_pair(K * (share + 1) / parts);
            for (int q = qb + tid; q < qe; q += TB) {
                const int pi = C.pij[q] >> 8, pj = C.pij[q] & 0xff, ij = pi * N + pj, ji = pj * N + pi;
                F[ij] = A0[ij]; F[ji] = A0[ji];
                F[N2 + ij] = A1[ij]; F[N2 + ji] = A1[ji];
            }
            __threadfence();
            __syncthreads();
            if (tid == 0) {
                s_last = atomicAdd(L.arrived + z, 1) == parts - 1;
                if (s_last) L.arrived[z] = 0;  // for the next launch
                __threadfence();
            }
            __syncthreads();
            if (!s_last) continue;
            for (int e = tid; e < N2; e += TB) {
                A0[e] = __ldcg(F + e);
                A1[e] = __ldcg(F + N2 + e);
            }
            __syncthreads();
        }
        const double c0 = 6.283185307179586 * C.norm * C.g2, c1 = 3.0 * c0;
        for (int e = tid; e < 4 * S * N; e += TB) {
            const int o = e / (S * N), s = (e / N) % S, i = e % N;
            const double *M = (o >> 1) ? A1 : A0;
            const bool prod = (o & 1) == 0;
            const double bI = C.bI64[s], bII = C.bII64[s];
            const double *v = vec + (size_t)(o * S + s) * N;
            double acc = 0.0;
            for (int j = 0; j < N; ++j) {
                double k = bI * M[i * N + j] + bII * M[j * N + i];
                acc += (prod ? em[i] * em[j] : 1.0) * k * v[j];
            }
            const double r = ((o >> 1) ? c1 : c0) * acc;
            double *dst = o == 0 ? L.j0 : o == 1 ? L.chi0 : o == 2 ? L.j1 : L.chi1;
            dst[((size_t)z * S + s) * N + i] = r;
            if (!isfinite(r)) atomicOr(L.flag, VX_FLAG_NONFINITE);
        }
        if (L.phi) {
            for (int e = tid; e < 4 * N2; e += TB) {
                const int d = e / (2 * N2), l = (e / N2) & 1, ij = e % N2, i = ij / N, j = ij % N;
                double a = l ? A1[ij] : A0[ij];
                L.phi[(size_t)z * 4 * N2 + e] = C.g2 * (d == 0 ? em[i] * em[j] * a : a);
            }
        }
        __syncthreads();
    }
}

const void *kernel_fp64_fwd() { return (const void *)k_pair_fp64; }

cudaError_t launch_fp64_fwd(const Launch64 &L, int grid, int block, size_t smem, cudaStream_t s) {
    k_pair_fp64<<<grid, block, smem, s>>>(L);
    return cudaGetLastError();
}

}  // namespace vx
