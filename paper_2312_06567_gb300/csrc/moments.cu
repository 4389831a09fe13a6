// Moments, entropy and totals of a stored state (Dzanic & Martinelli, arXiv
// 2312.06567, section "Governing equations": Q = int psi f, Pi = int f c c; the
// discrete entropy of section "Numerical method").
//
// All of these read every value of the state once and do little with it, so
// HBM bounds them once nothing else does.  What else there was: the FP64 pipe
// (2 instructions per SM and clock: a direct sum of the raw moments costs 17
// per value, a log() about 25), too few bytes in flight with one point per
// thread, and scalar error-free sums.  Here:
//   * raw moments are taken per first-axis velocity line: three (F) or four
//     (F, G) sums over centred indices jt = j - jc, folded per line and plane;
//   * the stepping path's line sums of an FP32 state are error-free FP32 pairs,
//     two points per thread on packed instructions; the diagnostic entry points
//     sum in FP64 about the node nearest u = 0;
//   * the entropy takes ln F from a table and a short series, the part that FP32
//     holds exactly or that lies far below the result on packed instructions.
// Times are on a GB300 for 16,384 points x 13,824 velocities (0.91 GB of FP32
// state): the stepping path's moments 1.16 -> 0.40 ms, the diagnostics'
// 7.18 -> 1.46, all of macro + moments + totals + entropy 22.6 -> 3.9.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "stage_f32_common.cuh"

namespace {

constexpr int MT = 256;          // threads per block
constexpr int MCH = 8;           // velocities loaded before they are used
// one plane quantity of two points: P += c * (s + e), error-free
__device__ __forceinline__ void plane_add2(float2 &P, float2 &Pe, float c, float2 s, float2 e) {
    const float2 c2 = dup2(c);
    const float2 pr = __fmul2_rn(c2, s);
    sum2x2(P, Pe, pr);
    Pe = __fadd2_rn(Pe, __ffma2_rn(c2, s, neg2(pr)));
    Pe = __ffma2_rn(c2, e, Pe);
}

// Raw moments of an FP32 state on the stepping path: lines' and planes' sums
// as FP32 pairs, the stage epilogue's operations in its velocity order, so the
// partials equal what an epilogue yields for the same values.  A thread takes
// the two points p and p + 256: one packed instruction serves both, loads stay
// coalesced for every P, and 2 x 8 loads per thread are in flight.  The FP64
// index moments of finished planes stay in the partials buffer, which the
// thread owns for its points (a block of lines spans few planes), leaving the
// registers to loads.  1.16 -> 0.40 ms for the state above (2.3 TB/s; latency
// of the sum chains at 24 warps per SM); with two blocks per SM 0.45, with 4
// velocities 0.43.
template <int C>
__global__ void __launch_bounds__(MT, 3) k_moments_f32(const float *f, double *part, VelGrid vg, int Nu, int P, int Kblk) {
    constexpr int NL = C == 2 ? 4 : 3, NQ = C == 2 ? 7 : 6;
    constexpr int MCH = C == 2 ? 4 : 8;                  // with G, eight spill 384 bytes, four 156
    const int pa = blockIdx.x * (2 * MT) + threadIdx.x, pb = pa + MT;
    if (pa >= P) return;
    const bool two = pb < P;
    const float *fa = f + pa, *fb = f + (two ? pb : pa);
    const int vb = blockIdx.y;
    const int k0 = vb * Kblk, k1 = min(Nu, k0 + Kblk);
    const int vn1 = vg.n[0], vn2 = vg.n[1];
    const int jc[3] = {(vn1 - 1) / 2, (vn2 - 1) / 2, (vg.n[2] - 1) / 2};
    const size_t GO = (size_t)Nu * P;                    // offset of the G component
    double *Ja = part + (size_t)vb * BGK_NMOM * P + pa;
    double *Jb = part + (size_t)vb * BGK_NMOM * P + (two ? pb : pa);
    float2 Pl[NQ], Pe[NQ];
#pragma unroll
    for (int i = 0; i < NQ; ++i) Pl[i] = Pe[i] = dup2(0.f);
    bool first = true;
    auto flush = [&](int j3) {
        const double c = trap3(j3, vg), t = (float)(j3 - jc[2]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h == 1 && !two) break;
            double d[7];
#pragma unroll
            for (int i = 0; i < 7; ++i)
                d[i] = i < NQ ? (double)(h ? Pl[i].y : Pl[i].x) + (double)(h ? Pe[i].y : Pe[i].x) : 0.0;
            plane_to_part(h ? Jb : Ja, P, c, t, d, first);
        }
#pragma unroll
        for (int i = 0; i < NQ; ++i) Pl[i] = Pe[i] = dup2(0.f);
        first = false;
    };
    int j3cur = (k0 / vn1) / vn2;
    for (int kl = k0; kl < k1; kl += vn1) {
        const int line = kl / vn1;
        const int j2 = line % vn2, j3 = line / vn2;
        if (j3 != j3cur) { flush(j3cur); j3cur = j3; }
        float2 L[NL], E[NL];
#pragma unroll
        for (int i = 0; i < NL; ++i) L[i] = E[i] = dup2(0.f);
        const size_t off = (size_t)kl * P;
        for (int j0 = 0; j0 < vn1; j0 += MCH) {
            float2 F[MCH], G[C == 2 ? MCH : 1];
#pragma unroll
            for (int i = 0; i < MCH; ++i) {
                if (j0 + i < vn1) {
                    const size_t o = off + (size_t)(j0 + i) * P;
                    F[i] = make_float2(__ldcs(fa + o), __ldcs(fb + o));
                    if (C == 2) G[C == 2 ? i : 0] = make_float2(__ldcs(fa + GO + o), __ldcs(fb + GO + o));
                }
            }
#pragma unroll
            for (int i = 0; i < MCH; ++i) {
                const int j1 = j0 + i;
                if (j1 < vn1) {
                    const float jt = (float)(j1 - jc[0]), cj = trap(j1, vn1);
                    const float2 cF = __fmul2_rn(dup2(cj), F[i]);
                    sum2x2(L[0], E[0], cF);
                    const float2 p1 = __fmul2_rn(cF, dup2(jt));
                    sum2x2(L[1], E[1], p1);
                    E[1] = sub2(E[1], __ffma2_rn(cF, dup2(-jt), p1));
                    const float jj = __fmul_rn(jt, jt);                  // exact
                    const float2 p2 = __fmul2_rn(cF, dup2(jj));
                    sum2x2(L[2], E[2], p2);
                    E[2] = sub2(E[2], __ffma2_rn(cF, dup2(-jj), p2));
                    if (C == 2) sum2x2(L[NL - 1], E[NL - 1], __fmul2_rn(dup2(cj), G[C == 2 ? i : 0]));
                }
            }
        }
        const float c2 = trap(j2, vn2), t2 = (float)(j2 - jc[1]);
        const float b = __fmul_rn(c2, t2), bb = __fmul_rn(b, t2);       // exact
        plane_add2(Pl[0], Pe[0], c2, L[0], E[0]);
        plane_add2(Pl[1], Pe[1], c2, L[1], E[1]);
        plane_add2(Pl[2], Pe[2], c2, L[2], E[2]);
        plane_add2(Pl[3], Pe[3], b, L[0], E[0]);
        plane_add2(Pl[4], Pe[4], b, L[1], E[1]);
        plane_add2(Pl[5], Pe[5], bb, L[0], E[0]);
        if (C == 2) plane_add2(Pl[NQ - 1], Pe[NQ - 1], c2, L[NL - 1], E[NL - 1]);
    }
    flush(j3cur);
    const double uc[3] = {vg.lo[0] + jc[0] * vg.h[0], vg.lo[1] + jc[1] * vg.h[1], vg.lo[2] + jc[2] * vg.h[2]};
    raw_in_place(Ja, P, vg, uc);
    if (two) raw_in_place(Jb, P, vg, uc);
}

// The node of each axis nearest u = 0, about which the diagnostics' sums are
// taken: index_to_raw then shifts by half a step at most (or by a distance that
// every velocity of the grid exceeds), so the raw moments come out as accurate as
// direct sums.  About the grid's middle a second moment is a difference of terms
// (half width / thermal speed)^2 times larger: on u = -2..60 with 64 nodes, a gas
// at rest with theta = 0.3 had 9e-13 for 1e-16.
__device__ __forceinline__ void zero_node(const VelGrid &vg, int (&jc)[3]) {
#pragma unroll
    for (int d = 0; d < 3; ++d) jc[d] = min(max((int)rint(-vg.lo[d] / vg.h[d]), 0), vg.n[d] - 1);
}

// The diagnostic entry points' second look: partials that are not finite (an
// infinity or NaN in the state, or sums out of range) are summed again directly
// in FP64: sums over centred indices make NaN of an infinite value (0 times it,
// or its difference in index_to_raw), which keeps its moments infinite here.
template <typename T>
__global__ void __launch_bounds__(MT) k_moments_redo(const T *f, double *part, const double *vtab, int Nu, int P,
                                                     int Kblk, int C) {
    const int p = blockIdx.x * MT + threadIdx.x, vb = blockIdx.y;
    if (p >= P) return;
    double *out = part + (size_t)vb * BGK_NMOM * P + p;
    if (isfinite(out[0] + out[(size_t)4 * P] + out[(size_t)5 * P] + out[(size_t)6 * P] + out[(size_t)10 * P])) return;
    const int k0 = vb * Kblk, k1 = min(Nu, k0 + Kblk);
    double m[BGK_NMOM];
#pragma unroll
    for (int j = 0; j < BGK_NMOM; ++j) m[j] = 0.0;
    for (int k = k0; k < k1; ++k) {
        const double *v = vtab + (size_t)k * BGK_VTAB;
        const double u1 = v[0], u2 = v[1], u3 = v[2], w = v[3];
        const double wF = w * (double)f[(size_t)k * P + p];
        m[0] += wF;
        m[1] = fma(wF, u1, m[1]);
        m[2] = fma(wF, u2, m[2]);
        m[3] = fma(wF, u3, m[3]);
        m[4] = fma(wF * u1, u1, m[4]);
        m[5] = fma(wF * u2, u2, m[5]);
        m[6] = fma(wF * u3, u3, m[6]);
        m[7] = fma(wF * u1, u2, m[7]);
        m[8] = fma(wF * u1, u3, m[8]);
        m[9] = fma(wF * u2, u3, m[9]);
        if (C == 2) m[10] = fma(w, (double)f[((size_t)Nu + k) * P + p], m[10]);
    }
#pragma unroll
    for (int j = 0; j < BGK_NMOM; ++j) out[(size_t)j * P] = m[j];
}

// Raw moments with FP64 sums: of an FP64 state, and of an FP32 state for the
// diagnostic entry points.  Per line T_m = sum_j c jt^m F (m <= 2) and sum_j c G
// with the exact factors c jt^m from a table, three (four) FP64 instructions per
// value instead of the 17 of a direct sum of the raw moments, folded per line into
// the plane's sums and per plane into the index moments in the partials buffer.
// FP32 values are widened by integer instructions.  The FP64 pipe bounds it (two
// instructions per multiprocessor and clock; two to four blocks, four or eight
// loads ahead all take the same time): 2.3e8 FP32 values 1.46 ms (7.2 for direct
// sums), with G 1.86, half as many FP64 ones 0.78 and 0.98.  Sums of eight FP32
// values as FP32 pairs before the FP64 ones took 0.90 ms, but lost five times what
// FP64 sums lose on lines of wide range.
template <typename T, int C>
__global__ void __launch_bounds__(MT, 2) k_moments_sums(const T *f, double *part, VelGrid vg, int Nu, int P, int Kblk) {
    constexpr int NQ = C == 2 ? 7 : 6;
    const int p = blockIdx.x * MT + threadIdx.x;
    // (c jt, c jt^2) and c of the first-axis nodes, c the trapezoid factor (exact)
    __shared__ double2 sj[BGK_MAXV];
    __shared__ double sc[BGK_MAXV];
    const int vn1 = vg.n[0], vn2 = vg.n[1];
    int jc[3];
    zero_node(vg, jc);
    for (int j = threadIdx.x; j < vn1; j += MT) {
        const double t = j - jc[0], c = trap(j, vn1);
        sj[j] = make_double2(c * t, c * t * t);
        sc[j] = c;
    }
    __syncthreads();
    if (p >= P) return;
    const int vb = blockIdx.y;
    const int k0 = vb * Kblk, k1 = min(Nu, k0 + Kblk);
    double *J = part + (size_t)vb * BGK_NMOM * P + p;
    double Pd[7];
#pragma unroll
    for (int i = 0; i < 7; ++i) Pd[i] = 0.0;
    bool first = true;
    auto flush = [&](int j3) {
        plane_to_part(J, P, trap3(j3, vg), (double)(j3 - jc[2]), Pd, first);
#pragma unroll
        for (int i = 0; i < 7; ++i) Pd[i] = 0.0;
        first = false;
    };
    int j3cur = (k0 / vn1) / vn2;
    for (int kl = k0; kl < k1; kl += vn1) {
        const int line = kl / vn1;
        const int j2 = line % vn2, j3 = line / vn2;
        if (j3 != j3cur) { flush(j3cur); j3cur = j3; }
        const T *fl = f + (size_t)kl * P + p, *gl = fl + (size_t)Nu * P;
        double T0 = 0.0, T1 = 0.0, T2 = 0.0, TG = 0.0;
        for (int j0 = 0; j0 < vn1; j0 += MCH) {
            T F[MCH], G[C == 2 ? MCH : 1];
#pragma unroll
            for (int i = 0; i < MCH; ++i)
                if (j0 + i < vn1) {
                    F[i] = __ldcs(fl + (size_t)(j0 + i) * P);
                    if (C == 2) G[C == 2 ? i : 0] = __ldcs(gl + (size_t)(j0 + i) * P);
                }
#pragma unroll
            for (int i = 0; i < MCH; ++i) {
                const int j1 = j0 + i;
                if (j1 < vn1) {
                    const double x = widen(F[i]), c = sc[j1];
                    const double2 t = sj[j1];
                    T0 = fma(c, x, T0);
                    T1 = fma(t.x, x, T1);
                    T2 = fma(t.y, x, T2);
                    if (C == 2) TG = fma(c, widen(G[C == 2 ? i : 0]), TG);
                }
            }
        }
        const double c = j2 == 0 || j2 == vn2 - 1 ? 0.5 : 1.0, t2 = (double)(j2 - jc[1]), b = c * t2, bb = b * t2;
        Pd[0] = fma(c, T0, Pd[0]); Pd[1] = fma(c, T1, Pd[1]); Pd[2] = fma(c, T2, Pd[2]);
        Pd[3] = fma(b, T0, Pd[3]); Pd[4] = fma(b, T1, Pd[4]); Pd[5] = fma(bb, T0, Pd[5]);
        if (C == 2) Pd[NQ - 1] = fma(c, TG, Pd[NQ - 1]);
    }
    flush(j3cur);
    const double uc[3] = {vg.lo[0] + jc[0] * vg.h[0], vg.lo[1] + jc[1] * vg.h[1], vg.lo[2] + jc[2] * vg.h[2]};
    raw_in_place(J, P, vg, uc);
}

// Sums over the velocity blocks, one thread per (slot, point): ACROSS writes
// m_out[p][slot] (bgk_moments), else out[slot][p] (a shard's partials).
template <bool ACROSS>
__global__ void __launch_bounds__(MT) k_reduce_moments(const double *part, int n_vblk, int P, double *out) {
    const int p = blockIdx.x * MT + threadIdx.x, j = blockIdx.y;
    if (p >= P) return;
    const double *q = part + (size_t)j * P + p;
    double s = 0.0;
#pragma unroll 8
    for (int vb = 0; vb < n_vblk; ++vb) s += q[(size_t)vb * BGK_NMOM * P];
    out[ACROSS ? (size_t)p * BGK_NMOM + j : (size_t)j * P + p] = s;
}

// ---- entropy ---------------------------------------------------------------
// ln x of a normal FP32 x (table-driven, after Tang 1990): x = 2^e m with m in
// [1, 2), k_i = 1/m to ten bits for the 1024 subintervals of m, so r = m k_i - 1
// is exact in FP32 (33 bits of m k_i less the 9 that cancel, |r| < 2^-9.6), and
//   ln x = (e ln2 - ln k_i) + (r - r^2/2) + r^3 (1/3 - r/4 + r^2/5):
// the first term in FP64, the second as an FP32 pair, the third, below 2^-30, in
// FP32 with the pair's low part and the rest of ln2.  Within 2^-50 of |ln x| for x
// outside [0.875, 1.125) (2^-54 root mean square, as log() has), where ln x itself
// is small; log() serves that interval.
constexpr int LOG_N = 1024;
struct LogTab { float k, pad; double l; };               // k_i, -ln k_i
// s + c = r - r^2/2 + r^3 (...) + e (ln2 - its FP64 value), on two values at once
__device__ __forceinline__ void log_tail2(float2 r, float2 e, float2 &s, float2 &c) {
    const float2 q = __fmul2_rn(r, r);
    const float2 qe = __ffma2_rn(r, r, neg2(q));                                     // r^2 = q + qe
    float2 t = __ffma2_rn(r, dup2(0.2f), dup2(-0.25f));
    t = __ffma2_rn(r, t, dup2(1.f / 3.f));
    t = __fmul2_rn(__fmul2_rn(r, q), t);
    s = __ffma2_rn(q, dup2(-0.5f), r);
    const float2 low = __ffma2_rn(q, dup2(-0.5f), sub2(r, s));                       // exact: |r| > q/2
    c = __fadd2_rn(__ffma2_rn(qe, dup2(-0.5f), t), low);
    c = __ffma2_rn(e, dup2(2.3190468138e-17f), c);
}
// the exact double of a normal FP32 value, halved for half = 1; of zero 2^-127,
// nothing beside the terms it is added to
__device__ __forceinline__ double widen_normal(float x, unsigned half = 0) {
    const unsigned b = __float_as_uint(x);
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + ((896u - half) << 20))), (int)(b << 29));
}

// Discrete entropy of the F component, partial over velocity blocks:
// part[vb][p] = sum_{k in block vb} w_k F ln F; a non-positive F (or NaN) has
// no entropy and is counted in *nonpos instead.  The sums are FP64 ones; two
// points per thread, so that what FP32 can do of the logarithm exactly or far
// below the result runs packed and four FP64 instructions per value remain (a
// library log and its sum take 25): 2.3e8 values 1.7 ms, 12 ms with log(), bound
// by the FP64 pipe at any occupancy from two to five blocks.  With ln F and the
// line sums as FP32 pairs 0.7 ms, but 2^-46 of F off where log() has 2^-53.
__global__ void __launch_bounds__(MT, 4) k_entropy_f32(const float *f, const LogTab *logs, VelGrid vg, int Nu, int P,
                                                       int Kblk, double *part, unsigned int *nonpos) {
    __shared__ __align__(16) LogTab tab[LOG_N];
    for (int i = threadIdx.x; i < LOG_N; i += MT)
        reinterpret_cast<float4 *>(tab)[i] = __ldg(reinterpret_cast<const float4 *>(logs) + i);
    __syncthreads();
    const int pa = blockIdx.x * (2 * MT) + threadIdx.x, pb = pa + MT;
    if (pa >= P) return;
    const bool two = pb < P;
    const float *fa = f + pa, *fb = f + (two ? pb : pa);
    const int vb = blockIdx.y;
    const int k0 = vb * Kblk, k1 = min(Nu, k0 + Kblk);
    const int vn1 = vg.n[0], vn2 = vg.n[1];
    double h[2] = {0.0, 0.0};
    unsigned int bad = 0;
    // not the table's: outside the positive normal range, or near 1
    auto other = [](float v) {
        const unsigned b = __float_as_uint(v);
        return b - 0x00800000u >= 0x7f000000u || b - 0x3f600000u < 0x00300000u;
    };
    for (int kl = k0; kl < k1; kl += vn1) {
        const int line = kl / vn1;
        const double c23 = (double)trap(line % vn2, vn2) * (double)trap3(line / vn2, vg);
        double T[2] = {0.0, 0.0}, S[2] = {0.0, 0.0};
        for (int j0 = 0; j0 < vn1; j0 += MCH) {
            float2 F[MCH];
#pragma unroll
            for (int i = 0; i < MCH; ++i)
                if (j0 + i < vn1) {
                    const size_t o = (size_t)(kl + j0 + i) * P;
                    F[i] = make_float2(__ldcs(fa + o), __ldcs(fb + o));
                }
#pragma unroll
            for (int i = 0; i < MCH; ++i) {
                if (j0 + i >= vn1) continue;
                const bool end = j0 + i == 0 || j0 + i == vn1 - 1;                   // trapezoid half weight
                double xa = widen_normal(F[i].x, end), xb = widen_normal(F[i].y, end);
                if (other(F[i].x) || other(F[i].y)) {
                    // positive values by log(), anything else is counted; their
                    // weight in the sums below is zero
                    for (int q = 0; q < 2; ++q) {
                        const float v = q ? F[i].y : F[i].x;
                        if (!other(v)) continue;
                        if (v > 0.f) h[q] = fma(c23 * (end ? 0.5 : 1.0) * (double)v, log((double)v), h[q]);
                        else if (q == 0 || two) ++bad;
                        if (q) { F[i].y = 1.f; xb = 0.0; }
                        else { F[i].x = 1.f; xa = 0.0; }
                    }
                }
                const unsigned ba = __float_as_uint(F[i].x), bb = __float_as_uint(F[i].y);
                const LogTab ta = tab[(ba >> 13) & (LOG_N - 1)], tb = tab[(bb >> 13) & (LOG_N - 1)];
                const float2 m = make_float2(__uint_as_float((ba & 0x007fffffu) | 0x3f800000u),
                                             __uint_as_float((bb & 0x007fffffu) | 0x3f800000u));
                // the exponent as a float: 2^23 + biased exponent, minus 2^23 + 127 (exact)
                const float2 e = __fadd2_rn(make_float2(__uint_as_float((ba >> 23) | 0x4b000000u),
                                                        __uint_as_float((bb >> 23) | 0x4b000000u)), dup2(-8388735.f));
                const float2 r = __ffma2_rn(m, make_float2(ta.k, tb.k), dup2(-1.f));             // exact
                float2 s, c;
                log_tail2(r, e, s, c);
                T[0] = fma(xa, fma(widen_normal(e.x), 0.69314718055994530942, ta.l), T[0]);
                T[1] = fma(xb, fma(widen_normal(e.y), 0.69314718055994530942, tb.l), T[1]);
                S[0] = fma(xa, widen_normal(s.x), S[0]);
                S[1] = fma(xb, widen_normal(s.y), S[1]);
                S[0] = fma(xa, widen_normal(c.x), S[0]);
                S[1] = fma(xb, widen_normal(c.y), S[1]);
            }
        }
        h[0] = fma(c23, T[0] + S[0], h[0]);
        h[1] = fma(c23, T[1] + S[1], h[1]);
    }
    const double W = vg.h[0] * vg.h[1] * vg.h[2];
    part[(size_t)vb * P + pa] = W * h[0];
    if (two) part[(size_t)vb * P + pb] = W * h[1];
    if (bad) atomicAdd(nonpos, bad);
}

// The same of an FP64 state.  ln F by a table of 256 subintervals in FP64, r =
// m k_i - 1 with one rounding and the series to r^7 (2^-67 of the next term): 12
// FP64 instructions per value in place of the library log()'s path (36 ms for
// 1.1e8 values); the FP64 pipe bounds it.
__global__ void __launch_bounds__(MT) k_entropy_f64(const double *f, VelGrid vg, int Nu, int P, int Kblk, double *part,
                                                    unsigned int *nonpos) {
    __shared__ double2 tab[256];                         // (k_i, -ln k_i)
    for (int i = threadIdx.x; i < 256; i += MT) {
        const double k = rint(512.0 / (1.0 + (i + 0.5) / 256.0)) / 512.0;
        tab[i] = make_double2(k, -log(k));
    }
    __syncthreads();
    const int p = blockIdx.x * MT + threadIdx.x;
    if (p >= P) return;
    const int vb = blockIdx.y;
    const int k0 = vb * Kblk, k1 = min(Nu, k0 + Kblk);
    const int vn1 = vg.n[0], vn2 = vg.n[1];
    double h = 0.0;
    unsigned int bad = 0;
    for (int kl = k0; kl < k1; kl += vn1) {
        const int line = kl / vn1;
        double T = 0.0;
        for (int j0 = 0; j0 < vn1; j0 += MCH) {
            double Fc[MCH];
#pragma unroll
            for (int i = 0; i < MCH; ++i)
                if (j0 + i < vn1) Fc[i] = __ldcs(f + (size_t)(kl + j0 + i) * P + p);
#pragma unroll
            for (int i = 0; i < MCH; ++i) {
                const int j1 = j0 + i;
                if (j1 >= vn1) continue;
                const double F = Fc[i];
                const unsigned hi = (unsigned)__double2hiint(F);
                double l;
                // not a positive normal value, or in [0.875, 1.125), where ln F
                // is small beside the table's roundings
                if (hi - 0x00100000u >= 0x7fe00000u || hi - 0x3fec0000u < 0x00060000u) {
                    if (!(F > 0.0)) { ++bad; continue; }
                    l = log(F);
                } else {
                    const double2 t = tab[(hi >> 12) & 255u];
                    const double m = __hiloint2double((hi & 0x000fffffu) | 0x3ff00000u, __double2loint(F));
                    // 2^52 + biased exponent, minus 2^52 + 1023 (exact)
                    const double e = __hiloint2double(0x43300000, hi >> 20) - 4503599627371519.0;
                    const double r = fma(m, t.x, -1.0);
                    double q = fma(r, 1.0 / 7.0, -1.0 / 6.0);
                    q = fma(r, q, 0.2);
                    q = fma(r, q, -0.25);
                    q = fma(r, q, 1.0 / 3.0);
                    q = fma(r, q, -0.5);
                    l = fma(e, 0.69314718055994530942, t.y) + fma(r * r, q, r);
                }
                T = fma(j1 == 0 || j1 == vn1 - 1 ? 0.5 * F : F, l, T);
            }
        }
        h = fma((double)trap(line % vn2, vn2) * (double)trap3(line / vn2, vg), T, h);
    }
    part[(size_t)vb * P + p] = vg.h[0] * vg.h[1] * vg.h[2] * h;
    if (bad) atomicAdd(nonpos, bad);
}

// ---- domain totals -----------------------------------------------------------
// sum_p W_p (rho, rho U, E) of the moments mom[P][11] and, with ent, sum_p W_p
// sum_vb ent[vb][p]: W_p the quadrature weight (node weights times |J_e| on the
// box, geo[p][10] on a curvilinear mesh).  Fixed grid and order, so equal
// states give equal totals; blocks write six sums each, one block adds them.
constexpr int TOT_BLOCKS = 152;
__global__ void __launch_bounds__(MT) k_totals(const double *mom, const double *ent, int n_vblk, int P, FROps fr,
                                               double jac, const double *geo, double *blk) {
    const int q = fr.q, Ns = q * q * q;
    double t[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int p = blockIdx.x * MT + threadIdx.x; p < P; p += gridDim.x * MT) {
        const int s = p % Ns;
        const double W = geo ? geo[(size_t)p * BGK_NGEO + 10] : fr.wq[s % q] * fr.wq[(s / q) % q] * fr.wq[s / (q * q)] * jac;
        const double *m = mom + (size_t)p * BGK_NMOM;
        t[0] = fma(W, m[0], t[0]); t[1] = fma(W, m[1], t[1]); t[2] = fma(W, m[2], t[2]); t[3] = fma(W, m[3], t[3]);
        t[4] = fma(W, 0.5 * (m[4] + m[5] + m[6]) + m[10], t[4]);
        if (ent) {
            double h = 0.0;
#pragma unroll 4
            for (int vb = 0; vb < n_vblk; ++vb) h += ent[(size_t)vb * P + p];
            t[5] = fma(W, h, t[5]);
        }
    }
    __shared__ double red[6][MT / 32];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        for (int o = 16; o > 0; o >>= 1) t[j] += __shfl_xor_sync(0xffffffffu, t[j], o);
        if ((threadIdx.x & 31) == 0) red[j][threadIdx.x >> 5] = t[j];
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        double s = 0.0;
        for (int w = 0; w < MT / 32; ++w) s += red[threadIdx.x][w];
        blk[(size_t)blockIdx.x * 6 + threadIdx.x] = s;
    }
}
__global__ void k_totals_sum(const double *blk, int n, double *out) {
    if (threadIdx.x < 6) {
        double s = 0.0;
        for (int b = 0; b < n; ++b) s += blk[(size_t)b * 6 + threadIdx.x];
        out[threadIdx.x] = s;
    }
}

}  // namespace

cudaError_t launch_moments_f64(const MomentArgs64 &a, const VelGrid &vg, int n_vblk, bool check, cudaStream_t s) {
    dim3 grid((a.P + MT - 1) / MT, n_vblk);
    if (a.C == 1) k_moments_sums<double, 1><<<grid, MT, 0, s>>>(a.f, a.part, vg, a.Nu, a.P, a.Kblk);
    else k_moments_sums<double, 2><<<grid, MT, 0, s>>>(a.f, a.part, vg, a.Nu, a.P, a.Kblk);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !check) return e;
    k_moments_redo<double><<<grid, MT, 0, s>>>(a.f, a.part, a.vtab, a.Nu, a.P, a.Kblk, a.C);
    return cudaGetLastError();
}

cudaError_t launch_moments_f32(const float *f, double *part, const double *vtab, const VelGrid &vg, int Nu, int P,
                               int Kblk, int C, int n_vblk, bool check, cudaStream_t s) {
    if (!check) {
        const dim3 grid((P + 2 * MT - 1) / (2 * MT), n_vblk);
        if (C == 1) k_moments_f32<1><<<grid, MT, 0, s>>>(f, part, vg, Nu, P, Kblk);
        else k_moments_f32<2><<<grid, MT, 0, s>>>(f, part, vg, Nu, P, Kblk);
        return cudaGetLastError();
    }
    const dim3 grid((P + MT - 1) / MT, n_vblk);
    if (C == 1) k_moments_sums<float, 1><<<grid, MT, 0, s>>>(f, part, vg, Nu, P, Kblk);
    else k_moments_sums<float, 2><<<grid, MT, 0, s>>>(f, part, vg, Nu, P, Kblk);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_moments_redo<float><<<grid, MT, 0, s>>>(f, part, vtab, Nu, P, Kblk, C);
    return cudaGetLastError();
}

cudaError_t launch_sum_partials(const double *part, int n_vblk, int P, double *out, cudaStream_t s) {
    k_reduce_moments<false><<<dim3((P + MT - 1) / MT, BGK_NMOM), MT, 0, s>>>(part, n_vblk, P, out);
    return cudaGetLastError();
}

cudaError_t launch_reduce_moments(const double *part, int n_vblk, int P, double *m_out, cudaStream_t s) {
    k_reduce_moments<true><<<dim3((P + MT - 1) / MT, BGK_NMOM), MT, 0, s>>>(part, n_vblk, P, m_out);
    return cudaGetLastError();
}

void entropy_log_table(std::vector<double> &out) {
    out.resize(2 * LOG_N);
    for (int i = 0; i < LOG_N; ++i) {
        LogTab t{};
        t.k = (float)(std::rint(LOG_N / (1.0 + (i + 0.5) / LOG_N)) / LOG_N);
        t.l = -std::log((double)t.k);
        std::memcpy(&out[2 * i], &t, sizeof t);
    }
}

cudaError_t launch_entropy_f32(const float *f, const double *logs, const VelGrid &vg, int Nu, int P, int Kblk, int n_vblk,
                               double *part, unsigned int *nonpos, cudaStream_t s) {
    k_entropy_f32<<<dim3((P + 2 * MT - 1) / (2 * MT), n_vblk), MT, 0, s>>>(f, reinterpret_cast<const LogTab *>(logs), vg, Nu, P,
                                                                           Kblk, part, nonpos);
    return cudaGetLastError();
}
cudaError_t launch_entropy_f64(const double *f, const VelGrid &vg, int Nu, int P, int Kblk, int n_vblk, double *part,
                               unsigned int *nonpos, cudaStream_t s) {
    k_entropy_f64<<<dim3((P + MT - 1) / MT, n_vblk), MT, 0, s>>>(f, vg, Nu, P, Kblk, part, nonpos);
    return cudaGetLastError();
}

size_t totals_scratch() { return (size_t)(TOT_BLOCKS + 1) * 6; }
cudaError_t launch_totals(const double *mom, const double *ent, int n_vblk, int P, const FROps &fr, double jac,
                          const double *geo, double *scratch, cudaStream_t s) {
    const int nb = std::min(TOT_BLOCKS, (P + MT - 1) / MT);
    k_totals<<<nb, MT, 0, s>>>(mom, ent, n_vblk, P, fr, jac, geo, scratch + 6);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_totals_sum<<<1, 32, 0, s>>>(scratch + 6, nb, scratch);
    return cudaGetLastError();
}
