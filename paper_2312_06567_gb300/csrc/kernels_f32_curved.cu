// Mixed-form fused stage on curvilinear meshes (FP32 state), one thread per
// group of first-axis node lines.
//
// The transformed-flux operator of CurvOps32 (bgk_internal.cuh): per direction
// and node i of a line, with a_j = u . S^d_j and the face normal velocities
// A = u . S_face,
//   t_i = sum_{j != i} kappa_ij a_j (f_j - f_i)
//       + g_R'_i A_R dev_R + g_L'_i A_L dev_L,
//   kappa_ij = D_ij - def_j - g_R'_i l_j(+1) - g_L'_i l_j(-1),
// dev = (upwind trace) - f_i: the own trace sum_j l_j (f_j - f_i) on an outflow
// face, the neighbour's sum_j l_j (nb_j - f_i) or the exterior value minus f_i
// on an inflow face, -f_i on a closed face (F^I = 0); then
//   div = (1/J) (sum_d t_d + f_i u . H).
// kappa is formed in FP64 from the FP32 tables and held as an FP32 pair, so
// kappa a_j is one rounding of the exact product and the telescoping of the
// tables survives; every rounding acts on deviations.
//
// What bounded the node-per-thread kernel this replaces was instructions (539
// per node and velocity with F and G) and the latency of neighbour values
// behind a block barrier (32% of the issue slots used).  Here:
//   * a thread owns LPT whole first-axis lines of an element (at Q = 2 a plane
//     of four nodes, else one line): a neighbour's values, the own line's and
//     the velocity bookkeeping serve all of them, and loads are vectors;
//   * neighbouring nodes of a line run as one packed FP32 pair, for F and again
//     for G, so geometry, coefficients and equilibrium are formed pairwise and
//     once for both components (pairing F with G instead needs every
//     coefficient twice in a register pair: 240 instructions per node);
//   * u . S is one packed FMA per two scalars: S's u_2 and u_3 parts are summed
//     once per velocity line into shared memory beside S's first component,
//     from a copy of the geometry in thread order (geop, coalesced);
//   * the volume term, the defect correction and the outflow faces' own traces
//     multiply the same deviation, so their coefficients are added first;
//   * no block barrier: each thread requests the values it needs itself (its own
//     and, on faces with inflow, the neighbours', mostly from L1 and L2) -- at
//     Q = 2 one velocity ahead through shared memory (without that: 8.3 ms), else
//     before any arithmetic.
// Stage of the sphere O-grid with 6 x 12 x 12 elements, p = 1, 40^3 velocities, F
// and G (4.4e8 points x velocities): 17.1 -> 5.8 ms (1.6 TB/s, 24% of HBM), 195
// instructions per node, 34% of the issue slots: eight warps per SM (registers
// and shared memory) do not cover the instruction latencies.  Warped box 6x5x6,
// p = 2, one component, 20^3: 1.17 -> 0.58 ms.  Small meshes keep the node-per-
// thread kernel (curved_node in kernels_f32.cu).
// Moments are the line kernel's: error-free line sums, plane pairs in
// thread-local memory (touched once per velocity line), FP64 index moments in the
// partials buffer.
// Dzanic & Martinelli, arXiv 2312.06567, section "Numerical method".

#include "stage_f32_common.cuh"

namespace {

using P2 = float2;                       // nodes 2 r and 2 r + 1 of a line

template <int Q, int C>
struct CurvGeom {
    // lines per thread: a plane of lines at Q = 2, one line else (more would
    // leave room for four warps per SM only)
    static constexpr int LPT = Q == 2 ? 2 : 1;
    static constexpr int TE = Q * Q / LPT;               // threads per element
    static constexpr int NR = (Q + 1) / 2;               // pairs per line (odd Q: the last lane is a copy)
    static constexpr int NPR = LPT * NR;                 // pairs per thread
    static constexpr int NN = Q * LPT;                   // nodes per thread
    // geometry records (two scalars each): S^1 of the line's other nodes in
    // rotated order, the line's two faces; S^2 of the other lines, their faces;
    // S^3 of the other planes, their faces; H
    static constexpr int O_A1 = 0, O_FX = O_A1 + LPT * (Q - 1) * NR, O_A2 = O_FX + LPT, O_FY = O_A2 + LPT * (Q - 1) * NR,
                         O_A3 = O_FY + 2 * NR, O_FZ = O_A3 + (Q - 1) * NPR, O_H = O_FZ + 2 * NPR, NG = O_H + NPR;
    static constexpr int NE = 6 * NPR;                   // equilibrium records, float4
    static constexpr int NQ = C == 2 ? 7 : 6;
    static constexpr int NT = 64;                        // two warps (96 threads at Q = 3: 8% slower)
    // Q = 2: a thread's values travel through a ring of two velocities in shared
    // memory, asynchronously (six 16-byte slots per component); else they are
    // read directly, both sides of every direction up front where that fits the
    // registers
    static constexpr bool BOTH = Q == 3 && C == 1;
    static constexpr int SLOTS = 5;
    static constexpr int MINB = Q == 3 && C == 1 ? 6 : Q <= 3 ? 4 : 3;
    template <bool RING>
    static size_t smem(int vn1) {
        return ((size_t)(NG + NE + LPT + (RING ? 2 * SLOTS * C : 0)) * 16) * NT + (size_t)(1 + 2 * C) * vn1 * sizeof(float2);
    }
};

// L consecutive node lines of one component as pairs
template <int Q, int L, bool VEC>
__device__ __forceinline__ void ld_lines(const float *p, P2 (&v)[L][(Q + 1) / 2]) {
    float x[L * Q];
    if constexpr (VEC && (L * Q) % 4 == 0) {
#pragma unroll
        for (int i = 0; i < L * Q; i += 4) {
            asm volatile("ld.global.nc.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(x[i]), "=f"(x[i + 1]), "=f"(x[i + 2]), "=f"(x[i + 3]) : "l"(p + i));
        }
    } else {
#pragma unroll
        for (int i = 0; i < L * Q; ++i) asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(x[i]) : "l"(p + i));
    }
#pragma unroll
    for (int l = 0; l < L; ++l)
#pragma unroll
        for (int r = 0; r < (Q + 1) / 2; ++r) v[l][r] = make_float2(x[l * Q + 2 * r], x[l * Q + (2 * r + 1 < Q ? 2 * r + 1 : Q - 1)]);
}
// node i of a line held as pairs
template <int N>
__device__ __forceinline__ float lane_of(const P2 (&v)[N], int i) { return i % 2 ? v[i / 2].y : v[i / 2].x; }

// Operator constants in shared memory, as pairs.  Row of node i towards its
// line's other nodes, j = (i + m) mod Q: (kappa_hi, kappa_lo), (l_j(-1), l_j(+1))
// and g = g_L'_i, -g_R'_i; crow[i][m]: both lanes node i (directions 2 and 3);
// cline[m][r]: lanes the nodes 2 r and 2 r + 1 (direction 1).
struct RowRec { float4 k, lo; float2 g[2]; };

template <int Q, int C, bool VEC>
__global__ void __launch_bounds__(CurvGeom<Q, C>::NT, CurvGeom<Q, C>::MINB) k_stage_f32_curved(StageArgs<float> a) {
    using G = CurvGeom<Q, C>;
    constexpr int NS = Q * Q * Q, LPT = G::LPT, NR = G::NR, NPR = G::NPR, NN = G::NN, NT = G::NT, NQ = G::NQ;
    extern __shared__ __align__(16) float4 dyn4[];
    __shared__ RowRec crow[Q][Q - 1], cline[Q - 1][NR];
    // trace weights, twice: of the left neighbour l(+1), of the right l(-1), and
    // of an exterior state held in the first place
    __shared__ float2 strace[3][Q];
    const int tid = threadIdx.x;
    float4 *sg = dyn4 + tid;                             // geometry records at sg[i * NT]
    float4 *se = dyn4 + G::NG * NT + tid;                // equilibrium records
    float4 *sw = dyn4 + (G::NG + G::NE) * NT + tid;      // wall densities at the lines' ends in direction 1, as pairs
    float4 *sr = dyn4 + (G::NG + G::NE + LPT) * NT + tid;      // the ring (RING): slot q of component c at sr[((st * SLOTS + q) * C + c) * NT]
    constexpr bool RING = Q == 2 && VEC;
    // after the threads' records: (u1, trapezoid factor) of the first-axis nodes,
    // and the exterior states of direction 1 on the current velocity line
    const int vn1 = a.vg.n[0], vn2 = a.vg.n[1];
    float2 *su1 = reinterpret_cast<float2 *>(dyn4 + (G::NG + G::NE + LPT + (RING ? 2 * G::SLOTS * C : 0)) * NT);
    float2 *sbc = su1 + vn1;                             // [side][component][vn1]
    // plane pairs: thread-local memory, touched once per velocity line
    float Pme[NN * 2 * NQ];
    const VelGrid &vg = a.vg;
    const CurvOps32 &co = a.cops;
    for (int j = tid; j < vn1; j += NT) su1[j] = make_float2(__ldg(a.vtab32 + j).x, trap(j, vn1));
    if (tid < Q * (Q - 1)) {
        const int i = tid / (Q - 1), m = tid % (Q - 1), j = (i + m + 1) % Q;
        crow[i][m].k = make_float4(co.kh[i][j], co.kh[i][j], co.kl[i][j], co.kl[i][j]);
        crow[i][m].lo = make_float4(co.lm[j], co.lm[j], co.lp[j], co.lp[j]);
        crow[i][m].g[0] = dup2(co.dgL[i]);
        crow[i][m].g[1] = dup2(-co.dgR[i]);
    }
    if (tid < (Q - 1) * NR) {
        const int m = tid / NR, r = tid % NR, i0 = 2 * r, i1 = min(2 * r + 1, Q - 1);
        const int j0 = (i0 + m + 1) % Q, j1 = (i1 + m + 1) % Q;
        cline[m][r].k = make_float4(co.kh[i0][j0], co.kh[i1][j1], co.kl[i0][j0], co.kl[i1][j1]);
        cline[m][r].lo = make_float4(co.lm[j0], co.lm[j1], co.lp[j0], co.lp[j1]);
        cline[m][r].g[0] = make_float2(co.dgL[i0], co.dgL[i1]);
        cline[m][r].g[1] = make_float2(-co.dgR[i0], -co.dgR[i1]);
    }
    if (tid < Q) {
        strace[0][tid] = dup2(co.lp[tid]);
        strace[1][tid] = dup2(co.lm[tid]);
        strace[2][tid] = dup2(tid == 0 ? 1.f : 0.f);
    }
    __syncthreads();
    const int n_th = a.mesh.Ne * G::TE;
    const int gt = blockIdx.x * NT + tid;                // thread among all elements' threads
    const bool active = gt < n_th;
    const int th = active ? gt : n_th - 1;               // an idle thread repeats the last one's work, without stores
    const int e = th / G::TE, rr = th - e * G::TE;
    const int jy0 = LPT == Q ? 0 : rr % Q, kz = LPT == Q ? rr : rr / Q;
    const int lin0 = Q * (jy0 + Q * kz);                 // first own node within the element (nodes are consecutive)
    const int own = e * NS + lin0;
    const int vb = blockIdx.y;
    const int k0 = vb * a.Kblk, k1 = min(a.Nu, k0 + a.Kblk);
    // face neighbours: element, or -1 on a boundary face
    int nb[6];
    {
        const int n1 = a.mesh.n[0], n2 = a.mesh.n[1], n3 = a.mesh.n[2];
        const int ec[3] = {e % n1, (e / n1) % n2, e / (n1 * n2)}, es[3] = {1, n1, n1 * n2}, nn[3] = {n1, n2, n3};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            nb[2 * d] = ec[d] > 0 ? e - es[d] : (a.mesh.periodic[d] ? e + (nn[d] - 1) * es[d] : -1);
            nb[2 * d + 1] = ec[d] < nn[d] - 1 ? e + es[d] : (a.mesh.periodic[d] ? e - (nn[d] - 1) * es[d] : -1);
        }
    }
    const size_t slab = (size_t)a.P, comp = (size_t)a.Nu * slab;
    const bool mom = a.part != nullptr;
    const int jc[3] = {(vn1 - 1) / 2, (vn2 - 1) / 2, (vg.n[2] - 1) / 2};
    const float fa = a.a32, fab = a.ab32, fc = a.c32;
    // own node of pair r of line l, lane h
    auto node_of = [&](int l, int r, int h) { return Q * l + (2 * r + h < Q ? 2 * r + h : Q - 1); };
#pragma unroll
    for (int p = 0; p < NPR; ++p) {
        const float4 *ra = reinterpret_cast<const float4 *>(a.eq32 + (size_t)(own + node_of(p / NR, p % NR, 0)) * BGK_NEQ32);
        const float4 *rb = reinterpret_cast<const float4 *>(a.eq32 + (size_t)(own + node_of(p / NR, p % NR, 1)) * BGK_NEQ32);
        const float4 a0 = __ldg(ra), b0 = __ldg(rb), a1 = __ldg(ra + 1), b1 = __ldg(rb + 1);
        se[(6 * p) * NT] = make_float4(a0.x, b0.x, a0.y, b0.y);             // E0, V1
        se[(6 * p + 1) * NT] = make_float4(a0.z, b0.z, a0.w, b0.w);         // A11, 1/tau
        se[(6 * p + 2) * NT] = make_float4(a1.x, b1.x, a1.y, b1.y);         // gamma1, gamma4/2
        se[(6 * p + 3) * NT] = make_float4(a1.z, b1.z, a1.w, b1.w);         // U0_1, G factor
    }
    // a face that is no wall: density 1
#pragma unroll
    for (int l = 0; l < LPT; ++l) {
        float2 w[2];
#pragma unroll
        for (int sd = 0; sd < 2; ++sd)
            w[sd] = nb[sd] < 0 && a.mesh.face_kind[sd] == BGK_FK_DIFFUSE
                        ? __ldg(a.rho_w2 + ((size_t)e * 6 + sd) * Q * Q + jy0 + l + Q * kz) : make_float2(1.f, 0.f);
        sw[l * NT] = make_float4(w[0].x, w[0].y, w[1].x, w[1].y);
    }
    if (mom)
#pragma unroll 1
        for (int q = 0; q < NN * 2 * NQ; ++q) Pme[q] = 0.f;
    int j3cur = -1;
    bool first_plane = true;
    auto flush_plane = [&](int j3) {
        const double c = trap3(j3, vg), t = (float)(j3 - jc[2]);
#pragma unroll 1
        for (int n = 0; n < NN; ++n) {
            float *P = Pme + n * 2 * NQ;
            double d[7];
#pragma unroll
            for (int q = 0; q < 7; ++q) {
                d[q] = 0.0;
                if (q < NQ) {
                    d[q] = (double)P[q] + (double)P[NQ + q];
                    P[q] = 0.f;
                    P[NQ + q] = 0.f;
                }
            }
            plane_to_part(a.part + (size_t)vb * BGK_NMOM * a.P + own + n, a.P, c, t, d, first_plane);
        }
        first_plane = false;
    };

    for (int kl = k0; kl < k1; kl += vn1) {
        const int line = kl / vn1;
        const int j2 = line % vn2, j3 = line / vn2;
        if (mom && active && j3 != j3cur) {
            if (j3cur >= 0) flush_plane(j3cur);
            j3cur = j3;
        }
        // ---- per velocity line: the u_2, u_3 parts of every u . S, and the
        // equilibrium's line constants
        {
            if (!a.mesh.periodic[0]) {                   // (closed along direction 1: every thread, uniform)
                __syncthreads();
                for (int i = tid; i < 2 * C * vn1; i += NT) {
                    const int q = i / vn1, j = i - q * vn1;
                    sbc[i] = __ldg(a.bc2 + (size_t)q * a.Nu + kl + j);
                }
                __syncthreads();
            }
            const float4 vl = __ldg(a.vtab32 + kl);
            const float u2 = vl.y, u3 = vl.z;
            const float *gp = a.geop + th;
#pragma unroll 4
            for (int i = 0; i < G::NG; ++i) {
                float s[2], b[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const size_t o = (size_t)(2 * i + h) * 3 * n_th;
                    s[h] = __ldg(gp + o);
                    b[h] = fmaf(u2, __ldg(gp + o + n_th), u3 * __ldg(gp + o + 2 * (size_t)n_th));
                }
                sg[i * NT] = make_float4(s[0], s[1], b[0], b[1]);
            }
#pragma unroll
            for (int p = 0; p < NPR; ++p) {
                float lc[2][4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int nd = own + node_of(p / NR, p % NR, h);
                    const float4 *rec = reinterpret_cast<const float4 *>(a.eq32 + (size_t)nd * BGK_NEQ32);
                    const float4 r2 = __ldg(rec + 2), r3 = __ldg(rec + 3), r4 = __ldg(rec + 4), r5 = __ldg(rec + 5);
                    Eq32 q;
                    q.V2 = r2.x; q.V3 = r2.y; q.A12 = r2.z; q.A13 = r2.w;
                    q.A22 = r3.x; q.A23 = r3.y; q.A33 = r3.z;
                    q.line(u2, u3, lc[h][0], lc[h][1]);
                    const float t2 = u2 - r4.z, t3 = u3 - r4.w;
                    lc[h][2] = fmaf(r4.x, t2, fmaf(r4.y, t3, fmaf(0.5f * r5.x, fmaf(t2, t2, t3 * t3), r3.w)));
                    lc[h][3] = __ldg(a.geo + (size_t)nd * BGK_NGEO32 + 9);
                }
                se[(6 * p + 4) * NT] = make_float4(lc[0][0], lc[1][0], lc[0][1], lc[1][1]);
                se[(6 * p + 5) * NT] = make_float4(lc[0][2], lc[1][2], lc[0][3], lc[1][3]);
            }
        }
        // line sums of each pair of nodes: F, F jt, F jt^2, G with their errors
        P2 L[NPR][C == 2 ? 4 : 3], E[NPR][C == 2 ? 4 : 3];
#pragma unroll
        for (int p = 0; p < NPR; ++p)
#pragma unroll
            for (int q = 0; q < (C == 2 ? 4 : 3); ++q) L[p][q] = E[p][q] = dup2(0.f);
        // the faces' normal velocities at first-axis node j: FX (left, right) of a
        // line, FY and FZ [side]; and which directions have inflow on which side
        struct Faces {
            P2 FX[LPT], FY[2][NR], FZ[2][LPT][NR];
            bool inL[3], inR[3];
        };
        auto us_at = [&](P2 u, int i) {
            const float4 t = sg[i * NT];
            return __ffma2_rn(u, make_float2(t.x, t.y), make_float2(t.z, t.w));
        };
        auto faces = [&](int j, Faces &A) {
            const P2 u = dup2(su1[j].x);
#pragma unroll
            for (int d = 0; d < 3; ++d) A.inL[d] = A.inR[d] = false;
#pragma unroll
            for (int l = 0; l < LPT; ++l) {
                A.FX[l] = us_at(u, G::O_FX + l);
                A.inL[0] |= A.FX[l].x > 0.f; A.inR[0] |= A.FX[l].y < 0.f;
            }
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                A.FY[0][r] = us_at(u, G::O_FY + r);
                A.FY[1][r] = us_at(u, G::O_FY + NR + r);
                A.inL[1] |= fmaxf(A.FY[0][r].x, A.FY[0][r].y) > 0.f;
                A.inR[1] |= fminf(A.FY[1][r].x, A.FY[1][r].y) < 0.f;
            }
#pragma unroll
            for (int l = 0; l < LPT; ++l)
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    A.FZ[0][l][r] = us_at(u, G::O_FZ + l * NR + r);
                    A.FZ[1][l][r] = us_at(u, G::O_FZ + NPR + l * NR + r);
                    A.inL[2] |= fmaxf(A.FZ[0][l][r].x, A.FZ[0][l][r].y) > 0.f;
                    A.inR[2] |= fminf(A.FZ[1][l][r].x, A.FZ[1][l][r].y) < 0.f;
                }
        };
        // RING: request the values of velocity kl + j into ring stage st: own, and
        // per direction those of the side with inflow (the left one first)
        auto request = [&](int j, const Faces &A, int st) {
            const float *fk = a.f_s + (size_t)(kl + j) * slab;
            auto cp = [&](int q, int c, const float *p) {
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_u32(sr + ((st * G::SLOTS + q) * C + c) * NT)), "l"(p) : "memory");
            };
            const int ne[3] = {A.inL[0] ? nb[0] : A.inR[0] ? nb[1] : -1, A.inL[1] ? nb[2] : A.inR[1] ? nb[3] : -1,
                               A.inL[2] ? nb[4] : A.inR[2] ? nb[5] : -1};
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const float *fc_ = fk + c * comp;
                cp(0, c, fc_ + own);
                if (ne[0] >= 0) cp(1, c, fc_ + (size_t)ne[0] * NS + lin0);
                if (ne[1] >= 0) cp(2, c, fc_ + (size_t)ne[1] * NS + Q * Q * kz);
                if (ne[2] >= 0) {
                    cp(3, c, fc_ + (size_t)ne[2] * NS);
                    cp(4, c, fc_ + (size_t)ne[2] * NS + Q * Q);
                }
            }
        };
        Faces A;
        if constexpr (RING) {
            faces(0, A);
            request(0, A, 0);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        float jt1 = (float)(-jc[0]);
        for (int j1 = 0; j1 < vn1; ++j1, jt1 += 1.f) {
            const int k = kl + j1;
            const float u1 = su1[j1].x;
            const P2 u12 = dup2(u1);
            const float *fk = a.f_s + (size_t)k * slab;
            auto us = [&](int i) { return us_at(u12, i); };      // the pair of scalars u . S of record i
            Faces An;
            if constexpr (RING) {
                if (j1 + 1 < vn1) {
                    faces(j1 + 1, An);
                    request(j1 + 1, An, (j1 + 1) & 1);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
                asm volatile("cp.async.wait_group 1;" ::: "memory");
                __syncwarp();                            // the partner plane's values are another lane's
            } else {
                // no ring: the own values two velocities ahead on their way to L2
                if (k + 2 < k1) {
#pragma unroll
                    for (int c = 0; c < C; ++c) asm volatile("prefetch.global.L2 [%0];" ::"l"(fk + c * comp + 2 * slab + own));
                }
                faces(j1, A);
            }
            const P2 (&FX)[LPT] = A.FX;
            const P2 (&FY)[2][NR] = A.FY;
            const P2 (&FZ)[2][LPT][NR] = A.FZ;
            const bool (&inL)[3] = A.inL, (&inR)[3] = A.inR;
            constexpr int NB = G::BOTH ? 2 : 1;
            P2 F[C][LPT][NR], T[C][LPT][NR], FN[C][LPT][NR];
            if (RING && fa != 0.f) {
#pragma unroll
                for (int c = 0; c < C; ++c) ld_lines<Q, LPT, VEC>(a.f_n + c * comp + (size_t)k * slab + own, FN[c]);
            }
            P2 X[NB][C][LPT][NR], Y[NB][C][Q][NR], Z[NB][Q][C][LPT][NR];
            P2 OZ[Q - 1][C][LPT][NR], OY[C][LPT == Q ? 1 : Q - 1][1][NR];
            // RING: two lines (16 bytes) from slot q, of this thread or the lane `of`
            auto slot = [&](int q, int c, int of, P2 (&v)[LPT][NR]) {
                const float4 t = sr[(((j1 & 1) * G::SLOTS + q) * C + c) * NT + of];
                v[0][0] = make_float2(t.x, t.y);
                v[LPT - 1][0] = make_float2(t.z, t.w);
            };
            // the exterior value (a Dirichlet state, or the wall's Maxwellian
            // times its density; closed faces have no flux, their face vectors
            // are zero): the product of two pairs, rounded once more
            auto pair_prod = [](float2 b, float2 w) {
                const float p = __fmul_rn(b.x, w.x);
                return __fadd_rn(p, fmaf(b.x, w.y, fmaf(b.y, w.x, fmaf(b.x, w.x, -p))));
            };
            auto exterior = [&](int fc, int fp, int c) {
                const float2 b = __ldg(a.bc2 + ((size_t)fc * C + c) * a.Nu + k);
                if (a.mesh.face_kind[fc] != BGK_FK_DIFFUSE) return b.x;
                return pair_prod(b, __ldg(a.rho_w2 + ((size_t)e * 6 + fc) * Q * Q + fp));
            };
            // the values behind face side sd of direction 1, 2, 3: the
            // neighbour's, or the exterior state in the first place of a line
            // (direction 1: from shared memory, where it is used)
            auto ld_x = [&](int ne, P2 (&v)[C][LPT][NR]) {
                if (ne >= 0) {
#pragma unroll
                    for (int c = 0; c < C; ++c) ld_lines<Q, LPT, VEC>(fk + c * comp + (size_t)ne * NS + lin0, v[c]);
                }
            };
            auto ld_y = [&](int sd, int ne, P2 (&v)[C][Q][NR]) {
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    if (ne >= 0) {
                        ld_lines<Q, Q, VEC>(fk + c * comp + (size_t)ne * NS + Q * Q * kz, v[c]);
                    } else {
#pragma unroll
                        for (int j = 0; j < Q; ++j)
#pragma unroll
                            for (int r = 0; r < NR; ++r)
                                v[c][j][r] = j ? dup2(0.f) : make_float2(exterior(2 + sd, node_of(0, r, 0) + Q * kz, c),
                                                                         exterior(2 + sd, node_of(0, r, 1) + Q * kz, c));
                    }
                }
            };
            auto ld_z = [&](int sd, int ne, P2 (&v)[Q][C][LPT][NR]) {
#pragma unroll
                for (int j = 0; j < Q; ++j)
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        if (ne >= 0) {
                            ld_lines<Q, LPT, VEC>(fk + c * comp + (size_t)ne * NS + Q * (jy0 + Q * j), v[j][c]);
                        } else {
#pragma unroll
                            for (int l = 0; l < LPT; ++l)
#pragma unroll
                                for (int r = 0; r < NR; ++r)
                                    v[j][c][l][r] = j ? dup2(0.f)
                                                      : make_float2(exterior(4 + sd, node_of(0, r, 0) + Q * (jy0 + l), c),
                                                                    exterior(4 + sd, node_of(0, r, 1) + Q * (jy0 + l), c));
                        }
                    }
            };
            const int s0[3] = {inL[0] ? 0 : 1, inL[1] ? 0 : 1, inL[2] ? 0 : 1};       // (not BOTH) the side first read
            if constexpr (RING) {
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    slot(0, c, 0, F[c]);
                    slot(0, c, (tid ^ 1) - tid, OZ[0][c]);
                    slot(1, c, 0, X[0][c]);
                    slot(2, c, 0, *reinterpret_cast<P2 (*)[LPT][NR]>(&Y[0][c]));
                    slot(3, c, 0, Z[0][0][c]);
                    slot(4, c, 0, Z[0][Q - 1][c]);
                }
                // boundary faces of directions 2 and 3 (direction 1's come from shared memory)
                if ((inL[1] && nb[2] < 0) || (inR[1] && !inL[1] && nb[3] < 0)) ld_y(s0[1], -1, Y[0]);
                if ((inL[2] && nb[4] < 0) || (inR[2] && !inL[2] && nb[5] < 0)) ld_z(s0[2], -1, Z[0]);
            } else {
#pragma unroll
                for (int c = 0; c < C; ++c) ld_lines<Q, LPT, VEC>(fk + c * comp + own, F[c]);
                if constexpr (G::BOTH) {
                    // a side without inflow reads the element itself (in cache, and
                    // finite; its inflow velocity is zero): no branch around loads
                    auto from = [&](bool in, int ne) { return in && ne >= 0 ? ne : e; };
                    ld_x(from(inL[0], nb[0]), X[0]);
                    ld_x(from(inR[0], nb[1]), X[NB - 1]);
                    ld_y(0, inL[1] ? nb[2] : e, Y[0]);
                    ld_y(1, inR[1] ? nb[3] : e, Y[NB - 1]);
                    ld_z(0, inL[2] ? nb[4] : e, Z[0]);
                    ld_z(1, inR[2] ? nb[5] : e, Z[NB - 1]);
                } else {
                    if (inL[0] || inR[0]) ld_x(s0[0] ? nb[1] : nb[0], X[0]);
                    if (inL[1] || inR[1]) ld_y(s0[1], s0[1] ? nb[3] : nb[2], Y[0]);
                    if (inL[2] || inR[2]) ld_z(s0[2], s0[2] ? nb[5] : nb[4], Z[0]);
                }
                // the element's other planes and the plane's other lines
#pragma unroll
                for (int m = 1; m < Q; ++m)
#pragma unroll
                    for (int c = 0; c < C; ++c)
                        ld_lines<Q, LPT, VEC>(fk + c * comp + (size_t)e * NS + Q * (jy0 + Q * ((kz + m) % Q)), OZ[m - 1][c]);
                if constexpr (LPT != Q) {
#pragma unroll
                    for (int m = 1; m < Q; ++m)
#pragma unroll
                        for (int c = 0; c < C; ++c)
                            ld_lines<Q, 1, VEC>(fk + c * comp + (size_t)e * NS + Q * ((jy0 + m) % Q + Q * kz), OY[c][m - 1]);
                }
                if (fa != 0.f) {
#pragma unroll
                    for (int c = 0; c < C; ++c) ld_lines<Q, LPT, VEC>(a.f_n + c * comp + (size_t)k * slab + own, FN[c]);
                }
            }
            // coefficient of a pair's deviations: the volume term (with defects)
            // and the outflow faces' own traces, gl = g_L' min(A_L, 0), gr = g_R' max(A_R, 0)
            auto coef = [&](const RowRec &w, P2 aj, P2 gl, P2 gr) {
                P2 c = __ffma2_rn(make_float2(w.k.x, w.k.y), aj, __fmul2_rn(make_float2(w.k.z, w.k.w), aj));
                c = __ffma2_rn(gr, make_float2(w.lo.z, w.lo.w), c);
                return __ffma2_rn(gl, make_float2(w.lo.x, w.lo.y), c);
            };
            auto neg_part = [](P2 v) { return make_float2(fminf(v.x, 0.f), fminf(v.y, 0.f)); };
            auto neg_of_neg = [](P2 v) { return make_float2(fminf(-v.x, 0.f), fminf(-v.y, 0.f)); };
            // inflow speed through side sd from its face velocities L or R
            auto inflow = [](int sd, P2 vL, P2 vR) {
                return make_float2(fmaxf(sd ? -vR.x : vL.x, 0.f), fmaxf(sd ? -vR.y : vL.y, 0.f));
            };
            // ---- first direction: the thread's own lines
#pragma unroll
            for (int l = 0; l < LPT; ++l) {
                const P2 oL = dup2(fminf(FX[l].x, 0.f)), oR = dup2(fminf(-FX[l].y, 0.f));
#pragma unroll
                for (int m = 1; m < Q; ++m)
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        const RowRec w = cline[m - 1][r];
                        const P2 cf = coef(w, us(G::O_A1 + (l * (Q - 1) + m - 1) * NR + r), __fmul2_rn(w.g[0], oL),
                                           __fmul2_rn(w.g[1], oR));
                        const int i0 = 2 * r, i1 = 2 * r + 1 < Q ? 2 * r + 1 : Q - 1;
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            const P2 fj = make_float2(lane_of(F[c][l], (i0 + m) % Q), lane_of(F[c][l], (i1 + m) % Q));
                            const P2 df = sub2(fj, F[c][l][r]);
                            T[c][l][r] = m == 1 ? __fmul2_rn(cf, df) : __ffma2_rn(cf, df, T[c][l][r]);
                        }
                    }
            }
            // inflow of side sd: g' A times (outer trace - f_i), A its inflow part
            auto in_x = [&](int sd, P2 (&v)[C][LPT][NR]) {
                const float2 *w = strace[(sd ? nb[1] : nb[0]) < 0 ? 2 : sd];
                if ((sd ? nb[1] : nb[0]) < 0) {
#pragma unroll
                    for (int l = 0; l < LPT; ++l) {
                        const float4 rw = sw[l * NT];
#pragma unroll
                        for (int c = 0; c < C; ++c) {
#pragma unroll
                            for (int r = 0; r < NR; ++r) v[c][l][r] = dup2(0.f);
                            v[c][l][0].x = pair_prod(sbc[(sd * C + c) * vn1 + j1], sd ? make_float2(rw.z, rw.w) : make_float2(rw.x, rw.y));
                        }
                    }
                }
#pragma unroll
                for (int l = 0; l < LPT; ++l) {
                    const P2 A = dup2(fmaxf(sd ? -FX[l].y : FX[l].x, 0.f));
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        const P2 gA = __fmul2_rn(cline[0][r].g[sd], A);
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            P2 q;
#pragma unroll
                            for (int j = 0; j < Q; ++j) {
                                const P2 dv = sub2(dup2(lane_of(v[c][l], j)), F[c][l][r]);
                                q = j == 0 ? __fmul2_rn(w[0], dv) : __ffma2_rn(w[j], dv, q);
                            }
                            T[c][l][r] = __ffma2_rn(gA, q, T[c][l][r]);
                        }
                    }
                }
            };
            if constexpr (G::BOTH) {
                if (__any_sync(0xffffffffu, inL[0])) in_x(0, X[0]);
                if (__any_sync(0xffffffffu, inR[0])) in_x(1, X[NB - 1]);
            } else {
                if (inL[0] || inR[0]) in_x(s0[0], X[0]);
                if (inL[0] && inR[0]) {
                    ld_x(nb[1], X[0]);
                    in_x(1, X[0]);
                }
            }
            // ---- second direction: lines across the element's rows of lines
#pragma unroll
            for (int l = 0; l < LPT; ++l)
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const RowRec *row = crow[LPT == Q ? l : jy0];
                    const P2 gl = __fmul2_rn(row[0].g[0], neg_part(FY[0][r])), gr = __fmul2_rn(row[0].g[1], neg_of_neg(FY[1][r]));
#pragma unroll
                    for (int m = 1; m < Q; ++m) {
                        const P2 cf = coef(row[m - 1], us(G::O_A2 + (l * (Q - 1) + m - 1) * NR + r), gl, gr);
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            const P2 fj = LPT == Q ? F[c][(l + m) % LPT][r] : OY[c][LPT == Q ? 0 : m - 1][0][r];
                            T[c][l][r] = __ffma2_rn(cf, sub2(fj, F[c][l][r]), T[c][l][r]);
                        }
                    }
                }
            auto in_y = [&](int sd, const P2 (&v)[C][Q][NR]) {
                const float2 *w = strace[(sd ? nb[3] : nb[2]) < 0 ? 2 : sd];
#pragma unroll
                for (int l = 0; l < LPT; ++l) {
                    const P2 g = crow[LPT == Q ? l : jy0][0].g[sd];
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        const P2 gA = __fmul2_rn(g, inflow(sd, FY[0][r], FY[1][r]));
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            P2 q;
#pragma unroll
                            for (int j = 0; j < Q; ++j) {
                                const P2 dv = sub2(v[c][j][r], F[c][l][r]);
                                q = j == 0 ? __fmul2_rn(w[0], dv) : __ffma2_rn(w[j], dv, q);
                            }
                            T[c][l][r] = __ffma2_rn(gA, q, T[c][l][r]);
                        }
                    }
                }
            };
            if constexpr (G::BOTH) {
                if (__any_sync(0xffffffffu, inL[1])) in_y(0, Y[0]);
                if (__any_sync(0xffffffffu, inR[1])) in_y(1, Y[NB - 1]);
            } else {
                if (inL[1] || inR[1]) in_y(s0[1], Y[0]);
                if (inL[1] && inR[1]) {
                    ld_y(1, nb[3], Y[0]);
                    in_y(1, Y[0]);
                }
            }
            // ---- third direction: lines across the element's planes
#pragma unroll
            for (int l = 0; l < LPT; ++l)
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const RowRec *row = crow[kz];
                    const P2 gl = __fmul2_rn(row[0].g[0], neg_part(FZ[0][l][r])), gr = __fmul2_rn(row[0].g[1], neg_of_neg(FZ[1][l][r]));
#pragma unroll
                    for (int m = 1; m < Q; ++m) {
                        const P2 cf = coef(row[m - 1], us(G::O_A3 + ((m - 1) * LPT + l) * NR + r), gl, gr);
#pragma unroll
                        for (int c = 0; c < C; ++c) T[c][l][r] = __ffma2_rn(cf, sub2(OZ[m - 1][c][l][r], F[c][l][r]), T[c][l][r]);
                    }
                }
            auto in_z = [&](int sd, const P2 (&v)[Q][C][LPT][NR]) {
                const float2 *w = strace[(sd ? nb[5] : nb[4]) < 0 ? 2 : sd];
                const P2 g = crow[kz][0].g[sd];
#pragma unroll
                for (int l = 0; l < LPT; ++l)
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        const P2 gA = __fmul2_rn(g, inflow(sd, FZ[0][l][r], FZ[1][l][r]));
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            P2 q;
#pragma unroll
                            for (int j = 0; j < Q; ++j) {
                                const P2 dv = sub2(v[j][c][l][r], F[c][l][r]);
                                q = j == 0 ? __fmul2_rn(w[0], dv) : __ffma2_rn(w[j], dv, q);
                            }
                            T[c][l][r] = __ffma2_rn(gA, q, T[c][l][r]);
                        }
                    }
            };
            if constexpr (G::BOTH) {
                if (__any_sync(0xffffffffu, inL[2])) in_z(0, Z[0]);
                if (__any_sync(0xffffffffu, inR[2])) in_z(1, Z[NB - 1]);
            } else {
                if (inL[2] || inR[2]) in_z(s0[2], Z[0]);
                if (inL[2] && inR[2]) {
                    ld_z(1, nb[5], Z[0]);
                    in_z(1, Z[0]);
                }
            }
            // ---- equilibrium, source, Runge--Kutta update, moments
            const float cj = su1[j1].y;
            float out[C][NN];
#pragma unroll
            for (int p = 0; p < NPR; ++p) {
                const int l = p / NR, r = p % NR;
                const float4 e0 = se[(6 * p) * NT], e1 = se[(6 * p + 1) * NT], e2 = se[(6 * p + 2) * NT], e3 = se[(6 * p + 3) * NT];
                const float4 e4 = se[(6 * p + 4) * NT], e5 = se[(6 * p + 5) * NT];
                const P2 c1 = sub2(u12, make_float2(e0.z, e0.w));
                const P2 ex = __ffma2_rn(c1, __ffma2_rn(make_float2(e1.x, e1.y), c1, make_float2(e4.x, e4.y)), make_float2(e4.z, e4.w));
                const P2 g32 = __fmul2_rn(make_float2(e0.x, e0.y), make_float2(Eq32::ex2(ex.x), Eq32::ex2(ex.y)));
                const P2 t1 = sub2(u12, make_float2(e3.x, e3.y));
                const P2 gc = __fmul2_rn(g32, __ffma2_rn(t1, __ffma2_rn(make_float2(e2.z, e2.w), t1, make_float2(e2.x, e2.y)),
                                                         make_float2(e5.x, e5.y)));
                const P2 uH = us(G::O_H + p), it = make_float2(e1.z, e1.w), ij = make_float2(e5.z, e5.w), gf = make_float2(e3.z, e3.w);
                P2 o[C];
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const P2 f = F[c][l][r];
                    const P2 div = __fmul2_rn(ij, __ffma2_rn(uH, f, T[c][l][r]));
                    const P2 eqv = c ? __fmul2_rn(gf, g32) : g32, eqc = c ? __fmul2_rn(gf, gc) : gc;
                    const P2 R = __ffma2_rn(sub2(eqv, f), it, sub2(__fmul2_rn(eqc, it), div));
                    o[c] = rk_update2(f, fa != 0.f ? FN[c][l][r] : dup2(0.f), R, fa, fab, fc, fa != 0.f);
                    out[c][node_of(l, r, 0)] = o[c].x;
                    if (2 * r + 1 < Q) out[c][node_of(l, r, 1)] = o[c].y;
                }
                if (mom) {
                    // the line kernels' error-free sums (LineAcc), two nodes at once
                    const P2 cF = __fmul2_rn(dup2(cj), o[0]);
                    sum2x2(L[p][0], E[p][0], cF);
                    const P2 p1 = __fmul2_rn(cF, dup2(jt1));
                    sum2x2(L[p][1], E[p][1], p1);
                    E[p][1] = sub2(E[p][1], __ffma2_rn(cF, dup2(-jt1), p1));
                    const float jj = __fmul_rn(jt1, jt1), njj = -jj;                 // exact
                    const P2 p2 = __fmul2_rn(cF, dup2(jj));
                    sum2x2(L[p][2], E[p][2], p2);
                    E[p][2] = sub2(E[p][2], __ffma2_rn(cF, dup2(njj), p2));
                    if (C == 2) sum2x2(L[p][C == 2 ? 3 : 0], E[p][C == 2 ? 3 : 0], __fmul2_rn(dup2(cj), o[C - 1]));
                }
            }
            if (active) {
                float *ok = a.f_out + (size_t)k * slab + own;
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    if constexpr (VEC && NN % 4 == 0) {
#pragma unroll
                        for (int n = 0; n < NN; n += 4)
                            *reinterpret_cast<float4 *>(ok + c * comp + n) = make_float4(out[c][n], out[c][n + 1], out[c][n + 2], out[c][n + 3]);
                    } else {
#pragma unroll
                        for (int n = 0; n < NN; ++n) ok[c * comp + n] = out[c][n];
                    }
                }
            }
            if constexpr (RING) {
                __syncwarp();                            // the partner has read this stage before it is filled again
                A = An;
            }
        }
        if (mom && active) {
            // end of the line: c2 jt2^b (line pair) into the plane pairs
            const float c2 = trap(j2, vn2), jt2 = (float)(j2 - jc[1]);
            const float bq = __fmul_rn(c2, jt2), bbq = __fmul_rn(bq, jt2);
#pragma unroll
            for (int n = 0; n < NN; ++n) {
                const int p = (n / Q) * NR + (n % Q) / 2, h = (n % Q) % 2;
                auto ln = [&](int q) { return h ? L[p][q].y : L[p][q].x; };
                auto er = [&](int q) { return h ? E[p][q].y : E[p][q].x; };
                float *P = Pme + n * 2 * NQ;
                plane_add_s<NQ>(P, 1, 0, c2, ln(0), er(0));
                plane_add_s<NQ>(P, 1, 1, c2, ln(1), er(1));
                plane_add_s<NQ>(P, 1, 2, c2, ln(2), er(2));
                plane_add_s<NQ>(P, 1, 3, bq, ln(0), er(0));
                plane_add_s<NQ>(P, 1, 4, bq, ln(1), er(1));
                plane_add_s<NQ>(P, 1, 5, bbq, ln(0), er(0));
                if (C == 2) plane_add_s<NQ>(P, 1, NQ - 1, c2, ln(C == 2 ? 3 : 0), er(C == 2 ? 3 : 0));
            }
        }
    }
    if (mom && active) {
        if (j3cur >= 0) flush_plane(j3cur);
        const double uc[3] = {vg.lo[0] + jc[0] * vg.h[0], vg.lo[1] + jc[1] * vg.h[1], vg.lo[2] + jc[2] * vg.h[2]};
        for (int n = 0; n < NN; ++n) raw_in_place(a.part + (size_t)vb * BGK_NMOM * a.P + own + n, a.P, vg, uc);
    }
}

template <int Q, int C, bool VEC>
cudaError_t curved_launch(const StageArgs<float> &a, int n_vblk, cudaStream_t s) {
    using G = CurvGeom<Q, C>;
    const size_t smem = G::template smem<Q == 2 && VEC>(a.vg.n[0]);
    static SmemLimit lim;
    size_t *attr = lim.slot();
    if (!attr) return cudaErrorInvalidDevice;
    if (smem > *attr) {
        const cudaError_t e = cudaFuncSetAttribute(k_stage_f32_curved<Q, C, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)smem);
        if (e != cudaSuccess) return e;
        *attr = smem;
    }
    const dim3 grid((a.mesh.Ne * G::TE + G::NT - 1) / G::NT, n_vblk);
    k_stage_f32_curved<Q, C, VEC><<<grid, G::NT, smem, s>>>(a);
    return cudaGetLastError();
}

template <int Q>
cudaError_t curved_q(const StageArgs<float> &a, int C, int n_vblk, cudaStream_t s) {
    // vector loads and stores need 16-byte aligned buffers (the caller's, in
    // bgk_stage) and whole 16-byte lines; at Q = 3, 5 there are none
    const auto al = [](const void *p) { return ((uintptr_t)p & 15u) == 0; };
    if constexpr (Q % 2 == 0) {
        if (al(a.f_s) && al(a.f_out) && (a.a32 == 0.f || al(a.f_n)))
            return C == 1 ? curved_launch<Q, 1, true>(a, n_vblk, s) : curved_launch<Q, 2, true>(a, n_vblk, s);
    }
    return C == 1 ? curved_launch<Q, 1, false>(a, n_vblk, s) : curved_launch<Q, 2, false>(a, n_vblk, s);
}

template <int Q>
void geop_fill(const float *geo32, const float *fvec32, const MeshInfo &mesh, const CurvOps32 &co, std::vector<float> &out) {
    using G = CurvGeom<Q, 1>;
    constexpr int NS = Q * Q * Q;
    const size_t n_th = (size_t)mesh.Ne * G::TE;
    out.assign((size_t)2 * G::NG * 3 * n_th, 0.f);
    for (size_t th = 0; th < n_th; ++th) {
        const int e = (int)(th / G::TE), r = (int)(th % G::TE);
        const int jy0 = G::LPT == Q ? 0 : r % Q, kz = G::LPT == Q ? r : r / Q;
        // closed faces: no flux, F^I = 0; with the face vector taken as zero the
        // only trace left of it is its share of H
        const int ec[3] = {e % mesh.n[0], (e / mesh.n[0]) % mesh.n[1], e / (mesh.n[0] * mesh.n[1])};
        bool closed[6];
        for (int f = 0; f < 6; ++f)
            closed[f] = !mesh.periodic[f / 2] && mesh.face_kind[f] == BGK_FK_CLOSED &&
                        ec[f / 2] == (f % 2 ? mesh.n[f / 2] - 1 : 0);
        const float zero[3] = {0.f, 0.f, 0.f};
        auto put = [&](int i, const float *v) {
            for (int c = 0; c < 3; ++c) out[((size_t)i * 3 + c) * n_th + th] = v[c];
        };
        auto node = [&](int i, int j, int k) { return geo32 + ((size_t)e * NS + i + Q * (j + Q * k)) * BGK_NGEO32; };
        auto fvec = [&](int f, int p) { return fvec32 + (((size_t)e * 6 + f) * Q * Q + p) * 3; };
        auto face = [&](int f, int p) { return closed[f] ? zero : fvec(f, p); };
        auto rest = [&](int o, int i, int j, int k) {
            const int id[3] = {i, j, k}, fp[3] = {j + Q * k, i + Q * k, i + Q * j};
            float H[3];
            for (int c = 0; c < 3; ++c) {
                double h = node(i, j, k)[28 + c];
                for (int f = 0; f < 6; ++f)
                    if (closed[f])
                        h -= (double)(f % 2 ? co.dgR[id[f / 2]] : co.dgL[id[f / 2]]) * (double)fvec(f, fp[f / 2])[c];
                H[c] = (float)h;
            }
            put(o, H);
        };
        // record i: two scalars, of the nodes (or faces) of a pair's lanes
        auto two = [&](int i, const float *v0, const float *v1) { put(2 * i, v0); put(2 * i + 1, v1); };
        for (int l = 0; l < G::LPT; ++l) {
            const int j = jy0 + l;
            two(G::O_FX + l, face(0, j + Q * kz), face(1, j + Q * kz));
            for (int r = 0; r < G::NR; ++r) {
                const int i0 = 2 * r, i1 = 2 * r + 1 < Q ? 2 * r + 1 : Q - 1;
                for (int m = 1; m < Q; ++m) {
                    two(G::O_A1 + (l * (Q - 1) + m - 1) * G::NR + r, node((i0 + m) % Q, j, kz), node((i1 + m) % Q, j, kz));
                    two(G::O_A2 + (l * (Q - 1) + m - 1) * G::NR + r, node(i0, (j + m) % Q, kz) + 3, node(i1, (j + m) % Q, kz) + 3);
                    two(G::O_A3 + ((m - 1) * G::LPT + l) * G::NR + r, node(i0, j, (kz + m) % Q) + 6, node(i1, j, (kz + m) % Q) + 6);
                }
                two(G::O_FZ + l * G::NR + r, face(4, i0 + Q * j), face(4, i1 + Q * j));
                two(G::O_FZ + G::NPR + l * G::NR + r, face(5, i0 + Q * j), face(5, i1 + Q * j));
                rest(2 * (G::O_H + l * G::NR + r), i0, j, kz);
                rest(2 * (G::O_H + l * G::NR + r) + 1, i1, j, kz);
            }
        }
        for (int r = 0; r < G::NR; ++r) {
            const int i0 = 2 * r, i1 = 2 * r + 1 < Q ? 2 * r + 1 : Q - 1;
            two(G::O_FY + r, face(2, i0 + Q * kz), face(2, i1 + Q * kz));
            two(G::O_FY + G::NR + r, face(3, i0 + Q * kz), face(3, i1 + Q * kz));
        }
    }
}

}  // namespace

void curved_geop(int q, const float *geo32, const float *fvec32, const MeshInfo &mesh, const CurvOps32 &co, std::vector<float> &out) {
    switch (q) {
        case 2: geop_fill<2>(geo32, fvec32, mesh, co, out); break;
        case 3: geop_fill<3>(geo32, fvec32, mesh, co, out); break;
        case 4: geop_fill<4>(geo32, fvec32, mesh, co, out); break;
        case 5: geop_fill<5>(geo32, fvec32, mesh, co, out); break;
    }
}

cudaError_t launch_stage_f32_curved(const StageArgs<float> &a, int C, int n_vblk, cudaStream_t s) {
    switch (a.fr.q) {
        case 2: return curved_q<2>(a, C, n_vblk, s);
        case 3: return curved_q<3>(a, C, n_vblk, s);
        case 4: return curved_q<4>(a, C, n_vblk, s);
        case 5: return C == 1 ? curved_launch<5, 1, false>(a, n_vblk, s) : cudaErrorInvalidValue;   // F and G: k_stage_f32
        default: return cudaErrorInvalidValue;
    }
}
