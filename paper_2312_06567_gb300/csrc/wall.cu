// Diffuse-wall densities (section "Implementation & problem setup": the wall
// is a weak boundary whose exterior state enters through the upwind flux).
// At every flux node of a diffuse face the particles entering the gas
// (u_n < 0, n the outward normal of the gas) are drawn from the wall
// Maxwellian rho_w M(u; U_w, theta_w); rho_w makes the node's net discrete
// mass flux vanish:
//     rho_w = - sum_{u_n > 0} w u_n F^- / sum_{u_n < 0} w u_n M(u; U_w, theta_w)
// with F^- the element's interior trace.
//
// The FP64 pipe bounds the kernel (the O-grid's wall elements, 144 x 8 nodes at
// 64,000 velocities, are 0.3 GB or 45 us of reading; their FP64 instructions
// take 0.35 ms), so the work is laid out to issue few of them: a thread keeps
// its first velocity index, so u1 n1 of its face points is formed once and u . n
// costs two FMAs; the weight goes into the Q trace coefficients; the sign of
// u . n is read from its bits; an FP32 value is widened by integer
// instructions; and at p = 1 one FMA goes into whichever sum the velocity
// belongs to, without a branch.  A cluster of WS blocks per (wall element, face)
// splits the velocities, so that a few dozen wall faces fill the GPU, and adds
// its partial sums through distributed shared memory in a fixed order.
// Mixed O-grid with 144 wall faces, p = 1, 40^3: 0.95 -> 0.43 ms; with 36 faces,
// 24^3, p = 1 / 2 / 3 / 4: 217 / 552 / 1056 / 1880 -> 40 / 120 / 184 / 557 us
// (FP64 form 195 / 494 / 895 / 1545 -> 45 / 121 / 194 / 449).
#include <cooperative_groups.h>

#include "bgk_internal.cuh"

namespace {

namespace cg = cooperative_groups;

constexpr int WT = 256, WS = 4;      // threads of a block, blocks of a cluster

template <typename T, int Q>
__global__ void __cluster_dims__(WS, 1, 1) __launch_bounds__(WT)
k_wall_density(const T *f, const T *fvec, const double *bcval, const double *vtab, const int *wall_ef, int Ne,
               int Nu, int n1, int C, FROps fr, double *rho_w, float2 *rho_w2) {
    constexpr int NS = Q * Q * Q, NF = Q * Q;
    constexpr bool KEEP = Q < 5;         // u1 n1 kept in registers (p = 4: would spill)
    __shared__ double red[WT / 32][2 * NF], part[2 * NF];
    __shared__ double nv[NF][3];
    __shared__ double lwr[Q];
    cg::cluster_group cluster = cg::this_cluster();
    const int wf = blockIdx.x / WS, split = blockIdx.x % WS;
    const int e = wall_ef[2 * wf], face = wall_ef[2 * wf + 1];
    const int d = face / 2, side = face % 2;
    for (int i = threadIdx.x; i < NF * 3; i += WT)
        nv[i / 3][i % 3] = (side ? 1.0 : -1.0) * (double)fvec[((size_t)e * 6 + face) * NF * 3 + i];
    if (threadIdx.x < Q) lwr[threadIdx.x] = side ? fr.lp[threadIdx.x] : fr.lm[threadIdx.x];
    __syncthreads();
    double num[NF], den[NF];
#pragma unroll
    for (int i = 0; i < NF; ++i) { num[i] = 0.0; den[i] = 0.0; }
    const size_t P = (size_t)Ne * NS;
    const int sd = d == 0 ? 1 : (d == 1 ? Q : Q * Q);           // node stride along the face normal
    const int sa = d == 0 ? Q : 1, sb = d == 2 ? Q : Q * Q;       // strides of the face point indices
    const double *Mf = bcval + (size_t)face * C * Nu;
    // a p = 1 element as two 16-byte loads (NS = 8) from an aligned state
    const bool vec = sizeof(T) == 4 && Q == 2 && (uintptr_t)f % 16 == 0;
    // velocities k = j1 + n1 * row (n1 <= 128): a thread keeps j1 and walks the rows
    const int rp = WT / n1, rows = Nu / n1, j1 = threadIdx.x % n1;
    const double u1 = vtab[(size_t)j1 * BGK_VTAB];
    double c1[KEEP ? NF : 1];
#pragma unroll
    for (int i = 0; i < (KEEP ? NF : 1); ++i) c1[i] = u1 * nv[i][0];
    if ((int)threadIdx.x < rp * n1)
#pragma unroll 2
        for (int r = split * rp + threadIdx.x / n1; r < rows; r += WS * rp) {
            const int k = j1 + n1 * r;
            const double *vt = vtab + (size_t)k * BGK_VTAB;
            const double u2 = vt[1], u3 = vt[2], w = vt[3], wM = w * Mf[k];
            const T *fe = f + (size_t)k * P + (size_t)e * NS;
            double lw[Q];
#pragma unroll
            for (int j = 0; j < Q; ++j) lw[j] = w * lwr[j];
            // u . n of face point i, and the trace where the velocity leaves
            // the gas (> 0 from the bits: neither zero nor negative)
            auto normal = [&](int i) { return fma(u3, nv[i][2], fma(u2, nv[i][1], KEEP ? c1[KEEP ? i : 0] : u1 * nv[i][0])); };
            auto leaves = [](double un) { return __double_as_longlong(un) > 0; };
            if constexpr (sizeof(T) == 4 && Q == 2) {
                if (vec) {
                    double un[NF];
                    bool any = false;
#pragma unroll
                    for (int i = 0; i < NF; ++i) {
                        un[i] = normal(i);
                        any |= leaves(un[i]);
                    }
                    float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
                    if (any) { lo = *(const float4 *)fe; hi = *(const float4 *)(fe + 4); }
                    const float v[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
                    for (int i = 0; i < NF; ++i) {
                        // the two nodes behind face point i, for normals along x, y, z
                        const int y = i % 2 + 4 * (i / 2);
                        const float v0 = d == 0 ? v[2 * i] : d == 1 ? v[y] : v[i];
                        const float v1 = d == 0 ? v[2 * i + 1] : d == 1 ? v[y + 2] : v[i + 4];
                        // one FMA into the sum this velocity belongs to
                        const bool out = leaves(un[i]);
                        const double tr = fma(lw[1], widen(v1), lw[0] * widen(v0));
                        const double r = fma(un[i], out ? tr : wM, out ? num[i] : den[i]);
                        num[i] = out ? r : num[i];
                        den[i] = out ? den[i] : r;
                    }
                    continue;
                }
            }
#pragma unroll
            for (int i = 0; i < NF; ++i) {
                const double un = normal(i);
                if (leaves(un)) {
                    // the line of nodes through face point (a, b) along axis d
                    const T *ln = fe + (i % Q) * sa + (i / Q) * sb;
                    double tr = 0.0;
#pragma unroll
                    for (int j = 0; j < Q; ++j) tr = fma(lw[j], widen(ln[j * sd]), tr);
                    num[i] = fma(un, tr, num[i]);
                } else {
                    den[i] = fma(un, wM, den[i]);
                }
            }
        }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < NF; ++i) {
        double a = num[i], b = den[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
        }
        if (lane == 0) { red[warp][i] = a; red[warp][NF + i] = b; }
    }
    __syncthreads();
    if (threadIdx.x < 2 * NF) {
        double a = 0.0;
        for (int w = 0; w < WT / 32; ++w) a += red[w][threadIdx.x];
        part[threadIdx.x] = a;
    }
    cluster.sync();
    if (split == 0 && threadIdx.x < NF) {
        double a = 0.0, b = 0.0;
        for (int s = 0; s < WS; ++s) {
            const double *p = cluster.map_shared_rank(part, s);
            a += p[threadIdx.x];
            b += p[NF + threadIdx.x];
        }
        const double r = b < 0.0 ? -a / b : 0.0;
        const size_t o = ((size_t)e * 6 + face) * NF + threadIdx.x;
        rho_w[o] = r;
        if (rho_w2) rho_w2[o] = make_float2((float)r, (float)(r - (double)(float)r));
    }
    cluster.sync();                  // the blocks' partial sums stay until they are read
}

template <typename T, int Q>
cudaError_t launch_q(const T *f, const T *fvec, const double *bcval, const double *vtab, const int *wall_ef,
                     int n_wall, int Ne, int Nu, int n1, int C, const FROps &fr, double *rho_w, float2 *rho_w2, cudaStream_t s) {
    k_wall_density<T, Q><<<n_wall * WS, WT, 0, s>>>(f, fvec, bcval, vtab, wall_ef, Ne, Nu, n1, C, fr, rho_w, rho_w2);
    return cudaGetLastError();
}

}  // namespace

template <typename T>
cudaError_t launch_wall_density(const T *f, const T *fvec, const double *bcval, const double *vtab,
                                const int *wall_ef, int n_wall, int q, int Ne, int Nu, int n1, int C, FROps fr,
                                double *rho_w, float2 *rho_w2, cudaStream_t s) {
    if (n_wall == 0) return cudaSuccess;
    switch (q) {
        case 2: return launch_q<T, 2>(f, fvec, bcval, vtab, wall_ef, n_wall, Ne, Nu, n1, C, fr, rho_w, rho_w2, s);
        case 3: return launch_q<T, 3>(f, fvec, bcval, vtab, wall_ef, n_wall, Ne, Nu, n1, C, fr, rho_w, rho_w2, s);
        case 4: return launch_q<T, 4>(f, fvec, bcval, vtab, wall_ef, n_wall, Ne, Nu, n1, C, fr, rho_w, rho_w2, s);
        case 5: return launch_q<T, 5>(f, fvec, bcval, vtab, wall_ef, n_wall, Ne, Nu, n1, C, fr, rho_w, rho_w2, s);
        default: return cudaErrorInvalidValue;
    }
}

template cudaError_t launch_wall_density<double>(const double *, const double *, const double *, const double *,
                                                 const int *, int, int, int, int, int, int, FROps, double *, float2 *, cudaStream_t);
template cudaError_t launch_wall_density<float>(const float *, const float *, const double *, const double *,
                                                const int *, int, int, int, int, int, int, FROps, double *, float2 *, cudaStream_t);
