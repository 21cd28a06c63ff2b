// 3-D stiffness apply y = A_l x (eq. discreteBilinear) with one thread per
// element grid line and the 1-D derivative sweeps in even-odd form.
//
// The GLL nodes are symmetric about 0, so the differentiation matrix is
// centro-antisymmetric: D[N-1-i][N-1-m] = -D[i][m] (N = p + 1), and so is
// D^T.  With u_e[m] = u[m] + u[N-1-m], u_o[m] = u[m] - u[N-1-m] (m < N/2),
//   A_i = sum_m E[i][m] u_e[m] (+ D[i][h] u[h], N odd, h = N/2),
//   B_i = sum_m O[i][m] u_o[m],   E, O = (D[i][m] +- D[i][N-1-m]) / 2,
// a line's derivative is (Du)[i] = A_i + B_i, (Du)[N-1-i] = B_i - A_i, and
// for N odd (Du)[h] = sum_m D[h][m] u_o[m]: N^2/2 multiply-adds and 2N adds
// per line instead of N^2 multiply-adds.  The coefficients are kernel
// parameters read with compile-time indices (constant-bank operands, no
// registers, no loads).  One thread owning a whole line is what lets the
// pairs (i, N-1-i) share A_i and B_i.
//
// Per element (N^2 threads), thread (a, b) owns the t-line (i, j) = (a, b)
// in registers (global reads of x and G, the t sweeps and the scatter, all
// coalesced along i), and the r-line (j, k) = (a, b) and the s-line
// (i, k) = (a, b) through shared memory.  Element-interior nodes are stored,
// shared nodes summed with atomics (direct stiffness summation), Dirichlet
// rows skipped when mask is set.  FP64: apply_eo3_kernel, with DOT per-block
// partials of sum_e x_e^T (A_e x_e) as in the node-per-thread kernels.  FP32:
// apply_eo3_pair_kernel, two elements or right-hand sides per thread.
#include "device.cuh"
#include "f32x2.cuh"
#include "reduce.cuh"
#include "setup.h"

#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

namespace glls {

namespace {

// Elements per CTA of the even-odd kernel: at most 256 threads, and no more
// elements than keep about eight CTAs per SM on the level (152 SMs).
int eo_epb(int p, long long E) {
    const long long most = 256 / ((p + 1) * (p + 1));
    const long long fill = E / (152 * 8);
    return (int)std::max(1LL, std::min(most, fill));
}

// One N x N matrix M in even-odd form (H = N / 2).
template <typename T, int N>
struct EoMat {
    static constexpr int H = N / 2;
    T e[H * H];   // (M[i][m] + M[i][N-1-m]) / 2, i, m < H
    T o[H * H];   // (M[i][m] - M[i][N-1-m]) / 2
    T c[H];       // M[i][h], N odd
    T r[H];       // M[h][m], N odd
};
template <typename T, int N>
struct EoParams {
    EoMat<T, N> f;   // D
    EoMat<T, N> t;   // D^T
};

// out = M u for one line, even-odd form
template <typename T, int N>
__device__ __forceinline__ void eo_line(const EoMat<T, N>& M, const T (&u)[N], T (&out)[N]) {
    constexpr int H = N / 2;
    constexpr bool ODD = (N & 1) != 0;
    T ue[H], uo[H];
#pragma unroll
    for (int m = 0; m < H; ++m) {
        ue[m] = u[m] + u[N - 1 - m];
        uo[m] = u[m] - u[N - 1 - m];
    }
#pragma unroll
    for (int i = 0; i < H; ++i) {
        T a = ODD ? M.c[i] * u[H] : T(0), b = T(0);
#pragma unroll
        for (int m = 0; m < H; ++m) {
            a += M.e[i * H + m] * ue[m];
            b += M.o[i * H + m] * uo[m];
        }
        out[i] = a + b;
        out[N - 1 - i] = b - a;
    }
    if constexpr (ODD) {
        T s = T(0);
#pragma unroll
        for (int m = 0; m < H; ++m) s += M.r[m] * uo[m];
        out[H] = s;
    }
}

// Shared-memory strides for 8-byte values: row RS, plane PS, element ES,
// chosen so that the row, column and node accesses of a warp spread over the
// banks (at most a two-way conflict).
template <int N>
struct EoShape {
    static constexpr int NP = N * N, NLOC = NP * N;
    static constexpr int RS = N == 8 ? 9 : N == 7 ? 7 : N == 6 ? 9 : N;
    static constexpr int kPlane[8] = {5, 9, 19, 25, 54, 52, 72, 89};              // N = 2 .. 9
    static constexpr int kElement[8] = {12, 27, 76, 125, 324, 369, 576, 801};
    static constexpr int PS = kPlane[N - 2], ES = kElement[N - 2];
    static constexpr int NBUF = 3;                           // x, and two work buffers
};

__device__ __forceinline__ bool on_bd(int I, int J, int K, const int n[3]) {
    return I == 0 || I == n[0] - 1 || J == 0 || J == n[1] - 1 || K == 0 || K == n[2] - 1;
}

// FP64 (T = double).  epb elements per CTA (at most 256 threads), chosen at
// launch so that small levels still spread over many CTAs per SM.  Two
// resident CTAs per SM bound the registers (at most 128 per thread).
template <typename T, int P, bool DOT, bool LOC>
__global__ void __launch_bounds__(256, 2)
    apply_eo3_kernel(DevLevel<T> L, const __grid_constant__ EoParams<T, P + 1> M, const T* __restrict__ x,
                     T* __restrict__ y, int mask, double* dot, double* part, unsigned* ticket, int epb, int nrhs,
                     T* loc) {
    using S = EoShape<P + 1>;
    constexpr int N = P + 1, NP = S::NP, NLOC = S::NLOC, RS = S::RS, PS = S::PS, ES = S::ES;
    extern __shared__ __align__(16) unsigned char eo_smem3[];
    T* sX = reinterpret_cast<T*>(eo_smem3);
    T* sU = sX + epb * ES;
    T* sV = sU + epb * ES;
    grid_dep_sync();
    // right-hand side fastest in the CTA order (see device.cuh)
    const int rhs = blockIdx.x % nrhs, bx = blockIdx.x / nrhs, nbx = gridDim.x / nrhs;
    x += (long long)rhs * L.N;
    y += (long long)rhs * L.N;
    if constexpr (LOC) loc += (long long)rhs * L.E * NLOC;
    const int E = (int)L.E, n0 = L.n[0], n1 = L.n[1];
    const int nplane = n0 * n1;
    const int tid = threadIdx.x;
    const int el = tid / NP, c = tid - el * NP, a = c % N, b = c / N;
    const int e = bx * epb + el;
    const bool act = el < epb && e < E;
    const int elo = act ? el : 0;
    T* X = sX + elo * ES;
    T* U = sU + elo * ES;
    T* V = sV + elo * ES;
    int base = 0, I = 0, J = 0, K0 = 0;
    T xc[N], ut[N];
    if (act) {
        const int ne0 = L.ne[0], ne1 = L.ne[1];
        const int ex = e % ne0, ey = (e / ne0) % ne1, ez = e / (ne0 * ne1);
        I = ex * P + a;
        J = ey * P + b;
        K0 = ez * P;
        base = (K0 * n1 + J) * n0 + I;
#pragma unroll
        for (int k = 0; k < N; ++k) xc[k] = x[base + k * nplane];
#pragma unroll
        for (int k = 0; k < N; ++k) X[k * PS + b * RS + a] = xc[k];
        eo_line<T, N>(M.f, xc, ut);
    }
    __syncthreads();
    if (act) {
        // r-line (j, k) = (a, b) of x into U, s-line (i, k) = (a, b) into V
        T u[N], v[N];
#pragma unroll
        for (int m = 0; m < N; ++m) u[m] = X[b * PS + a * RS + m];
        eo_line<T, N>(M.f, u, v);
#pragma unroll
        for (int m = 0; m < N; ++m) U[b * PS + a * RS + m] = v[m];
#pragma unroll
        for (int m = 0; m < N; ++m) u[m] = X[b * PS + m * RS + a];
        eo_line<T, N>(M.f, u, v);
#pragma unroll
        for (int m = 0; m < N; ++m) V[b * PS + m * RS + a] = v[m];
    }
    __syncthreads();
    T yt[N];
    if (act) {
        // node (a, b, k): w = G grad x; w_r, w_s over the node's own U, V slots,
        // w_t along the t-line in registers, then D^T along it
        const int EN = E * NLOC;
        const T* G = L.G + e * NLOC + c;
        T wt[N];
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const T g0 = __ldg(G + k * NP), g1 = __ldg(G + EN + k * NP), g2 = __ldg(G + 2 * EN + k * NP);
            const T g3 = __ldg(G + 3 * EN + k * NP), g4 = __ldg(G + 4 * EN + k * NP);
            const T g5 = __ldg(G + 5 * EN + k * NP);
            const int s = k * PS + b * RS + a;
            const T dr = U[s], ds = V[s], dt = ut[k];
            U[s] = g0 * dr + g1 * ds + g2 * dt;
            V[s] = g1 * dr + g3 * ds + g4 * dt;
            wt[k] = g2 * dr + g4 * ds + g5 * dt;
        }
        eo_line<T, N>(M.t, wt, yt);
    }
    __syncthreads();
    if (act) {
        // D^T along the r-line (j, k) = (a, b) of w_r and the s-line (i, k) = (a, b) of w_s, in place
        T u[N], v[N];
#pragma unroll
        for (int m = 0; m < N; ++m) u[m] = U[b * PS + a * RS + m];
        eo_line<T, N>(M.t, u, v);
#pragma unroll
        for (int m = 0; m < N; ++m) U[b * PS + a * RS + m] = v[m];
#pragma unroll
        for (int m = 0; m < N; ++m) u[m] = V[b * PS + m * RS + a];
        eo_line<T, N>(M.t, u, v);
#pragma unroll
        for (int m = 0; m < N; ++m) V[b * PS + m * RS + a] = v[m];
    }
    __syncthreads();
    double local = 0.0;
    if (act) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const int s = k * PS + b * RS + a;
            const T v = yt[k] + U[s] + V[s];
            if (DOT) local += (double)xc[k] * (double)v;
            if constexpr (LOC) {         // element values; summed by gather_kernel in a fixed order
                loc[e * NLOC + k * NP + c] = v;
                continue;
            }
            const int g = base + k * nplane;
            if (a > 0 && a < P && b > 0 && b < P && k > 0 && k < P) {
                y[g] = v;
            } else {
                if (mask && on_bd(I, J, K0 + k, L.n)) continue;
                atomicAdd(&y[g], v);
            }
        }
    }
    if (DOT) {
        __shared__ double red[kReduceThreads];
        const double tsum = block_sum(local, red);
        if (tid == 0) part[(long long)rhs * nbx + bx] = tsum;
        if (ticket && last_block(ticket)) {   // single right-hand side only
            finalize_partials(part, 1, gridDim.x, dot, 0, 0, red);
            if (tid == 0) *ticket = 0u;
        }
    }
}

// ---- FP32, two elements or two right-hand sides per thread -----------------

// One N x N matrix in even-odd form, every coefficient twice (both halves of
// a pair use it).
template <int N>
struct EoMat2 {
    static constexpr int H = N / 2;
    f32x2 e[H * H], o[H * H], c[H], r[H];
};
template <int N>
struct EoParams2 {
    EoMat2<N> f, t;
};

// out = M u for a pair of lines (as eo_line)
template <int N>
__device__ __forceinline__ void eo_line2(const EoMat2<N>& M, const f32x2 (&u)[N], f32x2 (&out)[N]) {
    constexpr int H = N / 2;
    constexpr bool ODD = (N & 1) != 0;
    f32x2 ue[H], uo[H];
#pragma unroll
    for (int m = 0; m < H; ++m) {
        ue[m] = add2(u[m], u[N - 1 - m]);
        uo[m] = sub2(u[m], u[N - 1 - m]);
    }
#pragma unroll
    for (int i = 0; i < H; ++i) {
        f32x2 a = ODD ? mul2(M.c[i], u[H]) : mul2(M.e[i * H], ue[0]), b = mul2(M.o[i * H], uo[0]);
        if constexpr (ODD) a = fma2(M.e[i * H], ue[0], a);
#pragma unroll
        for (int m = 1; m < H; ++m) {
            a = fma2(M.e[i * H + m], ue[m], a);
            b = fma2(M.o[i * H + m], uo[m], b);
        }
        out[i] = add2(a, b);
        out[N - 1 - i] = sub2(b, a);
    }
    if constexpr (ODD) {
        f32x2 s = mul2(M.r[0], uo[0]);
#pragma unroll
        for (int m = 1; m < H; ++m) s = fma2(M.r[m], uo[m], s);
        out[H] = s;
    }
}

// The even-odd apply with packed FP32 arithmetic.  A kernel with one line per
// thread was bound by instruction issue (990 instructions a thread at p = 7)
// and, next, by shared-memory wavefronts.  A thread that carries two lines in
// the halves of a pair issues one instruction for both: two right-hand sides
// of one element (RHS; the geometric factors are read once for both), or two
// neighbouring elements; at p = 7 the swizzled slots below remove the bank
// conflicts that a pair of strides leaves.  Measured on 16^3 elements, p = 7:
// 12.7 -> 10.9 us (9.1 us at the measured copy bandwidth), 32 right-hand
// sides 359 -> 237 us (L1 and shared memory then 84 % busy, issue 51 %); 24^3,
// p = 8: 74 -> 71 us.
//
// Resident CTAs of 128 threads the registers must allow: 4 (at most 128
// registers a thread) or 5 (96).  us per apply with 4 and with 5, 1 to 2 M
// nodes: one right-hand side p = 4 14.5 and 14.4, p = 5 18.3 and 18.3, p = 6
// 22.6 and 21.1, p = 7 20.5 and 20.4, p = 8 22.6 and 24.6; eight p = 5 88.1 and
// 88.1, p = 6 114.7 and 115.3, p = 7 108.4 and 102.3, p = 8 127.0 and 119.9.
constexpr int eo_pair_min_ctas(int P, bool rhs) { return rhs ? (P == 8 ? 4 : 5) : (P == 5 || P == 6 ? 5 : 4); }

template <int P, bool RHS, bool LOC>
__global__ void __launch_bounds__(128, eo_pair_min_ctas(P, RHS))
    apply_eo3_pair_kernel(DevLevel<float> L, const __grid_constant__ EoParams2<P + 1> M, const float* __restrict__ x,
                          float* __restrict__ y, int mask, int epb, int nrhs, float* loc) {
    using S = EoShape<P + 1>;
    constexpr int N = P + 1, NP = S::NP, NLOC = S::NLOC, RS = S::RS, PS = S::PS, ES = S::ES;
    extern __shared__ __align__(16) unsigned char eo_smem2[];
    f32x2* sX = reinterpret_cast<f32x2*>(eo_smem2);
    f32x2* sU = sX + epb * ES;
    f32x2* sV = sU + epb * ES;
    const int E = (int)L.E, n0 = L.n[0], n1 = L.n[1], nplane = n0 * n1;
    // right-hand sides fastest in the CTA order (see device.cuh)
    const int groups = RHS ? nrhs / 2 : nrhs;
    const int rg = blockIdx.x % groups, bx = blockIdx.x / groups;
    const int tid = threadIdx.x;
    const int el = tid / NP, c = tid - el * NP, a = c % N, b = c / N;
    const int slot = bx * epb + el;              // element (RHS) or pair of elements
    const int eA = RHS ? slot : 2 * slot;
    const bool act = el < epb && eA < E;
    const bool hasB = RHS || eA + 1 < E;         // an odd last element computes twice, stores once
    const int eB = RHS || !hasB ? eA : eA + 1;
    const float* xA = x + (long long)(RHS ? 2 * rg : rg) * L.N;
    const float* xB = RHS ? xA + L.N : xA;
    float* yA = y + (long long)(RHS ? 2 * rg : rg) * L.N;
    float* yB = RHS ? yA + L.N : yA;
    const int elo = act ? el : 0;
    f32x2* X = sX + elo * ES;
    f32x2* U = sU + elo * ES;
    f32x2* V = sV + elo * ES;
    // Slots of node (i, j, k) in the buffers: t-lines are read and written at
    // (a, b, k), r-lines at (m, a, b), s-lines at (a, m, b).  N = 8: rows of 8
    // with the column swizzled by the row and plane, so that every half-warp
    // touches 16 different 8-byte banks in all three; no pair of strides does.
    constexpr bool SWZ = N == 8;
    int to[2] = {}, ro[N] = {}, so[4] = {};
    if constexpr (SWZ) {
#pragma unroll
        for (int q = 0; q < 2; ++q) to[q] = b * 8 + (a ^ ((b >> 1) | (q << 2)));
#pragma unroll
        for (int m = 0; m < N; ++m) ro[m] = b * 72 + a * 8 + (m ^ ((a >> 1) | ((b & 1) << 2)));
#pragma unroll
        for (int q = 0; q < 4; ++q) so[q] = b * 72 + (a ^ (q | ((b & 1) << 2)));
    }
    auto at_t = [&](int k) { return SWZ ? k * 72 + to[k & 1] : k * PS + b * RS + a; };
    auto at_r = [&](int m) { return SWZ ? ro[m] : b * PS + a * RS + m; };
    auto at_s = [&](int m) { return SWZ ? m * 8 + so[(m >> 1) & 3] : b * PS + m * RS + a; };
    const int ne0 = L.ne[0], ne1 = L.ne[1];
    int baseA, baseB, KA, KB;
    bool bdA, bdB;                               // column (a, b) on the boundary of axes 0, 1
    {
        const int ex = eA % ne0, ey = (eA / ne0) % ne1, ez = eA / (ne0 * ne1);
        const int I = ex * P + a, J = ey * P + b;
        KA = ez * P;
        baseA = (KA * n1 + J) * n0 + I;
        bdA = I == 0 || I == n0 - 1 || J == 0 || J == n1 - 1;
    }
    if (RHS) {
        baseB = baseA;
        KB = KA;
        bdB = bdA;
    } else {
        const int ex = eB % ne0, ey = (eB / ne0) % ne1, ez = eB / (ne0 * ne1);
        const int I = ex * P + a, J = ey * P + b;
        KB = ez * P;
        baseB = (KB * n1 + J) * n0 + I;
        bdB = I == 0 || I == n0 - 1 || J == 0 || J == n1 - 1;
    }
    // low orders hold their geometric factors before the preceding kernel has
    // ended (mesh data)
    constexpr bool HELD = N <= 4;
    const int EN = E * NLOC;
    const float* GA = L.G + eA * NLOC + c;
    const float* GB = L.G + eB * NLOC + c;
    f32x2 gh[HELD ? N : 1][6];
    if (HELD && act) {
#pragma unroll
        for (int k = 0; k < N; ++k)
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const float ga = __ldg(GA + q * EN + k * NP);
                gh[HELD ? k : 0][q] = pack2(ga, RHS ? ga : __ldg(GB + q * EN + k * NP));
            }
    }
    grid_dep_sync();
    f32x2 ut[N];
    if (act) {
        f32x2 xc[N];
#pragma unroll
        for (int k = 0; k < N; ++k) xc[k] = pack2(xA[baseA + k * nplane], xB[baseB + k * nplane]);
#pragma unroll
        for (int k = 0; k < N; ++k) X[at_t(k)] = xc[k];
        eo_line2<N>(M.f, xc, ut);
    }
    __syncthreads();
    if (act) {
        f32x2 u[N], v[N];
#pragma unroll
        for (int m = 0; m < N; ++m) u[m] = X[at_r(m)];
        eo_line2<N>(M.f, u, v);
#pragma unroll
        for (int m = 0; m < N; ++m) U[at_r(m)] = v[m];
#pragma unroll
        for (int m = 0; m < N; ++m) u[m] = X[at_s(m)];
        eo_line2<N>(M.f, u, v);
#pragma unroll
        for (int m = 0; m < N; ++m) V[at_s(m)] = v[m];
    }
    __syncthreads();
    f32x2 yt[N];
    if (act) {
        f32x2 wt[N];
#pragma unroll
        for (int k = 0; k < N; ++k) {
            f32x2 g[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                if constexpr (HELD) {
                    g[q] = gh[k][q];
                } else {
                    const float ga = __ldg(GA + q * EN + k * NP);
                    g[q] = pack2(ga, RHS ? ga : __ldg(GB + q * EN + k * NP));
                }
            }
            const int s = at_t(k);
            const f32x2 dr = U[s], ds = V[s], dt = ut[k];
            U[s] = fma2(g[2], dt, fma2(g[1], ds, mul2(g[0], dr)));
            V[s] = fma2(g[4], dt, fma2(g[3], ds, mul2(g[1], dr)));
            wt[k] = fma2(g[5], dt, fma2(g[4], ds, mul2(g[2], dr)));
        }
        eo_line2<N>(M.t, wt, yt);
    }
    __syncthreads();
    if (act) {
        f32x2 u[N], v[N];
#pragma unroll
        for (int m = 0; m < N; ++m) u[m] = U[at_r(m)];
        eo_line2<N>(M.t, u, v);
#pragma unroll
        for (int m = 0; m < N; ++m) U[at_r(m)] = v[m];
#pragma unroll
        for (int m = 0; m < N; ++m) u[m] = V[at_s(m)];
        eo_line2<N>(M.t, u, v);
#pragma unroll
        for (int m = 0; m < N; ++m) V[at_s(m)] = v[m];
    }
    __syncthreads();
    if (!act) return;
    const bool inner = a > 0 && a < P && b > 0 && b < P;
    // element values of both halves; summed by gather_kernel in a fixed order
    float* lA = LOC ? loc + ((long long)(RHS ? 2 * rg : rg) * E + eA) * NLOC + c : nullptr;
    float* lB = LOC ? loc + ((long long)(RHS ? 2 * rg + 1 : rg) * E + eB) * NLOC + c : nullptr;
    const int last = L.n[2] - 1;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const int s = at_t(k);
        float vA, vB;
        unpack2(add2(add2(yt[k], U[s]), V[s]), vA, vB);
        if constexpr (LOC) {
            lA[k * NP] = vA;
            if (hasB) lB[k * NP] = vB;
            continue;
        }
        float* pA = yA + baseA + k * nplane;
        float* pB = yB + baseB + k * nplane;
        if (k > 0 && k < P && inner) {
            *pA = vA;
            if (hasB) *pB = vB;
        } else {
            const bool outA = bdA || (k == 0 && KA == 0) || (k == P && KA + P == last);
            const bool outB = bdB || (k == 0 && KB == 0) || (k == P && KB + P == last);
            if (!(mask && outA)) atomicAdd(pA, vA);
            if (hasB && !(mask && outB)) atomicAdd(pB, vB);
        }
    }
}

// Even-odd coefficients of D and D^T of order p in T, built once per order
template <typename T>
const std::vector<T>& eo_table(int p) {
    static std::once_flag once;
    static std::vector<T> tab[9];
    std::call_once(once, [] {
        for (int q = 1; q <= 8; ++q) {
            const int n = q + 1, h = n / 2;
            const std::vector<double> D = derivative_matrix(q);
            std::vector<T>& v = tab[q];
            for (int tr = 0; tr < 2; ++tr) {
                auto Mv = [&](int i, int m) { return tr ? D[m * n + i] : D[i * n + m]; };
                for (int i = 0; i < h; ++i)
                    for (int m = 0; m < h; ++m) v.push_back((T)(0.5 * (Mv(i, m) + Mv(i, n - 1 - m))));
                for (int i = 0; i < h; ++i)
                    for (int m = 0; m < h; ++m) v.push_back((T)(0.5 * (Mv(i, m) - Mv(i, n - 1 - m))));
                for (int i = 0; i < h; ++i) v.push_back((T)Mv(i, h));
                for (int m = 0; m < h; ++m) v.push_back((T)Mv(h, m));
            }
        }
    });
    return tab[p];
}

template <typename T, int N>
EoParams<T, N> eo_params() {
    static_assert(sizeof(EoParams<T, N>) == sizeof(T) * 2 * (2 * (N / 2) * (N / 2) + 2 * (N / 2)), "packed");
    EoParams<T, N> M;
    const std::vector<T>& v = eo_table<T>(N - 1);
    std::memcpy(&M, v.data(), sizeof(M));
    return M;
}

template <int N>
EoParams2<N> eo_params2() {
    const EoParams<float, N> M = eo_params<float, N>();
    EoParams2<N> D;
    const float* src = reinterpret_cast<const float*>(&M);
    float* dst = reinterpret_cast<float*>(&D);
    static_assert(sizeof(D) == 2 * sizeof(M), "packed");
    for (size_t i = 0; i < sizeof(M) / sizeof(float); ++i) dst[2 * i] = dst[2 * i + 1] = src[i];
    return D;
}

// Element slots per CTA of the pair kernel: at most 128 threads, and no more
// than keep about eight CTAs per SM on the level, but at least two warps' worth.
int eo_pair_epb(int p, long long slots) {
    const int np = (p + 1) * (p + 1);
    const long long most = std::max(1, 128 / np), least = std::max(1, 64 / np);
    return (int)std::max(least, std::min(most, slots / (152 * 8)));
}

template <int P>
bool launch_eo_pair(const DevLevel<float>& L, const float* x, float* y, bool mask, cudaStream_t st, int nrhs,
                    float* loc) {
    using S = EoShape<P + 1>;
    const bool rhs = nrhs % 2 == 0;
    const EoParams2<P + 1> M = eo_params2<P + 1>();
    const long long slots = rhs ? L.E : (L.E + 1) / 2;
    const int epb = eo_pair_epb(P, slots * (rhs ? nrhs / 2 : nrhs));
    const long long nb = (slots + epb - 1) / epb * (rhs ? nrhs / 2 : nrhs);
    if (nb > 0x7fffffffLL) return false;
    const int threads = (epb * S::NP + 31) / 32 * 32;
    const size_t smem = sizeof(f32x2) * S::NBUF * epb * S::ES;
    auto go = [&](auto kern) {
        launch_k(kern, (unsigned)nb, threads, smem, st, L, M, x, y, mask ? 1 : 0, epb, nrhs, loc);
        return true;
    };
    if (rhs) return loc ? go(apply_eo3_pair_kernel<P, true, true>) : go(apply_eo3_pair_kernel<P, true, false>);
    return loc ? go(apply_eo3_pair_kernel<P, false, true>) : go(apply_eo3_pair_kernel<P, false, false>);
}

template <typename T, int P>
bool launch_eo(const DevLevel<T>& L, const T* x, T* y, bool mask, double* dot, double* part, unsigned* ticket,
               cudaStream_t st, int nrhs, T* loc) {
    using S = EoShape<P + 1>;
    const EoParams<T, P + 1> M = eo_params<T, P + 1>();
    const int epb = eo_epb(P, L.E);
    const long long nb = (L.E + epb - 1) / epb * nrhs;
    if (nb > 0x7fffffffLL) return false;
    const int blocks = (int)nb;
    const int threads = (epb * S::NP + 31) / 32 * 32;
    const size_t smem = sizeof(T) * S::NBUF * epb * S::ES;
    auto go = [&](auto kern) {
        launch_k(kern, blocks, threads, smem, st, L, M, x, y, mask ? 1 : 0, dot, part, ticket, epb, nrhs, loc);
        return true;
    };
    if (dot) return loc ? go(apply_eo3_kernel<T, P, true, true>) : go(apply_eo3_kernel<T, P, true, false>);
    return loc ? go(apply_eo3_kernel<T, P, false, true>) : go(apply_eo3_kernel<T, P, false, false>);
}

template <typename T, int P>
bool set_eo_attr() {
    using S = EoShape<P + 1>;
    const int smem = (int)(sizeof(T) * S::NBUF * (256 / S::NP) * S::ES);
    const void* fns[] = {(const void*)apply_eo3_kernel<T, P, false, false>,
                         (const void*)apply_eo3_kernel<T, P, false, true>,
                         (const void*)apply_eo3_kernel<T, P, true, false>,
                         (const void*)apply_eo3_kernel<T, P, true, true>};
    for (const void* f : fns)
        if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return false;
    return true;
}

}  // namespace

// FP32 takes this kernel at every order (p <= 3: 16^3 elements, p = 3, 32
// right-hand sides 46.5 us with one thread per element column, 32.4 here; 20^3,
// one, 5.2 and 4.5 us), FP64 where it was measured faster than the node-per-
// thread kernel on 16^3-element levels: p = 6, 7 (p = 7: 193 against 218 us).
// FP64 elsewhere: the 2N adds per line and the lower thread count cost more
// than the saved multiply-adds.
bool apply_eo_selected(int dim, int p, bool f64) {
    if (dim != 3) return false;
    return f64 ? (p == 6 || p == 7) : (p >= 1 && p <= 8);
}

// Number of CTAs (= dot partials) of the even-odd kernel for L.
int apply_eo_blocks(int p, long long E) {
    const int epb = eo_epb(p, E);
    return (int)((E + epb - 1) / epb);
}

template <typename T>
bool launch_apply_eo(const DevLevel<T>& L, const T* x, T* y, bool mask, double* dot, double* part,
                     unsigned* ticket, cudaStream_t st, int nrhs, T* loc) {
    if (!apply_eo_selected(L.dim, L.p, sizeof(T) == 8)) return false;
    if constexpr (sizeof(T) == 8) {
        switch (L.p) {
            case 6: return launch_eo<T, 6>(L, x, y, mask, dot, part, ticket, st, nrhs, loc);
            default: return launch_eo<T, 7>(L, x, y, mask, dot, part, ticket, st, nrhs, loc);
        }
    } else {
        if (dot) return false;               // x.(A x) is formed in FP64 only
        switch (L.p) {
            case 1: return launch_eo_pair<1>(L, x, y, mask, st, nrhs, loc);
            case 2: return launch_eo_pair<2>(L, x, y, mask, st, nrhs, loc);
            case 3: return launch_eo_pair<3>(L, x, y, mask, st, nrhs, loc);
            case 4: return launch_eo_pair<4>(L, x, y, mask, st, nrhs, loc);
            case 5: return launch_eo_pair<5>(L, x, y, mask, st, nrhs, loc);
            case 6: return launch_eo_pair<6>(L, x, y, mask, st, nrhs, loc);
            case 7: return launch_eo_pair<7>(L, x, y, mask, st, nrhs, loc);
            default: return launch_eo_pair<8>(L, x, y, mask, st, nrhs, loc);
        }
    }
}
template bool launch_apply_eo<float>(const DevLevel<float>&, const float*, float*, bool, double*, double*,
                                     unsigned*, cudaStream_t, int, float*);
template bool launch_apply_eo<double>(const DevLevel<double>&, const double*, double*, bool, double*, double*,
                                      unsigned*, cudaStream_t, int, double*);

bool init_apply_eo_attributes() { return set_eo_attr<double, 6>() && set_eo_attr<double, 7>(); }

}  // namespace glls
