// Line smoothing with the Def. 3.2 line blocks R A_p P (GLL smoother,
// levels with p >= 2).
//
// A line's block couples every pair of its nodes that share an element, so it
// is the sum of (p+1) x (p+1) element-segment blocks overlapping at the
// element-boundary vertices.  The set-up (setup.cpp, line_blocks) condenses
// it: one step of Algorithm 1 with S = the block diagonal of the segment
// interiors K_I (Thm. 3.8: exact when S inverts those blocks exactly) leaves
// the Schur complement on the vertices (Prop. 3.7), which is tridiagonal and
// is solved by cyclic reduction (Cor. 3.9).  Per segment the set-up stores
// K_I^-1 (upper triangle) and w_L, w_R = K_I^-1 K_{I,v} for its two vertices;
// per vertex the multipliers of its elimination (Prop. 3.10, first variant).
// One application of the block inverse to g:
//   z   = K_I^-1 g_I                          every segment
//   c_v = g_v - w_R(v-1) . g_I(v-1) - w_L(v) . g_I(v)     (c = R (g - K x))
//   S nu = c                                  vertex CR, one lane group per line
//   x_I = z - w_L nu_left - w_R nu_right,  x_v = nu_v       (y = x + P e)
//
// A CTA owns LPC lines of one direction (a power of two, at most 16 lines and
// 256 segments), one segment task per thread (line_seg_body).  What bounds
// it: on levels far above L2 the bytes of the segment operators and the
// vectors, elsewhere the chain of dependent phases.  A thread reads its own
// nodes of r, y and x straight into registers, all loads back to back, and
// shared memory only carries the two dots and the vertex value of each
// segment.  In strided directions adjacent threads hold adjacent lines
// (coalesced across the lines; the operators are stored line fastest).  On
// x-lines adjacent threads hold adjacent segments (operators stored segment
// fastest): their loads share cache lines, which L1 serves, and the results
// go out through shared memory, coalesced along the line.
// The segment operators and the vertex multipliers are mesh data that no
// kernel writes, so they are loaded before the wait on the preceding kernel
// and overlap its end.
// P is the compile-time order (2..12); line_any_body takes the order at run
// time, with the operators in shared memory where one line's fit there.
#include "async_copy.cuh"
#include "cr_warp.cuh"
#include "device.cuh"

#include <algorithm>
#include <cstring>

namespace glls {

// The precision of this translation unit: FP32 here, FP64 in
// lines_block_f64.cu, which includes this file.
#ifdef GLLS_LINES_F64
using LineT = double;
#else
using LineT = float;
#endif

namespace {

template <typename T>
struct BlockLineArgs {
    int n, nlines, stride, m1, st1, st2, contiguous, mode;
    int p, E, span, cv, lpc, sub;   // sub: lanes per line of the vertex CR (a power of two, sub cv >= E - 1)
    int nrhs;           // right-hand sides (vectors of N values each)
    long long N;
    long long ntask;
    T alpha;
    const T* blk;                              // [ncoef][ntask]
    const T* vcr;                              // [3][nlines (E - 1)]
    const T* g;
    const T* r;
    T* y;
    T* x;
};

constexpr int kBlockThreads = 256;
constexpr int kMaxLinesPerCta = 16;

// SMs of the current device (cached per process: one device type).
int sm_count() {
    static const int n = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0 ? v : 152;
    }();
    return n;
}

// shared-memory index with one pad word per 32
__device__ __forceinline__ int padk(int k) { return k + (k >> 5); }

// Threads of a CTA of lpc lines of E segments.
__host__ __device__ __forceinline__ int block_threads(int lpc, int E) {
    const int t = (lpc * E + 31) / 32 * 32;
    return t > kBlockThreads ? kBlockThreads : t;
}

// ---- vertex systems -------------------------------------------------------
// Multipliers of a lane's C vertices (vertex k = C lane + j of the line):
// l/a, u/a and 1/a at the level that eliminates the vertex; zero past the end.
template <typename T, int C>
struct VertexCr {
    T la[C], ua[C], ia[C];
    __device__ __forceinline__ void load(const BlockLineArgs<T>& A, int line, bool valid, int slane) {
        const int nv = A.E - 1;
        const long long tot = (long long)A.nlines * nv;
        const T* v = A.vcr + (long long)line * nv;
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const int k = C * slane + j;
            const bool ok = valid && k < nv;
            la[j] = ok ? __ldg(v + k) : T(0);
            ua[j] = ok ? __ldg(v + tot + k) : T(0);
            ia[j] = ok ? __ldg(v + 2 * tot + k) : T(0);
        }
    }
};

// Cyclic reduction with stored multipliers, W lanes per system (W a power of
// two, several systems per warp): at level h the odd multiples of h are
// eliminated into the even ones (g_i -= (u/a)_{i-h} g_{i-h} + (l/a)_{i+h}
// g_{i+h}; the system is symmetric, so l_i = u_{i-h}), then restored
// (x_i = g_i/a_i - (l/a)_i x_{i-h} - (u/a)_i x_{i+h}).  A level costs two
// shuffles each way and no reciprocal; the coefficients' own recursion, which
// took six shuffles and a reciprocal a level, ran once at set-up.  All 32
// lanes of the warp take part.
template <typename T, int C>
__device__ __forceinline__ void vertex_cr(const VertexCr<T, C>& m, T (&g)[C], int slane, int W) {
#pragma unroll
    for (int h = 1; h < C; h *= 2) {
        T gr = __shfl_down_sync(kFullMask, m.la[h - 1] * g[h - 1], 1, W);
        if (slane == W - 1) gr = T(0);
#pragma unroll
        for (int j = 2 * h - 1; j < C; j += 2 * h) {
            const int jr = j + h < C ? j + h : 0;
            g[j] = g[j] - m.ua[j - h] * g[j - h] - (j + h < C ? m.la[jr] * g[jr] : gr);
        }
    }
    T G = g[C - 1];
    for (int d = 1; d < W; d *= 2) {
        const T fl = __shfl_up_sync(kFullMask, m.ua[C - 1] * G, d, W);
        const T fr = __shfl_down_sync(kFullMask, m.la[C - 1] * G, d, W);
        if (((slane + 1) & (2 * d - 1)) == 0) G -= fl + (slane + d < W ? fr : T(0));
    }
    const T Gi = G * m.ia[C - 1];
    T X = slane == W - 1 ? Gi : T(0);
    for (int d = W / 2; d >= 1; d /= 2) {
        T xl = __shfl_up_sync(kFullMask, X, d, W);
        const T xr = __shfl_down_sync(kFullMask, X, d, W);
        if (slane < d) xl = T(0);
        if (((slane + 1) & (2 * d - 1)) == d) X = Gi - m.la[C - 1] * xl - m.ua[C - 1] * xr;
    }
    g[C - 1] = X;
    if constexpr (C > 1) {
        T xprev = __shfl_up_sync(kFullMask, X, 1, W);
        if (slane == 0) xprev = T(0);
#pragma unroll
        for (int h = C / 2; h >= 1; h /= 2) {
#pragma unroll
            for (int j = h - 1; j < C; j += 2 * h) {
                const T xl = j - h >= 0 ? g[j - h >= 0 ? j - h : 0] : xprev;
                const T xr = g[j + h < C ? j + h : C - 1];
                g[j] = g[j] * m.ia[j] - m.la[j] * xl - m.ua[j] * xr;
            }
        }
    }
}

// The vertex phase of a CTA: sh[w SE + v] holds g_v - w_L . g_I of segment v
// (v >= 1) and sdr[w SE + v] w_R . g_I of segment v; the solution of vertex v
// replaces sh[w SE + v].  `first`: the multipliers of the lane group's first
// line, loaded at entry.
template <typename T, int C>
__device__ __forceinline__ void vertex_phase(const BlockLineArgs<T>& A, VertexCr<T, C>& first, T* sh, const T* sdr,
                                             int SE, int l0, int Wc) {
    const int W = A.sub, nv = A.E - 1;
    const int groups = (int)blockDim.x / W, slane = threadIdx.x & (W - 1);
    for (int w0 = 0; w0 < Wc; w0 += groups) {
        const int w = w0 + (int)threadIdx.x / W;
        if (w0 > 0) first.load(A, l0 + w, w < Wc, slane);
        T g[C];
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const int k = C * slane + j;
            g[j] = w < Wc && k < nv ? sh[w * SE + k + 1] - sdr[w * SE + k] : T(0);
        }
        vertex_cr<T, C>(first, g, slane, W);
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const int k = C * slane + j;
            if (w < Wc && k < nv) sh[w * SE + k + 1] = g[j];
        }
    }
}

// ---- segments ----------------------------------------------------------------
// Segment operator of one task, in registers from the kernel's entry (FP64 up
// to order 8; above, the values are read where they are used, K_I^-1 once and
// w_L, w_R twice).
template <typename T, int P>
struct SegOp {
    static constexpr int MI = P > 1 ? P - 1 : 1;
    static constexpr int NPK = MI * (MI + 1) / 2;
    static constexpr bool HELD = P <= (sizeof(T) == 8 ? 8 : 12);
    T t[HELD ? NPK : 1], wl[HELD ? MI : 1], wr[HELD ? MI : 1];
    const T* bp;
    long long nt;
    __device__ __forceinline__ void load(const T* p, long long ntask, bool valid) {
        bp = p;
        nt = ntask;
        if constexpr (HELD) {
            if (valid) {
#pragma unroll
                for (int c = 0; c < NPK; ++c) t[c] = __ldg(p + (long long)c * ntask);
#pragma unroll
                for (int i = 0; i < MI; ++i) {
                    wl[i] = __ldg(p + (long long)(NPK + i) * ntask);
                    wr[i] = __ldg(p + (long long)(NPK + MI + i) * ntask);
                }
            }
        }
    }
    __device__ __forceinline__ T tri(int c) const {
        if constexpr (HELD) return t[c];
        else return __ldg(bp + (long long)c * nt);
    }
    __device__ __forceinline__ T left(int i) const {
        if constexpr (HELD) return wl[i];
        else return __ldg(bp + (long long)(NPK + i) * nt);
    }
    __device__ __forceinline__ T right(int i) const {
        if constexpr (HELD) return wr[i];
        else return __ldg(bp + (long long)(NPK + MI + i) * nt);
    }
    // z = K_I^-1 g, dl = w_L . g, dr = w_R . g
    __device__ __forceinline__ void solve(const T (&g)[MI], T (&z)[MI], T& dl, T& dr) const {
#pragma unroll
        for (int i = 0; i < MI; ++i) z[i] = T(0);
        int c = 0;
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
            for (int j = i; j < MI; ++j) {
                const T v = tri(c++);
                z[i] += v * g[j];
                if (j != i) z[j] += v * g[i];
            }
        dl = dr = T(0);
#pragma unroll
        for (int i = 0; i < MI; ++i) {
            dl += left(i) * g[i];
            dr += right(i) * g[i];
        }
    }
};

// First line of CTA `blk` and the offset of its right-hand side's vectors (the
// right-hand side fastest in the CTA order, see device.cuh: the nrhs CTAs of
// one line group read the same segment operators).
template <typename T>
__device__ __forceinline__ int enter(const BlockLineArgs<T>& A, int blk, long long& vo) {
    const int rhs = A.nrhs == 1 ? 0 : blk % A.nrhs, bx = A.nrhs == 1 ? blk : blk / A.nrhs;
    vo = (long long)rhs * A.N;
    return bx * A.lpc;
}

// MODE 0: x = B^-1 g.  MODE 1: x += alpha B^-1 (r - y), and y is reset to 0
// on element-boundary nodes (the apply that produced y plain-stores element-
// interior nodes and adds into element-boundary ones).  MODE 2: x += alpha
// B^-1 r.  MODE 3: x = alpha B^-1 r.
template <typename T, int P, int C, bool CONTIG>
__device__ __forceinline__ void line_seg_body(const BlockLineArgs<T>& A, int blk, double stopped) {
    constexpr int MI = SegOp<T, P>::MI;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int E = A.E, LPC = A.lpc, SE = E | 1, mode = A.mode;
    T* sh = reinterpret_cast<T*>(smem_raw);   // [LPC][SE]
    T* sdr = sh + LPC * SE;                   // [LPC][SE]
    T* so = sdr + LPC * SE;                   // [padk(LPC n)]: new x (CONTIG)
    long long vo;
    const int l0 = enter(A, blk, vo);
    const T* src = (mode == 0 ? A.g : A.r) + vo;
    T* const yp = mode == 1 ? A.y + vo : nullptr;
    T* const xp = A.x + vo;
    const int Wc = min(LPC, A.nlines - l0);
    const int tid = threadIdx.x;
    // this thread's line w and segment e: segments adjacent for x-lines,
    // lines adjacent for strided directions
    int w, e;
    if constexpr (CONTIG) {
        w = tid / E;
        e = tid - w * E;
    } else {
        w = tid & (LPC - 1);
        e = tid >> (31 - __clz(LPC));
    }
    const bool act = w < Wc && e < E;
    const int li = l0 + (act ? w : 0);
    if (skip_item(stopped)) return;
    SegOp<T, P> op;
    op.load(A.blk + (CONTIG ? (long long)li * E + e : (long long)(act ? e : 0) * A.nlines + li), A.ntask, act);
    VertexCr<T, C> vc;
    {
        const int wg = tid / A.sub;
        vc.load(A, l0 + wg, wg < Wc, tid & (A.sub - 1));
    }
    const int stride = CONTIG ? 1 : A.stride;
    const int c2 = li / A.m1 + 1, c1 = li - (c2 - 1) * A.m1 + 1;
    const int v0 = c1 * A.st1 + c2 * A.st2 + e * P * stride;   // the segment's left vertex
    grid_dep_sync();

    T gi[MI], xi[MI], gv = T(0), xv = T(0);
    const bool vertex = act && e > 0;
    // one branch per mode, so that a thread's loads are issued back to back
#pragma unroll
    for (int i = 0; i < MI; ++i) gi[i] = xi[i] = T(0);
    if (act) {
        if (vertex) gv = src[v0];
#pragma unroll
        for (int i = 0; i < MI; ++i) gi[i] = src[v0 + (i + 1) * stride];
        if (mode == 1) {
            T yi[MI], yv = T(0);
            if (vertex) yv = yp[v0];
#pragma unroll
            for (int i = 0; i < MI; ++i) yi[i] = yp[v0 + (i + 1) * stride];
            if (vertex) xv = xp[v0];
#pragma unroll
            for (int i = 0; i < MI; ++i) xi[i] = xp[v0 + (i + 1) * stride];
            gv -= yv;
#pragma unroll
            for (int i = 0; i < MI; ++i) gi[i] -= yi[i];
        } else if (mode == 2) {
            if (vertex) xv = xp[v0];
#pragma unroll
            for (int i = 0; i < MI; ++i) xi[i] = xp[v0 + (i + 1) * stride];
        }
    }
    T z[MI], nl = T(0), nr = T(0);
    T dl, dr;
    op.solve(gi, z, dl, dr);
    if (E > 1) {
        if (act) {
            sdr[w * SE + e] = dr;
            sh[w * SE + e] = gv - dl;
        }
        __syncthreads();
        vertex_phase<T, C>(A, vc, sh, sdr, SE, l0, Wc);
        __syncthreads();
        if (act) {
            if (e > 0) nl = sh[w * SE + e];
            if (e < E - 1) nr = sh[w * SE + e + 1];
        }
    }
    const T scale = mode == 0 ? T(1) : A.alpha;
    // the next apply stores element-interior nodes and adds into the element-
    // boundary ones: only those must be reset
    const bool seam = mode == 1 && (c1 % P == 0 || (A.st2 != 0 && c2 % P == 0));
    if constexpr (!CONTIG) {
        if (!act) return;
#pragma unroll
        for (int i = 0; i < MI; ++i) {
            const int node = v0 + (i + 1) * stride;
            xp[node] = xi[i] + scale * (z[i] - (op.left(i) * nl + op.right(i) * nr));
            if (seam) yp[node] = T(0);
        }
        if (vertex) {
            xp[v0] = xv + scale * nl;
            if (mode == 1) yp[v0] = T(0);
        }
    } else {
        // a segment's nodes are adjacent: through shared memory, so that whole
        // warps write along the lines
        const int n = A.n, k0 = w * n + e * P;
        if (act) {
#pragma unroll
            for (int i = 0; i < MI; ++i)
                so[padk(k0 + i)] = xi[i] + scale * (z[i] - (op.left(i) * nl + op.right(i) * nr));
            if (vertex) {
                so[padk(k0 - 1)] = xv + scale * nl;
                if (mode == 1) yp[v0] = T(0);
            }
            if (seam) {
#pragma unroll
                for (int i = 0; i < MI; ++i) yp[v0 + i + 1] = T(0);
            }
        }
        __syncthreads();
        // value idx lies on line idx / n: exact by the rounded-up reciprocal
        // for idx < 2^15, n < 2^11
        const unsigned magic = n > 1 ? 0xffffffffu / (unsigned)n + 1u : 0u;
        const int total = Wc * n;
        const int q0 = l0 / A.m1, r0 = l0 - q0 * A.m1;      // plane and row of the CTA's first line
#pragma unroll
        for (int it = 0; it < P; ++it) {
            const int idx = tid + it * (int)blockDim.x;
            if (idx < total) {
                const int wl = n > 1 ? (int)__umulhi((unsigned)idx, magic) : idx;
                int row = r0 + wl, plane = q0;
                while (row >= A.m1) {
                    row -= A.m1;
                    ++plane;
                }
                xp[(row + 1) * A.st1 + (plane + 1) * A.st2 + 1 + idx - wl * n] = so[padk(idx)];
            }
        }
    }
}

// Any order and line length: the line values and the segment operators in
// shared memory (cp.async), z accumulated there.  STAGED = false reads the
// operators from global memory where they are used: the form of the lines
// whose operators alone pass the shared-memory limit (FP64 from p = 39 on one
// element, p = 16 on 97 elements a line; FP32 from p = 55).
template <typename T, int C, bool STAGED>
__device__ __forceinline__ void line_any_body(BlockLineArgs<T> A, int blk, double stopped) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = A.n, E = A.E, span = A.span, mode = A.mode, LPC = A.lpc, SE = E | 1;
    const int p = A.p, mi = p - 1, npk = mi * (mi + 1) / 2;
    const long long ntask = A.ntask;
    T* sg = reinterpret_cast<T*>(smem_raw);   // [LPC][span]: g, then z / nu, then B^-1 g
    T* sx = sg + LPC * span;                  // [LPC][span]: x on entry (MODE 1, 2)
    T* sy = sx + LPC * span;                  // [LPC][span]: y on entry (MODE 1)
    T* sz = sy + LPC * span;                  // [LPC][span]: z accumulation
    T* sh = sz + LPC * span;                  // [LPC][SE]
    T* sdr = sh + LPC * SE;                   // [LPC][SE]
    T* sop = sdr + LPC * SE;                  // [ncoef][threads of the item]: segment operators
    long long vo;
    const int l0 = enter(A, blk, vo);
    if (A.g) A.g += vo;
    if (A.r) A.r += vo;
    if (A.y) A.y += vo;
    A.x += vo;
    const int Wc = min(LPC, A.nlines - l0);
    const int tid = threadIdx.x;
    auto line_base = [&](int w) {
        const int li = l0 + w;
        return (li % A.m1 + 1) * A.st1 + (li / A.m1 + 1) * A.st2;
    };
    const bool has_task = tid < Wc * E;
    const int tw = has_task ? tid / E : 0, te = has_task ? tid - tw * E : 0;
    const bool contig = A.contiguous != 0;
    const T* bp = A.blk + (contig ? (long long)(l0 + tw) * E + te : (long long)te * A.nlines + l0 + tw);
    // operator rows are as long as this launch item's own thread count (a
    // work-list block may be larger; its extra threads have no segment)
    const int opstride = block_threads(LPC, E);
    if (skip_item(stopped)) return;
    VertexCr<T, C> vc;
    {
        const int wg = tid / A.sub;
        vc.load(A, l0 + wg, wg < Wc, tid & (A.sub - 1));
    }
    if (STAGED && has_task) {
        const int ncoef = npk + 2 * mi;
        for (int c = 0; c < ncoef; ++c) cp_async(sop + c * opstride + tid, bp + (long long)c * ntask);
    }
    auto opc = [&](int c) {   // coefficient c of this thread's segment
        if constexpr (STAGED) return sop[c * opstride + tid];
        else return __ldg(bp + (long long)c * ntask);
    };
    grid_dep_sync();
    // x-lines are walked along the line by whole warps; strided directions by
    // threads that each keep one line of the CTA and step over its rows,
    // adjacent threads on adjacent lines
    const int nthr = blockDim.x, nwarp = nthr >> 5;
    const int rows_per_pass = nthr / LPC;
    const int sw = contig ? 0 : tid % LPC, sk0 = contig ? 0 : tid / LPC;
    const bool s_active = !contig && sw < Wc && sk0 < rows_per_pass;
    const int s_base = s_active ? line_base(sw) : 0;
    auto stage = [&](int w, int k, int node) {
        const int o = w * span + padk(k);
        cp_async(sg + o, (mode == 0 ? A.g : A.r) + node);
        if (mode == 1) cp_async(sy + o, A.y + node);
        if (mode == 1 || mode == 2) cp_async(sx + o, A.x + node);
    };
    if (contig) {
        for (int w = tid >> 5; w < Wc; w += nwarp) {
            const int b = line_base(w);
            for (int k = tid & 31; k < n; k += 32) stage(w, k, b + (k + 1) * A.stride);
        }
    } else if (s_active) {
        for (int k = sk0; k < n; k += rows_per_pass) stage(sw, k, s_base + (k + 1) * A.stride);
    }
    cp_async_wait_all();
    __syncthreads();
    if (mode == 1) {          // g = r - y (pad slots hold unused values)
        for (int i = tid; i < Wc * span; i += nthr) sg[i] -= sy[i];
        __syncthreads();
    }
    if (has_task) {
        T* line = sg + tw * span;
        T* zz = sz + tw * span;
        const int base = te * p;   // line unknown of the segment's first interior node
        T dl = T(0), dr = T(0);
        for (int i = 0; i < mi; ++i) zz[padk(base + i)] = T(0);
        int c = 0;
        for (int i = 0; i < mi; ++i) {
            const T gi_ = line[padk(base + i)];
            T zi = T(0);
            for (int j = i; j < mi; ++j) {
                const T t = opc(c);
                ++c;
                zi += t * line[padk(base + j)];
                if (j != i) zz[padk(base + j)] += t * gi_;
            }
            zz[padk(base + i)] += zi;
            dl += opc(npk + i) * gi_;
            dr += opc(npk + mi + i) * gi_;
        }
        sdr[tw * SE + te] = dr;
        sh[tw * SE + te] = (te > 0 ? line[padk(base - 1)] : T(0)) - dl;
    }
    __syncthreads();
    if (E > 1) {
        vertex_phase<T, C>(A, vc, sh, sdr, SE, l0, Wc);
        __syncthreads();
    }
    if (has_task) {
        T* line = sg + tw * span;
        const T* zz = sz + tw * span;
        const int base = te * p;
        const T nl = te > 0 ? sh[tw * SE + te] : T(0);
        const T nr = te < E - 1 ? sh[tw * SE + te + 1] : T(0);
        for (int i = 0; i < mi; ++i)
            line[padk(base + i)] = zz[padk(base + i)] - (opc(npk + i) * nl + opc(npk + mi + i) * nr);
        if (te > 0) line[padk(base - 1)] = nl;
    }
    __syncthreads();
    // seam test: the line lies on an element boundary of another axis, or the
    // node is a vertex of the line
    auto put = [&](int w, int k, int base, bool line_seam) {
        const int node = base + (k + 1) * A.stride;
        const T v = sg[w * span + padk(k)];
        A.x[node] = mode == 0 ? v : (mode == 3 ? A.alpha * v : sx[w * span + padk(k)] + A.alpha * v);
        if (mode == 1 && (line_seam || (k + 1) % p == 0)) A.y[node] = T(0);
    };
    auto seam_of = [&](int w) {
        const int li = l0 + w;
        return ((li % A.m1 + 1) % p == 0) || (A.st2 != 0 && (li / A.m1 + 1) % p == 0);
    };
    if (contig) {
        for (int w = tid >> 5; w < Wc; w += nwarp) {
            const int b = line_base(w);
            const bool ls = seam_of(w);
            for (int k = tid & 31; k < n; k += 32) put(w, k, b, ls);
        }
    } else if (s_active) {
        const bool ls = seam_of(sw);
        for (int k = sk0; k < n; k += rows_per_pass) put(sw, k, s_base, ls);
    }
}

// FORM: x-lines (P > 0); operators in shared memory (P == 0, any direction).
template <typename T, int P, int CV, bool FORM>
__device__ __forceinline__ void line_block_body(const BlockLineArgs<T>& A, int blk, double stopped) {
    if constexpr (P == 0) line_any_body<T, CV, FORM>(A, blk, stopped);
    else line_seg_body<T, P, CV, FORM>(A, blk, stopped);
}

// Resident CTAs the registers must allow.  us per line update along the first
// and the second axis, with one fewer, as chosen and with one more: FP32 p = 8
// 2-D 64 x 64 4.1 4.7, 4.4 5.3, 5.2 7.1; 3-D 16^3 15.7 13.2, 14.0 12.5, 15.2
// 15.1; p = 6 20^3 12.4 14.2, 12.2 14.2, 12.0 12.9.  FP32 2-D 60 x 60 as chosen
// and with two: p = 9 4.3 4.9, 4.1 4.9; p = 11 4.5 9.8, 5.2 7.5; p = 12 7.4 10.8,
// 6.1 9.1.  FP64 p = 8 16^3 91 86, 80 75, 76 77; p = 6 20^3 71 72, 71 72, 73 78;
// 2-D 64 x 64 13.0 12.8, 12.8 13.2, 14.2 14.7.  Run-time order, FP32 2-D 200 x
// 200, p = 2: 11.7 9.1, 11.5 9.0, 7.7 7.2.
template <typename T, int P>
constexpr int line_min_ctas() {
    return sizeof(T) == 8 ? 2 : P == 0 ? 2 : P >= 9 ? 1 : 3;
}

template <typename T, int P, int CV, bool FORM>
__global__ void __launch_bounds__(kBlockThreads, line_min_ctas<T, P>())
    line_block_kernel(const __grid_constant__ BlockLineArgs<T> A) {
    line_block_body<T, P, CV, FORM>(A, blockIdx.x, 0.0);
}

// Work-list form: item j is one problem's level, direction and vectors.
template <typename T, int P, int CV, bool FORM>
__global__ void __launch_bounds__(kBlockThreads, line_min_ctas<T, P>())
    line_block_list_kernel(const BlockLineArgs<T>* __restrict__ items, WorkList w) {
    const int j = work_item(w, blockIdx.x);
    const double stopped = item_stopped(w, j);
    line_block_body<T, P, CV, FORM>(items[j], blockIdx.x - w.start[j], stopped);
}

// Shared memory of a CTA of lpc lines: the vertex arrays, with the line
// values once (x-lines) or four times (run-time order).
template <typename T>
size_t block_smem(int lpc, int n, int span, int E, bool contiguous, bool any_order) {
    const size_t tile = (size_t)lpc * n;
    const size_t values = any_order ? 4 * (size_t)lpc * span : contiguous ? tile + tile / 32 + 1 : 0;
    return sizeof(T) * (values + 2 * (size_t)lpc * (E | 1));
}

// Shared memory of the run-time-order instance's segment operators for a
// block of `threads` threads at order p.
template <typename T>
size_t op_smem(int p, int threads) {
    const size_t mi = (size_t)(p - 1);
    return sizeof(T) * (mi * (mi + 1) / 2 + 2 * mi) * (size_t)threads;
}

// Most lines of a CTA: a power of two, at most 16 lines and 256 segments.
int most_lines(int E) {
    int lpc = 1;
    while (2 * lpc <= kMaxLinesPerCta && 2 * lpc * E <= kBlockThreads) lpc *= 2;
    return lpc;
}

// Orders 2..12 are compiled for vertex chunks of 1 and 2 per lane (lines of
// up to 65 elements); longer lines and other orders take the run-time order.
template <typename T, int P, int CV>
bool launch_pc(BlockLineArgs<T> A, cudaStream_t st) {
    // lines per CTA: at most 256 segment tasks and 16 lines; the autotuner's
    // choice for the level and direction when it has made one (A.lpc > 0),
    // else fewer while the level would have less than about four CTAs per SM
    // (small levels are latency bound: more, smaller CTAs run their phases
    // side by side)
    const int most = most_lines(A.E);
    int lpc = most;
    if (A.lpc > 0) {
        while (lpc > A.lpc) lpc /= 2;
    } else {
        // strided directions keep four adjacent lines, half a 32-byte sector
        // of FP32 a row: below that the row reads, not the CTA count, bound
        // the launch (64 x 64 elements, p = 8: 4.7 us with four lines, 11 with one)
        const int least = A.contiguous ? 1 : 4;
        while (lpc > least && (long long)(A.nlines + lpc - 1) / lpc * A.nrhs < 4 * sm_count()) lpc /= 2;
    }
    // the run-time order's operators: in shared memory unless those of a
    // single line do not fit beside its values
    auto sm = [&](int c, bool staged) {
        return block_smem<T>(c, A.n, A.span, A.E, A.contiguous != 0, P == 0) +
               (staged ? op_smem<T>(A.p, block_threads(c, A.E)) : 0);
    };
    const bool staged = P == 0 && sm(1, true) <= kMaxDynSmemBytes;
    while (lpc > 1 && sm(lpc, staged) > kMaxDynSmemBytes) lpc /= 2;
    const size_t smem = sm(lpc, staged);
    if (smem > kMaxDynSmemBytes) return false;   // not reached: kMaxBlockLine, kMaxBlockSegments
    A.lpc = lpc;
    const int threads = block_threads(lpc, A.E);
    const long long blocks = (long long)(A.nlines + lpc - 1) / lpc * A.nrhs;
    if (blocks > 0x7fffffffLL) return false;
    if (P > 0 ? !A.contiguous : !staged)
        return launch_k(line_block_kernel<T, P, CV, false>, (unsigned)blocks, threads, smem, st, A) == cudaSuccess;
    return launch_k(line_block_kernel<T, P, CV, true>, (unsigned)blocks, threads, smem, st, A) == cudaSuccess;
}

template <typename T, int P>
bool launch_p(BlockLineArgs<T> A, cudaStream_t st) {
    if constexpr (P > 0) {
        if (A.cv == 1) return launch_pc<T, P, 1>(A, st);
        if (A.cv == 2) return launch_pc<T, P, 2>(A, st);
        return launch_p<T, 0>(A, st);
    } else {
        switch (A.cv) {
            case 1: return launch_pc<T, 0, 1>(A, st);
            case 2: return launch_pc<T, 0, 2>(A, st);
            case 4: return launch_pc<T, 0, 4>(A, st);
            default: return launch_pc<T, 0, 8>(A, st);
        }
    }
}

// Dynamic shared memory above 48 KB (the run-time order; the others stay below).
template <typename T>
bool set_attr_any() {
    const int lim = (int)kMaxDynSmemBytes;
    const void* fns[] = {(const void*)line_block_kernel<T, 0, 1, true>, (const void*)line_block_kernel<T, 0, 2, true>,
                         (const void*)line_block_kernel<T, 0, 4, true>, (const void*)line_block_kernel<T, 0, 8, true>,
                         (const void*)line_block_kernel<T, 0, 1, false>, (const void*)line_block_kernel<T, 0, 2, false>,
                         (const void*)line_block_kernel<T, 0, 4, false>, (const void*)line_block_kernel<T, 0, 8, false>,
                         (const void*)line_block_list_kernel<T, 0, 1, true>,
                         (const void*)line_block_list_kernel<T, 0, 2, true>,
                         (const void*)line_block_list_kernel<T, 0, 4, true>,
                         (const void*)line_block_list_kernel<T, 0, 8, true>};
    for (const void* f : fns)
        if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) != cudaSuccess) return false;
    return true;
}

}  // namespace

template <>
bool init_line_block_attributes<LineT>() {
    return set_attr_any<LineT>();
}

#ifndef GLLS_LINES_F64
bool line_block_supported(int n, int E) { return n <= kMaxBlockLine && E <= kMaxBlockSegments; }

// Whether launch_line_block_list(p, cv, ...) runs the order-specialised
// instance (smem[0] of the items) or the run-time-order one (smem[1]).
bool line_block_list_specialised(int p, int cv) { return p >= 2 && p <= 12 && cv <= 2; }
#endif

namespace {

// Fills A for a line solve of L along s; 0: nothing to do, -1: outside the
// supported range, 1: ready.
template <typename T>
int make_args(BlockLineArgs<T>& A, const DevLevel<T>& L, int s, int mode, const T* g, const T* r, T* y, T* x,
              T alpha, int nrhs) {
    A.nrhs = nrhs;
    A.N = L.N;
    A.n = L.n[s] - 2;
    if (A.n <= 0) return 0;
    A.E = L.ne[s];
    if (!line_block_supported(A.n, A.E) || L.N > (1LL << 31) - 1) return -1;
    int o1, o2;
    if (s == 0) { o1 = 1; o2 = 2; } else if (s == 1) { o1 = 0; o2 = 2; } else { o1 = 0; o2 = 1; }
    const int strides[3] = {1, L.n[0], L.n[0] * L.n[1]};
    A.m1 = L.n[o1] - 2;
    const int m2 = L.dim == 3 ? L.n[o2] - 2 : 1;
    A.nlines = A.m1 * m2;
    if (A.nlines <= 0) return 0;
    A.ntask = (long long)A.nlines * A.E;
    A.stride = strides[s];
    A.st1 = strides[o1];
    A.st2 = L.dim == 3 ? strides[o2] : 0;
    A.contiguous = s == 0;
    A.mode = mode;
    A.p = L.p;
    A.span = (A.n - 1) + ((A.n - 1) >> 5) + 1;
    A.span = (A.span + 3) / 4 * 4;
    A.lpc = L.lbc[s];                  // 0: the launch heuristic
    const int nv = A.E - 1;
    A.cv = nv <= 32 ? 1 : (nv <= 64 ? 2 : (nv <= 128 ? 4 : 8));
    A.sub = 1;                         // lanes per line of the vertex CR
    while (A.sub * A.cv < nv) A.sub *= 2;
    A.alpha = alpha;
    A.blk = L.blk[s];
    A.vcr = L.vcr[s];
    A.g = g;
    A.r = r;
    A.y = y;
    A.x = x;
    return 1;
}

template <typename T, int P, int CV>
bool launch_list_pc(int s, const void* items, const WorkList& w, int blocks, int threads, size_t smem,
                    cudaStream_t st) {
    const BlockLineArgs<T>* it = static_cast<const BlockLineArgs<T>*>(items);
    if (P > 0 && s != 0)
        return launch_k(line_block_list_kernel<T, P, CV, false>, (unsigned)blocks, threads, smem, st, it, w) ==
               cudaSuccess;
    return launch_k(line_block_list_kernel<T, P, CV, true>, (unsigned)blocks, threads, smem, st, it, w) == cudaSuccess;
}

template <typename T, int P>
bool launch_list_p(int s, int cv, const void* items, const WorkList& w, int blocks, int threads, size_t smem,
                   cudaStream_t st) {
    if constexpr (P > 0) {
        if (cv == 1) return launch_list_pc<T, P, 1>(s, items, w, blocks, threads, smem, st);
        if (cv == 2) return launch_list_pc<T, P, 2>(s, items, w, blocks, threads, smem, st);
        return launch_list_p<T, 0>(s, cv, items, w, blocks, threads, smem, st);
    } else {
        switch (cv) {
            case 1: return launch_list_pc<T, 0, 1>(s, items, w, blocks, threads, smem, st);
            case 2: return launch_list_pc<T, 0, 2>(s, items, w, blocks, threads, smem, st);
            case 4: return launch_list_pc<T, 0, 4>(s, items, w, blocks, threads, smem, st);
            default: return launch_list_pc<T, 0, 8>(s, items, w, blocks, threads, smem, st);
        }
    }
}

}  // namespace

template <typename T>
size_t line_block_item_bytes() {
    return sizeof(BlockLineArgs<T>);
}

// One work-list item: the line solve of L along s (as launch_line_block,
// one right-hand side), written into `item` (line_block_item_bytes bytes);
// its CTA count, block size, vertex chunk (cv, 1..8) and dynamic shared
// memory for the order-specialised instance (smem[0]) and the run-time-order
// instance (smem[1]).  Lines per CTA as for a single launch, without the
// small-level split (a work-list launch has the CTAs of all its items).
// 0: nothing to do; -1: unsupported.
template <typename T>
int line_block_list_item(const DevLevel<T>& L, int s, int mode, const T* g, const T* r, T* y, T* x, T alpha,
                         void* item, int* blocks, int* threads, size_t smem[2], int* cv) {
    BlockLineArgs<T> A;
    const int k = make_args<T>(A, L, s, mode, g, r, y, x, alpha, 1);
    if (k <= 0) return k;
    // the run-time-order instance also holds the segment operators of the
    // item's own threads
    auto sm1 = [&](int c) {
        return block_smem<T>(c, A.n, A.span, A.E, true, true) + op_smem<T>(A.p, block_threads(c, A.E));
    };
    int lpc = most_lines(A.E);
    while (lpc > 1 && sm1(lpc) > kMaxDynSmemBytes) lpc /= 2;
    if (sm1(lpc) > kMaxDynSmemBytes) return -1;
    A.lpc = lpc;
    smem[0] = block_smem<T>(lpc, A.n, A.span, A.E, A.contiguous != 0, false);
    smem[1] = sm1(lpc);
    *threads = block_threads(lpc, A.E);
    *blocks = (A.nlines + lpc - 1) / lpc;
    *cv = A.cv;
    std::memcpy(item, &A, sizeof(A));
    return 1;
}

// One launch over the items (all along axis s and of order p; cv: the largest
// vertex chunk of the items).
template <typename T>
bool launch_line_block_list(int p, int s, int cv, const void* items, const WorkList& w, int blocks, int threads,
                            size_t smem, cudaStream_t st) {
    if (w.nitems < 1 || blocks < 1) return true;
    switch (line_block_list_specialised(p, cv) ? p : 0) {
        case 2: return launch_list_p<T, 2>(s, cv, items, w, blocks, threads, smem, st);
        case 3: return launch_list_p<T, 3>(s, cv, items, w, blocks, threads, smem, st);
        case 4: return launch_list_p<T, 4>(s, cv, items, w, blocks, threads, smem, st);
        case 5: return launch_list_p<T, 5>(s, cv, items, w, blocks, threads, smem, st);
        case 6: return launch_list_p<T, 6>(s, cv, items, w, blocks, threads, smem, st);
        case 7: return launch_list_p<T, 7>(s, cv, items, w, blocks, threads, smem, st);
        case 8: return launch_list_p<T, 8>(s, cv, items, w, blocks, threads, smem, st);
        case 9: return launch_list_p<T, 9>(s, cv, items, w, blocks, threads, smem, st);
        case 10: return launch_list_p<T, 10>(s, cv, items, w, blocks, threads, smem, st);
        case 11: return launch_list_p<T, 11>(s, cv, items, w, blocks, threads, smem, st);
        case 12: return launch_list_p<T, 12>(s, cv, items, w, blocks, threads, smem, st);
        default: return launch_list_p<T, 0>(s, cv, items, w, blocks, threads, smem, st);
    }
}

template size_t line_block_item_bytes<LineT>();
template int line_block_list_item<LineT>(const DevLevel<LineT>&, int, int, const LineT*, const LineT*, LineT*, LineT*,
                                         LineT, void*, int*, int*, size_t*, int*);
template bool launch_line_block_list<LineT>(int, int, int, const void*, const WorkList&, int, int, size_t,
                                            cudaStream_t);

template <typename T>
bool launch_line_block(const DevLevel<T>& L, int s, int mode, const T* g, const T* r, T* y, T* x, T alpha,
                       cudaStream_t st, int nrhs) {
    BlockLineArgs<T> A;
    const int k = make_args<T>(A, L, s, mode, g, r, y, x, alpha, nrhs);
    if (k <= 0) return k == 0;
    switch (L.p) {
        case 2: return launch_p<T, 2>(A, st);
        case 3: return launch_p<T, 3>(A, st);
        case 4: return launch_p<T, 4>(A, st);
        case 5: return launch_p<T, 5>(A, st);
        case 6: return launch_p<T, 6>(A, st);
        case 7: return launch_p<T, 7>(A, st);
        case 8: return launch_p<T, 8>(A, st);
        case 9: return launch_p<T, 9>(A, st);
        case 10: return launch_p<T, 10>(A, st);
        case 11: return launch_p<T, 11>(A, st);
        case 12: return launch_p<T, 12>(A, st);
        default: return launch_p<T, 0>(A, st);
    }
}

template bool launch_line_block<LineT>(const DevLevel<LineT>&, int, int, const LineT*, const LineT*, LineT*, LineT*,
                                       LineT, cudaStream_t, int);

}  // namespace glls
