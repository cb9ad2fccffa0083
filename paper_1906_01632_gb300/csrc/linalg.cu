// linalg.cu -- batched linear algebra of the Newton/BiCGStab/multigrid solve
// (Section 2.3 and Section 5.1): 27-point 2x2-block stencil products,
// damped block-Jacobi smoothing, full-weighting restriction / trilinear
// prolongation on the vertex-centred 2:1 hierarchy, the dense coarse solve,
// the BiCGStab vector updates (van der Vorst; Templates, Sec. 2.3.8) with
// FP64 inner products, and the Newton line-search bookkeeping.
//
// Every node kernel runs one thread per node with grid.y = sample and skips
// samples whose mask flag is 0 (converged or failed samples).  Reductions are
// two-stage and deterministic: per-block partials [S][2][nblk], then one
// block per sample sums them in a fixed order.
//
// Solver vectors hold the unknowns of the interior system: Dirichlet
// components are kept at 0 by masking every kernel's output.
#include <algorithm>
#include <type_traits>
#include <cuda_pipeline.h>

#include "kernels.h"

namespace elder {

__device__ __forceinline__ bool on(const int* mask, int stride, int s)
{
    return mask == nullptr || mask[(size_t)s * stride] != 0;
}

static_assert(sizeof(KScal) % sizeof(int) == 0, "KScal layout");
static_assert(sizeof(NScal) % sizeof(int) == 0, "NScal layout");

// One neighbour term of the 27-point product.  The loads are unconditional
// (a missing neighbour reads node n itself and its term is selected to 0),
// so a thread issues all 54 loads of its row before the first use: the
// stencil kernels are memory-latency bound and need that parallelism.
template <class T, bool TRANS, class M>
__device__ __forceinline__ void stencil_term(const Grid& G, const B4<M>* __restrict__ J,
                                             const V2<T>* __restrict__ x, int n, int m,
                                             int slot, int tslot, bool ok, T& yp, T& yc,
                                             B4<M>* raw = nullptr)
{
    const int mm = ok ? m : n;
    const V2<T> xv = x[mm];
    const B4<M> b = !TRANS ? J[(size_t)slot * G.N + n] : J[(size_t)tslot * G.N + mm];
    if (raw) *raw = b;
    const T pp = ok ? mg_load<T>(b.pp) : T(0), pc = ok ? mg_load<T>(b.pc) : T(0);
    const T cp = ok ? mg_load<T>(b.cp) : T(0), cc = ok ? mg_load<T>(b.cc) : T(0);
    // explicit fused multiply-adds: every instantiation (one or two samples
    // per CTA) rounds the same way
    if (!TRANS) {
        yp = fma(pp, xv.p, fma(pc, xv.c, yp));
        yc = fma(cp, xv.p, fma(cc, xv.c, yc));
    } else {
        yp = fma(pp, xv.p, fma(cp, xv.c, yp));
        yc = fma(pc, xv.p, fma(cc, xv.c, yc));
    }
}

// y_n = sum over the 27 neighbours of the 2x2 block times x (or the
// transposed product, reading row m's block of offset -d).
template <class T, bool TRANS, class M>
__device__ __forceinline__ void stencil_apply(const Grid& G,
                                              const B4<M>* __restrict__ J,
                                              const V2<T>* __restrict__ x,
                                              int n, int i, int j, int k,
                                              T& yp, T& yc)
{
    const int sy = G.nx + 1, sz = (G.nx + 1) * (G.ny + 1);
    yp = T(0);
    yc = T(0);
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
                const bool ok = (dx < 0 ? i > 0 : (dx > 0 ? i < G.nx : true)) &&
                                (dy < 0 ? j > 0 : (dy > 0 ? j < G.ny : true)) &&
                                (dz < 0 ? k > 0 : (dz > 0 ? k < G.nz : true));
                stencil_term<T, TRANS, M>(G, J, x, n, n + dx + dy * sy + dz * sz,
                                          slot27(dx, dy, dz), slot27(-dx, -dy, -dz), ok, yp, yc);
            }
}

// ---------------------------------------------------------------------------
// SpMV with fused inner products
// ---------------------------------------------------------------------------

template <class T, bool TRANS, int MODE>
__global__ void __launch_bounds__(kMaxBS)
    k_spmv(Grid G, const B4<T>* __restrict__ J, const uint8_t* __restrict__ bc,
           const V2<T>* __restrict__ x, V2<T>* __restrict__ y,
           const V2<T>* __restrict__ a, double* __restrict__ partial,
           const int* mask, int mstride)
{
    const int s = blockIdx.y;
    if (!on(mask, mstride, s)) return;
    const size_t on_ = (size_t)s * G.N;
    J += (size_t)s * 27 * G.N;
    x += on_;
    y += on_;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    double d0 = 0.0, d1 = 0.0;
    if (n < G.N) {
        int i, j, k;
        node_ijk(G, n, i, j, k);
        T yp, yc;
        stencil_apply<T, TRANS, T>(G, J, x, n, i, j, k, yp, yc);
        if (MODE != 3) {
            const uint8_t b = bc[n];
            if (b & BC_P) yp = T(0);
            if (b & BC_C) yc = T(0);
        }
        y[n] = V2<T>{yp, yc};
        if (MODE == 1 || MODE == 2) {
            const V2<T> av = a[on_ + n];
            d0 = dot2(av.p, av.c, yp, yc);
        }
        if (MODE == 2) d1 = dot2(yp, yc, yp, yc);
    }
    // One partial per warp of 32 nodes, so the sums do not depend on the
    // (tuned) block size: the inner products are bitwise reproducible.
    if (MODE == 1 || MODE == 2) {
        const int W = (G.N + 31) >> 5;
        const int wg = n >> 5;
        const double t0 = warp_sum(d0);
        const double t1 = (MODE == 2) ? warp_sum(d1) : 0.0;
        if ((threadIdx.x & 31) == 0 && wg < W) {
            partial[((size_t)s * 2 + 0) * W + wg] = t0;
            if (MODE == 2) partial[((size_t)s * 2 + 1) * W + wg] = t1;
        }
    }
}

template <class T>
void launch_spmv(const Grid& G, const B4<T>* J, const uint8_t* bc,
                 const V2<T>* x, V2<T>* y, int trans, int mode,
                 const V2<T>* a, double* partial, const int* mask,
                 int mstride, int S, cudaStream_t st, int bs)
{
    count_launch(1);
    bs = spread_block(bs, G.N, S);
    dim3 grid(nblocks(G.N, bs), S);
#define ELDER_SPMV(TR, MO) \
    k_spmv<T, TR, MO><<<grid, bs, 0, st>>>(G, J, bc, x, y, a, partial, mask, mstride)
    if (!trans) {
        if (mode == 0) ELDER_SPMV(false, 0);
        else if (mode == 1) ELDER_SPMV(false, 1);
        else if (mode == 2) ELDER_SPMV(false, 2);
        else ELDER_SPMV(false, 3);
    } else {
        if (mode == 0) ELDER_SPMV(true, 0);
        else if (mode == 1) ELDER_SPMV(true, 1);
        else if (mode == 2) ELDER_SPMV(true, 2);
        else ELDER_SPMV(true, 3);
    }
#undef ELDER_SPMV
}

// ---------------------------------------------------------------------------
// multigrid: damped block-Jacobi smoother, residual, transfers, coarse solve
// ---------------------------------------------------------------------------

template <class T, class M, bool TRANS, bool ZEROX>
__global__ void __launch_bounds__(kMaxBS)
    k_smooth(Grid G, const B4<M>* __restrict__ J, const B4<T>* __restrict__ Dinv,
             const uint8_t* __restrict__ bc, const V2<T>* __restrict__ b,
             const V2<T>* __restrict__ x, V2<T>* __restrict__ xo, T omega,
             const int* mask, int mstride)
{
    const int s = blockIdx.y;
    if (!on(mask, mstride, s)) return;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= G.N) return;
    const size_t on_ = (size_t)s * G.N;
    const V2<T> bv = b[on_ + n];
    T rp = bv.p, rc = bv.c;
    V2<T> xn{T(0), T(0)};
    if (!ZEROX) {
        int i, j, k;
        node_ijk(G, n, i, j, k);
        T yp, yc;
        stencil_apply<T, TRANS, M>(G, J + (size_t)s * 27 * G.N, x + on_, n, i, j, k, yp, yc);
        rp -= yp;
        rc -= yc;
        xn = x[on_ + n];
    }
    const B4<T> d = Dinv[on_ + n];
    T zp, zc;
    if (!TRANS) { zp = d.pp * rp + d.pc * rc; zc = d.cp * rp + d.cc * rc; }
    else { zp = d.pp * rp + d.cp * rc; zc = d.pc * rp + d.cc * rc; }
    T op = xn.p + omega * zp, oc = xn.c + omega * zc;
    const uint8_t m = bc[n];
    if (m & BC_P) op = T(0);
    if (m & BC_C) oc = T(0);
    xo[on_ + n] = V2<T>{op, oc};
}

template <class T, class M>
void launch_smooth(const Grid& G, const B4<M>* J, const B4<T>* Dinv,
                   const uint8_t* bc, const V2<T>* b, const V2<T>* x,
                   V2<T>* xo, double omega, int trans, const int* mask,
                   int mstride, int S, cudaStream_t st, int bs)
{
    count_launch(1);
    dim3 grid(nblocks(G.N, bs), S);
    const T w = T(omega);
    if (x == nullptr) {
        if (trans) k_smooth<T, M, true, true><<<grid, bs, 0, st>>>(G, J, Dinv, bc, b, x, xo, w, mask, mstride);
        else k_smooth<T, M, false, true><<<grid, bs, 0, st>>>(G, J, Dinv, bc, b, x, xo, w, mask, mstride);
    } else {
        if (trans) k_smooth<T, M, true, false><<<grid, bs, 0, st>>>(G, J, Dinv, bc, b, x, xo, w, mask, mstride);
        else k_smooth<T, M, false, false><<<grid, bs, 0, st>>>(G, J, Dinv, bc, b, x, xo, w, mask, mstride);
    }
}

// ---------------------------------------------------------------------------
// z-line block Jacobi: x_out = x + omega L^{-1} (b - A x), L the block
// tridiagonal part of A along each vertical grid line (2x2 blocks of the
// offsets (0,0,-1), (0,0,0), (0,0,+1)).  One thread solves one line by the
// block Thomas algorithm.  It keeps the node-local pressure/salt coupling and
// the vertical (gravity) coupling implicit: next to a steep salt front on a
// rough permeability field the 2x2 diagonal blocks become nearly singular and
// point block Jacobi diverges locally, while the line solve stays stable.
// The diagonal block is recovered from Dinv (the inverse of the interior-
// masked block, kept in T precision); the off-diagonal line blocks come from
// the stored matrix, masked to the interior operator.
// ---------------------------------------------------------------------------

template <class T>
__device__ __forceinline__ B4<T> inv2(const B4<T>& a)
{
    const T det = a.pp * a.cc - a.pc * a.cp;
    const T r = T(1) / det;
    return B4<T>{a.cc * r, -a.pc * r, -a.cp * r, a.pp * r};
}

template <class T>
__device__ __forceinline__ B4<T> mul2(const B4<T>& a, const B4<T>& b)
{
    return B4<T>{a.pp * b.pp + a.pc * b.cp, a.pp * b.pc + a.pc * b.cc,
                 a.cp * b.pp + a.cc * b.cp, a.cp * b.pc + a.cc * b.cc};
}

// Raw (unmasked) line block of row n for the vertical offset dz = -1 or +1:
// the block of slot (0,0,dz) at row n, or for the transposed operator the
// block of slot (0,0,-dz) at row n + dz*sz read transposed.
template <class T, class M, bool TRANS>
__device__ __forceinline__ B4<T> raw_line_block(const B4<M>& q)
{
    if (!TRANS) return B4<T>{mg_load<T>(q.pp), mg_load<T>(q.pc), mg_load<T>(q.cp), mg_load<T>(q.cc)};
    return B4<T>{mg_load<T>(q.pp), mg_load<T>(q.cp), mg_load<T>(q.pc), mg_load<T>(q.cc)};
}

template <class T>
__device__ __forceinline__ B4<T> mask_block(B4<T> a, uint8_t row_bc, uint8_t col_bc)
{
    if (row_bc & BC_P) { a.pp = T(0); a.pc = T(0); }
    if (row_bc & BC_C) { a.cp = T(0); a.cc = T(0); }
    if (col_bc & BC_P) { a.pp = T(0); a.cp = T(0); }
    if (col_bc & BC_C) { a.pc = T(0); a.cc = T(0); }
    return a;
}

// Depth of the per-thread ring of line inputs in shared memory.
constexpr int kZlRing = 4;

// Asynchronous copy of one element (8, 16 or 32 bytes, naturally aligned)
// from global to shared memory.
template <class X>
__device__ __forceinline__ void async_copy(X* dst, const X* src)
{
    static_assert(sizeof(X) % 8 == 0 && sizeof(X) <= 32, "element size");
    constexpr int step = (sizeof(X) % 16 == 0) ? 16 : 8;
#pragma unroll
    for (int o = 0; o < (int)sizeof(X); o += step)
        __pipeline_memcpy_async(reinterpret_cast<char*>(dst) + o,
                                reinterpret_cast<const char*>(src) + o, step);
}

// The Thomas factors C_k = M_k^{-1} U_k and g_k of the forward sweep live in
// shared memory, [k][thread], for the backward sweep; the forward recursion
// carries C_{k-1} and g_{k-1} in registers.  The inputs of node k (rhs,
// inverse diagonal block, the two vertical line blocks) reach a per-thread
// ring of kZlRing slots in shared memory by asynchronous copies issued
// kZlRing nodes ahead: each thread walks its line serially, and the ring
// keeps several nodes' loads in flight per thread.
// MODE 1: x = 0, x_out = omega L^{-1} b;
// MODE 2: b holds the residual b - A x (masked), x_out = x + omega L^{-1} b.
// A sweep from a nonzero x is the multigrid residual kernel (all nodes in
// parallel, at stream rate) followed by MODE 2: folding the 27-point
// residual into the line kernel runs at a third of the bandwidth, because
// each thread walks its line serially and few warps fit an SM.
template <class T, class M, bool TRANS, int MODE>
__global__ void __launch_bounds__(kLineBS)
    k_smooth_zline(Grid G, const B4<M>* __restrict__ J, const B4<T>* __restrict__ Dinv,
                   const uint8_t* __restrict__ bc, const V2<T>* __restrict__ b,
                   const V2<T>* __restrict__ x, V2<T>* __restrict__ xo, T omega,
                   const int* mask, int mstride)
{
    extern __shared__ __align__(16) unsigned char zl_smem[];
    const int s = blockIdx.y;
    if (!on(mask, mstride, s)) return;
    const int bsz = blockDim.x, tx = threadIdx.x;
    B4<T>* Cs = reinterpret_cast<B4<T>*>(zl_smem);                  // [nz][bsz]
    V2<T>* gs = reinterpret_cast<V2<T>*>(Cs + (size_t)G.nz * bsz);   // [nz+1][bsz]
    B4<T>* Rdi = reinterpret_cast<B4<T>*>(gs + (size_t)(G.nz + 1) * bsz);  // [ring][bsz]
    V2<T>* Rb = reinterpret_cast<V2<T>*>(Rdi + (size_t)kZlRing * bsz);
    B4<M>* RL = reinterpret_cast<B4<M>*>(Rb + (size_t)kZlRing * bsz);
    B4<M>* RU = RL + (size_t)kZlRing * bsz;
    const int sz = (G.nx + 1) * (G.ny + 1);
    const int col = blockIdx.x * bsz + tx;
    if (col >= sz) return;
    const size_t on_ = (size_t)s * G.N;
    const B4<M>* Js = J + (size_t)s * 27 * G.N;
    const V2<T>* xs = (MODE == 1) ? nullptr : x + on_;
    // copies of node k into ring slot k % kZlRing (one commit group per node,
    // empty past the end of the line)
    auto issue = [&](int k) {
        if (k <= G.nz) {
            const int n = col + k * sz;
            const int q = (k % kZlRing) * bsz + tx;
            async_copy(Rb + q, b + on_ + n);
            async_copy(Rdi + q, Dinv + on_ + n);
            if (k > 0)
                async_copy(RL + q, !TRANS ? Js + (size_t)slot27(0, 0, -1) * G.N + n
                                          : Js + (size_t)slot27(0, 0, 1) * G.N + n - sz);
            if (k < G.nz)
                async_copy(RU + q, !TRANS ? Js + (size_t)slot27(0, 0, 1) * G.N + n
                                          : Js + (size_t)slot27(0, 0, -1) * G.N + n + sz);
        }
        __pipeline_commit();
    };
#pragma unroll
    for (int k = 0; k < kZlRing; ++k) issue(k);
    B4<T> Cp{T(0), T(0), T(0), T(0)};
    V2<T> gp{T(0), T(0)};
    uint8_t bc_prev = 0;
    uint8_t mk = bc[col];
    uint8_t bnext = (G.nz >= 1) ? bc[col + sz] : uint8_t(0);
    for (int k = 0; k <= G.nz; ++k) {
        const uint8_t bc_next = bnext;
        bnext = (k + 2 <= G.nz) ? bc[col + (k + 2) * sz] : uint8_t(0);
        // node k's group is complete once at most kZlRing - 1 newer ones pend
        __pipeline_wait_prior(kZlRing - 1);
        const int q = (k % kZlRing) * bsz + tx;
        const V2<T> bv = Rb[q];
        B4<T> di = Rdi[q];
        B4<M> qL{}, qU{};
        if (k > 0) qL = RL[q];
        if (k < G.nz) qU = RU[q];
        T rp = bv.p, rc = bv.c;
        if (mk & BC_P) rp = T(0);
        if (mk & BC_C) rc = T(0);
        if (TRANS) di = B4<T>{di.pp, di.cp, di.pc, di.cc};
        B4<T> Mk = inv2(di);
        if (k > 0) {
            const B4<T> L = mask_block(raw_line_block<T, M, TRANS>(qL), mk, bc_prev);
            const B4<T> LC = mul2(L, Cp);
            Mk.pp -= LC.pp; Mk.pc -= LC.pc; Mk.cp -= LC.cp; Mk.cc -= LC.cc;
            rp -= L.pp * gp.p + L.pc * gp.c;
            rc -= L.cp * gp.p + L.cc * gp.c;
        }
        const B4<T> Mi = inv2(Mk);
        if (k < G.nz) {
            const B4<T> U = mask_block(raw_line_block<T, M, TRANS>(qU), mk, bc_next);
            Cp = mul2(Mi, U);
            Cs[(size_t)k * bsz + tx] = Cp;
        }
        gp = V2<T>{Mi.pp * rp + Mi.pc * rc, Mi.cp * rp + Mi.cc * rc};
        gs[(size_t)k * bsz + tx] = gp;
        bc_prev = mk;
        mk = bc_next;
        // every value of slot q is in registers and used above: refill it
        issue(k + kZlRing);
    }
    __pipeline_wait_prior(0);
    V2<T> d = gp;
    for (int k = G.nz;; --k) {
        const int n = col + k * sz;
        if (k < G.nz) {
            const B4<T> C = Cs[(size_t)k * bsz + tx];
            const V2<T> g = gs[(size_t)k * bsz + tx];
            d = V2<T>{g.p - (C.pp * d.p + C.pc * d.c), g.c - (C.cp * d.p + C.cc * d.c)};
        }
        V2<T> xn{T(0), T(0)};
        if (MODE != 1) xn = xs[n];
        T op = xn.p + omega * d.p, oc = xn.c + omega * d.c;
        const uint8_t m = bc[n];
        if (m & BC_P) op = T(0);
        if (m & BC_C) oc = T(0);
        xo[on_ + n] = V2<T>{op, oc};
        if (k == 0) break;
    }
}

// Threads per block of the z-line sweep: as many as fit the per-thread
// Thomas storage and input ring in 96 KiB of shared memory (at least one
// warp).
template <class T, class M>
inline int zline_block(const Grid& G, size_t* smem)
{
    const size_t per = (size_t)G.nz * sizeof(B4<T>) + (size_t)(G.nz + 1) * sizeof(V2<T>) +
                       (size_t)kZlRing * (sizeof(B4<T>) + sizeof(V2<T>) + 2 * sizeof(B4<M>));
    int bs = (int)std::min<size_t>(kLineBS, (96 * 1024 / per) / 32 * 32);
    if (bs < 32) bs = 32;
    *smem = per * bs;
    return bs;
}

template <class T, class M>
void launch_smooth_zline(const Grid& G, const B4<M>* J, const B4<T>* Dinv, const uint8_t* bc,
                         const V2<T>* b, const V2<T>* x, V2<T>* xo, double omega, int trans,
                         const int* mask, int mstride, int S, cudaStream_t st, int mode)
{
    if (G.nz + 1 > kMaxLine) return;  // callers check the line limit first
    count_launch(1);
    size_t smem = 0;
    const int bs = zline_block<T, M>(G, &smem);
    dim3 grid(nblocks((G.nx + 1) * (G.ny + 1), bs), S);
    const T w = T(omega);
#define ELDER_ZL(TR, MO)                                                                       \
    do {                                                                                       \
        static bool attr_set = false;                                                          \
        if (!attr_set) {                                                                       \
            cudaFuncSetAttribute(k_smooth_zline<T, M, TR, MO>,                                 \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);     \
            attr_set = true;                                                                   \
        }                                                                                      \
        k_smooth_zline<T, M, TR, MO><<<grid, bs, smem, st>>>(G, J, Dinv, bc, b, x, xo, w, mask, \
                                                             mstride);                         \
    } while (0)
    if (mode == 1) {
        if (trans) ELDER_ZL(true, 1);
        else ELDER_ZL(false, 1);
    } else {
        if (trans) ELDER_ZL(true, 2);
        else ELDER_ZL(false, 2);
    }
#undef ELDER_ZL
}

// The lines of the sweeps.  FP32 (kLinePair): two threads per line, lanes 0-15
// of a warp walk 16 neighbouring lines up from the bottom, lanes 16-31 the same
// lines down from the top, both to the nodes next to the middle one, nz / 2: a
// line costs half its length in dependent steps and the launch has twice the
// threads.  FP64: one thread walks a line from the bottom, in the order of the
// textbook elimination; the FP64 solver's iterates do not change with the
// layout of its kernels (gradients of the adjoint switch with the sign of face
// fluxes that are zero to rounding, which makes another order visible).
template <class T> constexpr bool kLinePair = std::is_same<T, float>::value;

template <bool PAIR> struct LineThread {
    int col;    // the line (clamped to the last)
    bool up;    // the half above the middle
    bool live;  // the line exists
    int count;  // nodes of this thread's walk
    int end;    // its first node (the line's end)
    int step;   // to the next node
    __device__ __forceinline__ LineThread(const Grid& G, int sz)
    {
        const int t = blockIdx.x * blockDim.x + threadIdx.x;
        const int c = PAIR ? t / 32 * 16 + (t & 15) : t;
        live = c < sz;
        col = min(c, sz - 1);
        up = PAIR && (t & 16) != 0;
        const int m = G.nz >> 1;
        count = !PAIR ? G.nz + 1 : (up ? G.nz - m : m);
        end = up ? col + G.nz * sz : col;
        step = up ? -sz : sz;
    }
};

// Threads of a launch over all lines of a level.
template <class T> inline int line_threads(const Grid& G)
{
    return (kLinePair<T> ? 2 : 1) * (G.nx + 1) * (G.ny + 1);
}

// Factors of the vertical lines of a level's (non-transposed) operator, once
// per assembly.  FP32: a line is eliminated from both ends towards its middle node
// m = nz / 2: below it, with the diagonal blocks D and the masked line blocks L,
// U (lower, upper), M_k = D_k - L_k C_{k-1} and C_k = M_k^{-1} U_k, above it M_k =
// D_k - U_k C_{k+1} and C_k = M_k^{-1} L_k; the middle has both terms.  Stored
// per node: zMi = M_k^{-1}, zA = M_k^{-1} times the block towards the line's end
// (what the substitution needs of the previous node) and zC = C_k (the next
// one); at the middle zA = M_m^{-1} L_m and zC = M_m^{-1} U_m.  FP64: from the
// bottom to the top, zMi = M_k^{-1}, zA = L_k (masked), zC = C_k.  The serial walk,
// not the memory, is the time of these kernels on single samples and coarse
// levels.  D is the inverse of the stored inverse Dinv.
template <class T, class M>
__global__ void __launch_bounds__(128)
    k_zline_factor(Grid G, const B4<M>* __restrict__ Lz, const B4<M>* __restrict__ Uz,
                   size_t sst, const B4<T>* __restrict__ Dinv, const uint8_t* __restrict__ bc,
                   B4<T>* __restrict__ zMi, B4<T>* __restrict__ zA, B4<T>* __restrict__ zC,
                   const int* mask, int mstride)
{
    const int s = blockIdx.y;
    if (!on(mask, mstride, s)) return;
    const int sz = (G.nx + 1) * (G.ny + 1);
    const LineThread<kLinePair<T>> lt(G, sz);
    const size_t on_ = (size_t)s * G.N;
    const B4<M>* Lo = Lz + s * sst;
    const B4<M>* Up = Uz + s * sst;
    // towards the line's end (in) and towards the middle (to)
    const B4<M>*In = lt.up ? Up : Lo, *To = lt.up ? Lo : Up;
    B4<T> Cp{T(0), T(0), T(0), T(0)};
    uint8_t mprev = 0;
    int n = lt.end;
    if constexpr (!kLinePair<T>) {
        if (!lt.live) return;
        zA[on_ + n] = Cp;
        for (int k = 0; k <= G.nz; ++k) {
            const int n = lt.col + k * sz;
            const uint8_t mk = bc[n];
            B4<T> Mk = inv2(Dinv[on_ + n]);
            if (k > 0) {
                const B4<T> L = mask_block(raw_line_block<T, M, false>(Lo[n]), mk, mprev);
                const B4<T> LC = mul2(L, Cp);
                Mk.pp -= LC.pp; Mk.pc -= LC.pc; Mk.cp -= LC.cp; Mk.cc -= LC.cc;
                zA[on_ + n] = L;
            }
            const B4<T> Mi = inv2(Mk);
            zMi[on_ + n] = Mi;
            if (k < G.nz) {
                const uint8_t bn = bc[n + sz];
                const B4<T> U = mask_block(raw_line_block<T, M, false>(Up[n]), mk, bn);
                Cp = mul2(Mi, U);
                zC[on_ + n] = Cp;
            }
            mprev = mk;
        }
        return;
    }
#pragma unroll 4
    for (int i = 0; i < lt.count; ++i, n += lt.step) {
        const uint8_t mk = bc[n], mn = bc[n + lt.step];
        B4<T> Mk = inv2(Dinv[on_ + n]);
        const B4<T> A = mask_block(raw_line_block<T, M, false>(In[n]), mk, mprev);
        const B4<T> B = mask_block(raw_line_block<T, M, false>(To[n]), mk, mn);
        const bool inner = i > 0;  // (the block of a line's end points nowhere)
        const B4<T> AC = mul2(A, Cp);
        if (inner) { Mk.pp -= AC.pp; Mk.pc -= AC.pc; Mk.cp -= AC.cp; Mk.cc -= AC.cc; }
        const B4<T> Mi = inv2(Mk);
        Cp = mul2(Mi, B);
        if (lt.live) {
            zMi[on_ + n] = Mi;
            zA[on_ + n] = inner ? mul2(Mi, A) : B4<T>{T(0), T(0), T(0), T(0)};
            zC[on_ + n] = Cp;
        }
        mprev = mk;
    }
    // the middle node: the other half's last factor crosses the warp
    const int m = lt.col + (G.nz >> 1) * sz;
    const bool below = (G.nz >> 1) > 0, above = G.nz > (G.nz >> 1);
    const B4<T> Co{__shfl_xor_sync(0xffffffffu, Cp.pp, 16), __shfl_xor_sync(0xffffffffu, Cp.pc, 16),
                   __shfl_xor_sync(0xffffffffu, Cp.cp, 16),
                   __shfl_xor_sync(0xffffffffu, Cp.cc, 16)};
    if (lt.up || !lt.live) return;
    const uint8_t mk = bc[m];
    B4<T> Mk = inv2(Dinv[on_ + m]);
    B4<T> L{T(0), T(0), T(0), T(0)}, U = L;
    if (below) {
        L = mask_block(raw_line_block<T, M, false>(Lo[m]), mk, bc[m - sz]);
        const B4<T> LC = mul2(L, Cp);
        Mk.pp -= LC.pp; Mk.pc -= LC.pc; Mk.cp -= LC.cp; Mk.cc -= LC.cc;
    }
    if (above) {
        U = mask_block(raw_line_block<T, M, false>(Up[m]), mk, bc[m + sz]);
        const B4<T> UC = mul2(U, Co);
        Mk.pp -= UC.pp; Mk.pc -= UC.pc; Mk.cp -= UC.cp; Mk.cc -= UC.cc;
    }
    const B4<T> Mi = inv2(Mk);
    zMi[on_ + m] = Mi;
    zA[on_ + m] = mul2(Mi, L);
    zC[on_ + m] = mul2(Mi, U);
}

template <class T, class M>
void launch_zline_factor(const Grid& G, const B4<M>* Lz, const B4<M>* Uz, size_t sst,
                         const B4<T>* Dinv, const uint8_t* bc, B4<T>* zMi, B4<T>* zA, B4<T>* zC,
                         const int* mask, int mstride, int S, cudaStream_t st)
{
    count_launch(1);
    // (blocks for every SM, as the sweep)
    const int lines = line_threads<T>(G);
    const int bs = spread_block(128, lines, S);
    dim3 grid(nblocks(lines, bs), S);
    k_zline_factor<T, M><<<grid, bs, 0, st>>>(G, Lz, Uz, sst, Dinv, bc, zMi, zA, zC, mask,
                                              mstride);
}

// One damped z-line sweep with the factors of k_zline_factor: g_k = zMi_k r_k -
// zA_k g_{previous} from both ends to the middle (FP64: g_k = zMi_k (r_k - zA_k
// g_{k-1}) from the bottom), then d_k = g_k - zC_k d_{next} and x_out = x + omega d
// back out (x = 0 in MODE 1; in MODE 2 r is the masked residual b - A x).  A
// thread reads a chunk of kZaChunk nodes ahead of the recursion, so that a
// walk's time is its arithmetic (two dependent fused multiply-adds per node, FP64
// four) and not a memory latency per few nodes: 17 to 25 us per launch on single
// samples before.  g waits in shared memory, [i][thread].  An inactive line is
// clamped to the last one and not written.
constexpr int kZaChunk = 4;

template <class T, int MODE>
__global__ void __launch_bounds__(kBS)
    k_zline_apply(Grid G, const B4<T>* __restrict__ zMi, const B4<T>* __restrict__ zA,
                  const B4<T>* __restrict__ zC, const uint8_t* __restrict__ bc,
                  const V2<T>* __restrict__ r, const V2<T>* __restrict__ x, V2<T>* __restrict__ xo,
                  T omega, const int* mask, int mstride)
{
    extern __shared__ __align__(16) unsigned char za_smem[];
    V2<T>* gs = reinterpret_cast<V2<T>*>(za_smem) + threadIdx.x;
    const int s = blockIdx.y;
    if (!on(mask, mstride, s)) return;
    const int sz = (G.nx + 1) * (G.ny + 1), bs = blockDim.x;
    const LineThread<kLinePair<T>> lt(G, sz);
    const size_t on_ = (size_t)s * G.N;
    zMi += on_; zA += on_; zC += on_; r += on_; xo += on_;
    if (MODE != 1) x += on_;
    auto masked = [&](int n) {
        V2<T> v = r[n];
        const uint8_t m = bc[n];
        if (m & BC_P) v.p = T(0);
        if (m & BC_C) v.c = T(0);
        return v;
    };
    B4<T> mi[kZaChunk], za[kZaChunk];
    V2<T> rv[kZaChunk];
    auto fetch = [&](int i0) {
#pragma unroll
        for (int q = 0; q < kZaChunk; ++q) {
            const int n = lt.end + min(i0 + q, max(lt.count - 1, 0)) * lt.step;
            mi[q] = zMi[n];
            za[q] = zA[n];
            rv[q] = masked(n);
        }
    };
    fetch(0);
    V2<T> g{T(0), T(0)};
    for (int i0 = 0; i0 < lt.count; i0 += kZaChunk) {
        B4<T> a[kZaChunk], mc[kLinePair<T> ? 1 : kZaChunk];
        V2<T> h[kZaChunk];  // zMi r: off the recursion (FP64: r)
#pragma unroll
        for (int q = 0; q < kZaChunk; ++q) {
            a[q] = za[q];
            if (kLinePair<T>)
                h[q] = V2<T>{fma(mi[q].pp, rv[q].p, mi[q].pc * rv[q].c),
                             fma(mi[q].cp, rv[q].p, mi[q].cc * rv[q].c)};
            else {
                h[q] = rv[q];
                mc[q] = mi[q];
            }
        }
        if (i0 + kZaChunk < lt.count) fetch(i0 + kZaChunk);
#pragma unroll
        for (int q = 0; q < kZaChunk; ++q) {
            if (i0 + q < lt.count) {
                g = V2<T>{fma(-a[q].pp, g.p, fma(-a[q].pc, g.c, h[q].p)),
                          fma(-a[q].cp, g.p, fma(-a[q].cc, g.c, h[q].c))};
                if constexpr (!kLinePair<T>)
                    g = V2<T>{fma(mc[q].pp, g.p, mc[q].pc * g.c),
                              fma(mc[q].cp, g.p, mc[q].cc * g.c)};
                gs[(i0 + q) * bs] = g;
            }
        }
    }
    // backward factors of the nodes next to the middle, and the middle itself
    const int m = lt.col + (G.nz >> 1) * sz;
    V2<T> xv[kZaChunk];
    auto fetch_back = [&](int i1) {
#pragma unroll
        for (int q = 0; q < kZaChunk; ++q) {
            const int n = lt.end + max(i1 - q, 0) * lt.step;
            mi[q] = zC[n];
            if (MODE != 1) xv[q] = x[n];
        }
    };
    V2<T> d;
    auto put = [&](int n, V2<T> xn) {
        if (lt.live) xo[n] = V2<T>{fma(omega, d.p, xn.p), fma(omega, d.c, xn.c)};
    };
    // a whole walk ends at its last node, whose g is d
    int last = lt.count - 1;
    if constexpr (!kLinePair<T>) {
        d = g;
        const int n = lt.end + last * lt.step;
        put(n, MODE != 1 ? x[n] : V2<T>{T(0), T(0)});
        --last;
    }
    fetch_back(last);
    if constexpr (kLinePair<T>) {
        const B4<T> Mm = zMi[m], Am = zA[m], Cm = zC[m];
        const V2<T> rm = masked(m);
        const V2<T> o{__shfl_xor_sync(0xffffffffu, g.p, 16), __shfl_xor_sync(0xffffffffu, g.c, 16)};
        const V2<T> gl = lt.up ? o : g, gu = lt.up ? g : o;
        d.p = fma(-Am.pp, gl.p, fma(-Am.pc, gl.c, fma(Mm.pp, rm.p, Mm.pc * rm.c)));
        d.c = fma(-Am.cp, gl.p, fma(-Am.cc, gl.c, fma(Mm.cp, rm.p, Mm.cc * rm.c)));
        d.p = fma(-Cm.pp, gu.p, fma(-Cm.pc, gu.c, d.p));
        d.c = fma(-Cm.cp, gu.p, fma(-Cm.cc, gu.c, d.c));
        if (!lt.up) put(m, MODE != 1 ? x[m] : V2<T>{T(0), T(0)});
    }
    for (int i1 = last; i1 >= 0; i1 -= kZaChunk) {
        B4<T> c[kZaChunk];
        V2<T> xn[kZaChunk];
#pragma unroll
        for (int q = 0; q < kZaChunk; ++q) {
            c[q] = mi[q];
            xn[q] = MODE != 1 ? xv[q] : V2<T>{T(0), T(0)};
        }
        if (i1 - kZaChunk >= 0) fetch_back(i1 - kZaChunk);
#pragma unroll
        for (int q = 0; q < kZaChunk; ++q) {
            if (i1 - q >= 0) {
                const V2<T> gk = gs[(i1 - q) * bs];
                d = V2<T>{fma(-c[q].pp, d.p, fma(-c[q].pc, d.c, gk.p)),
                          fma(-c[q].cp, d.p, fma(-c[q].cc, d.c, gk.c))};
                put(lt.end + (i1 - q) * lt.step, xn[q]);
            }
        }
    }
}

template <class T>
void launch_zline_apply(const Grid& G, const B4<T>* zMi, const B4<T>* zA, const B4<T>* zC,
                        const uint8_t* bc, const V2<T>* r, const V2<T>* x, V2<T>* xo,
                        double omega, const int* mask, int mstride, int S, cudaStream_t st,
                        int mode, int bs)
{
    count_launch(1);
    // at most 64 KiB of waiting values per block, and blocks for every SM
    // where the grid has the lines (a walk is latency: it gains from an SM's
    // idle issue slots, not from neighbours)
    const int walk = kLinePair<T> ? G.nz - (G.nz >> 1) : G.nz + 1, lines = line_threads<T>(G);
    while (bs > 32 && sizeof(V2<T>) * walk * bs > 64 * 1024) bs /= 2;
    bs = spread_block(bs, lines, S);
    dim3 grid(nblocks(lines, bs), S);
    const size_t smem = sizeof(V2<T>) * walk * bs;
    if (mode == 1)
        launch_smem(k_zline_apply<T, 1>, grid, bs, smem, st, G, zMi, zA, zC, bc, r, x, xo,
                    T(omega), mask, mstride);
    else
        launch_smem(k_zline_apply<T, 2>, grid, bs, smem, st, G, zMi, zA, zC, bc, r, x, xo,
                    T(omega), mask, mstride);
}

// SPC samples per CTA: a thread forms the residual of its node in SPC
// samples, whose loads are independent (more loads in flight per thread at
// the price of registers); the autotuner picks SPC with the block size.  The
// loads of an inactive sample read sample s0's rows and its result is not
// stored.  At SPC = 1, at most 32 registers: every warp slot of an SM can
// then hold a warp, which this latency-bound stencil needs (at 34 a quarter
// stayed empty).
template <class T, class M, bool TRANS, int SPC>
__global__ void __launch_bounds__(kMaxBS, (2048 / kMaxBS) / SPC)
    k_mg_residual(Grid G, const B4<M>* __restrict__ J, const uint8_t* __restrict__ bc,
                  const V2<T>* __restrict__ b, const V2<T>* __restrict__ x,
                  V2<T>* __restrict__ r, const int* mask, int mstride, int S)
{
    const int s0 = blockIdx.y * SPC;
    bool act[SPC];
    bool any = false;
#pragma unroll
    for (int q = 0; q < SPC; ++q) {
        act[q] = s0 + q < S && on(mask, mstride, s0 + q);
        any = any || act[q];
    }
    if (!any) return;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= G.N) return;
    int i, j, k;
    node_ijk(G, n, i, j, k);
    T yp[SPC], yc[SPC];
#pragma unroll
    for (int q = 0; q < SPC; ++q) {
        const size_t s = act[q] ? s0 + q : s0;
        stencil_apply<T, TRANS, M>(G, J + s * 27 * G.N, x + s * G.N, n, i, j, k, yp[q], yc[q]);
    }
    const uint8_t m = bc[n];
#pragma unroll
    for (int q = 0; q < SPC; ++q) {
        if (!act[q]) continue;
        const size_t on_ = (size_t)(s0 + q) * G.N;
        const V2<T> bv = b[on_ + n];
        T rp = bv.p - yp[q], rc = bv.c - yc[q];
        if (m & BC_P) rp = T(0);
        if (m & BC_C) rc = T(0);
        r[on_ + n] = V2<T>{rp, rc};
    }
}

template <class T, class M>
void launch_mg_residual(const Grid& G, const B4<M>* J, const uint8_t* bc,
                        const V2<T>* b, const V2<T>* x, V2<T>* r, int trans,
                        const int* mask, int mstride, int S, cudaStream_t st, int bs, int spc)
{
    count_launch(1);
    bs = spread_block(bs, G.N, (S + spc - 1) / spc);
    dim3 grid(nblocks(G.N, bs), (S + spc - 1) / spc);
#define ELDER_MGR(TR, SP) \
    k_mg_residual<T, M, TR, SP><<<grid, bs, 0, st>>>(G, J, bc, b, x, r, mask, mstride, S)
    if (spc == 2) {
        if (trans) ELDER_MGR(true, 2);
        else ELDER_MGR(false, 2);
    } else {
        if (trans) ELDER_MGR(true, 1);
        else ELDER_MGR(false, 1);
    }
#undef ELDER_MGR
}

// Full weighting = transpose of trilinear interpolation on the vertex-centred
// 2:1 hierarchy (coarse node (I,J,K) is fine node (2I,2J,2K)).
template <class T>
__global__ void __launch_bounds__(kBS)
    k_restrict(Grid Gf, Grid Gc, const uint8_t* __restrict__ bcc,
               const V2<T>* __restrict__ rf, V2<T>* __restrict__ bco,
               const int* mask, int mstride)
{
    const int s = blockIdx.y;
    if (!on(mask, mstride, s)) return;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= Gc.N) return;
    int I, J, K;
    node_ijk_fast(Gc, n, I, J, K);
    rf += (size_t)s * Gf.N;
    T sp = T(0), sc = T(0);
#pragma unroll
    for (int c = -1; c <= 1; ++c)
#pragma unroll
        for (int b = -1; b <= 1; ++b)
#pragma unroll
            for (int a = -1; a <= 1; ++a) {
                const int fi = 2 * I + a, fj = 2 * J + b, fk = 2 * K + c;
                if (fi < 0 || fi > Gf.nx || fj < 0 || fj > Gf.ny || fk < 0 || fk > Gf.nz)
                    continue;
                const T w = T((a == 0 ? 1.0 : 0.5) * (b == 0 ? 1.0 : 0.5) * (c == 0 ? 1.0 : 0.5));
                const V2<T> v = rf[node_id(Gf, fi, fj, fk)];
                sp += w * v.p;
                sc += w * v.c;
            }
    const uint8_t m = bcc[n];
    if (m & BC_P) sp = T(0);
    if (m & BC_C) sc = T(0);
    bco[(size_t)s * Gc.N + n] = V2<T>{sp, sc};
}

template <class T>
void launch_restrict(const Grid& Gf, const Grid& Gc, const uint8_t* bcc,
                     const V2<T>* rf, V2<T>* bco, const int* mask, int mstride,
                     int S, cudaStream_t st)
{
    count_launch(1);
    const int bs = spread_block(kBS, Gc.N, S);
    dim3 grid(nblocks(Gc.N, bs), S);
    k_restrict<T><<<grid, bs, 0, st>>>(Gf, Gc, bcc, rf, bco, mask, mstride);
}

template <class T>
__global__ void __launch_bounds__(kBS)
    k_prolong_add(Grid Gf, Grid Gc, const uint8_t* __restrict__ bcf,
                  const V2<T>* __restrict__ xc, V2<T>* __restrict__ xf,
                  const int* mask, int mstride)
{
    const int s = blockIdx.y;
    if (!on(mask, mstride, s)) return;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= Gf.N) return;
    int i, j, k;
    node_ijk_fast(Gf, n, i, j, k);
    xc += (size_t)s * Gc.N;
    // trilinear interpolation as three nested averages of the 8 coarse
    // parents; for an even fine index both parents are the same node, whose
    // average is exact, so no branch depends on the parity
    const int sxc = Gc.nx + 1, szc = (Gc.nx + 1) * (Gc.ny + 1);
    const int c0 = (i >> 1) + sxc * (j >> 1) + szc * (k >> 1);
    const int di = i & 1, dj = (j & 1) * sxc, dk = (k & 1) * szc;
    V2<T> v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
        v[q] = xc[c0 + ((q & 1) ? di : 0) + ((q & 2) ? dj : 0) + ((q & 4) ? dk : 0)];
    const T h = T(0.5);
    T ap[4], ac[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        ap[q] = h * (v[2 * q].p + v[2 * q + 1].p);
        ac[q] = h * (v[2 * q].c + v[2 * q + 1].c);
    }
    const T bp0 = h * (ap[0] + ap[1]), bp1 = h * (ap[2] + ap[3]);
    const T bc0 = h * (ac[0] + ac[1]), bc1 = h * (ac[2] + ac[3]);
    const T sp = h * (bp0 + bp1), sc = h * (bc0 + bc1);
    const uint8_t m = bcf[n];
    V2<T> o = xf[(size_t)s * Gf.N + n];
    o.p = (m & BC_P) ? T(0) : o.p + sp;
    o.c = (m & BC_C) ? T(0) : o.c + sc;
    xf[(size_t)s * Gf.N + n] = o;
}

template <class T>
void launch_prolong_add(const Grid& Gf, const Grid& Gc, const uint8_t* bcf,
                        const V2<T>* xc, V2<T>* xf, const int* mask,
                        int mstride, int S, cudaStream_t st)
{
    count_launch(1);
    const int bs = spread_block(kBS, Gf.N, S);
    dim3 grid(nblocks(Gf.N, bs), S);
    k_prolong_add<T><<<grid, bs, 0, st>>>(Gf, Gc, bcf, xc, xf, mask, mstride);
}

// x = A_c^{-1} b on the coarsest grid, one block per sample; the inverse lies
// by columns.  Latency-bound (n loads of the inverse per unknown): kCaSplit
// threads share an unknown's sum, each over every kCaSplit-th term, so that a
// thread has n / kCaSplit independent loads.  The plain product reads a column
// per step (coalesced over the unknowns); the transposed one a row segment.
// FP64 keeps one running sum per unknown.
template <class T> constexpr int kCaSplit = std::is_same<T, float>::value ? 4 : 1;

template <class T>
__global__ void __launch_bounds__(1024)
    k_coarse_apply(int n, const T* __restrict__ Ainv, const V2<T>* __restrict__ b,
                   V2<T>* __restrict__ x, int trans, const int* mask, int mstride)
{
    extern __shared__ __align__(16) unsigned char ca_smem[];
    T* bs = reinterpret_cast<T*>(ca_smem);  // [n]
    T* part = bs + n;                       // [kCaSplit][n]
    const int s = blockIdx.x;
    if (!on(mask, mstride, s)) return;
    const T* bb = reinterpret_cast<const T*>(b + (size_t)s * (n / 2));
    for (int q = threadIdx.x; q < n; q += blockDim.x) bs[q] = bb[q];
    __syncthreads();
    const T* A = Ainv + (size_t)s * n * n;
    for (int e = threadIdx.x; e < n * kCaSplit<T>; e += blockDim.x) {
        // plain: consecutive threads take consecutive unknowns; transposed:
        // the kCaSplit threads of an unknown are neighbours
        const int r = trans ? e / kCaSplit<T> : e % n, c = trans ? e % kCaSplit<T> : e / n;
        T acc = T(0);
        if (!trans) {
#pragma unroll 8
            for (int q = c; q < n; q += kCaSplit<T>) acc = fma(A[(size_t)q * n + r], bs[q], acc);
        } else {
#pragma unroll 8
            for (int q = c; q < n; q += kCaSplit<T>) acc = fma(A[(size_t)r * n + q], bs[q], acc);
        }
        part[c * n + r] = acc;
    }
    __syncthreads();
    T* xx = reinterpret_cast<T*>(x + (size_t)s * (n / 2));
    for (int r = threadIdx.x; r < n; r += blockDim.x)
        xx[r] = kCaSplit<T> == 1 ? part[r]
                                 : (part[r] + part[n + r]) + (part[2 * n + r] + part[3 * n + r]);
}

template <class T>
void launch_coarse_apply(const Grid& G, const double* Ainv, const V2<T>* b,
                         V2<T>* x, int trans, const int* mask, int mstride,
                         int S, cudaStream_t st)
{
    count_launch(1);
    const int n = 2 * G.N;
    const int threads = std::min(1024, (n * kCaSplit<T> + 31) / 32 * 32);
    // the inverse is stored in the solver's arithmetic (CoarseType of its
    // multigrid storage type: FP32 for the mixed solver, FP64 otherwise)
    launch_smem(k_coarse_apply<T>, dim3(S), threads, sizeof(T) * n * (1 + kCaSplit<T>), st, n,
                reinterpret_cast<const T*>(Ainv), b, x, trans, mask, mstride);
}

// ---------------------------------------------------------------------------
// BiCGStab vector updates and per-sample scalars
// ---------------------------------------------------------------------------

template <class T>
__global__ void __launch_bounds__(kBS)
    k_bicg_init(Grid G, const uint8_t* __restrict__ bc, const V2<T>* __restrict__ b,
                V2<T>* x, V2<T>* r, V2<T>* rh, V2<T>* p, V2<T>* v,
                double* __restrict__ partial, const KScal* ks)
{
    __shared__ double red[32];
    const int s = blockIdx.y;
    if (!ks[s].active) return;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    double d = 0.0;
    if (n < G.N) {
        const size_t q = (size_t)s * G.N + n;
        V2<T> bv = b[q];
        const uint8_t m = bc[n];
        if (m & BC_P) bv.p = T(0);
        if (m & BC_C) bv.c = T(0);
        const V2<T> z{T(0), T(0)};
        x[q] = z;
        p[q] = z;
        v[q] = z;
        r[q] = bv;
        rh[q] = bv;
        d = dot2(bv.p, bv.c, bv.p, bv.c);
    }
    const double t = block_sum(d, red);
    if (threadIdx.x == 0) partial[((size_t)s * 2) * gridDim.x + blockIdx.x] = t;
}

template <class T>
void launch_bicg_init(const Grid& G, const uint8_t* bc, const V2<T>* b,
                      V2<T>* x, V2<T>* r, V2<T>* rh, V2<T>* p, V2<T>* v,
                      double* partial, KScal* ks, int S, cudaStream_t st)
{
    count_launch(1);
    dim3 grid(nblocks(G.N), S);
    k_bicg_init<T><<<grid, kBS, 0, st>>>(G, bc, b, x, r, rh, p, v, partial, ks);
}

template <class T>
__global__ void __launch_bounds__(kBS)
    k_bicg_p(int N, const V2<T>* __restrict__ r, const V2<T>* __restrict__ v,
             V2<T>* __restrict__ p, const KScal* ks)
{
    const int s = blockIdx.y;
    const KScal k = ks[s];
    if (!k.active) return;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const T b = ks_beta<T>(k), w = ks_omega<T>(k);
    const size_t q = (size_t)s * N + n;
    const V2<T> rv = r[q], vv = v[q];
    V2<T> pv = p[q];
    pv.p = rv.p + b * (pv.p - w * vv.p);
    pv.c = rv.c + b * (pv.c - w * vv.c);
    p[q] = pv;
}

template <class T>
void launch_bicg_p(const Grid& G, const V2<T>* r, const V2<T>* v, V2<T>* p,
                   const KScal* ks, int S, cudaStream_t st)
{
    count_launch(1);
    const int bs = spread_block(kBS, G.N, S);
    dim3 grid(nblocks(G.N, bs), S);
    k_bicg_p<T><<<grid, bs, 0, st>>>(G.N, r, v, p, ks);
}

template <class T>
__global__ void __launch_bounds__(kBS)
    k_bicg_s(int N, const V2<T>* __restrict__ r, const V2<T>* __restrict__ v,
             V2<T>* __restrict__ sv, const KScal* ks)
{
    const int s = blockIdx.y;
    const KScal k = ks[s];
    if (!k.active) return;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const T a = ks_alpha<T>(k);
    const size_t q = (size_t)s * N + n;
    const V2<T> rv = r[q], vv = v[q];
    sv[q] = V2<T>{rv.p - a * vv.p, rv.c - a * vv.c};
}

template <class T>
void launch_bicg_s(const Grid& G, const V2<T>* r, const V2<T>* v, V2<T>* s,
                   double* partial, const KScal* ks, int S, cudaStream_t st)
{
    count_launch(1);
    (void)partial;
    const int bs = spread_block(kBS, G.N, S);
    dim3 grid(nblocks(G.N, bs), S);
    k_bicg_s<T><<<grid, bs, 0, st>>>(G.N, r, v, s, ks);
}

// Each thread updates kXrNodes consecutive-stride nodes and sums its own
// terms of the two inner products before the FP64 block reduction (for the
// FP32 solver the per-thread sum is FP32, see dot2).
constexpr int kXrNodes = 4;

template <class T>
__global__ void __launch_bounds__(kBS)
    k_bicg_xr(int N, const V2<T>* __restrict__ ph, const V2<T>* __restrict__ sh,
              const V2<T>* __restrict__ sv, const V2<T>* __restrict__ t,
              const V2<T>* __restrict__ rh, V2<T>* __restrict__ x,
              V2<T>* __restrict__ r, double* __restrict__ partial,
              const KScal* ks)
{
    __shared__ double red[32];
    const int s = blockIdx.y;
    const KScal k = ks[s];
    if (!k.active) return;
    const T a = ks_alpha<T>(k), w = ks_omega<T>(k);
    T l0 = T(0), l1 = T(0);
    const int stride = gridDim.x * blockDim.x;
#pragma unroll
    for (int u = 0; u < kXrNodes; ++u) {
        const int n = blockIdx.x * blockDim.x + threadIdx.x + u * stride;
        if (n < N) {
            const size_t q = (size_t)s * N + n;
            const V2<T> pv = ph[q], shv = sh[q], svv = sv[q], tv = t[q], rhv = rh[q];
            V2<T> xv = x[q];
            xv.p += a * pv.p + w * shv.p;
            xv.c += a * pv.c + w * shv.c;
            x[q] = xv;
            const V2<T> rv{svv.p - w * tv.p, svv.c - w * tv.c};
            r[q] = rv;
            l0 += rv.p * rv.p + rv.c * rv.c;
            l1 += rhv.p * rv.p + rhv.c * rv.c;
        }
    }
    const double t0 = block_sum((double)l0, red);
    const double t1 = block_sum((double)l1, red);
    if (threadIdx.x == 0) {
        partial[((size_t)s * 2 + 0) * gridDim.x + blockIdx.x] = t0;
        partial[((size_t)s * 2 + 1) * gridDim.x + blockIdx.x] = t1;
    }
}

template <class T>
void launch_bicg_xr(const Grid& G, const V2<T>* ph, const V2<T>* sh,
                    const V2<T>* s, const V2<T>* t, const V2<T>* rh, V2<T>* x,
                    V2<T>* r, double* partial, const KScal* ks, int S,
                    cudaStream_t st)
{
    count_launch(1);
    dim3 grid(bicg_xr_blocks(G.N), S);
    k_bicg_xr<T><<<grid, kBS, 0, st>>>(G.N, ph, sh, s, t, rh, x, r, partial, ks);
}

// Threads of a block that sums nblk partials of one sample.  A block's time
// is its number of dependent load batches: at 256x256x64 the products leave
// 134 k partials per sum, which 128 threads read in 1,048 dependent rounds
// (391 us); 1024 threads with 8 loads in flight need 17.  Two samples of that
// grid: 302 -> 233 ms per step; one at 128x128x32: 30.3 -> 27.3 ms.  Up to 4096
// partials 128 threads take at most 4 batches and fix the order of the sums.
inline int finalize_threads(int nblk)
{
    int t = 128;
    while (nblk > 4096 && t < 1024 && 8 * t < nblk) t *= 2;
    return t;
}

// This thread's share of sum_q v[q], q < n: one running sum, 8 loads ahead.
__device__ __forceinline__ double strided_sum(const double* __restrict__ v, int n)
{
    double a = 0.0;
    const int st = blockDim.x;
    int q = threadIdx.x;
    for (; q + 7 * st < n; q += 8 * st) {
        double b[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) b[u] = v[q + u * st];
#pragma unroll
        for (int u = 0; u < 8; ++u) a += b[u];
    }
    for (; q < n; q += st) a += v[q];
    return a;
}

// This thread's share of the larger of 0 and max_q v[q], q < n.
__device__ __forceinline__ double strided_max(const double* __restrict__ v, int n)
{
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    const int st = blockDim.x;
    int q = threadIdx.x;
    for (; q + 3 * st < n; q += 4 * st) {
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = fmax(a[u], v[q + u * st]);
    }
    for (; q < n; q += st) a[0] = fmax(a[0], v[q]);
    return fmax(fmax(a[0], a[1]), fmax(a[2], a[3]));
}

// One block per sample: fixed-order sums of the partials and the BiCGStab
// scalar recurrences.
__global__ void k_bicg_finalize(int stage, const double* __restrict__ partial,
                                int nblk, KScal* ks, double rtol, int maxit)
{
    __shared__ double red[32];
    const int s = blockIdx.x;
    KScal k = ks[s];
    if (!k.active) return;
    // (stages 0 and 1 have one inner product; the second array is not written)
    const bool two = stage >= 2;
    double a0 = strided_sum(partial + ((size_t)s * 2 + 0) * nblk, nblk);
    double a1 = two ? strided_sum(partial + ((size_t)s * 2 + 1) * nblk, nblk) : 0.0;
    a0 = block_sum(a0, red);
    if (two) a1 = block_sum(a1, red);
    if (threadIdx.x != 0) return;
    if (stage == 0) {  // after init: ||b||^2 = (rh, r)
        k.bn2 = a0;
        k.rn2 = a0;
        k.rho = a0;
        k.rho_old = 1.0;
        k.alpha = 1.0;
        k.omega = 1.0;
        k.iters = 0;
        k.status = 0;
        k.best_rn2 = a0;
        k.improved = 0;
        k.beta = 0.0;  // p = v = 0: the first update sets p = r
        k.alpha_f = 1.0f;
        k.omega_f = 1.0f;
        k.beta_f = 0.0f;
        if (!(a0 > 0.0)) {
            k.active = 0;
            if (!isfinite(a0)) k.status = ELDER_SAMPLE_NONFINITE_;
        }
    } else if (stage == 1) {  // alpha = rho / (rh, v)
        if (a0 == 0.0 || !isfinite(a0)) {
            k.active = 0;
            k.status = ELDER_SAMPLE_BREAKDOWN_;
        } else {
            k.alpha = k.rho / a0;
            k.alpha_f = (float)k.alpha;
        }
    } else if (stage == 2) {  // omega = (t, s) / (t, t)
        k.omega = (a1 > 0.0) ? a0 / a1 : 0.0;
        k.omega_f = (float)k.omega;
    } else {  // end of iteration: ||r||^2 and the next rho = (rh, r)
        k.rn2 = a0;
        k.rho_old = k.rho;
        k.rho = a1;
        k.iters += 1;
        k.improved = a0 < k.best_rn2;
        if (k.improved) k.best_rn2 = a0;
        k.beta = (k.omega != 0.0 && k.rho_old != 0.0) ? (k.rho / k.rho_old) * (k.alpha / k.omega)
                                                      : 0.0;
        k.beta_f = (float)k.beta;
        if (!isfinite(a0)) {
            k.active = 0;
            k.status = ELDER_SAMPLE_NONFINITE_;
        } else if (a0 <= rtol * rtol * k.bn2) {
            k.active = 0;
        } else if (k.iters >= maxit) {
            k.active = 0;
            k.status = ELDER_SAMPLE_KRYLOV_MAXIT_;
        } else if (k.rho == 0.0 || k.omega == 0.0) {
            k.active = 0;
            k.status = ELDER_SAMPLE_BREAKDOWN_;
        }
    }
    ks[s] = k;
}

void launch_bicg_finalize(int stage, const double* partial, int nblk,
                          KScal* ks, double rtol, int maxit, int S,
                          cudaStream_t st)
{
    count_launch(1);
    k_bicg_finalize<<<S, finalize_threads(nblk), 0, st>>>(stage, partial, nblk, ks, rtol, maxit);
}

template <class T>
__global__ void k_bicg_keep(int N, V2<T>* __restrict__ x, V2<T>* __restrict__ xbest,
                            const KScal* ks, int keep)
{
    const int s = blockIdx.y;
    const KScal& k = ks[s];
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const size_t q = (size_t)s * N + n;
    if (keep == 1) {
        if (k.improved) xbest[q] = x[q];
    } else if (k.status != 0 || k.active) {
        x[q] = xbest[q];
    }
}

template <class T>
void launch_bicg_keep(const Grid& G, V2<T>* x, V2<T>* xbest, const KScal* ks, int keep, int S,
                      cudaStream_t st)
{
    count_launch(1);
    dim3 grid(nblocks(G.N), S);
    k_bicg_keep<T><<<grid, kBS, 0, st>>>(G.N, x, xbest, ks, keep);
}

// ---------------------------------------------------------------------------
// Newton with line search
// ---------------------------------------------------------------------------

// which = 0: ||R(u)||, res0 and the round-off floor of ||R|| (2 eps times the
// norm of the per-row sums of the magnitudes of the summed terms);
// which = 1: ||R(u_trial)|| and the floor at the trial state
__global__ void k_norm_finalize(const double* __restrict__ partial,
                                const double* __restrict__ act, int nblk, NScal* ns,
                                int which)
{
    __shared__ double red[32];
    const int s = blockIdx.x;
    if (which == 1 && !ns[s].ls_active) return;
    if (which == 0 && !ns[s].active) return;
    double a = strided_sum(partial + (size_t)s * nblk, nblk);
    double b = act ? strided_sum(act + (size_t)s * nblk, nblk) : 0.0;
    a = block_sum(a, red);
    b = block_sum(b, red);
    if (threadIdx.x != 0) return;
    const double r = sqrt(a);
    if (which == 0) {
        ns[s].rn = r;
        ns[s].res0 = r;
        ns[s].rfloor = 2.0 * 2.220446049250313e-16 * sqrt(b);
        if (!isfinite(r)) {
            ns[s].active = 0;
            ns[s].ls_active = 0;
            ns[s].status = ELDER_SAMPLE_NONFINITE_;
        } else if (r <= ns[s].rfloor) {  // already a solution to round-off
            ns[s].active = 0;
            ns[s].ls_active = 0;
            ns[s].status = 0;
        }
    } else {
        ns[s].rt = r;
        ns[s].rfloor_t = 2.0 * 2.220446049250313e-16 * sqrt(b);
    }
}

void launch_norm_finalize(const double* partial, const double* act, int nblk, NScal* ns,
                          int which, int S, cudaStream_t st)
{
    count_launch(1);
    k_norm_finalize<<<S, finalize_threads(nblk), 0, st>>>(partial, act, nblk, ns, which);
}

template <class T>
__global__ void __launch_bounds__(kBS)
    k_newton_rhs(int N, const V2<double>* __restrict__ R, V2<T>* __restrict__ b,
                 const NScal* ns)
{
    const int s = blockIdx.y;
    if (!ns[s].active) return;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const size_t q = (size_t)s * N + n;
    const V2<double> r = R[q];
    b[q] = V2<T>{T(-r.p), T(-r.c)};
}

template <class T>
void launch_newton_rhs(const Grid& G, const V2<double>* R, V2<T>* b,
                       const NScal* ns, int S, cudaStream_t st)
{
    count_launch(1);
    const int bs = spread_block(kBS, G.N, S);
    dim3 grid(nblocks(G.N, bs), S);
    k_newton_rhs<T><<<grid, bs, 0, st>>>(G.N, R, b, ns);
}

template <class T>
__global__ void __launch_bounds__(kBS)
    k_newton_trial(int N, const double* __restrict__ p, const double* __restrict__ c,
                   const V2<T>* __restrict__ dx, double* __restrict__ pt,
                   double* __restrict__ ct, double* __restrict__ partial,
                   const NScal* ns)
{
    __shared__ double red[32];
    const int s = blockIdx.y;
    if (!ns[s].ls_active) return;
    const double lam = ns[s].lambda;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (std::is_same<T, float>::value) {
        // FP32 correction: lambda is a power of two (1 halved by the line
        // search), so lambda d is exact in FP32 (above 2^-126 in magnitude;
        // below, it rounds to FP32's subnormals, far under the rounding of p
        // and c) and its widening exact; the maxima of the magnitudes are
        // integer maxima of their bit patterns.  Neither touches the FP64
        // pipe, and the values equal the FP64 form's, lambda (double) d.
        const float lamf = d2f_trunc(lam);
        unsigned up = 0u, uc = 0u;
        if (n < N) {
            const size_t q = (size_t)s * N + n;
            const V2<T> d = dx[q];
            const float dpf = lamf * d.p, dcf = lamf * d.c;
            pt[q] = p[q] + f2d_exact(dpf);
            ct[q] = c[q] + f2d_exact(dcf);
            // a non-finite correction must never meet the Newton stop: NaN
            // enters the maxima as +inf
            up = mag_bits(dpf);
            uc = mag_bits(dcf);
        }
        unsigned* ured = reinterpret_cast<unsigned*>(red);
        const unsigned t0 = block_max(up, ured);
        const unsigned t1 = block_max(uc, ured);
        if (threadIdx.x == 0) {
            partial[((size_t)s * 2 + 0) * gridDim.x + blockIdx.x] = f2d_exact(__uint_as_float(t0));
            partial[((size_t)s * 2 + 1) * gridDim.x + blockIdx.x] = f2d_exact(__uint_as_float(t1));
        }
        return;
    }
    double mp = 0.0, mc = 0.0;
    if (n < N) {
        const size_t q = (size_t)s * N + n;
        const V2<T> d = dx[q];
        const double dp = lam * (double)d.p, dc = lam * (double)d.c;
        pt[q] = p[q] + dp;
        ct[q] = c[q] + dc;
        // a non-finite correction must never meet the Newton stop: block_max
        // (fmax) would drop a NaN, so it enters the maxima as +inf
        mp = isfinite(dp) ? fabs(dp) : INFINITY;
        mc = isfinite(dc) ? fabs(dc) : INFINITY;
    }
    const double t0 = block_max(mp, red);
    const double t1 = block_max(mc, red);
    if (threadIdx.x == 0) {
        partial[((size_t)s * 2 + 0) * gridDim.x + blockIdx.x] = t0;
        partial[((size_t)s * 2 + 1) * gridDim.x + blockIdx.x] = t1;
    }
}

template <class T>
void launch_newton_trial(const Grid& G, const double* p, const double* c,
                         const V2<T>* dx, double* pt, double* ct,
                         double* partial, const NScal* ns, int S,
                         cudaStream_t st)
{
    count_launch(1);
    dim3 grid(nblocks(G.N), S);
    k_newton_trial<T><<<grid, kBS, 0, st>>>(G.N, p, c, dx, pt, ct, partial, ns);
}

// Armijo-type acceptance ||R(u + lambda d)|| < (1 - 1e-4 lambda) ||R(u)||;
// after ls_max halvings the last trial is taken.
__global__ void k_newton_ls_finalize(const double* __restrict__ pmax, int nblk,
                                     NScal* ns, int ls_max)
{
    __shared__ double red[32];
    const int s = blockIdx.x;
    if (!ns[s].ls_active) return;
    double a0 = strided_max(pmax + ((size_t)s * 2 + 0) * nblk, nblk);
    double a1 = strided_max(pmax + ((size_t)s * 2 + 1) * nblk, nblk);
    a0 = block_max(a0, red);
    a1 = block_max(a1, red);
    if (threadIdx.x != 0) return;
    NScal k = ns[s];
    k.dmax_p = a0;
    k.dmax_c = a1;
    const bool finite = isfinite(k.rt);
    // a trial at the round-off floor of ||R|| is accepted as it is: below
    // that level the decrease test compares rounding noise
    if (finite && (k.rt < (1.0 - 1e-4 * k.lambda) * k.rn || k.rt <= k.rfloor_t)) {
        k.ls_active = 0;
        k.accepted = 1;
    } else if (k.ls_count >= ls_max) {  // no step length decreased ||R||
        k.ls_active = 0;
        k.active = 0;
        k.status = ELDER_SAMPLE_LINESEARCH_;
    } else {
        k.lambda *= 0.5;
        k.ls_count += 1;
        k.ls_cuts += 1;
    }
    ns[s] = k;
}

void launch_newton_ls_finalize(const double* partial_res,
                               const double* partial_max, int nblk,
                               NScal* ns, int ls_max, int S, cudaStream_t st)
{
    count_launch(1);
    (void)partial_res;
    k_newton_ls_finalize<<<S, finalize_threads(nblk), 0, st>>>(partial_max, nblk, ns, ls_max);
}

__global__ void __launch_bounds__(kBS)
    k_newton_accept(int N, double* __restrict__ p, double* __restrict__ c,
                    const double* __restrict__ pt, const double* __restrict__ ct,
                    V2<double>* __restrict__ R, const V2<double>* __restrict__ Rt,
                    const NScal* ns)
{
    const int s = blockIdx.y;
    if (!ns[s].accepted) return;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const size_t q = (size_t)s * N + n;
    p[q] = pt[q];
    c[q] = ct[q];
    if (!ns[s].skip_res) R[q] = Rt[q];  // else R stays that of the last evaluated iterate
}

void launch_newton_accept(const Grid& G, double* p, double* c,
                          const double* pt, const double* ct, V2<double>* R,
                          const V2<double>* Rt, const NScal* ns, int S,
                          cudaStream_t st)
{
    count_launch(1);
    const int bs = spread_block(kBS, G.N, S);
    dim3 grid(nblocks(G.N, bs), S);
    k_newton_accept<<<grid, bs, 0, st>>>(G.N, p, c, pt, ct, R, Rt, ns);
}

// With inexact linear solves Newton converges linearly: from two
// consecutive full steps the contraction is theta = |d_k| / |d_{k-1}| and
// the remaining error about theta / (1 - theta) |d_k|.  A full step stops
// the iteration when that estimate, or the last correction itself, is
// within tolerance.
__device__ __forceinline__ bool newton_small(const NScal& k, double tol_p, double tol_c,
                                             int estimate)
{
    if (k.lambda != 1.0) return false;
    if (k.dmax_c <= tol_c && k.dmax_p <= tol_p) return true;
    if (estimate && k.full_prev && k.dprev_c > 0.0 && k.dprev_p > 0.0) {
        const double th = fmax(k.dmax_c / k.dprev_c, k.dmax_p / k.dprev_p);
        if (th < 0.5) {
            const double f = th / (1.0 - th);
            return f * k.dmax_c <= tol_c && f * k.dmax_p <= tol_p;
        }
    }
    return false;
}

// Before the trial residual of a full step (lambda = 1): the sizes of the
// correction (per-block maxima of k_newton_trial) decide the stop already,
// and a sample that meets it is accepted without its trial residual (its
// Armijo test would only compare a converged iterate).
__global__ void k_newton_predict(const double* __restrict__ pmax, int nblk, NScal* ns,
                                 double tol_p, double tol_c, int estimate)
{
    __shared__ double red[32];
    const int s = blockIdx.x;
    if (!ns[s].ls_active || ns[s].lambda != 1.0) return;
    double a0 = strided_max(pmax + ((size_t)s * 2 + 0) * nblk, nblk);
    double a1 = strided_max(pmax + ((size_t)s * 2 + 1) * nblk, nblk);
    a0 = block_max(a0, red);
    a1 = block_max(a1, red);
    if (threadIdx.x != 0) return;
    NScal k = ns[s];
    k.dmax_p = a0;
    k.dmax_c = a1;
    if (newton_small(k, tol_p, tol_c, estimate)) {
        k.ls_active = 0;
        k.accepted = 1;
        k.skip_res = 1;
        ns[s] = k;
    }
}

void launch_newton_predict(const double* partial_max, int nblk, NScal* ns, double tol_p,
                           double tol_c, int estimate, int S, cudaStream_t st)
{
    count_launch(1);
    k_newton_predict<<<S, finalize_threads(nblk), 0, st>>>(partial_max, nblk, ns, tol_p, tol_c, estimate);
}

__global__ void k_newton_check(NScal* ns, const KScal* ks, double tol_p,
                               double tol_c, int maxit, int estimate, int S)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    NScal k = ns[s];
    if (!k.active) return;
    k.kiters += ks[s].iters;
    if (k.accepted) {
        k.iters += 1;
        if (k.skip_res) {
            // accepted by k_newton_predict: its correction met the stop (rn
            // stays the norm of the last evaluated iterate)
            k.active = 0;
            k.status = 0;
        } else {
            k.rn = k.rt;
            k.rfloor = k.rfloor_t;
            // the correction-size stop (or R at its round-off floor)
            const bool small = newton_small(k, tol_p, tol_c, estimate);
            k.full_prev = (k.lambda == 1.0);
            k.dprev_c = k.dmax_c;
            k.dprev_p = k.dmax_p;
            if (small || k.rn <= k.rfloor) {
                k.active = 0;
                k.status = 0;
            } else if (k.iters >= maxit) {
                k.active = 0;
                k.status = ELDER_SAMPLE_NEWTON_MAXIT_;
            }
        }
    }
    k.skip_res = 0;
    k.accepted = 0;
    k.ls_count = 0;
    k.lambda = 1.0;
    k.ls_active = k.active;
    ns[s] = k;
}

void launch_newton_check(NScal* ns, const KScal* ks, double tol_p,
                         double tol_c, int maxit, int estimate, int S, cudaStream_t st)
{
    count_launch(1);
    k_newton_check<<<nblocks(S, 128), 128, 0, st>>>(ns, ks, tol_p, tol_c, maxit, estimate, S);
}

// Newton's starting point from the last states: order 1 the linear
// extrapolation 2 u^n - u^{n-1}, order 2 the quadratic 3 u^n - 3 u^{n-1} +
// u^{n-2}; the salt fraction clipped to [0, 1] (Dirichlet values are imposed
// afterwards).  h1, h2 hold u^{n-1}, u^{n-2}.
__global__ void k_extrapolate(int N, int order, const double* __restrict__ p_n,
                              const double* __restrict__ c_n, const double* __restrict__ p1,
                              const double* __restrict__ c1, const double* __restrict__ p2,
                              const double* __restrict__ c2, double* __restrict__ p,
                              double* __restrict__ c)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const size_t q = (size_t)blockIdx.y * N + n;
    double pe, ce;
    if (order == 2) {
        pe = 3.0 * (p_n[q] - p1[q]) + p2[q];
        ce = 3.0 * (c_n[q] - c1[q]) + c2[q];
    } else {
        pe = 2.0 * p_n[q] - p1[q];
        ce = 2.0 * c_n[q] - c1[q];
    }
    p[q] = pe;
    c[q] = fmin(1.0, fmax(0.0, ce));
}

void launch_extrapolate(const Grid& G, int order, const double* p_n, const double* c_n,
                        const double* p1, const double* c1, const double* p2, const double* c2,
                        double* p, double* c, int S, cudaStream_t st)
{
    count_launch(1);
    dim3 grid(nblocks(G.N), S);
    k_extrapolate<<<grid, kBS, 0, st>>>(G.N, order, p_n, c_n, p1, c1, p2, c2, p, c);
}

__global__ void k_newton_restore_failed(int N, double* __restrict__ p,
                                        double* __restrict__ c,
                                        const double* __restrict__ p_old,
                                        const double* __restrict__ c_old,
                                        const NScal* ns)
{
    const int s = blockIdx.y;
    if (ns[s].status == 0) return;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const size_t q = (size_t)s * N + n;
    p[q] = p_old[q];
    c[q] = c_old[q];
}

void launch_newton_restore_failed(const Grid& G, double* p, double* c,
                                  const double* p_old, const double* c_old,
                                  const NScal* ns, int S, cudaStream_t st)
{
    count_launch(1);
    dim3 grid(nblocks(G.N), S);
    k_newton_restore_failed<<<grid, kBS, 0, st>>>(G.N, p, c, p_old, c_old, ns);
}

// ---------------------------------------------------------------------------
// sample statistics (Section 3: eqs. pdestat, numer_var; exceedance estimate)
// ---------------------------------------------------------------------------
//
// One pass over the S fields per node, shifted by the first sample's value
// for stability: with d_i = c_i - c_0, S1 = sum w d, S2 = sum w d^2,
// W = sum w: mean = c_0 W + S1 and sum w (mean - c)^2 =
// (mean - c_0)^2 W - 2 (mean - c_0) S1 + S2.
//
// Bound by FP64 issue (1/64 of the FP32 rate here): 7 operations per value
// (difference, weighted difference, both sums, W, the threshold comparison
// and its sum) took 264 us for 256 fields of 71,825 nodes, 22 us of them
// memory time.  Now 3 for equal weights (the weight is applied to the sums; 158
// us) and 4 or 5 for given ones: W is formed once per block, the comparison is an
// integer one, the equal-weight count an integer.  kMomSplit threads of
// different warps share a node, each over every kMomSplit-th field, to keep
// the FP64 pipe fed; their sums meet in shared memory in a fixed order.
constexpr int kMomSplit = 4;
constexpr int kMomNodes = kBS / kMomSplit;  // nodes per block

// x > t for finite or infinite x, t of either sign, false for NaN (integer
// operations: bit patterns as two's-complement numbers order like the values)
__device__ __forceinline__ long long order_key(double x)
{
    const long long b = __double_as_longlong(x);
    return b < 0 ? (long long)(0x8000000000000000ull - (unsigned long long)b) : b;
}

__device__ __forceinline__ bool exceeds(double x, long long tkey)
{
    constexpr long long inf = 0x7FF0000000000000ll;
    const long long k = order_key(x);
    return k > tkey && k <= inf;
}

// neither infinite nor NaN (an integer test)
__device__ __forceinline__ bool finite_bits(double x)
{
    return (__double2hiint(x) & 0x7FF00000) != 0x7FF00000;
}

template <bool WEIGHTED>
__global__ void __launch_bounds__(kBS)
    k_moments(int N, int S, double inv, const double* __restrict__ c,
              const double* __restrict__ w, double threshold,
              double* __restrict__ mean, double* __restrict__ var,
              double* __restrict__ pexc)
{
    __shared__ double red[32];
    __shared__ double part[3][kMomSplit][kMomNodes];
    const int q = threadIdx.x / kMomNodes, l = threadIdx.x % kMomNodes;
    const int n = blockIdx.x * kMomNodes + l;
    double W = 1.0;
    if (WEIGHTED) {
        W = 0.0;
        for (int s = threadIdx.x; s < S; s += kBS) W += w[s];
        W = block_sum(W, red);
    }
    // (a NaN threshold is exceeded by nothing)
    const long long tkey = threshold == threshold ? order_key(threshold) : 0x7FFFFFFFFFFFFFFFll;
    double S1 = 0.0, S2 = 0.0, P = 0.0, c0 = 0.0;
    if (n < N) {
        c0 = c[n];
        int count = 0;
        const double* cn = c + n;
#pragma unroll 8
        for (int s = q; s < S; s += kMomSplit) {
            const double cv = __ldcs(cn + (size_t)s * N);
            const double d = cv - c0;
            if (WEIGHTED) {
                const double ws = __ldg(w + s), wd = ws * d;
                S1 += wd;
                S2 = fma(wd, d, S2);
                if (exceeds(cv, tkey)) P += ws;
            } else {
                S1 += d;
                S2 = fma(d, d, S2);
                count += exceeds(cv, tkey) ? 1 : 0;
            }
        }
        if (!WEIGHTED) P = (double)count;
    }
    part[0][q][l] = S1;
    part[1][q][l] = S2;
    part[2][q][l] = P;
    __syncthreads();
    if (q != 0 || n >= N) return;
#pragma unroll
    for (int r = 1; r < kMomSplit; ++r) {
        S1 += part[0][r][l];
        S2 += part[1][r][l];
        P += part[2][r][l];
    }
    if (!WEIGHTED) {  // (inv: 1 / S; all of S fields count exactly 1)
        P = P == (double)S ? 1.0 : P * inv;
        if (finite_bits(S1) && finite_bits(S2)) {
            S1 *= inv;
            S2 *= inv;
        } else {  // beyond the range before the weight (or not finite): weigh every term
            S1 = S2 = 0.0;
            for (int s = 0; s < S; ++s) {
                const double d = c[(size_t)s * N + n] - c0, wd = inv * d;
                S1 += wd;
                S2 = fma(wd, d, S2);
            }
        }
    }
    const double m = fma(c0, W, S1);
    const double dm = m - c0;
    mean[n] = m;
    var[n] = fmax(fma(dm * dm, W, fma(-2.0 * dm, S1, S2)), 0.0);
    pexc[n] = P;
}

void launch_moments(int N, int S, const double* c, const double* w,
                    double threshold, double* mean, double* var,
                    double* pexc, cudaStream_t st)
{
    count_launch(1);
    const int grid = nblocks(N, kMomNodes);
    if (w)
        k_moments<true><<<grid, kBS, 0, st>>>(N, S, 1.0 / S, c, w, threshold, mean, var, pexc);
    else
        k_moments<false><<<grid, kBS, 0, st>>>(N, S, 1.0 / S, c, w, threshold, mean, var, pexc);
}

// ---------------------------------------------------------------------------
// helpers
// ---------------------------------------------------------------------------

__global__ void k_sum_partials(const double* __restrict__ partial, int nblk,
                               double* __restrict__ out)
{
    __shared__ double red[32];
    double a = strided_sum(partial + (size_t)blockIdx.x * nblk, nblk);
    a = block_sum(a, red);
    if (threadIdx.x == 0) out[blockIdx.x] = a;
}

void launch_sum_partials(const double* partial, int nblk, double* out, int S,
                         cudaStream_t st)
{
    count_launch(1);
    k_sum_partials<<<S, finalize_threads(nblk), 0, st>>>(partial, nblk, out);
}

// which = 0: y = a x on Dirichlet components only, 0 elsewhere;
// which = 1: y += a x on Dirichlet components only;
// which = 2: y += a x on interior components only.
template <class T>
__global__ void k_axpy_mask(Grid G, const uint8_t* __restrict__ bc,
                            const V2<T>* __restrict__ x, V2<T>* __restrict__ y,
                            double a, int which)
{
    const int s = blockIdx.y;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= G.N) return;
    const size_t q = (size_t)s * G.N + n;
    const uint8_t m = bc[n];
    const V2<T> xv = x[q];
    V2<T> yv = (which == 0) ? V2<T>{T(0), T(0)} : y[q];
    const bool dp = (m & BC_P) != 0, dc = (m & BC_C) != 0;
    if (which <= 1) {
        if (dp) yv.p += T(a) * xv.p;
        if (dc) yv.c += T(a) * xv.c;
    } else {
        if (!dp) yv.p += T(a) * xv.p;
        if (!dc) yv.c += T(a) * xv.c;
    }
    y[q] = yv;
}

template <class T>
void launch_axpy_mask(const Grid& G, const uint8_t* bc, const V2<T>* x,
                      V2<T>* y, double a, int which, int S, cudaStream_t st)
{
    count_launch(1);
    dim3 grid(nblocks(G.N), S);
    k_axpy_mask<T><<<grid, kBS, 0, st>>>(G, bc, x, y, a, which);
}

template <class Ts, class Td>
__global__ void k_convert(const V2<Ts>* __restrict__ x, V2<Td>* __restrict__ y,
                          size_t n)
{
    const size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const V2<Ts> v = x[q];
    y[q] = V2<Td>{Td(v.p), Td(v.c)};
}

template <class Ts, class Td>
void launch_convert(const V2<Ts>* x, V2<Td>* y, size_t n, cudaStream_t st)
{
    count_launch(1);
    k_convert<Ts, Td><<<(unsigned)((n + kBS - 1) / kBS), kBS, 0, st>>>(x, y, n);
}

// ---------------------------------------------------------------------------
// explicit instantiations
// ---------------------------------------------------------------------------
#define ELDER_INST(T)                                                                    \
    template void launch_spmv<T>(const Grid&, const B4<T>*, const uint8_t*,              \
                                 const V2<T>*, V2<T>*, int, int, const V2<T>*,           \
                                 double*, const int*, int, int, cudaStream_t, int);      \
    template void launch_smooth<T, MgType<T>::type>(                                     \
        const Grid&, const B4<MgType<T>::type>*, const B4<T>*, const uint8_t*,           \
        const V2<T>*, const V2<T>*, V2<T>*, double, int, const int*, int, int,           \
        cudaStream_t, int);                                                              \
    template void launch_mg_residual<T, MgType<T>::type>(                                \
        const Grid&, const B4<MgType<T>::type>*, const uint8_t*, const V2<T>*,           \
        const V2<T>*, V2<T>*, int, const int*, int, int, cudaStream_t, int, int);        \
    template void launch_restrict<T>(const Grid&, const Grid&, const uint8_t*,           \
                                     const V2<T>*, V2<T>*, const int*, int, int,         \
                                     cudaStream_t);                                      \
    template void launch_prolong_add<T>(const Grid&, const Grid&, const uint8_t*,        \
                                        const V2<T>*, V2<T>*, const int*, int, int,      \
                                        cudaStream_t);                                   \
    template void launch_coarse_apply<T>(const Grid&, const double*, const V2<T>*,       \
                                         V2<T>*, int, const int*, int, int,              \
                                         cudaStream_t);                                  \
    template void launch_bicg_init<T>(const Grid&, const uint8_t*, const V2<T>*, V2<T>*, \
                                      V2<T>*, V2<T>*, V2<T>*, V2<T>*, double*, KScal*,   \
                                      int, cudaStream_t);                                \
    template void launch_bicg_p<T>(const Grid&, const V2<T>*, const V2<T>*, V2<T>*,      \
                                   const KScal*, int, cudaStream_t);                     \
    template void launch_bicg_s<T>(const Grid&, const V2<T>*, const V2<T>*, V2<T>*,      \
                                   double*, const KScal*, int, cudaStream_t);            \
    template void launch_bicg_xr<T>(const Grid&, const V2<T>*, const V2<T>*,             \
                                    const V2<T>*, const V2<T>*, const V2<T>*, V2<T>*,    \
                                    V2<T>*, double*, const KScal*, int, cudaStream_t);   \
    template void launch_newton_rhs<T>(const Grid&, const V2<double>*, V2<T>*,           \
                                       const NScal*, int, cudaStream_t);                 \
    template void launch_newton_trial<T>(const Grid&, const double*, const double*,      \
                                         const V2<T>*, double*, double*, double*,        \
                                         const NScal*, int, cudaStream_t);               \
    template void launch_axpy_mask<T>(const Grid&, const uint8_t*, const V2<T>*, V2<T>*, \
                                      double, int, int, cudaStream_t);                   \
    template void launch_bicg_keep<T>(const Grid&, V2<T>*, V2<T>*, const KScal*, int,    \
                                      int, cudaStream_t);                                \
    template void launch_smooth_zline<T, typename MgType<T>::type>(                      \
        const Grid&, const B4<typename MgType<T>::type>*, const B4<T>*, const uint8_t*,  \
        const V2<T>*, const V2<T>*, V2<T>*, double, int, const int*, int, int,           \
        cudaStream_t, int);
ELDER_INST(double)
ELDER_INST(float)
#undef ELDER_INST
// (line blocks stored with the multigrid matrix, or in FP32 beside the
// matrix-free finest level of the mixed solver)
#define ELDER_INST_ZLINE(T, M)                                                              \
    template void launch_zline_factor<T, M>(const Grid&, const B4<M>*, const B4<M>*, size_t, \
                                            const B4<T>*, const uint8_t*, B4<T>*, B4<T>*,    \
                                            B4<T>*, const int*, int, int, cudaStream_t);
ELDER_INST_ZLINE(double, double)
ELDER_INST_ZLINE(float, __nv_bfloat16)
ELDER_INST_ZLINE(float, float)
#undef ELDER_INST_ZLINE
template void launch_zline_apply<double>(const Grid&, const B4<double>*, const B4<double>*,
                                         const B4<double>*, const uint8_t*, const V2<double>*,
                                         const V2<double>*, V2<double>*, double, const int*, int,
                                         int, cudaStream_t, int, int);
template void launch_zline_apply<float>(const Grid&, const B4<float>*, const B4<float>*,
                                        const B4<float>*, const uint8_t*, const V2<float>*,
                                        const V2<float>*, V2<float>*, double, const int*, int,
                                        int, cudaStream_t, int, int);
template void launch_convert<double, float>(const V2<double>*, V2<float>*, size_t, cudaStream_t);
template void launch_convert<float, double>(const V2<float>*, V2<double>*, size_t, cudaStream_t);
template void launch_convert<double, double>(const V2<double>*, V2<double>*, size_t, cudaStream_t);

}  // namespace elder
