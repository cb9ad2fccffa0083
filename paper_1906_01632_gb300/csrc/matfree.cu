// matfree.cu -- products with the finest level's Jacobian in FP32 without the
// stored matrix.
//
// y = J x of the implicit step's linearisation at (p, c) is formed from the
// state, the cell coefficients and x: per cell the derivative of its 12
// quarter-face fluxes in the direction x, summed onto the cell's corners, plus
// the lumped storage term.  With the notation of k_jacobian (p' = p - rho0 g
// (Lz - z)) a face of direction D has
//   rho = rho0 + drho c_ip,  G = grad p'.e_D + [D=z] g drho c_ip,
//   m = -rho (K/mu) A G,
//   dm = -(K/mu) A (rho dG + drho dc_ip G),  dG = grad x_p.e_D + [D=z] g drho dc_ip,
//   dF = c_up dm + x_c,up m - phi Dm A (drho dc_ip grad c.e_D + rho grad x_c.e_D),
// d the directional derivative, the same as a product with the rows that
// k_jacobian assembles.
//
// What bounds it: FP32 issue.  The assembled product reads 432 B of matrix per
// node (FP32 Krylov operator; 216 B for the bfloat16 multigrid copy) and runs
// at the copy bandwidth; this form reads 8 B of state, 8 B of coefficients and
// the vectors, and issues about 450 FP32 instructions per cell.  The assembly
// then writes the three blocks of a node's vertical line only.  Steps against
// the stored matrix: 64x64x16 x 256: 210 -> 171 ms; 128x128x32 x 24 (dt = 0.005 yr):
// 74 -> 61 ms; 256x256x64 x 2: 233 -> 143 ms; 128x128x32: 22.3 -> 18.7 ms.
//
// Layout: a CTA owns a tile of (x, z) columns and marches along y.  A thread
// holds one cell column: the four corners of the row behind it stay in
// registers, the next row's come from a shared-memory row of (p', x_p, c, x_c).
// Rows, coefficients and the second operand arrive by asynchronous copies two
// layers' arithmetic ahead: with the loads one layer ahead in registers (and
// with 4 to 16 of them spilled) the warps waited for memory 2.4 of 7 cycles per
// instruction.  A quantity of the state and the same one of x share the packed
// FP32 instructions.  The contributions of a cell to the three corners owned by
// other threads cross through shared memory, double-buffered, so a row costs
// one __syncthreads.  The box is flat (nz is the short direction), so a tile
// holds whole z columns on most grids and only its x sides (and the ends of a
// y chunk) are computed twice.  256 threads of 128 registers, two CTAs per SM;
// three or four smaller CTAs of fewer registers spill and are slower (518 to
// 811 us).  64x64x16 x 256, the three kinds of product: 657, 684, 595 us with one
// value per instruction and register prefetch, 441, 477, 414 us now, 62 % of the
// issue slots, the FMA pipe throttling.
#include <algorithm>

#include "kernels.h"

namespace elder {

namespace {

constexpr int kMfThreads = 256;   // largest CTA
constexpr int kMfResident = 512;  // threads an SM holds (128 registers each)

// Tiling of a launch: ntx x ntz tiles of ox x oz output columns, nch chunks of
// oy output rows.
struct MfTiling {
    int ox, oz, oy, ntx, ntz, nch, threads;
};

// Constants of the face derivatives, formed on the host in FP64.  The (3,1)
// sums carry 16 (differences of p', x_p), 32 (differences of c, x_c) and 128
// (edge sums of c, x_c) times the Q1 weights.
struct MfConst {
    float kA[3];    // -A_d / (16 h_d)
    float dA[3];    // -Dm A_d / (32 h_d)
    float gz;       // 16 h_z g drho / 128
    float drho128;  // drho / 128
    float rho0, drho, drho2;
};

// Asynchronous copy of one word to shared memory (0 where `on` is false).
__device__ __forceinline__ void copy_word(float* dst, const float* src, bool on)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                     static_cast<unsigned>(__cvta_generic_to_shared(dst))),
                 "l"(src), "r"(on ? 4 : 0)
                 : "memory");
}

__device__ __forceinline__ void copy_pair(V2<float>* dst, const V2<float>* src, bool on)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(
                     static_cast<unsigned>(__cvta_generic_to_shared(dst))),
                 "l"(src), "r"(on ? 8 : 0)
                 : "memory");
}

__device__ __forceinline__ void copies_commit()
{
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// All but the newest group of copies have arrived.
__device__ __forceinline__ void copies_wait()
{
    asm volatile("cp.async.wait_group 1;" ::: "memory");
}

// Two FP32 operations per instruction (the packed forms of sm_103a): a pair
// holds a quantity of the state and the same one of x, whose sums and
// differences are formed alike.
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);
}

// (3,1) sums of two pairs: (a, b) -> (3 a + b, a + 3 b)
__device__ __forceinline__ void pass31(float2& a, float2& b)
{
    const float2 two = make_float2(2.0f, 2.0f), t = __fadd2_rn(a, b);
    a = __ffma2_rn(two, a, t);
    b = __ffma2_rn(two, b, t);
}

__device__ __forceinline__ void plane31(float2 (&q)[4])
{
    pass31(q[0], q[1]);
    pass31(q[2], q[3]);
    pass31(q[0], q[2]);
    pass31(q[1], q[3]);
}

// The four corners (x + 2 z) of one row of a cell column, p = (p', x_p) and c =
// (c, x_c).
struct MfRow {
    float2 p[4], c[4];
};

__device__ __forceinline__ void row_set(MfRow& r, const float4& a, const float4& b,
                                        const float4& d, const float4& e)
{
    r.p[0] = make_float2(a.x, a.y); r.c[0] = make_float2(a.z, a.w);
    r.p[1] = make_float2(b.x, b.y); r.c[1] = make_float2(b.z, b.w);
    r.p[2] = make_float2(d.x, d.y); r.c[2] = make_float2(d.z, d.w);
    r.p[3] = make_float2(e.x, e.y); r.c[3] = make_float2(e.z, e.w);
}

// Derivative (dm, dF) of one quarter face from its end A to B: g the weighted
// differences of p; zA, zB the cell sums of c at the ends; cA, cB the end
// values; kA, dA the cell's coefficients.
template <bool VERT>
__device__ __forceinline__ float2 face(const MfConst& k, float kA, float dA, float2 g, float2 zA,
                                       float2 zB, float2 cA, float2 cB)
{
    const float2 z = __fadd2_rn(zA, zB), dz = sub2(zB, zA);
    // (rho, its derivative) and (-(K/mu) A G, its derivative)
    const float2 rho = __ffma2_rn(make_float2(k.drho128, k.drho128), z, make_float2(k.rho0, 0.f));
    if (VERT) g = __ffma2_rn(make_float2(k.gz, k.gz), z, g);
    const float2 t = __fmul2_rn(make_float2(kA, kA), g);
    const float m = rho.x * t.x;
    const float dm = fmaf(rho.x, t.y, rho.y * t.x);
    const bool up = m >= 0.0f;
    const float cu = up ? cA.x : cB.x, vu = up ? cA.y : cB.y;
    const float w = fmaf(rho.y, dz.x, rho.x * dz.y);
    return make_float2(dm, fmaf(cu, dm, fmaf(vu, m, dA * w)));
}

// One cell between the rows lo (y = j) and hi (y = j + 1): adds the face
// derivatives to the corner sums al (row lo) and sets ah (row hi).
__device__ __forceinline__ void cell_apply(const MfConst& k, float phi, float km, const MfRow& lo,
                                           const MfRow& hi, float2 (&al)[4], float2 (&ah)[4])
{
    // y faces: one per (x, z) corner, from row lo to row hi
    float2 g[4], Zl[4], Zh[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        g[q] = sub2(hi.p[q], lo.p[q]);
        // cell sums of c: the (3,1) pass along y
        Zl[q] = lo.c[q];
        Zh[q] = hi.c[q];
        pass31(Zl[q], Zh[q]);
    }
    plane31(g);
    plane31(Zl); plane31(Zh);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 f = face<false>(k, km * k.kA[1], phi * k.dA[1], g[q], Zl[q], Zh[q], lo.c[q],
                                     hi.c[q]);
        al[q] = __fadd2_rn(al[q], f);
        ah[q] = make_float2(-f.x, -f.y);
    }
    float2 gx[4], gz[4];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        gx[q] = sub2(lo.p[2 * q + 1], lo.p[2 * q]);
        gz[q] = sub2(lo.p[q + 2], lo.p[q]);
        gx[q + 2] = sub2(hi.p[2 * q + 1], hi.p[2 * q]);
        gz[q + 2] = sub2(hi.p[q + 2], hi.p[q]);
    }
    plane31(gx);
    plane31(gz);
    // x faces (edge at (y, z)): corners 2 z and 2 z + 1 of a row
#pragma unroll
    for (int z = 0; z < 2; ++z) {
        const float kA = km * k.kA[0], dA = phi * k.dA[0];
        float2 gl = gx[z], gh = gx[z + 2];
        const int A = 2 * z, B = 2 * z + 1;
        const float2 f = face<false>(k, kA, dA, gl, Zl[A], Zl[B], lo.c[A], lo.c[B]);
        al[A] = __fadd2_rn(al[A], f);
        al[B] = sub2(al[B], f);
        const float2 h = face<false>(k, kA, dA, gh, Zh[A], Zh[B], hi.c[A], hi.c[B]);
        ah[A] = __fadd2_rn(ah[A], h);
        ah[B] = sub2(ah[B], h);
    }
    // z faces (edge at (x, y)): corners x and x + 2 of a row
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const float kA = km * k.kA[2], dA = phi * k.dA[2];
        float2 gl = gz[x], gh = gz[x + 2];
        const int A = x, B = x + 2;
        const float2 f = face<true>(k, kA, dA, gl, Zl[A], Zl[B], lo.c[A], lo.c[B]);
        al[A] = __fadd2_rn(al[A], f);
        al[B] = sub2(al[B], f);
        const float2 h = face<true>(k, kA, dA, gh, Zh[A], Zh[B], hi.c[A], hi.c[B]);
        ah[A] = __fadd2_rn(ah[A], h);
        ah[B] = sub2(ah[B], h);
    }
}

// MODE 0: y = A x; 1: also partial[0] = (a, y); 2: partial[0] = (y, a),
// partial[1] = (y, y) (partial [S][2][gridDim.x]); 3: y = a - A x.  Dirichlet
// components of y are 0.
template <int MODE>
__global__ void __launch_bounds__(kMfThreads, kMfResident / kMfThreads)
    k_mf_apply(Grid G, MfConst k, MfTiling t, const uint8_t* __restrict__ bc,
               const V2<float>* __restrict__ cellT, const V2<float>* __restrict__ nodeT,
               const V2<float>* __restrict__ x, V2<float>* __restrict__ y,
               const V2<float>* __restrict__ a, double* __restrict__ partial,
               const float* __restrict__ vs, const int* mask, int mstride)
{
    // the next row's (p', x_p, c, x_c); what a thread's cells add to the
    // corners of others: (1, 0) and (0, 1) in ca, (1, 1) in cb, the cells' phi in
    // cp; entry kMfThreads stays zero (a side without cells)
    __shared__ float4 nd[4][kMfThreads], ca[2][kMfThreads + 1];
    __shared__ float2 cb[2][kMfThreads + 1];
    __shared__ float cp[2][kMfThreads + 1];
    __shared__ V2<float> cl[4][kMfThreads], sa[4][kMfThreads];
    __shared__ double red[32];
    const int s = blockIdx.y;
    if (mask != nullptr && mask[(size_t)s * mstride] == 0) return;
    const float vscale = __ldg(vs);
    const int nx1 = G.nx + 1, pl = nx1 * (G.ny + 1);
    // the tile: output columns [x0, x1) x [z0, z1), threads on the columns
    // whose cells touch them
    const int bx = blockIdx.x % t.ntx, br = blockIdx.x / t.ntx;
    const int bz = br % t.ntz, bch = br / t.ntz;
    const int x0 = bx * t.ox, x1 = min(x0 + t.ox, nx1);
    const int z0 = bz * t.oz, z1 = min(z0 + t.oz, G.nz + 1);
    const int j0 = bch * t.oy, j1 = min(j0 + t.oy, G.ny + 1);
    const int xs = max(x0 - 1, 0), zs = max(z0 - 1, 0);
    const int wx = min(x1, G.nx) - xs + 1, wz = min(z1, G.nz) - zs + 1;
    const int tid = threadIdx.x;
    const int tz = tid / wx, tx = tid - tz * wx;
    const bool in = tz < wz;
    const int gx = xs + tx, gz = zs + tz;
    const bool cell = in && tx < wx - 1 && tz < wz - 1;
    const bool out = in && gx >= x0 && gx < x1 && gz >= z0 && gz < z1;
    // node and cell of row 0 (32-bit offsets: registers decide the occupancy
    // here; a batch of 2^32 nodes would not fit the device)
    const unsigned n0 = (unsigned)s * (unsigned)G.N + (in ? gx + pl * gz : 0);
    const unsigned e0 = (unsigned)s * (unsigned)G.C + (cell ? gx + G.nx * G.ny * gz : 0);
    const int js = max(j0 - 1, 0), je = min(j1 - 1, G.ny - 1);  // layers of cells
    // row j of the nodes, the coefficients of layer j - 1 and a's row j - 1 into
    // their buffers, one group per row (empty past the last); the nodes word
    // by word, into the order of the pairs
    auto copy_row = [&](int j) {
        const int b = j & 3;
        if (j <= je + 1) {
            float* d = &nd[b][tid].x;
            const V2<float>*st = nodeT + (n0 + nx1 * j), *w = x + (n0 + nx1 * j);
            copy_word(d, &st->p, in);
            copy_word(d + 1, &w->p, in);
            copy_word(d + 2, &st->c, in);
            copy_word(d + 3, &w->c, in);
        }
        if (j > js && j <= je + 1)
            copy_pair(&cl[b][tid], cellT + (e0 + G.nx * (j - 1)), cell);
        if (MODE != 0 && j > js && j <= j1)
            copy_pair(&sa[b][tid], a + (n0 + nx1 * (j - 1)), out);
        copies_commit();
    };
    // neighbours: the cell's corners ahead, the cells' sides behind
    const int R = tid + (cell ? 1 : 0), U = tid + (cell ? wx : 0),
              D = tid + (cell ? wx + 1 : 0);
    const int bX = tx > 0 ? tid - 1 : kMfThreads, bZ = tz > 0 ? tid - wx : kMfThreads,
              bD = tx > 0 && tz > 0 ? tid - wx - 1 : kMfThreads;
    double d0 = 0.0, d1 = 0.0;
    if (tid < 2) {
        ca[tid][kMfThreads] = make_float4(0.f, 0.f, 0.f, 0.f);
        cb[tid][kMfThreads] = make_float2(0.f, 0.f);
        cp[tid][kMfThreads] = 0.f;
    }
    copy_row(js);
    copy_row(js + 1);
    copy_row(js + 2);
    copies_wait();  // rows js and js + 1
    __syncthreads();
    MfRow r0, r1;
    row_set(r0, nd[js & 3][tid], nd[js & 3][R], nd[js & 3][U], nd[js & 3][D]);
    float2 al[4], ah[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) al[q] = make_float2(0.f, 0.f);
    float phl = 0.f;  // phi of the cell behind the row
    auto share = [&](int b, float phs) {
        ca[b][tid] = make_float4(al[1].x, al[1].y, al[2].x, al[2].y);
        cb[b][tid] = al[3];
        cp[b][tid] = phs;
    };
    // row j's sums gathered from the cells around it and written
    auto emit = [&](int j, float phs, float2 c, int mk) {
        const int b = j & 1;
        const float2 w0 = *reinterpret_cast<const float2*>(&ca[b][bX].x);
        const float2 w1 = *reinterpret_cast<const float2*>(&ca[b][bZ].z);
        const float2 w2 = cb[b][bD];
        float yp = (al[0].x + w0.x) + (w1.x + w2.x), yc = (al[0].y + w0.y) + (w1.y + w2.y);
        phs = (phs + cp[b][bX]) + (cp[b][bZ] + cp[b][bD]);
        if (!out) return;
        const float vd = phs * vscale * c.y;
        V2<float> av{0.f, 0.f};
        if (MODE != 0) av = sa[(j + 1) & 3][tid];
        yp = fmaf(vd, k.drho, yp);
        yc = fmaf(vd, fmaf(k.drho2, c.x, k.rho0), yc);
        if (MODE == 3) { yp = av.p - yp; yc = av.c - yc; }
        if (mk & BC_P) yp = 0.f;
        if (mk & BC_C) yc = 0.f;
        y[n0 + nx1 * j] = V2<float>{yp, yc};
        if (MODE == 1 || MODE == 2) d0 += dot2(av.p, av.c, yp, yc);
        if (MODE == 2) d1 += dot2(yp, yc, yp, yc);
    };
    // one layer: cells between row j (state lo) and row j + 1 (state hi)
    int mk = 0;  // the Dirichlet bits of row j
    auto layer = [&](int j, MfRow& lo, MfRow& hi) {
        // three rows ahead of the one behind: two layers' arithmetic hide the
        // copies (over row j - 1, whose last reader was the previous layer)
        copy_row(j + 3);
        if (out) mk = bc[gx + pl * gz + nx1 * j];
        const int b = j & 1, h = (j + 1) & 3;
        row_set(hi, nd[h][tid], nd[h][R], nd[h][U], nd[h][D]);
        const V2<float> co = cl[h][tid];
        cell_apply(k, co.p, co.c, lo, hi, al, ah);
        if (!cell) {
#pragma unroll
            for (int q = 0; q < 4; ++q) ah[q] = al[q] = make_float2(0.f, 0.f);
        }
        const float phs = phl + co.p;
        share(b, phs);
        copies_wait();
        __syncthreads();
        if (j >= j0) emit(j, phs, lo.c[0], mk);
#pragma unroll
        for (int q = 0; q < 4; ++q) al[q] = ah[q];
        phl = co.p;
    };
    int j = js;
    for (; j + 1 <= je; j += 2) {
        layer(j, r0, r1);
        layer(j + 1, r1, r0);
    }
    if (j <= je) {
        layer(j, r0, r1);
        r0.c[0] = r1.c[0];
    }
    if (j1 == G.ny + 1) {  // the last row of nodes has cells behind it only
        if (out) mk = bc[gx + pl * gz + nx1 * G.ny];
        share(G.ny & 1, phl);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        emit(G.ny, phl, r0.c[0], mk);
    }
    if (MODE == 1 || MODE == 2) {
        const double s0 = block_sum(d0, red);
        const double s1 = MODE == 2 ? block_sum(d1, red) : 0.0;
        if (tid == 0) {
            partial[((size_t)s * 2 + 0) * gridDim.x + blockIdx.x] = s0;
            if (MODE == 2) partial[((size_t)s * 2 + 1) * gridDim.x + blockIdx.x] = s1;
        }
    }
}

int tiles(int nodes, int out) { return (nodes + out - 1) / out; }

// Threads of the widest of nt tiles of `out` columns over `nodes`: a column
// more on each side that has a neighbouring tile.
int widest(int nodes, int out)
{
    const int nt = tiles(nodes, out);
    if (nt == 1) return nodes;
    if (nt == 2) return out + 1;
    return out + 2;
}

MfTiling choose_tiling(const Grid& G, int S)
{
    const int nx1 = G.nx + 1, ny1 = G.ny + 1, nz1 = G.nz + 1;
    MfTiling best{};
    double least = 1e300;
    for (int oz = nz1; oz >= 1; --oz) {
        if (oz < nz1 && tiles(nz1, oz) == tiles(nz1, oz + 1)) continue;
        const int ezs = (nz1 + tiles(nz1, oz) - 1) / tiles(nz1, oz);  // even shares
        for (int ntx = 1; ntx <= nx1; ++ntx) {
            const int ox = (nx1 + ntx - 1) / ntx;
            const int w = widest(nx1, ox) * widest(nz1, ezs);
            if (w > kMfThreads) continue;
            const int thr = (w + 31) / 32 * 32;
            const int res = std::max(1, kMfResident / thr);
            // thread slots of all tiles, scaled by the share of an SM's
            // thread slots that whole CTAs fill
            double c = (double)tiles(nx1, ox) * tiles(nz1, ezs) * thr * kMfResident / (res * thr);
            if (res == 1) c *= 1.15;  // a barrier then idles the SM
            if (c < least) {
                least = c;
                best = MfTiling{ox, ezs, ny1, tiles(nx1, ox), tiles(nz1, ezs), 1, thr};
            }
            if (thr <= 64) break;
        }
    }
    // chunks of rows: each adds a layer (and a start of about one more); the
    // launch's time goes with its waves times the layers of a chunk.  They follow
    // from the batch, and with them which rows a partial of the inner products
    // adds up: the values of y do not depend on them, the last bits of the FP64
    // sums do (partials of fixed groups of rows made the mixed steps 1 to 8 %
    // slower)
    const int slots = kSMs * std::max(1, kMfResident / best.threads);
    double lt = 1e300;
    const int base = best.ntx * best.ntz * S;
    for (int nch = 1; nch <= std::max(1, ny1 / 3); ++nch) {
        const int oy = (ny1 + nch - 1) / nch;
        // (the caller's partials hold one per 32 nodes)
        if (tiles(ny1, oy) != nch || best.ntx * best.ntz * nch > nblocks(G.N, 32)) continue;
        const long long ctas = (long long)base * nch;
        // many waves even out; below about 8 the last one counts whole
        const double waves = ctas > 8LL * slots ? (double)ctas / slots + 0.5
                                                : (double)((ctas + slots - 1) / slots);
        const double tt = waves * (oy + 2.5);
        if (tt < lt * 0.999) {
            lt = tt;
            best.oy = oy;
            best.nch = nch;
        }
    }
    return best;
}

// The tiling of a launch; the search runs once per grid and batch size in turn.
MfTiling mf_tiling(const Grid& G, int S)
{
    struct Last {
        int nx = 0, ny = 0, nz = 0, S = 0;
        MfTiling t{};
    };
    static thread_local Last last;
    if (last.nx != G.nx || last.ny != G.ny || last.nz != G.nz || last.S != S)
        last = Last{G.nx, G.ny, G.nz, S, choose_tiling(G, S)};
    return last.t;
}

MfConst mf_const(const Grid& G, const Phys& ph)
{
    const double h[3] = {G.hx, G.hy, G.hz};
    MfConst k;
    for (int d = 0; d < 3; ++d) {
        const double area = 0.25 * h[(d + 1) % 3] * h[(d + 2) % 3];
        k.kA[d] = (float)(-area / (16.0 * h[d]));
        k.dA[d] = (float)(-ph.Dm * area / (32.0 * h[d]));
    }
    k.gz = (float)(16.0 * G.hz * ph.g * ph.drho / 128.0);
    k.drho128 = (float)(ph.drho / 128.0);
    k.rho0 = (float)ph.rho0;
    k.drho = (float)ph.drho;
    k.drho2 = (float)(2.0 * ph.drho);
    return k;
}

}  // namespace

int mf_blocks(const Grid& G, int S)
{
    const MfTiling t = mf_tiling(G, S);
    return t.ntx * t.ntz * t.nch;
}

void launch_mf_apply(const Grid& G, const Phys& ph, const uint8_t* bc, const V2<float>* cellT,
                     const V2<float>* nodeT, const V2<float>* x, V2<float>* y, int mode,
                     const V2<float>* a, double* partial, const float* vs, const int* mask,
                     int mstride, int S, cudaStream_t st)
{
    count_launch(1);
    const MfTiling t = mf_tiling(G, S);
    const dim3 grid(t.ntx * t.ntz * t.nch, S);
    const MfConst k = mf_const(G, ph);
#define ELDER_MF(MO)                                                                        \
    k_mf_apply<MO><<<grid, t.threads, 0, st>>>(G, k, t, bc, cellT, nodeT, x, y, a, partial, \
                                               vs, mask, mstride)
    if (mode == 0) ELDER_MF(0);
    else if (mode == 1) ELDER_MF(1);
    else if (mode == 2) ELDER_MF(2);
    else ELDER_MF(3);
#undef ELDER_MF
}

}  // namespace elder
