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
// registers (as values and as (3,1)-weighted sums, so that each row's in-plane
// sums are formed once), the next row's corners come from a shared-memory row
// of float4 (p', c, x_p, x_c).  The contributions of a cell to the three
// corners owned by other threads cross through shared memory.  Both
// exchanges are double-buffered, so a row costs one __syncthreads.  The box
// is flat (nz is the short direction), so a tile holds whole z columns on most
// grids and only its x sides (and the ends of a y chunk) are computed twice.
#include <algorithm>

#include "kernels.h"

namespace elder {

namespace {

constexpr int kMfThreads = 512;   // largest CTA
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

// (3,1) sums of a pair: (a, b) -> (3 a + b, a + 3 b)
__device__ __forceinline__ void pass31(float& a, float& b)
{
    const float t = a + b;
    a = fmaf(2.0f, a, t);
    b = fmaf(2.0f, b, t);
}

// The four corners (x + 2 z) of one row of a cell column and the row's
// in-plane sums: gx[z], gz[x] the (3,1) sums of the x and z differences of p',
// dx, dz those of x_p; C, V the (3,1) x (3,1) sums of c and x_c.
struct MfRow {
    float p[4], c[4], u[4], v[4];
    float gx[2], gz[2], dx[2], dz[2];
    float C[4], V[4];
};

__device__ __forceinline__ void row_set(MfRow& r, const float4& a, const float4& b,
                                        const float4& d, const float4& e)
{
    r.p[0] = a.x; r.p[1] = b.x; r.p[2] = d.x; r.p[3] = e.x;
    r.c[0] = a.y; r.c[1] = b.y; r.c[2] = d.y; r.c[3] = e.y;
    r.u[0] = a.z; r.u[1] = b.z; r.u[2] = d.z; r.u[3] = e.z;
    r.v[0] = a.w; r.v[1] = b.w; r.v[2] = d.w; r.v[3] = e.w;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        r.gx[q] = r.p[2 * q + 1] - r.p[2 * q];
        r.dx[q] = r.u[2 * q + 1] - r.u[2 * q];
        r.gz[q] = r.p[q + 2] - r.p[q];
        r.dz[q] = r.u[q + 2] - r.u[q];
    }
    pass31(r.gx[0], r.gx[1]);
    pass31(r.dx[0], r.dx[1]);
    pass31(r.gz[0], r.gz[1]);
    pass31(r.dz[0], r.dz[1]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        r.C[q] = r.c[q];
        r.V[q] = r.v[q];
    }
    pass31(r.C[0], r.C[1]); pass31(r.C[2], r.C[3]);
    pass31(r.C[0], r.C[2]); pass31(r.C[1], r.C[3]);
    pass31(r.V[0], r.V[1]); pass31(r.V[2], r.V[3]);
    pass31(r.V[0], r.V[2]); pass31(r.V[1], r.V[3]);
}

// Derivative (dm, dF) of one quarter face from its end A to B: g, d the
// weighted differences of p' and x_p; zA, zB and wA, wB the cell sums of c and
// x_c at the ends; cA.. the end values; kA, dA the cell's coefficients.
template <bool VERT>
__device__ __forceinline__ void face(const MfConst& k, float kA, float dA, float g, float d,
                                     float zA, float zB, float wA, float wB, float cA, float cB,
                                     float vA, float vB, float& dm, float& dF)
{
    const float zs = zA + zB, ws = wA + wB;
    const float rho = fmaf(k.drho128, zs, k.rho0);
    const float drho = k.drho128 * ws;
    const float t = kA * (VERT ? fmaf(k.gz, zs, g) : g);
    const float s = kA * (VERT ? fmaf(k.gz, ws, d) : d);
    const float m = rho * t;
    dm = fmaf(rho, s, drho * t);
    const bool up = m >= 0.0f;
    const float cu = up ? cA : cB, vu = up ? vA : vB;
    const float w = fmaf(drho, zB - zA, rho * (wB - wA));
    dF = fmaf(cu, dm, fmaf(vu, m, dA * w));
}

// One cell between the rows lo (y = j) and hi (y = j + 1): adds the face
// derivatives to the corner sums al (row lo) and sets ah (row hi).
__device__ __forceinline__ void cell_apply(const MfConst& k, float phi, float km, const MfRow& lo,
                                           const MfRow& hi, float2 (&al)[4], float2 (&ah)[4])
{
    // cell sums of c and x_c: the (3,1) pass along y
    float Zl[4], Zh[4], Wl[4], Wh[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        Zl[q] = lo.C[q]; Zh[q] = hi.C[q];
        pass31(Zl[q], Zh[q]);
        Wl[q] = lo.V[q]; Wh[q] = hi.V[q];
        pass31(Wl[q], Wh[q]);
    }
    // y faces: one per (x, z) corner, from row lo to row hi
    {
        float g[4], d[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            g[q] = hi.p[q] - lo.p[q];
            d[q] = hi.u[q] - lo.u[q];
        }
        pass31(g[0], g[1]); pass31(g[2], g[3]); pass31(g[0], g[2]); pass31(g[1], g[3]);
        pass31(d[0], d[1]); pass31(d[2], d[3]); pass31(d[0], d[2]); pass31(d[1], d[3]);
        const float kA = km * k.kA[1], dA = phi * k.dA[1];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float dm, dF;
            face<false>(k, kA, dA, g[q], d[q], Zl[q], Zh[q], Wl[q], Wh[q], lo.c[q], hi.c[q],
                        lo.v[q], hi.v[q], dm, dF);
            al[q].x += dm;
            al[q].y += dF;
            ah[q].x = -dm;
            ah[q].y = -dF;
        }
    }
    // x faces (edge at (y, z)): corners 2 z and 2 z + 1 of a row
    {
        const float kA = km * k.kA[0], dA = phi * k.dA[0];
#pragma unroll
        for (int z = 0; z < 2; ++z) {
            float gl = lo.gx[z], gh = hi.gx[z], dl = lo.dx[z], dh = hi.dx[z];
            pass31(gl, gh);
            pass31(dl, dh);
            const int A = 2 * z, B = 2 * z + 1;
            float dm, dF;
            face<false>(k, kA, dA, gl, dl, Zl[A], Zl[B], Wl[A], Wl[B], lo.c[A], lo.c[B], lo.v[A],
                        lo.v[B], dm, dF);
            al[A].x += dm; al[A].y += dF; al[B].x -= dm; al[B].y -= dF;
            face<false>(k, kA, dA, gh, dh, Zh[A], Zh[B], Wh[A], Wh[B], hi.c[A], hi.c[B], hi.v[A],
                        hi.v[B], dm, dF);
            ah[A].x += dm; ah[A].y += dF; ah[B].x -= dm; ah[B].y -= dF;
        }
    }
    // z faces (edge at (x, y)): corners x and x + 2 of a row
    {
        const float kA = km * k.kA[2], dA = phi * k.dA[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            float gl = lo.gz[x], gh = hi.gz[x], dl = lo.dz[x], dh = hi.dz[x];
            pass31(gl, gh);
            pass31(dl, dh);
            const int A = x, B = x + 2;
            float dm, dF;
            face<true>(k, kA, dA, gl, dl, Zl[A], Zl[B], Wl[A], Wl[B], lo.c[A], lo.c[B], lo.v[A],
                       lo.v[B], dm, dF);
            al[A].x += dm; al[A].y += dF; al[B].x -= dm; al[B].y -= dF;
            face<true>(k, kA, dA, gh, dh, Zh[A], Zh[B], Wh[A], Wh[B], hi.c[A], hi.c[B], hi.v[A],
                       hi.v[B], dm, dF);
            ah[A].x += dm; ah[A].y += dF; ah[B].x -= dm; ah[B].y -= dF;
        }
    }
}

// MODE 0: y = A x; 1: also partial[0] = (a, y); 2: partial[0] = (y, a),
// partial[1] = (y, y) (partial [S][2][gridDim.x]); 3: y = a - A x.  Dirichlet
// components of y are 0.
template <int MODE>
__global__ void __launch_bounds__(kMfThreads)
    k_mf_apply(Grid G, MfConst k, MfTiling t, const uint8_t* __restrict__ bc,
               const V2<float>* __restrict__ cellT, const V2<float>* __restrict__ nodeT,
               const V2<float>* __restrict__ x, V2<float>* __restrict__ y,
               const V2<float>* __restrict__ a, double* __restrict__ partial,
               const float* __restrict__ vs, const int* mask, int mstride)
{
    __shared__ float4 nd[2][kMfThreads];
    __shared__ float2 ct[2][3][kMfThreads];
    __shared__ float ph[2][kMfThreads];
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
    const bool hasx = tx > 0, hasz = tz > 0;
    const size_t on = (size_t)s * G.N;
    const int n0 = in ? gx + pl * gz : 0;             // node of row 0
    const int e0 = cell ? gx + G.nx * G.ny * gz : 0;  // cell of row 0
    const V2<float>* ns = nodeT + on + n0;
    const V2<float>* xv = x + on + n0;
    const V2<float>* cs = cellT + (size_t)s * G.C + e0;
    const int js = max(j0 - 1, 0), je = min(j1 - 1, G.ny - 1);  // layers of cells
    auto load = [&](int j) {
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in) {
            const V2<float> st = ns[nx1 * j], w = xv[nx1 * j];
            q = make_float4(st.p, st.c, w.p, w.c);
        }
        return q;
    };
    const int R = tid + (cell ? 1 : 0), U = tid + (cell ? wx : 0),
              D = tid + (cell ? wx + 1 : 0);
    double d0 = 0.0, d1 = 0.0;
    float4 own = load(js), nxt = load(js + 1);
    nd[js & 1][tid] = own;
    nd[(js + 1) & 1][tid] = nxt;
    V2<float> co{0.f, 0.f};
    if (cell) co = cs[G.nx * js];
    __syncthreads();
    MfRow r0, r1;
    row_set(r0, own, nd[js & 1][R], nd[js & 1][U], nd[js & 1][D]);
    __syncthreads();  // the first layer overwrites row js
    float2 al[4], ah[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) al[q] = make_float2(0.f, 0.f);
    float phl = 0.f;  // phi of the cell behind the row
    // row j's sums gathered from the cells around it and written
    auto emit = [&](int j, const float2& mine, float cn, float vn) {
        const int b = j & 1;
        float yp = mine.x, yc = mine.y, phs = ph[b][tid];
        if (hasx) {
            const float2 w = ct[b][0][tid - 1];
            yp += w.x; yc += w.y;
            phs += ph[b][tid - 1];
        }
        if (hasz) {
            const float2 w = ct[b][1][tid - wx];
            yp += w.x; yc += w.y;
            phs += ph[b][tid - wx];
        }
        if (hasx && hasz) {
            const float2 w = ct[b][2][tid - wx - 1];
            yp += w.x; yc += w.y;
            phs += ph[b][tid - wx - 1];
        }
        if (!out) return;
        const int n = n0 + nx1 * j;
        const float vd = phs * vscale * vn;
        yp = fmaf(vd, k.drho, yp);
        yc = fmaf(vd, fmaf(k.drho2, cn, k.rho0), yc);
        V2<float> av{0.f, 0.f};
        if (MODE != 0) av = a[on + n];
        if (MODE == 3) { yp = av.p - yp; yc = av.c - yc; }
        const uint8_t m = bc[n];
        if (m & BC_P) yp = 0.f;
        if (m & BC_C) yc = 0.f;
        y[on + n] = V2<float>{yp, yc};
        if (MODE == 1 || MODE == 2) d0 += dot2(av.p, av.c, yp, yc);
        if (MODE == 2) d1 += dot2(yp, yc, yp, yc);
    };
    // one layer: cells between row j (state lo) and row j + 1 (state hi)
    auto layer = [&](int j, MfRow& lo, MfRow& hi) {
        // the row after next and the next layer's coefficients, used after
        // this layer's arithmetic
        float4 nn = nxt;
        V2<float> cn{0.f, 0.f};
        if (j < je) {
            nn = load(j + 2);
            if (cell) cn = cs[G.nx * (j + 1)];
        }
        const int b = j & 1, h = (j + 1) & 1;
        row_set(hi, nxt, nd[h][R], nd[h][U], nd[h][D]);
        cell_apply(k, co.p, co.c, lo, hi, al, ah);
        if (!cell) {
#pragma unroll
            for (int q = 0; q < 4; ++q) ah[q] = al[q] = make_float2(0.f, 0.f);
        }
        ct[b][0][tid] = al[1];
        ct[b][1][tid] = al[2];
        ct[b][2][tid] = al[3];
        ph[b][tid] = phl + co.p;
        nd[b][tid] = nn;  // row j was read as the previous layer's far row
        __syncthreads();
        if (j >= j0) emit(j, al[0], lo.c[0], lo.v[0]);
#pragma unroll
        for (int q = 0; q < 4; ++q) al[q] = ah[q];
        phl = co.p;
        co = cn;
        nxt = nn;
    };
    int j = js;
    for (; j + 1 <= je; j += 2) {
        layer(j, r0, r1);
        layer(j + 1, r1, r0);
    }
    if (j <= je) {
        layer(j, r0, r1);
        r0.c[0] = r1.c[0];
        r0.v[0] = r1.v[0];
    }
    if (j1 == G.ny + 1) {  // the last row of nodes has cells behind it only
        const int b = G.ny & 1;
        ct[b][0][tid] = al[1];
        ct[b][1][tid] = al[2];
        ct[b][2][tid] = al[3];
        ph[b][tid] = phl;
        __syncthreads();
        emit(G.ny, al[0], r0.c[0], r0.v[0]);
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
    // launch's time goes with its waves times the layers of a chunk
    const int slots = 152 * std::max(1, kMfResident / best.threads);
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
