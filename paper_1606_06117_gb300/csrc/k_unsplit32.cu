// k_unsplit32.cu -- fused unsplit CIR / FEC / BEC step, FP32, 3D, any size and
// alignment.
//
// The stages are those of k_unsplit.cu (L_U[Phi]; Phi_bar and the correction;
// L_U[Psi]), on a 32 x 16 column tile that marches along z, each stage one
// plane behind the one before and one cell narrower, and the same roundings.
// That kernel stages rows with 16-byte copies, which need rows of whole
// 16-byte chunks, and rebuilds each cell's position, Courant numbers and
// weights in every stage.  Here a thread owns the same two cells in every stage
// and on every plane (two of the tile, rows 8 apart, or two of the halo rings):
//  - velocities come straight from global memory, one plane ahead, so they need
//    neither shared memory nor alignment; Phi is staged element by element from
//    offsets computed once per tile, periodic wrap included;
//  - weights and corner offsets, made once, and the cells' own columns of Phi,
//    L_U[Phi] and Psi stay in registers for the three planes the stages need, so
//    two of the eight corners need no load;
//  - the plane loop is unrolled by three, so that these histories change roles
//    without moves and the L_U[Phi] and Psi planes sit at fixed addresses.
// Rows are 41 floats, odd, so that the rings' columns fall on distinct banks.
// CTAs take equal shares of the (column tile, plane) pairs however few.
//
// What bounds it: one CTA of 12 warps per SM reaches 93 % of what two reach
// (BEC, 256^3: 265 and 245 us), at 50 % issue activity and 44 % of the
// shared-memory pipe, each plane's three stages separated by barriers.
// Measured (CUDA events, us per step, k_unsplit.cu -> here):
//   rows of no 16-byte multiple, 187 x 150 x 131: CIR 88 -> 24, FEC 132 -> 41,
//   BEC 188 -> 56; 65 x 40 x 30: CIR 39.9 -> 4.8, BEC 33.7 -> 10.6;
//   whole chunks: 64^3 FEC 18.4 -> 8.5, BEC 14.0 -> 12.7, 188 x 150 x 131 BEC
//   60.5 -> 56.2; but 192^3 FEC 65 -> 82, BEC 102 -> 111, so larger grids of whole
//   chunks keep k_unsplit.cu (unsplit32_serves).
#include <type_traits>

#include "sl_internal.h"

namespace sl {
namespace {

constexpr int TX = 32, TY = 16, PW = 41;

// ring h of the tile (the cells that widening it from h - 1 to h adds) as a
// list: top row, bottom row, then the two sides in turn
constexpr int ring_size(int h) { return (TX + 2 * h) * (TY + 2 * h) - (TX + 2 * h - 2) * (TY + 2 * h - 2); }
__device__ __forceinline__ void ring_cell(int h, int i, int &x, int &y)
{
    const int W = TX + 2 * h;
    if (i < 2 * W) {
        x = i < W ? i - h : i - W - h;
        y = i < W ? -h : TY + h - 1;
    } else {
        i -= 2 * W;
        x = (i & 1) ? TX + h - 1 : -h;
        y = 1 - h + (i >> 1);
    }
}

__device__ __forceinline__ float lds(const char *sm, int at) { return *reinterpret_cast<const float *>(sm + at); }
__device__ __forceinline__ void sts(char *sm, int at, float v) { *reinterpret_cast<float *>(sm + at) = v; }

// Departures of a thread's two cells: W = 1 - |C| on x and y, C itself on z, and
// the byte offsets of the x and y neighbours at -sgn C (0 when C = 0), the x
// offset in the high half of a word and the y offset in the low half.
struct Dep {
    float2 wx, wy, cz;
    int off[2];
};
__device__ __forceinline__ Dep departure(const float2 (&u)[3], float sx, float sy, float sz, bool &bad)
{
    const float2 cx = make_float2(u[0].x * sx, u[0].y * sx), cy = make_float2(u[1].x * sy, u[1].y * sy);
    Dep d;
    d.cz = make_float2(u[2].x * sz, u[2].y * sz);
    bad = fabsf(cx.x) > 1.f || fabsf(cy.x) > 1.f || fabsf(d.cz.x) > 1.f || fabsf(cx.y) > 1.f || fabsf(cy.y) > 1.f ||
          fabsf(d.cz.y) > 1.f;
    d.wx = make_float2(1.f - fabsf(cx.x), 1.f - fabsf(cx.y));
    d.wy = make_float2(1.f - fabsf(cy.x), 1.f - fabsf(cy.y));
    d.off[0] = by_sign(cx.x, -4 * 65536, 4 * 65536, 0) | by_sign(cy.x, (-4 * PW) & 0xffff, 4 * PW, 0);
    d.off[1] = by_sign(cx.y, -4 * 65536, 4 * 65536, 0) | by_sign(cy.y, (-4 * PW) & 0xffff, 4 * PW, 0);
    return d;
}

// The three corners of a cell next to its own column in the plane at shared
// offset q: the neighbours along x, along y, and along both.
struct Corners {
    float x, y, xy;
};
__device__ __forceinline__ Corners corners(const char *sm, int ax, int ay, int axy)
{
    return Corners{lds(sm, ax), lds(sm, ay), lds(sm, axy)};
}

__device__ __forceinline__ float2 lerp2(float2 w, float2 a, float2 n)
{
    return make_float2(__fmaf_rn(w.x, __fsub_rn(a.x, n.x), n.x), __fmaf_rn(w.y, __fsub_rn(a.y, n.y), n.y));
}

// Trilinear values at the departure points of the two cells at shared offsets
// o (own plane at q0, z neighbour plane at qa (C_z > 0) or qb (C_z < 0)); v0, va
// and vb are the cells' own columns there.  S = 1 for L_U, -1 for L_{-U}.
template <int S>
__device__ __forceinline__ float2 trilinear(const char *sm, const Dep &d, const int (&o)[2], int q0, int qa, int qb,
                                            float2 v0, float2 va, float2 vb)
{
    Corners c[2], e[2];
    float2 own;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int ox = d.off[k] >> 16, oy = (int)(short)d.off[k];
        const int ax = S > 0 ? o[k] + ox : o[k] - ox, ay = S > 0 ? o[k] + oy : o[k] - oy;
        const int axy = S > 0 ? ax + oy : ax - oy;
        const float cz = k ? d.cz.y : d.cz.x;
        const int qz = by_sign(cz, qa, qb, q0);
        c[k] = corners(sm + q0, ax, ay, axy);
        e[k] = corners(sm + qz, ax, ay, axy);
        (k ? own.y : own.x) = k ? by_sign(cz, va.y, vb.y, v0.y) : by_sign(cz, va.x, vb.x, v0.x);
    }
    const float2 wz = make_float2(1.f - fabsf(d.cz.x), 1.f - fabsf(d.cz.y));
    const float2 b0 = lerp2(d.wx, v0, make_float2(c[0].x, c[1].x));
    const float2 b1 = lerp2(d.wx, make_float2(c[0].y, c[1].y), make_float2(c[0].xy, c[1].xy));
    const float2 f0 = lerp2(d.wx, own, make_float2(e[0].x, e[1].x));
    const float2 f1 = lerp2(d.wx, make_float2(e[0].y, e[1].y), make_float2(e[0].xy, e[1].xy));
    return lerp2(wz, lerp2(d.wy, b0, b1), lerp2(d.wy, f0, f1));
}

template <int NST>
struct Lay {
    static constexpr int PH = TY + 2 * NST;              // rows [-NST, TY + NST), columns [-4, TX + 5)
    static constexpr int PL = PH * PW * 4;               // bytes of a shared plane
    static constexpr int NPHI = 4;                       // Phi planes p-2, p-1, p and one ahead
    static constexpr int L0 = NPHI * PL;                 // L_U[Phi] ring (3 planes), then the Psi ring (3)
    static constexpr int P0 = L0 + (NST >= 2 ? 3 : 0) * PL;
    static constexpr int SMEM = P0 + (NST >= 3 ? 3 : 0) * PL;
    // threads: two cells each, the tile's first, then the rings'
    static constexpr int N1 = NST >= 2 ? ring_size(1) / 2 : 0, N2 = NST >= 3 ? ring_size(2) / 2 : 0;
    static constexpr int NT = (TX * TY / 2 + N1 + N2 + 31) / 32 * 32;
    static constexpr int K = (PH * PW + NT - 1) / NT;    // staged elements per thread
    static constexpr int CTAS = NST == 1 ? 3 : 2;        // per SM, by registers
};

// In-plane offsets: bytes, while those of a whole plane fit 32 bits (BIG false, planes
// of fewer than 2^30 cells), else elements (a plane holds fewer than 2^31 cells), whose
// scaling to 64-bit addresses costs a BEC step of 187 x 150 x 131 55.6 -> 58.6 us.
template <bool BIG>
__device__ __forceinline__ unsigned plane_off(int row, int col, int nx)
{
    return (BIG ? 1u : 4u) * (unsigned)(row * nx + col);
}
template <bool BIG, typename F>
__device__ __forceinline__ F *plane_at(F *plane, unsigned off)
{
    if constexpr (BIG)
        return plane + off;
    else
        return reinterpret_cast<F *>(reinterpret_cast<uintptr_t>(plane) + off);
}

template <int NST, bool BIG>
__global__ void __launch_bounds__(Lay<NST>::NT, Lay<NST>::CTAS)
k_unsplit32(const float *__restrict__ in, float *__restrict__ out, const float *__restrict__ vel, Geo g, float sx,
            float sy, float sz, int64_t fin, int64_t fout)
{
    using K = Lay<NST>;
    constexpr int PL = K::PL, NT = K::NT;
    in += (int64_t)blockIdx.y * fin;   // field of this CTA (FieldSet)
    out += (int64_t)blockIdx.y * fout;
    extern __shared__ __align__(16) char sm[];
    const int tid = threadIdx.x;
    bool bad = false;

    // this thread's cells and how many stages they take part in: rows r and
    // r + 8 of the tile (all), two cells of ring 1 (all but the last), two of
    // ring 2 (the first)
    int cx[2], cy[2], o[2], stages;
    if (tid < TX * TY / 2) {
        cx[0] = cx[1] = tid & 31;
        cy[0] = tid >> 5;
        cy[1] = cy[0] + TY / 2;
        stages = NST;
    } else {
        const int i = tid - TX * TY / 2, h = i < K::N1 ? 1 : 2;
        stages = i < K::N1 + K::N2 ? NST - h : 0;
        cx[0] = cx[1] = cy[0] = cy[1] = 0;
        if (stages)
            for (int k = 0; k < 2; ++k) ring_cell(h, h == 1 ? i + k * K::N1 : i - K::N1 + k * K::N2, cx[k], cy[k]);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) o[k] = 4 * ((cy[k] + NST) * PW + cx[k] + 4);

    // Work: with g.tz planes per item the items go round the grid; with
    // g.tz = 0 every CTA takes one equal share of the (column tile, plane) pairs,
    // numbered in each tile from a tile-dependent plane, so that the share
    // boundaries of all tiles fall on the same planes and neighbouring tiles,
    // processed at the same z, find their halo rows in L2.
    const bool shares = g.tz == 0;
    const int ntiles = g.tiles_x * g.tiles_y;
    const int64_t total = (int64_t)ntiles * (shares ? g.nz : g.chunks), G = gridDim.x;
    int64_t w = shares ? total * blockIdx.x / G : blockIdx.x;
    const int64_t wend = shares ? total * (blockIdx.x + 1) / G : total;
    const double share = (double)total / (double)G;

    while (w < wend) {
        int t, z0, z1;
        if (shares) {
            t = (int)(w / g.nz);
            const int64_t tile_w = (int64_t)t * g.nz;
            const int rot = g.nz < 8 ? 0 : (int)(fmod((double)tile_w, share) + 0.5) % g.nz;   // as k_unsplit.cu
            const int64_t e = wend < tile_w + g.nz ? wend : tile_w + g.nz;
            z0 = (int)(w - tile_w) + rot;   // planes are taken modulo nz
            z1 = z0 + (int)(e - w);
            w = e;
        } else {
            t = (int)(w % ntiles);
            z0 = (int)(w / ntiles) * g.tz;
            z1 = min(z0 + g.tz, g.nz);
            w += G;
        }
        const int x0 = (t % g.tiles_x) * TX, y0 = (t / g.tiles_x) * TY;
        // in-plane global offsets of the staged elements and of the cells
        unsigned src[K::K], go[2];
#pragma unroll
        for (int j = 0; j < K::K; ++j) {
            const int idx = tid + j * NT, row = idx / PW, col = idx - row * PW;
            src[j] = plane_off<BIG>(wrapi(y0 - NST + row, g.ny), wrapi(x0 - 4 + col, g.nx), g.nx);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) go[k] = plane_off<BIG>(wrapi(y0 + cy[k], g.ny), wrapi(x0 + cx[k], g.nx), g.nx);
        const bool tile = stages == NST;   // tile cells write the result
        const bool ok0 = tile && x0 + cx[0] < g.nx && y0 + cy[0] < g.ny, ok1 = tile && x0 + cx[1] < g.nx && y0 + cy[1] < g.ny;

        const int pfirst = z0 - NST, plast = z1 + NST - 1;
        auto stage = [&](int64_t z_off, int slot) {
            const float *s = in + z_off;
#pragma unroll
            for (int j = 0; j < K::K; ++j)
                if ((j + 1) * NT <= K::PH * PW || tid + j * NT < K::PH * PW)
                    cp_async4(sm + slot + 4 * (tid + j * NT), plane_at<BIG>(s, src[j]));
            cp_async_commit();
        };

        Dep dep[3];                            // planes p-1, p-2, p-3 in turn
        float2 ph[3], lu[3], ps[3];            // own columns
        float2 u[3];                           // velocity of plane p - 1
        int zc = wrapi(pfirst, g.nz);          // plane p modulo nz
        int sp = 0, s1 = 0, s2 = 0;            // shared planes of Phi_p, Phi_{p-1}, Phi_{p-2}
        stage((int64_t)zc * g.plane, 0);

        // the result of plane p - back for the thread's cells
        auto store = [&](int back, float2 v) {
            int q = zc - 1 - back;
            while (q < 0) q += g.nz;
            float *const dst = out + (int64_t)q * g.plane;
            if (ok0) *plane_at<BIG>(dst, go[0]) = v.x;
            if (ok1) *plane_at<BIG>(dst, go[1]) = v.y;
        };

        // iteration p; I0 = (p - pfirst) mod 3 is the turn of plane p in the histories
        auto plane = [&](auto turn, int p) {
            constexpr int I0 = decltype(turn)::value, I1 = (I0 + 2) % 3, I2 = (I0 + 1) % 3;
            cp_async_wait_all();
            __syncthreads();
            const int64_t zoff = (int64_t)zc * g.plane;
            zc = zc + 1 == g.nz ? 0 : zc + 1;
            const int nslot = sp + PL == K::NPHI * PL ? 0 : sp + PL;
            if (p < plast) stage((int64_t)zc * g.plane, nslot);
            // ---- stage 1 at plane p - 1: L_U[Phi]
            if (stages >= 1) {
                ph[I0] = make_float2(lds(sm, sp + o[0]), lds(sm, sp + o[1]));
                const bool on1 = p >= pfirst + 2;
                bool over = false;
                if (on1) dep[I0] = departure(u, sx, sy, sz, over);
                bad |= over && stages == NST;
                if (p < plast) {   // the velocity of plane p, for the next iteration
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const float *v = vel + d * g.ncell + zoff;
                        u[d] = make_float2(*plane_at<BIG>(v, go[0]), *plane_at<BIG>(v, go[1]));
                    }
                }
                if (on1) {
                    const float2 v = trilinear<1>(sm, dep[I0], o, s1, s2, sp, ph[I1], ph[I2], ph[I0]);
                    if constexpr (NST == 1) {
                        store(1, v);
                    } else {
                        lu[I0] = v;
                        sts(sm, K::L0 + I0 * PL + o[0], v.x);
                        sts(sm, K::L0 + I0 * PL + o[1], v.y);
                    }
                }
            }
            if constexpr (NST >= 2) {
                __syncthreads();
                // ---- stage 2 at plane p - 2: Phi_bar and the correction
                constexpr int Q0 = K::L0 + I1 * PL, QM = K::L0 + I2 * PL, QP = K::L0 + I0 * PL;
                if (p >= pfirst + 4 && stages >= 2) {
                    const float2 bar = trilinear<-1>(sm, dep[I1], o, Q0, QP, QM, lu[I1], lu[I0], lu[I2]);
                    const float2 f = ph[I2], to = NST == 2 ? lu[I1] : f;
                    const float2 r = make_float2(__fmaf_rn(f.x - bar.x, 0.5f, to.x), __fmaf_rn(f.y - bar.y, 0.5f, to.y));
                    if constexpr (NST == 2) {
                        store(2, r);
                    } else {
                        ps[I0] = r;
                        sts(sm, K::P0 + I0 * PL + o[0], r.x);
                        sts(sm, K::P0 + I0 * PL + o[1], r.y);
                    }
                }
            }
            if constexpr (NST >= 3) {
                __syncthreads();
                // ---- stage 3 at plane p - 3: L_U[Psi] (Psi planes p-4, p-3, p-2 in turn I2, I1, I0)
                constexpr int Q0 = K::P0 + I1 * PL, QM = K::P0 + I2 * PL, QP = K::P0 + I0 * PL;
                if (p >= pfirst + 6 && stages >= 3)
                    store(3, trilinear<1>(sm, dep[I2], o, Q0, QM, QP, ps[I1], ps[I2], ps[I0]));
            }
            s2 = s1;
            s1 = sp;
            sp = nslot;
        };
        for (int p = pfirst; p <= plast; p += 3) {
            plane(std::integral_constant<int, 0>{}, p);
            if (p + 1 <= plast) plane(std::integral_constant<int, 1>{}, p + 1);
            if (p + 2 <= plast) plane(std::integral_constant<int, 2>{}, p + 2);
        }
        __syncthreads();   // shared planes are reused by the next segment
    }
    flag_cfl(g.status, bad);
}

template <int NST, bool BIG>
cudaError_t go(Geo g, int grid, const float *in, float *out, const float *vel, const FieldSet &fs, cudaStream_t st)
{
    using K = Lay<NST>;
    auto kern = k_unsplit32<NST, BIG>;
    static ResidencyCache cache;
    Residency res;
    const cudaError_t e = residency(cache, kern, K::NT, K::SMEM, true, res);
    if (e != cudaSuccess) return e;
    g.tiles_x = (g.nx + TX - 1) / TX;
    g.tiles_y = (g.ny + TY - 1) / TY;
    const int64_t total = (int64_t)g.tiles_x * g.tiles_y * (g.tz > 0 ? g.chunks : g.nz);
    int64_t gr = total;
    // a plane of one CTA per SM takes 0.58 of a plane of two (BEC, 256^3)
    if (g.tz == 0)
        gr = plan_ctas((int64_t)g.tiles_x * g.tiles_y, g.nz, 2 * NST, 0.58, res.per_sm, res.sms, fs.n);
    if (grid > 0 && grid < total) gr = grid;
    if (gr < 1) gr = 1;
    if (gr > 0x7fffffff) return cudaErrorInvalidConfiguration;
    kern<<<dim3((unsigned)gr, fs.n), K::NT, K::SMEM, st>>>(in, out, vel, g, (float)g.sx, (float)g.sy, (float)g.sz, fs.fin,
                                                        fs.fout);
    return cudaGetLastError();
}

}  // namespace

bool unsplit32_serves(int scheme, int ndim, const int64_t dims[3], bool vec)
{
    if (ndim != 3) return false;
    if (!vec) return true;
    // by the (column tile, plane) pairs of the grid: FEC crosses over between 2600
    // (48 x 200 x 100: 20.4 against 21.6 us) and 4096 (128^3: 25.4 against 24.9), BEC
    // between 8000 (160^3: 61.3 against 62.6) and 11200 (256 x 100 x 200: 91 against 87).
    // Not where the tiles alone fill the SMs and have few planes: the equal shares then
    // cut most tiles, and each cut warms up again (FEC 300 x 300 x 7 16.1 against 13.7 us,
    // 512 x 512 x 5 27.4 against 18.0; BEC 512 x 512 x 8 50.8 against 48.3, x 11 59.5
    // against 62.2, 2048 x 2048 x 1 263 against 224).
    const int64_t tiles = ((dims[0] + TX - 1) / TX) * ((dims[1] + TY - 1) / TY);
    const bool few_tiles = tiles < 152;
    return scheme == 2 ? tiles * dims[2] < 9000 && (few_tiles || dims[2] >= 10) : tiles * dims[2] < 3000 && few_tiles;
}

cudaError_t launch_unsplit32(int scheme, Geo g, int grid, const void *in, void *out, const void *vel,
                             const FieldSet &fs, cudaStream_t st)
{
    const float *i = static_cast<const float *>(in), *v = static_cast<const float *>(vel);
    float *o = static_cast<float *>(out);
    const bool big = g.plane >= (int64_t)1 << 30;
    switch (scheme) {
    case 0: return big ? go<1, true>(g, grid, i, o, v, fs, st) : go<1, false>(g, grid, i, o, v, fs, st);
    case 1: return big ? go<2, true>(g, grid, i, o, v, fs, st) : go<2, false>(g, grid, i, o, v, fs, st);
    default: return big ? go<3, true>(g, grid, i, o, v, fs, st) : go<3, false>(g, grid, i, o, v, fs, st);
    }
}

}  // namespace sl
