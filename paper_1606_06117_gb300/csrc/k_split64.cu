// k_split64.cu -- fused directionally split third-order step (SL_CEC) with
// double arithmetic (SL_F64, and SL_F32_D64 with float storage), any size.
//
// What bounds it: the FP64 pipe.  GB300 issues about two double operations per
// clock and SM (measured: 0.62 T DFMA/s, 0.53 T/s of DADD, DMUL, DSETP or
// float-to-double conversions over the GPU), so one warp-wide double
// instruction costs as much as some 60 others, and HBM and the integer and
// shared-memory pipes idle next to it (256^3: 1 ms of double arithmetic at 33
// operations per cell against 0.1 ms of HBM traffic, per step).  Hence:
//  - every L_U[Phi] and delta of a sweep is computed once, by one thread, and
//    handed over through shared memory (runs held in registers compute them
//    again at both ends of every run);
//  - signs, comparisons with 1 and float-to-double widening use integer
//    operations on the bit patterns (a DSETP or F2F costs a double operation);
//  - the work of a phase is spread evenly over the CTA's warps, and so over the
//    four sub-partitions of the SM, each with its own FP64 pipe;
//  - persistent CTAs take equal shares of the (column tile, plane) pairs.
// Ten double operations per cell and sweep (sl_common.cuh's form takes eleven
// and its comparisons); with the halo about 38 (x,y,z) and 44 (z,y,x) per cell
// on 32 x 16 tiles, where register runs with double comparisons took 121 and
// more.  Two and three CTAs of 256 threads per SM cover each other's barriers.
// Measured (CUDA events), a step of each order: 256^3 SL_F64 6.56 ms before
// (32 x 16 and 32 x 8 tiles, 32-plane items), 2.90 ms now; the Rayleigh-Benard step of a 50 x 50 box, which
// advects three fields with this kernel, 29.9 -> 23.9 us.
#include "sl_internal.h"

namespace sl {
namespace {

constexpr int TX = 32;

// -------------------------------------------------- bit-pattern operations
__device__ __forceinline__ double pick(int s, double pos, double neg, double zero)
{
    return s > 0 ? pos : (s < 0 ? neg : zero);
}

// ------------------------------------------------------- the sweep's stages
// The 1D scheme of sl_common.cuh with L_U[Phi] written from the cell,
//   L_j = Phi_j - U_j (Phi_j - Phi_{j-s_j}),   delta_j = (Phi_j - L_j) - U_j (L_{j+s_j} - L_j),
// one operation less than from W = 1 - U.  U = 1 takes the neighbour itself, so
// that an integer Courant number stays an exact shift (delta is then exactly
// zero); equal neighbours keep constants and C = 0 exact.  delta starts from the rounded
// L_j: half of L_j's rounding error then cancels in the result (U ((Phi_j -
// Phi_{j-s_j}) - (L_{j+s_j} - L_j)), as many operations, left smooth fields 4 %
// further from the exact step).
__device__ __forceinline__ double lu(double c, double p, double nb)
{
    const bool unit = (__double2hiint(c) & 0x7fffffff) == 0x3ff00000 && __double2loint(c) == 0;
    return unit ? nb : fma(-fabs(c), p - nb, p);
}
__device__ __forceinline__ double delta_of(double c, double p, double L, double Ln)
{
    return fma(-fabs(c), Ln - L, p - L);
}
__device__ __forceinline__ double cec_of(double c, double L, double d, double dn)
{
    return fma(fma(fabs(c), 1.0 / 6.0, 1.0 / 6.0), dn - d, fma(0.5, d, L));
}

// Phi of a cell for the two stages of an in-plane sweep that use it: a float is widened
// once and kept in the cell's place for delta until delta replaces it (widened again,
// SL_F32_D64 took 3.98 ms for 3.86 at 256^3, a step of each order), a double is read again.
__device__ __forceinline__ double keep(double v, double &) { return v; }
__device__ __forceinline__ double keep(float v, double &place) { return place = widen(v); }
__device__ __forceinline__ double kept(const double &v, double) { return v; }
__device__ __forceinline__ double kept(const float &, double place) { return place; }

// Sliding window of the sweep along z for one column (ZWin of sl_common.cuh):
// after a push of Phi_p and C_{p-1} the result is the value at p - 3.
template <typename T>
struct ZWin64 {
    double ph[2], L[2], c[2], dl[2];   // Phi at p-2, p-1; L, C at p-3, p-2; delta at p-4, p-3

    __device__ __forceinline__ void init()
    {
        ph[0] = ph[1] = L[0] = L[1] = c[0] = c[1] = dl[0] = dl[1] = 0.0;
    }
    __device__ __forceinline__ T push(double phi, double cn)
    {
        const double Ln = lu(cn, ph[1], pick(sgn_bits(cn), ph[0], phi, ph[1]));
        const double dn = delta_of(c[1], ph[0], L[1], pick(sgn_bits(c[1]), Ln, L[0], L[1]));
        const T out = T(cec_of(c[0], L[0], dl[1], pick(sgn_bits(c[0]), dl[0], dn, dl[1])));
        ph[0] = ph[1];
        ph[1] = phi;
        L[0] = L[1];
        L[1] = Ln;
        c[0] = c[1];
        c[1] = cn;
        dl[0] = dl[1];
        dl[1] = dn;
        return out;
    }
};

// Stages rows [r0, r0 + NR) x columns [c0, c0 + NC) of one plane at row stride
// LD.  VEC: 16-byte copies of whole aligned chunks (nx a multiple of the chunk,
// c0 and x0 too), offsets computed once per segment.
template <typename T, int NT, int NR, int NC, int LD, bool VEC>
struct Stage64 {
    static constexpr int V = VEC ? 16 / sizeof(T) : 1, CPR = NC / V, N = NR * CPR, K = (N + NT - 1) / NT;
    int off[K];

    __device__ __forceinline__ void setup(int tid, int x0, int y0, int r0, int c0, int nx, int ny)
    {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int idx = tid + k * NT, row = idx / CPR, cc = idx - row * CPR;
            off[k] = idx < N ? wrapi(y0 + r0 + row, ny) * nx + wrapi(x0 + c0 + cc * V, nx) : -1;
        }
    }
    __device__ __forceinline__ void issue(int tid, T *dst, const T *src) const
    {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (off[k] < 0) continue;
            const int idx = tid + k * NT, row = idx / CPR, cc = idx - row * CPR;
            if constexpr (VEC)
                cp_async16(dst + row * LD + cc * V, src + off[k]);
            else
                cp_async_elem(dst + row * LD + cc, src + off[k]);
        }
    }
};

// One stage of an in-plane sweep over rows [0, NR) x columns [0, NC), a cell
// per thread and turn.
template <int NT, int NR, int NC, typename F>
__device__ __forceinline__ void each(int tid, F f)
{
#pragma unroll
    for (int k = 0; k < (NR * NC + NT - 1) / NT; ++k) {
        const int idx = tid + k * NT;
        if (NR * NC % NT == 0 || idx < NR * NC) f(idx / NC, idx - (idx / NC) * NC);
    }
}

// Shared memory of the two orders.  Staged planes in T, double-buffered; the
// sweeps' L_U[Phi], Courant numbers and delta in double.
template <typename T, int TY, bool HAS_Z, bool ZYX>
struct Lay {
    static constexpr int PW = TX + 8 + (sizeof(T) == 8 ? 2 : 4);      // staged row stride
    static constexpr int PHI = (TY + 6) * PW;                         // rows [-3, TY+3), columns [-4, TX+4)
    // x,y,z: u_x as Phi, u_y rows [-2, TY+2) and u_z rows [0, TY) of the tile's columns;
    // z,y,x: u_z as Phi, u_y rows [-2, TY+2) and u_x rows [0, TY) of the widened columns
    static constexpr int U1 = ZYX ? (HAS_Z ? PHI : 0) : PHI;
    static constexpr int U2 = (TY + 4) * (ZYX ? PW : TX);
    static constexpr int U3 = ZYX ? TY * PW : (HAS_Z ? TY * TX : 0);
    static constexpr int NB = HAS_Z ? 2 : 1;
    static constexpr int SLOT = PHI + U1 + U2 + U3;
    // sweep arrays: x,y,z runs its x sweep on TY + 6 rows; z,y,x its y sweep on TX + 6 columns
    static constexpr int CW = TX + 6;
    static constexpr int NL = ZYX ? (TY + 4) * CW : (TY + 6) * (TX + 4);
    static constexpr int NS = ZYX ? (TY + 6) * CW : (TY + 6) * TX;    // swept values handed on, in T
    static constexpr size_t smem() { return 8 * (size_t)(3 * NL) + sizeof(T) * (size_t)(NB * SLOT + NS); }
};

template <typename T, int TY, int NT, bool HAS_Z, bool VEC, bool ZYX>
__global__ void __launch_bounds__(NT, HAS_Z ? 2 : 1)
k_cec64(const T *__restrict__ in, T *__restrict__ out, const T *__restrict__ vel, Geo g, int64_t fin, int64_t fout)
{
    using K = Lay<T, TY, HAS_Z, ZYX>;
    constexpr int PW = K::PW, CW = K::CW, NB = K::NB;
    in += (int64_t)blockIdx.y * fin;   // field of this CTA (FieldSet)
    out += (int64_t)blockIdx.y * fout;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *const sL = reinterpret_cast<double *>(smem_raw), *const sC = sL + K::NL, *const sD = sC + K::NL;
    T *const buf = reinterpret_cast<T *>(sD + K::NL), *const sS = buf + NB * K::SLOT;
    const int tid = threadIdx.x;
    const double sx = g.sx, sy = g.sy, sz = g.sz;
    const int nzz = HAS_Z ? g.nz : 1;
    // Work: with g.tz planes per item the items go round the grid, with g.tz = 0
    // every CTA takes one equal share of the (column tile, plane) pairs.
    const bool shares = g.tz == 0;
    const int ntiles = g.tiles_x * g.tiles_y;
    const int64_t total = (int64_t)ntiles * (shares ? nzz : g.chunks), G = gridDim.x;
    int64_t w = shares ? total * blockIdx.x / G : blockIdx.x;
    const int64_t wend = shares ? total * (blockIdx.x + 1) / G : total;
    bool bad = false;
    pdl_release();
    pdl_wait();

    while (w < wend) {
        int t, z0, z1;
        if (shares) {
            t = (int)(w / nzz);
            z0 = (int)(w - (int64_t)t * nzz);
            z1 = (int)min((int64_t)nzz, z0 + (wend - w));
            w += z1 - z0;
        } else {
            t = (int)(w % ntiles);
            z0 = (int)(w / ntiles) * g.tz;
            z1 = min(z0 + g.tz, nzz);
            w += G;
        }
        const int x0 = (t % g.tiles_x) * TX, y0 = (t / g.tiles_x) * TY;
        Stage64<T, NT, TY + 6, TX + 8, PW, VEC> stP;
        Stage64<T, NT, TY + 4, ZYX ? TX + 8 : TX, ZYX ? PW : TX, VEC> stY;
        Stage64<T, NT, TY, ZYX ? TX + 8 : TX, ZYX ? PW : TX, VEC> stT;
        stP.setup(tid, x0, y0, -3, -4, g.nx, g.ny);
        stY.setup(tid, x0, y0, -2, ZYX ? -4 : 0, g.nx, g.ny);
        if (ZYX || HAS_Z) stT.setup(tid, x0, y0, 0, ZYX ? -4 : 0, g.nx, g.ny);

        const int pfirst = HAS_Z ? z0 - 3 : 0, plast = HAS_Z ? z1 + 2 : 0;
        auto issue = [&](int p, int slot) {
            T *const b = buf + slot * K::SLOT;
            const int64_t at = HAS_Z ? (int64_t)wrapi(p, g.nz) * g.plane : 0;
            stP.issue(tid, b, in + at);
            if constexpr (!ZYX) {
                stP.issue(tid, b + K::PHI, vel + at);
                stY.issue(tid, b + K::PHI + K::U1, vel + g.ncell + at);
                if constexpr (HAS_Z)
                    stT.issue(tid, b + K::PHI + K::U1 + K::U2,
                              vel + 2 * g.ncell + (int64_t)wrapi(p - 1, g.nz) * g.plane);
            } else {
                if constexpr (HAS_Z)
                    stP.issue(tid, b + K::PHI, vel + 2 * g.ncell + (int64_t)wrapi(p - 1, g.nz) * g.plane);
                const int64_t ak = HAS_Z ? (int64_t)wrapi(p - 3, g.nz) * g.plane : 0;
                stY.issue(tid, b + K::PHI + K::U1, vel + g.ncell + ak);
                stT.issue(tid, b + K::PHI + K::U1 + K::U2, vel + ak);
            }
            cp_async_commit();
        };

        // z windows of this thread's columns (x,y,z: the tile's cells; z,y,x: the
        // cells of the tile widened by the x and y halos)
        constexpr int NCOL = ZYX ? (TY + 6) * CW : TY * TX;
        constexpr int NW = HAS_Z ? (NCOL + NT - 1) / NT : 1;
        ZWin64<T> win[NW];
#pragma unroll
        for (int k = 0; k < NW; ++k) win[k].init();

        issue(pfirst, 0);
        for (int p = pfirst; p <= plast; ++p) {
            const int slot = (p - pfirst) & (NB - 1);
            cp_async_wait_all();
            __syncthreads();
            if (p < plast) issue(p + 1, slot ^ 1);
            const T *const sP = buf + slot * K::SLOT, *const s1 = sP + K::PHI, *const s2 = s1 + K::U1, *const s3 = s2 + K::U2;

            if constexpr (!ZYX) {
                // ---- x sweep: rows [-3, TY+3) -> sS
                each<NT, TY + 6, TX + 4>(tid, [&](int r, int j) {          // L at x = j - 2
                    const double c = widen(s1[r * PW + j + 2]) * sx;
                    const T *q = sP + r * PW + j + 2;
                    sC[r * (TX + 4) + j] = c;
                    sL[r * (TX + 4) + j] = lu(c, keep(q[0], sD[r * (TX + 4) + j]), widen(q[-sgn_bits(c)]));
                    if (j >= 2 && j < TX + 2) bad |= beyond_one(c);
                });
                __syncthreads();
                each<NT, TY + 6, TX + 2>(tid, [&](int r, int j) {          // delta at x = j - 1
                    const double c = sC[r * (TX + 4) + j + 1];
                    const double *l = sL + r * (TX + 4) + j + 1;
                    double &d = sD[r * (TX + 4) + j + 1];
                    d = delta_of(c, kept(sP[r * PW + j + 3], d), l[0], l[sgn_bits(c)]);
                });
                __syncthreads();
                each<NT, TY + 6, TX>(tid, [&](int r, int x) {
                    const double c = sC[r * (TX + 4) + x + 2];
                    const double *d = sD + r * (TX + 4) + x + 2;
                    sS[r * TX + x] = T(cec_of(c, sL[r * (TX + 4) + x + 2], d[0], d[-sgn_bits(c)]));
                });
                __syncthreads();
                // ---- y sweep on the tile's columns
                each<NT, TY + 4, TX>(tid, [&](int r, int x) {              // L at y = r - 2
                    const double c = widen(s2[r * TX + x]) * sy;
                    const T *q = sS + (r + 1) * TX + x;
                    sC[r * TX + x] = c;
                    sL[r * TX + x] = lu(c, keep(q[0], sD[r * TX + x]), widen(q[-sgn_bits(c) * TX]));
                    if (r >= 2 && r < TY + 2) bad |= beyond_one(c);
                });
                __syncthreads();
                each<NT, TY + 2, TX>(tid, [&](int r, int x) {              // delta at y = r - 1
                    const double c = sC[(r + 1) * TX + x];
                    const double *l = sL + (r + 1) * TX + x;
                    double &d = sD[(r + 1) * TX + x];
                    d = delta_of(c, kept(sS[(r + 2) * TX + x], d), l[0], l[sgn_bits(c) * TX]);
                });
                __syncthreads();
                // ---- the y sweep's value, then the cell's z window
#pragma unroll
                for (int k = 0; k < TY * TX / NT; ++k) {
                    const int idx = tid + k * NT, r = idx / TX, x = idx % TX;
                    const double c = sC[(r + 2) * TX + x];
                    const double *d = sD + (r + 2) * TX + x;
                    T v = T(cec_of(c, sL[(r + 2) * TX + x], d[0], d[-sgn_bits(c) * TX]));
                    if constexpr (HAS_Z) {
                        const double cz = widen(s3[idx]) * sz;
                        bad |= beyond_one(cz);
                        v = win[k].push(widen(v), cz);
                    }
                    if ((!HAS_Z || p - 3 >= z0) && x0 + x < g.nx && y0 + r < g.ny)
                        out[(HAS_Z ? (int64_t)(p - 3) * g.plane : 0) + (int64_t)(y0 + r) * g.nx + x0 + x] = v;
                }
            } else {
                // ---- z sweep on the widened columns -> sS (column j is x = j - 3)
                if constexpr (HAS_Z) {
#pragma unroll
                    for (int k = 0; k < NW; ++k) {
                        const int idx = tid + k * NT, r = idx / CW, j = idx - (idx / CW) * CW;
                        if (idx < NCOL) {
                            const double c = widen(s1[r * PW + j + 1]) * sz;
                            sS[idx] = win[k].push(widen(sP[r * PW + j + 1]), c);
                            if (r >= 3 && r < TY + 3 && j >= 3 && j < TX + 3) bad |= beyond_one(c);
                        }
                    }
                    __syncthreads();
                    if (p - 3 < z0) continue;
                }
                const T *const src = HAS_Z ? sS : sP + 1;
                constexpr int SW = HAS_Z ? CW : PW;
                // ---- y sweep on the widened columns
                each<NT, TY + 4, CW>(tid, [&](int r, int j) {              // L at y = r - 2
                    const double c = widen(s2[r * PW + j + 1]) * sy;
                    const T *q = src + (r + 1) * SW + j;
                    sC[r * CW + j] = c;
                    sL[r * CW + j] = lu(c, keep(q[0], sD[r * CW + j]), widen(q[-sgn_bits(c) * SW]));
                    if (r >= 2 && r < TY + 2 && j >= 3 && j < TX + 3) bad |= beyond_one(c);
                });
                __syncthreads();
                each<NT, TY + 2, CW>(tid, [&](int r, int j) {              // delta at y = r - 1
                    const double c = sC[(r + 1) * CW + j];
                    const double *l = sL + (r + 1) * CW + j;
                    double &d = sD[(r + 1) * CW + j];
                    d = delta_of(c, kept(src[(r + 2) * SW + j], d), l[0], l[sgn_bits(c) * CW]);
                });
                __syncthreads();
                each<NT, TY, CW>(tid, [&](int r, int j) {                  // over sS: its z-swept values are spent
                    const double c = sC[(r + 2) * CW + j];
                    const double *d = sD + (r + 2) * CW + j;
                    sS[r * CW + j] = T(cec_of(c, sL[(r + 2) * CW + j], d[0], d[-sgn_bits(c) * CW]));
                });
                __syncthreads();
                // ---- x sweep on the tile's rows
                each<NT, TY, TX + 4>(tid, [&](int r, int j) {              // L at x = j - 2
                    const double c = widen(s3[r * PW + j + 2]) * sx;
                    const T *q = sS + r * CW + j + 1;
                    sC[r * (TX + 4) + j] = c;
                    sL[r * (TX + 4) + j] = lu(c, keep(q[0], sD[r * (TX + 4) + j]), widen(q[-sgn_bits(c)]));
                    if (j >= 2 && j < TX + 2) bad |= beyond_one(c);
                });
                __syncthreads();
                each<NT, TY, TX + 2>(tid, [&](int r, int j) {              // delta at x = j - 1
                    const double c = sC[r * (TX + 4) + j + 1];
                    const double *l = sL + r * (TX + 4) + j + 1;
                    double &d = sD[r * (TX + 4) + j + 1];
                    d = delta_of(c, kept(sS[r * CW + j + 2], d), l[0], l[sgn_bits(c)]);
                });
                __syncthreads();
                each<NT, TY, TX>(tid, [&](int r, int x) {
                    const double c = sC[r * (TX + 4) + x + 2];
                    const double *d = sD + r * (TX + 4) + x + 2;
                    const T v = T(cec_of(c, sL[r * (TX + 4) + x + 2], d[0], d[-sgn_bits(c)]));
                    if (x0 + x < g.nx && y0 + r < g.ny)
                        out[(HAS_Z ? (int64_t)(p - 3) * g.plane : 0) + (int64_t)(y0 + r) * g.nx + x0 + x] = v;
                });
            }
        }
        __syncthreads();   // shared buffers are reused by the next segment
    }
    flag_cfl(g.status, bad);
}

template <typename T, int TY, int NT, bool HAS_Z, bool VEC, bool ZYX>
cudaError_t go(Geo g, const Launch &lc, const void *in, void *out, const void *vel, const FieldSet &fs, cudaStream_t st)
{
    using K = Lay<T, TY, HAS_Z, ZYX>;
    auto kern = k_cec64<T, TY, NT, HAS_Z, VEC, ZYX>;
    static ResidencyCache cache;
    Residency res;
    const cudaError_t e = residency(cache, kern, NT, K::smem(), true, res);
    if (e != cudaSuccess) return e;
    g.tiles_x = (g.nx + TX - 1) / TX;
    g.tiles_y = (g.ny + TY - 1) / TY;
    const int64_t tiles = (int64_t)g.tiles_x * g.tiles_y;
    const int64_t total = tiles * (g.tz > 0 ? g.chunks : g.nz);
    int64_t gr = total;
    if (HAS_Z && g.tz == 0)   // the FP64 pipe is shared: one CTA per SM is hardly slower per plane than half of two
        gr = plan_ctas(tiles, g.nz, 6, 0.55, res.per_sm, res.sms, fs.n);
    if (lc.grid > 0 && lc.grid < gr) gr = lc.grid;
    if (gr < 1) gr = 1;
    if (gr > 0x7fffffff) return cudaErrorInvalidConfiguration;
    return launch_kernel(kern, dim3((unsigned)gr, fs.n), NT, K::smem(), st, lc.pdl, static_cast<const T *>(in),
                         static_cast<T *>(out), static_cast<const T *>(vel), g, fs.fin, fs.fout);
}

template <typename T, bool HAS_Z, bool VEC>
cudaError_t by_order(int parity, const Geo &g, const Launch &lc, const void *in, void *out, const void *vel,
                     const FieldSet &fs, cudaStream_t st)
{
    if constexpr (HAS_Z) {
        return (parity & 1) ? go<T, 16, 256, true, VEC, true>(g, lc, in, out, vel, fs, st)
                            : go<T, 16, 256, true, VEC, false>(g, lc, in, out, vel, fs, st);
    } else {
        if (split64_tile_y(false, g.nx, g.ny, fs.n) == 4)
            return (parity & 1) ? go<T, 4, 128, false, VEC, true>(g, lc, in, out, vel, fs, st)
                                : go<T, 4, 128, false, VEC, false>(g, lc, in, out, vel, fs, st);
        return (parity & 1) ? go<T, 16, 256, false, VEC, true>(g, lc, in, out, vel, fs, st)
                            : go<T, 16, 256, false, VEC, false>(g, lc, in, out, vel, fs, st);
    }
}

}  // namespace

// Small planes take 4-row tiles, which spread them over more SMs: the 32 x 16 tiles of
// a 128^2 plane would leave 120 of 152 SMs idle, and the wider halo (about 38 double
// operations per cell in place of 24) costs less than that until the larger tiles
// give every SM two CTAs.
int split64_tile_y(bool has_z, int64_t nx, int64_t ny, int fields)
{
    return !has_z && (nx + TX - 1) / TX * ((ny + 15) / 16) * fields < 2 * 152 ? 4 : 16;
}

cudaError_t launch_split_cec64(bool f32_storage, Geo g, int parity, Launch lc, bool has_z, const void *in, void *out,
                               const void *vel, const FieldSet &fs, cudaStream_t st)
{
    const bool vec = lc.aligned && g.nx % (f32_storage ? 4 : 2) == 0;
    if (f32_storage) {
        if (has_z) return vec ? by_order<float, true, true>(parity, g, lc, in, out, vel, fs, st)
                              : by_order<float, true, false>(parity, g, lc, in, out, vel, fs, st);
        return vec ? by_order<float, false, true>(parity, g, lc, in, out, vel, fs, st)
                   : by_order<float, false, false>(parity, g, lc, in, out, vel, fs, st);
    }
    if (has_z) return vec ? by_order<double, true, true>(parity, g, lc, in, out, vel, fs, st)
                          : by_order<double, true, false>(parity, g, lc, in, out, vel, fs, st);
    return vec ? by_order<double, false, true>(parity, g, lc, in, out, vel, fs, st)
               : by_order<double, false, false>(parity, g, lc, in, out, vel, fs, st);
}

}  // namespace sl
