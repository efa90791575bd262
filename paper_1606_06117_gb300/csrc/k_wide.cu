// k_wide.cu -- steps at any Courant number, with non-local interpolation: the
// corners of L_U bracket the departure point X = i - C (cell units) however far
// it is, so |C| > 1 needs no wider stencil than |C| < 1, only a gather from
// further away (Sec. 4: semi-Lagrangian schemes may exceed CFL 1 when the
// interpolation uses non-neighbouring points).
//
//   CIR, FEC, BEC  the operator compositions of Sec. 2 (eqs. intro:FEC,
//                  intro:BEC) with the unsplit multilinear L_U (eq. CIR2D and
//                  its 3D tensor product).
//   CEC            split 1D sweeps (Sec. 5 eqs. split:1-2, order x,y,z on even
//                  steps and z,y,x on odd steps) with the weights of eq.
//                  intro:CECcoefSL, 3a = 2 - 1/(U % 1), b = 1 - a, and the
//                  correction of the local scheme taken at the departure cell:
//                  with m = trunc(C), r = C - m, j = i - m, s = sgn r,
//                  CEC_i = L_U[Phi]_i + delta_j/2 + (1 + |r|)/6 (delta_{j-s} - delta_j).
//                  For constant velocity this is the local CEC at Courant
//                  number r shifted by m cells (third order); for |C| < 1 it
//                  is the local CEC.
//
// A CEC sweep whose lines fit in shared memory is one kernel.  Otherwise one
// gather kernel per interpolation call, each with the scheme's pointwise
// combination as its epilogue, and one for the CEC correction.  Intermediate
// fields live in a caller-owned workspace.
#include <algorithm>
#include <type_traits>

#include "sl_internal.h"

namespace sl {
namespace {

enum Epi { EPI_NONE = 0, EPI_FEC = 1, EPI_BEC_IN = 2, EPI_DELTA = 3 };

constexpr int kWideBlock = 128;

struct WideGeo {
    int n[3];          // cells per axis (x, y, z)
    int64_t ncell;     // n[0] n[1] n[2]
    double s[3];       // dt / dx_d: Courant number = u_d s_d
    unsigned *status;  // SL_DEV_CFL: a non-finite or huge departure point
};

// Integer part and fraction of a displacement D (cell units): D = fl + f,
// f in [0, 1).  A non-finite displacement, or one of 2^30 cells or more, is
// flagged and replaced by 0, so that every index below stays in 32 bits and
// in bounds (grid sizes are at most 2^30).
template <typename T>
__device__ __forceinline__ int floor_split(T D, T &f, bool &bad)
{
    if (!(fabs(D) < T(1073741824.0))) {
        bad = true;
        D = T(0);
    }
    const T fl = floor(D);
    f = D - fl;
    return (int)fl;
}

// v reduced into [0, n), for v = a cell index (< n <= 2^30) plus an offset of
// magnitude below 2^30, so v and v - n fit in 32 bits.  Departure points
// within one period take a compare and an add; the remainder only runs beyond.
__device__ __forceinline__ int wrapn(int v, int n)
{
    if (v < 0) {
        v += n;
        if (v >= 0) return v;
    } else if (v < n) {
        return v;
    } else {
        v -= n;
        if (v < n) return v;
    }
    const int r = v % n;
    return r < 0 ? r + n : r;
}

// Index of a cell, in 32 bits (I = unsigned) on FP32 grids of fewer than 2^32 cells: the
// gathers are bound by instruction issue, and eight 64-bit products per cell were
// a sixth of their time (256^3 FP32, CIR / FEC / BEC: 131 / 270 / 403 us with 64-bit
// indices, 108 / 232 / 338 with 32).  All corners' places before all loads, so that
// every load of a thread is in flight at once, measured slower (148 / 280 / 425).
template <typename I = int64_t>
__device__ __forceinline__ I cell_at(const WideGeo &g, int x, int y, int z)
{
    return ((I)z * (I)g.n[1] + (I)y) * (I)g.n[0] + (I)x;
}

// Each thread takes the cells (x, y0 + k, z), k < kWideRows: a warp's loads of
// one k are coalesced along x, and the rows' loads are issued together (the
// velocity of all rows, then all corners), so that several independent gathers
// are in flight per thread.
constexpr int kWideRows = 4;

// out = epilogue(L_{dir U}[src]) at every cell.  AX < 0: the multilinear
// operator on NDIM axes; AX >= 0: the 1D operator along that axis.  dir = +1
// is L_U (departure i - C), dir = -1 is L_{-U} (departure i + C, -u at its own
// arrival cell).
template <typename T, typename I, int NDIM, int AX, int EPI>
__global__ void __launch_bounds__(kWideBlock)
k_wide_interp(T *__restrict__ out, const T *__restrict__ src, const T *__restrict__ vel, const T *__restrict__ aux0,
              const T *__restrict__ aux1, WideGeo g, int dir)
{
    constexpr int R = kWideRows;
    const int x = blockIdx.x * kWideBlock + threadIdx.x, y0 = blockIdx.y * R, z = blockIdx.z;
    bool bad = false;
    bool on[R];
    I cell[R];
    T C[R][3];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        on[k] = x < g.n[0] && y0 + k < g.n[1];
        cell[k] = on[k] ? cell_at<I>(g, x, y0 + k, z) : 0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const bool moves = AX < 0 ? d < NDIM : d == AX;
            C[k][d] = moves && on[k] ? vel[(int64_t)d * g.ncell + cell[k]] * T(g.s[d]) : T(0);
        }
    }
    T val[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const int pos[3] = {x, y0 + k, z};
        int b0[3] = {pos[0], pos[1], pos[2]}, b1[3] = {pos[0], pos[1], pos[2]};
        T f[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const bool moves = AX < 0 ? d < NDIM : d == AX;
            if (moves) {
                const int fl = floor_split<T>(T(-dir) * C[k][d], f[d], bad);
                b0[d] = wrapn(pos[d] + fl, g.n[d]);
                b1[d] = b0[d] + 1 == g.n[d] ? 0 : b0[d] + 1;
            }
        }
        val[k] = T(0);
        if (!on[k]) continue;
        if constexpr (AX >= 0) {
            int q0[3] = {pos[0], pos[1], pos[2]}, q1[3] = {pos[0], pos[1], pos[2]};
            q0[AX] = b0[AX];
            q1[AX] = b1[AX];
            const T a = src[cell_at<I>(g, q0[0], q0[1], q0[2])], b = src[cell_at<I>(g, q1[0], q1[1], q1[2])];
            val[k] = a + f[AX] * (b - a);
        } else {
            // corners weighted by prod_d (1 - f_d | f_d), lerped along x, then y, then z,
            // each lerp as a + f (b - a) so that a constant field stays exact
            T c[2];
#pragma unroll
            for (int h = 0; h < (NDIM == 3 ? 2 : 1); ++h) {
                const int zz = NDIM == 3 ? (h ? b1[2] : b0[2]) : z;
                const T a00 = src[cell_at<I>(g, b0[0], b0[1], zz)], a10 = src[cell_at<I>(g, b1[0], b0[1], zz)];
                const T a01 = src[cell_at<I>(g, b0[0], b1[1], zz)], a11 = src[cell_at<I>(g, b1[0], b1[1], zz)];
                const T e0 = a00 + f[0] * (a10 - a00);
                const T e1 = a01 + f[0] * (a11 - a01);
                c[h] = e0 + f[1] * (e1 - e0);
            }
            val[k] = NDIM == 3 ? c[0] + f[2] * (c[1] - c[0]) : c[0];
        }
    }
#pragma unroll
    for (int k = 0; k < R; ++k) {
        if (!on[k]) continue;
        const I i = cell[k];
        const T v = val[k];
        if constexpr (EPI == EPI_NONE) out[i] = v;
        if constexpr (EPI == EPI_FEC) out[i] = aux1[i] + (aux0[i] - v) * T(0.5);
        if constexpr (EPI == EPI_BEC_IN) out[i] = aux0[i] + (aux0[i] - v) * T(0.5);
        if constexpr (EPI == EPI_DELTA) out[i] = aux0[i] - v;
    }
    flag_cfl(g.status, bad);
}

// The CEC sweep's output along AX from L_U[Phi] (lphi) and delta = Phi - Phi_bar:
// CEC_i = lphi_i + delta_j/2 + (1 + |r|)/6 (delta_{j-s} - delta_j), m = trunc(C_i),
// r = C_i - m, j = i - m, s = sgn r.
template <typename T, int AX>
__global__ void __launch_bounds__(kWideBlock)
k_wide_cec(T *__restrict__ out, const T *__restrict__ lphi, const T *__restrict__ delta, const T *__restrict__ vel,
           WideGeo g)
{
    constexpr int R = kWideRows;
    const int x = blockIdx.x * kWideBlock + threadIdx.x, y0 = blockIdx.y * R, z = blockIdx.z;
    bool bad = false;
    bool on[R];
    int64_t cell[R];
    T C[R], L[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        on[k] = x < g.n[0] && y0 + k < g.n[1];
        cell[k] = on[k] ? cell_at(g, x, y0 + k, z) : 0;
        C[k] = on[k] ? vel[(int64_t)AX * g.ncell + cell[k]] * T(g.s[AX]) : T(0);
        L[k] = on[k] ? lphi[cell[k]] : T(0);
    }
    T dj[R], du[R], r[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        T c = C[k];
        if (!(fabs(c) < T(1073741824.0))) {
            bad = true;
            c = T(0);
        }
        const T m = trunc(c);
        r[k] = c - m;
        const int s = (r[k] > T(0)) - (r[k] < T(0));
        const int pos[3] = {x, y0 + k, z};
        int qj[3] = {pos[0], pos[1], pos[2]}, qu[3] = {pos[0], pos[1], pos[2]};
        qj[AX] = wrapn(pos[AX] - (int)m, g.n[AX]);
        qu[AX] = wrapn(pos[AX] - (int)m - s, g.n[AX]);
        dj[k] = on[k] ? delta[cell_at(g, qj[0], qj[1], qj[2])] : T(0);
        du[k] = on[k] ? delta[cell_at(g, qu[0], qu[1], qu[2])] : T(0);
    }
#pragma unroll
    for (int k = 0; k < R; ++k)
        if (on[k]) out[cell[k]] = L[k] + dj[k] * T(0.5) + (T(1) + fabs(r[k])) * T(1.0 / 6.0) * (du[k] - dj[k]);
    flag_cfl(g.status, bad);
}

dim3 wide_grid(const WideGeo &g)
{
    return dim3((g.n[0] + kWideBlock - 1) / kWideBlock, (g.n[1] + kWideRows - 1) / kWideRows, g.n[2]);
}

// --------------------------------------------- fused sweep on whole lines
// A CEC sweep along AX only reads the line it works on: L_U[Phi] at a cell
// gathers Phi near the cell's departure point, delta gathers L_U[Phi] near the
// reversed departure point, and the correction gathers delta near the
// departure cell.  So a CTA holds whole lines in shared memory (Phi, then
// delta in its place; L_U[Phi]) and writes the sweep's output: one read of Phi
// and u_AX and one write per cell (12 B in FP32), in place of the 44 B of the
// three gathers above.  Lines along x are rows (contiguous); lines along y or z
// are W adjacent x columns, so that every load and store of a warp is coalesced
// along x; the last column block of a row may be partial.
//
// What bounds it: instruction issue, so each cell's departure is worked out
// once, m = trunc C, r = C - m, and kept in registers with both gather
// positions.  With lo = i - m - [r > 0] the departure lies between lo and
// lo + 1 (fraction [r > 0] - r), and these two are also the departure cell and
// its upwind neighbour, which the correction reads; the reversed departure lies
// between lo' = i + m - [r < 0] and lo' + 1 (fraction [r < 0] + r).  Positions
// wrap by an unsigned minimum of p, p + n and p - n, and every line repeats its
// first element at its end, so that lo + 1 needs no wrap.  Courant numbers of n
// or more take a remainder first.
// Measured (256^3 FP32 at CFL 3.64, us per step of three sweeps): 291 with the
// Courant numbers in shared memory and three separate departure calculations
// (170-179 instructions per cell and sweep), 187 now (178 replayed from a graph).
// Cells per thread: with 4 a thread keeps to 64 registers, so that 32 warps fit an
// SM (8 took 98).
constexpr int kSweepCells = 4;

// unsigned wrap of p in [-n, 2 n) into [0, n)
__device__ __forceinline__ int wrap3(int p, int n)
{
    return (int)min(min((unsigned)p, (unsigned)(p + n)), (unsigned)(p - n));
}

// r > 0; a double's from its bits, since a double comparison costs as much as a
// double multiply-add, of which an SM issues two per clock
__device__ __forceinline__ bool positive(float r) { return r > 0.f; }
__device__ __forceinline__ bool positive(double r) { return __double_as_longlong(r) > 0; }
// |c| < n (false for a NaN)
__device__ __forceinline__ bool below(float c, int n) { return fabsf(c) < (float)n; }
__device__ __forceinline__ bool below(double c, int n)
{
    return (__double_as_longlong(c) & 0x7fffffffffffffffll) < __double_as_longlong((double)n);
}

// LW: log2 of the columns per tile (AX > 0).  For AX = 0 a tile is `rows` rows.
// Persistent CTAs; the loads of a CTA's next tile are issued before it works on
// the current one, so that DRAM latency runs under the three gathers (without
// that the y and z sweeps stalled on their loads).
// PART: tiles of so few cells that some warps have none in some turns; they skip these,
// which pays where double operations bound (8^3 SL_F64, a step of each order: 50.7 ->
// 17.9 us; with the test in full tiles, 256^3, 3438 -> 3871).
template <typename T, int AX, int LW, int NT, bool PART>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? 1024 / NT : 1)
k_wide_sweep(T *__restrict__ out, const T *__restrict__ src, const T *__restrict__ vel, WideGeo g, T sc, int rows,
             int tiles)
{
    constexpr int E = kSweepCells, W = 1 << LW;
    // Everything in shared memory is addressed in bytes: Phi, then delta, in lines
    // of n + 1 and a spare place; then L_U[Phi] the same way.
    extern __shared__ __align__(16) char sm[];
    constexpr int B = sizeof(T);
    const int n = g.n[AX];
    const int lines = AX == 0 ? rows : W;
    const int spare = lines * (n + 1) * B, LB = spare + B;
    const int tid = threadIdx.x;
    bool bad = false;
    const T *const va = vel + (int64_t)AX * g.ncell;
    constexpr int step = (AX == 0 ? 1 : W) * B;        // along a line
    const int period = n * step;
    const int xt = (g.n[0] + W - 1) >> LW;
    const int64_t stride = AX == 1 ? g.n[0] : (int64_t)g.n[0] * g.n[1];   // along a line (AX > 0)
    // Cell k of this thread has flat index e = tid + k NT of the tile: line e / n
    // and position e mod n of it (AX = 0), or column e mod W and position e / W.
    // pos: its distance from the line's start (AX = 0) or from column 0; own: its
    // place.  Cells beyond the tile's lines go to the spare place, and cells of a
    // partial tile beyond the grid work on zeros in places of their own.
    const int count = AX == 0 ? rows * n : n << LW;
    const int turns = (count - (tid & ~31) + NT - 1) / NT;   // of this warp
    auto has = [&](int k) { return !PART || k < turns; };
    int pos[E], line[E], own[E];
    bool rep[E];                                       // repeated at its line's end
    if constexpr (AX == 0) {
        int w = tid / n, i = tid - w * n;
        const int dw = NT / n, di = NT - dw * n;
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const bool in = tid + k * NT < count;
            pos[k] = in ? i * B : 0;
            line[k] = in ? w * (n + 1) * B : 0;
            own[k] = in ? line[k] + pos[k] : spare;
            rep[k] = in && i == 0;
            w += dw;
            i += di;
            if (i >= n) {
                i -= n;
                ++w;
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const int e = tid + k * NT;
            pos[k] = e < count ? e * B : 0;
            line[k] = 0;
            own[k] = e < count ? e * B : spare;
            rep[k] = k == 0 && tid < W;
        }
    }
    auto lds = [&](int q) { return *reinterpret_cast<const T *>(sm + q); };
    auto put = [&](int off, int k, T x) {
        *reinterpret_cast<T *>(sm + off + own[k]) = x;
        if ((AX == 0 || k == 0) && rep[k]) *reinterpret_cast<T *>(sm + off + own[k] + period) = x;
    };

    T v[E], c[E];
    int64_t q0;        // element of cell 0
    int limit;         // cells with k NT < limit are inside the grid
    const int64_t hop = AX == 0 ? NT : (int64_t)(NT >> LW) * stride;   // from cell k to k + 1
    const int64_t first = AX == 0 ? tid : (int64_t)(tid >> LW) * stride + (tid & (W - 1));
    auto load = [&](int b) {
        if constexpr (AX == 0) {
            const int64_t row0 = (int64_t)b * rows, all = (int64_t)g.n[1] * g.n[2];
            q0 = row0 * n + first;
            limit = (int)min((int64_t)rows, all - row0) * n - tid;
        } else {
            const int q = b / xt, x0 = (b - q * xt) << LW;   // q: z (AX = 1) or y (AX = 2)
            q0 = (AX == 1 ? (int64_t)q * g.n[0] * g.n[1] : (int64_t)q * g.n[0]) + x0 + first;
            limit = x0 + (tid & (W - 1)) < g.n[0] ? count - tid : 0;
        }
#pragma unroll
        for (int k = 0; k < E; ++k) {
            if (!has(k)) break;
            const bool ok = k * NT < limit;
            v[k] = ok ? src[q0 + k * hop] : T(0);
            c[k] = ok ? va[q0 + k * hop] : T(0);
        }
    };
    if (blockIdx.x < (unsigned)tiles) load(blockIdx.x);
    for (int b = blockIdx.x; b < tiles; b += gridDim.x) {
        int lo[E], back[E];           // places of the departure and of the reversed departure
        T r[E], phi[E], L[E];
        bool far = false;
#pragma unroll
        for (int k = 0; k < E; ++k) {
            if (!has(k)) break;
            c[k] *= sc;
            far |= !below(c[k], n);
        }
        int m[E];
        if (!__any_sync(0xffffffffu, far)) {
#pragma unroll
            for (int k = 0; k < E; ++k) {
            if (!has(k)) break;
                const T f = trunc(c[k]);
                m[k] = (int)f;
                r[k] = c[k] - f;
            }
        } else {   // a period or more somewhere, or a number that cannot be used
#pragma unroll
            for (int k = 0; k < E; ++k) {
            if (!has(k)) break;
                if (!(fabs(c[k]) < T(1073741824.0))) {
                    bad = true;
                    c[k] = T(0);
                }
                const T f = trunc(c[k]);
                m[k] = (int)f % n;
                r[k] = c[k] - f;
            }
        }
#pragma unroll
        for (int k = 0; k < E; ++k) {
            if (!has(k)) break;
            const int d = m[k] * step;
            lo[k] = line[k] + wrap3(pos[k] - d - (positive(r[k]) ? step : 0), period);
            back[k] = LB + line[k] + wrap3(pos[k] + d - (positive(-r[k]) ? step : 0), period);
            phi[k] = v[k];
        }
        T *const dst = out + q0;
        const int climit = limit;
        __syncthreads();   // the previous tile's delta has been read
#pragma unroll
        for (int k = 0; k < E; ++k)
            if (has(k)) put(0, k, phi[k]);
        if (b + (int)gridDim.x < tiles) load(b + gridDim.x);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < E; ++k) {                                     // L_U[Phi]
            if (!has(k)) break;
            const T a = lds(lo[k]), d = lds(lo[k] + step);
            L[k] = a + ((positive(r[k]) ? T(1) : T(0)) - r[k]) * (d - a);
        }
#pragma unroll
        for (int k = 0; k < E; ++k)
            if (has(k)) put(LB, k, L[k]);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < E; ++k) {                                     // delta = Phi - L_{-U}[L_U[Phi]]
            if (!has(k)) break;
            const T a = lds(back[k]), d = lds(back[k] + step);
            phi[k] -= a + ((positive(-r[k]) ? T(1) : T(0)) + r[k]) * (d - a);
        }
#pragma unroll
        for (int k = 0; k < E; ++k)
            if (has(k)) put(0, k, phi[k]);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < E; ++k) {                                     // departure-cell correction
            if (!has(k)) break;
            const T a = lds(lo[k]), d = lds(lo[k] + step);
            const T dj = positive(r[k]) ? d : a;
            const T du = positive(-r[k]) ? d : a;                             // r = 0: the cell itself
            const T res = L[k] + dj * T(0.5) + (T(1) + fabs(r[k])) * T(1.0 / 6.0) * (du - dj);
            if (k * NT < climit) dst[k * hop] = res;
        }
    }
    flag_cfl(g.status, bad);
}

template <typename T, int AX, int LW, int NT, bool PART>
cudaError_t go_sweep(T *dst, const T *src, const T *vel, const WideGeo &g, int rows, unsigned tiles, cudaStream_t st)
{
    // at most NT kSweepCells cells and their repeated elements, in two arrays
    constexpr size_t cap = 2 * sizeof(T) * (size_t)(NT * kSweepCells + 1 + (AX == 0 ? 256 : 1 << LW));
    static ResidencyCache cache;
    Residency res;
    const cudaError_t e = residency(cache, k_wide_sweep<T, AX, LW, NT, PART>, NT, cap, false, res);
    if (e != cudaSuccess) return e;
    const size_t lines = AX == 0 ? (size_t)rows : (size_t)1 << LW;
    const size_t smem = 2 * sizeof(T) * (lines * (size_t)(g.n[AX] + 1) + 1);
    const unsigned grid = std::min(tiles, (unsigned)(res.sms * res.per_sm));
    k_wide_sweep<T, AX, LW, NT, PART><<<grid, NT, smem, st>>>(dst, src, vel, g, T(g.s[AX]), rows, (int)tiles);
    return cudaGetLastError();
}

template <typename T, int AX, int LW, int NT>
cudaError_t sweep_tiles(T *dst, const T *src, const T *vel, const WideGeo &g, int rows, unsigned tiles, cudaStream_t st)
{
    if constexpr (sizeof(T) == 8) {
        const int64_t count = AX == 0 ? (int64_t)rows * g.n[0] : (int64_t)g.n[AX] << LW;
        if (count <= NT * (kSweepCells - 1)) return go_sweep<T, AX, LW, NT, true>(dst, src, vel, g, rows, tiles, st);
    }
    return go_sweep<T, AX, LW, NT, false>(dst, src, vel, g, rows, tiles, st);
}

// The fused sweep, with 512 threads (2048 cells); lines over 256 cells along y or
// z take 1024, where 2048 cells would leave column blocks of fewer than 32
// bytes, and lines of at most 32 cells 256.  False when a line has more than
// 4096 cells or the blocks do not fit a grid.
template <typename T, int AX>
bool sweep_fused(T *dst, const T *src, const T *vel, const WideGeo &g, cudaStream_t st, cudaError_t &e)
{
    const int n = g.n[AX];
    if (n > 1024 * kSweepCells) return false;
    const int64_t lines = g.ncell / n;
    // Few tiles in double precision, which the FP64 pipes bound: smaller ones, over all
    // SMs (16^3: two tiles of 128 rows and 16 column blocks, 51.2 us a step of each order,
    // now 18.5; a 512 x 300 plane 72.2, now 34.8).
    const DevCtx *const ctx = sizeof(T) == 8 ? ctx_get() : nullptr;
    const int sms = ctx ? ctx->num_sms : 0;
    if constexpr (AX == 0) {
        const int nt = n > 512 * kSweepCells ? 1024 : 512;
        int rows = (int)std::min<int64_t>(std::min(256, nt * kSweepCells / n), lines);
        if ((lines + rows - 1) / rows * 2 <= sms) rows = (int)((lines + sms - 1) / sms);
        const int64_t blocks = (lines + rows - 1) / rows;
        if (blocks > 0x7fffffff) return false;
        e = nt == 1024 ? sweep_tiles<T, 0, 0, 1024>(dst, src, vel, g, rows, (unsigned)blocks, st)
                       : sweep_tiles<T, 0, 0, 512>(dst, src, vel, g, rows, (unsigned)blocks, st);
    } else {
        int lw = n <= 64 ? 5 : n <= 128 ? 4 : n <= 512 ? 3 : n <= 1024 ? 2 : n <= 2048 ? 1 : 0;
        auto tiles = [&] { return (((int64_t)g.n[0] + (1 << lw) - 1) >> lw) * (lines / g.n[0]); };
        while (lw > 1 && tiles() * 2 <= sms) --lw;   // 16 bytes of a row at least
        const int64_t blocks = tiles();
        if (blocks > 0x7fffffff) return false;
        const unsigned b = (unsigned)blocks;
        switch (lw) {
        case 5: e = n <= 32 ? sweep_tiles<T, AX, 5, 256>(dst, src, vel, g, 0, b, st)
                            : sweep_tiles<T, AX, 5, 512>(dst, src, vel, g, 0, b, st); break;
        case 4: e = sweep_tiles<T, AX, 4, 512>(dst, src, vel, g, 0, b, st); break;
        case 3: e = n <= 256 ? sweep_tiles<T, AX, 3, 512>(dst, src, vel, g, 0, b, st)
                             : sweep_tiles<T, AX, 3, 1024>(dst, src, vel, g, 0, b, st); break;
        case 2: e = sweep_tiles<T, AX, 2, 1024>(dst, src, vel, g, 0, b, st); break;
        case 1: e = sweep_tiles<T, AX, 1, 1024>(dst, src, vel, g, 0, b, st); break;
        default: e = sweep_tiles<T, AX, 0, 1024>(dst, src, vel, g, 0, b, st); break;
        }
    }
    return true;
}

template <typename T, int NDIM, int AX, int EPI>
cudaError_t interp(T *out, const T *src, const T *vel, const T *aux0, const T *aux1, const WideGeo &g, int dir,
                   cudaStream_t st)
{
    // (FP64 gathers wait on the FP64 pipe: 256 x 256 x 128 FEC 1121 us with 64-bit indices, 1145 with 32)
    if (sizeof(T) == 4 && g.ncell <= (int64_t)UINT32_MAX)
        k_wide_interp<T, std::conditional_t<sizeof(T) == 4, unsigned, int64_t>, NDIM, AX, EPI>
            <<<wide_grid(g), kWideBlock, 0, st>>>(out, src, vel, aux0, aux1, g, dir);
    else
        k_wide_interp<T, int64_t, NDIM, AX, EPI><<<wide_grid(g), kWideBlock, 0, st>>>(out, src, vel, aux0, aux1, g, dir);
    return cudaGetLastError();
}

// One CEC sweep: fused on whole lines when they fit in shared memory, else the
// three gathers through the workspace fields w0 (L_U[Phi]) and w1 (delta).
template <typename T, int AX>
cudaError_t sweep(T *dst, const T *src, const T *vel, T *w0, T *w1, const WideGeo &g, cudaStream_t st)
{
    cudaError_t e = cudaSuccess;
    if (sweep_fused<T, AX>(dst, src, vel, g, st, e)) return e;
    e = interp<T, 3, AX, EPI_NONE>(w0, src, vel, nullptr, nullptr, g, +1, st);                        // L_U[Phi]
    if (e == cudaSuccess) e = interp<T, 3, AX, EPI_DELTA>(w1, w0, vel, src, nullptr, g, -1, st);       // delta
    if (e != cudaSuccess) return e;
    k_wide_cec<T, AX><<<wide_grid(g), kWideBlock, 0, st>>>(dst, w0, w1, vel, g);
    return cudaGetLastError();
}

template <typename T, int NDIM>
cudaError_t unsplit(int scheme, T *out, const T *in, const T *vel, T *w0, T *w1, const WideGeo &g, cudaStream_t st)
{
    if (scheme == 0) return interp<T, NDIM, -1, EPI_NONE>(out, in, vel, nullptr, nullptr, g, +1, st);
    cudaError_t e = interp<T, NDIM, -1, EPI_NONE>(w0, in, vel, nullptr, nullptr, g, +1, st);           // L_U[Phi]
    if (e != cudaSuccess) return e;
    if (scheme == 1) return interp<T, NDIM, -1, EPI_FEC>(out, w0, vel, in, w0, g, -1, st);
    e = interp<T, NDIM, -1, EPI_BEC_IN>(w1, w0, vel, in, nullptr, g, -1, st);                           // Phi + delta/2
    if (e != cudaSuccess) return e;
    return interp<T, NDIM, -1, EPI_NONE>(out, w1, vel, nullptr, nullptr, g, +1, st);
}

template <typename T>
cudaError_t run(int scheme, const void *in_v, void *out_v, const void *vel_v, int ndim, const WideGeo &g, int parity,
                void *work, cudaStream_t st)
{
    const T *in = static_cast<const T *>(in_v), *vel = static_cast<const T *>(vel_v);
    T *out = static_cast<T *>(out_v);
    const size_t fb = wide_field_bytes(g.ncell, sizeof(T));
    // the scheme's workspace fields (wide_fields of them; none for CIR, whose
    // workspace may be NULL)
    T *w[4] = {nullptr, nullptr, nullptr, nullptr};
    for (int k = 0; k < wide_fields(scheme, ndim); ++k) w[k] = reinterpret_cast<T *>(static_cast<char *>(work) + k * fb);
    if (scheme != 3) return ndim == 3 ? unsplit<T, 3>(scheme, out, in, vel, w[0], w[1], g, st)
                                      : unsplit<T, 2>(scheme, out, in, vel, w[0], w[1], g, st);
    // split CEC: in -> w2 (-> w3) -> out
    const T *src = in;
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < ndim && e == cudaSuccess; ++k) {
        const int axis = (parity & 1) ? ndim - 1 - k : k;
        T *dst = k == ndim - 1 ? out : w[2 + (k & 1)];
        e = axis == 0 ? sweep<T, 0>(dst, src, vel, w[0], w[1], g, st)
                      : (axis == 1 ? sweep<T, 1>(dst, src, vel, w[0], w[1], g, st)
                                   : sweep<T, 2>(dst, src, vel, w[0], w[1], g, st));
        src = dst;
    }
    return e;
}

}  // namespace

size_t wide_field_bytes(int64_t ncell, size_t elem) { return ((size_t)ncell * elem + 255) & ~(size_t)255; }

int wide_fields(int scheme, int ndim)
{
    switch (scheme) {
    case 0: return 0;
    case 1: return 1;
    case 2: return 2;
    default: return ndim == 3 ? 4 : 3;
    }
}

cudaError_t launch_wide(int dtype, int scheme, const void *in, void *out, const void *vel, int ndim,
                        const int64_t dims[3], const double s[3], int parity, void *work, unsigned *status,
                        cudaStream_t st)
{
    WideGeo g;
    for (int d = 0; d < 3; ++d) {
        g.n[d] = (int)dims[d];
        g.s[d] = d < ndim ? s[d] : 0.0;
    }
    g.ncell = dims[0] * dims[1] * dims[2];
    g.status = status;
    return dtype == 1 ? run<double>(scheme, in, out, vel, ndim, g, parity, work, st)
                      : run<float>(scheme, in, out, vel, ndim, g, parity, work, st);
}

}  // namespace sl
