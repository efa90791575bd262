// k_split.cu -- fused directionally split third-order step (SL_CEC) in FP32 on
// planes and on 3D grids of fewer than 8 planes, and the generic batched step
// (k_cec_fast.cu and k_split64.cu serve the rest).
//
// One kernel performs the three 1D CEC sweeps of a time step (Sec. 2 last
// paragraph, Sec. 5 eqs. split:1-2; per-axis coefficients of eq.
// intro:CECcoef) with a single HBM read of Phi and u and a single write of
// the result.  Each 1D sweep reads Phi three cells and u two cells away from
// its output, so the staged plane tiles carry a halo of 3 (Phi) and 2 (u).
//
//  - order x,y,z (even step): per plane, the x sweep runs on the staged tile
//    (rows widened by the y halo) into shared memory, the y sweep reads it and
//    feeds, per column, a register window that performs the z sweep three
//    planes behind the plane being loaded.
//  - order z,y,x (odd step): the z sweep runs first in register windows over
//    the halo-widened columns and writes each finished plane to shared
//    memory, where the y and x sweeps follow.
//
// Loads are 16-byte cp.async copies of whole aligned rows (x staged over
// [-4, TX+4)), double-buffered one plane ahead; periodic wrap-around is folded
// into per-thread source offsets computed once per work item.
#include <cmath>

#include "sl_internal.h"

namespace sl {
namespace {

template <int TX, int TY>
struct Shape {
    static constexpr int HW = TX + 8;                    // staged x in [-4, TX+4)
    static constexpr int PW = HW + 4;   // row stride
    static constexpr int PH = TY + 6;                    // staged y in [-3, TY+3)
};

// N consecutive elements from 16-byte aligned shared memory.
template <int N>
__device__ __forceinline__ void lds_vec(const float *src, float (&dst)[N])
{
    static_assert(N % 4 == 0, "");
#pragma unroll
    for (int i = 0; i < N / 4; ++i) {
        const float4 v = reinterpret_cast<const float4 *>(src)[i];
        dst[4 * i] = v.x; dst[4 * i + 1] = v.y; dst[4 * i + 2] = v.z; dst[4 * i + 3] = v.w;
    }
}

template <int N>
__device__ __forceinline__ void sts_vec(float *dst, const float (&src)[N])
{
#pragma unroll
    for (int i = 0; i < N / 4; ++i)
        reinterpret_cast<float4 *>(dst)[i] = make_float4(src[4 * i], src[4 * i + 1], src[4 * i + 2], src[4 * i + 3]);
}

// Stages a rectangle of rows [r0, r0+NR) (relative to the tile origin) and
// columns [c0, c0 + NC) of one plane into shared memory with row stride LD.
// VEC: 16-byte copies (NC and nx multiples of V, so every copy lies inside one
// period).  Otherwise 4-byte copies of whole shared rows (all LD columns: the
// destination of a thread's k-th copy is then tid + k NT elements in, with no
// row arithmetic).  The periodic wrap is in per-thread source offsets, computed
// once per work item; wrapping every element of every plane again took most of
// the time on grids whose rows are no multiple of 16 bytes (187 x 150 x 131,
// x,y,z / z,y,x: 123 / 173 us before, 55 / 79 after, when this kernel served it).
template <int NT, int NR, int NC, int LD, bool VEC>
struct Stager {
    static constexpr int V = VEC ? 16 / sizeof(float) : 1;
    static constexpr int CPR = VEC ? NC / V : LD;
    static constexpr int N = NR * CPR;
    static constexpr int K = (N + NT - 1) / NT;
    int off[K];

    __device__ __forceinline__ void setup(int tid, int x0, int y0, int r0, int c0, int nx, int ny)
    {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int idx = tid + k * NT;
            if (idx < N) {
                const int row = idx / CPR, cc = idx - (idx / CPR) * CPR;
                const int gy = wrapi(y0 + r0 + row, ny);
                const int gx = wrapi(x0 + c0 + cc * V, nx);
                off[k] = gy * nx + gx;
            } else {
                off[k] = -1;
            }
        }
    }

    __device__ __forceinline__ void issue(int tid, float *dst, const float *src) const
    {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int idx = tid + k * NT;
            if (off[k] < 0) continue;
            if constexpr (VEC) {
                const int row = idx / CPR, cc = idx - (idx / CPR) * CPR;
                cp_async16(dst + row * LD + cc * V, src + off[k]);
            } else {
                cp_async_elem(dst + idx, src + off[k]);
            }
        }
    }
};

__device__ __forceinline__ void decode_item(int item, const Geo &g, int TX, int TY, int &x0, int &y0, int &z0,
                                            int &z1)
{
    const int tx = item % g.tiles_x;
    const int rest = item / g.tiles_x;
    const int ty = rest % g.tiles_y;
    const int cz = rest / g.tiles_y;
    x0 = tx * TX;
    y0 = ty * TY;
    z0 = cz * g.tz;
    z1 = min(z0 + g.tz, g.nz);
}

// ============================================================ order x, y, z
template <int TX, int TY, bool HAS_Z, bool VEC>
struct XYZ {
    using S = Shape<TX, TY>;
    static constexpr int RX = 8, RY = 4;
    static constexpr int NT = TX * (TY / RY);
    static constexpr int NB = 2;
    static constexpr int SZ_PHI = S::PH * S::PW;
    static constexpr int SZ_CY = (TY + 4) * TX;
    static constexpr int SZ_CZ = HAS_Z ? TY * TX : 0;
    static constexpr int SZ_S1 = S::PH * TX;
    static constexpr size_t smem() { return sizeof(float) * (size_t)(NB * (2 * SZ_PHI + SZ_CY + SZ_CZ) + SZ_S1); }
};

template <int TX, int TY, bool HAS_Z, bool VEC>
__device__ __forceinline__ void xyz_item(const Geo &g, int item, const float *__restrict__ in, float *__restrict__ out,
                                         const float *__restrict__ vel, unsigned char *smem_raw, bool &bad)
{
    using K = XYZ<TX, TY, HAS_Z, VEC>;
    using S = typename K::S;
    constexpr int RX = K::RX, RY = K::RY, NT = K::NT, NB = K::NB;
    float *sPhi = reinterpret_cast<float *>(smem_raw);
    float *sCx = sPhi + NB * K::SZ_PHI;
    float *sCy = sCx + NB * K::SZ_PHI;
    float *sCz = sCy + NB * K::SZ_CY;
    float *sS1 = sCz + NB * K::SZ_CZ;

    const int tid = threadIdx.x;
    const float sx = (float)g.sx, sy = (float)g.sy, sz = (float)g.sz;

    Stager<NT, S::PH, S::HW, S::PW, VEC> stPhi;     // Phi and u_x: rows [-3,TY+3), cols [-4,TX+4)
    Stager<NT, TY + 4, TX, TX, VEC> stCy;           // u_y: rows [-2,TY+2), cols [0,TX)
    Stager<NT, TY, TX, TX, VEC> stCz;               // u_z: rows [0,TY), cols [0,TX)

    int x0, y0, z0, z1;
    decode_item(item, g, TX, TY, x0, y0, z0, z1);
    stPhi.setup(tid, x0, y0, -3, -4, g.nx, g.ny);
    stCy.setup(tid, x0, y0, -2, 0, g.nx, g.ny);
    if constexpr (HAS_Z) stCz.setup(tid, x0, y0, 0, 0, g.nx, g.ny);

    const int pfirst = HAS_Z ? z0 - 3 : 0;
    const int plast = HAS_Z ? z1 + 2 : 0;
    auto issue = [&](int p, int slot) {
        const int64_t base = (int64_t)wrapi(p, g.nz) * g.plane;
        stPhi.issue(tid, sPhi + slot * K::SZ_PHI, in + base);
        stPhi.issue(tid, sCx + slot * K::SZ_PHI, vel + base);
        stCy.issue(tid, sCy + slot * K::SZ_CY, vel + g.ncell + base);
        if constexpr (HAS_Z) {
            const int64_t bz = (int64_t)wrapi(p - 1, g.nz) * g.plane;
            stCz.issue(tid, sCz + slot * K::SZ_CZ, vel + 2 * g.ncell + bz);
        }
        cp_async_commit();
    };

    const int cx = tid % TX, yr = (tid / TX) * RY;     // y-sweep run / z columns of this thread
    ZWin win[RY];
#pragma unroll
    for (int i = 0; i < RY; ++i) win[i].init();

    issue(pfirst, 0);
    for (int p = pfirst; p <= plast; ++p) {
        const int slot = (p - pfirst) & 1;
        cp_async_wait_all();
        __syncthreads();
        if (p < plast) issue(p + 1, slot ^ 1);

        // ---- x sweep: rows [-3, TY+3) x cols [0, TX) -> sS1
        const float *phiP = sPhi + slot * K::SZ_PHI;
        const float *cxP = sCx + slot * K::SZ_PHI;
        constexpr int XR = TX / RX;
        for (int r = tid; r < S::PH * XR; r += NT) {
            const int row = r / XR, xr = (r - (r / XR) * XR) * RX;
            float blk[RX + 8];
            lds_vec<RX + 8>(phiP + row * S::PW + xr, blk);
            float pv[RX + 6];
#pragma unroll
            for (int k = 0; k < RX + 6; ++k) pv[k] = blk[k + 1];
            lds_vec<RX + 8>(cxP + row * S::PW + xr, blk);
            float cv[RX + 4];
#pragma unroll
            for (int k = 0; k < RX + 4; ++k) cv[k] = blk[k + 2] * sx;
#pragma unroll
            for (int k = 2; k < RX + 2; ++k) bad |= fabs(cv[k]) > 1.f;
            float o[RX];
            cec_line<RX>(pv, cv, o);
            sts_vec<RX>(sS1 + row * TX + xr, o);
        }
        __syncthreads();

        // ---- y sweep of this thread's run, then z windows
        const float *cyP = sCy + slot * K::SZ_CY;
        float pv[RY + 6];
#pragma unroll
        for (int k = 0; k < RY + 6; ++k) pv[k] = sS1[(yr + k) * TX + cx];
        float cv[RY + 4];
#pragma unroll
        for (int k = 0; k < RY + 4; ++k) cv[k] = cyP[(yr + k) * TX + cx] * sy;
#pragma unroll
        for (int k = 2; k < RY + 2; ++k) bad |= fabs(cv[k]) > 1.f;
        float o[RY];
        cec_line<RY>(pv, cv, o);
        const int gx = x0 + cx;
        if constexpr (HAS_Z) {
            const float *czP = sCz + slot * K::SZ_CZ;
            const int kz = p - 3;
#pragma unroll
            for (int i = 0; i < RY; ++i) {
                const float c = czP[(yr + i) * TX + cx] * sz;
                bad |= fabs(c) > 1.f;
                const float v = win[i].push(o[i], c);
                const int gy = y0 + yr + i;
                if (kz >= z0 && gx < g.nx && gy < g.ny) out[(int64_t)kz * g.plane + (int64_t)gy * g.nx + gx] = v;
            }
        } else {
#pragma unroll
            for (int i = 0; i < RY; ++i) {
                const int gy = y0 + yr + i;
                if (gx < g.nx && gy < g.ny) out[(int64_t)gy * g.nx + gx] = o[i];
            }
        }
    }
    __syncthreads();   // shared buffers are reused by the next item
}

template <int TX, int TY, bool HAS_Z, bool VEC>
__global__ void __launch_bounds__(XYZ<TX, TY, HAS_Z, VEC>::NT)
k_cec_xyz(const float *__restrict__ in, float *__restrict__ out, const float *__restrict__ vel, Geo g, int64_t fin,
          int64_t fout)
{
    in += (int64_t)blockIdx.y * fin;   // field of this CTA (FieldSet)
    out += (int64_t)blockIdx.y * fout;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nitems = g.tiles_x * g.tiles_y * g.chunks;
    bool bad = false;
    for (int item = blockIdx.x; item < nitems; item += gridDim.x)
        xyz_item<TX, TY, HAS_Z, VEC>(g, item, in, out, vel, smem_raw, bad);
    flag_cfl(g.status, bad);
}

// ============================================================ order z, y, x
template <int TX, int TY, bool HAS_Z, bool VEC>
struct ZYX {
    using S = Shape<TX, TY>;
    static constexpr int RX = 4, RY = 4;
    static constexpr int NT = 256;
    static constexpr int NB = 2;
    static constexpr int NZC = (TX + 6) * (TY + 6);           // z-swept columns
    static constexpr int NCOL = HAS_Z ? (NZC + NT - 1) / NT : 1;
    static constexpr int SZ_PHI = S::PH * S::PW;
    static constexpr int SZ_CZ = HAS_Z ? S::PH * S::PW : 0;
    static constexpr int SZ_Z = HAS_Z ? S::PH * S::PW : 0;
    static constexpr int SZ_CY = (TY + 4) * S::PW;
    static constexpr int SZ_S2 = TY * S::PW;
    static constexpr int SZ_CX = TY * S::PW;
    static constexpr size_t smem()
    {
        return sizeof(float) * (size_t)(NB * (SZ_PHI + SZ_CZ + SZ_CY + SZ_CX) + SZ_Z + SZ_S2);
    }
};

template <int TX, int TY, bool HAS_Z, bool VEC>
__device__ __forceinline__ void zyx_item(const Geo &g, int item, const float *__restrict__ in, float *__restrict__ out,
                                         const float *__restrict__ vel, unsigned char *smem_raw, bool &bad)
{
    using K = ZYX<TX, TY, HAS_Z, VEC>;
    using S = typename K::S;
    constexpr int RX = K::RX, RY = K::RY, NT = K::NT, NB = K::NB, NCOL = K::NCOL;
    float *sPhi = reinterpret_cast<float *>(smem_raw);
    float *sCz = sPhi + NB * K::SZ_PHI;
    float *sCy = sCz + NB * K::SZ_CZ;
    float *sCx = sCy + NB * K::SZ_CY;
    float *sZ = sCx + NB * K::SZ_CX;
    float *sS2 = sZ + K::SZ_Z;

    const int tid = threadIdx.x;
    const float sx = (float)g.sx, sy = (float)g.sy, sz = (float)g.sz;

    Stager<NT, S::PH, S::HW, S::PW, VEC> stPhi;     // Phi, u_z: rows [-3,TY+3), cols [-4,TX+4)
    Stager<NT, TY + 4, S::HW, S::PW, VEC> stCy;     // u_y: rows [-2,TY+2)
    Stager<NT, TY, S::HW, S::PW, VEC> stCx;         // u_x: rows [0,TY)

    int x0, y0, z0, z1;
    decode_item(item, g, TX, TY, x0, y0, z0, z1);
    stPhi.setup(tid, x0, y0, -3, -4, g.nx, g.ny);
    stCy.setup(tid, x0, y0, -2, -4, g.nx, g.ny);
    stCx.setup(tid, x0, y0, 0, -4, g.nx, g.ny);

    const int pfirst = HAS_Z ? z0 - 3 : 0;
    const int plast = HAS_Z ? z1 + 2 : 0;
    auto issue = [&](int p, int slot) {
        const int64_t base = (int64_t)wrapi(p, g.nz) * g.plane;
        stPhi.issue(tid, sPhi + slot * K::SZ_PHI, in + base);
        int64_t bk = base;
        if constexpr (HAS_Z) {
            const int64_t bz = (int64_t)wrapi(p - 1, g.nz) * g.plane;
            stPhi.issue(tid, sCz + slot * K::SZ_CZ, vel + 2 * g.ncell + bz);
            bk = (int64_t)wrapi(p - 3, g.nz) * g.plane;
        }
        stCy.issue(tid, sCy + slot * K::SZ_CY, vel + g.ncell + bk);
        stCx.issue(tid, sCx + slot * K::SZ_CX, vel + bk);
        cp_async_commit();
    };

    ZWin win[NCOL];
#pragma unroll
    for (int j = 0; j < NCOL; ++j) win[j].init();

    issue(pfirst, 0);
    for (int p = pfirst; p <= plast; ++p) {
        const int slot = (p - pfirst) & 1;
        cp_async_wait_all();
        __syncthreads();
        if (p < plast) issue(p + 1, slot ^ 1);

        const float *zsrc = sPhi + slot * K::SZ_PHI;
        int kz = 0;
        if constexpr (HAS_Z) {
            // ---- z sweep over columns x in [-3, TX+3), y in [-3, TY+3)
            const float *czP = sCz + slot * K::SZ_CZ;
#pragma unroll
            for (int j = 0; j < NCOL; ++j) {
                const int r = tid + j * NT;
                if (r < K::NZC) {
                    const int row = r / (TX + 6), col = r - (r / (TX + 6)) * (TX + 6) + 1;
                    const float c = czP[row * S::PW + col] * sz;
                    const float v = win[j].push(zsrc[row * S::PW + col], c);
                    sZ[row * S::PW + col] = v;
                    if (row >= 3 && row < TY + 3 && col >= 4 && col < TX + 4) bad |= fabs(c) > 1.f;
                }
            }
            __syncthreads();
            kz = p - 3;
            if (kz < z0) continue;
            zsrc = sZ;
        }

        // ---- y sweep: columns x in [-3, TX+3), rows [0, TY) -> sS2
        const float *cyP = sCy + slot * K::SZ_CY;
        for (int r = tid; r < (TX + 6) * (TY / RY); r += NT) {
            const int col = r % (TX + 6) + 1, yr = (r / (TX + 6)) * RY;
            float pv[RY + 6];
#pragma unroll
            for (int k = 0; k < RY + 6; ++k) pv[k] = zsrc[(yr + k) * S::PW + col];
            float cv[RY + 4];
#pragma unroll
            for (int k = 0; k < RY + 4; ++k) cv[k] = cyP[(yr + k) * S::PW + col] * sy;
            if (col >= 4 && col < TX + 4) {
#pragma unroll
                for (int k = 2; k < RY + 2; ++k) bad |= fabs(cv[k]) > 1.f;
            }
            float o[RY];
            cec_line<RY>(pv, cv, o);
#pragma unroll
            for (int i = 0; i < RY; ++i) sS2[(yr + i) * S::PW + col] = o[i];
        }
        __syncthreads();

        // ---- x sweep: rows [0, TY), cols [0, TX) -> global plane kz
        const float *cxP = sCx + slot * K::SZ_CX;
        constexpr int XR = TX / RX;
        for (int r = tid; r < TY * XR; r += NT) {
            const int row = r / XR, xr = (r - (r / XR) * XR) * RX;
            float blk[RX + 8];
            lds_vec<RX + 8>(sS2 + row * S::PW + xr, blk);
            float pv[RX + 6];
#pragma unroll
            for (int k = 0; k < RX + 6; ++k) pv[k] = blk[k + 1];
            lds_vec<RX + 8>(cxP + row * S::PW + xr, blk);
            float cv[RX + 4];
#pragma unroll
            for (int k = 0; k < RX + 4; ++k) cv[k] = blk[k + 2] * sx;
#pragma unroll
            for (int k = 2; k < RX + 2; ++k) bad |= fabs(cv[k]) > 1.f;
            float o[RX];
            cec_line<RX>(pv, cv, o);
            const int gy = y0 + row;
            if (gy < g.ny) {
                float *dst = out + (int64_t)kz * g.plane + (int64_t)gy * g.nx + x0 + xr;
                if (VEC && x0 + xr + RX <= g.nx) {
                    reinterpret_cast<float4 *>(dst)[0] = make_float4(o[0], o[1], o[2], o[3]);
                } else {
#pragma unroll
                    for (int i = 0; i < RX; ++i)
                        if (x0 + xr + i < g.nx) dst[i] = o[i];
                }
            }
        }
    }
    __syncthreads();
}

template <int TX, int TY, bool HAS_Z, bool VEC>
__global__ void __launch_bounds__(256)
k_cec_zyx(const float *__restrict__ in, float *__restrict__ out, const float *__restrict__ vel, Geo g, int64_t fin,
          int64_t fout)
{
    in += (int64_t)blockIdx.y * fin;   // field of this CTA (FieldSet)
    out += (int64_t)blockIdx.y * fout;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nitems = g.tiles_x * g.tiles_y * g.chunks;
    bool bad = false;
    for (int item = blockIdx.x; item < nitems; item += gridDim.x)
        zyx_item<TX, TY, HAS_Z, VEC>(g, item, in, out, vel, smem_raw, bad);
    flag_cfl(g.status, bad);
}

template <int TX, int TY, bool HAS_Z, bool VEC>
cudaError_t dispatch_order(int parity, const Geo &g, int grid, const void *in, void *out, const void *vel,
                           const FieldSet &fs, cudaStream_t st)
{
    const float *i = static_cast<const float *>(in);
    const float *v = static_cast<const float *>(vel);
    float *o = static_cast<float *>(out);
    if ((parity & 1) == 0) {
        using K = XYZ<TX, TY, HAS_Z, VEC>;
        auto kern = k_cec_xyz<TX, TY, HAS_Z, VEC>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::smem());
        if (e != cudaSuccess) return e;
        const int nitems = g.tiles_x * g.tiles_y * g.chunks;
        const int gr = grid > 0 && grid < nitems ? grid : nitems;
        kern<<<dim3(gr, fs.n), K::NT, K::smem(), st>>>(i, o, v, g, fs.fin, fs.fout);
    } else {
        using K = ZYX<TX, TY / 2, HAS_Z, VEC>;
        auto kern = k_cec_zyx<TX, TY / 2, HAS_Z, VEC>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::smem());
        if (e != cudaSuccess) return e;
        Geo g2 = g;
        g2.tiles_y = (g.ny + TY / 2 - 1) / (TY / 2);
        const int nitems = g2.tiles_x * g2.tiles_y * g2.chunks;
        const int gr = grid > 0 && grid < nitems ? grid : nitems;
        kern<<<dim3(gr, fs.n), K::NT, K::smem(), st>>>(i, o, v, g2, fs.fin, fs.fout);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------ batched
// Persistent CTAs take (instance, tile, z-chunk) items from a device counter
// until the batch is exhausted; every item is the same fused step as above.
template <int TX, int TY, int PAR>
__global__ void __launch_bounds__(256)
k_cec_batched(const BatchRec *__restrict__ recs, int ninst, int nitems, unsigned *counter, unsigned *status)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_item;
    bool bad = false;
    for (;;) {
        if (threadIdx.x == 0) s_item = (int)atomicAdd(counter, 1u);
        __syncthreads();
        const int it = s_item;
        __syncthreads();
        if (it >= nitems) break;
        int lo = 0, hi = ninst - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (recs[mid].item0[PAR] <= it) lo = mid; else hi = mid - 1;
        }
        const BatchRec &r = recs[lo];
        const Geo g = r.g[PAR];
        const float *in = static_cast<const float *>(PAR ? r.b : r.a);
        float *out = static_cast<float *>(PAR ? r.a : r.b);
        const float *vel = static_cast<const float *>(r.vel);
        if constexpr (PAR == 0)
            xyz_item<TX, TY, true, true>(g, it - r.item0[0], in, out, vel, smem_raw, bad);
        else
            zyx_item<TX, TY / 2, true, true>(g, it - r.item0[1], in, out, vel, smem_raw, bad);
    }
    flag_cfl(status, bad);
}

}  // namespace

int default_tz(int dtype, int ndim, const int64_t dims[3])
{
    (void)dtype;
    if (ndim == 2) return 1;
    // enough z chunks to give every SM two CTAs, but chunks of >= 16 planes
    const int64_t nz = dims[2];
    const int64_t cols = ((dims[0] + 31) / 32) * ((dims[1] + 31) / 32);
    int tz = (int)nz;
    const int64_t want = 2 * 152;
    while (tz > 16 && cols * ((nz + tz - 1) / tz) < want) tz = (tz + 1) / 2;
    return tz < 1 ? 1 : tz;
}

int64_t plan_ctas(int64_t tiles, int64_t nz, int warm, double alone, int per_sm, int sms, int fields)
{
    auto plane = [&](int64_t ctas) {
        const int64_t k = (ctas * fields + sms - 1) / sms;   // CTAs of the busiest SM
        return k <= 1 ? alone : 0.5 * (double)k;
    };
    const int64_t total = tiles * nz, all = (int64_t)per_sm * sms / fields;
    int64_t best = all < 1 ? 1 : (all < total ? all : total);
    const double share = (double)total / (double)best;
    double cost = (share + warm * (2.0 + floor(share / (double)nz))) * plane(best);
    for (int64_t c = 1; c <= nz && tiles * c <= all; ++c) {
        const double t = (double)((nz + c - 1) / c + warm) * plane(tiles * c);
        if (t < cost) {
            cost = t;
            best = tiles * c;
        }
    }
    return best;
}

cudaError_t launch_split_cec(int dtype, const void *in, void *out, const void *vel, int ndim,
                             const int64_t dims[3], const double s[3], int parity, Launch lc,
                             unsigned *status, cudaStream_t st, FieldSet fs)
{
    if (any_eligible(dims, ndim, dtype))
        return launch_cec_any(in, out, vel, dims, s, parity, lc, status, fs, st);
    constexpr int TX = 32;
    Geo g;
    g.nx = (int)dims[0];
    g.ny = (int)dims[1];
    g.nz = ndim == 3 ? (int)dims[2] : 1;
    g.plane = (int64_t)g.nx * g.ny;
    g.ncell = g.plane * g.nz;
    g.sx = s[0];
    g.sy = s[1];
    g.sz = ndim == 3 ? s[2] : 0.0;
    g.status = status;
    g.tz = ndim == 3 ? (lc.tz > 0 ? lc.tz : default_tz(dtype, ndim, dims)) : 1;
    if (g.tz > g.nz) g.tz = g.nz;
    g.chunks = (g.nz + g.tz - 1) / g.tz;
    g.tiles_x = (g.nx + TX - 1) / TX;
    const bool has_z = ndim == 3;
    if (dtype != 0) {   // SL_F64, SL_F32_D64
        g.tz = ndim == 3 && lc.tz > 0 ? g.tz : 0;   // default: equal shares
        return launch_split_cec64(dtype == 2, g, parity, lc, has_z, in, out, vel, fs, st);
    }
    constexpr int TY = 32;
    g.tiles_y = (g.ny + TY - 1) / TY;
    const bool vec = lc.aligned && g.nx % 4 == 0;
    if (has_z)
        return vec ? dispatch_order<TX, TY, true, true>(parity, g, lc.grid, in, out, vel, fs, st)
                   : dispatch_order<TX, TY, true, false>(parity, g, lc.grid, in, out, vel, fs, st);
    return vec ? dispatch_order<TX, TY, false, true>(parity, g, lc.grid, in, out, vel, fs, st)
               : dispatch_order<TX, TY, false, false>(parity, g, lc.grid, in, out, vel, fs, st);
}

size_t batched_smem(int parity)
{
    return parity ? ZYX<32, 16, true, true>::smem() : XYZ<32, 32, true, true>::smem();
}

void batched_tiles(int parity, int &tx, int &ty)
{
    tx = 32;
    ty = parity ? 16 : 32;
}

cudaError_t launch_batched_cec(const BatchRec *dev_recs, int ninst, int nitems, int parity, unsigned *counter,
                               unsigned *status, int grid, cudaStream_t st)
{
    const size_t smem = batched_smem(parity);
    if (parity) {
        auto kern = k_cec_batched<32, 32, 1>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<grid, 256, smem, st>>>(dev_recs, ninst, nitems, counter, status);
    } else {
        auto kern = k_cec_batched<32, 32, 0>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<grid, 256, smem, st>>>(dev_recs, ninst, nitems, counter, status);
    }
    return cudaGetLastError();
}

int batched_blocks_per_sm(int parity)
{
    int nb = 0;
    const size_t smem = batched_smem(parity);
    cudaError_t e;
    if (parity) {
        auto kern = k_cec_batched<32, 32, 1>;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, 256, smem);
    } else {
        auto kern = k_cec_batched<32, 32, 0>;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, 256, smem);
    }
    return e == cudaSuccess && nb > 0 ? nb : 1;
}

}  // namespace sl
