// sl_common.cuh -- device helpers shared by the fused advection kernels.
//
// Geometry of every fused kernel: the grid is cut into TX x TY columns of
// cells in the x-y plane and, in 3D, into chunks of TZ planes along z.  A CTA
// owns one (column tile, z chunk) item and marches along z, staging each x-y
// plane of the inputs (plus a periodic halo) in shared memory with 16-byte
// cp.async copies, so that every input element is read from HBM about once
// and every output element is written once.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace sl {

// ------------------------------------------------------------------ geometry
struct Geo {
    int nx, ny, nz;         // cells per axis
    int64_t plane;          // nx * ny
    int64_t ncell;          // nx * ny * nz
    double sx, sy, sz;      // dt / dx_d: Courant number = u_d * s_d
    int tiles_x, tiles_y;   // column tiles per axis
    int tz;                 // planes per z chunk
    int chunks;             // z chunks
    unsigned *status;       // device status word (SL_DEV_* bits)
};

__host__ __device__ __forceinline__ int wrapi(int v, int n)
{
    int r = v % n;
    return r < 0 ? r + n : r;
}

// ------------------------------------------------------------ async copies
__device__ __forceinline__ unsigned smem_u32(const void *p)
{
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(smem)), "l"(gmem));
}

__device__ __forceinline__ void cp_async4(void *smem, const void *gmem)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_u32(smem)), "l"(gmem));
}

__device__ __forceinline__ void cp_async8(void *smem, const void *gmem)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_u32(smem)), "l"(gmem));
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

template <typename T>
__device__ __forceinline__ void cp_async_elem(T *smem, const T *gmem)
{
    if constexpr (sizeof(T) == 4)
        cp_async4(smem, gmem);
    else
        cp_async8(smem, gmem);
}

// ------------------------------------------- programmatic dependent launch
// A kernel launched with the programmatic-serialisation attribute may start while
// its predecessor in the stream still runs; before it touches anything the
// predecessor reads or writes, every thread waits for the predecessor's end (its
// memory included).  Both are no-ops in a kernel launched without the attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ----------------------------------------------------------- 1D CEC kernels
//
// One directional sweep of the combined scheme (Sec. 2 eqs. intro:FEC,
// intro:BEC, intro:CEC, intro:CECcoef) along a line, for |C| <= 1, with
// s = sgn C, U = |C| and W = 1 - U.  The CIR operator of Sec. 3 is written from
// the upwind neighbour (s = 0: the cell itself),
//   L_j     = Phi_{j-s_j} + W_j (Phi_j - Phi_{j-s_j}),
//   delta_j = Phi_j - L_{-U}[L]_j = (Phi_j - L_j) - U_j (L_{j+s_j} - L_j),
//   CEC_i   = a FEC_i + b BEC_i (3a = 2 - 1/U, b = 1 - a)
//           = L_i + delta_i / 2 + (1 + U_i)/6 (delta_{i-s_i} - delta_i),
// exact algebra on the definitions without 1/U.  Constant fields stay exact
// (every difference is zero), C = +-1 is an exact shift (W = 0) and C = 0
// keeps the cell.  In FP32; k_split64.cu has the forms in double arithmetic.

// GB300 issues about two double operations per clock and SM, comparisons and
// float-to-double conversions included, so double signs, bounds and widenings go
// through the bit patterns.
//
// sgn C (a NaN counts as its sign bit says: every use ends in a NaN anyway)
__device__ __forceinline__ int sgn_bits(double c)
{
    const int hi = __double2hiint(c);
    return ((hi & 0x7fffffff) | __double2loint(c)) == 0 ? 0 : (hi < 0 ? -1 : 1);
}

// |C| > 1 (false for a NaN, like the comparison)
__device__ __forceinline__ bool beyond_one(float c) { return fabsf(c) > 1.f; }
__device__ __forceinline__ bool beyond_one(double c)
{
    const unsigned long long a = (unsigned long long)__double_as_longlong(c) & 0x7fffffffffffffffull;
    return a > 0x3ff0000000000000ull && a <= 0x7ff0000000000000ull;
}

// Exact conversion to the arithmetic type: float to double without the conversion
// instruction for normal numbers and zeros; denormals, infinities and NaN take it.
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v)
{
    const unsigned b = __float_as_uint(v), m = b & 0x7fffffffu;
    if (m - 1u < 0x007fffffu || m >= 0x7f800000u) return (double)v;
    const unsigned hi = (b & 0x80000000u) | (m ? (m >> 3) + (896u << 20) : 0u);
    return __hiloint2double((int)hi, (int)(b << 29));
}
template <typename D, typename T>
__device__ __forceinline__ D to(T v)
{
    if constexpr (sizeof(D) == 8)
        return widen(v);
    else
        return D(v);
}

// by the sign of C: C > 0, C < 0, C == 0
template <typename D, typename V>
__device__ __forceinline__ V by_sign(D C, V pos, V neg, V zero)
{
    if constexpr (sizeof(D) == 8) {
        const int s = sgn_bits(C);
        return s > 0 ? pos : (s < 0 ? neg : zero);
    } else {
        return C > D(0) ? pos : (C < D(0) ? neg : zero);
    }
}

// Outputs o[0..R) of a line segment from p[0..R+6) = Phi at offsets -3..R+2
// and c[0..R+4) = Courant numbers at offsets -2..R+1.
template <int R>
__device__ __forceinline__ void cec_line(const float (&p)[R + 6], const float (&c)[R + 4], float (&o)[R])
{
    float L[R + 4];                  // offsets -2..R+1 (index m <-> offset m-2, Phi at p[m+1])
#pragma unroll
    for (int m = 0; m < R + 4; ++m) {
        const float nb = by_sign(c[m], p[m], p[m + 2], p[m + 1]);
        L[m] = nb + (1.f - fabs(c[m])) * (p[m + 1] - nb);
    }
    float del[R + 2];                // offsets -1..R (index q <-> offset q-1)
#pragma unroll
    for (int q = 0; q < R + 2; ++q) {
        const int m = q + 1;
        const float Ln = by_sign(c[m], L[m + 1], L[m - 1], L[m]);
        del[q] = (p[m + 1] - L[m]) - fabs(c[m]) * (Ln - L[m]);
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int m = i + 2, q = i + 1;
        const float U = fabs(c[m]);
        const float dn = by_sign(c[m], del[q - 1], del[q + 1], del[q]);
        o[i] = L[m] + 0.5f * del[q] + (1.f + U) * (1.f / 6.f) * (dn - del[q]);
    }
}

// Sliding window of the same sweep along z for one column: feed planes in
// order with push(); after plane p is pushed, the result is the value at p - 3.
// State after a push of plane p: Phi at p-1, p; L at p-2, p-1; Courant at p-2,
// p-1; delta at p-3, p-2.
struct ZWin {
    float ph[2];   // Phi at p-2 (ph[0]), p-1 (ph[1])
    float L[2];    // L at p-3, p-2
    float c[2];    // Courant at p-3, p-2
    float dl[2];   // delta at p-4, p-3

    __device__ __forceinline__ void init()
    {
        ph[0] = ph[1] = L[0] = L[1] = c[0] = c[1] = dl[0] = dl[1] = 0.f;
    }

    // phi: Phi at plane p; c_pm1: Courant number at plane p-1.
    __device__ __forceinline__ float push(float phi, float c_pm1)
    {
        // L at p-1 (Phi at p-2, p-1, p; Courant at p-1)
        const float nb = by_sign(c_pm1, ph[0], phi, ph[1]);
        const float Ln = nb + (1.f - fabs(c_pm1)) * (ph[1] - nb);
        // delta at p-2 (Phi at p-2; L at p-3, p-2, p-1; Courant at p-2)
        const float C2 = c[1];
        const float Lb = by_sign(C2, Ln, L[0], L[1]);
        const float dn = (ph[0] - L[1]) - fabs(C2) * (Lb - L[1]);
        // CEC at p-3 (L at p-3; delta at p-4, p-3, p-2; Courant at p-3)
        const float C3 = c[0];
        const float dd = by_sign(C3, dl[0], dn, dl[1]);
        const float out = L[0] + 0.5f * dl[1] + (1.f + fabs(C3)) * (1.f / 6.f) * (dd - dl[1]);
        ph[0] = ph[1];
        ph[1] = phi;
        L[0] = L[1];
        L[1] = Ln;
        c[0] = C2;
        c[1] = c_pm1;
        dl[0] = dl[1];
        dl[1] = dn;
        return out;
    }
};

// ----------------------------------------------------------------- status
__device__ __forceinline__ void flag_cfl(unsigned *status, bool bad)
{
    // one atomic per warp that saw a violation
    const unsigned m = __ballot_sync(0xffffffffu, bad);
    if (m && (threadIdx.x & 31) == (__ffs(m) - 1)) atomicOr(status, 1u);
}

}  // namespace sl
