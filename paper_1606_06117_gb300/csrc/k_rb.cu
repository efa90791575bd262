// k_rb.cu -- the Rayleigh-Benard driver of Sec. 6 (eqs. e:nsnd, e:Tnd, e:mnd,
// e:poisson, e:proj) on the GPU: a 2D box with walls on all four sides, the
// velocity U = (u, w) and the temperature perturbation theta advected
// semi-Lagrangian by U with one of the paper's schemes, explicit buoyancy and
// diffusion, and a pressure-correction projection.
//
// Discretisation (cell-centred, nx x nz cells of Lx x Lz):
//  * the fields live on a grid padded by G = 3 ghost layers (the reach of the
//    split CEC stencil); before each step the ghosts are the walls' mirror
//    images: u and w change sign across every wall (no slip), theta changes
//    sign across the plates (theta = 0) and keeps it across the side walls
//    (d theta / dx = 0);
//  * the advection is sl_advect on the padded grid with the padded velocity:
//    the periodic wrap of the step kernels only ever reaches ghost cells;
//  * u2 = L[u] + dt Pr lap u, w2 = L[w] + dt (Ra Pr theta + Pr lap w),
//    theta' = L[theta] + dt (w + lap theta), 5-point Laplacians of the step-n
//    fields;
//  * projection: face velocities are averages of the two adjacent cells (zero
//    on the walls), their divergence D is the right-hand side of lap phi = D
//    with the compact Neumann Laplacian, solved in its eigenbasis: the
//    orthonormal DCT-II matrices C_x, C_z diagonalise it with eigenvalues
//    -(4/h^2) sin^2(pi j / 2 n) per axis, so phi = C_z^T [(C_z D C_x^T) / lam] C_x
//    with the constant mode set to zero.  Cells take the average of their
//    two faces' gradient corrections.
//
// GB300 runs FP64 at a small fraction of its FP32 rate (about two FMAs per
// clock and SM), so the step is arranged to spend few FP64 operations and to
// spread them over many SMs: each producer writes its cells' ghost images
// itself (no separate fill pass), the forces kernel also gives the divergence,
// the forces' CTAs hold 32 cells, and the transforms run one CTA per mode or
// row: all that stays within a z mode in one kernel (the x solve), the
// inverse z transform in the projection, which needs a row of phi and the
// difference of its neighbours only.  That makes four launches per step (the
// advection of the three fields in one).  At 50 x 50 the step is a chain of small
// kernels, so on small boxes each is launched while its predecessor runs (programmatic dependent
// launch), sets up what does not depend on it, copies its constant operands and
// then waits; long runs replay the step from a CUDA graph.  A kernel lets the next
// one in only when most of its work is done: CTAs that come in earlier take their
// places while the SMs are full, two or more end on one SM, and the FP64 pipe of
// that SM is what the step then waits for.
// Measured, FP64 CEC, us per step at 50 x 50 (128 x 128): 29.9 (65.5) with five
// launches one after the other, 23.9 with the double-precision sweeps of
// k_split64.cu, 23.0 (108) with four launches that overlap from their start, 21.5
// (100) with the forces' terms on warps of their own, 17.8 (58) with the late release,
// 16.3 (51) with one matrix per z mode for its x solve, 16.3 (42.5) with the overlap on
// small boxes only, 15.9 (42.6) now.  Boxes of one size differ by up to 3 % with where
// their memory lies.
#include <cmath>
#include <new>

#include "sl.h"
#include "sl_internal.h"

namespace sl {
namespace {

constexpr int RBG = 3;   // ghost layers

// Padded row length: G ghost columns on the left, G on the right and one more
// there when nx is odd, so that a padded plane has an even number of cells
// and the three state planes, back to back, share one 16-byte alignment.
__host__ __device__ constexpr int rb_px(int nx) { return nx + 2 * RBG + (nx & 1); }

// Ghost cell (k, i) of a padded (nz + 2G) x (nx + 2G) plane: the mirror image
// of an interior cell across the nearer wall(s), with sign sx per side-wall
// crossing and sz per plate crossing.  Interior cells are left alone.
template <typename T>
__global__ void k_rb_ghosts(T *p, int nplanes, int nx, int nz, int64_t pstride, const int *sx, const int *sz)
{
    const int px = rb_px(nx), pz = nz + 2 * RBG;
    const int64_t n = (int64_t)px * pz;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n * nplanes;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int f = (int)(idx / n);
        const int64_t r = idx - (int64_t)f * n;
        const int k = (int)(r / px), i = (int)(r - (int64_t)k * px);
        const int ki = k - RBG, ii = i - RBG;
        const bool gk = ki < 0 || ki >= nz, gi = ii < 0 || ii >= nx;
        if (!gk && !gi) continue;
        const int mk = ki < 0 ? -1 - ki : (ki >= nz ? 2 * nz - 1 - ki : ki);
        const int mi = ii < 0 ? -1 - ii : (ii >= nx ? 2 * nx - 1 - ii : ii);
        const int s = (gk ? sz[f] : 1) * (gi ? sx[f] : 1);
        T *pl = p + f * pstride;
        pl[r] = T(s) * pl[(int64_t)(mk + RBG) * px + mi + RBG];
    }
}

// Stores v at interior cell (k, i) of a padded plane and at each ghost cell
// whose mirror image it is (sign sx per side-wall crossing, sz per plate
// crossing): the same values the ghost fill gives, written by the producer.
template <typename T>
__device__ __forceinline__ void store_mirrored(T *pl, int k, int i, T v, int nx, int nz, T sx, T sz)
{
    const int px = rb_px(nx), gr = px - nx - RBG;   // gr ghost columns on the right
    pl[(int64_t)(k + RBG) * px + i + RBG] = v;
    const int gi = i < RBG ? -1 - i : (i >= nx - gr ? 2 * nx - 1 - i : INT32_MIN);
    const int gk = k < RBG ? -1 - k : (k >= nz - RBG ? 2 * nz - 1 - k : INT32_MIN);
    // a cell near both side walls (small nx) has two x images
    const int gi2 = (i < RBG && i >= nx - gr) ? 2 * nx - 1 - i : INT32_MIN;
    const int gk2 = (k < RBG && k >= nz - RBG) ? 2 * nz - 1 - k : INT32_MIN;
    const int xs[3] = {i, gi, gi2}, zs[3] = {k, gk, gk2};
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            if ((a == 0 && b == 0) || xs[a] == INT32_MIN || zs[b] == INT32_MIN) continue;
            const T sg = (a ? sx : T(1)) * (b ? sz : T(1));
            pl[(int64_t)(zs[b] + RBG) * px + xs[a] + RBG] = sg * v;
        }
}

// The explicit forces on the interior, from the advected fields a* and the
// step-n fields (ghosts filled): u2, w2 into o_u, o_w (interior only),
// theta' into o_t with its ghost images, and the divergence of the face
// velocities (averages of the adjacent cells of (u2, w2), zero on the walls)
// into d (nz x nx).  A cell evaluates u2 and w2 of its neighbours itself (the
// same expressions), so that no second pass is needed for the divergence.
// What bounds it at the paper's 50^2: FP64 issue, about 60 cycles of a scheduler per
// warp instruction, with one warp of 32 cells per SM.  So each of a CTA's 7 warps takes
// one of the terms (u2 here and on either side, w2 here and above and below, theta') of
// the same 32 cells, and the divergence is put together through shared memory.
// Measured, 50^2 FP64: 23.2 us per step with one thread per cell, 21.5 with
// the terms apart.
constexpr int kRbTerms = 7;
template <typename T>
__global__ void __launch_bounds__(32 * kRbTerms)
k_rb_forces(const T *u, const T *w, const T *th, const T *au, const T *aw, const T *at, T *o_u, T *o_w, T *o_t, T *d,
            int nx, int nz, T dt, T Ra, T Pr, T idx2, T idz2, T idx, T idz)
{
    __shared__ T val[kRbTerms][32];
    const int px = rb_px(nx), lane = threadIdx.x & 31, term = threadIdx.x >> 5;
    const int c = blockIdx.x * 32 + lane;
    const bool in = c < nx * nz;
    const int k = c / nx, i = c - k * nx;
    const int64_t o = (int64_t)(k + RBG) * px + i + RBG;
    auto lap = [&](const T *f, int64_t q) {
        return (f[q + 1] - T(2) * f[q] + f[q - 1]) * idx2 + (f[q + px] - T(2) * f[q] + f[q - px]) * idz2;
    };
    pdl_wait();
    if (term < 3) {
        // u2 at the cell (term 0), its east (1) and west neighbour (2)
        if (in && (term == 0 || (term == 1 ? i + 1 < nx : i > 0))) {
            const int64_t q = o + (term == 1) - (term == 2);
            const T v = au[q] + dt * (Pr * lap(u, q));
            val[term][lane] = v;
            if (term == 0) o_u[o] = v;
        }
    } else if (term < 6) {
        // w2 at the cell (term 3), above (4) and below it (5)
        if (in && (term == 3 || (term == 4 ? k + 1 < nz : k > 0))) {
            const int64_t q = o + (term == 4 ? px : 0) - (term == 5 ? px : 0);
            const T v = aw[q] + dt * (Ra * Pr * th[q] + Pr * lap(w, q));
            val[term][lane] = v;
            if (term == 3) o_w[o] = v;
        }
    } else if (in) {
        store_mirrored(o_t, k, i, at[o] + dt * (w[o] + lap(th, o)), nx, nz, T(1), T(-1));
    }
    pdl_release();
    __syncthreads();
    T part = T(0);
    if (term == 0 && in) {
        const T ue = i + 1 < nx ? T(0.5) * (val[0][lane] + val[1][lane]) : T(0);
        const T uw = i > 0 ? T(0.5) * (val[2][lane] + val[0][lane]) : T(0);
        part = (ue - uw) * idx;
    } else if (term == 3 && in) {
        const T wn = k + 1 < nz ? T(0.5) * (val[3][lane] + val[4][lane]) : T(0);
        const T ws = k > 0 ? T(0.5) * (val[5][lane] + val[3][lane]) : T(0);
        val[6][lane] = (wn - ws) * idz;
    }
    __syncthreads();
    if (term == 0 && in) d[c] = part + val[6][lane];
}

constexpr int kRbRowThreads = 256;

// out_q(c) = sum_{t < K} a_q[t] B[t * ldb + c * cs] for c < N and q < Q, by the
// CTA's 256 threads: 64 columns at a time, each column's sum split over four
// thread groups (t = g mod 4, two terms in flight per group) and combined in
// fixed order in shared memory (part, Q x 256 elements).
template <int Q, typename T, typename Store>
__device__ __forceinline__ void rb_vecmat(const T *const (&a)[Q], const T *B, int64_t ldb, int64_t cs, int K, int N,
                                          T *part, Store store)
{
    const int c = threadIdx.x & 63, g = threadIdx.x >> 6;
    for (int c0 = 0; c0 < N; c0 += 64) {
        const int col = c0 + c;
        T acc0[Q], acc1[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) acc0[q] = acc1[q] = T(0);
        if (col < N) {
            const T *b = B + col * cs;
            int t = g;
#pragma unroll 4
            for (; t + 4 < K; t += 8) {
                const T x = b[t * ldb], y = b[(t + 4) * ldb];
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    acc0[q] += a[q][t] * x;
                    acc1[q] += a[q][t + 4] * y;
                }
            }
            if (t < K) {
                const T x = b[t * ldb];
#pragma unroll
                for (int q = 0; q < Q; ++q) acc0[q] += a[q][t] * x;
            }
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) part[q * kRbRowThreads + g * 64 + c] = acc0[q] + acc1[q];
        __syncthreads();
        if (g < Q && col < N) {   // group q combines output q
            const T *p = part + g * kRbRowThreads + c;
            store(g, col, (p[0] + p[64]) + (p[128] + p[192]));
        }
        __syncthreads();
    }
}

// Copies n elements from global to shared memory: 16-byte chunks by cp.async
// (both bases 16-byte aligned), the tail by plain loads.
template <typename T>
__device__ __forceinline__ void rb_stage(T *dst, const T *src, int64_t n)
{
    constexpr int V = 16 / sizeof(T);
    const int64_t nv = n / V;
    for (int64_t c = threadIdx.x; c < nv; c += blockDim.x) cp_async16(dst + c * V, src + c * V);
    for (int64_t i = nv * V + threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

// Elements a staged operand block takes, rounded up to a 16-byte multiple.
template <typename T>
__host__ __device__ constexpr int64_t rb_pad(int64_t n)
{
    return (n + 16 / (int64_t)sizeof(T) - 1) / (16 / (int64_t)sizeof(T)) * (16 / (int64_t)sizeof(T));
}

// Everything of the Poisson solve that stays within one z mode, one CTA per mode k:
//   R[i] = sum_m C_z[k][m] D[m][i],  F[j] = sum_i R[i] C_x[j][i] / lam_kj,
//   G[k][i] = sum_j F[j] C_x[j][i]
// (lam_kj = lz[k] + lx[j]; the constant mode F[0] of k = 0 is 0); phi = C_z^T G is
// left to the projection.  The last two are one linear map of a row, so
//   G[k] = R M_k,  M_k[i][i'] = sum_{j, lam_kj != 0} C_x[j][i] C_x[j][i'] / lam_kj
// with the matrices M_k made once per box (k_rb_green): a third of the FP64 sums and all
// divisions less per step (FP64 CEC, 50 x 50: 17.8 -> 16.3 us per step, 128 x 128: 58 ->
// 51, 400 x 50: 175 -> 110).  Forms:
//   kLarge   M would take more than kRbGreenMax, or FP32 boxes that are not staged
//            (their sums are cheap and C_x stays closer than M: 128 x 128 33 us against
//            38): both x transforms, C_x entering transposed for the first, so that
//            every load is coalesced or a broadcast;
//   kGreen   M_k read from global memory;
//   kStaged  small boxes: D and M_k are copied to shared memory first, so that the
//            sums do not wait on L2; M_k while the predecessor still runs.
enum RbForm { kLarge, kGreen, kStaged };
template <typename T, int FORM>
__global__ void __launch_bounds__(kRbRowThreads)
k_rb_modes(const T *D, const T *cz, const T *cx, const T *cxT, const T *M, const T *lx, const T *lz, T *G, int nx, int nz)
{
    extern __shared__ __align__(16) unsigned char rb_smem[];
    T *part = reinterpret_cast<T *>(rb_smem), *R = part + kRbRowThreads, *F = R + rb_pad<T>(nx);
    T *az = F + rb_pad<T>(nx), *sD = az + rb_pad<T>(nz), *sM = sD + rb_pad<T>((int64_t)nz * nx);
    const int k = blockIdx.x;
    for (int m = threadIdx.x; m < nz; m += kRbRowThreads) az[m] = cz[(int64_t)k * nz + m];
    const T *const Mk = FORM == kLarge ? nullptr : M + k * rb_pad<T>((int64_t)nx * nx);
    if constexpr (FORM == kStaged) rb_stage(sM, Mk, (int64_t)nx * nx);
    pdl_wait();
    if constexpr (FORM == kStaged) {
        rb_stage(sD, D, (int64_t)nz * nx);
        cp_async_commit();
        cp_async_wait_all();
    }
    __syncthreads();
    const T *const a0[1] = {az}, *const a1[1] = {R}, *const a2[1] = {F};
    T *Gk = G + (int64_t)k * nx;
    rb_vecmat<1>(a0, FORM == kStaged ? sD : D, nx, 1, nz, nx, part, [&](int, int i, T v) { R[i] = v; });
    if constexpr (FORM == kLarge) {
        const T lk = lz[k];
        rb_vecmat<1>(a1, cxT, nx, 1, nx, nx, part,
                     [&](int, int j, T v) { F[j] = (k == 0 && j == 0) ? T(0) : v / (lk + lx[j]); });
    }
    pdl_release();
    rb_vecmat<1>(FORM == kLarge ? a2 : a1, FORM == kLarge ? cx : (FORM == kStaged ? sM : Mk), nx, 1, nx, nx, part,
                 [&](int, int i, T v) { Gk[i] = v; });
}

// The tables of a box, made on the device.  Measured, ms to create an FP64 box with host
// tables and no M, with host tables and M as a sum over the modes, and now: 50 x 50
// 0.12 / 0.17 / 0.06, 300 x 200 1.6 / 20.8 / 0.6, 1024 x 32 13 / 134 / 0.8, 48 x 4096
// 157 / 320 / 5.7.
//
// Element (j, i) of the orthonormal DCT-II matrix, s_j cos(pi j (i + 1/2) / n); the
// angle in units of pi / (2 n) is an integer, reduced to [0, n] exactly.
__device__ __forceinline__ double rb_cosine(int j, int i, int n)
{
    int r = (int)((int64_t)j * (2 * i + 1) % (4 * n));
    if (r > 2 * n) r = 4 * n - r;
    const bool neg = r > n;
    if (neg) r = 2 * n - r;
    const double c = sqrt((j == 0 ? 1.0 : 2.0) / n) * cospi((double)r / (2.0 * n));
    return neg ? -c : c;
}

// C (row j), and where they are wanted its transpose and, transposed, the differences
// of the rows around each (k_rb_project); the eigenvalues per axis.
template <typename T>
__global__ void k_rb_tables(T *c, T *ct, T *zt, T *lam, int n, double h)
{
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)n * n) return;
    const int a = (int)(e / n), b = (int)(e % n);
    c[e] = T(rb_cosine(a, b, n));
    if (ct) ct[e] = T(rb_cosine(b, a, n));
    if (zt) zt[e] = T(rb_cosine(b, a + 1 < n ? a + 1 : a, n) - rb_cosine(b, a > 0 ? a - 1 : a, n));
    if (a == 0) {
        const double s = sinpi((double)b / (2.0 * n));
        lam[b] = T(-4.0 / (h * h) * (s * s));
    }
}

// M of one box.  M_k inverts the tridiagonal matrix lap_x + lz_k, so it has a closed form:
// with s = dx / dz sin(pi k / (2 nz)), theta = 2 asinh(s), i <= i' (and symmetric)
//   M_k[i][i'] = -dx^2 cosh((i + 1/2) theta) cosh((nx - i' - 1/2) theta) / (sinh(theta) sinh(nx theta)),
// written with decaying exponentials; for k = 0 the inverse on vectors of zero mean,
//   dx^2 (max(x, x') - (x^2 + x'^2) / (2 nx) - nx / 3 + 1 / (12 nx)),   x = i + 1/2.
// (Its error against extended precision is a few units in the last place, that of the
// sum over the modes up to thirty.)  One CTA of mode k = blockIdx.y takes every
// gridDim.x-th row.
template <typename T>
__global__ void k_rb_green(T *M, int nx, int nz, double dx, double dz)
{
    extern __shared__ __align__(16) unsigned char rb_smem[];
    double *decay = reinterpret_cast<double *>(rb_smem);   // exp(-i theta)
    __shared__ double mode[3];
    const int k = blockIdx.y;
    if (k && threadIdx.x == 0) {   // once: every thread would wait for the FP64 pipe
        const double sn = sinpi((double)k / (2.0 * nz)), s = dx / dz * sn, theta = 2.0 * asinh(s);
        mode[0] = theta;
        mode[1] = dz / (2.0 * sn) * (dx / (2.0 * hypot(1.0, s))) / expm1(-2.0 * nx * theta);
        mode[2] = exp(-theta);
    }
    __syncthreads();
    if (k)
        for (int i = threadIdx.x; i < nx; i += blockDim.x) decay[i] = exp(-i * mode[0]);
    __syncthreads();
    const double scale = mode[1], half = mode[2];
    T *Mk = M + k * rb_pad<T>((int64_t)nx * nx);
    for (int i = blockIdx.x; i < nx; i += gridDim.x)
        for (int i2 = threadIdx.x; i2 < nx; i2 += blockDim.x) {
            const int lo = min(i, i2), hi = max(i, i2);
            double v;
            if (k) {
                const double p = decay[lo], q = decay[nx - 1 - hi];
                v = scale * decay[hi - lo] * (1.0 + p * p * half) * (1.0 + q * q * half);
            } else {
                const double x = lo + 0.5, y = hi + 0.5;
                v = dx * dx * (y - (x * x + y * y) / (2.0 * nx) - (nx / 3.0 - 1.0 / (12.0 * nx)));
            }
            Mk[(int64_t)i * nx + i2] = T(v);
        }
}

template <typename T>
cudaError_t rb_tables(void *cx, void *cxT, void *cz, void *czT, void *zT, void *lx, void *lz, void *M, int nx, int nz,
                      double dx, double dz)
{
    auto blocks = [](int n) { return (unsigned)(((int64_t)n * n + 63) / 64); };   // small, to spread over the SMs
    k_rb_tables<T><<<blocks(nx), 64>>>(static_cast<T *>(cx), static_cast<T *>(cxT), static_cast<T *>(nullptr),
                                        static_cast<T *>(lx), nx, dx);
    k_rb_tables<T><<<blocks(nz), 64>>>(static_cast<T *>(cz), static_cast<T *>(czT), static_cast<T *>(zT),
                                        static_cast<T *>(lz), nz, dz);
    if (M) k_rb_green<T><<<dim3(nx < 256 ? (nx + 7) / 8 : 32, nz), 256, sizeof(double) * nx>>>(static_cast<T *>(M), nx, nz, dx, dz);
    return cudaGetLastError();
}

// Projection, one CTA per row m: phi[m][i] = sum_k C_z[k][m] G[k][i] and the
// difference of the rows next to it, dphi[i] = sum_k Z[k][m] G[k][i] with Z[k][m] =
// C_z[k][m + 1] - C_z[k][m - 1] (rows beyond a wall replaced by m itself: no flux
// there).  Cells take the average of their two faces' gradient corrections
// (face gradient (phi_{i+1} - phi_i) / dx inside, zero on the walls); the result
// is the new u, w with their ghost images.  czT, zT: C_z and Z transposed.
// PAIR: one CTA for the rows m and nz - 1 - m, whose sums differ in the signs of the odd
// modes only (C_z[k][nz-1-m] = (-1)^k C_z[k][m], Z with a minus), so that the even
// and the odd half-sums serve both: half the FP64 work, on half as many CTAs.  It
// is for boxes of more rows than kRbPairRows, the SMs they would otherwise share.
// Measured, CEC, us per step without and with: 300 x 200 FP64 240 / 232, FP32 127 / 105.
constexpr int kRbPairRows = 152;
// Boxes of at most half as many rows as there are SMs launch each kernel while its
// predecessor runs: the CTAs of two kernels then find an SM each.  On larger boxes
// the next kernel's CTAs crowd on the SMs that finish first, and the FP64 pipe of
// those SMs is what the step waits for.  Measured, FP64 CEC, us per step with and
// without the overlap: 50 x 50 16.3 / 17.0, 80 x 80 30.6 / 29.9, 100 x 100 41.7 / 36.0,
// 128 x 128 50.9 / 42.5, 512 x 256 702 / 535.
constexpr int kRbEarlyRows = 76;
template <typename T, bool STAGED, bool PAIR>
__global__ void __launch_bounds__(kRbRowThreads)
k_rb_project(const T *u2, const T *w2, const T *G, const T *czT, const T *zT, T *u, T *w, int nx, int nz, T idx, T idz)
{
    extern __shared__ __align__(16) unsigned char rb_smem[];
    constexpr int H = PAIR ? 2 : 1;   // interleaved halves of the sums over k
    T *part = reinterpret_cast<T *>(rb_smem), *phi = part + 2 * kRbRowThreads, *dphi = phi + H * rb_pad<T>(nx);
    T *a = dphi + H * rb_pad<T>(nx), *z = a + rb_pad<T>(nz) + rb_pad<T>(H), *sG = z + rb_pad<T>(nz) + rb_pad<T>(H);
    const int m = blockIdx.x, px = rb_px(nx), nh = (nz + H - 1) / H;
    for (int k = threadIdx.x; k < nz; k += kRbRowThreads) {   // even k, then odd k
        const int at = PAIR ? (k & 1) * nh + (k >> 1) : k;
        a[at] = czT[(int64_t)m * nz + k];
        z[at] = zT[(int64_t)m * nz + k];
    }
    pdl_wait();
    if constexpr (STAGED) {
        rb_stage(sG, G, (int64_t)nz * nx);
        cp_async_commit();
        cp_async_wait_all();
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const T *const az[2] = {a + h * nh, z + h * nh};
        T *ph = phi + h * rb_pad<T>(nx), *dp = dphi + h * rb_pad<T>(nx);
        rb_vecmat<2>(az, (STAGED ? sG : G) + h * nx, H * nx, 1, h ? nz / 2 : nh, nx, part,
                     [&](int q, int i, T v) { (q ? dp : ph)[i] = v; });
    }
    pdl_release();
    auto correct = [&](int row, int i, T dx, T dz) {
        const int64_t o = (int64_t)(row + RBG) * px + i + RBG;
        store_mirrored(u, row, i, u2[o] - T(0.5) * (dx * idx), nx, nz, T(-1), T(-1));
        store_mirrored(w, row, i, w2[o] - T(0.5) * (dz * idz), nx, nz, T(-1), T(-1));
    };
    for (int i = threadIdx.x; i < nx; i += kRbRowThreads) {
        const int ie = i + 1 < nx ? i + 1 : i, iw = i > 0 ? i - 1 : i;
        const T dx = phi[ie] - phi[iw];
        if constexpr (!PAIR) {
            correct(m, i, dx, dphi[i]);
        } else {
            const T *po = phi + rb_pad<T>(nx);
            const T dxo = po[ie] - po[iw], dzo = dphi[rb_pad<T>(nx) + i];
            correct(m, i, dx + dxo, dphi[i] + dzo);
            if (nz - 1 - m != m) correct(nz - 1 - m, i, dx - dxo, dzo - dphi[i]);
        }
    }
}

// Dynamic shared memory of the two, and the most a box takes to stage its operands.
template <typename T>
size_t rb_modes_smem(int nx, int nz, bool staged)
{
    return sizeof(T) * (size_t)(kRbRowThreads + 2 * rb_pad<T>(nx) + rb_pad<T>(nz) +
                                (staged ? rb_pad<T>((int64_t)nz * nx) + rb_pad<T>((int64_t)nx * nx) : 0));
}
template <typename T>
size_t rb_project_smem(int nx, int nz, bool staged)
{
    const int h = nz > kRbPairRows ? 2 : 1;
    return sizeof(T) * (size_t)(2 * kRbRowThreads + 2 * h * rb_pad<T>(nx) + 2 * (rb_pad<T>(nz) + rb_pad<T>(2)) +
                                (staged ? rb_pad<T>((int64_t)nz * nx) : 0));
}
// (an unstaged FP64 box of 4096 x 4096 takes 197 KB in the projection)
constexpr size_t kRbStagedMax = 96 * 1024, kRbSmemMax = 200 * 1024;
// The most M takes.  FP64 boxes gain up to where it is read from HBM every step (144 MB,
// 300 x 200: 285 -> 240 us) and break even at 537 MB (512 x 256).  Every staged box is below.
constexpr size_t kRbGreenMax = 256u << 20;

// interior <-> padded copies
template <typename T>
__global__ void k_rb_copy(const T *src, T *dst, int nx, int nz, bool to_padded)
{
    const int px = rb_px(nx);
    const int n = nx * nz;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        const int k = c / nx, i = c - (c / nx) * nx;
        const int64_t o = (int64_t)(k + RBG) * px + i + RBG;
        if (to_padded)
            dst[o] = src[c];
        else
            dst[c] = src[o];
    }
}

int blocks_for(int64_t n) { return (int)std::min<int64_t>((n + 255) / 256, 4096); }

}  // namespace
}  // namespace sl

using namespace sl;

struct sl_rb {
    int device = -1;
    bool staged = false;   // transforms with staged operands (small boxes)
    int nx = 0, nz = 0, scheme = SL_CEC, dtype = SL_F64;
    double Lx = 2.0, Lz = 1.0, Ra = 0.0, Pr = 1.0;
    int64_t step = 0;
    size_t esz = 8;
    int64_t plane = 0;     // padded plane: rb_px(nx) (nz + 2G) elements
    int cur = 0;           // which of the two state buffers holds step n
    void *mem = nullptr;   // one device allocation
    // padded planes: two states (u, w, theta back to back, so that (u, w) is
    // the velocity argument of the advection), the advected fields, (u2, w2)
    void *S[2] = {nullptr, nullptr}, *A = nullptr, *W = nullptr;
    // interior arrays (nz x nx): the face divergence D, and phi in z modes (G)
    void *d = nullptr, *G = nullptr;
    // orthonormal DCT-II matrices C_x and C_z, their transposes (C_x's without M only), the
    // row differences of C_z (transposed, k_rb_project); eigenvalues per axis
    void *cx = nullptr, *cxT = nullptr, *cz = nullptr, *czT = nullptr, *zT = nullptr, *lx = nullptr, *lz = nullptr;
    void *M = nullptr;      // the z modes' x solves (k_rb_modes), unless too large
    int *signs = nullptr;   // sx of (u, w, theta), then sz of (u, w, theta)
    // long runs replay kRbGraphSteps steps from one CUDA graph, captured for
    // one dt and one starting buffer on a stream of the box's own
    cudaStream_t cs = nullptr;
    cudaGraphExec_t exec = nullptr;
    double graph_dt = 0.0;
    int graph_cur = -1;
};

namespace {

template <typename T>
int rb_step_t(sl_rb *r, double dt, int nsteps, cudaStream_t st)
{
    const int nx = r->nx, nz = r->nz, n = nx * nz;
    const int px = rb_px(nx), pz = nz + 2 * RBG;
    const int64_t P = r->plane;
    T *A = static_cast<T *>(r->A), *Wk = static_cast<T *>(r->W);
    T *d = static_cast<T *>(r->d), *G = static_cast<T *>(r->G);
    const T *cx = static_cast<const T *>(r->cx), *cxT = static_cast<const T *>(r->cxT);
    const T *cz = static_cast<const T *>(r->cz), *czT = static_cast<const T *>(r->czT), *zT = static_cast<const T *>(r->zT);
    const T *lx = static_cast<const T *>(r->lx), *lz = static_cast<const T *>(r->lz), *M = static_cast<const T *>(r->M);
    const double dx = r->Lx / nx, dz = r->Lz / nz;
    const int64_t pdims[3] = {px, pz, 1};
    const double sp[3] = {dx, dz, 1.0};
    const size_t msm = rb_modes_smem<T>(nx, nz, r->staged), psm = rb_project_smem<T>(nx, nz, r->staged);
    auto modes = r->staged ? k_rb_modes<T, kStaged> : (M ? k_rb_modes<T, kGreen> : k_rb_modes<T, kLarge>);
    const bool pair = nz > kRbPairRows, early = nz <= kRbEarlyRows;
    auto project = r->staged ? (pair ? k_rb_project<T, true, true> : k_rb_project<T, true, false>)
                             : (pair ? k_rb_project<T, false, true> : k_rb_project<T, false, false>);
    for (int s = 0; s < nsteps; ++s) {
        // S0 holds step n with its ghost layers (the walls' mirror images)
        T *S0 = static_cast<T *>(r->S[r->cur]), *S1 = static_cast<T *>(r->S[r->cur ^ 1]);
        // semi-Lagrangian advection of u, w, theta by U^n on the padded box;
        // CEC alternates its sweep order with the step index
        const void *ins[3] = {S0, S0 + P, S0 + 2 * P};
        void *outs[3] = {A, A + P, A + 2 * P};
        int rc = advect_fields(outs, ins, 3, S0, 2, pdims, sp, dt, r->scheme, r->dtype, (int)(r->step & 1), st, early);
        if (rc) return rc;
        // forces: u2, w2 into the work planes, theta' (with ghosts) into the
        // next state, the face divergence D into d
        cudaError_t e = launch_kernel(k_rb_forces<T>, dim3((n + 31) / 32), 32 * kRbTerms, 0, st, early, S0, S0 + P, S0 + 2 * P, A, A + P,
                                      A + 2 * P, Wk, Wk + P, S1 + 2 * P, d, nx, nz, T(dt), T(r->Ra), T(r->Pr),
                                      T(1.0 / (dx * dx)), T(1.0 / (dz * dz)), T(1.0 / dx), T(1.0 / dz));
        // G = [(C_z D C_x^T) / lam] C_x
        if (e == cudaSuccess)
            e = launch_kernel(modes, dim3(nz), kRbRowThreads, msm, st, early, d, cz, cx, cxT, M, lx, lz, G, nx, nz);
        // the projected u, w (with ghosts) of the next state
        if (e == cudaSuccess)
            e = launch_kernel(project, dim3(pair ? (nz + 1) / 2 : nz), kRbRowThreads, psm, st, early, Wk, Wk + P, G, czT, zT, S1, S1 + P, nx, nz,
                              T(1.0 / dx), T(1.0 / dz));
        if (e != cudaSuccess) return set_error(SL_ERR_CUDA, cudaGetErrorString(e));
        r->cur ^= 1;
        ++r->step;
    }
    return SL_OK;
}

template <typename T>
int rb_copy_t(sl_rb *r, const void *u, const void *w, const void *t, void *ou, void *ow, void *ot, cudaStream_t st)
{
    const int cb = blocks_for((int64_t)r->nx * r->nz);
    T *S = static_cast<T *>(r->S[r->cur]);
    const int64_t P = r->plane;
    if (u) {
        k_rb_copy<T><<<cb, 256, 0, st>>>(static_cast<const T *>(u), S, r->nx, r->nz, true);
        k_rb_copy<T><<<cb, 256, 0, st>>>(static_cast<const T *>(w), S + P, r->nx, r->nz, true);
        k_rb_copy<T><<<cb, 256, 0, st>>>(static_cast<const T *>(t), S + 2 * P, r->nx, r->nz, true);
        k_rb_ghosts<T><<<blocks_for(3 * P), 256, 0, st>>>(S, 3, r->nx, r->nz, P, r->signs, r->signs + 3);
    } else {
        k_rb_copy<T><<<cb, 256, 0, st>>>(S, static_cast<T *>(ou), r->nx, r->nz, false);
        k_rb_copy<T><<<cb, 256, 0, st>>>(S + P, static_cast<T *>(ow), r->nx, r->nz, false);
        k_rb_copy<T><<<cb, 256, 0, st>>>(S + 2 * P, static_cast<T *>(ot), r->nx, r->nz, false);
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? SL_OK : set_error(SL_ERR_CUDA, cudaGetErrorString(e));
}

constexpr int kRbGraphSteps = 8;   // even: the graph ends on the buffer and sweep order it starts on

int rb_eager(sl_rb *r, double dt, int nsteps, cudaStream_t st)
{
    return r->dtype == SL_F64 ? rb_step_t<double>(r, dt, nsteps, st) : rb_step_t<float>(r, dt, nsteps, st);
}

// The graph of kRbGraphSteps steps from the current buffer with this dt
// (captured again when either differs from the cached graph's).
int rb_graph(sl_rb *r, double dt)
{
    if (r->exec && r->graph_dt == dt && r->graph_cur == r->cur) return SL_OK;
    if (r->exec) {
        cudaGraphExecDestroy(r->exec);
        r->exec = nullptr;
    }
    cudaError_t e = cudaSuccess;
    if (!r->cs) e = cudaStreamCreateWithFlags(&r->cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) return set_error(SL_ERR_CUDA, cudaGetErrorString(e));
    const int cur0 = r->cur;
    const int64_t step0 = r->step;
    e = cudaStreamBeginCapture(r->cs, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return set_error(SL_ERR_CUDA, cudaGetErrorString(e));
    const int rc = rb_eager(r, dt, kRbGraphSteps, r->cs);
    cudaGraph_t g = nullptr;
    e = cudaStreamEndCapture(r->cs, &g);
    r->cur = cur0;   // nothing ran yet
    r->step = step0;
    if (rc != SL_OK || e != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        cudaGetLastError();
        return rc != SL_OK ? rc : set_error(SL_ERR_CUDA, cudaGetErrorString(e));
    }
    e = cudaGraphInstantiate(&r->exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        r->exec = nullptr;
        return set_error(SL_ERR_CUDA, cudaGetErrorString(e));
    }
    r->graph_dt = dt;
    r->graph_cur = cur0;
    return SL_OK;
}

}  // namespace

extern "C" {

int sl_rb_create(sl_rb **out, int nx, int nz, double Lx, double Lz, double Ra, double Pr, int scheme, int dtype)
{
    if (!out) return set_error(SL_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (nx < 4 || nz < 4 || nx > 4096 || nz > 4096) return set_error(SL_ERR_ARG, "nx and nz must be in [4, 4096]");
    if (!(Lx > 0) || !(Lz > 0) || !std::isfinite(Lx) || !std::isfinite(Lz) || !std::isfinite(Ra) ||
        !std::isfinite(Pr) || Pr < 0)
        return set_error(SL_ERR_ARG, "Lx, Lz must be > 0; Ra, Pr finite, Pr >= 0");
    if (scheme < SL_CIR || scheme > SL_CEC) return set_error(SL_ERR_ARG, "unknown scheme");
    if (dtype != SL_F32 && dtype != SL_F64) return set_error(SL_ERR_UNSUPPORTED, "the box runs in SL_F32 or SL_F64");
    DevCtx *c = ctx_get();
    if (!c) return set_error(SL_ERR_CUDA, "could not create the device context");
    sl_rb *r = new (std::nothrow) sl_rb();
    if (!r) return set_error(SL_ERR_NOMEM, "host allocation");
    r->device = c->device;
    r->nx = nx;
    r->nz = nz;
    r->Lx = Lx;
    r->Lz = Lz;
    r->Ra = Ra;
    r->Pr = Pr;
    r->scheme = scheme;
    r->dtype = dtype;
    r->esz = dtype == SL_F64 ? 8 : 4;
    // the planes of one state are contiguous (the advection's velocity is
    // (u, w)); every buffer starts on a 512-byte boundary
    r->plane = (int64_t)rb_px(nx) * (nz + 2 * RBG);
    auto round64 = [](int64_t k) { return (k + 63) / 64 * 64; };
    const int64_t n = (int64_t)nx * nz;
    const int64_t mstride = dtype == SL_F64 ? rb_pad<double>((int64_t)nx * nx) : rb_pad<float>((int64_t)nx * nx);
    r->staged = (dtype == SL_F64 ? rb_modes_smem<double>(nx, nz, true) : rb_modes_smem<float>(nx, nz, true)) <= kRbStagedMax;
    int64_t melems = r->staged || (dtype == SL_F64 && (size_t)(nz * mstride) * r->esz <= kRbGreenMax) ? nz * mstride : 0;
    auto elements = [&] {
        return (melems ? round64(melems) : round64((int64_t)nx * nx)) + round64((int64_t)nx * nx) + round64(nx) +
               round64(nz) + 4 * round64(3 * r->plane) + 2 * round64(n) + 3 * round64((int64_t)nz * nz) + 64;
    };
    auto allocate = [&] {
        if (cudaMalloc(&r->mem, r->esz * elements()) == cudaSuccess) return true;
        cudaGetLastError();
        return false;
    };
    bool got = allocate();
    if (!got && melems) {   // without M and staging the box takes less
        r->staged = false;
        melems = 0;
        got = allocate();
    }
    if (!got) {
        delete r;
        return set_error(SL_ERR_NOMEM, "device buffers of the box");
    }
    const int64_t elems = elements();
    char *p = static_cast<char *>(r->mem);
    auto take = [&](int64_t k) {
        void *q = p;
        p += r->esz * round64(k);
        return q;
    };
    r->S[0] = take(3 * r->plane);
    r->S[1] = take(3 * r->plane);
    r->A = take(3 * r->plane);
    r->W = take(3 * r->plane);
    r->d = take(n);
    r->G = take(n);
    r->cx = take((int64_t)nx * nx);
    if (!melems) r->cxT = take((int64_t)nx * nx);
    r->lx = take(nx);
    r->lz = take(nz);
    r->cz = take((int64_t)nz * nz);
    r->czT = take((int64_t)nz * nz);
    r->zT = take((int64_t)nz * nz);
    if (melems) r->M = take(melems);
    r->signs = reinterpret_cast<int *>(p);
    const double dx = Lx / nx, dz = Lz / nz;
    const int signs[6] = {-1, -1, 1, -1, -1, -1};   // sx of u, w, theta; sz of u, w, theta
    cudaError_t e = cudaMemset(r->mem, 0, r->esz * elems);
    if (e == cudaSuccess)
        e = dtype == SL_F64 ? rb_tables<double>(r->cx, r->cxT, r->cz, r->czT, r->zT, r->lx, r->lz, r->M, nx, nz, dx, dz)
                            : rb_tables<float>(r->cx, r->cxT, r->cz, r->czT, r->zT, r->lx, r->lz, r->M, nx, nz, dx, dz);
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
    if (e == cudaSuccess) e = cudaMemcpy(r->signs, signs, sizeof signs, cudaMemcpyHostToDevice);
    // small boxes stage the transforms' operands in shared memory; the kernels'
    // limit is per function, not per box, so it is raised to the cap that every
    // box fits under
    auto raise = [&](auto kern) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRbSmemMax);
    };
    if (dtype == SL_F64) {
        raise(k_rb_modes<double, kStaged>);
        raise(k_rb_modes<double, kGreen>);
        raise(k_rb_modes<double, kLarge>);
        raise(k_rb_project<double, true, false>);
        raise(k_rb_project<double, false, false>);
        raise(k_rb_project<double, true, true>);
        raise(k_rb_project<double, false, true>);
    } else {
        raise(k_rb_modes<float, kStaged>);
        raise(k_rb_modes<float, kGreen>);
        raise(k_rb_modes<float, kLarge>);
        raise(k_rb_project<float, true, false>);
        raise(k_rb_project<float, false, false>);
        raise(k_rb_project<float, true, true>);
        raise(k_rb_project<float, false, true>);
    }
    if (e != cudaSuccess) {
        cudaFree(r->mem);
        delete r;
        return set_error(SL_ERR_CUDA, cudaGetErrorString(e));
    }
    *out = r;
    return SL_OK;
}

int sl_rb_set_state(sl_rb *r, const void *u, const void *w, const void *theta, void *stream)
{
    if (!r || !u || !w || !theta) return set_error(SL_ERR_ARG, "NULL argument");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    r->step = 0;
    return r->dtype == SL_F64 ? rb_copy_t<double>(r, u, w, theta, nullptr, nullptr, nullptr, st)
                              : rb_copy_t<float>(r, u, w, theta, nullptr, nullptr, nullptr, st);
}

int sl_rb_get_state(sl_rb *r, void *u, void *w, void *theta, void *stream)
{
    if (!r || !u || !w || !theta) return set_error(SL_ERR_ARG, "NULL argument");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return r->dtype == SL_F64 ? rb_copy_t<double>(r, nullptr, nullptr, nullptr, u, w, theta, st)
                              : rb_copy_t<float>(r, nullptr, nullptr, nullptr, u, w, theta, st);
}

int sl_rb_step(sl_rb *r, double dt, int nsteps, void *stream)
{
    if (!r || nsteps < 0 || !std::isfinite(dt)) return set_error(SL_ERR_ARG, "bad argument");
    DevCtx *c = ctx_get();
    if (!c || c->device != r->device) return set_error(SL_ERR_ARG, "the box belongs to another device");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int left = nsteps, rc = SL_OK;
    if (left >= 2 * kRbGraphSteps) {
        if (r->step & 1) {   // graphs start on an even step (CEC's x-first sweep)
            rc = rb_eager(r, dt, 1, st);
            if (rc) return rc;
            --left;
        }
        rc = rb_graph(r, dt);
        if (rc) return rc;
        for (; left >= kRbGraphSteps; left -= kRbGraphSteps) {
            const cudaError_t e = cudaGraphLaunch(r->exec, st);
            if (e != cudaSuccess) return set_error(SL_ERR_CUDA, cudaGetErrorString(e));
            r->step += kRbGraphSteps;
        }
    }
    return left ? rb_eager(r, dt, left, st) : SL_OK;
}

int sl_rb_destroy(sl_rb *r)
{
    if (!r) return SL_OK;
    if (r->exec) cudaGraphExecDestroy(r->exec);
    if (r->cs) cudaStreamDestroy(r->cs);
    if (r->mem) cudaFree(r->mem);
    delete r;
    return SL_OK;
}

}  // extern "C"
