// k_learned.cu -- learned one-pass corrector: a 67 -> 64 -> 64 -> 1 MLP that
// maps each cell's 4 x 4 x 4 upwind neighbourhood and its fractional departure
// offsets to the third-order correction, so that one step is
//     Phi_new = L_U[Phi] + s * MLP(features),
// with L_U the multilinear (CIR) value at the departure point (Sec. 3, eq.
// CIR2D) and the target of training the combined scheme of eqs. intro:CEC /
// intro:CECcoef.  No counterpart in the paper: a throughput form whose error
// is judged against the plain scheme.
//
// Features of cell i (index space, |C| <= 1): X_d = i_d - C_d, base
// b_d = min(floor(X_d), i_d), f_d = X_d - b_d in [0, 1]; the 64 values
// Phi(b + (a, b', c)), a, b', c in {-1, 0, 1, 2} (x fastest); m = the trilinear
// value of the inner 2 x 2 x 2 at f (= CIR); s = max |Phi_k - m| (floored);
// inputs x_k = (Phi_k - m)/s, x_{64+d} = f_d - 1/2; output Phi_new = m + s y.
//
// Kernels: feature extraction for training samples, an FP32 minibatch
// forward/backward kernel with an Adam update, and the inference step whose
// two GEMMs run on the tensor cores (tcgen05.mma, BF16; the weights and the last 16 K
// columns of the activations in shared memory, the activations' first 64 columns and
// the FP32 accumulators in tensor memory).
#include <cuda_bf16.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <random>
#include <vector>

#include "sl.h"
#include "sl_internal.h"

namespace sl {
namespace lrn {

constexpr int NIN = 67, KP1 = 80, NH = 64;   // inputs, padded K of layer 1, hidden width
constexpr int NPARAM = NH * NIN + NH + NH * NH + NH + NH + 1;   // 8577
// offsets of the parameters in the FP32 parameter vector
constexpr int O_W1 = 0, O_B1 = O_W1 + NH * NIN, O_W2 = O_B1 + NH, O_B2 = O_W2 + NH * NH, O_W3 = O_B2 + NH,
              O_B3 = O_W3 + NH;

__device__ __forceinline__ uint32_t hash32(uint32_t x)
{
    x ^= x >> 16; x *= 0x7feb352dU; x ^= x >> 15; x *= 0x846ca68bU; x ^= x >> 16;
    return x;
}

// three-input max / min (one instruction each on sm_100 and later)
__device__ __forceinline__ float max3f(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float min3f(float a, float b, float c)
{
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// ------------------------------------------------------------- features
// Computes the 67 inputs, the CIR value m and the scale s of one cell from a
// periodic field; phi is read through `at(x, y, z)` (wrapped by the caller).
template <typename At>
__device__ __forceinline__ void cell_features(At at, int x, int y, int z, float cx, float cy, float cz,
                                              float (&feat)[NIN], float &m, float &s)
{
    const float X[3] = {x - cx, y - cy, z - cz};
    const int I[3] = {x, y, z};
    int b[3];
    float f[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        int fl = (int)floorf(X[d]);
        if (fl > I[d]) fl = I[d];
        b[d] = fl;
        f[d] = X[d] - (float)fl;
    }
    float v[64];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int bb = 0; bb < 4; ++bb)
#pragma unroll
            for (int a = 0; a < 4; ++a) v[a + 4 * bb + 16 * c] = at(b[0] - 1 + a, b[1] - 1 + bb, b[2] - 1 + c);
    // trilinear value of the inner cube (indices 1, 2 on each axis)
    float e[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {   // (y, z) pairs of the inner cube
        const int yy = 1 + (q & 1), zz = 1 + (q >> 1);
        const float lo = v[1 + 4 * yy + 16 * zz], hi = v[2 + 4 * yy + 16 * zz];
        e[q] = lo + f[0] * (hi - lo);
    }
    const float g0 = e[0] + f[1] * (e[1] - e[0]);
    const float g1 = e[2] + f[1] * (e[3] - e[2]);
    m = g0 + f[2] * (g1 - g0);
    // max |v_k - m| = max(max v - m, m - min v): rounding is monotonic, so this
    // is exactly the largest rounded difference; four chains each for ILP
    float hi[4], lo[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {   // chain c: v[c], v[c + 4], ..., v[c + 60]
        hi[c] = lo[c] = v[c + 60];
#pragma unroll
        for (int k = c; k < 60; k += 8) {
            hi[c] = max3f(hi[c], v[k], v[k + 4]);
            lo[c] = min3f(lo[c], v[k], v[k + 4]);
        }
    }
    const float vmax = fmaxf(fmaxf(hi[0], hi[1]), fmaxf(hi[2], hi[3]));
    const float vmin = fminf(fminf(lo[0], lo[1]), fminf(lo[2], lo[3]));
    s = fmaxf(fmaxf(vmax - m, m - vmin), 1e-30f);
    const float inv = 1.f / s;
    // feat = (v - m) / s as v inv - m inv, two cells' worth per packed FFMA2
    const float2 inv2 = make_float2(inv, inv), nm2 = make_float2(-m * inv, -m * inv);
#pragma unroll
    for (int k = 0; k < 64; k += 2) {
        const float2 r = __ffma2_rn(make_float2(v[k], v[k + 1]), inv2, nm2);
        feat[k] = r.x;
        feat[k + 1] = r.y;
    }
    feat[64] = f[0] - 0.5f;
    feat[65] = f[1] - 0.5f;
    feat[66] = f[2] - 0.5f;
}

__device__ __forceinline__ int wrapc(int v, int n)
{
    v %= n;
    return v < 0 ? v + n : v;
}

// Training samples at pseudo-random cells: rows of 68 floats (67 inputs, target
// y = (target_field - m) / s).
__global__ void k_samples(const float *__restrict__ phi, const float *__restrict__ target,
                          const float *__restrict__ vel, int nx, int ny, int nz, float sx, float sy, float sz,
                          int nsamples, uint32_t seed, float *__restrict__ rows)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nsamples) return;
    const int64_t plane = (int64_t)nx * ny, ncell = plane * nz;
    const uint32_t h = hash32(seed * 0x9E3779B9u + (uint32_t)j);
    const int64_t cell = (int64_t)(((uint64_t)h * (uint64_t)hash32(h ^ 0x5bd1e995u)) % (uint64_t)ncell);
    const int z = (int)(cell / plane), y = (int)((cell / nx) % ny), x = (int)(cell % nx);
    auto at = [&](int xx, int yy, int zz) {
        return phi[(int64_t)wrapc(zz, nz) * plane + (int64_t)wrapc(yy, ny) * nx + wrapc(xx, nx)];
    };
    float feat[NIN], m, s;
    cell_features(at, x, y, z, vel[cell] * sx, vel[ncell + cell] * sy, vel[2 * ncell + cell] * sz, feat, m, s);
    float *r = rows + (int64_t)j * 68;
#pragma unroll
    for (int k = 0; k < NIN; ++k) r[k] = feat[k];
    r[67] = (target[cell] - m) / s;
}

// --------------------------------------------------------------- training
// One minibatch: each CTA takes SB samples, runs forward and backward in FP32
// and adds its parameter gradients (and squared-error sum) into grad/loss.
constexpr int SB = 64, TT = 256;

__global__ void __launch_bounds__(TT) k_train(const float *__restrict__ params, const float *__restrict__ rows,
                                              int nrows, int batch, uint32_t seed, float *__restrict__ grad,
                                              float *__restrict__ loss)
{
    extern __shared__ __align__(16) float sm[];
    float *W = sm;                         // parameters, NPARAM
    float *X = W + ((NPARAM + 3) & ~3);    // SB x 68
    float *H1 = X + SB * 68;               // SB x NH
    float *H2 = H1 + SB * NH;
    float *D2 = H2 + SB * NH;              // dL/d(pre-activation 2)
    float *D1 = D2 + SB * NH;              // dL/d(pre-activation 1)
    float *DY = D1 + SB * NH;              // SB
    const int tid = threadIdx.x;
    for (int i = tid; i < NPARAM; i += TT) W[i] = params[i];
    const int s0 = blockIdx.x * SB;
    for (int i = tid; i < SB * 68; i += TT) {
        const int sidx = s0 + i / 68;
        float v = 0.f;
        if (sidx < batch) {
            const uint32_t r = hash32(seed * 0x85ebca6bu + (uint32_t)sidx) % (uint32_t)nrows;
            v = rows[(int64_t)r * 68 + i % 68];
        }
        X[i] = v;
    }
    __syncthreads();
    // layer 1
    for (int i = tid; i < SB * NH; i += TT) {
        const int s = i / NH, j = i % NH;
        float a = W[O_B1 + j];
        const float *w = W + O_W1 + j * NIN;
        const float *x = X + s * 68;
        for (int k = 0; k < NIN; ++k) a += w[k] * x[k];
        H1[i] = fmaxf(a, 0.f);
    }
    __syncthreads();
    for (int i = tid; i < SB * NH; i += TT) {
        const int s = i / NH, j = i % NH;
        float a = W[O_B2 + j];
        const float *w = W + O_W2 + j * NH;
        const float *h = H1 + s * NH;
        for (int k = 0; k < NH; ++k) a += w[k] * h[k];
        H2[i] = fmaxf(a, 0.f);
    }
    __syncthreads();
    if (tid < SB) {
        float y = W[O_B3];
        for (int k = 0; k < NH; ++k) y += W[O_W3 + k] * H2[tid * NH + k];
        const bool valid = s0 + tid < batch;
        const float e = valid ? y - X[tid * 68 + 67] : 0.f;
        DY[tid] = 2.f * e / (float)batch;
        atomicAdd(loss, e * e);
    }
    __syncthreads();
    for (int i = tid; i < SB * NH; i += TT) {
        const int s = i / NH, j = i % NH;
        D2[i] = H2[i] > 0.f ? DY[s] * W[O_W3 + j] : 0.f;
    }
    __syncthreads();
    for (int i = tid; i < SB * NH; i += TT) {
        const int s = i / NH, k = i % NH;
        float a = 0.f;
        for (int j = 0; j < NH; ++j) a += D2[s * NH + j] * W[O_W2 + j * NH + k];
        D1[i] = H1[i] > 0.f ? a : 0.f;
    }
    __syncthreads();
    // parameter gradients summed over the CTA's samples
    for (int p = tid; p < NPARAM; p += TT) {
        float g = 0.f;
        if (p < O_B1) {
            const int j = p / NIN, k = p % NIN;
            for (int s = 0; s < SB; ++s) g += D1[s * NH + j] * X[s * 68 + k];
        } else if (p < O_W2) {
            const int j = p - O_B1;
            for (int s = 0; s < SB; ++s) g += D1[s * NH + j];
        } else if (p < O_B2) {
            const int j = (p - O_W2) / NH, k = (p - O_W2) % NH;
            for (int s = 0; s < SB; ++s) g += D2[s * NH + j] * H1[s * NH + k];
        } else if (p < O_W3) {
            const int j = p - O_B2;
            for (int s = 0; s < SB; ++s) g += D2[s * NH + j];
        } else if (p < O_B3) {
            const int j = p - O_W3;
            for (int s = 0; s < SB; ++s) g += DY[s] * H2[s * NH + j];
        } else {
            for (int s = 0; s < SB; ++s) g += DY[s];
        }
        atomicAdd(grad + p, g);
    }
}

// Adam step on the FP32 parameters; clears the gradient.
__global__ void k_adam(float *__restrict__ params, float *__restrict__ grad, float *__restrict__ mom,
                       float *__restrict__ var, float lr, float b1, float b2, float eps, float c1, float c2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NPARAM) return;
    const float g = grad[i];
    const float m = b1 * mom[i] + (1.f - b1) * g;
    const float v = b2 * var[i] + (1.f - b2) * g * g;
    mom[i] = m;
    var[i] = v;
    params[i] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
    grad[i] = 0.f;
}

// ------------------------------------------------- inference (tensor cores)
// Shared-memory operand layout (no swizzle, K-major): 8 x 16-byte core
// matrices; the core matrix of rows [8r, 8r+8) and K elements [8k, 8k+8) sits
// at ((k * RG + r) * 128) bytes, RG = rows / 8.  Hence the byte distance
// between core matrices adjacent along K ("leading") is RG * 128 and along
// M/N ("stride") is 128.
__device__ __forceinline__ uint32_t core_off(int row, int kg, int rg) { return (uint32_t)((kg * rg + row / 8) * 128 + (row % 8) * 16); }

__host__ __device__ constexpr uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    // start >> 4 in bits 0-13, leading offset >> 4 in 16-29, stride offset >> 4
    // in 32-45, descriptor version 1 in bits 46-47, no swizzle (bits 61-63 = 0)
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor of kind::f16 with BF16 A and B, FP32 accumulator,
// both operands K-major, shape M x N.
__host__ __device__ constexpr uint32_t instr_desc(int M, int N)
{
    return (1u << 4)                          // D format: F32
           | (1u << 7)                        // A format: BF16
           | (1u << 10)                       // B format: BF16
           | ((uint32_t)(N >> 3) << 17)       // N / 8
           | ((uint32_t)(M >> 4) << 24);      // M / 16
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, int accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

// The same with A in tensor memory: row = lane, two BF16 elements along K per column.
__device__ __forceinline__ void mma_bf16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t b, uint32_t idesc, int accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "r"(tmem_a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                     smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

__device__ __forceinline__ void mbar_init1(uint64_t *bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}

__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, unsigned parity)
{
    for (unsigned it = 0; it < (1u << 20); ++it) {
        unsigned ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// 32 lanes x 64 consecutive TMEM columns into v[0..64) (this thread's lane), both
// loads in flight before the wait.
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
// Waits for the loads; the registers pass through the wait, so that nothing reads
// them before it.
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                   "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]),
                   "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]),
                   "+r"(r[30]), "+r"(r[31])::"memory");
}
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, float (&v)[64])
{
    uint32_t a[32], b[32];
    tmem_ld32_issue(taddr, a);
    tmem_ld32_issue(taddr + 32, b);
    tmem_wait(a);
    tmem_wait(b);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        v[i] = __uint_as_float(a[i]);
        v[32 + i] = __uint_as_float(b[i]);
    }
}

// 16 consecutive TMEM columns of this thread's lane <- r; tmem_wait_st before they are read.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n" ::"r"(
            taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// pack_bf16(max(a, 0), max(b, 0)) in one conversion (rounding and the clamp at
// zero commute, so the result is the same)
__device__ __forceinline__ uint32_t pack_bf16_relu(float a, float b)
{
    uint32_t d;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    return d;
}

constexpr int MT = 128;                      // cells per tile (MMA M)
constexpr int BX = 32, BY = 4;               // tile = 32 x 4 cells of one plane
constexpr int HX = 64, HY = BY + 4, HZ = 5;   // staged block: x halo 4 (16-byte chunks), y, z halo 2
static_assert(BX == 32 && HY == 8 && MT == 128, "the staging threads' shares");
constexpr int KS = KP1 - NH;                                     // K columns 64..79, staged in shared memory
constexpr int A_BYTES = MT * KS * 2, W_BYTES = NH * KP1 * 2;   // operand images, K = 80 in both layers
constexpr int BLK_FLOATS = HX * HY * HZ;
constexpr int STAGE_FLOATS = BLK_FLOATS + 3 * MT;              // Phi block + the tile's three u components
// One CTA per SM of WGS warpgroups that share the weights; each warpgroup works
// on tiles of its own (its operands, staging buffers, mbarrier, 96 TMEM columns
// and named barrier), so that one's gathers and epilogues run under another's
// tensor-core and copy latencies.
//  - A's columns 0 to 63 go from registers to tensor memory (BF16 pairs, one row per
//    lane) and are read there by the MMAs of both layers; only columns 64 to 79 pass
//    through shared memory, once.
//  - The biases enter through the GEMMs: K is padded from 67 to 80 anyway, columns
//    67 to 69 are 1, and the weight images hold each bias there as three BF16
//    parts that add up to its 24 bits.  Layer 2 overwrites columns 0 to 63 and leaves
//    those behind them as they are (its weights for columns 64 to 66 are zero).
//  - Layer 2 accumulates into the TMEM columns of layer 1, which the epilogue
//    between them has read.
//  - Rows of the staged block are 64 floats apart: a cell's bank depends on x alone,
//    so neighbours that step to different rows do not collide.
// What bounds it: instruction issue (about 60% of the cycles) with waits at the
// barriers of a tile's two GEMMs; registers allow no sixth warpgroup (80 each spill,
// 786 us).  Measured, 256^3: 825 us with four CTAs of one warpgroup and biases added
// from shared memory; 688 with five warpgroups in one CTA, 666 with 64 accumulators
// per TMEM read, 628 with A in tensor memory, 571 with whole lines per copy
// instruction and no divisions in the staging, 559 with rows 64 floats apart.
// Blocks staged two tiles ahead and one barrier less per tile took 568.
constexpr int WGS = 5, NT_STEP = WGS * MT, TM_COLS = 512, TM_WG = NH + NH / 2;   // D, then A's columns 0..63
static_assert(WGS * TM_WG <= TM_COLS, "tensor-memory columns of the warpgroups");
constexpr int S_A = 0, S_W1 = S_A + WGS * A_BYTES, S_W2 = S_W1 + W_BYTES;   // operands on 128-byte boundaries
constexpr int S_BLK = S_W2 + W_BYTES;                         // two stages per warpgroup
constexpr int S_F = S_BLK + WGS * 2 * 4 * STAGE_FLOATS;       // w3, b3 in FP32
constexpr int S_BAR = S_F + 4 * (NH + 4);
constexpr int S_TM = S_BAR + (8 * WGS + 15) / 16 * 16;
constexpr int SMEM_BYTES = S_TM + 16;
static_assert(A_BYTES % 128 == 0 && W_BYTES % 128 == 0 && S_F % 16 == 0, "alignment");
// a second resident CTA would wait forever for tensor-memory columns; its shared
// memory (with the 1 KB per-CTA reserve) cannot fit in the SM's 228 KB
static_assert(2 * (SMEM_BYTES + 1024) > 228 * 1024 && SMEM_BYTES <= 227 * 1024, "one resident CTA");

// The barrier of one warpgroup, and the same with an OR over its threads.
__device__ __forceinline__ void wg_sync(int g) { asm volatile("barrier.cta.sync %0, 128;\n" ::"r"(g + 1) : "memory"); }
__device__ __forceinline__ bool wg_or(int g, bool v)
{
    unsigned r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.or.pred q, %2, 128, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(r)
        : "r"((unsigned)v), "r"(g + 1)
        : "memory");
    return r != 0;
}

// One learned step over the grid; one cell per thread per tile.  wb points at
// the BF16 operand images of W1 and W2 (already in the core-matrix layout, biases
// included) followed by w3, b3 in FP32.
// A CTA's warpgroups take neighbouring tiles; SPREAD, for grids of at most a tile per
// warpgroup of the GPU: the CTAs take tiles in turn first, so that all SMs get some (32 x 16
// x 8: 7.2 us by neighbours, 5.4 in turn).  Two kernels: chosen at run time the order
// costs registers that spill (256^3 557 -> 614 us).
template <bool SPREAD>
__global__ void __launch_bounds__(NT_STEP, 1)
k_learned_step(const float *__restrict__ phi, float *__restrict__ out, const float *__restrict__ vel, int nx, int ny,
               int nz, float sx, float sy, float sz, const unsigned char *__restrict__ wb, unsigned *status)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    const int wg = threadIdx.x >> 7, tid = threadIdx.x & (MT - 1), warp = tid >> 5;   // within the warpgroup
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + S_BAR) + wg;
    uint32_t *tm_slot = reinterpret_cast<uint32_t *>(smem + S_TM);
    float *fw = reinterpret_cast<float *>(smem + S_F);
    float *blk = reinterpret_cast<float *>(smem + S_BLK) + wg * 2 * STAGE_FLOATS;
    unsigned char *A = smem + S_A + wg * A_BYTES;
    const int64_t plane = (int64_t)nx * ny, ncell = plane * nz;

    // weights once per CTA (operand images are copied verbatim)
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(wb);
        uint4 *dst = reinterpret_cast<uint4 *>(smem + S_W1);
        for (int i = threadIdx.x; i < 2 * W_BYTES / 16; i += NT_STEP) dst[i] = src[i];
        const float *fsrc = reinterpret_cast<const float *>(wb + 2 * W_BYTES);
        for (int i = threadIdx.x; i < NH + 1; i += NT_STEP) fw[i] = fsrc[i];
        *reinterpret_cast<uint4 *>(A + core_off(tid, 1, MT / 8)) = make_uint4(0u, 0u, 0u, 0u);   // columns 72..79
    }
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tm_slot)),
                     "n"(TM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
    }
    if (tid == 0) mbar_init1(bar);
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tm_slot + wg * TM_WG, tmem_a = tmem + NH;
    const uint32_t lanes = (uint32_t)(warp * 32) << 16;
    const uint32_t idesc = instr_desc(MT, NH);
    const uint32_t a0 = smem_u32(A), w1 = smem_u32(smem + S_W1), w2 = smem_u32(smem + S_W2);
    unsigned phase = 0;
    bool timeout = false;

    // tile (tx, ty, z) of this warpgroup, and the step to its next one
    const int tiles_x = nx / BX, tiles_y = ny / BY;
    const int64_t ntiles = (int64_t)tiles_x * tiles_y * nz, hop = (int64_t)gridDim.x * WGS;
    const int64_t first = SPREAD ? (int64_t)wg * gridDim.x + blockIdx.x : (int64_t)blockIdx.x * WGS + wg;
    const int hx = (int)(hop % tiles_x), hy = (int)(hop / tiles_x % tiles_y), hz = (int)(hop / ((int64_t)tiles_x * tiles_y));
    int tx = (int)(first % tiles_x), ty = (int)(first / tiles_x % tiles_y), z = (int)(first / ((int64_t)tiles_x * tiles_y));
    auto advance = [&](int &x, int &y, int &zz) {
        x += hx;
        y += hy;
        zz += hz;
        if (x >= tiles_x) {
            x -= tiles_x;
            ++y;
        }
        if (y >= tiles_y) {
            y -= tiles_y;
            ++zz;
        }
    };
    // the Phi block x in [x0-4, x0+36), y in [y0-2, y0+6), z in [z-2, z+3) and
    // the tile's velocity, staged with cp.async one tile ahead.  nx is a multiple of
    // 32, so a 16-byte chunk never straddles the periodic seam and every source is
    // aligned.  Chunk c of the 32 inner cells of rows (y, z) = (r, q), (r, q + 2),
    // (r, q + 4): eight threads read a whole line of a row; then the outer chunks,
    // two per row, by the first 80 threads.
    auto issue_block = [&](int tx_, int ty_, int z_, int b) {
        float *dst = blk + b * STAGE_FLOATS;
        auto wrapped = [](int v, int n) { return v + (v < 0 ? n : (v >= n ? -n : 0)); };   // at most one period away
        const int c = tid & 7, r = (tid >> 3) & 7, q = tid >> 6;
        const float *src = phi + (int64_t)wrapped(ty_ * BY - 2 + r, ny) * nx + tx_ * BX + 4 * c;
        float *d = dst + (q * HY + r) * HX + 4 + 4 * c;
#pragma unroll
        for (int k = 0; k < HZ; k += 2)
            if (q + k < HZ) cp_async16(d + k * HY * HX, src + wrapped(z_ - 2 + q + k, nz) * plane);
        if (tid < 2 * HY * HZ) {
            const int er = (tid >> 1) & 7, ez = tid >> 4, ex = (tid & 1) * (BX + 4);
            cp_async16(dst + (ez * HY + er) * HX + ex, phi + wrapped(z_ - 2 + ez, nz) * plane +
                                                           (int64_t)wrapped(ty_ * BY - 2 + er, ny) * nx +
                                                           wrapped(tx_ * BX - 4 + ex, nx));
        }
        const float *v = vel + (z_ * plane + (int64_t)(ty_ * BY + tid / BX) * nx + tx_ * BX + tid % BX);
        cp_async4(dst + BLK_FLOATS + tid, v);
        cp_async4(dst + BLK_FLOATS + MT + tid, v + ncell);
        cp_async4(dst + BLK_FLOATS + 2 * MT + tid, v + 2 * ncell);
        cp_async_commit();
    };
    // D = A (128 x 80) * W^T, both operands K-major, issued by one thread: columns
    // 64..79 of A first (shared memory), then 0..63 (tensor memory)
    auto gemm = [&](uint32_t w) {
        if (tid == 0) {
            auto db = [&](int k) { return smem_desc(w + k * 2 * (NH / 8) * 128, (NH / 8) * 128, 128); };
            mma_bf16(tmem, smem_desc(a0, (MT / 8) * 128, 128), db(NH / 16), idesc, 0);
#pragma unroll
            for (int k = 0; k < NH / 16; ++k) mma_bf16_ta(tmem, tmem_a + k * 8, db(k), idesc, 1);
            mma_commit(bar);
        }
        if (!mbar_wait_bounded(bar, phase)) timeout = true;
        phase ^= 1u;
        tc_fence_after();
    };
    if (first < ntiles) issue_block(tx, ty, z, 0);
    int it = 0;
    for (int64_t t = first; t < ntiles; t += hop, ++it) {
        const int x0 = tx * BX, y0 = ty * BY, z0 = z;
        const float *sb = blk + (it & 1) * STAGE_FLOATS;
        cp_async_wait_all();
        timeout = wg_or(wg, timeout);   // the block is there, and every warp is done with the tile before
        if (timeout) break;
        advance(tx, ty, z);
        if (t + hop < ntiles) issue_block(tx, ty, z, (it & 1) ^ 1);
        // ---- features of this thread's cell -> row tid of A (BF16)
        const int cxl = tid % BX, cyl = tid / BX;
        const int64_t cell = (int64_t)z0 * plane + (int64_t)(y0 + cyl) * nx + x0 + cxl;
        const float cx = sb[BLK_FLOATS + tid] * sx, cy = sb[BLK_FLOATS + MT + tid] * sy,
                    cz = sb[BLK_FLOATS + 2 * MT + tid] * sz;
        if (fabsf(cx) > 1.f || fabsf(cy) > 1.f || fabsf(cz) > 1.f) atomicOr(status, 1u);
        const float ccx = fminf(fmaxf(cx, -1.f), 1.f), ccy = fminf(fmaxf(cy, -1.f), 1.f),
                    ccz = fminf(fmaxf(cz, -1.f), 1.f);
        auto at = [&](int xx, int yy, int zz) {
            // xx, yy, zz are global indices within 2 cells of the cell
            return sb[((zz - z0 + 2) * HY + (yy - y0 + 2)) * HX + (xx - x0 + 4)];
        };
        float feat[NIN], m, s;
        cell_features(at, x0 + cxl, y0 + cyl, z0, ccx, ccy, ccz, feat, m, s);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t q[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) q[k] = pack_bf16(feat[32 * h + 2 * k], feat[32 * h + 2 * k + 1]);
            tmem_st16(tmem_a + lanes + 16 * h, q);
        }
        // columns 67..69 are the biases' ones
        *reinterpret_cast<uint4 *>(A + core_off(tid, 0, MT / 8)) =
            make_uint4(pack_bf16(feat[64], feat[65]), pack_bf16(feat[66], 1.f), pack_bf16(1.f, 1.f), 0u);
        tmem_wait_st();
        fence_async_smem();
        tc_fence_before();
        wg_sync(wg);
        tc_fence_after();
        gemm(w1);
        // ---- epilogue 1: ReLU, BF16 -> columns 0..63 of A
        {
            float v[NH];
            tmem_ld64(tmem + lanes, v);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t q[16];
#pragma unroll
                for (int k = 0; k < 16; ++k)   // ReLU folded into the conversion
                    q[k] = pack_bf16_relu(v[32 * h + 2 * k], v[32 * h + 2 * k + 1]);
                tmem_st16(tmem_a + lanes + 16 * h, q);
            }
            tmem_wait_st();
        }
        tc_fence_before();
        wg_sync(wg);
        tc_fence_after();
        gemm(w2);
        // ---- epilogue 2: ReLU, output layer, Phi_new = m + s y
        float2 ya01 = make_float2(fw[NH], 0.f), ya23 = make_float2(0.f, 0.f);   // four accumulation chains
        {
            float v[NH];
            tmem_ld64(tmem + lanes, v);
            const float4 *w3v = reinterpret_cast<const float4 *>(fw);
#pragma unroll
            for (int q = 0; q < NH / 4; ++q) {
                const float4 ww = w3v[q];
                const float2 h01 = make_float2(fmaxf(v[4 * q], 0.f), fmaxf(v[4 * q + 1], 0.f));
                const float2 h23 = make_float2(fmaxf(v[4 * q + 2], 0.f), fmaxf(v[4 * q + 3], 0.f));
                ya01 = __ffma2_rn(h01, make_float2(ww.x, ww.y), ya01);
                ya23 = __ffma2_rn(h23, make_float2(ww.z, ww.w), ya23);
            }
        }
        const float y = (ya01.x + ya01.y) + (ya23.x + ya23.y);
        out[cell] = m + s * y;
    }
    cp_async_wait_all();   // a block prefetched for a tile that was not run
    if (timeout) atomicOr(status, 2u);
    __syncthreads();
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(*tm_slot), "n"(TM_COLS));
}

// Failure-detection self-test: waits on an mbarrier that no thread or copy
// ever completes, gives up after `polls` polls like every bounded wait of the
// library, and records SL_DEV_TIMEOUT.  Faults, traps or hangs nothing.
__global__ void k_wait_selftest(unsigned polls, unsigned *status, unsigned *gave_up)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) mbar_init1(&bar);   // expects one arrival that never comes
    __syncthreads();
    bool ok = false;
    for (unsigned it = 0; it < polls && !ok; ++it) {
        unsigned r;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(r)
            : "r"(smem_u32(&bar)), "r"(0u)
            : "memory");
        ok = r != 0;
    }
    if (!ok && threadIdx.x == 0) {
        atomicOr(status, 2u);
        atomicAdd(gave_up, 1u);
    }
}

// Element (n, k) of a layer's weight image: its weight for k < nin, for k = 67 to
// 69 the three BF16 parts of its bias (cut off, not rounded, so that they add up to
// the FP32 value; a bias that is not finite stays whole), else 0.
__device__ __forceinline__ float image_value(const float *w, const float *b, int nin, int n, int k)
{
    if (k < nin) return w[n * nin + k];
    if (k < NIN || k >= NIN + 3) return 0.f;
    const float v = b[n];
    if (!isfinite(v)) return k == NIN ? v : 0.f;
    const float hi = __uint_as_float(__float_as_uint(v) & 0xffff0000u), r = v - hi;
    const float mid = __uint_as_float(__float_as_uint(r) & 0xffff0000u);
    return k == NIN ? hi : (k == NIN + 1 ? mid : r - mid);
}

// FP32 parameters -> the inference weight image: W1 and W2 (64 x 80 each, biases
// in columns 67 to 69) as BF16 K-major core matrices, then w3, b3 in FP32.
__global__ void k_pack(const float *__restrict__ params, unsigned char *__restrict__ wb)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    __nv_bfloat16 *w1 = reinterpret_cast<__nv_bfloat16 *>(wb);
    __nv_bfloat16 *w2 = reinterpret_cast<__nv_bfloat16 *>(wb + W_BYTES);
    float *f = reinterpret_cast<float *>(wb + 2 * W_BYTES);
    if (i < NH * KP1) {
        const int n = i / KP1, k = i % KP1, o = core_off(n, k / 8, NH / 8) / 2 + k % 8;
        w1[o] = __float2bfloat16_rn(image_value(params + O_W1, params + O_B1, NIN, n, k));
        w2[o] = __float2bfloat16_rn(image_value(params + O_W2, params + O_B2, NH, n, k));
    }
    if (i < NH) f[i] = params[O_W3 + i];
    if (i == 0) f[NH] = params[O_B3];
}

}  // namespace lrn
}  // namespace sl

// ============================================================== host side
using namespace sl;
using namespace sl::lrn;

struct sl_corrector {
    int device = -1;
    float *params = nullptr;   // NPARAM FP32 (layout: W1 64x67, b1, W2 64x64, b2, w3, b3)
    float *grad = nullptr;
    float *mom = nullptr;
    float *var = nullptr;
    float *loss = nullptr;     // 1 float
    unsigned char *wb = nullptr;   // inference weight image
    float *rows = nullptr;     // training rows, 68 floats each
    int64_t nrows = 0, cap = 0;
    int64_t adam_t = 0;
    void *scratch = nullptr;   // two fields for the checked step
    size_t scratch_bytes = 0;
    bool plain = false;        // sticky fallback to the plain scheme
};

namespace {

int lfail(int code, const char *msg) { return set_error(code, msg); }

bool learned_geometry_ok(int ndim, const int64_t dims[3]) {
    return ndim == 3 && dims[0] % BX == 0 && dims[1] % BY == 0 && dims[2] >= 3 && dims[0] >= 32 && dims[1] >= 4;
}

int pack(sl_corrector *c, cudaStream_t st) {
    k_pack<<<(NH * KP1 + 255) / 256, 256, 0, st>>>(c->params, c->wb);
    return cudaGetLastError() == cudaSuccess ? SL_OK : lfail(SL_ERR_CUDA, "weight packing launch failed");
}

}  // namespace

extern "C" {

int sl_corrector_create(sl_corrector **out, uint64_t seed)
{
    if (!out) return lfail(SL_ERR_ARG, "out must not be NULL");
    *out = nullptr;
    DevCtx *ctx = ctx_get();
    if (!ctx) return lfail(SL_ERR_CUDA, "could not create the device context");
    sl_corrector *c = new (std::nothrow) sl_corrector();
    if (!c) return lfail(SL_ERR_NOMEM, "host allocation");
    c->device = ctx->device;
    const size_t wbytes = 2 * W_BYTES + 4 * (NH + 4);
    void *p = nullptr;
    if (cudaMalloc(&p, 4 * (size_t)NPARAM * 4 + 256 + wbytes) != cudaSuccess) {
        delete c;
        return lfail(SL_ERR_NOMEM, "device parameters");
    }
    c->params = static_cast<float *>(p);
    c->grad = c->params + NPARAM;
    c->mom = c->grad + NPARAM;
    c->var = c->mom + NPARAM;
    c->loss = c->var + NPARAM;
    c->wb = reinterpret_cast<unsigned char *>(c->var + NPARAM) + 256;
    // He initialisation, zero biases (host RNG, seeded)
    std::vector<float> h(NPARAM, 0.f);
    std::mt19937_64 rng(seed);
    std::normal_distribution<float> nd(0.f, 1.f);
    for (int i = 0; i < NH * NIN; ++i) h[O_W1 + i] = nd(rng) * std::sqrt(2.f / NIN);
    for (int i = 0; i < NH * NH; ++i) h[O_W2 + i] = nd(rng) * std::sqrt(2.f / NH);
    for (int i = 0; i < NH; ++i) h[O_W3 + i] = nd(rng) * std::sqrt(1.f / NH);
    cudaError_t e = cudaMemcpy(c->params, h.data(), 4 * NPARAM, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(c->grad, 0, 4 * (size_t)NPARAM * 3 + 4);
    if (e != cudaSuccess || pack(c, nullptr) != SL_OK || cudaDeviceSynchronize() != cudaSuccess) {
        cudaFree(p);
        delete c;
        return lfail(SL_ERR_CUDA, "corrector initialisation");
    }
    *out = c;
    return SL_OK;
}

int sl_corrector_destroy(sl_corrector *c)
{
    if (!c) return SL_OK;
    cudaFree(c->params);
    if (c->rows) cudaFree(c->rows);
    if (c->scratch) cudaFree(c->scratch);
    delete c;
    return SL_OK;
}

int sl_corrector_param_count(void) { return NPARAM; }

int sl_corrector_get_params(sl_corrector *c, float *host, int n)
{
    if (!c || !host || n != NPARAM) return lfail(SL_ERR_ARG, "need the corrector and a buffer of sl_corrector_param_count() floats");
    return cudaMemcpy(host, c->params, 4 * NPARAM, cudaMemcpyDeviceToHost) == cudaSuccess ? SL_OK
                                                                                         : lfail(SL_ERR_CUDA, "copy");
}

int sl_corrector_set_params(sl_corrector *c, const float *host, int n)
{
    if (!c || !host || n != NPARAM) return lfail(SL_ERR_ARG, "need the corrector and sl_corrector_param_count() floats");
    if (cudaMemcpy(c->params, host, 4 * NPARAM, cudaMemcpyHostToDevice) != cudaSuccess) return lfail(SL_ERR_CUDA, "copy");
    c->plain = false;
    int rc = pack(c, nullptr);
    if (rc) return rc;
    return cudaDeviceSynchronize() == cudaSuccess ? SL_OK : lfail(SL_ERR_CUDA, "weight packing");
}

int sl_corrector_add_samples(sl_corrector *c, const void *phi, const void *target, const void *vel,
                             const int64_t dims[3], const double spacing[3], double dt, int nsamples, uint64_t seed,
                             void *stream)
{
    if (!c || !phi || !target || !vel || !dims || !spacing || nsamples < 1)
        return lfail(SL_ERR_ARG, "NULL argument or nsamples < 1");
    for (int d = 0; d < 3; ++d)
        if (dims[d] < 1 || !(spacing[d] > 0.0)) return lfail(SL_ERR_ARG, "bad dims or spacing");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (c->nrows + nsamples > c->cap) {
        const int64_t ncap = std::max<int64_t>(2 * c->cap, c->nrows + nsamples);
        float *nr = nullptr;
        if (cudaMalloc(&nr, (size_t)ncap * 68 * 4) != cudaSuccess) return lfail(SL_ERR_NOMEM, "sample buffer");
        if (c->rows) {
            if (cudaMemcpyAsync(nr, c->rows, (size_t)c->nrows * 68 * 4, cudaMemcpyDeviceToDevice, st) != cudaSuccess ||
                cudaStreamSynchronize(st) != cudaSuccess) {
                cudaFree(nr);
                return lfail(SL_ERR_CUDA, "sample copy");
            }
            cudaFree(c->rows);
        }
        c->rows = nr;
        c->cap = ncap;
    }
    k_samples<<<(nsamples + 255) / 256, 256, 0, st>>>(
        static_cast<const float *>(phi), static_cast<const float *>(target), static_cast<const float *>(vel),
        (int)dims[0], (int)dims[1], (int)dims[2], (float)(dt / spacing[0]), (float)(dt / spacing[1]),
        (float)(dt / spacing[2]), nsamples, (uint32_t)(seed ^ (seed >> 32)), c->rows + c->nrows * 68);
    if (cudaGetLastError() != cudaSuccess) return lfail(SL_ERR_CUDA, "sample launch");
    c->nrows += nsamples;
    return SL_OK;
}

int sl_corrector_get_rows(sl_corrector *c, float *host, int64_t first, int64_t n)
{
    if (!c || !host || first < 0 || n < 0 || first + n > c->nrows) return lfail(SL_ERR_ARG, "row range outside the training set");
    if (n == 0) return SL_OK;
    return cudaMemcpy(host, c->rows + first * 68, (size_t)n * 68 * 4, cudaMemcpyDeviceToHost) == cudaSuccess
               ? SL_OK
               : lfail(SL_ERR_CUDA, "copy");
}

int sl_corrector_train(sl_corrector *c, int iters, int batch, float lr, uint64_t seed, float *last_loss, void *stream)
{
    if (!c || iters < 1 || batch < 1 || !(lr > 0.f)) return lfail(SL_ERR_ARG, "bad training arguments");
    if (c->nrows < 1) return lfail(SL_ERR_ARG, "no training samples (sl_corrector_add_samples)");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t smem = 4 * (size_t)(((NPARAM + 3) & ~3) + SB * 68 + 4 * SB * NH + SB);
    if (cudaFuncSetAttribute(k_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return lfail(SL_ERR_CUDA, "training kernel shared memory");
    const float b1 = 0.9f, b2 = 0.999f;
    for (int it = 0; it < iters; ++it) {
        ++c->adam_t;
        const float c1 = 1.f - std::pow(b1, (float)c->adam_t), c2 = 1.f - std::pow(b2, (float)c->adam_t);
        if (cudaMemsetAsync(c->loss, 0, 4, st) != cudaSuccess) return lfail(SL_ERR_CUDA, "memset");
        k_train<<<(batch + SB - 1) / SB, TT, smem, st>>>(c->params, c->rows, (int)std::min<int64_t>(c->nrows, 1 << 30),
                                                        batch, (uint32_t)(seed * 2654435761u + it), c->grad, c->loss);
        k_adam<<<(NPARAM + 255) / 256, 256, 0, st>>>(c->params, c->grad, c->mom, c->var, lr, b1, b2, 1e-8f, c1, c2);
    }
    int rc = pack(c, st);
    if (rc) return rc;
    float l = 0.f;
    if (cudaMemcpyAsync(&l, c->loss, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
        return lfail(SL_ERR_CUDA, "training");
    if (last_loss) *last_loss = l / (float)batch;
    return SL_OK;
}

int sl_selftest_wait_timeout(unsigned polls, void *stream)
{
    if (polls < 1 || polls > (1u << 20)) return lfail(SL_ERR_ARG, "polls must be in [1, 2^20]");
    DevCtx *ctx = ctx_get();
    if (!ctx) return lfail(SL_ERR_CUDA, "no device context");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned *gave_up = ctx->counters + 255;
    if (cudaMemsetAsync(gave_up, 0, 4, st) != cudaSuccess) return lfail(SL_ERR_CUDA, "memset");
    k_wait_selftest<<<1, 32, 0, st>>>(polls, ctx->status, gave_up);
    unsigned h = 0;
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpyAsync(&h, gave_up, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return lfail(SL_ERR_CUDA, "self-test launch");
    return h == 1 ? SL_ERR_TIMEOUT : lfail(SL_ERR_CUDA, "the self-test wait completed unexpectedly");
}

int sl_corrector_reset(sl_corrector *c)
{
    if (!c) return lfail(SL_ERR_ARG, "corrector is NULL");
    c->plain = false;
    return SL_OK;
}

int sl_advect_learned(sl_corrector *c, void *out, const void *in, const void *vel, int ndim, const int64_t dims[3],
                      const double spacing[3], double dt, int step_parity, int check, double fallback_ratio,
                      int *used_plain, double errs[2], void *stream)
{
    if (!c || !out || !in || !vel || !dims || !spacing) return lfail(SL_ERR_ARG, "NULL argument");
    if (!learned_geometry_ok(ndim, dims))
        return lfail(SL_ERR_UNSUPPORTED, "learned steps need ndim = 3, dims[0] % 32 == 0, dims[1] % 4 == 0, dims[2] >= 3");
    if (reinterpret_cast<uintptr_t>(in) % 16 != 0)
        return lfail(SL_ERR_UNSUPPORTED, "learned steps need a 16-byte aligned input field");
    for (int d = 0; d < 3; ++d)
        if (!(spacing[d] > 0.0)) return lfail(SL_ERR_ARG, "spacing must be > 0");
    const int64_t n = dims[0] * dims[1] * dims[2];
    const size_t fb = (size_t)n * 4;
    const char *po = static_cast<const char *>(out), *pi = static_cast<const char *>(in);
    if (po < pi + fb && pi < po + fb) return lfail(SL_ERR_ALIAS, "out overlaps in");
    DevCtx *ctx = ctx_get();
    if (!ctx) return lfail(SL_ERR_CUDA, "no device context");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    auto learned = [&](void *dst) {
        const int64_t tiles = (dims[0] / BX) * (dims[1] / BY) * dims[2];
        const bool spread = tiles <= (int64_t)ctx->num_sms * WGS;
        const auto kern = spread ? k_learned_step<true> : k_learned_step<false>;
        static ResidencyCache cache[2];
        Residency res;
        const cudaError_t e = residency(cache[spread], kern, NT_STEP, SMEM_BYTES, true, res);
        if (e != cudaSuccess) return e;
        const int grid = tiles < res.sms ? (int)tiles : res.sms;   // one per SM: each holds its TMEM
        kern<<<grid, NT_STEP, SMEM_BYTES, st>>>(
            static_cast<const float *>(in), static_cast<float *>(dst), static_cast<const float *>(vel), (int)dims[0],
            (int)dims[1], (int)dims[2], (float)(dt / spacing[0]), (float)(dt / spacing[1]), (float)(dt / spacing[2]),
            c->wb, ctx->status);
        return cudaGetLastError();
    };
    if (used_plain) *used_plain = c->plain ? 1 : 0;
    if (!check) {
        if (c->plain) return sl_advect(out, in, vel, ndim, dims, spacing, dt, SL_CEC, SL_F32, step_parity, stream);
        return learned(out) == cudaSuccess ? SL_OK : lfail(SL_ERR_CUDA, "learned step launch");
    }
    // checked step: plain CEC into out, BEC and learned into scratch, compare
    if (c->scratch_bytes < 2 * fb + 256) {
        if (c->scratch) cudaFree(c->scratch);
        c->scratch = nullptr;
        c->scratch_bytes = 0;
        if (cudaMalloc(&c->scratch, 2 * fb + 256) != cudaSuccess) return lfail(SL_ERR_NOMEM, "check scratch");
        c->scratch_bytes = 2 * fb + 256;
    }
    char *s0 = static_cast<char *>(c->scratch);
    void *bec = s0, *lrn = s0 + ((fb + 255) & ~(size_t)255);
    int rc = sl_advect(out, in, vel, ndim, dims, spacing, dt, SL_CEC, SL_F32, step_parity, stream);
    if (rc) return rc;
    rc = sl_advect(bec, in, vel, ndim, dims, spacing, dt, SL_BEC, SL_F32, step_parity, stream);
    if (rc) return rc;
    if (learned(lrn) != cudaSuccess) return lfail(SL_ERR_CUDA, "learned step launch");
    double nl[3], np[3];
    rc = sl_norms(lrn, out, n, SL_F32, nl, stream);
    if (rc) return rc;
    rc = sl_norms(bec, out, n, SL_F32, np, stream);
    if (rc) return rc;
    if (errs) {
        errs[0] = nl[2];
        errs[1] = np[2];
    }
    if (!c->plain && nl[2] <= fallback_ratio * np[2]) {
        if (cudaMemcpyAsync(out, lrn, fb, cudaMemcpyDeviceToDevice, st) != cudaSuccess) return lfail(SL_ERR_CUDA, "copy");
    } else {
        c->plain = true;
    }
    if (used_plain) *used_plain = c->plain ? 1 : 0;
    return SL_OK;
}

}  // extern "C"
