// sl_internal.h -- declarations shared by the host entry points and the kernel
// translation units of libsl.  Not part of the public ABI (see include/sl.h).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "per_device.h"
#include "sl_common.cuh"

namespace sl {

// Per-device context: status word and small work areas.
struct DevCtx {
    int device = -1;
    unsigned *status = nullptr;      // SL_DEV_* bits
    double *partials = nullptr;      // reduction partials (kReduceBlocks x 4)
    unsigned *counters = nullptr;    // work counters for batched launches
    int num_sms = 0;
};

constexpr int kReduceBlocks = 1024;

DevCtx *ctx_get();   // context of the current device, created on demand

// Launch configuration chosen for a fused kernel.
struct Launch {
    int tz = 0;          // z chunk (planes per work item); 0 = default
    int ty = 0;          // column tile height among a kernel's compiled variants; 0 = default
    int grid = 0;        // CTAs; 0 = one per item (persistent kernels: their occupancy)
    bool aligned = true; // all base pointers 16-byte aligned (vector staging allowed)
    bool pdl = false;    // the kernel waits for its predecessor itself (kernels that know how)
};

// Launches kern; pdl: with programmatic stream serialisation, for a kernel that
// begins with pdl_wait() (sl_common.cuh).
template <typename... P, typename... A>
cudaError_t launch_kernel(void (*kern)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, bool pdl, A... args)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

// Shared-memory opt-in of a kernel on the current device (carveout: all of the SM's
// unified memory as shared, too) and its residency, once per device.
template <typename K>
cudaError_t residency(ResidencyCache &cache, K kern, int block, size_t smem, bool carveout, Residency &r)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= ResidencyCache::kDevices) return cudaErrorInvalidDevice;
    if (cache.get(dev, r)) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess && carveout) e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r.per_sm, kern, block, smem);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&r.sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (r.per_sm < 1) r.per_sm = 1;
    cache.set(dev, r);
    return cudaSuccess;
}

// Several fields advected by one velocity in one launch: field f reads
// in + f * fin and writes out + f * fout (elements); the launch's grid gains
// a y extent of n, and each field's CTAs do exactly what a launch for that
// field alone does.
struct FieldSet {
    int n = 1;
    int64_t fin = 0, fout = 0;
};

// Fused single-step kernels; return a cudaError_t of the launch.
cudaError_t launch_split_cec(int dtype, const void *in, void *out, const void *vel, int ndim,
                             const int64_t dims[3], const double s[3], int parity,
                             Launch lc, unsigned *status, cudaStream_t st, FieldSet fs = FieldSet());
// The same with double arithmetic (SL_F64, or float storage for SL_F32_D64);
// g carries the sizes, Courant factors and planes per work item (tz = 0: equal
// shares), its tiles are set by the launch (k_split64.cu).
cudaError_t launch_split_cec64(bool f32_storage, Geo g, int parity, Launch lc, bool has_z, const void *in, void *out,
                               const void *vel, const FieldSet &fs, cudaStream_t st);
int split64_tile_y(bool has_z, int64_t nx, int64_t ny, int fields);   // its tile height
cudaError_t launch_unsplit(int dtype, int scheme, const void *in, void *out, const void *vel,
                           int ndim, const int64_t dims[3], const double s[3], Launch lc,
                           unsigned *status, cudaStream_t st, FieldSet fs = FieldSet());
// The same for FP32 in 3D, any size and alignment (k_unsplit32.cu), and whether it
// serves a request (vec: 16-byte aligned buffers and rows of whole 16-byte
// chunks); g as for launch_split_cec64.
bool unsplit32_serves(int scheme, int ndim, const int64_t dims[3], bool vec);
cudaError_t launch_unsplit32(int scheme, Geo g, int grid, const void *in, void *out, const void *vel,
                             const FieldSet &fs, cudaStream_t st);
// FP32 3D CIR kernel on four-cell groups (k_cir_fast.cu); launch_unsplit routes
// eligible CIR steps to it.
bool cir_fast_eligible(int dtype, int ndim, const int64_t dims[3], bool aligned);
cudaError_t launch_cir_fast(const void *in, void *out, const void *vel, const int64_t dims[3], const double s[3],
                            Launch lc, unsigned *status, cudaStream_t st);

// Reductions (synchronous results through host pointers after a stream sync).
cudaError_t launch_norms(int dtype, const void *a, const void *b, int64_t n, double *partials,
                         cudaStream_t st);
cudaError_t launch_courant(int dtype, const void *vel, int ndim, int64_t n, const double s[3],
                           double *partials, cudaStream_t st);

// Batched persistent CEC step (FP32, 3D) over an instance table in device
// memory.  Record i owns global items [item0[par], item0[par] + items) of the
// x,y,z (par 0) or z,y,x (par 1) decomposition.
struct BatchRec {
    void *a;
    void *b;
    const void *vel;
    Geo g[2];
    int item0[2];
};
void batched_tiles(int parity, int &tx, int &ty);
int batched_blocks_per_sm(int parity);
cudaError_t launch_batched_cec(const BatchRec *dev_recs, int ninst, int nitems, int parity, unsigned *counter,
                               unsigned *status, int grid, cudaStream_t st);

int default_tz(int dtype, int ndim, const int64_t dims[3]);

// CTAs per field for a kernel whose CTAs take equal shares of the (column tile,
// plane) pairs of `tiles` tiles of nz planes and begin every run of planes with
// `warm` planes of warm-up.  A share that starts inside a tile and ends in the
// next warms up twice; tiles * c CTAs cut every tile into c runs of at most
// ceil(nz / c) planes that never do.  The cost of a choice is the planes its
// busiest CTA works on, warm-ups included, times what a plane takes with that many
// CTAs on an SM (two: 1, one: `alone`, k > 2: k / 2).
// Measured, CEC x,y,z / z,y,x us per step, equal shares of all resident CTAs and
// this: 187 x 150 x 131 59 / 68 and 49 / 58, 96^3 25 / 28 and 17.5 / 23, 192^3
// 58 / 72 and 51 / 68, 24 x 400 x 60 30 / 30 and 20 / 21.
int64_t plan_ctas(int64_t tiles, int64_t nz, int warm, double alone, int per_sm, int sms, int fields);

// Fast FP32 CEC path (k_cec_fast.cu): one periodic grid of whole 32 x 32 column
// tiles; w0 numbers its first (column tile, plane) pair in a batch.  A launch
// writes the output planes [zb, zb + nzr) (fast_fill: all nz planes) and reads
// the input planes [zb - 6, zb + nzr + 3), taken modulo nz.
// A single-instance launch may advance nf <= kFastFields fields with one
// velocity: its CTAs form groups of nf that take the same (column tile, plane)
// sequence, one field each, so the group's velocity reads are served from L2.
constexpr int kFastFields = 4;
struct FastInst {
    const float *in;
    float *out;
    const float *vel;
    int nx, ny, nz;
    int tiles_x, ntiles;
    int64_t plane, ncell;
    float sx, sy, sz;
    int64_t w0;
    const void *maps;   // batched tables: device address of this instance's tensor maps
    int zb, nzr;        // output planes [zb, zb + nzr); 0 <= zb, 1 <= nzr, zb + nzr <= nz
    int nf;             // fields (1 in batched tables); fin[0] = in, fout[0] = out
    const float *fin[kFastFields];
    float *fout[kFastFields];
};
// Input planes a fast launch reads below and above its output planes.
constexpr int kFastHaloBelow = 6, kFastHaloAbove = 3;
// Bytes of one instance's tensor maps (22 maps of the first field and the
// velocity, 9 for each further field; 128 bytes each, 64-byte aligned).
constexpr size_t kFastMapsBytes = (31 + 12 * (kFastFields - 1)) * 128;
// Encodes the tensor maps of an instance into dst (host memory, kFastMapsBytes).
cudaError_t fast_encode_maps(void *dst, const FastInst &f);
bool fast_eligible(const int64_t dims[3], int ndim, int dtype, bool aligned);
void fast_fill(FastInst &f, const void *in, void *out, const void *vel, const int64_t dims[3], const double s[3],
               int64_t w0);
cudaError_t launch_cec_fast(const FastInst &one, const FastInst *dev_table, int ninst, int64_t total, int parity,
                            unsigned *status, int grid_req, cudaStream_t st);
int fast_grid(int parity);
// The same kernels on FP32 3D grids of any x and y size and alignment (nz >= 8);
// lc.tz > 0: CTAs take shares of that many planes, except that any_default_tz planes
// stand for the kernels' own division (plan_ctas).  A tuned shape of this family is
// planes per work item, which the generic batched kernel takes too: its default, 32
// planes, there and here leaves each kernel its default.
bool any_eligible(const int64_t dims[3], int ndim, int dtype);
int any_default_tz(const int64_t dims[3]);
cudaError_t launch_cec_any(const void *in, void *out, const void *vel, const int64_t dims[3], const double s[3],
                           int parity, Launch lc, unsigned *status, const FieldSet &fs, cudaStream_t st);

// Steps at any Courant number (k_wide.cu): non-local interpolation, unfused
// kernels, intermediate fields in a caller-owned workspace of wide_fields()
// fields of wide_field_bytes() each (256-byte aligned).  Grids launch as
// (x blocks, ny, nz), so ny and nz must be at most 65535.
size_t wide_field_bytes(int64_t ncell, size_t elem);
int wide_fields(int scheme, int ndim);
cudaError_t launch_wide(int dtype, int scheme, const void *in, void *out, const void *vel, int ndim,
                        const int64_t dims[3], const double s[3], int parity, void *work, unsigned *status,
                        cudaStream_t st);

// sl_advect_multi; pdl as in Launch.
int advect_fields(void *const *outs, const void *const *ins, int nfields, const void *vel, int ndim,
                  const int64_t dims[3], const double spacing[3], double dt, int scheme, int dtype, int step_parity,
                  void *stream, bool pdl);

// Records a thread-local error message (read by sl_last_error) and returns code.
int set_error(int code, const char *msg);

// Largest element count sl_norms_static accepts.
constexpr int64_t kNormsStaticMaxElems = (int64_t)1 << 40;

}  // namespace sl
