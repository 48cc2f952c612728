// bridge.cu -- between the solver and the warm-start network: the training targets of a
// solved cavity, and a cavity started from the network's prediction (the equilibria of
// the predicted fields, lbm_set_fields), resampled trilinearly when the grids differ.
#include <algorithm>

#include "../context.h"
#include "lbm_net.h"
#include "nn.h"

using namespace lbm;

namespace {

// Trilinear resampling of a cell-centred m^3 prediction [voxel][4] onto the nx x ny x nz
// nodes of a context (node i at (i + 1/2) / nx of the box, clamped at the walls), scaled
// back to lattice units: u = p * U0, T = p / 2.
//
// FP64 arithmetic, of which GB300 issues two operations per clock and SM: the eight-corner sum
// per node took 0.57 ms at 64^3 -> 128^3 (three divisions, 32 conversions and 32 products a
// node).  A block therefore takes whole x-rows: the row of the prediction at the node row's
// (y, z) is interpolated once into shared memory (4 m values), and every node adds one
// interpolation in x with weights its thread keeps from row to row: about 30 operations a node
// instead of 170.  A warm start 64^3 -> 128^3 with 50 rounds and the fields read back, with
// the fused rounds (launch_step_imposed): 15.6 -> 4.5 ms.
constexpr int kResampleThreads = 128, kResampleRows = 16;

// Position of node i of n on an axis of m cells: cells lo and hi = lo + 1 with weights 1 - w
// and w.  A cell of weight 0 must not enter the sum (its value may not be finite): `one` is 1
// when only lo counts, 2 when only hi does.
struct AxisCell {
    double w, v;  // v = 1 - w
    int lo, hi, one;
};
__device__ __forceinline__ AxisCell axis_cell(int i, int n, int m) {
    const double s = (i + 0.5) * m / n - 0.5;
    const double p = fmin(fmax(s, 0.0), (double)(m - 1));
    AxisCell a;
    a.lo = min((int)floor(p), m - 2 < 0 ? 0 : m - 2);
    a.hi = min(a.lo + 1, m - 1);
    a.w = m == 1 ? 0.0 : p - a.lo;
    a.v = 1.0 - a.w;
    a.one = a.w == 0.0 ? 1 : a.v == 0.0 ? 2 : 0;
    return a;
}
__device__ __forceinline__ double mix(double l, double h, const AxisCell& a) {
    const double r = fma(a.w, h, a.v * l);
    return a.one == 0 ? r : a.one == 1 ? l : h;
}

__global__ void __launch_bounds__(kResampleThreads)
    resample_kernel(const float* __restrict__ pred, int m, int nx, int ny, int nz, double U0,
                    double* __restrict__ ux, double* __restrict__ uy, double* __restrict__ uz,
                    double* __restrict__ T) {
    extern __shared__ double row[];  // [4][m]
    __shared__ AxisCell cell[2][kResampleRows];
    const int i = blockIdx.x * kResampleThreads + threadIdx.x;
    const AxisCell x = axis_cell(i < nx ? i : 0, nx, m);
    const int64_t rows = (int64_t)ny * nz;
    for (int64_t r0 = (int64_t)blockIdx.y * kResampleRows; r0 < rows; r0 += (int64_t)gridDim.y * kResampleRows) {
        __syncthreads();  // the cells before are read
        if (threadIdx.x < 2 * kResampleRows) {
            const int64_t r = min(r0 + threadIdx.x % kResampleRows, rows - 1);
            const int k = (int)(r / ny), j = (int)(r - (int64_t)k * ny);
            if (threadIdx.x < kResampleRows) cell[0][threadIdx.x] = axis_cell(j, ny, m);
            else cell[1][threadIdx.x - kResampleRows] = axis_cell(k, nz, m);
        }
        for (int q = 0; q < kResampleRows && r0 + q < rows; ++q) {
            __syncthreads();  // the cells are there, the row before is read
            const AxisCell y = cell[0][q], z = cell[1][q];
            const float* p00 = pred + ((int64_t)z.lo * m + y.lo) * m * 4;
            const float* p01 = pred + ((int64_t)z.lo * m + y.hi) * m * 4;
            const float* p10 = pred + ((int64_t)z.hi * m + y.lo) * m * 4;
            const float* p11 = pred + ((int64_t)z.hi * m + y.hi) * m * 4;
            for (int e = threadIdx.x; e < 4 * m; e += kResampleThreads)
                row[(e & 3) * m + (e >> 2)] =
                    ((e & 3) == 3 ? 0.5 : U0) * mix(mix(p00[e], p01[e], y), mix(p10[e], p11[e], y), z);
            __syncthreads();
            if (i < nx) {
                const int64_t c = (r0 + q) * nx + i;
                ux[c] = mix(row[x.lo], row[x.hi], x);
                uy[c] = mix(row[m + x.lo], row[m + x.hi], x);
                uz[c] = mix(row[2 * m + x.lo], row[2 * m + x.hi], x);
                T[c] = mix(row[3 * m + x.lo], row[3 * m + x.hi], x);
            }
        }
    }
}

cudaError_t launch_resample(const float* pred, int m, const lbm_grid& g, double U0, double* out, int64_t n,
                            cudaStream_t st) {
    const size_t smem = (size_t)4 * m * sizeof(double);
    if (smem > 40 * 1024) {
        // one value for every caller: two threads may launch with different m
        const cudaError_t e =
            cudaFuncSetAttribute(resample_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
        if (e != cudaSuccess) return e;
    }
    const int64_t chunks = ((int64_t)g.ny * g.nz + kResampleRows - 1) / kResampleRows;
    const dim3 grid((g.nx + kResampleThreads - 1) / kResampleThreads, (unsigned)std::min<int64_t>(chunks, 65535));
    resample_kernel<<<grid, kResampleThreads, smem, st>>>(pred, m, g.nx, g.ny, g.nz, U0, out, out + n,
                                                          out + 2 * n, out + 3 * n);
    return cudaGetLastError();
}

}  // namespace

extern "C" int lbm_net_targets(lbm_ctx* c, float* out) {
    if (!c || !out) return fail(c, LBM_EINVAL, "NULL argument%s");
    if (!(c->params.U0 > 0)) return fail(c, LBM_EINVAL, "the context has no velocity scale U0%s");
    DeviceGuard g(c->device);
    int rc = with_storage(c->precision, [&](auto tag) {
        using S = decltype(tag);
        const ParamsOf<S> p = dev_params<typename Storage<S>::real>(c);
        CUDA_OR_FAIL(c, launch_targets<S>(c->dev, c->cur, p, 1.0 / c->params.U0, out, c->stream));
        return LBM_OK;
    });
    if (rc != LBM_OK) return rc;
    return wait_stream(c);
}

extern "C" int lbm_net_warm_start(lbm_ctx* c, const float* pred, int m, int iterations) {
    if (!c || !pred || m < 1 || iterations < 0)
        return fail(c, LBM_EINVAL, "NULL prediction, grid size < 1 or negative iterations%s");
    if (!(c->params.U0 > 0)) return fail(c, LBM_EINVAL, "the context has no velocity scale U0%s");
    DeviceGuard g(c->device);
    const int64_t n = c->ncell;
    // The FP64 fields go to the flow planes of the buffer the next step writes when nothing reads them
    // after the first round (FP32 and FP64), and the rounds take them packed from memory of the call's
    // own (16 bytes a node in FP32, where the fields themselves take 32); else the fields go there.
    // That memory is allocated and freed on each call (33 MB: 0.12 ms, half of it beside the resampling):
    // kept, it would be device memory that no arena counts.
    const bool dev16 = c->precision == LBM_FP16_DEV || c->precision == LBM_BF16_DEV;
    const bool lend = iterations == 0 ? !dev16 : rounds_fused(c);
    const size_t bytes = !lend ? (size_t)4 * n * sizeof(double) : iterations ? packed_bytes(c) : 0;
    double* buf = static_cast<double*>(c->dev.F[c->cur ^ 1]);
    void* own = nullptr;
    cudaError_t e = lend ? launch_resample(pred, m, c->grid, c->params.U0, buf, n, c->stream) : cudaSuccess;
    if (bytes && cudaMalloc(&own, bytes) != cudaSuccess)
        return fail(c, LBM_ENOMEM, "cudaMalloc failed: %s", cudaGetErrorString(cudaGetLastError()));
    if (!lend) {
        buf = static_cast<double*>(own);
        e = launch_resample(pred, m, c->grid, c->params.U0, buf, n, c->stream);
    }
    int rc = e == cudaSuccess
                 ? init_fields(c, nullptr, buf, buf + n, buf + 2 * n, buf + 3 * n, iterations, lend ? own : nullptr)
                 : fail(c, LBM_ECUDA, "resampling failed: %s", cudaGetErrorString(e));
    if (own) cudaFree(own);  // init_fields waited for the stream
    return rc;
}
