// Allocation-free dose SpMV with the objective epilogue.
//
// Some callers cannot allocate device memory at call time.  One example is a
// re-planning service that reserves and pins every device buffer before an
// online adaptive fraction starts, so that a fraction can neither fail on an
// out-of-memory error nor stall on the device-wide synchronisation that
// cudaMalloc and cudaFree may imply.  Another is an application whose own
// allocator owns the whole device.  This entry point computes the same
// quantities as dao_k_dose (z = D x, grad F(z) and F(z)) without a context
// and without any allocation: the caller passes the inputs and outputs, and
// the only scratch memory, the per-block partial sums of F and their
// ticket, lives in file-scope device arrays that every GPU loading the library keeps until the
// process exits.
#include <algorithm>
#include <mutex>

#include "dao_internal.h"

namespace {

constexpr int NA_MAX_VOXELS = 4194304;   // the entry point's limit
constexpr int NA_MAX_BLOCKS = 1024;      // size of the scratch array
constexpr int NA_THREADS = 512;
constexpr int NA_WARPS = NA_THREADS / 32;
constexpr int NA_CHUNK = 1024;           // products a warp holds at a time
constexpr int NA_AHEAD = 6;              // entries per lane requested together
constexpr int NA_MAX_DEVICES = 64;
constexpr int SMAX_TERMS = dao::SMAX;

// Per-block FP64 partial sums of the objective, and the ticket the blocks of a
// call take when they have written theirs (0 between calls).
static __device__ __align__(256) double dao_noalloc_scratch[NA_MAX_BLOCKS];
static __device__ unsigned dao_noalloc_ticket;

struct NoallocTerms {
    double t[SMAX_TERMS][4];  // alpha_s / |v_s|, T_s^-, beta_s / |v_s|, T_s^+
};

__device__ __forceinline__ double na_warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum of one double per thread over the block, valid in thread 0.
__device__ __forceinline__ double na_block_sum(double v, double* s_red) {
    v = na_warp_sum(v);
    __syncthreads();  // s_red may still be read from an earlier sum
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) {
        t = threadIdx.x < NA_WARPS ? s_red[threadIdx.x] : 0.0;
        t = na_warp_sum(t);
    }
    return t;
}

// A warp takes units of 32 consecutive rows (grid-stride): their entries are one
// contiguous range, read with consecutive entries on consecutive lanes, NA_AHEAD
// per lane in flight, the next ones (and the next unit's row offsets) requested
// before these are used; the products go to the warp's chunk of shared memory, and
// lane r sums row r's from there (four interleaved partial sums), so that every
// lane then has a row of its own for the FP64 epilogue.  The caller's rows have
// no padding, so wider loads would start off their alignment.  X: x in shared
// memory.  The block that takes the call's last ticket adds the blocks' partial
// sums in block order.
//
// Bound by the entries' bytes (8 nnz) in the limit; H&N-shaped FP32 matrix
// (304,184 voxels, 9.55 M entries).  With 8 lanes to a row the epilogue's FP64
// instructions (1/64 of the FP32 rate) ran with four lanes of 32 in use and each
// lane waited for its gather before its next entry: 104 us; the call took 158 us
// and takes 84 now (85.8 without the requests ahead), of which the kernel is the
// smaller part.
template <bool X>
__global__ void __launch_bounds__(NA_THREADS, 2) k_dose_noalloc(int V, int N, const int* __restrict__ rowptr,
                                                               const int* __restrict__ col,
                                                               const float* __restrict__ val,
                                                               const float* __restrict__ x,
                                                               const int* __restrict__ vstruct, int S,
                                                               const __grid_constant__ NoallocTerms terms,
                                                               float* __restrict__ z, float* __restrict__ grad,
                                                               double* partial, unsigned* ticket,
                                                               double* __restrict__ out) {
    extern __shared__ float s_na[];
    __shared__ double s_red[NA_WARPS];
    __shared__ double s_t[SMAX_TERMS][4];
    __shared__ float2 s_f[SMAX_TERMS];  // T^- rounded up, T^+ rounded down: an FP32 z compares with these as with the FP64
    __shared__ int s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* buf = s_na + warp * NA_CHUNK;
    float* sx = s_na + NA_WARPS * NA_CHUNK;
    const int units = (V + 31) / 32;
    const bool busy = (int)blockIdx.x * NA_WARPS < units;
    bool fin = true;
    for (int i = threadIdx.x; i < 4 * S && busy; i += NA_THREADS) {
        const double t = (&terms.t[0][0])[i];
        (&s_t[0][0])[i] = t;
        if ((i & 3) == 1) s_f[i >> 2].x = __double2float_ru(t);
        if ((i & 3) == 3) s_f[i >> 2].y = __double2float_rd(t);
        fin = fin && isfinite(t);
    }
    if (X && busy)
        for (int i = threadIdx.x; i < N; i += NA_THREADS) sx[i] = __ldg(x + i);
    const bool finite = __syncthreads_and(fin) != 0;
    double facc = 0.0;
    int rs_n = 0, re_n = 0, lab_n = 0;  // the next unit's row offsets and labels, requested ahead
    auto unit_in = [&](int u) {
        const int row = min(u, units) * 32 + lane;
        rs_n = __ldg(rowptr + min(row, V));
        re_n = __ldg(rowptr + min(row + 1, V));
        lab_n = row < V ? __ldg(vstruct + row) : 0;
    };
    const int u0 = blockIdx.x * NA_WARPS + warp;
    if (u0 < units) unit_in(u0);
    for (int u = u0; u < units; u += gridDim.x * NA_WARPS) {
        const int row = u * 32 + lane;
        const int rs = rs_n, re = re_n, lab = lab_n;
        unit_in(u + gridDim.x * NA_WARPS);
        const int e0 = __shfl_sync(0xffffffffu, rs, 0), e1 = __shfl_sync(0xffffffffu, re, 31);
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        for (int c0 = e0; c0 < e1; c0 += NA_CHUNK) {
            const int c1 = min(e1, c0 + NA_CHUNK);
            int cn[NA_AHEAD];
            float vn[NA_AHEAD];
            auto batch_in = [&](int p0) {
#pragma unroll
                for (int q = 0; q < NA_AHEAD; ++q) {
                    const int p = p0 + 32 * q + lane;
                    cn[q] = p < c1 ? __ldg(col + p) : 0;
                    vn[q] = p < c1 ? __ldg(val + p) : 0.f;
                }
            };
            batch_in(c0);
            for (int p0 = c0; p0 < c1; p0 += 32 * NA_AHEAD) {
                int c[NA_AHEAD];
                float v[NA_AHEAD];
#pragma unroll
                for (int q = 0; q < NA_AHEAD; ++q) {
                    c[q] = cn[q];
                    v[q] = vn[q];
                }
                batch_in(p0 + 32 * NA_AHEAD);
#pragma unroll
                for (int q = 0; q < NA_AHEAD; ++q) {
                    const int p = p0 + 32 * q + lane;
                    if (p < c1) buf[p - c0] = v[q] * (X ? sx[c[q]] : __ldg(x + c[q]));
                }
            }
            __syncwarp();
            const int a = max(rs, c0), b = min(re, c1);
            int p = a;
            for (; p + 3 < b; p += 4) {
                acc[0] += buf[p - c0];
                acc[1] += buf[p + 1 - c0];
                acc[2] += buf[p + 2 - c0];
                acc[3] += buf[p + 3 - c0];
            }
            for (; p < b; ++p) acc[0] += buf[p - c0];
            __syncwarp();
        }
        const float zr = (acc[0] + acc[1]) + (acc[2] + acc[3]);
        if (row < V) {
            z[row] = zr;
            if ((unsigned)lab >= (unsigned)S) {  // no such structure: flagged, never read
                if (grad != nullptr) grad[row] = __int_as_float(0x7fc00000);
                facc += __longlong_as_double(0x7ff8000000000000ll);  // the objective becomes NaN
            } else {
                float g = 0.f;
                if (zr < s_f[lab].x || zr > s_f[lab].y || !finite) {  // else both penalties are 0 (so most voxels)
                    const double* tt = s_t[lab];
                    const double zd = zr;
                    const double uu = fmax(0.0, tt[1] - zd), o = fmax(0.0, zd - tt[3]);
                    g = (float)(2.0 * (tt[2] * o - tt[0] * uu));
                    facc += tt[0] * uu * uu + tt[2] * o * o;
                }
                if (grad != nullptr) grad[row] = g;
            }
        }
    }
    const double t = na_block_sum(facc, s_red);
    if (threadIdx.x == 0) {
        partial[blockIdx.x] = t;
        // release: the partial sum before the ticket; acquire: the other blocks' sums.
        // The ticket wraps to 0 with the last block, and every launch has the same
        // number of blocks, so that it is 0 again whatever overlapped.
        unsigned old;
        asm volatile("atom.inc.acq_rel.gpu.global.u32 %0, [%1], %2;"
                     : "=r"(old)
                     : "l"(ticket), "r"(gridDim.x - 1u)
                     : "memory");
        s_last = old == gridDim.x - 1u;
    }
    __syncthreads();
    if (!s_last) return;
    double v = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += NA_THREADS) v += __ldcg(partial + i);
    v = na_block_sum(v, s_red);
    if (threadIdx.x == 0) *out = v;
}

std::mutex g_mu;
// per device: the scratch array, the ticket, the multiprocessors
struct NoallocDevice {
    double* scratch = nullptr;
    unsigned* ticket = nullptr;
    int sms = 0;
};
NoallocDevice g_na[NA_MAX_DEVICES];
// beamlets whose x fits shared memory beside the warps' chunks
constexpr int NA_MAX_X = (100 * 1024) / (int)sizeof(float) - NA_WARPS * NA_CHUNK;  // two blocks per SM
constexpr size_t na_smem(int n) { return sizeof(float) * ((size_t)NA_WARPS * NA_CHUNK + n); }

dao_status na_fail(dao_status s, const std::string& m) { return dao::set_error(s, m); }

}  // namespace

extern "C" {

dao_status dao_dose_objective_noalloc(int32_t n_voxels, int32_t n_beamlets, const int32_t* row_ptr,
                                      const int32_t* col, const float* val, const float* x,
                                      const int32_t* voxel_struct, int32_t n_structures, const double* terms,
                                      float* z, float* grad, double* objective, void* stream) {
    if (n_voxels < 1 || n_beamlets < 1 || !row_ptr || !col || !val || !x || !voxel_struct || !terms || !z ||
        !objective)
        return na_fail(DAO_EINVAL, "null pointer or empty problem");
    if (n_voxels > NA_MAX_VOXELS)
        return na_fail(DAO_EINVAL, "n_voxels exceeds the allocation-free limit of " + std::to_string(NA_MAX_VOXELS) +
                                       " voxels");
    if (n_structures < 1 || n_structures > SMAX_TERMS)
        return na_fail(DAO_EINVAL, "n_structures must be in [1, " + std::to_string(SMAX_TERMS) + "]");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return na_fail(DAO_ECUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= NA_MAX_DEVICES) return na_fail(DAO_EINVAL, "device ordinal out of range");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (st != nullptr) {  // the kernels run on the current device: the stream must belong to it
        int sdev = -1;
        e = cudaStreamGetDevice(st, &sdev);
        if (e != cudaSuccess) return na_fail(DAO_EINVAL, std::string("cudaStreamGetDevice: ") + cudaGetErrorString(e));
        if (sdev != dev)
            return na_fail(DAO_EINVAL, "the stream belongs to device " + std::to_string(sdev) +
                                           ", not to the current device " + std::to_string(dev));
    }
    NoallocDevice nd;
    {
        // set-up, once per device with that device current: the device addresses of
        // the file-scope array and ticket (their names are only host-side
        // stand-ins) and the kernels' shared memory limit.  The addresses belong
        // to the device's primary context as it was at that first call; after a
        // cudaDeviceReset they are stale, and a caller that resets the device must
        // not call this entry point again in the same process.
        std::lock_guard<std::mutex> lock(g_mu);
        NoallocDevice& g = g_na[dev];
        if (g.scratch == nullptr) {
            void *p = nullptr, *q = nullptr;
            int sms = 0;
            e = cudaGetSymbolAddress(&p, dao_noalloc_scratch);
            if (e == cudaSuccess) e = cudaGetSymbolAddress(&q, dao_noalloc_ticket);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(k_dose_noalloc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)na_smem(NA_MAX_X));
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(k_dose_noalloc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)na_smem(0));
            if (e != cudaSuccess) {
                cudaGetLastError();
                return na_fail(DAO_ECUDA, std::string("noalloc set-up: ") + cudaGetErrorString(e));
            }
            g.ticket = static_cast<unsigned*>(q);
            g.sms = sms;
            g.scratch = static_cast<double*>(p);
        }
        nd = g;
    }
    NoallocTerms t;
    for (int s = 0; s < SMAX_TERMS; ++s)
        for (int q = 0; q < 4; ++q) t.t[s][q] = s < n_structures ? terms[4 * s + q] : 0.0;
    const unsigned grid = (unsigned)std::min(2 * nd.sms, NA_MAX_BLOCKS);  // the same for every call: see the ticket
    if (n_beamlets <= NA_MAX_X)
        k_dose_noalloc<true><<<grid, NA_THREADS, na_smem(n_beamlets), st>>>(n_voxels, n_beamlets, row_ptr, col, val, x,
                                                                           voxel_struct, n_structures, t, z, grad,
                                                                           nd.scratch, nd.ticket, objective);
    else
        k_dose_noalloc<false><<<grid, NA_THREADS, na_smem(0), st>>>(n_voxels, n_beamlets, row_ptr, col, val, x,
                                                                   voxel_struct, n_structures, t, z, grad, nd.scratch,
                                                                   nd.ticket, objective);
    e = cudaGetLastError();
    if (e != cudaSuccess) return na_fail(DAO_ECUDA, std::string("k_dose_noalloc: ") + cudaGetErrorString(e));
    return DAO_OK;
}

}  // extern "C"
