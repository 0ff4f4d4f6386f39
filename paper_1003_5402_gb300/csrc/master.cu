// Master problem of column-generation DAO (arXiv:1003.5402, Sec. 2.2-2.3):
// min_y F(S y) subject to y >= 0 over the current aperture pool, where column k
// of the slab S (V x K, FP32) is the aperture dose D_kj of Eq. 2.  The slab is
// stored by groups of four columns, the four doses of a voxel together (entry
// (j, k) at ((k / 4) ld + j) 4 + k mod 4): one 16-byte load gives a voxel's
// doses of a group, and a warp's 32 voxels are 512 consecutive bytes.
//
// The paper uses gradient projection and gives no step or stopping rule.  This
// is a scaled gradient projection, the projected Newton method of Bertsekas
// (1982): variables with y_k <= eps and g_k > 0 take the plain gradient step,
// the others a Newton step on H = S_F^T diag(h) S_F (h = generalised second
// derivative of the piecewise-quadratic F), with Armijo backtracking along the
// projection arc.  One evaluation is four kernels:
//   k_master_eval   streams the slab in tiles of TILE voxels (2-D TMA bulk
//                   copies completing on an mbarrier) and computes z = S y as a
//                   compensated FP32 dot product (Ogita, Rump & Oishi,
//                   "Accurate sum and dot product", 2005; y split into two
//                   floats), pi = grad F(z), h and F; voxels with h > 0 are the
//                   only ones that contribute to g and H, and their rows, h and
//                   pi are written compacted, per tile, to an active list;
//   k_master_hess   the active list split evenly over the blocks: per-block
//                   partials of H (FP32), g and the rounding scale of g;
//   k_master_reduce fixed-order reduction of the partials;
//   k_master_step   one block: KKT test at the trial point, Armijo test, damped
//                   FP32 Cholesky of the free block of H, next trial point.
// Every kernel returns at once after the state is marked done, so evaluations
// can be queued ahead (or looped on the device by a graph while node).
//
// Stopping rule: |y_k - max(y_k - g_k, 0)| <= tol_rel * max|g(start)| +
// NOISE * u * sum_j |S_jk pi_j| for every k (u = 2^-24), i.e. KKT up to the
// FP32 rounding level of g.  A trial point that meets it is accepted without
// the Armijo test: near the optimum the objective's change is below its own
// rounding and the test would reject an optimal point.
#include <algorithm>

#include "dao_internal.h"

#include <cmath>

namespace dao {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int TILE = MASTER_TILE;   // voxels per evaluation tile = threads per block
constexpr int CH = 128;             // active voxels per Hessian sub-chunk
constexpr float U32 = 5.9604645e-8f;  // 2^-24
constexpr double NOISE = 64.0;
constexpr int WAIT_LIMIT = 1 << 20;   // mbarrier polls before a copy is declared lost
constexpr int HSTRIDE = KMAX * (KMAX + 1) / 2;  // packed curvature entries per block of the kept partial H

__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

__device__ __forceinline__ float warp_sum_f32(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

// ---- TMA / mbarrier (sm_90+ PTX) ----------------------------------------------
__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

// Bounded wait for the phase with the given parity; false if it never completed.
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity) {
    const unsigned a = smem_addr(bar);
    for (int i = 0; i < WAIT_LIMIT; ++i) {
        unsigned ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// 2-D tiled bulk copy of box (x, y) of the tensor map into shared memory.
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y,
                                            unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
            smem_addr(dst)),
        "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(smem_addr(bar))
        : "memory");
}

// TwoSum accumulation of a product a*y (y = yh + yl) into the pair (s, c).
__device__ __forceinline__ void dot2_step(float& s, float& c, float a, float yh, float yl) {
    const float p = a * yh;
    float pe = fmaf(a, yh, -p);  // a*yh = p + pe exactly
    pe = fmaf(a, yl, pe);
    const float t2 = s + p;      // TwoSum(s, p)
    const float bb = t2 - s;
    const float e = (s - (t2 - bb)) + (p - bb);
    s = t2;
    c += e + pe;
}

// (rb, cb) of the eb-th 4x4 block of the upper triangle, row-major
__device__ __forceinline__ void block_of(int eb, int KB, int& rb, int& cb) {
    int r = 0, rem = eb;
    while (rem >= KB - r) {
        rem -= KB - r;
        ++r;
    }
    rb = r;
    cb = r + rem;
}

// Packed index of entry (r, c), r <= c, of the upper triangle, column by column:
// c (c + 1) / 2 + r, the same for every pool size K (a partial H kept from one
// pool size to the next keeps its entries in place).
__device__ __forceinline__ int tri_index(int r, int c, int K) {
    (void)K;
    return c * (c + 1) / 2 + r;
}

__global__ void k_master_init(MasterDev* __restrict__ st, int K, const int* __restrict__ skip,
                              cudaGraphConditionalHandle cond, int use_cond, GridBar* __restrict__ gb) {
    const int t = threadIdx.x;
    if (t == 0 && gb != nullptr) {  // a barrier left by an aborted solve starts empty
        gb->count = 0;
        gb->broken = 0;
    }
    if (skip != nullptr && *skip) {  // the solve stopped before this round: nothing to iterate
        if (t == 0) {
            st->done = 1;
            if (use_cond) cudaGraphSetConditional(cond, 0u);
        }
        return;
    }
    if (t < K) {
        const double v = t < K - 1 ? st->y[t] : 0.0;  // warm start: previous optimum, new aperture at 0
        st->yt[t] = v;
        st->d[t] = 0.0;
    }
    if (t == 0) {
        st->K = K;
        st->iter = 0;
        st->phase = 0;
        st->done = 0;
        st->status = MASTER_RUNNING;
        st->alpha = 1.0;
        st->n_eval = 0;
        st->err = 0;
        st->ticket = 0;
        st->final_pending = 0;
        if (use_cond) cudaGraphSetConditional(cond, 1u);
    }
}

// Graph path: keep the statistics of the master solve that just finished.
__global__ void k_cg_record(const MasterDev* __restrict__ st, CGDev* __restrict__ cg, int K) {
    if (threadIdx.x != 0 || cg->idle) return;
    cg->trace[K - 1] = st->F;
    cg->res[K - 1] = st->res;
    cg->tol[K - 1] = st->tol;
    cg->evals[K - 1] = st->n_eval;
    cg->status[K - 1] = st->status;
}

// ---- evaluation: one slab tile per iteration --------------------------------
// A tile is TILE voxels x KP columns of the slab: two boxes of 128 voxels x KP / 4
// groups of columns, each landing in shared memory as [KP / 4][128][4].
__global__ void __launch_bounds__(TILE, 3) k_master_eval(const __grid_constant__ CUtensorMap tmap, int V, int K,
                                                         int KP, MasterDev* __restrict__ st,
                                                         float* __restrict__ act_rows, float2* __restrict__ act_hp,
                                                         int* __restrict__ act_count, double* __restrict__ F_part,
                                                         const uint8_t* __restrict__ vstruct,
                                                         const StructTermsF* __restrict__ tf, int S,
                                                         float* __restrict__ z_out, float* __restrict__ pi_out,
                                                         int mode, const int* __restrict__ skip) {
    if (skip != nullptr && *skip) return;
    if (mode == PASS_EVAL && st->done) return;
    const bool final_pass = mode == PASS_FINAL;
    extern __shared__ __align__(128) float4 As[];  // [2][KP / 4][TILE / 2]
    __shared__ __align__(8) unsigned long long bar;
    __shared__ float s_yh[KMAX], s_yl[KMAX];
    __shared__ int s_wcount[TILE / 32];
    __shared__ StructTermsF s_tf[SMAX];
    __shared__ float s_red[TILE / 32];
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    if (tid < KMAX) {
        const double yv = tid < K ? (final_pass ? st->y[tid] : st->yt[tid]) : 0.0;
        const float hi = (float)yv;
        s_yh[tid] = hi;
        s_yl[tid] = (float)(yv - (double)hi);
    }
    for (int i = tid; i < S; i += TILE) s_tf[i] = tf[i];
    if (tid == 0) mbar_init(&bar, 1);
    __syncthreads();
    float facc = 0.f;  // this thread's voxels: a few terms, FP32 is enough before the FP64 block sum
    unsigned parity = 0;
    bool lost = false;
    const int n_tiles = (V + TILE - 1) / TILE;
    const float4* av = As + (tid / (TILE / 2)) * (KP / 4) * (TILE / 2) + tid % (TILE / 2);  // this voxel, group 0
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        __syncthreads();  // every thread is done with the previous tile's buffers
        if (tid == 0 && KP > 0) {
            mbar_expect_tx(&bar, (unsigned)(TILE * KP * sizeof(float)));
            tma_load_2d(As, &tmap, tile * TILE * 2, 0, &bar);  // (8-byte elements)
            tma_load_2d(As + (KP / 4) * (TILE / 2), &tmap, tile * TILE * 2 + TILE, 0, &bar);
        }
        if (KP > 0) {
            if (!mbar_wait(&bar, parity)) {
                lost = true;
                break;
            }
            parity ^= 1u;
        }
        const int j = tile * TILE + tid;
        // ---- compensated z from this voxel's column of the tile, four chains
        float sc[4] = {0.f, 0.f, 0.f, 0.f}, cc[4] = {0.f, 0.f, 0.f, 0.f};
        for (int k = 0; k < KP; k += 4) {  // doses of columns K..KP-1 meet y = 0
            const float4 a = av[(k / 4) * (TILE / 2)];
            dot2_step(sc[0], cc[0], a.x, s_yh[k], s_yl[k]);
            dot2_step(sc[1], cc[1], a.y, s_yh[k + 1], s_yl[k + 1]);
            dot2_step(sc[2], cc[2], a.z, s_yh[k + 2], s_yl[k + 2]);
            dot2_step(sc[3], cc[3], a.w, s_yh[k + 3], s_yl[k + 3]);
        }
        float s = sc[0], c = cc[0];
#pragma unroll
        for (int q = 1; q < 4; ++q) {
            const float t2 = s + sc[q];
            const float bb = t2 - s;
            const float e = (s - (t2 - bb)) + (sc[q] - bb);
            s = t2;
            c += e + cc[q];
        }
        float h = 0.f, p = 0.f;
        if (j < V) {
            const StructTermsF t = S >= 0 ? s_tf[vstruct[j]] : voxel_terms(tf, j);
            const float du = (t.tu - s) - c;   // T^- - z, exact subtraction near the threshold
            const float dov = (s - t.to) + c;  // z - T^+
            const float u = fmaxf(du, 0.f), o = fmaxf(dov, 0.f);
            p = 2.f * (t.b * o - t.a * u);
            h = 2.f * ((du > 0.f ? t.a : 0.f) + (dov > 0.f ? t.b : 0.f));
            facc = fmaf(t.a * u, u, fmaf(t.b * o, o, facc));
            if (final_pass) {
                z_out[j] = s + c;
                pi_out[j] = p;
            }
        }
        if (final_pass) continue;
        // ---- compact the voxels with non-zero curvature into this tile's slots
        const bool act = h > 0.f;
        const unsigned bal = __ballot_sync(FULL, act);
        if (lane == 0) s_wcount[warp] = __popc(bal);
        __syncthreads();
        int base = 0, n_act = 0;
#pragma unroll
        for (int w = 0; w < TILE / 32; ++w) {
            const int cnt = s_wcount[w];
            base += w < warp ? cnt : 0;
            n_act += cnt;
        }
        if (act) {
            const size_t slot = (size_t)tile * TILE + base + __popc(bal & ((1u << lane) - 1u));
            float4* dst = reinterpret_cast<float4*>(act_rows + slot * KROW);
            for (int g = 0; g < KP / 4; ++g) dst[g] = av[g * (TILE / 2)];
            act_hp[slot] = make_float2(h, p);
        }
        if (tid == 0) act_count[tile] = n_act;
    }
    if (lost) {  // a tile copy never arrived: report it, the step kernel stops the solve
        if (tid == 0) st->err = 1;
        return;
    }
    if (final_pass) return;
    // F: FP32 within a warp (32 voxel terms), FP64 across the block's warps
    // (FP64 runs at 1/64 of the FP32 rate here: keep it to a few lanes)
    const float fw = warp_sum_f32(facc);
    if (lane == 0) s_red[warp] = fw;
    __syncthreads();
    if (tid < 32) {
        double t = tid < TILE / 32 ? (double)s_red[tid] : 0.0;
#pragma unroll
        for (int o = TILE / 64; o > 0; o >>= 1) t += __shfl_xor_sync(FULL, t, o);
        if (tid == 0) F_part[blockIdx.x] = t;
    }
}

// ---- curvature and gradient over the active list ----------------------------
// Block b takes active voxels [M b / G, M (b + 1) / G) in tile order, in
// sub-chunks of CH voxels copied to shared memory as rows of KW floats; thread
// (eb, v) accumulates the 4x4 block eb of H over voxel lane v, and the diagonal
// blocks also g and sum |S_jk pi_j|.
__global__ void __launch_bounds__(256) k_master_hess(const float* __restrict__ act_rows,
                                                     const float2* __restrict__ act_hp,
                                                     const int* __restrict__ act_count, int n_tiles, int K, int KW,
                                                     int NV, MasterDev* __restrict__ st, float* __restrict__ H_part,
                                                     double* __restrict__ g_part, float* __restrict__ gn_part, int G,
                                                     int mode) {
    if (mode == PASS_EVAL && st->done) return;
    // the partial arrays are overwritten: the persistent solve's kept partial H is gone
    if (blockIdx.x == 0 && threadIdx.x == 0) st->inc_G = 0;
    extern __shared__ __align__(16) float smem[];
    int* s_pref = reinterpret_cast<int*>(smem);                        // [n_tiles + 1]
    float* Ac = smem + ((n_tiles + 1 + 3) / 4) * 4;                    // [CH][KW]
    float* s_h = Ac + CH * KW;                                         // [CH]
    float* s_p = s_h + CH;                                             // [CH]
    __shared__ float s_scr[8 * 24];
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    // exclusive prefix of the per-tile active counts (integer sums: exact in any
    // order): contiguous chunks per thread, then a scan of the chunk totals
    __shared__ int s_wsum[8];
    {
        const int per = (n_tiles + 255) / 256;
        const int t0 = tid * per, t1 = min(n_tiles, t0 + per);
        int mine = 0;
        for (int t = t0; t < t1; ++t) mine += act_count[t];
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) s_wsum[warp] = incl;
        __syncthreads();
        int before = incl - mine;
        for (int w = 0; w < warp; ++w) before += s_wsum[w];
        for (int t = t0; t < t1; ++t) {
            s_pref[t] = before;
            before += act_count[t];
        }
        if (tid == 255) s_pref[n_tiles] = before;
    }
    const int KP = (K + 3) / 4 * 4;
    const int KB = KP / 4;
    const int nb = KB * (KB + 1) / 2;
    int rb = -1, cb = -1;
    const int v = tid % NV;
    if (tid < nb * NV) block_of(tid / NV, KB, rb, cb);
    __syncthreads();
    const int M = s_pref[n_tiles];
    const int m0 = (int)((long long)M * blockIdx.x / G), m1 = (int)((long long)M * (blockIdx.x + 1) / G);
    const int nq = KP / 4;
    float hs[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) hs[q] = 0.f;
    float gs[4] = {0.f, 0.f, 0.f, 0.f}, gns[4] = {0.f, 0.f, 0.f, 0.f};
    for (int c0 = m0; c0 < m1; c0 += CH) {
        const int n = min(CH, m1 - c0);
        __syncthreads();
        // copy the sub-chunk: two threads per voxel, alternate float4 groups
        {
            const int i = tid >> 1, half = tid & 1;
            if (i < n) {
                const int m = c0 + i;
                int lo = 0, hi = n_tiles;  // last tile with pref <= m
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (s_pref[mid] <= m) lo = mid; else hi = mid;
                }
                const size_t slot = (size_t)lo * TILE + (m - s_pref[lo]);
                const float4* src = reinterpret_cast<const float4*>(act_rows + slot * KROW);
                float4* dst = reinterpret_cast<float4*>(Ac + i * KW);
                for (int q = half; q < nq; q += 2) dst[q] = src[q];
                if (half == 0) {
                    const float2 hp = act_hp[slot];
                    s_h[i] = hp.x;
                    s_p[i] = hp.y;
                }
            }
        }
        __syncthreads();
        if (rb >= 0) {
            for (int i = v; i < n; i += NV) {
                const float4 ra = *reinterpret_cast<const float4*>(Ac + i * KW + 4 * rb);
                const float4 rc = *reinterpret_cast<const float4*>(Ac + i * KW + 4 * cb);
                const float hv = s_h[i];
                const float a0 = ra.x * hv, a1 = ra.y * hv, a2 = ra.z * hv, a3 = ra.w * hv;
                hs[0] = fmaf(a0, rc.x, hs[0]);
                hs[1] = fmaf(a0, rc.y, hs[1]);
                hs[2] = fmaf(a0, rc.z, hs[2]);
                hs[3] = fmaf(a0, rc.w, hs[3]);
                hs[4] = fmaf(a1, rc.x, hs[4]);
                hs[5] = fmaf(a1, rc.y, hs[5]);
                hs[6] = fmaf(a1, rc.z, hs[6]);
                hs[7] = fmaf(a1, rc.w, hs[7]);
                hs[8] = fmaf(a2, rc.x, hs[8]);
                hs[9] = fmaf(a2, rc.y, hs[9]);
                hs[10] = fmaf(a2, rc.z, hs[10]);
                hs[11] = fmaf(a2, rc.w, hs[11]);
                hs[12] = fmaf(a3, rc.x, hs[12]);
                hs[13] = fmaf(a3, rc.y, hs[13]);
                hs[14] = fmaf(a3, rc.z, hs[14]);
                hs[15] = fmaf(a3, rc.w, hs[15]);
                if (rb == cb) {
                    const float pv = s_p[i], pa = fabsf(pv);
                    gs[0] = fmaf(ra.x, pv, gs[0]);
                    gs[1] = fmaf(ra.y, pv, gs[1]);
                    gs[2] = fmaf(ra.z, pv, gs[2]);
                    gs[3] = fmaf(ra.w, pv, gs[3]);
                    gns[0] = fmaf(fabsf(ra.x), pa, gns[0]);
                    gns[1] = fmaf(fabsf(ra.y), pa, gns[1]);
                    gns[2] = fmaf(fabsf(ra.z), pa, gns[2]);
                    gns[3] = fmaf(fabsf(ra.w), pa, gns[3]);
                }
            }
        }
    }
    // fold the NV voxel lanes of each entry block (consecutive threads) with a
    // fixed shuffle tree, then across warps through shared memory when NV > 32
    float vals[24];
#pragma unroll
    for (int q = 0; q < 16; ++q) vals[q] = hs[q];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        vals[16 + q] = gs[q];
        vals[20 + q] = gns[q];
    }
    const int span = NV < 32 ? NV : 32;
    for (int o = span / 2; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < 24; ++q) vals[q] += __shfl_xor_sync(FULL, vals[q], o);
    if (NV > 32 && lane == 0)
#pragma unroll
        for (int q = 0; q < 24; ++q) s_scr[warp * 24 + q] = vals[q];
    __syncthreads();
    if ((tid % NV) == 0 && tid < nb * NV) {
        if (NV > 32) {
            const int w0 = tid >> 5, nw = NV >> 5;
#pragma unroll
            for (int q = 0; q < 24; ++q) {
                float t = 0.f;
                for (int w = 0; w < nw; ++w) t += s_scr[(w0 + w) * 24 + q];
                vals[q] = t;
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int r = 4 * rb + q, col = 4 * cb + e;
                if (r < K && col < K && r <= col) H_part[(size_t)tri_index(r, col, K) * G + blockIdx.x] = vals[q * 4 + e];
            }
        if (rb == cb) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = 4 * rb + q;
                if (r < K) {
                    g_part[(size_t)r * G + blockIdx.x] = (double)vals[16 + q];
                    gn_part[(size_t)r * G + blockIdx.x] = vals[20 + q];
                }
            }
        }
    }
}

// Reduction of the partial sums: one warp per output (packed H entries, then g,
// then the g rounding scale, then F), outputs strided over the grid's warps;
// lanes read the blocks' partials (contiguous per output) and combine them with
// a fixed shuffle tree in FP64.
// Lane's share src[lane], src[lane + 32], ... of n partial sums, added in that
// order (as a plain loop would), with the loads of up to RP_LANE of them issued
// before the first add: in-order issue would otherwise wait for each load at
// its add.  Through L2: the partials were written by other blocks.
constexpr int RP_LANE = 12;
template <class T>
__device__ __forceinline__ T lane_sum_strided(const T* __restrict__ src, int n, int lane) {
    T s = T(0);
    for (int b0 = 0; b0 < n; b0 += 32 * RP_LANE) {
        T v[RP_LANE];
#pragma unroll
        for (int q = 0; q < RP_LANE; ++q) {
            const int b = b0 + lane + 32 * q;
            v[q] = b < n ? __ldcg(src + b) : T(0);
        }
#pragma unroll
        for (int q = 0; q < RP_LANE; ++q) s += v[q];
    }
    return s;
}

// The partial arrays hold GC columns (the blocks that wrote them) at stride GH.
__device__ __forceinline__ void master_reduce_part(const float* __restrict__ H_part,
                                                   const double* __restrict__ g_part,
                                                   const float* __restrict__ gn_part,
                                                   const double* __restrict__ F_part, int GH, int GC, int GE, int K,
                                                   MasterDev* __restrict__ st, int bid, int nblocks) {
    const int E = K * (K + 1) / 2;
    const int lane = threadIdx.x & 31;
    const int n_out = E + 2 * K + 1;
    for (int o = (bid * (int)blockDim.x + (int)threadIdx.x) >> 5; o < n_out; o += (nblocks * (int)blockDim.x) >> 5) {
        if (o < E) {  // the factorisation is FP32: so is this sum
            float s = lane_sum_strided(H_part + (size_t)o * GH, GC, lane);
            s = warp_sum_f32(s);
            if (lane == 0) {  // o = c (c + 1) / 2 + r, r <= c
                int c = (int)((sqrtf(8.f * (float)o + 1.f) - 1.f) * 0.5f);
                while ((c + 1) * (c + 2) / 2 <= o) ++c;
                while (c * (c + 1) / 2 > o) --c;
                const int r = o - c * (c + 1) / 2;
                st->Ht[r * KMAX + c] = s;
                st->Ht[c * KMAX + r] = s;
            }
        } else if (o < E + K) {
            const int k = o - E;
            double s = lane_sum_strided(g_part + (size_t)k * GH, GC, lane);
            s = warp_sum_f64(s);
            if (lane == 0) st->gt[k] = s;
        } else if (o < E + 2 * K) {
            const int k = o - E - K;
            float s = lane_sum_strided(gn_part + (size_t)k * GH, GC, lane);
            s = warp_sum_f32(s);
            if (lane == 0) st->gn[k] = s;
        } else {
            double s = lane_sum_strided(F_part, GE, lane);
            s = warp_sum_f64(s);
            if (lane == 0) st->Ft = s;
        }
    }
}

// ---- tagged words ------------------------------------------------------------
// The persistent solve's reduced sums as 64-bit words, 32 bits of the value
// under the evaluation's number: a reader polls the words it needs, so that no
// barrier (release, counter, poll, then the loads) lies between the reduction and
// the step.  An aligned 64-bit access is single-copy atomic, so a word with the
// right number has its value.  Every word of an evaluation is read by every
// block before it arrives at the next evaluation's barrier, and rewritten only
// after that barrier.
__device__ __forceinline__ void word_put(unsigned long long* p, unsigned v, unsigned tag) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(((unsigned long long)tag << 32) | v) : "memory");
}
__device__ __forceinline__ unsigned long long word_get(const unsigned long long* p) {
    unsigned long long w;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
    return w;
}
__device__ __forceinline__ void word_put_f64(unsigned long long* p, double v, unsigned tag) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    word_put(p, (unsigned)b, tag);
    word_put(p + 1, (unsigned)(b >> 32), tag);
}
__device__ __forceinline__ double words_f64(unsigned long long lo, unsigned long long hi) {
    return __longlong_as_double((long long)((hi << 32) | (lo & 0xffffffffull)));
}

// Reduction of the partial sums of one evaluation (as master_reduce_part) into
// tagged words.  last_only: only the outputs of variable K - 1 (column K - 1 of H,
// its g and gn).
__device__ __forceinline__ void master_reduce_words(const float* __restrict__ H_part,
                                                    const double* __restrict__ g_part,
                                                    const float* __restrict__ gn_part,
                                                    const double* __restrict__ F_part, int GS, int G, int K,
                                                    MasterDev* st, int bid, bool last_only, unsigned tag) {
    const int E = K * (K + 1) / 2;
    const int lane = threadIdx.x & 31;
    const int n_out = last_only ? K + 2 : E + 2 * K + 1;
    // consecutive outputs on different blocks: the FP64 sums (g, F) are consecutive,
    // and an SM's FP64 pipe is slow
    for (int o_ = bid + G * ((int)threadIdx.x >> 5); o_ < n_out; o_ += G * ((int)blockDim.x >> 5)) {
        const int o = !last_only ? o_ : o_ < K ? E - K + o_ : o_ == K ? E + K - 1 : E + 2 * K - 1;
        if (o < E) {  // the factorisation is FP32: so is this sum
            const float x = warp_sum_f32(lane_sum_strided(H_part + (size_t)o * GS, G, lane));
            if (lane == 0) {  // o = c (c + 1) / 2 + r, r <= c: row c, column r of the lower triangle
                int c = (int)((sqrtf(8.f * (float)o + 1.f) - 1.f) * 0.5f);
                while ((c + 1) * (c + 2) / 2 <= o) ++c;
                while (c * (c + 1) / 2 > o) --c;
                word_put(&st->wH[c * KMAX + o - c * (c + 1) / 2], __float_as_uint(x), tag);
            }
        } else if (o < E + K) {
            const double x = warp_sum_f64(lane_sum_strided(g_part + (size_t)(o - E) * GS, G, lane));
            if (lane == 0) word_put_f64(&st->wg[2 * (o - E)], x, tag);
        } else if (o < E + 2 * K) {
            const float x = warp_sum_f32(lane_sum_strided(gn_part + (size_t)(o - E - K) * GS, G, lane));
            if (lane == 0) word_put(&st->wgn[o - E - K], __float_as_uint(x), tag);
        } else {
            const double x = warp_sum_f64(lane_sum_strided(F_part, G, lane));
            if (lane == 0) word_put_f64(&st->wF[0], x, tag);
        }
    }
}

// The step's threads: the first STEP_T of a block that may have more.
constexpr int STEP_T = 256;
constexpr int H_LD = KMAX + 4;  // row stride of H in the step's memory
static_assert(STEP_T == 256 && KMAX == 64, "the step maps a 16 x 16 thread grid onto 64 x 64 entries");

// Barrier of the step's threads.
__device__ __forceinline__ void step_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// The bit pattern of a non-negative double (0 for a NaN, as fmax would skip it).
// Patterns order like the values, so maxima and comparisons of non-negative
// doubles stay on the integer pipe: FP64 issues at 1/64 of the FP32 rate on
// this part, and the step is a chain of them.
constexpr unsigned long long INF_BITS = 0x7ff0000000000000ull;
__device__ __forceinline__ unsigned long long raw_bits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ unsigned long long nonneg_bits(double v) {
    const unsigned long long b = raw_bits(v);
    return b <= INF_BITS ? b : 0ull;
}
// fmax(v, 0.0) on the bit pattern.
__device__ __forceinline__ double relu_bits(double v) { return __longlong_as_double((long long)nonneg_bits(v)); }
// |v| as a bit pattern, 0 for a NaN.
__device__ __forceinline__ unsigned long long abs_bits(double v) {
    const unsigned long long b = raw_bits(v) & 0x7fffffffffffffffull;
    return b <= INF_BITS ? b : 0ull;
}
// A non-negative double rounded towards 0 to a float (0 below 2^-126, infinity from 2^128 on).
__device__ __forceinline__ float float_below(unsigned long long b) {
    const unsigned long long e = b >> 29;  // exponent and the first 23 fraction bits
    return e < (897ull << 23)   ? 0.f
           : e >= (1151ull << 23) ? __int_as_float(0x7f800000)
                                  : __uint_as_float((unsigned)(e - (896ull << 23)));
}
// Maximum over the warp: of the high words, then of the low words under it.
__device__ __forceinline__ unsigned long long warp_max_bits(unsigned long long b) {
    const unsigned hi = __reduce_max_sync(FULL, (unsigned)(b >> 32));
    const unsigned lo = __reduce_max_sync(FULL, (unsigned)(b >> 32) == hi ? (unsigned)b : 0u);
    return ((unsigned long long)hi << 32) | lo;
}

// Solver state of the persistent solve, one copy per block: every block takes
// the same step from the same reduced sums.
struct StepState {
    double y[KMAX], yt[KMAX], d[KMAX], g[KMAX];
    double F, alpha, tol, res;
    int iter, phase, done, status, n_eval, final_pending;
};

// Shared memory of the step.
struct StepMem {
    __align__(16) float H[KMAX][H_LD];      // H as reduced (lower triangle)
    __align__(16) float prow[2][2][KMAX];   // [step mod 2]: the pivot rows
    __align__(16) float pcol[2][2][KMAX];   // and the pivot columns
    __align__(16) float4 piv[2];            // the pivot block d00, d10, d11
    __align__(16) float2 pu[2];             // the right-hand side of the pivot rows
    float rhs[KMAX];                        // -g of the free variables in order, then the solution
    int fidx[KMAX];                         // free variables in order
    unsigned bal[2], diag[2];
    int viol[2], ok;
    unsigned long long res[2], gmax[2];
    float decf[2], absf[2], dF;
    double dec[2];
};

// Damped FP32 solve of (H_FF + lam I) x = b (nf free variables) by Gauss-Jordan
// elimination, two pivots a step; x in sm.rhs.  Returns false when a pivot is not
// in [2^-126, 2^126].  Thread (tr, tc) of a 16 x 16 grid holds the 4 x 4 entries
// from (4 tr, 4 tc) in registers, threads tc = 0 also the right-hand side of their
// rows.  Per step the owners publish the two pivot rows and columns (and the
// right-hand side's entries) in shared memory; after the step's one barrier
// every thread eliminates the pair as an L D L^T of its 2 x 2 block would (d0,
// l = d10 / d0, d1 = d11 - l d10) from its rows, those already eliminated
// included, so that no triangular solve is left: at the end each pair's 2 x 2
// system gives its x.  The chain of a step is a barrier, one shared-memory round
// trip and two reciprocals.  The whole step at 48 variables takes 8.8 us (64:
// 10.5), against 9.1 (11.7) with panels of four columns and a triangular solve.
// The reciprocals are the hardware approximation (__fdividef, within 2 ulp
// for pivots in [2^-126, 2^126]; others fail the check and the caller takes a
// larger shift).  H is symmetric positive definite up to rounding, and shifted,
// so the diagonal pivots need no search.
__device__ __forceinline__ bool step_solve(StepMem& sm, int k, int nf, const float (&H4)[4][4], const float (&b4)[4],
                                           float lam) {
    const int tr = k & 15, tc = k >> 4;
    float M[4][4], u[4], pi0[2] = {0.f, 0.f}, pl[2] = {0.f, 0.f}, pi1[2] = {0.f, 0.f};
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        u[a] = b4[a];
#pragma unroll
        for (int b = 0; b < 4; ++b) M[a][b] = H4[a][b] + (tr == tc && a == b ? lam : 0.f);
    }
    bool good = true;
    const int steps = (nf + 1) >> 1;
    const bool rows_in = 4 * tr < nf;
    for (int s0 = 0; s0 < steps; s0 += 2) {
        const int P = s0 >> 1;  // the pivot rows' thread row: two steps each
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (s0 + h < steps) {
                constexpr float ZERO = 0.f;
                if (tr == P && tc >= P) {
                    *reinterpret_cast<float4*>(&sm.prow[h][0][4 * tc]) =
                        make_float4(M[2 * h][0], M[2 * h][1], M[2 * h][2], M[2 * h][3]);
                    *reinterpret_cast<float4*>(&sm.prow[h][1][4 * tc]) =
                        make_float4(M[2 * h + 1][0], M[2 * h + 1][1], M[2 * h + 1][2], M[2 * h + 1][3]);
                }
                if (tc == P && rows_in) {
                    *reinterpret_cast<float4*>(&sm.pcol[h][0][4 * tr]) =
                        make_float4(M[0][2 * h], M[1][2 * h], M[2][2 * h], M[3][2 * h]);
                    *reinterpret_cast<float4*>(&sm.pcol[h][1][4 * tr]) =
                        make_float4(M[0][2 * h + 1], M[1][2 * h + 1], M[2][2 * h + 1], M[3][2 * h + 1]);
                    if (tr == P)
                        sm.piv[h] = make_float4(M[2 * h][2 * h], M[2 * h + 1][2 * h], M[2 * h + 1][2 * h + 1], ZERO);
                }
                if (tc == 0 && tr == P) sm.pu[h] = make_float2(u[2 * h], u[2 * h + 1]);
                step_sync();
                if (rows_in && (tc >= P || tc == 0)) {
                    const float4 d = sm.piv[h];
                    float4 c0 = *reinterpret_cast<const float4*>(&sm.pcol[h][0][4 * tr]);
                    float4 c1 = *reinterpret_cast<const float4*>(&sm.pcol[h][1][4 * tr]);
                    const float4 r0 = *reinterpret_cast<const float4*>(&sm.prow[h][0][4 * tc]);
                    float4 r1 = *reinterpret_cast<const float4*>(&sm.prow[h][1][4 * tc]);
                    const float2 e = sm.pu[h];
                    const float i0 = __fdividef(1.f, d.x);
                    const float l = d.y * i0;
                    const float d1 = fmaf(-l, d.y, d.z);
                    const float i1 = __fdividef(1.f, d1);
                    r1 = make_float4(fmaf(-l, r0.x, r1.x), fmaf(-l, r0.y, r1.y), fmaf(-l, r0.z, r1.z),
                                     fmaf(-l, r0.w, r1.w));
                    float m0[4] = {c0.x * i0, c0.y * i0, c0.z * i0, c0.w * i0};
                    float m1[4] = {fmaf(-l, c0.x, c1.x) * i1, fmaf(-l, c0.y, c1.y) * i1, fmaf(-l, c0.z, c1.z) * i1,
                                   fmaf(-l, c0.w, c1.w) * i1};
                    if (tr == P) {  // the pivot rows stay
                        m0[2 * h] = m0[2 * h + 1] = 0.f;
                        m1[2 * h] = m1[2 * h + 1] = 0.f;
                    }
                    const float q0[4] = {r0.x, r0.y, r0.z, r0.w}, q1[4] = {r1.x, r1.y, r1.z, r1.w};
                    if (tc >= P)
#pragma unroll
                        for (int a = 0; a < 4; ++a)
#pragma unroll
                            for (int b = 0; b < 4; ++b) M[a][b] = fmaf(-m1[a], q1[b], fmaf(-m0[a], q0[b], M[a][b]));
                    if (tc == 0) {
                        const float e1 = fmaf(-l, e.x, e.y);
#pragma unroll
                        for (int a = 0; a < 4; ++a) u[a] = fmaf(-m1[a], e1, fmaf(-m0[a], e.x, u[a]));
                        good = good && d.x >= 1.17549435e-38f && d.x <= 8.50705917e37f && d1 >= 1.17549435e-38f &&
                               d1 <= 8.50705917e37f;
                        if (tr == P) {
                            pi0[h] = i0;
                            pl[h] = l;
                            pi1[h] = i1;
                        }
                    }
                }
            }
        }
    }
    if (tc == 0) {  // half a warp
        if (rows_in)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float x1 = fmaf(-pl[h], u[2 * h], u[2 * h + 1]) * pi1[h];
                sm.rhs[4 * tr + 2 * h] = fmaf(-pl[h], x1, u[2 * h] * pi0[h]);
                sm.rhs[4 * tr + 2 * h + 1] = x1;
            }
        if (tr == 0) sm.ok = good;  // thread (0, 0) takes part in every step
    }
    step_sync();
    return sm.ok != 0;
}

// The projected-Newton step: variable v = k mod 64 of thread k; warps 0 and 1 test
// the KKT conditions, warps 2 and 3 the decrease, all threads share the
// factorisation.  LOCAL: the state is the block's shared copy (persistent solve);
// else it is the plan's, in device memory, read through L2.  The reduced sums:
// Ft, gt and gn of variable v, and H's lower triangle in sm.H (visible after the
// first barrier).  The caller synchronises the block before and after it.
//
// A chain of dependent block phases, so latency is all that counts: FP64 only
// where a decision needs it (the tests are made in FP32 with their error
// margins and repeated in FP64 when they fall inside).
template <bool LOCAL, class ST>
__device__ __forceinline__ void master_step_body(ST* st, int K, double Ft, double gt_, float gn_, int max_iter,
                                                 double tol_rel, double sigma, StepMem& sm) {
    auto get = [](const auto* p) {
        if constexpr (LOCAL)
            return *p;
        else
            return __ldcg(p);
    };
    const int k = threadIdx.x, lane = k & 31, warp = k >> 5;
    const int v = k & (KMAX - 1);
    const double yt_ = get(&st->yt[v]), y_ = get(&st->y[v]), g_ = get(&st->g[v]);
    const int phase = get(&st->phase), iter0 = get(&st->iter), n_eval0 = get(&st->n_eval);
    const double tol0 = get(&st->tol), F0 = get(&st->F), alpha0 = get(&st->alpha);
    const bool own = v < K;
    const bool lead = k < KMAX && own;  // thread k < K owns variable k
    const double yt = own ? yt_ : 0.0, gt = own ? gt_ : 0.0;
    const float bneg = -(float)gt;
    // tolerance of this solve from the gradient at the warm start
    double tol = tol0;
    if (phase == 0) {
        if (warp < 2) {
            const unsigned long long m = warp_max_bits(own ? abs_bits(gt) : 0ull);
            if (lane == 0) sm.gmax[warp] = m;
        }
        step_sync();
        if (warp < 2) tol = tol_rel * fmax(__longlong_as_double((long long)max(sm.gmax[0], sm.gmax[1])), 1e-300);
    }
    if (warp < 2) {
        // |y - P(y - g)| = |min(y, g)| (y >= 0)
        const unsigned long long yb = raw_bits(yt), gb = raw_bits(gt), ga = gb & 0x7fffffffffffffffull;
        const unsigned long long rt = !own ? 0ull : (gb >> 63) ? (ga <= INF_BITS ? ga : yb) : min(gb, yb);
        const float rf = float_below(rt), lf = fmaf((float)(NOISE * (double)U32), own ? gn_ : 0.f, float_below(raw_bits(tol)));
        bool vi = own && rf > lf * (1.f + 1e-6f);
        const bool sure = !own || vi || rf * (1.f + 1e-6f) <= lf;
        if (__any_sync(FULL, !sure))
            if (!sure) vi = rt > raw_bits(tol + NOISE * (double)U32 * (double)gn_);
        const int viol = __any_sync(FULL, vi) ? 1 : 0;
        const unsigned long long rm = warp_max_bits(rt);
        if (lane == 0) {
            sm.res[warp] = rm;
            sm.viol[warp] = viol;
        }
    } else if (warp < 4 && phase != 0) {
        // g^T (y_t - y) in FP32, with the sum of its terms' magnitudes
        const float t = own ? (float)g_ * (float)(yt - y_) : 0.f;
        float s = warp_sum_f32(t), a = warp_sum_f32(fabsf(t));
        if (lane == 0) {
            sm.decf[warp - 2] = s;
            sm.absf[warp - 2] = a;
            if (warp == 2) sm.dF = (float)(Ft - F0);
        }
    }
    step_sync();
    const unsigned long long rb = max(sm.res[0], sm.res[1]);
    const int viol = sm.viol[0] | sm.viol[1];
    const bool cap = iter0 >= max_iter + 64;
    bool accept = !cap;
    if (accept && phase != 0 && viol) {  // Armijo: F_t <= F + sigma g^T (y_t - y)
        const float sg = (float)sigma, dF = sm.dF;
        const float thr = sg * (sm.decf[0] + sm.decf[1]);
        const float m = 1e-5f * (sg * (sm.absf[0] + sm.absf[1]) + fabsf(dF));
        accept = dF <= thr - m;
        if (!accept && !(dF > thr + m)) {  // too close to tell in FP32 (the same for every thread)
            if (warp < 2) {
                double dec = own ? g_ * (yt - y_) : 0.0;
                dec = warp_sum_f64(dec);
                if (lane == 0) sm.dec[warp] = dec;
            }
            step_sync();
            accept = Ft <= F0 + sigma * (sm.dec[0] + sm.dec[1]);
        }
    }
    if (k == 0) {
        st->n_eval = n_eval0 + 1;
        if (phase == 0) st->tol = tol;
    }
    if (cap) {
        if (k == 0) {
            st->status = MASTER_MAXITER;
            st->final_pending = 1;
            st->done = 1;
        }
        return;
    }
    if (!accept) {
        const double alpha = alpha0 * 0.5;
        if (alpha < 9.3e-10) {  // 2^-30: the line search found no decrease
            if (k == 0) {
                st->status = MASTER_STALLED;
                st->final_pending = 1;
                st->done = 1;
            }
            return;
        }
        if (lead) st->yt[k] = fmax(y_ + alpha * get(&st->d[k]), 0.0);
        if (k == 0) {
            st->alpha = alpha;
            st->iter = iter0 + 1;
            st->phase = 1;
        }
        return;
    }
    // accept the trial point
    if (lead) {
        st->y[k] = yt;
        st->g[k] = gt;
    }
    if (k == 0) {
        st->F = Ft;
        st->res = __longlong_as_double((long long)rb);
    }
    if (!viol || iter0 >= max_iter) {
        if (k == 0) {
            st->status = viol ? MASTER_MAXITER : MASTER_CONVERGED;
            st->done = 1;
        }
        return;
    }
    // epsilon-active set, free variables compacted in order
    const bool active = lead && raw_bits(yt) <= min(raw_bits(1e-3), rb) && nonneg_bits(gt) > 0ull;
    const bool fr = lead && !active;
    const float hd = fr ? sm.H[k][k] : 0.f;
    if (k < KMAX) {
        const unsigned bal = __ballot_sync(FULL, fr);
        const unsigned md = __reduce_max_sync(FULL, hd > 0.f ? __float_as_uint(hd) : 0u);
        if (lane == 0) {
            sm.bal[warp] = bal;
            sm.diag[warp] = md;
        }
    }
    step_sync();
    const int nf = __popc(sm.bal[0]) + __popc(sm.bal[1]);
    const float maxdiag = __uint_as_float(max(sm.diag[0], sm.diag[1]));
    int pos = 0;
    if (fr) {
        pos = (warp ? __popc(sm.bal[0]) : 0) + __popc(sm.bal[warp] & ((1u << lane) - 1u));
        sm.fidx[pos] = k;
        sm.rhs[pos] = bneg;
    }
    double d = active ? -gt : 0.0;
    step_sync();
    const int r0 = 4 * (k & 15), q0 = 4 * (k >> 4);  // this thread's 4 x 4 entries
    float H4[4][4], b4[4];
    {
        int fi[4], fq[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            fi[a] = r0 + a < nf ? sm.fidx[r0 + a] : -1;
            fq[a] = q0 + a < nf ? sm.fidx[q0 + a] : -1;
            b4[a] = r0 + a < nf ? sm.rhs[r0 + a] : 0.f;
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b)
                H4[a][b] = fi[a] >= 0 && fq[b] >= 0 ? sm.H[max(fi[a], fq[b])][min(fi[a], fq[b])] : 0.f;
    }
    float lam = 1e-6f * maxdiag + 1e-30f;
    bool ok = false;
    for (int attempt = 0; attempt < 6 && !ok; ++attempt) {  // a failed pivot: a 100x larger shift
        ok = step_solve(sm, k, nf, H4, b4, lam);
        lam *= 100.f;
    }
    if (fr) {
        if (ok)
            d = (double)sm.rhs[pos];
        else
            d = -gt / (hd > 0.f ? (double)hd : 1.0);
    }
    if (lead) {
        st->d[k] = d;
        st->yt[k] = relu_bits(yt + d);
    }
    if (k == 0) {
        st->alpha = 1.0;
        st->iter = iter0 + 1;
        st->phase = 1;
    }
}

// Reduction of the evaluation's partial sums, then the step: every block reduces
// its share of the outputs, and the block that finishes last (a ticket taken
// after a memory fence, so all outputs are visible to it) takes the step.  No
// block waits for another.  The while-node condition is set to "not done" on
// every path that continues; the evaluation cap inside the step guarantees that
// done is reached.
__global__ void __launch_bounds__(STEP_T, 1) k_master_reduce_step(const float* __restrict__ H_part,
                                                               const double* __restrict__ g_part,
                                                               const float* __restrict__ gn_part,
                                                               const double* __restrict__ F_part, int GH, int GE,
                                                               MasterDev* __restrict__ st, int max_iter,
                                                               double tol_rel, double sigma,
                                                               cudaGraphConditionalHandle cond, int use_cond) {
    __shared__ int s_last;
    __shared__ StepMem sm;
    if (st->done) {  // the same for every block: only the last block of a launch changes it
        if (use_cond && blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(cond, 0u);
        return;
    }
    master_reduce_part(H_part, g_part, gn_part, F_part, GH, GH, GE, st->K, st, blockIdx.x, gridDim.x);
    __syncthreads();
    if (threadIdx.x == 0) s_last = atom_add_acq_rel_gpu(&st->ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    if (threadIdx.x == 0) st->ticket = 0;
    if (__ldcg(&st->err)) {  // a tile copy was lost in an evaluation: stop with the last accepted point
        if (threadIdx.x == 0) {
            st->status = MASTER_ERROR;
            st->final_pending = 1;
            st->done = 1;
        }
    } else {
        const int K = __ldcg(&st->K), tid = threadIdx.x, v = tid & (KMAX - 1);
        const double Ft = __ldcg(&st->Ft), gt = __ldcg(&st->gt[v]);
        const float gn = __ldcg(&st->gn[v]);
#pragma unroll
        for (int m = 0; m < KMAX * KMAX / STEP_T; ++m) {
            const int r = 4 * m + (tid >> 6);
            if (v <= r && r < K) sm.H[r][v] = __ldcg(&st->Ht[r * KMAX + v]);
        }
        __syncthreads();
        master_step_body<false>(st, K, Ft, gt, gn, max_iter, tol_rel, sigma, sm);
    }
    if (use_cond && threadIdx.x == 0) cudaGraphSetConditional(cond, st->done ? 0u : 1u);
}

// ---- the master solve as one persistent cooperative kernel -------------------
// One block of 16 warps per SM, all co-resident (cooperative launch).  A warp
// owns tiles of 32 voxels, one per lane, interleaved over the grid's warps (so the
// active voxels of a compact target spread over them), and meets the other
// warps of its block only when its tiles are done.  A tile's doses (512 bytes per
// group of four columns) come to the warp's ring in shared memory by 16-byte
// asynchronous copies, tiles ahead; they stay there from one evaluation to
// the next where the ring holds all of the warp's tiles.  Per Newton iteration:
//   A. per tile: the lanes form the compensated z of their voxel, then pi, h, F
//      and the voxel's curvature state; the voxels with h > 0 then add to g and
//      its rounding scale, a lane per voxel and group of columns; the
//      voxels whose h changed go to the warp's list and, while there is room,
//      their doses to a block-wide pool of rows.  After its tiles the block adds
//      the listed changes to its kept partial H (Delta h s s^T, a 2x2 block of H
//      per thread) and writes its partials to column b of the partial arrays;
//   grid barrier;
//   B. every block reduces its share of the outputs in a fixed order, into words
//      tagged with the evaluation's number;
//   C. every block collects the words and takes the same Newton step from them, on
//      its own copy of the solver state, so no block waits for another's step.
// The first evaluation of a solve that follows a converged one on the same
// grid, with one more aperture at intensity 0, is at the point the last one ended
// on: z, pi, F, g and H of the older apertures stand, and only the new
// aperture's g and its column of H are formed (MODE_EXT).
// One plan of 50 apertures, H&N-shaped (304,184 voxels), FP16 storage: 6.64 ms,
// against 8.70 with blocks of 256 threads on 128-voxel chunks copied by TMA, five
// block barriers to a chunk, and the step taken by one block between two grid
// barriers; 8 prostate-shaped plans of 20 apertures at once 8.33 ms (10.96).  An
// evaluation now takes 20.6 us on average (28 before): tiles 6.3, the update of
// H 1.6, partials 0.7, waiting for the last block 2.5, reduction and collection
// 4.0, step 5.0.  The pass is bound by instruction issue, the rest by latency.
// Every wait is bounded: after GRID_WAIT_LIMIT polls the block reports st->err = 2,
// marks the barrier broken (later launches of the solve return at entry) and every
// block leaves at its next wait.
constexpr int PT = 512;            // threads per block (the step takes the first STEP_T)
constexpr int PW = PT / 32;
// Up to this many blocks each thread of the step polls its own words at once (20
// apertures on 19,200 voxels, 38 blocks: 1.93 ms, 1.97 if a warp polls one word
// first, which is a second trip to L2); on more, their polls keep the L2 from the
// reducing warps (152 blocks, 50 apertures: 6.70 ms, 6.64 after one word).
constexpr int DIRECT_BLOCKS = 64;
constexpr int RING = 21;           // groups of four columns of a tile in a warp's ring
constexpr int RING_LD = 132;       // floats of a group in the ring: 32 voxels x 4, and 4 against bank conflicts
constexpr size_t RING_BYTES = (size_t)PW * RING * RING_LD * sizeof(float);
constexpr int LIST = 128;          // listed voxels of a warp: four tiles
constexpr int HB = KMAX;           // rows of changed voxels held at a time for the update of H (the step's matrix A)
enum { MODE_FULL = 0, MODE_EXT = 1, MODE_INC = 2 };  // the kept partial H: rebuilt, extended by a column, updated
constexpr int GRID_WAIT_LIMIT = 1 << 22;

__device__ __forceinline__ void copy16_async(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// A warp's tiles in its ring: copy n (n = 0, 1, ... over the launch) is tile n
// mod tiles; group g of copy n sits at position (n KG + g) mod size.  size is a
// whole number of tiles (two to four ahead, or all of them: nothing is copied
// twice), or, where the ring holds fewer than two, the whole ring: then the next
// tile's first RING - KG groups are ahead and its others follow when the tile is
// released.  A group's 32 x 16 bytes are followed by 16 unused ones, so that
// the same voxel of eight groups, as the gradient reads it, falls on different
// banks.
struct TileRing {
    float* buf;
    const float* src;            // the lane's voxel of the warp's first tile, group 0
    size_t gstride, tstride;     // floats from one group to the next, from one tile to the next
    int KG, size, tiles, slots;  // slots: tiles the ring holds; 0: the fractional form
    int n, pos;                  // the copy in use and its position
    int iss_tile, iss_pos;       // next tile to issue (index in the warp's), position of its next group
    bool resident;

    __device__ __forceinline__ void issue(int g0, int g1) {  // groups [g0, g1) of tile iss_tile
        const float* p = src + (size_t)iss_tile * tstride + (size_t)g0 * gstride;
        float* d = buf + iss_pos * RING_LD + (threadIdx.x & 31) * 4;
        for (int g = g0; g < g1; ++g, p += gstride) {
            copy16_async(d, p);
            d += RING_LD;
            if (++iss_pos == size) {
                iss_pos = 0;
                d -= size * RING_LD;
            }
        }
        copies_commit();
    }
    __device__ __forceinline__ void next_tile() {
        if (++iss_tile == tiles) iss_tile = 0;
    }
    __device__ __forceinline__ void init(float* b, const float* slab, int ld, int KG_, int t0, int stride, int n32) {
        buf = b;
        src = slab + ((size_t)t0 * 32 + (threadIdx.x & 31)) * 4;
        gstride = (size_t)ld * 4;
        tstride = (size_t)stride * 128;
        KG = KG_;
        tiles = t0 < n32 ? (n32 - 1 - t0) / stride + 1 : 0;
        const int fit = RING / KG;
        resident = tiles <= fit;
        slots = resident ? tiles : fit >= 2 ? min(fit, 4) : 0;
        size = slots ? slots * KG : RING;
        n = pos = iss_tile = iss_pos = 0;
        if (tiles == 0) return;
        for (int k = 0; k < max(slots, 1); ++k) {
            issue(0, KG);
            next_tile();
        }
        if (slots == 0) issue(0, RING - KG);  // the first groups of the next tile
    }
    // Copy n has arrived (every lane; the lanes see each other's pieces).
    __device__ __forceinline__ void wait() {
        if (resident)
            copies_wait<0>();
        else if (slots == 4)
            copies_wait<3>();
        else if (slots == 3)
            copies_wait<2>();
        else
            copies_wait<1>();
        __syncwarp();
    }
    // Copy n has been read (by the whole warp): its place is refilled.
    __device__ __forceinline__ void release() {
        ++n;
        pos += KG;
        if (resident) {
            if (n == tiles) n = pos = 0;
            return;
        }
        if (pos >= size) pos -= size;
        __syncwarp();
        if (slots) {
            issue(0, KG);
            next_tile();
        } else {
            issue(RING - KG, KG);
            next_tile();
            issue(0, RING - KG);
        }
    }
    // Group g of the copy in use: its 32 voxels' float4 each.
    __device__ __forceinline__ const float* group(int g) const {
        const int x = pos + g;
        return buf + (x >= size ? x - size : x) * RING_LD;
    }
};

// Barrier over the blocks of one cooperative launch with one acquire-release
// atomic per arrival.  The counter only grows: barrier e of a launch completes when it
// reaches base + (e + 1) G.  base, the counter at launch, is a multiple of G
// (each completed barrier adds exactly G), and every block reads it before its
// first arrival, when fewer than G arrivals can have happened, so
// base = c - c % G for whatever value c it reads.  Waiters poll the counter.
// The host zeroes it before each solve; a solve's barriers stay far below
// 2^32 arrivals.  *s_target is the block's next target.
__device__ __forceinline__ bool grid_sync(GridBar* gb, unsigned nblocks, unsigned* s_target, int* s_flag) {
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned target = *s_target + nblocks;
        *s_target = target;
        // release: the block's writes (ordered by the __syncthreads above)
        // before the arrival; acquire: the other blocks' writes after it
        const unsigned arrived = atom_add_acq_rel_gpu(&gb->count, 1u) + 1u;
        int ok = 1;
        if (arrived != target) {
            int i = 0;
            while ((int)(ld_acquire_gpu(&gb->count) - target) < 0 && ++i < GRID_WAIT_LIMIT) {
                __nanosleep(64);
                if ((i & 4095) == 0 && ld_acquire_gpu(&gb->broken)) i = GRID_WAIT_LIMIT - 1;  // another gave up
            }
            ok = i < GRID_WAIT_LIMIT;
            if (!ok) atomicExch(&gb->broken, 1u);
        }
        *s_flag = ok;
    }
    __syncthreads();
    return *s_flag != 0;
}

// s + c of four chains as a pair.
__device__ __forceinline__ void chains_sum(const float (&sc)[4], const float (&cc)[4], float& s, float& c) {
    s = sc[0];
    c = cc[0];
#pragma unroll
    for (int q = 1; q < 4; ++q) {
        const float t2 = s + sc[q];
        const float bb = t2 - s;
        const float e = (s - (t2 - bb)) + (sc[q] - bb);
        s = t2;
        c += e + cc[q];
    }
}

// z of one voxel: the compensated dot product of its doses dose4(c), c < KP
// (columns K .. KP - 1 meet y = 0), with y, in four chains, as a pair (s, c).
// s_y: (yh, yl) of two columns per entry.
template <class Dose4>
__device__ __forceinline__ void voxel_dot(int KP, const float4* s_y, float& s, float& c, Dose4 dose4) {
    float sc[4] = {0.f, 0.f, 0.f, 0.f}, cc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int k = 0; k < KP; k += 4) {
        const float4 a = dose4(k);
        const float4 y0 = s_y[k >> 1], y1 = s_y[(k >> 1) + 1];
        dot2_step(sc[0], cc[0], a.x, y0.x, y0.y);
        dot2_step(sc[1], cc[1], a.y, y0.z, y0.w);
        dot2_step(sc[2], cc[2], a.z, y1.x, y1.y);
        dot2_step(sc[3], cc[3], a.w, y1.z, y1.w);
    }
    chains_sum(sc, cc, s, c);
}

// The same where every dose is >= 0 and z is known to within a factor: the chains
// start at C, a power of two at least 4 |z_last| (z_last: the voxel's dose at the
// previous evaluation).  While a chain's own sum stays within C / 2, every
// partial sum lies in [C, 1.5 C], so t = RN(s + a yh) differs from s by an exact
// float d, the rounding error a yh - d has at most ulp(C) / 2 and one FMA gives it:
// five operations a term instead of dot2_step's eleven, with the same second-order
// error (terms of size u ulp(z)).  Sums of non-negative terms only grow, so
// the last one within C / 2 proves the others; returns false otherwise
// (also for a NaN), and the caller takes voxel_dot.
__device__ __forceinline__ void dot2_biased(float& s, float& c, float a, float yh, float yl) {
    const float t = fmaf(a, yh, s);
    const float d = t - s;
    c += fmaf(a, yl, fmaf(a, yh, -d));
    s = t;
}
template <class Dose4>
__device__ __forceinline__ bool voxel_dot_biased(int KP, const float4* s_y, float z_last, float& s, float& c,
                                                 Dose4 dose4) {
    const float C = __uint_as_float((__float_as_uint(z_last) & 0x7f800000u) + (3u << 23));
    float sc[4] = {C, C, C, C}, cc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
    for (int k = 0; k < KP; k += 4) {
        const float4 a = dose4(k);
        const float4 y0 = s_y[k >> 1], y1 = s_y[(k >> 1) + 1];
        dot2_biased(sc[0], cc[0], a.x, y0.x, y0.y);
        dot2_biased(sc[1], cc[1], a.y, y0.z, y0.w);
        dot2_biased(sc[2], cc[2], a.z, y1.x, y1.y);
        dot2_biased(sc[3], cc[3], a.w, y1.z, y1.w);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) sc[q] -= C;  // exact
    chains_sum(sc, cc, s, c);
    return sc[0] + sc[1] + sc[2] + sc[3] <= 0.5f * C;
}

// BATCH: one launch for several plans, blocks [g GB, (g + 1) GB) solving the
// master problem of tasks[g] with its own barrier and partial arrays (the
// plans' solves run side by side, each on GB blocks); otherwise one plan, t1,
// on the whole grid.  Every other difference is the block's index within its
// group (bid) and the group's size (G).
// The master solve of one plan (a task) by a group of G co-resident blocks, bid
// the block's index in it; ring_mem the dynamic shared memory; s_target / s_flag the
// group barrier's shared state (s_target: the block's next target, already based
// on the barrier counter).
// Every block of the group calls it with the same K.
__device__ __forceinline__ void master_solve_group(
    const float* __restrict__ slab, int ld, int V, int GS, int S, int max_iter, MasterDev* st,
    GridBar* __restrict__ gb, float* __restrict__ H_part, double* __restrict__ g_part, float* __restrict__ gn_part,
    double* __restrict__ F_part, const uint8_t* __restrict__ vstruct, const StructTermsF* __restrict__ tf,
    double tol_rel, float* __restrict__ z_out, float* __restrict__ pi_out, CGDev* __restrict__ cg,
    uint8_t* __restrict__ vstate, float* __restrict__ H_keep, bool nonneg, int bid, int G, int K, double sigma,
    float* ring_mem, unsigned* s_target, int* s_flag) {
    // the step's memory; its H holds rows of changed voxels between steps
    __shared__ StepMem sm;
    __shared__ StepState ss;
    __shared__ __align__(16) float2 s_y[KMAX];
    __shared__ StructTermsF s_tf[SMAX];
    __shared__ float2 s_al[PW][32];  // a tile's active voxels: pi (EXT: h times the new column's dose), offset in a group
    __shared__ float s_red[2][PW];
    // a warp's list: the changed voxels, their change of h and their row of the
    // pool; then the warps' gradient sums
    __shared__ __align__(16) int s_dj[PW][LIST];
    __shared__ __align__(16) float s_dh[PW][LIST];
    __shared__ unsigned char s_ds[PW][LIST];
    __shared__ float s_ch[HB];  // change of h of the rows in hand
    __shared__ int s_row[HB];   // their rows of A
    __shared__ int s_nd[PW];
    __shared__ int s_mode0, s_pool, s_lost;
    float(*A)[H_LD] = sm.H;
    float(*s_g)[KMAX] = reinterpret_cast<float(*)[KMAX]>(&s_dj[0][0]);    // g or the new column of H
    float(*s_gn)[KMAX] = reinterpret_cast<float(*)[KMAX]>(&s_dh[0][0]);  // gn
    static_assert(KMAX <= LIST && HB <= KMAX && HB < 256, "scratch fits");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int i = tid; i < S; i += PT) s_tf[i] = tf[i];
    const int KP = (K + 3) / 4 * 4;
    // update of H: thread (eb, vl) the 2x2 blocks eb, eb + PT / NV, ... of the upper
    // triangle over every NV-th row
    const int NV = persist_lanes(K);
    const int KB = KP / 2;
    const int nb = KB * (KB + 1) / 2;
    const int vl = tid % NV;
    int rb0 = 0, cb0 = 0;
    if (tid / NV < nb) block_of(tid / NV, KB, rb0, cb0);
    // gradient: lane (vs, gl) takes the column group gl of every (32 / LP)-th active voxel
    const int KG = KP / 4;
    const int LP = KG <= 1 ? 1 : KG <= 2 ? 2 : KG <= 4 ? 4 : KG <= 8 ? 8 : 16;
    const int gl = lane & (LP - 1), vs = lane / LP;
    // tile i of this warp: bid + G (warp + PW i); warp 0 has the most
    const int n32 = (V + 31) / 32;
    const int rounds = bid < n32 ? (n32 - 1 - bid) / (PW * G) + 1 : 0;
    TileRing ring;
    ring.init(ring_mem + warp * (RING * RING_LD), slab, ld, KG, bid + G * warp, PW * G, n32);
    const float4* y4 = reinterpret_cast<const float4*>(s_y);
    int n_ev = 0;  // evaluations of this solve so far
    const unsigned tag0 = __ldcg(&st->epoch);  // evaluations of the plan before this solve
    // warm start (every block): the previous optimum, the new aperture K - 1 at 0
    if (tid < KMAX) {
        const double yv = tid < K - 1 ? __ldcg(&st->y[tid]) : 0.0;
        ss.y[tid] = yv;
        ss.yt[tid] = yv;
        ss.d[tid] = 0.0;
        ss.g[tid] = 0.0;
    }
    if (tid == 0) {
        ss.F = 0.0;
        ss.alpha = 1.0;
        ss.tol = 0.0;
        ss.res = 0.0;
        ss.iter = ss.phase = ss.done = ss.n_eval = ss.final_pending = 0;
        ss.status = MASTER_RUNNING;
        s_pool = 0;
        s_lost = 0;
        // the kept partial H: extended by the new column, kept, or rebuilt
        const int iG = __ldcg(&st->inc_G), iK = __ldcg(&st->inc_K);
        s_mode0 = iG == G && iK == K - 1 ? MODE_EXT : iG == G && iK == K ? MODE_INC : MODE_FULL;
        if (bid == 0) {  // a solve that ends early leaves these
            st->K = K;
            st->done = 0;
            st->status = MASTER_RUNNING;
            st->err = 0;
        }
    }
    __syncthreads();
    bool broken = false;
    for (;;) {
        if (tid < KMAX) {
            const double yv = tid < K ? ss.yt[tid] : 0.0;
            const float hi = (float)yv;
            s_y[tid] = make_float2(hi, (float)(yv - (double)hi));
        }
        __syncthreads();
        // ---- A. the warp's tiles
        const int mode = n_ev == 0 ? s_mode0 : MODE_INC;
        float facc = 0.f, gk = 0.f, gnk = 0.f;
        float4 ga = make_float4(0.f, 0.f, 0.f, 0.f), gna = ga;  // EXT: ga holds the new column of H
        int nd_w = 0;           // voxels in the warp's list
        bool h_written = false;
        // the lane's voxel of tile i: its label and curvature state, and its dose at
        // the last evaluation (EXT: its pi), requested one tile ahead
        auto voxel_in = [&](int i, int& lab_, unsigned& osv_, float& x_) {
            const int jj = (bid + G * (warp + PW * i)) * 32 + lane;
            const bool in = i < ring.tiles && jj < V;
            lab_ = in && S >= 0 ? (int)vstruct[jj] : 0;
            osv_ = in && mode != MODE_FULL ? (unsigned)vstate[jj] : 0u;
            x_ = in && mode != MODE_FULL ? __ldcg((mode == MODE_EXT ? pi_out : z_out) + jj) : 0.f;
        };
        int lab_n;
        unsigned osv_n;
        float x_n;
        voxel_in(0, lab_n, osv_n, x_n);
        // adds the n_a listed voxels of the tile in use: their doses times the listed
        // value to ga (and the product of the magnitudes to gna)
        auto add_rows = [&](int n_a, bool scale_too) {
            if (gl < KG) {
                const float* base = ring.group(gl);
                for (int r = vs; r < n_a; r += 32 / LP) {
                    const float2 e = s_al[warp][r];
                    const float4 a = *reinterpret_cast<const float4*>(base + __float_as_int(e.y));
                    ga.x = fmaf(a.x, e.x, ga.x);
                    ga.y = fmaf(a.y, e.x, ga.y);
                    ga.z = fmaf(a.z, e.x, ga.z);
                    ga.w = fmaf(a.w, e.x, ga.w);
                    if (scale_too) {
                        const float pa = fabsf(e.x);
                        gna.x = fmaf(fabsf(a.x), pa, gna.x);
                        gna.y = fmaf(fabsf(a.y), pa, gna.y);
                        gna.z = fmaf(fabsf(a.z), pa, gna.z);
                        gna.w = fmaf(fabsf(a.w), pa, gna.w);
                    }
                }
            }
        };
        for (int i = 0; i < rounds; ++i) {
            const bool mine = i < ring.tiles;
            const int j = (bid + G * (warp + PW * i)) * 32 + lane;
            const int lab = lab_n;
            const unsigned osv = osv_n;
            const float x_in = x_n;
            voxel_in(i + 1, lab_n, osv_n, x_n);
            if (mine && mode == MODE_EXT) {
                ring.wait();
                float hs = 0.f;
                if (j < V) {
                    const StructTermsF tt = S >= 0 ? s_tf[lab] : voxel_terms(tf, j);
                    const float a = ring.group(KG - 1)[4 * lane + ((K - 1) & 3)];
                    hs = 2.f * (((osv & 1u) ? tt.a : 0.f) + ((osv & 2u) ? tt.b : 0.f)) * a;
                    gk = fmaf(a, x_in, gk);
                    gnk = fmaf(fabsf(a), fabsf(x_in), gnk);
                }
                const unsigned am = __ballot_sync(FULL, hs != 0.f);
                if (hs != 0.f) s_al[warp][__popc(am & lt)] = make_float2(hs, __int_as_float(4 * lane));
                __syncwarp();
                add_rows(__popc(am), false);
                ring.release();
            } else if (mine) {
                ring.wait();
                auto dose4 = [&](int k) { return *reinterpret_cast<const float4*>(ring.group(k >> 2) + 4 * lane); };
                float s = 0.f, c = 0.f;
                const bool fast = nonneg && mode != MODE_FULL && voxel_dot_biased(KP, y4, x_in, s, c, dose4);
                if (__any_sync(FULL, !fast && j < V)) {
                    float s2, c2;
                    voxel_dot(KP, y4, s2, c2, dose4);
                    if (!fast) {
                        s = s2;
                        c = c2;
                    }
                }
                float p = 0.f, h = 0.f, dh = 0.f;
                if (j < V) {
                    const StructTermsF tt = S >= 0 ? s_tf[lab] : voxel_terms(tf, j);
                    const float du = (tt.tu - s) - c;
                    const float dov = (s - tt.to) + c;
                    const float u = fmaxf(du, 0.f), o = fmaxf(dov, 0.f);
                    p = 2.f * (tt.b * o - tt.a * u);
                    h = 2.f * ((du > 0.f ? tt.a : 0.f) + (dov > 0.f ? tt.b : 0.f));
                    facc = fmaf(tt.a * u, u, fmaf(tt.b * o, o, facc));
                    z_out[j] = s + c;  // the state of the round when this point is the final one
                    pi_out[j] = p;
                    const unsigned nsv = (du > 0.f ? 1u : 0u) | (dov > 0.f ? 2u : 0u);
                    dh = h - 2.f * (((osv & 1u) ? tt.a : 0.f) + ((osv & 2u) ? tt.b : 0.f));
                    if (nsv != osv || mode == MODE_FULL) vstate[j] = (uint8_t)nsv;
                }
                const unsigned am = __ballot_sync(FULL, h > 0.f);
                const unsigned dm = __ballot_sync(FULL, dh != 0.f);
                if (h > 0.f) s_al[warp][__popc(am & lt)] = make_float2(p, __int_as_float(4 * lane));
                if (dm) {
                    int slot0 = HB;
                    if (mode != MODE_FULL) {  // rows of the pool, in any order: the list gives the order of the sums
                        if (lane == 0) slot0 = min(atomicAdd(&s_pool, __popc(dm)), HB);
                        slot0 = __shfl_sync(FULL, slot0, 0);
                    }
                    if (dh != 0.f) {
                        const int r = __popc(dm & lt);
                        s_dj[warp][nd_w + r] = j;
                        s_dh[warp][nd_w + r] = dh;
                        s_ds[warp][nd_w + r] = (unsigned char)min(slot0 + r, HB);
                    }
                    nd_w += __popc(dm);
                    for (unsigned m = dm; m && slot0 < HB; m &= m - 1u, ++slot0) {
                        if (lane < KG)
                            *reinterpret_cast<float4*>(&A[slot0][4 * lane]) =
                                *reinterpret_cast<const float4*>(ring.group(lane) + 4 * (__ffs(m) - 1));
                    }
                }
                __syncwarp();
                add_rows(__popc(am), true);
                ring.release();
            }
            if (mode == MODE_EXT) continue;
            // the listed changes into the kept partial H: once, after the last tile,
            // unless a list could overflow before
            const bool end = i == rounds - 1;
            if (!end && (i < LIST / 32 - 1 || !__syncthreads_or(nd_w > LIST - 32))) continue;
            if (lane == 0) s_nd[warp] = nd_w;
            const bool any = __syncthreads_or(nd_w > 0) != 0;
            nd_w = 0;
            const bool rebuild = mode == MODE_FULL && !h_written;
            if (!any && !rebuild) continue;
            h_written = true;
            int n_d = 0;
#pragma unroll
            for (int w = 0; w < PW; ++w) n_d += s_nd[w];
            const bool pooled = mode != MODE_FULL && n_d <= HB;  // every row is in the pool
            for (int eb = tid / NV; eb - tid / NV < nb; eb += PT / NV) {  // (uniform count: barriers inside)
                const bool act = eb < nb;
                int rb = rb0, cb = cb0;
                if (act && eb >= PT / NV) block_of(eb, KB, rb, cb);
                rb *= 2;
                cb *= 2;
                // entries (rb, cb), (rb, cb + 1), (rb + 1, cb), (rb + 1, cb + 1): those of the
                // upper triangle, requested before the rows are summed
                const bool wr = act && vl == 0;
                float* keep = H_keep + (size_t)bid * HSTRIDE;
                const bool e0 = wr && cb < K, e1 = wr && cb + 1 < K, e2 = e0 && rb < cb, e3 = e1;
                const int i0 = tri_index(rb, cb, K), i1 = tri_index(rb, cb + 1, K);
                float old[4] = {0.f, 0.f, 0.f, 0.f};
                if (!rebuild) {
                    if (e0) old[0] = keep[i0];
                    if (e1) old[1] = keep[i1];
                    if (e2) old[2] = keep[i0 + 1];
                    if (e3) old[3] = keep[i1 + 1];
                }
                float hs[4] = {0.f, 0.f, 0.f, 0.f};
                for (int r0 = 0; r0 < n_d; r0 += HB) {
                    const int n = min(HB, n_d - r0);
                    if (eb - tid / NV == 0 || n_d > HB) {  // the rows in hand: their change of h, their place in A
                        __syncthreads();  // the rows before are summed
                        if (tid < n || !pooled) {
                            const int r = tid & (HB - 1);
                            int w = 0, x = r0 + r;
                            if (r < n) {
                                while (x >= s_nd[w]) x -= s_nd[w++];
                                if (tid < HB) {
                                    s_ch[r] = s_dh[w][x];
                                    s_row[r] = pooled ? (int)s_ds[w][x] : r;
                                }
                                if (!pooled) {
                                    const float4* row = reinterpret_cast<const float4*>(slab) + s_dj[w][x];
                                    for (int g = tid / HB; g < KG; g += PT / HB)
                                        *reinterpret_cast<float4*>(&A[r][4 * g]) = __ldg(row + (size_t)g * ld);
                                }
                            }
                        }
                        __syncthreads();
                    }
                    if (act)
                        for (int r = vl; r < n; r += NV) {
                            const float* row = A[s_row[r]];
                            const float2 ra = *reinterpret_cast<const float2*>(row + rb);
                            const float2 rc = *reinterpret_cast<const float2*>(row + cb);
                            const float hv = s_ch[r];
                            const float a0 = ra.x * hv, a1 = ra.y * hv;
                            hs[0] = fmaf(a0, rc.x, hs[0]);
                            hs[1] = fmaf(a0, rc.y, hs[1]);
                            hs[2] = fmaf(a1, rc.x, hs[2]);
                            hs[3] = fmaf(a1, rc.y, hs[3]);
                        }
                }
                for (int o = NV / 2; o > 0; o >>= 1)
#pragma unroll
                    for (int q = 0; q < 4; ++q) hs[q] += __shfl_xor_sync(FULL, hs[q], o);
                auto put = [&](int idx, float v) {
                    keep[idx] = v;
                    H_part[(size_t)idx * GS + bid] = v;
                };
                if (e0) put(i0, old[0] + hs[0]);
                if (e1) put(i1, old[1] + hs[1]);
                if (e2) put(i0 + 1, old[2] + hs[2]);
                if (e3) put(i1 + 1, old[3] + hs[3]);
            }
            if (tid == 0) s_pool = 0;
            __syncthreads();  // the rows and lists are free
        }
        if (rounds == 0 && mode == MODE_FULL)  // a block without voxels: its part of H is 0
            for (int e = tid; e < K * (K + 1) / 2; e += PT) {
                H_keep[(size_t)bid * HSTRIDE + e] = 0.f;
                H_part[(size_t)e * GS + bid] = 0.f;
            }
        ++n_ev;
        // ---- the block's partials: F; g and its rounding scale (or the new
        // aperture's, and its column of H), the warps in order
        const float f0 = warp_sum_f32(mode == MODE_EXT ? gk : facc);
        if (lane == 0) s_red[0][warp] = f0;
        if (mode == MODE_EXT) {
            const float f1 = warp_sum_f32(gnk);
            if (lane == 0) s_red[1][warp] = f1;
        }
        for (int o = LP; o < 32; o <<= 1) {
            ga.x += __shfl_xor_sync(FULL, ga.x, o);
            ga.y += __shfl_xor_sync(FULL, ga.y, o);
            ga.z += __shfl_xor_sync(FULL, ga.z, o);
            ga.w += __shfl_xor_sync(FULL, ga.w, o);
            gna.x += __shfl_xor_sync(FULL, gna.x, o);
            gna.y += __shfl_xor_sync(FULL, gna.y, o);
            gna.z += __shfl_xor_sync(FULL, gna.z, o);
            gna.w += __shfl_xor_sync(FULL, gna.w, o);
        }
        if (lane < KG) {  // (lanes below LP)
            *reinterpret_cast<float4*>(&s_g[warp][4 * lane]) = ga;
            *reinterpret_cast<float4*>(&s_gn[warp][4 * lane]) = gna;
        }
        __syncthreads();
        if (tid < 2 * KMAX) {  // g (or the new column of H), gn
            const int k = tid & (KMAX - 1), a = tid / KMAX;
            if (k < K) {
                float x = 0.f;
#pragma unroll
                for (int w = 0; w < PW; ++w) x += a ? s_gn[w][k] : s_g[w][k];
                if (mode == MODE_EXT) {
                    if (a == 0) {
                        H_keep[(size_t)bid * HSTRIDE + tri_index(k, K - 1, K)] = x;
                        H_part[(size_t)tri_index(k, K - 1, K) * GS + bid] = x;
                    }
                } else if (a == 0) {
                    g_part[(size_t)k * GS + bid] = (double)x;
                } else {
                    gn_part[(size_t)k * GS + bid] = x;
                }
            }
        } else if (warp == PW - 1) {  // F in FP64 (or the new aperture's g and gn) over the warps
            if (mode == MODE_EXT) {
                float x = lane < PW ? s_red[0][lane] : 0.f, y = lane < PW ? s_red[1][lane] : 0.f;
                x = warp_sum_f32(x);
                y = warp_sum_f32(y);
                if (lane == 0) {
                    g_part[(size_t)(K - 1) * GS + bid] = (double)x;
                    gn_part[(size_t)(K - 1) * GS + bid] = y;
                }
            } else {
                double x = lane < PW ? (double)s_red[0][lane] : 0.0;
#pragma unroll
                for (int o = PW / 2; o > 0; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
                if (lane == 0) F_part[bid] = x;
            }
        }
        if (!grid_sync(gb, G, s_target, s_flag)) {
            broken = true;
            break;
        }
        // ---- B. reduction by every block
        const unsigned tag = tag0 + (unsigned)n_ev;
        master_reduce_words(H_part, g_part, gn_part, F_part, GS, G, K, st, bid, mode == MODE_EXT, tag);
        // ---- C. the step, by every block on its own copy of the state.  Every
        // word of this evaluation is waited for (EXT: those of variable K - 1; the
        // others are the last evaluation's).
        if (tid < STEP_T) {
            const int v = tid & (KMAX - 1);
            unsigned long long w[KMAX * KMAX / STEP_T], x[5];
            auto waits = [&](int r) { return r < K && v <= r && (mode != MODE_EXT || r == K - 1); };
            // on many blocks first one of the words that take longest, polled by one warp
            int tries = 0;
            auto again = [&]() {
                if (++tries < GRID_WAIT_LIMIT && ((tries & 4095) || !ld_acquire_gpu(&gb->broken))) return true;
                s_lost = 1;
                return false;
            };
            if (G > DIRECT_BLOCKS) {
                if (warp == 0) {
                    const unsigned long long* probe = mode == MODE_EXT ? &st->wg[2 * K - 1] : &st->wF[1];
                    while ((unsigned)(word_get(probe) >> 32) != tag && again()) {
                    }
                }
                step_sync();
            }
            for (bool ok = false; !ok;) {
                ok = true;
#pragma unroll
                for (int m = 0; m < KMAX * KMAX / STEP_T; ++m) {
                    const int r = 4 * m + (tid >> 6);
                    if (r < K && v <= r) w[m] = word_get(&st->wH[r * KMAX + v]);
                }
                if (v < K) {
                    x[0] = word_get(&st->wg[2 * v]);
                    x[1] = word_get(&st->wg[2 * v + 1]);
                    x[2] = word_get(&st->wgn[v]);
                }
                x[3] = word_get(&st->wF[0]);
                x[4] = word_get(&st->wF[1]);
#pragma unroll
                for (int m = 0; m < KMAX * KMAX / STEP_T; ++m)
                    if (waits(4 * m + (tid >> 6))) ok = ok && (unsigned)(w[m] >> 32) == tag;
                if (v < K && (mode != MODE_EXT || v == K - 1))
                    ok = ok && (unsigned)(x[0] >> 32) == tag && (unsigned)(x[1] >> 32) == tag &&
                         (unsigned)(x[2] >> 32) == tag;
                if (mode != MODE_EXT) ok = ok && (unsigned)(x[3] >> 32) == tag && (unsigned)(x[4] >> 32) == tag;
                if (!ok && !again()) break;
            }
#pragma unroll
            for (int m = 0; m < KMAX * KMAX / STEP_T; ++m) {
                const int r = 4 * m + (tid >> 6);
                if (r < K && v <= r) sm.H[r][v] = __uint_as_float((unsigned)w[m]);
            }
            step_sync();
            if (!s_lost)
                master_step_body<true>(&ss, K, words_f64(x[3], x[4]), v < K ? words_f64(x[0], x[1]) : 0.0,
                                       v < K ? __uint_as_float((unsigned)x[2]) : 0.f, max_iter, tol_rel, sigma, sm);
        }
        __syncthreads();
        if (s_lost) {
            if (tid == 0) atomicExch(&gb->broken, 1u);
            broken = true;
            break;
        }
        if (ss.done) break;
    }
    copies_wait<0>();  // no copy outlives the launch
    if (broken) {      // a wait ran out: the host reports it
        if (tid == 0) {
            st->err = 2;
            if (bid == 0) {
                st->inc_G = 0;
                st->epoch = tag0 + (unsigned)n_ev + 1u;
            }
        }
        return;
    }
    if (bid == 0) {  // the solver state, and the round's record
        if (tid < K) {
            st->y[tid] = ss.y[tid];
            st->yt[tid] = ss.yt[tid];
            st->d[tid] = ss.d[tid];
            st->g[tid] = ss.g[tid];
        }
        if (tid == 0) {
            st->F = ss.F;
            st->alpha = ss.alpha;
            st->tol = ss.tol;
            st->res = ss.res;
            st->iter = ss.iter;
            st->phase = ss.phase;
            st->status = ss.status;
            st->n_eval = ss.n_eval;
            st->ticket = 0;
            st->final_pending = ss.final_pending;
            st->epoch = tag0 + (unsigned)n_ev;
            // the kept partial H, the voxel states, z, pi and the reduced sums are
            // those of the last evaluation: of the accepted point, or not kept
            st->inc_G = ss.final_pending ? 0 : G;
            st->inc_K = K;
            st->done = 1;
            if (cg != nullptr) {
                cg->trace[K - 1] = ss.F;
                cg->res[K - 1] = ss.res;
                cg->tol[K - 1] = ss.tol;
                cg->evals[K - 1] = ss.n_eval;
                cg->status[K - 1] = ss.status;
            }
        }
    }
    // the solve stopped at an accepted point other than the last one evaluated:
    // z and pi of that point
    if (ss.final_pending) {
        if (tid < KMAX) {
            const double yv = tid < K ? ss.y[tid] : 0.0;
            const float hi = (float)yv;
            s_y[tid] = make_float2(hi, (float)(yv - (double)hi));
        }
        __syncthreads();
        for (int t = bid + G * warp; t < n32; t += PW * G) {
            const int j = t * 32 + lane;
            float s, c;
            voxel_dot(KP, y4, s, c, [&](int k) {  // the slab's columns are padded past V
                return __ldg(reinterpret_cast<const float4*>(slab) + (size_t)(k >> 2) * ld + j);
            });
            if (j < V) {
                const StructTermsF tt = S >= 0 ? s_tf[vstruct[j]] : voxel_terms(tf, j);
                const float u = fmaxf((tt.tu - s) - c, 0.f), o = fmaxf((s - tt.to) + c, 0.f);
                z_out[j] = s + c;
                pi_out[j] = 2.f * (tt.b * o - tt.a * u);
            }
        }
    }
}


template <bool BATCH>
__global__ void __launch_bounds__(PT, 1) k_master_persist(const __grid_constant__ MasterTask t1,
                                                          const MasterTask* __restrict__ tasks, int GB, int K,
                                                          double sigma) {
    const MasterTask& t = BATCH ? tasks[blockIdx.x / GB] : t1;
    const int bid = BATCH ? (int)(blockIdx.x % GB) : (int)blockIdx.x;
    extern __shared__ __align__(128) float ring_mem[];
    __shared__ int s_flag, s_stop0;
    __shared__ unsigned s_target;
    const int* skip = t.skip;
    if (skip != nullptr && *skip) return;  // the same for every block
    if (K <= 0) K = __ldcg(&t.cg->K);      // pool size from the device (one graph for every round)
    const int G = BATCH ? GB : (int)gridDim.x;
    if (threadIdx.x == 0) {  // barrier base; a solve whose barrier broke runs no further master solve
        const unsigned c = *reinterpret_cast<volatile unsigned*>(&t.gb->count);
        s_target = c - c % (unsigned)G;
        s_stop0 = *reinterpret_cast<volatile unsigned*>(&t.gb->broken) != 0;
    }
    __syncthreads();
    if (s_stop0) return;
    master_solve_group(t.slab, t.ld, t.V, t.GS, t.S, t.max_iter, t.st, t.gb, t.H_part, t.g_part, t.gn_part, t.F_part,
                       t.vstruct, t.tf, t.tol_rel, t.z_out, t.pi_out, t.cg, t.vstate, t.H_keep, t.nonneg != 0, bid, G, K, sigma,
                       ring_mem, &s_target, &s_flag);
}

}  // namespace

__host__ __device__ int master_kw(int K) {
    const int KP = (K + 3) / 4 * 4;
    int kw = KP < 4 ? 4 : KP;
    if (((kw / 4) & 1) == 0) kw += 4;  // odd float4 count per row: conflict-free row-per-thread loads
    return kw;
}

size_t master_eval_smem(int K) {
    const int KP = (K + 3) / 4 * 4;
    return (size_t)TILE * (KP > 0 ? KP : 4) * sizeof(float);
}

size_t master_hess_smem(int K, int n_tiles) {
    return (size_t)((n_tiles + 1 + 3) / 4 * 4) * sizeof(int) + (size_t)CH * master_kw(K) * sizeof(float) +
           2 * CH * sizeof(float);
}

// Row lanes per 2x2 block of H in the persistent solve: the most (a power of
// two, within a warp) for which every block of the triangle has its lanes among
// the threads.
__host__ __device__ int persist_lanes(int K) {
    const int KB = (K + 3) / 4 * 2;
    const int nb = KB * (KB + 1) / 2;
    int nv = 1;
    while (nb > 0 && nv < 32 && nv * 2 * nb <= PT) nv *= 2;
    return nv;
}

__host__ __device__ int master_lanes(int K) {
    const int KP = (K + 3) / 4 * 4;
    const int KB = KP / 4;
    const int nb = KB * (KB + 1) / 2;
    int nv = 1;
    while (nb > 0 && nv * 2 * nb <= 256) nv *= 2;
    return nv;
}

// Blocks of the evaluation kernel for pool size K: all resident at once.
int master_grid(int V, int num_sms, int K) {
    const int n_tiles = (V + TILE - 1) / TILE;
    int occ = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_master_eval, TILE, master_eval_smem(K)) != cudaSuccess ||
        occ < 1) {
        cudaGetLastError();
        occ = 1;
    }
    const int gmax = num_sms * (occ < 4 ? occ : 4);
    return n_tiles < gmax ? (n_tiles > 0 ? n_tiles : 1) : gmax;
}

int master_grid_max(int num_sms) { return 4 * num_sms; }

int master_hess_grid(int num_sms) { return 2 * num_sms; }

// Diagnostic of the bounded barrier wait: a cooperative launch of `blocks`
// blocks meets at grid_sync, except block `absent`, which leaves without
// arriving.  The others must give up after GRID_WAIT_LIMIT polls, mark the
// barrier broken and report (out[0] = blocks that gave up, out[1] = blocks
// that passed).  Nothing faults and every wait ends.
__global__ void k_barrier_check(GridBar* gb, int absent, int* out) {
    __shared__ unsigned s_target;
    __shared__ int s_flag;
    if (threadIdx.x == 0) s_target = 0;
    if ((int)blockIdx.x == absent) return;  // the whole block leaves: it never arrives
    const bool ok = grid_sync(gb, gridDim.x, &s_target, &s_flag);
    if (threadIdx.x == 0) atomicAdd(&out[ok ? 1 : 0], 1);
}

cudaError_t launch_barrier_check(GridBar* gb, int blocks, int absent, int* out, cudaStream_t stream) {
    void* args[] = {(void*)&gb, (void*)&absent, (void*)&out};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(32);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, (const void*)k_barrier_check, args);
}

cudaError_t master_configure() {
    cudaError_t e = cudaFuncSetAttribute(k_master_eval, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)master_eval_smem(KMAX));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_master_persist<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RING_BYTES);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_master_persist<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RING_BYTES);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_master_hess, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
}

cudaError_t launch_master_init(MasterDev* st, int K, const int* skip, cudaGraphConditionalHandle cond,
                               int use_cond, cudaStream_t stream, int* launches, GridBar* gb) {
    k_master_init<<<1, KMAX, 0, stream>>>(st, K, skip, cond, use_cond, gb);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_master_eval(const MasterBuffers& mb, int V, int K, const uint8_t* vstruct, const StructTermsF* tf,
                               int S, float* z_out, float* pi_out, int mode, const int* skip, cudaStream_t stream,
                               int* launches) {
    const int KP = (K + 3) / 4 * 4;
    k_master_eval<<<mb.grid[K], TILE, master_eval_smem(K), stream>>>(
        mb.tmap[KP / 4], V, K, KP, mb.st, mb.act_rows, mb.act_hp, mb.act_count, mb.F_part, vstruct, tf, S, z_out,
        pi_out, mode, skip);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_master_hess(const MasterBuffers& mb, int K, int mode, cudaStream_t stream, int* launches) {
    k_master_hess<<<mb.GH, 256, master_hess_smem(K, mb.n_tiles), stream>>>(
        mb.act_rows, mb.act_hp, mb.act_count, mb.n_tiles, K, master_kw(K), master_lanes(K), mb.st, mb.H_part,
        mb.g_part, mb.gn_part, mb.GH, mode);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_master_step(int K, const MasterBuffers& mb, int max_iter, double tol_rel,
                               cudaGraphConditionalHandle cond, int use_cond, cudaStream_t stream, int* launches) {
    const int outs = K * (K + 1) / 2 + 2 * K + 1;
    k_master_reduce_step<<<(outs + STEP_T / 32 - 1) / (STEP_T / 32), STEP_T, 0, stream>>>(
        mb.H_part, mb.g_part, mb.gn_part, mb.F_part, mb.GH, mb.grid[K], mb.st, max_iter, tol_rel, 1e-4, cond,
        use_cond);
    ++*launches;
    return cudaGetLastError();
}

// Co-resident blocks of the persistent solve: one per SM, and no more than give
// every warp a tile of 32 voxels (fewer blocks have fewer partials to reduce
// and arrivals to wait for); 0 when a cooperative launch is not possible.
// want > 0: that many blocks, at most one per SM.
int master_persist_grid(int V, int num_sms, int want) {
    int dev = 0, coop = 0, occ = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_master_persist<false>, PT, RING_BYTES) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (occ < 1) return 0;
    const int need = (V + 32 * PW - 1) / (32 * PW);
    return std::min(num_sms, want > 0 ? want : std::max(need, 1));
}

cudaError_t launch_master_persist(const MasterBuffers& mb, const float* slab, int ld, int V, int K,
                                  const uint8_t* vstruct, const StructTermsF* tf, int S, int max_iter, double tol_rel,
                                  const int* skip, float* z_out, float* pi_out, CGDev* cg, cudaStream_t stream,
                                  int* launches) {
    const int G = mb.GP;
    if (G < 1) return cudaErrorInvalidConfiguration;
    if (K <= 0 && cg == nullptr) return cudaErrorInvalidValue;
    MasterTask t{};
    t.vstate = mb.vstate;
    t.H_keep = mb.H_keep;
    t.slab = slab;
    t.ld = ld;
    t.V = V;
    t.GS = mb.GH;  // partial arrays: stride GH >= G
    t.S = S;
    t.max_iter = max_iter;
    t.st = mb.st;
    t.gb = mb.bar;
    t.H_part = mb.H_part;
    t.g_part = mb.g_part;
    t.gn_part = mb.gn_part;
    t.F_part = mb.F_part;
    t.vstruct = vstruct;
    t.tf = tf;
    t.tol_rel = tol_rel;
    t.skip = skip;
    t.z_out = z_out;
    t.pi_out = pi_out;
    t.cg = cg;
    t.nonneg = mb.nonneg;
    const MasterTask* none = nullptr;
    int GB = 0;
    double sigma = 1e-4;
    void* args[] = {(void*)&t, (void*)&none, (void*)&GB, (void*)&K, (void*)&sigma};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(G);
    cfg.blockDim = dim3(PT);
    cfg.dynamicSmemBytes = RING_BYTES;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelExC(&cfg, (const void*)k_master_persist<false>, args);
    ++*launches;
    return e;
}

int master_batch_group(int n_tasks, int num_sms) {
    // one co-resident block per SM shared out evenly; more plans than SMs (up to
    // two per SM) run one block each, in two launches
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_master_persist<true>, PT, RING_BYTES) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (occ < 1 || n_tasks < 1 || n_tasks > 2 * num_sms) return 0;
    return std::max(1, num_sms / n_tasks);
}

cudaError_t launch_master_persist_batch(const MasterTask* tasks, int n_tasks, int GB, int num_sms,
                                        cudaStream_t stream, int* launches) {
    if (n_tasks < 1 || GB < 1 || GB > num_sms) return cudaErrorInvalidConfiguration;
    int K = 0;  // each group reads its pool size from its plan's device state
    MasterTask none{};
    double sigma = 1e-4;
    const int most = num_sms / GB;  // plans of one launch: every block resident
    for (int t0 = 0; t0 < n_tasks; t0 += most) {
        const MasterTask* part = tasks + t0;
        void* args[] = {(void*)&none, (void*)&part, (void*)&GB, (void*)&K, (void*)&sigma};
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(std::min(most, n_tasks - t0) * GB);
        cfg.blockDim = dim3(PT);
        cfg.dynamicSmemBytes = RING_BYTES;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelExC(&cfg, (const void*)k_master_persist<true>, args);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    return cudaSuccess;
}

cudaError_t launch_cg_record(const MasterDev* st, CGDev* cg, int K, cudaStream_t stream, int* launches) {
    k_cg_record<<<1, 32, 0, stream>>>(st, cg, K);
    ++*launches;
    return cudaGetLastError();
}

}  // namespace dao
