// Device-side construction of a plan's matrices from the caller's CSR of D
// (uploaded as is): the checks of the caller's rows and labels, the padded
// row offsets (a scan), the padded voxel-major layout, the per-row beam segments,
// the per-beamlet scales of the 16-bit storage, and the beamlet-major
// transpose D^T by a stable counting sort.
//
// The transpose keeps every row of D^T in increasing voxel order, the order a
// sequential counting sort gives, without sorting: the voxel rows are cut into
// chunks; C[chunk][i] counts chunk's entries of beamlet i (shared-memory
// integer atomics, so the counts are exact); a scan over chunks turns the
// counts into each chunk's first slot in every row of D^T; then a block per
// chunk places its entries, each at its beamlet's first slot plus the number of
// the chunk's earlier rows that hold the beamlet, counted in a bitmap of rows.
//
// The passes over the entries are bound by latency, not by bytes, unless each
// warp keeps many loads in flight.  They therefore give a warp several consecutive
// rows whose entries it reads as one stretch, several per lane requested
// together, with each lane keeping track of the row that its entry is in.
#include <algorithm>
#include <climits>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "dao_internal.h"

namespace dao {

namespace {

constexpr unsigned FULL = 0xffffffffu;

template <int PREC>
__device__ __forceinline__ unsigned short to16(float r) {
    if (PREC == DAO_PREC_FP16) return __half_as_ushort(__float2half_rn(r));
    return __bfloat16_as_ushort(__float2bfloat16_rn(r));
}

// scale_i = s_i, or 1 for a beamlet without entries; dmax = max_i s_i.
__global__ void k_scale_fix(unsigned* __restrict__ smax, int N, unsigned* __restrict__ dmax) {
    __shared__ unsigned s_m[8];
    unsigned m = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        const unsigned b = smax[i];
        m = max(m, b);
        const float s = __uint_as_float(b);
        reinterpret_cast<float*>(smax)[i] = s > 0.f ? s : 1.f;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(FULL, m, o));
    if ((threadIdx.x & 31) == 0) s_m[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = max(t, s_m[w]);
        atomicMax(dmax, t);
    }
}

constexpr int RW_T = 256, RW_W = RW_T / 32;  // threads and warps of a block
constexpr int RW_ROWS = 8;                   // rows per warp: with 32 the warps of the longest rows end last
constexpr int RW_U = 4;                      // entries per lane requested together

// Padded voxel-major D (padding repeats the row's last column with value 0) and
// its beam segments: seg[b][j] = first padded position of row j with column >=
// beam_off[b], seg[B][j] = the end of row j's real entries.  A warp per RW_ROWS
// rows; the segments by a binary search per (row, beam) over columns that the warp
// has just read.  Prostate-shaped FP32 matrix (7.4 M entries, 9 beams): a warp per
// row, and a thread per row that walked it again for the segments, took 38 + 49 us;
// with a search for every entry's beam 59, bound by issue; now 31.
template <int PREC>
__global__ void __launch_bounds__(RW_T) k_fill_d(const int64_t* __restrict__ rp, const int* __restrict__ col,
                                                 const float* __restrict__ val, const int* __restrict__ prow, int V,
                                                 const float* __restrict__ scale, const int* __restrict__ beam_off,
                                                 int B, int* __restrict__ seg, int* __restrict__ dcol,
                                                 float* __restrict__ dval, unsigned short* __restrict__ dcol16,
                                                 unsigned short* __restrict__ dval16) {
    __shared__ int s_start[RW_W][RW_ROWS + 1], s_shift[RW_W][RW_ROWS + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t w = (int64_t)blockIdx.x * RW_W + warp;
    if (w * RW_ROWS >= V) return;
    const int j0 = (int)(w * RW_ROWS), j = min(j0 + min(lane, RW_ROWS), V);  // lane RW_ROWS: the end
    const bool own = lane < RW_ROWS && j < V;
    const int64_t p0 = rp[j], s0 = __shfl_sync(FULL, p0, 0);
    const int len = own ? (int)(rp[j + 1] - p0) : 0;
    const int q0 = prow[j], pl = own ? prow[j + 1] - q0 : 0;
    if (lane <= RW_ROWS) {
        s_start[warp][lane] = (int)(p0 - s0);
        s_shift[warp][lane] = q0 - (int)(p0 - s0);
    }
    __syncwarp();
    auto put = [&](int q, int c, float v) {
        if (PREC == DAO_PREC_FP32) {
            dcol[q] = c;
            dval[q] = v;
        } else {
            dcol16[q] = (unsigned short)c;
            dval16[q] = to16<PREC>(v / scale[c]);
        }
    };
    const int n = s_start[warp][RW_ROWS];
    int r = 0;  // the row of the lane's entry
    for (int t0 = 0; t0 < n; t0 += 32 * RW_U) {
        int c[RW_U];
        float v[RW_U];
#pragma unroll
        for (int u = 0; u < RW_U; ++u) {
            const int t = t0 + 32 * u + lane;
            c[u] = t < n ? col[s0 + t] : 0;
            v[u] = t < n ? val[s0 + t] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < RW_U; ++u) {
            const int t = t0 + 32 * u + lane;
            if (t < n) {
                while (t >= s_start[warp][r + 1]) ++r;
                put(s_shift[warp][r] + t, c[u], v[u]);
            }
        }
    }
    if (own) {
        const int last = len > 0 ? col[p0 + len - 1] : 0;
        for (int t = len; t < pl; ++t) put(q0 + t, last, 0.f);
    }
    for (int i = lane; i < RW_ROWS * (B + 1); i += 32) {
        const int rr = i % RW_ROWS, b = i / RW_ROWS;
        if (j0 + rr >= V) continue;
        const int a = s_start[warp][rr];
        int lo = a, hi = s_start[warp][rr + 1];
        if (b == B) {
            lo = hi;
        } else {
            const int first = beam_off[b];
            while (lo < hi) {
                const int m = (lo + hi) >> 1;
                if (col[s0 + m] < first)
                    lo = m + 1;
                else
                    hi = m;
            }
        }
        seg[(size_t)b * V + j0 + rr] = s_shift[warp][rr] + lo;
    }
}

// Beamlet counters of one block live in shared memory for a tile of TILE_N
// beamlets; a matrix with more beamlets runs a grid of (chunk, tile) blocks.
constexpr int TILE_N = 12288;
constexpr int STATS_T = 512, STATS_U = 8;

// Per (chunk, beamlet tile): C[chunk][i] = the chunk's entries of beamlet i,
// counted in shared memory, and s_i = max |D_ij| over them folded into smax
// (bits of a non-negative float, ordered like the floats).  Both maxima only grow,
// so a value that is not above the one read needs no atomic.  STATS_U entries per
// thread in flight: 65 us with one on a prostate-shaped FP32 matrix, now 24.
__global__ void __launch_bounds__(STATS_T) k_chunk_stats(const int64_t* __restrict__ rp, const int* __restrict__ col,
                                                         const float* __restrict__ val, int V, int CH, int N,
                                                         int* __restrict__ C, unsigned* __restrict__ smax) {
    extern __shared__ unsigned s_stats[];
    const int ch = blockIdx.x, i0 = blockIdx.y * TILE_N;
    const int nt = min(TILE_N, N - i0);
    unsigned* s_cnt = s_stats;
    unsigned* s_mx = s_stats + nt;
    for (int t = threadIdx.x; t < 2 * nt; t += STATS_T) s_stats[t] = 0u;
    __syncthreads();
    const int64_t p0 = rp[(int64_t)ch * CH], p1 = rp[min((int64_t)V, (int64_t)(ch + 1) * CH)];
    for (int64_t q = p0; q < p1; q += STATS_T * STATS_U) {
        int c[STATS_U];
        float v[STATS_U];
#pragma unroll
        for (int u = 0; u < STATS_U; ++u) {
            const int64_t p = q + u * STATS_T + threadIdx.x;
            c[u] = p < p1 ? col[p] - i0 : -1;
            v[u] = p < p1 ? val[p] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < STATS_U; ++u)
            if (c[u] >= 0 && c[u] < nt) {
                const unsigned m = __float_as_uint(fabsf(v[u]));
                atomicAdd(&s_cnt[c[u]], 1u);
                if (m > *(volatile unsigned*)&s_mx[c[u]]) atomicMax(&s_mx[c[u]], m);
            }
    }
    __syncthreads();
    int* Cc = C + (size_t)ch * N + i0;
    for (int t = threadIdx.x; t < nt; t += STATS_T) {
        const unsigned n = s_cnt[t];
        Cc[t] = (int)n;
        if (n && s_mx[t] > __ldcg(&smax[i0 + t])) atomicMax(&smax[i0 + t], s_mx[t]);
    }
}

// Column i of C becomes each chunk's first slot relative to the start of row
// i of D^T, and cnt[i] its total.  Block of 32 beamlets x 32 chunk segments:
// segment sums, a scan over the segments in shared memory, then each segment
// rewritten from its offset.
__global__ void __launch_bounds__(1024) k_chunk_scan(int* __restrict__ C, int n_ch, int N, int* __restrict__ cnt) {
    __shared__ int s_sum[32][33];
    const int x = threadIdx.x, y = threadIdx.y;
    const int i = blockIdx.x * 32 + x;
    const int per = (n_ch + 31) / 32;
    const int c0 = min(n_ch, y * per), c1 = min(n_ch, c0 + per);
    int sum = 0;
    if (i < N)
        for (int ch = c0; ch < c1; ++ch) sum += C[(size_t)ch * N + i];
    s_sum[y][x] = sum;
    __syncthreads();
    int run = 0;
    for (int t = 0; t < y; ++t) run += s_sum[t][x];
    if (i < N) {
        if (y == 31) cnt[i] = run + sum;
        for (int ch = c0; ch < c1; ++ch) {
            const int v = C[(size_t)ch * N + i];
            C[(size_t)ch * N + i] = run;
            run += v;
        }
    }
}

// Placement: a block per (chunk, beamlet tile of width tw) takes PL_ROWS voxel rows
// at a time: a bitmap of the rows that hold each beamlet (PL_ROWS bits in words of
// 32 rows, word-major so that consecutive beamlets lie in consecutive banks), then
// each entry at its beamlet's next slot plus the bits below its row, which is the
// order of a walk in CSR order without the walk.  Equal stretches of entries per warp,
// PL_U entries per lane requested together; the second reading of the columns
// comes from cache.  A warp per (chunk, narrower tile) that walked the rows one
// after another took 198 us on a prostate-shaped FP32 matrix (7.4 M entries, 3600
// beamlets); now 128, bound by the scattered 4-byte writes.
constexpr int PL_T = 1024, PL_ROWS = 256, PL_WORDS = PL_ROWS / 32, PL_U = 8;
constexpr int PL_TILE = 6000;  // beamlets per tile: 36 bytes of shared memory each

size_t place_smem(int tw) { return sizeof(int) * (size_t)tw * (PL_WORDS + 1); }

__global__ void __launch_bounds__(PL_T) k_chunk_place(const int64_t* __restrict__ rp, const int* __restrict__ col,
                                                      const float* __restrict__ val, int V, int CH, int N, int tw,
                                                      const int* __restrict__ C, const int* __restrict__ trow,
                                                      int* __restrict__ tcol, float* __restrict__ tval) {
    extern __shared__ int s_pl[];
    __shared__ int s_row[PL_ROWS + 1];  // row starts, relative to the window's first entry
    const int ch = blockIdx.x, i0 = blockIdx.y * tw;
    const int nt = min(tw, N - i0);
    int* s_slot = s_pl;                                          // next slots
    unsigned* s_bits = reinterpret_cast<unsigned*>(s_pl) + tw;   // PL_WORDS x tw
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int t = tid; t < nt; t += PL_T) s_slot[t] = trow[i0 + t] + C[(size_t)ch * N + i0 + t];
    const int j0 = ch * CH, j1 = (int)min((int64_t)V, (int64_t)j0 + CH);
    for (int w0 = j0; w0 < j1; w0 += PL_ROWS) {
        const int nr = min(PL_ROWS, j1 - w0);
        const int64_t e0 = rp[w0];
        for (int r = tid; r <= nr; r += PL_T) s_row[r] = (int)(rp[w0 + r] - e0);
        for (int t = tid; t < PL_WORDS * tw / 4; t += PL_T) reinterpret_cast<uint4*>(s_bits)[t] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        // an equal stretch of the entries per warp
        const int per = (s_row[nr] + PL_T / 32 - 1) / (PL_T / 32);
        const int tb = min(warp * per, s_row[nr]), te = min(tb + per, s_row[nr]);
        int r0 = 0;  // the row of entry tb: the last that starts at or before it
        for (int lo = 0, hi = nr; hi - lo > 1;) {
            const int m = (lo + hi) >> 1;
            if (s_row[m] <= tb)
                lo = m;
            else
                hi = m;
            r0 = lo;
        }
        int r = r0;
        for (int t0 = tb; t0 < te; t0 += 32 * PL_U) {
            int c[PL_U];
#pragma unroll
            for (int u = 0; u < PL_U; ++u) {
                const int t = t0 + 32 * u + lane;
                c[u] = t < te ? col[e0 + t] - i0 : -1;
            }
#pragma unroll
            for (int u = 0; u < PL_U; ++u) {
                const int t = t0 + 32 * u + lane;
                if (c[u] >= 0 && c[u] < nt) {
                    while (t >= s_row[r + 1]) ++r;
                    atomicOr(&s_bits[(r >> 5) * tw + c[u]], 1u << (r & 31));
                }
            }
        }
        __syncthreads();
        r = r0;
        for (int t0 = tb; t0 < te; t0 += 32 * PL_U) {
            int c[PL_U];
            float v[PL_U];
#pragma unroll
            for (int u = 0; u < PL_U; ++u) {
                const int t = t0 + 32 * u + lane;
                c[u] = t < te ? col[e0 + t] - i0 : -1;
                v[u] = t < te ? val[e0 + t] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < PL_U; ++u) {
                const int t = t0 + 32 * u + lane;
                if (c[u] >= 0 && c[u] < nt) {
                    while (t >= s_row[r + 1]) ++r;
                    const int rw = r >> 5;
                    int pos = s_slot[c[u]] + __popc(s_bits[rw * tw + c[u]] & ((1u << (r & 31)) - 1u));
                    for (int q = 0; q < rw; ++q) pos += __popc(s_bits[q * tw + c[u]]);
                    tcol[pos] = w0 + r;
                    tval[pos] = v[u];
                }
            }
        }
        if (w0 + PL_ROWS < j1) {  // the next rows' first slots
            __syncthreads();
            for (int t = tid; t < nt; t += PL_T) {
                int n = 0;
                for (int q = 0; q < PL_WORDS; ++q) n += __popc(s_bits[q * tw + t]);
                s_slot[t] += n;
            }
            __syncthreads();
        }
    }
}

// Padding of the rows of D^T: the row's last voxel with value 0.
__global__ void k_pad_t(const int* __restrict__ trow, const int* __restrict__ cnt, int N, int* __restrict__ tcol,
                        float* __restrict__ tval) {
    const int lane = threadIdx.x & 31;
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= N) return;
    const int q0 = trow[i], real = cnt[i], q1 = trow[i + 1];
    const int last = real > 0 ? tcol[q0 + real - 1] : 0;
    for (int q = q0 + real + lane; q < q1; q += 32) {
        tcol[q] = last;
        tval[q] = 0.f;
    }
}

// 16-bit values of D^T, row i scaled by 1 / s_i.
template <int PREC>
__global__ void k_quant_t(const float* __restrict__ tval, const int* __restrict__ trow, int N,
                          const float* __restrict__ scale, unsigned short* __restrict__ tval16) {
    const int lane = threadIdx.x & 31;
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= N) return;
    const float s = scale[i];
    for (int q = trow[i] + lane; q < trow[i + 1]; q += 32) tval16[q] = to16<PREC>(tval[q] / s);
}

// The caller's CSR and labels: row bounds inside [0, nnz], columns in [0, N) and
// strictly increasing, finite values, label in [0, S).  A bad row or label is
// recorded as V - j under atomicMax (so the lowest index wins); a good row writes
// its padded length, a good label its byte and one count for its structure.  Every
// read of col / val is inside checked bounds.
//
// A warp per RW_ROWS rows: where all their bounds hold, the rows' entries are one
// stretch, and the columns increase strictly inside every row exactly when the
// stretch has no more places that do not increase than there are among the rows'
// starts.  Only where that, a column or a value fails are the rows looked at one by
// one.  Prostate-shaped matrix (7.4 M entries): 50 us with a warp per row, now 23.
__global__ void __launch_bounds__(RW_T) k_check(const int64_t* __restrict__ rp, const int* __restrict__ col,
                                                const float* __restrict__ val, int64_t nnz, int V, int N,
                                                const int* __restrict__ label, int S, int pad,
                                                int64_t* __restrict__ plen, uint8_t* __restrict__ vs8,
                                                BuildCheck* __restrict__ chk) {
    __shared__ int s_cnt[SMAX];
    for (int k = threadIdx.x; k < SMAX; k += blockDim.x) s_cnt[k] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t w = (int64_t)blockIdx.x * RW_W + (threadIdx.x >> 5);
    if (w * RW_ROWS < V) {
        const int j0 = (int)(w * RW_ROWS), j = min(j0 + min(lane, RW_ROWS), V);  // lane RW_ROWS: the end
        const bool own = lane < RW_ROWS && j < V;
        const int64_t p0 = rp[j], p1 = own ? rp[j + 1] : p0;
        const bool bounds = !own || (p0 >= 0 && p1 >= p0 && p1 <= nnz);
        bool ok = bounds, neg = false;
        if (__all_sync(FULL, bounds)) {
            const int64_t s0 = __shfl_sync(FULL, p0, 0), e0 = __shfl_sync(FULL, p0, RW_ROWS);
            const bool down = p1 > p0 && p0 > s0 && col[p0] <= col[p0 - 1];
            int extra = 0, carry = INT_MIN;
            bool bad = false;
            for (int64_t q = s0; q < e0; q += 32 * RW_U) {
                int c[RW_U];
                float v[RW_U];
#pragma unroll
                for (int u = 0; u < RW_U; ++u) {
                    const int64_t p = q + 32 * u + lane;
                    c[u] = p < e0 ? col[p] : 0;
                    v[u] = p < e0 ? val[p] : 0.f;
                }
#pragma unroll
                for (int u = 0; u < RW_U; ++u) {
                    int prev = __shfl_up_sync(FULL, c[u], 1);
                    if (lane == 0) prev = carry;
                    carry = __shfl_sync(FULL, c[u], 31);
                    if (q + 32 * u + lane < e0) {
                        bad |= c[u] < 0 || c[u] >= N || !isfinite(v[u]);
                        neg |= v[u] < 0.f;
                        extra += c[u] <= prev;
                    }
                }
            }
            extra = (int)__reduce_add_sync(FULL, (unsigned)extra) - __popc(__ballot_sync(FULL, down));
            ok = extra == 0 && !__any_sync(FULL, bad);
        } else {
            ok = false;
        }
        if (!__all_sync(FULL, ok)) {  // which rows
            for (int r = 0; r < RW_ROWS; ++r) {
                const int64_t a = __shfl_sync(FULL, p0, r), b = __shfl_sync(FULL, p1, r);
                bool good = __shfl_sync(FULL, (int)bounds, r) != 0;
                if (good) {
                    bool bad = false;
                    for (int64_t p = a + lane; p < b; p += 32) {
                        const int c = col[p];
                        const float v = val[p];
                        bad |= c < 0 || c >= N || !isfinite(v);
                        if (p > a) bad |= c <= col[p - 1];
                    }
                    good = !__any_sync(FULL, bad);
                }
                if (lane == r) ok = good;
            }
        }
        if (__any_sync(FULL, neg) && lane == 0) chk->negative = 1;
        if (own) {
            plen[j] = ok ? (p1 - p0 + pad - 1) / pad * pad : 0;
            if (!ok) atomicMax(&chk->bad_row, V - j);
            const int l = label[j];
            if (l < 0 || l >= S) {
                atomicMax(&chk->bad_label, V - j);
            } else {
                vs8[j] = (uint8_t)l;
                atomicAdd(&s_cnt[l], 1);
            }
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < S; k += blockDim.x)
        if (s_cnt[k]) atomicAdd(&chk->count[k], s_cnt[k]);
}

// Exclusive scan of plen in three steps: block totals, a scan of the totals
// (one block), then each block's scan plus its offset.  SCAN_T threads with
// SCAN_E consecutive elements each per block.
constexpr int SCAN_T = 1024, SCAN_E = 4, SCAN_B = SCAN_T * SCAN_E;

// Exclusive scan of one value per thread across the block; returns the block total.
__device__ __forceinline__ int64_t block_exscan(int64_t v, int64_t* ex) {
    __shared__ int64_t s_w[SCAN_T / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int64_t t = lane < SCAN_T / 32 ? s_w[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(FULL, t, o);
            if (lane >= o) t += y;
        }
        if (lane < SCAN_T / 32) s_w[lane] = t;  // inclusive over warps
    }
    __syncthreads();
    const int64_t before = wid > 0 ? s_w[wid - 1] : 0;
    *ex = before + x - v;
    const int64_t total = s_w[SCAN_T / 32 - 1];
    __syncthreads();  // s_w reused by the next call
    return total;
}

__global__ void __launch_bounds__(SCAN_T) k_scan_totals(const int64_t* __restrict__ plen, int V,
                                                         int64_t* __restrict__ bsum) {
    const int64_t i0 = (int64_t)blockIdx.x * SCAN_B + (int64_t)threadIdx.x * SCAN_E;
    int64_t v = 0;
#pragma unroll
    for (int e = 0; e < SCAN_E; ++e)
        if (i0 + e < V) v += plen[i0 + e];
    int64_t ex;
    const int64_t t = block_exscan(v, &ex);
    if (threadIdx.x == 0) bsum[blockIdx.x] = t;
}

// One block: bsum becomes exclusive; the grand total goes to chk->padded and
// (clamped) to prow[V].
__global__ void __launch_bounds__(SCAN_T) k_scan_offsets(int64_t* __restrict__ bsum, int nb, int V,
                                                          int* __restrict__ prow, BuildCheck* __restrict__ chk) {
    int64_t carry = 0;
    for (int b0 = 0; b0 < nb; b0 += SCAN_T) {
        const int b = b0 + threadIdx.x;
        const int64_t v = b < nb ? bsum[b] : 0;
        int64_t ex;
        const int64_t t = block_exscan(v, &ex);
        if (b < nb) bsum[b] = carry + ex;
        carry += t;
    }
    if (threadIdx.x == 0) {
        chk->padded = carry;
        prow[V] = (int)min(carry, (int64_t)INT_MAX);
    }
}

__global__ void __launch_bounds__(SCAN_T) k_scan_apply(const int64_t* __restrict__ plen, int V,
                                                        const int64_t* __restrict__ bsum, int* __restrict__ prow) {
    const int64_t i0 = (int64_t)blockIdx.x * SCAN_B + (int64_t)threadIdx.x * SCAN_E;
    int64_t v[SCAN_E], tot = 0;
#pragma unroll
    for (int e = 0; e < SCAN_E; ++e) {
        v[e] = i0 + e < V ? plen[i0 + e] : 0;
        tot += v[e];
    }
    int64_t ex;
    block_exscan(tot, &ex);
    int64_t run = bsum[blockIdx.x] + ex;
#pragma unroll
    for (int e = 0; e < SCAN_E; ++e)
        if (i0 + e < V) {
            prow[i0 + e] = (int)min(run, (int64_t)INT_MAX);
            run += v[e];
        }
}

inline unsigned blocks_for(int64_t threads, int bs) { return (unsigned)((threads + bs - 1) / bs); }
inline unsigned row_warp_blocks(int V) { return blocks_for(((int64_t)V + RW_ROWS - 1) / RW_ROWS * 32, RW_T); }

}  // namespace

int check_scan_blocks(int V) { return (int)blocks_for(V, SCAN_B); }

cudaError_t build_check(const int64_t* rp, const int* col, const float* val, int64_t nnz, int V, int N,
                        const int* label, int S, int pad, int64_t* plen, int64_t* bsum, uint8_t* vs8, int* prow,
                        BuildCheck* chk, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(chk, 0, sizeof(BuildCheck), s);
    if (e != cudaSuccess) return e;
    k_check<<<row_warp_blocks(V), RW_T, 0, s>>>(rp, col, val, nnz, V, N, label, S, pad, plen, vs8, chk);
    const int nb = check_scan_blocks(V);
    k_scan_totals<<<nb, SCAN_T, 0, s>>>(plen, V, bsum);
    k_scan_offsets<<<1, SCAN_T, 0, s>>>(bsum, nb, V, prow, chk);
    k_scan_apply<<<nb, SCAN_T, 0, s>>>(plen, V, bsum, prow);
    return cudaGetLastError();
}

cudaError_t build_stats(const int64_t* rp, const int* col, const float* val, int V, int CH, int N, int n_ch,
                        int* C, int* cnt, unsigned* smax, unsigned* dmax, int num_sms, cudaStream_t s) {
    const int n_tile = (N + TILE_N - 1) / TILE_N;
    const size_t sm_stats = 2 * sizeof(unsigned) * (size_t)std::min(N, TILE_N);
    // the attribute is process-wide and plans may be created from several threads at
    // once: always the largest size any launch asks for, never this plan's own
    cudaError_t e = cudaFuncSetAttribute(k_chunk_stats, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(2 * sizeof(unsigned) * TILE_N));
    if (e == cudaSuccess) e = cudaMemsetAsync(smax, 0, sizeof(unsigned) * N, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(dmax, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    k_chunk_stats<<<dim3(n_ch, n_tile), STATS_T, sm_stats, s>>>(rp, col, val, V, CH, N, C, smax);
    k_chunk_scan<<<(N + 31) / 32, dim3(32, 32), 0, s>>>(C, n_ch, N, cnt);
    k_scale_fix<<<num_sms, 256, 0, s>>>(smax, N, dmax);
    return cudaGetLastError();
}

cudaError_t build_fill_d(int prec, const int64_t* rp, const int* col, const float* val, const int* prow, int V,
                         const float* scale, const int* beam_off, int B, int* seg, DevCSR& D, cudaStream_t s) {
    const unsigned g = row_warp_blocks(V);
    if (prec == DAO_PREC_FP32)
        k_fill_d<DAO_PREC_FP32><<<g, RW_T, 0, s>>>(rp, col, val, prow, V, scale, beam_off, B, seg, D.col, D.val,
                                                   nullptr, nullptr);
    else if (prec == DAO_PREC_FP16)
        k_fill_d<DAO_PREC_FP16><<<g, RW_T, 0, s>>>(rp, col, val, prow, V, scale, beam_off, B, seg, nullptr, nullptr,
                                                   D.col16, D.val16);
    else
        k_fill_d<DAO_PREC_BF16><<<g, RW_T, 0, s>>>(rp, col, val, prow, V, scale, beam_off, B, seg, nullptr, nullptr,
                                                   D.col16, D.val16);
    return cudaGetLastError();
}

namespace {
// One thread per unit of 32 rows: its group count, the largest into out[0];
// the largest row into out[1].
__global__ void k_unit_max(const int* __restrict__ prow, int V, int epg, int* __restrict__ out) {
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    const int r0 = u * 32;
    if (r0 >= V) return;
    const int r1 = min(r0 + 32, V);
    atomicMax(out, (prow[r1] - prow[r0]) / epg);
    int m = 0;
    for (int r = r0; r < r1; ++r) m = max(m, prow[r + 1] - prow[r]);
    atomicMax(out + 1, m / epg);
}

// One thread per split of the merge form: at diagonal d the largest i in
// [max(0, d - G), min(d, V)] whose row i - 1 ends within the first d - i groups
// (binary search: the condition holds up to that i and fails after it).
__global__ void k_merge_path(const int* __restrict__ prow, int V, int epg, int chunk, int n_warps,
                             int2* __restrict__ out) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v > n_warps) return;
    const long long G = prow[V] / epg;
    const long long d = min((long long)v * chunk, (long long)V + G);
    long long lo = max(0LL, d - G), hi = min(d, (long long)V);
    while (lo < hi) {
        const long long mid = (lo + hi + 1) >> 1;
        if ((long long)(prow[mid] / epg) <= d - mid)  // row mid - 1 ends within d - mid groups
            lo = mid;
        else
            hi = mid - 1;
    }
    out[v] = make_int2((int)lo, (int)(d - lo));
}
}  // namespace

namespace {
constexpr int BEAM_TILE = 1024;  // rows per tile of the beams' row-offset scan

// Inclusive sum over the block of one int per thread (BEAM_TILE threads);
// *total receives the block's sum.
__device__ __forceinline__ int block_scan_incl(int v, int* s_w, int* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) s_w[w] = v;
    __syncthreads();
    if (w == 0) {
        int x = s_w[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += u;
        }
        s_w[lane] = x;  // inclusive sums of the warps' totals
    }
    __syncthreads();
    const int r = v + (w > 0 ? s_w[w - 1] : 0);
    *total = s_w[BEAM_TILE / 32 - 1];
    __syncthreads();
    return r;
}

__device__ __forceinline__ int beam_seg_len(const int* __restrict__ seg, int V, int b, int j) {
    return j < V ? seg[(size_t)(b + 1) * V + j] - seg[(size_t)b * V + j] : 0;
}

// Per (tile, beam): the sum of the tile's segment lengths of the beam.
__global__ void __launch_bounds__(BEAM_TILE) k_beam_tiles(const int* __restrict__ seg, int V, int n_tiles,
                                                         int* __restrict__ tsum) {
    __shared__ int s_w[BEAM_TILE / 32];
    const int b = blockIdx.y, t = blockIdx.x;
    int total = 0;
    block_scan_incl(beam_seg_len(seg, V, b, t * BEAM_TILE + (int)threadIdx.x), s_w, &total);
    if (threadIdx.x == 0) tsum[(size_t)b * n_tiles + t] = total;
}

// Per beam: the tile sums turned into the tiles' first offsets (in place),
// the beam's total into brp[b][V].
__global__ void __launch_bounds__(BEAM_TILE) k_beam_tile_scan(int* __restrict__ tsum, int n_tiles, int V,
                                                             int* __restrict__ brp) {
    __shared__ int s_w[BEAM_TILE / 32];
    const int b = blockIdx.x;
    int carry = 0;
    for (int c0 = 0; c0 < n_tiles; c0 += BEAM_TILE) {
        const int i = c0 + (int)threadIdx.x;
        const int v = i < n_tiles ? tsum[(size_t)b * n_tiles + i] : 0;
        int total = 0;
        const int incl = block_scan_incl(v, s_w, &total);
        if (i < n_tiles) tsum[(size_t)b * n_tiles + i] = carry + incl - v;
        carry += total;
    }
    if (threadIdx.x == 0) brp[(size_t)b * (V + 1) + V] = carry;
}

// Per (tile, beam): the row offsets of the tile's rows, counted from the
// beam's first entry; beam b's entries follow those of beams 0 .. b - 1 (the
// totals brp[b'][V]).
__global__ void __launch_bounds__(BEAM_TILE) k_beam_offsets(const int* __restrict__ seg, int V, int n_tiles,
                                                           const int* __restrict__ toff, int* __restrict__ brp) {
    __shared__ int s_w[BEAM_TILE / 32];
    const int b = blockIdx.y, t = blockIdx.x;
    const int j = t * BEAM_TILE + (int)threadIdx.x;
    const int len = beam_seg_len(seg, V, b, j);
    int total = 0;
    const int incl = block_scan_incl(len, s_w, &total);
    if (j < V) brp[(size_t)b * (V + 1) + j] = toff[(size_t)b * n_tiles + t] + incl - len;
}

// D by beams: the rows' segments of each beam one after the other, with the beamlet
// index local to the beam.  A warp per 32 rows of one beam, whose entries are one
// stretch of the beam's range.  A thread per (beam, row) that copied its segment
// took 84 us on a prostate-shaped FP32 matrix (7.4 M entries, 9 beams); now 30.
template <int PREC>
__global__ void __launch_bounds__(RW_T) k_beam_fill(const int* __restrict__ seg, int V,
                                                    const int* __restrict__ beam_off,
                                                    const int* __restrict__ brp, const int* __restrict__ col,
                                                    const float* __restrict__ val,
                                                    const unsigned short* __restrict__ col16,
                                                    const unsigned short* __restrict__ val16,
                                                    unsigned short* __restrict__ bcol, float* __restrict__ bval32,
                                                    unsigned short* __restrict__ bval16) {
    __shared__ int s_start[RW_W][33], s_src[RW_W][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = blockIdx.y;
    const int j = (int)min((int64_t)V, ((int64_t)blockIdx.x * RW_W + warp) * 32 + lane);
    if (__shfl_sync(FULL, j, 0) >= V) return;  // uniform
    const int* bp = brp + (size_t)b * (V + 1);
    const int d = bp[j];
    int before = 0;  // the entries of the beams before b
    for (int bb = lane; bb < b; bb += 32) before += brp[(size_t)bb * (V + 1) + V];
    before = (int)__reduce_add_sync(FULL, (unsigned)before);
    const int d0 = __shfl_sync(FULL, d, 0), base = beam_off[b];
    const int64_t out = (int64_t)before + d0;
    s_start[warp][lane] = d - d0;
    s_src[warp][lane] = j < V ? seg[(size_t)b * V + j] - (d - d0) : 0;
    if (lane == 31) s_start[warp][32] = bp[min(j + 1, V)] - d0;
    __syncwarp();
    const int n = s_start[warp][32];
    int r = 0;
    for (int t0 = 0; t0 < n; t0 += 32 * RW_U) {
        int c[RW_U];
        float v[RW_U];
        unsigned short h[RW_U];
#pragma unroll
        for (int u = 0; u < RW_U; ++u) {
            const int t = t0 + 32 * u + lane;
            if (t >= n) continue;
            while (t >= s_start[warp][r + 1]) ++r;
            const int q = s_src[warp][r] + t;
            if (PREC == DAO_PREC_FP32) {
                c[u] = __ldg(col + q);
                v[u] = __ldg(val + q);
            } else {
                c[u] = __ldg(col16 + q);
                h[u] = __ldg(val16 + q);
            }
        }
#pragma unroll
        for (int u = 0; u < RW_U; ++u) {
            const int t = t0 + 32 * u + lane;
            if (t >= n) continue;
            bcol[out + t] = (unsigned short)(c[u] - base);
            if (PREC == DAO_PREC_FP32)
                bval32[out + t] = v[u];
            else
                bval16[out + t] = h[u];
        }
    }
}
}  // namespace

int beam_scan_tiles(int V) { return (V + BEAM_TILE - 1) / BEAM_TILE; }

cudaError_t build_beam_rows(const int* seg, int V, int B, int* brp, int* tmp, cudaStream_t s) {
    if (B < 1 || V < 1) return cudaSuccess;
    const int nt = beam_scan_tiles(V);
    k_beam_tiles<<<dim3(nt, B), BEAM_TILE, 0, s>>>(seg, V, nt, tmp);
    k_beam_tile_scan<<<B, BEAM_TILE, 0, s>>>(tmp, nt, V, brp);
    k_beam_offsets<<<dim3(nt, B), BEAM_TILE, 0, s>>>(seg, V, nt, tmp, brp);
    return cudaGetLastError();
}

cudaError_t build_beam_fill(int prec, const int* seg, int V, int B, const int* beam_off, const DevCSR& D,
                            cudaStream_t s) {
    if (B < 1 || V < 1) return cudaSuccess;
    const dim3 g((unsigned)(((int64_t)V + RW_T - 1) / RW_T), (unsigned)B);  // RW_W warps of 32 rows
    if (prec == DAO_PREC_FP32)
        k_beam_fill<DAO_PREC_FP32><<<g, RW_T, 0, s>>>(seg, V, beam_off, D.beam_rowptr, D.col, D.val,
                                                      nullptr, nullptr, D.beam_col, D.beam_val32, nullptr);
    else
        k_beam_fill<DAO_PREC_FP16><<<g, RW_T, 0, s>>>(seg, V, beam_off, D.beam_rowptr, nullptr, nullptr,
                                                      D.col16, D.val16, D.beam_col, nullptr, D.beam_val16);
    return cudaGetLastError();
}

cudaError_t build_merge_path(const int* prow, int V, int epg, int chunk, int n_warps, int2* out, cudaStream_t s) {
    k_merge_path<<<(n_warps + 1 + 255) / 256, 256, 0, s>>>(prow, V, epg, chunk, n_warps, out);
    return cudaGetLastError();
}

cudaError_t build_unit_max(const int* prow, int V, int epg, int* out, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(out, 0, 2 * sizeof(int), s);
    if (e != cudaSuccess || V < 1) return e;
    const int units = (V + 31) / 32;
    k_unit_max<<<(units + 255) / 256, 256, 0, s>>>(prow, V, epg, out);
    return cudaGetLastError();
}

cudaError_t build_transpose_place(int prec, const int64_t* rp, const int* col, const float* val, int V, int CH, int N,
                                  int n_ch, int* C, const int* cnt, const float* scale, DevCSR& Dt, float* tval,
                                  cudaStream_t s) {
    const int n_tile = (N + PL_TILE - 1) / PL_TILE;
    const int tw = ((N + n_tile - 1) / n_tile + 3) / 4 * 4;  // the bitmap is cleared 16 bytes at a time
    // process-wide: the largest size any launch asks for (see build_stats)
    cudaError_t e = cudaFuncSetAttribute(k_chunk_place, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)place_smem(PL_TILE));
    if (e != cudaSuccess) return e;
    k_chunk_place<<<dim3(n_ch, n_tile), PL_T, place_smem(tw), s>>>(rp, col, val, V, CH, N, tw, C, Dt.rowptr, Dt.col,
                                                                   tval);
    k_pad_t<<<blocks_for((int64_t)N * 32, 256), 256, 0, s>>>(Dt.rowptr, cnt, N, Dt.col, tval);
    if (prec == DAO_PREC_FP16)
        k_quant_t<DAO_PREC_FP16><<<blocks_for((int64_t)N * 32, 256), 256, 0, s>>>(tval, Dt.rowptr, N, scale,
                                                                                   Dt.val16);
    else if (prec == DAO_PREC_BF16)
        k_quant_t<DAO_PREC_BF16><<<blocks_for((int64_t)N * 32, 256), 256, 0, s>>>(tval, Dt.rowptr, N, scale,
                                                                                   Dt.val16);
    return cudaGetLastError();
}

}  // namespace dao
