// Pricing under MLC hardware constraints (arXiv:1003.5402, Sec. 4, last
// paragraph: besides the consecutiveness of each row's open beamlets the
// method handles interdigitation, connectedness and jaws-only delivery).
//
// One block per beam.  Every mode works on the FP64 prefix sums of the beam's
// rows, P_r[0] = 0, P_r[c + 1] = P_r[c] + w_c (column order), an interval's
// sum being P_r[R] - P_r[L]; the arithmetic and the tie rules below are fixed
// so that the result is reproducible bit for bit:
//   - interdigitation (adjacent rows' leaves may not cross: L_r <= R_{r+1} and
//     L_{r+1} <= R_r, a closed row's leaves together at some position p):
//     dynamic programme over the rows on the leaf states (L, R), 0 <= L <= R
//     <= C, f_0(s) = I_0(s), f_r(s') = I_r(s') + min over compatible s of
//     f_{r-1}(s); the minimum over the compatible states {L <= R', R >= L'} is
//     read from a two-dimensional running minimum (a suffix minimum over R,
//     then a prefix minimum over L) that keeps the smallest state index on
//     equal values, so every choice, and the trace back from the smallest
//     final state, takes the smallest index among equal values;
//   - connectedness (the open rows form one contiguous block): each row's
//     best non-empty interval (smallest (L, R) in L-major order on ties), then
//     the paper's one-pass search over those row values picks the block;
//   - jaws-only (a rectangle): for every column range [L, R) the paper's
//     one-pass search over the rows' interval sums, then the smallest value
//     over the column ranges, the earliest range on ties.
// A beam whose best value is not negative is closed (value 0).  The beam's
// value is written at its first MLC row of row_v and 0 at the others, so that
// the beam decision, which sums row_v over a beam's rows in row order, sees
// exactly the beam's value; closed rows are written as (0, 0).
#include <climits>

#include "dao_internal.h"

namespace dao {

namespace {

constexpr int MLC_THREADS = 256;
// Interdigitation: each MLC row's step takes two tables of prefix minima (at most 33
// lines of 33), a warp to a line.  A thread to a line walks 33 dependent
// comparisons: the pricing call of 9 beams of 20 x 20 took 98 us so, 79 with a warp
// scanning each line.
constexpr int MLC_THREADS_IL = 1024;
constexpr int mlc_threads(int mode) { return mode == DAO_MLC_INTERDIGITATION ? MLC_THREADS_IL : MLC_THREADS; }

// A double as an integer that orders like it (a NaN above infinity, so that it is
// never the smaller; -0 as 0): the dynamic programme's minima are chains of
// comparisons, and FP64 ones issue at 1/64 of the FP32 rate on this part (the
// pricing call under interdigitation, 9 beams of 20 x 20: 163 us with them, 98
// without, other changes to the call 7 us of that).
typedef unsigned long long mlc_key;
__device__ __forceinline__ mlc_key mlc_to_key(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned long long m = b & 0x7fffffffffffffffull;
    if (m > 0x7ff0000000000000ull) return ~0ull;
    return (b >> 63) ? 0x8000000000000000ull - m : 0x8000000000000000ull + m;
}
__device__ __forceinline__ double mlc_from_key(mlc_key k) {
    const unsigned long long h = 0x8000000000000000ull;
    return __longlong_as_double((long long)(k >= h ? k - h : (h - k) | h));
}
constexpr mlc_key MLC_KEY_INF = 0xfff0000000000000ull;  // mlc_to_key(infinity)

__device__ __forceinline__ bool mlc_better(mlc_key v, int i, mlc_key bv, int bi) {
    return v < bv || (v == bv && i < bi);
}

// index of the leaf state (L, R), 0 <= L <= R <= C (C1 = C + 1), L-major
__device__ __forceinline__ int mlc_state(int L, int R, int C1) { return L * C1 - L * (L - 1) / 2 + (R - L); }

// Inclusive running minimum over the warp's lanes of (value, index): by value, the
// smaller index on equal ones, so the same in whatever order the scan combines.
__device__ __forceinline__ void mlc_scan(mlc_key& m, int& mi) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const mlc_key om = __shfl_up_sync(0xffffffffu, m, o);
        const int oi = __shfl_up_sync(0xffffffffu, mi, o);
        if (lane >= o && mlc_better(om, oi, m, mi)) {
            m = om;
            mi = oi;
        }
    }
}

// The paper's one-pass search (Sec. 2.3) over n values v(1..n): running sum,
// largest running sum with its earliest position, best difference with the
// earliest end; returns v* and the block [a, b) (v* = 0: none).
template <class Get>
__device__ __forceinline__ double mlc_row_search(int n, Get get, int* a, int* b) {
    double s = 0.0, vbar = 0.0, best = 0.0;
    int l = 0, ls = 0, rs = 1;
    for (int r = 1; r <= n; ++r) {
        s = s + get(r - 1);
        if (s > vbar) {
            vbar = s;
            l = r;
        }
        if (s - vbar < best) {
            best = s - vbar;
            ls = l;
            rs = r + 1;
        }
    }
    *a = ls;
    *b = rs - 1;
    return best;
}

template <int MODE>
__global__ void __launch_bounds__(mlc_threads(MODE)) k_price_mlc(const float* __restrict__ w,
                                                           const int* __restrict__ beam_off,
                                                           const int* __restrict__ rows,
                                                           const int* __restrict__ cols,
                                                           const int* __restrict__ beam_row0,
                                                           double* __restrict__ row_v, int2* __restrict__ row_lr,
                                                           const int* __restrict__ skip) {
    extern __shared__ __align__(16) double sm[];
    if (skip != nullptr && *skip) return;
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    (void)lane;
    (void)warp;
    const int R = rows[b], C = cols[b], C1 = C + 1, off = beam_off[b], r0 = beam_row0[b];
    double* P = sm;  // [R][C1]
    // the rows' prices, converted by all threads; then their sums in column order
    for (int i = tid; i < R * C; i += blockDim.x) P[i / C * C1 + i % C + 1] = (double)w[off + i];
    __syncthreads();
    for (int r = tid; r < R; r += blockDim.x) {
        double acc = 0.0;
        P[r * C1] = 0.0;
        for (int c = 0; c < C; ++c) {
            acc = acc + P[r * C1 + c + 1];
            P[r * C1 + c + 1] = acc;
        }
    }
    __syncthreads();
    __shared__ double s_val;
    __shared__ int s_a, s_b, s_L, s_R;

    if constexpr (MODE == DAO_MLC_INTERDIGITATION) {
        const int NS = C1 * (C1 + 1) / 2;
        mlc_key* f = reinterpret_cast<mlc_key*>(P + R * C1);                   // [NS] of the row before, as keys
        mlc_key* Gv = f + NS;                                                   // [C1][C1]
        int* Gi = reinterpret_cast<int*>(Gv + C1 * C1);                         // [C1][C1]
        unsigned short* back = reinterpret_cast<unsigned short*>(Gi + C1 * C1);  // [R][NS]
        unsigned char* sL = reinterpret_cast<unsigned char*>(back + R * NS);     // [NS]
        unsigned char* sR = sL + NS;                                            // [NS]
        __shared__ mlc_key s_key[MLC_THREADS_IL / 32];
        __shared__ int s_idx[MLC_THREADS_IL / 32];
        __shared__ unsigned short s_path[64];  // the rows' states (at most 64 rows)
        for (int L = tid; L <= C; L += blockDim.x)
            for (int Rr = L; Rr <= C; ++Rr) {
                const int s = mlc_state(L, Rr, C1);
                sL[s] = (unsigned char)L;
                sR[s] = (unsigned char)Rr;
            }
        __syncthreads();
        for (int s = tid; s < NS; s += blockDim.x) f[s] = mlc_to_key(P[sR[s]] - P[sL[s]]);
        __syncthreads();
        for (int r = 1; r < R; ++r) {
            // H[a][x] = min over R >= max(a, x) of f(a, R): a warp per a, lane l
            // the entry R = C - l (and, of 33 entries, lane 31 also R = 0)
            for (int a = warp; a <= C; a += MLC_THREADS_IL / 32) {
                const int s0 = mlc_state(a, a, C1) - a, Rr = C - lane;
                mlc_key m = MLC_KEY_INF;
                int mi = INT_MAX;
                if (Rr >= a && mlc_better(f[s0 + Rr], s0 + Rr, m, mi)) {
                    m = f[s0 + Rr];
                    mi = s0 + Rr;
                }
                mlc_scan(m, mi);
                if (Rr >= a) {
                    Gv[a * C1 + Rr] = m;
                    Gi[a * C1 + Rr] = mi;
                }
                // below a the value at R = a stands
                const mlc_key ma = __shfl_sync(0xffffffffu, m, min(C - a, 31));
                const int ia = __shfl_sync(0xffffffffu, mi, min(C - a, 31));
                if (lane < a) {
                    Gv[a * C1 + lane] = ma;
                    Gi[a * C1 + lane] = ia;
                }
                if (C == 32 && a == 0 && lane == 31) {  // R = 0 after R = 1
                    const bool b0 = mlc_better(f[s0], s0, m, mi);
                    Gv[0] = b0 ? f[s0] : m;
                    Gi[0] = b0 ? s0 : mi;
                }
            }
            __syncthreads();
            // G[a][x] = min over a' <= a of H[a'][x]: min over L <= a, R >= x; a warp
            // per x, lane l the entry a = l (and, of 33 entries, lane 31 also a = 32)
            for (int x = warp; x <= C; x += MLC_THREADS_IL / 32) {
                mlc_key m = MLC_KEY_INF;
                int mi = INT_MAX;
                if (lane <= C) {
                    const mlc_key v = Gv[lane * C1 + x];
                    const int i = Gi[lane * C1 + x];
                    if (mlc_better(v, i, m, mi)) {
                        m = v;
                        mi = i;
                    }
                }
                mlc_scan(m, mi);
                if (lane <= C) {
                    Gv[lane * C1 + x] = m;
                    Gi[lane * C1 + x] = mi;
                }
                if (C == 32 && lane == 31) {
                    const mlc_key v = Gv[32 * C1 + x];
                    const int i = Gi[32 * C1 + x];
                    const bool b0 = mlc_better(v, i, m, mi);
                    Gv[32 * C1 + x] = b0 ? v : m;
                    Gi[32 * C1 + x] = b0 ? i : mi;
                }
            }
            __syncthreads();
            // the states compatible with (L', R') are {L <= R', R >= L'}: G[R'][L']
            const double* Pr = P + r * C1;
            for (int s = tid; s < NS; s += blockDim.x) {
                const int L = sL[s], Rr = sR[s];
                f[s] = mlc_to_key((Pr[Rr] - Pr[L]) + mlc_from_key(Gv[Rr * C1 + L]));
                const int from = Gi[Rr * C1 + L];
                back[r * NS + s] = from == INT_MAX ? (unsigned short)0 : (unsigned short)from;  // (no number before it)
            }
            __syncthreads();
        }
        // the smallest state value, the earliest among equal ones (state 0 if its value is no number)
        {
            mlc_key m = ~0ull;
            int mi = INT_MAX;
            for (int s = tid; s < NS; s += blockDim.x)
                if (mlc_better(f[s], s, m, mi)) {
                    m = f[s];
                    mi = s;
                }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const mlc_key om = __shfl_xor_sync(0xffffffffu, m, o);
                const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
                if (mlc_better(om, oi, m, mi)) {
                    m = om;
                    mi = oi;
                }
            }
            if ((tid & 31) == 0) {
                s_key[tid >> 5] = m;
                s_idx[tid >> 5] = mi;
            }
        }
        __syncthreads();
        if (tid == 0) {
            mlc_key m = s_key[0];
            int best = s_idx[0];
            for (int q = 1; q < MLC_THREADS_IL / 32; ++q)
                if (mlc_better(s_key[q], s_idx[q], m, best)) {
                    m = s_key[q];
                    best = s_idx[q];
                }
            if (f[0] == ~0ull) best = 0;
            const double v = f[best] == ~0ull ? 0.0 : mlc_from_key(f[best]);
            s_val = v;
            row_v[r0] = v < 0.0 ? v : 0.0;
            int s = best;
            for (int r = R - 1; r >= 0; --r) {
                s_path[r] = (unsigned short)s;
                if (r > 0) s = back[r * NS + s];
            }
        }
        __syncthreads();
        const bool open = s_val < 0.0;
        for (int r = tid; r < R; r += blockDim.x) {
            const int L = sL[s_path[r]], Rr = sR[s_path[r]];
            row_lr[r0 + r] = (open && L < Rr) ? make_int2(L, Rr) : make_int2(0, 0);
            if (r > 0) row_v[r0 + r] = 0.0;
        }
    } else if constexpr (MODE == DAO_MLC_CONNECTED) {
        double* m = P + R * C1;                                  // [R]
        int* lr = reinterpret_cast<int*>(m + R);                 // [R][2]
        for (int r = tid; r < R; r += blockDim.x) {
            const double* Pr = P + r * C1;
            double best = INFINITY;
            int bl = 0, br = 0;
            for (int L = 0; L < C; ++L)
                for (int Rr = L + 1; Rr <= C; ++Rr) {
                    const double v = Pr[Rr] - Pr[L];
                    if (v < best) {
                        best = v;
                        bl = L;
                        br = Rr;
                    }
                }
            m[r] = best;
            lr[2 * r] = bl;
            lr[2 * r + 1] = br;
        }
        __syncthreads();
        if (tid == 0) {
            int a = 0, e = 0;
            const double v = mlc_row_search(R, [&](int q) { return m[q]; }, &a, &e);
            const bool open = v < 0.0;
            row_v[r0] = open ? v : 0.0;
            for (int r = 0; r < R; ++r) {
                if (r > 0) row_v[r0 + r] = 0.0;
                row_lr[r0 + r] = (open && r >= a && r < e) ? make_int2(lr[2 * r], lr[2 * r + 1]) : make_int2(0, 0);
            }
        }
    } else {  // DAO_MLC_JAWS
        const int NP = C * C1 / 2;                               // column ranges L < R
        double* pv = P + R * C1;                                 // [NP]
        int* pab = reinterpret_cast<int*>(pv + NP);              // [NP][2]
        for (int p = tid; p < NP; p += blockDim.x) {
            int L = 0, q = p;
            while (q >= C - L) {
                q -= C - L;
                ++L;
            }
            const int Rr = L + 1 + q;
            int a = 0, e = 0;
            pv[p] = mlc_row_search(R, [&](int k) { return P[k * C1 + Rr] - P[k * C1 + L]; }, &a, &e);
            pab[2 * p] = a;
            pab[2 * p + 1] = e;
        }
        __syncthreads();
        if (tid == 0) {
            int best = 0;
            for (int p = 1; p < NP; ++p)
                if (pv[p] < pv[best]) best = p;
            const double v = pv[best];
            const bool open = v < 0.0;
            int L = 0, q = best;
            while (q >= C - L) {
                q -= C - L;
                ++L;
            }
            s_val = v;
            s_L = L;
            s_R = L + 1 + q;
            s_a = open ? pab[2 * best] : 0;
            s_b = open ? pab[2 * best + 1] : 0;
            row_v[r0] = open ? v : 0.0;
        }
        __syncthreads();
        for (int r = tid; r < R; r += blockDim.x) {
            if (r > 0) row_v[r0 + r] = 0.0;
            row_lr[r0 + r] = (r >= s_a && r < s_b) ? make_int2(s_L, s_R) : make_int2(0, 0);
        }
    }
}

template <int MODE>
cudaError_t mlc_launch(const float* w, const int* beam_off, const int* rows, const int* cols, const int* beam_row0,
                       int n_beams, size_t smem, double* row_v, int2* row_lr, const int* skip, cudaStream_t stream) {
    k_price_mlc<MODE><<<n_beams, mlc_threads(MODE), smem, stream>>>(w, beam_off, rows, cols, beam_row0, row_v, row_lr,
                                                              skip);
    return cudaGetLastError();
}

}  // namespace

size_t mlc_smem_bytes(int mode, int max_rows, int max_cols) {
    const size_t R = (size_t)max_rows, C = (size_t)max_cols, C1 = C + 1;
    switch (mode) {
        case DAO_MLC_INTERDIGITATION: {
            const size_t NS = C1 * (C1 + 1) / 2;
            return 8 * (R * C1 + NS + C1 * C1) + 4 * C1 * C1 + 2 * R * NS + 2 * NS;
        }
        case DAO_MLC_CONNECTED:
            return 8 * (R * C1 + R) + 8 * R;
        case DAO_MLC_JAWS: {
            const size_t NP = C * C1 / 2;
            return 8 * (R * C1 + NP) + 8 * NP;
        }
    }
    return 0;
}

cudaError_t mlc_configure(int mode, size_t smem) {
    // the attribute is process-wide and plans may be created from several threads
    // at once: the largest size of any plan (64 rows of 32 beamlets), never this
    // plan's own, which another thread's smaller plan could otherwise lower
    if (smem > mlc_smem_bytes(mode, 64, 32)) return cudaErrorInvalidValue;
    smem = mlc_smem_bytes(mode, 64, 32);
    switch (mode) {
        case DAO_MLC_INTERDIGITATION:
            return cudaFuncSetAttribute(k_price_mlc<DAO_MLC_INTERDIGITATION>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        case DAO_MLC_CONNECTED:
            return cudaFuncSetAttribute(k_price_mlc<DAO_MLC_CONNECTED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)smem);
        case DAO_MLC_JAWS:
            return cudaFuncSetAttribute(k_price_mlc<DAO_MLC_JAWS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)smem);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_price_mlc(int mode, const float* w, const int* beam_off, const int* rows, const int* cols,
                             const int* beam_row0, int n_beams, size_t smem, double* row_v, int2* row_lr,
                             const int* skip, cudaStream_t stream, int* launches) {
    if (n_beams == 0) return cudaSuccess;
    cudaError_t e = cudaErrorInvalidValue;
    switch (mode) {
        case DAO_MLC_INTERDIGITATION:
            e = mlc_launch<DAO_MLC_INTERDIGITATION>(w, beam_off, rows, cols, beam_row0, n_beams, smem, row_v, row_lr,
                                                    skip, stream);
            break;
        case DAO_MLC_CONNECTED:
            e = mlc_launch<DAO_MLC_CONNECTED>(w, beam_off, rows, cols, beam_row0, n_beams, smem, row_v, row_lr, skip,
                                              stream);
            break;
        case DAO_MLC_JAWS:
            e = mlc_launch<DAO_MLC_JAWS>(w, beam_off, rows, cols, beam_row0, n_beams, smem, row_v, row_lr, skip,
                                         stream);
            break;
    }
    ++*launches;
    return e;
}

}  // namespace dao
