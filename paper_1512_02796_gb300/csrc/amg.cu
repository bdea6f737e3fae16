// Device side of the smoothed-aggregation multigrid preconditioner (see
// amg.h): the numeric set-up of the hierarchy from the assembled FP64
// operator, the V-cycle, and the conjugate-gradient driver that uses it.
//
// Layout: vectors are node-major with R right-hand sides interleaved
// (x[i * R + r]), as everywhere in the library.  The K operator has one value
// set for all right-hand sides; M_delta has two (its blocks, R = 2, column r
// uses set r), and every level of its hierarchy keeps two sets over one
// pattern.  All sums run in a fixed order: results are identical from run
// to run.
#include <algorithm>
#include <array>
#include <cmath>
#include <cstdio>
#include <exception>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "abi_internal.h"
#include "amg.h"

namespace qpat {

struct SellDev {
    int64_t n = 0;
    const int64_t* ptr = nullptr;
    const int32_t* col = nullptr;
    const uint16_t* len = nullptr;  // nullptr (row-major only): ptr[i + 1] - ptr[i]
    int64_t entries = 0;
    int maxlen = 0;
    int rowmajor = 0;  // layout (see SellPattern)
};

struct LevelDev {
    SellDev A;
    const int32_t* diag = nullptr;
    int64_t nc = 0;
    SellDev P;
    const uint16_t* a2p = nullptr;
    const uint16_t* pself = nullptr;
    const int64_t* ap_ptr = nullptr;
    const int32_t* ap_col = nullptr;
    const int64_t* ap_sptr = nullptr;
    const uint16_t* ap_slot = nullptr;
    int64_t ap_nnz = 0;
    int ap_maxlen = 0;
    SellDev R;
    const int64_t* r_src = nullptr;
    const int64_t* g_ptr = nullptr;
    const uint16_t* g_slot = nullptr;
};

namespace {

__device__ __forceinline__ int row_len(const SellDev& S, int64_t i) {
    return S.len ? int(S.len[i]) : int(S.ptr[i + 1] - S.ptr[i]);
}

__device__ __forceinline__ int64_t spos(const SellDev& S, int64_t row, int k) {
    return S.rowmajor ? S.ptr[row] + k : (S.ptr[row >> 5] + k) * 32 + (row & 31);
}

// ---------------------------------------------------------------- set-up kernels

// The fine operator of K's cycle: the entries of K in the prior's pattern (a
// subset of each row, in the same order), the others added to the diagonal.
__global__ void __launch_bounds__(256) k_lump(SellDev K, const int* ent_edge, const uint8_t* in_prior, SellDev F,
                                              const int32_t* diag, const double* val, double* out) {
    const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (i >= K.n) return;
    const int L = K.len[i];
    double lump = 0.0;
    int k2 = 0;
    for (int k = 0; k < L; ++k) {
        const int64_t at = spos(K, i, k);
        const int e = ent_edge[at];
        if (e < 0 || in_prior[e])
            out[spos(F, i, k2++)] = val[at];
        else
            lump += val[at];
    }
    out[spos(F, i, diag[i])] += lump;
}

// Inverse diagonal (n x NV, interleaved) and the Gershgorin bound
// max_i sum_j |a_ij| / a_ii of D^-1 A per value set (hi must start at 0; the
// bound is >= 1, so the bits of the positive doubles order like integers).
template <int NV>
__global__ void __launch_bounds__(256) k_dinv_hi(SellDev A, const int32_t* diag, const double* v0, const double* v1,
                                                 double* dinv, double* hi) {
    __shared__ double bmax[NV][8];
    const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        double ratio = 0.0;
        if (i < A.n) {
            const double* val = v == 0 ? v0 : v1;
            const int L = A.len[i];
            double s = 0.0;
            for (int k = 0; k < L; ++k) s += fabs(val[spos(A, i, k)]);
            const double d = val[spos(A, i, diag[i])];
            dinv[i * NV + v] = 1.0 / d;
            ratio = s / fabs(d);
        }
        // the largest ratio of the block (max is exact in any order), then one atomic per block
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ratio = fmax(ratio, __shfl_xor_sync(0xffffffffu, ratio, o));
        if (lane == 0) bmax[v][warp] = ratio;
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        double m = 0.0;
        for (int w = 0; w < int(blockDim.x >> 5); ++w) m = fmax(m, bmax[threadIdx.x][w]);
        atomicMax(reinterpret_cast<unsigned long long*>(hi + threadIdx.x), __double_as_longlong(m));
    }
}

// Upper end of the smoothing interval: the Gershgorin bound with a margin.
// A single step (degree 1) multiplies the top of the spectrum by
// 1 - 2 / (1 + 1 / ratio) = -0.94 without it, so error there (the checkerboard
// of a structured grid, which reaches the bound) would hardly decay; with 1.13
// it is -0.71 and the 128^3 solves take half the iterations.
constexpr double kSmoothMargin = 1.13;

// Weighted inverse diagonal of the degree-1 smoother, wd = D^-1 / theta, and the scaled operator A diag(wd), so that
// one gather forms b - A (wd b).
template <int NV>
__global__ void __launch_bounds__(256) k_weights(int64_t n, const double* dinv, const double* hi, double ratio,
                                                 double* wd) {
    __shared__ double w[NV];
    if (threadIdx.x < NV) {
        const double h = kSmoothMargin * hi[threadIdx.x];
        w[threadIdx.x] = 1.0 / (0.5 * (h + h / ratio));
    }
    __syncthreads();
    const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (i < n * NV) wd[i] = w[i % NV] * dinv[i];
}
template <int NV>
__global__ void __launch_bounds__(256) k_scaled(int64_t entries, const int32_t* col, const double* wd, const double* v0,
                                                const double* v1, double* s0, double* s1) {
    const int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (e >= entries) return;
    const int64_t j = col[e];
    s0[e] = v0[e] * wd[j * NV];
    if (NV == 2) s1[e] = v1[e] * wd[j * NV + 1];
}

// Row i of P: 1 - omega on the row's own aggregate and omega shared out over
// the aggregates of its graph neighbours by their couplings -a_ij (only
// negative ones count).  For a row that sums to 0 this is one damped Jacobi
// step on P_tent; for every row it keeps the constants exactly, which is what
// the 1 / delta mode of M_delta needs.  omega: amg.h.
template <int NV>
__global__ void __launch_bounds__(256) k_prolong(SellDev A, SellDev P, const int32_t* diag, const uint16_t* a2p,
                                                 const uint16_t* pself, const double* v0, const double* v1, double* p0,
                                                 double* p1) {
    const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (i >= A.n) return;
    const int L = A.len[i], LP = P.len[i], dk = diag[i];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const double* val = v == 0 ? v0 : v1;
        double* pv = v == 0 ? p0 : p1;
        double sum = 0.0;
        for (int k = 0; k < L; ++k) {
            const int64_t at = spos(A, i, k);
            if (k != dk && a2p[at] != kAmgDropped) sum += fmax(-val[at], 0.0);
        }
        for (int k = 0; k < LP; ++k) pv[spos(P, i, k)] = 0.0;
        const bool any = sum > 0.0;
        pv[spos(P, i, pself[i])] = any ? 1.0 - kAmgOmega : 1.0;
        if (!any) continue;
        const double w = kAmgOmega / sum;
        for (int k = 0; k < L; ++k) {
            const int64_t at = spos(A, i, k);
            if (k != dk && a2p[at] != kAmgDropped) pv[spos(P, i, a2p[at])] += w * fmax(-val[at], 0.0);
        }
    }
}

// Row i of A P = sum over the entries a_ij of row i of A of a_ij (row j of
// P), 8 lanes per row and value set (4 rows per warp): the entries of row i
// of A are taken one after the other and the 8 lanes add a_ij P[j, :] into
// the row's shared accumulator; the columns of one P row differ, so no two
// lanes meet on a slot and every value is summed in the same order on every
// run.  Also writes P2 = P - wd (A P), the prolongation followed by the
// degree-1 smoother's step, in the pattern of A P (wd: nullptr = not wanted).
constexpr int kApLanes = 8;
template <int NV>
__global__ void k_ap(SellDev A, SellDev P, const int32_t* diag, const int64_t* ap_ptr, const int64_t* ap_sptr,
                     const uint16_t* ap_slot, int64_t ap_nnz, int ap_maxlen, const double* v0, const double* v1,
                     const double* p0, const double* p1, const double* wd, double* ap, double* p2) {
    extern __shared__ double acc_all[];
    const int grp = threadIdx.x / kApLanes, sub = threadIdx.x % kApLanes;
    const int64_t task = blockIdx.x * int64_t(blockDim.x / kApLanes) + grp;
    const bool valid = task < A.n * NV;
    const int64_t i = valid ? task / NV : 0;
    const int v = valid ? int(task % NV) : 0;
    double* acc = acc_all + int64_t(grp) * ap_maxlen;
    const double* val = v == 0 ? v0 : v1;
    const double* pv = v == 0 ? p0 : p1;
    const int64_t b = valid ? ap_ptr[i] : 0, cnt = valid ? ap_ptr[i + 1] - b : 0;
    for (int64_t t = sub; t < cnt; t += kApLanes) acc[t] = 0.0;
    __syncwarp();
    int64_t o = valid ? ap_sptr[i] : 0, own = 0;
    const int L = valid ? A.len[i] : 0, dk = valid ? diag[i] : 0;
    // the longest row of the warp sets the step count, so that every lane reaches each __syncwarp
    int Lw = L;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) Lw = max(Lw, __shfl_xor_sync(0xffffffffu, Lw, s));
    for (int k = 0; k < Lw; ++k) {
        if (k < L) {
            const int64_t at = spos(A, i, k);
            const int64_t j = A.col[at];
            const double a = val[at];
            const int LPj = P.len[j];
            if (k == dk) own = o;
            for (int kk = sub; kk < LPj; kk += kApLanes) acc[ap_slot[o + kk]] += a * pv[spos(P, j, kk)];
            o += LPj;
        }
        __syncwarp();
    }
    double* out = ap + v * ap_nnz + b;
    for (int64_t t = sub; t < cnt; t += kApLanes) out[t] = acc[t];
    if (wd) {
        const double w = valid ? wd[i * NV + v] : 0.0;
        for (int64_t t = sub; t < cnt; t += kApLanes) acc[t] *= -w;
        __syncwarp();
        const int LP = valid ? P.len[i] : 0;
        for (int kk = sub; kk < LP; kk += kApLanes) acc[ap_slot[own + kk]] += pv[spos(P, i, kk)];
        __syncwarp();
        double* out2 = p2 + v * ap_nnz + b;
        for (int64_t t = sub; t < cnt; t += kApLanes) out2[t] = acc[t];
    }
}

// R = P^T values gathered from P (padding 0).
template <int NV>
__global__ void k_rvals(int64_t entries, const int64_t* r_src, const double* p0, const double* p1, double* r0,
                        double* r1) {
    const int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (e >= entries) return;
    const int64_t s = r_src[e];
    r0[e] = s >= 0 ? p0[s] : 0.0;
    if (NV == 2) r1[e] = s >= 0 ? p1[s] : 0.0;
}

// Coarse row I of P^T (A P), one warp per row and value set: the R entries
// (fine rows i, ascending) are taken one after the other and the lanes add
// the entries of row i of A P into the row's shared accumulator; within one
// fine row the columns differ, so no two lanes meet on a slot and every
// coarse value is summed in the same order on every run.
template <int NV>
__global__ void k_galerkin(SellDev R, SellDev C, const int64_t* r_src, const int64_t* ap_ptr, const int64_t* g_ptr,
                           const uint16_t* g_slot, int64_t ap_nnz, const double* p0, const double* p1,
                           const double* ap, double* c0, double* c1) {
    extern __shared__ double acc_all[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    const int64_t task = blockIdx.x * int64_t(wpb) + warp;
    if (task >= C.n * NV) return;
    const int64_t I = task / NV;
    const int v = int(task % NV);
    double* acc = acc_all + int64_t(warp) * C.maxlen;
    const double* pv = v == 0 ? p0 : p1;
    const double* apv = ap + v * ap_nnz;
    double* out = v == 0 ? c0 : c1;
    const int LC = C.len[I], LR = R.len[I];
    for (int k = lane; k < LC; k += 32) acc[k] = 0.0;
    __syncwarp();
    int64_t o = g_ptr[I];
    for (int k = 0; k < LR; ++k) {
        const int64_t at = spos(R, I, k);
        const int64_t i = R.col[at];
        const double p = pv[r_src[at]];
        const int64_t b = ap_ptr[i], cnt = ap_ptr[i + 1] - b;
        for (int64_t t = lane; t < cnt; t += 32) acc[g_slot[o + t]] += p * apv[b + t];
        o += cnt;
        __syncwarp();
    }
    for (int k = lane; k < LC; k += 32) out[spos(C, I, k)] = acc[k];
}

// Gauss-Jordan inversion of the (symmetric positive definite) coarsest
// operator, one CTA per value set, without pivoting: the pivots of an SPD
// matrix are its positive Schur complements.  The matrix stays in registers
// (thread (w, lane) holds rows w + 32 u, columns lane + 32 v); a step passes
// its pivot row and column through shared memory, double-buffered, with one
// barrier.  n^3 multiply-adds on one SM's FP64 pipe bound it (64 rows: ~70 us).
constexpr int kInvTiles = kAmgCoarsest / 32;
template <int NV>
__global__ void __launch_bounds__(1024) k_dense_inv(SellDev A, const double* v0, const double* v1, double* inv) {
    extern __shared__ double dense[];
    __shared__ double row[2][kAmgCoarsest], col[2][kAmgCoarsest], piv[2];
    const int n = int(A.n), w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double* val = blockIdx.x == 0 ? v0 : v1;
    for (int t = threadIdx.x; t < n * n; t += blockDim.x) dense[t] = 0.0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        for (int k = 0; k < A.len[i]; ++k) {
            const int64_t at = spos(A, i, k);
            dense[i * n + A.col[at]] += val[at];
        }
    __syncthreads();
    double a[kInvTiles][kInvTiles];
#pragma unroll
    for (int u = 0; u < kInvTiles; ++u)
#pragma unroll
        for (int v = 0; v < kInvTiles; ++v) {
            const int i = w + 32 * u, j = lane + 32 * v;
            a[u][v] = i < n && j < n ? dense[i * n + j] : 0.0;
        }
    auto publish = [&](int k) {
        const int b = k & 1;
#pragma unroll
        for (int u = 0; u < kInvTiles; ++u)
#pragma unroll
            for (int v = 0; v < kInvTiles; ++v) {
                const int i = w + 32 * u, j = lane + 32 * v;
                if (i == k) row[b][j] = a[u][v];
                if (j == k) col[b][i] = a[u][v];
                if (i == k && j == k) piv[b] = 1.0 / a[u][v];
            }
    };
    publish(0);
    for (int k = 0; k < n; ++k) {
        __syncthreads();
        const int b = k & 1;
        const double rp = piv[b];
        double r[kInvTiles];
#pragma unroll
        for (int v = 0; v < kInvTiles; ++v) r[v] = row[b][lane + 32 * v] * rp;
#pragma unroll
        for (int u = 0; u < kInvTiles; ++u) {
            const int i = w + 32 * u;
            const double c = col[b][i];
#pragma unroll
            for (int v = 0; v < kInvTiles; ++v) {
                const int j = lane + 32 * v;
                a[u][v] = i == k ? (j == k ? rp : r[v]) : j == k ? -c * rp : fma(-c, r[v], a[u][v]);
            }
        }
        if (k + 1 < n) publish(k + 1);
    }
#pragma unroll
    for (int u = 0; u < kInvTiles; ++u)
#pragma unroll
        for (int v = 0; v < kInvTiles; ++v) {
            const int i = w + 32 * u, j = lane + 32 * v;
            if (i < n && j < n) inv[int64_t(blockIdx.x) * n * n + i * n + j] = a[u][v];
        }
}

__global__ void k_d2f(int64_t n, const double* in, float* out) {
    const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (i < n) out[i] = float(in[i]);
}

}  // namespace

namespace {

// ---------------------------------------------------------------- solve kernels

constexpr int kRedMaxGrid = 152 * 8;  // blocks of the reducing kernels

template <typename T, int R>
__device__ __forceinline__ void ldR(const T* p, T* v) {
    if constexpr (std::is_same<T, double>::value && R % 2 == 0) {
#pragma unroll
        for (int r = 0; r < R; r += 2) {
            const double2 t = *reinterpret_cast<const double2*>(p + r);
            v[r] = t.x;
            v[r + 1] = t.y;
        }
    } else if constexpr (std::is_same<T, float>::value && R % 4 == 0) {
#pragma unroll
        for (int r = 0; r < R; r += 4) {
            const float4 t = *reinterpret_cast<const float4*>(p + r);
            v[r] = t.x;
            v[r + 1] = t.y;
            v[r + 2] = t.z;
            v[r + 3] = t.w;
        }
    } else if constexpr (std::is_same<T, float>::value && R == 2) {
        const float2 t = *reinterpret_cast<const float2*>(p);
        v[0] = t.x;
        v[1] = t.y;
    } else {
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = p[r];
    }
}

template <typename T, int R>
__device__ __forceinline__ void stR(T* p, const T* v) {
    if constexpr (std::is_same<T, double>::value && R % 2 == 0) {
#pragma unroll
        for (int r = 0; r < R; r += 2) *reinterpret_cast<double2*>(p + r) = make_double2(v[r], v[r + 1]);
    } else if constexpr (std::is_same<T, float>::value && R % 4 == 0) {
#pragma unroll
        for (int r = 0; r < R; r += 4) *reinterpret_cast<float4*>(p + r) = make_float4(v[r], v[r + 1], v[r + 2], v[r + 3]);
    } else {
#pragma unroll
        for (int r = 0; r < R; ++r) p[r] = v[r];
    }
}

// acc = (A x)_i for the R columns of row i (NV = 2: column r uses value set r), by one thread.
template <typename T, int R, int NV>
__device__ __forceinline__ void row_apply(const SellDev& A, const T* v0, const T* v1, const T* x, int64_t i, T* acc) {
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = T(0);
    const int L = row_len(A, i);
    for (int k = 0; k < L; ++k) {
        const int64_t at = spos(A, i, k);
        const int64_t c = A.col[at];
        T xv[R];
        ldR<T, R>(x + c * R, xv);
        if constexpr (NV == 1) {
            const T a = v0[at];
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fma(a, xv[r], acc[r]);
        } else {
            acc[0] = fma(v0[at], xv[0], acc[0]);
            acc[1] = fma(v1[at], xv[1], acc[1]);
        }
    }
}

// x = A^-1 b on the coarsest level (dense inverse, n <= kAmgCoarsest).
template <typename T, int R, int NV>
__global__ void k_dense_apply(int n, const T* inv, const T* b, T* x) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n * R; t += gridDim.x * blockDim.x) {
        const int i = t / R, r = t % R;
        const T* row = inv + int64_t(NV == 2 ? r : 0) * n * n + int64_t(i) * n;
        T s = T(0);
        for (int j = 0; j < n; ++j) s = fma(row[j], b[j * R + r], s);
        x[t] = s;
    }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Block totals of Q per-thread values, in a fixed order, to part[blockIdx * Q + q].
template <int Q>
__device__ __forceinline__ void block_partials(double* v, double* part) {
    __shared__ double red[8][Q];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const double t = warp_sum(v[q]);
        if (lane == 0) red[warp][q] = t;
    }
    __syncthreads();
    if (threadIdx.x < Q) {
        double s = 0.0;
        for (int w = 0; w < int(blockDim.x >> 5); ++w) s += red[w][threadIdx.x];
        part[int64_t(blockIdx.x) * Q + threadIdx.x] = s;
    }
}

// Total of quantity q over G block partials (a full warp calls it; every lane gets it).
__device__ __forceinline__ double total_of(const double* part, int G, int Q, int q) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};  // four loads in flight
    const int lane = threadIdx.x & 31;
    for (int g = lane; g < G; g += 128)
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (g + 32 * u < G) s[u] += __ldcg(part + int64_t(g + 32 * u) * Q + q);
    return warp_sum((s[0] + s[1]) + (s[2] + s[3]));
}

// Grid totals of the block partials by the block that finishes last (the
// counter wraps back to 0): true in that block only, tot[q] then holds the
// totals, summed in the same order whichever block it is.
template <int Q>
__device__ __forceinline__ bool last_block_totals(const double* part, unsigned* count, double* tot) {
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(count, gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    if (!last) return false;
    __threadfence();
    for (int q = threadIdx.x >> 5; q < Q; q += int(blockDim.x >> 5)) {
        const double t = total_of(part, gridDim.x, Q, q);
        if ((threadIdx.x & 31) == 0) tot[q] = t;
    }
    __syncthreads();
    return true;
}

// ---- rows with several lanes: lanes x C right-hand sides (16-byte accesses) x G groups that share a row's entries
// (G may span the warps of a block).  The group's sums are combined by an xor tree, then over the warps in order.
template <typename T, int R>
constexpr int kLaneRhs = R == 1 ? 1 : sizeof(T) == 8 ? 2 : R % 4 == 0 ? 4 : 2;

template <typename T, int R, int NV>
__device__ __forceinline__ void row_part(const SellDev& A, const T* v0, const T* v1, const T* x, int64_t i, int c0, int g,
                                         int G, bool valid, T* acc) {
    constexpr int C = kLaneRhs<T, R>, U = 4;  // U entries in flight
#pragma unroll
    for (int r = 0; r < C; ++r) acc[r] = T(0);
    const int L = valid ? row_len(A, i) : 0;
    const int64_t base = !valid ? 0 : A.rowmajor ? A.ptr[i] : A.ptr[i >> 5] * 32 + (i & 31);
    const int64_t stride = A.rowmajor ? 1 : 32;
    for (int k0 = g; k0 < L; k0 += U * G) {
        T a0[U], a1[U], xv[U][C];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = k0 + u * G;
            const int64_t at = base + int64_t(k < L ? k : k0) * stride;
            a0[u] = k < L ? __ldg(v0 + at) : T(0);
            if (NV == 2) a1[u] = k < L ? __ldg(v1 + at) : T(0);
            ldR<T, C>(x + int64_t(__ldg(A.col + at)) * R + c0, xv[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (k0 + u * G >= L) break;
            if constexpr (NV == 1) {
#pragma unroll
                for (int r = 0; r < C; ++r) acc[r] = fma(a0[u], xv[u][r], acc[r]);
            } else {
                acc[0] = fma(a0[u], xv[u][0], acc[0]);
                acc[1] = fma(a1[u], xv[u][1], acc[1]);
            }
        }
    }
}

// Threads of a block over rows: LPR lanes of one row's right-hand sides, GW
// entry groups in a warp, W warps per row.  rows() per block.
template <typename T, int R, int GW, int W>
struct RowMap {
    static constexpr int C = kLaneRhs<T, R>, LPR = R / C, PER = LPR * GW, RPB = W > 1 ? 8 / W : 256 / PER;
    static_assert(PER <= 32 && (W == 1 || PER == 32), "a row's lanes fill whole warps when it spans several");
    int lane, warp, c0, g, slot;  // slot: row within the block
    __device__ RowMap() {
        lane = threadIdx.x & 31;
        warp = threadIdx.x >> 5;
        c0 = (lane % LPR) * C;
        g = (lane % PER) / LPR + (W > 1 ? (warp % W) * GW : 0);
        slot = W > 1 ? warp / W : threadIdx.x / PER;
    }
    // sums the groups of the row; valid in lanes with g == 0
    __device__ void combine(T* acc) const {
        if constexpr (GW > 1) {
#pragma unroll
            for (int r = 0; r < C; ++r)
#pragma unroll
                for (int o = PER / 2; o >= LPR; o >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
        }
        if constexpr (W > 1) {
            __shared__ T part[8][R];
            if (lane < LPR)
#pragma unroll
                for (int r = 0; r < C; ++r) part[warp][c0 + r] = acc[r];
            __syncthreads();
            if (g == 0)
                for (int w = 1; w < W; ++w)
#pragma unroll
                    for (int r = 0; r < C; ++r) acc[r] += part[warp + w][c0 + r];
            __syncthreads();
        }
    }
    // block totals of NQ quantities per right-hand side (acc[q * C + r] in the lanes with g == 0; 0 elsewhere)
    template <int NQ>
    __device__ void block_totals(const double* acc, double* part) const {
        __shared__ double red[8][NQ * R];
#pragma unroll
        for (int q = 0; q < NQ; ++q)
#pragma unroll
            for (int r = 0; r < C; ++r) {
                double v = acc[q * C + r];
#pragma unroll
                for (int o = 16; o >= LPR; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane < LPR) red[warp][q * R + c0 + r] = v;
            }
        __syncthreads();
        if (threadIdx.x < NQ * R) {
            double t = 0.0;
            for (int w = 0; w < 8; ++w) t += red[w][threadIdx.x];
            part[int64_t(blockIdx.x) * NQ * R + threadIdx.x] = t;
        }
    }
};

// Degree-1 cycle on one level (b the level's right-hand side, wd the weighted inverse diagonal, see k_weights):
//   MODE 0: y = b - (A diag(wd)) b           (residual after the pre-smoothing step from zero)
//   MODE 1: y = R x                          (restriction)
//   MODE 2: y = P2 e + wd (b + res)          (prolongation, correction and post-smoothing step: with x = wd b + P e,
//                                             x + wd (b - A x) = wd (b + res) + (P - wd A P) e)
//   MODE 3: y = b + A x
// Three kernels a level; the smoothed iterate itself is never stored.  FP64: bound by FP64 issue (A, P and P2 rows
// hold 7, 4 and 10 entries on a Kuhn mesh, 21 multiply-adds a node and right-hand side).
template <typename T, int R, int NV, int MODE, int GW, int W>
__global__ void __launch_bounds__(256) k_level(SellDev A, const T* __restrict__ v0, const T* __restrict__ v1,
                                               const T* __restrict__ x, const T* __restrict__ wd,
                                               const T* __restrict__ b, const T* __restrict__ res, T* __restrict__ y) {
    const RowMap<T, R, GW, W> m;
    constexpr int C = RowMap<T, R, GW, W>::C;
    const int64_t i = blockIdx.x * int64_t(m.RPB) + m.slot;
    T acc[C];
    row_part<T, R, NV>(A, v0, v1, x, i, m.c0, m.g, GW * W, i < A.n, acc);
    m.combine(acc);
    if (i >= A.n || m.g != 0) return;
    const int64_t o = i * R + m.c0;
    if constexpr (MODE == 0) {
        T bv[C];
        ldR<T, C>(b + o, bv);
#pragma unroll
        for (int r = 0; r < C; ++r) acc[r] = bv[r] - acc[r];
    } else if constexpr (MODE == 3) {
        T bv[C];
        ldR<T, C>(b + o, bv);
#pragma unroll
        for (int r = 0; r < C; ++r) acc[r] = bv[r] + acc[r];
    } else if constexpr (MODE == 2) {
        T bv[C], rv[C];
        ldR<T, C>(b + o, bv);
        ldR<T, C>(res + o, rv);
#pragma unroll
        for (int r = 0; r < C; ++r) acc[r] = fma(wd[i * NV + (NV == 2 ? m.c0 + r : 0)], bv[r] + rv[r], acc[r]);
    }
    stR<T, C>(y + o, acc);
}

// Chebyshev smoothing step k (of a polynomial in D^-1 A on [hi / ratio, hi], hi with its margin):
//   res = b - A x_in  (FIRST: x_in = 0, res = b),
//   d = c_d d + c_r D^-1 res,  x_out = x_in + d,
// with the coefficients of the three-term recurrence (Saad, Iterative
// Methods for Sparse Linear Systems, Alg. 12.1): theta, delta the centre and
// half-width of the interval, sigma = theta / delta, rho_0 = 1 / sigma,
// rho_k = 1 / (2 sigma - rho_{k-1}); step 0: c_d = 0, c_r = 1 / theta;
// step k: c_d = rho_k rho_{k-1}, c_r = 2 rho_k / delta.
template <typename T, int R, int NV, bool FIRST, int GW>
__global__ void __launch_bounds__(256) k_cheb(SellDev A, const T* v0, const T* v1, const T* dinv, const double* hi,
                                              double ratio, int k, const T* x_in, T* x_out, T* d, const T* b) {
    const RowMap<T, R, GW, 1> m;
    constexpr int C = RowMap<T, R, GW, 1>::C;
    __shared__ T cd[NV], cr[NV];  // a block's threads share the divisions
    if (threadIdx.x < NV) {
        const double h = kSmoothMargin * hi[threadIdx.x], lo = h / ratio;
        const double theta = 0.5 * (h + lo), delta = 0.5 * (h - lo), sigma = theta / delta;
        double rho_prev = 1.0 / sigma, rho = rho_prev;
        for (int j = 1; j <= k; ++j) {
            rho_prev = rho;
            rho = 1.0 / (2.0 * sigma - rho_prev);
        }
        cd[threadIdx.x] = k == 0 ? T(0) : T(rho * rho_prev);
        cr[threadIdx.x] = k == 0 ? T(1.0 / theta) : T(2.0 * rho / delta);
    }
    __syncthreads();
    const int64_t i = blockIdx.x * int64_t(m.RPB) + m.slot;
    T res[C], bv[C], dv[C], xv[C];
    if constexpr (!FIRST) {
        row_part<T, R, NV>(A, v0, v1, x_in, i, m.c0, m.g, GW, i < A.n, res);
        m.combine(res);
    }
    if (i >= A.n || m.g != 0) return;
    const int64_t o = i * R + m.c0;
    ldR<T, C>(b + o, bv);
    if constexpr (FIRST) {
#pragma unroll
        for (int r = 0; r < C; ++r) {
            res[r] = bv[r];
            xv[r] = T(0);
        }
    } else {
        ldR<T, C>(x_in + o, xv);
#pragma unroll
        for (int r = 0; r < C; ++r) res[r] = bv[r] - res[r];
    }
    if (k > 0) ldR<T, C>(d + o, dv);
#pragma unroll
    for (int r = 0; r < C; ++r) {
        const int v = NV == 2 ? m.c0 + r : 0;
        const T upd = cr[v] * dinv[i * NV + v] * res[r];
        dv[r] = k > 0 ? fma(cd[v], dv[r], upd) : upd;
        xv[r] += dv[r];
    }
    stR<T, C>(d + o, dv);
    stR<T, C>(x_out + o, xv);
}

// ---- conjugate gradients (FP64), R right-hand sides; ctl[0] status, ctl[1] RHS still running

// x = 0, r = b, partials of b.b
template <int R>
__global__ void __launch_bounds__(256) k_cg_init(int64_t n, const double* b, double* x, double* r, double* part) {
    double acc[R];
#pragma unroll
    for (int q = 0; q < R; ++q) acc[q] = 0.0;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        double bv[R], z[R];
        ldR<double, R>(b + i * R, bv);
#pragma unroll
        for (int q = 0; q < R; ++q) {
            acc[q] = fma(bv[q], bv[q], acc[q]);
            z[q] = 0.0;
        }
        stR<double, R>(r + i * R, bv);
        stR<double, R>(x + i * R, z);
    }
    block_partials<R>(acc, part);
}

// x = x0, r = b - A x0, partials of b.b and of r.r (the stopping target stays rtol |b|); x0 may be x
template <int R, int NV>
__global__ void __launch_bounds__(256) k_cg_init_x0(SellDev A, const double* v0, const double* v1, const double* b,
                                                    const double* x0, double* x, double* r, double* part) {
    double acc[2 * R];
#pragma unroll
    for (int q = 0; q < 2 * R; ++q) acc[q] = 0.0;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < A.n; i += int64_t(gridDim.x) * blockDim.x) {
        double bv[R], av[R], xv[R];
        row_apply<double, R, NV>(A, v0, v1, x0, i, av);
        ldR<double, R>(b + i * R, bv);
        ldR<double, R>(x0 + i * R, xv);
#pragma unroll
        for (int q = 0; q < R; ++q) {
            acc[q] = fma(bv[q], bv[q], acc[q]);
            av[q] = bv[q] - av[q];
            acc[R + q] = fma(av[q], av[q], acc[R + q]);
        }
        stR<double, R>(r + i * R, av);
        if (x != x0) stR<double, R>(x + i * R, xv);
    }
    block_partials<2 * R>(acc, part);
}

// x = r = 0 on the right-hand sides with b = 0, whatever the guess was
template <int R>
__global__ void __launch_bounds__(256) k_cg_clear(int64_t n, const double* bb, double* x, double* r) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n * R; i += int64_t(gridDim.x) * blockDim.x)
        if (bb[i % R] == 0.0) x[i] = r[i] = 0.0;
}

// Control words of a CG solve (int ctl[]): [0] status, [1] right-hand sides
// still running, [2] iterations done, [3] 1 before the first direction,
// [4] iteration cap, [5] right-hand sides with b = 0 and a residual (from a
// guess), [6] right-hand sides with a scale other than 1; the per-RHS running
// flags follow at ctl + kCtlActive.
constexpr int kCtlActive = 8;

// bb = totals of b.b.  A right-hand side with b = 0 is solved by x = 0, and
// one whose guess already meets the target by that guess: neither runs (a
// residual of 0 would have no direction).  Q: quantities per right-hand side
// in the partials (2: r.r behind b.b; 1: r = b).  scale: the FP32 cycle works on
// scale r, so that neither small nor large right-hand sides leave FP32's range:
// 1 where |r| lies in [2^-20, 2^60] (53 binary digits less at the end of a solve,
// and as many again between entries, still lie above 2^-126), else the
// power of two that brings |r| to [1, 2).  z, p and q then carry it too, alpha
// its inverse, and beta and the iterates are the same to the bit.
// stop: the |r|^2 at which the iteration leaves a right-hand side: the target
// tol[0] |b|^2, or, in sweeps (tol[1] > 0), tol[1] times |r|^2 at the sweep's
// start, but no less than two such sweeps from |b|^2 would leave.
template <int R, int Q>
__global__ void k_cg_start(const double* part, int G, const double* tol, double* bb, double* stop, double* scale,
                           int* ctl) {
    int* active = ctl + kCtlActive;
    __shared__ int clear[R];
    const int r = threadIdx.x >> 5;
    const double t = total_of(part, G, Q * R, r);
    const double rr = Q == 1 ? t : total_of(part, G, Q * R, (Q - 1) * R + r);
    if ((threadIdx.x & 31) == 0) {
        bb[r] = t;
        const int e = rr > 0.0 && isfinite(rr) ? ilogb(rr) >> 1 : 0;
        scale[r] = e >= -20 && e < 60 ? 1.0 : scalbn(1.0, -e);
        stop[r] = tol[1] > 0.0 ? fmax(tol[1] * rr, tol[1] * tol[1] * t) : tol[0] * t;
        active[r] = t > 0.0 && rr > tol[0] * t ? 1 : 0;
        clear[r] = t == 0.0 && rr > 0.0 ? 1 : 0;
        if (!isfinite(t))
            atomicExch(ctl, int(QPAT_EINVAL));
        else if (!isfinite(rr))
            atomicExch(ctl, int(QPAT_EBREAKDOWN));
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int c = 0, z = 0, s = 0;
        for (int q = 0; q < R; ++q) {
            c += active[q];
            z += clear[q];
            s += scale[q] != 1.0;
        }
        ctl[1] = c;
        ctl[2] = 0;
        ctl[3] = 1;
        ctl[5] = z;
        ctl[6] = s;
    }
}

// q = A p, p.q; the last block forms alpha = r.z / p.q on the running right-hand sides (0 on the others)
template <int R, int NV, int GW>
__global__ void __launch_bounds__(256) k_cg_apply(SellDev A, const double* __restrict__ v0, const double* __restrict__ v1,
                                                  const double* __restrict__ p, double* __restrict__ q, double* part,
                                                  unsigned* count, const double* rz, double* alpha, int* ctl) {
    const RowMap<double, R, GW, 1> m;
    constexpr int C = RowMap<double, R, GW, 1>::C;
    __shared__ double tot[R];
    double dot[C];
#pragma unroll
    for (int r = 0; r < C; ++r) dot[r] = 0.0;
    for (int64_t i0 = int64_t(blockIdx.x) * m.RPB; i0 < A.n; i0 += int64_t(gridDim.x) * m.RPB) {
        const int64_t i = i0 + m.slot;
        double acc[C];
        row_part<double, R, NV>(A, v0, v1, p, i, m.c0, m.g, GW, i < A.n, acc);
        m.combine(acc);
        if (i < A.n && m.g == 0) {
            double pv[C];
            ldR<double, C>(p + i * R + m.c0, pv);
#pragma unroll
            for (int r = 0; r < C; ++r) dot[r] = fma(pv[r], acc[r], dot[r]);
            stR<double, C>(q + i * R + m.c0, acc);
        }
    }
    m.template block_totals<1>(dot, part);
    if (!last_block_totals<R>(part, count, tot)) return;
    if (threadIdx.x < R) {
        const int* active = ctl + kCtlActive;
        const int r = threadIdx.x;
        const double pq = tot[r];
        double a = 0.0;
        if (active[r]) {
            if (!(pq > 0.0) || !isfinite(pq) || !isfinite(rz[r]))
                atomicExch(ctl, int(QPAT_EBREAKDOWN));
            else
                a = rz[r] / pq;
        }
        alpha[r] = a;
    }
}

// beta = r.z / (r.z)_old from the totals of r.z; FLEX: z.(r - r_old) / (r.z)_old with r - r_old = -alpha q (the form
// that tolerates a preconditioner that varies slightly between applications), tot[R ..] = q.z.  0 before the first
// direction (ctl[3], cleared here).  rz <- r.z.  By the threads of one block.
template <int R, bool FLEX>
__device__ __forceinline__ void cg_beta(const double* tot, double* rz, const double* alpha, double* beta, int* ctl) {
    const int first = ctl[3];
    if (threadIdx.x < R) {
        const int* active = ctl + kCtlActive;
        const int r = threadIdx.x;
        const double t = tot[r];
        double b = 0.0;
        if (!first && active[r]) b = (FLEX ? -alpha[r] * tot[R + r] : t) / rz[r];
        if (active[r] && (!isfinite(t) || !(t > 0.0))) atomicExch(ctl, int(QPAT_EBREAKDOWN));
        beta[r] = b;
        rz[r] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) ctl[3] = 0;
}

// The fine level's MODE 2 of k_level with z in FP64, the dots r.z (FLEX, the FP32 cycle: and q.z) and, in the last
// block, beta.
template <typename T, int R, int NV, int GW>
__global__ void __launch_bounds__(256) k_top(SellDev P2, const T* __restrict__ v0, const T* __restrict__ v1,
                                             const T* __restrict__ e, const T* __restrict__ wd, const T* __restrict__ b,
                                             const T* __restrict__ res, const double* __restrict__ rr,
                                             const double* __restrict__ q, double* __restrict__ z, double* part,
                                             unsigned* count, double* rz, const double* alpha, double* beta, int* ctl) {
    constexpr bool FLEX = !std::is_same<T, double>::value;
    constexpr int NQ = FLEX ? 2 : 1;
    const RowMap<T, R, GW, 1> m;
    constexpr int C = RowMap<T, R, GW, 1>::C;
    __shared__ double tot[NQ * R];
    double dot[NQ * C];
#pragma unroll
    for (int r = 0; r < NQ * C; ++r) dot[r] = 0.0;
    for (int64_t i0 = int64_t(blockIdx.x) * m.RPB; i0 < P2.n; i0 += int64_t(gridDim.x) * m.RPB) {
        const int64_t i = i0 + m.slot;
        T acc[C];
        row_part<T, R, NV>(P2, v0, v1, e, i, m.c0, m.g, GW, i < P2.n, acc);
        m.combine(acc);
        if (i < P2.n && m.g == 0) {
            const int64_t o = i * R + m.c0;
            T bv[C], rv[C];
            ldR<T, C>(b + o, bv);
            ldR<T, C>(res + o, rv);
            double zv[C], rd[C];
#pragma unroll
            for (int r = 0; r < C; ++r) {
                zv[r] = double(fma(wd[i * NV + (NV == 2 ? m.c0 + r : 0)], bv[r] + rv[r], acc[r]));
                if constexpr (!FLEX) rd[r] = bv[r];
            }
            if constexpr (FLEX) ldR<double, C>(rr + o, rd);
#pragma unroll
            for (int r = 0; r < C; ++r) dot[r] = fma(rd[r], zv[r], dot[r]);
            if constexpr (FLEX) {
                ldR<double, C>(q + o, rd);
#pragma unroll
                for (int r = 0; r < C; ++r) dot[C + r] = fma(rd[r], zv[r], dot[C + r]);
            }
            stR<double, C>(z + o, zv);
        }
    }
    m.template block_totals<NQ>(dot, part);
    if (last_block_totals<NQ * R>(part, count, tot)) cg_beta<R, FLEX>(tot, rz, alpha, beta, ctl);
}

// The vector passes: thread per two right-hand sides of a node (16-byte accesses; the same right-hand sides in every
// step of the grid).  Bound by HBM.
template <int R>
using FlatMap = RowMap<double, R, 1, 1>;
#define FOR_FLAT(n, R)                                                                                  \
    for (int64_t o = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) * C; o < (n) * (R);               \
         o += int64_t(gridDim.x) * blockDim.x * C)

// r.z (FLEX: and q.z) and, in the last block, beta, where no fused kernel has formed them
template <int R, bool FLEX>
__global__ void __launch_bounds__(256) k_cg_dots(int64_t n, const double* __restrict__ r, const double* __restrict__ z,
                                                 const double* __restrict__ qv, double* part, unsigned* count, double* rz,
                                                 const double* alpha, double* beta, int* ctl) {
    constexpr int C = FlatMap<R>::C, NQ = FLEX ? 2 : 1;
    const FlatMap<R> m;
    __shared__ double tot[NQ * R];
    double dot[NQ * C];
#pragma unroll
    for (int t = 0; t < NQ * C; ++t) dot[t] = 0.0;
    FOR_FLAT(n, R) {
        double a[C], zv[C];
        ldR<double, C>(r + o, a);
        ldR<double, C>(z + o, zv);
#pragma unroll
        for (int t = 0; t < C; ++t) dot[t] = fma(a[t], zv[t], dot[t]);
        if constexpr (FLEX) {
            ldR<double, C>(qv + o, a);
#pragma unroll
            for (int t = 0; t < C; ++t) dot[C + t] = fma(a[t], zv[t], dot[C + t]);
        }
    }
    m.template block_totals<NQ>(dot, part);
    if (last_block_totals<NQ * R>(part, count, tot)) cg_beta<R, FLEX>(tot, rz, alpha, beta, ctl);
}

// p = z + beta p
template <int R>
__global__ void __launch_bounds__(256) k_cg_dir(int64_t n, const double* beta, const double* __restrict__ z,
                                                double* __restrict__ p) {
    constexpr int C = FlatMap<R>::C;
    const FlatMap<R> m;
    double be[C];
#pragma unroll
    for (int t = 0; t < C; ++t) be[t] = beta[m.c0 + t];
    FOR_FLAT(n, R) {
        double zv[C], pv[C];
        ldR<double, C>(z + o, zv);
        ldR<double, C>(p + o, pv);
#pragma unroll
        for (int t = 0; t < C; ++t) pv[t] = fma(be[t], pv[t], zv[t]);
        stR<double, C>(p + o, pv);
    }
}

// x += alpha p, r -= alpha q (b32: and the FP32 copy of r, SCALED: of scale r;
// a multiplication by 1 for every entry would cost a fifth of this kernel), r.r.  The last
// block checks: a right-hand side stops once |r|^2 <= stop; one more
// iteration is done.  Inside a graph (use_graph) it also sets the loop's
// condition: go on while some right-hand side runs, the status is clean and
// the cap is not reached (reaching it with a running right-hand side is
// QPAT_ENOCONV).
template <int R, bool SCALED>
__global__ void __launch_bounds__(256) k_cg_update(int64_t n, const double* alpha, const double* __restrict__ p,
                                                   const double* __restrict__ q, double* __restrict__ x,
                                                   double* __restrict__ r, const double* scale,
                                                   float* __restrict__ b32, double* part, unsigned* count,
                                                   const double* stop, double* rr, int* ctl,
                                                   cudaGraphConditionalHandle cond, int use_graph) {
    constexpr int C = FlatMap<R>::C;
    const FlatMap<R> m;
    __shared__ double tot[R];
    double al[C], sc[C], dot[C];
#pragma unroll
    for (int t = 0; t < C; ++t) {
        al[t] = alpha[m.c0 + t];
        if (SCALED) sc[t] = scale[m.c0 + t];
        dot[t] = 0.0;
    }
    FOR_FLAT(n, R) {
        double pv[C], qv[C], xv[C], rv[C];
        ldR<double, C>(p + o, pv);
        ldR<double, C>(q + o, qv);
        ldR<double, C>(x + o, xv);
        ldR<double, C>(r + o, rv);
#pragma unroll
        for (int t = 0; t < C; ++t) {
            xv[t] = fma(al[t], pv[t], xv[t]);
            rv[t] = fma(-al[t], qv[t], rv[t]);
            dot[t] = fma(rv[t], rv[t], dot[t]);
        }
        stR<double, C>(x + o, xv);
        stR<double, C>(r + o, rv);
        if (b32)
#pragma unroll
            for (int t = 0; t < C; ++t) b32[o + t] = float(SCALED ? sc[t] * rv[t] : rv[t]);
    }
    m.template block_totals<1>(dot, part);
    if (!last_block_totals<R>(part, count, tot)) return;
    int* active = ctl + kCtlActive;
    if (threadIdx.x < R) {
        const double t = tot[threadIdx.x];
        rr[threadIdx.x] = t;
        if (!isfinite(t)) atomicExch(ctl, int(QPAT_EBREAKDOWN));
        if (active[threadIdx.x] && t <= stop[threadIdx.x]) active[threadIdx.x] = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int c = 0;
        for (int k = 0; k < R; ++k) c += active[k];
        ctl[1] = c;
        const int it = ++ctl[2];
        if (c > 0 && it >= ctl[4] && ctl[0] == QPAT_OK) ctl[0] = QPAT_ENOCONV;
        if (use_graph) cudaGraphSetConditional(cond, (c > 0 && ctl[0] == QPAT_OK) ? 1u : 0u);
    }
}

// b32 = scale r in FP32, N x R
template <int R>
__global__ void __launch_bounds__(256) k_cg_cast(int64_t n, const double* scale, const double* r, float* b32) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n * R; i += int64_t(gridDim.x) * blockDim.x)
        b32[i] = float(scale[i % R] * r[i]);
}
__global__ void k_f2d_vec(int64_t n, const float* in, double* out) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
        out[i] = double(in[i]);
}

}  // namespace

// ---------------------------------------------------------------- host side

// Device memory that the multigrid solver of a mesh holds, and the most that
// it may hold (0: no limit).
struct MemLedger {
    size_t used = 0, limit = 0;
    bool refused = false;  // an allocation failed
};

// A set of device allocations that is released as a whole.  Every part of the
// state below is allocated into a local one and put in its place only when all
// of it is there, so that a failed allocation leaves nothing half-built.
class DevMem {
  public:
    explicit DevMem(MemLedger* l) : ledger_(l) {}
    DevMem(DevMem&& o) noexcept : ledger_(o.ledger_) { list_.swap(o.list_); }
    DevMem& operator=(DevMem&& o) noexcept {
        std::swap(ledger_, o.ledger_);
        list_.swap(o.list_);
        return *this;
    }
    ~DevMem() {
        for (const auto& a : list_) {
            cudaFree(a.first);
            ledger_->used -= a.second;
        }
    }
    // count values of T; nothing (and e unchanged) once e reports a failure
    template <typename T>
    T* get(size_t count, cudaError_t& e) {
        if (e != cudaSuccess) return nullptr;
        const size_t bytes = std::max<size_t>(count, 1) * sizeof(T);
        if (ledger_->limit && ledger_->used + bytes > ledger_->limit) {
            e = cudaErrorMemoryAllocation;
            ledger_->refused = true;
            return nullptr;
        }
        list_.emplace_back(nullptr, 0);
        void* p = nullptr;
        if ((e = cudaMalloc(&p, bytes)) != cudaSuccess) {
            list_.pop_back();
            ledger_->refused = e == cudaErrorMemoryAllocation;
            return nullptr;
        }
        list_.back() = {p, bytes};
        ledger_->used += bytes;
        return static_cast<T*>(p);
    }
    template <typename T>
    const T* put(const std::vector<T>& h, cudaError_t& e) {
        T* d = get<T>(h.size(), e);
        if (e == cudaSuccess && !h.empty()) e = cudaMemcpy(d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice);
        return d;
    }

  private:
    MemLedger* ledger_;
    std::vector<std::pair<void*, size_t>> list_;
};

struct AmgHierDev {
    explicit AmgHierDev(MemLedger* l) : mem(l) {}
    bool ready = false;
    bool used[2] = {false, false};  // a K (M_delta) solve has run on it
    std::string error;              // non-empty: this mesh has no hierarchy
    std::vector<LevelDev> lv;
    SellDev K;                      // the full pattern of K (the products of its CG)
    DevMem mem;
};

// One CG iteration captured once as the body of a graph "while" node, per
// operator values, right-hand-side count and cycle settings; the check
// kernel of the body sets the loop condition on the device.
struct AmgGraph {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    int body_kernels = 0;
    AmgGraph() = default;
    AmgGraph(AmgGraph&& o) noexcept : graph(o.graph), exec(o.exec), body_kernels(o.body_kernels) {
        o.graph = nullptr;
        o.exec = nullptr;
    }
    AmgGraph& operator=(AmgGraph&&) = delete;
    ~AmgGraph() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
    }
};

struct AmgValues {
    explicit AmgValues(MemLedger* l) : mem(l) {}
    uint64_t stamp = 0;
    bool valid = false;
    bool has32 = false;
    double ratio = 0.0;     // mg_ratio of S, wd and P2
    std::vector<std::array<double*, 2>> A, P, R;  // A[0]: K taken into the fine pattern (M_delta: its own values)
    std::vector<std::array<double*, 2>> S, P2;    // degree-1 cycle: A diag(wd), P - wd A P
    std::vector<double*> AP, dinv, wd;
    double* hi = nullptr;   // 2 per level
    double* inv = nullptr;  // coarsest inverse, NV x n x n
    std::vector<std::array<float*, 2>> A32, P32, R32, S32, P232;
    std::vector<float*> dinv32, wd32;
    float* inv32 = nullptr;
    std::map<std::string, AmgGraph> graphs;  // iterations captured on these values
    DevMem mem;
};

struct AmgVecs {
    explicit AmgVecs(MemLedger* l) : mem(l) {}
    std::vector<void*> b, xa, xb, d, r;  // nullptr where the form of the cycle has no use for one
    DevMem mem;
};

struct AmgCg {
    explicit AmgCg(MemLedger* l) : mem(l) {}
    double *x = nullptr, *r = nullptr, *p = nullptr, *q = nullptr, *z = nullptr, *part = nullptr;
    double *bb = nullptr, *rz = nullptr, *alpha = nullptr, *beta = nullptr, *rr = nullptr, *scale = nullptr;
    double *stop = nullptr, *tol = nullptr;
    int* ctl = nullptr;  // control words (see k_cg_start)
    unsigned* count = nullptr;  // blocks that have finished (see last_block_totals)
    DevMem mem;
};

struct AmgState {
    MemLedger ledger;
    AmgHierDev hier{&ledger};     // on the prior's pattern, for K and M_delta
    std::map<std::array<int, 3>, AmgVecs> vecs;   // (R, FP32 cycle, degree 1)
    std::map<int, AmgCg> cg;                       // R
    std::map<const void*, AmgValues> vals;         // per operator; their graphs work on vecs and cg too
    cudaStream_t capture = nullptr;                // a non-default stream to capture on
};

namespace {

SellDev upload_sell(DevMem& mem, const SellPattern& S, cudaError_t& e) {
    SellDev d;
    d.n = S.n;
    d.ptr = mem.put(S.ptr, e);
    d.col = mem.put(S.col, e);
    d.len = mem.put(S.len, e);
    d.entries = S.entries();
    d.maxlen = S.maxlen;
    d.rowmajor = S.rowmajor ? 1 : 0;
    return d;
}

// Grid of a kernel that strides over its work: every resident block of the
// device (a grid between one and two waves would leave half of it idle at the
// end), at most `most`.
template <typename K>
int full_grid(K kernel, int most) {
    int dev = 0, nsm = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, 256, 0) != cudaSuccess || nsm * per < 1)
        return most;
    return std::min(most, nsm * per);
}

inline int blocks_of(int64_t n, int per = 256) { return int(std::max<int64_t>(1, (n + per - 1) / per)); }

int build_hier(qpat_mesh_s* M, AmgHierDev& H, MemLedger& ledger) {
    AmgPlan plan;
    try {
        const SellPattern fine = amg_fine_pattern(M->h);
        plan = amg_build_plan(fine, amg_fine_graph(M->h, fine));
    } catch (const std::exception& ex) {  // host memory
        ledger.refused = true;
        return fail(QPAT_ENOMEM, std::string("multigrid plan: ") + ex.what());
    }
    if (!plan.error.empty()) {
        H.error = plan.error;
        return fail(QPAT_EINVAL, plan.error);
    }
    cudaError_t e = cudaSuccess;
    for (const AmgLevelPlan& L : plan.levels) {
        LevelDev d;
        d.A = upload_sell(H.mem, L.A, e);
        d.diag = H.mem.put(L.diag, e);
        d.nc = L.nc;
        if (L.nc > 0) {
            d.P = upload_sell(H.mem, L.P, e);
            d.a2p = H.mem.put(L.a2p, e);
            d.pself = H.mem.put(L.pself, e);
            d.ap_ptr = H.mem.put(L.ap_ptr, e);
            d.ap_col = H.mem.put(L.ap_col, e);
            d.ap_sptr = H.mem.put(L.ap_sptr, e);
            d.ap_slot = H.mem.put(L.ap_slot, e);
            d.ap_nnz = int64_t(L.ap_col.size());
            for (size_t i = 0; i + 1 < L.ap_ptr.size(); ++i)
                d.ap_maxlen = std::max<int>(d.ap_maxlen, int(L.ap_ptr[i + 1] - L.ap_ptr[i]));
            d.R = upload_sell(H.mem, L.R, e);
            d.r_src = H.mem.put(L.r_src, e);
            d.g_ptr = H.mem.put(L.g_ptr, e);
            d.g_slot = H.mem.put(L.g_slot, e);
        }
        H.lv.push_back(d);
    }
    const std::vector<uint16_t> len(M->h.sell_len.begin(), M->h.sell_len.end());
    H.K.n = M->h.N;
    H.K.ptr = M->d.sell_ptr;
    H.K.col = M->el.ent_col;
    H.K.len = H.mem.put(len, e);
    H.K.entries = M->d.sell_entries;
    H.K.maxlen = M->d.sell_wmax;
    if (e != cudaSuccess) return cuda_fail(e, "multigrid upload");
    H.ready = true;
    return QPAT_OK;
}

template <int NV>
cudaError_t numeric_levels(const qpat_mesh_s* M, const AmgHierDev& H, const OpState& st, AmgValues& V, double ratio,
                           cudaStream_t s) {
    const int L = int(H.lv.size());
    cudaError_t e = cudaMemsetAsync(V.hi, 0, sizeof(double) * 2 * L, s);
    if (e != cudaSuccess) return e;
    if (NV == 1) {
        note_launch(1);
        k_lump<<<blocks_of(H.K.n), 256, 0, s>>>(H.K, M->el.ent_edge, M->el.in_prior, H.lv[0].A, H.lv[0].diag, st.v64[0],
                                                V.A[0][0]);
    }
    for (int l = 0; l < L; ++l) {
        const LevelDev& d = H.lv[size_t(l)];
        const double *a0 = V.A[size_t(l)][0], *a1 = V.A[size_t(l)][1];
        double* hi = V.hi + 2 * l;
        note_launch(1);
        k_dinv_hi<NV><<<blocks_of(d.A.n), 256, 0, s>>>(d.A, d.diag, a0, a1, V.dinv[size_t(l)], hi);
        if (l + 1 == L) break;
        const auto& Pv = V.P[size_t(l)];
        const auto& Rv = V.R[size_t(l)];
        if (V.wd[size_t(l)]) {
            note_launch(2);
            k_weights<NV><<<blocks_of(d.A.n * NV), 256, 0, s>>>(d.A.n, V.dinv[size_t(l)], hi, ratio, V.wd[size_t(l)]);
            k_scaled<NV><<<blocks_of(d.A.entries), 256, 0, s>>>(d.A.entries, d.A.col, V.wd[size_t(l)], a0, a1,
                                                                V.S[size_t(l)][0], V.S[size_t(l)][1]);
        }
        note_launch(4);
        k_prolong<NV><<<blocks_of(d.A.n), 256, 0, s>>>(d.A, d.P, d.diag, d.a2p, d.pself, a0, a1, Pv[0], Pv[1]);
        k_rvals<NV><<<blocks_of(d.R.entries), 256, 0, s>>>(d.R.entries, d.r_src, Pv[0], Pv[1], Rv[0], Rv[1]);
        {
            int wpb = 8;  // warps per block, kApLanes lanes per row
            const int rpw = 32 / kApLanes;
            while (wpb > 1 && size_t(wpb * rpw) * size_t(d.ap_maxlen) * sizeof(double) > 96 * 1024) wpb >>= 1;
            const size_t smem = size_t(wpb * rpw) * size_t(d.ap_maxlen) * sizeof(double);
            if ((e = allow_smem(reinterpret_cast<const void*>(&k_ap<NV>), smem)) != cudaSuccess) return e;
            k_ap<NV><<<blocks_of(d.A.n * NV, wpb * rpw), 32 * wpb, smem, s>>>(
                d.A, d.P, d.diag, d.ap_ptr, d.ap_sptr, d.ap_slot, d.ap_nnz, d.ap_maxlen, a0, a1, Pv[0], Pv[1],
                V.wd[size_t(l)], V.AP[size_t(l)], V.P2[size_t(l)][0]);
        }
        const LevelDev& c = H.lv[size_t(l + 1)];
        int wpb = 8;
        while (wpb > 1 && size_t(wpb) * size_t(c.A.maxlen) * sizeof(double) > 96 * 1024) wpb >>= 1;
        const size_t smem = size_t(wpb) * size_t(c.A.maxlen) * sizeof(double);
        if ((e = allow_smem(reinterpret_cast<const void*>(&k_galerkin<NV>), smem)) != cudaSuccess) return e;
        k_galerkin<NV><<<blocks_of(c.A.n * NV, wpb), 32 * wpb, smem, s>>>(
            d.R, c.A, d.r_src, d.ap_ptr, d.g_ptr, d.g_slot, d.ap_nnz, Pv[0], Pv[1], V.AP[size_t(l)],
            V.A[size_t(l + 1)][0], V.A[size_t(l + 1)][1]);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    const LevelDev& c = H.lv[size_t(L - 1)];
    const int n = int(c.A.n);
    const size_t smem = size_t(n) * size_t(n) * sizeof(double);
    if ((e = allow_smem(reinterpret_cast<const void*>(&k_dense_inv<NV>), smem)) != cudaSuccess) return e;
    const double *a0 = V.A[size_t(L - 1)][0], *a1 = V.A[size_t(L - 1)][1];
    note_launch(1);
    k_dense_inv<NV><<<NV, 1024, smem, s>>>(c.A, a0, a1, V.inv);
    return cudaGetLastError();
}

cudaError_t cast_to_f32(const double* in, float* out, int64_t n, cudaStream_t s) {
    note_launch(1);
    k_d2f<<<blocks_of(n), 256, 0, s>>>(n, in, out);
    return cudaGetLastError();
}

// Values of the hierarchy for the operator st (allocated once per operator
// buffer, recomputed when st was prepared again or the cycle's form changed).
// fast: S, wd and P2 of the fine level too (degree 1; the coarser levels always
// have theirs).  After a failure V is incomplete and must be dropped.
int numeric(qpat_mesh_s* M, const AmgHierDev& H, const OpState& st, AmgValues& V, bool fast, double ratio, bool need32,
            cudaStream_t s) {
    const int L = int(H.lv.size());
    const int NV = st.nv;
    cudaError_t e = cudaSuccess;
    auto set = [&](auto& list) { list.assign(size_t(L), {nullptr, nullptr}); };
    // room for S, P2 and wd of a level with a transfer, and for their FP32 copies
    auto smoothing = [&](int l) {
        if (l + 1 == L) return;
        const LevelDev& d = H.lv[size_t(l)];
        for (int v = 0; v < NV; ++v) V.S[size_t(l)][size_t(v)] = V.mem.get<double>(size_t(d.A.entries), e);
        double* p2 = V.mem.get<double>(size_t(d.ap_nnz) * NV, e);
        V.P2[size_t(l)] = {p2, NV == 2 && p2 ? p2 + d.ap_nnz : nullptr};
        V.wd[size_t(l)] = V.mem.get<double>(size_t(d.A.n) * NV, e);
    };
    auto smoothing32 = [&](int l) {
        if (l + 1 == L) return;
        const LevelDev& d = H.lv[size_t(l)];
        for (int v = 0; v < NV; ++v) {
            V.S32[size_t(l)][size_t(v)] = V.mem.get<float>(size_t(d.A.entries), e);
            V.P232[size_t(l)][size_t(v)] = V.mem.get<float>(size_t(d.ap_nnz), e);
        }
        V.wd32[size_t(l)] = V.mem.get<float>(size_t(d.A.n) * NV, e);
    };
    if (V.A.empty()) {
        set(V.A);
        set(V.P);
        set(V.R);
        set(V.S);
        set(V.P2);
        V.wd.assign(size_t(L), nullptr);
        V.AP.assign(size_t(L), nullptr);
        V.dinv.assign(size_t(L), nullptr);
        for (int l = 0; l < L; ++l) {
            const LevelDev& d = H.lv[size_t(l)];
            for (int v = 0; v < NV; ++v) {
                V.A[size_t(l)][size_t(v)] =
                    l == 0 && NV == 2 ? st.v64[v] : V.mem.get<double>(size_t(d.A.entries), e);
                if (l + 1 < L) {
                    V.P[size_t(l)][size_t(v)] = V.mem.get<double>(size_t(d.P.entries), e);
                    V.R[size_t(l)][size_t(v)] = V.mem.get<double>(size_t(d.R.entries), e);
                }
            }
            if (l + 1 < L) V.AP[size_t(l)] = V.mem.get<double>(size_t(d.ap_nnz) * NV, e);
            V.dinv[size_t(l)] = V.mem.get<double>(size_t(d.A.n) * NV, e);
            if (l > 0) smoothing(l);
        }
        V.hi = V.mem.get<double>(size_t(2 * L), e);
        const int64_t nco = H.lv.back().A.n;
        V.inv = V.mem.get<double>(size_t(NV * nco * nco), e);
        if (e != cudaSuccess) return cuda_fail(e, "multigrid workspace");
        // padding entries are never written: keep them 0
        for (int l = 0; l < L && e == cudaSuccess; ++l)
            for (int v = 0; v < NV && e == cudaSuccess; ++v) {
                const LevelDev& d = H.lv[size_t(l)];
                if (l + 1 < L) e = cudaMemsetAsync(V.P[size_t(l)][size_t(v)], 0, sizeof(double) * d.P.entries, s);
                if (e == cudaSuccess && !(l == 0 && NV == 2))
                    e = cudaMemsetAsync(V.A[size_t(l)][size_t(v)], 0, sizeof(double) * d.A.entries, s);
            }
        if (e != cudaSuccess) return cuda_fail(e, "multigrid memset");
    }
    if (NV == 2) V.A[0] = {st.v64[0], st.v64[1]};
    if (fast && L > 1 && !V.wd[0]) {
        smoothing(0);
        if (e != cudaSuccess) return cuda_fail(e, "multigrid workspace");
        V.valid = false;
    }
    if (need32 && !V.has32) {
        set(V.A32);
        set(V.P32);
        set(V.R32);
        set(V.S32);
        set(V.P232);
        V.wd32.assign(size_t(L), nullptr);
        V.dinv32.assign(size_t(L), nullptr);
        for (int l = 0; l < L; ++l) {
            const LevelDev& d = H.lv[size_t(l)];
            for (int v = 0; v < NV; ++v) {
                V.A32[size_t(l)][size_t(v)] = V.mem.get<float>(size_t(d.A.entries), e);
                if (l + 1 < L) {
                    V.P32[size_t(l)][size_t(v)] = V.mem.get<float>(size_t(d.P.entries), e);
                    V.R32[size_t(l)][size_t(v)] = V.mem.get<float>(size_t(d.R.entries), e);
                }
            }
            V.dinv32[size_t(l)] = V.mem.get<float>(size_t(d.A.n) * NV, e);
            if (l > 0) smoothing32(l);
        }
        const int64_t nco = H.lv.back().A.n;
        V.inv32 = V.mem.get<float>(size_t(NV * nco * nco), e);
        if (e != cudaSuccess) return cuda_fail(e, "multigrid workspace");
        V.has32 = true;
        V.valid = false;
    }
    if (fast && L > 1 && V.has32 && !V.wd32[0]) {
        smoothing32(0);
        if (e != cudaSuccess) return cuda_fail(e, "multigrid workspace");
        V.valid = false;
    }
    if (V.valid && V.stamp == st.stamp && V.ratio == ratio) return QPAT_OK;
    V.ratio = ratio;
    e = NV == 1 ? numeric_levels<1>(M, H, st, V, ratio, s) : numeric_levels<2>(M, H, st, V, ratio, s);
    if (e != cudaSuccess) return cuda_fail(e, "multigrid set-up");
    if (V.has32) {
        auto cast = [&](const double* in, float* out, int64_t n) {
            if (e == cudaSuccess && out) e = cast_to_f32(in, out, n, s);
        };
        for (int l = 0; l < L; ++l) {
            const LevelDev& d = H.lv[size_t(l)];
            for (int v = 0; v < NV; ++v) {
                const size_t i = size_t(l), j = size_t(v);
                cast(V.A[i][j], V.A32[i][j], d.A.entries);
                cast(V.P[i][j], V.P32[i][j], d.P.entries);
                cast(V.R[i][j], V.R32[i][j], d.R.entries);
                cast(V.S[i][j], V.S32[i][j], d.A.entries);
                cast(V.P2[i][j], V.P232[i][j], d.ap_nnz);
            }
            cast(V.dinv[size_t(l)], V.dinv32[size_t(l)], d.A.n * NV);
            cast(V.wd[size_t(l)], V.wd32[size_t(l)], d.A.n * NV);
        }
        const int64_t nco = H.lv.back().A.n;
        cast(V.inv, V.inv32, NV * nco * nco);
        if (e != cudaSuccess) return cuda_fail(e, "multigrid set-up");
    }
    V.stamp = st.stamp;
    V.valid = true;
    return QPAT_OK;
}

}  // namespace

namespace {

// Optional CUDA-event timing of the fine level's smoothing products (degree 1:
// its residual kernel; higher degrees: the smoothing steps); the events of one cycle are read after
// the next stream synchronisation of the CG loop.
struct FineTimer {
    bool on = false;
    cudaStream_t s = nullptr;
    std::vector<cudaEvent_t> ev;
    int used = 0;
    double ms = 0.0;
    int64_t launches = 0;
    void before() {
        if (!on) return;
        if (used + 2 > int(ev.size())) {
            cudaEvent_t a, b;
            cudaEventCreate(&a);
            cudaEventCreate(&b);
            ev.push_back(a);
            ev.push_back(b);
        }
        cudaEventRecord(ev[size_t(used)], s);
    }
    void after() {
        if (!on) return;
        cudaEventRecord(ev[size_t(used + 1)], s);
        used += 2;
    }
    void collect() {  // after a synchronisation of the stream
        for (int k = 0; k < used; k += 2) {
            float t = 0.f;
            if (cudaEventElapsedTime(&t, ev[size_t(k)], ev[size_t(k + 1)]) == cudaSuccess) ms += t;
            ++launches;
        }
        used = 0;
    }
    ~FineTimer() {
        for (cudaEvent_t e : ev) cudaEventDestroy(e);
    }
};

// The degree-1 cycle (see k_level): per level the residual, its restriction
// and, on the way back, prolongation with the post-smoothing step; the fine
// level's last kernel (k_top) belongs to the CG.
template <typename T, int R, int NV>
struct FastCycle {
    const AmgHierDev& H;
    const AmgValues& V;
    AmgVecs& W;
    cudaStream_t s;
    FineTimer* timer = nullptr;

    static constexpr bool F64 = std::is_same<T, double>::value;
    static constexpr int LPR = R / kLaneRhs<T, R>, GX = 32 / LPR, GM = GX < 8 ? GX : 8;
    const T* val(const std::vector<std::array<double*, 2>>& a, const std::vector<std::array<float*, 2>>& b, int l,
                 int v) const {
        if constexpr (F64) return a[size_t(l)][size_t(v)];
        else return b[size_t(l)][size_t(v)];
    }
    const T* wd(int l) const {
        if constexpr (F64) return V.wd[size_t(l)];
        else return V.wd32[size_t(l)];
    }
    SellDev p2(int l) const {
        const LevelDev& d = H.lv[size_t(l)];
        SellDev p;
        p.n = d.A.n;
        p.ptr = d.ap_ptr;
        p.col = d.ap_col;
        p.entries = d.ap_nnz;
        p.maxlen = d.ap_maxlen;
        p.rowmajor = 1;
        return p;
    }
    // Groups that share a row's entries.  FP64 issue is the scarce resource
    // (16 cycles of an SM for each warp instruction, idle lanes included), so
    // rows are shared by several groups only as far as the GPU would not be
    // filled otherwise, or two where rows of one lane lie row by row in memory
    // (coalescing); FP32 shares row-major rows by up to 8.  Long rows of the
    // smallest levels get a block each.
    template <int MODE>
    void launch(const SellDev& A, const T* v0, const T* v1, const T* x, const T* w, const T* b, const T* res, T* y) {
        note_launch(1);
        const double avg = double(A.entries) / double(std::max<int64_t>(1, A.n));
        const int64_t fill = 152 * 1024, threads = A.n * LPR;
        auto go = [&](auto gw, auto wpr) {
            using Map = RowMap<T, R, decltype(gw)::value, decltype(wpr)::value>;
            k_level<T, R, NV, MODE, decltype(gw)::value, decltype(wpr)::value>
                <<<blocks_of(A.n, Map::RPB), 256, 0, s>>>(A, v0, v1, x, w, b, res, y);
        };
        using std::integral_constant;
        constexpr int GS = F64 ? (LPR == 1 ? 2 : 1) : GM;
        if (A.n <= 1024 && avg >= 8 * GX)
            go(integral_constant<int, GX>(), integral_constant<int, 8>());
        else if (threads * GM < fill && avg >= 2 * GX)
            go(integral_constant<int, GX>(), integral_constant<int, 1>());
        else if (threads * GS < fill)
            go(integral_constant<int, GM>(), integral_constant<int, 1>());
        else if (A.rowmajor)
            go(integral_constant<int, GS>(), integral_constant<int, 1>());
        else
            go(integral_constant<int, 1>(), integral_constant<int, 1>());
    }

    // From the fine level (from = 0, right-hand side b0): leaves its residual in W.r[0] and returns the correction on
    // level 1.  From level 1 (right-hand side in W.b[1]): returns the cycle's result there.
    const T* run(const T* b0, int from) {
        const int L = int(H.lv.size());
        for (int l = from; l + 1 < L; ++l) {
            const LevelDev& d = H.lv[size_t(l)];
            const T* b = l == 0 ? b0 : static_cast<const T*>(W.b[size_t(l)]);
            T* res = static_cast<T*>(W.r[size_t(l)]);
            if (l == 0 && timer) timer->before();
            launch<0>(d.A, val(V.S, V.S32, l, 0), val(V.S, V.S32, l, 1), b, nullptr, b, nullptr, res);
            if (l == 0 && timer) timer->after();
            launch<1>(d.R, val(V.R, V.R32, l, 0), val(V.R, V.R32, l, 1), res, nullptr, nullptr, nullptr,
                      static_cast<T*>(W.b[size_t(l + 1)]));
        }
        const T* inv;
        if constexpr (F64) inv = V.inv;
        else inv = V.inv32;
        const int nc = int(H.lv.back().A.n);
        T* x = static_cast<T*>(W.xa[size_t(L - 1)]);
        note_launch(1);
        k_dense_apply<T, R, NV><<<blocks_of(nc * R, 128), 128, 0, s>>>(nc, inv, static_cast<const T*>(W.b[size_t(L - 1)]), x);
        for (int l = L - 2; l >= 1; --l) {
            T* y = static_cast<T*>(W.xa[size_t(l)]);
            launch<2>(p2(l), val(V.P2, V.P232, l, 0), val(V.P2, V.P232, l, 1), x, wd(l), static_cast<const T*>(W.b[size_t(l)]),
                      static_cast<const T*>(W.r[size_t(l)]), y);
            x = y;
        }
        return x;
    }
};

// The cycle with a smoothing polynomial of higher degree on the fine level
// (pre-smoothing from x = 0, residual, restriction, the degree-1 cycle of the
// coarser levels, prolongation, post-smoothing with the same polynomial: B is
// symmetric).  The coarser levels are bound by the number of their kernels: with
// the polynomial there too (7 kernels a level at degree 2, 3 now), K with 4
// right-hand sides on the 33 x 33 x 41 cylinder took 11.4 ms at degree 2, 7.0 now; at
// degree 8 on 40^3 13.5 and 6.2; M_delta on 64^3 at degree 2 16.0 and 8.6.
template <typename T, int R, int NV>
struct PolyCycle {
    const AmgHierDev& H;
    const AmgValues& V;
    AmgVecs& W;
    int deg;
    double ratio;
    cudaStream_t s;
    FineTimer* timer = nullptr;

    static constexpr bool F64 = std::is_same<T, double>::value;
    const T* av(int l, int v) const {
        if constexpr (F64)
            return V.A[size_t(l)][size_t(v)];
        else
            return V.A32[size_t(l)][size_t(v)];
    }
    const T* pv(int l, int v) const {
        if constexpr (F64) return V.P[size_t(l)][size_t(v)];
        else return V.P32[size_t(l)][size_t(v)];
    }
    const T* rv(int l, int v) const {
        if constexpr (F64) return V.R[size_t(l)][size_t(v)];
        else return V.R32[size_t(l)][size_t(v)];
    }
    const T* dinv(int l) const {
        if constexpr (F64) return V.dinv[size_t(l)];
        else return V.dinv32[size_t(l)];
    }
    const T* inv() const {
        if constexpr (F64) return V.inv;
        else return V.inv32;
    }

    const T* run(const T* b) {
        const LevelDev& d = H.lv[0];
        FastCycle<T, R, NV> coarse{H, V, W, s};
        T* x = static_cast<T*>(W.xa[0]);
        T* y = static_cast<T*>(W.xb[0]);
        T* dd = static_cast<T*>(W.d[0]);
        if (H.lv.size() == 1) {
            note_launch(1);
            k_dense_apply<T, R, NV><<<1, 256, 0, s>>>(int(d.A.n), inv(), b, x);
            return x;
        }
        const T *a0 = av(0, 0), *a1 = av(0, 1);
        note_launch(1);
        k_cheb<T, R, NV, true, 1><<<blocks_of(d.A.n, RowMap<T, R, 1, 1>::RPB), 256, 0, s>>>(d.A, a0, a1, dinv(0), V.hi, ratio,
                                                                                       0, nullptr, x, dd, b);
        auto step = [&](int k) {
            if (timer) timer->before();
            note_launch(1);
            auto go = [&](auto gw) {
                constexpr int GW = decltype(gw)::value;
                k_cheb<T, R, NV, false, GW><<<blocks_of(d.A.n, RowMap<T, R, GW, 1>::RPB), 256, 0, s>>>(
                    d.A, a0, a1, dinv(0), V.hi, ratio, k, x, y, dd, b);
            };
            // a row's entries are shared by several groups only where the GPU would not be filled otherwise, in FP64 by two
            // as soon as eight would fill it (see FastCycle::launch)
            constexpr int GM = FastCycle<T, R, NV>::GM;
            const int64_t fill = 152 * 1024, threads = d.A.n * coarse.LPR;
            if (threads * (F64 ? GM : 1) < fill) go(std::integral_constant<int, GM>());
            else if (threads < fill) go(std::integral_constant<int, 2>());
            else go(std::integral_constant<int, 1>());
            if (timer) timer->after();
            std::swap(x, y);
        };
        for (int k = 1; k < deg; ++k) step(k);
        T* res = static_cast<T*>(W.r[0]);
        coarse.template launch<0>(d.A, a0, a1, x, nullptr, b, nullptr, res);
        coarse.template launch<1>(d.R, rv(0, 0), rv(0, 1), res, nullptr, nullptr, nullptr, static_cast<T*>(W.b[1]));
        const T* xc = coarse.run(nullptr, 1);
        coarse.template launch<3>(d.P, pv(0, 0), pv(0, 1), xc, nullptr, x, nullptr, y);
        std::swap(x, y);
        for (int k = 0; k < deg; ++k) step(k);
        return x;
    }
};

// What a solve took: iterations, the sweeps they came in, and whether the
// refinement ended above its target.
struct CgCount {
    int iters = 0, sweeps = 0;
    bool stalled = false;
};

// Conjugate gradients on the fine operator with one V-cycle per iteration
// as the preconditioner; X0 (or 0) to start, each right-hand side stops at
// |r| <= rtol |b| (the recursive residual, as the persistent PCG does).
// After the start, every iteration is
//   z = B r, beta = r.z / (r.z)_old, p = z + beta p, q = A p,
//   alpha = r.z / p.q, x += alpha p, r -= alpha q, check,
// launched from the host one kernel at a time when the fine level is being
// timed, and otherwise replayed from a captured graph whose "while" node runs
// on the device until the check ends it (no host round trip per iteration).
// Both forms launch the same kernels on the same data.
template <int R, int NV>
struct CgSolve {
    qpat_mesh_s* M;
    const OpState& st;
    const SolveOpts& so;
    const AmgHierDev& H;
    AmgValues& V;
    bool f32;
    AmgVecs& W;
    AmgCg& C;
    cudaStream_t s;
    FineTimer* timer;
    int64_t n = 0;
    int G = 0;

    bool fast() const { return so.mg_degree <= 1 && H.lv.size() > 1; }

    // z = B r and beta on stream t; returns the kernels launched beyond those that the cycles count themselves
    template <typename T>
    void precondition(cudaStream_t t) {
        constexpr bool F32 = std::is_same<T, float>::value;
        const T* b;
        if constexpr (F32) b = static_cast<const T*>(W.b[0]);
        else b = C.r;
        note_launch(1);
        if (fast()) {
            FastCycle<T, R, NV> c{H, V, W, t, timer};
            const T* e = c.run(b, 0);
            k_top<T, R, NV, 1><<<full_grid(k_top<T, R, NV, 1>, G), 256, 0, t>>>(c.p2(0), c.val(V.P2, V.P232, 0, 0), c.val(V.P2, V.P232, 0, 1), e, c.wd(0), b,
                                                  static_cast<const T*>(W.r[0]), C.r, C.q, C.z, C.part, C.count, C.rz,
                                                  C.alpha, C.beta, C.ctl);
            return;
        }
        PolyCycle<T, R, NV> c{H, V, W, std::max(1, so.mg_degree), so.mg_ratio, t, timer};
        const T* x = c.run(b);
        const double* z;
        if constexpr (F32) {
            note_launch(1);
            k_f2d_vec<<<G, 256, 0, t>>>(n * R, x, C.z);
            z = C.z;
        } else {
            z = x;
        }
        k_cg_dots<R, F32><<<full_grid(k_cg_dots<R, F32>, G), 256, 0, t>>>(n, C.r, z, C.q, C.part, C.count, C.rz, C.alpha, C.beta, C.ctl);
        zp = z;
    }
    const double* zp = nullptr;  // z where it is not C.z
    bool scaled = false;         // some right-hand side goes into the FP32 cycle with a scale

    // one iteration on stream t; use_graph: the check sets the loop condition
    void body(cudaStream_t t, cudaGraphConditionalHandle cond, int use_graph) {
        zp = C.z;
        if (f32) precondition<float>(t);
        else precondition<double>(t);
        note_launch(3);
        k_cg_dir<R><<<full_grid(k_cg_dir<R>, G), 256, 0, t>>>(n, C.beta, zp, C.p);
        // K's rows hold 15 entries, M_delta's 7: one group per row, the lanes of its right-hand sides side by side
        k_cg_apply<R, NV, 1><<<full_grid(k_cg_apply<R, NV, 1>, G), 256, 0, t>>>(NV == 1 ? H.K : H.lv[0].A, st.v64[0], st.v64[1], C.p, C.q, C.part, C.count,
                                               C.rz, C.alpha, C.ctl);
        float* const b32 = f32 ? static_cast<float*>(W.b[0]) : nullptr;
        auto update = [&](auto kernel) {
            kernel<<<full_grid(kernel, G), 256, 0, t>>>(n, C.alpha, C.p, C.q, C.x, C.r, C.scale, b32, C.part, C.count, C.stop,
                                                        C.rr, C.ctl, cond, use_graph);
        };
        if (scaled) update(k_cg_update<R, true>);
        else update(k_cg_update<R, false>);
    }

    // With so.sweep_rtol the solve is a refinement: sweeps of the iteration,
    // each to sweep_rtol of the residual b - A x that is formed at its start,
    // until that residual meets the target or max_sweeps are over.  The
    // iterates are FP64, so that what is left then is their rounding.
    int run(AmgState& A, const std::string& key, const double* B, double* X, const double* X0, CgCount* count) {
        const SellDev& A0 = NV == 1 ? H.K : H.lv[0].A;
        n = A0.n;
        G = int(std::min<int64_t>(blocks_of(n * R, 512), kRedMaxGrid));
        int* hc = reinterpret_cast<int*>(M->host_scratch + 240);
        cudaError_t e = cudaSuccess;
        auto read_ctl = [&]() -> cudaError_t {
            cudaError_t x = cudaMemcpyAsync(hc, C.ctl, 7 * sizeof(int), cudaMemcpyDeviceToHost, s);
            if (x == cudaSuccess) x = cudaStreamSynchronize(s);
            return x;
        };
        const bool refine = so.sweep_rtol > 0.0;
        const double tol[2] = {so.rtol * so.rtol, refine ? so.sweep_rtol * so.sweep_rtol : 0.0};
        const int cap[1] = {so.maxit};
        if ((e = cudaMemsetAsync(C.ctl, 0, 8 * sizeof(int), s)) != cudaSuccess ||
            (e = cudaMemcpyAsync(C.ctl + 4, cap, sizeof(int), cudaMemcpyHostToDevice, s)) != cudaSuccess ||
            (e = cudaMemcpyAsync(C.tol, tol, sizeof(tol), cudaMemcpyHostToDevice, s)) != cudaSuccess ||
            (e = cudaMemsetAsync(C.p, 0, sizeof(double) * n * R, s)) != cudaSuccess)
            return cuda_fail(e, "multigrid start");
        for (const double* from = X0;; from = C.x) {
            note_launch(2);
            if (from) {
                k_cg_init_x0<R, NV><<<G, 256, 0, s>>>(A0, st.v64[0], st.v64[1], B, from, C.x, C.r, C.part);
                k_cg_start<R, 2><<<1, 32 * R, 0, s>>>(C.part, G, C.tol, C.bb, C.stop, C.scale, C.ctl);
            } else {
                k_cg_init<R><<<G, 256, 0, s>>>(n, B, C.x, C.r, C.part);
                k_cg_start<R, 1><<<1, 32 * R, 0, s>>>(C.part, G, C.tol, C.bb, C.stop, C.scale, C.ctl);
            }
            if ((e = read_ctl()) != cudaSuccess) return cuda_fail(e, "multigrid cg");
            if (hc[0] != QPAT_OK)
                return fail(hc[0], hc[0] == QPAT_EINVAL ? "multigrid cg: right-hand side not finite"
                                                        : "multigrid cg: residual at the start not finite");
            if (hc[5] > 0) {
                note_launch(1);
                k_cg_clear<R><<<G, 256, 0, s>>>(n, C.bb, C.x, C.r);
            }
            if (hc[1] == 0) break;
            if (refine && count->sweeps >= so.max_sweeps) {
                count->stalled = true;
                break;
            }
            ++count->sweeps;
            scaled = f32 && hc[6] > 0;
            if (f32) {
                note_launch(1);
                k_cg_cast<R><<<G, 256, 0, s>>>(n, C.scale, C.r, static_cast<float*>(W.b[0]));
            }
            if (!timer->on) {
                const std::string name = scaled ? key + "/scaled" : key;
                auto g = V.graphs.find(name);
                if (g == V.graphs.end()) {
                    AmgGraph fresh;
                    const int rc = capture(A, fresh);
                    if (rc != QPAT_OK) return rc;
                    g = V.graphs.emplace(name, std::move(fresh)).first;
                }
                if ((e = cudaGraphLaunch(g->second.exec, s)) != cudaSuccess) return cuda_fail(e, "multigrid graph");
                if ((e = read_ctl()) != cudaSuccess) return cuda_fail(e, "multigrid cg");
                note_launch(hc[2] * g->second.body_kernels);
            } else {
                while (true) {
                    body(s, 0, 0);
                    if ((e = read_ctl()) != cudaSuccess) return cuda_fail(e, "multigrid cg");
                    timer->collect();
                    if (hc[0] != QPAT_OK || hc[1] == 0) break;
                }
            }
            count->iters += hc[2];
            if (hc[0] == QPAT_ENOCONV) return fail(QPAT_ENOCONV, "multigrid cg: iteration cap reached");
            if (hc[0] != QPAT_OK) return fail(hc[0], "multigrid cg: breakdown (p.Ap <= 0 or not finite)");
            if (!refine) break;
        }
        if ((e = cudaMemcpyAsync(X, C.x, sizeof(double) * n * R, cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
            return cuda_fail(e, "copy");
        return QPAT_OK;
    }

    int capture(AmgState& A, AmgGraph& g) {
        cudaError_t e = cudaSuccess;
        if (!A.capture && (e = cudaStreamCreateWithFlags(&A.capture, cudaStreamNonBlocking)) != cudaSuccess)
            return cuda_fail(e, "multigrid capture stream");
        if ((e = cudaGraphCreate(&g.graph, 0)) != cudaSuccess) return cuda_fail(e, "multigrid graph");
        cudaGraphConditionalHandle cond;
        if ((e = cudaGraphConditionalHandleCreate(&cond, g.graph, 1, cudaGraphCondAssignDefault)) != cudaSuccess)
            return cuda_fail(e, "multigrid graph");
        cudaGraphNodeParams np = {};
        np.type = cudaGraphNodeTypeConditional;
        np.conditional.handle = cond;
        np.conditional.type = cudaGraphCondTypeWhile;
        np.conditional.size = 1;
        cudaGraphNode_t node;
        if ((e = cudaGraphAddNode(&node, g.graph, nullptr, nullptr, 0, &np)) != cudaSuccess)
            return cuda_fail(e, "multigrid graph");
        cudaGraph_t bodyg = np.conditional.phGraph_out[0];
        if ((e = cudaStreamBeginCaptureToGraph(A.capture, bodyg, nullptr, nullptr, 0,
                                               cudaStreamCaptureModeThreadLocal)) != cudaSuccess)
            return cuda_fail(e, "multigrid capture");
        const int64_t before = thread_launches();
        body(A.capture, cond, 1);
        g.body_kernels = int(thread_launches() - before);
        cudaGraph_t out = nullptr;
        const cudaError_t e1 = cudaGetLastError();
        e = cudaStreamEndCapture(A.capture, &out);
        // capturing counted the body's launches once; replays are counted per iteration
        note_launch(-g.body_kernels);
        if (e1 != cudaSuccess) return cuda_fail(e1, "multigrid capture");
        if (e != cudaSuccess) return cuda_fail(e, "multigrid capture");
        if ((e = cudaGraphInstantiate(&g.exec, g.graph, 0)) != cudaSuccess) return cuda_fail(e, "multigrid graph");
        return QPAT_OK;
    }
};

template <int NV>
int dispatch(int R, AmgState& A, const std::string& key, qpat_mesh_s* M, const OpState& st, const SolveOpts& so,
             const AmgHierDev& H, AmgValues& V, bool f32, AmgVecs& W, AmgCg& C, const double* B, double* X,
             const double* X0, cudaStream_t s, FineTimer* timer, CgCount* count) {
    if constexpr (NV == 2) {
        return CgSolve<2, 2>{M, st, so, H, V, f32, W, C, s, timer}.run(A, key, B, X, X0, count);
    } else {
        switch (R) {
            case 1: return CgSolve<1, 1>{M, st, so, H, V, f32, W, C, s, timer}.run(A, key, B, X, X0, count);
            case 2: return CgSolve<2, 1>{M, st, so, H, V, f32, W, C, s, timer}.run(A, key, B, X, X0, count);
            case 4: return CgSolve<4, 1>{M, st, so, H, V, f32, W, C, s, timer}.run(A, key, B, X, X0, count);
            case 8: return CgSolve<8, 1>{M, st, so, H, V, f32, W, C, s, timer}.run(A, key, B, X, X0, count);
            default: return CgSolve<16, 1>{M, st, so, H, V, f32, W, C, s, timer}.run(A, key, B, X, X0, count);
        }
    }
}

}  // namespace

int amg_solve(qpat_mesh_s* M, const OpState& st, const SolveOpts& so, int R, const double* B, double* X,
              cudaStream_t s, const double* X0) {
    if (R != 1 && R != 2 && R != 4 && R != 8 && R != 16) return fail(QPAT_EINVAL, "multigrid: R must be 1, 2, 4, 8 or 16");
    if (st.nv == 2 && R != 2) return fail(QPAT_EINVAL, "multigrid: M_delta is solved as 2 right-hand sides");
    if (!(so.mg_ratio > 1.0) || so.mg_degree < 1 || so.mg_degree > 8)
        return fail(QPAT_EINVAL, "multigrid: mg_degree must lie in [1, 8] and mg_ratio exceed 1");
    if (!M->amg) M->amg = new AmgState();
    AmgState& A = *M->amg;
    A.ledger.refused = false;
    AmgHierDev& H = A.hier;
    if (!H.ready) {
        if (!H.error.empty()) return fail(QPAT_EINVAL, H.error);
        AmgHierDev fresh(&A.ledger);
        const int rc = build_hier(M, fresh, A.ledger);
        if (rc != QPAT_OK) {
            H.error = fresh.error;  // no hierarchy for this mesh; empty where only memory is short
            return rc;
        }
        H = std::move(fresh);
    }
    const bool f32 = so.multigrid == 2 && st.kind == OP_K;
    const bool fast = so.mg_degree <= 1 && H.lv.size() > 1;
    H.used[st.kind == OP_PRIOR] = true;
    const void* const op = st.v64[0];
    AmgValues& V = A.vals.try_emplace(op, &A.ledger).first->second;
    int rc = numeric(M, H, st, V, fast, so.mg_ratio, f32, s);
    if (rc != QPAT_OK) {
        A.vals.erase(op);
        return rc;
    }
    cudaError_t e = cudaSuccess;
    const std::array<int, 3> form{R, f32 ? 1 : 0, fast ? 1 : 0};
    auto vecs = A.vecs.find(form);
    if (vecs == A.vecs.end()) {
        AmgVecs fresh(&A.ledger);
        const size_t esz = f32 ? sizeof(float) : sizeof(double), L = H.lv.size();
        // the fine level's iterate and its partners belong to the polynomial (or, alone, to the dense solve), its
        // right-hand side is CG's residual unless the cycle wants that in FP32
        for (size_t l = 0; l < L; ++l) {
            auto vec = [&](bool used) {
                return used ? fresh.mem.get<char>(size_t(H.lv[l].A.n) * R * esz, e) : nullptr;
            };
            fresh.b.push_back(vec(l > 0 || f32));
            fresh.xa.push_back(vec(l > 0 || !fast));
            fresh.xb.push_back(vec(l == 0 && !fast));
            fresh.d.push_back(vec(l == 0 && !fast));
            fresh.r.push_back(vec(l + 1 < L));
        }
        if (e != cudaSuccess) return cuda_fail(e, "multigrid workspace");
        vecs = A.vecs.emplace(form, std::move(fresh)).first;
    }
    AmgVecs& W = vecs->second;
    auto cg = A.cg.find(R);
    if (cg == A.cg.end()) {
        AmgCg C(&A.ledger);
        const size_t nR = size_t(M->h.N) * R;
        C.x = C.mem.get<double>(nR, e);
        C.r = C.mem.get<double>(nR, e);
        C.p = C.mem.get<double>(nR, e);
        C.q = C.mem.get<double>(nR, e);
        C.z = C.mem.get<double>(nR, e);
        C.part = C.mem.get<double>(size_t(kRedMaxGrid) * 32, e);
        double* sc = C.mem.get<double>(7 * 16 + 2, e);
        C.ctl = C.mem.get<int>(kCtlActive + 16, e);
        C.count = C.mem.get<unsigned>(1, e);
        if (e == cudaSuccess) e = cudaMemsetAsync(C.count, 0, sizeof(unsigned), s);
        if (e == cudaSuccess) e = cudaMemsetAsync(C.q, 0, sizeof(double) * nR, s);
        if (e != cudaSuccess) return cuda_fail(e, "multigrid workspace");
        C.bb = sc;
        C.rz = sc + 16;
        C.alpha = sc + 32;
        C.beta = sc + 48;
        C.rr = sc + 64;
        C.scale = sc + 80;
        C.stop = sc + 96;
        C.tol = sc + 112;
        cg = A.cg.emplace(R, std::move(C)).first;
    }
    AmgCg& C = cg->second;
    // an iteration captured on V depends on these settings and buffers beside it
    char key[256];
    std::snprintf(key, sizeof key, "%d/%d/%d/%d/%.17g/%p", R, st.nv, int(f32), so.mg_degree, so.mg_ratio,
                  static_cast<const void*>(st.v64[1]));
    FineTimer timer;
    timer.on = M->timing != 0;
    timer.s = s;
    if (M->timing) cudaEventRecord(M->ev0, s);
    CgCount count;
    rc = st.nv == 2 ? dispatch<2>(R, A, key, M, st, so, H, V, f32, W, C, B, X, X0, s, &timer, &count)
                    : dispatch<1>(R, A, key, M, st, so, H, V, f32, W, C, B, X, X0, s, &timer, &count);
    if (timer.on) {
        cudaStreamSynchronize(s);
        timer.collect();
        M->mg_fine_ms += timer.ms;
        M->mg_fine_launches += timer.launches;
    }
    if ((e = cudaGetLastError()) != cudaSuccess && rc == QPAT_OK) rc = cuda_fail(e, "multigrid launch");
    if (M->timing) {
        cudaEventRecord(M->ev1, s);
        cudaEventSynchronize(M->ev1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, M->ev0, M->ev1);
        M->pcg_ms += ms;
    }
    M->stats.pcg_iters += count.iters;
    M->stats.rhs_iters += int64_t(count.iters) * R;
    M->stats.solves += R;
    M->stats.launches += std::max(1, count.sweeps);
    if (so.sweep_rtol > 0.0) M->stats.refinements += count.sweeps;
    if (count.stalled) M->stats.fp64_fallbacks += 1;
    return rc;
}

int amg_levels(qpat_mesh_s* M, int prior, int64_t* rows, int max_levels) {
    if (!M->amg) return 0;
    const AmgHierDev& H = M->amg->hier;
    if (!H.used[prior ? 1 : 0]) return 0;
    const int L = int(H.lv.size());
    for (int l = 0; l < std::min(L, max_levels); ++l) rows[l] = H.lv[size_t(l)].A.n;
    return L;
}

void amg_set_limit(qpat_mesh_s* M, size_t bytes) {
    if (!M->amg) M->amg = new AmgState();
    M->amg->ledger.limit = bytes;
}

AmgOutcome amg_outcome(const qpat_mesh_s* M) {
    if (!M->amg || M->amg->ledger.refused) return AmgOutcome::no_memory;
    return M->amg->hier.ready ? AmgOutcome::ran : AmgOutcome::no_hierarchy;
}

size_t amg_bytes(const qpat_mesh_s* M) { return M->amg ? M->amg->ledger.used : 0; }

void amg_release(qpat_mesh_s* M) {
    if (!M->amg) return;
    if (M->amg->capture) cudaStreamDestroy(M->amg->capture);
    delete M->amg;
    M->amg = nullptr;
}

}  // namespace qpat
