// One-pass patch kernels (operator applies, diagonals, Jacobian pieces),
// the load vector, layout conversions and reductions.
#include "launch.h"

namespace qpat {

namespace {

constexpr int kRedBlocks = 608;  // 4 x 152 SMs

// ---------------------------------------------------------------- operator apply
// One CTA per patch: stage, element loop, write the owned rows.  Columns
// [c0, c0 + R) of N x ldx node-major x and y (large RHS counts are applied in
// column chunks so that the staging fits in shared memory).
template <typename T, int R, int OP>
__global__ void __launch_bounds__(kThreads) k_apply(MeshDev m, OpParams<T> op, T sign, const T* __restrict__ x,
                                                    T* __restrict__ y, int ldx, int c0) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PatchSmem<T, R> s;
    s.carve(reinterpret_cast<T*>(smem_raw), m.max_touched, m.max_own);
    const int p = blockIdx.x;
    const int nb = m.node_ptr[p], nt = m.node_ptr[p + 1] - nb;
    const int ob = m.own_begin[p], nown = m.own_begin[p + 1] - ob;
    stage_static<T, R>(m, nb, nt, s, op);
    for (int i = threadIdx.x; i < nt * R; i += blockDim.x) {
        const int g = __ldg(m.nodes + nb + i / R);
        s.xin[i] = __ldg(x + size_t(g) * ldx + c0 + (i % R));
    }
    for (int i = threadIdx.x; i < nown * R; i += blockDim.x) s.yout[i] = T(0);
    __syncthreads();
    patch_elements<T, R, OP, true>(m, p, nown, s, op);  // coloured: run-to-run identical
    __syncthreads();
    for (int i = threadIdx.x; i < nown * R; i += blockDim.x) {
        T v = s.yout[i];
        if (OP == OP_PRIOR) v += op.delta * s.xin[i];
        y[size_t(ob + i / R) * ldx + c0 + (i % R)] = sign * v;
    }
}

constexpr size_t kSmemBudget = 200 * 1024;

template <typename T, int R, int OP>
cudaError_t apply_t(const MeshDev& m, const OpParams<T>& op, T sign, const T* x, T* y, int ldx, int c0,
                    cudaStream_t st) {
    const size_t smem = PatchSmem<T, R>::bytes(m.max_touched, m.max_own);
    auto kern = k_apply<T, R, OP>;
    cudaError_t e = qpat::allow_smem((const void*)kern, size_t(smem));
    if (e != cudaSuccess) return e;
    qpat::note_launch(1);
    kern<<<m.P, kThreads, smem, st>>>(m, op, sign, x, y, ldx, c0);
    return cudaGetLastError();
}

// largest chunk of {16, 8, 4, 2, 1} dividing R whose staging fits the budget
template <typename T>
int apply_chunk(const MeshDev& m, int R, size_t per_node_extra) {
    for (int c : {16, 8, 4, 2, 1}) {
        if (c > R || R % c) continue;
        const size_t bytes = sizeof(T) * (size_t(m.max_touched) * (per_node_extra + size_t(c)) +
                                          size_t(m.max_own) * c);
        if (bytes <= kSmemBudget) return c;
    }
    return 1;
}

// ---------------------------------------------------------------- diagonals (FP64)
// diag K_ii = sum_T [ S_kappa/4 |c_i|^2/(6|det|) + |T|/120 (2 S_mu + 4 mu_i) ] + sum_F |F|/12
__global__ void __launch_bounds__(kThreads) k_diag_K(MeshDev m, const double* __restrict__ kappa,
                                                     const double* __restrict__ mu, double* inv64, float* inv32) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PatchSmem<double, 1> s;
    s.carve(reinterpret_cast<double*>(smem_raw), m.max_touched, m.max_own);
    const int p = blockIdx.x;
    const int nb = m.node_ptr[p], nt = m.node_ptr[p + 1] - nb;
    const int ob = m.own_begin[p], nown = m.own_begin[p + 1] - ob;
    OpParams<double> op{kappa, mu, 0, 0, 0, 1};
    stage_static<double, 1>(m, nb, nt, s, op);
    for (int i = threadIdx.x; i < nown; i += blockDim.x) s.yout[i] = 0.0;
    __syncthreads();
    // colour by colour: plain sums in a fixed order (see for_each_coloured)
    for_each_coloured(m.tcol_beg, m.tcol_off, p, [&](int t) {
        const ushort4 lv = m.tet_loc[t];
        const int v[4] = {lv.x, lv.y, lv.z, lv.w};
        double pc[4][3], c[4][3], ad;
        load_tet(s, lv, pc);
        tet_cofactors(pc, c, ad);
        double ks = 0, Sm = 0;
        for (int a = 0; a < 4; ++a) {
            ks += s.c1[v[a]];
            Sm += s.c2[v[a]];
        }
        const double sk = ks / (24.0 * ad), vm = ad / 720.0;
        for (int a = 0; a < 4; ++a)
            if (v[a] < nown) {
                const double c2 = c[a][0] * c[a][0] + c[a][1] * c[a][1] + c[a][2] * c[a][2];
                s.yout[v[a]] += sk * c2 + vm * (2.0 * Sm + 4.0 * s.c2[v[a]]);
            }
    });
    for_each_coloured(m.fcol_beg, m.fcol_off, p, [&](int f) {
        const ushort4 lv = m.face_loc[f];
        const int v[3] = {lv.x, lv.y, lv.z};
        const double w = m.pface_area64[f] / 12.0;
        for (int a = 0; a < 3; ++a)
            if (v[a] < nown) s.yout[v[a]] += w;
    });
    for (int i = threadIdx.x; i < nown; i += blockDim.x) {
        const double d = 1.0 / s.yout[i];
        inv64[ob + i] = d;
        if (inv32) inv32[ob + i] = float(d);
    }
}

// diag M_delta: block r: scale_r c_T |c_i|^2 / (6 |det|) + delta
__global__ void __launch_bounds__(kThreads) k_diag_prior(MeshDev m, const double* __restrict__ u1,
                                                         const double* __restrict__ u2, double inv_T2,
                                                         int kind, double q, double scale1, double delta,
                                                         double* inv64, float* inv32) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PatchSmem<double, 2> s;
    s.carve(reinterpret_cast<double*>(smem_raw), m.max_touched, m.max_own);
    const int p = blockIdx.x;
    const int nb = m.node_ptr[p], nt = m.node_ptr[p + 1] - nb;
    const int ob = m.own_begin[p], nown = m.own_begin[p + 1] - ob;
    OpParams<double> op{u1, u2, inv_T2, scale1, delta, 0, nullptr, nullptr, kind, q};
    stage_static<double, 2>(m, nb, nt, s, op);
    for (int i = threadIdx.x; i < 2 * nown; i += blockDim.x) s.yout[i] = 0.0;
    __syncthreads();
    for_each_coloured(m.tcol_beg, m.tcol_off, p, [&](int t) {
        const ushort4 lv = m.tet_loc[t];
        const int v[4] = {lv.x, lv.y, lv.z, lv.w};
        double pc[4][3], c[4][3], ad;
        load_tet(s, lv, pc);
        tet_cofactors(pc, c, ad);
        for (int r = 0; r < 2; ++r) {
            const double* uc = r == 0 ? s.c1 : s.c2;
            double u[4], Gu[3];
            for (int a = 0; a < 4; ++a) u[a] = uc[v[a]];
            grad_vec(c, u, Gu);
            const double g2 = (Gu[0] * Gu[0] + Gu[1] * Gu[1] + Gu[2] * Gu[2]) / (ad * ad);
            const double cT = prior_weight<double>(kind, g2, inv_T2, q);
            const double sk = (r == 0 ? 1.0 : scale1) * cT / (6.0 * ad);
            for (int a = 0; a < 4; ++a)
                if (v[a] < nown) s.yout[2 * v[a] + r] += sk * (c[a][0] * c[a][0] + c[a][1] * c[a][1] + c[a][2] * c[a][2]);
        }
    });
    for (int i = threadIdx.x; i < 2 * nown; i += blockDim.x) {
        const double d = 1.0 / (s.yout[i] + delta);
        inv64[2 * ob + i] = d;
        if (inv32) inv32[2 * ob + i] = float(d);
    }
}

// y = A x with an assembled operator: one CTA per patch, x staged on the
// touched nodes in shared memory, thread-per-row sliced-ELLPACK rows.
template <typename T, int R, int NV>
__global__ void __launch_bounds__(kThreads) k_apply_csr(MeshDev m, const T* __restrict__ v0,
                                                        const T* __restrict__ v1, const T* __restrict__ x,
                                                        T* __restrict__ y) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* xin = reinterpret_cast<T*>(smem_raw);
    const int p = blockIdx.x;
    const int nb = m.node_ptr[p], nt = m.node_ptr[p + 1] - nb;
    const int ob = m.own_begin[p], nown = m.own_begin[p + 1] - ob;
    for (int i = threadIdx.x; i < nt * R; i += blockDim.x) {
        const int g = __ldg(m.nodes + nb + i / R);
        xin[i] = __ldg(x + size_t(g) * R + (i % R));
    }
    __syncthreads();
    csr_rows<T, R, NV>(m, ob, nown, v0, v1, xin, [&](int i, int r, T v) { y[size_t(ob + i) * R + r] = v; });
}

template <typename T, int R, int NV>
cudaError_t apply_csr_t(const MeshDev& m, const T* v0, const T* v1, const T* x, T* y, cudaStream_t st) {
    const size_t smem = sizeof(T) * size_t(m.max_touched) * R;
    auto kern = k_apply_csr<T, R, NV>;
    cudaError_t e = qpat::allow_smem((const void*)kern, size_t(smem));
    if (e != cudaSuccess) return e;
    qpat::note_launch(1);
    kern<<<m.P, kThreads, smem, st>>>(m, v0, v1, x, y);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- load vector
// f_i += 2/3 sum over the boundary faces F of node i of Phi_F |F|, gathered per
// (node, illumination) over the node's faces in a fixed order.  Bound by the
// latency of a face's two loads behind its index and of FP64: three faces in
// flight and one division a node (91,125 nodes x 4: 16 us; one face at a time
// with a division each: 49).
__global__ void k_load(MeshDev m, int K, int R, const double* __restrict__ flux, double* f) {
    constexpr int U = 3;
    const int64_t total = int64_t(m.N) * K;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
        const int g = int(i / K), k = int(i % K);
        const int q0 = __ldg(m.nface_ptr + g), q1 = __ldg(m.nface_ptr + g + 1);
        if (q0 == q1) continue;
        double acc = 0.0;
        for (int q = q0; q < q1; q += U) {
            double v[U], w[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int fi = __ldg(m.nface + min(q + u, q1 - 1));
                v[u] = __ldg(flux + size_t(k) * m.F + fi);
                w[u] = __ldg(m.farea + fi);
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (q + u < q1) acc = fma(v[u], w[u], acc);
        }
        f[size_t(g) * R + k] += 2.0 * acc / 3.0;
    }
}

// ---------------------------------------------------------------- layout helpers
// out[l*R + r] = in[r*N + perm[l]] for r < K, 0 for K <= r < R
template <typename Tin, typename Tout>
__global__ void k_to_lib(int N, int K, int R, const int* __restrict__ perm, const Tin* __restrict__ in,
                         Tout* __restrict__ out) {
    const int64_t total = int64_t(N) * R;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
        const int l = int(i / R), r = int(i % R);
        out[i] = r < K ? Tout(in[int64_t(r) * N + perm[l]]) : Tout(0);
    }
}

// out[r*N + perm[l]] = in[l*R + r] for r < K
template <typename Tin, typename Tout>
__global__ void k_from_lib(int N, int K, int R, const int* __restrict__ perm, const Tin* __restrict__ in,
                           Tout* __restrict__ out) {
    const int64_t total = int64_t(N) * K;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
        const int l = int(i / K), r = int(i % K);
        out[int64_t(r) * N + perm[l]] = Tout(in[int64_t(l) * R + r]);
    }
}

int grid_for(int64_t n) {
    int64_t g = (n + 255) / 256;
    if (g > 152 * 16) g = 152 * 16;
    if (g < 1) g = 1;
    return int(g);
}

// ---------------------------------------------------------------- reductions
template <typename T>
__global__ void k_dot_partial(int64_t n, int R, const T* __restrict__ a, const T* __restrict__ b, double* partial) {
    // thread t handles entries i with i % R == t % R (blockDim multiple of R)
    __shared__ double sm[256];
    double acc = 0.0;
    const int64_t total = n * R;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x)
        acc += double(a[i]) * double(b[i]);
    sm[threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.x < R) {
        double s = 0.0;
        for (int j = threadIdx.x; j < blockDim.x; j += R) s += sm[j];
        partial[size_t(blockIdx.x) * R + threadIdx.x] = s;
    }
}

// A warp per right-hand side, eight loads of a lane in flight (one thread
// adding 608 partial sums in a row: 36 us).
__global__ void k_dot_final(int nblk, int R, const double* partial, double* out) {
    const int r = blockIdx.x;
    double a[8] = {};
    for (int j0 = threadIdx.x; j0 < nblk; j0 += 8 * 32)
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (j0 + 32 * u < nblk) a[u] += partial[size_t(j0 + 32 * u) * R + r];
    double s = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) out[r] = s;
}

__global__ void k_cast_d2f_scaled(int64_t n, int R, const double* in, const double* scale, float* out) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n * R; i += int64_t(gridDim.x) * blockDim.x) {
        const double s = scale[i % R];
        out[i] = s > 0.0 ? float(in[i] / s) : 0.0f;
    }
}

__global__ void k_axpy_f2d_scaled(int64_t n, int R, const float* d, const double* scale, double* x) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n * R; i += int64_t(gridDim.x) * blockDim.x)
        x[i] += scale[i % R] * double(d[i]);
}

__global__ void k_sub(int64_t n, const double* a, const double* b, double* out) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
        out[i] = a[i] - b[i];
}

__global__ void k_cast_d2f(int64_t n, const double* in, float* out) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
        out[i] = float(in[i]);
}

}  // namespace

template <typename T>
cudaError_t launch_apply_K(const MeshDev& m, int R, const T* c1, const T* c2, int robin, T sign, const T* x, T* y,
                           cudaStream_t s) {
    OpParams<T> op{c1, c2, T(0), T(0), T(0), robin};
    if (R != 1 && R != 2 && R != 4 && R != 8 && R != 16) return cudaErrorInvalidValue;
    const int C = apply_chunk<T>(m, R, 5);
    for (int c0 = 0; c0 < R; c0 += C) {
        cudaError_t e = cudaErrorInvalidValue;
        switch (C) {
            case 1: e = apply_t<T, 1, OP_K>(m, op, sign, x, y, R, c0, s); break;
            case 2: e = apply_t<T, 2, OP_K>(m, op, sign, x, y, R, c0, s); break;
            case 4: e = apply_t<T, 4, OP_K>(m, op, sign, x, y, R, c0, s); break;
            case 8: e = apply_t<T, 8, OP_K>(m, op, sign, x, y, R, c0, s); break;
            case 16: e = apply_t<T, 16, OP_K>(m, op, sign, x, y, R, c0, s); break;
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t launch_apply_prior(const MeshDev& m, const T* u1, const T* u2, T inv_T2, int kind, T q, T scale1,
                               T delta, const T* x, T* y, cudaStream_t s) {
    OpParams<T> op{u1, u2, inv_T2, scale1, delta, 0, nullptr, nullptr, kind, q};
    return apply_t<T, 2, OP_PRIOR>(m, op, T(1), x, y, 2, 0, s);
}

cudaError_t launch_invdiag_K(const MeshDev& m, const double* kappa, const double* mu, double* inv64, float* inv32,
                             cudaStream_t s) {
    const size_t smem = PatchSmem<double, 1>::bytes(m.max_touched, m.max_own);
    cudaError_t e = qpat::allow_smem((const void*)k_diag_K, size_t(smem));
    if (e != cudaSuccess) return e;
    qpat::note_launch(1);
    k_diag_K<<<m.P, kThreads, smem, s>>>(m, kappa, mu, inv64, inv32);
    return cudaGetLastError();
}

cudaError_t launch_invdiag_prior(const MeshDev& m, const double* u1, const double* u2, double inv_T2, int kind,
                                 double q, double scale1, double delta, double* inv64, float* inv32,
                                 cudaStream_t s) {
    const size_t smem = PatchSmem<double, 2>::bytes(m.max_touched, m.max_own);
    cudaError_t e = qpat::allow_smem((const void*)k_diag_prior, size_t(smem));
    if (e != cudaSuccess) return e;
    qpat::note_launch(1);
    k_diag_prior<<<m.P, kThreads, smem, s>>>(m, u1, u2, inv_T2, kind, q, scale1, delta, inv64, inv32);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_apply_csr(const MeshDev& m, int NV, int R, const T* v0, const T* v1, const T* x, T* y,
                             cudaStream_t s) {
    if (NV == 2) {
        if (R != 2) return cudaErrorInvalidValue;
        return apply_csr_t<T, 2, 2>(m, v0, v1, x, y, s);
    }
    switch (R) {
        case 1: return apply_csr_t<T, 1, 1>(m, v0, v1, x, y, s);
        case 2: return apply_csr_t<T, 2, 1>(m, v0, v1, x, y, s);
        case 4: return apply_csr_t<T, 4, 1>(m, v0, v1, x, y, s);
        case 8: return apply_csr_t<T, 8, 1>(m, v0, v1, x, y, s);
        case 16: return apply_csr_t<T, 16, 1>(m, v0, v1, x, y, s);
        default: return cudaErrorInvalidValue;
    }
}

// Whether k_apply_csr for R right-hand sides fits the device's per-block
// shared memory (the input vector is staged on the patch's touched nodes).
template <typename T>
bool apply_csr_fits(const MeshDev& m, int R) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return true;
    }
    return sizeof(T) * size_t(m.max_touched) * size_t(R) <= size_t(optin);
}
template bool apply_csr_fits<double>(const MeshDev&, int);
template bool apply_csr_fits<float>(const MeshDev&, int);

template cudaError_t launch_apply_csr<double>(const MeshDev&, int, int, const double*, const double*, const double*,
                                              double*, cudaStream_t);
template cudaError_t launch_apply_csr<float>(const MeshDev&, int, int, const float*, const float*, const float*,
                                             float*, cudaStream_t);

cudaError_t launch_load(const MeshDev& m, int K, int R, const double* flux, double* f, cudaStream_t s) {
    qpat::note_launch(1);
    k_load<<<grid_for(int64_t(m.N) * K), 256, 0, s>>>(m, K, R, flux, f);
    return cudaGetLastError();
}

template <typename Tin, typename Tout>
cudaError_t launch_to_lib(const MeshDev& m, int K, int R, const Tin* in, Tout* out, cudaStream_t s) {
    qpat::note_launch(1);
    k_to_lib<Tin, Tout><<<grid_for(int64_t(m.N) * R), 256, 0, s>>>(m.N, K, R, m.perm, in, out);
    return cudaGetLastError();
}

template <typename Tin, typename Tout>
cudaError_t launch_from_lib(const MeshDev& m, int K, int R, const Tin* in, Tout* out, cudaStream_t s) {
    qpat::note_launch(1);
    k_from_lib<Tin, Tout><<<grid_for(int64_t(m.N) * K), 256, 0, s>>>(m.N, K, R, m.perm, in, out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_dots(int64_t n, int R, const T* a, const T* b, double* partial, double* out, cudaStream_t s) {
    qpat::note_launch(1);
    k_dot_partial<T><<<kRedBlocks, 256, 0, s>>>(n, R, a, b, partial);
    qpat::note_launch(1);
    k_dot_final<<<R, 32, 0, s>>>(kRedBlocks, R, partial, out);
    return cudaGetLastError();
}

cudaError_t launch_cast_d2f_scaled(int64_t n, int R, const double* in, const double* scale, float* out,
                                   cudaStream_t s) {
    qpat::note_launch(1);
    k_cast_d2f_scaled<<<grid_for(n * R), 256, 0, s>>>(n, R, in, scale, out);
    return cudaGetLastError();
}

cudaError_t launch_axpy_f2d_scaled(int64_t n, int R, const float* d, const double* scale, double* x,
                                   cudaStream_t s) {
    qpat::note_launch(1);
    k_axpy_f2d_scaled<<<grid_for(n * R), 256, 0, s>>>(n, R, d, scale, x);
    return cudaGetLastError();
}

cudaError_t launch_sub(int64_t n, const double* a, const double* b, double* out, cudaStream_t s) {
    qpat::note_launch(1);
    k_sub<<<grid_for(n), 256, 0, s>>>(n, a, b, out);
    return cudaGetLastError();
}

cudaError_t launch_cast_d2f(int64_t n, const double* in, float* out, cudaStream_t s) {
    qpat::note_launch(1);
    k_cast_d2f<<<grid_for(n), 256, 0, s>>>(n, in, out);
    return cudaGetLastError();
}

template cudaError_t launch_apply_K<double>(const MeshDev&, int, const double*, const double*, int, double,
                                            const double*, double*, cudaStream_t);
template cudaError_t launch_apply_K<float>(const MeshDev&, int, const float*, const float*, int, float, const float*,
                                           float*, cudaStream_t);
template cudaError_t launch_apply_prior<double>(const MeshDev&, const double*, const double*, double, int, double,
                                                double, double, const double*, double*, cudaStream_t);
template cudaError_t launch_apply_prior<float>(const MeshDev&, const float*, const float*, float, int, float, float,
                                               float, const float*, float*, cudaStream_t);
template cudaError_t launch_to_lib<double, double>(const MeshDev&, int, int, const double*, double*, cudaStream_t);
template cudaError_t launch_to_lib<double, float>(const MeshDev&, int, int, const double*, float*, cudaStream_t);
template cudaError_t launch_from_lib<double, double>(const MeshDev&, int, int, const double*, double*, cudaStream_t);
template cudaError_t launch_from_lib<float, double>(const MeshDev&, int, int, const float*, double*, cudaStream_t);
template cudaError_t launch_dots<double>(int64_t, int, const double*, const double*, double*, double*, cudaStream_t);
template cudaError_t launch_dots<float>(int64_t, int, const float*, const float*, double*, double*, cudaStream_t);

}  // namespace qpat
