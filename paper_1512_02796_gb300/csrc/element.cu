// Element sums as gathers over the element plan (see element.h): assembly of
// K and of the two M_delta blocks, the right-hand sides of J s and the
// accumulation of J^T t.
//
// Each is two or three short kernels: per tet (or per edge) the products that
// its tets share, per edge the sum over the tets around it, per row the
// entries of the row.  Every sum runs in the order of the plan, so results
// are the same from run to run, with no atomics, no colours and no barriers.
//
// Bound: FP64 issue and the plan's bytes about equally.  At 128^3 (2.1 M
// nodes, 12.3 M tets) K takes ~200 FP64 operations and ~1.5 KB a node (per tet
// 144 bytes with the lists that name it, per edge 64, per entry 16);
// the element-by-element form that this replaces recomputed the geometry of
// every tet (some 150 FP64 operations, for each patch that lists it),
// searched the row for every entry and waited at ~26 barriers a patch.
#include "element.h"
#include "launch.h"

namespace qpat {
namespace {

constexpr int kT = 256;
inline unsigned blocks(int64_t n) { return unsigned((n + kT - 1) / kT); }
__device__ __forceinline__ int64_t thread_id() { return blockIdx.x * int64_t(blockDim.x) + threadIdx.x; }

// Off-diagonal stiffness factors s_ab = c_a . c_b / (24 |det|) and vm = |det| / 720.
__global__ void __launch_bounds__(kT) k_geometry(ElemDev el, const double* __restrict__ xyz) {
    const int64_t t = thread_id();
    if (t >= el.E) return;
    const int4 v = el.tet[t];
    const int id[4] = {v.x, v.y, v.z, v.w};
    double p[4][3], c[4][3], ad;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int k = 0; k < 3; ++k) p[a][k] = xyz[3 * int64_t(id[a]) + k];
    tet_cofactors(p, c, ad);
    const double f = 1.0 / (24.0 * ad);
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        const int a = edge_a(q), b = edge_b(q);
        el.s[6 * t + q] = f * (c[a][0] * c[b][0] + c[a][1] * c[b][1] + c[a][2] * c[b][2]);
    }
    el.vm[t] = ad / 720.0;
}

__global__ void __launch_bounds__(kT) k_geometry_sums(ElemDev el, int64_t N) {
    const int64_t i = thread_id();
    if (i < el.NE) {
        double a = 0.0;
        for (int64_t q = el.edge_ptr[i]; q < el.edge_ptr[i + 1]; ++q) a += el.vm[el.edge_tet[q] >> 3];
        el.edge_vr[i].x = a;
    }
    if (i < N) {
        double a = 0.0;
        for (int64_t q = el.node_ptr[i]; q < el.node_ptr[i + 1]; ++q) a += el.vm[el.node_tet[q]];
        el.node_vr[i].x = a;
    }
}

// ---------------------------------------------------------------- K(c1, c2)

// Per tet: (sum of c1, vm x sum of c2).
__global__ void __launch_bounds__(kT) k_tet_K(ElemDev el, const double* __restrict__ c1, const double* __restrict__ c2,
                                              double2* __restrict__ tq) {
    const int64_t t = thread_id();
    if (t >= el.E) return;
    const int4 v = __ldg(el.tet + t);
    tq[t] = make_double2((c1[v.x] + c1[v.y]) + (c1[v.z] + c1[v.w]),
                         el.vm[t] * ((c2[v.x] + c2[v.y]) + (c2[v.z] + c2[v.w])));
}

// Per edge: (stiffness, mass and Robin part) of its entry.
__global__ void __launch_bounds__(kT) k_edge_K(ElemDev el, const double2* __restrict__ tq, const double* __restrict__ c2,
                                               double robin, double2* __restrict__ ev) {
    const int64_t e = thread_id();
    if (e >= el.NE) return;
    double st = 0.0, ma = 0.0;
    const int64_t q1 = el.edge_ptr[e + 1];
    for (int64_t q = el.edge_ptr[e]; q < q1; ++q) {
        const uint32_t code = __ldg(el.edge_tet + q);
        const int64_t t = code >> 3;
        const double2 w = __ldg(tq + t);
        st = fma(el.s[6 * t + (code & 7)], w.x, st);
        ma += w.y;
    }
    const int2 v = __ldg(el.edge + e);
    const double2 vr = el.edge_vr[e];
    ev[e] = make_double2(st, fma(vr.x, c2[v.x] + c2[v.y], ma) + robin * vr.y);
}

// Mass and Robin part of a row's diagonal: sum over its tets of vm (2 Sm + 4 mu_i).
__device__ __forceinline__ double diag_mass(const ElemDev& el, const double2* __restrict__ tq,
                                            const double* __restrict__ c2, double robin, int64_t i) {
    double a = 0.0;
    const int64_t q1 = el.node_ptr[i + 1];
    for (int64_t q = el.node_ptr[i]; q < q1; ++q) a += __ldg(&tq[__ldg(el.node_tet + q)].y);
    const double2 vr = el.node_vr[i];
    return fma(4.0 * vr.x, c2[i], 2.0 * a) + robin * vr.y;
}

// Largest value of the block into *to (non-negative doubles order like their bits; max is exact in any order).
__device__ __forceinline__ void block_max(double v, double* to) {
    __shared__ double part[kT / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kT / 32; ++w) v = fmax(v, part[w]);
        atomicMax(reinterpret_cast<unsigned long long*>(to), static_cast<unsigned long long>(__double_as_longlong(v)));
    }
}

// Rows of the sliced-ELLPACK values (padding 0), the inverse diagonal, the FP32 copies and the Gershgorin bound.
// The rows of the stiffness sum to 0, which gives its diagonal.
__global__ void __launch_bounds__(kT) k_row_K(MeshDev m, ElemDev el, const double2* __restrict__ tq,
                                              const double2* __restrict__ ev, const double* __restrict__ c2,
                                              double robin, double* __restrict__ val, float* __restrict__ val32,
                                              double* __restrict__ inv64, float* __restrict__ inv32, double* gbound) {
    const int64_t i = thread_id();
    double ratio = 0.0;
    if (i < ((int64_t(m.N) + 31) & ~int64_t(31))) {
        const int64_t p0 = m.sell_ptr[i >> 5] * 32 + (i & 31), p1 = m.sell_ptr[(i >> 5) + 1] * 32;
        double st = 0.0, off = 0.0;
        for (int64_t at = p0; at < p1; at += 32) {
            const int e = __ldg(el.ent_edge + at);
            double v = 0.0;
            if (e >= 0) {
                const double2 w = __ldg(ev + e);
                v = w.x + w.y;
                st += w.x;
                off += fabs(v);
            }
            val[at] = v;
            if (val32) val32[at] = float(v);
        }
        if (i < m.N) {
            const double d = diag_mass(el, tq, c2, robin, i) - st;
            const int64_t at = p0 + int64_t(m.sell_diag[i]) * 32;
            val[at] = d;
            if (val32) val32[at] = float(d);
            const double inv = 1.0 / d;
            inv64[i] = inv;
            if (inv32) inv32[i] = float(inv);
            ratio = 1.0 + off * inv;
        }
    }
    if (gbound) block_max(ratio, gbound);
}

// y = -K(c1, c2) x without the Robin term, for R right-hand sides, from the edge values: thread per row and chunk
// of C right-hand sides.  Taken as sum_j a_ij (x_j - x_i) + (row sum) x_i, so that the gradient of a smooth x comes
// from differences of x, as in an element-by-element product.
template <int R>
__global__ void __launch_bounds__(kT) k_rhs_jv(MeshDev m, ElemDev el, const double2* __restrict__ tq,
                                               const double2* __restrict__ ev, const double* __restrict__ c2,
                                               const double* __restrict__ x, double* __restrict__ y) {
    constexpr int C = R > 4 ? 4 : R, NCH = R / C;
    const int64_t g = thread_id();
    const int64_t i = g / NCH;
    const int c0 = int(g % NCH) * C;
    if (i >= m.N) return;
    double xi[C], acc[C], row = diag_mass(el, tq, c2, 0.0, i);
#pragma unroll
    for (int r = 0; r < C; ++r) {
        xi[r] = x[i * R + c0 + r];
        acc[r] = 0.0;
    }
    const int64_t p0 = m.sell_ptr[i >> 5] * 32 + (i & 31);
    const int len = m.sell_len[i];
    for (int k = 0; k < len; ++k) {
        const int e = __ldg(el.ent_edge + p0 + 32 * k);
        if (e < 0) continue;
        const double2 w = __ldg(ev + e);
        const double a = w.x + w.y;
        row += w.y;
        const double* xj = x + int64_t(__ldg(el.ent_col + p0 + 32 * k)) * R + c0;
#pragma unroll
        for (int r = 0; r < C; ++r) acc[r] = fma(a, xj[r] - xi[r], acc[r]);
    }
#pragma unroll
    for (int r = 0; r < C; ++r) y[i * R + c0 + r] = -fma(row, xi[r], acc[r]);
}

// ---------------------------------------------------------------- prior

// |grad u|^2 on a tet from coordinates: infinite only where it is beyond the range, never the difference of infinities.
__device__ __noinline__ double tet_grad2(const double* xyz, const double* u, int4 v) {
    const int id[4] = {v.x, v.y, v.z, v.w};
    double p[4][3], c[4][3], x[4], g[3], ad;
    for (int a = 0; a < 4; ++a) {
        for (int k = 0; k < 3; ++k) p[a][k] = xyz[3 * int64_t(id[a]) + k];
        x[a] = u[id[a]];
    }
    tet_cofactors(p, c, ad);
    grad_vec(c, x, g);
    return (g[0] * g[0] + g[1] * g[1] + g[2] * g[2]) / (ad * ad);
}

// Per tet: 4 x the lagged weight of each block.  Two weights by one division
// where their products stay well inside the range; any other field, T or size
// of tet (gradients of 1e70 and more against T) goes by the general formulas.
__global__ void __launch_bounds__(kT) k_tet_prior(ElemDev el, const double* __restrict__ xyz,
                                                  const double* __restrict__ u1,
                                                  const double* __restrict__ u2, double inv_T2, int kind, double q,
                                                  double scale1, double2* __restrict__ tq) {
    const int64_t t = thread_id();
    if (t >= el.E) return;
    const int4 v = __ldg(el.tet + t);
    double s[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) s[c] = el.s[6 * t + c];
    // |grad u|^2 = e / vm with e = -sum_ab s_ab (u_a - u_b)^2 / 30
    const double vm = el.vm[t];
    double e[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const double* u = r == 0 ? u1 : u2;
        const double x[4] = {u[v.x], u[v.y], u[v.z], u[v.w]};
        double a = 0.0;
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const double d = x[edge_a(c)] - x[edge_b(c)];
            a = fma(s[c] * d, d, a);
        }
        e[r] = a * (-1.0 / 30.0);
        if (e[r] < 0.0) e[r] = 0.0;
    }
    double w[2];
    // 1 / (1 + |grad u|^2 / T^2) = vm / (vm + e / T^2)
    const double a = fma(e[0], inv_T2, vm), b = fma(e[1], inv_T2, vm), ab = a * b;
    if (!(ab > 1e-280 && ab < 1e280)) {  // NaN too
        w[0] = 4.0 * prior_weight<double>(kind, tet_grad2(xyz, u1, v), inv_T2, q);
        w[1] = 4.0 * scale1 * prior_weight<double>(kind, tet_grad2(xyz, u2, v), inv_T2, q);
    } else if (kind == 0) {
        const double f = 4.0 * vm / ab;
        w[0] = f * b;
        w[1] = scale1 * (f * a);
    } else {
        w[0] = 4.0 * prior_weight<double>(kind, e[0] / vm, inv_T2, q);
        w[1] = 4.0 * scale1 * prior_weight<double>(kind, e[1] / vm, inv_T2, q);
    }
    tq[t] = make_double2(w[0], w[1]);
}

// Per edge of the prior's pattern: the entry of both blocks.
__global__ void __launch_bounds__(kT) k_edge_prior(ElemDev el, const double2* __restrict__ tq,
                                                   double2* __restrict__ ev) {
    const int64_t e = thread_id();
    if (e >= el.NE || !__ldg(el.in_prior + e)) return;
    double a = 0.0, b = 0.0;
    const int64_t q1 = el.edge_ptr[e + 1];
    for (int64_t q = el.edge_ptr[e]; q < q1; ++q) {
        const uint32_t code = __ldg(el.edge_tet + q);
        const int64_t t = code >> 3;
        const double2 w = __ldg(tq + t);
        const double s = el.s[6 * t + (code & 7)];
        a = fma(s, w.x, a);
        b = fma(s, w.y, b);
    }
    ev[e] = make_double2(a, b);
}

// Rows of both blocks: the stiffness diagonal is minus the row's other entries, plus delta.
__global__ void __launch_bounds__(kT) k_row_prior(MeshDev m, ElemDev el, const double2* __restrict__ ev, double delta,
                                                  double* __restrict__ val0, double* __restrict__ val1,
                                                  double* __restrict__ inv64, float* __restrict__ inv32,
                                                  double* gbound) {
    const int64_t i = thread_id();
    double ratio = 0.0;
    if (i < ((int64_t(m.N) + 31) & ~int64_t(31))) {
        const int64_t p0 = m.sell_ptr[i >> 5] * 32 + (i & 31), p1 = m.sell_ptr[(i >> 5) + 1] * 32;
        double sa = 0.0, sb = 0.0, oa = 0.0, ob = 0.0;
        for (int64_t at = p0; at < p1; at += 32) {
            const int e = __ldg(el.pent_edge + at);
            double2 w = make_double2(0.0, 0.0);
            if (e >= 0) {
                w = __ldg(ev + e);
                sa += w.x;
                sb += w.y;
                oa += fabs(w.x);
                ob += fabs(w.y);
            }
            val0[at] = w.x;
            val1[at] = w.y;
        }
        if (i < m.N) {
            const int64_t at = p0 + int64_t(m.sell_diag[i]) * 32;
            const double da = delta - sa, db = delta - sb;
            val0[at] = da;
            val1[at] = db;
            const double ia = 1.0 / da, ib = 1.0 / db;
            inv64[2 * i] = ia;
            inv64[2 * i + 1] = ib;
            if (inv32) {
                inv32[2 * i] = float(ia);
                inv32[2 * i + 1] = float(ib);
            }
            ratio = fmax(1.0 + oa * ia, 1.0 + ob * ib);
        }
    }
    if (gbound) block_max(ratio, gbound);
}

// ---------------------------------------------------------------- J^T
//   y_i0 = -sum_k sum_T (|T| / 4) grad f_k . grad z_k      = sum_T sum_ab s_ab E_ab
//   y_i1 = -sum_k (M(f_k) z_k)_i = -[ sum_T vm (sum_ab P_ab + 2 sum_a D_a) + sum_ij (sum vm) P_ij + 4 (sum vm) D_i ]
// with, over the K right-hand sides, E_ab = sum_k (f_a - f_b)(z_a - z_b), P_ab = sum_k (f_a z_b + f_b z_a) per edge
// and D_a = sum_k f_a z_a per node.  The sums over k are taken once per edge (7 a node on Kuhn meshes) instead of
// once per tet and vertex (24 a node): ~290 K/8 FP64 operations a node.

template <int R>
__global__ void __launch_bounds__(kT) k_edge_vjp(MeshDev m, ElemDev el, const double* __restrict__ f,
                                                 const double* __restrict__ z, double2* __restrict__ ep,
                                                 double* __restrict__ dn) {
    constexpr int C = R > 8 ? 8 : R, NCH = R / C;
    const int64_t i = thread_id();
    if (i >= m.N) return;
    double fi[C], zi[C], d = 0.0;
    auto own = [&](int c) {
#pragma unroll
        for (int r = 0; r < C; ++r) {
            fi[r] = f[i * R + c * C + r];
            zi[r] = z[i * R + c * C + r];
        }
    };
    for (int c = 0; c < NCH; ++c) {
        own(c);
#pragma unroll
        for (int r = 0; r < C; ++r) d = fma(fi[r], zi[r], d);
    }
    dn[i] = d;
    const int64_t p0 = m.sell_ptr[i >> 5] * 32 + (i & 31);
    const int len = m.sell_len[i];
    for (int k = 0; k < len; ++k) {
        const int64_t j = __ldg(el.ent_col + p0 + 32 * k);
        if (j <= i) continue;
        double e = 0.0, p = 0.0;
        for (int c = 0; c < NCH; ++c) {
            if (NCH > 1) own(c);
            const double* fj = f + j * R + c * C;
            const double* zj = z + j * R + c * C;
#pragma unroll
            for (int r = 0; r < C; ++r) {
                const double a = fj[r], b = zj[r];
                e = fma(a - fi[r], b - zi[r], e);
                p = fma(fi[r], b, fma(a, zi[r], p));
            }
        }
        ep[__ldg(el.ent_edge + p0 + 32 * k)] = make_double2(e, p);
    }
}

__global__ void __launch_bounds__(kT) k_tet_vjp(ElemDev el, const double2* __restrict__ ep,
                                                const double* __restrict__ dn, double2* __restrict__ tq) {
    const int64_t t = thread_id();
    if (t >= el.E) return;
    const int4 v = __ldg(el.tet + t);
    double g = 0.0, p = 2.0 * ((dn[v.x] + dn[v.y]) + (dn[v.z] + dn[v.w]));
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const double2 w = __ldg(ep + __ldg(el.tet_edge + 6 * t + c));
        g = fma(el.s[6 * t + c], w.x, g);
        p += w.y;
    }
    tq[t] = make_double2(g, el.vm[t] * p);
}

__global__ void __launch_bounds__(kT) k_row_vjp(MeshDev m, ElemDev el, const double2* __restrict__ ep,
                                                const double* __restrict__ dn, const double2* __restrict__ tq,
                                                double* __restrict__ y) {
    const int64_t i = thread_id();
    if (i >= m.N) return;
    double a = 0.0, b = 4.0 * el.node_vr[i].x * dn[i];
    const int64_t p0 = m.sell_ptr[i >> 5] * 32 + (i & 31);
    const int len = m.sell_len[i];
    for (int k = 0; k < len; ++k) {
        const int e = __ldg(el.ent_edge + p0 + 32 * k);
        if (e >= 0) b = fma(el.edge_vr[e].x, __ldg(&ep[e].y), b);
    }
    const int64_t q1 = el.node_ptr[i + 1];
    for (int64_t q = el.node_ptr[i]; q < q1; ++q) {
        const double2 w = __ldg(tq + __ldg(el.node_tet + q));
        a += w.x;
        b += w.y;
    }
    *reinterpret_cast<double2*>(y + 2 * i) = make_double2(a, -b);
}

}  // namespace

cudaError_t launch_element_geometry(const MeshDev& m, const ElemDev& el, cudaStream_t s) {
    note_launch(2);
    k_geometry<<<blocks(el.E), kT, 0, s>>>(el, m.xyz64);
    k_geometry_sums<<<blocks(std::max<int64_t>(el.NE, m.N)), kT, 0, s>>>(el, m.N);
    return cudaGetLastError();
}

cudaError_t launch_assemble_K(const MeshDev& m, const ElemDev& el, const ElemScratch& w, const double* kappa,
                              const double* mu, double* val, float* val32, double* inv64, float* inv32, cudaStream_t s,
                              double* gbound) {
    if (gbound) {
        const cudaError_t e = cudaMemsetAsync(gbound, 0, sizeof(double), s);
        if (e != cudaSuccess) return e;
    }
    note_launch(3);
    k_tet_K<<<blocks(el.E), kT, 0, s>>>(el, kappa, mu, w.tet);
    k_edge_K<<<blocks(el.NE), kT, 0, s>>>(el, w.tet, mu, 1.0, w.edge);
    k_row_K<<<blocks(m.N), kT, 0, s>>>(m, el, w.tet, w.edge, mu, 1.0, val, val32, inv64, inv32, gbound);
    return cudaGetLastError();
}

cudaError_t launch_assemble_prior(const MeshDev& m, const ElemDev& el, const ElemScratch& w, const double* u1,
                                  const double* u2, double inv_T2, int kind, double q, double scale1, double delta,
                                  double* val0, double* val1, double* inv64, float* inv32, cudaStream_t s,
                                  double* gbound) {
    if (gbound) {
        const cudaError_t e = cudaMemsetAsync(gbound, 0, sizeof(double), s);
        if (e != cudaSuccess) return e;
    }
    note_launch(3);
    k_tet_prior<<<blocks(el.E), kT, 0, s>>>(el, m.xyz64, u1, u2, inv_T2, kind, q, scale1, w.tet);
    k_edge_prior<<<blocks(el.NE), kT, 0, s>>>(el, w.tet, w.edge);
    k_row_prior<<<blocks(m.N), kT, 0, s>>>(m, el, w.edge, delta, val0, val1, inv64, inv32, gbound);
    return cudaGetLastError();
}

cudaError_t launch_rhs_jv(const MeshDev& m, const ElemDev& el, const ElemScratch& w, int R, const double* c1,
                          const double* c2, const double* x, double* y, cudaStream_t s) {
    note_launch(3);
    k_tet_K<<<blocks(el.E), kT, 0, s>>>(el, c1, c2, w.tet);
    k_edge_K<<<blocks(el.NE), kT, 0, s>>>(el, w.tet, c2, 0.0, w.edge);
    switch (R) {
        case 1: k_rhs_jv<1><<<blocks(m.N), kT, 0, s>>>(m, el, w.tet, w.edge, c2, x, y); break;
        case 2: k_rhs_jv<2><<<blocks(m.N), kT, 0, s>>>(m, el, w.tet, w.edge, c2, x, y); break;
        case 4: k_rhs_jv<4><<<blocks(m.N), kT, 0, s>>>(m, el, w.tet, w.edge, c2, x, y); break;
        case 8: k_rhs_jv<8><<<blocks(int64_t(m.N) * 2), kT, 0, s>>>(m, el, w.tet, w.edge, c2, x, y); break;
        case 16: k_rhs_jv<16><<<blocks(int64_t(m.N) * 4), kT, 0, s>>>(m, el, w.tet, w.edge, c2, x, y); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_vjp_accum(const MeshDev& m, const ElemDev& el, const ElemScratch& w, double* node, int R,
                             const double* phi, const double* z, double* y, cudaStream_t s) {
    note_launch(3);
    switch (R) {
        case 1: k_edge_vjp<1><<<blocks(m.N), kT, 0, s>>>(m, el, phi, z, w.edge, node); break;
        case 2: k_edge_vjp<2><<<blocks(m.N), kT, 0, s>>>(m, el, phi, z, w.edge, node); break;
        case 4: k_edge_vjp<4><<<blocks(m.N), kT, 0, s>>>(m, el, phi, z, w.edge, node); break;
        case 8: k_edge_vjp<8><<<blocks(m.N), kT, 0, s>>>(m, el, phi, z, w.edge, node); break;
        case 16: k_edge_vjp<16><<<blocks(m.N), kT, 0, s>>>(m, el, phi, z, w.edge, node); break;
        default: return cudaErrorInvalidValue;
    }
    k_tet_vjp<<<blocks(el.E), kT, 0, s>>>(el, w.edge, node, w.tet);
    k_row_vjp<<<blocks(m.N), kT, 0, s>>>(m, el, w.edge, node, w.tet, y);
    return cudaGetLastError();
}

}  // namespace qpat
