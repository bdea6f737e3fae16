// BF16 tensor-core kernels of the 3D U-Net (see unet_kernels.cuh).
#include <algorithm>

#include "unet_kernels.cuh"

namespace qpat {
namespace unet {

namespace {

using bf16 = __nv_bfloat16;

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ uint32_t ld32(const bf16* p) { return *reinterpret_cast<const uint32_t*>(p); }

__device__ __forceinline__ uint32_t pack2(bf16 lo, bf16 hi) {
    return uint32_t(__bfloat16_as_ushort(lo)) | (uint32_t(__bfloat16_as_ushort(hi)) << 16);
}

// neighbour of linear voxel v = (z, y, x) across tap, or -1 outside the grid
__device__ __forceinline__ int nbr(int z, int y, int x, int tap, int n) {
    const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
    const int zz = z + dz, yy = y + dy, xx = x + dx;
    if (zz < 0 || yy < 0 || xx < 0 || zz >= n || yy >= n || xx >= n) return -1;
    return (zz * n + yy) * n + xx;
}

constexpr int kConvWarps = 8;  // 128 voxels per CTA

// out[v][co] = act( bias[co] + sum_{tap, ci} in[nbr(v, tap)][ci] * w[tap][co][ci] )
template <int NT>
__global__ void __launch_bounds__(kConvWarps * 32) k_conv_fwd(const bf16* __restrict__ in, int Cin,
                                                              const bf16* __restrict__ w,
                                                              const float* __restrict__ bias, int Cout, int relu,
                                                              bf16* __restrict__ out, float* __restrict__ out32,
                                                              int n) {
    extern __shared__ uint32_t sw[];  // one tap: Cout rows of (Cin + 8) bf16
    const int nvox = n * n * n;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int v0 = (blockIdx.x * kConvWarps + warp) * 16;
    const bool live = v0 < nvox;
    const int rA = v0 + g, rB = v0 + g + 8;
    const int zA = rA / (n * n), yA = (rA / n) % n, xA = rA % n;
    const int zB = rB / (n * n), yB = (rB / n) % n, xB = rB % n;
    const int ldw = (Cin + 8) / 2;
    const int cw = Cin / 2;
    float acc[NT][4];
#pragma unroll
    for (int i = 0; i < NT; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
    for (int tap = 0; tap < 27; ++tap) {
        __syncthreads();
        const uint32_t* wt = reinterpret_cast<const uint32_t*>(w + size_t(tap) * Cout * Cin);
        for (int i = threadIdx.x; i < Cout * cw; i += blockDim.x) sw[(i / cw) * ldw + (i % cw)] = wt[i];
        __syncthreads();
        if (!live) continue;
        const int nA = rA < nvox ? nbr(zA, yA, xA, tap, n) : -1;
        const int nB = rB < nvox ? nbr(zB, yB, xB, tap, n) : -1;
        const bf16* pA = in + size_t(nA < 0 ? 0 : nA) * Cin + 2 * t;
        const bf16* pB = in + size_t(nB < 0 ? 0 : nB) * Cin + 2 * t;
        for (int c0 = 0; c0 < Cin; c0 += 16) {
            uint32_t a[4];
            a[0] = nA >= 0 ? ld32(pA + c0) : 0u;
            a[1] = nB >= 0 ? ld32(pB + c0) : 0u;
            a[2] = nA >= 0 ? ld32(pA + c0 + 8) : 0u;
            a[3] = nB >= 0 ? ld32(pB + c0 + 8) : 0u;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const uint32_t* row = sw + (nt * 8 + g) * ldw + c0 / 2 + t;
                const uint32_t b[2] = {row[0], row[4]};
                mma_bf16(acc[nt], a, b);
            }
        }
    }
    if (!live) return;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        const int co = nt * 8 + 2 * t;
        const float b0 = bias ? bias[co] : 0.f, b1 = bias ? bias[co + 1] : 0.f;
        float v[4] = {acc[nt][0] + b0, acc[nt][1] + b1, acc[nt][2] + b0, acc[nt][3] + b1};
        if (relu)
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = fmaxf(v[k], 0.f);
        if (rA < nvox) {
            *reinterpret_cast<uint32_t*>(out + size_t(rA) * Cout + co) =
                pack2(__float2bfloat16(v[0]), __float2bfloat16(v[1]));
            if (out32) {
                out32[size_t(rA) * Cout + co] = v[0];
                out32[size_t(rA) * Cout + co + 1] = v[1];
            }
        }
        if (rB < nvox) {
            *reinterpret_cast<uint32_t*>(out + size_t(rB) * Cout + co) =
                pack2(__float2bfloat16(v[2]), __float2bfloat16(v[3]));
            if (out32) {
                out32[size_t(rB) * Cout + co] = v[2];
                out32[size_t(rB) * Cout + co + 1] = v[3];
            }
        }
    }
}

template <int NT>
cudaError_t conv_fwd_t(const bf16* in, int Cin, const bf16* w, const float* bias, int Cout, int relu, bf16* out,
                       float* out32, int n, cudaStream_t s) {
    const size_t smem = sizeof(uint32_t) * size_t(Cout) * ((Cin + 8) / 2);
    cudaError_t e = qpat::allow_smem((const void*)k_conv_fwd<NT>, size_t(smem));
    if (e != cudaSuccess) return e;
    const int nvox = n * n * n;
    const int grid = (nvox + 16 * kConvWarps - 1) / (16 * kConvWarps);
    qpat::note_launch(1);
    k_conv_fwd<NT><<<grid, kConvWarps * 32, smem, s>>>(in, Cin, w, bias, Cout, relu, out, out32, n);
    return cudaGetLastError();
}

// Weight gradient: partial[chunk][tap][co][ci] = sum_{v in chunk} dy[v][co] in[nbr(v, tap)][ci]
// and, from the centre tap's CTAs, bias[chunk][co] = sum dy[v][co].  A CTA
// takes a chunk of voxels, a tap and 16 output channels; 64 voxels at a time
// are copied to shared memory (16-byte cp.async, zeros outside the grid, the
// next 64 under the current ones' MMAs), and each warp multiplies 16 of them:
// both operands lie voxel by voxel, so their fragments come by transposed
// ldmatrix.  Chunks are sized so that the CTAs fill the GPU (a grid of 4^3
// voxels as well as one of 128^3); their sums are added in order by
// k_sum_chunks.  Bound: shared-memory and L2 reads of `in`, once per tap.
constexpr int kWgThreads = 128, kWgStep = 64;
constexpr int kWgradVoxMin = 256, kWgradVoxMax = 8192;

int64_t wgrad_chunk_voxels(int64_t voxels, int Cout) {
    int64_t c = kWgradVoxMax;
    while (c > kWgradVoxMin && (voxels + c - 1) / c * 27 * (Cout / 16) < 1024) c /= 2;
    return c;
}

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const bf16* p) {
    const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p));
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}

__device__ __forceinline__ void copy16(bf16* dst, const bf16* src, bool ok) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
}

// v / d for v < 2^31 by a multiplication (Granlund and Montgomery 1994)
struct FastDiv {
    uint32_t d, m, s;
    explicit FastDiv(uint32_t div) : d(div), m(0), s(0) {
        while ((uint64_t(1) << s) < d) ++s;
        m = uint32_t(((uint64_t(1) << 32) * ((uint64_t(1) << s) - d)) / d + 1);
    }
    __device__ __forceinline__ uint32_t div(uint32_t v) const { return (__umulhi(m, v) + v) >> s; }
};

// The same 16 bytes from an address that is a multiple of a bf16's size only.
__device__ __forceinline__ void copy_bf16(bf16* dst, const bf16* src, bool ok) {
    for (int e = 0; e < 8; ++e) dst[e] = ok ? src[e] : __float2bfloat16(0.f);
}

// kAligned: in and dy lie on 16-byte boundaries (a caller's tensors need not)
template <int NCI, bool kAligned>
__global__ void __launch_bounds__(kWgThreads) k_conv_wgrad(const bf16* __restrict__ in, const bf16* __restrict__ dy,
                                                           int Cout, float* __restrict__ partial,
                                                           float* __restrict__ bias, int n, FastDiv dn, int64_t voxels,
                                                           int64_t chunk_voxels) {
    constexpr int Cin = 8 * NCI, LI = Cin + 8, LD = 16 + 8;  // padded rows: fragment rows fall into different banks
    extern __shared__ __align__(16) unsigned char wg_smem[];
    bf16* sIn = reinterpret_cast<bf16*>(wg_smem);         // 2 x kWgStep x LI
    bf16* sDy = sIn + 2 * kWgStep * LI;                   // 2 x kWgStep x LD
    __shared__ float red[16][Cin + 1];
    const int chunk = blockIdx.x, tap = blockIdx.y, co0 = blockIdx.z * 16;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int64_t vbeg = chunk * chunk_voxels, vend = min(voxels, vbeg + chunk_voxels);
    const int64_t shift = (int64_t(tap / 9 - 1) * n + (tap / 3 % 3 - 1)) * n + (tap % 3 - 1);
    auto copy = [](bf16* dst, const bf16* src, bool ok) {
        if constexpr (kAligned)
            copy16(dst, src, ok);
        else
            copy_bf16(dst, src, ok);
    };
    auto load = [&](int64_t v0, int st) {
        for (int i = threadIdx.x; i < kWgStep * NCI; i += kWgThreads) {
            const int64_t v = v0 + i / NCI;
            bool ok = v < vend;
            if (ok) {
                const uint32_t q = dn.div(uint32_t(v)), r = dn.div(q), w = dn.div(r);  // rows, planes, samples before v
                const int x = int(uint32_t(v) - q * n) + tap % 3 - 1, y = int(q - r * n) + tap / 3 % 3 - 1,
                          z = int(r - w * n) + tap / 9 - 1;
                ok = x >= 0 && y >= 0 && z >= 0 && x < n && y < n && z < n;
            }
            copy(sIn + (st * kWgStep + i / NCI) * LI + i % NCI * 8, ok ? in + (v + shift) * Cin + i % NCI * 8 : in, ok);
        }
        for (int i = threadIdx.x; i < kWgStep * 2; i += kWgThreads) {
            const int64_t v = v0 + i / 2;
            const bool ok = v < vend;
            copy(sDy + (st * kWgStep + i / 2) * LD + i % 2 * 8, ok ? dy + v * Cout + co0 + i % 2 * 8 : dy, ok);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[NCI][4];
#pragma unroll
    for (int i = 0; i < NCI; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
    float db = 0.f;
    load(vbeg, 0);
    int st = 0;
    for (int64_t v0 = vbeg; v0 < vend; v0 += kWgStep, st ^= 1) {
        load(v0 + kWgStep, st ^ 1);  // past the end: zeros
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        const bf16* d = sDy + (st * kWgStep + warp * 16) * LD;
        const bf16* x = sIn + (st * kWgStep + warp * 16) * LI;
        // the four 8 x 8 blocks of a 16 (voxels) x 16 (channels) tile, transposed: lane l addresses row l % 8 of block l / 8
        const int vr = lane & 7, hi8 = (lane >> 3) & 1, hi16 = lane >> 4;
        uint32_t a[4];
        ldsm4t(a, d + (vr + 8 * hi16) * LD + 8 * hi8);  // A[co][v]: blocks (co 0-7, v 0-7), (co 8-15, v 0-7), (.., v 8-15)
#pragma unroll
        for (int c = 0; c < NCI; c += 2) {
            uint32_t b[4];
            ldsm4t(b, x + (vr + 8 * hi8) * LI + 8 * (c + hi16));  // B[v][ci]: (v 0-7, v 8-15) of ci block c, then of c + 1
            const uint32_t b0[2] = {b[0], b[1]}, b1[2] = {b[2], b[3]};
            mma_bf16(acc[c], a, b0);
            mma_bf16(acc[c + 1], a, b1);
        }
        if (tap == 13) {
            const int co = threadIdx.x & 15, part = threadIdx.x >> 4;
            for (int v = part; v < kWgStep; v += kWgThreads / 16) db += __bfloat162float(sDy[(st * kWgStep + v) * LD + co]);
        }
        __syncthreads();
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    // reduce the 4 warps in turn: C fragment rows co (g, g+8), columns ci (2t, 2t+1)
    for (int w = 0; w < 4; ++w) {
        if (warp == w) {
#pragma unroll
            for (int nc = 0; nc < NCI; ++nc) {
                const int c = nc * 8 + 2 * t;
                red[g][c] = (w ? red[g][c] : 0.f) + acc[nc][0];
                red[g][c + 1] = (w ? red[g][c + 1] : 0.f) + acc[nc][1];
                red[g + 8][c] = (w ? red[g + 8][c] : 0.f) + acc[nc][2];
                red[g + 8][c + 1] = (w ? red[g + 8][c + 1] : 0.f) + acc[nc][3];
            }
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < 16 * Cin; i += blockDim.x) {
        const int r = i / Cin, c = i % Cin;
        partial[((size_t(chunk) * 27 + tap) * Cout + co0 + r) * Cin + c] = red[r][c];
    }
    if (tap == 13) {
        __syncthreads();
        float* part = &red[0][0];  // 16 x (Cin + 1) floats, 128 of them used
        part[threadIdx.x] = db;
        __syncthreads();
        if (threadIdx.x < 16) {
            float s = 0.f;
            for (int k = 0; k < kWgThreads / 16; ++k) s += part[16 * k + threadIdx.x];
            bias[size_t(chunk) * Cout + co0 + threadIdx.x] = s;
        }
    }
}

// dw (27 Cout Cin) and db (Cout): sums over the chunks in order, added to what is there when add is set
__global__ void k_sum_chunks(const float* __restrict__ partial, const float* __restrict__ bias, int chunks, int64_t count,
                             int Cout, int add, float* __restrict__ dw, float* __restrict__ db) {
    const int64_t total = count + (db ? Cout : 0);
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
        const bool w = i < count;
        const float* src = w ? partial + i : bias + (i - count);
        const int64_t stride = w ? count : Cout;
        float* to = w ? dw + i : db + (i - count);
        float s = 0.f;
        for (int c = 0; c < chunks; ++c) s += src[c * stride];
        *to = add ? *to + s : s;
    }
}

template <int NCI>
cudaError_t wgrad_t(const bf16* in, const bf16* dy, int Cout, float* partial, float* bias, int n, int64_t voxels,
                    int64_t chunk, cudaStream_t s) {
    const size_t smem = sizeof(bf16) * 2 * kWgStep * size_t(8 * NCI + 8 + 16 + 8);
    const bool aligned = ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(dy)) & 15) == 0;
    const auto kernel = aligned ? k_conv_wgrad<NCI, true> : k_conv_wgrad<NCI, false>;
    const cudaError_t e = qpat::allow_smem((const void*)kernel, smem);
    if (e != cudaSuccess) return e;
    const dim3 grid(unsigned((voxels + chunk - 1) / chunk), 27, unsigned(Cout / 16));
    qpat::note_launch(1);
    kernel<<<grid, kWgThreads, smem, s>>>(in, dy, Cout, partial, bias, n, FastDiv(uint32_t(n)), voxels, chunk);
    return cudaGetLastError();
}

__global__ void k_flip(const bf16* w, int Cin, int Cout, bf16* wt) {
    const int64_t total = int64_t(27) * Cin * Cout;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
        // wt[tap][ci][co] = w[26 - tap][co][ci]
        const int tap = int(i / (int64_t(Cin) * Cout));
        const int rem = int(i % (int64_t(Cin) * Cout));
        const int ci = rem / Cout, co = rem % Cout;
        wt[i] = w[(size_t(26 - tap) * Cout + co) * Cin + ci];
    }
}

// The element-wise kernels take 8 channels (16 bytes) a thread; every channel
// count of the network is a multiple of 8.  Bound by HBM.
struct Oct {
    float f[8];
};
__device__ __forceinline__ Oct ld8(const bf16* p) {
    const uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
    Oct o;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        o.f[2 * k] = __uint_as_float(w[k] << 16);
        o.f[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
    }
    return o;
}
__device__ __forceinline__ void st8(bf16* p, const Oct& o) {
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) w[k] = pack2(__float2bfloat16(o.f[2 * k]), __float2bfloat16(o.f[2 * k + 1]));
    *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
}
#define FOR_OCT(total) \
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < (total); i += int64_t(gridDim.x) * blockDim.x)

__global__ void k_relu_mask(bf16* dy, const bf16* y, int64_t count) {
    FOR_OCT(count / 8) {
        const uint4 u = __ldg(reinterpret_cast<const uint4*>(y) + i);
        uint4 d = reinterpret_cast<uint4*>(dy)[i];
        auto keep = [](uint32_t v, uint32_t g) {  // halves of g whose v is above 0
            return (__uint_as_float(v << 16) > 0.f ? g & 0xffffu : 0u) |
                   (__uint_as_float(v & 0xffff0000u) > 0.f ? g & 0xffff0000u : 0u);
        };
        d = make_uint4(keep(u.x, d.x), keep(u.y, d.y), keep(u.z, d.z), keep(u.w, d.w));
        reinterpret_cast<uint4*>(dy)[i] = d;
    }
}

// The pooling and concatenation kernels take B samples as one grid of B n planes: n is even, so no pair of planes
// straddles two samples.
__global__ void k_avgpool(const bf16* in, int C, int n, int B, bf16* out) {
    const int m = n / 2, c8 = C / 8;
    FOR_OCT(int64_t(m) * m * m * c8 * B) {
        const int c = int(i % c8) * 8;
        const int64_t v = i / c8;
        const int x = int(v % m), y = int(v / m % m);
        const int64_t z = v / (int64_t(m) * m);
        Oct s{};
        for (int d = 0; d < 8; ++d) {
            const Oct q = ld8(in + (((2 * z + (d >> 2)) * n + 2 * y + ((d >> 1) & 1)) * n + 2 * x + (d & 1)) * C + c);
#pragma unroll
            for (int k = 0; k < 8; ++k) s.f[k] += q.f[k];
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) s.f[k] *= 0.125f;
        st8(out + v * C + c, s);
    }
}

__global__ void k_avgpool_bwd(const bf16* dout, int C, int n, int B, bf16* din, int accumulate) {
    const int m = n / 2, c8 = C / 8;
    FOR_OCT(int64_t(n) * n * n * c8 * B) {
        const int c = int(i % c8) * 8;
        const int64_t v = i / c8;
        const int x = int(v % n), y = int(v / n % n);
        const int64_t z = v / (int64_t(n) * n);
        Oct g = ld8(dout + (((z / 2) * m + y / 2) * m + x / 2) * C + c);
        Oct old{};
        if (accumulate) old = ld8(din + v * C + c);
#pragma unroll
        for (int k = 0; k < 8; ++k) g.f[k] = accumulate ? 0.125f * g.f[k] + old.f[k] : 0.125f * g.f[k];
        st8(din + v * C + c, g);
    }
}

__global__ void k_upcat(const bf16* lo, int Clo, const bf16* skip, int Cs, int n, int B, bf16* cat) {
    const int m = n / 2, C = Clo + Cs, c8 = C / 8;
    FOR_OCT(int64_t(n) * n * n * c8 * B) {
        const int c = int(i % c8) * 8;
        const int64_t v = i / c8;
        const bf16* src = skip + v * Cs + (c - Clo);
        if (c < Clo) {
            const int x = int(v % n), y = int(v / n % n);
            const int64_t z = v / (int64_t(n) * n);
            src = lo + (((z / 2) * m + y / 2) * m + x / 2) * Clo + c;
        }
        reinterpret_cast<uint4*>(cat)[i] = __ldg(reinterpret_cast<const uint4*>(src));
    }
}

__global__ void k_upcat_bwd_lo(const bf16* dcat, int Clo, int Cs, int n, int B, bf16* dlo) {
    const int m = n / 2, C = Clo + Cs, c8 = Clo / 8;
    FOR_OCT(int64_t(m) * m * m * c8 * B) {
        const int c = int(i % c8) * 8;
        const int64_t v = i / c8;
        const int x = int(v % m), y = int(v / m % m);
        const int64_t z = v / (int64_t(m) * m);
        Oct s{};
        for (int d = 0; d < 8; ++d) {
            const Oct q = ld8(dcat + (((2 * z + (d >> 2)) * n + 2 * y + ((d >> 1) & 1)) * n + 2 * x + (d & 1)) * C + c);
#pragma unroll
            for (int k = 0; k < 8; ++k) s.f[k] += q.f[k];
        }
        st8(dlo + v * Clo + c, s);
    }
}

__global__ void k_upcat_bwd_skip(const bf16* dcat, int Clo, int Cs, int n, int B, bf16* dskip, int accumulate) {
    const int C = Clo + Cs, c8 = Cs / 8;
    FOR_OCT(int64_t(n) * n * n * c8 * B) {
        const int c = int(i % c8) * 8;
        const int64_t v = i / c8;
        Oct g = ld8(dcat + v * C + Clo + c);
        if (accumulate) {
            const Oct old = ld8(dskip + v * Cs + c);
#pragma unroll
            for (int k = 0; k < 8; ++k) g.f[k] += old.f[k];
        }
        st8(dskip + v * Cs + c, g);
    }
}

__global__ void k_adam(float* w, bf16* wb, const float* g, float* m, float* v, int64_t count, float lr, float b1,
                       float b2, float eps, float c1, float c2) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < count; i += int64_t(gridDim.x) * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        w[i] = wi;
        if (wb) wb[i] = __float2bfloat16(wi);
    }
}

__global__ void k_f2b(const float* in, bf16* out, int64_t count) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < count; i += int64_t(gridDim.x) * blockDim.x)
        out[i] = __float2bfloat16(in[i]);
}

__global__ void k_b2f(const bf16* in, float* out, int64_t count) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < count; i += int64_t(gridDim.x) * blockDim.x)
        out[i] = __bfloat162float(in[i]);
}

int grid1d(int64_t n) {
    return int(std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16)));
}

}  // namespace

static int g_conv_engine = 0;
void set_conv_engine(int engine) { g_conv_engine = engine; }
int conv_engine() { return g_conv_engine; }

cudaError_t conv3d_fwd(const bf16* in, int Cin, const bf16* w, const float* bias, int Cout, int relu, bf16* out,
                       float* out32, int n, cudaStream_t s) {
    if (Cin % 16 || Cout % 8 || n % 2) return cudaErrorInvalidValue;
    if (g_conv_engine == 0 && conv3d_fwd_tc_supported(Cin, Cout))
        return conv3d_fwd_tc(ConvInput{in, Cin}, w, bias, Cout, relu, ConvOutput{out, out32}, n, 1, s);
    switch (Cout / 8) {
        case 1: return conv_fwd_t<1>(in, Cin, w, bias, Cout, relu, out, out32, n, s);
        case 2: return conv_fwd_t<2>(in, Cin, w, bias, Cout, relu, out, out32, n, s);
        case 4: return conv_fwd_t<4>(in, Cin, w, bias, Cout, relu, out, out32, n, s);
        case 6: return conv_fwd_t<6>(in, Cin, w, bias, Cout, relu, out, out32, n, s);
        case 8: return conv_fwd_t<8>(in, Cin, w, bias, Cout, relu, out, out32, n, s);
        case 12: return conv_fwd_t<12>(in, Cin, w, bias, Cout, relu, out, out32, n, s);
        case 16: return conv_fwd_t<16>(in, Cin, w, bias, Cout, relu, out, out32, n, s);
        case 24: return conv_fwd_t<24>(in, Cin, w, bias, Cout, relu, out, out32, n, s);
        default: return cudaErrorInvalidValue;
    }
}

size_t wgrad_scratch(int n, int Cin, int Cout, int B) {
    const int64_t voxels = int64_t(n) * n * n * B, chunk = wgrad_chunk_voxels(voxels, Cout);
    return size_t((voxels + chunk - 1) / chunk) * (size_t(27) * Cin * Cout + size_t(Cout));
}

cudaError_t conv3d_wgrad(const bf16* in, int Cin, const bf16* dy, int Cout, float* dw, float* db, float* partial,
                         int n, int B, int add, cudaStream_t s) {
    if (Cin % 8 || Cout % 16 || (n * n * n) % 16) return cudaErrorInvalidValue;
    if (int64_t(n) * n * n * B >= int64_t(1) << 31) return cudaErrorInvalidValue;  // 32-bit voxel numbers
    const int64_t voxels = int64_t(n) * n * n * B, chunk = wgrad_chunk_voxels(voxels, Cout);
    const int chunks = int((voxels + chunk - 1) / chunk);
    const int64_t count = int64_t(27) * Cout * Cin;
    float* bias = partial + chunks * count;
    cudaError_t e = cudaErrorInvalidValue;
    switch (Cin / 8) {
        case 2: e = wgrad_t<2>(in, dy, Cout, partial, bias, n, voxels, chunk, s); break;
        case 4: e = wgrad_t<4>(in, dy, Cout, partial, bias, n, voxels, chunk, s); break;
        case 6: e = wgrad_t<6>(in, dy, Cout, partial, bias, n, voxels, chunk, s); break;
        case 8: e = wgrad_t<8>(in, dy, Cout, partial, bias, n, voxels, chunk, s); break;
        case 12: e = wgrad_t<12>(in, dy, Cout, partial, bias, n, voxels, chunk, s); break;
        case 16: e = wgrad_t<16>(in, dy, Cout, partial, bias, n, voxels, chunk, s); break;
        case 24: e = wgrad_t<24>(in, dy, Cout, partial, bias, n, voxels, chunk, s); break;
        default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    qpat::note_launch(1);
    k_sum_chunks<<<grid1d(count + Cout), 256, 0, s>>>(partial, bias, chunks, count, Cout, add, dw, db);
    return cudaGetLastError();
}

cudaError_t flip_weights(const bf16* w, int Cin, int Cout, bf16* w_t, cudaStream_t s) {
    qpat::note_launch(1);
    k_flip<<<grid1d(int64_t(27) * Cin * Cout), 256, 0, s>>>(w, Cin, Cout, w_t);
    return cudaGetLastError();
}

cudaError_t relu_mask(bf16* dy, const bf16* y, int64_t count, cudaStream_t s) {
    qpat::note_launch(1);
    k_relu_mask<<<grid1d(count / 8), 256, 0, s>>>(dy, y, count);
    return cudaGetLastError();
}

cudaError_t avgpool(const bf16* in, int C, int n, int B, bf16* out, cudaStream_t s) {
    qpat::note_launch(1);
    k_avgpool<<<grid1d(int64_t(n / 2) * (n / 2) * (n / 2) * C / 8 * B), 256, 0, s>>>(in, C, n, B, out);
    return cudaGetLastError();
}

cudaError_t avgpool_bwd(const bf16* dout, int C, int n, int B, bf16* din, int accumulate, cudaStream_t s) {
    qpat::note_launch(1);
    k_avgpool_bwd<<<grid1d(int64_t(n) * n * n * C / 8 * B), 256, 0, s>>>(dout, C, n, B, din, accumulate);
    return cudaGetLastError();
}

cudaError_t upcat(const bf16* lo, int Clo, const bf16* skip, int Cs, int n, int B, bf16* cat, cudaStream_t s) {
    qpat::note_launch(1);
    k_upcat<<<grid1d(int64_t(n) * n * n * (Clo + Cs) / 8 * B), 256, 0, s>>>(lo, Clo, skip, Cs, n, B, cat);
    return cudaGetLastError();
}

cudaError_t upcat_bwd(const bf16* dcat, int Clo, int Cs, int n, int B, bf16* dlo, bf16* dskip, int accumulate_skip,
                      cudaStream_t s) {
    qpat::note_launch(1);
    k_upcat_bwd_lo<<<grid1d(int64_t(n / 2) * (n / 2) * (n / 2) * Clo / 8 * B), 256, 0, s>>>(dcat, Clo, Cs, n, B, dlo);
    qpat::note_launch(1);
    k_upcat_bwd_skip<<<grid1d(int64_t(n) * n * n * Cs / 8 * B), 256, 0, s>>>(dcat, Clo, Cs, n, B, dskip, accumulate_skip);
    return cudaGetLastError();
}

cudaError_t adam(float* w, bf16* wb, const float* g, float* m, float* v, int64_t count, float lr, float b1, float b2,
                 float eps, int step, cudaStream_t s) {
    const float c1 = 1.f - powf(b1, float(step)), c2 = 1.f - powf(b2, float(step));
    qpat::note_launch(1);
    k_adam<<<grid1d(count), 256, 0, s>>>(w, wb, g, m, v, count, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

cudaError_t f32_to_bf16(const float* in, bf16* out, int64_t count, cudaStream_t s) {
    qpat::note_launch(1);
    k_f2b<<<grid1d(count), 256, 0, s>>>(in, out, count);
    return cudaGetLastError();
}

cudaError_t bf16_to_f32(const bf16* in, float* out, int64_t count, cudaStream_t s) {
    qpat::note_launch(1);
    k_b2f<<<grid1d(count), 256, 0, s>>>(in, out, count);
    return cudaGetLastError();
}

}  // namespace unet
}  // namespace qpat
