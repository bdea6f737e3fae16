// 3x3x3 BF16 convolution of the U-Net on the 5th-generation tensor cores
// (tcgen05.mma, accumulator in tensor memory), the forward kernel the
// U-Net's inference and data-gradient passes use on sm_100-class GPUs.
//
// Implicit GEMM: D[128 voxels][Cout] += A_tap[128 voxels][Cin] x B_tap[Cin][Cout]
// over 27 taps, without gathering a tile per tap.  A CTA loads the input of a
// Tx x Ty x Tz box of voxels with its halo once into shared memory, laid out
// as [8-channel chunk][voxel of the padded box] in 16-byte units: the
// canonical no-swizzle K-major layout (8 rows x 16 bytes) with its row groups
// 128 bytes apart, so that consecutive voxels are consecutive rows.  A tap is
// then a shift of the start address by its distance in the padded box, and
// any 128 consecutive voxels of the box form the rows of one MMA; rows that
// fall on the padding are computed and dropped.  Weights ([Cout][Cin] per tap,
// the same layout) stay in shared memory when all 27 taps take at most
// kResident bytes, else they are streamed through a ring of taps.  One thread
// of a warp issues the MMAs (M = 128, N = Cout, K = 16) of the warp's 128-row
// tiles, taps in order and channels in order within a tap, into the tile's
// own columns of tensor memory; the halo arrives in three groups of planes, and the taps
// of a plane start when it has arrived.  Each warp then reads its quarter of
// the lanes with tcgen05.ld, adds the bias, applies ReLU and stores.
// The input may be the concatenation of an upsampled coarser grid and a skip
// tensor, read directly from both.
//
// Bound: an MMA with few output channels reads its 4 KB of A at 128 bytes a
// cycle (32 cycles) whatever N is, so a layer takes at least
// 27 Cin / 16 x 32 cycles per 128 voxels; the form before this one copied
// 27 x 128 rows per tile and waited for each copy.
//
// Tensor memory is allocated by warp 0 and freed on every exit path.  A wait
// that gives up writes NaN into the tiles (the caller's parity checks see it)
// and counts the event in g_tc_timeouts.
#include <algorithm>
#include <array>
#include <cstdint>
#include <map>
#include <mutex>

#include "unet_kernels.cuh"

namespace qpat {
namespace unet {

namespace {

using bf16 = __nv_bfloat16;

constexpr int kTcThreads = 256;
constexpr int kTcRows = 128;  // MMA M
constexpr int kResident = 64 * 1024;  // weights kept in shared memory as a whole
constexpr int kTcSmem = 220 * 1024;   // dynamic shared memory a CTA may take
constexpr long long kTcSpin = 1LL << 22;

__device__ int g_tc_timeouts;

__device__ __forceinline__ uint32_t s_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// shared-memory matrix descriptor: no swizzle, K-major; lbo = byte distance
// of K-adjacent core matrices, sbo = byte distance of 8-row groups
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= uint64_t((addr & 0x3FFFF) >> 4);          // bits  0-13: start address / 16
    d |= uint64_t((lbo & 0x3FFFF) >> 4) << 16;     // bits 16-29: leading byte offset / 16
    d |= uint64_t((sbo & 0x3FFFF) >> 4) << 32;     // bits 32-45: stride byte offset / 16
    d |= uint64_t(1) << 46;                        // bits 46-47: descriptor version (sm_100)
    return d;                                      // base offset 0, no swizzle
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major
__host__ __device__ constexpr uint32_t instr_desc(int M, int N) {
    return (1u << 4)                      // D format: F32
           | (1u << 7)                    // A format: BF16
           | (1u << 10)                   // B format: BF16
           | (uint32_t(N >> 3) << 17)     // N / 8
           | (uint32_t(M >> 4) << 24);    // M / 16
}

__device__ __forceinline__ bool mbar_wait_parity(uint64_t* bar, uint32_t parity) {
    for (long long i = 0; i < kTcSpin; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(s_addr(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// 16 bytes into shared memory, zeros where ok is false (src stays a valid address)
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Geometry of a launch (host and device).
struct TcBox {
    int n, Tx, Ty, Tz;
    int P, RY;          // padded row (Tx + 2), padded rows per plane (Ty + 2)
    int tiles;          // 128-row tiles per CTA
    int lbo;            // bytes between 8-channel chunks of the halo
    int wlbo, wtap;     // bytes between chunks of a tap's weights, bytes of a tap
    int stages;         // 27: weights resident; else the ring's taps
    int ncols;          // tensor-memory columns
    int nx, ny;         // boxes along x and y
};

struct TcArgs {
    TcBox g;
    const bf16* skip;   // n^3 x Cskip per sample
    const bf16* lo;     // (n / 2)^3 x Clo per sample in front of it, or nullptr
    int Cskip, Clo;
    const bf16* w;
    const float* bias;
    int Cout, relu;
    bf16* out;          // may be nullptr
    float* out32;       // may be nullptr
    float* first;       // channel 0 only (n^3 floats per sample), or nullptr
    int first_exp;      //   its exponential
};

__global__ void __launch_bounds__(kTcThreads) k_conv_fwd_tc(const TcArgs a) {
    extern __shared__ __align__(128) unsigned char tc_smem[];
    __shared__ uint64_t mbar[3];
    __shared__ uint32_t tmem_base_s;
    const TcBox& g = a.g;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = g.n, Cin = a.Clo + a.Cskip, kc = Cin / 8, lc = a.Clo / 8;
    const int x0 = int(blockIdx.x % g.nx) * g.Tx, y0 = int(blockIdx.x / g.nx) * g.Ty, z0 = int(blockIdx.y) * g.Tz;
    const int64_t nvox = int64_t(n) * n * n, sample = blockIdx.z;
    unsigned char* sA = tc_smem;
    unsigned char* sW = sA + size_t(kc) * g.lbo;
    const uint32_t uA = s_addr(sA), uW = s_addr(sW);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_addr(&tmem_base_s)),
                     "r"(g.ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < 3; ++i)  // one arrival per issuing warp
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s_addr(&mbar[i])), "r"(min(g.tiles, kTcThreads / 32))
                         : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }

    // halo planes [p0, p1) of the box: a warp per padded row, 16 bytes per lane
    auto load_planes = [&](int p0, int p1) {
        const bf16* skip = a.skip + sample * nvox * a.Cskip;
        const bf16* lo = a.lo ? a.lo + sample * (nvox >> 3) * a.Clo : nullptr;
        const int m = n >> 1, dx = 32 / kc, dc = 32 % kc;
        for (int row = p0 * g.RY + warp; row < p1 * g.RY; row += kTcThreads / 32) {
            const int z = z0 + row / g.RY - 1, y = y0 + row % g.RY - 1;
            const bool in = z >= 0 && z < n && y >= 0 && y < n;
            int x = lane / kc, c = lane % kc;
            for (; x < g.P; ) {
                const int xx = x0 + x - 1;
                const bool ok = in && xx >= 0 && xx < n;
                const void* src = a.skip;
                if (ok)
                    src = c < lc ? static_cast<const void*>(lo + ((int64_t(z >> 1) * m + (y >> 1)) * m + (xx >> 1)) * a.Clo + c * 8)
                                 : static_cast<const void*>(skip + ((int64_t(z) * n + y) * n + xx) * a.Cskip + (c - lc) * 8);
                cp16(uA + uint32_t(c * g.lbo + (row * g.P + x) * 16), src, ok);
                x += dx;
                c += dc;
                if (c >= kc) {
                    c -= kc;
                    ++x;
                }
            }
        }
    };
    auto load_weights = [&](int tap, int stage) {
        const bf16* src = a.w + size_t(tap) * a.Cout * Cin;
        const uint32_t dst = uW + uint32_t(stage * g.wtap);
        for (int i = threadIdx.x; i < a.Cout * kc; i += kTcThreads)
            cp16(dst + uint32_t((i % kc) * g.wlbo + (i / kc) * 16), src + size_t(i) * 8, true);
    };
    const bool resident = g.stages == 27;
    load_planes(0, g.Tz);
    if (resident) {
        for (int t = 0; t < 27; ++t) load_weights(t, t);
        cp_commit();
        load_planes(g.Tz, g.Tz + 1);
        cp_commit();
        load_planes(g.Tz + 1, g.Tz + 2);
        cp_commit();
    } else {
        load_planes(g.Tz, g.Tz + 2);
        load_weights(0, 0);
        cp_commit();
        load_weights(1, 1);
        cp_commit();
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_s;
    const uint32_t idesc = instr_desc(kTcRows, a.Cout);

    // MMAs of one tap.  Issuing one takes a thread far longer than the tensor core takes to run it at N = 16 when the
    // descriptors are built anew (150 cycles against 32), so the tiles go round the warps (a tile's MMAs stay with one
    // thread and in order) and a descriptor is its predecessor plus a constant in the address field.
    const int issuers = min(g.tiles, kTcThreads / 32);
    const bool issuer = lane == 0 && warp < issuers;
    const uint64_t descA = smem_desc(uA, uint32_t(g.lbo), 128u), descB = smem_desc(uW, uint32_t(g.wlbo), 128u);
    const uint32_t stepA = uint32_t(2 * g.lbo) >> 4, stepB = uint32_t(2 * g.wlbo) >> 4;
    auto issue = [&](int tap, int stage) {
        const uint64_t da0 = descA + uint32_t((tap / 9 * g.RY + tap / 3 % 3) * g.P + tap % 3);
        const uint64_t db0 = descB + (uint32_t(stage * g.wtap) >> 4);
        for (int t = warp; t < g.tiles; t += issuers) {
            uint64_t da = da0 + uint32_t(t * kTcRows), db = db0;
            const uint32_t d = tmem + uint32_t(t * a.Cout);
            uint32_t acc = tap > 0 ? 1u : 0u;
            for (int k = 0; k < Cin / 16; ++k) {
                asm volatile(
                    "{\n\t.reg .pred p;\n\t"
                    "setp.ne.b32 p, %4, 0;\n\t"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
                    "l"(da), "l"(db), "r"(idesc), "r"(acc)
                    : "memory");
                da += stepA;
                db += stepB;
                acc = 1u;
            }
        }
    };
    auto commit = [&](int i) {
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s_addr(&mbar[i]))
                     : "memory");
    };
    // this thread's copies have arrived -> visible to the tensor core (async proxy) for everybody; false (in every
    // thread) once a wait of some thread has given up
    bool mine = true;
    auto publish = [&]() -> bool {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        const bool all = __syncthreads_and(mine);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        return all;
    };
    if (resident) {
        for (int dz = 0; dz < 3; ++dz) {
            if (dz == 0) cp_wait<2>();
            else if (dz == 1) cp_wait<1>();
            else cp_wait<0>();
            publish();
            if (issuer) {
                for (int t = 0; t < 9; ++t) issue(9 * dz + t, 9 * dz + t);
                if (dz == 2) commit(0);
            }
        }
        mine = mbar_wait_parity(&mbar[0], 0u);
    } else {
        // ring of 2 or 3 taps; completion of tap t is phase t / stages of mbar[t % stages]
        const int S = g.stages;
        int tap = 0;
        for (; tap < 27; ++tap) {
            cp_wait<1>();
            if (!publish()) break;
            if (issuer) {
                issue(tap, tap % S);
                commit(tap % S);
            }
            const int next = tap + 2;  // goes to the stage of tap next - S, whose MMAs must have read it
            if (next >= S && next < 27 && !mbar_wait_parity(&mbar[(next - S) % S], uint32_t(((next - S) / S) & 1))) mine = false;
            if (next < 27) load_weights(next, next % S);
            cp_commit();
        }
        cp_wait<0>();
        // the last taps' MMAs (or, after a give-up, those in flight) finish before TMEM is read and freed
        for (int t = max(0, tap - S); t < tap; ++t)
            if (!mbar_wait_parity(&mbar[t % S], uint32_t((t / S) & 1))) mine = false;
    }
    const bool ok = __syncthreads_and(mine);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    // ---- epilogue: warps w and w + 4 own TMEM lanes 32 (w % 4) .. + 31 and take the tiles in turn
    if (!ok && threadIdx.x == 0) atomicAdd(&g_tc_timeouts, 1);
    for (int t = warp >> 2; t < g.tiles; t += 2) {
        const int p = t * kTcRows + (warp & 3) * 32 + lane;
        const int x = p % g.P, y = p / g.P % g.RY, z = p / (g.P * g.RY);
        const bool valid = x < g.Tx && y < g.Ty && z < g.Tz && x0 + x < n && y0 + y < n && z0 + z < n;
        const int64_t v = sample * nvox + (int64_t(z0 + z) * n + (y0 + y)) * n + x0 + x;
        for (int c0 = 0; c0 < a.Cout; c0 += 16) {
            uint32_t r[16];
            const uint32_t taddr = tmem + (uint32_t((warp & 3) * 32) << 16) + uint32_t(t * a.Cout + c0);
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                "[%16];"
                : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                  "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                  "=r"(r[15])
                : "r"(taddr)
                : "memory");
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (!valid) continue;
            float f[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                float q = ok ? __uint_as_float(r[j]) : __int_as_float(0x7fc00000);
                if (a.bias) q += __ldg(a.bias + c0 + j);
                if (a.relu) q = fmaxf(q, 0.f);
                f[j] = q;
            }
            if (a.first && c0 == 0) a.first[v] = a.first_exp ? expf(f[0]) : f[0];
            if (a.out) {
                uint32_t packed[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * j], f[2 * j + 1]);
                    packed[j] = *reinterpret_cast<const uint32_t*>(&h);
                }
                uint4* o = reinterpret_cast<uint4*>(a.out + v * a.Cout + c0);
                o[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
                o[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
            }
            if (a.out32) {
                float4* o32 = reinterpret_cast<float4*>(a.out32 + v * a.Cout + c0);
#pragma unroll
                for (int j = 0; j < 4; ++j) o32[j] = make_float4(f[4 * j], f[4 * j + 1], f[4 * j + 2], f[4 * j + 3]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(g.ncols) : "memory");
}

// The box of a launch with the least estimated time per SM: whole waves of
// CTAs, each its halo's bytes at ~48 a cycle, its MMAs at 32 cycles (more
// above 128 output channels) and its stores; two CTAs share an SM where their
// shared memory (<= half) lets one's loads run under the other's MMAs.
// false: no box fits.
bool search_box(int n, int Cin, int Cout, int B, TcBox& best, size_t& best_smem) {
    const int kc = Cin / 8;
    const int wlbo = Cout * 16 + 16, wtap = kc * wlbo;
    double best_t = 0.0;
    bool found = false;
    for (int sx = 0; sx < 10; ++sx) {
        const int Tx = (n + (1 << sx) - 1) >> sx;
        if (sx > 0 && Tx < 8) break;
        for (int Tz : {1, 2, 4, 8})
            for (int Ty = 1; Ty <= std::min(n, 64); ++Ty) {
                if (Tz > n && Tz > 1) continue;
                TcBox g{};
                g.n = n;
                g.Tx = Tx;
                g.Ty = Ty;
                g.Tz = Tz;
                g.P = Tx + 2;
                g.RY = Ty + 2;
                const int span = ((Tz - 1) * g.RY + Ty - 1) * g.P + Tx;
                g.tiles = (span + kTcRows - 1) / kTcRows;
                if (g.tiles * Cout > 512) break;
                // every row that an MMA reads (the last tap shifts the last tile by this much) lies in the buffer
                const int rows = std::max((Tz + 2) * g.RY * g.P, g.tiles * kTcRows + (2 * g.RY + 2) * g.P + 2);
                g.lbo = (rows * 16 + 127) / 128 * 128 + 64;
                g.wlbo = wlbo;
                g.wtap = wtap;
                g.stages = 27 * wtap <= kResident ? 27 : 3;
                size_t smem = size_t(kc) * g.lbo + size_t(g.stages) * wtap;
                if (smem > size_t(kTcSmem) && g.stages == 3) {
                    g.stages = 2;
                    smem -= wtap;
                }
                if (smem > size_t(kTcSmem)) break;
                g.ncols = 32;
                while (g.ncols < g.tiles * Cout) g.ncols *= 2;
                g.nx = (n + Tx - 1) / Tx;
                g.ny = (n + Ty - 1) / Ty;
                const double ctas = double(g.nx) * g.ny * ((n + Tz - 1) / Tz) * B;
                const int share = smem <= size_t(kTcSmem) / 2 && g.ncols <= 256 ? 2 : 1;
                const double mma = g.tiles * 27.0 * (Cin / 16) * std::max(32.0, Cout / 4.0);
                const double load = ((Tz + 2.0) * g.RY * g.P * Cin * 2 + 27.0 * wtap) / 48.0 + 1500.0;
                const double store = g.tiles * 128.0 * Cout * 2 / 32.0 + 500.0;
                const double waves = std::max(1.0, double(int64_t((ctas + 152 * share - 1) / (152 * share))));
                const double t = waves * (share == 2 ? std::max(2 * mma, mma + load + store) : mma + load + store);
                if (!found || t < best_t) {
                    found = true;
                    best_t = t;
                    best = g;
                    best_smem = smem;
                }
            }
    }
    return found;
}

// The search's answers by shape (a function of the shape alone); the table starts afresh when it grows beyond a
// program's handful of layers.
bool choose_box(int n, int Cin, int Cout, int B, TcBox& box, size_t& smem) {
    struct Found {
        bool ok;
        TcBox box;
        size_t smem;
    };
    static std::mutex mu;
    static std::map<std::array<int, 4>, Found> known;
    std::lock_guard<std::mutex> lock(mu);
    const std::array<int, 4> key{n, Cin, Cout, B};
    auto it = known.find(key);
    if (it == known.end()) {
        if (known.size() >= 1024) known.clear();
        Found f{};
        f.ok = search_box(n, Cin, Cout, B, f.box, f.smem);
        it = known.emplace(key, f).first;
    }
    box = it->second.box;
    smem = it->second.smem;
    return it->second.ok;
}

}  // namespace

bool conv3d_fwd_tc_supported(int Cin, int Cout) {
    // M = 128 needs N = Cout a multiple of 16 in [16, 256]; K steps of 16; the smallest box (8 x 1 x 1) with two taps
    // of weights fits whenever this bound holds
    return Cin % 16 == 0 && Cout % 16 == 0 && Cout >= 16 && Cout <= 256 &&
           2 * (size_t(kTcRows) * Cin * 2 + size_t(Cout) * Cin * 2) <= 200 * 1024;
}

cudaError_t conv3d_fwd_tc(const ConvInput& in, const bf16* w, const float* bias, int Cout, int relu, const ConvOutput& out,
                          int n, int B, cudaStream_t s) {
    const int Cin = in.Clo + in.Cskip;
    TcArgs a{};
    size_t smem = 0;
    if (!conv3d_fwd_tc_supported(Cin, Cout) || in.Clo % 8 || in.Cskip % 8 || B < 1 || B > 65535 || n > 65535 ||
        !choose_box(n, Cin, Cout, B, a.g, smem))
        return cudaErrorInvalidValue;
    cudaError_t e = qpat::allow_smem((const void*)k_conv_fwd_tc, smem);
    if (e != cudaSuccess) return e;
    a.skip = in.skip;
    a.lo = in.lo;
    a.Cskip = in.Cskip;
    a.Clo = in.Clo;
    a.w = w;
    a.bias = bias;
    a.Cout = Cout;
    a.relu = relu;
    a.out = out.bf;
    a.out32 = out.f32;
    a.first = out.first;
    a.first_exp = out.first_exp;
    qpat::note_launch(1);
    k_conv_fwd_tc<<<dim3(unsigned(a.g.nx * a.g.ny), unsigned((n + a.g.Tz - 1) / a.g.Tz), unsigned(B)), kTcThreads, smem, s>>>(a);
    return cudaGetLastError();
}

int tc_timeouts() {
    int h = 0;
    cudaMemcpyFromSymbol(&h, g_tc_timeouts, sizeof(int));
    return h;
}

}  // namespace unet
}  // namespace qpat
