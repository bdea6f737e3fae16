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
// kResident bytes, else they are streamed through a ring of taps.  A warp's
// elected lane issues the MMAs (M = 128, N = Cout, K = 16) of the warp's 128-row
// tiles, taps in order and channels in order within a tap, into the tile's
// own columns of tensor memory.  Each warp then reads its quarter of the lanes
// with tcgen05.ld, adds the bias, applies ReLU and stores.
// The input may be the concatenation of an upsampled coarser grid and a skip
// tensor, read directly from both.
//
// Bound: an MMA with few output channels reads its 4 KB of A at 128 bytes a
// cycle (32 cycles) whatever N is, so a layer takes at least
// 27 Cin / 16 x 32 cycles per 128 voxels: 49 us for 16 -> 16 channels at 128^3.
// Measured there, one sample: MMAs alone 75 us over the empty kernel's 26, copies
// alone 62, stores 23, together 137 (one box per CTA and no overlap: 192);
// 48 -> 16: 374 (651); 64^3, 32 -> 32: 48 (97); 64^3, 96 -> 32, streamed: 212 (341).
// With boxes chosen by those rates and a ring of four taps, 8 samples through all
// layers at 128^3 went from 11.2 to 8.9 ms; eight issuing warps instead of four: 9.0.
//
// Tensor memory is allocated by warp 0 and freed on every exit path, after the
// MMAs in flight are done (or have been waited for as long as any wait lasts).
// A wait that gives up counts the event in g_tc_timeouts and writes NaN into the
// tiles (0 behind a ReLU, whose maximum with 0 drops it).
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
    int tiles;          // 128-row tiles per box
    int lbo;            // bytes between 8-channel chunks of the halo
    int wlbo, wtap;     // bytes between chunks of a tap's weights, bytes of a tap
    int stages;         // 27: weights resident; else the ring's taps
    int ncols;          // tensor-memory columns
    int nx, ny, nz;     // boxes along x, y, z
    int boxes;          // of all samples
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

struct Corner {
    int x, y, z, sample;
};
__device__ __forceinline__ Corner corner_of(const TcBox& g, int box) {
    Corner c;
    c.x = box % g.nx * g.Tx;
    box /= g.nx;
    c.y = box % g.ny * g.Ty;
    box /= g.ny;
    c.z = box % g.nz * g.Tz;
    c.sample = box / g.nz;
    return c;
}

// One tensor's rows of the halo, kt 16-byte chunks a voxel, to shared address dst.  A row of voxels lies in one piece in memory, so a lane's address
// advances by 32 chunks; up = 1: the row of the grid of half the side, every
// voxel twice.
__device__ __forceinline__ void load_rows(const TcBox& g, const Corner& c, const bf16* t, int kt, int up, uint32_t dst) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n = g.n, m = n >> up;
    const int dx = 32 / kt, dk = 32 % kt, x0 = lane / kt, q0 = lane % kt;
    const int xa = c.x == 0 ? 1 : 0, xb = min(g.P, n - c.x + 1);  // padded columns inside the grid
    const bf16* base = t + int64_t(c.sample) * m * m * m * kt * 8;
    for (int row = warp; row < (g.Tz + 2) * g.RY; row += kTcThreads / 32) {
        const int z = c.z + row / g.RY - 1, y = c.y + row % g.RY - 1;
        const bool in = z >= 0 && z < n && y >= 0 && y < n;
        const bf16* src = base + (in ? (int64_t(z >> up) * m + (y >> up)) * m * kt * 8 : 0);
        const uint32_t to = dst + uint32_t(row * g.P * 16);
        for (int x = x0, q = q0; x < g.P;) {
            const bool ok = in && x >= xa && x < xb;
            cp16(to + uint32_t(q * g.lbo + x * 16), src + (ok ? (((c.x + x - 1) >> up) * kt + q) * 8 : 0), ok);
            x += dx;
            q += dk;
            if (q >= kt) {
                q -= kt;
                ++x;
            }
        }
    }
}

// The halo of box c to shared address dst.
__device__ __forceinline__ void load_halo(const TcArgs& a, const Corner& c, uint32_t dst) {
    if (a.Clo) load_rows(a.g, c, a.lo, a.Clo / 8, 1, dst);
    load_rows(a.g, c, a.skip, a.Cskip / 8, 0, dst + uint32_t(a.Clo / 8 * a.g.lbo));
}

// Weights of taps [t0, t0 + taps) to shared address dst.
__device__ __forceinline__ void load_weights(const TcArgs& a, int t0, int taps, uint32_t dst) {
    const int kc = (a.Clo + a.Cskip) / 8, per = a.Cout * kc;
    const bf16* src = a.w + size_t(t0) * per * 8;
    for (int i = threadIdx.x; i < taps * per; i += kTcThreads) {
        const int tap = i / per, j = i - tap * per, row = j / kc;
        cp16(dst + uint32_t(tap * a.g.wtap + (j - row * kc) * a.g.wlbo + row * 16), src + size_t(i) * 8, true);
    }
}

// The results of box c from tensor memory: warps w and w + 4 own lanes 32 (w % 4) .. + 31 and take the tiles in turn.
__device__ __forceinline__ void store_box(const TcArgs& a, const Corner& c, uint32_t tmem, bool ok) {
    const TcBox& g = a.g;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n = g.n;
    const int64_t nvox = int64_t(n) * n * n;
    for (int t = warp >> 2; t < g.tiles; t += kTcThreads / 128) {
        const int p = t * kTcRows + (warp & 3) * 32 + lane;
        const int x = p % g.P, y = p / g.P % g.RY, z = p / (g.P * g.RY);
        const bool valid = x < g.Tx && y < g.Ty && z < g.Tz && c.x + x < n && c.y + y < n && c.z + z < n;
        const int64_t v = c.sample * nvox + (int64_t(c.z + z) * n + (c.y + y)) * n + c.x + x;
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
}

__device__ __forceinline__ void tmem_alloc(uint32_t* base, int ncols) {  // one warp
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_addr(base)), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t base, int ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(ncols) : "memory");
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s_addr(bar)) : "memory");
}
// Executed by a whole warp, issued by its elected lane: bar completes a phase when that lane's MMAs so far are done.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(s_addr(bar))
        : "memory");
}
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void to_async_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// The MMAs of one tap for tiles first, first + step, ... of a box, by one warp:
// every lane walks the loop with warp-uniform values and the elected one
// issues, so that the descriptors stay in uniform registers (a single lane
// that builds them takes 100 to 200 cycles an MMA, several times what the
// tensor core takes at N = 16); each descriptor is its predecessor plus a
// constant in the address field.
struct TapIssue {
    uint64_t descA, descB;
    uint32_t stepA, stepB, idesc;
    __device__ TapIssue(const TcArgs& a, uint32_t uA, uint32_t uW)
        : descA(smem_desc(uA, uint32_t(a.g.lbo), 128u)), descB(smem_desc(uW, uint32_t(a.g.wlbo), 128u)),
          stepA(uint32_t(2 * a.g.lbo) >> 4), stepB(uint32_t(2 * a.g.wlbo) >> 4), idesc(instr_desc(kTcRows, a.Cout)) {}
    __device__ __forceinline__ void operator()(const TcArgs& a, int tap, uint32_t halo_off, uint32_t w_off, uint32_t acc_at,
                                               int first, int step) const {
        const TcBox& g = a.g;
        const int ks = (a.Clo + a.Cskip) / 16;
        const uint64_t da0 = descA + (halo_off >> 4) + uint32_t((tap / 9 * g.RY + tap / 3 % 3) * g.P + tap % 3);
        const uint64_t db0 = descB + (w_off >> 4);
        for (int t = first; t < g.tiles; t += step) {
            uint64_t da = da0 + uint32_t(t * kTcRows), db = db0;
            const uint32_t d = acc_at + uint32_t(t * a.Cout);
            uint32_t acc = tap > 0 ? 1u : 0u;
            for (int k = 0; k < ks; ++k) {
                asm volatile(
                    "{\n\t.reg .pred p, q;\n\t"
                    "elect.sync _|q, 0xffffffff;\n\t"
                    "setp.ne.b32 p, %4, 0;\n\t"
                    "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
                    "l"(da), "l"(db), "r"(idesc), "r"(acc)
                    : "memory");
                da += stepA;
                db += stepB;
                acc = 1u;
            }
        }
    }
};

// Resident weights: a CTA goes through its boxes with two halos and two sets of
// accumulators.  Eight warps copy halos and store results; four more only issue
// MMAs (a thread that issues waits while the tensor core's queue is full, so it
// cannot be one that copies).  Box `it` uses halo, accumulators and barriers
// it % 2: full (its halo is there), done (its MMAs are over), stored (its
// accumulators have been read).  Every wait is bounded; once one gives up, no
// thread waits again and what is stored is NaN.
constexpr int kIssueWarps = 4;
constexpr int kStayThreads = kTcThreads + 32 * kIssueWarps;

__global__ void __launch_bounds__(kStayThreads) k_conv_fwd_tc_stay(const TcArgs a) {
    extern __shared__ __align__(128) unsigned char tc_smem[];
    __shared__ uint64_t full[2], done[2], stored[2], drained[kIssueWarps];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int gave_up;
    const TcBox& g = a.g;
    const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0);  // warp-uniform for the compiler
    const int halo = (a.Clo + a.Cskip) / 8 * g.lbo, set = g.tiles * a.Cout;
    const uint32_t uA = s_addr(tc_smem), uW = uA + uint32_t(halo * 2);
    if (warp == 0) tmem_alloc(&tmem_base_s, g.ncols);
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&full[i], kTcThreads);
            mbar_init(&done[i], kIssueWarps);
            mbar_init(&stored[i], kTcThreads);
        }
        for (int i = 0; i < kIssueWarps; ++i) mbar_init(&drained[i], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        gave_up = 0;
    }
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_base_s, 0);
    auto wait = [&](uint64_t* bar, int phase) {
        if (!gave_up && !mbar_wait_parity(bar, uint32_t(phase & 1))) {
            gave_up = 1;
            atomicAdd(&g_tc_timeouts, 1);
        }
    };
    const int boxes = g.boxes, stride = int(gridDim.x), mine = int(blockIdx.x);
    const int count = mine < boxes ? (boxes - 1 - mine) / stride + 1 : 0;
    if (warp >= kTcThreads / 32) {
        const TapIssue issue(a, uA, uW);
        for (int it = 0; it < count; ++it) {
            const int buf = it & 1;
            wait(&full[buf], it >> 1);
            if (it >= 2) wait(&stored[buf], (it >> 1) - 1);
            __syncwarp();
            tc_after();
            for (int t = 0; t < 27; ++t)
                issue(a, t, uint32_t(buf * halo), uint32_t(t * g.wtap), tmem + uint32_t(buf * set), warp - kTcThreads / 32,
                      kIssueWarps);
            mma_commit(&done[buf]);
        }
    } else {
        load_halo(a, corner_of(g, mine), uA);
        load_weights(a, 0, 27, uW);
        cp_commit();
        for (int it = 0; it <= count; ++it) {
            const int buf = it & 1;
            if (it < count) {
                cp_wait<0>();
                to_async_proxy();
                mbar_arrive(&full[buf]);
            }
            if (it > 0) {
                wait(&done[buf ^ 1], (it - 1) >> 1);
                tc_after();
            }
            if (it + 1 < count) {
                load_halo(a, corner_of(g, mine + (it + 1) * stride), uA + uint32_t((buf ^ 1) * halo));
                cp_commit();
            }
            if (it > 0) {
                store_box(a, corner_of(g, mine + (it - 1) * stride), tmem + uint32_t((buf ^ 1) * set), !gave_up);
                tc_before();
                mbar_arrive(&stored[buf ^ 1]);
            }
        }
    }
    tc_before();
    __syncthreads();
    if (gave_up) {  // nobody has waited for the MMAs since: they end before tensor memory is freed
        if (warp >= kTcThreads / 32) {
            uint64_t* const end = &drained[warp - kTcThreads / 32];
            mma_commit(end);
            if (!mbar_wait_parity(end, 0u)) atomicAdd(&g_tc_timeouts, 1);
        }
        __syncthreads();
    }
    if (warp == 0) tmem_free(tmem, g.ncols);
}

// Streamed weights: one box per CTA, a ring of 2 to 4 taps (with 4, the stage that a copy goes to was read by the
// MMAs of two taps ago, so that nothing waits for the tap just issued); the tiles go round
// the warps (a tile's MMAs stay with one lane, in order).
__global__ void __launch_bounds__(kTcThreads) k_conv_fwd_tc(const TcArgs a) {
    extern __shared__ __align__(128) unsigned char tc_smem[];
    __shared__ uint64_t mbar[4];
    __shared__ uint32_t tmem_base_s;
    const TcBox& g = a.g;
    const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0);
    const int halo = (a.Clo + a.Cskip) / 8 * g.lbo;
    const uint32_t uA = s_addr(tc_smem), uW = uA + uint32_t(halo);
    const int issuers = min(g.tiles, kTcThreads / 32);
    const bool issuer = warp < issuers;
    if (warp == 0) tmem_alloc(&tmem_base_s, g.ncols);
    if (threadIdx.x == 0) {
        for (int i = 0; i < 4; ++i) mbar_init(&mbar[i], issuers);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const Corner at = corner_of(g, blockIdx.x);
    load_halo(a, at, uA);
    load_weights(a, 0, 1, uW);
    cp_commit();
    load_weights(a, 1, 1, uW + uint32_t(g.wtap));
    cp_commit();
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_base_s, 0);
    const TapIssue issue(a, uA, uW);
    // completion of tap t is phase t / S of mbar[t % S]; a thread whose wait gives up says so at the next barrier,
    // where all leave together
    const int S = g.stages;
    bool mine = true;
    int tap = 0;
    for (; tap < 27; ++tap) {
        cp_wait<1>();
        to_async_proxy();
        if (!__syncthreads_and(mine)) break;
        if (issuer) {
            tc_after();
            issue(a, tap, 0u, uint32_t(tap % S * g.wtap), tmem, warp, issuers);
            mma_commit(&mbar[tap % S]);
        }
        const int next = tap + 2;  // goes to the stage of tap next - S, whose MMAs must have read it
        if (next >= S && next < 27 && !mbar_wait_parity(&mbar[(next - S) % S], uint32_t(((next - S) / S) & 1))) mine = false;
        if (next < 27) load_weights(a, next, 1, uW + uint32_t(next % S * g.wtap));
        cp_commit();
    }
    cp_wait<0>();
    // the last taps' MMAs (or, after a give-up, those in flight) finish before TMEM is read and freed
    for (int t = max(0, tap - S); t < tap; ++t)
        if (!mbar_wait_parity(&mbar[t % S], uint32_t((t / S) & 1))) mine = false;
    const bool good = __syncthreads_and(mine);
    tc_after();
    if (!good && threadIdx.x == 0) atomicAdd(&g_tc_timeouts, 1);
    store_box(a, at, tmem, good);
    tc_before();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, g.ncols);
}

// The box of a launch with the least estimated time, in cycles as measured at
// 128^3 (16 -> 16 and 48 -> 16 channels, one part at a time): an MMA 40 (more
// above 160 output channels), but a warp issues one every 118, halos come in at
// 13 bytes a cycle, results leave at 16.  Resident weights: per box the larger
// of the MMAs and the copies with their waits; streamed: the sum, ~8,000 for a
// CTA's start and its first tap and, where the ring has fewer than 4 taps,
// ~1,000 a tap for the MMAs that a copy waits for; two CTAs share an SM where
// their shared memory allows.  false: no box fits.
bool search_box(int n, int Cin, int Cout, int B, TcBox& best, size_t& best_smem) {
    const int kc = Cin / 8;
    const int wlbo = Cout * 16 + 16, wtap = kc * wlbo;
    const bool stay = 27 * wtap <= kResident;
    double best_t = 0.0;
    bool found = false;
    for (int sx = 0; sx < 10; ++sx) {
        const int Tx = (n + (1 << sx) - 1) >> sx;
        if (sx > 0 && Tx < 8) break;
        for (int Tz : {1, 2, 3, 4, 6, 8})
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
                const int cols = g.tiles * Cout * (stay ? 2 : 1);
                if (cols > 512) break;
                // every row that an MMA reads (the last tap shifts the last tile by this much) lies in the buffer
                const int rows = std::max((Tz + 2) * g.RY * g.P, g.tiles * kTcRows + (2 * g.RY + 2) * g.P + 2);
                g.lbo = (rows * 16 + 127) / 128 * 128 + 64;
                g.wlbo = wlbo;
                g.wtap = wtap;
                g.stages = stay ? 27 : 4;
                size_t smem = size_t(kc) * g.lbo * (stay ? 2 : 1) + size_t(g.stages) * wtap;
                while (smem > size_t(kTcSmem) && !stay && g.stages > 2) {
                    --g.stages;
                    smem -= wtap;
                }
                if (smem > size_t(kTcSmem)) break;
                g.ncols = 32;
                while (g.ncols < cols) g.ncols *= 2;
                g.nx = (n + Tx - 1) / Tx;
                g.ny = (n + Ty - 1) / Ty;
                g.nz = (n + Tz - 1) / Tz;
                const double boxes = double(g.nx) * g.ny * g.nz * B;
                if (boxes >= 2147483648.0) continue;
                g.boxes = int(boxes);
                const int issuers = stay ? kIssueWarps : kTcThreads / 32;
                const double mma = 27.0 * (Cin / 16) * std::max(g.tiles * std::max(40.0, Cout / 4.0),
                                                                118.0 * ((g.tiles + issuers - 1) / issuers));
                const double load = (Tz + 2.0) * g.RY * g.P * Cin * 2 / 13.0 + 800.0;
                const double store = g.tiles * 128.0 * Cout * 2 / 16.0 + 300.0;
                const int share = !stay && smem <= size_t(kTcSmem) / 2 && g.ncols <= 256 ? 2 : 1;
                const double waves = std::max(1.0, double(int64_t((boxes + 152 * share - 1) / (152 * share))));
                const double tap = g.stages < 4 ? 1000.0 : 0.0;
                const double t = stay ? waves * std::max(mma + 600.0, load + store + 2500.0) + load + store
                                      : waves * (share * std::max(mma, 27.0 * wtap / 24.0) + 27.0 * tap + load + store + 8000.0);
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
    if (!conv3d_fwd_tc_supported(Cin, Cout) || in.Clo % 8 || in.Cskip % 8 || B < 1 || n < 1 ||
        !choose_box(n, Cin, Cout, B, a.g, smem))
        return cudaErrorInvalidValue;
    const bool stay = a.g.stages == 27;
    cudaError_t e = qpat::allow_smem(stay ? (const void*)k_conv_fwd_tc_stay : (const void*)k_conv_fwd_tc, smem);
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
    if (stay) {
        int dev = 0, nsm = 0, per = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
            (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
            (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_conv_fwd_tc_stay, kStayThreads, smem)) != cudaSuccess)
            return e;
        per = std::max(1, std::min(per, 512 / a.g.ncols));  // resident CTAs share the 512 columns of tensor memory
        k_conv_fwd_tc_stay<<<std::min(a.g.boxes, nsm * per), kStayThreads, smem, s>>>(a);
    } else {
        k_conv_fwd_tc<<<a.g.boxes, kTcThreads, smem, s>>>(a);
    }
    return cudaGetLastError();
}

int tc_timeouts() {
    int h = 0;
    cudaMemcpyFromSymbol(&h, g_tc_timeouts, sizeof(int));
    return h;
}

}  // namespace unet
}  // namespace qpat
