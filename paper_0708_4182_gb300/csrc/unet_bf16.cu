// unet_bf16.cu -- hand-written kernels of the warm-start U-Net (sm_103a).
//
// The surrogate maps a channel's wall mask, electric-force level and fill
// fraction to its steady density and velocity, which then initialise the
// lattice Boltzmann run (the warm start). Activations are BF16, channels-last
// (NHWC); every sum accumulates in FP32; the optimizer keeps FP32 master
// weights and moments.
//
// The 3x3 convolutions run on the 5th-generation tensor cores: tcgen05.mma
// (kind::f16, BF16 operands from shared memory, FP32 accumulator in tensor
// memory) issued by one elected thread per CTA, operands staged by cp.async and
// cp.async.bulk into the canonical no-swizzle layout (8-row x 16-byte core
// matrices), completion tracked by tcgen05.commit on mbarriers, the accumulator
// read back with tcgen05.ld for the epilogue. Forward and input-gradient
// convolutions are an implicit GEMM with M = 128 consecutive pixels of the
// padded image, N = a tile of output channels, K = 16 input channels of one of
// the 9 taps per MMA (both operands K-major: channels are contiguous per
// pixel). The weight gradient is a GEMM per tap with M = 128 channels of the
// wider side, N = a tile of the other and K = 16 pixels per MMA (both operands
// MN-major), the 9 taps sharing a CTA's staged operands.
//
// A tensor "view" is (pointer to its first channel, channels per pixel of
// the underlying buffer), so a layer reads or writes a channel range of a
// larger buffer (the decoder's concatenations); nothing is copied. Padding of
// the 3x3 convolutions: circular in x (the channels are periodic along the
// flow), zero in y (walls).
#include "unet_bf16.h"

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

namespace unet {
namespace {

using bf16 = __nv_bfloat16;

constexpr int kT = 256;                      // threads of the SIMT kernels
constexpr uint32_t kWaitLimit = 1u << 18;    // try_wait rounds before giving up (about 1 s on a GB300)
constexpr int kSmemPerSm = 233472;           // shared memory of one SM (bytes)

__device__ __forceinline__ float ld(const bf16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ int wrapx(int x, int w) { return x < 0 ? x + w : (x >= w ? x - w : x); }

// ------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// Bounded wait on one phase of an mbarrier. On timeout raise *err and set
// alive = false: the thread waits no more (each later call returns at once),
// so a kernel that lost a phase ends after one time limit per thread rather
// than one per wait, and nothing hangs.
__device__ __forceinline__ void mbar_wait_alive(uint64_t* bar, uint32_t parity, int* err, bool& alive)
{
    if (!alive) return;
    for (uint32_t i = 0; i < kWaitLimit; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (ok) return;
    }
    atomicOr(err, 1);
    alive = false;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(bar))
                 : "memory");
}

// One arrival that also announces `bytes` of bulk copies to come.
__device__ __forceinline__ void mbar_expect_arrive(uint64_t* bar, uint32_t bytes)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

// Contiguous global -> shared copy (16-byte multiples) counted on `bar`.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// 16-byte global -> shared copy; src_bytes = 0 fills zeros (src is not read)
__device__ __forceinline__ void cp_async16_ca(void* dst, const void* src, uint32_t src_bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async16_cg(void* dst, const void* src, uint32_t src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// shared-memory matrix descriptor, no swizzle: core matrix (8 rows x 16 B)
// (i, j) at start + i * sbo + j * lbo, j along K, i along M (or N)
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return uint64_t((addr >> 4) & 0x3FFF) | (uint64_t((lbo >> 4) & 0x3FFF) << 16) |
           (uint64_t((sbo >> 4) & 0x3FFF) << 32) | (uint64_t(1) << 46);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B,
// M = 128, N = n; a_mn / b_mn select MN-major operands
__host__ __device__ constexpr uint32_t idesc_bf16(int n, bool a_mn, bool b_mn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (a_mn ? 1u << 15 : 0u) | (b_mn ? 1u << 16 : 0u) |
           (uint32_t(n >> 3) << 17) | (uint32_t(128 >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
        "l"(da), "l"(db), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// One thread of the converged warp. The MMA issue loops branch on this, and on
// a warp index that is uniform to the compiler (warp_index): behind a plain
// "lane == 0" it takes 157 cycles to issue an MMA whatever its size (operands
// of the uniform datapath in divergent code), behind elect 66 for N <= 128, 98
// for 192 and 130 for 256, the MMA's own rate (measured, one CTA).
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\tselp.u32 %0, 1, 0, e;\n\t}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0); }

// 32 lanes x 16 consecutive FP32 columns: thread t of the warp gets lane t
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Shared address `at` in the cluster's CTA `rank`, and the float at such an address.
__device__ __forceinline__ uint32_t map_cluster(uint32_t at, uint32_t rank)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(at), "r"(rank));
    return a;
}
__device__ __forceinline__ float ld_cluster(uint32_t at)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
    return v;
}

// 32 lanes x 4 columns; the values are there after tmem_ld_wait
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float (&v)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// TMEM columns to allocate for accumulators spanning n FP32 columns (a power
// of two >= 32, at most the 512 of an SM; n > 512 cannot be allocated)
__host__ __device__ constexpr uint32_t tmem_cols(int n)
{
    return n <= 32 ? 32u : (n <= 64 ? 64u : (n <= 128 ? 128u : (n <= 256 ? 256u : 512u)));
}

// Dynamic shared memory that lets at most 512 / cols CTAs share an SM, so
// their tensor-memory allocations (cols columns each) always fit in the 512.
__host__ constexpr int smem_for_tmem(int cols, int needed)
{
    const int ctas = 512 / cols;
    const int cap = kSmemPerSm / (ctas + 1) + 1024;
    return needed > cap ? needed : cap;
}

// output-channel tile of a convolution with n output channels
__host__ __device__ constexpr int conv_ntile(int n) { return n % 128 == 0 ? 128 : (n % 64 == 0 ? 64 : 32); }

// ------------------------------------------------------------------ tensor-core 3x3 convolution
// y[b, p, co] = act(bias[co] + sum_{tap, k} B[co][k](tap) x[b, p + off(tap), k])
// x: NHWC view (channels per pixel ct_in, K = 16 kc channels used), y: NHWC
// view (ct_out per pixel), wt: packed weights (conv_pack_kernel).
//
// The image (or a strip of S of its columns, conv_strip) is taken with one halo column on
// each side, pitch = S + 2 pixels a row, and its padded pixels are numbered row
// by row. A CTA computes MT x 128 consecutive padded pixels (M = 128 a tile) x
// NT output channels; the results on halo columns are dropped (3% of a 64-wide
// image, 6% of a 32-wide one). In this numbering tap (dy, dx) of every pixel is
// the pixel dy pitch + dx further on, so one window of MT 128 + 2 pitch + 2
// pixels of a 16-channel chunk, staged once at a uniform 16-byte pixel pitch
// (two planes of 8 channels: LBO the plane distance, SBO 8 pixels), serves all
// nine taps: the A descriptors of the taps only differ in their start. (Staging
// the 128 pixels once per tap, as 4 rows x 32 columns, took 9 times the copies;
// staging 3 halo rows per output row, 3 times, and the weights once per row.)
//
// K runs over (group of CK chunks, tap, chunk). Warps 2-7 stage the windows of
// a group with 16-byte cp.async into a ring of slots and arrive on the slot's
// "full" mbarrier when their own copies have landed and are fenced for the
// tensor core's proxy; warp 1 brings the weights, contiguous in the packing,
// with cp.async.bulk into a ring of slots of TW taps; one thread of warp 0
// issues the MMAs and commits them to the slots' "empty" mbarriers. All eight
// warps read the accumulators back. NG blocks of NT output channels share one
// MMA (32 channels take as long as 96: 64 cycles for N <= 128).
//
// Bound by the issue chain (a wait on two barriers and a commit per weight slot
// around MMAs of 64 cycles each) and, for 32 output channels, by the MMAs
// themselves. Clusters of 4 that share the weights by multicast, deeper weight
// rings and 4 window slots were not faster. Measured on 16 images (us, before ->
// now): 384 -> 128 channels at 16x64 66 -> 21, 128 -> 128 27 -> 12.5, 256 -> 256
// at 8x32 46 -> 17, 192 -> 64 at 32x128 39 -> 35, 64 -> 192 49 -> 29, 96 -> 32 at
// 64x256 56 -> 41, 32 -> 96 72 -> 37, 32 -> 32 30 -> 21; on 8 images 96 -> 32 32 -> 24,
// 32 -> 32 16.5 -> 14.4; on one, 32 -> 32 7.0 -> 7.2, 256 -> 256 43 -> 15. The sums run in the
// order of the earlier kernels, so the outputs are the same bits.
constexpr int kCvThreads = 256;
constexpr int kCvProducers = kCvThreads - 64;
constexpr int kWSlotsMax = 12;
constexpr int kXSlots = 2;  // window slots
// weight taps per ring slot
template <int CK> __host__ __device__ constexpr int conv_tw() { return CK == 1 ? 3 : 1; }
// window pixels for a strip of S columns, rounded up to 1 mod 8 so that the
// planes of a pixel lie in different banks
__host__ __device__ constexpr int conv_npx(int S, int mt) { return (128 * mt + 2 * (S + 2) + 2 + 6) / 8 * 8 + 1; }
template <int NT, int NG, int CK> __host__ __device__ constexpr int conv_wbytes() { return conv_tw<CK>() * CK * NT * NG * 32; }
template <int NT, int NG, int CK, int MT> __host__ __device__ constexpr size_t conv_smem(int S, int wslots)
{
    return size_t(kXSlots) * CK * conv_npx(S, MT) * 32 + size_t(wslots) * conv_wbytes<NT, NG, CK>() +
           (2 * kXSlots + 2 * kWSlotsMax + 1) * 8 + 16 + size_t(conv_npx(S, MT)) * 4;
}

template <int NT, int NG, int CK, int MT>
__global__ void __launch_bounds__(kCvThreads) conv3x3_tc_kernel(const bf16* __restrict__ x, int ct_in, int kc,
                                                                const bf16* __restrict__ wt,
                                                                const float* __restrict__ bias,
                                                                bf16* __restrict__ y, int ct_out, int H, int W, int S,
                                                                int relu, int wslots, int* __restrict__ err)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int N = NT * NG;
    static_assert(MT * N <= 512, "the accumulators must fit the tensor memory");
    constexpr int XS = kXSlots, TW = conv_tw<CK>();
    constexpr uint32_t kCols = tmem_cols(MT * N);
    constexpr int kWBytes = conv_wbytes<NT, NG, CK>();  // one weight slot: TW taps x CK chunks of N x 16
    const int npx = conv_npx(S, MT);
    const int xbytes = CK * npx * 32;           // one window slot
    unsigned char* sw = smem;                   // [wslots][kWBytes]
    unsigned char* sx = sw + wslots * kWBytes;  // [XS][chunk][plane][pixel] of 16 bytes
    uint64_t* xfull = reinterpret_cast<uint64_t*>(sx + size_t(XS) * xbytes);
    uint64_t* xempty = xfull + XS;
    uint64_t* wfull = xempty + XS;
    uint64_t* wempty = wfull + kWSlotsMax;
    uint64_t* done = wempty + kWSlotsMax;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    uint32_t* pix = reinterpret_cast<uint32_t*>(tmem_slot + 4);  // the image's pixel at each window position, or kZeroPix
    constexpr uint32_t kZeroPix = 0xffffffffu;

    __shared__ float sbias[N];
    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const int strips = W / S, strip = blockIdx.x % strips;
    const int pitch = S + 2, s0 = (blockIdx.x / strips) * (128 * MT);
    const int nb = blockIdx.y, b = blockIdx.z;
    const int groups = kc / CK;
    const size_t nstride = size_t(kc) * 9 * NT * 16;  // between the packed blocks of NT channels
    const bf16* wblk = wt + size_t(nb) * NG * nstride;

    if (tid == 0) {
        for (int s = 0; s < XS; ++s) {
            mbar_init(&xfull[s], kCvProducers);
            mbar_init(&xempty[s], 1);
        }
        for (int s = 0; s < wslots; ++s) {
            mbar_init(&wfull[s], 1);
            mbar_init(&wempty[s], 1);
        }
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(tmem_slot, kCols);
    for (int i = tid; i < N; i += kCvThreads) sbias[i] = bias ? bias[nb * N + i] : 0.f;
    // window position i is padded pixel s0 - pitch - 1 + i
    for (int i = tid; i < npx; i += kCvThreads) {
        const int q = s0 - pitch - 1 + i + 2 * pitch;
        const int r = q / pitch, yy = r - 2, xx = wrapx(strip * S + (q - r * pitch) - 1, W);
        pix[i] = (yy >= 0 && yy < H) ? uint32_t(yy) * uint32_t(W) + uint32_t(xx) : kZeroPix;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    bool alive = true;

    if (warp == 0) {
        if (elect_one()) {
            constexpr uint32_t idesc = idesc_bf16(N, false, false);
            const uint32_t lbo = uint32_t(npx) * 16;
            uint32_t acc = 0;
            int ws = 0;
            uint32_t wph = 0;
#pragma unroll 1
            for (int g = 0; g < groups; ++g) {
                const int s = g % XS;
                mbar_wait_alive(&xfull[s], uint32_t(g / XS) & 1u, err, alive);
                const uint32_t xa = smem_u32(sx + size_t(s) * xbytes);
#pragma unroll 1
                for (int t0 = 0; t0 < 9; t0 += TW) {
                    mbar_wait_alive(&wfull[ws], wph, err, alive);
                    tc_fence_after();
                    const uint32_t wa = smem_u32(sw + ws * kWBytes);
#pragma unroll
                    for (int tt = 0; tt < TW; ++tt) {
                        const int t = t0 + tt, dy = t / 3, dx = t - 3 * dy;
                        const uint32_t off = uint32_t(dy * pitch + dx) * 16;
#pragma unroll
                        for (int j = 0; j < CK; ++j) {
                            const uint64_t db = smem_desc(wa + (tt * CK + j) * N * 32, 128, 256);
#pragma unroll
                            for (int m = 0; m < MT; ++m)
                                mma_bf16(tmem + m * N, smem_desc(xa + j * npx * 32 + off + m * 2048, lbo, 128), db,
                                         idesc, acc);
                            acc = 1;
                        }
                    }
                    mma_commit(&wempty[ws]);
                    if (++ws == wslots) {
                        ws = 0;
                        wph ^= 1u;
                    }
                }
                mma_commit(&xempty[s]);
            }
            mma_commit(done);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (elect_one()) {
            int ws = 0;
            uint32_t wph = 1;
#pragma unroll 1
            for (int g = 0; g < groups; ++g) {
#pragma unroll 1
                for (int t0 = 0; t0 < 9; t0 += TW) {
                    // the slot's earlier MMAs (the first pass over the ring finds the slots free)
                    if (g * (9 / TW) + t0 / TW >= wslots) mbar_wait_alive(&wempty[ws], wph, err, alive);
                    mbar_expect_arrive(&wfull[ws], kWBytes);
                    unsigned char* dst = sw + ws * kWBytes;
                    if constexpr (CK == 1) {
                        if constexpr (NG == 1) {  // TW consecutive taps of a chunk are one block
                            bulk_g2s(dst, wblk + size_t(g * 9 + t0) * NT * 16, kWBytes, &wfull[ws]);
                        } else {
                            for (int tt = 0; tt < TW; ++tt)
                                for (int q = 0; q < NG; ++q)
                                    bulk_g2s(dst + (tt * NG + q) * NT * 32,
                                             wblk + q * nstride + size_t(g * 9 + t0 + tt) * NT * 16, NT * 32, &wfull[ws]);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < CK; ++j)
                            bulk_g2s(dst + j * NT * 32, wblk + size_t((g * CK + j) * 9 + t0) * NT * 16, NT * 32, &wfull[ws]);
                    }
                    if (++ws == wslots) {
                        ws = 0;
                        wph ^= 1u;
                    }
                }
            }
            // no copy is in flight when the CTA ends, also after a timeout
            bool drain = true;
            const int uses = groups * (9 / TW);
            for (int u = uses > wslots ? uses - wslots : 0; u < uses; ++u)
                mbar_wait_alive(&wfull[u % wslots], uint32_t(u / wslots) & 1u, err, drain);
        }
        __syncwarp();
    } else {
        const int pt = tid - 64;
        constexpr int PP = 2 * CK;   // 16-byte pieces of a pixel
        constexpr int LAG = XS - 1;  // groups between a thread's copies and their arrival
#pragma unroll 1
        for (int g = 0; g < groups; ++g) {
            const int s = g % XS;
            if (g >= LAG) {  // hand a landed group over before waiting for a slot
                cp_async_wait<LAG - 1>();
                fence_proxy_async();
                mbar_arrive(&xfull[(g - LAG) % XS]);
            }
            if (g >= XS) mbar_wait_alive(&xempty[s], uint32_t(g / XS - 1) & 1u, err, alive);
            unsigned char* dst = sx + size_t(s) * xbytes + (pt % PP) * npx * 16;
            const bf16* src = x + size_t(b) * H * W * ct_in + g * CK * 16 + (pt % PP) * 8;
#pragma unroll 4
            for (int i = pt / PP; i < npx; i += kCvProducers / PP) {
                const uint32_t o = pix[i];
                const bool in = o != kZeroPix;
                cp_async16_ca(dst + i * 16, in ? src + size_t(o) * ct_in : x, in ? 16u : 0u);
            }
            cp_async_commit();
        }
        cp_async_wait<0>();
        fence_proxy_async();
        for (int g = groups > LAG ? groups - LAG : 0; g < groups; ++g) mbar_arrive(&xfull[g % XS]);
    }
    mbar_wait_alive(done, 0, err, alive);
    tc_fence_after();

    // epilogue: warp w reads tensor-memory lanes 32 (w % 4) .. + 31 (pixels of
    // each tile) and every second 16-channel block of the MT tiles
    const int quad = warp & 3;
#pragma unroll 1
    for (int m = 0; m < MT; ++m) {
        const int q = s0 + m * 128 + quad * 32 + lane;
        const int yy = q / pitch, cc = q - yy * pitch;
        const bool ok = cc >= 1 && cc <= S && yy < H;
        bf16* out = y + (size_t(b * H + yy) * W + strip * S + cc - 1) * ct_out + nb * N;
#pragma unroll 1
        for (int n0 = 16 * (warp >> 2); n0 < N; n0 += 32) {
            float v[16];
            tmem_ld16(tmem + (uint32_t(quad * 32) << 16) + m * N + n0, v);
            __align__(16) bf16 o[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                float a = v[j] + sbias[n0 + j];
                if (relu) a = fmaxf(a, 0.f);
                o[j] = __float2bfloat16_rn(a);
            }
            if (ok) {
                uint4* dst = reinterpret_cast<uint4*>(out + n0);
                dst[0] = reinterpret_cast<const uint4*>(o)[0];
                dst[1] = reinterpret_cast<const uint4*>(o)[1];
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kCols);
}

// Packed B operand of the tensor-core convolution. Forward (transpose = 0):
// row n = output channel, column k = input channel, B[n][k](tap) =
// w[n][k][tap]. Input gradient (transpose = 1): row n = input channel of the
// forward layer, column k = its output channel, B[n][k](tap) = w[k][n][8 - tap]
// (the transposed, flipped kernel). w: FP32 master weights [co][ci][9]. Out:
// blocks [n tile][k chunk of 16][tap] of NT x 16 BF16 in core-matrix order
// (row group i at 256 B, k half j at 128 B, row r at 16 B); k beyond the real
// channels is 0.
//
// A thread takes the nine taps of one (n, k), which are contiguous in w, and
// consecutive threads consecutive k, whose outputs lie in 16-byte runs (a thread
// per output element found its place by 64-bit divisions and read 4 of every 36
// bytes: 50 us for all layers of the network, now 20).
__device__ __forceinline__ void pack_pair(const float* __restrict__ w, int co, int ci, int transpose, int nt, int kc,
                                          int i, bf16* __restrict__ out)
{
    const int kreal = transpose ? co : ci, kp = kc * 16;
    const int n = i / kp, k = i - n * kp;
    const float* src = w + (transpose ? size_t(k) * ci + n : size_t(n) * ci + k) * 9;
    const int nbk = n / nt, nn = n - nbk * nt, c = k >> 4, kk = k & 15;
    bf16* dst = out + (size_t(nbk) * kc + c) * 9 * nt * 16 + ((nn >> 3) * 2 + (kk >> 3)) * 64 + (nn & 7) * 8 + (kk & 7);
#pragma unroll
    for (int t = 0; t < 9; ++t)
        dst[size_t(t) * nt * 16] = __float2bfloat16_rn(k < kreal ? src[transpose ? 8 - t : t] : 0.f);
}

__global__ void conv_pack_kernel(const float* __restrict__ w, int co, int ci, int transpose, int nt, int kc,
                                 bf16* __restrict__ out)
{
    const int pairs = (transpose ? ci : co) * kc * 16;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < pairs; i += gridDim.x * blockDim.x)
        pack_pair(w, co, ci, transpose, nt, kc, i, out);
}

// Several packings in one launch: job blockIdx.y is the record
// jobs[5 y .. 5 y + 4] = (address of w, co, ci, transpose, address of out).
__global__ void conv_pack_many_kernel(const long long* __restrict__ jobs)
{
    const long long* j = jobs + 5 * blockIdx.y;
    const float* w = reinterpret_cast<const float*>(j[0]);
    const int co = int(j[1]), ci = int(j[2]), transpose = int(j[3]);
    bf16* out = reinterpret_cast<bf16*>(j[4]);
    const int nrows = transpose ? ci : co, kreal = transpose ? co : ci;
    const int kc = (kreal + 15) / 16, nt = conv_ntile(nrows), pairs = nrows * kc * 16;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < pairs; i += gridDim.x * blockDim.x)
        pack_pair(w, co, ci, transpose, nt, kc, i, out);
}

// ------------------------------------------------------------------ tensor-core weight gradient
// dw[co][ci][tap] += sum over pixels p of dy[p][co] x[p + off(tap)][ci]: per
// tap a GEMM whose K runs over the pixels, 16 a MMA, both operands MN-major (8
// channels of a pixel in 16 bytes, pixels at a 16-byte pitch: LBO = 8 pixels,
// SBO = the distance of two channel groups). The wider of the two channel
// counts is the MMA's M (tiles of 128 rows: dy, or x with SW), the narrower
// its N (tiles of NT = 32 or 16).
//
// A CTA marches down columns of P pixels (P = 64, 32 or 16, dividing the row)
// with all nine taps: row y of dy meets rows y - 1, y and y + 1 of x (halo rows
// of P + 2 pixels), each into its own accumulator (9 NT <= 512 tensor-memory
// columns), so every row of dy and of x is staged once per column; a tap's dx
// only moves the start of the x descriptor. (One tap row per CTA staged both
// three times, and its epilogue added three floats in every nine.) Rows
// outside the image are skipped.
//
// Warps 1-7 stage row r of x and row r - 1 of dy with 16-byte cp.async into
// slot r of a ring and arrive on its "full" mbarrier kWgLag rows later (their
// own copies landed and fenced for the tensor core's proxy); one thread of
// warp 0 issues the MMAs of row r - 1 and commits them to the "empty" mbarrier
// of the slot that held row r - 2. The grid is one wave, or as many as keep the
// sums of an accumulator to kWgChain pixels: each CTA takes an equal share of the
// rows of all columns, crossing from column to column.
//
// The epilogue lays the accumulators out in shared memory as dw has them; the
// CTAs of a cluster add them up through distributed shared memory and add the
// sums to dw with atomics on consecutive floats, a warp's 32 in 4 sectors. (Lane
// by lane, and once per CTA, they took 26 of 45 us at 128 x 128 channels.)
// An MMA of N <= 128 takes 64 cycles, which bounds the narrow layers (32 x 32
// channels at 64x256: 32 us of MMAs). Measured on 16 images (us, before -> now):
// 32 -> 32 at 64x256 54 -> 35, 96 -> 32 92 -> 39, 64 -> 64 at 32x128 46 -> 25,
// 192 -> 64 101 -> 39, 128 -> 128 at 16x64 48 -> 19, 384 -> 128 56 -> 35,
// 256 -> 256 at 8x32 46 -> 21.
constexpr int kWgSlots = 6;
constexpr int kWgLag = 2;                       // rows between a producer's copies and their "full" arrival
constexpr int kWgThreads = 256;                 // 8 warps: one issues the MMAs, seven stage operands
constexpr int kWgProducers = kWgThreads - 32;
template <int P> __host__ __device__ constexpr int wgrad_halo_pix() { return P + 2; }
// dy and x channels per CTA
template <int NT, bool SW> __host__ __device__ constexpr int wgrad_co_tile() { return SW ? NT : 128; }
template <int NT, bool SW> __host__ __device__ constexpr int wgrad_ci_tile() { return SW ? 128 : NT; }
// The accumulators in shared memory, for the sum over a cluster: per output
// channel the 9 taps of the tile's input channels in a row, plus one float of
// padding (bank conflicts).
template <int NT, bool SW> __host__ __device__ constexpr int wgrad_red_pitch() { return wgrad_ci_tile<NT, SW>() * 9 + 1; }
template <int NT, bool SW> __host__ __device__ constexpr int wgrad_red_bytes() { return wgrad_co_tile<NT, SW>() * wgrad_red_pitch<NT, SW>() * 4; }
constexpr int kWgCluster = 8;                   // CTAs whose sums are added before they reach dw, at most
// Pixels summed in one accumulator at most. The tensor core adds each MMA's 16
// pixels to the FP32 accumulator with truncation, so the error grows with the
// length of the chain: relative L2 of dw on positive operands, 32 -> 32 channels
// at 64x256, 512 images, 3.0e-4 in chains of 55,000 pixels.
constexpr int kWgChain = 4096;
template <int NT, int P, bool SW> __host__ __device__ constexpr int wgrad_smem_needed()
{
    const int ring = kWgSlots * (wgrad_co_tile<NT, SW>() * P * 2 + (wgrad_ci_tile<NT, SW>() / 8) * wgrad_halo_pix<P>() * 16);
    const int red = (wgrad_red_bytes<NT, SW>() + 15) / 16 * 16;
    return (ring > red ? ring : red) + 2 * kWgSlots * 8 + 8 + 16;
}

template <int NT, int P, bool SW>
__global__ void __launch_bounds__(kWgThreads) wgrad_tc_kernel(const bf16* __restrict__ x, int ct_x, int ci,
                                                              const bf16* __restrict__ dy, int ct_dy, int co,
                                                              float* __restrict__ dw, int H, int W, long long rows,
                                                              long long per, int cs, int* __restrict__ err)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    static_assert(9 * NT <= 512, "nine accumulators must fit the tensor memory");
    static_assert(P == 16 || P == 32 || P == 64, "columns of 16, 32 or 64 pixels");
    static_assert(kWgLag + 3 <= kWgSlots, "a row's three x slots, and those on their way");
    constexpr int COT = wgrad_co_tile<NT, SW>(), CIT = wgrad_ci_tile<NT, SW>();
    constexpr int HP = wgrad_halo_pix<P>();                // halo row pixels
    constexpr int kDBytes = COT * P * 2;                   // dy: COT output channels x P pixels
    constexpr int kXBytes = (CIT / 8) * HP * 16;           // x: one halo row of CIT input channels
    constexpr int kSlot = kDBytes + kXBytes;
    constexpr int kRing = kWgSlots * kSlot, kRed = (wgrad_red_bytes<NT, SW>() + 15) / 16 * 16;
    constexpr uint32_t kCols = tmem_cols(9 * NT);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + (kRing > kRed ? kRing : kRed));
    uint64_t* empty = full + kWgSlots;
    uint64_t* done = empty + kWgSlots;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);

    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const int co0 = blockIdx.x * COT, ci0 = blockIdx.y * CIT;
    const int co_here = co - co0 < COT ? co - co0 : COT;
    const int ci_here = ci - ci0 < CIT ? ci - ci0 : CIT;
    // rows k_begin .. k_end - 1 of all columns' rows (column k / H, image row k % H)
    const long long k_begin = blockIdx.z * per, k_end = k_begin + per < rows ? k_begin + per : rows;
    const int cols_x = W / P;

    // channel groups beyond co_here and ci_here are never loaded: they only reach
    // accumulators that are not read
    if (tid == 0) {
        for (int s = 0; s < kWgSlots; ++s) {
            mbar_init(&full[s], kWgProducers);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(tmem_slot, kCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    bool alive = true;

    if (warp == 0) {
        if (elect_one()) {
            constexpr uint32_t idesc = idesc_bf16(NT, true, true);
            const uint32_t s0 = smem_u32(smem);
            uint32_t acc[3] = {0, 0, 0};  // per tap row: its accumulators have been written
            int slot = 0;
            uint32_t ph = 0;
#pragma unroll 1
            for (long long k = k_begin; k < k_end;) {
                const int ya = int(k % H), n = int(k_end - k < H - ya ? k_end - k : H - ya), yb = ya + n;
                k += n;
#pragma unroll 1
                for (int r = ya - 1; r <= yb; ++r) {
                    mbar_wait_alive(&full[slot], ph, err, alive);
                    tc_fence_after();
                    const int sm1 = slot == 0 ? kWgSlots - 1 : slot - 1, sm2 = sm1 == 0 ? kWgSlots - 1 : sm1 - 1;
                    if (r > ya) {
                        // row y = r - 1: dy in this slot, x rows y - 1, y, y + 1 in the last three
                        const uint32_t da = s0 + slot * kSlot;
#pragma unroll
                        for (int t = 0; t < 3; ++t) {
                            const int xr = r - 2 + t;
                            if (xr < 0 || xr >= H) continue;
                            const uint32_t xa = s0 + (t == 0 ? sm2 : t == 1 ? sm1 : slot) * kSlot + kDBytes;
#pragma unroll
                            for (int j = 0; j < P / 16; ++j) {
                                const uint64_t dd = smem_desc(da + j * 256, 128, P * 16);  // dy, 16-pixel piece j
#pragma unroll
                                for (int dx = 0; dx < 3; ++dx) {
                                    const uint64_t dh = smem_desc(xa + (16 * j + dx) * 16, 128, HP * 16);  // x, shifted dx
                                    mma_bf16(tmem + (3 * t + dx) * NT, SW ? dh : dd, SW ? dd : dh, idesc,
                                             j > 0 ? 1u : acc[t]);
                                }
                            }
                            acc[t] = 1;
                        }
                        mma_commit(&empty[sm2]);
                        if (r == yb) {  // the column's last row: its other slots as well
                            mma_commit(&empty[sm1]);
                            mma_commit(&empty[slot]);
                        }
                    }
                    if (++slot == kWgSlots) {
                        slot = 0;
                        ph ^= 1u;
                    }
                }
            }
            mma_commit(done);
        }
        __syncwarp();
    } else {
        const int pt = tid - 32;  // producer thread
        const int gd = (co_here + 7) / 8, gx = (ci_here + 7) / 8;
        int slot = 0, lslot = 0;  // slot of this row, and of the row to hand over
        uint32_t ph = 1;          // (the first pass over the ring finds the slots free)
        long long step = 0;
#pragma unroll 1
        for (long long k = k_begin; k < k_end;) {
            const long long col = k / H;
            const int ya = int(k - col * H), n = int(k_end - k < H - ya ? k_end - k : H - ya), yb = ya + n;
            k += n;
            const long long img = (col / cols_x) * H;  // the image's first row
            const int x0 = int(col % cols_x) * P;
#pragma unroll 1
            for (int r = ya - 1; r <= yb; ++r, ++step) {
                if (step >= kWgSlots) mbar_wait_alive(&empty[slot], ph, err, alive);
                unsigned char* sd = smem + slot * kSlot;
                unsigned char* sx = sd + kDBytes;
                if (r > ya) {
                    const bf16* drow = dy + (size_t(img + r - 1) * W + x0) * ct_dy + co0;
                    for (int q = pt; q < P * gd; q += kWgProducers) {
                        const int kk = q % P, g = q / P;
                        cp_async16_cg(sd + g * (P * 16) + kk * 16, drow + size_t(kk) * ct_dy + g * 8, 16u);
                    }
                }
                if (r >= 0 && r < H) {
                    const bf16* xrow = x + size_t(img + r) * W * ct_x + ci0;
                    for (int q = pt; q < HP * gx; q += kWgProducers) {
                        const int pix = q % HP, g = q / HP;
                        const int xs = wrapx(x0 + pix - 1, W);
                        cp_async16_ca(sx + g * (HP * 16) + pix * 16, xrow + size_t(xs) * ct_x + g * 8, 16u);
                    }
                }
                cp_async_commit();
                if (step >= kWgLag) {
                    cp_async_wait<kWgLag>();
                    fence_proxy_async();
                    mbar_arrive(&full[lslot]);
                    lslot = lslot + 1 == kWgSlots ? 0 : lslot + 1;
                }
                if (++slot == kWgSlots) {
                    slot = 0;
                    ph ^= 1u;
                }
            }
        }
        cp_async_wait<0>();
        fence_proxy_async();
        for (long long s = step > kWgLag ? step - kWgLag : 0; s < step; ++s) {
            mbar_arrive(&full[lslot]);
            lslot = lslot + 1 == kWgSlots ? 0 : lslot + 1;
        }
    }
    // every warp: the last commit completes when all MMAs have
    mbar_wait_alive(done, 0, err, alive);
    tc_fence_after();
    // the ring becomes the exchange space: nobody copies into it any more
    __syncthreads();

    // warp w reads tensor-memory lanes 32 (w % 4) .. + 31 and every second
    // block of 4 columns, nine taps of each
    constexpr int RP = wgrad_red_pitch<NT, SW>();
    float* red = reinterpret_cast<float*>(smem);
    const int m = (warp & 3) * 32 + lane;
    // a tap row that lay outside the image for every row of this CTA was never
    // written (nor anything by a CTA without rows)
    const bool any = k_end > k_begin, many = H > 1 && k_end - k_begin > 1;
    const bool up = many || (any && k_begin % H > 0), down = many || (any && k_begin % H < H - 1);
#pragma unroll 1
    for (int n0 = 4 * (warp >> 2); n0 < NT; n0 += 8) {
        float v[9][4];
#pragma unroll
        for (int t = 0; t < 9; ++t) tmem_ld4(tmem + (uint32_t((warp & 3) * 32) << 16) + t * NT + n0, v[t]);
        tmem_ld_wait();
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const bool ok = t < 3 ? up : t < 6 ? any : down;
                red[SW ? (n0 + c) * RP + m * 9 + t : m * RP + (n0 + c) * 9 + t] = ok ? v[t][c] : 0.f;
            }
    }
    // Tensor memory goes back before any wait for the cluster: a peer may still
    // wait for its own allocation, behind a CTA of another launch that holds the
    // columns and waits for a peer in its turn.
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kCols);
    if (cs > 1) cluster_sync();
    const int len = ci_here * 9;
    if (cs == 1) {
        // a warp per output channel
        for (int row = warp; row < co_here; row += kWgThreads / 32) {
            float* dst = dw + (size_t(co0 + row) * ci + ci0) * 9;
            const float* src = red + row * RP;
#pragma unroll 9
            for (int i = lane; i < len; i += 32) atomicAdd(dst + i, src[i]);
        }
        return;
    }
    // each CTA of the cluster adds its share of the output channels over all of
    // them, in the order of their ranks, and the sums to dw
    const int rank = int(blockIdx.z) % cs, share = (co_here + cs - 1) / cs, o_end = min(co_here - rank * share, share);
    const uint32_t red0 = smem_u32(red);
    uint32_t peer[kWgCluster];  // red of each rank
#pragma unroll
    for (int q = 0; q < kWgCluster; ++q) peer[q] = map_cluster(red0, q < cs ? q : 0);
#pragma unroll 2
    for (int i = tid; i < o_end * len; i += kWgThreads) {
        const int o = i / len, e = i - o * len, row = rank * share + o;
        const uint32_t at = uint32_t(row * RP + e) * 4;
        float v[kWgCluster];
#pragma unroll
        for (int q = 0; q < kWgCluster; ++q) v[q] = q < cs ? ld_cluster(peer[q] + at) : 0.f;
        float sum = v[0];
#pragma unroll
        for (int q = 1; q < kWgCluster; ++q) sum += v[q];
        atomicAdd(dw + (size_t(co0 + row) * ci + ci0) * 9 + e, sum);
    }
    cluster_sync();  // a peer may still be reading this CTA's sums
}

// ------------------------------------------------------------------ SIMT kernels (NHWC)
// db[c] += sum over pixels of dy[p, c]; block = channels, grid over pixel ranges
__global__ void bias_grad_kernel(const bf16* __restrict__ dy, int ct, int C, long long npix, int per_block,
                                 float* __restrict__ db)
{
    const int c = threadIdx.x;
    if (c >= C) return;
    const long long p0 = (long long)blockIdx.x * per_block;
    const long long p1 = p0 + per_block < npix ? p0 + per_block : npix;
    float s = 0.f;
    for (long long p = p0; p < p1; ++p) s += ld(dy + p * ct + c);
    atomicAdd(&db[c], s);
}

// 8 BF16 values (16 bytes) <-> FP32
__device__ __forceinline__ void unpack8(const uint4& q, float (&v)[8])
{
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[2 * k] = __uint_as_float(w[k] << 16);
        v[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
    }
}
__device__ __forceinline__ uint4 pack8(const float (&v)[8])
{
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
        w[k] = *reinterpret_cast<const uint32_t*>(&h);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// 1x1 head: y[b, o, p] = bias[o] + sum_i w[o][i] x[b, p, i] (x NHWC view, y FP32 NCHW)
__global__ void head_fwd_kernel(const bf16* __restrict__ x, int ct, int Ci, const bf16* __restrict__ w,
                                const float* __restrict__ bias, float* __restrict__ y, int Co, int HW, int B)
{
    // the Co x Ci weights (at most 8 x 64) once per block, read as broadcasts
    __shared__ float ws[8 * 64];
    for (int k = threadIdx.x; k < Co * Ci; k += blockDim.x) ws[k] = ld(w + k);
    __syncthreads();
    const long long n = (long long)B * HW;
    const bool vec = (Ci % 8 == 0) && (ct % 8 == 0) && ((reinterpret_cast<uintptr_t>(x) & 15) == 0);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int b = int(i / HW), p = int(i % HW);
        const bf16* xp = x + i * ct;
        float s[8];
        for (int o = 0; o < Co; ++o) s[o] = bias[o];
        if (vec) {
            // the pixel's channels 8 at a time (16-byte loads), each used by every output
            for (int c0 = 0; c0 < Ci; c0 += 8) {
                float xv[8];
                unpack8(*reinterpret_cast<const uint4*>(xp + c0), xv);
                for (int o = 0; o < Co; ++o) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) s[o] = fmaf(ws[o * Ci + c0 + k], xv[k], s[o]);
                }
            }
        } else {
            for (int c = 0; c < Ci; ++c) {
                const float xv = ld(xp + c);
                for (int o = 0; o < Co; ++o) s[o] = fmaf(ws[o * Ci + c], xv, s[o]);
            }
        }
        for (int o = 0; o < Co; ++o) y[((long long)b * Co + o) * HW + p] = s[o];
    }
}

// head backward: dx[b, p, i] = sum_o w[o][i] dy[b, o, p] (NHWC BF16 out);
// dw[o][i] += sum dy x, db[o] += sum dy (FP32). Block: Ci channels x
// (256 / Ci) pixel lanes; each thread keeps its CO partial sums of dw and db
// in registers, reduced per block in shared memory.
template <int CO>
__global__ void head_bwd_kernel(const bf16* __restrict__ x, int ct, int Ci, const bf16* __restrict__ w,
                                const float* __restrict__ dy, int HW, int B, bf16* __restrict__ dx, int ct_dx,
                                float* __restrict__ dw, float* __restrict__ db)
{
    __shared__ float red[kT][CO];
    const int lanes = kT / Ci;
    const int c = threadIdx.x % Ci, lane = threadIdx.x / Ci;
    float wc[CO], sw[CO], sb[CO];
#pragma unroll
    for (int o = 0; o < CO; ++o) {
        wc[o] = ld(w + o * Ci + c);
        sw[o] = sb[o] = 0.f;
    }
    const long long n = (long long)B * HW;
    if (lane < lanes) {
        for (long long i = (long long)blockIdx.x * lanes + lane; i < n; i += (long long)gridDim.x * lanes) {
            const int b = int(i / HW), p = int(i % HW);
            const float xv = ld(x + i * ct + c);
            float s = 0.f;
#pragma unroll
            for (int o = 0; o < CO; ++o) {
                const float g = dy[((long long)b * CO + o) * HW + p];
                s = fmaf(wc[o], g, s);
                sw[o] = fmaf(g, xv, sw[o]);
                sb[o] += g;
            }
            dx[i * ct_dx + c] = __float2bfloat16_rn(s);
        }
    }
#pragma unroll
    for (int o = 0; o < CO; ++o) red[threadIdx.x][o] = lane < lanes ? sw[o] : 0.f;
    __syncthreads();
    if (lane == 0) {
        for (int o = 0; o < CO; ++o) {
            float t = red[c][o];
            for (int k = 1; k < lanes; ++k) t += red[k * Ci + c][o];
            atomicAdd(&dw[o * Ci + c], t);
        }
    }
    __syncthreads();
    // db: every channel's thread saw the same dy values, so channel 0's lanes suffice
#pragma unroll
    for (int o = 0; o < CO; ++o) red[threadIdx.x][o] = (c == 0 && lane < lanes) ? sb[o] : 0.f;
    __syncthreads();
    if (threadIdx.x < CO) {
        float t = 0.f;
        for (int k = 0; k < lanes; ++k) t += red[k * Ci][threadIdx.x];
        atomicAdd(&db[threadIdx.x], t);
    }
}

// The same with 8 channels of a pixel per thread (16-byte accesses; Ci = 8, 16,
// 32 or 64, views 16-byte aligned): the products of dx run in the same order;
// the sums of dw and db go over the warp's lanes of one channel group by
// shuffles, then over the warps. Memory bound; a channel a thread took 43 us for
// 16 tiles of 64x256 and 32 channels, now 24.
template <int CO>
__global__ void __launch_bounds__(kT) head_bwd8_kernel(const bf16* __restrict__ x, int ct, int Ci,
                                                       const bf16* __restrict__ w, const float* __restrict__ dy, int HW,
                                                       int B, bf16* __restrict__ dx, int ct_dx, float* __restrict__ dw,
                                                       float* __restrict__ db)
{
    __shared__ float red[kT / 32][8][CO * 8 + CO];
    const int G = Ci / 8, grp = threadIdx.x % G, lanes = kT / G;
    float wc[CO][8], sw[CO][8], sb[CO];
#pragma unroll
    for (int o = 0; o < CO; ++o) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            wc[o][k] = ld(w + o * Ci + grp * 8 + k);
            sw[o][k] = 0.f;
        }
        sb[o] = 0.f;
    }
    const long long n = (long long)B * HW;
    for (long long i = (long long)blockIdx.x * lanes + threadIdx.x / G; i < n; i += (long long)gridDim.x * lanes) {
        const int b = int(i / HW), p = int(i - (long long)b * HW);
        float xv[8], s[8];
        unpack8(*reinterpret_cast<const uint4*>(x + i * ct + grp * 8), xv);
#pragma unroll
        for (int k = 0; k < 8; ++k) s[k] = 0.f;
#pragma unroll
        for (int o = 0; o < CO; ++o) {
            const float g = dy[((long long)b * CO + o) * HW + p];
            sb[o] += g;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                s[k] = fmaf(wc[o][k], g, s[k]);
                sw[o][k] = fmaf(g, xv[k], sw[o][k]);
            }
        }
        *reinterpret_cast<uint4*>(dx + i * ct_dx + grp * 8) = pack8(s);
    }
    // lanes l and l ^ m (m = G, 2 G, ..) hold the same channel group
    const int wl = threadIdx.x & 31, wp = threadIdx.x >> 5;
    for (int m = G; m < 32; m <<= 1) {
#pragma unroll
        for (int o = 0; o < CO; ++o) {
            sb[o] += __shfl_xor_sync(0xffffffffu, sb[o], m);
#pragma unroll
            for (int k = 0; k < 8; ++k) sw[o][k] += __shfl_xor_sync(0xffffffffu, sw[o][k], m);
        }
    }
    if (wl < G) {
#pragma unroll
        for (int o = 0; o < CO; ++o) {
            red[wp][wl][CO * 8 + o] = sb[o];
#pragma unroll
            for (int k = 0; k < 8; ++k) red[wp][wl][o * 8 + k] = sw[o][k];
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < CO * Ci + CO; i += kT) {
        // db from the first channel group (every group saw the same dy)
        const int o = i < CO * Ci ? i / Ci : i - CO * Ci, c = i < CO * Ci ? i % Ci : 0;
        const int e = i < CO * Ci ? o * 8 + c % 8 : CO * 8 + o;
        float t = 0.f;
        for (int q = 0; q < kT / 32; ++q) t += red[q][c / 8][e];
        atomicAdd(i < CO * Ci ? &dw[o * Ci + c] : &db[o], t);
    }
}

// 2x2 average pooling of an (H, W) NHWC view and its adjoint
// 2x2 average pooling of an (H, W) NHWC view and its adjoint. One thread per
// coarse pixel and 8 channels (16-byte accesses): C, ctx, cty multiples of 8,
// views 16-byte aligned (checked by the host entries).
__global__ void pool2_fwd_kernel(const bf16* __restrict__ x, int ctx, bf16* __restrict__ y, int cty, int C, int H,
                                 int W, int B)
{
    const int h = H / 2, w = W / 2, C8 = C / 8;
    const int n = B * h * w * C8;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int c = (i % C8) * 8, pix = i / C8;
        const int xx = pix % w, r = pix / w;  // r = b * h + yy
        const bf16* s = x + (size_t(2 * r) * W + 2 * xx) * ctx + c;
        float a[8], b2[8], c2[8], d[8];
        unpack8(*reinterpret_cast<const uint4*>(s), a);
        unpack8(*reinterpret_cast<const uint4*>(s + ctx), b2);
        unpack8(*reinterpret_cast<const uint4*>(s + size_t(W) * ctx), c2);
        unpack8(*reinterpret_cast<const uint4*>(s + size_t(W + 1) * ctx), d);
        float o[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) o[k] = 0.25f * ((a[k] + b2[k]) + (c2[k] + d[k]));
        *reinterpret_cast<uint4*>(y + size_t(pix) * cty + c) = pack8(o);
    }
}

__global__ void pool2_bwd_kernel(const bf16* __restrict__ dy, int cty, bf16* __restrict__ dx, int ctx, int C, int H,
                                 int W, int B, int accumulate)
{
    const int h = H / 2, w = W / 2, C8 = C / 8;
    const int n = B * h * w * C8;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int c = (i % C8) * 8, pix = i / C8;
        const int xx = pix % w, r = pix / w;
        float g[8];
        unpack8(*reinterpret_cast<const uint4*>(dy + size_t(pix) * cty + c), g);
#pragma unroll
        for (int k = 0; k < 8; ++k) g[k] *= 0.25f;
        bf16* o = dx + (size_t(2 * r) * W + 2 * xx) * ctx + c;
        const size_t offs[4] = {0, size_t(ctx), size_t(W) * ctx, size_t(W + 1) * ctx};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint4* dst = reinterpret_cast<uint4*>(o + offs[q]);
            float v[8];
            if (accumulate) {
                unpack8(*dst, v);
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] += g[k];
            } else {
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = g[k];
            }
            *dst = pack8(v);
        }
    }
}

// nearest 2x upsampling of an (h, w) NHWC view and its adjoint (sum over the
// 4 copies); a thread reads 8 channels (16 bytes) of a coarse pixel and writes
// them four times, so C, ctx, cty must be multiples of 8 and the views 16-byte
// aligned. (A thread per copy, placed by 64-bit divisions: 34 us for the three
// upsamplings of 16 tiles of 64x256, now 19.)
__global__ void up2_fwd_kernel(const bf16* __restrict__ x, int ctx, bf16* __restrict__ y, int cty, int C, int h,
                               int w, int B)
{
    const int W = 2 * w, C8 = C / 8;
    const long long n = (long long)B * h * w * C8;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        long long pix;
        int c;
        if (n < (1LL << 31)) {
            const uint32_t q = uint32_t(i) / uint32_t(C8);
            pix = q;
            c = int(uint32_t(i) - q * uint32_t(C8)) * 8;
        } else {
            pix = i / C8;
            c = int(i % C8) * 8;
        }
        const long long r = n < (1LL << 31) ? (long long)(uint32_t(pix) / uint32_t(w)) : pix / w;  // b * h + y
        const int xx = int(pix - r * w);
        const uint4 v = *reinterpret_cast<const uint4*>(x + size_t(pix) * ctx + c);
        bf16* o = y + (size_t(2 * r) * W + 2 * xx) * cty + c;
        *reinterpret_cast<uint4*>(o) = v;
        *reinterpret_cast<uint4*>(o + cty) = v;
        *reinterpret_cast<uint4*>(o + size_t(W) * cty) = v;
        *reinterpret_cast<uint4*>(o + size_t(W + 1) * cty) = v;
    }
}

__global__ void up2_bwd_kernel(const bf16* __restrict__ dy, int cty, bf16* __restrict__ dx, int ctx, int C, int h,
                               int w, int B)
{
    const int W = 2 * w, C8 = C / 8;
    const int n = B * h * w * C8;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int c = (i % C8) * 8, pix = i / C8;
        const int xx = pix % w, r = pix / w;
        const bf16* s = dy + (size_t(2 * r) * W + 2 * xx) * cty + c;
        float a[8], b2[8], c2[8], d[8];
        unpack8(*reinterpret_cast<const uint4*>(s), a);
        unpack8(*reinterpret_cast<const uint4*>(s + cty), b2);
        unpack8(*reinterpret_cast<const uint4*>(s + size_t(W) * cty), c2);
        unpack8(*reinterpret_cast<const uint4*>(s + size_t(W + 1) * cty), d);
        float o[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) o[k] = (a[k] + b2[k]) + (c2[k] + d[k]);
        *reinterpret_cast<uint4*>(dx + size_t(pix) * ctx + c) = pack8(o);
    }
}

// dy <- dy * (y > 0): gradient through a ReLU whose output is y (NHWC views,
// C <= 256 channels, C, cty, ctd multiples of 8, 16-byte aligned); with db !=
// NULL also db[c] += sum over pixels of the masked dy (the bias gradient of the
// layer that produced y). A thread handles 8 channels of a pixel with 16-byte
// loads and keeps 8 partial sums; the block sums them per channel in shared
// memory, one atomic per channel.
__global__ void relu_bwd_kernel(const bf16* __restrict__ y, int cty, bf16* __restrict__ dy, int ctd, int C,
                                long long npix, float* __restrict__ db)
{
    __shared__ float red[kT][8];
    const int G = C / 8, lanes = kT / G;
    const int grp = threadIdx.x % G, lane = threadIdx.x / G;
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    // each pixel's 8 gradients: zero where y <= 0, else kept and summed
    auto step = [&](const uint4& yv, uint4& gv) {
        const bf16* ye = reinterpret_cast<const bf16*>(&yv);
        bf16* ge = reinterpret_cast<bf16*>(&gv);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (__bfloat162float(ye[j]) > 0.f)
                s[j] += __bfloat162float(ge[j]);
            else
                ge[j] = __float2bfloat16_rn(0.f);
        }
    };
    if (lane < lanes) {
        // four pixels per round, their loads issued together
        const long long stride = (long long)gridDim.x * lanes;
        long long p = (long long)blockIdx.x * lanes + lane;
        for (; p + 3 * stride < npix; p += 4 * stride) {
            uint4 yv[4], gv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                yv[u] = *reinterpret_cast<const uint4*>(y + (p + u * stride) * cty + grp * 8);
                gv[u] = *reinterpret_cast<const uint4*>(dy + (p + u * stride) * ctd + grp * 8);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                step(yv[u], gv[u]);
                *reinterpret_cast<uint4*>(dy + (p + u * stride) * ctd + grp * 8) = gv[u];
            }
        }
        for (; p < npix; p += stride) {
            const uint4 yv = *reinterpret_cast<const uint4*>(y + p * cty + grp * 8);
            uint4 gv = *reinterpret_cast<const uint4*>(dy + p * ctd + grp * 8);
            step(yv, gv);
            *reinterpret_cast<uint4*>(dy + p * ctd + grp * 8) = gv;
        }
    }
    if (!db) return;
    if (lane >= lanes) {
#pragma unroll
        for (int j = 0; j < 8; ++j) s[j] = 0.f;
    }
    // bias gradient: the partial sums of group grp over the block's pixels
    const int tid = threadIdx.x;
    if ((G & (G - 1)) == 0) {
        // G divides 32: threads tid ^ m (m = G, 2G, .., 16) hold the same
        // group, so shuffles sum a warp's lanes; then one value per warp and
        // group goes through shared memory
        for (int m = G; m < 32; m <<= 1) {
#pragma unroll
            for (int j = 0; j < 8; ++j) s[j] += __shfl_xor_sync(0xffffffffu, s[j], m);
        }
        const int wl = tid & 31, wp = tid >> 5;
        if (wl < G) {
#pragma unroll
            for (int j = 0; j < 8; ++j) red[wp * G + wl][j] = s[j];
        }
        __syncthreads();
        if (tid < C) {
            const int g = tid / 8, j = tid % 8;
            float t = 0.f;
            for (int w = 0; w < kT / 32; ++w) t += red[w * G + g][j];
            atomicAdd(&db[g * 8 + j], t);
        }
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) red[tid][j] = s[j];
        __syncthreads();
        if (tid < C) {
            const int g = tid / 8, j = tid % 8;
            float t = 0.f;
            for (int k = 0; k < lanes; ++k) t += red[k * G + g][j];
            atomicAdd(&db[g * 8 + j], t);
        }
    }
}

// FP32 NCHW planes -> BF16 NHWC with ct channels per pixel (channels >= c are
// 0). V: a thread writes 8 channels of a pixel in 16 bytes (ct a multiple of 8,
// y 16-byte aligned; an element a thread took 18 us for 16 tiles of 64x256, now
// 5).
template <bool V>
__global__ void input_nhwc_kernel(const float* __restrict__ x, int C, int HW, int B, bf16* __restrict__ y, int ct)
{
    if constexpr (V) {
        const int groups = ct / 8;
        const long long n = (long long)B * HW;
        for (long long pix = blockIdx.x * (long long)blockDim.x + threadIdx.x; pix < n;
             pix += (long long)gridDim.x * blockDim.x) {
            const int b = int(pix / HW), p = int(pix - (long long)b * HW);
            for (int g = 0; g < groups; ++g) {
                float v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = g * 8 + k < C ? x[((long long)b * C + g * 8 + k) * HW + p] : 0.f;
                *reinterpret_cast<uint4*>(y + pix * ct + g * 8) = pack8(v);
            }
        }
    } else {
        const long long n = (long long)B * HW * ct;
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
            const int c = int(i % ct);
            const long long pix = i / ct;
            const int b = int(pix / HW), p = int(pix % HW);
            y[i] = __float2bfloat16_rn(c < C ? x[((long long)b * C + c) * HW + p] : 0.f);
        }
    }
}

// weighted mean squared error over n = B*C*HW values, weight per channel:
// loss = sum_i wc (p - t)^2 / n; grad = 2 wc (p - t) / n (FP32, NCHW)
__global__ void mse_kernel(const float* __restrict__ p, const float* __restrict__ t, const float* __restrict__ wc,
                           int C, int HW, long long n, float* __restrict__ grad, double* __restrict__ loss)
{
    __shared__ double red[kT];
    double s = 0.0;
    // four values in flight per thread
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x; i0 < n; i0 += 4 * stride) {
        float d[4], w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const long long i = i0 + u * stride;
            const bool in = i < n;
            // 32-bit divisions where the count allows
            const int c = !in ? 0 : n < (1LL << 31) ? int((uint32_t(i) / uint32_t(HW)) % uint32_t(C)) : int((i / HW) % C);
            w[u] = wc[c];
            d[u] = in ? p[i] - t[i] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const long long i = i0 + u * stride;
            if (i >= n) continue;  // (an infinite weight times the padding's 0 would be NaN)
            s += double(w[u]) * d[u] * d[u];
            grad[i] = 2.f * w[u] * d[u] / float(n);
        }
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int h = kT / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, red[0] / double(n));
}

// Adam on FP32 master weights; writes the BF16 compute copy if wb != NULL
// hyper (may be NULL): lr, c1 = 1 - b1^t, c2 = 1 - b2^t read from device
// memory instead of the arguments (a replayable graph of training steps)
__global__ void adam_kernel(float* __restrict__ wm, bf16* __restrict__ wb, const float* __restrict__ g,
                            float* __restrict__ m, float* __restrict__ v, long long n, float lr, float b1, float b2,
                            float eps, float c1, float c2, float wd, const float* __restrict__ hyper)
{
    if (hyper) {
        lr = hyper[0];
        c1 = hyper[1];
        c2 = hyper[2];
    }
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i] + wd * wm[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float w = wm[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        wm[i] = w;
        if (wb) wb[i] = __float2bfloat16_rn(w);
    }
}

// One training step's Adam scalars on the device. state: [0] t, [1] b1^t,
// [2] b2^t (running products, multiplied in FP32 as the host entry does),
// then the step's [3] lr = lr_sched[t - 1] (the last entry beyond the end),
// [4] 1 - b1^t, [5] 1 - b2^t.
__global__ void adam_hyper_kernel(float* __restrict__ state, const float* __restrict__ lr_sched, int n, float b1,
                                  float b2)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int t = int(state[0]) + 1;
    const float p1 = state[1] * b1, p2 = state[2] * b2;
    state[0] = float(t);
    state[1] = p1;
    state[2] = p2;
    state[3] = lr_sched[t - 1 < n ? t - 1 : n - 1];
    state[4] = 1.f - p1;
    state[5] = 1.f - p2;
}

__global__ void f32_to_bf16_kernel(const float* __restrict__ x, bf16* __restrict__ y, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16_rn(x[i]);
}

// Warm-start fields from the network output y [n][3][hw] (normalised): on
// fluid nodes (mask 0) rho = clamp(y0 rho_std + rho_mean, lo, hi), u = y1,2
// u_scale; 0 on solids. out [n][3][hw] FP64; sums[b] += sum of rho over image b.
__global__ void warm_decode_kernel(const float* __restrict__ y, int hw, int n, const uint8_t* __restrict__ mask,
                                   float rho_mean, float rho_std, float u_scale, double lo, double hi,
                                   double* __restrict__ out, double* __restrict__ sums)
{
    __shared__ double red[kT];
    const int b = blockIdx.y;
    double s = 0.0;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < hw; p += gridDim.x * blockDim.x) {
        const bool fluid = mask[(size_t)b * hw + p] == 0;
        const float* yb = y + (size_t)b * 3 * hw;
        double r = double(yb[p]) * rho_std + rho_mean;
        r = fluid ? fmin(fmax(r, lo), hi) : 0.0;
        double* ob = out + (size_t)b * 3 * hw;
        ob[p] = r;
        ob[hw + p] = fluid ? double(yb[hw + p]) * u_scale : 0.0;
        ob[2 * hw + p] = fluid ? double(yb[2 * hw + p]) * u_scale : 0.0;
        s += r;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int h = kT / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(&sums[b], red[0]);
}

// rho of image b scaled by mass[b] / sums[b]
__global__ void warm_scale_kernel(int hw, const double* __restrict__ mass, const double* __restrict__ sums,
                                  double* __restrict__ out)
{
    const int b = blockIdx.y;
    const double k = sums[b] > 0.0 ? mass[b] / sums[b] : 1.0;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < hw; p += gridDim.x * blockDim.x)
        out[(size_t)b * 3 * hw + p] *= k;
}

int blocks_for(long long n) { return int(n / kT + 1 < 4096 ? n / kT + 1 : 4096); }

int status(cudaError_t e) { return e == cudaSuccess ? 0 : int(e); }

__device__ int g_err = 0;  // set by a tensor-core kernel whose mbarrier wait timed out

int* err_ptr()
{
    static int* p = nullptr;
    if (!p) cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_err);
    return p;
}

// columns of a strip for CTAs of mt tiles. A CTA stages two rows more than its
// 128 mt pixels, so few tiles go with short rows: 128 columns where they divide
// the row (one image of 64x256, 32 -> 32 channels, forward 7.2 us, 8.3 on whole
// rows; 96 -> 32, 8 images, 24 and 35 us). Else, and for 4 tiles (96 -> 32, 16
// images: 41 us on whole rows, 47 on 128 columns), the whole row up to 256 columns,
// or the largest multiple of 32 up to 256 that divides it.
int conv_strip(int wd, int mt)
{
    if (mt < 4 && wd % 128 == 0) return 128;
    if (wd <= 256) return wd;
    int s = 256;
    while (wd % s) s -= 32;
    return s;
}

template <int NT, int NG, int CK, int MT>
int launch_conv_mt(const void* x, int ct_in, int kc, const void* wt, const float* bias, void* y, int ct_out, int cout,
                   int n, int h, int wd, int relu, cudaStream_t st)
{
    const int S = conv_strip(wd, MT);
    constexpr int cols = int(tmem_cols(MT * NT * NG));
    // weight slots: what fits beside a second CTA on the SM (or alone, where
    // the accumulators or 4 slots leave no room for one), up to the K loop's uses
    const int budget = cols <= 256 && 2 * (conv_smem<NT, NG, CK, MT>(S, 4) + 1024) <= kSmemPerSm ? kSmemPerSm / 2 - 1024
                                                                                                 : kSmemPerSm - 1024;
    constexpr int WMAX = CK == 1 ? 4 : kWSlotsMax;
    int wslots = 4;
    while (wslots < WMAX && wslots < (kc / CK) * (9 / conv_tw<CK>()) &&
           conv_smem<NT, NG, CK, MT>(S, wslots + 1) <= size_t(budget))
        ++wslots;
    const int smem = smem_for_tmem(cols, int(conv_smem<NT, NG, CK, MT>(S, wslots)));
    auto k = conv3x3_tc_kernel<NT, NG, CK, MT>;
    // the instance's limit, the same in every call (not this width's need): calls
    // of other widths may run in other threads
    static std::atomic<int> known{0};
    int limit = known.load(std::memory_order_relaxed);
    cudaError_t e = cudaSuccess;
    if (limit == 0) {
        cudaFuncAttributes at{};
        if ((e = cudaFuncGetAttributes(&at, k)) != cudaSuccess) return int(e);
        limit = kSmemPerSm - 1024 - int(at.sharedSizeBytes);
        known.store(limit, std::memory_order_relaxed);
    }
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, limit)) != cudaSuccess) return int(e);
    dim3 grid((wd / S) * ((h * (S + 2) + 128 * MT - 1) / (128 * MT)), cout / (NT * NG), n);
    k<<<grid, kCvThreads, smem, st>>>((const bf16*)x, ct_in, kc, (const bf16*)wt, bias, (bf16*)y, ct_out, h, wd, S,
                                      relu, wslots, err_ptr());
    return status(cudaGetLastError());
}

// CTAs of mt tiles and n_cta output channels each
long long conv_ctas(int mt, int n_cta, int cout, int n, int h, int wd)
{
    const int S = conv_strip(wd, mt);
    return (long long)(wd / S) * ((h * (S + 2) + 128 * mt - 1) / (128 * mt)) * (cout / n_cta) * n;
}

// Rows of a multiple of 128 pixels (CK = 1): MT tiles per CTA, the most of 4, 2
// and 1 that leave two CTAs per SM; more tiles reuse the staged weights and the
// window's two extra rows.
template <int NT, int NG>
int launch_conv_wide(const void* x, int ct_in, int kc, const void* wt, const float* bias, void* y, int ct_out,
                     int cout, int n, int h, int wd, int relu, cudaStream_t st)
{
    constexpr int N = NT * NG;
    auto ctas = [&](int mt) { return conv_ctas(mt, N, cout, n, h, wd); };
    if (N <= 64 && ctas(4) >= 304)
        return launch_conv_mt<NT, NG, 1, N <= 64 ? 4 : 1>(x, ct_in, kc, wt, bias, y, ct_out, cout, n, h, wd, relu, st);
    if (ctas(2) >= 304) return launch_conv_mt<NT, NG, 1, 2>(x, ct_in, kc, wt, bias, y, ct_out, cout, n, h, wd, relu, st);
    return launch_conv_mt<NT, NG, 1, 1>(x, ct_in, kc, wt, bias, y, ct_out, cout, n, h, wd, relu, st);
}

template <int NT>
int launch_conv(const void* x, int ct_in, int kc, const void* wt, const float* bias, void* y, int ct_out, int cout,
                int n, int h, int wd, int relu, cudaStream_t st)
{
    // K in groups of 4, 2 or 1 chunks of 16 channels (rows of whole 128-pixel
    // tiles: 1); the order of the sums, and so the result, depends on it
    if (wd % 128 == 0) {
        // three blocks of 32 or 64 output channels in one MMA: one of N = 32
        // takes as long as one of N = 96, three of N = 64 twice as long as one of
        // 192 (unless that leaves half of the SMs without a CTA: 64 -> 192 at
        // 32x128, one image, 12.3 us with, 10.3 without)
        if constexpr (NT <= 64)
            if (cout % (3 * NT) == 0 && (NT == 32 || conv_ctas(1, 3 * NT, cout, n, h, wd) >= 76))
                return launch_conv_wide<NT, 3>(x, ct_in, kc, wt, bias, y, ct_out, cout, n, h, wd, relu, st);
        return launch_conv_wide<NT, 1>(x, ct_in, kc, wt, bias, y, ct_out, cout, n, h, wd, relu, st);
    }
    if (kc % 4 == 0) return launch_conv_mt<NT, 1, 4, 1>(x, ct_in, kc, wt, bias, y, ct_out, cout, n, h, wd, relu, st);
    if (kc % 2 == 0) return launch_conv_mt<NT, 1, 2, 1>(x, ct_in, kc, wt, bias, y, ct_out, cout, n, h, wd, relu, st);
    return launch_conv_mt<NT, 1, 1, 1>(x, ct_in, kc, wt, bias, y, ct_out, cout, n, h, wd, relu, st);
}

template <int NT, int P, bool SW>
int launch_wgrad_p(const void* x, int ct_x, int ci, const void* dy, int ct_dy, int co, float* dw, int n, int h,
                   int wd, cudaStream_t st)
{
    constexpr int COT = wgrad_co_tile<NT, SW>(), CIT = wgrad_ci_tile<NT, SW>();
    const int smem = smem_for_tmem(int(tmem_cols(9 * NT)), wgrad_smem_needed<NT, P, SW>());
    auto k = wgrad_tc_kernel<NT, P, SW>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return int(e);
    const int tx = (co + COT - 1) / COT, ty = (ci + CIT - 1) / CIT;
    const long long rows = (long long)n * (wd / P) * h;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = at.val.clusterDim.y = 1;
    cfg.blockDim = dim3(kWgThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    // clusters of the largest size that run at once on this device
    at.val.clusterDim.z = kWgCluster;
    cfg.gridDim = dim3(1, 1, kWgCluster);
    int dev = 0, sms = 0, at_once = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return int(e);
    // known per device; a query that fails is asked again, and the call goes
    // without clusters
    constexpr int kDevices = 32;
    static std::atomic<int> known[kDevices];
    if (dev < kDevices) at_once = known[dev].load(std::memory_order_relaxed);
    if (at_once == 0) {
        if (cudaOccupancyMaxActiveClusters(&at_once, k, &cfg) != cudaSuccess || at_once < 0) {
            cudaGetLastError();
            at_once = 0;
        }
        if (dev < kDevices) known[dev].store(at_once, std::memory_order_relaxed);
    }
    // Whole waves of CTAs (mostly one) that share the rows of all columns equally,
    // at least 4 rows each (a shorter CTA is mostly prologue and epilogue). Where that
    // leaves SMs free, up to 8 CTAs form a cluster that adds its sums in a fixed
    // order before the atomics, so that dw gets few addends (with at most two
    // the result does not depend on their order). Clusters of 8 do not fill the
    // SMs, so larger layers go without: 192 -> 64 channels at 32x128, 16 images,
    // 41 us, with clusters 60.
    const long long most = (rows + 3) / 4, tiles = (long long)tx * ty;
    const bool few = most * tiles <= (long long)at_once * kWgCluster;
    const long long wave = sms * (9 * NT <= 256 ? 2 : 1) / tiles;
    long long splits = few ? most : wave;
    if (splits > most) splits = most;
    if (splits < 1) splits = 1;
    // more waves where one would make the chains too long
    const long long least = (rows + kWgChain / P - 1) / (kWgChain / P);
    if (splits < least) splits = wave > 1 ? (least + wave - 1) / wave * wave : least;
    if (splits > 65535) splits = 65535;
    int cs = 1;
    while (few && cs < kWgCluster && 2 * cs <= splits) cs *= 2;
    splits = splits / cs * cs;
    const long long per = (rows + splits - 1) / splits;
    at.val.clusterDim.z = cs;
    cfg.gridDim = dim3(tx, ty, int(splits));
    return status(cudaLaunchKernelEx(&cfg, k, (const bf16*)x, ct_x, ci, (const bf16*)dy, ct_dy, co, dw, h, wd, rows, per,
                                     cs, err_ptr()));
}

template <int NT, bool SW>
int launch_wgrad(const void* x, int ct_x, int ci, const void* dy, int ct_dy, int co, float* dw, int n, int h,
                 int wd, cudaStream_t st)
{
    // columns of the widest of 64, 32 and 16 pixels that divides the row
    if (wd % 64 == 0) return launch_wgrad_p<NT, 64, SW>(x, ct_x, ci, dy, ct_dy, co, dw, n, h, wd, st);
    if (wd % 32 == 0) return launch_wgrad_p<NT, 32, SW>(x, ct_x, ci, dy, ct_dy, co, dw, n, h, wd, st);
    return launch_wgrad_p<NT, 16, SW>(x, ct_x, ci, dy, ct_dy, co, dw, n, h, wd, st);
}

}  // namespace
}  // namespace unet

using namespace unet;

extern "C" {

int unet_conv_ntile(int channels) { return conv_ntile(channels); }

size_t unet_conv_pack_elems(int co, int ci, int transpose)
{
    const int nrows = transpose ? ci : co, kreal = transpose ? co : ci;
    const int kc = (kreal + 15) / 16;
    return size_t(nrows) * kc * 16 * 9;
}

int unet_conv_pack(const float* w, int co, int ci, int transpose, void* out, void* stream)
{
    const int nrows = transpose ? ci : co, kreal = transpose ? co : ci;
    if (nrows % 32) return -1;
    const int kc = (kreal + 15) / 16;
    conv_pack_kernel<<<blocks_for((long long)nrows * kc * 16), kT, 0, (cudaStream_t)stream>>>(w, co, ci, transpose, conv_ntile(nrows), kc,
                                                                        (bf16*)out);
    return status(cudaGetLastError());
}

int unet_conv_pack_many(const long long* jobs, int njobs, long max_elems, void* stream)
{
    if (!jobs || njobs < 1 || njobs > 65535 || max_elems < 1) return -1;
    conv_pack_many_kernel<<<dim3(blocks_for(max_elems / 9), njobs), kT, 0, (cudaStream_t)stream>>>(jobs);
    return status(cudaGetLastError());
}

int unet_conv3x3(const void* x, int ct_in, int cin, const void* wt, const float* bias, void* y, int ct_out, int cout,
                 int n, int h, int wd, int relu, void* stream)
{
    // K runs over kc chunks of 16 channels: cin a multiple of 16, or cin < 16
    // in a view whose first 16 channels are readable (channels >= cin zero)
    const int kc = (cin + 15) / 16;
    if (wd % 32 || h % 4 || cout % 32 || ct_in % 8 || ct_out % 8 || cin < 1 ||
        (cin % 16 && cin > 16) || kc * 16 > ct_in ||
        (reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(wt)) & 15)
        return -1;
    cudaStream_t st = (cudaStream_t)stream;
    switch (conv_ntile(cout)) {
    case 128: return launch_conv<128>(x, ct_in, kc, wt, bias, y, ct_out, cout, n, h, wd, relu, st);
    case 64: return launch_conv<64>(x, ct_in, kc, wt, bias, y, ct_out, cout, n, h, wd, relu, st);
    default: return launch_conv<32>(x, ct_in, kc, wt, bias, y, ct_out, cout, n, h, wd, relu, st);
    }
}

int unet_conv3x3_bwd_weight(const void* x, int ct_x, int ci, const void* dy, int ct_dy, int co, float* dw, float* db,
                            int n, int h, int wd, void* stream)
{
    if (wd % 16 || co % 8 || ct_x % 8 || ct_dy % 8 ||
        (reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(dy)) & 15)
        return -1;
    cudaStream_t st = (cudaStream_t)stream;
    // the wider of the two channel counts on the MMA's 128 rows
    int rc;
    if (ci > co)
        rc = launch_wgrad<32, true>(x, ct_x, ci, dy, ct_dy, co, dw, n, h, wd, st);
    else if (ci > 16)
        rc = launch_wgrad<32, false>(x, ct_x, ci, dy, ct_dy, co, dw, n, h, wd, st);
    else
        rc = launch_wgrad<16, false>(x, ct_x, ci, dy, ct_dy, co, dw, n, h, wd, st);
    if (rc || !db) return rc;
    const long long npix = (long long)n * h * wd;
    const int per = 1024;
    bias_grad_kernel<<<int((npix + per - 1) / per), co <= kT ? co : kT, 0, st>>>((const bf16*)dy, ct_dy, co, npix, per,
                                                                                db);
    return status(cudaGetLastError());
}

int unet_tc_error(void* stream, int reset)
{
    int h = 0;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = cudaMemcpyAsync(&h, err_ptr(), sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return -int(e);
    if (reset && h) {
        const int z = 0;
        cudaMemcpyAsync(err_ptr(), &z, sizeof(int), cudaMemcpyHostToDevice, st);
        cudaStreamSynchronize(st);
    }
    return h;
}

int unet_head_fwd(const void* x, int ct, int ci, const void* w, const float* bias, float* y, int co, int n, int hw,
                  void* stream)
{
    if (co < 1 || co > 8 || ci < 1 || ci > 64) return -1;
    head_fwd_kernel<<<blocks_for((long long)n * hw), kT, 0, (cudaStream_t)stream>>>((const bf16*)x, ct, ci,
                                                                                   (const bf16*)w, bias, y, co, hw, n);
    return status(cudaGetLastError());
}

int unet_head_bwd(const void* x, int ct, int ci, const void* w, const float* dy, int co, int n, int hw, void* dx,
                  int ct_dx, float* dw, float* db, void* stream)
{
    if (co != 3 || ci < 1 || ci > kT) return -1;
    if ((ci == 8 || ci == 16 || ci == 32 || ci == 64) && ct % 8 == 0 && ct_dx % 8 == 0 &&
        ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(dx)) & 15) == 0) {
        // about 8 pixels per thread, at most 4 blocks per SM
        long long blocks8 = (long long)n * hw * (ci / 8) / (kT * 8) + 1;
        if (blocks8 > 608) blocks8 = 608;
        head_bwd8_kernel<3><<<int(blocks8), kT, 0, (cudaStream_t)stream>>>((const bf16*)x, ct, ci, (const bf16*)w, dy, hw,
                                                                          n, (bf16*)dx, ct_dx, dw, db);
        return status(cudaGetLastError());
    }
    // at most 8 blocks per SM: each block adds its partial sums into the same
    // 3 (ci + 1) addresses of dw and db
    long long blocks = (long long)n * hw * ci / (kT * 4) + 1;
    if (blocks > 1184) blocks = 1184;
    head_bwd_kernel<3><<<int(blocks), kT, 0, (cudaStream_t)stream>>>(
        (const bf16*)x, ct, ci, (const bf16*)w, dy, hw, n, (bf16*)dx, ct_dx, dw, db);
    return status(cudaGetLastError());
}

// the vector pooling/upsampling kernels: 8-channel groups, 16-byte aligned
// views, 32-bit element counts
static bool vec8_ok(const void* a, int cta, const void* b, int ctb, int c, long long elems)
{
    return c % 8 == 0 && cta % 8 == 0 && ctb % 8 == 0 && elems / 8 < (1LL << 31) &&
           ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0;
}

int unet_pool2_fwd(const void* x, int ctx, void* y, int cty, int c, int n, int h, int wd, void* stream)
{
    if (!vec8_ok(x, ctx, y, cty, c, (long long)n * c * h * wd) || h % 2 || wd % 2) return -1;
    pool2_fwd_kernel<<<blocks_for((long long)n * c / 8 * h * wd / 4), kT, 0, (cudaStream_t)stream>>>(
        (const bf16*)x, ctx, (bf16*)y, cty, c, h, wd, n);
    return status(cudaGetLastError());
}

int unet_pool2_bwd(const void* dy, int cty, void* dx, int ctx, int c, int n, int h, int wd, int accumulate,
                   void* stream)
{
    if (!vec8_ok(dy, cty, dx, ctx, c, (long long)n * c * h * wd) || h % 2 || wd % 2) return -1;
    pool2_bwd_kernel<<<blocks_for((long long)n * c / 8 * h * wd / 4), kT, 0, (cudaStream_t)stream>>>(
        (const bf16*)dy, cty, (bf16*)dx, ctx, c, h, wd, n, accumulate);
    return status(cudaGetLastError());
}

int unet_up2_fwd(const void* x, int ctx, void* y, int cty, int c, int n, int h, int wd, void* stream)
{
    if (c % 8 || ctx % 8 || cty % 8 || (reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15)
        return -1;
    up2_fwd_kernel<<<blocks_for((long long)n * c / 8 * h * wd), kT, 0, (cudaStream_t)stream>>>(
        (const bf16*)x, ctx, (bf16*)y, cty, c, h, wd, n);
    return status(cudaGetLastError());
}

int unet_up2_bwd(const void* dy, int cty, void* dx, int ctx, int c, int n, int h, int wd, void* stream)
{
    if (!vec8_ok(dy, cty, dx, ctx, c, (long long)n * c * h * wd * 4)) return -1;
    up2_bwd_kernel<<<blocks_for((long long)n * c / 8 * h * wd), kT, 0, (cudaStream_t)stream>>>(
        (const bf16*)dy, cty, (bf16*)dx, ctx, c, h, wd, n);
    return status(cudaGetLastError());
}

int unet_relu_bwd(const void* y, int cty, void* dy, int ctd, int c, long npix, float* db, void* stream)
{
    if (c < 8 || c > kT || c % 8 || cty % 8 || ctd % 8 ||
        (reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(dy)) & 15)
        return -1;
    long long blocks = (long long)npix * (c / 8) / (kT * 4) + 1;  // about 4 pixels per thread: one round
    if (blocks > 1184) blocks = 1184;                                 // 8 per SM
    relu_bwd_kernel<<<int(blocks), kT, 0, (cudaStream_t)stream>>>((const bf16*)y, cty, (bf16*)dy, ctd, c, npix, db);
    return status(cudaGetLastError());
}

int unet_input_nhwc(const float* x, int c, int hw, int n, void* y, int ct, void* stream)
{
    if (ct % 8 == 0 && (reinterpret_cast<uintptr_t>(y) & 15) == 0)
        input_nhwc_kernel<true><<<blocks_for((long long)n * hw), kT, 0, (cudaStream_t)stream>>>(x, c, hw, n, (bf16*)y, ct);
    else
        input_nhwc_kernel<false><<<blocks_for((long long)n * hw * ct), kT, 0, (cudaStream_t)stream>>>(x, c, hw, n, (bf16*)y, ct);
    return status(cudaGetLastError());
}

int unet_mse(const float* pred, const float* target, const float* wc, int c, int hw, long count, float* grad,
             double* loss, void* stream)
{
    mse_kernel<<<blocks_for(count) / 8 + 1, kT, 0, (cudaStream_t)stream>>>(pred, target, wc, c, hw, count, grad,
                                                                           loss);
    return status(cudaGetLastError());
}

int unet_adam(float* w_master, void* w_bf16, const float* grad, float* m, float* v, long count, float lr,
              float beta1, float beta2, float eps, int step, float weight_decay, void* stream)
{
    float c1 = 1.f, c2 = 1.f;
    for (int k = 0; k < step; ++k) {
        c1 *= beta1;
        c2 *= beta2;
    }
    adam_kernel<<<blocks_for(count), kT, 0, (cudaStream_t)stream>>>(w_master, (bf16*)w_bf16, grad, m, v, count, lr,
                                                                    beta1, beta2, eps, 1.f - c1, 1.f - c2,
                                                                    weight_decay, nullptr);
    return status(cudaGetLastError());
}

int unet_adam_dev(float* w_master, void* w_bf16, const float* grad, float* m, float* v, long count,
                  const float* hyper, float beta1, float beta2, float eps, float weight_decay, void* stream)
{
    if (!hyper) return -1;
    adam_kernel<<<blocks_for(count), kT, 0, (cudaStream_t)stream>>>(w_master, (bf16*)w_bf16, grad, m, v, count, 0.f,
                                                                    beta1, beta2, eps, 1.f, 1.f, weight_decay, hyper);
    return status(cudaGetLastError());
}

int unet_adam_hyper(float* state, const float* lr_schedule, int n, float beta1, float beta2, void* stream)
{
    if (!state || !lr_schedule || n < 1) return -1;
    adam_hyper_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(state, lr_schedule, n, beta1, beta2);
    return status(cudaGetLastError());
}

int unet_warm_fields(const float* y, int n, int hw, const uint8_t* mask, const double* mass, float rho_mean,
                     float rho_std, float u_scale, double lo, double hi, double* out, double* sums, void* stream)
{
    if (n < 1 || n > 65535 || hw < 1) return -1;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = cudaMemsetAsync(sums, 0, size_t(n) * sizeof(double), st);
    if (e != cudaSuccess) return int(e);
    const int bx = (hw + kT - 1) / kT < 64 ? (hw + kT - 1) / kT : 64;
    warm_decode_kernel<<<dim3(bx, n), kT, 0, st>>>(y, hw, n, mask, rho_mean, rho_std, u_scale, lo, hi, out, sums);
    warm_scale_kernel<<<dim3(bx, n), kT, 0, st>>>(hw, mass, sums, out);
    return status(cudaGetLastError());
}

int unet_f32_to_bf16(const float* x, void* y, long count, void* stream)
{
    f32_to_bf16_kernel<<<blocks_for(count), kT, 0, (cudaStream_t)stream>>>(x, (bf16*)y, count);
    return status(cudaGetLastError());
}

}  // extern "C"
