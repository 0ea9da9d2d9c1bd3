// Training and inference kernels of the warm-start U-Net (no counterpart in the
// paper): 3x3 convolutions as implicit GEMMs on the tensor cores (BF16 operands,
// FP32 accumulation, mma.sync m16n8k16), their data and weight gradients, pooling,
// upsampling, channel concatenation, the 1x1 head, the MSE loss and Adam.
// Activations are NHWC bfloat16 with channel counts that are multiples of 32;
// 3x3 weights are [9][Cout][Cin] (tap = (dh + 1) * 3 + (dw + 1)).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <stdint.h>

#include <algorithm>

#include "../../include/tpflbm.h"
#include "../../include/tpfnet.h"

namespace {

typedef __nv_bfloat16 bf16;

// Programmatic dependent launch: every kernel here is launched so that its CTAs may start
// while the kernel before it on the stream drains, and waits for that kernel's end (and its
// memory) before it touches global memory.  What runs ahead is the launch itself and a tensor
// core kernel's set-up (barriers, tensor memory, descriptors), about 2 us of each of the 20 to
// 60 short kernels of a forward or training step.  pdl_next lets the next kernel start; the
// tensor core kernels say so once they hold their tensor memory (a waiting successor must
// not take it from a CTA that has yet to allocate).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_enter()
{
    pdl_wait();
    pdl_next();
}
// The mma.sync kernels run for tens of microseconds and at one CTA after another on an SM: where
// they have more CTAs than SMs, early ones pile up on the SMs that the kernel before left first, and
// the kernel takes longer than its launch saved ((4, 15, 60, 256, 256) data gradient 148 us against
// 88, (8, 30, 120, 128, 128) forward 83 against 68; with at most one CTA per SM (1, 31, 33, 64, 64)
// forward 17.3 against 18.6).  So they start early, and let others, up to that many CTAs only.
constexpr unsigned kPdlCtas = 152;
__device__ __forceinline__ void pdl_enter_small()
{
    pdl_wait();
    if (gridDim.x * gridDim.y * gridDim.z <= kPdlCtas) pdl_next();
}
template <class... K, class... A>
cudaError_t launch_pdl(void (*kernel)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, K(args)...);
}
template <class... K, class... A>
void launch_pdl_small(void (*kernel)(K...), dim3 grid, dim3 block, cudaStream_t s, A... args)
{
    if ((unsigned long long)grid.x * grid.y * grid.z <= kPdlCtas)
        launch_pdl(kernel, grid, block, 0, s, args...);
    else
        kernel<<<grid, block, 0, s>>>(K(args)...);
}

constexpr int kBM = 64;  // output pixels per CTA (one row segment)
constexpr int kKC = 32;  // input channels per K chunk
constexpr int kPad = 8;  // smem row padding (bf16) against bank conflicts

__device__ __forceinline__ uint32_t ld_pair(const bf16* p) { return *reinterpret_cast<const uint32_t*>(p); }

__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, const uint32_t* b)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// y[n, h, w, co] = act(b[co] + sum_tap sum_ci x[n, h+dh, w+dw, ci] W[tap][co][ci]).
// CTA: 64 pixels of one image row x BN output channels; 4 warps, 16 pixels each.
template <int BN>
__global__ void __launch_bounds__(128)
k_conv3x3(const bf16* __restrict__ x, int N, int H, int W, int Cin, const bf16* __restrict__ wt,
          const float* __restrict__ bias, int Cout, int relu, bf16* __restrict__ y, int ldy,
          const bf16* __restrict__ mask)
{
    pdl_enter_small();
    __shared__ __align__(16) bf16 As[kBM][kKC + kPad];
    __shared__ __align__(16) bf16 Bs[BN][kKC + kPad];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, tig = lane & 3;
    const int wblocks = (W + kBM - 1) / kBM;
    const int row = blockIdx.x / wblocks, w0 = (blockIdx.x % wblocks) * kBM;
    const int n = row / H, h = row % H;
    const int co0 = blockIdx.y * BN;
    constexpr int NT = BN / 8;
    float acc[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;

    for (int tap = 0; tap < 9; ++tap) {
        const int dh = tap / 3 - 1, dw = tap % 3 - 1;
        const int hh = h + dh;
        for (int c0 = 0; c0 < Cin; c0 += kKC) {
            // A: 64 pixels x 32 channels (4 x 16-byte pieces per pixel)
            for (int k = tid; k < kBM * 4; k += 128) {
                const int m = k >> 2, q = k & 3;
                const int ww = w0 + m + dw;
                uint4 v = make_uint4(0, 0, 0, 0);
                if (hh >= 0 && hh < H && ww >= 0 && ww < W)
                    v = *reinterpret_cast<const uint4*>(x + (((size_t)n * H + hh) * W + ww) * Cin + c0 + q * 8);
                *reinterpret_cast<uint4*>(&As[m][q * 8]) = v;
            }
            // B: BN output channels x 32 input channels
            for (int k = tid; k < BN * 4; k += 128) {
                const int co = k >> 2, q = k & 3;
                *reinterpret_cast<uint4*>(&Bs[co][q * 8]) =
                    *reinterpret_cast<const uint4*>(wt + ((size_t)tap * Cout + co0 + co) * Cin + c0 + q * 8);
            }
            __syncthreads();
#pragma unroll
            for (int ks = 0; ks < kKC; ks += 16) {
                uint32_t a[4];
                const int r0 = warp * 16 + g;
                a[0] = ld_pair(&As[r0][ks + 2 * tig]);
                a[1] = ld_pair(&As[r0 + 8][ks + 2 * tig]);
                a[2] = ld_pair(&As[r0][ks + 2 * tig + 8]);
                a[3] = ld_pair(&As[r0 + 8][ks + 2 * tig + 8]);
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    uint32_t b[2];
                    b[0] = ld_pair(&Bs[j * 8 + g][ks + 2 * tig]);
                    b[1] = ld_pair(&Bs[j * 8 + g][ks + 2 * tig + 8]);
                    mma_bf16(acc[j], a, b);
                }
            }
            __syncthreads();
        }
    }
    // epilogue: bias, optional ReLU, bf16 store
#pragma unroll
    for (int j = 0; j < NT; ++j) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int m = warp * 16 + g + 8 * r;
            const int ww = w0 + m;
            if (ww >= W) continue;
            const int co = co0 + j * 8 + 2 * tig;
            float v0 = acc[j][2 * r] + (bias ? bias[co] : 0.f);
            float v1 = acc[j][2 * r + 1] + (bias ? bias[co + 1] : 0.f);
            if (relu) {
                v0 = fmaxf(v0, 0.f);
                v1 = fmaxf(v1, 0.f);
            }
            const size_t px = ((size_t)n * H + h) * W + ww;
            if (mask) {
                if (!(__bfloat162float(mask[px * Cout + co]) > 0.f)) v0 = 0.f;
                if (!(__bfloat162float(mask[px * Cout + co + 1]) > 0.f)) v1 = 0.f;
            }
            __nv_bfloat162 o;
            o.x = __float2bfloat16_rn(v0);
            o.y = __float2bfloat16_rn(v1);
            *reinterpret_cast<__nv_bfloat162*>(y + px * ldy + co) = o;
        }
    }
}

// ------------------------------------------------ tcgen05 forward convolution
//
// The same convolution on the fifth-generation tensor cores: an implicit GEMM with
// M = 128 output pixels (a BW x BH block of one image, BW * BH = 128), N = BN output
// channels and K = 9 taps x Cin.  Operands are staged by TMA in swizzled K-major tiles
// of KC channels per row (64 channels: 128-byte rows and swizzle when Cin allows, else
// 32 channels: 64-byte rows and swizzle): the activation tile of a tap is the
// pixel block shifted by (dh, dw), read through a 4-D tensor map whose out-of-range
// rows and columns come back as zeros (the padding); the weight tile is BN rows of
// [9 Cout][Cin].  One thread issues the copies into a ring of kTcStages stages, one
// thread issues tcgen05.mma (M = 128, N = BN, K = 16, BF16 in, FP32 accumulated in
// tensor memory) and frees each stage with tcgen05.commit; the four warps then read
// the accumulator (warp w owns TMEM lanes 32w..32w+31, i.e. pixels), add the bias,
// apply the ReLU and store bf16.  Every wait is bounded; a wait that runs out sets
// the error flag and the CTA still releases its tensor memory.
constexpr int kTcStages = 4;
__device__ int g_tc_err;                     // a bounded wait of the tcgen05 kernel ran out

__device__ __forceinline__ uint32_t sa(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mb_init(uint64_t* b, uint32_t n)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sa(b)), "r"(n) : "memory");
}
// one lane of a converged warp.  The warps that issue copies and MMAs run their loops with
// all lanes and pick the issuing one with this around each issue: tcgen05.mma and the bulk
// copies take their operands from uniform registers, and in a branch that one lane took by
// its number the compiler cannot know them to be uniform (an MMA of 128 x 32 x 16 then took
// 210 cycles to issue).
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n selp.u32 %0, 1, 0, q;\n}\n" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void mb_expect_tx(uint64_t* b, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(sa(b)), "r"(bytes) : "memory");
}
// Bounded wait of a whole warp: false, on every lane, when the polls of any lane ran out.  (Lanes
// poll each for itself; one that gave up alone would leave the others in an elect.sync or a
// __syncwarp that waits for it.)
constexpr uint32_t kMbPolls = 1u << 22;
__device__ __forceinline__ bool mb_wait(uint64_t* b, uint32_t parity, uint32_t polls = kMbPolls, int* err = &g_tc_err)
{
    uint32_t ok = 0;
    for (uint32_t it = 0; it < polls && !ok; ++it)
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(sa(b)), "r"(parity)
            : "memory");
    if (__all_sync(0xffffffffu, ok != 0)) return true;
    atomicExch(err, 1);
    return false;
}
__device__ __forceinline__ void tma_3d(void* dst, const CUtensorMap* m, uint64_t* b, int c0, int c1, int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
            sa(dst)),
        "l"((uint64_t)m), "r"(c0), "r"(c1), "r"(c2), "r"(sa(b))
        : "memory");
}
__device__ __forceinline__ void tma_4d(void* dst, const CUtensorMap* m, uint64_t* b, int c0, int c1, int c2, int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(sa(dst)),
        "l"((uint64_t)m), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(sa(b))
        : "memory");
}
// shared-memory matrix descriptor of a K-major tile with KC bf16 (2 KC bytes) per row,
// swizzled over the row width (64 bytes: mode 4, 128 bytes: mode 2), 8-row groups
// 16 KC bytes apart (start address and strides in 16-byte units; descriptor version 1)
template <int KC>
__device__ __forceinline__ uint64_t kmajor_desc(uint32_t addr)
{
    static_assert(KC == 32 || KC == 64, "64- or 128-byte rows");
    constexpr uint64_t mode = KC == 64 ? 2 : 4;
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(16 * KC >> 4) << 32) |
           ((uint64_t)1 << 46) | (mode << 61);
}
// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// d (+)= A B; and an arrival on bar once every MMA issued so far has finished
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate)
        : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(sa(bar)) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

template <int BN, int KC>
__global__ void __launch_bounds__(128, 1)
k_conv3x3_tc(const __grid_constant__ CUtensorMap mx, const __grid_constant__ CUtensorMap mw, int H, int W, int Cin,
             int Cout, int BW, int BH, const float* __restrict__ bias, int relu, bf16* __restrict__ y, int ldy,
             const bf16* __restrict__ mask)
{
    static_assert(BN == 32 || BN == 64 || BN == 128 || BN == 256, "TMEM columns: a power of two from 32");
    constexpr int kABytes = 128 * KC * 2, kBBytes = BN * KC * 2;
    constexpr int kStage = kABytes + kBBytes;  // multiple of 1024
    extern __shared__ __align__(1024) unsigned char tsm[];
    __shared__ __align__(8) uint64_t full[kTcStages], empty[kTcStages], done;
    __shared__ uint32_t tmem_base;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    // 1024-byte aligned stages (the swizzle pattern repeats every 512 bytes)
    unsigned char* st0 = tsm + ((1024 - (sa(tsm) & 1023)) & 1023);
    const int bpr = W / BW, bpi = bpr * (H / BH);  // pixel blocks per row of blocks, per image
    const int n = blockIdx.x / bpi, rem = blockIdx.x % bpi;
    const int h0 = (rem / bpr) * BH, w0 = (rem % bpr) * BW;
    const int co0 = blockIdx.y * BN;
    const int kc = Cin / KC, ksteps = 9 * kc;

    if (tid == 0) {
        for (int s = 0; s < kTcStages; ++s) {
            mb_init(&full[s], 1);
            mb_init(&empty[s], 1);
        }
        mb_init(&done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sa(&tmem_base)),
                     "r"(BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    pdl_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_next();
    const uint32_t tmem = tmem_base;

    if (warp == 0) {
        // producer: stage k % S holds tap k / kc, channels (k % kc) * 32
        int issued = 0;
        for (int k = 0; k < ksteps; ++k) {
            const int s = k % kTcStages;
            if (k >= kTcStages && !mb_wait(&empty[s], ((k / kTcStages) - 1) & 1)) break;
            unsigned char* a = st0 + s * kStage;
            const int tap = k / kc, c0 = (k % kc) * KC;
            if (elect_one()) {
                mb_expect_tx(&full[s], kStage);
                tma_4d(a, &mx, &full[s], c0, w0 + tap % 3 - 1, h0 + tap / 3 - 1, n);
                tma_3d(a + kABytes, &mw, &full[s], c0, co0, tap);
            }
            __syncwarp();
            issued = k + 1;
        }
        // copies still in flight (only after a wait ran out) land before the CTA ends
        for (int k = issued > kTcStages ? issued - kTcStages : 0; k < issued; ++k)
            mb_wait(&full[k % kTcStages], (k / kTcStages) & 1);
    } else if (warp == 1) {
        // MMA issuer
        constexpr uint32_t idesc = tc_idesc(128, BN);
        for (int k = 0; k < ksteps; ++k) {
            const int s = k % kTcStages;
            if (!mb_wait(&full[s], (k / kTcStages) & 1)) break;
            tc_fence_after();
            const uint32_t a = sa(st0 + s * kStage), b = a + kABytes;
            if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < KC / 16; ++kk)
                    tc_mma(tmem, kmajor_desc<KC>(a + 32 * kk), kmajor_desc<KC>(b + 32 * kk), idesc, (k | kk) != 0);
                tc_commit(&empty[s]);  // stage s is free once these MMAs have read it
            }
            __syncwarp();
        }
        // the accumulator is complete once every MMA issued has finished
        if (elect_one()) tc_commit(&done);
    }
    __syncwarp();

    // epilogue: thread (warp w, lane l) owns pixel 32 w + l of the block
    mb_wait(&done, 0);
    tc_fence_after();
    const int m = warp * 32 + lane;
    const int hh = h0 + m / BW, ww = w0 + m % BW;
    const size_t px = ((size_t)n * H + hh) * W + ww;
    bf16* out = y + px * ldy + co0;
    const bf16* mrow = mask ? mask + px * Cout + co0 : nullptr;
#pragma unroll 1
    for (int c = 0; c < BN; c += 8) {
        uint32_t r[8];
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                     : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        uint32_t o[4];
        uint4 mk = make_uint4(0, 0, 0, 0);
        if (mrow) mk = *reinterpret_cast<const uint4*>(mrow + c);
        const uint32_t mu[4] = {mk.x, mk.y, mk.z, mk.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float v0 = __uint_as_float(r[2 * j]) + (bias ? bias[co0 + c + 2 * j] : 0.f);
            float v1 = __uint_as_float(r[2 * j + 1]) + (bias ? bias[co0 + c + 2 * j + 1] : 0.f);
            if (relu) {
                v0 = fmaxf(v0, 0.f);
                v1 = fmaxf(v1, 0.f);
            }
            if (mrow) {  // bf16 is the upper half of float32
                if (!(__uint_as_float(mu[j] << 16) > 0.f)) v0 = 0.f;
                if (!(__uint_as_float(mu[j] & 0xffff0000u) > 0.f)) v1 = 0.f;
            }
            __nv_bfloat162 t;
            t.x = __float2bfloat16_rn(v0);
            t.y = __float2bfloat16_rn(v1);
            o[j] = *reinterpret_cast<uint32_t*>(&t);
        }
        *reinterpret_cast<uint4*>(out + c) = make_uint4(o[0], o[1], o[2], o[3]);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(BN) : "memory");
}

// ------------------------------------------ tcgen05 convolution on halo tiles
//
// The same GEMMs with the activations staged once per CTA instead of once per tap.  A CTA
// takes MT (1 or 2) blocks of 8 x 16 output pixels side by side (M = 128 each) and BN output
// channels.  One TMA box per KC channels brings the block's pixels and their one-pixel
// frame, (8 MT + 2) x 18 rows of KC channels, zero outside the image.  A tap's operand is
// then a window into that box: 16 groups (image rows) of 8 rows (pixels), the groups one row
// of the box apart, starting (dh + 1) box rows and dw + 1 pixels in.  The box starts on a
// swizzle boundary and the swizzle follows the address bits, so a window may start at any of
// its rows.  Images of other extents have blocks that reach past their edge: the box is zero
// there and nothing is stored.  The weights of each (tap, channel chunk) come through a ring of stages; taps
// outermost, as in k_conv3x3_tc, so that the FP32 sums are the same bit for bit.
//
// What this saves is the way from L2 to the SM, which bounded the per-tap form: 184 MB of
// copies for (4, 128, 512, 32, 32) against 40 MB here, 113 MB against 30 MB for (4, 64, 256,
// 64, 64).
constexpr int kHaloChunks = 12;  // channel chunks of a box (Cin <= 768)
constexpr int kHaloStages = 8;   // weight stages at most
constexpr int kHaloRows = 18;    // box rows: 16 image rows and the frame
// dynamic shared memory at most: what 227 KB leave beside the kernel's own 1.3 KB, in whole KB
constexpr int kHaloSmem = 225 * 1024;

// K-major descriptor with 8-row groups sbo bytes apart (kmajor_desc: 16 KC)
template <int KC>
__device__ __forceinline__ uint64_t kmajor_desc_sbo(uint32_t addr, uint32_t sbo)
{
    constexpr uint64_t mode = KC == 64 ? 2 : 4;
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(sbo >> 4) << 32) |
           ((uint64_t)1 << 46) | (mode << 61);
}
// bytes of one chunk's box, a multiple of the swizzle's 1024
__host__ __device__ constexpr int halo_bytes(int MT, int KC)
{
    return ((8 * MT + 2) * kHaloRows * 2 * KC + 1023) / 1024 * 1024;
}

// The weights' way through shared memory: a stage holds T taps (1, 3 or 9) of CC channel chunks
// of the BN output channels, S stages in use.
struct HaloStages {
    int T, CC, S;
};

template <int KC, int MT>
__global__ void __launch_bounds__(128 * MT)
k_conv3x3_halo(const __grid_constant__ CUtensorMap mx, const __grid_constant__ CUtensorMap mw, int H, int W, int Cin,
               int Cout, int BN, const HaloStages st, const float* __restrict__ bias, int relu, bf16* __restrict__ y,
               int ldy, const bf16* __restrict__ mask)
{
    constexpr int kPitch = 8 * MT + 2, kABytes = halo_bytes(MT, KC), kABox = kPitch * kHaloRows * 2 * KC;
    extern __shared__ __align__(1024) unsigned char tsm[];
    __shared__ __align__(8) uint64_t fullA[kHaloChunks], fullB[kHaloStages], emptyB[kHaloStages], done;
    __shared__ uint32_t tmem_base;
    __shared__ __align__(16) float sbias[256];
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    unsigned char* sA = tsm + ((1024 - (sa(tsm) & 1023)) & 1023);
    const int kc = Cin / KC, kBBytes = BN * KC * 2, kStage = st.T * st.CC * kBBytes;
    unsigned char* sB = sA + kc * kABytes;
    const int bpr = (W + 8 * MT - 1) / (8 * MT), bpi = bpr * ((H + 15) / 16);
    const int n = blockIdx.x / bpi, rem = blockIdx.x % bpi;
    const int h0 = (rem / bpr) * 16, w0 = (rem % bpr) * 8 * MT;
    const int co0 = blockIdx.y * BN;
    uint32_t cols = 32;
    while ((int)cols < MT * BN) cols *= 2;

    if (tid == 0) {
        for (int c = 0; c < kc; ++c) mb_init(&fullA[c], 1);
        for (int s = 0; s < st.S; ++s) {
            mb_init(&fullB[s], 1);
            mb_init(&emptyB[s], 1);
        }
        mb_init(&done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sa(&tmem_base)),
                     "r"(cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    pdl_wait();
    for (int k = tid; k < BN; k += 128 * MT) sbias[k] = bias ? bias[co0 + k] : 0.f;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_next();
    const uint32_t tmem = tmem_base;

    // Stage k covers taps t .. t + T - 1 and chunks c .. c + CC - 1.  All counters advance by
    // additions: divisions by the runtime counts cost more than a stage's MMAs.
    if (warp == 0) {
        // producer: a chunk's box ahead of the weights that need it first
        int s = 0, t = 0, c = 0, issued = 0;
        uint32_t round = 0;  // times the ring has gone round
        for (; t < 9; ++issued) {
            if (round && !mb_wait(&emptyB[s], (round - 1) & 1)) break;
            if (elect_one()) {
                if (t == 0)
                    for (int j = c; j < c + st.CC; ++j) {
                        mb_expect_tx(&fullA[j], kABox);
                        tma_4d(sA + j * kABytes, &mx, &fullA[j], j * KC, w0 - 1, h0 - 1, n);
                    }
                mb_expect_tx(&fullB[s], kStage);
                for (int j = 0; j < st.CC; ++j)
                    tma_3d(sB + s * kStage + j * st.T * kBBytes, &mw, &fullB[s], (c + j) * KC, co0, t);
            }
            __syncwarp();
            if (++s == st.S) { s = 0; ++round; }
            c += st.CC;
            if (c == kc) { c = 0; t += st.T; }
        }
        if (t < 9) {  // a wait ran out: the copies still in flight land before the CTA ends
            for (int j = 0; j < kc && j < issued * st.CC; ++j) mb_wait(&fullA[j], 0);
            for (int k = issued > st.S ? issued - st.S : 0; k < issued; ++k)
                mb_wait(&fullB[k % st.S], (k / st.S) & 1);
        }
    } else if (warp == 1) {
        const uint32_t idesc = tc_idesc(128, BN);
        int s = 0, t = 0, c = 0;
        uint32_t round = 0;
        bool ok = true;
        while (t < 9 && ok) {
            if (t == 0)
                for (int j = c; j < c + st.CC && ok; ++j) ok = mb_wait(&fullA[j], 0);
            ok = ok && mb_wait(&fullB[s], round & 1);
            if (!ok) break;
            tc_fence_after();
            if (elect_one()) {
                // a tap's window starts t / 3 = dh + 1 box rows and t % 3 = dw + 1 pixels in
                int row = t / 3 * kPitch + t % 3, tw = t % 3;
                for (int u = 0; u < st.T; ++u) {
                    uint32_t a0 = sa(sA) + (uint32_t)(c * kABytes + row * 2 * KC);
                    uint32_t b0 = sa(sB) + (uint32_t)(s * kStage + u * kBBytes);
                    for (int j = 0; j < st.CC; ++j) {
                        const uint64_t ad = kmajor_desc_sbo<KC>(a0, kPitch * 2 * KC), bd = kmajor_desc<KC>(b0);
                        const bool first = (t | u | c | j) == 0;
                        // (the address is the descriptor's low field: no step leaves it)
#pragma unroll
                        for (int kk = 0; kk < KC / 16; ++kk)
#pragma unroll
                            for (int q = 0; q < MT; ++q)
                                tc_mma(tmem + (uint32_t)(q * BN), ad + (16 * KC * q + 32 * kk) / 16, bd + 2 * kk, idesc,
                                       !(first && kk == 0));
                        a0 += kABytes;
                        b0 += st.T * kBBytes;
                    }
                    ++row;
                    if (++tw == 3) { tw = 0; row += kPitch - 3; }
                }
                tc_commit(&emptyB[s]);
            }
            __syncwarp();
            if (++s == st.S) { s = 0; ++round; }
            c += st.CC;
            if (c == kc) { c = 0; t += st.T; }
        }
        if (elect_one()) tc_commit(&done);
    }
    __syncwarp();

    // epilogue: warps 4 q .. 4 q + 3 hold block q; thread (warp w, lane l) its pixel m = 32 (w % 4)
    // + l, at row m / 8 and column m % 8 of the block
    const int q = warp >> 2, m = (warp & 3) * 32 + lane;
    const int hh = h0 + m / 8, ww = w0 + 8 * q + m % 8;
    const bool inside = hh < H && ww < W;  // (not so for the last blocks of other extents)
    const size_t px = inside ? ((size_t)n * H + hh) * W + ww : 0;
    bf16* out = y + px * ldy + co0;
    const bf16* mrow = mask ? mask + px * Cout + co0 : nullptr;
    mb_wait(&done, 0);
    tc_fence_after();
#pragma unroll 1
    for (int c = 0; c < BN; c += 32) {
        uint32_t r[32];
        const uint32_t at = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(q * BN + c);
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
            "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
              "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
              "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
              "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
            : "r"(at));
        uint4 mk[4];
        if (mrow) {
#pragma unroll
            for (int j = 0; j < 4; ++j) mk[j] = *reinterpret_cast<const uint4*>(mrow + c + 8 * j);
        }
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t o[4];
            const uint32_t mu[4] = {mk[j].x, mk[j].y, mk[j].z, mk[j].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 bb = *reinterpret_cast<const float2*>(&sbias[c + 8 * j + 2 * e]);
                float v0 = __uint_as_float(r[8 * j + 2 * e]) + bb.x, v1 = __uint_as_float(r[8 * j + 2 * e + 1]) + bb.y;
                if (relu) {
                    v0 = fmaxf(v0, 0.f);
                    v1 = fmaxf(v1, 0.f);
                }
                if (mrow) {  // bf16 is the upper half of float32
                    if (!(__uint_as_float(mu[e] << 16) > 0.f)) v0 = 0.f;
                    if (!(__uint_as_float(mu[e] & 0xffff0000u) > 0.f)) v1 = 0.f;
                }
                const __nv_bfloat162 t2 = __floats2bfloat162_rn(v0, v1);
                o[e] = *reinterpret_cast<const uint32_t*>(&t2);
            }
            if (inside) *reinterpret_cast<uint4*>(out + c + 8 * j) = make_uint4(o[0], o[1], o[2], o[3]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}

// dW[tap][co][ci] += sum_p dz[p][co] x[p + off(tap)][ci], db[co] += sum_p dz[p][co].
// CTA: one tap, WM co x 32 ci, a chunk of 32 pixels at a time over its pixel range;
// accumulates in FP32 and adds into dW with atomics.  4 warps: WM/16 row blocks of
// 16 output channels times 64/WM groups of n-tiles.
constexpr int kWN = 32, kWK = 32;
template <int WM, bool PART>
__global__ void __launch_bounds__(128)
k_conv3x3_wgrad(const bf16* __restrict__ x, const bf16* __restrict__ dz, int N, int H, int W, int Cin, int Cout,
                int pix_per_cta, float* __restrict__ dw, float* __restrict__ db, float* __restrict__ part)
{
    pdl_enter_small();
    constexpr int RB = WM / 16;        // row blocks
    constexpr int NG = 4 / RB;         // n-tile groups
    constexpr int NTW = 4 / NG;        // n-tiles (of 8 ci) per warp
    __shared__ __align__(16) bf16 Az[WM][kWK + kPad];   // [co][p]
    __shared__ __align__(16) bf16 Bx[kWN][kWK + kPad];  // [ci][p]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, tig = lane & 3;
    const int rb = warp % RB, ng = warp / RB;
    const int tap = blockIdx.z % 9, split = blockIdx.z / 9;
    const int dh = tap / 3 - 1, dwd = tap % 3 - 1;
    const int co0 = blockIdx.y * WM, ci0 = blockIdx.x * kWN;
    const long long P = (long long)N * H * W;
    const long long p_begin = (long long)split * pix_per_cta;
    const long long p_end = p_begin + pix_per_cta < P ? p_begin + pix_per_cta : P;
    float acc[NTW][4];
#pragma unroll
    for (int j = 0; j < NTW; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
    float bacc = 0.f;
    if constexpr (PART) {  // this split's own sums, stored (as in k_conv3x3_wgrad_tc)
        dw = part + (size_t)split * ((size_t)9 * Cout * Cin + Cout);
        db = dw + (size_t)9 * Cout * Cin;
    }
    const bool do_bias = db && tap == 4 && blockIdx.x == 0;

    for (long long p0 = p_begin; p0 < p_end; p0 += kWK) {
        // dz tile: 32 pixels x WM co -> Az[co][p]
        for (int k = tid; k < kWK * WM; k += 128) {
            const int pl = k / WM, co = k % WM;
            const long long p = p0 + pl;
            bf16 v = __float2bfloat16_rn(0.f);
            if (p < p_end) v = dz[p * Cout + co0 + co];
            Az[co][pl] = v;
        }
        // x tile at the tap offset: 32 pixels x 32 ci -> Bx[ci][p]
        for (int k = tid; k < kWK * kWN; k += 128) {
            const int pl = k / kWN, ci = k % kWN;
            const long long p = p0 + pl;
            bf16 v = __float2bfloat16_rn(0.f);
            if (p < p_end) {
                const int w = (int)(p % W), hrow = (int)((p / W) % H), nn = (int)(p / ((long long)W * H));
                const int hh = hrow + dh, ww = w + dwd;
                if (hh >= 0 && hh < H && ww >= 0 && ww < W) v = x[(((long long)nn * H + hh) * W + ww) * Cin + ci0 + ci];
            }
            Bx[ci][pl] = v;
        }
        __syncthreads();
        if (do_bias && tid < WM) {
            for (int pl = 0; pl < kWK; ++pl) bacc += __bfloat162float(Az[tid][pl]);
        }
#pragma unroll
        for (int ks = 0; ks < kWK; ks += 16) {
            uint32_t a[4];
            const int r0 = rb * 16 + g;
            a[0] = ld_pair(&Az[r0][ks + 2 * tig]);
            a[1] = ld_pair(&Az[r0 + 8][ks + 2 * tig]);
            a[2] = ld_pair(&Az[r0][ks + 2 * tig + 8]);
            a[3] = ld_pair(&Az[r0 + 8][ks + 2 * tig + 8]);
#pragma unroll
            for (int j = 0; j < NTW; ++j) {
                const int nt = ng * NTW + j;
                uint32_t b[2];
                b[0] = ld_pair(&Bx[nt * 8 + g][ks + 2 * tig]);
                b[1] = ld_pair(&Bx[nt * 8 + g][ks + 2 * tig + 8]);
                mma_bf16(acc[j], a, b);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < NTW; ++j) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int co = co0 + rb * 16 + g + 8 * r;
            const int ci = ci0 + (ng * NTW + j) * 8 + 2 * tig;
            float* dst = dw + ((size_t)tap * Cout + co) * Cin + ci;
            if constexpr (PART) {
                dst[0] = acc[j][2 * r];
                dst[1] = acc[j][2 * r + 1];
            } else {
                atomicAdd(dst, acc[j][2 * r]);
                atomicAdd(dst + 1, acc[j][2 * r + 1]);
            }
        }
    }
    if (do_bias && tid < WM) {
        if constexpr (PART) db[co0 + tid] = bacc;
        else atomicAdd(db + co0 + tid, bacc);
    }
}

// flipped transposes for the data gradients: wd[tap][ci][co] = w[8 - tap][co][ci], of up to
// kMaxFlips layers in one launch (blockIdx.y; 3 us each on its own)
constexpr int kMaxFlips = 16;
struct FlipList {
    const bf16* w[kMaxFlips];
    bf16* wd[kMaxFlips];
    int cin[kMaxFlips], cout[kMaxFlips];
};
__global__ void __launch_bounds__(256) k_flip_weights(const FlipList L)
{
    pdl_enter();
    // 32 x 32 (co, ci) tiles of one tap through shared memory, so that both sides are read
    // and written in whole rows
    __shared__ bf16 t[32][33];
    const int l = blockIdx.y, cin = L.cin[l], cout = L.cout[l];
    const int ti = cin / 32, to = cout / 32;
    const bf16* w = L.w[l];
    bf16* wd = L.wd[l];
    for (int k = blockIdx.x; k < 9 * ti * to; k += gridDim.x) {
        const int tap = k / (ti * to), ci0 = 32 * ((k / to) % ti), co0 = 32 * (k % to);
        for (int r = threadIdx.x >> 5; r < 32; r += 8)
            t[r][threadIdx.x & 31] = w[((size_t)(8 - tap) * cout + co0 + r) * cin + ci0 + (threadIdx.x & 31)];
        __syncthreads();
        for (int r = threadIdx.x >> 5; r < 32; r += 8)
            wd[((size_t)tap * cin + ci0 + r) * cout + co0 + (threadIdx.x & 31)] = t[threadIdx.x & 31][r];
        __syncthreads();
    }
}

// The element-wise kernels come in two forms: eight channels (one 16-byte piece) per thread
// where every channel count and offset is a multiple of eight and every tensor 16-byte
// aligned (all of the network's calls), and one element per thread for the rest.  They
// move memory and nothing else; the scalar forms spent their time on 2-byte accesses and
// 64-bit divisions per element (a training step of batch 4 at 512 x 128: upsampling 144 us,
// now 16; pooling's gradient 75, now 15).
struct Piece {
    float v[8];
};
__device__ __forceinline__ Piece ld8(const bf16* p)
{
    const uint4 q = *reinterpret_cast<const uint4*>(p);
    const uint32_t u[4] = {q.x, q.y, q.z, q.w};
    Piece r;
#pragma unroll
    for (int j = 0; j < 4; ++j) {  // bf16 is the upper half of float32
        r.v[2 * j] = __uint_as_float(u[j] << 16);
        r.v[2 * j + 1] = __uint_as_float(u[j] & 0xffff0000u);
    }
    return r;
}
__device__ __forceinline__ void st8(bf16* p, const Piece& r)
{
    uint32_t u[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const __nv_bfloat162 t = __floats2bfloat162_rn(r.v[2 * j], r.v[2 * j + 1]);
        u[j] = *reinterpret_cast<const uint32_t*>(&t);
    }
    *reinterpret_cast<uint4*>(p) = make_uint4(u[0], u[1], u[2], u[3]);
}
// zero where the mask's element is not positive
__device__ __forceinline__ void relu_back8(Piece& d, const Piece& y)
{
#pragma unroll
    for (int j = 0; j < 8; ++j)
        if (!(y.v[j] > 0.f)) d.v[j] = 0.f;
}

// ------------------------------------------------ tcgen05 weight gradient
//
// dW[tap][co][ci] += sum_p dz[p][co] x[p + off(tap)][ci], with blocks of BW x BH pixels as K steps
// and one column offset dw of the taps per CTA: a stage holds the block of dz (64 output channels
// per box, two boxes when there are more) and the block of x shifted by dw with a row above and
// below, BH + 2 rows of BW pixels by CK input channels.  Both are MN-major, one pixel's channels
// per row.  The three taps of the column are one MMA: its N runs over three blocks of CK channels
// that lie one image row (BW rows of shared memory) apart, so the operand's windows are the taps'
// shifts and dz is read from shared memory once for the three.  M = 128 output channels (past the
// boxes that exist, lanes hold sums that are not read), N = 3 CK, K = 16 pixels, 16 rows of the
// block.  db is summed from the dz boxes by four more warps in the CTAs of dw = -1 and the first
// input channels, each thread eight channels of every fourth pixel.  Partial sums of a CTA go to
// dw in vector reductions (dw off the 16-byte rule: one by one).  Blocks that reach past an image's
// edge add nothing: dz is zero there.  With PART the sums of each split are stored instead, for
// k_sum_parts to add up in one order.
//
// Blocks: segments of 64 x 1 where the width allows, else 8 x 16.  The segments' order and their
// split over CTAs decide which products meet in which float32 sum, and training amplifies that: a
// first step of Adam turns a change of a gradient near zero into one of up to a whole step, and
// sums over 8 x 16 blocks, as accurate as these, moved the second step's gradients by 1e-4.  So the
// order is fixed (wgrad_splits): every tap's sum runs through its CTA's segments from left to right
// and from top to bottom, 16 pixels at a time.
//
// Weight and bias gradient, batch 4 (us, against one tap or column of taps per MMA in the same
// order): 512 x 128 32 -> 32 82 -> 30, 96 -> 32 188 -> 57; 256 x 64 64 -> 64 35 -> 13, 192 -> 64 78 ->
// 28; 64 x 16 256 -> 256 37 -> 10 (8 x 16 blocks, which stage x 1.1 times instead of 3: 17, 40, 11, 19
// and 9).  Bound by staging from L2 and by the reductions at the end.
constexpr int kWgStages = 4;
constexpr int kWgPix = 64;  // pixels of a row segment
// bytes of a dz box (BW x BH pixels of 64 channels) and of the x box
__host__ __device__ constexpr int wg_dz(int BW, int BH) { return BW * BH * 128; }
__host__ __device__ constexpr int wg_x(int BW, int BH, int CK) { return BW * (BH + 2) * 2 * CK; }

// MN-major descriptor: rows of CK channels (64 or 128 bytes, swizzled over the row), groups of
// eight rows sbo bytes apart along K, blocks of a row's channels lbo bytes apart along M or N
template <int CK>
__device__ __forceinline__ uint64_t mnmajor_desc2(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    constexpr uint64_t mode = CK == 64 ? 2 : 4;
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           ((uint64_t)1 << 46) | (mode << 61);
}
__device__ __forceinline__ void red_add4(float* p, const uint32_t* r)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(__uint_as_float(r[0])),
                 "f"(__uint_as_float(r[1])), "f"(__uint_as_float(r[2])), "f"(__uint_as_float(r[3]))
                 : "memory");
}

template <int CK, int BW, int BH, bool PART>
__global__ void __launch_bounds__(256)
k_conv3x3_wgrad_tc(const __grid_constant__ CUtensorMap mdz, const __grid_constant__ CUtensorMap mx, int N, int H,
                   int W, int Cin, int Cout, int tiles_per_cta, float* __restrict__ dw, float* __restrict__ db,
                   float* __restrict__ part)
{
    static_assert(BW % 8 == 0 && BW * BH % 64 == 0, "whole groups of eight rows, sixteen pixels per MMA and bias warp");
    constexpr int kPix = BW * BH, kDz = wg_dz(BW, BH), kX = wg_x(BW, BH, CK);
    constexpr int kRow = BW * 2 * CK;  // one image row of the x box
    constexpr uint32_t kCols = CK == 64 ? 256 : 128;        // TMEM columns: 3 CK in use
    // MN-major A and B (transpose bits)
    constexpr uint32_t idesc = tc_idesc(128, 3 * CK) | (1u << 15) | (1u << 16);
    extern __shared__ __align__(1024) unsigned char tsm[];
    __shared__ __align__(8) uint64_t full[kWgStages], empty[kWgStages], done;
    __shared__ uint32_t tmem_base;
    __shared__ float sdb[4][128];
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    unsigned char* st0 = tsm + ((1024 - (sa(tsm) & 1023)) & 1023);
    const int co0 = blockIdx.x * 128, ci0 = blockIdx.y * CK;
    const int g = blockIdx.z % 3, split = blockIdx.z / 3;
    const int nb = co0 + 64 < Cout ? 2 : 1;  // dz boxes
    const int boxes = Cout > 64 ? 2 : 1;     // room for them
    const int kStage = boxes * kDz + kX;
    const int bpr = (W + BW - 1) / BW, bpi = bpr * ((H + BH - 1) / BH), tiles = N * bpi;
    const int begin = split * tiles_per_cta, end = min(begin + tiles_per_cta, tiles), steps = max(end - begin, 0);
    if constexpr (PART) {  // this split's own sums (of all taps, then of the bias), stored
        dw = part + (size_t)split * ((size_t)9 * Cout * Cin + Cout);
        db = dw + (size_t)9 * Cout * Cin;
    }
    const bool bias = db && g == 0 && blockIdx.y == 0;

    if (tid == 0) {
        for (int s = 0; s < kWgStages; ++s) {
            mb_init(&full[s], 1);
            mb_init(&empty[s], bias ? 5 : 1);  // the MMAs and, with the bias, its four warps
        }
        mb_init(&done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sa(&tmem_base)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    pdl_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_next();
    const uint32_t tmem = tmem_base;

    if (warp == 0) {
        int n = begin / bpi, rem = begin - n * bpi, row = rem / bpr, col = rem - row * bpr, issued = 0;
        for (; issued < steps; ++issued) {
            const int s = issued % kWgStages;
            if (issued >= kWgStages && !mb_wait(&empty[s], (issued / kWgStages - 1) & 1)) break;
            if (elect_one()) {
                unsigned char* a = st0 + s * kStage;
                mb_expect_tx(&full[s], nb * kDz + kX);
                tma_4d(a, &mdz, &full[s], co0, BW * col, BH * row, n);
                if (nb == 2) tma_4d(a + kDz, &mdz, &full[s], co0 + 64, BW * col, BH * row, n);
                tma_4d(a + boxes * kDz, &mx, &full[s], ci0, BW * col + g - 1, BH * row - 1, n);
            }
            __syncwarp();
            if (++col == bpr) {
                col = 0;
                if (++row * bpr == bpi) { row = 0; ++n; }
            }
        }
        if (issued < steps)  // a wait ran out: the copies still in flight land before the CTA ends
            for (int k = max(issued - kWgStages, 0); k < issued; ++k) mb_wait(&full[k % kWgStages], (k / kWgStages) & 1);
    } else if (warp == 1) {
        for (int k = 0; k < steps; ++k) {
            const int s = k % kWgStages;
            if (!mb_wait(&full[s], (k / kWgStages) & 1)) break;
            tc_fence_after();
            if (elect_one()) {
                const uint32_t a = sa(st0 + s * kStage), b = a + boxes * kDz;
                // (with one dz box the second block of M is the first one's rows 8 and on)
                const uint64_t ad = mnmajor_desc2<64>(a, nb == 2 ? kDz : 1024, 1024);
                const uint64_t bd = mnmajor_desc2<CK>(b, kRow, 8 * 2 * CK);
#pragma unroll
                for (int kk = 0; kk < kPix / 16; ++kk)
                    tc_mma(tmem, ad + 16 * 128 / 16 * kk, bd + 16 * 2 * CK / 16 * kk, idesc, (k | kk) != 0);
                tc_commit(&empty[s]);
            }
            __syncwarp();
        }
        if (elect_one()) tc_commit(&done);
    } else if (warp >= 4 && bias) {
        // lane: 16-byte piece lane % 8 of a row, pixels kPix / 4 (warp - 4) + 4 j + lane / 8
        const int piece = lane & 7, p0 = kPix / 4 * (warp - 4) + (lane >> 3);
        float acc[2][8] = {};
        for (int k = 0; k < steps; ++k) {
            const int s = k % kWgStages;
            if (!mb_wait(&full[s], (k / kWgStages) & 1)) break;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if (q >= nb) break;
                const unsigned char* a = st0 + s * kStage + q * kDz;
                float part[8] = {};
#pragma unroll
                for (int j = 0; j < kPix / 16; ++j) {
                    const int p = p0 + 4 * j;
                    const Piece v = ld8(reinterpret_cast<const bf16*>(a + 128 * p + 16 * (piece ^ (p & 7))));
#pragma unroll
                    for (int e = 0; e < 8; ++e) part[e] += v.v[e];
                }
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[q][e] += part[e];
            }
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sa(&empty[s])) : "memory");
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                float v = acc[q][e];
                v += __shfl_xor_sync(0xffffffffu, v, 8);
                v += __shfl_xor_sync(0xffffffffu, v, 16);
                if (lane < 8) sdb[warp - 4][64 * q + 8 * piece + e] = v;
            }
        }
    }
    __syncwarp();

    // thread (warp w, lane l) owns output channel co0 + 32 (w % 4) + l (its TMEM lane); warps 4-7
    // take the second half of the columns
    mb_wait(&done, 0);
    tc_fence_after();
    const int co = co0 + (warp & 3) * 32 + lane;
    const bool mine = steps > 0 && co < Cout, vec = ((uintptr_t)dw & 15) == 0;
    constexpr int kHalf = 3 * CK / 2;
#pragma unroll 1
    for (int c = (warp >> 2) * kHalf; c < ((warp >> 2) + 1) * kHalf; c += 16) {
        uint32_t r[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
            "%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
              "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (mine) {
            // columns c .. c + 15: tap 3 (c / CK) + g, input channels ci0 + c % CK and on
            float* dst = dw + ((size_t)(3 * (c / CK) + g) * Cout + co) * Cin + ci0 + c % CK;
#pragma unroll
            for (int j = 0; j < 16; j += 4) {
                if constexpr (PART) {
                    *reinterpret_cast<uint4*>(dst + j) = make_uint4(r[j], r[j + 1], r[j + 2], r[j + 3]);
                } else if (vec) {
                    red_add4(dst + j, r + j);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e) atomicAdd(dst + j + e, __uint_as_float(r[j + e]));
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (bias && tid < 128 && co0 + tid < Cout) {  // one atomic per CTA and channel
        const float v = (sdb[0][tid] + sdb[1][tid]) + (sdb[2][tid] + sdb[3][tid]);
        if constexpr (PART) db[co0 + tid] = v;
        else atomicAdd(db + co0 + tid, v);
    }
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

// dst[k] += the sum over p of part[p * stride + k], for up to kMaxSums ranges in one launch: the
// parameter gradients of a backward pass from the partial sums that its kernels stored.  Added in
// one order, with the rounding errors carried along, so the result is the same on every run and the
// nearest float32 to the partial sums' sum but for one rounding.  A thread takes four words of a
// range of up to 64 partial sums that allows it, a warp one word of any other (the head's: 304).  Bound by
// reading the partial sums (22 M words, 88 MB, for the whole network at batch 4).
constexpr int kMaxSums = 32;
struct SumList {
    const float* part[kMaxSums];
    float* dst[kMaxSums];
    long long stride[kMaxSums];
    int count[kMaxSums], parts[kMaxSums];
    int first[kMaxSums + 1];  // first block of each range
    uint32_t four;            // bit i: range i goes by four words
};
struct Carried {  // a float32 sum and the rounding errors it left
    float s, c;
    __device__ __forceinline__ void add(float v)
    {
        const float t = s + v, b = t - s;
        c += (s - (t - b)) + (v - b);
        s = t;
    }
};
__global__ void __launch_bounds__(256) k_sum_parts(const SumList L, int n)
{
    pdl_enter();
    int i = 0;
    while (i + 1 < n && (int)blockIdx.x >= L.first[i + 1]) ++i;
    const int block = (int)blockIdx.x - L.first[i], parts = L.parts[i];
    const long long stride = L.stride[i];
    if (L.four >> i & 1) {
        const int k = 4 * (block * 256 + (int)threadIdx.x);
        if (k >= L.count[i]) return;
        float4* dst = reinterpret_cast<float4*>(L.dst[i] + k);
        const float* p = L.part[i] + k;
        const float4 d = *dst;
        Carried a[4] = {{d.x, 0.f}, {d.y, 0.f}, {d.z, 0.f}, {d.w, 0.f}};
        for (int q = 0; q < parts; q += 8, p += 8 * stride) {
            float4 v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                v[j] = q + j < parts ? *reinterpret_cast<const float4*>(p + j * stride) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 8; ++j) {  // (adding zero changes nothing)
                a[0].add(v[j].x);
                a[1].add(v[j].y);
                a[2].add(v[j].z);
                a[3].add(v[j].w);
            }
        }
        *dst = make_float4(a[0].s + a[0].c, a[1].s + a[1].c, a[2].s + a[2].c, a[3].s + a[3].c);
        return;
    }
    const int k = block * 8 + (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (k >= L.count[i]) return;
    const float* p = L.part[i] + k;
    Carried a{lane == 0 ? L.dst[i][k] : 0.f, 0.f};
    for (int q = lane; q < parts; q += 32) a.add(p[q * stride]);
    for (int o = 16; o > 0; o >>= 1) {
        const float s = __shfl_down_sync(0xffffffffu, a.s, o), c = __shfl_down_sync(0xffffffffu, a.c, o);
        a.add(s);
        a.c += c;
    }
    if (lane == 0) L.dst[i][k] = a.s + a.c;
}

__global__ void k_relu_mask8(bf16* __restrict__ d, const bf16* __restrict__ y, long long pieces)
{
    pdl_enter();
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < pieces; k += (long long)gridDim.x * blockDim.x) {
        Piece v = ld8(d + 8 * k);
        relu_back8(v, ld8(y + 8 * k));
        st8(d + 8 * k, v);
    }
}
// The image kernels below: blockIdx.y walks the rows (of all images), threads the pieces of
// a row; C8 pieces per pixel.
// x: ldx channels per pixel
__global__ void k_pool8(const bf16* __restrict__ x, int rows, int W, int C8, int ldx, bf16* __restrict__ y)
{
    pdl_enter();
    const int Wo = W / 2, C = 8 * C8;
    for (int r = blockIdx.y; r < rows; r += gridDim.y)  // output row: image rows 2 r, 2 r + 1
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < Wo * C8; k += gridDim.x * blockDim.x) {
            const int w = k / C8, c = 8 * (k - w * C8);
            const bf16* b = x + ((size_t)2 * r * W + 2 * w) * ldx + c;
            const Piece p0 = ld8(b), p1 = ld8(b + ldx), p2 = ld8(b + (size_t)W * ldx),
                        p3 = ld8(b + (size_t)W * ldx + ldx);
            Piece o;
#pragma unroll
            for (int j = 0; j < 8; ++j) o.v[j] = 0.25f * (p0.v[j] + p1.v[j] + p2.v[j] + p3.v[j]);
            st8(y + ((size_t)r * Wo + w) * C + c, o);
        }
}
// rows: coarse rows; one thread serves the 2 x 2 fine pixels of a coarse one.  dx = dy / 4,
// plus `add` (lda channels per pixel; may be dx itself) when given, zero where `mask` (ldm
// channels per pixel) is not positive when given.
__global__ void k_pool_back8(const bf16* __restrict__ dy, int rows, int W, int C8, const bf16* add, int lda,
                             const bf16* __restrict__ mask, int ldm, bf16* dx)
{
    pdl_enter();
    const int Wo = W / 2, C = 8 * C8;
    for (int r = blockIdx.y; r < rows; r += gridDim.y)
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < Wo * C8; k += gridDim.x * blockDim.x) {
            const int w = k / C8, c = 8 * (k - w * C8);
            const Piece g = ld8(dy + ((size_t)r * Wo + w) * C + c);
            Piece old[4], mk[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const size_t px = (size_t)(2 * r + q / 2) * W + 2 * w + q % 2;
                if (add) old[q] = ld8(add + px * lda + c);
                if (mask) mk[q] = ld8(mask + px * ldm + c);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const size_t px = (size_t)(2 * r + q / 2) * W + 2 * w + q % 2;
                Piece v;
#pragma unroll
                for (int j = 0; j < 8; ++j) v.v[j] = add ? 0.25f * g.v[j] + old[q].v[j] : 0.25f * g.v[j];
                if (mask) relu_back8(v, mk[q]);
                st8(dx + px * C + c, v);
            }
        }
}
__global__ void k_up_into8(const bf16* __restrict__ x, int rows, int W, int C8, bf16* __restrict__ y, int Ctot, int cofs)
{
    pdl_enter();
    const int Wo = W / 2, C = 8 * C8;
    for (int r = blockIdx.y; r < rows; r += gridDim.y)
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < Wo * C8; k += gridDim.x * blockDim.x) {
            const int w = k / C8, c = 8 * (k - w * C8);
            const uint4 v = *reinterpret_cast<const uint4*>(x + ((size_t)r * Wo + w) * C + c);
            bf16* d = y + ((size_t)2 * r * W + 2 * w) * Ctot + cofs + c;
            *reinterpret_cast<uint4*>(d) = v;
            *reinterpret_cast<uint4*>(d + Ctot) = v;
            *reinterpret_cast<uint4*>(d + (size_t)W * Ctot) = v;
            *reinterpret_cast<uint4*>(d + (size_t)W * Ctot + Ctot) = v;
        }
}
// zero where `mask` (laid out as dx) is not positive, when given
__global__ void k_up_back8(const bf16* __restrict__ dy, int rows, int W, int Ctot, int cofs, int C8,
                           const bf16* __restrict__ mask, bf16* __restrict__ dx)
{
    pdl_enter();
    const int Wo = W / 2, C = 8 * C8;
    for (int r = blockIdx.y; r < rows; r += gridDim.y)
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < Wo * C8; k += gridDim.x * blockDim.x) {
            const int w = k / C8, c = 8 * (k - w * C8);
            const bf16* b = dy + ((size_t)2 * r * W + 2 * w) * Ctot + cofs + c;
            const Piece p0 = ld8(b), p1 = ld8(b + Ctot), p2 = ld8(b + (size_t)W * Ctot),
                        p3 = ld8(b + (size_t)W * Ctot + Ctot);
            Piece o;
#pragma unroll
            for (int j = 0; j < 8; ++j) o.v[j] = p0.v[j] + p1.v[j] + p2.v[j] + p3.v[j];
            const size_t at = ((size_t)r * Wo + w) * C + c;
            if (mask) relu_back8(o, ld8(mask + at));
            st8(dx + at, o);
        }
}
__global__ void k_channels8(const bf16* __restrict__ src, int Sc, int sofs, long long pixels, int C8,
                            bf16* __restrict__ dst, int Dc, int dofs, int accumulate)
{
    pdl_enter();
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < pixels * C8; k += (long long)gridDim.x * blockDim.x) {
        const long long p = k / C8;
        const int c = 8 * (int)(k - p * C8);
        const bf16* a = src + p * Sc + sofs + c;
        bf16* d = dst + p * Dc + dofs + c;
        if (!accumulate) {
            *reinterpret_cast<uint4*>(d) = *reinterpret_cast<const uint4*>(a);
            continue;
        }
        Piece v = ld8(a);
        const Piece old = ld8(d);
#pragma unroll
        for (int j = 0; j < 8; ++j) v.v[j] += old.v[j];
        st8(d, v);
    }
}

__global__ void k_relu_mask(bf16* __restrict__ d, const bf16* __restrict__ y, long long count)
{
    pdl_enter();
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < count; k += (long long)gridDim.x * blockDim.x)
        if (!(__bfloat162float(y[k]) > 0.f)) d[k] = __float2bfloat16_rn(0.f);
}

// 2x2 average pooling and its adjoint; nearest upsampling and its adjoint
__global__ void k_pool(const bf16* __restrict__ x, int N, int H, int W, int C, bf16* __restrict__ y)
{
    pdl_enter();
    const int Ho = H / 2, Wo = W / 2;
    const long long total = (long long)N * Ho * Wo * C;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < total; k += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(k % C);
        long long r = k / C;
        const int wo = (int)(r % Wo); r /= Wo;
        const int ho = (int)(r % Ho);
        const int n = (int)(r / Ho);
        const size_t b = (((size_t)n * H + 2 * ho) * W + 2 * wo) * C + c;
        const float s = __bfloat162float(x[b]) + __bfloat162float(x[b + C]) + __bfloat162float(x[b + (size_t)W * C]) +
                        __bfloat162float(x[b + (size_t)W * C + C]);
        y[k] = __float2bfloat16_rn(0.25f * s);
    }
}
// dx[fine] (+)= dy[coarse] / 4
__global__ void k_pool_back(const bf16* __restrict__ dy, int N, int H, int W, int C, bf16* __restrict__ dx, int accumulate)
{
    pdl_enter();
    const long long total = (long long)N * H * W * C;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < total; k += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(k % C);
        long long r = k / C;
        const int w = (int)(r % W); r /= W;
        const int hh = (int)(r % H);
        const int n = (int)(r / H);
        float v = 0.25f * __bfloat162float(dy[(((size_t)n * (H / 2) + hh / 2) * (W / 2) + w / 2) * C + c]);
        if (accumulate) v += __bfloat162float(dx[k]);
        dx[k] = __float2bfloat16_rn(v);
    }
}
// y[n, h, w, cofs + c] = x[n, h/2, w/2, c] : upsampled x into channels [cofs, cofs + C) of a Ctot tensor
__global__ void k_up_into(const bf16* __restrict__ x, int N, int H, int W, int C, bf16* __restrict__ y, int Ctot, int cofs)
{
    pdl_enter();
    const long long total = (long long)N * H * W * C;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < total; k += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(k % C);
        long long r = k / C;
        const int w = (int)(r % W); r /= W;
        const int hh = (int)(r % H);
        const int n = (int)(r / H);
        y[(((size_t)n * H + hh) * W + w) * Ctot + cofs + c] = x[(((size_t)n * (H / 2) + hh / 2) * (W / 2) + w / 2) * C + c];
    }
}
// dx[coarse] = sum of the 4 fine dy values in channels [cofs, cofs + C) of a Ctot tensor
__global__ void k_up_back(const bf16* __restrict__ dy, int N, int H, int W, int Ctot, int cofs, int C, bf16* __restrict__ dx)
{
    pdl_enter();
    const int Ho = H / 2, Wo = W / 2;
    const long long total = (long long)N * Ho * Wo * C;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < total; k += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(k % C);
        long long r = k / C;
        const int wo = (int)(r % Wo); r /= Wo;
        const int ho = (int)(r % Ho);
        const int n = (int)(r / Ho);
        const size_t b = (((size_t)n * H + 2 * ho) * W + 2 * wo) * Ctot + cofs + c;
        const float s = __bfloat162float(dy[b]) + __bfloat162float(dy[b + Ctot]) +
                        __bfloat162float(dy[b + (size_t)W * Ctot]) + __bfloat162float(dy[b + (size_t)W * Ctot + Ctot]);
        dx[k] = __float2bfloat16_rn(s);
    }
}
// copy channels [sofs, sofs + C) of an Sc-channel tensor into channels [dofs, dofs + C) of a Dc-channel
// tensor (concatenation and its adjoint split); accumulate adds into the destination
__global__ void k_channels(const bf16* __restrict__ src, int Sc, int sofs, long long pixels, int C, bf16* __restrict__ dst,
                           int Dc, int dofs, int accumulate)
{
    pdl_enter();
    const long long total = pixels * C;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < total; k += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(k % C);
        const long long p = k / C;
        float v = __bfloat162float(src[p * Sc + sofs + c]);
        bf16* d = dst + p * Dc + dofs + c;
        if (accumulate) v += __bfloat162float(*d);
        *d = __float2bfloat16_rn(v);
    }
}

// The head with one pixel per thread: its C channels in 16-byte pieces, the weights in
// shared memory, the outputs of a block leaving through shared memory in one run.  C a
// multiple of 8, at most 8 outputs, 16-byte aligned x.
template <int CO>
__global__ void __launch_bounds__(256)
k_head8(const bf16* __restrict__ x, long long pixels, int C, const float* __restrict__ Wt, const float* __restrict__ b,
        float* __restrict__ out)
{
    pdl_enter();
    extern __shared__ float shw[];  // C x CO weights, then 256 x CO outputs
    float* sho = shw + C * CO;
    for (int k = threadIdx.x; k < C * CO; k += 256) shw[k] = Wt[k];
    float bo[CO];
#pragma unroll
    for (int o = 0; o < CO; ++o) bo[o] = b[o];
    __syncthreads();
    for (long long p0 = blockIdx.x * 256LL; p0 < pixels; p0 += gridDim.x * 256LL) {
        const long long p = p0 + threadIdx.x;
        if (p < pixels) {
            float s[CO];
#pragma unroll
            for (int o = 0; o < CO; ++o) s[o] = bo[o];
            for (int c = 0; c < C; c += 8) {
                const Piece v = ld8(x + p * C + c);
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int o = 0; o < CO; ++o) s[o] = fmaf(v.v[j], shw[(c + j) * CO + o], s[o]);
            }
#pragma unroll
            for (int o = 0; o < CO; ++o) sho[threadIdx.x * CO + o] = s[o];
        }
        __syncthreads();
        const int m = (int)(pixels - p0 < 256 ? pixels - p0 : 256) * CO;
        for (int k = threadIdx.x; k < m; k += 256) out[p0 * CO + k] = sho[k];
        __syncthreads();
    }
}
// Head gradients, C = 8 G with G a power of two up to 32: lane l of a warp holds channels
// 8 (l % G) .. + 7 of pixel l / G, their weights and the FP32 partial sums of dW and db in
// registers over all its pixels; shuffles, shared memory and one atomic per block and
// parameter add them up (with `part` a block stores its sums, of dW and then of db).  Bound by reading x and dout and writing dx.  (Adding every
// pixel's products into shared memory with atomics serialised each warp on the same C x CO
// words: 1,147 us at 262,144 pixels, C = 32, 5 outputs.)
template <int CO>
__global__ void __launch_bounds__(256)
k_head_back8(const bf16* __restrict__ x, const float* __restrict__ dout, long long pixels, int C,
             const float* __restrict__ Wt, bf16* __restrict__ dx, float* __restrict__ dW, float* __restrict__ db,
             int relu, float* __restrict__ part)
{
    pdl_enter();
    extern __shared__ float sh[];  // C * CO + CO sums
    const int G = C >> 3, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cg = lane & (G - 1), ps = lane / G, PP = 32 / G;
    float w[8][CO], acc[8][CO], accb[CO];
#pragma unroll
    for (int o = 0; o < CO; ++o) {
        accb[o] = 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            w[j][o] = Wt[(8 * cg + j) * CO + o];
            acc[j][o] = 0.f;
        }
    }
    for (int k = threadIdx.x; k < (C + 1) * CO; k += 256) sh[k] = 0.f;
    __syncthreads();
    for (long long p = ((long long)blockIdx.x * 8 + warp) * PP + ps; p < pixels; p += (long long)gridDim.x * 8 * PP) {
        float d[CO];
#pragma unroll
        for (int o = 0; o < CO; ++o) d[o] = dout[p * CO + o];
        const Piece v = ld8(x + p * C + 8 * cg);
        Piece r;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float s = 0.f;
#pragma unroll
            for (int o = 0; o < CO; ++o) {
                s = fmaf(d[o], w[j][o], s);
                acc[j][o] = fmaf(v.v[j], d[o], acc[j][o]);
            }
            r.v[j] = s;
        }
        if (relu) relu_back8(r, v);
        st8(dx + p * C + 8 * cg, r);
#pragma unroll
        for (int o = 0; o < CO; ++o) accb[o] += d[o];
    }
    for (int m = G; m < 32; m <<= 1) {
#pragma unroll
        for (int o = 0; o < CO; ++o) {
            accb[o] += __shfl_xor_sync(0xffffffffu, accb[o], m);
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j][o] += __shfl_xor_sync(0xffffffffu, acc[j][o], m);
        }
    }
    for (int q = 0; q < 8; ++q) {  // warp by warp, in one order
        if (warp == q && ps == 0) {
#pragma unroll
            for (int o = 0; o < CO; ++o) {
#pragma unroll
                for (int j = 0; j < 8; ++j) sh[(8 * cg + j) * CO + o] += acc[j][o];
                if (cg == 0) sh[C * CO + o] += accb[o];
            }
        }
        __syncthreads();
    }
    if (part) {
        for (int k = threadIdx.x; k < (C + 1) * CO; k += 256) part[(size_t)blockIdx.x * ((C + 1) * CO) + k] = sh[k];
        return;
    }
    for (int k = threadIdx.x; k < C * CO; k += 256) atomicAdd(&dW[k], sh[k]);
    for (int k = threadIdx.x; k < CO; k += 256) atomicAdd(&db[k], sh[C * CO + k]);
}

// 1x1 head: out[p][o] = b[o] + sum_c x[p][c] W[c][o] (FP32 weights and output)
__global__ void k_head(const bf16* __restrict__ x, long long pixels, int C, const float* __restrict__ Wt,
                       const float* __restrict__ b, int Cout, float* __restrict__ out)
{
    pdl_enter();
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < pixels * Cout; k += (long long)gridDim.x * blockDim.x) {
        const int o = (int)(k % Cout);
        const long long p = k / Cout;
        float s = b[o];
        for (int c = 0; c < C; ++c) s = fmaf(__bfloat162float(x[p * C + c]), Wt[c * Cout + o], s);
        out[k] = s;
    }
}
// head gradients: dx[p][c] = sum_o dout[p][o] W[c][o]; dW[c][o] += sum_p x[p][c] dout[p][o]; db[o] += sum_p dout[p][o]
__global__ void k_head_back(const bf16* __restrict__ x, const float* __restrict__ dout, long long pixels, int C,
                            const float* __restrict__ Wt, int Cout, bf16* __restrict__ dx, float* __restrict__ dW,
                            float* __restrict__ db)
{
    pdl_enter();
    extern __shared__ float sh[];  // C * Cout + Cout partial sums
    for (int k = threadIdx.x; k < C * Cout + Cout; k += blockDim.x) sh[k] = 0.f;
    __syncthreads();
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < pixels; p += (long long)gridDim.x * blockDim.x) {
        for (int c = 0; c < C; ++c) {
            float s = 0.f;
            const float xv = __bfloat162float(x[p * C + c]);
            for (int o = 0; o < Cout; ++o) {
                const float d = dout[p * Cout + o];
                s = fmaf(d, Wt[c * Cout + o], s);
                atomicAdd(&sh[c * Cout + o], xv * d);
            }
            dx[p * C + c] = __float2bfloat16_rn(s);
        }
        for (int o = 0; o < Cout; ++o) atomicAdd(&sh[C * Cout + o], dout[p * Cout + o]);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < C * Cout; k += blockDim.x) atomicAdd(&dW[k], sh[k]);
    for (int k = threadIdx.x; k < Cout; k += blockDim.x) atomicAdd(&db[k], sh[C * Cout + k]);
}

// mean squared error with channel weights; grad = d loss / d pred; loss accumulated in FP64
__global__ void __launch_bounds__(256) k_mse(const float* __restrict__ pred, const float* __restrict__ target, const float* __restrict__ wch,
                      long long count, int C, float* __restrict__ grad, double* __restrict__ loss)
{
    pdl_enter();
    double acc = 0.0;
    const float inv = 1.f / (float)count;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < count; k += (long long)gridDim.x * blockDim.x) {
        const float wc = wch ? wch[k % C] : 1.f;
        const float d = pred[k] - target[k];
        acc += (double)d * d * wc;
        if (grad) grad[k] = 2.f * d * wc * inv;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    // one atomic per block: they queue up on the one word (one per warp of 1,024 blocks took
    // 19 us at 1.3 M elements)
    __shared__ double part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) acc += part[w];
        atomicAdd(loss, acc / (double)count);
    }
}

// Adam on FP32 master weights, refreshing the bf16 copy used by the convolutions
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ gr, float* __restrict__ m, float* __restrict__ v,
                       long long count, float lr, float b1, float b2, float eps, float c1, float c2,
                       bf16* __restrict__ pb)
{
    pdl_enter();
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < count; k += (long long)gridDim.x * blockDim.x) {
        const float gk = gr[k];
        const float mk = b1 * m[k] + (1.f - b1) * gk;
        const float vk = b2 * v[k] + (1.f - b2) * gk * gk;
        m[k] = mk;
        v[k] = vk;
        const float pk = p[k] - lr * (mk * c1) / (sqrtf(vk * c2) + eps);
        p[k] = pk;
        if (pb) pb[k] = __float2bfloat16_rn(pk);
    }
}

__global__ void k_to_bf16(const float* __restrict__ x, long long count, bf16* __restrict__ y)
{
    pdl_enter();
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < count; k += (long long)gridDim.x * blockDim.x)
        y[k] = __float2bfloat16_rn(x[k]);
}

// planar float fields <-> interleaved NHWC tensors, with a per-channel affine map
constexpr int kMaxPackC = 8;
struct Affine {
    float scale[kMaxPackC], shift[kMaxPackC];
};
__global__ void k_pack(const float* __restrict__ src, const float* __restrict__ base, long long plane, int C,
                       long long pixels, Affine a, void* __restrict__ dst, int Cd, int bf)
{
    pdl_enter();
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < pixels * C; k += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(k % C);
        const long long p = k / C;
        const float d = src[c * plane + p] - (base ? base[c * plane + p] : 0.f);
        const float v = fmaf(d, a.scale[c], a.shift[c]);
        if (bf) ((bf16*)dst)[p * Cd + c] = __float2bfloat16_rn(v);
        else ((float*)dst)[p * Cd + c] = v;
    }
}
__global__ void k_unpack(const float* __restrict__ src, long long pixels, int C, Affine a, const float* __restrict__ base,
                         float* __restrict__ dst, long long plane)
{
    pdl_enter();
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < pixels * C; k += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(k % C);
        const long long p = k / C;
        dst[c * plane + p] = fmaf(src[k], a.scale[c], a.shift[c]) + (base ? base[c * plane + p] : 0.f);
    }
}

// One warp waits in the manner of the issuing warps' loops on a barrier that completes: in block
// 0 with every lane's polls, in block 1 with one lane that has none.  out[2 block]: lanes that
// left the loop, out[2 block + 1]: the error flag.
__global__ void __launch_bounds__(64) k_wait_check(uint32_t polls, int* out)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mb_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 32) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sa(&bar)) : "memory");
    if (threadIdx.x >= 32) return;
    bool left = false;
    for (int k = 0; k < 2; ++k) {
        if (!mb_wait(&bar, 0, blockIdx.x == 1 && threadIdx.x == 5 ? 0 : polls, out + 2 * blockIdx.x + 1)) {
            left = true;
            break;
        }
        elect_one();
        __syncwarp();
    }
    const unsigned m = __ballot_sync(0xffffffffu, left);
    if (threadIdx.x == 0) out[2 * blockIdx.x] = __popc(m);
}

int grid_of(long long count)
{
    long long b = (count + 255) / 256;
    return (int)(b < 152 * 32 ? (b < 1 ? 1 : b) : 152 * 32);
}

// whether tensors and channel counts allow 16-byte pieces
template <class... P>
bool pieces(int channels, P... p)
{
    return channels % 8 == 0 && ((... | (uintptr_t)p) & 15) == 0;
}
// grid of the row kernels: `per_row` pieces in each of `rows` rows (one idle block for none: an
// empty batch is no error)
dim3 grid_rows(int rows, int per_row)
{
    return dim3(std::max(1, (per_row + 255) / 256), std::max(1, std::min(rows, 65535)));
}

int status(cudaError_t e) { return e == cudaSuccess ? TPF_OK : TPF_ERR_CUDA; }

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
        else
            cudaGetLastError();
    }
    return fn;
}

// Images of fewer pixels whose blocks do not divide evenly stay on the mma.sync kernels: no level
// of a network has them, and they keep those kernels in use.  It is not where the two are level
// (us forward and weight gradient, tcgen05 / mma.sync: 31 x 33, 64 -> 64 4.9/17.5 and 4.4/9.1, 9 x 11
// 4.8/16.1 and 4.3/7.1).
constexpr long long kRaggedPixels = 1024;

// Shapes the tcgen05 convolutions take: images that divide into pixel blocks of BW x BH = 128
// (BW = W up to 128, dividing W; BH dividing H; BW 0 where they do not), and any other of at
// least kRaggedPixels pixels (halo form).  BN: the largest of 256, 128, 64, 32 that divides
// Cout and still gives at least one CTA per SM (else 32).  0 when the shape is not taken.
int tc_bn(int N, int H, int W, int Cout, int& BW, int& BH)
{
    BW = W < 128 ? W : 128;
    BH = BW > 0 && 128 % BW == 0 ? 128 / BW : 0;
    if (BH == 0 || W % BW != 0 || H % BH != 0) {
        BW = BH = 0;
        if ((long long)N * H * W < kRaggedPixels) return 0;
    }
    const long long mtiles = BW ? (long long)N * (H / BH) * (W / BW) : (long long)N * ((H + 15) / 16) * ((W + 7) / 8);
    for (int bn = 256; bn > 32; bn /= 2)
        if (Cout % bn == 0 && mtiles * (Cout / bn) >= 152) return bn;
    return 32;
}

// tensor maps of the convolutions: pixel boxes of an NHWC tensor
bool pixel_map(CUtensorMap* m, const bf16* x, int N, int H, int W, int C, int KC, int bw, int bh)
{
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)N};
    cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2};
    cuuint32_t box[4] = {(cuuint32_t)KC, (cuuint32_t)bw, (cuuint32_t)bh, 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void*)x, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
              KC == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// and KC channels x BN output channels x T taps of the [9][Cout][Cin] weights
bool weight_map(CUtensorMap* m, const bf16* wt, int Cin, int Cout, int KC, int BN, int T)
{
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {(cuuint64_t)Cin, (cuuint64_t)Cout, 9};
    cuuint64_t strides[2] = {(cuuint64_t)Cin * 2, (cuuint64_t)Cout * Cin * 2};
    cuuint32_t box[3] = {(cuuint32_t)KC, (cuuint32_t)BN, (cuuint32_t)T};
    cuuint32_t es[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)wt, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
              KC == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The tcgen05 convolution for 16-byte aligned tensors of a shape tc_bn takes; returns
// false (nothing launched) otherwise.
template <int BN, int KC>
bool launch_tc(const bf16* x, int N, int H, int W, int Cin, const bf16* wt, const float* bias, int Cout, int relu,
               bf16* y, int ldy, const bf16* mask, cudaStream_t s, int BW, int BH)
{
    CUtensorMap mx, mw;
    if (!pixel_map(&mx, x, N, H, W, Cin, KC, BW, BH) || !weight_map(&mw, wt, Cin, Cout, KC, BN, 1)) return false;
    const int smem = kTcStages * (128 + BN) * KC * 2 + 1024;
    // set on every call: the attribute belongs to the current device
    if (cudaFuncSetAttribute(k_conv3x3_tc<BN, KC>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    dim3 grd(N * (H / BH) * (W / BW), Cout / BN);
    launch_pdl(k_conv3x3_tc<BN, KC>, grd, 128, smem, s, mx, mw, H, W, Cin, Cout, BW, BH, bias, relu, y, ldy, mask);
    return true;
}

// The kernel that a convolution of 16-byte aligned tensors takes: bn output channels per tile (0:
// the mma.sync kernel), KC channels per chunk, and the halo form (MT blocks per CTA, its weight
// stages, its shared memory) or the per-tap one (st.S = 0; blocks of BW x BH).  The one place
// where this is decided, for the launches and for tpfnet_conv3x3_tcgen05.
struct ConvPlan {
    int bn, KC, MT, smem, BW, BH;
    HaloStages st;
};
ConvPlan plan_conv(int N, int H, int W, int Cin, int Cout)
{
    ConvPlan p{};
    p.bn = tc_bn(N, H, W, Cout, p.BW, p.BH);
    p.KC = Cin % 64 == 0 ? 64 : 32;
    const int kc = Cin / p.KC;
    if (!p.bn || kc < 1) return ConvPlan{};
    const bool any = p.BW == 0;  // an extent that only the halo form takes
    if ((H % 16 == 0 && W % 8 == 0) || any) {
        // two blocks per CTA where that still gives every SM a CTA (half the weight traffic)
        const long long pairs = (long long)N * ((H + 15) / 16) * ((W + 15) / 16);
        p.MT = (W % 16 == 0 || any) && pairs * (Cout / p.bn) >= 152 ? 2 : 1;
        const int a = kc * halo_bytes(p.MT, p.KC) + 1024, b = p.bn * p.KC * 2;
        // The fewest and largest weight stages that fit: a wait and its loop cost about as much as
        // eight MMAs.  With more CTAs than SMs, two to an SM: all nine taps at once, three at a
        // time, or one; where the boxes leave no room for that, the per-tap kernel is the better
        // one ((4, 32, 128, 384, 128): 22.9 us against 31.1, (4, 16, 64, 256, 256): 16.8 against
        // 17.7).  With at most one CTA per SM its whole shared memory, and parts of a tap if need be.
        const long long blocks = (long long)N * ((H + 15) / 16) * ((W + 8 * p.MT - 1) / (8 * p.MT));
        const long long ctas = blocks * (Cout / p.bn);
        const int limit = ctas > 152 ? 112 * 1024 : kHaloSmem;
        auto take = [&](int T, int CC, int S) {
            if (p.st.S || CC < 1 || kc % CC || (long long)a + (long long)S * T * CC * b > limit) return;
            p.st = {T, CC, S};
        };
        if (kc <= kHaloChunks) {
            take(9, kc, 1);
            take(3, kc, 3);
            take(1, kc, 4);
            take(1, kc, 3);
            if (ctas <= 152) {
                take(1, kc / 2, 4);
                take(1, kc / 3, 4);
                take(1, 1, 4);
            }
        }
        p.smem = a + p.st.S * p.st.T * p.st.CC * b;
        if (!p.st.S && any) return ConvPlan{};
    }
    return p;
}

// The halo form; false (nothing launched) when it cannot be.
template <int KC, int MT>
bool launch_halo(const ConvPlan& p, const bf16* x, int N, int H, int W, int Cin, const bf16* wt, const float* bias, int Cout,
                 int relu, bf16* y, int ldy, const bf16* mask, cudaStream_t s)
{
    CUtensorMap mx, mw;
    if (!pixel_map(&mx, x, N, H, W, Cin, KC, 8 * MT + 2, kHaloRows) || !weight_map(&mw, wt, Cin, Cout, KC, p.bn, p.st.T))
        return false;
    // set on every call (the attribute belongs to the current device), and always to the same size:
    // another thread may be between its setting and its launch
    if (cudaFuncSetAttribute(k_conv3x3_halo<KC, MT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kHaloSmem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    const dim3 grd((unsigned)(N * ((H + 15) / 16) * ((W + 8 * MT - 1) / (8 * MT))), Cout / p.bn);
    launch_pdl(k_conv3x3_halo<KC, MT>, grd, 128 * MT, p.smem, s, mx, mw, H, W, Cin, Cout, p.bn, p.st, bias, relu, y, ldy, mask);
    return true;
}

bool conv_tc(const bf16* x, int N, int H, int W, int Cin, const bf16* wt, const float* bias, int Cout, int relu,
             bf16* y, int ldy, const bf16* mask, cudaStream_t s)
{
    if ((((uintptr_t)x | (uintptr_t)wt | (uintptr_t)y | (uintptr_t)mask) & 15) || ldy % 8) return false;
    const ConvPlan p = plan_conv(N, H, W, Cin, Cout);
    if (!p.bn) return false;
    if (p.st.S) {
        const auto f = p.KC == 64 ? (p.MT == 2 ? launch_halo<64, 2> : launch_halo<64, 1>)
                                  : (p.MT == 2 ? launch_halo<32, 2> : launch_halo<32, 1>);
        return f(p, x, N, H, W, Cin, wt, bias, Cout, relu, y, ldy, mask, s);
    }
    const auto f = p.KC == 64 ? (p.bn == 256 ? launch_tc<256, 64> : p.bn == 128 ? launch_tc<128, 64>
                                 : p.bn == 64 ? launch_tc<64, 64> : launch_tc<32, 64>)
                              : (p.bn == 256 ? launch_tc<256, 32> : p.bn == 128 ? launch_tc<128, 32>
                                 : p.bn == 64 ? launch_tc<64, 32> : launch_tc<32, 32>);
    return f(x, N, H, W, Cin, wt, bias, Cout, relu, y, ldy, mask, s, p.BW, p.BH);
}

// CTAs over which the 64 x 1 segments of an image batch are split, `per` segments each: about as
// many as run at once when each takes 64 input channels of one tap (from kWgTaps3Pixels pixels up
// of three).  Part of the results (see k_conv3x3_wgrad_tc), not of the launch: what a CTA takes
// otherwise does not move it.
constexpr long long kWgTaps3Pixels = 1 << 17;
long long wgrad_splits(int N, int H, int W, int Cin, int Cout, long long& per)
{
    const long long P = (long long)N * H * W, nchunks = (long long)N * H * (W / kWgPix);
    const int taps = P >= kWgTaps3Pixels ? 3 : 1;
    const long long base = (9 / taps) * (long long)((Cout + 127) / 128) * ((Cin + 63) / 64);
    const long long target = taps == 1 ? 2 * 152 : 152;
    const long long splits = std::max(1LL, std::min(nchunks, (target + base - 1) / base));
    per = (nchunks + splits - 1) / splits;
    return (nchunks + per - 1) / per;
}

// Which weight gradient a shape takes, for 16-byte aligned x and dz, and how its pixels are split
// over CTAs: rows of whole segments, images that divide into blocks of 8 x 16, and any other large
// enough take the tcgen05 kernel with CK input channels per CTA (CK = 0: the mma.sync kernel, WM
// output channels per CTA), in `splits` runs of `per` blocks (pixels).
struct WgradPlan {
    int CK, WM, splits, per;
    bool rows;
};
WgradPlan plan_wgrad(int N, int H, int W, int Cin, int Cout, bool aligned)
{
    WgradPlan p{};
    const long long P = (long long)N * H * W;
    long long splits, per;
    p.rows = W % kWgPix == 0;
    if (!aligned || !encode_fn() || (!p.rows && !(H % 16 == 0 && W % 8 == 0) && P < kRaggedPixels)) {
        p.WM = Cout % 64 == 0 ? 64 : 32;
        // split the pixels so that the grid fills the GPU a few times over
        const long long base = 9LL * (Cin / kWN) * (Cout / p.WM);
        splits = std::max(1LL, std::min((152LL * 8 + base - 1) / base, (P + kWK - 1) / kWK));
        per = ((P + splits - 1) / splits + kWK - 1) / kWK * kWK;
        splits = (P + per - 1) / per;
    } else {
        p.CK = Cin % 64 == 0 ? 64 : 32;
        if (p.rows) {
            splits = wgrad_splits(N, H, W, Cin, Cout, per);
        } else {
            // split the blocks over about as many CTAs as run at once
            const int stage = (Cout > 64 ? 2 : 1) * wg_dz(8, 16) + wg_x(8, 16, p.CK);
            const long long tiles = (long long)N * ((H + 15) / 16) * ((W + 7) / 8);
            const long long base = 3LL * ((Cout + 127) / 128) * (Cin / p.CK);
            const long long target = kWgStages * stage + 1024 <= 112 * 1024 ? 304 : 152;
            splits = std::max(1LL, std::min(tiles, target / base));
            per = (tiles + splits - 1) / splits;
            splits = (tiles + per - 1) / per;
        }
    }
    p.splits = (int)splits;
    p.per = (int)per;
    return p;
}

// The weight gradient on blocks of BW x BH; false (nothing launched) when it cannot be.
template <int CK, int BW, int BH>
bool launch_wgrad(const WgradPlan& p, const bf16* x, const bf16* dz, int N, int H, int W, int Cin, int Cout, float* dw,
                  float* db, float* part, cudaStream_t s)
{
    const auto kern = part ? k_conv3x3_wgrad_tc<CK, BW, BH, true> : k_conv3x3_wgrad_tc<CK, BW, BH, false>;
    CUtensorMap mdz, mx;
    if (!pixel_map(&mdz, dz, N, H, W, Cout, 64, BW, BH) || !pixel_map(&mx, x, N, H, W, Cin, CK, BW, BH + 2)) return false;
    const int smem = kWgStages * ((Cout > 64 ? 2 : 1) * wg_dz(BW, BH) + wg_x(BW, BH, CK)) + 1024;
    // (always the size of two dz boxes: another thread may be between its setting and its launch)
    constexpr int kMost = kWgStages * (2 * wg_dz(BW, BH) + wg_x(BW, BH, CK)) + 1024;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    launch_pdl(kern, dim3((Cout + 127) / 128, Cin / CK, 3 * (unsigned)p.splits), 256, smem, s, mdz, mx, N, H, W, Cin, Cout,
               p.per, dw, db, part);
    return true;
}

// The weight gradient by p; false (nothing launched) when that cannot be.  Adds into dw (and db),
// or stores the splits' sums into part.
bool wgrad(const WgradPlan& p, const bf16* x, const bf16* dz, int N, int H, int W, int Cin, int Cout, float* dw, float* db,
           float* part, cudaStream_t s)
{
    if (p.CK) {
        const auto f = p.rows ? (p.CK == 64 ? launch_wgrad<64, kWgPix, 1> : launch_wgrad<32, kWgPix, 1>)
                              : (p.CK == 64 ? launch_wgrad<64, 8, 16> : launch_wgrad<32, 8, 16>);
        return f(p, x, dz, N, H, W, Cin, Cout, dw, db, part, s);
    }
    const dim3 grd(Cin / kWN, Cout / p.WM, 9 * p.splits);
    const auto f = part ? (p.WM == 64 ? k_conv3x3_wgrad<64, true> : k_conv3x3_wgrad<32, true>)
                        : (p.WM == 64 ? k_conv3x3_wgrad<64, false> : k_conv3x3_wgrad<32, false>);
    launch_pdl_small(f, grd, 128, s, x, dz, N, H, W, Cin, Cout, p.per, dw, db, part);
    return true;
}

}  // namespace

extern "C" {

static int conv_any(const void* x, int N, int H, int W, int Cin, const void* wt, const float* bias, int Cout, int relu,
                    void* y, int ldy, const void* mask, void* stream)
{
    if (!x || !wt || !y || N < 1 || H < 1 || W < 1 || Cin % kKC || Cout % 32) return TPF_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (conv_tc((const bf16*)x, N, H, W, Cin, (const bf16*)wt, bias, Cout, relu, (bf16*)y, ldy, (const bf16*)mask, s))
        return status(cudaGetLastError());
    // the mma.sync kernel reads 16-byte pieces and writes pairs of channels
    if ((((uintptr_t)x | (uintptr_t)wt) & 15) || ((uintptr_t)y & 3) || ldy % 2) return TPF_ERR_INVALID_ARG;
    const int wblocks = (W + kBM - 1) / kBM;
    if (Cout % 64 == 0) {
        dim3 grd(wblocks * N * H, Cout / 64);
        launch_pdl_small(k_conv3x3<64>, grd, 128, s, (const bf16*)x, N, H, W, Cin, (const bf16*)wt, bias, Cout, relu, (bf16*)y,
                                      ldy, (const bf16*)mask);
    } else {
        dim3 grd(wblocks * N * H, Cout / 32);
        launch_pdl_small(k_conv3x3<32>, grd, 128, s, (const bf16*)x, N, H, W, Cin, (const bf16*)wt, bias, Cout, relu, (bf16*)y,
                                      ldy, (const bf16*)mask);
    }
    return status(cudaGetLastError());
}

int tpfnet_conv3x3(const void* x, int N, int H, int W, int Cin, const void* wt, const float* bias, int Cout, int relu,
                   void* y, void* stream)
{
    return conv_any(x, N, H, W, Cin, wt, bias, Cout, relu, y, Cout, nullptr, stream);
}

int tpfnet_conv3x3_into(const void* x, int N, int H, int W, int Cin, const void* wt, const float* bias, int Cout,
                        int relu, void* y, int ldy, void* stream)
{
    if (ldy < Cout || ldy % 2) return TPF_ERR_INVALID_ARG;
    return conv_any(x, N, H, W, Cin, wt, bias, Cout, relu, y, ldy, nullptr, stream);
}

int tpfnet_conv3x3_dgrad_masked(const void* dz, int N, int H, int W, int Cout, const void* wflip, int Cin,
                                const void* mask, void* dx, void* stream)
{
    return conv_any(dz, N, H, W, Cout, wflip, nullptr, Cin, 0, dx, Cin, mask, stream);
}

int tpfnet_flip_weights(int layers, const void* const* wt, const int* cin, const int* cout, void* const* wflip,
                        void* stream)
{
    if (layers < 1 || layers > kMaxFlips || !wt || !cin || !cout || !wflip) return TPF_ERR_INVALID_ARG;
    FlipList L{};
    int most = 0;
    for (int l = 0; l < layers; ++l) {
        if (!wt[l] || !wflip[l] || cin[l] < 32 || cout[l] < 32 || cin[l] % 32 || cout[l] % 32) return TPF_ERR_INVALID_ARG;
        L.w[l] = (const bf16*)wt[l];
        L.wd[l] = (bf16*)wflip[l];
        L.cin[l] = cin[l];
        L.cout[l] = cout[l];
        const int tiles = 9 * (cin[l] / 32) * (cout[l] / 32);
        if (tiles > most) most = tiles;
    }
    launch_pdl(k_flip_weights, dim3(most < 304 ? most : 304, layers), 256, 0, (cudaStream_t)stream, L);
    return status(cudaGetLastError());
}

int tpfnet_conv3x3_tcgen05(int N, int H, int W, int Cin, int Cout)
{
    if (N < 1 || H < 1 || W < 1 || Cin % kKC || Cout % 32 || !encode_fn()) return 0;
    return plan_conv(N, H, W, Cin, Cout).bn;
}

int tpfnet_wgrad_parts(int N, int H, int W, int Cin, int Cout)
{
    if (N < 1 || H < 1 || W < 1 || Cin < 32 || Cout < 32 || Cin % 32 || Cout % 32) return 0;
    return plan_wgrad(N, H, W, Cin, Cout, true).splits;
}

int tpfnet_conv3x3_wgrad_tcgen05(int N, int H, int W, int Cin, int Cout)
{
    if (N < 1 || H < 1 || W < 1 || Cin < 32 || Cout < 32 || Cin % 32 || Cout % 32) return 0;
    return plan_wgrad(N, H, W, Cin, Cout, true).CK > 0 ? 1 : 0;
}

int tpfnet_status(void)
{
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_tc_err, sizeof(int)) != cudaSuccess) return TPF_ERR_CUDA;
    return v ? TPF_ERR_TIMEOUT : TPF_OK;
}

int tpfnet_check_bounded_wait(int polls, int out[4])
{
    if (polls < 1 || !out) return TPF_ERR_INVALID_ARG;
    int* d = nullptr;
    cudaError_t e = cudaMalloc(&d, 4 * sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(d, 0, 4 * sizeof(int));
    if (e == cudaSuccess) {
        k_wait_check<<<2, 64>>>((uint32_t)polls, d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, d, 4 * sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return status(e);
}

int tpfnet_conv3x3_dgrad(const void* dz, int N, int H, int W, int Cout, const void* wt, int Cin, void* wflip, void* dx,
                         void* stream)
{
    if (!dz || !wt || !wflip || !dx || Cin % 32 || Cout % kKC) return TPF_ERR_INVALID_ARG;
    int rc = tpfnet_flip_weights(1, &wt, &Cin, &Cout, &wflip, stream);
    if (rc) return rc;
    return tpfnet_conv3x3(dz, N, H, W, Cout, wflip, nullptr, Cin, 0, dx, stream);
}

int tpfnet_conv3x3_wgrad(const void* x, const void* dz, int N, int H, int W, int Cin, int Cout, float* dw, float* db,
                         void* stream)
{
    if (!x || !dz || !dw || N < 1 || H < 1 || W < 1 || Cin < kWN || Cout < 32 || Cin % kWN || Cout % 32)
        return TPF_ERR_INVALID_ARG;
    const bool aligned = !(((uintptr_t)x | (uintptr_t)dz) & 15);
    for (const bool tc : {aligned, false})  // (the mma.sync kernel where the other cannot be launched)
        if (wgrad(plan_wgrad(N, H, W, Cin, Cout, tc), (const bf16*)x, (const bf16*)dz, N, H, W, Cin, Cout, dw, db, nullptr,
                  (cudaStream_t)stream))
            break;
    return status(cudaGetLastError());
}

int tpfnet_conv3x3_wgrad_part(const void* x, const void* dz, int N, int H, int W, int Cin, int Cout, float* part,
                              void* stream)
{
    if (!x || !dz || !part || !tpfnet_wgrad_parts(N, H, W, Cin, Cout) ||
        (((uintptr_t)x | (uintptr_t)dz | (uintptr_t)part) & 15))
        return TPF_ERR_INVALID_ARG;
    const bool ok = wgrad(plan_wgrad(N, H, W, Cin, Cout, true), (const bf16*)x, (const bf16*)dz, N, H, W, Cin, Cout, nullptr,
                          nullptr, part, (cudaStream_t)stream);
    return ok ? status(cudaGetLastError()) : TPF_ERR_CUDA;
}

int tpfnet_sum_parts(int n, const float* const* part, const long long* stride, const int* count, const int* parts,
                     float* const* dst, void* stream)
{
    if (n < 1 || n > kMaxSums || !part || !stride || !count || !parts || !dst) return TPF_ERR_INVALID_ARG;
    SumList L{};
    for (int i = 0; i < n; ++i) {
        if (!part[i] || !dst[i] || count[i] < 1 || parts[i] < 1 || stride[i] < count[i]) return TPF_ERR_INVALID_ARG;
        L.part[i] = part[i];
        L.dst[i] = dst[i];
        L.stride[i] = stride[i];
        L.count[i] = count[i];
        L.parts[i] = parts[i];
        // (more partial sums than that are a chain too long for one thread)
        const bool four = parts[i] <= 64 && ((uintptr_t)part[i] & 15) == 0 && ((uintptr_t)dst[i] & 15) == 0 &&
                          stride[i] % 4 == 0 && count[i] % 4 == 0;
        L.four |= (uint32_t)four << i;
        L.first[i + 1] = L.first[i] + (four ? (count[i] + 1023) / 1024 : (count[i] + 7) / 8);
    }
    launch_pdl(k_sum_parts, L.first[n], 256, 0, (cudaStream_t)stream, L, n);
    return status(cudaGetLastError());
}

int tpfnet_relu_mask(void* d, const void* y, long long count, void* stream)
{
    if (pieces((int)(count % 8), d, y)) {
        launch_pdl(k_relu_mask8, grid_of(count / 8), 256, 0, (cudaStream_t)stream, (bf16*)d, (const bf16*)y, count / 8);
        return status(cudaGetLastError());
    }
    launch_pdl(k_relu_mask, grid_of(count), 256, 0, (cudaStream_t)stream, (bf16*)d, (const bf16*)y, count);
    return status(cudaGetLastError());
}

int tpfnet_pool(const void* x, int N, int H, int W, int C, void* y, void* stream)
{
    if (H % 2 || W % 2) return TPF_ERR_INVALID_ARG;
    if (pieces(C, x, y)) {
        launch_pdl(k_pool8, grid_rows(N * (H / 2), W / 2 * (C / 8)), 256, 0, (cudaStream_t)stream, (const bf16*)x, N * (H / 2), W,
                                                                                         C / 8, C, (bf16*)y);
        return status(cudaGetLastError());
    }
    launch_pdl(k_pool, grid_of((long long)N * H * W * C / 4), 256, 0, (cudaStream_t)stream, (const bf16*)x, N, H, W, C, (bf16*)y);
    return status(cudaGetLastError());
}

int tpfnet_pool_back(const void* dy, int N, int H, int W, int C, void* dx, int accumulate, void* stream)
{
    if (H % 2 == 0 && W % 2 == 0 && pieces(C, dy, dx)) {
        launch_pdl(k_pool_back8, grid_rows(N * (H / 2), W / 2 * (C / 8)), 256, 0, (cudaStream_t)stream, 
            (const bf16*)dy, N * (H / 2), W, C / 8, accumulate ? (const bf16*)dx : nullptr, C, nullptr, 0, (bf16*)dx);
        return status(cudaGetLastError());
    }
    launch_pdl(k_pool_back, grid_of((long long)N * H * W * C), 256, 0, (cudaStream_t)stream, (const bf16*)dy, N, H, W, C, (bf16*)dx,
                                                                                    accumulate);
    return status(cudaGetLastError());
}

int tpfnet_up_into(const void* x, int N, int H, int W, int C, void* y, int Ctot, int cofs, void* stream)
{
    if (H % 2 == 0 && W % 2 == 0 && pieces(C | Ctot | cofs, x, y)) {
        launch_pdl(k_up_into8, grid_rows(N * (H / 2), W / 2 * (C / 8)), 256, 0, (cudaStream_t)stream, 
            (const bf16*)x, N * (H / 2), W, C / 8, (bf16*)y, Ctot, cofs);
        return status(cudaGetLastError());
    }
    launch_pdl(k_up_into, grid_of((long long)N * H * W * C), 256, 0, (cudaStream_t)stream, (const bf16*)x, N, H, W, C, (bf16*)y,
                                                                                  Ctot, cofs);
    return status(cudaGetLastError());
}

int tpfnet_up_back(const void* dy, int N, int H, int W, int Ctot, int cofs, int C, void* dx, void* stream)
{
    if (H % 2 == 0 && W % 2 == 0 && pieces(C | Ctot | cofs, dy, dx)) {
        launch_pdl(k_up_back8, grid_rows(N * (H / 2), W / 2 * (C / 8)), 256, 0, (cudaStream_t)stream, 
            (const bf16*)dy, N * (H / 2), W, Ctot, cofs, C / 8, nullptr, (bf16*)dx);
        return status(cudaGetLastError());
    }
    launch_pdl(k_up_back, grid_of((long long)N * H * W * C / 4), 256, 0, (cudaStream_t)stream, (const bf16*)dy, N, H, W, Ctot, cofs,
                                                                                       C, (bf16*)dx);
    return status(cudaGetLastError());
}

int tpfnet_pool_from(const void* x, int N, int H, int W, int C, int ldx, void* y, void* stream)
{
    if (!x || !y || N < 1 || H < 2 || W < 2 || H % 2 || W % 2 || C < 8 || ldx < C || !pieces(C | ldx, x, y))
        return TPF_ERR_INVALID_ARG;
    launch_pdl(k_pool8, grid_rows(N * (H / 2), W / 2 * (C / 8)), 256, 0, (cudaStream_t)stream, (const bf16*)x, N * (H / 2), W, C / 8,
                                                                                     ldx, (bf16*)y);
    return status(cudaGetLastError());
}

int tpfnet_pool_back_skip(const void* dy, int N, int H, int W, int C, const void* skip, int lds, const void* mask,
                          int ldm, void* dx, void* stream)
{
    if (!dy || !skip || !mask || !dx || N < 1 || H < 2 || W < 2 || H % 2 || W % 2 || C < 8 || lds < C || ldm < C ||
        !pieces(C | lds | ldm, dy, skip, mask, dx))
        return TPF_ERR_INVALID_ARG;
    launch_pdl(k_pool_back8, grid_rows(N * (H / 2), W / 2 * (C / 8)), 256, 0, (cudaStream_t)stream, 
        (const bf16*)dy, N * (H / 2), W, C / 8, (const bf16*)skip, lds, (const bf16*)mask, ldm, (bf16*)dx);
    return status(cudaGetLastError());
}

int tpfnet_up_back_masked(const void* dy, int N, int H, int W, int Ctot, int cofs, int C, const void* mask, void* dx,
                          void* stream)
{
    if (!dy || !mask || !dx || N < 1 || H < 2 || W < 2 || H % 2 || W % 2 || C < 8 || cofs < 0 || cofs + C > Ctot ||
        !pieces(C | Ctot | cofs, dy, mask, dx))
        return TPF_ERR_INVALID_ARG;
    launch_pdl(k_up_back8, grid_rows(N * (H / 2), W / 2 * (C / 8)), 256, 0, (cudaStream_t)stream, 
        (const bf16*)dy, N * (H / 2), W, Ctot, cofs, C / 8, (const bf16*)mask, (bf16*)dx);
    return status(cudaGetLastError());
}

int tpfnet_channels(const void* src, int Sc, int sofs, long long pixels, int C, void* dst, int Dc, int dofs,
                    int accumulate, void* stream)
{
    if (pieces(C | Sc | sofs | Dc | dofs, src, dst)) {
        launch_pdl(k_channels8, grid_of(pixels * (C / 8)), 256, 0, (cudaStream_t)stream, (const bf16*)src, Sc, sofs, pixels, C / 8,
                                                                               (bf16*)dst, Dc, dofs, accumulate);
        return status(cudaGetLastError());
    }
    launch_pdl(k_channels, grid_of(pixels * C), 256, 0, (cudaStream_t)stream, (const bf16*)src, Sc, sofs, pixels, C, (bf16*)dst, Dc,
                                                                     dofs, accumulate);
    return status(cudaGetLastError());
}

int tpfnet_head(const void* x, long long pixels, int C, const float* Wt, const float* b, int Cout, float* out,
                void* stream)
{
    const int blocks = (int)((pixels + 255) / 256 < 152 * 8 ? (pixels + 255) / 256 : 152 * 8);
    const int smem = (C + 256) * Cout * (int)sizeof(float);
    if (pixels > 0 && Cout >= 1 && Cout <= 8 && smem <= 48 * 1024 && pieces(C, x)) {
        cudaStream_t s = (cudaStream_t)stream;
        auto run = [&](auto kern) { launch_pdl(kern, blocks, 256, smem, s, (const bf16*)x, pixels, C, Wt, b, out); };
        switch (Cout) {
        case 1: run(k_head8<1>); break;
        case 2: run(k_head8<2>); break;
        case 3: run(k_head8<3>); break;
        case 4: run(k_head8<4>); break;
        case 5: run(k_head8<5>); break;
        case 6: run(k_head8<6>); break;
        case 7: run(k_head8<7>); break;
        default: run(k_head8<8>); break;
        }
        return status(cudaGetLastError());
    }
    launch_pdl(k_head, grid_of(pixels * Cout), 256, 0, (cudaStream_t)stream, (const bf16*)x, pixels, C, Wt, b, Cout, out);
    return status(cudaGetLastError());
}

// blocks of k_head_back8, 0 where it does not take the shape
int tpfnet_head_parts(long long pixels, int C, int Cout)
{
    const int G = C / 8;
    if (pixels < 1 || Cout < 1 || Cout > 8 || C % 8 || G < 1 || G > 32 || (G & (G - 1))) return 0;
    const long long per = 8 * (32 / G);  // pixels per block and turn
    return (int)((pixels + per - 1) / per < 152 * 2 ? (pixels + per - 1) / per : 152 * 2);
}

static int head_back_any(const void* x, const float* dout, long long pixels, int C, const float* Wt, int Cout, void* dx,
                         float* dW, float* db, int relu, float* part, void* stream)
{
    const int smem = (C * Cout + Cout) * (int)sizeof(float);
    if (smem > 48 * 1024) return TPF_ERR_INVALID_ARG;
    const int blocks = pieces(C, x, dx) ? tpfnet_head_parts(pixels, C, Cout) : 0;
    if (part && !blocks) return TPF_ERR_INVALID_ARG;
    if (blocks) {
        cudaStream_t s = (cudaStream_t)stream;
        auto run = [&](auto kern) {
            launch_pdl(kern, blocks, 256, smem, s, (const bf16*)x, dout, pixels, C, Wt, (bf16*)dx, dW, db, relu, part);
        };
        switch (Cout) {
        case 1: run(k_head_back8<1>); break;
        case 2: run(k_head_back8<2>); break;
        case 3: run(k_head_back8<3>); break;
        case 4: run(k_head_back8<4>); break;
        case 5: run(k_head_back8<5>); break;
        case 6: run(k_head_back8<6>); break;
        case 7: run(k_head_back8<7>); break;
        default: run(k_head_back8<8>); break;
        }
        return status(cudaGetLastError());
    }
    launch_pdl(k_head_back, grid_of(pixels) < 304 ? grid_of(pixels) : 304, 256, smem, (cudaStream_t)stream, 
        (const bf16*)x, dout, pixels, C, Wt, Cout, (bf16*)dx, dW, db);
    const int rc = status(cudaGetLastError());
    return rc || !relu ? rc : tpfnet_relu_mask(dx, x, pixels * C, stream);
}

int tpfnet_head_back(const void* x, const float* dout, long long pixels, int C, const float* Wt, int Cout, void* dx,
                     float* dW, float* db, void* stream)
{
    return head_back_any(x, dout, pixels, C, Wt, Cout, dx, dW, db, 0, nullptr, stream);
}

int tpfnet_head_back_masked(const void* x, const float* dout, long long pixels, int C, const float* Wt, int Cout,
                            void* dx, float* dW, float* db, void* stream)
{
    return head_back_any(x, dout, pixels, C, Wt, Cout, dx, dW, db, 1, nullptr, stream);
}

int tpfnet_head_back_part(const void* x, const float* dout, long long pixels, int C, const float* Wt, int Cout,
                          void* dx, float* part, void* stream)
{
    if (!part) return TPF_ERR_INVALID_ARG;
    return head_back_any(x, dout, pixels, C, Wt, Cout, dx, nullptr, nullptr, 1, part, stream);
}

int tpfnet_unet_forward(const tpfnet_unet* u, const void* x, int N, int H, int W, float* out, void* stream)
{
    if (!u || !x || !out || N < 1 || H < 8 || W < 8 || H % 8 || W % 8) return TPF_ERR_INVALID_ARG;
    const int* c = u->ch;
    int rc = TPF_OK, k = 0;  // k: the 3x3 layer that is next
    auto conv = [&](const void* in, int lvl, int cin, int cout, void* y, int ldy) {
        if (rc == TPF_OK)
            rc = tpfnet_conv3x3_into(in, N, H >> lvl, W >> lvl, cin, u->weight[k], u->bias[k], cout, 1, y, ldy, stream);
        ++k;
    };
    // encoder: each level's output goes into its half of the concatenation (the bottleneck's
    // into a tensor of its own)
    const void* in = x;
    int cin = u->cin;
    for (int l = 0; l < 4; ++l) {
        const int ld = l < 3 ? c[l + 1] + c[l] : c[3];
        bf16* y = l < 3 ? (bf16*)u->cat[l] + c[l + 1] : (bf16*)u->deep;
        conv(in, l, cin, c[l], u->enc[l], c[l]);
        conv(u->enc[l], l, c[l], c[l], y, ld);
        if (l == 3) break;
        if (rc == TPF_OK) rc = tpfnet_pool_from(y, N, H >> l, W >> l, c[l], ld, u->pool[l], stream);
        in = u->pool[l];
        cin = c[l];
    }
    // decoder
    const void* up = u->deep;
    for (int l = 2; l >= 0; --l) {
        const int ct = c[l + 1] + c[l];
        if (rc == TPF_OK) rc = tpfnet_up_into(up, N, H >> l, W >> l, c[l + 1], u->cat[l], ct, 0, stream);
        conv(u->cat[l], l, ct, c[l], u->dec_a[l], c[l]);
        conv(u->dec_a[l], l, c[l], c[l], u->dec[l], c[l]);
        up = u->dec[l];
    }
    if (rc == TPF_OK) rc = tpfnet_head(u->dec[0], (long long)N * H * W, c[0], u->head_w, u->head_b, u->cout, out, stream);
    return rc;
}

int tpfnet_mse(const float* pred, const float* target, const float* wch, long long count, int C, float* grad,
               double* loss, void* stream)
{
    launch_pdl(k_mse, grid_of(count) < 304 ? grid_of(count) : 304, 256, 0, (cudaStream_t)stream, pred, target, wch, count, C, grad,
                                                                                          loss);
    return status(cudaGetLastError());
}

int tpfnet_adam(float* p, const float* g, float* m, float* v, long long count, float lr, float b1, float b2, float eps,
                int step, void* pb, void* stream)
{
    const float c1 = 1.f / (1.f - powf(b1, (float)step)), c2 = 1.f / (1.f - powf(b2, (float)step));
    launch_pdl(k_adam, grid_of(count), 256, 0, (cudaStream_t)stream, p, g, m, v, count, lr, b1, b2, eps, c1, c2, (bf16*)pb);
    return status(cudaGetLastError());
}

static int affine_of(int C, const float* scale, const float* shift, Affine* a)
{
    if (C < 1 || C > kMaxPackC) return TPF_ERR_INVALID_ARG;
    for (int c = 0; c < C; ++c) {
        a->scale[c] = scale ? scale[c] : 1.f;
        a->shift[c] = shift ? shift[c] : 0.f;
    }
    return TPF_OK;
}

int tpfnet_pack(const float* src, const float* base, long long plane, int C, long long pixels, const float* scale,
                const float* shift, void* dst, int Cd, int dst_bf16, void* stream)
{
    Affine a;
    if (!src || !dst || Cd < C || plane < pixels || affine_of(C, scale, shift, &a)) return TPF_ERR_INVALID_ARG;
    launch_pdl(k_pack, grid_of(pixels * C), 256, 0, (cudaStream_t)stream, src, base, plane, C, pixels, a, dst, Cd,
                                                                 dst_bf16 ? 1 : 0);
    return status(cudaGetLastError());
}

int tpfnet_unpack(const float* src, long long pixels, int C, const float* scale, const float* shift, const float* base,
                  float* dst, long long plane, void* stream)
{
    Affine a;
    if (!src || !dst || plane < pixels || affine_of(C, scale, shift, &a)) return TPF_ERR_INVALID_ARG;
    launch_pdl(k_unpack, grid_of(pixels * C), 256, 0, (cudaStream_t)stream, src, pixels, C, a, base, dst, plane);
    return status(cudaGetLastError());
}

int tpfnet_to_bf16(const float* x, long long count, void* y, void* stream)
{
    launch_pdl(k_to_bf16, grid_of(count), 256, 0, (cudaStream_t)stream, x, count, (bf16*)y);
    return status(cudaGetLastError());
}

}  // extern "C"
