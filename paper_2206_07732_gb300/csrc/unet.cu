// Learned warm start of the pressure solve: a 4-level convolutional U-Net in
// BF16 on the tensor cores with FP32 accumulation, its training (forward,
// backward, Adam) and its use as the initial guess of a tank's solve.
//
// Every convolution is an implicit GEMM on tcgen05 with the accumulator in
// tensor memory: rows are output pixels, columns output channels, the reduction
// runs over (tap, input channel).  Activations and gradients are chunk-planar
// BF16 tensors ([rows][C / 8][W][8]).  The forward convolutions (3x3, nearest
// upsampling + 3x3, 2x2 stride 2) and the 3x3 input gradients (the 3x3
// convolution of the output gradient with the flipped, transposed weights) run
// in the halo kernels (k_conv_rows where its weights fit and the image fills the GPU,
// else k_conv_halo; both persistent and warp-specialised): a stage holds one input row of one channel chunk,
// staged by bulk copy, and every horizontal tap reads it through a shifted descriptor;
// the weights arrive pre-packed by bulk copy.  The stride-2
// layer's input gradient is one GEMM for all four sub-pixels (k_down_dx).  Weight
// gradients reduce over pixels, split
// across CTAs (k_wgrad_tc); their partial tiles are summed in a fixed order, so
// results are reproducible bit for bit.  ReLU masks, biases,
// the skip gradient and the BF16 rounding are fused into the GEMM epilogues.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "internal.cuh"
#include "poisson_op.cuh"
#include "tank.cuh"

typedef __nv_bfloat16 bf16;
typedef __nv_bfloat162 bf162;

namespace wec {
namespace {

// ------------------------------------------------------------ architecture --
enum LayerKind { L_CONV3 = 0, L_UP3 = 1, L_DOWN2 = 2, L_HEAD = 3 };

struct LayerDef {
    int kind, ci, co, level;  // level of the output tensor (0 = full resolution)
};

constexpr int kNumLayers = 21;
constexpr int kInCh = 2;   // features per cell
constexpr int kInPad = 16; // channels of the stored BF16 input (two 16-byte chunks per pixel)
const LayerDef kLayers[kNumLayers] = {
    {L_CONV3, 2, 32, 0},    {L_CONV3, 32, 32, 0},                           // enc0a, enc0b
    {L_DOWN2, 32, 64, 1},   {L_CONV3, 64, 64, 1},   {L_CONV3, 64, 64, 1},   // down0, enc1a, enc1b
    {L_DOWN2, 64, 128, 2},  {L_CONV3, 128, 128, 2}, {L_CONV3, 128, 128, 2}, // down1, enc2a, enc2b
    {L_DOWN2, 128, 256, 3}, {L_CONV3, 256, 256, 3}, {L_CONV3, 256, 256, 3}, // down2, enc3a, enc3b
    {L_UP3, 256, 128, 2},   {L_CONV3, 256, 128, 2}, {L_CONV3, 128, 128, 2}, // up2, cat2, dec2
    {L_UP3, 128, 64, 1},    {L_CONV3, 128, 64, 1},  {L_CONV3, 64, 64, 1},   // up1, cat1, dec1
    {L_UP3, 64, 32, 0},     {L_CONV3, 64, 32, 0},   {L_CONV3, 32, 32, 0},   // up0, cat0, dec0
    {L_HEAD, 32, 1, 0}};                                                    // head
constexpr int kHead = 20;
inline int enc_a(int l) { return 3 * l; }
inline int enc_b(int l) { return 3 * l + 1; }
inline int down(int l) { return 3 * l + 2; }      // l = 0..2: level l -> l + 1
inline int up(int l) { return 11 + 3 * (2 - l); }  // l = 2..0: level l + 1 -> l
inline int cat(int l) { return up(l) + 1; }
inline int dec(int l) { return up(l) + 2; }

inline int taps(int kind) { return kind == L_DOWN2 ? 4 : (kind == L_HEAD ? 1 : 9); }
inline int cin_pad(int ci) { return ci == kInCh ? kInPad : ci; }
inline int round_up(int a, int b) { return (a + b - 1) / b * b; }
inline size_t round_up_z(size_t a, size_t b) { return (a + b - 1) / b * b; }

// ----------------------------------------------------------- tile constants --
constexpr int kBM = 128;     // GEMM rows (pixels, or weight rows in k_wgrad_tc) per CTA

enum EpiKind { E_FWD = 0, E_DX = 1, E_DOWNDX = 2, E_POOL = 3 };

// The input tensors of a layer and its output grid: channel c < c0 comes from in0,
// the rest from in1 (concatenation).
struct Gat {
    const bf16 *in0, *in1;
    int c0, c1;
    int N, H, W;       // output grid
    int Hi, Wi;        // grid of the input tensors
    int K;             // taps * (c0 + c1)
};

// Fused epilogue.  E_FWD: out0 = bf16(relu(acc + bias)).  E_DX: input gradient;
// columns < nsplit: out0 = bf16(acc * (mask0 > 0)), the rest: out1 = bf16(acc).
// E_DOWNDX: the stride-2 layer's input gradient, column z ld0 + c
// channel c at sub-pixel z of each half-grid pixel's 2x2 block:
// out0 = bf16((acc + add) * (mask0 > 0)).
// E_POOL (row-block tiles): an upsampling layer's input gradient on the half grid,
// out0 = bf16(sum of acc over the 2x2 block * (mask0 > 0)).
struct Epi {
    int kind;
    const float *bias;
    bf16 *out0;
    const bf16 *mask0;
    int ld0;
    bf16 *out1;
    int ld1, nsplit;
    const bf16 *add;
};

// ------------------------------------------------------------- PTX helpers --
__device__ __forceinline__ unsigned smem_u32(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

// 16-byte global -> shared copy; src_bytes = 0 fills the destination with zeros.
__device__ __forceinline__ void cp16(void *dst, const void *src, int src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// ---------------------------------------------------------- tensor layout --
// Activations and their gradients are chunk-planar BF16 tensors
// [rows][C / 8][W][8] (row = n H + y): the 8 channels [8q, 8q + 8) of a whole
// image row are contiguous, so a row segment of one channel chunk is one
// contiguous block (what the convolutions stage with bulk copies).
__device__ __forceinline__ size_t cofs(size_t row, int x, int c, int C, int W)
{
    return ((row * (size_t)(C >> 3) + (size_t)(c >> 3)) * (size_t)W + (size_t)x) * 8 + (size_t)(c & 7);
}

// ---------------------------------------------------------------- tcgen05 --
// Tensor-core tiles: one CTA owns 128 pixels x BN channels whose FP32 accumulator
// lives in tensor memory; operands in shared memory in the no-swizzle K-major
// core-matrix layout (8 rows x 16 bytes per core matrix); one thread issues
// tcgen05.mma (M = 128, N = BN, K = 16, BF16 x BF16 -> FP32).  Every wait is bounded:
// on expiry the kernel raises *err, drains its copies, frees its tensor memory and
// returns.
constexpr int kTcK = 64;               // reduction elements per stage
constexpr int kTcThreads = 160;        // warps 0-3: producers / epilogue; warp 4: MMA
constexpr long long kWaitLimit = 1LL << 22;  // polls; far above any legitimate wait here

__device__ __forceinline__ void mbar_init(unsigned a, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(a), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned a)
{
    asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(a) : "memory");
}
// Wait for the phase with the given parity to complete; false after kWaitLimit polls.
__device__ __forceinline__ bool mbar_wait(unsigned a, unsigned parity)
{
    for (long long it = 0; it < kWaitLimit; ++it) {
        unsigned ok;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ uint64_t umma_desc(unsigned saddr)
{
    // start address, K-direction core-matrix stride 128 B, 8-row-group stride
    // 1024 B (both >> 4), descriptor version 1 (bit 46), no swizzle
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           (1ull << 46);
}

template <int BN>
__host__ __device__ constexpr unsigned umma_idesc()
{
    // kind::f16: D F32 (bits 4-5 = 1), A BF16 (bits 7-9 = 1), B BF16 (bits 10-12 = 1),
    // both K-major, N >> 3 at bit 17, M >> 4 at bit 24
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(BN >> 3) << 17) | ((unsigned)(kBM >> 4) << 24);
}

// Epilogue of a tensor-core tile: the calling warp (warp = TMEM lane quarter)
// reads its 32 tile rows; tile row r is pixel m0 + r ps, valid below M.  The
// BF16 results are stored an 8-channel chunk of a row at a time, as one 16-byte
// vector: the warp's 32 rows are consecutive pixels of one image row, so in the
// chunk-planar layout a warp's store of one chunk is contiguous.  go is warp-uniform (tcgen05.ld is warp-collective).
template <int BN>
__device__ __forceinline__ void tc_epilogue(const Epi &e, const Gat &g, unsigned tmem, int m0, int n0, int M,
                                            int warp, int lane, bool go, int ps = 1)
{
    if (!go) return;
    const int row = warp * 32 + lane, p = m0 + row * ps;
    const size_t prow = (size_t)(p / g.W);
    const int px = p - (int)prow * g.W;
#pragma unroll 1
    for (int c0 = 0; c0 < BN; c0 += 16) {
        unsigned v[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
            "[%16];\n"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
              "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
            : "r"(tmem + ((unsigned)(warp * 32) << 16) + (unsigned)c0));
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        if (p >= M) continue;
        const int col = n0 + c0;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {  // two 8-channel chunks
            const int cc = col + 8 * hh;
            float f[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) f[q] = __uint_as_float(v[8 * hh + q]);
            bf16 *dst;
            if (e.kind == E_FWD) {
#pragma unroll
                for (int q = 0; q < 8; ++q) f[q] = fmaxf(f[q] + e.bias[cc + q], 0.0f);
                dst = e.out0 + cofs(prow, px, cc, e.ld0, g.W);
            } else if (e.kind == E_DOWNDX) {
                const int z = cc / e.ld0;
                const size_t o = cofs(2 * prow + (z >> 1), 2 * px + (z & 1), cc - z * e.ld0, e.ld0, 2 * g.W);
                const uint4 mv = *reinterpret_cast<const uint4 *>(e.mask0 + o);
                const uint4 av = *reinterpret_cast<const uint4 *>(e.add + o);
                const bf16 *m = reinterpret_cast<const bf16 *>(&mv), *a = reinterpret_cast<const bf16 *>(&av);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    f[q] = __bfloat162float(m[q]) > 0.0f ? f[q] + __bfloat162float(a[q]) : 0.0f;
                dst = e.out0 + o;
            } else if (cc < e.nsplit) {
                const uint4 mv = *reinterpret_cast<const uint4 *>(e.mask0 + cofs(prow, px, cc, e.ld0, g.W));
                const bf16 *m = reinterpret_cast<const bf16 *>(&mv);
#pragma unroll
                for (int q = 0; q < 8; ++q) f[q] = __bfloat162float(m[q]) > 0.0f ? f[q] : 0.0f;
                dst = e.out0 + cofs(prow, px, cc, e.ld0, g.W);
            } else {
                dst = e.out1 + cofs(prow, px, cc - e.nsplit, e.ld1, g.W);
            }
            __align__(16) bf162 hv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) hv[q] = __floats2bfloat162_rn(f[2 * q], f[2 * q + 1]);
            *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(hv);
        }
    }
}

// Input gradient of a stride-2 layer: every half-grid pixel's K = 2C output gradients
// times the 4C x K matrix B (row z C + c: sub-pixel z of the pixel's 2x2 block) gives
// the C input gradients of its four sub-pixels (E_DOWNDX).  The four sub-pixels are
// columns of one product, so a pixel is staged once for all of them, and K <= 256
// fits in shared memory whole.  Bound by the epilogue's traffic (reads the mask and
// the skip gradient, writes the result: 6 bytes per value); four images of
// 256 x 512, C = 32: 38 us for 118 MB (105 with a launch plane per sub-pixel and
// 4-byte accesses).
template <int BN>
__global__ void __launch_bounds__(kTcThreads) k_down_dx(const bf16 *__restrict__ G, int K, int M, int W,
                                                        const bf16 *__restrict__ B, Epi e, int *err)
{
    pdl_entry();
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int KT = K / kTcK;
    constexpr int kA = kBM * kTcK * 2, kStage = kA + BN * kTcK * 2;
    unsigned char *bar_base = smem + KT * kStage;
    const unsigned full = smem_u32(bar_base), done = full + 8;
    unsigned *tmem_slot = reinterpret_cast<unsigned *>(bar_base + 16);
    const int m0 = blockIdx.x * kBM, n0 = blockIdx.y * BN;

    if (tid == 0) {
        mbar_init(full, 128);
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                     "r"(BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned tmem = *tmem_slot;
    bool ok = true;

    if (warp < 4) {
        // ---- staging: thread t takes tile pixel t (a chunk is one contiguous run of
        // pixels), and of the weights 8 rows x 16 bytes per 8 threads ----
        const int p = m0 + tid;
        const bool v = p < M;
        const size_t row = v ? (size_t)(p / W) : 0;
        const bf16 *src = G + cofs(row, v ? p - (int)row * W : 0, 0, K, W);
        for (int kt = 0; kt < KT; ++kt) {
            unsigned char *As = smem + kt * kStage, *Bs = As + kA;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                cp16(As + ((tid >> 3) * 8 + q) * 128 + (tid & 7) * 16, src + (size_t)(8 * kt + q) * W * 8, v ? 16 : 0);
#pragma unroll
            for (int rr = 0; rr < BN / 16; ++rr) {
                const int c = tid + 128 * rr, nn = c >> 3, q = c & 7;
                cp16(Bs + ((nn >> 3) * 8 + q) * 128 + (nn & 7) * 16, B + (size_t)(n0 + nn) * K + kt * kTcK + q * 8, 16);
            }
        }
        cp_commit();
        cp_wait<0>();
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        mbar_arrive(full);
    } else if (lane == 0) {
        // ---- MMA issuer ----
        constexpr unsigned idesc = umma_idesc<BN>();
        ok = mbar_wait(full, 0);
        if (ok) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            for (int kt = 0; kt < KT; ++kt) {
                const unsigned a0 = smem_u32(smem + kt * kStage), b0 = a0 + kA;
#pragma unroll
                for (int kk = 0; kk < kTcK / 16; ++kk) {
                    const uint64_t ad = umma_desc(a0 + kk * 256), bd = umma_desc(b0 + kk * 256);
                    const unsigned acc = (kt > 0 || kk > 0) ? 1u : 0u;
                    asm volatile(
                        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                        "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                        : "memory");
                }
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(done)
                         : "memory");
            if (!mbar_wait(done, 0)) ok = false;  // no MMA in flight past this point
        }
    }

    if (warp < 4) {
        // ---- epilogue: TMEM lanes 32 warp .. +31 are this warp's rows ----
        ok = mbar_wait(done, 0);
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        Gat g{};  // the epilogue needs only the row length
        g.W = W;
        tc_epilogue<BN>(e, g, tmem, m0, n0, M, warp, lane, __all_sync(0xffffffffu, ok));
    }
    if (!ok) atomicExch(err, 1);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 4) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(BN) : "memory");
    }
}

// ------------------------------------------------ tcgen05 halo convolution --
// A convolution whose CTA tile is 128 consecutive pixels of one output image
// row (n, i, x0 .. x0 + 127) by BN output channels, the accumulator in tensor
// memory.  The reduction runs in stages of CS input channels x one vertical
// tap: a stage holds the input row of that tap once, K-chunk by K-chunk (16
// bytes per pixel slot, the next chunk LBO bytes on), and the horizontal taps
// read it through descriptors whose start addresses differ by one slot (8-row
// groups 128 B apart).  Modes:
//   3x3 (stride 1, zero border): slots x0 - 1 .. x0 + 134 of input row i + ta - 1;
//   up: the same over the nearest-upsampled input (slot x reads pixel x / 2 of
//       row (i + ta - 1) / 2 of the half-resolution tensor);
//   down (2x2, stride 2): input row 2 i + ta, even pixels 2 (x0 + r) in slots
//       0 .. 127 and odd pixels in slots 128 .. 255, one array per horizontal tap.
// The stage's weights for all its horizontal taps arrive in one bulk copy,
// pre-packed in core-matrix order (k_pack_halo).
enum HaloMode { H_CONV3 = 0, H_UP3 = 1, H_DOWN2 = 2 };

struct Halo {
    const bf16 *in0, *in1;  // channels [0, c0) from in0, [c0, c0 + c1) from in1 (concatenation)
    int c0, c1;
    int N, H, W, xtiles;    // output image grid; 128-pixel tiles per image row
    int Hi, Wi;             // input tensor grid
    int mode, nst;          // HaloMode; stages: (c0 + c1) / CS x vertical taps
    int ncols;              // output channels (column tiles of BN)
};

template <int BN, int CS, bool DOWN>
struct HaloSmem {
    static constexpr int kSlots = DOWN ? 256 : 136;       // pixel slots per K-chunk (a multiple of 8)
    static constexpr int kLBO = (kSlots + 1) * 16;         // one padding slot: chunks fall in different banks
    static constexpr int kTH = DOWN ? 2 : 3;               // horizontal taps per stage
    static constexpr int kA = (CS / 8) * kLBO;
    static constexpr int kB = kTH * BN * CS * 2;
    static constexpr int kStage = kA + kB;
    static constexpr int kFit = (227 * 1024 - 512) / kStage;
    static constexpr int kStages = kFit >= 4 ? 4 : (kFit >= 2 ? kFit : 2);
    static constexpr int kBytes = kStages * kStage + 512;  // + barriers and the TMEM address
};

__device__ __forceinline__ uint64_t umma_desc_s(unsigned saddr, unsigned lbo, unsigned sbo)
{
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

__device__ __forceinline__ void mbar_expect_tx(unsigned a, unsigned bytes)
{
    asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(a), "r"(bytes)
                 : "memory");
}

// Contiguous global -> shared bulk copy completing on an mbarrier (tx bytes).
__device__ __forceinline__ void bulk_g2s(unsigned dst, const void *src, unsigned bytes, unsigned mbar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(mbar)
        : "memory");
}

// Persistent and warp-specialised: a CTA walks the tiles blockIdx.x,
// blockIdx.x + gridDim.x, ...; warps 0-3 stage operands through the stage ring
// (continuing across tiles), one thread of warp 8 issues the MMAs into one of
// two tensor-memory accumulator buffers, and warps 4-7 drain the other buffer
// (epilogue of tile t overlapping the loads and MMAs of tile t + 1).
constexpr int kPThreads = 288;  // warps 0-3 producers, 4-7 epilogue, 8 MMA issue

template <int BN, int CS, bool DOWN>
__global__ void __launch_bounds__(kPThreads, 1) k_conv_halo(Halo h, const bf16 *__restrict__ Bp, Epi e, int *err)
{
    pdl_entry();
    extern __shared__ __align__(1024) unsigned char smem[];
    using S = HaloSmem<BN, CS, DOWN>;
    constexpr int TH = S::kTH, TV = DOWN ? 2 : 3, NS = S::kStages, CH = CS / 8;
    // cp.async stages a producer keeps in flight before signalling: one stage of
    // slack between the MMA being waited for and the one being fed
    constexpr int LAG = NS >= 3 ? NS - 2 : 0;
    constexpr int kCols = DOWN ? 2 * BN : 4 * BN;  // two tile buffers (x two parities for the up mode)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char *bar_base = smem + NS * S::kStage;
    const unsigned full0 = smem_u32(bar_base), empty0 = full0 + 8 * NS;
    const unsigned accf0 = empty0 + 8 * NS, acce0 = accf0 + 16;  // accumulator full[2] / empty[2]
    unsigned *tmem_slot = reinterpret_cast<unsigned *>(bar_base + 8 * (2 * NS + 4));
    const bool up = !DOWN && h.mode == H_UP3;
    const int nacc = up ? 2 : 1;
    const int ntn = h.ncols / BN, ntiles = h.N * h.H * h.xtiles * ntn, KT = h.nst;

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(full0 + 8 * s, DOWN ? 129 : 5);  // producers (or their warps) + the bulk copies' expect_tx arrival
            mbar_init(empty0 + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(accf0 + 8 * b, 1);
            mbar_init(acce0 + 8 * b, 128);
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned tmem = *tmem_slot;
    bool ok = true;

    // tile t: column tile nt (fastest), then 128-column tile xt of image row rowid
    auto decode = [&](int t, int &nt, int &rowid, int &x0) {
        nt = t % ntn;
        const int r = t / ntn;
        x0 = (r % h.xtiles) * kBM;
        rowid = r / h.xtiles;
    };

    if (warp < 4) {
        // ---- producers ----
        long long g = 0, sig = 0;  // stages staged / signalled by this thread
        // Stages whose slots outside the row are zero for the column tile zx.  (One thread
        // issuing all of a stage's copies, the zero slots stored again for every stage and
        // 128 arrivals took 3 % of the network's time.)
        unsigned zeroed = 0;
        int zx = -1;
        for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
            int nt, rowid, x0;
            decode(t, nt, rowid, x0);
            const int i = rowid % h.H, n = rowid / h.H;
            const bf16 *Bt = Bp + (size_t)nt * h.nst * TH * BN * CS;
            for (int kt = 0; kt < KT && ok; ++kt, ++g) {
                const int s = (int)(g % NS);
                if (g >= NS)  // (the warp goes on or stops as one)
                    ok = __all_sync(0xffffffffu, mbar_wait(empty0 + 8 * s, (unsigned)(((g / NS) - 1) & 1)));
                if (!ok) break;
                unsigned char *As = smem + s * S::kStage, *Bs = As + S::kA;
                const int cc = kt / TV, ta = kt - TV * cc, cb = cc * CS;
                int y = DOWN ? 2 * i + ta : i + ta - 1;  // input row (output grid for the up mode)
                const bool row_ok = y >= 0 && y < (DOWN ? h.Hi : h.H);
                if (up) y >>= 1;
                const bf16 *tbase;
                int tC, coff;
                if (cb < h.c0) {
                    tbase = h.in0;
                    tC = h.c0;
                    coff = cb;
                } else {
                    tbase = h.in1;
                    tC = h.c1;
                    coff = cb - h.c0;
                }
                const size_t trow = (size_t)n * h.Hi + (row_ok ? y : 0);
                if (!DOWN) {
                    // slots x0 - 1 + sl of the input row: the columns inside [0, Wi)
                    // arrive by one bulk copy per channel chunk (a contiguous row
                    // segment of its plane), the others are zero
                    const int xs = max(x0 - 1, 0), xe = min(x0 - 1 + S::kSlots, h.Wi), s0 = xs - (x0 - 1);
                    if (tid == 0) {
                        mbar_expect_tx(full0 + 8 * s, S::kB + (row_ok ? (unsigned)(xe - xs) * 16u * CH : 0u));
                        bulk_g2s(smem_u32(Bs), Bt + (size_t)kt * TH * BN * CS, S::kB, full0 + 8 * s);
                    }
                    if (row_ok && tid >= 32 && tid < 32 + CH) {
                        const int q = tid - 32;
                        bulk_g2s(smem_u32(As + q * S::kLBO + s0 * 16), tbase + cofs(trow, xs, coff + 8 * q, tC, h.Wi),
                                 (unsigned)(xe - xs) * 16u, full0 + 8 * s);
                    }
                    if (x0 != zx) {
                        zx = x0;
                        zeroed = 0;
                    }
                    if (!row_ok || !(zeroed >> s & 1)) {
                        for (int idx = tid; idx < S::kSlots * CH; idx += 128) {
                            const int q = idx % CH, sl = idx / CH;
                            if (!(row_ok && sl >= s0 && sl < s0 + (xe - xs)))
                                *reinterpret_cast<uint4 *>(As + q * S::kLBO + sl * 16) = make_uint4(0u, 0u, 0u, 0u);
                        }
                        zeroed |= 1u << s;
                        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                    }
                    // only bulk copies (tracked by the byte count) and the warp's zero
                    // stores: signal at once
                    __syncwarp();
                    if (lane == 0) mbar_arrive(full0 + 8 * s);
                    sig = g + 1;
                } else {
                    if (tid == 0) {
                        mbar_expect_tx(full0 + 8 * s, S::kB);
                        bulk_g2s(smem_u32(Bs), Bt + (size_t)kt * TH * BN * CS, S::kB, full0 + 8 * s);
                    }
                    for (int idx = tid; idx < S::kSlots * CH; idx += 128) {
                        const int q = idx % CH, sl = idx / CH;
                        const int r = sl & (kBM - 1), x = 2 * (x0 + r) + (sl >> 7);  // even / odd input pixels
                        const bool v = row_ok && x0 + r < h.W;
                        cp16(As + q * S::kLBO + sl * 16, v ? tbase + cofs(trow, x, coff + 8 * q, tC, h.Wi) : h.in0,
                             v ? 16 : 0);
                    }
                    cp_commit();
                    if (g >= LAG) {
                        cp_wait<LAG>();
                        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                        mbar_arrive(full0 + 8 * (int)((g - LAG) % NS));
                        sig = g - LAG + 1;
                    }
                }
            }
        }
        cp_wait<0>();
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        if (ok)
            for (; sig < g; ++sig) mbar_arrive(full0 + 8 * (int)(sig % NS));
    } else if (warp == 8) {
        if (lane == 0) {
            // ---- MMA issue: per stage TH taps x CS / 16 K-steps (x 2 parities for up) ----
            constexpr unsigned idesc = umma_idesc<BN>();
            long long g = 0;
            int lt = 0;
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++lt) {
                const int buf = lt & 1;
                if (lt >= 2) ok = mbar_wait(acce0 + 8 * buf, (unsigned)(((lt >> 1) - 1) & 1));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const unsigned acc0 = tmem + (unsigned)(buf * nacc * BN);
                for (int kt = 0; kt < KT && ok; ++kt, ++g) {
                    const int s = (int)(g % NS);
                    ok = mbar_wait(full0 + 8 * s, (unsigned)((g / NS) & 1));
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const unsigned a0 = smem_u32(smem + s * S::kStage), b0 = a0 + S::kA;
                    for (int b = 0; b < nacc; ++b)
#pragma unroll
                        for (int tb = 0; tb < TH; ++tb) {
                            // slot offset of the tap: tb (3x3), the even / odd input array
                            // (down), (b + tb + 1) / 2 (up: output column 2 (x0 + r) + b
                            // reads input column x0 + r + that - 1)
                            const int so = DOWN ? tb * kBM : (up ? (b + tb + 1) >> 1 : tb);
#pragma unroll
                            for (int kk = 0; kk < CS / 16; ++kk) {
                                const uint64_t ad = umma_desc_s(a0 + 2 * kk * S::kLBO + so * 16, S::kLBO, 128);
                                const uint64_t bd =
                                    umma_desc_s(b0 + tb * (BN * CS * 2) + 2 * kk * 128, 128, CH * 128);
                                const unsigned acc = (kt > 0 || tb > 0 || kk > 0) ? 1u : 0u;
                                asm volatile(
                                    "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                                        acc0 + (unsigned)(b * BN)),
                                    "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                                    : "memory");
                            }
                        }
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                                     empty0 + 8 * s)
                                 : "memory");
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                                 accf0 + 8 * buf)
                             : "memory");
            }
            // no MMA in flight past this point (the last tile's commit completed)
            if (lt > 0 && !mbar_wait(accf0 + 8 * ((lt - 1) & 1), (unsigned)(((lt - 1) >> 1) & 1))) ok = false;
        }
    } else {
        // ---- epilogue (warps 4-7: TMEM lanes 32 (warp - 4) .. +31) ----
        const int ew = warp - 4;
        Gat g{};  // the epilogue needs only the output grid
        g.N = h.N;
        g.H = h.H;
        g.W = h.W;
        int lt = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++lt) {
            const int buf = lt & 1;
            const bool ok2 = ok && mbar_wait(accf0 + 8 * buf, (unsigned)((lt >> 1) & 1));
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const bool go = __all_sync(0xffffffffu, ok2);
            int nt, rowid, x0;
            decode(t, nt, rowid, x0);
            const int ps = up ? 2 : 1, nvalid = min(kBM, (up ? h.Wi : h.W) - x0);
            for (int b = 0; b < nacc; ++b) {
                const int m0 = rowid * h.W + ps * x0 + b;
                tc_epilogue<BN>(e, g, tmem + (unsigned)((buf * nacc + b) * BN), m0, nt * BN, m0 + ps * nvalid, ew,
                                lane, go, ps);
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            mbar_arrive(acce0 + 8 * buf);
            if (!go) {
                ok = false;
                break;
            }
        }
    }
    if (!ok) atomicExch(err, 1);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 8) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kCols) : "memory");
    }
}

// E_POOL epilogue of two image rows (accumulators t0 and t1 = rows 2i, 2i + 1): the
// sum over each 2x2 block, rounded once, masked; lanes 2j and 2j + 1 hold a block's
// columns and store one of its two 8-channel chunks each.  m: first pixel of the tile
// in the half grid, nvalid: its pixels there, W2: the half grid's row length.
template <int BN>
__device__ __forceinline__ void pool_epilogue(const Epi &e, unsigned t0, unsigned t1, int m, int nvalid, int W2, int n0,
                                              int warp, int lane)
{
    const int row = (warp * 32 + lane) >> 1, p = m + row;
    const size_t prow = (size_t)(p / W2);
    const int px = p - (int)prow * W2;
#pragma unroll 1
    for (int c0 = 0; c0 < BN; c0 += 16) {
        float f[8];
#pragma unroll
        for (int i = 0; i < 2; ++i) {  // the step's two chunks; a lane keeps the one that it stores
            float v[2][8];
#pragma unroll
            for (int a = 0; a < 2; ++a)
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                             : "=f"(v[a][0]), "=f"(v[a][1]), "=f"(v[a][2]), "=f"(v[a][3]), "=f"(v[a][4]), "=f"(v[a][5]),
                               "=f"(v[a][6]), "=f"(v[a][7])
                             : "r"((a ? t1 : t0) + ((unsigned)(warp * 32) << 16) + (unsigned)(c0 + 8 * i)));
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float s = (v[0][q] + __shfl_xor_sync(0xffffffffu, v[0][q], 1)) +
                                (v[1][q] + __shfl_xor_sync(0xffffffffu, v[1][q], 1));
                if ((lane & 1) == i) f[q] = s;
            }
        }
        if (row >= nvalid) continue;
        const size_t o = cofs(prow, px, n0 + c0 + 8 * (lane & 1), e.ld0, W2);
        const uint4 mv = *reinterpret_cast<const uint4 *>(e.mask0 + o);
        const bf16 *mk = reinterpret_cast<const bf16 *>(&mv);
#pragma unroll
        for (int q = 0; q < 8; ++q) f[q] = __bfloat162float(mk[q]) > 0.0f ? f[q] : 0.0f;
        __align__(16) bf162 hv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) hv[q] = __floats2bfloat162_rn(f[2 * q], f[2 * q + 1]);
        *reinterpret_cast<uint4 *>(e.out0 + o) = *reinterpret_cast<const uint4 *>(hv);
    }
}

// Stride-1 and upsampling convolutions of the finer levels (rows_bn): a CTA's tile is
// 128 pixels of R consecutive image rows, with an accumulator per row (two for the
// column parities of the up mode), and the weights of all taps stay in shared
// memory.  An input row is staged once and feeds the (up to three) output rows
// around it, where the one-row tiles (k_conv_halo) stage it once per vertical tap
// and fetch the weights with every stage -- at 64 channels more bytes than the
// pixels.  The products of an output are added in the same order (channels, vertical
// tap, horizontal tap), so the values are the same.  Persistent and
// warp-specialised: producers (warps 0-3), MMA (warp 8), epilogue (warps 4-7), which
// takes a row as soon as its last tap is in; a row's accumulator goes back to the
// MMA by itself.  80 registers, so that two CTAs fit on an SM (with 100 the 32 -> 32
// channel layer took 24 us, with 78 13).  Bound by the latency of the staged rows and
// the epilogue's stores: 32 -> 32 channels at 256 x 1024 13 us (one-row tiles: 21) for
// 34 MB, 64 -> 32 22 us (34); four images of 256 x 512, input gradients 32 -> 64 53 us
// (87) and, pooled, 32 -> 64 31 us (116 + 55 with the pooling pass).
template <int BN, int CS, bool UP, int NS>
struct RowsCfg {
    static constexpr int kLBO = 137 * 16;             // 136 pixel slots per chunk and one of padding
    static constexpr int kStage = (CS / 8) * kLBO;    // an input row
    static constexpr int kAcc = UP ? 2 : 1;           // accumulators per output row
    static constexpr int kRows = 256 / (BN * kAcc);   // output rows per tile, at most (256 accumulator columns)
    static int bytes(int cin) { return (9 * cin * BN * 2 + 1023) / 1024 * 1024 + NS * kStage + 256; }
};

template <int BN, int CS, bool UP, int NS>
__global__ void __maxnreg__(80)
    k_conv_rows(Halo h, int R, const bf16 *__restrict__ Bp, Epi e, int *err)
{
    pdl_entry();
    extern __shared__ __align__(1024) unsigned char smem[];
    using S = RowsCfg<BN, CS, UP, NS>;
    constexpr int CH = CS / 8, RM = S::kRows, NA = S::kAcc;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wbytes = h.nst * 3 * BN * CS * 2, ncc = h.nst / 3;
    unsigned char *const ring = smem + (wbytes + 1023) / 1024 * 1024;
    unsigned char *const bars = ring + NS * S::kStage;
    const unsigned full0 = smem_u32(bars), empty0 = full0 + 8 * NS, accf0 = empty0 + 8 * NS, acce0 = accf0 + 8 * RM,
                   wfull = acce0 + 8 * RM;
    unsigned *const tmem_slot = reinterpret_cast<unsigned *>(bars + 8 * (2 * NS + 2 * RM + 1));
    const int rblocks = (h.H + R - 1) / R, ntiles = h.N * rblocks * h.xtiles, nt = blockIdx.y;

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(full0 + 8 * s, 5);  // the producers' warps + the bulk copies' expect_tx arrival
            mbar_init(empty0 + 8 * s, 1);
        }
        for (int q = 0; q < RM; ++q) {  // per output row: accumulator full, and read
            mbar_init(accf0 + 8 * q, 1);
            mbar_init(acce0 + 8 * q, 128);
        }
        mbar_init(wfull, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                     "r"(256)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned tmem = *tmem_slot;
    bool ok = true;

    // tile t: column tile xt (fastest) of row block rb of image n
    auto decode = [&](int t, int &n, int &i0, int &rv, int &x0) {
        const int r = t / h.xtiles;
        x0 = (t - r * h.xtiles) * kBM;
        n = r / rblocks;
        i0 = (r - n * rblocks) * R;
        rv = min(R, h.H - i0);
    };

    // input rows of a tile (the up mode reads the half grid)
    auto first_row = [&](int i0) { return UP ? (i0 >> 1) - 1 : i0 - 1; };
    auto row_count = [&](int rv) { return UP ? (rv >> 1) + 2 : rv + 2; };

    if (warp < 4) {
        // ---- producers
        if (tid == 0) {
            mbar_expect_tx(wfull, (unsigned)wbytes);
            bulk_g2s(smem_u32(smem), Bp + (size_t)nt * h.nst * 3 * BN * CS, (unsigned)wbytes, wfull);
        }
        unsigned zeroed = 0;  // stages whose slots outside the row are zero for the column tile zx
        int zx = -1;
        int g = 0;
        for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
            int n, i0, rv, x0;
            decode(t, n, i0, rv, x0);
            if (x0 != zx) {
                zx = x0;
                zeroed = 0;
            }
            const int xs = max(x0 - 1, 0), xe = min(x0 - 1 + 136, h.Wi), s0 = xs - (x0 - 1);
            for (int cc = 0; cc < ncc && ok; ++cc) {
                const int cb = cc * CS;
                const bf16 *tbase = cb < h.c0 ? h.in0 : h.in1;
                const int tC = cb < h.c0 ? h.c0 : h.c1, coff = cb < h.c0 ? cb : cb - h.c0;
                for (int q = 0; q < row_count(rv); ++q, ++g) {
                    const int s = g % NS, y = first_row(i0) + q;
                    if (g >= NS)  // (the warp goes on or stops as one)
                        ok = __all_sync(0xffffffffu, mbar_wait(empty0 + 8 * s, (unsigned)((g / NS - 1) & 1)));
                    if (!ok) break;
                    unsigned char *const As = ring + s * S::kStage;
                    const bool row_ok = y >= 0 && y < h.Hi;
                    if (tid == 0) mbar_expect_tx(full0 + 8 * s, row_ok ? (unsigned)(xe - xs) * 16u * CH : 0u);
                    if (row_ok && tid >= 32 && tid < 32 + CH) {
                        const int c = tid - 32;
                        bulk_g2s(smem_u32(As + c * S::kLBO + s0 * 16),
                                 tbase + cofs((size_t)n * h.Hi + y, xs, coff + 8 * c, tC, h.Wi), (unsigned)(xe - xs) * 16u,
                                 full0 + 8 * s);
                    }
                    if (!row_ok || !(zeroed >> s & 1)) {
                        for (int idx = tid; idx < 136 * CH; idx += 128) {
                            const int c = idx % CH, sl = idx / CH;
                            if (!(row_ok && sl >= s0 && sl < s0 + (xe - xs)))
                                *reinterpret_cast<uint4 *>(As + c * S::kLBO + sl * 16) = make_uint4(0u, 0u, 0u, 0u);
                        }
                        zeroed |= 1u << s;
                        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(full0 + 8 * s);
                }
            }
        }
        if (!ok)  // drain what is in flight
            for (int q = max(0, g - NS); q < g; ++q) mbar_wait(full0 + 8 * (q % NS), (unsigned)((q / NS) & 1));
    } else if (warp == 8) {
        if (lane == 0) {
            // ---- MMA issue
            constexpr unsigned idesc = umma_idesc<BN>();
            ok = mbar_wait(wfull, 0u);
            const unsigned w0 = smem_u32(smem);
            unsigned used = 0;  // per output row: parity of the uses of its accumulator
            int g = 0;
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
                int n, i0, rv, x0;
                decode(t, n, i0, rv, x0);
                for (int cc = 0; cc < ncc && ok; ++cc)
                    for (int q = 0; q < row_count(rv) && ok; ++q, ++g) {
                        const int s = g % NS; // input row first_row + q
                        ok = mbar_wait(full0 + 8 * s, (unsigned)((g / NS) & 1));
                        if (!ok) break;
                        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        const unsigned a0 = smem_u32(ring + s * S::kStage);
                        // output row r reads it with vertical tap q - r; in the up mode with those of
                        // r + ta = 2q - 1 and 2q
                        for (int r = max(0, (UP ? 2 * q : q) - (UP ? 3 : 2)); r < min(rv, (UP ? 2 * q : q) + 1) && ok; ++r) {
                            const int ta0 = UP ? max(2 * q - 1 - r, 0) : q - r, ta1 = UP ? min(2 * q - r, 2) : q - r;
                            for (int ta = ta0; ta <= ta1; ++ta) {
                                if (cc == 0 && ta == 0) {  // the last tile's row r has been read
                                    ok = mbar_wait(acce0 + 8 * r, (~used >> r) & 1u);
                                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                                    if (!ok) break;
                                }
                                const unsigned b0 = w0 + (unsigned)((cc * 3 + ta) * 3) * (BN * CS * 2);
#pragma unroll
                                for (int b = 0; b < NA; ++b)
#pragma unroll
                                    for (int tb = 0; tb < 3; ++tb) {
                                        const int so = UP ? (b + tb + 1) >> 1 : tb;
#pragma unroll
                                        for (int kk = 0; kk < CS / 16; ++kk) {
                                            const uint64_t ad = umma_desc_s(a0 + 2 * kk * S::kLBO + so * 16, S::kLBO, 128);
                                            const uint64_t bd =
                                                umma_desc_s(b0 + tb * (BN * CS * 2) + 2 * kk * 128, 128, CH * 128);
                                            const unsigned acc = (cc > 0 || ta > 0 || tb > 0 || kk > 0) ? 1u : 0u;
                                            asm volatile(
                                                "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                                                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                                                    tmem + (unsigned)((r * NA + b) * BN)),
                                                "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                                                : "memory");
                                        }
                                    }
                            }
                        }
                        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                                         empty0 + 8 * s)
                                     : "memory");
                        if (cc == ncc - 1)  // rows that took their last tap here
                            for (int r = max(0, UP ? 2 * q - 3 : q - 2); r < min(rv, UP ? 2 * q - 1 : q - 1); ++r) {
                                used ^= 1u << r;
                                asm volatile(
                                    "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                                        accf0 + 8 * r)
                                    : "memory");
                            }
                    }
            }
            // no MMA in flight past this point (the last stage's commit covers all before it)
            if (g > 0 && !mbar_wait(empty0 + 8 * ((g - 1) % NS), (unsigned)(((g - 1) / NS) & 1))) ok = false;
        }
    } else {
        // ---- epilogue (warps 4-7: TMEM lanes 32 (warp - 4) .. +31)
        Gat g{};  // the epilogue needs only the output grid
        g.N = h.N;
        g.H = h.H;
        g.W = h.W;
        unsigned used = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
            int n, i0, rv, x0;
            decode(t, n, i0, rv, x0);
            const bool pool = e.kind == E_POOL;
            const int ps = UP ? 2 : 1, nvalid = min(kBM, (UP ? h.Wi : h.W) - x0);
            bool go = true;
            for (int r = 0; r < rv && go; ++r) {
                const bool ok2 = mbar_wait(accf0 + 8 * r, (used >> r) & 1u);
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                go = __all_sync(0xffffffffu, ok2);
                used ^= 1u << r;
                if (pool) {  // rows in pairs (rv is even)
                    if (!(r & 1) || !go) continue;
                    const int W2 = h.W >> 1, m = (n * (h.H >> 1) + ((i0 + r) >> 1)) * W2 + (x0 >> 1);
                    pool_epilogue<BN>(e, tmem + (unsigned)((r - 1) * BN), tmem + (unsigned)(r * BN), m, nvalid >> 1, W2,
                                      nt * BN, warp - 4, lane);
                } else {
#pragma unroll
                    for (int b = 0; b < NA; ++b) {
                        const int m0 = (n * h.H + i0 + r) * h.W + ps * x0 + b;
                        tc_epilogue<BN>(e, g, tmem + (unsigned)((r * NA + b) * BN), m0, nt * BN, m0 + ps * nvalid, warp - 4,
                                        lane, go, ps);
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                if (pool) mbar_arrive(acce0 + 8 * (r - 1));
                mbar_arrive(acce0 + 8 * r);
            }
            if (!go) {
                ok = false;
                break;
            }
        }
    }
    if (!ok) atomicExch(err, 1);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 8) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(256) : "memory");
    }
}

// Weight gradient on tcgen05: part[z][k][n] = sum over the pixels of split z of
// A(p, k) G[p][n], A the layer's forward gather.  The reduction runs over pixels,
// and a chunk-planar row holds 8 channels of consecutive pixels 16 bytes apart:
// both operands are MN-major core matrices (8 pixels x 8 channels in 128 bytes)
// exactly as the tensors lie in memory, so a stage is one bulk copy per channel
// chunk of a row segment.  M is the weight row (vertical tap, input channel) --
// the 128-row tile stacks the chunks of the input rows of all vertical taps -- and
// N the output channel; each horizontal tap is the same stage read through a
// descriptor shifted by one 16-byte slot, into an accumulator of its own in tensor
// memory.  An upsampling layer reads its half-grid input with the output gradient
// de-interleaved by column parity, a stride-2 layer its input de-interleaved
// likewise.  Units (one row segment of kWgP pixels) are split over blockIdx.z; the
// partials are summed in split order.  Bound by the staging (an input row is read
// once per vertical tap, from L2).  The m16n8k16 form with a per-pixel gather took
// 2.5 ms for the 20 layers at 4 x 256 x 512; this one 0.86 (each launch timed on its
// own).
struct Wg {
    const bf16 *in0, *in1, *G;
    int c0, c1, cin;         // channels of the two tensors, and together
    int H, W, Hi, Wi;        // output grid, input grid
    int co, rows, Kpad;      // output channels; weight rows (vertical taps x cin; stride 2: taps x cin)
    int xt, units, ups;      // segments per image row, units, units per split
};
enum WgKind { WG_CONV3 = 0, WG_UP3 = 1, WG_DOWN2 = 2 };
constexpr int kWgP = 64;                   // reduction pixels per stage
constexpr int kWgStages = 4;
constexpr int kWgAcs = (kWgP + 3) * 16;    // a chunk's slots: one halo slot on either side, one of padding
constexpr int kWgBcs = (kWgP + 1) * 16;

template <int KIND, int BN>
struct WgCfg {
    static constexpr int kShifts = KIND == WG_DOWN2 ? 1 : 3;
    static constexpr int kPar = KIND == WG_UP3 ? 2 : 1;  // column parities of G
    static constexpr int kA = 16 * kWgAcs;
    static constexpr int kB = kPar * (BN / 8) * kWgBcs;
    static constexpr int kStage = (kA + kB + 127) / 128 * 128;
    static constexpr int kBytes = kWgStages * kStage + 256;
    static constexpr int kUsed = kShifts * BN;
    static constexpr int kCols = kUsed <= 64 ? 64 : kUsed <= 128 ? 128 : kUsed <= 256 ? 256 : 512;
    static_assert(kUsed <= 512, "accumulators exceed tensor memory");
};

template <int KIND, int BN>
__global__ void __launch_bounds__(kTcThreads, 1) k_wgrad_tc(Wg w, float *__restrict__ part, int *err)
{
    pdl_entry();
    using C = WgCfg<KIND, BN>;
    constexpr int NS = kWgStages;
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *const bars = smem + NS * C::kStage;
    const unsigned full0 = smem_u32(bars), empty0 = full0 + 8 * NS, done = empty0 + 8 * NS;
    unsigned *const tmem_slot = reinterpret_cast<unsigned *>(bars + 8 * (2 * NS + 1));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n0 = blockIdx.y * BN, u0 = blockIdx.z * w.ups, u1 = min(u0 + w.ups, w.units);
    const int Kw = KIND == WG_UP3 ? w.Wi : w.W;  // reduction pixels of a row
    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(full0 + 8 * s, 128);
            mbar_init(empty0 + 8 * s, 1);
        }
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                     "r"(C::kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned tmem = *tmem_slot;
    bool ok = true;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);

    if (warp < 4) {
        // ---- producers: thread t < 16 stages chunk t of A, the next BN / 8 (one parity) those of B
        const int cq = w.cin >> 3;
        auto a_chunk = [&](int m, int &tg, const bf16 *&base, int &Ct, int &ch) {  // false: rows past the last
            const int gc = blockIdx.x * 16 + m;
            tg = gc / cq;
            ch = (gc - tg * cq) * 8;
            base = ch < w.c0 ? w.in0 : w.in1;
            Ct = ch < w.c0 ? w.c0 : w.c1;
            if (ch >= w.c0) ch -= w.c0;
            return gc * 8 < w.rows;
        };
        int g = 0;
        for (int un = u0; un < u1; ++un, ++g) {
            const int s = g % NS;
            if (g >= NS) ok = mbar_wait(empty0 + 8 * s, (unsigned)((g / NS - 1) & 1));
            if (!ok) break;
            unsigned char *const As = smem + s * C::kStage, *const Bs = As + C::kA;
            const int rowid = un / w.xt, x0 = (un - rowid * w.xt) * kWgP, n = rowid / w.H, i = rowid - n * w.H;
            unsigned bytes = 0, dst = 0;
            const bf16 *src = nullptr;
            if (KIND != WG_DOWN2 && tid < 16) {
                int tg, Ct, ch;
                const bf16 *base;
                const bool valid = a_chunk(tid, tg, base, Ct, ch);
                int y = i + tg - 1;
                const bool in = valid && y >= 0 && y < w.H;
                if (KIND == WG_UP3) y >>= 1;
                unsigned char *const a = As + tid * kWgAcs;
                const int xs = max(x0 - 1, 0), xe = in ? min(x0 + kWgP + 1, w.Wi) : xs, s0 = xs - (x0 - 1);
                for (int sl = 0; sl < s0; ++sl) *reinterpret_cast<uint4 *>(a + sl * 16) = zero;
                for (int sl = s0 + xe - xs; sl < kWgP + 2; ++sl) *reinterpret_cast<uint4 *>(a + sl * 16) = zero;
                if (in) {
                    bytes = (unsigned)(xe - xs) * 16u;
                    dst = smem_u32(a + s0 * 16);
                    src = base + cofs((size_t)n * w.Hi + y, xs, ch, Ct, w.Wi);
                }
            }
            if (KIND == WG_DOWN2) {
                // the input's even / odd columns, rows 2 i and 2 i + 1
                for (int idx = tid; idx < 16 * kWgP; idx += 128) {
                    const int m = idx / kWgP, k = idx - m * kWgP;
                    int tg, Ct, ch;
                    const bf16 *base;
                    const bool v = a_chunk(m, tg, base, Ct, ch) && x0 + k < w.W;
                    uint4 val = zero;
                    if (v)
                        val = *reinterpret_cast<const uint4 *>(
                            base + cofs((size_t)n * w.Hi + 2 * i + (tg >> 1), 2 * (x0 + k) + (tg & 1), ch, Ct, w.Wi));
                    *reinterpret_cast<uint4 *>(As + m * kWgAcs + k * 16) = val;
                }
            }
            const int tb = tid - (KIND == WG_DOWN2 ? 0 : 16);
            if (KIND != WG_UP3 && tb >= 0 && tb < BN / 8) {
                unsigned char *const b = Bs + tb * kWgBcs;
                const int nk = min(kWgP, w.W - x0);
                for (int k = nk; k < kWgP; ++k) *reinterpret_cast<uint4 *>(b + k * 16) = zero;
                bytes = (unsigned)nk * 16u;
                dst = smem_u32(b);
                src = w.G + cofs((size_t)rowid, x0, n0 + 8 * tb, w.co, w.W);
            }
            if (KIND == WG_UP3) {
                for (int idx = tid; idx < 2 * (BN / 8) * kWgP; idx += 128) {
                    const int r = idx / kWgP, k = idx - r * kWgP, b = r & 1, q = r >> 1;
                    uint4 val = zero;
                    if (x0 + k < w.Wi)
                        val = *reinterpret_cast<const uint4 *>(
                            w.G + cofs((size_t)rowid, 2 * (x0 + k) + b, n0 + 8 * q, w.co, w.W));
                    *reinterpret_cast<uint4 *>(Bs + (b * (BN / 8) + q) * kWgBcs + k * 16) = val;
                }
            }
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            if (bytes) {
                mbar_expect_tx(full0 + 8 * s, bytes);
                bulk_g2s(dst, src, bytes, full0 + 8 * s);
            } else {
                mbar_arrive(full0 + 8 * s);
            }
        }
        if (!ok)  // drain what is in flight
            for (int q = max(0, g - NS); q < g; ++q) mbar_wait(full0 + 8 * (q % NS), (unsigned)((q / NS) & 1));
    } else if (lane == 0) {
        // ---- MMA issue: both operands MN-major (bits 15, 16), BF16 x BF16 -> FP32
        constexpr unsigned idesc = umma_idesc<BN>() | (1u << 15) | (1u << 16);
        int g = 0;
        for (int un = u0; un < u1; ++un, ++g) {
            const int s = g % NS;
            ok = mbar_wait(full0 + 8 * s, (unsigned)((g / NS) & 1));
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const unsigned a0 = smem_u32(smem + s * C::kStage), b0 = a0 + C::kA;
            const int x0 = (un % w.xt) * kWgP, ks = (min(kWgP, Kw - x0) + 15) / 16;
            for (int par = 0; par < C::kPar; ++par)
                for (int tb = 0; tb < C::kShifts; ++tb) {
                    const int so = KIND == WG_CONV3 ? tb : KIND == WG_UP3 ? (par + tb + 1) >> 1 : 0;
                    for (int k = 0; k < ks; ++k) {
                        // K step 128 B (8 pixels), M / N step one chunk
                        const uint64_t ad = umma_desc_s(a0 + (so + 16 * k) * 16, 128, kWgAcs);
                        const uint64_t bd = umma_desc_s(b0 + par * (BN / 8) * kWgBcs + 16 * k * 16, 128, kWgBcs);
                        const unsigned acc = (g > 0 || par > 0 || k > 0) ? 1u : 0u;
                        asm volatile(
                            "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem + (unsigned)(tb * BN)),
                            "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                            : "memory");
                    }
                }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(empty0 + 8 * s)
                         : "memory");
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(done) : "memory");
    }
    // ---- the accumulators to this split's partial tile
    const bool drained = mbar_wait(done, 0u);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const bool go = __all_sync(0xffffffffu, ok && drained);
    if (warp < 4 && go) {
        const int row = blockIdx.x * 128 + warp * 32 + lane, ta = row / w.cin, ci = row - ta * w.cin;
        for (int tb = 0; tb < C::kShifts; ++tb) {
            const int k = KIND == WG_DOWN2 ? row : (ta * 3 + tb) * w.cin + ci;
            float *const o = part + ((size_t)blockIdx.z * w.Kpad + k) * w.co + n0;
#pragma unroll 1
            for (int c = 0; c < BN; c += 16) {
                unsigned v[16];
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                    "[%16];\n"
                    : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                      "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                    : "r"(tmem + ((unsigned)(warp * 32) << 16) + (unsigned)(tb * BN + c)));
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                if (row < w.rows)
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        *reinterpret_cast<uint4 *>(o + c + 4 * q) = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2],
                                                                               v[4 * q + 3]);
            }
        }
    }
    if (!(ok && drained)) atomicExch(err, 1);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 4) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(C::kCols) : "memory");
    }
}

// ------------------------------------------------------------ small kernels --
constexpr int kT = 256;
constexpr int kHeadVals = 34;  // per-block partials of the head: dw[32], db, loss

// x FP32 [M][2] (pixel p = row W + x) -> chunk-planar BF16 with kInPad channels, channels 2.. zero.
__global__ void k_input(const float *__restrict__ x, long long M, int W, bf16 *__restrict__ xin)
{
    pdl_entry();
    const long long p = blockIdx.x * (long long)kT + threadIdx.x;
    if (p >= M) return;
    const size_t prow = (size_t)(p / W);
    const int px = (int)(p - (long long)prow * W);
    const float2 v = *reinterpret_cast<const float2 *>(x + 2 * p);
    __align__(16) bf16 row[kInPad];
    row[0] = __float2bfloat16_rn(v.x);
    row[1] = __float2bfloat16_rn(v.y);
#pragma unroll
    for (int c = 2; c < kInPad; ++c) row[c] = __float2bfloat16_rn(0.0f);
#pragma unroll
    for (int q = 0; q < kInPad / 8; ++q)
        *reinterpret_cast<uint4 *>(xin + cofs(prow, px, 8 * q, kInPad, W)) = reinterpret_cast<const uint4 *>(row)[q];
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// 1x1 FP32 head over the 32-channel tensor a: out = a . w + b.  With a target
// (training): dout = 2 (out - t) / M, the gradient of the head input's
// pre-activation G = bf16(dout w * (a > 0)), and per-block partials of dw, db and
// the squared error (kHeadVals per block).
__global__ void __launch_bounds__(kT) k_head(const bf16 *__restrict__ a, const float *__restrict__ w, long long M,
                                             int W, float *__restrict__ out, const float *__restrict__ target,
                                             float inv_m, bf16 *__restrict__ G, float *__restrict__ part)
{
    pdl_entry();
    __shared__ float sh[kT / 32][kHeadVals];
    const long long p = blockIdx.x * (long long)kT + threadIdx.x;
    float av[32];
    float o = 0.0f;
    const size_t prow = (size_t)(p / W);
    const int px = (int)(p - (long long)prow * W);
    if (p < M) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint4 u = *reinterpret_cast<const uint4 *>(a + cofs(prow, px, 8 * q, 32, W));
            const bf16 *h = reinterpret_cast<const bf16 *>(&u);
#pragma unroll
            for (int c = 0; c < 8; ++c) av[8 * q + c] = __bfloat162float(h[c]);
        }
        o = w[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) o = fmaf(av[c], w[c], o);
        out[p] = o;
    }
    if (!target) return;
    float d = 0.0f, se = 0.0f;
    if (p < M) {
        const float r = o - target[p];
        d = 2.0f * r * inv_m;
        se = r * r;
        __align__(16) bf16 g[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) g[c] = __float2bfloat16_rn(av[c] > 0.0f ? d * w[c] : 0.0f);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            *reinterpret_cast<uint4 *>(G + cofs(prow, px, 8 * q, 32, W)) = reinterpret_cast<const uint4 *>(g)[q];
    } else {
#pragma unroll
        for (int c = 0; c < 32; ++c) av[c] = 0.0f;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        const float s = warp_sum(d * av[c]);
        if (lane == 0) sh[warp][c] = s;
    }
    {
        const float s = warp_sum(d);
        if (lane == 0) sh[warp][32] = s;
        const float q = warp_sum(se);
        if (lane == 0) sh[warp][33] = q;
    }
    __syncthreads();
    if (threadIdx.x < kHeadVals) {
        float s = 0.0f;
        for (int wv = 0; wv < kT / 32; ++wv) s += sh[wv][threadIdx.x];
        part[(size_t)blockIdx.x * kHeadVals + threadIdx.x] = s;
    }
}

// Head gradient and loss from the per-block partials: a CTA per value, in a
// fixed order (one thread per value walked 2048 partials in 90 us).
__global__ void __launch_bounds__(kT) k_head_final(const float *__restrict__ part, int nblocks, float *__restrict__ gw,
                                                   double *loss, double inv_m)
{
    pdl_entry();
    __shared__ double sh[kT];
    const int v = blockIdx.x;
    double s = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += kT) s += part[(size_t)b * kHeadVals + v];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int h = kT / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) sh[threadIdx.x] += sh[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x) return;
    if (v < 33)
        gw[v] = (float)sh[0];
    else
        *loss = sh[0] * inv_m;
}

// Column sums of a chunk-planar G [rows][C / 8][W][8] (bias gradient): block (q, b)
// sums chunk q over rows [b rpb, (b + 1) rpb) into part[b][8 q ..], 16 bytes a load.
__global__ void __launch_bounds__(kT) k_colsum(const bf16 *__restrict__ G, int rows, int W, int C, int rpb,
                                               float *__restrict__ part)
{
    pdl_entry();
    __shared__ float sh[kT / 32][8];
    const int nq = C / 8, q = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float acc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = 0.0f;
    const int r0 = blockIdx.y * rpb, r1 = min(r0 + rpb, rows);
    for (int r = r0; r < r1; ++r) {
        const uint4 *seg = reinterpret_cast<const uint4 *>(G + ((size_t)r * nq + q) * (size_t)W * 8);
        for (int x = threadIdx.x; x < W; x += kT) {
            const uint4 u = seg[x];
            const bf16 *h = reinterpret_cast<const bf16 *>(&u);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] += __bfloat162float(h[c]);
        }
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float s = warp_sum(acc[c]);
        if (lane == 0) sh[warp][c] = s;
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        float s = 0.0f;
        for (int v = 0; v < kT / 32; ++v) s += sh[v][threadIdx.x];
        part[(size_t)blockIdx.y * C + 8 * q + threadIdx.x] = s;
    }
}

// A layer's gradient from its partials, in fixed order: weights gw[(t ci + c) co +
// o] = sum_z part[z][t cinp + c][o], then the bias gw[nw + o] = sum_b cpart[b][o].
// 32 values per CTA, the partials over 8 warps.
__global__ void __launch_bounds__(kT) k_wgrad_reduce(const float *__restrict__ part, int splits, int Kpad, int co,
                                                     int cinp, int ci, int nw, const float *__restrict__ cpart, int nb,
                                                     float *__restrict__ gw)
{
    pdl_entry();
    __shared__ float sh[kT / 32][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, idx = blockIdx.x * 32 + lane;
    float s = 0.0f;
    if (idx < nw) {
        const int r = idx / co, o = idx - r * co, t = r / ci, c = r - t * ci;
        const float *p = part + (size_t)(t * cinp + c) * co + o;
        const size_t zs = (size_t)Kpad * co;
#pragma unroll 4
        for (int z = warp; z < splits; z += kT / 32) s += p[z * zs];
    } else if (idx < nw + co) {
        const float *p = cpart + (idx - nw);
#pragma unroll 4
        for (int b = warp; b < nb; b += kT / 32) s += p[(size_t)b * co];
    }
    sh[warp][lane] = s;
    __syncthreads();
    if (warp || idx >= nw + co) return;
    s = 0.0f;
    for (int v = 0; v < kT / 32; ++v) s += sh[v][lane];
    gw[idx] = s;
}

// Adam with bias correction (b1t = 1 - beta1^t, b2t = 1 - beta2^t).
__global__ void k_adam(float *__restrict__ th, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, long long n, float lr, float b1t, float b2t)
{
    pdl_entry();
    const long long k = blockIdx.x * (long long)kT + threadIdx.x;
    if (k >= n) return;
    const float gk = g[k];
    const float mk = 0.9f * m[k] + 0.1f * gk;
    const float vk = 0.999f * v[k] + 0.001f * gk * gk;
    m[k] = mk;
    v[k] = vk;
    th[k] -= lr * (mk / b1t) / (sqrtf(vk / b2t) + 1e-8f);
}

// Halo-ordered BF16 weights of a halo GEMM: for each column tile nt (BN wide),
// stage (cc, ta) and horizontal tap tb (tv x th taps, tap t = th ta + tb), a
// BN x CS block in core-matrix order: element (n, ch) at
// ((n / 8) (CS / 8) + ch / 8) 64 + (n % 8) 8 + ch % 8.  Forward (flip = 0):
// value W[t][cc CS + ch][nt BN + n] (zero for channels >= ci, the input
// layer's padding); 3x3 input gradient (flip = 1): W[8 - t][nt BN + n][cc CS + ch].
// W is [tv th][ci][co] FP32.
__global__ void k_pack_halo(const float *__restrict__ W, int ci, int co, int kin, int ncols, int BN, int CS, int tv,
                            int th, int flip, bf16 *__restrict__ out)
{
    pdl_entry();
    const long long idx = blockIdx.x * (long long)kT + threadIdx.x;
    const long long nst = (long long)(kin / CS) * tv;
    const long long blk = (long long)BN * CS;
    if (idx >= (long long)(ncols / BN) * nst * th * blk) return;
    const long long b = idx / blk;
    const int w = (int)(idx - b * blk);
    const int tb = (int)(b % th), st = (int)((b / th) % nst), nt = (int)(b / (th * nst));
    const int cc = st / tv, ta = st - tv * cc;
    const int rb = w / 64, r = w - rb * 64, nb = rb / (CS / 8), qb = rb - nb * (CS / 8);
    const int nn = nb * 8 + r / 8, ch = qb * 8 + r % 8;
    const int col = nt * BN + nn, kc = cc * CS + ch, t = th * ta + tb;
    float v;
    if (!flip)
        v = kc < ci ? W[((size_t)t * ci + kc) * co + col] : 0.0f;
    else
        v = W[((size_t)(8 - t) * ci + col) * co + kc];
    out[idx] = __float2bfloat16_rn(v);
}

// BF16 copy of a stride-2 layer's weights W [4][ci][co]: the K-major matrices
// [t][c][o] of its input-gradient GEMMs (one per sub-pixel t).
__global__ void k_pack_down(const float *__restrict__ W, long long n, bf16 *__restrict__ Bk)
{
    pdl_entry();
    const long long q = blockIdx.x * (long long)kT + threadIdx.x;
    if (q < n) Bk[q] = __float2bfloat16_rn(W[q]);
}

// ------------------------------------------------- features of a pressure problem --
// part[b] = sum of b^2 over block b's cells (FP64).
__global__ void __launch_bounds__(kT) k_feat_bsum(const double *__restrict__ b, int n, double *__restrict__ part)
{
    pdl_entry();
    __shared__ double sh[kT / 32];
    double s = 0.0;
    for (int c = blockIdx.x * kT + threadIdx.x; c < n; c += gridDim.x * kT) s += b[c] * b[c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kT / 32; ++w) t += sh[w];
        part[blockIdx.x] = t;
    }
}

// Sum of n partials, computed once per block (warp 0, fixed order) and shared:
// the same value in every block.  Call from all threads of the block.
__device__ double block_sum_parts(const double *part, int n)
{
    __shared__ double r;
    if (threadIdx.x < 32) {
        double s = 0.0;
        for (int k = threadIdx.x; k < n; k += 32) s += part[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) r = s;
    }
    __syncthreads();
    const double v = r;
    __syncthreads();  // r may be written again by the next call
    return v;
}

__device__ __forceinline__ double cell_beta(const double *bu, const double *bv, int nx, int i, int j)
{
    return 0.25 * (bu[j * (nx + 1) + i] + bu[j * (nx + 1) + i + 1] + bv[j * nx + i] + bv[(j + 1) * nx + i]);
}

// Features x [n][2] (and, if phi is given, the target t [n]) of A phi = b.
__global__ void k_features(int nx, int ny, const double *__restrict__ b, const double *__restrict__ bu,
                           const double *__restrict__ bv, const double *__restrict__ inp, double rho_w,
                           const double *__restrict__ part, int nparts, const double *__restrict__ phi,
                           float *__restrict__ x, float *__restrict__ t)
{
    pdl_entry();
    const double s2 = block_sum_parts(part, nparts);
    const int c = blockIdx.x * kT + threadIdx.x;
    if (c >= nx * ny) return;
    const int i = c % nx, j = c / nx;
    const double beta = cell_beta(bu, bv, nx, i, j);
    float x0 = 0.0f, x1 = 0.0f, tt = 0.0f;
    if (s2 > 0.0 && beta > 0.0) {  // FP32 arithmetic: the features are FP32 network inputs
        const float irms = (float)(1.0 / sqrt(s2 / (double(nx) * ny)));
        x0 = (float)b[c] * irms;
        x1 = 0.25f * logf((float)(rho_w * beta) / (float)inp[0]);
        if (phi) tt = (float)phi[c] * (float)beta * irms;
    }
    *reinterpret_cast<float2 *>(x + 2 * (size_t)c) = make_float2(x0, x1);
    if (phi) t[c] = tt;
}

// phi0 = out rms(b) / beta_c; then part2[b] = sum of (b - A phi0)^2 over block b.
__global__ void k_guess(int nx, int ny, const double *__restrict__ b, const double *__restrict__ bu,
                        const double *__restrict__ bv, const double *__restrict__ part, int nparts,
                        const float *__restrict__ out, double *__restrict__ phi)
{
    pdl_entry();
    const double s2 = block_sum_parts(part, nparts);
    const int c = blockIdx.x * kT + threadIdx.x;
    if (c >= nx * ny) return;
    const int i = c % nx, j = c / nx;
    const double beta = cell_beta(bu, bv, nx, i, j);
    const float rms = (float)sqrt(s2 / (double(nx) * ny));  // FP32: an initial guess, judged by its FP64 residual
    phi[c] = (s2 > 0.0 && beta > 0.0) ? double(out[c] * rms / (float)beta) : 0.0;
}

__global__ void __launch_bounds__(kT) k_guess_resid(int nx, int ny, const double *__restrict__ b,
                                                    const double *__restrict__ bu, const double *__restrict__ bv,
                                                    const double *__restrict__ phi, double *__restrict__ part)
{
    pdl_entry();
    __shared__ double sh[kT / 32];
    double s = 0.0;
    for (int c = blockIdx.x * kT + threadIdx.x; c < nx * ny; c += gridDim.x * kT) {
        const int i = c % nx, j = c / nx;
        const double r = b[c] - (diag_at(bu, bv, nx, ny, i, j) * phi[c] - offsum_at(bu, bv, phi, nx, ny, i, j));
        s += r * r;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kT / 32; ++w) t += sh[w];
        part[blockIdx.x] = t;
    }
}

// Keep phi0 only if ||b - A phi0|| < ||b|| (else phi0 = 0); count tried / kept.
__global__ void k_guess_select(int n, const double *__restrict__ pb, const double *__restrict__ pr, int nparts,
                               double *__restrict__ phi, long long *stats)
{
    pdl_entry();
    const double b2 = block_sum_parts(pb, nparts);
    const double r2 = block_sum_parts(pr, nparts);
    const bool keep = r2 < b2;
    const int c = blockIdx.x * kT + threadIdx.x;
    if (!keep && c < n) phi[c] = 0.0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        stats[0] += 1;
        stats[1] += keep ? 1 : 0;
    }
}

}  // namespace
}  // namespace wec

struct wec_net {
    int H = 0, W = 0, maxb = 0;
    cudaStream_t st = nullptr;
    size_t nparam = 0;
    float *theta = nullptr, *grad = nullptr, *am = nullptr, *av = nullptr;  // FP32 [nparam] each
    long long adam_t = 0;
    bool wdirty = true;                       // BF16 matrices older than theta
    bf16 *wmat = nullptr;                     // every layer's BF16 matrices
    size_t flat[wec::kNumLayers] = {};        // layer weights in theta (bias follows)
    size_t wb[wec::kNumLayers] = {};          // stride-2 layers: input-gradient matrices in wmat
    size_t hf[wec::kNumLayers] = {}, hb[wec::kNumLayers] = {};  // halo-ordered 3x3 matrices (forward / input gradient)
    int bnf[wec::kNumLayers] = {}, bnb[wec::kNumLayers] = {};   // their column-tile widths
    bf16 *xin = nullptr;                      // [maxb][H][W][8]
    bf16 *act[wec::kNumLayers] = {};          // layer outputs
    float *out = nullptr;                     // [maxb][H][W]
    bf16 *gA[4] = {}, *gB[4] = {}, *skip[3] = {};  // gradients per level
    float *part = nullptr;                    // split-K partials of the weight gradients
    size_t part_n = 0;
    float *cpart = nullptr;                   // column-sum / head partials
    float *xb = nullptr, *tb = nullptr;       // gathered batch (or a tank's features)
    double *loss = nullptr, *lossh = nullptr; // device / pinned host
    double *dpart = nullptr;                  // FP64 partials of the tank guess (2 x kRedBlocks)
    int *err = nullptr;                       // device: set when a tensor-core pipeline wait expired
    std::vector<void *> allocs;
};

namespace wec {
namespace {

constexpr int kCsumBlocks = 912;   // CTAs of a bias-gradient launch (6 per SM)

size_t weight_count(int L) { return (size_t)taps(kLayers[L].kind) * kLayers[L].ci * kLayers[L].co; }
int fwd_K(int L) { return taps(kLayers[L].kind) * cin_pad(kLayers[L].ci); }
int level_h(const wec_net *N, int l) { return N->H >> l; }
int level_w(const wec_net *N, int l) { return N->W >> l; }
int chans(int l) { return 32 << l; }

void layer_inputs(const wec_net *N, int L, const bf16 **in0, const bf16 **in1)
{
    *in1 = nullptr;
    for (int l = 0; l < 4; ++l) {
        if (L == enc_a(l)) *in0 = l == 0 ? N->xin : N->act[down(l - 1)];
        if (L == enc_b(l)) *in0 = N->act[enc_a(l)];
        if (l < 3 && L == down(l)) *in0 = N->act[enc_b(l)];
        if (l < 3 && L == up(l)) *in0 = l == 2 ? N->act[enc_b(3)] : N->act[dec(l + 1)];
        if (l < 3 && L == cat(l)) {
            *in0 = N->act[up(l)];
            *in1 = N->act[enc_b(l)];
        }
        if (l < 3 && L == dec(l)) *in0 = N->act[cat(l)];
    }
}

// Layer L's input tensors and output grid.
Gat fwd_gather(const wec_net *N, int L, int batch)
{
    const LayerDef &d = kLayers[L];
    const int cinp = cin_pad(d.ci), H = level_h(N, d.level), W = level_w(N, d.level);
    Gat g{};
    layer_inputs(N, L, &g.in0, &g.in1);
    g.c0 = g.in1 ? cinp / 2 : cinp;
    g.c1 = g.in1 ? cinp / 2 : 0;
    g.N = batch;
    g.H = H;
    g.W = W;
    g.Hi = d.kind == L_UP3 ? H / 2 : (d.kind == L_DOWN2 ? 2 * H : H);
    g.Wi = d.kind == L_UP3 ? W / 2 : (d.kind == L_DOWN2 ? 2 * W : W);
    g.K = fwd_K(L);
    return g;
}

template <int BN>
int launch_down_dx(cudaStream_t st, unsigned mt, const bf16 *G, int K, int ncols, int M, int W, const bf16 *B, const Epi &e,
                   int *err)
{
    const int smem = K / kTcK * (kBM + BN) * kTcK * 2 + 256;
    static bool attr = false;  // dynamic shared memory above 48 KB, set once per instantiation
    if (!attr) {
        WEC_CK(cudaFuncSetAttribute(k_down_dx<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        attr = true;
    }
    WEC_CK(launch_k(k_down_dx<BN>, dim3(mt, (unsigned)(ncols / BN)), kTcThreads, smem, st, G, K, M, W, B, e, err));
    return WEC_OK;
}

// Input gradient of down(l) (profile level 100 + layer) from its output gradient G on
// the half grid.  Tile width: the widest of 256/128/64/32 dividing the 4C columns
// that still gives >= 256 CTAs (about two per SM), else 32.
int down_dx(wec_net *N, int l, int batch, const bf16 *G, const Epi &e)
{
    const int C = chans(l), K = 2 * C, ncols = 4 * C, W = level_w(N, l + 1), M = batch * level_h(N, l + 1) * W;
    const unsigned mt = (unsigned)((M + kBM - 1) / kBM);
    int bn = 32;
    for (int c : {256, 128, 64})
        if (ncols % c == 0 && mt * (ncols / c) >= 256) {
            bn = c;
            break;
        }
    const bf16 *B = N->wmat + N->wb[down(l)];
    WEC_PROF("net_conv", 100 + down(l), 2.0 * M * (K + 3.0 * ncols) + 2.0 * K * ncols, N->st);
    switch (bn) {
    case 256: return launch_down_dx<256>(N->st, mt, G, K, ncols, M, W, B, e, N->err);
    case 128: return launch_down_dx<128>(N->st, mt, G, K, ncols, M, W, B, e, N->err);
    case 64: return launch_down_dx<64>(N->st, mt, G, K, ncols, M, W, B, e, N->err);
    default: return launch_down_dx<32>(N->st, mt, G, K, ncols, M, W, B, e, N->err);
    }
}

// ---- convolutions with the halo kernel ----
inline int halo_cs(int c) { return c >= 64 ? 64 : c; }  // channels per stage (c: channels of one input tensor)
inline bool halo_fwd(int L) { return kLayers[L].kind != L_HEAD; }
inline bool halo_bwd(int L) { return L != enc_a(0) && (kLayers[L].kind == L_CONV3 || kLayers[L].kind == L_UP3); }
inline int halo_kin(int L, bool bwd) { return bwd ? kLayers[L].co : cin_pad(kLayers[L].ci); }
inline int halo_mode(int kind) { return kind == L_UP3 ? H_UP3 : (kind == L_DOWN2 ? H_DOWN2 : H_CONV3); }

// one-row tiles of an image; the up mode tiles the half-resolution row
long long halo_tiles(const wec_net *N, int level, bool up)
{
    const int w = up ? level_w(N, level) / 2 : level_w(N, level);
    return (long long)level_h(N, level) * ((w + kBM - 1) / kBM);
}

// Column-tile width: the widest of 128 / 64 dividing ncols that still gives >= 128
// tiles for one image (measured: wider tiles beat more, narrower ones down to
// about one tile per SM), else 32.  The up mode tiles the half-resolution row.
int halo_bn(const wec_net *N, int level, int ncols, bool up = false)
{
    const long long tiles = halo_tiles(N, level, up);
    for (int c : {128, 64})
        if (ncols % c == 0 && tiles * (ncols / c) >= 128) return c;
    return 32;
}

// Persistent grid: as many CTAs as fit on the GPU at once (shared memory and
// tensor-memory columns), at most one per tile.
template <int BN, int CS, bool DOWN>
int launch_halo_t(cudaStream_t st, long long ntiles, const Halo &h, const bf16 *B, const Epi &e, int *err)
{
    using S = HaloSmem<BN, CS, DOWN>;
    static int ctas = 0;  // resident CTAs on the device, computed once per instantiation
    if (!ctas) {
        WEC_CK(cudaFuncSetAttribute(k_conv_halo<BN, CS, DOWN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    S::kBytes));
        int occ = 0;
        WEC_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_conv_halo<BN, CS, DOWN>, kPThreads, S::kBytes));
        const int cols = DOWN ? 2 * BN : 4 * BN;
        ctas = sm_count() * std::max(1, std::min(occ, 512 / cols));
    }
    const unsigned grid = (unsigned)std::min<long long>(ntiles, ctas);
    WEC_CK(launch_k(k_conv_halo<BN, CS, DOWN>, grid, kPThreads, S::kBytes, st, h, B, e, err));
    return WEC_OK;
}

template <int BN>
int launch_halo_cs(int CS, bool down, cudaStream_t st, long long ntiles, const Halo &h, const bf16 *B, const Epi &e,
                   int *err)
{
    if (down) {
        if (CS == 64) return launch_halo_t<BN, 64, true>(st, ntiles, h, B, e, err);
        if (CS == 32) return launch_halo_t<BN, 32, true>(st, ntiles, h, B, e, err);
    } else {
        if (CS == 64) return launch_halo_t<BN, 64, false>(st, ntiles, h, B, e, err);
        if (CS == 32) return launch_halo_t<BN, 32, false>(st, ntiles, h, B, e, err);
        if (CS == 16) return launch_halo_t<BN, 16, false>(st, ntiles, h, B, e, err);
    }
    return fail(WEC_ERR_INVALID, "net: unsupported channels per stage");
}

// Column-tile width of the row-block kernel (k_conv_rows), or 0 where it does not
// apply: above the coarsest level, the widest tile whose weights take at most 76 KB
// (beside the staged rows of a second CTA), and as many columns as the layers of the
// level have outputs -- twice as many lose: 64 -> 128 channels at level 1 took 49 us
// against 46 with the one-row tiles, four images of 256 x 512.  At level 2,
// 128 -> 128 channels take 26 us (30).  E_POOL always (level 1: 27 us; an FP32 full
// grid and a pooling pass took 55 + 30).  The up mode only with three stages: with
// two, 128 -> 64 channels took 25 us against 22.  And only where the one-row tiles of
// the largest batch are more than the SMs: up to there each has a CTA of its own, and
// half as many CTAs with twice the work lose -- 64 -> 64 channels at 32 x 64 to 64 x
// 128 pixels 13 us against 10, 128 -> 128 at 16 x 32 15 against 12, a forward pass at
// 64 x 128 200 against 170 (E_POOL has the row blocks alone).
int rows_bn(const wec_net *N, int mode, int level, int cin, int ncols, bool pool = false)
{
    if (mode == H_DOWN2 || level > 2 || (ncols > std::max(64, chans(level)) && !pool)) return 0;
    const bool up = mode == H_UP3;
    if (!pool && N->maxb * halo_tiles(N, level, up) * (ncols / halo_bn(N, level, ncols, up)) <= sm_count()) return 0;
    if (mode == H_UP3) return cin == 64 && ncols == 32 ? 32 : 0;
    for (int bn : {64, 32})
        if (ncols % bn == 0 && 9 * cin * bn * 2 <= 76 * 1024) return bn;
    return 0;
}

template <int BN, int CS, bool UP, int NS>
int launch_rows_t(cudaStream_t st, const Halo &h, const bf16 *B, const Epi &e, int *err)
{
    using S = RowsCfg<BN, CS, UP, NS>;
    auto kern = k_conv_rows<BN, CS, UP, NS>;
    const int smem = S::bytes(h.c0 + h.c1);
    static bool attr = false;
    if (!attr) {
        WEC_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 113 * 1024));
        attr = true;
    }
    const int ntn = h.ncols / BN, slots = std::max(1, 2 * sm_count() / ntn);
    // rows per tile: as many as the accumulators hold, fewer where the tiles would not fill the GPU
    int R = S::kRows;
    auto tiles = [&](int r) { return (long long)h.N * ((h.H + r - 1) / r) * h.xtiles; };
    while (R > 2 && tiles(R) < slots) R /= 2;
    const dim3 grid((unsigned)std::min<long long>(tiles(R), slots), (unsigned)ntn);
    WEC_CK(launch_k(kern, grid, kPThreads, smem, st, h, R, B, e, err));
    return WEC_OK;
}

int launch_rows(int BN, int CS, cudaStream_t st, const Halo &h, const bf16 *B, const Epi &e, int *err)
{
    const bool wide = 9 * (h.c0 + h.c1) * BN * 2 > 56 * 1024;  // two stages beside the weights, else three or four
    if (h.mode == H_UP3) return launch_rows_t<32, 64, true, 3>(st, h, B, e, err);
    if (BN == 64)
        return wide ? launch_rows_t<64, 64, false, 2>(st, h, B, e, err) : launch_rows_t<64, 32, false, 4>(st, h, B, e, err);
    if (CS == 64)
        return wide ? launch_rows_t<32, 64, false, 2>(st, h, B, e, err) : launch_rows_t<32, 64, false, 3>(st, h, B, e, err);
    return CS == 32 ? launch_rows_t<32, 32, false, 4>(st, h, B, e, err) : launch_rows_t<32, 16, false, 4>(st, h, B, e, err);
}

// A convolution of the given HaloMode whose output grid is the level's: input
// channels [0, c0) from in0 and [c0, c0 + c1) from in1 (concatenation; c1 = 0:
// one tensor), ncols output channels, halo-ordered weights B of tile width BN.
int conv_halo(wec_net *N, cudaStream_t st, int tag, int mode, int batch, int level, const bf16 *in0, int c0,
              const bf16 *in1, int c1, const bf16 *B, int BN, int ncols, const Epi &e)
{
    Halo h{};
    h.in0 = in0;
    h.in1 = in1 ? in1 : in0;
    h.c0 = c0;
    h.c1 = in1 ? c1 : 0;
    h.N = batch;
    h.H = level_h(N, level);
    h.W = level_w(N, level);
    h.Hi = mode == H_UP3 ? h.H / 2 : (mode == H_DOWN2 ? 2 * h.H : h.H);
    h.Wi = mode == H_UP3 ? h.W / 2 : (mode == H_DOWN2 ? 2 * h.W : h.W);
    h.xtiles = ((mode == H_UP3 ? h.Wi : h.W) + kBM - 1) / kBM;  // the up mode tiles its input row
    h.mode = mode;
    const int CS = halo_cs(c0), tv = mode == H_DOWN2 ? 2 : 3;
    h.nst = (h.c0 + h.c1) / CS * tv;
    h.ncols = ncols;
    const long long ntiles = (long long)batch * h.H * h.xtiles * (ncols / BN);
    const double M = (double)batch * h.H * h.W;
    WEC_PROF("net_conv", tag, 2.0 * M * ((double)(h.c0 + h.c1) + ncols) + 2.0 * tv * tv * (h.c0 + h.c1) * ncols, st);
    if (rows_bn(N, mode, level, h.c0 + h.c1, ncols, e.kind == E_POOL)) return launch_rows(BN, CS, st, h, B, e, N->err);
    switch (BN) {
    case 128: return launch_halo_cs<128>(CS, mode == H_DOWN2, st, ntiles, h, B, e, N->err);
    case 64: return launch_halo_cs<64>(CS, mode == H_DOWN2, st, ntiles, h, B, e, N->err);
    default: return launch_halo_cs<32>(CS, mode == H_DOWN2, st, ntiles, h, B, e, N->err);
    }
}

// The weight-gradient GEMM of layer L: columns per CTA, CTAs per SM (by shared
// memory), and the weight rows its 128-row tiles cover.
struct WgShape {
    int bn, occ, rows;
};
WgShape wgrad_shape(int L)
{
    const LayerDef &d = kLayers[L];
    const int bn = std::min(d.co, 128);
    return {bn, bn == 32 || (bn == 64 && d.kind != L_UP3) ? 2 : 1, (d.kind == L_DOWN2 ? 4 : 3) * cin_pad(d.ci)};
}

// Splits of its units (row segments) over blockIdx.z: at most as many CTAs as are resident.
int wgrad_max_splits(long long units, int L)
{
    const WgShape w = wgrad_shape(L);
    const int tiles = (w.rows + 127) / 128 * (kLayers[L].co / w.bn);
    return (int)std::min<long long>(std::max(1, sm_count() * w.occ / tiles), units);
}
int wgrad_splits(long long units, int L, int *ups)
{
    const int splits = wgrad_max_splits(units, L);
    *ups = (int)((units + splits - 1) / splits);
    return (int)((units + *ups - 1) / *ups);
}

// Row segments of layer L over `rows` image rows of its output grid
long long wgrad_units(const wec_net *N, int L, long long rows)
{
    const LayerDef &d = kLayers[L];
    const int kw = level_w(N, d.level) / (d.kind == L_UP3 ? 2 : 1);
    return rows * ((kw + kWgP - 1) / kWgP);
}

template <int KIND, int BN>
int launch_wgrad_t(wec_net *N, const Wg &w, int splits)
{
    using C = WgCfg<KIND, BN>;
    static bool set = false;
    if (!set) {
        WEC_CK(cudaFuncSetAttribute(k_wgrad_tc<KIND, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kBytes));
        set = true;
    }
    const dim3 grid((unsigned)((w.rows + 127) / 128), (unsigned)(w.co / BN), (unsigned)splits);
    WEC_CK(launch_k(k_wgrad_tc<KIND, BN>, grid, kTcThreads, C::kBytes, N->st, w, N->part, N->err));
    return WEC_OK;
}

template <int KIND>
int launch_wgrad(wec_net *N, const Wg &w, int bn, int splits)
{
    if constexpr (KIND != WG_DOWN2)  // (no stride-2 layer has 32 output channels)
        if (bn == 32) return launch_wgrad_t<KIND, 32>(N, w, splits);
    return bn == 64 ? launch_wgrad_t<KIND, 64>(N, w, splits) : launch_wgrad_t<KIND, 128>(N, w, splits);
}

// grad of layer L's weights and bias from its output gradient G.
int wgrad(wec_net *N, int L, int batch, const bf16 *G)
{
    const LayerDef &d = kLayers[L];
    const Gat g = fwd_gather(N, L, batch);
    const long long M = (long long)g.N * g.H * g.W;
    const WgShape sh = wgrad_shape(L);
    const int rows = g.N * g.H;
    Wg w{};
    w.in0 = g.in0;
    w.in1 = g.in1;
    w.G = G;
    w.c0 = g.c0;
    w.c1 = g.c1;
    w.cin = g.c0 + g.c1;
    w.H = g.H;
    w.W = g.W;
    w.Hi = g.Hi;
    w.Wi = g.Wi;
    w.co = d.co;
    w.rows = sh.rows;
    w.Kpad = round_up(g.K, kBM);
    const long long units = wgrad_units(N, L, rows);
    w.xt = (int)(units / rows);
    w.units = (int)units;
    const int splits = wgrad_splits(units, L, &w.ups);
    cudaStream_t st = N->st;
    {
        WEC_PROF("net_wgrad", L, 2.0 * M * ((double)w.cin + d.co), st);
        const int e = d.kind == L_CONV3 ? launch_wgrad<WG_CONV3>(N, w, sh.bn, splits)
                      : d.kind == L_UP3 ? launch_wgrad<WG_UP3>(N, w, sh.bn, splits)
                                        : launch_wgrad<WG_DOWN2>(N, w, sh.bn, splits);
        if (e) return e;
    }
    const int nq = d.co / 8, want = std::min(rows, std::max(1, kCsumBlocks / nq));
    const int rpb = (rows + want - 1) / want, nb = (rows + rpb - 1) / rpb;
    {
        WEC_PROF("net_bias_grad", -1, 2.0 * M * d.co, st);
        WEC_CK(launch_k(k_colsum, dim3(nq, nb), kT, 0, st, G, rows, g.W, d.co, rpb, N->cpart));
    }
    const int nw = (int)weight_count(L);
    WEC_PROF("net_wgrad_reduce", -1, 4.0 * nw * (splits + 1), st);
    WEC_CK(launch_k(k_wgrad_reduce, nblk(nw + d.co, 32), kT, 0, st, (const float *)N->part, splits, w.Kpad, d.co,
                    cin_pad(d.ci), d.ci, nw, (const float *)N->cpart, nb, N->grad + N->flat[L]));
    return WEC_OK;
}

// Input gradient of a 3x3 layer (conv or up): the 3x3 convolution of G (its
// output gradient, level grid) with the flipped, transposed weights.
int dx_conv(wec_net *N, int L, int batch, const bf16 *G, const Epi &e)
{
    const LayerDef &d = kLayers[L];
    return conv_halo(N, N->st, 100 + L, H_CONV3, batch, d.level, G, d.co, nullptr, 0, N->wmat + N->hb[L], N->bnb[L],
                     d.ci, e);
}

int pack_weights(wec_net *N)
{
    for (int L = 0; L < kHead; ++L) {
        const LayerDef &d = kLayers[L];
        if (d.kind == L_DOWN2) {
            const long long n = (long long)weight_count(L);
            WEC_PROF("net_pack", -1, 6.0 * n, N->st);
            WEC_CK(launch_k(k_pack_down, nblk(n, kT), kT, 0, N->st, (const float *)(N->theta + N->flat[L]), n,
                            N->wmat + N->wb[L]));
        }
        for (int bwd = 0; bwd < 2; ++bwd) {
            if (!(bwd ? halo_bwd(L) : halo_fwd(L))) continue;
            const int kin = halo_kin(L, bwd), ncols = bwd ? d.ci : d.co, BN = bwd ? N->bnb[L] : N->bnf[L];
            const bool concat = L == cat(0) || L == cat(1) || L == cat(2);
            const int cs = halo_cs(bwd ? d.co : (concat ? d.ci / 2 : kin));
            const int tv = (!bwd && d.kind == L_DOWN2) ? 2 : 3;
            const long long nh = (long long)tv * tv * kin * ncols;
            WEC_PROF("net_pack", -1, 4.0 * weight_count(L) + 2.0 * nh, N->st);
            WEC_CK(launch_k(k_pack_halo, nblk(nh, kT), kT, 0, N->st, (const float *)(N->theta + N->flat[L]), d.ci,
                            d.co, kin, ncols, BN, cs, tv, tv, bwd, N->wmat + (bwd ? N->hb[L] : N->hf[L])));
        }
    }
    N->wdirty = false;
    return WEC_OK;
}

// Forward pass of batch images x (FP32 [batch][H][W][2]) into out; with a
// target, also the head's gradient, loss partials and G of dec0 (in gA[0]).
int forward(wec_net *N, int batch, const float *x, float *out, const float *target)
{
    cudaStream_t st = N->st;
    if (N->wdirty)
        if (int e = pack_weights(N)) return e;
    const long long M = (long long)batch * N->H * N->W;
    {
        WEC_PROF("net_input", -1, 8.0 * M + 16.0 * M, st);
        WEC_CK(launch_k(k_input, nblk(M, kT), kT, 0, st, x, M, N->W, N->xin));
    }
    for (int L = 0; L < kHead; ++L) {
        const LayerDef &d = kLayers[L];
        Epi e{};
        e.kind = E_FWD;
        e.bias = N->theta + N->flat[L] + weight_count(L);
        e.out0 = N->act[L];
        e.ld0 = d.co;
        const Gat g = fwd_gather(N, L, batch);
        if (int r = conv_halo(N, st, L, halo_mode(d.kind), batch, d.level, g.in0, g.c0, g.in1, g.c1,
                              N->wmat + N->hf[L], N->bnf[L], d.co, e))
            return r;
    }
    const int nb = nblk(M, kT);
    {
        WEC_PROF("net_head", -1, 64.0 * M + 8.0 * M, st);
        WEC_CK(launch_k(k_head, nb, kT, 0, st, (const bf16 *)N->act[dec(0)], (const float *)(N->theta + N->flat[kHead]),
                        M, N->W, out, target, (float)(1.0 / (double)M), N->gA[0], N->cpart));
    }
    if (target) {
        WEC_PROF("net_head", -1, 4.0 * kHeadVals * nb, st);
        WEC_CK(launch_k(k_head_final, kHeadVals, kT, 0, st, (const float *)N->cpart, nb, N->grad + N->flat[kHead], N->loss,
                        1.0 / (double)M));
    }
    return WEC_OK;
}

int backward(wec_net *N, int batch)
{
    for (int l = 0; l < 3; ++l) {  // decoder, last level first; G of dec(l) is in gA[l]
        const int C = chans(l);
        if (int r = wgrad(N, dec(l), batch, N->gA[l])) return r;
        Epi e{};
        e.kind = E_DX;
        e.out0 = N->gB[l];
        e.mask0 = N->act[cat(l)];
        e.ld0 = C;
        e.nsplit = C;
        if (int r = dx_conv(N, dec(l), batch, N->gA[l], e)) return r;
        if (int r = wgrad(N, cat(l), batch, N->gB[l])) return r;
        e.out0 = N->gA[l];
        e.mask0 = N->act[up(l)];
        e.out1 = N->skip[l];
        e.ld1 = C;
        if (int r = dx_conv(N, cat(l), batch, N->gB[l], e)) return r;
        if (int r = wgrad(N, up(l), batch, N->gA[l])) return r;
        Epi f{};
        f.ld0 = 2 * C;
        f.kind = E_POOL;  // the 2x2 sums in the epilogue
        f.out0 = N->gA[l + 1];
        f.mask0 = l == 2 ? N->act[enc_b(3)] : N->act[dec(l + 1)];
        if (int r = dx_conv(N, up(l), batch, N->gA[l], f)) return r;
    }
    for (int l = 3; l >= 0; --l) {  // encoder; G of down(l)'s output is in gA[l + 1]
        const int C = chans(l);
        if (l < 3) {
            if (int r = wgrad(N, down(l), batch, N->gA[l + 1])) return r;
            Epi e{};
            e.kind = E_DOWNDX;
            e.out0 = N->gA[l];
            e.mask0 = N->act[enc_b(l)];
            e.ld0 = C;
            e.add = N->skip[l];
            if (int r = down_dx(N, l, batch, N->gA[l + 1], e)) return r;
        }
        if (int r = wgrad(N, enc_b(l), batch, N->gA[l])) return r;
        Epi e{};
        e.kind = E_DX;
        e.out0 = N->gB[l];
        e.mask0 = N->act[enc_a(l)];
        e.ld0 = C;
        e.nsplit = C;
        if (int r = dx_conv(N, enc_b(l), batch, N->gA[l], e)) return r;
        if (int r = wgrad(N, enc_a(l), batch, N->gB[l])) return r;
        if (l > 0) {
            e.out0 = N->gA[l];
            e.mask0 = N->act[down(l - 1)];
            if (int r = dx_conv(N, enc_a(l), batch, N->gB[l], e)) return r;
        }
    }
    return WEC_OK;
}

int net_alloc(wec_net *N, void **p, size_t bytes)
{
    cudaError_t e = cudaMalloc(p, std::max<size_t>(bytes, 256));
    if (e != cudaSuccess) return cuda_fail(e, "net: device allocation");
    N->allocs.push_back(*p);
    return WEC_OK;
}

void net_free(wec_net *N)
{
    if (!N) return;
    if (N->st) cudaStreamSynchronize(N->st);
    for (void *p : N->allocs) cudaFree(p);
    if (N->lossh) cudaFreeHost(N->lossh);
    delete N;
}

}  // namespace

size_t net_param_count()
{
    size_t n = 0;
    for (int L = 0; L < kNumLayers; ++L) n += weight_count(L) + kLayers[L].co;
    return n;
}

int net_sync_weights(wec_net *N)
{
    if (!N->wdirty) return WEC_OK;
    if (int r = pack_weights(N)) return r;
    WEC_CK(cudaStreamSynchronize(N->st));
    return WEC_OK;
}

// Enqueue the net's guess for the tank's increment phi (step front, after the
// pressure problem is built).
int net_enqueue_guess(wec_tank *T, cudaStream_t st)
{
    wec_net *N = T->net;
    if (N->wdirty) return fail(WEC_ERR_INVALID, "net guess: BF16 weights not packed");
    const int nx = T->P.nx, ny = T->P.ny, nc = nx * ny;
    const double *bu = T->solver.L64[0].bu, *bv = T->solver.L64[0].bv;
    cudaStream_t keep = N->st;
    N->st = st;
    {
        WEC_PROF("net_features", -1, 8.0 * nc, st);
        WEC_CK(launch_k(k_feat_bsum, kRedBlocks, kT, 0, st, (const double *)T->rhs, nc, N->dpart));
    }
    {
        WEC_PROF("net_features", -1, 8.0 * nc * 4 + 8.0 * nc, st);
        WEC_CK(launch_k(k_features, nblk(nc, kT), kT, 0, st, nx, ny, (const double *)T->rhs, bu, bv,
                        (const double *)T->inp, T->P.rho_w, (const double *)N->dpart, kRedBlocks,
                        (const double *)nullptr, N->xb, (float *)nullptr));
    }
    int r = forward(N, 1, N->xb, N->out, nullptr);
    N->st = keep;
    if (r) return r;
    {
        WEC_PROF("net_guess", -1, 8.0 * nc * 4 + 4.0 * nc, st);
        WEC_CK(launch_k(k_guess, nblk(nc, kT), kT, 0, st, nx, ny, (const double *)T->rhs, bu, bv,
                        (const double *)N->dpart, kRedBlocks, (const float *)N->out, T->phi));
    }
    {
        WEC_PROF("net_guess", -1, 8.0 * nc * 5, st);
        WEC_CK(launch_k(k_guess_resid, kRedBlocks, kT, 0, st, nx, ny, (const double *)T->rhs, bu, bv,
                        (const double *)T->phi, N->dpart + kRedBlocks));
    }
    {
        WEC_PROF("net_guess", -1, 8.0 * nc, st);
        WEC_CK(launch_k(k_guess_select, nblk(nc, kT), kT, 0, st, nc, (const double *)N->dpart,
                        (const double *)(N->dpart + kRedBlocks), kRedBlocks, T->phi, T->net_stats));
    }
    return WEC_OK;
}

}  // namespace wec

using namespace wec;

extern "C" {

size_t wec_net_param_count(void) { return net_param_count(); }

int wec_net_create(int H, int W, int max_batch, void *cuda_stream, wec_net **out)
{
    if (!out) return fail(WEC_ERR_INVALID, "net_create: out is NULL");
    *out = nullptr;
    if (H < 8 || W < 8 || H % 8 || W % 8 || max_batch < 1)
        return fail(WEC_ERR_INVALID, "net_create: H, W must be multiples of 8 (>= 8) and max_batch >= 1");
    if ((long long)H * W * max_batch > (1LL << 26))
        return fail(WEC_ERR_INVALID, "net_create: max_batch * H * W above 2^26 pixels");
    wec_net *N = new (std::nothrow) wec_net();
    if (!N) return fail(WEC_ERR_NOMEM, "net_create: host allocation failed");
    N->H = H;
    N->W = W;
    N->maxb = max_batch;
    N->st = (cudaStream_t)cuda_stream;
    N->nparam = net_param_count();
    size_t nw = 0, off = 0;
    for (int L = 0; L < kNumLayers; ++L) {
        N->flat[L] = off;
        off += weight_count(L) + kLayers[L].co;
        if (L == kHead) break;
        const LayerDef &d = kLayers[L];
        if (d.kind == L_DOWN2) {
            N->wb[L] = nw;
            nw = round_up_z(nw + weight_count(L), 64);
        }
        if (halo_fwd(L)) {
            N->bnf[L] = rows_bn(N, halo_mode(d.kind), d.level, cin_pad(d.ci), d.co);
            if (!N->bnf[L]) N->bnf[L] = halo_bn(N, d.level, d.co, d.kind == L_UP3);
            N->hf[L] = nw;
            nw = round_up_z(nw + (size_t)taps(d.kind) * halo_kin(L, false) * d.co, 64);
        }
        if (halo_bwd(L)) {
            N->bnb[L] = rows_bn(N, H_CONV3, d.level, d.co, d.ci, d.kind == L_UP3);
            if (!N->bnb[L]) N->bnb[L] = halo_bn(N, d.level, d.ci);
            N->hb[L] = nw;
            nw = round_up_z(nw + 9 * (size_t)halo_kin(L, true) * d.ci, 64);
        }
    }
    const size_t P0 = (size_t)max_batch * H * W;
    auto pix = [&](int l) { return P0 >> (2 * l); };
    size_t part_n = 0;
    for (int L = 0; L < kHead; ++L) {
        // (a smaller batch may round to more splits than the largest, never above the cap)
        const int s = wgrad_max_splits(wgrad_units(N, L, (long long)max_batch * level_h(N, kLayers[L].level)), L);
        part_n = std::max(part_n, (size_t)s * round_up(fwd_K(L), kBM) * kLayers[L].co);
    }
    int r = WEC_OK;
    auto A = [&](void **p, size_t bytes) {
        if (!r) r = net_alloc(N, p, bytes);
    };
    A((void **)&N->theta, 4 * N->nparam);
    A((void **)&N->grad, 4 * N->nparam);
    A((void **)&N->am, 4 * N->nparam);
    A((void **)&N->av, 4 * N->nparam);
    A((void **)&N->wmat, 2 * nw);
    A((void **)&N->xin, 2 * P0 * kInPad);
    for (int L = 0; L < kHead; ++L) A((void **)&N->act[L], 2 * pix(kLayers[L].level) * kLayers[L].co);
    A((void **)&N->out, 4 * P0);
    for (int l = 0; l < 4; ++l) {
        A((void **)&N->gA[l], 2 * pix(l) * chans(l));
        A((void **)&N->gB[l], 2 * pix(l) * chans(l));
        if (l < 3) A((void **)&N->skip[l], 2 * pix(l) * chans(l));
    }
    A((void **)&N->part, 4 * part_n);
    A((void **)&N->cpart, 4 * (size_t)std::max(kCsumBlocks * 8, nblk((long long)P0, kT) * kHeadVals));
    A((void **)&N->xb, 4 * P0 * kInCh);
    A((void **)&N->tb, 4 * P0);
    A((void **)&N->loss, 8);
    A((void **)&N->dpart, 8 * 2 * kRedBlocks);
    A((void **)&N->err, sizeof(int));
    N->part_n = part_n;
    if (!r) {
        cudaError_t ce = cudaMallocHost((void **)&N->lossh, 8);
        if (ce != cudaSuccess) r = cuda_fail(ce, "net_create: pinned allocation");
    }
    if (!r) {
        cudaError_t ce = cudaMemsetAsync(N->theta, 0, 4 * N->nparam, N->st);
        if (ce == cudaSuccess) ce = cudaMemsetAsync(N->grad, 0, 4 * N->nparam, N->st);
        if (ce == cudaSuccess) ce = cudaMemsetAsync(N->am, 0, 4 * N->nparam, N->st);
        if (ce == cudaSuccess) ce = cudaMemsetAsync(N->av, 0, 4 * N->nparam, N->st);
        if (ce == cudaSuccess) ce = cudaMemsetAsync(N->err, 0, sizeof(int), N->st);
        if (ce == cudaSuccess) ce = cudaStreamSynchronize(N->st);
        if (ce != cudaSuccess) r = cuda_fail(ce, "net_create: initialisation");
    }
    if (r) {
        net_free(N);
        return r;
    }
    *out = N;
    return WEC_OK;
}

void wec_net_destroy(wec_net *N) { net_free(N); }

int wec_net_set_params(wec_net *N, const float *host, size_t n)
{
    if (!N || !host) return fail(WEC_ERR_INVALID, "net_set_params: NULL argument");
    if (n != N->nparam) return fail(WEC_ERR_INVALID, "net_set_params: n must equal wec_net_param_count()");
    for (size_t k = 0; k < n; ++k)
        if (!std::isfinite(host[k])) return fail(WEC_ERR_INVALID, "net_set_params: non-finite parameter");
    WEC_CK(cudaMemcpyAsync(N->theta, host, 4 * n, cudaMemcpyHostToDevice, N->st));
    WEC_CK(cudaMemsetAsync(N->am, 0, 4 * n, N->st));
    WEC_CK(cudaMemsetAsync(N->av, 0, 4 * n, N->st));
    WEC_CK(cudaStreamSynchronize(N->st));
    N->adam_t = 0;
    N->wdirty = true;
    return WEC_OK;
}

// After a synchronising call: a tensor-core pipeline wait that expired is an error.
static int check_pipeline(wec_net *N, const char *what)
{
    int h = 0;
    WEC_CK(cudaMemcpy(&h, N->err, sizeof(int), cudaMemcpyDeviceToHost));
    if (!h) return WEC_OK;
    WEC_CK(cudaMemset(N->err, 0, sizeof(int)));
    return fail(WEC_ERR_CUDA, std::string(what) + ": a tensor-core pipeline wait expired");
}

static int copy_out(const wec_net *N, const float *src, float *host, size_t n, const char *what)
{
    if (!N || !host) return fail(WEC_ERR_INVALID, std::string(what) + ": NULL argument");
    if (n != N->nparam) return fail(WEC_ERR_INVALID, std::string(what) + ": n must equal wec_net_param_count()");
    WEC_CK(cudaMemcpyAsync(host, src, 4 * n, cudaMemcpyDeviceToHost, N->st));
    WEC_CK(cudaStreamSynchronize(N->st));
    return WEC_OK;
}

int wec_net_get_params(const wec_net *N, float *host, size_t n)
{
    return copy_out(N, N ? N->theta : nullptr, host, n, "net_get_params");
}

int wec_net_get_grads(const wec_net *N, float *host, size_t n)
{
    return copy_out(N, N ? N->grad : nullptr, host, n, "net_get_grads");
}

int wec_net_get_activation(const wec_net *N, int layer, int batch, unsigned short *host, size_t n)
{
    if (!N || !host) return fail(WEC_ERR_INVALID, "net_get_activation: NULL argument");
    if (layer < 0 || layer >= kHead || batch < 1 || batch > N->maxb)
        return fail(WEC_ERR_INVALID, "net_get_activation: layer outside [0, 19] or batch outside [1, max_batch]");
    const LayerDef &d = kLayers[layer];
    const size_t want = (size_t)batch * level_h(N, d.level) * level_w(N, d.level) * d.co;
    if (n != want) return fail(WEC_ERR_INVALID, "net_get_activation: n does not match the layer's tensor");
    WEC_CK(cudaMemcpyAsync(host, N->act[layer], 2 * n, cudaMemcpyDeviceToHost, N->st));
    WEC_CK(cudaStreamSynchronize(N->st));
    return WEC_OK;
}

int wec_net_forward(wec_net *N, int batch, const float *x, float *out)
{
    if (!N || !x || !out) return fail(WEC_ERR_INVALID, "net_forward: NULL argument");
    if (batch < 1 || batch > N->maxb) return fail(WEC_ERR_INVALID, "net_forward: batch outside [1, max_batch]");
    if (int r = forward(N, batch, x, out, nullptr)) return r;
    WEC_CK(cudaStreamSynchronize(N->st));
    return check_pipeline(N, "net_forward");
}

int wec_net_loss_grad(wec_net *N, int batch, const float *x, const float *target, double *loss)
{
    if (!N || !x || !target || !loss) return fail(WEC_ERR_INVALID, "net_loss_grad: NULL argument");
    if (batch < 1 || batch > N->maxb) return fail(WEC_ERR_INVALID, "net_loss_grad: batch outside [1, max_batch]");
    if (int r = forward(N, batch, x, N->out, target)) return r;
    if (int r = backward(N, batch)) return r;
    WEC_CK(cudaMemcpyAsync(N->lossh, N->loss, 8, cudaMemcpyDeviceToHost, N->st));
    WEC_CK(cudaStreamSynchronize(N->st));
    if (int r = check_pipeline(N, "net_loss_grad")) return r;
    *loss = *N->lossh;
    return std::isfinite(*loss) ? WEC_OK : fail(WEC_ERR_NONFINITE, "net_loss_grad: non-finite loss");
}

int wec_net_adam(wec_net *N, float lr)
{
    if (!N) return fail(WEC_ERR_INVALID, "net_adam: NULL net");
    if (!(lr > 0.0f) || !std::isfinite(lr)) return fail(WEC_ERR_INVALID, "net_adam: lr must be finite and > 0");
    N->adam_t += 1;
    const float b1t = (float)(1.0 - std::pow(0.9, (double)N->adam_t));
    const float b2t = (float)(1.0 - std::pow(0.999, (double)N->adam_t));
    {
        WEC_PROF("net_adam", -1, 4.0 * 7 * N->nparam, N->st);
        WEC_CK(launch_k(k_adam, nblk((long long)N->nparam, kT), kT, 0, N->st, N->theta, (const float *)N->grad, N->am,
                        N->av, (long long)N->nparam, lr, b1t, b2t));
    }
    N->wdirty = true;
    return WEC_OK;
}

int wec_net_train_step(wec_net *N, const float *xs, const float *ts, const int *idx, int batch, float lr,
                       double *loss)
{
    if (!N || !xs || !ts || !idx || !loss) return fail(WEC_ERR_INVALID, "net_train_step: NULL argument");
    if (batch < 1 || batch > N->maxb) return fail(WEC_ERR_INVALID, "net_train_step: batch outside [1, max_batch]");
    const size_t px = (size_t)N->H * N->W;
    for (int b = 0; b < batch; ++b) {
        if (idx[b] < 0) return fail(WEC_ERR_INVALID, "net_train_step: negative sample index");
        WEC_CK(cudaMemcpyAsync(N->xb + b * px * kInCh, xs + (size_t)idx[b] * px * kInCh, 4 * px * kInCh,
                               cudaMemcpyDeviceToDevice, N->st));
        WEC_CK(cudaMemcpyAsync(N->tb + b * px, ts + (size_t)idx[b] * px, 4 * px, cudaMemcpyDeviceToDevice, N->st));
    }
    if (int r = wec_net_loss_grad(N, batch, N->xb, N->tb, loss)) return r;
    return wec_net_adam(N, lr);
}

int wec_net_sample(wec_tank *T, float *x, float *t)
{
    if (!T || !x || !t) return fail(WEC_ERR_INVALID, "net_sample: NULL argument");
    if (!T->stepped) return fail(WEC_ERR_INVALID, "net_sample: the tank has not stepped yet");
    const int nx = T->P.nx, ny = T->P.ny, nc = nx * ny;
    cudaStream_t st = T->gst;
    {
        WEC_PROF("net_features", -1, 8.0 * nc, st);
        WEC_CK(launch_k(k_feat_bsum, kRedBlocks, kT, 0, st, (const double *)T->rhs, nc, T->part));
    }
    {
        WEC_PROF("net_features", -1, 8.0 * nc * 6 + 12.0 * nc, st);
        WEC_CK(launch_k(k_features, nblk(nc, kT), kT, 0, st, nx, ny, (const double *)T->rhs,
                        (const double *)T->solver.L64[0].bu, (const double *)T->solver.L64[0].bv,
                        (const double *)T->inp, T->P.rho_w, (const double *)T->part, kRedBlocks,
                        (const double *)T->phi, x, t));
    }
    WEC_CK(cudaStreamSynchronize(st));
    return WEC_OK;
}

int wec_tank_set_net(wec_tank *T, wec_net *N)
{
    if (!T) return fail(WEC_ERR_INVALID, "tank_set_net: NULL tank");
    if (N && (N->H != T->P.ny || N->W != T->P.nx))
        return fail(WEC_ERR_INVALID, "tank_set_net: the net's H x W must be the tank's ny x nx");
    if (!T->inp_owned) return fail(WEC_ERR_INVALID, "tank_set_net: tanks of a batch take no net");
    if (N)
        if (int r = net_sync_weights(N)) return r;
    if (!T->net_stats) {
        WEC_CK(cudaMalloc(&T->net_stats, 2 * sizeof(long long)));
        WEC_CK(cudaMemsetAsync(T->net_stats, 0, 2 * sizeof(long long), T->gst));
        WEC_CK(cudaStreamSynchronize(T->gst));
    }
    WEC_CK(cudaStreamSynchronize(T->gst));
    if (T->exec) cudaGraphExecDestroy(T->exec);
    if (T->graph) cudaGraphDestroy(T->graph);
    T->exec = nullptr;
    T->graph = nullptr;
    T->net = N;
    return WEC_OK;
}

int wec_tank_net_stats(const wec_tank *T, long long *tried, long long *kept)
{
    if (!T || !tried || !kept) return fail(WEC_ERR_INVALID, "tank_net_stats: NULL argument");
    long long h[2] = {0, 0};
    if (T->net_stats) {
        WEC_CK(cudaMemcpyAsync(h, T->net_stats, sizeof(h), cudaMemcpyDeviceToHost, T->gst));
        WEC_CK(cudaStreamSynchronize(T->gst));
    }
    *tried = h[0];
    *kept = h[1];
    return WEC_OK;
}

}  // extern "C"
