// cnn.cu -- learned localiser: a 4-layer 3x3 convolutional network mapping a
// projection plane (XDoppler amplitude / frame maximum) to a microbubble
// heatmap on a 4x finer grid, with BF16 tensor-core forward, input-gradient
// and weight-gradient kernels (FP32 accumulation), MSE loss, Adam on FP32
// master weights.  The paper names learned localisation as future work
// (Sec. IV); the network is the build's reading of that form.
//
//   L1 conv3x3(1 -> 32) + ReLU     FP32 CUDA cores (K = 9)
//   L2 conv3x3(32 -> 32) + ReLU    tcgen05 MMA (BF16, FP32 accumulators in TMEM)
//   L3 conv3x3(32 -> 32) + ReLU    idem
//   L4 conv3x3(32 -> 16)           idem, epilogue = pixel shuffle to 4x
// The forward pass is one kernel (cnn_stream.cuh).  The input gradients are
// tcgen05 convolutions with flipped weights (k_conv_tc); the weight gradients
// (M = COUT is below the tcgen05 minimum of 64) use mma.sync m16n8k16.
//
// Activations NHWC BF16; weights [Cout][9 taps][Cin] (tap = 3 (dy+1) + dx+1).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "rca_internal.cuh"

#define CNN_C 32
#define CNN_UP 4
#define CNN_LOSS_BLOCKS 1024
#define CONV_TH 8   // tile rows (one warp each)
#define CONV_TW 16  // tile columns (the 16 rows of one mma A fragment)

namespace {

struct ParamLayout {
    // offsets (floats) into the flat parameter vector
    int w[4], b[4], total;
};

inline ParamLayout param_layout()
{
    ParamLayout p;
    const int cin[4] = {1, CNN_C, CNN_C, CNN_C}, cout[4] = {CNN_C, CNN_C, CNN_C, CNN_UP * CNN_UP};
    int o = 0;
    for (int l = 0; l < 4; ++l) {
        p.w[l] = o;
        o += cout[l] * 9 * cin[l];
        p.b[l] = o;
        o += cout[l];
    }
    p.total = o;
    return p;
}

__device__ __forceinline__ unsigned pack_bf2(float a, float b)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<unsigned*>(&v);
}

__device__ __forceinline__ float2 unpack_bf2(unsigned u)
{
    return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}

__device__ __forceinline__ void mma_bf16(float c[4], const unsigned a[4], const unsigned b[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// ---------------------------------------------------------------------------
// Input gradient of a 3x3 layer on the 5th-generation tensor cores (tcgen05,
// TMEM): the convolution of the output gradient with the flipped weights, times
// (mask > 0) of the layer's BF16 NHWC input, BF16 NHWC out.
// A CTA of 128 threads owns a tile of 8 rows x 16 columns (M = 128 pixels,
// ordered column-major: pixel m = 8 x + y), so that one image column of the
// tile is one 8-row core matrix of the MMA's A operand.  The input tile with
// its one-pixel halo (10 x 18 pixels, CIN channels) sits in shared memory in
// the K-major, no-swizzle core-matrix layout
//   [CIN / 8][18 columns][10 rows][8 channels] (16-byte rows),
// so the A operand of tap (dy, dx) is the same array seen from start offset
// dx x 160 + dy x 16 bytes: a column step is 160 bytes (SBO) and an 8-channel
// step 18 x 160 bytes (LBO).  No im2col copy is made.  The weights of all nine
// taps (B operand, [9][CIN / 8][COUT / 8][8 outputs][8 channels]) are staged
// once per CTA.  One thread issues the 9 x CIN / 16 MMAs (M = 128, N = COUT,
// K = 16, BF16 in, FP32 accumulators in TMEM) and commits them to an
// mbarrier; each warp then reads its 32 pixels' rows of the accumulator with
// tcgen05.ld for the epilogue.
// ---------------------------------------------------------------------------
#define TC_HALO_C 18                        // tile columns + halo
#define TC_HALO_R 10                        // tile rows + halo
#define TC_CM_BYTES (TC_HALO_R * 16)        // one column of the halo tile: 10 rows x 16 bytes

__device__ __forceinline__ uint64_t tc_sdesc(unsigned saddr, unsigned lbo, unsigned sbo)
{
    // shared-memory matrix descriptor: start, leading (K) and stride (M/N) byte
    // offsets in 16-byte units, descriptor version 1, no swizzle
    return (uint64_t)((saddr >> 4) & 0x3fff) | ((uint64_t)((lbo >> 4) & 0x3fff) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3fff) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: D FP32, A and B BF16, both K-major
__host__ __device__ constexpr unsigned tc_idesc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(unsigned tmem_d, uint64_t da, uint64_t db, unsigned idesc, int accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
        : "memory");
}

// one lane of a converged warp
__device__ __forceinline__ bool elect_one()
{
    unsigned p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

template <int NC>
__device__ __forceinline__ void tc_ld(unsigned taddr, float* v);
template <>
__device__ __forceinline__ void tc_ld<16>(unsigned taddr, float* v)
{
    unsigned r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = __uint_as_float(r[q]);
}
template <>
__device__ __forceinline__ void tc_ld<32>(unsigned taddr, float* v)
{
    unsigned r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
          "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
          "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 32; ++q) v[q] = __uint_as_float(r[q]);
}

#include "cnn_stream.cuh"

template <int CIN, int COUT>
__global__ void __launch_bounds__(128) k_conv_tc(const __nv_bfloat16* __restrict__ x,
                                                 const __nv_bfloat16* __restrict__ wt,
                                                 const __nv_bfloat16* __restrict__ mask, int B, int H, int W,
                                                 __nv_bfloat16* __restrict__ out, unsigned* __restrict__ status)
{
    grid_wait();
    static_assert(CIN % 16 == 0 && COUT % 16 == 0 && COUT <= 32, "shapes of the 3x3 layers");
    constexpr int KC = CIN / 8, NG = COUT / 8;
    constexpr int TAPB = KC * NG * 128;                 // bytes of one tap's weights
    constexpr int ABYTES = KC * TC_HALO_C * TC_CM_BYTES;
    constexpr unsigned IDESC = tc_idesc(128, COUT);
    constexpr unsigned TMEM_COLS = 64;                  // two 32-column accumulators
    extern __shared__ __align__(16) unsigned char smtc[];
    unsigned char* sB = smtc;                           // [9][KC][NG][8][8] bf16
    unsigned char* sA = smtc + 9 * TAPB;                // [3][KC][18][10][8] bf16
    __shared__ uint64_t bars[2];
    __shared__ unsigned s_tmem;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // weights: element (o, t, c) of [COUT][9][CIN] -> tap t, core (c / 8, o / 8), row o % 8, column c % 8
    for (int q = threadIdx.x; q < COUT * 9 * KC; q += blockDim.x) {
        const int o = q / (9 * KC), r = q % (9 * KC), t = r / KC, kc = r % KC;
        const uint4 v = reinterpret_cast<const uint4*>(wt)[q];   // 8 channels kc*8 .. of (o, t)
        *reinterpret_cast<uint4*>(sB + t * TAPB + (kc * NG + o / 8) * 128 + (o % 8) * 16) = v;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        mbar_fence_init();
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = s_tmem;
    const unsigned sAa = smem_u32(sA), sBa = smem_u32(sB);
    const int tiles_i = (H + CONV_TH - 1) / CONV_TH, tiles_j = (W + CONV_TW - 1) / CONV_TW;
    const int ntiles = B * tiles_i * tiles_j;
    auto coords = [&](int tile, int& b, int& i0, int& j0) {
        b = tile / (tiles_i * tiles_j);
        const int tij = tile % (tiles_i * tiles_j);
        i0 = (tij / tiles_j) * CONV_TH;
        j0 = (tij % tiles_j) * CONV_TW;
    };
    // halo tile of `tile` into buffer `buf` by 16-byte cp.async copies (zero-filled
    // outside the plane), one commit group per call (empty when tile >= ntiles):
    // 8-channel chunk kc of pixel (row yr, column xg)
    auto load = [&](int tile, int buf) {
        if (tile < ntiles) {
            int b, i0, j0;
            coords(tile, b, i0, j0);
            const unsigned dst = sAa + (unsigned)(buf * ABYTES);
            for (int q = threadIdx.x; q < TC_HALO_R * TC_HALO_C * KC; q += blockDim.x) {
                const int kc = q % KC, p = q / KC, xg = p % TC_HALO_C, yr = p / TC_HALO_C;
                const int ii = i0 - 1 + yr, jj = j0 - 1 + xg;
                const bool in = ii >= 0 && ii < H && jj >= 0 && jj < W;
                const void* src = in ? (const void*)(x + (((size_t)b * H + ii) * W + jj) * CIN + kc * 8) : (const void*)x;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                                 dst + (unsigned)((kc * TC_HALO_C + xg) * TC_CM_BYTES + yr * 16)),
                             "l"(src), "r"(in ? 16u : 0u)
                             : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // this thread's copies of every group but the newest are done; then the
    // generic-proxy writes are ordered before the tensor cores read the tile
    auto wait_older = [&]() {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        fence_proxy_async();
    };
    // the 9 x CIN / 16 MMAs of halo buffer `ab` into accumulator `buf` (one thread)
    auto issue = [&](int ab, int buf) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const unsigned aB = sAa + ab * ABYTES, dcol = tmem + (unsigned)(32 * buf);
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int dy = t / 3, dx = t % 3;
#pragma unroll
            for (int kk = 0; kk < CIN / 16; ++kk) {
                const uint64_t da = tc_sdesc(aB + (2 * kk * TC_HALO_C + dx) * TC_CM_BYTES + dy * 16,
                                             TC_HALO_C * TC_CM_BYTES, TC_CM_BYTES);
                const uint64_t db = tc_sdesc(sBa + t * TAPB + 2 * kk * NG * 128, NG * 128, 128);
                tc_mma(dcol, da, db, IDESC, (t | kk) != 0);
            }
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         smem_u32(&bars[buf]))
                     : "memory");
    };
    // software pipeline over three halo buffers and two accumulators: the copies
    // of tile k + 2 and the MMAs of tile k + 1 run while tile k's epilogue drains
    unsigned phase = 0;   // bit b: parity of the next completion of bars[b]
    bool ok = true;
    int tile = blockIdx.x;
    load(tile, 0);
    load(tile + gridDim.x, 1);
    if (tile < ntiles) {
        wait_older();
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (threadIdx.x == 0) issue(0, 0);
    }
    for (int k = 0; tile < ntiles; ++k, tile += gridDim.x) {
        const int cur = k & 1, nxt = cur ^ 1;
        const int ntile = tile + gridDim.x;
        // buffer (k + 2) mod 3 held tile k - 1, whose MMAs completed before its epilogue
        load(ntile + gridDim.x, (k + 2) % 3);
        wait_older();
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (ntile < ntiles && threadIdx.x == 0) issue((k + 1) % 3, nxt);
        // bounded wait for tile k's accumulators
        if (!mbar_wait_bounded(&bars[cur], (phase >> cur) & 1u)) ok = false;
        if (__syncthreads_or(!ok)) {
            if (threadIdx.x == 0) atomicOr(status, ST_TIMEOUT);
            // the MMAs in flight finish (bounded) before the accumulators are freed
            mbar_wait_bounded(&bars[cur], (phase >> cur) & 1u);
            if (ntile < ntiles) mbar_wait_bounded(&bars[nxt], (phase >> nxt) & 1u);
            asm volatile("cp.async.wait_all;" ::: "memory");
            break;
        }
        phase ^= 1u << cur;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        int b, i0, j0;
        coords(tile, b, i0, j0);
        // epilogue: warp w reads TMEM lanes 32 w .. 32 w + 31 = pixels m of the tile
        float v[COUT];
        tc_ld<COUT>(tmem + ((unsigned)(32 * warp) << 16) + (unsigned)(32 * cur), v);
        const int m = 32 * warp + lane;
        const int i = i0 + (m & 7), j = j0 + (m >> 3);
        if (i < H && j < W) {
            const size_t pix = ((size_t)b * H + i) * W + j;
            const unsigned* mk = reinterpret_cast<const unsigned*>(mask) + pix * (COUT / 2);
            unsigned pk[COUT / 2];
#pragma unroll
            for (int o = 0; o < COUT; o += 2) {
                const float2 mm = unpack_bf2(mk[o / 2]);
                pk[o / 2] = pack_bf2(mm.x > 0.f ? v[o] : 0.f, mm.y > 0.f ? v[o + 1] : 0.f);
            }
#pragma unroll
            for (int q = 0; q < COUT / 8; ++q)
                reinterpret_cast<uint4*>(out)[pix * (COUT / 8) + q] =
                    make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
        }
        // every warp's reads of accumulator `cur` are done before MMAs write it again
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) {
        mbar_inval(&bars[0]);
        mbar_inval(&bars[1]);
    }
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// ---------------------------------------------------------------------------
// Weight gradient on tensor cores: dW[o][t][c] = sum_p dY[p][o] X[p + t][c],
// a GEMM with M = COUT, N = 9 x CIN and the reduction over pixels.  Each CTA
// accumulates its tiles in registers and writes one partial [COUT][9 CIN]
// (plus the bias partial) to scratch; k_reduce_grads adds the partials in a
// fixed order (deterministic).  Both operands are reduced over their slow
// index, so the tiles stay as they lie in memory (pixel-major, 16-byte cp.async
// copies, two buffers) and ldmatrix transposes them into the fragments; a tap is
// a shift of whole pixel rows.  One warp per tap; pixel rows are padded by 16
// bytes, which puts the eight rows of a matrix in different banks.  (With
// 2-byte transposing stores and gathers: 50 us for 64 planes of 80 x 32, 17 us here.)
// ---------------------------------------------------------------------------
#define WG_XS (CNN_C * 2 + 16)                          // bytes of one staged input pixel
#define WG_DS(COUT) ((COUT) * 2 + 16)                   // of one staged output-gradient pixel
#define WG_HALO ((CONV_TH + 2) * (CONV_TW + 2))
#define WG_BUF(COUT) (CONV_TH * CONV_TW * WG_DS(COUT) + WG_HALO * WG_XS)

__device__ __forceinline__ void ldsm_x4_trans(unsigned addr, unsigned r[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

__device__ __forceinline__ void cp_async16(unsigned dst, const void* src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16u : 0u) : "memory");
}

template <int COUT>
__global__ void __launch_bounds__(288, 3) k_wgrad_mma(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ dy,
                                                      int B, int H, int W, float* __restrict__ part)
{
    grid_wait();
    constexpr int MT = COUT / 16, DC = COUT / 8, DS = WG_DS(COUT), XOFF = CONV_TH * CONV_TW * DS, HW2 = CONV_TW + 2;
    constexpr int N = 9 * CNN_C;
    extern __shared__ __align__(16) unsigned char smraw[];   // [2][dY tile, X tile with halo]
    const int lane = threadIdx.x & 31, tap = threadIdx.x >> 5;
    const int g = lane >> 2, tig = lane & 3;
    const unsigned sm = smem_u32(smraw);
    float acc[MT][4][4], db[MT][2];
#pragma unroll
    for (int m = 0; m < MT; ++m) {
        db[m][0] = db[m][1] = 0.f;
#pragma unroll
        for (int n = 0; n < 4; ++n) acc[m][n][0] = acc[m][n][1] = acc[m][n][2] = acc[m][n][3] = 0.f;
    }
    const int tiles_i = (H + CONV_TH - 1) / CONV_TH, tiles_j = (W + CONV_TW - 1) / CONV_TW;
    const int ntiles = B * tiles_i * tiles_j;
    auto load = [&](int tile, int buf) {
        if (tile < ntiles) {
            const int b = tile / (tiles_i * tiles_j), tij = tile % (tiles_i * tiles_j);
            const int i0 = (tij / tiles_j) * CONV_TH, j0 = (tij % tiles_j) * CONV_TW;
            const unsigned dst = sm + (unsigned)(buf * WG_BUF(COUT));
            for (int q = threadIdx.x; q < CONV_TH * CONV_TW * DC; q += blockDim.x) {
                const int c = q % DC, p = q / DC, ii = i0 + p / CONV_TW, jj = j0 + p % CONV_TW;
                const bool in = ii < H && jj < W;
                cp_async16(dst + p * DS + c * 16, in ? dy + (((size_t)b * H + ii) * W + jj) * COUT + c * 8 : dy, in);
            }
            for (int q = threadIdx.x; q < WG_HALO * (CNN_C / 8); q += blockDim.x) {
                const int c = q % (CNN_C / 8), p = q / (CNN_C / 8), ii = i0 - 1 + p / HW2, jj = j0 - 1 + p % HW2;
                const bool in = ii >= 0 && ii < H && jj >= 0 && jj < W;
                cp_async16(dst + XOFF + p * WG_XS + c * 16, in ? x + (((size_t)b * H + ii) * W + jj) * CNN_C + c * 8 : x, in);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // fragment addresses of this lane: dY (pixel, 8-output chunk) and X (pixel, 8-channel chunk)
    const unsigned la = (unsigned)(((lane >> 4) * 8 + (lane & 7)) * DS + (lane >> 3 & 1) * 16);
    const unsigned lb = (unsigned)(XOFF + ((tap / 3) * HW2 + tap % 3 + (lane >> 3 & 1) * 8 + (lane & 7)) * WG_XS +
                                   (lane >> 4) * 16);
    int buf = 0;
    load(blockIdx.x, 0);
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, buf ^= 1) {
        load(tile + gridDim.x, buf ^ 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        const unsigned base = sm + (unsigned)(buf * WG_BUF(COUT));
#pragma unroll 2
        for (int rr = 0; rr < CONV_TH; ++rr) {                 // k-steps: the 16 pixels of a tile row
            unsigned a[MT][4], bb[2][4];
#pragma unroll
            for (int m = 0; m < MT; ++m) ldsm_x4_trans(base + la + rr * CONV_TW * DS + m * 32, a[m]);
#pragma unroll
            for (int j = 0; j < 2; ++j) ldsm_x4_trans(base + lb + rr * HW2 * WG_XS + j * 32, bb[j]);
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int n = 0; n < 4; ++n) mma_bf16(acc[m][n], a[m], bb[n >> 1] + 2 * (n & 1));
            if (tap == 0) {
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float2 v = unpack_bf2(a[m][q]);
                        db[m][q & 1] += v.x + v.y;
                    }
            }
        }
        __syncthreads();                                       // the buffer is filled again two tiles on
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    // partial of this CTA: rows (o) g, g + 8 of each m-tile, columns tap * 32 + n * 8 + 2 tig (+1)
    float* dst = part + (size_t)blockIdx.x * (COUT * N + COUT);
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int o = m * 16 + g + 8 * h;
#pragma unroll
            for (int n = 0; n < 4; ++n)
                *reinterpret_cast<float2*>(dst + o * N + tap * CNN_C + n * 8 + 2 * tig) =
                    make_float2(acc[m][n][2 * h], acc[m][n][2 * h + 1]);
            float s = db[m][h];
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (tap == 0 && tig == 0) dst[COUT * N + o] = s;
        }
}

// L1 weight gradient (CIN = 1), FP32: per-CTA partials of dW1[o][t], db1[o].  A
// warp walks one plane row, its lanes being the 32 output channels: one 64-byte
// load of the output gradient and three broadcast loads of the input per pixel
// feed ten sums in registers.  (With a thread per (o, t) and one pixel at a
// time: 288 us for 64 planes of 80 x 32, 14 us here.)
__global__ void __launch_bounds__(256) k_wgrad1(const float* __restrict__ x, const __nv_bfloat16* __restrict__ dy, int rows,
                                                int H, int W, float* __restrict__ part)
{
    grid_wait();
    __shared__ float red[8][CNN_C * 10];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float s[10];
#pragma unroll
    for (int t = 0; t < 10; ++t) s[t] = 0.f;
    for (int r = blockIdx.x * 8 + warp; r < rows; r += gridDim.x * 8) {
        const int i = r % H;
        const float* xr = x + (size_t)r * W;
        const __nv_bfloat16* dr = dy + (size_t)r * W * CNN_C + lane;
        const bool up = i > 0, dn = i + 1 < H;
        float v[3][3];                                         // [row][column j - 1, j, j + 1]
#pragma unroll
        for (int q = 0; q < 3; ++q) v[q][0] = v[q][1] = 0.f;
        v[0][2] = up ? xr[-W] : 0.f, v[1][2] = xr[0], v[2][2] = dn ? xr[W] : 0.f;
#pragma unroll 4
        for (int j = 0; j < W; ++j) {
            const bool in = j + 1 < W;
#pragma unroll
            for (int q = 0; q < 3; ++q) v[q][0] = v[q][1], v[q][1] = v[q][2];
            v[0][2] = up && in ? xr[j + 1 - W] : 0.f;
            v[1][2] = in ? xr[j + 1] : 0.f;
            v[2][2] = dn && in ? xr[j + 1 + W] : 0.f;
            const float d = __bfloat162float(dr[(size_t)j * CNN_C]);
#pragma unroll
            for (int t = 0; t < 9; ++t) s[t] = fmaf(d, v[t / 3][t % 3], s[t]);
            s[9] += d;
        }
    }
#pragma unroll
    for (int t = 0; t < 10; ++t) red[warp][t < 9 ? lane * 9 + t : CNN_C * 9 + lane] = s[t];
    __syncthreads();
    for (int k = threadIdx.x; k < CNN_C * 10; k += 256) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) t += red[w][k];
        part[(size_t)blockIdx.x * (CNN_C * 10) + k] = t;
    }
}

// Sums of the CTAs' partials in a fixed order: every layer's gradients and the
// loss in one launch.  A block adds 32 columns, eight warps taking every
// eighth partial, so that a column's loads are not one serial chain (four launches
// of one thread per column, 608 partials: 157 us; 456 partials here: 10 us).
struct GradSums {
    const float* part[5];
    int nparts[5], len[5], block0[6];   // layers 1..4, then the loss (one column); first block of each
    float* out[5];
    float scale[5];
};

__global__ void __launch_bounds__(256) k_reduce_grads(const GradSums g)
{
    grid_wait();
    __shared__ float red[8][32];
    int seg = 0;
    while (seg < 4 && (int)blockIdx.x >= g.block0[seg + 1]) ++seg;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int len = g.len[seg], np = g.nparts[seg], k = ((int)blockIdx.x - g.block0[seg]) * 32 + lane;
    const float* p = g.part[seg];
    float s = 0.f;
    if (seg == 4) {                                            // one column: spread its partials over the block
        for (int c = threadIdx.x; c < np; c += 256) s += p[c];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    } else if (k < len) {
#pragma unroll 8
        for (int c = warp; c < np; c += 8) s += p[(size_t)c * len + k];
    }
    red[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && k < len) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) t += red[w][lane];
        g.out[seg][k] = t * g.scale[seg];
    }
}

// MSE loss: per-CTA partial sums of (heat - target)^2 and dZ4 (un-shuffled
// 2 (heat - target) / n, BF16 NHWC with 16 channels).  A thread owns one plane
// pixel: four 16-byte runs of the heatmap and of the target, one 32-byte gradient
// (element by element with its divisions: 18 us for 64 planes of 80 x 32, 6 us here).
template <bool ALIGNED>
__global__ void __launch_bounds__(256) k_loss(const float* __restrict__ heat, const float* __restrict__ target, int rows,
                                              int W, float scale, __nv_bfloat16* __restrict__ dz, float* __restrict__ part)
{
    grid_wait();
    __shared__ float red[8];
    const unsigned np = (unsigned)rows * W;                    // within the network's capacity, an int
    float s = 0.f;
    for (unsigned p = blockIdx.x * 256 + threadIdx.x; p < np; p += gridDim.x * 256) {
        const unsigned r = p / W, j = p - r * W;
        const size_t at = ((size_t)r * CNN_UP * W + j) * CNN_UP;
        float4 h[CNN_UP], t[CNN_UP];
#pragma unroll
        for (int a = 0; a < CNN_UP; ++a) {
            const size_t q = at + (size_t)a * W * CNN_UP;
            h[a] = __ldg(reinterpret_cast<const float4*>(heat + q));
            t[a] = ALIGNED ? __ldg(reinterpret_cast<const float4*>(target + q))
                           : make_float4(target[q], target[q + 1], target[q + 2], target[q + 3]);
        }
        unsigned pk[2 * CNN_UP];
#pragma unroll
        for (int a = 0; a < CNN_UP; ++a) {
            const float d0 = h[a].x - t[a].x, d1 = h[a].y - t[a].y, d2 = h[a].z - t[a].z, d3 = h[a].w - t[a].w;
            s = fmaf(d0, d0, s), s = fmaf(d1, d1, s), s = fmaf(d2, d2, s), s = fmaf(d3, d3, s);
            pk[2 * a] = pack_bf2(d0 * scale, d1 * scale);
            pk[2 * a + 1] = pack_bf2(d2 * scale, d3 * scale);
        }
        uint4* o = reinterpret_cast<uint4*>(dz + (size_t)p * (CNN_UP * CNN_UP));
        o[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        o[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < 8; ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}

// Adam on the FP32 masters (bias-corrected step sizes computed on the host),
// then the BF16 copies of the updated weights (as k_pack_weights)
struct PackedWeights {
    ParamLayout lay;
    __nv_bfloat16 *fwd[4], *flip[4];
};

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ gr, float* __restrict__ m, float* __restrict__ v,
                       const PackedWeights w, float lr_t, float b1, float b2, float eps_t)
{
    grid_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= w.lay.total) return;
    const float g = gr[i];
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    const float pn = p[i] - lr_t * mi / (sqrtf(vi) + eps_t);
    p[i] = pn;
#pragma unroll
    for (int l = 1; l < 4; ++l) {
        const int q = i - w.lay.w[l], O = l == 3 ? CNN_UP * CNN_UP : CNN_C;
        if (q < 0 || q >= O * 9 * CNN_C) continue;
        const int o = q / (9 * CNN_C), t = (q / CNN_C) % 9, c = q % CNN_C;
        const __nv_bfloat16 h = __float2bfloat16(pn);
        w.fwd[l][q] = h;
        w.flip[l][((size_t)c * 9 + (8 - t)) * O + o] = h;
    }
}

// BF16 copies of the weights: forward layout [O][9][I] and, for the input
// gradient, the transposed and tap-flipped [I][9][O] (tap 8 - t).
__global__ void k_pack_weights(const float* __restrict__ w, int O, int I, __nv_bfloat16* __restrict__ fwd,
                               __nv_bfloat16* __restrict__ flip)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= O * 9 * I) return;
    const int o = q / (9 * I), t = (q / I) % 9, c = q % I;
    const __nv_bfloat16 v = __float2bfloat16(w[q]);
    fwd[q] = v;
    if (flip) flip[((size_t)c * 9 + (8 - t)) * O + o] = v;
}

// Gaussian targets: target[b][y][x] = sum over the plane's points of
// exp(-((y - z4)^2 + (x - x4)^2) / (2 sigma^2)); pts [n][3] = (plane, z4, x4),
// grouped by plane with offsets off[B + 1].
__global__ void k_target(const float* __restrict__ pts, const int* __restrict__ off, int H4, int W4, float sigma,
                         float* __restrict__ target)
{
    const int b = blockIdx.y;
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= H4 * W4) return;
    const int y = q / W4, x = q % W4;
    const float inv = 1.f / (2.f * sigma * sigma);
    float s = 0.f;
    for (int k = off[b]; k < off[b + 1]; ++k) {
        const float dz = (float)y - pts[3 * k + 1], dx = (float)x - pts[3 * k + 2];
        s += __expf(-(dz * dz + dx * dx) * inv);
    }
    target[(size_t)b * H4 * W4 + q] = s;
}

__global__ void k_count_offsets(const float* __restrict__ pts, int n, int B, int* __restrict__ off)
{
    // off[b] = first point with plane >= b (points sorted by plane)
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b > B) return;
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if ((int)pts[3 * mid] < b) lo = mid + 1;
        else hi = mid;
    }
    off[b] = lo;
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct ulm_cnn {
    rca_handle* h = nullptr;
    ulm_cnn_desc desc{};
    ParamLayout lay{};
    float* params = nullptr;   // FP32 masters
    float* grads = nullptr;
    float* m = nullptr;
    float* v = nullptr;
    __nv_bfloat16* wbf[4] = {nullptr, nullptr, nullptr, nullptr};  // forward copies (layers 2..4)
    __nv_bfloat16* wfl[4] = {nullptr, nullptr, nullptr, nullptr};  // flipped copies (layers 2..4)
    long long step = 0;
    // activations for the largest batch
    size_t cap_px = 0;
    float* x0 = nullptr;
    __nv_bfloat16 *a1 = nullptr, *a2 = nullptr, *a3 = nullptr;
    __nv_bfloat16 *g1 = nullptr, *g2 = nullptr, *g3 = nullptr, *gz = nullptr;
    float* heat = nullptr;
    float* part = nullptr;  // scratch for per-CTA partials
    size_t part_len = 0;
    int sms = 0;
    int grid_conv_tc = 0;   // input-gradient CTAs: four per SM (64 TMEM columns each)
    int grid_wgrad = 0;     // weight-gradient CTAs, each with one partial: three per SM
};

static rca_status cnn_check_shape(ulm_cnn* c, int B, int H, int W)
{
    if (B <= 0 || H <= 0 || W <= 0) return set_error(c->h, RCA_ERR_SHAPE, "batch and plane sizes must be positive");
    if ((size_t)B * H * W > c->cap_px)
        return set_error(c->h, RCA_ERR_SHAPE, "batch of %d planes %dx%d exceeds the network's capacity (%zu pixels)", B, H, W,
                         c->cap_px);
    return RCA_OK;
}

static rca_status cnn_pack(ulm_cnn* c)
{
    const int cin[4] = {1, CNN_C, CNN_C, CNN_C}, cout[4] = {CNN_C, CNN_C, CNN_C, CNN_UP * CNN_UP};
    for (int l = 1; l < 4; ++l) {
        const int n = cout[l] * 9 * cin[l];
        k_pack_weights<<<(n + 255) / 256, 256, 0, c->h->stream>>>(c->params + c->lay.w[l], cout[l], cin[l], c->wbf[l],
                                                                c->wfl[l]);
    }
    return cuda_check(c->h, cudaGetLastError(), "cnn pack");
}

template <int CIN, int COUT>
static rca_status conv_launch(ulm_cnn* c, const __nv_bfloat16* x, const __nv_bfloat16* w, const __nv_bfloat16* mask,
                              int B, int H, int W, __nv_bfloat16* out)
{
    // weights of the nine taps + three halo tiles
    constexpr size_t smem = (size_t)9 * CIN * COUT * 2 + (size_t)3 * (CIN / 8) * TC_HALO_C * TC_CM_BYTES;
    static_assert(smem <= 100 * 1024, "conv tile exceeds its shared-memory budget");
    auto kern = k_conv_tc<CIN, COUT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_check(c->h, e, "conv smem attribute");
    const int ntiles = B * ((H + CONV_TH - 1) / CONV_TH) * ((W + CONV_TW - 1) / CONV_TW);
    const int grid = std::min(ntiles, c->grid_conv_tc);
    launch_chain(kern, dim3(grid), dim3(128), smem, c->h->stream, x, w, mask, B, H, W, out, c->h->d_status);
    return cuda_check(c->h, cudaGetLastError(), "conv kernel");
}

// weight gradient partials of layer l + 1 into their part of the scratch
template <int COUT>
static rca_status wgrad_launch(ulm_cnn* c, const __nv_bfloat16* x, const __nv_bfloat16* dy, int B, int H, int W, int l,
                               GradSums& sums, size_t& at)
{
    auto kern = k_wgrad_mma<COUT>;
    const int smem = 2 * WG_BUF(COUT);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return cuda_check(c->h, e, "wgrad smem attribute");
    const int ntiles = B * ((H + CONV_TH - 1) / CONV_TH) * ((W + CONV_TW - 1) / CONV_TW);
    sums.part[l] = c->part + at, sums.nparts[l] = std::min(ntiles, c->grid_wgrad), sums.len[l] = COUT * 9 * CNN_C + COUT;
    launch_chain(kern, dim3(sums.nparts[l]), dim3(288), smem, c->h->stream, x, dy, B, H, W, c->part + at);
    at += (size_t)c->grid_wgrad * sums.len[l];
    return cuda_check(c->h, cudaGetLastError(), "wgrad kernel");
}

// the four layers in one launch; KEEP: the activations the backward pass reads
template <bool KEEP>
static rca_status cnn_forward(ulm_cnn* c, const float* A, const float* M, int ppf, int B, int H, int W, float* heat)
{
    const int sms = c->sms;
    StreamArgs g{};
    g.A = A, g.M = M, g.ppf = ppf > 0 ? ppf : 1, g.B = B, g.H = H, g.W = W;
    g.plan = stream_plan(B, H, W, sms);
    g.w1 = c->params + c->lay.w[0], g.b1 = c->params + c->lay.b[0];
    g.w2 = c->wbf[1], g.w3 = c->wbf[2], g.w4 = c->wbf[3];
    g.b2 = c->params + c->lay.b[1], g.b3 = c->params + c->lay.b[2], g.b4 = c->params + c->lay.b[3];
    g.heat = heat, g.x0 = c->x0, g.a1 = c->a1, g.a2 = c->a2, g.a3 = c->a3, g.status = c->h->d_status;
    auto kern = k_cnn_stream<KEEP>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, StreamSmem::bytes);
    if (e != cudaSuccess) return cuda_check(c->h, e, "cnn smem attribute");
    launch_chain(kern, dim3(std::min(g.plan.nruns, sms)), dim3(ST_THREADS), StreamSmem::bytes, c->h->stream, g);
    return cuda_check(c->h, cudaGetLastError(), "cnn forward");
}

extern "C" rca_status ulm_cnn_create(rca_handle* h, const ulm_cnn_desc* d, ulm_cnn** out)
{
    if (!h) return RCA_ERR_INVALID_ARG;
    if (!d || !out) return set_error(h, RCA_ERR_INVALID_ARG, "null descriptor or output");
    *out = nullptr;
    if (d->channels != CNN_C) return set_error(h, RCA_ERR_UNSUPPORTED, "only %d channels are built", CNN_C);
    if (d->max_pixels <= 0) return set_error(h, RCA_ERR_INVALID_ARG, "max_pixels must be positive");
    ulm_cnn* c = new (std::nothrow) ulm_cnn();
    if (!c) return set_error(h, RCA_ERR_CUDA, "out of host memory");
    c->h = h;
    c->desc = *d;
    c->lay = param_layout();
    c->cap_px = (size_t)d->max_pixels;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    c->sms = sms;
    c->grid_conv_tc = 4 * sms;
    c->grid_wgrad = 3 * sms;
    // partials of layers 4, 3, 2 and 1, then of the loss
    c->part_len = (size_t)c->grid_wgrad * (CNN_UP * CNN_UP * (9 * CNN_C + 1) + 2 * CNN_C * (9 * CNN_C + 1) + CNN_C * 10) +
                  CNN_LOSS_BLOCKS;
    const size_t P = c->lay.total, px = c->cap_px;
    bool ok = cudaMalloc(&c->params, P * 4) == cudaSuccess && cudaMalloc(&c->grads, P * 4) == cudaSuccess &&
              cudaMalloc(&c->m, P * 4) == cudaSuccess && cudaMalloc(&c->v, P * 4) == cudaSuccess &&
              cudaMalloc(&c->x0, px * 4) == cudaSuccess && cudaMalloc(&c->a1, px * CNN_C * 2) == cudaSuccess &&
              cudaMalloc(&c->a2, px * CNN_C * 2) == cudaSuccess && cudaMalloc(&c->a3, px * CNN_C * 2) == cudaSuccess &&
              cudaMalloc(&c->g1, px * CNN_C * 2) == cudaSuccess && cudaMalloc(&c->g2, px * CNN_C * 2) == cudaSuccess &&
              cudaMalloc(&c->g3, px * CNN_C * 2) == cudaSuccess &&
              cudaMalloc(&c->gz, px * CNN_UP * CNN_UP * 2) == cudaSuccess &&
              cudaMalloc(&c->heat, px * CNN_UP * CNN_UP * 4) == cudaSuccess &&
              cudaMalloc(&c->part, c->part_len * 4) == cudaSuccess;
    for (int l = 1; l < 4 && ok; ++l) {
        const int n = (l == 3 ? CNN_UP * CNN_UP : CNN_C) * 9 * CNN_C;
        ok = cudaMalloc(&c->wbf[l], n * 2) == cudaSuccess && cudaMalloc(&c->wfl[l], n * 2) == cudaSuccess;
    }
    if (!ok) {
        ulm_cnn_destroy(c);
        return set_error(h, RCA_ERR_CUDA, "cnn allocation failed");
    }
    // He-normal initial weights, zero biases (seeded, host generated)
    std::vector<float> init(P, 0.f);
    std::mt19937_64 rng(d->seed);
    std::normal_distribution<double> nd(0.0, 1.0);
    const int cin[4] = {1, CNN_C, CNN_C, CNN_C}, cout[4] = {CNN_C, CNN_C, CNN_C, CNN_UP * CNN_UP};
    for (int l = 0; l < 4; ++l) {
        const double sd = std::sqrt(2.0 / (9.0 * cin[l]));
        for (int q = 0; q < cout[l] * 9 * cin[l]; ++q) init[c->lay.w[l] + q] = (float)(nd(rng) * sd);
    }
    rca_status st = ulm_cnn_set_params(c, init.data(), P);
    if (st != RCA_OK) {
        ulm_cnn_destroy(c);
        return st;
    }
    *out = c;
    return RCA_OK;
}

extern "C" rca_status ulm_cnn_destroy(ulm_cnn* c)
{
    if (!c) return RCA_ERR_INVALID_ARG;
    cudaStreamSynchronize(c->h->stream);
    void* ptrs[] = {c->params, c->grads, c->m, c->v, c->x0, c->a1, c->a2, c->a3, c->g1, c->g2, c->g3, c->gz, c->heat,
                    c->part, c->wbf[1], c->wbf[2], c->wbf[3], c->wfl[1], c->wfl[2], c->wfl[3]};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    delete c;
    return RCA_OK;
}

extern "C" rca_status ulm_cnn_param_count(const ulm_cnn* c, size_t* n)
{
    if (!c || !n) return RCA_ERR_INVALID_ARG;
    *n = (size_t)c->lay.total;
    return RCA_OK;
}

extern "C" rca_status ulm_cnn_set_params(ulm_cnn* c, const float* host, size_t n)
{
    if (!c || !host) return RCA_ERR_INVALID_ARG;
    if (n != (size_t)c->lay.total) return set_error(c->h, RCA_ERR_SHAPE, "expected %d parameters", c->lay.total);
    rca_status st = cuda_check(c->h, cudaMemcpy(c->params, host, n * 4, cudaMemcpyHostToDevice), "set params");
    if (st != RCA_OK) return st;
    cudaMemset(c->m, 0, n * 4);
    cudaMemset(c->v, 0, n * 4);
    cudaMemset(c->grads, 0, n * 4);
    c->step = 0;
    return cnn_pack(c);
}

extern "C" rca_status ulm_cnn_get_params(const ulm_cnn* c, float* host, size_t n)
{
    if (!c || !host) return RCA_ERR_INVALID_ARG;
    if (n != (size_t)c->lay.total) return set_error(c->h, RCA_ERR_SHAPE, "expected %d parameters", c->lay.total);
    cudaStreamSynchronize(c->h->stream);
    return cuda_check(c->h, cudaMemcpy(host, c->params, n * 4, cudaMemcpyDeviceToHost), "get params");
}

extern "C" rca_status ulm_cnn_get_grads(const ulm_cnn* c, float* host, size_t n)
{
    if (!c || !host) return RCA_ERR_INVALID_ARG;
    if (n != (size_t)c->lay.total) return set_error(c->h, RCA_ERR_SHAPE, "expected %d parameters", c->lay.total);
    cudaStreamSynchronize(c->h->stream);
    return cuda_check(c->h, cudaMemcpy(host, c->grads, n * 4, cudaMemcpyDeviceToHost), "get grads");
}

extern "C" rca_status ulm_cnn_forward(ulm_cnn* c, const float* A, const float* M, int ppf, int B, int H, int W,
                                      float* heat)
{
    if (!c) return RCA_ERR_INVALID_ARG;
    if (!A || !heat) return set_error(c->h, RCA_ERR_INVALID_ARG, "null input or heatmap");
    rca_status st = cnn_check_shape(c, B, H, W);
    if (st != RCA_OK) return st;
    // the kernel stores 16-byte vectors, and stores while other blocks still read: a heatmap at another alignment, or over
    // the memory of the input or its maxima, is copied out of the network's own
    const size_t px = (size_t)B * H * W, nM = M ? ((size_t)B + std::max(ppf, 1) - 1) / std::max(ppf, 1) : 0;
    auto over = [&](const float* p, size_t n) {
        const uintptr_t a = reinterpret_cast<uintptr_t>(heat), b = reinterpret_cast<uintptr_t>(p);
        return a < b + n * 4 && b < a + px * CNN_UP * CNN_UP * 4;
    };
    float* direct = (reinterpret_cast<uintptr_t>(heat) & 15) == 0 && !over(A, px) && !over(M, nM) ? heat : c->heat;
    if ((st = cnn_forward<false>(c, A, M, ppf, B, H, W, direct)) != RCA_OK || direct == heat) return st;
    return cuda_check(c->h,
                      cudaMemcpyAsync(heat, c->heat, px * CNN_UP * CNN_UP * 4, cudaMemcpyDeviceToDevice, c->h->stream),
                      "heatmap copy");
}

extern "C" rca_status ulm_cnn_infer(ulm_cnn* c, const float* A, const float* M, int ppf, int B, int H, int W,
                                    float* heat)
{
    return ulm_cnn_forward(c, A, M, ppf, B, H, W, heat);
}

extern "C" rca_status ulm_cnn_train_step(ulm_cnn* c, const float* A, const float* M, int ppf, int B, int H, int W,
                                         const float* target, float* loss_dev, int apply_update)
{
    if (!c) return RCA_ERR_INVALID_ARG;
    if (!A || !target || !loss_dev) return set_error(c->h, RCA_ERR_INVALID_ARG, "null input, target or loss");
    rca_status st = cnn_check_shape(c, B, H, W);
    if (st != RCA_OK) return st;
    cudaStream_t s = c->h->stream;
    if ((st = cnn_forward<true>(c, A, M, ppf, B, H, W, c->heat)) != RCA_OK) return st;
    const ParamLayout& L = c->lay;
    const size_t px = (size_t)B * H * W;
    const float n = (float)(px * CNN_UP * CNN_UP);
    GradSums sums{};
    size_t at = 0;
    const int lgrid = (int)std::min<size_t>((px + 255) / 256, CNN_LOSS_BLOCKS);
    float* lpart = c->part + (c->part_len - CNN_LOSS_BLOCKS);
    if ((reinterpret_cast<uintptr_t>(target) & 15) == 0)
        launch_chain(k_loss<true>, dim3(lgrid), dim3(256), 0, s, c->heat, target, B * H, W, 2.0f / n, c->gz, lpart);
    else
        launch_chain(k_loss<false>, dim3(lgrid), dim3(256), 0, s, c->heat, target, B * H, W, 2.0f / n, c->gz, lpart);
    // layer 4: dW4 from (a3, dz); dgrad -> g3 masked by a3 > 0
    if ((st = wgrad_launch<CNN_UP * CNN_UP>(c, c->a3, c->gz, B, H, W, 3, sums, at)) != RCA_OK) return st;
    if ((st = conv_launch<CNN_UP * CNN_UP, CNN_C>(c, c->gz, c->wfl[3], c->a3, B, H, W, c->g3)) != RCA_OK) return st;
    // layer 3
    if ((st = wgrad_launch<CNN_C>(c, c->a2, c->g3, B, H, W, 2, sums, at)) != RCA_OK) return st;
    if ((st = conv_launch<CNN_C, CNN_C>(c, c->g3, c->wfl[2], c->a2, B, H, W, c->g2)) != RCA_OK) return st;
    // layer 2
    if ((st = wgrad_launch<CNN_C>(c, c->a1, c->g2, B, H, W, 1, sums, at)) != RCA_OK) return st;
    if ((st = conv_launch<CNN_C, CNN_C>(c, c->g2, c->wfl[1], c->a1, B, H, W, c->g1)) != RCA_OK) return st;
    // layer 1 (FP32)
    sums.part[0] = c->part + at, sums.nparts[0] = std::min(c->grid_wgrad, (B * H + 7) / 8), sums.len[0] = CNN_C * 10;
    launch_chain(k_wgrad1, dim3(sums.nparts[0]), dim3(256), 0, s, c->x0, c->g1, B * H, H, W, c->part + at);
    // every layer's sums and the loss
    sums.part[4] = lpart, sums.nparts[4] = lgrid, sums.len[4] = 1, sums.out[4] = loss_dev, sums.scale[4] = 1.0f / n;
    for (int l = 0; l < 4; ++l) sums.out[l] = c->grads + L.w[l], sums.scale[l] = 1.f;
    for (int l = 0; l < 5; ++l) sums.block0[l + 1] = sums.block0[l] + (sums.len[l] + 31) / 32;
    launch_chain(k_reduce_grads, dim3(sums.block0[5]), dim3(256), 0, s, sums);
    if ((st = cuda_check(c->h, cudaGetLastError(), "backward kernels")) != RCA_OK) return st;
    if (!apply_update) return RCA_OK;
    c->step += 1;
    const double b1 = c->desc.beta1, b2 = c->desc.beta2;
    const double bc1 = 1.0 - std::pow(b1, (double)c->step), bc2 = 1.0 - std::pow(b2, (double)c->step);
    // p -= lr * (m / bc1) / (sqrt(v / bc2) + eps)  ==  lr_t * m / (sqrt(v) + eps_t)
    const float lr_t = (float)(c->desc.lr * std::sqrt(bc2) / bc1);
    const float eps_t = (float)(c->desc.eps * std::sqrt(bc2));
    PackedWeights w{};
    w.lay = L;
    for (int l = 1; l < 4; ++l) w.fwd[l] = c->wbf[l], w.flip[l] = c->wfl[l];
    launch_chain(k_adam, dim3((L.total + 255) / 256), dim3(256), 0, s, c->params, c->grads, c->m, c->v, w, lr_t, (float)b1, (float)b2, eps_t);
    return cuda_check(c->h, cudaGetLastError(), "adam");
}

extern "C" rca_status ulm_cnn_target(rca_handle* h, const float* pts, int n, int B, int H4, int W4, float sigma,
                                     float* target)
{
    if (!h) return RCA_ERR_INVALID_ARG;
    if (!target || (n > 0 && !pts) || n < 0 || B <= 0 || H4 <= 0 || W4 <= 0 || !(sigma > 0))
        return set_error(h, RCA_ERR_INVALID_ARG, "bad target arguments");
    rca_status st = RCA_OK;
    int* off = (int*)ws_get(h, WS_MISC, (size_t)(B + 1) * sizeof(int), &st);
    if (!off) return st;
    k_count_offsets<<<(B + 1 + 255) / 256, 256, 0, h->stream>>>(pts, n, B, off);
    dim3 grid((H4 * W4 + 255) / 256, B);
    k_target<<<grid, 256, 0, h->stream>>>(pts, off, H4, W4, sigma, target);
    return cuda_check(h, cudaGetLastError(), "target kernels");
}

extern "C" rca_status ulm_cnn_save(const ulm_cnn* c, const char* path)
{
    if (!c || !path) return RCA_ERR_INVALID_ARG;
    const size_t P = c->lay.total;
    std::vector<float> buf(4 * P);
    cudaStreamSynchronize(c->h->stream);
    cudaMemcpy(buf.data(), c->params, P * 4, cudaMemcpyDeviceToHost);
    cudaMemcpy(buf.data() + P, c->m, P * 4, cudaMemcpyDeviceToHost);
    cudaMemcpy(buf.data() + 2 * P, c->v, P * 4, cudaMemcpyDeviceToHost);
    FILE* f = fopen(path, "wb");
    if (!f) return set_error(c->h, RCA_ERR_INVALID_ARG, "cannot open %s", path);
    const char magic[8] = {'U', 'L', 'M', 'C', 'N', 'N', '1', 0};
    long long hdr[3] = {(long long)P, c->step, CNN_C};
    bool ok = fwrite(magic, 1, 8, f) == 8 && fwrite(hdr, sizeof hdr, 1, f) == 1 && fwrite(buf.data(), 4, 3 * P, f) == 3 * P;
    fclose(f);
    return ok ? RCA_OK : set_error(c->h, RCA_ERR_INVALID_ARG, "write failed: %s", path);
}

extern "C" rca_status ulm_cnn_load(ulm_cnn* c, const char* path)
{
    if (!c || !path) return RCA_ERR_INVALID_ARG;
    const size_t P = c->lay.total;
    FILE* f = fopen(path, "rb");
    if (!f) return set_error(c->h, RCA_ERR_INVALID_ARG, "cannot open %s", path);
    char magic[8];
    long long hdr[3];
    std::vector<float> buf(3 * P);
    bool ok = fread(magic, 1, 8, f) == 8 && memcmp(magic, "ULMCNN1", 7) == 0 && fread(hdr, sizeof hdr, 1, f) == 1 &&
              hdr[0] == (long long)P && hdr[2] == CNN_C && fread(buf.data(), 4, 3 * P, f) == 3 * P;
    fclose(f);
    if (!ok) return set_error(c->h, RCA_ERR_SHAPE, "%s is not a checkpoint of this network", path);
    cudaMemcpy(c->params, buf.data(), P * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(c->m, buf.data() + P, P * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(c->v, buf.data() + 2 * P, P * 4, cudaMemcpyHostToDevice);
    c->step = hdr[1];
    return cnn_pack(c);
}
