// Eigen-based SVD clutter filter on the Stage-1 slices (Sec. II-A2): for each
// transmission k, the frames' slices form the Casorati matrix X_k (pixels x
// frames); the filter removes the subspace of the n_c largest eigenvalues of
// the frame covariance C_k = X_k^H X_k:  X_k <- X_k - X_k Q Q^H.
//   k_svd_cov_tc   partial covariance tiles of 128 x 128 frames over one split
//                  of the pixels on the tensor cores (tcgen05, kind::tf32, FP32
//                  accumulators in TMEM), FP32-accurate by three TF32 products
//   k_svd_covsum   deterministic sum of the splits, Hermitian completion
//   k_svd_iterate  orthogonal iteration Q <- orth(C Q) towards the n_c-dim
//                  dominant eigenspace, one cluster of CTAs per transmission
//                  (orthonormalisation: classical Gram-Schmidt applied twice); the
//                  projection needs the subspace only.  Beyond 512 frames the same
//                  as two kernels per step: k_svd_cq, k_svd_orth
//   k_svd_project  thread per pixel pair: t = X[p] Q, then X[p] -= t Q^H (in place)
//   k_svd_info     (on request) Rayleigh quotients of the removed basis and of
//                  one extra iterated vector, and the invariance residual
//                  ||C Q - Q (Q^H C Q)||_F of the removed subspace
// The iteration carries nc + 1 vectors (one beyond the rank, when F allows):
// Gram-Schmidt keeps the first nc columns independent of the last, so the
// removed subspace is that of an nc-vector iteration, and the extra column's
// Rayleigh quotient estimates the first eigenvalue left in the data.
#include <algorithm>
#include <cmath>

#include "rca_internal.cuh"

namespace {

#define SV_THREADS 512     // subspace CTA

__device__ __forceinline__ float2 sv_cmul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }

// ---------------------------------------------------------------------------
// Covariance on the tensor cores.  With X = Xr + i Xi (pixels x frames),
//   Re C = Xr^T Xr + Xi^T Xi,   Im C = Xr^T Xi - Xi^T Xr,
// as K-major GEMMs over the pixels (a frame's slice is contiguous in pixels).
// FP32 accuracy from TF32 operands: x = hi + lo with hi = tf32(x), lo = tf32(x -
// hi), and a product a b taken as hi hi + hi lo + lo hi (the dropped lo lo term is
// 2^-22 of it).
// CTA = (frame tile pair ta <= tb, transmission, pixel split): A is 128 frames,
// B is n <= 128 frames (a multiple of 16: the last tile is only as wide as its
// frames).  Operand tiles K-major, no swizzle: 8-row core matrices, the k group kg
// of 4 pixels at byte kg LBO (32 bytes of padding put the four k groups of a store
// in different banks).  B holds [Br | Bi] as 2 n rows, and the accumulators are
// [N | Re | P] with n columns each: Ar [Br | Bi] adds to [Re | P] and
// Ai [Br | Bi] to [N | Re], six MMAs of N = 2 n per 8 pixels; Im = P - N.  On the
// diagonal A is B's own tile.
// Eight converter warps (lane = 4 pixels of one of 8 frames, so that a load
// covers whole 128-byte lines) split a chunk of 16 pixels into a stage and arrive
// on its `full` barrier; a ninth warp issues the chunk's MMAs and commits them to
// the stage's `empty` barrier.  The partial sums are stored transposed (lanes
// along a): part[k][split][b][a] for a <= b.
// Bound: shared memory (144 KB of operand reads and 64 KB of stores per chunk,
// 1660 cycles, against 1540 of the tensor pipe).  300 frames of the paper's slices:
// 2.33 ms with a thread per frame row (32 lines a load), four products of N = 128
// and 128-wide last tiles; now 1.17 ms, with the same sums in the same order.
// (FP16 pairs under a power-of-two scale: 1.06 ms and a 0.18 ms scan for the largest
// value; their sums round half as often in TMEM, which moved the filtered slices by
// up to 4e-5 of the blood, most of what they were off before.)
// Every mbarrier wait is bounded; on a timeout the CTA records ST_TIMEOUT,
// waits once more (bounded) for the commit of its MMAs in flight, frees TMEM
// and returns.  If that second wait also runs out, MMAs may still be in
// flight when TMEM is freed: nothing then guarantees the CTA's accumulators,
// and the status word says the call failed.
// ---------------------------------------------------------------------------
#define SVT_M 128
#define SVT_PC 16                           // pixels per chunk (two K steps)
#define SVT_ALBO (SVT_M * 16 + 32)
#define SVT_BLBO (2 * SVT_M * 16 + 32)
#define SVT_ATILE (4 * SVT_ALBO)            // one of Ar hi, Ar lo, Ai hi, Ai lo
#define SVT_BTILE (4 * SVT_BLBO)            // [Br | Bi] hi or lo
#define SVT_STAGE (4 * SVT_ATILE + 2 * SVT_BTILE)
#define SVT_STAGES 3
#define SVT_SMEM (SVT_STAGES * SVT_STAGE)
#define SVT_CONV 256                        // converter threads
#define SVT_THREADS (SVT_CONV + 32)
#define SVT_TMEM_COLS 512
#define SVT_KMAX 1024                       // pixels per split at most
static_assert(SVT_STAGE % 128 == 0 && SVT_SMEM <= 227 * 1024, "stage size");

__device__ __forceinline__ unsigned svt_tf32(float x)
{
    unsigned r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

// hi and lo TF32 parts of four values
__device__ __forceinline__ void svt_split(float x0, float x1, float x2, float x3, uint4& hi, uint4& lo)
{
    hi = make_uint4(svt_tf32(x0), svt_tf32(x1), svt_tf32(x2), svt_tf32(x3));
    lo = make_uint4(svt_tf32(x0 - __uint_as_float(hi.x)), svt_tf32(x1 - __uint_as_float(hi.y)),
                    svt_tf32(x2 - __uint_as_float(hi.z)), svt_tf32(x3 - __uint_as_float(hi.w)));
}

__device__ __forceinline__ void svt_st16(unsigned addr, uint4 v)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}

// shared-memory matrix descriptor: start, leading (K) and stride (M / N) byte
// offsets in 16-byte units, descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t svt_sdesc(unsigned saddr, unsigned lbo)
{
    return (uint64_t)((saddr >> 4) & 0x3fff) | ((uint64_t)((lbo >> 4) & 0x3fff) << 16) | ((uint64_t)(128 >> 4) << 32) |
           (1ull << 46);
}

// instruction descriptor of kind::tf32: D FP32, A and B TF32 (format 2), both K-major, M = 128
__device__ __forceinline__ unsigned svt_idesc(int N)
{
    return (1u << 4) | (2u << 7) | (2u << 10) | ((unsigned)(N >> 3) << 17) | ((unsigned)(SVT_M >> 4) << 24);
}

__device__ __forceinline__ void svt_mma(unsigned tmem_d, uint64_t da, uint64_t db, unsigned idesc, int accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
        : "memory");
}

// 16 consecutive FP32 accumulator columns of this warp's 32 TMEM lanes
__device__ __forceinline__ void svt_ld16(unsigned taddr, float* v)
{
    unsigned r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = __uint_as_float(r[q]);
}

__device__ __forceinline__ void svt_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__global__ void __launch_bounds__(SVT_THREADS, 1) k_svd_cov_tc(const float2* __restrict__ sl, int F, int nt, int P,
                                                               int ntile, int psplit, float2* __restrict__ part,
                                                               unsigned* __restrict__ status)
{
    extern __shared__ __align__(128) unsigned char svsm[];
    __shared__ uint64_t full[SVT_STAGES], empty[SVT_STAGES], done;
    __shared__ unsigned s_tmem;
    __shared__ volatile int abort_flag;
    int pair = blockIdx.x, ta = 0;
    while (pair >= ntile - ta) {
        pair -= ntile - ta;
        ++ta;
    }
    const int tb = ta + pair;
    const bool diag = ta == tb;
    const int k = blockIdx.y, split = blockIdx.z;
    const int a0 = ta * SVT_M, b0 = tb * SVT_M;
    const int n = min(SVT_M, (F - b0 + 15) / 16 * 16);        // columns of the B tile
    const int p0 = split * psplit, p1 = min(P, p0 + psplit);
    const int nch = p1 > p0 ? (p1 - p0 + SVT_PC - 1) / SVT_PC : 0;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(SVT_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int q = 0; q < SVT_STAGES; ++q) {
            mbar_init(&full[q], SVT_CONV);
            mbar_init(&empty[q], 1);
        }
        mbar_init(&done, 1);
        abort_flag = 0;
        mbar_fence_init();
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = s_tmem;
    const unsigned sbase = smem_u32(svsm);
    if (warp < SVT_CONV / 32) {
        // pass i of a chunk: rows 64 i + 8 warp + lane / 4 of the 256 rows (A, then B), pixels 4 (lane % 4) .. + 3
        const int rw = 8 * warp + (lane >> 2), qp = lane & 3;
        const float4* g[4];
        unsigned dst[4];
        int lo_r[4];                                          // byte distance from the hi to the lo tile
        int re_im[4];                                         // and from the real to the imaginary rows
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = 64 * (i & 1) + rw, f = (i < 2 ? a0 : b0) + r;
            const bool skip = (i < 2 && diag) || (i >= 2 && r >= n);
            g[i] = !skip && f < F ? reinterpret_cast<const float4*>(sl + ((size_t)f * nt + k) * P) : nullptr;
            dst[i] = (unsigned)(r * 16 + (i < 2 ? qp * SVT_ALBO : qp * SVT_BLBO + 4 * SVT_ATILE));
            if (skip) dst[i] = 0xffffffffu;
            lo_r[i] = i < 2 ? SVT_ATILE : SVT_BTILE;
            re_im[i] = i < 2 ? 2 * SVT_ATILE : n * 16;
        }
        auto load = [&](int c, float4 (&x)[4][2]) {
            const int p = p0 + c * SVT_PC + 4 * qp;           // pixel quads are either inside [p0, p1) or outside
            const bool in = c < nch && p < p1;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    x[i][h] = (g[i] && in) ? __ldg(g[i] + p / 2 + h) : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        float4 x[4][2], nx[4][2];
        load(0, x);
        for (int c = 0; c < nch; ++c) {
            const int q = c % SVT_STAGES, u = c / SVT_STAGES;
            load(c + 1, nx);
            // use u of stage q waits until the MMAs of use u - 1 have read it
            if (u > 0 && !mbar_wait_bounded(&empty[q], (unsigned)(u - 1) & 1u)) abort_flag = 1;
            if (abort_flag) break;
            const unsigned st = sbase + (unsigned)(q * SVT_STAGE);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (dst[i] == 0xffffffffu) continue;
                const float4 v = x[i][0], w = x[i][1];
                uint4 h, l;
                svt_split(v.x, v.z, w.x, w.z, h, l);
                svt_st16(st + dst[i], h);
                svt_st16(st + dst[i] + lo_r[i], l);
                svt_split(v.y, v.w, w.y, w.w, h, l);
                svt_st16(st + dst[i] + re_im[i], h);
                svt_st16(st + dst[i] + re_im[i] + lo_r[i], l);
            }
            // this thread's generic-proxy writes before the tensor cores read them
            fence_proxy_async();
            svt_arrive(&full[q]);
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i][0] = nx[i][0], x[i][1] = nx[i][1];
        }
    } else {
        unsigned el;
        asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(el));
        if (el) {
            // the MMAs of chunk c once its stage is full, committed to the stage's
            // empty barrier; the final commit (all MMAs) to `done`
            const unsigned id2 = svt_idesc(2 * n), id1 = svt_idesc(n);
            const unsigned dN = tmem, dRe = tmem + n;
            for (int c = 0; c < nch; ++c) {
                const int q = c % SVT_STAGES, u = c / SVT_STAGES;
                if (!mbar_wait_bounded(&full[q], (unsigned)u & 1u)) abort_flag = 1;
                if (abort_flag) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    const unsigned sa = sbase + (unsigned)(q * SVT_STAGE) + 2 * ks * SVT_ALBO;
                    const unsigned sb = sbase + (unsigned)(q * SVT_STAGE) + 4 * SVT_ATILE + 2 * ks * SVT_BLBO;
                    const uint64_t bh = svt_sdesc(sb, SVT_BLBO), bl = svt_sdesc(sb + SVT_BTILE, SVT_BLBO);
                    uint64_t rh, rl, ih, il;                  // A: real hi, lo, imaginary hi, lo
                    if (diag) {
                        rh = bh, rl = bl;
                        ih = svt_sdesc(sb + n * 16, SVT_BLBO), il = svt_sdesc(sb + SVT_BTILE + n * 16, SVT_BLBO);
                    } else {
                        rh = svt_sdesc(sa, SVT_ALBO), rl = svt_sdesc(sa + SVT_ATILE, SVT_ALBO);
                        ih = svt_sdesc(sa + 2 * SVT_ATILE, SVT_ALBO), il = svt_sdesc(sa + 3 * SVT_ATILE, SVT_ALBO);
                    }
                    const bool first = c == 0 && ks == 0;
                    svt_mma(dRe, rh, bh, id2, !first);
                    svt_mma(dRe, rh, bl, id2, 1);
                    svt_mma(dRe, rl, bh, id2, 1);
                    if (first) {                              // N starts here, Re goes on
                        svt_mma(dN, ih, bh, id1, 0);
                        svt_mma(dRe, ih, svt_sdesc(sb + n * 16, SVT_BLBO), id1, 1);
                    } else {
                        svt_mma(dN, ih, bh, id2, 1);
                    }
                    svt_mma(dN, ih, bl, id2, 1);
                    svt_mma(dN, il, bh, id2, 1);
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 smem_u32(&empty[q]))
                             : "memory");
            }
            // arrives once every MMA issued above has completed (none issued: at once)
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&done))
                         : "memory");
        }
        __syncwarp();
    }
    // every thread: the MMAs complete (bounded) before the accumulators are read or freed
    const bool fin = mbar_wait_bounded(&done, 0u);
    if (__syncthreads_or(!fin || abort_flag)) {
        if (threadIdx.x == 0) atomicOr(status, ST_TIMEOUT);
        // one more bounded wait for the MMAs still in flight before the
        // barriers are invalidated and TMEM is freed (the MMA thread commits
        // `done` after its last issue even when it stopped early)
        if (!fin) mbar_wait_bounded(&done, 0u);
        __syncthreads();
    } else if (nch > 0 && warp < SVT_CONV / 32) {
        // warps w and w + 4 read the same TMEM lanes (rows a), every other 16 columns each
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        float2* dst = part + (((size_t)k * gridDim.z + split) * F) * F;
        const int a = a0 + 32 * (warp & 3) + lane;
        const unsigned lrow = (unsigned)(32 * (warp & 3)) << 16;
#pragma unroll 1
        for (int cg = warp >> 2; cg < n / 16; cg += 2) {
            float re[16], ip[16], in[16];
            svt_ld16(tmem + lrow + (unsigned)(16 * cg), in);
            svt_ld16(tmem + lrow + (unsigned)(n + 16 * cg), re);
            svt_ld16(tmem + lrow + (unsigned)(2 * n + 16 * cg), ip);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const int b = b0 + 16 * cg + j;
                if (a <= b && b < F) dst[(size_t)b * F + a] = make_float2(re[j], ip[j] - in[j]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 0; q < SVT_STAGES; ++q) {
            mbar_inval(&full[q]);
            mbar_inval(&empty[q]);
        }
        mbar_inval(&done);
    }
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(SVT_TMEM_COLS)
                     : "memory");
    }
}

// C[k][a][b] = sum over splits for a <= b, C[b][a] = conj(C[a][b]), so that C is exactly Hermitian
__global__ void k_svd_covsum(const float2* __restrict__ part, int F, int nsplit, float2* __restrict__ C)
{
    const int k = blockIdx.y;
    float2* Ck = C + (size_t)k * F * F;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < F * F; idx += gridDim.x * blockDim.x) {
        const int b = idx / F, a = idx - b * F;
        if (a > b) continue;
        float2 s = make_float2(0.f, 0.f);
#pragma unroll 8
        for (int q = 0; q < nsplit; ++q) {
            const float2 v = part[(((size_t)k * nsplit + q) * F + b) * F + a];
            s.x += v.x;
            s.y += v.y;
        }
        Ck[(size_t)a * F + b] = s;
        if (a < b) Ck[(size_t)b * F + a] = make_float2(s.x, -s.y);
    }
}

// deterministic start vectors in [-1, 1]
__device__ __forceinline__ float sv_hash(unsigned x)
{
    x ^= x >> 16;
    x *= 0x7feb352du;
    x ^= x >> 15;
    x *= 0x846ca68bu;
    x ^= x >> 16;
    return (float)(x & 0xffffff) * (2.0f / 16777216.0f) - 1.0f;
}

// block sum of one float (all threads get the result)
__device__ __forceinline__ float sv_bsum(float v, float* red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    float s = 0.f;
    for (int w = 0; w < nw; ++w) s += red[w];
    return s;
}

// Orthonormalise the nc columns of Y (pitch ld) into Q by classical
// Gram-Schmidt applied twice per column.
__device__ void sv_orth(float2* Y, float2* Q, int F, int nc, int ld, float2* rbuf, float* red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int j = 0; j < nc; ++j) {
        for (int pass = 0; pass < 2; ++pass) {
            // r_i = Q_i^H y_j, one warp per previous column
            for (int i = warp; i < j; i += nw) {
                float2 s = make_float2(0.f, 0.f);
                for (int g = lane; g < F; g += 32) {
                    const float2 q = Q[g * ld + i], y = Y[g * ld + j];
                    s.x += q.x * y.x + q.y * y.y;
                    s.y += q.x * y.y - q.y * y.x;
                }
                for (int o = 16; o > 0; o >>= 1) {
                    s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
                    s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
                }
                if (lane == 0) rbuf[i] = s;
            }
            __syncthreads();
            for (int g = threadIdx.x; g < F; g += blockDim.x) {
                float2 y = Y[g * ld + j];
                for (int i = 0; i < j; ++i) {
                    const float2 t = sv_cmul(rbuf[i], Q[g * ld + i]);
                    y.x -= t.x;
                    y.y -= t.y;
                }
                Y[g * ld + j] = y;
            }
            __syncthreads();
        }
        float e = 0.f;
        for (int g = threadIdx.x; g < F; g += blockDim.x) {
            const float2 y = Y[g * ld + j];
            e += y.x * y.x + y.y * y.y;
        }
        const float nrm = sqrtf(sv_bsum(e, red));
        const float inv = nrm > 0.f ? 1.0f / nrm : 0.f;
        for (int g = threadIdx.x; g < F; g += blockDim.x) {
            const float2 y = Y[g * ld + j];
            Q[g * ld + j] = make_float2(y.x * inv, y.y * inv);
        }
        __syncthreads();
    }
}

// Orthogonal iteration for the nc-dimensional dominant eigenspace of each
// C_k, one step = k_svd_cq (Y = C Q over many CTAs) then k_svd_orth (one CTA
// per transmission: Y -> orthonormal Q); k_svd_orth with `start` set builds
// the fixed start basis.  Q, Y: [k][F][nc] in global memory.
__global__ void __launch_bounds__(SV_THREADS) k_svd_orth(float2* __restrict__ Yg, float2* __restrict__ Qg, int F,
                                                         int nc, int start)
{
    extern __shared__ float2 ssv[];
    __shared__ float red[32];
    __shared__ float2 rbuf[32];
    const int ld = nc + 1;                             // padded: lanes over g spread over the banks
    float2* Q = ssv;                                   // [F][ld]
    float2* Y = ssv + (size_t)F * ld;                  // [F][ld]
    const int k = blockIdx.x;
    for (int idx = threadIdx.x; idx < F * nc; idx += blockDim.x) {
        const int g = idx / nc, j = idx - g * nc;
        Y[g * ld + j] = start ? make_float2(sv_hash(2u * (unsigned)idx + 1u), sv_hash(2u * (unsigned)idx + 2u))
                              : Yg[((size_t)k * F + g) * nc + j];
    }
    __syncthreads();
    sv_orth(Y, Q, F, nc, ld, rbuf, red);
    for (int idx = threadIdx.x; idx < F * nc; idx += blockDim.x) {
        const int g = idx / nc, j = idx - g * nc;
        Qg[((size_t)k * F + g) * nc + j] = Q[g * ld + j];
    }
}

// ---------------------------------------------------------------------------
// The whole orthogonal iteration of one transmission in one cluster of eight
// CTAs.  Each CTA owns an eighth of the rows of C_k (up to 320 frames, ten rows per
// lane, they fit its shared memory; beyond, each step reads them from L2) and holds
// the whole basis V; a step is
//   product   the CTA's rows of C V, one row and three columns per thread
//   exchange  its rows to every CTA's V (distributed shared memory), between two
//             cluster barriers: V is read by the product until the first
//   basis     Gram-Schmidt in every CTA alike
// Latency-bound by the basis chain.  As two kernels per step (product over many
// CTAs, basis in one) 30 steps of 300 frames and 17 vectors took 2.66 ms, launches
// included; now 1.24 ms, with the same sums in the same order (400 frames, one
// transmission pair of 199 x 64 pixels: the whole filter 3.31 and 2.30 ms).  (Modified
// Gram-Schmidt with one barrier per column and the product in four quarters: 0.69
// ms, but its rounding moved the filtered slices by 1e-5 of the blood.)
// ---------------------------------------------------------------------------
#define SVI_CTAS 8
#define SVI_FMAX 512                                   // 32 lanes x 16 rows of a column
#define SVI_FSMEM 320                                  // C's rows in shared memory up to here (10 rows of a column)

__device__ __forceinline__ void svi_cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

struct SviSmem {
    int ld, ldc, rows, v, part, c, bytes;              // leading dimensions, rows per CTA, byte offsets
    bool c_in;                                         // C's rows in shared memory
};

inline SviSmem svi_smem(int F, int nb)
{
    SviSmem s;
    s.ld = nb | 1;                                     // odd: a column's lanes hit different banks
    s.ldc = F | 1;
    s.rows = (F + SVI_CTAS - 1) / SVI_CTAS;
    s.v = 0;
    s.part = s.v + F * s.ld * 8;
    s.c = s.part + s.rows * nb * 8;
    s.c_in = F <= SVI_FSMEM;                           // 197 KB at most (33 columns)
    s.bytes = s.c + (s.c_in ? s.rows * s.ldc * 8 : 0);
    return s;
}

// Classical Gram-Schmidt, twice per column, of the nb columns of V in place: the
// sums of sv_orth in its order (dot products over a warp's lanes, updates over the
// earlier columns, the norm over the block), with the finished columns in their
// warps' registers as well.
template <int RPL, int CPW>                            // rows per lane, columns per warp
__device__ __forceinline__ void svi_basis(float2* __restrict__ V, int F, int nb, int ld, float2* rbuf, float* red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = threadIdx.x;
    float2 q[CPW][RPL];
#pragma unroll
    for (int c = 0; c < CPW; ++c)
#pragma unroll
        for (int r = 0; r < RPL; ++r) q[c][r] = make_float2(0.f, 0.f);
    for (int j = 0; j < nb; ++j) {
        float2 y = g < F ? V[g * ld + j] : make_float2(0.f, 0.f);
        for (int pass = 0; pass < 2 && j > 0; ++pass) {
            // r_i = q_i^H y, the warp that owns column i
            if (warp < j) {
                float2 yy[RPL];
#pragma unroll
                for (int r = 0; r < RPL; ++r)
                    yy[r] = lane + 32 * r < F ? V[(lane + 32 * r) * ld + j] : make_float2(0.f, 0.f);
#pragma unroll
                for (int c = 0; c < CPW; ++c) {
                    if (warp + 16 * c >= j) continue;
                    float2 s = make_float2(0.f, 0.f);
#pragma unroll
                    for (int r = 0; r < RPL; ++r) {
                        s.x += q[c][r].x * yy[r].x + q[c][r].y * yy[r].y;
                        s.y += q[c][r].x * yy[r].y - q[c][r].y * yy[r].x;
                    }
                    for (int o = 16; o > 0; o >>= 1) {
                        s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
                        s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
                    }
                    if (lane == 0) rbuf[warp + 16 * c] = s;
                }
            }
            __syncthreads();
            if (g < F) {
#pragma unroll 4
                for (int i = 0; i < j; ++i) {
                    const float2 t = sv_cmul(rbuf[i], V[g * ld + i]);
                    y.x -= t.x;
                    y.y -= t.y;
                }
                if (pass == 0) V[g * ld + j] = y;
            }
            if (pass == 0) __syncthreads();
        }
        float e = 0.f;
        if (g < F) e += y.x * y.x + y.y * y.y;
        const float nrm = sqrtf(sv_bsum(e, red));
        const float inv = nrm > 0.f ? 1.0f / nrm : 0.f;
        if (g < F) V[g * ld + j] = make_float2(y.x * inv, y.y * inv);
        __syncthreads();
#pragma unroll
        for (int c = 0; c < CPW; ++c) {
            if (warp + 16 * c != j) continue;
#pragma unroll
            for (int r = 0; r < RPL; ++r)
                q[c][r] = lane + 32 * r < F ? V[(lane + 32 * r) * ld + j] : make_float2(0.f, 0.f);
        }
    }
}

template <int RPL, int CPW, bool CIN>
__global__ void __cluster_dims__(SVI_CTAS, 1, 1) __launch_bounds__(SV_THREADS, 1)
    k_svd_iterate(const float2* __restrict__ Call, int F, int nb, int iters, const SviSmem L, float2* __restrict__ Qg)
{
    extern __shared__ __align__(16) unsigned char svi[];
    __shared__ float2 rbuf[34];
    __shared__ float red[32];
    float2* V = reinterpret_cast<float2*>(svi + L.v);       // [F][ld]
    float2* part = reinterpret_cast<float2*>(svi + L.part); // [rows][nb]
    const int k = blockIdx.y, rank = blockIdx.x, r0 = rank * L.rows, nr = min(L.rows, F - r0);   // nr may be < 1
    const float2* Cg = Call + ((size_t)k * F + r0) * F;
    float2* Cs = reinterpret_cast<float2*>(svi + L.c);      // [rows][ldc]
    if (CIN)
        for (int r = threadIdx.x >> 5; r < nr; r += SV_THREADS / 32)
            for (int g = threadIdx.x & 31; g < F; g += 32) Cs[r * L.ldc + g] = Cg[(size_t)r * F + g];
    for (int idx = threadIdx.x; idx < F * nb; idx += SV_THREADS)
        V[idx / nb * L.ld + idx % nb] = make_float2(sv_hash(2u * (unsigned)idx + 1u), sv_hash(2u * (unsigned)idx + 2u));
    __syncthreads();
    svi_basis<RPL, CPW>(V, F, nb, L.ld, rbuf, red);
    const int ntc = (nb + 2) / 3, nrr = max(nr, 0);
    for (int it = 0; it < iters; ++it) {
        for (int t = threadIdx.x; t < nrr * ntc; t += SV_THREADS) {
            // row a, columns b .. b + 2 (the edge repeats the last column)
            const int a = t / ntc, b = 3 * (t % ntc), b1 = min(b + 1, nb - 1), b2 = min(b + 2, nb - 1);
            const float2* cr = CIN ? Cs + a * L.ldc : Cg + (size_t)a * F;
            float2 acc[3];
#pragma unroll
            for (int w = 0; w < 3; ++w) acc[w] = make_float2(0.f, 0.f);
#pragma unroll 4
            for (int g = 0; g < F; ++g) {
                const float2 c = cr[g];
                const float2* v = V + g * L.ld;
                const float2 q[3] = {v[b], v[b1], v[b2]};
#pragma unroll
                for (int w = 0; w < 3; ++w) {
                    acc[w].x = fmaf(c.x, q[w].x, fmaf(-c.y, q[w].y, acc[w].x));
                    acc[w].y = fmaf(c.x, q[w].y, fmaf(c.y, q[w].x, acc[w].y));
                }
            }
#pragma unroll
            for (int w = 0; w < 3; ++w)
                if (b + w < nb) part[a * nb + b + w] = acc[w];
        }
        svi_cluster_sync();                            // every CTA of the cluster has read V
        for (int idx = threadIdx.x; idx < nrr * nb; idx += SV_THREADS) {
            const float2 y = part[idx];
            const unsigned at = smem_u32(V + (r0 + idx / nb) * L.ld + idx % nb);
#pragma unroll
            for (int c = 0; c < SVI_CTAS; ++c) {
                unsigned to;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(at), "r"(c));
                asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(to), "f"(y.x), "f"(y.y) : "memory");
            }
        }
        svi_cluster_sync();                            // V is C V in every CTA
        svi_basis<RPL, CPW>(V, F, nb, L.ld, rbuf, red);
    }
    if (rank == 0)
        for (int idx = threadIdx.x; idx < F * nb; idx += SV_THREADS)
            Qg[(size_t)k * F * nb + idx] = V[idx / nb * L.ld + idx % nb];
}

// Y[k] = C_k Q[k]: a thread per (row, column) of Y, rows in blocks of
// SV_THREADS / nc per CTA; Q[k] staged in shared memory
__global__ void __launch_bounds__(SV_THREADS) k_svd_cq(const float2* __restrict__ C, const float2* __restrict__ Qg,
                                                       int F, int nc, float2* __restrict__ Yg)
{
    extern __shared__ float2 ssv[];                    // Q[k] [F][nc]
    const int k = blockIdx.y;
    const float2* Qk = Qg + (size_t)k * F * nc;
    for (int idx = threadIdx.x; idx < F * nc; idx += blockDim.x) ssv[idx] = Qk[idx];
    __syncthreads();
    const int rows = blockDim.x / nc;
    const int f = blockIdx.x * rows + threadIdx.x / nc, j = threadIdx.x % nc;
    if (threadIdx.x >= rows * nc || f >= F) return;
    const float2* Crow = C + ((size_t)k * F + f) * F;
    float2 acc = make_float2(0.f, 0.f);
    for (int g = 0; g < F; ++g) {
        const float2 c = __ldg(Crow + g), q = ssv[g * nc + j];
        acc.x = fmaf(c.x, q.x, fmaf(-c.y, q.y, acc.x));
        acc.y = fmaf(c.x, q.y, fmaf(c.y, q.x, acc.y));
    }
    Yg[((size_t)k * F + f) * nc + j] = acc;
}

// Two adjacent pixels per thread: t = X[p] Q over the frames, then X[p] -= t Q^H
// (in place).  The two pixels are the halves of packed FP32 pairs, so that a
// basis value read from shared memory feeds four packed FMAs, and NC (the rank
// rounded up to a multiple of four, the basis padded with zeros) keeps t in
// registers.  Frames in blocks of SV_FB, the next block's loads in flight while
// one is worked on.  Bound: FP32 pipe (39 GFLOP for the paper's ensemble at rank
// 16, 0.5 ms) beside three passes over the slices in HBM (0.54 ms).  One pixel per
// thread with scalar FMAs and a test per column: 2.30 ms; now 0.84 ms, with the
// same sums in the same order.
#define SV_FB 4
template <int NC>
__global__ void __launch_bounds__(128) k_svd_project(float2* __restrict__ sl, int F, int nt, int P, int nc, int nb,
                                                     const float2* __restrict__ Qall)
{
    extern __shared__ __align__(16) float2 ssv[];          // [F][NC]
    const int k = blockIdx.y;
    const float2* Qk = Qall + (size_t)k * F * nb;          // [F][nb]; the first nc columns are removed
    for (int idx = threadIdx.x; idx < F * NC; idx += blockDim.x) {
        const int f = idx / NC, j = idx % NC;
        ssv[idx] = j < nc ? Qk[f * nb + j] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const int p = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (p >= P) return;                                    // P is even: both pixels inside
    const size_t fs = (size_t)nt * P / 2;                  // frame stride in pixel pairs
    float4* base = reinterpret_cast<float4*>(sl + (size_t)k * P + p);
    uint64_t tr[NC], ti[NC];                               // (pixel 0, pixel 1)
#pragma unroll
    for (int j = 0; j < NC; ++j) tr[j] = ti[j] = 0ull;
    const unsigned qa = smem_u32(ssv);
    float4 x[SV_FB], nx[SV_FB];
    auto load = [&](int f0, float4 (&v)[SV_FB]) {
#pragma unroll
        for (int u = 0; u < SV_FB; ++u)
            v[u] = f0 + u < F ? base[(size_t)(f0 + u) * fs] : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    load(0, x);
    for (int f0 = 0; f0 < F; f0 += SV_FB) {
        load(f0 + SV_FB, nx);
#pragma unroll
        for (int u = 0; u < SV_FB; ++u) {
            if (f0 + u >= F) break;
            const uint64_t xr = f2_pack(x[u].x, x[u].z), xi = f2_pack(x[u].y, x[u].w), xn = f2_pack(-x[u].y, -x[u].w);
            const unsigned qf = qa + (unsigned)((f0 + u) * NC * 8);
#pragma unroll
            for (int j = 0; j < NC; j += 2) {
                uint64_t q2[2];
                lds_u64x2(qf + j * 8, q2[0], q2[1]);
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const float2 q = f2_unpack(q2[v]);
                    const uint64_t qr = f2_pack(q.x, q.x), qi = f2_pack(q.y, q.y);
                    tr[j + v] = f2_fma(xr, qr, f2_fma(xn, qi, tr[j + v]));
                    ti[j + v] = f2_fma(xr, qi, f2_fma(xi, qr, ti[j + v]));
                }
            }
        }
#pragma unroll
        for (int u = 0; u < SV_FB; ++u) x[u] = nx[u];
    }
    load(0, x);
    for (int f0 = 0; f0 < F; f0 += SV_FB) {
        load(f0 + SV_FB, nx);
#pragma unroll
        for (int u = 0; u < SV_FB; ++u) {
            if (f0 + u >= F) break;
            // the negated pixels gather sum_j t_j conj(q_j) = (tr qr + ti qi, ti qr - tr qi)
            uint64_t nr = f2_pack(-x[u].x, -x[u].z), ni = f2_pack(-x[u].y, -x[u].w);
            const unsigned qf = qa + (unsigned)((f0 + u) * NC * 8);
#pragma unroll
            for (int j = 0; j < NC; j += 2) {
                uint64_t q2[2];
                lds_u64x2(qf + j * 8, q2[0], q2[1]);
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const float2 q = f2_unpack(q2[v]);
                    const uint64_t qr = f2_pack(q.x, q.x), qi = f2_pack(q.y, q.y), qn = f2_pack(-q.y, -q.y);
                    nr = f2_fma(tr[j + v], qr, f2_fma(ti[j + v], qi, nr));
                    ni = f2_fma(ti[j + v], qr, f2_fma(tr[j + v], qn, ni));
                }
            }
            const float2 r = f2_unpack(nr), i = f2_unpack(ni);
            base[(size_t)(f0 + u) * fs] = make_float4(-r.x, -i.x, -r.y, -i.y);
        }
#pragma unroll
        for (int u = 0; u < SV_FB; ++u) x[u] = nx[u];
    }
}

// One CTA per transmission, after Y = C Q (nb columns): H = Q^H Y, the
// Rayleigh quotients theta_j = Re H_jj, and the residual of the removed
// subspace R = Y_nc - Q_nc H_nc (first nc columns).  info[k] = {max and min
// theta_j over j < nc, theta_nc of the extra column (0 without one),
// ||R||_F / min_j theta_j}.
__global__ void __launch_bounds__(SV_THREADS) k_svd_info(const float2* __restrict__ Qg, const float2* __restrict__ Yg,
                                                        int F, int nc, int nb, float* __restrict__ info)
{
    extern __shared__ float2 ssv[];
    __shared__ float red[32];
    __shared__ float2 H[33 * 33];
    const int ld = nb + 1;
    float2* Q = ssv;                                   // [F][ld]
    float2* Y = ssv + (size_t)F * ld;                  // [F][ld]
    const int k = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int idx = threadIdx.x; idx < F * nb; idx += blockDim.x) {
        const int g = idx / nb, j = idx - g * nb;
        Q[g * ld + j] = Qg[((size_t)k * F + g) * nb + j];
        Y[g * ld + j] = Yg[((size_t)k * F + g) * nb + j];
    }
    __syncthreads();
    for (int e = warp; e < nb * nb; e += nw) {
        const int i = e / nb, j = e - i * nb;
        float2 acc = make_float2(0.f, 0.f);
        for (int g = lane; g < F; g += 32) {
            const float2 q = Q[g * ld + i], y = Y[g * ld + j];    // conj(q) y
            acc.x += q.x * y.x + q.y * y.y;
            acc.y += q.x * y.y - q.y * y.x;
        }
        for (int o = 16; o > 0; o >>= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
        }
        if (lane == 0) H[i * nb + j] = acc;
    }
    __syncthreads();
    float r2 = 0.f;
    for (int idx = threadIdx.x; idx < F * nc; idx += blockDim.x) {
        const int g = idx / nc, j = idx - g * nc;
        float2 r = Y[g * ld + j];
        for (int i = 0; i < nc; ++i) {
            const float2 t = sv_cmul(Q[g * ld + i], H[i * nb + j]);
            r.x -= t.x;
            r.y -= t.y;
        }
        r2 += r.x * r.x + r.y * r.y;
    }
    r2 = sv_bsum(r2, red);
    if (threadIdx.x == 0) {
        float tmax = -INFINITY, tmin = INFINITY;
        for (int j = 0; j < nc; ++j) {
            tmax = fmaxf(tmax, H[j * nb + j].x);
            tmin = fminf(tmin, H[j * nb + j].x);
        }
        info[4 * k + 0] = tmax;
        info[4 * k + 1] = tmin;
        info[4 * k + 2] = nb > nc ? H[nc * nb + nc].x : 0.f;
        info[4 * k + 3] = tmin > 0.f ? sqrtf(r2) / tmin : INFINITY;
    }
}

}  // namespace

size_t svd_subspace_smem(int F, int nb) { return 2 * (size_t)F * (nb + 1) * sizeof(float2); }

rca_status launch_clutter_svd(rca_handle* h, const rca_tables* t, float2* slices, int F, int nc, int iters,
                              float* info)
{
    const GeomDev& g = t->gd;
    const int nt = 2 * g.K, P = g.nzs * g.N;
    if (nc < 0 || nc > 32) return set_error(h, RCA_ERR_INVALID_ARG, "clutter rank %d outside [0, 32]", nc);
    if (nc >= F) return set_error(h, RCA_ERR_INVALID_ARG, "clutter rank %d must be below the frame count %d", nc, F);
    if (iters < 1 || iters > 1000) return set_error(h, RCA_ERR_INVALID_ARG, "iterations %d outside [1, 1000]", iters);
    if (nc == 0) {
        if (info) {
            cudaError_t e0 = cudaMemsetAsync(info, 0, (size_t)4 * nt * sizeof(float), h->stream);
            if (e0 != cudaSuccess) return cuda_check(h, e0, "clutter info clear");
        }
        return RCA_OK;
    }
    const int nb = std::min(nc + 1, F);                 // iterated vectors: the rank plus one
    const size_t smem_sub = svd_subspace_smem(F, nb);
    if (smem_sub > 200 * 1024)
        return set_error(h, RCA_ERR_UNSUPPORTED, "frames x (rank + 2) = %d x %d exceeds the subspace kernel", F, nb + 1);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // the covariance's pixel quads stay whole: N is a multiple of 4 (geometry rule)
    if (P % 4 != 0) return set_error(h, RCA_ERR_UNSUPPORTED, "slice pixel count %d not a multiple of 4", P);
    // (tile pair, transmission, pixel split) CTAs, at least one wave, and at
    // most SVT_KMAX pixels per split, added on the CUDA cores (k_svd_covsum):
    // the error of one TMEM accumulation grows with its length (measured on the
    // 300-frame paper stack: 2.6e-5 of the input with 21 280 pixels per split,
    // 1.6e-6 with 1 024; 5.7e-7 for the CUDA-core FP32 covariance it replaced)
    const int ntile = (F + SVT_M - 1) / SVT_M, npair = ntile * (ntile + 1) / 2;
    int nsplit = std::max({1, sms / (npair * nt), (P + SVT_KMAX - 1) / SVT_KMAX});
    nsplit = std::min(nsplit, (P + SVT_PC - 1) / SVT_PC);
    const int psplit = ((P + nsplit - 1) / nsplit + SVT_PC - 1) / SVT_PC * SVT_PC;
    nsplit = (P + psplit - 1) / psplit;
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t n_part = (size_t)nt * nsplit * F * F, n_C = (size_t)nt * F * F, n_Q = (size_t)nt * F * nb;
    const size_t bytes = up(n_part * 8) + up(n_C * 8) + 2 * up(n_Q * 8);
    rca_status st = RCA_OK;
    char* ws = (char*)ws_get(h, WS_SVD, bytes, &st);
    if (!ws) return st;
    float2* part = reinterpret_cast<float2*>(ws);
    float2* C = reinterpret_cast<float2*>(ws + up(n_part * 8));
    float2* Q = reinterpret_cast<float2*>((char*)C + up(n_C * 8));
    float2* Y = reinterpret_cast<float2*>((char*)Q + up(n_Q * 8));
    cudaError_t ea = cudaFuncSetAttribute(k_svd_cov_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, SVT_SMEM);
    if (ea != cudaSuccess) return cuda_check(h, ea, "covariance smem attribute");
    k_svd_cov_tc<<<dim3(npair, nt, nsplit), SVT_THREADS, SVT_SMEM, h->stream>>>(slices, F, nt, P, ntile, psplit,
                                                                                 part, h->d_status);
    k_svd_covsum<<<dim3((unsigned)std::min<size_t>(((size_t)F * F + 255) / 256, 1024), nt), 256, 0, h->stream>>>(
        part, F, nsplit, C);
    cudaError_t e = cudaFuncSetAttribute(k_svd_orth, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_sub);
    if (e != cudaSuccess) return cuda_check(h, e, "subspace smem attribute");
    const size_t smem_q = (size_t)F * nb * sizeof(float2);
    e = cudaFuncSetAttribute(k_svd_cq, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_q);
    if (e != cudaSuccess) return cuda_check(h, e, "subspace product smem attribute");
    const int rows_cq = SV_THREADS / nb;
    // the cluster kernel keeps a column in a warp's registers, 16 rows per lane at most
    if (F <= SVI_FMAX) {
        const SviSmem L = svi_smem(F, nb);
        auto kern = L.c_in ? (nb <= 32 ? k_svd_iterate<10, 2, true> : k_svd_iterate<10, 3, true>)
                           : (nb <= 32 ? k_svd_iterate<16, 2, false> : k_svd_iterate<16, 3, false>);
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L.bytes);
        if (e != cudaSuccess) return cuda_check(h, e, "subspace smem attribute");
        kern<<<dim3(SVI_CTAS, nt), SV_THREADS, L.bytes, h->stream>>>(C, F, nb, iters, L, Q);
    } else {
        k_svd_orth<<<nt, SV_THREADS, smem_sub, h->stream>>>(Y, Q, F, nb, 1);
        for (int it = 0; it < iters; ++it) {
            k_svd_cq<<<dim3((F + rows_cq - 1) / rows_cq, nt), SV_THREADS, smem_q, h->stream>>>(C, Q, F, nb, Y);
            k_svd_orth<<<nt, SV_THREADS, smem_sub, h->stream>>>(Y, Q, F, nb, 0);
        }
    }
    if (info) {
        k_svd_cq<<<dim3((F + rows_cq - 1) / rows_cq, nt), SV_THREADS, smem_q, h->stream>>>(C, Q, F, nb, Y);
        e = cudaFuncSetAttribute(k_svd_info, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_sub);
        if (e != cudaSuccess) return cuda_check(h, e, "clutter info smem attribute");
        k_svd_info<<<nt, SV_THREADS, smem_sub, h->stream>>>(Q, Y, F, nc, nb, info);
    }
    static constexpr decltype(&k_svd_project<4>) project[8] = {
        k_svd_project<4>,  k_svd_project<8>,  k_svd_project<12>, k_svd_project<16>,
        k_svd_project<20>, k_svd_project<24>, k_svd_project<28>, k_svd_project<32>};
    const int nq = (nc + 3) / 4;
    const size_t smem_proj = (size_t)F * nq * 4 * sizeof(float2);
    e = cudaFuncSetAttribute(project[nq - 1], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_proj);
    if (e != cudaSuccess) return cuda_check(h, e, "projection smem attribute");
    project[nq - 1]<<<dim3((P / 2 + 127) / 128, nt), 128, smem_proj, h->stream>>>(slices, F, nt, P, nc, nb, Q);
    return cuda_check(h, cudaGetLastError(), "clutter filter kernels");
}
