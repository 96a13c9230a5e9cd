// localize.cu -- XDoppler enhancement, separable NCC, sub-pixel peaks and
// XZ / YZ pairing (Sec. II-A4, Fig. 1e, Fig. 1g).
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <mutex>

#include "rca_internal.cuh"

namespace {

// ---------------------------------------------------------------------------
// XDoppler: each thread owns one pixel (axis, slab, row, lateral) and walks
// the frames with a sliding 3-frame window, so every plane is read once:
//   Q_t = P_RC,t conj(P_CR,t),  A_t = sqrt(|Q_{t-1} + Q_t + Q_{t+1}|).
// The planes of frame t+2 are loaded while frame t is finished.  Frames are
// split into chunks across blockIdx.y (each chunk re-reads the frame before
// it) when the planes alone would give too few blocks.  M_t = max A_t: warp
// max, shared-memory atomicMax per frame, one global atomicMax per block and
// frame at the end (non-negative floats order like their bits).
// ---------------------------------------------------------------------------
// plane element i of compile-time dtype PT as float2 (read-only path)
template <int PT>
__device__ __forceinline__ float2 ld_plane(const void* __restrict__ p, size_t i)
{
    if constexpr (PT == RCA_C32) {
        return __ldg(reinterpret_cast<const float2*>(p) + i);
    } else {
        const unsigned u = __ldg(reinterpret_cast<const unsigned*>(p) + i);
        if constexpr (PT == RCA_C16F) return __half22float2(*reinterpret_cast<const __half2*>(&u));
        else return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u));
    }
}

template <int PT>
__global__ void __launch_bounds__(256) k_enhance(const void* __restrict__ planes, int F, int S, size_t plane_sz,
                                                 int enh, int tf, float* __restrict__ A, unsigned* __restrict__ M)
{
    grid_wait();
    extern __shared__ unsigned mx[];  // [tf] maxima of this chunk's frames
    const int t0 = blockIdx.y * tf, t1 = min(F, t0 + tf);
    for (int t = threadIdx.x; t < t1 - t0; t += blockDim.x) mx[t] = 0u;
    __syncthreads();
    const size_t per_axis = (size_t)S * plane_sz;
    const size_t npx = 2 * per_axis;
    const size_t FS = 2 * npx;                       // elements per frame: [axis][family][S][nz][N]
    const size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool act = p < npx;
    const size_t axis = act ? p / per_axis : 0, rest = act ? p % per_axis : 0;
    const int lane = threadIdx.x & 31;
    // element of the RC plane of frame t is t FS + oR; its CR plane lies per_axis further
    const size_t oR = axis * 2 * per_axis + rest;
    auto ld = [&](int t, int fam) {
        return (act && t < F) ? ld_plane<PT>(planes, (size_t)t * FS + oR + (fam ? per_axis : 0))
                              : make_float2(0.f, 0.f);
    };
    auto xq = [](float2 a, float2 b) { return make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y); };
    float2 r0 = ld(t0, 0), c0 = ld(t0, 1), r1 = ld(t0 + 1, 0), c1 = ld(t0 + 1, 1);
    float2 r2 = ld(t0 + 2, 0), c2 = ld(t0 + 2, 1);
    float2 qm = make_float2(0.f, 0.f);
    if (t0 > 0 && enh == ULM_ENH_XDOPPLER) qm = xq(ld(t0 - 1, 0), ld(t0 - 1, 1));
    // prefetch index of frame t + 3 and output pointer of frame t, advanced per frame
    size_t i3 = (size_t)(t0 + 3) * FS + oR;
    float* out = A + (size_t)t0 * npx + p;
    for (int t = t0; t < t1; ++t) {
        float2 r3 = make_float2(0.f, 0.f), c3 = r3;
        if (act && t + 3 < F) {
            r3 = ld_plane<PT>(planes, i3);
            c3 = ld_plane<PT>(planes, i3 + per_axis);
        }
        i3 += FS;
        float a;
        if (enh == ULM_ENH_XDOPPLER) {
            const float2 q0 = xq(r0, c0), qp = xq(r1, c1);
            const float re = qm.x + q0.x + qp.x, im = qm.y + q0.y + qp.y;
            a = sqrtf(sqrtf(re * re + im * im));
            qm = q0;
        } else {
            const float re = r0.x + c0.x, im = r0.y + c0.y;
            a = sqrtf(re * re + im * im);
        }
        if (act) __stcs(out, a);
        out += npx;
        // warp maximum on the bits (non-negative floats order like their bits)
        const unsigned m = __reduce_max_sync(0xffffffffu, act ? __float_as_uint(a) : 0u);
        if (lane == 0) atomicMax(mx + (t - t0), m);
        r0 = r1; c0 = c1; r1 = r2; c1 = c2; r2 = r3; c2 = c3;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < t1 - t0; t += blockDim.x) atomicMax(M + t0 + t, mx[t]);
}

// ---------------------------------------------------------------------------
// NCC + regional peaks.  CTA = (row strip of NCC_RS rows, plane).  NCC via
// separable 1D correlations (Fig. 1g):
//   s1 = box(A), s2 = box(A^2), sg = (g_z x g_l) * A,
//   NCC = (sg - mu_G s1) / sqrt((s2 - s1^2 / d^2) * ss_G),
// computed on the strip plus one row above and below for the 3x3 test.
// Candidates are compacted in raster order into a fixed-capacity slot of
// the strip; the true count is kept.
//
// Box sums by split points: for a run of B <= d consecutive outputs every
// window contains the run's last first-row m, so
//   box(r) = Suf(r) + Pre(r + d - 1),  Suf(r) = x_r + ... + x_{m-1},
//   Pre(k) = x_m + ... + x_k,
// about three adds per output instead of d, and every output is the sum of
// two partial sums over its own window only (no running sum carries the
// rounding of values that have left the window).  The Gaussian-weighted sums
// keep their d taps.
//
// Vertical pass first, on column pairs (one 64-bit shared load gives two
// columns of an input row; thread task = column pair x VB output rows); its
// three sums are stored transposed into row pairs, so the horizontal pass
// works on two output rows at once (thread task = row pair x HB output
// columns).  Thread-to-data maps keep both passes free of bank conflicts:
// consecutive lanes take consecutive column pairs in the vertical pass and
// consecutive row pairs (row-pair stride of N + 1 pairs) in the horizontal
// pass.
// ---------------------------------------------------------------------------
#define NCC_THREADS 256   // 128 for planes of up to 64 columns, whose passes have no more tasks

// float2 columns of one padded vertical-sum row pair (see k_detect)
__host__ __device__ inline int det_npad(int N, int H, int HB)
{
    const int w = (N + HB - 1) / HB * HB + 2 * H;
    return w | 1;
}
__host__ __device__ inline int det_hb(int H) { return H >= 4 ? 8 : 2 * H; }

// split-point box sums of NB consecutive outputs from the NB + 2H inputs
// in[0 ..]: out[r] = in[r] + ... + in[r + 2H]  (NB <= 2H + 1)
template <int H, int NB, typename LOAD>
__device__ __forceinline__ void split_box(LOAD in, uint64_t (&out)[NB])
{
    static_assert(NB >= 1 && NB <= 2 * H + 1, "a run of outputs must share a split row");
    constexpr int m = NB - 1;
    uint64_t suf[NB];
    if constexpr (m >= 1) {
        suf[m - 1] = in(m - 1);
#pragma unroll
        for (int k = m - 2; k >= 0; --k) suf[k] = f2_add(in(k), suf[k + 1]);
    }
    uint64_t pre = in(m);
#pragma unroll
    for (int k = m + 1; k <= m + 2 * H; ++k) {
        pre = f2_add(pre, in(k));
        const int r = k - 2 * H;
        if (r >= 0) out[r] = r < m ? f2_add(suf[r], pre) : pre;
    }
}

// the count of candidate slot s: kept in full, added to the kept total of its
// chunk of GATHER_SLOTS slots (for the gather's offsets), to the true total and,
// what does not fit the slot, to the dropped total (total[1])
__device__ __forceinline__ void slot_count(int* __restrict__ cnt, int* __restrict__ part,
                                           unsigned long long* __restrict__ total, int s, int n, unsigned* __restrict__ status)
{
    cnt[s] = n;
    if (n > 0) {
        atomicAdd(part + s / GATHER_SLOTS, min(n, CAND_CAP));
        atomicAdd(total, (unsigned long long)n);
    }
    if (n > CAND_CAP) {
        atomicAdd(total + 1, (unsigned long long)(n - CAND_CAP));
        atomicOr(status, ST_CAPACITY);
    }
}

// Whether NCC row ro, column l of the NCC rows sN is a 3 x 3 regional maximum.
__device__ __forceinline__ bool ncc_peak(const float* __restrict__ sN, int NS, int ro, int l)
{
    const float c = sN[ro * NS + l];
    bool pk = true;
#pragma unroll
    for (int a = -1; a <= 1; ++a)
#pragma unroll
        for (int b = -1; b <= 1; ++b) {
            if (a == 0 && b == 0) continue;
            const float v = sN[(ro + a) * NS + l + b];
            const bool earlier = (a < 0) || (a == 0 && b < 0);
            pk = pk && (earlier ? (c > v) : (c >= v));
        }
    return pk;
}

// NT threads run the two correlation passes; one warp more serves them: it fetches
// the strips, and while the others are at the next strip it tests the last one's
// few pixels over the thresholds and writes the peaks.  (With all threads walking
// the pixels for peaks, compacting and fetching between barriers, the paper's 300
// frames at d = 11 took 1.40 ms, now 1.18.)  What is left is the two passes: issue
// slots half used, the barriers after either pass the largest stall.
#define DET_LIST 1024   // pixels over the thresholds that the serving warp takes; beyond, all threads test
template <int H, int NC, int NT>
__global__ void __launch_bounds__(NT + 32, 512 / NT) k_detect(const float* __restrict__ A, const float* __restrict__ Mf,
                                                          int S, int nz, int Nrt, int nplanes, NccConst nc,
                                                          ulm_loc2d* __restrict__ cand, int* __restrict__ cnt,
                                                          int* __restrict__ part, unsigned long long* __restrict__ total,
                                                          float* __restrict__ ncc_out, unsigned* __restrict__ status)
{
    constexpr int D = 2 * H + 1;
    constexpr int RN = NCC_RS + 2;          // NCC rows: the strip and one row above and below
    constexpr int RP = RN / 2;              // row pairs
    constexpr int VB = H >= 4 ? 8 : (H >= 2 ? 4 : 2);   // output rows per vertical task
    constexpr int HB = H >= 4 ? 8 : 2 * H;  // output columns per horizontal task (det_hb)
    constexpr int NW = (NCC_RS * 256 + 31) / 32;   // bitmap words of the strip's pixels (N <= 256)
    static_assert(RN % VB == 0 && VB % 2 == 0 && VB <= D, "vertical runs must tile the NCC rows in pairs");
    const int N = NC > 0 ? NC : Nrt;        // lateral pixels (compile-time for the usual widths)
    extern __shared__ __align__(128) float sm[];
    const int nstrip = (nz + NCC_RS - 1) / NCC_RS;
    const int items = nplanes * nstrip;
    const int rin = RN + 2 * H;
    // columns of a padded vertical-sum row pair: column c at c + H, zero pads on
    // both sides, room for the last horizontal block's overhang, odd (conflict-free)
    const int NPAD = det_npad(N, H, HB);
    const int VS = 2 * NPAD;                // floats per row pair of a vertical-sum array
    const int NS = N + 1;                   // NCC row stride
    const size_t abuf = max((size_t)rin * N, (size_t)RN * NS);
    // sm + bb abuf (bb = 0, 1): [rin][N] amplitude rows i0-1-H ..., double-buffered
    float* sV = sm + 2 * abuf;              // [3][RP][NPAD][2]; column c at c + H
    // [RN][N] flags A >= alpha M_t of the NCC rows' pixels, set by the vertical pass
    // (which holds the amplitudes), so that the horizontal pass reads no global memory
    unsigned char* aflag = reinterpret_cast<unsigned char*>(sV + (size_t)3 * RP * NPAD * 2);
    // of the items of either buffer: the pixels with NCC >= ncc_min and their flag set,
    // in no order; their peaks, in raster order
    __shared__ unsigned short list[2][DET_LIST];
    __shared__ unsigned bits[2][NW];
    __shared__ unsigned short order[CAND_CAP];
    __shared__ int nlist[2];
    __shared__ uint64_t full[2], done[2];   // rows fetched; NCC rows and list complete
    const int nwords = (NCC_RS * N + 31) / 32;
    if (threadIdx.x == 0) {
        for (int q = 0; q < 2; ++q) {
            mbar_init(&full[q], 1);
            mbar_init(&done[q], NT / 32);   // one arrival per warp: an arrival is a serialised access
            nlist[q] = 0;
        }
        mbar_fence_init();
    }
    for (int idx = threadIdx.x; idx < 2 * NW; idx += blockDim.x) bits[idx / NW][idx % NW] = 0u;
    {
        const int npad = NPAD - N;          // H on the left, the rest on the right
        for (int idx = threadIdx.x; idx < 3 * RP * npad; idx += blockDim.x) {
            const int ar = idx / npad, q = idx - ar * npad;
            const int col = q < H ? q : N + q;
            reinterpret_cast<float2*>(sV)[(size_t)ar * NPAD + col] = make_float2(0.f, 0.f);
        }
    }
    __syncthreads();
    grid_wait();
    if (threadIdx.x >= NT) {
        // ---- serving warp
        const int lane = threadIdx.x - NT;
        // rows [i0-1-H, i0+NCC_RS+1+H) of item `it`'s plane into buffer bb: zero
        // outside the plane, one bulk copy inside
        auto fetch = [&](int it, int bb) {
            const int plane = it / nstrip, strip = it - plane * nstrip;
            const int rlo = strip * NCC_RS - 1 - H;
            const int lo = max(rlo, 0), hi = max(lo, min(rlo + rin, nz));
            const int z0 = min(lo - rlo, rin), z1 = hi - rlo;
            float* sA = sm + bb * abuf;
            for (int idx = lane; idx < z0 * N; idx += 32) sA[idx] = 0.f;
            for (int idx = lane; idx < (rin - z1) * N; idx += 32) sA[(size_t)z1 * N + idx] = 0.f;
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
                // the copied rows land inside the buffer's rin rows (checked build; else nothing is copied)
                const bool in = chk(lo >= rlo && hi - rlo <= rin && plane < nplanes, status);
                const unsigned bytes = in ? (unsigned)((hi - lo) * N * sizeof(float)) : 0u;
                mbar_arrive_expect_tx(&full[bb], bytes);
                if (bytes)
                    bulk_g2s(sA + (size_t)(lo - rlo) * N, A + ((size_t)plane * nz + lo) * N, bytes, &full[bb]);
            }
            __syncwarp();
        };
        const int stride = gridDim.x;
        int fetched = 0;                    // items fetched so far
        for (int it = blockIdx.x; it < items && fetched < 2; it += stride, ++fetched) fetch(it, fetched);
        int k = 0;
        for (int it = blockIdx.x; it < items; it += stride, ++k) {
            const int bb = k & 1;
            if (!mbar_wait_bounded(&done[bb], (unsigned)(k >> 1) & 1u)) {
                if (lane == 0) atomicOr(status, ST_TIMEOUT);
                break;
            }
            const float* sN = sm + bb * abuf;
            const int plane = it / nstrip, strip = it - plane * nstrip;
            const int t = plane / (2 * S), axis = (plane / S) % 2, b = plane % S, i0 = strip * NCC_RS;
            const int n_over = nlist[bb];
            if (n_over <= DET_LIST)
                for (int q = lane; q < n_over; q += 32) {
                    const int p = list[bb][q], ro = 1 + p / N;
                    if (ncc_peak(sN, NS, ro, p - (ro - 1) * N) && chk((p >> 5) < NW && ro + 1 < RN, status))
                        atomicOr(&bits[bb][p >> 5], 1u << (p & 31));
                }
            __syncwarp();
            // lane: a run of bitmap words; their counts scanned over the warp
            const int wpl = (nwords + 31) / 32, w0 = lane * wpl, w1 = min(nwords, w0 + wpl);
            int x = 0;
            for (int w = w0; w < w1; ++w) x += __popc(bits[bb][w]);
            int before = -x;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            before += x;
            if (lane == 31) slot_count(cnt, part, total, it, x, status);
            for (int w = w0; w < w1; ++w) {
                unsigned m = bits[bb][w];
                bits[bb][w] = 0u;
                for (; m; m &= m - 1, ++before)
                    if (before < CAND_CAP) order[before] = (unsigned short)(w * 32 + __ffs(m) - 1);
            }
            __syncwarp();
            const int npk = min(__shfl_sync(0xffffffffu, x, 31), CAND_CAP);
            for (int q = lane; q < npk; q += 32) {
                const int p = order[q], ro = 1 + p / N, l = p - (ro - 1) * N, i = i0 - 1 + ro;
                const float c = sN[ro * NS + l];
                auto para = [](float fm, float f0, float fp) {
                    const float den = fm - 2.f * f0 + fp;
                    if (den >= 0.f) return 0.f;
                    const float dl = (fm - fp) / (2.f * den);
                    return fminf(0.5f, fmaxf(-0.5f, dl));
                };
                ulm_loc2d e;
                e.frame = t;
                e.axis = axis;
                e.slab = b;
                e.iz = i;
                e.ilat = l;
                e.z = (float)i + para(sN[(ro - 1) * NS + l], c, sN[(ro + 1) * NS + l]);
                e.lat = (float)l + para(sN[ro * NS + l - 1], c, sN[ro * NS + l + 1]);
                e.ncc = c;
                e.amp = 0.f;        // filled from A by the gather
                e.reserved = 0;
                cand[(size_t)it * CAND_CAP + q] = e;
            }
            if (lane == 0) nlist[bb] = 0;
            __syncwarp();
            // the buffer, its list and its bitmap are free: the item after the next
            if (it + 2 * stride < items) {
                fetch(it + 2 * stride, bb);
                ++fetched;
            }
        }
        // a wait ran out: the copies in flight end (bounded) before the block may
        for (int q = k; q < fetched; ++q) mbar_wait_bounded(&full[q & 1], (unsigned)(q >> 1) & 1u);
    } else {
        // packed Gaussian taps, held for every item
        uint64_t gz[D], gl[D];
#pragma unroll
        for (int q = 0; q < D; ++q) {
            gz[q] = f2_pack(nc.gz[q], nc.gz[q]);
            gl[q] = f2_pack(nc.gl[q], nc.gl[q]);
        }
        int k = 0;
        // strip, plane of its frame and frame of the item, advanced without divisions
        const int dstrip = gridDim.x % nstrip, dpl = gridDim.x / nstrip % (2 * S), dt = gridDim.x / nstrip / (2 * S);
        int strip = blockIdx.x % nstrip, pl = blockIdx.x / nstrip % (2 * S), t = blockIdx.x / nstrip / (2 * S);
        float Mnext = blockIdx.x < items ? __ldg(Mf + t) : 0.f;
        for (int it = blockIdx.x; it < items; it += gridDim.x, ++k) {
            const int bb = k & 1;
            const float Mt = Mnext;
            const int plane = t * 2 * S + pl, i0 = strip * NCC_RS;
            strip += dstrip, pl += dpl, t += dt;
            if (strip >= nstrip) strip -= nstrip, ++pl;
            if (pl >= 2 * S) pl -= 2 * S, ++t;
            if (it + (int)gridDim.x < items) Mnext = __ldg(Mf + t);
            const int late = !mbar_wait_bounded(&full[bb], (unsigned)(k >> 1) & 1u);
            float* sA = sm + bb * abuf;
            float* sN = sA;                     // NCC rows over the amplitude rows once the vertical pass is done
            const float athr = nc.alpha * Mt;
            // NCC rows whose plane row i = i0 - 1 + ro lies in [1, nz - 2]
            const int ro_lo = max(1, 2 - i0), ro_hi = min(NCC_RS, nz - 1 - i0);
            // ---- vertical pass: thread = (column pair, VB output rows)
            {
                const int NP = N / 2;
                const unsigned sAa = smem_u32(sA), sVa = smem_u32(sV);
                for (int task = threadIdx.x; task < NP * (RN / VB); task += NT) {
                    const int cp = task % NP, rb = task / NP;
                    const int ro0 = rb * VB;
                    // NCC rows ro0 .. ro0 + VB - 1 use amplitude rows ro0 .. ro0 + VB - 1 + 2H
                    uint64_t x[VB + 2 * H];
                    const unsigned src = sAa + (unsigned)((ro0 * N + 2 * cp) * 4);
#pragma unroll
                    for (int m = 0; m < VB + 2 * H; ++m) x[m] = lds_u64(src + (unsigned)(m * N * 4));
#pragma unroll
                    for (int r = 0; r < VB; ++r) {
                        // the centre amplitude of NCC row ro0 + r, both columns of the pair
                        const float2 ac = f2_unpack(x[r + H]);
                        const unsigned short fl = (unsigned short)((ac.x >= athr ? 1u : 0u) | (ac.y >= athr ? 0x100u : 0u));
                        if (chk((ro0 + r) * N + 2 * cp + 1 < RN * N, status))
                            *reinterpret_cast<unsigned short*>(aflag + (ro0 + r) * N + 2 * cp) = fl;
                    }
                    uint64_t v1[VB], v2[VB], vg[VB];
                    split_box<H, VB>([&](int q) { return x[q]; }, v1);
                    split_box<H, VB>([&](int q) { return f2_mul(x[q], x[q]); }, v2);
#pragma unroll
                    for (int r = 0; r < VB; ++r) {
                        uint64_t a = f2_mul(gz[0], x[r]);
#pragma unroll
                        for (int q = 1; q < D; ++q) a = f2_fma(gz[q], x[r + q], a);
                        vg[r] = a;
                    }
                    // transpose 2 x 2 blocks into row pairs: [arr][rp][H + column][row parity]
                    const unsigned dst0 = sVa + (unsigned)(((ro0 / 2) * VS + 2 * (2 * cp + H)) * 4);
#pragma unroll
                    for (int j = 0; j < VB; j += 2) {
                        const uint64_t* arrs[3] = {v1, v2, vg};
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            const float2 r0 = f2_unpack(arrs[a][j]), r1 = f2_unpack(arrs[a][j + 1]);
                            const unsigned dst = dst0 + (unsigned)(((a * RP + j / 2) * VS) * 4);
                            asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(dst), "f"(r0.x), "f"(r1.x) : "memory");
                            asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(dst + 8u), "f"(r0.y), "f"(r1.y) : "memory");
                        }
                    }
                }
            }
            // the vertical sums are complete; every thread's wait for the rows succeeded
            int any;
            asm volatile(
                "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 q, %1, 0;\n\tbarrier.cta.red.or.pred p, 1, %2, q;\n\tselp.s32 %0, 1, 0, p;\n\t}"
                : "=r"(any)
                : "r"(late), "n"(NT)
                : "memory");
            if (any) {
                if (threadIdx.x == 0) atomicOr(status, ST_TIMEOUT);
                break;
            }
            // ---- horizontal pass + NCC: thread = (row pair, HB output columns);
            // the amplitude rows are no longer read, so the NCC rows take their place
            {
                const float flat = nc.flat_coef * Mt * Mt;
                const float inv_d2 = 1.0f / (float)(D * D);
                const int ncb = (N + HB - 1) / HB;
                const uint64_t nid2 = f2_pack(-inv_d2, -inv_d2), nmu = f2_pack(-nc.muG, -nc.muG);
                const unsigned sVa = smem_u32(sV);
                for (int task = threadIdx.x; task < RP * ncb; task += NT) {
                    const int rp = task % RP, cb = task / RP;
                    const int c0 = cb * HB;
                    // padded input columns c0 - H .. c0 + HB - 1 + H start at pad index c0; past N they
                    // read the right pad (zero) or feed only outputs past N
                    const unsigned at = sVa + (unsigned)((rp * VS + 2 * c0) * 4);
                    uint64_t s1[HB], s2[HB], sg[HB];
                    {
                        uint64_t a[HB + 2 * H];
#pragma unroll
                        for (int m = 0; m < HB + 2 * H; ++m) a[m] = lds_u64(at + (unsigned)(m * 8));
                        split_box<H, HB>([&](int q) { return a[q]; }, s1);
#pragma unroll
                        for (int m = 0; m < HB + 2 * H; ++m) a[m] = lds_u64(at + (unsigned)(RP * VS * 4 + m * 8));
                        split_box<H, HB>([&](int q) { return a[q]; }, s2);
#pragma unroll
                        for (int m = 0; m < HB + 2 * H; ++m) a[m] = lds_u64(at + (unsigned)(2 * RP * VS * 4 + m * 8));
#pragma unroll
                        for (int r = 0; r < HB; ++r) {
                            uint64_t g = f2_mul(gl[0], a[r]);
#pragma unroll
                            for (int q = 1; q < D; ++q) g = f2_fma(gl[q], a[r + q], g);
                            sg[r] = g;
                        }
                    }
                    const int ia = i0 - 1 + 2 * rp;    // plane row of the pair's first row
                    const bool row0 = ia >= H && ia < nz - H && Mt > 0.f;
                    const bool row1 = ia + 1 >= H && ia + 1 < nz - H && Mt > 0.f;
                    float* nrow = sN + (2 * rp) * NS + c0;
                    unsigned over = 0u;                // pixels with NCC >= ncc_min: bits j (first row) and HB + j
#pragma unroll
                    for (int j = 0; j < HB; ++j) {
                        const int c = c0 + j;
                        if (c >= N) break;
                        // ssA = s2 - s1^2 / d^2, numerator = sg - mu_G s1 (both rows of the pair)
                        const float2 ss = f2_unpack(f2_fma(f2_mul(s1[j], s1[j]), nid2, s2[j]));
                        const float2 nu = f2_unpack(f2_fma(nmu, s1[j], sg[j]));
                        const bool colok = c >= H && c < N - H;
                        const float v0 = (colok && row0 && ss.x > flat) ? nu.x * nc.inv_ssG_sqrt * rsqrtf(ss.x) : 0.f;
                        const float v1 = (colok && row1 && ss.y > flat) ? nu.y * nc.inv_ssG_sqrt * rsqrtf(ss.y) : 0.f;
                        nrow[j] = v0;
                        nrow[NS + j] = v1;
                        if (v0 >= nc.ncc_min) over |= 1u << j;
                        if (v1 >= nc.ncc_min) over |= 1u << (HB + j);
                        if (ncc_out) {
                            if (2 * rp >= 1 && 2 * rp <= NCC_RS && ia < nz) ncc_out[((size_t)plane * nz + ia) * N + c] = v0;
                            if (2 * rp + 1 <= NCC_RS && ia + 1 < nz) ncc_out[((size_t)plane * nz + ia + 1) * N + c] = v1;
                        }
                    }
                    // the rows and columns a peak may lie in
                    constexpr unsigned RM = (1u << HB) - 1u;
                    if (2 * rp < ro_lo || 2 * rp > ro_hi) over &= ~RM;
                    if (2 * rp + 1 < ro_lo || 2 * rp + 1 > ro_hi) over &= RM;
                    if (c0 == 0) over &= ~(1u | 1u << HB);
                    if (c0 + HB >= N) over &= ~(1u << (N - 1 - c0) | 1u << (HB + N - 1 - c0));
                    while (over) {
                        const int bit = __ffs(over) - 1;
                        over &= over - 1;
                        const int ro = 2 * rp + (bit >= HB), l = c0 + (bit >= HB ? bit - HB : bit);
                        if (!aflag[ro * N + l]) continue;
                        const int at = atomicAdd(&nlist[bb], 1);
                        if (at < DET_LIST) list[bb][at] = (unsigned short)((ro - 1) * N + l);
                    }
                }
            }
            asm volatile("barrier.cta.sync 1, %0;" ::"n"(NT) : "memory");
            if (nlist[bb] > DET_LIST) {
                // many pixels over the thresholds: every thread tests the strip's pixels
                constexpr int MAXL = NT;
                const int RG = MAXL / N > 0 ? MAXL / N : 1;
                for (int l = threadIdx.x % min(N, MAXL); l < N; l += MAXL)
                    for (int ro = ro_lo + (N < MAXL ? threadIdx.x / N : 0); ro <= ro_hi; ro += RG)
                        if ((N >= MAXL || threadIdx.x / N < RG) && l >= 1 && l < N - 1 && sN[ro * NS + l] >= nc.ncc_min &&
                            aflag[ro * N + l] && ncc_peak(sN, NS, ro, l)) {
                            const int p = (ro - 1) * N + l;
                            if (chk(p >= 0 && (p >> 5) < NW && ro + 1 < RN, status)) atomicOr(&bits[bb][p >> 5], 1u << (p & 31));
                        }
                // the flags are overwritten by the next item's vertical pass
                asm volatile("barrier.cta.sync 1, %0;" ::"n"(NT) : "memory");
            }
            __syncwarp();
            if ((threadIdx.x & 31) == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&done[bb])) : "memory");
        }
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int q = 0; q < 2; ++q) {
            mbar_inval(&full[q]);
            mbar_inval(&done[q]);
        }
}

// ---------------------------------------------------------------------------
// Peaks of score maps on a finer grid (the learned localiser's heatmaps).
// CTA = (strip of DET_RS fine rows, plane); same raster-order compaction as
// k_detect.  Positions are converted to plane pixels for pairing.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_detect_map(const float* __restrict__ map, int up, const float* __restrict__ A,
                                                    const float* __restrict__ Mf, int S, int nz, int N, float score_min,
                                                    float alpha, ulm_loc2d* __restrict__ cand, int* __restrict__ cnt,
                                                    int* __restrict__ part, unsigned long long* __restrict__ total,
                                                    unsigned* __restrict__ status)
{
    grid_wait();
    extern __shared__ __align__(128) float smf[];
    __shared__ int wsum[32];
    __shared__ uint64_t bar;
    const int H4 = nz * up, W4 = N * up;
    const int strip = blockIdx.x, plane = blockIdx.y, nstrip = gridDim.x;
    const int t = plane / (2 * S), axis = (plane / S) % 2, b = plane % S;
    const int i0 = strip * DET_RS, rin = DET_RS + 2;
    const float* mp = map + (size_t)plane * H4 * W4;
    const float* Ap = A + (size_t)plane * nz * N;
    const float Mt = Mf[t];
    {
        const int rlo = i0 - 1;
        const int lo = max(rlo, 0), hi = max(lo, min(rlo + rin, H4));
        if (threadIdx.x == 0) {
            mbar_init(&bar, 1);
            mbar_fence_init();
        }
        __syncthreads();
        const int z0 = min(lo - rlo, rin), z1 = hi - rlo;
        for (int idx = threadIdx.x; idx < z0 * W4; idx += blockDim.x) smf[idx] = 0.f;
        for (int idx = threadIdx.x; idx < (rin - z1) * W4; idx += blockDim.x) smf[(size_t)z1 * W4 + idx] = 0.f;
        if (threadIdx.x == 0) {
            fence_proxy_async();
            const unsigned bytes = (unsigned)((hi - lo) * W4 * sizeof(float));
            mbar_arrive_expect_tx(&bar, bytes);
            if (bytes) bulk_g2s(smf + (size_t)(lo - rlo) * W4, mp + (size_t)lo * W4, bytes, &bar);
        }
        if (!cta_wait_copies(&bar, 0, status)) return;
    }
    const float athr = alpha * Mt;
    ulm_loc2d* slot = cand + ((size_t)plane * nstrip + strip) * CAND_CAP;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int npx = DET_RS * W4;
    const int nwords = (npx + 31) / 32;
    // candidate bitmap of the strip's pixels in raster order (cleared, then set by
    // the test: consecutive lanes take consecutive pixels, conflict-free on the rows)
    unsigned* bits = reinterpret_cast<unsigned*>(smf + (size_t)rin * W4);
    for (int w = threadIdx.x; w < nwords; w += blockDim.x) bits[w] = 0u;
    __syncthreads();
    // rows in turn, consecutive lanes on consecutive columns (no division per pixel)
    const int ro_lo = max(1, 2 - i0), ro_hi = min(DET_RS, H4 - 1 - i0);   // rows with 1 <= i <= H4 - 2
    for (int ro = ro_lo; ro <= ro_hi; ++ro) {
#pragma unroll 2
        for (int j = threadIdx.x; j < W4; j += blockDim.x) {
            const int i = i0 - 1 + ro, p = (ro - 1) * W4 + j;
            if (j < 1 || j >= W4 - 1) continue;
            const float c = smf[ro * W4 + j];
            if (!(c >= score_min)) continue;
            bool pk = true;
#pragma unroll
            for (int a = -1; a <= 1; ++a)
#pragma unroll
                for (int bb = -1; bb <= 1; ++bb) {
                    if (a == 0 && bb == 0) continue;
                    const float q = smf[(ro + a) * W4 + j + bb];
                    const bool earlier = (a < 0) || (a == 0 && bb < 0);
                    pk = pk && (earlier ? (c > q) : (c >= q));
                }
            // the amplitude (global memory) only for regional maxima
            if (pk && Ap[(size_t)(i / up) * N + j / up] >= athr) atomicOr(&bits[p >> 5], 1u << (p & 31));
        }
    }
    __syncthreads();
    // compaction: consecutive bitmap words per thread, a block-wide exclusive scan of their counts
    const int wpt = (nwords + blockDim.x - 1) / blockDim.x;
    const int w0 = threadIdx.x * wpt, w1 = min(nwords, w0 + wpt);
    int mine = 0;
    for (int w = w0; w < w1; ++w) mine += __popc(bits[w]);
    int x = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    int before = x - mine;
    for (int w = 0; w < warp; ++w) before += wsum[w];
    const float half = 0.5f * (float)(up - 1), inv = 1.f / (float)up;
    for (int w = w0; w < w1; ++w) {
        unsigned m = bits[w];
        while (m) {
            const int bit = __ffs(m) - 1;
            m &= m - 1;
            if (before < CAND_CAP) {
                const int p = w * 32 + bit;
                const int ro = 1 + p / W4, j = p - (ro - 1) * W4, i = i0 - 1 + ro;
                const float c = smf[ro * W4 + j];
                auto para = [](float fm, float f0, float fp) {
                    const float den = fm - 2.f * f0 + fp;
                    if (den >= 0.f) return 0.f;
                    const float dl = (fm - fp) / (2.f * den);
                    return fminf(0.5f, fmaxf(-0.5f, dl));
                };
                ulm_loc2d e;
                e.frame = t;
                e.axis = axis;
                e.slab = b;
                e.iz = i / up;
                e.ilat = j / up;
                e.z = ((float)i + para(smf[(ro - 1) * W4 + j], c, smf[(ro + 1) * W4 + j]) - half) * inv;
                e.lat = ((float)j + para(smf[ro * W4 + j - 1], c, smf[ro * W4 + j + 1]) - half) * inv;
                e.ncc = c;
                e.amp = Ap[(size_t)e.iz * N + e.ilat];
                e.reserved = 0;
                slot[before] = e;
            }
            ++before;
        }
    }
    // the last thread's running index is the strip's count
    if (threadIdx.x == blockDim.x - 1) slot_count(cnt, part, total, plane * nstrip + strip, before, status);
}

#define SCAN_MAX (1024 * 4096)   // entries of one compaction at most

// sum over the block of part[0 .. n) plus `own` of every thread before this one:
// the exclusive offset of this thread's first entry; *all: the sum with every
// thread's own (256 threads)
__device__ __forceinline__ int block_offset(const int* __restrict__ part, int n, int own, int* red, int* all)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int p = 0, x = own;
    for (int q = threadIdx.x; q < n; q += blockDim.x) p += part[q];
    p = __reduce_add_sync(0xffffffffu, p);
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();                                   // red is free
    if (lane == 31) red[warp] = x, red[8 + warp] = p;
    __syncthreads();
    int before = 0, sum = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        before += red[8 + w];
        sum += red[w] + red[8 + w];
        if (w < warp) before += red[w];
    }
    *all = sum;
    return before + x - own;
}

// Copy the kept candidates of a chunk of slots to their place in the output list:
// the chunk's offset is the sum of the totals before it, a slot's a scan of the
// counts in the block (one launch instead of three scan kernels and a gather), and
// the chunk's entries are spread over the threads of gridDim.y blocks, which scan
// alike (slots_gather's rule).  A non-null: each entry's amplitude is read here from
// A [plane][nz][N] at its pixel (the detection kernel leaves it to this highly
// parallel pass).  poff (optional): the list offset of
// every plane, of nstrip slots each.  Where slots dropped candidates, the count
// goes past the entries kept; what it covers beyond them becomes entries of frame F,
// which sort last and pair with nothing, so that a list is in order over its count
// (with whatever the buffer held there, the pairing's plane offsets were wrong and
// its searches ran over the whole list: 58 ms instead of 0.58 for a count of 1.31 million, 0.49 million kept).
__global__ void __launch_bounds__(256) k_gather(const ulm_loc2d* __restrict__ cand, const int* __restrict__ cnt,
                                                const int* __restrict__ part, const unsigned long long* __restrict__ total,
                                                int nslots, int nstrip, ulm_loc2d* __restrict__ out, int cap,
                                                int* __restrict__ n_out, int* __restrict__ poff, const float* __restrict__ A,
                                                int S, int nz, int N, unsigned* __restrict__ status)
{
    grid_wait();
    static_assert(GATHER_SLOTS == 256, "a thread per slot");
    __shared__ int red[16], off[GATHER_SLOTS + 1];
    const int s0 = blockIdx.x * GATHER_SLOTS, s = s0 + threadIdx.x;
    const int own = s < nslots ? min(cnt[s], CAND_CAP) : 0;
    int all;
    const int at = block_offset(part, blockIdx.x, own, red, &all);
    off[threadIdx.x] = at;
    if (threadIdx.x == 0) off[GATHER_SLOTS] = all;
    if (poff && blockIdx.y == 0) {
        if (s < nslots && s % nstrip == 0) poff[s / nstrip] = at;
        if (s == nslots - 1) poff[nslots / nstrip] = at + own;
    }
    const int turn = 256 * gridDim.y, first = 256 * blockIdx.y + threadIdx.x;
    if (blockIdx.x == 0 && first == 0) *n_out = (int)min(*total, 0x7fffffffull);
    if (total[1] != 0) {
        // word by word: entry by entry (40 bytes a lane) took ten times as long
        constexpr int EW = sizeof(ulm_loc2d) / 4;
        const int F = nslots / nstrip / (2 * S);
        int* w = reinterpret_cast<int*>(out);
        const long long end = (long long)min(*total, (unsigned long long)cap) * EW;
        for (long long i = (long long)(*total - total[1]) * EW + blockIdx.x * turn + first; i < end; i += turn * gridDim.x)
            w[i] = i % EW == offsetof(ulm_loc2d, frame) / 4 ? F : 0;
    }
    __syncthreads();
    const int base = off[0], n = all - base;
    for (int i = first; i < n; i += turn) {
        const int dst = base + i;
        if (dst >= cap) {
            atomicOr(status, ST_CAPACITY);
            break;
        }
        int lo = 0;                                    // the last slot with off <= dst
#pragma unroll
        for (int h = GATHER_SLOTS / 2; h > 0; h >>= 1)
            if (off[lo + h] <= dst) lo += h;
        ulm_loc2d e = cand[(size_t)(s0 + lo) * CAND_CAP + (dst - off[lo])];
        if (A && chk(e.iz >= 0 && e.iz < nz && e.ilat >= 0 && e.ilat < N && e.slab >= 0 && e.slab < S &&
                         (unsigned)((e.frame * 2 + e.axis) * S + e.slab) < (unsigned)(nslots / nstrip), status))
            e.amp = __ldg(A + (((size_t)(e.frame * 2 + e.axis) * S + e.slab) * nz + e.iz) * N + e.ilat);
        out[dst] = e;
    }
}

// ---------------------------------------------------------------------------
// pairing
// ---------------------------------------------------------------------------
__device__ __forceinline__ int plane_key(const ulm_loc2d& e, int S) { return (e.frame * 2 + e.axis) * S + e.slab; }

__global__ void k_list_plane_offsets(const ulm_loc2d* __restrict__ L, const int* __restrict__ n2d, int cap2d, int S,
                                     int nplanes, int* __restrict__ poff)
{
    grid_wait();
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p > nplanes) return;
    int n = min(*n2d, cap2d);
    int lo = 0, hi = n;  // first index with key >= p
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (plane_key(L[mid], S) < p) lo = mid + 1;
        else hi = mid;
    }
    poff[p] = lo;
}

// XZ / YZ eligibility and cost in double precision: same frame and
// sub-block, |dz| <= 1 pixel, ratio I_xz / I_yz in [0.9, 1.11];
// cost max(I) / min(I) (orders pairs like |ln ratio|).
// The decisions are those of FP64 arithmetic on the FP32 inputs (the oracle's).
// GB300's FP64 rate is low, so each test is first taken in FP32 where that
// provably gives the same answer (rounding to nearest is monotonic, so
// fl32(e) > 1 implies e > 1 and fl32(e) < 1 implies e < 1; a ratio more than
// 0.01 inside or outside a bound is on the same side in FP64), and in FP64
// only when the FP32 value sits at the bound.
__device__ __forceinline__ bool pair_ok(const ulm_loc2d& x, const ulm_loc2d& y, int P)
{
    if (x.frame != y.frame) return false;
    // x.ilat / P == y.slab and y.ilat / P == x.slab (non-negative indexes), without divisions
    const int xl = y.slab * P, yl = x.slab * P;
    if (x.ilat < xl || x.ilat >= xl + P || y.ilat < yl || y.ilat >= yl + P) return false;
    const float dz = fabsf(x.z - y.z);
    if (dz > 1.0f) return false;
    if (dz == 1.0f && fabs((double)x.z - (double)y.z) > 1.0) return false;
    const float r32 = x.amp / y.amp;
    const bool lo_sure = r32 >= 0.91f, hi_sure = r32 <= 1.10f;
    if (r32 <= 0.89f || r32 >= 1.12f || !(r32 == r32)) return false;
    const double ax = x.amp, ay = y.amp;
    if (!(lo_sure && hi_sure)) {
        const double r = ax / ay;
        if (!(r >= 0.9 && r <= 1.11)) return false;
    }
    return true;
}

// whether partner p (amplitude pa) of an entry of amplitude a beats partner q (qa):
// the lower FP64 cost max / min, ties to the lower index.  The FP32 costs (1 to 1.12,
// within 1.4e-7 of the quotient) decide unless they are closer than 4e-7.
__device__ __forceinline__ bool pair_better(float a, int p, float pa, int q, float qa)
{
    const float c = a > pa ? a / pa : pa / a, d = a > qa ? a / qa : qa / a;
    if (c < d - 4e-7f) return true;
    if (c > d + 4e-7f) return false;
    const double A = a, C = pa, D = qa;
    const double c64 = A > C ? A / C : C / A, d64 = A > D ? A / D : D / A;
    return c64 < d64 || (c64 == d64 && p < q);
}

// The partner of entry e: the eligible entry of the least cost in the plane of its
// slab's counterpart on the other axis, ties to the lower index (0x7fffffff: none, or
// !act).  LANES consecutive lanes share an entry.
template <int LANES>
__device__ __forceinline__ int pair_search(const ulm_loc2d* __restrict__ L, int n, const ulm_loc2d& e, bool act, int F, int S,
                                           int P, const int* __restrict__ poff)
{
    int b = 0x7fffffff;
    float pa = 0.f;
    const int slab = e.ilat / P;
    if (act && (unsigned)e.axis < 2u && e.frame >= 0 && e.frame < F && e.ilat >= 0 && slab < S) {
        const int pl = (e.frame * 2 + 1 - e.axis) * S + slab;
        const int q1 = min(poff[pl + 1], n);
        for (int q = poff[pl] + (int)(threadIdx.x % LANES); q < q1; q += LANES) {
            const ulm_loc2d y = L[q];
            if ((e.axis == 0 ? pair_ok(e, y, P) : pair_ok(y, e, P)) &&
                (b == 0x7fffffff || pair_better(e.amp, q, y.amp, b, pa))) {
                b = q;
                pa = y.amp;
            }
        }
    }
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1) {
        const int ob = __shfl_xor_sync(0xffffffffu, b, o);
        const float oa = __shfl_xor_sync(0xffffffffu, pa, o);
        if (ob != 0x7fffffff && (b == 0x7fffffff || pair_better(e.amp, ob, oa, b, pa))) {
            b = ob;
            pa = oa;
        }
    }
    return b;
}

// match[a]: the partner of XZ entry a where a is that one's partner too, else -1
template <int LANES>
__device__ __forceinline__ void pair_match(const ulm_loc2d* __restrict__ L, int n, int F, int S, int P,
                                           const int* __restrict__ poff, int* __restrict__ match)
{
    constexpr int PER = 256 / LANES;
    for (int a0 = blockIdx.x * PER; a0 < n; a0 += gridDim.x * PER) {
        const int a = a0 + threadIdx.x / LANES;
        ulm_loc2d x{}, y{};
        if (a < n) x = L[a];
        const bool xz = a < n && x.axis == 0;
        int m = -1;
        if (__any_sync(0xffffffffu, xz)) {
            const int b = pair_search<LANES>(L, n, x, xz, F, S, P, poff);
            const bool found = b != 0x7fffffff;
            if (__any_sync(0xffffffffu, found)) {
                if (found) y = L[b];
                if (pair_search<LANES>(L, n, y, found, F, S, P, poff) == a) m = b;
            }
        }
        if (a < n && threadIdx.x % LANES == 0) match[a] = m;
    }
}

// Matches of a list: every XZ entry searches its partner, and that one back.  Sixteen
// lanes share an entry (with one, a serial chain of loads and FP64 divisions, 2 392
// entries took 53 us, now 13) until the entries alone fill the chip, then two: 270 570
// entries of the paper's ensemble 267 us with one lane, 104 with sixteen, 86 with
// eight, 80 with two; 41 226 of a small geometry 114, 29, 30 and 50.  (Searches from
// both axes, so that none follows another, do twice the tests where few entries have a
// partner: 537 122 entries of which 820 match took 195 us; one lane 132, two 101.)
// Times of ulm_pair3d.
#define PAIR_LANES 16
#define PAIR_WIDE (1 << 18)   // entries from which on two lanes share one
__global__ void __launch_bounds__(256) k_pair_match(const ulm_loc2d* __restrict__ L, const int* __restrict__ n2d, int cap2d,
                                                    int F, int S, int P, const int* __restrict__ poff, int* __restrict__ match)
{
    grid_wait();
    const int n = min(*n2d, cap2d);
    if (n < PAIR_WIDE) pair_match<PAIR_LANES>(L, n, F, S, P, poff, match);
    else pair_match<2>(L, n, F, S, P, poff, match);
}

#define PAIR_CHUNK 1024   // list entries whose matches are counted together

__global__ void __launch_bounds__(256) k_pair_count(const int* __restrict__ n2d, int cap2d, const int* __restrict__ match,
                                                    int* __restrict__ part)
{
    grid_wait();
    __shared__ int red[8];
    const int n = min(*n2d, cap2d);
    for (int c = blockIdx.x; c * PAIR_CHUNK < n; c += gridDim.x) {
        int m = 0;
#pragma unroll
        for (int q = 0; q < PAIR_CHUNK; q += 256) {
            const int a = c * PAIR_CHUNK + q + threadIdx.x;
            if (a < n && match[a] >= 0) ++m;
        }
        m = __reduce_add_sync(0xffffffffu, m);
        __syncthreads();
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
        __syncthreads();
        if (threadIdx.x == 0) {
            int t = 0;
            for (int w = 0; w < 8; ++w) t += red[w];
            part[c] = t;
        }
    }
}

__global__ void __launch_bounds__(256) k_pair_write(const ulm_loc2d* __restrict__ L, const int* __restrict__ n2d, int cap2d,
                                                    const int* __restrict__ match, const int* __restrict__ part,
                                                    ulm_loc3d* __restrict__ out, int cap3d, int* __restrict__ n3d,
                                                    unsigned* __restrict__ status)
{
    grid_wait();
    __shared__ int red[16];
    constexpr int PER = PAIR_CHUNK / 256;
    const int n = min(*n2d, cap2d);
    if (n <= 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *n3d = 0;
        return;
    }
    for (int c = blockIdx.x; c * PAIR_CHUNK < n; c += gridDim.x) {
        const int a0 = c * PAIR_CHUNK + PER * threadIdx.x;
        unsigned m = 0u;
#pragma unroll
        for (int q = 0; q < PER; ++q)
            if (a0 + q < n && match[a0 + q] >= 0) m |= 1u << q;
        int all;
        int dst = block_offset(part, c, __popc(m), red, &all);
        if (threadIdx.x == 0 && (c + 1) * PAIR_CHUNK >= n) *n3d = all;
        while (m) {
            const int a = a0 + __ffs(m) - 1, b = match[a];
            m &= m - 1;
            if (dst >= cap3d) {
                atomicOr(status, ST_CAPACITY);
                break;
            }
            const ulm_loc2d x = L[a], y = L[b];
            ulm_loc3d o;
            o.frame = x.frame;
            o.i_xz = a;
            o.i_yz = b;
            o.reserved = 0;
            o.x = x.lat;
            o.y = y.lat;
            o.z = 0.5f * (x.z + y.z);
            o.amp_xz = x.amp;
            o.amp_yz = y.amp;
            o.reserved2 = 0.f;
            out[dst++] = o;
        }
    }
}

}  // namespace

// candidate slots of a detection, then their gather
struct Slots {
    ulm_loc2d* cand;
    int *cnt, *part;
    unsigned long long* total;
};

static rca_status slots_get(rca_handle* h, int nslots, Slots* o)
{
    rca_status st = RCA_OK;
    o->cand = (ulm_loc2d*)ws_get(h, WS_CAND, (size_t)nslots * CAND_CAP * sizeof(ulm_loc2d), &st);
    if (!o->cand) return st;
    // the true total, the chunks' kept totals, then the slots' counts.  All are cleared: a block whose wait runs out
    // counts nothing in the slots that it leaves, and the gather has to find those empty
    const size_t bytes = slots_bytes(nslots);
    char* p = (char*)ws_get(h, WS_CANDCNT, bytes, &st);
    if (!p) return st;
    o->total = reinterpret_cast<unsigned long long*>(p);
    o->part = reinterpret_cast<int*>(p + 16);
    o->cnt = o->part + (nslots + GATHER_SLOTS - 1) / GATHER_SLOTS;
    return cuda_check(h, cudaMemsetAsync(p, 0, bytes, h->stream), "candidate counts");
}

static rca_status slots_gather(rca_handle* h, const Slots& o, int nslots, int nstrip, ulm_loc2d* out, int cap, int* n2d,
                               int* poff, const float* A, const GeomDev& g)
{
    if (nslots > SCAN_MAX) return set_error(h, RCA_ERR_UNSUPPORTED, "scan over more than %d entries", SCAN_MAX);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // up to eight blocks a chunk, as long as there are no more than four per SM: with one, 20 frames of 250 x 128
    // planes have 23 blocks, which took 70 us for the 150 000 entries of 26 a slot (detection 162 us, now 104)
    const int chunks = (nslots + GATHER_SLOTS - 1) / GATHER_SLOTS;
    const int ny = std::max(1, std::min(8, 4 * sms / chunks));
    launch_chain(k_gather, dim3(chunks, ny), dim3(256), 0, h->stream,
        o.cand, o.cnt, o.part, o.total, nslots, nstrip, out, cap, n2d, poff, A, g.S, g.nz, g.N, h->d_status);
    return cuda_check(h, cudaGetLastError(), "gather kernel");
}

// pairing on scratch: match [cap2d], part [chunks of PAIR_CHUNK]
static rca_status pair_launch(rca_handle* h, const GeomDev& g, const ulm_loc2d* L, const int* n2d, int cap2d, int F,
                              const int* poff, int* match, int* part, ulm_loc3d* out, int cap3d, int* n3d)
{
    const int nn = std::max(cap2d, 1);
    if (nn > SCAN_MAX) return set_error(h, RCA_ERR_UNSUPPORTED, "scan over more than %d entries", SCAN_MAX);
    // the list's length is known on the device only: grids of a few waves at most walk it
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int cap_blocks = 16 * sms;
    const int nb = std::min(cap_blocks, (nn + 256 / PAIR_LANES - 1) / (256 / PAIR_LANES));
    const int nc = std::min(cap_blocks, (nn + PAIR_CHUNK - 1) / PAIR_CHUNK);
    launch_chain(k_pair_match, dim3(nb), dim3(256), 0, h->stream, L, n2d, cap2d, F, g.S, g.P, poff, match);
    launch_chain(k_pair_count, dim3(nc), dim3(256), 0, h->stream, n2d, cap2d, match, part);
    launch_chain(k_pair_write, dim3(nc), dim3(256), 0, h->stream, L, n2d, cap2d, match, part, out, cap3d, n3d, h->d_status);
    return cuda_check(h, cudaGetLastError(), "pair kernels");
}

rca_status launch_enhance(rca_handle* h, const rca_tables* t, const void* planes, rca_dtype pt, int F, int enh,
                          float* A, float* M)
{
    const GeomDev& g = t->gd;
    if (enh != ULM_ENH_XDOPPLER && enh != ULM_ENH_COHERENT) return set_error(h, RCA_ERR_INVALID_ARG, "bad enhancement mode");
    const size_t plane_sz = (size_t)g.nz * g.N;
    const size_t npx = 2 * (size_t)g.S * plane_sz;
    if (F > 48 * 1024) return set_error(h, RCA_ERR_UNSUPPORTED, "more than 49152 frames in one call");
    cudaMemsetAsync(M, 0, sizeof(float) * F, h->stream);
    // Every block walks all frames of its chunk, so the last wave of blocks
    // sets the tail: split the frames into chunks until the grid holds at
    // least eight waves of resident blocks (each chunk re-reads one frame;
    // at least 16 frames per chunk)
    const unsigned pblocks = (unsigned)((npx + 255) / 256);
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    auto kern = pt == RCA_C32 ? k_enhance<RCA_C32> : pt == RCA_C16F ? k_enhance<RCA_C16F> : k_enhance<RCA_C16BF>;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, (size_t)std::min(F, 16) * sizeof(unsigned));
    const unsigned resident = (unsigned)(std::max(1, per_sm) * sms);
    const int want = std::max(1, (int)((8u * resident + pblocks - 1) / pblocks));
    const int nchunk = std::min(want, std::max(1, F / 16));
    const int tf = (F + nchunk - 1) / nchunk;
    const size_t smem = (size_t)tf * sizeof(unsigned);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_check(h, e, "enhance smem attribute");
    dim3 grid(pblocks, (unsigned)((F + tf - 1) / tf));
    launch_chain(kern, grid, dim3(256), smem, h->stream, planes, F, g.S, plane_sz, enh, tf, A, reinterpret_cast<unsigned*>(M));
    return cuda_check(h, cudaGetLastError(), "enhance kernel");
}

rca_status launch_detect2d(rca_handle* h, const rca_tables* t, const float* A, const float* M, int F,
                           const ulm_params* prm, ulm_loc2d* out, int cap, int* n2d, float* ncc_out, int* plane_off)
{
    const GeomDev& g = t->gd;
    const int d = prm->d, hh = (d - 1) / 2;
    NccConst nc;
    nc.d = d;
    nc.h = hh;
    double G[RCA_MAX_NCC_D * RCA_MAX_NCC_D];
    double muG = 0.0;
    for (int a = -hh; a <= hh; ++a) {
        nc.gz[a + hh] = (float)std::exp(-(double)(a * a) / (2.0 * (double)prm->sig_z * prm->sig_z));
        nc.gl[a + hh] = (float)std::exp(-(double)(a * a) / (2.0 * (double)prm->sig_lat * prm->sig_lat));
    }
    for (int a = 0; a < d; ++a)
        for (int b = 0; b < d; ++b) {
            G[a * d + b] = (double)nc.gz[a] * (double)nc.gl[b];
            muG += G[a * d + b];
        }
    muG /= (double)(d * d);
    double ssG = 0.0;
    for (int q = 0; q < d * d; ++q) ssG += (G[q] - muG) * (G[q] - muG);
    nc.muG = (float)muG;
    nc.inv_ssG_sqrt = (float)(1.0 / std::sqrt(ssG));
    nc.flat_coef = (float)(1e-5 * d * d);
    nc.alpha = prm->alpha;
    nc.ncc_min = prm->ncc_min;

    const int nstrip = (g.nz + NCC_RS - 1) / NCC_RS;
    const int nplanes = F * 2 * g.S;
    const int nslots = nplanes * nstrip;
    rca_status st = RCA_OK;
    if (g.N % 2 != 0 || g.N > 256) return set_error(h, RCA_ERR_UNSUPPORTED, "NCC detection needs an even N <= 256");
    Slots slots;
    if ((st = slots_get(h, nslots, &slots)) != RCA_OK) return st;
    const int rin = NCC_RS + 2 + 2 * hh;
    // two buffers of amplitude rows (later the NCC rows, stride N + 1) + three
    // padded vertical-sum arrays of row pairs
    // + the amplitude flags of the NCC rows ([NCC_RS + 2][N] bytes)
    size_t smem = (2 * std::max((size_t)rin * g.N, (size_t)(NCC_RS + 2) * (g.N + 1)) +
                   (size_t)3 * ((NCC_RS + 2) / 2) * det_npad(g.N, hh, det_hb(hh)) * 2) * sizeof(float) +
                  (size_t)(NCC_RS + 2) * g.N;
    // persistent CTAs (as many as fit on an SM, each walking (plane, strip)
    // items with the next item's rows in flight), never more CTAs than items
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaSuccess;
    switch (hh) {
#define RCA_DETECT_LAUNCH(HV, NV, TV)                                                                      \
    do {                                                                                                   \
        auto kern = k_detect<HV, NV, TV>;                                                                  \
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);            \
        if (e != cudaSuccess) return cuda_check(h, e, "detect smem attribute");                          \
        int per_sm = 0;                                                                                    \
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, TV + 32, smem);                       \
        const dim3 grid((unsigned)std::max(1, std::min(nslots, std::max(1, per_sm) * sms)));               \
        launch_chain(kern, grid, dim3(TV + 32), smem, h->stream, A, M, g.S, g.nz, g.N, nplanes, nc, slots.cand, slots.cnt,      \
                                            slots.part, slots.total, ncc_out, h->d_status);                \
    } while (0)
#define RCA_DETECT_CASE(HV)                                                                                \
    case HV:                                                                                               \
        if (g.N == 128) RCA_DETECT_LAUNCH(HV, 128, NCC_THREADS);                                           \
        else if (g.N == 32) RCA_DETECT_LAUNCH(HV, 32, NCC_THREADS / 2);                                    \
        else if (g.N <= 64) RCA_DETECT_LAUNCH(HV, 0, NCC_THREADS / 2);                                     \
        else RCA_DETECT_LAUNCH(HV, 0, NCC_THREADS);                                                        \
        break;
        RCA_DETECT_CASE(1)
        RCA_DETECT_CASE(2)
        RCA_DETECT_CASE(3)
        RCA_DETECT_CASE(4)
        RCA_DETECT_CASE(5)
        RCA_DETECT_CASE(6)
        RCA_DETECT_CASE(7)
#undef RCA_DETECT_CASE
#undef RCA_DETECT_LAUNCH
    default: return set_error(h, RCA_ERR_INVALID_ARG, "NCC kernel length out of range");
    }
    if ((st = cuda_check(h, cudaGetLastError(), "detect kernel")) != RCA_OK) return st;
    return slots_gather(h, slots, nslots, nstrip, out, cap, n2d, plane_off, A, g);
}

rca_status launch_pair3d(rca_handle* h, const rca_tables* t, const ulm_loc2d* L, const int* n2d, int cap2d, int F,
                         ulm_loc3d* out, int cap3d, int* n3d, const int* plane_off)
{
    const GeomDev& g = t->gd;
    const int nplanes = F * 2 * g.S;
    rca_status st = RCA_OK;
    const int nn = std::max(cap2d, 1);
    int* match = (int*)ws_get(h, WS_FLAGS, (size_t)nn * sizeof(int), &st);
    if (!match) return st;
    int* part = (int*)ws_get(h, WS_MISC, (size_t)((nn + PAIR_CHUNK - 1) / PAIR_CHUNK) * sizeof(int), &st);
    if (!part) return st;
    if (!plane_off) {
        int* poff = (int*)ws_get(h, WS_PLANEOFF, (size_t)(nplanes + 1) * sizeof(int), &st);
        if (!poff) return st;
        launch_chain(k_list_plane_offsets, dim3((nplanes + 1 + 255) / 256), dim3(256), 0, h->stream, L, n2d, cap2d, g.S, nplanes, poff);
        plane_off = poff;
    }
    return pair_launch(h, g, L, n2d, cap2d, F, plane_off, match, part, out, cap3d, n3d);
}

// detection and pairing of one ensemble: the detection's gather writes the plane
// offsets that the pairing needs
rca_status launch_detect_pair(rca_handle* h, const rca_tables* t, const float* A, const float* M, int F,
                              const ulm_params* prm, ulm_loc2d* out2d, int cap2d, int* n2d, ulm_loc3d* out3d, int cap3d,
                              int* n3d)
{
    rca_status st = RCA_OK;
    int* poff = (int*)ws_get(h, WS_PLANEOFF, ((size_t)F * 2 * t->gd.S + 1) * sizeof(int), &st);
    if (!poff) return st;
    if ((st = launch_detect2d(h, t, A, M, F, prm, out2d, cap2d, n2d, nullptr, poff)) != RCA_OK) return st;
    return launch_pair3d(h, t, out2d, n2d, cap2d, F, out3d, cap3d, n3d, poff);
}

// ---------------------------------------------------------------------------
// Pairing without allocation (ulm_pair3d_noalloc).
//
// ulm_pair3d takes its scratch from the handle's workspace, which grows with
// cudaMalloc the first time a longer list arrives.  Some callers must not
// allocate once they are running: an acquisition loop that sized its device
// memory before the first ensemble cannot afford the device-wide stall of an
// allocation, or its failure, in the middle of a scan; a program whose own
// memory pool already holds the free HBM would see the allocation fail.
// For them the same kernels run on a fixed scratch array compiled into this
// file.  Being a file-scope __device__ variable, the array exists once per
// device, shared by every handle and call on it: calls whose work overlaps
// on the GPU race on it.  Its address is looked up once per device, on the
// first call made with that device current, and kept for the life of the
// process (a device reset makes the kept address stale; rca.h says so).
//
// Nothing in it needs clearing between calls: each call writes every entry
// it reads (plane offsets for all planes, matches for all live entries, one
// count per live chunk), so the previous call's contents are never seen.
// ---------------------------------------------------------------------------
namespace {

constexpr size_t na_round(size_t b) { return (b + 255) & ~(size_t)255; }
constexpr int NA_CHUNKS = (ULM_PAIR3D_NOALLOC_MAX_2D + PAIR_CHUNK - 1) / PAIR_CHUNK;
constexpr size_t NA_POFF = 0;
constexpr size_t NA_MATCH = NA_POFF + na_round((size_t)(ULM_PAIR3D_NOALLOC_MAX_PLANES + 1) * sizeof(int));
constexpr size_t NA_PART = NA_MATCH + na_round((size_t)ULM_PAIR3D_NOALLOC_MAX_2D * sizeof(int));
constexpr size_t NA_BYTES = ULM_PAIR3D_NOALLOC_SCRATCH_BYTES;   // the size that rca.h states
static_assert(NA_PART + na_round((size_t)NA_CHUNKS * sizeof(int)) <= NA_BYTES, "scratch size stated in rca.h is too small");

constexpr int NA_MAX_DEVICES = 64;

}  // namespace

static __device__ __align__(256) unsigned char g_pair_scratch[NA_BYTES];

static std::mutex g_pair_scratch_mu;
static unsigned char* g_pair_scratch_dev[NA_MAX_DEVICES];  // per device, null until looked up

// device address of g_pair_scratch on the handle's device (which is current)
static rca_status pair_scratch(rca_handle* h, unsigned char** base)
{
    if (h->device < 0 || h->device >= NA_MAX_DEVICES)
        return set_error(h, RCA_ERR_UNSUPPORTED, "ulm_pair3d_noalloc: device %d beyond %d", h->device, NA_MAX_DEVICES);
    std::lock_guard<std::mutex> lock(g_pair_scratch_mu);
    if (!g_pair_scratch_dev[h->device]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_pair_scratch);
        if (e != cudaSuccess) return cuda_check(h, e, "ulm_pair3d_noalloc scratch address");
        if (!p) return set_error(h, RCA_ERR_CUDA, "ulm_pair3d_noalloc: null scratch address");
        g_pair_scratch_dev[h->device] = static_cast<unsigned char*>(p);
    }
    *base = g_pair_scratch_dev[h->device];
    return RCA_OK;
}

rca_status launch_pair3d_noalloc(rca_handle* h, const rca_tables* t, const ulm_loc2d* L, const int* n2d, int cap2d,
                                 int F, ulm_loc3d* out, int cap3d, int* n3d)
{
    const GeomDev& g = t->gd;
    const long long nplanes = (long long)F * 2 * g.S;
    if (cap2d > ULM_PAIR3D_NOALLOC_MAX_2D)
        return set_error(h, RCA_ERR_UNSUPPORTED, "ulm_pair3d_noalloc: cap2d %d exceeds its fixed scratch of %d entries",
                         cap2d, ULM_PAIR3D_NOALLOC_MAX_2D);
    if (nplanes > ULM_PAIR3D_NOALLOC_MAX_PLANES)
        return set_error(h, RCA_ERR_UNSUPPORTED, "ulm_pair3d_noalloc: %lld planes exceed its fixed scratch of %d planes",
                         nplanes, ULM_PAIR3D_NOALLOC_MAX_PLANES);
    unsigned char* base = nullptr;
    rca_status st = pair_scratch(h, &base);
    if (st != RCA_OK) return st;
    int* poff = reinterpret_cast<int*>(base + NA_POFF);
    int* match = reinterpret_cast<int*>(base + NA_MATCH);
    int* part = reinterpret_cast<int*>(base + NA_PART);
    const int np = (int)nplanes;
    launch_chain(k_list_plane_offsets, dim3((np + 1 + 255) / 256), dim3(256), 0, h->stream, L, n2d, cap2d, g.S, np, poff);
    return pair_launch(h, g, L, n2d, cap2d, F, poff, match, part, out, cap3d, n3d);
}

rca_status launch_detect_map(rca_handle* h, const rca_tables* t, const float* map, int up, const float* A, const float* M,
                             int F, float score_min, float alpha, ulm_loc2d* out, int cap, int* n2d)
{
    const GeomDev& g = t->gd;
    const int H4 = g.nz * up, W4 = g.N * up;
    const int nstrip = (H4 + DET_RS - 1) / DET_RS;
    const int nplanes = F * 2 * g.S;
    const int nslots = nplanes * nstrip;
    rca_status st = RCA_OK;
    Slots slots;
    if ((st = slots_get(h, nslots, &slots)) != RCA_OK) return st;
    // the strip's rows plus the candidate bitmap of its pixels
    const size_t smem = (size_t)(DET_RS + 2) * W4 * sizeof(float) + (size_t)((DET_RS * W4 + 31) / 32) * sizeof(unsigned);
    if (smem > 200 * 1024) return set_error(h, RCA_ERR_UNSUPPORTED, "map rows of %d fine pixels exceed shared memory", W4);
    cudaError_t e = cudaFuncSetAttribute(k_detect_map, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_check(h, e, "detect_map smem attribute");
    dim3 grid(nstrip, nplanes);
    launch_chain(k_detect_map, dim3(grid), dim3(256), smem, h->stream, map, up, A, M, g.S, g.nz, g.N, score_min, alpha, slots.cand, slots.cnt,
                                                 slots.part, slots.total, h->d_status);
    if ((st = cuda_check(h, cudaGetLastError(), "detect_map kernel")) != RCA_OK) return st;
    return slots_gather(h, slots, nslots, nstrip, out, cap, n2d, nullptr, nullptr, g);
}
