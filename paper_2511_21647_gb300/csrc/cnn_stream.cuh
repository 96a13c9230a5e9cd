// cnn_stream.cuh -- the whole forward pass of the learned localiser in one
// kernel: the four 3x3 layers are streamed row by row, so that no activation
// leaves the SM (included by cnn.cu, which holds the tcgen05 helpers).
#pragma once

// ---------------------------------------------------------------------------
// A strip is 128 pixel slots wide (the M = 128 rows of one MMA): one window of
// a plane row, or the same row of several narrow planes side by side with one
// zero column between them.  Four warps walk a strip down the rows; at step t
// they run
//   layer 1 on row y (FP32, CUDA cores, weights in registers),
//   the MMAs of layer 2 on row y - 1, layer 3 on row y - 3, layer 4 on row
//   y - 5 (each the row its previous layer finished one step before),
//   the epilogues of the three output rows that those MMAs complete.
// Every input row is multiplied once: its three horizontal taps go as MMAs of
// N = 3 x COUT into the accumulators of the three output rows it touches
// (TMEM slots row mod 3), the weights being staged along N in the order
// ky = 2 1 0 2 1 so that each of the three rotations is a start offset.  The
// first of the row's MMAs is split per output row, because the newest of the
// three starts its sum there.  The order of the additions into an output is
// that of k_conv_tc (ky, kx, channels), and so are its bits.
//
// What bounds it: shared-memory bandwidth.  A 128 x 96 x 16 MMA reads 7 KB of
// operands (56 cycles at 128 B per clock, against 48 of the tensor pipe; as
// three MMAs of N = 32 it would read 15 KB), about 1040 cycles per row of 128
// pixels for the three layers, and the CUDA cores' accesses add about half as
// much (ncu, 16 frames of the paper's planes: the operand reads 67 % of the elapsed
// cycles, those accesses 38 %, the tensor pipe 43 %).  Two strips per CTA share the
// 77 KB of weights and fill each other's waits; 240 of 512 TMEM columns each.
// Separate warps for the edge layers, the hidden layers and the issue of MMAs
// keep a step short: one set of four warps that also issued took 5 800 cycles a
// step, an issuing warp of its own 3 700, all three 3 100.
// 16 frames of the paper's planes (512 of 250 x 128): 3.36 ms as five kernels
// (activations through HBM, heatmap copied), 0.73 ms here.
// ---------------------------------------------------------------------------
#define ST_M 128
#define ST_SLOTS (ST_M + 2)                       // one zero slot on either side
#define ST_KC 4                                   // 8-channel chunks of an activation row
#define ST_ROWB (ST_KC * ST_SLOTS * 16)           // bytes of one activation row
#define ST_WB(COUT) (3 * ST_KC * 5 * (COUT) * 16) // bytes of one layer's staged weights
#define ST_XW 132                                 // floats of one staged input row
#define ST_EDGE 4                                 // slots a window loses on either side to its halos
#define ST_STRIPS 2
#define ST_THREADS (ST_STRIPS * 288)              // per strip: four "edge" warps (layers 1 and 4), four "hidden"
                                                  // warps (layers 2 and 3), one MMA-issuing warp

struct StreamPlan {
    int np;       // planes side by side in a strip (narrow planes), else 1
    int nwin;     // windows per plane row (wide planes), else 1
    int ngrp;     // plane groups
    int R, nruns; // the rows of all windows of all groups, one after another, are cut into nruns runs of R
};

struct StreamSmem {
    static constexpr int w2 = 0, w3 = w2 + ST_WB(32), w4 = w3 + ST_WB(32), ring = w4 + ST_WB(16);
    static constexpr int xrow = ring + ST_STRIPS * 6 * ST_ROWB;
    static constexpr int bias = xrow + ST_STRIPS * 4 * ST_XW * 4;
    static constexpr int bytes = bias + (32 + 16) * 4;
};

struct StreamArgs {
    const float *A, *M;
    int ppf, B, H, W;
    StreamPlan plan;
    const float *w1, *b1, *b2, *b3, *b4;
    const __nv_bfloat16 *w2, *w3, *w4;
    float* heat;
    // KEEP: the normalised input and the activations, as the backward pass reads them
    float* x0;
    __nv_bfloat16 *a1, *a2, *a3;
    unsigned* status;
};

// weights [COUT][9][32] -> [kx][kc][ky order 2 1 0 2 1][COUT / 8][8 outputs][8 channels]
template <int COUT>
__device__ __forceinline__ void st_stage_weights(unsigned char* dst, const __nv_bfloat16* __restrict__ w)
{
    for (int q = threadIdx.x; q < 3 * ST_KC * 5 * COUT; q += blockDim.x) {
        const int o = q % COUT, r = q / COUT, blk = r % 5, kc = (r / 5) % ST_KC, kx = r / (5 * ST_KC);
        const int ky = (blk == 0 || blk == 3) ? 2 : (blk == 2 ? 0 : 1);
        const uint4 v = reinterpret_cast<const uint4*>(w)[(o * 9 + 3 * ky + kx) * ST_KC + kc];
        *reinterpret_cast<uint4*>(dst + ((kx * ST_KC + kc) * 5 + blk) * COUT * 16 + o * 16) = v;
    }
}

// the MMAs of one input row (one thread): ring row at `a`, weights at `b`,
// accumulators of the three output rows in TMEM columns tcol + COUT * (row mod 3)
template <int COUT>
__device__ __forceinline__ void st_issue(unsigned a, unsigned b, unsigned tcol, int row, bool first, uint64_t* bar)
{
    constexpr unsigned LB = 5 * COUT * 16;
    const int p = row % 3;
    const unsigned off = (p == 1 ? 0u : (p == 0 ? 1u : 2u)) * COUT * 16;
#pragma unroll
    for (int kx = 0; kx < 3; ++kx)
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
            const uint64_t da = tc_sdesc(a + kx * 16 + 2 * kk * ST_SLOTS * 16, ST_SLOTS * 16, 128);
            const unsigned bb = b + (unsigned)(kx * ST_KC + 2 * kk) * LB + off;
            if (kx == 0 && kk == 0) {
                const int fresh = (p + 1) % 3;   // output row `row + 1` starts here
#pragma unroll
                for (int s = 0; s < 3; ++s)
                    tc_mma(tcol + s * COUT, da, tc_sdesc(bb + s * COUT * 16, LB, 128), tc_idesc(ST_M, COUT),
                           !first && s != fresh);
            } else {
                tc_mma(tcol, da, tc_sdesc(bb, LB, 128), tc_idesc(ST_M, 3 * COUT), 1);
            }
        }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

template <bool KEEP>
__global__ void __launch_bounds__(ST_THREADS, 1) k_cnn_stream(const StreamArgs g)
{
    extern __shared__ __align__(128) unsigned char sms[];
    __shared__ uint64_t bars[ST_STRIPS][3];
    __shared__ unsigned s_tmem;
    __shared__ int s_err[ST_STRIPS][2];                             // a wait of step t ran out: [t & 1]
    // warp-uniform by a shuffle, so that the issuing warps' descriptors stay in uniform registers
    const int wid = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const bool issuer = wid >= 8 * ST_STRIPS, inner = wid >= 4 * ST_STRIPS;
    const int strip = issuer ? wid - 8 * ST_STRIPS : wid / 4 % ST_STRIPS, warp = wid & 3;
    const int lane = threadIdx.x & 31, tid = 32 * warp + lane;
    const int H = g.H, W = g.W;
    grid_wait();
    st_stage_weights<32>(sms + StreamSmem::w2, g.w2);
    st_stage_weights<32>(sms + StreamSmem::w3, g.w3);
    st_stage_weights<16>(sms + StreamSmem::w4, g.w4);
    for (int q = threadIdx.x; q < (StreamSmem::bias - StreamSmem::ring) / 16; q += blockDim.x)
        reinterpret_cast<uint4*>(sms + StreamSmem::ring)[q] = make_uint4(0, 0, 0, 0);
    float* sbias = reinterpret_cast<float*>(sms + StreamSmem::bias);
    if (threadIdx.x < 32) {                           // layers 1 and 4
        sbias[threadIdx.x] = g.b1[threadIdx.x];
        if (threadIdx.x < 16) sbias[32 + threadIdx.x] = g.b4[threadIdx.x];
    }
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < ST_STRIPS; ++s) {
            for (int l = 0; l < 3; ++l) mbar_init(&bars[s][l], 1);
            s_err[s][0] = s_err[s][1] = 0;
        }
        mbar_fence_init();
    }
    fence_proxy_async();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tm = s_tmem + (unsigned)(256 * strip);            // layers 2, 3, 4 at columns 0, 96, 192
    const unsigned tlane = tm + ((unsigned)(32 * warp) << 16);
    unsigned char* ring = sms + StreamSmem::ring + strip * 6 * ST_ROWB;   // [layer 1..3][2][ST_ROWB]
    const unsigned ringa = smem_u32(ring), wa = smem_u32(sms), b1a = smem_u32(sbias + 8 * warp);
    float* xs = reinterpret_cast<float*>(sms + StreamSmem::xrow) + strip * 4 * ST_XW;   // rows y & 3
    auto sync = [&]() { asm volatile("bar.sync %0, 288;" ::"r"(strip + 1) : "memory"); };   // a strip's nine warps
    unsigned phase = 0;                                              // bit l: parity of bars[strip][l]
    // 36 register pairs: an edge warp w's layer-1 weights of channels 8 w .. 8 w + 7, [channel pair][tap];
    // a hidden warp's biases of layers 2 and 3, [layer][channel pair]
    uint64_t reg[36];
#pragma unroll
    for (int p = 0; p < 36; ++p) {
        if (inner) {
            reg[p] = p < 16 ? f2_pack(g.b2[2 * p], g.b2[2 * p + 1])
                            : (p < 32 ? f2_pack(g.b3[2 * p - 32], g.b3[2 * p - 31]) : 0ull);
        } else {
            const int o = 8 * warp + 2 * (p / 9), t = p % 9;
            reg[p] = f2_pack(g.w1[o * 9 + t], g.w1[(o + 1) * 9 + t]);
        }
    }
    bool dead = false;
    const long long rows_all = (long long)g.plan.ngrp * g.plan.nwin * H;
    const long long run = blockIdx.x + (long long)gridDim.x * strip, run_end = min(rows_all, (run + 1) * g.plan.R);
    for (long long row = run * g.plan.R; row < run_end && !dead;) {
        // the part of the run that lies in one window
        const int gw = (int)(row / H), win = gw % g.plan.nwin, grp = gw / g.plan.nwin;
        const int r0 = (int)(row % H), r1 = (int)min((long long)H, r0 + (run_end - row));
        row += r1 - r0;
        const int lo2 = max(0, r0 - 3), hi2 = min(H - 1, r1 + 2);    // rows that layers 2, 3, 4 read
        const int lo3 = max(0, r0 - 2), hi3 = min(H - 1, r1 + 1);
        const int lo4 = max(0, r0 - 1), hi4 = min(H - 1, r1);
        const int t_end = r1 + 5 - lo2;                              // layer 4's row r1 - 1 is written here
        if (issuer) {
            for (int t = 0; t <= t_end; ++t) {
                sync();                                              // the rows of step t - 1 are in the rings
                if (*(volatile int*)&s_err[strip][(t + 1) & 1]) {
                    dead = true;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int i2 = lo2 + t - 1, i3 = i2 - 2, i4 = i3 - 2, rd = (t + 1) & 1;
                if (elect_one()) {
                    if (i2 >= lo2 && i2 <= hi2)
                        st_issue<32>(ringa + rd * ST_ROWB, wa + StreamSmem::w2, tm, i2, i2 == lo2, &bars[strip][0]);
                    if (i3 >= lo3 && i3 <= hi3)
                        st_issue<32>(ringa + (2 + rd) * ST_ROWB, wa + StreamSmem::w3, tm + 96, i3, i3 == lo3, &bars[strip][1]);
                    if (i4 >= lo4 && i4 <= hi4)
                        st_issue<16>(ringa + (4 + rd) * ST_ROWB, wa + StreamSmem::w4, tm + 192, i4, i4 == lo4, &bars[strip][2]);
                }
                __syncwarp();
            }
            if (!dead) {
                sync();                                              // the last step's
                dead = *(volatile int*)&s_err[strip][t_end & 1] != 0;
            }
            continue;
        }
        // this slot's plane and column; `live`: inside the plane, `own`: its outputs are written
        auto slot_pos = [&](int s, int& b, int& col) {
            if (g.plan.nwin > 1) {
                b = grp;
                col = win * (ST_M - 2 * ST_EDGE) - ST_EDGE + s;
                return col >= 0 && col < W;
            }
            b = grp * g.plan.np + s / (W + 1);
            col = s % (W + 1);
            return s / (W + 1) < g.plan.np && col < W && b < g.B;
        };
        auto slot_own = [&](int s) { return g.plan.nwin == 1 || (s >= ST_EDGE && s < ST_M - ST_EDGE); };
        int b, col;
        const bool live = slot_pos(tid, b, col), own = live && slot_own(tid);
        const size_t pix0 = live ? (size_t)b * H * W + col : 0;
        // after the step's barrier: a wait that ran out makes every warp of the strip leave
        auto gave_up = [&](int t, int first, int last) {
            if (*(volatile int*)&s_err[strip][t & 1] == 0) return false;
            if (tid == 0) {
                atomicOr(g.status, ST_TIMEOUT);
                for (int l = first; l <= last; ++l) mbar_wait_bounded(&bars[strip][l], (phase >> l & 1u) ^ 1u);
            }
            return true;
        };
        if (inner) {
            sync();
            for (int t = 0; t <= t_end; ++t) {
                const int i2 = lo2 + t - 1, i3 = i2 - 2, wr = t & 1;
                bool ok = true;
                // the output row that layer `layer`'s MMAs on input row i completed: bias, ReLU, BF16 -> next ring
                auto hidden = [&](int layer, int i, int i_lo, int i_hi, int o_lo, int o_hi, __nv_bfloat16* keep_to) {
                    if (i >= i_lo && i <= i_hi) {
                        ok = mbar_wait_bounded(&bars[strip][layer], phase >> layer & 1u) && ok;
                        phase ^= 1u << layer;
                    }
                    const int o = i - 1;
                    if (o < o_lo || o > o_hi) return;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    float v[32];
                    tc_ld<32>(tlane + (unsigned)(96 * layer + 32 * (o % 3)), v);
                    unsigned pk[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        const float2 y = f2_unpack(f2_add(f2_pack(v[2 * c], v[2 * c + 1]), reg[16 * layer + c]));
                        pk[c] = pack_bf2(fmaxf(y.x, 0.f), fmaxf(y.y, 0.f));
                    }
                    unsigned char* dst = ring + (2 * (layer + 1) + wr) * ST_ROWB + (tid + 1) * 16;
                    const bool keep = KEEP && own && o >= r0 && o < r1;
#pragma unroll
                    for (int c = 0; c < ST_KC; ++c) {
                        const uint4 q = live ? make_uint4(pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3])
                                             : make_uint4(0, 0, 0, 0);
                        *reinterpret_cast<uint4*>(dst + c * ST_SLOTS * 16) = q;
                        if (keep) reinterpret_cast<uint4*>(keep_to)[(pix0 + (size_t)o * W) * ST_KC + c] = q;
                    }
                };
                hidden(0, i2, lo2, hi2, lo3, hi3, g.a2);
                hidden(1, i3, lo3, hi3, lo4, hi4, g.a3);
                if (!ok) s_err[strip][t & 1] = 1;
                fence_proxy_async();
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                sync();
                if ((dead = gave_up(t, 0, 1))) break;
            }
            continue;
        }
        float scale = 1.f;
        if (live && g.M) {
            const float m = g.M[b / g.ppf];
            scale = m > 0.f ? 1.f / m : 0.f;
        }
        // layer 1 works on slots lane + 32 q: bit q live, bit q + 4 written out (KEEP)
        unsigned m1 = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int bq, cq;
            const bool lv = slot_pos(lane + 32 * q, bq, cq);
            if (lv) m1 |= 1u << q;
            if (lv && slot_own(lane + 32 * q)) m1 |= 16u << q;
        }
        auto x_at = [&](int y) { return (live && y >= 0 && y < H) ? __ldg(g.A + pix0 + (size_t)y * W) * scale : 0.f; };
#pragma unroll
        for (int q = -1; q <= 1; ++q) xs[((lo2 + q) & 3) * ST_XW + tid + 1] = x_at(lo2 + q);
        sync();
        for (int t = 0; t <= t_end; ++t) {
            const int y1 = lo2 + t, i4 = y1 - 5, o4 = i4 - 1;
            const float xn = (y1 + 2 <= hi2 + 1) ? x_at(y1 + 2) : 0.f;
            if (y1 <= hi2) {
                const bool keep = KEEP && y1 >= r0 && y1 < r1;
                const float* xr[3] = {xs + ((y1 - 1) & 3) * ST_XW, xs + (y1 & 3) * ST_XW, xs + ((y1 + 1) & 3) * ST_XW};
                unsigned char* dst = ring + (t & 1) * ST_ROWB + warp * ST_SLOTS * 16;
                if (KEEP && keep && own) g.x0[pix0 + (size_t)y1 * W] = xr[1][tid + 1];
                uint64_t bias[4];
                lds_u64x2(b1a, bias[0], bias[1]);
                lds_u64x2(b1a + 16, bias[2], bias[3]);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int s = lane + 32 * q;
                    uint64_t acc[4] = {bias[0], bias[1], bias[2], bias[3]};
#pragma unroll
                    for (int k = 0; k < 9; ++k) {
                        const float x = xr[k / 3][s + k % 3];
                        const uint64_t xx = f2_pack(x, x);
#pragma unroll
                        for (int p = 0; p < 4; ++p) acc[p] = f2_fma(reg[9 * p + k], xx, acc[p]);
                    }
                    unsigned pk[4];
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const float2 v = f2_unpack(acc[p]);
                        pk[p] = (m1 >> q & 1u) ? pack_bf2(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f)) : 0u;
                    }
                    const uint4 o = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    *reinterpret_cast<uint4*>(dst + (s + 1) * 16) = o;
                    if (KEEP && keep && (m1 >> q & 16u)) {
                        int bq, cq;
                        slot_pos(s, bq, cq);
                        reinterpret_cast<uint4*>(g.a1)[(((size_t)bq * H + y1) * W + cq) * ST_KC + warp] = o;
                    }
                }
            }
            if (i4 >= lo4 && i4 <= hi4) {
                if (!mbar_wait_bounded(&bars[strip][2], phase >> 2 & 1u)) s_err[strip][t & 1] = 1;
                phase ^= 4u;
            }
            if (o4 >= r0 && o4 < r1) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                float v[16];
                tc_ld<16>(tlane + (unsigned)(192 + 16 * (o4 % 3)), v);
                if (own) {
                    // channel c = 4 a + s -> heatmap pixel (4 i + a, 4 j + s)
                    const float4* bs = reinterpret_cast<const float4*>(sbias + 32);
                    const size_t W4 = (size_t)W * CNN_UP;
                    float* hp = g.heat + ((size_t)b * H + o4) * CNN_UP * W4 + (size_t)col * CNN_UP;
#pragma unroll
                    for (int a = 0; a < CNN_UP; ++a) {
                        const float4 bb = bs[a];
                        __stcs(reinterpret_cast<float4*>(hp + a * W4),
                               make_float4(v[4 * a] + bb.x, v[4 * a + 1] + bb.y, v[4 * a + 2] + bb.z, v[4 * a + 3] + bb.w));
                    }
                }
            }
            xs[((y1 + 2) & 3) * ST_XW + tid + 1] = xn;               // row y1 - 2 is no longer read
            fence_proxy_async();
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            sync();
            if ((dead = gave_up(t, 2, 2))) break;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int s = 0; s < ST_STRIPS; ++s)
            for (int l = 0; l < 3; ++l) mbar_inval(&bars[s][l]);
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(512) : "memory");
    }
}

// How a batch is cut.  Planes of up to 63 columns share a strip (one zero column
// apart), planes wider than 128 are cut into windows of 120 columns whose edges
// are recomputed.  Every strip of the chip gets one run of rows of the same
// length; a run pays about nine steps more for each window that it enters
// (three rows of halo and the pipeline's depth), so equal runs beat whole row
// segments dealt out in turns (512 planes of 250 rows on 304 strips: 421 rows
// and 2.7 windows each, about 446 steps, against 7 turns of 72).
inline StreamPlan stream_plan(int B, int H, int W, int sms)
{
    StreamPlan p;
    p.np = W < ST_M ? (ST_M + 1) / (W + 1) : 1;
    p.nwin = W > ST_M ? (W + ST_M - 2 * ST_EDGE - 1) / (ST_M - 2 * ST_EDGE) : 1;
    p.ngrp = (B + p.np - 1) / p.np;
    const long long rows = (long long)p.ngrp * p.nwin * H, strips = (long long)ST_STRIPS * sms;
    p.R = (int)((rows + strips - 1) / strips);
    p.nruns = (int)((rows + p.R - 1) / p.R);
    return p;
}
