// Microbubble separation on the projection planes (Sec. II-A5): each plane
// pixel's slow-time signal over the F frames is Fourier transformed, split by
// rectangular masks into 2 nb speed / direction subsets and transformed back.
//
// k_separate<MX, OUT> is persistent.  A CTA loops over groups of SP_TL
// consecutive lateral pixels of one plane row; the group's 2 SP_TL slow-time
// signals (RC and CR family of each pixel, interleaved: signal 2 l + fam) sit
// in shared memory as [F][SP_G] complex.  Transforms are mixed-radix Stockham
// passes (self-sorting, ping-pong between two buffers) whose radices (2, 3,
// 4, 5 and products of two of them up to 20) are evaluated in registers:
//   forward transform, spectrum kept in registers (MX values per thread);
//   per subset: the masked spectrum, scaled by 1/F, is written back and
//   transformed inversely; then either the complex subset is stored
//   (SP_OUT_COMPLEX) or its XDoppler (SP_OUT_XDOPPLER) or coherent
//   (SP_OUT_COHERENT) amplitude and per-frame maxima, which is what a
//   subset's localisation reads.
// Shared-memory traffic per subset and group: one write of the masked
// spectrum, two accesses per element per pass, one read for the output.
//
// k_separate_win<R1, OUT> is the form for frame counts with a two-pass plan
// (win_radix), among them the paper's 300.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "rca_internal.cuh"

namespace {

#define SP_TL 8                 // lateral pixels per group
#define SP_G (2 * SP_TL)        // signals per group
#define SP_THREADS 256
#define SP_MAXP 10              // passes
#define SP_MAXF 512
#define SP_WR 56                // W_R^m tables of 8, 12, 16 and 20 points
#define SP_OUT_COMPLEX 0
#define SP_OUT_XDOPPLER 1
#define SP_OUT_COHERENT 2

struct SepConst {
    int F, npass, nsub, enh;
    int radix[SP_MAXP];
    int twoff[SP_MAXP];             // pass p's twiddle table in shared memory (float2 offset)
    int ntw;                        // entries of all pass tables
    float s3, c51, c52, s51, s52;   // sin(2pi/3); cos, sin of 2pi/5 and 4pi/5
    float2 wr[SP_WR];               // exp(-2 pi i m / R), m < R
    signed char bin[SP_MAXF];       // subset of DFT bin j, -1 none
    short lo[2 * ULM_SEP_MAX_BANDS], hi[2 * ULM_SEP_MAX_BANDS];   // first and last bin of each subset (hi < lo: none)
    signed char r0[2 * ULM_SEP_MAX_BANDS], nw[2 * ULM_SEP_MAX_BANDS];   // k_separate_win: its window
};

// offset of R's table in SepConst::wr
__host__ __device__ constexpr int wr_off(int R)
{
    return R == 8 ? 0 : R == 12 ? 8 : R == 16 ? 20 : R == 20 ? 36 : -1;
}

// complex sums, differences and real multiples.  PK: as packed pairs, one issue slot instead of two, the same rounding;
// else scalar: k_separate's largest form, one CTA of eight warps an SM, waits for results rather than for issue slots
// (60 rows of 512 frames, 32 elements, six subsets: 648 us packed, 613 scalar)
template <bool PK>
__device__ __forceinline__ float2 f2add(float2 a, float2 b)
{
    if constexpr (PK) return f2_unpack(f2_add(f2_pack(a.x, a.y), f2_pack(b.x, b.y)));
    else return make_float2(a.x + b.x, a.y + b.y);
}
template <bool PK>
__device__ __forceinline__ float2 f2sub(float2 a, float2 b)
{
    if constexpr (PK) return f2_unpack(f2_sub(f2_pack(a.x, a.y), f2_pack(b.x, b.y)));
    else return make_float2(a.x - b.x, a.y - b.y);
}
template <bool PK>
__device__ __forceinline__ float2 f2scale(float2 a, float s)
{
    if constexpr (PK) return f2_unpack(f2_mul(f2_pack(a.x, a.y), f2_pack(s, s)));
    else return make_float2(a.x * s, a.y * s);
}
template <bool PK>
__device__ __forceinline__ float2 f2fma(float2 a, float s, float2 b)
{
    if constexpr (PK) return f2_unpack(f2_fma(f2_pack(a.x, a.y), f2_pack(s, s), f2_pack(b.x, b.y)));
    else return make_float2(fmaf(a.x, s, b.x), fmaf(a.y, s, b.y));
}
// a + i^e b, e known at compile time; the odd quarter turns in scalar operations, whose operands need no swap
template <bool PK>
__device__ __forceinline__ float2 addq(float2 a, float2 b, int e)
{
    e &= 3;
    return e == 0   ? f2add<PK>(a, b)
           : e == 1 ? make_float2(a.x - b.y, a.y + b.x)
           : e == 2 ? f2sub<PK>(a, b)
                    : make_float2(a.x + b.y, a.y - b.x);
}
// a w (forward) or a conj(w) (inverse)
template <bool INV>
__device__ __forceinline__ float2 twmul(float2 a, float2 w)
{
    return INV ? make_float2(fmaf(a.x, w.x, a.y * w.y), fmaf(a.y, w.x, -a.x * w.y))
               : make_float2(fmaf(a.x, w.x, -a.y * w.y), fmaf(a.x, w.y, a.y * w.x));
}
__device__ __forceinline__ float sqrt_approx_ftz(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// sqrt.approx (relative error about 2^-23; 0 -> 0)
__device__ __forceinline__ float sqrt_approx(float x)
{
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// R-point DFT in registers, y_k = sum_n x_n exp(-+2 pi i n k / R)
template <int R, bool INV, bool PK> struct Dft;

template <bool INV, bool PK> struct Dft<2, INV, PK> {
    static __device__ __forceinline__ void run(float2 (&v)[2], const SepConst&)
    {
        const float2 a = v[0];
        v[0] = f2add<PK>(a, v[1]);
        v[1] = f2sub<PK>(a, v[1]);
    }
};

// from the sum and difference of inputs 1 and 2, st t and sd d with signs known at compile time
template <bool INV, bool PK>
__device__ __forceinline__ void core3(float2 (&v)[3], float2 t, float2 d, float st, int sd, const SepConst& c)
{
    const float2 m = f2fma<PK>(t, -0.5f * st, v[0]);
    const float k = INV == (sd > 0) ? c.s3 : -c.s3;                            // v1, v2 = m +- i k d
    v[0] = st > 0.f ? f2add<PK>(v[0], t) : f2sub<PK>(v[0], t);
    v[1] = make_float2(fmaf(-k, d.y, m.x), fmaf(k, d.x, m.y));
    v[2] = make_float2(fmaf(k, d.y, m.x), fmaf(-k, d.x, m.y));
}

template <bool INV, bool PK> struct Dft<3, INV, PK> {
    static __device__ __forceinline__ void run(float2 (&v)[3], const SepConst& c)
    {
        core3<INV, PK>(v, f2add<PK>(v[1], v[2]), f2sub<PK>(v[1], v[2]), 1.f, 1, c);
    }
};

template <bool INV, bool PK> struct Dft<4, INV, PK> {
    static __device__ __forceinline__ void run(float2 (&v)[4], const SepConst&)
    {
        const float2 t0 = f2add<PK>(v[0], v[2]), t1 = f2sub<PK>(v[0], v[2]);
        const float2 t2 = f2add<PK>(v[1], v[3]), t3 = f2sub<PK>(v[1], v[3]);
        v[0] = f2add<PK>(t0, t2);
        v[2] = f2sub<PK>(t0, t2);
        v[1] = addq<PK>(t1, t3, INV ? 1 : 3);
        v[3] = addq<PK>(t1, t3, INV ? 3 : 1);
    }
};

// from the sums and differences of inputs 1, 4 (a1, s1 b1) and 2, 3 (a2, b2), s1 = +-1 known at compile time
template <bool INV, bool PK>
__device__ __forceinline__ void core5(float2 (&v)[5], float2 a1, float2 b1, float2 a2, float2 b2, int s1, const SepConst& c)
{
    const float2 m1 = f2fma<PK>(a2, c.c52, f2fma<PK>(a1, c.c51, v[0]));
    const float2 m2 = f2fma<PK>(a2, c.c51, f2fma<PK>(a1, c.c52, v[0]));
    const float2 r1 = s1 > 0 ? f2fma<PK>(b2, c.s52, f2scale<PK>(b1, c.s51)) : f2fma<PK>(b1, -c.s51, f2scale<PK>(b2, c.s52));
    const float2 r2 = s1 > 0 ? f2fma<PK>(b2, -c.s51, f2scale<PK>(b1, c.s52)) : f2fma<PK>(b1, c.s52, f2scale<PK>(b2, c.s51));   // s1 r2
    const int e1 = INV ? 1 : 3, e2 = e1 + (s1 > 0 ? 0 : 2);
    v[0] = f2add<PK>(v[0], f2add<PK>(a1, a2));
    v[1] = addq<PK>(m1, r1, e1);
    v[4] = addq<PK>(m1, r1, e1 + 2);
    v[2] = addq<PK>(m2, r2, e2);
    v[3] = addq<PK>(m2, r2, e2 + 2);
}

template <bool INV, bool PK> struct Dft<5, INV, PK> {
    static __device__ __forceinline__ void run(float2 (&v)[5], const SepConst& c)
    {
        core5<INV, PK>(v, f2add<PK>(v[1], v[4]), f2sub<PK>(v[1], v[4]), f2add<PK>(v[2], v[3]), f2sub<PK>(v[2], v[3]), 1, c);
    }
};

// R = R1 R2 by one Cooley-Tukey split in registers: n = R2 n1 + n2,
// k = k1 + R1 k2; the inner twiddles W_R^(n2 k1) are kernel-parameter
// constants at compile-time offsets.
template <int R1, int R2, bool INV, bool PK> struct DftC {
    static __device__ __forceinline__ void run(float2 (&v)[R1 * R2], const SepConst& c)
    {
        constexpr int W0 = wr_off(R1 * R2);
#pragma unroll
        for (int n2 = 0; n2 < R2; ++n2) {
            float2 a[R1];
#pragma unroll
            for (int n1 = 0; n1 < R1; ++n1) a[n1] = v[R2 * n1 + n2];
            Dft<R1, INV, PK>::run(a, c);
#pragma unroll
            for (int k1 = 0; k1 < R1; ++k1)
                v[R2 * k1 + n2] = (n2 * k1 == 0) ? a[k1] : twmul<INV>(a[k1], c.wr[W0 + n2 * k1]);
        }
        float2 o[R1 * R2];
#pragma unroll
        for (int k1 = 0; k1 < R1; ++k1) {
            float2 b[R2];
#pragma unroll
            for (int n2 = 0; n2 < R2; ++n2) b[n2] = v[R2 * k1 + n2];
            Dft<R2, INV, PK>::run(b, c);
#pragma unroll
            for (int k2 = 0; k2 < R2; ++k2) o[k1 + R1 * k2] = b[k2];
        }
#pragma unroll
        for (int k = 0; k < R1 * R2; ++k) v[k] = o[k];
    }
};

// coprime R1, R2 (Good and Thomas): input n goes by its remainders (n mod R1, n mod R2), output k = (R2 k1 + R1 k2) mod R;
// W_R^(n k) = W_R1^(n1 k1) W_R2^(n2 k2), so nothing is multiplied between the two steps
__host__ __device__ constexpr int crt_unit(int a, int b)      // 1 mod a, 0 mod b
{
    int n = 0;
    while (n % a != 1 % a) n += b;
    return n;
}
template <int R1, int R2, bool INV, bool PK> struct DftP {
    static __device__ __forceinline__ void run(float2 (&v)[R1 * R2], const SepConst& c)
    {
        constexpr int R = R1 * R2, E1 = crt_unit(R1, R2), E2 = crt_unit(R2, R1);
        float2 w[R];
#pragma unroll
        for (int n2 = 0; n2 < R2; ++n2) {
            float2 a[R1];
#pragma unroll
            for (int n1 = 0; n1 < R1; ++n1) a[n1] = v[(E1 * n1 + E2 * n2) % R];
            Dft<R1, INV, PK>::run(a, c);
#pragma unroll
            for (int k1 = 0; k1 < R1; ++k1) w[R2 * k1 + n2] = a[k1];
        }
#pragma unroll
        for (int k1 = 0; k1 < R1; ++k1) {
            float2 b[R2];
#pragma unroll
            for (int n2 = 0; n2 < R2; ++n2) b[n2] = w[R2 * k1 + n2];
            Dft<R2, INV, PK>::run(b, c);
#pragma unroll
            for (int k2 = 0; k2 < R2; ++k2) v[(R2 * k1 + R1 * k2) % R] = b[k2];
        }
    }
};

template <int R, bool INV, bool PK> struct Radix { using T = Dft<R, INV, PK>; };
template <bool INV, bool PK> struct Radix<6, INV, PK> { using T = DftP<2, 3, INV, PK>; };
template <bool INV, bool PK> struct Radix<8, INV, PK> { using T = DftC<2, 4, INV, PK>; };
template <bool INV, bool PK> struct Radix<10, INV, PK> { using T = DftP<2, 5, INV, PK>; };
template <bool INV, bool PK> struct Radix<12, INV, PK> { using T = DftP<4, 3, INV, PK>; };
template <bool INV, bool PK> struct Radix<15, INV, PK> { using T = DftP<3, 5, INV, PK>; };
template <bool INV, bool PK> struct Radix<16, INV, PK> { using T = DftC<4, 4, INV, PK>; };
template <bool INV, bool PK> struct Radix<20, INV, PK> { using T = DftP<4, 5, INV, PK>; };

// twiddle-table row pitch of a radix-R pass (R - 1 entries, even for 16-byte pairs)
__host__ __device__ constexpr int tw_pitch(int R) { return (R - 1 + 1) & ~1; }

// One Stockham pass of radix R over the SP_G signals: after the passes with
// radices before this one (product Ns), butterfly idx (k = idx mod Ns) takes
// in[idx + r F / R], twiddles them by W_F^(k r F / (Ns R)) = T[k pitch + r - 1],
// transforms and stores output u at (idx - k) R + k + u Ns.
template <int R, bool INV, bool PK>
__device__ __forceinline__ void sp_pass(const float2* __restrict__ in, float2* __restrict__ out, int F, int Ns,
                                        const float2* __restrict__ T, const SepConst& c)
{
    constexpr int P = tw_pitch(R);
    const int nb = F / R;
    for (int it = threadIdx.x; it < nb * SP_G; it += SP_THREADS) {
        const int g = it & (SP_G - 1), idx = it / SP_G;
        const int k = idx % Ns;
        const float2* src = in + idx * SP_G + g;
        float2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = src[r * nb * SP_G];
        if (k != 0) {
            const float4* t4 = reinterpret_cast<const float4*>(T + k * P);
#pragma unroll
            for (int r = 1; r < R; r += 2) {
                const float4 w = t4[(r - 1) / 2];
                v[r] = twmul<INV>(v[r], make_float2(w.x, w.y));
                if (r + 1 < R) v[r + 1] = twmul<INV>(v[r + 1], make_float2(w.z, w.w));
            }
        }
        Radix<R, INV, PK>::T::run(v, c);
        float2* dst = out + ((idx - k) * R + k) * SP_G + g;
#pragma unroll
        for (int u = 0; u < R; ++u) dst[u * Ns * SP_G] = v[u];
    }
}

// all passes; returns the buffer that holds the result
template <bool INV, bool PK>
__device__ float2* sp_fft(float2* a, float2* b, const SepConst& sc, const float2* tws)
{
    int Ns = 1;
    const int F = sc.F;
    for (int p = 0; p < sc.npass; ++p) {
        const int R = sc.radix[p];
        const float2* T = tws + sc.twoff[p];
        switch (R) {
            case 2: sp_pass<2, INV, PK>(a, b, F, Ns, T, sc); break;
            case 3: sp_pass<3, INV, PK>(a, b, F, Ns, T, sc); break;
            case 4: sp_pass<4, INV, PK>(a, b, F, Ns, T, sc); break;
            case 5: sp_pass<5, INV, PK>(a, b, F, Ns, T, sc); break;
            case 6: sp_pass<6, INV, PK>(a, b, F, Ns, T, sc); break;
            case 8: sp_pass<8, INV, PK>(a, b, F, Ns, T, sc); break;
            case 10: sp_pass<10, INV, PK>(a, b, F, Ns, T, sc); break;
            case 12: sp_pass<12, INV, PK>(a, b, F, Ns, T, sc); break;
            case 15: sp_pass<15, INV, PK>(a, b, F, Ns, T, sc); break;
            case 16: sp_pass<16, INV, PK>(a, b, F, Ns, T, sc); break;
            default: sp_pass<20, INV, PK>(a, b, F, Ns, T, sc); break;
        }
        __syncthreads();
        float2* t = a;
        a = b;
        b = t;
        Ns *= R;
    }
    return a;
}

// planes [F][2][2][S][nz][N] -> OUT_COMPLEX: sub [nsub][F][2][2][S][nz][N] C32;
// OUT_XDOPPLER / OUT_COHERENT: A [nsub][F][2][S][nz][N], M [nsub][F] (float bits, >= 0)
template <int MX, int OUT>
__global__ void __launch_bounds__(SP_THREADS, MX <= 19 ? 2 : 1)
    k_separate(const void* __restrict__ planes, int pt, const __grid_constant__ SepConst sc, int S, int nz, int N,
               float2* __restrict__ sub, float* __restrict__ A, unsigned* __restrict__ M)
{
    constexpr bool PK = MX <= 19;
    extern __shared__ __align__(16) float2 smem[];
    const int F = sc.F, nsub = sc.nsub;
    float2* B0 = smem;
    float2* B1 = B0 + (size_t)F * SP_G;
    float2* tws = B1 + (size_t)F * SP_G;                                      // pass twiddle tables
    unsigned* mx = reinterpret_cast<unsigned*>(tws + sc.ntw);                 // [nsub][F] frame maxima (amplitude outputs)
    signed char* sbin = reinterpret_cast<signed char*>(mx + (OUT != SP_OUT_COMPLEX ? nsub * F : 0));

    // pass p (Ns > 1): T_p[k pitch + r - 1] = exp(-2 pi i k r / (Ns R)), double then rounded
    {
        int Ns = 1;
        for (int p = 0; p < sc.npass; ++p) {
            const int R = sc.radix[p], P = tw_pitch(R);
            if (Ns > 1)
                for (int e = threadIdx.x; e < Ns * P; e += SP_THREADS) {
                    const int k = e / P, r = e % P + 1;
                    float2 w = make_float2(0.f, 0.f);
                    if (r < R) {
                        double sn, cs;
                        sincospi(-2.0 * (double)(k * r) / (double)(Ns * R), &sn, &cs);
                        w = make_float2((float)cs, (float)sn);
                    }
                    tws[sc.twoff[p] + e] = w;
                }
            Ns *= R;
        }
    }
    for (int m = threadIdx.x; m < F; m += SP_THREADS) sbin[m] = sc.bin[m];
    if (OUT != SP_OUT_COMPLEX)
        for (int i = threadIdx.x; i < nsub * F; i += SP_THREADS) mx[i] = 0u;
    __syncthreads();

    const int ngl = (N + SP_TL - 1) / SP_TL;
    const size_t rows_axis = (size_t)S * nz, per_axis = rows_axis * N;
    const long long ngroups = 2LL * (long long)rows_axis * ngl;
    const int n_el = F * SP_G;
    const float invF = 1.0f / (float)F;

    for (long long grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
        const int lg = (int)(grp % ngl);
        const long long row = grp / ngl;
        const int axis = (int)(row / (long long)rows_axis);
        const int lat0 = lg * SP_TL;
        const size_t rest0 = (size_t)(row % (long long)rows_axis) * N + lat0;

        // slow-time signals of the group: element t * SP_G + 2 l + fam; all of a
        // thread's loads are issued before its shared-memory stores
        float2 xr[MX];
#pragma unroll
        for (int m = 0; m < MX; ++m) {
            const int i = threadIdx.x + m * SP_THREADS;
            const int t = i / SP_G, gg = i & (SP_G - 1), l = gg >> 1, fam = gg & 1;
            xr[m] = make_float2(0.f, 0.f);
            if (i < n_el && lat0 + l < N)
                xr[m] = load_c(planes, (((size_t)t * 2 + axis) * 2 + fam) * per_axis + rest0 + l, pt);
        }
#pragma unroll
        for (int m = 0; m < MX; ++m) {
            const int i = threadIdx.x + m * SP_THREADS;
            if (i < n_el) B0[i] = xr[m];
        }
        __syncthreads();
        // each thread keeps the spectrum's elements threadIdx.x + m SP_THREADS; per subset the masked spectrum is written
        // back for the inverse transform
        const float2* X = sp_fft<false, PK>(B0, B1, sc, tws);
#pragma unroll
        for (int m = 0; m < MX; ++m) {
            const int e = threadIdx.x + m * SP_THREADS;
            xr[m] = e < n_el ? X[e] : make_float2(0.f, 0.f);
        }
        __syncthreads();

        for (int s = 0; s < nsub; ++s) {
#pragma unroll
            for (int m = 0; m < MX; ++m) {
                const int e = threadIdx.x + m * SP_THREADS;
                if (e < n_el) B0[e] = sbin[e / SP_G] == s ? f2scale<PK>(xr[m], invF) : make_float2(0.f, 0.f);
            }
            __syncthreads();
            const float2* Y = sp_fft<true, PK>(B0, B1, sc, tws);
            if (OUT == SP_OUT_COMPLEX) {
                float2* dst = sub + (size_t)s * F * 4 * per_axis;
                for (int i = threadIdx.x; i < n_el; i += SP_THREADS) {
                    const int t = i / SP_G, gg = i & (SP_G - 1), l = gg >> 1, fam = gg & 1;
                    if (lat0 + l < N) dst[(((size_t)t * 2 + axis) * 2 + fam) * per_axis + rest0 + l] = Y[i];
                }
            } else {
                // thread = (frame chunk ch, lateral pair lp): frames [ch per, ch per + per)
                // of lateral pixels la = lp + 4 (ch & 1) and lb = lp + 4 (1 - (ch & 1))
                // (the two chunks of a quarter-warp read opposite halves of their rows);
                // the three-frame window slides along the chunk.  Y4[t SP_TL + l] =
                // (RC, CR) of pixel l at frame t.
                constexpr int NLP = SP_TL / 2, NCH = SP_THREADS / NLP;
                const float4* Y4 = reinterpret_cast<const float4*>(Y);
                float* dstA = A + (size_t)s * F * 2 * per_axis;
                const int lp = threadIdx.x & (NLP - 1), ch = threadIdx.x / NLP;
                const int la = lp + NLP * (ch & 1), lb = lp + NLP * (1 - (ch & 1));
                const bool oka = lat0 + la < N, okb = lat0 + lb < N;
                const int per = (F + NCH - 1) / NCH, t0 = ch * per;
                auto ld = [&](int t, int l) -> float4 {
                    return (t >= 0 && t < F) ? Y4[t * SP_TL + l] : make_float4(0.f, 0.f, 0.f, 0.f);
                };
                auto qf = [](float4 v) { return make_float2(v.x * v.z + v.y * v.w, v.y * v.z - v.x * v.w); };
                float2 qma = qf(ld(t0 - 1, la)), qmb = qf(ld(t0 - 1, lb));
                float2 q0a = qf(ld(t0, la)), q0b = qf(ld(t0, lb));
                float4 ya = ld(t0, la), yb = ld(t0, lb);
#pragma unroll
                for (int i = 0; i < per; ++i) {
                    const int t = t0 + i;
                    float aa, ab;
                    if (OUT == SP_OUT_XDOPPLER) {
                        const float2 qpa = qf(ld(t + 1, la)), qpb = qf(ld(t + 1, lb));
                        const float ra = qma.x + q0a.x + qpa.x, ia = qma.y + q0a.y + qpa.y;
                        const float rb = qmb.x + q0b.x + qpb.x, ib = qmb.y + q0b.y + qpb.y;
                        aa = sqrt_approx(sqrt_approx(ra * ra + ia * ia));
                        ab = sqrt_approx(sqrt_approx(rb * rb + ib * ib));
                        qma = q0a;
                        q0a = qpa;
                        qmb = q0b;
                        q0b = qpb;
                    } else {
                        const float ra = ya.x + ya.z, ia = ya.y + ya.w, rb = yb.x + yb.z, ib = yb.y + yb.w;
                        aa = sqrt_approx(ra * ra + ia * ia);
                        ab = sqrt_approx(rb * rb + ib * ib);
                        ya = ld(t + 1, la);
                        yb = ld(t + 1, lb);
                    }
                    float mm = 0.f;
                    if (t < F) {
                        float* d = dstA + ((size_t)t * 2 + axis) * per_axis + rest0;
                        if (oka) {
                            __stcs(d + la, aa);
                            mm = aa;
                        }
                        if (okb) {
                            __stcs(d + lb, ab);
                            mm = fmaxf(mm, ab);
                        }
                    }
                    mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, 1));
                    mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, 2));
                    if (lp == 0 && t < F) atomicMax(mx + s * F + t, __float_as_uint(mm));
                }
            }
            __syncthreads();
        }
    }
    if (OUT != SP_OUT_COMPLEX)
        for (int i = threadIdx.x; i < nsub * F; i += SP_THREADS)
            if (mx[i]) atomicMax(M + i, mx[i]);
}

// frame counts with a plan of two passes R1 = 4 Q (20, 16, 12) and R2 (an instantiated radix), R2 <= R1 where there is
// one (a thread per butterfly in both passes): R1, else 0 (k_separate).  Paper geometry, FP32 planes, three bands: 300
// frames (250 rows) 11.82 ms in k_separate with its passes fixed at compile time, 9.58 ms here; 60 rows of 60 frames 1553
// and 532 us, 128 frames 1761 and 902, 144 frames 2986 and 945, 256 frames 3063 and 1901.
__host__ __device__ constexpr int win_radix(int F)
{
    for (int pass = 0; pass < 2; ++pass)
        for (int R1 = 12; R1 <= 20; R1 += 4) {
            const int R2 = F / R1;
            const bool menu = R2 == 4 || R2 == 5 || R2 == 6 || R2 == 8 || R2 == 10 || R2 == 12 || R2 == 15 || R2 == 16;
            if (F % R1 == 0 && menu && (R2 <= R1 || pass == 1)) return R1;
        }
    return 0;
}

// y_k = sum_{m < NW Q} x_m exp(2 pi i m k / (4 Q)) to dst[k], k < 4 Q: the 4 Q-point inverse transform of inputs of which
// all but the first NW Q are zero.  The four-point step has one or two inputs (m and m + Q), so its output k1 is a sum at
// most and a quarter turn.  Q = 3, 5: coprime split; the quarter turns i^(m k1) go into the signs and swaps of the first
// sums (74 issue slots of arithmetic for 12 and 96 for 20 points).  Q = 4: the inner twiddles W_16^(n2 k1) remain.
template <int Q, int NW, typename St>
__device__ __forceinline__ void win_idft(const float2 (&x)[NW * Q], const SepConst& c, St store)
{
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
        float2 b[Q];
        // b[m] = i^(m k1) z[m] (Q = 3, 5); z[m] = x[m] + i^(Q k1) x[m + Q]
#pragma unroll
        for (int m = 0; m < Q; ++m) b[m] = NW == 1 ? x[m] : addq<true>(x[m], x[(NW - 1) * Q + m], (Q == 4 ? 1 : Q) * k1);
        if constexpr (Q == 5) {
            // inputs 1, 4: i^k1 z1 and z4; inputs 2, 3: i^(2 k1) (z2 + i^k1 z3), i^(2 k1) = -1 for odd k1
            const float2 a1 = addq<true>(b[4], b[1], k1), n1 = addq<true>(b[4], b[1], k1 + 2);      // n1 = -(i^k1 z1 - z4)
            float2 a2 = addq<true>(b[2], b[3], k1), b2 = addq<true>(b[2], b[3], k1 + 2);
            if (k1 & 1) {
                a2 = make_float2(-a2.x, -a2.y);
                b2 = make_float2(-b2.x, -b2.y);
            }
            core5<true, true>(b, a1, n1, a2, b2, -1, c);
        } else if constexpr (Q == 3) {
            // input 2: i^(2 k1) z2 = s z2, s = +-1; input 1: i^k1 z1 = s i^(-k1) z1
            const float2 t = addq<true>(b[2], b[1], -k1), d = addq<true>(b[2], b[1], 2 - k1);
            core3<true, true>(b, t, d, k1 & 1 ? -1.f : 1.f, k1 & 1 ? 1 : -1, c);
        } else {
#pragma unroll
            for (int m = 1; m < Q; ++m)
                if (k1) b[m] = twmul<true>(b[m], c.wr[wr_off(16) + m * k1]);
            Dft<Q, true, true>::run(b, c);
        }
#pragma unroll
        for (int k2 = 0; k2 < Q; ++k2) store(Q == 4 ? k1 + 4 * k2 : (Q * k1 + 4 * k2) % (4 * Q), b[k2]);
    }
}

// first inverse pass of one subset: butterfly idx reads bins idx + R2 (r0 + m) of the spectrum, those of [lo, hi]
template <int R1, int NW>
__device__ __forceinline__ void win_pass1(const float2* X, float2* B, int R2, int r0, int lo, int hi, const SepConst& c)
{
    constexpr int Q = R1 / 4;
    for (int it = threadIdx.x; it < R2 * SP_G; it += R1 * SP_G) {
        const int g = it & (SP_G - 1), idx = it / SP_G;
        float2 x[NW * Q];
#pragma unroll
        for (int m = 0; m < NW * Q; ++m) {
            const int j = idx + R2 * (r0 + m);
            x[m] = (unsigned)(j - lo) < (unsigned)(hi + 1 - lo) ? X[j * SP_G + g] : make_float2(0.f, 0.f);
        }
        float2* dst = B + idx * R1 * SP_G + g;
        win_idft<Q, NW>(x, c, [&](int k, float2 y) { dst[k * SP_G] = y; });
    }
}

// second pass in registers: thread (idx, g) holds, twiddles and transforms the elements idx + R1 r', which are also the
// frames (or bins) idx + R1 u that it produces
template <int R1, int R2, bool INV>
__device__ __forceinline__ void win_pass2(float2 (&v)[R2], const float2* B, const float2* T, const SepConst& c)
{
    const int idx = threadIdx.x / SP_G;
#pragma unroll
    for (int r = 0; r < R2; ++r) v[r] = B[threadIdx.x + r * R1 * SP_G];
    const float4* t4 = reinterpret_cast<const float4*>(T + idx * tw_pitch(R2));
#pragma unroll
    for (int r = 1; r < R2; r += 2) {
        const float4 w = t4[(r - 1) / 2];
        v[r] = twmul<INV>(v[r], make_float2(w.x, w.y));
        if (r + 1 < R2) v[r + 1] = twmul<INV>(v[r + 1], make_float2(w.z, w.w));
    }
    Radix<R2, INV, true>::T::run(v, c);
}

// amplitudes of one subset from its frames Y [F][SP_G]: thread (lateral pixel l, chunk of PER frames); the frame maxima
// are only reduced when a warp holds a value that its CTA's maximum does not bound (NaN among them)
template <int F, int NT, int PER, int OUT>
__device__ __forceinline__ void win_output(const float2* Y, float* dst, size_t frame_pitch, bool ok, unsigned* mx)
{
    const int l = threadIdx.x & (SP_TL - 1), t0 = threadIdx.x / SP_TL * PER;
    const float4* Y4 = reinterpret_cast<const float4*>(Y) + l;                // Y4[t SP_TL]: (RC, CR) of pixel l
    static_assert(NT / SP_TL * PER >= F && NT % 32 == 0, "chunks cover the frames");
    float a[PER];
    auto ld = [&](int t) { return t >= 0 && t < F ? Y4[t * SP_TL] : make_float4(0.f, 0.f, 0.f, 0.f); };
    if (OUT == SP_OUT_XDOPPLER) {
        auto qf = [](float4 v) { return make_float2(v.x * v.z + v.y * v.w, v.y * v.z - v.x * v.w); };
        float2 qm = qf(ld(t0 - 1)), q0 = qf(ld(t0));
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const float2 qp = qf(ld(t0 + i + 1));
            const float re = qm.x + q0.x + qp.x, im = qm.y + q0.y + qp.y;
            a[i] = sqrt_approx_ftz(sqrt_approx(re * re + im * im));    // the inner root is 0 or above 2^-75
            qm = q0;
            q0 = qp;
        }
    } else {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const float4 y = ld(t0 + i);
            const float re = y.x + y.z, im = y.y + y.w;
            a[i] = sqrt_approx(re * re + im * im);
        }
    }
    bool above = false;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        if (t0 + i >= F) break;
        if (ok) __stcs(dst + (size_t)(t0 + i) * frame_pitch + l, a[i]);
        above |= ok && !(a[i] <= __uint_as_float(mx[t0 + i]));
    }
    if (__any_sync(0xffffffffu, above)) {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            float m = ok ? a[i] : 0.f;
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 4));
            if (l == 0 && t0 + i < F) atomicMax(mx + t0 + i, __float_as_uint(m));
        }
    }
}

// k_separate for frame counts F = R1 R2 in two passes, with three changes.
// (1) A subset's bins are consecutive, so the first inverse pass (R1 points, inputs R2 bins apart) reads a window of
// R1 / 4 or R1 / 2 consecutive inputs r0 .. (at most half: up and down bins lie in either half).  The window is taken
// as if it began at input 0, which multiplies frame t by exp(-2 pi i r0 t / R1): the amplitudes of the two families'
// product or sum do not see it, the complex output is multiplied back.
// (2) The second pass reads and writes the same elements in one thread, in place, so the spectrum stays in the other
// buffer instead of in 40 registers, and R1 SP_G threads have one butterfly each.
// (3) The frame maxima are reduced only where one rises.
// What bounds it at 300 frames: issue slots and the shared-memory pipe together, with barriers between the phases
// (without samples read and amplitudes written it takes 7.9 ms of 9.6).  Slower here: groups of four pixels (15.3 ms,
// half the bytes per request), both families in a thread (11.0, a third fewer instructions but 10 warps an SM),
// amplitudes and the next first pass in one phase with the families exchanged by shuffles (10.0), samples copied ahead
// asynchronously or prefetched to L2 (10.0, 10.7); 16 pixels a group measure the same.
template <int R1, int OUT>
__global__ void __launch_bounds__(R1* SP_G, R1 == 20 ? 2 : R1 == 16 ? 3 : 4)
    k_separate_win(const void* __restrict__ planes, int pt, const __grid_constant__ SepConst sc, int S, int nz, int N,
                   float2* __restrict__ sub, float* __restrict__ A, unsigned* __restrict__ M)
{
    constexpr int NT = R1 * SP_G;
    extern __shared__ __align__(16) float2 smem[];
    const int F = sc.F, nsub = sc.nsub, R2 = F / R1;
    float2* X = smem;
    float2* B = X + (size_t)F * SP_G;
    float2* tws = B + (size_t)F * SP_G;                                       // exp(-2 pi i k r / F), k < R1, r < R2
    unsigned* mx = reinterpret_cast<unsigned*>(tws + sc.ntw);                 // [nsub][F] frame maxima (amplitude outputs)
    const int P = tw_pitch(R2);
    for (int e = threadIdx.x; e < R1 * P; e += NT) {
        const int k = e / P, r = e % P + 1;
        double sn = 0.0, cs = 0.0;
        if (r < R2) sincospi(-2.0 * (double)(k * r) / (double)F, &sn, &cs);
        tws[e] = make_float2((float)cs, (float)sn);
    }
    if (OUT != SP_OUT_COMPLEX)
        for (int i = threadIdx.x; i < nsub * F; i += NT) mx[i] = 0u;
    __syncthreads();

    const int ngl = (N + SP_TL - 1) / SP_TL;
    const size_t rows_axis = (size_t)S * nz, per_axis = rows_axis * N;
    const unsigned ngroups = (unsigned)(2 * rows_axis * ngl);     // planes of 2^32 groups of 48 and more frames fit no memory
    const float invF = 1.0f / (float)F;

    for (unsigned grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
        const unsigned row = grp / ngl;
        const int axis = row >= rows_axis, lat0 = (int)(grp - row * ngl) * SP_TL;
        const size_t rest0 = (row - axis * rows_axis) * N + lat0;

        // forward: the first pass reads the planes (signal g = 2 l + family), all of a thread's loads before its arithmetic
        for (int it = threadIdx.x; it < R2 * SP_G; it += NT) {
            const int g = it & (SP_G - 1), idx = it / SP_G, l = g >> 1;
            const size_t base = ((size_t)idx * 4 + axis * 2 + (g & 1)) * per_axis + rest0 + l, step = (size_t)R2 * 4 * per_axis;
            float2 v[R1];
            if (lat0 + l >= N) {
#pragma unroll
                for (int r = 0; r < R1; ++r) v[r] = make_float2(0.f, 0.f);
            } else if (pt == RCA_C32) {
                const float2* p = reinterpret_cast<const float2*>(planes) + base;
#pragma unroll
                for (int r = 0; r < R1; ++r) v[r] = p[r * step];
            } else {
                const unsigned* p = reinterpret_cast<const unsigned*>(planes) + base;
                unsigned w[R1];
#pragma unroll
                for (int r = 0; r < R1; ++r) w[r] = p[r * step];
#pragma unroll
                for (int r = 0; r < R1; ++r) v[r] = load_c(w + r, 0, pt);
            }
            Radix<R1, false, true>::T::run(v, sc);
            float2* dst = X + idx * R1 * SP_G + g;
#pragma unroll
            for (int u = 0; u < R1; ++u) dst[u * SP_G] = v[u];
        }
        __syncthreads();
        auto second = [&](auto r2) {
            constexpr int RR = decltype(r2)::value;
            float2 v[RR];
            win_pass2<R1, RR, false>(v, X, tws, sc);
#pragma unroll
            for (int u = 0; u < RR; ++u) X[threadIdx.x + u * NT] = f2scale<true>(v[u], invF);
        };
        auto subset = [&](auto r2, int s) {
            constexpr int RR = decltype(r2)::value;
            float2 v[RR];
            win_pass2<R1, RR, true>(v, B, tws, sc);
            if (OUT == SP_OUT_COMPLEX) {
                const int g = threadIdx.x & (SP_G - 1), idx = threadIdx.x / SP_G, l = g >> 1;
                const float2 w = sc.wr[wr_off(R1) + sc.r0[s] * idx % R1];     // exp(-2 pi i r0 t / R1), t = idx + R1 u
                float2* dst = sub + ((size_t)s * F + idx) * 4 * per_axis + (axis * 2 + (g & 1)) * per_axis + rest0 + l;
                if (lat0 + l < N)
#pragma unroll
                    for (int u = 0; u < RR; ++u) dst[(size_t)u * R1 * 4 * per_axis] = twmul<true>(v[u], w);
            } else {
#pragma unroll
                for (int u = 0; u < RR; ++u) B[threadIdx.x + u * NT] = v[u];
                __syncthreads();
                constexpr int PER = (RR + 1) / 2;
                win_output<R1 * RR, NT, PER, OUT>(B, A + ((size_t)s * F * 2 + axis) * per_axis + rest0, 2 * per_axis,
                                                  lat0 + (int)(threadIdx.x & (SP_TL - 1)) < N, mx + s * F);
            }
        };
#define SP_R2(RR, CALL)                                                                                         \
    case RR:                                                                                                    \
        if constexpr (win_radix(R1 * RR) == R1) CALL;                                                           \
        break
#define SP_SWITCH(CALL)                                                                                         \
    switch (R2) {                                                                                               \
        SP_R2(4, CALL(4));                                                                                      \
        SP_R2(5, CALL(5));                                                                                      \
        SP_R2(6, CALL(6));                                                                                      \
        SP_R2(8, CALL(8));                                                                                      \
        SP_R2(10, CALL(10));                                                                                    \
        SP_R2(12, CALL(12));                                                                                    \
        SP_R2(15, CALL(15));                                                                                    \
        SP_R2(16, CALL(16));                                                                                    \
    }
#define SP_SECOND(RR) second(std::integral_constant<int, RR>())
#define SP_SUBSET(RR) subset(std::integral_constant<int, RR>(), s)
        SP_SWITCH(SP_SECOND)
        __syncthreads();
        for (int s = 0; s < nsub; ++s) {
            if (sc.nw[s] == 1)
                win_pass1<R1, 1>(X, B, R2, sc.r0[s], sc.lo[s], sc.hi[s], sc);
            else
                win_pass1<R1, 2>(X, B, R2, sc.r0[s], sc.lo[s], sc.hi[s], sc);
            __syncthreads();
            SP_SWITCH(SP_SUBSET)
            __syncthreads();
        }
#undef SP_SUBSET
#undef SP_SECOND
#undef SP_SWITCH
#undef SP_R2
    }
    if (OUT != SP_OUT_COMPLEX)
        for (int i = threadIdx.x; i < nsub * F; i += NT)
            if (mx[i]) atomicMax(M + i, mx[i]);
}

// radix plan: F = product of the passes' radices, largest first from the menu
bool plan_radices(int F, int* radix, int* npass)
{
    static const int menu[] = {20, 16, 15, 12, 10, 8, 6, 5, 4, 3, 2};
    int n = 0, rem = F;
    while (rem > 1) {
        int pick = 0;
        for (int r : menu)
            if (rem % r == 0) {
                pick = r;
                break;
            }
        if (!pick || n == SP_MAXP) return false;
        radix[n++] = pick;
        rem /= pick;
    }
    *npass = n;
    return true;
}

template <typename K>
rca_status launch_sep(rca_handle* h, K kern, int threads, const void* planes, int pt, const SepConst& sc, int S, int nz, int N,
                      float2* sub, float* A, unsigned* M, size_t smem, long long ngroups)
{
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_check(h, e, "separation smem attribute");
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    if (e != cudaSuccess) return cuda_check(h, e, "separation occupancy");
    if (per_sm < 1) return set_error(h, RCA_ERR_UNSUPPORTED, "separation kernel does not fit an SM");
    const long long grid = std::min<long long>(ngroups, (long long)per_sm * sms);
    if (grid > 0) kern<<<(unsigned)grid, threads, smem, h->stream>>>(planes, pt, sc, S, nz, N, sub, A, M);
    return cuda_check(h, cudaGetLastError(), "separation kernel");
}

}  // namespace

rca_status launch_separate(rca_handle* h, const rca_tables* t, const void* planes, rca_dtype pt, int F,
                           const ulm_sep_params* prm, int enh, float2* sub, float* A, float* M)
{
    const GeomDev& g = t->gd;
    const int nb = prm->n_bands;
    if (!(prm->prf_hz > 0.0) || nb < 1 || nb > ULM_SEP_MAX_BANDS)
        return set_error(h, RCA_ERR_INVALID_ARG, "separation needs prf_hz > 0 and 1 .. %d bands", ULM_SEP_MAX_BANDS);
    if (!(prm->edges_hz[0] >= 0.0)) return set_error(h, RCA_ERR_INVALID_ARG, "band edges must start at >= 0");
    for (int b = 0; b < nb; ++b)
        if (!(prm->edges_hz[b + 1] > prm->edges_hz[b]))
            return set_error(h, RCA_ERR_INVALID_ARG, "band edges must increase");
    if (A && enh != ULM_ENH_XDOPPLER && enh != ULM_ENH_COHERENT)
        return set_error(h, RCA_ERR_INVALID_ARG, "bad enhancement mode");
    if (F > SP_MAXF) return set_error(h, RCA_ERR_UNSUPPORTED, "separation supports at most %d frames", SP_MAXF);
    SepConst sc;
    std::memset(&sc, 0, sizeof(sc));
    sc.F = F;
    sc.nsub = 2 * nb;
    sc.enh = enh;
    const int R1 = win_radix(F);
    if (R1) {
        sc.npass = 2;
        sc.radix[0] = R1;
        sc.radix[1] = F / R1;
    } else if (!plan_radices(F, sc.radix, &sc.npass))
        return set_error(h, RCA_ERR_UNSUPPORTED, "separation needs a frame count with prime factors 2, 3, 5 (F = %d)", F);
    const double pi = 3.14159265358979323846;
    sc.s3 = (float)std::sin(2.0 * pi / 3.0);
    sc.c51 = (float)std::cos(2.0 * pi / 5.0);
    sc.c52 = (float)std::cos(4.0 * pi / 5.0);
    sc.s51 = (float)std::sin(2.0 * pi / 5.0);
    sc.s52 = (float)std::sin(4.0 * pi / 5.0);
    for (int R : {8, 12, 16, 20})
        for (int m = 0; m < R; ++m)
            sc.wr[wr_off(R) + m] = make_float2((float)std::cos(2.0 * pi * m / R), (float)-std::sin(2.0 * pi * m / R));
    // pass twiddle tables: rows of tw_pitch(R) entries per k < Ns (passes with Ns > 1)
    {
        int Ns = 1, off = 0;
        for (int p = 0; p < sc.npass; ++p) {
            sc.twoff[p] = off;
            if (Ns > 1) off += Ns * tw_pitch(sc.radix[p]);
            Ns *= sc.radix[p];
        }
        sc.ntw = off;
    }
    // bin -> subset: signed index k, |k| prf / F against the edges (upper edge
    // inclusive), k > 0 up (subsets 0 .. nb-1), k < 0 down (nb .. 2 nb - 1);
    // DC and the Nyquist bin in none
    for (int j = 0; j < F; ++j) {
        sc.bin[j] = -1;
        if (j == 0 || 2 * j == F) continue;
        const int k = 2 * j < F ? j : j - F;
        const double f = (double)std::abs(k) * prm->prf_hz / (double)F;
        for (int b = 0; b < nb; ++b)
            if (prm->edges_hz[b] < f && f <= prm->edges_hz[b + 1]) {
                sc.bin[j] = (signed char)((k > 0 ? 0 : 1) * nb + b);
                break;
            }
    }
    for (int k = 0; k < sc.nsub; ++k) {
        sc.lo[k] = 0;
        sc.hi[k] = -1;
    }
    for (int j = 0; j < F; ++j)
        if (sc.bin[j] >= 0) {
            const int k = sc.bin[j];
            if (sc.hi[k] < 0) sc.lo[k] = (short)j;
            sc.hi[k] = (short)j;
        }
    for (int k = 0; R1 && k < sc.nsub; ++k) {
        const int R2 = F / R1, first = sc.lo[k] / R2, last = std::max<int>(sc.hi[k], 0) / R2;
        sc.nw[k] = last - first < R1 / 4 ? 1 : 2;
        sc.r0[k] = (signed char)std::min(first, R1 - sc.nw[k] * (R1 / 4));
    }
    const int out = !A ? SP_OUT_COMPLEX : enh == ULM_ENH_XDOPPLER ? SP_OUT_XDOPPLER : SP_OUT_COHERENT;
    const size_t smem = (size_t)2 * F * SP_G * sizeof(float2) + (size_t)sc.ntw * sizeof(float2) +
                        (out != SP_OUT_COMPLEX ? (size_t)sc.nsub * F * sizeof(unsigned) : 0) + (size_t)F;
    const long long ngroups = 2LL * g.S * g.nz * ((g.N + SP_TL - 1) / SP_TL);
    unsigned* Mu = reinterpret_cast<unsigned*>(M);
    if (out != SP_OUT_COMPLEX) {
        cudaError_t e = cudaMemsetAsync(M, 0, sizeof(float) * (size_t)sc.nsub * F, h->stream);
        if (e != cudaSuccess) return cuda_check(h, e, "separation maxima");
    }
    const int mx = (F * SP_G + SP_THREADS - 1) / SP_THREADS;
#define SP_ARGS h, kern, threads, planes, (int)pt, sc, g.S, g.nz, g.N, sub, A, Mu, smem, ngroups
#define SP_LAUNCH(KERN, V, THREADS)                                                                             \
    {                                                                                                           \
        auto kern = out == SP_OUT_XDOPPLER   ? KERN<V, SP_OUT_XDOPPLER>                                         \
                    : out == SP_OUT_COHERENT ? KERN<V, SP_OUT_COHERENT>                                         \
                                             : KERN<V, SP_OUT_COMPLEX>;                                         \
        const int threads = THREADS;                                                                            \
        return launch_sep(SP_ARGS);                                                                             \
    }
    if (R1 == 20) SP_LAUNCH(k_separate_win, 20, 20 * SP_G)
    if (R1 == 16) SP_LAUNCH(k_separate_win, 16, 16 * SP_G)
    if (R1 == 12) SP_LAUNCH(k_separate_win, 12, 12 * SP_G)
    if (mx <= 8) SP_LAUNCH(k_separate, 8, SP_THREADS)
    if (mx <= 19) SP_LAUNCH(k_separate, 19, SP_THREADS)
    SP_LAUNCH(k_separate, 32, SP_THREADS)
#undef SP_LAUNCH
#undef SP_ARGS
}
