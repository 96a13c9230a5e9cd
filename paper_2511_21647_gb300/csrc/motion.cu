// Projection-based rigid motion estimation (Sec. II-A3, Fig. 1d): Fourier-
// domain cross-correlation of every frame's Stage-1 slices with frame 0.
//
// The slices are zero-padded to Zp x Xp (Zp the next power of two >= nzs,
// Xp = N) and transformed by hand-written FFTs in registers: 16 points per thread,
// n = 16 T points by T threads, one exchange through shared memory per transform.
//   k_mo_twiddles   exp(-2 pi i k / n) for both axes (double, rounded)
//   k_mo_rows       forward FFT of every slice row and the row energies
//   k_mo_cols       per 16-column tile of one slice: forward FFT of each column; for
//                   frame 0 the 2D spectrum is kept as the reference, otherwise it is
//                   multiplied by the reference's conjugate and transformed back
//                   along the columns, in place
//   k_mo_peak       inverse FFT of a share of a slice's rows and the peak of |R| in
//                   them (first in row-major order on ties); the last share of a slice
//                   takes the peak of all, its four neighbours for the parabolic
//                   sub-pixel refinement, the NCC
//   k_mo_combine    RC / CR averaging into one 3D displacement per frame
// No scaling in either direction: R comes out Zp Xp times the correlation.  A
// spectrum stays in the order the forward transform leaves it in (positions along
// x, registers along z): the pointwise product and the inverse take it as it is.
// Frames go through in chunks whose spectra stay in the L2 cache, so that HBM sees
// the slices once.  300 frames of the paper's slices: 4.5 ms with radix-4 passes in
// shared memory (rows 0.92, columns 2.43, peak 1.15) and 64-frame chunks; 1.77 with these
// kernels, 1.66 with dependent launches (chunks of 32 MB: 2.30, too few CTAs per
// launch; of 96 MB: 1.99, past the L2; both without those).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "rca_internal.cuh"

namespace {

#define MO_TILE 16        // columns per k_mo_cols CTA
#define MO_TP (MO_TILE + 1)  // padded tile row: a warp's column walk spreads over the banks
#define MO_PEAK_ROWS 128   // rows per k_mo_peak CTA
#define MO_CHUNK_BYTES (size_t)(64 << 20)   // spectra of one chunk of frames (L2: 129 MB)

__device__ __forceinline__ float2 c_add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 c_sub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 c_mul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ float2 c_mulc(float2 a, float2 b) { return make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y); }

// twiddles w_n^k = exp(-2 pi i k / n), k < n, for n = Xp and then n = Zp
__global__ void k_mo_twiddles(int xp, int zp, float2* __restrict__ tw)
{
    grid_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= xp + zp) return;
    const int n = i < xp ? xp : zp, k = i < xp ? i : i - xp;
    double s, c;
    sincospi(-2.0 * (double)k / (double)n, &s, &c);
    tw[i] = make_float2((float)c, (float)s);
}

// ---------------------------------------------------------------------------
// transforms of N values in registers, natural order in and out, no scaling
// ---------------------------------------------------------------------------
// v times w_32^m (forward, exp(-2 pi i m / 32)) or its conjugate
template <bool INV>
__device__ __forceinline__ float2 mul_w32(float2 v, int m)
{
    // cos(pi m / 16), m = 0 .. 8
    constexpr float C[9] = {1.0f, 0.98078528040323044913f, 0.92387953251128675613f, 0.83146961230254523708f,
                            0.70710678118654752440f, 0.55557023301960222474f, 0.38268343236508977173f,
                            0.19509032201612826785f, 0.0f};
    m &= 31;
    if (m == 0) return v;
    if (m == 16) return make_float2(-v.x, -v.y);
    if (m == 8) return INV ? make_float2(-v.y, v.x) : make_float2(v.y, -v.x);
    if (m == 24) return INV ? make_float2(v.y, -v.x) : make_float2(-v.y, v.x);
    const int q = m & 15;
    float c = q <= 8 ? C[q] : -C[16 - q], s = q <= 8 ? C[8 - q] : C[q - 8];   // cos, sin of pi q / 16
    if (m > 16) c = -c, s = -s;
    return c_mul(v, make_float2(c, INV ? s : -s));
}

template <bool INV>
__device__ __forceinline__ void dft4(float2& a, float2& b, float2& c, float2& d)
{
    const float2 s = c_add(a, c), t = c_sub(a, c), u = c_add(b, d), w = c_sub(b, d);
    const float2 r = INV ? make_float2(-w.y, w.x) : make_float2(w.y, -w.x);
    a = c_add(s, u), b = c_add(t, r), c = c_sub(s, u), d = c_sub(t, r);
}

template <int N, bool INV>
__device__ __forceinline__ void dft(float2* v)
{
    if constexpr (N == 2) {
        const float2 a = v[0], b = v[1];
        v[0] = c_add(a, b), v[1] = c_sub(a, b);
    } else if constexpr (N == 4) {
        dft4<INV>(v[0], v[1], v[2], v[3]);
    } else if constexpr (N == 8) {
        float2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        dft4<INV>(e[0], e[1], e[2], e[3]);
        dft4<INV>(o[0], o[1], o[2], o[3]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 t = mul_w32<INV>(o[k], 4 * k);
            v[k] = c_add(e[k], t), v[k + 4] = c_sub(e[k], t);
        }
    } else if constexpr (N == 16) {
        float2 u[16];
#pragma unroll
        for (int b = 0; b < 4; ++b) {            // over n = 4 a + b
            float2 w[4] = {v[b], v[4 + b], v[8 + b], v[12 + b]};
            dft4<INV>(w[0], w[1], w[2], w[3]);
#pragma unroll
            for (int k = 0; k < 4; ++k) u[4 * k + b] = mul_w32<INV>(w[k], 2 * b * k);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            dft4<INV>(u[4 * k], u[4 * k + 1], u[4 * k + 2], u[4 * k + 3]);
#pragma unroll
            for (int b = 0; b < 4; ++b) v[k + 4 * b] = u[4 * k + b];
        }
    }
}

// ---------------------------------------------------------------------------
// n = 16 T points by T threads of a warp (T = 2 .. 32).  Thread t holds the points
// t + T j; over j they become A[t][k1] w_n^{t k1}, and over t, X[k1 + 16 k2].
// After the exchange a thread holds, for T <= 16, all k2 of k1 = t + T g
// (register g T + k2), for T = 32 k2 = 16 (t & 1) .. + 15 of k1 = t / 2 (the two
// halves of the 32-point sum meet in one shuffle).  `buf(k1, t)` is the address
// of the exchange cell; w[k1] = w_n^{t k1}.
// ---------------------------------------------------------------------------
template <int T, typename Buf>
__device__ __forceinline__ void fft_fwd(float2 v[16], const float2 w[16], int t, Buf buf)
{
    dft<16, false>(v);
    __syncwarp();                                // the buffer's last readers are done
#pragma unroll
    for (int k = 0; k < 16; ++k) *buf(k, t) = k ? c_mul(v[k], w[k]) : v[0];
    __syncwarp();
    if constexpr (T <= 16) {
#pragma unroll
        for (int g = 0; g < 16 / T; ++g) {
#pragma unroll
            for (int u = 0; u < T; ++u) v[g * T + u] = *buf(t + T * g, u);
            dft<T, false>(v + g * T);
        }
    } else {
        const int s = t & 1;
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = *buf(t >> 1, 2 * u + s);
        dft<16, false>(v);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const float2 x = mul_w32<false>(v[k], k);
            const float2 m = make_float2(s ? x.x : v[k].x, s ? x.y : v[k].y);
            const float2 o = make_float2(__shfl_xor_sync(0xffffffffu, m.x, 1), __shfl_xor_sync(0xffffffffu, m.y, 1));
            v[k] = s ? c_sub(o, m) : c_add(m, o);
        }
    }
}

template <int T, typename Buf>
__device__ __forceinline__ void fft_inv(float2 v[16], const float2 w[16], int t, Buf buf)
{
    __syncwarp();                                // the buffer's last readers are done
    if constexpr (T <= 16) {
#pragma unroll
        for (int g = 0; g < 16 / T; ++g) {
            dft<T, true>(v + g * T);
#pragma unroll
            for (int u = 0; u < T; ++u) *buf(t + T * g, u) = v[g * T + u];
        }
    } else {
        const int s = t & 1;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const float2 o = make_float2(__shfl_xor_sync(0xffffffffu, v[k].x, 1), __shfl_xor_sync(0xffffffffu, v[k].y, 1));
            const float2 d = mul_w32<true>(c_sub(o, v[k]), k), e = c_add(v[k], o);
            v[k] = make_float2(s ? d.x : e.x, s ? d.y : e.y);
        }
        dft<16, true>(v);
#pragma unroll
        for (int u = 0; u < 16; ++u) *buf(t >> 1, 2 * u + s) = v[u];
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float2 x = *buf(k, t);
        v[k] = k ? c_mulc(x, w[k]) : x;
    }
    dft<16, true>(v);
}

template <int T>
__device__ __forceinline__ void load_twiddles(float2 w[16], const float2* __restrict__ tw, int t)
{
#pragma unroll
    for (int k = 0; k < 16; ++k) w[k] = __ldg(tw + t * k);     // t k < 16 T
}

// exchange cells of one row transform: [k1][t], the rows of a warp 16 banks apart
template <int T>
struct RowBuf {
    static constexpr int LD = T + 1, RS = (16 * LD + 15) / 16 * 16 + 8;
    float2* p;
    __device__ __forceinline__ float2* operator()(int k, int t) const { return p + k * LD + t; }
};

// warps per row-transform CTA (the exchange cells of short rows take more space)
template <int T>
constexpr int ROW_WARPS = T <= 4 ? 4 : 8;

// position of register r of thread t in a row's spectrum
template <int T>
__device__ __forceinline__ int spec_pos(int r, int t)
{
    return r * T + t;
}

// forward FFT of the slice rows of frames frame_base ..; B[f - frame_base][k][zp rows][Xp] (rows < nzs),
// E[f][k][z] = sum |s|^2
template <int T>
__global__ void __launch_bounds__(32 * ROW_WARPS<T>) k_mo_rows(const float2* __restrict__ sl, int nt, int nzs, int zp,
                                                 const float2* __restrict__ tw, int frame_base, float2* __restrict__ B,
                                                 float* __restrict__ E)
{
    grid_wait();
    constexpr int XP = 16 * T, RW = 32 / T;              // rows per warp
    __shared__ float2 smo[ROW_WARPS<T> * RW * RowBuf<T>::RS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t = lane % T, r = lane / T;
    const RowBuf<T> buf{smo + (warp * RW + r) * RowBuf<T>::RS};
    const size_t fk = (size_t)(frame_base + blockIdx.z) * nt + blockIdx.y, lk = (size_t)blockIdx.z * nt + blockIdx.y;
    float2 w[16];
    load_twiddles<T>(w, tw, t);
    const int z = (blockIdx.x * ROW_WARPS<T> + warp) * RW + r;
    const bool in = z < nzs;
    float2 v[16];
    float e = 0.f;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        v[j] = in ? __ldcs(sl + (fk * nzs + z) * XP + t + T * j) : make_float2(0.f, 0.f);
        e = fmaf(v[j].x, v[j].x, fmaf(v[j].y, v[j].y, e));
    }
#pragma unroll
    for (int o = T / 2; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    fft_fwd<T>(v, w, t, buf);
    if (!in) return;
    float2* dst = B + (lk * zp + z) * XP;
#pragma unroll
    for (int q = 0; q < 16; ++q) dst[spec_pos<T>(q, t)] = v[q];
    if (t == 0) E[fk * nzs + z] = e;
}

// Column pass over a 16-column tile of one slice, in place on B (zp rows per slice).
// KEEP: frame 0, the 2D spectrum goes to ref, in register order: pair q of thread t of
// column x of transmission k at ((k Xp + x) 8 + q) T + t.  Otherwise multiply by
// conj(ref) and transform back.
template <int T, bool KEEP>
__global__ void __launch_bounds__(T < 16 ? 16 * T : 256, 2) k_mo_cols(float2* __restrict__ B, int nt, int nzs, int xp,
                                                                      const float2* __restrict__ twz,
                                                                      float4* __restrict__ ref)
{
    grid_wait();
    constexpr int ZP = 16 * T, LDZ = T + 2;              // exchange cell (k1, t) in tile row k1 LDZ + t
    extern __shared__ float2 tile[];                     // [16 LDZ][MO_TP]
    const int x0 = blockIdx.x * MO_TILE, k = blockIdx.y;
    float2* Bk = B + ((size_t)blockIdx.z * nt + k) * ZP * xp + x0;
    // element i of the tile: row i / MO_TILE, column i % MO_TILE
    for (int i = threadIdx.x; i < ZP * MO_TILE; i += blockDim.x) {
        const int z = i / MO_TILE, c = i % MO_TILE;
        tile[z * MO_TP + c] = z < nzs ? Bk[(size_t)z * xp + c] : make_float2(0.f, 0.f);
    }
    const int t = threadIdx.x % T;
    float2 w[16];
    load_twiddles<T>(w, twz, t);
    __syncthreads();
    for (int c = threadIdx.x / T; c < MO_TILE; c += blockDim.x / T) {
        float2* col = tile + c;
        auto buf = [&](int k1, int u) { return col + (k1 * LDZ + u) * MO_TP; };
        float2 v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = col[(t + T * j) * MO_TP];
        fft_fwd<T>(v, w, t, buf);
        float4* rc = ref + ((size_t)k * xp + x0 + c) * 8 * T + t;
        if constexpr (KEEP) {
#pragma unroll
            for (int q = 0; q < 8; ++q) rc[q * T] = make_float4(v[2 * q].x, v[2 * q].y, v[2 * q + 1].x, v[2 * q + 1].y);
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 r = __ldg(rc + q * T);
                v[2 * q] = c_mulc(v[2 * q], make_float2(r.x, r.y));
                v[2 * q + 1] = c_mulc(v[2 * q + 1], make_float2(r.z, r.w));
            }
            fft_inv<T>(v, w, t, buf);
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 16; ++j) col[(t + T * j) * MO_TP] = v[j];
        }
    }
    if constexpr (!KEEP) {
        __syncthreads();
        for (int i = threadIdx.x; i < ZP * MO_TILE; i += blockDim.x) {
            const int z = i / MO_TILE, c = i % MO_TILE;
            Bk[(size_t)z * xp + c] = tile[z * MO_TP + c];
        }
    }
}

// the column pass of up to 16 rows: a thread per column
template <int ZP, bool KEEP>
__global__ void k_mo_cols_short(float2* __restrict__ B, int nt, int nzs, int xp, float2* __restrict__ ref)
{
    grid_wait();
    const int x = threadIdx.x, k = blockIdx.y;
    float2* Bk = B + ((size_t)blockIdx.z * nt + k) * ZP * xp + x;
    float2 v[ZP];
#pragma unroll
    for (int z = 0; z < ZP; ++z) v[z] = z < nzs ? Bk[(size_t)z * xp] : make_float2(0.f, 0.f);
    dft<ZP, false>(v);
#pragma unroll
    for (int z = 0; z < ZP; ++z) {
        float2* r = ref + ((size_t)k * ZP + z) * xp + x;
        if constexpr (KEEP) *r = v[z];
        else v[z] = c_mulc(v[z], *r);
    }
    if constexpr (!KEEP) {
        dft<ZP, true>(v);
#pragma unroll
        for (int z = 0; z < ZP; ++z) Bk[(size_t)z * xp] = v[z];
    }
}

// inverse FFT of the row at `src` (spectrum positions) into v[j] = R[t + T j]
template <int T>
__device__ __forceinline__ void mo_row_inv(const float2* __restrict__ src, float2 v[16], const float2 w[16], int t,
                                           const RowBuf<T>& buf)
{
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = src[spec_pos<T>(q, t)];
    fft_inv<T>(v, w, t, buf);
}

__device__ __forceinline__ void mo_better(float& best, int& idx, float m, int i)
{
    if (m > best || (m == best && i < idx)) {
        best = m;
        idx = i;
    }
}

// sub-pixel peak and NCC of one slice from the peaks of its shares (one warp)
template <int T>
__device__ __forceinline__ void mo_finish(const float2* __restrict__ Cs, const float* __restrict__ E, int k, int f, int nt,
                                          int nzs, int zp, const float2 w[16], const RowBuf<T>& buf, float (*mag)[16 * T],
                                          int npart, const float* pbest, const int* pidx, float* __restrict__ shifts,
                                          int* __restrict__ peaks)
{
    constexpr int XP = 16 * T;
    const int lane = threadIdx.x & 31, t = lane % T, r = lane / T;
    float best = -1.f;
    int idx = 0x7fffffff;
    for (int q = lane; q < npart; q += 32) mo_better(best, idx, __ldcg(pbest + q), __ldcg(pidx + q));
    float e0 = 0.f, e1 = 0.f;                            // frame energies (row sums of |s|^2)
    for (int z = lane; z < nzs; z += 32) {
        e0 += E[((size_t)f * nt + k) * nzs + z];
        e1 += E[(size_t)k * nzs + z];
    }
    for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
        mo_better(best, idx, ob, oi);
        e0 += __shfl_xor_sync(0xffffffffu, e0, o);
        e1 += __shfl_xor_sync(0xffffffffu, e1, o);
    }
    if (idx == 0x7fffffff) idx = 0;                      // no comparable value (NaN throughout)
    const int iz = idx / XP, ix = idx % XP;
    // neighbours: rows iz - 1 and iz + 1 at ix, row iz at ix - 1 and ix + 1 (circular)
#pragma unroll 1
    for (int q = 0; q < 3; ++q) {
        float2 v[16];
        mo_row_inv<T>(Cs + (size_t)((iz + q + zp - 1) & (zp - 1)) * XP, v, w, t, buf);
        if (r == 0)
#pragma unroll
            for (int j = 0; j < 16; ++j) mag[q][t + T * j] = sqrtf(v[j].x * v[j].x + v[j].y * v[j].y);
    }
    __syncwarp();
    if (lane != 0) return;
    const float m0 = sqrtf(best);
    auto para = [](float mm, float m, float mp) {
        const float den = mm - 2.f * m + mp;
        if (den >= 0.f) return 0.f;
        return fminf(0.5f, fmaxf(-0.5f, (mm - mp) / (2.f * den)));
    };
    const int dz = iz < zp / 2 ? iz : iz - zp, dx = ix < XP / 2 ? ix : ix - XP;
    const float den = sqrtf(e0) * sqrtf(e1) * (float)zp * (float)XP;
    float* o = shifts + ((size_t)f * nt + k) * 3;
    o[0] = (float)dz + para(mag[0][ix], m0, mag[2][ix]);
    o[1] = (float)dx + para(mag[1][(ix + XP - 1) & (XP - 1)], m0, mag[1][(ix + 1) & (XP - 1)]);
    o[2] = den > 0.f ? m0 / den : 0.f;
    if (peaks) {
        peaks[((size_t)f * nt + k) * 2] = dz;
        peaks[((size_t)f * nt + k) * 2 + 1] = dx;
    }
}

// peak of |R|^2 over MO_PEAK_ROWS rows of one slice; the CTA that is the last of its
// slice to write its share finishes the slice (`count`: zero before the first launch,
// and again after every slice)
template <int T>
__global__ void __launch_bounds__(32 * ROW_WARPS<T>) k_mo_peak(const float2* __restrict__ C, const float* __restrict__ E,
                                                               int nt, int nzs, int zp, const float2* __restrict__ tw,
                                                               int frame_base, float* pbest, int* pidx,
                                                               unsigned* __restrict__ count, float* __restrict__ shifts,
                                                               int* __restrict__ peaks)
{
    grid_wait();
    constexpr int XP = 16 * T, RW = 32 / T;
    __shared__ float2 smo[ROW_WARPS<T> * RW * RowBuf<T>::RS];
    __shared__ float s_best[8];
    __shared__ int s_idx[8];
    __shared__ bool s_last;
    __shared__ float mag[3][XP];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t = lane % T, r = lane / T;
    const RowBuf<T> buf{smo + (warp * RW + r) * RowBuf<T>::RS};
    float2 w[16];
    load_twiddles<T>(w, tw, t);
    const size_t slice = (size_t)blockIdx.z * nt + blockIdx.y;
    const float2* Cs = C + slice * zp * XP;
    float best = -1.f;
    int idx = 0x7fffffff;
    const int z1 = min(zp, (int)(blockIdx.x + 1) * MO_PEAK_ROWS);
    for (int zb = blockIdx.x * MO_PEAK_ROWS + warp * RW; zb < z1; zb += ROW_WARPS<T> * RW) {
        const int z = zb + r;                            // past the slice only for fewer rows than a warp takes
        float2 v[16];
        mo_row_inv<T>(Cs + (size_t)min(z, zp - 1) * XP, v, w, t, buf);
        if (z < zp)
#pragma unroll
            for (int j = 0; j < 16; ++j) mo_better(best, idx, v[j].x * v[j].x + v[j].y * v[j].y, z * XP + t + T * j);
    }
    for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
        mo_better(best, idx, ob, oi);
    }
    if (lane == 0) {
        s_best[warp] = best;
        s_idx[warp] = idx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < ROW_WARPS<T>; ++q) mo_better(best, idx, s_best[q], s_idx[q]);
        pbest[slice * gridDim.x + blockIdx.x] = best;
        pidx[slice * gridDim.x + blockIdx.x] = idx;
        __threadfence();
        s_last = atomicAdd(count + slice, 1u) == gridDim.x - 1;
        if (s_last) count[slice] = 0;
        __threadfence();
    }
    __syncthreads();
    if (s_last && warp == 0)
        mo_finish<T>(Cs, E, blockIdx.y, frame_base + blockIdx.z, nt, nzs, zp, w, buf, mag, gridDim.x,
                     pbest + slice * gridDim.x, pidx + slice * gridDim.x, shifts, peaks);
}

// motion[f] = (x_RC pitch, y_CR pitch, (z_RC + z_CR) / 2 dz / us), averages over each family's K
__global__ void k_mo_combine(const float* __restrict__ shifts, int F, int K, double pitch, double row_m,
                             float* __restrict__ motion)
{
    grid_wait();
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= F) return;
    const float* s = shifts + (size_t)f * 2 * K * 3;
    double zr = 0.0, xr = 0.0, zc = 0.0, yc = 0.0;
    for (int k = 0; k < K; ++k) {
        zr += s[k * 3];
        xr += s[k * 3 + 1];
        zc += s[(K + k) * 3];
        yc += s[(K + k) * 3 + 1];
    }
    motion[f * 3] = (float)(xr / K * pitch);
    motion[f * 3 + 1] = (float)(yc / K * pitch);
    motion[f * 3 + 2] = (float)(0.5 * (zr + zc) / K * row_m);
}

int ilog2(int v)
{
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

struct MotionBufs {
    float2 *tw, *B;
    float4* ref;
    float *E, *shifts, *pbest;
    int *pidx, *peaks;
    unsigned* count;
};

// the column pass of nf frames (KEEP: of frame 0, into the reference)
template <bool KEEP>
cudaError_t launch_cols(cudaStream_t s, const MotionBufs& b, int nt, int nzs, int xp, int logz, int nf)
{
    const float2* twz = b.tw + xp;
    auto tiled = [&](auto tc) {
        constexpr int T = decltype(tc)::value;
        const int smem = 16 * (T + 2) * MO_TP * (int)sizeof(float2);
        const cudaError_t e = cudaFuncSetAttribute(k_mo_cols<T, KEEP>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        launch_chain(k_mo_cols<T, KEEP>, dim3(xp / MO_TILE, nt, nf), dim3(T < 16 ? 16 * T : 256), smem, s, b.B, nt, nzs, xp, twz, b.ref);
        return cudaGetLastError();
    };
    auto few = [&](auto zc) {
        launch_chain(k_mo_cols_short<decltype(zc)::value, KEEP>, dim3(1, nt, nf), dim3(xp), 0, s, b.B, nt, nzs, xp, (float2*)b.ref);
        return cudaGetLastError();
    };
    switch (logz) {
    case 1: return few(std::integral_constant<int, 2>());
    case 2: return few(std::integral_constant<int, 4>());
    case 3: return few(std::integral_constant<int, 8>());
    case 4: return few(std::integral_constant<int, 16>());
    case 5: return tiled(std::integral_constant<int, 2>());
    case 6: return tiled(std::integral_constant<int, 4>());
    case 7: return tiled(std::integral_constant<int, 8>());
    case 8: return tiled(std::integral_constant<int, 16>());
    default: return tiled(std::integral_constant<int, 32>());
    }
}

// all frames, T threads per row
template <int T>
cudaError_t run_motion(cudaStream_t s, const MotionBufs& b, const float2* slices, int F, int nt, int nzs, int logz, int chunk)
{
    constexpr int XP = 16 * T, RB = ROW_WARPS<T> * (32 / T);   // rows per k_mo_rows CTA
    const int zp = 1 << logz, npart = (zp + MO_PEAK_ROWS - 1) / MO_PEAK_ROWS;
    launch_chain(k_mo_twiddles, dim3((XP + zp + 255) / 256), dim3(256), 0, s, XP, zp, b.tw);
    for (int f0 = 0; f0 < F; f0 += chunk) {
        const int nf = std::min(chunk, F - f0);
        launch_chain(k_mo_rows<T>, dim3((nzs + RB - 1) / RB, nt, nf), dim3(32 * ROW_WARPS<T>), 0, s, slices, nt, nzs, zp, b.tw, f0, b.B, b.E);
        cudaError_t e = cudaSuccess;
        if (f0 == 0 && (e = launch_cols<true>(s, b, nt, nzs, XP, logz, 1)) != cudaSuccess) return e;
        if ((e = launch_cols<false>(s, b, nt, nzs, XP, logz, nf)) != cudaSuccess) return e;
        launch_chain(k_mo_peak<T>, dim3(npart, nt, nf), dim3(32 * ROW_WARPS<T>), 0, s, b.B, b.E, nt, nzs, zp, b.tw, f0, b.pbest, b.pidx,
                                                                       b.count, b.shifts, b.peaks);
    }
    return cudaGetLastError();
}

}  // namespace

rca_status launch_motion(rca_handle* h, const rca_tables* t, const float2* slices, int F, float* motion,
                         float* shifts_out, int* peaks)
{
    const GeomDev& g = t->gd;
    const int nt = 2 * g.K, nzs = g.nzs, xp = g.N;
    if (xp < 32 || xp > 256 || (xp & (xp - 1)))
        return set_error(h, RCA_ERR_UNSUPPORTED, "motion estimation needs a power-of-two N in [32, 256] (N = %d)", xp);
    const int logz = ilog2(nzs), zp = 1 << logz;
    // a column is 16 points in each of at most 32 threads
    if (zp > 512) return set_error(h, RCA_ERR_UNSUPPORTED, "motion estimation supports at most 512 slice rows");
    // workspace: twiddles, B [chunk][2K][Zp][Xp], the reference spectrum [2K][Xp][Zp], E [F][2K][nzs],
    // shifts [F][2K][3], peaks of the shares and their counts
    const size_t frame = (size_t)nt * zp * xp * 8;
    const int chunk = (int)std::min<size_t>(F, std::max<size_t>(1, MO_CHUNK_BYTES / frame));
    const int npart = (zp + MO_PEAK_ROWS - 1) / MO_PEAK_ROWS;
    const size_t n_part = (size_t)chunk * nt * npart;
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t sizes[8] = {up((size_t)(xp + zp) * 8), up(chunk * frame), up(frame), up((size_t)F * nt * nzs * 4),
                             up((size_t)F * nt * 3 * 4), up(n_part * 4), up(n_part * 4),
                             up((size_t)chunk * nt * 4)};
    size_t bytes = 0;
    for (size_t s : sizes) bytes += s;
    rca_status st = RCA_OK;
    char* ws = (char*)ws_get(h, WS_MOTION, bytes, &st);
    if (!ws) return st;
    char* at[8];
    for (int q = 0; q < 8; ++q) {
        at[q] = ws;
        ws += sizes[q];
    }
    MotionBufs b{(float2*)at[0], (float2*)at[1], (float4*)at[2], (float*)at[3], shifts_out ? shifts_out : (float*)at[4],
                 (float*)at[5], (int*)at[6], peaks, (unsigned*)at[7]};
    cudaError_t e = cudaMemsetAsync(b.count, 0, (size_t)chunk * nt * 4, h->stream);
    if (e != cudaSuccess) return cuda_check(h, e, "motion counters");
    switch (xp) {
    case 32: e = run_motion<2>(h->stream, b, slices, F, nt, nzs, logz, chunk); break;
    case 64: e = run_motion<4>(h->stream, b, slices, F, nt, nzs, logz, chunk); break;
    case 128: e = run_motion<8>(h->stream, b, slices, F, nt, nzs, logz, chunk); break;
    default: e = run_motion<16>(h->stream, b, slices, F, nt, nzs, logz, chunk); break;
    }
    if (e != cudaSuccess) return cuda_check(h, e, "motion kernels");
    launch_chain(k_mo_combine, dim3((F + 127) / 128), dim3(128), 0, h->stream, b.shifts, F, g.K, g.pitch, g.dz / g.us, motion);
    return cuda_check(h, cudaGetLastError(), "motion kernels");
}
