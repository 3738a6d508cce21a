// What the paper's fitter takes besides the NLL and its gradient (Sec. 4, 5:
// FUMILI needs the gradient and an approximation of the Hessian; plots of the
// fit weight the accepted MC events with the fitted intensity).
//
// FUMILI's approximation of the NLL Hessian in the real parameters
// p = (Re V_0..Re V_{N-1}, Im V_0..): the second derivatives of the intensity
// are dropped in both terms of Eq. 3 (they cancel in expectation at the
// minimum), leaving
//   H = sum_i d_i d_i^T,   d_i = grad_p ln I_i = 2 (Re, Im) of conj(A_a(i)) S_i / I_i.
// One half of a block's warps forms d_i, one event to a thread (S by a
// compensated dot product with V as a float pair), into a shared-memory tile J
// of 256 events x 2NP columns (Re parts at 0..NP-1, Im parts at NP..2NP-1,
// zero-padded), one tile ahead of the other half, which adds up the upper
// triangle of J^T J in 8x8 blocks over event groups: FP32 within a run of tiles,
// float pairs across runs, event groups and blocks, summed in a fixed order. This kernel serves samples of
// more than 20 waves (and PWA_HESS_KERNEL=generic); up to 20 waves the tensor-
// core kernel of k_hess_tc.cu forms the same sum.
//
// Projection weights: w_j = I(Omega_j) / N_gen per accepted MC event (their
// sum is V^H M V), and fit fractions F_ab = Re(conj(V_a) M_ab V_b) / V^H M V.
#include "amp_kernel.cuh"
#include "ff.cuh"
#include "pwa_internal.cuh"

namespace pwa {

namespace {

constexpr int kHT = 256;     // events per tile = threads per block
constexpr int kFlush = 8;    // tiles summed in FP32 before the float-float add

// Amplitudes of event i into ar, ai (zero for padded waves a >= N). Every
// load is unconditional (a padded wave re-reads wave 0, then is zeroed by a
// select) so that all 2NP loads are in flight together.
template <int NP>
__device__ __forceinline__ void load_event(const float *__restrict__ pl, int64_t pitch, int64_t i,
                                           int N, float *ar, float *ai)
{
#pragma unroll
    for (int w = 0; w < NP; ++w) {
        const int64_t o = (w < N ? 2 * w : 0) * pitch + i;
        const float x = __ldg(pl + o), y = __ldg(pl + o + pitch);
        ar[w] = w < N ? x : 0.f;
        ai[w] = w < N ? y : 0.f;
    }
}

// S = sum_a V_a A_a in FP32, in four independent FMA chains (waves a = c mod 4
// in chain c) joined pairwise. |S - S_exact| <= gamma_{N/4+3} sum_a |V_a A_a|
// per component, V rounded to float. Padded waves have A = 0 and V = 0.
template <int NP>
__device__ __forceinline__ void dot4(const float *ar, const float *ai, const float *vf, float &sr,
                                     float &si)
{
    float r[4] = {0.f, 0.f, 0.f, 0.f}, m[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int w = 0; w < NP; ++w) {
        const float x = ar[w], y = ai[w], vr = vf[2 * w], vi = vf[2 * w + 1];
        r[w & 3] = fmaf(x, vr, fmaf(-y, vi, r[w & 3]));
        m[w & 3] = fmaf(x, vi, fmaf(y, vr, m[w & 3]));
    }
    sr = (r[0] + r[1]) + (r[2] + r[3]);
    si = (m[0] + m[1]) + (m[2] + m[3]);
}

// V as float pairs for dot2x4: per wave (vr, vi, -vr, -vi), (-vi, vr, vi, -vr)
// of the high parts and (lr, li, -li, lr) of the low ones.
__device__ __forceinline__ void load_v2(const double *V, int N, int np, float4 *vt)
{
    for (int w = threadIdx.x; w < np; w += blockDim.x) {
        const double r = w < N ? V[2 * w] : 0.0, i = w < N ? V[2 * w + 1] : 0.0;
        const float hr = (float)r, hi = (float)i;
        const float lr = (float)(r - (double)hr), li = (float)(i - (double)hi);
        vt[3 * w] = make_float4(hr, hi, -hr, -hi);
        vt[3 * w + 1] = make_float4(-hi, hr, hi, -hr);
        vt[3 * w + 2] = make_float4(lr, li, -li, lr);
    }
}

// S = sum_a (Vh + Vl)_a A_a, compensated (Dot2 of Ogita, Rump and Oishi: each
// product split exactly by FMA, TwoSum of the high parts) in four chains
// (waves a = c mod 4) joined by TwoSum, Re S and Im S as a packed pair; the Vl
// terms in plain FMA. The result is within about 2^-24 |S| + N^2 2^-48
// sum_a |V_a A_a| of the exact sum.
template <int NP>
__device__ __forceinline__ void dot2x4(const float *ar, const float *ai, const float4 *vt, float &sr,
                                       float &si)
{
    f2 s[4] = {0, 0, 0, 0}, c[4] = {0, 0, 0, 0}, l = 0;
#pragma unroll
    for (int w = 0; w < NP; ++w) {
        const int j = w & 3;
        const f2 x = dup2(ar[w]), y = dup2(ai[w]);
        const float4 a = vt[3 * w], b = vt[3 * w + 1], d = vt[3 * w + 2];
        dot2_step(s[j], c[j], x, pk2(a.x, a.y), pk2(a.z, a.w));  // (x vr, x vi)
        dot2_step(s[j], c[j], y, pk2(b.x, b.y), pk2(b.z, b.w));  // (-y vi, y vr)
        l = fma2(x, pk2(d.x, d.y), fma2(y, pk2(d.z, d.w), l));
    }
#pragma unroll
    for (int j = 1; j < 4; ++j) {
        const ff t = ff_two_sum(s[0], s[j]);
        s[0] = t.h;
        c[0] = add2(c[0], add2(t.l, c[j]));
    }
    upk2(add2(s[0], add2(c[0], l)), sr, si);
}

__device__ __forceinline__ void load_v(const double *V, int N, int np2, float *vf)
{
    for (int c = threadIdx.x; c < np2; c += blockDim.x)
        vf[c] = c < 2 * N ? __double2float_rn(V[c]) : 0.f;
}

// Work split of the Hessian kernel for np padded waves: PP = 2 np padded
// parameters in B 4-column blocks, NB 4x4 blocks of the upper triangle, whose
// sums run over EG groups of events (event e of a tile to group e mod EG, added
// in order: the groups fix the order of the FP32 sums).
constexpr int hess_blocks(int np) { return np / 2; }
constexpr int hess_nb(int np) { return hess_blocks(np) * (hess_blocks(np) + 1) / 2; }
// events handled by the busiest of kHT threads per tile with `it` items (block,
// group) each, plus `it` for the per-item overhead
constexpr int hess_cost(int np, int it)
{
    return (it * kHT / hess_nb(np)) < 1
               ? (1 << 20)
               : it * ((kHT + it * kHT / hess_nb(np) - 1) / (it * kHT / hess_nb(np))) + it;
}
constexpr int hess_groups(int np)
{
    const int c1 = hess_cost(np, 1), c2 = hess_cost(np, 2), c3 = hess_cost(np, 3);
    const int it = (c1 <= c2 && c1 <= c3) ? 1 : (c2 <= c3) ? 2 : 3;
    return it * kHT / hess_nb(np) > kHT ? kHT : it * kHT / hess_nb(np);
}
// 8x8 superblocks (two block rows and columns) of the upper triangle.
constexpr int hess_super(int np) { return (np / 4) * (np / 4 + 1) / 2; }
// Rows of a product thread's piece of a superblock (8 columns wide): the whole,
// or a half where two threads for each superblock and group still fit.
constexpr int hess_rows(int np)
{
    return 2 * hess_super(np) * hess_groups(np) <= kHT ? 4 : 8;
}

template <int NP>
struct HessCfg {
    static constexpr int B = hess_blocks(NP), NB = hess_nb(NP), EG = hess_groups(NP);
    static constexpr int SB = B / 2, NS = hess_super(NP);
    static constexpr int R = hess_rows(NP), PT = NS * (8 / R) * EG;
    // float4s between the rows of a tile: odd, so that the stores of 8 threads (one
    // row each) fall into different banks
    static constexpr int LD = B + 1;
    static constexpr size_t TILES = 2 * (size_t)kHT * LD * sizeof(float4);
    static constexpr size_t SUMS = (size_t)EG * NS * 64 * sizeof(float2);
    static constexpr size_t SMEM = TILES > SUMS ? TILES : SUMS;
    // Warps 0 .. PW - 1 add products. A fifth and sixth one make their two of the
    // SM's four schedulers carry twice the products of the others, which then get
    // three of the warps that form J, and the first two one each (two warps idle).
    static constexpr int PW = (PT + 31) / 32, WARPS = PW > 4 ? 16 : 12;
    static_assert(PW <= 6, "more product warps than there are");
    // the warp's place among those that form J, -1 for the others
    static __device__ __forceinline__ int j_warp(int warp)
    {
        if (PW <= 4)
            return warp - 4 < 0 ? -1 : warp - 4;
        return warp < 6 ? -1 : warp < 12 ? warp - 6 : warp < 14 ? -1 : warp - 8;
    }
};

// Place of block column x in a row of J: the even ones first, so that the
// loads of neighbouring superblocks are neighbours in the banks.
__device__ __forceinline__ constexpr int hess_place(int x, int sb) { return (x & 1) * sb + (x >> 1); }

// The sums of many FP32 runs are float pairs (this part's FP64 pipe has 1/64 of
// the FP32 rate: as doubles the conversions and sums of one block took 15 us). Every
// FP32 sum is a multiple of 2^-149, so that a pair loses nothing to underflow that
// its terms had not lost; a total that a float may not hold is added in FP64.
__device__ __forceinline__ bool is_wide(float h) { return !(fabsf(h) < 0x1p100f); }

__device__ __forceinline__ float half_of(f2 v, int odd)
{
    return __uint_as_float((unsigned)(odd ? v >> 32 : v));
}

// (h, l) += x, h + l kept to the rounding of l
__device__ __forceinline__ void sum2(float &h, float &l, float x)
{
    const float t = h + x, z = t - h;
    const float e = (h - (t - z)) + (x - z);
    l += e;
    h = t;
}

// The sum of n pairs, `stride` apart, in FP64. (A call, so that the kernels' own code
// stays as it is without it.)
__device__ __noinline__ double wide_sum(const float2 *v, int n, int stride)
{
    double d = 0.0;
#pragma unroll 1
    for (int i = 0; i < n; ++i)
        d += (double)v[(size_t)i * stride].x + (double)v[(size_t)i * stride].y;
    return d;
}

// Eight warps form J of the next tile (one event per thread, the tile after that
// being loaded) while up to six add the products of the current one; two tile
// buffers, one barrier per tile. Every kFlush tiles the FP32 sums go to float pairs
// in global scratch (they would take twice the registers of the products).
//
// Bound by instruction issue of the two parts together: at 32 waves the products
// alone take 4.3 us a tile and SM (packed FMAs, two to an instruction; single
// ones made the call a third slower), forming J alone 4.3 to 5.8, both 6.9. One
// call at 333k events x 29 waves 172 to 98 us, at 1M x 32 404 to 245 us, at 500k
// x 48 494 to 212 us, against one 256-thread role that did both in turn, with
// 4x4 blocks (two 16-byte loads for 16 products, here four for 64).
template <int NP>
__global__ void __launch_bounds__(HessCfg<NP>::WARPS * 32, 1)
    hess_kernel(const float *__restrict__ pl, int64_t pitch, int64_t n, int N, const double *V,
                float2 *partials, float2 *scratch, int *status)
{
    using C = HessCfg<NP>;
    extern __shared__ __align__(16) float J[];   // [2][kHT][LD float4s]
    __shared__ float4 vt[3 * NP];
    __shared__ int s_bad;
    load_v2(V, N, NP, vt);
    if (threadIdx.x == 0)
        s_bad = 0;
    __syncthreads();
    const int n_tiles = (int)((n + kHT - 1) / kHT);
    const int n_my = (n_tiles > (int)blockIdx.x) ? (n_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    auto tile_of = [&](int k) { return (int64_t)blockIdx.x + (int64_t)k * gridDim.x; };
    const int j_warp = C::j_warp(threadIdx.x >> 5), je = j_warp * 32 + (threadIdx.x & 31);
    // product threads: rows 8 bx + row0 .. + R - 1 and columns 8 by .. + 7 of the
    // events of group grp
    const int p = threadIdx.x;
    const bool p_thread = p < C::PT;
    int grp = 0, bx = 0, by = 0, sup = 0, half = 0;
    if (p_thread) {
        half = p % (8 / C::R);
        sup = p / (8 / C::R) % C::NS;
        grp = p / (8 / C::R * C::NS);
        by = sup;
        while (by >= C::SB - bx) {
            by -= C::SB - bx;
            ++bx;
        }
        by += bx;
    }

    if (j_warp >= 0) {
        int bad = 0;
        float xr[NP], xi[NP];
        // this thread's event of tile k (events past n read event n - 1 and are dropped)
        auto load = [&](int k) {
            load_event<NP>(pl, pitch, min(tile_of(k) * kHT + je, n - 1), N, xr, xi);
        };
        auto form = [&](int k) {
            const int64_t i = tile_of(k) * kHT + je;
            float4 *J4 = reinterpret_cast<float4 *>(J) + (size_t)(k & 1) * kHT * C::LD;
            float rr = 0.f, ri = 0.f;
            if (i < n) {
                float sr, si;
                dot2x4<NP>(xr, xi, vt, sr, si);
                const float I = fmaf(sr, sr, si * si);
                if (I > 0.f && I < INFINITY) {
                    rr = 2.f * sr / I;
                    ri = 2.f * si / I;
                } else {
                    bad = 1;
                }
            }
            // 2 Re(conj(A) S) / I and 2 Im(conj(A) S) / I (zero rows past n)
#pragma unroll
            for (int q = 0; q < NP / 4; ++q) {
                float4 re, im;
                re.x = fmaf(xr[4 * q], rr, xi[4 * q] * ri);
                re.y = fmaf(xr[4 * q + 1], rr, xi[4 * q + 1] * ri);
                re.z = fmaf(xr[4 * q + 2], rr, xi[4 * q + 2] * ri);
                re.w = fmaf(xr[4 * q + 3], rr, xi[4 * q + 3] * ri);
                im.x = fmaf(xr[4 * q], ri, -xi[4 * q] * rr);
                im.y = fmaf(xr[4 * q + 1], ri, -xi[4 * q + 1] * rr);
                im.z = fmaf(xr[4 * q + 2], ri, -xi[4 * q + 2] * rr);
                im.w = fmaf(xr[4 * q + 3], ri, -xi[4 * q + 3] * rr);
                J4[je * C::LD + hess_place(q, C::SB)] = re;
                J4[je * C::LD + hess_place(NP / 4 + q, C::SB)] = im;
            }
        };
        if (n_my > 0) {
            load(0);
            form(0);
        }
        if (n_my > 1)
            load(1);
        __syncthreads();
        for (int k = 0; k < n_my; ++k) {
            if (k + 1 < n_my)
                form(k + 1);
            if (k + 2 < n_my)
                load(k + 2);
            if (C::PW > 4 && k + 3 < n_my) {
                // 128-byte lines of the tile after that: where three of these warps share a
                // scheduler the loads are late otherwise (1M events: 32 waves 258 to 248 us,
                // 48 waves at half of them 235 to 210; 24 and 40 waves, two on each, were
                // slower by 10 us)
                const int64_t e0 = tile_of(k + 3) * kHT;
                for (int q = je; q < 2 * N * 8; q += kHT)
                    if (e0 + (q & 7) * 32 < n)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(pl + (q >> 3) * pitch + e0 +
                                                                     (q & 7) * 32));
            }
            __syncthreads();
        }
        if (bad)
            s_bad = 1;
    } else {
        f2 s[C::R][4];
#pragma unroll
        for (int r = 0; r < C::R; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                s[r][q] = 0;
        // sums of the earlier runs of tiles: [R * 8][kHT] float pairs
        float2 *acc = scratch + (size_t)blockIdx.x * (64 * kHT) + p;
        int run = 0;
        bool flushed = false;
        __syncthreads();
        for (int k = 0; k < n_my; ++k) {
            const int64_t left = n - tile_of(k) * kHT;
            const int rows = left < kHT ? (int)left : kHT;
            if (p_thread) {
                const float4 *J4 = reinterpret_cast<const float4 *>(J) + (size_t)(k & 1) * kHT * C::LD;
                const float4 *ja = J4 + half * C::SB + bx, *jb = J4 + by;
#pragma unroll 2
                for (int e = grp; e < rows; e += C::EG) {
                    float a[C::R];
                    f2 b[4];
#pragma unroll
                    for (int h = 0; h < C::R / 4; ++h) {
                        const float4 v = ja[e * C::LD + h * C::SB];
                        a[4 * h] = v.x, a[4 * h + 1] = v.y, a[4 * h + 2] = v.z, a[4 * h + 3] = v.w;
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float4 v = jb[e * C::LD + h * C::SB];
                        b[2 * h] = pk2(v.x, v.y), b[2 * h + 1] = pk2(v.z, v.w);
                    }
#pragma unroll
                    for (int r = 0; r < C::R; ++r)
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            s[r][q] = fma2(dup2(a[r]), b[q], s[r][q]);
                }
                if (++run == kFlush && k + 1 < n_my) {
                    run = 0;
#pragma unroll
                    for (int r = 0; r < C::R; ++r)
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            float2 *x = acc + (size_t)(8 * r + q) * kHT;
                            float2 v = flushed ? *x : make_float2(0.f, 0.f);
                            sum2(v.x, v.y, half_of(s[r][q >> 1], q & 1));
                            *x = v;
                        }
#pragma unroll
                    for (int r = 0; r < C::R; ++r)
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            s[r][q] = 0;
                    flushed = true;
                }
            }
            __syncthreads();
        }
        // the groups' sums: [EG][64][NS] float pairs (the tiles are free now)
        if (p_thread) {
            float2 *sums = reinterpret_cast<float2 *>(J) + (size_t)grp * 64 * C::NS + sup;
#pragma unroll
            for (int r = 0; r < C::R; ++r)
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    float2 v = flushed ? acc[(size_t)(8 * r + q) * kHT] : make_float2(0.f, 0.f);
                    sum2(v.x, v.y, half_of(s[r][q >> 1], q & 1));
                    sums[(size_t)((half * C::R + r) * 8 + q) * C::NS] = v;
                }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_bad)
        atomicOr(status, FLAG_DOMAIN);
    const float2 *sums = reinterpret_cast<const float2 *>(J);
    float2 *out = partials + (size_t)blockIdx.x * C::NS * 64;
    for (int q = threadIdx.x; q < C::NS * 64; q += C::WARPS * 32) {
        float h = 0.f, l = 0.f;
        for (int g = 0; g < C::EG; ++g) {
            const float2 v = sums[(size_t)g * 64 * C::NS + q];
            sum2(h, l, v.x);
            l += v.y;
        }
        if (is_wide(h)) {  // in FP64 at the block's scratch, which is free now
            reinterpret_cast<double *>(scratch)[(size_t)blockIdx.x * (64 * kHT) + q] =
                wide_sum(sums + q, C::EG, 64 * C::NS);
            h = INFINITY;
            l = 0.f;
        }
        out[q] = make_float2(h, l);
    }
}

// H[r][c] over the real parameters (Re V at 0..N-1, Im V at N..2N-1) from the
// blocks' sums [grid][64][NS] (infinite: a double in the block's scratch): 32 entries
// per block, one per lane, its 8 warps taking every eighth of the grid, then added in
// order, so that the order is the same on every run; zero when a data intensity was
// not positive. With async_or set, the status bits of the call are also OR-ed into
// *async_or.
__global__ void __launch_bounds__(256)
    hess_finalize(const float2 *partials, const float2 *scratch, int grid, int NP, int N,
                  const int *status, double *H, int *async_or)
{
    __shared__ float2 part[8][32];
    __shared__ double part_wide[8][32];
    const int flags = *status;
    if (async_or && blockIdx.x == 0 && threadIdx.x == 0 && flags)
        atomicOr(async_or, flags);
    const int SB = NP / 4, NS = SB * (SB + 1) / 2, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int o = blockIdx.x * 32 + lane;
    float h = 0.f, l = 0.f;
    if (o < NS * 64) {
#pragma unroll 4
        for (int b = warp; b < grid; b += 8) {
            const float2 v = partials[(size_t)b * NS * 64 + o];
            sum2(h, l, v.x);
            l += v.y;
        }
        if (!(fabsf(h) < INFINITY)) {  // a block's sum in FP64 was among them
            double d = 0.0;
#pragma unroll 1
            for (int b = warp; b < grid; b += 8) {
                const float2 v = partials[(size_t)b * NS * 64 + o];
                d += isinf(v.x) ? reinterpret_cast<const double *>(scratch)[(size_t)b * (64 * kHT) + o]
                                  : (double)v.x + (double)v.y;
            }
            part_wide[warp][lane] = d;
            h = INFINITY;
            l = 0.f;
        }
    }
    part[warp][lane] = make_float2(h, l);
    __syncthreads();
    if (warp || o >= NS * 64)
        return;
    for (int w = 1; w < 8; ++w) {
        sum2(h, l, part[w][lane].x);
        l += part[w][lane].y;
    }
    double total = (double)h + (double)l;
    if (!(fabsf(h) < INFINITY)) {
        total = 0.0;
#pragma unroll 1
        for (int w = 0; w < 8; ++w) {
            const float2 v = part[w][lane];
            total += isinf(v.x) ? part_wide[w][lane] : (double)v.x + (double)v.y;
        }
    }
    int y = o % NS, x = 0;
    const int q = o / NS;
    while (y >= SB - x) {
        y -= SB - x;
        ++x;
    }
    const int pr = 8 * x + (q >> 3), pc = 8 * (x + y) + (q & 7);
    const int r = pr < NP ? pr : pr - NP, c = pc < NP ? pc : pc - NP;
    if (r >= N || c >= N || pr > pc)
        return;
    const int hr = pr < NP ? r : N + r, hc = pc < NP ? c : N + c, P = 2 * N;
    const double v = (flags & FLAG_DOMAIN) ? 0.0 : total;
    H[hr * P + hc] = v;
    H[hc * P + hr] = v;
}

// Blocks per SM the weights kernel is compiled for (the register cap that
// gave no spills per size).
constexpr int weights_min_blocks(int np) { return np == 16 ? 2 : np <= 24 ? 3 : 1; }

// One event per thread and iteration; its 2N loads are issued together (an L1
// prefetch of the next iteration's lines, as in the likelihood kernels, made
// this kernel slower: 190 -> 242 us at 5M events, three CTAs per SM).
template <int NP>
__global__ void __launch_bounds__(256, weights_min_blocks(NP))
    mc_weights_kernel(const float *__restrict__ pl, int64_t pitch, int64_t n, int N,
                      const double *V, float inv_ngen, float *__restrict__ w)
{
    __shared__ float vf[2 * NP];
    load_v(V, N, 2 * NP, vf);
    __syncthreads();
#pragma unroll 1
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        float ar[NP], ai[NP], sr, si;
        load_event<NP>(pl, pitch, i, N, ar, ai);
        dot4<NP>(ar, ai, vf, sr, si);
        w[i] = fmaf(sr, sr, si * si) * inv_ngen;
    }
}

// F[a][b] = Re(conj(V_a) M_ab V_b) / V^H M V; the denominator is the sum of
// the numerators (M is Hermitian), summed in a fixed order.
__global__ void fit_fractions_kernel(const double *M, const double *V, int N, double *F)
{
    __shared__ double part[256];
    double mine = 0.0;
    for (int o = threadIdx.x; o < N * N; o += blockDim.x) {
        const int a = o / N, b = o % N;
        const double mr = M[2 * o], mi = M[2 * o + 1];
        const double pr = mr * V[2 * b] - mi * V[2 * b + 1], pi = mr * V[2 * b + 1] + mi * V[2 * b];
        const double num = V[2 * a] * pr + V[2 * a + 1] * pi;
        F[o] = num;
        mine += num;
    }
    part[threadIdx.x] = mine;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h)
            part[threadIdx.x] += part[threadIdx.x + h];
        __syncthreads();
    }
    const double nv = part[0];
    for (int o = threadIdx.x; o < N * N; o += blockDim.x)
        F[o] /= nv;
}

template <int NP>
cudaError_t hess_np(const Planes &d, const double *V, double *part, int grid, int *status,
                    double *H, int *async_or, cudaStream_t s)
{
    using C = HessCfg<NP>;
    cudaError_t e = cudaFuncSetAttribute(hess_kernel<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)C::SMEM);
    if (e != cudaSuccess)
        return e;
    const int64_t n_tiles = (d.n + kHT - 1) / kHT;
    if (grid > n_tiles)
        grid = (int)n_tiles;
    float2 *sums = reinterpret_cast<float2 *>(part);
    hess_kernel<NP><<<grid, C::WARPS * 32, C::SMEM, s>>>(d.ptr, d.pitch, d.n, d.n_waves, V, sums,
                                                   sums + (size_t)grid * C::NS * 64, status);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    hess_finalize<<<C::NS * 2, 256, 0, s>>>(sums, sums + (size_t)grid * C::NS * 64, grid, NP, d.n_waves,
                                            status, H, async_or);
    return cudaGetLastError();
}

template <int NP>
cudaError_t weights_np(const Planes &mc, const double *V, float inv_ngen, float *w, int grid,
                       cudaStream_t s)
{
    mc_weights_kernel<NP><<<grid, 256, 0, s>>>(mc.ptr, mc.pitch, mc.n, mc.n_waves, V, inv_ngen, w);
    return cudaGetLastError();
}

int pad_np(int n)
{
    for (int p : {4, 8, 12, 16, 20, 24, 32, 40, 48})
        if (n <= p)
            return p;
    return -1;
}

}  // namespace

size_t hess_partials_doubles(int n_waves, int grid)
{
    const int np = pad_np(n_waves);
    return (size_t)grid * 64 * (hess_super(np) + kHT);  // float pairs: the sums, the scratch
}

cudaError_t launch_hessian(const Planes &d, const double *V, double *partials, int grid, int *status,
                           double *H, int *async_or, cudaStream_t s)
{
    switch (pad_np(d.n_waves)) {
    case 4: return hess_np<4>(d, V, partials, grid, status, H, async_or, s);
    case 8: return hess_np<8>(d, V, partials, grid, status, H, async_or, s);
    case 12: return hess_np<12>(d, V, partials, grid, status, H, async_or, s);
    case 16: return hess_np<16>(d, V, partials, grid, status, H, async_or, s);
    case 20: return hess_np<20>(d, V, partials, grid, status, H, async_or, s);
    case 24: return hess_np<24>(d, V, partials, grid, status, H, async_or, s);
    case 32: return hess_np<32>(d, V, partials, grid, status, H, async_or, s);
    case 40: return hess_np<40>(d, V, partials, grid, status, H, async_or, s);
    case 48: return hess_np<48>(d, V, partials, grid, status, H, async_or, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_mc_weights(const Planes &mc, const double *V, double n_gen, float *w, int grid,
                              cudaStream_t s)
{
    const float ig = (float)(1.0 / n_gen);
    switch (pad_np(mc.n_waves)) {
    case 4: return weights_np<4>(mc, V, ig, w, grid, s);
    case 8: return weights_np<8>(mc, V, ig, w, grid, s);
    case 12: return weights_np<12>(mc, V, ig, w, grid, s);
    case 16: return weights_np<16>(mc, V, ig, w, grid, s);
    case 20: return weights_np<20>(mc, V, ig, w, grid, s);
    case 24: return weights_np<24>(mc, V, ig, w, grid, s);
    case 32: return weights_np<32>(mc, V, ig, w, grid, s);
    case 40: return weights_np<40>(mc, V, ig, w, grid, s);
    case 48: return weights_np<48>(mc, V, ig, w, grid, s);
    }
    return cudaErrorInvalidValue;
}

namespace {
__global__ void or_flags_kernel(const int *src, int *dst)
{
    if (*src)
        atomicOr(dst, *src);
}
}  // namespace

cudaError_t launch_or_flags(const int *src, int *dst, cudaStream_t s)
{
    or_flags_kernel<<<1, 1, 0, s>>>(src, dst);
    return cudaGetLastError();
}

namespace {
template <int N>
cudaError_t weights_tma_n(const CUtensorMap *map, const EvalArgs &a, int grid, cudaStream_t s)
{
    using C = AmpCfg<N, 2>;
    cudaError_t e = cudaFuncSetAttribute(nll_amp_kernel<N, 2, true>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (e != cudaSuccess)
        return e;
    const int n_tiles = (int)((a.n_events + C::TE - 1) / C::TE);
    nll_amp_kernel<N, 2, true><<<grid, C::THREADS, C::SMEM, s>>>(*map, a, n_tiles, nullptr);
    return cudaGetLastError();
}
}  // namespace

// Projection weights through the TMA-fed direct-form kernel (its weights
// mode): map over the MC planes as for the data (the same box: 256 events,
// 192 from 40 waves on, x 2n rows), amax over the MC sample; S by the exact
// product split.
cudaError_t launch_mc_weights_tma(const CUtensorMap *map, const Planes &mc, const double *V,
                                  const float *amax, double n_gen, float *w, int *status, int grid,
                                  cudaStream_t s)
{
    EvalArgs a{};
    a.n_waves = mc.n_waves;
    a.n_events = mc.n;
    a.V = V;
    a.amax = amax;
    a.status = status;
    a.weights = w;
    a.inv_ngen = (float)(1.0 / n_gen);
    switch (pad_np(mc.n_waves)) {
    case 4: return weights_tma_n<4>(map, a, grid, s);
    case 8: return weights_tma_n<8>(map, a, grid, s);
    case 12: return weights_tma_n<12>(map, a, grid, s);
    case 16: return weights_tma_n<16>(map, a, grid, s);
    case 20: return weights_tma_n<20>(map, a, grid, s);
    case 24: return weights_tma_n<24>(map, a, grid, s);
    case 32: return weights_tma_n<32>(map, a, grid, s);
    case 40: return weights_tma_n<40>(map, a, grid, s);
    case 48: return weights_tma_n<48>(map, a, grid, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_fit_fractions(const double *M, const double *V, int N, double *F, cudaStream_t s)
{
    fit_fractions_kernel<<<1, 256, 0, s>>>(M, V, N, F);
    return cudaGetLastError();
}

}  // namespace pwa
