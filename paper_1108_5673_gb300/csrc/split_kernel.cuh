// The direct form's evaluation (amp_kernel.cuh: the same sums in the same
// order) for incoherent sums of L components, I = sum_l |S^l|^2, gradient
// - sum_i sum_l conj(A^l) S^l / I, with S and the gradient in warps of their own.
//
// A CTA's events come in units of 64, two adjacent ones per lane packed in
// FP32x2 registers; each unit is one TMA copy of 2 L n rows into a ring slot.
// Twelve S warps take the units' components in turn and hand S^l to the unit's
// gradient warps (even and odd waves; one for few waves) through shared memory.
// A gradient warp keeps the sums of its two events per lane over all its units,
// tiles of three units going to two groups in turn.
//
// Bound by HBM and the time a unit holds its slot: copies of these boxes alone
// stream 1M events x 20 waves x 2 components (320 MB) in 53 us, 49 with boxes of
// 192 events. Eight warps that did S and then the gradient of 192-event tiles (a
// 61 KB slot, three of them) took 74 us, at 35% of the issue slots; with whole
// units as the S warps' items the 80-row units still held the nine slots too long
// (76 us whatever the number of warps). One call, us, before and now (with the
// results written to pinned memory instead of a stream synchronisation, which is
// 4 to 10 of it): 1M events, 20 waves x 2 components 90 to 72, 24 x 2 138 to 91,
// 12 x 4 117 to 84, 16 x 3 125 to 86, 8 x 2 53 to 41, 4 x 2 43 to 36. Nine S warps
// 77 at 20 x 2, fifteen 76; three producer warps no faster.
#pragma once

#include <numeric>

#include "amp_kernel.cuh"

namespace pwa {

namespace {

template <int N, int L>
struct SplitCfg {
    static constexpr int G = 2, GW = 3;                // groups, units per tile
    static constexpr int UNITS = G * GW;               // units with sums of their own
    // gradient warps per unit, waves of one (at 8 waves and below a second warp is
    // not worth its waits: 41 against 42 us at 1M events x 8 waves x 2 components)
    static constexpr int GH = N <= 8 ? 1 : 2, NH = N / GH;
    static constexpr int SWARPS = 12;
    static constexpr int UE = 64;                      // events per unit
    static constexpr int ROWS = 2 * N * L;
    static constexpr uint32_t SLOT_BYTES = ROWS * UE * 4;
    static constexpr uint32_t RS_BYTES = L * 32 * 16;  // r^l of a slot's events, 16 bytes per lane
    // ring slots: as many as fit 200 KB, of those with few barriers below
    static constexpr int pick_slots()
    {
        for (int n : {18, 12, 9, 6, 4})
            if (n * (SLOT_BYTES + RS_BYTES) <= 200 * 1024)
                return n;
        return 3;
    }
    static constexpr int SLOTS = pick_slots();
    // Barriers: unit q has slot q % SLOTS and barriers q % BARS. BARS is a multiple of
    // every number of warps that take the units in turn, so that the successive uses
    // of a barrier are waited for by the same warps: a parity wait then never sees a
    // phase more than one away, however far one warp falls behind another.
    static constexpr int BARS = std::lcm(SLOTS, std::lcm(SWARPS, UNITS));
    static constexpr int WARPS = 1 + SWARPS + GH * UNITS + 1;  // producer, S, gradient, helper
    static constexpr int THREADS = WARPS * 32;
    static constexpr int NF = 2 * N + 1;
    static constexpr size_t RING_BYTES = (size_t)SLOTS * SLOT_BYTES;
    static constexpr size_t SMEM =
        RING_BYTES + (size_t)SLOTS * RS_BYTES + 3 * BARS * sizeof(uint64_t);
    static_assert(SMEM <= 210 * 1024, "the ring does not fit");
    static_assert((size_t)(2 * N + 3) * 8 + 8 * (2 * N + 1) <= RING_BYTES, "the last CTA's sums");
};

template <int N, int L>
__global__ void __launch_bounds__(SplitCfg<N, L>::THREADS, 1)
    nll_split_kernel(const __grid_constant__ CUtensorMap map, const EvalArgs a, const int n_tiles,
                     int *work_flags)
{
    using C = SplitCfg<N, L>;
    constexpr int UE = C::UE, GW = C::GW, GH = C::GH, NH = C::NH, NF = C::NF, BARS = C::BARS;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *ring = reinterpret_cast<float *>(smem_raw);
    float4 *rs = reinterpret_cast<float4 *>(smem_raw + C::RING_BYTES);  // [SLOTS][L][32]
    uint64_t *full = reinterpret_cast<uint64_t *>(rs + (size_t)C::SLOTS * L * 32);
    uint64_t *rfull = full + BARS, *empty = rfull + BARS;

    __shared__ WaveCoef Vc[N];
    __shared__ double sV[2 * N];   // the helper warp's copy of V
    __shared__ float s_sigma, s_unit;
    __shared__ long long red_i[C::UNITS][2];
    __shared__ float red_f[C::UNITS][NF];
    __shared__ int s_flags, s_last;
    AmpScratch sc = amp_scratch(a.partials, gridDim.x);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // tiles of this CTA: blockIdx.x, blockIdx.x + gridDim.x, ...; unit q is the
    // (q % GW)-th of its tile q / GW (those past the last event are left out)
    const int n_my =
        (n_tiles > (int)blockIdx.x) ? (n_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    auto event0 = [&](int q) {
        return ((int64_t)blockIdx.x + (int64_t)(q / GW) * gridDim.x) * (GW * UE) + (q % GW) * UE;
    };
    int n_units = n_my * GW;
    while (n_units > 0 && event0(n_units - 1) >= a.n_events)
        --n_units;
    const uint32_t slot_tx = 2u * (uint32_t)a.n_waves * L * UE * 4u;
    auto parity = [](int q) { return (uint32_t)(q / BARS) & 1u; };
    auto issue = [&](int q) {
        mbar_arrive_expect_tx(&full[q % BARS], slot_tx);
        tma_load_2d(ring + (size_t)(q % C::SLOTS) * C::ROWS * UE, &map, (int)event0(q), 0,
                    &full[q % BARS]);
    };
    // units the producer issues (none when the timeout path is being tested)
    const int n_issue = a.stall_ns ? 0 : n_units;
    const unsigned long long wait_ns = a.stall_ns ? a.stall_ns : kWaitLimitNs;
    for (int b = threadIdx.x; b < BARS; b += blockDim.x) {
        mbar_init(&full[b], 1);
        mbar_init(&rfull[b], L);
        mbar_init(&empty[b], L + GH);
    }
    fence_barrier_init();
    if (threadIdx.x == 0)
        s_flags = 0;
    __syncthreads();
    // start streaming before the prologue below (its global loads take ~1 us)
    const int n_first = n_issue < C::SLOTS ? n_issue : C::SLOTS;
    if (threadIdx.x == 0)
        for (int q = 0; q < n_first; ++q)
            issue(q);
    // Rows of padded waves (n_waves < N) are never written by TMA: zero them
    // once so that they contribute nothing (their V is zero as well).
    for (int s = 0; s < C::SLOTS; ++s)
        for (int i = 2 * a.n_waves * L * UE + threadIdx.x; i < C::ROWS * UE; i += blockDim.x)
            ring[(size_t)s * C::ROWS * UE + i] = 0.f;
    if (threadIdx.x < N)
        wave_coef(a.V, a.n_waves, threadIdx.x, Vc[threadIdx.x]);
    if (warp == C::WARPS - 1)
        exact_scale(a.V, a.amax, a.n_waves, lane, &s_sigma, &s_unit);
    __syncthreads();

    int flags = 0;
    // component l of wave w sits at rows 2 (l n + w), 2 (l n + w) + 1 (padded
    // waves w >= n carry V = 0: their products are exactly 0)
    const int comp_rows = 2 * a.n_waves * UE;
    if (warp == 0) {
        if (lane == 0) {
            // ---- producer --------------------------------------------------------
            int q = n_first;
            for (; q < n_issue; ++q) {
                const int before = q - C::SLOTS;  // the slot's last unit
                if (!mbar_wait(&empty[before % BARS], parity(before))) {
                    flags |= FLAG_TIMEOUT;
                    break;
                }
                issue(q);
            }
            // no copy may still be landing in shared memory when the CTA exits
            // (the last SLOTS units issued are the latest use of every slot)
            for (int k = (q > C::SLOTS ? q - C::SLOTS : 0); k < q; ++k)
                if (!mbar_wait(&full[k % BARS], parity(k)))
                    flags |= FLAG_TIMEOUT;
        }
    } else if (warp <= C::SWARPS) {
        // ---- S^l: item k is component k % L of unit k / L ---------------------
        const int sw = warp - 1;
        const float sigma = s_sigma, unit = s_unit;
        const f2 SG = pk2(sigma, sigma);
        // bits(t) - bits(sigma) summed over the 2N terms of Im S: remove the offset once
        const unsigned im_offset = 2u * (unsigned)N * __float_as_uint(sigma);
        for (int k = sw; k < n_units * L; k += C::SWARPS) {
            const int q = k / L, l = k % L, s = q % C::SLOTS;
            if (!mbar_wait(&full[q % BARS], parity(q), wait_ns)) {
                flags |= FLAG_TIMEOUT;
                break;
            }
            const float *T = ring + (size_t)s * C::ROWS * UE + 2 * lane + l * comp_rows;
            float sr[2], si[2];
            exact_sum2<N>(
                [&](int w, f2 &ar, f2 &ai) {
                    ar = lds2(T + (2 * w) * UE);
                    ai = lds2(T + (2 * w + 1) * UE);
                },
                Vc, SG, unit, im_offset, sr, si);
            rs[(s * L + l) * 32 + lane] = make_float4(sr[0], sr[1], si[0], si[1]);
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&rfull[q % BARS]);
                mbar_arrive(&empty[q % BARS]);
            }
        }
    } else if (warp < C::WARPS - 1) {
        // ---- ln I (gh = 0) and the gradient of waves gh, gh + GH, ... of the units
        // u, u + UNITS, ... --
        const int gi = warp - 1 - C::SWARPS, u = gi / GH, gh = gi % GH;
        float gs[2 * NH];
#pragma unroll
        for (int c = 0; c < 2 * NH; ++c)
            gs[c] = 0.f;
        long long l_int = 0;      // sum of round(2^23 ln f)
        int eacc = 0;             // sum of exponents
        float l_frac = 0.f;       // sum of the remainders (units of 2^-23)
        int bad = 0;
        for (int q = u; q < n_units; q += C::UNITS) {
            const int s = q % C::SLOTS;
            if (!mbar_wait(&full[q % BARS], parity(q), wait_ns) ||
                !mbar_wait(&rfull[q % BARS], parity(q), wait_ns)) {
                flags |= FLAG_TIMEOUT;
                break;
            }
            const float *T = ring + (size_t)s * C::ROWS * UE + 2 * lane + 2 * gh * UE;
            const int64_t ev0 = event0(q) + 2 * lane;
            float4 r[L];
#pragma unroll
            for (int l = 0; l < L; ++l)
                r[l] = rs[(s * L + l) * 32 + lane];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float I = 0.f;
#pragma unroll
                for (int l = 0; l < L; ++l) {
                    const float sr = e ? r[l].y : r[l].x, si = e ? r[l].w : r[l].z;
                    const float Il = fmaf(sr, sr, si * si);
                    I = l ? I + Il : Il;
                }
                const bool in = (ev0 + e) < a.n_events;
                const bool ok = in && (I > 0.f) && (I < INFINITY);
                const float rI = __frcp_rn(I);
#pragma unroll
                for (int l = 0; l < L; ++l) {
                    float &sr = e ? r[l].y : r[l].x, &si = e ? r[l].w : r[l].z;
                    sr = ok ? sr * rI : 0.f;
                    si = ok ? si * rI : 0.f;
                }
                if (gh == 0) {
                    if (ok) {
                        int ex;
                        const float f = split_exponent(I, ex);
                        // 2^23 ln f = k + r exactly: k integer (|k| < 2^22), |r| <= 1/2
                        const float y = logf(f) * 8388608.0f;
                        const float t = y + 12582912.0f;  // 1.5 * 2^23: rounds y to an integer
                        l_int += __float_as_int(t) - 0x4B400000;
                        l_frac += y - (t - 12582912.0f);
                        eacc += ex;
                    } else if (in) {
                        bad = 1;
                    }
                }
            }
#pragma unroll
            for (int l = 0; l < L; ++l) {
                const float *Tl = T + l * comp_rows;
#pragma unroll
                for (int i = 0; i < NH; ++i) {
                    float a0, a1, b0, b1;
                    upk2(lds2(Tl + (2 * GH * i) * UE), a0, a1);
                    upk2(lds2(Tl + (2 * GH * i + 1) * UE), b0, b1);
                    // conj(A) r = (ar rr + ai ri) + i (ar ri - ai rr)
                    gs[2 * i] = fmaf(a0, r[l].x, fmaf(b0, r[l].z, gs[2 * i]));
                    gs[2 * i] = fmaf(a1, r[l].y, fmaf(b1, r[l].w, gs[2 * i]));
                    gs[2 * i + 1] = fmaf(a0, r[l].z, fmaf(-b0, r[l].x, gs[2 * i + 1]));
                    gs[2 * i + 1] = fmaf(a1, r[l].w, fmaf(-b1, r[l].y, gs[2 * i + 1]));
                }
            }
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&empty[q % BARS]);
        }
        if (bad)
            flags |= FLAG_DOMAIN;
        // sums over the warp (fixed order)
        if (gh == 0) {
            const long long li = warp_sum(l_int);
            const long long ei = warp_sum((long long)eacc);
            const float lf = warp_sum(l_frac);
            if (lane == 0) {
                red_i[u][0] = li;
                red_i[u][1] = ei;
                red_f[u][0] = lf;
            }
        }
        warp_transpose_sum<2 * NH>(gs, lane);
#pragma unroll
        for (int b = 0; b < (2 * NH + 31) / 32; ++b) {
            const int c = 32 * b + lane;
            if (c < 2 * NH)
                red_f[u][1 + 2 * (GH * (c / 2) + gh) + (c & 1)] = gs[32 * b];
        }
    } else if (blockIdx.x == 0) {
        // ---- helper warp of CTA 0: M V and V^H M V in FP64, one row per lane ----
        const int Nw = a.n_waves;
        for (int i = lane; i < 2 * Nw; i += 32)
            sV[i] = a.V[i];
        __syncwarp();
        double nv = 0.0;
        for (int row = lane; row < Nw; row += 32) {
            double re = 0.0, im = 0.0;
            for (int b = 0; b < Nw; ++b) {
                const double mr = a.M[2 * (row * Nw + b)], mi = a.M[2 * (row * Nw + b) + 1];
                const double vr = sV[2 * b], vi = sV[2 * b + 1];
                re = fma(mr, vr, fma(-mi, vi, re));
                im = fma(mr, vi, fma(mi, vr, im));
            }
            sc.mv[2 * row] = re;
            sc.mv[2 * row + 1] = im;
            nv = fma(sV[2 * row], re, fma(sV[2 * row + 1], im, nv));  // Re(conj(V) (M V))
        }
        nv = warp_sum(nv);
        if (lane == 0)
            sc.mv[2 * kMaxWaves] = nv;
    }
    if (flags)
        atomicOr(&s_flags, flags);
    __syncthreads();

    // ---- block partial, fixed order over warps -------------------------
    if (threadIdx.x < 2) {
        long long v = 0;
        for (int w = 0; w < C::UNITS; ++w)
            v += red_i[w][threadIdx.x];
        sc.pi[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = v;
    }
    for (int c = threadIdx.x; c < NF; c += blockDim.x) {
        dfloat v = {0.f, 0.f};
        for (int w = 0; w < C::UNITS; ++w)
            v = df_add(v, dfloat{red_f[w][c], 0.f});
        sc.pf[(size_t)c * gridDim.x + blockIdx.x] = make_float2(v.hi, v.lo);
    }
    float *tiles = ring;
#include "direct_finish.cuh"
}

}  // namespace

}  // namespace pwa
