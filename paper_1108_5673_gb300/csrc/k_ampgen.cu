// Amplitudes on the device (Sec. 4: the framework computes its amplitudes on
// the GPU), for the amplitude model of the samples here:
//   A_a(Omega) = BW(m; M_a, G_a) Y_{l_a}^{m_a}(theta, phi),
//   BW(m; M, G) = 1 / (M^2 - m^2 - i M G) = (D + i M G) / (D^2 + (M G)^2), D = M^2 - m^2,
//   Y_l^m = N_lm P_l^m(cos theta) e^{i m phi} for m >= 0 (Condon-Shortley phase
//   in P_l^m), Y_l^{-m} = (-1)^m conj(Y_l^m).
// Each component is the float nearest to the model's value in FP64.
//
// FP64 arithmetic throughout held the FP64 pipe (1/64 of the FP32 rate) at 87%
// and took 6.35 ms for 5M events x 20 waves. Here the values are formed in
// float-float (ff.cuh, ~44 bits, two events per thread in packed FP32) with a
// bound on their error, and rounded where the bound leaves no doubt which
// float is nearest (Ziv's test). An amplitude in doubt (one in 1240 at 20
// waves with l up to 4, in 240 at 40 with l up to 10), and an event whose inputs or
// products leave the float-float range, go to a queue per
// warp and are evaluated in FP64 a warp's worth at a time: one by one, by the
// lane concerned, they took as long as the rest (1.35 ms in all). Measured at
// 5M x 20: 0.69 ms (1.3 TB/s of the 0.92 GB), at 2M x 40 with l up to 10: 0.86
// ms against 7.6, at 5M x 4: 0.22 ms against 1.48; bound by instruction issue
// (60% of the slots, most of the rest packed FP32 instructions that take two).
//
// The waves are visited in order of (|m|, l), so that
// e^{i m phi}, P_m^m and the upward recurrence in l continue from wave to wave
// (each P_l^m is formed once however many waves share it); the order, the
// recurrence's coefficients and the waves' constants form a table that the
// host builds once per call, passes as a kernel argument (10 KB) and each block
// keeps in shared memory. e^{i phi}:
// phi reduced by multiples of pi/2 in FP64, then the Taylor series of sine
// and cosine on [-pi/4, pi/4], the terms above 2^-19 in float-float. Event-
// major output goes through shared memory, a warp's 64 events at a time,
// so that global stores are whole rows; planes are written directly.
#include <algorithm>
#include <cmath>
#include <vector>

#include "ff.cuh"

namespace pwa {

namespace {

constexpr int kGenThreads = 128;
constexpr int kMaxL = 16;

// 1 / k for the recurrence's divisor l - m (k = 1 .. kMaxL), rounded to double
__constant__ double c_inv[kMaxL + 1] = {
    0.0, 1.0, 1.0 / 2, 1.0 / 3, 1.0 / 4, 1.0 / 5, 1.0 / 6, 1.0 / 7, 1.0 / 8, 1.0 / 9, 1.0 / 10,
    1.0 / 11, 1.0 / 12, 1.0 / 13, 1.0 / 14, 1.0 / 15, 1.0 / 16};

// One amplitude in FP64 (the components and events the float-float path
// leaves).
__device__ __noinline__ float2 amplitude_fp64(double m, double x, double phi, const GenWave *w)
{
    const int l = w->l, mm = w->m, am = mm < 0 ? -mm : mm;
    const double s = sqrt(fmax(0.0, 1.0 - x * x));
    double c1, s1, er = 1.0, ei = 0.0;
    sincos(phi, &s1, &c1);
    // P_l^am(x), Condon-Shortley phase, and e^{i am phi}
    double pmm = 1.0;
    for (int k = 1; k <= am; ++k) {
        pmm *= -(2.0 * k - 1.0) * s;
        const double t = er * c1 - ei * s1;
        ei = er * s1 + ei * c1;
        er = t;
    }
    double p = pmm;
    if (l > am) {
        double p2 = pmm, p1 = x * (2.0 * am + 1.0) * pmm;
        for (int ll = am + 2; ll <= l; ++ll) {
            const double q = ((2.0 * ll - 1.0) * x * p1 - (ll + am - 1.0) * p2) * c_inv[ll - am];
            p2 = p1;
            p1 = q;
        }
        p = p1;
    }
    const double y = w->norm * p;
    double yr = y * er, yi = y * ei;
    if (mm < 0) {
        const double sign = (am & 1) ? -1.0 : 1.0;
        yr *= sign;
        yi *= -sign;
    }
    const double D = w->mass * w->mass - m * m, G = w->mass * w->width;
    const double rden = 1.0 / (D * D + G * G);
    const double br = D * rden, bi = G * rden;
    return make_float2(__double2float_rn(br * yr - bi * yi), __double2float_rn(br * yi + bi * yr));
}

// phi = r + k pi/2 with |r| <= pi/4, in FP64; ok cleared for |phi| > 2^20
__device__ __forceinline__ double reduce(double phi, int &k, bool &ok)
{
    // (compared as bits: FP64 comparisons are FP64 instructions)
    ok = ok && (unsigned)(__double2hiint(phi) & 0x7fffffff) < 0x41300000u;
    const double magic = 6755399441055744.0;  // 1.5 2^52: rounds to an integer
    const double t = fma(phi, 0.63661977236758134308, magic);  // 2 / pi
    k = __double2loint(t);
    const double kd = t - magic;
    // pi/2 as the nearest double and the remainder
    const double r = fma(-kd, 1.57079632679489661923, phi);
    return fma(-kd, 6.12323399573676588614e-17, r);
}

// e^{i phi} to 2^-43.5
__device__ __forceinline__ void expi(double phi0, double phi1, ff &c, ff &s, bool &ok0, bool &ok1)
{
    int k0, k1;
    const double r0 = reduce(phi0, k0, ok0), r1 = reduce(phi1, k1, ok1);
    const ff r = ff_split(r0, r1, ok0, ok1);
    const ff z = ff_norm(ff_sqr(r));  // r^2 <= 0.617
    // sin r = r - r^3/3! + r^5/5! - r^7/7! + (r^9/9! ...), the last in FP32
    f2 q = fma2(z.h, dup2(1.0f / 6227020800.0f), dup2(-1.0f / 39916800.0f));
    q = fma2(z.h, q, dup2(1.0f / 362880.0f));
    ff p = ff_add(ff_const(-1.0 / 5040), ff_mul(z, q));
    p = ff_add(ff_const(1.0 / 120), ff_mul(z, p));
    p = ff_add(ff_const(-1.0 / 6), ff_mul(z, p));
    const ff sr = ff_add(r, ff_mul(ff_norm(ff_mul(z, r)), p));
    // cos r = 1 - r^2/2! + r^4/4! - r^6/6! + r^8/8! - (r^10/10! ...)
    f2 g = fma2(z.h, dup2(1.0f / 87178291200.0f), dup2(-1.0f / 479001600.0f));
    g = fma2(z.h, g, dup2(1.0f / 3628800.0f));
    ff u = ff_sub(ff_const(1.0 / 40320), ff_mul(z, g));
    u = ff_add(ff_const(-1.0 / 720), ff_mul(z, u));
    u = ff_add(ff_const(1.0 / 24), ff_mul(z, u));
    u = ff_add(ff_const(-0.5), ff_mul(z, u));
    const ff cr = ff_add(ff_dup(1.0f, 0.0f), ff_mul(z, u));
    // swap and signs by the quadrant of each event
    auto turn = [&](f2 a, f2 b, int add) {
        float a0, a1, b0, b1;
        upk2(a, a0, a1);
        upk2(b, b0, b1);
        const float v0 = (k0 & 1) ? b0 : a0, v1 = (k1 & 1) ? b1 : a1;
        return pk2(__uint_as_float(__float_as_uint(v0) ^ ((unsigned)((k0 + add) & 2) << 30)),
                   __uint_as_float(__float_as_uint(v1) ^ ((unsigned)((k1 + add) & 2) << 30)));
    };
    c = {turn(cr.h, sr.h, 1), turn(cr.l, sr.l, 1)};
    s = {turn(sr.h, cr.h, 0), turn(sr.l, cr.l, 0)};
}

__device__ __forceinline__ ff load_pair(const GenPair &p)
{
    const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(&p);
    return {v.x, v.y};
}

template <bool SOA>
__global__ void __launch_bounds__(kGenThreads, 4)
    amp_gen_kernel(const double *__restrict__ kin, int64_t n, int N,
                   const __grid_constant__ GenTable table, bool fp64_only, float *__restrict__ out,
                   int64_t pitch)
{
    extern __shared__ float2 rows[];  // event-major: [warps][64][N | 1]
    __shared__ GenWave w[kMaxWaves];
    __shared__ GenStep steps[kGenMaxSteps];
    __shared__ uint2 queue[kGenThreads / 32][96];  // (event, wave) pairs left to FP64, per warp
    const int n_steps = table.n_steps;
    for (int i = threadIdx.x; i < (int)(N * sizeof(GenWave) / 4); i += blockDim.x)
        reinterpret_cast<int *>(w)[i] = reinterpret_cast<const int *>(table.w)[i];
    for (int i = threadIdx.x; i < (int)(n_steps * sizeof(GenStep) / 4); i += blockDim.x)
        reinterpret_cast<int *>(steps)[i] = reinterpret_cast<const int *>(table.steps)[i];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ld = N | 1;  // odd row length: conflict-free 8-byte columns
    float2 *my = rows + (size_t)warp * 64 * ld;
    uint2 *q = queue[warp];
    int queued = 0;  // the same in every lane
    // FP64 values of the last (up to 32) queued amplitudes, one per lane, over
    // the provisional ones in the output (event-major: in the rows still held
    // for the batch that starts at e0)
    auto drain = [&](int64_t e0) {
        const int take = queued < 32 ? queued : 32;
        queued -= take;
        if (lane < take) {
            const uint2 it = q[queued + lane];
            const int64_t i = it.x;
            const GenWave *W = &w[it.y];
            const float2 A = amplitude_fp64(kin[3 * i], kin[3 * i + 1], kin[3 * i + 2], W);
            if (SOA) {
                out[(int64_t)(2 * W->index) * pitch + i] = A.x;
                out[(int64_t)(2 * W->index + 1) * pitch + i] = A.y;
            } else if (i >= e0) {
                my[(int)(i - e0) * ld + W->index] = A;
            } else {
                reinterpret_cast<float2 *>(out)[i * N + W->index] = A;
            }
        }
        __syncwarp();
    };
    const bool pairs = !fp64_only && !table.fp64_only;
    const int64_t stride = (int64_t)gridDim.x * (2 * kGenThreads);
    for (int64_t e0 = ((int64_t)blockIdx.x * (kGenThreads / 32) + warp) * 64; e0 < n; e0 += stride) {
        // this lane's events; past the end the last one is repeated (nothing
        // of it is stored)
        const bool in0 = e0 + lane < n, in1 = e0 + 32 + lane < n;
        const int64_t i0 = in0 ? e0 + lane : n - 1, i1 = in1 ? e0 + 32 + lane : n - 1;
        bool ok0 = pairs, ok1 = pairs;
        const double x0 = kin[3 * i0 + 1], x1 = kin[3 * i1 + 1];
        const ff x = ff_split(x0, x1, ok0, ok1);
        const double ma = kin[3 * i0], mb = kin[3 * i1];
        const ff m2 = ff_split(ma * ma, mb * mb, ok0, ok1);
        // sin^2 theta; at and beyond the poles (and below 2^-40, where the
        // rounding of x matters) FP64
        const double w0 = fma(-x0, x0, 1.0), w1 = fma(-x1, x1, 1.0);
        ok0 = ok0 && __double2hiint(w0) >= 0x3d700000;  // w0 >= 2^-40
        ok1 = ok1 && __double2hiint(w1) >= 0x3d700000;
        const ff s = ff_sqrt(ff_split(w0, w1, ok0, ok1));
        ff c1, s1;
        expi(kin[3 * i0 + 2], kin[3 * i1 + 2], c1, s1, ok0, ok1);

        // e^{i m phi}, P_m^m, the recurrence's last two values with
        // bounds on their errors, and y = N_lm P_l^m with its bound
        ff er = ff_dup(1.f, 0.f), ei = ff_dup(0.f, 0.f), pmm = er, p1 = er,
           p2 = ei, y = ei;
        f2 e1 = 0ull, e2 = 0ull, y_err = 0ull;
        bool y0 = false, y1 = false;
        int step = 0, am = 0;
        for (int a = 0; a < N; ++a) {
            const GenWave &W = w[a];
            if (W.m_inc >= 0) {  // a new |m|
                for (int k = 0; k < W.m_inc; ++k) {
                    const ff t = ff_norm(ff_det(er, c1, ei, s1));
                    ei = ff_norm(ff_dot(er, s1, ei, c1));
                    er = t;
                    pmm = ff_norm(ff_mul(ff_mul(s, dup2(-(float)(2 * am + 1))), pmm));
                    ++am;
                }
                p1 = pmm;
                p2 = ff_dup(0.f, 0.f);
                e1 = mul2(dup2((float)am * 0x1p-43f), abs2(pmm.h));
                e2 = 0ull;
            }
            for (int k = 0; k < W.l_steps; ++k, ++step) {
                // P_l = a x P_{l-1} - b P_{l-2}
                const ff sa = load_pair(steps[step].a), sb = load_pair(steps[step].b);
                const ff xp = ff_norm(ff_mul(x, p1));
                const ff u = ff_mul(sa, xp), v = ff_mul(sb, p2);
                const ff sm = ff_two_diff(u.h, v.h);
                const f2 eps = dup2(0x1p-43f);
                const f2 ex = fma2(abs2(x.h), e1, mul2(eps, abs2(xp.h)));
                const f2 eq = fma2(sa.h, ex, fma2(sb.h, e2, mul2(eps, abs2(v.h))));
                p2 = p1;
                e2 = e1;
                p1 = ff_fast(sm.h, add2(sm.l, sub2(u.l, v.l)));
                e1 = eq;
            }
            if (W.new_y) {
                // (the sign (-1)^m of m < 0 is in N_lm); |y| >= 2^-60: no product
                // behind it has lost bits to underflow
                const ff nrm = load_pair(W.nrm);
                y = ff_norm(ff_mul(nrm, p1));
                const f2 ay = abs2(y.h);
                float a0, a1;
                upk2(ay, a0, a1);
                y0 = a0 >= 0x1p-60f && ok0;
                y1 = a1 >= 0x1p-60f && ok1;
                // the relative errors of the products (2^-42.2 in all) and of
                // e^{i m phi} (m 2^-42.7), and P's
                y_err = fma2(ay, dup2(fmaf((float)am, 0x1p-42f, 0x1p-42f)),
                             mul2(mul2(dup2(1.001f), abs2(nrm.h)), e1));
            }
            // A = y (D + i G) e^{i m phi} / (D^2 + G^2); for m < 0 the conjugate of
            // the same with G negated (in the table), conjugated at the end
            const ff M2 = load_pair(W.m2), G = load_pair(W.g), G2 = load_pair(W.g2);
            const ff D = ff_sub(M2, m2);
            const ff dd = ff_sqr(D);
            const ff den = ff_two_sum(dd.h, G2.h);
            const ff inv = ff_rcp(ff{den.h, add2(den.l, add2(dd.l, G2.l))});
            ff Er = D, Ei = G;
            if (am > 0) {
                Er = ff_det(D, er, G, ei);
                Ei = ff_dot(D, ei, G, er);
            }
            const ff f = ff_mul(y, inv);
            // below 2^-100 f's low part has lost bits, which the product with a large E shows
            // in the result (in keV, MeV^2 and the like: 1 / (D^2 + G^2) is tiny there)
            float f0, f1;
            upk2(abs2(f.h), f0, f1);
            const ff re = ff_mul(Er, f), im = ff_mul(Ei, f);
            // error bound: y's, and D's rounding (2^-46 of M^2 + m^2, times |BW|)
            const f2 b = mul2(add2(abs2(D.h), abs2(G.h)), inv.h);
            const f2 dm = mul2(dup2(0x1p-46f), add2(M2.h, m2.h));
            const f2 err = mul2(b, fma2(mul2(dm, b), abs2(y.h), y_err));
            float2 A0, A1;
            bool r0, r1, j0, j1;
            ff_round(re, err, A0.x, A1.x, r0, r1);
            ff_round(im, err, A0.y, A1.y, j0, j1);
            A0.y = __uint_as_float(__float_as_uint(A0.y) ^ W.conj);
            A1.y = __uint_as_float(__float_as_uint(A1.y) ^ W.conj);
            if (SOA) {
                float *o = out + (int64_t)(2 * W.index) * pitch + e0 + lane;
                if (in0) {
                    o[0] = A0.x;
                    o[pitch] = A0.y;
                }
                if (in1) {
                    o[32] = A1.x;
                    o[pitch + 32] = A1.y;
                }
            } else {
                my[lane * ld + W.index] = A0;
                my[(lane + 32) * ld + W.index] = A1;
            }
            // amplitudes in doubt wait for a warp's worth of them: FP64
            // instructions cost the same for one lane as for 32
            const bool d0 = !(r0 && j0 && y0 && f0 >= 0x1p-100f) && in0,
                       d1 = !(r1 && j1 && y1 && f1 >= 0x1p-100f) && in1;
            if (__any_sync(0xffffffffu, d0 || d1)) {
                const unsigned below = (1u << lane) - 1;
                unsigned doubt = __ballot_sync(0xffffffffu, d0);
                if (d0)
                    q[queued + __popc(doubt & below)] = make_uint2((unsigned)i0, (unsigned)a);
                queued += __popc(doubt);
                doubt = __ballot_sync(0xffffffffu, d1);
                if (d1)
                    q[queued + __popc(doubt & below)] = make_uint2((unsigned)i1, (unsigned)a);
                queued += __popc(doubt);
                __syncwarp();
                while (queued >= 32)
                    drain(e0);
            }
        }
        if (!SOA) {
            // the warp's rows, contiguous in the output
            __syncwarp();
            const int cnt = (int)(n - e0 < 64 ? n - e0 : 64) * N;
            float2 *dst = reinterpret_cast<float2 *>(out) + e0 * N;
            int r = lane / N, c = lane - r * N;
            const int dr = 32 / N, dc = 32 - dr * N;
            for (int k = lane; k < cnt; k += 32) {
                dst[k] = my[r * ld + c];
                r += dr;
                c += dc;
                if (c >= N) {
                    c -= N;
                    ++r;
                }
            }
            __syncwarp();
        }
    }
    while (queued > 0)
        drain(n);
}

}  // namespace

int ampgen_max_l() { return kMaxL; }

void ampgen_table(const pwa_wave *waves, int N, GenTable *t)
{
    std::vector<int> order(N);
    for (int a = 0; a < N; ++a)
        order[a] = a;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        const int ma = std::abs(waves[a].m), mb = std::abs(waves[b].m);
        if (ma != mb)
            return ma < mb;
        return waves[a].l != waves[b].l ? waves[a].l < waves[b].l : waves[a].m < waves[b].m;
    });
    int cur_m = 0, cur_l = 0;
    t->n_steps = 0;
    t->fp64_only = 0;
    for (int k = 0; k < N; ++k) {
        const pwa_wave &s = waves[order[k]];
        const int am = std::abs(s.m);
        GenWave &w = t->w[k];
        double ratio = 1.0;  // (l - |m|)! / (l + |m|)!
        for (int j = s.l - am + 1; j <= s.l + am; ++j)
            ratio /= j;
        w.mass = s.mass;
        w.width = s.width;
        w.norm = std::sqrt((2.0 * s.l + 1.0) / (4.0 * 3.14159265358979323846) * ratio);
        w.l = s.l;
        w.m = s.m;
        w.index = order[k];
        w.m_inc = k == 0 || am != cur_m ? am - (k == 0 ? 0 : cur_m) : -1;
        if (w.m_inc >= 0) {
            cur_m = am;
            cur_l = am;
        }
        w.l_steps = s.l - cur_l;
        for (; cur_l < s.l; ++cur_l) {
            const int l = cur_l + 1;
            t->steps[t->n_steps++] =
                GenStep{gen_pair((2.0 * l - 1.0) / (l - am)), gen_pair((l + am - 1.0) / (l - am))};
        }
        const double g = s.mass * s.width;
        // scales whose squares would leave the float range in D^2 + G^2
        if (!(g * g >= 0x1p-80 && g * g <= 0x1p80 && s.mass * s.mass <= 0x1p60))
            t->fp64_only = 1;
        w.m2 = gen_pair(s.mass * s.mass);
        w.g = gen_pair(s.m < 0 ? -g : g);
        w.g2 = gen_pair(g * g);
        w.nrm = gen_pair(s.m < 0 && (am & 1) ? -w.norm : w.norm);
        w.conj = s.m < 0 ? 0x80000000u : 0u;
        w.new_y = k == 0 || s.l != t->w[k - 1].l || s.m != t->w[k - 1].m;
    }
}

cudaError_t launch_amp_gen(const double *kin, int64_t n, int N, const GenTable &table, bool fp64_only,
                           float *out, bool soa, int64_t pitch, int num_sms, cudaStream_t s)
{
    if (n <= 0)
        return cudaSuccess;
    if (N < 1 || N > kMaxWaves)
        return cudaErrorInvalidValue;
    const int64_t need = (n + 2 * kGenThreads - 1) / (2 * kGenThreads);
    const unsigned grid = (unsigned)std::min<int64_t>(need, (int64_t)num_sms * 4);
    if (soa) {
        amp_gen_kernel<true><<<grid, kGenThreads, 0, s>>>(kin, n, N, table, fp64_only, out, pitch);
    } else {
        const auto rows = [](int waves) { return (size_t)2 * kGenThreads * (waves | 1) * sizeof(float2); };
        const size_t smem = rows(N);
        // the same limit at every call: contexts in other threads launch it too
        const cudaError_t e = cudaFuncSetAttribute(
            amp_gen_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rows(kMaxWaves));
        if (e != cudaSuccess)
            return e;
        amp_gen_kernel<false><<<grid, kGenThreads, smem, s>>>(kin, n, N, table, fp64_only, out, 0);
    }
    return cudaGetLastError();
}

}  // namespace pwa
