// Covariant tensor amplitudes on the device (Sec. 4: the framework builds its
// amplitudes on the GPU in the covariant tensor formalism), for the radiative
// decay J/psi -> gamma X, X -> K+ K-:
//   4-vectors in the J/psi rest frame, metric (+,-,-,-); per event the
//   photon q and the kaons k1, k2 (from their 3-momenta, mK = 0.493677 GeV),
//   p = k1 + k2, r = k1 - k2, rt = r - (r.p / p.p) p;
//   unobserved components l = 2 (M index) + (photon polarization index):
//   J/psi helicity M = +1, -1 along z, psi(+1) = (0, -1, -i, 0)/sqrt2,
//   psi(-1) = (0, 1, -i, 0)/sqrt2; photon e1 = (0, z x q / |z x q|) (x when q
//   lies along z), e2 = (0, q/|q| x e1);
//   spin 0: A = BW(p.p) psi.e;
//   spin 2: A = BW(p.p) B2(Q) [(psi.rt)(e.rt) - (1/3)(rt.rt)(psi.e - (psi.p)(e.p)/p.p)],
//     Q^2 = p.p/4 - mK^2, B2 = sqrt(13 / (Q^4 + 3 Q^2 Q0^2 + 9 Q0^4)), Q0 = 0.197327 GeV;
//   BW(s) = 1 / (M^2 - s - i M G).
// Each component is the float nearest to the formalism's value in FP64.
//
// FP64 arithmetic throughout held the FP64 pipe (1/64 of the FP32 rate) at 88%:
// 5.96 ms for 5M events x 12 waves. As in the generator of BW x Y_l^m, the
// values are formed in float-float, two events per thread, with a bound on
// their error, and rounded where it decides the nearest float; an event and
// wave in doubt goes to a queue per warp that FP64 serves 32 at a time.
// Measured, generation into the planes with the maxima, 1M + 2.5M events x 12
// waves: 0.77 ms (4.2 in FP64, event-major); an event and wave in doubt is one
// in a hundred (where p.p cancels and near a wave's pole), and FP64 still takes
// 39% of its pipe's time.
//
// Two identities of the formalism shorten the pair path (both hold exactly,
// the FP64 evaluation to its rounding): r.p = k1.k1 - k2.k2 = 0, so rt = r and
// rt.rt = 4 mK^2 - p.p; and psi(-1) has the real part of psi(+1) negated, so
// component M = -1 of a contraction (Re, Im) is (-Re, Im), and the four values
// of a wave and a polarization are sums and differences of four products.
//
// Output: event-major [n][4][N] complex64; or the planes of an incoherent
// sample (plane 2 (l N + a) = Re A_a^l); or the planes that M is built from
// (n 4 pseudo-events of N waves: plane 2a = Re A_a, event 4i + l), as a load
// needs them, without an event-major copy in between. With amax, the largest
// |Re| + |Im| of each wave over events and components is taken on the way.
#include <algorithm>

#include "ff.cuh"

namespace pwa {

namespace {

constexpr int kCovThreads = 128;

__device__ __forceinline__ double mdot(const double (&a)[4], const double (&b)[4])
{
    return a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3];
}

// The four components of one event and wave in FP64: A[l] = (re, im).
__device__ __noinline__ void cov_fp64(const double *v, double mass, double width, bool spin2,
                                      float2 (&A)[4])
{
    const double mK = 0.493677, Q0 = 0.197327, isq2 = 0.70710678118654752440;
    double q[4], k1[4], k2[4], p[4], r[4], rt[4];
    q[1] = v[0];
    q[2] = v[1];
    q[3] = v[2];
    const double qq = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    q[0] = qq;
    k1[0] = sqrt(mK * mK + v[3] * v[3] + v[4] * v[4] + v[5] * v[5]);
    k2[0] = sqrt(mK * mK + v[6] * v[6] + v[7] * v[7] + v[8] * v[8]);
    for (int c = 0; c < 3; ++c) {
        k1[c + 1] = v[3 + c];
        k2[c + 1] = v[6 + c];
    }
    for (int c = 0; c < 4; ++c) {
        p[c] = k1[c] + k2[c];
        r[c] = k1[c] - k2[c];
    }
    const double pp = mdot(p, p), rp = mdot(r, p);
    for (int c = 0; c < 4; ++c)
        rt[c] = r[c] - rp / pp * p[c];
    const double rr = mdot(rt, rt);
    const double Q2 = pp / 4.0 - mK * mK;
    const double b2 = sqrt(13.0 / (Q2 * Q2 + 3.0 * Q2 * Q0 * Q0 + 9.0 * Q0 * Q0 * Q0 * Q0));
    double e[2][4];
    const double ux = -q[2], uy = q[1];  // z x q
    const double un = sqrt(ux * ux + uy * uy);
    e[0][0] = 0.0;
    e[0][3] = 0.0;
    if (un > 1e-12 * qq) {
        e[0][1] = ux / un;
        e[0][2] = uy / un;
    } else {
        e[0][1] = 1.0;
        e[0][2] = 0.0;
    }
    const double qh0 = q[1] / qq, qh1 = q[2] / qq, qh2 = q[3] / qq;
    e[1][0] = 0.0;
    e[1][1] = qh1 * e[0][3] - qh2 * e[0][2];
    e[1][2] = qh2 * e[0][1] - qh0 * e[0][3];
    e[1][3] = qh0 * e[0][2] - qh1 * e[0][1];
    const double D = mass * mass - pp, G = mass * width;
    const double inv = 1.0 / (D * D + G * G);
    const double br = D * inv, bi = G * inv;
#pragma unroll
    for (int im = 0; im < 2; ++im) {
        const double psr[4] = {0.0, im == 0 ? -isq2 : isq2, 0.0, 0.0};
        const double psi[4] = {0.0, 0.0, -isq2, 0.0};
#pragma unroll
        for (int il = 0; il < 2; ++il) {
            const double(&ww)[4] = e[il];
            double cr = mdot(psr, ww), ci = mdot(psi, ww);
            if (spin2) {
                const double prw = mdot(ww, rt), pwp = mdot(ww, p);
                const double ar = mdot(psr, rt), ai = mdot(psi, rt);
                const double apr = mdot(psr, p), api = mdot(psi, p);
                cr = b2 * (ar * prw - rr / 3.0 * (cr - apr * pwp / pp));
                ci = b2 * (ai * prw - rr / 3.0 * (ci - api * pwp / pp));
            }
            A[2 * im + il] = make_float2(__double2float_rn(br * cr - bi * ci),
                                         __double2float_rn(br * ci + bi * cr));
        }
    }
}

__device__ __forceinline__ ff ff_sum3(ff a, ff b, ff c) { return ff_add(ff_add(a, b), c); }

// Contractions of one event pair and polarization: (X, Y) = -(r_x, r_y) (e.r) +
// (4/3) Q^2 ((e_x, e_y) + (p_x, p_y) (e.p) / p.p), so that the spin-2 contraction
// of psi(+1) is B2 (X + i Y) / sqrt2 (e.r and e.p: products of 3-vectors).
__device__ __forceinline__ void spin2(const ff (&e)[3], bool has_z, const ff (&r)[3], const ff (&p)[3],
                                      ff q43, ff ipp, ff &X, ff &Y)
{
    ff er = ff_norm(ff_dot(e[0], r[0], e[1], r[1])), ep = ff_norm(ff_dot(e[0], p[0], e[1], p[1]));
    if (has_z) {
        er = ff_add(er, ff_mul(e[2], r[2]));
        ep = ff_add(ep, ff_mul(e[2], p[2]));
    }
    const ff t = ff_norm(ff_mul(ep, ipp));
    const ff x = ff_add(e[0], ff_mul(p[0], t)), y = ff_add(e[1], ff_mul(p[1], t));
    X = ff_norm(ff_det(q43, x, r[0], er));
    Y = ff_norm(ff_det(q43, y, r[1], er));
}

template <int MODE>
__global__ void __launch_bounds__(kCovThreads, 4)
    cov_amp_kernel(const double *__restrict__ p3, int64_t n, int N, const __grid_constant__ CovTable table,
                   bool fp64_only, float *__restrict__ out, int64_t pitch, float *__restrict__ amax)
{
    __shared__ CovWave w[kMaxWaves];
    __shared__ uint2 queue[kCovThreads / 32][96];  // (event, wave) pairs left to FP64, per warp
    __shared__ unsigned wave_max[kMaxWaves];       // bits of non-negative floats
    for (int i = threadIdx.x; i < (int)(N * sizeof(CovWave) / 4); i += blockDim.x)
        reinterpret_cast<int *>(w)[i] = reinterpret_cast<const int *>(table.w)[i];
    for (int i = threadIdx.x; i < N; i += blockDim.x)
        wave_max[i] = 0u;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint2 *q = queue[warp];
    int queued = 0;  // the same in every lane
    auto store = [&](int64_t i, int a, const float2 (&A)[4]) {
        if (MODE == kCovEventMajor) {
            float2 *o = reinterpret_cast<float2 *>(out) + i * 4 * N + a;
#pragma unroll
            for (int l = 0; l < 4; ++l)
                o[(int64_t)l * N] = A[l];
        } else if (MODE == kCovPlanes) {
#pragma unroll
            for (int l = 0; l < 4; ++l) {
                out[(int64_t)(2 * (l * N + a)) * pitch + i] = A[l].x;
                out[(int64_t)(2 * (l * N + a) + 1) * pitch + i] = A[l].y;
            }
        } else {
            *reinterpret_cast<float4 *>(out + (int64_t)(2 * a) * pitch + 4 * i) =
                make_float4(A[0].x, A[1].x, A[2].x, A[3].x);
            *reinterpret_cast<float4 *>(out + (int64_t)(2 * a + 1) * pitch + 4 * i) =
                make_float4(A[0].y, A[1].y, A[2].y, A[3].y);
        }
    };
    auto largest = [](const float2 (&A)[4]) {
        float m = 0.f;
#pragma unroll
        for (int l = 0; l < 4; ++l)
            m = fmaxf(m, fabsf(A[l].x) + fabsf(A[l].y));
        return m;
    };
    // FP64 values of the last (up to 32) queued pairs, one per lane, over the
    // provisional ones in the output
    auto drain = [&]() {
        const int take = queued < 32 ? queued : 32;
        queued -= take;
        if (lane < take) {
            const uint2 it = q[queued + lane];
            const CovWave &W = w[it.y];
            float2 A[4];
            cov_fp64(p3 + 9 * (int64_t)it.x, W.mass, W.width, W.spin == 2, A);
            store(it.x, W.index, A);
            if (amax)
                atomicMax(&wave_max[W.index], __float_as_uint(largest(A)));
        }
        __syncwarp();
    };
    const bool pairs = !fp64_only && !table.fp64_only;
    const double mK2d = 0.493677 * 0.493677, Q02 = 0.197327 * 0.197327;
    const int64_t stride = (int64_t)gridDim.x * (2 * kCovThreads);
    for (int64_t e0 = ((int64_t)blockIdx.x * (kCovThreads / 32) + warp) * 64; e0 < n; e0 += stride) {
        // this lane's events; past the end the last one is repeated (nothing
        // of it is stored)
        const bool in0 = e0 + lane < n, in1 = e0 + 32 + lane < n;
        const int64_t i0 = in0 ? e0 + lane : n - 1, i1 = in1 ? e0 + 32 + lane : n - 1;
        bool ok0 = pairs, ok1 = pairs;
        const double *v0 = p3 + 9 * i0, *v1 = p3 + 9 * i1;
        auto split = [&](int c) { return ff_split(v0[c], v1[c], ok0, ok1); };
        // the polarizations: e1 = (-q_y, q_x, 0) / un, e2 = (-c e1_y, c e1_x, un / |q|), c = q_z / |q|
        ff e1[3], e2[3];
        {
            const ff qx = split(0), qy = split(1), qz = split(2);
            const ff un2 = ff_add(ff_sqr(qx), ff_sqr(qy)), qq2 = ff_add(un2, ff_sqr(qz));
            float u0, u1, s0, s1;
            upk2(un2.h, u0, u1);
            upk2(qq2.h, s0, s1);
            // photons within 2^-20 of the axis, or without momentum: FP64
            ok0 = ok0 && u0 >= 0x1p-40f * s0 && u0 >= 0x1p-60f;
            ok1 = ok1 && u1 >= 0x1p-40f * s1 && u1 >= 0x1p-60f;
            const ff un = ff_sqrt(un2), iun = ff_norm(ff_rcp(un)), iqq = ff_norm(ff_rcp(ff_sqrt(qq2)));
            e1[0] = ff_neg(ff_norm(ff_mul(qy, iun)));
            e1[1] = ff_norm(ff_mul(qx, iun));
            const ff c = ff_norm(ff_mul(qz, iqq));
            e2[0] = ff_neg(ff_norm(ff_mul(c, e1[1])));
            e2[1] = ff_norm(ff_mul(c, e1[0]));
            e2[2] = ff_norm(ff_mul(un, iqq));
        }
        // p = k1 + k2, r = k1 - k2, p.p, and the largest sizes for the bounds
        ff p[3], r[3], p0;
        {
            const ff mk = ff_const(mK2d);
            ff k1s = mk, k2s = mk;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const ff a = split(3 + c), b = split(6 + c);
                k1s = ff_add(k1s, ff_sqr(a));
                k2s = ff_add(k2s, ff_sqr(b));
                p[c] = ff_add(a, b);
                r[c] = ff_sub(a, b);
            }
            p0 = ff_add(ff_sqrt(k1s), ff_sqrt(k2s));
        }
        const ff p02 = ff_norm(ff_sqr(p0));
        const ff pp = ff_sub(p02, ff_sum3(ff_norm(ff_sqr(p[0])), ff_sqr(p[1]), ff_sqr(p[2])));
        // p.p to 2^-42 of p_0^2 (p_0 to 2^-44.8, the sums to 2^-43.5 of p_0^2), so
        // Q^2 = p.p / 4 - mK^2 to 2^-44 of it
        const f2 eps_q = mul2(p02.h, dup2(0x1p-44f));
        const ff Q2 = ff_sub(ff{mul2(pp.h, dup2(0.25f)), mul2(pp.l, dup2(0.25f))}, ff_const(mK2d));
        const ff ipp = ff_norm(ff_rcp(pp));
        // B2 / sqrt2 = sqrt(13 / 2 / den), den = Q^2 (Q^2 + 3 Q0^2) + 9 Q0^4
        const ff den = ff_add(ff_mul(Q2, ff_add(Q2, ff_const(3.0 * Q02))), ff_const(9.0 * Q02 * Q02));
        const ff iden = ff_norm(ff_rcp(den));
        const ff b2 = ff_sqrt(ff_norm(ff_mul(iden, ff_const(6.5))));
        const ff q43 = ff_norm(ff_mul(Q2, ff_const(4.0 / 3.0)));
        // the contractions (re, im) of psi(+1) with e1 and e2
        const ff isq2 = ff_const(0.70710678118654752440);
        ff c0[2][2], c2[2][2];
        spin2(e1, false, r, p, q43, ipp, c2[0][0], c2[0][1]);
        spin2(e2, true, r, p, q43, ipp, c2[1][0], c2[1][1]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            c2[0][k] = ff_norm(ff_mul(b2, c2[0][k]));
            c2[1][k] = ff_norm(ff_mul(b2, c2[1][k]));
            c0[0][k] = ff_norm(ff_mul(isq2, e1[k]));
            c0[1][k] = ff_norm(ff_mul(isq2, e2[k]));
        }
        // error of the spin-2 contractions: with |e| = 1 and g = p_0^2 / p.p, the
        // products of X and Y are below S = r.r + (4/3) |Q^2| (1 + g) (3-vectors)
        // and wrong by at most 2^-42.5 of that (e.r by 2^-43 |r|) and (4/3) (1 + g)
        // times Q^2's error; B2 by 2^-43 and (Q^2 + 3/2 Q0^2) / den times Q^2's error
        f2 err2;
        {
            const f2 R2 = fma2(r[0].h, r[0].h, fma2(r[1].h, r[1].h, mul2(r[2].h, r[2].h)));
            const f2 g1 = mul2(fma2(p02.h, abs2(ipp.h), dup2(1.0f)), dup2(1.34f));
            const f2 S = fma2(g1, abs2(Q2.h), mul2(R2, dup2(1.01f)));
            const f2 rel = fma2(mul2(eps_q, abs2(iden.h)), add2(abs2(Q2.h), dup2(0.0585f)), dup2(0x1.8p-42f));
            err2 = mul2(abs2(b2.h), fma2(S, rel, mul2(g1, eps_q)));
        }
        const f2 eps_pp = mul2(p02.h, dup2(0x1p-42f));

        for (int a = 0; a < N; ++a) {
            const CovWave &W = w[a];
            const bool sp2 = W.spin == 2;
            // BW = (D + i G) / (D^2 + G^2)
            const ulonglong2 m2 = *reinterpret_cast<const ulonglong2 *>(&W.m2),
                             gg = *reinterpret_cast<const ulonglong2 *>(&W.g),
                             g2 = *reinterpret_cast<const ulonglong2 *>(&W.g2);
            const ff D = ff_sub(ff{m2.x, m2.y}, pp);
            const ff dd = ff_sqr(D);
            const ff dn = ff_two_sum(dd.h, g2.x);
            const ff inv = ff_rcp(ff{dn.h, add2(dn.l, add2(dd.l, g2.y))});
            const ff br = ff_norm(ff_mul(D, inv)), bi = ff_norm(ff_mul(ff{gg.x, gg.y}, inv));
            const f2 b = add2(abs2(br.h), abs2(bi.h));
            // relative error: the products' (BW to 2^-43.7, C to 2^-43.2, their product
            // and sums 2^-45), and D's rounding times |BW|
            const f2 rel = fma2(b, fma2(m2.x, dup2(0x1p-46f), eps_pp), dup2(0x1p-42f));
            float2 A0[4], A1[4];
            bool s0 = ok0, s1 = ok1;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const ff cr = sp2 ? c2[k][0] : c0[k][0], ci = sp2 ? c2[k][1] : c0[k][1];
                const ff x = ff_mul(br, cr), y = ff_mul(bi, ci), z = ff_mul(br, ci), v = ff_mul(bi, cr);
                const f2 size = add2(abs2(cr.h), abs2(ci.h));
                const f2 err = mul2(b, sp2 ? fma2(size, rel, err2) : mul2(size, rel));
                float t0, t1;
                bool a0, a1;
                // M = +1: (x - y, z + v); M = -1: (-(x + y), z - v)
                ff u = ff_two_diff(x.h, y.h);
                ff_round(ff{u.h, add2(u.l, sub2(x.l, y.l))}, err, A0[k].x, A1[k].x, a0, a1);
                s0 = s0 && a0;
                s1 = s1 && a1;
                u = ff_two_sum(z.h, v.h);
                ff_round(ff{u.h, add2(u.l, add2(z.l, v.l))}, err, A0[k].y, A1[k].y, a0, a1);
                s0 = s0 && a0;
                s1 = s1 && a1;
                u = ff_two_sum(x.h, y.h);
                ff_round(ff{u.h, add2(u.l, add2(x.l, y.l))}, err, t0, t1, a0, a1);
                A0[2 + k].x = -t0;
                A1[2 + k].x = -t1;
                s0 = s0 && a0;
                s1 = s1 && a1;
                u = ff_two_diff(z.h, v.h);
                ff_round(ff{u.h, add2(u.l, sub2(z.l, v.l))}, err, A0[2 + k].y, A1[2 + k].y, a0, a1);
                s0 = s0 && a0;
                s1 = s1 && a1;
            }
            if (in0)
                store(i0, W.index, A0);
            if (in1)
                store(i1, W.index, A1);
            if (amax) {
                const float t = fmaxf(in0 && s0 ? largest(A0) : 0.f, in1 && s1 ? largest(A1) : 0.f);
                const unsigned u = __reduce_max_sync(0xffffffffu, __float_as_uint(t));
                if (lane == 0)
                    atomicMax(&wave_max[W.index], u);
            }
            // pairs in doubt wait for a warp's worth of them
            const bool d0 = !s0 && in0, d1 = !s1 && in1;
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
                    drain();
            }
        }
    }
    while (queued > 0)
        drain();
    if (amax) {
        __syncthreads();
        for (int i = threadIdx.x; i < N; i += blockDim.x)
            if (wave_max[i])
                atomicMax(reinterpret_cast<int *>(amax + i), (int)wave_max[i]);
    }
}

}  // namespace

void cov_table(const pwa_cov_wave *waves, int N, CovTable *t)
{
    t->fp64_only = 0;
    for (int a = 0; a < N; ++a) {
        const double m = waves[a].mass, g = m * waves[a].width;
        CovWave &w = t->w[a];
        w.m2 = gen_pair(m * m);
        w.g = gen_pair(g);
        w.g2 = gen_pair(g * g);
        w.mass = m;
        w.width = waves[a].width;
        w.spin = waves[a].spin;
        w.index = a;
        // scales whose squares would leave the float range in D^2 + G^2
        if (!(g * g >= 0x1p-60 && g * g <= 0x1p60 && m * m <= 0x1p30))
            t->fp64_only = 1;
    }
}

cudaError_t launch_cov_amp_gen(const double *p3, int64_t n, int N, const CovTable &table, bool fp64_only,
                               float *out, int mode, int64_t pitch, float *amax, int num_sms,
                               cudaStream_t s)
{
    if (n < 1 || N < 1 || N > kMaxWaves)
        return cudaErrorInvalidValue;
    const int64_t need = (n + 2 * kCovThreads - 1) / (2 * kCovThreads);
    const unsigned g = (unsigned)std::min<int64_t>(need, (int64_t)num_sms * 4);
    if (mode == kCovEventMajor)
        cov_amp_kernel<kCovEventMajor><<<g, kCovThreads, 0, s>>>(p3, n, N, table, fp64_only, out, pitch, amax);
    else if (mode == kCovPlanes)
        cov_amp_kernel<kCovPlanes><<<g, kCovThreads, 0, s>>>(p3, n, N, table, fp64_only, out, pitch, amax);
    else
        cov_amp_kernel<kCovPseudoEvents><<<g, kCovThreads, 0, s>>>(p3, n, N, table, fp64_only, out, pitch, amax);
    return cudaGetLastError();
}

}  // namespace pwa
