// No header, but the end of a direct-form evaluation kernel, part of its body (a function,
// inlined, cost the coherent kernel 2 of 44 us at 1M events x 20 waves): with
// each CTA's partial sums in `sc`, the last CTA adds them up and writes the
// results. Uses the kernel's a, sc, work_flags, s_flags, s_last, warp, lane, N,
// NF, C::THREADS and, once idle, the shared memory at `tiles`.
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_flags)
            atomicOr(work_flags, s_flags);
        __threadfence();
        const unsigned t = atomicAdd(a.ticket, 1u);
        s_last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last)
        return;

    // ---- last CTA: deterministic final sum + normalisation term ---------
    // One warp per component (2N+1 float-float ones, then the 2 integer
    // ones): lane l adds CTAs l, l + 32, ... (coalesced loads, all issued
    // before the adds, with M V and the launch's flags: one L2 round trip),
    // then a fixed shuffle tree. (The partials are read with L2 loads after
    // the ticket, so no further fence is needed.)
    const int Nw = a.n_waves;
    const int G_ = gridDim.x;
    constexpr int NWARPS = C::THREADS / 32;
    constexpr int CPW = (NF + 2 + NWARPS - 1) / NWARPS;  // components per warp
    constexpr int QB = 5;                                 // loads per lane and component in flight
    dfloat *tot_f = reinterpret_cast<dfloat *>(tiles);                  // [NF]
    long long *tot_i = reinterpret_cast<long long *>(tot_f + NF);       // [2]
    double *smv = reinterpret_cast<double *>(tot_i + 2);                // [2N] M V, V^H M V
    const double mv_i = threadIdx.x < 2 * Nw ? __ldcg(&sc.mv[threadIdx.x])
                                             : threadIdx.x == 2 * Nw ? __ldcg(&sc.mv[2 * kMaxWaves])
                                                                      : 0.0;
    const int wf = __ldcg(work_flags);
    {
        // a partial is 8 bytes either way: a float pair (hi in the low word)
        // or an integer
        const unsigned long long *pf64 = reinterpret_cast<const unsigned long long *>(sc.pf);
        const unsigned long long *pi64 = reinterpret_cast<const unsigned long long *>(sc.pi);
        dfloat acc[CPW];
        long long iacc[CPW];
#pragma unroll
        for (int k = 0; k < CPW; ++k) {
            acc[k] = dfloat{0.f, 0.f};
            iacc[k] = 0;
        }
        for (int b0 = 0; b0 < G_; b0 += 32 * QB) {
            unsigned long long r[CPW][QB];
#pragma unroll
            for (int k = 0; k < CPW; ++k) {
                const int comp = warp + k * NWARPS;
                const unsigned long long *src =
                    comp < NF ? pf64 + (size_t)comp * G_ : pi64 + (size_t)(comp - NF) * G_;
#pragma unroll
                for (int q = 0; q < QB; ++q) {
                    const int b = b0 + lane + 32 * q;
                    r[k][q] = (b < G_ && comp < NF + 2) ? __ldcg(src + b) : 0ull;
                }
            }
#pragma unroll
            for (int k = 0; k < CPW; ++k) {
                if (warp + k * NWARPS < NF) {
#pragma unroll
                    for (int q = 0; q < QB; ++q)
                        acc[k] = df_add(acc[k], dfloat{__uint_as_float((unsigned)r[k][q]),
                                                       __uint_as_float((unsigned)(r[k][q] >> 32))});
                } else {
#pragma unroll
                    for (int q = 0; q < QB; ++q)
                        iacc[k] += (long long)r[k][q];
                }
            }
        }
#pragma unroll
        for (int k = 0; k < CPW; ++k) {
            const int comp = warp + k * NWARPS;
            if (comp < NF) {
                const dfloat v = warp_sum(acc[k]);
                if (lane == 0)
                    tot_f[comp] = v;
            } else if (comp < NF + 2) {
                const long long v = warp_sum(iacc[k]);
                if (lane == 0)
                    tot_i[comp - NF] = v;
            }
        }
    }
    if (threadIdx.x <= 2 * Nw)
        smv[threadIdx.x] = mv_i;
    __syncthreads();
    const bool invalid = (wf & (FLAG_DOMAIN | FLAG_TIMEOUT)) != 0;
    for (int c = threadIdx.x; c < 2 * Nw + 1; c += blockDim.x) {  // padded waves excluded
        const dfloat v = tot_f[c];
        if (c > 0) {
            // gradient: - sum_i conj(A) S / I + (M V)
            if (a.grad)
                a.grad[c - 1] = invalid ? 0.0 : (smv[c - 1] - (double)v.hi) - (double)v.lo;
        } else {
            // ln sum: integer part and exponents are exact; the rest is small
            const long long li = tot_i[0], ei = tot_i[1];
            const double lnsum =
                fma((double)ei, kLn2, ((double)li + ((double)v.hi + (double)v.lo)) * 0x1p-23);
            double nll = smv[2 * Nw] - lnsum;
            if (wf & FLAG_DOMAIN)
                nll = INFINITY;
            if (wf & FLAG_TIMEOUT)
                nll = NAN;
            a.nll[0] = nll;
            if (wf)
                atomicOr(a.status, wf);
            if (a.done)
                atomicAdd(a.done, 1);
        }
    }
    if (a.host_flag)
        __threadfence_system();  // this thread's results reach the host before the flag
    __syncthreads();
    if (threadIdx.x == 0) {
        *work_flags = 0;
        *a.ticket = 0u;
        if (a.host_flag)
            *reinterpret_cast<volatile unsigned long long *>(a.host_flag) =
                ((unsigned long long)a.seq << 32) | (unsigned)wf;
    }
