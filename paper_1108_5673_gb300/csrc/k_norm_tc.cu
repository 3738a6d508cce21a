// MC normalisation matrix on the tensor cores (the inner bracket of the
// second term of Eq. 3, built once per sample as Sec. 2 says it can be when
// masses and widths are fixed):
//
//   M[a][b] = (1/N_gen) sum_{j in accepted MC} conj(A_a(j)) A_b(j).
//
// With the real rows x_p(j), p = 2a (Re A_a) and 2a + 1 (Im A_a), this is the
// symmetric contraction over the events G = X X^T, G[p][q] = sum_j x_p(j)
// x_q(j), and Re M_ab = G[2a][2b] + G[2a+1][2b+1], Im M_ab = G[2a][2b+1] -
// G[2a+1][2b].
//
// Exact digits. Each wave a gets one power of two 2^r_a > 2 max_j (|Re A_a| +
// |Im A_a|) for the whole sample. Every float x of rows 2a, 2a+1 is written
// as five fixed-point digits x = sum_{s=1..5} t_s + rest, t_s = c_s 2^(r_a -
// 8s) with integers |c_s| <= 128 and |rest| <= 2^(r_a - 41). The kernel works on
// x 2^-r_a (an exact product), so that every wave's digits lie at the same place
// whatever its unit, and the sums get 2^(r_a + r_b) back in FP64 at the end. Digit s
// is the remainder rounded to the nearest multiple of 2^-8s (by adding and
// subtracting 1.5 2^(23 - 8s)), an exact float operation, and t_s has
// at most 8 significant bits, so it is an exact BF16 value. Any x with |x| >=
// 2^(r_a - 17) is a multiple of 2^(r_a - 40) and has rest = 0. A product of
// digits s and t of rows p and q is c c' 2^(r_p + r_q - 8(s + t)): within one
// accumulator entry (p, q) of one digit pair all products are integer
// multiples of one quantum and at most 2^14 of it, so the tensor cores' FP32
// sum over 1024 events (at most 2^24 quanta) is exact.
//
// Digit blocks D_st[p][q] = sum_j t_s(p, j) t_t(q, j), R rows each, from MMAs on
// the same digits in shared memory. Up to 20 waves: one or two per tile, the first
// with as many digits as fit M = 128 rows (S1 = 5 up to 12 waves, 3 up to 20) against
// all five, the second [X4; X5] against X4. An M = 128 MMA reads its 128 A rows
// whatever the number of columns, which is what a small model's tile costs, hence
// one MMA where everything fits. With D_ts = D_st^T these are all pairs (all but
// (5,5) beyond 12 waves), all exact, drained every 1024 events:
//   G = T + U + U^T, T the products whose transposes are among them too (a
//   symmetric sum), U the others,
// so that one sum W = T/2 + U per (row, column) serves, G = W + W^T: float-
// float for the first accumulator's blocks, plain FP32 for the second's, which are
// below 2^-28 of the leading one. Per event and real entry of G the error is
// at most 2^-41 (|x_p| 2^r_q [|x_q| < 2^(r_q - 17)] + |x_q| 2^r_p [|x_p| <
// 2^(r_p - 17)]) + 2^(r_p + r_q - 61), with unbiased signs apart from the last
// term.
//
// Beyond 20 waves, where M used to come from exact FP64 products, the rest is kept
// too: Z = rest rounded to BF16 (a float: 8 bits of its own, whatever its size) is a
// sixth row block, and the MMAs are [X1; X2] against [X1; X2; X3; X4] into the first
// accumulator, [X1; X2] and [X3; X4] against [X5; Z] and [X3; X4] against [X3; X4]
// into the second: every pair but (5,5), (5,Z) and (Z,Z). (The second's sums are
// FP32 sums, no longer all exact: (1,5) and the products with Z are at most 2^-28 of
// G.) The error above shrinks by 2^-9.
//
// Largest error of M relative to sqrt(M_aa M_bb), against double-double sums, for
// uniform m and the harmonics and widths of the benchmark's waves (0.05 to 0.4 GeV),
// 50k / 200k / 1M events: 20 waves 3e-14 / 2e-14 / 7e-15; 21 and more 2.7e-16 / 3e-16 /
// 7e-16 (without Z 5e-14 / 3e-14 / 1e-14), FP64 sums of the exact products 1.5e-15 /
// 1.4e-15 / 1.4e-15. Where a wave's largest amplitude is so far above its rms that this
// would not hold (norm_tc_spread_ok), M is built again by the FP64 kernel.
//
// More than 32 waves: the accumulators no longer fit tensor memory, so the
// waves are cut into three blocks and three launches take two blocks each
// (two TMA boxes per tile); between them every pair of waves is covered, at
// twice the one-pass traffic and digit work.
//
// Per CTA (persistent, one per SM), sixteen warps (128 registers a thread): a
// TMA warp streams 64-event tiles of the planes; six consumer warps in GROUPS
// groups (tile j to group j mod GROUPS, its row pairs shared by the group's
// warps: one-warp groups for the few rows of a small model, so that several
// tiles are in flight, three-warp groups from 16 waves on) write the digits
// K-major with 128-byte swizzle into a ring of digit buffers; one thread
// issues the MMAs (kind::f16, K = 16, four steps per tile); eight drain warps
// (two per lane quarter, half of each block's columns) add the accumulators
// into W. Up to 20 waves two accumulator sets alternate; beyond, one set, whose
// two accumulators hand over separately, so that the first MMA of the next period
// runs while the second accumulator is drained. The CTA's share of M goes to
// global memory with the CTA index innermost; norm_tc_finalize adds the CTAs
// in a fixed order, divides by N_gen and fills the Hermitian matrix.
//
// Bound: the digit split (30 packed FP32 operations per two rows and four
// events, on six warps) and the MMAs, about 1300 and 1280 cycles per tile at
// 32 waves, overlapping in part; at few waves the fixed cost of a tile, ~600 cycles
// (a copy 430, a step of the issuer). Producer and issuer run as converged warps
// with one elected lane issuing, so that their addresses and descriptors stay in
// uniform registers: as single lanes they took 5M x 4 from 183 to 207 us a call, 5M
// x 16 from 305 to 340, 10M x 12 from 381 to 404. Waiting for the loads before a stage
// is released took 5M x 20 from 339 to 349. Per call of pwa_build_norm: 10M x 32 in
// 0.99 ms (2.6 TB/s of amplitudes), 5M x 24 0.45, 5M x 20 0.35, 10M x 12 0.38, 4M x 48
// 1.24; without Z 0.92, 0.39 and 1.15 at 32, 24 and 48 waves; on the FP64 pipe beyond 20
// waves 81 ms at 10M x 32 and 69 ms at 4M x 48. Digit buffers and stages: with Z at 32
// waves four buffers leave two stages; two buffers and eight stages 1.19 ms, three
// two-warp groups with a buffer and a stage each 1.03, one group of six warps 1.03.
#include <string.h>

#include "pwa_internal.cuh"

namespace pwa {

namespace {

constexpr int kNTE = 64;         // events per tile (one K-atom)
constexpr int kNCons = 6;        // consumer warps
constexpr int kNDrain = 8;       // drain warps (warps 2..9: lane quarter = warp % 4)
constexpr int kNFirstDrain = 2;
constexpr int kNFirstCons = kNFirstDrain + kNDrain;
constexpr int kNWarps = kNFirstCons + kNCons;  // 0 TMA, 1 MMA, 2-9 drain, 10-15 consumers
constexpr int kNThreads = kNWarps * 32;
constexpr int kNDigits = 5;
constexpr int kNPeriod = 16;     // tiles per accumulation period (1024 events: sums <= 2^24)
constexpr uint32_t kNTmemCols = 512;
constexpr int kNFinMaxRounds = 8;    // CTAs up to 32 x 8
constexpr int kNMaxOnePass = 32;     // waves of one launch

constexpr int round_up16(int x) { return (x + 15) / 16 * 16; }
constexpr int cmax(int a, int b) { return a > b ? a : b; }
constexpr int cmin(int a, int b) { return a < b ? a : b; }

template <int NW>
struct NormTcCfg {
    static constexpr int R = 2 * NW;                         // real rows (padded waves)
    // digits in the first MMA's A operand; B1 digits in its B operand; column
    // blocks of the second accumulator (see the header); row blocks of a buffer
    static constexpr int S1 = NW <= 12 ? 5 : NW <= 20 ? 3 : 2;
    static constexpr bool REST = S1 == 2;                    // the rest of x as a sixth digit
    static constexpr int B1 = REST ? 4 : kNDigits;
    static constexpr int B2 = S1 == 5 ? 0 : S1 == 3 ? 1 : 4;
    static constexpr int ROWBLOCKS = REST ? kNDigits + 1 : kNDigits;
    static constexpr int N1 = round_up16(B1 * R);            // columns of the first accumulator
    static constexpr int N2 = round_up16(B2 * R);            // of the second
    static constexpr int NI2 = REST ? 2 * R : N2;            // one instruction's columns in it
    static constexpr int NI1 = N1 > 256 ? N1 / 2 : N1;       // one instruction's columns
    static constexpr int WPG = NW <= 8 ? 1 : NW <= 12 ? 2 : 3;  // warps per consumer group
    static constexpr int GROUPS = kNCons / WPG;
    static constexpr int ITERS = (NW + WPG - 1) / WPG;       // row pairs per warp and tile
    static constexpr int NBUF = NW <= 12 ? 6 : 4;
    static constexpr int NACC = 2 * (N1 + N2) <= (int)kNTmemCols ? 2 : 1;
    // buffer rows: the digits, the B operands' padding, and the 128 rows that
    // each A operand reads
    static constexpr int BUFROWS =
        REST ? ROWBLOCKS * R : cmax(cmax(N1, 128), B2 ? cmax(S1 * R + N2, S1 * R + 128) : 0);
    static constexpr uint32_t JBYTES = BUFROWS * 128;        // one 64-event K-atom of every row
    static constexpr uint32_t STAGE_BYTES = R * kNTE * 4;
    static constexpr int STAGES =
        cmin(18, (int)((224 * 1024 - NBUF * JBYTES) / STAGE_BYTES)) / GROUPS * GROUPS;
    static constexpr size_t SMEM = (size_t)NBUF * JBYTES + (size_t)STAGES * STAGE_BYTES + 1024;
    // the CTA's sums W[S1 R][R] as doubles reuse the digit buffers
    static constexpr size_t SUMS_BYTES = (size_t)S1 * R * R * sizeof(double);
    static_assert(S1 * R <= 128, "S1 digits of every row fit M = 128");
    static_assert(NI1 % 16 == 0 && NI1 <= 256 && NI2 % 16 == 0 && NI2 <= 256 && N1 % NI1 == 0,
                  "N of the MMA");
    static_assert(!REST || BUFROWS >= S1 * R + 128, "rows of the second A operand");
    static_assert(NACC * (N1 + N2) <= (int)kNTmemCols, "tensor memory");
    static_assert(NW % 4 == 0, "drain in 4-column steps, 8-row swizzle atoms per digit");
    // Stages and buffers belong to one group each: a group's parity wait on
    // the phase of use k is then on a barrier whose use k - 1 it consumed
    // itself. Shared ones would let a wait pass one phase too early, because
    // copies can land out of order and groups can drift apart.
    static_assert(STAGES >= GROUPS && STAGES % GROUPS == 0 && NBUF % GROUPS == 0, "owned rings");
    static_assert(JBYTES % 1024 == 0 && STAGE_BYTES % 1024 == 0, "swizzle atoms stay 1 KB aligned");
    static_assert(SMEM <= 227 * 1024, "shared memory");
    static_assert(SUMS_BYTES <= (size_t)NBUF * JBYTES, "sums fit in the digit buffers");
};

// The waves of one launch: box k of blk waves starts at wave first[k]; local
// wave w is wave first[w / blk] + w % blk (past the model's end: a zero wave).
struct NormBlocks {
    int n_box, blk, first[2];
    __host__ __device__ int local() const { return n_box * blk; }
    __host__ __device__ int global(int w) const { return w < blk ? first[0] + w : first[1] + w - blk; }
};

// Byte offset of (row, byte b of the row) in a K-major operand with 128-byte
// swizzle: 128-byte rows in 8-row (1 KB) atoms, the 16-byte chunk index
// XOR-ed with the row within the atom.
__device__ __forceinline__ uint32_t sw128(int row, uint32_t b)
{
    return (uint32_t)(row >> 3) * 1024 + (uint32_t)(row & 7) * 128 +
           ((((b >> 4) ^ (uint32_t)(row & 7)) & 7) << 4) + (b & 15);
}

// Two floats (events e, e + 1) to a packed BF16 pair, event e in the low
// half (the smaller K index). The inputs are exact BF16 values here.
__device__ __forceinline__ uint32_t to_bf16x2(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

__device__ __forceinline__ void st_shared_v2(uint32_t addr, uint32_t a, uint32_t b)
{
    // no memory clobber: loads of the next rows may move above it; the proxy
    // fence that follows the stores is ordered after them (both volatile)
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b));
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t *r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}

// (hi, lo) += x for two float-float sums at once (Knuth's TwoSum).
__device__ __forceinline__ void two_sum2(f2 &hi, f2 &lo, f2 x)
{
    const f2 s = add2(hi, x);
    const f2 bb = sub2(s, hi);
    lo = add2(lo, add2(sub2(hi, sub2(s, bb)), sub2(x, bb)));
    hi = s;
}

// The scale of wave a's digits: r = floor(log2 amax) + 2 (so that every |x| <
// 2^(r - 1)); a wave that is zero throughout gets r = 0.
__host__ __device__ __forceinline__ int wave_exponent(float amax)
{
    int bits;
    memcpy(&bits, &amax, sizeof bits);
    return amax > 0.f ? ((bits >> 23) & 0xff) - 125 : 0;
}

// NW columns (this thread's half of a block) of its lane's row at `taddr`.
template <int NW>
__device__ __forceinline__ void tmem_row_half(uint32_t taddr, uint32_t (&v)[NW])
{
    if constexpr (NW % 16 == 0) {
#pragma unroll
        for (int c = 0; c < NW / 16; ++c)
            tmem_ld16(taddr + (uint32_t)(16 * c), *reinterpret_cast<uint32_t(*)[16]>(v + 16 * c));
    } else if constexpr (NW % 8 == 0) {
#pragma unroll
        for (int c = 0; c < NW / 8; ++c)
            tmem_ld8(taddr + (uint32_t)(8 * c), *reinterpret_cast<uint32_t(*)[8]>(v + 8 * c));
    } else {
#pragma unroll
        for (int c = 0; c < NW / 4; ++c)
            tmem_ld4(taddr + (uint32_t)(4 * c), v + 4 * c);
    }
}

template <int NW>
__global__ void __launch_bounds__(kNThreads, 1)
    norm_tc_kernel(const __grid_constant__ CUtensorMap map, const float *__restrict__ amax,
                   int n_waves, NormBlocks blocks, int n_tiles, double *__restrict__ part,
                   int *status)
{
    using C = NormTcCfg<NW>;
    constexpr int R = C::R, S1 = C::S1, STAGES = C::STAGES, NBUF = C::NBUF, NACC = C::NACC;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    const uint32_t jbase = smem_u32(base);
    float *stages = reinterpret_cast<float *>(base + (size_t)NBUF * C::JBYTES);
    __shared__ uint64_t full[STAGES], empty[STAGES], jfull[NBUF], jempty[NBUF];
    __shared__ uint64_t accfull[2 * NACC], accempty[2 * NACC], g_done;
    __shared__ float s_scale[R];   // 2^-r of the row's wave
    __shared__ uint32_t tmem_base;
    __shared__ int s_flags;

    // the warp's number as a value the compiler knows to be the same in every lane:
    // what the producer and the issuer compute can then stay in uniform registers
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    // tiles of this CTA: blockIdx.x + j gridDim.x, j < n_my; tile j goes to
    // consumer group j % GROUPS, TMA stage j % STAGES, digit buffer j % NBUF
    const int n_my =
        (n_tiles > (int)blockIdx.x) ? (n_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int box_rows = 2 * blocks.blk;
    const uint32_t stage_tx = (uint32_t)(blocks.n_box * box_rows) * kNTE * 4u;
    const int n_first = n_my < STAGES ? n_my : STAGES;
    auto issue = [&](int j) {
        const int s = j % STAGES;
        float *dst = stages + (size_t)s * (C::STAGE_BYTES / 4);
        const int x = ((int)blockIdx.x + j * (int)gridDim.x) * kNTE;
        mbar_arrive_expect_tx(&full[s], stage_tx);
        for (int k = 0; k < blocks.n_box; ++k)
            tma_load_2d(dst + k * box_rows * kNTE, &map, x, 2 * blocks.first[k], &full[s]);
    };
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], C::WPG);
        }
        for (int b = 0; b < NBUF; ++b) {
            mbar_init(&jfull[b], C::WPG);
            mbar_init(&jempty[b], 1);
        }
        for (int b = 0; b < 2 * NACC; ++b) {
            mbar_init(&accfull[b], 1);
            mbar_init(&accempty[b], kNDrain);
        }
        mbar_init(&g_done, 1);
        fence_barrier_init();
        s_flags = 0;
        for (int j = 0; j < n_first; ++j)
            issue(j);
    }
    // rows of padded waves are never written by TMA: zero them once; so are
    // the buffer rows past the digits, which the MMAs read as padding
    const int in_rows = blocks.n_box * box_rows;
    for (int s = 0; s < STAGES; ++s)
        for (int i = in_rows * kNTE + threadIdx.x; i < R * kNTE; i += blockDim.x)
            stages[(size_t)s * (C::STAGE_BYTES / 4) + i] = 0.f;
    for (int b = 0; b < NBUF; ++b)
        for (uint32_t i = C::ROWBLOCKS * R * 32 + threadIdx.x; i < C::JBYTES / 4; i += blockDim.x)
            reinterpret_cast<uint32_t *>(base + (size_t)b * C::JBYTES)[i] = 0u;
    if (threadIdx.x < R) {
        const int w = threadIdx.x / 2;
        const int g = w < blocks.local() ? blocks.global(w) : n_waves;
        s_scale[threadIdx.x] = g < n_waves ? __int_as_float((127 - wave_exponent(amax[g])) << 23) : 1.f;
    }
    if (warp == 1)
        tmem_alloc(&tmem_base, kNTmemCols);
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_base, 0);
    int flags = 0;

    if (warp == 0) {
        // ---- producer: the warp runs as one, an elected lane issues the copies ----
        const bool lead = elect_one();
        int j = n_first;
        for (; j < n_my; ++j) {
            if (!warp_wait(&empty[j % STAGES], (uint32_t)(j / STAGES - 1) & 1)) {
                flags |= FLAG_TIMEOUT;
                break;
            }
            if (lead)
                issue(j);
            __syncwarp();
        }
        // no copy may still be landing in shared memory when the CTA exits
        for (int q = (j > STAGES ? j - STAGES : 0); q < j; ++q)
            if (!mbar_wait(&full[q % STAGES], (uint32_t)(q / STAGES) & 1))
                flags |= FLAG_TIMEOUT;
    } else if (warp == 1) {
        // ---- MMA issuer: as the producer -----------------------------------
        const bool lead = elect_one();
        const uint32_t id1 = umma_idesc_bf16(128, C::NI1, 0, 0);
        const uint32_t id2 = umma_idesc_bf16(128, C::NI2, 0, 0);
        const uint64_t dK = umma_desc_sw128(0, 16, 1024);
        const uint32_t row2 = (uint32_t)(S1 * R) * 128u;  // byte offset of digit S1 + 1's rows
        bool ok = true;
        for (int j = 0; j < n_my; ++j) {
            const int b = j % NBUF;
            if (!warp_wait(&jfull[b], (uint32_t)(j / NBUF) & 1)) {
                ok = false;
                break;
            }
            const int P = j / kNPeriod, set = P % NACC;
            const bool first = (j % kNPeriod) == 0;
            const bool last = (j % kNPeriod) == kNPeriod - 1 || j == n_my - 1;
            const uint32_t jb = jbase + (uint32_t)b * C::JBYTES;
            const uint32_t acc1 = tmem + (uint32_t)set * (C::N1 + C::N2), acc2 = acc1 + C::N1;
            // an accumulator is free once the period NACC before has been drained
            if (first && P >= NACC && !warp_wait(&accempty[2 * set], (uint32_t)(P / NACC - 1) & 1)) {
                ok = false;
                break;
            }
            tc_fence_after();
            if (lead) {
#pragma unroll
                for (int ks = 0; ks < kNTE / 16; ++ks) {
                    const uint32_t a = jb + (uint32_t)ks * 32;  // 16 events = 32 bytes of a row
#pragma unroll
                    for (int h = 0; h < C::N1 / C::NI1; ++h)
                        umma_bf16(acc1 + (uint32_t)(h * C::NI1), dK + (a >> 4),
                                  dK + ((a + (uint32_t)(h * C::NI1) * 128u) >> 4), id1,
                                  (first && ks == 0) ? 0u : 1u);
                }
                if (last)
                    umma_commit(&accfull[2 * set]);
            }
            __syncwarp();
            if constexpr (C::B2 > 0) {
                if (first && P >= NACC &&
                    !warp_wait(&accempty[2 * set + 1], (uint32_t)(P / NACC - 1) & 1)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                if (lead) {
#pragma unroll
                    for (int ks = 0; ks < kNTE / 16; ++ks) {
                        const uint32_t a = jb + row2 + (uint32_t)ks * 32;
                        const uint32_t acc = (first && ks == 0) ? 0u : 1u;
                        if constexpr (C::REST) {
                            const uint32_t a1 = jb + (uint32_t)ks * 32, b5 = a1 + (uint32_t)(4 * R) * 128u;
                            umma_bf16(acc2, dK + (a1 >> 4), dK + (b5 >> 4), id2, acc);
                            umma_bf16(acc2, dK + (a >> 4), dK + (b5 >> 4), id2, 1u);
                            umma_bf16(acc2 + (uint32_t)C::NI2, dK + (a >> 4), dK + (a >> 4), id2, acc);
                        } else {
                            umma_bf16(acc2, dK + (a >> 4), dK + (a >> 4), id2, acc);
                        }
                    }
                }
                __syncwarp();
            }
            if (lead) {
                // on completion the digit buffer is free again
                umma_commit(&jempty[b]);
                if (C::B2 > 0 && last)
                    umma_commit(&accfull[2 * set + 1]);
            }
            __syncwarp();
        }
        if (lead)
            umma_commit(&g_done);
        __syncwarp();
        // tensor memory is released only after every product has finished
        if (!mbar_wait(&g_done, 0))
            ok = false;
        if (!ok)
            flags |= FLAG_TIMEOUT;
    } else if (warp < kNFirstCons) {
        // ---- drain: lane quarter q, rows m = 32 q + lane, columns half h ----
        // Row m holds row p = m % R of digit m / R of each MMA's A operand;
        // block t of an accumulator is columns t R ... of it. Blocks whose
        // transpose is among the products too count half (T/2): t < S1 of the
        // first, the A digits' own of the second (its last two when there are four).
        const int q = warp & 3, h = (warp - kNFirstDrain) >> 2, m = q * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
        constexpr int HC = NW / 2;  // packed column pairs per thread and block (NW columns)
        constexpr int CH = NW <= 24 ? NW : 16;  // columns read at a time
        const f2 HALF = pk2(0.5f, 0.5f);
        // B2 = 1: D_44 counts half, D_54 (rows of the second A digit) in full
        const float w54 = m < R ? 0.5f : 1.0f;
        const f2 W54 = pk2(w54, w54);
        // (wh, wl): the first accumulator's blocks; w2: the second's, below 2^-28 of the
        // leading one (2^-48 for B2 = 1), whose FP32 roundings are below 2^-52 of it.
        // Added to (wh, wl) they would fall below its last bit, one-sidedly.
        f2 wh[HC], wl[HC], w2[C::B2 > 0 ? HC : 1];
#pragma unroll
        for (int c = 0; c < HC; ++c)
            wh[c] = wl[c] = 0ull;
#pragma unroll
        for (int c = 0; c < (C::B2 > 0 ? HC : 1); ++c)
            w2[c] = 0ull;
        const int n_periods = (n_my + kNPeriod - 1) / kNPeriod;
        bool ok = true;
        for (int P = 0; P < n_periods && ok; ++P) {
            const int set = P % NACC;
#pragma unroll
            for (int half = 0; half < (C::B2 > 0 ? 2 : 1); ++half) {
                if (!mbar_wait(&accfull[2 * set + half], (uint32_t)(P / NACC) & 1)) {
                    flags |= FLAG_TIMEOUT;
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t acc = tmem + lane_addr + (uint32_t)set * (C::N1 + C::N2) +
                                     (half ? (uint32_t)C::N1 : 0u) + (uint32_t)(h * NW);
                const int n_blocks = half ? C::B2 : C::B1;
#pragma unroll
                for (int t = 0; t < n_blocks; ++t) {
#pragma unroll
                    for (int c0 = 0; c0 < NW; c0 += CH) {
                        uint32_t v[CH];
                        tmem_row_half<CH>(acc + (uint32_t)(t * R + c0), v);
                        tmem_ld_wait();
                        if (t == n_blocks - 1 && c0 + CH == NW) {
                            // every column is in registers: the accumulator may be reused
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0)
                                mbar_arrive(&accempty[2 * set + half]);
                        }
#pragma unroll
                        for (int i = 0; i < CH / 2; ++i) {
                            const int c = c0 / 2 + i;
                            const f2 x = pk2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
                            if (half == 0)
                                two_sum2(wh[c], wl[c], t < S1 ? mul2(x, HALF) : x);
                            else if (C::B2 == 1)
                                w2[c] = fma2(x, W54, w2[c]);
                            else
                                w2[c] = t < 2 ? add2(w2[c], x) : fma2(x, HALF, w2[c]);
                        }
                    }
                }
            }
        }
        // ---- this CTA's share of M -----------------------------------------
        // W goes through shared memory (the digit buffers are free once the
        // last period is drained: every MMA has completed); then G[p][q] =
        // sum over the digit rows d < S1 of W[dR + p][q] + W[dR + q][p].
        double *Ws = reinterpret_cast<double *>(base);
        if (m < S1 * R) {
#pragma unroll
            for (int c = 0; c < HC; ++c) {
                float a0, a1, b0, b1;
                upk2(wh[c], a0, a1);
                upk2(wl[c], b0, b1);
                double x0 = (double)a0 + (double)b0, x1 = (double)a1 + (double)b1;
                if (C::B2 > 0 && m < 2 * R) {
                    float d0, d1;
                    upk2(w2[C::B2 > 0 ? c : 0], d0, d1);
                    x0 += (double)d0;
                    x1 += (double)d1;
                }
                Ws[m * R + h * NW + 2 * c] = x0;
                Ws[m * R + h * NW + 2 * c + 1] = x1;
            }
        }
        asm volatile("bar.sync 1, %0;" ::"r"(kNDrain * 32) : "memory");
        // entries e of the upper triangle (a <= b) of the local waves, real and imaginary parts
        const int nl = blocks.local(), E = nl * (nl + 1) / 2;
        for (int ec = (warp - kNFirstDrain) * 32 + lane; ec < 2 * E; ec += kNDrain * 32) {
            const int e = ec >> 1, comp = ec & 1;
            int a = 0, o = e;
            while (o >= nl - a) {
                o -= nl - a;
                ++a;
            }
            const int b = a + o;
            auto G = [&](int p, int r) {
                double v = 0.0;
#pragma unroll
                for (int d = 0; d < S1; ++d)
                    v += Ws[(d * R + p) * R + r] + Ws[(d * R + r) * R + p];
                return v;
            };
            const double v = comp == 0 ? G(2 * a, 2 * b) + G(2 * a + 1, 2 * b + 1)
                                       : G(2 * a, 2 * b + 1) - G(2 * a + 1, 2 * b);
            part[(size_t)ec * gridDim.x + blockIdx.x] = v;
        }
    } else {
        // ---- consumers: group g takes tiles j = g, g + GROUPS, ... ----------
        // A half warp holds one row of the tile (four events a lane); warp w of
        // the group takes row pairs w, w + WPG, ...
        const int cw = warp - kNFirstCons, g = cw / C::WPG, wg = cw % C::WPG;
        const unsigned zero = (unsigned)blocks.n_box >> 4;  // what the compiler does not know
        const int half = lane >> 4, l16 = lane & 15;
        for (int j = g; j < n_my; j += C::GROUPS) {
            const int st = j % STAGES, b = j % NBUF, k = j / NBUF;
            if (!mbar_wait(&full[st], (uint32_t)(j / STAGES) & 1)) {
                flags |= FLAG_TIMEOUT;
                break;
            }
            const float *T = stages + (size_t)st * (C::STAGE_BYTES / 4) + 4 * l16;
            float4 xs[C::ITERS];
            unsigned seen = 0;
#pragma unroll
            for (int it = 0; it < C::ITERS; ++it) {
                const int rp = wg + it * C::WPG;
                if (rp < NW) {
                    xs[it] = *reinterpret_cast<const float4 *>(T + (2 * rp + half) * kNTE);
                    seen |= __float_as_uint(xs[it].x);
                }
            }
            // Once the amplitudes are in registers the stage may be refilled. The
            // arrival's address depends on every load's result: loads that were only issued
            // can be overtaken by it, since the products' operand reads, which can fill shared
            // memory's bandwidth, hold them up for longer than a refill takes (single rows of a
            // tile then came from the tile after: seen with three products of 128 columns
            // a step).
            __syncwarp();
            if (lane == 0)
                mbar_arrive(empty + st + (seen & zero));
            // the buffer is free once the products of its previous tile are done
            if (k > 0 && !mbar_wait(&jempty[b], (uint32_t)(k - 1) & 1)) {
                flags |= FLAG_TIMEOUT;
                break;
            }
            const uint32_t jb = jbase + (uint32_t)b * C::JBYTES;
#pragma unroll
            for (int it = 0; it < C::ITERS; ++it) {
                const int rp = wg + it * C::WPG;
                if (rp < NW) {
                    const int p = 2 * rp + half;
                    const float scale = s_scale[p], sig = 1.5f * 32768.f;
                    const f2 S0 = pk2(sig, sig), SC = pk2(scale, scale);
                    f2 z0 = mul2(pk2(xs[it].x, xs[it].y), SC), z1 = mul2(pk2(xs[it].z, xs[it].w), SC);
                    const uint32_t dst = jb + sw128(p, (uint32_t)l16 * 8);
                    float step = 1.0f;
#pragma unroll
                    for (int d = 0; d < kNDigits; ++d) {
                        // z rounded to a multiple of 2^-8(d+1): z + S - S with S = S0 2^-8d
                        // (the products by powers of two are exact), and the exact
                        // remainder
                        const f2 up = pk2(step, step), dn = pk2(-step, -step);
                        const f2 t0 = fma2(S0, dn, fma2(S0, up, z0));
                        const f2 t1 = fma2(S0, dn, fma2(S0, up, z1));
                        z0 = sub2(z0, t0);
                        z1 = sub2(z1, t1);
                        float a0, a1, a2, a3;
                        upk2(t0, a0, a1);
                        upk2(t1, a2, a3);
                        st_shared_v2(dst + (uint32_t)(d * R) * 128u, to_bf16x2(a0, a1),
                                     to_bf16x2(a2, a3));
                        step *= 0x1p-8f;
                    }
                    if constexpr (C::REST) {  // what is left, to 8 bits of its own
                        float a0, a1, a2, a3;
                        upk2(z0, a0, a1);
                        upk2(z1, a2, a3);
                        st_shared_v2(dst + (uint32_t)(kNDigits * R) * 128u, to_bf16x2(a0, a1),
                                     to_bf16x2(a2, a3));
                    }
                }
            }
            // generic-proxy writes become visible to the tensor core, then signal
            fence_async_smem();
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&jfull[b]);
        }
    }
    if (flags)
        atomicOr(&s_flags, flags);
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && s_flags)
        atomicOr(status, s_flags);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, kNTmemCols);
    }
}

// M from the CTAs' shares: one warp per (entry, part) of the launch's upper
// triangle; lane k adds CTAs k, k + 32, ... (all loads issued first), then a
// fixed shuffle tree; scaled back by the two waves' 2^r, divided by N_gen, written
// to (a, b) and conjugated to (b, a), the diagonal's imaginary part zero. With a
// timeout flagged, M is NaN.
__global__ void norm_tc_finalize(const double *__restrict__ part, int grid, int N,
                                 NormBlocks blocks, const float *__restrict__ amax, double n_gen,
                                 const int *status, double *__restrict__ M)
{
    const int ec = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int nl = blocks.local(), E = nl * (nl + 1) / 2;
    if (ec >= 2 * E)
        return;
    const int e = ec >> 1, comp = ec & 1;
    int la = 0, o = e;
    while (o >= nl - la) {
        o -= nl - la;
        ++la;
    }
    const int a = blocks.global(la), b = blocks.global(la + o);
    if (a >= N || b >= N)
        return;
    const double *pe = part + (size_t)ec * grid;
    double x[kNFinMaxRounds];
#pragma unroll
    for (int k = 0; k < kNFinMaxRounds; ++k) {
        const int g = lane + 32 * k;
        x[k] = g < grid ? pe[g] : 0.0;
    }
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < kNFinMaxRounds; ++k)
        v += x[k];
    v = warp_sum(v);
    if (lane == 0) {
        double r = ldexp(v, wave_exponent(amax[a]) + wave_exponent(amax[b])) / n_gen;
        if (*status & FLAG_TIMEOUT)
            r = NAN;
        if (a == b) {
            M[2 * (a * N + a) + comp] = comp ? 0.0 : r;
        } else {
            M[2 * (a * N + b) + comp] = r;
            M[2 * (b * N + a) + comp] = comp ? -r : r;
        }
    }
}

template <int NW>
cudaError_t norm_tc_nw(const CUtensorMap *map, const Planes &mc, const NormBlocks &blocks,
                       const float *amax, double n_gen, double *part, int grid, int *status,
                       double *M, cudaStream_t s)
{
    using C = NormTcCfg<NW>;
    const int n_tiles = (int)((mc.n + kNTE - 1) / kNTE);
    if (grid > n_tiles)
        grid = n_tiles;
    if (grid > 32 * kNFinMaxRounds)
        grid = 32 * kNFinMaxRounds;
    cudaError_t e = cudaFuncSetAttribute(norm_tc_kernel<NW>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (e != cudaSuccess)
        return e;
    norm_tc_kernel<NW><<<grid, kNThreads, C::SMEM, s>>>(*map, amax, mc.n_waves, blocks, n_tiles,
                                                        part, status);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    const int E2 = blocks.local() * (blocks.local() + 1);
    norm_tc_finalize<<<(E2 + 7) / 8, 256, 0, s>>>(part, grid, mc.n_waves, blocks, amax, n_gen, status,
                                                  M);
    return cudaGetLastError();
}

// waves per block: all of them in one launch, or a third
int norm_tc_block(int n_waves) { return n_waves <= kNMaxOnePass ? n_waves : (n_waves + 2) / 3; }

cudaError_t norm_tc_pass(const CUtensorMap *map, const Planes &mc, const NormBlocks &blocks,
                         const float *amax, double n_gen, double *part, int grid, int *status,
                         double *M, cudaStream_t s)
{
    const int n = blocks.local();
    if (n <= 4)
        return norm_tc_nw<4>(map, mc, blocks, amax, n_gen, part, grid, status, M, s);
    if (n <= 8)
        return norm_tc_nw<8>(map, mc, blocks, amax, n_gen, part, grid, status, M, s);
    if (n <= 12)
        return norm_tc_nw<12>(map, mc, blocks, amax, n_gen, part, grid, status, M, s);
    if (n <= 16)
        return norm_tc_nw<16>(map, mc, blocks, amax, n_gen, part, grid, status, M, s);
    if (n <= 20)
        return norm_tc_nw<20>(map, mc, blocks, amax, n_gen, part, grid, status, M, s);
    if (n <= 24)
        return norm_tc_nw<24>(map, mc, blocks, amax, n_gen, part, grid, status, M, s);
    return norm_tc_nw<32>(map, mc, blocks, amax, n_gen, part, grid, status, M, s);
}

}  // namespace

bool norm_tc_available(int n_waves) { return n_waves >= 1 && n_waves <= kMaxWaves; }

int norm_tc_box_events() { return kNTE; }

int norm_tc_box_rows(int n_waves) { return 2 * norm_tc_block(n_waves); }

bool norm_tc_scale_ok(float amax)
{
    // above, the FP64 kernel, whose error is the smaller one (the digits would serve up
    // to 2^125: beyond, and below 2^-124, 2^-r is no normal float); far below, where
    // amplitudes become subnormal, their own last bits limit the digits
    return amax == 0.f || (amax >= 0x1p-100f && amax < 0x1p53f);
}

bool norm_tc_checks_spread(int n_waves) { return n_waves > 20; }

bool norm_tc_spread_ok(int n_waves, const float *amax, int64_t n, double n_gen, const double *diag)
{
    // Beyond 20 waves the standard is the FP64 kernel's error. The dropped squares of
    // the fifth digits add up to k^2 2^-67.6 of M_aa, k = 2^r_a / rms of the wave: k is
    // at most 47 for widths of 0.05 GeV (error 3e-16 measured), 120 for 0.01 GeV
    // (2e-15; FP64 1e-15), 900 for 1e-4 GeV (5e-14).
    for (int a = 0; a < n_waves; ++a)
        if (amax[a] > 0.f &&
            !(ldexp((double)n / n_gen, 2 * wave_exponent(amax[a])) <= 0x1p14 * diag[a]))
            return false;
    return true;
}

size_t norm_tc_partials_doubles(int n_waves, int grid)
{
    const int n = n_waves <= kNMaxOnePass ? n_waves : 2 * norm_tc_block(n_waves);
    return (size_t)grid * n * (n + 1);
}

cudaError_t launch_build_norm_tc(const CUtensorMap *map, const Planes &mc, const float *amax,
                                 double n_gen, double *partials, int grid, int *status, double *M,
                                 cudaStream_t s)
{
    if (mc.n < 1 || !norm_tc_available(mc.n_waves))
        return cudaErrorInvalidValue;
    const int blk = norm_tc_block(mc.n_waves);
    if (blk == mc.n_waves)
        return norm_tc_pass(map, mc, NormBlocks{1, blk, {0, 0}}, amax, n_gen, partials, grid, status,
                            M, s);
    for (int i = 0; i < 3; ++i)
        for (int k = i + 1; k < 3; ++k) {
            const cudaError_t e = norm_tc_pass(map, mc, NormBlocks{2, blk, {i * blk, k * blk}}, amax,
                                               n_gen, partials, grid, status, M, s);
            if (e != cudaSuccess)
                return e;
        }
    return cudaSuccess;
}

}  // namespace pwa
