// Loading the sample into the device store (Sec. 2: amplitudes are computed
// once per event and kept; Sec. 5, Table 1: "Start-up" and "Lookup table
// creation").
//
//  pack:  event-major interleaved complex [n][N] (float or double pairs) ->
//         structure-of-arrays planes, plane 2a = Re A_a, plane 2a+1 = Im A_a,
//         events contiguous. Doubles are rounded to nearest float.
//  table: planes -> per-event Hermitian table of Sec. 2, coefficient-major
//         t[p][i]: p < N holds |A_a|^2, then for each pair a < b in
//         row-major order two planes Re(A_a conj A_b), Im(A_a conj A_b).
#include <cuda_bf16.h>

#include <algorithm>

#include "pwa_internal.cuh"

namespace pwa {

namespace {

constexpr int kPackWarps = 8;
constexpr int kPackUnroll = 8;  // loads in flight per lane
constexpr int kPackMaxWaves = 2 * kMaxWaves;  // an incoherent sample's waves times components

constexpr size_t pack_smem(int n_waves, int n_max)
{
    return ((size_t)kPackWarps * 2 * n_waves * 33 + n_max) * sizeof(float);
}
static_assert(pack_smem(kPackMaxWaves, kPackMaxWaves) <= 227 * 1024, "shared memory");

// One warp takes 32 events: their rows are contiguous in the source, so they
// are read 32 elements at a time (a load's lanes next to each other, eight
// loads in flight), turned through the warp's own piece of shared memory
// (rows of 33 floats, all real parts before all imaginary ones: neither side
// conflicts) and written as 128-byte pieces of the planes. With amax, the
// largest |Re| + |Im| of each wave (index w mod n_max) is taken on the way, so
// that no second pass over the planes is needed.
//
// Bound by HBM: the bytes are read once and written once. 14M events x 32
// waves in 1.43 ms with the maxima (5.0 TB/s); with a divided index per element,
// 64 events per block and the maxima in a pass of their own 2.03 ms.
template <typename T2>
__global__ void __launch_bounds__(kPackWarps * 32)
    pack_kernel(const T2 *__restrict__ src, int64_t n, int N, float *__restrict__ planes, int64_t pitch,
                float *__restrict__ amax, int n_max)
{
    extern __shared__ float sm[];  // [warps][2N][33], then the block's maxima [n_max]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *my = sm + (size_t)warp * 2 * N * 33;
    unsigned *mx = reinterpret_cast<unsigned *>(sm + (size_t)kPackWarps * 2 * N * 33);
    for (int i = threadIdx.x; amax && i < n_max; i += blockDim.x)
        mx[i] = 0u;
    __syncthreads();
    const int64_t groups = (n + 31) / 32, stride = (int64_t)gridDim.x * kPackWarps;
    // this lane's first element of a group: event e_0, wave w_0; 32 elements on:
    const int w_0 = lane % N, e_0 = lane / N, dw = 32 % N, de = 32 / N;
    for (int64_t g = (int64_t)blockIdx.x * kPackWarps + warp; g < groups; g += stride) {
        const int64_t e0 = g * 32;
        const int cnt = (int)(n - e0 < 32 ? n - e0 : 32), total = cnt * N;
        const T2 *in = src + e0 * N;
        int w = w_0, e = e_0;
        for (int k0 = lane; k0 < total; k0 += 32 * kPackUnroll) {
            T2 v[kPackUnroll];
#pragma unroll
            for (int j = 0; j < kPackUnroll; ++j)
                if (k0 + 32 * j < total)
                    v[j] = __ldcs(in + k0 + 32 * j);
#pragma unroll
            for (int j = 0; j < kPackUnroll; ++j) {
                if (k0 + 32 * j < total) {
                    my[w * 33 + e] = (float)v[j].x;  // round to nearest for doubles
                    my[(N + w) * 33 + e] = (float)v[j].y;
                }
                w += dw;
                e += de;
                if (w >= N) {
                    w -= N;
                    ++e;
                }
            }
        }
        __syncwarp();
        float *out = planes + e0 + lane;
        int slot = 0;
        for (int r = 0; r < N; ++r) {
            const float re = my[r * 33 + lane], im = my[(N + r) * 33 + lane];
            if (lane < cnt) {
                out[(int64_t)(2 * r) * pitch] = re;
                out[(int64_t)(2 * r + 1) * pitch] = im;
            }
            if (amax) {
                const float t = lane < cnt ? fmaxf(0.f, fabsf(re) + fabsf(im)) : 0.f;
                const unsigned u = __reduce_max_sync(0xffffffffu, __float_as_uint(t));
                if (lane == 0 && u > mx[slot])
                    atomicMax(&mx[slot], u);  // non-negative floats order like their bit patterns
                slot = slot + 1 == n_max ? 0 : slot + 1;
            }
        }
        __syncwarp();
    }
    if (amax) {
        __syncthreads();
        for (int i = threadIdx.x; i < n_max; i += blockDim.x)
            if (mx[i])
                atomicMax(reinterpret_cast<int *>(amax + i), (int)mx[i]);
    }
}

template <typename T2>
cudaError_t pack(const void *src, int64_t n, int N, float *planes, int64_t pitch, float *amax,
                 int n_max, int num_sms, cudaStream_t s)
{
    const size_t smem = pack_smem(N, n_max);
    // the same limit at every call: contexts in other threads launch it too
    cudaError_t e = cudaFuncSetAttribute(pack_kernel<T2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)pack_smem(kPackMaxWaves, kPackMaxWaves));
    if (e != cudaSuccess)
        return e;
    // as many blocks as shared memory (and 2048 threads an SM) keeps resident
    const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(8, (224 * 1024) / (smem + 1024)));
    const int64_t need = (n + 32 * kPackWarps - 1) / (32 * kPackWarps);
    const unsigned grid = (unsigned)std::min<int64_t>(need, (int64_t)num_sms * per_sm);
    pack_kernel<T2><<<grid, kPackWarps * 32, smem, s>>>(static_cast<const T2 *>(src), n, N, planes,
                                                        pitch, amax, n_max);
    return cudaGetLastError();
}

// Each entry is the float nearest to its exact value: the products of two
// floats are exact in double and each entry adds two of them, so the double
// result carries one rounding and the final rounding to float is the only
// one that matters. (One-time work; FP64 is acceptable here.)
__global__ void table_kernel(const float *__restrict__ planes, int64_t pitch, int64_t n, int N,
                             float *__restrict__ table, int64_t tpitch)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    for (int w = 0; w < N; ++w) {
        const double ar = planes[(2 * w) * pitch + i], ai = planes[(2 * w + 1) * pitch + i];
        table[w * tpitch + i] = __double2float_rn(ar * ar + ai * ai);
    }
    int p = N;
    for (int x = 0; x < N; ++x) {
        const double xr = planes[(2 * x) * pitch + i], xi = planes[(2 * x + 1) * pitch + i];
        for (int y = x + 1; y < N; ++y) {
            const double yr = planes[(2 * y) * pitch + i], yi = planes[(2 * y + 1) * pitch + i];
            // A_x conj(A_y) = (xr yr + xi yi) + i (xi yr - xr yi)
            table[(int64_t)p * tpitch + i] = __double2float_rn(xr * yr + xi * yi);
            table[(int64_t)(p + 1) * tpitch + i] = __double2float_rn(xi * yr - xr * yi);
            p += 2;
        }
    }
}

// Per-event table of an incoherent sum over L components (planes of L N
// waves, component l of wave a at plane 2 (l N + a)): products of floats are
// exact in double, summed over components in double and rounded once.
__global__ void table_incoh_kernel(const float *__restrict__ planes, int64_t pitch, int64_t n,
                                   int N, int L, float *__restrict__ table, int64_t tpitch)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    auto re = [&](int l, int w) { return (double)planes[(2 * (l * N + w)) * pitch + i]; };
    auto im = [&](int l, int w) { return (double)planes[(2 * (l * N + w) + 1) * pitch + i]; };
    for (int w = 0; w < N; ++w) {
        double d = 0.0;
        for (int l = 0; l < L; ++l)
            d += re(l, w) * re(l, w) + im(l, w) * im(l, w);
        table[w * tpitch + i] = __double2float_rn(d);
    }
    int p = N;
    for (int x = 0; x < N; ++x)
        for (int y = x + 1; y < N; ++y) {
            double tr = 0.0, ti = 0.0;
            for (int l = 0; l < L; ++l) {
                // A_x conj(A_y) = (xr yr + xi yi) + i (xi yr - xr yi)
                tr += re(l, x) * re(l, y) + im(l, x) * im(l, y);
                ti += im(l, x) * re(l, y) - re(l, x) * im(l, y);
            }
            table[(int64_t)p * tpitch + i] = __double2float_rn(tr);
            table[(int64_t)(p + 1) * tpitch + i] = __double2float_rn(ti);
            p += 2;
        }
}

__global__ void amp_max_kernel(const float *__restrict__ planes, int64_t pitch, int64_t n, int N,
                               float *__restrict__ amax)
{
    const int w = blockIdx.y;
    float m = 0.f;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(planes[(2 * w) * pitch + i]) + fabsf(planes[(2 * w + 1) * pitch + i]));
    for (int o = 16; o > 0; o >>= 1)
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0)  // non-negative floats order like their bit patterns
        atomicMax(reinterpret_cast<int *>(amax + w), __float_as_int(m));
}

__global__ void plane_absmax_kernel(const float *__restrict__ planes, int64_t pitch, int64_t n,
                                    float *__restrict__ out)
{
    const int r = blockIdx.y;
    float m = 0.f;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(planes[(int64_t)r * pitch + i]));
    for (int o = 16; o > 0; o >>= 1)
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0)
        atomicMax(reinterpret_cast<int *>(out + r), __float_as_int(m));
}

__global__ void to_float_kernel(const double *__restrict__ src, int64_t n, float *__restrict__ dst)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = __double2float_rn(src[i]);
}

}  // namespace

cudaError_t launch_to_float(const double *src, int64_t n, float *dst, cudaStream_t s)
{
    if (n <= 0)
        return cudaSuccess;
    to_float_kernel<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, s>>>(src, n, dst);
    return cudaGetLastError();
}

cudaError_t launch_plane_absmax(const float *planes, int64_t pitch, int64_t n, int rows, float *out,
                                cudaStream_t s)
{
    if (n <= 0)
        return cudaSuccess;
    dim3 grid((unsigned)std::min<int64_t>((n + 255) / 256, 64), (unsigned)rows);
    plane_absmax_kernel<<<grid, 256, 0, s>>>(planes, pitch, n, out);
    return cudaGetLastError();
}

cudaError_t launch_amp_max(const Planes &amp, float *amax, cudaStream_t s)
{
    if (amp.n <= 0)
        return cudaSuccess;
    dim3 grid((unsigned)std::min<int64_t>((amp.n + 255) / 256, 256), (unsigned)amp.n_waves);
    amp_max_kernel<<<grid, 256, 0, s>>>(amp.ptr, amp.pitch, amp.n, amp.n_waves, amax);
    return cudaGetLastError();
}

cudaError_t launch_pack(const void *src, int dtype, int64_t n, int n_waves, float *planes,
                        int64_t pitch, float *amax, int n_max, int num_sms, cudaStream_t s)
{
    if (n <= 0)
        return cudaSuccess;
    if (n_waves < 1 || n_waves > kPackMaxWaves || n_max < 1 || n_waves % n_max)
        return cudaErrorInvalidValue;
    return dtype == PWA_C64
               ? pack<float2>(src, n, n_waves, planes, pitch, amax, n_max, num_sms, s)
               : pack<double2>(src, n, n_waves, planes, pitch, amax, n_max, num_sms, s);
}

cudaError_t launch_table_build(const Planes &amp, float *table, int64_t table_pitch, cudaStream_t s)
{
    if (amp.n <= 0)
        return cudaSuccess;
    const int64_t blocks = (amp.n + 127) / 128;
    table_kernel<<<(unsigned)blocks, 128, 0, s>>>(amp.ptr, amp.pitch, amp.n, amp.n_waves, table,
                                                   table_pitch);
    return cudaGetLastError();
}

cudaError_t launch_table_build_incoh(const Planes &amp, int n_lambda, float *table,
                                     int64_t table_pitch, cudaStream_t s)
{
    if (amp.n <= 0)
        return cudaSuccess;
    if (n_lambda < 1 || amp.n_waves % n_lambda)
        return cudaErrorInvalidValue;
    const int64_t blocks = (amp.n + 127) / 128;
    table_incoh_kernel<<<(unsigned)blocks, 128, 0, s>>>(amp.ptr, amp.pitch, amp.n,
                                                        amp.n_waves / n_lambda, n_lambda, table,
                                                        table_pitch);
    return cudaGetLastError();
}

}  // namespace pwa
