// vacf_noalloc.cu -- a velocity-autocorrelation entry point that allocates no
// device memory.
//
// Who needs it: callers that cannot call cudaMalloc at the point where they
// want the correlation -- for example code running inside a memory pool or
// arena they do not control, a host process that has handed all device memory
// to another framework's caching allocator, or a real-time loop that must not
// risk an allocation's implicit synchronisation or failure.  They pass their
// own sample and output buffers; the only scratch this routine needs (the
// per-chunk partial sums of the correlator) lives in a fixed array compiled
// into the library, which every GPU that loads the library keeps until the
// process exits.
//
// The correlation itself is the same blocked all-origin estimator as the
// library's stateful VACF (vacf_kernels.cu): for every block of up to 64 new
// samples t and every lag k <= max_lag it adds V(t).V(t - k).  Products are
// FP32; each lane sums the products of one component over one block (at most
// 64 terms) in FP32 and adds that to an FP64 accumulator, and everything
// above that (components, chunks, blocks) is summed in FP64.  Here the
// samples are the caller's whole trajectory instead of the library's ring.
//
// k_corr_noalloc: a CTA owns 128 lags and a run of work units, a unit being 64
// samples x 64 components.  The units of a lag tile (blocks inner, component
// groups outer) are dealt in equal runs to the CTAs of that tile, as many as
// fill the chip and the scratch holds, so one launch covers the trajectory
// whatever its shape.  Along a run the window of 192 samples slides by 64: one
// new window block and the 64 new samples per unit are copied (cp.async) while
// the previous unit computes, into a ring of four window blocks and two
// sample buffers.  A lane holds two components and 16 lags as packed FP32
// pairs (fma.rn.f32x2: the two components' FMAs, each rounded as fmaf), and
// the 16-sample window groups stay in registers from one group to the next,
// so 256 packed FMAs take 32 shared loads.  Bound: the packed FMAs with their
// shared loads (0.26 of the 0.39 ms below with the FP64 additions left out)
// and then the FP64 pipe (2 lanes per clock and SM), which takes one addition
// per lag, component and block; the widening to FP64 is done on the bits.
// Spreading those additions over the next unit's FMAs (twice the registers,
// one CTA per SM) measured 0.38 ms, and 0.052 against 0.036 ms with 1000
// samples x 300 components: not kept.
// Measured with 4096 samples x 1536 components, lags to 1000: 14.3 -> 0.39 ms
// (before: one launch of 16 CTAs per 64 samples).
#include <cuda_runtime.h>

#include <mutex>

#include "lbp_internal.cuh"

namespace {

constexpr int NB = 64;       // samples per correlation block
constexpr int NKT = 128;     // lags per CTA
constexpr int NLW = 16;      // lags per warp
constexpr int NJ = 64;       // components per work unit (two per lane)
constexpr int NJCH = 1024;   // components per chunk of the sizes the call takes
constexpr int NT = 256;      // threads
constexpr int NWB = 4;       // window blocks in the ring
constexpr int MAX_RUNS = 512;  // CTAs per lag tile
constexpr int SMEM = (2 + NWB) * NB * NJ * (int)sizeof(float);  // two sample buffers and the ring

// Scratch: partial sums [runs][max_lag + 1], 4 MiB.
constexpr long long SCRATCH_DOUBLES = 524288;
static __device__ __align__(256) double g_vacf_scratch[SCRATCH_DOUBLES];

// Address of g_vacf_scratch and the SM count per device, looked up once per device.
constexpr int MAX_DEVICES = 64;
std::mutex g_mu;
double *g_scratch_ptr[MAX_DEVICES] = {};
int g_sms[MAX_DEVICES] = {};

using Pair = unsigned long long;  // two FP32 values
__device__ __forceinline__ Pair fma2(Pair a, Pair b, Pair c) {
    Pair d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// One block of 64 samples x 64 components (samples [64 q, 64 q + 64), zeros
// outside the trajectory) to shared memory, asynchronously.  VEC: 16 bytes at
// a time (rows 16-byte aligned), else 4.
template <bool VEC>
__device__ __forceinline__ void load_block(float *dst, const float *__restrict__ samples, long long T, int ncomp,
                                           long long q, int j0) {
    constexpr int W = VEC ? 4 : 1, PER_ROW = NJ / W;
    const unsigned base = (unsigned)__cvta_generic_to_shared(dst);
#pragma unroll
    for (int e = threadIdx.x; e < NB * PER_ROW; e += NT) {
        const int row = e / PER_ROW, col = (e - row * PER_ROW) * W;
        const long long s = q * NB + row;
        const bool in = s >= 0 && s < T && j0 + col < ncomp;
        const float *src = in ? samples + s * ncomp + j0 + col : samples;
        const unsigned d = base + (unsigned)(row * NJ + col) * 4u;
        if (VEC)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(in ? 16 : 0) : "memory");
        else
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(in ? 4 : 0) : "memory");
    }
}

template <bool VEC>
__global__ void __launch_bounds__(NT, 2) k_corr_noalloc(const float *__restrict__ samples, long long T, int ncomp,
                                                        int K, int nblk, int nsub, double *part) {
    extern __shared__ __align__(16) float sm[];
    float *sA = sm, *sW = sm + 2 * NB * NJ;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k0 = blockIdx.x * NKT, kb = k0 / NB;
    // blocks before kb end before the tile's first lag: no pairs
    const int nb = nblk - kb;
    const long long units = nb > 0 ? (long long)nb * nsub : 0;
    const long long u0 = units * blockIdx.y / gridDim.y, u1 = units * (blockIdx.y + 1) / gridDim.y;
    double dacc[NLW];
#pragma unroll
    for (int m = 0; m < NLW; ++m) dacc[m] = 0.0;
    int sub = nb > 0 ? (int)(u0 / nb) : 0, b = nb > 0 ? kb + (int)(u0 - (long long)sub * nb) : 0;
    // the sample buffer and the three window blocks of a unit whose predecessor
    // has not loaded them
    auto load_all = [&](int buf, int bb, int ss) {
        load_block<VEC>(sA + buf * NB * NJ, samples, T, ncomp, bb, ss * NJ);
        for (int w = 0; w < 3; ++w) {
            const int q = bb - kb - 2 + w;
            load_block<VEC>(sW + (q & (NWB - 1)) * NB * NJ, samples, T, ncomp, q, ss * NJ);
        }
    };
    if (u0 < u1) load_all(0, b, sub);
    int buf = 0;
    bool fresh = true;
    Pair wp[NLW];  // the 16 window samples before the current group
    for (long long u = u0; u < u1; ++u) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        const bool more = u + 1 < u1, wrap = b + 1 == nblk;
        if (more && !wrap) {
            load_block<VEC>(sA + (buf ^ 1) * NB * NJ, samples, T, ncomp, b + 1, sub * NJ);
            const int q = b + 1 - kb;
            load_block<VEC>(sW + (q & (NWB - 1)) * NB * NJ, samples, T, ncomp, q, sub * NJ);
        }
        // row r of the 192-row window holds sample 64 (b - kb - 2) + r; sample t
        // of the block and lag k0 + 16 warp + m meet at r = t + 128 - 16 warp - m
        const int qlo = b - kb - 2;
        const int g0 = NKT - NLW * warp;
        auto group = [&](int r0) {  // this lane's pair of the group of 16 rows at r0
            const int q = qlo + (r0 >> 6);
            return reinterpret_cast<const Pair *>(sW + ((q & (NWB - 1)) * NB + (r0 & 63)) * NJ) + lane;
        };
        if (fresh) {
            const Pair *w = group(g0 - NLW);
#pragma unroll
            for (int i = 0; i < NLW; ++i) wp[i] = w[i * (NJ / 2)];
        }
        Pair acc[NLW];  // one component's products over this block only
#pragma unroll
        for (int m = 0; m < NLW; ++m) acc[m] = 0ull;
        const Pair *pa = reinterpret_cast<const Pair *>(sA + buf * NB * NJ) + lane;
#pragma unroll
        for (int tc = 0; tc < NB; tc += NLW) {
            const Pair *w = group(g0 + tc);
            Pair wc[NLW];
#pragma unroll
            for (int i = 0; i < NLW; ++i) wc[i] = w[i * (NJ / 2)];
#pragma unroll
            for (int i = 0; i < NLW; ++i) {
                const Pair a = pa[(tc + i) * (NJ / 2)];
#pragma unroll
                for (int m = 0; m < NLW; ++m) acc[m] = fma2(a, i >= m ? wc[i - m] : wp[NLW + i - m], acc[m]);
            }
#pragma unroll
            for (int i = 0; i < NLW; ++i) wp[i] = wc[i];
        }
#pragma unroll
        for (int m = 0; m < NLW; ++m) {
            dacc[m] += lbp::widen_f32(__uint_as_float((unsigned)acc[m]));
            dacc[m] += lbp::widen_f32(__uint_as_float((unsigned)(acc[m] >> 32)));
        }
        buf ^= 1;
        fresh = wrap;
        if (++b == nblk) {
            b = kb;
            ++sub;
            if (more) {
                __syncthreads();  // the window blocks are still being read
                load_all(buf, b, sub);
            }
        }
    }
#pragma unroll
    for (int m = 0; m < NLW; ++m) {
        double v = dacc[m];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        const int k = k0 + NLW * warp + m;
        if (lane == 0 && k <= K) part[(long long)blockIdx.y * (K + 1) + k] = v;
    }
}

// one warp per lag: the runs' partial sums in a fixed order, and the pair counts
__global__ void __launch_bounds__(NT) k_reduce_noalloc(const double *part, int runs, int K, long long T, int npairs,
                                                       double *csum, long long *counts) {
    const int k = (int)((blockIdx.x * (long long)NT + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (k > K) return;
    double s = 0.0;
    for (int c = lane; c < runs; c += 32) s += part[(long long)c * (K + 1) + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
        csum[k] = s;
        counts[k] = T > k ? (long long)npairs * (T - k) : 0;
    }
}

}  // namespace

// sets the thread's lbp_last_error message (lbp_api.cu)
lbp_status lbp_set_error_for_noalloc(lbp_status st, const char *msg);

// One-time set-up per device happens inside the first call on that device
// (cudaGetSymbolAddress with the device current): make that first call
// before any CUDA graph capture that includes this routine.  The address is
// kept for the life of the process, so the routine must not be used on a
// device after cudaDeviceReset has torn down its context.
extern "C" lbp_status lbp_vacf_correlate_noalloc(const float *samples, int64_t T, int ncomp,
                                                 int max_lag, int npairs, double *csum,
                                                 int64_t *counts, void *stream) {
    if (T < 0 || ncomp < 1 || max_lag < 0 || npairs < 0)
        return lbp_set_error_for_noalloc(LBP_EINVAL,
                                         "lbp_vacf_correlate_noalloc: need T >= 0, ncomp >= 1, max_lag >= 0, npairs >= 0");
    if (!csum || !counts || (T > 0 && !samples))
        return lbp_set_error_for_noalloc(LBP_EINVAL, "lbp_vacf_correlate_noalloc: null pointer");
    const long long nchunks = ((long long)ncomp + NJCH - 1) / NJCH;
    // the limits of the interface, from a layout with a scratch row per chunk and a
    // grid row each.  Today's needs max_lag below the scratch size, and with it the
    // grid sizes below bounded, which follows: both factors are at least 1
    if (nchunks * ((long long)max_lag + 1) > SCRATCH_DOUBLES)
        return lbp_set_error_for_noalloc(
            LBP_EINVAL,
            "lbp_vacf_correlate_noalloc: ceil(ncomp / 1024) * (max_lag + 1) exceeds the 524288-entry scratch");
    if (nchunks > 65535)
        return lbp_set_error_for_noalloc(LBP_EINVAL,
                                         "lbp_vacf_correlate_noalloc: ncomp > 65535 * 1024 (one grid row per chunk)");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return lbp_set_error_for_noalloc(LBP_ECUDA, cudaGetErrorString(e));
    if (dev < 0 || dev >= MAX_DEVICES)
        return lbp_set_error_for_noalloc(LBP_EINVAL, "lbp_vacf_correlate_noalloc: device index >= 64");
    double *part = nullptr;
    int sms = 0;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (!g_scratch_ptr[dev]) {
            void *p = nullptr;
            e = cudaGetSymbolAddress(&p, g_vacf_scratch);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g_sms[dev], cudaDevAttrMultiProcessorCount, dev);
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(k_corr_noalloc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(k_corr_noalloc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
            if (e != cudaSuccess)
                return lbp_set_error_for_noalloc(LBP_ECUDA, cudaGetErrorString(e));
            g_scratch_ptr[dev] = static_cast<double *>(p);
        }
        part = g_scratch_ptr[dev];
        sms = g_sms[dev];
    }
    cudaStream_t st = (cudaStream_t)stream;
    const long long nblk = (T + NB - 1) / NB, nsub = ((long long)ncomp + NJ - 1) / NJ;
    if (nblk > 2147483647ll)
        return lbp_set_error_for_noalloc(LBP_EINVAL, "lbp_vacf_correlate_noalloc: T > 2^37");
    int runs = 0;
    if (T > 0) {
        // about four CTAs per SM over all lag tiles (two are resident), so that
        // the runs of the later tiles, shorter by the blocks before their first
        // lag, leave no SM idle for long
        const int tiles = (max_lag + NKT) / NKT;
        long long n = (4ll * sms + tiles - 1) / tiles;
        if (n > SCRATCH_DOUBLES / ((long long)max_lag + 1)) n = SCRATCH_DOUBLES / ((long long)max_lag + 1);
        if (n > nblk * nsub) n = nblk * nsub;
        runs = (int)(n > MAX_RUNS ? MAX_RUNS : n);
        const dim3 grid((unsigned)tiles, (unsigned)runs);
        const bool vec = ncomp % 4 == 0 && reinterpret_cast<uintptr_t>(samples) % 16 == 0;
        auto kern = vec ? k_corr_noalloc<true> : k_corr_noalloc<false>;
        kern<<<grid, NT, SMEM, st>>>(samples, T, ncomp, max_lag, (int)nblk, (int)nsub, part);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        const unsigned blocks = (unsigned)((32ll * ((long long)max_lag + 1) + NT - 1) / NT);
        k_reduce_noalloc<<<blocks, NT, 0, st>>>(part, runs, max_lag, T, npairs, csum, (long long *)counts);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return lbp_set_error_for_noalloc(LBP_ECUDA, cudaGetErrorString(e));
    return LBP_OK;
}
