// Standardised scores (Eq. 7 for iHS, Eq. 11 for XPEHH): each unstandardised
// score is centred and scaled by the mean and standard deviation of its
// frequency bin, over all markers passed in (the caller's genome).
//
// Deterministic reduction, two forms.  Up to kNormPrivMaxBins bins: CTA s reads
// segment s of the markers once; each of its threads adds its markers (thread
// stride) into its own per-bin accumulators in shared memory, then one thread
// per bin adds the threads' values (from thread b on, so that the threads read
// distinct banks), and the CTA that finishes last adds the segments (first the
// last CTA of each dozen those of its dozen) and, for a whole standardisation,
// makes the bin's mean or SD: three launches (one kernel per step took seven, and
// one thread per bin added 304 segments one after the other; 1M scores, 100 bins:
// 0.142 ms, now 0.078).  More bins: CTA (b, s) sums bin b over segment s (thread
// stride, then a fixed tree), and a second launch adds the segments.  FP64
// additions are slow here (two lanes per SM cycle, some hundred cycles for a
// dependent one), so every sum is short or runs in several chains.  Every order
// is fixed (the segments' number too, whatever the GPU), so the results are the
// same whichever CTA is last.  Two passes: the mean, then the sum of squared
// deviations about it (no cancellation of E[x^2] - E[x]^2).
#include <limits.h>
#include <math.h>

#include "../../include/selscan.h"
#include "internal.h"

namespace selscan {

namespace {

constexpr int kNormThreads = 256;
constexpr int kNormSegments = 16;           // per-bin form: segments per bin
constexpr int kNormPrivThreads = 128;       // private-accumulator form
constexpr int kNormPrivMaxBins = 128;       // its accumulators: 128 x 128 x 12 B = 192 KB
constexpr int kNormPrivSegments = 152;
constexpr int kNormDozen = 12;              // segments added by the last CTA among their own
constexpr int kNormDozens = (kNormPrivSegments + kNormDozen - 1) / kNormDozen;
constexpr int kNormMaxSegments = kNormPrivSegments + kNormDozens;    // parts per bin in the workspace
constexpr int kNormCounters = kNormDozens + 1;                       // per pass

__device__ __forceinline__ int bin_of(int32_t n1, int n, int nbins)
{
    // derived-allele frequency n1 / n in nbins equal bins, decided in integers
    if (nbins == 1) return 0;
    long long b = ((long long)n1 * nbins) / n;
    return b >= nbins ? nbins - 1 : (b < 0 ? 0 : (int)b);
}

template <typename T>
__device__ __forceinline__ T block_sum(T v, T *red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    T t = 0;
    if (threadIdx.x == 0)
        for (int w = 0; w < kNormThreads / 32; ++w) t += red[w];
    __syncthreads();
    return t;                       // valid in thread 0
}

// What a pass leaves per bin: the totals, and for a whole standardisation the
// statistic made from them (mean after pass 0, sample SD after pass 1).
struct BinOut {
    long long *count;
    double *sum, *mean, *sd;
    int finish;
    unsigned *done;                 // counters of the pass, zero: CTAs (dozens) done, then per dozen
};

__device__ __forceinline__ void finish_bin(int pass, long long c, double s, double *mean, double *sd)
{
    if (pass == 0) *mean = c > 0 ? s / (double)c : __longlong_as_double(0x7ff8000000000000ll);
    else *sd = c > 1 ? sqrt(s / (double)(c - 1)) : __longlong_as_double(0x7ff8000000000000ll);
}

// True in the CTA that is the last of `of` to get here; what the others wrote
// before is then visible to it.  Every thread of the CTA calls it.
__device__ __forceinline__ bool last_of(unsigned *done, unsigned of)
{
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(done, 1u) == of - 1u;
    __syncthreads();
    const bool r = last;
    if (r) __threadfence();
    return r;
}

// Sum of the parts [q0, q1) (at most 16) of bin b, part q at q * nbins + b.
__device__ __forceinline__ void sum_parts(int nbins, int pass, int b, int q0, int q1, const double *part_sum,
                                          const long long *part_cnt, double &s, long long &c)
{
    constexpr int U = 16;
    double v[U];
    long long k[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const bool on = q0 + u < q1;
        v[u] = on ? __ldcg(part_sum + (size_t)(q0 + u) * nbins + b) : 0.0;
        k[u] = on && pass == 0 ? __ldcg(part_cnt + (size_t)(q0 + u) * nbins + b) : 0ll;
    }
#pragma unroll
    for (int d = 1; d < U; d <<= 1) {
#pragma unroll
        for (int u = 0; u < U; u += 2 * d) {
            v[u] += v[u + d];
            k[u] += k[u + d];
        }
    }
    s = v[0];
    c = k[0];
}

// The totals of the bins first, first + step, ..., from their parts [q0, q1).
__device__ __forceinline__ void put_totals(int first, int step, int nbins, int pass, int q0, int q1,
                                           const double *part_sum, const long long *part_cnt, const BinOut &out)
{
    for (int b = first; b < nbins; b += step) {
        double s;
        long long c;
        sum_parts(nbins, pass, b, q0, q1, part_sum, part_cnt, s, c);
        out.sum[b] = s;
        if (pass == 0) out.count[b] = c;
        if (out.finish) finish_bin(pass, pass == 0 ? c : out.count[b], s, out.mean + b, out.sd + b);
    }
}

// The markers of bin b are those with n1 in [lo, hi): bin_of(n1) = b exactly
// when b n <= n1 nbins < (b + 1) n, i.e. ceil(b n / nbins) <= n1 <
// ceil((b + 1) n / nbins), the first bin open below and the last open above
// (bin_of clamps).  One interval per CTA, two compares per marker.
__device__ __forceinline__ void bin_interval(int b, int n, int nbins, long long &lo, long long &hi)
{
    lo = b == 0 ? LLONG_MIN : ((long long)b * n + nbins - 1) / nbins;
    hi = b == nbins - 1 ? LLONG_MAX : ((long long)(b + 1) * n + nbins - 1) / nbins;
}

// pass 0: count and sum per (bin, segment); pass 1: squared deviations about mean[bin]
__global__ void __launch_bounds__(kNormThreads) norm_partial_kernel(
    const double *score, const int8_t *status, const int32_t *n1, long long m, int n, int nbins,
    int pass, const double *mean, double *part_sum, long long *part_cnt)
{
    __shared__ double red_d[kNormThreads / 32];
    __shared__ long long red_c[kNormThreads / 32];
    const int b = blockIdx.x / kNormSegments, seg = blockIdx.x % kNormSegments;
    const long long per = (m + kNormSegments - 1) / kNormSegments;
    const long long lo = (long long)seg * per, hi = lo + per < m ? lo + per : m;
    long long n1lo, n1hi;
    bin_interval(b, n, nbins, n1lo, n1hi);
    double acc = 0.0;
    long long cnt = 0;
    const double mu = pass == 1 ? mean[b] : 0.0;
    for (long long k = lo + threadIdx.x; k < hi; k += kNormThreads) {
        if (status[k] != (int8_t)SELSCAN_LOCUS_OK) continue;
        const long long c = n1[k];
        if (c < n1lo || c >= n1hi) continue;
        const double x = score[k];
        if (pass == 0) { acc += x; ++cnt; }
        else { const double d = x - mu; acc += d * d; }
    }
    const double s = block_sum(acc, red_d);
    const long long c = block_sum(cnt, red_c);
    if (threadIdx.x == 0) {
        part_sum[(size_t)seg * nbins + b] = s;
        if (pass == 0) part_cnt[(size_t)seg * nbins + b] = c;
    }
}

// The totals of every bin from its segments, after norm_partial_kernel.  A launch
// of its own: there are 16 CTAs a bin, and a tally in each of them cost more than
// it saved (1,024 bins, 1,000 scores, whole call: 0.242 ms against 0.159).
__global__ void __launch_bounds__(32) norm_totals_kernel(int nbins, int pass, const double *part_sum,
                                                         const long long *part_cnt, BinOut out)
{
    static_assert(kNormSegments <= 16, "one sum of the parts");
    put_totals(blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, nbins, pass, 0, kNormSegments, part_sum,
               part_cnt, out);
}

// pass 0: count and sum per (segment, bin); pass 1: squared deviations about
// mean[bin].  Shared memory: sums [nbins + 1][128] (double), counts [nbins + 1][128]
// (the last row takes the markers that count in no bin).
__global__ void __launch_bounds__(kNormPrivThreads) norm_partial_private_kernel(
    const double *score, const int8_t *status, const int32_t *n1, long long m, int n, int nbins,
    int pass, const double *mean, double *part_sum, long long *part_cnt, BinOut out)
{
    extern __shared__ double psum[];
    int *pcnt = (int *)(psum + (size_t)(nbins + 1) * kNormPrivThreads);
    const int t = threadIdx.x;
    for (int b = 0; b <= nbins; ++b) {           // the last one takes what has no bin
        psum[b * kNormPrivThreads + t] = 0.0;
        pcnt[b * kNormPrivThreads + t] = 0;
    }
    const long long per = (m + kNormPrivSegments - 1) / kNormPrivSegments;
    const long long lo = (long long)blockIdx.x * per, hi = lo + per < m ? lo + per : m;
    const bool small = (unsigned long long)n * (unsigned long long)nbins < (1ull << 32);
    constexpr int U = 8;                         // markers whose loads are in flight together
    for (long long k0 = lo + t; k0 < hi; k0 += U * kNormPrivThreads) {
        int8_t st[U];
        int32_t c1[U];
        double x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long k = k0 + (long long)u * kNormPrivThreads;
            st[u] = k < hi ? status[k] : (int8_t)-1;
            c1[u] = k < hi ? n1[k] : 0;
            x[u] = k < hi ? score[k] : 0.0;
        }
        // two markers at a time: their additions overlap unless they meet in a bin
#pragma unroll
        for (int u = 0; u < U; u += 2) {
            int b[2];
            double v[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                // bin_of in 32 bits where n nbins fits them (0 <= n1 < n): n1 >= n is
                // the last bin, n1 <= 0 the first
                const int32_t c = c1[u + h];
                b[h] = -1;
                v[h] = 0.0;
                if (st[u + h] == (int8_t)SELSCAN_LOCUS_OK) {
                    if (!small) b[h] = bin_of(c, n, nbins);
                    else if (c <= 0) b[h] = 0;
                    else if (c >= n) b[h] = nbins - 1;
                    else b[h] = (int)((unsigned)c * (unsigned)nbins / (unsigned)n);
                    v[h] = x[u + h];
                    if (pass == 1) { const double d = v[h] - mean[b[h]]; v[h] = d * d; }
                }
            }
            if (b[0] == b[1]) {
                if (b[0] < 0) continue;
                v[0] += v[1];
            }
            const int i0 = (b[0] < 0 ? nbins : b[0]) * kNormPrivThreads + t;      // this thread's slots:
            const int i1 = (b[1] < 0 || b[1] == b[0] ? nbins : b[1]) * kNormPrivThreads + t;   // no other writer
            const double a0 = psum[i0], a1 = psum[i1];
            const int k0_ = pcnt[i0], k1_ = pcnt[i1];
            psum[i0] = a0 + v[0];
            pcnt[i0] = k0_ + (b[0] == b[1] ? 2 : 1);
            psum[i1] = a1 + v[1];
            pcnt[i1] = k1_ + 1;
        }
    }
    __syncthreads();
    for (int b = t; b < nbins; b += kNormPrivThreads) {
        double ch[8];                            // eight chains
        long long c = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) ch[u] = 0.0;
#pragma unroll 2
        for (int j = 0; j < kNormPrivThreads; j += 8) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int k = b * kNormPrivThreads + ((j + u + b) & (kNormPrivThreads - 1));
                ch[u] += psum[k];
                c += pcnt[k];
            }
        }
        const double sum = ((ch[0] + ch[1]) + (ch[2] + ch[3])) + ((ch[4] + ch[5]) + (ch[6] + ch[7]));
        part_sum[(size_t)blockIdx.x * nbins + b] = sum;
        if (pass == 0) part_cnt[(size_t)blockIdx.x * nbins + b] = c;
    }
    static_assert(kNormDozen <= 16 && kNormDozens <= 16, "two levels of sums of the parts");
    const int dz = blockIdx.x / kNormDozen, q0 = dz * kNormDozen;
    const int q1 = q0 + kNormDozen < kNormPrivSegments ? q0 + kNormDozen : kNormPrivSegments;
    if (!last_of(out.done + 1 + dz, (unsigned)(q1 - q0))) return;
    for (int b = t; b < nbins; b += kNormPrivThreads) {
        double s;
        long long c;
        sum_parts(nbins, pass, b, q0, q1, part_sum, part_cnt, s, c);
        part_sum[(size_t)(kNormPrivSegments + dz) * nbins + b] = s;
        if (pass == 0) part_cnt[(size_t)(kNormPrivSegments + dz) * nbins + b] = c;
    }
    if (last_of(out.done, kNormDozens))
        put_totals(t, kNormPrivThreads, nbins, pass, kNormPrivSegments, kNormPrivSegments + kNormDozens, part_sum,
                   part_cnt, out);
}

// Mean (pass 0) or sample SD (pass 1) of each bin from its totals.
__global__ void norm_finish_kernel(int nbins, int pass, const long long *bin_count,
                                   const double *bin_sum, double *bin_mean, double *bin_sd)
{
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nbins; b += gridDim.x * blockDim.x) {
        finish_bin(pass, bin_count[b], bin_sum[b], bin_mean + b, bin_sd + b);
    }
}

// out = (score - mean) / SD.  FP64 is a narrow pipe on this GPU (two lanes per SM
// cycle) and the divide is what the kernel spends its time on: the bin's
// reciprocal is taken once per CTA, and a quotient is one product corrected by
// its exact remainder (Markstein's method: correctly rounded, like the divide);
// quotients that are not in the ordinary range, and bins whose reciprocal is not
// (an SD that overflowed to infinity has 0, a subnormal one infinity), take the
// divide.
__device__ __forceinline__ bool ordinary(double v)
{
    // 2^-767 <= |v| < 2^768, on the integer pipe: a compare would take the FP64 pipe
    return ((unsigned)__double2hiint(v) & 0x7FFFFFFFu) - 0x10000000u < 0x60000000u;
}
__device__ __forceinline__ double quotient(double a, double d, double inv)
{
    const double q = a * inv;
    if (!ordinary(q) || !ordinary(a)) return a / d;
    return fma(fma(-q, d, a), inv, q);
}

constexpr int kApplyThreads = 256, kApplyU = 4;
__global__ void __launch_bounds__(kApplyThreads) norm_apply_kernel(const double *score, const int8_t *status,
                                                                   const int32_t *n1, long long m, int n,
                                                                   int nbins, const double *bin_mean,
                                                                   const double *bin_sd,
                                                                   const long long *bin_count, double *out)
{
    extern __shared__ double tab[];              // per bin: mean, SD, 1 / SD (0: no score; NaN: divide)
    for (int b = threadIdx.x; b < nbins; b += kApplyThreads) {
        const double sd = bin_sd[b];
        const bool ok = bin_count[b] >= 2 && sd > 0.0;
        tab[3 * b] = bin_mean[b];
        tab[3 * b + 1] = sd;
        const double inv = 1.0 / sd;
        tab[3 * b + 2] = !ok ? 0.0 : ordinary(inv) ? inv : __longlong_as_double(0x7ff8000000000000ll);
    }
    __syncthreads();
    const bool small = (unsigned long long)n * (unsigned long long)nbins < (1ull << 32);
    const long long stride = (long long)gridDim.x * kApplyThreads;
    for (long long k0 = blockIdx.x * (long long)kApplyThreads + threadIdx.x; k0 < m; k0 += kApplyU * stride) {
        int8_t st[kApplyU];
        int32_t c1[kApplyU];
        double x[kApplyU];
#pragma unroll
        for (int u = 0; u < kApplyU; ++u) {
            const long long k = k0 + u * stride;
            st[u] = k < m ? status[k] : (int8_t)-1;
            c1[u] = k < m ? n1[k] : 0;
            x[u] = k < m ? score[k] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kApplyU; ++u) {
            const long long k = k0 + u * stride;
            double r = __longlong_as_double(0x7ff8000000000000ll);
            if (st[u] == (int8_t)SELSCAN_LOCUS_OK) {
                int b;
                if (!small) b = bin_of(c1[u], n, nbins);
                else if (c1[u] <= 0) b = 0;
                else if (c1[u] >= n) b = nbins - 1;
                else b = (int)((unsigned)c1[u] * (unsigned)nbins / (unsigned)n);
                const double inv = tab[3 * b + 2];
                if (__double2hiint(inv) != 0) r = quotient(x[u] - tab[3 * b], tab[3 * b + 1], inv);
            }
            if (k < m) out[k] = r;
        }
    }
}

}  // namespace

}  // namespace selscan

using namespace selscan;

namespace {

size_t parts_bytes(int nbins)
{
    return ((size_t)nbins * kNormMaxSegments * 8 + 255) & ~(size_t)255;
}

bool norm_args_ok(const double *score, const int8_t *status, const int32_t *n1, int64_t m,
                  int32_t n, int32_t nbins)
{
    return score && status && n1 && m >= 1 && n >= 1 && nbins >= 1 && nbins <= SELSCAN_NORM_MAX_BINS;
}

// pass 0: bin_count and bin_sum (sum of the scores); pass 1: bin_sum = sum of
// squared deviations about bin_mean.  part_sum / part_cnt: workspace; out.done
// must be 0.
void launch_bin_sums(const double *score, const int8_t *status, const int32_t *n1, int64_t m,
                     int32_t n, int32_t nbins, int pass, const double *bin_mean, double *part_sum,
                     long long *part_cnt, const BinOut &out, cudaStream_t s)
{
    if (nbins <= kNormPrivMaxBins) {
        const size_t smem = (size_t)(nbins + 1) * kNormPrivThreads * (sizeof(double) + sizeof(int));
        cudaFuncSetAttribute(norm_partial_private_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)((size_t)(kNormPrivMaxBins + 1) * kNormPrivThreads * 12));
        norm_partial_private_kernel<<<kNormPrivSegments, kNormPrivThreads, smem, s>>>(
            score, status, n1, m, n, nbins, pass, bin_mean, part_sum, part_cnt, out);
    } else {
        const unsigned grid = (unsigned)(nbins * kNormSegments);
        norm_partial_kernel<<<grid, kNormThreads, 0, s>>>(score, status, n1, m, n, nbins, pass,
                                                          bin_mean, part_sum, part_cnt);
        norm_totals_kernel<<<(nbins + 31) / 32, 32, 0, s>>>(nbins, pass, part_sum, part_cnt, out);
    }
}

void launch_apply(const double *score, const int8_t *status, const int32_t *n1, int64_t m,
                  int32_t n, int32_t nbins, const double *bin_mean, const double *bin_sd,
                  const long long *bin_count, double *out, cudaStream_t s)
{
    // eight CTAs per SM at most
    long long blocks = (m + kApplyThreads * kApplyU - 1) / (kApplyThreads * kApplyU);
    const long long most = 8ll * device_sms();
    if (blocks > most) blocks = most;
    norm_apply_kernel<<<(unsigned)blocks, kApplyThreads, (size_t)nbins * 24, s>>>(
        score, status, n1, m, n, nbins, bin_mean, bin_sd, bin_count, out);
}

}  // namespace

extern "C" {

size_t selscan_normalize_workspace_bytes(int32_t nbins)
{
    if (nbins < 1 || nbins > SELSCAN_NORM_MAX_BINS) return 0;
    return parts_bytes(nbins) * 2 + (((size_t)nbins * 8 + 255) & ~(size_t)255) + 256;
}

int selscan_normalize(const double *score, const int8_t *status, const int32_t *n1, int64_t m,
                      int32_t n, int32_t nbins, double *out, int64_t *bin_count, double *bin_mean,
                      double *bin_sd, void *workspace, size_t ws_bytes, void *stream)
{
    if (!norm_args_ok(score, status, n1, m, n, nbins) || !out || !bin_count || !bin_mean || !bin_sd)
        return SELSCAN_ERR_INVALID_ARG;
    const size_t need = selscan_normalize_workspace_bytes(nbins);
    if (!workspace || ws_bytes < need || ((uintptr_t)workspace & 255)) return SELSCAN_ERR_WORKSPACE;
    cudaStream_t s = (cudaStream_t)stream;
    double *part_sum = (double *)workspace;
    long long *part_cnt = (long long *)((unsigned char *)workspace + parts_bytes(nbins));
    double *bin_sum = (double *)((unsigned char *)workspace + 2 * parts_bytes(nbins));
    long long *cnt = (long long *)bin_count;
    unsigned *done = (unsigned *)((unsigned char *)workspace + need - 256);
    if (cudaMemsetAsync(done, 0, 2 * kNormCounters * sizeof(unsigned), s) != cudaSuccess) return SELSCAN_ERR_CUDA;
    for (int pass = 0; pass < 2; ++pass)
        launch_bin_sums(score, status, n1, m, n, nbins, pass, bin_mean, part_sum, part_cnt,
                        BinOut{cnt, bin_sum, bin_mean, bin_sd, 1, done + pass * kNormCounters}, s);
    launch_apply(score, status, n1, m, n, nbins, bin_mean, bin_sd, cnt, out, s);
    return cudaGetLastError() == cudaSuccess ? SELSCAN_OK : SELSCAN_ERR_CUDA;
}

int selscan_normalize_bin_sums(const double *score, const int8_t *status, const int32_t *n1,
                               int64_t m, int32_t n, int32_t nbins, int32_t pass,
                               const double *bin_mean, int64_t *bin_count, double *bin_sum,
                               void *workspace, size_t ws_bytes, void *stream)
{
    if (!norm_args_ok(score, status, n1, m, n, nbins) || !bin_sum || (pass != 0 && pass != 1) ||
        (pass == 0 && !bin_count) || (pass == 1 && !bin_mean))
        return SELSCAN_ERR_INVALID_ARG;
    const size_t need = selscan_normalize_workspace_bytes(nbins);
    if (!workspace || ws_bytes < need || ((uintptr_t)workspace & 255)) return SELSCAN_ERR_WORKSPACE;
    double *part_sum = (double *)workspace;
    long long *part_cnt = (long long *)((unsigned char *)workspace + parts_bytes(nbins));
    unsigned *done = (unsigned *)((unsigned char *)workspace + need - 256);
    if (cudaMemsetAsync(done, 0, kNormCounters * sizeof(unsigned), (cudaStream_t)stream) != cudaSuccess) return SELSCAN_ERR_CUDA;
    launch_bin_sums(score, status, n1, m, n, nbins, pass, bin_mean, part_sum, part_cnt,
                    BinOut{(long long *)bin_count, bin_sum, nullptr, nullptr, 0, done}, (cudaStream_t)stream);
    return cudaGetLastError() == cudaSuccess ? SELSCAN_OK : SELSCAN_ERR_CUDA;
}

int selscan_normalize_finish(int32_t nbins, int32_t pass, const int64_t *bin_count,
                             const double *bin_sum, double *bin_mean, double *bin_sd, void *stream)
{
    if (nbins < 1 || nbins > SELSCAN_NORM_MAX_BINS || (pass != 0 && pass != 1) || !bin_count ||
        !bin_sum || (pass == 0 && !bin_mean) || (pass == 1 && !bin_sd))
        return SELSCAN_ERR_INVALID_ARG;
    norm_finish_kernel<<<(nbins + 127) / 128, 128, 0, (cudaStream_t)stream>>>(
        nbins, pass, (const long long *)bin_count, bin_sum, bin_mean, bin_sd);
    return cudaGetLastError() == cudaSuccess ? SELSCAN_OK : SELSCAN_ERR_CUDA;
}

int selscan_normalize_apply(const double *score, const int8_t *status, const int32_t *n1,
                            int64_t m, int32_t n, int32_t nbins, const int64_t *bin_count,
                            const double *bin_mean, const double *bin_sd, double *out, void *stream)
{
    if (!norm_args_ok(score, status, n1, m, n, nbins) || !bin_count || !bin_mean || !bin_sd || !out)
        return SELSCAN_ERR_INVALID_ARG;
    launch_apply(score, status, n1, m, n, nbins, bin_mean, bin_sd, (const long long *)bin_count, out,
                 (cudaStream_t)stream);
    return cudaGetLastError() == cudaSuccess ? SELSCAN_OK : SELSCAN_ERR_CUDA;
}

}  // extern "C"
