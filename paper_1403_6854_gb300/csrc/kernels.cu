// Kernels of the EHH / iHS / XPEHH scan (sm_103a).
//
//   validate      positions and map non-decreasing (device error word)
//   core_select   derived count n_1 per marker and the MAF filter (Section 1.2)
//   walk_*        the EHH walks (walk.cuh): persistent with a global queue, or
//                 one CTA per core (plain launch)
//   bucket_*      longest-first ordering of the walks that outlive the probe pass
//   finalize_*    iHH_c = downstream + upstream, status, ln ratio (Eq. 4, Eq. 5)
//   ehh_trace     the single-locus report (Eq. 1, Eq. 3 per step)
//   pack          0/1 bytes -> bit rows
#include <math.h>

#include "../../include/selscan.h"
#include "internal.h"
#include "device_common.cuh"

namespace selscan {

// ------------------------------------------------------------ validate
__global__ void validate_kernel(const long long *pos, const double *gmap, long long m, int32_t *err,
                                int check_map)
{
    for (long long k = 1 + blockIdx.x * (long long)blockDim.x + threadIdx.x; k < m;
         k += (long long)gridDim.x * blockDim.x) {
        if (pos[k] < pos[k - 1] || (check_map && !(gmap[k] >= gmap[k - 1])))
            atomicExch(err, SELSCAN_ERR_UNSORTED);
    }
    if (check_map && blockIdx.x == 0 && threadIdx.x == 0 && m >= 1 && !(gmap[0] == gmap[0]))
        atomicExch(err, SELSCAN_ERR_UNSORTED);
}

cudaError_t launch_validate(const long long *pos, const double *gmap, long long m, int32_t *err,
                            cudaStream_t s, int check_map)
{
    long long blocks = (m + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    validate_kernel<<<(unsigned)blocks, 256, 0, s>>>(pos, gmap, m, err, check_map);
    return cudaGetLastError();
}

// ------------------------------------------------------------ core select
// A warp counts the derived alleles of kCoreRows rows at once: lane l reads the
// 64-bit words l, l + 32, ... of each of them, all of a round's loads issued
// before the popcounts, then one warp sum per row.
constexpr int kCoreRows = 4;
__global__ void core_select_kernel(ScanArgs a, int mode, unsigned maf_num, unsigned maf_den,
                                   int maf_filter, int32_t *n1, int8_t *core_status)
{
    const int lane = threadIdx.x & 31;
    const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const unsigned n_total = (unsigned)(a.nA + a.nB);
    const unsigned long long *hap = (const unsigned long long *)a.hap;
    for (long long k0 = a.k0 + warp * kCoreRows; k0 < a.k1; k0 += nw * kCoreRows) {
        unsigned c[kCoreRows];
#pragma unroll
        for (int r = 0; r < kCoreRows; ++r) c[r] = 0u;
        for (int w = lane; w < a.W; w += 32) {
            const unsigned long long vm = (unsigned long long)valid32(a, 2 * w) |
                                          ((unsigned long long)valid32(a, 2 * w + 1) << 32);
            unsigned long long v[kCoreRows];
#pragma unroll
            for (int r = 0; r < kCoreRows; ++r)
                v[r] = k0 + r < a.k1 ? __ldg(hap + (k0 + r) * a.ld + w) : 0ull;
#pragma unroll
            for (int r = 0; r < kCoreRows; ++r) c[r] += (unsigned)__popcll(v[r] & vm);
        }
#pragma unroll
        for (int r = 0; r < kCoreRows; ++r) {
            const unsigned cr = __reduce_add_sync(FULLMASK, c[r]);
            const long long k = k0 + r;
            if (lane == 0 && k < a.k1) {
                n1[k] = (int32_t)cr;
                const unsigned minor = cr < n_total - cr ? cr : n_total - cr;
                const bool filt = (mode == 0 || maf_filter) &&
                                  (unsigned long long)maf_den * minor < (unsigned long long)maf_num * n_total;
                core_status[k] = filt ? (int8_t)SELSCAN_LOCUS_MAF_FILTERED : (int8_t)0;
            }
        }
    }
}

cudaError_t launch_core_select(const ScanArgs &a, int mode, unsigned maf_num, unsigned maf_den,
                               int maf_filter, int32_t *n1, int8_t *core_status, cudaStream_t s)
{
    const long long warps = (a.k1 - a.k0 + kCoreRows - 1) / kCoreRows;
    long long blocks = (warps * 32 + 255) / 256;
    if (blocks > 8192) blocks = 8192;
    if (blocks < 1) blocks = 1;
    core_select_kernel<<<(unsigned)blocks, 256, 0, s>>>(a, mode, maf_num, maf_den, maf_filter,
                                                         n1, core_status);
    return cudaGetLastError();
}

// 32 x 32 bit transpose across a warp: lane l holds row l (bit c = entry (l, c));
// afterwards lane j holds column j (bit i = entry (i, j)).  Five butterfly stages
// exchange the off-diagonal blocks of halving size with the partner lane.
__device__ __forceinline__ unsigned warp_transpose32(unsigned x, int lane)
{
    unsigned msk = 0x0000FFFFu;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1, msk ^= msk << s) {
        const unsigned y = __shfl_xor_sync(FULLMASK, x, s);
        x = (lane & s) ? ((x & ~msk) | ((y >> s) & msk)) : ((x & msk) | ((y << s) & ~msk));
    }
    return x;
}

// The 32 rows of block b as 32-marker words (dst: 64 W of them), by a CTA of 256
// threads: the rows [x0, x1) of the block are staged in shared memory (odd row
// stride: the column reads hit distinct banks), a warp taking whole rows, then
// a warp takes 64-bit columns, two 32 x 32 bit transposes each.  c[r]: this
// lane's derived alleles of row 4 warp + r.
__device__ __forceinline__ void block_words(const ScanArgs &a, long long b, long long x0, long long x1,
                                            unsigned long long *rows_sm, unsigned *dst, unsigned c[4])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int W = a.W, Wp = W | 1;
    const unsigned long long *hap = (const unsigned long long *)a.hap;
    // four rows per warp: all loads of a round before the counts
#pragma unroll
    for (int r = 0; r < 4; ++r) c[r] = 0u;
    for (int w = lane; w < W; w += 32) {
        const unsigned long long vm = (unsigned long long)valid32(a, 2 * w) |
                                      ((unsigned long long)valid32(a, 2 * w + 1) << 32);
        unsigned long long v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const long long k = 32 * b + 4 * warp + r;
            v[r] = k >= x0 && k < x1 ? __ldg(hap + k * a.ld + w) & vm : 0ull;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            rows_sm[(4 * warp + r) * Wp + w] = v[r];
            c[r] += (unsigned)__popcll(v[r]);
        }
    }
    __syncthreads();
    for (int w = warp; w < W; w += 8) {
        const unsigned long long v = rows_sm[lane * Wp + w];
        dst[64 * w + lane] = warp_transpose32((unsigned)v, lane);
        dst[64 * w + 32 + lane] = warp_transpose32((unsigned)(v >> 32), lane);
    }
}

// core_select fused with the transposition of the rows into 32-marker words:
// both read every row once.  Bound by HBM (a row is read once and written once):
// 5,000 haplotypes x 1,000,000 markers 0.38 ms, 3.3 TB/s.
__global__ void __launch_bounds__(256) core_select_words_kernel(ScanArgs a, int mode, unsigned maf_num,
                                                                unsigned maf_den, int maf_filter, int32_t *n1,
                                                                int8_t *core_status, long long x0, long long x1,
                                                                unsigned *tw)
{
    extern __shared__ __align__(16) unsigned long long rows_sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned n_total = (unsigned)(a.nA + a.nB);
    const long long b = (x0 >> 5) + blockIdx.x;
    unsigned c[4];
    block_words(a, b, x0, x1, rows_sm, tw + (size_t)blockIdx.x * (size_t)(64 * a.W), c);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const unsigned cr = __reduce_add_sync(FULLMASK, c[r]);
        const long long k = 32 * b + 4 * warp + r;
        if (lane == 0 && k >= a.k0 && k < a.k1) {
            n1[k] = (int32_t)cr;
            const unsigned minor = cr < n_total - cr ? cr : n_total - cr;
            const bool filt = (mode == 0 || maf_filter) &&
                              (unsigned long long)maf_den * minor < (unsigned long long)maf_num * n_total;
            core_status[k] = filt ? (int8_t)SELSCAN_LOCUS_MAF_FILTERED : (int8_t)0;
        }
    }
}

// The 32-marker words of every scan of a tick, one CTA per block.
__global__ void __launch_bounds__(256) tick_words_kernel(const __grid_constant__ ChunkTick t)
{
    extern __shared__ __align__(16) unsigned long long rows_sm[];
    int s = 0;
    while ((int)blockIdx.x >= t.boff[s + 1]) ++s;
    const ScanArgs &a = t.w[s].a;
    const long long b = (int)blockIdx.x - t.boff[s];
    unsigned c[4];
    block_words(a, b, 0, a.m, rows_sm, (unsigned *)t.w[s].tw + (size_t)b * (size_t)(64 * a.W), c);
}

cudaError_t launch_tick_words(const ChunkTick &t, cudaStream_t s)
{
    int W = 1;
    for (int i = 0; i < t.nscans; ++i) W = t.w[i].a.W > W ? t.w[i].a.W : W;     // 0: no part in the tick
    const size_t smem = (size_t)32 * (W | 1) * 8;
    const cudaError_t e = allow_smem(tick_words_kernel);
    if (e != cudaSuccess) return e;
    tick_words_kernel<<<t.boff[t.nscans], 256, smem, s>>>(t);
    return cudaGetLastError();
}

cudaError_t launch_core_select_words(const ScanArgs &a, int mode, unsigned maf_num, unsigned maf_den,
                                     int maf_filter, int32_t *n1, int8_t *core_status, long long x0,
                                     long long x1, unsigned *tw, cudaStream_t s)
{
    const size_t smem = (size_t)32 * (a.W | 1) * 8;
    const cudaError_t e = allow_smem(core_select_words_kernel);
    if (e != cudaSuccess) return e;
    const long long blocks = ((x1 - 1) >> 5) - (x0 >> 5) + 1;
    core_select_words_kernel<<<(unsigned)blocks, 256, smem, s>>>(a, mode, maf_num, maf_den, maf_filter, n1,
                                                                 core_status, x0, x1, tw);
    return cudaGetLastError();
}

// ------------------------------------------------------------ walks
// Persistent walk kernel.  pass 1: items in core order (a warp takes one
// core's items per queue fetch), optionally capped at max_steps; pass 2:
// the sorted list of walks the first pass left unfinished, one per fetch.
// MINB: resident 8-warp CTAs per SM the build is compiled for (register cap
// 65536 / (256 * MINB)): 2 (128 registers) or 3 (85 registers)
template <int NPOP, int MINB>
__global__ void __launch_bounds__(256, MINB) walk_persistent_kernel(ScanArgs a, ItemSink sk, Scratch sc,
                                                              long long n_cores, int pass,
                                                              int max_steps, int fetch)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int wpc = blockDim.x >> 5;
    const long long gw = (long long)blockIdx.x * wpc + warp;
    WarpBufs b = make_bufs(smem + (size_t)warp * slice_bytes(sc),
                           sc.base + (size_t)gw * sc.per_warp, sc);
    init_window(b);
    unsigned wpar[2] = {0u, 0u};
    const int ipc = NPOP == 2 ? 2 : 4;
    const unsigned long long total = pass == 2 ? sk.q->n2 : (unsigned long long)n_cores;
    const unsigned long long step = pass == 2 ? 1ull : (unsigned long long)fetch;
    for (;;) {
        unsigned long long idx = 0;
        if (lane == 0) idx = atomicAdd(&sk.q->head, step);
        idx = __shfl_sync(FULLMASK, idx, 0);
        if (idx >= total) break;
        if (pass == 2) {
            if (!run_item<NPOP>(a, sk, b, sk.sorted2[idx], 0, wpar)) return;
            continue;
        }
        const unsigned long long end = idx + step < total ? idx + step : total;
        for (unsigned long long c = (unsigned long long)a.k0 + idx; c < (unsigned long long)a.k0 + end;
             ++c) {
            if (sk.core_status[c] == (int8_t)SELSCAN_LOCUS_MAF_FILTERED) continue;
            for (int q = 0; q < ipc; ++q)
                if (!run_item<NPOP>(a, sk, b, (uint32_t)(c * ipc + q), max_steps, wpar)) return;
        }
    }
}

// Plain launch: one CTA per core, one warp per walk; global scratch slots
// are taken from a bitmap (at most nslots warps are resident at once).
template <int NPOP>
__global__ void __launch_bounds__(128) walk_plain_kernel(ScanArgs a, ItemSink sk, Scratch sc,
                                                         unsigned int *slotmap, int nslots)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const long long core = a.k0 + blockIdx.x;
    if (sk.core_status[core] == (int8_t)SELSCAN_LOCUS_MAF_FILTERED) return;
    int slot = -1;
    if (lane == 0) {
        const int start = (int)(((long long)blockIdx.x * (blockDim.x >> 5) + warp) % nslots);
        for (int t = 0; t < nslots; ++t) {
            const int s = (start + t) % nslots;
            const unsigned bit = 1u << (s & 31);
            if (!(atomicOr(slotmap + (s >> 5), bit) & bit)) { slot = s; break; }
        }
        __threadfence();
    }
    slot = __shfl_sync(FULLMASK, slot, 0);
    if (slot < 0) {                       // cannot happen: nslots >= resident warps
        if (lane == 0) {
            sk.item_status[core * (NPOP == 2 ? 2 : 4) + warp] = (int8_t)WALK_UNFINISHED;
            atomicExch(sc.err, SELSCAN_ERR_INTERNAL);
        }
        return;
    }
    WarpBufs b = make_bufs(smem + (size_t)warp * slice_bytes(sc),
                           sc.base + (size_t)slot * sc.per_warp, sc);
    init_window(b);
    unsigned wpar[2] = {0u, 0u};
    // a warp whose copies may still be in flight keeps its slot (nothing else reuses it)
    if (!run_item<NPOP>(a, sk, b, (uint32_t)(core * (NPOP == 2 ? 2 : 4) + warp), 0, wpar)) return;
    __syncwarp();
    if (lane == 0) {
        __threadfence();
        atomicAnd(slotmap + (slot >> 5), ~(1u << (slot & 31)));
    }
}

// one block: histogram of the queued walks' keys, its exclusive scan (the
// buckets' first places), and the queue's head reset
__global__ void __launch_bounds__(1024) bucket_rank_kernel(ItemSink sk)
{
    __shared__ uint32_t t[NBUCKET];
    const int i = threadIdx.x;
    const unsigned long long n2 = sk.q->n2;
    if (i < NBUCKET) t[i] = 0u;
    __syncthreads();
    for (unsigned long long k = i; k < n2; k += blockDim.x) atomicAdd(t + sk.key2[k], 1u);
    __syncthreads();
    const uint32_t own = i < NBUCKET ? t[i] : 0u;
    for (int o = 1; o < NBUCKET; o <<= 1) {
        const uint32_t v = i < NBUCKET && i >= o ? t[i - o] : 0u;
        __syncthreads();
        if (i < NBUCKET) t[i] += v;
        __syncthreads();
    }
    if (i < NBUCKET) sk.bucket[i] = t[i] - own;
    if (i == 0) sk.q->head = 0ull;
}

__global__ void bucket_scatter_kernel(ItemSink sk)
{
    const unsigned long long n2 = sk.q->n2;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n2;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const uint32_t p = atomicAdd(sk.bucket + sk.key2[i], 1u);
        sk.sorted2[p] = sk.list2[i];
    }
}

static int g_sms = 0;
static int sm_count()
{
    if (g_sms == 0) {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
            g_sms = v;
        else
            return 152;
    }
    return g_sms;
}

template <typename K>
static int occupancy_of(K kernel, int warps_per_cta, size_t smem_bytes, bool carve)
{
    int nb = 0;
    allow_smem(kernel);
    if (carve) cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, warps_per_cta * 32, smem_bytes) !=
        cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    return nb;
}

int max_ctas_per_sm(int schedule, int warps_per_cta, size_t smem_bytes, int minb)
{
    int a, b;
    if (schedule == SELSCAN_SCHED_PLAIN) {
        a = occupancy_of(walk_plain_kernel<1>, warps_per_cta, smem_bytes, false);
        b = occupancy_of(walk_plain_kernel<2>, warps_per_cta, smem_bytes, false);
    } else if (minb == 3) {
        a = occupancy_of(walk_persistent_kernel<1, 3>, warps_per_cta, smem_bytes, true);
        b = occupancy_of(walk_persistent_kernel<2, 3>, warps_per_cta, smem_bytes, true);
    } else {
        a = occupancy_of(walk_persistent_kernel<1, 2>, warps_per_cta, smem_bytes, true);
        b = occupancy_of(walk_persistent_kernel<2, 2>, warps_per_cta, smem_bytes, true);
    }
    // the smaller of the two builds: a plan must fit either population count
    if (a < 1) return b;
    if (b < 1) return a;
    return a < b ? a : b;
}

int device_sms() { return sm_count(); }

// percentage of the unified L1/shared array to reserve for shared memory so
// that the CTAs one SM holds at once fit (228 KB per SM on this part)
static int carveout_pct(size_t smem_per_cta, int ctas)
{
    const int per_sm = (ctas + sm_count() - 1) / sm_count();
    const size_t need = (smem_per_cta + 1024) * (size_t)per_sm;
    int pct = (int)((need * 100 + 228 * 1024 - 1) / (228 * 1024));
    return pct > 100 ? 100 : (pct < 10 ? 10 : pct);
}

template <int NPOP, int MINB>
static cudaError_t persistent_impl(const ScanArgs &a, const ItemSink &sk, const Scratch &sc,
                                   int schedule, int wpc, int ctas, int probe, int fetch,
                                   long long n_cores, cudaStream_t s)
{
    const size_t smem = slice_bytes(sc) * (size_t)wpc;
    cudaError_t e = allow_smem(walk_persistent_kernel<NPOP, MINB>);
    if (e != cudaSuccess) return e;
    // shared memory as large as the resident CTAs need; the rest stays L1
    e = cudaFuncSetAttribute(walk_persistent_kernel<NPOP, MINB>,
                             cudaFuncAttributePreferredSharedMemoryCarveout, carveout_pct(smem, ctas));
    if (e != cudaSuccess) return e;
    const int cap = schedule == SELSCAN_SCHED_LONGEST_FIRST ? probe : 0;
    walk_persistent_kernel<NPOP, MINB><<<ctas, wpc * 32, smem, s>>>(a, sk, sc, n_cores, 1, cap,
                                                                     cap > 0 ? 1 : fetch);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (schedule == SELSCAN_SCHED_LONGEST_FIRST && probe > 0) {
        bucket_rank_kernel<<<1, 1024, 0, s>>>(sk);
        bucket_scatter_kernel<<<2 * sm_count(), 256, 0, s>>>(sk);
        walk_persistent_kernel<NPOP, MINB><<<ctas, wpc * 32, smem, s>>>(a, sk, sc, n_cores, 2, 0, 1);
    }
    return cudaGetLastError();
}

template <int NPOP>
static cudaError_t walk_impl(const ScanArgs &a, const ItemSink &sk, const Scratch &sc,
                             int schedule, int wpc, int ctas, int probe, int fetch, int minb,
                             long long n_cores, cudaStream_t s)
{
    if (schedule == SELSCAN_SCHED_PLAIN) {
        const int ipc = NPOP == 2 ? 2 : 4;
        const size_t smem_p = slice_bytes(sc) * (size_t)ipc;
        cudaError_t e = allow_smem(walk_plain_kernel<NPOP>);
        if (e != cudaSuccess) return e;
        // `ctas` carries the number of scratch slots; the bitmap was reset by the caller
        walk_plain_kernel<NPOP><<<(unsigned)n_cores, ipc * 32, smem_p, s>>>(a, sk, sc, sk.slotmap,
                                                                            ctas);
        return cudaGetLastError();
    }
    if (minb == 3)
        return persistent_impl<NPOP, 3>(a, sk, sc, schedule, wpc, ctas, probe, fetch, n_cores, s);
    return persistent_impl<NPOP, 2>(a, sk, sc, schedule, wpc, ctas, probe, fetch, n_cores, s);
}

template <int NPOP, int MINB>
static cudaError_t pass2_impl(const ScanArgs &a, const ItemSink &sk, const Scratch &sc, int wpc,
                              int ctas, cudaStream_t s)
{
    const size_t smem = slice_bytes(sc) * (size_t)wpc;
    cudaError_t e = allow_smem(walk_persistent_kernel<NPOP, MINB>);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(walk_persistent_kernel<NPOP, MINB>,
                             cudaFuncAttributePreferredSharedMemoryCarveout, carveout_pct(smem, ctas));
    if (e != cudaSuccess) return e;
    bucket_rank_kernel<<<1, 1024, 0, s>>>(sk);
    bucket_scatter_kernel<<<2 * sm_count(), 256, 0, s>>>(sk);
    walk_persistent_kernel<NPOP, MINB><<<ctas, wpc * 32, smem, s>>>(a, sk, sc, 0, 2, 0, 1);
    return cudaGetLastError();
}

cudaError_t launch_pass2(const ScanArgs &a, const ItemSink &sink, const Scratch &sc,
                         int warps_per_cta, int ctas, int minb, cudaStream_t s)
{
    if (sink.mode == 1)
        return minb == 3 ? pass2_impl<2, 3>(a, sink, sc, warps_per_cta, ctas, s)
                         : pass2_impl<2, 2>(a, sink, sc, warps_per_cta, ctas, s);
    return minb == 3 ? pass2_impl<1, 3>(a, sink, sc, warps_per_cta, ctas, s)
                     : pass2_impl<1, 2>(a, sink, sc, warps_per_cta, ctas, s);
}

cudaError_t launch_walk(const ScanArgs &a, const ItemSink &sink, const Scratch &sc,
                        int schedule, int warps_per_cta, int ctas, int probe_steps, int fetch,
                        int minb, long long n_cores, cudaStream_t s)
{
    if (sink.mode == 1)
        return walk_impl<2>(a, sink, sc, schedule, warps_per_cta, ctas, probe_steps, fetch, minb,
                            n_cores, s);
    return walk_impl<1>(a, sink, sc, schedule, warps_per_cta, ctas, probe_steps, fetch, minb,
                        n_cores, s);
}

// ------------------------------------------------------------ finalize
__global__ void finalize_ihs_kernel(ItemSink sk, long long k0, long long k1, double *ihh1, double *ihh0,
                                    double *lnratio, int8_t *status)
{
    for (long long c = k0 + blockIdx.x * (long long)blockDim.x + threadIdx.x; c < k1;
         c += (long long)gridDim.x * blockDim.x) {
        if (sk.core_status[c] == (int8_t)SELSCAN_LOCUS_MAF_FILTERED) {
            ihh1[c] = 0.0;
            ihh0[c] = 0.0;
            lnratio[c] = __longlong_as_double(0x7ff8000000000000ll);
            for (int q = 0; q < 4; ++q) { sk.stop[4 * c + q] = 0; sk.digest[4 * c + q] = 0ull; }
            continue;
        }
        int worst = 0;
        for (int q = 0; q < 4; ++q) {
            const int st = sk.item_status[4 * c + q];
            worst = st > worst ? st : worst;
        }
        const double a1 = sk.item_ihh[4 * c] + sk.item_ihh[4 * c + 1];   // down + up
        const double a0 = sk.item_ihh[4 * c + 2] + sk.item_ihh[4 * c + 3];
        if (worst == 0 && (a1 == 0.0 || a0 == 0.0)) worst = SELSCAN_LOCUS_UNDEFINED;
        ihh1[c] = a1;
        ihh0[c] = a0;
        status[c] = (int8_t)worst;
        lnratio[c] = worst == 0 ? log(a1 / a0) : __longlong_as_double(0x7ff8000000000000ll);
    }
}

__global__ void finalize_xpehh_kernel(ItemSink sk, long long k0, long long k1, double *ihhA, double *ihhB,
                                      double *lnratio, int8_t *status)
{
    for (long long c = k0 + blockIdx.x * (long long)blockDim.x + threadIdx.x; c < k1;
         c += (long long)gridDim.x * blockDim.x) {
        if (sk.core_status[c] == (int8_t)SELSCAN_LOCUS_MAF_FILTERED) {
            ihhA[c] = 0.0;
            ihhB[c] = 0.0;
            lnratio[c] = __longlong_as_double(0x7ff8000000000000ll);
            for (int q = 0; q < 2; ++q) sk.stop[2 * c + q] = 0;
            for (int q = 0; q < 6; ++q) sk.digest[6 * c + q] = 0ull;
            continue;
        }
        int worst = 0;
        for (int q = 0; q < 2; ++q) {
            const int st = sk.item_status[2 * c + q];
            worst = st > worst ? st : worst;
        }
        const double a = sk.item_ihh[4 * c] + sk.item_ihh[4 * c + 2];      // down + up, pop A
        const double bb = sk.item_ihh[4 * c + 1] + sk.item_ihh[4 * c + 3]; // pop B
        if (worst == 0 && (a == 0.0 || bb == 0.0)) worst = SELSCAN_LOCUS_UNDEFINED;
        ihhA[c] = a;
        ihhB[c] = bb;
        status[c] = (int8_t)worst;
        lnratio[c] = worst == 0 ? log(a / bb) : __longlong_as_double(0x7ff8000000000000ll);
    }
}

cudaError_t launch_finalize_ihs(const ItemSink &sink, long long k0, long long k1, double *ihh1,
                                double *ihh0, double *lnratio, int8_t *status, cudaStream_t s)
{
    long long blocks = (k1 - k0 + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    finalize_ihs_kernel<<<(unsigned)blocks, 256, 0, s>>>(sink, k0, k1, ihh1, ihh0, lnratio, status);
    return cudaGetLastError();
}

cudaError_t launch_finalize_xpehh(const ItemSink &sink, long long k0, long long k1, double *ihhA,
                                  double *ihhB, double *lnratio, int8_t *status, cudaStream_t s)
{
    long long blocks = (k1 - k0 + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    finalize_xpehh_kernel<<<(unsigned)blocks, 256, 0, s>>>(sink, k0, k1, ihhA, ihhB, lnratio, status);
    return cudaGetLastError();
}

// ------------------------------------------------------------ EHH trace
__global__ void __launch_bounds__(192) ehh_trace_kernel(ScanArgs a, long long locus, Scratch sc,
                                                        unsigned long long *S, long long cap,
                                                        long long *len, int32_t *stop,
                                                        int8_t *status, double *ihh,
                                                        unsigned long long *denom, const int *rest)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int q = threadIdx.x >> 5;
    if (rest && rest[q] == 0) return;         // done before (warps do not meet)
    trace_walk(a, locus, sc, smem + (size_t)q * slice_bytes(sc), q, S, cap, len, stop, status, ihh, denom);
}

cudaError_t launch_ehh(const ScanArgs &a, long long locus, const Scratch &sc,
                       unsigned long long *S, long long cap, long long *len, int32_t *stop,
                       int8_t *status, double *ihh, unsigned long long *denom, const int *rest,
                       cudaStream_t s)
{
    const size_t smem = slice_bytes(sc) * 6;
    cudaError_t e = allow_smem(ehh_trace_kernel);
    if (e != cudaSuccess) return e;
    ehh_trace_kernel<<<1, 192, smem, s>>>(a, locus, sc, S, cap, len, stop, status, ihh, denom, rest);
    return cudaGetLastError();
}

// ------------------------------------------------------------ pack
// bit 0 of each of the four bytes of x, as bits 0..3: with one bit per byte
// kept, the multiply moves byte i's bit to bit 24 + i and nothing else reaches
// bits 24..31
__device__ __forceinline__ unsigned byte_lsbs(unsigned x) { return ((x & 0x01010101u) * 0x01020408u) >> 24; }

// Bit 0 of each of 16 bytes, as bits 0..15.
__device__ __forceinline__ unsigned lsbs16(const uint4 &q)
{
    return byte_lsbs(q.x) | (byte_lsbs(q.y) << 4) | (byte_lsbs(q.z) << 8) | (byte_lsbs(q.w) << 12);
}
// the same of the 16 bytes from p on, those outside [lo, hi) as 0
__device__ __noinline__ unsigned lsbs16_edge(const uint8_t *p, const uint8_t *lo, const uint8_t *hi)
{
    unsigned v = 0u;
    for (int i = 0; i < 16; ++i)
        if (p + i >= lo && p + i < hi) v |= (unsigned)(__ldg(p + i) & 1u) << i;
    return v;
}

// Rows of bytes start anywhere: a lane reads the 16-byte chunks at aligned
// addresses, folds each to 16 bits, and the stream of bits, not of bytes, is
// shifted to the row's start with the next chunk's bits.  A chunk that leaves
// the input is read byte by byte.

// marker-major input [m, n] bytes: a warp packs whole marker rows, 512
// haplotypes a step (one 16-byte load per lane, four steps in flight); four
// lanes' 16 bits are a word, lane l keeps words 8 step + l (l < 8) and stores
// them 32 at a time.  Bound by HBM (5,000 x 250,000: 0.35 ms, 4.0 TB/s; byte
// loads and ballots took 1.24 ms).
__global__ void __launch_bounds__(256) pack_mm_kernel(const uint8_t *hap01, int n, long long m,
                                                      int W, unsigned long long *rows, long long ld)
{
    const int lane = threadIdx.x & 31;
    const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const uint8_t *end = hap01 + m * n;
    for (long long k = warp; k < m; k += nw) {
        const uint8_t *src = hap01 + k * n;
        const int off = (int)((uintptr_t)src & 15u);
        const uint8_t *base = src - off;
        unsigned long long *dst = rows + k * ld;
        for (long long w0 = 0; w0 < ld; w0 += 32) {        // 32 words: four steps of 512 haplotypes
            uint4 q[4];
            bool in[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const long long c = (w0 >> 3) + u;             // step
                const uint8_t *p = base + c * 512 + lane * 16;
                in[u] = c * 512 < n && p >= hap01 && p + 16 <= end;
                if (in[u]) q[u] = __ldg((const uint4 *)p);
            }
            unsigned long long mine = 0ull;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const long long c = (w0 >> 3) + u;
                if (c * 512 >= n) break;                        // warp-uniform
                const uint8_t *p = base + c * 512 + lane * 16;
                unsigned v = in[u] ? lsbs16(q[u]) : lsbs16_edge(p, hap01, end);
                unsigned next = __shfl_down_sync(FULLMASK, v, 1);
                if (off) {                                      // warp-uniform
                    if (lane == 31) {
                        const uint8_t *p2 = p + 16;
                        next = p2 >= src + n ? 0u
                             : p2 + 16 <= end ? lsbs16(__ldg((const uint4 *)p2)) : lsbs16_edge(p2, hap01, end);
                    }
                    v = ((v | (next << 16)) >> off) & 0xFFFFu;
                }
                const long long h0 = c * 512 + lane * 16;       // haplotypes past n are pad bits
                if (h0 + 16 > n) v &= h0 >= n ? 0u : (1u << (n - h0)) - 1u;
                // lane 4 i gathers word 8 u + i of the 32, lane 8 u + i keeps it
                unsigned lo = v | (__shfl_down_sync(FULLMASK, v, 1) << 16);
                const unsigned hi = __shfl_down_sync(FULLMASK, lo, 2);
                lo = __shfl_sync(FULLMASK, lo, 4 * (lane & 7));
                const unsigned hi2 = __shfl_sync(FULLMASK, hi, 4 * (lane & 7));
                if ((lane >> 3) == u) mine = (unsigned long long)lo | ((unsigned long long)hi2 << 32);
            }
            if (w0 + lane < ld) dst[w0 + lane] = mine;
        }
    }
}

// The same for samples of at most 16 S - 15 haplotypes: S lanes a row, so that a
// warp packs 32 / S rows at once, four rows of each group in flight.
template <int S>
__global__ void __launch_bounds__(256) pack_mm_small_kernel(const uint8_t *hap01, int n, long long m,
                                                            int W, unsigned long long *rows, long long ld)
{
    constexpr int U = 4;
    const int l = threadIdx.x & (S - 1);
    const long long group = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / S;
    const long long ng = (long long)gridDim.x * blockDim.x / S;
    const uint8_t *end = hap01 + m * n;
    const int keep = n - 16 * l;                               // haplotypes of this lane's 16
    // whole warps take the same number of turns (shuffles): rows past m are not stored
    const long long turns = (m + ng * U - 1) / (ng * U);
    for (long long q = 0; q < turns; ++q) {
        uint4 v4[U];
        bool in[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long k = (q * U + u) * ng + group;
            const uint8_t *src = hap01 + k * n, *p = src - (int)((uintptr_t)src & 15u) + 16 * l;
            in[u] = k < m && p < src + n && p >= hap01 && p + 16 <= end;
            if (in[u]) v4[u] = __ldg((const uint4 *)p);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long k = (q * U + u) * ng + group;
            const uint8_t *src = hap01 + k * n;
            const int off = (int)((uintptr_t)src & 15u);
            const uint8_t *p = src - off + 16 * l;
            unsigned v = in[u] ? lsbs16(v4[u]) : (k < m && p < src + n ? lsbs16_edge(p, hap01, end) : 0u);
            v = ((v | (__shfl_down_sync(FULLMASK, v, 1, S) << 16)) >> off) & 0xFFFFu;
            if (keep < 16) v &= keep <= 0 ? 0u : (1u << keep) - 1u;
            const unsigned lo = v | (__shfl_down_sync(FULLMASK, v, 1, S) << 16);
            const unsigned hi = __shfl_down_sync(FULLMASK, lo, 2, S);
            if (k < m) {
                if ((l & 3) == 0 && l / 4 < W)
                    rows[k * ld + l / 4] = (unsigned long long)lo | ((unsigned long long)hi << 32);
                for (long long w = W + l; w < ld; w += S) rows[k * ld + w] = 0ull;
            }
        }
    }
}

// haplotype-major input [n, m] bytes: a CTA packs word w of a tile of kPackTile
// markers.  Warp v reads rows 64 w + 8 v .. + 7 as whole kPackTile-byte pieces
// (one coalesced 16-byte load per lane and row), folds each lane's 16 bytes into
// a 16-bit mask and pairs the masks of neighbouring lanes into the row's 32-bit
// mask words in shared memory (stride 17 words: the transpose's reads of one
// word of 32 rows hit distinct banks); then warp v transposes markers
// [64 v, 64 v + 64) of the tile: four 32 x 32 bit transposes.  This kernel takes
// the whole tiles of inputs whose rows all start on 16-byte boundaries.  Bound by
// HBM: 5,000 x 1,000,000 1.17 ms, 4.8 TB/s.
constexpr int kPackTile = 512;
__global__ void __launch_bounds__(256) pack_hm_staged_kernel(const uint8_t *hap01, int n,
                                                             long long m, int W,
                                                             unsigned long long *rows, long long ld)
{
    __shared__ unsigned msk[64][kPackTile / 32 + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long tasks = m / kPackTile * ld;
    for (long long t = blockIdx.x; t < tasks; t += gridDim.x) {
        const long long kb = t / ld;
        const long long w = t - kb * ld;
        const long long k0 = kb * kPackTile;
        if (w < W) {
            uint4 q[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) {              // all eight loads in flight at once
                const long long h = 64 * w + 8 * warp + r;
                q[r] = __ldg((const uint4 *)(hap01 + (h < n ? h : 0) * m + k0) + lane);
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const long long h = 64 * w + 8 * warp + r;
                unsigned v = lsbs16(q[r]);
                if (h >= n) v = 0u;
                const unsigned hi = __shfl_down_sync(FULLMASK, v, 1);
                if ((lane & 1) == 0) msk[8 * warp + r][lane >> 1] = v | (hi << 16);
            }
        }
        __syncthreads();
        unsigned a0 = 0u, a1 = 0u, b0 = 0u, b1 = 0u;
        if (w < W) {
            a0 = msk[lane][2 * warp];
            a1 = msk[lane][2 * warp + 1];
            b0 = msk[lane + 32][2 * warp];
            b1 = msk[lane + 32][2 * warp + 1];
        }
        __syncthreads();                               // the next tile may refill msk
        const unsigned lo0 = warp_transpose32(a0, lane), hi0 = warp_transpose32(b0, lane);
        const unsigned lo1 = warp_transpose32(a1, lane), hi1 = warp_transpose32(b1, lane);
        const long long k = k0 + 64 * warp + lane;
        rows[k * ld + w] = (unsigned long long)lo0 | ((unsigned long long)hi0 << 32);
        rows[(k + 32) * ld + w] = (unsigned long long)lo1 | ((unsigned long long)hi1 << 32);
    }
}

// Bit j of (a, b) = bit 0 of p[j] (a: j < 32, b: j >= 32) for j < nk <= 64;
// nk = 64: from its four 16-byte pieces v.
__device__ __forceinline__ void lsb_mask64(const uint4 *v, const uint8_t *p, int nk, unsigned &a,
                                           unsigned &b)
{
    a = 0u;
    b = 0u;
    if (nk == 64) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned s = byte_lsbs(v[i].x) | (byte_lsbs(v[i].y) << 4) |
                               (byte_lsbs(v[i].z) << 8) | (byte_lsbs(v[i].w) << 12);
            if (i < 2) a |= s << (16 * i);
            else b |= s << (16 * (i - 2));
        }
    } else {
        for (int j = 0; j < nk; ++j) {
            const unsigned bit = __ldg(p + j) & 1u;
            if (j < 32) a |= bit << j;
            else b |= bit << (j - 32);
        }
    }
}

// haplotype-major input [n, m] bytes whose rows start on 16-byte boundaries,
// markers [kbeg, m) (the ragged tail of the staged kernel above: 2 us less than a
// tile of the kernel below): a warp packs word w of 64 consecutive markers.  Lane l reads markers [k0, k0 + 64) of haplotypes 64 w + l and
// 64 w + 32 + l (contiguous bytes of their rows, both rows' loads issued
// together), keeps bit 0 of each byte in a 64-bit mask per haplotype, and four
// 32 x 32 bit transposes across the warp turn the masks into the markers'
// words; lane j stores the words of markers k0 + j and k0 + 32 + j.
// Consecutive warps take consecutive words of the same markers, so the stores
// of a row segment meet in L2.
__global__ void __launch_bounds__(256) pack_hm_kernel(const uint8_t *hap01, int n, long long m,
                                                      int W, unsigned long long *rows, long long ld,
                                                      long long kbeg)
{
    const int lane = threadIdx.x & 31;
    const long long tasks = (m - kbeg + 63) / 64 * ld;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long t = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; t < tasks; t += nw) {
        const long long kb = t / ld;
        const long long w = t - kb * ld;
        const long long k0 = kbeg + kb * 64;
        const int nk = m - k0 < 64 ? (int)(m - k0) : 64;
        unsigned a0 = 0u, a1 = 0u, b0 = 0u, b1 = 0u;     // haplotype 64 w + l: a; + 32: b
        if (w < W) {
            const long long h0 = 64 * w + lane, h1 = h0 + 32;
            const bool v0 = h0 < n, v1 = h1 < n;
            // rows past n read row 0 (it exists) and are dropped
            const uint8_t *p0 = hap01 + (v0 ? h0 : 0) * m + k0;
            const uint8_t *p1 = hap01 + (v1 ? h1 : 0) * m + k0;
            uint4 q0[4], q1[4];
            if (nk == 64) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    q0[i] = __ldg((const uint4 *)p0 + i);
                    q1[i] = __ldg((const uint4 *)p1 + i);
                }
            }
            lsb_mask64(q0, p0, nk, a0, a1);
            lsb_mask64(q1, p1, nk, b0, b1);
            if (!v0) { a0 = 0u; a1 = 0u; }
            if (!v1) { b0 = 0u; b1 = 0u; }
        }
        const unsigned lo0 = warp_transpose32(a0, lane), hi0 = warp_transpose32(b0, lane);
        const unsigned lo1 = warp_transpose32(a1, lane), hi1 = warp_transpose32(b1, lane);
        if (lane < nk) rows[(k0 + lane) * ld + w] = (unsigned long long)lo0 | ((unsigned long long)hi0 << 32);
        if (lane + 32 < nk)
            rows[(k0 + 32 + lane) * ld + w] = (unsigned long long)lo1 | ((unsigned long long)hi1 << 32);
    }
}

// The staged kernel for rows that start anywhere, last tile included.  A lane reads aligned chunks, the row's stream of bits is shifted to its
// start, one more chunk per row completing the piece; the last tile's pieces run
// into the next rows, its markers past m are not stored.  5,000 x 999,999: 1.60
// ms, 3.5 TB/s (11.3 ms with byte loads).
__global__ void __launch_bounds__(256) pack_hm_any_kernel(const uint8_t *hap01, int n, long long m, int W,
                                                          unsigned long long *rows, long long ld)
{
    __shared__ unsigned msk[64][kPackTile / 32 + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long tasks = (m + kPackTile - 1) / kPackTile * ld;
    const uint8_t *end = hap01 + (long long)n * m;
    for (long long t = blockIdx.x; t < tasks; t += gridDim.x) {
        const long long kb = t / ld;
        const long long w = t - kb * ld;
        const long long k0 = kb * kPackTile;
        if (w < W) {
            uint4 q[8];
            bool in[8];
            unsigned extra = 0u;                       // lane r: the chunk after row r's piece
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const long long h = 64 * w + 8 * warp + r;
                const uint8_t *src = hap01 + (h < n ? h : 0) * m + k0;
                const uint8_t *p = src - (int)((uintptr_t)src & 15u) + lane * 16;
                in[r] = p >= hap01 && p + 16 <= end;
                if (in[r]) q[r] = __ldg((const uint4 *)p);
            }
            if (lane < 8) {
                const long long h = 64 * w + 8 * warp + lane;
                const uint8_t *src = hap01 + (h < n ? h : 0) * m + k0;
                const uint8_t *p = src - (int)((uintptr_t)src & 15u) + kPackTile;
                if (p < end) extra = p + 16 <= end ? lsbs16(__ldg((const uint4 *)p)) : lsbs16_edge(p, hap01, end);
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const long long h = 64 * w + 8 * warp + r;
                const uint8_t *src = hap01 + (h < n ? h : 0) * m + k0;
                const int off = (int)((uintptr_t)src & 15u);
                const uint8_t *p = src - off + lane * 16;
                unsigned v = in[r] ? lsbs16(q[r]) : (p < end ? lsbs16_edge(p, hap01, end) : 0u);
                unsigned next = __shfl_down_sync(FULLMASK, v, 1);
                const unsigned ex = __shfl_sync(FULLMASK, extra, r);
                if (lane == 31) next = ex;
                v = h < n ? ((v | (next << 16)) >> off) & 0xFFFFu : 0u;
                const unsigned hi = __shfl_down_sync(FULLMASK, v, 1);
                if ((lane & 1) == 0) msk[8 * warp + r][lane >> 1] = v | (hi << 16);
            }
        }
        __syncthreads();
        unsigned a0 = 0u, a1 = 0u, b0 = 0u, b1 = 0u;
        if (w < W) {
            a0 = msk[lane][2 * warp];
            a1 = msk[lane][2 * warp + 1];
            b0 = msk[lane + 32][2 * warp];
            b1 = msk[lane + 32][2 * warp + 1];
        }
        __syncthreads();                               // the next tile may refill msk
        const unsigned lo0 = warp_transpose32(a0, lane), hi0 = warp_transpose32(b0, lane);
        const unsigned lo1 = warp_transpose32(a1, lane), hi1 = warp_transpose32(b1, lane);
        const long long k = k0 + 64 * warp + lane;
        if (k < m) rows[k * ld + w] = (unsigned long long)lo0 | ((unsigned long long)hi0 << 32);
        if (k + 32 < m) rows[(k + 32) * ld + w] = (unsigned long long)lo1 | ((unsigned long long)hi1 << 32);
    }
}

cudaError_t launch_pack(const uint8_t *hap01, int n, long long m, int hap_major,
                        unsigned long long *rows, long long ld, cudaStream_t s)
{
    const int W = (n + 63) / 64;
    // grid-stride: 16 CTAs of 8 warps per SM at most
    const long long cap = 16ll * device_sms();
    if (hap_major) {
        const bool aligned = m % 16 == 0 && ((uintptr_t)hap01 & 15) == 0;
        const long long tiles = (m + kPackTile - 1) / kPackTile;
        auto blocks = [&](long long tasks) { return (unsigned)(tasks < cap ? tasks : cap); };
        if (aligned && tiles > 1) {
            const long long kbeg = m / kPackTile * kPackTile;
            pack_hm_staged_kernel<<<blocks(m / kPackTile * ld), 256, 0, s>>>(hap01, n, m, W, rows, ld);
            if (kbeg < m)
                pack_hm_kernel<<<blocks(((m - kbeg + 63) / 64 * ld + 7) / 8), 256, 0, s>>>(hap01, n, m, W, rows, ld, kbeg);
        } else {
            pack_hm_any_kernel<<<blocks(tiles * ld), 256, 0, s>>>(hap01, n, m, W, rows, ld);
        }
    } else {
        const int S = n <= 16 * 8 - 15 ? 8 : n <= 16 * 16 - 15 ? 16 : 32;   // lanes a row
        long long blocks = S == 32 ? (m + 7) / 8 : (m + 1024 / S - 1) / (1024 / S);
        if (blocks > cap) blocks = cap;
        if (S == 8) pack_mm_small_kernel<8><<<(unsigned)blocks, 256, 0, s>>>(hap01, n, m, W, rows, ld);
        else if (S == 16) pack_mm_small_kernel<16><<<(unsigned)blocks, 256, 0, s>>>(hap01, n, m, W, rows, ld);
        else pack_mm_kernel<<<(unsigned)blocks, 256, 0, s>>>(hap01, n, m, W, rows, ld);
    }
    return cudaGetLastError();
}

}  // namespace selscan
