// Sorted-sweep form of the EHH walks (iHS Eq. 3-5, XPEHH Eq. 6-7).
//
// Every statistic of a walk is a function of S(i), the number of pairs of the
// walk's sample that are identical over the markers between the core and
// x_i (Section 1.2: EHH(x_i) = S(i) / C(N, 2)).  If the haplotypes are kept
// sorted by their sequence read outward from the core (the prefix order of a
// positional Burrows-Wheeler sweep), the haplotypes identical over
// [core, x_i] are contiguous runs of that order, and two neighbours t-1, t
// part at the first marker where they differ, i.e. at walk step M[t] = the
// length of their common run ending at the core.  So S(0) = C(n_c, 2) per
// core class, and step i only has to apply the boundaries t with M[t] = i:
// splitting a run [l, r) at t lowers S by (t - l)(r - t).  The cost of a walk
// becomes the number of boundaries it crosses, not the number of groups it
// carries at every step.
//
// Two kernels per stage:
//  * sweep_kernel: one CTA per chunk of cores and direction keeps the order A
//    and the run lengths M of all haplotypes in shared memory and advances them
//    marker by marker (a stable partition by allele; the new run length of a
//    neighbour pair is 1 + the minimum over the old pairs it spans).  At every
//    core of the stage it writes M, the class boundary n0 (and, for XPEHH, the
//    population of each sorted position) to a slot.  A chunk's state at its
//    first core holds `warmup` markers of history, so its sort is exact for
//    walks that stay within it: start_kernel sorts the haplotypes by that
//    history's 32-marker words directly (samples too large for its shared
//    memory take the history's markers through the sweep instead).
//  * split_walk_kernel: one warp per slot runs the walks of that core (both
//    allele classes of iHS, or the pooled XPEHH walk) 32 or 64 steps at a
//    time, lane l taking step l of the window: S of every step of the window
//    comes from one pass over the window's boundaries, then gaps, the map, the
//    cutoff and the trapezoid apply to all its steps at once, exactly as the
//    per-step walk applies them.  A walk that would step beyond its chunk's
//    history is handed to the per-step walk kernel (second pass).
#include <cooperative_groups.h>
#include <limits.h>

#include "../../include/selscan.h"
#include "device_common.cuh"
#include "internal.h"

namespace selscan {

namespace {

constexpr unsigned kInf16 = 0xFFFFu;
constexpr int kRowRing = 4;                 // rows in flight ahead of the sort (cp.async)
// Window boundaries a walking warp keeps on chip (a multiple of 4; a window with
// more new ones than that is not taken one boundary per lane), and the steps of a
// window after the first (whole blocks of 32).  An XPEHH boundary takes 8 bytes
// and its walks are short: 1,024 of them left too little of the SM's memory to L1
// for the slots the walk reads twice (1M: walks 17.2 ms; 512 and 32 steps, four CTAs
// per SM, 12.7).
__host__ __device__ constexpr int tok_smem(int xpehh) { return xpehh ? 512 : 1024; }
__host__ __device__ constexpr int win_steps(int xpehh) { return xpehh ? 32 : 64; }

__host__ __device__ inline int sweep_e(int n, int T)
{
    int e = (n + T - 1) / T;
    return (e + 3) & ~3;                    // a multiple of 4: elements are read 4 at a time
}
__host__ __device__ inline int sweep_npad(int n, int T) { return sweep_e(n, T) * T; }
__host__ __device__ inline int split_nw(int n) { return (n + 32) >> 5; }   // bits 0..n

// ---- prefix-state algebra of the stable partition --------------------------
// A segment of the current order summarised as: the running minimum of the
// run lengths since its last allele-0 / allele-1 element (or over the whole
// segment if it has none) -- the "tails" -- the minimum over the segment, the
// number of allele-0 elements, and whether each allele occurs.  Three words:
// A = tail0 | tail1 << 16; B = the minimum in both halves; C = zeros |
// seen0 << 15 | seen1 << 31 (zeros < 2^14; the flags sit on byte sign bits,
// so one byte permute in sign-replicate mode turns them into the halfword
// mask of the tails that R decides).  compose(L, R) replaces R by the summary
// of L followed by R: both tails are continued through R with one 16-bit
// SIMD minimum.
__device__ __forceinline__ unsigned seen_mask(unsigned c)
{
    unsigned r;   // bytes 0, 1 <- sign of byte 1 (seen0); bytes 2, 3 <- sign of byte 3 (seen1)
    asm("prmt.b32 %0, %1, 0, 0xBB99;" : "=r"(r) : "r"(c));
    return r;
}
__device__ __forceinline__ void compose(unsigned lA, unsigned lB, unsigned lC, unsigned &rA,
                                        unsigned &rB, unsigned &rC)
{
    const unsigned cont = __vminu2(lA, rB);                        // L's tails continued through R
    const unsigned keep = seen_mask(rC);                           // the tails R decides
    rA = (rA & keep) | (cont & ~keep);
    rB = __vminu2(lB, rB);
    rC = ((lC + rC) & 0x3FFFu) | ((lC | rC) & 0x80008000u);
}
constexpr unsigned kIdA = 0xFFFFFFFFu;
constexpr unsigned kIdB = 0xFFFFFFFFu;
constexpr unsigned kIdC = 0u;

// Asynchronous global -> shared copies of 8 bytes (rows start on 8-byte
// boundaries whatever their stride), in per-thread commit groups.
__device__ __forceinline__ void cp_async8(void *smem_dst, const void *gsrc)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

__device__ __forceinline__ unsigned bit_index(const SweepArgs &w, int h)
{
    // position of haplotype h (pooled numbering, A first) in the row's bits
    return h < w.a.nA ? (unsigned)h : (unsigned)(64 * w.a.WA + (h - w.a.nA));
}

}  // namespace

// Slot of one core: header {n0, history horizon, 0, 0}, the run lengths M and,
// for XPEHH, the population-A flags of the sorted positions.  M is kept in
// groups of 32 positions (16 words, u16 pairs): word j of group g holds the run
// lengths of positions 32 g + j (low half) and 32 g + 16 + j (high half), so
// that the walker turns a group into a 32-bit mask in position order with
// 16-bit SIMD operations alone.
namespace {
__host__ __device__ inline size_t slot_isa_at(int n) { return 16 + (size_t)((n + 31) / 32) * 64; }
}  // namespace

size_t sweep_smem_bytes(int n, int W, int T, int R)
{
    const int W32 = ((2 * W) + 4) & ~3;
    return (size_t)sweep_npad(n, T) * 4 * 2 + (size_t)W32 * 4 * kRowRing + T / 32 * 12 +
           (size_t)((R + 31) / 32) * 4;
}

size_t sweep_slot_bytes(int n, int xpehh)
{
    // a multiple of 16 bytes: every slot's M region is read and written in 16-byte units
    return slot_isa_at(n) + (xpehh ? (((size_t)split_nw(n) * 4 + 15) & ~(size_t)15) : 0);
}

size_t sweep_state_bytes(int n, int T) { return (size_t)sweep_npad(n, T) * 4; }
__host__ __device__ size_t sweep_elements(int n, int T) { return (size_t)sweep_npad(n, T); }


// ---- the sweep ---------------------------------------------------------------
// Shared memory: two buffers of np packed elements (bit index of the haplotype
// in the row | run length with its predecessor << 16), a ring of kRowRing row
// buffers (filled by cp.async, each with one extra all-ones word), the warp
// totals and the stage's core bitmap.  Positions n..np-1 hold padding elements whose allele is that
// all-ones word: they sort after every real haplotype and never touch a real
// element's run length.  T threads (32 to 512); EMAX bounds the elements per
// thread (at most 32, one allele bit each in a 32-bit mask), up to 24 stay in
// registers between the two passes.
// XP: 1 an XPEHH scan, 0 iHS, -1 told by nB.
// `sync` is a barrier of the T threads that sort; `done(r)` is called once every
// thread has written its part of the slots of the stage's first r markers.
template <int T, int EMAX, bool EXACT, int XP, class Sync, class Done>
__device__ __forceinline__ void sort_chunk(const SweepArgs &w, unsigned char *smem, int dir, long long c0,
                                           long long c1, int blk, Sync sync, Done done)
{
    constexpr bool CACHE = EMAX <= 24;
    const int n = w.n;
    // EXACT: every thread holds exactly EMAX elements (no per-element guards)
    const int E = EXACT ? EMAX : sweep_e(n, T);
    const int np = E * T;
    const int W32 = 2 * w.a.W;
    const int W32r = (W32 + 4) & ~3;             // >= W32 + 1
    const unsigned pad_bi = 32u * (unsigned)W32; // bit index of the padding elements
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NW = T / 32;
    unsigned *P0 = (unsigned *)smem;             // buffer b at P0 + b * np
    unsigned *R0 = P0 + 2 * np;                  // row ring: slot r at R0 + r * W32r
    unsigned *wsum = R0 + kRowRing * W32r;
    unsigned *cbits = wsum + 3 * NW;             // the stage's cores that pass the filter

    // dir 0: walks toward lower indices.  The chunk covers cores [c0, c1); blk is
    // the index of its state and of its slots
    const long long m = w.a.m;
    long long klo, khi;                          // this stage's cores [klo, khi)
    if (dir == 0) {
        klo = c0 + (long long)w.stage * w.R;
        khi = klo + w.R < c1 ? klo + w.R : c1;
        if (klo >= c1) return;
    } else {
        khi = c1 - (long long)w.stage * w.R;
        klo = khi - w.R > c0 ? khi - w.R : c0;
        if (khi <= c0) return;
    }
    // history origin of the chunk: the sort is exact for runs inside it
    const long long s0 = c0 - w.L > 0 ? c0 - w.L : 0;
    const long long e0 = c1 - 1 + w.L < m - 1 ? c1 - 1 + w.L : m - 1;
    long long xfirst, xlast;                     // markers of this launch, in sweep order
    if (dir == 0) {
        xfirst = w.stage == 0 && !w.started ? s0 : klo;
        xlast = khi - 1;
    } else {
        xfirst = w.stage == 0 && !w.started ? e0 : khi - 1;
        xlast = klo;
    }
    const long long step = dir == 0 ? 1 : -1;
    unsigned *st = (unsigned *)w.st + (size_t)blk * np;

    // ---- state in: the identity order, the chunk's starting state, or the last stage's
    if (w.stage == 0 && !w.started) {
        for (int t = tid; t < np; t += T) P0[t] = t < n ? bit_index(w, t) : pad_bi;
    } else {
        for (int t = tid; t < np; t += T) P0[t] = st[t];
    }
    const unsigned long long *hap64 = (const unsigned long long *)w.a.hap;
    const long long ld = w.a.ld;
    const int W = w.a.W;
    const long long nq = (xlast - xfirst) * step + 1;   // markers of this launch
    // row q (in sweep order) goes to ring slot q % kRowRing, kRowRing - 1 rows ahead
    auto fetch_row = [&](long long q) {
        if (q < nq) {
            unsigned *dst = R0 + (q & (kRowRing - 1)) * W32r;
            const unsigned long long *src = hap64 + (xfirst + q * step) * ld;
            for (int t = tid; t < W; t += T) cp_async8(dst + 2 * t, src + t);
        }
        cp_async_commit();
    };
    for (int q = 0; q < kRowRing; ++q) fetch_row(q);
    for (int r = 0; r < kRowRing; ++r)          // the padding elements' all-ones word
        if (tid < W32r - W32) R0[r * W32r + W32 + tid] = 0xFFFFFFFFu;
    {
        const int nrc = (int)(khi - klo);
        for (int r0 = 0; r0 < nrc; r0 += T) {
            const int r = r0 + tid;
            const bool v = r < nrc && w.sk.core_status[klo + r] != (int8_t)SELSCAN_LOCUS_MAF_FILTERED;
            const unsigned bits = __ballot_sync(FULLMASK, v);
            if (lane == 0 && r0 + warp * 32 < nrc) cbits[(r0 >> 5) + warp] = bits;
        }
    }
    cp_async_wait<kRowRing - 1>();               // row 0
    sync();

    int cur = 0;
    const int base = tid * E;
    unsigned val[CACHE ? EMAX : 1];
    long long q = 0;
    for (long long x = xfirst;; x += step, ++q) {
        const bool more = x != xlast;
        const bool is_core = x >= klo && x < khi;
        const bool wr = is_core && ((cbits[(x - klo) >> 5] >> ((x - klo) & 31)) & 1u);

        const unsigned *Pc = P0 + cur * np;
        const unsigned *row = R0 + (q & (kRowRing - 1)) * W32r;
        // pass 1: alleles, the new run lengths as far as this segment decides
        // them, and the segment summary.  Both tails live in one word (allele
        // 0 low, 1 high).  Run lengths stay at most 65,000 (a chunk plus its
        // warm-up spans at most 65,000 markers), so adding one to each half
        // never carries.  The first element of each allele in the segment gets
        // its prefix tail after placement.
        unsigned vmask = 0u, allw = 0xFFFFFFFFu, mn01 = 0xFFFFFFFFu;
#pragma unroll
        for (int e = 0; e < EMAX; e += 4) {
            if (e < E) {
                // 16-byte loads: a thread's segment starts at 16 E bytes, and
                // eight lanes at that stride cover distinct banks
                const uint4 q = *(const uint4 *)(Pc + base + e);
                const unsigned q4[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const unsigned pv = q4[h];
                    // the word of bit index pv & 0xFFFF, (pv & 0xFFFF) >> 5, by multiplies
                    const unsigned wd = row[__umulhi(pv * 65536u, 2048u)];
                    const unsigned v = __funnelshift_r(wd, wd, pv) & 1u;   // bit pv % 32
                    vmask = vmask + vmask + v;            // element e at bit E - 1 - e
                    allw = min(allw, pv);                 // high half: the segment minimum
                    mn01 = __vminu2(mn01, __byte_perm(pv, 0u, 0x3232u));
                    // the selector by multiply-add (v ? 0x7610 : 0x5410), and the tail
                    // of allele v restarted by a 16x2 maximum with 0xFFFF in its half
                    if (CACHE) val[e + h] = __byte_perm(pv, mn01 + 0x00010001u, 0x5410u + v * 0x2200u);
                    mn01 = __vmaxu2(mn01, 0x0000FFFFu + v * 0xFFFE0001u);
                }
            }
        }
        const unsigned ones = (unsigned)__popc(vmask);
        vmask <<= 32 - E;                         // element e at bit 31 - e
        const unsigned zeros = (unsigned)E - ones;
        const unsigned hp0 = zeros != 0u, hp1 = ones != 0u;
        unsigned p0 = mn01;
        unsigned p1 = (allw >> 16) * 0x00010001u;
        unsigned p2 = zeros | (hp0 << 15) | (hp1 << 31);
        // warp inclusive scan
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned o0 = __shfl_up_sync(FULLMASK, p0, d);
            const unsigned o1 = __shfl_up_sync(FULLMASK, p1, d);
            const unsigned o2 = __shfl_up_sync(FULLMASK, p2, d);
            if (lane >= d) compose(o0, o1, o2, p0, p1, p2);
        }
        unsigned x0 = __shfl_up_sync(FULLMASK, p0, 1), x1 = __shfl_up_sync(FULLMASK, p1, 1);
        unsigned x2 = __shfl_up_sync(FULLMASK, p2, 1);
        if (lane == 0) { x0 = kIdA; x1 = kIdB; x2 = kIdC; }
        if (lane == 31) { wsum[3 * warp] = p0; wsum[3 * warp + 1] = p1; wsum[3 * warp + 2] = p2; }
        sync();
        if (is_core) done(dir == 0 ? (int)(x - klo) : (int)(khi - 1 - x));
        fetch_row(q + kRowRing);                  // every thread is done with this row's slot
        // every warp scans the warp totals: its own prefix and the block total
        unsigned q0 = lane < NW ? wsum[3 * lane] : kIdA;
        unsigned q1 = lane < NW ? wsum[3 * lane + 1] : kIdB;
        unsigned q2 = lane < NW ? wsum[3 * lane + 2] : kIdC;
#pragma unroll
        for (int d = 1; d < NW; d <<= 1) {
            const unsigned o0 = __shfl_up_sync(FULLMASK, q0, d);
            const unsigned o1 = __shfl_up_sync(FULLMASK, q1, d);
            const unsigned o2 = __shfl_up_sync(FULLMASK, q2, d);
            if (lane >= d) compose(o0, o1, o2, q0, q1, q2);
        }
        unsigned w0 = __shfl_sync(FULLMASK, q0, (warp + 31) & 31);
        unsigned w1 = __shfl_sync(FULLMASK, q1, (warp + 31) & 31);
        unsigned w2 = __shfl_sync(FULLMASK, q2, (warp + 31) & 31);
        if (warp == 0) { w0 = kIdA; w1 = kIdB; w2 = kIdC; }
        const unsigned tot2 = __shfl_sync(FULLMASK, q2, NW - 1);
        const unsigned n0 = tot2 & 0x3FFFu;
        compose(w0, w1, w2, x0, x1, x2);          // this thread's exclusive prefix
        // pass 2: place the elements; the first allele-0 / allele-1 element of
        // the segment takes its run length from the prefix (0 if it is the
        // first of its allele overall)
        const unsigned zs = x2 & 0x3FFFu;
        const unsigned os = n0 + (unsigned)base - zs;
        unsigned z = zs, o = os;
        unsigned *Pn = P0 + (cur ^ 1) * np;
        if (CACHE) {
            // allele-0 elements go to zs + (elements so far) - (ones so far)
            const unsigned zk = zs + os;
#pragma unroll
            for (int e = 0; e < EMAX; ++e) {
                if (e < E) {
                    const unsigned one = (vmask >> (31 - e)) & 1u;
                    Pn[one ? o : zk + (unsigned)e - o] = val[CACHE ? e : 0];
                    o += one;
                }
            }
        }
        if (!CACHE) {
            // second sweep over the segment for the run lengths (large samples)
            unsigned a0 = x0 & 0xFFFFu, a1 = x0 >> 16;
            unsigned h0 = (x2 >> 15) & 1u, h1 = x2 >> 31;
            z = zs;
            o = os;
            for (int e = 0; e < E; ++e) {
                const unsigned q = Pc[base + e];
                const unsigned mv = q >> 16;
                a0 = min(a0, mv);
                a1 = min(a1, mv);
                const unsigned one = (vmask >> (31 - e)) & 1u;
                const unsigned mnv = one ? a1 : a0;
                const unsigned hpv = one ? h1 : h0;
                const unsigned out = hpv ? min(mnv + 1u, kInf16) : 0u;
                const unsigned p = one ? o : z;
                o += one;
                z += one ^ 1u;
                a1 = one ? kInf16 : a1;
                a0 = one ? a0 : kInf16;
                h1 |= one;
                h0 |= one ^ 1u;
                Pn[p] = (q & 0xFFFFu) | (out << 16);
            }
        } else {
            // the first allele-0 / allele-1 element of the segment (placed at zs
            // / os): 1 + the minimum over the prefix tail and its own span
            if (hp0) {
                const unsigned u = Pn[zs];
                const unsigned out = ((x2 >> 15) & 1u) ? min((x0 & 0xFFFFu) + 1u, u >> 16) : 0u;
                Pn[zs] = (u & 0xFFFFu) | (out << 16);
            }
            if (hp1) {
                const unsigned u = Pn[os];
                const unsigned out = (x2 >> 31) ? min((x0 >> 16) + 1u, u >> 16) : 0u;
                Pn[os] = (u & 0xFFFFu) | (out << 16);
            }
        }
        cp_async_wait<kRowRing - 1>();           // row q + 1 has landed
        sync();
        cur ^= 1;

        // ---- a core of this stage: hand its sorted state to the walk
        if (wr) {
            const int r = dir == 0 ? (int)(x - klo) : (int)(khi - 1 - x);
            unsigned char *slot = w.slots + ((size_t)blk * w.R + r) * w.slot_bytes;
            const bool xp = XP < 0 ? w.a.nB > 0 : XP == 1;
            if (tid == 0) {
                int *hdr = (int *)slot;
                hdr[0] = (int)n0;
                long long hz;
                if (dir == 0) hz = s0 == 0 ? INT_MAX : x - s0;
                else hz = e0 == m - 1 ? INT_MAX : e0 - x;
                hdr[1] = (int)hz;
            }
            const unsigned *Ps = P0 + cur * np;
            // run lengths, 8 per 16-byte store (the padding elements fill the last
            // group; np is a multiple of 32).  Nothing waits for the stores: the
            // next marker's partition reads this buffer and writes the other one.
            // XPEHH: the same thread makes the population flags of its 8 positions
            // (16x2 clamps of the bit indices, as the walker marks windows) and four
            // neighbours' make a word: a third of the instructions of a ballot per
            // word (1M: sort 19.0 -> 17.5 ms)
            const uint4 *P4 = (const uint4 *)Ps;
            uint4 *M4 = (uint4 *)(slot + 16);
            const int items = (n + 31) / 32 * 4;
            if (!xp) {
                for (int t = tid; t < items; t += T) {
                    const uint4 lo = P4[(t >> 2) * 8 + (t & 3)], hi = P4[(t >> 2) * 8 + 4 + (t & 3)];
                    M4[t] = make_uint4(__byte_perm(lo.x, hi.x, 0x7632u), __byte_perm(lo.y, hi.y, 0x7632u),
                                       __byte_perm(lo.z, hi.z, 0x7632u), __byte_perm(lo.w, hi.w, 0x7632u));
                }
            } else {
                unsigned *isA = (unsigned *)(slot + slot_isa_at(n));
                const unsigned L = 64u * (unsigned)w.a.WA * 0x00010001u, L1 = L - 0x00010001u;
                for (int t0 = 0; t0 < items; t0 += T) {      // whole warps: items is a multiple of 4
                    const int t = t0 + tid;
                    unsigned f = 0u;                          // bits j, 16 + j: the position is in B
                    if (t < items) {
                        const uint4 lo = P4[(t >> 2) * 8 + (t & 3)], hi = P4[(t >> 2) * 8 + 4 + (t & 3)];
                        M4[t] = make_uint4(__byte_perm(lo.x, hi.x, 0x7632u), __byte_perm(lo.y, hi.y, 0x7632u),
                                           __byte_perm(lo.z, hi.z, 0x7632u), __byte_perm(lo.w, hi.w, 0x7632u));
                        f = __vmaxu2(__vminu2(__byte_perm(lo.w, hi.w, 0x5410u), L), L1) - L1;
                        f = f + f + (__vmaxu2(__vminu2(__byte_perm(lo.z, hi.z, 0x5410u), L), L1) - L1);
                        f = f + f + (__vmaxu2(__vminu2(__byte_perm(lo.y, hi.y, 0x5410u), L), L1) - L1);
                        f = f + f + (__vmaxu2(__vminu2(__byte_perm(lo.x, hi.x, 0x5410u), L), L1) - L1);
                        f = (f ^ 0x000F000Fu) << (4 * (t & 3));
                    }
                    f |= __shfl_xor_sync(FULLMASK, f, 1);
                    f |= __shfl_xor_sync(FULLMASK, f, 2);
                    if (t < items && (t & 3) == 0) isA[t >> 2] = f;
                }
                if (tid == 0 && (n & 31) == 0) isA[n >> 5] = 0u;   // the word of position n
            }
        }
        if (!more) break;
    }
    // ---- state out for the next stage
    if (w.stage + 1 < w.nstages) {
        const unsigned *Ps = P0 + cur * np;
        for (int t = tid; t < np; t += T) st[t] = Ps[t];
    }
}

template <int T, int EMAX, bool EXACT = false, int XP = -1>
__global__ void __launch_bounds__(T, T == 512 ? 2 : (T == 256 ? 3 : 512 / T)) sweep_kernel(SweepArgs w)
{
    extern __shared__ __align__(16) unsigned char smem[];
    if (w.quit && *w.quit >= 6) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) *w.walk_head = 0ull;   // the next walk launch's slot counter
    const int dir = blockIdx.x / w.nch, c = blockIdx.x % w.nch;
    const long long c0 = w.a.k0 + (long long)c * w.B;   // chunk c of [k0, k1)
    if (c0 >= w.a.k1) return;
    const long long c1 = c0 + w.B < w.a.k1 ? c0 + w.B : w.a.k1;
    sort_chunk<T, EMAX, EXACT, XP>(w, smem, dir, c0, c1, blockIdx.x, [] { __syncthreads(); }, [](int) {});
}

// ---- the split walk ----------------------------------------------------------
namespace {

// Per-warp shared memory: the window's boundaries in position order (position |
// M << 16) with, for XPEHH, the number of population-A haplotypes before each;
// the run starts older than the window (O) and those of it (N) as bitmaps over
// positions 0..n, one summary bit per non-zero word of O (S); the drops of S
// per step of a sparse window; and for XPEHH the population-A flags of the
// sorted positions with their per-word prefix counts.
struct SplitSmem {
    unsigned *tk;                         // window list on chip, first tok_smem entries (XPEHH: pairs)
    unsigned *gtk;                        // the rest, global: entry k at gtk[k]
    unsigned *O, *N, *S, *dec;
    unsigned *isA, *PA;
    int nw, ns;
};

__host__ __device__ inline int split_words(int n, int xpehh)
{
    const int nw = split_nw(n), ns = (nw + 31) >> 5;
    return tok_smem(xpehh) * (xpehh ? 2 : 1) + 2 * nw + ns + win_steps(xpehh) * (xpehh ? 3 : 2) + (xpehh ? 2 * nw : 0);
}

__device__ inline SplitSmem split_smem(unsigned char *base, unsigned char *scratch, int n, int xpehh)
{
    SplitSmem s;
    s.nw = split_nw(n);
    s.ns = (s.nw + 31) >> 5;
    unsigned *p = (unsigned *)base;
    s.tk = p; p += tok_smem(xpehh) * (xpehh ? 2 : 1);
    s.dec = p; p += win_steps(xpehh) * (xpehh ? 3 : 2);
    s.O = p; p += s.nw;
    s.N = p; p += s.nw;
    s.S = p; p += s.ns;
    s.isA = p; p += xpehh ? s.nw : 0;
    s.PA = p;
    s.gtk = (unsigned *)scratch;
    return s;
}

__device__ __forceinline__ int c2i(unsigned k) { return (int)(k * (k - 1u) / 2u); }

// Bitmap searches with a third level: `sup` has bit q set when summary word q
// is non-zero (at most 16 summary words: n <= 16383), so neither search loops.
// last set position < b (b > 0; position 0 is always set)
__device__ __forceinline__ int prev_start(const unsigned *B, const unsigned *S, unsigned sup, int b)
{
    const int wd = b >> 5;
    const unsigned bits = B[wd] & ((1u << (b & 31)) - 1u);
    if (bits) return (wd << 5) + 31 - __clz(bits);
    const int sw = wd - 1;                       // >= 0: word 0 holds position 0
    int q = sw >> 5;
    unsigned sb = S[q] & (0xFFFFFFFFu >> (31 - (sw & 31)));
    if (!sb) {                                   // q > 0 here: summary word 0 has bit 0
        q = 31 - __clz(sup & ((1u << q) - 1u));
        sb = S[q];
    }
    const int ww = (q << 5) + 31 - __clz(sb);
    return (ww << 5) + 31 - __clz(B[ww]);
}

// first set position > b (b < n; position n is always set)
__device__ __forceinline__ int next_start(const unsigned *B, const unsigned *S, unsigned sup, int b)
{
    const int wd = b >> 5;
    const unsigned bits = B[wd] & ~((2u << (b & 31)) - 1u);
    if (bits) return (wd << 5) + __ffs(bits) - 1;
    const int sw = wd + 1;                       // a word up to the one of position n
    int q = sw >> 5;
    unsigned sb = S[q] & (0xFFFFFFFFu << (sw & 31));
    if (!sb) {
        q = __ffs(sup & ~((2u << q) - 1u)) - 1;
        sb = S[q];
    }
    const int ww = (q << 5) + __ffs(sb) - 1;
    return (ww << 5) + __ffs(B[ww]) - 1;
}

__device__ __forceinline__ unsigned count_a(const SplitSmem &s, int x)
{
    return s.PA[x >> 5] + (unsigned)__popc(s.isA[x >> 5] & ((1u << (x & 31)) - 1u));
}

// The run boundaries of a window in position order: positions t with M[t] <=
// hi (ALL), or only those that are no older run start (M[t] >= the window's
// first step).  Each lane turns 32 neighbouring run lengths into a bitmap word:
// the 16x2 clamp to [hi, hi + 1] less hi leaves the bit "not yet parted", the
// slot's layout puts the bits in position order.  `merge` first adds the
// previous window's boundaries (N) to the older run starts (O).  Only positions
// in [pa, pb) are looked at (the classes whose walks still run).  Returns the
// number of boundaries, K0 of them before position n0; sup gets one bit per
// summary word of O (at most 17 words: n <= 16383).
template <int NPOP, typename Tile>
__device__ __forceinline__ unsigned mark_window(const Tile &tile, const SplitSmem &s, const uint4 *M4,
                                                int n, int n0, int hi, bool all, bool merge,
                                                int pa, int pb, unsigned &K0, unsigned &sup)
{
    const int lane = tile.thread_rank();
    const unsigned short *M16 = (const unsigned short *)M4;
    const unsigned PP = (unsigned)(hi + 1) * 0x00010001u, P1 = PP - 0x00010001u;
    unsigned K = 0u, c0 = 0u;
    sup = 0u;
    for (int it = 0; it < s.ns; ++it) {
        const int wd = it * 32 + lane;
        unsigned o = 0u, hit = 0u;
        if (wd < s.nw) {
            o = s.O[wd];
            if (merge) {
                o |= s.N[wd];
                s.O[wd] = o;
            }
            if (32 * wd < pb && 32 * wd + 32 > pa) {
                uint4 q[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) q[u] = M4[4 * wd + u];
                unsigned acc = 0u;               // word j's bits land at j and 16 + j
#pragma unroll
                for (int u = 3; u >= 0; --u) {
                    acc = acc + acc + (__vmaxu2(__vminu2(q[u].w, PP), P1) - P1);
                    acc = acc + acc + (__vmaxu2(__vminu2(q[u].z, PP), P1) - P1);
                    acc = acc + acc + (__vmaxu2(__vminu2(q[u].y, PP), P1) - P1);
                    acc = acc + acc + (__vmaxu2(__vminu2(q[u].x, PP), P1) - P1);
                }
                hit = ~acc & (pb - 32 * wd >= 32 ? 0xFFFFFFFFu : (1u << (pb - 32 * wd)) - 1u);
                if (pa > 32 * wd) hit &= 0xFFFFFFFFu << (pa - 32 * wd);
                s.N[wd] = hit & ~o;
                if (!all) hit &= ~o;
            }
        }
        const unsigned bal = tile.ballot(o != 0u);
        if (lane == 0) s.S[it] = bal;
        sup |= bal ? 1u << it : 0u;
        const int below = n0 - 32 * wd;          // positions of this word before n0
        c0 += (unsigned)__popc(hit & (below >= 32 ? 0xFFFFFFFFu : below > 0 ? (1u << below) - 1u : 0u));
        const unsigned c = (unsigned)__popc(hit);
        unsigned incl = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned v = tile.shfl_up(incl, d);
            if (lane >= d) incl += v;
        }
        unsigned at = K + incl - c;
        while (hit) {
            const int b = __ffs(hit) - 1;
            hit &= hit - 1u;
            const int t = 32 * wd + b;
            const unsigned tok = (unsigned)t | ((unsigned)M16[32 * wd + ((b & 15) << 1 | b >> 4)] << 16);
            unsigned *dst = at < (unsigned)tok_smem(NPOP == 2) ? s.tk : s.gtk;
            if (NPOP == 2) *(uint2 *)(dst + 2 * at) = make_uint2(tok, count_a(s, t));
            else dst[at] = tok;
            ++at;
        }
        K += tile.shfl(incl, 31);
    }
    K0 = (unsigned)__reduce_add_sync(0xFFFFFFFFu, (int)c0);
    tile.sync();
    return K;
}

// Sums of squared run lengths over the list entries [ka, kb), cut at the
// boundaries of steps up to this lane's step (token < lim): d[0] all
// haplotypes, for XPEHH d[1] population A, d[2] population B.  last / lastA:
// the run start so far (position, population-A haplotypes before it).
template <int NPOP>
struct RunCut {
    unsigned lim, last, lastA, d[NPOP == 2 ? 3 : 1];
    __device__ __forceinline__ void cut(unsigned t, unsigned ta)
    {
        const unsigned p = t & 0xFFFFu, l = p - last;
        if (NPOP == 2) {
            const unsigned la = ta - lastA, lb = l - la;
            if (t < lim) {
                d[0] += l * l;
                d[NPOP == 2 ? 1 : 0] += la * la;
                d[NPOP == 2 ? 2 : 0] += lb * lb;
                last = p;
                lastA = ta;
            }
        } else if (t < lim) {
            d[0] += l * l;
            last = p;
        }
    }
    // list entry k
    __device__ __forceinline__ void one(const SplitSmem &s, unsigned k)
    {
        const unsigned *src = k < (unsigned)tok_smem(NPOP == 2) ? s.tk : s.gtk;
        if (NPOP == 2) {
            const uint2 t = *(const uint2 *)(src + 2 * k);
            cut(t.x, t.y);
        } else {
            cut(src[k], 0u);
        }
    }
    // iHS: entries [ka, kb), upward
    __device__ __forceinline__ void range(const SplitSmem &s, unsigned ka, unsigned kb)
    {
        unsigned k = ka;
        const unsigned kv = kb < (unsigned)tok_smem(NPOP == 2) ? kb : (unsigned)tok_smem(NPOP == 2);
        for (; k < kv && (k & 3u); ++k) one(s, k);
#pragma unroll 2
        for (; k + 4 <= kv; k += 4) {
            const uint4 t = *(const uint4 *)(s.tk + k);
            cut(t.x, 0u);
            cut(t.y, 0u);
            cut(t.z, 0u);
            cut(t.w, 0u);
        }
        for (; k < kb; ++k) one(s, k);
    }
    // XPEHH: entries [0, K) from both ends at once: the lower half of the warp
    // runs upward from position 0, the upper half downward from position n (the
    // squares do not see the sign); the run between their last cuts closes it
    template <typename Tile>
    __device__ __forceinline__ void both_ends(const Tile &tile, const SplitSmem &s, unsigned K, unsigned n,
                                              unsigned nA)
    {
        const bool up = tile.thread_rank() < 16;
        last = up ? 0u : n;
        lastA = up ? 0u : nA;
        const unsigned half = K >> 1;
        if (K <= (unsigned)tok_smem(NPOP == 2)) {
            const uint2 *q = (const uint2 *)s.tk + (up ? 0u : K - 1u);
            const int st = up ? 1 : -1;
#pragma unroll 4
            for (unsigned x = 0; x < half; ++x, q += st) cut(q->x, q->y);
        } else {
            for (unsigned x = 0; x < half; ++x) one(s, up ? x : K - 1u - x);
        }
        if ((K & 1u) && up) one(s, half);
        const unsigned l = last - (unsigned)__shfl_xor_sync(0xFFFFFFFFu, last, 16);
        const unsigned la = lastA - (unsigned)__shfl_xor_sync(0xFFFFFFFFu, lastA, 16), lb = l - la;
#pragma unroll
        for (int q = 0; q < (NPOP == 2 ? 3 : 1); ++q) d[q] += __shfl_xor_sync(0xFFFFFFFFu, d[q], 16);
        d[0] += l * l;
        d[NPOP == 2 ? 1 : 0] += la * la;
        d[NPOP == 2 ? 2 : 0] += lb * lb;
    }
};

// Drops of S by step (s.dec) from a window's K new boundaries, one per lane:
// the pairs whose common run ends exactly at step v are counted once, at the
// leftmost boundary b of their span with M[b] = v: the first member lies in
// [p, b), p the last run start before b with M <= v, the second in [b, e), e
// the first run start after b with M < v.  p and e are the nearest older run
// start (bitmap O) or a nearer boundary of the window itself (the neighbours
// in the list).  So boundary b removes (b - p)(e - b) pairs at step v, and per
// population the products of its members on either side.
template <int NPOP, typename Tile>
__device__ __forceinline__ void sparse_terms(const Tile &tile, const SplitSmem &s, unsigned K, int lo, int n0,
                                             unsigned sup)
{
    constexpr int kWin = win_steps(NPOP == 2);
    const int lane = tile.thread_rank();
    for (int q = lane; q < kWin * (NPOP == 2 ? 3 : 2); q += 32) s.dec[q] = 0u;
    tile.sync();
    for (unsigned k = lane; k < K; k += 32) {
        const unsigned t = s.tk[NPOP * k];
        const int b = (int)(t & 0xFFFFu);
        const unsigned v = t >> 16;
        int p = prev_start(s.O, s.S, sup, b), e = next_start(s.O, s.S, sup, b);
        for (int q = (int)k - 1; q >= 0; --q) {
            const unsigned u = s.tk[NPOP * q];
            const int x = (int)(u & 0xFFFFu);
            if (x < p) break;
            if (u >> 16 <= v) { p = x; break; }
        }
        for (unsigned q = k + 1; q < K; ++q) {
            const unsigned u = s.tk[NPOP * q];
            const int x = (int)(u & 0xFFFFu);
            if (x > e) break;
            if (u >> 16 < v) { e = x; break; }
        }
        unsigned *dec = s.dec + (v - (unsigned)lo);
        const unsigned dd = (unsigned)((b - p) * (e - b));
        if (NPOP == 2) {
            const unsigned ab = s.tk[NPOP * k + 1];
            const unsigned la = ab - count_a(s, p), ra = count_a(s, e) - ab;
            atomicAdd(dec, la * ra);
            atomicAdd(dec + kWin, ((unsigned)(b - p) - la) * ((unsigned)(e - b) - ra));
            atomicAdd(dec + 2 * kWin, dd);
        } else {
            atomicAdd(dec + (b < n0 ? 0 : kWin), dd);
        }
    }
    tile.sync();
}

// iHS, windows of kNarrow steps: S of the two classes at the step of this lane
// (number lane mod 8 of the window; M <= that step <=> token < lim) from the K
// listed boundaries, K0 of class 0.  Four lanes a step run over a quarter of a
// class's list each; their first and last cuts join the quarters.
constexpr int kNarrow = 8;
__device__ __forceinline__ uint2 narrow_counts(const unsigned *tk, const unsigned *gtk, unsigned K0, unsigned K,
                                            unsigned n0, unsigned n, unsigned lim)
{
    constexpr unsigned kTok = (unsigned)tok_smem(0), kNone = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    unsigned S[2];
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
        const unsigned ka = c ? K0 : 0u, kb = c ? K : K0, start = c ? n0 : 0u, end = c ? n : n0;
        const unsigned per = (kb - ka + 3u) / 4u, from = ka + (unsigned)(lane >> 3) * per;
        unsigned d = 0u, last = 0u, first = kNone;
        if (K <= kTok) {
#pragma unroll 4
            for (unsigned x = 0; x < per; ++x) {
                const unsigned k = from + x, t = k < kb ? tk[k] : kNone;
                if (t < lim) {
                    const unsigned p = t & 0xFFFFu, l = p - last;
                    d += l * l;
                    first = min(first, p);
                    last = p;
                }
            }
        } else {
#pragma unroll 4
            for (unsigned x = 0; x < per; ++x) {
                const unsigned k = from + x, t = k < kb ? (k < kTok ? tk : gtk)[k] : kNone;
                if (t < lim) {
                    const unsigned p = t & 0xFFFFu, l = p - last;
                    d += l * l;
                    first = min(first, p);
                    last = p;
                }
            }
        }
        unsigned sum = 0u, cur = start;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int src = (lane & 7) + 8 * q;
            const unsigned f = __shfl_sync(0xFFFFFFFFu, first, src), e = __shfl_sync(0xFFFFFFFFu, last, src);
            const unsigned dq = __shfl_sync(0xFFFFFFFFu, d, src);
            if (f != kNone) {                         // a quarter's first cut was measured from 0
                sum += dq - f * f + (f - cur) * (f - cur);
                cur = e;
            }
        }
        sum += (end - cur) * (end - cur);
        S[c] = (sum - (end - start)) >> 1;
    }
    return make_uint2(S[0], S[1]);
}

}  // namespace

size_t split_smem_per_warp(int n, int xpehh)
{
    return ((size_t)split_words(n, xpehh) * 4 + 15) & ~(size_t)15;
}

// the list holds at most n boundaries, the first tok_smem of them on chip
size_t split_scratch_per_warp(int n) { return n <= tok_smem(1) ? 0 : (((size_t)n * 8) + 255) & ~(size_t)255; }

// The walks of one core, by one warp.  The first window is the steps 1..32:
// every lane runs over all boundaries with M <= 32 (shared memory, broadcast
// reads) and cuts at those of its own step, so S(i) = (sum of squared run
// lengths - haplotypes) / 2 of 32 steps costs about six instructions per
// boundary, where a step at a time needs two bitmap searches, three shared
// atomics and two warp sums per step with most lanes idle (1M iHS: 13.5 ms ->
// 7.4).  The pooled XPEHH walk, three counts per boundary and few steps long,
// takes 16 steps at a time, two lanes a step from both ends of the list (1M:
// 17.2 ms against 24.1 with 32; 12.7 since its list is shorter, tok_smem).  Later
// windows (win_steps) hold few boundaries among many older run starts: there each lane takes one boundary
// (sparse_terms); a window with more than tok_smem of them is cut like the
// first one.  NARROW (iHS): windows of kNarrow steps instead, for slots most of
// whose boundaries part within the first 32 steps (wide_slot).
// Pair counts fit 32 bits (C(16383, 2) < 2^32); the digest is 64-bit.  Lane
// (i - 1) mod 32 adds step i's trapezoid term to its own FP64 partial sum, and
// the partial sums meet in a fixed butterfly when the walk ends: the order of
// the per-step walk, so a walk handed over to it gives the same bits.
template <int NPOP, bool NARROW = false, typename Tile>
__device__ __forceinline__ void walk_slot(const SweepArgs &w, const Tile &tile, const SplitSmem &s,
                                          const unsigned char *slot, long long k, int dir)
{
    constexpr int G = 32;
    constexpr int NV = NPOP == 2 ? 3 : 2;     // S values: class 0, class 1; or A, B, pooled
    constexpr int NWK = NPOP == 2 ? 1 : 2;    // walks of a slot
    constexpr int kDense = NARROW ? kNarrow : NPOP == 2 ? 16 : 32;   // steps of a window cut boundary by boundary
    constexpr int kWin = win_steps(NPOP == 2);    // and of one taken one boundary per lane
    const int lane = tile.thread_rank();
    const int n = w.n;
    const long long m = w.a.m;
    const int n0 = ((const int *)slot)[0];
    const int hz = ((const int *)slot)[1];
    const uint4 *M4 = (const uint4 *)(slot + 16);

    for (int q = lane; q < s.nw; q += G) {   // run starts before step 1: 0, n0, n
        unsigned o = q == 0 ? 1u : 0u;
        if (q == n0 >> 5) o |= 1u << (n0 & 31);
        if (q == n >> 5) o |= 1u << (n & 31);
        s.O[q] = o;
        s.N[q] = 0u;
    }
    if (NPOP == 2) {
        const unsigned *isA = (const unsigned *)(slot + slot_isa_at(n));
        unsigned carry = 0u;
        for (int base = 0; base < s.nw; base += G) {
            const int q = base + lane;
            const unsigned v = q < s.nw ? isA[q] : 0u;
            const unsigned pc = (unsigned)__popc(v);
            unsigned incl = pc;
#pragma unroll
            for (int d = 1; d < G; d <<= 1) {
                const unsigned u = tile.shfl_up(incl, d);
                if (lane >= d) incl += u;
            }
            if (q < s.nw) { s.isA[q] = v; s.PA[q] = carry + incl - pc; }
            carry += tile.shfl(incl, G - 1);
        }
    }
    tile.sync();

    // ---- step 0 (the core marker splits the sample into its allele classes)
    unsigned S[NV], prev[NV];             // S of this lane's step; S of the step before the block
    unsigned D[NV];                       // C(N, 2)
    unsigned long long cutD[NWK];         // a walk stops at the first cut_den S < cut_num D
    if (NPOP == 2) {
        const unsigned nA = (unsigned)w.a.nA, nB = (unsigned)w.a.nB;
        const unsigned a0 = count_a(s, n0), a1 = nA - a0;
        const unsigned b0 = (unsigned)n0 - a0, b1 = nB - b0;
        prev[0] = (unsigned)(c2i(a0) + c2i(a1));
        prev[1] = (unsigned)(c2i(b0) + c2i(b1));
        prev[NV - 1] = (unsigned)(c2i((unsigned)n0) + c2i((unsigned)(n - n0)));
        D[0] = (unsigned)c2i(nA);
        D[1] = (unsigned)c2i(nB);
        D[NV - 1] = (unsigned)c2i((unsigned)n);
    } else {
        prev[0] = D[0] = (unsigned)c2i((unsigned)n0);             // allele 0: positions [0, n0)
        prev[1] = D[1] = (unsigned)c2i((unsigned)(n - n0));       // allele 1: positions [n0, n)
    }
    unsigned long long dig[NV];           // this lane's part of the digests
    double acc[2] = {0.0, 0.0};           // this lane's partial trapezoid sums
    bool act[NWK];
    int stop[NWK];
    unsigned skey[NWK];                   // S where an unfinished walk left off
    bool any = false;
#pragma unroll
    for (int q = 0; q < NV; ++q) dig[q] = lane == 0 ? prev[q] : 0u;
#pragma unroll
    for (int q = 0; q < NWK; ++q) {
        const unsigned Dq = D[NPOP == 2 ? NV - 1 : q];
        cutD[q] = (unsigned long long)w.a.cut_num * Dq;
        stop[q] = 0;
        skey[q] = 0u;
        act[q] = Dq != 0u;
        any |= act[q];
    }
    int fin = WALK_OK;                    // how the still-active walks end
    int endstep = 0;
    int lo = 1;                           // first step of the window
    bool dense = true, merge = false;
    while (any) {
        unsigned K0, sup;
        const int hi = lo + (dense ? kDense - 1 : kWin - 1);
        const int pa = NPOP == 1 && !act[0] ? n0 : 0, pb = NPOP == 1 && !act[NWK - 1] ? n0 : n;
        const unsigned K = mark_window<NPOP>(tile, s, M4, n, n0, hi, dense, merge, pa, pb, K0, sup);
        if (!dense && K > (unsigned)tok_smem(NPOP == 2)) {    // redo as a window of fewer steps
            dense = true;
            merge = false;
            continue;
        }
        if (!dense) sparse_terms<NPOP>(tile, s, K, lo, n0, sup);
        for (int b0 = lo; b0 <= hi; b0 += 32) {
            // the step of this lane: its map distance g, or how the walk ends
            // there.  Step i belongs to lane (i - 1) mod 32; the block is the
            // lanes [la, lb)
            const int la = (b0 - 1) & 31, i0 = b0 - la, i = i0 + lane;
            const int lb = la + (hi - b0 + 1 < 32 ? hi - b0 + 1 : 32);
            const bool mine = lane >= la && lane < lb;
            double gq = 0.0;
            int gk = 0;                   // 0 a step, WALK_EDGE past the array end, WALK_GAP a gap abort
            const long long step = dir ? 1 : -1;
            const long long xl = k + step * i, xp = xl - step;
            if (xl < 0 || xl >= m) gk = WALK_EDGE;
            else {
                const long long p1 = __ldg(w.a.pos + xl), p0 = __ldg(w.a.pos + xp);
                const long long bp = dir ? p1 - p0 : p0 - p1;
                if (bp > w.a.max_gap) gk = WALK_GAP;
                else {
                    double gg;
                    if (w.a.physical) gg = (double)bp;
                    else {
                        const double g1 = __ldg(w.a.gmap + xl), g0 = __ldg(w.a.gmap + xp);
                        gg = dir ? g1 - g0 : g0 - g1;
                    }
                    if (bp > w.a.gap_scale) gg = gg * ((double)w.a.gap_scale / (double)bp);
                    gq = gg;
                }
            }
            // S of this lane's step
            if (dense) {
                RunCut<NPOP> rc;
                if (NPOP == 2) {
                    // 16 steps, each by two lanes
                    rc.lim = (unsigned)(i0 + la + (lane & 15) + 1) << 16;   // M <= i  <=>  token < lim
                    rc.d[0] = rc.d[NPOP == 2 ? 1 : 0] = rc.d[NPOP == 2 ? 2 : 0] = 0u;
                    rc.both_ends(tile, s, K, (unsigned)n, (unsigned)w.a.nA);
                    S[0] = (rc.d[NPOP == 2 ? 1 : 0] - (unsigned)w.a.nA) >> 1;
                    S[1] = (rc.d[NPOP == 2 ? 2 : 0] - (unsigned)w.a.nB) >> 1;
                    S[NV - 1] = (rc.d[0] - (unsigned)n) >> 1;
                } else if (NARROW) {
                    const uint2 c = narrow_counts(s.tk, s.gtk, K0, K, (unsigned)n0, (unsigned)n,
                                                  (unsigned)(i0 + la + (lane & 7) + 1) << 16);
                    S[0] = c.x;
                    S[1] = c.y;
                } else {
                    rc.lim = (unsigned)(i + 1) << 16;
                    S[0] = S[1] = 0u;
                    if (act[0]) {
                        rc.last = 0u;
                        rc.d[0] = 0u;
                        rc.range(s, 0u, K0);
                        rc.cut((unsigned)n0, 0u);
                        S[0] = (rc.d[0] - (unsigned)n0) >> 1;
                    }
                    if (act[NWK - 1]) {
                        rc.last = (unsigned)n0;
                        rc.d[0] = 0u;
                        rc.range(s, K0, K);
                        rc.cut((unsigned)n, 0u);
                        S[1] = (rc.d[0] - (unsigned)(n - n0)) >> 1;
                    }
                }
            } else {
#pragma unroll
                for (int q = 0; q < NV; ++q) {
                    unsigned dd = mine ? s.dec[q * kWin + (i - lo)] : 0u;
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        const unsigned v = tile.shfl_up(dd, d);
                        if (lane >= d) dd += v;
                    }
                    S[q] = prev[q] - dd;
                }
            }
            // where the block ends for the walks still running: a gap or the
            // array end (tested before a step's S), else the history's end
            const unsigned km = tile.ballot(mine && gk != 0), hm = tile.ballot(mine && i > hz);
            const int ke = km ? __ffs(km) - 1 : lb, he = hm ? __ffs(hm) - 1 : lb;
            const int end = ke <= he ? ke : he;
            const int kfin = tile.shfl(gk, ke & 31);
            any = false;
#pragma unroll
            for (int q = 0; q < NWK; ++q) {
                if (!act[q]) continue;
                const int sd = NPOP == 2 ? NV - 1 : q;
                const unsigned sm = tile.ballot(mine && (unsigned long long)w.a.cut_den * S[sd] < cutD[q]);
                const int sl = sm ? __ffs(sm) - 1 : lb;
                const bool stops = sl < end;
                const int full = stops ? sl : end;       // lanes below: whole steps
                const bool cnt = lane >= la && lane < full + (stops ? 1 : 0);
                const bool term = lane >= la && lane < full + (stops && w.a.crossing ? 1 : 0);
                if (end < lb) skey[q] = end > la ? tile.shfl(S[sd], (end - 1) & 31) : prev[sd];
#pragma unroll
                for (int v = NPOP == 2 ? 0 : q; v <= (NPOP == 2 ? NV - 1 : q); ++v) {
                    unsigned sp = tile.shfl_up(S[v], 1);
                    if (lane == la) sp = prev[v];
                    if (cnt) dig[v] += (unsigned long long)(unsigned)(i + 1) * S[v];
                    if (term && v < 2) acc[v < 2 ? v : 0] += (double)(sp + S[v]) * gq;
                    prev[v] = tile.shfl(S[v], lb - 1);
                }
                if (stops) {
                    stop[q] = i0 + sl;
                    act[q] = false;
                }
                any |= act[q];
            }
            if (!any) break;
            if (end < lb) {
                fin = ke <= he ? kfin : WALK_UNFINISHED;
                endstep = i0 + end;
                any = false;
                break;
            }
        }
        lo = hi + 1;
        dense = (lo & 31) != 1;           // whole blocks of 32 from here on
        merge = true;
    }
    // ---- the lanes' partial sums, then the results (lane 0)
#pragma unroll
    for (int q = 0; q < 2; ++q) acc[q] = lane_sum_f64<G>(acc[q]);
#pragma unroll
    for (int q = 0; q < NV; ++q) {
#pragma unroll
        for (int d = G / 2; d > 0; d >>= 1) dig[q] += __shfl_xor_sync(0xFFFFFFFFu, dig[q], d);
    }
    if (lane == 0) {
        const ItemSink &sk = w.sk;
#pragma unroll
        for (int q = 0; q < NWK; ++q) {
            const unsigned Dq = D[NPOP == 2 ? NV - 1 : q];
            // iHS items: (allele 1, down), (allele 1, up), (allele 0, down), (allele 0, up)
            const uint32_t item = NPOP == 2 ? (uint32_t)(k * 2 + dir)
                                            : (uint32_t)(k * 4 + (q == 1 ? 0 : 2) + dir);
            int status = Dq == 0u ? WALK_UNDEFINED : WALK_OK;
            if (act[q]) {
                if (fin == WALK_UNFINISHED) {
                    const unsigned long long slot2 = atomicAdd(&sk.q->n2, 1ull);
                    sk.list2[slot2] = item;
                    sk.key2[slot2] = bucket_of((float)((double)skey[q] / (double)Dq));
                    continue;
                }
                status = fin;
                stop[q] = endstep;
            }
            sk.item_status[item] = (int8_t)status;
            sk.stop[item] = stop[q];
            if (NPOP == 2) {
                sk.item_ihh[2 * (size_t)item] = D[0] ? acc[0] / (2.0 * (double)D[0]) : 0.0;
                sk.item_ihh[2 * (size_t)item + 1] = D[1] ? acc[1] / (2.0 * (double)D[1]) : 0.0;
                sk.digest[3 * (size_t)item] = dig[0];
                sk.digest[3 * (size_t)item + 1] = dig[1];
                sk.digest[3 * (size_t)item + 2] = dig[NV - 1];
            } else {
                sk.item_ihh[item] = Dq ? acc[q] / (2.0 * (double)Dq) : 0.0;
                sk.digest[item] = Dq ? dig[q] : 0ull;
            }
        }
    }
    tile.sync();
}

// iHS in samples of more than kWideBoundaries haplotypes: whether more than that many
// run boundaries part within the first 32 steps, told from 256 run lengths (eight a
// lane, spread over the slot).  Their walks last a dozen steps (unlinked alleles),
// and a window of 32 that runs over all of them, mostly in global memory, takes
// longer than windows of kNarrow steps with short lists: 5,000 x 100,000 unlinked
// 11.3 ms against 6.4, 10,000 x 75,000 18.4 against 7.8.  Up to twice the on-chip
// list the window of 32 is the faster one (8,000 haplotypes of 320 founders: 5.0
// ms against 5.6).
constexpr int kWideBoundaries = 2048;
__device__ __forceinline__ bool wide_slot(const unsigned char *slot, int n, int lane)
{
    const uint4 v = __ldg((const uint4 *)(slot + 16) + (unsigned)lane * ((unsigned)n >> 8));
    const unsigned P1 = 32u * 0x00010001u, PP = P1 + 0x00010001u;     // 16x2 clamps, as in mark_window
    const unsigned f = (__vmaxu2(__vminu2(v.x, PP), P1) - P1) + (__vmaxu2(__vminu2(v.y, PP), P1) - P1) +
                       (__vmaxu2(__vminu2(v.z, PP), P1) - P1) + (__vmaxu2(__vminu2(v.w, PP), P1) - P1);
    const unsigned over = (unsigned)__reduce_add_sync(0xFFFFFFFFu, (int)((f & 0xFFFFu) + (f >> 16)));
    return (256u - over) * (unsigned)n > 256u * (unsigned)kWideBoundaries;
}

// Walks the slots that a warp has put by: a list through a word per core and
// direction (w.sk.sorted2, which the second pass fills later), from put_by - 1 on.
__device__ __noinline__ void walk_put_by(const SweepArgs &w, unsigned *tk, unsigned *gtk, unsigned put_by)
{
    namespace cg = cooperative_groups;
    const cg::thread_block_tile<32> tile = cg::tiled_partition<32>(cg::this_thread_block());
    const int lane = tile.thread_rank();
    const SplitSmem s = split_smem((unsigned char *)tk, (unsigned char *)gtk, w.n, 0);
    while (put_by != 0u) {
        const unsigned id = put_by - 1u;
        const int dir = (int)(id & 1u);
        const long long q = (long long)(id >> 1), c = q / w.B;
        const long long c1 = (c + 1) * w.B < w.a.k1 - w.a.k0 ? (c + 1) * w.B : w.a.k1 - w.a.k0;
        const long long r = (dir == 0 ? q - c * w.B : c1 - 1 - q) - (long long)w.stage * w.R;
        walk_slot<1, true>(w, tile, s, w.slots + (size_t)((dir * w.nch + c) * w.R + r) * w.slot_bytes, w.a.k0 + q, dir);
        unsigned nxt = 0u;
        if (lane == 0) nxt = w.sk.sorted2[id];
        put_by = tile.shfl(nxt, 0);
    }
}

// Persistent: each warp takes slots of this stage (both directions) from a
// counter.  WIDE: puts wide slots by and walks them at the end, out of line; in the
// common walk's place their code cost it registers (1M iHS 25.3 ms; so 24.5, and
// 24.2 without).
template <int NPOP, int G, bool WIDE>
__device__ __forceinline__ void split_walks(const SweepArgs &w, unsigned char *smem)
{
    static_assert(G == 32, "lane l owns step l of a block of 32");
    namespace cg = cooperative_groups;
    const cg::thread_block_tile<G> tile = cg::tiled_partition<G>(cg::this_thread_block());
    const int lane = tile.thread_rank(), tix = threadIdx.x / G;
    const int n = w.n;
    const SplitSmem s = split_smem(smem + (size_t)tix * w.split_bytes,
                                   w.wscratch + ((size_t)blockIdx.x * kSplitWarps + tix) * w.wscratch_bytes,
                                   n, NPOP == 2);
    const long long per_dir = (long long)w.nch * w.R;
    unsigned put_by = 0u;                     // 1 + the last slot put by
    unsigned long long nxt = 0;               // the slot after this one, fetched ahead
    if (lane == 0) nxt = atomicAdd(w.walk_head, 1ull);
    for (;;) {
        const unsigned long long gs = tile.shfl(nxt, 0);
        if (gs >= (unsigned long long)(2 * per_dir)) break;
        if (lane == 0) nxt = atomicAdd(w.walk_head, 1ull);
        // slot counts are below 2^31 (2 x chunks x stage cores): 32-bit decode
        const unsigned gsl = (unsigned)gs;
        const long long gslot = (long long)gs;
        const unsigned cr = gsl / (unsigned)w.R;
        const int r = (int)(gsl - cr * (unsigned)w.R);
        const int dir = cr >= (unsigned)w.nch ? 1 : 0;
        const int c = (int)(cr - (unsigned)dir * (unsigned)w.nch);
        const long long c0 = w.a.k0 + (long long)c * w.B;
        if (c0 >= w.a.k1) continue;
        const long long c1 = c0 + w.B < w.a.k1 ? c0 + w.B : w.a.k1;
        long long k;
        if (dir == 0) {
            const long long klo = c0 + (long long)w.stage * w.R;
            const long long khi = klo + w.R < c1 ? klo + w.R : c1;
            k = klo + r;
            if (k >= khi) continue;
        } else {
            const long long khi = c1 - (long long)w.stage * w.R;
            const long long klo = khi - w.R > c0 ? khi - w.R : c0;
            k = khi - 1 - r;
            if (k < klo) continue;
        }
        if (w.sk.core_status[k] == (int8_t)SELSCAN_LOCUS_MAF_FILTERED) continue;

        const unsigned char *slot = w.slots + (size_t)gslot * w.slot_bytes;
        if (WIDE && wide_slot(slot, n, lane)) {
            const unsigned id = (unsigned)(2 * (k - w.a.k0) + dir);
            if (lane == 0) w.sk.sorted2[id] = put_by;
            put_by = id + 1u;
        } else {
            walk_slot<NPOP>(w, tile, s, slot, k, dir);
        }
    }
    if (WIDE && put_by != 0u) walk_put_by(w, s.tk, s.gtk, put_by);
}

#ifndef SPLIT_MIN_CTAS
#define SPLIT_MIN_CTAS 4
#endif
template <int NPOP, int G>
__global__ void __launch_bounds__(kSplitWarps * 32, SPLIT_MIN_CTAS) split_walk_kernel(SweepArgs w)
{
    extern __shared__ __align__(16) unsigned char smem[];
    split_walks<NPOP, G, false>(w, smem);
}

template <int G>
static void (*walk_kernel_for(int xpehh))(SweepArgs)
{
    return xpehh ? split_walk_kernel<2, G> : split_walk_kernel<1, G>;
}

__global__ void __launch_bounds__(kSplitWarps * 32, SPLIT_MIN_CTAS)
    split_walk_wide_kernel(const __grid_constant__ SweepArgs w)
{
    extern __shared__ __align__(16) unsigned char smem[];
    split_walks<1, 32, true>(w, smem);
}

// the walk kernel of a sample
static void (*walk_kernel_of(int n, int xpehh))(SweepArgs)
{
    return !xpehh && n > kWideBoundaries ? split_walk_wide_kernel : walk_kernel_for<32>(xpehh);
}

// ---- the starting state of a chunk ----------------------------------------------
// The order and run lengths that the sweep would have after stepping through
// the history [s0, c0) (toward lower indices; [c1, e0] the other way) from the
// identity order: the haplotypes sorted by their sequence read from the nearest
// history marker outward, ties by index, M = the common length of neighbours.
// A multikey quicksort over the 32-marker words of w.tw, all groups of all
// levels at once: per round every unresolved group splits three ways, stably,
// about its middle element's word (the equal part goes on to the next word),
// by one prefix sum over the CTA; once few are left, only they take part.
// About 40 rounds (19 of all elements, 20 late ones at 1M) replace 1,536 marker passes.
// Shared memory per haplotype: element (bit index | group start << 16) and
// group (at its start: end | word level << 16) twice, the prefix sums, and the
// level at which each boundary arose.
__host__ __device__ size_t start_smem_bytes(int n, int T) { return (size_t)n * 22 + 8 + (size_t)(T / 32) * 4; }

namespace {

// QUIT: looked at once a round, w.quit ends it without a state (then false);
// `quitting` is a word of shared memory of its own, zero.
template <int T, bool QUIT = false>
__device__ bool start_state(const SweepArgs &w, unsigned char *smem, int dir, long long c0, long long c1,
                            unsigned *st, int np, volatile int *quitting = nullptr)
{
    const int n = w.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned *el = (unsigned *)smem;             // [2][n]
    unsigned *inf = el + 2 * n;                  // [2][n]
    unsigned *pre = inf + 2 * n;                 // [n + 1]
    unsigned *wsum = pre + n + 1;                // [T / 32]
    unsigned short *bw = (unsigned short *)(wsum + T / 32);   // [n]
    const long long m = w.a.m;
    const long long near = dir == 0 ? c0 - 1 : c1;
    const long long s0 = c0 - w.L > 0 ? c0 - w.L : 0;
    const long long e0 = c1 - 1 + w.L < m - 1 ? c1 - 1 + w.L : m - 1;
    const long long far = dir == 0 ? s0 : e0;
    const int H = (int)(dir == 0 ? c0 - s0 : e0 - c1 + 1);    // history markers
    const int bn = (int)((near >> 5) - w.tb0), bf = (int)((far >> 5) - w.tb0);   // blocks in tw
    const int nlev = H == 0 ? 0 : (dir == 0 ? bn - bf : bf - bn) + 1;
    const unsigned kn = (unsigned)near & 31u, kf = (unsigned)far & 31u;
    const unsigned mnear = dir == 0 ? 0xFFFFFFFFu >> (31u - kn) : 0xFFFFFFFFu << kn;
    const unsigned mfar = dir == 0 ? 0xFFFFFFFFu << kf : 0xFFFFFFFFu >> (31u - kf);
    // word l of haplotype bit index bi, the nearest marker in the top bit
    auto key = [&](unsigned bi, int l) {
        unsigned v = __ldg(w.tw + (size_t)(dir == 0 ? bn - l : bn + l) * (size_t)w.tld + bi);
        if (l == 0) v &= mnear;
        if (l == nlev - 1) v &= mfar;
        return dir == 0 ? v : __brev(v);
    };
    // exclusive prefix of v over the CTA's threads, and the total (two barriers)
    unsigned total = 0u;
    auto block_prefix = [&](unsigned v) {
        unsigned incl = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned u = __shfl_up_sync(FULLMASK, incl, d);
            if (lane >= d) incl += u;
        }
        __syncthreads();                          // the last totals have been read
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        unsigned off = incl - v;
        total = 0u;
#pragma unroll
        for (int q = 0; q < T / 32; ++q) {
            const unsigned u = wsum[q];
            off += q < warp ? u : 0u;
            total += u;
        }
        return off;
    };
    const int E = ((n + T - 1) / T) | 1;         // odd: a segment's strided reads hit distinct banks
    const int base = tid * E;
    constexpr int EC = 4;                        // late rounds: active elements per thread,
    constexpr int LW = 4;                        // and words compared at once
    const int few = n <= EC * T ? n : (EC * T < n * 5 / 8 ? EC * T : n * 5 / 8);
    for (int t = tid; t < n; t += T) el[t] = bit_index(w, t);
    if (tid == 0) inf[0] = (unsigned)n;
    __syncthreads();
    int cur = 0;
    int na = nlev > 0 && n > 1 ? n : 0;          // elements in unresolved groups
    constexpr unsigned kQuit = 1u << 30;         // far above any count of elements
    while (na > few) {
        const int walked = QUIT && tid == 0 ? *(const volatile int *)w.quit : 0;   // used at the round's end
        const unsigned *elc = el + cur * n, *ifc = inf + cur * n;
        // pass 1: this segment's elements below (low half) / equal to (high
        // half) their group's pivot, counted exclusively into pre
        unsigned cnt = 0u;
        for (int e0_ = 0; e0_ < E; e0_ += 4) {
            unsigned ka[4], kp[4];
            bool un[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int p = base + e0_ + u;
                un[u] = false;
                ka[u] = kp[u] = 0u;
                if (e0_ + u < E && p < n) {
                    const unsigned v = elc[p], g = v >> 16, f = ifc[g];
                    const unsigned end = f & 0xFFFFu;
                    const int l = (int)(f >> 16);
                    un[u] = end - g > 1u && l < nlev;
                    if (un[u]) {
                        ka[u] = key(v & 0xFFFFu, l);
                        kp[u] = key(elc[g + ((end - g) >> 1)] & 0xFFFFu, l);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int p = base + e0_ + u;
                if (e0_ + u < E && p < n) {
                    pre[p] = cnt;
                    if (un[u]) cnt += ka[u] < kp[u] ? 1u : (ka[u] == kp[u] ? 0x10000u : 0u);
                }
            }
        }
        const unsigned off = block_prefix(cnt);
        for (int e = 0; e < E; ++e)
            if (base + e < n) pre[base + e] += off;
        if (tid == 0) pre[n] = total;
        __syncthreads();
        // pass 2: place the elements; the first of each part describes its group
        unsigned *eln = el + (cur ^ 1) * n, *ifn = inf + (cur ^ 1) * n;
        unsigned left = 0u;
#pragma unroll 4
        for (int p = tid; p < n; p += T) {
            const unsigned v = elc[p], g = v >> 16, f = ifc[g];
            const unsigned end = f & 0xFFFFu, l = f >> 16;
            unsigned np_ = (unsigned)p, g2 = g, end2 = end, l2 = l;
            if (end - g > 1u && (int)l < nlev) {
                const unsigned pg = pre[g], me = pre[p], d = pre[p + 1] - me;
                const unsigned tot = pre[end] - pg, mine = me - pg;
                const unsigned L = tot & 0xFFFFu, Q = tot >> 16, ml = mine & 0xFFFFu, mq = mine >> 16;
                if (d == 1u) { np_ = g + ml; end2 = g + L; }
                else if (d != 0u) { g2 = g + L; np_ = g2 + mq; end2 = g2 + Q; l2 = l + 1u; }
                else { g2 = g + L + Q; np_ = g2 + ((unsigned)p - g - ml - mq); }
                left += end2 - g2 > 1u && (int)l2 < nlev ? 1u : 0u;
            }
            eln[np_] = (v & 0xFFFFu) | (g2 << 16);
            if (np_ == g2) {
                ifn[g2] = end2 | (l2 << 16);
                if (g2 != g) bw[g2] = (unsigned short)l;
            }
        }
        if (QUIT && walked >= 6) left += kQuit;
        block_prefix(left);
        if (QUIT && total >= kQuit) return false;
        na = (int)total;
        cur ^= 1;
    }
    if (na > 0) {
        // late rounds: the unresolved elements alone, listed in position order
        // (a group stays contiguous in the list), at most EC per thread; a
        // round reads them into registers and writes them back in place
        unsigned *fin = el + cur * n;             // by position: bit index | group start << 16
        const unsigned *ifc = inf + cur * n;
        unsigned *ael = el + (cur ^ 1) * n;       // by list index: bit index | list index of the group << 16
        unsigned *ainf = inf + (cur ^ 1) * n;     // at a group's first index: end | level << 16
        unsigned short *ap = na < n ? (unsigned short *)(pre + na + 1)     // positions
                                    : (unsigned short *)(inf + n);
        if (na < n) {
            unsigned cnt = 0u;
            for (int e = 0; e < E; ++e) {
                const int p = base + e;
                if (p < n) {
                    const unsigned g = fin[p] >> 16, f = ifc[g];
                    cnt += (f & 0xFFFFu) - g > 1u && (int)(f >> 16) < nlev ? 1u : 0u;
                }
            }
            unsigned at = block_prefix(cnt);
            for (int e = 0; e < E; ++e) {
                const int p = base + e;
                if (p < n) {
                    const unsigned v = fin[p], g = v >> 16, f = ifc[g];
                    if ((f & 0xFFFFu) - g > 1u && (int)(f >> 16) < nlev) {
                        const unsigned ag = at - ((unsigned)p - g);
                        ael[at] = (v & 0xFFFFu) | (ag << 16);
                        ap[at] = (unsigned short)p;
                        if ((unsigned)p == g) ainf[ag] = (at + (f & 0xFFFFu) - g) | (f & 0xFFFF0000u);
                        ++at;
                    }
                }
            }
        } else {
            ainf = inf;                           // one group: every haplotype at word 0
            for (int t = tid; t < n; t += T) {
                ael[t] = fin[t];
                ap[t] = (unsigned short)t;
            }
        }
        bool more = true;
        __syncthreads();
        while (more) {
            const int walked = QUIT && tid == 0 ? *(const volatile int *)w.quit : 0;
            unsigned v[EC], f[EC], d[EC];
            unsigned cnt = 0u;
#pragma unroll
            for (int u = 0; u < EC; ++u) {
                const int i = EC * tid + u;
                f[u] = 0u;                        // resolved (or no element)
                d[u] = 0u;
                if (i < na) {
                    v[u] = ael[i];
                    const unsigned g = v[u] >> 16;
                    f[u] = ainf[g];
                    const unsigned end = f[u] & 0xFFFFu;
                    const int l = (int)(f[u] >> 16);
                    if (end - g > 1u && l < nlev) {
                        const unsigned bi = v[u] & 0xFFFFu, bp = ael[g + ((end - g) >> 1)] & 0xFFFFu;
                        unsigned ka[LW], kp[LW];
#pragma unroll
                        for (int j = 0; j < LW; ++j) ka[j] = l + j < nlev ? key(bi, l + j) : 0u;
#pragma unroll
                        for (int j = 0; j < LW; ++j) kp[j] = l + j < nlev ? key(bp, l + j) : 0u;
                        d[u] = 0x10000u;
#pragma unroll
                        for (int j = LW - 1; j >= 0; --j)
                            d[u] = ka[j] < kp[j] ? 1u : (ka[j] == kp[j] ? d[u] : 0u);
                    } else {
                        f[u] = 0u;
                    }
                }
                cnt += d[u];
            }
            unsigned me = block_prefix(cnt);
#pragma unroll
            for (int u = 0; u < EC; ++u) {
                if (EC * tid + u < na) pre[EC * tid + u] = me;
                me += d[u];
            }
            // group ends look up pre one past the list's last index too; the
            // position list follows at pre + na + 1
            if (tid == 0) pre[na] = total;
            __syncthreads();
            bool left = false;
#pragma unroll
            for (int u = 0; u < EC; ++u) {
                if (f[u] == 0u) continue;
                const unsigned i = (unsigned)(EC * tid + u), g = v[u] >> 16, end = f[u] & 0xFFFFu, l = f[u] >> 16;
                const unsigned pg = pre[g], tot = pre[end] - pg, mine = pre[i] - pg;
                const unsigned L = tot & 0xFFFFu, Q = tot >> 16, ml = mine & 0xFFFFu, mq = mine >> 16;
                unsigned ni, g2 = g, end2, l2 = l;
                if (d[u] == 1u) { ni = g + ml; end2 = g + L; }
                else if (d[u] != 0u) { g2 = g + L; ni = g2 + mq; end2 = g2 + Q; l2 = l + LW; }
                else { g2 = g + L + Q; ni = g2 + (i - g - ml - mq); end2 = end; }
                left = left || (end2 - g2 > 1u && (int)l2 < nlev);
                ael[ni] = (v[u] & 0xFFFFu) | (g2 << 16);
                fin[ap[ni]] = (v[u] & 0xFFFFu) | ((unsigned)ap[g2] << 16);
                if (ni == g2) {
                    ainf[g2] = end2 | (l2 << 16);
                    if (g2 != g) bw[ap[g2]] = (unsigned short)l;
                }
            }
            // every thread has read `quitting` of the last round: block_prefix's
            // barriers lie between
            if (QUIT && walked >= 6) *quitting = 1;
            more = __syncthreads_or(left) != 0;
            if (QUIT && *quitting) return false;
        }
    }
    // run lengths: neighbours of one group share the whole history, others part
    // in the word at which their boundary arose
    const unsigned *elc = el + cur * n;
    const unsigned pad_bi = 64u * (unsigned)w.a.W;
    const int off0 = dir == 0 ? 31 - (int)kn : (int)kn;       // bits of word 0 nearer than `near`
    for (int p = tid; p < np; p += T) {
        unsigned M = 0u, bi = pad_bi;
        if (p < n) {
            const unsigned v = elc[p];
            bi = v & 0xFFFFu;
            if (p > 0) {
                if ((int)(v >> 16) == p) {
                    int l = bw[p];                // or one of the next LW - 1
                    unsigned x = key(bi, l) ^ key(elc[p - 1] & 0xFFFFu, l);
                    while (x == 0u && l + 1 < nlev) {
                        ++l;
                        x = key(bi, l) ^ key(elc[p - 1] & 0xFFFFu, l);
                    }
                    M = (unsigned)(32 * l - off0 + __clz((int)x));
                } else {
                    M = (unsigned)H;
                }
            }
        }
        st[p] = bi | (M << 16);
    }
    return true;
}

}  // namespace

template <int T>
__global__ void __launch_bounds__(T) start_kernel(SweepArgs w)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int dir = blockIdx.x / w.nch, c = blockIdx.x % w.nch;
    const long long c0 = w.a.k0 + (long long)c * w.B;
    if (c0 >= w.a.k1) return;
    const long long c1 = c0 + w.B < w.a.k1 ? c0 + w.B : w.a.k1;
    const int np = (int)sweep_elements(w.n, w.threads);
    start_state<T>(w, smem, dir, c0, c1, (unsigned *)w.st + (size_t)blockIdx.x * np, np);
}

// ---- a whole short scan in one launch ----------------------------------------------
// Short chromosomes (the in-order schedule): one CTA per chunk and direction.
// All of its TC threads make the chunk's starting state (the whole arm as
// history, so no walk is ever handed on); the first TS then sort the cores one
// after the other into slots of their own, while the other warps walk each core
// as soon as its slot is written.  When the sort is done its warps walk too, and
// warps that run out of work take slots of any chunk whose sort is done.
// Waits are inside the CTA only (a walking warp for its own sorting warps, with
// a limit); a chunk that is not ready is left to its owner.
// w.heads[chunk]: 0 until the chunk's sort is done, then 1 + the next slot.
// Bound by latency (one chunk's serial chain of rounds, marker passes and walks),
// so the chromosome is cut into as many chunks as the GPU holds CTAs at once.
constexpr int kChunkClosed = 1 << 24;        // added to a chunk's own counter when its sort is done
constexpr int kChunkPolls = 1 << 24;

template <int TS>
__device__ __forceinline__ void sort_barrier()
{
    if (TS == 32) __syncwarp();
    else asm volatile("bar.sync 1, %0;" ::"n"(TS) : "memory");
}

// Waits until the CTA's sorting warps have written slot r, `limit` looks at the
// most.  Each lane looks, the warp decides together: lanes that left on their own
// count could part when the slot is written around the last look.  (One lane
// looking for its warp takes chr22 iHS from 0.33 to 0.62 ms.)
__device__ __forceinline__ bool wait_slot(const volatile int *ready, int r, int limit)
{
    int looks = 0;
    while (*ready <= r && ++looks < limit) __nanosleep(64);
    const bool ok = !__any_sync(FULLMASK, looks >= limit);
    __threadfence_block();                    // the flag before the slot
    __syncwarp();
    return ok;
}

// One chunk and direction of one scan.
struct ChunkTask { const SweepArgs *w; long long c0, c1; int dir, blk, cnt; };

// The chunks of one scan.
struct ScanChunks {
    SweepArgs w;
    __device__ int count() const { return 2 * w.nch; }
    __device__ int most() const { return w.R; }          // cores of a whole chunk
    __device__ unsigned *heads() const { return w.heads; }
    __device__ ChunkTask task(int id) const
    {
        ChunkTask t;
        t.w = &w;
        t.dir = id / w.nch;
        t.blk = id;
        t.c0 = w.a.k0 + (long long)(id % w.nch) * w.B;
        t.c1 = t.c0 + w.B < w.a.k1 ? t.c0 + w.B : w.a.k1;
        t.cnt = t.c0 < t.c1 ? (int)(t.c1 - t.c0) : 0;
        return t;
    }
};

// The chunks of a tick's units (ChunkTick): unit u's chunks are the tasks
// [first[u], first[u + 1]), both directions.
struct TickChunks {
    ChunkTick t;
    __device__ int count() const { return t.first[t.nunits]; }
    __device__ int most() const { return t.B; }
    __device__ unsigned *heads() const { return t.heads; }
    __device__ ChunkTask task(int id) const
    {
        int lo = 0, hi = t.nunits - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (t.first[mid] <= id) lo = mid;
            else hi = mid - 1;
        }
        const int local = id - t.first[lo], nch = (t.first[lo + 1] - t.first[lo]) >> 1;
        ChunkTask r;
        r.w = t.w + t.scan[lo];
        r.dir = local >= nch;
        r.blk = t.blk0[lo] + local;
        r.c0 = t.c0[lo] + (long long)(local - r.dir * nch) * t.B;
        r.c1 = r.c0 + t.B < t.c1[lo] ? r.c0 + t.B : t.c1[lo];
        r.cnt = (int)(r.c1 - r.c0);
        return r;
    }
};

// NPOP 1: iHS scans, 2: XPEHH scans, 0: both kinds.
template <int TS, int TC, int EMAX, int MINB, int NPOP, class Chunks>
__global__ void __launch_bounds__(TC, MINB) chunk_scan_kernel(const __grid_constant__ Chunks ch)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int own_next;                  // next slot of this chunk while it is being sorted
    __shared__ volatile int own_ready;        // slots written
    namespace cg = cooperative_groups;
    const cg::thread_block_tile<32> tile = cg::tiled_partition<32>(cg::this_thread_block());
    const int lane = tile.thread_rank(), warp = threadIdx.x >> 5;
    const int me = (int)blockIdx.x;
    unsigned *heads = ch.heads();
    auto walk_one = [&](const ChunkTask &t, int r) {
        const SweepArgs &w = *t.w;
        const long long k = t.dir == 0 ? t.c0 + r : t.c1 - 1 - r;
        if (w.sk.core_status[k] == (int8_t)SELSCAN_LOCUS_MAF_FILTERED) return;
        const unsigned char *slot = w.slots + ((size_t)t.blk * w.R + r) * w.slot_bytes;
        const bool xp = NPOP == 2 || (NPOP == 0 && w.a.nB > 0);
        const SplitSmem s = split_smem(smem + w.split_off + (size_t)warp * w.split_bytes,
                                       w.wscratch + ((size_t)me * (TC / 32) + warp) * w.wscratch_bytes, w.n, xp);
        if (NPOP != 1 && xp) walk_slot<2>(w, tile, s, slot, k, t.dir);
        if (NPOP != 2 && !xp) walk_slot<1>(w, tile, s, slot, k, t.dir);
    };
    const ChunkTask mine = ch.task(me);
    bool own = false;                         // this chunk's remaining slots are this warp's to drain
    if (mine.cnt > 0) {                       // uniform over the CTA
        const SweepArgs &w = *mine.w;
        const int np = (int)sweep_elements(w.n, TS);
        start_state<TC>(w, smem, mine.dir, mine.c0, mine.c1, (unsigned *)w.st + (size_t)mine.blk * np, np);
        if (threadIdx.x == 0) {
            own_next = 0;
            own_ready = 0;
        }
        __syncthreads();
        if (threadIdx.x < TS) {
            sort_chunk<TS, EMAX, false, NPOP == 0 ? -1 : NPOP - 1>(w, smem, mine.dir, mine.c0, mine.c1, mine.blk,
                                        [] { sort_barrier<TS>(); },
                                        [&](int r) {
                                            if (threadIdx.x == 0) {
                                                __threadfence_block();
                                                own_ready = r;
                                            }
                                        });
            sort_barrier<TS>();
            if (threadIdx.x == 0) {
                __threadfence();              // the slots before the flags
                own_ready = mine.cnt;
                const int next = atomicAdd(&own_next, kChunkClosed);
                atomicExch(heads + me, 1u + (unsigned)(next < mine.cnt ? next : mine.cnt));
            }
            sort_barrier<TS>();
            own = true;
        } else {
            for (;;) {
                int r = 0;
                if (lane == 0) r = atomicAdd(&own_next, 1);
                r = __shfl_sync(FULLMASK, r, 0);
                if (r >= mine.cnt) break;
                if (!wait_slot(&own_ready, r, kChunkPolls)) {
                    if (lane == 0) atomicExch(w.err, SELSCAN_ERR_TIMEOUT);
                    break;
                }
                walk_one(mine, r);
            }
        }
    }
    // own chunk first, then whatever is ready (128 chunks looked at per step,
    // heads padded to a multiple of 128), until a full look finds nothing
    int first = me & ~127;
    const int span = (ch.count() + 127) & ~127;
    const unsigned most = (unsigned)ch.most();
    for (;;) {
        int id = own ? me : -1;
        own = false;
        for (int q = 0; q < span && id < 0; q += 128) {
            const int at = first + q < span ? first + q : first + q - span;
            const volatile unsigned *h = heads + at + 4 * lane;
            unsigned avail = 0u;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned v = h[u];
                if (v != 0u && v <= most) avail |= 1u << u;
            }
            const unsigned any = __ballot_sync(FULLMASK, avail != 0u);
            if (any) {
                const int l = __ffs(any) - 1;
                id = at + 4 * l + __ffs((int)__shfl_sync(FULLMASK, avail, l)) - 1;
                first = at;
                __threadfence();                  // the flag before the slots
            }
        }
        if (id < 0) break;
        const ChunkTask t = ch.task(id);
        unsigned nxt = 0u;
        if (lane == 0) nxt = atomicAdd(heads + id, 1u);
        for (;;) {
            const int r = (int)__shfl_sync(FULLMASK, nxt, 0) - 1;
            if (r >= t.cnt) break;
            if (lane == 0) nxt = atomicAdd(heads + id, 1u);
            walk_one(t, r);
        }
        // a chunk shorter than the others: mark it used up for the scan above
        if (lane == 0) atomicMax(heads + id, most + 1u);
    }
}

typedef void (*ChunkKernel)(ScanChunks);

// Threads that sort a chunk, threads of its CTA, CTAs per SM.  Chunks of many
// cores: a narrow sort with walking warps beside it (204 haplotypes x 22,147
// markers 0.34 ms: one warp of six, four CTAs per SM; all four of four warps
// sorting, then walking: 0.39).  Chunks of few cores: every warp sorts, then
// walks (100 x 2,000: 0.127 ms, against 0.185 with one sorting warp of six).
struct ChunkShape { int ts, tc, ctas; ChunkKernel ihs, xpehh; };
static ChunkShape chunk_shape(int n, long long m)
{
    if (n <= 1024 && m < 16 * 2 * device_sms())
        return {128, 128, 5, chunk_scan_kernel<128, 128, 8, 5, 1, ScanChunks>, chunk_scan_kernel<128, 128, 8, 5, 2, ScanChunks>};
    if (n <= 256)
        return {32, 192, 4, chunk_scan_kernel<32, 192, 8, 4, 1, ScanChunks>, chunk_scan_kernel<32, 192, 8, 4, 2, ScanChunks>};
    if (n <= 512)
        return {64, 192, 4, chunk_scan_kernel<64, 192, 8, 4, 1, ScanChunks>, chunk_scan_kernel<64, 192, 8, 4, 2, ScanChunks>};
    if (n <= 2048)
        return {128, 256, 2, chunk_scan_kernel<128, 256, 16, 2, 1, ScanChunks>, chunk_scan_kernel<128, 256, 16, 2, 2, ScanChunks>};
    return {256, 320, 2, chunk_scan_kernel<256, 320, 24, 2, 1, ScanChunks>, chunk_scan_kernel<256, 320, 24, 2, 2, ScanChunks>};
}
int chunk_sort_threads(int n, long long m) { return chunk_shape(n, m).ts; }
int chunk_warps(int n, long long m) { return chunk_shape(n, m).tc / 32; }

// the walking warps' shared memory follows the sort's (they run side by side);
// the starting state's is gone by then
static int chunk_split_off(int n, int W, int ts, int R) { return (int)((sweep_smem_bytes(n, W, ts, R) + 15) & ~(size_t)15); }
size_t chunk_smem_bytes(int n, long long m, int W, int R, int xpehh)
{
    const ChunkShape c = chunk_shape(n, m);
    const size_t a = start_smem_bytes(n, c.tc);
    const size_t b = (size_t)chunk_split_off(n, W, c.ts, R) + split_smem_per_warp(n, xpehh) * (size_t)(c.tc / 32);
    return a > b ? a : b;
}

int chunk_ctas_per_sm(int n, long long m, size_t smem, int xpehh)
{
    const ChunkShape c = chunk_shape(n, m);
    int per_sm = 0;
    const ChunkKernel k = xpehh ? c.xpehh : c.ihs;
    if (allow_smem(k, kFixedSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, c.tc, smem) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    return per_sm < c.ctas ? per_sm : c.ctas;
}

cudaError_t launch_chunk_scan(const SweepArgs &w0, cudaStream_t s)
{
    ScanChunks sc;
    sc.w = w0;
    SweepArgs &w = sc.w;
    const int xp = w.a.nB > 0;
    const ChunkShape c = chunk_shape(w.n, w.a.m);
    const size_t smem = chunk_smem_bytes(w.n, w.a.m, w.a.W, w.R, xp);
    w.split_off = chunk_split_off(w.n, w.a.W, c.ts, w.R);
    const ChunkKernel k = xp ? c.xpehh : c.ihs;
    const cudaError_t e = allow_smem(k, kFixedSmem);
    if (e != cudaSuccess) return e;
    k<<<2 * w.nch, c.tc, smem, s>>>(sc);
    return cudaGetLastError();
}

// ---- a tick's core ranges (batched scans) -----------------------------------------
// Shapes by the largest sample of the tick: a scan's smaller sample sorts on the
// same threads.
struct TickShape { int ts, tc, ctas; void (*kernel)(TickChunks); };
static TickShape tick_shape(int max_n)
{
    if (max_n <= 512) return {64, 192, 4, chunk_scan_kernel<64, 192, 8, 4, 0, TickChunks>};
    if (max_n <= 1024) return {128, 256, 2, chunk_scan_kernel<128, 256, 8, 2, 0, TickChunks>};
    if (max_n <= 2048) return {128, 320, 2, chunk_scan_kernel<128, 320, 16, 2, 0, TickChunks>};
    return {256, 320, 2, chunk_scan_kernel<256, 320, 24, 2, 0, TickChunks>};
}
int tick_sort_threads(int max_n) { return tick_shape(max_n).ts; }
int tick_warps(int max_n) { return tick_shape(max_n).tc / 32; }
int tick_ctas(int max_n) { return tick_shape(max_n).ctas; }

size_t tick_smem_bytes(int max_n, int n, int W, int R, int xpehh, int *split_off)
{
    const TickShape c = tick_shape(max_n);
    *split_off = chunk_split_off(n, W, c.ts, R);
    const size_t a = start_smem_bytes(n, c.tc);
    const size_t b = (size_t)*split_off + split_smem_per_warp(n, xpehh) * (size_t)(c.tc / 32);
    return a > b ? a : b;
}

cudaError_t launch_chunk_tick(const ChunkTick &t, int max_n, size_t smem, cudaStream_t s)
{
    static_assert(sizeof(TickChunks) <= 32000, "tick parameter block too large");
    const TickShape c = tick_shape(max_n);
    const cudaError_t e = allow_smem(c.kernel, kFixedSmem);
    if (e != cudaSuccess) return e;
    // static: the block is large, and the launch consumes it before this returns
    static thread_local TickChunks tc;
    tc.t = t;
    c.kernel<<<t.first[t.nunits], c.tc, smem, s>>>(tc);
    return cudaGetLastError();
}

int split_walk_ctas(int n, int xpehh)
{
    // resident CTAs of the persistent walker
    int per_sm = 0;
    const size_t smem = split_smem_per_warp(n, xpehh) * kSplitWarps;
    allow_smem(walk_kernel_of(n, xpehh));
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, walk_kernel_of(n, xpehh), kSplitWarps * 32, smem);
    if (e != cudaSuccess || per_sm < 1) per_sm = 1;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return per_sm * (sms > 0 ? sms : 1);
}

// The sorting kernel of a sample and CTA width.  The 256-thread sorts of the large
// scans are compiled for each kind of scan (iHS beside XPEHH's population flags in
// one kernel: 1M iHS sort 15.2 ms against 14.5).
template <int XP>
static void (*sort256(int E))(SweepArgs)
{
    return E == 4 ? sweep_kernel<256, 4, true, XP> : E == 8 ? sweep_kernel<256, 8, true, XP>
         : E == 12 ? sweep_kernel<256, 12, true, XP> : E == 16 ? sweep_kernel<256, 16, true, XP>
         : E == 20 ? sweep_kernel<256, 20, true, XP> : E == 24 ? sweep_kernel<256, 24, true, XP>
         : sweep_kernel<256, 32>;
}
static void (*sort_kernel(int n, int threads, bool xpehh))(SweepArgs)
{
    const int E = sweep_e(n, threads);
    if (threads == 256) return xpehh ? sort256<1>(E) : sort256<0>(E);
    if (threads == 512)
        return E <= 4 ? sweep_kernel<512, 4> : E <= 8 ? sweep_kernel<512, 8>
             : E <= 16 ? sweep_kernel<512, 16> : E <= 24 ? sweep_kernel<512, 24>
             : sweep_kernel<512, 32>;
    if (threads == 128)
        return E <= 8 ? sweep_kernel<128, 8> : E <= 16 ? sweep_kernel<128, 16> : sweep_kernel<128, 32>;
    if (threads == 64)
        return E <= 8 ? sweep_kernel<64, 8> : E <= 16 ? sweep_kernel<64, 16> : sweep_kernel<64, 32>;
    return E <= 8 ? sweep_kernel<32, 8> : E <= 16 ? sweep_kernel<32, 16> : sweep_kernel<32, 32>;
}

// narrow CTAs for small samples: a round is a few elements per thread
static int start_threads(int n) { return n <= 512 ? 128 : n <= 2048 ? 256 : 512; }

static cudaError_t launch_start(const SweepArgs &w, cudaStream_t s)
{
    const int T = start_threads(w.n);
    void (*start)(SweepArgs) = T == 128 ? start_kernel<128> : T == 256 ? start_kernel<256> : start_kernel<512>;
    const size_t smem = start_smem_bytes(w.n, T);
    const cudaError_t e = allow_smem(start);
    if (e != cudaSuccess) return e;
    start<<<2 * w.nch, T, smem, s>>>(w);
    return cudaGetLastError();
}

cudaError_t launch_sweep_path(const SweepArgs &w0, cudaStream_t s)
{
    SweepArgs w = w0;
    const size_t ssm = sweep_smem_bytes(w.n, w.a.W, w.threads, w.R);
    void (*sweep)(SweepArgs) = sort_kernel(w.n, w.threads, w.a.nB > 0);
    cudaError_t e = allow_smem(sweep);
    if (e != cudaSuccess) return e;
    const size_t wsm = (size_t)w.split_bytes * kSplitWarps;
    void (*walk)(SweepArgs) = walk_kernel_of(w.n, w.a.nB > 0);
    if ((e = allow_smem(walk)) != cudaSuccess) return e;
    if (w.started && (e = launch_start(w, s)) != cudaSuccess) return e;
    for (int st = 0; st < w.nstages; ++st) {
        w.stage = st;
        sweep<<<2 * w.nch, w.threads, ssm, s>>>(w);
        if (st == 0 && w.sweep_done_event &&
            (e = cudaEventRecord((cudaEvent_t)w.sweep_done_event, s)) != cudaSuccess)
            return e;
        walk<<<w.walk_ctas, kSplitWarps * 32, wsm, s>>>(w);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// ---- the single-locus report --------------------------------------------------------
// The locus is a chunk of one core with kReportSteps markers of history on either
// side: its starting states and one marker of the sort give the run lengths of
// both directions, and then every step's S is independent of the others: a warp
// counts 32 steps from the boundaries with M up to its last one (RunCut).  The CTA
// that finishes last runs the six walks over those counts, 32 steps a turn, with
// the rules of walk_slot (the whole sample's S is the sum of the two classes').
// A walk that outlives the history is left to the per-step kernel (rest[q] = 1).
// Bound by the chain of launches and rounds, not by a step at a time (204
// haplotypes, 22,147 markers, a locus in a sweep: 269 us by the per-step kernel).
//
// How long the walks are shows only while they run, and walks of a dozen or two
// steps are done step by step before the starting states are (2,000 haplotypes, 80
// founders: 107 us step by step, 281 sorted; in a sweep 2,975 and 380).  So the two
// CTAs of the starting states run beside the six per-step walks, whichever is done
// first ends the other, and the results are the same (130 and 312 us).  Neither
// waits for the other: each looks at a counter as it goes.
struct QuitWhenStarted {
    const volatile int *started;
    // answer with the look of a step ago: its load holds nothing up, and the step
    // may be the last (5,000 haplotypes, 10 steps: 226 us against 369); not where a
    // step takes 60 us (10,000: 1,000 us against 830)
    bool late;
    int seen;
    __device__ __forceinline__ bool operator()()
    {
        const int before = seen;
        seen = *started;
        return __shfl_sync(FULLMASK, late ? before : seen, 0) >= 2;
    }
};

// where the word that start_state<T, true> quits by lies
static __host__ __device__ size_t report_quit_at(int n, int T) { return (start_smem_bytes(n, T) + 15) & ~(size_t)15; }
size_t report_start_smem(int n, int T) { return report_quit_at(n, T) + 16; }

template <int T>
__global__ void __launch_bounds__(T, 1) report_start_kernel(ReportArgs r, Scratch sc)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const SweepArgs &w = r.w;
    if (blockIdx.x < 2) {
        volatile int *quitting = (volatile int *)(smem + report_quit_at(w.n, T));
        if (threadIdx.x == 0) *quitting = 0;
        __syncthreads();
        const int np = (int)sweep_elements(w.n, w.threads);
        if (!start_state<T, true>(w, smem, blockIdx.x, w.a.k0, w.a.k1, (unsigned *)w.st + (size_t)blockIdx.x * np, np,
                                  quitting))
            return;
        if (threadIdx.x == 0) atomicAdd(r.started, 1);
        return;
    }
    const int q = (int)(blockIdx.x - 2) * (T / 32) + (int)(threadIdx.x >> 5);
    if (q >= 6) return;
    const bool done = trace_walk(w.a, w.a.k0, sc, smem + (size_t)(threadIdx.x >> 5) * slice_bytes(sc), q,
                                 (unsigned long long *)r.out.S, r.capacity, (long long *)r.out.len, r.out.stop, r.out.status,
                                 r.out.ihh, (unsigned long long *)r.out.denom, QuitWhenStarted{r.started, w.n <= 6144, 0});
    if (done && (threadIdx.x & 31) == 0) atomicAdd(r.walked, 1);
}
__global__ void __launch_bounds__(kSplitWarps * 32) report_kernel(ReportArgs r)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ bool last;
    namespace cg = cooperative_groups;
    const cg::thread_block_tile<32> tile = cg::tiled_partition<32>(cg::this_thread_block());
    const int lane = tile.thread_rank(), warp = threadIdx.x >> 5;
    const SweepArgs &w = r.w;
    if (*r.walked >= 6) return;                   // done step by step
    const int n = w.n;
    const long long m = w.a.m, x0 = w.a.k0;
    {
        const int dir = blockIdx.y;
        const int blk = blockIdx.x * kSplitWarps + warp, lo = 32 * blk + 1;
        const long long most = dir ? m - 1 - x0 : x0;            // steps inside the array
        if (lo <= most && lo <= kReportSteps) {                  // uniform over the warp
            const unsigned char *slot = w.slots + (size_t)dir * w.slot_bytes;
            const int n0 = ((const int *)slot)[0];
            const SplitSmem s = split_smem(smem + (size_t)warp * w.split_bytes,
                                           w.wscratch + ((size_t)(dir * gridDim.x + blockIdx.x) * kSplitWarps + warp) *
                                                            w.wscratch_bytes, n, false);
            for (int q = lane; q < s.nw; q += 32) s.O[q] = s.N[q] = 0u;
            tile.sync();
            unsigned K0, sup;
            const unsigned K = mark_window<1>(tile, s, (const uint4 *)(slot + 16), n, n0, lo + 31, true, false, 0, n,
                                              K0, sup);
            RunCut<1> rc;
            rc.lim = (unsigned)(lo + lane + 1) << 16;
            rc.last = 0u;
            rc.d[0] = 0u;
            rc.range(s, 0u, K0);
            rc.cut((unsigned)n0, 0u);
            r.S[(size_t)(2 * dir) * kReportSteps + lo - 1 + lane] = (rc.d[0] - (unsigned)n0) >> 1;
            rc.last = (unsigned)n0;
            rc.d[0] = 0u;
            rc.range(s, K0, K);
            rc.cut((unsigned)n, 0u);
            r.S[(size_t)(2 * dir + 1) * kReportSteps + lo - 1 + lane] = (rc.d[0] - (unsigned)(n - n0)) >> 1;
        }
    }
    __threadfence();                              // the counts before the tally
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(r.done, 1u) == gridDim.x * gridDim.y - 1u;
    __syncthreads();
    if (!last || warp >= 6) return;
    __threadfence();
    // ---- walk w = q / 2 (allele 1, allele 0, the whole sample), direction q % 2
    const int q = warp, wk = q >> 1, dir = q & 1;
    const unsigned n0 = ((const unsigned *)(w.slots + (size_t)dir * w.slot_bytes))[0], n1 = (unsigned)n - n0;
    const int hz = ((const int *)(w.slots + (size_t)dir * w.slot_bytes))[1];
    const unsigned D = (unsigned)c2i(wk == 0 ? n1 : wk == 1 ? n0 : (unsigned)n);
    if (q < 3 && lane == 0) r.out.denom[q] = (uint64_t)(unsigned)c2i(q == 0 ? n1 : q == 1 ? n0 : (unsigned)n);
    int status = D == 0u ? WALK_UNDEFINED : WALK_OK, stop = 0;
    double acc = 0.0;
    if (D != 0u) {
        const unsigned long long cutD = (unsigned long long)w.a.cut_num * D;
        unsigned prev = wk == 2 ? (unsigned)(c2i(n0) + c2i(n1)) : D;
        uint64_t *trace = r.out.S + (size_t)q * r.capacity;
        if (lane == 0 && r.capacity > 0) trace[0] = prev;
        const unsigned *Sd = r.S + (size_t)(2 * dir) * kReportSteps;
        bool walking = true;
        for (int i0 = 1; walking; i0 += 32) {
            const int i = i0 + lane;
            double gq = 0.0;
            int gk = 0;
            const long long step = dir ? 1 : -1, xl = x0 + step * i, xp = xl - step;
            if (xl < 0 || xl >= m) gk = WALK_EDGE;
            else {
                const long long p1 = __ldg(w.a.pos + xl), p0 = __ldg(w.a.pos + xp);
                const long long bp = dir ? p1 - p0 : p0 - p1;
                if (bp > w.a.max_gap) gk = WALK_GAP;
                else {
                    double gg;
                    if (w.a.physical) gg = (double)bp;
                    else {
                        const double g1 = __ldg(w.a.gmap + xl), g0 = __ldg(w.a.gmap + xp);
                        gg = dir ? g1 - g0 : g0 - g1;
                    }
                    if (bp > w.a.gap_scale) gg = gg * ((double)w.a.gap_scale / (double)bp);
                    gq = gg;
                }
            }
            unsigned S = 0u;
            if (gk != WALK_EDGE && i <= kReportSteps) {
                const unsigned s0 = __ldcg(Sd + i - 1), s1 = __ldcg(Sd + kReportSteps + i - 1);
                S = wk == 0 ? s1 : wk == 1 ? s0 : s0 + s1;
            }
            const unsigned km = tile.ballot(gk != 0), hm = tile.ballot(i > hz || i > kReportSteps);
            const int ke = km ? __ffs(km) - 1 : 32, he = hm ? __ffs(hm) - 1 : 32;
            const int end = ke <= he ? ke : he;
            const unsigned sm = tile.ballot((unsigned long long)w.a.cut_den * S < cutD);
            const int sl = sm ? __ffs(sm) - 1 : 32;
            const bool stops = sl < end;
            const int full = stops ? sl : end;
            unsigned sp = tile.shfl_up(S, 1);
            if (lane == 0) sp = prev;
            if (lane < full + (stops ? 1 : 0) && i < r.capacity) trace[i] = S;
            if (lane < full + (stops && w.a.crossing ? 1 : 0)) acc += (double)(sp + S) * gq;
            prev = tile.shfl(S, 31);
            if (stops) {
                stop = i0 + sl;
                walking = false;
            } else if (end < 32) {
                status = ke <= he ? tile.shfl(gk, ke & 31) : WALK_UNFINISHED;
                stop = i0 + end;
                walking = false;
            }
        }
    }
    acc = lane_sum_f64<32>(acc);
    if (lane != 0) return;
    r.rest[q] = status == WALK_UNFINISHED ? 1 : 0;
    if (status == WALK_UNFINISHED) return;
    r.out.len[q] = status == WALK_OK ? stop + 1 : status == WALK_UNDEFINED ? 0 : stop;
    r.out.stop[q] = stop;
    r.out.status[q] = (int8_t)status;
    r.out.ihh[q] = D ? acc / (2.0 * (double)D) : 0.0;
}

cudaError_t launch_report(const ReportArgs &r, const Scratch &sc, cudaStream_t s)
{
    const SweepArgs &w = r.w;
    const int T = start_threads(w.n), per = T / 32 < 6 ? T / 32 : 6;      // walks of a CTA
    void (*start)(ReportArgs, Scratch) = T == 128 ? report_start_kernel<128> : T == 256 ? report_start_kernel<256>
                                       : report_start_kernel<512>;
    const size_t a = report_start_smem(w.n, T), b = slice_bytes(sc) * (size_t)per;
    cudaError_t e = allow_smem(start);
    if (e != cudaSuccess) return e;
    start<<<2 + (6 + per - 1) / per, T, a > b ? a : b, s>>>(r, sc);
    void (*sweep)(SweepArgs) = sort_kernel(w.n, w.threads, w.a.nB > 0);
    const size_t ssm = sweep_smem_bytes(w.n, w.a.W, w.threads, 1);
    if ((e = allow_smem(sweep)) != cudaSuccess) return e;
    sweep<<<2, w.threads, ssm, s>>>(w);
    const size_t wsm = (size_t)w.split_bytes * kSplitWarps;
    if ((e = allow_smem(report_kernel, kFixedSmem)) != cudaSuccess) return e;
    report_kernel<<<dim3(kReportSteps / 32 / kSplitWarps, 2), kSplitWarps * 32, wsm, s>>>(r);
    return cudaGetLastError();
}

}  // namespace selscan
