// Device parts of the numeric pass that its kernels share: block scans, the
// row sort, the prune rule and the end of a column (mcl_numeric.cu,
// mcl_direct.cu).
#pragma once

#include <cfloat>
#include <climits>
#include <cstdint>

#include "mcl_device.cuh"
#include "mcl_internal.h"

namespace mcl {

__device__ __forceinline__ void set_err2(DevCounters* c, unsigned bit) { atomicOr(&c->err, bit); }

struct WinShared {
    BlockScratch bs;
    int wsm[34];
    int item;
    double red;    // result of a mass
    double sum4[2][4];  // partial sums of the warps
    float max4[4];
    Quotient quo;       // by the sum
    double chaos;
    int flag;
};

// Exclusive block scan of one int per thread; *total gets the sum.  Three
// barriers (the last protects the scratch for the next call).
template <int T>
__device__ __forceinline__ int block_scan_excl(int x, int* total, int* wsm) {
    constexpr int NW = T / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wsm[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int w = lane < NW ? wsm[lane] : 0;
        int wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < NW) wsm[lane] = wi - w;
        if (lane == 31) wsm[32] = wi;
    }
    __syncthreads();
    const int res = wsm[warp] + incl - x;
    *total = wsm[32];
    __syncthreads();
    return res;
}

// Radix select by count over the distinct keys of A ++ B (bit 63 clear):
// returns kappa with #{x : x >= kappa} == M exactly (1 <= M <= na + nb).  Most
// significant digit first; stops as soon as the chosen bin holds exactly the
// keys still needed, returning its prefix with zero low bits.  Digits of 11
// bits: two passes for the values of a column where eight-bit digits take four
// (the first of which sees two or three different exponents), and one shared
// atomic per key.  bins: SEL_BINS counters, zero on entry and on return.
constexpr int SEL_BINS = 2048;
template <int T>
__device__ uint64_t block_select_wide(const uint64_t* A, int na, const uint64_t* B, int nb, int M,
                                      unsigned* bins, BlockScratch* bs, int* wsm) {
    constexpr int PER = SEL_BINS / T;
    const int tid = threadIdx.x, tot = na + nb;
    uint64_t prefix = 0;
    int need = M;
    for (int shift = 52, bits = 11;;) {
        const uint64_t himask = ~0ull << (shift + bits);
        const unsigned dmask = (1u << bits) - 1u;
        for (int i = tid; i < tot; i += T) {
            const uint64_t x = cat_at(A, na, B, i);
            if ((x & himask) == prefix) atomicAdd(bins + ((unsigned)(x >> shift) & dmask), 1u);
        }
        __syncthreads();
        // thread t owns the bins from SEL_BINS - 1 - t PER down
        int c[PER], sum = 0;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            unsigned* bin = bins + (SEL_BINS - 1 - tid * PER - q);
            c[q] = (int)*bin;
            *bin = 0u;
            sum += c[q];
        }
        int total;
        int before = block_scan_excl<T>(sum, &total, wsm);
        if (before < need && before + sum >= need) {
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                if (before < need && before + c[q] >= need) {
                    bs->sel_prefix = prefix | ((uint64_t)(SEL_BINS - 1 - tid * PER - q) << shift);
                    bs->sel_need = need - before;
                    bs->sel_done = c[q] == need - before;
                }
                before += c[q];
            }
        }
        __syncthreads();
        prefix = bs->sel_prefix;
        need = bs->sel_need;
        const bool done = bs->sel_done != 0;
        __syncthreads();
        if (done || shift == 0) break;
        bits = shift < 11 ? shift : 11;
        shift -= bits;
    }
    return prefix;
}

// Stable in-place compaction of a[0..n) keeping keys >= cut; returns the
// new length.  Each thread owns IPT consecutive elements per round; all
// reads of a round precede its writes (the scan's barriers), and outputs
// never land past the round's inputs.
template <int T, int IPT>
__device__ int compact_stable(uint64_t* a, int n, uint64_t cut, int* wsm) {
    int outpos = 0;
    for (int base = 0; base < n; base += T * IPT) {
        uint64_t x[IPT];
        int c = 0;
        const int i0 = base + threadIdx.x * IPT;
#pragma unroll
        for (int q = 0; q < IPT; ++q) {
            const int i = i0 + q;
            x[q] = i < n ? a[i] : 0ull;
            if (i < n && x[q] >= cut) ++c;
        }
        int tot;
        int o = outpos + block_scan_excl<T>(c, &tot, wsm);
#pragma unroll
        for (int q = 0; q < IPT; ++q)
            if (i0 + q < n && x[q] >= cut) a[o++] = x[q];
        outpos += tot;
        __syncthreads();
    }
    return outpos;
}

// Scratch per CTA in global memory (stride = cur_stride sources): source
// column start (int64), length, two cursor arrays (read / write; swapped
// after a window succeeds) and a_kj.
struct SrcMeta {
    int64_t* ks;
    int32_t* len;
    int32_t* cur;
    int32_t* nxt;
    float* akj;
    __device__ SrcMeta(int32_t* base, int64_t stride) {
        ks = reinterpret_cast<int64_t*>(base);
        len = base + 2 * stride;
        cur = len + stride;
        nxt = cur + stride;
        akj = reinterpret_cast<float*>(nxt + stride);
    }
};

// Stable LSD radix sort of s[0..n) ascending by the field s[i] >> 32, whose
// values are below 2^bits, eight bits per pass.  Warp w owns a contiguous
// segment; per pass each warp counts its digits (whist[w][digit]), one block
// scan over (digit, warp) turns the counts into start offsets, and each warp
// scatters its segment in order (equal digits of a 32-element chunk are
// ranked by lane), so the sort is stable.  tmp holds n elements; whist holds
// (T / 32) * 256 counters.  Ends with a barrier.
template <int T>
__device__ void block_radix_sort_hi(uint64_t* s, uint64_t* tmp, int n, int bits, unsigned* whist,
                                    int* wsm) {
    constexpr int NW = T / 32;
    constexpr int DPT = T >= 256 ? 1 : 256 / T;  // digits per thread in the offset scan
    static_assert(T >= 256 ? T % 256 == 0 : 256 % T == 0, "digits per thread");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int seg = ((n + NW - 1) / NW + 31) & ~31;
    const int w0 = min(n, warp * seg), w1 = min(n, w0 + seg);
    uint64_t* src = s;
    uint64_t* dst = tmp;
    for (int sh = 0; sh < bits; sh += 8) {
        for (int i = tid; i < NW * 256; i += T) whist[i] = 0u;
        __syncthreads();
        for (int base = w0; base < w1; base += 32) {
            const int i = base + lane;
            const bool v = i < w1;
            const unsigned dg = v ? (unsigned)(src[i] >> (32 + sh)) & 255u : 0u;
            const unsigned act = __ballot_sync(FULL, v);
            if (v) {
                const unsigned grp = __match_any_sync(act, dg);
                if (__ffs(grp) - 1 == lane) whist[warp * 256 + dg] += (unsigned)__popc(grp);
            }
            __syncwarp();
        }
        __syncthreads();
        {
            const bool own = tid * DPT < 256;  // threads beyond the 256 digits scan zeros
            unsigned c[DPT][NW];
            int tot = 0;
#pragma unroll
            for (int q = 0; q < DPT; ++q)
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    c[q][w] = own ? whist[w * 256 + tid * DPT + q] : 0u;
                    tot += (int)c[q][w];
                }
            int total;
            int run = block_scan_excl<T>(tot, &total, wsm);
            if (own) {
#pragma unroll
                for (int q = 0; q < DPT; ++q)
#pragma unroll
                    for (int w = 0; w < NW; ++w) {
                        whist[w * 256 + tid * DPT + q] = (unsigned)run;
                        run += (int)c[q][w];
                    }
            }
        }
        __syncthreads();
        for (int base = w0; base < w1; base += 32) {
            const int i = base + lane;
            const bool v = i < w1;
            uint64_t x = 0;
            unsigned dg = 0;
            if (v) {
                x = src[i];
                dg = (unsigned)(x >> (32 + sh)) & 255u;
            }
            const unsigned act = __ballot_sync(FULL, v);
            if (v) {
                const unsigned grp = __match_any_sync(act, dg);
                dst[whist[warp * 256 + dg] + __popc(grp & lanemask_lt())] = x;
                __syncwarp(act);
                if (__ffs(grp) - 1 == lane) whist[warp * 256 + dg] += (unsigned)__popc(grp);
            }
            __syncwarp();
        }
        __syncthreads();
        uint64_t* t = src;
        src = dst;
        dst = t;
    }
    if (src != s) {
        for (int i = tid; i < n; i += T) s[i] = src[i];
        __syncthreads();
    }
}

// Sorts s[0..n) ascending by the field s[i] >> 32 (distinct values below
// span) by distribution: NB buckets of equal width, a scan of their counts, and
// a thread per bucket for the few keys in it.  About eight barriers, where
// three radix passes take twenty-four.  Returns false, with s as it was, when a
// bucket has more than BSORT_MAX keys (rows bunched together).  tmp holds n
// elements; cnt holds NB counters, NB a multiple of T.  Power-law graphs of 20k,
// 200k and 600k vertices: 4.65, 58.9 and 141 ms an iteration, 4.89, 61.1 and 146
// with radix passes alone; 6 and 24 keys a bucket the same as 12.
constexpr int BSORT_MAX = 12;
template <int T>
__device__ bool block_bucket_sort_hi(uint64_t* s, uint64_t* tmp, int n, unsigned span, unsigned* cnt,
                                     int* wsm, int* flag) {
    constexpr int NB = T / 32 * 256, PER = NB / T;
    const int tid = threadIdx.x;
    // bucket = floor(x scale / 2^32) < NB for x < span <= 2^31
    const unsigned scale = span > (unsigned)NB ? (unsigned)(((unsigned long long)NB << 32) / span) : 0u;
    auto bucket = [&](uint64_t x) {
        const unsigned r = (unsigned)(x >> 32);
        return scale ? __umulhi(r, scale) : r;
    };
    for (int i = tid; i < NB; i += T) cnt[i] = 0u;
    if (tid == 0) *flag = 0;
    __syncthreads();
    for (int i = tid; i < n; i += T)
        if (atomicAdd(cnt + bucket(s[i]), 1u) >= (unsigned)BSORT_MAX) *flag = 1;
    __syncthreads();
    if (*flag) {
        __syncthreads();
        return false;
    }
    unsigned c[PER];
    int sum = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        c[q] = cnt[tid * PER + q];
        sum += (int)c[q];
    }
    int total;
    int at = block_scan_excl<T>(sum, &total, wsm);
    const int first = at;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        cnt[tid * PER + q] = (unsigned)at;
        at += (int)c[q];
    }
    __syncthreads();
    for (int i = tid; i < n; i += T) {
        const uint64_t x = s[i];
        tmp[atomicAdd(cnt + bucket(x), 1u)] = x;
    }
    __syncthreads();
    // this thread's buckets, ordered by insertion, back to s
    at = first;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int m = (int)c[q];
        for (int a = 0; a < m; ++a) {
            const uint64_t x = tmp[at + a];
            int b = a;
            for (; b > 0 && s[at + b - 1] > x; --b) s[at + b] = s[at + b - 1];
            s[at + b] = x;
        }
        at += m;
    }
    __syncthreads();
    return true;
}

// Value mass of the keys >= cut in a[0..n), as an exact integer sum of the
// values in fixed point (each truncated at 2^-50 of the largest value), so
// that it does not depend on the order of a's elements.  Warp 0 sums; the
// result is broadcast to the block.
template <int T>
__device__ double mass_at_or_above(const uint64_t* a, int n, uint64_t cut, WinShared* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t kmax = 0;
    for (int i = threadIdx.x; i < n; i += T) kmax = a[i] > kmax ? a[i] : kmax;
    kmax = warp_max(kmax);
    if (lane == 0) sh->bs.q[3][warp] = (long long)kmax;
    __syncthreads();
    if (warp == 0) {
        uint64_t y = lane < T / 32 ? (uint64_t)sh->bs.q[3][lane] : 0ull;
        y = warp_max(y);
        const float maxv = key_val(y);
        int e = 0;
        frexpf(maxv > 0.0f ? maxv : 1.0f, &e);  // every value < 2^e
        const int s50 = 50 - e;
        unsigned long long acc = 0;
        for (int i = lane; i < n; i += 32)
            if (a[i] >= cut) acc += fixed_of(key_val(a[i]), s50);
        acc = warp_sum(acc);
        if (lane == 0) sh->red = ldexp((double)acc, -s50);
    }
    __syncthreads();
    const double r = sh->red;
    __syncthreads();
    return r;
}

constexpr int SUM_T = 128;  // threads that add a column's powers

// Few keys: every rank by counting.  FEW_KEYS keys at most (one per thread).
// 300k vertices of 8 entries (up to some 90 candidates): 8.6 ms, 9.7 with at most
// 64 keys, 10.1 without; 2M of 2: 52.9 ms, 60.0 without; the third iteration of a
// 10k-vertex planted partition 1.61 ms, 1.71 without.
constexpr int FEW_KEYS = 128;

// The prune rule (below) on top[0..ntop), ntop <= FEW_KEYS: on return the kept
// keys are the first m* of top, in row order.  Where the cut is the threshold
// a key needs no rank; otherwise it is compared with every other: its rank,
// and the mass of the keys from it up in the fixed point of block_select_mass
// (mhist holds the keys' masses), give the same cuts as the radix selects,
// whose passes cost more than this column's whole work.
template <int T>
__device__ int finish_few(uint64_t* top, int ntop, const PruneParams& pp, double S, bool theta_cut,
                          long long Tt, int64_t cap, unsigned* hist, unsigned long long* mhist, WinShared* sh,
                          DevCounters* ctr) {
    static_assert(FEW_KEYS <= T && FEW_KEYS <= 256, "one key per thread");
    const int tid = threadIdx.x;
    const bool mine = tid < ntop;
    const uint64_t x = mine ? top[tid] : 0ull;
    const int q = (int)(Tt < (long long)pp.K ? Tt : (long long)pp.K);
    int mstar;
    bool kept;
    if (theta_cut) {
        mstar = (int)Tt;  // the entries >= theta, all among the candidates
        kept = mine && x >= ((uint64_t)__float_as_uint(pp.theta) << 32);
    } else {
        int rank = 0;
        if (q >= pp.Krec) {
            mstar = pp.Krec;
            if (mine)
                for (int k = 0; k < ntop; ++k) rank += top[k] > x;
        } else {
            // scale of the masses: the largest value below 2^e
            if (tid < FEW_KEYS) {
                const uint64_t y = warp_max(x);
                if ((tid & 31) == 0) sh->bs.q[3][tid >> 5] = (long long)y;
            }
            __syncthreads();
            uint64_t kmax = 0;
#pragma unroll
            for (int w = 0; w < FEW_KEYS / 32; ++w) {
                const uint64_t y = (uint64_t)sh->bs.q[3][w];
                kmax = y > kmax ? y : kmax;
            }
            int e = 0;
            const float maxv = key_val(kmax);
            frexpf(maxv > 0.0f ? maxv : 1.0f, &e);
            const int s50 = 50 - e;
            if (mine) mhist[tid] = fixed_of(key_val(x), s50);
            if (tid == 0) {
                sh->red = 0.0;
                sh->flag = INT_MAX;
            }
            __syncthreads();
            unsigned long long mass = 0;
            if (mine)
                for (int k = 0; k < ntop; ++k) {
                    const uint64_t y = top[k];
                    rank += y > x;
                    mass += y >= x ? mhist[k] : 0ull;
                }
            const double target = (double)pp.p * S;
            bool enough = false;  // Tt <= K: known to fall short
            if (Tt > pp.K) {
                if (mine && rank == pp.K - 1) sh->red = ldexp((double)mass, -s50);
                __syncthreads();
                enough = target <= 0.0 || sh->red >= target;
            }
            if (enough) {
                mstar = q;
            } else {
                const double tf = ceil(ldexp(target, s50));
                if (tf < 9.0e18 && mine && mass >= (unsigned long long)tf) atomicMin(&sh->flag, rank + 1);
                __syncthreads();
                mstar = min(sh->flag, ntop);
            }
        }
        if (mstar > pp.Krec) mstar = pp.Krec;
        if (mstar > ntop) mstar = ntop;
        if ((int64_t)mstar > cap) {  // cannot happen for validated input; never write past cap
            if (tid == 0) set_err2(ctr, ERR_INTERNAL);
            mstar = (int)cap;
        }
        kept = mine && rank < mstar;
    }
    // positions: the kept keys' low words are larger for smaller rows, and never 0
    if (tid < FEW_KEYS) hist[tid] = kept ? (uint32_t)x : 0u;
    __syncthreads();
    int at = 0;
    if (kept) {
        const uint32_t r = (uint32_t)x;
        const uint4* h4 = reinterpret_cast<const uint4*>(hist);
        for (int k = 0; k < ntop; k += 4) {
            const uint4 y = h4[k >> 2];
            at += (y.x > r) + (y.y > r) + (y.z > r) + (y.w > r);
        }
    }
    __syncthreads();
    if (kept && (int64_t)at < cap) top[at] = x;
    __syncthreads();
    return (int64_t)mstar > cap ? (int)cap : mstar;
}

// Finish a column: prune rule on the candidate keys top[0..ntop) plus exact
// statistics, then the kept keys in row order (sorted here unless the
// buffer is already row-ordered) written with inflation (pp.inflate) or
// their B values; returns m* and chaos_j via the pointers.
// For an unordered buffer, rows lie in [row_lo, row_lo + row_span); the
// row sort uses top[m .. topcap) and rscratch ((T / 32) * 256 counters)
// as scratch when they suffice, the bitonic network otherwise.
template <int T, int IPT, bool ROW_ORDERED>
__device__ void finish_column(uint64_t* top, int ntop, int topcap, const PruneParams& pp, double S,
                              unsigned long long mt, int f, long long Tt, int64_t cap, int32_t* out_row,
                              float* out_val, unsigned* hist, unsigned long long* mhist,
                              unsigned* bins, WinShared* sh, DevCounters* ctr, int row_lo, int row_span,
                              unsigned* rscratch, int* mstar_out, double* chaos_out) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // FP64 sums, quotients and the test of the mass at or above theta are one
    // warp's, not every warp's: their instructions take 16 clocks of the SM each,
    // and a column of a few entries took 23k clocks in here (the recovery's
    // targets, where that test fails, are computed by every warp)
    const int q = (int)(Tt < (long long)pp.K ? Tt : (long long)pp.K);
    bool theta_cut = false;  // the entries >= theta are at most K and carry the mass to recover
    if (q < pp.Krec && Tt <= pp.K) {
        if (tid == 0) {
            const double goal = (double)pp.p * S;
            sh->flag = goal <= 0.0 || ldexp((double)mt, -f) >= goal;
        }
        __syncthreads();
        theta_cut = sh->flag != 0;
        __syncthreads();
    }
    int m;
    if (ntop <= FEW_KEYS) {
        m = finish_few<T>(top, ntop, pp, S, theta_cut, Tt, cap, hist, mhist, sh, ctr);
    } else {
    double mq = 0.0;
    uint64_t kq = 0;
    // q >= Krec: m* = min(Krec, max(q, m_rec)) = Krec whatever the recovery
    // finds, so neither the top-q mass nor m_rec is needed
    const bool krec_bound = q >= pp.Krec;
    if (!krec_bound && Tt > pp.K) {
        kq = block_select_wide<T>(top, ntop, top, 0, pp.K, bins, &sh->bs, sh->wsm);
        mq = mass_at_or_above<T>(top, ntop, kq, sh);
    }
    int mstar;
    uint64_t cut;
    bool have_cut = false;
    if (krec_bound) {
        mstar = pp.Krec;
    } else if (theta_cut || (Tt > pp.K && ((double)pp.p * S <= 0.0 || mq >= (double)pp.p * S))) {
        mstar = q;
        if (mstar <= pp.Krec) {
            if (Tt <= pp.K) {
                cut = (uint64_t)__float_as_uint(pp.theta) << 32;  // exactly the entries >= theta
            } else {
                cut = kq;
            }
            have_cut = true;
        }
    } else {
        uint64_t kr = 0;
        int mr = 0;
        const int found =
            block_select_mass<T>(top, ntop, (double)pp.p * S, &kr, &mr, hist, mhist, &sh->bs);
        mstar = found ? mr : ntop;
        if (found && mstar <= pp.Krec) {
            cut = kr;
            have_cut = true;
        }
    }
    if (mstar > pp.Krec) mstar = pp.Krec;
    if (mstar > ntop) mstar = ntop;
    if ((int64_t)mstar > cap) {  // cannot happen for validated input; never write past cap
        if (tid == 0) set_err2(ctr, ERR_INTERNAL);
        mstar = (int)cap;
        have_cut = false;
    }
    if (!have_cut || mstar == 0) {
        if (mstar == 0)
            cut = ~0ull;
        else if (mstar >= ntop)
            cut = 0ull;
        else
            cut = block_select_wide<T>(top, ntop, top, 0, mstar, bins, &sh->bs, sh->wsm);
    }
    // the kept keys (exactly m* of them: keys are distinct) to the front
    m = mstar > 0 ? compact_stable<T, IPT>(top, ntop, cut, sh->wsm) : 0;
    if (m != mstar) {
        if (tid == 0) set_err2(ctr, ERR_INTERNAL);
        m = m < mstar ? m : mstar;
    }
    if (!ROW_ORDERED && m > 1) {
        // re-key as (row - row_lo, value bits) and sort ascending: rows are distinct
        for (int i = tid; i < m; i += T) {
            const uint64_t x = top[i];
            top[i] = ((uint64_t)(uint32_t)(key_row(x) - row_lo) << 32) | (x >> 32);
        }
        __syncthreads();
        if (rscratch != nullptr && topcap - m >= m) {
            const int bits = 32 - __clz(row_span - 1);
            if (!block_bucket_sort_hi<T>(top, top + m, m, (unsigned)row_span, rscratch, sh->wsm, &sh->flag))
                block_radix_sort_hi<T>(top, top + m, m, bits, rscratch, sh->wsm);
        } else {
            block_sort_asc<T>(top, m);
        }
        for (int i = tid; i < m; i += T) {
            const uint64_t x = top[i];
            top[i] = make_key(__uint_as_float((uint32_t)x), (int)(x >> 32) + row_lo);
        }
        __syncthreads();
    }
    }
    // ---- inflation, renormalisation, chaos_j and the output ----
    // U = sum u and the sum of u^2 over the kept u = v^r, in an order that does not depend on
    // the block size: thread t of the first SUM_T takes i = t, t + SUM_T, ..., a warp's lanes
    // are added by a fixed butterfly and the warps' sums in turn (warps beyond m add 0).
    // a = u (1 / U) in FP64, rounded to FP32.
    const float rr = pp.r;
    if (!pp.inflate) {
        for (int i = tid; i < m; i += T) {
            const uint64_t x = top[i];
            out_row[i] = key_row(x);
            out_val[i] = key_val(x);
        }
        if (tid == 0) {
            *mstar_out = m;
            *chaos_out = 0.0;
        }
        __syncthreads();
        return;
    }
    if (tid < SUM_T) {
        double su = 0.0, su2 = 0.0;
        float mu = 0.0f;
        if (warp * 32 < m) {
            for (int i = tid; i < m; i += SUM_T) {
                const float u = inflate_value(key_val(top[i]), rr);
                const double x = float_to_double(u);
                su += x;
                su2 += x * x;
                mu = fmaxf(mu, u);
            }
            su = warp_sum(su);
            su2 = warp_sum(su2);
            mu = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(mu)));  // mu >= 0
        }
        if (lane == 0) {
            sh->sum4[0][warp] = su;
            sh->sum4[1][warp] = su2;
            sh->max4[warp] = mu;
        }
    }
    __syncthreads();
    if (tid == 0) {
        const double U = ((sh->sum4[0][0] + sh->sum4[0][1]) + sh->sum4[0][2]) + sh->sum4[0][3];
        const double U2 = ((sh->sum4[1][0] + sh->sum4[1][1]) + sh->sum4[1][2]) + sh->sum4[1][3];
        const float mu = fmaxf(fmaxf(sh->max4[0], sh->max4[1]), fmaxf(sh->max4[2], sh->max4[3]));
        Quotient quo;
        quo.init(U);
        sh->quo = quo;
        const double inv = quo.inv;
        // max a - sum a^2; the largest u gives the largest a
        const double ch = (double)mu * inv - (U2 * inv) * inv;
        sh->chaos = ch < 0.0 ? 0.0 : ch;
        *mstar_out = m;
        *chaos_out = sh->chaos;
    }
    __syncthreads();
    const Quotient quo = sh->quo;
    for (int i = tid; i < m; i += T) {
        const uint64_t x = top[i];
        const float u = inflate_value(key_val(x), rr);
        float a;
        if (!quo.plain() || !quo.quick(u, &a)) a = (float)((double)u * quo.inv);
        out_row[i] = key_row(x);
        out_val[i] = a;
    }
    __syncthreads();
}

// Exact unsigned 32-bit division by a run-time constant d >= 1 with one
// multiply-high (the round-up method of Granlund and Montgomery, 1994):
// l = ceil(log2 d), m = floor(2^32 (2^l - d) / d) + 1,
// q = (t + ((x - t) >> 1)) >> (l - 1) with t = mulhi(m, x); d = 1 is x.
struct FastDiv {
    uint32_t m;
    int l;
    __device__ void init(uint32_t d) {
        l = 0;
        while ((1ull << l) < d) ++l;
        m = l == 0 ? 0u : (uint32_t)((((1ull << l) - d) << 32) / d + 1ull);
    }
    __device__ __forceinline__ uint32_t div(uint32_t x) const {
        if (l == 0) return x;
        const uint32_t t = __umulhi(m, x);
        return (t + ((x - t) >> 1)) >> (l - 1);
    }
};

}  // namespace mcl
