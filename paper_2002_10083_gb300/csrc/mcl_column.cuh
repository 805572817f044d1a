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
    int next;
    // window plan published by thread 0 (rows [pr0, pr1) when prs)
    int pf0, pf1, pr0, pr1, prs, pdone;
    // per-window flags, double-buffered by window parity
    int ovf2[2];   // the window exceeded its table
    int went2[2];  // entries of the window's table
    int next2[2];  // source counter of the warp-per-source insert
    double red;    // result of a mass
    double red4[4];  // partial results of an ordered sum
    int flag;
};

// Sum of f(i) over i < m in an order that does not depend on the block size
// (at least SUM_T threads): thread t of the first SUM_T takes i = t, t + SUM_T,
// ..., each warp adds its lanes by a fixed butterfly and the warps' sums are
// added in turn; the result is broadcast to the block.  Two barriers.
constexpr int SUM_T = 128;
template <class F>
__device__ __forceinline__ double ordered_sum(int m, F f, double* slots) {
    if (threadIdx.x < SUM_T) {
        double x = 0.0;
        for (int i = threadIdx.x; i < m; i += SUM_T) x += f(i);
        x = warp_sum(x);
        if ((threadIdx.x & 31) == 0) slots[threadIdx.x >> 5] = x;
    }
    __syncthreads();
    const double r = ((slots[0] + slots[1]) + slots[2]) + slots[3];
    __syncthreads();
    return r;
}

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
// elements; cnt holds NB counters, NB a multiple of T.
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
            if (a[i] >= cut) acc += __float2ull_rz(ldexpf(key_val(a[i]), s50));
        acc = warp_sum(acc);
        if (lane == 0) sh->red = ldexp((double)acc, -s50);
    }
    __syncthreads();
    const double r = sh->red;
    __syncthreads();
    return r;
}

// Few keys: every rank by counting.  FEW_KEYS keys at most (one per thread).
constexpr int FEW_KEYS = 128;

// The prune rule (below) on top[0..ntop), ntop <= FEW_KEYS: on return the kept
// keys are the first m* of top, in row order.  Where the cut is the threshold
// a key needs no rank; otherwise it is compared with every other: its rank,
// and the mass of the keys from it up in the fixed point of block_select_mass
// (mhist holds the keys' masses), give the same cuts as the radix selects,
// whose passes cost more than this column's whole work.
template <int T>
__device__ int finish_few(uint64_t* top, int ntop, const PruneParams& pp, double S, double MT, long long Tt,
                          int64_t cap, unsigned* hist, unsigned long long* mhist, WinShared* sh,
                          DevCounters* ctr) {
    static_assert(FEW_KEYS <= T && FEW_KEYS <= 256, "one key per thread");
    const int tid = threadIdx.x;
    const bool mine = tid < ntop;
    const uint64_t x = mine ? top[tid] : 0ull;
    const double target = (double)pp.p * S;
    const int q = (int)(Tt < (long long)pp.K ? Tt : (long long)pp.K);
    int mstar;
    bool kept;
    if (q < pp.Krec && Tt <= pp.K && (target <= 0.0 || MT >= target)) {
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
            if (mine) mhist[tid] = __float2ull_rz(ldexpf(key_val(x), s50));
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
            double mq = MT;
            if (Tt > pp.K) {
                if (mine && rank == pp.K - 1) sh->red = ldexp((double)mass, -s50);
                __syncthreads();
                mq = sh->red;
            }
            if (target <= 0.0 || mq >= target) {
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
                              double MT, long long Tt, int64_t cap, int32_t* out_row,
                              float* out_val, unsigned* hist, unsigned long long* mhist,
                              WinShared* sh, DevCounters* ctr, int row_lo, int row_span,
                              unsigned* rscratch, int* mstar_out, double* chaos_out) {
    const int tid = threadIdx.x;
    int m;
    if (ntop <= FEW_KEYS) {
        m = finish_few<T>(top, ntop, pp, S, MT, Tt, cap, hist, mhist, sh, ctr);
    } else {
    const double target = (double)pp.p * S;
    const int q = (int)(Tt < (long long)pp.K ? Tt : (long long)pp.K);
    double mq = 0.0;
    uint64_t kq = 0;
    // q >= Krec: m* = min(Krec, max(q, m_rec)) = Krec whatever the recovery
    // finds, so neither the top-q mass nor m_rec is needed
    const bool krec_bound = q >= pp.Krec;
    if (krec_bound) {
    } else if (Tt <= pp.K) {
        mq = MT;
    } else {
        kq = block_select_count<T>(top, ntop, top, 0, pp.K, hist, &sh->bs);
        mq = mass_at_or_above<T>(top, ntop, kq, sh);
    }
    int mstar;
    uint64_t cut;
    bool have_cut = false;
    if (krec_bound) {
        mstar = pp.Krec;
    } else if (target <= 0.0 || mq >= target) {
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
        const int f = block_select_mass<T>(top, ntop, target, &kr, &mr, hist, mhist, &sh->bs);
        mstar = f ? mr : ntop;
        if (f && mstar <= pp.Krec) {
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
            cut = block_select_count<T>(top, ntop, top, 0, mstar, hist, &sh->bs);
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
    const float rr = pp.r;
    const double U = pp.inflate ? ordered_sum(m, [top, rr](int i) {
        return float_to_double(inflate_value(key_val(top[i]), rr)); }, sh->red4) : 0.0;
    const double invU = U > 0.0 ? 1.0 / U : 0.0;
    double ch = 0.0;
    if (pp.inflate) {
        float umax = 0.0f;
        const double sq = ordered_sum(m, [&](int i) {
            const uint64_t x = top[i];
            const float u = inflate_value(key_val(x), rr);
            const double a = float_to_double(u) * invU;
            umax = fmaxf(umax, u);
            out_row[i] = key_row(x);
            out_val[i] = (float)a;
            return a * a; }, sh->red4);
        // the largest u gives the largest a (rounding is monotone)
        const double mx = block_max_d<T>((double)umax * invU, &sh->bs);
        ch = mx - sq;
        if (ch < 0.0) ch = 0.0;
    } else {
        for (int i = tid; i < m; i += T) {
            const uint64_t x = top[i];
            out_row[i] = key_row(x);
            out_val[i] = key_val(x);
        }
    }
    if (tid == 0) {
        *mstar_out = m;
        *chaos_out = ch;
    }
    __syncthreads();
}

// Append the candidates an enumerator yields to top[0..ntop); first cuts
// the buffer back to ksel entries if they would not fit.  `count(tau)`
// returns this thread's number of keys > tau; `emit(tau, dst, base)` writes
// this thread's keys at dst[base ...] (base: its exclusive scan offset).
template <int T, int IPT, class Enum>
__device__ __forceinline__ void append_candidates(Enum& en, uint64_t* top, int topcap, int ksel,
                                                  int& ntop, uint64_t& tau, int c, unsigned* hist,
                                                  WinShared* sh) {
    int C;
    int base = block_scan_excl<T>(c, &C, sh->wsm);
    if (ntop + C > topcap) {
        // invariant: C <= window capacity = topcap - ksel, so ntop > ksel here
        const uint64_t kap = block_select_count<T>(top, ntop, top, 0, ksel, hist, &sh->bs);
        ntop = compact_stable<T, IPT>(top, ntop, kap, sh->wsm);
        tau = kap;
        c = en.count(tau);
        base = block_scan_excl<T>(c, &C, sh->wsm);
    }
    en.emit(tau, top + ntop, base);
    ntop += C;
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
