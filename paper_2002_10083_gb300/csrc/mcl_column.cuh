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
    double red;    // result of an ordered sum
};

// Sum of f(s[i]) over i < m in an order that does not depend on the block
// size: warp 0 alone, lane l taking i = l, l + 32, ..., then a fixed
// butterfly; the result is broadcast to the block.  Two barriers.
template <class F>
__device__ __forceinline__ double ordered_sum(const uint64_t* s, int m, F f, double* slot) {
    if (threadIdx.x < 32) {
        double x = 0.0;
        for (int i = threadIdx.x; i < m; i += 32) x += f(s[i]);
        x = warp_sum(x);
        if (threadIdx.x == 0) *slot = x;
    }
    __syncthreads();
    const double r = *slot;
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

// Finish a column: prune rule on the candidate keys top[0..ntop) plus exact
// statistics, then the kept keys in row order (sorted here unless the
// buffer is already row-ordered) written with inflation (pp.inflate) or
// their B values; returns m* and chaos_j via the pointers.
// For an unordered buffer, rows lie in [row_lo, row_lo + row_span); the
// radix sort uses top[m .. topcap) and rscratch ((T / 32) * 256 counters)
// as scratch when they suffice, the bitonic network otherwise.
template <int T, int IPT, bool ROW_ORDERED>
__device__ void finish_column(uint64_t* top, int ntop, int topcap, const PruneParams& pp, double S,
                              double MT, long long Tt, int64_t cap, int32_t* out_row,
                              float* out_val, unsigned* hist, unsigned long long* mhist,
                              WinShared* sh, DevCounters* ctr, int row_lo, int row_span,
                              unsigned* rscratch, int* mstar_out, double* chaos_out) {
    const int tid = threadIdx.x;
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
    int m = mstar > 0 ? compact_stable<T, IPT>(top, ntop, cut, sh->wsm) : 0;
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
    const float rr = pp.r;
    const double U = pp.inflate ? ordered_sum(top, m, [rr](uint64_t x) {
        return (double)inflate_value(key_val(x), rr); }, &sh->red) : 0.0;
    const double invU = U > 0.0 ? 1.0 / U : 0.0;
    double amax = 0.0;
    for (int i = tid; i < m; i += T) {
        const uint64_t x = top[i];
        const float v = key_val(x);
        float outv = v;
        if (pp.inflate) {
            const double a = (double)inflate_value(v, pp.r) * invU;
            outv = (float)a;
            amax = a > amax ? a : amax;
        }
        out_row[i] = key_row(x);
        out_val[i] = outv;
    }
    double ch = 0.0;
    if (pp.inflate) {
        const double mx = block_max_d<T>(amax, &sh->bs);
        const double sq = ordered_sum(top, m, [rr, invU](uint64_t x) {
            const double a = (double)inflate_value(key_val(x), rr) * invU;
            return a * a; }, &sh->red);
        ch = mx - sq;
        if (ch < 0.0) ch = 0.0;
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
