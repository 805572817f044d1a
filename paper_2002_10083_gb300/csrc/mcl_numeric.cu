// The fused numeric pass of one MCL iteration (Algorithm 1: expansion,
// Prune, inflation) with a shared-memory accumulator of exact fixed-point
// sums.
//
// One CTA owns one output column j at a time (persistent grid, work list in
// longest-first order).  Products a_ik * a_kj are formed in FP32 and added
// as 64-bit integers: each product is scaled by 2^f_j, where 2^(62 - f_j)
// bounds the column sum s_j = sum_k a_kj colsum_k(A) (known before any
// product and bounding every product and every entry, all values being
// >= 0), and truncated.  Integer addition is associative, so an entry of
// B_*j does not depend on the order of its additions, on the window plan or
// on the CTA shape: runs are bit-identical.  The sum is exact up to the
// truncation of each product (below 2^-62 s_j), far below FP32 resolution
// for any entry that can survive the prune.
//
// The column's row span is cut into row windows sized from the output-size
// estimate (about PLAN entries each; windows of at most HS rows give every
// row its own slot, no hashing):
//
//   1. insert:  every product of the window is added into its slot: row - r0
//               in a window of at most HS rows, else linear probing from a
//               multiplicative hash (keys claimed by compare-and-swap), the
//               sum as two 32-bit words.  Four products per lane and round:
//               their first probes are issued together, then their low words'
//               additions, then the high words' with the carries;
//   2. extract: one scan of the table, which clears it: sums below both the
//               threshold and the running top-k bound are only counted, the
//               others update the statistics, and ranking keys (FP32 value
//               bits, row) above the bound go to a candidate buffer and past
//               its end to a spill in global memory; when the buffer was too
//               small it is cut back to the top ksel keys (radix select).
//
// A window takes two or three barriers.  (With the plan of each window
// published by one thread, a block scan for the candidates' positions and
// separate passes for extraction, emission and clearing there were ten.)
//
// Bound by instruction issue and the latency of the probes: 55% of issue
// slots busy at 32 warps per SM (64 registers), DRAM at 6%; about 2.3 clocks
// of an SM per hashed product.  First iteration of the 1M-vertex power-law
// graph, columns that are not dense in their span: 448 ms before the two
// barriers, the FP64-free column end and the wide selects, 394 ms with them.
// Not faster: the four probe chains of a lane advanced together (583 ms the
// iteration against 524), windows of 5,120 slots in 512-thread CTAs (696
// against 606), windows planned for 896 or 1,280 entries (501 and 494 against
// 492).
//
// Windows come from per-window product buckets (a counting pass and a
// scatter of (row, FP32 product) into window order); a column that is one
// small window from its sources, product by product; without bucket space
// from per-source cursors over the sorted rows (a warp or a lane per source).  A hashed window whose
// probe runs exceed PMAX slots is split by rows and redone (counted as a
// split), and the rest of the column starts at the width that fitted;
// results never depend on the size estimate.  Finally the prune rule picks
// m* (threshold / top-k / recovery), the kept keys are sorted by row,
// inflated, renormalised with an FP64 sum and written with chaos_j.
#include <climits>
#include <cstdint>

#include "mcl_column.cuh"
#include "mcl_device.cuh"
#include "mcl_internal.h"

namespace mcl {

constexpr int PMAX = 64;          // probe run that marks a hashed window as overflowed
// Products per source and window below which the walk over the sources gives
// each lane a source, and 4 of its products a round, instead of each warp one and
// 128.  Power-law graphs through the small configuration alone, 20k, 200k and
// 600k vertices: 26, 420 and 1,007 ms without lanes; 16.1, 131 and 340 ms with
// the line at 12; 11.6, 134 and 347 at 16; 10.6, 138 and 356 at 20.  Only for
// launches where columns can be many windows without buckets (WALK): its
// registers cost the others 1% (1M vertices: 505 -> 511 ms).
constexpr int LANE_MAX = 16;
// A column of so few sources and products in one window: every lane finds its own
// products' sources, with a search each, instead of a warp walking one source at a
// time.  300k vertices of 8 entries: 9.6 ms with the walk, 8.6 with the search;
// 1,000 of 250 (62,500 products a column): 0.42 ms with the walk, 0.63 with the
// search.  With the line at 65,536, 16,384, 8,192, 4,096 and 2,048 iteration 2 of
// the 2,000-vertex planted partition takes 0.43, 0.43, 0.39, 0.37 and 0.37 ms.
constexpr int FLAT_SOURCES = 256, FLAT_PRODUCTS = 4096;

struct ExpandShared {
    WinShared w;
    int cand;       // candidates of the window
    int went[2];    // entries of the window, by window parity
    int next[2];    // source counters, by window parity
    int full;       // a bucket, or a hashed window, was too small
    int upre[FLAT_SOURCES + 1];  // first product of each source
};

struct ExpandArgs {
    CscView A;
    PruneParams pp;
    ExpandBuffers b;
    int conf;
    int plan;
};

template <int T, int HS>
struct ExpandLayout {
    static constexpr size_t bytes(int ksel) {
        return (size_t)HS * 12 + 2 * 32 * 4 + 256 * 4 + 256 * 8 + sizeof(ExpandShared) + (size_t)(ksel + HS) * 8;
    }
};

template <int T, int HS, int MINB, bool WALK>
__global__ void __launch_bounds__(T, MINB) k_expand(ExpandArgs a) {
    const int PLAN = a.plan;  // distinct rows a window is planned for
    constexpr int IPT = 8, NW = T / 32;
    static_assert(HS >= (T / 32) * 256, "the row sort's counters fit in the key array");
    static_assert(HS % (T * 4) == 0, "the scan takes four slots per thread");
    static_assert(2 * HS >= SEL_BINS, "the selects' counters fit in the (empty) table");
    extern __shared__ __align__(16) unsigned char smem[];
    // sums' words and keys (row + 1, 0 = empty); idle lanes add 0 beyond the slots
    unsigned* lo32 = reinterpret_cast<unsigned*>(smem);
    unsigned* hi32 = lo32 + HS + 32;
    int* keys = reinterpret_cast<int*>(hi32 + HS + 32);
    unsigned long long* mhist = reinterpret_cast<unsigned long long*>(keys + HS);
    unsigned* hist = reinterpret_cast<unsigned*>(mhist + 256);
    const int ksel = a.pp.ksel;
    const int topcap = ksel + HS;
    uint64_t* top = reinterpret_cast<uint64_t*>(hist + 256);
    ExpandShared* es = reinterpret_cast<ExpandShared*>(top + topcap);
    WinShared* sh = &es->w;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const CscView& A = a.A;
    const ExpandBuffers& b = a.b;
    DevCounters* ctr = b.ctr;
    SrcMeta meta(b.cursors + (int64_t)blockIdx.x * 6 * b.cur_stride, b.cur_stride);
    // per-CTA bucket of (row, bits(product)) pairs
    int2* bkt = b.bucket_row ? reinterpret_cast<int2*>(b.bucket_row) + (int64_t)blockIdx.x * b.bucket_cap
                             : nullptr;
    // window starts and ends in the bucket (per CTA: WINDOW_MAX + 1 of each)
    int32_t* woff = b.woff ? b.woff + (int64_t)blockIdx.x * 2 * (WINDOW_MAX + 1) : nullptr;
    int32_t* wlim = woff ? woff + (WINDOW_MAX + 1) : nullptr;
    uint64_t* spill = b.spill + (int64_t)blockIdx.x * HS;
    const int wbeg = ctr->bin_off[a.conf * NZ], wend = ctr->bin_off[a.conf * NZ + NZ];
    if (ctr->err & ERR_STAGING) return;  // the iteration is redone without the graph

    for (int i = tid; i < HS + 32; i += T) lo32[i] = hi32[i] = 0u;
    for (int i = tid; i < HS; i += T) keys[i] = 0;
    const float theta = a.pp.theta;
    for (;;) {
        if (tid == 0) {
            sh->item = atomicAdd(&ctr->conf_ctr[a.conf], 1);
            es->cand = 0;
            es->went[0] = 0;
            es->went[1] = 0;
            es->next[0] = 0;
            es->full = 0;
        }
        __syncthreads();
        const int item = sh->item;
        if (wbeg + item >= wend) break;
        const int j = b.work[wbeg + item];
        const int64_t cb = A.colptr[j], ce = A.colptr[j + 1];
        const int d = (int)(ce - cb);
        const int lo = b.rlo[j], hiE = b.rhi[j] + 1;
        const bool empty = d == 0 || hiE <= lo;
        if (empty || d > b.cur_stride) {
            if (tid == 0) {
                if (!empty) set_err2(ctr, ERR_CURSOR);
                b.kept[j] = 0;
                b.chaos[j] = 0.0;
                b.bnnz[j] = 0;
            }
            __syncthreads();
            continue;
        }
        const int span = hiE - lo;
        const int64_t flops_j = b.flops[j];
        const double S = b.bsum[j];
        int64_t est = b.est[j];
        if (est < 1) est = 1;
        // ---- plan: about est / PLAN windows of equal row width.  With bucket
        // space the products go to per-window buckets, and a window that
        // overflows the table is split by rows (later windows of the column
        // then start at the split width).  Otherwise the window width adapts
        // to the entries seen. ----
        int64_t nw64 = (est + PLAN - 1) / PLAN;
        if (nw64 < 1) nw64 = 1;
        if (nw64 > span) nw64 = span;
        bool bucket = false;
        if (nw64 > 1 && bkt != nullptr && flops_j <= b.bucket_cap) {
            const int64_t wmax = WINDOW_MAX < HS ? WINDOW_MAX : HS;
            if (nw64 > wmax) nw64 = wmax;
            bucket = true;
        }
        int width = (int)(((int64_t)span + nw64 - 1) / nw64);
        if (width < HS && span > width) {
            // a window of at most HS rows has a slot per row (no hashing): use the
            // widest such windows
            const int64_t nid = ((int64_t)span + HS - 1) / HS;
            if (nid < nw64) {
                nw64 = nid;
                width = (int)(((int64_t)span + nw64 - 1) / nw64);
            }
        }
        const int nwin = (int)(((int64_t)span + width - 1) / width);
        if (nwin == 1) bucket = false;  // one window: straight from the sources
        const bool flat = nwin == 1 && d <= FLAT_SOURCES && flops_j <= FLAT_PRODUCTS;
        if (flat) {
            // the sources' first products by a scan over the block
            constexpr int PER = (FLAT_SOURCES + T - 1) / T;
            int len[PER], sum = 0;
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int i = tid * PER + q;
                len[q] = 0;
                if (i < d) {
                    const int k = A.rowidx[cb + i];
                    const int64_t ks = A.colptr[k];
                    len[q] = (int)(A.colptr[k + 1] - ks);
                    meta.ks[i] = ks;
                    meta.len[i] = len[q];
                    meta.cur[i] = 0;
                    meta.akj[i] = A.val[cb + i];
                }
                sum += len[q];
            }
            int tot;
            int at = block_scan_excl<T>(sum, &tot, sh->wsm);
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int i = tid * PER + q;
                if (i < d) es->upre[i] = at;
                at += len[q];
            }
            if (tid == 0) es->upre[d] = tot;
        } else {
            for (int i = tid; i < d; i += T) {
                const int k = A.rowidx[cb + i];
                const int64_t ks = A.colptr[k];
                meta.ks[i] = ks;
                meta.len[i] = (int)(A.colptr[k + 1] - ks);
                meta.cur[i] = 0;
                meta.akj[i] = A.val[cb + i];
            }
        }
        int ntop = 0;
        uint64_t tau = 0;
        unsigned long long qmin = 0;  // sums below it are neither candidates nor >= theta
        unsigned long long s_mt = 0;
        long long s_t = 0;
        unsigned s_n = 0;
        FixScale fx;
        fx.init(S);
        const bool plain = fx.plain();
        __syncthreads();

        if (bucket) {
            int* wcnt = reinterpret_cast<int*>(lo32);  // nwin <= HS counters each
            int* wcur = reinterpret_cast<int*>(hi32);
            FastDiv fdiv;
            fdiv.init((uint32_t)width);
            // Scatter (row, a_ik * a_kj) into the window buckets from the cursors wcur;
            // with a capacity capw per window (window w owns [w capw, (w + 1) capw))
            // a run that would pass its window's end sets es->full and writes
            // nothing past it.
            auto scatter = [&](int capw) {
                if (tid == 0) es->next[1] = 0;
                __syncthreads();
                for (;;) {
                    int kidx = 0;
                    if (lane == 0) kidx = atomicAdd(&es->next[1], 1);
                    kidx = __shfl_sync(FULL, kidx, 0);
                    if (kidx >= d) break;
                    const int len = meta.len[kidx];
                    const int64_t ks = meta.ks[kidx];
                    const int32_t* rows = A.rowidx + ks;
                    const float* vv = A.val + ks;
                    const float akj = meta.akj[kidx];
                    // the next 128 products are loaded while this chunk is routed
                    int rr[4];
                    float pv[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int p = 32 * c + lane;
                        rr[c] = p < len ? __ldg(rows + p) : 0;
                        pv[c] = p < len ? __ldg(vv + p) : 0.0f;
                    }
                    for (int pb = 0; pb < len; pb += 128) {
                        int nr[4];
                        float nv[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const int p = pb + 128 + 32 * c + lane;
                            nr[c] = p < len ? __ldg(rows + p) : 0;
                            nv[c] = p < len ? __ldg(vv + p) : 0.0f;
                        }
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const bool v = pb + 32 * c + lane < len;
                            const unsigned act = __ballot_sync(FULL, v);  // a prefix of the lanes
                            if (act == 0u) break;
                            const int row = rr[c];
                            const uint32_t w = v ? fdiv.div((uint32_t)(row - lo)) : 0xFFFFFFFFu;
                            const uint32_t wp = __shfl_up_sync(FULL, w, 1);
                            const bool head = v && (lane == 0 || wp != w);
                            const unsigned heads = __ballot_sync(FULL, head);
                            int base = 0;
                            if (head) {
                                const unsigned after = heads & ~((2u << lane) - 1u);
                                const int end = after ? __ffs(after) - 1 : __popc(act);
                                base = atomicAdd(wcur + w, end - lane);
                                if (capw > 0 && base + (end - lane) > ((int)w + 1) * capw)
                                    es->full = 1;
                            }
                            // the head of this lane's run: the highest head at or below it
                            const int hl = 31 - __clz(heads & ((2u << lane) - 1u));
                            base = __shfl_sync(FULL, base, hl);
                            if (v) {
                                const int pos = base + lane - hl;
                                if (capw == 0 || pos < ((int)w + 1) * capw)
                                    bkt[pos] = make_int2(row, __float_as_int(pv[c] * akj));
                            }
                        }
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            rr[c] = nr[c];
                            pv[c] = nv[c];
                        }
                    }
                }
                __syncthreads();
            };
            // products per window of equal row width are near their mean for
            // rows spread over the span: try fixed capacities of twice the mean
            // share first (1.25x left 13.5k of the 1M-vertex graph's columns to
            // the counting pass, 2x 1.6k)
            const int64_t capw64 = ((flops_j + nwin - 1) / nwin) * 2 + 64;
            bool counted = true;
            if (capw64 * nwin <= b.bucket_cap) {
                const int capw = (int)capw64;
                for (int i = tid; i < nwin; i += T) wcur[i] = i * capw;
                if (tid == 0) es->full = 0;
                __syncthreads();
                scatter(capw);
                counted = es->full != 0;  // a window was fuller than its capacity
                if (!counted)
                    for (int i = tid; i < nwin; i += T) {
                        woff[i] = i * capw;
                        wlim[i] = wcur[i];
                    }
                __syncthreads();
            }
            if (counted) {
                // ---- count the products of every window ----
                for (int i = tid; i < nwin; i += T) wcnt[i] = 0;
                if (tid == 0) es->next[1] = 0;
                __syncthreads();
                for (;;) {
                    int kidx = 0;
                    if (lane == 0) kidx = atomicAdd(&es->next[1], 1);
                    kidx = __shfl_sync(FULL, kidx, 0);
                    if (kidx >= d) break;
                    const int len = meta.len[kidx];
                    const int32_t* rows = A.rowidx + meta.ks[kidx];
                    for (int pb = 0; pb < len; pb += 128) {
                        int rr[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const int p = pb + 32 * c + lane;
                            rr[c] = p < len ? __ldg(rows + p) : 0;
                        }
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            // rows are sorted, so equal windows form runs of lanes
                            const bool v = pb + 32 * c + lane < len;
                            const unsigned act = __ballot_sync(FULL, v);  // a prefix of the lanes
                            if (act == 0u) break;
                            const uint32_t w = v ? fdiv.div((uint32_t)(rr[c] - lo)) : 0xFFFFFFFFu;
                            const uint32_t wp = __shfl_up_sync(FULL, w, 1);
                            const bool head = v && (lane == 0 || wp != w);
                            const unsigned heads = __ballot_sync(FULL, head);
                            if (head) {
                                const unsigned after = heads & ~((2u << lane) - 1u);
                                const int end = after ? __ffs(after) - 1 : __popc(act);
                                atomicAdd(wcnt + w, end - lane);
                            }
                        }
                    }
                }
                __syncthreads();
                // ---- window offsets (exclusive scan), scatter cursors ----
                {
                    const int per = (nwin + T - 1) / T;
                    const int i0 = min(nwin, tid * per), i1 = min(nwin, i0 + per);
                    int c = 0;
                    for (int i = i0; i < i1; ++i) c += wcnt[i];
                    int tot;
                    int run = block_scan_excl<T>(c, &tot, sh->wsm);
                    for (int i = i0; i < i1; ++i) {
                        woff[i] = run;
                        wcur[i] = run;
                        run += wcnt[i];
                        wlim[i] = run;
                    }
                    if (tid == 0 && (int64_t)tot != flops_j) set_err2(ctr, ERR_INTERNAL);
                }
                __syncthreads();
                scatter(0);
            }
            for (int i = tid; i < nwin; i += T) {
                wcnt[i] = 0;
                wcur[i] = 0;
            }
            if (tid == 0) es->full = 0;
            __syncthreads();
        }

        // four products per lane (row h + r0 of the window for h < wr) into their slots' sums
        auto add4 = [&](const unsigned (&h)[4], const float (&v)[4], unsigned wr, int r0, bool hash) {
            unsigned slot[4], ql[4], qh[4], old[4];
            int key[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const bool in = h[c] < wr;
                const unsigned long long q = plain ? fx.qplain(v[c]) : fx.qv(v[c]);
                ql[c] = in ? (unsigned)q : 0u;
                qh[c] = in ? (unsigned)(q >> 32) : 0u;
                key[c] = in ? (int)h[c] + r0 + 1 : 0;
                slot[c] = hash ? __umulhi((unsigned)key[c] * 0x9E3779B1u, (unsigned)HS) : h[c];
            }
            if (hash) {
                int got[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) got[c] = key[c] ? atomicCAS(keys + slot[c], 0, key[c]) : 0;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    for (int p = 0; got[c] != 0 && got[c] != key[c]; ++p) {
                        if (p == PMAX) {
                            es->full = 1;
                            key[c] = 0;
                            ql[c] = 0u;
                            qh[c] = 0u;
                            break;
                        }
                        slot[c] = slot[c] + 1 == HS ? 0 : slot[c] + 1;
                        got[c] = atomicCAS(keys + slot[c], 0, key[c]);
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (!hash && key[c]) keys[slot[c]] = key[c];
                slot[c] = key[c] ? slot[c] : (unsigned)(HS + lane);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) old[c] = atomicAdd(lo32 + slot[c], ql[c]);
#pragma unroll
            for (int c = 0; c < 4; ++c) atomicAdd(hi32 + slot[c], qh[c] + (old[c] + ql[c] < old[c] ? 1u : 0u));
        };

        // ---- windows: w counts the bucket windows; pw rows at once of the window's rows up to
        // we (all of them unless it has to be split); without buckets one window, pw rows at once ----
        int32_t* cur = meta.cur;
        int32_t* nxt = meta.nxt;
        const int batch = max(1, min(32, d / (4 * NW)));  // sources a warp takes at once
        const bool lanes = WALK && !bucket &&
                           (float)flops_j * (float)width < (float)LANE_MAX * (float)d * (float)span;
        int w = 0, pw = width;
        int we = bucket ? (int)min((int64_t)lo + width, (int64_t)hiE) : hiE;
        int r0 = lo, r1 = (int)min((int64_t)r0 + pw, (int64_t)we);
        for (int it = 0; r0 < hiE; ++it) {
            const unsigned wr = (unsigned)(r1 - r0);
            const bool hash = wr > (unsigned)HS;
            if (tid == 0) {
                es->next[(it + 1) & 1] = 0;
                es->went[(it + 1) & 1] = 0;
            }
            // ---- 1. insert the products of the window ----
            if (bucket) {
                const int be = wlim[w];
                int pb = woff[w] + warp * 128;
                int2 cx[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int p = pb + 32 * u + lane;
                    cx[u] = p < be ? bkt[p] : make_int2(INT_MAX, 0);
                }
                while (pb < be) {
                    unsigned h[4];
                    float v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        h[u] = (unsigned)(cx[u].x - r0);
                        v[u] = __int_as_float(cx[u].y);
                    }
                    pb += T * 4;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {  // the next round's, while these are added
                        const int p = pb + 32 * u + lane;
                        cx[u] = p < be ? bkt[p] : make_int2(INT_MAX, 0);
                    }
                    add4(h, v, wr, r0, hash);
                }
            } else if (flat && r0 == lo && r1 == hiE) {
                const int F = (int)flops_j;
                for (int tb = warp * 128; tb < F; tb += T * 4) {
                    unsigned h[4];
                    float v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int t = tb + 32 * u + lane;
                        h[u] = 0xFFFFFFFFu;
                        v[u] = 0.0f;
                        if (t < F) {
                            int s0 = 0, s1 = d;  // upre[s0] <= t < upre[s1]
                            while (s1 - s0 > 1) {
                                const int m = (s0 + s1) >> 1;
                                if (es->upre[m] <= t) s0 = m; else s1 = m;
                            }
                            const int64_t p = meta.ks[s0] + (t - es->upre[s0]);
                            h[u] = (unsigned)(__ldg(A.rowidx + p) - r0);
                            v[u] = __fmul_rn(__ldg(A.val + p), meta.akj[s0]);
                        }
                    }
                    add4(h, v, wr, r0, hash);
                }
            } else {
                // a warp per source and 128 of its products a round; with few products per
                // source and window a lane per source and four
                int* next = &es->next[it & 1];
                const int take = lanes ? 32 : batch;
                const int step = lanes ? 1 : 32;
                for (;;) {
                    int k0 = 0;
                    if (lane == 0) k0 = atomicAdd(next, take);
                    k0 = __shfl_sync(FULL, k0, 0);
                    if (k0 >= d) break;
                    const int k1 = min(k0 + take, d);
                    for (int s = lanes ? k0 + lane : k0; s < k1; s += lanes ? 32 : 1) {
                        const int len = meta.len[s];
                        const int64_t ks = meta.ks[s];
                        const float akj = meta.akj[s];
                        int pos = cur[s];
                        while (pos < len) {
                            unsigned h[4];
                            float v[4];
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const int p = pos + step * c + (lanes ? 0 : lane);
                                h[c] = (unsigned)((p < len ? __ldg(A.rowidx + ks + p) : INT_MAX) - r0);
                                v[c] = p < len ? __ldg(A.val + ks + p) : 0.0f;
                            }
                            int nin = 0;
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                v[c] = __fmul_rn(v[c], akj);
                                nin += lanes ? (int)(h[c] < wr) : __popc(__ballot_sync(FULL, h[c] < wr));
                            }
                            add4(h, v, wr, r0, hash);
                            pos += nin;
                            if (nin < 4 * step) break;
                        }
                        if (lanes || lane == 0) nxt[s] = pos;
                    }
                }
            }
            __syncthreads();
            if (es->full) {  // split: a quarter of the rows at once from here on
                __syncthreads();  // every thread has read the flag
                for (int i = tid; i < HS; i += T) {
                    lo32[i] = 0u;
                    hi32[i] = 0u;
                    keys[i] = 0;
                }
                if (tid == 0) {
                    es->full = 0;  // before the barrier: the redone window may set it again
                    atomicAdd(&ctr->splits, 1ull);
                }
                __syncthreads();
                pw = max(1, (r1 - r0) / 4);
                r1 = r0 + pw;
                continue;
            }
            // ---- 2. extract: one scan of the table, which it clears ----
            const unsigned slots = hash ? (unsigned)HS : (wr + 127u) & ~127u;
            unsigned n0 = s_n;
            for (unsigned h = tid * 4; h < slots; h += T * 4) {  // four slots; whole warps
                uint4* pl = reinterpret_cast<uint4*>(lo32 + h);
                uint4* ph = reinterpret_cast<uint4*>(hi32 + h);
                int4* pk = reinterpret_cast<int4*>(keys + h);
                const uint4 l4 = *pl, h4 = *ph;
                const int4 k4 = *pk;
                const unsigned xl[4] = {l4.x, l4.y, l4.z, l4.w}, xh[4] = {h4.x, h4.y, h4.z, h4.w};
                const int kk[4] = {k4.x, k4.y, k4.z, k4.w};
                unsigned big = 0;  // slots to look at
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const unsigned long long q = ((unsigned long long)xh[u] << 32) | xl[u];
                    s_n += kk[u] != 0;
                    big |= kk[u] != 0 && q >= qmin ? 1u << u : 0u;
                }
                while (__any_sync(FULL, big != 0u)) {  // one slot per lane and round
                    uint64_t key = 0;
                    if (big) {
                        const unsigned g = h + (unsigned)__ffs(big) - 1u;
                        big &= big - 1u;
                        const unsigned long long q = ((unsigned long long)hi32[g] << 32) | lo32[g];
                        const float v = fx.value(q);
                        if (v >= theta) {
                            ++s_t;
                            s_mt += q;
                        }
                        key = make_key(v, keys[g] - 1);
                    }
                    const bool take = key > tau;
                    const unsigned m = __ballot_sync(FULL, take);
                    if (m) {
                        int base = 0;
                        if (lane == 0) base = atomicAdd(&es->cand, __popc(m));
                        const int at = ntop + __shfl_sync(FULL, base, 0) + __popc(m & lanemask_lt());
                        if (take) {
                            if (at < topcap)
                                top[at] = key;
                            else
                                spill[at - topcap] = key;
                        }
                    }
                }
                *pl = make_uint4(0u, 0u, 0u, 0u);
                *ph = make_uint4(0u, 0u, 0u, 0u);
                *pk = make_int4(0, 0, 0, 0);
            }
            n0 = __reduce_add_sync(FULL, s_n - n0);
            if (lane == 0 && n0) atomicAdd(&es->went[it & 1], (int)n0);
            __syncthreads();
            const int have = ntop + es->cand, went = es->went[it & 1];
            __syncthreads();
            if (tid == 0) es->cand = 0;
            if (have > topcap) {  // cut back to the ksel largest
                const int over = have - topcap;
                tau = block_select_wide<T>(top, topcap, spill, over, ksel, lo32, &sh->bs, sh->wsm);
                ntop = compact_stable<T, IPT>(top, topcap, tau, sh->wsm);
                for (int i = tid; i < over; i += T) {
                    const uint64_t x = spill[i];
                    if (x >= tau) top[ntop + atomicAdd(&es->cand, 1)] = x;
                }
                __syncthreads();
                ntop = ksel;
                if (tid == 0) es->cand = 0;
                qmin = fx.lower(fminf(theta, key_val(tau)));
                __syncthreads();
            } else {
                ntop = have;
            }
            // ---- 3. next window ----
            int32_t* t = cur;  // cursors advance past the window
            cur = nxt;
            nxt = t;
            const bool whole = r1 - r0 >= width;
            if (went < PLAN / 2 && (bucket ? !whole : pw < (1 << 29))) {
                pw = bucket ? min(width, pw * 2) : pw * 2;
            } else if (!bucket && went > PLAN + PLAN / 2 && pw > 1) {
                pw /= 2;
            }
            r0 = r1;
            if (bucket && r0 >= we) {
                do ++w; while (w < nwin && wlim[w] == woff[w]);  // empty windows
                r0 = w < nwin ? lo + w * width : hiE;
                we = (int)min((int64_t)r0 + width, (int64_t)hiE);
            }
            r1 = (int)min((int64_t)r0 + pw, (int64_t)we);
        }
        double dv[1] = {0.0};
        long long qv[3] = {s_t, (long long)s_n, (long long)s_mt};
        block_sum<T>(dv, 0, qv, 3, &sh->bs);
        int mstar = 0;
        double ch = 0.0;
        const int64_t obase = b.off[j];
        // the table's key array is free here: counters of the row sort
        finish_column<T, IPT, false>(top, ntop, topcap, a.pp, S, (unsigned long long)qv[2], fx.f, qv[0], b.cap[j],
                                     b.tmp_row + (obase - b.tmp_off0),
                                     b.tmp_val + (obase - b.tmp_off0), hist, mhist, lo32, sh, ctr,
                                     lo, span, reinterpret_cast<unsigned*>(keys), &mstar, &ch);
        for (int i = tid; i < (T / 32) * 256; i += T) keys[i] = 0;
        if (tid == 0) {
            b.kept[j] = mstar;
            b.chaos[j] = ch;
            b.bnnz[j] = qv[1];
            if (qv[1] > est) atomicAdd(&ctr->misses, 1ull);
        }
    }
}

// Configurations: 0 = small columns (128 threads, 1024 slots, windows of
// 512 rows, 8 CTAs per SM); 1 = everything else, in one of three shapes
// that the autotuner picks from (threads, table slots, CTAs per SM):
//   table 0: 256 x 2048 x 4,  table 1: 512 x 4096 x 2,  table 2: 256 x 4096 x 2.
// The candidate buffer holds ksel + HS keys (a window adds at most HS).
template <int T_, int HS_, int MINB_>
struct Conf {
    static constexpr int T = T_, HS = HS_, MINB = MINB_;
};
using Conf0 = Conf<128, 1024, 8>;
using Conf1a = Conf<256, 2048, 4>;
using Conf1b = Conf<512, 4096, 2>;
using Conf1c = Conf<256, 4096, 2>;

template <class C>
static size_t conf_smem(int ksel) { return ExpandLayout<C::T, C::HS>::bytes(ksel); }

template <class C>
static int conf_grid(int ksel, int num_sms) {
    const size_t smem = conf_smem<C>(ksel);
    auto kern = k_expand<C::T, C::HS, C::MINB, false>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, C::T, smem);
    if (occ < 1) occ = 1;
    return occ * num_sms;
}

template <class C>
static void conf_launch(int conf, const CscView& A, const PruneParams& pp, const ExpandBuffers& b,
                        int grid, bool walk, cudaStream_t s) {
    int plan = conf == 0 ? C::HS / 2 : (pp.plan > 0 ? pp.plan : C::HS / 2);
    if (plan > (3 * C::HS) / 4) plan = (3 * C::HS) / 4;
    if (plan < 64) plan = 64;
    ExpandArgs a{A, pp, b, conf, plan};
    const size_t smem = conf_smem<C>(pp.ksel);
    auto kern = walk ? k_expand<C::T, C::HS, C::MINB, true> : k_expand<C::T, C::HS, C::MINB, false>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<grid, C::T, smem, s>>>(a);
}

// Bytes of candidate spill: a window's slots for every CTA of the largest configuration.
size_t numeric_spill_bytes(const PruneParams& pp, int num_sms) {
    const size_t hs = pp.table == 0 ? Conf1a::HS : Conf1b::HS;
    static_assert(Conf1b::HS == Conf1c::HS, "one size for both wide shapes");
    const size_t b0 = (size_t)numeric_grid(0, pp, num_sms) * Conf0::HS * 8;
    const size_t b1 = (size_t)numeric_grid(CONF_LARGE, pp, num_sms) * hs * 8;
    const size_t b2 = direct_spill_bytes(direct_grid(pp.ksel, num_sms));
    return b0 > b1 ? (b0 > b2 ? b0 : b2) : (b1 > b2 ? b1 : b2);
}

int numeric_grid(int conf, const PruneParams& pp, int num_sms) {
    if (conf == CONF_DIRECT) return direct_grid(pp.ksel, num_sms);
    if (conf == 0) return conf_grid<Conf0>(pp.ksel, num_sms);
    return pp.table == 1 ? conf_grid<Conf1b>(pp.ksel, num_sms)
                         : pp.table == 2 ? conf_grid<Conf1c>(pp.ksel, num_sms)
                                         : conf_grid<Conf1a>(pp.ksel, num_sms);
}

void launch_numeric(int conf, const CscView& A, const PruneParams& pp, const ExpandBuffers& b,
                    int grid, bool walk, cudaStream_t s) {
    if (conf == CONF_DIRECT)
        launch_direct(A, pp, b, grid, s);
    else if (conf == 0)
        conf_launch<Conf0>(conf, A, pp, b, grid, walk, s);
    else if (pp.table == 1)
        conf_launch<Conf1b>(conf, A, pp, b, grid, walk, s);
    else if (pp.table == 2)
        conf_launch<Conf1c>(conf, A, pp, b, grid, walk, s);
    else
        conf_launch<Conf1a>(conf, A, pp, b, grid, walk, s);
    count_launches(1);
}

// ---------------------------------------------------------------------------
// the prune rule alone on a materialised matrix (same candidate machinery;
// a column's entries are already row-ordered)
// ---------------------------------------------------------------------------

constexpr int PR_MINB = 4;  // 64 registers: the selects and scans need the warps
constexpr int PR_T = 256, PR_IPT = 8, PR_VC = PR_T * PR_IPT;

struct PruneShared {
    WinShared w;
    int cnt[2][PR_IPT * PR_T / 32];  // candidates per round and warp, by chunk parity
    unsigned bins[SEL_BINS];         // counters of the selects, zero between them
};

// The candidates and statistics of one column of m entries, in row order.
// load(i, &row, &q) gives entry i with its fixed-point value; a chunk of 2,048
// entries is read once, coalesced, and kept in registers while the positions
// of its candidates are counted (ballots per round and warp, in entry order).
template <class Load>
__device__ __forceinline__ void prune_candidates(int64_t m, const FixScale& fx, float theta, Load load,
                                                 uint64_t* top, int topcap, int ksel, PruneShared* ps, int& ntop, long long& s_t,
                                                 unsigned long long& s_mt) {
    constexpr int NW = PR_T / 32;
    static_assert(PR_IPT * NW == 64, "two counts per lane");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint64_t tau = 0;
    int par = 0;
    for (int64_t base = 0; base < m; base += PR_VC, par ^= 1) {
        uint64_t key[PR_IPT];
#pragma unroll
        for (int u = 0; u < PR_IPT; ++u) {
            const int64_t i = base + u * PR_T + tid;
            key[u] = 0;
            if (i < m) {
                int row;
                float v;
                unsigned long long q;
                load(i, row, v, q);
                if (v >= theta) {
                    ++s_t;
                    s_mt += q;
                }
                key[u] = make_key(v, row);
            }
        }
        auto count = [&](int* cnt, int& at) {  // at: this lane's two counts' exclusive offset
#pragma unroll
            for (int u = 0; u < PR_IPT; ++u) {
                const unsigned b = __ballot_sync(FULL, key[u] > tau);
                if (lane == 0) cnt[u * NW + warp] = __popc(b);
            }
            __syncthreads();
            const int c0 = cnt[2 * lane], c1 = cnt[2 * lane + 1];
            int incl = c0 + c1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += y;
            }
            at = incl - c0 - c1;
            return __shfl_sync(FULL, incl, 31);
        };
        int* cnt = ps->cnt[par];
        int at;
        int C = count(cnt, at);
        if (ntop + C > topcap) {  // C <= PR_VC = topcap - ksel, so ntop > ksel here
            tau = block_select_wide<PR_T>(top, ntop, top, 0, ksel, ps->bins, &ps->w.bs, ps->w.wsm);
            ntop = compact_stable<PR_T, PR_IPT>(top, ntop, tau, ps->w.wsm);
            C = count(cnt, at);
        }
#pragma unroll
        for (int u = 0; u < PR_IPT; ++u) {
            const int f = u * NW + warp;  // its offset: lane f / 2, plus the lane's first count if odd
            int o = __shfl_sync(FULL, at, f >> 1);
            if (f & 1) o += cnt[f - 1];
            const bool take = key[u] > tau;
            const unsigned b = __ballot_sync(FULL, take);
            if (take) top[ntop + o + __popc(b & lanemask_lt())] = key[u];
        }
        ntop += C;
        __syncthreads();
    }
}

// FIXED: a merged product whose entries are the exact 64-bit fixed-point sums
// of the numeric pass (rows sorted per column; column j's scale from the
// column sum bsum[j]): the statistics and keys of the numeric pass, so the
// same iteration.  Otherwise FP32 values, whose mass at or above the threshold
// is summed in the fixed point of the column's own sum.
struct PruneArgs {
    int32_t n;
    const int64_t* colptr;
    const int32_t* rowidx;
    const float* val;
    const unsigned long long* q;
    const double* sum;
    PruneParams pp;
    ExpandBuffers b;
};

template <bool FIXED>
__global__ void __launch_bounds__(PR_T, PR_MINB) k_prune(PruneArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int ksel = a.pp.ksel;
    const int topcap = ksel + PR_VC;
    unsigned long long* mhist = reinterpret_cast<unsigned long long*>(smem);
    unsigned* hist = reinterpret_cast<unsigned*>(mhist + 256);  // 16-byte aligned whatever ksel is
    uint64_t* top = reinterpret_cast<uint64_t*>(hist + 256);
    PruneShared* ps = reinterpret_cast<PruneShared*>(top + topcap);
    WinShared* sh = &ps->w;
    const int tid = threadIdx.x;
    const ExpandBuffers& b = a.b;
    for (int i = tid; i < SEL_BINS; i += PR_T) ps->bins[i] = 0u;
    for (;;) {
        if (tid == 0) sh->item = atomicAdd(&b.ctr->work_ctr, 1);
        __syncthreads();
        const int64_t j = sh->item;
        __syncthreads();
        if (j >= a.n) break;
        const int64_t cb = a.colptr[j], m = a.colptr[j + 1] - cb;
        const double S = a.sum[j];
        FixScale fx;
        fx.init(S);
        int ntop = 0;
        unsigned long long s_mt = 0;
        long long s_t = 0;
        const int32_t* rows = a.rowidx + cb;
        const float* vals = FIXED ? nullptr : a.val + cb;
        const unsigned long long* qs = FIXED ? a.q + cb : nullptr;
        prune_candidates(
            m, fx, a.pp.theta,
            [&](int64_t i, int& row, float& v, unsigned long long& q) {
                row = rows[i];
                if (FIXED) {
                    q = qs[i];
                    v = fx.value(q);
                } else {
                    v = vals[i];
                    q = fx.qv(v);
                }
            },
            top, topcap, ksel, ps, ntop, s_t, s_mt);
        double dv[1] = {0.0};
        long long qv[2] = {s_t, (long long)s_mt};
        block_sum<PR_T>(dv, 0, qv, 2, &sh->bs);
        int mstar = 0;
        double ch = 0.0;
        const int64_t obase = b.off[j];
        finish_column<PR_T, 8, true>(top, ntop, topcap, a.pp, S, (unsigned long long)qv[1], fx.f, qv[0], b.cap[j],
                                     b.tmp_row + (obase - b.tmp_off0),
                                     b.tmp_val + (obase - b.tmp_off0), hist, mhist, ps->bins, sh, b.ctr, 0,
                                     0, nullptr, &mstar, &ch);
        if (tid == 0) {
            b.kept[j] = mstar;
            b.chaos[j] = ch;
            b.bnnz[j] = m;
        }
    }
}

template <bool FIXED>
static void prune_launch(const PruneArgs& a, int num_sms, cudaStream_t s) {
    if (a.n == 0) return;
    const size_t smem = (size_t)(a.pp.ksel + PR_VC) * 8 + 256 * 4 + 256 * 8 + sizeof(PruneShared);
    cudaFuncSetAttribute(k_prune<FIXED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_prune<FIXED>, PR_T, smem);
    if (occ < 1) occ = 1;
    int grid = occ * num_sms;
    if ((int64_t)grid > a.n) grid = (int)a.n;
    cudaMemsetAsync(&a.b.ctr->work_ctr, 0, sizeof(int), s);
    k_prune<FIXED><<<grid, PR_T, smem, s>>>(a);
    count_launches(1);
}

void launch_prune_fixed(int32_t n, const int64_t* colptr, const int32_t* rowidx,
                        const unsigned long long* q, const double* bsum, const PruneParams& pp,
                        const ExpandBuffers& b, int num_sms, cudaStream_t s) {
    prune_launch<true>(PruneArgs{n, colptr, rowidx, nullptr, q, bsum, pp, b}, num_sms, s);
}

// Column sums of B in b.colsum.
void launch_prune(const CscView& B, const PruneParams& pp, const ExpandBuffers& b, int num_sms,
                  cudaStream_t s) {
    prune_launch<false>(PruneArgs{B.n, B.colptr, B.rowidx, B.val, nullptr, b.colsum, pp, b}, num_sms, s);
}

}  // namespace mcl

