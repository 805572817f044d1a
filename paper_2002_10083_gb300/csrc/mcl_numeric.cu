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
//               multiplicative hash (int32 row keys claimed by
//               compare-and-swap, uint64 sums added with integer atomics);
//   2. extract: over the table, the ranking key (FP32 value bits, row) of
//               every entry replaces its sum in place, with the exact column
//               statistics (count, count and mass at or above the
//               threshold); the keys above the running top-k bound tau go to
//               a candidate buffer that is cut back to the top ksel keys
//               (radix select) when full;
//   3. clear:   the table.
//
// Windows come from per-window product buckets (a counting pass and a
// scatter of (row, FP32 product) into window order) or, without bucket
// space, from per-source cursors over the sorted rows.  A hashed window whose
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

// ---------------------------------------------------------------------------
// the accumulator: int32 row keys and uint64 fixed-point sums per slot
// ---------------------------------------------------------------------------

constexpr int KEY_EMPTY = -1;
constexpr int PMAX = 64;  // probe run that marks a hashed window as overflowed

// *p += v in shared memory, as two 32-bit atomics: the low word's returns the
// old value, whose carry goes into the high word's.  A 64-bit shared-memory
// addition is a compare-and-swap loop on this GPU: 1.7 per clock and SM at
// random slots against 3.9 (11 for a 32-bit one).
__device__ __forceinline__ void red_add_u64(unsigned long long* p, unsigned long long v) {
    unsigned* w = reinterpret_cast<unsigned*>(p);
    const unsigned lo = (unsigned)v;
    const unsigned old = atomicAdd(w, lo);
    const unsigned hi = (unsigned)(v >> 32) + (old + lo < old ? 1u : 0u);
    if (hi) atomicAdd(w + 1, hi);
}

__device__ __forceinline__ int cas_shared(int* p, int cmp, int val) {
    int old;
    asm volatile("atom.shared.cas.b32 %0, [%1], %2, %3;"
                 : "=r"(old)
                 : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(cmp), "r"(val)
                 : "memory");
    return old;
}

// Home slot of a row in a hashed window: multiplicative hash scaled to HS
// slots (any HS).
template <int HS>
__device__ __forceinline__ int table_home(int row) {
    return (int)(((uint64_t)((uint32_t)row * 0x9E3779B1u) * (uint64_t)HS) >> 32);
}

// Add q at `row`: slot row - r0 in an identity window (rows of the window
// span at most HS slots; every writer of a slot stores the same row), else
// linear probing from the row's hash, an empty slot claimed by
// compare-and-swap.  A probe run of PMAX slots sets *ovf and adds nothing.
template <int HS, bool IDENT>
__device__ __forceinline__ void acc_add(int row, unsigned long long q, int r0, int* keys,
                                        unsigned long long* vals, int* ovf) {
    if (IDENT) {
        const unsigned h = (unsigned)(row - r0);
        if (h >= (unsigned)HS) {  // cannot happen: a window's segments hold rows in [r0, r1)
            *ovf = 2;
            return;
        }
        keys[h] = row;
        red_add_u64(vals + h, q);
        return;
    }
    int h = table_home<HS>(row);
    for (int p = 0; p < PMAX; ++p) {
        int k = *reinterpret_cast<volatile int*>(keys + h);
        if (k == KEY_EMPTY) {
            k = cas_shared(keys + h, KEY_EMPTY, row);
            if (k == KEY_EMPTY) k = row;
        }
        if (k == row) {
            red_add_u64(vals + h, q);
            return;
        }
        if (++h == HS) h = 0;
    }
    *ovf = 1;
}

// Expected entries per source and window below which a window walks its
// sources one per lane instead of one per warp.
constexpr int LANE_MODE_MAX = 12;

// The ranking keys of a window's table after extraction (0: empty slot;
// thread t takes slots t, t + T, ...).
template <int T, int HS>
struct KeyEnum {
    const uint64_t* vk;
    __device__ int count(uint64_t tau) const {
        int c = 0;
        for (int h = threadIdx.x; h < HS; h += T) c += vk[h] > tau;
        return c;
    }
    __device__ void emit(uint64_t tau, uint64_t* dst, int base) const {
        for (int h = threadIdx.x; h < HS; h += T) {
            const uint64_t k = vk[h];
            if (k > tau) dst[base++] = k;
        }
    }
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
        return (size_t)HS * 12 + (size_t)(ksel + HS) * 8 + 256 * 4 + 256 * 8 + sizeof(WinShared);
    }
};

template <int T, int HS, int MINB>
__global__ void __launch_bounds__(T, MINB) k_expand(ExpandArgs a) {
    const int PLAN = a.plan;  // distinct rows a window is planned for
    constexpr int IPT = 8;
    static_assert(HS >= (T / 32) * 256, "the row sort's counters fit in the key array");
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned long long* vals = reinterpret_cast<unsigned long long*>(smem);
    int* keys = reinterpret_cast<int*>(vals + HS);
    uint64_t* vkeys = reinterpret_cast<uint64_t*>(vals);  // ranking keys after extraction
    uint64_t* top = reinterpret_cast<uint64_t*>(keys + HS);
    const int ksel = a.pp.ksel;
    const int topcap = ksel + HS;  // a window adds at most HS candidates
    unsigned* hist = reinterpret_cast<unsigned*>(top + topcap);
    unsigned long long* mhist = reinterpret_cast<unsigned long long*>(hist + 256);
    WinShared* sh = reinterpret_cast<WinShared*>(mhist + 256);

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
    const int wbeg = ctr->bin_off[a.conf * NZ], wend = ctr->bin_off[a.conf * NZ + NZ];
    if (ctr->err & ERR_STAGING) return;  // the iteration is redone without the graph

    for (int i = tid; i < HS; i += T) {
        keys[i] = KEY_EMPTY;
        vals[i] = 0ull;
    }
    const float theta = a.pp.theta;
    for (;;) {
        if (tid == 0) sh->item = atomicAdd(&ctr->conf_ctr[a.conf], 1);
        __syncthreads();
        const int item = sh->item;
        __syncthreads();
        if (wbeg + item >= wend) break;
        const int j = b.work[wbeg + item];
        const int64_t cb = A.colptr[j], ce = A.colptr[j + 1];
        const int d = (int)(ce - cb);
        const int lo = b.rlo[j], hiE = b.rhi[j] + 1;
        if (d == 0 || hiE <= lo) {
            if (tid == 0) {
                b.kept[j] = 0;
                b.chaos[j] = 0.0;
                b.bnnz[j] = 0;
            }
            continue;
        }
        if (d > b.cur_stride) {
            if (tid == 0) {
                set_err2(ctr, ERR_CURSOR);
                b.kept[j] = 0;
                b.chaos[j] = 0.0;
                b.bnnz[j] = 0;
            }
            continue;
        }
        const int span = hiE - lo;
        const int64_t flops_j = b.flops[j];
        int64_t est = b.est[j];
        if (est < 1) est = 1;
        for (int i = tid; i < d; i += T) {
            const int k = A.rowidx[cb + i];
            const int64_t ks = A.colptr[k];
            const float akj = A.val[cb + i];
            meta.ks[i] = ks;
            meta.len[i] = (int)(A.colptr[k + 1] - ks);
            meta.cur[i] = 0;
            meta.akj[i] = akj;
        }
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
        int ntop = 0;
        uint64_t tau = 0;
        unsigned long long s_mt = 0;
        long long s_t = 0, s_n = 0;
        FastDiv fdiv;
        fdiv.init((uint32_t)width);
        __syncthreads();
        const double S = b.bsum[j];
        FixScale fx;
        fx.init(S);

        if (bucket) {
            int* wcnt = reinterpret_cast<int*>(vals);  // nwin <= HS counters each
            int* wcur = wcnt + HS;
            // Scatter (row, a_ik * a_kj) into the window buckets from the cursors wcur;
            // with a capacity capw per window (window w owns [w capw, (w + 1) capw))
            // a run that would pass its window's end sets sh->next2[1] and writes
            // nothing past it.
            auto scatter = [&](int capw) {
                if (tid == 0) sh->next = 0;
                __syncthreads();
                for (;;) {
                    int kidx = 0;
                    if (lane == 0) kidx = atomicAdd(&sh->next, 1);
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
                                    sh->next2[1] = 1;
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
                if (tid == 0) sh->next2[1] = 0;
                __syncthreads();
                scatter(capw);
                counted = sh->next2[1] != 0;  // a window was fuller than its capacity
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
                if (tid == 0) sh->next = 0;
                __syncthreads();
                for (;;) {
                    int kidx = 0;
                    if (lane == 0) kidx = atomicAdd(&sh->next, 1);
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
            for (int i = tid; i < HS; i += T) vals[i] = 0ull;
        }

        // ---- windows ----
        // Thread 0 plans every window and publishes it; bucket mode: bucket
        // window f0 = [f0, f1) (rows [r0, r1) of it while it is split);
        // cursor mode: rows [r0, r1).
        int f0 = 0, f1 = 0;
        bool rowsplit = false;
        int split_w = 0;  // > 0: rows per piece when windows are being split
        int r0 = lo, r1 = lo;
        int cwidth = width;  // cursor mode: current window width
        int32_t* cur = meta.cur;
        int32_t* nxt = meta.nxt;
        const bool lane_mode =
            !bucket && (double)flops_j * (double)width < (double)LANE_MODE_MAX * (double)d * (double)span;
        auto plan = [&](int f) {  // thread 0 only
            while (f < nwin && wlim[f] == woff[f]) ++f;  // empty windows
            f0 = f;
            f1 = f;
            rowsplit = false;
            if (f >= nwin) return;
            if (split_w > 0) {
                const int ws = lo + f * width;
                const int we = (int)min((int64_t)ws + width, (int64_t)hiE);
                if (split_w < we - ws) {
                    rowsplit = true;
                    f1 = f + 1;
                    r0 = ws;
                    r1 = ws + split_w;
                    return;
                }
                split_w = 0;
            }
            f1 = f + 1;
        };
        auto publish = [&](int nextpar) {  // thread 0 only
            sh->pf0 = f0;
            sh->pf1 = f1;
            sh->pr0 = r0;
            sh->pr1 = r1;
            sh->prs = rowsplit ? 1 : 0;
            sh->pdone = bucket ? f0 >= nwin : r0 >= hiE;
            sh->ovf2[nextpar] = 0;
            sh->went2[nextpar] = 0;
            sh->next2[nextpar] = 0;
        };
        if (tid == 0) {
            if (bucket)
                plan(0);
            else
                r1 = (int)min((int64_t)lo + cwidth, (int64_t)hiE);
            publish(0);
        }
        for (int it = 0;; ++it) {
            const int par = it & 1;
            __syncthreads();  // this window's plan and flags are published
            if (sh->pdone) break;
            const int F0 = sh->pf0, R0 = sh->pr0, R1 = sh->pr1;
            const bool RS = sh->prs != 0;
            int* ovfp = &sh->ovf2[par];
            // rows of this window: a bucket window (or its split piece) or the cursor range;
            // at most HS rows wide, it maps row - wr0 to its slot (no hashing)
            const int wr0 = bucket ? (RS ? R0 : lo + F0 * width) : R0;
            const int wr1 =
                bucket ? (RS ? R1 : (int)min((int64_t)lo + (int64_t)(F0 + 1) * width, (int64_t)hiE))
                       : R1;
            const bool ident = wr1 - wr0 <= HS;
            auto add = [&](int row, unsigned long long q) {
                if (ident)
                    acc_add<HS, true>(row, q, wr0, keys, vals, ovfp);
                else
                    acc_add<HS, false>(row, q, wr0, keys, vals, ovfp);
            };
            // ---- 1. insert the products of the window ----
            if (bucket) {
                const int bs = woff[F0], be = wlim[F0];
                // four products per lane in flight while the previous four update
                // the table (the loads are issued before the shared atomics)
                int2 cx[4];
                int pb = bs + warp * 128;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int p = pb + 32 * u + lane;
                    cx[u] = p < be ? bkt[p] : make_int2(-1, 0);
                }
                for (; pb < be; pb += T * 4) {
                    int2 nx[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int p = pb + T * 4 + 32 * u + lane;
                        nx[u] = p < be ? bkt[p] : make_int2(-1, 0);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int row = cx[u].x;
                        bool valid = row >= 0;
                        if (RS) valid = valid && row >= R0 && row < R1;
                        if (valid) add(row, fx.qv(__int_as_float(cx[u].y)));
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) cx[u] = nx[u];
                }
            } else if (lane_mode) {
                for (int kidx = tid; kidx < d; kidx += T) {
                    const int64_t ks = meta.ks[kidx];
                    const int32_t* rows = A.rowidx + ks;
                    const float* vv = A.val + ks;
                    const float akj = meta.akj[kidx];
                    const int len = meta.len[kidx];
                    int pos = cur[kidx];
                    for (; pos < len; ++pos) {
                        const int row = __ldg(rows + pos);
                        if (row >= R1) break;
                        add(row, fx.q(__ldg(vv + pos), akj));
                    }
                    nxt[kidx] = pos;
                }
            } else {
                for (;;) {
                    int kidx = 0;
                    if (lane == 0) kidx = atomicAdd(&sh->next2[par], 1);
                    kidx = __shfl_sync(FULL, kidx, 0);
                    if (kidx >= d) break;
                    const int64_t ks = meta.ks[kidx];
                    const int32_t* rows = A.rowidx + ks;
                    const float* vv = A.val + ks;
                    const float akj = meta.akj[kidx];
                    const int len = meta.len[kidx];
                    int pos = cur[kidx];
                    while (pos < len) {
                        const int p = pos + lane;
                        const int row = p < len ? __ldg(rows + p) : INT_MAX;
                        const bool valid = row < R1;
                        if (valid) add(row, fx.q(__ldg(vv + p), akj));
                        const int nin = __popc(__ballot_sync(FULL, valid));
                        pos += nin;
                        if (nin < 32) break;
                    }
                    if (lane == 0) nxt[kidx] = pos;
                }
            }
            __syncthreads();
            if (*ovfp) {
                for (int i = tid; i < HS; i += T) {
                    keys[i] = KEY_EMPTY;
                    vals[i] = 0ull;
                }
                if (*ovfp == 2 && tid == 0) set_err2(ctr, ERR_INTERNAL);  // cannot happen
                if (tid == 0) {
                    atomicAdd(&ctr->splits, 1ull);
                    if (bucket && !rowsplit) {
                        // split the window's rows (a single row never overflows)
                        rowsplit = true;
                        r0 = lo + f0 * width;
                        const int we = (int)min((int64_t)r0 + width, (int64_t)hiE);
                        r1 = r0 + (we - r0) / 2;
                    } else {
                        r1 = r0 + (r1 - r0) / 2;
                        cwidth = r1 - r0;
                    }
                    publish(par ^ 1);
                }
                continue;
            }
            // ---- 2. statistics and candidates: every entry becomes its ranking key
            // in place (exact statistics from the fixed-point sums), row keys cleared ----
            KeyEnum<T, HS> en{vkeys};
            int c = 0, cnt = 0;
            for (int h = tid; h < HS; h += T) {
                const int row = keys[h];
                if (row != KEY_EMPTY) {
                    const unsigned long long q = vals[h];
                    const float v = fx.value(q);
                    const uint64_t key = make_key(v, row);
                    ++cnt;
                    if (v >= theta) {
                        ++s_t;
                        s_mt += q;
                    }
                    c += key > tau;
                    vkeys[h] = key;
                    keys[h] = KEY_EMPTY;
                }
            }
            s_n += cnt;
            {
                const int wc = warp_sum(cnt);
                if (lane == 0 && wc) atomicAdd(&sh->went2[par], wc);
            }
            append_candidates<T, IPT>(en, top, topcap, ksel, ntop, tau, c, hist, sh);
            // ---- 3. clear the table ----
            for (int i = tid; i < HS; i += T) vkeys[i] = 0ull;
            if (!bucket) {  // cursors advance past the window
                int32_t* t = cur;
                cur = nxt;
                nxt = t;
            }
            // ---- 4. next window ----
            if (tid == 0) {
                const int went = sh->went2[par];  // complete: append_candidates ends with a barrier
                if (bucket) {
                    if (rowsplit) {
                        const int we =
                            (int)min((int64_t)lo + (int64_t)(f0 + 1) * width, (int64_t)hiE);
                        int wd = r1 - r0;
                        if (went < PLAN / 2 && wd < width) wd *= 2;
                        r0 = r1;
                        if (r0 >= we) {
                            split_w = wd;
                            plan(f0 + 1);
                        } else {
                            r1 = min(we, r0 + wd);
                        }
                    } else {
                        plan(f1);
                    }
                } else {
                    r0 = r1;
                    if (went < PLAN / 2 && cwidth < (1 << 29))
                        cwidth *= 2;
                    else if (went > PLAN + PLAN / 2 && cwidth > 1)
                        cwidth /= 2;
                    r1 = (int)min((int64_t)r0 + cwidth, (int64_t)hiE);
                }
                publish(par ^ 1);
            }
        }
        double dv[1] = {0.0};
        long long qv[3] = {s_t, s_n, (long long)s_mt};
        block_sum<T>(dv, 0, qv, 3, &sh->bs);
        const double MT = ldexp((double)(unsigned long long)qv[2], -fx.f);
        int mstar = 0;
        double ch = 0.0;
        const int64_t obase = b.off[j];
        // the table's key array is free here: radix counters of the row sort
        finish_column<T, IPT, false>(top, ntop, topcap, a.pp, S, MT, qv[0], b.cap[j],
                                     b.tmp_row + (obase - b.tmp_off0),
                                     b.tmp_val + (obase - b.tmp_off0), hist, mhist, sh, ctr, lo,
                                     span, reinterpret_cast<unsigned*>(keys), &mstar, &ch);
        for (int i = tid; i < (T / 32) * 256; i += T) keys[i] = KEY_EMPTY;
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
    auto kern = k_expand<C::T, C::HS, C::MINB>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, C::T, smem);
    if (occ < 1) occ = 1;
    return occ * num_sms;
}

template <class C>
static void conf_launch(int conf, const CscView& A, const PruneParams& pp, const ExpandBuffers& b,
                        int grid, cudaStream_t s) {
    int plan = conf == 0 ? C::HS / 2 : (pp.plan > 0 ? pp.plan : C::HS / 2);
    if (plan > (3 * C::HS) / 4) plan = (3 * C::HS) / 4;
    if (plan < 64) plan = 64;
    ExpandArgs a{A, pp, b, conf, plan};
    k_expand<C::T, C::HS, C::MINB><<<grid, C::T, conf_smem<C>(pp.ksel), s>>>(a);
}

int numeric_grid(int conf, const PruneParams& pp, int num_sms) {
    if (conf == CONF_DIRECT) return direct_grid(pp.ksel, num_sms);
    if (conf == 0) return conf_grid<Conf0>(pp.ksel, num_sms);
    return pp.table == 1 ? conf_grid<Conf1b>(pp.ksel, num_sms)
                         : pp.table == 2 ? conf_grid<Conf1c>(pp.ksel, num_sms)
                                         : conf_grid<Conf1a>(pp.ksel, num_sms);
}

void launch_numeric(int conf, const CscView& A, const PruneParams& pp, const ExpandBuffers& b,
                    int grid, cudaStream_t s) {
    if (conf == CONF_DIRECT)
        launch_direct(A, pp, b, grid, s);
    else if (conf == 0)
        conf_launch<Conf0>(conf, A, pp, b, grid, s);
    else if (pp.table == 1)
        conf_launch<Conf1b>(conf, A, pp, b, grid, s);
    else if (pp.table == 2)
        conf_launch<Conf1c>(conf, A, pp, b, grid, s);
    else
        conf_launch<Conf1a>(conf, A, pp, b, grid, s);
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
};

// The candidates and statistics of one column of m entries, in row order.
// load(i, &row, &q) gives entry i with its fixed-point value; a chunk of 2,048
// entries is read once, coalesced, and kept in registers while the positions
// of its candidates are counted (ballots per round and warp, in entry order).
template <class Load>
__device__ __forceinline__ void prune_candidates(int64_t m, const FixScale& fx, float theta, Load load,
                                                 uint64_t* top, int topcap, int ksel, unsigned* hist,
                                                 PruneShared* ps, int& ntop, long long& s_t,
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
            tau = block_select_count<PR_T>(top, ntop, top, 0, ksel, hist, &ps->w.bs);
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
            top, topcap, ksel, hist, ps, ntop, s_t, s_mt);
        double dv[1] = {0.0};
        long long qv[2] = {s_t, (long long)s_mt};
        block_sum<PR_T>(dv, 0, qv, 2, &sh->bs);
        const double MT = ldexp((double)(unsigned long long)qv[1], -fx.f);
        int mstar = 0;
        double ch = 0.0;
        const int64_t obase = b.off[j];
        finish_column<PR_T, 8, true>(top, ntop, topcap, a.pp, S, MT, qv[0], b.cap[j],
                                     b.tmp_row + (obase - b.tmp_off0),
                                     b.tmp_val + (obase - b.tmp_off0), hist, mhist, sh, b.ctr, 0,
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

