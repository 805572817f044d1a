// The numeric pass for columns that are dense in their row span: windows of
// consecutive rows with a 64-bit sum per row in shared memory, no hashing.
//
// Two CTAs share an SM, each with a table of 10,240 rows, so that one's scans
// and selects overlap the other's inserts (one CTA with 24,576 rows: the same
// on 40k-row columns, 5-30% slower on shorter or sparser ones, whose time goes
// into the phases between barriers).  The candidate buffer grows with K: above
// about 1,200 one CTA fits an SM (iteration 2 of a 30k-vertex power-law graph
// with K = 1,100, 1,500 and 4,096: 28.9, 40.1 and 41.5 ms; 72.7, 82.9 and 112 ms
// with hashed windows).
//
//   insert:  the products of the window's rows, from per-source cursors over
//            the sorted rows of A (one or more windows: a source is visited
//            once per window), or, where a source has few products per window,
//            from per-window product buckets.  A product is two 32-bit shared
//            atomics and about 20 instructions: four per lane and round, no
//            branches, the next round's loads issued first;
//   extract: one scan of the table, which clears it.  Almost every sum is
//            below both the threshold and the running top-k bound and is only
//            counted, by a comparison of integers.  Candidates go to a shared
//            buffer, and beyond its end to a per-CTA spill in global memory;
//            past that end the buffer is cut back to the ksel largest once per
//            window.
//
// The sums are those of mcl_numeric.cu (exact fixed point), as are the
// candidate keys and the end of a column, so a column's result does not
// depend on the kernel that takes it.  A sum can be zero although its row has
// products (they were 0 or truncated to 0): such products mark their row in a
// bitmap, so that the entry still counts.
//
// Bound by the instructions of the insert (78% of issue slots when it took
// about 95 per product; 8% of DRAM peak).  Iteration 2 of the 40k-vertex
// power-law graph (4.4e10 products): 240 ms with the hashed windows that
// mcl_numeric.cu then had, 95 ms here; iteration 2 of 16 planted partitions of
// up to 50k vertices (4.8e10): 401 ms and 121 ms.
#include <cfloat>
#include <climits>
#include <cstdint>
#include <type_traits>

#include "mcl_column.cuh"
#include "mcl_device.cuh"
#include "mcl_internal.h"

namespace mcl {

constexpr int DIR_T = 512;        // threads of the CTA
constexpr int DIR_MINB = 2;       // CTAs per SM
constexpr int DIR_W = 10240;      // rows of a window
constexpr int DIR_HEAD = 2048;    // candidates beyond ksel that the buffer holds
constexpr int DIR_LONG = 64;      // sources shared by all warps
// Below this many products per source and window, the products go through
// window buckets: a visit costs a warp a round of 128 products whatever it
// finds (200k-vertex graph, columns of 200k-800k products: 1.32M-3.73M clocks
// per CTA with cursors at 41 products per visit, 1.03M-2.61M with buckets).
constexpr int DIR_BUCKET_MAX = 128;
// The sums' low and high words are two arrays (all banks serve each), each
// followed by 32 words that idle lanes add 0 to.
constexpr int DIR_HI = DIR_W + 32;

struct __align__(16) DirShared {
    WinShared w;
    int cand;      // candidates of the window
    int zany;      // some product of the window was zero
    int nlong;
    int next[2];   // source counters, by window parity
    int full;      // a bucket was fuller than its capacity
    int longs[DIR_LONG];
    unsigned zbm[DIR_W / 32];  // rows of zero products
};

struct DirectArgs {
    CscView A;
    PruneParams pp;
    ExpandBuffers b;
    uint64_t* spill;  // per CTA: DIR_W candidates that the buffer had no room for
};

static size_t direct_smem(int ksel) {
    return (size_t)2 * DIR_HI * 4 + sizeof(DirShared) + 256 * 4 + 256 * 8 + (size_t)(ksel + DIR_HEAD) * 8;
}

__device__ __forceinline__ unsigned atom_add_shared(unsigned addr, unsigned v) {
    unsigned old;
    asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(addr), "r"(v) : "memory");
    return old;
}

// hi word at addr + DIR_HI words: += qh + carry(old + ql)
__device__ __forceinline__ void red_high(unsigned addr, unsigned old, unsigned ql, unsigned qh) {
    asm volatile("{ .reg .u32 t, h;\n\tadd.cc.u32 t, %1, %2;\n\taddc.u32 h, %3, 0;\n\t"
                 "red.shared.add.u32 [%0 + %4], h; }" ::"r"(addr), "r"(old), "r"(ql), "r"(qh),
                 "n"(DIR_HI * 4)
                 : "memory");
}

__global__ void __launch_bounds__(DIR_T, DIR_MINB) k_expand_direct(DirectArgs a) {
    constexpr int T = DIR_T, NW = T / 32, IPT = 4;
    extern __shared__ __align__(16) unsigned char smem[];
    const int ksel = a.pp.ksel;
    const int topcap = ksel + DIR_HEAD;
    unsigned* lo32 = reinterpret_cast<unsigned*>(smem);
    unsigned* hi32 = lo32 + DIR_HI;
    DirShared* ds = reinterpret_cast<DirShared*>(hi32 + DIR_HI);
    unsigned long long* mhist = reinterpret_cast<unsigned long long*>(ds + 1);
    unsigned* hist = reinterpret_cast<unsigned*>(mhist + 256);
    uint64_t* top = reinterpret_cast<uint64_t*>(hist + 256);
    unsigned* zbm = ds->zbm;
    WinShared* sh = &ds->w;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const CscView& A = a.A;
    const ExpandBuffers& b = a.b;
    DevCounters* ctr = b.ctr;
    if (ctr->err & ERR_STAGING) return;  // the iteration is redone without the graph
    SrcMeta meta(b.cursors + (int64_t)blockIdx.x * 6 * b.cur_stride, b.cur_stride);
    int2* bkt = b.bucket_row ? reinterpret_cast<int2*>(b.bucket_row) + (int64_t)blockIdx.x * b.bucket_cap
                             : nullptr;
    int32_t* woff = b.woff ? b.woff + (int64_t)blockIdx.x * 2 * (WINDOW_MAX + 1) : nullptr;
    int32_t* wlim = woff ? woff + (WINDOW_MAX + 1) : nullptr;
    const int wbeg = ctr->bin_off[CONF_DIRECT * NZ], wend = ctr->bin_off[CONF_DIRECT * NZ + NZ];
    uint64_t* spill = a.spill + (int64_t)blockIdx.x * DIR_W;
    const unsigned table = (unsigned)__cvta_generic_to_shared(lo32);
    for (int i = tid; i < 2 * DIR_HI; i += T) lo32[i] = 0u;
    for (int i = tid; i < DIR_W / 32; i += T) zbm[i] = 0u;
    const float theta = a.pp.theta;
    for (;;) {
        if (tid == 0) {
            sh->item = atomicAdd(&ctr->conf_ctr[CONF_DIRECT], 1);
            ds->nlong = 0;
            ds->next[0] = 0;
            ds->zany = 0;
            ds->cand = 0;
        }
        __syncthreads();
        const int item = sh->item;
        if (wbeg + item >= wend) break;
        const int j = b.work[wbeg + item];
        const int64_t cb = A.colptr[j];
        const int d = (int)(A.colptr[j + 1] - cb);
        const int lo = b.rlo[j], hiE = b.rhi[j] + 1;
        const int span = hiE - lo;
        if (d > b.cur_stride || d < 1 || span < 1) {  // cannot happen: the columns binned here
            if (tid == 0) {
                atomicOr(&ctr->err, ERR_CURSOR);
                b.kept[j] = 0;
                b.chaos[j] = 0.0;
                b.bnnz[j] = 0;
            }
            __syncthreads();
            continue;
        }
        const int64_t flops_j = b.flops[j];
        const double S = b.bsum[j];
        FixScale fx;
        fx.init(S);
        // ---- windows of equal row width ----
        int nwin = (int)(((int64_t)span + DIR_W - 1) / DIR_W);
        const int width = (int)(((int64_t)span + nwin - 1) / nwin);
        nwin = (int)(((int64_t)span + width - 1) / width);
        const bool bucket = nwin > 1 && bkt != nullptr && flops_j <= b.bucket_cap && nwin <= WINDOW_MAX &&
                            flops_j < (int64_t)DIR_BUCKET_MAX * d * nwin;
        for (int i = tid; i < d; i += T) {
            const int k = A.rowidx[cb + i];
            const int64_t ks = A.colptr[k];
            const int len = (int)(A.colptr[k + 1] - ks);
            meta.ks[i] = ks;
            meta.len[i] = len;
            meta.cur[i] = 0;
            meta.akj[i] = A.val[cb + i];
            if (nwin == 1 && len >= T) {  // every warp takes a share of a long source
                const int l = atomicAdd(&ds->nlong, 1);
                if (l < DIR_LONG) {
                    ds->longs[l] = i;
                    meta.cur[i] = -1;
                }
            }
        }
        __syncthreads();

        const bool plain = fx.plain();
        // a product below it may be 0
        const float vmin = plain ? ldexpf(1.0f, -fx.f) : FLT_MAX;
        const unsigned idle = table + (DIR_W + lane) * 4;
        // Four products per lane into their rows' sums, without branches: the low words'
        // atomics are issued together, then the high words' with their carries.  whole: every
        // lane has four products of the window (h < wr); else lanes without one add 0 to a
        // word of their own beside the table.
        auto add4 = [&](const unsigned (&h)[4], const float (&v)[4], unsigned wr, auto whole) {
            unsigned at[4], ql[4], qh[4], old[4];
            bool zero = false;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const unsigned long long q = plain ? fx.qplain(v[c]) : fx.qv(v[c]);
                at[c] = table + h[c] * 4;
                ql[c] = (unsigned)q;
                qh[c] = (unsigned)(q >> 32);
                if (decltype(whole)::value) {
                    zero |= v[c] < vmin;
                } else {
                    const bool in = h[c] < wr;
                    zero |= in && v[c] < vmin;
                    at[c] = in ? at[c] : idle;
                    ql[c] = in ? ql[c] : 0u;
                    qh[c] = in ? qh[c] : 0u;
                }
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) old[c] = atom_add_shared(at[c], ql[c]);
#pragma unroll
            for (int c = 0; c < 4; ++c) red_high(at[c], old[c], ql[c], qh[c]);
            if (zero) {  // rare: the exact test
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (h[c] < wr && fx.qv(v[c]) == 0ull) {
                        atomicOr(zbm + (h[c] >> 5), 1u << (h[c] & 31));
                        ds->zany = 1;
                    }
            }
        };

        if (bucket) {
            int* wcnt = reinterpret_cast<int*>(lo32);  // nwin <= WINDOW_MAX counters each
            int* wcur = reinterpret_cast<int*>(hi32);
            FastDiv fdiv;
            fdiv.init((uint32_t)width);
            // (row, a_ik a_kj) into the buckets from the cursors wcur; with a capacity capw per
            // window a run that would pass its window's end sets ds->full and writes nothing past it.
            // capw < 0 only counts.
            auto scatter = [&](int capw, int* next) {
                for (;;) {
                    int kidx = 0;
                    if (lane == 0) kidx = atomicAdd(next, 1);
                    kidx = __shfl_sync(FULL, kidx, 0);
                    if (kidx >= d) break;
                    const int len = meta.len[kidx];
                    const int64_t ks = meta.ks[kidx];
                    const int32_t* rows = A.rowidx + ks;
                    const float* vv = A.val + ks;
                    const float akj = meta.akj[kidx];
                    int rr[4];
                    float pv[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int p = 32 * c + lane;
                        rr[c] = p < len ? __ldg(rows + p) : 0;
                        pv[c] = p < len && capw >= 0 ? __ldg(vv + p) : 0.0f;
                    }
                    for (int pb = 0; pb < len; pb += 128) {
                        int nr[4];
                        float nv[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const int p = pb + 128 + 32 * c + lane;
                            nr[c] = p < len ? __ldg(rows + p) : 0;
                            nv[c] = p < len && capw >= 0 ? __ldg(vv + p) : 0.0f;
                        }
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            // rows are sorted: equal windows form runs of lanes
                            const bool v = pb + 32 * c + lane < len;
                            const unsigned act = __ballot_sync(FULL, v);
                            if (act == 0u) break;
                            const uint32_t w = v ? fdiv.div((uint32_t)(rr[c] - lo)) : 0xFFFFFFFFu;
                            const uint32_t wp = __shfl_up_sync(FULL, w, 1);
                            const bool head = v && (lane == 0 || wp != w);
                            const unsigned heads = __ballot_sync(FULL, head);
                            int base = 0;
                            if (head) {
                                const unsigned after = heads & ~((2u << lane) - 1u);
                                const int end = after ? __ffs(after) - 1 : __popc(act);
                                base = atomicAdd(wcur + w, end - lane);
                                if (capw > 0 && base + (end - lane) > ((int)w + 1) * capw) ds->full = 1;
                            }
                            if (capw < 0) continue;
                            const int hl = 31 - __clz(heads & ((2u << lane) - 1u));
                            base = __shfl_sync(FULL, base, hl);
                            if (v) {
                                const int pos = base + lane - hl;
                                if (capw == 0 || pos < ((int)w + 1) * capw)
                                    bkt[pos] = make_int2(rr[c], __float_as_int(pv[c] * akj));
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
            // twice the mean share of the products per window first; only a column where some
            // window is fuller counts and scatters again
            const int64_t capw64 = ((flops_j + nwin - 1) / nwin) * 2 + 64;
            bool counted = true;
            if (capw64 * nwin <= b.bucket_cap) {
                const int capw = (int)capw64;
                for (int i = tid; i < nwin; i += T) wcur[i] = i * capw;
                if (tid == 0) {
                    ds->full = 0;
                    ds->next[1] = 0;
                }
                __syncthreads();
                scatter(capw, &ds->next[0]);
                counted = ds->full != 0;
                if (!counted)
                    for (int i = tid; i < nwin; i += T) {
                        woff[i] = i * capw;
                        wlim[i] = wcur[i];
                    }
                __syncthreads();
            }
            if (counted) {
                for (int i = tid; i < nwin; i += T) wcur[i] = 0;
                if (tid == 0) {
                    ds->next[0] = 0;
                    ds->next[1] = 0;
                }
                __syncthreads();
                scatter(-1, &ds->next[0]);
                for (int i = tid; i < nwin; i += T) wcnt[i] = wcur[i];
                __syncthreads();
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
                if (tid == 0 && (int64_t)tot != flops_j) atomicOr(&ctr->err, ERR_INTERNAL);
                __syncthreads();
                scatter(0, &ds->next[1]);
            }
            for (int i = tid; i < nwin; i += T) {
                wcnt[i] = 0;
                wcur[i] = 0;
            }
            __syncthreads();
        }

        // ---- windows ----
        int ntop = 0;
        uint64_t tau = 0;
        unsigned long long qmin = 0;  // sums below it are neither candidates nor >= theta
        unsigned long long s_mt = 0;
        long long s_t = 0;
        unsigned s_n = 0;
        int32_t* cur = meta.cur;
        int32_t* nxt = meta.nxt;
        const int batch = max(1, min(32, d / (4 * NW)));  // sources a warp takes at once
        for (int w = 0; w < nwin; ++w) {
            const int r0 = lo + w * width;
            const int r1 = (int)min((int64_t)r0 + width, (int64_t)hiE);
            const unsigned wr = (unsigned)(r1 - r0);
            if (tid == 0) ds->next[(w + 1) & 1] = 0;
            // ---- insert ----
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
                    const bool whole = pb + 128 <= be;
                    pb += T * 4;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int p = pb + 32 * u + lane;
                        cx[u] = p < be ? bkt[p] : make_int2(INT_MAX, 0);
                    }
                    if (whole)
                        add4(h, v, wr, std::true_type{});
                    else
                        add4(h, v, wr, std::false_type{});
                }
            } else {
                if (nwin == 1) {
                    const int nl = min(ds->nlong, DIR_LONG);
                    for (int l = 0; l < nl; ++l) {
                        const int kidx = ds->longs[l];
                        const int len = meta.len[kidx];
                        const int32_t* rows = A.rowidx + meta.ks[kidx];
                        const float* vv = A.val + meta.ks[kidx];
                        const float akj = meta.akj[kidx];
                        for (int pb = warp * 128; pb < len; pb += T * 4) {
                            unsigned h[4];
                            float v[4];
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const int p = pb + 32 * c + lane;
                                h[c] = p < len ? (unsigned)(__ldg(rows + p) - r0) : 0xFFFFFFFFu;
                                v[c] = p < len ? __ldg(vv + p) : 0.0f;
                            }
#pragma unroll
                            for (int c = 0; c < 4; ++c) v[c] = __fmul_rn(v[c], akj);
                            add4(h, v, wr, std::false_type{});
                        }
                    }
                }
                int* next = &ds->next[w & 1];
                for (;;) {
                    int k0 = 0;
                    if (lane == 0) k0 = atomicAdd(next, batch);
                    k0 = __shfl_sync(FULL, k0, 0);
                    if (k0 >= d) break;
                    const int nb = min(batch, d - k0);
                    // lane l holds source k0 + l of the batch
                    int64_t mks = 0;
                    int mlen = 0, mcur = -1;
                    float makj = 0.0f;
                    if (lane < nb) {
                        mcur = cur[k0 + lane];
                        mks = meta.ks[k0 + lane];
                        mlen = meta.len[k0 + lane];
                        makj = meta.akj[k0 + lane];
                    }
                    unsigned left = __ballot_sync(FULL, mcur >= 0 && mcur < mlen);
                    int mnxt = mcur;
                    if (left != 0u) {
                        // this lane's next entry of the current source, and the entries from it on
                        const int32_t* prow;
                        const float* pval;
                        int rem, s;
                        float akj;
                        int rr[4];
                        float pv[4];
                        auto source = [&]() {
                            s = __ffs(left) - 1;
                            const int pos = __shfl_sync(FULL, mcur, s) + lane;
                            const int64_t at = __shfl_sync(FULL, mks, s) + pos;
                            rem = __shfl_sync(FULL, mlen, s) - pos;
                            akj = __shfl_sync(FULL, makj, s);
                            prow = A.rowidx + at;
                            pval = A.val + at;
                        };
                        auto load = [&]() {
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                rr[c] = 32 * c < rem ? __ldg(prow + 32 * c) : INT_MAX;
                                pv[c] = 32 * c < rem ? __ldg(pval + 32 * c) : 0.0f;
                            }
                        };
                        source();
                        load();
                        for (bool more = true; more;) {
                            unsigned h[4];
                            float v[4];
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                h[c] = (unsigned)(rr[c] - r0);
                                v[c] = __fmul_rn(pv[c], akj);
                            }
                            const bool whole = __all_sync(FULL, h[3] < wr);  // rows are sorted
                            if (whole) {
                                prow += 128;
                                pval += 128;
                                rem -= 128;
                            }
                            const int rem0 = __shfl_sync(FULL, rem, 0);
                            if (!whole || rem0 <= 0) {  // the source has no more in this window
                                int nin = 0;
                                if (!whole)
#pragma unroll
                                    for (int c = 0; c < 4; ++c)
                                        nin += __popc(__ballot_sync(FULL, h[c] < wr));
                                // lane 0's position: length - rem0, and the entries taken now
                                if (lane == s) mnxt = mlen - rem0 + nin;
                                left &= left - 1u;
                                more = left != 0u;
                                if (more) source();
                            }
                            if (more) load();  // the next chunk, while this one is added
                            if (whole)
                                add4(h, v, wr, std::true_type{});
                            else
                                add4(h, v, wr, std::false_type{});
                        }
                    }
                    if (nwin > 1 && lane < nb) nxt[k0 + lane] = mnxt;
                }
            }
            __syncthreads();
            // ---- extract: one scan of the table, which it clears ----
            const bool zany = ds->zany != 0;
            for (unsigned h = tid * 4; h < (wr + 127 & ~127u); h += T * 4) {  // four rows; whole warps
                uint4* pl = reinterpret_cast<uint4*>(lo32 + h);
                uint4* ph = reinterpret_cast<uint4*>(hi32 + h);
                const uint4 l4 = *pl, h4 = *ph;
                const unsigned xl[4] = {l4.x, l4.y, l4.z, l4.w}, xh[4] = {h4.x, h4.y, h4.z, h4.w};
                const unsigned zb = zany ? (zbm[h >> 5] >> (h & 31)) & 15u : 0u;
                unsigned big = 0;  // rows to look at
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const unsigned long long q = ((unsigned long long)xh[u] << 32) | xl[u];
                    const bool here = q != 0ull || ((zb >> u) & 1u);
                    s_n += here;
                    big |= here && q >= qmin ? 1u << u : 0u;
                }
                while (__any_sync(FULL, big != 0u)) {  // one row per lane and round: few have any
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
                        key = make_key(v, r0 + (int)g);
                    }
                    // candidates to the buffer, in any order; those it has no room for to the spill
                    const bool take = key > tau;
                    const unsigned m = __ballot_sync(FULL, take);
                    if (m) {
                        int base = 0;
                        if (lane == 0) base = atomicAdd(&ds->cand, __popc(m));
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
            }
            __syncthreads();
            const int have = ntop + ds->cand;
            __syncthreads();
            if (tid == 0) {
                ds->cand = 0;
                ds->zany = 0;
            }
            if (have > topcap) {  // cut back to the ksel largest
                const int over = have - topcap;
                tau = block_select_wide<T>(top, topcap, spill, over, ksel, lo32, &sh->bs, sh->wsm);
                ntop = compact_stable<T, IPT>(top, topcap, tau, sh->wsm);
                for (int i = tid; i < over; i += T) {
                    const uint64_t x = spill[i];
                    if (x >= tau) top[ntop + atomicAdd(&ds->cand, 1)] = x;
                }
                __syncthreads();
                ntop = ksel;
                if (tid == 0) ds->cand = 0;
                qmin = fx.lower(fminf(theta, key_val(tau)));
            } else {
                ntop = have;
            }
            if (zany)
                for (unsigned i = tid; i < (wr + 31) / 32; i += T) zbm[i] = 0u;
            __syncthreads();
            int32_t* t = cur;
            cur = nxt;
            nxt = t;
        }
        double dv[1] = {0.0};
        long long qv[3] = {s_t, (long long)s_n, (long long)s_mt};
        block_sum<T>(dv, 0, qv, 3, &sh->bs);
        int mstar = 0;
        double ch = 0.0;
        const int64_t obase = b.off[j];
        // the table is free (and zero) here: radix counters of the row sort
        finish_column<T, IPT, false>(top, ntop, topcap, a.pp, S, (unsigned long long)qv[2], fx.f, qv[0], b.cap[j],
                                     b.tmp_row + (obase - b.tmp_off0), b.tmp_val + (obase - b.tmp_off0),
                                     hist, mhist, hi32, sh, ctr, lo, span, lo32, &mstar, &ch);
        for (int i = tid; i < NW * 256; i += T) lo32[i] = 0u;
        if (tid == 0) {
            b.kept[j] = mstar;
            b.chaos[j] = ch;
            b.bnnz[j] = qv[1];
            if (qv[1] > b.est[j]) atomicAdd(&ctr->misses, 1ull);
        }
    }
}

int direct_grid(int ksel, int num_sms) {
    const size_t smem = direct_smem(ksel);
    cudaFuncSetAttribute(k_expand_direct, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_expand_direct, DIR_T, smem);
    return (occ < 1 ? 1 : occ) * num_sms;
}

size_t direct_spill_bytes(int grid) { return (size_t)grid * DIR_W * 8; }

void launch_direct(const CscView& A, const PruneParams& pp, const ExpandBuffers& b, int grid,
                   cudaStream_t s) {
    k_expand_direct<<<grid, DIR_T, direct_smem(pp.ksel), s>>>(DirectArgs{A, pp, b, b.spill});
}

}  // namespace mcl
