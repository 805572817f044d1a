// The expansion with its inner dimension split into stages, and the binary
// merge of the stages' partial products (Section IV, "Binary merge";
// Algorithm 2).
//
// B = A A = sum_t P_t, where stage t multiplies the columns of A by the rows
// k of A in block t of the inner index: P_t(:, j) = sum over k in block t of
// a_kj A(:, k).  A partial product is unpruned, its columns sorted by row,
// and its entries are the exact 64-bit fixed-point sums the numeric pass
// uses (every column's scale comes from the same column sum s_j =
// sum_k a_kj colsum_k(A), in the same order), so partial products add
// exactly and the merged product, pruned, equals the one-pass iteration bit
// for bit.
//
// One kernel does both jobs on row-sorted inputs: for each output column a
// CTA walks its sources (the columns of A of one stage, scaled by a_kj, or
// the columns of the partial products being merged) in windows of rows; a
// shared bitmap marks the rows present (count mode: their number) and a prefix
// count of the bitmap gives each row its position in the output column.  Fill
// mode adds the values at their positions in a shared array of 64-bit sums (or
// in the output itself, where the window has more entries than the array) and
// writes the window's entries out in order, so the output comes out sorted and
// its sums do not depend on the order of the additions.
//
// The sources are cut into units of 128 entries that the warps take in turn:
// a merge has 2 to 5 sources and a stage of a sparse column a handful, which
// would leave most warps idle with a source per warp.  20k-vertex power-law
// graph (3.8e8 products) in 8 stages: 96 ms with a source per warp and every
// product a global atomic, 17 ms with units and shared sums, 15 ms with the
// small CTAs, 11.1 ms without passes over the sources for parts of a window.
#include <climits>
#include <cstdint>

#include "mcl_device.cuh"
#include "mcl_internal.h"

namespace mcl {

// Column sums of B from the identity sum_i (AA)_ij = sum_k a_kj colsum_k(A):
// warp per column, lane l taking the column's entries l, l + 32, ..., then a
// butterfly -- the order of the numeric pass, so the same doubles.
__global__ void k_bsum(CscView A, const double* colsum, double* bsum) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t j = gw; j < A.n; j += nw) {
        const int64_t cb = A.colptr[j];
        const int d = (int)(A.colptr[j + 1] - cb);
        double s = 0.0;
        for (int i = lane; i < d; i += 32) s += (double)A.val[cb + i] * colsum[A.rowidx[cb + i]];
        s = warp_sum(s);
        if (lane == 0) bsum[j] = s;
    }
}

void launch_bsum(const CscView& A, const double* colsum, double* bsum, cudaStream_t s) {
    if (A.n == 0) return;
    int64_t blocks = ((int64_t)A.n * 32 + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    k_bsum<<<(unsigned)blocks, 256, 0, s>>>(A, colsum, bsum);
    count_launches(1);
}

constexpr int RA_UNIT = 128;   // entries a warp takes at once
// Shapes by the rows of the output: threads, bitmap words (32 rows each), sums,
// CTAs per SM.  A column's steps are short and separated by barriers, so small
// outputs take many small CTAs (16.4 -> 15.2 ms against RankSmall at 20k rows);
// a wider bitmap leaves room for fewer.  With a source per warp and every product
// a global atomic, power-law graphs in 4 stages: 60k rows 170 ms (RankSmall: 26.9),
// 400k rows 1,793 ms (RankLarge: 401).
template <int T_, int WORDS_, int CAP_, int MINB_>
struct RankShape {
    static constexpr int T = T_, WORDS = WORDS_, CAP = CAP_, MINB = MINB_;
};
using RankTiny = RankShape<256, 1024, 4096, 5>;
using RankSmall = RankShape<512, 4096, 8192, 2>;
using RankLarge = RankShape<512, 16384, 8192, 1>;
// A window with more entries than the array of sums holds adds in global memory
// (the L2).  Walking its sources again for every arrayful was no better anywhere:
// 100k vertices of 400 entries, 2 stages: 557 ms with up to eight passes, 390 with
// two, 389 with one; 12k of 130, 4 stages: 6.6 and 5.9 ms; 140k of 100: 120 and 116.

template <int T>
struct RankShared {
    BlockScratch bs;
    int wsm[34];
    int item;
    int lo, hi;               // row span of the column's sources
    int upre[T + 1];          // first unit of each source of a batch of T
};

// Sources of one output column, per CTA in global scratch (stride entries):
// row arrays, value arrays (FP32 of A or uint64 sums), lengths, a_kj and
// the cursors of the window walk.
struct RankScratch {
    const int32_t** rows;
    const void** vals;
    int32_t* len;
    float* akj;
    int32_t* cur;
    int32_t* nxt;
};

// Exclusive block scan of x; the total to all threads.  Ends with a barrier.
template <int T>
__device__ __forceinline__ int ra_scan(int x, int* total, int* wsm) {
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
        const int w0 = lane < T / 32 ? wsm[lane] : 0;
        int wi = w0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < T / 32) wsm[lane] = wi - w0;
        if (lane == 31) wsm[32] = wi;
    }
    __syncthreads();
    const int res = wsm[warp] + incl - x;
    *total = wsm[32];
    __syncthreads();
    return res;
}

// STAGE: sources are the columns k of A in [k0, k1) referenced by column j;
// otherwise the columns j of the partial products.  FILL: write the output
// (else count it).
template <bool STAGE, bool FILL, class SH>
__global__ void __launch_bounds__(SH::T, SH::MINB) k_rank_acc(RankArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int RA_T = SH::T;
    constexpr int WORDS = SH::WORDS, CAP = SH::CAP, WB = WORDS * 32;
    uint32_t* bm = reinterpret_cast<uint32_t*>(smem);
    int32_t* wpre = reinterpret_cast<int32_t*>(bm + WORDS);  // from here FILL only, up to sh
    unsigned* lo32 = reinterpret_cast<unsigned*>(wpre + WORDS);
    unsigned* hi32 = lo32 + CAP;
    RankShared<RA_T>* sh = reinterpret_cast<RankShared<RA_T>*>(FILL ? reinterpret_cast<unsigned char*>(hi32 + CAP)
                                                        : reinterpret_cast<unsigned char*>(bm + WORDS));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NWP = RA_T / 32;
    unsigned long long* sb = reinterpret_cast<unsigned long long*>(a.scratch) +
                             (int64_t)blockIdx.x * 6 * a.stride;
    RankScratch rs{reinterpret_cast<const int32_t**>(sb),
                   reinterpret_cast<const void**>(sb + a.stride),
                   reinterpret_cast<int32_t*>(sb + 2 * a.stride),
                   reinterpret_cast<float*>(sb + 3 * a.stride),
                   reinterpret_cast<int32_t*>(sb + 4 * a.stride),
                   reinterpret_cast<int32_t*>(sb + 5 * a.stride)};
    if (FILL)
        for (int i = tid; i < 2 * CAP; i += RA_T) lo32[i] = 0u;
    for (;;) {
        if (tid == 0) {
            sh->item = atomicAdd(&a.ctr->work_ctr, 1);
            sh->lo = INT_MAX;
            sh->hi = -1;
        }
        __syncthreads();
        const int64_t j = sh->item;
        if (j >= a.n) break;
        // ---- the column's sources ----
        int ns = 0;
        int64_t i0 = 0;
        if (STAGE) {
            // rows are sorted: those below k0, and below k1, lead the column
            const int64_t cb = a.A.colptr[j], ce = a.A.colptr[j + 1];
            int below = 0, within = 0;
            for (int64_t base = cb; base < ce; base += RA_T) {
                const int k = base + tid < ce ? a.A.rowidx[base + tid] : INT_MAX;
                below += __syncthreads_count(k < a.k0);
                within += __syncthreads_count(k < a.k1);
            }
            ns = within - below;
            i0 = cb + below;
        } else {
            ns = a.nparts;
        }
        if (ns > a.stride) {  // cannot happen: the stride exceeds the longest column
            if (tid == 0) {
                atomicOr(&a.ctr->err, ERR_CURSOR);
                if (!FILL) a.nnz_out[j] = 0;
            }
            __syncthreads();
            continue;
        }
        int mn = INT_MAX, mx = -1;
        for (int s = tid; s < ns; s += RA_T) {
            const int32_t* rows;
            const void* vals;
            int len;
            float f = 1.0f;
            if (STAGE) {
                const int k = a.A.rowidx[i0 + s];
                const int64_t ks = a.A.colptr[k];
                rows = a.A.rowidx + ks;
                vals = a.A.val + ks;
                len = (int)(a.A.colptr[k + 1] - ks);
                f = a.A.val[i0 + s];
            } else {
                const int64_t ps = a.pcol[s][j];
                rows = a.prow[s] + ps;
                vals = a.pval[s] + ps;
                len = (int)(a.pcol[s][j + 1] - ps);
            }
            rs.rows[s] = rows;
            rs.vals[s] = vals;
            rs.len[s] = len;
            rs.akj[s] = f;
            rs.nxt[s] = 0;
            if (len > 0) {
                mn = min(mn, rows[0]);
                mx = max(mx, rows[len - 1]);
            }
        }
        if (mx >= 0) {
            atomicMin(&sh->lo, mn);
            atomicMax(&sh->hi, mx);
        }
        __syncthreads();
        const int lo = sh->lo;
        const int hiE = sh->hi + 1;
        FixScale fx;
        fx.init(STAGE ? a.bsum[j] : 1.0);
        long long cnt = 0;
        int64_t obase = FILL ? a.colptr_out[j] : 0;
        for (int r0 = lo; r0 < hiE && hiE > lo;) {
            const int r1 = (int)min((int64_t)r0 + WB, (int64_t)hiE);
            const int nwords = (r1 - r0 + 31) >> 5;
            const bool last = r1 == hiE;
            for (int i = tid; i < nwords; i += RA_T) bm[i] = 0u;
            // each source's entries of the window: [cur, nxt)
            for (int s = tid; s < ns; s += RA_T) {
                const int c0 = rs.nxt[s], len = rs.len[s];
                int x = len;
                if (!last) {
                    int h = len;  // first entry at or beyond r1
                    x = c0;
                    const int32_t* rows = rs.rows[s];
                    while (x < h) {
                        const int m = (x + h) >> 1;
                        if (rows[m] < r1) x = m + 1; else h = m;
                    }
                }
                rs.cur[s] = c0;
                rs.nxt[s] = x;
            }
            __syncthreads();
            // f(s, p0, end) for every unit [p0, p0 + RA_UNIT) of the sources' entries
            auto each_unit = [&](auto f) {
                for (int b0 = 0; b0 < ns; b0 += RA_T) {
                    const int m = min(RA_T, ns - b0);
                    const int u = tid < m ? (rs.nxt[b0 + tid] - rs.cur[b0 + tid] + RA_UNIT - 1) / RA_UNIT : 0;
                    int tot;
                    const int at = ra_scan<RA_T>(u, &tot, sh->wsm);
                    if (tid < m) sh->upre[tid] = at;
                    if (tid == 0) sh->upre[m] = tot;
                    __syncthreads();
                    const int units = sh->upre[m];
                    int s = 0;
                    for (int u = warp; u < units; u += NWP) {
                        while (sh->upre[s + 1] <= u) ++s;
                        f(b0 + s, rs.cur[b0 + s] + (u - sh->upre[s]) * RA_UNIT, rs.nxt[b0 + s]);
                    }
                    __syncthreads();
                }
            };
            // ---- mark the rows of the window ----
            each_unit([&](int s, int p0, int end) {
                const int32_t* rows = rs.rows[s] + lane;
                int rr[RA_UNIT / 32];
#pragma unroll
                for (int c = 0; c < RA_UNIT / 32; ++c)
                    rr[c] = p0 + 32 * c + lane < end ? __ldg(rows + p0 + 32 * c) : -1;
#pragma unroll
                for (int c = 0; c < RA_UNIT / 32; ++c)
                    if (rr[c] >= 0) {
                        const int off = rr[c] - r0;
                        atomicOr(bm + (off >> 5), 1u << (off & 31));
                    }
            });
            if (!FILL) {
                for (int i = tid; i < nwords; i += RA_T) cnt += __popc(bm[i]);
                __syncthreads();
            } else {
                // ---- positions: exclusive prefix counts of the bitmap words ----
                int wtot = 0;
                // Four words per thread and scan: with one, the 32 scans of a wide bitmap were most
                // of a sparse column (1M vertices of 8 entries, 2 stages: 696 ms, now 444).
                for (int w0 = 0; w0 < nwords; w0 += RA_T * 4) {
                    const int w = w0 + tid * 4;
                    int c[4], sum = 0, tot;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        c[q] = w + q < nwords ? __popc(bm[w + q]) : 0;
                        sum += c[q];
                    }
                    int at = wtot + ra_scan<RA_T>(sum, &tot, sh->wsm);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (w + q < nwords) wpre[w + q] = at;
                        at += c[q];
                    }
                    wtot += tot;
                }
                __syncthreads();
                // rows of the entries, in order
                for (int w = tid; w < nwords; w += RA_T) {
                    int64_t at = obase + wpre[w];
                    for (uint32_t x = bm[w]; x; x &= x - 1u) a.row_out[at++] = r0 + 32 * w + __ffs(x) - 1;
                }
                // ---- sums ----
                auto products = [&](auto put) {  // put(position, sum)
                    each_unit([&](int s, int p0, int end) {
                        const int32_t* rows = rs.rows[s];
                        const float akj = rs.akj[s];
                        int rr[RA_UNIT / 32];
                        unsigned long long q[RA_UNIT / 32];
#pragma unroll
                        for (int c = 0; c < RA_UNIT / 32; ++c) {
                            const int p = p0 + 32 * c + lane;
                            rr[c] = p < end ? __ldg(rows + p) : -1;
                            if (STAGE)
                                q[c] = __float_as_uint(
                                    p < end ? __ldg(reinterpret_cast<const float*>(rs.vals[s]) + p) : 0.0f);
                            else
                                q[c] = p < end ? reinterpret_cast<const unsigned long long*>(rs.vals[s])[p] : 0ull;
                        }
#pragma unroll
                        for (int c = 0; c < RA_UNIT / 32; ++c)
                            if (rr[c] >= 0) {
                                const int off = rr[c] - r0;
                                const int rank = wpre[off >> 5] +
                                                 __popc(bm[off >> 5] & ((1u << (off & 31)) - 1u));
                                put(rank, STAGE ? fx.q(__uint_as_float((unsigned)q[c]), akj) : q[c]);
                            }
                    });
                };
                if (wtot <= CAP) {
                    products([&](int rank, unsigned long long q) {
                        const unsigned ql = (unsigned)q;
                        const unsigned old = atomicAdd(lo32 + rank, ql);
                        const unsigned qh = (unsigned)(q >> 32) + (old + ql < old ? 1u : 0u);
                        if (qh) atomicAdd(hi32 + rank, qh);
                    });
                    for (int e = tid; e < wtot; e += RA_T) {
                        a.val_out[obase + e] = ((unsigned long long)hi32[e] << 32) | lo32[e];
                        lo32[e] = 0u;
                        hi32[e] = 0u;
                    }
                    __syncthreads();
                } else {  // 64-bit atomics in global memory
                    for (int e = tid; e < wtot; e += RA_T) a.val_out[obase + e] = 0ull;
                    __syncthreads();
                    products([&](int rank, unsigned long long q) { atomicAdd(a.val_out + obase + rank, q); });
                }
                obase += wtot;
                __syncthreads();
            }
            r0 = r1;
        }
        if (!FILL) {
            double dd[1] = {0.0};
            long long qq[1] = {cnt};
            block_sum<RA_T>(dd, 0, qq, 1, &sh->bs);
            if (tid == 0) a.nnz_out[j] = qq[0];
        }
        __syncthreads();
    }
}

template <bool STAGE, bool FILL, class SH>
static void rank_launch(const RankArgs& a, int num_sms, cudaStream_t s) {
    const size_t smem = (size_t)SH::WORDS * 4 * (FILL ? 2 : 1) + (FILL ? (size_t)SH::CAP * 8 : 0) + sizeof(RankShared<SH::T>);
    auto kern = k_rank_acc<STAGE, FILL, SH>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, SH::T, smem);
    if (occ < 1) occ = 1;
    int grid = occ * num_sms;
    if (grid > a.grid_cap) grid = a.grid_cap;
    if ((int64_t)grid > a.n) grid = a.n > 0 ? (int)a.n : 1;
    cudaMemsetAsync(&a.ctr->work_ctr, 0, sizeof(int), s);
    kern<<<grid, SH::T, smem, s>>>(a);
    count_launches(1);
}

template <class SH>
static void rank_any(const RankArgs& a, bool stage, bool fill, int num_sms, cudaStream_t s) {
    if (stage)
        fill ? rank_launch<true, true, SH>(a, num_sms, s) : rank_launch<true, false, SH>(a, num_sms, s);
    else
        fill ? rank_launch<false, true, SH>(a, num_sms, s) : rank_launch<false, false, SH>(a, num_sms, s);
}

static void rank_shape(const RankArgs& a, bool stage, bool fill, int num_sms, cudaStream_t s) {
    if (a.n == 0) return;
    if (a.n <= RankTiny::WORDS * 32)
        rank_any<RankTiny>(a, stage, fill, num_sms, s);
    else if (a.n <= RankSmall::WORDS * 32)
        rank_any<RankSmall>(a, stage, fill, num_sms, s);
    else
        rank_any<RankLarge>(a, stage, fill, num_sms, s);
}

int split_grid_cap(int64_t n, int num_sms) {
    return num_sms * (n <= RankTiny::WORDS * 32 ? RankTiny::MINB : 4);
}

void launch_split_count(const RankArgs& a, bool stage, int num_sms, cudaStream_t s) {
    rank_shape(a, stage, false, num_sms, s);
}

void launch_split_fill(const RankArgs& a, bool stage, int num_sms, cudaStream_t s) {
    rank_shape(a, stage, true, num_sms, s);
}

}  // namespace mcl
