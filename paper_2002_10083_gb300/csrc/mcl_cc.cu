// Connected components of the final matrix's undirected pattern
// (Algorithm 1, "return the connected components of A").
//
// Lock-free union-find: every stored entry (i, j) hooks the larger of the
// two roots under the smaller with atomicCAS, so every root is the
// smallest vertex of its set and the final label of a vertex is the
// smallest vertex id of its component.  Retry loops make global progress
// (a failed CAS means another thread linked a root), and every loop is
// bounded; exhausting a bound raises ERR_TIMEOUT instead of spinning.
#include <cstdint>

#include "mcl_device.cuh"
#include "mcl_internal.h"

namespace mcl {

constexpr int CC_FIND_LIMIT = 1 << 22;
constexpr int CC_LINK_LIMIT = 1 << 20;

// The root of x's tree, or -1 after `limit` steps.
__device__ __forceinline__ int cc_find_within(int* parent, int x, int limit) {
    for (int it = 0; it < limit; ++it) {
        const int p = *reinterpret_cast<volatile int*>(parent + x);
        if (p == x) return x;
        const int gp = *reinterpret_cast<volatile int*>(parent + p);
        if (gp != p) atomicCAS(parent + x, p, gp);  // path halving, benign if it loses
        x = gp;
    }
    return -1;
}

__device__ __forceinline__ int cc_find(int* parent, int x, DevCounters* ctr) {
    const int r = cc_find_within(parent, x, CC_FIND_LIMIT);
    if (r < 0) atomicOr(&ctr->err, ERR_TIMEOUT);
    return r < 0 ? x : r;
}

__global__ void k_cc_init(int32_t n, int* parent) {
    int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v < n) parent[v] = (int)v;
}

__device__ __forceinline__ void cc_link(int* parent, int a, int b, DevCounters* ctr) {
    int it = 0;
    for (; it < CC_LINK_LIMIT; ++it) {
        a = cc_find(parent, a, ctr);
        b = cc_find(parent, b, ctr);
        if (a == b) break;
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        // a > b: hang root a under root b
        if (atomicCAS(parent + a, a, b) == a) break;
    }
    if (it == CC_LINK_LIMIT) atomicOr(&ctr->err, ERR_TIMEOUT);
}

// The components are found in three steps, as in Afforest (Sutton, Ben-Nun and
// Barak, 2018): a few entries of every column are linked, all paths are
// compressed, and then every entry is looked at: most already have the same
// parent as their column and need no walk.  Linking every entry from the start
// took 755 us on 13.5M entries, all warps contending for the same few roots.
// With one first entry, 1M vertices banded from the diagonal take 0.99 ms instead of
// 0.38 (their columns begin with themselves); with four, 2M random columns of 3
// take 0.79 instead of 0.72.
constexpr int CC_FIRST = 2;
// The first step gives up after so many steps of a walk and leaves the entry to
// the last: on a ring, all threads at once build a path of 300k vertices, and
// those of the next wave walked it one step after the other (1M vertices: 119 ms
// without the limit, 0.5 with it, 3.1 to 4.3 with every entry linked from the
// start).  8: 0.31 ms instead of 0.39 on a ring in both directions, but 1.2 to
// 1.5 times as long on shallow trees; 64: 0.67 instead of 0.45 on a band of five.
constexpr int CC_FIRST_WALK = 16;
// Few entries, or few per column (a converged matrix), are linked at once: two
// launches less (300 columns of 30 entries: 52 us against 60; 1,000 of 16: 77
// against 70; 20,000 of one: 51 against 60).
constexpr int64_t CC_FEW = 12288, CC_FEW_SPARSE = 65536;

// thread per column: link its first CC_FIRST entries and its last
__global__ void k_cc_first(CscView A, int* parent, DevCounters* ctr) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= A.n) return;
    const int64_t cb = A.colptr[j], ce = A.colptr[j + 1];
    auto link = [&](int b) {
        int a = (int)j;
        if (a == b) return;
        for (int it = 0; it < CC_FIRST_WALK; ++it) {
            a = cc_find_within(parent, a, CC_FIRST_WALK);
            b = cc_find_within(parent, b, CC_FIRST_WALK);
            if (a < 0 || b < 0) break;
            if (a == b) return;
            if (a < b) {
                const int t = a;
                a = b;
                b = t;
            }
            if (atomicCAS(parent + a, a, b) == a) return;
        }
        ctr->cc_left = 1;
    };
    for (int64_t p = cb; p < ce && p < cb + CC_FIRST; ++p) link(A.rowidx[p]);
    if (ce > cb + CC_FIRST) link(A.rowidx[ce - 1]);
}

__global__ void k_cc_compress(int32_t n, int* parent, DevCounters* ctr) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const int p = parent[v], r = cc_find(parent, (int)v, ctr);
    if (r != p) parent[v] = r;
}

// warp per column: link every stored (row, column) pair; after k_cc_first those
// whose ends do not already have one parent (a parent read from a cache may be
// an old one: two vertices that once had the same are in one set all the same)
template <bool FIRST>
__global__ void k_cc_hook(CscView A, int* parent, DevCounters* ctr) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int done = FIRST && !ctr->cc_left ? CC_FIRST + 1 : 0;  // columns of so few entries are linked
    for (int64_t j = gw; j < A.n; j += nw) {
        const int64_t cb = A.colptr[j], ce = A.colptr[j + 1];
        if (ce - cb <= done) continue;
        if (FIRST) {
            const int pj = parent[j];
            for (int64_t p = cb + lane; p < ce; p += 128) {
                int b[4], q[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) b[c] = p + 32 * c < ce ? A.rowidx[p + 32 * c] : (int)j;
#pragma unroll
                for (int c = 0; c < 4; ++c) q[c] = parent[b[c]];
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (q[c] != pj && b[c] != (int)j) cc_link(parent, (int)j, b[c], ctr);
            }
        } else {
            for (int64_t p = cb + lane; p < ce; p += 32) {
                const int b = A.rowidx[p];
                if (b != (int)j) cc_link(parent, (int)j, b, ctr);
            }
        }
    }
}

__global__ void k_cc_label(int32_t n, int* parent, int32_t* labels, DevCounters* ctr) {
    int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v < n) labels[v] = cc_find(parent, (int)v, ctr);
}

void launch_components(const CscView& A, int32_t* labels, DevCounters* ctr, cudaStream_t s) {
    if (A.n == 0) return;
    // labels doubles as the parent array (int32, same length)
    int* parent = reinterpret_cast<int*>(labels);
    const unsigned nb = (unsigned)((A.n + 255) / 256);
    k_cc_init<<<nb, 256, 0, s>>>(A.n, parent);
    count_launches(1);
    int64_t blocks = ((int64_t)A.n * 32 + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (A.nnz <= CC_FEW || (A.nnz <= CC_FEW_SPARSE && A.nnz <= 2 * (int64_t)A.n)) {
        k_cc_hook<false><<<(unsigned)blocks, 256, 0, s>>>(A, parent, ctr);
    } else {
        k_cc_first<<<nb, 256, 0, s>>>(A, parent, ctr);
        k_cc_compress<<<nb, 256, 0, s>>>(A.n, parent, ctr);
        k_cc_hook<true><<<(unsigned)blocks, 256, 0, s>>>(A, parent, ctr);
        count_launches(2);
    }
    count_launches(1);
    k_cc_label<<<nb, 256, 0, s>>>(A.n, parent, labels, ctr);
    count_launches(1);
}

}  // namespace mcl
