// Source-cluster tree, target batches, interaction lists and work items
// (Section 5.1, Eq. MAC, Algorithm 3), built on the GPU level by level.
//
// Every level runs point-parallel passes over the positions of the clusters
// being split: bounding boxes (order-preserving 64-bit min/max), child codes,
// a stable partition by code (block counts + one global scan), and the child
// records.  Geometric decisions use explicitly rounded float64 operations
// (__dadd_rn and friends are never contracted into FMAs) so they round exactly
// as the formulas are written.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <initializer_list>
#include <cstring>
#include <utility>

#include "tagi_internal.cuh"

namespace tagi {

namespace {

constexpr double kSqrt2 = 1.4142135623730951;
constexpr int kScanThreads = 1024;
constexpr int kBlk = 1024;  // positions per block in the partition passes

__device__ __forceinline__ unsigned long long ord64(double v)
{
    v = v + 0.0;  // -0 -> +0
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double unord64(unsigned long long o)
{
    unsigned long long b = (o >> 63) ? (o & 0x7fffffffffffffffull) : ~o;
    return __longlong_as_double((long long)b);
}

// ---------------------------------------------------------------- scans
__global__ void __launch_bounds__(kScanThreads) k_scan_i64(const int64_t* __restrict__ in, int64_t* __restrict__ out,
                                                           int64_t n)
{
    __shared__ int64_t ws[kScanThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t per = (n + kScanThreads - 1) / kScanThreads;
    const int64_t a = min(n, (int64_t)tid * per), b = min(n, a + per);
    int64_t s = 0;
    for (int64_t i = a; i < b; i++) s += in[i];
    int64_t x = s;  // inclusive over the warp
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t v = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += v;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int64_t y = ws[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t v = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += v;
        }
        ws[lane] = y;
    }
    __syncthreads();
    int64_t run = x - s + (warp > 0 ? ws[warp - 1] : 0);
    for (int64_t i = a; i < b; i++) {
        const int64_t v = in[i];
        out[i] = run;
        run += v;
    }
    if (tid == kScanThreads - 1) out[n] = run;
}

// ---------------------------------------------------------------- level passes
__global__ void k_init(int* pos, int* seg, int64_t n)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) {
        pos[i] = (int)i;
        seg[i] = 0;
    }
}

__global__ void k_init_root(int n, int* begin, int* end, int* parent, int* level, int* nchild,
                            unsigned long long* blo, unsigned long long* bhi)
{
    begin[0] = 0;
    end[0] = n;
    parent[0] = -1;
    level[0] = 0;
    nchild[0] = 0;
    for (int d = 0; d < 3; d++) {
        blo[d] = ~0ull;
        bhi[d] = 0ull;
    }
}

// Bounding boxes of the clusters owning seg[p] >= 0.  Positions of a cluster
// are consecutive, so most blocks hold one cluster: its warps reduce by
// shuffles, the block in shared memory, and six atomics go out instead of six a
// warp (which serialise on the root's six words).
constexpr int kBoxThreads = 256;
__global__ void __launch_bounds__(kBoxThreads) k_bbox(const int* __restrict__ pos, const int* __restrict__ seg,
                                                      const double* __restrict__ xyz, int64_t n,
                                                      unsigned long long* blo, unsigned long long* bhi)
{
    __shared__ unsigned long long smn[kBoxThreads / 32][3], smx[kBoxThreads / 32][3];
    const int64_t p = blockIdx.x * (int64_t)kBoxThreads + threadIdx.x;
    const int c = p < n ? seg[p] : -1;
    unsigned long long v[3] = {0, 0, 0};
    if (c >= 0) {
        const int i = pos[p];
        v[0] = ord64(xyz[i]);
        v[1] = ord64(xyz[n + i]);
        v[2] = ord64(xyz[2 * n + i]);
    }
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ int sc;
    if (threadIdx.x == 0) sc = c;
    __syncthreads();
    const bool one = __syncthreads_and(c == sc);
    if (one && sc < 0) return;
    if (one || __all_sync(full, c == __shfl_sync(full, c, 0))) {
        unsigned long long mn[3] = {v[0], v[1], v[2]}, mx[3] = {v[0], v[1], v[2]};
        for (int off = 16; off > 0; off >>= 1)
            for (int d = 0; d < 3; d++) {
                const unsigned long long a = __shfl_down_sync(full, mn[d], off), b = __shfl_down_sync(full, mx[d], off);
                mn[d] = min(mn[d], a);
                mx[d] = max(mx[d], b);
            }
        if (one) {
            if (lane == 0)
                for (int d = 0; d < 3; d++) {
                    smn[warp][d] = mn[d];
                    smx[warp][d] = mx[d];
                }
        } else if (lane == 0 && c >= 0) {
            for (int d = 0; d < 3; d++) {
                atomicMin(&blo[3 * c + d], mn[d]);
                atomicMax(&bhi[3 * c + d], mx[d]);
            }
        }
    } else if (c >= 0) {
        for (int d = 0; d < 3; d++) {
            atomicMin(&blo[3 * c + d], v[d]);
            atomicMax(&bhi[3 * c + d], v[d]);
        }
    }
    if (!one) return;
    __syncthreads();
    if (threadIdx.x < 3) {
        const int d = threadIdx.x;
        unsigned long long mn = smn[0][d], mx = smx[0][d];
        for (int w = 1; w < kBoxThreads / 32; w++) {
            mn = min(mn, smn[w][d]);
            mx = max(mx, smx[w][d]);
        }
        atomicMin(&blo[3 * c + d], mn);
        atomicMax(&bhi[3 * c + d], mx);
    }
}

// Finish boxes of clusters [first, last): lo/hi, center, radius; decide the split.
__global__ void k_finalize(int first, int last, const unsigned long long* blo, const unsigned long long* bhi,
                           const int* begin, const int* end, int leaf_size, double* lo, double* hi,
                           double* cen, double* rad, double* mid, int* smask)
{
    int c = first + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= last) return;
    double l[3], h[3], e[3], emax = 0.0;
    for (int d = 0; d < 3; d++) {
        l[d] = unord64(blo[3 * c + d]);
        h[d] = unord64(bhi[3 * c + d]);
        lo[3 * c + d] = l[d];
        hi[3 * c + d] = h[d];
        cen[3 * c + d] = __dmul_rn(__dadd_rn(l[d], h[d]), 0.5);
        e[d] = __dsub_rn(h[d], l[d]);
        if (e[d] > emax) emax = e[d];
    }
    rad[c] = __dmul_rn(__dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(e[0], e[0]), __dmul_rn(e[1], e[1])),
                                             __dmul_rn(e[2], e[2]))),
                       0.5);
    int m = 0;
    if (end[c] - begin[c] > leaf_size && emax > 0.0) {
        for (int d = 0; d < 3; d++)
            if (__dmul_rn(e[d], kSqrt2) >= emax) m |= 1 << d;
    }
    smask[c] = m;
    for (int d = 0; d < 3; d++) mid[3 * c + d] = cen[3 * c + d];
}

// Child code of every position (-1 outside the clusters being split), and per
// block of kBlk positions the number of positions with each code, stored
// bin-major: cnt[b * nblk + blk].
__global__ void __launch_bounds__(kBlk) k_codes(const int* __restrict__ pos, const int* __restrict__ seg,
                                                const double* __restrict__ xyz, int64_t n,
                                                const int* __restrict__ smask, const double* __restrict__ mid,
                                                signed char* code, int64_t nblk, int64_t* cnt)
{
    __shared__ int wc[kBlk / 32][8];
    const int64_t p = blockIdx.x * (int64_t)kBlk + threadIdx.x;
    int k = -1;
    const int c = p < n ? seg[p] : -1;
    if (c >= 0) {
        const int m = smask[c];
        if (m) {
            const int i = pos[p];
            k = 0;
            for (int d = 0; d < 3; d++)
                if ((m >> d) & 1)
                    if (xyz[d * n + i] >= mid[3 * c + d]) k |= 1 << d;
        }
    }
    code[p] = (signed char)k;  // the array holds whole blocks
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int b = 0; b < 8; b++) {
        const unsigned m = __ballot_sync(0xffffffffu, k == b);
        if (lane == 0) wc[warp][b] = __popc(m);
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        int s = 0;
        for (int w = 0; w < kBlk / 32; w++) s += wc[w][threadIdx.x];
        cnt[threadIdx.x * nblk + blockIdx.x] = s;
    }
}

// One warp per cluster of the level: per-bin counts between begin and end and
// the bin prefix at begin (block offsets plus a warp-parallel partial count).
__device__ void prefix8(const int64_t* off, const signed char* code, int64_t nblk, int64_t x, int lane, int64_t (&pf)[8])
{
    const int64_t blk = x / kBlk;
    int cnt[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    // four codes a load; bytes at or beyond x do not count
#pragma unroll
    for (int i = 0; i < kBlk / 128; i++) {
        const int64_t q = blk * kBlk + 4 * lane + 128 * i;
        if (q >= x) continue;
        unsigned w = *reinterpret_cast<const unsigned*>(code + q);
        if (x - q < 4) w |= 0xffffffffu << (8 * (int)(x - q));
#pragma unroll
        for (int b = 0; b < 8; b++) cnt[b] += __popc(__vcmpeq4(w, b * 0x01010101u)) >> 3;
    }
#pragma unroll
    for (int b = 0; b < 8; b++) {
        int v = cnt[b];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        pf[b] = off[b * nblk + blk] + v;
    }
}

__global__ void k_counts(int first, int last, const int* begin, const int* end, const int* smask,
                         const signed char* code, const int64_t* off, int64_t nblk, int* cnt, int64_t* pfx,
                         int64_t* nnz)
{
    const int c = first + (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32);
    const int lane = threadIdx.x & 31;
    if (c >= last) return;  // uniform per warp
    const int j = c - first;
    int64_t pb[8], pe[8];
    if (smask[c]) {
        prefix8(off, code, nblk, begin[c], lane, pb);
        prefix8(off, code, nblk, end[c], lane, pe);
    } else {
        for (int b = 0; b < 8; b++) pb[b] = pe[b] = 0;
    }
    if (lane == 0) {
        int z = 0;
        for (int b = 0; b < 8; b++) {
            const int v = (int)(pe[b] - pb[b]);
            cnt[8 * j + b] = v;
            pfx[8 * j + b] = pb[b];
            z += v > 0;
        }
        nnz[j] = z;
    }
}

__global__ void k_children(int first, int last, int nc0, const int64_t* cbase, const int* begin, const int* cnt,
                           int lvl, int* cbeg, int* cend, int* cpar, int* clev, int* cnch, int* cchild,
                           int* bfirst, int* bid, unsigned long long* blo, unsigned long long* bhi)
{
    int c = first + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= last) return;
    int j = c - first;
    int id = nc0 + (int)cbase[j];
    int start = begin[c];
    int q = 0;
    for (int b = 0; b < 8; b++) {
        int v = cnt[8 * j + b];
        bfirst[8 * j + b] = start;
        bid[8 * j + b] = -1;
        if (v > 0) {
            cbeg[id] = start;
            cend[id] = start + v;
            cpar[id] = c;
            clev[id] = lvl + 1;
            cnch[id] = 0;
            for (int d = 0; d < 3; d++) {
                blo[3 * id + d] = ~0ull;
                bhi[3 * id + d] = 0ull;
            }
            cchild[8 * c + q] = id;
            bid[8 * j + b] = id;
            q++;
            id++;
        }
        start += v;
    }
    cnch[c] = q;
}

// Stable scatter of the positions of split clusters into their children.
__global__ void k_scatter(const int* __restrict__ posA, const int* __restrict__ segA,
                          const signed char* __restrict__ code, int64_t n, int64_t nblk, const int64_t* off,
                          int first, const int64_t* pfx, const int* bfirst, const int* bid, const int* cnt,
                          int* posB, int* segB, int* err)
{
    __shared__ int wc[kBlk / 32][8];
    int64_t p = blockIdx.x * (int64_t)kBlk + threadIdx.x;
    int k = p < n ? code[p] : -1;
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned mine = 0;
    for (int b = 0; b < 8; b++) {
        unsigned m = __ballot_sync(0xffffffffu, k == b);
        if (lane == 0) wc[warp][b] = __popc(m);
        if (k == b) mine = m;
    }
    __syncthreads();
    if (p >= n) return;
    if (k < 0) {
        posB[p] = posA[p];
        segB[p] = -1;
        return;
    }
    int before = 0;
    for (int w = 0; w < warp; w++) before += wc[w][k];
    before += __popc(mine & ((1u << lane) - 1u));
    int c = segA[p];
    int j = c - first;
    int64_t rank = off[k * nblk + blockIdx.x] + before - pfx[8 * j + k];
    if (rank < 0 || rank >= cnt[8 * j + k]) {  // cannot happen; guards the write
        atomicOr(err, 2);
        return;
    }
    int64_t dest = bfirst[8 * j + k] + rank;
    posB[dest] = posA[p];
    segB[dest] = bid[8 * j + k];
}

__global__ void k_gather_points(const int* pos, const double* xyz, const double* w, int64_t n, double* px,
                                double* py, double* pz, double* pw)
{
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    int i = pos[p];
    px[p] = xyz[i];
    py[p] = xyz[n + i];
    pz[p] = xyz[2 * n + i];
    pw[p] = w[i];
}

__global__ void k_is_leaf(int nc, const int* nch, int64_t* flag)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < nc) flag[c] = nch[c] == 0;
}

// flag[c] = approximated, size[c] = its points (0 otherwise)
__global__ void k_far_flags(int nc, const int* is_far, const int* begin, const int* end, int64_t* flag, int64_t* size)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nc) return;
    flag[c] = is_far[c];
    size[c] = is_far[c] ? end[c] - begin[c] : 0;
}

// Values that the host reads together: one launch and one wait for all of them.
constexpr int kReadMax = 8;
struct ReadList {
    const int64_t* p64[kReadMax];
    const int* p32[kReadMax];
    int n;
};
__global__ void k_collect(ReadList L, int64_t* out)
{
    const int i = threadIdx.x;
    if (i < L.n) out[i] = L.p64[i] ? *L.p64[i] : (int64_t)*L.p32[i];
}

__global__ void k_compact(int nc, const int64_t* flag, const int64_t* off, int* out, int* idx_of)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nc) return;
    if (flag[c]) {
        out[off[c]] = c;
        if (idx_of) idx_of[c] = (int)off[c];
    } else if (idx_of) {
        idx_of[c] = -1;
    }
}

__global__ void k_fill_leaf(const int* leaves, const int* begin, const int* end, int* pt_leaf)
{
    int c = leaves[blockIdx.x];
    for (int p = begin[c] + threadIdx.x; p < end[c]; p += blockDim.x) pt_leaf[p] = c;
}

// ---------------------------------------------------------------- lists
struct ListArgs {
    const int *begin, *end, *nch, *child, *pt_leaf, *leaves;
    const double *cen, *rad;
    double theta;
    int P;
};

// Algorithm 3's ComputePotential for one batch, one warp per batch: the
// clusters to visit form a frontier (level by level from the root), each lane
// applies the MAC to one cluster, and warp prefix sums place the entries and
// the opened children in lane order, so the output order is deterministic.
// In count mode (FILL false) only counts are produced.  The MAC arithmetic is
// the float64 expression of the oracle, without contraction.
constexpr int kListWarps = 2;      // warps (batches) per CTA
constexpr int kFront = 1024;       // frontier capacity per warp and level

__device__ __forceinline__ int warp_excl(int v, int lane, int* total)
{
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    *total = __shfl_sync(0xffffffffu, x, 31);
    return x - v;
}

template <bool FILL>
__device__ void walk_warp(const ListArgs a, int batch, int limit, int* front, int* nent, int64_t* near_src,
                          int64_t* far_src, Entry* out, int* out_batch, int* out_clus, int* is_far, int* err)
{
    const int lane = threadIdx.x & 31;
    int* cur = front;
    int* nxt = front + kFront;
    if (lane == 0) cur[0] = 0;
    __syncwarp();
    int ncur = 1, cnt = 0;
    int64_t sn = 0, sf = 0;  // per lane
    const double bx = a.cen[3 * batch], by = a.cen[3 * batch + 1], bz = a.cen[3 * batch + 2];
    const double rb = a.rad[batch];
    while (ncur > 0) {
        int nnext = 0;
        for (int base = 0; base < ncur; base += 32) {
            const int i = base + lane;
            int c = -1, kind = 0, ne = 0, nch = 0;  // kind: 1 far, 2 open, 3 direct
            if (i < ncur) {
                c = cur[i];
                const double dx = __dsub_rn(bx, a.cen[3 * c]), dy = __dsub_rn(by, a.cen[3 * c + 1]),
                             dz = __dsub_rn(bz, a.cen[3 * c + 2]);
                const double R =
                    __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
                const bool theta_ok = __ddiv_rn(__dadd_rn(rb, a.rad[c]), R) < a.theta;
                const bool size_ok = a.P < a.end[c] - a.begin[c];
                if (theta_ok && size_ok) {
                    kind = 1;
                    ne = 1;
                } else if (!theta_ok && a.nch[c] > 0) {
                    kind = 2;
                    nch = a.nch[c];
                } else {
                    // direct sum with every point of c: one entry per leaf below it
                    kind = 3;
                    for (int p = a.begin[c]; p < a.end[c]; p = a.end[a.pt_leaf[p]]) ne++;
                }
            }
            int etot, ctot;
            const int eoff = warp_excl(ne, lane, &etot);
            const int coff = warp_excl(nch, lane, &ctot);
            if ((FILL && cnt + etot > limit) || nnext + ctot > kFront) {
                if (lane == 0) *err = 1;
                return;
            }
            if (kind == 2)
                for (int q = 0; q < nch; q++) nxt[nnext + coff + q] = a.child[8 * c + q];
            if (kind == 1) {
                sf += a.P;
                if (FILL) {
                    out[cnt + eoff] = Entry{0, 0, c, 2};
                    out_batch[cnt + eoff] = batch;
                    out_clus[cnt + eoff] = c;
                    is_far[c] = 1;
                }
            } else if (kind == 3) {
                int t = 0;
                for (int p = a.begin[c]; p < a.end[c];) {
                    const int leaf = a.pt_leaf[p];
                    const int e = a.end[leaf];
                    if (FILL) {
                        out[cnt + eoff + t] = Entry{a.begin[leaf], e, leaf, leaf == batch ? 1 : 0};
                        out_batch[cnt + eoff + t] = batch;
                        out_clus[cnt + eoff + t] = leaf;
                    }
                    sn += e - a.begin[leaf];
                    t++;
                    p = e;
                }
            }
            cnt += etot;
            nnext += ctot;
        }
        __syncwarp();
        int* t = cur;
        cur = nxt;
        nxt = t;
        ncur = nnext;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sn += __shfl_down_sync(0xffffffffu, sn, o);
        sf += __shfl_down_sync(0xffffffffu, sf, o);
    }
    *nent = cnt;
    *near_src = sn;  // lane 0 holds the sums
    *far_src = sf;
}

__global__ void __launch_bounds__(32 * kListWarps) k_list_count(ListArgs a, int nleaf, int64_t* cnt,
                                                                 int64_t* near_pairs, int64_t* far_pairs, int* err)
{
    __shared__ int front[kListWarps][2 * kFront];
    const int w = threadIdx.x >> 5;
    const int j = blockIdx.x * kListWarps + w;
    if (j >= nleaf) return;
    const int b = a.leaves[j];
    int ne = 0;
    int64_t sn = 0, sf = 0;
    walk_warp<false>(a, b, 0, front[w], &ne, &sn, &sf, nullptr, nullptr, nullptr, nullptr, err);
    if ((threadIdx.x & 31) == 0) {
        cnt[j] = ne;
        const int64_t nb = a.end[b] - a.begin[b];
        near_pairs[j] = nb * sn;
        far_pairs[j] = nb * sf;
    }
}

__global__ void __launch_bounds__(32 * kListWarps) k_list_fill(ListArgs a, int nleaf, const int64_t* off, Entry* ent,
                                                                int* eb, int* ec, int* is_far, int* err)
{
    __shared__ int front[kListWarps][2 * kFront];
    const int w = threadIdx.x >> 5;
    const int j = blockIdx.x * kListWarps + w;
    if (j >= nleaf) return;
    const int b = a.leaves[j];
    int ne;
    int64_t sn, sf;
    const int64_t o = off[j];
    walk_warp<true>(a, b, (int)(off[j + 1] - o), front[w], &ne, &sn, &sf, ent + o, eb + o, ec + o, is_far, err);
}

__global__ void k_far_ranges(int64_t nent, Entry* ent, const int* cl_far, int64_t n, int P)
{
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= nent) return;
    Entry x = ent[e];
    if (x.flags & 2) {
        int64_t s0 = n + (int64_t)cl_far[x.frame] * P;
        x.src0 = (int)s0;
        x.src1 = (int)(s0 + P);
        ent[e] = x;
    }
}

// flags bit2: the boxes of the batch and of the source cluster are at least
// sqrt(42) alpha apart, so exp(-r^2/alpha^2) <= 2^-60 for every pair of the
// entry and the Gaussian of the Coulomb SS is below float32 resolution there
// (the FP32C kernel leaves it out; the float64 kernel ignores the bit).
// pairs[0], pairs[1]: near and far pairs of the flagged entries.
__global__ void k_gauss_flags(int64_t nent, Entry* ent, const int* eb, const int* ec, const double* lo,
                              const double* hi, const int* begin, const int* end, double alpha,
                              unsigned long long* pairs)
{
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= nent) return;
    const int b = eb[e], c = ec[e];
    double d2 = 0.0;
    for (int k = 0; k < 3; k++) {
        const double g = fmax(0.0, fmax(lo[3 * c + k] - hi[3 * b + k], lo[3 * b + k] - hi[3 * c + k]));
        d2 += g * g;
    }
    if (d2 >= 42.0 * alpha * alpha) {
        Entry x = ent[e];
        x.flags |= 4;
        ent[e] = x;
        const unsigned long long np = (unsigned long long)(end[b] - begin[b]) * (unsigned long long)(x.src1 - x.src0);
        atomicAdd(pairs + ((x.flags & 2) ? 1 : 0), np);
    }
}

// Offset of each entry's frame from its batch's center, as a two-float, so
// that the near/far kernel shifts positions without float64.
__global__ void k_entry_shift(int64_t nent, const Entry* __restrict__ ent, const int* __restrict__ eb,
                              const double* __restrict__ cen, float4* __restrict__ out)
{
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= nent) return;
    const int f = ent[e].frame, b = eb[e];
    float h[3], l[3];
    for (int d = 0; d < 3; d++) {
        const double o = cen[3 * f + d] - cen[3 * b + d];
        h[d] = (float)o;
        l[d] = (float)(o - (double)h[d]);
    }
    out[2 * e] = make_float4(h[0], h[1], h[2], 0.0f);
    out[2 * e + 1] = make_float4(l[0], l[1], l[2], 0.0f);
}

// ---------------------------------------------------------------- work items
// A target chunk's items are runs of its batch's list.  Two ways to cut it:
//   whole: an item takes whole entries until they hold at least seg sources
//     (padded to 8), the next begins after them;
//   split: each entry is padded to whole folds of 16 and cut into units where
//     an item may begin -- every kItemUnit sources of a direct entry (the
//     kernel's tile), an approximated cluster as one unit -- and item s starts
//     at the first unit at or after position s * seg.  A unit is no longer
//     than seg, so no item is empty, and units are whole folds, so the cut
//     moves no float32 sum.
constexpr int kItemUnit = 128;
constexpr int kSegment = 8192, kItemsWanted = 8192, kItemsFew = 2000;
constexpr int kAntChunkMin = 256, kAntItemsWanted = 1216;
static_assert(kItemUnit % 16 == 0, "whole folds");

__host__ __device__ __forceinline__ int padded(int v) { return (v + 15) & ~15; }
// offset of the entry's last unit from its start
__device__ __forceinline__ int last_unit(const Entry& x)
{
    return (x.flags & 2) ? 0 : (x.src1 - x.src0 - 1) / kItemUnit * kItemUnit;
}

// The segments of one batch's list, by one warp, 32 entries at a time with a
// warp prefix sum of their lengths.  start(s, e, skip) is called by one lane
// for each segment s: it begins at source skip of entry e.  Returns their
// number (all lanes).
template <class F>
__device__ int walk_segments(const Entry* __restrict__ ent, int64_t e0, int64_t e1, int seg, bool split, F&& start)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    if (e0 == e1 && lane == 0) start(0, (int)e0, 0);
    int64_t at = 0, prev = -1;  // split: start of this round's first entry; of the unit before it
    int nseg = e0 == e1 ? 1 : 0;
    int64_t open = -1;          // whole: position where the open segment began
    for (int64_t base = e0; base < e1; base += 32) {
        const int64_t e = base + lane;
        const bool live = e < e1;
        const Entry x = live ? ent[e] : Entry{0, 0, 0, 2};
        const int len = split ? padded(x.src1 - x.src0) : (x.src1 - x.src0 + 7) & ~7;
        int64_t incl = len;
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t v = __shfl_up_sync(full, incl, o);
            if (lane >= o) incl += v;
        }
        incl += at;
        const int m = (int)min((int64_t)31, e1 - 1 - base);
        if (split) {
            const int64_t a = incl - len, last = a + (live ? last_unit(x) : 0);
            int64_t before = __shfl_up_sync(full, last, 1);
            if (lane == 0) before = prev;
            if (live)
                for (int64_t s = before < 0 ? 0 : before / seg + 1; s <= last / seg; s++) {
                    const int64_t off = s * seg - a;  // first unit at or after off
                    start((int)s, (int)e, off <= 0 ? 0 : (int)((off + kItemUnit - 1) / kItemUnit * kItemUnit));
                }
            prev = __shfl_sync(full, last, m);
            nseg = (int)(prev / seg) + 1;
        } else {
            int first = 0;  // lane where the next segment begins, 32: not in this round
            while (first <= m) {
                if (open < 0) {
                    open = first == 0 ? at : __shfl_sync(full, incl, first - 1);
                    if (lane == first) start(nseg, (int)e, 0);
                    nseg++;
                }
                const unsigned done = __ballot_sync(full, live && lane >= first && incl - open >= seg);
                if (!done) break;
                first = __ffs(done);  // the lane after the one that fills it
                open = -1;
            }
        }
        at = __shfl_sync(full, incl, m);
    }
    return nseg;
}

// One warp per batch: target chunks and items (chunks times segments).
__global__ void k_item_counts(int nleaf, const int* leaves, const int* begin, const int* end, const int64_t* eoff,
                              const Entry* ent, int seg, int split, int64_t* nchunk, int64_t* nitem)
{
    const int j = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32);
    if (j >= nleaf) return;  // uniform per warp
    const int segs = walk_segments(ent, eoff[j], eoff[j + 1], seg, split, [](int, int, int) {});
    if ((threadIdx.x & 31) == 0) {
        const int b = leaves[j];
        const int ch = (end[b] - begin[b] + kTargetsPerItem - 1) / kTargetsPerItem;
        nchunk[j] = ch;
        nitem[j] = (int64_t)ch * segs;
    }
}

// One block per batch.  Its warp 0 leaves the start of every segment in the
// first chunk's items; then all threads complete the items of all chunks and
// the order in which CTAs take them: an item runs for a millisecond on a large
// tree, so the chunks' last items, which are shorter, come last.
__global__ void __launch_bounds__(128) k_item_fill(int nleaf, const int* leaves, const int* begin, const int* end,
                                                   const int64_t* eoff, const Entry* ent, int seg, int split,
                                                   const int64_t* chunk_off, const int64_t* item_off, Item* items,
                                                   int64_t nitems, int64_t ntchunk, int* order, int* tc_item0, int* tc_t0, int* tc_t1, int* tc_batch)
{
    const int j = blockIdx.x;
    const int b = leaves[j];
    const int nb = end[b] - begin[b];
    const int64_t c0 = chunk_off[j], i0 = item_off[j], e1 = eoff[j + 1];
    const int ch = (int)(chunk_off[j + 1] - c0);
    const int segs = (int)((item_off[j + 1] - i0) / ch);
    if (threadIdx.x < 32)
        walk_segments(ent, eoff[j], e1, seg, split, [&](int s, int e, int skip) {
            if (s < segs) {
                items[i0 + s].e0 = e;
                items[i0 + s].skip = skip;
            }
        });
    __syncthreads();
    for (int q = threadIdx.x; q < ch * segs; q += blockDim.x) {
        const int ci = q / segs, s = q % segs;
        const int64_t tc = c0 + ci;
        const int t0 = begin[b] + ci * kTargetsPerItem, t1 = min(begin[b] + nb, t0 + kTargetsPerItem);
        const int64_t first = i0 + (int64_t)ci * segs;
        int f0 = items[i0 + s].e0, skip = items[i0 + s].skip, f1 = (int)e1, stop = 0;
        if (s + 1 < segs) {  // up to where the next segment starts
            f1 = items[i0 + s + 1].e0;
            stop = items[i0 + s + 1].skip;
            if (stop > 0) f1++;
        }
        Item& it = items[first + s];
        it.t0 = t0;
        it.t1 = t1;
        it.e1 = f1;
        it.stop = stop;
        it.batch = b;
        it.tchunk = (int)tc;
        it.i0 = (int)first;
        it.ni = segs;
        if (ci > 0) {
            it.e0 = f0;
            it.skip = skip;
        }
        // the CTA that takes it: the last, shorter item of every chunk after all others
        order[s < segs - 1 ? first + s - tc : nitems - ntchunk + tc] = (int)(first + s);
        if (tc == ntchunk - 1 && s == 0) tc_item0[ntchunk] = (int)nitems;
        if (s == 0) {
            tc_item0[tc] = (int)first;
            tc_t0[tc] = t0;
            tc_t1[tc] = t1;
            tc_batch[tc] = b;
        }
    }
}

__global__ void k_ant_counts(int nfar, const int* far_cl, const int* begin, const int* end, int chunk, int64_t* cnt)
{
    int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= nfar) return;
    int c = far_cl[f];
    cnt[f] = (end[c] - begin[c] + chunk - 1) / chunk;
}

__global__ void k_ant_fill(int nfar, const int* far_cl, const int* begin, const int* end, int chunk,
                           const int64_t* off, AntItem* items, int* far_ant0)
{
    int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f > nfar) return;
    far_ant0[f] = (int)off[f];
    if (f == nfar) return;
    int c = far_cl[f];
    int64_t o = off[f];
    for (int p = begin[c]; p < end[c]; p += chunk) items[o++] = AntItem{p, min(end[c], p + chunk), c, f};
}

// ---------------------------------------------------------------- records
// Mesh-point records: position relative to the center of the point's leaf
// and quadrature weight, each as a two-float (hi in rec4, lo in rec4lo).
__global__ void k_point_records(int64_t n, const double* px, const double* py, const double* pz, const double* pw,
                                const int* pt_leaf, const double* cen, float4* rec4, float4* rec4lo, double* rx,
                                double* ry, double* rz, double* rw)
{
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    if (rec4) {
        int c = pt_leaf[p];
        double d[3] = {px[p] - cen[3 * c], py[p] - cen[3 * c + 1], pz[p] - cen[3 * c + 2]};
        float h[3], l[3];
        for (int k = 0; k < 3; k++) {
            h[k] = (float)d[k];
            l[k] = (float)(d[k] - (double)h[k]);
        }
        const float wh = (float)pw[p];
        rec4[p] = make_float4(h[0], h[1], h[2], wh);
        rec4lo[p] = make_float4(l[0], l[1], l[2], (float)(pw[p] - (double)wh));
    }
    if (rx) {
        rx[p] = px[p];
        ry[p] = py[p];
        rz[p] = pz[p];
        rw[p] = pw[p];
    }
}

// Proxy positions: Chebyshev points of the second kind cos(pi k / n) mapped
// to each approximated cluster's box (Section 5.2).  Index (k1 (n+1) + k2)(n+1) + k3.
__global__ void k_proxy_records(int nfar, const int* far_cl, int degree, int64_t n, const double* lo,
                                const double* hi, float4* rec4, double* rx, double* ry, double* rz)
{
    __shared__ double node[kMaxDegree + 1];
    int f = blockIdx.x;
    int c = far_cl[f];
    int m = degree + 1, P = m * m * m;
    if (threadIdx.x < m) node[threadIdx.x] = cos(M_PI * threadIdx.x / degree);
    __syncthreads();
    double cc[3], hh[3];
    for (int d = 0; d < 3; d++) {
        cc[d] = (lo[3 * c + d] + hi[3 * c + d]) * 0.5;
        hh[d] = (hi[3 * c + d] - lo[3 * c + d]) * 0.5;
    }
    for (int k = threadIdx.x; k < P; k += blockDim.x) {
        int k1 = k / (m * m), k2 = (k / m) % m, k3 = k % m;
        double s1 = node[k1], s2 = node[k2], s3 = node[k3];
        int64_t r = n + (int64_t)f * P + k;
        if (rec4) {
            // the float32 anterpolation interpolates on the float32-rounded
            // nodes; the proxies sit on exactly those nodes
            s1 = (double)(float)s1;
            s2 = (double)(float)s2;
            s3 = (double)(float)s3;
            rec4[r] = make_float4((float)(hh[0] * s1), (float)(hh[1] * s2), (float)(hh[2] * s3), 0.0f);
        }
        if (rx) {
            rx[r] = cc[0] + hh[0] * s1;
            ry[r] = cc[1] + hh[1] * s2;
            rz[r] = cc[2] + hh[2] * s3;
        }
    }
}

__global__ void k_check_finite(const double* a, int64_t n, int* bad)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n && !isfinite(a[i])) atomicOr(bad, 1);
}

inline int nblocks(int64_t n, int t) { return (int)((n + t - 1) / t); }

// Pinned host words for values read back, once per host thread; the device
// writes them itself (pinned memory is mapped), so there is no copy to wait for.
struct Host1 {
    int64_t* h = nullptr;
    Host1()
    {
        thread_local int64_t* buf = nullptr;
        if (!buf) TAGI_CUDA(cudaMallocHost(&buf, kReadMax * sizeof(int64_t)));
        h = buf;
    }
    // the values at the given device addresses into h[0], h[1], ...
    void read(cudaStream_t s, std::initializer_list<const int64_t*> p64, std::initializer_list<const int*> p32 = {})
    {
        ReadList L{};
        for (const int64_t* p : p64) L.p64[L.n++] = p;
        for (const int* p : p32) L.p32[L.n++] = p;
        launch(k_collect, 1, 32, 0, s, L, h);
        TAGI_LAUNCH_CHECK();
        TAGI_CUDA(cudaStreamSynchronize(s));
    }
};

}  // namespace

void exclusive_scan_i64(const int64_t* in, int64_t* out, int64_t n, cudaStream_t s)
{
    launch(k_scan_i64, 1, kScanThreads, 0, s, in, out, n);
    TAGI_LAUNCH_CHECK();
}

// Grow every per-cluster array to hold `cap` clusters, keeping contents.
static void grow_clusters(Tree& T, int cur, int cap, DevBuf& blo, DevBuf& bhi, cudaStream_t s)
{
    struct G {
        DevBuf* b;
        size_t per;
    } g[] = {{&T.cl_begin, 4},  {&T.cl_end, 4}, {&T.cl_parent, 4}, {&T.cl_level, 4}, {&T.cl_nchild, 4},
             {&T.cl_child, 32}, {&T.cl_lo, 24}, {&T.cl_hi, 24},     {&T.cl_cen, 24},  {&T.cl_rad, 8},
             {&blo, 24},        {&bhi, 24}};
    for (auto& x : g) {
        if (x.b->bytes >= x.per * (size_t)cap) continue;
        DevBuf nb;
        nb.ensure(x.per * (size_t)cap);
        if (x.b->p && cur > 0) TAGI_CUDA(cudaMemcpyAsync(nb.p, x.b->p, x.per * (size_t)cur, cudaMemcpyDeviceToDevice, s));
        *x.b = std::move(nb);  // the old block goes back to this stream's cache, behind the copy
    }
}

void build_tree(Tree& T, const double* xyz, const double* w)
{
    cudaStream_t s = T.stream;
    const int64_t n = T.n;
    TAGI_REQUIRE(n <= (int64_t)0x3fffffff, "n too large for 32-bit tree positions");
    Host1 H;
    // ---- input validation (non-finite coordinates or weights): flag[0], read
    // with the first level's result; flag[1]: partition consistency
    DevBuf flag;
    flag.ensure(64);
    TAGI_CUDA(cudaMemsetAsync(flag.p, 0, 64, s));
    launch(k_check_finite, nblocks(3 * n, 256), 256, 0, s, xyz, 3 * n, flag.as<int>());
    launch(k_check_finite, nblocks(n, 256), 256, 0, s, w, n, flag.as<int>());
    TAGI_LAUNCH_CHECK();

    DevBuf posA, posB, segA, segB, code, blo, bhi, mid, smask;
    posA.ensure(4 * n);
    posB.ensure(4 * n);
    segA.ensure(4 * n);
    segB.ensure(4 * n);
    const int64_t nblk = (n + kBlk - 1) / kBlk;
    code.ensure((size_t)nblk * kBlk);
    DevBuf bcnt, boff;
    bcnt.ensure(8 * 8 * nblk);
    boff.ensure(8 * (8 * nblk + 1));

    int cap = 1024;
    grow_clusters(T, 0, cap, blo, bhi, s);
    mid.ensure(24 * (size_t)cap);
    smask.ensure(4 * (size_t)cap);

    launch(k_init, nblocks(n, 256), 256, 0, s, posA.as<int>(), segA.as<int>(), n);
    launch(k_init_root, 1, 1, 0, s, (int)n, T.cl_begin.as<int>(), T.cl_end.as<int>(), T.cl_parent.as<int>(),
           T.cl_level.as<int>(), T.cl_nchild.as<int>(), blo.as<unsigned long long>(), bhi.as<unsigned long long>());
    TAGI_LAUNCH_CHECK();

    // One wait per level: the number of new clusters, which sizes the arrays
    // that the next kernels write and ends the loop when it is zero.
    int first = 0, last = 1, nc = 1, lvl = 0;
    DevBuf cnt, pfx, nnz, cbase, bfirst, bid;
    while (true) {
        const int nl = last - first;
        launch(k_bbox, nblocks(n, kBoxThreads), kBoxThreads, 0, s, posA.as<int>(), segA.as<int>(), xyz, n,
               blo.as<unsigned long long>(), bhi.as<unsigned long long>());
        launch(k_finalize, nblocks(nl, 128), 128, 0, s, first, last, blo.as<unsigned long long>(),
               bhi.as<unsigned long long>(), T.cl_begin.as<int>(), T.cl_end.as<int>(), T.leaf_size,
               T.cl_lo.as<double>(), T.cl_hi.as<double>(), T.cl_cen.as<double>(), T.cl_rad.as<double>(),
               mid.as<double>(), smask.as<int>());
        launch(k_codes, (int)nblk, kBlk, 0, s, posA.as<int>(), segA.as<int>(), xyz, n, smask.as<int>(),
               mid.as<double>(), code.as<signed char>(), nblk, bcnt.as<int64_t>());
        exclusive_scan_i64(bcnt.as<int64_t>(), boff.as<int64_t>(), 8 * nblk, s);
        cnt.ensure(32 * (size_t)nl);
        pfx.ensure(64 * (size_t)nl);
        nnz.ensure(8 * (size_t)nl);
        cbase.ensure(8 * ((size_t)nl + 1));
        bfirst.ensure(32 * (size_t)nl);
        bid.ensure(32 * (size_t)nl);
        launch(k_counts, nblocks(32 * (int64_t)nl, 128), 128, 0, s, first, last, T.cl_begin.as<int>(),
               T.cl_end.as<int>(), smask.as<int>(), code.as<signed char>(), boff.as<int64_t>(), nblk, cnt.as<int>(),
               pfx.as<int64_t>(), nnz.as<int64_t>());
        exclusive_scan_i64(nnz.as<int64_t>(), cbase.as<int64_t>(), nl, s);
        TAGI_LAUNCH_CHECK();
        H.read(s, {cbase.as<int64_t>() + nl}, {flag.as<int>(), flag.as<int>() + 1});
        TAGI_REQUIRE(H.h[1] == 0, "xyz or w holds a non-finite value");
        TAGI_REQUIRE(H.h[2] == 0, "tree partition consistency check failed");
        const int nnew = (int)H.h[0];
        if (nnew == 0) {
            // the last level are all leaves
            TAGI_CUDA(cudaMemsetAsync(T.cl_nchild.as<int>() + first, 0, 4 * (size_t)nl, s));
            break;
        }
        TAGI_REQUIRE(lvl < kMaxDepth, "tree deeper than 64 levels (degenerate point set)");
        if (nc + nnew > cap) {
            const int ncap = std::max(2 * cap, nc + nnew);
            grow_clusters(T, nc, ncap, blo, bhi, s);
            // both are written again for the next level before they are read
            mid.ensure(24 * (size_t)ncap);
            smask.ensure(4 * (size_t)ncap);
            cap = ncap;
        }
        launch(k_children, nblocks(nl, 128), 128, 0, s, first, last, nc, cbase.as<int64_t>(), T.cl_begin.as<int>(),
               cnt.as<int>(), lvl, T.cl_begin.as<int>(), T.cl_end.as<int>(), T.cl_parent.as<int>(),
               T.cl_level.as<int>(), T.cl_nchild.as<int>(), T.cl_child.as<int>(), bfirst.as<int>(), bid.as<int>(),
               blo.as<unsigned long long>(), bhi.as<unsigned long long>());
        launch(k_scatter, (int)nblk, kBlk, 0, s, posA.as<int>(), segA.as<int>(), code.as<signed char>(), n, nblk,
               boff.as<int64_t>(), first, pfx.as<int64_t>(), bfirst.as<int>(), bid.as<int>(), cnt.as<int>(),
               posB.as<int>(), segB.as<int>(), flag.as<int>() + 1);
        TAGI_LAUNCH_CHECK();
        std::swap(posA, posB);
        std::swap(segA, segB);
        first = nc;
        nc += nnew;
        last = nc;
        lvl++;
    }
    T.nc = nc;
    T.depth = lvl;

    // ---- points in tree order
    T.perm.ensure(4 * n);
    TAGI_CUDA(cudaMemcpyAsync(T.perm.p, posA.p, 4 * n, cudaMemcpyDeviceToDevice, s));
    T.px.ensure(8 * n);
    T.py.ensure(8 * n);
    T.pz.ensure(8 * n);
    T.pw.ensure(8 * n);
    launch(k_gather_points, nblocks(n, 256), 256, 0, s, posA.as<int>(), xyz, w, n, T.px.as<double>(), T.py.as<double>(),
                                                    T.pz.as<double>(), T.pw.as<double>());
    TAGI_LAUNCH_CHECK();
    posA.release();
    posB.release();
    segA.release();
    segB.release();
    code.release();
    bcnt.release();
    boff.release();
    blo.release();
    bhi.release();

    // ---- leaves (batches)
    DevBuf fl, fo;
    fl.ensure(8 * (size_t)nc);
    fo.ensure(8 * ((size_t)nc + 1));
    launch(k_is_leaf, nblocks(nc, 256), 256, 0, s, nc, T.cl_nchild.as<int>(), fl.as<int64_t>());
    exclusive_scan_i64(fl.as<int64_t>(), fo.as<int64_t>(), nc, s);
    H.read(s, {fo.as<int64_t>() + nc});
    T.nleaf = (int)H.h[0];
    T.leaves.ensure(4 * (size_t)T.nleaf);
    launch(k_compact, nblocks(nc, 256), 256, 0, s, nc, fl.as<int64_t>(), fo.as<int64_t>(), T.leaves.as<int>(), nullptr);
    T.pt_leaf.ensure(4 * n);
    launch(k_fill_leaf, T.nleaf, 256, 0, s, T.leaves.as<int>(), T.cl_begin.as<int>(), T.cl_end.as<int>(),
                                        T.pt_leaf.as<int>());
    TAGI_LAUNCH_CHECK();

    // ---- interaction lists (Algorithm 3, MAC of Eq. MAC)
    ListArgs la{T.cl_begin.as<int>(), T.cl_end.as<int>(),  T.cl_nchild.as<int>(), T.cl_child.as<int>(),
                T.pt_leaf.as<int>(),  T.leaves.as<int>(),   T.cl_cen.as<double>(), T.cl_rad.as<double>(),
                T.theta,              T.P};
    const int nleaf = T.nleaf;
    DevBuf lc, lo_, npair, fpair, err;
    lc.ensure(8 * (size_t)nleaf);
    lo_.ensure(8 * ((size_t)nleaf + 1));
    npair.ensure(8 * ((size_t)nleaf + 1));
    fpair.ensure(8 * ((size_t)nleaf + 1));
    err.ensure(16);
    TAGI_CUDA(cudaMemsetAsync(err.p, 0, 16, s));
    launch(k_list_count, nblocks(nleaf, kListWarps), 32 * kListWarps, 0, s, la, nleaf, lc.as<int64_t>(), npair.as<int64_t>(),
                                                   fpair.as<int64_t>(), err.as<int>());
    exclusive_scan_i64(lc.as<int64_t>(), lo_.as<int64_t>(), nleaf, s);
    TAGI_LAUNCH_CHECK();
    {
        DevBuf t1, t2;
        t1.ensure(8 * ((size_t)nleaf + 1));
        t2.ensure(8 * ((size_t)nleaf + 1));
        exclusive_scan_i64(npair.as<int64_t>(), t1.as<int64_t>(), nleaf, s);
        exclusive_scan_i64(fpair.as<int64_t>(), t2.as<int64_t>(), nleaf, s);
        H.read(s, {lo_.as<int64_t>() + nleaf, t1.as<int64_t>() + nleaf, t2.as<int64_t>() + nleaf}, {err.as<int>()});
        TAGI_REQUIRE(H.h[3] == 0, "interaction-list stack overflow");
        T.nent = H.h[0];
        T.near_pairs = H.h[1];
        T.far_pairs = H.h[2];
    }
    TAGI_REQUIRE(T.nent < (int64_t)0x7fffffff, "too many interaction entries");
    T.ent.ensure(sizeof(Entry) * (size_t)std::max<int64_t>(T.nent, 1));
    T.ent_batch.ensure(4 * (size_t)std::max<int64_t>(T.nent, 1));
    T.ent_clus.ensure(4 * (size_t)std::max<int64_t>(T.nent, 1));
    T.ent_off.ensure(8 * ((size_t)nleaf + 1));
    TAGI_CUDA(cudaMemcpyAsync(T.ent_off.p, lo_.p, 8 * ((size_t)nleaf + 1), cudaMemcpyDeviceToDevice, s));
    DevBuf isfar;
    isfar.ensure(4 * (size_t)nc);
    TAGI_CUDA(cudaMemsetAsync(isfar.p, 0, 4 * (size_t)nc, s));
    launch(k_list_fill, nblocks(nleaf, kListWarps), 32 * kListWarps, 0, s, la, nleaf, lo_.as<int64_t>(), T.ent.as<Entry>(),
                                                  T.ent_batch.as<int>(), T.ent_clus.as<int>(), isfar.as<int>(),
                                                  err.as<int>());
    TAGI_LAUNCH_CHECK();

    // ---- approximated clusters
    {
        DevBuf f64, o64, z64, zo;
        f64.ensure(8 * (size_t)nc);
        o64.ensure(8 * ((size_t)nc + 1));
        z64.ensure(8 * (size_t)nc);
        zo.ensure(8 * ((size_t)nc + 1));
        T.far_cl.ensure(4 * (size_t)nc);
        T.cl_far.ensure(4 * (size_t)nc);
        launch(k_far_flags, nblocks(nc, 256), 256, 0, s, nc, isfar.as<int>(), T.cl_begin.as<int>(), T.cl_end.as<int>(),
               f64.as<int64_t>(), z64.as<int64_t>());
        exclusive_scan_i64(f64.as<int64_t>(), o64.as<int64_t>(), nc, s);
        exclusive_scan_i64(z64.as<int64_t>(), zo.as<int64_t>(), nc, s);
        launch(k_compact, nblocks(nc, 256), 256, 0, s, nc, f64.as<int64_t>(), o64.as<int64_t>(), T.far_cl.as<int>(),
                                                   T.cl_far.as<int>());
        TAGI_LAUNCH_CHECK();
        // ant_points: sum of N_S over approximated clusters (anterpolation
        // work, reported by tagi_tree_info)
        H.read(s, {o64.as<int64_t>() + nc, zo.as<int64_t>() + nc}, {err.as<int>()});
        TAGI_REQUIRE(H.h[2] == 0, "interaction-list fill disagrees with its count");
        T.nfar = (int)H.h[0];
        T.ant_points = H.h[1];
    }
    T.nrec = n + (int64_t)T.nfar * T.P;
    TAGI_REQUIRE(T.nrec < (int64_t)0x7fffffff, "too many source records");
    if (T.nent > 0)
        launch(k_far_ranges, nblocks(T.nent, 256), 256, 0, s, T.nent, T.ent.as<Entry>(), T.cl_far.as<int>(), n, T.P);
    if (T.prec == TAGI_FP32C && T.nent > 0) {
        T.ent_shift.ensure(2 * sizeof(float4) * (size_t)T.nent);
        launch(k_entry_shift, nblocks(T.nent, 256), 256, 0, s, T.nent, T.ent.as<Entry>(), T.ent_batch.as<int>(),
               T.cl_cen.as<double>(), T.ent_shift.as<float4>());
    }
    DevBuf ng;
    ng.ensure(2 * sizeof(int64_t));
    TAGI_CUDA(cudaMemsetAsync(ng.p, 0, 2 * sizeof(int64_t), s));
    if (T.nent > 0)
        launch(k_gauss_flags, nblocks(T.nent, 256), 256, 0, s, T.nent, T.ent.as<Entry>(), T.ent_batch.as<int>(),
               T.ent_clus.as<int>(), T.cl_lo.as<double>(), T.cl_hi.as<double>(), T.cl_begin.as<int>(),
               T.cl_end.as<int>(), T.alpha, ng.as<unsigned long long>());
    TAGI_LAUNCH_CHECK();

    // ---- anterpolation items (counted here, with the work items)
    DevBuf ac, ao;
    ac.ensure(8 * (size_t)std::max(T.nfar, 1));
    ao.ensure(8 * ((size_t)T.nfar + 1));
    // shorter items until there are kAntItemsWanted (four waves of two CTAs on
    // 152 SMs): an item is a serial chain of point tiles
    T.ant_chunk = kAntChunk;
    while (T.ant_chunk > kAntChunkMin && T.ant_points / T.ant_chunk < kAntItemsWanted) T.ant_chunk /= 2;
    if (T.nfar > 0)
        launch(k_ant_counts, nblocks(T.nfar, 128), 128, 0, s, T.nfar, T.far_cl.as<int>(), T.cl_begin.as<int>(),
               T.cl_end.as<int>(), T.ant_chunk, ac.as<int64_t>());
    exclusive_scan_i64(ac.as<int64_t>(), ao.as<int64_t>(), T.nfar, s);
    TAGI_LAUNCH_CHECK();

    // ---- work items of the near/far kernel
    // Whole entries, the caller's number of sources an item or kSegment: the
    // order in which a target's two-float sums are added follows from the
    // segment and the list alone.  Where no number was given and kSegment leaves
    // fewer than kItemsFew items (1.3 waves of 152 SMs at the 10 CTAs of the
    // three-field kernel) the SMs would wait for a few long ones: there the
    // items are split until there are kItemsWanted.  The 5,003 point cube ran 64
    // CTAs over 5,003 sources each, 334 us a call at first, 82 split; the
    // uniform hydrogen mesh (400 items) 689 -> 446 us.
    const int64_t rows = (T.near_pairs + T.far_pairs) / kTargetsPerItem;
    int seg_src = T.segment ? T.segment : kSegment;
    T.split_items = T.segment == 0 && rows / seg_src < kItemsFew;
    if (T.split_items) {
        const int unit = std::max(kItemUnit, padded(T.P));  // no unit is longer than an item
        seg_src = (int)std::max<int64_t>(std::min<int64_t>(seg_src, rows / kItemsWanted), unit);
    }
    DevBuf nch, nit, choff, itoff;
    nch.ensure(8 * (size_t)nleaf);
    nit.ensure(8 * (size_t)nleaf);
    choff.ensure(8 * ((size_t)nleaf + 1));
    itoff.ensure(8 * ((size_t)nleaf + 1));
    launch(k_item_counts, nblocks(32 * (int64_t)nleaf, 128), 128, 0, s, nleaf, T.leaves.as<int>(), T.cl_begin.as<int>(),
                                                      T.cl_end.as<int>(), T.ent_off.as<int64_t>(), T.ent.as<Entry>(),
                                                      seg_src, T.split_items ? 1 : 0, nch.as<int64_t>(),
                                                      nit.as<int64_t>());
    exclusive_scan_i64(nch.as<int64_t>(), choff.as<int64_t>(), nleaf, s);
    exclusive_scan_i64(nit.as<int64_t>(), itoff.as<int64_t>(), nleaf, s);
    TAGI_LAUNCH_CHECK();
    H.read(s, {choff.as<int64_t>() + nleaf, itoff.as<int64_t>() + nleaf, ng.as<int64_t>(), ng.as<int64_t>() + 1,
               ao.as<int64_t>() + T.nfar});
    T.ntchunk = H.h[0];
    T.nitems = H.h[1];
    T.near_pairs_ng = H.h[2];
    T.far_pairs_ng = H.h[3];
    T.nant = H.h[4];
    T.items.ensure(sizeof(Item) * (size_t)std::max<int64_t>(T.nitems, 1));
    T.item_order.ensure(4 * (size_t)std::max<int64_t>(T.nitems, 1));
    T.tc_item0.ensure(4 * ((size_t)T.ntchunk + 1));
    T.tc_t0.ensure(4 * (size_t)T.ntchunk);
    T.tc_t1.ensure(4 * (size_t)T.ntchunk);
    T.tc_batch.ensure(4 * (size_t)T.ntchunk);
    launch(k_item_fill, nleaf, 128, 0, s, nleaf, T.leaves.as<int>(), T.cl_begin.as<int>(),
                                                    T.cl_end.as<int>(), T.ent_off.as<int64_t>(), T.ent.as<Entry>(),
                                                    seg_src, T.split_items ? 1 : 0, choff.as<int64_t>(),
                                                    itoff.as<int64_t>(),
                                                    T.items.as<Item>(), T.nitems, T.ntchunk,
                                                    T.item_order.as<int>(), T.tc_item0.as<int>(), T.tc_t0.as<int>(),
                                                    T.tc_t1.as<int>(), T.tc_batch.as<int>());
    TAGI_LAUNCH_CHECK();
    if (T.nfar > 0) {
        T.ant_items.ensure(sizeof(AntItem) * (size_t)T.nant);
        T.far_ant0.ensure(4 * ((size_t)T.nfar + 1));
        launch(k_ant_fill, nblocks(T.nfar + 1, 128), 128, 0, s, T.nfar, T.far_cl.as<int>(), T.cl_begin.as<int>(),
                                                            T.cl_end.as<int>(), T.ant_chunk, ao.as<int64_t>(),
                                                            T.ant_items.as<AntItem>(), T.far_ant0.as<int>());
        TAGI_LAUNCH_CHECK();
    }

    // ---- source records
    const bool fp32 = T.prec == TAGI_FP32C;
    if (fp32) {
        T.rec4.ensure(16 * (size_t)T.nrec);
        T.rec4lo.ensure(16 * (size_t)n);
    } else {
        T.rx.ensure(8 * (size_t)T.nrec);
        T.ry.ensure(8 * (size_t)T.nrec);
        T.rz.ensure(8 * (size_t)T.nrec);
        T.rw.ensure(8 * (size_t)T.nrec);
    }
    launch(k_point_records, nblocks(n, 256), 256, 0, s, 
        n, T.px.as<double>(), T.py.as<double>(), T.pz.as<double>(), T.pw.as<double>(), T.pt_leaf.as<int>(),
        T.cl_cen.as<double>(), fp32 ? T.rec4.as<float4>() : nullptr, fp32 ? T.rec4lo.as<float4>() : nullptr,
        fp32 ? nullptr : T.rx.as<double>(),
        fp32 ? nullptr : T.ry.as<double>(), fp32 ? nullptr : T.rz.as<double>(), fp32 ? nullptr : T.rw.as<double>());
    if (T.nfar > 0)
        launch(k_proxy_records, T.nfar, 256, 0, s, T.nfar, T.far_cl.as<int>(), T.degree, n, T.cl_lo.as<double>(),
                                               T.cl_hi.as<double>(), fp32 ? T.rec4.as<float4>() : nullptr,
                                               fp32 ? nullptr : T.rx.as<double>(), fp32 ? nullptr : T.ry.as<double>(),
                                               fp32 ? nullptr : T.rz.as<double>());
    TAGI_LAUNCH_CHECK();
    anterpolate_weights(T);
}

}  // namespace tagi
