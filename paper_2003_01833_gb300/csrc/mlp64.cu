// Warm-start MLP with H = 64 hidden units on the tensor cores: bfloat16
// operands, tcgen05.mma kind::f16 with float32 accumulation in tensor memory.
//
// Model (F = 8 features, two tanh layers of 64, one output), per point p:
//   z1 = W1 x + b1, h1 = tanh z1, z2 = W2 bf16(h1) + b2, h2 = tanh z2,
//   y = W3 . h2 + b3,
// with x, W1, W2, W3 in bfloat16 (rounded from the float64 master weights),
// b1, b2, b3 and every activation in float32; the input of the second layer
// is rounded to bfloat16 as the tensor cores take it.  Gradient of
// L = sum_p wt_p (y_p - t_p)^2:
//   dy = 2 wt (y - t), dz2 = dy W3 (1 - h2^2), dz1 = (bf16(dz2) W2)(1 - h1^2),
//   dW2 = sum bf16(dz2) bf16(h1)^T, db2 = sum bf16(dz2),
//   dW1 = sum bf16(dz1) x^T,        db1 = sum bf16(dz1),
//   dW3 = sum bf16(dy) bf16(h2),    db3 = sum bf16(dy).
//
// Tiles of 128 points; point p of a tile is TMEM lane p of the per-point
// products, and warpgroup g of a CTA's two handles hidden units [32 g, 32 g +
// 32) of every point (a warp reads its own 32-lane quarter of TMEM).  The
// products are
//   Z1 = X W1^T           (M 128 points, N 64, K 16: features padded)
//   Z2 = H1 W2^T          (M 128, N 64, K 64)
//   dH1 = dZ2 W2          (M 128, N 64, K 64)
// and the weight gradients contractions over the tile's points, accumulated
// in TMEM over up to kFold tiles:
//   D1 = [dZ2 dZ1]^T [H1 X 1]   (M 128 = 64 + 64, N 128 of which 73 are used, K 128)
//   D2 = [H2 X 1]^T dy          (M 128 of which 65 are used, N 16, K 128)
// then added to a float64 partial row in global memory.
//
// What bounds it: a tile is a chain of four products with the activations of
// 128 points between them, about 3,500 issue slots a scheduler (64 accurate
// tanh a unit pair), so the tensor pipe idles and latency shows.  Every
// activation is stored once, one 128-byte row of 64 units a point with the
// 128-byte swizzle, in 16-byte pieces: read along its rows it is the K-major A
// operand of the next product, read across (MN-major) the operand of the
// weight gradients, whose K are the points; W2 likewise serves Z2 and dH1.
// That takes 100 KB, so two CTAs share an SM and one computes while the other
// waits.  With transposed copies stored value by value (160 KB, one CTA of 512
// threads) a training step over 10.9M points took 4.63 ms, now 1.74 (131 and 49
// SM clocks a point), the same bits.
//
// The float32 sums in TMEM are those of one CTA per SM: virtual CTA v owns
// tiles v, v + V, ..., in groups of kFold, and the two CTAs of an SM's worth of
// work take its groups in turn (mlp64_plan).
//
// Every wait is bounded; one that gives up sets *err and the CTA returns after
// a bounded wait for its MMAs.
#include <cuda_runtime.h>

#include "bf16.cuh"
#include "mlp64.cuh"
#include "tagi_internal.cuh"
#include "tc.cuh"

namespace tagi {

namespace {

using namespace mlp64;
constexpr int kT = 128;        // points per tile
constexpr int kWG = 2;         // warpgroups per CTA
constexpr int kCB = 64 / kWG;  // hidden units per thread
constexpr int kThreads = kT * kWG;
constexpr int kFold = 8;       // tiles accumulated in tensor memory between float64 folds
constexpr long long kWait = 2000000000LL;

// byte layout of the shared memory (every tile 1024-aligned).  Point tiles:
// 128 rows x 128 B.
constexpr int kPointTile = 128 * 128;
constexpr int sDZ2 = 0;                  // bf16(dz2)
constexpr int sDZ1 = sDZ2 + kPointTile;  // bf16(dz1)
constexpr int sH2 = sDZ1 + kPointTile;   // bf16(h2)
constexpr int sB2 = sH2 + kPointTile;    // 2 tiles of 16 rows ([dy; 0]) x 64 points
constexpr int sFwd = sB2 + 2 * 16 * 128; // from here on: what the forward pass needs
constexpr int sH1 = sFwd;                // bf16(h1)
constexpr int sX = sH1 + kPointTile;     // features 0..7, 1, zeros
constexpr int sW1 = sX + kPointTile;     // 64 rows (units) x 128 B: W1 row, zeros
constexpr int sW2 = sW1 + 64 * 128;      // 64 rows (out j) x 64 (in i)
constexpr int kSmem = sW2 + 64 * 128;
static_assert(sFwd % 1024 == 0, "tiles are 1024-aligned");
// TMEM columns
constexpr uint32_t cZ = 0, cD1 = 64, cD2 = 192;

__device__ __forceinline__ uint32_t swz2(int r, int k)  // bf16 element k of row r, 128B swizzle
{
    return r * 128 + ((((k >> 3) ^ (r & 7))) << 4) + ((k & 7) << 1);
}

__device__ __forceinline__ void st16(uint8_t* sm, uint32_t off, uint16_t v) { *reinterpret_cast<uint16_t*>(sm + off) = v; }

// units [c0, c0 + N) of row r, rounded to bfloat16
template <int N>
__device__ __forceinline__ void store_row(uint8_t* tile, int r, int c0, const float (&v)[N])
{
#pragma unroll
    for (int c = 0; c < N; c += 8)
        *reinterpret_cast<uint4*>(tile + swz2(r, c0 + c)) =
            make_uint4(bf16x2(v[c], v[c + 1]), bf16x2(v[c + 2], v[c + 3]), bf16x2(v[c + 4], v[c + 5]),
                       bf16x2(v[c + 6], v[c + 7]));
}

struct __align__(16) Bias {
    float b1[kH], b2[kH], w3[kH], b3;
};

// 16 consecutive values from shared memory, four a load (all lanes of a warp
// read the same ones; one by one they were a tenth of a tile's instructions)
__device__ __forceinline__ void load16(const float* p, float (&v)[16])
{
#pragma unroll
    for (int c = 0; c < 16; c += 4) {
        const float4 t = *reinterpret_cast<const float4*>(p + c);
        v[c] = t.x;
        v[c + 1] = t.y;
        v[c + 2] = t.z;
        v[c + 3] = t.w;
    }
}

// MMAs of one stage, issued by thread 0, then all threads wait for them
struct Sync {
    uint64_t* bar;
    uint32_t phase;
    bool ok;
    __device__ void wait()
    {
        if (ok && !tc::mbar_wait(bar, phase, kWait)) ok = false;
        phase ^= 1;
        tc::fence_after_sync();
    }
};

// After a wait that gave up, thread 0: flag it, and wait (bounded) for every
// MMA it has issued, whichever commits they belong to
__device__ __noinline__ void give_up(uint64_t* drained, int* err)
{
    atomicOr(err, 1);
    tc::commit(drained);
    tc::mbar_wait(drained, 0, kWait);
}

// A and B K-major, `ksteps` K-steps of 16 from the start of a row
__device__ __forceinline__ void mma_chain(uint32_t d, uint32_t a, uint32_t b, int ksteps, uint32_t idesc)
{
    const uint64_t da = tc::sdesc_sw128(a), db = tc::sdesc_sw128(b);
    for (int k = 0; k < ksteps; k++) tc::mma_bf16(d, da + 2 * k, db + 2 * k, idesc, k > 0 ? 1u : 0u);
}

// the thread's place: point (TMEM lane) pl of the tile, hidden units
// [c0, c0 + kCB) of warpgroup g
struct Who {
    int t, pl, g, c0;
    uint32_t lane_base;
    __device__ explicit Who(uint32_t tmem)
    {
        t = threadIdx.x;
        pl = t & (kT - 1);
        g = t / kT;
        c0 = g * kCB;
        lane_base = tmem + ((uint32_t)((pl >> 5) * 32) << 16);
    }
};

// Weights (bf16 operand tiles) and float32 biases from the float64 master
// weights; zero the operand tiles from byte `from` on; the column of ones.
__device__ void setup(uint8_t* sm, int from, Bias* B, const double* __restrict__ master)
{
    for (int e = from / 16 + threadIdx.x; e < kSmem / 16; e += kThreads)
        reinterpret_cast<uint4*>(sm)[e] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    for (int e = threadIdx.x; e < kH * kF; e += kThreads)
        st16(sm, sW1 + swz2(e / kF, e % kF), bf16_of_double(master[oW1 + e]));
    for (int e = threadIdx.x; e < kH * kH; e += kThreads)
        st16(sm, sW2 + swz2(e / kH, e % kH), bf16_of_double(master[oW2 + e]));
    for (int e = threadIdx.x; e < kH; e += kThreads) {
        B->b1[e] = (float)master[oB1 + e];
        B->b2[e] = (float)master[oB2 + e];
        B->w3[e] = bf16_float(bf16_of_double(master[oW3 + e]));
    }
    if (threadIdx.x == 0) B->b3 = (float)master[oB3];
    // W1's column 8 is zero, so the ones do not enter Z1
    for (int e = threadIdx.x; e < kT; e += kThreads) st16(sm, sX + swz2(e, kF), 0x3F80);
}

// tanh(z + b) of this thread's units of the product in TMEM column cZ
__device__ __forceinline__ void activate(const Who& w, const float* b, float (&h)[kCB])
{
#pragma unroll
    for (int c = 0; c < kCB; c += 16) {
        float v[16], bc[16];
        load16(b + w.c0 + c, bc);
        tc::tmem_ld16(w.lane_base + cZ + w.c0 + c, v);
#pragma unroll
        for (int i = 0; i < 16; i++) h[c + i] = tanhf(v[i] + bc[i]);
    }
}

// Forward pass of point pl of the tile whose features xv (warpgroup 0) holds:
// y.  Returns false, in all threads, if a wait of any thread gave up before this
// tile; callers leave their loops on that alone, since sy.ok, the thread's own,
// may differ between threads from the tile's first wait on.  h1, h2: this
// thread's activations (float32).  ypart: [4][kT] shared partial sums of W3 . h2
// over 16 units each, added in unit order.
__device__ bool forward_tile(uint8_t* sm, const Bias& B, uint4 xv, const Who& w, uint32_t tmem, Sync& sy,
                             float* ypart, float (&h1)[kCB], float (&h2)[kCB], float& y)
{
    if (w.g == 0) *reinterpret_cast<uint4*>(sm + sX + swz2(w.pl, 0)) = xv;
    tc::fence_async_smem();
    tc::fence_before_sync();
    sy.ok = __syncthreads_and(sy.ok);
    if (!sy.ok) return false;
    if (w.t == 0) {
        tc::fence_after_sync();
        mma_chain(tmem + cZ, tc::smem_u32(sm + sX), tc::smem_u32(sm + sW1), 1, tc::idesc_bf16(128, 64));
        tc::commit(sy.bar);
    }
    sy.wait();
    activate(w, B.b1, h1);
    store_row<kCB>(sm + sH1, w.pl, w.c0, h1);
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    if (w.t == 0) {
        tc::fence_after_sync();
        mma_chain(tmem + cZ, tc::smem_u32(sm + sH1), tc::smem_u32(sm + sW2), 4, tc::idesc_bf16(128, 64));
        tc::commit(sy.bar);
    }
    sy.wait();
    activate(w, B.b2, h2);
#pragma unroll
    for (int c = 0; c < kCB; c += 16) {
        float yp = 0.0f, w3[16];
        load16(B.w3 + w.c0 + c, w3);
#pragma unroll
        for (int i = 0; i < 16; i++) yp = fmaf(w3[i], h2[c + i], yp);
        ypart[(w.c0 + c) / 16 * kT + w.pl] = yp;
    }
    tc::fence_before_sync();
    __syncthreads();
    y = B.b3;
#pragma unroll
    for (int q = 0; q < 4; q++) y += ypart[q * kT + w.pl];
    return true;
}

// features of point p (zeros beyond n)
__device__ __forceinline__ uint4 load_features(const uint16_t* __restrict__ feat, int64_t p, int64_t n)
{
    return p < n ? *reinterpret_cast<const uint4*>(feat + p * kF) : make_uint4(0, 0, 0, 0);
}

constexpr uint32_t kColsFwd = 64, kColsGrad = 256;

// dynamic shared memory: the tiles from sFwd on (four CTAs of 48 KB fit an SM;
// 4 x 64 TMEM columns)
__global__ void __launch_bounds__(kThreads, 2) k_mlp64_fwd(const uint16_t* __restrict__ feat, int64_t n,
                                                           const double* __restrict__ master, float* __restrict__ y,
                                                           int* __restrict__ err)
{
    extern __shared__ uint8_t raw[];
    uint8_t* sm =
        reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023)) - sFwd;
    __shared__ Bias B;
    __shared__ uint64_t bar, drained;
    __shared__ uint32_t slot;
    __shared__ float ypart[4 * kT];
    const int t = threadIdx.x;
    setup(sm, sFwd, &B, master);
    if ((t >> 5) == 0) tc::tmem_alloc(&slot, kColsFwd);
    if (t == 0) {
        tc::mbar_init(&bar, 1);
        tc::mbar_init(&drained, 1);
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = slot;
    const Who w(tmem);
    Sync sy{&bar, 0, true};
    const int64_t ntiles = (n + kT - 1) / kT;
    uint4 next = make_uint4(0, 0, 0, 0);
    if (w.g == 0) next = load_features(feat, (int64_t)blockIdx.x * kT + w.pl, n);
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t p = tile * kT + w.pl;
        const uint4 xv = next;
        if (w.g == 0) next = load_features(feat, p + (int64_t)gridDim.x * kT, n);
        float h1[kCB], h2[kCB], out;
        if (!forward_tile(sm, B, xv, w, tmem, sy, ypart, h1, h2, out)) break;
        if (w.g == 0 && p < n) y[p] = out;
    }
    if (!__syncthreads_and(sy.ok) && t == 0) give_up(&drained, err);
    tc::fence_before_sync();
    __syncthreads();
    if ((t >> 5) == 0) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, kColsFwd);
    }
}

// partial[blockIdx.x][kParams + 1]: this CTA's gradient sums and loss (in the
// order of mlp64.cuh).  Block b works for virtual CTA b % V of V, on its groups of
// kFold tiles b / V, b / V + gridDim.x / V, ...
__global__ void __launch_bounds__(kThreads, 2) k_mlp64_grad(const uint16_t* __restrict__ feat,
                                                            const float* __restrict__ target,
                                                            const float* __restrict__ wt, int64_t n,
                                                            const double* __restrict__ master,
                                                            double* __restrict__ partial, int V, int* __restrict__ err)
{
    extern __shared__ uint8_t raw[];
    uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
    __shared__ Bias B;
    __shared__ uint64_t bar, drained;
    __shared__ uint32_t slot;
    __shared__ float ypart[4 * kT];
    __shared__ double lsum[kT];
    const int t = threadIdx.x;
    double* out = partial + (size_t)blockIdx.x * (kParams + 1);
    for (int e = t; e <= kParams; e += kThreads) out[e] = 0.0;
    setup(sm, 0, &B, master);
    if ((t >> 5) == 0) tc::tmem_alloc(&slot, kColsGrad);
    if (t == 0) {
        tc::mbar_init(&bar, 1);
        tc::mbar_init(&drained, 1);
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = slot;
    const Who w(tmem);
    Sync sy{&bar, 0, true};
    double loss = 0.0;
    const int64_t ntiles = (n + kT - 1) / kT;
    const int vcta = blockIdx.x % V, split = gridDim.x / V;
    // tiles vcta, vcta + V, ... of the virtual CTA
    const int64_t mine = ntiles > vcta ? (ntiles - 1 - vcta) / V + 1 : 0;

    // TMEM lane r of D1 and D2 into the partial row; every entry has one writer
    auto fold = [&]() {
        const int r = w.pl;
        if (r < 64) {
#pragma unroll 1
            for (int c = w.g * 16; c < 64; c += 16 * kWG) {
                float v[16];
                double s[16];
#pragma unroll
                for (int i = 0; i < 16; i++) s[i] = out[pW2 + (c + i) * kH + r];
                tc::tmem_ld16(w.lane_base + cD1 + c, v);
#pragma unroll
                for (int i = 0; i < 16; i++) out[pW2 + (c + i) * kH + r] = s[i] + (double)v[i];
            }
        }
        float v[16];  // columns 64..71: W1, 72: the biases
        tc::tmem_ld16(w.lane_base + cD1 + 64, v);
        if (w.g == 0) {
            if (r < 64) {
                out[pB2 + r] += (double)v[8];
            } else {
#pragma unroll
                for (int f = 0; f < kF; f++) out[pW1 + f * kH + r - 64] += (double)v[f];
                out[pB1 + r - 64] += (double)v[8];
            }
        } else {
            float d[8];
            tc::tmem_ld8(w.lane_base + cD2, d);
            if (r < 64) out[pW3 + r] += (double)d[0];
            if (r == 64 + kF) out[pB3] += (double)d[0];  // the column of ones
        }
    };

    // the k-th tile of the virtual CTA after k in this CTA's order
    auto after = [&](int64_t k) { return (k % kFold) == kFold - 1 ? k + 1 + (int64_t)(split - 1) * kFold : k + 1; };
    int64_t k = (int64_t)(blockIdx.x / V) * kFold;
    uint4 nx = make_uint4(0, 0, 0, 0);
    float nt = 0.0f, nw = 0.0f;
    auto load = [&](int64_t kk) {
        const int64_t p = (vcta + kk * V) * kT + w.pl;
        const bool valid = kk < mine && p < n;
        if (w.g == 0) nx = load_features(feat, valid ? p : n, n);
        nt = valid ? target[p] : 0.0f;
        nw = valid ? wt[p] : 0.0f;
    };
    load(k);
    while (k < mine) {
        const int64_t p = (vcta + k * V) * kT + w.pl;
        const uint4 xv = nx;
        const float tv = nt, wv = nw;
        const int64_t knext = after(k);
        load(knext);
        float h1[kCB], h2[kCB], yv;
        if (!forward_tile(sm, B, xv, w, tmem, sy, ypart, h1, h2, yv)) break;
        const float r = p < n ? yv - tv : 0.0f;
        if (w.g == 0) loss += (double)wv * (double)r * (double)r;
        const float dy = 2.0f * wv * r;
        // h2 and dz2 = dy W3 (1 - h2^2)
        store_row<kCB>(sm + sH2, w.pl, w.c0, h2);
#pragma unroll
        for (int c = 0; c < kCB; c += 16) {
            float w3[16];
            load16(B.w3 + w.c0 + c, w3);
#pragma unroll
            for (int i = 0; i < 16; i++) h2[c + i] = dy * w3[i] * (1.0f - h2[c + i] * h2[c + i]);
        }
        store_row<kCB>(sm + sDZ2, w.pl, w.c0, h2);
        if (w.g == 0)
            st16(sm, sB2 + (w.pl >> 6) * 16 * 128 + swz2(0, w.pl & 63), (uint16_t)(bf16x2(dy, 0.0f) & 0xFFFFu));
        tc::fence_async_smem();
        tc::fence_before_sync();
        __syncthreads();
        if (w.t == 0) {
            tc::fence_after_sync();
            const uint64_t da = tc::sdesc_sw128(tc::smem_u32(sm + sDZ2));
            const uint64_t db = tc::sdesc_mn_sw128(tc::smem_u32(sm + sW2), 0);
#pragma unroll
            for (int q = 0; q < 4; q++)  // 16 rows j of W2 a step
                tc::mma_bf16(tmem + cZ, da + 2 * q, db + 128 * q, tc::idesc_bf16(128, 64, false, true), q > 0);
            tc::commit(sy.bar);
        }
        sy.wait();
        // dz1 = dh1 (1 - h1^2)
#pragma unroll
        for (int c = 0; c < kCB; c += 16) {
            float a[16];
            tc::tmem_ld16(w.lane_base + cZ + w.c0 + c, a);
#pragma unroll
            for (int i = 0; i < 16; i++) h1[c + i] = a[i] * (1.0f - h1[c + i] * h1[c + i]);
        }
        store_row<kCB>(sm + sDZ1, w.pl, w.c0, h1);
        tc::fence_async_smem();
        tc::fence_before_sync();
        __syncthreads();
        if (w.t == 0) {
            tc::fence_after_sync();
            const bool acc = (k % kFold) != 0;
            const uint64_t a1 = tc::sdesc_mn_sw128(tc::smem_u32(sm + sDZ2), sDZ1 - sDZ2);
            const uint64_t b1 = tc::sdesc_mn_sw128(tc::smem_u32(sm + sH1), sX - sH1);
            const uint64_t a2 = tc::sdesc_mn_sw128(tc::smem_u32(sm + sH2), sX - sH2);
            const uint64_t b2 = tc::sdesc_sw128(tc::smem_u32(sm + sB2));
            // K = 128 points, 16 rows of the point tiles a step; dy: two tiles of 64
#pragma unroll
            for (int q = 0; q < 8; q++)
                tc::mma_bf16(tmem + cD1, a1 + 128 * q, b1 + 128 * q, tc::idesc_bf16(128, 128, true, true),
                             q > 0 || acc);
#pragma unroll
            for (int q = 0; q < 8; q++)
                tc::mma_bf16(tmem + cD2, a2 + 128 * q, b2 + 128 * (q >> 2) + 2 * (q & 3),
                             tc::idesc_bf16(128, 16, true, false), q > 0 || acc);
            tc::commit(sy.bar);
        }
        // the next tile rewrites these operand tiles: wait here
        sy.wait();
        if ((k % kFold) == kFold - 1 || k == mine - 1) fold();
        tc::fence_before_sync();
        k = knext;
    }
    if (w.g == 0) lsum[w.pl] = loss;
    const bool ok = __syncthreads_and(sy.ok);
    if (!ok && t == 0) give_up(&drained, err);
    if (ok && t == 0) {
        double s = 0.0;
        for (int q = 0; q < kT; q++) s += lsum[q];
        out[pLoss] = s;
    }
    tc::fence_before_sync();
    __syncthreads();
    if ((t >> 5) == 0) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, kColsGrad);
    }
}

template <class K>
void allow_smem(K kern, int bytes, bool (&set)[64])
{
    int dev = 0;
    TAGI_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64 || !set[dev]) {
        TAGI_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
        if (dev >= 0 && dev < 64) set[dev] = true;
    }
}

}  // namespace

int mlp64_params() { return kParams; }

// y[n] of the network.  err: device int.
void mlp64_forward(const uint16_t* feat, int64_t n, const double* master, float* y, int* err, int sms, cudaStream_t s)
{
    static bool set[64] = {};
    const int smem = kSmem - sFwd + 1024;
    allow_smem(k_mlp64_fwd, smem, set);
    const int64_t tiles = (n + kT - 1) / kT;
    const int64_t most = 2LL * sms;
    launch(k_mlp64_fwd, (int)(tiles < most ? tiles : most), kThreads, smem, s, feat, n, master, y, err);
    TAGI_LAUNCH_CHECK();
}

// Virtual CTAs (one per SM) and CTAs that share each one's groups of kFold
// tiles: two where it has more than one group.
static void mlp64_plan(int64_t n, int sms, int* virt, int* split)
{
    const int64_t tiles = (n + kT - 1) / kT;
    *virt = (int)(tiles < sms ? tiles : sms);
    *split = (tiles + *virt - 1) / *virt > kFold ? 2 : 1;
}

int mlp64_grad_grid(int64_t n, int sms)
{
    int v, split;
    mlp64_plan(n, sms, &v, &split);
    return v * split;
}

// per-CTA gradient partials [mlp64_grad_grid][kParams + 1]
void mlp64_gradient(const uint16_t* feat, const float* target, const float* wt, int64_t n, const double* master,
                    double* partial, int sms, int* err, cudaStream_t s)
{
    static bool set[64] = {};
    allow_smem(k_mlp64_grad, kSmem + 1024, set);
    int v, split;
    mlp64_plan(n, sms, &v, &split);
    launch(k_mlp64_grad, v * split, kThreads, kSmem + 1024, s, feat, target, wt, n, master, partial, v, err);
    TAGI_LAUNCH_CHECK();
}

}  // namespace tagi
