// Learned warm start for SCF runs of molecules: point features, a per-point
// MLP (F = 8 inputs, two tanh layers of H = 32 here, one output), its
// gradient and Adam.  The H = 64 network runs on the tensor cores
// (mlp64.cu); this file holds the entry points of both.  Weights enter the products rounded to bfloat16 and features are
// stored as bfloat16; the arithmetic of a point is float32, gradients are
// accumulated over points in float64 in a fixed order (deterministic for a
// given device), and Adam keeps float64 master weights.
//
// Not a method of the paper: its SCF runs start from superposed atomic data
// (Section 6).  The model predicts a relative correction y of the normalised
// superposition start s, psi = s (1 + y).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>

#include "bf16.cuh"
#include "mlp64.cuh"
#include "pair64.cuh"
#include "tagi_internal.cuh"

namespace tagi {
namespace {

constexpr int kF = 8;
constexpr int kH = 32;
constexpr int oW1 = 0, oB1 = kH * kF, oW2 = oB1 + kH, oB2 = oW2 + kH * kH, oW3 = oB2 + kH, oB3 = oW3 + kH;
constexpr int kP = oB3 + 1;  // 1377 parameters
constexpr int kPPad = 1380;  // float slots of the weights in shared memory (keeps the stash 16-byte aligned)
constexpr int kThreads = 128;
// Stash row of one point for the gradient reduction: x | h1 | h2 | dz1 | dz2 |
// dy | 1.  Written four values at a time: a stride of 35 16-byte words keeps
// eight rows in different banks.
constexpr int cX = 0, cH1 = 8, cH2 = 40, cD1 = 72, cD2 = 104, cDy = 136, cOne = 137, kStride = 140;
// Gradient entries per thread: a 2 x 4 tile of W2 (rows j0, j0+1; columns
// i0..i0+3), two entries of one row of W1, and one of the other 97 (b1, b2, W3,
// b3): six shared loads per point for its eleven products.
constexpr int kRest = 3 * kH + 1;
static_assert(kThreads == (kH / 2) * (kH / 4) && kH * kF == 2 * kThreads && kRest <= kThreads, "entries per thread");
constexpr int kMaxNuclei = 16;
constexpr size_t kGradSmem = sizeof(float) * (kPPad + (size_t)kThreads * kStride);

struct Nuclei {
    double x[kMaxNuclei], y[kMaxNuclei], z[kMaxNuclei];
    double zs[kMaxNuclei];  // decay rate of each nucleus's exponential features (1 by default)
    int m;
    int ordered;  // 1: two nuclei taken in list order (r1 to the first) instead of by distance
};

__device__ __forceinline__ bool is_weight(int e)
{
    return (e >= oW1 && e < oB1) || (e >= oW2 && e < oB2) || (e >= oW3 && e < oB3);
}

// Weights rounded to bfloat16, biases as float32, into shared memory.
__device__ __forceinline__ void load_params(float* sw, const double* __restrict__ master)
{
    for (int e = threadIdx.x; e < kP; e += blockDim.x)
        sw[e] = is_weight(e) ? bf16_float(bf16_of_double(master[e])) : (float)master[e];
}

__device__ __forceinline__ void load_x(const uint16_t* __restrict__ feat, int64_t i, float x[kF])
{
    const uint4 v = *reinterpret_cast<const uint4*>(feat + i * kF);
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < 4; k++) {
        x[2 * k] = bf16_float(u[k] & 0xFFFFu);
        x[2 * k + 1] = bf16_float(u[k] >> 16);
    }
}

// Weights are read from shared memory four at a time (the same address for
// the whole warp): one by one these reads, not the products, set the pace.
__device__ __forceinline__ void weights4(const float* w, float (&v)[4])
{
    const float4 t = *reinterpret_cast<const float4*>(w);
    v[0] = t.x;
    v[1] = t.y;
    v[2] = t.z;
    v[3] = t.w;
}

__device__ __forceinline__ void layer1(const float* sw, const float x[kF], float h1[kH])
{
#pragma unroll
    for (int i = 0; i < kH; i++) {
        float z = sw[oB1 + i];
#pragma unroll
        for (int f = 0; f < kF; f += 4) {
            float w[4];
            weights4(sw + oW1 + i * kF + f, w);
#pragma unroll
            for (int c = 0; c < 4; c++) z = fmaf(w[c], x[f + c], z);
        }
        h1[i] = tanhf(z);
    }
}

__device__ __forceinline__ float layer2_unit(const float* sw, const float h1[kH], int j)
{
    float z = sw[oB2 + j];
#pragma unroll
    for (int i = 0; i < kH; i += 4) {
        float w[4];
        weights4(sw + oW2 + j * kH + i, w);
#pragma unroll
        for (int c = 0; c < 4; c++) z = fmaf(w[c], h1[i + c], z);
    }
    return tanhf(z);
}

// ------------------------------------------------------------------ kernels
// Features of a point (float64, rounded once to bfloat16): with r1 <= r2 the
// distances to the two nearest nuclei (the lower index first on ties), z1
// and z2 those nuclei's decay rates (1 unless given) and R their
// separation, [e^-(z1 r1), e^-(z2 r2), tanh r1, tanh r2, (r2 - r1)/R,
// tanh((r1 + r2)/R - 1), R - 1.5, e^-(r1 + r2 - R)].  Sums of squares are
// formed left to right without contraction.
//
// Only 8 bits of each value are kept, and float64 runs at 1/73 of the float32
// rate here: the distances are float64 (pair64.cuh's root), the exponentials
// and tangents float32 with a bound on their relative error.  A value whose
// bound reaches a rounding boundary of bfloat16 (one in a thousand) is
// evaluated again in float64, a point whose distances tie or cancel to within
// rounding takes the float64 form throughout (features_exact), so the bits
// are those of the float64 form.  192,000 points take 22 us, 130 in float64 alone.
struct Pair {
    double R, invR;
    uint16_t f6;
};

__device__ __forceinline__ double distance2(const Nuclei& nuc, int a, double px, double py, double pz)
{
    const double dx = px - nuc.x[a], dy = py - nuc.y[a], dz = pz - nuc.z[a];
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

__device__ __forceinline__ double separation(const Nuclei& nuc, int a1, int a2)
{
    return sqrt(distance2(nuc, a2, nuc.x[a1], nuc.y[a1], nuc.z[a1]));
}

__device__ __noinline__ uint4 features_exact(const Nuclei& nuc, double px, double py, double pz)
{
    double d1 = INFINITY, d2 = INFINITY;
    int a1 = 0, a2 = 1;
    for (int a = 0; a < (nuc.ordered ? 0 : nuc.m); a++) {
        const double d = sqrt(distance2(nuc, a, px, py, pz));
        if (d < d1) {
            d2 = d1;
            a2 = a1;
            d1 = d;
            a1 = a;
        } else if (d < d2) {
            d2 = d;
            a2 = a;
        }
    }
    if (nuc.ordered) {
        d1 = sqrt(distance2(nuc, 0, px, py, pz));
        d2 = sqrt(distance2(nuc, 1, px, py, pz));
    }
    const double R = separation(nuc, a1, a2);
    const double s12 = __dadd_rn(d1, d2);
    const double f[kF] = {exp(-__dmul_rn(nuc.zs[a1], d1)),
                          exp(-__dmul_rn(nuc.zs[a2], d2)),
                          tanh(d1),
                          tanh(d2),
                          __dsub_rn(d2, d1) / R,
                          tanh(__dsub_rn(s12 / R, 1.0)),
                          __dsub_rn(R, 1.5),
                          exp(-__dsub_rn(s12, R))};
    uint32_t u[4];
#pragma unroll
    for (int k = 0; k < 4; k++)
        u[k] = (uint32_t)bf16_of_double(f[2 * k]) | ((uint32_t)bf16_of_double(f[2 * k + 1]) << 16);
    return make_uint4(u[0], u[1], u[2], u[3]);
}

// bfloat16 of a float32 in normal range, if `units` of its last place do not
// reach a rounding boundary
__device__ __forceinline__ bool round_safe(float v, float units, uint32_t& b)
{
    const uint32_t u = __float_as_uint(v);
    b = (u + 0x8000u) >> 16;
    return (float)abs((int)(u & 0xffffu) - 0x8000) > units + 1.0f;
}

__device__ __noinline__ uint32_t exp_exact(double x) { return bf16_of_double(exp(-x)); }
__device__ __noinline__ uint32_t tanh_exact(double x) { return bf16_of_double(tanh(x)); }

// e^-x, x to 2^-22: float32 argument and product within x 2^-22, expf within
// 2^-21 (units of the last place are at most 2^-24 of the value each)
__device__ __forceinline__ uint32_t exp_bits(double x)
{
    const float xf = (float)x;
    if (xf >= 94.0f) return 0;  // below half the least bfloat16, 2^-133
    uint32_t b;
    if (xf < 69.0f && round_safe(expf(-xf), 8.0f + 4.0f * fabsf(xf), b)) return b;
    return exp_exact(x);
}

// tanh x, x to 2^-22: tanhf within 2^-22, tanh no steeper than x relatively
__device__ __forceinline__ uint32_t tanh_bits(double x)
{
    uint32_t b;
    const float xf = (float)x;
    if (fabsf(xf) > 1e-30f && round_safe(tanhf(xf), 16.0f, b)) return b;
    return tanh_exact(x);
}

__global__ void __launch_bounds__(256) k_features(const double* __restrict__ xyz, int64_t n,
                                                  const __grid_constant__ Nuclei nuc, uint16_t* __restrict__ feat)
{
    __shared__ Pair pairs[kMaxNuclei * kMaxNuclei];
    for (int q = threadIdx.x; q < nuc.m * nuc.m; q += blockDim.x) {
        const double R = separation(nuc, q / nuc.m, q % nuc.m);
        pairs[q] = Pair{R, 1.0 / R, bf16_of_double(__dsub_rn(R, 1.5))};
    }
    __syncthreads();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double px = xyz[i], py = xyz[n + i], pz = xyz[2 * n + i];
    // the two nearest by squared distance (positive float64 compare as
    // integers); squares a few units apart may have equal roots: not safe
    long long q1 = 0x7ff0000000000000ll, q2 = q1;
    int a1 = 0, a2 = 1;
    bool safe = true;
    if (nuc.ordered) {
        q1 = __double_as_longlong(distance2(nuc, 0, px, py, pz));
        q2 = __double_as_longlong(distance2(nuc, 1, px, py, pz));
    } else {
        for (int a = 0; a < nuc.m; a++) {
            const long long q = __double_as_longlong(distance2(nuc, a, px, py, pz));
            safe = safe && (q == q1 || llabs(q - q1) > 8) && (q == q2 || llabs(q - q2) > 8);
            if (q < q1) {
                q2 = q1;
                a2 = a1;
                q1 = q;
                a1 = a;
            } else if (q < q2) {
                q2 = q;
                a2 = a;
            }
        }
    }
    const double r21 = __longlong_as_double(q1), r22 = __longlong_as_double(q2);
    uint4 out = make_uint4(0, 0, 0, 0);
    safe = safe && p64::fast_range(r21) && p64::fast_range(r22);
    if (safe) {
        const Pair pr = pairs[a1 * nuc.m + a2];
        double ri, d1, d2;
        p64::inv_sqrt(r21, ri, d1);
        p64::inv_sqrt(r22, ri, d2);
        const double s12 = d1 + d2, diff = d2 - d1, x5 = fma(s12, pr.invR, -1.0);
        const double f4 = diff * pr.invR;
        // the roots are within 2^-51 of their values: not safe where the
        // difference cancels below 2^-26 of them, or where f4 is as near a
        // rounding boundary (the middle of its 45 dropped bits) as the
        // cancellation has left it exact
        const long long b4 = __double_as_longlong(f4);
        const float s32 = (float)s12, rest = fabsf((float)diff);
        safe = fabsf((float)x5) > 1.5e-8f &&
               (q1 == q2 || (rest > 1.5e-8f * s32 &&
                             (float)llabs((b4 & 0x1fffffffffffll) - 0x100000000000ll) > 64.0f + 8.0f * s32 / rest));
        if (safe) {
            const uint32_t f0 = exp_bits(nuc.zs[a1] * d1), f1 = exp_bits(nuc.zs[a2] * d2);
            const uint32_t f2 = tanh_bits(d1), f3 = tanh_bits(d2);
            const uint32_t f5 = tanh_bits(x5), f7 = exp_bits(s12 - pr.R);
            out = make_uint4(f0 | f1 << 16, f2 | f3 << 16, bf16_of_double(f4) | f5 << 16, pr.f6 | f7 << 16);
        }
    }
    if (!safe) out = features_exact(nuc, px, py, pz);
    *reinterpret_cast<uint4*>(feat + i * kF) = out;
}

__global__ void __launch_bounds__(kThreads) k_mlp_forward(const uint16_t* __restrict__ feat, int64_t n,
                                                          const double* __restrict__ master, float* __restrict__ y)
{
    __shared__ __align__(16) float sw[kPPad];
    load_params(sw, master);
    __syncthreads();
#pragma unroll 1
    for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads) {
        // the weights are read from shared memory in every iteration rather
        // than all 1377 held in registers across the loop
        asm volatile("" ::: "memory");
        float x[kF], h1[kH];
        load_x(feat, i, x);
        layer1(sw, x, h1);
        float out = sw[oB3];
#pragma unroll 1
        for (int j = 0; j < kH; j++) out = fmaf(sw[oW3 + j], layer2_unit(sw, h1, j), out);
        y[i] = out;
    }
}

// Loss L = sum_p wt_p (y_p - t_p)^2 and its gradient: each thread runs the
// forward and backward pass of one point of a 128-point tile and stashes
// (x, h1, h2, dz1, dz2, dy) in shared memory; then each thread forms its own
// gradient entries (outer-product sums over the tile in point order, float32)
// and adds them to float64 accumulators.  Tiles are strided over a fixed grid;
// per-block partials [grid][kP + 1] (the loss last) are reduced by k_mlp_adam.
// Bound by shared-memory loads: they come four (two) values at a time, a
// quarter of what one by one took: loss and gradient of 192,000 points 157 ->
// 130 us, the same bits.
__global__ void __launch_bounds__(kThreads) k_mlp_grad(const uint16_t* __restrict__ feat,
                                                       const float* __restrict__ target, const float* __restrict__ wt,
                                                       int64_t n, const double* __restrict__ master,
                                                       double* __restrict__ partial)
{
    extern __shared__ __align__(16) float sm[];
    float* sw = sm;
    float* st = sm + kPPad;
    __shared__ double sl[kThreads];
    const int tid = threadIdx.x;
    load_params(sw, master);

    const int j0 = 2 * (tid >> 3), i0 = 4 * (tid & 7);
    const int r1 = tid >> 2, f1 = 2 * (tid & 3);  // W1 row, first of two features
    // the other entry: rp[ca] * rp[cb]; threads past them compute and drop one
    const int ce = tid < kH ? oB1 + tid : tid < 2 * kH ? oB2 + tid - kH : tid < 3 * kH ? oW3 + tid - 2 * kH : oB3;
    const int ca = tid < kH ? cD1 + tid : tid < 2 * kH ? cD2 + tid - kH : cDy;
    const int cb = tid >= 2 * kH && tid < 3 * kH ? cH2 + tid - 2 * kH : cOne;
    double accw[8], acc1[2] = {0.0, 0.0}, accr = 0.0;
#pragma unroll
    for (int k = 0; k < 8; k++) accw[k] = 0.0;
    double lsum = 0.0;
    __syncthreads();

    const int64_t ntiles = (n + kThreads - 1) / kThreads;
    float* row = st + tid * kStride;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t i = tile * kThreads + tid;
        if (i < n) {
            float x[kF], h1[kH];
            load_x(feat, i, x);
            layer1(sw, x, h1);
            float y = sw[oB3];
#pragma unroll 1
            for (int j = 0; j < kH; j += 4) {
                float a[4];
#pragma unroll
                for (int c = 0; c < 4; c++) {
                    a[c] = layer2_unit(sw, h1, j + c);
                    y = fmaf(sw[oW3 + j + c], a[c], y);
                }
                *reinterpret_cast<float4*>(row + cH2 + j) = make_float4(a[0], a[1], a[2], a[3]);
            }
            const float r = y - target[i];
            const float dy = 2.0f * wt[i] * r;
            lsum += (double)wt[i] * (double)r * (double)r;
            float g1[kH];
#pragma unroll
            for (int q = 0; q < kH; q++) g1[q] = 0.0f;
#pragma unroll 1
            for (int j = 0; j < kH; j += 4) {
                float a[4], d2[4];
                weights4(row + cH2 + j, a);
#pragma unroll
                for (int c = 0; c < 4; c++) {
                    d2[c] = dy * sw[oW3 + j + c] * (1.0f - a[c] * a[c]);
#pragma unroll
                    for (int q = 0; q < kH; q += 4) {
                        float w[4];
                        weights4(sw + oW2 + (j + c) * kH + q, w);
#pragma unroll
                        for (int u = 0; u < 4; u++) g1[q + u] = fmaf(w[u], d2[c], g1[q + u]);
                    }
                }
                *reinterpret_cast<float4*>(row + cD2 + j) = make_float4(d2[0], d2[1], d2[2], d2[3]);
            }
#pragma unroll
            for (int q = 0; q < kH; q += 4) {
                *reinterpret_cast<float4*>(row + cH1 + q) = make_float4(h1[q], h1[q + 1], h1[q + 2], h1[q + 3]);
                float d1[4];
#pragma unroll
                for (int u = 0; u < 4; u++) d1[u] = g1[q + u] * (1.0f - h1[q + u] * h1[q + u]);
                *reinterpret_cast<float4*>(row + cD1 + q) = make_float4(d1[0], d1[1], d1[2], d1[3]);
            }
#pragma unroll
            for (int f = 0; f < kF; f += 4)
                *reinterpret_cast<float4*>(row + cX + f) = make_float4(x[f], x[f + 1], x[f + 2], x[f + 3]);
            *reinterpret_cast<float4*>(row + cDy) = make_float4(dy, 1.0f, 0.0f, 0.0f);
        } else {
            for (int c = 0; c < kStride; c += 4)
                *reinterpret_cast<float4*>(row + c) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        __syncthreads();
        {
            float s[8], s1[2] = {0.0f, 0.0f}, sr = 0.0f;
#pragma unroll
            for (int k = 0; k < 8; k++) s[k] = 0.0f;
#pragma unroll 4
            for (int p = 0; p < kThreads; p++) {
                const float* rp = st + p * kStride;
                const float2 d = *reinterpret_cast<const float2*>(rp + cD2 + j0);
                float h[4];
                weights4(rp + cH1 + i0, h);
#pragma unroll
                for (int c = 0; c < 4; c++) {
                    s[c] = fmaf(d.x, h[c], s[c]);
                    s[4 + c] = fmaf(d.y, h[c], s[4 + c]);
                }
                const float e = rp[cD1 + r1];
                const float2 xf = *reinterpret_cast<const float2*>(rp + cX + f1);
                s1[0] = fmaf(e, xf.x, s1[0]);
                s1[1] = fmaf(e, xf.y, s1[1]);
                sr = fmaf(rp[ca], rp[cb], sr);
            }
#pragma unroll
            for (int k = 0; k < 8; k++) accw[k] += (double)s[k];
            acc1[0] += (double)s1[0];
            acc1[1] += (double)s1[1];
            accr += (double)sr;
        }
        __syncthreads();
    }
    double* out = partial + (size_t)blockIdx.x * (kP + 1);
#pragma unroll
    for (int c = 0; c < 4; c++) {
        out[oW2 + j0 * kH + i0 + c] = accw[c];
        out[oW2 + (j0 + 1) * kH + i0 + c] = accw[4 + c];
    }
    out[oW1 + r1 * kF + f1] = acc1[0];
    out[oW1 + r1 * kF + f1 + 1] = acc1[1];
    if (tid < kRest) out[ce] = accr;
    sl[tid] = lsum;
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        for (int t = 0; t < kThreads; t++) s += sl[t];
        out[kP] = s;
    }
}

// Gradient and loss from the per-block partials [nblk][np + 1], then, if
// apply, one Adam step on the float64 master weights (c1 = 1 - beta1^t, c2 =
// 1 - beta2^t).  A block sums 32 entries, each by kAdamSlices threads over
// every kAdamSlices-th row whose sums are then added in order: one thread
// alone waits for one row after another (38 us for 304 rows).  tc: the rows
// are in the order of mlp64.cuh.
constexpr int kAdamSlices = 16;
__global__ void __launch_bounds__(32 * kAdamSlices) k_mlp_adam(const double* __restrict__ partial, int nblk, int np,
                                                               int tc, double* __restrict__ master,
                                                               double* __restrict__ m, double* __restrict__ v,
                                                               double lr, double beta1, double beta2, double eps,
                                                               double c1, double c2, int apply,
                                                               double* __restrict__ grad_out,
                                                               double* __restrict__ loss_out)
{
    __shared__ double part[kAdamSlices][32];
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + lane;
    double g = 0.0;
    if (e <= np) {
        const double* row = partial + (tc ? mlp64::slot(e) : e);
        for (int b = slice; b < nblk; b += kAdamSlices) g += row[(size_t)b * (np + 1)];
    }
    part[slice][lane] = g;
    __syncthreads();
    if (slice > 0 || e > np) return;
#pragma unroll
    for (int q = 1; q < kAdamSlices; q++) g += part[q][lane];
    if (e == np) {
        *loss_out = g;
        return;
    }
    grad_out[e] = g;
    if (!apply) return;
    const double mm = beta1 * m[e] + (1.0 - beta1) * g;
    const double vv = beta2 * v[e] + (1.0 - beta2) * g * g;
    m[e] = mm;
    v[e] = vv;
    master[e] -= (lr * (mm / c1)) / (sqrt(vv / c2) + eps);
}

// psi = s (1 + y) and per-block partial sums of psi^2 w (block order).
__global__ void __launch_bounds__(256) k_warm_apply(const float* __restrict__ y, const double* __restrict__ s,
                                                    const double* __restrict__ w, int64_t n,
                                                    double* __restrict__ psi, double* __restrict__ part)
{
    __shared__ double red[256];
    double acc = 0.0;
    for (int64_t i = blockIdx.x * 256LL + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const double p = s[i] * (1.0 + (double)y[i]);
        psi[i] = p;
        acc += p * p * w[i];
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// psi /= sqrt(sum of the partials): every block sums them in the same order
// (256 strided sums, then a tree), so every block has the same factor.  One
// thread that adds 608 partials one after another took 35 of this kernel's 39
// us.
__global__ void __launch_bounds__(256) k_warm_scale(double* __restrict__ psi, int64_t n,
                                                    const double* __restrict__ part, int nblk)
{
    __shared__ double red[256];
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += 256) s += part[b];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    const double inv = 1.0 / sqrt(red[0]);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        psi[i] *= inv;
}

// ------------------------------------------------------------------ object
struct Mlp {
    int dev = 0;
    int sms = 0;
    int H = kH;     // 32: SIMT kernels of this file; 64: tensor-core kernels (mlp64.cu)
    int np = kP;    // parameters
    int64_t step = 0;
    DevBuf master, m, v, partial, grad, loss, part, errd;
    std::string err;
};

int grad_grid(const Mlp& M, int64_t n)
{
    const int64_t tiles = (n + kThreads - 1) / kThreads;
    return (int)std::min<int64_t>(tiles, 2LL * M.sms);
}

thread_local std::string g_mlp_err;

template <class F>
tagi_status guarded_mlp(F&& f)
{
    try {
        report_error(TAGI_OK, "");
        f();
        return TAGI_OK;
    } catch (const Error& e) {
        g_mlp_err = e.what();
        return report_error(e.status, g_mlp_err.c_str());
    } catch (const std::bad_alloc&) {
        return report_error(TAGI_ERR_OOM, "host allocation failed");
    } catch (const std::exception& e) {
        g_mlp_err = e.what();
        return report_error(TAGI_ERR_CUDA, g_mlp_err.c_str());
    }
}

Mlp* as_mlp(const tagi_mlp* p)
{
    TAGI_REQUIRE(p != nullptr, "mlp is NULL");
    return reinterpret_cast<Mlp*>(const_cast<tagi_mlp*>(p));
}

void check_data(const void* feat, int64_t n)
{
    TAGI_REQUIRE(feat != nullptr, "feat is NULL");
    TAGI_REQUIRE(n >= 1, "n must be >= 1");
    TAGI_REQUIRE(((uintptr_t)feat & 15) == 0, "feat must be 16-byte aligned");
}

// Gradient (and loss) of the current master weights into M.grad / M.loss;
// with apply, one Adam step as well.
void grad_pass(Mlp& M, const uint16_t* feat, const float* target, const float* wt, int64_t n,
               const tagi_adam_params* a, bool apply, cudaStream_t s)
{
    const int grid = M.H == 64 ? mlp64_grad_grid(n, M.sms) : grad_grid(M, n);
    M.partial.ensure(sizeof(double) * (size_t)grid * (M.np + 1));
    if (M.H == 64)
        mlp64_gradient(feat, target, wt, n, M.master.as<double>(), M.partial.as<double>(), M.sms, M.errd.as<int>(), s);
    else
        launch(k_mlp_grad, grid, kThreads, kGradSmem, s, feat, target, wt, n, M.master.as<double>(),
               M.partial.as<double>());
    double c1 = 1.0, c2 = 1.0, lr = 0.0, b1 = 0.9, b2 = 0.999, eps = 1e-8;
    if (apply) {
        M.step += 1;
        lr = a->lr;
        b1 = a->beta1;
        b2 = a->beta2;
        eps = a->eps;
        c1 = 1.0 - std::pow(b1, (double)M.step);
        c2 = 1.0 - std::pow(b2, (double)M.step);
    }
    launch(k_mlp_adam, M.np / 32 + 1, 32 * kAdamSlices, 0, s, M.partial.as<double>(), grid, M.np, M.H == 64 ? 1 : 0,
           M.master.as<double>(), M.m.as<double>(), M.v.as<double>(), lr, b1, b2, eps, c1, c2, apply ? 1 : 0, M.grad.as<double>(),
           M.loss.as<double>());
    TAGI_LAUNCH_CHECK();
}

// y of the network for n points (the H = 32 or the H = 64 kernels)
void run_forward(Mlp& M, const uint16_t* feat, int64_t n, float* y, cudaStream_t s)
{
    if (M.H == 64) {
        mlp64_forward(feat, n, M.master.as<double>(), y, M.errd.as<int>(), M.sms, s);
    } else {
        const int64_t blocks = std::min<int64_t>((n + kThreads - 1) / kThreads, 8LL * M.sms);
        launch(k_mlp_forward, (unsigned)blocks, kThreads, 0, s, feat, n, M.master.as<double>(), y);
        TAGI_LAUNCH_CHECK();
    }
}

// after a synchronisation: a bounded wait of the tensor-core kernels gave up
void check_mlp_err(Mlp& M, cudaStream_t s)
{
    if (M.H != 64) return;
    int h = 0;
    TAGI_CUDA(cudaMemcpyAsync(&h, M.errd.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    TAGI_CUDA(cudaStreamSynchronize(s));
    if (h) throw Error(TAGI_ERR_TIMEOUT, "a bounded wait of the tensor-core MLP kernels gave up");
}

}  // namespace
}  // namespace tagi

using namespace tagi;

extern "C" {

tagi_status tagi_mlp_create(int n_features, int hidden, const double* params, int64_t n_params, tagi_mlp** out)
{
    return guarded_mlp([&] {
        TAGI_REQUIRE(out != nullptr, "out is NULL");
        *out = nullptr;
        TAGI_REQUIRE(n_features == kF && (hidden == kH || hidden == 64),
                     "the model has 8 features and 32 or 64 hidden units");
        const int np = hidden == 64 ? mlp64_params() : kP;
        TAGI_REQUIRE(params != nullptr && n_params == np, "params must hold 1377 (H = 32) or 4801 (H = 64) values");
        for (int64_t e = 0; e < n_params; e++) TAGI_REQUIRE(std::isfinite(params[e]), "params must be finite");
        TAGI_CUDA(cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGradSmem));
        auto* M = new Mlp();
        M->H = hidden;
        M->np = np;
        try {
            TAGI_CUDA(cudaGetDevice(&M->dev));
            TAGI_CUDA(cudaDeviceGetAttribute(&M->sms, cudaDevAttrMultiProcessorCount, M->dev));
            AllocStream as(nullptr);
            M->master.ensure(sizeof(double) * np);
            M->m.ensure(sizeof(double) * np);
            M->v.ensure(sizeof(double) * np);
            M->grad.ensure(sizeof(double) * np);
            M->loss.ensure(sizeof(double));
            M->errd.ensure(sizeof(int));
            TAGI_CUDA(cudaMemcpy(M->master.p, params, sizeof(double) * np, cudaMemcpyHostToDevice));
            TAGI_CUDA(cudaMemset(M->m.p, 0, sizeof(double) * np));
            TAGI_CUDA(cudaMemset(M->v.p, 0, sizeof(double) * np));
            TAGI_CUDA(cudaMemset(M->errd.p, 0, sizeof(int)));
        } catch (...) {
            delete M;
            throw;
        }
        *out = reinterpret_cast<tagi_mlp*>(M);
    });
}

tagi_status tagi_mlp_get_params(const tagi_mlp* mlp, double* params, int64_t n_params, void* stream)
{
    return guarded_mlp([&] {
        Mlp* M = as_mlp(mlp);
        TAGI_REQUIRE(params != nullptr && n_params == M->np, "params must hold the model's parameter count");
        cudaStream_t s = (cudaStream_t)stream;
        TAGI_CUDA(cudaMemcpyAsync(params, M->master.p, sizeof(double) * M->np, cudaMemcpyDeviceToHost, s));
        TAGI_CUDA(cudaStreamSynchronize(s));
        check_mlp_err(*M, s);
    });
}

static tagi_status features_call(const double* xyz, int64_t n, const double* nuclei, const double* scale,
                                 int n_nuclei, int ordered, uint16_t* feat, void* stream)
{
    return guarded_mlp([&] {
        TAGI_REQUIRE(xyz != nullptr && nuclei != nullptr, "xyz or nuclei is NULL");
        check_data(feat, n);
        TAGI_REQUIRE(n_nuclei >= 2 && n_nuclei <= kMaxNuclei, "need 2 to 16 nuclei");
        TAGI_REQUIRE(!ordered || n_nuclei == 2, "list order needs exactly two nuclei");
        Nuclei nu{};
        nu.m = n_nuclei;
        nu.ordered = ordered;
        for (int a = 0; a < n_nuclei; a++) {
            nu.x[a] = nuclei[3 * a];
            nu.y[a] = nuclei[3 * a + 1];
            nu.z[a] = nuclei[3 * a + 2];
            nu.zs[a] = scale ? scale[a] : 1.0;
            TAGI_REQUIRE(std::isfinite(nu.x[a]) && std::isfinite(nu.y[a]) && std::isfinite(nu.z[a]),
                         "nuclei must be finite");
            TAGI_REQUIRE(std::isfinite(nu.zs[a]) && nu.zs[a] > 0.0, "decay rates must be finite and positive");
        }
        for (int a = 0; a < n_nuclei; a++)
            for (int b = 0; b < a; b++)
                TAGI_REQUIRE(nu.x[a] != nu.x[b] || nu.y[a] != nu.y[b] || nu.z[a] != nu.z[b],
                             "nuclei must be distinct");
        launch(k_features, (unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream, xyz, n, nu, feat);
        TAGI_LAUNCH_CHECK();
    });
}

tagi_status tagi_mlp_features(const double* xyz, int64_t n, const double* nuclei, int n_nuclei, uint16_t* feat,
                              void* stream)
{
    return features_call(xyz, n, nuclei, nullptr, n_nuclei, 0, feat, stream);
}

tagi_status tagi_mlp_features_ordered(const double* xyz, int64_t n, const double* nuclei, uint16_t* feat,
                                      void* stream)
{
    return features_call(xyz, n, nuclei, nullptr, 2, 1, feat, stream);
}

tagi_status tagi_mlp_features_scaled(const double* xyz, int64_t n, const double* nuclei, const double* scale,
                                     int n_nuclei, int ordered, uint16_t* feat, void* stream)
{
    if (!scale) return report_error(TAGI_ERR_INVALID_ARG, "scale is NULL");
    return features_call(xyz, n, nuclei, scale, n_nuclei, ordered ? 1 : 0, feat, stream);
}

tagi_status tagi_mlp_forward(const tagi_mlp* mlp, const uint16_t* feat, int64_t n, float* y, void* stream)
{
    return guarded_mlp([&] {
        Mlp* M = as_mlp(mlp);
        check_data(feat, n);
        TAGI_REQUIRE(y != nullptr, "y is NULL");
        run_forward(*M, feat, n, y, (cudaStream_t)stream);
    });
}

tagi_status tagi_mlp_gradient(tagi_mlp* mlp, const uint16_t* feat, const float* target, const float* wt, int64_t n,
                              double* grad, double* loss, void* stream)
{
    return guarded_mlp([&] {
        Mlp* M = as_mlp(mlp);
        check_data(feat, n);
        TAGI_REQUIRE(target != nullptr && wt != nullptr, "target or wt is NULL");
        TAGI_REQUIRE(grad != nullptr && loss != nullptr, "grad or loss is NULL");
        cudaStream_t s = (cudaStream_t)stream;
        AllocStream as(s);
        grad_pass(*M, feat, target, wt, n, nullptr, false, s);
        TAGI_CUDA(cudaMemcpyAsync(grad, M->grad.p, sizeof(double) * M->np, cudaMemcpyDeviceToHost, s));
        TAGI_CUDA(cudaMemcpyAsync(loss, M->loss.p, sizeof(double), cudaMemcpyDeviceToHost, s));
        TAGI_CUDA(cudaStreamSynchronize(s));
        check_mlp_err(*M, s);
    });
}

tagi_status tagi_mlp_train_step(tagi_mlp* mlp, const uint16_t* feat, const float* target, const float* wt,
                                int64_t n, const tagi_adam_params* adam, double* loss, void* stream)
{
    return guarded_mlp([&] {
        Mlp* M = as_mlp(mlp);
        check_data(feat, n);
        TAGI_REQUIRE(target != nullptr && wt != nullptr && adam != nullptr, "target, wt or adam is NULL");
        TAGI_REQUIRE(std::isfinite(adam->lr) && adam->lr >= 0.0, "lr must be >= 0");
        TAGI_REQUIRE(adam->beta1 >= 0.0 && adam->beta1 < 1.0 && adam->beta2 >= 0.0 && adam->beta2 < 1.0,
                     "beta1 and beta2 must be in [0, 1)");
        TAGI_REQUIRE(adam->eps > 0.0, "eps must be > 0");
        cudaStream_t s = (cudaStream_t)stream;
        AllocStream as(s);
        grad_pass(*M, feat, target, wt, n, adam, true, s);
        if (loss) {
            TAGI_CUDA(cudaMemcpyAsync(loss, M->loss.p, sizeof(double), cudaMemcpyDeviceToHost, s));
            TAGI_CUDA(cudaStreamSynchronize(s));
            check_mlp_err(*M, s);
        }
    });
}

tagi_status tagi_mlp_warm_start(const tagi_mlp* mlp, const uint16_t* feat, const double* s0, const double* w,
                                int64_t n, double* psi, void* stream)
{
    return guarded_mlp([&] {
        Mlp* M = as_mlp(mlp);
        check_data(feat, n);
        TAGI_REQUIRE(s0 != nullptr && w != nullptr && psi != nullptr, "s, w or psi is NULL");
        cudaStream_t s = (cudaStream_t)stream;
        AllocStream as(s);
        DevBuf y;
        y.ensure(sizeof(float) * (size_t)n);
        run_forward(*M, feat, n, y.as<float>(), s);
        const int nb = (int)std::min<int64_t>((n + 255) / 256, 4LL * M->sms);
        M->part.ensure(sizeof(double) * nb);
        launch(k_warm_apply, nb, 256, 0, s, (const float*)y.as<float>(), s0, w, n, psi, M->part.as<double>());
        launch(k_warm_scale, (unsigned)std::min<int64_t>((n + 255) / 256, 2LL * M->sms), 256, 0, s, psi, n,
               (const double*)M->part.as<double>(), nb);
        TAGI_LAUNCH_CHECK();
    });
}

tagi_status tagi_mlp_destroy(tagi_mlp* mlp)
{
    return guarded_mlp([&] {
        if (!mlp) return;
        Mlp* M = reinterpret_cast<Mlp*>(mlp);
        TAGI_CUDA(cudaDeviceSynchronize());
        delete M;
    });
}

}  // extern "C"
