"""The H = 64 network's kernels when a bounded wait runs out, on the host.

mlp64.cu is compiled with g++ against stand-ins for the CUDA names it uses: a
CTA is 256 threads, __syncthreads a barrier that checks that every thread stands
at the same line, and the mbarrier's waits give up where a scenario says so.
Whatever threads see the limit first, they have to leave the tile loop together:
no thread may return from the kernel, or stand at another barrier, while others
wait, and tensor memory goes back only after a wait for every product issued.
"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2003_01833_gb300", "csrc")

CUDA = r"""
#pragma once
#include <math.h>
#include <pthread.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <time.h>
#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __noinline__
#define __launch_bounds__(...)
#define __restrict__
#define __align__(n) alignas(n)
#define __shared__ static
#define __syncthreads() emu::barrier(__LINE__, true)
#define __syncthreads_and(x) emu::barrier(__LINE__, (x))
#define asm(...) r = 0
using std::isnan;
struct uint4 { uint32_t x, y, z, w; };
struct float4 { float x, y, z, w; };
struct dim { unsigned x, y, z; };
static inline uint4 make_uint4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) { return uint4{a, b, c, d}; }
template <class T, class U> T bits(U u) { T t; memcpy(&t, &u, sizeof t); return t; }
static inline long long __double_as_longlong(double x) { return bits<long long>(x); }
static inline uint32_t __float_as_uint(float x) { return bits<uint32_t>(x); }
static inline float __uint_as_float(uint32_t x) { return bits<float>(x); }
typedef void* cudaStream_t;
static thread_local dim threadIdx;
static dim blockIdx, gridDim;

namespace emu {
constexpr int kThreads = 256;
alignas(1024) static uint8_t smem[1 << 18];
static pthread_mutex_t mu = PTHREAD_MUTEX_INITIALIZER;
static pthread_cond_t cv = PTHREAD_COND_INITIALIZER;
static int waiting, at_line, round_, result, value = 1, left;
// Products complete in order, at once, except that those of commit `stuck` take
// longer than the limit of the threads that late() names and hold up all behind
static int stuck, mode, issued;
static bool held, freed;
struct Bar {
    uint64_t* p;
    int done, pending;
};
static Bar bars[2];
static thread_local int waits;  // on the first barrier

static Bar& bar_of(uint64_t* p)
{
    for (Bar& b : bars)
        if (!b.p || b.p == p) {
            b.p = p;
            return b;
        }
    abort();
}
static void release()
{
    held = false;
    for (Bar& b : bars) {
        b.done += b.pending;
        b.pending = 0;
    }
}

static void fail(const char* what)
{
    printf("commit %d mode %d: %s\n", stuck, mode, what);
    fflush(stdout);
    _Exit(1);
}
static timespec in(double s)
{
    timespec t;
    clock_gettime(CLOCK_REALTIME, &t);
    t.tv_nsec += (long)(s * 1e9);
    t.tv_sec += t.tv_nsec / 1000000000;
    t.tv_nsec %= 1000000000;
    return t;
}
static bool barrier(int line, bool x)
{
    pthread_mutex_lock(&mu);
    if (left) fail("a thread has returned, others are at a barrier");
    if (waiting && line != at_line) fail("threads at different barriers");
    at_line = line;
    value &= x;
    const int mine = round_;
    if (++waiting == kThreads) {
        waiting = 0;
        result = value;
        value = 1;
        round_++;
        pthread_cond_broadcast(&cv);
    } else {
        const timespec t = in(20.0);
        while (mine == round_)
            if (pthread_cond_timedwait(&cv, &mu, &t)) fail("a barrier that not all threads reach");
    }
    const bool r = result;
    pthread_mutex_unlock(&mu);
    return r;
}
static void commit(uint64_t* p)
{
    pthread_mutex_lock(&mu);
    if (issued++ == stuck) held = true;
    (held ? bar_of(p).pending : bar_of(p).done)++;
    pthread_cond_broadcast(&cv);
    pthread_mutex_unlock(&mu);
}
// whether thread t gives up on commit `stuck`
static bool late(int t)
{
    switch (mode) {
        case 0: return true;
        case 1: return t & 1;
        case 2: return t < 32;
        case 3: return t >= 128;
        case 4: return t != 0;
        default: return t == 0;
    }
}
static bool wait(uint64_t* p, uint32_t parity)
{
    pthread_mutex_lock(&mu);
    Bar& b = bar_of(p);
    const bool give_up = &b == bars && waits++ == stuck && late(threadIdx.x);
    const timespec limit = in(0.1);
    bool ok;
    while (!(ok = (uint32_t)(b.done & 1) != parity)) {
        if (held) {
            if (give_up) break;
            release();  // the others' limit is longer
            pthread_cond_broadcast(&cv);
        } else if (pthread_cond_timedwait(&cv, &mu, &limit)) {
            break;
        }
    }
    pthread_mutex_unlock(&mu);
    return ok && !give_up;
}
}  // namespace emu
static inline int atomicOr(int* p, int v) { return __atomic_fetch_or(p, v, __ATOMIC_SEQ_CST); }
"""

INTERNAL = r"""
#pragma once
#define TAGI_CUDA(x) (x)
#define TAGI_LAUNCH_CHECK()
constexpr int cudaFuncAttributeMaxDynamicSharedMemorySize = 8;
static inline int cudaGetDevice(int* d) { return *d = 0; }
template <class K> int cudaFuncSetAttribute(K, int, int) { return 0; }
template <class K, class... A> void launch(K, A...) {}
"""

TC = r"""
#pragma once
namespace tagi { namespace tc {
static inline uint32_t smem_u32(const void*) { return 0; }
static inline uint64_t sdesc_sw128(uint32_t) { return 0; }
static inline uint64_t sdesc_mn_sw128(uint32_t, uint32_t) { return 0; }
static inline uint32_t idesc_bf16(int, int, bool = false, bool = false) { return 0; }
static inline void mma_bf16(uint32_t, uint64_t, uint64_t, uint32_t, uint32_t) {}
static inline void commit(uint64_t* b) { emu::commit(b); }
static inline bool mbar_wait(uint64_t* b, uint32_t parity, long long) { return emu::wait(b, parity); }
static inline void mbar_init(uint64_t* b, uint32_t) { emu::bar_of(b); }
static inline void tmem_alloc(uint32_t* slot, uint32_t) { *slot = 0; }
static inline void tmem_dealloc(uint32_t, uint32_t)
{
    if (emu::held) emu::fail("tensor memory freed with products in flight");
    emu::freed = true;
}
template <int N> void ld(float* v)
{
    if (emu::freed) emu::fail("tensor memory read after it was freed");
    for (int i = 0; i < N; i++) v[i] = 0.0f;
}
static inline void tmem_ld8(uint32_t, float* v) { ld<8>(v); }
static inline void tmem_ld16(uint32_t, float* v) { ld<16>(v); }
static inline void fence_async_smem() {}
static inline void fence_before_sync() {}
static inline void fence_after_sync() {}
}}
"""

MAIN = r"""
#include "mlp64.cu"
using namespace tagi;
constexpr int N = 300;  // three tiles of one CTA
static uint16_t feat[N * 8];
static float target[N], wt[N], y[N];
static double master[mlp64::kParams], partial[mlp64::kParams + 1];
static int err;
static bool grad;
static void* thread(void* arg)
{
    threadIdx.x = (unsigned)(intptr_t)arg;
    if (grad)
        k_mlp64_grad(feat, target, wt, N, master, partial, 1, &err);
    else
        k_mlp64_fwd(feat, N, master, y, &err);
    pthread_mutex_lock(&emu::mu);
    emu::left++;
    if (emu::waiting) emu::fail("a thread returns, others are at a barrier");
    pthread_mutex_unlock(&emu::mu);
    return nullptr;
}
int main(int argc, char** argv)
{
    grad = atoi(argv[1]);
    gridDim.x = 1;
    const int commits = grad ? 12 : 6;
    for (emu::stuck = 0; emu::stuck <= commits; emu::stuck++)
        for (emu::mode = 0; emu::mode < 6; emu::mode++) {
            emu::issued = emu::left = err = 0;
            emu::held = emu::freed = false;
            for (emu::Bar& b : emu::bars) b = emu::Bar{};
            pthread_t t[emu::kThreads];
            for (int i = 0; i < emu::kThreads; i++) pthread_create(&t[i], nullptr, thread, (void*)(intptr_t)i);
            for (int i = 0; i < emu::kThreads; i++) pthread_join(t[i], nullptr);
            if (err != (emu::stuck < commits)) emu::fail("the error flag is wrong");
            if (!emu::freed) emu::fail("tensor memory kept");
        }
    puts("ok");
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("mlp64")
    for name in ("mlp64.cu", "mlp64.cuh", "bf16.cuh"):
        with open(os.path.join(CSRC, name)) as f:
            s = f.read()
        (d / name).write_text(s.replace("extern __shared__ uint8_t raw[];", "uint8_t* raw = emu::smem;"))
    (d / "cuda_runtime.h").write_text(CUDA)
    (d / "tagi_internal.cuh").write_text(INTERNAL)
    (d / "tc.cuh").write_text(TC)
    (d / "main.cpp").write_text(MAIN)
    exe = str(d / "mlp64_waits")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-w", "-pthread", "-I", str(d), str(d / "main.cpp"), "-o", exe])
    return exe


@pytest.mark.parametrize("kernel", ["forward", "gradient"])
def test_threads_leave_together(program, kernel):
    r = subprocess.run([program, str(int(kernel == "gradient"))], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
