// The threads of one block as fibers on the host, in an order the test chooses:
// enough of CUDA to run device code that meets at barriers and trades values in
// warps.  A fiber runs until it meets others; emu_run reports the fibers that
// wait for ones that never come.
#pragma once
#include <ucontext.h>

#include <climits>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <functional>
#include <type_traits>
#include <vector>

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#undef __shared__
#undef __global__
#undef __launch_bounds__
#undef __restrict__
#undef __grid_constant__
#undef __cluster_dims__
#define __shared__ static
#define __global__ inline
#define __launch_bounds__(...)
#define __restrict__
#define __grid_constant__
#define __cluster_dims__(...)
#define __noinline__

struct EmuIndex { unsigned x = 0, y = 0, z = 0; };
inline EmuIndex threadIdx, blockIdx, blockDim, gridDim;

namespace emu {
struct Fiber {
    ucontext_t uc;
    std::vector<char> stack;
    bool done = false;
    int wait = -1;  // -1: ready; 0: at the block's barrier; 1: at its warp's
};
inline std::vector<Fiber> fibers;
inline ucontext_t main_uc;
inline int cur = 0;
inline uint64_t lane_val[4096];

inline void meet(int what) {
    fibers[cur].wait = what;
    swapcontext(&fibers[cur].uc, &main_uc);
}
inline std::function<void(int)> body;
inline void entry() {
    body(cur);
    fibers[cur].done = true;
    swapcontext(&fibers[cur].uc, &main_uc);
}
// Runs `n` threads; `order` lists them as they get their turns, `started(k)` is
// called after the k-th of the first round.  Returns how many are left waiting.
inline int run(int n, const std::vector<int> &order, std::function<void(int)> f,
               std::function<void(int)> started = {}) {
    body = f;
    fibers = std::vector<Fiber>(n);
    for (auto &fb : fibers) {
        fb.stack.resize(128 << 10);
        getcontext(&fb.uc);
        fb.uc.uc_stack.ss_sp = fb.stack.data();
        fb.uc.uc_stack.ss_size = fb.stack.size();
        fb.uc.uc_link = &main_uc;
        makecontext(&fb.uc, entry, 0);
    }
    bool first = true;
    for (;;) {
        bool ran = false;
        int k = 0;
        for (int t : order) {
            if (!fibers[t].done && fibers[t].wait < 0) {
                ran = true;
                cur = t;
                threadIdx.x = static_cast<unsigned>(t);
                swapcontext(&main_uc, &fibers[t].uc);
            }
            if (first && started) started(k);
            ++k;
        }
        first = false;
        // barriers that every thread has reached
        int at_block = 0;
        for (auto &fb : fibers) at_block += !fb.done && fb.wait == 0;
        if (at_block == n)
            for (auto &fb : fibers) fb.wait = -1;
        bool freed = at_block == n;
        for (int w = 0; w < n; w += 32) {
            const int m = n - w < 32 ? n - w : 32;
            int c = 0;
            for (int t = w; t < w + m; ++t) c += !fibers[t].done && fibers[t].wait == 1;
            if (c == m) {
                for (int t = w; t < w + m; ++t) fibers[t].wait = -1;
                freed = true;
            }
        }
        if (!ran && !freed) break;
    }
    int stuck = 0;
    for (auto &fb : fibers) stuck += !fb.done;
    return stuck;
}
template <class T>
T trade(T v, int src) {
    static_assert(sizeof(T) <= 8, "");
    const int me = cur;
    lane_val[me] = 0;
    memcpy(&lane_val[me], &v, sizeof(T));
    meet(1);
    T r;
    memcpy(&r, &lane_val[(me & ~31) | (src & 31)], sizeof(T));
    meet(1);
    return r;
}
}  // namespace emu

inline void __syncthreads() { emu::meet(0); }
inline void __syncwarp(unsigned = 0xffffffffu) { emu::meet(1); }
template <class T> T __shfl_xor_sync(unsigned, T v, int o) { return emu::trade(v, (emu::cur & 31) ^ o); }
template <class T> T __shfl_sync(unsigned, T v, int s) { return emu::trade(v, s); }
inline bool __any_sync(unsigned, bool p) {
    bool r = false;
    for (int l = 0; l < 32; ++l) r = emu::trade(p, l) || r;
    return r;
}
inline void __threadfence() {}
inline void __nanosleep(unsigned) {}
template <class T, class U> T atomicOr(T *p, U v) { T o = *p; *p = o | v; return o; }
template <class T, class U> T atomicAdd(T *p, U v) { T o = *p; *p = o + v; return o; }
template <class T, class U> T atomicExch(T *p, U v) { T o = *p; *p = v; return o; }
template <class T> T atomicCAS(T *p, T c, T v) { T o = *p; if (o == c) *p = v; return o; }
template <class T> T __ldcg(const T *p) { return *p; }
inline long long clock64() { return 0; }
template <class A, class B> A emu_bits(B b) { A a; static_assert(sizeof(A) == sizeof(B), ""); memcpy(&a, &b, sizeof a); return a; }
inline int __double2hiint(double x) { return static_cast<int>(emu_bits<uint64_t>(x) >> 32); }
inline int __double2loint(double x) { return static_cast<int>(emu_bits<uint64_t>(x)); }
inline long long __double_as_longlong(double x) { return emu_bits<long long>(x); }
inline double __longlong_as_double(long long x) { return emu_bits<double>(x); }
inline float __uint_as_float(unsigned x) { return emu_bits<float>(x); }
inline float __int_as_float(int x) { return emu_bits<float>(x); }
inline unsigned __float_as_uint(float x) { return emu_bits<unsigned>(x); }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) { return s ? (hi << s) | (lo >> (32 - s)) : hi; }
inline size_t __cvta_generic_to_shared(const void *p) { return reinterpret_cast<size_t>(p); }
inline void emu_set_conditional(cudaGraphConditionalHandle, unsigned) {}
#define cudaGraphSetConditional emu_set_conditional
using std::max;
using std::min;
