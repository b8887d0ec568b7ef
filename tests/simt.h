// Runs a CUDA kernel's source as host C++, one block at a time: a thread of the
// block is a coroutine, a barrier or a warp shuffle is where it gives way.  One
// warp may be held back (`late`): it runs only when no other thread can, which is
// the latest a scheduler may run it.  Enough of CUDA for the kernels that the
// tests take through it.
#pragma once
#include <ucontext.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <functional>
#include <vector>

#define __global__
#define __device__
#define __forceinline__ inline
#define __launch_bounds__(n)
#define __restrict__
#define __shared__ static
using std::max;
using std::min;

struct Index {
    unsigned x;
};
static Index threadIdx, blockIdx;
struct alignas(16) float4 {
    float x, y, z, w;
};
inline float4 make_float4(float x, float y, float z, float w) { return {x, y, z, w}; }
template <class T>
T __ldg(const T* p) { return *p; }
template <class T>
T __ldcg(const T* p) { return *p; }
inline int __float_as_int(float f) { int i; memcpy(&i, &f, 4); return i; }
inline float __int_as_float(int i) { float f; memcpy(&f, &i, 4); return f; }
inline unsigned atomicOr(unsigned* p, unsigned v) { unsigned o = *p; *p |= v; return o; }
inline unsigned long long atomicAdd(unsigned long long* p, unsigned long long v) {
    unsigned long long o = *p;
    *p += v;
    return o;
}

namespace simt {
struct Group {  // a block or a warp: its live threads meet here
    int live = 0, here = 0;
    unsigned gen = 0, any = 0, all = 0;
    void arrive() {
        if (here == live && live) {
            here = 0;
            all = any;
            any = 0;
            ++gen;
        }
    }
};
static std::vector<ucontext_t> ctx;
static std::vector<char> gone, waits;
static std::vector<Group*> at;
static std::vector<unsigned> want;
static ucontext_t home;
static Group block;
static std::vector<Group> warps;
static std::vector<uint32_t> lane_word;
static const std::function<void()>* body;

inline void give_way() { swapcontext(&ctx[threadIdx.x], &home); }
inline unsigned meet(Group& g, unsigned v) {
    const unsigned t = threadIdx.x;
    g.any |= v;
    ++g.here;
    at[t] = &g;
    want[t] = g.gen + 1;
    waits[t] = 1;
    g.arrive();
    give_way();
    return g.all;
}
inline Group& my_warp() { return warps[threadIdx.x / 32]; }
inline void start() {
    const unsigned t = threadIdx.x;
    (*body)();
    gone[t] = 1;
    --block.live;
    --warps[t / 32].live;
    block.arrive();
    warps[t / 32].arrive();
}
inline void run_block(int n, int late, const std::function<void()>& f) {
    static std::vector<std::vector<char>> stacks;
    body = &f;
    ctx.resize(n);
    stacks.resize(n);
    gone.assign(n, 0);
    waits.assign(n, 0);
    at.assign(n, nullptr);
    want.assign(n, 0);
    lane_word.assign(n, 0);
    block = Group();
    block.live = n;
    warps.assign(n / 32, Group());
    for (auto& w : warps) w.live = 32;
    for (int t = 0; t < n; ++t) {
        stacks[t].resize(64 << 10);
        getcontext(&ctx[t]);
        ctx[t].uc_stack.ss_sp = stacks[t].data();
        ctx[t].uc_stack.ss_size = stacks[t].size();
        ctx[t].uc_link = &home;
        makecontext(&ctx[t], start, 0);
    }
    for (int left = n; left;) {
        bool ran = false;
        for (int pass = 0; pass < 2 && !ran; ++pass)  // the late warp only if nobody else could go on
            for (int t = 0; t < n; ++t) {
                if (gone[t] || (t / 32 == late) != (pass == 1)) continue;
                if (waits[t] && at[t]->gen != want[t]) continue;
                waits[t] = 0;
                ran = true;
                threadIdx.x = t;
                swapcontext(&home, &ctx[t]);
                left -= gone[t];
            }
        if (!ran) abort();  // a barrier that nobody can complete
    }
}
}  // namespace simt

inline void __syncthreads() { simt::meet(simt::block, 0); }
inline int __syncthreads_or(int p) { return simt::meet(simt::block, p != 0) != 0; }
inline unsigned __reduce_or_sync(unsigned, unsigned v) { return simt::meet(simt::my_warp(), v); }
inline int simt_shfl(int v, int from) {
    const int t = threadIdx.x, base = t & ~31;
    simt::lane_word[t] = (uint32_t)v;
    simt::meet(simt::my_warp(), 0);
    const int got = (int)simt::lane_word[base + from];
    simt::meet(simt::my_warp(), 0);
    return got;
}
inline int __shfl_up_sync(unsigned, int v, int d) { const int l = threadIdx.x & 31; return simt_shfl(v, l < d ? l : l - d); }
inline int __shfl_down_sync(unsigned, int v, int d) { const int l = threadIdx.x & 31; return simt_shfl(v, l + d > 31 ? l : l + d); }
