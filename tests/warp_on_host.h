// Runs device code of one warp on the host: the 32 lanes are coroutines, each of which runs on its own
// until its next warp-wide operation, in a given order.  Code that reads shared memory which another
// lane may already have overwritten (no warp-wide operation between the two) gives wrong results under some
// order, and the same ones every time.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>
#include <ucontext.h>

#include <functional>
#include <vector>

#undef __shared__
#define __shared__ static

static struct { unsigned x; } threadIdx, blockDim{32};

template <typename T, typename F> static T bits_as(F v) {
    static_assert(sizeof(T) == sizeof(F), "");
    T r;
    memcpy(&r, &v, sizeof r);
    return r;
}
static inline long long __double_as_longlong(double v) { return bits_as<long long>(v); }
static inline unsigned __float_as_uint(float v) { return bits_as<unsigned>(v); }
static inline float __uint_as_float(unsigned v) { return bits_as<float>(v); }
static inline double __hiloint2double(int hi, int lo) { return bits_as<double>(((unsigned long long)(unsigned)hi << 32) | (unsigned)lo); }
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
    return (unsigned)(((((unsigned long long)hi << 32) | lo) << (s & 31)) >> 32);
}
static inline float __fdividef(float a, float b) { return a / b; }
template <typename T> static inline T __ldg(const T *p) { return *p; }

struct Warp {
    ucontext_t main, lane[32];
    std::vector<char> stack[32];
    double slot[2][32];
    unsigned step[32];
    bool done[32];
    unsigned now;
    std::function<void()> body;
};
static Warp W;

static void warp_yield() { swapcontext(&W.lane[W.now], &W.main); }
static void warp_entry() {
    W.body();
    W.done[W.now] = true;
    warp_yield();
}
// body by every lane, the lanes taking their steps in the order order[0], order[1], ...
static void run_warp(const int *order, std::function<void()> body) {
    W.body = body;
    for (int l = 0; l < 32; l++) {
        W.stack[l].resize(256 * 1024);
        W.step[l] = 0;
        W.done[l] = false;
        getcontext(&W.lane[l]);
        W.lane[l].uc_stack.ss_sp = W.stack[l].data();
        W.lane[l].uc_stack.ss_size = W.stack[l].size();
        W.lane[l].uc_link = &W.main;
        makecontext(&W.lane[l], warp_entry, 0);
    }
    for (bool live = true; live;) {
        live = false;
        for (int q = 0; q < 32; q++) {
            const int l = order[q];
            if (W.done[l]) continue;
            live = true;
            W.now = threadIdx.x = (unsigned)l;
            swapcontext(&W.main, &W.lane[l]);
        }
    }
}
static inline void __syncwarp(unsigned = 0xffffffffu) {
    W.step[W.now]++;
    warp_yield();
    threadIdx.x = W.now;
}
static inline double __shfl_sync(unsigned, double v, int src) {
    double *s = W.slot[W.step[W.now] & 1];  // a lane reaches the next such operation only after all have read
    s[W.now] = v;
    __syncwarp();
    return s[src & 31];
}
