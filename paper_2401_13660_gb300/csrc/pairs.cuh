// Helpers of the scans that put two adjacent steps into each packed fp32 operation (forward.cu, backward.cu).
#pragma once

#include "common.cuh"
#include "tma.cuh"

namespace mbscan {

__device__ __forceinline__ float2 splat(float v) { return make_float2(v, v); }

__device__ __forceinline__ float2 shfl2(float2 v, int mask) {
    return make_float2(__shfl_xor_sync(kFull, v.x, mask), __shfl_xor_sync(kFull, v.y, mask));
}

// Byte offset of channels c, c + 1 at step t in a token tile of kCh channels, swizzled by TMA in its rows of 64 or
// 128 bytes (16-byte chunk j of row t at chunk j ^ (t / 2 % 4), j ^ (t % 8))
template <typename T, int kCh>
__device__ __forceinline__ int tile_off(int t, int c) {
    constexpr int kRow = kCh * (int)sizeof(T);
    static_assert(kRow == 64 || kRow == 128, "rows of a swizzle pattern");
    const int by = c * (int)sizeof(T), x = kRow == 128 ? t & 7 : (t >> 1) & 3;
    return t * kRow + (((by >> 4) ^ x) << 4) + (by & 15);
}

// Two adjacent elements of the input dtype at a byte offset of a shared tile, as fp32
template <typename T>
__device__ __forceinline__ float2 ld2(const void *base, int off) {
    if constexpr (sizeof(T) == 2) {
        const unsigned u = *reinterpret_cast<const unsigned *>(static_cast<const char *>(base) + off);
        return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
    } else {
        return *reinterpret_cast<const float2 *>(static_cast<const char *>(base) + off);
    }
}
template <typename T>
__device__ __forceinline__ void st2(void *base, int off, float2 v) {
    if constexpr (sizeof(T) == 2)
        *reinterpret_cast<__nv_bfloat162 *>(static_cast<char *>(base) + off) = __floats2bfloat162_rn(v.x, v.y);
    else
        *reinterpret_cast<float2 *>(static_cast<char *>(base) + off) = v;
}

__device__ __forceinline__ float rcp(float x) {   // 1 / x on the SFU
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// softplus(v) of a pair given u = e^v and o = 1 + u: the same three ranges as softplus() of common.cuh
__device__ __forceinline__ float2 softplus_of(float2 v, float2 u, float2 o) {
    float2 r = fma2(u, splat(0.33333334f), splat(-0.5f));
    r = mul2(u, fma2(u, r, splat(1.f)));
    const float2 lw = mul2(make_float2(lg2(o.x), lg2(o.y)), splat(kLn2));
    r.x = u.x < 0.03125f ? r.x : lw.x;
    r.y = u.y < 0.03125f ? r.y : lw.y;
    r.x = v.x > 15.f ? v.x : r.x;
    r.y = v.y > 15.f ? v.y : r.y;
    return r;
}
__device__ __forceinline__ float2 softplus2(float2 v) {
    const float2 w = mul2(v, splat(kLog2e));
    const float2 u = make_float2(ex2(w.x), ex2(w.y));
    return softplus_of(v, u, add2(u, splat(1.f)));
}

// silu(z) of a pair
__device__ __forceinline__ float2 silu2(float2 z) {
    const float2 w = mul2(z, splat(-kLog2e));
    const float2 o = add2(make_float2(ex2(w.x), ex2(w.y)), splat(1.f));
    return mul2(z, make_float2(rcp(o.x), rcp(o.y)));
}

// A state (adjoint) h carried over a segment with decays p and end state (adjoint) e from zero. A zero one stays out of
// it: where states grow (A > 0) p overflows, and step by step no infinity would have met it. (The mask is on p: selecting
// e instead makes the loop over the segments wait for its loads, 1 x 8192 x 2048 123.2 us instead of 121.9.)
__device__ __forceinline__ float fold(float p, float h, float e) { return fmaf(h == 0.f ? 0.f : p, h, e); }

// A share's flag in global memory: set after its state has been written, and waited for (bounded).
__device__ __forceinline__ void flag_set(int *f) {
    asm volatile("st.release.gpu.global.s32 [%0], 1;" ::"l"(f) : "memory");
}
__device__ __forceinline__ bool flag_wait(const int *f) {
    const long long t0 = clock64();
    for (;;) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
        if (v) return true;
        if (clock64() - t0 > kWaitCycles) return false;
    }
}

}  // namespace mbscan
