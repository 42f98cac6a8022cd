// Shared by the line-pass AX kernels (nek_ax_fx.cuh, nek_ax_dx.cuh): the shared-memory layout of an element whose threads walk
// its lines, asynchronous copies, and the integer arithmetic of their block fixed point.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace nek {

namespace {

// Shared-memory layout of an element's points (8-byte words): point (i, j, k) at i + row j + plane k.  The
// pitches are those with the fewest bank conflicts over the three line directions and the point-wise passes (counted for
// every nx over the lanes of a warp): dense except where nx is a multiple of 4.
template <int NX>
struct FxGrid {
    static constexpr int ROW = NX == 16 ? 17 : NX;
    static constexpr int PAD = NX == 4 ? 4 : NX == 8 ? 2 : NX == 12 ? 12 : 0;
    static constexpr int PLANE = NX * ROW + PAD;
    static constexpr int SIZE = NX * PLANE;
    // r lines are nx words apart from lane to lane: every second run of REV lanes walks its lines backwards
    // (with the sign of the input flipped, D[n-1-i][n-1-l] = -D[i][l]), so that the two runs meet different banks
    static constexpr int REV = NX % 2 ? 0 : NX == 16 ? 0 : NX % 4 ? 8 : 4;
    __device__ static __forceinline__ int at(int p)
    {
        int a = p;
        if constexpr (ROW != NX) a += (ROW - NX) * (p / NX);
        if constexpr (PAD != 0) a += PAD * (p / (NX * NX));
        return a;
    }
};

constexpr int kSMs = 152;  // of a GB300

__device__ __forceinline__ void cp_async8(void* dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

__device__ __forceinline__ long long madw(int a, int b, long long c) { return (long long)a * b + c; }

// z 2^x as a double (round to nearest even; x such that nothing overflows or underflows), from the bit pattern: no
// FP64 instruction.
__device__ __forceinline__ double fx_ldexp(long long z, int x)
{
    const long long sg = z >> 63;
    const unsigned long long a = (unsigned long long)((z ^ sg) - sg);
    const int lz = __clzll((long long)a);
    const unsigned long long f = a << lz >> 1;
    const unsigned long long m = (f + 0x1FFull + ((unsigned)(f >> 10) & 1u)) >> 10;  // leading one at bit 52 (53 after a carry)
    const unsigned hi = (unsigned)(m >> 32) + ((unsigned)(1085 + x - lz) << 20);  // the leading one adds 1
    return a == 0 ? 0.0 : __hiloint2double((int)(hi | ((unsigned)sg & 0x80000000u)), (int)(unsigned)m);
}

// n doubles from p into L2 (a hint: the whole 16-byte units among them).
__device__ __forceinline__ void l2_prefetch(const double* p, int64_t n)
{
    const uintptr_t a = (reinterpret_cast<uintptr_t>(p) + 15) & ~(uintptr_t)15;
    const int64_t bytes = (int64_t)(reinterpret_cast<uintptr_t>(p + n) - a) & ~(int64_t)15;
    if (bytes > 0)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((unsigned)bytes) : "memory");
}

}  // namespace

}  // namespace nek
