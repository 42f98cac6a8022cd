// Learned element preconditioner: a small 3D convolutional network applied to
// every nx = 8 element block, its training kernels, and flexible CG using it.
//
// The network (no counterpart in the paper, which uses Nekbone's fixed
// preconditioner): input channels r/rms(r) and (Jacobi r)/rms(Jacobi r) of one
// element; three 3x3x3 convolutions with zero padding inside the element,
// 16 hidden channels and GELU after the first two; BF16 weights (FP32 master
// copy, rounded when staged), FP32 activations and accumulation.  The output,
// times rms(Jacobi r) and 1/multiplicity, summed over elements by dssum and
// masked, is the preconditioned residual.
//
// Parameter vector (FP32): W1 [16][2][27], b1 [16], W2 [16][16][27], b2 [16],
// W3 [1][16][27], b3 [1]; tap t = (dk+1)*9 + (dj+1)*3 + (di+1) reads the point
// (i+di, j+dj, k+dk).
#include <cuda_bf16.h>

#include <vector>

#include "nek_internal.h"
#include "nek_pcg.cuh"

namespace nek {

namespace {

constexpr int NXN = 8, NP = 512, CIN = 2, CH = 16;
constexpr int OW1 = 0, OB1 = OW1 + CH * CIN * 27, OW2 = OB1 + CH, OB2 = OW2 + CH * CH * 27, OW3 = OB2 + CH,
              OB3 = OW3 + CH * 27, NPARAM = OB3 + 1;

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float gelu(float v) { return 0.5f * v * (1.f + erff(v * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float v)
{
    return 0.5f * (1.f + erff(v * 0.70710678118654752f)) + v * expf(-0.5f * v * v) * 0.39894228040143268f;
}

// Weights staged in shared memory as [cin][27][cout] (BF16-rounded floats).
template <int CI, int CO>
__device__ __forceinline__ void stage_weights(const float* __restrict__ W, float* sW)
{
    for (int q = threadIdx.x; q < CI * 27 * CO; q += blockDim.x) {
        const int o = q % CO, t = (q / CO) % 27, c = q / (CO * 27);
        sW[q] = bf16r(W[(o * CI + c) * 27 + t]);
    }
}

// Two points per thread, p and p + NP/2 (planes k and k + 4): every weight read
// from shared memory feeds two FMAs.
template <int CI, int CO>
__device__ __forceinline__ void conv_2pts(const float* xin, const float* sW, const float* sb, int i, int j, int k,
                                          float (&acc0)[CO], float (&acc1)[CO])
{
#pragma unroll
    for (int o = 0; o < CO; o++) acc0[o] = acc1[o] = sb[o];
#pragma unroll
    for (int t = 0; t < 27; t++) {
        const int dk = t / 9 - 1, dj = (t / 3) % 3 - 1, di = t % 3 - 1;
        const int ii = i + di, jj = j + dj, k0 = k + dk, k1 = k + 4 + dk;
        if (ii < 0 || ii >= NXN || jj < 0 || jj >= NXN) continue;
        const bool v0 = k0 >= 0, v1 = k1 < NXN;  // k0 < 8 and k1 >= 0 always hold for k in [0,4)
        const int q0 = ii + NXN * (jj + NXN * k0), q1 = ii + NXN * (jj + NXN * k1);
#pragma unroll 4
        for (int c = 0; c < CI; c++) {
            const float x0 = v0 ? xin[c * NP + q0] : 0.f;
            const float x1 = v1 ? xin[c * NP + q1] : 0.f;
            const float* w = sW + (c * 27 + t) * CO;
#pragma unroll
            for (int o = 0; o < CO; o++) {
                const float wo = w[o];
                acc0[o] = fmaf(wo, x0, acc0[o]);
                acc1[o] = fmaf(wo, x1, acc1[o]);
            }
        }
    }
}

// ------------------------------------------------------------------ prep
// xin[e][0][p] = r/rms(r), xin[e][1][p] = (minv r)/rms(minv r); scale[e] = rms(minv r).
// One warp per element: lane l holds points l + 32 q (q = 0..15, coalesced), sums
// its FP64 squares, the warp sums the lanes with a fixed shuffle tree, and lane 0
// forms the two RMS values and their reciprocals (FP64 square root and division
// on one lane); no block-wide barrier, so the warps of a CTA work on different
// elements independently.
//
// Bound by the FP64 pipe (2 operations a clock and SM; a conversion between the types counts as one): 5 operations a point,
// and 5 additions, a root and two quotients a warp and element.  4096 elements: 46.8 -> 35.8 us with the two
// trees and roots in the same instructions and the conversions on the integer pipe; the same values bit for bit.
constexpr int kPrepWarps = 8;

// (float)x, rounded to nearest even, without the conversion instruction where the result is a normal number.
__device__ __forceinline__ float to_f32(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned a = hi & 0x7FFFFFFFu;
    if (a - (897u << 20) >= (1150u - 897u) << 20) return (float)x;  // subnormal, zero, large, infinite, NaN
    const unsigned f = (__funnelshift_l(lo, hi, 3) - (896u << 23)) & 0x7FFFFFFFu, rest = lo << 3;  // truncated; what is cut off
    const unsigned r = f + (rest > 0x80000000u || (rest == 0x80000000u && (f & 1u)));
    return __uint_as_float(r | (hi & 0x80000000u));
}

__global__ void __launch_bounds__(32 * kPrepWarps) k_net_prep(int64_t nelt, const double* __restrict__ r,
                                                               const double* __restrict__ minv,
                                                               float* __restrict__ xin, float* __restrict__ scale)
{
    const int lane = threadIdx.x & 31;
    for (int64_t e = (int64_t)blockIdx.x * kPrepWarps + (threadIdx.x >> 5); e < nelt;
         e += (int64_t)gridDim.x * kPrepWarps) {
        double rv[NP / 32], jv[NP / 32];
#pragma unroll
        for (int q = 0; q < NP / 32; q++) {
            const int64_t o = e * NP + lane + 32 * q;
            rv[q] = r[o];
            jv[q] = minv[o] * rv[q];
        }
        double a = 0.0, b = 0.0;
#pragma unroll
        for (int q = 0; q < NP / 32; q++) {
            a += rv[q] * rv[q];
            b += jv[q] * jv[q];
        }
        // the two shuffle trees in one: after the first step (the same pairs of lanes as in a tree of their own) lanes
        // below 16 go on with a, the others with b
        const bool up = lane >= 16;
        const double other = __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
        double t = (up ? b : a) + other;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        double inv = 0.0;
        if ((lane & 15) == 0) {  // both roots and quotients by the same instructions
            const double rms = sqrt(t / NP);
            inv = rms > 0.0 ? 1.0 / rms : 0.0;
            if (up) scale[e] = (float)rms;
        }
        const double ia = __shfl_sync(0xffffffffu, inv, 0), ib = __shfl_sync(0xffffffffu, inv, 16);
#pragma unroll
        for (int q = 0; q < NP / 32; q++) {
            xin[(e * CIN + 0) * NP + lane + 32 * q] = to_f32(rv[q] * ia);
            xin[(e * CIN + 1) * NP + lane + 32 * q] = to_f32(jv[q] * ib);
        }
    }
}

// ------------------------------------------------------------------ inference
struct ApplySmem {
    float x[CIN * NP];
    float a1[CH * NP];
    float a2[CH * NP];
    float w1[CIN * 27 * CH];
    float w2[CH * 27 * CH];
    float w3[CH * 27];
    float b1[CH], b2[CH], b3[4];
};

// z[e][p] = net(xin[e])[p] * scale[e] * c[e][p] (FP64 out).  NP/2 threads per
// element, each computing points p and p + NP/2.
constexpr int NT_APPLY = NP / 2;
__global__ void __launch_bounds__(NT_APPLY) k_net_apply(int64_t nelt, const float* __restrict__ theta,
                                                        const float* __restrict__ xin,
                                                        const float* __restrict__ scale,
                                                        const double* __restrict__ c, double* __restrict__ z)
{
    extern __shared__ __align__(16) unsigned char raw[];
    ApplySmem& S = *reinterpret_cast<ApplySmem*>(raw);
    stage_weights<CIN, CH>(theta + OW1, S.w1);
    stage_weights<CH, CH>(theta + OW2, S.w2);
    stage_weights<CH, 1>(theta + OW3, S.w3);
    if (threadIdx.x < CH) {
        S.b1[threadIdx.x] = bf16r(theta[OB1 + threadIdx.x]);
        S.b2[threadIdx.x] = bf16r(theta[OB2 + threadIdx.x]);
    }
    if (threadIdx.x == 0) S.b3[0] = bf16r(theta[OB3]);
    const int p = threadIdx.x, p1 = p + NT_APPLY;
    const int i = p % NXN, j = (p / NXN) % NXN, k = p / (NXN * NXN);  // k in [0, 4)
    for (int64_t e = blockIdx.x; e < nelt; e += gridDim.x) {
        __syncthreads();
        S.x[p] = xin[(e * CIN + 0) * NP + p];
        S.x[p1] = xin[(e * CIN + 0) * NP + p1];
        S.x[NP + p] = xin[(e * CIN + 1) * NP + p];
        S.x[NP + p1] = xin[(e * CIN + 1) * NP + p1];
        __syncthreads();
        {
            float a0[CH], a1[CH];
            conv_2pts<CIN, CH>(S.x, S.w1, S.b1, i, j, k, a0, a1);
#pragma unroll
            for (int o = 0; o < CH; o++) {
                S.a1[o * NP + p] = gelu(a0[o]);
                S.a1[o * NP + p1] = gelu(a1[o]);
            }
        }
        __syncthreads();
        {
            float a0[CH], a1[CH];
            conv_2pts<CH, CH>(S.a1, S.w2, S.b2, i, j, k, a0, a1);
#pragma unroll
            for (int o = 0; o < CH; o++) {
                S.a2[o * NP + p] = gelu(a0[o]);
                S.a2[o * NP + p1] = gelu(a1[o]);
            }
        }
        __syncthreads();
        float y0[1], y1[1];
        conv_2pts<CH, 1>(S.a2, S.w3, S.b3, i, j, k, y0, y1);
        z[e * NP + p] = (double)y0[0] * (double)scale[e] * c[e * NP + p];
        z[e * NP + p1] = (double)y1[0] * (double)scale[e] * c[e * NP + p1];
    }
}

// ------------------------------------------------------------------ training
//
// The convolutions and their gradients work on lines of 8 points along i.  A thread holds a line of one input
// channel in registers and feeds 22 multiply-adds (three taps along i, the zero padding at its ends left out) from it
// for each of four output channels: 88 multiply-adds for five 16-byte shared-memory loads (convolution), or 22 for each of
// 16 channel pairs from 16 loads (weight gradient).  A block is one sample and a quarter of the output channels, 256
// threads, so that a batch of 256 spreads evenly (1024 blocks over 152 SMs) and a small one still fills the chip; the
// 16 input channels are shared out over four groups of 64 threads, whose sums are added through shared memory.
//
// What bounds it: the FP32 pipe (12 M multiply-adds a sample and their recomputed part, 80 us a batch of 256 at the
// pipe's rate).  A batch of 256: forward 62 + 10 us, backward 15 + 96 us, a whole energy-norm gradient 209 us; one block of 512
// threads a sample, one point or one 4 x 4 tile of channel pairs a thread, took 91, 536 and 654 us.
constexpr int NTT = 256;    // threads of the training kernels: 64 lines x 4 groups
constexpr int CS = 520;     // floats of one channel in shared memory: 64 lines and a zero line
constexpr int kZeroLine = 512;

// The two 16-byte halves of a line are exchanged in lines j = 4..7, so that eight lanes on consecutive lines meet all banks:
// place of the first half (float index; the second is at ^ 4).
__device__ __forceinline__ int line_at(int j, int k) { return 8 * (j + 8 * k) + ((j & 4) ? 4 : 0); }
// The nine neighbours (dj, dk) of line (j, k); the zero line outside the element.
__device__ __forceinline__ void line_neighbours(int j, int k, int (&off)[9])
{
#pragma unroll
    for (int q = 0; q < 9; q++) {
        const int jj = j + q % 3 - 1, kk = k + q / 3 - 1;
        off[q] = jj >= 0 && jj < 8 && kk >= 0 && kk < 8 ? line_at(jj, kk) : kZeroLine;
    }
}
__device__ __forceinline__ void line_load(const float* s, int at, float (&x)[8])
{
    const float4 a = *reinterpret_cast<const float4*>(s + at), b = *reinterpret_cast<const float4*>(s + (at ^ 4));
    x[0] = a.x, x[1] = a.y, x[2] = a.z, x[3] = a.w;
    x[4] = b.x, x[5] = b.y, x[6] = b.z, x[7] = b.w;
}
__device__ __forceinline__ void line_store(float* s, int at, const float (&x)[8])
{
    *reinterpret_cast<float4*>(s + at) = make_float4(x[0], x[1], x[2], x[3]);
    *reinterpret_cast<float4*>(s + (at ^ 4)) = make_float4(x[4], x[5], x[6], x[7]);
}
__device__ __forceinline__ void line_load_global(const float* g, float (&x)[8])
{
#pragma unroll
    for (int i = 0; i < 8; i++) x[i] = g[i];
}

// The same for the workspace's arrays, which are 16-byte aligned.
__device__ __forceinline__ void line_load_ws(const float* g, float (&x)[8])
{
    const float4 a = *reinterpret_cast<const float4*>(g), b = *reinterpret_cast<const float4*>(g + 4);
    x[0] = a.x, x[1] = a.y, x[2] = a.z, x[3] = a.w;
    x[4] = b.x, x[5] = b.y, x[6] = b.z, x[7] = b.w;
}
__device__ __forceinline__ void line_store_ws(float* g, const float (&x)[8])
{
    *reinterpret_cast<float4*>(g) = make_float4(x[0], x[1], x[2], x[3]);
    *reinterpret_cast<float4*>(g + 4) = make_float4(x[4], x[5], x[6], x[7]);
}

// acc[o][p] += sum over the CN channels from s on and the 27 taps of w x: four output channels of one line.  sW:
// [channel][dj, dk][di][4 outputs].
template <int CN>
__device__ __forceinline__ void conv4(const float* s, const float* sW, const int (&off)[9], float (&acc)[4][8])
{
#pragma unroll 1
    for (int c = 0; c < CN; c++) {
#pragma unroll
        for (int q = 0; q < 9; q++) {
            float x[8];
            line_load(s + c * CS, off[q], x);
            const float4* wq = reinterpret_cast<const float4*>(sW) + (c * 9 + q) * 3;
            const float4 wm = wq[0], w0 = wq[1], wp = wq[2];
            const float m[4] = {wm.x, wm.y, wm.z, wm.w}, z[4] = {w0.x, w0.y, w0.z, w0.w}, n[4] = {wp.x, wp.y, wp.z, wp.w};
#pragma unroll
            for (int o = 0; o < 4; o++)
#pragma unroll
                for (int p = 0; p < 8; p++) {
                    if (p > 0) acc[o][p] = fmaf(m[o], x[p - 1], acc[o][p]);
                    acc[o][p] = fmaf(z[o], x[p], acc[o][p]);
                    if (p < 7) acc[o][p] = fmaf(n[o], x[p + 1], acc[o][p]);
                }
        }
    }
}

// acc[di] += sum_p g[p] x[p + di] over one line.
__device__ __forceinline__ void corr3(const float (&g)[8], const float (&x)[8], float (&acc)[3])
{
#pragma unroll
    for (int p = 0; p < 8; p++) {
        if (p > 0) acc[0] = fmaf(g[p], x[p - 1], acc[0]);
        acc[1] = fmaf(g[p], x[p], acc[1]);
        if (p < 7) acc[2] = fmaf(g[p], x[p + 1], acc[2]);
    }
}

// Sums the four groups' acc of output channel `grp` through red (4 x 4 x 512 floats); every thread gets its line of it.
__device__ __forceinline__ void group_sum(float* red, int grp, int at, const float (&acc)[4][8], float (&out)[8])
{
    __syncthreads();
#pragma unroll
    for (int o = 0; o < 4; o++) line_store(red + (grp * 4 + o) * 512, at, acc[o]);
    __syncthreads();
#pragma unroll
    for (int p = 0; p < 8; p++) out[p] = 0.f;
#pragma unroll
    for (int g = 0; g < 4; g++) {
        float x[8];
        line_load(red + (g * 4 + grp) * 512, at, x);
#pragma unroll
        for (int p = 0; p < 8; p++) out[p] += x[p];
    }
}

// Weights of four outputs o0 .. o0 + 3 over CI channels as [channel][dj, dk][di][4]; FLIP: the taps of the transposed
// convolution, with W's roles exchanged (W[channel][o] read at the mirrored tap).
template <int CI, bool FLIP>
__device__ __forceinline__ void stage_conv4(const float* __restrict__ W, int o0, int nin, float* sW)
{
    for (int q = threadIdx.x; q < CI * 27 * 4; q += NTT) {
        const int o = o0 + (q & 3), t = (q >> 2) % 27, c = q / 108;
        sW[q] = bf16r(FLIP ? W[(c * nin + o) * 27 + 26 - t] : W[(o * nin + c) * 27 + t]);
    }
}

struct Fwd12Smem {
    float a1[CH * CS];  // later the group sums
    float x[CIN * CS];
    float w1[4 * CIN * 108];
    float w2[CH * 108];
    float b1[CH], b2[4];
};

// Layers 1 and 2 of sample blockIdx.x / 4; writes channels 4 q .. 4 q + 3 (q = blockIdx.x % 4) of the pre-activations h1, h2.
__global__ void __launch_bounds__(NTT, 3) k_net_fwd12(const float* __restrict__ theta, const float* __restrict__ xin,
                                                      float* __restrict__ h1, float* __restrict__ h2)
{
    extern __shared__ __align__(16) unsigned char raw[];
    Fwd12Smem& S = *reinterpret_cast<Fwd12Smem*>(raw);
    const int64_t b = blockIdx.x >> 2;
    const int part = blockIdx.x & 3, tid = threadIdx.x, grp = tid >> 6, l = tid & 63, j = l & 7, k = l >> 3;
    for (int g = 0; g < 4; g++) stage_conv4<CIN, false>(theta + OW1, 4 * g, CIN, S.w1 + g * CIN * 108);
    stage_conv4<CH, false>(theta + OW2, 4 * part, CH, S.w2);
    if (tid < CH) S.b1[tid] = bf16r(theta[OB1 + tid]);
    if (tid < 4) S.b2[tid] = bf16r(theta[OB2 + 4 * part + tid]);
    const int at = line_at(j, k);
    if (grp < CIN) {
        float v[8];
        line_load_global(xin + (b * CIN + grp) * NP + 8 * l, v);
        line_store(S.x + grp * CS, at, v);
    }
    if (tid < CIN * 8) S.x[(tid >> 3) * CS + kZeroLine + (tid & 7)] = 0.f;
    if (tid < CH * 8) S.a1[(tid >> 3) * CS + kZeroLine + (tid & 7)] = 0.f;
    int off[9];
    line_neighbours(j, k, off);
    __syncthreads();
    float acc[4][8];
#pragma unroll
    for (int o = 0; o < 4; o++)
#pragma unroll
        for (int p = 0; p < 8; p++) acc[o][p] = S.b1[4 * grp + o];
    conv4<CIN>(S.x, S.w1 + grp * CIN * 108, off, acc);
#pragma unroll
    for (int o = 0; o < 4; o++) {
        if (grp == part) line_store_ws(h1 + (b * CH + 4 * grp + o) * NP + 8 * l, acc[o]);
#pragma unroll
        for (int p = 0; p < 8; p++) acc[o][p] = gelu(acc[o][p]);
        line_store(S.a1 + (4 * grp + o) * CS, at, acc[o]);
    }
    __syncthreads();
#pragma unroll
    for (int o = 0; o < 4; o++)
#pragma unroll
        for (int p = 0; p < 8; p++) acc[o][p] = 0.f;
    conv4<4>(S.a1 + 4 * grp * CS, S.w2 + 4 * grp * 108, off, acc);
    float out[8];
    group_sum(S.a1, grp, at, acc, out);
    const float bias = S.b2[grp];
#pragma unroll
    for (int p = 0; p < 8; p++) out[p] += bias;
    line_store_ws(h2 + (b * CH + 4 * part + grp) * NP + 8 * l, out);
}

struct Fwd3Smem {
    float a2[CH * CS];
    float red[4 * 512];
    float w3[CH * 28];  // [channel][tap], padded
    float b3[4];
};

// Layer 3 of sample blockIdx.x: y from the pre-activations h2.
__global__ void __launch_bounds__(NTT) k_net_fwd3(const float* __restrict__ theta, const float* __restrict__ h2,
                                                  float* __restrict__ y)
{
    extern __shared__ __align__(16) unsigned char raw[];
    Fwd3Smem& S = *reinterpret_cast<Fwd3Smem*>(raw);
    const int64_t b = blockIdx.x;
    const int tid = threadIdx.x, grp = tid >> 6, l = tid & 63, j = l & 7, k = l >> 3, at = line_at(j, k);
    for (int q = tid; q < CH * 27; q += NTT) S.w3[q / 27 * 28 + q % 27] = bf16r(theta[OW3 + q]);
    if (tid == 0) S.b3[0] = bf16r(theta[OB3]);
    if (tid < CH * 8) S.a2[(tid >> 3) * CS + kZeroLine + (tid & 7)] = 0.f;
#pragma unroll
    for (int a = 0; a < 4; a++) {
        float v[8];
        line_load_ws(h2 + (b * CH + 4 * grp + a) * NP + 8 * l, v);
#pragma unroll
        for (int p = 0; p < 8; p++) v[p] = gelu(v[p]);
        line_store(S.a2 + (4 * grp + a) * CS, at, v);
    }
    int off[9];
    line_neighbours(j, k, off);
    __syncthreads();
    float acc[8] = {};
#pragma unroll 1
    for (int c = 4 * grp; c < 4 * grp + 4; c++) {
#pragma unroll
        for (int q = 0; q < 9; q++) {
            float x[8];
            line_load(S.a2 + c * CS, off[q], x);
            const float* w = S.w3 + c * 28 + 3 * q;
#pragma unroll
            for (int p = 0; p < 8; p++) {
                if (p > 0) acc[p] = fmaf(w[0], x[p - 1], acc[p]);
                acc[p] = fmaf(w[1], x[p], acc[p]);
                if (p < 7) acc[p] = fmaf(w[2], x[p + 1], acc[p]);
            }
        }
    }
    line_store(S.red + grp * 512, at, acc);
    __syncthreads();
    for (int q = tid; q < NP; q += NTT) {
        const int i = q & 7, jj = (q >> 3) & 7, a = line_at(jj, q >> 6), r = (i < 4 ? a : a ^ 4) + (i & 3);
        y[b * NP + q] = ((S.red[r] + S.red[512 + r]) + (S.red[1024 + r] + S.red[1536 + r])) + S.b3[0];
    }
}

// Per sample: loss_b = |y - t|^2 / |t|^2 ; dy = (2/B) (y - t) / |t|^2.
__global__ void __launch_bounds__(NP) k_net_loss(int B, const float* __restrict__ y, const float* __restrict__ t,
                                                 float* __restrict__ dy, float* __restrict__ loss_b)
{
    __shared__ float sh[2][NP / 32];
    const int p = threadIdx.x;
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
        const float d = y[(int64_t)b * NP + p] - t[(int64_t)b * NP + p];
        const float tv = t[(int64_t)b * NP + p];
        float a = d * d, c = tv * tv;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        if ((p & 31) == 0) {
            sh[0][p >> 5] = a;
            sh[1][p >> 5] = c;
        }
        __syncthreads();
        float num = 0.f, den = 0.f;
        for (int q = 0; q < NP / 32; q++) {
            num += sh[0][q];
            den += sh[1][q];
        }
        __syncthreads();
        den = den > 0.f ? den : 1.f;
        dy[(int64_t)b * NP + p] = 2.f / (float)B * d / den;
        if (p == 0) loss_b[b] = num / den;
    }
}

// d = y - t (FP32, in place into d)
__global__ void k_net_diff(int64_t n, const float* __restrict__ y, const float* __restrict__ t, float* __restrict__ d)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
        d[q] = y[q] - t[q];
}

// Per sample: loss_b = d.Ad / t.At ; dy = (2/B) Ad / t.At  (A = the sample element's operator).
__global__ void __launch_bounds__(NP) k_net_energy_loss(int B, const float* __restrict__ d, const float* __restrict__ Ad,
                                                        const float* __restrict__ t, const float* __restrict__ At,
                                                        float* __restrict__ dy, float* __restrict__ loss_b)
{
    __shared__ float sh[2][NP / 32];
    const int p = threadIdx.x;
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
        const int64_t o = (int64_t)b * NP + p;
        float a = d[o] * Ad[o], c = t[o] * At[o];
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, s);
            c += __shfl_xor_sync(0xffffffffu, c, s);
        }
        if ((p & 31) == 0) {
            sh[0][p >> 5] = a;
            sh[1][p >> 5] = c;
        }
        __syncthreads();
        float num = 0.f, den = 0.f;
        for (int q = 0; q < NP / 32; q++) {
            num += sh[0][q];
            den += sh[1][q];
        }
        __syncthreads();
        den = den > 0.f ? den : 1.f;
        dy[o] = 2.f / (float)B * Ad[o] / den;
        if (p == 0) loss_b[b] = num / den;
    }
}

// Weight-gradient tasks: (dj, dk) x channel tile x line group, 9 x 4 x 7 of the 256 threads.  A tile holds the
// channels ct, ct + 4, ct + 8, ct + 12, which lie on different banks.
constexpr int kLineGroups = 7;

struct Bwd3Smem {
    float a2[CH * CS];
    float dy[CS];
    float w3[4 * 108];
    float red[36 * 12 * kLineGroups];
    float sum[NTT / 32];
};

// Backward of layer 3 of sample blockIdx.x: dW3, db3 into gs, and h2 (the pre-activations) replaced by
// dh2 = gelu'(h2) convT(dy; W3).
__global__ void __launch_bounds__(NTT, 2) k_net_bwd3(const float* __restrict__ theta, const float* __restrict__ dy,
                                                     float* __restrict__ h2, float* __restrict__ gs)
{
    extern __shared__ __align__(16) unsigned char raw[];
    Bwd3Smem& S = *reinterpret_cast<Bwd3Smem*>(raw);
    const int64_t b = blockIdx.x;
    float* g = gs + b * NPARAM;
    const int tid = threadIdx.x, grp = tid >> 6, l = tid & 63, j = l & 7, k = l >> 3, at = line_at(j, k);
    // [group][dj, dk][di][4 channels] of the mirrored taps
    for (int q = tid; q < 4 * 108; q += NTT) {
        const int c = 4 * (q / 108) + (q & 3), t = (q % 108) >> 2;
        S.w3[q] = bf16r(theta[OW3 + c * 27 + 26 - t]);
    }
    float sdy = 0.f;
    if (grp == 0) {
        float v[8];
        line_load_ws(dy + b * NP + 8 * l, v);
        line_store(S.dy, at, v);
#pragma unroll
        for (int p = 0; p < 8; p++) sdy += v[p];
    }
    if (tid < 8) S.dy[kZeroLine + tid] = 0.f;
    if (tid < CH * 8) S.a2[(tid >> 3) * CS + kZeroLine + (tid & 7)] = 0.f;
    float gp[4][8];
#pragma unroll
    for (int a = 0; a < 4; a++) {
        float v[8];
        line_load_ws(h2 + (b * CH + 4 * grp + a) * NP + 8 * l, v);
#pragma unroll
        for (int p = 0; p < 8; p++) {
            gp[a][p] = gelu_grad(v[p]);
            v[p] = gelu(v[p]);
        }
        line_store(S.a2 + (4 * grp + a) * CS, at, v);
    }
    if (grp == 0) {  // db3: two warps
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sdy += __shfl_xor_sync(0xffffffffu, sdy, o);
        if ((tid & 31) == 0) S.sum[tid >> 5] = sdy;
    }
    int off[9];
    line_neighbours(j, k, off);
    __syncthreads();
    if (tid == 0) g[OB3] = S.sum[0] + S.sum[1];
    {
        float acc[4][8] = {};
        conv4<1>(S.dy, S.w3 + grp * 108, off, acc);
#pragma unroll
        for (int a = 0; a < 4; a++) {
#pragma unroll
            for (int p = 0; p < 8; p++) acc[a][p] *= gp[a][p];
            line_store_ws(h2 + (b * CH + 4 * grp + a) * NP + 8 * l, acc[a]);
        }
    }
    // dW3[c][t] = sum_p dy a2(p + t)
    if (tid < 36 * kLineGroups) {
        const int ct = tid & 3, q = (tid >> 2) % 9, lg = tid / 36, dj = q % 3 - 1, dk = q / 3 - 1;
        float acc[4][3] = {};
#pragma unroll 1
        for (int m = lg; m < 64; m += kLineGroups) {
            const int jj = (m & 7) + dj, kk = (m >> 3) + dk;
            const int xo = jj >= 0 && jj < 8 && kk >= 0 && kk < 8 ? line_at(jj, kk) : kZeroLine;
            float gv[8];
            line_load(S.dy, line_at(m & 7, m >> 3), gv);
#pragma unroll
            for (int a = 0; a < 4; a++) {
                float x[8];
                line_load(S.a2 + (ct + 4 * a) * CS, xo, x);
                corr3(gv, x, acc[a]);
            }
        }
#pragma unroll
        for (int a = 0; a < 4; a++)
#pragma unroll
            for (int d = 0; d < 3; d++) S.red[lg * 432 + (ct + 4 * a) * 27 + 3 * q + d] = acc[a][d];
    }
    __syncthreads();
    for (int q = tid; q < CH * 27; q += NTT) {
        float v = 0.f;
#pragma unroll
        for (int lg = 0; lg < kLineGroups; lg++) v += S.red[lg * 432 + q];
        g[OW3 + q] = v;
    }
}

struct Bwd12Smem {
    float g2[CH * CS];  // dh2
    float a1[CH * CS];  // gelu(h1); later the partial sums
    float x[CIN * CS];
    float g1[4 * CS];   // dh1, this quarter's channels
    float w2[CH * 108];
};
static_assert(36 * 24 * kLineGroups <= CH * CS && 16 * 512 <= CH * CS && 9 * 24 * 28 <= CH * CS, "partial sums fit");

// Backward of layers 2 and 1 of sample blockIdx.x / 4 for a quarter q = blockIdx.x % 4 of the channels: dW2 and db2 of the
// outputs 4 q .. 4 q + 3, and dh1 = gelu'(h1) convT(dh2; W2), dW1 and db1 of the hidden channels 4 q .. 4 q + 3.
__global__ void __launch_bounds__(NTT, 2)
    k_net_bwd12(const float* __restrict__ theta, const float* __restrict__ xin, const float* __restrict__ h1,
                const float* __restrict__ dh2, float* __restrict__ gs)
{
    extern __shared__ __align__(16) unsigned char raw[];
    Bwd12Smem& S = *reinterpret_cast<Bwd12Smem*>(raw);
    const int64_t b = blockIdx.x >> 2;
    float* g = gs + b * NPARAM;
    const int part = blockIdx.x & 3, tid = threadIdx.x, grp = tid >> 6, l = tid & 63, j = l & 7, k = l >> 3;
    const int at = line_at(j, k);
    stage_conv4<CH, true>(theta + OW2, 4 * part, CH, S.w2);
    if (grp < CIN) {
        float v[8];
        line_load_global(xin + (b * CIN + grp) * NP + 8 * l, v);
        line_store(S.x + grp * CS, at, v);
    }
    if (tid < CIN * 8) S.x[(tid >> 3) * CS + kZeroLine + (tid & 7)] = 0.f;
    if (tid < CH * 8) {
        S.g2[(tid >> 3) * CS + kZeroLine + (tid & 7)] = 0.f;
        S.a1[(tid >> 3) * CS + kZeroLine + (tid & 7)] = 0.f;
    }
#pragma unroll 2
    for (int a = 0; a < 4; a++) {
        float v[8];
        line_load_ws(dh2 + (b * CH + 4 * grp + a) * NP + 8 * l, v);
        line_store(S.g2 + (4 * grp + a) * CS, at, v);
        line_load_ws(h1 + (b * CH + 4 * grp + a) * NP + 8 * l, v);
#pragma unroll
        for (int p = 0; p < 8; p++) v[p] = gelu(v[p]);
        line_store(S.a1 + (4 * grp + a) * CS, at, v);
    }
    __syncthreads();
    // ---- dW2[o][c][t] = sum_p dh2[o] a1[c](p + t): four outputs x a tile of four channels x three taps a thread
    const int ct = tid & 3, q9 = (tid >> 2) % 9, lg = tid / 36, dj = q9 % 3 - 1, dk = q9 / 3 - 1;
    {
        float acc[4][4][3] = {};
        if (tid < 36 * kLineGroups) {
#pragma unroll 1
            for (int m = lg; m < 64; m += kLineGroups) {
                const int jj = (m & 7) + dj, kk = (m >> 3) + dk;
                const int xo = jj >= 0 && jj < 8 && kk >= 0 && kk < 8 ? line_at(jj, kk) : kZeroLine;
                const int go = line_at(m & 7, m >> 3);
                float gv[4][8];
#pragma unroll
                for (int o = 0; o < 4; o++) line_load(S.g2 + (4 * part + o) * CS, go, gv[o]);
#pragma unroll
                for (int a = 0; a < 4; a++) {
                    float x[8];
                    line_load(S.a1 + (ct + 4 * a) * CS, xo, x);
#pragma unroll
                    for (int o = 0; o < 4; o++) corr3(gv[o], x, acc[o][a]);
                }
            }
        }
#pragma unroll
        for (int h = 0; h < 2; h++) {  // two outputs at a time through the space of a1
            __syncthreads();
            if (tid < 36 * kLineGroups) {
#pragma unroll
                for (int o = 0; o < 2; o++)
#pragma unroll
                    for (int a = 0; a < 4; a++)
#pragma unroll
                        for (int d = 0; d < 3; d++)
                            S.a1[lg * 864 + (o * CH + ct + 4 * a) * 27 + 3 * q9 + d] = acc[2 * h + o][a][d];
            }
            __syncthreads();
            for (int q = tid; q < 864; q += NTT) {
                float v = 0.f;
#pragma unroll
                for (int n = 0; n < kLineGroups; n++) v += S.a1[n * 864 + q];
                g[OW2 + (4 * part + 2 * h) * CH * 27 + q] = v;
            }
        }
    }
    // ---- dh1 of this quarter
    {
        int off[9];
        line_neighbours(j, k, off);
        float acc[4][8] = {};
        conv4<4>(S.g2 + 4 * grp * CS, S.w2 + 4 * grp * 108, off, acc);
        float out[8], hv[8];
        group_sum(S.a1, grp, at, acc, out);
        line_load_ws(h1 + (b * CH + 4 * part + grp) * NP + 8 * l, hv);
#pragma unroll
        for (int p = 0; p < 8; p++) out[p] *= gelu_grad(hv[p]);
        line_store(S.g1 + grp * CS, at, out);
    }
    __syncthreads();
    // ---- biases: a warp for each of the quarter's channels of dh2 and dh1
    {
        const int w = tid >> 5, lane = tid & 31;
        const float* src = w < 4 ? S.g2 + (4 * part + w) * CS : S.g1 + (w - 4) * CS;
        float v = 0.f;
#pragma unroll
        for (int q = 0; q < NP / 32; q++) v += src[lane + 32 * q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) g[w < 4 ? OB2 + 4 * part + w : OB1 + 4 * part + w - 4] = v;
    }
    // ---- dW1[o][c][t] = sum_p dh1[o] x[c](p + t): all 24 of a (dj, dk) a thread, 28 line groups
    if (tid < 9 * 28) {
        const int q = tid % 9, n = tid / 9, d1 = q % 3 - 1, d2 = q / 3 - 1;
        float acc[4][CIN][3] = {};
#pragma unroll 1
        for (int m = n; m < 64; m += 28) {
            const int jj = (m & 7) + d1, kk = (m >> 3) + d2;
            const int xo = jj >= 0 && jj < 8 && kk >= 0 && kk < 8 ? line_at(jj, kk) : kZeroLine;
            const int go = line_at(m & 7, m >> 3);
            float x[CIN][8];
#pragma unroll
            for (int c = 0; c < CIN; c++) line_load(S.x + c * CS, xo, x[c]);
#pragma unroll
            for (int o = 0; o < 4; o++) {
                float gv[8];
                line_load(S.g1 + o * CS, go, gv);
#pragma unroll
                for (int c = 0; c < CIN; c++) corr3(gv, x[c], acc[o][c]);
            }
        }
#pragma unroll
        for (int o = 0; o < 4; o++)
#pragma unroll
            for (int c = 0; c < CIN; c++)
#pragma unroll
                for (int d = 0; d < 3; d++) S.a1[n * 216 + (o * CIN + c) * 27 + 3 * q + d] = acc[o][c][d];
    }
    __syncthreads();
    for (int q = tid; q < 4 * CIN * 27; q += NTT) {
        float v = 0.f;
#pragma unroll
        for (int n = 0; n < 28; n++) v += S.a1[n * 216 + q];
        g[OW1 + 4 * part * CIN * 27 + q] = v;
    }
}

// grad[q] = sum_b gs[b][q], loss = sum_b loss_b / B: 32 parameters a block, the samples shared out over eight warps
// (warp w takes b = w, w + 8, ...), whose sums are added in order.  The loads' latency is what a thread waits
// for: 256 samples one after the other took 17 us.
constexpr int kReduceWarps = 8;
__global__ void __launch_bounds__(32 * kReduceWarps) k_net_reduce(int B, const float* __restrict__ gs,
                                                                  const float* __restrict__ loss_b,
                                                                  float* __restrict__ grad, float* __restrict__ loss)
{
    __shared__ float sh[2][kReduceWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, q = blockIdx.x * 32 + lane;
    const bool with_loss = blockIdx.x == 0 && loss;
    float s = 0.f, sl = 0.f;
    if (q < NPARAM) {
#pragma unroll 16
        for (int b = w; b < B; b += kReduceWarps) s += gs[(int64_t)b * NPARAM + q];
    }
    if (with_loss && lane == 0) {
#pragma unroll 16
        for (int b = w; b < B; b += kReduceWarps) sl += loss_b[b];
    }
    sh[0][w][lane] = s;
    sh[1][w][lane] = sl;
    __syncthreads();
    if (w == 0) {
        for (int k = 1; k < kReduceWarps; k++) {
            s += sh[0][k][lane];
            sl += sh[1][k][lane];
        }
        if (q < NPARAM) grad[q] = s;
        if (with_loss && lane == 0) loss[0] = sl / (float)B;
    }
}

__global__ void k_adam(int n, float* __restrict__ th, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const float gq = g[q];
    const float mq = b1 * m[q] + (1.f - b1) * gq;
    const float vq = b2 * v[q] + (1.f - b2) * gq * gq;
    m[q] = mq;
    v[q] = vq;
    th[q] -= lr * (mq / c1) / (sqrtf(vq / c2) + eps);
}

std::atomic<uint64_t> g_apply_conf{0}, g_fwd12_conf{0}, g_fwd3_conf{0}, g_bwd3_conf{0}, g_bwd12_conf{0};

int grid_for(int64_t n) { return static_cast<int>(n < 152 * 2 ? n : 152 * 2); }

// Forward pass of a batch, keeping the pre-activations.
nek_status launch_train_forward(int batch, const float* theta, const float* xin, float* h1, float* h2, float* y,
                                cudaStream_t s)
{
    nek_status st = ensure_dyn_smem(k_net_fwd12, sizeof(Fwd12Smem), g_fwd12_conf);
    if (st == NEK_OK) st = ensure_dyn_smem(k_net_fwd3, sizeof(Fwd3Smem), g_fwd3_conf);
    if (st != NEK_OK) return st;
    k_net_fwd12<<<4u * (unsigned)batch, NTT, sizeof(Fwd12Smem), s>>>(theta, xin, h1, h2);
    k_net_fwd3<<<(unsigned)batch, NTT, sizeof(Fwd3Smem), s>>>(theta, h2, y);
    return check_launch();
}

// Backward pass from dy: each sample's gradient into gs; h2 is overwritten.  Then the sums over the batch.
nek_status launch_train_backward(int batch, const float* theta, const float* xin, const float* h1, float* h2,
                                 const float* dy, float* gs, const float* lossb, float* grad, float* loss,
                                 cudaStream_t s)
{
    nek_status st = ensure_dyn_smem(k_net_bwd3, sizeof(Bwd3Smem), g_bwd3_conf);
    if (st == NEK_OK) st = ensure_dyn_smem(k_net_bwd12, sizeof(Bwd12Smem), g_bwd12_conf);
    if (st != NEK_OK) return st;
    k_net_bwd3<<<(unsigned)batch, NTT, sizeof(Bwd3Smem), s>>>(theta, dy, h2, gs);
    k_net_bwd12<<<4u * (unsigned)batch, NTT, sizeof(Bwd12Smem), s>>>(theta, xin, h1, h2, gs);
    k_net_reduce<<<(NPARAM + 31) / 32, 32 * kReduceWarps, 0, s>>>(batch, gs, lossb, grad, loss);
    return check_launch();
}

}  // namespace

nek_status launch_net_apply(int64_t nelt, const float* theta, const float* xin, const float* scale, const double* c,
                            double* z, cudaStream_t s)
{
    nek_status st = ensure_dyn_smem(k_net_apply, sizeof(ApplySmem), g_apply_conf);
    if (st != NEK_OK) return st;
    k_net_apply<<<static_cast<int>(nelt < 152 * 2 ? nelt : 152 * 2), NT_APPLY, sizeof(ApplySmem), s>>>(nelt, theta,
                                                                                                  xin, scale, c, z);
    return check_launch();
}

// target[e][p] = (xs - xk)[e][p] / scale[e] (FP64 difference and quotient, one FP32 rounding); 0 where
// the element's scale is 0.
__global__ void k_net_target(int64_t n, const double* __restrict__ xs, const double* __restrict__ xk,
                             const float* __restrict__ scale, float* __restrict__ target)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const double s = (double)scale[q / NP];
        target[q] = s > 0.0 ? (float)((xs[q] - xk[q]) / s) : 0.f;
    }
}

nek_status launch_net_prep(int64_t nelt, const double* r, const double* minv, float* xin, float* scale,
                           cudaStream_t s)
{
    const int64_t nb = (nelt + kPrepWarps - 1) / kPrepWarps;
    k_net_prep<<<static_cast<int>(nb < 152 * 16 ? nb : 152 * 16), 32 * kPrepWarps, 0, s>>>(nelt, r, minv, xin, scale);
    return check_launch();
}

}  // namespace nek

using namespace nek;

namespace {

inline size_t al256(size_t b) { return (b + 255) & ~size_t(255); }

struct TrainLayout {
    float *h1, *h2, *y, *dy, *lossb, *gs, *d, *Ad, *At;
    size_t bytes;
};

TrainLayout train_layout(char* base, int B)
{
    TrainLayout L{};
    size_t off = 0;
    auto take = [&](size_t n) {
        char* q = base ? base + off : nullptr;
        off += al256(n);
        return reinterpret_cast<float*>(q);
    };
    L.h1 = take(sizeof(float) * (size_t)B * CH * NP);
    L.h2 = take(sizeof(float) * (size_t)B * CH * NP);
    L.y = take(sizeof(float) * (size_t)B * NP);
    L.dy = take(sizeof(float) * (size_t)B * NP);
    L.lossb = take(sizeof(float) * (size_t)B);
    L.gs = take(sizeof(float) * (size_t)B * NPARAM);
    L.d = take(sizeof(float) * (size_t)B * NP);
    L.Ad = take(sizeof(float) * (size_t)B * NP);
    L.At = take(sizeof(float) * (size_t)B * NP);
    L.bytes = off;
    return L;
}

}  // namespace

extern "C" {

int nek_net_param_count(void) { return NPARAM; }

nek_status nek_net_prep(int64_t nelt, int nx, const double* r, const double* minv, float* xin, float* scale,
                        void* stream)
{
    if (nx != NXN) return NEK_ERR_UNSUPPORTED_NX;
    if (nelt < 0) return NEK_ERR_INVALID_ARG;
    if (nelt == 0) return NEK_OK;
    if (!r || !minv || !xin || !scale) return NEK_ERR_INVALID_ARG;
    return launch_net_prep(nelt, r, minv, xin, scale, static_cast<cudaStream_t>(stream));
}

nek_status nek_net_target(int64_t nelt, int nx, const double* xs, const double* xk, const float* scale,
                          float* target, void* stream)
{
    if (nx != NXN) return NEK_ERR_UNSUPPORTED_NX;
    if (nelt < 0) return NEK_ERR_INVALID_ARG;
    if (nelt == 0) return NEK_OK;
    if (!xs || !xk || !scale || !target) return NEK_ERR_INVALID_ARG;
    const int64_t n = nelt * NP;
    k_net_target<<<pcg::stream_blocks(n), 256, 0, static_cast<cudaStream_t>(stream)>>>(n, xs, xk, scale, target);
    return check_launch();
}

nek_status nek_net_apply(int64_t nelt, int nx, const float* theta, const float* xin, const float* scale,
                         const double* c, double* z, void* stream)
{
    if (nx != NXN) return NEK_ERR_UNSUPPORTED_NX;
    if (nelt < 0) return NEK_ERR_INVALID_ARG;
    if (nelt == 0) return NEK_OK;
    if (!theta || !xin || !scale || !c || !z) return NEK_ERR_INVALID_ARG;
    return launch_net_apply(nelt, theta, xin, scale, c, z, static_cast<cudaStream_t>(stream));
}

size_t nek_net_train_workspace_bytes(int batch) { return batch > 0 ? train_layout(nullptr, batch).bytes : 0; }

nek_status nek_net_forward_batch(int batch, const float* theta, const float* xin, float* y, void* workspace,
                                 void* stream)
{
    if (batch <= 0 || !theta || !xin || !y || !workspace || !is_aligned(workspace, 256)) return NEK_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    TrainLayout L = train_layout(static_cast<char*>(workspace), batch);
    return launch_train_forward(batch, theta, xin, L.h1, L.h2, y, s);
}

nek_status nek_net_train_grad(int batch, const float* theta, const float* xin, const float* target, float* grad,
                              float* loss, void* workspace, void* stream)
{
    if (batch <= 0 || !theta || !xin || !target || !grad || !workspace || !is_aligned(workspace, 256))
        return NEK_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    TrainLayout L = train_layout(static_cast<char*>(workspace), batch);
    const nek_status st = launch_train_forward(batch, theta, xin, L.h1, L.h2, L.y, s);
    if (st != NEK_OK) return st;
    k_net_loss<<<grid_for(batch), NP, 0, s>>>(batch, L.y, target, L.dy, L.lossb);
    return launch_train_backward(batch, theta, xin, L.h1, L.h2, L.dy, L.gs, L.lossb, grad, loss, s);
}

nek_status nek_net_train_grad_energy(int batch, const float* theta, const float* xin, const float* target,
                                     const double* D, const float* Glp32, const float* gscale, float* grad,
                                     float* loss, void* workspace, void* stream)
{
    if (batch <= 0 || !theta || !xin || !target || !D || !Glp32 || !gscale || !grad || !workspace ||
        !is_aligned(workspace, 256))
        return NEK_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    TrainLayout L = train_layout(static_cast<char*>(workspace), batch);
    const int64_t n = (int64_t)batch * NP;
    nek_status st = launch_train_forward(batch, theta, xin, L.h1, L.h2, L.y, s);
    if (st != NEK_OK) return st;
    k_net_diff<<<pcg::stream_blocks(n), 256, 0, s>>>(n, L.y, target, L.d);
    if ((st = check_launch()) != NEK_OK) return st;
    if ((st = launch_ax_lowp(NEK_PREC_F32, batch, NXN, D, Glp32, gscale, L.d, L.Ad, s)) != NEK_OK) return st;
    if ((st = launch_ax_lowp(NEK_PREC_F32, batch, NXN, D, Glp32, gscale, target, L.At, s)) != NEK_OK) return st;
    k_net_energy_loss<<<grid_for(batch), NP, 0, s>>>(batch, L.d, L.Ad, target, L.At, L.dy, L.lossb);
    return launch_train_backward(batch, theta, xin, L.h1, L.h2, L.dy, L.gs, L.lossb, grad, loss, s);
}

nek_status nek_adam_step(int n, float* theta, const float* grad, float* m, float* v, float lr, float beta1,
                         float beta2, float eps, int step, void* stream)
{
    if (n <= 0 || !theta || !grad || !m || !v || step < 1 || !(lr > 0.f)) return NEK_ERR_INVALID_ARG;
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    k_adam<<<(n + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(n, theta, grad, m, v, lr, beta1, beta2,
                                                                           eps, c1, c2);
    return check_launch();
}

}  // extern "C"
