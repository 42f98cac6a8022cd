// Learned-preconditioner inference on the 5th-generation tensor cores (tcgen05):
// BF16 operands in shared memory, FP32 accumulators in tensor memory (TMEM).
//
// Each 3x3x3 convolution of the per-element network is an implicit GEMM whose rows are the lines of points along i.
// Two elements at a time make one M = 128 tile: row m = 8 (2 k + e) + j is line (j, k) of element e.  The
// activations of point i of every line lie together,
//     point i, K half h, padded plane kk = k + 1, element e, padded line jj = j + 1:
//     16-byte row (8 BF16 channels) at 5184 i + 2592 h + 144 (2 kk + e) + 16 jj,
// on a zero-padded grid of (jj, kk) whose last zero line and plane are the next one's first, so the A operand of a
// tap (dj, dk) is one descriptor with the strides LBO = 2592 B, SBO = 144 B, shifted by
// 16 (1 + dj) + 288 (1 + dk).  The three taps along i go to N: the MMA of input point i multiplies by a 16 x 48
// operand (di = +1, 0, -1) into the TMEM columns of the output points i - 1, i and i + 1 (16 channels each, 128 columns
// a tile): 78 MMAs a layer and two elements, where one MMA per tap takes 270 of N = 16.  An MMA of so few columns takes
// the time to read its 4 KB of A from shared memory, so the reads are what counts.  Every output still sums its 27 taps
// in the order (dk, dj, di), one MMA each: the sums are bit-identical to those of one MMA per tap.  The first (dj, dk)
// overwrites: the point i + 1 that an MMA reaches first is a 16-column MMA of its own there.
//
// A CTA has four groups of eight warps, each with its own tile (41 KB of activations, 128 TMEM columns) and
// mbarrier; the weights (41 KB) are shared.  A group is a chain of MMAs, wait and epilogue per layer; the groups'
// chains overlap.  One CTA per SM, persistent over pairs of elements.
//
// The epilogue reads each thread's TMEM lane (one line) with tcgen05.ld, adds the bias, applies GELU in FP32,
// rounds to BF16 and writes the rows back in place (the next layer's input; every MMA of the layer has
// completed by then).  The last layer writes z = y * scale * c in FP64.
//
// What bounds it (13 824 elements, 362 us against 975 before; 320 TFLOP/s of useful work; tensor pipe 33 %, issue
// 53 %): the MMAs alone, with the GELUs left out, take 263 us, about 50 cycles each for the 42 shared-memory wavefronts of
// their operands; the GELUs alone (25 instructions, ten of them on the half-rate ALU pipe) about 200 us of issue.  Three
// groups of four warps took 500 us, three of eight 440, four of eight 418, and 362 once one elected thread issues all MMAs
// with operands in uniform registers (20 instructions an MMA before, which the issuing warp did not get through between
// the GELUs).
//
// Numerics are those of nek_net_apply_bf16's contract: BF16 weights, the input
// and both hidden activations rounded to BF16 (nearest even) before each
// convolution, products exact and sums FP32 in the tensor core.
//
// Every wait on the mbarrier is bounded (~2 s of global time).  A wait that runs
// out sets a device flag (read by nek_fcg_solve_trunc, which returns
// NEK_ERR_TIMEOUT), writes NaN into the tile's outputs (so the solve that uses
// it stops on a non-finite value), waits once more and ends its group; the CTA then frees its TMEM and
// returns.
#include <cuda_bf16.h>

#include "nek_internal.h"
#include "nek_tc5.cuh"

namespace nek {

namespace {

constexpr int NP = 512, CIN = 2, CH = 16;
constexpr int NPARAM_TC5 = CH * CIN * 27 + CH + CH * CH * 27 + CH + CH * 27 + 1;
constexpr int OW1 = 0, OB1 = OW1 + CH * CIN * 27, OW2 = OB1 + CH, OB2 = OW2 + CH * CH * 27, OW3 = OB2 + CH,
              OB3 = OW3 + CH * 27;
constexpr int kGroups = 4, kGroupThreads = 256;  // eight warps: two per 32-lane TMEM sub-partition
constexpr int kLine8 = 144;                      // bytes between the two elements' groups of 8 lines (and a zero one)
constexpr int kPlane2 = 2 * kLine8;              // between planes
constexpr int kHalf = 9 * kPlane2;               // K half (8 channels) of one point's activations; the plane after it is the
constexpr int kPoint = 2 * kHalf;                // next one's zero plane
constexpr int kTile = 8 * kPoint + kPlane2 + 16;
constexpr int kTapHalf = 48 * 16, kTap = 2 * kTapHalf;  // B operand of one (dj, dk): [K half][n][8 channels]
constexpr uint32_t kHint = 1000;  // ns that a wait may sleep at a time
constexpr uint32_t kTmemCols = 128 * kGroups;
constexpr long long kWaitNs = 2000000000LL;             // default bound of every mbarrier wait

struct __align__(128) Tc5Smem {
    unsigned char w[3][9][kTap];
    unsigned char act[kGroups][kTile];
    float b1[16], b2[16], b3[4];
    unsigned long long mbar[kGroups];
    uint32_t tmem_base;
};

__device__ int g_net_tc5_timeout = 0;  // set by a bounded wait that ran out

__device__ __forceinline__ float gelu5(float v) { return 0.5f * v * (1.f + erff(v * 0.70710678118654752f)); }

// Barrier of one group (ids 1 ..), and the same with the disjunction of a predicate.
__device__ __forceinline__ void group_sync(int g)
{
    asm volatile("barrier.cta.sync %0, %1;" ::"r"(g + 1), "r"(kGroupThreads) : "memory");
}
__device__ __forceinline__ bool group_or(int g, bool v)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %3, 0;\n\t"
        "barrier.cta.red.or.pred q, %1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(r)
        : "r"(g + 1), "r"(kGroupThreads), "r"((uint32_t)v)
        : "memory");
    return r != 0;
}

// Channel 0 of four consecutive points of the lane (columns 0, 16, 32, 48 from t), loads and wait in one statement.
__device__ __forceinline__ void tmem_ld_points(uint32_t t, float (&y)[4])
{
    uint32_t r[4];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%4];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x1.b32 {%1}, [%5];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x1.b32 {%2}, [%6];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x1.b32 {%3}, [%7];\n\t"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3])
        : "r"(t), "r"(t + 16), "r"(t + 32), "r"(t + 48)
        : "memory");
#pragma unroll
    for (int i = 0; i < 4; i++) y[i] = __uint_as_float(r[i]);
}

// The MMAs of one layer (one elected thread): every tap of every point into the tile's 128 columns.
__device__ __forceinline__ void layer_mmas(uint32_t d, uint64_t a0, uint64_t b0)
{
    constexpr uint32_t i16 = tc5::idesc_bf16_f32(128, 16), i32 = tc5::idesc_bf16_f32(128, 32),
                       i48 = tc5::idesc_bf16_f32(128, 48);
    // the first (dj, dk): point i reaches output i + 1 for the first time
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const uint64_t a = a0 + (uint64_t)(i * (kPoint >> 4));
        if (i == 0)
            tc5::mma_bf16(d, a, b0 + 16, i32, 0u);  // outputs 0 and 1
        else {
            tc5::mma_bf16(d + 16u * (i - 1), a, b0, i32, 1u);  // outputs i - 1 and i
            if (i < 7) tc5::mma_bf16(d + 16u * (i + 1), a, b0 + 32, i16, 0u);
        }
    }
#pragma unroll 1
    for (int q = 1; q < 9; q++) {
        const uint64_t aq = a0 + (uint64_t)((q / 3) * (kPlane2 >> 4) + q % 3), b = b0 + (uint64_t)(q * (kTap >> 4));
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const uint64_t a = aq + (uint64_t)(i * (kPoint >> 4));
            if (i == 0)
                tc5::mma_bf16(d, a, b + 16, i32, 1u);
            else
                tc5::mma_bf16(d + 16u * (i - 1), a, b, i < 7 ? i48 : i32, 1u);
        }
    }
}

// arrivals: arrivals the mbarriers expect per phase (1: the commit of the MMAs;
// the self-test passes 2, which no phase ever gets, so every wait runs out).
__global__ void __launch_bounds__(kGroups* kGroupThreads, 1)
    k_net_apply_tc5(int64_t nelt, const float* __restrict__ theta, const float* __restrict__ xin,
                    const float* __restrict__ scale, const double* __restrict__ c, double* __restrict__ z,
                    long long wait_ns, int arrivals)
{
    extern __shared__ __align__(128) unsigned char raw5[];
    Tc5Smem& S = *reinterpret_cast<Tc5Smem*>(raw5);
    constexpr int NT = kGroups * kGroupThreads;
    const int tid = threadIdx.x, warp = tid >> 5, grp = tid / kGroupThreads;

    // ---- set-up: weights as BF16 B operands, zero grids, biases, mbarriers, TMEM
    for (int q = tid; q < 3 * 9 * 2 * 48 * 8; q += NT) {
        const int k8 = q & 7, n = (q >> 3) % 48, h = (q / (8 * 48)) & 1, t9 = (q / (16 * 48)) % 9, l = q / (16 * 48 * 9);
        const int ch = 8 * h + k8, o = n & 15, t = 3 * t9 + 2 - (n >> 4);  // n = 0..15: di = +1
        float v = 0.f;
        if (l == 0 && ch < CIN) v = theta[OW1 + (o * CIN + ch) * 27 + t];
        if (l == 1) v = theta[OW2 + (o * CH + ch) * 27 + t];
        if (l == 2 && o == 0) v = theta[OW3 + ch * 27 + t];
        reinterpret_cast<__nv_bfloat16*>(S.w)[q] = __float2bfloat16_rn(v);
    }
    for (int q = tid; q < kGroups * kTile / 16; q += NT) reinterpret_cast<uint4*>(S.act)[q] = make_uint4(0, 0, 0, 0);
    if (tid < CH) {
        S.b1[tid] = __bfloat162float(__float2bfloat16_rn(theta[OB1 + tid]));
        S.b2[tid] = __bfloat162float(__float2bfloat16_rn(theta[OB2 + tid]));
    }
    if (tid == 0) {
        S.b3[0] = __bfloat162float(__float2bfloat16_rn(theta[OB3]));
        for (int g = 0; g < kGroups; g++) tc5::mbar_init(tc5::smem_u32(&S.mbar[g]), arrivals);
    }
    if (warp == 0) tc5::tmem_alloc(&S.tmem_base, kTmemCols);
    tc5::fence_async_smem();
    tc5::fence_before();
    __syncthreads();
    tc5::fence_after();
    // warp-uniform by construction (broadcast from lane 0), so that the MMAs' operands live in uniform registers
    const int ugrp = __shfl_sync(0xffffffffu, grp, 0);
    const uint32_t tmem = __shfl_sync(0xffffffffu, S.tmem_base, 0), d_tile = tmem + 128u * (uint32_t)ugrp;
    const uint32_t mbar = tc5::smem_u32(&S.mbar[ugrp]);
    unsigned char* act = S.act[ugrp];
    const uint64_t a0 = tc5::smem_desc(tc5::smem_u32(act), kHalf, kLine8);  // tap (dj, dk) = (-1, -1) of point 0
    const uint64_t b0 = tc5::smem_desc(tc5::smem_u32(S.w), kTapHalf, 128);
    uint32_t parity = 0;
    // this thread's line (its TMEM lane m: element e of the pair, j, k), the four points i0 .. i0 + 3 of it, and the
    // place of its rows at point i0
    const int m = tid & 127, e = (m >> 3) & 1, j = m & 7, k = m >> 4, i0 = (tid >> 5) & 4;
    const uint32_t lane_addr = d_tile + ((uint32_t)(32 * (warp & 3)) << 16) + 16u * (uint32_t)i0;
    unsigned char* rows = act + kPoint * i0 + kPlane2 * (k + 1) + kLine8 * e + 16 * (j + 1);
    const bool vec = (reinterpret_cast<uintptr_t>(xin) & 15) == 0;
    const bool vecz = ((reinterpret_cast<uintptr_t>(z) | reinterpret_cast<uintptr_t>(c)) & 15) == 0;

    const int64_t npair = (nelt + 1) / 2, step = (int64_t)gridDim.x * kGroups;
    // the points' two input channels (zero where the pair has no second element)
    float x[2][4];
    auto load_line = [&](int64_t pair) {
        const int64_t el = 2 * pair + e;
#pragma unroll
        for (int ci = 0; ci < 2; ci++) {
            if (pair < npair && el < nelt) {
                const float* q = xin + (el * CIN + ci) * NP + 8 * (j + 8 * k) + i0;
                if (vec) {
                    const float4 u = __ldg(reinterpret_cast<const float4*>(q));
                    x[ci][0] = u.x, x[ci][1] = u.y, x[ci][2] = u.z, x[ci][3] = u.w;
                } else {
#pragma unroll
                    for (int i = 0; i < 4; i++) x[ci][i] = __ldg(q + i);
                }
            } else {
#pragma unroll
                for (int i = 0; i < 4; i++) x[ci][i] = 0.f;
            }
        }
    };
    int64_t pair = blockIdx.x + (int64_t)gridDim.x * grp;
    load_line(pair);
    for (; pair < npair; pair += step) {
        const int64_t el = 2 * pair + e;
        const bool live = el < nelt;
        // input: channels 0, 1 of the line's rows (rounded to BF16), channels 2..15 zero
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const __nv_bfloat162 x01 = __floats2bfloat162_rn(x[0][i], x[1][i]);
            *reinterpret_cast<uint4*>(rows + i * kPoint) =
                make_uint4(*reinterpret_cast<const uint32_t*>(&x01), 0u, 0u, 0u);
            *reinterpret_cast<uint4*>(rows + i * kPoint + kHalf) = make_uint4(0, 0, 0, 0);
        }
        bool failed = false;  // uniform across the group (decided by its barrier)
        for (int layer = 0; layer < 3; layer++) {
            tc5::fence_async_smem();  // the rows, written by this group's threads, are read by the tensor core
            tc5::fence_before();
            group_sync(grp);
            tc5::fence_after();
            if ((warp & 7) == 0) {
                if (tc5::elect_one()) {
                    layer_mmas(d_tile, a0, b0 + (uint64_t)(layer * (9 * kTap >> 4)));
                    tc5::mma_commit(mbar);
                }
                __syncwarp();
            }
            double2 cv[2];
            double sc = 0.0;
            if (layer == 2) {  // under the last layer's MMAs: the next pair's input, this pair's output factors
                load_line(pair + step);
                if (live) {
                    sc = (double)scale[el];
                    const double* cl = c + el * NP + 8 * (j + 8 * k) + i0;
#pragma unroll
                    for (int i = 0; i < 4; i += 2)
                        cv[i / 2] = vecz ? __ldg(reinterpret_cast<const double2*>(cl + i))
                                         : make_double2(__ldg(cl + i), __ldg(cl + i + 1));
                }
            }
            // the group's first warp waits for the MMAs, the others for it at the barrier
            const bool ok = (warp & 7) != 0 || tc5::mbar_wait_bounded(mbar, parity, wait_ns, kHint);
            if (group_or(grp, !ok)) {
                // a wait ran out: flag it, poison the pair's outputs, wait once more for the MMAs in
                // flight, then leave the loop (TMEM is freed below)
                failed = true;
                if (m == 0) atomicExch(&g_net_tc5_timeout, 1);
                if (j == 0 && k == 0 && i0 == 0 && live) z[el * NP] = __longlong_as_double(0x7FF8000000000000LL);
                tc5::mbar_wait_bounded(mbar, parity, wait_ns);
                break;
            }
            parity ^= 1u;
            __syncwarp();
            tc5::fence_after();
            if (layer < 2) {
                const float* b = layer == 0 ? S.b1 : S.b2;
#pragma unroll 1
                for (int i = 0; i < 4; i++) {
                    float v[16];
                    tc5::tmem_ld16(lane_addr + 16u * (uint32_t)i, v);
                    uint32_t packed[8];
#pragma unroll
                    for (int q = 0; q < 8; q++) {
                        const __nv_bfloat162 h2 =
                            __floats2bfloat162_rn(gelu5(v[2 * q] + b[2 * q]), gelu5(v[2 * q + 1] + b[2 * q + 1]));
                        packed[q] = *reinterpret_cast<const uint32_t*>(&h2);
                    }
                    *reinterpret_cast<uint4*>(rows + i * kPoint) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
                    *reinterpret_cast<uint4*>(rows + i * kPoint + kHalf) =
                        make_uint4(packed[4], packed[5], packed[6], packed[7]);
                }
            } else {
                float y[4];
                tmem_ld_points(lane_addr, y);
                if (live) {
                    double* zl = z + el * NP + 8 * (j + 8 * k) + i0;
#pragma unroll
                    for (int i = 0; i < 4; i += 2) {
                        const double2 v = make_double2((double)(y[i] + S.b3[0]) * sc * cv[i / 2].x,
                                                       (double)(y[i + 1] + S.b3[0]) * sc * cv[i / 2].y);
                        if (vecz)
                            *reinterpret_cast<double2*>(zl + i) = v;
                        else
                            zl[i] = v.x, zl[i + 1] = v.y;
                    }
                }
            }
            tc5::fence_before();
        }
        if (failed) break;
    }
    tc5::fence_before();
    __syncthreads();
    tc5::fence_after();
    if (warp == 0) tc5::tmem_dealloc(tmem, kTmemCols);
}

int sm_count()
{
    static int n = 0;
    if (!n) {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) ==
                                                      cudaSuccess && v > 0)
            n = v;
        else
            n = 152;
    }
    return n;
}

}  // namespace

nek_status launch_net_apply_tc5_ex(int64_t nelt, const float* theta, const float* xin, const float* scale,
                                   const double* c, double* z, cudaStream_t s, long long wait_ns, int arrivals)
{
    static std::atomic<uint64_t> configured{0};
    nek_status st = ensure_dyn_smem(k_net_apply_tc5, sizeof(Tc5Smem), configured);
    if (st != NEK_OK) return st;
    const int64_t npair = (nelt + 1) / 2, cap = sm_count();  // one CTA per SM, a pair for every SM before a second group's
    const int grid = static_cast<int>(npair < cap ? npair : cap);
    k_net_apply_tc5<<<grid, kGroups * kGroupThreads, sizeof(Tc5Smem), s>>>(nelt, theta, xin, scale, c, z, wait_ns,
                                                                          arrivals);
    return check_launch();
}

nek_status launch_net_apply_tc5(int64_t nelt, const float* theta, const float* xin, const float* scale,
                                const double* c, double* z, cudaStream_t s)
{
    return launch_net_apply_tc5_ex(nelt, theta, xin, scale, c, z, s, kWaitNs, 1);
}

// Reads and clears the flag that a bounded wait of the kernel ran out (synchronous).
nek_status net_tc5_take_timeout(bool* timed_out)
{
    int v = 0, zero = 0;
    nek_status st = check_cuda(cudaMemcpyFromSymbol(&v, g_net_tc5_timeout, sizeof(int)));
    if (st == NEK_OK && v) st = check_cuda(cudaMemcpyToSymbol(g_net_tc5_timeout, &zero, sizeof(int)));
    *timed_out = v != 0;
    return st;
}

}  // namespace nek

using namespace nek;

extern "C" {

nek_status nek_net_apply_bf16(int64_t nelt, int nx, const float* theta, const float* xin, const float* scale,
                              const double* c, double* z, void* stream)
{
    if (nx != 8) return NEK_ERR_UNSUPPORTED_NX;
    if (nelt < 0) return NEK_ERR_INVALID_ARG;
    if (nelt == 0) return NEK_OK;
    if (!theta || !xin || !scale || !c || !z || !is_aligned(xin, 4) || !is_aligned(z, 8) || !is_aligned(c, 8))
        return NEK_ERR_INVALID_ARG;
    return launch_net_apply_tc5(nelt, theta, xin, scale, c, z, static_cast<cudaStream_t>(stream));
}

nek_status nek_net_tc_selftest(int force_timeout, int64_t wait_us, int* timed_out)
{
    if (!timed_out || wait_us < 1 || wait_us > 2000000) return NEK_ERR_INVALID_ARG;
    *timed_out = 0;
    bool stale = false;
    nek_status st = net_tc5_take_timeout(&stale);  // clear a flag left by an earlier call
    if (st != NEK_OK) return st;
    // two elements with zero weights and inputs: z = 0 unless the wait ran out (then z[0] is NaN)
    const int64_t ne = 2;
    float* buf = nullptr;
    double* dbuf = nullptr;
    const size_t nf = NPARAM_TC5 + ne * CIN * NP + ne;
    if ((st = check_cuda(cudaMalloc(&buf, sizeof(float) * nf))) != NEK_OK) return NEK_ERR_NOMEM;
    if ((st = check_cuda(cudaMalloc(&dbuf, sizeof(double) * 2 * ne * NP))) != NEK_OK) {
        cudaFree(buf);
        return NEK_ERR_NOMEM;
    }
    st = check_cuda(cudaMemset(buf, 0, sizeof(float) * nf));
    if (st == NEK_OK) st = check_cuda(cudaMemset(dbuf, 0, sizeof(double) * 2 * ne * NP));
    if (st == NEK_OK)
        st = launch_net_apply_tc5_ex(ne, buf, buf + NPARAM_TC5, buf + NPARAM_TC5 + ne * CIN * NP, dbuf,
                                     dbuf + ne * NP, nullptr, wait_us * 1000LL, force_timeout ? 2 : 1);
    if (st == NEK_OK) st = check_cuda(cudaDeviceSynchronize());
    bool to = false;
    if (st == NEK_OK) st = net_tc5_take_timeout(&to);
    double z0 = 0.0;
    if (st == NEK_OK) st = check_cuda(cudaMemcpy(&z0, dbuf + ne * NP, sizeof(double), cudaMemcpyDeviceToHost));
    cudaFree(buf);
    cudaFree(dbuf);
    if (st != NEK_OK) return st;
    *timed_out = to ? 1 : 0;
    if (to != (z0 != z0)) return NEK_ERR_CUDA;  // the flag and the poisoned output must agree
    return to ? NEK_ERR_TIMEOUT : NEK_OK;
}

}  // extern "C"
