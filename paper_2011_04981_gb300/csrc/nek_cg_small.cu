// The FP64 solve of few elements as one cooperative kernel.
//
// A Jacobi-PCG iteration on 64 elements of nx = 8 is 7 launches and a read-back of a few microseconds each around half a
// megabyte of work; it is bound by those.  Where every element can have a CTA of its own resident (nelt up to
// dx_small_blocks x SMs), one launch runs all iterations: r, x, minv and the point flags of a CTA's element stay in registers
// and its p in shared memory, the operator is k_ax_dx's, and the CTAs meet three times an iteration at a barrier in
// global memory:
//   w = A_e p to memory | each point sums its own copies of w (the plan's members, in dssum's order), partial <p,w> |
//   alpha, r, x, partials of <r,r> and <r,z> | beta, the residual test, p.
// Every CTA adds the same partials in the same order, so all hold the same scalars and take the same exit; the host reads
// them once.  The operations on a point are those of the kernels in nek_pcg.cuh.
//
// A call of 64 elements of nx = 8 takes 15.3 us an iteration (53 us as 7 launches and a read-back, 43 with a read-back every
// tenth); 456 elements of nx = 8 26 (60), 150 of nx = 5 16 (60), of nx = 16 57 (84), general loop timed with read-backs every
// tenth iteration and events; faster on every size that fits, so the rule is that it fits.  What bounds it is latency, in
// clocks of 32000 an iteration (64 elements, nx = 8): operator 10000, waits at the barriers 8500, sums over copies and
// <p,w> 5900, alpha 2300, updates 2300, beta 2600; an FP64 instruction holds a warp's pipe 64 of them.
#include "nek_ax_dx.cuh"
#include "nek_pcg.cuh"

namespace nek {
namespace pcg {

struct SmallArgs {
    int nelt;
    const double *D, *G, *minv;
    const uint8_t* flags;
    const int32_t* grp;  // group of each point or -1 (in the memory of w); null without groups
    const int32_t *off, *mem;
    const double *r0, *p0;
    double *x, *w, *pwparts, *parts;
    Scalars* sc;
    unsigned* bar;  // arrivals, zero at the start
    int max_iter;
    long long wait_ns;
};

// Iterations of one launch at most: about a second (1.1 s at nx = 16).
constexpr int kSmallMaxIter = 20000;

namespace {

constexpr int dx_small_blocks(int nx)
{
    const int by_smem = (int)((227 * 1024) / (sizeof(double) * 5 * nx * nx * nx + 5120));
    const int by_warps = 20 / (dx_threads(nx, 1, 1) / 32);
    const int b = by_smem < by_warps ? by_smem : by_warps;
    return b < 1 ? 1 : b;
}

__device__ __forceinline__ long long now_ns()
{
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The barrier of all CTAs, in two halves.  The launch is cooperative, so every CTA is resident and the wait is met; one
// that is not within wait_ns is false, which ends the kernel, and the general loop solves instead.
__device__ __forceinline__ void small_arrive(unsigned* bar)
{
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
}

__device__ __forceinline__ bool small_wait(unsigned* bar, unsigned target, long long wait_ns)
{
    bool late = false;
    if (threadIdx.x == 0) {
        long long t0 = 0;
        for (unsigned n = 1;; n++) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if ((int)(v - target) >= 0) break;
            if ((n & 63u) == 0u) {  // the clock is looked at from the 64th poll on (some 50 us)
                const long long t = now_ns();
                if (t0 == 0)
                    t0 = t;
                else if (t - t0 > wait_ns) {
                    late = true;
                    break;
                }
            }
        }
    }
    return !__syncthreads_or(late);
}

__device__ __forceinline__ bool small_barrier(unsigned* bar, unsigned target, long long wait_ns)
{
    small_arrive(bar);
    return small_wait(bar, target, wait_ns);
}

// Sum of n values by one warp, in a fixed order, in every lane; past the L1 (other CTAs wrote them).
__device__ __forceinline__ double small_sum(const double* __restrict__ v, int n)
{
    double t = 0.0;
#pragma unroll 4
    for (int q = threadIdx.x & 31; q < n; q += 32) t += __ldcg(v + q);
    return warp_tree(t);
}

// The group of every member of a plan's groups.
__global__ void k_point_groups(int64_t ngroups, const int32_t* __restrict__ off, const int32_t* __restrict__ mem,
                               int32_t* __restrict__ grp)
{
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < ngroups; g += (int64_t)gridDim.x * blockDim.x)
        for (int32_t m = off[g]; m < off[g + 1]; m++) grp[mem[m]] = (int32_t)g;
}

template <int NX>
__global__ void __launch_bounds__(dx_threads(NX, 1, 1), (dx_small_blocks(NX))) k_cg_small(SmallArgs A)
{
    using Grid = FxGrid<NX>;
    constexpr int NP = Grid::SIZE, N3 = NX * NX * NX;
    constexpr int TPE = dx_tpe(NX, 1), NB = dx_threads(NX, 1, 1), B = (N3 + TPE - 1) / TPE;
    static_assert(2 * NB <= 3 * NP && NB >= 64, "the sums' staging takes the place of A");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DxSmem<NX, 1>& S = *reinterpret_cast<DxSmem<NX, 1>*>(smem_raw);
    __shared__ Scalars sc;
    const int tid = threadIdx.x;
    const bool active = tid < TPE;
    const int t = active ? tid : 0;
    double* sh = S.A[0];
    if (tid == 0) sc = *A.sc;
    bool sym;
    const bool bad = dx_build<NX>(A.D, S.D, S.tab, tid, NB, sym);
    const DxLines<NX, 1> ln(S.U, S.A[0], NP, 0, t, sym);
    double* At[3];
#pragma unroll
    for (int d = 0; d < 3; d++) At[d] = S.A[d] + Grid::at(t);
    double* Ut = S.U + Grid::at(t);
    const int64_t e0 = blockIdx.x * (int64_t)N3;
    const double* Ge = A.G + e0 * 6;

    // this thread's points t, t + TPE, ...
    double x[B], r[B], mi[B];
    int ga[B], gn[B];  // its copies: mem[ga .. ga + gn), gn = 0 for a point without others
    unsigned fl = 0u;  // two flag bits a point
    auto has = [&](int b) { return active && (b < B - 1 || t + b * TPE < N3); };
    auto off = [&](int b) { return Grid::at(t + b * TPE) - Grid::at(t); };
#pragma unroll
    for (int b = 0; b < B; b++) {
        x[b] = r[b] = mi[b] = 0.0;
        ga[b] = gn[b] = 0;
        if (has(b)) {
            const int64_t q = e0 + t + b * TPE;
            r[b] = A.r0[q];
            mi[b] = A.minv[q];
            Ut[off(b)] = A.p0[q];
            fl |= (unsigned)(A.flags[q] & (kFree | kOwner)) << (2 * b);
            const int g = A.grp ? A.grp[q] : -1;
            if (g >= 0) {
                ga[b] = A.off[g];
                gn[b] = A.off[g + 1] - ga[b];
            }
        }
    }
    // thread 0: a residual norm^2 in (above, huge] is neither within the tolerance nor without a finite quotient; relres, with
    // its square root and division, is then formed at the end only
    const double bt = sc.tol * sc.bnorm, b2 = bt * bt, bh = sc.bnorm * 1e300;
    const double above = sc.tol == 0.0 ? 0.0 : b2 > 1e-280 ? b2 * (1.0 + 1e-13) : INFINITY, huge = fmin(bh * bh, 1e300);
    bool near = true;
    const int rshift = sc.rshift;
    unsigned target = gridDim.x;
    bool late = !small_barrier(A.bar, target, A.wait_ns);  // every CTA has read the map: w may be written
    for (int it = 0; it < A.max_iter && !late && !halted(&sc); it++) {
        // ---- w = A_e p
        if (active) dx_lines<NX, false, 1>(ln.u, ln.a, ln.str, ln.sgn, S.tab[0], S.D, sym, bad);
        __syncthreads();
        if (active) dx_geom<NX, TPE>(Ge, At, t);
        __syncthreads();
        if (active) dx_lines<NX, true, 1>(ln.in, ln.a, ln.str, ln.sgn, S.tab[1], S.D, sym, bad);
        __syncthreads();
        double w[B];
#pragma unroll
        for (int b = 0; b < B; b++) {
            w[b] = 0.0;
            if (has(b)) {
                w[b] = (At[0][off(b)] + At[1][off(b)]) + At[2][off(b)];
                if (gn[b]) A.w[e0 + t + b * TPE] = w[b];
            }
        }
        if ((late = !small_barrier(A.bar, target += gridDim.x, A.wait_ns))) break;
        // ---- dssum of the own points, <p,w>
        double pw[1] = {0.0}, o1[B];
#pragma unroll
        for (int b = 0; b < B; b++) {  // the first two copies of every point together
            o1[b] = 0.0;
            if (gn[b]) {
                w[b] = __ldcg(A.w + A.mem[ga[b]]);
                o1[b] = __ldcg(A.w + A.mem[ga[b] + 1]);
            }
        }
#pragma unroll
        for (int b = 0; b < B; b++) {
            if (gn[b]) {
                w[b] += o1[b];
                for (int o = 2; o < gn[b]; o += 2) {
                    const double v0 = __ldcg(A.w + A.mem[ga[b] + o]);
                    const double v1 = o + 1 < gn[b] ? __ldcg(A.w + A.mem[ga[b] + o + 1]) : 0.0;
                    w[b] += v0;
                    if (o + 1 < gn[b]) w[b] += v1;
                }
            }
            if (has(b) && (fl >> (2 * b) & 3u) == (kFree | kOwner)) pw[0] += Ut[off(b)] * w[b];
        }
        {
            const double v = block_sums<NB, 1>(pw, sh);
            if (tid == 0) A.pwparts[blockIdx.x] = v;
        }
        if ((late = !small_barrier(A.bar, target += gridDim.x, A.wait_ns))) break;
        if (tid < 32) {
            const double s = small_sum(A.pwparts, A.nelt);
            if (tid == 0) set_alpha(s, &sc);
        }
        __syncthreads();
        if (sc.status != NEK_OK) break;
        // ---- x, r, their sums
        const double alpha = sc.alpha;
        double v2[2] = {0.0, 0.0};
        float s_hi = 0.f, s_lo = 0.f, s_c = 0.f;  // <r,r> in float pairs, as in k_update
#pragma unroll
        for (int b = 0; b < B; b++) {
            if (has(b)) {
                const unsigned f = fl >> (2 * b);
                r[b] = fma(-alpha, f & kFree ? w[b] : 0.0, r[b]);
                if (f & kOwner) {
                    sq_pair_add(r[b], rshift, s_hi, s_lo, s_c);
                    v2[1] += r[b] * (mi[b] * r[b]);
                }
            }
        }
        v2[0] = (widen(s_hi) + widen(s_lo)) + widen(s_c);
        {
            const double v = block_sums<NB, 2>(v2, sh);
            if ((tid & 31) == 0 && tid < 64) A.parts[(tid >> 5) * A.nelt + blockIdx.x] = v;
        }
        small_arrive(A.bar);
#pragma unroll
        for (int b = 0; b < B; b++)
            if (has(b)) x[b] = fma(alpha, Ut[off(b)], x[b]);
        if ((late = !small_wait(A.bar, target += gridDim.x, A.wait_ns))) break;
        // the residual test and beta, the same operations as set_beta, one warp each
        if (tid < 32) {
            const double rr = small_sum(A.parts, A.nelt) * sc.rback;
            if (tid == 0) {
                sc.rr = rr;
                near = !(rr > above && rr <= huge);
                if (near) sc.relres = sqrt(rr) / sc.bnorm;
            }
        } else if (tid < 64) {
            const double rz = small_sum(A.parts + A.nelt, A.nelt);
            if (tid == 32) {
                sc.beta = rz / sc.rz;
                sc.rz = rz;
            }
        }
        __syncthreads();
        if (tid == 0) {
            if ((near && !isfinite(sc.relres)) || !isfinite(sc.rz)) {
                sc.status = NEK_ERR_BREAKDOWN;
                sc.iters = sc.it;
            } else if (near && sc.tol > 0.0 && sc.relres <= sc.tol) {
                sc.done = 1;
                sc.iters = sc.it;
            }
        }
        __syncthreads();
        // ---- the next direction
        if (!halted(&sc)) {
            const double beta = sc.beta;
#pragma unroll
            for (int b = 0; b < B; b++)
                if (has(b)) Ut[off(b)] = fma(beta, Ut[off(b)], mi[b] * r[b]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int b = 0; b < B; b++)
        if (has(b)) A.x[e0 + t + b * TPE] = x[b];
    if (blockIdx.x == 0 && tid == 0) {
        if (late) sc.status = NEK_ERR_CUDA;
        sc.xpend = 0;
        if (sc.it > 0) sc.relres = sqrt(sc.rr) / sc.bnorm;
        *A.sc = sc;
    }
}

template <int NX>
nek_status launch_small(const SmallArgs& a, cudaStream_t s, bool& ran)
{
    constexpr size_t smem = sizeof(DxSmem<NX, 1>);
    static_assert(dx_small_blocks(NX) * (smem + 1024 + 256) <= 228 * 1024, "the CTAs counted on are resident");
    static std::atomic<uint64_t> configured{0};
    nek_status st = ensure_dyn_smem(k_cg_small<NX>, smem, configured);
    if (st != NEK_OK) return st;
    SmallArgs args = a;
    void* params[] = {&args};
    const cudaError_t e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_cg_small<NX>), dim3((unsigned)a.nelt),
                                                      dim3(dx_threads(NX, 1, 1)), params, smem, s);
    if (e == cudaErrorCooperativeLaunchTooLarge) {  // fewer SMs than counted on: the general loop takes it
        cudaGetLastError();
        return NEK_OK;
    }
    ran = e == cudaSuccess;
    return check_cuda(e);
}

}  // namespace

nek_status run_small(const nek_gs* gs, int64_t nelt, int nx, const double* D, const double* G, const uint8_t* mask,
                     const double* minv, const uint8_t* flags, const double* f, double* x, const Buffers<double>& b,
                     double* edot, double tol, int max_iter, cudaStream_t s, Result* res, bool& ran, const double*& rhs,
                     const SmallWait& wait)
{
    ran = false;
    if (nx < 4 || nelt > (int64_t)kSMs * dx_small_blocks(nx) || nelt > kMaxReduceBlocks || max_iter > kSmallMaxIter)
        return NEK_OK;
    const int64_t n = nelt * nx * nx * nx;
    const int nb = reduce_blocks(n);
    static_assert(sizeof(Scalars) + sizeof(unsigned) <= 256, "the barrier's counter follows the scalars");
    SmallArgs a{};
    a.nelt = (int)nelt;
    a.D = D;
    a.G = G;
    a.minv = minv;
    a.flags = flags;
    a.r0 = b.r;
    a.p0 = b.p;
    a.x = x;
    a.w = b.w;
    a.pwparts = edot;
    a.parts = b.parts;
    a.sc = b.sc;
    a.bar = reinterpret_cast<unsigned*>(b.sc + 1);
    a.max_iter = max_iter;
    a.wait_ns = wait.ns;
    k_init<double><<<nb, NT, 0, s>>>(n, gs->d_c, mask, minv, f, x, b.r, b.p, b.parts, flags);
    k_init_finish<<<1, NT, 0, s>>>(b.parts, nb, tol, b.sc);
    rhs = b.r;  // masked f, which the kernel leaves as it is; f itself may lie where x is
    int launches = 2;
    // (for the self-test: the counter one short, so that no wait is met)
    nek_status st = check_cuda(cudaMemsetAsync(a.bar, wait.force_timeout ? 0xFF : 0, sizeof(unsigned), s));
    if (st != NEK_OK) return st;
    if (gs->ngroups > 0) {
        if ((st = check_cuda(cudaMemsetAsync(b.w, 0xFF, sizeof(int32_t) * n, s))) != NEK_OK) return st;
        k_point_groups<<<stream_blocks(gs->ngroups), 256, 0, s>>>(gs->ngroups, gs->d_offsets, gs->d_members,
                                                                  reinterpret_cast<int32_t*>(b.w));
        a.grp = reinterpret_cast<const int32_t*>(b.w);
        a.off = gs->d_offsets;
        a.mem = gs->d_members;
        launches++;
    }
    if ((st = check_launch()) != NEK_OK) return st;
    switch (nx) {
        case 4: st = launch_small<4>(a, s, ran); break;
        case 5: st = launch_small<5>(a, s, ran); break;
        case 6: st = launch_small<6>(a, s, ran); break;
        case 7: st = launch_small<7>(a, s, ran); break;
        case 8: st = launch_small<8>(a, s, ran); break;
        case 9: st = launch_small<9>(a, s, ran); break;
        case 10: st = launch_small<10>(a, s, ran); break;
        case 11: st = launch_small<11>(a, s, ran); break;
        case 12: st = launch_small<12>(a, s, ran); break;
        case 13: st = launch_small<13>(a, s, ran); break;
        case 14: st = launch_small<14>(a, s, ran); break;
        case 15: st = launch_small<15>(a, s, ran); break;
        case 16: st = launch_small<16>(a, s, ran); break;
        default: return NEK_OK;
    }
    res->launches = launches + (ran ? 1 : 0);
    if (st != NEK_OK || !ran) return st;
    Scalars h{};
    if ((st = check_cuda(cudaMemcpyAsync(&h, b.sc, sizeof(h), cudaMemcpyDeviceToHost, s))) != NEK_OK) return st;
    if ((st = check_cuda(cudaStreamSynchronize(s))) != NEK_OK) return st;
    if (h.status == NEK_ERR_CUDA) {
        ran = false;
        return NEK_OK;
    }
    return result_of(h, tol, res);
}

}  // namespace pcg
}  // namespace nek
