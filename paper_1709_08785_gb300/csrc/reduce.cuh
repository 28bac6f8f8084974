// Single-pass grid reduction with a deterministic order, and the BiCGStab
// scalar updates that its last block performs.
//
// Each block reduces its threads' values (warp shuffles, then one warp over
// the warp sums, the other warps leaving through a non-blocking barrier
// arrival) and writes one partial per block; all blocks but the last count
// themselves with a release add and retire, and the highest-indexed block
// (dispatched last) waits, bounded, for that count, adds the partials in
// block order and runs the finaliser on the solver state.  The sum order
// depends only on the launch shape, so results repeat bit for bit from run
// to run.  This replaces the paper's MPI_Allreduce of every dot product and
// norm (Sec. IV-B).
#pragma once

#include "ctx.cuh"

namespace qcd {

__device__ __forceinline__ bool finite_d(double x) { return isfinite(x); }

// The scalar recurrences of BiCGStab (Alg. 2, with alpha = rho0/<r~|q> and
// beta = (rho1/rho0)(alpha/omega), the standard reading of the printed
// formulas), run by one thread at the end of a grid reduction, on the
// critical path between two kernels: each quotient takes one FP64 division
// (a long dependent sequence on GB300, whose FP64 rate is 1/64 of FP32) and
// the breakdown test compares squares instead of taking square roots.
__device__ inline void finalize(int op, SolverState *st)
{
    const double *s = st->sum;
    switch (op) {
    case FIN_ALPHA: {
        const double dr = s[0], di = s[1];
        const double den = dr * dr + di * di;
        st->iter += 1;
        if (!(den > 0.0) || !finite_d(den)) {
            st->done = 1;
            st->status = finite_d(den) ? QCD_EBREAKDOWN : QCD_ENONFINITE;
            break;
        }
        const double inv = 1.0 / den;
        st->alpha[0] = (st->rho0[0] * dr + st->rho0[1] * di) * inv;
        st->alpha[1] = (st->rho0[1] * dr - st->rho0[0] * di) * inv;
        break;
    }
    case FIN_S:
        st->rr = s[0];
        if (!finite_d(s[0])) {
            st->done = 1;
            st->status = QCD_ENONFINITE;
        } else if (s[0] < st->tol2) {
            st->done = 1;
            st->status = QCD_OK;
            st->exit_half = 1;
        }
        break;
    case FIN_OMEGA: {
        const double tt = s[2];
        if (!(tt > 0.0) || !finite_d(tt) || !finite_d(s[0]) || !finite_d(s[1])) {
            st->done = 1;
            st->status = finite_d(tt) ? QCD_EBREAKDOWN : QCD_ENONFINITE;
            st->exit_half = 1;
            break;
        }
        const double inv = 1.0 / tt;
        st->omega[0] = s[0] * inv;
        st->omega[1] = s[1] * inv;
        if (st->omega[0] == 0.0 && st->omega[1] == 0.0) {
            st->done = 1;
            st->status = QCD_EBREAKDOWN;
            st->exit_half = 1;
        }
        break;
    }
    case FIN_X: {
        const double rr = s[0], r1r = s[1], r1i = s[2];
        st->rr = rr;
        st->exit_half = 0;
        if (!finite_d(rr) || !finite_d(r1r) || !finite_d(r1i)) {
            st->done = 1;
            st->status = QCD_ENONFINITE;
        } else if (rr < st->tol2) {
            st->done = 1;
            st->status = QCD_OK;
        } else if (st->bd_eps >= 0.0 && r1r * r1r + r1i * r1i <= st->bd_eps * st->bd_eps * (st->rt2 * rr)) {
            st->done = 1;
            st->status = QCD_EBREAKDOWN;
        } else if (st->iter >= st->maxit) {
            st->done = 1;
            st->status = QCD_ENOTCONV;
        } else {
            // beta = (rho1/rho0) * (alpha/omega) = (rho1 alpha) / (rho0 omega)
            const double nr = r1r * st->alpha[0] - r1i * st->alpha[1];
            const double ni = r1r * st->alpha[1] + r1i * st->alpha[0];
            const double dr = st->rho0[0] * st->omega[0] - st->rho0[1] * st->omega[1];
            const double di = st->rho0[0] * st->omega[1] + st->rho0[1] * st->omega[0];
            const double inv = 1.0 / (dr * dr + di * di);
            st->beta[0] = (nr * dr + ni * di) * inv;
            st->beta[1] = (ni * dr - nr * di) * inv;
            st->rho0[0] = r1r;
            st->rho0[1] = r1i;
        }
        break;
    }
    case FIN_INIT:
    case FIN_RESTART:
        // r = r~ = p = b: rho0 = |b|^2; a zero right-hand side is converged
        if (op == FIN_INIT && st->tol2_rel > 0.0) st->tol2 = st->tol2_rel * s[0];
        st->norm2[1] = s[0];
        st->rr = s[0];
        st->rt2 = s[0];
        st->rho0[0] = s[0];
        st->rho0[1] = 0.0;
        st->exit_half = 0;
        if (!finite_d(s[0])) {
            st->done = 1;
            st->status = QCD_ENONFINITE;
        } else if (s[0] <= st->tol2 || s[0] == 0.0) {
            st->done = 1;
            st->status = QCD_OK;
        } else {
            st->done = 0;
            st->status = QCD_OK;
        }
        break;
    default:
        if (op >= FIN_SETN && op < FIN_SETN + 4) st->norm2[op - FIN_SETN] = s[0];
        else if (op >= FIN_ADDN && op < FIN_ADDN + 4) st->norm2[op - FIN_ADDN] += s[0];
        break;
    }
    for (int k = 0; k < 2; ++k) {
        st->coef[k] = (float)st->alpha[k];
        st->coef[2 + k] = (float)st->omega[k];
        st->coef[4 + k] = (float)st->beta[k];
    }
}

// A sum beyond the warp, by the accumulator type A of the threads.  FP64 for
// the FP64 and DF64 levels.  For the FP32 and FP16 levels, whose warp sums are
// floats, a pair of floats (double-float, 2^-48): an FP64 instruction keeps a
// warp scheduler's FP64 lanes busy for 64 cycles, and the FP64 tree of a block and
// of its grid held each fused-dot kernel for some 2 us (two-level solves at one
// launch shape: 8^4 2.94 -> 2.58 ms, 12^3x24 4.42 -> 3.97, 24^3x48 17.65 -> 17.27).
// A pair's 2^-48 is far below the 2^-24 of the warp sums that it adds.  Its range is
// FP32's, so the warp sums enter times 2^-5 (up to 32 a block; exact down to
// 2^-121) and a grid's sum beyond 3.4e38 is taken again in FP64: only a warp sum
// itself can leave the range.  (Three-level solves at 4^4 and 8^4 with no care for
// the range 2.62 / 2.23 ms, so 2.63 / 2.21, with the FP64 sum inlined 2.66 / 2.25, with a
// check in every block instead of the factor 2% more at 16^3x32.)
template <class A>
struct WideOf {
    using type = double;
};
template <>
struct WideOf<float> {
    using type = df;
};
__device__ __forceinline__ double wide_shfl(double v, int off) { return __shfl_xor_sync(0xffffffffu, v, off); }
__device__ __forceinline__ df wide_shfl(df v, int off)
{
    return df(__shfl_xor_sync(0xffffffffu, v.hi, off), __shfl_xor_sync(0xffffffffu, v.lo, off));
}
// a partial in its 8-byte slot
__device__ __forceinline__ double wide_pack(double v) { return v; }
__device__ __forceinline__ double wide_pack(df v)
{
    return __hiloint2double(__float_as_int(v.hi), __float_as_int(v.lo));
}
// a warp sum as a term of the block's; a total back to its own scale, and
// whether it is finite there
__device__ __forceinline__ double wide_in(double v) { return v; }
__device__ __forceinline__ df wide_in(float v) { return df(v * 0x1p-5f); }
__device__ __forceinline__ bool wide_out(double v, double &sum)
{
    sum = v;
    return true;
}
__device__ __forceinline__ bool wide_out(df v, double &sum)
{
    const df t(v.hi * 0x1p5f, v.lo * 0x1p5f);
    sum = (double)t;
    return isfinite(t.hi);
}
template <class W>
__device__ __forceinline__ W wide_unpack(double d)
{
    if constexpr (std::is_same<W, df>::value)
        return df(__int_as_float(__double2hiint(d)), __int_as_float(__double2loint(d)));
    else return d;
}

// The sums over nw warps of the values src(warp, k), k < N <= 4, by one warp:
// lane 8 k + j adds the warps j, j + 8, ..., then three steps add the eight
// lanes of every k at once; all of lanes 8 k .. 8 k + 7 return sum k.
template <int N, class W, class Src>
__device__ __forceinline__ W warps_sum(int nw, const Src &src)
{
    const int lane = threadIdx.x + threadIdx.y * blockDim.x & 31, k = lane >> 3;
    W t = W(0.f);
    if (k < N)
        for (int w = lane & 7; w < nw; w += 8) t = t + src(w, k);
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) t = t + wide_shfl(t, off);
    return t;
}

// The grid's sums from the float-pair partials in FP64, lanes 8 k .. 8 k + 7 sum k
// (a function of its own and rolled: inlined, it slowed the path beside it)
template <int N>
__device__ __noinline__ double pairs_sum_slow(const double *partials, int nblk)
{
    const int lane = threadIdx.x + threadIdx.y * blockDim.x & 31, k = lane >> 3;
    double t = 0.0;
    if (k < N)
#pragma unroll 1
        for (int b = lane & 7; b < nblk; b += 8) t += (double)wide_unpack<df>(__ldcg(partials + (size_t)b * 4 + k));
#pragma unroll 1
    for (int off = 4; off > 0; off >>= 1) t += wide_shfl(t, off);
    return 32.0 * t;
}

// Reduce N values over the grid; blocks may be 1-D or 2-D.  The per-thread
// values and the warp stage are in the accumulator type A (float for the
// FP32 and FP16 levels, whose sums feed FP32 recurrences: GB300's FP64 rate
// is 1/64 of its FP32 rate, and per-thread FP64 adds slowed those kernels
// in proportion to their size); the warp sums and everything after are in
// WideOf<A>.
// bidx / nblk: the block's index among the nblk blocks of this reduction
// (blockIdx.x / gridDim.x, or another grid dimension when several
// reductions share one launch); the block with index nblk - 1 is dispatched
// after every other block of its reduction.
template <int N, class A>
__device__ __forceinline__ void grid_reduce_ex(A v[N], const RedArgs &ra, int bidx, int nblk)
{
    using W = typename WideOf<A>::type;
    __shared__ A sh[32][4];
    __shared__ double sw[32][4];
    __shared__ int last;
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int nthr = blockDim.x * blockDim.y;
    const int lane = tid & 31, wid = tid >> 5, nw = (nthr + 31) >> 5;
#pragma unroll
    for (int k = 0; k < N; ++k)
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], off);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < N; ++k) sh[wid][k] = v[k];
    const auto mine = [&](int w, int k) { return wide_in(sh[w][k]); };
    if (bidx != nblk - 1) {
        // Every block but the last: warps 1.. post their sums and leave at
        // once (bar.arrive does not wait; their output stores proceed), warp
        // 0 waits for them (bar.sync on the same named barrier), adds the
        // sums in warp order, writes the block's partial and counts it.
        // Nothing holds a block at a full-block barrier.
        if (wid != 0) {
            asm volatile("bar.arrive 1, %0;" ::"r"(nthr) : "memory");
            return;
        }
        asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
        const W t = warps_sum<N, W>(nw, mine);
        if ((lane & 7) == 0 && (lane >> 3) < N) ra.partials[(size_t)bidx * 4 + (lane >> 3)] = wide_pack(t);
        __syncwarp();
        if (lane == 0)  // the partial ordered before the count; no reply awaited
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ra.counter) : "memory");
        return;
    }
    // the solver state, a word a lane, on its way while the other blocks finish
    constexpr int WORDS = sizeof(SolverState) / 8;
    static_assert(sizeof(SolverState) % 8 == 0 && WORDS <= 32, "one warp moves the state");
    __shared__ double sst[WORDS];
    const double word = tid < WORDS ? __ldcg((const double *)ra.st + tid) : 0.0;
    __syncthreads();
    if (wid == 0) {
        const W t = warps_sum<N, W>(nw, mine);
        if ((lane & 7) == 0 && (lane >> 3) < N) ra.partials[(size_t)bidx * 4 + (lane >> 3)] = wide_pack(t);
        __syncwarp();
        if (lane == 0) {
            // the highest-indexed block is dispatched last: it waits
            // (bounded) until every other block has counted
            const unsigned want = (unsigned)nblk - 1;
            long long n = 0;
            unsigned got;
            for (;;) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(got) : "l"(ra.counter) : "memory");
                if (got >= want || ++n > (1ll << 26)) break;
                __nanosleep(32);
            }
            last = got >= want ? 1 : 0;
        }
    }
    __syncthreads();
    if (!last) {  // the other blocks never all counted: report, do not hang
        if (tid == 0) {
            ra.st->status = QCD_ETIMEOUT;
            ra.st->done = 1;
            *ra.counter = 0u;
            __threadfence();
        }
        return;
    }
    // the partials in rows of four 8-byte slots, two slots a thread; eight loads
    // in flight per thread, added as a tree
    const bool hi = tid & 1;
    const int rows = nthr >> 1;
    W s0 = W(0.f), s1 = W(0.f);
    if (N > 2 || !hi)
        for (int b0 = tid >> 1; b0 < nblk; b0 += 8 * rows) {
            double2 t[8];  // all zero bits are zero in either form
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int b = b0 + u * rows;
                t[u] = b < nblk ? __ldcg((const double2 *)ra.partials + (size_t)b * 2 + hi) : make_double2(0.0, 0.0);
            }
            W x[8], y[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                x[u] = wide_unpack<W>(t[u].x);
                y[u] = wide_unpack<W>(t[u].y);
            }
#pragma unroll
            for (int d = 4; d > 0; d >>= 1)
#pragma unroll
                for (int u = 0; u < d; ++u) {
                    x[u] = x[u] + x[u + d];
                    if (N > 1) y[u] = y[u] + y[u + d];
                }
            s0 = s0 + x[0];
            if (N > 1) s1 = s1 + y[0];
        }
#pragma unroll
    for (int off = 16; off > 1; off >>= 1) {
        s0 = s0 + wide_shfl(s0, off);
        if (N > 1) s1 = s1 + wide_shfl(s1, off);
    }
    if (lane < 2) {
        sw[wid][2 * lane] = wide_pack(s0);
        sw[wid][2 * lane + 1] = wide_pack(s1);
    }
    if (tid < WORDS) sst[tid] = word;
    __syncthreads();
    if (wid == 0) {
        const W t = warps_sum<N, W>(nw, [&](int w, int k) { return wide_unpack<W>(sw[w][k]); });
        double sum;
        const bool fin = wide_out(t, sum);
        if constexpr (std::is_same<W, df>::value)
            if (__any_sync(0xffffffffu, !fin))  // (rare)
                sum = pairs_sum_slow<N>(ra.partials, nblk);
        SolverState *st = (SolverState *)sst;
        if ((lane & 7) == 0) st->sum[lane >> 3] = (lane >> 3) < N ? sum : 0.0;
        __syncwarp();
        if (lane == 0) finalize(ra.op, st);
        __syncwarp();
        // no fence: the kernel ends here, and its completion publishes the
        // state and the counter to the next kernel in stream order
        if (lane < WORDS) ((double *)ra.st)[lane] = sst[lane];
        if (lane == 0) *ra.counter = 0u;
    }
}

template <int N, class A>
__device__ __forceinline__ void grid_reduce(A v[N], const RedArgs &ra)
{
    grid_reduce_ex<N, A>(v, ra, (int)blockIdx.x, (int)gridDim.x);
}

}  // namespace qcd
