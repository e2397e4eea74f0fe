// Whole CG solves of small matrix-free systems in one launch (Section 7.5): a
// persistent cooperative kernel runs every phase of every iteration -- SpMV with
// p.q, residual update with r.r, solution and direction update -- for up to
// kCgSmallSystems systems at a time, with a grid barrier (gridbar.cuh) between
// phases.
//
// Three launches per iteration cost a small system far more than its work: at
// 64^3 an iteration took 33.8 us, most of it in the hundreds of blocks of each
// kernel queueing on the reduction's ticket, for 12 FP64 instructions per row
// on a pipe that does 0.6 T of them per second (5 us).  Here a block takes a
// contiguous range of the bricks (64 x 8 x 4 or 32 x 16 x 4 points) of the
// systems still running, every brick leaves one partial sum, and every block
// sums the partials of its own systems after the barrier, in brick order: no
// ticket, no last block, and the result does not depend on which block took
// which brick, so a system solved in a batch equals the same system alone bit
// for bit.  The SpMV is the exact-sum form (xsum.cuh): 5.6 FP64 instructions
// per row and iteration in all, where the row kernel's iteration takes 12.  x
// is updated together with p, which saves one read of p.  Rows of r, p and q
// have an even pitch, so every access is 16 bytes wide.
//
// Measured per iteration: 64^3 11.7 us (k_cg_one: latency of three barriers, two
// sums and the halo loads), 96^3 25.2, 128^3 44.9 (start: 33.8, 49.2, 73.2); 64
// systems of 22.9 M unknowns in all 149 ms, start 429: 1.8 x what their vectors'
// 80 bytes per row take at the copy rate, the FP64 pipe 55% and DRAM 43% busy --
// each phase waits on its loads part of the time.  Three blocks per SM (80
// registers, 152 bytes of spill); four (64 registers, more spill) took 155 ms.
//
// Vectors change hands between SMs from phase to phase, so they are read with
// ld.global.cg (L2), never through L1.
#include <algorithm>

#include "cg_small.cuh"
#include "gridbar.cuh"

namespace hcg {

namespace {

constexpr int kNT = kCgBlock, kKZ = kCgSmallKZ;
constexpr int kPlane = 680;   // shared words per plane: 10 rows of 68 or 18 of 36 (648)

// In alpha's place: A is not positive definite on p (p.q <= 0, or NaN).  alpha
// itself is never negative; it is 0 where p.q overflows and r.r does not, and
// the solve then goes on to max_iter, as with three launches per iteration.
constexpr double kBreakdown = -1.0;

// The thread's place in a brick of a system.
struct Place {
    int X, Y, k0;
    int nk;            // planes of the brick inside the grid
    int64_t at;        // index of the thread's first point in r, p and q (rows of `pitch`)
    int64_t dense;     // its index in x and b
    bool ok0, ok1;     // its two x points inside the grid
};

__device__ __forceinline__ Place place_of(const CgSmallSys& s, int brick, int tid)
{
    Place c;
    const int lpr = 1 << s.lg, rows = kNT >> s.lg;
    const int t = brick / s.tiles_x;
    const int x0 = (brick - t * s.tiles_x) * (2 * lpr);
    const int tz = t / s.tiles_y;
    c.X = x0 + 2 * (tid & (lpr - 1));
    c.Y = (t - tz * s.tiles_y) * rows + (tid >> s.lg);
    c.k0 = tz * kKZ;
    c.nk = min(kKZ, s.nz - c.k0);
    const int64_t line = (int64_t)c.k0 * s.ny + c.Y;
    c.at = line * s.pitch + c.X;
    c.dense = line * s.nx + c.X;
    c.ok0 = c.X < s.nx && c.Y < s.ny;
    c.ok1 = c.ok0 && c.X + 1 < s.nx;
    return c;
}

// Two consecutive values of r, p or q, zeros where !ok.  Their rows have an even
// pitch and start 16-byte aligned; the pad of an odd row holds zeros.
template <typename T>
__device__ __forceinline__ void ld_pair(const T* p, bool ok, T (&o)[2])
{
    using W = typename std::conditional<std::is_same<T, double>::value, double2, longlong2>::type;
    o[0] = o[1] = T(0);
    if (ok) {
        const W v = __ldcg(reinterpret_cast<const W*>(p));
        o[0] = v.x;
        o[1] = v.y;
    }
}

__device__ __forceinline__ void st_pair(double* p, bool ok, const double (&v)[2])
{
    if (ok) *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
}

// Two values of the caller's x: 16 bytes at a time when its rows allow.
__device__ __forceinline__ void ld_x(const double* p, bool vec, bool ok0, bool ok1, double (&o)[2])
{
    if (vec) return ld_pair(p, ok0, o);
    o[0] = ok0 ? __ldcg(p) : 0.0;
    o[1] = ok1 ? __ldcg(p + 1) : 0.0;
}

__device__ __forceinline__ void st_x(double* p, bool vec, bool ok0, bool ok1, const double (&v)[2])
{
    if (vec) return st_pair(p, ok0, v);
    if (ok0) p[0] = v[0];
    if (ok1) p[1] = v[1];
}

// Sum of 256 values in shared memory by one warp, a tree of eight levels; valid in lane 0.
__device__ __forceinline__ double warp_of_rows(const double* red)
{
    static_assert(kNT == 256, "eight rows of 32");
    const int lane = threadIdx.x & 31;
    double a[8];
#pragma unroll
    for (int w = 0; w < 8; ++w) a[w] = red[lane + 32 * w];
    double s = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    return s;
}

// The brick's sum of v over its 256 threads, in a fixed order, into *dst.  The
// threads' values meet in shared memory and one warp adds them (12 FP64
// instructions per brick instead of 43 by shuffles in every warp).  `red` is
// the buffer of this turn; callers alternate between two.
__device__ __forceinline__ void brick_sum(double v, double* red, int turn, double* dst)
{
    const int tid = threadIdx.x;
    red[tid] = v;
    __syncthreads();
    if ((tid >> 5) == (turn & 7)) {
        const double s = warp_of_rows(red);
        if ((tid & 31) == 0) *dst = s;
    }
}

// Sum of a system's brick partials in a fixed order, in thread 0 only: each
// thread its own strided partials, one warp the threads' sums.  (The FP64 pipe
// does one warp instruction in 16 cycles: a division or a shuffle tree in all
// eight warps of every block costs microseconds.)  All threads call it.
__device__ __forceinline__ double sys_sum(const double* part, int n, double* red)
{
    const int tid = threadIdx.x;
    double v = 0.0;
    if (tid < n) v = __ldcg(part + tid);
    for (int t = tid + kNT; t < n; t += kNT) v += __ldcg(part + t);
    red[tid] = v;
    __syncthreads();
    return tid < 32 ? warp_of_rows(red) : 0.0;
}

// Whether sqrt(rho) / ||b|| <= rtol; t2 = (rtol ||b||)^2 decides without a root
// and a division (a microsecond of one thread's FP64) unless rho is within
// rounding of it or t2 near the ends of the range.
__device__ __forceinline__ bool cg_stops(double rho, double bnorm, double rtol, double t2)
{
    if (t2 > 1e-280 && t2 < 1e280) {
        if (rho > t2 * (1.0 + 1e-12)) return false;
        if (rho < t2 * (1.0 - 1e-12)) return true;
    }
    return sqrt(rho) / bnorm <= rtol;
}

// q = A p on a brick; returns the thread's share of p.q.  CONV: the exact-sum
// form (emax = p's largest exponent field), else FP64 arithmetic.  REG: the
// thread's own values of p are in pv and q stays in qv; otherwise p is read and
// q written.
template <bool CONV, bool REG>
__device__ __forceinline__ double spmv_brick(const CgSmallSys& s, const Place& c, int emax, long long* sm,
                                             const double (&pv)[kKZ][2], double (&qv)[kKZ][2])
{
    const int tid = threadIdx.x;
    const int lpr = 1 << s.lg, rows = kNT >> s.lg;
    const int bw = 2 * lpr + 4, pl = (rows + 2) * bw;
    const int64_t sxy = (int64_t)s.pitch * s.ny;
    const long long* p = reinterpret_cast<const long long*>(s.p);
    const int lx = tid & (lpr - 1), row = tid >> s.lg;
    long long v[kKZ + 2][2];
#pragma unroll
    for (int q = 0; q < kKZ + 2; ++q) {
        if (REG && q > 0 && q <= kKZ) {
            v[q][0] = __double_as_longlong(pv[q - 1][0]);
            v[q][1] = __double_as_longlong(pv[q - 1][1]);
            continue;
        }
        const int k = c.k0 - 1 + q;
        const bool in = k >= 0 && k < s.nz;
        ld_pair(p + c.at + (q - 1) * sxy, in && c.ok0, v[q]);
    }
    // halo rows (sides 0, 1: a pair of each plane per thread) and columns
    const int yk = (tid >> s.lg) & (kKZ - 1), yside = tid >> (s.lg + 2);
    const int y0 = c.Y - row, x0 = c.X - 2 * lx;
    long long hy[2] = {0, 0}, hx = 0;
    if (yside < 2) {
        const int Yh = yside ? y0 + rows : y0 - 1;
        const bool in = Yh >= 0 && Yh < s.ny && yk < c.nk;
        ld_pair(p + ((int64_t)(c.k0 + yk) * s.ny + Yh) * s.pitch + c.X, in && c.X < s.nx, hy);
    }
    const int lr = 8 - s.lg;   // log2(rows)
    const int xr = tid & (rows - 1), xk = (tid >> lr) & (kKZ - 1), xside = tid >> (lr + 2);
    if (xside < 2) {
        const int Xh = xside ? x0 + 2 * lpr : x0 - 1;
        if (Xh >= 0 && Xh < s.nx && y0 + xr < s.ny && xk < c.nk)
            hx = __ldcg(p + ((int64_t)(c.k0 + xk) * s.ny + y0 + xr) * s.pitch + Xh);
    }
    auto fix = [emax](long long b) -> long long { return CONV ? xs_fix(b, emax) : b; };
    const int own = (row + 1) * bw + 2 + 2 * lx;
    long long u[kKZ + 2][2];
#pragma unroll
    for (int q = 0; q < kKZ + 2; ++q)
#pragma unroll
        for (int i = 0; i < 2; ++i) u[q][i] = fix(v[q][i]);
#pragma unroll
    for (int kk = 0; kk < kKZ; ++kk)
        *reinterpret_cast<longlong2*>(sm + kk * pl + own) = make_longlong2(u[kk + 1][0], u[kk + 1][1]);
    if (yside < 2)
        *reinterpret_cast<longlong2*>(sm + yk * pl + (yside ? rows + 1 : 0) * bw + 2 + 2 * lx) =
            make_longlong2(fix(hy[0]), fix(hy[1]));
    if (xside < 2) sm[xk * pl + (xr + 1) * bw + (xside ? 2 + 2 * lpr : 1)] = fix(hx);
    __syncthreads();
    double pq = 0.0;
#pragma unroll
    for (int kk = 0; kk < kKZ; ++kk) {
        if (!c.ok0 || kk >= c.nk) {
            qv[kk][0] = qv[kk][1] = 0.0;
            continue;
        }
        const long long* pc = sm + kk * pl + own;
        const longlong2 ymv = *reinterpret_cast<const longlong2*>(pc - bw);
        const longlong2 ypv = *reinterpret_cast<const longlong2*>(pc + bw);
        const long long ym[2] = {ymv.x, ymv.y}, yp[2] = {ypv.x, ypv.y};
        const long long left = pc[-1], right = pc[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const long long C = u[kk + 1][i], B = u[kk][i], Ab = u[kk + 2][i];
            const long long xm = i == 0 ? left : u[kk + 1][0], xp = i == 1 ? right : u[kk + 1][1];
            if constexpr (CONV) {
                const long long L = 6 * C - (((B + ym[i]) + (xm + xp)) + (yp[i] + Ab));
                qv[kk][i] = (i == 0 && (kk & 1) == 0) ? xs_unfix_dp(L, emax) : xs_unfix(L, emax);
            } else {
                auto d = [](long long b) { return __longlong_as_double(b); };
                const double sv = ((d(B) + d(ym[i])) + (d(xm) + d(xp))) + (d(yp[i]) + d(Ab));
                qv[kk][i] = __fma_rn(6.0, d(C), -sv);
            }
        }
        if (!c.ok1) qv[kk][1] = 0.0;
        if constexpr (!REG) st_pair(s.q + c.at + kk * sxy, true, qv[kk]);
        pq = __fma_rn(__longlong_as_double(v[kk + 1][0]), qv[kk][0], pq);
        pq = __fma_rn(__longlong_as_double(v[kk + 1][1]), qv[kk][1], pq);
    }
    return pq;
}

// (A v)[i, j, k] on the FP64 pipe, v read through L2 (start and true residual).
__device__ __forceinline__ double row_apply(const CgSmallSys& s, const double* v, int i, int j, int k, int64_t at)
{
    const int64_t sxy = (int64_t)s.nx * s.ny;
    const double zm = k > 0 ? __ldcg(v + at - sxy) : 0.0;
    const double ym = j > 0 ? __ldcg(v + at - s.nx) : 0.0;
    const double xm = i > 0 ? __ldcg(v + at - 1) : 0.0;
    const double xp = i < s.nx - 1 ? __ldcg(v + at + 1) : 0.0;
    const double yp = j < s.ny - 1 ? __ldcg(v + at + s.nx) : 0.0;
    const double zp = k < s.nz - 1 ? __ldcg(v + at + sxy) : 0.0;
    return __fma_rn(6.0, __ldcg(v + at), -(((zm + ym) + (xm + xp)) + (yp + zp)));
}

}  // namespace

// The block's share of the bricks of the listed systems, and the walk over it.
struct Walk {
    int lo, hi;      // bricks of the list this block takes
    int first;       // list entry that holds brick lo
};

__global__ void __launch_bounds__(kNT, 3)
    k_cg_small(const CgSmallSys* __restrict__ all, const CgSmallGroup* __restrict__ groups, int ngroups,
               unsigned long long* bar, int* err)
{
    __shared__ __align__(16) long long sm[kKZ * kPlane];   // free again at the brick sum's barrier
    __shared__ double red[2][kNT];
    __shared__ double s_alpha[kCgSmallSystems], s_beta;
    __shared__ int s_stop;
    __shared__ int s_first[kCgSmallSystems + 1];   // first brick of each listed system
    __shared__ short s_id[kCgSmallSystems];
    __shared__ int s_n;
    __shared__ unsigned s_pm[kNT / 32], s_any;
    const int tid = threadIdx.x, warp = tid >> 5;
    int ph = 0, turn = 0;
    const CgSmallSys* sys = all;
    int nsys = 0;

    // lists the systems that take part -- all of them, or those still running
    // after `it` iterations -- and returns this block's share of their bricks
    auto list = [&](bool all, int it) -> Walk {
        __syncthreads();
        if (warp == 0) {
            int n = 0, bricks = 0;
            for (int b = 0; b < nsys; b += 32) {
                const int i = b + tid;
                const bool in = i < nsys && (all || (__ldcg(&sys[i].S->done) == 0 && it < sys[i].max_iter));
                const int mine = in ? sys[i].bricks : 0;
                int incl = mine;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int up = __shfl_up_sync(0xffffffffu, incl, o);
                    if (tid >= o) incl += up;
                }
                const unsigned mask = __ballot_sync(0xffffffffu, in);
                if (in) {
                    const int e = n + __popc(mask & ((1u << tid) - 1u));
                    s_id[e] = (short)i;
                    s_first[e] = bricks + incl - mine;
                }
                n += __popc(mask);
                bricks += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (tid == 0) {
                s_n = n;
                s_first[n] = bricks;
            }
        }
        __syncthreads();
        Walk w;
        const long long total = s_first[s_n];
        w.lo = (int)(total * blockIdx.x / gridDim.x);
        w.hi = (int)(total * (blockIdx.x + 1) / gridDim.x);
        w.first = 0;
        while (w.first + 1 < s_n && s_first[w.first + 1] <= w.lo) ++w.first;
        return w;
    };
    // barrier between phases; *any becomes whether some block's flag (thread
    // 0's) was set; false: a wait ran out here or in another block
    auto sync = [&](unsigned flag = 0, bool* any = nullptr) -> bool {
        __syncthreads();
        bool ok = true;
        if (tid == 0) {
            grid_arrive(bar, ph, flag, 0u);
            ok = grid_wait(bar, ph, 0u, &s_any, err);
        }
        ++ph;
        const bool good = __syncthreads_or(!ok) == 0;
        if (any) *any = s_any != 0;
        return good;
    };
    // folds the threads' largest |p| high word into a slot of the system
    auto fold_pmax = [&](unsigned pm, unsigned long long* slot) {
        pm = __reduce_max_sync(0xffffffffu, pm);
        if ((tid & 31) == 0) s_pm[warp] = pm;
        __syncthreads();
        if (tid == 0) {
            unsigned b = 0;
            for (int w = 0; w < kNT / 32; ++w) b = max(b, s_pm[w]);
            atomicMax(slot, (unsigned long long)b << 32);
        }
    };

    for (int gi = 0; gi < ngroups; ++gi) {
        sys = all + groups[gi].first;
        nsys = groups[gi].count;
        // r = b - A x0, p = r; partials of r.r and b.b
        Walk w = list(true, 0);
        for (int e = w.first; e < s_n && s_first[e] < w.hi; ++e) {
            const CgSmallSys& s = sys[s_id[e]];
            const int64_t sxy = (int64_t)s.pitch * s.ny, sd = (int64_t)s.nx * s.ny;
            unsigned pm = 0;
            for (int g = max(w.lo, s_first[e]); g < min(w.hi, s_first[e + 1]); ++g) {
                const int brick = g - s_first[e];
                const Place c = place_of(s, brick, tid);
                double rr = 0.0, bb = 0.0;
                for (int kk = 0; kk < c.nk; ++kk) {
                    double rv[2] = {0.0, 0.0};
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        if (i ? c.ok1 : c.ok0) {
                            const int64_t at = c.dense + kk * sd + i;
                            const double bt = __ldg(s.b + at);
                            rv[i] = bt - row_apply(s, s.x, c.X + i, c.Y, c.k0 + kk, at);
                            rr = __fma_rn(rv[i], rv[i], rr);
                            bb = __fma_rn(bt, bt, bb);
                            pm = max(pm, xs_abs_hi(rv[i]));
                        }
                    st_pair(s.r + c.at + kk * sxy, c.ok0, rv);
                    st_pair(s.p + c.at + kk * sxy, c.ok0, rv);
                }
                brick_sum(rr, red[turn & 1], turn, s.part + brick);
                ++turn;
                brick_sum(bb, red[turn & 1], turn, s.part + s.bricks + brick);
                ++turn;
            }
            fold_pmax(pm, &s.S->pmax[0]);
            __syncthreads();
        }
        if (!sync()) return;
        for (int e = w.first; e < s_n && s_first[e] < w.hi; ++e) {
            const CgSmallSys& s = sys[s_id[e]];
            if (s_first[e] < w.lo) continue;   // the block with the system's first brick keeps its scalars
            const double rho = sys_sum(s.part, s.bricks, red[0]);
            const double bn2 = sys_sum(s.part + s.bricks, s.bricks, red[1]);
            if (tid == 0) {
                CgScalars* S = s.S;
                S->rho2[0] = rho;
                S->bnorm = sqrt(bn2);
                S->zero_rhs = bn2 == 0.0;
                S->relres = bn2 == 0.0 ? 0.0 : sqrt(rho) / S->bnorm;
                if (bn2 == 0.0 || S->relres <= S->rtol) S->done = 1;
            }
            __syncthreads();
        }
        if (!sync()) return;

        int most = 0;   // iterations any system of the group may take: ends the loop whatever its scalars say
        for (int i = 0; i < nsys; ++i) most = max(most, sys[i].max_iter);
        bool relist = true;   // some system stopped: the others' bricks are shared out anew
        for (int it = 0; it < most; ++it) {
            if (relist) w = list(false, it);
            if (s_n == 0) break;   // the same in every block
            unsigned ended = 0;    // thread 0: a system this block keeps the scalars of stops with this iteration
            // q = A p, partials of p.q
            for (int e = w.first; e < s_n && s_first[e] < w.hi; ++e) {
                const CgSmallSys& s = sys[s_id[e]];
                const int emax = (int)(__ldcg(&s.S->pmax[it % 3]) >> 52);
                const bool conv = cg_xs_ok(emax);
                for (int g = max(w.lo, s_first[e]); g < min(w.hi, s_first[e + 1]); ++g) {
                    const int brick = g - s_first[e];
                    const Place c = place_of(s, brick, tid);
                    double none[kKZ][2], qv[kKZ][2];
                    const double pq = conv ? spmv_brick<true, false>(s, c, emax, sm, none, qv)
                                           : spmv_brick<false, false>(s, c, emax, sm, none, qv);
                    brick_sum(pq, red[turn & 1], turn, s.part + brick);
                    ++turn;
                }
            }
            if (!sync()) return;
            // alpha; r -= alpha q, partials of r.r
            for (int e = w.first; e < s_n && s_first[e] < w.hi; ++e) {
                const CgSmallSys& s = sys[s_id[e]];
                const int64_t sxy = (int64_t)s.pitch * s.ny;
                const double rho = tid == 0 ? __ldcg(&s.S->rho2[it & 1]) : 0.0;
                const double pq = sys_sum(s.part, s.bricks, red[turn & 1]);
                ++turn;
                if (tid == 0) {
                    s_alpha[e] = pq > 0.0 ? rho / pq : kBreakdown;
                    if (s_first[e] >= w.lo && !(pq > 0.0)) {
                        s.S->done = 2;
                        ended = 1;
                    }
                }
                __syncthreads();
                const double alpha = s_alpha[e];
                if (alpha == kBreakdown) continue;   // nothing more is updated
                for (int g = max(w.lo, s_first[e]); g < min(w.hi, s_first[e + 1]); ++g) {
                    const int brick = g - s_first[e];
                    const Place c = place_of(s, brick, tid);
                    double rv[kKZ][2], qv[kKZ][2];
#pragma unroll
                    for (int kk = 0; kk < kKZ; ++kk) {
                        const bool in = kk < c.nk && c.ok0;
                        ld_pair((const double*)s.r + c.at + kk * sxy, in, rv[kk]);
                        ld_pair((const double*)s.q + c.at + kk * sxy, in, qv[kk]);
                    }
                    double rr = 0.0;
#pragma unroll
                    for (int kk = 0; kk < kKZ; ++kk) {
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            rv[kk][i] = __fma_rn(-alpha, qv[kk][i], rv[kk][i]);
                            rr = __fma_rn(rv[kk][i], rv[kk][i], rr);
                        }
                        st_pair(s.r + c.at + kk * sxy, kk < c.nk && c.ok0, rv[kk]);
                    }
                    brick_sum(rr, red[turn & 1], turn, s.part + s.bricks + brick);
                    ++turn;
                }
            }
            if (!sync()) return;
            // beta and the stop test; x += alpha p, p = r + beta p
            for (int e = w.first; e < s_n && s_first[e] < w.hi; ++e) {
                const CgSmallSys& s = sys[s_id[e]];
                CgScalars* S = s.S;
                const bool xvec = (s.nx & 1) == 0 && (reinterpret_cast<uintptr_t>(s.x) & 15) == 0;
                const int64_t sxy = (int64_t)s.pitch * s.ny, sd = (int64_t)s.nx * s.ny;
                const double alpha = s_alpha[e];
                if (alpha == kBreakdown) continue;   // the block that keeps its scalars has ended it
                double rho = 0.0, bnorm = 0.0, rtol = 0.0;
                if (tid == 0) {
                    rho = __ldcg(&S->rho2[it & 1]);
                    bnorm = __ldcg(&S->bnorm);
                    rtol = __ldcg(&S->rtol);
                }
                const double rho_new = sys_sum(s.part + s.bricks, s.bricks, red[turn & 1]);
                ++turn;
                if (tid == 0) {
                    const double t = rtol * bnorm;
                    s_stop = cg_stops(rho_new, bnorm, rtol, t * t);
                    s_beta = rho_new / rho;
                }
                __syncthreads();
                const bool stop = s_stop != 0;
                const double beta = s_beta;
                unsigned pm = 0;
                for (int g = max(w.lo, s_first[e]); g < min(w.hi, s_first[e + 1]); ++g) {
                    const int brick = g - s_first[e];
                    const Place c = place_of(s, brick, tid);
                    double xv[kKZ][2], pv[kKZ][2], rv[kKZ][2];
#pragma unroll
                    for (int kk = 0; kk < kKZ; ++kk) {
                        const bool in = kk < c.nk && c.ok0;
                        ld_pair((const double*)s.p + c.at + kk * sxy, in, pv[kk]);
                        ld_x(s.x + c.dense + kk * sd, xvec, in, in && c.ok1, xv[kk]);
                        ld_pair((const double*)s.r + c.at + kk * sxy, in, rv[kk]);
                    }
#pragma unroll
                    for (int kk = 0; kk < kKZ; ++kk) {
                        const bool in = kk < c.nk && c.ok0;
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            xv[kk][i] = __fma_rn(alpha, pv[kk][i], xv[kk][i]);
                            pv[kk][i] = __fma_rn(beta, pv[kk][i], rv[kk][i]);
                            pm = max(pm, xs_abs_hi(pv[kk][i]));
                        }
                        st_x(s.x + c.dense + kk * sd, xvec, in, in && c.ok1, xv[kk]);
                        if (!stop) st_pair(s.p + c.at + kk * sxy, in, pv[kk]);
                    }
                }
                fold_pmax(pm, &S->pmax[(it + 1) % 3]);
                if (tid == 0 && s_first[e] >= w.lo) {
                    S->pmax[(it + 2) % 3] = 0;   // last read by the SpMV of iteration it - 1
                    S->rho2[(it + 1) & 1] = rho_new;
                    S->iters = it + 1;
                    if (stop) S->done = 1;
                    if (stop || it + 1 >= s.max_iter) ended = 1;
                }
                __syncthreads();
            }
            if (!sync(ended, &relist)) return;
        }

        // the true residual ||b - A x||^2 of every system; a zero right-hand side has the solution 0
        w = list(true, 0);
        for (int e = w.first; e < s_n && s_first[e] < w.hi; ++e) {
            const CgSmallSys& s = sys[s_id[e]];
            const int64_t sd = (int64_t)s.nx * s.ny;
            const bool zero = __ldcg(&s.S->zero_rhs) != 0;
            for (int g = max(w.lo, s_first[e]); g < min(w.hi, s_first[e + 1]); ++g) {
                const int brick = g - s_first[e];
                const Place c = place_of(s, brick, tid);
                double rr = 0.0;
                for (int kk = 0; kk < c.nk; ++kk)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        if (i ? c.ok1 : c.ok0) {
                            const int64_t at = c.dense + kk * sd + i;
                            if (zero) {
                                s.x[at] = 0.0;
                            } else {
                                const double d = __ldg(s.b + at) - row_apply(s, s.x, c.X + i, c.Y, c.k0 + kk, at);
                                rr = __fma_rn(d, d, rr);
                            }
                        }
                brick_sum(rr, red[turn & 1], turn, s.part + brick);
                ++turn;
            }
        }
        if (!sync()) return;
        for (int e = w.first; e < s_n && s_first[e] < w.hi; ++e) {
            const CgSmallSys& s = sys[s_id[e]];
            if (s_first[e] < w.lo) continue;
            const double rr = sys_sum(s.part, s.bricks, red[turn & 1]);
            ++turn;
            if (tid == 0) {
                CgScalars* S = s.S;
                S->rr_true = rr;
                const int its = __ldcg(&S->iters);
                if (its > 0) S->relres = sqrt(__ldcg(&S->rho2[its & 1])) / __ldcg(&S->bnorm);
            }
        }
    }
}

// One system whose bricks all have a block of their own: the same phases with
// the block's part of x, r, p and q in registers; only p goes through memory,
// for the neighbours.  The brick partials and their order are k_cg_small's, so
// the result is the same bit for bit.  Bound by latency: three barriers, two
// sums over the partials and the loads of p's halo per iteration.
template <int MINB>
__global__ void __launch_bounds__(kNT, MINB) k_cg_one(const CgSmallSys* __restrict__ sys, unsigned long long* bar, int* err)
{
    __shared__ __align__(16) long long sm[kKZ * kPlane];
    __shared__ double red[2][kNT];
    __shared__ double s_val;
    __shared__ int s_flag;
    __shared__ unsigned s_pm[kNT / 32], s_m;
    const int tid = threadIdx.x;
    const CgSmallSys s = *sys;
    CgScalars* S = s.S;
    const Place c = place_of(s, blockIdx.x, tid);
    const int64_t sxy = (int64_t)s.pitch * s.ny, sd = (int64_t)s.nx * s.ny;
    double* const part_pq = s.part + blockIdx.x;
    double* const part_rr = part_pq + s.bricks;
    int ph = 0;
    unsigned m = 0;   // the direction's largest exponent field
    // barrier between phases; NEW: every block brings its values' exponent and m becomes the largest
    auto sync = [&](bool fresh, unsigned pm) -> bool {
        if (fresh) {
            pm = __reduce_max_sync(0xffffffffu, pm);
            if ((tid & 31) == 0) s_pm[tid >> 5] = pm;
        }
        __syncthreads();
        bool ok = true;
        if (tid == 0) {
            unsigned mine = m;
            if (fresh) {
                mine = s_pm[0];
                for (int w = 1; w < kNT / 32; ++w) mine = max(mine, s_pm[w]);
                mine >>= 20;
            }
            grid_arrive(bar, ph, mine, m);
            ok = grid_wait(bar, ph, m, &s_m, err);
        }
        ++ph;
        const bool all = __syncthreads_or(!ok) == 0;
        m = s_m;
        return all;
    };

    double xv[kKZ][2], rv[kKZ][2], pv[kKZ][2], qv[kKZ][2];
    double rr = 0.0, bb = 0.0;
    unsigned pm = 0;
#pragma unroll
    for (int kk = 0; kk < kKZ; ++kk)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            xv[kk][i] = rv[kk][i] = 0.0;
            if (kk < c.nk && (i ? c.ok1 : c.ok0)) {
                const int64_t at = c.dense + kk * sd + i;
                const double bt = __ldg(s.b + at);
                xv[kk][i] = s.x[at];
                rv[kk][i] = bt - row_apply(s, s.x, c.X + i, c.Y, c.k0 + kk, at);
                rr = __fma_rn(rv[kk][i], rv[kk][i], rr);
                bb = __fma_rn(bt, bt, bb);
                pm = max(pm, xs_abs_hi(rv[kk][i]));
            }
            pv[kk][i] = rv[kk][i];
        }
    auto store_p = [&] {
#pragma unroll
        for (int kk = 0; kk < kKZ; ++kk)
            st_pair(s.p + c.at + kk * sxy, kk < c.nk && c.ok0, pv[kk]);
    };
    store_p();
    brick_sum(rr, red[0], 0, part_pq);
    brick_sum(bb, red[1], 1, part_rr);
    if (!sync(true, pm)) return;
    const double rho0 = sys_sum(s.part, s.bricks, red[0]);
    const double bn2 = sys_sum(s.part + s.bricks, s.bricks, red[1]);
    // the scalars live in thread 0 of every block, the same in each
    double rho = rho0, bnorm = 0.0, rtol = 0.0, t2 = 0.0;
    if (tid == 0) {
        bnorm = sqrt(bn2);
        rtol = __ldcg(&S->rtol);
        t2 = rtol * bnorm;
        t2 *= t2;
        s_flag = bn2 == 0.0 ? 2 : sqrt(rho) / bnorm <= rtol ? 1 : 0;
    }
    __syncthreads();
    const bool zero = s_flag == 2;
    int done = s_flag != 0 ? 1 : 0, it = 0;
    // both reads of part_* are over everywhere before the first phase writes them again
    if (!sync(false, 0u)) return;
    while (!done && it < s.max_iter) {
        const double pq_t = cg_xs_ok((int)m) ? spmv_brick<true, true>(s, c, (int)m, sm, pv, qv)
                                             : spmv_brick<false, true>(s, c, (int)m, sm, pv, qv);
        brick_sum(pq_t, red[0], it, part_pq);
        if (!sync(false, 0u)) return;
        const double pq = sys_sum(s.part, s.bricks, red[1]);
        if (tid == 0) s_val = pq > 0.0 ? rho / pq : kBreakdown;
        __syncthreads();
        const double alpha = s_val;
        if (alpha == kBreakdown) {
            done = 2;
            break;
        }
        rr = 0.0;
#pragma unroll
        for (int kk = 0; kk < kKZ; ++kk)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                rv[kk][i] = __fma_rn(-alpha, qv[kk][i], rv[kk][i]);
                rr = __fma_rn(rv[kk][i], rv[kk][i], rr);
            }
        brick_sum(rr, red[0], it + 1, part_rr);
        // x waits for nothing: its update fills the barrier's wait
#pragma unroll
        for (int kk = 0; kk < kKZ; ++kk)
#pragma unroll
            for (int i = 0; i < 2; ++i) xv[kk][i] = __fma_rn(alpha, pv[kk][i], xv[kk][i]);
        if (!sync(false, 0u)) return;
        const double rho_new = sys_sum(s.part + s.bricks, s.bricks, red[1]);
        if (tid == 0) {
            s_val = rho_new / rho;
            s_flag = cg_stops(rho_new, bnorm, rtol, t2);
            rho = rho_new;
        }
        __syncthreads();
        const double beta = s_val;
        done = s_flag;
        ++it;
        if (done || it == s.max_iter) break;
        pm = 0;
#pragma unroll
        for (int kk = 0; kk < kKZ; ++kk)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                pv[kk][i] = __fma_rn(beta, pv[kk][i], rv[kk][i]);
                pm = max(pm, xs_abs_hi(pv[kk][i]));
            }
        store_p();
        if (!sync(true, pm)) return;
    }
    const bool xvec = (s.nx & 1) == 0 && (reinterpret_cast<uintptr_t>(s.x) & 15) == 0;
#pragma unroll
    for (int kk = 0; kk < kKZ; ++kk) {
        if (zero) xv[kk][0] = xv[kk][1] = 0.0;
        if (kk < c.nk) st_x(s.x + c.dense + kk * sd, xvec, c.ok0, c.ok1, xv[kk]);
    }
    if (!sync(false, 0u)) return;
    rr = 0.0;
    if (!zero)
        for (int kk = 0; kk < c.nk; ++kk)
#pragma unroll
            for (int i = 0; i < 2; ++i)
                if (i ? c.ok1 : c.ok0) {
                    const int64_t at = c.dense + kk * sd + i;
                    const double d = __ldg(s.b + at) - row_apply(s, s.x, c.X + i, c.Y, c.k0 + kk, at);
                    rr = __fma_rn(d, d, rr);
                }
    brick_sum(rr, red[0], 0, part_pq);
    if (!sync(false, 0u)) return;
    if (blockIdx.x != 0) return;
    const double rr_true = sys_sum(s.part, s.bricks, red[1]);
    if (tid == 0) {
        S->bnorm = bnorm;
        S->zero_rhs = zero;
        S->relres = zero ? 0.0 : sqrt(rho) / bnorm;
        S->done = done;
        S->iters = it;
        S->rr_true = rr_true;
    }
}

// Blocks of a kernel resident at once on the GPU, 0 if that cannot be told.
template <typename K>
int resident_blocks(K kern)
{
    int per_sm = 0, dev = 0, sms = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kNT, 0) != cudaSuccess ||
        cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return per_sm * sms;
}

bool cg_small_shape(const OpDev& A, CgSmallSys* s)
{
    if (A.kind != HS_OP_STENCIL7 || A.n < kCgSmallMinN || A.n >= kCgSmallMaxN || A.nx < kCgSmallMinNx) return false;
    int best = 0;
    for (int lg = 5; lg >= 4; --lg) {   // 64 x 8 columns, or 32 x 16 where those need fewer bricks
        const int tx = (A.nx + (2 << lg) - 1) / (2 << lg), rows = kNT >> lg, ty = (A.ny + rows - 1) / rows;
        const int64_t bricks = (int64_t)tx * ty * ((A.nz + kKZ - 1) / kKZ);
        if (bricks > kCgSmallMaxBricks || (best && bricks >= best)) continue;
        best = (int)bricks;
        s->lg = lg;
        s->tiles_x = tx;
        s->tiles_y = ty;
        s->bricks = best;
    }
    s->pitch = (A.nx + 1) & ~1;
    s->nx = A.nx;
    s->ny = A.ny;
    s->nz = A.nz;
    return best > 0;
}

int cg_small_launch(const CgSmallSys* sys, const CgSmallGroup* groups, int ngroups, bool single, int64_t bricks,
                    unsigned long long* bar, int* err, cudaStream_t stream)
{
    // asked once per process (a single GPU)
    static const int slots = resident_blocks(k_cg_small), slots_one = resident_blocks(k_cg_one<2>),
                     slots_sm = resident_blocks(k_cg_one<1>);
    if (slots < 1) return fail(HS_ECUDA, "cg: no resident block of the small-system kernel");
    // a block per brick in registers: one per SM with all the registers it likes
    // (64^3 11.25 us per iteration), or two (11.73; 80^3 15.5 against 18.9 in k_cg_small)
    const bool one = single && bricks <= slots_one;
    const void* kern = !one ? (const void*)k_cg_small
                       : bricks <= slots_sm ? (const void*)k_cg_one<1> : (const void*)k_cg_one<2>;
    const int blocks = one ? (int)bricks : (int)std::min<int64_t>(bricks, slots);
    void* args_one[] = {(void*)&sys, (void*)&bar, (void*)&err};
    void* args[] = {(void*)&sys, (void*)&groups, (void*)&ngroups, (void*)&bar, (void*)&err};
    const cudaError_t e = cudaLaunchCooperativeKernel(kern, dim3((unsigned)blocks), dim3(kNT), one ? args_one : args, 0,
                                                      stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return cuda_fail(e, "cg: small-system kernel");
    }
    HS_CHECK_LAUNCH("cg: small-system kernel");
    return HS_OK;
}

}  // namespace hcg
