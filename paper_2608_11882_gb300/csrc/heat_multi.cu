// Many steps of the update of Section 4, Eq. 4 in one launch, for grids whose
// fields stay in L2: a persistent cooperative kernel whose blocks exchange the
// step's maximum with the barrier between two steps (gridbar.cuh).
//
// A step of such a grid takes a few microseconds, less than launching the
// Interior and Boundary kernels for it and draining them (14.4 us per 64^3 FP64
// step, however small the grid).  Here the blocks stay: each takes a fixed set
// of bricks of 64 x ROWS x kMuKZ points, every step loads a brick with its
// one-point halo from L2 (ld.global.cg: a block must not see another SM's new
// values through its own stale L1 lines), converts it once, and stores the new
// values; all loads of a brick are in flight at once, where the streaming
// kernel waits plane by plane.  A step of a grid with one brick per block is
// bound by latency: load, convert, store, barrier (64^3 FP64 3.5 us, FP32 2.5);
// with several, by instruction issue, the z halo converted twice per four
// planes.  At least two blocks per SM, every block resident, so that one loads
// while the other computes (held to three the kernel took 17.7 us instead of
// 15.4 per FP64 step of 191 x 101 x 150).  The per-point arithmetic is that of the
// other heat kernels, so results match them bit for bit, and the whole grid --
// Interior and Boundary planes -- is one step's work.
#include <algorithm>

#include "gridbar.cuh"
#include "heat_common.cuh"

namespace hcg {

constexpr int kMuNT = 256, kMuKZ = 4, kMuTW = 64, kMuMinBlocks = 2;

template <typename T>
struct MultiShape {
    static constexpr int V = Vec<T>::V;
    static constexpr int LPR = kMuTW / V;        // threads per row
    static constexpr int ROWS = kMuNT / LPR;     // 8 rows of doubles, 16 of floats
    static constexpr int A = 16 / (int)sizeof(T);
    static constexpr int BW = kMuTW + 2 * A;     // shared row: the brick's row at column A
};

template <typename T>
__device__ __forceinline__ void ldcg_vec(const T* p, T (&o)[Vec<T>::V])
{
    const typename Vec<T>::type v = __ldcg(reinterpret_cast<const typename Vec<T>::type*>(p));
    if constexpr (Vec<T>::V == 4) {
        o[0] = v.x;
        o[1] = v.y;
        o[2] = v.z;
        o[3] = v.w;
    } else {
        o[0] = v.x;
        o[1] = v.y;
    }
}

template <typename T>
struct MultiArgs {
    T* buf[2];
    HeatGeom g;
    T r;                 // FIXED64: r 2^64
    FxState* fx;
    int cur, m3;
    int steps;
    int tiles_x, tiles_y, bricks;
    unsigned long long* bar;
    int* err;
};

// One brick of one step; returns what joins the step's maximum (high words of
// |u| for the exact sum, |U| for FIXED64).
template <typename T, bool XS, bool CONV>
__device__ __forceinline__ void multi_brick(const MultiArgs<T>& a, const T* src, T* dst, int brick, int emax, int ks,
                                            typename std::conditional<XS, long long, T>::type* sm,
                                            unsigned long long& mx)
{
    using S = MultiShape<T>;
    using Q = typename std::conditional<XS, long long, T>::type;   // fixed-point integers, or the values
    constexpr int V = S::V, LPR = S::LPR, ROWS = S::ROWS, A = S::A, BW = S::BW, KZ = kMuKZ;
    constexpr int PL = (ROWS + 2) * BW;
    const HeatGeom& g = a.g;
    const int tid = threadIdx.x;
    const int lx = tid % LPR, row = tid / LPR;
    const int t = brick / a.tiles_x;
    const int x0 = (brick - t * a.tiles_x) * kMuTW;
    const int tz = t / a.tiles_y;
    const int y0 = (t - tz * a.tiles_y) * ROWS, k0 = tz * KZ;
    const int X = x0 + V * lx, Y = y0 + row;
    const bool in = X < g.nx && Y < g.ny;
    const int64_t own = g.at(X, Y, k0);

    // the thread's column of planes k0-1 .. k0+KZ, a vector of the halo rows and
    // a value of the halo columns; cells outside the grid read the zero
    // boundary layer, those outside the buffer are not read
    T v[KZ + 2][V], hy[V], hx = T(0);
#pragma unroll
    for (int q = 0; q < KZ + 2; ++q) {
        if (in && k0 - 1 + q <= g.nz) {
            ldcg_vec(src + own + (q - 1) * g.plane, v[q]);
        } else {
#pragma unroll
            for (int i = 0; i < V; ++i) v[q][i] = T(0);
        }
    }
    const int yk = (tid / LPR) % KZ, yside = tid / (LPR * KZ);   // sides 0, 1: one vector each
    {
        const int Yh = yside ? y0 + ROWS : y0 - 1;
        if (yside < 2 && X < g.nx && Yh <= g.ny && k0 + yk < g.nz) {
            ldcg_vec(src + g.at(X, Yh, k0 + yk), hy);
        } else {
#pragma unroll
            for (int i = 0; i < V; ++i) hy[i] = T(0);
        }
    }
    const int xr = tid % ROWS, xk = (tid / ROWS) % KZ, xside = tid / (ROWS * KZ);
    if (xside < 2) {
        const int Xh = xside ? x0 + kMuTW : x0 - 1;
        if (Xh <= g.nx && y0 + xr < g.ny && k0 + xk < g.nz) hx = __ldcg(src + g.at(Xh, y0 + xr, k0 + xk));
    }

    auto fix = [emax](T w) -> Q {
        if constexpr (XS) {
            if constexpr (CONV) return xs_fix(__double_as_longlong(w), emax);
            return __double_as_longlong(w);
        } else {
            return w;
        }
    };
    Q u[KZ + 2][V];
#pragma unroll
    for (int q = 0; q < KZ + 2; ++q)
#pragma unroll
        for (int i = 0; i < V; ++i) u[q][i] = fix(v[q][i]);
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk) st_vec(sm + kk * PL + (row + 1) * BW + A + V * lx, u[kk + 1]);
    if (yside < 2) {
        Q h[V];
#pragma unroll
        for (int i = 0; i < V; ++i) h[i] = fix(hy[i]);
        st_vec(sm + yk * PL + (yside ? ROWS + 1 : 0) * BW + A + V * lx, h);
    }
    if (xside < 2) sm[xk * PL + (xr + 1) * BW + (xside ? A + kMuTW : A - 1)] = fix(hx);
    __syncthreads();

    if (!in) return;
    const int nvalid = min(V, g.nx - X);
    double r2 = 0.0;
    if constexpr (CONV) r2 = xs_r2(a.r, emax);
    T* o = dst + own;
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk) {
        if (k0 + kk >= g.nz) break;
        const Q* pc = sm + kk * PL + (row + 1) * BW + A + V * lx;
        Q ym[V], yp[V];
        ld_vec(pc - BW, ym);
        ld_vec(pc + BW, yp);
        const Q left = pc[-1], right = pc[V];
        T w[V];
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const Q c = u[kk + 1][i], zm = u[kk][i], zp = u[kk + 2][i];
            const Q xm = i == 0 ? left : u[kk + 1][i - 1], xp = i == V - 1 ? right : u[kk + 1][i + 1];
            if constexpr (XS) {
                if constexpr (CONV) {
                    // one point in four back on the FP64 pipe, as in the streaming kernel
                    const long long L = xs_numerator(c, xm, xp, ym[i], yp[i], zm, zp);
                    w[i] = (i == 0 && (kk & 1) == 0) ? xs_apply<true>(v[kk + 1][i], L, a.r, r2, emax)
                                                     : xs_apply<false>(v[kk + 1][i], L, a.r, r2, emax);
                } else {
                    auto d = [](long long b) { return __longlong_as_double(b); };
                    w[i] = Point<double, false>::update(v[kk + 1][i], d(xm), d(xp), d(ym[i]), d(yp[i]), d(zm), d(zp),
                                                        a.r, 0);
                }
            } else {
                w[i] = Point<T, false>::update(c, xm, xp, ym[i], yp[i], zm, zp, a.r, ks);
            }
        }
        if (nvalid == V) {
            st_vec(o, w);
        } else {
#pragma unroll
            for (int i = 0; i < V; ++i)
                if (i < nvalid) o[i] = w[i];
        }
        if constexpr (XS || kIsFixed<T>) {
#pragma unroll
            for (int i = 0; i < V; ++i) {
                unsigned long long m;
                if constexpr (XS) m = xs_abs_hi(w[i]);
                else m = fx_abs(w[i]);
                if (i < nvalid && m > mx) mx = m;
            }
        }
        o += g.plane;
    }
}

template <typename T, bool XS>
__global__ void __launch_bounds__(kMuNT, kMuMinBlocks) k_heat_multi(const __grid_constant__ MultiArgs<T> a)
{
    using S = MultiShape<T>;
    using Q = typename std::conditional<XS, long long, T>::type;
    constexpr int SM = kMuKZ * (S::ROWS + 2) * S::BW;
    __shared__ __align__(16) Q sm[2 * SM];   // two bricks: the next one is staged while slow warps read
    __shared__ unsigned wout[kMuNT / 32];
    __shared__ unsigned s_m;
    const int tid = threadIdx.x;
    // a launch after a wait that ran out does no work at all
    if (__syncthreads_or(tid == 0 && *(volatile int*)a.err != 0)) return;
    // the field's scale at the first step: its largest exponent (exact sum) or
    // the bit length of max|U| (FIXED64); the barrier carries it from step to step
    unsigned m = 0;
    int E = 0;
    if constexpr (XS) m = (unsigned)xs_emax(a.fx, a.m3);
    if constexpr (kIsFixed<T>) {
        m = 64 - __clzll((long long)__ldcg(&a.fx->slot[a.m3].maxU));
        E = __ldcg(&a.fx->slot[a.m3].E);
    }
    int parity = 0;
    for (int s = 0; s < a.steps; ++s) {
        const T* src = a.buf[(a.cur + s) & 1];
        T* dst = a.buf[(a.cur + s + 1) & 1];
        const int emax = (int)m;
        const int ks = kIsFixed<T> && m != 0 && m < 57 ? 57 - (int)m : 0;   // fx_shift
        E += ks;
        unsigned long long mx = 0;
        bool conv = false;
        if constexpr (XS) conv = !xs_native(emax, a.r);
        for (int b = blockIdx.x; b < a.bricks; b += gridDim.x, parity ^= 1) {
            if constexpr (XS) {
                if (conv)
                    multi_brick<T, XS, true>(a, src, dst, b, emax, ks, sm + parity * SM, mx);
                else
                    multi_brick<T, XS, false>(a, src, dst, b, emax, ks, sm + parity * SM, mx);
            } else {
                multi_brick<T, XS, false>(a, src, dst, b, emax, ks, sm + parity * SM, mx);
            }
        }
        unsigned out = 0;
        if constexpr (XS) out = (unsigned)mx >> 20;
        if constexpr (kIsFixed<T>) out = 64 - __clzll((long long)mx);
        if constexpr (XS || kIsFixed<T>) {
            out = __reduce_max_sync(0xffffffffu, out);
            if ((tid & 31) == 0) wout[tid >> 5] = out;
        }
        __syncthreads();
        bool ok = true;
        if (tid == 0) {
            if constexpr (XS || kIsFixed<T>) {
#pragma unroll
                for (int w = 1; w < kMuNT / 32; ++w) out = wout[w] > out ? wout[w] : out;
            }
            grid_arrive(a.bar, s, out, m);
            // after the last step only block 0 waits, to record the field's state
            if (s + 1 < a.steps || blockIdx.x == 0) ok = grid_wait(a.bar, s, m, &s_m, a.err);
        }
        if (__syncthreads_or(!ok)) return;
        if (s + 1 < a.steps || blockIdx.x == 0) m = s_m;
    }
    if (blockIdx.x == 0 && tid == 0) {
        grid_reset(a.bar);
        if constexpr (XS || kIsFixed<T>) {
            // only the exponent, or the bit length, of a slot's maximum is ever read
            FxSlot* now = &a.fx->slot[(a.m3 + a.steps) % 3];
            if constexpr (XS) now->maxU = (unsigned long long)m << 52;
            else now->maxU = m ? 1ull << (m - 1) : 0ull;
            now->E = E;
            a.fx->slot[(a.m3 + a.steps + 1) % 3].maxU = 0;
        }
    }
}

template <typename T, bool XS>
int multi_launch_t(const MultiCall& c)
{
    using S = MultiShape<T>;
    auto kern = k_heat_multi<T, XS>;
    // blocks resident at once, asked once per process (a single GPU)
    static const int slots = [kern] {
        int per_sm = 0, dev = 0, sms = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kMuNT, 0) != cudaSuccess ||
            cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            (void)cudaGetLastError();
            return 0;
        }
        return per_sm * sms;
    }();
    if (slots < 1) return fail(HS_ECUDA, "heat: no resident block of the multi-step kernel");
    const HeatGeom& g = *c.g;
    MultiArgs<T> a;
    a.buf[0] = (T*)c.buf[0];
    a.buf[1] = (T*)c.buf[1];
    a.g = g;
    if constexpr (kIsFixed<T>) a.r = c.R;
    else a.r = (T)c.r;
    a.fx = c.fx;
    a.cur = c.cur;
    a.m3 = c.m3;
    a.steps = c.steps;
    a.tiles_x = (g.nx + kMuTW - 1) / kMuTW;
    a.tiles_y = (g.ny + S::ROWS - 1) / S::ROWS;
    a.bricks = (int)multi_bricks(c.arith, g);
    a.bar = (unsigned long long*)c.sync;
    a.err = c.err;
    const int blocks = std::min(a.bricks, slots);
    void* args[] = {&a};
    const cudaError_t e =
        cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)blocks), dim3(kMuNT), args, 0, c.stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return cuda_fail(e, "heat multi-step kernel");
    }
    HS_CHECK_LAUNCH("heat multi-step kernel");
    return HS_OK;
}

int64_t multi_bricks(int arith, const HeatGeom& g)
{
    const int rows = arith == A_F32 ? MultiShape<float>::ROWS : MultiShape<double>::ROWS;
    return (int64_t)((g.nx + kMuTW - 1) / kMuTW) * ((g.ny + rows - 1) / rows) * ((g.nz + kMuKZ - 1) / kMuKZ);
}

int multi_launch(const MultiCall& c)
{
    switch (c.arith) {
    case A_F32: return multi_launch_t<float, false>(c);
    case A_FX64: return multi_launch_t<long long, false>(c);
    case A_F64_XS: return multi_launch_t<double, true>(c);
    }
    return fail(HS_EINVAL, "heat: arithmetic without a multi-step kernel");
}

}  // namespace hcg
