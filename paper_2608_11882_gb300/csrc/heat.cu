// Explicit 7-point heat stepping on one GPU: the Interior and Boundary kernels
// of Algorithms INTERIOR and BOUNDARY, the full-step kernel of Algorithm
// COMPUTE_SINGLE_GPU, and the heat_* entry points of the C ABI.
//
// Update (Section 4, Eq. 4 with kappa = 1 and f = 0, r = alpha dt / h^2):
//     u' = u + r * (((u[i-1] + u[i+1]) + (u[j-1] + u[j+1])) + (u[k-1] + u[k+1]) - 6 u)
// on interior points; the boundary layer stays zero (Dirichlet).
//
// Arithmetic, chosen per handle:
//   FP64      (default) FP64 fields, the six-neighbour sum and S - 6u exact in
//             64-bit fixed point on the field's current scale, rounded back to
//             a double and applied with one FP64 fused multiply-add
//             (heat_common.cuh);
//   FP64 pipe (HS_FP64_PIPE, and temporal blocking) the update in double
//             precision with two fused multiply-adds;
//   FP64 exact one rounding per operation in the written order (no FMA), the
//             oracle's rounding sequence bit for bit;
//   FP32      the update in single precision (storage and arithmetic);
//   FIXED64   FP64 interface, field held as 64-bit fixed-point integers
//             U = round(u 2^E).  The six-neighbour sum and S - 6U are exact;
//             r is held as R = r 2^64 (exactly for r >= 2^-11); the one rounding
//             per point is of R (S - 6U) / 2^64 to the nearest integer.  E is set
//             at upload from max|u0| so that 12 max|U| < 2^61, and grows during
//             the run: every step's kernels track max|U| of their output, and
//             when the field has shrunk the next step shifts all values left by
//             k bits (exact), keeping max|U| in [2^56, 2^57) -- about 57
//             significant bits relative to the current maximum.  For r <= 1/6
//             the update is a convex combination, so |U| never grows and
//             nothing overflows.  GB300's integer pipes run about 60x the rate
//             of its FP64 pipe, which makes this the FP64-accuracy form that is
//             bound by HBM rather than by FP64 issue.
//
// Layout in HBM: each field buffer holds (nz+2) planes of (ny+2) rows.  A row
// has `pitch` elements (a multiple of 128 bytes); interior x = 0 sits at
// element `lead` (32 bytes in), so interior rows start 32-byte aligned, and
// the x-boundary cells sit at lead-1 and lead+nx.  Planes 0 and nz+1, rows 0
// and ny+1 and the x-boundary cells hold the Dirichlet zeros in both buffers
// and are never written after creation, so a pointer swap keeps them intact.
#include <algorithm>
#include <cmath>
#include <vector>
#include <cstdlib>
#include <new>
#include <type_traits>

#include "gridbar.cuh"
#include "heat_common.cuh"
#include "tma.cuh"

namespace hcg {

// ---- Interior kernel ----------------------------------------------------------
// One thread per (i, j) column marches up a chunk of k-planes, keeping the
// values at k-1, k and k+1 in registers (rotated each plane); the four
// in-plane neighbours come through the read-only cache, where the block's
// neighbouring columns have just loaded them.
constexpr int kBX = 32, kBY = 8;

template <typename T, bool EXACT>
__global__ void __launch_bounds__(kBX* kBY)
    k_heat_interior(const T* __restrict__ src, T* __restrict__ dst, HeatGeom g, T r, int kbeg,
                    int kend, int kchunk, FxState* fx, int m3)
{
    const int i = blockIdx.x * kBX + threadIdx.x;
    const int j = blockIdx.y * kBY + threadIdx.y;
    const int k0 = kbeg + (int)blockIdx.z * kchunk;
    const int k1 = min(k0 + kchunk, kend);
    int ks = 0;
    if constexpr (kIsFixed<T>) ks = fx_shift(fx, m3);
    unsigned long long mx = 0;
    if (i < g.nx && j < g.ny && k0 < k1) {
        const int64_t P = g.plane, Y = g.pitch;
        int64_t c = g.at(i, j, k0);
        T below = __ldg(src + c - P);
        T cur = __ldg(src + c);
        for (int k = k0; k < k1; ++k) {
            const T above = __ldg(src + c + P);
            const T xm = __ldg(src + c - 1), xp = __ldg(src + c + 1);
            const T ym = __ldg(src + c - Y), yp = __ldg(src + c + Y);
            const T v = Point<T, EXACT>::update(cur, xm, xp, ym, yp, below, above, r, ks);
            dst[c] = v;
            if constexpr (kIsFixed<T>) {
                const unsigned long long a = fx_abs(v);
                mx = a > mx ? a : mx;
            }
            below = cur;
            cur = above;
            c += P;
        }
    }
    if constexpr (kIsFixed<T>)
        fx_finish<kBX * kBY>(mx, fx, m3, ks,
                             blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0);
}

// ---- Boundary kernel ------------------------------------------------------------
// The outermost interior k-planes (k = 0 and k = nz-1): the planes a k-split
// across devices would exchange.  blockIdx.z selects the plane.
template <typename T, bool EXACT>
__global__ void __launch_bounds__(kBX* kBY)
    k_heat_boundary(const T* __restrict__ src, T* __restrict__ dst, HeatGeom g, T r, FxState* fx,
                    int m3)
{
    const int i = blockIdx.x * kBX + threadIdx.x;
    const int j = blockIdx.y * kBY + threadIdx.y;
    int ks = 0;
    if constexpr (kIsFixed<T>) ks = fx_shift(fx, m3);
    unsigned long long mx = 0;
    if (i < g.nx && j < g.ny) {
        const int k = (blockIdx.z == 0) ? 0 : g.nz - 1;
        const int64_t P = g.plane, Y = g.pitch;
        const int64_t c = g.at(i, j, k);
        const T v = Point<T, EXACT>::update(__ldg(src + c), __ldg(src + c - 1), __ldg(src + c + 1),
                                            __ldg(src + c - Y), __ldg(src + c + Y),
                                            __ldg(src + c - P), __ldg(src + c + P), r, ks);
        dst[c] = v;
        if constexpr (kIsFixed<T>) mx = fx_abs(v);
    }
    if constexpr (kIsFixed<T>)
        fx_finish<kBX * kBY>(mx, fx, m3, ks,
                             blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0);
}

// ---- full-step kernel -------------------------------------------------------------
// Algorithm COMPUTE_SINGLE_GPU: one thread per interior point over the whole
// box, all seven values loaded directly.  A separate code path from the
// Interior/Boundary pair, used to cross-check it bit for bit.
template <typename T, bool EXACT>
__global__ void __launch_bounds__(256)
    k_heat_full(const T* __restrict__ src, T* __restrict__ dst, HeatGeom g, T r, FxState* fx,
                int m3)
{
    const int64_t n = (int64_t)g.nx * g.ny * g.nz;
    const int64_t P = g.plane, Y = g.pitch;
    int ks = 0;
    if constexpr (kIsFixed<T>) ks = fx_shift(fx, m3);
    unsigned long long mx = 0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t % g.nx);
        const int64_t jk = t / g.nx;
        const int j = (int)(jk % g.ny);
        const int k = (int)(jk / g.ny);
        const int64_t c = g.at(i, j, k);
        const T v = Point<T, EXACT>::update(src[c], src[c - 1], src[c + 1], src[c - Y], src[c + Y],
                                            src[c - P], src[c + P], r, ks);
        dst[c] = v;
        if constexpr (kIsFixed<T>) {
            const unsigned long long a = fx_abs(v);
            mx = a > mx ? a : mx;
        }
    }
    if constexpr (kIsFixed<T>) fx_finish<256>(mx, fx, m3, ks, blockIdx.x == 0);
}

// ---- Boundary and full-step kernels in the FP64 exact-sum arithmetic ------------------
// Per point the seven doubles are converted, then updated as in the streaming
// Interior kernel (xs_point); every output joins the step's maximum.
__global__ void __launch_bounds__(kBX* kBY)
    k_heat_boundary_xs(const double* __restrict__ src, double* __restrict__ dst, HeatGeom g, double r,
                       FxState* fx, int m3)
{
    const int i = blockIdx.x * kBX + threadIdx.x;
    const int j = blockIdx.y * kBY + threadIdx.y;
    const int emax = xs_emax(fx, m3);
    unsigned mx = 0;
    if (i < g.nx && j < g.ny) {
        const int k = (blockIdx.z == 0) ? 0 : g.nz - 1;
        const int64_t P = g.plane, Y = g.pitch;
        const int64_t c = g.at(i, j, k);
        const double v = xs_point(__ldg(src + c), __ldg(src + c - 1), __ldg(src + c + 1),
                                  __ldg(src + c - Y), __ldg(src + c + Y), __ldg(src + c - P),
                                  __ldg(src + c + P), r, emax);
        dst[c] = v;
        mx = xs_abs_hi(v);
    }
    fx_finish<kBX * kBY>((unsigned long long)mx << 32, fx, m3, 0,
                         blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0);
}

__global__ void __launch_bounds__(256)
    k_heat_full_xs(const double* __restrict__ src, double* __restrict__ dst, HeatGeom g, double r,
                   FxState* fx, int m3)
{
    const int64_t n = (int64_t)g.nx * g.ny * g.nz;
    const int64_t P = g.plane, Y = g.pitch;
    const int emax = xs_emax(fx, m3);
    unsigned mx = 0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t % g.nx);
        const int64_t jk = t / g.nx;
        const int j = (int)(jk % g.ny);
        const int k = (int)(jk / g.ny);
        const int64_t c = g.at(i, j, k);
        const double v = xs_point(src[c], src[c - 1], src[c + 1], src[c - Y], src[c + Y], src[c - P],
                                  src[c + P], r, emax);
        dst[c] = v;
        const unsigned a = xs_abs_hi(v);
        mx = a > mx ? a : mx;
    }
    fx_finish<256>((unsigned long long)mx << 32, fx, m3, 0, blockIdx.x == 0);
}

// ---- FIXED64 conversions (at upload and read only) --------------------------------
// Grid-stride over the interior points of a padded buffer.
__global__ void __launch_bounds__(256) k_fx_maxabs(const double* __restrict__ buf, HeatGeom g,
                                                   FxState* st)
{
    const int64_t n = (int64_t)g.nx * g.ny * g.nz;
    unsigned long long m = 0;
    int bad = 0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t % g.nx);
        const int64_t jk = t / g.nx;
        const double v = buf[g.at(i, (int)(jk % g.ny), (int)(jk / g.ny))];
        if (!isfinite(v)) bad = 1;
        const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(v));
        m = b > m ? b : m;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_down_sync(0xffffffffu, m, o);
        m = other > m ? other : m;
        bad |= __shfl_down_sync(0xffffffffu, bad, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&st->maxabs_bits, m);
        atomicMax(&st->slot[0].maxU, m);   // the exact-sum FP64 arithmetic's step-0 maximum
        if (bad) atomicOr(&st->nonfinite, 1);
    }
}

// E such that 12 max|u| 2^E < 2^61: with 12 M = f 2^e, f in [0.5, 1), E = 61 - e.
__device__ __forceinline__ int fx_scale_exp(const FxState* st)
{
    const double m = __longlong_as_double((long long)st->maxabs_bits);
    if (st->nonfinite || !(m > 0.0)) return 0;
    int e = 0;
    (void)frexp(12.0 * m, &e);
    return 61 - e;
}

// In place: the interior doubles of buf become round(u 2^E); slot 0 describes
// the encoded field, slot 1 is cleared for the first step.
__global__ void __launch_bounds__(256) k_fx_encode(double* __restrict__ buf, HeatGeom g,
                                                   FxState* st)
{
    const int E = fx_scale_exp(st);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const double m = __longlong_as_double((long long)st->maxabs_bits);
        st->slot[0].E = E;
        st->slot[0].maxU = (st->nonfinite || !(m > 0.0))
                               ? 0ull
                               : (unsigned long long)__double2ll_rn(scalbn(m, E));
        st->slot[1].maxU = 0;
    }
    long long* out = reinterpret_cast<long long*>(buf);
    const int64_t n = (int64_t)g.nx * g.ny * g.nz;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t % g.nx);
        const int64_t jk = t / g.nx;
        const int64_t c = g.at(i, (int)(jk % g.ny), (int)(jk / g.ny));
        const double v = buf[c];
        out[c] = isfinite(v) ? __double2ll_rn(scalbn(v, E)) : 0;
    }
}

// The interior of src (fixed point, the field of slot m3) as doubles u = U 2^-E in dst.
__global__ void __launch_bounds__(256) k_fx_decode(const long long* __restrict__ src,
                                                   double* __restrict__ dst, HeatGeom g,
                                                   const FxState* st, int m3)
{
    const int E = st->slot[m3].E;
    const int64_t n = (int64_t)g.nx * g.ny * g.nz;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t % g.nx);
        const int64_t jk = t / g.nx;
        const int64_t c = g.at(i, (int)(jk % g.ny), (int)(jk / g.ny));
        dst[c] = scalbn(__ll2double_rn(src[c]), -E);
    }
}

}  // namespace hcg

using namespace hcg;

struct hs_heat {
    HeatGeom g;
    int32_t dtype;
    Arith arith;
    size_t elem;
    double r;
    long long R;       // FIXED64: r 2^64
    uint32_t flags;
    cudaStream_t stream;
    void* arena;       // the handle's device allocation: err, fx, msync and, if it owns them, buf[]
    void* buf[2];
    bool owns_buf;     // false: buf[] are the caller's dev_buf0/dev_buf1
    FxState* fx;       // FIXED64 only
    int* err;          // device error word: 1 when a bounded device wait ran out
    int cur;           // buffer holding the current time level
    int64_t steps;     // steps since the last upload
    int64_t fxseq;     // fields produced since the last upload (FIXED64 slot = fxseq % 3)
    int kchunk;        // planes per Interior-kernel block
    int tdepth;        // steps per pass of the temporally blocked kernel (1: Interior + Boundary)
    bool deep;         // the library chose the depth, and passes of four steps are faster here
    CUtensorMap maps[2];   // TMA maps of the two buffers (temporal blocking)
    CUtensorMap smaps[2];  // TMA maps of the two buffers (streaming Interior kernel)
    uint32_t tbox[2];      // box of maps[]
    uint32_t sbox[2];      // box of smaps[]
    int kc_stream;         // k-planes per block of the streaming Interior kernel
    void* kap;             // HS_VARKAPPA: kappa on every padded node
    void* fdt;             // HS_VARKAPPA: dt f on the interior
    double vbx, vby, vbz;  // HS_VARKAPPA: dt / (2 h_d^2)
    int kappa_ok;          // HS_VARKAPPA, FP64: kappa allows the exact-sum form
    CUtensorMap vmaps[4];  // HS_VARKAPPA, FP64: TMA maps of the two buffers, kappa and dt f
    // Large grids run each step's Boundary kernel on a side stream, beside the
    // Interior kernel: forked from `stream` after the previous step (ev_fork)
    // and joined back before the next one (ev_join).  Null: one stream.
    cudaStream_t bstream;
    cudaEvent_t ev_fork, ev_join;
    void* msync;           // grid-barrier memory of the multi-step kernel; null: the handle does not use it
    // heat_time_interior: event pairs around the Interior launches of heat_step
    bool timing;
    std::vector<cudaEvent_t> tev;   // 2 per recorded launch, reused
    size_t tev_used;                // pairs recorded since the last heat_interior_time
};

namespace {

// Layout of the words at the start of a handle's allocation.
constexpr size_t kHeatFxOffset = 128, kHeatBarOffset = 256;
constexpr size_t kHeatStateBytes = (kHeatBarOffset + kGridBarBytes + 255) / 256 * 256;
static_assert(sizeof(FxState) <= kHeatBarOffset - kHeatFxOffset, "the per-step state fits its slot");

constexpr int64_t kForkMinPoints = (int64_t)1 << 22;
constexpr size_t kMaxTimedLaunches = 8192;   // event pairs a handle keeps for heat_interior_time

constexpr uint32_t kKnownFlags =
    HS_ALLOW_UNSTABLE | HS_EXACT_ROUNDING | HS_SCHED_FULL | HS_FIXED64 | HS_VARKAPPA | HS_FP64_PIPE;
constexpr double kKappaMax = 0.95;   // max of 0.5 + 0.45 sin sin sin (Section 4, Eq. 2)

int check_desc(const hs_heat_desc* d)
{
    if (!d) return fail(HS_EINVAL, "heat: desc is NULL");
    if (d->nx < 1 || d->ny < 1 || d->nz < 1)
        return fail(HS_EINVAL, "heat: grid %d x %d x %d must have at least one interior point per axis",
                    d->nx, d->ny, d->nz);
    if (d->nx > (1 << 30) || d->ny > 65535 * kBY || d->nz > (1 << 30))
        return fail(HS_EINVAL, "heat: grid axis too large (ny <= %d)", 65535 * kBY);
    if (!std::isfinite(d->r) || d->r < 0.0)
        return fail(HS_EINVAL, "heat: r = %g must be finite and >= 0", d->r);
    if (d->flags & ~kKnownFlags) return fail(HS_EINVAL, "heat: unknown flag bits 0x%x", d->flags);
    if (d->dtype != HS_F64 && d->dtype != HS_F32)
        return fail(HS_EINVAL, "heat: dtype %d is not HS_F64 or HS_F32", d->dtype);
    if ((d->flags & HS_EXACT_ROUNDING) && d->dtype != HS_F64)
        return fail(HS_EINVAL, "heat: HS_EXACT_ROUNDING applies to HS_F64 only");
    if ((d->flags & HS_FP64_PIPE) && (d->dtype != HS_F64 || (d->flags & HS_FIXED64)))
        return fail(HS_EINVAL, "heat: HS_FP64_PIPE applies to plain HS_F64 only");
    if (d->flags & HS_FIXED64) {
        if (d->dtype != HS_F64) return fail(HS_EINVAL, "heat: HS_FIXED64 applies to HS_F64 only");
        if (d->flags & HS_EXACT_ROUNDING)
            return fail(HS_EINVAL, "heat: HS_FIXED64 and HS_EXACT_ROUNDING exclude each other");
        if (d->flags & HS_ALLOW_UNSTABLE)
            return fail(HS_EINVAL, "heat: HS_FIXED64 needs r <= 1/6 (a growing field would overflow)");
    }
    if (d->tdepth < 0 || d->tdepth > 4)
        return fail(HS_EINVAL, "heat: tdepth %d not in {0, 1, 2, 3, 4}", d->tdepth);
    if ((d->flags & HS_SCHED_FULL) && d->tdepth > 1)
        return fail(HS_EINVAL, "heat: HS_SCHED_FULL runs one step per pass (tdepth 0 or 1)");
    if (d->flags & HS_VARKAPPA) {
        if (d->flags & (HS_FIXED64 | HS_EXACT_ROUNDING | HS_SCHED_FULL))
            return fail(HS_EINVAL, "heat: HS_VARKAPPA runs plain FP64 or FP32, Interior + Boundary");
        if (d->tdepth > 1) return fail(HS_EINVAL, "heat: HS_VARKAPPA runs one step per pass");
        // the update stays a convex combination (without the source) while
        // dt (kappa_max) sum_d 2/h_d^2 <= 1, which r = dt/h_min^2 <= 1/(6 kappa_max) ensures
        if (d->r > 1.0 / (6.0 * kKappaMax) && !(d->flags & HS_ALLOW_UNSTABLE))
            return fail(HS_EUNSTABLE, "heat: r = %.17g exceeds 1/(6 kappa_max) = %.6g", d->r,
                        1.0 / (6.0 * kKappaMax));
        return HS_OK;
    }
    // Three-dimensional stability of the explicit update: r <= 1/6.
    if (d->r > 1.0 / 6.0 && !(d->flags & HS_ALLOW_UNSTABLE))
        return fail(HS_EUNSTABLE, "heat: r = %.17g exceeds the stability bound 1/6", d->r);
    return HS_OK;
}

size_t elem_size(int dtype) { return dtype == HS_F64 ? sizeof(double) : sizeof(float); }

// Caller-owned time-level buffers: both or neither, distinct, not
// overlapping, 256-byte aligned (TMA and the 16-byte vector accesses need
// less; every CUDA allocator gives this).
int check_user_buffers(const hs_heat_desc* d, size_t bytes)
{
    if (!d->dev_buf0 && !d->dev_buf1) return HS_OK;
    if (!d->dev_buf0 || !d->dev_buf1)
        return fail(HS_EINVAL, "heat: give both dev_buf0 and dev_buf1, or neither");
    const uintptr_t a = reinterpret_cast<uintptr_t>(d->dev_buf0), b = reinterpret_cast<uintptr_t>(d->dev_buf1);
    if ((a | b) & 255) return fail(HS_EINVAL, "heat: dev_buf0 and dev_buf1 must be 256-byte aligned");
    if ((a < b ? b - a : a - b) < bytes)
        return fail(HS_EINVAL, "heat: dev_buf0 and dev_buf1 overlap (each needs %zu bytes)", bytes);
    return HS_OK;
}

// Plain FP64 runs the exact-sum arithmetic, except where a kernel has only the
// FP64-pipe form: temporal blocking and the variable-coefficient problem.
Arith pick_arith(const hs_heat_desc* d)
{
    const int depth = d->tdepth ? d->tdepth : 1;
    if (d->flags & HS_FIXED64) return A_FX64;
    if (d->flags & HS_EXACT_ROUNDING) return A_F64_EXACT;
    if (d->dtype == HS_F32) return A_F32;
    if ((d->flags & (HS_FP64_PIPE | HS_VARKAPPA)) || depth > 1) return A_F64;
    return A_F64_XS;
}

int pick_kchunk(const HeatGeom& g, uint32_t flags = 0, int dtype = HS_F64)
{
    // the FP32 variable-kappa kernel waits on its loads: short chunks (more
    // blocks in flight) measured 340 GLUP/s at 8 planes against 265 at the
    // 102 planes of the rule below (510^3)
    if ((flags & HS_VARKAPPA) && dtype == HS_F32) return g.nz > 2 ? std::min(8, g.nz - 2) : 1;
    // the FP64 variable-kappa kernel: about eight waves of three blocks per SM, in
    // chunks of 4 to 64 planes (510^3: 64 planes 140 GLUP/s, 32 139, 16 135, 128
    // 135; 96^3: 4 planes 16.5 us per step, 16 20.7, 32 35)
    if (flags & HS_VARKAPPA) {
        const int64_t tiles = (int64_t)((g.nx + 63) / 64) * ((g.ny + 7) / 8);
        const int64_t kc = (tiles * g.nz + kNumSMs * 24 - 1) / (kNumSMs * 24);
        return (int)std::min<int64_t>(std::max<int64_t>(4, std::min<int64_t>(kc, 64)), g.nz);
    }
    const int64_t blocks_xy = (int64_t)((g.nx + kBX - 1) / kBX) * ((g.ny + kBY - 1) / kBY);
    const int64_t target = (int64_t)kNumSMs * 8 * 4;   // about four waves of 8 blocks per SM
    const int64_t nzi = g.nz > 2 ? g.nz - 2 : 1;
    int64_t chunks = (target + blocks_xy - 1) / blocks_xy;
    if (chunks < 1) chunks = 1;
    int64_t kc = (nzi + chunks - 1) / chunks;
    if (kc < 8) kc = 8;
    if (kc > nzi) kc = nzi;
    return (int)kc;
}

template <typename T, bool EXACT>
int launch_interior_t(hs_heat* h, T param)
{
    const HeatGeom& g = h->g;
    if (g.nz < 3) return HS_OK;   // no plane lies strictly between the boundary planes
    const int kbeg = 1, kend = g.nz - 1;
    const int nchunks = (kend - kbeg + h->kchunk - 1) / h->kchunk;
    dim3 block(kBX, kBY, 1);
    dim3 grid((g.nx + kBX - 1) / kBX, (g.ny + kBY - 1) / kBY, nchunks);
    k_heat_interior<T, EXACT><<<grid, block, 0, h->stream>>>(
        (const T*)h->buf[h->cur], (T*)h->buf[1 - h->cur], g, param, kbeg, kend, h->kchunk, h->fx,
        (int)(h->fxseq % 3));
    HS_CHECK_LAUNCH("heat interior kernel");
    return HS_OK;
}

template <typename T, bool EXACT>
int launch_boundary_t(hs_heat* h, T param, cudaStream_t s)
{
    const HeatGeom& g = h->g;
    dim3 block(kBX, kBY, 1);
    dim3 grid((g.nx + kBX - 1) / kBX, (g.ny + kBY - 1) / kBY, g.nz >= 2 ? 2 : 1);
    k_heat_boundary<T, EXACT><<<grid, block, 0, s>>>(
        (const T*)h->buf[h->cur], (T*)h->buf[1 - h->cur], g, param, h->fx, (int)(h->fxseq % 3));
    HS_CHECK_LAUNCH("heat boundary kernel");
    return HS_OK;
}

template <typename T, bool EXACT>
int launch_full_t(hs_heat* h, T param)
{
    const HeatGeom& g = h->g;
    const int64_t n = (int64_t)g.nx * g.ny * g.nz;
    int64_t blocks = (n + 255) / 256;
    if (blocks > (int64_t)kNumSMs * 64) blocks = (int64_t)kNumSMs * 64;
    k_heat_full<T, EXACT><<<(unsigned)blocks, 256, 0, h->stream>>>(
        (const T*)h->buf[h->cur], (T*)h->buf[1 - h->cur], g, param, h->fx, (int)(h->fxseq % 3));
    HS_CHECK_LAUNCH("heat full-step kernel");
    return HS_OK;
}

enum Part { P_INTERIOR, P_BOUNDARY, P_FULL };

// The Interior kernel: planes 1 .. nz-2, staged through shared memory by TMA.
int launch_stream_interior(hs_heat* h)
{
    if (h->g.nz < 3) return HS_OK;   // no plane lies strictly between the boundary planes
    StreamCall c;
    c.arith = h->arith;
    c.kbeg = 1;
    c.kend = h->g.nz - 1;
    c.kc = h->kc_stream;
    c.map = &h->smaps[h->cur];
    c.dst = h->buf[1 - h->cur];
    c.g = &h->g;
    c.r = h->r;
    c.R = h->R;
    c.fx = h->fx;
    c.m3 = (int)(h->fxseq % 3);
    c.err = h->err;
    c.stream = h->stream;
    c.box[0] = h->sbox[0];
    c.box[1] = h->sbox[1];
    return stream_launch(c);
}

int launch_part_xs(hs_heat* h, Part p, cudaStream_t s)
{
    const HeatGeom& g = h->g;
    const double* src = (const double*)h->buf[h->cur];
    double* dst = (double*)h->buf[1 - h->cur];
    const int m3 = (int)(h->fxseq % 3);
    if (p == P_INTERIOR) return launch_stream_interior(h);
    if (p == P_BOUNDARY) {
        dim3 grid((g.nx + kBX - 1) / kBX, (g.ny + kBY - 1) / kBY, g.nz >= 2 ? 2 : 1);
        k_heat_boundary_xs<<<grid, dim3(kBX, kBY, 1), 0, s>>>(src, dst, g, h->r, h->fx, m3);
        HS_CHECK_LAUNCH("heat boundary kernel (FP64 exact sum)");
        return HS_OK;
    }
    const int64_t n = (int64_t)g.nx * g.ny * g.nz;
    int64_t blocks = (n + 255) / 256;
    if (blocks > (int64_t)kNumSMs * 64) blocks = (int64_t)kNumSMs * 64;
    k_heat_full_xs<<<(unsigned)blocks, 256, 0, h->stream>>>(src, dst, g, h->r, h->fx, m3);
    HS_CHECK_LAUNCH("heat full-step kernel (FP64 exact sum)");
    return HS_OK;
}

template <typename T, bool EXACT>
int launch_part(hs_heat* h, Part p, T param, cudaStream_t s)
{
    // FP64 is bound by the FP64 pipe, where the register z-march issues the
    // fewest extra instructions; the HBM-bound arithmetics stream through TMA.
    if (p == P_INTERIOR)
        return std::is_same<T, double>::value ? launch_interior_t<T, EXACT>(h, param)
                                              : launch_stream_interior(h);
    if (p == P_BOUNDARY) return launch_boundary_t<T, EXACT>(h, param, s);
    return launch_full_t<T, EXACT>(h, param);
}

// Planes [kbeg, kend) of a step of the variable-coefficient problem.
int vk_planes(hs_heat* h, int kbeg, int kend, cudaStream_t s)
{
    VkCall c = {};
    c.kbeg = kbeg;
    c.kend = kend;
    c.f64 = h->dtype == HS_F64;
    c.src = h->buf[h->cur];
    c.dst = h->buf[1 - h->cur];
    c.kap = h->kap;
    c.fdt = h->fdt;
    c.g = &h->g;
    c.bx = h->vbx;
    c.by = h->vby;
    c.bz = h->vbz;
    c.kchunk = h->kchunk;
    c.stream = s;
    c.fx = h->fx;   // FP64 only
    c.m3 = (int)(h->fxseq % 3);
    c.err = h->err;
    c.umap = &h->vmaps[h->cur];
    c.kmap = &h->vmaps[2];
    c.fmap = &h->vmaps[3];
    c.exact = h->kappa_ok;
    return vk_launch(c);
}

int vk_part(hs_heat* h, Part p, cudaStream_t s)
{
    const int nz = h->g.nz;
    if (p == P_FULL) return vk_planes(h, 0, nz, s);
    if (p == P_INTERIOR) return vk_planes(h, 1, nz - 1, s);
    const int rc = vk_planes(h, 0, 1, s);
    return rc != HS_OK || nz < 2 ? rc : vk_planes(h, nz - 1, nz, s);
}

// Launches one part of a step.  The Boundary kernel goes to stream s (the
// handle's own stream unless given); the other parts always to h->stream.
int do_part(hs_heat* h, Part p, cudaStream_t s = nullptr)
{
    if (!s || p != P_BOUNDARY) s = h->stream;
    if (h->flags & HS_VARKAPPA) return vk_part(h, p, s);
    switch (h->arith) {
    case A_F64: return launch_part<double, false>(h, p, h->r, s);
    case A_F64_EXACT: return launch_part<double, true>(h, p, h->r, s);
    case A_F32: return launch_part<float, false>(h, p, (float)h->r, s);
    case A_FX64: return launch_part<long long, false>(h, p, h->R, s);
    case A_F64_XS: return launch_part_xs(h, p, s);
    }
    return fail(HS_EINVAL, "heat: unknown arithmetic");
}

// The Interior part of a heat_step step, between a pair of timing events on
// the handle's stream while heat_time_interior is on.
int timed_interior(hs_heat* h)
{
    // past kMaxTimedLaunches unread records the launches go untimed
    if (!h->timing || h->tev_used >= kMaxTimedLaunches) return do_part(h, P_INTERIOR);
    const size_t i = 2 * h->tev_used;
    while (h->tev.size() < i + 2) {
        cudaEvent_t e;
        HS_TRY_CUDA(cudaEventCreate(&e), "heat_step: timing event");
        h->tev.push_back(e);
    }
    HS_TRY_CUDA(cudaEventRecord(h->tev[i], h->stream), "heat_step: timing event");
    const int rc = do_part(h, P_INTERIOR);
    if (rc != HS_OK) return rc;
    HS_TRY_CUDA(cudaEventRecord(h->tev[i + 1], h->stream), "heat_step: timing event");
    h->tev_used += 1;
    return HS_OK;
}

// Temporal depth when the descriptor leaves it to the library.  One step per
// pass of FP32 is bound by HBM (174 us at 512^3); two steps per pass move half
// the bytes (122 us), and where the tiles of 32-thread rows are the better
// ones heat_step takes passes of four steps while that many remain (112 us;
// tb_deep).  FP64 and FIXED64 are bound by the FP64 pipe and the integer pipes:
// blocking saves only bytes and adds the halo's work.  The variable-coefficient
// problem runs one step per pass.
int default_tdepth(Arith a, uint32_t flags)
{
    return (a == A_F32 && !(flags & HS_VARKAPPA)) ? 2 : 1;
}

int pick_kc_tb(const HeatGeom& g, int arith, int L)
{
    int TX = 0, TY = 0;
    tb_tile(arith, L, g.nx, &TX, &TY);
    const int64_t tiles = (int64_t)((g.nx + TX - 1) / TX) * ((g.ny + TY - 1) / TY);
    // Whole waves of resident blocks (two per SM at depth 2, one above), against
    // chunks long enough that the 2 L halo planes and the ring's start (about
    // three planes) stay cheap: the chunk length with the fewest planes in all,
    // where that saves 5% or more of those of about 1824 blocks (without that
    // margin FIXED64 at depth 4, 512^3, went from 571 to 616 us for a count 1%
    // lower).  Chunks of more than 64 L planes are left out: their blocks drift
    // apart and stop sharing halos in L2 (512^3 FP32 at depth 2: 121.9 us per
    // step, 124.1 with 256-plane chunks).  Against the fixed count: 123.1 ->
    // 121.9 there, 384^3 65.5 -> 56.5, depth 4 at 512^3 127.9 -> 112.3.
    const int64_t slots = (int64_t)kNumSMs * (L == 2 ? 2 : 1);
    auto planes = [&](int64_t kc) {
        const int64_t blocks = tiles * ((g.nz + kc - 1) / kc);
        return (blocks + slots - 1) / slots * (kc + 2 * L + 3);
    };
    // A grid too small to fill the GPU with chunks of 8 L planes takes chunks of 4 L
    // and up: with one wave or less, the planes of one chunk are the time of a pass
    // (96^3, 24 steps: FP32 at depth 2 240 -> 152 us, where tiles of 28 rows had made
    // it slower than those of 20 at 225; FIXED64 at depth 4 497 -> 311).
    // A launch holds 65535 chunks.
    const int64_t fit = ((int64_t)g.nz + 65534) / 65535;
    const int64_t floor_kc = tiles * ((g.nz + 8 * L - 1) / (8 * L)) < slots ? 4 * L : 8 * L;
    const int64_t shortest = std::max(fit, std::min<int64_t>(g.nz, floor_kc)), longest = std::min<int64_t>(g.nz, 64 * L);
    const int64_t chunks = (12 * (int64_t)kNumSMs + tiles - 1) / tiles;
    int64_t best = std::max(shortest, (g.nz + chunks - 1) / chunks);
    int64_t least = planes(best) * 19 / 20;
    for (int64_t kc = longest; kc >= shortest; --kc) {
        const int64_t p = planes(kc);
        if (p < least) {
            least = p;
            best = kc;
        }
    }
    return (int)best;
}

int pick_kc_stream(const HeatGeom& g, int arith)
{
    const int tw = 512 / (int)g.elem;                  // tile width: 32 threads x one 16-byte vector
    const int ry = stream_rows_for(arith);
    const int64_t tiles = (int64_t)((g.nx + tw - 1) / tw) * ((g.ny + ry - 1) / ry);
    // about four waves of 3 blocks of 16 rows per SM; the exact-sum kernel (8 rows,
    // 7 resident blocks of 128 threads per SM) gets 64 blocks per SM, about 9
    // waves of 27-plane chunks at 512^3 -- measured ahead of 4 waves of longer
    // chunks and 12 waves of shorter ones
    const int64_t target = (int64_t)kNumSMs * (arith == A_F64_XS ? 16 : 3) * 4;
    const int64_t planes = g.nz > 2 ? g.nz - 2 : 1;
    int64_t chunks = (target + tiles - 1) / tiles;
    if (chunks < 1) chunks = 1;
    int64_t kc = (planes + chunks - 1) / chunks;
    // every chunk stages two planes more than it writes: 8 planes at least, and
    // in the exact-sum kernel up to 16 where three waves remain
    int64_t lo = 8;
    if (arith == A_F64_XS) {
        const int64_t wave = (int64_t)kNumSMs * 7;
        lo = planes * tiles / (3 * wave);
        lo = lo < 8 ? 8 : (lo > 16 ? 16 : lo);
    }
    if (kc < lo) kc = lo;
    if (kc > planes) kc = planes;
    return (int)kc;
}

// Steps of one launch of the multi-step kernel, whose blocks may fill the GPU: at
// 3 to 40 us per step other streams' kernels wait 40 ms at most, and a launch in
// 1024 steps costs less than 0.2%.
constexpr int64_t kMultiSteps = 1024;

// Whether heat_step advances this handle with the multi-step kernel, unless the
// caller asked for another schedule or depth.  Its time goes with its bricks, the
// streaming kernel's and the blocked pass's only above a floor; thin grids leave
// bricks and tiles alike partly empty.  Per step, launches / multi-step kernel:
//   FP64, to 24 bricks per SM: 64^3 14.4 / 3.4 us, 160^3 28.3 / 22.5, 500 x 9 x 900
//     (3600) 33.8 / 32.3; 66 x 200 x 310 (3900) 35.7 / 36.0, 20 x 400 x 400 (5000)
//     43.8 / 45.6, 16 x 640 x 400 (8000) 63.6 / 74.7.  From 2^22 points 176^3 (2904)
//     28.0 / 30.7.
//   FIXED64, to 40: 160^3 24.7 / 19.5, 20 x 400 x 400 43.7 / 39.0; 17 x 600 x 380
//     (7125) 57.3 / 58.7.  From 2^22 points 176^3 25.3 / 25.8.
//   FP32 against the blocked pass, four steps deep, to 6: 64^3 7.3 / 2.6, 128^3 7.2 /
//     6.1, 60 x 200 x 260 (845) 7.8 / 6.4; 144^3 (972) 7.3 / 7.8, 160^3 7.3 / 8.2, 65
//     x 340 x 340 (3740) 13.4 / 23.0.  Two deep (tb_deep), to 9: 250 x 140 x 140
//     (1260) 10.3 / 8.8; 370 x 120 x 120 (1440) 10.3 / 11.2.  Thin grids, whose tiles
//     hold 7/4 of the bricks' points and more: 60 x 260 x 260 (1105) 8.8 / 8.2, 16 x
//     640 x 400 (4000) 24.7 / 17.4; from 2^22 points only the narrowest: 20 x 600 x 600
//     30.3 / 27.6, 60 x 360 x 370 13.4 / 18.8; 640 x 640 x 10, mostly z halo, 10.4 / 7.6.
//   FP32 one step at a time (tdepth 1): 192^3 15.9 / 10.7, 65 x 340 x 340 22.8 / 22.5.
bool use_multi(const hs_heat_desc* d, const hs_heat* h)
{
    if (d->flags & (HS_SCHED_FULL | HS_VARKAPPA)) return false;
    if (h->arith != A_F32 && h->arith != A_FX64 && h->arith != A_F64_XS) return false;
    if (d->tdepth > 1) return false;   // the caller asked for temporal blocking
    const HeatGeom& g = h->g;
    const int64_t npts = (int64_t)g.nx * g.ny * g.nz, bricks = multi_bricks(h->arith, g);
    const bool below22 = npts < ((int64_t)1 << 22);
    if (h->arith == A_F64_XS) return below22 && bricks <= 24 * kNumSMs;
    if (h->arith == A_FX64) return below22 && bricks <= 40 * kNumSMs;
    if (npts >= ((int64_t)1 << 23)) return false;
    if (d->tdepth == 1 || bricks <= (h->deep ? 6 : 9) * kNumSMs || g.nx <= 24) return true;
    int TX = 0, TY = 0;
    const int L = h->deep ? 4 : 2;
    tb_tile(A_F32, L, g.nx, &TX, &TY);
    const int64_t tiles =
        (int64_t)((g.nx + TX - 1) / TX) * TX * ((g.ny + TY - 1) / TY) * TY * ((int64_t)g.nz + 2 * L + 3);
    return below22 && 7 * 4096 * bricks <= 4 * tiles;
}

// n_steps steps in one launch of the multi-step kernel.
int multi_steps(hs_heat* h, int n_steps)
{
    MultiCall c;
    c.arith = h->arith;
    c.buf[0] = h->buf[0];
    c.buf[1] = h->buf[1];
    c.cur = h->cur;
    c.g = &h->g;
    c.r = h->r;
    c.R = h->R;
    c.fx = h->fx;
    c.m3 = (int)(h->fxseq % 3);
    c.steps = n_steps;
    c.sync = h->msync;
    c.err = h->err;
    c.stream = h->stream;
    const int rc = multi_launch(c);
    if (rc != HS_OK) return rc;
    h->cur = (int)((h->cur + n_steps) & 1);
    h->steps += n_steps;
    h->fxseq += n_steps;
    return HS_OK;
}

// One pass of L steps with the temporally blocked kernel.
int tb_pass(hs_heat* h, int L)
{
    TbCall c;
    c.arith = h->arith;
    c.L = L;
    c.kc = pick_kc_tb(h->g, h->arith, L);
    c.map = &h->maps[h->cur];
    c.dst = h->buf[1 - h->cur];
    c.g = &h->g;
    c.r = h->r;
    c.R = h->R;
    c.fx = h->fx;
    c.m3 = (int)(h->fxseq % 3);
    c.err = h->err;
    c.stream = h->stream;
    c.box[0] = h->tbox[0];
    c.box[1] = h->tbox[1];
    int rc = tb_launch(c);
    if (rc != HS_OK) return rc;
    h->cur = 1 - h->cur;
    h->steps += L;
    h->fxseq += 1;
    return HS_OK;
}

// Copies between a dense nx*ny*nz array and the interior of a padded buffer.
int copy_interior(hs_heat* h, void* buf, const void* dense, void* dense_out, cudaMemcpyKind kind)
{
    const HeatGeom& g = h->g;
    const size_t e = h->elem;
    cudaMemcpy3DParms p = {};
    p.extent = make_cudaExtent((size_t)g.nx * e, (size_t)g.ny, (size_t)g.nz);
    cudaPitchedPtr padded = make_cudaPitchedPtr(buf, (size_t)g.pitch * e, (size_t)g.pitch,
                                                (size_t)(g.ny + 2));
    cudaPos inner = make_cudaPos((size_t)g.lead * e, 1, 1);
    if (dense) {   // dense -> padded
        p.srcPtr = make_cudaPitchedPtr(const_cast<void*>(dense), (size_t)g.nx * e, (size_t)g.nx,
                                       (size_t)g.ny);
        p.dstPtr = padded;
        p.dstPos = inner;
    } else {       // padded -> dense
        p.srcPtr = padded;
        p.srcPos = inner;
        p.dstPtr = make_cudaPitchedPtr(dense_out, (size_t)g.nx * e, (size_t)g.nx, (size_t)g.ny);
    }
    p.kind = kind;
    HS_TRY_CUDA(cudaMemcpy3DAsync(&p, h->stream), "heat: interior copy");
    return HS_OK;
}

// The interior between the dense layout (x fastest, nx * ny * nz) and the
// padded one, a row of x per block step, as raw W-sized words (16-byte words
// when a row and the dense base allow; every padded interior row starts
// 16-byte aligned).  All sizes and offsets are in words.
template <typename W>
__global__ void __launch_bounds__(256)
    k_interior_copy(const W* __restrict__ src, W* __restrict__ dst, int64_t nxw, int64_t pitch_w,
                    int64_t plane_w, int64_t lead_w, int ny, int nz, int to_padded)
{
    const int64_t rows = (int64_t)ny * nz;
    for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {
        const int64_t j = r % ny, k = r / ny;
        const int64_t pd = (k + 1) * plane_w + (j + 1) * pitch_w + lead_w, dn = r * nxw;
        const W* s = src + (to_padded ? dn : pd);
        W* d = dst + (to_padded ? pd : dn);
        for (int64_t i = threadIdx.x; i < nxw; i += blockDim.x) d[i] = s[i];
    }
}

// Device-side re-layout of the interior: dense -> padded (to_padded) or back.
int interior_copy(hs_heat* h, const void* src, void* dst, bool to_padded)
{
    const HeatGeom& g = h->g;
    const int64_t e = (int64_t)h->elem;
    const void* dense = to_padded ? src : dst;
    const int64_t rows = (int64_t)g.ny * g.nz;
    const unsigned blocks = (unsigned)(rows < (int64_t)kNumSMs * 16 ? rows : (int64_t)kNumSMs * 16);
    if ((g.nx * e) % 16 == 0 && (reinterpret_cast<uintptr_t>(dense) & 15) == 0) {
        k_interior_copy<uint4><<<blocks, 256, 0, h->stream>>>(
            (const uint4*)src, (uint4*)dst, g.nx * e / 16, g.pitch * e / 16, g.plane * e / 16, g.lead * e / 16,
            g.ny, g.nz, to_padded);
    } else if (e == 8) {
        k_interior_copy<unsigned long long><<<blocks, 256, 0, h->stream>>>(
            (const unsigned long long*)src, (unsigned long long*)dst, g.nx, g.pitch, g.plane, g.lead, g.ny, g.nz,
            to_padded);
    } else {
        k_interior_copy<unsigned><<<blocks, 256, 0, h->stream>>>((const unsigned*)src, (unsigned*)dst, g.nx, g.pitch,
                                                                 g.plane, g.lead, g.ny, g.nz, to_padded);
    }
    HS_CHECK_LAUNCH("heat: interior copy kernel");
    return HS_OK;
}

unsigned conv_blocks(const HeatGeom& g)
{
    const int64_t n = (int64_t)g.nx * g.ny * g.nz;
    int64_t b = (n + 255) / 256;
    const int64_t cap = (int64_t)kNumSMs * 16;
    return (unsigned)(b < cap ? (b < 1 ? 1 : b) : cap);
}

}  // namespace

namespace hcg {

int heat_batch_view(hs_heat_t h, HeatBatchView* v)
{
    if (!h || !v) return fail(HS_EINVAL, "heat batch: NULL handle");
    v->g = h->g;
    v->buf[0] = h->buf[0];
    v->buf[1] = h->buf[1];
    v->r = h->r;
    v->arith = h->arith;
    v->cur = h->cur;
    v->vk = (h->flags & HS_VARKAPPA) ? 1 : 0;
    v->fx = h->fx;
    v->m3 = (int)(h->fxseq % 3);
    v->stream = h->stream;
    return HS_OK;
}

int heat_batch_advance(hs_heat_t h, int64_t steps)
{
    if (!h) return fail(HS_EINVAL, "heat batch: NULL handle");
    h->cur = (int)((h->cur + steps) & 1);
    h->steps += steps;
    h->fxseq += steps;
    return HS_OK;
}

}  // namespace hcg

extern "C" {

int heat_buffer_bytes(const hs_heat_desc* desc, size_t* bytes)
{
    int rc = check_desc(desc);
    if (rc != HS_OK) return rc;
    if (!bytes) return fail(HS_EINVAL, "heat_buffer_bytes: bytes is NULL");
    const HeatGeom g = make_geom(desc->nx, desc->ny, desc->nz, elem_size(desc->dtype));
    *bytes = (size_t)g.total * elem_size(desc->dtype);
    return HS_OK;
}

int heat_device_bytes(const hs_heat_desc* desc, size_t* bytes)
{
    int rc = check_desc(desc);
    if (rc != HS_OK) return rc;
    if (!bytes) return fail(HS_EINVAL, "heat_device_bytes: bytes is NULL");
    const HeatGeom g = make_geom(desc->nx, desc->ny, desc->nz, elem_size(desc->dtype));
    const bool user_bufs = desc->dev_buf0 || desc->dev_buf1;
    *bytes = user_bufs ? 0 : 2 * (size_t)g.total * elem_size(desc->dtype);
    const Arith a = pick_arith(desc);
    if (a == A_FX64 || a == A_F64_XS) *bytes += sizeof(FxState);
    if (desc->flags & HS_VARKAPPA)   // kappa and dt f
        *bytes += 2 * (size_t)g.total * elem_size(desc->dtype) + (desc->dtype == HS_F64 ? sizeof(FxState) : 0);
    return HS_OK;
}

int heat_create(hs_heat_t* out, const hs_heat_desc* desc)
{
    if (!out) return fail(HS_EINVAL, "heat_create: out is NULL");
    *out = nullptr;
    int rc = check_desc(desc);
    if (rc != HS_OK) return rc;
    hs_heat* h = new (std::nothrow) hs_heat();
    if (!h) return fail(HS_ENOMEM, "heat_create: host allocation failed");
    h->dtype = desc->dtype;
    h->elem = elem_size(desc->dtype);
    h->g = make_geom(desc->nx, desc->ny, desc->nz, h->elem);
    h->r = desc->r;
    h->flags = desc->flags;
    h->arith = pick_arith(desc);
    // r <= 1/6 < 1/2, so r 2^64 < 2^63.  For r >= 2^-11 it is an integer (r's
    // last bit is worth at least 2^-64), so R holds r exactly; a smaller r is
    // rounded to the nearest multiple of 2^-64.
    h->R = (h->arith == A_FX64) ? std::llrint(std::ldexp(desc->r, 64)) : 0;
    h->stream = (cudaStream_t)desc->stream;
    h->cur = 0;
    h->steps = 0;
    h->kchunk = pick_kchunk(h->g, desc->flags, desc->dtype);
    h->tdepth = desc->tdepth ? desc->tdepth : default_tdepth(h->arith, desc->flags);
    if (h->flags & HS_SCHED_FULL) h->tdepth = 1;
    h->deep = desc->tdepth == 0 && h->tdepth > 1 && tb_deep(h->arith, h->g.nx);
    const size_t bytes = (size_t)h->g.total * h->elem;
    rc = check_user_buffers(desc, bytes);
    if (rc != HS_OK) {
        delete h;
        return rc;
    }
    h->owns_buf = !desc->dev_buf0;
    // one allocation holds the handle's words (error word, per-step state, grid
    // barrier) and, unless the caller owns them, the two buffers
    const size_t fbytes = (bytes + 255) & ~(size_t)255;
    const size_t total = kHeatStateBytes + (h->owns_buf ? 2 * fbytes : 0);
    cudaError_t ea = dev_alloc(&h->arena, total, h->stream);
    if (ea != cudaSuccess) {
        h->arena = nullptr;
        rc = cuda_fail(ea, "heat_create: device allocation");
        heat_destroy(h);
        return rc;
    }
    char* const base = (char*)h->arena;
    h->err = (int*)base;
    FxState* const fx_state = (FxState*)(base + kHeatFxOffset);
    if (use_multi(desc, h)) h->msync = base + kHeatBarOffset;
    h->buf[0] = h->owns_buf ? (void*)(base + kHeatStateBytes) : desc->dev_buf0;
    h->buf[1] = h->owns_buf ? (void*)(base + kHeatStateBytes + fbytes) : desc->dev_buf1;
    ea = cudaMemsetAsync(h->arena, 0, total, h->stream);
    for (int b = 0; b < 2 && !h->owns_buf && ea == cudaSuccess; ++b)
        ea = cudaMemsetAsync(h->buf[b], 0, bytes, h->stream);
    if (ea != cudaSuccess) {
        rc = cuda_fail(ea, "heat_create: cudaMemsetAsync");
        heat_destroy(h);
        return rc;
    }
    {
        const CUtensorMapDataType dt = h->arith == A_FX64   ? CU_TENSOR_MAP_DATA_TYPE_INT64
                                       : h->dtype == HS_F64 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64
                                                            : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
        uint32_t bx = 0, by = 0;
        stream_box(h->arith, &bx, &by);
        h->sbox[0] = bx;
        h->sbox[1] = by;
        for (int b = 0; b < 2; ++b) {
            const int e = encode_field_map(&h->smaps[b], h->buf[b], dt, h->elem, (uint64_t)h->g.pitch,
                                           (uint64_t)(h->g.ny + 2), (uint64_t)(h->g.nz + 2), bx, by);
            if (e != 0) {
                rc = cuda_fail((cudaError_t)e, "heat_create: TMA tensor map (streaming)");
                heat_destroy(h);
                return rc;
            }
        }
        h->kc_stream = pick_kc_stream(h->g, h->arith);
    }
    if (h->tdepth > 1) {
        const CUtensorMapDataType dt = h->arith == A_FX64   ? CU_TENSOR_MAP_DATA_TYPE_INT64
                                       : h->dtype == HS_F64 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64
                                                            : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
        uint32_t box_x = 0, box_y = 0;
        tb_box(h->arith, h->g.nx, &box_x, &box_y);
        h->tbox[0] = box_x;
        h->tbox[1] = box_y;
        for (int b = 0; b < 2; ++b) {
            const int e = encode_field_map(&h->maps[b], h->buf[b], dt, h->elem, (uint64_t)h->g.pitch,
                                           (uint64_t)(h->g.ny + 2), (uint64_t)(h->g.nz + 2), box_x,
                                           box_y);
            if (e != 0) {
                rc = cuda_fail((cudaError_t)e, "heat_create: TMA tensor map");
                heat_destroy(h);
                return rc;
            }
        }
    }
    if (h->arith == A_FX64 || h->arith == A_F64_XS) h->fx = fx_state;
    if (h->flags & HS_VARKAPPA) {
        const size_t bytes = (size_t)h->g.total * h->elem;
        cudaError_t e = dev_alloc(&h->kap, bytes, h->stream);
        if (e == cudaSuccess) e = dev_alloc(&h->fdt, bytes, h->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(h->kap, 0, bytes, h->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(h->fdt, 0, bytes, h->stream);
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "heat_create: kappa/source arrays");
            heat_destroy(h);
            return rc;
        }
        const double hx = 1.0 / (h->g.nx + 1), hy = 1.0 / (h->g.ny + 1), hz = 1.0 / (h->g.nz + 1);
        const double hmin = std::fmin(hx, std::fmin(hy, hz));
        const double dt = desc->r * hmin * hmin;
        h->vbx = dt / (2.0 * hx * hx);
        h->vby = dt / (2.0 * hy * hy);
        h->vbz = dt / (2.0 * hz * hz);
        VkCall c = {};
        c.f64 = h->dtype == HS_F64;
        c.kap = h->kap;
        c.fdt = h->fdt;
        c.g = &h->g;
        c.stream = h->stream;
        int kappa_off = 1;
        if (c.f64) {
            e = dev_alloc((void**)&c.kappa_off, sizeof(int), h->stream);
            if (e == cudaSuccess) e = cudaMemsetAsync(c.kappa_off, 0, sizeof(int), h->stream);
            if (e != cudaSuccess) {
                rc = cuda_fail(e, "heat_create: kappa check word");
                heat_destroy(h);
                return rc;
            }
        }
        rc = vk_init(c, dt);
        if (rc == HS_OK && c.f64) {
            cudaError_t e2 = cudaMemcpyAsync(&kappa_off, c.kappa_off, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
            if (e2 == cudaSuccess) e2 = cudaStreamSynchronize(h->stream);
            if (e2 != cudaSuccess) rc = cuda_fail(e2, "heat_create: kappa check");
        }
        if (c.kappa_off) dev_free(c.kappa_off, h->stream);
        if (rc != HS_OK) {
            heat_destroy(h);
            return rc;
        }
        if (h->dtype == HS_F64) h->fx = fx_state;   // the exact-sum form tracks the field's largest exponent
        h->kappa_ok = kappa_off == 0;
        if (h->dtype == HS_F64) {
            const int em = vk_maps(h->vmaps, h->buf, h->kap, h->fdt, h->g);
            if (em != 0) {
                rc = cuda_fail((cudaError_t)em, "heat_create: TMA tensor map (variable kappa)");
                heat_destroy(h);
                return rc;
            }
        }
    }
    // A Boundary kernel beside the Interior one pays for its extra API calls
    // once the Interior kernel takes tens of microseconds (2^22 points and up).
    const int64_t npts = (int64_t)h->g.nx * h->g.ny * h->g.nz;
    if (!(h->flags & (HS_SCHED_FULL | HS_VARKAPPA)) && h->tdepth == 1 && npts >= kForkMinPoints && h->g.nz >= 3) {
        cudaError_t e = cudaStreamCreateWithFlags(&h->bstream, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->ev_join, cudaEventDisableTiming);
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "heat_create: side stream");
            heat_destroy(h);
            return rc;
        }
    }
    *out = h;
    return HS_OK;
}

int heat_upload(hs_heat_t h, const void* u, int src_is_device)
{
    if (!h || !u) return fail(HS_EINVAL, "heat_upload: NULL handle or field");
    // The field goes to buffer 0 only.  The spare buffer needs no copy: every
    // interior value of it is written by the next step before it is read, and
    // its boundary layer has been zero since creation -- the same state the
    // paper reaches by uploading u_old and u_new alike.
    // device sources and pinned, mapped host sources are re-laid out by a
    // kernel (the latter reading host memory directly); pageable host sources
    // go through one strided 3-D copy (measured faster over the host link than
    // a contiguous copy into a staging buffer plus the re-layout)
    const void* mapped = src_is_device ? nullptr : mapped_host_ptr(u);
    int rc = src_is_device ? interior_copy(h, u, h->buf[0], true)
             : mapped      ? interior_copy(h, mapped, h->buf[0], true)
                           : copy_interior(h, h->buf[0], u, nullptr, cudaMemcpyHostToDevice);
    if (rc != HS_OK) return rc;
    if (h->arith == A_FX64) {
        HS_TRY_CUDA(cudaMemsetAsync(h->fx, 0, sizeof(FxState), h->stream), "heat_upload: memset");
        const unsigned blocks = conv_blocks(h->g);
        k_fx_maxabs<<<blocks, 256, 0, h->stream>>>((const double*)h->buf[0], h->g, h->fx);
        HS_CHECK_LAUNCH("heat_upload: max|u| kernel");
        k_fx_encode<<<blocks, 256, 0, h->stream>>>((double*)h->buf[0], h->g, h->fx);
        HS_CHECK_LAUNCH("heat_upload: fixed-point encode kernel");
    } else if (h->arith == A_F64_XS || (h->fx && (h->flags & HS_VARKAPPA))) {
        // slot 0: the largest |u| bit pattern of the uploaded field
        HS_TRY_CUDA(cudaMemsetAsync(h->fx, 0, sizeof(FxState), h->stream), "heat_upload: memset");
        k_fx_maxabs<<<conv_blocks(h->g), 256, 0, h->stream>>>((const double*)h->buf[0], h->g, h->fx);
        HS_CHECK_LAUNCH("heat_upload: max|u| kernel");
    }
    h->cur = 0;
    h->steps = 0;
    h->fxseq = 0;
    return HS_OK;
}

int heat_interior(hs_heat_t h)
{
    if (!h) return fail(HS_EINVAL, "heat_interior: NULL handle");
    return do_part(h, P_INTERIOR);
}

int heat_boundary(hs_heat_t h)
{
    if (!h) return fail(HS_EINVAL, "heat_boundary: NULL handle");
    return do_part(h, P_BOUNDARY);
}

int heat_swap(hs_heat_t h)
{
    if (!h) return fail(HS_EINVAL, "heat_swap: NULL handle");
    h->cur = 1 - h->cur;
    h->steps += 1;
    h->fxseq += 1;
    return HS_OK;
}

int heat_step(hs_heat_t h, int64_t n_steps)
{
    if (!h) return fail(HS_EINVAL, "heat_step: NULL handle");
    if (n_steps < 0) return fail(HS_EINVAL, "heat_step: n_steps = %lld < 0", (long long)n_steps);
    if (h->msync && !h->timing) {
        while (n_steps > 0) {
            const int part = (int)std::min<int64_t>(n_steps, kMultiSteps);
            const int rc = multi_steps(h, part);
            if (rc != HS_OK) return rc;
            n_steps -= part;
        }
        return HS_OK;
    }
    if (h->tdepth > 1) {
        // passes of the handle's depth, then the remainder in the largest built depths
        const int top = h->deep ? 4 : h->tdepth;
        int64_t left = n_steps;
        static const int depths[] = {4, 3, 2};
        for (int L : depths) {
            if (L > top) continue;
            for (; left >= L; left -= L) {
                const int rc = tb_pass(h, L);
                if (rc != HS_OK) return rc;
            }
        }
        for (; left > 0; --left) {   // a last single step: Boundary + Interior
            int rc = do_part(h, P_BOUNDARY);
            if (rc == HS_OK) rc = do_part(h, P_INTERIOR);
            if (rc != HS_OK) return rc;
            h->cur = 1 - h->cur;
            h->steps += 1;
            h->fxseq += 1;
        }
        return HS_OK;
    }
    for (int64_t m = 0; m < n_steps; ++m) {
        int rc;
        if ((h->flags & HS_SCHED_FULL) || ((h->flags & HS_VARKAPPA) && !h->timing)) {
            rc = do_part(h, P_FULL);   // variable kappa: all planes in one launch
        } else if (h->bstream) {
            // Interior on the handle's stream, Boundary beside it on the side
            // stream (the two write disjoint planes of the new level and fold
            // into the step maximum with atomics); the next step starts after both
            HS_TRY_CUDA(cudaEventRecord(h->ev_fork, h->stream), "heat_step: fork event");
            rc = timed_interior(h);
            if (rc != HS_OK) return rc;
            HS_TRY_CUDA(cudaStreamWaitEvent(h->bstream, h->ev_fork, 0), "heat_step: fork wait");
            rc = do_part(h, P_BOUNDARY, h->bstream);
            if (rc != HS_OK) return rc;
            HS_TRY_CUDA(cudaEventRecord(h->ev_join, h->bstream), "heat_step: join event");
            HS_TRY_CUDA(cudaStreamWaitEvent(h->stream, h->ev_join, 0), "heat_step: join wait");
        } else {
            rc = do_part(h, P_BOUNDARY);
            if (rc == HS_OK) rc = timed_interior(h);
        }
        if (rc != HS_OK) return rc;
        h->cur = 1 - h->cur;
        h->steps += 1;
        h->fxseq += 1;
    }
    return HS_OK;
}

int heat_time_interior(hs_heat_t h, int enable)
{
    if (!h) return fail(HS_EINVAL, "heat_time_interior: NULL handle");
    h->timing = enable != 0;
    return HS_OK;
}

int heat_interior_time(hs_heat_t h, double* mean_ms, int64_t* launches)
{
    if (!h) return fail(HS_EINVAL, "heat_interior_time: NULL handle");
    double total = 0.0;
    const size_t n = h->tev_used;
    if (n > 0) HS_TRY_CUDA(cudaEventSynchronize(h->tev[2 * n - 1]), "heat_interior_time: synchronize");
    for (size_t i = 0; i < n; ++i) {
        float ms = 0.0f;
        HS_TRY_CUDA(cudaEventElapsedTime(&ms, h->tev[2 * i], h->tev[2 * i + 1]),
                    "heat_interior_time: elapsed time");
        total += ms;
    }
    h->tev_used = 0;
    if (mean_ms) *mean_ms = n ? total / (double)n : 0.0;
    if (launches) *launches = (int64_t)n;
    return HS_OK;
}

int heat_read(hs_heat_t h, void* dst, int dst_is_device)
{
    if (!h || !dst) return fail(HS_EINVAL, "heat_read: NULL handle or destination");
    void* src = h->buf[h->cur];
    void* spare = h->buf[1 - h->cur];
    if (h->arith == A_FX64) {
        // Decode into the spare buffer's interior; the next step overwrites
        // all of it, and its boundary layer stays zero.
        k_fx_decode<<<conv_blocks(h->g), 256, 0, h->stream>>>(
            (const long long*)h->buf[h->cur], (double*)spare, h->g, h->fx, (int)(h->fxseq % 3));
        HS_CHECK_LAUNCH("heat_read: fixed-point decode kernel");
        src = spare;
    }
    // device and pinned, mapped host destinations by a kernel, pageable host
    // ones by one strided 3-D copy
    void* mapped = dst_is_device ? nullptr : mapped_host_ptr(dst);
    int rc = dst_is_device ? interior_copy(h, src, dst, false)
             : mapped      ? interior_copy(h, src, mapped, false)
                           : copy_interior(h, src, nullptr, dst, cudaMemcpyDeviceToHost);
    if (rc != HS_OK) return rc;
    // status reads on the handle's own stream (a legacy-stream copy would also
    // wait for every other blocking stream, e.g. a batch running elsewhere)
    int err = 0;
    HS_TRY_CUDA(cudaMemcpyAsync(&err, h->err, sizeof(int), cudaMemcpyDeviceToHost, h->stream),
                "heat_read: error word");
    HS_TRY_CUDA(cudaStreamSynchronize(h->stream), "heat_read: stream synchronize");
    if (err == 2)
        return fail(HS_ECUDA, "heat_read: a bounded wait inside a TMA-staged heat kernel ran out and "
                              "the block's loads in flight did not complete in time; the field is not "
                              "valid and the CUDA context should be treated as suspect");
    if (err)
        return fail(HS_ETIMEOUT, "heat_read: a bounded wait inside a heat kernel (for a TMA load, or at the "
                                 "multi-step kernel's barrier) ran out; the field is not valid");
    if (h->arith == A_FX64) {
        FxState st;
        HS_TRY_CUDA(cudaMemcpyAsync(&st, h->fx, sizeof(st), cudaMemcpyDeviceToHost, h->stream),
                    "heat_read: state");
        HS_TRY_CUDA(cudaStreamSynchronize(h->stream), "heat_read: stream synchronize");
        if (st.nonfinite)
            return fail(HS_ERANGE, "heat_read: the uploaded field held NaN or Inf, which the "
                                   "fixed-point form cannot carry");
    }
    return HS_OK;
}

int heat_steps_done(hs_heat_t h, int64_t* steps)
{
    if (!h || !steps) return fail(HS_EINVAL, "heat_steps_done: NULL argument");
    *steps = h->steps;
    return HS_OK;
}

int heat_set_kchunk(hs_heat_t h, int32_t planes)
{
    if (!h) return fail(HS_EINVAL, "heat_set_kchunk: NULL handle");
    if (planes < 0) return fail(HS_EINVAL, "heat_set_kchunk: planes = %d < 0", planes);
    const int interior = h->g.nz > 2 ? h->g.nz - 2 : 1;
    if (planes == 0) {
        h->kchunk = pick_kchunk(h->g, h->flags, h->dtype);
        h->kc_stream = pick_kc_stream(h->g, h->arith);
    } else {
        h->kchunk = h->kc_stream = planes < interior ? planes : interior;
    }
    return HS_OK;
}

int heat_get_kchunk(hs_heat_t h, int32_t* planes)
{
    if (!h || !planes) return fail(HS_EINVAL, "heat_get_kchunk: NULL argument");
    const bool streaming = !(h->flags & HS_VARKAPPA) && h->arith != A_F64 && h->arith != A_F64_EXACT;
    *planes = streaming ? h->kc_stream : h->kchunk;
    return HS_OK;
}

int heat_get_tdepth(hs_heat_t h, int32_t* tdepth)
{
    if (!h || !tdepth) return fail(HS_EINVAL, "heat_get_tdepth: NULL argument");
    *tdepth = h->tdepth;
    return HS_OK;
}

int heat_destroy(hs_heat_t h)
{
    if (!h) return HS_OK;
    int rc = HS_OK;
    if (h->arena) {
        cudaError_t e = cudaStreamSynchronize(h->stream);
        if (e != cudaSuccess) rc = cuda_fail(e, "heat_destroy: stream synchronize");
    }
    if (h->bstream) {
        cudaError_t e = cudaStreamSynchronize(h->bstream);
        if (e != cudaSuccess && rc == HS_OK) rc = cuda_fail(e, "heat_destroy: side stream synchronize");
        (void)cudaStreamDestroy(h->bstream);
    }
    for (cudaEvent_t e : h->tev) (void)cudaEventDestroy(e);
    if (h->ev_fork) (void)cudaEventDestroy(h->ev_fork);
    if (h->ev_join) (void)cudaEventDestroy(h->ev_join);
    dev_free(h->arena, h->stream);
    dev_free(h->kap, h->stream);
    dev_free(h->fdt, h->stream);
    delete h;
    return rc;
}

}  // extern "C"
