// The paper's variable-coefficient heat problem (Section 4, Eqs. 1-4):
//     du/dt = div(kappa grad u) + f,  kappa = 0.5 + 0.45 sin(pi x) sin(pi y) sin(pi z),
//     f = 1 + cos(pi x) cos(pi y) cos(pi z),
//     u' = u + dt f + sum_d dt/(2 h_d^2) D_d(u),
//     D_x = (k[i+1] + k[i]) (u[i+1] - u[i]) - (k[i] + k[i-1]) (u[i] - u[i-1])
// (face-averaged kappa: the reading of the unprinted D that matches
// beta = dt/(2h^2)).  As in the paper's Algorithm "1-GPU Baseline", the
// coefficients and dt f are arrays resident beside u, dt f on the interior.
// Interior and Boundary kernels as for the constant-coefficient update.
//
// Every node of the padded box keeps its kappa: u, kappa and dt f in, u' out, 32
// bytes per FP64 update and 16 per FP32 update.  FP64 forms the operator sum in
// integers on the field's fixed-point scale -- each face's flux kappa dU from
// three 32-bit products, the six fluxes summed in 64 bits and rounded to a
// double once -- and spends two or three FP64 instructions per update, where
// the formula takes 23.  Fields outside that form's exponent range use the
// formula itself.
#include <algorithm>
#include <cmath>

#include "heat_common.cuh"
#include "tma.cuh"

namespace hcg {

constexpr int kVkBX = 32, kVkBY = 8;

// kappa on every padded node, dt f on interior nodes (zero on the boundary).
// Sets *off = 1 if a kappa lies outside [0.5, 1), where xs_flux would not hold it
// (0.5 + 0.45 s with s in [0, 1] never does).
template <typename T>
__global__ void __launch_bounds__(256) k_vk_init(T* __restrict__ kap, T* __restrict__ fdt, HeatGeom g,
                                                 double dt, int* off)
{
    const double hx = 1.0 / (g.nx + 1), hy = 1.0 / (g.ny + 1), hz = 1.0 / (g.nz + 1);
    const int64_t n = (int64_t)(g.nx + 2) * (g.ny + 2) * (g.nz + 2);
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int I = (int)(t % (g.nx + 2));
        const int64_t jk = t / (g.nx + 2);
        const int J = (int)(jk % (g.ny + 2));
        const int K = (int)(jk / (g.ny + 2));
        const int64_t c = (int64_t)K * g.plane + (int64_t)J * g.pitch + g.lead - 1 + I;
        const double x = I * hx, y = J * hy, z = K * hz;
        const double k = 0.5 + 0.45 * sinpi(x) * sinpi(y) * sinpi(z);
        kap[c] = (T)k;
        if (off && !(k >= 0.5 && k < 1.0)) atomicOr(off, 1);
        const bool interior = I >= 1 && I <= g.nx && J >= 1 && J <= g.ny && K >= 1 && K <= g.nz;
        fdt[c] = interior ? (T)(dt * (1.0 + cospi(x) * cospi(y) * cospi(z))) : (T)0;
    }
}

template <typename T>
__device__ __forceinline__ T vk_point(T uc, T uxm, T uxp, T uym, T uyp, T uzm, T uzp, T kc, T kxm, T kxp,
                                      T kym, T kyp, T kzm, T kzp, T f, T bx, T by, T bz)
{
    const T dx = (kxp + kc) * (uxp - uc) - (kc + kxm) * (uc - uxm);
    const T dy = (kyp + kc) * (uyp - uc) - (kc + kym) * (uc - uym);
    const T dz = (kzp + kc) * (uzp - uc) - (kc + kzm) * (uc - uzm);
    return (uc + f) + ((bx * dx + by * dy) + bz * dz);
}

// ---- FP64, exact-sum form --------------------------------------------------
// u' = (u + dt f) + beta D with D = sum over the faces of (kappa + kappa_nb)
// (u_nb - u): the differences of the field's fixed-point integers (SH = 7: units
// of 2^-60 of the field's largest binade) times the face sums in xs_flux, summed
// in 64 bits, L = D 2^(1080 - e) to within 15 units of 4 2^-60 each rounded to a
// double once.  One beta for every axis (a cubic grid) needs nothing more;
// otherwise the axis sums are first scaled by beta_d / beta_max in 62-bit fixed
// point.  The error against the formula in exact arithmetic is below 30 2^-57
// max|u| beta plus a few roundings.  e is tracked per step in the handle's
// FxState like the default FP64 arithmetic's.  Fields whose exponent lies outside
// [kVkEmaxLo, kVkEmaxHi] (all-zero or tiny fields, values near overflow, NaN,
// Inf) take vk_point.
constexpr int kVkEmaxLo = 120, kVkEmaxHi = 2030;

struct VkBeta {
    double bx, by, bz;        // dt / (2 h_d^2)
    double b;                 // the largest
    int wh[3], wl[3];         // beta_d / b times 2^62, as xs_mulhi3 takes it
    long long low;            // what the three products fall short by on average
    int exact;                // every kappa is in [0.5, 1)
};

__device__ __forceinline__ bool vk_exact_ok(int emax, double b)
{
    return emax >= max(kVkEmaxLo, xs_emax_lo(b)) && emax <= kVkEmaxHi;
}

// A block of 32 x 8 threads owns 64 x 8 columns and marches up its planes, every
// thread two consecutive x points.  Each plane of the tile -- u and kappa with a
// one-point halo, dt f without -- arrives by TMA into a ring of kVkNst stages, up
// to kVkNst - 2 planes ahead of use; once plane k+1 lands, the block converts its
// u in place (every thread its own two values, warps 0 and 1 the halo rows, warp
// 2 the halo columns), so each value is converted once and no load waits on
// memory inside the march.  The flux through the face between a thread's two
// points and through the face below a plane are formed once.  One of a thread's
// two points converts its sum on the FP64 pipe.  Every mbarrier wait is bounded,
// as in heat_stream.cu.
//
// Instruction issue (62%), the FP64 pipe (57%) and DRAM (58%) share the time, 174
// instructions per point.  510^3: 856 us per step, 155 GLUP/s = 4.96 TB/s of the
// 32 bytes per update (890 before xs_fix's shorter form, which the figures below
// and 520 x 510 x 500's 1176 us go with).  Before: face sums in three arrays
// (48 bytes), their products summed in 128 bits, every neighbour converted where
// it was used, 265 instructions: 1541 us and 2400 us.  Loads through L1 instead
// of TMA: 1178 us.  Three resident blocks either way, but held to 80 registers
// by the launch bound the compiler's schedule took 946 us; a 3-stage ring 1250,
// 6 stages (two blocks) 1030; both points on the FP64 pipe 906, none 890.
constexpr int kVkTW = 64, kVkBW = 68, kVkD = 2, kVkNst = 4;
constexpr uint32_t kVkBoxBytes = (kVkBY + 2) * kVkBW * 8, kVkSrcBytes = kVkBY * kVkTW * 8;
constexpr int kVkPlane = (int)((kVkBoxBytes + 127) / 128 * 128 / 8);   // words of a staged plane of u or kappa
constexpr int kVkStage = 2 * kVkPlane + (int)(kVkSrcBytes / 8);        // u, kappa, dt f
constexpr size_t kVkSmem = (size_t)kVkNst * (kVkStage * 8 + sizeof(uint64_t));

template <bool CUBIC, bool EXACT>
__device__ __forceinline__ unsigned vk_march(const CUtensorMap* umap, const CUtensorMap* kmap, const CUtensorMap* fmap,
                                             double* __restrict__ dst, const HeatGeom& g, const VkBeta& B, int kb,
                                             int ke, int emax, long long* stage, uint64_t* bars, int& s_abort, int* err)
{
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kVkBX + tx;
    const int x0 = blockIdx.x * kVkTW, y0 = blockIdx.y * kVkBY;
    const int X = x0 + 2 * tx, Y = y0 + ty;
    const bool in = X < g.nx && Y < g.ny, two = X + 1 < g.nx;
    const int own = (ty + 1) * kVkBW + kVkD + 2 * tx;
    const int p_first = kb - 1, p_last = ke;
    // converted besides the thread's own values: a pair of halo row 0 (warp 0) or
    // 9 (warp 1), or one halo-column value (warp 2)
    int extra = -1;
    if (ty == 0) extra = kVkD + 2 * tx;
    else if (ty == 1) extra = (kVkBY + 1) * kVkBW + kVkD + 2 * tx;
    else if (ty == 2 && tx < 2 * kVkBY)
        extra = tx < kVkBY ? (tx + 1) * kVkBW + kVkD - 1 : (tx - kVkBY + 1) * kVkBW + kVkD + kVkTW;
    auto fix = [emax](long long b) -> long long { return EXACT ? xs_fix<7>(b, emax) : b; };
    auto dbl = [](long long v) { return __longlong_as_double(v); };
    const double r2 = EXACT ? xs_r2(B.b, emax) : 0.0;
    auto issue = [&](int p, int slot) {   // plane p into its slot (thread 0)
        long long* st = stage + slot * kVkStage;
        mbar_arrive_expect_tx(&bars[slot], 2 * kVkBoxBytes + kVkSrcBytes);
        tma_load_3d(st, umap, g.lead + x0 - kVkD, y0, p + 1, &bars[slot]);
        tma_load_3d(st + kVkPlane, kmap, g.lead + x0 - kVkD, y0, p + 1, &bars[slot]);
        tma_load_3d(st + 2 * kVkPlane, fmap, g.lead + x0, y0 + 1, p + 1, &bars[slot]);
    };
    // converts this thread's part of a staged plane; its own values before and after
    auto convert = [&](long long* pl, double (&raw)[2], long long (&U)[2]) {
        const longlong2 v = *reinterpret_cast<const longlong2*>(pl + own);
        raw[0] = dbl(v.x);
        raw[1] = dbl(v.y);
        U[0] = fix(v.x);
        U[1] = fix(v.y);
        if constexpr (EXACT) {
            *reinterpret_cast<longlong2*>(pl + own) = make_longlong2(U[0], U[1]);
            if (ty < 2) {
                const longlong2 h = *reinterpret_cast<const longlong2*>(pl + extra);
                *reinterpret_cast<longlong2*>(pl + extra) = make_longlong2(fix(h.x), fix(h.y));
            } else if (extra >= 0) {
                pl[extra] = fix(pl[extra]);
            }
        }
    };

    int issued = p_first - 1, drain_from = p_first;
    if (tid == 0)
        for (int s = 0; s < kVkNst && p_first + s <= p_last; ++s) {
            issue(p_first + s, s);
            issued = p_first + s;
        }
    unsigned mx = 0;
    double uc[2], un[2];
    long long Uc[2], Un[2], kc[2], fb[2] = {0, 0};
    bool ok = mbar_wait_bounded(&bars[0], 0) && mbar_wait_bounded(&bars[1], 0);
    {
        const longlong2 ub = *reinterpret_cast<const longlong2*>(stage + own);
        const longlong2 kl = *reinterpret_cast<const longlong2*>(stage + kVkPlane + own);
        const longlong2 kv = *reinterpret_cast<const longlong2*>(stage + kVkStage + kVkPlane + own);
        kc[0] = kv.x;
        kc[1] = kv.y;
        convert(stage + kVkStage, uc, Uc);
        if constexpr (EXACT) {   // the flux through the face below the first plane
            fb[0] = xs_flux(kl.x, kc[0], Uc[0] - fix(ub.x));
            fb[1] = xs_flux(kl.y, kc[1], Uc[1] - fix(ub.y));
            fence_proxy_async_smem();   // before the barrier after which TMA may refill the slot
        }
    }
    if (!ok) {
        atomicExch(err, 1);
        s_abort = 1;
    }
    __syncthreads();
    int s_cur = 1, n_cur = 0;
    double* out = dst + g.at(in ? X : 0, in ? Y : 0, kb);
    if (!s_abort) {
        for (int k = kb; k < ke; ++k) {
            const int s_nxt = s_cur + 1 == kVkNst ? 0 : s_cur + 1, s_prev = s_cur == 0 ? kVkNst - 1 : s_cur - 1;
            const int n_nxt = s_nxt == 0 ? n_cur + 1 : n_cur;
            if (!mbar_wait_bounded(&bars[s_nxt], (uint32_t)n_nxt & 1u)) {
                atomicExch(err, 1);
                s_abort = 1;
            }
            convert(stage + s_nxt * kVkStage, un, Un);
            const long long* pu = stage + s_cur * kVkStage + own;
            const long long* pk = pu + kVkPlane;
            const longlong2 kav = *reinterpret_cast<const longlong2*>(stage + s_nxt * kVkStage + kVkPlane + own);
            const longlong2 kym = *reinterpret_cast<const longlong2*>(pk - kVkBW);
            const longlong2 kyp = *reinterpret_cast<const longlong2*>(pk + kVkBW);
            const longlong2 uym = *reinterpret_cast<const longlong2*>(pu - kVkBW);
            const longlong2 uyp = *reinterpret_cast<const longlong2*>(pu + kVkBW);
            const double2 f = *reinterpret_cast<const double2*>(stage + s_cur * kVkStage + 2 * kVkPlane + ty * kVkTW +
                                                                2 * tx);
            const long long Ul = pu[-1], Ur = pu[2], kl = pk[-1], kr = pk[2];
            double w[2];
            if constexpr (EXACT) {
                const long long fl = xs_flux(kl, kc[0], Uc[0] - Ul);
                const long long fm = xs_flux(kc[0], kc[1], Uc[1] - Uc[0]);
                const long long fr = xs_flux(kc[1], kr, Ur - Uc[1]);
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const long long fa = xs_flux(kc[q], q ? kav.y : kav.x, Un[q] - Uc[q]);
                    const long long dx = q == 0 ? fm - fl : fr - fm;
                    const long long dy = xs_flux(kc[q], q ? kyp.y : kyp.x, (q ? uyp.y : uyp.x) - Uc[q]) -
                                         xs_flux(kc[q], q ? kym.y : kym.x, Uc[q] - (q ? uym.y : uym.x));
                    const long long dz = fa - fb[q];
                    fb[q] = fa;
                    const long long L = CUBIC ? dx + dy + dz
                                              : B.low + xs_mulhi3(dx << 2, B.wh[0], B.wl[0]) +
                                                    xs_mulhi3(dy << 2, B.wh[1], B.wl[1]) +
                                                    xs_mulhi3(dz << 2, B.wh[2], B.wl[2]);
                    const double uf = __dadd_rn(uc[q], q ? f.y : f.x);
                    w[q] = q == 0 ? xs_apply<true>(uf, L, B.b, r2, emax) : xs_apply<false>(uf, L, B.b, r2, emax);
                }
            } else {
                const long long* pb = stage + s_prev * kVkStage + own;
                const longlong2 ub = *reinterpret_cast<const longlong2*>(pb);
                const longlong2 kbv = *reinterpret_cast<const longlong2*>(pb + kVkPlane);
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    w[q] = vk_point<double>(uc[q], q ? uc[0] : dbl(Ul), q ? dbl(Ur) : uc[1], dbl(q ? uym.y : uym.x),
                                            dbl(q ? uyp.y : uyp.x), dbl(q ? ub.y : ub.x), un[q], dbl(kc[q]),
                                            dbl(q ? kc[0] : kl), dbl(q ? kr : kc[1]), dbl(q ? kym.y : kym.x),
                                            dbl(q ? kyp.y : kyp.x), dbl(q ? kbv.y : kbv.x), dbl(q ? kav.y : kav.x),
                                            q ? f.y : f.x, B.bx, B.by, B.bz);
            }
            if (in) {
                if (two) {
                    *reinterpret_cast<double2*>(out) = make_double2(w[0], w[1]);
                } else {
                    out[0] = w[0];
                    w[1] = 0.0;
                }
                mx = max(mx, max(xs_abs_hi(w[0]), xs_abs_hi(w[1])));
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uc[q] = un[q];
                Uc[q] = Un[q];
            }
            kc[0] = kav.x;
            kc[1] = kav.y;
            out += g.plane;
            if constexpr (EXACT) fence_proxy_async_smem();
            __syncthreads();
            if (s_abort) {
                drain_from = k + 1;
                break;
            }
            if (tid == 0 && issued < p_last) {   // plane k-1's slot is free
                fence_proxy_async_smem();
                issue(issued + 1, s_prev);
                ++issued;
            }
            s_cur = s_nxt;
            n_cur = n_nxt;
        }
    }
    if (s_abort && tid == 0) {
        const long long t0 = clock64();   // one time budget for the whole drain
        for (int p = drain_from; p <= issued; ++p) {
            const int i = p - p_first;
            if (!mbar_wait_until(&bars[i % kVkNst], (uint32_t)(i / kVkNst) & 1u, t0, kWaitCycles)) {
                atomicExch(err, 2);   // loads may still be landing: the context is suspect
                break;
            }
        }
    }
    return mx;
}

template <bool CUBIC>
__global__ void __launch_bounds__(kVkBX* kVkBY, 2)
    k_vk_xs(const __grid_constant__ CUtensorMap umap, const __grid_constant__ CUtensorMap kmap,
            const __grid_constant__ CUtensorMap fmap, double* __restrict__ dst, HeatGeom g, VkBeta B, int kbeg, int kend,
            int kchunk, FxState* fx, int m3, int* err)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    long long* stage = reinterpret_cast<long long*>(smem_raw);
    uint64_t* bars = reinterpret_cast<uint64_t*>(stage + kVkNst * kVkStage);
    __shared__ int s_abort;
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        // a block that starts after another one gave up does no work at all
        s_abort = *(volatile int*)err;
        for (int s = 0; s < kVkNst; ++s) mbar_init(&bars[s], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (s_abort) return;
    const int kb = kbeg + (int)blockIdx.z * kchunk;
    const int ke = min(kb + kchunk, kend);
    const int emax = xs_emax(fx, m3);
    const unsigned mx =
        B.exact && vk_exact_ok(emax, B.b)
            ? vk_march<CUBIC, true>(&umap, &kmap, &fmap, dst, g, B, kb, ke, emax, stage, bars, s_abort, err)
            : vk_march<CUBIC, false>(&umap, &kmap, &fmap, dst, g, B, kb, ke, emax, stage, bars, s_abort, err);
    if (s_abort) return;   // uniform: every thread passed the barrier that saw it
    fx_finish<kVkBX * kVkBY>((unsigned long long)mx << 32, fx, m3, 0,
                             blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0);
}

// The tensor maps of an FP64 handle: its two buffers, kappa, dt f.
int vk_maps(CUtensorMap (&maps)[4], void* const (&buf)[2], void* kap, void* fdt, const HeatGeom& g)
{
    void* const base[4] = {buf[0], buf[1], kap, fdt};
    for (int i = 0; i < 4; ++i) {
        const int e = encode_field_map(&maps[i], base[i], CU_TENSOR_MAP_DATA_TYPE_INT64, sizeof(double),
                                       (uint64_t)g.pitch, (uint64_t)(g.ny + 2), (uint64_t)(g.nz + 2),
                                       i < 3 ? kVkBW : kVkTW, i < 3 ? kVkBY + 2 : kVkBY);
        if (e != 0) return e;
    }
    return 0;
}

// FP32: every thread four consecutive x points (one 16-byte vector
// of u, kappa and dt f per row), so a point costs about 3.5 load instructions
// instead of 11; the update of each point is vk_point's.  A thread whose four
// points run past nx loads element by element up to the boundary node nx (u
// zero there, kappa not) and computes only its interior points.  The kernel
// waits on its loads (long-scoreboard stalls): four blocks per SM at 64
// registers, with 8-plane chunks, ran 340 GLUP/s at 510^3 against 265 with
// three blocks at 80 registers.
__global__ void __launch_bounds__(kVkBX* kVkBY, 4)
    k_vk_f4(const float* __restrict__ src, float* __restrict__ dst, const float* __restrict__ kap,
                     const float* __restrict__ fdt, HeatGeom g, float bx, float by, float bz, int kbeg, int kend,
                     int kchunk)
{
    const int i0 = (blockIdx.x * kVkBX + threadIdx.x) * 4;
    const int j = blockIdx.y * kVkBY + threadIdx.y;
    if (i0 >= g.nx || j >= g.ny) return;
    const int k0 = kbeg + (int)blockIdx.z * kchunk;
    const int k1 = min(k0 + kchunk, kend);
    if (k0 >= k1) return;
    const int64_t P = g.plane, Y = g.pitch;
    const bool full = i0 + 3 < g.nx;
    const int nv = min(4, g.nx - i0);   // interior points of this thread
    auto ld4 = [&](const float* p, float (&o)[4]) {
        if (full) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(p));
            o[0] = v.x;
            o[1] = v.y;
            o[2] = v.z;
            o[3] = v.w;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) o[q] = i0 + q <= g.nx ? __ldg(p + q) : 0.0f;
        }
    };
    int64_t c = g.at(i0, j, k0);
    float ub[4], uc[4], kb[4], kc[4];
    ld4(src + c - P, ub);
    ld4(src + c, uc);
    ld4(kap + c - P, kb);
    ld4(kap + c, kc);
    for (int k = k0; k < k1; ++k) {
        float ua[4], ka[4], uym[4], uyp[4], kym[4], kyp[4], f[4];
        ld4(src + c + P, ua);
        ld4(kap + c + P, ka);
        ld4(src + c - Y, uym);
        ld4(src + c + Y, uyp);
        ld4(kap + c - Y, kym);
        ld4(kap + c + Y, kyp);
        ld4(fdt + c, f);
        const float uL = __ldg(src + c - 1), kL = __ldg(kap + c - 1);
        const float uR = full ? __ldg(src + c + 4) : 0.0f, kR = full ? __ldg(kap + c + 4) : 0.0f;
        float o[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float uxm = q == 0 ? uL : uc[q - 1], uxp = q == 3 ? uR : uc[q + 1];
            const float kxm = q == 0 ? kL : kc[q - 1], kxp = q == 3 ? kR : kc[q + 1];
            o[q] = vk_point<float>(uc[q], uxm, uxp, uym[q], uyp[q], ub[q], ua[q], kc[q], kxm, kxp, kym[q], kyp[q],
                                   kb[q], ka[q], f[q], bx, by, bz);
        }
        if (full) {
            *reinterpret_cast<float4*>(dst + c) = make_float4(o[0], o[1], o[2], o[3]);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (q < nv) dst[c + q] = o[q];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            ub[q] = uc[q];
            uc[q] = ua[q];
            kb[q] = kc[q];
            kc[q] = ka[q];
        }
        c += P;
    }
}

int vk_init(const VkCall& c, double dt)
{
    const int64_t n = (int64_t)(c.g->nx + 2) * (c.g->ny + 2) * (c.g->nz + 2);
    int64_t blocks = (n + 255) / 256;
    if (blocks > (int64_t)kNumSMs * 16) blocks = (int64_t)kNumSMs * 16;
    if (c.f64)
        k_vk_init<double><<<(unsigned)blocks, 256, 0, c.stream>>>((double*)c.kap, (double*)c.fdt, *c.g, dt, c.kappa_off);
    else
        k_vk_init<float><<<(unsigned)blocks, 256, 0, c.stream>>>((float*)c.kap, (float*)c.fdt, *c.g, dt, nullptr);
    HS_CHECK_LAUNCH("heat: kappa/source init kernel");
    return HS_OK;
}

int vk_launch(const VkCall& c)
{
    const HeatGeom& g = *c.g;
    if (c.kend <= c.kbeg) return HS_OK;
    const int planes = c.kend - c.kbeg;
    const int kchunk = std::max(c.kchunk, (planes + 65534) / 65535);   // a launch holds 65535 chunks
    const int nchunks = (planes + kchunk - 1) / kchunk;
    const dim3 block(kVkBX, kVkBY, 1);
    const unsigned by = (g.ny + kVkBY - 1) / kVkBY;
    if (c.f64) {
        VkBeta B;
        B.bx = c.bx;
        B.by = c.by;
        B.bz = c.bz;
        B.b = std::fmax(c.bx, std::fmax(c.by, c.bz));
        const double axis[3] = {c.bx, c.by, c.bz};
        // xs_mulhi3 rounds two partial products down and leaves out the third, in the
        // mean one unit and wl / 2^33; with the largest beta's 2^62 it is exact here.
        // Fluxes round down alike and their bias cancels in a face's difference, this
        // one would add up from step to step.
        double low = 0.0;
        for (int d = 0; d < 3; ++d) {
            const long long w = B.b > 0.0 ? std::llrint(std::ldexp(axis[d] / B.b, 62)) : 0ll;
            B.wl[d] = (int)(unsigned)w;
            B.wh[d] = (int)((w - B.wl[d]) >> 32);
            if (w != 0 && w != 1ll << 62) low += 1.0 + std::ldexp((double)B.wl[d], -33);
        }
        B.low = std::llrint(low);
        B.exact = c.exact;
        const bool cubic = c.bx == c.by && c.by == c.bz;
        auto kern = cubic ? k_vk_xs<true> : k_vk_xs<false>;
        // once per process, under the thread-safe initialisation of a local static
        static const cudaError_t configured = [] {
            const cudaError_t e = cudaFuncSetAttribute(k_vk_xs<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kVkSmem);
            return e != cudaSuccess ? e
                                    : cudaFuncSetAttribute(k_vk_xs<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                           (int)kVkSmem);
        }();
        HS_TRY_CUDA(configured, "heat: variable-kappa kernel smem attribute");
        const dim3 grid((g.nx + kVkTW - 1) / kVkTW, by, nchunks);
        kern<<<grid, block, kVkSmem, c.stream>>>(*c.umap, *c.kmap, *c.fmap, (double*)c.dst, g, B, c.kbeg, c.kend, kchunk,
                                                 c.fx, c.m3, c.err);
    } else {
        const dim3 grid((g.nx + 4 * kVkBX - 1) / (4 * kVkBX), by, nchunks);
        k_vk_f4<<<grid, block, 0, c.stream>>>((const float*)c.src, (float*)c.dst, (const float*)c.kap,
                                                       (const float*)c.fdt, g, (float)c.bx, (float)c.by, (float)c.bz,
                                                       c.kbeg, c.kend, kchunk);
    }
    HS_CHECK_LAUNCH("heat variable-kappa kernel");
    return HS_OK;
}

}  // namespace hcg
