// Batched CG: many independent systems A_s x_s = b_s (7-point Laplacians of
// different grids, matrix-free or CSR) solved together.  Stencil systems of 2^14
// to 2^22 unknowns go through one launch for whole solves (cg_small.cu), the
// others through an update, a direction and up to three SpMV launches (one per
// kind present) per iteration for all of them.
//
// Each of those others gets the same number of blocks and the same grid-stride row
// partition as its own cg_run would use, its own reduction partials, ticket
// and device scalars, so its iterates -- and results -- equal a solve of it
// alone bit for bit.  Systems that have converged (or hit max_iter) stop at
// the top of each kernel; the host reads all stop flags once per chunk of
// iterations.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "cg_small.cuh"

namespace hcg {

struct SysDev {
    OpDev A;
    const double* b;
    double* x;
    double* r;
    double* p;
    double* q;
    double* partials;   // 2 * nblocks
    CgScalars* S;
    int32_t block0;     // first block of this system in the batch grid
    int32_t nblocks;
    int32_t max_iter;
    int32_t mode;       // SpmvMode of the operator with this block count
    int32_t nshares;    // SP_STAGED: shares of the SpMV (spmv_shares(nblocks)), else nblocks
};

// System of this block (binary search over block0) and the block's index in it.
__device__ __forceinline__ int sys_of_block(const SysDev* sys, int nsys, int* local)
{
    int lo = 0, hi = nsys - 1;
    const int b = (int)blockIdx.x;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (sys[mid].block0 <= b) lo = mid; else hi = mid - 1;
    }
    *local = b - sys[lo].block0;
    return lo;
}

// arrive_last for a block range: partial at [local], ticket of the system.
__device__ __forceinline__ bool arrive_last_sys(double total, double* partials, uint32_t* ticket,
                                                int local, int nblocks)
{
    __shared__ bool last;
    if (threadIdx.x == 0) {
        partials[local] = total;
        __threadfence();
        const uint32_t t = atomicAdd(ticket, 1u);
        last = (t == (uint32_t)nblocks - 1);
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

__device__ __forceinline__ double sum_partials_n(const double* partials, int m, double* sh)
{
    double v = 0.0;
    for (int t = threadIdx.x; t < m; t += kCgBlock) v += __ldcg(partials + t);
    return block_sum<kCgBlock>(v, sh);
}

__device__ __forceinline__ double apply_sys(const OpDev& A, const double* __restrict__ p, int64_t row)
{
    return A.kind == HS_OP_STENCIL7 ? apply_stencil_row(A, p, row) : apply_csr_row(A, p, row);
}

// q = A x0 (start), then r = b - q, p = r, rho, ||b||.
__global__ void __launch_bounds__(kCgBlock) k_cgb_apply_x(const SysDev* sys, int nsys)
{
    int local;
    const SysDev& s = sys[sys_of_block(sys, nsys, &local)];
    for (int64_t row = (int64_t)local * kCgBlock + threadIdx.x; row < s.A.n;
         row += (int64_t)s.nblocks * kCgBlock)
        s.q[row] = apply_sys(s.A, s.x, row);
}

__global__ void __launch_bounds__(kCgBlock) k_cgb_start(const SysDev* sys, int nsys)
{
    int local;
    const SysDev& s = sys[sys_of_block(sys, nsys, &local)];
    __shared__ double sh[kCgBlock / 32];
    double rr = 0.0, bb = 0.0;
    unsigned pm = 0;
    for (int64_t t = (int64_t)local * kCgBlock + threadIdx.x; t < s.A.n;
         t += (int64_t)s.nblocks * kCgBlock) {
        const double bt = s.b[t];
        const double rt = bt - s.q[t];
        s.r[t] = rt;
        s.p[t] = rt;
        rr = __fma_rn(rt, rt, rr);
        bb = __fma_rn(bt, bt, bb);
        pm = max(pm, xs_abs_hi(rt));
    }
    const double rr_blk = block_sum<kCgBlock>(rr, sh);
    const double bb_blk = block_sum<kCgBlock>(bb, sh);
    if (s.mode == SP_STAGED) cg_fold_pmax(pm, s.S, 0, local == 0);
    if (threadIdx.x == 0) s.partials[s.nblocks + local] = bb_blk;
    if (!arrive_last_sys(rr_blk, s.partials, &s.S->ticket, local, s.nblocks)) return;
    const double rho = sum_partials_n(s.partials, s.nblocks, sh);
    const double bnorm2 = sum_partials_n(s.partials + s.nblocks, s.nblocks, sh);
    if (threadIdx.x == 0) {
        CgScalars* S = s.S;
        S->ticket = 0;
        S->rho = rho;
        S->bnorm = sqrt(bnorm2);
        S->iters = 0;
        S->zero_rhs = (bnorm2 == 0.0);
        if (bnorm2 == 0.0) {
            S->relres = 0.0;
            S->done = 1;
        } else {
            S->relres = sqrt(rho) / S->bnorm;
            S->done = (S->relres <= S->rtol) ? 1 : 0;
        }
    }
}

// One kernel per SpmvMode, so each has its own register budget (and, for the
// staged mode, block size); blocks of the other modes' systems return at once.
template <int MODE, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_cgb_spmv_dot(const SysDev* sys, int nsys)
{
    grid_dependency_wait();
    int local;
    const SysDev& s = sys[sys_of_block(sys, nsys, &local)];
    if (s.mode != MODE || *(volatile int32_t*)&s.S->done || s.S->iters >= s.max_iter) return;
    __shared__ double sh[NT / 32];
    double pq = 0.0;
    // as k_cg_spmv_dot / k_cg_spmv_staged: the same points per thread and the
    // same arithmetic, so the same results
    const int64_t row0 = (int64_t)local * NT + threadIdx.x;
    const int64_t stride = (int64_t)s.nblocks * NT;
    if (MODE == SP_STAGED) {
        // share `local` of a single solve's launch; the blocks beyond the shares add 0
        if (local < s.nshares) pq = spmv_stencil_share(s.A, s.p, s.q, cg_pemax(s.S), local, s.nshares);
    } else for (int64_t row = row0; row < s.A.n; row += stride) {
        const double qv = MODE == SP_CSR ? apply_csr_row(s.A, s.p, row) : apply_stencil_row(s.A, s.p, row);
        s.q[row] = qv;
        pq = __fma_rn(__ldg(s.p + row), qv, pq);
    }
    allow_dependents();
    const double blk = block_sum<NT>(pq, sh);
    if (!arrive_last_sys(blk, s.partials, &s.S->ticket, local, s.nblocks)) return;
    const double tot = sum_partials_nt<NT>(s.partials, s.nshares, sh);
    if (threadIdx.x == 0) {
        CgScalars* S = s.S;
        S->ticket = 0;
        S->pq = tot;
        if (!(tot > 0.0))
            S->done = 2;
        else
            S->alpha = S->rho / tot;
    }
}

// WITH_X: x += alpha p too, as k_cg_update; batches with a large system leave that to
// k_cgb_direction (80 bytes per row and iteration instead of 88: one of 200^3
// 123.7 -> 107.5 ms, 16 CSR systems of 64^3 116 -> 128).
template <bool WITH_X>
__global__ void __launch_bounds__(kCgBlock) k_cgb_update(const SysDev* sys, int nsys)
{
    grid_dependency_wait();
    int local;
    const SysDev& s = sys[sys_of_block(sys, nsys, &local)];
    if (*(volatile int32_t*)&s.S->done || s.S->iters >= s.max_iter) return;
    __shared__ double sh[kCgBlock / 32];
    const double alpha = s.S->alpha;
    const int64_t t0 = (int64_t)local * kCgBlock + threadIdx.x, stride = (int64_t)s.nblocks * kCgBlock;
    const double rr = WITH_X ? cg_update_xr_rows(s.A.n, s.x, s.r, s.p, s.q, alpha, t0, stride)
                             : cg_update_rows(s.A.n, s.r, s.q, alpha, t0, stride);
    allow_dependents();
    const double blk = block_sum<kCgBlock>(rr, sh);
    if (!arrive_last_sys(blk, s.partials, &s.S->ticket, local, s.nblocks)) return;
    const double rho_new = sum_partials_n(s.partials, s.nblocks, sh);
    if (threadIdx.x == 0) {
        CgScalars* S = s.S;
        S->ticket = 0;
        S->iters += 1;
        S->relres = sqrt(rho_new) / S->bnorm;
        if (S->relres <= S->rtol)
            S->done = 1;
        else
            S->beta = rho_new / S->rho;
        S->rho = rho_new;
    }
}

// x += alpha p and, unless the system has stopped, p = r + beta p, for the
// systems that took iteration `it`.
__global__ void __launch_bounds__(kCgBlock) k_cgb_direction(const SysDev* sys, int nsys, int it)
{
    grid_dependency_wait();
    int local;
    const SysDev& s = sys[sys_of_block(sys, nsys, &local)];
    // the update kernel of this iteration has already counted it
    if (*(volatile int32_t*)&s.S->iters != it + 1) return;
    const bool next = *(volatile int32_t*)&s.S->done == 0;
    const unsigned pm = cg_direction_rows<X_ONE>(s.A.n, s.r, s.p, nullptr, s.p, s.x, s.S->alpha, 0.0, s.S->beta, next,
                                                 (int64_t)local * kCgBlock + threadIdx.x, (int64_t)s.nblocks * kCgBlock);
    allow_dependents();
    if (s.mode == SP_STAGED && next) cg_fold_pmax(pm, s.S, (it + 1) % 3, local == 0);
}

// p = r + beta p.
__global__ void __launch_bounds__(kCgBlock) k_cgb_pupdate(const SysDev* sys, int nsys)
{
    grid_dependency_wait();
    int local;
    const SysDev& s = sys[sys_of_block(sys, nsys, &local)];
    // the update kernel of this iteration has already counted it
    if (*(volatile int32_t*)&s.S->done) return;
    const double beta = s.S->beta;
    const unsigned pm = cg_pupdate_rows(s.A.n, s.r, s.p, beta, (int64_t)local * kCgBlock + threadIdx.x,
                                        (int64_t)s.nblocks * kCgBlock);
    allow_dependents();
    if (s.mode == SP_STAGED) cg_fold_pmax(pm, s.S, s.S->iters % 3, local == 0);
}

// ||b - A x||^2 into rr_true (q = A x from k_cgb_apply_x).
__global__ void __launch_bounds__(kCgBlock) k_cgb_resid(const SysDev* sys, int nsys)
{
    int local;
    const SysDev& s = sys[sys_of_block(sys, nsys, &local)];
    __shared__ double sh[kCgBlock / 32];
    double rr = 0.0;
    for (int64_t t = (int64_t)local * kCgBlock + threadIdx.x; t < s.A.n;
         t += (int64_t)s.nblocks * kCgBlock) {
        const double d = s.b[t] - s.q[t];
        rr = __fma_rn(d, d, rr);
    }
    const double blk = block_sum<kCgBlock>(rr, sh);
    if (!arrive_last_sys(blk, s.partials, &s.S->ticket, local, s.nblocks)) return;
    const double tot = sum_partials_n(s.partials, s.nblocks, sh);
    if (threadIdx.x == 0) {
        s.S->ticket = 0;
        s.S->rr_true = tot;
    }
}

}  // namespace hcg

using namespace hcg;

// Control words of the small systems' launch, uploaded whole before a run.
struct SmallCtl {
    unsigned long long bar[6 * kGridBarStride];
    int32_t err;
    int32_t pad[31];
};

struct hs_cg_batch {
    cudaStream_t stream;
    int32_t n;
    // systems that run three kernels per iteration
    std::vector<int32_t> big;  // their places in the batch
    int32_t total_blocks;
    bool has_mode[3];          // SpmvModes present (one SpMV kernel each)
    bool x_late;               // x is updated with p, not with r: some system is large (cg_x_late)
    std::vector<SysDev> sys;   // host copy (b, x filled per run)
    SysDev* d_sys;
    // small matrix-free systems, solved whole in one launch (cg_small.cu)
    std::vector<int32_t> small;         // their places in the batch, group after group
    std::vector<CgSmallSys> ssys;       // host copy (b, x filled per run)
    std::vector<CgSmallGroup> groups;
    SmallCtl ctl;                       // host copy of the control words
    int64_t sbricks;                    // bricks of the largest group
    CgSmallSys* d_ssys;
    CgSmallGroup* d_groups;
    SmallCtl* d_ctl;
    int32_t h_err;
    std::vector<int64_t> rows, len;   // unknowns of each system, values of its r, p and q
    void* arena;               // r, p, q, partials, scalars and tables of all systems
    CgScalars* d_S;
    CgScalars* h_S;            // host mirror of the scalars, n entries
};

extern "C" {

int cg_batch_destroy(hs_cg_batch_t b)
{
    if (!b) return HS_OK;
    int rc = HS_OK;
    cudaError_t e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) rc = cuda_fail(e, "cg_batch_destroy: synchronize");
    dev_free(b->arena, b->stream);
    delete[] b->h_S;
    delete b;
    return rc;
}

// Lays out a new batch and allocates its device memory.
static int cg_batch_fill(hs_cg_batch* b, const hs_op* ops, int32_t n)
{
    b->rows.resize((size_t)n);
    int64_t vec_total = 0, part_total = 0;
    int64_t blocks = 0;
    for (int32_t i = 0; i < n; ++i) {
        const OpDev A = to_dev(&ops[i]);
        b->rows[(size_t)i] = A.n;
        b->len.push_back((cg_vector_len(A) + 1) & ~(int64_t)1);   // every vector starts 16-byte aligned
        vec_total += b->len.back();
        CgSmallSys ss;
        memset(&ss, 0, sizeof(ss));
        if (cg_small_shape(A, &ss)) {
            b->small.push_back(i);
            part_total += 2 * (int64_t)ss.bricks;
            continue;
        }
        SysDev s;
        memset(&s, 0, sizeof(s));
        s.A = A;
        s.nblocks = grid_for(s.A.n);
        s.mode = spmv_mode(s.A, s.nblocks);
        s.nshares = s.mode == SP_STAGED ? spmv_shares(s.nblocks) : s.nblocks;
        b->has_mode[s.mode] = true;
        if (cg_x_late(s.A)) b->x_late = true;
        s.block0 = (int32_t)blocks;
        blocks += s.nblocks;
        part_total += 2 * (int64_t)s.nblocks;
        b->big.push_back(i);
        b->sys.push_back(s);
    }
    if (blocks > INT32_MAX) {
        return fail(HS_EINVAL, "cg_batch_create: batch too large");
    }
    b->total_blocks = (int32_t)blocks;
    // Small systems that advance in step share a group, at most kCgSmallSystems
    // (groups of fewer unknowns, whose vectors would stay in L2, measured slower:
    // 64 systems of 22.9 M unknowns 149 ms in one group, 165 in groups of 6 M, 179
    // of 3 M -- the phases' fixed costs weigh more), those with about equally many
    // iterations ahead together: the count grows with 1 / sum_d 1/n_d^2.
    auto difficulty = [&](int32_t i) {
        const double x = ops[i].nx, y = ops[i].ny, z = ops[i].nz;
        return 1.0 / (1.0 / (x * x) + 1.0 / (y * y) + 1.0 / (z * z));
    };
    std::stable_sort(b->small.begin(), b->small.end(),
                     [&](int32_t p, int32_t q) { return difficulty(p) > difficulty(q); });
    int64_t bricks = 0;
    for (size_t k = 0; k < b->small.size(); ++k) {
        if (k % kCgSmallSystems == 0) {
            b->groups.push_back(CgSmallGroup{(int32_t)k, 0});
            bricks = 0;
        }
        CgSmallSys ss;
        memset(&ss, 0, sizeof(ss));
        (void)cg_small_shape(to_dev(&ops[b->small[k]]), &ss);
        b->ssys.push_back(ss);
        b->groups.back().count += 1;
        bricks += ss.bricks;
        b->sbricks = std::max(b->sbricks, bricks);
    }
    auto align = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t s_vec = align(sizeof(double) * 3 * (size_t)vec_total), s_part = align(sizeof(double) * (size_t)part_total);
    const size_t s_S = align(sizeof(CgScalars) * (size_t)n), s_sys = align(sizeof(SysDev) * b->sys.size());
    const size_t s_ssys = align(sizeof(CgSmallSys) * b->ssys.size());
    const size_t s_groups = align(sizeof(CgSmallGroup) * b->groups.size());
    const size_t bytes = s_vec + s_part + s_S + s_sys + s_ssys + s_groups + sizeof(SmallCtl);
    cudaError_t e = dev_alloc(&b->arena, bytes, b->stream);
    if (e != cudaSuccess) b->arena = nullptr;
    if (e == cudaSuccess) {
        b->h_S = new (std::nothrow) CgScalars[(size_t)n]();
        if (!b->h_S) e = cudaErrorMemoryAllocation;
    }
    if (e != cudaSuccess) return cuda_fail(e, "cg_batch_create: allocation");
    char* base = (char*)b->arena;
    double* vec = (double*)base;
    double* part = (double*)(base + s_vec);
    b->d_S = (CgScalars*)(base + s_vec + s_part);
    b->d_sys = (SysDev*)(base + s_vec + s_part + s_S);
    b->d_ssys = (CgSmallSys*)(base + s_vec + s_part + s_S + s_sys);
    b->d_groups = (CgSmallGroup*)(base + s_vec + s_part + s_S + s_sys + s_ssys);
    b->d_ctl = (SmallCtl*)(base + s_vec + s_part + s_S + s_sys + s_ssys + s_groups);
    auto take = [&](auto& s, int32_t i, int64_t partials) {
        const int64_t len = b->len[(size_t)i];
        s.r = vec;
        s.p = vec + len;
        s.q = vec + 2 * len;
        vec += 3 * len;
        s.S = b->d_S + i;
        double* const p0 = part;
        part += partials;
        return p0;
    };
    for (size_t k = 0; k < b->sys.size(); ++k)
        b->sys[k].partials = take(b->sys[k], b->big[k], 2 * (int64_t)b->sys[k].nblocks);
    for (size_t k = 0; k < b->ssys.size(); ++k)
        b->ssys[k].part = take(b->ssys[k], b->small[k], 2 * (int64_t)b->ssys[k].bricks);
    return HS_OK;
}

int cg_batch_create(hs_cg_batch_t* out, const hs_op* ops, int32_t n, void* stream)
{
    if (!out) return fail(HS_EINVAL, "cg_batch_create: out is NULL");
    *out = nullptr;
    if (!ops || n < 1) return fail(HS_EINVAL, "cg_batch_create: no systems");
    for (int32_t i = 0; i < n; ++i) {
        const int rc = check_op(&ops[i]);
        if (rc != HS_OK) return rc;
        if (ops[i].host) return fail(HS_EINVAL, "cg_batch_create: operator %d must be device memory", i);
    }
    hs_cg_batch* b = new (std::nothrow) hs_cg_batch();
    if (!b) return fail(HS_ENOMEM, "cg_batch_create: host allocation failed");
    b->stream = (cudaStream_t)stream;
    b->n = n;
    int rc = HS_OK;
    try {
        rc = cg_batch_fill(b, ops, n);
    } catch (const std::bad_alloc&) {
        rc = fail(HS_ENOMEM, "cg_batch_create: host allocation failed");
    }
    if (rc != HS_OK) {
        cg_batch_destroy(b);
        return rc;
    }
    *out = b;
    return HS_OK;
}

int cg_batch_run(hs_cg_batch_t b, const void* const* bs, void* const* xs, double rtol, int32_t max_iter,
                 hs_cg_info* infos)
{
    if (!b || !bs || !xs) return fail(HS_EINVAL, "cg_batch_run: NULL argument");
    if (!(rtol >= 0.0) || !std::isfinite(rtol)) return fail(HS_EINVAL, "cg_batch_run: bad rtol");
    if (max_iter < 0) return fail(HS_EINVAL, "cg_batch_run: max_iter < 0");
    const int n = b->n;
    for (int i = 0; i < n; ++i)
        if (!bs[i] || !xs[i]) return fail(HS_EINVAL, "cg_batch_run: NULL vector of system %d", i);
    for (size_t k = 0; k < b->sys.size(); ++k) {
        b->sys[k].b = (const double*)bs[b->big[k]];
        b->sys[k].x = (double*)xs[b->big[k]];
        b->sys[k].max_iter = max_iter;
    }
    for (size_t k = 0; k < b->ssys.size(); ++k) {
        b->ssys[k].b = (const double*)bs[b->small[k]];
        b->ssys[k].x = (double*)xs[b->small[k]];
        b->ssys[k].max_iter = max_iter;
    }
    if (!b->sys.empty())
        HS_TRY_CUDA(cudaMemcpyAsync(b->d_sys, b->sys.data(), sizeof(SysDev) * b->sys.size(), cudaMemcpyHostToDevice,
                                    b->stream),
                    "cg_batch_run: system table");
    if (!b->ssys.empty()) {
        HS_TRY_CUDA(cudaMemcpyAsync(b->d_ssys, b->ssys.data(), sizeof(CgSmallSys) * b->ssys.size(),
                                    cudaMemcpyHostToDevice, b->stream),
                    "cg_batch_run: system table");
        HS_TRY_CUDA(cudaMemcpyAsync(b->d_groups, b->groups.data(), sizeof(CgSmallGroup) * b->groups.size(),
                                    cudaMemcpyHostToDevice, b->stream),
                    "cg_batch_run: group table");
        HS_TRY_CUDA(cudaMemcpyAsync(b->d_ctl, &b->ctl, sizeof(SmallCtl), cudaMemcpyHostToDevice, b->stream),
                    "cg_batch_run: control words");
    }
    for (int i = 0; i < n; ++i) {
        memset(&b->h_S[i], 0, sizeof(CgScalars));
        b->h_S[i].rtol = rtol;
    }
    HS_TRY_CUDA(cudaMemcpyAsync(b->d_S, b->h_S, sizeof(CgScalars) * (size_t)n, cudaMemcpyHostToDevice,
                                b->stream),
                "cg_batch_run: scalars");
    const int G = b->total_blocks;
#define CGB_LAUNCH(kern, what)                                                 \
    do {                                                                       \
        kern<<<G, kCgBlock, 0, b->stream>>>(b->d_sys, nbig);                      \
        HS_CHECK_LAUNCH(what);                                                 \
    } while (0)
    // the iteration kernels launch as dependent launches: each waits on entry
    // for the kernel before it, and its launch overlaps that kernel's tail
#define CGB_LAUNCH_DEP(kern, what)                                                             \
    do {                                                                                       \
        HS_TRY_CUDA(launch_dependent(kern, G, kCgBlock, b->stream, b->d_sys, nbig), "cg batch: kernel launch"); \
        HS_CHECK_LAUNCH(what);                                                                 \
    } while (0)
    if (!b->ssys.empty()) {
        const int rc_ = cg_small_launch(b->d_ssys, b->d_groups, (int)b->groups.size(), b->ssys.size() == 1, b->sbricks,
                                        b->d_ctl->bar, &b->d_ctl->err, b->stream);
        if (rc_ != HS_OK) return rc_;
    }
    const int nbig = (int)b->sys.size();
    if (nbig) {
        CGB_LAUNCH(k_cgb_apply_x, "cg batch: A x0 kernel");
        CGB_LAUNCH(k_cgb_start, "cg batch: start kernel");
    }
    int32_t enqueued = 0;
    int chunk = 4;
    for (;;) {
        HS_TRY_CUDA(cudaMemcpyAsync(b->h_S, b->d_S, sizeof(CgScalars) * (size_t)n, cudaMemcpyDeviceToHost,
                                    b->stream),
                    "cg_batch_run: scalar readback");
        HS_TRY_CUDA(cudaStreamSynchronize(b->stream), "cg_batch_run: synchronize");
        bool all = true;
        for (int32_t i : b->big)
            if (!b->h_S[i].done && b->h_S[i].iters < max_iter) all = false;
        if (all || enqueued >= max_iter) break;
        const int32_t todo = (max_iter - enqueued < chunk) ? max_iter - enqueued : chunk;
        for (int32_t t = 0; t < todo; ++t) {
            if (b->has_mode[SP_STAGED]) {
                HS_TRY_CUDA(launch_dependent(k_cgb_spmv_dot<SP_STAGED, kSpBlock, kSpMinBlocks>, G, kSpBlock, b->stream, b->d_sys,
                                             nbig),
                            "cg batch: kernel launch");
                HS_CHECK_LAUNCH("cg batch: spmv+dot kernel");
            }
            if (b->has_mode[SP_ROWS]) CGB_LAUNCH_DEP((k_cgb_spmv_dot<SP_ROWS, kCgBlock, 1>), "cg batch: spmv+dot kernel");
            if (b->has_mode[SP_CSR]) CGB_LAUNCH_DEP((k_cgb_spmv_dot<SP_CSR, kCgBlock, 1>), "cg batch: spmv+dot kernel");
            if (b->x_late) {
                CGB_LAUNCH_DEP(k_cgb_update<false>, "cg batch: update kernel");
                HS_TRY_CUDA(launch_dependent(k_cgb_direction, G, kCgBlock, b->stream, b->d_sys, nbig, enqueued + t),
                            "cg batch: kernel launch");
                HS_CHECK_LAUNCH("cg batch: direction kernel");
            } else {
                CGB_LAUNCH_DEP(k_cgb_update<true>, "cg batch: update kernel");
                CGB_LAUNCH_DEP(k_cgb_pupdate, "cg batch: p update kernel");
            }
        }
        enqueued += todo;
        if (chunk < 32) chunk *= 2;
    }
    // zero right-hand sides have the solution 0
    for (int32_t i : b->big)
        if (b->h_S[i].zero_rhs)
            HS_TRY_CUDA(cudaMemsetAsync(xs[i], 0, sizeof(double) * (size_t)b->rows[(size_t)i], b->stream),
                        "cg_batch_run: zero solution");
    if (nbig) {
        CGB_LAUNCH(k_cgb_apply_x, "cg batch: A x kernel");
        CGB_LAUNCH(k_cgb_resid, "cg batch: residual kernel");
    }
#undef CGB_LAUNCH
#undef CGB_LAUNCH_DEP
    HS_TRY_CUDA(cudaMemcpyAsync(b->h_S, b->d_S, sizeof(CgScalars) * (size_t)n, cudaMemcpyDeviceToHost,
                                b->stream),
                "cg_batch_run: scalar readback");
    b->h_err = 0;
    if (!b->ssys.empty())
        HS_TRY_CUDA(cudaMemcpyAsync(&b->h_err, &b->d_ctl->err, sizeof(int32_t), cudaMemcpyDeviceToHost, b->stream),
                    "cg_batch_run: control words");
    HS_TRY_CUDA(cudaStreamSynchronize(b->stream), "cg_batch_run: synchronize");
    if (b->h_err) return fail(HS_ETIMEOUT, "cg_batch_run: a bounded wait in the small-system kernel ran out");
    int rc = HS_OK;
    for (int i = 0; i < n; ++i) {
        const CgScalars& f = b->h_S[i];
        if (f.done == 2) return fail(HS_ECUDA, "cg_batch_run: breakdown in system %d", i);
        const bool conv = (f.done == 1);
        if (!conv) rc = HS_ENOCONV;
        if (infos) {
            infos[i].iters = f.iters;
            infos[i].status = conv ? HS_OK : HS_ENOCONV;
            infos[i].relres_recur = f.relres;
            infos[i].relres_true = f.zero_rhs ? 0.0 : sqrt(f.rr_true) / f.bnorm;
            infos[i].refinements = 0;
            infos[i].reserved = 0;
        }
    }
    if (rc == HS_ENOCONV) set_error("cg_batch_run: some systems did not reach rtol %g in %d iterations", rtol,
                                    max_iter);
    return rc;
}

}  // extern "C"
