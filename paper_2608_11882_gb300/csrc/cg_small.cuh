// Whole solves of small matrix-free systems in one launch (cg_small.cu).
#pragma once
#include "cg_common.cuh"
#include "gridbar.cuh"

namespace hcg {

constexpr int kCgSmallKZ = 4;
constexpr int kCgSmallSystems = 64;      // systems of one launch
constexpr int kCgSmallMaxBricks = 4096;  // bricks of one system
// Sizes that take this path.  Upper end: per iteration 44.9 us against 73.2 for
// three launches at 128^3, 84.6 against 86.4 at 160^3.  Lower end: smaller solves
// keep the three launches per iteration that hs_launch_count reports for them
// (the kernel would take about 12 us per iteration there too, against 16).
constexpr int64_t kCgSmallMinN = (int64_t)1 << 14, kCgSmallMaxN = (int64_t)1 << 22;
constexpr int kCgSmallMinNx = 16;        // also bounds what the padding of odd rows adds
struct CgSmallSys {
    int32_t nx, ny, nz;
    int32_t lg;                  // log2 of the threads per brick row: 5 (64 x 8 x 4) or 4 (32 x 16 x 4)
    int32_t tiles_x, tiles_y, bricks;
    int32_t max_iter;
    int32_t pitch;               // row length of r, p and q: nx made even, the pad zero
    int32_t pad_;
    const double* b;
    double* x;
    double* r;                   // r, p, q: 16-byte aligned
    double* p;
    double* q;
    double* part;                // 2 * bricks
    CgScalars* S;
};

// Systems [first, first + count) of a launch, solved in step with one another.
struct CgSmallGroup {
    int32_t first, count;   // count <= kCgSmallSystems
};

// Control block of a single solve.  Uploaded whole before the launch; the error
// word and what follows it are read back after.
struct CgSmallCtl {
    unsigned long long bar[6 * kGridBarStride];   // the grid barrier's words, zero before a launch
    CgSmallGroup group;
    int32_t err;
    int32_t pad[29];
    CgSmallSys sys;
    CgScalars S;
};

// Fills the geometry of a system that takes this path; false for any other.
bool cg_small_shape(const OpDev& A, CgSmallSys* s);
// Values each of r, p and q holds: rows of even pitch on this path, else n, made even.
inline int64_t cg_vector_len(const OpDev& A)
{
    CgSmallSys s;
    return cg_small_shape(A, &s) ? (int64_t)s.pitch * A.ny * A.nz : (A.n + 1) & ~(int64_t)1;
}
// One launch over ngroups groups, one after the other.  single: one system in
// all; bricks: of the largest group.  *err is set to 1 when a bounded wait ran out.
int cg_small_launch(const CgSmallSys* sys, const CgSmallGroup* groups, int ngroups, bool single, int64_t bricks,
                    unsigned long long* bar, int* err, cudaStream_t stream);

}  // namespace hcg
