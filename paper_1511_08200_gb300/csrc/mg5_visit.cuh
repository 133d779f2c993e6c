// mg5_visit.cuh -- arguments of the coarse-grid visit in one cluster (k_visit.cu).
#pragma once
#include "mg5_kernels.cuh"

namespace mg5 {

constexpr int kVisitCtas = 16;
constexpr int kVisitLevels = 6;
// Cells of the largest grid taken.  A half-sweep of 32^3 costs 16 SMs 4.9 us (450 instructions a cell)
// where a launch over all SMs takes 3.1 us (patch 5.2): a 64^3 refinement took 1497 us with the 32^3
// grid in the cluster and 1423 without; 24 x 20 x 36 (2.2 us a half-sweep) gained 5% in it.  The planes are
// dealt along the first axis only, so a slab that is thin there uses few CTAs, one at 8 planes and
// fewer.  That is slower than the same slab on its side, and still faster than launches (a relaxation
// to 1e-10, launches -> cluster): 16 x 48 x 40 2181 -> 1511 us, 48 x 40 x 16 2188 -> 1085, 16 x 48 x 48
// 2670 -> 1411, 20 x 72 x 72 7122 -> 2554, 16 x 96 x 16 1666 -> 1330, 16 x 20 x 24 1126 -> 897.
constexpr int kVisitCells = 20000;
constexpr int kVisitCoarsest = 2048;          // cells of a coarsest grid CTA 0 iterates
constexpr int kVisitSmem = 222 * 1024;        // dynamic shared memory a CTA may use
constexpr int kVisitHeadroom = 2;             // bits: rounding, and a nonlinear correction above the linear one

struct VisitLevel {
    int id, n0, n1, n2;    // interior sides
    int P, act, single;    // planes per CTA, CTAs that own planes, held by CTA 0 alone
    int wq, sz;            // cells of a row of one colour, of an array
    int pieces, F;         // offsets in shared memory (16 bytes)
    int ring;              // ghosts around a plane (box)
    unsigned mq, m1, m2, mring;   // reciprocals of (n2 + 1) / 2, n1, n2, ring
    int nmax2;             // 2 floor(log2 of the largest side)
    int Hq;                // h^2 = H 2^Hq
    float Hh, Hl;
    float wh, wl;          // omega / 6
    float inv_h, inv_l;    // 1 / cells
    float w[3][2];         // ghost weights w, w^2, w^3 (box)
    double h2, k;          // k = (2 alpha / 3) / h^2
    double *v, *v0;
    const double *f;       // the top grid's restricted residual
    float2 *x;             // scratch: residuals on the way down, corrections on the way up
};

struct VisitArgs {
    int nlev, nu1, nu2, nu_coarse, smem;
    int headroom;          // bits above the largest value that the first attempt's unit leaves
    double rtol;
    const double *m_up;    // mean residual of the grid above (periodic)
    double *c_out;         // c of the top grid (periodic)
    unsigned long long *clamp;
    int *sweeps;
    VisitLevel lev[kVisitLevels];
};

// Fills sides, distribution and shared-memory layout; false: the grids do not fit.  (Whether the device
// takes the cluster at all is the context's to know: prepare_visit_kernels.)
bool visit_plan(const int (*q)[3], int nlev, bool box, VisitArgs *A);
// ... and a level's constants (w: extrapolation weight of a box's ghosts).
void visit_level_consts(VisitLevel *L, const CoefT<double> &cf, double w);
// Sets the kernels' attributes on the current device; *fits: it can hold a cluster of kVisitCtas CTAs.
cudaError_t prepare_visit_kernels(bool *fits);
cudaError_t launch_visit(const VisitArgs &A, bool box, cudaStream_t st);

}  // namespace mg5
