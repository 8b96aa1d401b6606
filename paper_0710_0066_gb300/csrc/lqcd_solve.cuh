// lqcd_solve.cuh -- what the persistent solver kernels share: the argument
// block of one launch, the per-system state and the launch plan.
#pragma once
#include "lqcd_common.cuh"

constexpr int NSYS_MAX = 64;
constexpr int NQ = 3;
constexpr int SPLIT_NQ = 4;  // partial sums per CTA in lqcd_split.cu
constexpr int NACC = 5;  // iteration sums kept beside the sticky status

// per-system state codes in the flag arrays
enum { F_ACTIVE = 0, F_DONE = 1, F_NAN = 2, F_MAXIT = 3 };

struct SolveArgs {
    Geo g;
    int mode;  // MODE_INTRA: slabs, MODE_ALL: whole lattice
    double k2;
    double diag;  // the system is diag - k2 H_eo H_oe (1, or 1 + rho for W3,eo)
    int method;   // SOLVER_BICGSTAB or SOLVER_SERIES (inner iteration)
    int guess;    // 1: x holds an initial guess on entry, 0: start from x = 0
    int nsys, cps;
    int ngrp;   // groups of cps CTAs; group k solves the systems k, k + ngrp, ...
    // order of a system's groups of 32 sites (lqcd_split.cu): as the sites, or
    // in tiles of 2^lt[0] slices x 2^lt[1] planes x 2^lt[2] groups of a plane,
    // 2^nt[0] tiles along x1 and 2^nt[1] along a plane's groups
    int tiled, lt[3], nt[2];
    int chunk;  // sites of one system handled by one CTA (the last CTA may get fewer)
    int slab0, slabstep;
    int nsite;
    GaugeF U64, UP;
    SpinorF b, x, r64;  // double, parity 0
    SpinorF t64;        // parity 1: double (double solve) or df pairs (mixed)
    SpinorF r, rh, p, v, s, t;  // inner precision, parity 0
    SpinorF tmp;        // inner precision, parity 1
    SpinorF e;          // inner solution (single; double for the double solver)
    SpinorF eb;         // its best iterate (lqcd_split.cu)
    double tol, inner_tol;
    int max_iter, max_outer, max_inner;
    double* part;       // double-buffered partial sums of every CTA
    unsigned* bar;      // one barrier counter per system, BAR_STRIDE apart
    int* status;
    int* sticky;        // first failure of any solve since the host last read it
    unsigned long long* acc;  // [5] inner iterations, BiCGstab iterations x sites,
                              // outer cycles x sites, series iterations x sites,
                              // Schwarz-preconditioned iterations x sites
    int* iters;         // [nsys]
    double* resid;      // [nsys]
    int* outer_out;
    long long spin_limit;  // clock64 cycles of one barrier wait before LQCD_ERR_TIMEOUT
    // Schwarz-preconditioned inner solve of the whole lattice (SOLVER_SAP):
    // full-lattice vectors in the inner precision, [0] the even, [1] the odd
    // parity block; fy (the inner solution) in the precision of e, whose
    // even block it is
    double kappa;
    int nsap;  // geometric-series terms of every block solve of the preconditioner
    // SOLVER_SAPB: 4-D Schwarz blocks of extents bk[mu] (2 or 4, lbk = log2),
    // nbk[mu] = L[mu] / bk[mu] blocks per direction, nblk in all, bvh sites
    // of one parity in a block
    int bk[4], lbk[4], nbk[4], nblk, bvh;
    SpinorF fr[2], frh[2], fp[2], fv[2], fs[2], ft[2], fzp[2], fzs[2], fw1[2], fw2[2], fy[2];
};

struct SysSt {  // the CTA's own system
    double bn2, rn2, rr, itol2;
    double2 rho, alpha, omega, beta;
    int active, idone, it, itc, flag;
};

// barrier counters of different systems sit on different 128-byte lines
constexpr int BAR_STRIDE = 32;

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}


// lqcd_split.cu: the persistent solver of single- and double-precision inner
// storage.  split_init sets its kernels' attributes and reads their occupancy
// (gmax: the largest grid) and the bytes of the L2; split_plan picks the
// kernel for the systems of A (spt: lqcd_set_solver_schedule) and sets cps,
// ngrp, chunk and the tiling.
constexpr int SPLIT_NVAR = 6;
struct SplitPlan {
    const void* fn;
    int grid, block, smem;
};
cudaError_t split_init(int num_sms, int occ[SPLIT_NVAR][2], int* gmax, int* l2);
SplitPlan split_plan(SolveArgs& A, int prec, int method, int spt, int num_sms, const int occ[SPLIT_NVAR][2],
                     int l2);
