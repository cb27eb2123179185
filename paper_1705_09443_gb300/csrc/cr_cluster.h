// Slab solves of the sweeps by cyclic reduction on thread-block clusters (cr_cluster.cu).
#pragma once
#include "lss_ctx.h"

enum CrcMode { CRC_A = 0, CRC_E = 1 };   // first pass (first and last layers kept), second pass (couplings subtracted, D_i written)

constexpr int kCrcLevels = 18;
struct CrcLv { int K, dinv, cbe, dcdb; };   // as CrLevelOffs, in blocks

struct CrcArgs {
    // the caller's: right-hand sides, vectors of the mode and direction
    int R;
    const void* f;           // forward: R x n_tot^2 sparsified right-hand side, x2 index slowest
    const double2* yin;      // transposed: R x n^2 vectors on I
    void *a_first, *a_last;  // CRC_A outputs, [slab][k][R]
    const void *lam, *phi;   // CRC_E couplings, [slab][k][R]
    double2* y;              // forward CRC_E output, R x n^2 (or R x n_tot^2 when y_grid)
    int y_grid;
    void* X;                 // transposed CRC_E output: R x n_tot^2 grid, x2 index slowest
    int beside;              // the pass's 16-wide slabs run beside this launch (block LU)
    // filled by lss_cr_cluster
    const SlabDev* slabs;
    int n_slabs, n_tot, n, b, slab0, L, P;
    const void *fac, *coef;
    long long t0[2], p0[2];  // entry offsets of the level-0 bands and D^{-1} rows, 16- and 32-wide slabs
    CrcLv lv[kCrcLevels];
};

// One pass over the slabs [s0, s0 + nsl) of block width ldw (16 or 32);
// LSS_ERR_UNSUPPORTED when a slab's rows do not fit a cluster's shared memory.
int lss_cr_cluster(lss_ctx* c, int mode, bool transpose, CrcArgs A, int s0, int nsl, int ldw, cudaStream_t s);

// Right-hand sides that share a cluster in the forward passes over 16-wide slabs.
int lss_cr_cluster_rhs(const lss_ctx* c, int R);
