// Passes of the zero-padded FFT convolution in 64-bit fixed point
// (fx_line.cuh), for the 2D and the 3D LS operator.
#pragma once
#include <cuda_runtime.h>
#include "fx_line.cuh"

// What a pass does with its lines.
enum FxMode {
    FX_FWD_IN = 0,    // n complex doubles per line (m.*u, u or m.*u_I) -> transformed line
    FX_FWD_MID = 1,   // n fixed-point entries -> transformed line
    FX_CONV = 2,      // n entries: transform, multiply by the kernel transform, back; n entries out
    FX_INV_MID = 3,   // L entries of a transformed line -> n entries
    FX_INV_OUT = 4    // L entries -> n complex doubles through the operator's epilogue
};

// Lines of one pass.  Line l = a * lb + b of right-hand side r has entry j at
// r * in_r + a * in_a + b * in_b + j * in_s (output alike); the exponent of
// entry j is ein[r * ein_r + a * ein_a + b * ein_b + j * ein_s] and the line's
// own goes to eout[r * nlines + l].
struct FxArgs {
    int nlines, lb, n;
    const longlong2* in;
    longlong2* out;
    long long in_r, in_a, in_b, in_s, out_r, out_a, out_b, out_s;
    const int* ein;
    int* eout;
    long long ein_r;
    int ein_a, ein_b, ein_s;
    const void* tw;         // twiddle digits in the form of the line length's plan
    const fx_tw* khat;      // FX_CONV: [line][L], storage order along the line
    const int* ek;          // its exponent per line
    // FX_FWD_IN / FX_INV_OUT: vectors on I (line l, entry j at r * N + l * n + j)
    const double2* x;
    const double* m;
    double2* y;
    double2* uI;
    const double2* phase;   // FX_FWD_IN, plane waves: exp(i omega d_a p_a), [r][axis][n]
    long long N;
    int dim, in_mode, out_mode;
};

bool lss_fx_supported(int lg);
int lss_fx_lines(int lg);   // lines per CTA
// Entries per thread for an operator of the given line length whose widest
// pass transforms `entries` entries.  Every pass of one application takes the same.
int lss_fx_entries(int lg, long long entries, int num_sms);
// R right-hand sides; lg = log2 of the line length, E entries per thread.
cudaError_t lss_fx_pass(int mode, int lg, int E, const FxArgs& A, int R, cudaStream_t s);
cudaError_t lss_fx_phases(const double* dirs, double2* phase, int dim, int n, int R, double omega, double h,
                          cudaStream_t s);
