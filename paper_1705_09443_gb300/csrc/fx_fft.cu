// Kernels of the fixed-point FFT convolution (fx_line.cuh, fx_fft.cuh).
//
// A CTA transforms C lines, 4 or 8 entries per thread in registers, the lines
// interleaved in shared memory: neighbouring threads are the C lines, so that
// a strided pass (lines = columns) reads and writes C x 16 contiguous bytes
// and a pass along contiguous lines still covers whole 128-byte segments.
// Transformed lines are kept in the digit-reversed order in which the last
// butterflies leave them (the kernel transform is stored in the same order),
// so a forward and a backward transform need no reordering pass, and the
// convolution pass multiplies by the kernel in registers.
#include <cmath>
#include <vector>

#include "fx_fft.cuh"
#include "lss_ctx.h"

namespace {

// This CTA's lines and the reductions over a line: threads with the same
// line are C lanes apart.
template <int LG, int E>
struct FxCta {
    using PL = FxPlan<LG, E>;
    fx2* sm;          // C x L entries
    unsigned* red;    // reduction words, C per slot
    int c, t;

    __device__ unsigned line_or(unsigned f) const {
#pragma unroll
        for (int o = PL::C; o < 32; o <<= 1) f |= __shfl_xor_sync(0xffffffffu, f, o);
        return f;
    }
    __device__ int line_max(int f) const {
#pragma unroll
        for (int o = PL::C; o < 32; o <<= 1) f = max(f, __shfl_xor_sync(0xffffffffu, f, o));
        return f;
    }
    __device__ bool first_lane() const { return (threadIdx.x & 31) < PL::C; }

    // largest e over the line (slot holds e + 2^30, zero before)
    __device__ int reduce_max(int slot, int e) const {
        e = line_max(e);
        if (first_lane()) atomicMax(&red[slot * PL::C + c], (unsigned)(e + (1 << 30)));
        __syncthreads();
        return (int)red[slot * PL::C + c] - (1 << 30);
    }
    __device__ static unsigned fold(const fx2* v) {
        unsigned f = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) f |= fx_fold(v[e]);
        return f;
    }
    // Entries of pass A to the threads that take them in pass B, the line
    // shifted to the bits of pass B.
    template <int A, int B>
    __device__ void exchange(int slot, fx2* v, int& ex) const {
#pragma unroll
        for (int e = 0; e < E; ++e) sm[fx_sidx<LG, E>(fx_pos<LG, E, A>(t, e), c)] = v[e];
        const unsigned f = line_or(fold(v));
        if (first_lane()) atomicOr(&red[slot * PL::C + c], f);
        __syncthreads();
        const int s = min(PL::bits(B) - fx_bits(red[slot * PL::C + c]), 31);
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = sm[fx_sidx<LG, E>(fx_pos<LG, E, B>(t, e), c)];
        fx_shift_line<E>(v, s);
        ex -= s;
    }
    // passes P .. NP-1, the exchange before pass P uses slot + P - 1
    template <int P>
    __device__ void forward(fx2* v, int& ex, int slot, const typename PL::Tw* __restrict__ tw) const {
        if constexpr (P > 0) exchange<P - 1, P>(slot + P - 1, v, ex);
        fx_fwd_pass<LG, E, P>(v, t, tw);
        if constexpr (P + 1 < PL::NP) {
            ex += 2;
            forward<P + 1>(v, ex, slot, tw);
        }
    }
    // passes P .. 0 of the inverse on entries with their parts exchanged
    template <int P>
    __device__ void inverse(fx2* v, int& ex, int slot, const typename PL::Tw* __restrict__ tw) const {
        if constexpr (P + 1 < PL::NP) {
            exchange<P + 1, P>(slot + P, v, ex);
            ex += 2;
        }
        fx_inv_pass<LG, E, P>(v, t, tw);
        if constexpr (P > 0) inverse<P - 1>(v, ex, slot, tw);
    }
    __device__ static void swap(fx2* v) {
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = fx_swap(v[e]);
    }
};

// v 2^E
__device__ __forceinline__ double fx_to_double(long long v, int E) {
    if (E > -1000 && E < 900) return (double)v * __hiloint2double((1023 + E) << 20, 0);
    return scalbn((double)v, E);
}

constexpr int fx_min_ctas(int tpb) { return 1024 / tpb; }   // 64 registers per thread

template <int LG, int E, int MODE>
__global__ void __launch_bounds__(FxPlan<LG, E>::TPB, fx_min_ctas(FxPlan<LG, E>::TPB)) fx_kernel(const FxArgs A) {
    using PL = FxPlan<LG, E>;
    constexpr int L = PL::L, C = PL::C, r0 = 1 << PL::lg(0);
    constexpr bool kFwd = MODE == FX_FWD_IN || MODE == FX_FWD_MID || MODE == FX_CONV;
    constexpr int kSlots = 2 + 2 * (PL::NP - 1);   // reduction words per line, each used once
    extern __shared__ __align__(16) unsigned char fx_smem[];
    FxCta<LG, E> K;
    K.sm = reinterpret_cast<fx2*>(fx_smem);
    K.red = reinterpret_cast<unsigned*>(fx_smem + (size_t)C * L * sizeof(fx2));
    K.c = threadIdx.x % C;
    K.t = threadIdx.x / C;
    for (int i = threadIdx.x; i < kSlots * C; i += PL::TPB) K.red[i] = 0;
    const int t = K.t, n = A.n;
    const int line = blockIdx.x * C + K.c;
    const long long r = blockIdx.y;
    const bool live = line < A.nlines;
    const int la = live ? line / A.lb : 0, lb = live ? line % A.lb : 0;
    const typename PL::Tw* __restrict__ tw = (const typename PL::Tw*)A.tw;

    fx2 v[E];
    int xl;   // the line's exponent
    bool bad;
    if constexpr (MODE == FX_FWD_IN) {
        int ex[E], ey[E], emax = -100000;
        const long long base = r * A.N + (long long)line * n;
        double2 ph = mk(1.0, 0.0);
        if (A.in_mode == MV_IN_PLANEWAVE && live) {   // the factors of the axes before the last
            const double2* p = A.phase + r * A.dim * n;
            ph = A.dim == 2 ? p[line] : p[line / n] * p[n + line % n];
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            v[e] = {0, 0};
            ex[e] = ey[e] = 0;
            const int j = fx_pos<LG, E, 0>(t, e);
            if (e % r0 < r0 / 2 && live && j < n) {
                double2 d;
                if (A.in_mode == MV_IN_PLANEWAVE) {
                    d = ph * A.phase[(r * A.dim + A.dim - 1) * n + j];
                    if (A.uI) A.uI[base + j] = d;
                    d = A.m[(long long)line * n + j] * d;
                } else {
                    d = A.x[base + j];
                    if (A.in_mode == MV_IN_MU) d = A.m[(long long)line * n + j] * d;
                }
                v[e].x = fx_from_double(d.x, ex[e]);
                v[e].y = fx_from_double(d.y, ey[e]);
                if (d.x != 0.0) emax = max(emax, ex[e] + 53);   // (true for NaN)
                if (d.y != 0.0) emax = max(emax, ey[e] + 53);
            }
        }
        __syncthreads();   // the reduction words are zero
        emax = K.reduce_max(0, emax);
        bad = emax >= kFxBad;
        xl = emax - PL::bits_half();
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (e % r0 < r0 / 2) v[e] = {fx_shift(v[e].x, ex[e] - xl), fx_shift(v[e].y, ey[e] - xl)};
    } else {
        int ex[E], emax = -200000;
        const longlong2* in = A.in + r * A.in_r + la * A.in_a + lb * A.in_b;
        const int* ein = A.ein + r * A.ein_r + (long long)la * A.ein_a + (long long)lb * A.ein_b;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            v[e] = {0, 0};
            ex[e] = -200000;
            const int j = kFwd ? fx_pos<LG, E, 0>(t, e) : fx_spos<LG, E>(t, e);
            if (live && (kFwd ? e % r0 < r0 / 2 && j < n : true)) {
                const longlong2 q = in[j * A.in_s];
                v[e] = {q.x, q.y};
                ex[e] = ein[(long long)j * A.ein_s];
            }
        }
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (!kFwd || e % r0 < r0 / 2) emax = max(emax, ex[e] + fx_bits(fx_fold(v[e])));
        __syncthreads();
        emax = K.reduce_max(0, emax);
        bad = emax >= kFxBad;
        xl = emax - (kFwd ? PL::bits_half() : PL::bits(PL::NP - 1));
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (!kFwd || e % r0 < r0 / 2) v[e] = {fx_shift(v[e].x, ex[e] - xl), fx_shift(v[e].y, ex[e] - xl)};
    }

    if constexpr (kFwd) K.template forward<0>(v, xl, 2, tw);
    if constexpr (MODE == FX_FWD_IN || MODE == FX_FWD_MID) {
        if (live) {
            longlong2* out = A.out + r * A.out_r + la * A.out_a + lb * A.out_b;
#pragma unroll
            for (int e = 0; e < E; ++e) out[fx_spos<LG, E>(t, e) * A.out_s] = make_longlong2(v[e].x, v[e].y);
            if (t == 0) A.eout[r * A.nlines + line] = bad ? kFxBad : xl;
        }
        return;
    }
    if constexpr (MODE == FX_CONV) {
        // the product and 16 more bits of each part, so that a line whose
        // entries are small where the kernel is large loses none when it is
        // shifted up for the way back
        constexpr int PS = PL::lg(PL::NP - 1) - 1;
        int kl = live ? line : 0;
        if constexpr (E != kFxBase) {   // the table keeps the order of the kFxBase plan
            constexpr int m = L - 1;
            if (A.dim == 2) kl = fx_store<LG, kFxBase>(fx_freq<LG, E>(kl));
            else kl = (fx_store<LG, kFxBase>(fx_freq<LG, E>(kl >> LG)) << LG) + fx_store<LG, kFxBase>(fx_freq<LG, E>(kl & m));
        }
        const fx_tw* __restrict__ kh = A.khat + (long long)kl * L;
        unsigned frac[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            unsigned fx, fy;
            int ks = fx_spos<LG, E>(t, e);
            if constexpr (E != kFxBase) ks = fx_store<LG, kFxBase>(fx_freq<LG, E>(ks));
            fx_kmul<PS>(v[e], kh[ks], v[e], fx, fy);
            frac[e] = __byte_perm(fx, fy, 0x7632);
        }
        const unsigned f = K.line_or(FxCta<LG, E>::fold(v));
        if (K.first_lane()) atomicOr(&K.red[C + K.c], f);
        __syncthreads();
        const int s = min(PL::bits(PL::NP - 1) - fx_bits(K.red[C + K.c]), 31);
#pragma unroll
        for (int e = 0; e < E; ++e)
            v[e] = {fx_lift(v[e].x, frac[e] << 16, s), fx_lift(v[e].y, frac[e] & 0xffff0000u, s)};
        xl += A.ek[kl] + 64 + PS - s;
    }
    K.swap(v);
    K.template inverse<PL::NP - 1>(v, xl, MODE == FX_CONV ? 2 + (PL::NP - 1) : 2, tw);
    K.swap(v);
    if (!live) return;
    if constexpr (MODE == FX_CONV || MODE == FX_INV_MID) {
        longlong2* out = A.out + r * A.out_r + la * A.out_a + lb * A.out_b;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int j = fx_pos<LG, E, 0>(t, e);
            if (e % r0 < r0 / 2 && j < n) out[j * A.out_s] = make_longlong2(v[e].x, v[e].y);
        }
        if (t == 0) A.eout[r * A.nlines + line] = bad ? kFxBad : xl;
    } else {
        const long long base = r * A.N + (long long)line * n;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int j = fx_pos<LG, E, 0>(t, e);
            if (!(e % r0 < r0 / 2 && j < n)) continue;
            double2 d = mk(fx_to_double(v[e].x, xl), fx_to_double(v[e].y, xl));
            if (bad) d = mk(nan(""), nan(""));
            if (A.out_mode == MV_OUT_A) {
                A.y[base + j] = A.x[base + j] + d;
            } else if (A.out_mode == MV_OUT_AT) {
                A.y[base + j] = A.x[base + j] + A.m[(long long)line * n + j] * d;
            } else {
                A.y[base + j] = mk(-d.x, -d.y);
            }
        }
    }
}

// One CTA per line of the kernel transform (storage order): its largest part
// sets the exponent of the line's digits.
template <int LG>
__global__ void __launch_bounds__(128) fx_khat_kernel(const double2* __restrict__ khat, fx_tw* __restrict__ out,
                                                      int* __restrict__ ek, int dim) {
    constexpr int L = 1 << LG;
    __shared__ unsigned big;
    const int line = blockIdx.x;
    long long src;
    if (dim == 2) src = (long long)fx_freq<LG, kFxBase>(line) * L;
    else src = ((long long)fx_freq<LG, kFxBase>(line >> LG) * L + fx_freq<LG, kFxBase>(line & (L - 1))) * L;
    if (threadIdx.x == 0) big = 0;
    __syncthreads();
    unsigned e = 0;
    for (int j = threadIdx.x; j < L; j += blockDim.x) {
        const double2 k = khat[src + j];
        e = max(e, max((unsigned)(__double2hiint(k.x) & 0x7fffffff), (unsigned)(__double2hiint(k.y) & 0x7fffffff)) >> 20);
    }
    atomicMax(&big, e);
    __syncthreads();
    const int x = fx_kernel_exp(big);
    if (threadIdx.x == 0) ek[line] = x;
    for (int s = threadIdx.x; s < L; s += blockDim.x) {
        const double2 k = khat[src + fx_freq<LG, kFxBase>(s)];
        out[(long long)line * L + s] =
            fx_kernel_digits(__double2ll_rn(scalbn(k.x, -x)), __double2ll_rn(scalbn(k.y, -x)));
    }
}

__global__ void fx_phase_kernel(const double* __restrict__ dirs, double2* __restrict__ phase, int n, int tot,
                                double omega, double h) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= tot) return;
    double sn, cs;
    sincos(omega * dirs[i / n] * ((i % n + 1) * h), &sn, &cs);
    phase[i] = mk(cs, sn);
}

template <int LG, int E, int MODE>
cudaError_t launch(const FxArgs& A, int R, cudaStream_t s) {
    using PL = FxPlan<LG, E>;
    constexpr size_t sh = (size_t)PL::C * PL::L * sizeof(fx2) + (2 + 2 * (PL::NP - 1)) * PL::C * sizeof(unsigned);
    if constexpr (sh > 48 * 1024) {
        std::lock_guard<std::mutex> lock(lss_config_mutex());
        long long& done = lss_dev_cache((const void*)fx_kernel<LG, E, MODE>, 0);
        if (!done) {
            const cudaError_t e =
                cudaFuncSetAttribute(fx_kernel<LG, E, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
            if (e) return e;
            done = 1;
        }
    }
    fx_kernel<LG, E, MODE><<<dim3((A.nlines + PL::C - 1) / PL::C, R), PL::TPB, sh, s>>>(A);
    return cudaGetLastError();
}

template <int LG, int E>
cudaError_t launch_mode(int mode, const FxArgs& A, int R, cudaStream_t s) {
    switch (mode) {
        case FX_FWD_IN: return launch<LG, E, FX_FWD_IN>(A, R, s);
        case FX_CONV: return launch<LG, E, FX_CONV>(A, R, s);
        case FX_INV_OUT: return launch<LG, E, FX_INV_OUT>(A, R, s);
        default: break;
    }
    if constexpr (LG <= 8) {   // 3D: n <= 128
        if (mode == FX_FWD_MID) return launch<LG, E, FX_FWD_MID>(A, R, s);
        if (mode == FX_INV_MID) return launch<LG, E, FX_INV_MID>(A, R, s);
    }
    return cudaErrorInvalidValue;
}

template <int LG>
cudaError_t launch_plan(int mode, int E, const FxArgs& A, int R, cudaStream_t s) {
    if constexpr (LG <= 10)
        if (E == 4) return launch_mode<LG, 4>(mode, A, R, s);
    return launch_mode<LG, 8>(mode, A, R, s);
}

}  // namespace

bool lss_fx_supported(int lg) { return lg >= kFxMinLg && lg <= kFxMaxLg; }

int lss_fx_lines(int lg) {
    static_assert(FxPlan<6, 8>::C == FxPlan<9, 8>::C && FxPlan<10, 8>::C == FxPlan<11, 8>::C, "lines per CTA");
    return lg <= 9 ? FxPlan<9, 8>::C : FxPlan<11, 8>::C;
}

// Eight entries per thread unless that leaves fewer than 256 threads per SM in
// the widest pass, then four (n = 64: 22.5 against 30.7 us per application,
// n = 128: 24.6 against 32.8; equal at n = 256 with one right-hand side, and
// with two 53.2 against 47.1).
int lss_fx_entries(int lg, long long entries, int num_sms) {
    return lg <= 10 && entries / 8 < 256LL * num_sms ? 4 : 8;
}

cudaError_t lss_fx_pass(int mode, int lg, int E, const FxArgs& A, int R, cudaStream_t s) {
    switch (lg) {
        case 6: return launch_plan<6>(mode, E, A, R, s);
        case 7: return launch_plan<7>(mode, E, A, R, s);
        case 8: return launch_plan<8>(mode, E, A, R, s);
        case 9: return launch_plan<9>(mode, E, A, R, s);
        case 10: return launch_plan<10>(mode, E, A, R, s);
        case 11: return launch_plan<11>(mode, E, A, R, s);
        default: return cudaErrorInvalidValue;
    }
}

namespace {

// khat (L^(d-1) lines of L entries, natural order on every axis, the last axis
// contiguous) -> digits in storage order on every axis, an exponent per line
cudaError_t khat_digits(int lg, int dim, const double2* khat, fx_tw* out, int* ek, cudaStream_t s) {
    const unsigned lines = dim == 2 ? 1u << lg : 1u << (2 * lg);
    switch (lg) {
        case 6: fx_khat_kernel<6><<<lines, 128, 0, s>>>(khat, out, ek, dim); break;
        case 7: fx_khat_kernel<7><<<lines, 128, 0, s>>>(khat, out, ek, dim); break;
        case 8: fx_khat_kernel<8><<<lines, 128, 0, s>>>(khat, out, ek, dim); break;
        case 9: fx_khat_kernel<9><<<lines, 128, 0, s>>>(khat, out, ek, dim); break;
        case 10: fx_khat_kernel<10><<<lines, 128, 0, s>>>(khat, out, ek, dim); break;
        case 11: fx_khat_kernel<11><<<lines, 128, 0, s>>>(khat, out, ek, dim); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace

int lss_fx_tables(lss_ctx* c, const double2* khat, cudaStream_t s) {
    const int lg = c->lgL, L = c->L;
    const size_t lines = c->dim == 3 ? (size_t)L * L : (size_t)L;
    static_assert(FxPlan<7, 8>::kThree == false && FxPlan<8, 8>::kThree && FxPlan<10, 8>::kThree &&
                  FxPlan<11, 8>::kThree == false, "twiddle forms below");
    const bool three = lg >= 8 && lg <= 10;   // FxPlan::kThree
    const size_t tws = three ? sizeof(fx_tw3) : sizeof(fx_tw);
    c->fx_host.resize(L * tws / sizeof(int));
    std::vector<long double> re(L), im(L);
    fx_host_roots(L, re.data(), im.data());
    for (int k = 0; k < L; ++k) {
        if (three) fx_host_tw(re[k], im[k], ((fx_tw3*)c->fx_host.data())[k]);
        else fx_host_tw(re[k], im[k], ((fx_tw*)c->fx_host.data())[k]);
    }
    cudaError_t e = cudaMalloc(&c->fx_tw, L * tws + lines * sizeof(int));
    if (e) {
        cudaGetLastError();
        return lss_fail(c, LSS_ERR_OOM, "device allocation failed: fixed-point operator tables");
    }
    c->fx_ek = (int*)((char*)c->fx_tw + L * tws);
    e = cudaMemcpyAsync(c->fx_tw, c->fx_host.data(), L * tws, cudaMemcpyHostToDevice, s);
    if (!e) {
        ProfScope ps(c, s, LSS_PROF_SETUP, 1);
        e = khat_digits(lg, c->dim, khat, (fx_tw*)c->fx_khat, c->fx_ek, s);
    }
    return lss_check_cuda(c, e, "fixed-point operator tables");
}

cudaError_t lss_fx_phases(const double* dirs, double2* phase, int dim, int n, int R, double omega, double h,
                          cudaStream_t s) {
    const int tot = R * dim * n;
    fx_phase_kernel<<<(tot + 255) / 256, 256, 0, s>>>(dirs, phase, n, tot, omega, h);
    return cudaGetLastError();
}
