// Interface recurrences of the sweep for many right-hand sides: one
// cooperative kernel over all slabs (Sec. 2.3-2.4; the recurrences are stated
// in slab.cu, those of two fronts in launch_recur2_chains).
//
// Only the chains lambda and phi depend on the slab before; mu, nu and the
// middle slab's couplings are formed for all slabs at once between the two
// chain passes, with no barrier inside.  A chain step is one product of an
// n_tot x n_tot map with the n_tot x R vectors (two with two fronts), a grid
// barrier closes it.  What bounds a step is latency and, in FP64, the FP64
// pipe (2 multiply-adds per clock and SM), so a step has to reach every SM: a
// task is only TRC = 8, 4, 2 or 1 rows of CW columns, its length-n_tot sums
// split over the 16 warps of a CTA (lanes along the columns, so vector rows
// are read coalesced and map entries are broadcast from shared memory, a
// partial sum per warp added up at the end).  A CTA's next map rows do not
// depend on the chain and are copied by cp.async before the barrier.
// FP64, n = 256, 16 right-hand sides, one front: 2.4 ms per sweep (the FP64 pipe
// 70 % busy) against 19.1 of 16-column tiles of 32 rows, which left 18 CTAs per
// step; FP32, n = 512, 64 right-hand
// sides, two fronts: 2.05 ms against 3.35.
#include <algorithm>
#include <mutex>

#include "lss_common.cuh"
#include "lss_ctx.h"

namespace {

constexpr int kRwThreads = 512, kRwWarps = kRwThreads / 32;

template <typename C>
struct RwArgs {
    int ns, mid, n_tot, R, two;
    int trc_tiles, col_tiles;   // row and column tiles of one product
    const C* maps;              // Lambda, Gamma, Phi (Psi with two fronts): n_slabs x n_tot^2 each
    const C* a_first;
    const C* a_last;
    C* lam;
    C* phi;
    unsigned* bar;
    int* err;
};

// out = base - M x (- M2 x2)
template <typename C>
struct RwProd {
    const C *M, *x, *base, *M2, *x2;
    C* out;
};

// Steps: the forward chains, one step of independent products, the backward chains.
template <typename C>
struct RwPlan {
    const RwArgs<C>& A;
    long long nt2, vec;
    int S;
    __device__ explicit RwPlan(const RwArgs<C>& a) : A(a), nt2((long long)a.n_tot * a.n_tot), vec((long long)a.n_tot * a.R) {
        S = A.two ? max(A.mid - 1, A.ns - 2 - A.mid) : A.ns - 2;
        if (S < 0) S = 0;
    }
    __device__ int steps() const { return 2 * S + 1; }
    __device__ const C* map(int which, int i) const { return A.maps + ((long long)which * A.ns + i) * nt2; }
    // current vectors of the chains' first slabs are the a_i themselves
    __device__ const C* lam(int i) const { return i == 0 ? A.a_last : A.lam + i * vec; }
    __device__ const C* phi_end(int i) const { return i == A.ns - 1 ? A.a_first + i * vec : A.phi + i * vec; }
    __device__ int products(int st) const {
        if (st == S) return A.two ? max(0, A.mid - 1) + (A.ns - 2 - A.mid) + 2 : A.ns - 1;
        if (!A.two) return 1;
        const int s = st < S ? st : st - S - 1;
        return (A.mid - 1 - s >= 1 ? 1 : 0) + (A.ns - 2 - A.mid - s >= 1 ? 1 : 0);
    }
    __device__ RwProd<C> product(int st, int p) const {
        RwProd<C> q;
        q.M2 = q.x2 = nullptr;
        const int ns = A.ns, c = A.mid;
        if (!A.two) {
            if (st < S) {                       // lambda_i = last(a_i) - Lambda_i lambda_{i-1}
                const int i = st + 1;
                q.M = map(0, i); q.x = lam(i - 1); q.base = A.a_last + i * vec; q.out = A.lam + i * vec;
            } else if (st == S) {               // mu_i = first(a_i) - Gamma_i lambda_{i-1}
                const int i = p + 1;
                q.M = map(1, i); q.x = lam(i - 1); q.base = A.a_first + i * vec; q.out = A.phi + i * vec;
            } else {                            // phi_i = mu_i - Phi_i phi_{i+1}
                const int i = ns - 2 - (st - S - 1);
                q.M = map(2, i); q.x = A.phi + (i + 1) * vec; q.base = q.out = A.phi + i * vec;
            }
            return q;
        }
        if (st == S) {
            const int nmu = max(0, c - 1);
            if (p < nmu) {                      // mu_i left of the middle slab
                const int i = p + 1;
                q.M = map(1, i); q.x = lam(i - 1); q.base = A.a_first + i * vec; q.out = A.phi + i * vec;
            } else if (p < nmu + ns - 2 - c) {  // nu_i right of it
                const int i = c + 1 + p - nmu;
                q.M = map(3, i); q.x = phi_end(i + 1); q.base = A.a_last + i * vec; q.out = A.lam + i * vec;
            } else {                            // the middle slab: first layer (p last), last layer
                const bool first = p == nmu + ns - 2 - c;
                q.M = map(first ? 2 : 3, c); q.x = phi_end(c + 1);
                if (c > 0) { q.M2 = map(first ? 1 : 0, c); q.x2 = lam(c - 1); }
                q.base = (first ? A.a_first : A.a_last) + c * vec;
                q.out = (first ? A.phi : A.lam) + c * vec;
            }
            return q;
        }
        const bool fwd = st < S;
        const int s = fwd ? st : st - S - 1;
        const bool left = p == 0 && c - 1 - s >= 1;
        if (fwd && left) {
            const int i = 1 + s;
            q.M = map(0, i); q.x = lam(i - 1); q.base = A.a_last + i * vec; q.out = A.lam + i * vec;
        } else if (fwd) {
            const int i = ns - 2 - s;
            q.M = map(2, i); q.x = phi_end(i + 1); q.base = A.a_first + i * vec; q.out = A.phi + i * vec;
        } else if (left) {
            const int i = c - 1 - s;
            q.M = map(2, i); q.x = A.phi + (i + 1) * vec; q.base = q.out = A.phi + i * vec;
        } else {
            const int i = c + 1 + s;
            q.M = map(0, i); q.x = A.lam + (i - 1) * vec; q.base = q.out = A.lam + i * vec;
        }
        return q;
    }
};

template <typename T, int CW, int TRC>
__global__ void __launch_bounds__(kRwThreads) recur_wide_kernel(const RwArgs<cx<T>> A) {
    using C = cx<T>;
    constexpr int LPC = CW < 32 ? CW : 32;    // lanes along the columns
    constexpr int NC = CW / LPC;              // columns per lane
    constexpr int SUB = 32 / LPC;             // slices of a sum per warp
    constexpr int NS = kRwWarps * SUB;
    extern __shared__ __align__(16) unsigned char rws[];
    const int K = A.n_tot, R = A.R, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    C* Mb = reinterpret_cast<C*>(rws);        // 2 x TRC x K: map rows of this and the next task
    C* red = Mb + 2 * TRC * K;                // kRwWarps x TRC x CW partial sums
    const RwPlan<C> P(A);
    const int nsteps = P.steps(), per = A.trc_tiles * A.col_tiles;

    for (long long e = blockIdx.x * (long long)kRwThreads + tid; e < P.vec; e += (long long)gridDim.x * kRwThreads) {
        if (!A.two || A.mid > 0) A.lam[e] = A.a_last[e];   // (the middle slab's is a product)
        if (A.two) A.phi[(A.ns - 1) * P.vec + e] = A.a_first[(A.ns - 1) * P.vec + e];
    }
    // this CTA's tasks in order
    int st = 0, task = blockIdx.x;
    auto settle = [&] {   // to the next step that has a task for this CTA
        while (st < nsteps && task >= P.products(st) * per) { ++st; task = blockIdx.x; }
    };
    auto copy_rows = [&](const C* M, int row0, C* dst) {
        for (int e = tid; e < TRC * K; e += kRwThreads) {
            const bool ok = row0 + e / K < K;
            cp_async_entry(dst + e, ok ? M + (long long)row0 * K + e : M, ok);
        }
        cp_async_commit();
    };
    auto prefetch = [&](C* dst) {
        if (st < nsteps) copy_rows(P.product(st, task / per).M, task % per / A.col_tiles * TRC, dst);
        else cp_async_commit();
    };
    settle();
    prefetch(Mb);
    int buf = 0, nbar = 0;
    const int col0 = lane % LPC, slice = warp * SUB + lane / LPC;
    while (st < nsteps) {
        const RwProd<C> q = P.product(st, task / per);
        const int row0 = task % per / A.col_tiles * TRC, cb = task % A.col_tiles * CW;
        const int cst = st;
        task += gridDim.x;
        settle();
        prefetch(Mb + (buf ^ 1) * TRC * K);
        for (; nbar < cst; ++nbar) grid_barrier_count(A.bar, (nbar + 1) * gridDim.x, A.err);
        // the outputs' base values, read while the sums form
        C bv[(TRC * CW + kRwThreads - 1) / kRwThreads];
        constexpr int NB = (TRC * CW + kRwThreads - 1) / kRwThreads;
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int e = tid + u * kRwThreads, row = row0 + e / CW, col = cb + e % CW;
            bv[u] = e < TRC * CW && row < K && col < R ? q.base[(long long)row * R + col] : czero<C>();
        }
        C acc[TRC][NC];
#pragma unroll
        for (int a = 0; a < TRC; ++a)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[a][c] = czero<C>();
        bool on[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) on[c] = cb + col0 + 32 * c < R;
        auto sums = [&](const C* Ms, const C* x) {
#pragma unroll 4
            for (int k = slice; k < K; k += NS) {
                C xv[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) xv[c] = on[c] ? x[(long long)k * R + cb + col0 + 32 * c] : czero<C>();
#pragma unroll
                for (int a = 0; a < TRC; ++a) {
                    const C m = Ms[a * K + k];
#pragma unroll
                    for (int c = 0; c < NC; ++c) acc[a][c] = cfma(m, xv[c], acc[a][c]);
                }
            }
        };
        cp_async_wait<1>();
        __syncthreads();
        C* Ms = Mb + buf * TRC * K;
        sums(Ms, q.x);
        if (q.M2) {   // the middle slab's second coupling: its rows through the same buffer
            __syncthreads();
            copy_rows(q.M2, row0, Ms);
            cp_async_wait<0>();
            __syncthreads();
            sums(Ms, q.x2);
        }
#pragma unroll
        for (int o = LPC; o < 32; o <<= 1)
#pragma unroll
            for (int a = 0; a < TRC; ++a)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    acc[a][c].x += __shfl_xor_sync(0xffffffffu, acc[a][c].x, o);
                    acc[a][c].y += __shfl_xor_sync(0xffffffffu, acc[a][c].y, o);
                }
        if (lane < LPC)
#pragma unroll
            for (int a = 0; a < TRC; ++a)
#pragma unroll
                for (int c = 0; c < NC; ++c) red[(warp * TRC + a) * CW + col0 + 32 * c] = acc[a][c];
        __syncthreads();
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int e = tid + u * kRwThreads, row = row0 + e / CW, col = cb + e % CW;
            if (e < TRC * CW && row < K && col < R) {
                C s = red[e];
#pragma unroll
                for (int w = 1; w < kRwWarps; ++w) s = s + red[w * TRC * CW + e];
                q.out[(long long)row * R + col] = bv[u] - s;
            }
        }
        __syncthreads();   // partial sums and map rows may be overwritten
        buf ^= 1;
    }
    cp_async_wait<0>();
    for (; nbar < nsteps - 1; ++nbar) grid_barrier_count(A.bar, (nbar + 1) * gridDim.x, A.err);
}

template <typename T, int CW>
const void* rw_kernel(int trc) {
    switch (trc) {
        case 8: return (const void*)recur_wide_kernel<T, CW, 8>;
        case 4: return (const void*)recur_wide_kernel<T, CW, 4>;
        case 2: return (const void*)recur_wide_kernel<T, CW, 2>;
        default: return (const void*)recur_wide_kernel<T, CW, 1>;
    }
}

template <typename T>
int recur_wide(lss_ctx* c, const cx<T>* maps, cx<T>* lam, cx<T>* phi, const cx<T>* a_first, const cx<T>* a_last, int R,
               cudaStream_t s) {
    using C = cx<T>;
    const int K = c->n_tot, CW = R <= 16 ? 16 : R <= 32 ? 32 : 64;
    const bool two = c->fronts == 2;
    const int nct = (R + CW - 1) / CW, chains = two ? 2 : 1;
    auto smem_of = [&](int trc) { return sizeof(C) * ((size_t)2 * trc * K + (size_t)kRwWarps * trc * CW); };
    // the most rows per task (the vectors are read once per task) that leave a
    // chain step tasks for three quarters of the SMs
    int trc = 8;
    while (trc > 1 && (4LL * chains * ((K + trc - 1) / trc) * nct < 3LL * c->num_sms || smem_of(trc) > 220 * 1024)) trc /= 2;
    const size_t smem = smem_of(trc);
    const void* k = CW == 16 ? rw_kernel<T, 16>(trc) : CW == 32 ? rw_kernel<T, 32>(trc) : rw_kernel<T, 64>(trc);
    int per = 0;
    {
        std::lock_guard<std::mutex> lock(lss_config_mutex());
        long long& cfg = lss_dev_cache(k, 0);   // shared memory opted into
        if ((long long)smem > cfg) {
            const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)std::max<size_t>(smem, 48 * 1024));
            if (e) return lss_check_cuda(c, e, "recurrence attribute");
            cfg = (long long)smem;
        }
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, kRwThreads, smem);
        if (e || per < 1) return lss_check_cuda(c, e ? e : cudaErrorInvalidConfiguration, "recurrence occupancy");
    }
    RwArgs<C> A{};
    A.ns = c->n_slabs;
    A.mid = c->mid;
    A.n_tot = K;
    A.R = R;
    A.two = two;
    A.trc_tiles = (K + trc - 1) / trc;
    A.col_tiles = nct;
    A.maps = maps;
    A.a_first = a_first;
    A.a_last = a_last;
    A.lam = lam;
    A.phi = phi;
    A.bar = c->d_bar;
    A.err = c->d_err;
    // (the independent products of the middle step fill whatever grid the chains leave)
    const long long tasks = (long long)A.trc_tiles * nct * std::max(chains, c->n_slabs);
    const int nb = (int)std::min<long long>((long long)per * c->num_sms, std::max<long long>(1, tasks));
    ProfScope ps(c, s, LSS_PROF_RECUR, 1);
    cudaError_t e = cudaMemsetAsync(A.bar, 0, sizeof(unsigned), s);   // the barriers' arrival counter
    void* args[] = {&A};
    if (!e) e = cudaLaunchCooperativeKernel(k, dim3(nb), dim3(kRwThreads), args, smem, s);
    return lss_check_cuda(c, e, "recurrence launch");
}

}  // namespace

int lss_recur_wide(lss_ctx* c, const void* maps, void* lam, void* phi, const void* a_first, const void* a_last, int R,
                   cudaStream_t s) {
    if (c->prec == LSS_FP64)
        return recur_wide<double>(c, (const double2*)maps, (double2*)lam, (double2*)phi, (const double2*)a_first,
                                  (const double2*)a_last, R, s);
    return recur_wide<float>(c, (const float2*)maps, (float2*)lam, (float2*)phi, (const float2*)a_first,
                             (const float2*)a_last, R, s);
}
