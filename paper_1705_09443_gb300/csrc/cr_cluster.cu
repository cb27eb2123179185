// Cyclic-reduction slab solves on thread-block clusters: the two passes of the
// sweep (slab.cu) and of the transposed sweep (adjoint.cu).
//
// A solve is a chain of 2 log2(n_tot) levels; within a level every block row
// is independent.  A cluster of CL CTAs solves NR right-hand sides of one slab:
// CTA q owns the block rows [q P, (q + 1) P) in its shared memory, reads the
// neighbour rows of other CTAs through distributed shared memory, and the
// levels are separated by one cluster barrier each.  A task is one block row:
// its blocks are read straight into registers (16 entries of the two coupling
// blocks and 8 of the inverse per lane, coalesced), those of a level's first
// task before the barrier, so that the factor latency overlaps it.  A 16-wide
// row is a warp's task (a half warp per block), a 32-wide row that of four
// warps (block x half of the columns, partial sums through shared memory).  A CTA
// has 256 threads for 16-wide slabs, 512 or 256 for 32-wide ones (launch).
//
// Forward operator, level by level:
//   P0     y_o = D_o^{-1} b_o on the odd rows
//   F(l)   b_e -= C_e y_{e-1} + B_e y_{e+1} on the even rows, then
//          y = D^{-1} b where the row is odd in level l + 1 or the last one left
//   B(l)   x_o = y_o - D^{-1}C x_{o-1} - D^{-1}B x_{o+1}
//   B(0)   x_o = y_o - D_o^{-1} (C_o x_{o-1} + B_o x_{o+1}), bands
// Transposed (adjoint.cu's formulas), the inverses of levels >= 1 on the way back:
//   F(0)   bands of the odd neighbours;  F(l) b_e -= (D^{-1}B)_{e-1}^T b_{e-1} + (D^{-1}C)_{e+1}^T b_{e+1}
//   B(l)   x_o = D_o^{-T} (b_o - B_{o-1}^T x_{o-1} - C_{o+1}^T x_{o+1})
#include <algorithm>

#include <cooperative_groups.h>

#include "cr_cluster.h"
#include "lss_common.cuh"

namespace {

namespace cg = cooperative_groups;

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

template <typename C>
__device__ __forceinline__ C shfl_xor_c(C v, int o) {
    v.x = __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y = __shfl_xor_sync(0xffffffffu, v.y, o);
    return v;
}

template <typename T, int MODE, bool TR, int G, int NR, int NT>
struct Crc {
    using C = cx<T>;
    static constexpr int TW = G == 16 ? 1 : 4;                 // warps per task
    static constexpr int kTeams = NT / 32 / TW;
    // Columns beyond the layers of a 32-wide slab are zero.  FP64 is bound by its
    // pipe and neither reads nor multiplies them (20 layers, n = 64, 16 right-hand
    // sides: P 1.33 -> 1.16 ms); in FP32 the test takes longer than it saves.
    static constexpr bool kSkip = G == 32 && sizeof(T) == 8;
    static constexpr int XS = 18;                              // staged entries of one vector (16, padded for the banks)
    static constexpr int kStage = (G == 16 ? 2 : 1) * NR * XS; // per warp
    static constexpr int kPart = G == 16 ? 0 : 2 * 4 * NR * 32;   // per team: partial sums, two buffers
    static constexpr int kFixed = NT / 32 * kStage + kTeams * kPart;

    const CrcArgs& A;
    const SlabDev& sd;
    cg::cluster_group cl;
    C* b;        // own block rows, [row][NR][G]
    C* st;       // this warp's staged vectors
    C* part;     // this team's partial sums
    const C* F;
    int K, P, rank, lo, hi;   // own rows [lo, hi)
    int lane, p, sub, team;   // p: layer; sub: which part of a task this half warp / warp has
    int nc;                   // right-hand sides
    int kp, ki;               // columns within the slab's layers of this lane's part of a pair, of an inverse
    int buf = 0;

    C m[16], d[8];

    __device__ Crc(const CrcArgs& A_, const SlabDev& sd_, C* sm) : A(A_), sd(sd_), cl(cg::this_cluster()) {
        const int warp = threadIdx.x >> 5;
        lane = threadIdx.x & 31;
        team = warp / TW;
        p = lane % G;
        sub = G == 16 ? lane / 16 : warp % 4;
        st = sm + warp * kStage;
        part = sm + NT / 32 * kStage + team * kPart;
        b = sm + kFixed;
        F = (const C*)A.fac + sd.fac_off;
        K = A.n_tot;
        P = A.P;
        rank = (int)cl.block_rank();
        lo = min(K, rank * P);
        hi = min(K, lo + P);
        kp = max(0, min(16, sd.w - ca()));
        ki = max(0, min(8, sd.w - sub * 8));
    }
    // column c of the block row at position k, in whichever CTA owns it
    __device__ const C* row(int k, int c) const {
        const int q = k / P;
        const C* base = q == rank ? b : cl.map_shared_rank(b, q);
        return base + ((long long)(k - q * P) * NR + c) * G;
    }
    __device__ C* own(int k, int c) const { return b + ((long long)(k - lo) * NR + c) * G; }

    // entry (p, a) of a block or of its transpose
    __device__ static C ent(const C* M, int p, int a) { return TR ? M[p * G + a] : M[a * G + p]; }
    __device__ void load_inv(long long block) {
        const C* M = F + block * (G * G);
#pragma unroll
        for (int u = 0; u < 8; ++u) d[u] = !kSkip || u < ki ? ent(M, p, sub * 8 + u) : czero<C>();
    }
    // the part of a pair of blocks that this lane multiplies: the left
    // neighbour's block or the right one's, columns ca .. ca + 15
    __device__ int side() const { return G == 16 ? sub : sub >> 1; }
    __device__ int ca() const { return G == 16 ? 0 : (sub & 1) * 16; }
    __device__ void load_pair(const C* left, const C* right, bool hl, bool hr) {
        const bool has = side() ? hr : hl;
        const C* M = side() ? right : left;
#pragma unroll
        for (int u = 0; u < 16; ++u) m[u] = has && (!kSkip || u < kp) ? ent(M, p, ca() + u) : czero<C>();
    }
    // acc[c] = this lane's part of  (left) x_{kl} + (right) x_{kr}
    __device__ void pair(int kl, int kr, bool hl, bool hr, C (&acc)[NR]) {
        const bool has = side() ? hr : hl;
        const int kn = side() ? kr : kl;
        C* s = st + (G == 16 ? sub * NR * XS : 0);
        __syncwarp();
        if (G == 16 || lane < 16) {
#pragma unroll
            for (int c = 0; c < NR; ++c)
                if (c < nc) s[c * XS + (lane & 15)] = has ? row(kn, c)[ca() + (lane & 15)] : czero<C>();
        }
        __syncwarp();
#pragma unroll
        for (int c = 0; c < NR; ++c) {
            acc[c] = czero<C>();
            if (c < nc) {
                C s1 = czero<C>();
#pragma unroll
                for (int u = 0; u < 16; u += 2) {
                    if (kSkip && u >= kp) break;
                    acc[c] = cfma(m[u], s[c * XS + u], acc[c]);
                    s1 = cfma(m[u + 1], s[c * XS + u + 1], s1);
                }
                acc[c] = acc[c] + s1;
            }
        }
    }
    // acc[c] = this lane's part of  D^{-1} v  (v: every lane of the team holds entry p)
    __device__ void inv(const C (&v)[NR], C (&acc)[NR]) {
        __syncwarp();
        if (p / 8 == sub || G == 16) {
            if (G == 16) {
                if (p / 8 == sub)
#pragma unroll
                    for (int c = 0; c < NR; ++c) st[sub * NR * XS + c * XS + (p & 7)] = v[c];
            } else {
#pragma unroll
                for (int c = 0; c < NR; ++c) st[c * XS + (p & 7)] = v[c];
            }
        }
        __syncwarp();
        const C* s = st + (G == 16 ? sub * NR * XS : 0);
#pragma unroll
        for (int c = 0; c < NR; ++c) {
            acc[c] = czero<C>();
            if (c < nc) {
                C s1 = czero<C>();
#pragma unroll
                for (int u = 0; u < 8; u += 2) {
                    if (kSkip && u >= ki) break;
                    acc[c] = cfma(d[u], s[c * XS + u], acc[c]);
                    s1 = cfma(d[u + 1], s[c * XS + u + 1], s1);
                }
                acc[c] = acc[c] + s1;
            }
        }
    }
    // the parts of a task summed: afterwards every lane holds entry p
    __device__ void combine(C (&acc)[NR]) {
        if constexpr (G == 16) {
#pragma unroll
            for (int c = 0; c < NR; ++c) acc[c] = acc[c] + shfl_xor_c(acc[c], 16);
        } else {
            C* q = part + buf * (4 * NR * 32);   // two buffers: the other one may still be read
            buf ^= 1;
#pragma unroll
            for (int c = 0; c < NR; ++c) q[(sub * NR + c) * 32 + lane] = acc[c];
            asm volatile("bar.sync %0, 128;" ::"r"(team + 1) : "memory");
#pragma unroll
            for (int c = 0; c < NR; ++c)
                acc[c] = (q[c * 32 + lane] + q[(NR + c) * 32 + lane]) +
                         (q[(2 * NR + c) * 32 + lane] + q[(3 * NR + c) * 32 + lane]);
        }
    }
    __device__ bool writer() const { return sub == 0; }
    __device__ void get_own(int k, C (&v)[NR]) const {
#pragma unroll
        for (int c = 0; c < NR; ++c) v[c] = own(k, c)[p];
    }
    // (all lanes of the team have read the row: a combine lies between)
    __device__ void put(int k, const C (&v)[NR]) const {
        if (writer())
#pragma unroll
            for (int c = 0; c < NR; ++c) own(k, c)[p] = v[c];
    }

    // rows j = first + 2 i of level l (first = 0: even, 1: odd) that this CTA owns
    __device__ void range(int l, int first, int& i0, int& i1) const {
        auto lower = [&](int pos) {   // least i with (first + 2 i) << l >= pos
            const int j = (pos + (1 << l) - 1) >> l;
            return max(0, (j - first + 1) >> 1);
        };
        i0 = lower(lo);
        i1 = lower(hi);
    }

    // tridiagonal couplings of level 0: this lane's part (side 0: left
    // neighbour, 1: right) of  C x_{k-1} + B x_{k+1}  from the bands
    __device__ void band(const C* bl, const C* br, bool hl, bool hr, int k, C (&acc)[NR]) const {
#pragma unroll
        for (int c = 0; c < NR; ++c) acc[c] = czero<C>();
        const bool one = G == 16 || (sub & 1) == 0;   // two of the four warps of a 32-wide row
        const bool has = (side() ? hr : hl) && one;
        if (!has) return;
        const C* bd = side() ? br : bl;
#pragma unroll
        for (int da = -1; da <= 1; ++da) {
            const int a = TR ? p - da : p + da;
            if (a < 0 || a >= G) continue;
            const C cv = bd[(da + 1) * G + (TR ? a : p)];
#pragma unroll
            for (int c = 0; c < NR; ++c)
                if (c < nc) acc[c] = cfma(cv, row(side() ? k + 1 : k - 1, c)[a], acc[c]);
        }
    }

    __device__ void rhs(int i, int r0) {
        const int na = sd.na, w = sd.w;
        const long long nt2 = (long long)K * K;
        for (int e = threadIdx.x; e < (hi - lo) * NR * G; e += NT) {
            const int pp = e % G, c = (e / G) % NR, k = lo + e / (G * NR), r = r0 + c;
            C v = czero<C>();
            if (pp < w && c < nc) {
                const long long vec = (long long)K * A.R;
                const C* lam = (const C*)A.lam;
                const C* phi = (const C*)A.phi;
                if (!TR) {
                    if (pp >= na && pp <= sd.ll) v = ((const C*)A.f)[(long long)r * nt2 + (long long)k * K + sd.s + A.b + (pp - na)];
                } else {
                    const int x1 = sd.s + (pp - na), i2 = k - A.b;
                    if (pp >= na && x1 >= 1 && x1 <= A.n && i2 >= 1 && i2 <= A.n)
                        v = to_c<C>(A.yin[(long long)r * A.n * A.n + (long long)(x1 - 1) * A.n + (i2 - 1)]);
                }
                if (MODE == CRC_E && pp == na && i > 0) {   // the left neighbour's coupling
                    const SlabDev& so = TR ? A.slabs[i - 1] : sd;
                    const C* cf = (const C*)A.coef + so.coef_off;
                    for (int dk = -1; dk <= 1; ++dk) {
                        const int kk = TR ? k - dk : k + dk;
                        if (kk < 0 || kk >= K) continue;
                        const C cv = TR ? cf[(long long)kk * so.cstride + (so.w - 1) * 9 + 6 + dk + 1]
                                        : cf[(long long)k * so.cstride + pp * 9 + dk + 1];
                        const C xv = lam[(long long)(i - 1) * vec + (long long)kk * A.R + r];
                        v = cfma(mk(-cv.x, -cv.y), xv, v);
                    }
                }
                if (MODE == CRC_E && pp == sd.ll && i < A.n_slabs - 1) {   // the right neighbour's
                    const SlabDev& so = TR ? A.slabs[i + 1] : sd;
                    const C* cf = (const C*)A.coef + so.coef_off;
                    for (int dk = -1; dk <= 1; ++dk) {
                        const int kk = TR ? k - dk : k + dk;
                        if (kk < 0 || kk >= K) continue;
                        const C cv = TR ? cf[(long long)kk * so.cstride + so.na * 9 + dk + 1]
                                        : cf[(long long)k * so.cstride + pp * 9 + 6 + dk + 1];
                        const C xv = phi[(long long)(i + 1) * vec + (long long)kk * A.R + r];
                        v = cfma(mk(-cv.x, -cv.y), xv, v);
                    }
                }
            }
            b[e] = v;
        }
    }

    __device__ void solve(int i, int r0) {
        const CrcLv* lv = A.lv;
        const int L = A.L, Kh = (K + 1) / 2;
        const C* t0 = F + A.t0[G == 32];
        const C* p0 = F + A.p0[G == 32];
        int i0, i1;
        C v[NR], acc[NR];
        // ---- P0: y_o = D_o^{-1} b_o
        range(0, 1, i0, i1);
        int t = i0 + team;
        if (L > 0 && t < i1) load_inv(lv[0].dinv + t);
        rhs(i, r0);
        __syncthreads();
        if (L > 0)
            for (; t < i1; t += kTeams) {
                if (t != i0 + team) load_inv(lv[0].dinv + t);
                get_own(2 * t + 1, v);
                inv(v, acc);
                combine(acc);
                put(2 * t + 1, acc);
            }
        // ---- F(l); one row left: the top
        for (int l = 0; l < L; ++l) {
            const int Kl = lv[l].K;
            range(l, 0, i0, i1);
            t = i0 + team;
            auto load = [&](int t_) {
                const int e = 2 * t_;
                if (l > 0) {
                    if (TR)
                        load_pair(F + (lv[l].dcdb + 2LL * (t_ - 1) + 1) * (G * G), F + (lv[l].dcdb + 2LL * t_) * (G * G),
                                  e >= 1, e + 1 < Kl);
                    else
                        load_pair(F + (lv[l].cbe + 2LL * t_) * (G * G), F + (lv[l].cbe + 2LL * t_ + 1) * (G * G), e >= 1,
                                  e + 1 < Kl);
                }
                if (l + 1 == L) load_inv(lv[L].dinv);
                else if (!TR && (t_ & 1)) load_inv(lv[l + 1].dinv + (t_ >> 1));
            };
            cluster_arrive();
            if (t < i1) load(t);
            cluster_wait();
            for (; t < i1; t += kTeams) {
                if (t != i0 + team) load(t);
                const int e = 2 * t, k = e << l;
                const bool hl = e >= 1, hr = e + 1 < Kl;
                if (l == 0) {
                    const C *bl, *br;
                    if (TR) {
                        bl = t0 + ((long long)Kh + t - 1) * 6 * G + 3 * G;
                        br = t0 + ((long long)Kh + t) * 6 * G;
                    } else {
                        bl = t0 + (long long)t * 6 * G;
                        br = bl + 3 * G;
                    }
                    band(bl, br, hl, hr, k, acc);
                } else {
                    pair((e - 1) << l, (e + 1) << l, hl, hr, acc);
                }
                get_own(k, v);
                combine(acc);
#pragma unroll
                for (int c = 0; c < NR; ++c) v[c] = v[c] - acc[c];
                if (l + 1 == L || (!TR && (t & 1))) {
                    inv(v, acc);
                    combine(acc);
                    put(k, acc);
                } else {
                    put(k, v);
                }
            }
        }
        if (L == 0) {   // a single block row
            if (lo == 0 && team == 0) {
                load_inv(lv[0].dinv);
                get_own(0, v);
                inv(v, acc);
                combine(acc);
                put(0, acc);
            }
        }
        // ---- B(l)
        for (int l = L - 1; l >= 1; --l) {
            const int Kl = lv[l].K;
            range(l, 1, i0, i1);
            t = i0 + team;
            auto load = [&](int t_) {
                const int j = 2 * t_ + 1;
                if (TR) {
                    load_pair(F + (lv[l].cbe + 2LL * t_ + 1) * (G * G), F + (lv[l].cbe + 2LL * (t_ + 1)) * (G * G), true,
                              j + 1 < Kl);
                    load_inv(lv[l].dinv + t_);
                } else {
                    load_pair(F + (lv[l].dcdb + 2LL * t_) * (G * G), F + (lv[l].dcdb + 2LL * t_ + 1) * (G * G), true,
                              j + 1 < Kl);
                }
            };
            cluster_arrive();
            if (t < i1) load(t);
            cluster_wait();
            for (; t < i1; t += kTeams) {
                if (t != i0 + team) load(t);
                const int j = 2 * t + 1, k = j << l;
                pair((j - 1) << l, (j + 1) << l, true, j + 1 < Kl, acc);
                get_own(k, v);
                combine(acc);
#pragma unroll
                for (int c = 0; c < NR; ++c) v[c] = v[c] - acc[c];
                if (TR) {
                    inv(v, acc);
                    combine(acc);
                    put(k, acc);
                } else {
                    put(k, v);
                }
            }
        }
        // ---- B(0)
        if (L > 0) {
            constexpr bool kTwo = MODE == CRC_A && !TR;   // layers na and ll only
            range(0, 1, i0, i1);
            t = i0 + team;
            cluster_arrive();
            if (!kTwo && t < i1) load_inv(lv[0].dinv + t);
            cluster_wait();
            for (; t < i1; t += kTeams) {
                if (!kTwo && t != i0 + team) load_inv(lv[0].dinv + t);
                const int k = 2 * t + 1;
                const C *bl, *br;
                if (TR) {
                    bl = t0 + (long long)t * 6 * G + 3 * G;
                    br = t0 + (long long)(t + 1) * 6 * G;
                } else {
                    bl = t0 + ((long long)Kh + t) * 6 * G;
                    br = bl + 3 * G;
                }
                band(bl, br, true, k + 1 < K, k, acc);
                get_own(k, v);
                combine(acc);
                C dv[NR];
                if constexpr (!kTwo) {
                    inv(acc, dv);
                    combine(dv);
#pragma unroll
                    for (int c = 0; c < NR; ++c) v[c] = v[c] - dv[c];
                    put(k, v);
                } else {
                    const C* pr = p0 + (long long)t * 2 * G;
                    const C q0 = pr[p], q1 = pr[G + p];
#pragma unroll
                    for (int c = 0; c < NR; ++c) {
                        C d0 = cfma(q0, acc[c], czero<C>()), d1 = cfma(q1, acc[c], czero<C>());
#pragma unroll
                        for (int off = G / 2; off > 0; off >>= 1) {
                            d0 = d0 + shfl_xor_c(d0, off);
                            d1 = d1 + shfl_xor_c(d1, off);
                        }
                        if (writer() && p == sd.na) own(k, c)[p] = v[c] - d0;
                        if (writer() && p == sd.ll && sd.ll != sd.na) own(k, c)[p] = v[c] - d1;
                    }
                }
            }
        }
        cluster_arrive();   // every read of this CTA's rows is done before it leaves
        cluster_wait();
        __syncthreads();
        // ---- outputs
        const int rows = hi - lo;
        if (MODE == CRC_A) {
            C* af = (C*)A.a_first;
            C* al = (C*)A.a_last;
            const long long base = (long long)i * K * A.R + r0;
            for (int e = threadIdx.x; e < rows * nc; e += NT) {
                const int c = e % nc, k = lo + e / nc;
                af[base + (long long)k * A.R + c] = own(k, c)[sd.na];
                al[base + (long long)k * A.R + c] = own(k, c)[sd.ll];
            }
        } else if (TR || A.y_grid) {   // layers fastest
            const long long nt2 = (long long)K * K;
            for (int e = threadIdx.x; e < sd.nl * rows * nc; e += NT) {
                const int pl = e % sd.nl, k = lo + (e / sd.nl) % rows, c = e / (sd.nl * rows);
                const C x = own(k, c)[sd.na + pl];
                const long long o = (long long)(r0 + c) * nt2 + (long long)k * K + sd.s + A.b + pl;
                if (TR) ((C*)A.X)[o] = x;
                else A.y[o] = to_d(x);
            }
        } else {
            for (int e = threadIdx.x; e < sd.nl * rows * nc; e += NT) {
                const int k = lo + e % rows, pl = (e / rows) % sd.nl, c = e / (rows * sd.nl);
                const int x1 = sd.s + pl, i2 = k - A.b;
                if (x1 >= 1 && x1 <= A.n && i2 >= 1 && i2 <= A.n)
                    A.y[(long long)(r0 + c) * A.n * A.n + (long long)(x1 - 1) * A.n + (i2 - 1)] = to_d(own(k, c)[sd.na + pl]);
            }
        }
    }
};

template <typename T, int MODE, bool TR, int G, int NR, int NT>
__global__ void __launch_bounds__(NT, 512 / NT) cr_cluster_kernel(const __grid_constant__ CrcArgs A) {
    extern __shared__ __align__(128) unsigned char crc_smem[];
    const int i = A.slab0 + blockIdx.y;
    __shared__ SlabDev sd;
    if (threadIdx.x == 0) sd = A.slabs[i];
    __syncthreads();
    Crc<T, MODE, TR, G, NR, NT> S(A, sd, reinterpret_cast<cx<T>*>(crc_smem));
    const int r0 = (int)(blockIdx.x / S.cl.num_blocks()) * NR;
    S.nc = min(NR, A.R - r0);
    S.solve(i, r0);
}

constexpr size_t kCrcSmem = size_t(220) * 1024;

// Clusters of a pass's slabs of one width.
int crc_clusters(const lss_ctx* c, int ldw, int R, int nr) {
    int total = 0;   // (its runs share the SMs)
    for (const SlabDev& q : c->slabs) total += q.ldw == ldw;
    return total * ((R + nr - 1) / nr);
}
// Clusters of cl CTAs that the GPU holds at once, a CTA per SM: a cluster lies in
// one GPC (18 to 20 SMs), so 16 clusters of 8 or 36 of 4 fill it.
bool crc_one_wave(const lss_ctx* c, long long clusters, int cl) {
    return clusters * cl <= (cl == 8 ? c->num_sms * 6 / 7 : c->num_sms * 19 / 20);
}

template <typename T, int MODE, bool TR, int G, int NR, int NT>
int launch(lss_ctx* c, CrcArgs A, int nsl, cudaStream_t s) {
    using S = Crc<T, MODE, TR, G, NR, NT>;
    auto kern = cr_cluster_kernel<T, MODE, TR, G, NR, NT>;
    const int K = A.n_tot, groups = (A.R + NR - 1) / NR;
    const long long N = crc_clusters(c, G, A.R, NR);
    auto smem = [&](int P) { return sizeof(cx<T>) * ((size_t)S::kFixed + (size_t)P * NR * G); };
    // Cluster size.  More CTAs per slab shorten the chain of the low levels but
    // make the barriers of the high ones dearer, and once the pass fills the
    // SMs they add nothing.  Passes A + E of one application, us, 1 / 2 / 4 CTAs
    // per 16-wide slab: FP64 n = 64, 2 right-hand sides 300 / 200 / 330,
    // n = 181, 1 680 / 410 / 400, n = 256, 8 3170 / 3110 / 3350; mixed n = 256,
    // 1 (two fronts) 320 / 200 / 245, n = 512, 1 600 / 630 / 410 (few CTAs of
    // many rows lack loads in flight: at least two CTAs where 128 rows remain).
    // A 32-wide slab is four times the work.  Where they are few, theirs is the
    // longest chain: 8 CTAs as long as all clusters run at once, then 4 (FP64
    // n = 256, 1: 1000 us, with 4 1070 and with 2 1490; clusters of 16 take longer
    // in mixed precision, n = 256: 360 us against 200).  More clusters than that
    // come in waves, and two CTAs of 256 threads share an SM to overlap their
    // barriers, in clusters of 4, of 2 once the SMs are full without (P, ms, 512
    // threads with 1 / 2 / 4 / 8 CTAs | 256 threads: FP64, all slabs 20 layers wide,
    // n = 64, 6 right-hand sides 1.01 / 0.65 / 0.71 / 0.88 | 1.12 / 0.71 / 0.62 / 0.69,
    // 40: 3.12 / 2.92 / 3.36 / 4.92 | 3.11 / 2.77 / 2.87 / 3.44, n = 256, 10:
    // 8.1 / 7.2 / 7.7 / 9.9 | 7.0 / 7.0 / 6.5 / 7.3; mixed, n = 64, 3:
    // 0.36 / 0.24 / 0.18 / 0.15, n = 100, 40: 0.86 / 0.90 / 0.97 / 1.17 | 0.83 / 0.83 / 0.84 / 0.93).
    // Beside a block LU of the other slabs the SMs are not theirs alone: 4 CTAs
    // of more than 32 rows each (P, mixed, ms, with 8 / 4 / 2 CTAs: n = 64, 64
    // right-hand sides 1.47 / 1.47 / 1.39, n = 128, 64 3.31 / 3.08 / 3.07 and 96
    // 1.36 / 1.30 / 1.43, n = 256, 32 2.13 / 1.95 / 1.95).
    int cl = 1;
    if (G == 16) {
        while (cl < 4 && K > 4 * cl && (N * cl < c->num_sms * 3 / 4 || K / (2 * cl) >= 128))
            cl *= 2;
    } else if (A.beside) {
        while (cl < 4 && K > 64 * cl && N * cl < c->num_sms) cl *= 2;
    } else {
        cl = NT == 256 ? (N <= 2 * c->num_sms ? 4 : 2) : crc_one_wave(c, N, 8) ? 8 : 4;
        while (cl > 1 && K <= 2 * cl) cl /= 2;
    }
    // two CTAs of 256 threads per SM; past 8 CTAs only where the rows fit no other way
    while (cl < 8 && smem((K + cl - 1) / cl) > (NT == 256 ? kCrcSmem / 2 : kCrcSmem)) cl *= 2;
    if (smem((K + cl - 1) / cl) > kCrcSmem) cl = 16;
    A.P = (K + cl - 1) / cl;
    const size_t sh = smem(A.P);
    if (sh > kCrcSmem) return lss_fail(c, LSS_ERR_UNSUPPORTED, "slab solve: a slab's rows do not fit a cluster's shared memory");
    {
        std::lock_guard<std::mutex> lock(lss_config_mutex());
        long long& cfg = lss_dev_cache((const void*)kern, 0);
        if (!cfg) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCrcSmem);
            if (!e) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e) return lss_check_cuda(c, e, "slab solve attribute");
            cfg = 1;
        }
    }
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3(cl * groups, nsl);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = sh;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return lss_check_cuda(c, cudaLaunchKernelEx(&cfg, kern, A), "slab solve launch");
}

template <typename T, int MODE, bool TR, int NR>
int launch_wide(lss_ctx* c, const CrcArgs& A, int nsl, cudaStream_t s) {
    if (!A.beside && !crc_one_wave(c, crc_clusters(c, 32, A.R, NR), 4)) return launch<T, MODE, TR, 32, NR, 256>(c, A, nsl, s);
    return launch<T, MODE, TR, 32, NR, 512>(c, A, nsl, s);
}

template <typename T, int MODE, bool TR>
int dispatch(lss_ctx* c, const CrcArgs& A, int nsl, int ldw, cudaStream_t s) {
    if constexpr (!TR)
        if (ldw == 16 && lss_cr_cluster_rhs(c, A.R) == 2) return launch<T, MODE, TR, 16, 2, 256>(c, A, nsl, s);
    if constexpr (sizeof(T) == 4)
        if (A.R > 1 && c->n_tot <= 1400)   // (their rows of a 32-wide slab fit 8 CTAs)
            return ldw == 16 ? launch<T, MODE, TR, 16, 4, 256>(c, A, nsl, s) : launch_wide<T, MODE, TR, 4>(c, A, nsl, s);
    return ldw == 16 ? launch<T, MODE, TR, 16, 1, 256>(c, A, nsl, s) : launch_wide<T, MODE, TR, 1>(c, A, nsl, s);
}

}  // namespace

// Single precision is bound by the factor stream and by latency: four
// right-hand sides share every factor entry (n = 512, 12: 7.0 against 12.3 ms
// of pass A per solve).  Double precision is bound by the FP64 pipe: one per
// cluster leaves more warps to fill it (n = 256, 8: 1.53 against 2.16 ms with four).
int lss_cr_cluster_rhs(const lss_ctx* c, int R) {
    if (R > 1 && c->tune.solve_nr == 2) return 2;
    return c->prec == LSS_MIXED && R > 1 && c->n_tot <= 1400 ? 4 : 1;
}

int lss_cr_cluster(lss_ctx* c, int mode, bool transpose, CrcArgs A, int s0, int nsl, int ldw, cudaStream_t s) {
    A.slabs = c->d_slabs;
    A.n_slabs = c->n_slabs;
    A.n_tot = c->n_tot;
    A.n = c->n;
    A.b = c->b;
    A.fac = c->fac;
    A.coef = c->coef;
    A.slab0 = s0;
    A.L = cr_levels(c->n_tot);
    if (A.L + 1 > kCrcLevels) return LSS_ERR_UNSUPPORTED;
    for (int l = 0; l <= A.L; ++l) {
        const CrLevelOffs o = cr_level(c->n_tot, l);
        A.lv[l] = CrcLv{o.K, (int)o.dinv, (int)o.cbe, (int)o.dcdb};
    }
    for (int w = 0; w < 2; ++w) {
        const int g = w ? 32 : 16;
        A.t0[w] = cr_t0_off(c->n_tot, g * g);
        A.p0[w] = cr_p0_off(c->n_tot, g * g, g);
    }
    const bool d = c->prec == LSS_FP64;
    if (transpose) {
        if (mode == CRC_A)
            return d ? dispatch<double, CRC_A, true>(c, A, nsl, ldw, s) : dispatch<float, CRC_A, true>(c, A, nsl, ldw, s);
        return d ? dispatch<double, CRC_E, true>(c, A, nsl, ldw, s) : dispatch<float, CRC_E, true>(c, A, nsl, ldw, s);
    }
    if (mode == CRC_A)
        return d ? dispatch<double, CRC_A, false>(c, A, nsl, ldw, s) : dispatch<float, CRC_A, false>(c, A, nsl, ldw, s);
    return d ? dispatch<double, CRC_E, false>(c, A, nsl, ldw, s) : dispatch<float, CRC_E, false>(c, A, nsl, ldw, s);
}
