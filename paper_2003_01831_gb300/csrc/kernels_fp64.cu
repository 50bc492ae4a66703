// FP64 kernels of the AFQMC walker step: batched complex GEMM (its tensor-core form is in
// gemm_slices.cu), Gauss-Jordan
// inverse / log-det, trace epilogue, local energy and force bias, Philox fields,
// phaseless weights, Gram-Schmidt re-orthonormalisation, estimator reduction.
//
// The formulas follow the phaseless algorithm the paper cites in Sec. V (Zhang &
// Krakauer 2003; Motta & Zhang 2018) for the Hamiltonian of Sec. V, Eq. (1) with
// the Cholesky factorisation of Eq. (3).  All reductions run in a fixed order for
// a fixed launch shape, so results are bitwise reproducible run to run.
#include <cuda_runtime.h>
#include <float.h>
#include <math.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "ffc.cuh"
#include "kernels_fp64.cuh"
#include "kernels_tc.cuh"

namespace afqmc {

namespace {

constexpr int kThreads = 256;

// Fixed-order block reduction of a complex value (all threads get the result).
__device__ cplx block_sum(cplx v, cplx* sh) {
    const int t = threadIdx.x;
    sh[t] = v;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (t < s) sh[t] = sh[t] + sh[t + s];
        __syncthreads();
    }
    cplx r = sh[0];
    __syncthreads();
    return r;
}

__device__ double block_sum_d(double v, double* sh) {
    const int t = threadIdx.x;
    sh[t] = v;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (t < s) sh[t] += sh[t + s];
        __syncthreads();
    }
    double r = sh[0];
    __syncthreads();
    return r;
}

__device__ __forceinline__ bool finite_c(cplx a) { return isfinite(a.re) && isfinite(a.im); }

// ------------------------------------------------------------------ batched GEMM
template <bool R>
struct Elem {
    using T = cplx;
};
template <>
struct Elem<true> {
    using T = double;
};

__device__ __forceinline__ void load_elem(double& dst, const void* base, int64_t idx, bool conj) {
    dst = static_cast<const double*>(base)[idx];
}
__device__ __forceinline__ void load_elem(cplx& dst, const void* base, int64_t idx, bool conj) {
    const double2 v = static_cast<const double2*>(base)[idx];
    dst.re = v.x;
    dst.im = conj ? -v.y : v.y;
}
__device__ __forceinline__ void zero_elem(double& d) { d = 0.0; }
__device__ __forceinline__ void zero_elem(cplx& d) { d = cplx{0.0, 0.0}; }

__device__ __forceinline__ void mac(cplx& acc, double a, double b) { acc.re = fma(a, b, acc.re); }
__device__ __forceinline__ void mac(cplx& acc, double a, cplx b) {
    acc.re = fma(a, b.re, acc.re);
    acc.im = fma(a, b.im, acc.im);
}
__device__ __forceinline__ void mac(cplx& acc, cplx a, double b) {
    acc.re = fma(a.re, b, acc.re);
    acc.im = fma(a.im, b, acc.im);
}
__device__ __forceinline__ void mac(cplx& acc, cplx a, cplx b) { cfma(acc, a, b); }

// Tiles of TS x TS outputs (TS = 64: 4 x 4 per thread; TS = 32: 2 x 2 per thread, for the small
// blocks of few-electron systems, e.g. the 32 x 32 T_n = Ltilde_n Theta blocks), K in steps of
// 512 / TS, so each operand tile holds 512 elements either way.
template <bool AR, bool BR, int TS>
__global__ void __launch_bounds__(kThreads) zgemm_kernel(GemmArgs g) {
    constexpr int BM = TS, BN = TS, BK = 512 / TS, R = TS / 16;
    using TA = typename Elem<AR>::T;
    using TB = typename Elem<BR>::T;
    __shared__ TA As[BK][BM + 1];
    __shared__ TB Bs[BK][BN + 1];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int64_t nbatch = (int64_t)g.nb0 * g.nb1 * g.nb2;
    for (int64_t b = blockIdx.z; b < nbatch; b += gridDim.z) {
        const int64_t b0 = b / ((int64_t)g.nb1 * g.nb2);
        const int64_t r12 = b % ((int64_t)g.nb1 * g.nb2);
        const int64_t b1 = r12 / g.nb2, b2 = r12 % g.nb2;
        const int64_t offA = b0 * g.A.s0 + b1 * g.A.s1 + b2 * g.A.s2;
        const int64_t offB = b0 * g.B.s0 + b1 * g.B.s1 + b2 * g.B.s2;
        cplx acc[R][R];
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < R; ++j) acc[i][j] = cplx{0.0, 0.0};

        for (int k0 = 0; k0 < g.k; k0 += BK) {
            for (int e = threadIdx.x; e < BM * BK; e += kThreads) {
                int r, kk;
                if (g.A.op == OP_N) { r = e / BK; kk = e % BK; }
                else { kk = e / BM; r = e % BM; }
                const int gr = m0 + r, gk = k0 + kk;
                TA v;
                zero_elem(v);
                if (gr < g.m && gk < g.k) {
                    const int64_t idx = offA + (g.A.op == OP_N ? (int64_t)gr * g.A.ld + gk
                                                                : (int64_t)gk * g.A.ld + gr);
                    load_elem(v, g.A.ptr, idx, g.A.op == OP_C);
                }
                As[kk][r] = v;
            }
            for (int e = threadIdx.x; e < BN * BK; e += kThreads) {
                int c, kk;
                if (g.B.op == OP_N) { kk = e / BN; c = e % BN; }
                else { c = e / BK; kk = e % BK; }
                const int gc = n0 + c, gk = k0 + kk;
                TB v;
                zero_elem(v);
                if (gc < g.n && gk < g.k) {
                    const int64_t idx = offB + (g.B.op == OP_N ? (int64_t)gk * g.B.ld + gc
                                                                : (int64_t)gc * g.B.ld + gk);
                    load_elem(v, g.B.ptr, idx, g.B.op == OP_C);
                }
                Bs[kk][c] = v;
            }
            __syncthreads();
#pragma unroll
            for (int kk = 0; kk < BK; ++kk) {
                TA a[R];
                TB bv[R];
#pragma unroll
                for (int i = 0; i < R; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
                for (int j = 0; j < R; ++j) bv[j] = Bs[kk][tx + 16 * j];
#pragma unroll
                for (int i = 0; i < R; ++i)
#pragma unroll
                    for (int j = 0; j < R; ++j) mac(acc[i][j], a[i], bv[j]);
            }
            __syncthreads();
        }
        const bool use_beta = (g.beta.re != 0.0 || g.beta.im != 0.0);
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int r = m0 + ty + 16 * i;
            if (r >= g.m) continue;
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const int c = n0 + tx + 16 * j;
                if (c >= g.n) continue;
                cplx v = g.alpha * acc[i][j];
                cplx* cp = g.C + b0 * g.sc0 + b1 * g.sc1 + b2 * g.sc2 + (int64_t)r * g.ldc + c;
                if (use_beta) v = v + g.beta * (*cp);
                *cp = v;
                if (g.D) {
                    cplx* dp = g.D + b0 * g.sd0 + b1 * g.sd1 + b2 * g.sd2 + (int64_t)r * g.ldd + c;
                    *dp = *dp + v;
                }
            }
        }
    }
}

// One output per thread, or by P neighbouring threads that share its contraction, for products too
// small to fill tiles (few electrons, few walkers): a 64 x 64 or 32 x 32 tile does its padding's
// multiply-adds too, on one SM (25 us for a 24 x 5 output and K = 24), where this spreads the outputs
// alone over all SMs.  Neighbouring outputs run along a row, so A is a broadcast and B coalesced for
// op N.  An FP64 instruction holds its scheduler's pipe for 64 cycles and its result takes 200, so
// P > 1 takes fewer steps of the chain as long as it finds idle schedulers (zgemm_form): 9.2 us
// with one thread for 16 x 24 x 5 outputs and K = 24, 4.0 with eight.
constexpr int kSmallT = 64;
template <int P>
struct SmallSum {   // P = 1: zgemm_kernel's order of sums; P > 1: the products of a complex one apart
    cplx a{0.0, 0.0}, b{0.0, 0.0};
    template <class X, class Y>
    __device__ __forceinline__ void add(const X& x, const Y& y) {
        if constexpr (P > 1 && std::is_same<X, cplx>::value && std::is_same<Y, cplx>::value) {
            a.re = fma(x.re, y.re, a.re);
            b.re = fma(x.im, y.im, b.re);
            a.im = fma(x.re, y.im, a.im);
            b.im = fma(x.im, y.re, b.im);
        } else {
            mac(a, x, y);
        }
    }
    __device__ __forceinline__ cplx total() const { return P > 1 ? cplx{a.re - b.re, a.im + b.im} : a; }
};
template <bool AR, bool BR, int P>
__global__ void __launch_bounds__(kSmallT) zgemm_small_kernel(GemmArgs g, uint32_t outputs) {
    using TA = typename Elem<AR>::T;
    using TB = typename Elem<BR>::T;
    const uint32_t id = (blockIdx.x * kSmallT + threadIdx.x) / P;
    const int part = threadIdx.x % P;
    const unsigned all = __ballot_sync(0xffffffffu, id < outputs);   // whole groups of P
    if (id >= outputs) return;
    const uint32_t n = (uint32_t)g.n, m = (uint32_t)g.m, nb1 = (uint32_t)g.nb1, nb2 = (uint32_t)g.nb2;
    const uint32_t rc = id / n, b = rc / m, b01 = b / nb2;
    const int c = (int)(id - rc * n), r = (int)(rc - b * m);
    const int64_t b2 = b - b01 * nb2, b0 = b01 / nb1, b1 = b01 - b0 * nb1;
    const int64_t sa = (g.A.op == OP_N ? 1 : g.A.ld) * (int64_t)P, sb = (g.B.op == OP_N ? g.B.ld : 1) * (int64_t)P;
    int64_t ia = b0 * g.A.s0 + b1 * g.A.s1 + b2 * g.A.s2 + (int64_t)r * (g.A.op == OP_N ? g.A.ld : 1) + part * (sa / P);
    int64_t ib = b0 * g.B.s0 + b1 * g.B.s1 + b2 * g.B.s2 + (int64_t)c * (g.B.op == OP_N ? 1 : g.B.ld) + part * (sb / P);
    SmallSum<P> acc;
    const bool ca = g.A.op == OP_C, cb = g.B.op == OP_C;
    constexpr int U = P == 1 ? 8 : 4;   // loads of each operand in flight
    int k = part;
    for (; k + (U - 1) * P < g.k; k += U * P) {
        TA a[U];
        TB v[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            load_elem(a[q], g.A.ptr, ia + q * sa, ca);
            load_elem(v[q], g.B.ptr, ib + q * sb, cb);
        }
#pragma unroll
        for (int q = 0; q < U; ++q) acc.add(a[q], v[q]);
        ia += U * sa;
        ib += U * sb;
    }
#pragma unroll
    for (int q = 0; q < U - 1; ++q) {   // the rest, loads in flight too
        if (k + q * P >= g.k) break;
        TA a;
        TB v;
        load_elem(a, g.A.ptr, ia + q * sa, ca);
        load_elem(v, g.B.ptr, ib + q * sb, cb);
        acc.add(a, v);
    }
    cplx sum = acc.total();
#pragma unroll
    for (int o = P / 2; o > 0; o >>= 1) {
        sum.re += __shfl_xor_sync(all, sum.re, o);
        if (!AR || !BR) sum.im += __shfl_xor_sync(all, sum.im, o);
    }
    if (part != 0) return;
    cplx v = g.alpha * sum;
    cplx* cp = g.C + b0 * g.sc0 + b1 * g.sc1 + b2 * g.sc2 + (int64_t)r * g.ldc + c;
    if (g.beta.re != 0.0 || g.beta.im != 0.0) v = v + g.beta * (*cp);
    *cp = v;
    if (g.D) {
        cplx* dp = g.D + b0 * g.sd0 + b1 * g.sd1 + b2 * g.sd2 + (int64_t)r * g.ldd + c;
        *dp = *dp + v;
    }
}

// ------------------------------------------------------------------ Gauss-Jordan
constexpr int kGJU = 8;   // element updates in flight per thread
__global__ void __launch_bounds__(kThreads)
    gj_kernel(cplx* Sbase, int64_t stride, int N, cplx* logdet, int with_inverse, unsigned* flags) {
    extern __shared__ unsigned char smem_raw[];
    cplx* prow = reinterpret_cast<cplx*>(smem_raw);  // N (scaled pivot row)
    cplx* pcol = prow + N;                           // N (pivot column)
    int* perm = reinterpret_cast<int*>(pcol + N);    // N
    __shared__ double red_v[kThreads];
    __shared__ int red_i[kThreads];
    __shared__ int s_piv;
    __shared__ int s_singular;
    cplx* A = Sbase + (int64_t)blockIdx.x * stride;
    const int t = threadIdx.x;
    double logabs = 0.0, phase = 0.0;  // meaningful in thread 0
    if (t == 0) s_singular = 0;
    __syncthreads();
    for (int k = 0; k < N; ++k) {
        // pivot: max |re|+|im| over rows k..N-1 of column k, lowest index on ties
        // (warp shuffles, then one pass over the per-warp winners)
        double best = -1.0;
        int bi = N;
        for (int i = k + t; i < N; i += kThreads) {
            const double v = abs1(A[(int64_t)i * N + k]);
            if (v > best || (v != v && best == best)) { best = v; bi = i; }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const double v2 = __shfl_xor_sync(0xffffffffu, best, o);
            const int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
            if (v2 > best || (v2 == best && i2 < bi) || (v2 != v2 && best == best)) { best = v2; bi = i2; }
        }
        if ((t & 31) == 0) {
            red_v[t >> 5] = best;
            red_i[t >> 5] = bi;
        }
        __syncthreads();
        if (t == 0) {
            double bv = red_v[0];
            int bidx = red_i[0];
            for (int q = 1; q < kThreads / 32; ++q) {
                const double v2 = red_v[q];
                const int i2 = red_i[q];
                if (v2 > bv || (v2 == bv && i2 < bidx) || (v2 != v2 && bv == bv)) { bv = v2; bidx = i2; }
            }
            s_piv = bidx;
            if (!(bv > 0.0)) s_singular = (bv != bv) ? 2 : 1;
            perm[k] = bidx;
        }
        __syncthreads();
        if (s_singular) break;
        const int p = s_piv;
        if (p != k) {
            for (int j = t; j < N; j += kThreads) {
                const cplx a = A[(int64_t)k * N + j];
                A[(int64_t)k * N + j] = A[(int64_t)p * N + j];
                A[(int64_t)p * N + j] = a;
            }
            __syncthreads();
        }
        const cplx piv = A[(int64_t)k * N + k];
        const cplx inv = cdiv(cplx{1.0, 0.0}, piv);
        if (t == 0) {
            logabs += log(hypot(piv.re, piv.im));
            phase += atan2(piv.im, piv.re) + (p != k ? M_PI : 0.0);
        }
        for (int j = t; j < N; j += kThreads) {
            prow[j] = A[(int64_t)k * N + j] * inv;
            pcol[j] = A[(int64_t)j * N + k];
        }
        __syncthreads();
        // Element updates, kGJU per thread in flight: all loads are issued before any
        // arithmetic, so a thread waits on the memory system once per batch, not per element.
        if (with_inverse) {
            const int64_t NN = (int64_t)N * N;
            for (int64_t e0 = t; e0 < NN; e0 += (int64_t)kThreads * kGJU) {
                cplx v[kGJU];
#pragma unroll
                for (int u = 0; u < kGJU; ++u) {
                    const int64_t e = e0 + (int64_t)u * kThreads;
                    if (e < NN) v[u] = A[e];
                }
#pragma unroll
                for (int u = 0; u < kGJU; ++u) {
                    const int64_t e = e0 + (int64_t)u * kThreads;
                    if (e >= NN) continue;
                    const int i = (int)(e / N), j = (int)(e % N);
                    if (i == k) v[u] = (j == k) ? inv : prow[j];
                    else if (j == k) v[u] = cplx{0.0, 0.0} - pcol[i] * inv;
                    else cfma(v[u], cplx{0.0, 0.0} - pcol[i], prow[j]);
                    A[e] = v[u];
                }
            }
        } else {
            const int nr = N - k - 1;
            const int64_t nn = (int64_t)nr * nr;
            for (int64_t e0 = t; e0 < nn; e0 += (int64_t)kThreads * kGJU) {
                cplx v[kGJU];
#pragma unroll
                for (int u = 0; u < kGJU; ++u) {
                    const int64_t e = e0 + (int64_t)u * kThreads;
                    if (e < nn) v[u] = A[(int64_t)(k + 1 + e / nr) * N + k + 1 + e % nr];
                }
#pragma unroll
                for (int u = 0; u < kGJU; ++u) {
                    const int64_t e = e0 + (int64_t)u * kThreads;
                    if (e >= nn) continue;
                    const int i = k + 1 + (int)(e / nr), j = k + 1 + (int)(e % nr);
                    cfma(v[u], cplx{0.0, 0.0} - pcol[i], prow[j]);
                    A[(int64_t)i * N + j] = v[u];
                }
            }
        }
        __syncthreads();
    }
    if (s_singular) {
        if (t == 0) {
            logdet[blockIdx.x] = cplx{-INFINITY, 0.0};
            atomicOr(flags, s_singular == 2 ? FLAG_NONFINITE : FLAG_SINGULAR);
        }
        return;
    }
    if (with_inverse) {
        for (int k = N - 1; k >= 0; --k) {
            const int p = perm[k];
            if (p != k) {
                for (int i = t; i < N; i += kThreads) {
                    const cplx a = A[(int64_t)i * N + k];
                    A[(int64_t)i * N + k] = A[(int64_t)i * N + p];
                    A[(int64_t)i * N + p] = a;
                }
            }
            __syncthreads();
        }
    }
    if (t == 0) logdet[blockIdx.x] = cplx{logabs, atan2(sin(phase), cos(phase))};
}

// ------------------------------------------------------- Gauss-Jordan in shared memory
// The same elimination (pivot max |re|+|im|, lowest index on ties; physical row swaps; the
// in-place inverse with its column permutation undone at the end) with the matrix held on
// chip: one CTA for N <= kGJSmemOne, else a cluster of two CTAs that own alternate columns
// (column j lives in CTA j % 2 at local column j / 2) and exchange the pivot column and the
// pivot index through distributed shared memory, two cluster barriers per elimination step.
// FP64 throughput, not memory latency, then bounds the elimination.
constexpr int kGJSmemOne = 96;      // largest N done by one CTA (N^2 complex in shared memory)
constexpr int kGJSmemMax = 128;     // largest N done by the two-CTA cluster
constexpr int kGJT = 512;           // threads per CTA
// local columns per lane: COLS = ceil(H / 32) <= 3 (template parameter)

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// address of the same shared variable in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
    uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p)), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_peer_f64(uint32_t addr, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void st_peer_s32(uint32_t addr, int v) {
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

template <int C>
__device__ __forceinline__ void gj_sync() {
    if (C == 1) __syncthreads();
    else cluster_sync_all();
}

template <int C, int COLS>
__global__ void __launch_bounds__(kGJT)
    gj_smem_kernel(cplx* Sbase, int64_t stride, int N, cplx* logdet, int with_inverse, unsigned* flags) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int H = (N + C - 1) / C;                   // local columns
    cplx* A = reinterpret_cast<cplx*>(smem_raw);     // [N][H]
    cplx* pcol = A + (size_t)N * H;                  // pivot column (before this step's swap)
    cplx* prow = pcol + N;                           // scaled pivot row, local columns
    int* perm = reinterpret_cast<int*>(prow + H);    // pivot row of every step
    int* pos = perm + N;                             // final column of each stored column
    __shared__ double red_v[kGJT / 32];
    __shared__ int red_i[kGJT / 32];
    __shared__ int s_piv;
    __shared__ int s_singular;
    constexpr int R = COLS <= 2 ? 4 : 2;               // rows per warp in flight
    const int rank = C == 1 ? 0 : (int)cluster_rank();
    const int64_t mat = C == 1 ? blockIdx.x : blockIdx.x / C;
    cplx* G = Sbase + mat * stride;
    const int t = threadIdx.x;
    const int NH = N * H;
    // load my columns: global column j = c*C + rank
    for (int e = t; e < NH; e += kGJT) {
        const int i = e / H, c = e % H, j = c * C + rank;
        A[e] = j < N ? G[(int64_t)i * N + j] : cplx{0.0, 0.0};
    }
    if (t == 0) s_singular = 0;
    double logabs = 0.0, phase = 0.0;   // thread 0 of rank 0
    gj_sync<C>();
    for (int k = 0; k < N; ++k) {
        const int owner = k % C, lk = k / C;
        if (rank == owner) {
            double best = -1.0;
            int bi = N;
            for (int i = k + t; i < N; i += kGJT) {
                const double v = abs1(A[i * H + lk]);
                if (v > best || (v != v && best == best)) { best = v; bi = i; }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const double v2 = __shfl_xor_sync(0xffffffffu, best, o);
                const int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
                if (v2 > best || (v2 == best && i2 < bi) || (v2 != v2 && best == best)) { best = v2; bi = i2; }
            }
            if ((t & 31) == 0) { red_v[t >> 5] = best; red_i[t >> 5] = bi; }
            // the pivot column (pre-swap) to both CTAs
            for (int i = t; i < N; i += kGJT) {
                const cplx v = A[i * H + lk];
                pcol[i] = v;
                if (C > 1) {
                    const uint32_t a = peer_addr(&pcol[i], (uint32_t)(owner ^ 1));
                    st_peer_f64(a, v.re);
                    st_peer_f64(a + 8, v.im);
                }
            }
            __syncthreads();
            if (t == 0) {
                double bv = red_v[0];
                int bidx = red_i[0];
                for (int q = 1; q < kGJT / 32; ++q) {
                    const double v2 = red_v[q];
                    const int i2 = red_i[q];
                    if (v2 > bv || (v2 == bv && i2 < bidx) || (v2 != v2 && bv == bv)) { bv = v2; bidx = i2; }
                }
                const int sing = (bv > 0.0) ? 0 : ((bv != bv) ? 2 : 1);
                s_piv = bidx;
                s_singular = sing;
                if (C > 1) {
                    st_peer_s32(peer_addr(&s_piv, (uint32_t)(owner ^ 1)), bidx);
                    st_peer_s32(peer_addr(&s_singular, (uint32_t)(owner ^ 1)), sing);
                }
            }
        }
        gj_sync<C>();
        if (s_singular) break;
        const int p = s_piv;
        if (p != k) {
            for (int c = t; c < H; c += kGJT) {
                const cplx a = A[k * H + c];
                A[k * H + c] = A[p * H + c];
                A[p * H + c] = a;
            }
        }
        __syncthreads();
        if (t == 0) {
            perm[k] = p;
            if (p != k) {
                const cplx a = pcol[k];
                pcol[k] = pcol[p];
                pcol[p] = a;
            }
        }
        __syncthreads();
        const cplx piv = pcol[k];
        const cplx inv = cdiv(cplx{1.0, 0.0}, piv);
        if (t == 0 && rank == 0) {
            logabs += log(hypot(piv.re, piv.im));
            phase += atan2(piv.im, piv.re) + (p != k ? M_PI : 0.0);
        }
        for (int c = t; c < H; c += kGJT) prow[c] = A[k * H + c] * inv;
        __syncthreads();
        // Rank-1 update: warps over rows, lanes over (at most COLS) local columns, so the
        // multiplier pcol[i] is one broadcast per row and the pivot row sits in registers.
        // Padding columns (j >= N) hold zeros and stay zero.
        const int warp = t >> 5, lane = t & 31;
        const bool own_k = rank == owner;
        // R rows per warp at a time: all their loads are issued before any arithmetic, so
        // a lane has R * COLS independent updates in flight.
        if (with_inverse) {
            cplx pr[COLS];
#pragma unroll
            for (int u = 0; u < COLS; ++u) pr[u] = (lane + 32 * u < H) ? prow[lane + 32 * u] : cplx{0.0, 0.0};
            for (int i0 = warp; i0 < N; i0 += R * (kGJT / 32)) {
                cplx m[R], a[R][COLS];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = i0 + r * (kGJT / 32);
                    const bool live = i < N && i != k;
                    m[r] = live ? cplx{0.0, 0.0} - pcol[i] : cplx{0.0, 0.0};
#pragma unroll
                    for (int u = 0; u < COLS; ++u) {
                        const int c = lane + 32 * u;
                        if (live && c < H) a[r][u] = A[i * H + c];
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = i0 + r * (kGJT / 32);
                    if (i >= N || i == k) continue;
#pragma unroll
                    for (int u = 0; u < COLS; ++u) {
                        const int c = lane + 32 * u;
                        if (c >= H) continue;
                        if (own_k && c == lk) a[r][u] = m[r] * inv;   // column k of the inverse
                        else cfma(a[r][u], m[r], pr[u]);
                        A[i * H + c] = a[r][u];
                    }
                }
            }
            for (int c = t; c < H; c += kGJT) A[k * H + c] = (own_k && c == lk) ? inv : prow[c];
        } else {
            // trailing block only: rows i > k, columns j > k
            const int c0 = (k + 1 - rank + C - 1) / C;   // first local column with j > k
            cplx pr[COLS];
#pragma unroll
            for (int u = 0; u < COLS; ++u) {
                const int c = c0 + lane + 32 * u;
                pr[u] = c < H ? prow[c] : cplx{0.0, 0.0};
            }
            for (int i0 = k + 1 + warp; i0 < N; i0 += R * (kGJT / 32)) {
                cplx m[R], a[R][COLS];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = i0 + r * (kGJT / 32);
                    m[r] = i < N ? cplx{0.0, 0.0} - pcol[i] : cplx{0.0, 0.0};
#pragma unroll
                    for (int u = 0; u < COLS; ++u) {
                        const int c = c0 + lane + 32 * u;
                        if (i < N && c < H) a[r][u] = A[i * H + c];
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = i0 + r * (kGJT / 32);
                    if (i >= N) continue;
#pragma unroll
                    for (int u = 0; u < COLS; ++u) {
                        const int c = c0 + lane + 32 * u;
                        if (c >= H) continue;
                        cfma(a[r][u], m[r], pr[u]);
                        A[i * H + c] = a[r][u];
                    }
                }
            }
        }
        gj_sync<C>();
    }
    if (s_singular) {
        if (t == 0 && rank == 0) {
            logdet[mat] = cplx{-INFINITY, 0.0};
            atomicOr(flags, s_singular == 2 ? FLAG_NONFINITE : FLAG_SINGULAR);
        }
        if (C > 1) cluster_sync_all();   // keep the peer's shared memory alive until both are done
        return;
    }
    if (with_inverse) {
        // undo the pivoting on the columns: for k = N-1..0 swap columns k and perm[k]
        if (t == 0) {
            for (int j = 0; j < N; ++j) pos[j] = j;    // pos: stored column -> final column, via idx
            int* idx = pos;                             // idx[j] = stored column at final position j
            for (int k = N - 1; k >= 0; --k) {
                const int q = perm[k];
                const int a = idx[k];
                idx[k] = idx[q];
                idx[q] = a;
            }
        }
        __syncthreads();
        // pos currently holds idx; write stored column s = idx[j] to final column j
        for (int e = t; e < N * N; e += kGJT) {
            const int i = e / N, j = e % N;
            const int sc = pos[j];
            if (sc % C != rank) continue;
            G[(int64_t)i * N + j] = A[i * H + sc / C];
        }
    }
    if (t == 0 && rank == 0) logdet[mat] = cplx{logabs, atan2(sin(phase), cos(phase))};
    if (C > 1) cluster_sync_all();
}

// ------------------------------------------------------- Gauss-Jordan in registers
// The inverse and log-determinant of an N x N complex matrix, 32 < N <= 128, held entirely in
// registers: one CTA for N <= 64, else a cluster of two CTAs (the two halves of a 128 x 128
// complex matrix fill two register files).  CTA r owns the 64 consecutive columns
// [64 r, 64 r + 64); warp w of it owns CW of them, and lane l holds rows l, l + 32, ... (RQ of
// them), so the thread's block is RQ x CW.  Pivoting is implicit: step k picks, among the rows
// not pivoted yet, the one with the largest |re| + |im| in column k (lowest row on ties), scales
// it and eliminates column k from every other row, in place, so that after N steps the stored
// array X satisfies X[p_k][j] = inverse[k][p_j] for the pivot rows p_k.  det = sign(p) prod(pivot).
// Four columns are a panel.  Its four steps are taken first, on the panel alone, by RQ neighbouring
// warps, the owner among them (one row a lane, so the chain from one pivot to the next is short:
// search, reciprocal, one row's update), which publish each step's column, pivot row and pivot (to both CTAs'
// shared memory); then all other warps take the same steps, in the same order, on their columns, each
// warp by itself (the pivot row reaches its lanes by shuffles, the multipliers come from shared
// memory), and the next panel's warps go on to that panel.  One barrier per panel orders them.
// Steps that each had a barrier, with the next column updated and searched by its one owner warp,
// left the fp32 pipe idle for two thirds of the time.  32 < N <= 64 runs two matrices an SM
// (CW = 8, 256 threads; a panel of eight columns would spill).  Float pairs are packed two columns to a 64-bit register, which halves the
// instructions; conversions from and to FP64 are by integer operations where they can be (the FP64
// pipe takes 64 cycles for a warp's instruction).
// Measured, a barrier per step -> this: 2048 inverses of N = 128 25.5 -> 13.2 ms in float pairs (the
// fp32 pipe's 6.6 ms for the updates, the panels' chains the rest) and 45.7 -> 37.4 ms in FP64 (the
// FP64 pipe's 28 ms); 512 of N = 64 1.38 -> 0.54 and 2.13 -> 1.74 ms.
constexpr int kGJRegCols = 64;      // columns per CTA
constexpr int kGJPanel = 4;         // columns per panel
template <int CW>
constexpr int kGJRegThreads = 32 * (kGJRegCols / CW);   // a warp per CW columns

// Element arithmetic of the register Gauss-Jordan kernel.  NumD: FP64 complex.  NumFF: each of
// re, im a float pair hi + lo (~2^-44 relative, the TwoProduct / TwoSum error-free transforms on
// the fp32 pipe, which is ~64x GB300's FP64 pipe), pivot reciprocals as exact as FP64 rounded to
// such a pair; the read-out and the log-determinant are FP64 either way.
struct NumD {
    using T = cplx;
    __device__ static T from(cplx v) { return v; }
    __device__ static cplx to(const T& v) { return v; }
    // |re| + |im| as two words ordered like the value (non-negative; infinities, NaN on top)
    __device__ static void key(const T& v, unsigned& hi, unsigned& lo) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(abs1(v));
        hi = (unsigned)(b >> 32);
        lo = (unsigned)b;
    }
    static constexpr bool kTwoWords = true;
    static constexpr unsigned kInf = 0x7ff00000u;   // high word of infinity
    __device__ static T recip(const T& v);
    __device__ static T mul(const T& a, const T& b) { return a * b; }
    template <int RQ, int CW>
    struct Tile {   // a thread's RQ x CW block
        T a[RQ][CW];
        __device__ T get(int q, int u) const { return a[q][u]; }
        __device__ void set(int q, int u, const T& v) { a[q][u] = v; }
    };
    template <int RQ, int CW>   // row q: a -= m p
    __device__ static void upd(Tile<RQ, CW>& t, int q, const T& m, const Tile<1, CW>& p) {
#pragma unroll
        for (int u = 0; u < CW; ++u) cfma(t.a[q][u], cplx{-m.re, -m.im}, p.a[0][u]);
    }
    __device__ static T negmul(const T& m, const T& b) { const cplx w = m * b; return cplx{-w.re, -w.im}; }
    __device__ static T shfl(const T& v, int src) {
        return cplx{__shfl_sync(0xffffffffu, v.re, src), __shfl_sync(0xffffffffu, v.im, src)};
    }
    __device__ static void st_peer(uint32_t ad, const T& v) {
        st_peer_f64(ad, v.re);
        st_peer_f64(ad + 8, v.im);
    }
};
struct NumFF {
    using T = ffc;
    __device__ static T from(cplx v) {
        ffc r;
        ff_split(v.re, r.rh, r.rl);
        ff_split(v.im, r.ih, r.il);
        return r;
    }
    __device__ static cplx to(const T& v) { return cplx{widen(v.rh) + widen(v.rl), widen(v.ih) + widen(v.il)}; }
    __device__ static void key(const T& v, unsigned& hi, unsigned& lo) {
        hi = __float_as_uint(fabsf(v.rh) + fabsf(v.ih));
        lo = 0u;
    }
    static constexpr bool kTwoWords = false;
    static constexpr unsigned kInf = 0x7f800000u;
    __device__ static T recip(const T& v);
    __device__ static T mul(const T& a, const T& b) {
        T r{0.f, 0.f, 0.f, 0.f};
        ff_fma(r.rh, r.rl, a.rh, a.rl, b.rh, b.rl);
        ff_fma(r.rh, r.rl, -a.ih, -a.il, b.ih, b.il);
        ff_fma(r.ih, r.il, a.rh, a.rl, b.ih, b.il);
        ff_fma(r.ih, r.il, a.ih, a.il, b.rh, b.rl);
        return r;
    }
    template <int RQ, int CW>
    struct Tile {   // a thread's RQ x CW block, columns 2 j and 2 j + 1 packed
        f32x2 rh[RQ][CW / 2], rl[RQ][CW / 2], ih[RQ][CW / 2], il[RQ][CW / 2];
        __device__ T get(int q, int u) const {
            return ffc{part(rh[q][u / 2], u), part(rl[q][u / 2], u), part(ih[q][u / 2], u), part(il[q][u / 2], u)};
        }
        __device__ void set(int q, int u, const T& v) {
            put(rh[q][u / 2], u, v.rh);
            put(rl[q][u / 2], u, v.rl);
            put(ih[q][u / 2], u, v.ih);
            put(il[q][u / 2], u, v.il);
        }
        __device__ static float part(f32x2 x, int u) { return u & 1 ? f2_hi(x) : f2_lo(x); }
        __device__ static void put(f32x2& x, int u, float v) { x = u & 1 ? f2(f2_lo(x), v) : f2(v, f2_hi(x)); }
    };
    template <int RQ, int CW>   // row q: a -= m p
    __device__ static void upd(Tile<RQ, CW>& t, int q, const T& m, const Tile<1, CW>& p) {
        const f32x2 rh = f2(m.rh, m.rh), nrh = f2(-m.rh, -m.rh), nrl = f2(-m.rl, -m.rl);
        const f32x2 ih = f2(m.ih, m.ih), nih = f2(-m.ih, -m.ih), il = f2(m.il, m.il), nil = f2(-m.il, -m.il);
#pragma unroll
        for (int j = 0; j < CW / 2; ++j) {
            ff_fma2(t.rh[q][j], t.rl[q][j], nrh, rh, nrl, p.rh[0][j], p.rl[0][j]);
            ff_fma2(t.rh[q][j], t.rl[q][j], ih, nih, il, p.ih[0][j], p.il[0][j]);
            ff_fma2(t.ih[q][j], t.il[q][j], nrh, rh, nrl, p.ih[0][j], p.il[0][j]);
            ff_fma2(t.ih[q][j], t.il[q][j], nih, ih, nil, p.rh[0][j], p.rl[0][j]);
        }
    }
    __device__ static T negmul(const T& m, const T& b) {
        const T w = mul(m, b);
        return ffc{-w.rh, -w.rl, -w.ih, -w.il};
    }
    __device__ static T shfl(const T& v, int src) {
        return ffc{__shfl_sync(0xffffffffu, v.rh, src), __shfl_sync(0xffffffffu, v.rl, src),
                   __shfl_sync(0xffffffffu, v.ih, src), __shfl_sync(0xffffffffu, v.il, src)};
    }
    __device__ static void st_peer(uint32_t ad, const T& v) {
        asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(ad), "f"(v.rh), "f"(v.rl), "f"(v.ih),
                     "f"(v.il)
                     : "memory");
    }
};

// v 2^n, by the exponent field where v and the result are normal.
__device__ __forceinline__ double scale2(double v, int n) {
    const int hi = __double2hiint(v), lo = __double2loint(v), e = (hi >> 20) & 0x7ff;
    if (((hi << 1) | lo) == 0) return v;
    if (e == 0 || e == 0x7ff || (unsigned)(e + n - 1) >= 2046u) return ldexp(v, n);
    return __hiloint2double(hi + (n << 20), lo);
}
// z scaled by a power of two so that its larger component lies in [1, 2); returns the exponent taken
// out.  z finite and not zero.
__device__ __forceinline__ int cnormalise(cplx& z) {
    int e = max((__double2hiint(z.re) >> 20) & 0x7ff, (__double2hiint(z.im) >> 20) & 0x7ff) - 1023;
    if (e == -1023) {   // both subnormal
        frexp(fmax(fabs(z.re), fabs(z.im)), &e);
        --e;
    }
    z = cplx{scale2(z.re, -e), scale2(z.im, -e)};
    return e;
}
// 1 / z: |z|^2 of z scaled as above, which keeps it away from overflow and underflow, and 1 / |z|^2
// as r (1 + e + e^2), e = 1 - |z|^2 r, from the float reciprocal r (e^3 < 2^-66, so the last rounding
// is all the error).  Six dependent FP64 operations, at 200 cycles each, where frexp, ldexp and the
// division took some twenty.
__device__ __forceinline__ cplx crecip(cplx z) {
    const int n = -cnormalise(z);
    const double d = fma(z.re, z.re, z.im * z.im);   // in [1, 8)
    const float df = __uint_as_float((unsigned)((unsigned long long)__double_as_longlong(d) >> 29) - (896u << 23));
    const double r0 = widen(__frcp_rn(df));
    const double e = fma(-d, r0, 1.0);
    const double r = fma(r0, fma(e, e, e), r0);
    return cplx{scale2(z.re * r, n), scale2(-z.im * r, n)};
}
// log det from the product of the pivots v (scaled, exponent ex apart)
__device__ __forceinline__ cplx log_of_product(cplx v, int ex) {
    return cplx{0.5 * log(fma(v.re, v.re, v.im * v.im)) + ex * M_LN2, atan2(v.im, v.re)};
}

// entry (q, u) of a tile with q (sel_q) or u (sel_u) known at run time only
template <class Num, int RQ, int CW>
__device__ __forceinline__ typename Num::T sel_q(const typename Num::template Tile<RQ, CW>& t, int q, int u) {
    typename Num::T r = t.get(0, u);
#pragma unroll
    for (int i = 1; i < RQ; ++i)
        if (q == i) r = t.get(i, u);
    return r;
}
template <class Num, int RQ, int CW>
__device__ __forceinline__ typename Num::T sel_u(const typename Num::template Tile<RQ, CW>& t, int q, int u) {
    typename Num::T r = t.get(q, 0);
#pragma unroll
    for (int i = 1; i < CW; ++i)
        if (u == i) r = t.get(q, i);
    return r;
}

__device__ __forceinline__ cplx NumD::recip(const cplx& v) { return crecip(v); }
// 1 / z for a float pair, on the fp32 pipe: z scaled by a power of two as in crecip, q = conj(z) / |z|^2
// in single precision, then one Newton step q (1 + e + e^2), e = 1 - z q, with e and the product as
// float pairs (2^-22 -> 2^-50, as FP64 rounded to a pair).  In FP64 (an instruction of its pipe takes 200 cycles of a chain) this
// was two thirds of the way from one pivot to the next.
__device__ __forceinline__ ffc NumFF::recip(const ffc& z) {
    const float mx = fmaxf(fabsf(z.rh), fabsf(z.ih));
    const int ex = (int)((__float_as_uint(mx) >> 23) & 0xffu);          // biased exponent
    const int es = min(max(254 - ex, 1), 253);                          // 2^(es - 127) mx in [1, 2)
    const float s = __uint_as_float((unsigned)es << 23);
    const float ah = z.rh * s, al = z.rl * s, bh = z.ih * s, bl = z.il * s;
    const float r = __frcp_rn(fmaf(ah, ah, bh * bh));
    const float qr = ah * r, qi = -(bh * r);
    // e = 1 - (ah + al + i (bh + bl)) (qr + i qi): the leading products' and sums' errors and the low
    // products gathered with their own errors (without those, four times the error of FP64)
    auto low = [](float a, float b, float ga, float gb, float ha, float hb, float c, float& lead) {
        // lead + (a + b + ga gb + ha hb + c) as a float pair; returns the low half
        const float g = ga * gb, ge = fmaf(ga, gb, -g), h = ha * hb, he = fmaf(ha, hb, -h);
        float l1, c1, l2, c2, l3, c3, l4, c4, c5;
        two_sum(a, b, l1, c1);
        two_sum(g, h, l2, c2);
        two_sum(l1, l2, l3, c3);
        two_sum(l3, c, l4, c4);
        two_sum(lead, l4, lead, c5);
        return c5 + ((c1 + c2) + (c3 + c4) + (ge + he));
    };
    const float p1 = ah * qr, e1 = fmaf(ah, qr, -p1), p2 = bh * qi, e2 = fmaf(bh, qi, -p2);
    float s1, t1, xh, t2, s3, t3;
    two_sum(1.0f, -p1, s1, t1);
    two_sum(s1, p2, xh, t2);
    const float xl = low(e2, -e1, -al, qr, bl, qi, t1 + t2, xh);
    const float p3 = ah * qi, e3 = fmaf(ah, qi, -p3), p4 = bh * qr, e4 = fmaf(bh, qr, -p4);
    two_sum(p3, p4, s3, t3);
    const float nl = low(e3, e4, al, qi, bl, qr, t3, s3);
    const float yh = -s3, yl = -nl;
    // f = e + e^2, q (1 + f)
    const float fl = fmaf(xh, xh, fmaf(-yh, yh, xl)), gl = fmaf(2.0f * xh, yh, yl);
    auto add = [&](float q, float a, float b, float c, float d, float bl2, float dl) {   // q + a (b + bl2) + c (d + dl)
        const float m1 = a * b, h1 = fmaf(a, b, -m1), m2 = c * d, h2 = fmaf(c, d, -m2);
        float u, v, h, l;
        two_sum(m1, m2, u, v);
        v = fmaf(a, bl2, fmaf(c, dl, v + (h1 + h2)));
        two_sum(q, u, h, l);
        l += v;
        const float hi = h + l;
        return make_float2(hi * s, (l - (hi - h)) * s);
    };
    const float2 re = add(qr, qr, xh, -qi, yh, fl, gl), im = add(qi, qr, yh, qi, xh, gl, fl);
    return ffc{re.x, re.y, im.x, im.y};
}

// barrier of the RQ warps that work on a panel (a group at a time, ordered by the CTA's barriers)
template <int RQ>
__device__ __forceinline__ void gj_panel_sync() {
    asm volatile("bar.sync 1, %0;" ::"n"(32 * RQ) : "memory");
}
// Shared memory of a CTA: the panel being applied and the next one being published (buffers b and
// b ^ 1), the panel's columns on their way between its owner and the warps that work on it, and for
// each of these the best pivot and its row (two steps in turn).
template <class Num, int RQ>
struct GJShared {
    using T = typename Num::T;
    T col[2][kGJPanel][32 * RQ];            // columns before their elimination: the multipliers
    T inv[2][kGJPanel], piv[2][kGJPanel];   // pivots and their reciprocals
    int p[2][kGJPanel];                     // pivot rows (or -1 singular, -2 non-finite)
    T x[2][kGJPanel][32 * RQ];
    T row[2][RQ][kGJPanel];
    unsigned key[2][RQ][3];
    T pivs[32 * RQ];
    int perm[32 * RQ], pinv[32 * RQ];
    cplx det[RQ];
    int dexp[RQ];
};
// The steps of one panel (columns c0 ...), by RQ warps: warp q has the rows 32 q ... + 31.  used:
// bit q, row lane + 32 q is a pivot row already.
template <class Num, int C, int RQ>
__device__ __forceinline__ void gj_panel(GJShared<Num, RQ>& sh, int b, int c0, int N, int q, int lane, int rank,
                                         unsigned& used) {
    constexpr int CW = kGJPanel;
    using T = typename Num::T;
    const int i = lane + 32 * q;
    typename Num::template Tile<1, CW> x;
#pragma unroll
    for (int u = 0; u < CW; ++u) x.set(0, u, sh.x[b][u][i]);
#pragma unroll 1
    for (int s = 0; s < CW && c0 + s < N; ++s) {
        const int e = s & 1;
        const T m = sel_u<Num, 1, CW>(x, 0, s);
        sh.col[b][s][i] = m;
        if (C > 1) Num::st_peer(peer_addr(&sh.col[b][s][i], (uint32_t)(rank ^ 1)), m);
        // the warp's largest unused entry, lowest row on ties
        const bool open = i < N && !((used >> q) & 1u);
        unsigned kh = 0u, kl = 0u;
        if (open) Num::key(m, kh, kl);
        const unsigned mh = __reduce_max_sync(0xffffffffu, kh);
        const unsigned ml = Num::kTwoWords ? __reduce_max_sync(0xffffffffu, kh == mh ? kl : 0u) : 0u;
        const unsigned hit = __ballot_sync(0xffffffffu, open && kh == mh && kl == ml);
        const int wl = hit ? __ffs(hit) - 1 : 0;
        if (lane == wl) {
            sh.key[e][q][0] = hit ? mh : 0u;
            sh.key[e][q][1] = hit ? ml : 0u;
            sh.key[e][q][2] = hit ? (unsigned)i : 0xffffffffu;
#pragma unroll
            for (int u = 0; u < CW; ++u) sh.row[e][q][u] = x.get(0, u);
        }
        gj_panel_sync<RQ>();
        unsigned bh = sh.key[e][0][0], bl = sh.key[e][0][1], bi = sh.key[e][0][2];
#pragma unroll
        for (int w = 1; w < RQ; ++w) {
            const unsigned h = sh.key[e][w][0], l = sh.key[e][w][1], r = sh.key[e][w][2];
            if (r != 0xffffffffu && (bi == 0xffffffffu || h > bh || (h == bh && l > bl))) { bh = h; bl = l; bi = r; }
        }
        // a zero column is singular; a NaN or infinite pivot magnitude is non-finite
        const int p = bh >= Num::kInf ? -2 : ((bh | bl) == 0u ? -1 : (int)bi);
        if (p < 0) {   // the same in all RQ warps
            if (q == 0 && lane == 0) {
                sh.p[b][s] = p;
                if (C > 1) st_peer_s32(peer_addr(&sh.p[b][s], (uint32_t)(rank ^ 1)), p);
            }
            break;
        }
        const int pl = p & 31, pq = p >> 5;
        const T pv = sh.row[e][pq][s];
        const T inv = Num::recip(pv);
        if (q == 0 && lane == 0) {
            sh.p[b][s] = p;
            sh.inv[b][s] = inv;
            sh.piv[b][s] = pv;
            if (C > 1) {
                st_peer_s32(peer_addr(&sh.p[b][s], (uint32_t)(rank ^ 1)), p);
                Num::st_peer(peer_addr(&sh.inv[b][s], (uint32_t)(rank ^ 1)), inv);
                Num::st_peer(peer_addr(&sh.piv[b][s], (uint32_t)(rank ^ 1)), pv);
            }
        }
        const T mine = Num::mul(sh.row[e][pq][lane & (CW - 1)], inv);   // lane u scales entry u
        typename Num::template Tile<1, CW> prow;
#pragma unroll
        for (int u = 0; u < CW; ++u) prow.set(0, u, Num::shfl(mine, u));
        Num::upd(x, 0, m, prow);
        const T val = i == p ? inv : Num::negmul(m, inv);   // column c0 + s of the inverse
#pragma unroll
        for (int u = 0; u < CW; ++u) {
            const T w = i == p ? prow.get(0, u) : x.get(0, u);
            x.set(0, u, u == s ? val : w);
        }
        if (lane == pl) used |= 1u << pq;
    }
#pragma unroll
    for (int u = 0; u < CW; ++u) sh.x[b][u][i] = x.get(0, u);
}

template <class Num, int C, int RQ, int CW>
__global__ void __launch_bounds__(kGJRegThreads<CW>, CW / 4)
    gj_reg_kernel(cplx* Sbase, int64_t stride, int N, cplx* logdet, unsigned* flags) {
    using T = typename Num::T;
    __shared__ GJShared<Num, RQ> sh;
    const int rank = C == 1 ? 0 : (int)cluster_rank();
    const int64_t mat = C == 1 ? blockIdx.x : blockIdx.x / C;
    cplx* G = Sbase + mat * stride;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c0 = rank * kGJRegCols + warp * CW;                                  // first global column of this warp
    const int g0 = rank * kGJRegCols + warp / RQ * RQ * CW, g1 = g0 + RQ * CW;     // columns of its group of RQ warps
    typename Num::template Tile<RQ, CW> a;
#pragma unroll
    for (int q = 0; q < RQ; ++q) {
        const int i = lane + 32 * q;
#pragma unroll
        for (int u = 0; u < CW; ++u) {
            const int j = c0 + u;
            a.set(q, u, Num::from((i < N && j < N) ? G[(int64_t)i * N + j] : cplx{0.0, 0.0}));
        }
    }
    unsigned used = 0;   // bit q: row lane + 32 q is a pivot row already
    // step s of the panel published in buffer b, on this warp's columns: a -= m prow, prow in the
    // pivot row
    auto step = [&](int b, int s) {
        const int p = sh.p[b][s];
        const T inv = sh.inv[b][s];
        const int pl = p & 31, pq = p >> 5;
        if (lane == pl) used |= 1u << pq;
        // the warp's pivot-row entries: gathered from lane pl, each scaled by one lane (lane
        // u % CW scales entry u), then shared again
        T mine = Num::shfl(sel_q<Num, RQ, CW>(a, pq, 0), pl);
#pragma unroll
        for (int u = 1; u < CW; ++u) {
            const T e = Num::shfl(sel_q<Num, RQ, CW>(a, pq, u), pl);
            if ((lane & (CW - 1)) == u) mine = e;
        }
        mine = Num::mul(mine, inv);
        typename Num::template Tile<1, CW> prow;
#pragma unroll
        for (int u = 0; u < CW; ++u) prow.set(0, u, Num::shfl(mine, u));
#pragma unroll
        for (int q = 0; q < RQ; ++q) {
            if (32 * q >= N) break;
            Num::upd(a, q, sh.col[b][s][lane + 32 * q], prow);
            if (q == pq) {   // the same in every thread
#pragma unroll
                for (int u = 0; u < CW; ++u) a.set(q, u, lane == pl ? prow.get(0, u) : a.get(q, u));
            }
        }
    };
    // panel t, published in buffer b: by the owner's group of RQ warps.  The owner's columns wait in
    // sh.x until it has taken the panel's steps on its others.
    auto panel = [&](int t, int b) {
        const int pc = t * kGJPanel;
        if (pc < g0 || pc >= g1 || pc >= N) return;
#pragma unroll
        for (int o = 0; o < CW; o += kGJPanel)
            if (pc == c0 + o) {
#pragma unroll
                for (int q = 0; q < RQ; ++q)
#pragma unroll
                    for (int u = 0; u < kGJPanel; ++u) sh.x[b][u][lane + 32 * q] = a.get(q, o + u);
            }
        gj_panel_sync<RQ>();
        gj_panel<Num, C, RQ>(sh, b, pc, N, warp % RQ, lane, rank, used);
    };
    if (C > 1) gj_sync<C>();   // the peer runs before anything is written to its shared memory
    panel(0, 0);
    gj_sync<C>();
    int singular = 0;
    for (int t = 0; t * kGJPanel < N; ++t) {
        const int b = t & 1, pc = t * kGJPanel, ns = min(kGJPanel, N - pc);
        for (int s = 0; s < ns && !singular; ++s) {
            const int p = sh.p[b][s];
            if (p < 0) singular = p;
            else if (threadIdx.x == 0) { sh.perm[pc + s] = p; sh.pivs[pc + s] = sh.piv[b][s]; }
        }
        if (singular) break;
        if (g0 < N && (CW > kGJPanel || pc != c0)) {
#pragma unroll 1
            for (int s = 0; s < ns; ++s) step(b, s);
        }
#pragma unroll
        for (int o = 0; o < CW; o += kGJPanel)
            if (pc == c0 + o) {
#pragma unroll
                for (int q = 0; q < RQ; ++q)
#pragma unroll
                    for (int u = 0; u < kGJPanel; ++u) a.set(q, o + u, sh.x[b][u][lane + 32 * q]);
            }
        panel(t + 1, b ^ 1);
        gj_sync<C>();
    }
    if (singular) {
        if (threadIdx.x == 0 && rank == 0) {
            logdet[mat] = cplx{-INFINITY, 0.0};
            atomicOr(flags, singular == -2 ? FLAG_NONFINITE : FLAG_SINGULAR);
        }
        if (C > 1) cluster_sync_all();   // keep shared memory alive until the peer is done
        return;
    }
    __syncthreads();
    if (threadIdx.x < N) sh.pinv[sh.perm[threadIdx.x]] = threadIdx.x;
    // log|det| and arg det from the product of the pivots (fixed order: a lane each, a tree over the
    // warp, the RQ warps in turn), the exponents apart, times -1 for an odd pivot permutation, whose
    // sign is that of its inversions (pairs of steps whose pivot rows are out of order)
    int odd = 0;
    if (rank == 0 && warp < RQ) {
        const int k = (int)threadIdx.x;
        cplx v{1.0, 0.0};
        int ex = 0;
        if (k < N) {
            v = Num::to(sh.pivs[k]);
            ex = cnormalise(v);
            const int pk = sh.perm[k];
            for (int j = 0; j < k; ++j) odd ^= sh.perm[j] > pk ? 1 : 0;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            v = v * cplx{__shfl_xor_sync(0xffffffffu, v.re, o), __shfl_xor_sync(0xffffffffu, v.im, o)};
            ex += __shfl_xor_sync(0xffffffffu, ex, o);
        }
        ex += cnormalise(v);
        odd = __popc(__ballot_sync(0xffffffffu, odd)) & 1;
        if (lane == 0) {
            sh.det[warp] = v;
            sh.dexp[warp] = 2 * ex + odd;
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < RQ; ++q) {
        const int i = lane + 32 * q;
        if (i >= N) continue;
        const int64_t orow = (int64_t)sh.pinv[i] * N;
#pragma unroll
        for (int u = 0; u < CW; ++u) {
            const int j = c0 + u;
            if (j < N) G[orow + sh.perm[j]] = Num::to(a.get(q, u));
        }
    }
    if (rank == 0 && warp == 0) {
        cplx v = sh.det[0];
        int ex = sh.dexp[0] >> 1, sign = sh.dexp[0];
#pragma unroll
        for (int w = 1; w < RQ; ++w) {
            v = v * sh.det[w];
            ex += sh.dexp[w] >> 1;
            sign += sh.dexp[w];
        }
        ex += cnormalise(v);
        if (sign & 1) v = cplx{-v.re, -v.im};
        const cplx ld = log_of_product(v, ex);
        if (lane == 0) logdet[mat] = ld;
    }
    if (C > 1) cluster_sync_all();
}

// ------------------------------------------------------- Gauss-Jordan, one warp per matrix
// The inverse and log-determinant of an N x N complex matrix, N <= 32, by one warp: lane i holds
// row i in registers, padded to NC columns with the identity (which changes neither the true
// block nor the determinant), so the elimination needs no block barrier and an SM runs as many
// matrices as warps fit.  Pivoting is implicit as in gj_reg_kernel (max |re| + |im| among the rows
// not used yet, lowest row on ties); the pivot row passes through shared memory, where lane j
// scales entry j, and every lane reads it back as broadcasts.  Each step's pivot column is always
// register column 0: the update writes column j to j - 1 and the new column of the inverse
// to NC - 1, so the step is one loop body with static register indices.  INV = false stops at the log-determinant and updates the trailing columns
// only (in groups of 8).
// Bound by the FP64 pipe (2 multiply-adds per SM and clock: 0.22 ms for the inverses of 1024
// matrices of N = 32), which the 512-thread shared-memory kernel missed by its four barriers
// a step on blocks of one matrix each.  Measured, the shared-memory kernel -> this one: 1024
// inverses of N = 32 3.79 -> 0.33 ms, N = 16 1.79 -> 0.10 ms; log-determinants alone 3.28 -> 0.22 ms.
constexpr int kGJWarpMax = 32;
constexpr int kGJWarps = 2;   // matrices per CTA

// log det of one warp's matrix: lane k has the pivot of step k and its row (1 and 0 past N).
template <int NC>
__device__ __forceinline__ cplx gj_warp_logdet(cplx piv, int perm, int N) {
    const int lane = threadIdx.x & 31;
    // log|det| and arg det from the product of the pivots, times -1 for an odd pivot permutation,
    // whose sign is that of its inversions (pairs of steps whose pivot rows are out of order)
    cplx v = piv;
    int ex = cnormalise(v);
    int odd = 0;
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        const int pj = __shfl_sync(0xffffffffu, perm, j);
        if (lane < N && j < lane && pj > perm) odd ^= 1;
    }
    odd = __popc(__ballot_sync(0xffffffffu, odd)) & 1;
#pragma unroll
    for (int o = NC > 16 ? 16 : NC / 2; o > 0; o >>= 1) {   // the first NC lanes' pivots; the others' are 1
        v = v * cplx{__shfl_xor_sync(0xffffffffu, v.re, o), __shfl_xor_sync(0xffffffffu, v.im, o)};
        ex += __shfl_xor_sync(0xffffffffu, ex, o);
    }
    ex += cnormalise(v);
    if (odd) v = cplx{-v.re, -v.im};
    return log_of_product(v, ex);
}

template <int NC, bool INV>
__global__ void __launch_bounds__(32 * kGJWarps)
    gj_warp_kernel(cplx* Sbase, int64_t stride, int N, int count, cplx* logdet, unsigned* flags) {
    __shared__ __align__(16) cplx rowbuf[kGJWarps][NC];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t mat = (int64_t)blockIdx.x * kGJWarps + warp;
    if (mat >= count) return;
    cplx* G = Sbase + mat * stride;
    cplx* row = rowbuf[warp];
    cplx a[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        a[j] = cplx{lane == j ? 1.0 : 0.0, 0.0};
        if (lane < N && j < N) a[j] = G[(int64_t)lane * N + j];
    }
    bool used = lane >= N;
    int mystep = 0, myperm = 0;         // lane i: step that used row i; lane k: pivot row of step k
    cplx mypiv{1.0, 0.0};               // lane k: pivot of step k
    int bad = 0;
#pragma unroll 1
    for (int k = 0; k < N; ++k) {
        // largest |re| + |im| by its bit pattern (ordered for non-negative doubles; infinities and
        // NaN come out on top)
        const unsigned long long key = used ? 0ull : (unsigned long long)__double_as_longlong(abs1(a[0]));
        const unsigned kh = (unsigned)(key >> 32);
        const unsigned mh = __reduce_max_sync(0xffffffffu, kh);
        const unsigned kl = kh == mh ? (unsigned)key : 0u;
        const unsigned ml = __reduce_max_sync(0xffffffffu, kl);
        const unsigned hit = __ballot_sync(0xffffffffu, !used && kh == mh && kl == ml);
        if (mh >= 0x7ff00000u) { bad = 2; break; }
        if ((mh | ml) == 0u) { bad = 1; break; }
        const int p = __ffs(hit) - 1;
        if (lane == p) {
#pragma unroll
            for (int j = 0; j < NC; ++j) row[j] = a[j];
        }
        __syncwarp();
        const cplx piv = row[0];
        const cplx inv = crecip(piv);
        cplx mine{0.0, 0.0};
        if (lane < NC) mine = lane == 0 ? inv : row[lane] * inv;
        __syncwarp();
        if (lane < NC) row[lane] = mine;
        if (lane == k) { mypiv = piv; myperm = p; }
        if (lane == p) { used = true; mystep = k; }
        __syncwarp();
        const bool isp = lane == p;
        const cplx nm{-a[0].re, -a[0].im};
        cplx last{0.0, 0.0};
        if (INV) {   // column k of the inverse: -m / piv, 1 / piv in the pivot row
            last = nm * inv;
            if (isp) last = inv;
        }
#pragma unroll
        for (int j0 = 0; j0 < NC; j0 += 8) {
            if (INV || j0 < NC - k) {
#pragma unroll
                for (int j = j0 < 1 ? 1 : j0; j < (j0 + 8 < NC ? j0 + 8 : NC); ++j) {
                    const cplx pr = row[j];
                    cplx v = a[j];
                    cfma(v, nm, pr);
                    a[j - 1] = isp ? pr : v;
                }
            }
        }
        a[NC - 1] = last;
        __syncwarp();
    }
    if (bad) {
        if (lane == 0) {
            logdet[mat] = cplx{-INFINITY, 0.0};
            atomicOr(flags, bad == 2 ? FLAG_NONFINITE : FLAG_SINGULAR);
        }
        return;
    }
    const cplx ld = gj_warp_logdet<NC>(mypiv, myperm, N);
    if (lane == 0) logdet[mat] = ld;
    if (INV) {   // row i of the array is row mystep of the inverse; column j is its column perm[j]
#pragma unroll
        for (int u = 0; u < NC; ++u) {
            const int j = u + N < NC ? u + N : u + N - NC;   // N steps moved column j to register u
            const int c = __shfl_sync(0xffffffffu, myperm, j);
            if (lane < N && j < N) G[(int64_t)mystep * N + c] = a[u];
        }
    }
}

// The same by a team of four warps, for counts that leave schedulers without a matrix: warp w holds the
// columns [w NC / 4, (w + 1) NC / 4), so a step's updates take a quarter of one pipe's time on four.  The
// warp of column k + 1 updates that first, finds its pivot and publishes it with the column before the
// rest of its update; one barrier a step.  The arithmetic is gj_warp_kernel's, bit for bit.
// Measured, one warp -> team, inverses (ms): 128 of N = 32 0.240 -> 0.100, 122 of N = 23 0.135 -> 0.065,
// 128 of N = 16 0.079 -> 0.043, 16 of N = 5 0.028 -> 0.021.
constexpr int kGJTeam = 4;
template <int NC, bool INV>
__global__ void __launch_bounds__(32 * kGJTeam)
    gj_team_kernel(cplx* Sbase, int64_t stride, int N, cplx* logdet, unsigned* flags) {
    constexpr int CW = NC / kGJTeam;
    __shared__ __align__(16) cplx col[2][32];       // the pivot column, before its elimination
    __shared__ __align__(16) cplx row[kGJTeam][CW];
    __shared__ cplx inv_s[2], piv_s[2], pivs[32];
    __shared__ int p_s[2], perm[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c0 = warp * CW;
    const int64_t mat = blockIdx.x;
    cplx* G = Sbase + mat * stride;
    cplx a[CW];
#pragma unroll
    for (int u = 0; u < CW; ++u) {
        a[u] = cplx{lane == c0 + u ? 1.0 : 0.0, 0.0};
        if (lane < N && c0 + u < N) a[u] = G[(int64_t)lane * N + c0 + u];
    }
    bool used = lane >= N;
    int mystep = 0;
    // pivot search in a column (entry v of this lane's row) and publication in buffer b
    auto publish = [&](int b, const cplx& v) {
        const unsigned long long key = used ? 0ull : (unsigned long long)__double_as_longlong(abs1(v));
        const unsigned kh = (unsigned)(key >> 32);
        const unsigned mh = __reduce_max_sync(0xffffffffu, kh);
        const unsigned kl = kh == mh ? (unsigned)key : 0u;
        const unsigned ml = __reduce_max_sync(0xffffffffu, kl);
        const unsigned hit = __ballot_sync(0xffffffffu, !used && kh == mh && kl == ml);
        const int p = mh >= 0x7ff00000u ? -2 : ((mh | ml) == 0u ? -1 : __ffs(hit) - 1);
        col[b][lane] = v;
        if (p >= 0) {   // the same in every lane
            const cplx piv{__shfl_sync(0xffffffffu, v.re, p), __shfl_sync(0xffffffffu, v.im, p)};
            const cplx inv = crecip(piv);
            if (lane == 0) {
                inv_s[b] = inv;
                piv_s[b] = piv;
            }
        }
        if (lane == 0) p_s[b] = p;
    };
    if (warp == 0) publish(0, a[0]);
    __syncthreads();
    int bad = 0;
#pragma unroll 1
    for (int k = 0; k < N; ++k) {
        const int b = k & 1, p = p_s[b];
        if (p < 0) { bad = p; break; }
        const cplx inv = inv_s[b], m = col[b][lane], nm{-m.re, -m.im};
        const bool isp = lane == p;
        if (threadIdx.x == 0) {
            perm[k] = p;
            pivs[k] = piv_s[b];
        }
        if (isp) {
            used = true;
            mystep = k;
#pragma unroll
            for (int u = 0; u < CW; ++u) row[warp][u] = a[u];
        }
        __syncwarp();
        cplx mine{0.0, 0.0};
        if (lane < CW) mine = row[warp][lane] * inv;
        __syncwarp();
        if (lane < CW) row[warp][lane] = mine;
        __syncwarp();
        const int uk = k - c0, u1 = uk + 1;
        auto update = [&](int u) {
            const cplx pr = row[warp][u];
            cplx v = a[u];
            cfma(v, nm, pr);
            a[u] = isp ? pr : v;
        };
        const bool next = u1 >= 0 && u1 < CW && k + 1 < N;
        if (next) {
#pragma unroll
            for (int u = 0; u < CW; ++u)
                if (u == u1) {
                    update(u);
                    publish(b ^ 1, a[u]);
                }
        }
#pragma unroll
        for (int u = 0; u < CW; ++u) {
            if ((next && u == u1) || (!INV && u <= uk)) continue;
            if (u == uk) {   // column k of the inverse: -m / piv, 1 / piv in the pivot row
                const cplx last = nm * inv;
                a[u] = isp ? inv : last;
            } else {
                update(u);
            }
        }
        __syncthreads();
    }
    if (bad) {
        if (threadIdx.x == 0) {
            logdet[mat] = cplx{-INFINITY, 0.0};
            atomicOr(flags, bad == -2 ? FLAG_NONFINITE : FLAG_SINGULAR);
        }
        return;
    }
    if (warp == 0) {
        const cplx ld = gj_warp_logdet<NC>(lane < N ? pivs[lane] : cplx{1.0, 0.0}, lane < N ? perm[lane] : 0, N);
        if (lane == 0) logdet[mat] = ld;
    }
    if (INV) {
#pragma unroll
        for (int u = 0; u < CW; ++u)
            if (lane < N && c0 + u < N) G[(int64_t)mystep * N + perm[c0 + u]] = a[u];
    }
}

// ------------------------------------------------------------------ traces of T
// t = Tr T and X = Tr(T T) of each matrix.  T_ab T_ba counts twice off the diagonal, so the pairs
// (a, a + s mod N) with s = 1 .. (N - 1) / 2 (and, for even N, half of s = N / 2) cover X with half the
// multiply-adds.  GROUP threads (a warp for N <= 32, a CTA above) stage one matrix in shared
// memory at an even row pitch, which makes the reads of T_a,a+s and T_a+s,a (lanes over a) free of
// bank conflicts, and leave four sums.  Bound by the FP64 pipe (2 N^2 multiply-adds, 16 cycles a
// warp instruction) beside the read of T; the old form, which read T_ba with a stride from global
// memory and did every product twice, took 16.8 ms for the 655,360 matrices of a step at M = 128,
// W = 512; this one 3.6 ms, with twelve matrices an SM in flight (3.9 with eight).
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
template <int GROUP, int T_>
__global__ void __launch_bounds__(T_)
    trace_pairs_kernel(const cplx* T, int64_t count, int W, int N, int n0, cplx* t_out, cplx* X_out, int64_t ldo) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[kThreads / 32][4];
    const int P = N + (N & 1);
    const int grp = threadIdx.x / GROUP, l = threadIdx.x % GROUP, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    cplx* m = reinterpret_cast<cplx*>(smem_raw) + (size_t)grp * N * P;
    auto sync = [] {
        if (GROUP == 32) __syncwarp();
        else __syncthreads();
    };
    constexpr int kGroups = T_ / GROUP;
    const int64_t NN = (int64_t)N * N;
    for (int64_t i0 = (int64_t)blockIdx.x * kGroups; i0 < count; i0 += (int64_t)gridDim.x * kGroups) {
        const int64_t i = i0 + grp;   // matrix (c, w)
        if (GROUP == 32 && i >= count) break;
        for (int e = l; e < N * N; e += GROUP) {
            const int a = e / N;
            cp_async16(m + a * P + (e - a * N), T + i * NN + e);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        sync();
        cplx tr{0.0, 0.0}, x{0.0, 0.0};   // x: the pairs, to be counted twice
        double xr = 0.0, xi = 0.0;        // products counted once
        for (int a = l; a < N; a += GROUP) {
            const cplx d = m[a * P + a];
            tr = tr + d;
            xr += fma(d.re, d.re, -d.im * d.im);
            xi += 2.0 * d.re * d.im;
        }
        const int half = (N - 1) / 2;
        if (GROUP == 32) {
            if (l < N) {
                int b = l;
                for (int s = 1; s <= half; ++s) {
                    b = b + 1 == N ? 0 : b + 1;
                    cfma(x, m[l * P + b], m[b * P + l]);
                }
                if (!(N & 1) && l < N / 2) cfma(x, m[l * P + l + N / 2], m[(l + N / 2) * P + l]);
            }
        } else {   // thread (a, slice of the shifts): kThreads / 128 or more slices
            const int lanes = N <= 64 ? 64 : 128, slices = kThreads / lanes;
            const int a = l % lanes, q = l / lanes;
            if (a < N) {
                for (int s = 1 + q; s <= half; s += slices) {
                    const int b = a + s < N ? a + s : a + s - N;
                    cfma(x, m[a * P + b], m[b * P + a]);
                }
                if (!(N & 1) && q == 0 && a < N / 2) cfma(x, m[a * P + a + N / 2], m[(a + N / 2) * P + a]);
            }
        }
        // four sums over the lanes: two exchanges halve the values a lane carries, three more add
        double v[4] = {tr.re, tr.im, fma(2.0, x.re, xr), fma(2.0, x.im, xi)};
        {
            const bool up = (lane & 16) != 0;
            const double s0 = up ? v[0] : v[2], s1 = up ? v[1] : v[3];
            v[0] = (up ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, s0, 16);
            v[1] = (up ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, s1, 16);
            const bool odd = (lane & 8) != 0;
            const double s2 = odd ? v[0] : v[1];
            v[0] = (odd ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, s2, 8);
        }
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 4);
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
        // lane 0: t.re, 8: t.im, 16: X.re, 24: X.im
        const int64_t o = (i % W) * ldo + n0 + i / W;
        if (GROUP == 32) {
            if ((lane & 7) == 0) reinterpret_cast<double*>((lane & 16) ? X_out + o : t_out + o)[(lane >> 3) & 1] = v[0];
            __syncwarp();
        } else {
            if ((lane & 7) == 0) red[warp][lane >> 3] = v[0];
            __syncthreads();
            if (threadIdx.x < 4) {
                double s = red[0][threadIdx.x];
                for (int q = 1; q < kThreads / 32; ++q) s += red[q][threadIdx.x];
                reinterpret_cast<double*>(threadIdx.x >= 2 ? X_out + o : t_out + o)[threadIdx.x & 1] = s;
            }
            __syncthreads();
        }
    }
}
// N above what shared memory holds
__global__ void __launch_bounds__(kThreads)
    trace_kernel(const cplx* T, int W, int N, int n0, cplx* t_out, cplx* X_out, int64_t ldo) {
    __shared__ cplx sh[kThreads];
    const int w = blockIdx.x, c = blockIdx.y;
    const cplx* Tm = T + ((int64_t)c * W + w) * N * N;
    cplx tr{0.0, 0.0}, x{0.0, 0.0};
    for (int64_t e = threadIdx.x; e < (int64_t)N * N; e += kThreads) {
        const int a = (int)(e / N), b = (int)(e % N);
        const cplx tab = Tm[e];
        cfma(x, tab, Tm[(int64_t)b * N + a]);
        if (a == b) tr = tr + tab;
    }
    tr = block_sum(tr, sh);
    x = block_sum(x, sh);
    if (threadIdx.x == 0) {
        t_out[(int64_t)w * ldo + n0 + c] = tr;
        X_out[(int64_t)w * ldo + n0 + c] = x;
    }
}

// ------------------------------------------------------------------ local energy
__global__ void __launch_bounds__(kThreads) local_energy_kernel(LocalEnergyArgs a) {
    __shared__ cplx sh[kThreads];
    const int w = blockIdx.x;
    cplx e1{0.0, 0.0};
    for (int s = 0; s < 2; ++s) {
        const int Ns = s == 0 ? a.Nup : a.Ndn;
        const cplx* Th = a.Theta[s] + (int64_t)w * a.M * Ns;
        const cplx* ht = a.ht[s] + (a.wper > 0 ? (int64_t)(w / a.wper) * a.ht_stride[s] : 0);
        for (int64_t e = threadIdx.x; e < (int64_t)a.M * Ns; e += kThreads) {
            const int k = (int)(e / Ns), b = (int)(e % Ns);
            cfma(e1, ht[(int64_t)b * a.M + k], Th[e]);
        }
    }
    const double sq = sqrt(a.tau);
    cplx e2{0.0, 0.0};
    const bool energy = a.X[0] != nullptr || a.exch[0] != nullptr;
    for (int n = threadIdx.x; n < a.Nchol; n += kThreads) {
        const int64_t i = (int64_t)w * a.Nchol + n;
        const cplx ts = a.t[0][i] + a.t[1][i];
        if (energy) {
            cfma(e2, ts, ts);
            if (a.X[0]) e2 = e2 - a.X[0][i] - a.X[1][i];
        }
        cplx xb{sq * ts.im, -sq * ts.re};  // -i sqrt(tau) ts
        if (a.fb_cap > 0.0) {
            const double mag = hypot(xb.re, xb.im);
            if (mag > a.fb_cap) xb = (a.fb_cap / mag) * xb;
        }
        if (a.xbar) a.xbar[i] = xb;
    }
    if (energy) {
        e1 = block_sum(e1, sh);
        e2 = block_sum(e2, sh);
        if (threadIdx.x == 0) {
            if (a.exch[0]) e2 = e2 - a.exch[0][w] - a.exch[1][w];
            const cplx E = cplx{a.E0 + e1.re + 0.5 * e2.re, e1.im + 0.5 * e2.im};
            a.E_L[w] = E;
            if (!finite_c(E)) atomicOr(a.flags, FLAG_NONFINITE);
        }
    }
}

// ------------------------------------------------------------------ Philox4x32-10
__device__ __forceinline__ void philox_round(uint32_t& c0, uint32_t& c1, uint32_t& c2, uint32_t& c3,
                                             uint32_t k0, uint32_t k1) {
    const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
    const uint64_t p1 = (uint64_t)0xCD9E8D57u * c2;
    const uint32_t hi0 = (uint32_t)(p0 >> 32), lo0 = (uint32_t)p0;
    const uint32_t hi1 = (uint32_t)(p1 >> 32), lo1 = (uint32_t)p1;
    const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
}

// params (optional, device): {seed, step} read at run time (graph replays), the key being
// params[0] + seed; otherwise seed and step as given.
__global__ void philox_kernel(uint64_t seed, int64_t step, const int64_t* params, int W, int w0, int Nchol,
                              double* x) {
    const int nq = (Nchol + 3) / 4;
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (int64_t)W * nq) return;
    if (params) {
        seed += (uint64_t)params[0];
        step = params[1];
    }
    const int w = (int)(id / nq), q = (int)(id % nq);
    uint32_t c0 = (uint32_t)q, c1 = (uint32_t)(w0 + w), c2 = (uint32_t)step, c3 = 0u;
    uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    for (int r = 0; r < 10; ++r) {
        if (r > 0) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        philox_round(c0, c1, c2, c3, k0, k1);
    }
    const double inv = 2.3283064365386963e-10;  // 2^-32
    const uint32_t o[4] = {c0, c1, c2, c3};
    double* xr = x + (int64_t)w * Nchol;
    for (int p = 0; p < 2; ++p) {
        const double u1 = ((double)o[2 * p] + 0.5) * inv;
        const double u2 = ((double)o[2 * p + 1] + 0.5) * inv;
        const double r = sqrt(-2.0 * log(u1));
        double sn, cs;
        sincospi(2.0 * u2, &sn, &cs);
        const int n = 4 * q + 2 * p;
        if (n < Nchol) xr[n] = r * cs;
        if (n + 1 < Nchol) xr[n + 1] = r * sn;
    }
}

// ------------------------------------------------------------------ small kernels
__global__ void hs_coeff_kernel(const double* x, const cplx* xbar, const cplx* weight, int W, int Nchol,
                                cplx* c, unsigned* flags) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (int64_t)W * Nchol) return;
    const int w = (int)(id / Nchol);
    const double xv = x[id];
    if (!isfinite(xv)) atomicOr(flags, FLAG_NONFINITE);
    const bool alive = weight[w].re != 0.0 || weight[w].im != 0.0;
    c[id] = alive ? cplx{xv - xbar[id].re, -xbar[id].im} : cplx{0.0, 0.0};
}

__global__ void __launch_bounds__(kThreads) weight_kernel(WeightArgs a) {
    __shared__ cplx sh[kThreads];
    const int w = blockIdx.x;
    cplx s{0.0, 0.0};
    for (int n = threadIdx.x; n < a.Nchol; n += kThreads) {
        const int64_t i = (int64_t)w * a.Nchol + n;
        const cplx xb = a.xbar[i];
        // x xbar - xbar^2 / 2
        s = s + a.x[i] * xb;
        cfma(s, cplx{-0.5, 0.0} * xb, xb);
    }
    s = block_sum(s, sh);
    if (threadIdx.x != 0) return;
    const cplx w0 = a.weight[w];
    const bool alive = w0.re != 0.0 || w0.im != 0.0;
    if (!alive) { a.accept[w] = 0; return; }
    const cplx ln = a.logS_new[w];
    if (!finite_c(ln)) { a.accept[w] = 0; a.weight[w] = cplx{0.0, 0.0}; return; }
    const cplx dl = ln - a.logS_old[w];
    const cplx ex = cplx{dl.re + s.re + a.tau * (a.E_T - a.E0), dl.im + s.im};
    if (a.mode == AFQMC_WEIGHT_FREE) {
        const double m = exp(ex.re);
        a.weight[w] = w0 * cplx{m * cos(ex.im), m * sin(ex.im)};
    } else if (a.mode == AFQMC_WEIGHT_LOCAL) {
        // exp(-tau (E_b - E_T)), E_b the pre-step Re E_L bounded to E_T +- ebound
        const double el = a.E_L[w].re;
        if (!(el == el)) { a.accept[w] = 0; a.weight[w] = cplx{0.0, 0.0}; return; }
        const double eb = fmin(fmax(el, a.E_T - a.ebound), a.E_T + a.ebound);
        const double c = cos(dl.im);
        a.weight[w] = cplx{w0.re * exp(-a.tau * (eb - a.E_T)) * (c > 0.0 ? c : 0.0), 0.0};
    } else {
        const double c = cos(dl.im);
        a.weight[w] = cplx{w0.re * exp(ex.re) * (c > 0.0 ? c : 0.0), 0.0};
    }
    a.accept[w] = 1;
}

__global__ void commit_kernel(cplx* Phi, const cplx* Phi_new, const int* accept, int W, int64_t per) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (int64_t)W * per) return;
    if (accept[id / per]) Phi[id] = Phi_new[id];
}

__global__ void __launch_bounds__(kThreads)
    qr_kernel(cplx* Phi, int64_t stride, int M, int N, const cplx* weight) {
    extern __shared__ unsigned char smem_raw[];
    cplx* v = reinterpret_cast<cplx*>(smem_raw);  // M
    cplx* r = v + M;                              // N
    __shared__ double shd[kThreads];
    const int w = blockIdx.x;
    if (weight[w].re == 0.0 && weight[w].im == 0.0) return;
    cplx* Q = Phi + (int64_t)w * stride;
    const int t = threadIdx.x;
    for (int j = 0; j < N; ++j) {
        for (int k = t; k < M; k += kThreads) v[k] = Q[(int64_t)k * N + j];
        __syncthreads();
        for (int pass = 0; pass < 2; ++pass) {
            for (int i = t; i < j; i += kThreads) {
                cplx acc{0.0, 0.0};
                for (int k = 0; k < M; ++k) cfma(acc, conjg(Q[(int64_t)k * N + i]), v[k]);
                r[i] = acc;
            }
            __syncthreads();
            for (int k = t; k < M; k += kThreads) {
                cplx acc = v[k];
                for (int i = 0; i < j; ++i) cfma(acc, cplx{0.0, 0.0} - Q[(int64_t)k * N + i], r[i]);
                v[k] = acc;
            }
            __syncthreads();
        }
        double nrm = 0.0;
        for (int k = t; k < M; k += kThreads) nrm += v[k].re * v[k].re + v[k].im * v[k].im;
        nrm = block_sum_d(nrm, shd);
        const double inv = 1.0 / sqrt(nrm);
        for (int k = t; k < M; k += kThreads) Q[(int64_t)k * N + j] = inv * v[k];
        __syncthreads();
    }
}

// E_mix = sum_w w E_L / sum_w w (fixed-order FP64); with `sums` also the two partial sums, from
// which processes holding parts of one population combine their E_mix.
__global__ void __launch_bounds__(kThreads) emix_kernel(const cplx* weight, const cplx* E_L, int W, cplx* out,
                                                        cplx* sums) {
    __shared__ cplx sh[kThreads];
    cplx num{0.0, 0.0}, den{0.0, 0.0};
    for (int w = threadIdx.x; w < W; w += kThreads) {
        cfma(num, weight[w], E_L[w]);
        den = den + weight[w];
    }
    num = block_sum(num, sh);
    den = block_sum(den, sh);
    if (threadIdx.x == 0) {
        out[0] = cdiv(num, den);
        if (sums) {
            sums[0] = num;
            sums[1] = den;
        }
    }
}

__global__ void fill_kernel(cplx* p, int64_t n, cplx v) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id < n) p[id] = v;
}

__global__ void replicate_kernel(cplx* dst, const cplx* src, int64_t n, int copies, int64_t dst_stride) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= n * copies) return;
    const int c = (int)(id / n);
    const int64_t e = id % n;
    dst[c * dst_stride + e] = src[e];
}

__global__ void r2c_kernel(const double* s, cplx* d, int64_t n) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id < n) d[id] = cplx{s[id], 0.0};
}

__global__ void finite_kernel(const double* p, int64_t n, unsigned* flags) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id < n && !isfinite(p[id])) atomicOr(flags, FLAG_NONFINITE);
}

__global__ void sym_kernel(const double* L, int M, int Nchol, unsigned* flags) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (int64_t)Nchol * M * M) return;
    const int n = (int)(id / ((int64_t)M * M));
    const int64_t e = id % ((int64_t)M * M);
    const int i = (int)(e / M), k = (int)(e % M);
    if (k <= i) return;
    const double a = L[id], b = L[(int64_t)n * M * M + (int64_t)k * M + i];
    if (fabs(a - b) > 1e-10 * fmax(1.0, fabs(a))) atomicOr(flags, 8u);
}

__global__ void hprime_reduce_kernel(const double* h, const cplx* parts, int nparts, int M, double* hp) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (int64_t)M * M) return;
    double acc = 0.0;
    for (int p = 0; p < nparts; ++p) acc += parts[(int64_t)p * M * M + id].re;
    hp[id] = h[id] - 0.5 * acc;
}

// Hermitian split of general complex Cholesky vectors (Sec. V, Eq. (3) with complex L_n):
// V[2n] = (L_n + L_n^+)/2, V[2n+1] = (L_n - L_n^+)/(2i).  Both are Hermitian and
// sum_m V_m (x) V_m is the two-body operator of sum_n L_n (x) L_n^+ up to the exchange of the
// two electrons, which the antisymmetric fermion pair cannot see.
__global__ void herm_split_kernel(const cplx* L, int M, int Nchol, cplx* V) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t mm = (int64_t)M * M;
    if (id >= (int64_t)Nchol * mm) return;
    const int64_t n = id / mm, e = id % mm;
    const int i = (int)(e / M), k = (int)(e % M);
    const cplx a = L[id];
    const cplx b = conjg(L[n * mm + (int64_t)k * M + i]);   // (L_n^+)_ik
    const cplx d = a - b;
    V[2 * n * mm + e] = 0.5 * (a + b);
    V[(2 * n + 1) * mm + e] = cplx{0.5 * d.im, -0.5 * d.re};   // d / (2i)
}

__global__ void hprime_reduce_c_kernel(const double* h, const cplx* parts, int nparts, int M, cplx* hp) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (int64_t)M * M) return;
    cplx acc{0.0, 0.0};
    for (int p = 0; p < nparts; ++p) acc = acc + parts[(int64_t)p * M * M + id];
    hp[id] = cplx{h[id] - 0.5 * acc.re, -0.5 * acc.im};
}

__device__ __forceinline__ cplx clog(cplx z) { return cplx{log(hypot(z.re, z.im)), atan2(z.im, z.re)}; }
__device__ __forceinline__ cplx cexp(cplx z) {
    const double r = exp(z.re);
    return cplx{r * cos(z.im), r * sin(z.im)};
}
__device__ __forceinline__ bool usable(cplx c, cplx l) {
    return (c.re != 0.0 || c.im != 0.0) && isfinite(l.re) && isfinite(l.im);
}

__global__ void __launch_bounds__(kThreads) msd_combine_kernel(MsdArgs a) {
    __shared__ cplx u[kMaxDets];
    __shared__ cplx sh[kThreads];
    const int w = blockIdx.x;
    if (w == 0 && threadIdx.x == 0 && a.inv_flags && (*a.inv_flags & FLAG_NONFINITE))
        atomicOr(a.flags, FLAG_NONFINITE);
    if (threadIdx.x == 0) {
        double m = -INFINITY;
        for (int I = 0; I < a.ND; ++I) {
            const cplx l = a.ls[(int64_t)I * a.ldw + w];
            if (usable(a.cc[I], l)) m = fmax(m, (clog(a.cc[I]) + l).re);
        }
        cplx Z{0.0, 0.0};
        for (int I = 0; I < a.ND; ++I) {
            const cplx l = a.ls[(int64_t)I * a.ldw + w];
            u[I] = usable(a.cc[I], l) ? cexp(clog(a.cc[I]) + l - cplx{m, 0.0}) : cplx{0.0, 0.0};
            Z = Z + u[I];
        }
        if (Z.re == 0.0 && Z.im == 0.0) {
            atomicOr(a.flags, FLAG_SINGULAR);
            a.logS[w] = cplx{-INFINITY, 0.0};
        } else {
            const cplx lz = clog(Z);
            a.logS[w] = cplx{m + lz.re, lz.im};
            for (int I = 0; I < a.ND; ++I) u[I] = cdiv(u[I], Z);
        }
    }
    __syncthreads();
    if (a.E) {
        cplx e{0.0, 0.0};
        for (int I = threadIdx.x; I < a.ND; I += kThreads)
            if (u[I].re != 0.0 || u[I].im != 0.0) e = e + u[I] * a.E[(int64_t)I * a.ldw + w];
        e = block_sum(e, sh);
        if (threadIdx.x == 0) {
            a.E_L[w] = e;
            if (!finite_c(e)) atomicOr(a.flags, FLAG_NONFINITE);
        }
    }
    if (a.t) {
        const double sq = sqrt(a.tau);
        for (int n = threadIdx.x; n < a.Nchol; n += kThreads) {
            cplx ts{0.0, 0.0};
            for (int I = 0; I < a.ND; ++I)
                if (u[I].re != 0.0 || u[I].im != 0.0) ts = ts + u[I] * a.t[((int64_t)I * a.ldw + w) * a.Nchol + n];
            cplx xb{sq * ts.im, -sq * ts.re};  // -i sqrt(tau) t
            if (a.fb_cap > 0.0) {
                const double mag = hypot(xb.re, xb.im);
                if (mag > a.fb_cap) xb = (a.fb_cap / mag) * xb;
            }
            a.xbar[(int64_t)w * a.Nchol + n] = xb;
        }
    }
}

__global__ void msd_variational_kernel(const cplx* cc, const cplx* E, const cplx* L, int ND, cplx* out) {
    double m = -INFINITY;
    for (int I = 0; I < ND; ++I)
        for (int J = 0; J < ND; ++J) {
            const cplx l = L[(int64_t)I * ND + J];
            if (usable(cc[I], l) && (cc[J].re != 0.0 || cc[J].im != 0.0))
                m = fmax(m, (clog(cc[I]) + clog(conjg(cc[J])) + l).re);
        }
    cplx num{0.0, 0.0}, den{0.0, 0.0};
    for (int I = 0; I < ND; ++I)
        for (int J = 0; J < ND; ++J) {
            const cplx l = L[(int64_t)I * ND + J];
            if (!usable(cc[I], l) || (cc[J].re == 0.0 && cc[J].im == 0.0)) continue;
            const cplx f = cexp(clog(cc[I]) + clog(conjg(cc[J])) + l - cplx{m, 0.0});
            num = num + f * E[(int64_t)I * ND + J];
            den = den + f;
        }
    *out = cdiv(num, den);
}

__global__ void cplx_add_kernel(const cplx* a, const cplx* b, cplx* d, int64_t n) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id < n) d[id] = a[id] + b[id];
}

__global__ void c2r_scale_kernel(const cplx* s, double* d, int64_t n) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id < n) d[id] = s[id].re;
}

__global__ void add_identity_kernel(cplx* A, int M, double s) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < M) A[(int64_t)i * M + i].re += s;
}

__global__ void raise_status_kernel(unsigned* flags, unsigned bits) { atomicOr(flags, bits); }

inline unsigned blocks_for(int64_t n, int t = kThreads) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// ================================================================== launchers
// 32 x 32 tiles when they cover the output with at most 60% of the 64 x 64 tiles' area (small
// blocks of few-electron systems), 64 x 64 otherwise.
static int zgemm_tile(const GemmArgs& g) {
    const int64_t a64 = (int64_t)((g.m + 63) / 64) * ((g.n + 63) / 64) * 4096;
    const int64_t a32 = (int64_t)((g.m + 31) / 32) * ((g.n + 31) / 32) * 1024;
    return 10 * a32 <= 6 * a64 ? 32 : 64;
}

// The form of a product, by estimated time (microseconds; constants fitted to products of M = 24 to
// 128, N = 5 to 32, W = 2 to 512):
//   * 0, tiles: the padded multiply-adds at 85% of the FP64 pipe (5.2e5 a microsecond over all SMs), no less than one
//     tile's on its SM;
//   * 2, one output per thread (3, 4: by four or eight): the multiply-adds alone, at 3.0e5 a microsecond, and the latency of
//     its loads along K;
//   * 1, the tensor cores (where the caller gives a workspace): slice_gemm_us, gemm_slices.cu.
int zgemm_form(const GemmArgs& g, const SliceScratch* ws) {
    const double nbatch = (double)g.nb0 * g.nb1 * g.nb2;
    const double per = (g.A.real ? 1.0 : 2.0) * (g.B.real ? 1.0 : 2.0) * g.k;   // multiply-adds an output
    const int ts = zgemm_tile(g);
    const double tiles = nbatch * ((g.m + ts - 1) / ts) * ((g.n + ts - 1) / ts);
    const double tiled_us = 3.0 + ceil(tiles / tc_num_sms()) * ts * ts * per / 3.4e3;
    const double outputs = nbatch * g.m * g.n;
    const double thread_us = outputs < 2e9 ? 3.0 + std::max(outputs * per / 3.0e5, 0.05 * g.k) + 0.01 * g.k : 1e30;
    const double slice_us = ws && ws->buf && g.k > 0 ? slice_gemm_us(g) : 1e30;
    if (slice_us < std::min(tiled_us, thread_us)) return 1;
    if (thread_us >= tiled_us) return 0;
    // threads to an output while one each would leave schedulers without a warp: their pipes' work is
    // the same, in more and shorter chains
    const double room = 128.0 * tc_num_sms();
    return outputs * 4 <= room && g.k >= 16 ? 4 : (outputs <= room && g.k >= 8 ? 3 : 2);
}

void zgemm_as(const GemmArgs& g, int form, cudaStream_t st) {
    if (g.m <= 0 || g.n <= 0) return;
    if (form == 1) {
        slice_gemm(g, g.ws, st);
        return;
    }
    if (g.ws) g.ws->a = g.ws->b = SliceScratch::Packed{};   // no slices for the next product to keep
    const int64_t nbatch = (int64_t)g.nb0 * g.nb1 * g.nb2;
    count_launch();
    if (form >= 2) {
        const int64_t outputs = nbatch * g.m * g.n;
        auto go = [&](auto p1, auto p4, auto p8) {
            const int p = form == 4 ? 8 : form == 3 ? 4 : 1;
            const unsigned blocks = (unsigned)((outputs * p + kSmallT - 1) / kSmallT);
            (p == 8 ? p8 : p == 4 ? p4 : p1)<<<blocks, kSmallT, 0, st>>>(g, (uint32_t)outputs);
        };
        if (g.A.real && g.B.real) go(zgemm_small_kernel<true, true, 1>, zgemm_small_kernel<true, true, 4>, zgemm_small_kernel<true, true, 8>);
        else if (g.A.real) go(zgemm_small_kernel<true, false, 1>, zgemm_small_kernel<true, false, 4>, zgemm_small_kernel<true, false, 8>);
        else if (g.B.real) go(zgemm_small_kernel<false, true, 1>, zgemm_small_kernel<false, true, 4>, zgemm_small_kernel<false, true, 8>);
        else go(zgemm_small_kernel<false, false, 1>, zgemm_small_kernel<false, false, 4>, zgemm_small_kernel<false, false, 8>);
        return;
    }
    const int ts = zgemm_tile(g);
    dim3 grid((g.n + ts - 1) / ts, (g.m + ts - 1) / ts, (unsigned)std::min<int64_t>(nbatch, 65535));
    auto go = [&](auto k32, auto k64) {
        if (ts == 32) k32<<<grid, kThreads, 0, st>>>(g);
        else k64<<<grid, kThreads, 0, st>>>(g);
    };
    if (g.A.real && g.B.real) go(zgemm_kernel<true, true, 32>, zgemm_kernel<true, true, 64>);
    else if (g.A.real) go(zgemm_kernel<true, false, 32>, zgemm_kernel<true, false, 64>);
    else if (g.B.real) go(zgemm_kernel<false, true, 32>, zgemm_kernel<false, true, 64>);
    else go(zgemm_kernel<false, false, 32>, zgemm_kernel<false, false, 64>);
}

void raise_status(unsigned* flags, unsigned bits, cudaStream_t st) {
    count_launch();
    raise_status_kernel<<<1, 1, 0, st>>>(flags, bits);
}

void zgemm(const GemmArgs& g, cudaStream_t st) {
    if (g.m <= 0 || g.n <= 0) return;
    zgemm_as(g, zgemm_form(g, g.ws), st);
}

void batched_inverse_logdet(cplx* S, int64_t stride, int N, int count, cplx* logdet, bool with_inverse,
                            unsigned* flags, cudaStream_t st, bool float_float) {
    if (count <= 0) return;
    const int variant = launch_policy().gj_variant;   // 0 auto, 1 shared memory, 2 registers, 3 float-float
    if (with_inverse && N > 32 && N <= 2 * kGJRegCols && variant != 1) {
        const bool ff = variant == 3 || (variant == 0 && float_float);
        count_launch();
        if (N <= kGJRegCols) {
            if (ff) gj_reg_kernel<NumFF, 1, 2, 8><<<count, kGJRegThreads<8>, 0, st>>>(S, stride, N, logdet, flags);
            else gj_reg_kernel<NumD, 1, 2, 4><<<count, kGJRegThreads<4>, 0, st>>>(S, stride, N, logdet, flags);
            return;
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)count * 2);
        cfg.blockDim = dim3(kGJRegThreads<4>);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        if (ff) cudaLaunchKernelEx(&cfg, gj_reg_kernel<NumFF, 2, 4, 4>, S, stride, N, logdet, flags);
        else cudaLaunchKernelEx(&cfg, gj_reg_kernel<NumD, 2, 4, 4>, S, stride, N, logdet, flags);
        return;
    }
    // one warp per matrix up to 32 rows (variant 1 keeps the shared-memory kernel reachable for
    // comparison; it serves log-determinants of 32 < N <= 128)
    if (N <= kGJWarpMax && variant != 1) {
        const unsigned grid = (unsigned)((count + kGJWarps - 1) / kGJWarps);
        count_launch();
        // a team of warps to a matrix while the matrices leave schedulers idle (up to 4 an SM: 512
        // of N = 32 0.25 -> 0.20 ms, 1024 0.33 -> 0.38)
        if (variant != 4 && (variant == 5 || count <= 4 * tc_num_sms())) {
            auto team = [&](auto inv, auto log_only) {
                if (with_inverse) inv<<<(unsigned)count, 32 * kGJTeam, 0, st>>>(S, stride, N, logdet, flags);
                else log_only<<<(unsigned)count, 32 * kGJTeam, 0, st>>>(S, stride, N, logdet, flags);
            };
            if (N <= 8) team(gj_team_kernel<8, true>, gj_team_kernel<8, false>);
            else if (N <= 16) team(gj_team_kernel<16, true>, gj_team_kernel<16, false>);
            else if (N <= 24) team(gj_team_kernel<24, true>, gj_team_kernel<24, false>);
            else team(gj_team_kernel<32, true>, gj_team_kernel<32, false>);
            return;
        }
        auto go = [&](auto inv, auto log_only) {
            if (with_inverse) inv<<<grid, 32 * kGJWarps, 0, st>>>(S, stride, N, count, logdet, flags);
            else log_only<<<grid, 32 * kGJWarps, 0, st>>>(S, stride, N, count, logdet, flags);
        };
        if (N <= 8) go(gj_warp_kernel<8, true>, gj_warp_kernel<8, false>);
        else if (N <= 16) go(gj_warp_kernel<16, true>, gj_warp_kernel<16, false>);
        else if (N <= 24) go(gj_warp_kernel<24, true>, gj_warp_kernel<24, false>);
        else go(gj_warp_kernel<32, true>, gj_warp_kernel<32, false>);
        return;
    }
    if (N <= kGJSmemMax) {
        const int C = N <= kGJSmemOne ? 1 : 2;
        const int H = (N + C - 1) / C;
        const int cols = (H + 31) / 32;
        const size_t sm = (size_t)N * H * sizeof(cplx) + (size_t)(N + H) * sizeof(cplx) + 2 * N * sizeof(int);
        const int wi = with_inverse ? 1 : 0;
        count_launch();
        if (C == 1) {
            auto launch1 = [&](auto kern) {
                raise_dyn_smem(kern, sm);
                kern<<<count, kGJT, sm, st>>>(S, stride, N, logdet, wi, flags);
            };
            if (cols == 1) launch1(gj_smem_kernel<1, 1>);
            else if (cols == 2) launch1(gj_smem_kernel<1, 2>);
            else launch1(gj_smem_kernel<1, 3>);
        } else {
            raise_dyn_smem(gj_smem_kernel<2, 2>, sm);
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)count * 2);
            cfg.blockDim = dim3(kGJT);
            cfg.dynamicSmemBytes = sm;
            cfg.stream = st;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = 2;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            cudaLaunchKernelEx(&cfg, gj_smem_kernel<2, 2>, S, stride, N, logdet, wi, flags);   // H <= 64
        }
        return;
    }
    const size_t sm = (size_t)N * (2 * sizeof(cplx) + sizeof(int));
    count_launch();
    gj_kernel<<<count, kThreads, sm, st>>>(S, stride, N, logdet, with_inverse ? 1 : 0, flags);
}

void trace_terms(const cplx* T, int nc, int W, int N, int n0, cplx* t_out, cplx* X_out, int64_t ldo,
                 cudaStream_t st) {
    const int64_t count = (int64_t)nc * W;
    if (count <= 0) return;
    const int P = N + (N & 1);
    const size_t one = (size_t)N * P * sizeof(cplx);
    auto go = [&](auto kern, int threads, int groups, int ctas) {
        raise_dyn_smem(kern, one * groups);
        const int64_t grid = std::min<int64_t>((count + groups - 1) / groups, ctas);
        count_launch();
        kern<<<(unsigned)grid, threads, one * groups, st>>>(T, count, W, N, n0, t_out, X_out, ldo);
    };
    // CTAs: as many as shared memory lets an SM hold, on every SM, a few rounds each
    const int sms = tc_num_sms();
    if (N <= 32) {
        // one CTA of twelve matrices where two of eight do not fit an SM (N = 32: 3.9 -> 3.6 ms a step)
        if (2 * 8 * one > 220000)
            go(trace_pairs_kernel<32, 384>, 384, 12, sms * 4);
        else
            go(trace_pairs_kernel<32, kThreads>, kThreads, kThreads / 32,
               sms * std::max(1, std::min(8, (int)(220000 / (one * (kThreads / 32))))) * 4);
        return;
    }
    if (one <= 220000) {   // N <= 117
        go(trace_pairs_kernel<kThreads, kThreads>, kThreads, 1, sms * std::max(1, std::min(8, (int)(220000 / one))) * 4);
        return;
    }
    dim3 grid(W, nc);
    count_launch();
    trace_kernel<<<grid, kThreads, 0, st>>>(T, W, N, n0, t_out, X_out, ldo);
}

void msd_combine(const MsdArgs& a, cudaStream_t st) {
    count_launch();
    msd_combine_kernel<<<a.W, kThreads, 0, st>>>(a);
}

void msd_variational_energy(const cplx* cc, const cplx* E, const cplx* logS, int ND, cplx* out, cudaStream_t st) {
    count_launch();
    msd_variational_kernel<<<1, 1, 0, st>>>(cc, E, logS, ND, out);
}

void cplx_add(const cplx* a, const cplx* b, cplx* dst, int64_t n, cudaStream_t st) {
    count_launch();
    cplx_add_kernel<<<blocks_for(n), kThreads, 0, st>>>(a, b, dst, n);
}

void local_energy_forcebias(const LocalEnergyArgs& a, cudaStream_t st) {
    count_launch();
    local_energy_kernel<<<a.W, kThreads, 0, st>>>(a);
}

void philox_fields(uint64_t seed, int64_t step, int W, int Nchol, double* x, cudaStream_t st, int w0) {
    const int64_t n = (int64_t)W * ((Nchol + 3) / 4);
    count_launch();
    philox_kernel<<<blocks_for(n), kThreads, 0, st>>>(seed, step, nullptr, W, w0, Nchol, x);
}

void philox_fields_dev(const int64_t* params, uint64_t seed_add, int W, int Nchol, double* x, cudaStream_t st,
                       int w0) {
    const int64_t n = (int64_t)W * ((Nchol + 3) / 4);
    count_launch();
    philox_kernel<<<blocks_for(n), kThreads, 0, st>>>(seed_add, 0, params, W, w0, Nchol, x);
}

void hs_coefficients(const double* x, const cplx* xbar, const cplx* weight, int W, int Nchol, cplx* c,
                     unsigned* flags, cudaStream_t st) {
    count_launch();
    hs_coeff_kernel<<<blocks_for((int64_t)W * Nchol), kThreads, 0, st>>>(x, xbar, weight, W, Nchol, c, flags);
}

// Comb population control on one thread: the running sums must be formed left to right in
// FP64 so that every slot falls in the same interval as in any other implementation of the same
// definition.  Slot k sits at (k + xi) total / W (no fused multiply-add can form here).
__global__ void comb_kernel(const cplx* weight, int W, double xi, int* idx, double* total_out) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double total = 0.0;
    int last = W - 1;
    bool any = false;
    for (int j = 0; j < W; ++j) {
        total += weight[j].re;
        if (weight[j].re > 0.0) { last = j; any = true; }
    }
    if (!any) last = W - 1;
    *total_out = total;
    int j = 0;
    double c = weight[0].re;
    for (int k = 0; k < W; ++k) {
        const double u = ((double)k + xi) * total / (double)W;
        while (j < last && !(c > u)) c += weight[++j].re;
        idx[k] = j;
    }
}
__global__ void gather_rows_kernel(const cplx* src, int64_t per, const int* idx, int W, cplx* dst) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)W * per) return;
    const int64_t w = i / per, e = i % per;
    dst[i] = src[(int64_t)idx[w] * per + e];
}
__global__ void equal_weights_kernel(cplx* weight, int W, const double* total) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w < W) weight[w] = cplx{*total / (double)W, 0.0};
}

void comb_indices(const cplx* weight, int W, double xi, int* idx, double* total, cudaStream_t st) {
    count_launch();
    comb_kernel<<<1, 32, 0, st>>>(weight, W, xi, idx, total);
}
void gather_rows(const cplx* src, int64_t per, const int* idx, int W, cplx* dst, cudaStream_t st) {
    const int64_t n = (int64_t)W * per;
    if (n <= 0) return;
    count_launch();
    gather_rows_kernel<<<(unsigned)((n + kThreads - 1) / kThreads), kThreads, 0, st>>>(src, per, idx, W, dst);
}
void equal_weights(cplx* weight, int W, const double* total, cudaStream_t st) {
    count_launch();
    equal_weights_kernel<<<(W + kThreads - 1) / kThreads, kThreads, 0, st>>>(weight, W, total);
}

void weight_update(const WeightArgs& a, cudaStream_t st) {
    count_launch();
    weight_kernel<<<a.W, kThreads, 0, st>>>(a);
}

void commit_walkers(cplx* Phi, const cplx* Phi_new, const int* accept, int W, int64_t per, cudaStream_t st) {
    count_launch();
    commit_kernel<<<blocks_for((int64_t)W * per), kThreads, 0, st>>>(Phi, Phi_new, accept, W, per);
}

void qr_reorthonormalise(cplx* Phi, int64_t stride, int M, int N, int W, const cplx* weight,
                         cudaStream_t st) {
    const size_t sm = (size_t)(M + N) * sizeof(cplx);
    count_launch();
    qr_kernel<<<W, kThreads, sm, st>>>(Phi, stride, M, N, weight);
}

void mixed_energy(const cplx* weight, const cplx* E_L, int W, cplx* out, cudaStream_t st, cplx* sums) {
    count_launch();
    emix_kernel<<<1, kThreads, 0, st>>>(weight, E_L, W, out, sums);
}

void fill_cplx(cplx* p, int64_t n, cplx v, cudaStream_t st) {
    if (n > 0) count_launch();
    if (n > 0) fill_kernel<<<blocks_for(n), kThreads, 0, st>>>(p, n, v);
}

void replicate(cplx* dst, const cplx* src, int64_t n, int copies, int64_t dst_stride, cudaStream_t st) {
    count_launch();
    replicate_kernel<<<blocks_for(n * copies), kThreads, 0, st>>>(dst, src, n, copies, dst_stride);
}

void real_to_cplx(const double* src, cplx* dst, int64_t n, cudaStream_t st) {
    count_launch();
    r2c_kernel<<<blocks_for(n), kThreads, 0, st>>>(src, dst, n);
}

void check_finite(const double* p, int64_t n, unsigned* flags, cudaStream_t st) {
    if (n > 0) count_launch();
    if (n > 0) finite_kernel<<<blocks_for(n), kThreads, 0, st>>>(p, n, flags);
}

void check_symmetric(const double* L, int M, int Nchol, unsigned* flags, cudaStream_t st) {
    const int64_t n = (int64_t)Nchol * M * M;
    count_launch();
    sym_kernel<<<blocks_for(n), kThreads, 0, st>>>(L, M, Nchol, flags);
}

namespace {

// sum_n L_n L_n^+ for symmetric (real) or Hermitian (complex) L_n, in `parts` partial sums:
// for such L_n it equals X^+ X with X[(n, k)][i] = L[n][k][i], a contiguous [Nchol*M][M]
// matrix.  The K = Nchol*M reduction is split into `parts` GEMMs (fixed split, reduced in a
// fixed order by the caller's kernel) to fill the GPU.  gram_parts: two CTAs a SM over the
// output's tiles, at least 4 vectors a part beyond 16; and 16 in any case, which bounds the length of a part's
// sum (2560 vectors of M = 512 in five parts: errors of 1.9e-14 relative on the diagonal, in sixteen
// 0.75e-14).  Returns the workspace, or NULL.
int gram_parts(int M, int Nchol) {
    const int tiles = ((M + 63) / 64) * ((M + 63) / 64), fill = (2 * tc_num_sms() + tiles - 1) / tiles;
    return std::max({1, std::min(Nchol, 16), std::min({Nchol, fill, Nchol / 4})});
}

cplx* gram_of_cholesky(const void* L, bool real, int M, int Nchol, int parts, cudaStream_t st) {
    const int per = (Nchol + parts - 1) / parts;  // Cholesky vectors per part
    cplx* buf = nullptr;
    if (cudaMallocAsync(&buf, sizeof(cplx) * (size_t)parts * M * M, st) != cudaSuccess) {
        fail(AFQMC_ERR_OOM, "hprime workspace");
        return nullptr;
    }
    fill_cplx(buf, (int64_t)parts * M * M, cplx{0.0, 0.0}, st);
    // every full part in one launch (64 x 64 tiles of one part alone would leave most SMs idle),
    // then the rest
    const int whole = Nchol / per, rest = Nchol - whole * per;
    auto run = [&](int first, int count, int vectors) {
        if (count < 1 || vectors < 1) return;
        GemmArgs g;
        g.m = g.n = M;
        g.k = vectors * M;
        g.nb1 = count;
        const int64_t off = (int64_t)first * per * M * M;
        const void* X = real ? (const void*)(static_cast<const double*>(L) + off)
                             : (const void*)(static_cast<const cplx*>(L) + off);
        g.A.ptr = X; g.A.real = real; g.A.op = real ? OP_T : OP_C; g.A.ld = M; g.A.s1 = (int64_t)per * M * M;
        g.B.ptr = X; g.B.real = real; g.B.op = OP_N; g.B.ld = M; g.B.s1 = (int64_t)per * M * M;
        g.C = buf + (int64_t)first * M * M; g.ldc = M; g.sc1 = (int64_t)M * M;
        zgemm(g, st);
    };
    run(0, whole, per);
    run(whole, 1, rest);
    return buf;
}

}  // namespace

void build_hprime(const double* h, const double* L, int M, int Nchol, double* hp, cudaStream_t st) {
    const int parts = gram_parts(M, Nchol);
    cplx* buf = gram_of_cholesky(L, true, M, Nchol, parts, st);
    if (!buf) return;
    count_launch();
    hprime_reduce_kernel<<<blocks_for((int64_t)M * M), kThreads, 0, st>>>(h, buf, parts, M, hp);
    cudaFreeAsync(buf, st);
}

void build_hprime_hermitian(const double* h, const cplx* V, int M, int Nv, cplx* hp, cudaStream_t st) {
    const int parts = gram_parts(M, Nv);
    cplx* buf = gram_of_cholesky(V, false, M, Nv, parts, st);
    if (!buf) return;
    count_launch();
    hprime_reduce_c_kernel<<<blocks_for((int64_t)M * M), kThreads, 0, st>>>(h, buf, parts, M, hp);
    cudaFreeAsync(buf, st);
}

void hermitian_split(const cplx* L, int M, int Nchol, cplx* V, cudaStream_t st) {
    const int64_t n = (int64_t)Nchol * M * M;
    count_launch();
    herm_split_kernel<<<blocks_for(n), kThreads, 0, st>>>(L, M, Nchol, V);
}

namespace {

// ||X||_1 (largest column sum of |x|) of a device M x M matrix, read on the host.
int norm1_on_host(const void* X, bool real, int M, cudaStream_t st, double* nrm) {
    const size_t n = (size_t)M * M;
    std::vector<cplx> hX(real ? 0 : n);
    std::vector<double> hR(real ? n : 0);
    cudaError_t e = real ? cudaMemcpyAsync(hR.data(), X, sizeof(double) * n, cudaMemcpyDefault, st)
                         : cudaMemcpyAsync(hX.data(), X, sizeof(cplx) * n, cudaMemcpyDefault, st);
    if (e != cudaSuccess) return fail(AFQMC_ERR_CUDA, "expm copy");
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return fail(AFQMC_ERR_CUDA, "expm sync");
    *nrm = 0.0;
    for (int j = 0; j < M; ++j) {
        double c = 0.0;
        for (int i = 0; i < M; ++i)
            c += real ? fabs(hR[(size_t)i * M + j]) : hypot(hX[(size_t)i * M + j].re, hX[(size_t)i * M + j].im);
        *nrm = std::max(*nrm, c);
    }
    return AFQMC_OK;
}

// E = exp(s Y) for a complex device matrix Y with ||Y||_1 = nrm:
// (T_q(s Y / 2^j))^(2^j), Taylor order 18 by Horner, j squarings so that ||s Y / 2^j||_1 <= 1/4
// (truncation error below 1e-20 relative).  E must not alias Y.
int expm_taylor_squaring(const cplx* Y, double nrm, double s, int M, cplx* E, cudaStream_t st) {
    nrm *= fabs(s);
    int sq = 0;
    while (nrm > 0.25 && sq < 60) { nrm *= 0.5; ++sq; }
    const double sc = s / ldexp(1.0, sq);
    cplx* Tm = nullptr;
    cplx* E0 = E;
    if (cudaMallocAsync(&Tm, sizeof(cplx) * M * M, st) != cudaSuccess) return fail(AFQMC_ERR_OOM, "expm workspace");
    // E = I
    fill_cplx(E, (int64_t)M * M, cplx{0.0, 0.0}, st);
    count_launch();
    add_identity_kernel<<<blocks_for(M), kThreads, 0, st>>>(E, M, 1.0);
    const int order = 18;
    for (int k = order; k >= 1; --k) {
        // E <- I + (sc / k) Y E
        GemmArgs g;
        g.m = g.n = g.k = M;
        g.A.ptr = Y; g.A.ld = M;
        g.B.ptr = E; g.B.ld = M;
        g.alpha = cplx{sc / k, 0.0};
        g.C = Tm; g.ldc = M;
        zgemm(g, st);
        count_launch();
        add_identity_kernel<<<blocks_for(M), kThreads, 0, st>>>(Tm, M, 1.0);
        std::swap(E, Tm);
    }
    for (int q = 0; q < sq; ++q) {
        GemmArgs g;
        g.m = g.n = g.k = M;
        g.A.ptr = E; g.A.ld = M;
        g.B.ptr = E; g.B.ld = M;
        g.C = Tm; g.ldc = M;
        zgemm(g, st);
        std::swap(E, Tm);
    }
    if (E != E0) {   // the result sits in the workspace: move it to the caller's buffer
        cudaMemcpyAsync(E0, E, sizeof(cplx) * M * M, cudaMemcpyDeviceToDevice, st);
        Tm = E;
    }
    cudaFreeAsync(Tm, st);
    return AFQMC_OK;
}

}  // namespace

int expm_real(const double* X, double s, int M, double* out, cudaStream_t st) {
    double nrm = 0.0;
    AFQMC_TRY(norm1_on_host(X, true, M, st, &nrm));
    cplx *Y = nullptr, *E = nullptr;
    const size_t bytes = sizeof(cplx) * M * M;
    if (cudaMallocAsync(&Y, bytes, st) != cudaSuccess || cudaMallocAsync(&E, bytes, st) != cudaSuccess) {
        if (Y) cudaFreeAsync(Y, st);
        return fail(AFQMC_ERR_OOM, "expm workspace");
    }
    real_to_cplx(X, Y, (int64_t)M * M, st);
    const int rc = expm_taylor_squaring(Y, nrm, s, M, E, st);
    if (rc == AFQMC_OK) {
        count_launch();
        c2r_scale_kernel<<<blocks_for((int64_t)M * M), kThreads, 0, st>>>(E, out, (int64_t)M * M);
    }
    cudaFreeAsync(Y, st);
    cudaFreeAsync(E, st);
    return rc;
}

int expm_complex(const cplx* X, double s, int M, cplx* out, cudaStream_t st) {
    double nrm = 0.0;
    AFQMC_TRY(norm1_on_host(X, false, M, st, &nrm));
    return expm_taylor_squaring(X, nrm, s, M, out, st);
}

}  // namespace afqmc
