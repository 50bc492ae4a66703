// FP64 matrix products on the tensor cores.
//
// GB300's FP64 pipe does 2 multiply-adds per SM and clock, its fp16 tensor cores ~4096, so a
// product of integers small enough to be summed exactly in fp32 is worth some thirty of them for
// each FP64 one (the splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59 (2012), with
// digits sized for fp16 operands and fp32 accumulators):
//   * Every row of an operand (along the contracted index) gets the exponent e of its largest
//     entry (|x| < 2^e) and each entry is rounded to a fixed-point number of 58 or 59 bits below
//     2^e, cut into S signed digits d_p of BETA bits (|d_p| <= 2^(BETA-1)), the last with 11 bits
//     (its fraction bits included): x = 2^(e - BETA + 1) sum_p d_p 2^(-BETA p).  Every digit is
//     exact in fp16.
//   * The products of digits p and q of equal weight p + q = d go to one tensor-memory accumulator
//     per d < D.  With BETA = 8 for K <= 128 and BETA = 7 for K <= 512 at most 8 x 2^21 bounds
//     every partial sum, so the accumulators are exact integers (the last one, which the
//     fractional digits reach, is rounded 24 bits below its own small weight).  Dropped weights
//     d >= D lie 2^-56 and less below |a||b|.
//   * The epilogue adds the accumulators as one 64-bit integer (its unit 2^-53 of the product of the
//     rows' largest entries, or less) and rounds it to FP64 in integer instructions (a few FP64
//     operations per output would cost as much as the tile's MMAs).
// The result carries the rounding of its operands to 2^-59 of their rows' largest entries, the
// dropped weights and one rounding: against a 128-bit sum the error measured is at most that of
// the multiply-add loop of zgemm_kernel (tests/test_gpu_gemm_slices.py).  Longer contractions run in
// pieces of at most 512, each with its own exponents, added in FP64.
//
// Complex operands become real ones: a real operand times a complex one has the complex one's re
// and im as separate rows; two complex operands are contracted over [re | im] rows of the one
// against the rows [re | -im], [im | re] of the other, the "expanded" one.
// A NaN or infinity anywhere in a row gives NaN in all of its results.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "kernels_fp64.cuh"
#include "kernels_tc.cuh"
#include "tc_ptx.cuh"

namespace afqmc {

using namespace tc;

namespace {

constexpr int kRows = 128;      // tile rows (operand R)
constexpr int kCols = 64;       // tile columns (operand Q): D accumulators of 64 fill tensor memory
constexpr int kChunk = 32;      // contracted entries per stage (64-byte swizzle)
constexpr int kMaxStages = 3;
constexpr int kEpiWarps = 16;   // four per tensor-memory lane quadrant, 16 columns each
constexpr int kThreadsG = 64 + 32 * kEpiWarps;
constexpr int kNanExp = 1 << 20;   // exponent of a row with a NaN or an infinity

// K <= 128: eight-bit digits, 7 slices, 28 products; K <= 512: seven bits, 8 slices, 36 products.
template <int S_>
struct Digits {
    static constexpr int S = S_;
    static constexpr int BETA = S_ == 7 ? 8 : 7;
    static constexpr int D = S_;                       // accumulators (weights 0 .. D - 1)
    static constexpr int kTail = 11;                   // bits of the last digit
    static constexpr int kFrac = kTail - BETA;         // fraction bits of the last digit
    // fixed-point value v = x 2^(kPoint - e): BETA - 1 bits above the first digit's unit
    static constexpr int kPoint = BETA - 1 + BETA * (S - 1) + kFrac;
};
// A stage of one CTA: the R rows of its tile and the Q rows, or half of them for a CTA pair.
template <int S, bool PAIR>
struct Stage {
    static constexpr int kQRows = PAIR ? kCols / 2 : kCols;
    static constexpr int kBytes = S * (kRows + kQRows) * kChunk * 2;
    static constexpr int kCount = 216 * 1024 / kBytes < kMaxStages ? 216 * 1024 / kBytes : kMaxStages;
    static_assert(kCount >= 2, "stage ring");
};
// Place in the ring of stages and the parity of its turn.
template <int N>
struct Ring {
    int st = 0;
    uint32_t phase = 0;
    __device__ __forceinline__ void next() {
        if (++st == N) {
            st = 0;
            phase ^= 1u;
        }
    }
};

// Division of 0 <= x < 2^31 by a fixed divisor d: x / d = (x mul) >> (32 + shift) with mul =
// ceil(2^(32 + shift) / d), shift = ceil(log2 d) - 1 (d > 1), which is exact for such x
// (Granlund and Montgomery, PLDI 1994).
struct Div {
    uint32_t mul = 0, d = 1;
    int shift = 0;
    Div() = default;
    explicit Div(int64_t n) : d((uint32_t)n) {
        if (d <= 1) return;
        while ((1u << (shift + 1)) < d) ++shift;
        mul = (uint32_t)(((1ull << (32 + shift)) + d - 1) / d);
    }
    __device__ __forceinline__ uint32_t div(uint32_t x) const { return d <= 1 ? x : __umulhi(x, mul) >> shift; }
    __device__ __forceinline__ void divmod(uint32_t x, uint32_t& q, uint32_t& r) const {
        q = div(x);
        r = x - q * d;
    }
};

// Index spaces: up to three batch dimensions, each with its count and stride.
struct Dims {
    int64_t cnt[3], str[3];
};
// The same for the device: index i -> sum of digit times stride.
struct Strides {
    Div c1, c2;
    int64_t str[3] = {0, 0, 0};
    Strides() = default;
    explicit Strides(const Dims& d) : c1(d.cnt[1]), c2(d.cnt[2]) {
        for (int i = 0; i < 3; ++i) str[i] = d.str[i];
    }
    __device__ __forceinline__ int64_t at(uint32_t i) const {
        uint32_t q, i0, i1, i2;
        c2.divmod(i, q, i2);
        c1.divmod(q, i0, i1);
        return (int64_t)i0 * str[0] + (int64_t)i1 * str[1] + (int64_t)i2 * str[2];
    }
};

struct PackArgs {
    const void* ptr;
    int real, conj, expand, parts, idx_contig, scale;   // scale: multiply by alpha
    int64_t si, sk;            // element strides of the row index and of the contracted index
    int n, k, koff;            // row index count, contracted length, padded length of one part
    int klen, pieces;          // the contracted index in `pieces` pieces of klen (<= koff)
    int64_t Kp;                // row pitch of the slices (parts x koff)
    Strides own, shared;       // batch dimensions folded into the rows / kept as batches
    Div dn, dbatch;            // by n, by nbatch
    int64_t own_rows;          // rows before expansion
    int64_t nbatch;
    __half* out;               // [S][pieces][nbatch][own_rows (x 2)][Kp]
    int64_t plane;             // elements per slice
    int* exps;                 // [pieces][nbatch][own_rows]
    cplx alpha;
};

__device__ __forceinline__ cplx pack_load(const PackArgs& a, int64_t off) {
    cplx v;
    if (a.real) {
        v = cplx{static_cast<const double*>(a.ptr)[off], 0.0};
    } else {
        const double2 t = static_cast<const double2*>(a.ptr)[off];
        v = cplx{t.x, a.conj ? -t.y : t.y};
    }
    if (a.scale) v = a.real ? cplx{a.alpha.re * v.re, 0.0} : a.alpha * v;
    return v;
}
__device__ __forceinline__ int exp_field(double x) {
    return (int)(((uint32_t)((unsigned long long)__double_as_longlong(x) >> 32) >> 20) & 0x7ffu);
}

// The S digits of x at the row exponent e as fp16 bit patterns.
template <int S>
__device__ __forceinline__ void digits_of(double x, int e, unsigned short (&d)[S]) {
    using P = Digits<S>;
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int E = (int)((b >> 52) & 0x7ffu);
    long long v = 0;
    if (E != 0 && e != kNanExp) {   // subnormals count as zero
        const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
        const int sh = E - 1075 + P::kPoint - e;   // x = m 2^(E - 1075); at most 6
        if (sh >= 0) v = (long long)(m << sh);
        else if (sh > -56) v = (long long)((m + (1ull << (-sh - 1))) >> -sh);
        if (b >> 63) v = -v;
    }
    {   // last digit: 11 bits, in units of 2^-kFrac
        const int t = (int)((v + 1024) & 2047) - 1024;
        v = (v - t) >> 11;
        d[S - 1] = __half_as_ushort(__float2half_rn((float)t * (1.0f / (1 << P::kFrac))));
    }
#pragma unroll
    for (int p = S - 2; p > 0; --p) {
        constexpr int h = 1 << (P::BETA - 1);
        const int t = (int)((v + h) & (2 * h - 1)) - h;
        v = (v - t) >> P::BETA;
        d[p] = __half_as_ushort(__float2half_rn((float)t));
    }
    d[0] = __half_as_ushort(__float2half_rn((float)(int)v));
}

// RB rows per block (8, or 32 of at most 64 entries).  Pass 1 finds each row's exponent, pass 2 takes
// 2048 entries at a time from shared memory (filled coalesced along whichever index is contiguous,
// by pass 1 already if the rows fit) and writes the digits, two neighbours per store.  Most calls
// have a few hundred rows, so a block's chain of loads and digits is the time, not the bytes
// (8 in and 2 S out per entry): 32 rows a block of any length took 83 us for 1024 complex rows of
// 3072 (55 now), 25 for 64 x 32 rows of 128 (9), 13 for 90 real rows of 90 (4).
constexpr int kPackT = 256;
template <int S, int RB>
__global__ void __launch_bounds__(kPackT) pack_slices_kernel(PackArgs a) {
    constexpr int KB = 2048 / RB, KS = kPackT / RB;
    __shared__ cplx tile[RB][KB + 1];
    __shared__ int64_t off[RB];
    __shared__ int rowexp[RB];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t r0 = (int64_t)blockIdx.x * RB, bt = blockIdx.y;   // bt = (piece, shared batch)
    uint32_t piece, sb;
    a.dbatch.divmod(blockIdx.y, piece, sb);
    const int kn = min(a.klen, a.k - (int)piece * a.klen);
    if (tid < RB) {
        const int64_t r = r0 + tid;
        uint32_t ob, i;
        a.dn.divmod((uint32_t)r, ob, i);
        off[tid] = r < a.own_rows ? a.shared.at(sb) + a.own.at(ob) + i * a.si + (int64_t)piece * a.klen * a.sk : -1;
        rowexp[tid] = 0;
    }
    __syncthreads();
    const bool once = a.koff <= KB;
    if (a.idx_contig) {
        const int i = tid % RB;
        int m = 0;
        if (off[i] >= 0) {
#pragma unroll 4
            for (int kk = tid / RB; kk < kn; kk += KS) {
                const cplx v = pack_load(a, off[i] + kk * a.sk);
                m = max(m, max(exp_field(v.re), exp_field(v.im)));
                if (once) tile[i][kk] = v;
            }
            atomicMax(&rowexp[i], m);
        }
    } else {
        for (int i = warp; i < RB; i += kPackT / 32) {
            int m = 0;
            if (off[i] >= 0) {
#pragma unroll 4
                for (int kk = lane; kk < kn; kk += 32) {
                    const cplx v = pack_load(a, off[i] + kk * a.sk);
                    m = max(m, max(exp_field(v.re), exp_field(v.im)));
                    if (once) tile[i][kk] = v;
                }
            }
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) rowexp[i] = m;
        }
    }
    if (once) {
        const int pad = a.koff - kn;   // a few entries
        for (int q = tid; q < RB * pad; q += kPackT) tile[q % RB][kn + q / RB] = cplx{0.0, 0.0};
    }
    __syncthreads();
    if (tid < RB) {
        const int m = rowexp[tid];
        const int e = m == 0x7ff ? kNanExp : (m == 0 ? 0 : m - 1022);   // largest entry < 2^e
        rowexp[tid] = e;
        if (off[tid] >= 0) a.exps[bt * a.own_rows + r0 + tid] = e;
    }
    const int64_t rows = a.own_rows * (a.expand ? 2 : 1);
    for (int k0 = 0; k0 < a.koff; k0 += KB) {
        const int kc = min(KB, a.koff - k0);   // even, as koff is
        __syncthreads();
        if (!once) {
            if (a.idx_contig) {
                const int i = tid % RB;
#pragma unroll 4
                for (int kk = tid / RB; kk < kc; kk += KS) {
                    cplx v{0.0, 0.0};
                    if (off[i] >= 0 && k0 + kk < kn) v = pack_load(a, off[i] + (k0 + kk) * a.sk);
                    tile[i][kk] = v;
                }
            } else {
                for (int i = warp; i < RB; i += kPackT / 32) {
#pragma unroll 4
                    for (int kk = lane; kk < kc; kk += 32) {
                        cplx v{0.0, 0.0};
                        if (off[i] >= 0 && k0 + kk < kn) v = pack_load(a, off[i] + (k0 + kk) * a.sk);
                        tile[i][kk] = v;
                    }
                }
            }
            __syncthreads();
        }
        const int half = kc / 2;
#pragma unroll 1
        for (int q = tid; q < RB * half; q += kPackT) {
            const int i = q / half, kk = 2 * (q - i * half);
            if (off[i] < 0) break;
            const int e = rowexp[i];
            const cplx v0 = tile[i][kk], v1 = tile[i][kk + 1];
            unsigned short x[S], y[S];
            unsigned re[S], im[S];
            digits_of<S>(v0.re, e, x);
            digits_of<S>(v1.re, e, y);
#pragma unroll
            for (int p = 0; p < S; ++p) re[p] = (unsigned)x[p] | ((unsigned)y[p] << 16);
            if (!a.real) {
                digits_of<S>(v0.im, e, x);
                digits_of<S>(v1.im, e, y);
#pragma unroll
                for (int p = 0; p < S; ++p) im[p] = (unsigned)x[p] | ((unsigned)y[p] << 16);
            }
            const int64_t r = r0 + i;
            const int64_t row = (bt * rows + (a.expand ? 2 * r : r)) * a.Kp + k0 + kk;
#pragma unroll
            for (int p = 0; p < S; ++p) {
                __half* o = a.out + p * a.plane + row;
                *reinterpret_cast<unsigned*>(o) = re[p];
                if (a.real) continue;
                if (a.parts == 2) *reinterpret_cast<unsigned*>(o + a.koff) = a.expand ? im[p] ^ 0x80008000u : im[p];
                if (a.expand) {
                    *reinterpret_cast<unsigned*>(o + a.Kp) = im[p];
                    if (a.parts == 2) *reinterpret_cast<unsigned*>(o + a.Kp + a.koff) = re[p];
                }
            }
        }
    }
}

struct OutArgs {
    int64_t rows, cols;        // per batch, after expansion
    int rexp, cexp;            // which side is expanded (at most one)
    Div rn, cn;                // row / column index counts within one own batch
    int64_t rs, cs;            // output strides of the row / column index (complex elements)
    Strides rown, cown, shared;    // output strides of the batch dimensions
    Strides drown, dcown, dshared;
    int64_t drs, dcs;
    const int *er, *ec;        // exponents [pieces][nbatch][rows before expansion]
    cplx *C, *D;
    double beta;
    int64_t tiles;             // row tiles x column tiles x batches
    Div drt, dper, dtiles;     // by row tiles, tiles of a batch, all tiles
    int nk;                    // stages of one piece
    int pieces;                // pieces of the contracted index
    int64_t nbatch;            // shared batches
    // few tiles and a long contraction: `groups` CTAs share a tile's pieces (pg each) and write
    // their sums to C + group * gstride
    int groups, pg;
    int64_t gstride;
    __device__ __forceinline__ void tile(uint32_t t, uint32_t& b, uint32_t& ct, uint32_t& rt) const {
        uint32_t q;
        dper.divmod(t, b, q);
        drt.divmod(q, ct, rt);
    }
};

struct Ctl {
    uint64_t full[kMaxStages], empty[kMaxStages], tfull, tempty, done;
    uint32_t tmem_base;
    int abort;
};

// FP64 value of I 2^x, rounded to nearest.  The common case, a result well inside the exponent range
// with |I| >= 2^32, takes one count of leading zeros and two funnel shifts; the other (small and zero
// I; x beyond the range: 0, infinity or, from a row marked kNanExp, NaN) is out of line.
__device__ __noinline__ double round64_rare(unsigned hi0, unsigned lo0, unsigned sign, int x) {
    const unsigned long long X0 = ((unsigned long long)hi0 << 32) | lo0;
    if (x > kNanExp / 2) return __longlong_as_double(0x7ff8000000000000ll);
    if (X0 == 0) return 0.0;
    const int lz = __clzll((long long)X0);
    const unsigned long long X = X0 << lz, m = (X >> 11) + ((X >> 10) & 1ull);   // 2^52 .. 2^53
    const int eb = 1023 + 63 - lz + x;
    const unsigned long long r = eb < 1 ? 0ull : (eb > 2046 ? 0x7ff0000000000000ull : ((unsigned long long)(eb - 1) << 52) + m);
    return __longlong_as_double((long long)(r | ((unsigned long long)sign << 32)));
}
__device__ __forceinline__ double round64(long long I, int x) {
    const int s = (int)(I >> 63);
    const unsigned long long X = (unsigned long long)((I ^ s) - s);
    const unsigned hi0 = (unsigned)(X >> 32), lo0 = (unsigned)X, sign = (unsigned)s & 0x80000000u;
    const int lz = __clz((int)hi0);
    const int eb1 = 1023 + 63 - 1 + x - lz;   // biased exponent - 1
    if (hi0 == 0u || (unsigned)eb1 > 2045u) return round64_rare(hi0, lo0, sign, x);
    const unsigned hi = __funnelshift_l(lo0, hi0, lz), lo = lo0 << lz;
    // bits 63 .. 11 plus the rounding bit; the leading one carries into the exponent field
    const unsigned long long m = (((unsigned long long)(hi >> 11) << 32) | __funnelshift_r(lo, hi, 11)) + ((lo >> 10) & 1u);
    return __hiloint2double((int)(((unsigned)(m >> 32) + ((unsigned)eb1 << 20)) | sign), (int)(unsigned)m);
}

// Barrier of the epilogue warps with the conjunction of `pred`.
__device__ __forceinline__ int epi_and(int pred) {
    int r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.s32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 2, 512, p;\n\t"
        "selp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(pred)
        : "memory");
    return r;
}

// One output's accumulators a_d 2^(-BETA d) as an integer in units of 2^-kGather of accumulator 0's:
// 62 or 63 bits, the lowest 2^-54 (S = 7) or 2^-53 (S = 8) of the product of the rows' largest
// entries.  Every sum below is exact but the last, of the two smallest accumulators.
template <int S>
struct Gather {
    static constexpr int kPoint = S == 7 ? 40 : 41;
    __device__ static long long of(const uint32_t (&a)[S][8], int j) {
        auto f = [&](int d) { return __uint_as_float(a[d][j]); };
        auto in = [&](int d) { return __float2int_rn(f(d)); };
        if (S == 7) {   // BETA = 8: a0 2^40 + a1 2^32 + ... + a5 + a6 2^-8
            long long I = (long long)((in(0) << 8) + in(1)) << 32;
            I += (long long)((in(2) << 8) + in(3)) * 65536;
            I += (long long)in(4) * 256;
            return I + __float2int_rn(fmaf(f(6), 0x1p-8f, f(5)));
        }
        // BETA = 7: a0 2^41 + a1 2^34 + ... + a6 2^-1 + a7 2^-8
        long long I = (long long)((in(0) << 7) + in(1)) << 34;
        I += (long long)((in(2) << 7) + in(3)) * (1 << 20);
        I += (long long)in(4) * (1 << 13);
        I += (long long)in(5) * 64;
        return I + __float2int_rn(0.5f * fmaf(f(S - 1), 0x1p-7f, f(6)));
    }
};

// Where a thread's results go: its row's offsets, the tile's column tables.
struct RowOut {
    int64_t roff, rdof;
    int comp;      // re / im row of an expanded row operand
    bool ok;
};

// Columns c and c + 1 of the row: z0, z1 into C (and D).
__device__ __forceinline__ void store_pair(const OutArgs& o, const RowOut& r, const int64_t* coff, const int64_t* cdof,
                                           int c, double z0, double z1) {
    if (!r.ok || coff[c] < 0) return;
    if (o.cexp) {   // re and im of one element
        double2* w = reinterpret_cast<double2*>(o.C + r.roff + coff[c]);
        double2 z = make_double2(z0, z1);
        if (o.beta != 0.0) {
            const double2 old = *w;
            z.x = fma(o.beta, old.x, z.x);
            z.y = fma(o.beta, old.y, z.y);
        }
        *w = z;
        if (o.D) {
            double2* u = reinterpret_cast<double2*>(o.D + r.rdof + cdof[c]);
            const double2 old = *u;
            *u = make_double2(old.x + z.x, old.y + z.y);
        }
        return;
    }
    double* C = reinterpret_cast<double*>(o.C);
    double* D = reinterpret_cast<double*>(o.D);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if (coff[c + q] < 0) return;
        const int64_t i = 2 * (r.roff + coff[c + q]) + r.comp, id = 2 * (r.rdof + cdof[c + q]) + r.comp;
        double z = q == 0 ? z0 : z1;
        if (o.beta != 0.0) z = fma(o.beta, C[i], z);
        if (o.rexp) {
            C[i] = z;
        } else {   // both operands real
            const double im = o.beta != 0.0 ? o.beta * C[i + 1] : 0.0;
            *reinterpret_cast<double2*>(C + i) = make_double2(z, im);
            if (o.D) D[id + 1] += im;
        }
        if (o.D) D[id] += z;
    }
}

// One persistent CTA per SM: warp 0 loads stages of all slices of both operands (one TMA copy
// each), warp 1 issues the S (S + 1) / 2 MMAs (N = 64) of every 16 contracted entries, the
// other sixteen warps turn the accumulators into FP64.  An N of 64 leaves the tensor core waiting
// for shared memory (47 cycles an MMA of 128 rows, 32 of them its products); a wider tile
// has no room for its accumulators.  PAIR: two CTAs take two neighbouring row tiles with one MMA of
// M = 256, each with half of the Q rows in its shared memory, which are then read and copied once
// for both, in stages that leave room for a third.  For lack of tensor memory the accumulators
// have one buffer: the epilogue first folds each output's accumulators into a 64-bit integer in
// registers, releases tensor memory, and rounds and stores while the next tile's products run.
// MULTI: the contracted index in several pieces, whose rounded results are added in registers.
// Measured (T_n = Ltilde_n Theta of M = 128, N = 32, 64 vectors x 512 walkers): 14.3 ms by
// the multiply-add tiles, 0.54 ms here without pairs (80 cycles an MMA before A stayed in the
// collector and one elected lane issued from uniform registers), 0.48 ms with them; of a tile's
// 17600 cycles without pairs 10500 issued MMAs, 2750 waited for copies and 3200 for the
// accumulators to be read.  Copies of 128-byte rows (two slices side by side) and more, shorter stages
// gained nothing (0.55, 0.68 ms).
template <int S, bool MULTI, bool PAIR>
__global__ void __launch_bounds__(kThreadsG, 1)
    slice_gemm_kernel(const __grid_constant__ CUtensorMap tR, const __grid_constant__ CUtensorMap tQ, OutArgs o,
                      unsigned* flags) {
    using P = Digits<S>;
    using St = Stage<S, PAIR>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sbase = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Ctl* ctl = reinterpret_cast<Ctl*>(sbase + St::kCount * St::kBytes);
    // output offsets (C, D) and exponents of the tile's columns, for two pieces in turn
    int64_t* coff2 = reinterpret_cast<int64_t*>(ctl + 1);
    int64_t* cdof2 = coff2 + 2 * kCols;
    int* cexp2 = reinterpret_cast<int*>(cdof2 + 2 * kCols);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = PAIR ? cluster_ctarank() : 0;
    const uint32_t first = PAIR ? cluster_id_x() : blockIdx.x, stride = PAIR ? ncluster_x() : gridDim.x;
    if (warp == 0 && lane == 0) {
        tma_prefetch_desc(&tR);
        tma_prefetch_desc(&tQ);
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < St::kCount; ++i) {
            mbar_init(&ctl->full[i], 1);
            mbar_init(&ctl->empty[i], 1);
        }
        mbar_init(&ctl->tfull, 1);
        mbar_init(&ctl->tempty, (PAIR ? 2 : 1) * kEpiWarps);
        mbar_init(&ctl->done, 1);
        ctl->abort = 0;
        fence_mbar_init();
    }
    if (PAIR) {
        __syncthreads();
        cluster_sync();   // both CTAs' barriers exist before any copy or arrival reaches them
    }
    if (warp == 1) {
        if (PAIR) {
            tmem_alloc_pair(&ctl->tmem_base, 512);
            tmem_relinquish_pair();
        } else {
            tmem_alloc(&ctl->tmem_base, 512);
            tmem_relinquish();
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (PAIR) cluster_sync();   // tensor memory allocated in both CTAs before the first MMA
    const uint32_t work = (uint32_t)(MULTI ? o.tiles * o.groups : o.tiles);
    if (warp == 0) {
        if (lane == 0) {
            int64_t g = 0;
            Ring<St::kCount> ring;
            bool ok = true;
            for (uint32_t w = first; w < work && ok; w += stride) {
                uint32_t grp, t, b, ct, rt;
                o.dtiles.divmod(w, grp, t);
                o.tile(t, b, ct, rt);
                const int p0 = MULTI ? (int)grp * o.pg : 0, p1 = MULTI ? min(o.pieces, p0 + o.pg) : 1;
                for (int pc = p0; pc < p1 && ok; ++pc)
                    for (int kb = 0; kb < o.nk; ++kb, ++g, ring.next()) {
                        const int st = ring.st;
                        if (!mbar_wait(&ctl->empty[st], ring.phase ^ 1u, &ctl->abort)) { ok = false; break; }
                        uint8_t *s = sbase + (size_t)st * St::kBytes, *sq = s + S * kRows * kChunk * 2;
                        const int z = (int)(pc * o.nbatch + b), x = kb * kChunk;
                        if (PAIR) {   // rank 0's barrier counts both CTAs' bytes
                            if (rank == 0) mbar_arrive_expect_tx(&ctl->full[st], 2 * St::kBytes);
                            const uint32_t fb = mapa_shared(&ctl->full[st], 0);
                            tma_load_4d_pair(s, &tR, fb, x, (int)(2 * rt + rank) * kRows, z, 0);
                            tma_load_4d_pair(sq, &tQ, fb, x, (int)ct * kCols + (int)rank * St::kQRows, z, 0);
                        } else {
                            mbar_arrive_expect_tx(&ctl->full[st], St::kBytes);
                            tma_load_4d(s, &tR, &ctl->full[st], x, (int)rt * kRows, z, 0);
                            tma_load_4d(sq, &tQ, &ctl->full[st], x, (int)ct * kCols, z, 0);
                        }
                    }
            }
            if (!ok && rank == 0)
                for (int64_t j = g > St::kCount ? g - St::kCount : 0; j < g; ++j)
                    wait_drain(&ctl->full[j % St::kCount], (uint32_t)((j / St::kCount) & 1));
            if (!ok && rank != 0) {   // the peer cannot wait on rank 0's barriers: its copies get time to land
                const long long t0 = clock64();
                while (clock64() - t0 < (1LL << 22)) {
                }
            }
        }
    } else if (warp == 1) {
      if (rank == 0) {
        // the whole warp runs the loop, one elected lane issues: the MMAs follow each other as fast as
        // the tensor core takes them only while their descriptors stay in uniform registers
        constexpr uint32_t idesc = idesc_bf16(PAIR ? 2 * kRows : kRows, kCols, true);
        const uint32_t tmem = ctl->tmem_base;
        const uint64_t d0 = desc_sw64(smem_u32(sbase));
        const uint32_t lo0 = (uint32_t)d0, hi0 = (uint32_t)(d0 >> 32);
        Ring<St::kCount> ring;
        int it = 0;
        bool ok = true;
        for (uint32_t w = first; w < work && ok; w += stride) {
            const int p0 = MULTI ? (int)o.dtiles.div(w) * o.pg : 0, p1 = MULTI ? min(o.pieces, p0 + o.pg) : 1;
            for (int pc = p0; pc < p1 && ok; ++pc, ++it) {
                if (!warp_wait(&ctl->tempty, ((uint32_t)it & 1u) ^ 1u, &ctl->abort)) { ok = false; break; }
                tc_fence_after();
                for (int kb = 0; kb < o.nk; ++kb, ring.next()) {
                    const int st = ring.st;
                    if (!warp_wait(&ctl->full[st], ring.phase, &ctl->abort)) { ok = false; break; }
                    tc_fence_after();
                    if (elect_one()) {
                        const uint32_t sr = lo0 + st * (St::kBytes >> 4);
                        const uint32_t sq = sr + (S * kRows * kChunk * 2 >> 4);
#pragma unroll
                        for (int kk = 0; kk < kChunk / 16; ++kk)
#pragma unroll
                            for (int p = 0; p < S; ++p)   // slice p of R stays in the collector
#pragma unroll
                                for (int d = p; d < P::D; ++d) {
                                    const uint32_t D = tmem + d * kCols, a = sr + ((p * kRows * kChunk * 2 + kk * 32) >> 4),
                                                   b = sq + (((d - p) * St::kQRows * kChunk * 2 + kk * 32) >> 4),
                                                   acc = (kk | p) != 0 ? 1u : (kb != 0 ? 1u : 0u);
                                    if (p == S - 1) mma_f16_lo<kKeepNone, PAIR>(D, a, b, hi0, idesc, acc);
                                    else if (d == p) mma_f16_lo<kKeepFirst, PAIR>(D, a, b, hi0, idesc, acc);
                                    else if (d < P::D - 1) mma_f16_lo<kKeepMore, PAIR>(D, a, b, hi0, idesc, acc);
                                    else mma_f16_lo<kKeepLast, PAIR>(D, a, b, hi0, idesc, acc);
                                }
                        if (PAIR) mma_commit_pair(&ctl->empty[st], 3);   // free in both CTAs
                        else mma_commit(&ctl->empty[st]);
                    }
                    __syncwarp();
                }
                if (!ok) break;
                if (elect_one()) {
                    if (PAIR) mma_commit_pair(&ctl->tfull, 3);
                    else mma_commit(&ctl->tfull);
                }
                __syncwarp();
            }
        }
        if (elect_one()) {
            if (PAIR) mma_commit_pair(&ctl->done, 1);
            else mma_commit(&ctl->done);
            wait_drain(&ctl->done, 0);
        }
        __syncwarp();
      }
    } else {
        const int q = warp & 3, h = (warp - 2) >> 2;   // lane quadrant, columns [16 h, 16 h + 16)
        const int et = threadIdx.x - 64;
        const uint32_t tq = ctl->tmem_base + ((uint32_t)(q * 32) << 16) + 16 * h;
        const int rx = o.rexp ? 1 : 0, cx = o.cexp ? 1 : 0;
        constexpr int kShift = -2 * (P::BETA - 1) - Gather<S>::kPoint;
        int it = 0;
        bool ok = true;
        for (uint32_t w = first; w < work && ok; w += stride) {
            uint32_t grp, t, b, ct, rt, ob, i;
            o.dtiles.divmod(w, grp, t);
            o.tile(t, b, ct, rt);
            const int p0 = MULTI ? (int)grp * o.pg : 0, p1 = MULTI ? min(o.pieces, p0 + o.pg) : 1;
            const int64_t r = (int64_t)(PAIR ? 2 * rt + rank : rt) * kRows + q * 32 + lane;
            const uint32_t ri = (uint32_t)r >> rx;
            RowOut ro;
            ro.ok = r < o.rows;
            o.rn.divmod(ri, ob, i);
            ro.roff = ro.ok ? o.shared.at(b) + o.rown.at(ob) + i * o.rs : 0;
            ro.rdof = ro.ok && o.D ? o.dshared.at(b) + o.drown.at(ob) + i * o.drs : 0;
            if (MULTI && ro.ok) ro.roff += grp * o.gstride;
            ro.comp = o.rexp ? (int)(r & 1) : 0;
            double acc[MULTI ? 16 : 1];
            if (MULTI) {
#pragma unroll
                for (int j = 0; j < 16; ++j) acc[MULTI ? j : 0] = 0.0;
            }
#pragma unroll 1
            for (int pc = p0; pc < p1; ++pc, ++it) {
                int64_t* coff = coff2 + (it & 1) * kCols;
                int64_t* cdof = cdof2 + (it & 1) * kCols;
                int* cexp = cexp2 + (it & 1) * kCols;
                const int64_t z = pc * o.nbatch + b;
                if (et < kCols) {
                    const int64_t c = (int64_t)ct * kCols + et;
                    const uint32_t ci = (uint32_t)c >> cx;
                    const bool in = c < o.cols;
                    uint32_t cob, cj;
                    o.cn.divmod(ci, cob, cj);
                    coff[et] = in ? o.cown.at(cob) + cj * o.cs : -1;
                    cdof[et] = in && o.D ? o.dcown.at(cob) + cj * o.dcs : 0;
                    cexp[et] = in ? o.ec[z * (o.cols >> cx) + ci] : 0;
                }
                const int er = ro.ok ? o.er[z * (o.rows >> rx) + ri] : 0;
                int got = 1;
                if (lane == 0) got = mbar_wait(&ctl->tfull, (uint32_t)it & 1u, &ctl->abort) ? 1 : 0;
                got = __shfl_sync(0xffffffffu, got, 0);
                // the tables are written; if any warp's wait gave up, all sixteen leave together.  (A
                // warp reaches this barrier of the next piece only after reading this one's tables,
                // so two sets suffice.)
                if (!epi_and(got)) { ok = false; break; }
                tc_fence_after();
                auto value = [&](int j, long long I) { return round64(I, er + cexp[16 * h + j] + kShift); };
                auto release = [&]() {   // every accumulator of this warp is in registers
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        if (PAIR) mbar_arrive_cluster_relaxed(mapa_shared(&ctl->tempty, 0));
                        else mbar_arrive(&ctl->tempty);
                    }
                };
                if (MULTI) {
#pragma unroll
                    for (int c8 = 0; c8 < 2; ++c8) {
                        uint32_t a[S][8];
#pragma unroll
                        for (int d = 0; d < S; ++d) tmem_ld8_nw(tq + d * kCols + 8 * c8, a[d]);
                        tmem_ld_wait();
                        if (c8 == 1) release();
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            acc[MULTI ? 8 * c8 + j : 0] += value(8 * c8 + j, Gather<S>::of(a, j));
                        }
                    }
                    if (pc + 1 < p1) continue;
#pragma unroll
                    for (int j = 0; j < 16; j += 2)
                        store_pair(o, ro, coff, cdof, 16 * h + j, acc[MULTI ? j : 0], acc[MULTI ? j + 1 : 0]);
                } else {
                    long long I[16];
#pragma unroll
                    for (int c8 = 0; c8 < 2; ++c8) {
                        uint32_t a[S][8];
#pragma unroll
                        for (int d = 0; d < S; ++d) tmem_ld8_nw(tq + d * kCols + 8 * c8, a[d]);
                        tmem_ld_wait();
                        if (c8 == 1) release();
#pragma unroll
                        for (int j = 0; j < 8; ++j) I[8 * c8 + j] = Gather<S>::of(a, j);
                    }
#pragma unroll
                    for (int j = 0; j < 16; j += 2)
                        store_pair(o, ro, coff, cdof, 16 * h + j, value(j, I[j]), value(j + 1, I[j + 1]));
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync();   // both CTAs are done with tensor memory and each other's shared memory
    if (warp == 1) {
        tc_fence_after();
        if (PAIR) tmem_dealloc_pair(ctl->tmem_base, 512);
        else tmem_dealloc(ctl->tmem_base, 512);
    }
    if (threadIdx.x == 0 && ctl->abort) atomicOr(flags, FLAG_TIMEOUT);
}

// ------------------------------------------------------------------------------------ host side
int64_t up(int64_t n, int64_t m) { return (n + m - 1) / m * m; }

// How one product runs: which batch dimensions fold into which operand's rows, which operand is
// expanded and which one supplies the tile rows.
struct Plan {
    Dims aown{{1, 1, 1}, {0, 0, 0}}, bown = aown, shared_a = aown, shared_b = aown, shared_c = aown, shared_d = aown,
        aown_c = aown, bown_c = aown, aown_d = aown, bown_d = aown;
    int64_t na = 1, nb = 1, ns = 1;       // own batches of A and B, shared batches
    int parts = 1, koff = 0, klen = 0, pieces = 1, S = 7;
    bool exp_a = false, exp_b = false, swap = false;   // swap: A supplies the tile rows
    int64_t rows_a = 0, rows_b = 0;       // after expansion
    int64_t tiles = 0;                    // pairs of row tiles with `pair`
    bool pair = false;                    // a CTA pair to two neighbouring row tiles
    int groups = 1, pg = 1;               // CTAs that share a tile's pieces, pieces of each
    size_t bytes_p = 0;                   // their partial outputs
    size_t bytes_a = 0, bytes_b = 0, bytes = 0;
};

constexpr int kMaxK = 512;

int64_t tile_count(int64_t r, int64_t c) { return (up(r, kRows) / kRows) * (up(c, kCols) / kCols); }

Plan make_plan(const GemmArgs& g) {
    Plan p;
    const int64_t cnt[3] = {g.nb0, g.nb1, g.nb2}, sa[3] = {g.A.s0, g.A.s1, g.A.s2}, sb[3] = {g.B.s0, g.B.s1, g.B.s2},
                  sc[3] = {g.sc0, g.sc1, g.sc2}, sd[3] = {g.sd0, g.sd1, g.sd2};
    for (int i = 0; i < 3; ++i) {
        if (cnt[i] == 1) continue;
        if (sa[i] != 0 && sb[i] == 0) {
            p.aown.cnt[i] = p.aown_c.cnt[i] = p.aown_d.cnt[i] = cnt[i];
            p.aown.str[i] = sa[i]; p.aown_c.str[i] = sc[i]; p.aown_d.str[i] = sd[i];
            p.na *= cnt[i];
        } else if (sb[i] != 0 && sa[i] == 0) {
            p.bown.cnt[i] = p.bown_c.cnt[i] = p.bown_d.cnt[i] = cnt[i];
            p.bown.str[i] = sb[i]; p.bown_c.str[i] = sc[i]; p.bown_d.str[i] = sd[i];
            p.nb *= cnt[i];
        } else {
            p.shared_a.cnt[i] = p.shared_b.cnt[i] = p.shared_c.cnt[i] = p.shared_d.cnt[i] = cnt[i];
            p.shared_a.str[i] = sa[i]; p.shared_b.str[i] = sb[i]; p.shared_c.str[i] = sc[i]; p.shared_d.str[i] = sd[i];
            p.ns *= cnt[i];
        }
    }
    p.parts = !g.A.real && !g.B.real ? 2 : 1;
    const int most = kMaxK / p.parts;
    p.pieces = std::max(1, (g.k + most - 1) / most);   // of equal length, at most kMaxK with both parts
    p.klen = (g.k + p.pieces - 1) / p.pieces;
    p.koff = (int)up(p.klen, 8);
    p.S = p.parts * p.koff <= 128 ? 7 : 8;
    // orientation and expansion with the fewest tiles; ties keep B's rows on the tile rows (the
    // output's contiguous index across lanes)
    int64_t best = -1;
    for (int sw = 0; sw < 2; ++sw)
        for (int ea = 0; ea < 2; ++ea) {
            const bool xa = p.parts == 2 ? ea == 1 : !g.A.real;
            const bool xb = p.parts == 2 ? ea == 0 : !g.B.real;
            if (p.parts == 1 && ea) continue;
            const int64_t ra = p.na * g.m * (xa ? 2 : 1), rb = p.nb * g.n * (xb ? 2 : 1);
            const int64_t t = p.ns * (sw ? tile_count(ra, rb) : tile_count(rb, ra));
            if (best < 0 || t < best) {
                best = t;
                p.swap = sw == 1;
                p.exp_a = xa; p.exp_b = xb;
                p.rows_a = ra; p.rows_b = rb;
            }
        }
    p.tiles = best;
    {   // pairs where they leave at most one row tile in ten empty
        const int64_t rt = up(p.swap ? p.rows_a : p.rows_b, kRows) / kRows, pt = (rt + 1) / 2;
        p.pair = rt >= 2 && (rt % 2 == 0 || rt >= 9);
        if (p.pair) p.tiles = p.tiles / rt * pt;
    }
    const int64_t Kp = (int64_t)p.parts * p.koff;
    const int64_t nz = p.ns * p.pieces;
    p.bytes_a = up((int64_t)p.S * nz * p.rows_a * Kp * 2, 1024) + up(4 * nz * p.na * g.m, 1024);
    p.bytes_b = up((int64_t)p.S * nz * p.rows_b * Kp * 2, 1024) + up(4 * nz * p.nb * g.n, 1024);
    p.groups = (int)std::max<int64_t>(1, std::min<int64_t>(p.pieces, tc_num_sms() / (p.pair ? 2 : 1) / std::max<int64_t>(p.tiles, 1)));
    p.pg = (p.pieces + p.groups - 1) / p.groups;
    p.groups = (p.pieces + p.pg - 1) / p.pg;
    if (p.groups > 1) p.bytes_p = up((int64_t)p.groups * p.na * p.nb * p.ns * g.m * g.n * 16, 1024);
    p.bytes = p.bytes_a + p.bytes_b + p.bytes_p;
    return p;
}

template <int S>
void launch_pack(const PackArgs& a, cudaStream_t st) {
    count_launch();
    const int rb = a.koff <= 64 ? 32 : 8;
    const dim3 grid((unsigned)((a.own_rows + rb - 1) / rb), (unsigned)(a.nbatch * a.pieces));
    if (rb == 32) pack_slices_kernel<S, 32><<<grid, kPackT, 0, st>>>(a);
    else pack_slices_kernel<S, 8><<<grid, kPackT, 0, st>>>(a);
}

PackArgs pack_args(const GemmOperand& X, bool is_a, int n, int k, const Plan& p, void* buf, cplx alpha) {
    PackArgs a{};
    a.ptr = X.ptr;
    a.real = X.real;
    a.conj = X.op == OP_C;
    a.expand = is_a ? p.exp_a : p.exp_b;
    a.parts = p.parts;
    // A: row index i at i ld (N) or i (T, C); B: row index j at j (N) or j ld (T, C)
    const bool idx_fast = (X.op == OP_N) != is_a;
    a.idx_contig = idx_fast;
    a.si = idx_fast ? 1 : X.ld;
    a.sk = idx_fast ? X.ld : 1;
    a.n = n;
    a.k = k;
    a.koff = p.koff;
    a.klen = p.klen;
    a.pieces = p.pieces;
    a.Kp = (int64_t)p.parts * p.koff;
    a.own = Strides(is_a ? p.aown : p.bown);
    a.shared = Strides(is_a ? p.shared_a : p.shared_b);
    a.dn = Div(n);
    a.dbatch = Div(p.ns);
    a.own_rows = (is_a ? p.na : p.nb) * n;
    a.nbatch = p.ns;
    const int64_t rows = is_a ? p.rows_a : p.rows_b;
    a.plane = p.ns * p.pieces * rows * a.Kp;
    a.out = static_cast<__half*>(buf);
    a.exps = reinterpret_cast<int*>(static_cast<uint8_t*>(buf) + up((int64_t)p.S * a.plane * 2, 1024));
    a.alpha = alpha;
    a.scale = alpha.re != 1.0 || alpha.im != 0.0;
    return a;
}

// C = beta C + the groups' sums in order (and D += C)
__global__ void __launch_bounds__(256) sum_groups_kernel(const cplx* part, int groups, int64_t total, GemmArgs g) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= total) return;
    cplx v = part[i];
    for (int q = 1; q < groups; ++q) v = v + part[q * total + i];
    const int64_t c = i % g.n, r = i / g.n % g.m, b = i / ((int64_t)g.m * g.n);
    const int64_t b2 = b % g.nb2, b1 = b / g.nb2 % g.nb1, b0 = b / g.nb2 / g.nb1;
    cplx* C = g.C + b0 * g.sc0 + b1 * g.sc1 + b2 * g.sc2 + r * g.ldc + c;
    if (g.beta.re != 0.0) v = cplx{fma(g.beta.re, C->re, v.re), fma(g.beta.re, C->im, v.im)};
    *C = v;
    if (g.D) {
        cplx* D = g.D + b0 * g.sd0 + b1 * g.sd1 + b2 * g.sd2 + r * g.ldd + c;
        *D = *D + v;
    }
}

template <int S, bool PAIR>
int launch_gemm(const CUtensorMap& r, const CUtensorMap& q, const OutArgs& o, unsigned* flags, cudaStream_t st) {
    using St = Stage<S, PAIR>;
    auto kern = o.pieces > 1 ? slice_gemm_kernel<S, true, PAIR> : slice_gemm_kernel<S, false, PAIR>;
    const size_t sm = 1024 + (size_t)St::kCount * St::kBytes + sizeof(Ctl) + 2 * kCols * (2 * sizeof(int64_t) + sizeof(int));
    raise_dyn_smem(kern, sm);
    constexpr int C = PAIR ? 2 : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(C * std::min<int64_t>(o.tiles * o.groups, tc_num_sms() / C)));
    cfg.blockDim = dim3(kThreadsG);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    count_launch();
    cudaLaunchKernelEx(&cfg, kern, r, q, o, flags);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(AFQMC_ERR_CUDA, std::string("slice_gemm launch: ") + cudaGetErrorString(e));
    return AFQMC_OK;
}
int launch_gemm(const Plan& p, const CUtensorMap& r, const CUtensorMap& q, const OutArgs& o, unsigned* flags, cudaStream_t st) {
    if (p.pair) return p.S == 7 ? launch_gemm<7, true>(r, q, o, flags, st) : launch_gemm<8, true>(r, q, o, flags, st);
    return p.S == 7 ? launch_gemm<7, false>(r, q, o, flags, st) : launch_gemm<8, false>(r, q, o, flags, st);
}

// One product that fits the workspace: B's slices at its start, A's at its end,
// partial outputs between them.
int run_plan(const GemmArgs& g, const Plan& p, SliceScratch* ws, cudaStream_t st) {
    uint8_t* buf = static_cast<uint8_t*>(ws->buf);
    // alpha multiplies B, or A where alpha is complex and B real
    const bool on_a = g.B.real && g.alpha.im != 0.0;
    const cplx one{1.0, 0.0};
    const PackArgs pb = pack_args(g.B, false, g.n, g.k, p, buf, on_a ? one : g.alpha);
    const PackArgs pa = pack_args(g.A, true, g.m, g.k, p, buf + (ws->bytes - p.bytes_a) / 1024 * 1024, on_a ? g.alpha : one);
    const int64_t nz = p.ns * p.pieces;
    auto kept = [&](bool keep, SliceScratch::Packed& have, const PackArgs& x, int64_t rows) {
        const bool same = keep && have.rows == rows && have.pitch == x.Kp && have.batches == nz;
        have = SliceScratch::Packed{rows, x.Kp, nz};
        if (same) return;
        if (p.S == 7) launch_pack<7>(x, st);
        else launch_pack<8>(x, st);
    };
    kept(g.keep_b, ws->b, pb, p.rows_b);
    kept(g.keep_a, ws->a, pa, p.rows_a);
    const PackArgs &R = p.swap ? pa : pb, &Q = p.swap ? pb : pa;
    const int64_t rr = p.swap ? p.rows_a : p.rows_b, rc = p.swap ? p.rows_b : p.rows_a;
    CUtensorMap mr, mq;
    auto encode = [&](CUtensorMap* m, const PackArgs& x, int64_t rows, int box_rows) {
        const uint64_t dims[4] = {(uint64_t)x.Kp, (uint64_t)rows, (uint64_t)nz, (uint64_t)p.S};
        const uint64_t str[3] = {(uint64_t)x.Kp * 2, (uint64_t)rows * x.Kp * 2, (uint64_t)x.plane * 2};
        const uint32_t box[4] = {kChunk, (uint32_t)box_rows, 1, (uint32_t)p.S};
        return make_map4(m, x.out, dims, str, box, 64);
    };
    AFQMC_TRY(encode(&mr, R, rr, kRows));
    AFQMC_TRY(encode(&mq, Q, rc, p.pair ? kCols / 2 : kCols));
    OutArgs o{};
    o.rows = rr;
    o.cols = rc;
    o.rexp = p.swap ? p.exp_a : p.exp_b;
    o.cexp = p.swap ? p.exp_b : p.exp_a;
    o.rn = Div(p.swap ? g.m : g.n);
    o.cn = Div(p.swap ? g.n : g.m);
    o.rs = p.swap ? g.ldc : 1;
    o.cs = p.swap ? 1 : g.ldc;
    o.drs = p.swap ? g.ldd : 1;
    o.dcs = p.swap ? 1 : g.ldd;
    Dims rown = p.swap ? p.aown_c : p.bown_c, cown = p.swap ? p.bown_c : p.aown_c, shared = p.shared_c;
    o.drown = Strides(p.swap ? p.aown_d : p.bown_d);
    o.dcown = Strides(p.swap ? p.bown_d : p.aown_d);
    o.dshared = Strides(p.shared_d);
    o.er = R.exps;
    o.ec = Q.exps;
    o.C = g.C;
    o.D = g.D;
    o.beta = g.beta.re;
    o.tiles = p.tiles;
    o.drt = Div(up(rr, p.pair ? 2 * kRows : kRows) / (p.pair ? 2 * kRows : kRows));
    o.dper = Div(p.tiles / p.ns);
    o.dtiles = Div(p.tiles);
    o.nk = (int)(up((int64_t)p.parts * p.koff, kChunk) / kChunk);
    o.pieces = p.pieces;
    o.nbatch = p.ns;
    o.groups = p.groups;
    o.pg = p.pg;
    auto place = [&] {
        o.rown = Strides(rown);
        o.cown = Strides(cown);
        o.shared = Strides(shared);
    };
    place();
    const int64_t mn = (int64_t)g.m * g.n, total = (int64_t)g.nb0 * g.nb1 * g.nb2 * mn;
    if (p.groups > 1) {   // the groups' sums side by side, dense, then added in order
        o.C = reinterpret_cast<cplx*>(buf + p.bytes_b);
        o.D = nullptr;
        o.beta = 0.0;
        o.gstride = total;
        const int64_t dense[3] = {(int64_t)g.nb1 * g.nb2 * mn, (int64_t)g.nb2 * mn, mn};
        (p.swap ? o.rs : o.cs) = g.n;
        for (int i = 0; i < 3; ++i)
            for (Dims* d : {&rown, &cown, &shared})
                if (d->cnt[i] > 1) d->str[i] = dense[i];
        place();
        AFQMC_TRY(launch_gemm(p, mr, mq, o, ws->flags, st));
        count_launch();
        sum_groups_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(o.C, p.groups, total, g);
        return AFQMC_OK;
    }
    return launch_gemm(p, mr, mq, o, ws->flags, st);
}

}  // namespace

size_t slice_gemm_bytes(const GemmArgs& g) { return make_plan(g).bytes + 1024; }

// Expected time in microseconds: three launches with little in each, the persistent tiles at 65 (pairs: 56) cycles an MMA and 6000
// for the epilogue, and the operands' packing.
double slice_gemm_us(const GemmArgs& g) {
    if (g.beta.im != 0.0 || (g.A.real && g.B.real && g.alpha.im != 0.0)) return 1e30;
    const Plan p = make_plan(g);
    // the pack kernel's grid, 31-bit indices
    if (p.ns * p.pieces > 65535 || std::max(p.rows_a, p.rows_b) >= 1ll << 31 || p.tiles * p.groups >= 1ll << 31) return 1e30;
    const double cyc = p.S * (p.S + 1) / 2 * (up((int64_t)p.parts * p.koff, 16) / 16) * (p.pair ? 56.0 : 65.0) + 6000.0;
    const int ctas = tc_num_sms() / (p.pair ? 2 : 1);
    const double waves = (double)((p.tiles * p.groups + ctas - 1) / ctas);
    return 26.0 + p.pg * waves * cyc / 1.9e3 + (double)p.bytes / 2.0e6 + (p.groups > 1 ? 4.0 : 0.0);
}

int slice_gemm(const GemmArgs& g, SliceScratch* ws, cudaStream_t st) {
    const Plan p = make_plan(g);
    if (p.bytes + 1024 <= ws->bytes) return run_plan(g, p, ws, st);
    // too large for the workspace: cut a long contraction (the output is then added up in rounds) after
    // as many pieces as fit, in equal shares for the CTAs of a tile where that is possible; else
    // halve the largest of the batch dimensions, n and m
    GemmArgs lo = g, hi = g;
    lo.keep_a = lo.keep_b = hi.keep_a = hi.keep_b = false;
    const int64_t big = std::max<int64_t>({g.nb0, g.nb1, g.nb2});
    const size_t esa = g.A.real ? sizeof(double) : sizeof(cplx), esb = g.B.real ? sizeof(double) : sizeof(cplx);
    auto shift = [&](int64_t da, int64_t db, int64_t dc, int64_t dd) {
        hi.A.ptr = static_cast<const char*>(g.A.ptr) + esa * (size_t)da;
        hi.B.ptr = static_cast<const char*>(g.B.ptr) + esb * (size_t)db;
        hi.C = g.C + dc;
        hi.D = g.D ? g.D + dd : nullptr;
    };
    if (p.pieces >= 8) {
        const int64_t fit = (int64_t)(ws->bytes / ((p.bytes + 1024) / p.pieces + 1));
        const int64_t share = std::max<int64_t>(1, tc_num_sms() / (p.pair ? 2 : 1) / std::max<int64_t>(p.tiles, 1));
        const int64_t n = fit > share ? fit / share * share : std::max<int64_t>(1, fit);
        // (at least a 64th, which may be cut again: bounds the depth of the cuts)
        lo.k = (int)std::min<int64_t>(std::max<int64_t>(n, p.pieces / 64), p.pieces - 1) * p.klen;
        hi.k = g.k - lo.k;
        shift(lo.k * (g.A.op == OP_N ? 1 : g.A.ld), lo.k * (g.B.op == OP_N ? g.B.ld : 1), 0, 0);
        lo.D = nullptr;
        hi.beta = cplx{1.0, 0.0};
    } else if (big > 1) {
        if (big == g.nb0) {
            lo.nb0 = g.nb0 / 2; hi.nb0 = g.nb0 - lo.nb0;
            shift(lo.nb0 * g.A.s0, lo.nb0 * g.B.s0, lo.nb0 * g.sc0, lo.nb0 * g.sd0);
        } else if (big == g.nb1) {
            lo.nb1 = g.nb1 / 2; hi.nb1 = g.nb1 - lo.nb1;
            shift(lo.nb1 * g.A.s1, lo.nb1 * g.B.s1, lo.nb1 * g.sc1, lo.nb1 * g.sd1);
        } else {
            lo.nb2 = g.nb2 / 2; hi.nb2 = g.nb2 - lo.nb2;
            shift(lo.nb2 * g.A.s2, lo.nb2 * g.B.s2, lo.nb2 * g.sc2, lo.nb2 * g.sd2);
        }
    } else if (g.n >= g.m && g.n > 1) {
        lo.n = g.n / 2; hi.n = g.n - lo.n;
        shift(0, lo.n * (g.B.op == OP_N ? 1 : g.B.ld), lo.n, lo.n);
    } else if (g.m > 1) {
        lo.m = g.m / 2; hi.m = g.m - lo.m;
        shift(lo.m * (g.A.op == OP_N ? g.A.ld : 1), 0, lo.m * g.ldc, lo.m * g.ldd);
    } else {
        return fail(AFQMC_ERR_OOM, "slice_gemm: workspace too small");
    }
    AFQMC_TRY(slice_gemm(lo, ws, st));
    return slice_gemm(hi, ws, st);
}

}  // namespace afqmc
