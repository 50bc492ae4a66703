// FP64 matrix products on the tensor cores.
//
// GB300's FP64 pipe does 2 multiply-adds per SM and clock, its fp16 tensor cores ~4096, so a
// product of integers small enough to be summed exactly in fp32 is worth some thirty of them for
// each FP64 one (the splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59 (2012), with
// digits sized for fp16 operands and fp32 accumulators):
//   * The contraction runs in pieces of at most 128 real products.  Every row of an operand (along
//     the contracted index) gets, in each piece, the exponent e of its largest entry (|x| < 2^e), and
//     each entry is rounded to a fixed-point number of 58 bits below 2^e, cut into 7 signed digits
//     d_p of 8 bits (|d_p| <= 2^7), the last with 11 bits (its fraction bits included): x = 2^(e - 7)
//     sum_p d_p 2^(-8 p).  Every digit is exact in fp16.
//   * The products of digits p and q of equal weight p + q = d go to one tensor-memory accumulator
//     per d < 8.  At most 8 x 2^21 bounds every partial sum, so the accumulators are exact integers
//     (the last two, which the fractional digits reach, are rounded 24 bits below their own small
//     weight).  Dropped weights d >= 8 lie 2^-64 and less below |a||b|.
//   * The epilogue adds the accumulators as one 64-bit integer and rounds it to FP64 in integer
//     instructions (a few FP64 operations per output would cost as much as the tile's MMAs).
// What that loses are the operands' roundings, 2^-59 of their rows' largest entries: next to nothing
// in a sum that contains products near 2^(ea + eb), the scale of its row and column, but everything
// in one whose large a_k meet small b_k throughout.  So each output is certified by a lower bound
// of sum_k |a_k b_k|, the product of the first digits' sizes less half a unit (by mma.sync, while
// the tensor core works on the tile's digits): where that is at least 2^-4 of 2^(ea + eb), the result lies
// within (k + 1) 2^-53 sum_k |a_k b_k|, the bound of the multiply-add loop, and the errors measured are
// a third of that loop's and less.  All other outputs, and the rows and columns that digits cannot hold
// (infinities, NaN, numbers near the ends of the FP64 range), are listed and formed by the multiply-add
// loop in a second kernel, over all SMs (in the tile's epilogue they pile up on a few).
// The rms error / (2^-53 sum |a_k b_k|) of 128 products, of the loop -> of digits (in exact arithmetic;
// tests/test_gpu_graded_products.py holds the kernels to the loop's): normal entries 0.39 -> 0.05; one operand decaying as e^(-k / 20) 1.1 -> 0.13; entries
// graded oppositely over 1 to 1e2 0.47 -> 0.13, over 1 to 1e4 and more 0.5 -> 0.5 (by the loop).
//
// Complex operands become real ones: a real operand times a complex one has the complex one's re
// and im as separate rows; two complex operands are contracted over [re | im] rows of the one
// against the rows [re | -im], [im | re] of the other, the "expanded" one.
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
// A row's word: its exponent times 4 and a bit for each half of the row ([re | im], or the whole row) that
// is zero throughout.
constexpr int kLoopExp = 1 << 22;     // exponent of a row that digits cannot hold: its outputs by the loop
constexpr int kZeroRow = 3;           // word of a row of zeros
constexpr int kMaxExp = 900;          // sums of two exponents beyond this: by the loop
constexpr float kEven = 1024.0f;      // certificate: 2^-4 in units of the first digits' products, 2^-14

constexpr int S = 7;                            // digits
constexpr int BETA = 8;                         // bits of a digit
constexpr int D = 8;                            // accumulators (weights 0 .. D - 1)
constexpr int kTail = 11;                       // bits of the last digit
constexpr int kFrac = kTail - BETA;             // fraction bits of the last digit
// fixed-point value v = x 2^(kPoint - e): BETA - 1 bits above the first digit's unit
constexpr int kPoint = BETA - 1 + BETA * (S - 1) + kFrac;
constexpr int kMaxK = 128;                      // contracted real products of a piece
constexpr int kMmas = S * (S + 1) / 2 + (S - 1);   // of 16 contracted entries

// A stage of one CTA: the R rows of its tile and the Q rows, or half of them for a CTA pair.
template <bool PAIR>
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
    Div dblocks;               // by the blocks of one (piece, batch)
    __half* out;               // [S][pieces][nbatch][own_rows (x 2)][Kp]
    int64_t plane;             // elements per slice
    int* exps;                 // words of the rows [pieces][nbatch][own_rows (x 2)]
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
// The exponent field; 1, that of the smallest normal number, for subnormal ones, 0 for zero.
__device__ __forceinline__ int exp_field(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), e = (hi >> 20) & 0x7ffu;
    return e != 0u ? (int)e : (((hi << 1) | (uint32_t)__double2loint(x)) != 0u ? 1 : 0);
}
// Row exponent from the largest field m: largest entry < 2^e.
__device__ __forceinline__ int row_exp(int m) { return m == 0 ? 0 : (m < 64 || m == 0x7ff ? kLoopExp : m - 1022); }

// The S digits of x at the row exponent e as fp16 bit patterns.
__device__ __forceinline__ void digits_of(double x, int e, unsigned short (&d)[S]) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int E = (int)((b >> 52) & 0x7ffu);
    long long v = 0;
    if (E != 0 && e != kLoopExp) {   // subnormals are less than half a unit
        const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
        const int sh = E - 1075 + kPoint - e;   // x = m 2^(E - 1075); at most 5
        if (sh >= 0) v = (long long)(m << sh);
        else if (sh > -56) v = (long long)((m + (1ull << (-sh - 1))) >> -sh);
        if (b >> 63) v = -v;
    }
    {   // last digit: 11 bits, in units of 2^-kFrac
        const int t = (int)((v + 1024) & 2047) - 1024;
        v = (v - t) >> 11;
        d[S - 1] = __half_as_ushort(__float2half_rn((float)t * (1.0f / (1 << kFrac))));
    }
#pragma unroll
    for (int p = S - 2; p > 0; --p) {
        constexpr int h = 1 << (BETA - 1);
        const int t = (int)((v + h) & (2 * h - 1)) - h;
        v = (v - t) >> BETA;
        d[p] = __half_as_ushort(__float2half_rn((float)t));
    }
    d[0] = __half_as_ushort(__float2half_rn((float)(int)v));
}

// RB rows per block (8, or 32 of at most 64 entries).  The rows of one piece are read once, coalesced along
// whichever index is contiguous, into shared memory; their exponents found; and the digits
// written, two neighbours per store.  Most calls have a few hundred rows, so a block's chain of
// loads and digits is the time, not the bytes (8 in, 14 out per entry): 32 rows a block of any length
// took 83 us for 1024 complex rows of 3072 (55 with 8 rows a block), 25 for 64 x 32 rows of 128 (9), 13 for 90 real
// rows of 90 (4).
constexpr int kPackT = 256;
template <int RB>
__global__ void __launch_bounds__(kPackT) pack_slices_kernel(PackArgs a) {
    constexpr int KB = RB == 32 ? 64 : kMaxK, KS = kPackT / RB;
    __shared__ cplx tile[RB][KB + 1];
    __shared__ int64_t off[RB];
    __shared__ int rowexp[2][RB];   // of re and im (of both where they share a row)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t btu, blk, piece, sb;
    a.dblocks.divmod(blockIdx.x, btu, blk);
    a.dbatch.divmod(btu, piece, sb);
    const int64_t r0 = (int64_t)blk * RB, bt = btu;   // bt = (piece, shared batch)
    const int kn = min(a.klen, a.k - (int)piece * a.klen);
    if (tid < RB) {
        const int64_t r = r0 + tid;
        uint32_t ob, i;
        a.dn.divmod((uint32_t)r, ob, i);
        off[tid] = r < a.own_rows ? a.shared.at(sb) + a.own.at(ob) + i * a.si + (int64_t)piece * a.klen * a.sk : -1;
        rowexp[0][tid] = rowexp[1][tid] = 0;
    }
    __syncthreads();
    if (a.idx_contig) {
        const int i = tid % RB;
        int mr = 0, mi = 0;
        if (off[i] >= 0) {
#pragma unroll 4
            for (int kk = tid / RB; kk < kn; kk += KS) {
                const cplx v = pack_load(a, off[i] + kk * a.sk);
                mr = max(mr, exp_field(v.re));
                mi = max(mi, exp_field(v.im));
                tile[i][kk] = v;
            }
            atomicMax(&rowexp[0][i], mr);
            if (!a.real) atomicMax(&rowexp[1][i], mi);
        }
    } else {
        for (int i = warp; i < RB; i += kPackT / 32) {
            int mr = 0, mi = 0;
            if (off[i] >= 0) {
#pragma unroll 4
                for (int kk = lane; kk < kn; kk += 32) {
                    const cplx v = pack_load(a, off[i] + kk * a.sk);
                    mr = max(mr, exp_field(v.re));
                    mi = max(mi, exp_field(v.im));
                    tile[i][kk] = v;
                }
            }
            mr = __reduce_max_sync(0xffffffffu, mr);
            mi = __reduce_max_sync(0xffffffffu, mi);
            if (lane == 0) {
                rowexp[0][i] = mr;
                rowexp[1][i] = mi;
            }
        }
    }
    {
        const int pad = a.koff - kn;   // a few entries
        for (int q = tid; q < RB * pad; q += kPackT) tile[q % RB][kn + q / RB] = cplx{0.0, 0.0};
    }
    __syncthreads();
    const int ex = a.expand ? 2 : 1;
    const int64_t rows = a.own_rows * ex;
    if (tid < RB) {
        int mr = rowexp[0][tid], mi = rowexp[1][tid];
        int zr = mr == 0 ? 3 : 0, zi = mi == 0 ? 3 : 0;   // the zero halves of the rows of re and of im
        if (a.parts == 2) {
            const int re = mr == 0, im = mi == 0;
            zr = re | im << 1;
            zi = im | re << 1;
            mr = mi = max(mr, mi);
        }
        const int er = row_exp(mr), ei = row_exp(mi);
        rowexp[0][tid] = er;
        rowexp[1][tid] = ei;
        if (off[tid] >= 0) {
            int* e = a.exps + bt * rows + ex * (r0 + tid);
            e[0] = 4 * er + zr;
            if (a.expand) e[1] = 4 * ei + zi;
        }
    }
    __syncthreads();
    const int half = a.koff / 2;   // koff is even
#pragma unroll 1
    for (int q = tid; q < RB * half; q += kPackT) {
        const int i = q / half, kk = 2 * (q - i * half);
        if (off[i] < 0) break;
        const cplx v0 = tile[i][kk], v1 = tile[i][kk + 1];
        unsigned short x[S], y[S];
        unsigned re[S], im[S];
        digits_of(v0.re, rowexp[0][i], x);
        digits_of(v1.re, rowexp[0][i], y);
#pragma unroll
        for (int p = 0; p < S; ++p) re[p] = (unsigned)x[p] | ((unsigned)y[p] << 16);
        if (!a.real) {
            digits_of(v0.im, rowexp[1][i], x);
            digits_of(v1.im, rowexp[1][i], y);
#pragma unroll
            for (int p = 0; p < S; ++p) im[p] = (unsigned)x[p] | ((unsigned)y[p] << 16);
        }
        const int64_t row = (bt * rows + ex * (r0 + i)) * a.Kp + kk;
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

// An operand as the multiply-add loop reads it.
struct Source {
    const void* ptr;
    int real, conj;
    int64_t si, sk;
    Strides own, shared;
};
struct OutArgs {
    int64_t rows, cols;        // per batch, after expansion
    int rexp, cexp;            // which side is expanded (at most one)
    Div rn, cn;                // row / column index counts within one own batch
    int64_t rs, cs;            // output strides of the row / column index (complex elements)
    Strides rown, cown, shared;    // output strides of the batch dimensions
    Strides drown, dcown, dshared;
    int64_t drs, dcs;
    const int *er, *ec;        // words of the rows and columns [pieces][nbatch][rows]
    const __half *dr, *dc;     // their first digits [pieces][nbatch][rows][Kp]
    int Kp;
    // for the outputs by the multiply-add loop: the operands of the rows and of the columns
    Source srow, scol;
    int k, klen;
    cplx alpha;
    uint32_t *list, *head;     // pairs of outputs for the loop (see slice_gemm_kernel), [entries listed, CTAs done]
    uint32_t room;
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

// FP64 value of I 2^x, rounded to nearest; x is such that the result is zero or well inside the exponent
// range.
__device__ __forceinline__ double round64(long long I, int x) {
    const int s = (int)(I >> 63);
    const unsigned long long X = (unsigned long long)((I ^ s) - s);
    const unsigned sign = (unsigned)s & 0x80000000u;
    const bool big = (X >> 32) != 0ull;
    const unsigned h = big ? (unsigned)(X >> 32) : (unsigned)X, l = big ? (unsigned)X : 0u;
    const int lz = __clz((int)h);
    const int eb1 = (big ? 1023 + 63 - 1 : 1023 + 31 - 1) + x - lz;   // biased exponent - 1
    const unsigned hi = __funnelshift_l(l, h, lz), lo = l << lz;
    // bits 63 .. 11 plus the rounding bit; the leading one carries into the exponent field
    const unsigned long long m = (((unsigned long long)(hi >> 11) << 32) | __funnelshift_r(lo, hi, 11)) + ((lo >> 10) & 1u);
    const unsigned top = ((unsigned)(m >> 32) + ((unsigned)eb1 << 20)) | sign;
    return __hiloint2double(h != 0u ? (int)top : 0, (int)(unsigned)m);
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

// Eight outputs' accumulators a_d 2^(-8 d) as integers in units of 2^-kGather of accumulator 0's, 2^-55 of
// the scale 2^(ea + eb); below 2^53 of them (a quarter of the scale) in units 2^-8 of that, whose bit in
// `fine` is set.  Every sum is exact but that of the two smallest accumulators.  Two accumulators at a
// time, to hold few of them in registers.  Conversion to integers by adding 1.5 2^23, which leaves the
// integer in the low bits (the conversion instruction has an eighth of the rate); beyond 2^22, which only
// accumulators 2 to 5 of all but equal entries reach, by the instruction.  Bound by the reads of tensor memory:
// 4300 cycles for its 256 KB; half of the instructions here gained nothing.
constexpr int kGather = 41;
constexpr float kMagic = 12582912.0f;
constexpr int kMagicBits = 0x4b400000;
template <int STEP>
__device__ __forceinline__ void gather(long long (&I)[16], int c0, const uint32_t (&a)[2][8], unsigned& fine) {
    auto f = [&](int d, int j) { return __uint_as_float(a[d][j]); };
    if (STEP < 3) {   // a0 2^41 + a1 2^33, a2 2^25 + a3 2^17, a4 2^9 + a5 2
        int top[8];
        unsigned over = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int r0 = __float_as_int(f(0, j) + kMagic), r1 = __float_as_int(f(1, j) + kMagic);
            over |= (unsigned)((r0 ^ kMagicBits) | (r1 ^ kMagicBits));
            top[j] = (int)(((unsigned)(r0 - kMagicBits) << 8) + (unsigned)(r1 - kMagicBits));
        }
        constexpr long long unit = STEP == 0 ? 1ll << 33 : (STEP == 1 ? 1ll << 17 : 2ll);
        if (STEP > 0 && (over >> 23) != 0u) {   // a pair may be beyond 32 bits
#pragma unroll
            for (int j = 0; j < 8; ++j) I[c0 + j] += (256ll * __float2int_rn(f(0, j)) + __float2int_rn(f(1, j))) * unit;
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) I[c0 + j] = (STEP == 0 ? 0ll : I[c0 + j]) + top[j] * unit;
        }
    } else {          // a6 2^-7 + a7 2^-15
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float s = fmaf(f(1, j), 0x1p-15f, f(0, j) * 0x1p-7f), m = s + kMagic;
            long long v = I[c0 + j] + (__float_as_int(m) - kMagicBits);
            const int hi = (int)(v >> 32);
            if ((unsigned)(hi ^ (hi >> 31)) < 1u << 21) {
                v = v * 256 + (__float_as_int(fmaf(s - (m - kMagic), 256.0f, kMagic)) - kMagicBits);
                fine |= 1u << (c0 + j);
            }
            I[c0 + j] = v;
        }
    }
}

// Bit j: the certificate of this lane's row and column 16 h + j, for the warp's 32 rows from r0 and 16 columns
// from c0 (rows and columns past the last repeat that, unused).  A lane of a quad takes eight entries of every 32
// of a row or column, the same ones of both.  The sums only grow: where entries are alike 32 of them are
// enough for all outputs, and the rest is left out (mma.sync keeps the tensor core from the tile's MMAs: all 128
// cost 20% of the kernel's time).
__device__ __forceinline__ void mma_sync(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t digit_size(uint32_t d) {   // max(|d| - 1/2, 0) of two digits
    const uint32_t a = d & 0x7fff7fffu;
    uint32_t r;
    asm("fma.rn.relu.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(0x3c003c00u), "r"(0xb800b800u));
    return r;
}
__device__ __forceinline__ unsigned certificates(const OutArgs& o, int64_t z, int64_t r0, int64_t c0) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const __half *x[4], *y[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = o.dr + (z * o.rows + min(r0 + 8 * i + g, o.rows - 1)) * o.Kp + 8 * t;
#pragma unroll
    for (int n = 0; n < 2; ++n) y[n] = o.dc + (z * o.cols + min(c0 + 8 * n + g, o.cols - 1)) * o.Kp + 8 * t;
    float d[2][2][4] = {};
    for (int k = 0; k < o.Kp; k += 32) {
        uint4 a[4], b[2];
        const bool in = k + 8 * t < o.Kp;
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = in ? __ldg(reinterpret_cast<const uint4*>(x[i] + k)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int n = 0; n < 2; ++n) b[n] = in ? __ldg(reinterpret_cast<const uint4*>(y[n] + k)) : make_uint4(0u, 0u, 0u, 0u);
        auto size = [](uint4& v) { v = make_uint4(digit_size(v.x), digit_size(v.y), digit_size(v.z), digit_size(v.w)); };
#pragma unroll
        for (int i = 0; i < 4; ++i) size(a[i]);
#pragma unroll
        for (int n = 0; n < 2; ++n) size(b[n]);
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                mma_sync(d[m][n], a[2 * m].x, a[2 * m + 1].x, a[2 * m].y, a[2 * m + 1].y, b[n].x, b[n].y);
                mma_sync(d[m][n], a[2 * m].z, a[2 * m + 1].z, a[2 * m].w, a[2 * m + 1].w, b[n].z, b[n].w);
            }
        float least = d[0][0][0];
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int c = 0; c < 4; ++c) least = fminf(least, d[m][n][c]);
        if (__all_sync(0xffffffffu, least >= kEven)) return 0xffffu;
    }
    // element c of d[m][n]: row 16 m + 8 (c / 2) + g, column 8 n + 2 t + c % 2; to row = lane
    unsigned even = 0;
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const unsigned b0 = __ballot_sync(0xffffffffu, d[0][n][c] >= kEven), b1 = __ballot_sync(0xffffffffu, d[0][n][2 + c] >= kEven);
            const unsigned b2 = __ballot_sync(0xffffffffu, d[1][n][c] >= kEven), b3 = __ballot_sync(0xffffffffu, d[1][n][2 + c] >= kEven);
            const unsigned w = lane < 16 ? (lane < 8 ? b0 : b1) : (lane < 24 ? b2 : b3);
            unsigned v = (w >> (4 * (lane & 7))) & 15u;
            v = (v | v << 2) & 0x33u;
            v = (v | v << 1) & 0x55u;
            even |= v << (8 * n + c);
        }
    return even;
}
// Whether the digits' result stands, from the words of its row and column and the certificate: a sum of zeros
// is exact, the rest needs the certificate and room around the result.
__device__ __forceinline__ bool stands(int wr, int wc, bool even) {
    const int x = (wr >> 2) + (wc >> 2);
    return abs(x) <= kMaxExp ? even || ((wr | wc) & 3) == 3 : false;
}

// The outputs of row r and columns c, c + 1 (batch b) by the multiply-add loop over contracted entries k0
// .. k1 - 1, as real sums of real products: which parts of the row's and the columns' elements meet is the
// form's; turn: times i (of the side with separate parts).  lane < 0: by one thread; else by the warp, entries lane, lane + 32, ... in each lane, and all lanes return
// the sums.
enum Form { kReal, kRowParts, kColParts, kRowComplex, kColComplex };   // the side whose re and im are separate rows
__device__ __forceinline__ double flip(double x, bool neg) {   // -x, off the FP64 pipe
    return __hiloint2double(__double2hiint(x) ^ (neg ? 0x80000000 : 0), __double2loint(x));
}
template <bool REAL>
__device__ __forceinline__ cplx source_load(const Source& s, int64_t at) {
    if (REAL) return cplx{__ldg(static_cast<const double*>(s.ptr) + at), 0.0};
    const double2 v = __ldg(static_cast<const double2*>(s.ptr) + at);
    return cplx{v.x, flip(v.y, s.conj)};
}
template <int FORM>
__device__ __forceinline__ double2 loop_form(const OutArgs& o, int64_t ix, int64_t iy, int64_t iy1, int kn, bool odd, int lane,
                                             bool turn) {
    constexpr bool ROWS = FORM == kRowParts || FORM == kRowComplex, COLS = FORM == kColParts || FORM == kColComplex;
    constexpr bool XR = FORM == kReal || FORM == kColParts, YR = FORM == kReal || FORM == kRowParts;
    const Source &X = o.srow, &Y = o.scol;
    const int first = lane < 0 ? 0 : lane, step = lane < 0 ? 1 : 32;
    const int64_t sx = step * X.sk, sy = step * Y.sk;
    ix += first * X.sk;
    iy += first * Y.sk;
    iy1 += first * Y.sk;
    auto scaled = [&](cplx v) { return turn ? cplx{flip(v.im, true), v.re} : v; };
    auto mac = [&](double2& z, cplx x, cplx y, cplx y1) {
        if (ROWS) x = scaled(x);
        if (COLS) y = scaled(y);
        double u = x.re, v = x.im;
        if (ROWS) u = odd ? x.im : x.re;
        if (FORM == kRowComplex) v = odd ? x.re : flip(x.im, true);
        z.x = fma(u, y.re, z.x);
        z.y = fma(u, COLS ? y.im : y1.re, z.y);
        if (FORM == kRowComplex) {
            z.x = fma(v, y.im, z.x);
            z.y = fma(v, y1.im, z.y);
        } else if (FORM == kColComplex) {
            z.x = fma(-v, y.im, z.x);
            z.y = fma(v, y.re, z.y);
        }
    };
    double2 s[4] = {};   // four sums: shorter chains, and fewer roundings in each
    int k = first;
    for (; k + 3 * step < kn; k += 4 * step, ix += 4 * sx, iy += 4 * sy, iy1 += 4 * sy) {
        cplx x[4], y[4], y1[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            x[u] = source_load<XR>(X, ix + u * sx);
            y[u] = source_load<YR>(Y, iy + u * sy);
            if (!COLS) y1[u] = source_load<YR>(Y, iy1 + u * sy);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) mac(s[u], x[u], y[u], COLS ? cplx{0.0, 0.0} : y1[u]);
    }
    for (; k < kn; k += step, ix += sx, iy += sy, iy1 += sy)
        mac(s[0], source_load<XR>(X, ix), source_load<YR>(Y, iy), COLS ? cplx{0.0, 0.0} : source_load<YR>(Y, iy1));
    double2 z = make_double2((s[0].x + s[1].x) + (s[2].x + s[3].x), (s[0].y + s[1].y) + (s[2].y + s[3].y));
    if (lane >= 0) {
#pragma unroll
        for (int h = 16; h > 0; h >>= 1) {
            z.x += __shfl_xor_sync(0xffffffffu, z.x, h);
            z.y += __shfl_xor_sync(0xffffffffu, z.y, h);
        }
    }
    return z;
}
__device__ __forceinline__ double2 loop_pair(const OutArgs& o, uint32_t b, int k0, int k1, uint32_t r, uint32_t c, int lane) {
    uint32_t q, i;
    o.rn.divmod(o.rexp ? r >> 1 : r, q, i);
    const int64_t ix = o.srow.shared.at(b) + o.srow.own.at(q) + i * o.srow.si + k0 * o.srow.sk;
    auto col = [&](uint32_t cc) {
        o.cn.divmod(cc, q, i);
        return o.scol.shared.at(b) + o.scol.own.at(q) + i * o.scol.si + k0 * o.scol.sk;
    };
    const int64_t iy = col(o.cexp ? c >> 1 : c), iy1 = o.cexp || c + 1 >= o.cols ? iy : col(c + 1);
    const int kn = k1 - k0;
    const bool odd = r & 1u;
    auto sums = [&](bool turn) {
        if (o.cexp)
            return o.srow.real ? loop_form<kColParts>(o, ix, iy, iy1, kn, odd, lane, turn)
                               : loop_form<kColComplex>(o, ix, iy, iy1, kn, odd, lane, turn);
        if (o.rexp)
            return o.scol.real ? loop_form<kRowParts>(o, ix, iy, iy1, kn, odd, lane, turn)
                               : loop_form<kRowComplex>(o, ix, iy, iy1, kn, odd, lane, turn);
        return loop_form<kReal>(o, ix, iy, iy1, kn, odd, lane, false);
    };
    double2 z = make_double2(0.0, 0.0);
#pragma unroll 1
    for (int part = 0; part < 2; ++part) {   // alpha = a + i b: most often one of them
        const double a = part ? o.alpha.im : o.alpha.re;
        if (a == 0.0 && !(part == 0 && o.alpha.im == 0.0)) continue;
        const double2 v = sums(part == 1);
        z = make_double2(fma(a, v.x, z.x), fma(a, v.y, z.y));
    }
    return z;
}

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

// z0, z1 added to what store_pair stored.
__device__ __forceinline__ void add_pair(const OutArgs& o, const RowOut& r, const int64_t* coff, const int64_t* cdof, int c,
                                         double z0, double z1) {
    double* C = reinterpret_cast<double*>(o.C);
    double* D = reinterpret_cast<double*>(o.D);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int e = o.cexp ? c : c + q, part = o.cexp ? q : r.comp;
        if (coff[e] < 0) return;
        const double z = q == 0 ? z0 : z1;
        C[2 * (r.roff + coff[e]) + part] += z;
        if (o.D) D[2 * (r.rdof + cdof[e]) + part] += z;
    }
}

// One persistent CTA per SM: warp 0 loads stages of all slices of both operands (one TMA copy
// each), warp 1 issues the 34 MMAs (N = 64) of every 16 contracted entries, the
// other sixteen warps turn the accumulators into FP64.  An N of 64 leaves the tensor core waiting
// for shared memory (47 cycles an MMA of 128 rows, 32 of them its products); a wider tile
// has no room for its accumulators.  PAIR: two CTAs take two neighbouring row tiles with one MMA of
// M = 256, each with half of the Q rows in its shared memory, which are then read and copied once
// for both, in stages that leave room for a third.  For lack of tensor memory the accumulators
// have one buffer: the epilogue first folds each output's accumulators into a 64-bit integer in
// registers, releases tensor memory, and rounds and stores while the next tile's products run.
// MULTI: the contracted index in several pieces, whose rounded results are added in registers.  While the
// MMAs of a tile or piece run, the epilogue warps certify its outputs (see the top of the file) and list
// those that do not stand (a pair of columns with one is left out; its other pieces are added up all the same).
// Measured (T_n = Ltilde_n Theta of M = 128, N = 32, 64 vectors x 512 walkers): 14.3 ms by the
// multiply-add tiles, 0.54 ms here (0.45 with 28 products of digits and no certificates, whose errors were
// at the loop's and, in graded sums, far above); of a tile's 17900 cycles 10700 issue MMAs, 2700 wait
// for copies and 4400 for the accumulators to be read, while the epilogue warps take 2400 for the certificates
// and 7000 for rounding.  Contractions of several pieces are bound by these epilogues (N = 32, K = 128
// complex, 682 vectors x 48 walkers: 1.18 ms, 0.93 when a piece held 512 entries).
// Copies of 128-byte rows (two slices side by side) and more, shorter stages gained nothing (0.55, 0.68 ms when
// it was 0.54 without pairs).
template <bool MULTI, bool PAIR>
__global__ void __launch_bounds__(kThreadsG, 1)
    slice_gemm_kernel(const __grid_constant__ CUtensorMap tR, const __grid_constant__ CUtensorMap tQ,
                      const __grid_constant__ OutArgs o, unsigned* flags) {
    using St = Stage<PAIR>;
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
                            for (int p = 0; p < S; ++p) {   // slice p of R stays in the collector
                                const int last = p + S < D ? p + S - 1 : D - 1;
#pragma unroll
                                for (int d = p; d <= last; ++d) {
                                    // accumulator d begins with slice 0, the last one with slice 1
                                    const bool begun = kk != 0 || p != (d < S ? 0 : d - S + 1);
                                    const uint32_t dst = tmem + d * kCols, a = sr + ((p * kRows * kChunk * 2 + kk * 32) >> 4),
                                                   b = sq + (((d - p) * St::kQRows * kChunk * 2 + kk * 32) >> 4),
                                                   acc = begun ? 1u : (kb != 0 ? 1u : 0u);
                                    if (d == p) mma_f16_lo<kKeepFirst, PAIR>(dst, a, b, hi0, idesc, acc);
                                    else if (d < last) mma_f16_lo<kKeepMore, PAIR>(dst, a, b, hi0, idesc, acc);
                                    else mma_f16_lo<kKeepLast, PAIR>(dst, a, b, hi0, idesc, acc);
                                }
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
        constexpr int kShift = -2 * (BETA - 1) - kGather;
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
            unsigned redo = 0;   // pairs of outputs of which some piece does not stand
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
                    cexp[et] = in ? o.ec[z * o.cols + c] : kZeroRow;
                }
                const int er = ro.ok ? o.er[z * o.rows + r] : kZeroRow;
                __syncwarp();
                const unsigned even = certificates(o, z, r - lane, (int64_t)ct * kCols + 16 * h);
                int got = 1;
                if (lane == 0) got = mbar_wait(&ctl->tfull, (uint32_t)it & 1u, &ctl->abort) ? 1 : 0;
                got = __shfl_sync(0xffffffffu, got, 0);
                // the tables are written; if any warp's wait gave up, all sixteen leave together.  (A
                // warp reaches this barrier of the next piece only after reading this one's tables,
                // so two sets suffice.)
                if (!epi_and(got)) { ok = false; break; }
                tc_fence_after();
                long long I[16];
                unsigned fine = 0;
#pragma unroll
                for (int c8 = 0; c8 < 16; c8 += 8) {
                    uint32_t a[2][8];
                    auto load = [&](int d) {
                        tmem_ld8_nw(tq + d * kCols + c8, a[0]);
                        tmem_ld8_nw(tq + (d + 1) * kCols + c8, a[1]);
                        tmem_ld_wait();
                    };
                    load(0);
                    gather<0>(I, c8, a, fine);
                    load(2);
                    gather<1>(I, c8, a, fine);
                    load(4);
                    gather<2>(I, c8, a, fine);
                    load(6);
                    if (c8 == 8) {   // every accumulator of this warp is in registers
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) {
                            if (PAIR) mbar_arrive_cluster_relaxed(mapa_shared(&ctl->tempty, 0));
                            else mbar_arrive(&ctl->tempty);
                        }
                    }
                    gather<3>(I, c8, a, fine);
                }
                unsigned bad = 0;   // pairs of outputs that do not stand
                const bool plain = even == 0xffffu && max(abs(er >> 2), abs(cexp[16 * h + (lane & 15)] >> 2)) <= kMaxExp / 2;
                if (!__all_sync(0xffffffffu, plain)) {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (!stands(er, cexp[16 * h + j], (even >> j) & 1u)) bad |= 1u << (j & ~1);
                    if (!ro.ok) bad = 0;
                }
                auto value = [&](int j) {
                    return round64(I[j], (er >> 2) + (cexp[16 * h + j] >> 2) + kShift - 8 * (int)((fine >> j) & 1u));
                };
#pragma unroll
                for (int j = 0; j < 16; j += 2) {
                    const double z0 = value(j), z1 = value(j + 1);
                    const bool skip = (bad >> j) & 1u;
                    if (MULTI) {
                        acc[MULTI ? j : 0] += skip ? 0.0 : z0;
                        acc[MULTI ? j + 1 : 0] += skip ? 0.0 : z1;
                    } else if (!skip) {
                        store_pair(o, ro, coff, cdof, 16 * h + j, z0, z1);
                    }
                }
                redo |= bad;
                if (MULTI && pc + 1 < p1) continue;
                if (MULTI) {
#pragma unroll
                    for (int j = 0; j < 16; j += 2)
                        store_pair(o, ro, coff, cdof, 16 * h + j, acc[MULTI ? j : 0], acc[MULTI ? j + 1 : 0]);
                }
                const unsigned any = __reduce_or_sync(0xffffffffu, redo);
                if (any) {   // entry: (tile, warp, pair of columns)
                    uint32_t at = 0;
                    if (lane == 0) at = atomicAdd(o.head, (uint32_t)__popc(any));
                    at = __shfl_sync(0xffffffffu, at, 0) + __popc(any & ((1u << lane) - 1u));
                    if (((any >> lane) & 1u) && at < o.room)
                        o.list[at] = (((PAIR ? 2 * w + rank : w) * 16 + 4 * h + q) * 8) + (lane >> 1);
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

// The listed outputs by the multiply-add loop, a warp to an entry: 32 rows by two columns, of which it
// finds again the ones that do not stand (the certificates are exact sums, so it finds the same).  One piece:
// stores them; several: adds the loop over the pieces that do not stand to what was stored.  A lane takes an
// output where at least twelve of the warp's need the loop (its operations take 64 cycles each for the warp
// either way), else the warp takes them one by one.  Bound by the FP64 pipe where many are listed: a product
// of 512 x (128 x 32) outputs and K = 128, real by complex, all of them listed, takes 1.16 ms in all, 0.94 by the
// tiles and 0.09 where none is listed; one of complex operands 1.25, 0.93 and 0.16 (256 x (128 x 32)); real by complex
// products of K = 1024 and more, where the tiles' padding or few CTAs cost more, 4.4, 4.3 and 0.29 (64 x (128 x 128)).
// Graded over a factor of 100 they take 0.51, and 2.7 ms.
template <bool MULTI, bool PAIR>
__global__ void __launch_bounds__(256, 2) slice_loop_kernel(const __grid_constant__ OutArgs o) {
    const int lane = threadIdx.x & 31;
    const uint32_t count = min(*reinterpret_cast<volatile uint32_t*>(o.head), o.room);
    for (uint32_t e = blockIdx.x * 8 + (threadIdx.x >> 5); e < count; e += gridDim.x * 8) {
        const uint32_t id = o.list[e];
        const int j = 2 * (int)(id & 7), warp = (int)(id >> 3) & 15, h = warp >> 2, q = warp & 3;
        const uint32_t tile = id >> 7, w = PAIR ? tile >> 1 : tile;
        uint32_t grp, t, b, ct, rt, ob, i;
        o.dtiles.divmod(w, grp, t);
        o.tile(t, b, ct, rt);
        const int p0 = MULTI ? (int)grp * o.pg : 0, p1 = MULTI ? min(o.pieces, p0 + o.pg) : 1;
        const int64_t r0 = (int64_t)(PAIR ? 2 * rt + (tile & 1u) : rt) * kRows + q * 32, r = r0 + lane;
        const int64_t c0 = (int64_t)ct * kCols + 16 * h, c = c0 + j;
        if (c >= o.cols) continue;
        const bool ok = r < o.rows, two = c + 1 < o.cols;
        double2 sum = make_double2(0.0, 0.0);
        unsigned redo = 0;
#pragma unroll 1
        for (int pc = p0; pc < p1; ++pc) {
            const int64_t z = pc * o.nbatch + b;
            __syncwarp();
            const unsigned even = certificates(o, z, r0, c0) >> j;
            const int er = ok ? o.er[z * o.rows + r] : kZeroRow;
            const int ec0 = o.ec[z * o.cols + c], ec1 = two ? o.ec[z * o.cols + c + 1] : kZeroRow;
            const bool mine = ok && !(stands(er, ec0, even & 1u) && stands(er, ec1, even & 2u));
            const unsigned who = __ballot_sync(0xffffffffu, mine);
            const int k0 = pc * o.klen, k1 = min(o.k, k0 + o.klen);
            double2 y = make_double2(0.0, 0.0);
            if (__popc(who) >= 12) {
                if (mine) y = loop_pair(o, b, k0, k1, (uint32_t)r, (uint32_t)c, -1);
            } else {
#pragma unroll 1
                for (unsigned left = who; left; left &= left - 1u) {
                    const int l = __ffs((int)left) - 1;
                    const double2 v = loop_pair(o, b, k0, k1, (uint32_t)(r0 + l), (uint32_t)c, lane);
                    if (lane == l) y = v;
                }
            }
            if (mine) {
                redo = 1;
                sum = make_double2(sum.x + y.x, sum.y + y.y);
            }
        }
        if (!redo) continue;
        // as in slice_gemm_kernel: offsets of the row and of the columns
        RowOut ro;
        ro.ok = true;
        o.rn.divmod((uint32_t)r >> (o.rexp ? 1 : 0), ob, i);
        ro.roff = o.shared.at(b) + o.rown.at(ob) + i * o.rs + (MULTI ? grp * o.gstride : 0);
        ro.rdof = o.D ? o.dshared.at(b) + o.drown.at(ob) + i * o.drs : 0;
        ro.comp = o.rexp ? (int)(r & 1) : 0;
        int64_t coff[2] = {-1, -1}, cdof[2] = {0, 0};
        for (int u = 0; u < (two ? 2 : 1); ++u) {
            o.cn.divmod((uint32_t)(c + u) >> (o.cexp ? 1 : 0), ob, i);
            coff[u] = o.cown.at(ob) + i * o.cs;
            cdof[u] = o.D ? o.dcown.at(ob) + i * o.dcs : 0;
        }
        if (MULTI) add_pair(o, ro, coff, cdof, 0, sum.x, sum.y);
        else store_pair(o, ro, coff, cdof, 0, sum.x, sum.y);
    }
    // the last CTA empties the list for the next product
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(o.head + 1, 1u) == gridDim.x - 1) {
            o.head[0] = 0u;
            o.head[1] = 0u;
        }
    }
}

// ------------------------------------------------------------------------------------ host side
int64_t up(int64_t n, int64_t m) { return (n + m - 1) / m * m; }

// How one product runs: which batch dimensions fold into which operand's rows, which operand is
// expanded and which one supplies the tile rows.
struct Plan {
    Dims aown{{1, 1, 1}, {0, 0, 0}}, bown = aown, shared_a = aown, shared_b = aown, shared_c = aown, shared_d = aown,
        aown_c = aown, bown_c = aown, aown_d = aown, bown_d = aown;
    int64_t na = 1, nb = 1, ns = 1;       // own batches of A and B, shared batches
    int parts = 1, koff = 0, klen = 0, pieces = 1;
    bool exp_a = false, exp_b = false, swap = false;   // swap: A supplies the tile rows
    int64_t rows_a = 0, rows_b = 0;       // after expansion
    int64_t tiles = 0;                    // pairs of row tiles with `pair`
    bool pair = false;                    // a CTA pair to two neighbouring row tiles
    int groups = 1, pg = 1;               // CTAs that share a tile's pieces, pieces of each
    size_t bytes_p = 0;                   // their partial outputs
    int64_t room = 0;                     // most entries of the list of outputs for the loop
    size_t bytes_a = 0, bytes_b = 0, bytes_l = 0, bytes = 0;
};

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
    p.koff = (int)up(p.klen, 16 / p.parts);   // a row of parts x koff entries is a multiple of 16
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
    auto bytes = [&](int64_t rows) { return up(S * nz * rows * Kp * 2, 1024) + up(4 * nz * rows, 1024); };
    p.bytes_a = bytes(p.rows_a);
    p.bytes_b = bytes(p.rows_b);
    p.groups = (int)std::max<int64_t>(1, std::min<int64_t>(p.pieces, tc_num_sms() / (p.pair ? 2 : 1) / std::max<int64_t>(p.tiles, 1)));
    p.pg = (p.pieces + p.groups - 1) / p.groups;
    p.groups = (p.pieces + p.pg - 1) / p.pg;
    if (p.groups > 1) p.bytes_p = up((int64_t)p.groups * p.na * p.nb * p.ns * g.m * g.n * 16, 1024);
    p.room = p.tiles * (p.pair ? 2 : 1) * p.groups * 128;
    p.bytes_l = up(4 * p.room, 1024);
    p.bytes = p.bytes_a + p.bytes_b + p.bytes_p + p.bytes_l + kSliceHead;
    return p;
}

void launch_pack(PackArgs a, cudaStream_t st) {
    count_launch();
    const int rb = a.koff <= 64 ? 32 : 8;
    const int64_t blocks = (a.own_rows + rb - 1) / rb;
    a.dblocks = Div(blocks);
    const unsigned grid = (unsigned)(blocks * a.nbatch * a.pieces);
    if (rb == 32) pack_slices_kernel<32><<<grid, kPackT, 0, st>>>(a);
    else pack_slices_kernel<8><<<grid, kPackT, 0, st>>>(a);
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
    a.exps = reinterpret_cast<int*>(static_cast<uint8_t*>(buf) + up(S * a.plane * 2, 1024));
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

template <bool PAIR>
void launch_gemm(const CUtensorMap& r, const CUtensorMap& q, const OutArgs& o, unsigned* flags, cudaStream_t st) {
    using St = Stage<PAIR>;
    auto kern = o.pieces > 1 ? slice_gemm_kernel<true, PAIR> : slice_gemm_kernel<false, PAIR>;
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
    count_launch();
    const unsigned grid = 2 * (unsigned)tc_num_sms();
    if (o.pieces > 1) slice_loop_kernel<true, PAIR><<<grid, 256, 0, st>>>(o);
    else slice_loop_kernel<false, PAIR><<<grid, 256, 0, st>>>(o);
}
void launch_gemm(const Plan& p, const CUtensorMap& r, const CUtensorMap& q, const OutArgs& o, unsigned* flags, cudaStream_t st) {
    p.pair ? launch_gemm<true>(r, q, o, flags, st) : launch_gemm<false>(r, q, o, flags, st);
}

// One product that fits the workspace: B's slices at its start, then partial outputs and the list, A's slices
// before the last kSliceHead bytes, the list's counts.  False, with nothing launched, where a tensor map cannot be made.
bool run_plan(const GemmArgs& g, const Plan& p, SliceScratch* ws, cudaStream_t st) {
    uint8_t* buf = static_cast<uint8_t*>(ws->buf);
    // alpha multiplies B, or A where alpha is complex and B real
    const bool on_a = g.B.real && g.alpha.im != 0.0;
    const cplx one{1.0, 0.0};
    const PackArgs pb = pack_args(g.B, false, g.n, g.k, p, buf, on_a ? one : g.alpha);
    const PackArgs pa = pack_args(g.A, true, g.m, g.k, p, buf + (ws->bytes - kSliceHead - p.bytes_a) / 1024 * 1024, on_a ? g.alpha : one);
    const int64_t nz = p.ns * p.pieces;
    const PackArgs &R = p.swap ? pa : pb, &Q = p.swap ? pb : pa;
    const int64_t rr = p.swap ? p.rows_a : p.rows_b, rc = p.swap ? p.rows_b : p.rows_a;
    CUtensorMap mr, mq;
    auto encode = [&](CUtensorMap* m, const PackArgs& x, int64_t rows, int box_rows) {
        const uint64_t dims[4] = {(uint64_t)x.Kp, (uint64_t)rows, (uint64_t)nz, (uint64_t)S};
        const uint64_t str[3] = {(uint64_t)x.Kp * 2, (uint64_t)rows * x.Kp * 2, (uint64_t)x.plane * 2};
        const uint32_t box[4] = {kChunk, (uint32_t)box_rows, 1, (uint32_t)S};
        return make_map4(m, x.out, dims, str, box, 64);
    };
    if (encode(&mr, R, rr, kRows) != AFQMC_OK || encode(&mq, Q, rc, p.pair ? kCols / 2 : kCols) != AFQMC_OK) return false;
    auto kept = [&](bool keep, SliceScratch::Packed& have, const PackArgs& x, int64_t rows, bool is_a) {
        const Dims &own = is_a ? p.aown : p.bown, &shared = is_a ? p.shared_a : p.shared_b;
        SliceScratch::Packed now{x.ptr, x.out, {rows, x.Kp, nz, x.n, x.k, x.klen, x.si, x.sk}, {}, x.scale ? x.alpha : one,
                                 x.real | x.conj << 1 | x.expand << 2 | x.scale << 3};
        for (int i = 0; i < 3; ++i) {
            now.batch[i] = own.cnt[i];
            now.batch[3 + i] = own.str[i];
            now.batch[6 + i] = shared.cnt[i];
            now.batch[9 + i] = shared.str[i];
        }
        const bool same = keep && have == now;
        have = now;
        if (!same) launch_pack(x, st);
    };
    kept(g.keep_b, ws->b, pb, p.rows_b, false);
    kept(g.keep_a, ws->a, pa, p.rows_a, true);
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
    o.dr = R.out;
    o.dc = Q.out;
    o.Kp = (int)R.Kp;
    auto source = [](const PackArgs& x) { return Source{x.ptr, x.real, x.conj, x.si, x.sk, x.own, x.shared}; };
    o.srow = source(R);
    o.scol = source(Q);
    o.k = g.k;
    o.klen = p.klen;
    o.alpha = g.alpha;
    o.list = reinterpret_cast<uint32_t*>(buf + p.bytes_b + p.bytes_p);
    o.head = reinterpret_cast<uint32_t*>(buf + ws->bytes / 1024 * 1024 - kSliceHead);
    o.room = (uint32_t)p.room;
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
        launch_gemm(p, mr, mq, o, ws->flags, st);
        count_launch();
        sum_groups_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(o.C, p.groups, total, g);
    } else {
        launch_gemm(p, mr, mq, o, ws->flags, st);
    }
    return true;
}

}  // namespace

size_t slice_gemm_bytes(const GemmArgs& g) { return make_plan(g).bytes + 1024; }

// Expected time in microseconds: four launches with little in each, the persistent tiles at 65 (pairs: 56) cycles an MMA and 6000
// for the epilogue of each piece, and the operands' packing.
double slice_gemm_us(const GemmArgs& g) {
    if (g.beta.im != 0.0 || (g.A.real && g.B.real && g.alpha.im != 0.0)) return 1e30;
    const Plan p = make_plan(g);
    // 31-bit indices
    const int64_t nz = p.ns * p.pieces, most = 1ll << 31;
    if (std::max(p.rows_a, p.rows_b) >= most || nz * (std::max(p.rows_a, p.rows_b) / 8 + 1) >= most || p.room >= 2 * most)
        return 1e30;
    const double cyc = kMmas * (up((int64_t)p.parts * p.koff, kChunk) / 16) * (p.pair ? 56.0 : 65.0) + 6000.0;
    const int ctas = tc_num_sms() / (p.pair ? 2 : 1);
    const double waves = (double)((p.tiles * p.groups + ctas - 1) / ctas);
    return 29.0 + p.pg * waves * cyc / 1.9e3 + (double)p.bytes / 2.0e6 + (p.groups > 1 ? 4.0 : 0.0);
}

int slice_scratch_init(SliceScratch* ws) {
    if (ws->bytes < 2 * kSliceHead) return AFQMC_OK;   // holds no product
    if (cudaMemset(static_cast<uint8_t*>(ws->buf) + ws->bytes / 1024 * 1024 - kSliceHead, 0, kSliceHead) != cudaSuccess ||
        cudaStreamSynchronize(cudaStreamLegacy) != cudaSuccess)   // before any stream uses it
        return fail(AFQMC_ERR_CUDA, "slice workspace");
    return AFQMC_OK;
}

// Each part of a product that has been cut takes this form or, where it cannot, the tiles: what earlier parts have
// added to C and D is never added again.
void slice_gemm(const GemmArgs& g, SliceScratch* ws, cudaStream_t st) {
    const Plan p = make_plan(g);
    if (p.bytes + 1024 <= ws->bytes) {
        if (!run_plan(g, p, ws, st)) zgemm_as(g, 0, st);
        return;
    }
    // too large for the workspace: cut a long contraction (the output is then added up in rounds) after
    // as many pieces as fit, in equal shares for the CTAs of a tile where that is possible; else
    // halve the largest of the batch dimensions, n and m, and in the end the contraction again
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
    auto cut_k = [&](int k) {
        lo.k = k;
        hi.k = g.k - k;
        shift(k * (g.A.op == OP_N ? 1 : g.A.ld), k * (g.B.op == OP_N ? g.B.ld : 1), 0, 0);
        lo.D = nullptr;
        hi.beta = cplx{1.0, 0.0};
    };
    if (p.pieces >= 32) {
        const int64_t fit = (int64_t)(ws->bytes / ((p.bytes + 1024) / p.pieces + 1));
        const int64_t share = std::max<int64_t>(1, tc_num_sms() / (p.pair ? 2 : 1) / std::max<int64_t>(p.tiles, 1));
        const int64_t n = fit > share ? fit / share * share : std::max<int64_t>(1, fit);
        // (at least a 64th, which may be cut again: bounds the depth of the cuts)
        cut_k((int)std::min<int64_t>(std::max<int64_t>(n, p.pieces / 64), p.pieces - 1) * p.klen);
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
    } else if (p.pieces > 1) {
        cut_k(p.pieces / 2 * p.klen);
    } else {
        zgemm_as(g, 0, st);
        return;
    }
    slice_gemm(lo, ws, st);
    slice_gemm(hi, ws, st);
}

}  // namespace afqmc
