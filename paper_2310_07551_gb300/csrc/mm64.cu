// FP64 mode products on the 5th-generation tensor cores.
//
// GB300's FP64 pipe does 2 FMA per clock and SM (1.25 TFLOP/s in all), three
// orders of magnitude below its FP16 tensor rate, so an FP64 contraction is
// formed here from exact digit products.  Every fibre of an operand (the
// entries that one output sums over) is scaled by a power of two to a 62-bit
// fixed-point number and cut into eight balanced 8-bit digits, held as FP16
// integers: x = 2^(e - 6) (d0 + d1 2^-8 + ... + d7 2^-56), |d0| <= 64,
// |d1..7| <= 128.  The digit products of weight class t = p + q <= 7 (36 of
// 64) run as FP16 MMAs into one FP32 tensor-memory accumulator per class, the
// epilogue recombines the classes in integers and rounds once to FP64.  (The error-free
// splitting of matrix products of Ozaki, Ogita, Oishi and Rump, 2012, with digits of
// a fixed radix.)
//
// What it loses, per contracted entry and in units of the product 2^(ex + el) of the
// two fibres' powers of two: the dropped classes, below 2^-59.2 (seven digit products of
// at most 2^14 at 2^-76); the operands' rounding, 2^-62.  Accumulators: at most 256
// entries are contracted between drains, which bounds class t by t 2^22: classes 0 to
// 4 stay below 2^24 and are exact; 5 to 7 may pass it, where nearly all of more than 200
// entries have extreme digits of the same sign, and then lose a unit (2^-52, 2^-60,
// 2^-68) per MMA.  The drain keeps 2^-66 of class 7 and 2^-60 of the sum.  A chain of
// n FMAs loses 2^-53 of a partial sum per entry, so the digits are the better where
// the sum S of the terms' magnitudes is not small against 2^(ex + el).  Where it is
// (identity or graded matrices, localised states), small entries have few digits of
// their own: such outputs, S below 2^-8, become FMA chains (k_settle), so that every
// output is within n 2^-51 S of its sum, as a chain is within n 2^-53 S.
//
// A fibre holding Inf or NaN carries a flag instead of an exponent: outputs
// of a NaN fibre are NaN, those of an Inf fibre are recomputed by the FP64
// FMA chain in the epilogue.  So are the outputs behind a bounded wait that gave
// up: a call that meets one is slow, and its results are right.
#include <cuda_fp16.h>
#include <limits.h>
#include <stdlib.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "mm64.h"
#include "ptx.cuh"

namespace ds {
namespace mm {

using namespace ptx;

namespace {
constexpr int kNanRow = 32767, kInfRow = 32766, kZeroRow = -16384;   // exponents of non-finite and zero fibres
// Digit sums below 2^-kWeak of their fibres' 2^exponents are looked into (settle).  At
// 2^-8 the dropped classes weigh about as much as an FMA chain's roundings (a random
// walk: 2^-54 sqrt(n) of S); one power of two more would send 4 to 8 times as many outputs of
// a smooth state to the chains (Schnakenberg 301 x 150 at step 1200, second mode: 0.09 %
// of them, 0.5 % at 2^-7).
// entries of at least 2^-kBig of their fibre's are flagged as big, so that one that is
// big in both fibres is a term of 2^-kWeak.
constexpr int kWeak = 8, kBig = kWeak / 2;
constexpr int kChunkSlabs = 16;                           // slabs between drains: 256 entries
constexpr int kSms = 152;

// ---------------------------------------------------------------------------
// Digit images.  One warp takes 2E rows of one slab: lane = (row, E consecutive
// contracted entries), so that every digit plane is written as 64 E contiguous
// bytes.  Up to 16 warps share the slabs of a row group, each
// keeping the first slab it reads in registers, so a fibre of up to 256 entries
// is read once.  24 bytes per entry pass through memory, which bounds large
// tensors; blocks are as small as the slabs allow, so that one block's loads run
// behind another's stores.
// ---------------------------------------------------------------------------
struct SplitArgs {
    int count;
    int *reset;                // set to zero (the products' count of outputs left to k_settle)
    int first[kMaxProd + 1];   // block prefix
    View v[kMaxProd];
    Image im[kMaxProd];
};
constexpr int kSplitWarps = 16;

__host__ __device__ inline int split_warps(int slabs) { return slabs < kSplitWarps ? slabs : kSplitWarps; }

template <int E>
__device__ __forceinline__ void load_entries(const View &v, int64_t base, bool row_ok, int slab, int chunk, int spc,
                                             unsigned long long (&x)[E])
{
    const int t = slab / spc, k0 = (slab - t * spc) * kSlab + chunk * E, left = row_ok ? v.n - k0 : 0;
    const double *src = v.src[t] + base + v.I * k0;
    const double sc = v.scale[t];
    if (v.I == 1 && left >= E && ((uintptr_t)src & 15) == 0) {
#pragma unroll
        for (int j = 0; j < E; j += 2) {
            const longlong2 d = *reinterpret_cast<const longlong2 *>(src + j);
            x[j] = (unsigned long long)d.x;
            x[j + 1] = (unsigned long long)d.y;
        }
    } else {
#pragma unroll
        for (int j = 0; j < E; ++j)
            x[j] = j < left ? (unsigned long long)__double_as_longlong(src[v.I * j]) : 0ULL;
    }
    if (sc != 1.0) {
#pragma unroll
        for (int j = 0; j < E; ++j)
            x[j] = (unsigned long long)__double_as_longlong(__dmul_rn(__longlong_as_double((long long)x[j]), sc));
    }
}

// exponent e with max < 2^e of a fibre's largest magnitude (its bits)
__device__ __forceinline__ int fibre_exp(unsigned long long mx)
{
    const int ef = (int)(mx >> 52);
    if (ef == 0x7FF) return (mx & 0xFFFFFFFFFFFFFULL) ? kNanRow : kInfRow;
    if (ef > 0) return ef - 1022;
    return mx ? (64 - __clzll((long long)mx)) - 1074 : kZeroRow;
}
// magnitude of a slab whose largest entry has these bits: below 2^(code - 1023); 0: all zero
__device__ __forceinline__ uint32_t slab_code(unsigned long long mx) { return mx ? (uint32_t)(mx >> 52) + 1 : 0u; }

// the eight digits of E consecutive entries: bytes of x 2^(62 - e) + 128 in
// every byte, one chunk of 2 E bytes per digit plane.  Returns a bit per big entry.
template <int E>
__device__ __forceinline__ uint32_t store_digits(const unsigned long long (&x)[E], int e, uint8_t *dst, int64_t plane)
{
    uint32_t lo[E], hi[E], big = 0;
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const unsigned long long b = x[j];
        int ef = (int)(b >> 52) & 0x7FF;
        unsigned long long m = b & 0xFFFFFFFFFFFFFULL;
        if (ef) m |= 1ULL << 52; else ef = 1;
        const int sh = ef - 1013 - e;   // <= 9 (<= 61 for subnormal fibres)
        unsigned long long f;
        if (sh >= 0) f = m << (sh & 63);
        else f = sh < -60 ? 0ULL : (m + (1ULL << (-sh - 1))) >> -sh;
        if (e >= kInfRow) f = 0ULL;
        if (f >> (62 - kBig)) big |= 1u << j;
        if ((long long)b < 0) f = 0ULL - f;
        f += 0x8080808080808080ULL;
        lo[j] = (uint32_t)f;
        hi[j] = (uint32_t)(f >> 32);
    }
    const __half2 off = __half2half2(__ushort_as_half((unsigned short)0xE480));   // -1152 = -(1024 + 128)
#pragma unroll
    for (int p = 0; p < kDigits; ++p) {
        uint32_t q[E / 2];
#pragma unroll
        for (int j = 0; j < E / 2; ++j) {
            const uint32_t w0 = p < 4 ? hi[2 * j] : lo[2 * j], w1 = p < 4 ? hi[2 * j + 1] : lo[2 * j + 1];
            const int b = 3 - (p & 3);
            // FP16 1024 + byte, two entries per word
            const uint32_t w = (__byte_perm(w0, w1, b | (b << 4) | ((4 + b) << 8) | ((4 + b) << 12)) & 0x00FF00FFu) |
                               0x64006400u;
            const __half2 h = __hadd2(*reinterpret_cast<const __half2 *>(&w), off);
            q[j] = *reinterpret_cast<const uint32_t *>(&h);
        }
        if constexpr (E == 8) *reinterpret_cast<uint4 *>(dst + p * plane) = make_uint4(q[0], q[1], q[2], q[3]);
        else *reinterpret_cast<uint2 *>(dst + p * plane) = make_uint2(q[0], q[1]);
    }
    return big;
}

template <int E>
__device__ __forceinline__ unsigned long long largest(unsigned long long mx, const unsigned long long (&x)[E])
{
#pragma unroll
    for (int j = 0; j < E; ++j) mx = max(mx, x[j] & 0x7FFFFFFFFFFFFFFFULL);
    return mx;
}

// a slab's mask and code of a row from its lanes' parts; all lanes of a warp
template <int E>
__device__ __forceinline__ void join_lanes(uint32_t &big, uint32_t &code, int chunk)
{
    big <<= chunk * E;
#pragma unroll
    for (int w = 1; w < kSlab / E; w *= 2) {
        big |= __shfl_xor_sync(0xffffffffu, big, w);
        code = max(code, __shfl_xor_sync(0xffffffffu, code, w));
    }
}

// IT: 32-bit row indices where every view allows it (their divisions are a
// good part of a small launch)
template <typename IT, int E>
__global__ void __launch_bounds__(kSplitWarps * 32, 2) k_digits(const __grid_constant__ SplitArgs a)
{
    static_assert(E == 8 || E == 4, "16 or 8 bytes of a digit plane per thread");
    constexpr int kRows = 2 * E, kLaneBits = E == 8 ? 1 : 2;   // rows per warp, log2 of the lanes per row
    __shared__ unsigned long long smax[kSplitWarps][kRows];
    __shared__ int speak[kSplitWarps][kRows];   // the slab of that entry
    int q = 0;
    while (q + 1 < a.count && (int)blockIdx.x >= a.first[q + 1]) ++q;
    const View &v = a.v[q];
    const Image &im = a.im[q];
    const int S = im.slabs, WS = split_warps(S), G = blockDim.x / 32 / WS, spc = S / v.ncat;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int gi = warp / WS, sub = warp % WS;
    const IT rows = (IT)im.rows, rb = (IT)im.rb, I = (IT)v.I;
    const IT groups = (rows + kRows - 1) / kRows, g = (IT)(blockIdx.x - a.first[q]) * G + gi;
    const IT entry = g / groups, group = g - entry * groups;   // batch entry, row group in it
    const int row = lane >> kLaneBits, chunk = lane & ((1 << kLaneBits) - 1);
    const IT r = group * kRows + row, rg = (IT)v.r0 + r;
    const bool in = gi < G && entry < (IT)v.batch, row_ok = in && r < rows;
    const IT o = rg / I;
    const int64_t base = (int64_t)entry * v.stride + (int64_t)o * (v.I * v.n) + (rg - o * I);
    const IT first = r / rb, blocks = (rows + rb - 1) / rb;
    const int rr = (int)(r - first * rb);
    const int64_t plane = (int64_t)im.rb * 32;
    uint8_t *dst = im.data + ((int64_t)entry * blocks + first) * S * kDigits * plane + rr * 32 +
                   (E == 8 ? (chunk ^ ((rr >> 2) & 1)) << 4 : (((chunk >> 1) ^ ((rr >> 2) & 1)) << 4) + ((chunk & 1) << 3));
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0 && a.reset) *a.reset = 0;
    unsigned long long x[E];
    load_entries(v, base, row_ok, min(sub, S - 1), chunk, spc, x);
    unsigned long long mx = largest(0ULL, x);
    const uint32_t code = slab_code(mx);
    int peak = min(sub, S - 1);
    for (int s = sub + WS; s < S; s += WS) {
        unsigned long long w[E];
        load_entries(v, base, row_ok, s, chunk, spc, w);
        const unsigned long long m = largest(0ULL, w);
        if (m > mx) {
            mx = m;
            peak = s;
        }
    }
#pragma unroll
    for (int w = 1; w < kSlab / E; w *= 2) {
        const unsigned long long m = __shfl_xor_sync(0xffffffffu, mx, w);
        const int o = __shfl_xor_sync(0xffffffffu, peak, w);
        if (m > mx) {
            mx = m;
            peak = o;
        }
    }
    if (chunk == 0) {
        smax[warp][row] = mx;
        speak[warp][row] = peak;
    }
    __syncthreads();
    pdl_trigger();
    if (!in) return;
    for (int w = 0; w < WS; ++w) mx = max(mx, smax[gi * WS + w][row]);
    const int e = fibre_exp(mx);
    if (sub == 0 && chunk == 0 && row_ok) {
        int w = 0;
        while (w < WS - 1 && smax[gi * WS + w][row] != mx) ++w;
        im.exps[(int64_t)entry * blocks * rb + r] = speak[gi * WS + w][row] << 16 | (e & 0xFFFF);
    }
    const int64_t at = ((int64_t)entry * blocks + first) * S * im.rb + rr;   // of the row's mask and code in slab 0
    auto note = [&](int s, uint32_t big, uint32_t code) {
        join_lanes<E>(big, code, chunk);
        if (chunk == 0 && row_ok) {
            im.masks[at + (int64_t)s * im.rb] = (uint16_t)big;
            im.codes[at + (int64_t)s * im.rb] = (uint16_t)code;
        }
    };
    if (sub < S) note(sub, store_digits(x, e, dst + (int64_t)sub * kDigits * plane, plane), code);
    for (int s = sub + WS; s < S; s += WS) {
        unsigned long long w[E];
        load_entries(v, base, row_ok, s, chunk, spc, w);
        note(s, store_digits(w, e, dst + (int64_t)s * kDigits * plane, plane), slab_code(largest(0ULL, w)));
    }
}

// ---------------------------------------------------------------------------
// The digit products.  One persistent CTA per SM; warp 0 copies digit blocks (one
// contiguous block per operand and slab) into a four-stage ring, warp 1 issues
// the MMAs, four warpgroups drain.  A tile is 128 rows by `nt` <=
// 64 columns: eight classes of 64 FP32 columns are all 512 columns of tensor
// memory.  Such a tile reads 48 KiB of digits per 1152 clocks of MMAs, 42 bytes
// per clock and SM, which the L2 does not always give; but sharing the row block
// between two CTAs costs more than it saves.  Each CTA for itself: 301 x 150 four
// steps 570 us, complex 150 x 150 305 us, Tucker 201 x 150 x 67 142 us, 96^3 with
// adjoint 9.98 ms; a cluster of two that loads half of the rows each and multicasts
// them: 616, 311, 153, 10.06; halves passed on from shared memory to shared memory:
// 893, 513, 189, 13.1.  (Multicast loads are out of the library in any case: it also
// runs on several GPUs.)  The digit planes of
// B lie one after the other in shared memory, so digit p of A meets up to
// 256 / nt digits of B in one MMA, whose output columns are the adjacent classes.
// ---------------------------------------------------------------------------
struct GProd {
    const uint8_t *A, *B;
    const int *eA, *eB;
    const uint16_t *mA, *mB, *cA, *cB;   // masks and codes
    double *out;
    int slabs, nt, ntiles, mtiles, cols, accumulate, ncat, n;
    int64_t rows, r0, I, IB, sA, sB, sOut;   // strides of a batch
    const double *X[kMaxCat], *L[kMaxCat];
    double sc[kMaxCat];
};
// Outputs of a tile that a drain leaves to k_settle: column c of it, the rows of a lane
// quarter that have a bit in `rows`; exps: the column's exponent and slab (Image::exps).
struct Left {
    uint16_t prod, c;
    int entry, mi, ni;         // (ni: tile times four, plus the quarter)
    uint32_t rows;
    int exps;
};
static_assert(sizeof(Left) == 24, "as left_bytes has it");
struct GArgs {
    int count;
    int first[kMaxProd + 1];   // prefix of tiles
    int *nleft;
    Left *left;                // room for every tile's
    long long wait_limit;
    GProd p[kMaxProd];
};

// Five warpgroups: copies and MMAs (warps 0, 1; 2 and 3 idle), then four that
// drain, of a quarter of the columns each.  The first gives registers up: 128 x
// 32 + 512 x 112 = 640 x 96, the launch's total; a drain thread holds up to 16
// outputs as two 64-bit integers.
constexpr int kThreads = 640, kEpiThreads = 512, kStages = 4, kEpiCols = 16;
constexpr uint32_t kPlaneA = kRowBlock * 32, kStageA = kDigits * kPlaneA, kStageB = kDigits * 64 * 32;
constexpr uint32_t kStageBytes = kStageA + kStageB;
constexpr uint32_t kBars = 2 * kStages + 3;
constexpr uint32_t kSmem = kStages * kStageBytes + 128 + 1024;
static_assert(8 * kBars + 8 <= 128, "barriers and two words behind the ring");

// tile u: its product (q: the product of an earlier one), batch entry, row tile and
// column tile
__device__ __forceinline__ const GProd &find_tile(const GArgs &a, int u, int &q, int &entry, int &mi, int &ni)
{
    while (q + 1 < a.count && u >= a.first[q + 1]) ++q;
    const GProd &p = a.p[q];
    const int t = u - a.first[q], row = t / p.ntiles;
    ni = t - row * p.ntiles;
    entry = row / p.mtiles;
    mi = row - entry * p.mtiles;
    return p;
}

// The MMAs of one slab: 36 digit products, in 12 (8, for at most 32 columns)
// instructions.  Digit p of A stays in the collector buffer across the
// instructions that share it.  fresh: the accumulators start at zero (digit 0 of
// A meets every digit of B, that is every class, first).  Issued from compile-
// time tables: with the descriptors formed in a loop one thread took 400 clocks
// per instruction, three times the MMAs' own time.
template <int NT>
__device__ __forceinline__ void issue_slab(uint32_t tmem, uint32_t sA, uint32_t sB, bool fresh)
{
    constexpr int PER = 256 / NT < kDigits ? 256 / NT : kDigits;   // digits of B per MMA
    const uint64_t a0 = desc_sw32(sA), b0 = desc_sw32(sB);
#pragma unroll
    for (int p = 0; p < kDigits; ++p) {
        const uint64_t ad = a0 + (uint64_t)(p * kPlaneA >> 4);
        const uint32_t acc = p == 0 && fresh ? 0u : 1u;
        const int nq = kDigits - p;
#pragma unroll
        for (int q = 0; q < nq; q += PER) {
            const int w = nq - q < PER ? nq - q : PER;
            const uint64_t bd = b0 + (uint64_t)(q * NT * 32 >> 4);
            const uint32_t d = tmem + (p + q) * NT, id = idesc_f16(kRowBlock, w * NT);
            if (nq <= PER) mma_f16<0>(d, ad, bd, id, acc);
            else if (q == 0) mma_f16<1>(d, ad, bd, id, acc);
            else if (q + PER < nq) mma_f16<2>(d, ad, bd, id, acc);
            else mma_f16<3>(d, ad, bd, id, acc);
        }
    }
}

// all eight classes of four columns, complete on return
__device__ __forceinline__ void load_classes(uint32_t taddr, uint32_t cs, uint32_t (&v)[32])
{
    asm volatile(
        "{\n\t.reg .b32 t;\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%32];\n\t"
        "add.u32 t, %32, %33;\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4, %5, %6, %7}, [t];\n\t"
        "add.u32 t, t, %33;\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8, %9, %10, %11}, [t];\n\t"
        "add.u32 t, t, %33;\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12, %13, %14, %15}, [t];\n\t"
        "add.u32 t, t, %33;\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16, %17, %18, %19}, [t];\n\t"
        "add.u32 t, t, %33;\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%20, %21, %22, %23}, [t];\n\t"
        "add.u32 t, t, %33;\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%24, %25, %26, %27}, [t];\n\t"
        "add.u32 t, t, %33;\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%28, %29, %30, %31}, [t];\n\t"
        "tcgen05.wait::ld.sync.aligned;\n\t}\n"
        : "=&r"(v[0]), "=&r"(v[1]), "=&r"(v[2]), "=&r"(v[3]), "=&r"(v[4]), "=&r"(v[5]), "=&r"(v[6]), "=&r"(v[7]),
          "=&r"(v[8]), "=&r"(v[9]), "=&r"(v[10]), "=&r"(v[11]), "=&r"(v[12]), "=&r"(v[13]), "=&r"(v[14]),
          "=&r"(v[15]), "=&r"(v[16]), "=&r"(v[17]), "=&r"(v[18]), "=&r"(v[19]), "=&r"(v[20]), "=&r"(v[21]),
          "=&r"(v[22]), "=&r"(v[23]), "=&r"(v[24]), "=&r"(v[25]), "=&r"(v[26]), "=&r"(v[27]), "=&r"(v[28]),
          "=&r"(v[29]), "=&r"(v[30]), "=&r"(v[31])
        : "r"(taddr), "r"(cs)
        : "memory");
}

// The classes of a thread's `hc` columns as P 2^38 + Q in units of 2^-14 of class
// 5: classes 0 .. 2 in P, the rest in Q.  ADD: on top of the earlier entries'.
template <bool ADD>
__device__ __forceinline__ void drain(uint32_t taddr, uint32_t cs, int hc, long long (&P)[kEpiCols], long long (&Q)[kEpiCols])
{
#pragma unroll
    for (int g = 0; g < kEpiCols / 4; ++g) {
        if (g * 4 < hc) {
            uint32_t v[32];
            load_classes(taddr + g * 4, cs, v);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                auto cls = [&](int t) { return __uint_as_float(v[t * 4 + j]); };
                // |class 0| <= 2^20, |class 1| <= 2^22: integers by adding 1.5 2^23
                // (the conversion unit takes 16 values per clock and SM, as long for
                // six classes as the MMAs of 96 entries)
                const int c0 = __float_as_int(cls(0) + 12582912.0f) - 0x4B400000;
                const int c1 = __float_as_int(cls(1) + 12582912.0f) - 0x4B400000;
                const int c2 = __float2int_rn(cls(2)), c3 = __float2int_rn(cls(3)), c4 = __float2int_rn(cls(4));
                const int c5 = __float2int_rn(cls(5)), c6 = __float2int_rn(fmaf(cls(7), 0.25f, 64.0f * cls(6)));
                const long long hp = (long long)c0 * 65536 + (c1 * 256 + c2);
                const long long lp = (long long)c3 * 1073741824 + ((long long)c4 * 4194304 + ((long long)c5 * 16384 + c6));
                P[g * 4 + j] = ADD ? P[g * 4 + j] + hp : hp;
                Q[g * 4 + j] = ADD ? Q[g * 4 + j] + lp : lp;
            }
        }
    }
}

// P 2^38 + Q rounded to 53 bits, in 32-bit integers without branches (the FP64
// pipe would take longer than the digit products).  The value is hi:lo, with the
// leading bit at bit 52, times 2^(E - 52) and the sign.
struct Rounded {
    uint32_t lo, hi, sign;
    int E;
};
__device__ __forceinline__ Rounded round_sum(long long P, long long Q, int e)
{
    // 96 bits: H = P + (Q >> 38) above 32 of the low 38 bits of Q; their
    // magnitude
    const long long H = P + (Q >> 38);
    uint32_t w0 = (uint32_t)(Q >> 6), w1 = (uint32_t)H, w2 = (uint32_t)((unsigned long long)H >> 32);
    const uint32_t neg = (uint32_t)((int)w2 >> 31);
    asm("{\n\t.reg .u32 a, b, c;\n\txor.b32 a, %0, %3;\n\txor.b32 b, %1, %3;\n\txor.b32 c, %2, %3;\n\t"
        "sub.cc.u32 %0, a, %3;\n\tsubc.cc.u32 %1, b, %3;\n\tsubc.u32 %2, c, %3;\n\t}"
        : "+r"(w0), "+r"(w1), "+r"(w2)
        : "r"(neg));
    // leading word up, then the leading bit
    const bool z = w2 == 0;
    w2 = z ? w1 : w2;
    w1 = z ? w0 : w1;
    w0 = z ? 0u : w0;
    const int lz = __clz((int)w2);
    const uint32_t m1 = __funnelshift_l(w1, w2, lz), m0 = __funnelshift_l(w0, w1, lz);
    Rounded r;
    // 53 of the 64 leading bits, to nearest; a carry moves up into the exponent
    asm("{\n\t.reg .u32 a, b, c;\n\tadd.cc.u32 a, %2, 0x400;\n\taddc.cc.u32 b, %3, 0;\n\taddc.u32 c, 0, 0;\n\t"
        "shf.r.clamp.b32 %0, a, b, 11;\n\tshf.r.clamp.b32 %1, b, c, 11;\n\t}"
        : "=r"(r.lo), "=r"(r.hi)
        : "r"(m0), "r"(m1));
    r.sign = neg & 0x80000000u;
    r.E = e + 93 - lz - (z ? 32 : 0);
    if (w2 == 0) r.E = INT_MIN / 2;   // |H| = 0: left to round_rare
    return r;
}
// what round_sum leaves: zero, sums below 2^-30 of class 2's unit, results
// outside the normal range
__device__ __noinline__ double round_rare(long long P, long long Q, int e)
{
    const long long H = P + (Q >> 38), L = Q & 0x3FFFFFFFFF;
    const bool neg = H < 0;
    // |H| 2^38 + |L|; the low bits go where it is 2^63 or more
    const long long h = neg ? -H - (L ? 1 : 0) : H, l = neg && L ? 0x4000000000 - L : L;
    int sh = 0;
    while (h >> (25 + sh)) ++sh;
    unsigned long long V = ((unsigned long long)h << (38 - sh)) | ((unsigned long long)l >> sh);
    if (V == 0) return 0.0;
    const int lz = __clzll((long long)V);
    V <<= lz;
    unsigned long long m = (V >> 11) + (V >> 10 & 1);
    const int E = e - 8 + sh - lz + 63;   // m 2^(E - 52)
    if (E < -1200) return neg ? -0.0 : 0.0;
    const double r = scalbn((double)m, max(-2000, min(2000, E)) - 52);
    return neg ? -r : r;
}

// the FP64 FMA chain of one output
__device__ __forceinline__ double fma_chain(const GProd &p, int64_t entry, int64_t r, int i)
{
    double total = 0.0;
    const int64_t xa = entry * p.sA + (r / p.I) * (p.I * p.n) + r % p.I;
    const int64_t lb = entry * p.sB + (i / p.IB) * (p.IB * p.n) + i % p.IB;
    for (int t = 0; t < p.ncat; ++t) {
        const double *x = p.X[t] + xa, *l = p.L[t] + lb;
        double s = 0.0;
        for (int k = 0; k < p.n; ++k) s = fma(x[p.I * k], l[p.IB * k], s);
        total = t ? total + p.sc[t] * s : p.sc[t] * s;
    }
    return total;
}

// Lower bound, in units of 2^-28 of the fibres' 2^exponents, of the summed magnitudes of
// the terms of slab s (of every concatenated operand) of row m and column c of a tile,
// from its two leading digits v = 256 d0 + d1: |v| stands for at least |v| - 1/2.
__device__ __forceinline__ float leading_terms(const GProd &p, const uint8_t *A, const uint8_t *B, int spc, int s, int m, int c)
{
    const int nt = p.nt, sa = (m >> 2) & 1, sb = (c >> 2) & 1;
    float sum = 0.0f;
    for (int t = 0; t < p.ncat; ++t) {
        const uint4 *a = reinterpret_cast<const uint4 *>(A + (int64_t)(t * spc + s) * kStageA + m * 32);
        const uint4 *b = reinterpret_cast<const uint4 *>(B + (int64_t)(t * spc + s) * (nt * 32 * kDigits) + c * 32);
        uint4 x[2][2], y[2][2];   // digit, half of the slab
#pragma unroll
        for (int d = 0; d < 2; ++d)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                x[d][h] = __ldg(a + d * (kPlaneA / 16) + (h ^ sa));
                y[d][h] = __ldg(b + d * (nt * 2) + (h ^ sb));
            }
        auto pair = [](uint32_t lead, uint32_t next) {   // two entries' |v| - 1/2, not negative
            const float2 u = __half22float2(*reinterpret_cast<const __half2 *>(&lead)), w = __half22float2(*reinterpret_cast<const __half2 *>(&next));
            return make_float2(fmaxf(fabsf(fmaf(256.0f, u.x, w.x)) - 0.5f, 0.0f), fmaxf(fabsf(fmaf(256.0f, u.y, w.y)) - 0.5f, 0.0f));
        };
        auto quad = [&](const uint4 &x0, const uint4 &x1, const uint4 &y0, const uint4 &y1) {
            const uint32_t xl[4] = {x0.x, x0.y, x0.z, x0.w}, xn[4] = {x1.x, x1.y, x1.z, x1.w};
            const uint32_t yl[4] = {y0.x, y0.y, y0.z, y0.w}, yn[4] = {y1.x, y1.y, y1.z, y1.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 u = pair(xl[q], xn[q]), v = pair(yl[q], yn[q]);
                sum = fmaf(u.x, v.x, fmaf(u.y, v.y, sum));
            }
        };
        quad(x[0][0], x[1][0], y[0][0], y[1][0]);
        quad(x[0][1], x[1][1], y[0][1], y[1][1]);
    }
    return sum;
}

// Outputs that are small against the largest entries of their fibres (Left), by W warps.
// The digit sum stands where the leading digits, in the slab with the column's largest
// entry, show terms that add up to 2^-kWeak of the fibres' 2^exponents (a zero crossing
// of a smooth state has them, but none that is big in both fibres).  The others become
// FMA chains.  (accumulate: all of them; their digit sums were not added.)
//   Few of them: sixteen lanes for an output, each with eight entries on their way.
// Many (graded operands): a lane per row, its chain over every fourth slab (in each of
// four warps), first those whose bounds are within 2^-24 of the largest, then those that
// are not beyond 2^-56 of the sums so far.  The FP64 pipe bounds that: a DFMA of a
// warp takes its quarter of the SM 64 clocks.  W does not change a sum's order.
constexpr int kFew = 8, kSettleThreads = 128, kSettleBlocks = 4;   // (blocks per SM)
struct SettleShared {
    int most[4][32];
    double part[4][32];   // warp, row
};
template <int W>
__device__ __forceinline__ void settle(const GProd &p, const Left &g, SettleShared &sh)
{
    const uint32_t all = 0xffffffffu;
    const int tid = threadIdx.x % (32 * W), warp = tid / 32, lane = tid % 32;
    const int S = p.slabs, ncat = p.ncat, spc = S / ncat, n = p.n, nt = p.nt;
    const int mi = g.mi, ni = g.ni / 4, m0 = g.ni % 4 * 32, c = g.c;
    const int64_t I = p.I, IB = p.IB, entry = g.entry, ta = entry * p.mtiles + mi, tb = entry * p.ntiles + ni;
    uint32_t rows = g.rows;
    if (!p.accumulate) {
        const int s = (g.exps >> 16) % spc, ec = (int16_t)g.exps;
        bool look = true;
        if constexpr (W == 1) {
            // (graded operands: the slab's bound says no as soon)
            const int er = (int16_t)__ldg(p.eA + ta * kRowBlock + m0 + lane);
            int b = 0;
            for (int t = 0; t < ncat; ++t)
                b = max(b, (int)__ldg(p.cA + (ta * S + t * spc + s) * kRowBlock + m0 + lane) + (int)__ldg(p.cB + (tb * S + t * spc + s) * nt + c));
            // 16 ncat <= 96 products below 2^(b - 2046)
            look = __any_sync(all, (rows >> lane & 1) && b - 2046 + 7 > er + ec - kWeak);
        }
        if (look)
            rows &= __ballot_sync(all, leading_terms(p, p.A + ta * S * kStageA, p.B + tb * S * (nt * 32 * kDigits), spc, s, m0 + lane, c) <
                                           1.001f * (float)(1 << (28 - kWeak)));
        if (rows == 0) return;
    }
    auto place = [&](int row, int64_t &x, int64_t &y) {   // a row's first entry, its output
        const int64_t rg = p.r0 + (int64_t)mi * kRowBlock + m0 + row;
        const int64_t ro = (rg | I) >> 32 ? rg / I : (int64_t)((uint32_t)rg / (uint32_t)I);
        x = entry * p.sA + ro * (I * n) + (rg - ro * I);
        y = entry * p.sOut + ro * (I * p.cols) + (rg - ro * I) + I * (ni * nt + c);
    };
    auto put = [&](int64_t y, double t) { p.out[y] = p.accumulate ? __dadd_rn(p.out[y], t) : t; };
    const uint32_t col = (uint32_t)(ni * nt + c), co = col / (uint32_t)IB;
    const int64_t ls = entry * p.sB + co * (IB * n) + (col - co * (uint32_t)IB);   // the column's first entry
    int64_t xs, ys;
    const int count = __popc(rows);
    if (count <= kFew) {
        constexpr int step = 16, share = 32 * W / step;
        const int sub = tid % step;
        for (int first = 0; first < count; first += share) {
            const int mine = first + tid / step;
            place((int)__fns(rows, 0, min(mine, count - 1) + 1), xs, ys);   // (the last one again where they run out)
            double total = 0.0;
            for (int t = 0; t < ncat; ++t) {
                const double *x = p.X[t] + xs, *l = p.L[t] + ls;
                double sum = 0.0;
                for (int k0 = sub; k0 - sub < n; k0 += 8 * step) {
                    double xv[8], lv[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int k = k0 + i * step;
                        xv[i] = k < n ? x[I * k] : 0.0;
                        lv[i] = k < n ? l[IB * k] : 0.0;
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (k0 - sub + i * step < n) sum = fma(xv[i], lv[i], sum);
                }
                total = fma(p.sc[t], sum, total);
            }
#pragma unroll
            for (int w = step / 2; w; w /= 2) total += __shfl_xor_sync(all, total, w);
            if (sub == 0 && mine < count) put(ys, total);
        }
        return;
    }
    const bool weak = rows >> lane & 1;
    const uint16_t *ca = p.cA + ta * S * kRowBlock + m0 + lane, *cb = p.cB + tb * S * nt + c;
    // products of slab s are below 2^(bound - 2046); 0: all zero
    auto bound = [&](int s) {
        const int b = __ldg(cb + s * nt), r = __ldg(ca + s * kRowBlock);
        return weak && r && b ? r + b : 0;
    };
    int most = 0;
#pragma unroll 8
    for (int s = warp; s < S; s += W) most = max(most, bound(s));
    if constexpr (W > 1) {
        __syncthreads();   // (the outputs before are done with the shared memory)
        sh.most[warp][lane] = most;
        __syncthreads();
        most = max(max(sh.most[0][lane], sh.most[1][lane]), max(sh.most[2][lane], sh.most[3][lane]));
    }
    place(lane, xs, ys);
    const int from = max(most - 24, 1);
    int floor = from;   // slabs of a smaller bound do not matter (yet)
    double total = 0.0;
    for (int pass = 0; pass < 2; ++pass) {
        double half = 0.0, quarter = 0.0;   // (W = 1) parts 0 (+ 1), part 2
#pragma unroll 1
        for (int first = W == 1 ? 0 : warp; first < (W == 1 ? 4 : warp + 1); ++first) {
            double mine = 0.0, sum = 0.0;
            int t = 0;
            for (int s = first; s < S; s += 4) {
                const int b = bound(s), u = s / spc;
                if (!__any_sync(all, b && b >= floor) || (pass && __any_sync(all, b >= from))) continue;
                if (u != t) {
                    mine = fma(p.sc[t], sum, mine);
                    sum = 0.0;
                    t = u;
                }
                const int k0 = (s - u * spc) * kSlab, ki = lane % kSlab;
                const double *x = p.X[u] + xs;
                double xv[kSlab];
#pragma unroll
                for (int i = 0; i < kSlab; ++i) xv[i] = weak && k0 + i < n ? x[I * (k0 + i)] : 0.0;
                const double lk = k0 + ki < n ? p.L[u][ls + IB * (k0 + ki)] : 0.0;
#pragma unroll
                for (int i = 0; i < kSlab; ++i) sum = fma(xv[i], __shfl_sync(all, lk, i), sum);
            }
            mine = fma(p.sc[t], sum, mine);
            if constexpr (W > 1) {
                sh.part[warp][lane] = mine;
            } else {
                if (first == 0) half = mine;
                else if (first == 1) half += mine;
                else if (first == 2) quarter = mine;
                else total += half + (quarter + mine);
            }
        }
        if constexpr (W > 1) {
            __syncthreads();
            total += (sh.part[0][lane] + sh.part[1][lane]) + (sh.part[2][lane] + sh.part[3][lane]);
            __syncthreads();
        }
        // S slabs of 16 products below 2^(b - 2046) are below 2^-56 of |total|
        if (pass == 0 && weak) floor = min(floor, (total == 0.0 ? -100000 : ilogb(total)) - 56 + 2046 - 4 - (32 - __clz(S)));
    }
    if (warp == 0 && weak) put(ys, total);
}

// A kernel of its own because what is left to it clusters: settled by the CTA of their
// tile, ten groups of outputs took 240k clocks where the other CTAs took 40k.  A block
// takes a column's where they are few (latency), each of its warps one where they are
// many.  (301 x 150 four steps, late: 818 us, with four columns to a block 890; complex
// 150 x 150 469, 496; the phi setup of 256 x 200, where they are many, 26.2 ms, 24.8.)
__global__ void __launch_bounds__(kSettleThreads, kSettleBlocks) k_settle(const __grid_constant__ GArgs a)
{
    __shared__ SettleShared sh;
    pdl_trigger();
    pdl_wait();
    const int items = *a.nleft;
    if (items <= 4 * (int)gridDim.x) {
        for (int i = blockIdx.x; i < items; i += gridDim.x) settle<4>(a.p[a.left[i].prod], a.left[i], sh);
    } else {
        for (int i = blockIdx.x * 4 + threadIdx.x / 32; i < items; i += gridDim.x * 4) settle<1>(a.p[a.left[i].prod], a.left[i], sh);
    }
}

__global__ void __launch_bounds__(kThreads, 1) k_digit_products(const __grid_constant__ GArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_addr(smem_raw), base = (raw + 1023u) & ~1023u;
    const uint32_t bars = base + kStages * kStageBytes;
    uint32_t *tmem_slot = (uint32_t *)(smem_raw + (bars - raw) + 8 * kBars);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
    const uint32_t FULL = bars, EMPTY = FULL + 8 * kStages, TFULL = EMPTY + 8 * kStages, TEMPTY = TFULL + 8, DRAIN = TFULL + 16;
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x / 32, 0), lane = threadIdx.x % 32;
    const int tiles = a.first[a.count];
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2 * kStages; ++s) bar_init(bars + 8 * s, 1);
        bar_init(TFULL, 1);
        bar_init(TEMPTY, kEpiThreads);
        bar_init(DRAIN, 1);
        *abort_flag = 0;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = *tmem_slot;
    pdl_trigger();
    pdl_wait();

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
        if (warp == 0) {
            int stage = 0, q = 0, issued = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int u = blockIdx.x; ok && u < tiles; u += gridDim.x) {
                int be, mi, ni;
                const GProd &p = find_tile(a, u, q, be, mi, ni);
                const uint32_t nb = (uint32_t)p.nt * 32 * kDigits;
                const int slabs = p.slabs;
                const uint8_t *A = p.A + ((int64_t)be * p.mtiles + mi) * slabs * kStageA;
                const uint8_t *B = p.B + ((int64_t)be * p.ntiles + ni) * slabs * nb;
                for (int s = 0; s < slabs; ++s) {
                    ok = __all_sync(0xffffffffu, bar_wait(EMPTY + 8 * stage, phase ^ 1u, abort_flag, a.wait_limit));
                    if (!ok) break;
                    if (elect_one()) {
                        const uint32_t sA = base + stage * kStageBytes;
                        bar_expect(FULL + 8 * stage, kStageA + nb);
                        bulk_load(sA, A, kStageA, FULL + 8 * stage);
                        bulk_load(sA + kStageA, B, nb, FULL + 8 * stage);
                    }
                    __syncwarp();
                    A += kStageA;
                    B += nb;
                    ++issued;
                    if (++stage == kStages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            // every issued copy lands before the CTA exits
            volatile int never = 0;
            for (int s = max(0, issued - kStages); s < issued; ++s)
                bar_wait(FULL + 8 * (s % kStages), s / kStages & 1, &never, kWaitCycles);
        }
        if (warp == 1) {
            int stage = 0, q = 0;
            uint32_t phase = 0, tphase = 0;
            bool ok = true;
            for (int u = blockIdx.x; ok && u < tiles; u += gridDim.x) {
                int be, mi, ni;
                const GProd &p = find_tile(a, u, q, be, mi, ni);
                const int nt = p.nt, slabs = p.slabs;
                for (int s = 0; s < slabs; ++s) {
                    const bool fresh = s % kChunkSlabs == 0;
                    if (fresh) {
                        ok = __all_sync(0xffffffffu, bar_wait(TEMPTY, tphase ^ 1u, abort_flag, a.wait_limit));
                        if (!ok) break;
                        tphase ^= 1u;
                    }
                    ok = __all_sync(0xffffffffu, bar_wait(FULL + 8 * stage, phase, abort_flag, a.wait_limit));
                    if (!ok) break;
                    tc_after();
                    const uint32_t sA = base + stage * kStageBytes, sB = sA + kStageA;
                    if (elect_one()) {
                        switch (nt) {
                        case 64: issue_slab<64>(tmem, sA, sB, fresh); break;
                        case 48: issue_slab<48>(tmem, sA, sB, fresh); break;
                        case 32: issue_slab<32>(tmem, sA, sB, fresh); break;
                        default: issue_slab<16>(tmem, sA, sB, fresh); break;
                        }
                        mma_commit_to(EMPTY + 8 * stage);
                        if (s + 1 == slabs || s % kChunkSlabs == kChunkSlabs - 1) mma_commit_to(TFULL);
                    }
                    __syncwarp();
                    if (++stage == kStages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            if (elect_one()) mma_commit_to(DRAIN);
            __syncwarp();
            volatile int never = 0;
            bar_wait(DRAIN, 0, &never, kWaitCycles);
        }
    } else {
        // warp w reads the tensor-memory lanes 32 (w % 4) ..; the four warps of a
        // lane quarter take a quarter of the columns each
        asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
        const int quarter = warp % 4, part = (warp - 4) / 4;
        const int m = quarter * 32 + lane;
        uint32_t tphase = 0;
        bool ok = true;
        int q = 0;
        for (int u = blockIdx.x; u < tiles; u += gridDim.x) {
            int be, mi, ni;
            const GProd &p = find_tile(a, u, q, be, mi, ni);
            const int nt = p.nt, hc = nt / 4, cw = part * hc;   // the warp's first column in the tile
            const int64_t r = (int64_t)mi * kRowBlock + m;
            const bool row_ok = r < p.rows;
            const int c0 = ni * nt + cw;
            const int64_t rg = p.r0 + r, ro = (rg | p.I) >> 32 ? rg / p.I : (int64_t)((uint32_t)rg / (uint32_t)p.I);
            double *const out = p.out + be * p.sOut + ro * (p.I * p.cols) + (rg - ro * p.I) + p.I * c0;
            // exponents, and where the columns have their largest entries, while the MMAs run
            const int er = row_ok ? (int16_t)__ldg(p.eA + (int64_t)be * p.mtiles * kRowBlock + r) : 0;
            const int wc = lane < hc && c0 + lane < p.cols ? __ldg(p.eB + (int64_t)be * p.ntiles * nt + c0 + lane) : 0;
            // a column of the warp's that is not finite: every row takes the slow form
            const bool odd_col = __any_sync(0xffffffffu, (int16_t)wc >= kInfRow);
            long long P[kEpiCols], Q[kEpiCols];
            for (int s0 = 0; s0 < p.slabs; s0 += kChunkSlabs) {
                ok = ok && __all_sync(0xffffffffu, bar_wait(TFULL, tphase, abort_flag, a.wait_limit));
                if (!ok) break;
                tphase ^= 1u;
                tc_after();
                const uint32_t tq = tmem + (uint32_t)cw + ((uint32_t)(quarter * 32) << 16);
                if (s0 == 0) drain<false>(tq, (uint32_t)nt, hc, P, Q);
                else drain<true>(tq, (uint32_t)nt, hc, P, Q);
                tc_before();
                bar_arrive(TEMPTY);
            }
            const bool odd = !ok || odd_col || er >= kInfRow;
            // (every lane takes part in the shuffles of the column exponents)
            if (!__all_sync(0xffffffffu, odd)) {
                uint32_t weak = 0;   // columns whose sums are small against their fibres
                const bool mine = row_ok && !odd;
#pragma unroll
                for (int g = 0; g < kEpiCols / 4; ++g) {
                    if (g * 4 < hc && c0 + g * 4 < p.cols) {
                        double z[4];
                        bool rare = false;
                        int e[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            e[j] = er + (int16_t)__shfl_sync(0xffffffffu, wc, g * 4 + j) - 58;
                            const Rounded y = round_sum(P[g * 4 + j], Q[g * 4 + j], e[j]);
                            const uint32_t x = (uint32_t)(y.E + 1022);   // biased exponent - 1
                            rare |= x >= 2045u;
                            if (y.E < e[j] + 58 - kWeak) weak |= 1u << (g * 4 + j);
                            z[j] = __hiloint2double((int)((y.hi + (x << 20)) | y.sign), (int)y.lo);
                        }
                        if (rare) {
#pragma unroll 1
                            for (int j = 0; j < 4; ++j) {
                                const long long pj = j == 0 ? P[g * 4] : j == 1 ? P[g * 4 + 1] : j == 2 ? P[g * 4 + 2] : P[g * 4 + 3];
                                const long long qj = j == 0 ? Q[g * 4] : j == 1 ? Q[g * 4 + 1] : j == 2 ? Q[g * 4 + 2] : Q[g * 4 + 3];
                                const int ej = j == 0 ? e[0] : j == 1 ? e[1] : j == 2 ? e[2] : e[3];
                                const double r = round_rare(pj, qj, ej);
                                if (j == 0) z[0] = r;
                                else if (j == 1) z[1] = r;
                                else if (j == 2) z[2] = r;
                                else z[3] = r;
                            }
                        }
                        double *o = out + p.I * (g * 4);
                        if (!mine) continue;
                        if (c0 + g * 4 + 3 < p.cols && !p.accumulate) {
                            if (p.I == 1 && ((uintptr_t)o & 31) == 0) {
                                asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(o), "d"(z[0]), "d"(z[1]),
                                             "d"(z[2]), "d"(z[3])
                                             : "memory");
                            } else {
                                o[0] = z[0];
                                o[p.I] = z[1];
                                o[2 * p.I] = z[2];
                                o[3 * p.I] = z[3];
                            }
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                if (c0 + g * 4 + j < p.cols) {
                                    // (weak sums are not added: settle does that)
                                    if (!p.accumulate) o[p.I * j] = z[j];
                                    else if (er == kZeroRow || !(weak >> (g * 4 + j) & 1)) o[p.I * j] = __dadd_rn(o[p.I * j], z[j]);
                                }
                        }
                    }
                }
                if (!mine || er == kZeroRow) weak = 0;
                // Small by cancellation, or because the terms are?  The digits stand where
                // an entry is big in both fibres, in the slab where the column has its
                // largest (of any concatenated operand).
                uint32_t hold = 0;   // (lane: column) rows left to settle
                uint32_t cols = __reduce_or_sync(0xffffffffu, weak);
                if (cols && !p.accumulate) {
                    const int S = p.slabs, spc = S / p.ncat, s = (wc >> 16) % spc;
                    const uint16_t *const ma = p.mA + ((int64_t)be * p.mtiles + mi) * S * kRowBlock + m;
                    const uint16_t *const mb = p.mB + ((int64_t)be * p.ntiles + ni) * S * nt + cw + lane;
                    for (int t0 = 0; t0 < p.ncat; t0 += 3) {
                        uint32_t b[3];
#pragma unroll
                        for (int t = 0; t < 3; ++t)
                            b[t] = (cols >> lane & 1) && t0 + t < p.ncat ? __ldg(mb + (int64_t)((t0 + t) * spc + s) * nt) : 0u;
                        // (columns that have it in the same slab together)
                        for (uint32_t left = cols; left;) {
                            const int at = __shfl_sync(0xffffffffu, s, __ffs((int)left) - 1);
                            uint32_t same = __ballot_sync(0xffffffffu, s == at) & left, r[3];
                            left &= ~same;
#pragma unroll
                            for (int t = 0; t < 3; ++t) r[t] = t0 + t < p.ncat ? __ldg(ma + (int64_t)((t0 + t) * spc + at) * kRowBlock) : 0u;
                            for (; same; same &= same - 1) {
                                const int j = __ffs((int)same) - 1;
                                uint32_t found = 0;
#pragma unroll
                                for (int t = 0; t < 3; ++t) found |= r[t] & __shfl_sync(0xffffffffu, b[t], j);
                                if (found) weak &= ~(1u << j);
                            }
                        }
                    }
                    cols = __reduce_or_sync(0xffffffffu, weak);
                }
                for (; cols; cols &= cols - 1) {
                    const int j = __ffs((int)cols) - 1;
                    const bool zero = (int16_t)__shfl_sync(0xffffffffu, wc, j) == kZeroRow;
                    const uint32_t rows = __ballot_sync(0xffffffffu, !zero && c0 + j < p.cols && (weak >> j & 1));
                    if (lane == j) hold = rows;
                }
                const uint32_t some = __ballot_sync(0xffffffffu, hold);
                if (some) {
                    int at = lane == 0 ? atomicAdd(a.nleft, __popc(some)) : 0;
                    at = __shfl_sync(0xffffffffu, at, 0) + __popc(some & ((1u << lane) - 1));
                    if (hold) a.left[at] = {(uint16_t)q, (uint16_t)(cw + lane), be, mi, ni * 4 + quarter, hold, wc};
                    __syncwarp();
                }
            }
            if (odd && row_ok) {
                // non-finite entries, or a wait gave up (every later output of this warp)
#pragma unroll 1
                for (int j = 0; j < hc && c0 + j < p.cols; ++j) {
                    const int e = (int16_t)__ldg(p.eB + (int64_t)be * p.ntiles * nt + c0 + j);
                    const double z = er == kNanRow || e == kNanRow ? __longlong_as_double(0x7FF8000000000000LL)
                                                                   : fma_chain(p, be, rg, c0 + j);
                    double *o = out + p.I * j;
                    *o = p.accumulate ? __dadd_rn(*o, z) : z;
                }
            }
        }
    }
    tc_before();
    __syncthreads();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// ---------------------------------------------------------------------------
// The FP64 pipe's own kernel for small products: four lanes per output, each
// with every fourth entry of the contraction, so that even a 64 x 64 product
// spreads over every SM (a 64 x 64 tile would keep one SM's FP64 pipe busy for
// 63 us) and the chain of dependent FMAs is a quarter of the contraction.
// ---------------------------------------------------------------------------
struct FArgs {
    int count;
    int64_t first[kMaxProd + 1];   // output prefix
    GProd p[kMaxProd];
};
constexpr int kLanes = 4;

// IT: 32-bit indices where the launch allows them (its divisions cost as much as
// a short contraction)
template <typename IT>
__global__ void __launch_bounds__(128) k_fma_products(const __grid_constant__ FArgs a)
{
    const IT total = (IT)a.first[a.count];
    const int sub = threadIdx.x % kLanes;
    pdl_trigger();
    pdl_wait();
    // whole warps stay in the loop for the shuffles
    for (IT e0 = ((IT)blockIdx.x * blockDim.x + threadIdx.x) / 32 * (32 / kLanes); e0 < total;
         e0 += (IT)gridDim.x * blockDim.x / kLanes) {
        const IT e = min(e0 + (IT)(threadIdx.x % 32 / kLanes), total - 1);
        int q = 0;
        while (q + 1 < a.count && e >= (IT)a.first[q + 1]) ++q;
        const GProd &p = a.p[q];
        const IT I = (IT)p.I, cols = (IT)p.cols, IB = (IT)p.IB;
        const IT size = (IT)p.rows * cols, entry = (e - (IT)a.first[q]) / size, t = e - (IT)a.first[q] - entry * size;
        // neighbouring lanes: neighbouring outputs in memory
        IT o, x0, i;
        if (I == 1) {
            o = t / cols;
            i = t - o * cols;
            x0 = 0;
        } else {
            o = t / (I * cols);
            const IT w = t - o * (I * cols);
            i = w / I;
            x0 = w - i * I;
        }
        const int64_t xa = (int64_t)entry * p.sA + (int64_t)o * (p.I * p.n) + x0;
        const IT ob = i / IB;
        const int64_t lb = (int64_t)entry * p.sB + (int64_t)ob * (p.IB * p.n) + (i - ob * IB);
        double y = 0.0;
        for (int c = 0; c < p.ncat; ++c) {
            const double *x = p.X[c] + xa, *l = p.L[c] + lb;
            double s = 0.0;
            int k = sub;
            for (; k + 3 * kLanes < p.n; k += 4 * kLanes) {
                double xv[4], lv[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    xv[j] = x[p.I * (k + j * kLanes)];
                    lv[j] = l[p.IB * (k + j * kLanes)];
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) s = fma(xv[j], lv[j], s);
            }
            for (; k < p.n; k += kLanes) s = fma(x[p.I * k], l[p.IB * k], s);
            y = p.sc[c] == 1.0 && c == 0 ? s : fma(p.sc[c], s, y);
        }
#pragma unroll
        for (int w = 1; w < kLanes; w *= 2) y += __shfl_xor_sync(0xffffffffu, y, w);
        if (sub == 0 && e0 + (IT)(threadIdx.x % 32 / kLanes) < total) {
            double *z = p.out + (int64_t)entry * p.sOut + t;
            *z = p.accumulate ? __dadd_rn(*z, y) : y;
        }
    }
}

GProd to_gprod(const Product &s)
{
    GProd p{};
    p.A = s.ia.data;
    p.B = s.ib.data;
    p.eA = s.ia.exps;
    p.eB = s.ib.exps;
    p.mA = s.ia.masks;
    p.mB = s.ib.masks;
    p.cA = s.ia.codes;
    p.cB = s.ib.codes;
    p.out = s.out;
    p.slabs = s.ia.slabs;
    p.nt = s.ib.rb;
    p.cols = (int)s.B.rows;
    p.ntiles = p.nt ? (p.cols + p.nt - 1) / p.nt : 0;
    p.mtiles = (int)((s.A.rows + kRowBlock - 1) / kRowBlock);
    p.sA = s.A.stride;
    p.sB = s.B.stride;
    p.sOut = s.stride;
    p.accumulate = s.accumulate;
    p.ncat = s.A.ncat;
    p.n = s.A.n;
    p.rows = s.A.rows;
    p.r0 = s.A.r0;
    p.I = s.A.I;
    p.IB = s.B.I;
    for (int t = 0; t < s.A.ncat; ++t) {
        p.X[t] = s.A.src[t];
        p.L[t] = s.B.src[t];
        p.sc[t] = s.A.scale[t] * s.B.scale[t];
    }
    return p;
}
}  // namespace

int tile_cols(int64_t rows, int cols, int products, int slabs)
{
    // the width whose waves take the least: clocks per tile of 6 and of 16 slabs over
    // ten and fifty waves (15110 and 26818 at 64 columns, 12645 and 21823 at 48, 9219 and
    // 16247 at 32, 6341 and 12415 at 16), as a share per slab and one per tile
    static const struct {
        int nt, slab, tile;
    } kCost[] = {{64, 1171, 8085}, {48, 918, 7138}, {32, 703, 5002}, {16, 607, 2696}};
    const int64_t mt = (rows + kRowBlock - 1) / kRowBlock * products;
    int best = 16;
    double least = 0.0;
    for (const auto &c : kCost) {
        const int64_t tiles = mt * ((cols + c.nt - 1) / c.nt);
        const double t = (double)((tiles + kSms - 1) / kSms) * ((double)slabs * c.slab + c.tile);
        if (least == 0.0 || t < least) {
            least = t;
            best = c.nt;
        }
    }
    // the same number of tiles, evenly wide
    const int nb = (cols + best - 1) / best;
    return std::min(best, ((cols + nb - 1) / nb + 15) / 16 * 16);
}

bool use_digits(int64_t rows, int n, int count)
{
    // Up to 2^20 points ds_tucker_static gives the same bits as ds_tucker, and its 20 MiB
    // hold the digits of a 1024 x 1024 matrix and of a row block, not of a larger one; so
    // 2048 x 400 runs its long mode on the FP64 pipe, 2990 us (tiled FMA chains before:
    // 5227).  Beyond, 4096, the dense scheme's largest matrix.
    const int most = rows * n > ((int64_t)1 << 20) ? 4096 : 1024;
    // 1.5e6 FMAs take the FP64 pipe about as long as the launches of a digit
    // product take at least (7, 9 + 5 and 3 us); row tiles of 128 that are mostly padding
    // move the line (twelve products of 64 x 64: 9 against 14 us)
    return n >= 12 && n <= most && rows >= 16 && (double)rows * n * n * count > 1.5e6 * std::max(1.0, 160.0 / rows);
}

template <int E>
static void split_as(const View *v, const Image *im, int count, int *reset, cudaStream_t st)
{
    SplitArgs a{};
    a.count = count;
    a.reset = reset;
    bool wide = false;
    int warps = 1;
    for (int q = 0; q < count; ++q) warps = std::max(warps, split_warps(im[q].slabs));
    warps *= std::max(1, 8 / warps);
    for (int q = 0; q < count; ++q) {
        a.v[q] = v[q];
        a.im[q] = im[q];
        const int G = warps / split_warps(im[q].slabs);
        const int64_t groups = (im[q].rows + 2 * E - 1) / (2 * E) * v[q].batch;
        a.first[q + 1] = a.first[q] + (int)((groups + G - 1) / G);
        wide = wide || (v[q].r0 + im[q].rows + 2 * E * 32) * std::max(1, v[q].batch) > INT32_MAX || v[q].I > INT32_MAX;
    }
    const dim3 grid(a.first[count]), block(warps * 32);
    if (wide) pdl_launch(k_digits<int64_t, E>, grid, block, 0, st, a);
    else pdl_launch(k_digits<int, E>, grid, block, 0, st, a);
}

void launch_split(const View *v, const Image *im, int count, int *reset, cudaStream_t st)
{
    // Where eight entries per thread leave half of the SMs' warps empty, four: a
    // chain of dependent work half as long (301 x 150, 150 x 301 and their matrices
    // 8.4 -> 7.0 us; eighteen tensors of 96^3, with warps for all SMs, 45 -> 49 us).
    int64_t threads = 0;
    for (int q = 0; q < count; ++q) threads += im[q].rows * v[q].batch * im[q].slabs * (kSlab / 8);
    if (threads < (int64_t)kSms * 512) split_as<4>(v, im, count, reset, st);
    else split_as<8>(v, im, count, reset, st);
}

int launch_products(const Product *s, int count, uint8_t *left, long long wait_limit, cudaStream_t st)
{
    static std::atomic<uint64_t> ready{0};   // devices whose shared-memory limit is raised
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 64 || !(ready.load() >> dev & 1)) {
        cudaFuncSetAttribute(k_digit_products, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
        if (dev < 64) ready.fetch_or((uint64_t)1 << dev);
    }
    GArgs a{};
    a.count = count;
    a.wait_limit = wait_limit;
    for (int q = 0; q < count; ++q) {
        a.p[q] = to_gprod(s[q]);
        a.first[q + 1] = a.first[q] + a.p[q].mtiles * a.p[q].ntiles * s[q].A.batch;
    }
    const int tiles = a.first[count];
    if (tiles == 0) return 0;
    a.nleft = (int *)left;
    a.left = (Left *)(left + kAlign);
    pdl_launch(k_digit_products, dim3(std::min(tiles, kSms)), dim3(kThreads), kSmem, st, a);
    pdl_launch(k_settle, dim3((int)std::min<int64_t>(kSms * kSettleBlocks, (int64_t)tiles * 64)), dim3(kSettleThreads), 0, st, a);
    return 2;
}

void launch_products_fma(const Product *s, int count, cudaStream_t st)
{
    FArgs a{};
    a.count = count;
    for (int q = 0; q < count; ++q) {
        a.p[q] = to_gprod(s[q]);
        a.first[q + 1] = a.first[q] + a.p[q].rows * a.p[q].cols * s[q].A.batch;
    }
    const int64_t total = a.first[count];
    if (total == 0) return;
    const dim3 grid((int)std::min<int64_t>((total * kLanes + 127) / 128, kSms * 16));
    // (headroom for the stride past the end and the thread index)
    if (total < (int64_t)1 << 28) pdl_launch(k_fma_products<int>, grid, dim3(128), 0, st, a);
    else pdl_launch(k_fma_products<int64_t>, grid, dim3(128), 0, st, a);
}

View tensor_view(int d, const int64_t *n, int mu, const double *X)
{
    View v{};
    v.src[0] = X;
    v.scale[0] = 1.0;
    v.ncat = v.batch = 1;
    v.n = (int)n[mu];
    v.I = v.rows = 1;
    for (int q = 0; q < d; ++q) {
        if (q < mu) v.I *= n[q];
        if (q != mu) v.rows *= n[q];
    }
    return v;
}

View matrix_view(int64_t n, const double *L, int transpose, double scale)
{
    View v{};
    v.src[0] = L;
    v.scale[0] = scale;
    v.ncat = v.batch = 1;
    v.n = (int)n;
    v.I = transpose ? 1 : n;
    v.rows = n;
    return v;
}

size_t scratch_bytes(int64_t N, int64_t n, int count, int cat, bool matrices)
{
    const int slabs = slabs_of((int)n, cat);
    const size_t a = aligned(image_total(N / n, kRowBlock, slabs) + left_bytes(N / n, (int)n, 1));
    // (the padding to whole tiles is below 64 columns)
    const size_t b = matrices ? aligned(image_total(n + 64, 1, slabs)) : 0;
    // beyond 1 GiB a launch fills the GPU many times over: row blocks cost nothing
    const size_t most = (size_t)1 << 30;
    return kAlign + std::min(count * a, std::max(most, 2 * a / (pad_rows(N / n, kRowBlock) / kRowBlock) + kAlign)) + count * b;
}

namespace {
bool same_view(const View &a, const View &b)
{
    if (a.ncat != b.ncat || a.n != b.n || a.I != b.I || a.rows != b.rows || a.r0 != b.r0 || a.batch != b.batch || a.stride != b.stride) return false;
    for (int t = 0; t < a.ncat; ++t)
        if (a.src[t] != b.src[t] || a.scale[t] != b.scale[t]) return false;
    return true;
}
double product_flops(const Product &p) { return 2.0 * p.A.batch * p.A.rows * p.B.rows * p.A.n * p.A.ncat; }
}  // namespace

int run_products(const Context &c, const Product *ps, int count, cudaStream_t st)
{
    int launches = 0;
    for (int i = 0; i < count;) {
        const int many = count * ps[i].A.batch;   // products in a launch
        const bool digits = use_digits(ps[i].A.rows, ps[i].A.n, many);
        Product p[kMaxProd];
        View sv[kMaxProd];
        Image si[kMaxProd];
        int np = 0, ns = 0;
        size_t used = 0, lists = kAlign;   // (from the start of the scratch) images; at its end: left outputs
        double flops = 0.0;
        auto place = [&](const View &v, int rb, Image &im) {   // scratch for v's image; false: no room
            for (int q = 0; q < ns; ++q)
                if (si[q].rb == rb && same_view(sv[q], v)) {
                    im = si[q];
                    return true;
                }
            im.rb = rb;
            im.slabs = slabs_of(v.n, v.ncat);
            im.rows = v.rows;
            const size_t all = image_total(v, rb);
            if (used + lists + all > c.ws_bytes || ns == kMaxProd) return false;
            im.place(c.ws + used, v.batch);
            used += all;
            sv[ns] = v;
            si[ns++] = im;
            return true;
        };
        auto add = [&](const Product &q, bool with_b) {
            Product t = q;
            const size_t u0 = used, l0 = lists;
            const int n0 = ns;
            lists += left_bytes(t.A.rows, (int)t.B.rows, t.A.batch);
            if (used + lists > c.ws_bytes || (with_b && !place(t.B, tile_cols(t.A.rows, (int)t.B.rows, many, slabs_of(t.A.n, t.A.ncat)), t.ib)) ||
                !place(t.A, kRowBlock, t.ia)) {
                used = u0;
                lists = l0;
                ns = n0;
                return false;
            }
            p[np++] = t;
            flops += product_flops(t);
            return true;
        };
        auto flush = [&] {
            if (ns) {
                if (c.prof) c.prof->begin(st, 1, 0.0);
                launch_split(sv, si, ns, (int *)(c.ws + (c.ws_bytes - lists) / kAlign * kAlign), st);
                if (c.prof) c.prof->end(st);
                ++launches;
            }
            if (c.prof) c.prof->begin(st, 1, flops);
            launches += launch_products(p, np, c.ws + (c.ws_bytes - lists) / kAlign * kAlign, c.wait_limit, st);
            if (c.prof) c.prof->end(st);
        };
        int j = i;
        if (digits)
            while (j < count && np < kMaxProd && add(ps[j], ps[j].ib.data == nullptr)) ++j;
        if (j > i) {
            flush();
            i = j;
            continue;
        }
        // one product whose images do not fit together: B's once (where it is cut
        // per call), A's in row blocks
        bool done = false;
        if (digits && ps[i].A.batch == 1) {
            Product t = ps[i];
            const size_t per = image_total(kRowBlock, kRowBlock, slabs_of(t.A.n, t.A.ncat)) + left_bytes(kRowBlock, (int)t.B.rows, 1);
            const bool ok = t.ib.data || place(t.B, tile_cols(t.A.rows, (int)t.B.rows, 1, slabs_of(t.A.n, t.A.ncat)), t.ib);
            if (ok && used + per + 2 * kAlign <= c.ws_bytes) {
                const int64_t fit = (int64_t)((c.ws_bytes - used - 2 * kAlign) / per) * kRowBlock;
                const size_t u0 = used;
                for (int64_t r = 0; r < ps[i].A.rows; r += fit) {
                    Product part = t;
                    part.A.r0 = t.A.r0 + r;
                    part.A.rows = std::min(fit, t.A.rows - r);
                    if (r) ns = 0;   // B's image stays
                    used = u0;
                    lists = kAlign;
                    np = 0;
                    flops = 0.0;
                    add(part, false);
                    flush();
                }
                done = true;
            }
        }
        if (!done) {
            // the FP64 pipe: every remaining product of a small phase in one launch
            np = 0;
            flops = 0.0;
            const int most = digits ? 1 : kMaxProd;
            for (j = i; j < count && np < most; ++j) {
                p[np++] = ps[j];
                flops += product_flops(ps[j]);
            }
            if (c.prof) c.prof->begin(st, 1, flops);
            launch_products_fma(p, np, st);
            if (c.prof) c.prof->end(st);
            ++launches;
        } else
            j = i + 1;
        i = j;
    }
    return launches;
}

void tucker_f64(const Context &c, int d, const int64_t *n, const double *X, double *Y, const double *const *L,
                int transpose, double *tmp, cudaStream_t st)
{
    int64_t N = 1;
    for (int q = 0; q < d; ++q) N *= n[q];
    const double *in = X;
    for (int mu = 0; mu < d; ++mu) {
        Product p{};
        p.A = tensor_view(d, n, mu, in);
        p.B = matrix_view(n[mu], L[mu], transpose);
        p.out = mu == d - 1 ? Y : tmp + (mu % 2) * N;
        run_products(c, &p, 1, st);
        in = p.out;
    }
}

long long wait_limit_default()
{
    const char *e = getenv("DS_WAIT_LIMIT_CYCLES");
    const long long v = e ? atoll(e) : 0;
    return v > 0 ? v : kWaitCycles;
}

}  // namespace mm
}  // namespace ds
