// FP32 Linear layers on the tensor cores, for the FP32 path's MLPs.
//
// An FP32 number has 24 significant bits, so it is exactly the sum of three
// BF16 numbers of 8 bits each: hi = x rounded to BF16, mid = x - hi rounded,
// lo = the rest (both differences are exact; numbers are scaled first, see kUp,
// so that this holds for the smallest ones, and from 2^104 on and for infinities
// FP32 FMAs take over). A product x w is then the sum of
// nine BF16 products, each exact in FP32; the six largest are accumulated in
// FP32 by tcgen05.mma and the three left out (mid lo, lo mid, lo lo) are below
// 2^-25 |x w|, of either sign. (Splitting by clearing bits costs the same but
// makes every piece agree in sign with x: the parts left out then add up.)
// The tensor core truncates its running sums, so a sum must not carry terms far below it: a Linear's hi hi
// products have an accumulator of their own up to width 64 (above, and in weight gradients of 65 to 128
// inputs, the small products come first in a common one), the epilogue adds the accumulators up in FP32 and
// gives back what truncation takes in the mean (kTruncation). Sums in tensor memory run over at most 256
// products per output (inputs) or one tile of rows (weight gradients, continued in FP32 registers, rounding
// to nearest).
//
// What bounds it: at width 64 a Linear moves 512 bytes per row for 49 kFLOP of
// BF16 products, 96 FLOP per byte, far below the ridge: HBM, if the splitting
// (about 6 instructions per element) and the epilogue are hidden. So the block
// is specialised: four warps load FP32 rows, split them and write the three
// operand tiles (swizzled K-major rows); one warp issues the MMAs; two
// groups of four warps take alternate tiles from two sets of tensor-memory
// accumulators, through a per-warp staging tile so that every global access of
// an epilogue (bias, residual, gathers, stores) is a run of whole 64-byte
// pieces of rows. A Linear with ELU of 1.34M rows at width 64 takes 0.16 ms,
// 4.3 TB/s (HBM alone: 0.10). A third epilogue group (16 warps, each group
// issuing its own MMAs) gave the same there and cost the narrow widths 12 %.

#include <algorithm>

#include "device_common.cuh"
#include "fused_common.cuh"
#include "lin3.h"
#include "profiler.h"

namespace gnn {
namespace lin3 {

using namespace tc;
using fused::align_up;
using fused::aligned_smem;
using fused::desc_step;
using fused::kmajor_off;
using fused::span_of;

cudaError_t take_device_error(unsigned int* out) { return take_device_error_word(out); }

namespace {

// k_lin3: 4 producer warps, 8 epilogue warps, one MMA warp: 13 warps leave each
// thread 128 registers (at 17 it is 96), which the epilogue's operands need.
// k_wgrad3: two operands to split and little to do at the end, 8 + 8 + 1 warps.
constexpr int kProducers = 128, kEpilogue = 256;
constexpr int kThreads = kProducers + kEpilogue + 32;
constexpr int kProducerWarps = kProducers / 32, kEpilogueWarps = kEpilogue / 32;
constexpr int kSide = 128;   // k_wgrad3: producer threads of one operand
constexpr int kWThreads = 2 * kSide + kEpilogue + 32;
constexpr int kWProducerWarps = 2 * kSide / 32;
constexpr int kStageLd = 20;                      // floats per row of a 32 x 16 staging tile: 16-byte rows, no conflicts
constexpr uint32_t kStageBytes = 32 * kStageLd * 4;
constexpr uint32_t kSmemMax = 227 * 1024;

__host__ __device__ inline int pad16(int n) { return (n + 15) / 16 * 16; }
__host__ __device__ inline int pow2_width(int n) { return n <= 16 ? 16 : (n <= 32 ? 32 : (n <= 64 ? 64 : 128)); }
__host__ __device__ inline uint32_t pow2_cols(uint32_t n) {
    uint32_t c = 32;
    while (c < n) c <<= 1;
    return c;
}

// ------------------------------------------------------------------ device helpers

// The ends of the range. Streamed operands are split at 2^24 of their size, so that the last bit of the
// smallest FP32 number is a normal BF16 number, and weights at 2^-24, which leaves a Linear's sums as they
// are; a weight gradient's two streamed operands leave 2^48, taken off where its tiles are added. No bit of
// a sum in the middle of the range changes by it.
//
// The other end cannot be split. From 2^104 on, and for infinities, hi is infinite, and every sum that the
// number is in is a NaN: all columns of its row. So the epilogue looks at one column of each row (LayerNorm:
// at the mean), and a tile in which that is not finite is begun again after a function out of line has
// replaced the sums that are not finite by FP32 FMAs. Weights are looked at when they are split, eight
// at a time: one above 2^16 (below, a sum that overflows has a number above 2^104 in it), or eight
// below 2^-80, whose pieces lose bits and one of which is made a NaN, send every tile of the block there. A
// weight gradient's sums are looked at when the block is done. A training step at width 64 takes 9.58 -> 9.69 ms
// with it, a 4-cube forward 77.5 -> 81.4 us (checking all sums in the epilogue, or the numbers in the
// producers, cost 9 and 4 % more of the step).
constexpr float kUp = 16777216.f, kDown = 1.f / 16777216.f, kUnscale = kDown * kDown;
constexpr float kBigWeight = 65536.f;                     // 2^16
constexpr float kTinyWeights = 8.271806125530277e-25f;    // 2^-80

__device__ __forceinline__ bool finite(float v) { return fabsf(v) <= 3.402823466e38f; }

// Eight FP32 values times 2^24 (DOWN: 2^-24) as three BF16 octets whose sum they are.
template <bool DOWN = false>
__device__ __forceinline__ void split8(const float* v, uint4& hi, uint4& mid, uint4& lo) {
    uint32_t h[4], m[4], l[4];
    constexpr float kS = DOWN ? kDown : kUp;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 t = __fmul2_rn(make_float2(v[2 * i], v[2 * i + 1]), make_float2(kS, kS));
        float a = t.x, b = t.y, x, y;
        h[i] = pack_bf16x2(a, b);
        unpack_bf16x2(h[i], x, y);
        a -= x;
        b -= y;
        m[i] = pack_bf16x2(a, b);
        unpack_bf16x2(m[i], x, y);
        l[i] = pack_bf16x2(a - x, b - y);
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    mid = make_uint4(m[0], m[1], m[2], m[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// Eight weights of a row: true if they are special.
__device__ __forceinline__ bool check_weights(float* v) {
    const float m = fmaxf(fmaxf(fmaxf(fabsf(v[0]), fabsf(v[1])), fmaxf(fabsf(v[2]), fabsf(v[3]))),
                          fmaxf(fmaxf(fabsf(v[4]), fabsf(v[5])), fmaxf(fabsf(v[6]), fabsf(v[7]))));
    const bool tiny = m > 0.f && m < kTinyWeights;
    if (tiny) v[0] = __uint_as_float(0x7fffffffu);
    return tiny || !(m <= kBigWeight);
}

// Up to n (may be <= 0) of the 8 values at p, the rest zero. VEC: p is 16-byte
// aligned and n is a multiple of 4.
template <bool VEC>
__device__ __forceinline__ void load8(const float* p, int n, float* v) {
    if constexpr (VEC) {
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 a = n > 0 ? __ldg(reinterpret_cast<const float4*>(p)) : z;
        const float4 b = n > 4 ? __ldg(reinterpret_cast<const float4*>(p) + 1) : z;
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = i < n ? __ldg(p + i) : 0.f;
    }
}

// Four values of a row, of which n exist (VEC: all four or none). The loads are
// plain ones: an epilogue may read the buffer it writes (same lane, same address).
template <bool VEC>
__device__ __forceinline__ float4 load4(const float* p, int n) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (VEC) {
        if (n > 0) v = *reinterpret_cast<const float4*>(p);
    } else {
        if (n > 0) v.x = p[0];
        if (n > 1) v.y = p[1];
        if (n > 2) v.z = p[2];
        if (n > 3) v.w = p[3];
    }
    return v;
}
template <bool VEC>
__device__ __forceinline__ void store4(float* p, int n, float4 v) {
    if constexpr (VEC) {
        if (n > 0) *reinterpret_cast<float4*>(p) = v;
    } else {
        if (n > 0) p[0] = v.x;
        if (n > 1) p[1] = v.y;
        if (n > 2) p[2] = v.z;
        if (n > 3) p[3] = v.w;
    }
}
__device__ __forceinline__ float4 add4(float4 a, float4 b) {
    const float2 l = __fadd2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
    const float2 h = __fadd2_rn(make_float2(a.z, a.w), make_float2(b.z, b.w));
    return make_float4(l.x, l.y, h.x, h.y);
}

template <int V>
struct Int {
    static constexpr int value = V;
};

// One lane of the warp waits, the warp agrees (and is converged afterwards).
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, int lane) {
    int ok = 1;
    if (lane == 0) ok = mbar_wait(bar, parity) ? 1 : 0;
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

// 16 values into 16 consecutive TMEM columns of this thread's lane.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float* v) {
    uint32_t r[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) r[i] = __float_as_uint(v[i]);
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

// Accumulators of a row tile, NP columns each: what they hold, in the order in which they lie.
enum Acc {
    kAccAll,     // all six products
    kAccHalves,  // all six products of the first | of the second half of the steps
    kAccSmall,   // hi hi | the five small products
    kAccThree    // hi hi | 2^-8 terms | 2^-16 terms
};
__host__ __device__ constexpr int acc_count(Acc acc) { return acc == kAccAll ? 1 : (acc == kAccThree ? 3 : 2); }

// 16 columns of the lane's row: the accumulators' sum, with gain times the large products given back.
template <Acc ACC>
__device__ __forceinline__ void load_acc16(uint32_t taddr, int NP, float gain, float* v) {
    float u[16], w[16];
    tmem_ld16(taddr, v);
    if constexpr (ACC != kAccAll) tmem_ld16(taddr + NP, u);
    if constexpr (ACC == kAccThree) tmem_ld16(taddr + 2 * NP, w);
    tmem_ld_wait();
    const float2 g = make_float2(gain, gain);
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
        const float2 a = make_float2(v[i], v[i + 1]);
        float2 b = make_float2(u[i], u[i + 1]);
        if constexpr (ACC == kAccThree) b = __fadd2_rn(b, make_float2(w[i], w[i + 1]));
        const float2 r = ACC == kAccAll ? __fmul2_rn(g, a) : __ffma2_rn(g, ACC == kAccHalves ? __fadd2_rn(a, b) : a, b);
        const float2 z = __fadd2_rn(a, r);
        v[i] = z.x;
        v[i + 1] = z.y;
    }
}
__device__ __forceinline__ void load_sum16(uint32_t taddr, int NP, Acc acc, float gain, float* v) {
    if (acc == kAccThree) load_acc16<kAccThree>(taddr, NP, gain, v);
    else if (acc == kAccHalves) load_acc16<kAccHalves>(taddr, NP, gain, v);
    else load_acc16<kAccAll>(taddr, NP, gain, v);
}

// Sums that are not finite, by FP32 FMAs from global memory, in order.
struct LinSum {   // of a row of a Linear
    const Args& A;
    int64_t row;
    __device__ float operator()(int n) const {
        const int64_t off = n >= A.nsplit ? A.noff + (int64_t)(n - A.nsplit) * A.sn : (int64_t)n * A.sn;
        float t = 0.f;
        for (int s = 0; s < 2 && n < A.N; ++s) {
#pragma unroll 8
            for (int k = 0; k < A.K[s]; ++k) t = fmaf(A.A[s][row * A.lda[s] + k], A.W[s][off + k * A.sk], t);
        }
        return t;
    }
};
struct RowSum {   // sum over j < n of a[j] b[j ld + i], zero for i >= ld
    const float* a;
    const float* b;
    int n, ld;
    __device__ float operator()(int i) const {
        float t = 0.f;
        if (i >= ld) return t;
#pragma unroll 8
        for (int j = 0; j < n; ++j) t = fmaf(a[j], b[(int64_t)j * ld + i], t);
        return t;
    }
};

// The accumulators (NP columns of the warp's rows) with every sum that is not finite replaced.
template <class F>
__device__ __noinline__ void patch_sums(const F& exact, bool mine, uint32_t taddr, int NP, Acc acc, float gain) {
    for (int c0 = 0; c0 < NP; c0 += 16) {
        float v[16], w[16];
        uint32_t bad = 0;
        load_sum16(taddr + c0, NP, acc, gain, v);
#pragma unroll
        for (int i = 0; i < 16; ++i) bad |= (mine && !finite(v[i])) ? 1u << i : 0u;
        if (!__any_sync(0xffffffffu, bad != 0)) continue;
        for (int i = 0; i < 16; ++i) {
            const float t = (bad >> i) & 1u ? exact(c0 + i) : 0.f;
            w[i] = finite(t) ? fmaf(-gain, t, t) : t;   // (the gain is given back when it is read)
        }
        __syncwarp();
        for (int a = 0; a < acc_count(acc); ++a) {
            tmem_ld16(taddr + (uint32_t)(a * NP + c0), v);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if ((bad >> i) & 1u) v[i] = a == 0 ? w[i] : 0.f;
            tmem_st16(taddr + (uint32_t)(a * NP + c0), v);
        }
        tmem_st_wait();
    }
}
// sum over the block's row tiles (RT rows each) of G[r ldg] X[r ldx]
__device__ __noinline__ float dw_sum(const float* G, int64_t ldg, const float* X, int64_t ldx, int64_t rows, int n_tiles,
                                     int RT) {
    float s = 0.f;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        const int64_t r1 = std::min<int64_t>(rows, (int64_t)(t + 1) * RT);
        float a = 0.f;
#pragma unroll 8
        for (int64_t r = (int64_t)t * RT; r < r1; ++r) a = fmaf(G[r * ldg], X[r * ldx], a);
        s += a;
    }
    return s;
}

// ELU (alpha 1) of two values: z above zero, e^z - 1 at and below it, by the
// usual two steps: Cody and Waite's reduction z = n ln 2 + r, |r| <= ln 2 / 2
// (ln 2 in two parts, n by adding and subtracting 1.5 * 2^23), and Taylor's
// series of e^r - 1 up to r^8 (the rest is below 6e-10 r); then
// e^z - 1 = 2^n (e^r - 1) + (2^n - 1), exact in its last term for n >= -24. On
// the packed FP32 pipe it is 12 instructions per value where a call of expm1f
// is about 40. Below -87 it is -1; a NaN stays one (the select is on z <= 0).
__device__ __forceinline__ float2 elu_pair(float2 z) {
    const float2 c = make_float2(fmaxf(z.x, -87.f), fmaxf(z.y, -87.f));
    auto both = [](float v) { return make_float2(v, v); };
    const float2 t = __ffma2_rn(c, both(1.4426950408889634f), both(12582912.f));
    const float2 n = __fadd2_rn(t, both(-12582912.f));
    float2 r = __ffma2_rn(n, both(-0.693145751953125f), c);
    r = __ffma2_rn(n, both(-1.4286068203094172e-6f), r);
    float2 q = __ffma2_rn(r, both(1.f / 40320.f), both(1.f / 5040.f));
    q = __ffma2_rn(q, r, both(1.f / 720.f));
    q = __ffma2_rn(q, r, both(1.f / 120.f));
    q = __ffma2_rn(q, r, both(1.f / 24.f));
    q = __ffma2_rn(q, r, both(1.f / 6.f));
    q = __ffma2_rn(q, r, both(0.5f));
    q = __ffma2_rn(__fmul2_rn(q, r), r, r);
    const float2 p2 = make_float2(__uint_as_float((__float_as_uint(t.x) << 23) + 0x3f800000u),
                                  __uint_as_float((__float_as_uint(t.y) << 23) + 0x3f800000u));
    const float2 e = __ffma2_rn(p2, q, __fadd2_rn(p2, both(-1.f)));
    return make_float2(z.x <= 0.f ? e.x : z.x, z.y <= 0.f ? e.y : z.y);
}

// The six products of a split pair, smallest first: (term of A, term of B).
__device__ constexpr int kTermA[6] = {2, 0, 1, 1, 0, 0};
__device__ constexpr int kTermB[6] = {0, 2, 1, 0, 1, 0};

// An MMA of 128 x 64 x 16 needs 32 cycles of the tensor core, but one follows the other at 110
// whatever its width when one lane of a diverged warp issues them, and at 85 when the whole warp
// goes through the loop and one lane acts. So the warp stays together, and the terms of B lie one
// after the other as rows of one tile: up to width 80 three MMAs do the six products, hi of A with
// [hi | mid | lo] of B, mid with [hi | mid], lo with [hi], into three sums [hi hi | 2^-8 terms |
// 2^-16 terms]. Per row tile at width 64: 1,650 cycles where the 24 narrow ones took 2,630. For a
// weight gradient the terms of X are consecutive blocks of one MN-major operand, up to width 64
// (1.0 -> 0.83 of the time at 64).
//
// Every step (16 of the contraction) cuts the running sum toward zero. Measured against 64 bits, 16 to 128
// products: with normal or ELU operands a sum of n steps loses (n + 1) / 2 times 1.6e-8 to 1.9e-8 of its value
// (up to 3.4e-8 where magnitudes are spread, nothing where all are alike). For one Linear that is below
// FP32's rounding, but every row and layer loses in the same direction: on a network of width 64 (128) the
// parameter gradients were 1.7 (3.5) times as far from 64 bits as with FP32 FMAs. So the epilogue of a Linear
// gives the mean back (kTruncation: at most 4.5e-8 of a sum, below a unit in the last place), and above
// width 64 the steps are halved between two accumulators. Networks of widths 8 to 128 against 64 bits, the
// gradients' largest error over the FMAs': 0.57, their geometric mean 0.80. Weight gradients stay as
// summed: their tiles are added in FP32, and their errors were below the FMAs' already.
constexpr float kTruncation = 1.8e-8f;
__host__ __device__ constexpr float gain_of(int steps) { return kTruncation * 0.5f * (float)(steps + 1); }

// Two tiles' accumulators fit 512 columns. Up to width 64 three wide sums. Above, two of all six products
// (smallest first): with two blocks a block each. With more blocks (two sources, up to width 80), where a
// block's small products would follow another's large ones, three sums again. (Halves beside the small sums
// up to width 64 too: errors 2 to 5 % smaller, a training step 2 %, a small call 6 % slower; not kept.)
__host__ __device__ inline Acc acc_of(int NP, int KB, int nkb) {
    if (NP <= 64 || nkb > 2) return kAccThree;
    return nkb * KB > 16 ? kAccHalves : kAccAll;
}

// ------------------------------------------------------------------ shared memory

struct Smem {
    uint32_t w, a, stg, sums, par, bar, tm, total;
    uint32_t wterm, aterm;
};

// W: nkb blocks x 3 terms of [NP x KB]; a: stages x 3 terms of [128 x KB].
__host__ __device__ inline Smem lin_smem(int NP, int KB, int nkb, int stages) {
    Smem s;
    s.wterm = (uint32_t)NP * KB * 2;
    s.aterm = 128u * KB * 2;
    s.w = 0;
    s.a = align_up((uint32_t)nkb * 3 * s.wterm, 1024);
    s.stg = s.a + (uint32_t)stages * 3 * s.aterm;
    s.sums = s.stg + kEpilogueWarps * kStageBytes;           // [8 warps][2 NP]
    s.par = s.sums + kEpilogueWarps * 2 * (uint32_t)NP * 4;  // bias, gamma, beta
    s.bar = align_up(s.par + 3 * (uint32_t)NP * 4, 8);       // full[4], empty[4], acc_full[2], acc_empty[2]
    s.tm = s.bar + 12 * 8;
    s.total = s.tm + 16 + 1024;
    return s;
}

// ------------------------------------------------------------------ k_lin3

// Producer warps: load FP32 rows (every block of W columns of every source),
// split them, write the three operand tiles of a stage.
template <int W, bool VEC, int MODE>
__device__ __forceinline__ void lin_producer(const Args& A, const Smem& P, uint8_t* sm, uint64_t* full,
                                             uint64_t* empty, int tid, int lane) {
    constexpr int U = W / 8, RS = kProducers / U, IT = 128 / RS;   // pieces of 8 columns per row; rows per step; steps
    constexpr int B = IT < 8 ? IT : 8;                             // pieces in flight per thread
    constexpr int S = span_of(W);
    static_assert((RS * S) % 1024 == 0, "the swizzle repeats every RS rows");
    const int c = (tid % U) * 8, row0 = tid / U;
    const uint32_t off0 = tile_off(row0, c, 128, S);
    const int stages = A.stages, nkb = A.nkb[0] + A.nkb[1];
    int st = 0, use = 0;
    for (int t = blockIdx.x; t < A.n_tiles; t += gridDim.x) {
        if (VEC && tid == 0 && t + (int)gridDim.x < A.n_tiles) {   // the next tile's rows into L2
            const int64_t rn = (int64_t)(t + (int)gridDim.x) * 128;
            const int64_t nr = std::min<int64_t>(128, A.rows - rn);
            for (int s = 0; s < 2; ++s)
                if (A.K[s] && A.lda[s] == A.K[s]) prefetch_l2(A.A[s] + rn * A.lda[s], (uint32_t)(nr * A.K[s] * 4));
            if (A.add && A.ldadd == A.N) prefetch_l2(A.add + rn * A.N, (uint32_t)(nr * A.N * 4));
            if ((MODE == kLnAdjoint || MODE == kAdd) && A.g0) prefetch_l2(A.g0 + rn * A.N, (uint32_t)(nr * A.N * 4));
        }
        const int left = (int)std::min<int64_t>(128, A.rows - (int64_t)t * 128);
        for (int b = 0; b < nkb; ++b) {
            const int s = b < A.nkb[0] ? 0 : 1;
            const int kc = (b - (s ? A.nkb[0] : 0)) * W + c;
            const int nk = A.K[s] - kc;
            const float* src = A.A[s] + ((int64_t)t * 128 + row0) * A.lda[s] + kc;
            const int64_t step = RS * A.lda[s];
            uint8_t* dst = sm + P.a + (uint32_t)st * 3 * P.aterm + off0;
            const bool whole = left == 128 && A.K[s] % W == 0;
#pragma unroll
            for (int i0 = 0; i0 < IT; i0 += B) {
                float v[B][8];
                if (whole) {
#pragma unroll
                    for (int i = 0; i < B; ++i) load8<VEC>(src + (i0 + i) * step, 8, v[i]);
                } else {
#pragma unroll
                    for (int i = 0; i < B; ++i)
                        load8<VEC>(src + (i0 + i) * step, row0 + (i0 + i) * RS < left ? nk : 0, v[i]);
                }
                if (i0 == 0 && use > 0 && !warp_wait(empty + st, (uint32_t)(use - 1) & 1u, lane)) return;
#pragma unroll
                for (int i = 0; i < B; ++i) {
                    uint4 h, m, l;
                    split8(v[i], h, m, l);
                    uint8_t* q = dst + (i0 + i) * RS * S;
                    *reinterpret_cast<uint4*>(q) = h;
                    *reinterpret_cast<uint4*>(q + 128 * S) = m;
                    *reinterpret_cast<uint4*>(q + 2 * 128 * S) = l;
                }
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(full + st);
            if (++st == stages) {
                st = 0;
                ++use;
            }
        }
    }
}

// OPS: what an epilogue adds or needs of other rows: nothing, one row (add), or gathered rows
// (P, Q of kElu; da, w of kLnAdjoint and kAdd).
enum Ops { kOpsNone = 0, kOpsRow, kOpsGather };

template <int MODE, int OPS, bool VEC>
__global__ void __launch_bounds__(kThreads, 1) k_lin3(const __grid_constant__ Args A) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = aligned_smem(smem_raw);
    const int NP = A.NP, KB = A.KB, S = span_of(KB), stages = A.stages, nkb = A.nkb[0] + A.nkb[1], N = A.N;
    const Smem P = lin_smem(NP, KB, nkb, stages);
    float* sPar = reinterpret_cast<float*>(sm + P.par);
    uint64_t* full = reinterpret_cast<uint64_t*>(sm + P.bar);
    uint64_t* empty = full + 4;
    uint64_t* acc_full = full + 8;
    uint64_t* acc_empty = full + 10;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + P.tm);
    const Acc acc = acc_of(NP, KB, nkb);
    const int ACC = acc_count(acc) * NP;                        // columns of a tile's accumulators
    const uint32_t NCOLS = pow2_cols(2 * (uint32_t)ACC);        // two tiles
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == 0) {
        tmem_alloc(tslot, NCOLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < stages; ++i) {
            mbar_init(full + i, kProducerWarps);
            mbar_init(empty + i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(acc_full + i, 1);
            mbar_init(acc_empty + i, 4);
        }
        fence_mbar_init();
    }
    bool special_w = false;
    {   // the weights, split, for the block's lifetime
        const int upr = KB / 8, per = NP * upr;
        for (int i = tid; i < nkb * per; i += kThreads) {
            const int b = i / per, n = (i - b * per) / upr, k8 = (i % upr) * 8;
            const int s = b < A.nkb[0] ? 0 : 1;
            const int k0 = (b - (s ? A.nkb[0] : 0)) * KB + k8;
            const bool second = n >= A.nsplit;
            const float* w = A.W[s] + (second ? A.noff + (int64_t)(n - A.nsplit) * A.sn : (int64_t)n * A.sn);
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = (n < N && k0 + j < A.K[s]) ? __ldg(w + (k0 + j) * A.sk) : 0.f;
            special_w |= check_weights(v);
            uint4 t[3];
            split8<true>(v, t[0], t[1], t[2]);
            const uint32_t off = tile_off(n, k8, NP, S);
#pragma unroll
            for (int j = 0; j < 3; ++j) *reinterpret_cast<uint4*>(sm + P.w + (b * 3 + j) * P.wterm + off) = t[j];
        }
        for (int i = tid; i < NP; i += kThreads) {
            sPar[i] = (A.bias && i < N) ? A.bias[i] : 0.f;
            if (MODE == kLayerNorm || MODE == kLnAdjoint) {
                sPar[NP + i] = i < N ? A.gamma[i] : 0.f;
                sPar[2 * NP + i] = i < N ? A.beta[i] : 0.f;
            }
        }
        if (MODE == kLnAdjoint) {
            float* z = reinterpret_cast<float*>(sm + P.sums);
            for (int i = tid; i < kEpilogueWarps * 2 * NP; i += kThreads) z[i] = 0.f;
        }
    }
    fence_proxy_async();
    tc_fence_before();
    const float spoil = __syncthreads_or(special_w) ? __uint_as_float(0x7fffffffu) : 0.f;   // not finite if special
    tc_fence_after();
    const uint32_t tmem = *tslot;

    if (warp < kProducerWarps) {
        if (KB == 64) lin_producer<64, VEC, MODE>(A, P, sm, full, empty, tid, lane);
        else if (KB == 32) lin_producer<32, VEC, MODE>(A, P, sm, full, empty, tid, lane);
        else lin_producer<16, VEC, MODE>(A, P, sm, full, empty, tid, lane);
    } else if (warp == kProducerWarps + kEpilogueWarps) {
        // ---- one lane of a converged warp issues the MMAs
        {
            const uint32_t lead = elect_one();
            const uint32_t id = idesc_bf16(128, NP), id2 = idesc_bf16(128, 2 * NP), id3 = idesc_bf16(128, 3 * NP);
            const uint64_t a0 = kmajor_desc(smem_u32(sm + P.a), 128, S, 0);
            const uint64_t w0 = kmajor_desc(smem_u32(sm + P.w), NP, S, 0);
            int n = 0, j = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < A.n_tiles && ok; t += gridDim.x, ++j) {
                const int buf = j & 1;
                const uint32_t d = tmem + (uint32_t)(buf * ACC);
                if (j >= 2) ok = mbar_wait(acc_empty + buf, (uint32_t)((j >> 1) - 1) & 1u);
                for (int b = 0; b < nkb && ok; ++b, ++n) {
                    const int st = n % stages, use = n / stages;
                    ok = mbar_wait(full + st, (uint32_t)use & 1u);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t ao = (uint32_t)st * 3 * P.aterm, wo = (uint32_t)b * 3 * P.wterm;
                    auto issue = [&](auto kb) {
                        constexpr int NS = decltype(kb)::value / 16;   // steps: one swizzle block, 32 bytes each
                        const int half = nkb * NS / 2, s0 = b * NS;    // of the tile's steps; this block's first
                        if (acc == kAccThree) {
                            const uint64_t wp = desc_step(w0, wo);
#pragma unroll
                            for (int p = 0; p < 3; ++p) {
                                const uint64_t ap = desc_step(a0, ao + p * P.aterm);
#pragma unroll
                                for (int k = 0; k < NS; ++k)
                                    mma_bf16_warp(lead, d + p * NP, desc_step(ap, k * 32), desc_step(wp, k * 32),
                                                  p == 0 ? id3 : (p == 1 ? id2 : id), (s0 + k > 0 || p > 0) ? 1u : 0u);
                            }
                            return;
                        }
#pragma unroll
                        for (int p = 0; p < 6; ++p) {
                            const uint64_t ap = desc_step(a0, ao + kTermA[p] * P.aterm);
                            const uint64_t wp = desc_step(w0, wo + kTermB[p] * P.wterm);
#pragma unroll
                            for (int k = 0; k < NS; ++k) {
                                const bool second = acc == kAccHalves && s0 + k >= half;
                                mma_bf16_warp(lead, second ? d + NP : d, desc_step(ap, k * 32), desc_step(wp, k * 32), id,
                                              (p > 0 || s0 + k > (second ? half : 0)) ? 1u : 0u);
                            }
                        }
                    };
                    if (KB == 64) issue(Int<64>());
                    else if (KB == 32) issue(Int<32>());
                    else issue(Int<16>());
                    mma_commit_warp(lead, empty + st);
                }
                if (ok) mma_commit_warp(lead, acc_full + buf);
            }
            // the last stage's release has arrived before the block may end
            if (ok && n > 0) mbar_wait(empty + (n - 1) % stages, (uint32_t)((n - 1) / stages) & 1u);
        }
        __syncwarp();
    } else {
        // ---- epilogue: group eg takes the tiles of accumulator eg. A warp has 32 rows; it reads
        // the accumulator by rows (lane = row) and everything else by pieces of 8 rows x 16 columns
        const int ew = warp - kProducerWarps, eg = ew >> 2, q = ew & 3;
        float* stg = reinterpret_cast<float*>(sm + P.stg + ew * kStageBytes);
        float* sums = reinterpret_cast<float*>(sm + P.sums) + ew * 2 * NP;
        const uint32_t tacc = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(eg * ACC);
        const int rs = lane >> 2, c4 = (lane & 3) * 4;
        const int steps = (A.K[0] + 15) / 16 + (A.K[1] + 15) / 16;
        const float gain = gain_of(acc == kAccHalves ? (steps + 1) / 2 : steps);
        constexpr bool kGather = MODE == kElu && OPS == kOpsGather, kEdge = MODE != kElu && OPS == kOpsGather;
        bool ok = true;
        int j = 0, t = blockIdx.x;
        // a tile that turns out to be special (nothing of it has been written by then) is patched and begun again
        bool patched = false;
        auto next = [&] {
            t += gridDim.x;
            ++j;
            patched = false;
        };
        while (t < A.n_tiles && ok) {
            if ((j & 1) != eg) {
                next();
                continue;
            }
            const int64_t rb = (int64_t)t * 128 + 32 * q;
            const int nv = (int)std::min<int64_t>(32, std::max<int64_t>(0, A.rows - rb));
            // this lane's rows (clamped to the last one: loads need no test, stores have it) and their
            // receivers, senders and weights
            int64_t row[4];
            int rv[4] = {0, 0, 0, 0}, sv[4] = {0, 0, 0, 0};
            float wv[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                row[i] = nv > 0 ? rb + std::min(8 * i + rs, nv - 1) : 0;
                if (kGather || kEdge) rv[i] = A.recv[row[i]];
                if (kGather) sv[i] = A.snd[row[i]];
                if (kEdge) wv[i] = A.w[row[i]];
            }
            // the upstream gradient of one piece of the four rows, g0 or g0 + w da[recv]. It is formed wherever
            // it is needed: a buffer for it would be the caller's gradient output, which may be one of the inputs
            auto load_g = [&](int c0, float4* g) {
                const int nc = N - (c0 + c4), col = VEC ? std::min(c0 + c4, N - 4) : c0 + c4;
#pragma unroll
                for (int i = 0; i < 4; ++i) g[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (A.g0) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) g[i] = load4<VEC>(A.g0 + row[i] * N + col, VEC ? 4 : nc);
                }
                if constexpr (kEdge) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 d = load4<VEC>(A.da + (int64_t)rv[i] * N + col, VEC ? 4 : nc);
                        g[i] = make_float4(fmaf(wv[i], d.x, g[i].x), fmaf(wv[i], d.y, g[i].y), fmaf(wv[i], d.z, g[i].z),
                                           fmaf(wv[i], d.w, g[i].w));
                    }
                }
            };
            // operands of one piece of the four rows
            auto load_ops = [&](int c0, float4* x, float4* y) {
                const int nc = N - (c0 + c4), col = VEC ? std::min(c0 + c4, N - 4) : c0 + c4;
                (void)y;
                if constexpr (MODE == kAdd && kEdge) {
                    load_g(c0, x);
                } else if constexpr (kGather) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        x[i] = load4<VEC>(A.P + (int64_t)rv[i] * A.ldpq + col, VEC ? 4 : nc);
                        y[i] = load4<VEC>(A.Q + (int64_t)sv[i] * A.ldpq + col, VEC ? 4 : nc);
                    }
                } else if constexpr (MODE != kLnAdjoint && OPS == kOpsRow) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) x[i] = load4<VEC>(A.add + row[i] * A.ldadd + col, VEC ? 4 : nc);
                }
            };
            float4 x[4], y[4];
            load_ops(0, x, y);   // before the wait: the first piece's operands
            ok = warp_wait(acc_full + eg, (uint32_t)(j >> 1) & 1u, lane);
            if (!ok) break;
            tc_fence_after();
            auto special = [&](float v) {
                if (patched || !__any_sync(0xffffffffu, lane < nv && !finite(v + spoil))) return false;
                patch_sums(LinSum{A, lane < nv ? rb + lane : 0}, lane < nv, tacc, NP, acc, gain);
                return patched = true;
            };
            float mean = 0.f, rstd = 0.f, m1 = 0.f, m2 = 0.f;
            if constexpr (MODE == kLayerNorm || MODE == kLnAdjoint) {
                // row statistics: the lane's row, two passes over the accumulator
                float s4[4] = {0.f, 0.f, 0.f, 0.f};
                for (int c0 = 0; c0 < N; c0 += 16) {
                    float v[16];
                    load_sum16(tacc + c0, NP, acc, gain, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) s4[i & 3] += v[i] + sPar[c0 + i];   // padding columns are zero
                }
                mean = ((s4[0] + s4[1]) + (s4[2] + s4[3])) / N;
                if (special(mean)) continue;
                float q4[4] = {0.f, 0.f, 0.f, 0.f};
                for (int c0 = 0; c0 < N; c0 += 16) {
                    float v[16];
                    load_sum16(tacc + c0, NP, acc, gain, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float d = c0 + i < N ? v[i] + sPar[c0 + i] - mean : 0.f;
                        q4[i & 3] = fmaf(d, d, q4[i & 3]);
                    }
                }
                rstd = rsqrtf(((q4[0] + q4[1]) + (q4[2] + q4[3])) / N + A.eps);
            }
            if constexpr (MODE == kLnAdjoint) {
                // g, and its two row sums against gamma and gamma * xhat
                for (int c0 = 0; c0 < N; c0 += 16) {
                    float4 g[4];
                    load_g(c0, g);
#pragma unroll
                    for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(stg + (8 * i + rs) * kStageLd + c4) = g[i];
                    float v[16];
                    load_sum16(tacc + c0, NP, acc, gain, v);
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 16; i += 4) {
                        const float4 g4 = *reinterpret_cast<const float4*>(stg + lane * kStageLd + i);
                        const float gg[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            // (a clamped piece past the last column repeats real values: not counted)
                            const float d = c0 + i + k < N ? __fmul_rn(gg[k], sPar[NP + c0 + i + k]) : 0.f;
                            m1 += d;
                            m2 = fmaf(d, (v[i + k] + sPar[c0 + i + k] - mean) * rstd, m2);
                        }
                    }
                    __syncwarp();
                }
                m1 /= N;
                m2 /= N;
            }
            bool again = false;
            for (int c0 = 0; c0 < NP; c0 += 16) {
                const int col = c0 + c4, nc = N - col;
                float v[16];
                load_sum16(tacc + c0, NP, acc, gain, v);
                if (MODE != kLayerNorm && MODE != kLnAdjoint && c0 == 0 && (again = special(v[0]))) break;
                if constexpr (MODE == kLayerNorm || MODE == kLnAdjoint) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[i] = (v[i] + sPar[c0 + i] - mean) * rstd;   // xhat
                }
#pragma unroll
                for (int i = 0; i < 16; i += 4)
                    *reinterpret_cast<float4*>(stg + lane * kStageLd + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                const float4 b = *reinterpret_cast<const float4*>(sPar + col);
                float4 ga = b, be = b;
                if constexpr (MODE == kLayerNorm || MODE == kLnAdjoint) {
                    ga = *reinterpret_cast<const float4*>(sPar + NP + col);
                    be = *reinterpret_cast<const float4*>(sPar + 2 * NP + col);
                }
                if constexpr (MODE == kLnAdjoint) load_g(c0, x);
                __syncwarp();
                float4 u[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) u[i] = *reinterpret_cast<const float4*>(stg + (8 * i + rs) * kStageLd + c4);
                if constexpr (MODE == kElu) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        u[i] = add4(u[i], b);
                        if constexpr (OPS == kOpsRow) u[i] = add4(u[i], x[i]);
                        if constexpr (OPS == kOpsGather) u[i] = add4(u[i], add4(x[i], y[i]));
                    }
                } else if constexpr (MODE == kLayerNorm) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        u[i] = make_float4(u[i].x * ga.x + be.x, u[i].y * ga.y + be.y, u[i].z * ga.z + be.z,
                                           u[i].w * ga.w + be.w);
                        if constexpr (OPS == kOpsRow) u[i] = add4(u[i], x[i]);
                    }
                } else if constexpr (MODE == kLnAdjoint) {
                    float4 sg = make_float4(0.f, 0.f, 0.f, 0.f), sb = sg;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int r = 8 * i + rs;
                        const float rr = __shfl_sync(0xffffffffu, rstd, r);
                        const float a1 = __shfl_sync(0xffffffffu, m1, r), a2 = __shfl_sync(0xffffffffu, m2, r);
                        const float4 g = x[i], xh = u[i];
                        if (r < nv) {   // clamped rows are not counted
                            sg = make_float4(sg.x + g.x * xh.x, sg.y + g.y * xh.y, sg.z + g.z * xh.z, sg.w + g.w * xh.w);
                            sb = add4(sb, g);
                        }
                        // g gamma as rounded for the sums: equal terms cancel exactly (one column: dz = 0)
                        auto dz = [&](float gg, float gm, float h) { return rr * (__fmul_rn(gg, gm) - a1 - h * a2); };
                        u[i] = make_float4(dz(g.x, ga.x, xh.x), dz(g.y, ga.y, xh.y), dz(g.z, ga.z, xh.z),
                                           dz(g.w, ga.w, xh.w));
                    }
                    // column sums over the warp's rows
                    float cs[8] = {sg.x, sg.y, sg.z, sg.w, sb.x, sb.y, sb.z, sb.w};
#pragma unroll
                    for (int o = 4; o < 32; o <<= 1) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) cs[i] += __shfl_xor_sync(0xffffffffu, cs[i], o);
                    }
                    if (lane < 4) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            sums[col + i] += cs[i];
                            sums[NP + col + i] += cs[4 + i];
                        }
                    }
                } else if constexpr (MODE == kEluAdjoint) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        u[i] = make_float4(u[i].x * elu1_deriv_from_out(x[i].x), u[i].y * elu1_deriv_from_out(x[i].y),
                                           u[i].z * elu1_deriv_from_out(x[i].z), u[i].w * elu1_deriv_from_out(x[i].w));
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        u[i] = add4(u[i], b);
                        if constexpr (OPS != kOpsNone) u[i] = add4(u[i], x[i]);
                    }
                }
                // the next piece's operands (an in-place sum reads other columns than it has written)
                if (MODE != kLnAdjoint && c0 + 16 < NP) load_ops(c0 + 16, x, y);
                if constexpr (MODE == kElu) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float2 lo = elu_pair(make_float2(u[i].x, u[i].y)), hi = elu_pair(make_float2(u[i].z, u[i].w));
                        u[i] = make_float4(lo.x, lo.y, hi.x, hi.y);
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (8 * i + rs < nv) store4<VEC>(A.out + row[i] * A.ldo + col, nc, u[i]);
                __syncwarp();
            }
            if (again) continue;
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty + eg);
            next();
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if constexpr (MODE == kLnAdjoint) {
        const float* z = reinterpret_cast<const float*>(sm + P.sums);
        for (int i = tid; i < 2 * N; i += kThreads) {
            const int o = (i < N) ? i : NP + (i - N);
            float s = 0.f;
            for (int w = 0; w < kEpilogueWarps; ++w) s += z[w * 2 * NP + o];
            A.part[(int64_t)blockIdx.x * 2 * N + i] = s;
        }
    }
    if (warp == 0) tmem_dealloc(tmem, NCOLS);
}

// ------------------------------------------------------------------ k_wgrad3

struct WArgs {
    int64_t rows;
    int n_tiles;               // of RT rows
    int RT;                    // rows per stage: 128, or 64 when an operand is 128 wide
    const float* G;
    const float* X;
    int64_t ldg, ldx;
    int N, K, NP, db, vec_g, vec_x, stages;
    float* part;
};

struct WSmem {
    uint32_t st, red, bar, tm, total, gterm, xterm, stage;
};

__host__ __device__ inline WSmem wgrad_smem(int NP, int KP, int RT, int stages) {
    WSmem s;
    s.gterm = (uint32_t)RT * NP * 2;
    s.xterm = (uint32_t)RT * KP * 2;
    s.stage = 3 * (s.gterm + s.xterm);
    s.st = 0;
    // M = 128 views of a narrower G read up to 256 RT bytes from a term's start: inside the
    // stages, or in the pad behind the last one
    uint32_t end = (uint32_t)stages * s.stage;
    end = std::max(end, (uint32_t)(stages - 1) * s.stage + 2 * s.gterm + 256u * RT);
    s.red = align_up(end, 16);                        // db: [128 threads][8]
    s.bar = align_up(s.red + kSide * 8 * 4, 8);  // full[4], empty[4], acc_full[2], acc_empty[2]
    s.tm = s.bar + 12 * 8;
    s.total = s.tm + 16 + 1024;
    return s;
}

struct WSide {
    const float* src;
    int64_t ld;
    int cols;
    uint32_t dst;   // of stage 0
};

// Load, split and write one operand's rows of every stage: [R x W], and their
// column sums (cs: the thread's 8 columns, rows in order).
template <int W, int R, bool VEC>
__device__ __forceinline__ void wgrad_producer(const WArgs& A, const WSmem& P, const WSide& d, uint8_t* sm,
                                               uint64_t* full, uint64_t* empty, int pt, int lane, float* cs) {
    constexpr int U = W / 8, RS = kSide / U, IT = R / RS, B = IT < 4 ? IT : 4, S = span_of(W);
    constexpr uint32_t TERM = R * W * 2;
    const int c = (pt % U) * 8, row0 = pt / U, nc = d.cols - c;
    const uint32_t off0 = tile_off(row0, c, R, S);
    // rows RS apart: whole swizzle periods (1024 bytes) except the 128-wide rows, 8 apart, with the same period
    static_assert((RS * S) % 1024 == 0, "the swizzle repeats every RS rows");
    const int64_t step = RS * d.ld;
    int st = 0, use = 0;
    for (int t = blockIdx.x; t < A.n_tiles; t += gridDim.x) {
        if (VEC && pt == 0 && d.ld == d.cols && t + (int)gridDim.x < A.n_tiles) {   // the next tile's rows into L2
            const int64_t rn = (int64_t)(t + (int)gridDim.x) * R;
            prefetch_l2(d.src + rn * d.ld, (uint32_t)(std::min<int64_t>(R, A.rows - rn) * d.cols * 4));
        }
        const int left = (int)std::min<int64_t>(R, A.rows - (int64_t)t * R);
        const float* src = d.src + ((int64_t)t * R + row0) * d.ld + c;
        uint8_t* dst = sm + d.dst + (uint32_t)st * P.stage + off0;
#pragma unroll
        for (int i0 = 0; i0 < IT; i0 += B) {
            float v[B][8];
            if (left == R && d.cols == W) {
#pragma unroll
                for (int i = 0; i < B; ++i) load8<VEC>(src + (i0 + i) * step, 8, v[i]);
            } else {
#pragma unroll
                for (int i = 0; i < B; ++i)
                    load8<VEC>(src + (i0 + i) * step, row0 + (i0 + i) * RS < left ? nc : 0, v[i]);
            }
            if (i0 == 0 && use > 0 && !warp_wait(empty + st, (uint32_t)(use - 1) & 1u, lane)) return;
#pragma unroll
            for (int i = 0; i < B; ++i) {
#pragma unroll
                for (int k = 0; k < 8; ++k) cs[k] += v[i][k];
                uint4 h, m, l;
                split8(v[i], h, m, l);
                uint8_t* q = dst + (i0 + i) * RS * S;
                *reinterpret_cast<uint4*>(q) = h;
                *reinterpret_cast<uint4*>(q + TERM) = m;
                *reinterpret_cast<uint4*>(q + 2 * TERM) = l;
            }
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(full + st);
        if (++st == A.stages) {
            st = 0;
            ++use;
        }
    }
}

// dW = G^T X over the CTA's row tiles: both operands are MN-major views of the
// same split row tiles (rows = the contraction). The sums of one tile (RT rows)
// are added to FP32 registers by the epilogue warps, so no tensor-core
// sum runs over more than RT rows.
template <int KP>
__global__ void __launch_bounds__(kWThreads, 1) k_wgrad3(const __grid_constant__ WArgs A) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = aligned_smem(smem_raw);
    const int NP = A.NP, RT = A.RT, stages = A.stages, N = A.N, K = A.K;
    const int Sg = span_of(NP);
    constexpr int Sx = span_of(KP);
    const WSmem P = wgrad_smem(NP, KP, RT, stages);
    uint64_t* full = reinterpret_cast<uint64_t*>(sm + P.bar);
    uint64_t* empty = full + 4;
    uint64_t* acc_full = full + 8;
    uint64_t* acc_empty = full + 10;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + P.tm);
    float* sRed = reinterpret_cast<float*>(sm + P.red);
    constexpr int SUMS = KP <= 64 ? 3 : 1;              // accumulators of a tile (of width 128: one)
    constexpr uint32_t NCOLS = 2 * SUMS * KP <= 128 ? 128 : (2 * SUMS * KP <= 256 ? 256 : 512);
    constexpr int CW = KP >= 32 ? KP / 2 : 16;      // accumulator columns per epilogue thread
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == 0) {
        tmem_alloc(tslot, NCOLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < stages; ++i) {
            mbar_init(full + i, kWProducerWarps);
            mbar_init(empty + i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(acc_full + i, 1);
            mbar_init(acc_empty + i, kEpilogueWarps);
        }
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    float* part = A.part + (int64_t)blockIdx.x * (N * K + (A.db ? N : 0));

    if (warp < kWProducerWarps) {
        // half of the producer warps split G, half X
        const bool x = warp >= kWProducerWarps / 2;
        const int pt = tid & (kSide - 1);
        const WSide d{x ? A.X : A.G, x ? A.ldx : A.ldg, x ? K : N, P.st + (x ? 3 * P.gterm : 0u)};
        float cs[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) cs[i] = 0.f;
        auto go = [&](auto w, auto rt) {
            constexpr int W = decltype(w)::value, R = decltype(rt)::value;
            if (x ? A.vec_x : A.vec_g) wgrad_producer<W, R, true>(A, P, d, sm, full, empty, pt, lane, cs);
            else wgrad_producer<W, R, false>(A, P, d, sm, full, empty, pt, lane, cs);
        };
        const int w = x ? KP : NP;
        if (RT == 64) {
            if (w == 128) go(Int<128>(), Int<64>());
            else if (w == 64) go(Int<64>(), Int<64>());
            else if (w == 32) go(Int<32>(), Int<64>());
            else go(Int<16>(), Int<64>());
        } else {
            if (w == 64) go(Int<64>(), Int<128>());
            else if (w == 32) go(Int<32>(), Int<128>());
            else go(Int<16>(), Int<128>());
        }
        if (A.db && !x) {   // column sums of G: threads of one column group in thread order
            const int gu = NP / 8;
#pragma unroll
            for (int k = 0; k < 8; ++k) sRed[pt * 8 + k] = cs[k];
            named_sync(1, kSide);
            for (int c = pt; c < N; c += kSide) {
                float s = 0.f;
                for (int i = c / 8; i < kSide; i += gu) s += sRed[i * 8 + (c & 7)];
                part[(int64_t)N * K + c] = s;
            }
        }
    } else if (warp == kWProducerWarps + kEpilogueWarps) {
        {
            const uint32_t lead = elect_one();
            constexpr uint32_t id = idesc_bf16(128, KP, 1, 1);
            const uint32_t base = smem_u32(sm + P.st);
            const uint64_t g0 = sdesc(base, (uint32_t)RT * Sg, 8 * Sg, swz_code(Sg));
            const uint64_t x0 = sdesc(base + 3 * P.gterm, (uint32_t)RT * Sx, 8 * Sx, swz_code(Sx));
            int n = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < A.n_tiles && ok; t += gridDim.x, ++n) {
                const int st = n % stages, use = n / stages, buf = n & 1;
                if (n >= 2) ok = mbar_wait(acc_empty + buf, (uint32_t)((n >> 1) - 1) & 1u);
                ok = ok && mbar_wait(full + st, (uint32_t)use & 1u);
                if (!ok) break;
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(buf * SUMS * KP), so = (uint32_t)st * P.stage;
                auto issue = [&](auto rt) {
                    if constexpr (SUMS == 3) {   // the terms of X are consecutive blocks of one MN-major operand
                        const uint64_t xp = desc_step(x0, so);
#pragma unroll
                        for (int p = 0; p < 3; ++p) {
                            const uint64_t gp = desc_step(g0, so + p * P.gterm);
                            constexpr uint32_t ids[3] = {idesc_bf16(128, 3 * KP, 1, 1), idesc_bf16(128, 2 * KP, 1, 1), id};
#pragma unroll
                            for (int k0 = 0; k0 < decltype(rt)::value; k0 += 16)
                                mma_bf16_warp(lead, d + p * KP, desc_step(gp, (uint32_t)(k0 * Sg)), desc_step(xp, (uint32_t)(k0 * Sx)),
                                         ids[p], (p > 0 || k0 > 0) ? 1u : 0u);
                        }
                    } else {
#pragma unroll
                        for (int p = 0; p < 6; ++p) {
                            const uint64_t gp = desc_step(g0, so + kTermA[p] * P.gterm);
                            const uint64_t xp = desc_step(x0, so + kTermB[p] * P.xterm);
#pragma unroll
                            for (int k0 = 0; k0 < decltype(rt)::value; k0 += 16)
                                mma_bf16_warp(lead, d, desc_step(gp, (uint32_t)(k0 * Sg)), desc_step(xp, (uint32_t)(k0 * Sx)), id,
                                         (p > 0 || k0 > 0) ? 1u : 0u);
                        }
                    }
                };
                if (RT == 64) issue(Int<64>());
                else issue(Int<128>());
                mma_commit_warp(lead, empty + st);
                mma_commit_warp(lead, acc_full + buf);
            }
            if (ok && n > 0) mbar_wait(empty + (n - 1) % stages, (uint32_t)((n - 1) / stages) & 1u);
        }
        __syncwarp();
    } else {
        const int ew = warp - kWProducerWarps, q = ew & 3, half = ew >> 2;
        const int c0 = half * CW;
        const bool work = c0 < KP;
        float acc[CW];
#pragma unroll
        for (int i = 0; i < CW; ++i) acc[i] = 0.f;
        int n = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < A.n_tiles && ok; t += gridDim.x, ++n) {
            const int buf = n & 1;
            ok = warp_wait(acc_full + buf, (uint32_t)(n >> 1) & 1u, lane);
            if (!ok) break;
            tc_fence_after();
            if (work) {
#pragma unroll
                for (int i = 0; i < CW; i += 16) {
                    float v[16];
                    const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * SUMS * KP + c0 + i);
                    load_acc16<SUMS == 3 ? kAccThree : kAccAll>(ta, KP, 0.f, v);
#pragma unroll
                    for (int k = 0; k < 16; ++k) acc[i + k] = fmaf(v[k], kUnscale, acc[i + k]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty + buf);
        }
        const int r = 32 * q + lane;
        if (work && r < N) {
#pragma unroll
            for (int i = 0; i < CW; ++i) {
                if (c0 + i >= K) continue;
                float* o = part + (int64_t)r * K + c0 + i;
                *o = acc[i];
                if (!finite(acc[i])) *o = dw_sum(A.G + r, A.ldg, A.X + c0 + i, A.ldx, A.rows, A.n_tiles, RT);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, NCOLS);
}

// ------------------------------------------------------------------ k_chain3

// One Linear of the adjoint chain at widths <= 64, both halves in one pass over
// dz [rows x N] and h [rows x K]: dz' = (dz W) ELU'(h) and dW += dz^T h,
// db += column sums of dz. dz is split once for both products (its row tile is
// the K-major operand of the first and the MN-major one of the second), h once,
// and each row is read once instead of twice (three tensors moved instead of
// five). Two stages of dz and one of h fill shared memory beside W; the widths
// above 64 need twice that and keep the two launches. 3.23M edge rows at width
// 64: 0.72 ms (0.84 with one MMA per product) against 0.49 + 0.48 for the two
// launches: the four producer warps split both operands and set the pace (HBM
// alone: 0.37).
struct CArgs {
    int64_t rows;
    int n_tiles;
    const float* G;      // dz [rows x N]
    const float* H;      // h [rows x K]
    const float* W;      // [N x K]
    float* out;          // dz' [rows x K]
    int N, K, db, vec;
    float* part;         // per CTA: dW [N x K], then db [N]
};

struct CSmem {
    uint32_t w, g, h, stg, red, bar, tm, total, wterm, gterm, hterm;
};

template <int NW, int KW>
__host__ __device__ constexpr CSmem chain_smem() {
    CSmem s{};
    s.wterm = KW * NW * 2;
    s.gterm = 128 * NW * 2;
    s.hterm = 128 * KW * 2;
    s.w = 0;
    s.g = align_up(3 * s.wterm, 1024);
    s.h = s.g + 2 * 3 * s.gterm;
    // M = 128 views of a narrower dz tile read 32 KB from a term's start: the h stage and what follows
    uint32_t end = s.h + 3 * s.hterm;
    const uint32_t view = s.h - s.gterm + 32768;
    end = end > view ? end : view;
    s.stg = align_up(end, 16);
    s.red = s.stg + kEpilogueWarps * kStageBytes;        // db: [128 threads][8]
    s.bar = align_up(s.red + kProducers * 8 * 4, 8);     // full_g[2], empty_g[2], full_h, empty_h, acc_full[2], acc_empty[2], w_full[2], w_empty[2]
    s.tm = s.bar + 14 * 8;
    s.total = s.tm + 16 + 1024;
    return s;
}

// Load, split and write the [128 x W] rows of one operand tile; cs: column sums (or NULL).
template <int W, bool VEC, bool SUM>
__device__ __forceinline__ void chain_fill(const float* src, int64_t ld, int cols, int left, uint8_t* dst, int tid,
                                           float* cs, uint64_t* empty, bool wait, uint32_t parity, int lane, bool& ok) {
    constexpr int U = W / 8, RS = kProducers / U, IT = 128 / RS, B = IT < 8 ? IT : 8, S = span_of(W);
    static_assert((RS * S) % 1024 == 0, "the swizzle repeats every RS rows");
    const int c = (tid % U) * 8, row0 = tid / U;
    uint8_t* d0 = dst + tile_off(row0, c, 128, S);
    const float* p = src + (int64_t)row0 * ld + c;
    const int64_t step = RS * ld;
#pragma unroll
    for (int i0 = 0; i0 < IT; i0 += B) {
        float v[B][8];
        if (left == 128 && cols == W) {
#pragma unroll
            for (int i = 0; i < B; ++i) load8<VEC>(p + (i0 + i) * step, 8, v[i]);
        } else {
#pragma unroll
            for (int i = 0; i < B; ++i) load8<VEC>(p + (i0 + i) * step, row0 + (i0 + i) * RS < left ? cols - c : 0, v[i]);
        }
        if (i0 == 0 && wait) {
            ok = warp_wait(empty, parity, lane);
            if (!ok) return;
        }
#pragma unroll
        for (int i = 0; i < B; ++i) {
            if constexpr (SUM) {
#pragma unroll
                for (int k = 0; k < 8; ++k) cs[k] += v[i][k];
            }
            uint4 h, m, l;
            split8(v[i], h, m, l);
            uint8_t* q = d0 + (i0 + i) * RS * S;
            *reinterpret_cast<uint4*>(q) = h;
            *reinterpret_cast<uint4*>(q + 128 * S) = m;
            *reinterpret_cast<uint4*>(q + 2 * 128 * S) = l;
        }
    }
    fence_proxy_async();
    __syncwarp();
}

// NW, KW: N and K rounded up to 16, 32 or 64.
template <int NW, int KW, bool VEC>
__global__ void __launch_bounds__(kThreads, 1) k_chain3(const __grid_constant__ CArgs A) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = aligned_smem(smem_raw);
    constexpr CSmem P = chain_smem<NW, KW>();
    constexpr int Sg = span_of(NW), Sh = span_of(KW);
    uint64_t* full_g = reinterpret_cast<uint64_t*>(sm + P.bar);
    uint64_t* empty_g = full_g + 2;
    uint64_t* full_h = full_g + 4;
    uint64_t* empty_h = full_g + 5;
    uint64_t* acc_full = full_g + 6;
    uint64_t* acc_empty = full_g + 8;
    uint64_t* w_full = full_g + 10;
    uint64_t* w_empty = full_g + 12;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + P.tm);
    float* sRed = reinterpret_cast<float*>(sm + P.red);
    // TMEM: dz' of two tiles, three sums each (at KW = 64 two: five MMAs a K-step), then dW, three
    // sums, of two tiles (at KW = 64 of one: the next tile's dz' is under way while it is read)
    constexpr Acc ZA = KW <= 32 ? kAccThree : kAccSmall;
    constexpr int ZS = acc_count(ZA), WB = KW <= 32 ? 2 : 1;
    constexpr uint32_t WCOL = 2 * ZS * KW;
    constexpr uint32_t NCOLS = WCOL + WB * 3 * KW <= 256 ? 256 : 512;
    static_assert(WCOL + WB * 3 * KW <= 512, "tensor memory");
    constexpr int CW = KW >= 32 ? KW / 2 : 16;   // dW columns per epilogue thread
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, N = A.N, K = A.K;

    if (warp == 0) {
        tmem_alloc(tslot, NCOLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(full_g + i, kProducerWarps);
            mbar_init(empty_g + i, 1);
            mbar_init(acc_full + i, 1);
            mbar_init(acc_empty + i, 4);
            mbar_init(w_full + i, 1);
            mbar_init(w_empty + i, kEpilogueWarps);
        }
        mbar_init(full_h, kProducerWarps);
        mbar_init(empty_h, 1);
        fence_mbar_init();
    }
    bool special_w = false;
    // W^T as the [KW x NW] K-major operand of dz W: row k, column n
    for (int i = tid; i < KW * (NW / 8); i += kThreads) {
        const int k = i / (NW / 8), n8 = (i % (NW / 8)) * 8;
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = (k < K && n8 + j < N) ? __ldg(A.W + (int64_t)(n8 + j) * K + k) : 0.f;
        special_w |= check_weights(v);
        uint4 t[3];
        split8<true>(v, t[0], t[1], t[2]);
        const uint32_t off = tile_off(k, n8, KW, Sg);
#pragma unroll
        for (int j = 0; j < 3; ++j) *reinterpret_cast<uint4*>(sm + P.w + j * P.wterm + off) = t[j];
    }
    fence_proxy_async();
    tc_fence_before();
    const float spoil = __syncthreads_or(special_w) ? __uint_as_float(0x7fffffffu) : 0.f;   // not finite if special
    tc_fence_after();
    const uint32_t tmem = *tslot;
    float* part = A.part + (int64_t)blockIdx.x * (N * K + (A.db ? N : 0));

    if (warp < kProducerWarps) {
        float cs[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) cs[i] = 0.f;
        bool ok = true;
        int j = 0;
        for (int t = blockIdx.x; t < A.n_tiles && ok; t += gridDim.x, ++j) {
            if (VEC && tid == 0 && t + (int)gridDim.x < A.n_tiles) {   // the next tile's rows into L2
                const int64_t rn = (int64_t)(t + (int)gridDim.x) * 128, nr = std::min<int64_t>(128, A.rows - rn);
                prefetch_l2(A.G + rn * N, (uint32_t)(nr * N * 4));
                prefetch_l2(A.H + rn * K, (uint32_t)(nr * K * 4));
            }
            const int64_t r0 = (int64_t)t * 128;
            const int left = (int)std::min<int64_t>(128, A.rows - r0), st = j & 1;
            chain_fill<NW, VEC, true>(A.G + r0 * N, N, N, left, sm + P.g + st * 3 * P.gterm, tid, cs, empty_g + st, j >= 2,
                                      (uint32_t)((j >> 1) - 1) & 1u, lane, ok);
            if (!ok) break;
            if (lane == 0) mbar_arrive(full_g + st);
            chain_fill<KW, VEC, false>(A.H + r0 * K, K, K, left, sm + P.h, tid, nullptr, empty_h, j >= 1,
                                       (uint32_t)(j - 1) & 1u, lane, ok);
            if (!ok) break;
            if (lane == 0) mbar_arrive(full_h);
        }
        if (A.db) {   // column sums of dz: threads of one column group in thread order
            constexpr int GU = NW / 8;
#pragma unroll
            for (int k = 0; k < 8; ++k) sRed[tid * 8 + k] = cs[k];
            named_sync(1, kProducers);
            for (int c = tid; c < N; c += kProducers) {
                float s = 0.f;
                for (int i = c / 8; i < kProducers; i += GU) s += sRed[i * 8 + (c & 7)];
                part[(int64_t)N * K + c] = s;
            }
        }
    } else if (warp == kProducerWarps + kEpilogueWarps) {
        {
            const uint32_t lead = elect_one();
            const uint32_t gb = smem_u32(sm + P.g), hb = smem_u32(sm + P.h);
            const uint64_t gk = kmajor_desc(gb, 128, Sg, 0), wk = kmajor_desc(smem_u32(sm + P.w), KW, Sg, 0);
            const uint64_t gm = sdesc(gb, 128u * Sg, 8 * Sg, swz_code(Sg)), hm = sdesc(hb, 128u * Sh, 8 * Sh, swz_code(Sh));
            constexpr uint32_t idz[3] = {idesc_bf16(128, ZS * KW), idesc_bf16(128, (ZS - 1) * KW), idesc_bf16(128, KW)};
            constexpr uint32_t idw[3] = {idesc_bf16(128, 3 * KW, 1, 1), idesc_bf16(128, 2 * KW, 1, 1), idesc_bf16(128, KW, 1, 1)};
            bool ok = true;
            int j = 0;
            for (int t = blockIdx.x; t < A.n_tiles && ok; t += gridDim.x, ++j) {
                const int b = j & 1;
                const uint32_t go = (uint32_t)b * 3 * P.gterm, par = (uint32_t)((j >> 1) - 1) & 1u;
                if (j >= 2) ok = mbar_wait(acc_empty + b, par);
                ok = ok && mbar_wait(full_g + b, (uint32_t)(j >> 1) & 1u);
                if (!ok) break;
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(b * ZS * KW);
                auto z = [&](int col, int ta, int tw, uint32_t id, bool add) {
                    const uint64_t a = desc_step(gk, go + ta * P.gterm), w = desc_step(wk, tw * P.wterm);
#pragma unroll
                    for (int k0 = 0; k0 < NW; k0 += 16)
                        mma_bf16_warp(lead, d + col * KW, desc_step(a, k0 * 2), desc_step(w, k0 * 2), id, (add || k0 > 0) ? 1u : 0u);
                };
                z(0, 0, 0, idz[0], false);
                z(1, 1, 0, idz[1], true);
                if constexpr (ZS == 3) {
                    z(2, 2, 0, idz[2], true);
                } else {
                    z(1, 2, 0, idz[2], true);
                    z(1, 1, 1, idz[2], true);
                    z(1, 0, 2, idz[2], true);
                }
                mma_commit_warp(lead, acc_full + b);
                const int wb = j % WB;
                if (j >= WB) ok = mbar_wait(w_empty + wb, (uint32_t)(j / WB - 1) & 1u);
                ok = ok && mbar_wait(full_h, (uint32_t)j & 1u);
                if (!ok) break;
                tc_fence_after();
                const uint32_t dw = tmem + WCOL + (uint32_t)(wb * 3 * KW);
#pragma unroll
                for (int p = 0; p < 3; ++p) {
                    const uint64_t a = desc_step(gm, go + p * P.gterm);
#pragma unroll
                    for (int k0 = 0; k0 < 128; k0 += 16)
                        mma_bf16_warp(lead, dw + p * KW, desc_step(a, (uint32_t)(k0 * Sg)), desc_step(hm, (uint32_t)(k0 * Sh)), idw[p],
                                 (p > 0 || k0 > 0) ? 1u : 0u);
                }
                mma_commit_warp(lead, empty_g + b);
                mma_commit_warp(lead, empty_h);
                mma_commit_warp(lead, w_full + wb);
            }
            // the last releases have arrived before the block may end
            if (ok && j > 0) {
                mbar_wait(empty_h, (uint32_t)(j - 1) & 1u);
                mbar_wait(empty_g + ((j - 1) & 1), (uint32_t)((j - 1) >> 1) & 1u);
            }
        }
        __syncwarp();
    } else {
        const int ew = warp - kProducerWarps, eg = ew >> 2, q = ew & 3;
        float* stg = reinterpret_cast<float*>(sm + P.stg + ew * kStageBytes);
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        const int rs = lane >> 2, c4 = (lane & 3) * 4;
        const int c0w = eg * CW;               // this thread's dW columns (row 32 q + lane)
        float acc[CW];
#pragma unroll
        for (int i = 0; i < CW; ++i) acc[i] = 0.f;
        bool ok = true;
        const float zgain = gain_of((N + 15) / 16);
        // dW of tile j into the registers: by the tile's own group halfway through it, by the other
        // one after its tile before, at about the same time
        auto read_w = [&](int j) {
            const int wb = j % WB;
            ok = warp_wait(w_full + wb, (uint32_t)(j / WB) & 1u, lane);
            if (!ok) return;
            tc_fence_after();
            if (c0w < KW) {
#pragma unroll
                for (int i = 0; i < CW; i += 16) {
                    float v[16];
                    load_acc16<kAccThree>(tmem + lane_base + WCOL + (uint32_t)(wb * 3 * KW + c0w + i), KW, 0.f, v);
#pragma unroll
                    for (int k = 0; k < 16; ++k) acc[i + k] = fmaf(v[k], kUnscale, acc[i + k]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(w_empty + wb);
        };
        int j = 0, t = blockIdx.x;
        bool patched = false;   // as in k_lin3; a special tile is begun again before its dW is read
        while (t < A.n_tiles && ok) {
            const int b = j & 1;
            if (b == eg) {   // this group's tile: dz' = acc ELU'(h)
                const int64_t rb = (int64_t)t * 128 + 32 * q;
                const int nv = (int)std::min<int64_t>(32, std::max<int64_t>(0, A.rows - rb));
                int64_t row[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) row[i] = nv > 0 ? rb + std::min(8 * i + rs, nv - 1) : 0;
                auto load_h = [&](int c0, float4* x) {
                    const int nc = K - (c0 + c4), col = VEC ? std::min(c0 + c4, K - 4) : c0 + c4;
#pragma unroll
                    for (int i = 0; i < 4; ++i) x[i] = load4<VEC>(A.H + row[i] * K + col, VEC ? 4 : nc);
                };
                float4 x[4];
                load_h(0, x);
                ok = warp_wait(acc_full + b, (uint32_t)(j >> 1) & 1u, lane);
                if (!ok) break;
                tc_fence_after();
                const uint32_t tacc = tmem + lane_base + (uint32_t)(b * ZS * KW);
                bool again = false;
#pragma unroll
                for (int c0 = 0; c0 < KW; c0 += 16) {
                    float v[16];
                    load_acc16<ZA>(tacc + c0, KW, zgain, v);
                    if (c0 == 0 && !patched && __any_sync(0xffffffffu, lane < nv && !finite(v[0] + spoil))) {
                        patch_sums(RowSum{A.G + (lane < nv ? rb + lane : 0) * N, A.W, N, K}, lane < nv, tacc, KW, ZA, zgain);
                        again = patched = true;
                        break;
                    }
#pragma unroll
                    for (int i = 0; i < 16; i += 4)
                        *reinterpret_cast<float4*>(stg + lane * kStageLd + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                    __syncwarp();
                    float4 u[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 z = *reinterpret_cast<const float4*>(stg + (8 * i + rs) * kStageLd + c4);
                        u[i] = make_float4(z.x * elu1_deriv_from_out(x[i].x), z.y * elu1_deriv_from_out(x[i].y),
                                           z.z * elu1_deriv_from_out(x[i].z), z.w * elu1_deriv_from_out(x[i].w));
                    }
                    if (c0 + 16 < KW) load_h(c0 + 16, x);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (8 * i + rs < nv) store4<VEC>(A.out + row[i] * K + c0 + c4, K - (c0 + c4), u[i]);
                    __syncwarp();
                    if (c0 == (KW == 64 ? 16 : 0)) read_w(j);
                }
                if (again) continue;
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acc_empty + b);
            }
            if (b != eg) read_w(j);
            t += gridDim.x;
            ++j;
            patched = false;
        }
        const int r = 32 * q + lane;
        if (c0w < KW && r < N) {
#pragma unroll
            for (int i = 0; i < CW; ++i) {
                if (c0w + i >= K) continue;
                float* o = part + (int64_t)r * K + c0w + i;
                *o = acc[i];
                if (!finite(acc[i])) *o = dw_sum(A.G + r, N, A.H + c0w + i, K, A.rows, A.n_tiles, 128);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, NCOLS);
}

// ------------------------------------------------------------------ k_reduce3

struct RedArgs {
    Sum s[kMaxReduce];
    int first[kMaxReduce + 1];   // first block of each sum
    int n;
};

// 32 elements x 8 lanes over the partials of a block: lane l sums the partials
// l, l + 8, ... in order, and the lanes are combined in order.
__global__ void __launch_bounds__(256) k_reduce3(const __grid_constant__ RedArgs A) {
    __shared__ float red[8][33];
    int i = 0;
    while (i + 1 < A.n && (int)blockIdx.x >= A.first[i + 1]) ++i;
    const Sum& S = A.s[i];
    const int cx = threadIdx.x & 31, l = threadIdx.x >> 5;
    const int e = ((int)blockIdx.x - A.first[i]) * 32 + cx;
    float s = 0.f;
    if (e < S.N * S.K) {
        const float* p = S.part + e;
#pragma unroll 4
        for (int z = l; z < S.nz; z += 8) s += p[(int64_t)z * S.stride];
    }
    red[l][cx] = s;
    __syncthreads();
    if (l == 0 && e < S.N * S.K) {
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) t += red[k][cx];
        float* d = S.dst + (int64_t)(e / S.K) * S.ldd + e % S.K;
        *d += t;
    }
}

inline bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

template <class Kern>
int set_smem(Kern k, uint32_t bytes) {
    GNN_CUDA_CHECK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes),
                   "cudaFuncSetAttribute");
    return GNN_OK;
}

int pick_stages(int NP, int KB, int nkb) {
    for (int s = 4; s >= 2; --s)
        if (lin_smem(NP, KB, nkb, s).total <= kSmemMax) return s;
    return 0;
}

int blocks_of(int K, int KB) { return K ? (pow2_width(K) + KB - 1) / KB : 0; }
int block_width(int K) { return std::min(64, pow2_width(K)); }

}  // namespace

bool fits(int N, int K, int sources) {
    if (N > kMaxWidth || K > kMaxWidth) return false;
    const int KB = block_width(K);
    return pick_stages(pad16(N), KB, sources * blocks_of(K, KB)) != 0;
}

int run(Mode mode, Args a, cudaStream_t s, int* ctas) {
    if (ctas) *ctas = 0;
    if (a.rows == 0 || a.N == 0) return GNN_OK;
    const int64_t nt = (a.rows + 127) / 128;
    GNN_REQUIRE(nt <= 0x7fffffff - 2 * kMaxCtas, GNN_ESHAPE, "lin3: too many rows");
    a.n_tiles = (int)nt;
    a.NP = pad16(a.N);
    a.KB = block_width(std::max(a.K[0], a.K[1]));
    a.nkb[0] = blocks_of(a.K[0], a.KB);
    a.nkb[1] = blocks_of(a.K[1], a.KB);
    a.stages = pick_stages(a.NP, a.KB, a.nkb[0] + a.nkb[1]);
    GNN_REQUIRE(a.stages > 0 && a.N <= kMaxWidth, GNN_EUNSUPPORTED, "lin3: shape %d x (%d + %d) does not fit", a.N,
                a.K[0], a.K[1]);
    // 16-byte accesses only where every row of every operand starts on a 16-byte boundary
    bool vec = a.N % 4 == 0 && aligned16(a.out) && a.ldo % 4 == 0;
    for (int i = 0; i < 2; ++i)
        if (a.K[i]) vec = vec && a.K[i] % 4 == 0 && a.lda[i] % 4 == 0 && aligned16(a.A[i]);
    vec = vec && (!a.add || (aligned16(a.add) && a.ldadd % 4 == 0));
    vec = vec && (!a.P || (aligned16(a.P) && aligned16(a.Q) && a.ldpq % 4 == 0));
    vec = vec && aligned16(a.g0) && aligned16(a.da);
    if (a.nsplit <= 0) a.nsplit = a.NP;
    const uint32_t smem = lin_smem(a.NP, a.KB, a.nkb[0] + a.nkb[1], a.stages).total;
    const int grid = (int)std::min<int64_t>(nt, std::min(kMaxCtas, fused::host::num_sms()));
    if (ctas) *ctas = grid;
    int rc = GNN_OK;
    auto launch = [&](auto mode_c, auto ops_c, const char* name) {
        constexpr int M = decltype(mode_c)::value, O = decltype(ops_c)::value;
        auto kern = vec ? k_lin3<M, O, true> : k_lin3<M, O, false>;
        if ((rc = set_smem(kern, smem))) return;
        ProfScope _ps(s, name);
        kern<<<grid, kThreads, smem, s>>>(a);
    };
    constexpr Int<kOpsNone> none;
    constexpr Int<kOpsRow> one_row;
    constexpr Int<kOpsGather> gather;
    switch (mode) {
        case kElu:
            if (a.P) launch(Int<kElu>(), gather, "k_lin3_elu");
            else if (a.add) launch(Int<kElu>(), one_row, "k_lin3_elu");
            else launch(Int<kElu>(), none, "k_lin3_elu");
            break;
        case kLayerNorm:
            if (a.add) launch(Int<kLayerNorm>(), one_row, "k_lin3_ln");
            else launch(Int<kLayerNorm>(), none, "k_lin3_ln");
            break;
        case kLnAdjoint:
            if (a.da) launch(Int<kLnAdjoint>(), gather, "k_lin3_ln_adj");
            else launch(Int<kLnAdjoint>(), none, "k_lin3_ln_adj");
            break;
        case kEluAdjoint: launch(Int<kEluAdjoint>(), one_row, "k_lin3_elu_adj"); break;
        case kAdd:
            if (a.da) launch(Int<kAdd>(), gather, "k_lin3_add");
            else if (a.add) launch(Int<kAdd>(), one_row, "k_lin3_add");
            else launch(Int<kAdd>(), none, "k_lin3_add");
            break;
    }
    if (rc) return rc;
    GNN_LAUNCH_CHECK("k_lin3");
    return GNN_OK;
}

int wgrad(int64_t rows, const float* G, int64_t ldg, int N, const float* X, int64_t ldx, int K, bool db, float* part,
          cudaStream_t s, int* ctas) {
    *ctas = 0;
    if (rows == 0) return GNN_OK;
    GNN_REQUIRE(N <= kMaxWidth && K <= kMaxWidth, GNN_EUNSUPPORTED, "lin3: weight gradient %d x %d does not fit", N, K);
    WArgs a{};
    a.rows = rows;
    a.G = G; a.ldg = ldg; a.N = N;
    a.X = X; a.ldx = ldx; a.K = K;
    a.NP = pow2_width(N);
    const int KP = pow2_width(K);
    a.RT = (a.NP > 64 || KP > 64) ? 64 : 128;
    const int64_t nt = (rows + a.RT - 1) / a.RT;
    GNN_REQUIRE(nt <= 0x7fffffff - 2 * kMaxCtas, GNN_ESHAPE, "lin3: too many rows");
    a.n_tiles = (int)nt;
    a.db = db ? 1 : 0;
    a.vec_g = N % 4 == 0 && ldg % 4 == 0 && aligned16(G);
    a.vec_x = K % 4 == 0 && ldx % 4 == 0 && aligned16(X);
    a.stages = 4;
    while (wgrad_smem(a.NP, KP, a.RT, a.stages).total > kSmemMax) --a.stages;
    a.part = part;
    const uint32_t smem = wgrad_smem(a.NP, KP, a.RT, a.stages).total;
    const int grid = (int)std::min<int64_t>(nt, std::min(kMaxCtas, fused::host::num_sms()));
    *ctas = grid;
    int rc = GNN_OK;
    auto launch = [&](auto kern) {
        if ((rc = set_smem(kern, smem))) return;
        ProfScope _ps(s, "k_wgrad3");
        kern<<<grid, kWThreads, smem, s>>>(a);
    };
    if (KP == 16) launch(k_wgrad3<16>);
    else if (KP == 32) launch(k_wgrad3<32>);
    else if (KP == 64) launch(k_wgrad3<64>);
    else launch(k_wgrad3<128>);
    if (rc) return rc;
    GNN_LAUNCH_CHECK("k_wgrad3");
    return GNN_OK;
}

bool chain_fits(int N, int K) { return N <= 64 && K <= 64; }

int chain(int64_t rows, const float* G, int N, const float* H, int K, const float* W, float* out, bool db, float* part,
          cudaStream_t s, int* ctas) {
    *ctas = 0;
    if (rows == 0) return GNN_OK;
    GNN_REQUIRE(chain_fits(N, K), GNN_EUNSUPPORTED, "lin3: chain %d x %d does not fit", N, K);
    CArgs a{};
    a.rows = rows;
    const int64_t nt = (rows + 127) / 128;
    GNN_REQUIRE(nt <= 0x7fffffff - 2 * kMaxCtas, GNN_ESHAPE, "lin3: too many rows");
    a.n_tiles = (int)nt;
    a.G = G; a.N = N;
    a.H = H; a.K = K;
    a.W = W; a.out = out; a.db = db ? 1 : 0; a.part = part;
    const bool vec = N % 4 == 0 && K % 4 == 0 && aligned16(G) && aligned16(H) && aligned16(out);
    const int grid = (int)std::min<int64_t>(nt, std::min(kMaxCtas, fused::host::num_sms()));
    *ctas = grid;
    int rc = GNN_OK;
    auto launch = [&](auto nw, auto kw) {
        constexpr int NW = decltype(nw)::value, KW = decltype(kw)::value;
        constexpr uint32_t smem = chain_smem<NW, KW>().total;
        static_assert(smem <= kSmemMax, "one block per SM");
        auto kern = vec ? k_chain3<NW, KW, true> : k_chain3<NW, KW, false>;
        if ((rc = set_smem(kern, smem))) return;
        ProfScope _ps(s, "k_chain3");
        kern<<<grid, kThreads, smem, s>>>(a);
    };
    auto with_k = [&](auto nw) {
        const int kw = pow2_width(K);
        if (kw == 16) launch(nw, Int<16>());
        else if (kw == 32) launch(nw, Int<32>());
        else launch(nw, Int<64>());
    };
    const int nw = pow2_width(N);
    if (nw == 16) with_k(Int<16>());
    else if (nw == 32) with_k(Int<32>());
    else with_k(Int<64>());
    if (rc) return rc;
    GNN_LAUNCH_CHECK("k_chain3");
    return GNN_OK;
}

int reduce(const Sum* sums, int n, cudaStream_t s) {
    RedArgs a{};
    int blocks = 0;
    auto flush = [&]() -> int {
        if (blocks == 0) return GNN_OK;
        a.first[a.n] = blocks;
        {
            ProfScope _ps(s, "k_reduce3");
            k_reduce3<<<blocks, 256, 0, s>>>(a);
        }
        a.n = blocks = 0;
        GNN_LAUNCH_CHECK("k_reduce3");
        return GNN_OK;
    };
    auto dest = [](const Sum& q) { return Dest{q.dst, q.ldd, q.N, q.K}; };
    int rc;
    for (int i = 0; i < n; ++i) {
        if (sums[i].nz == 0 || !sums[i].dst) continue;
        bool apart = a.n < kMaxReduce;
        for (int k = 0; k < a.n; ++k) apart = apart && !may_overlap(dest(a.s[k]), dest(sums[i]));
        if (!apart && (rc = flush())) return rc;
        a.s[a.n] = sums[i];
        a.first[a.n++] = blocks;
        blocks += (sums[i].N * sums[i].K + 31) / 32;
    }
    return flush();
}

}  // namespace lin3
}  // namespace gnn
