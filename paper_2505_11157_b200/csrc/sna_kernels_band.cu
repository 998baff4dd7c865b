// Band kernels (sm_100a, mma.sync): the windows of Eq. (s2_attention_discrete_detailed) that are too narrow for the
// 128-row tiles of the dense kernels.  Every contraction runs on FP16 tensor-core instructions with fp32-level accuracy:
// operands are scaled by powers of two and split into two FP16 numbers, x = hi + lo with 22 significant bits; a product is the
// three m16n8k16 terms lo*hi + hi*lo + hi*hi summed in fp32 (the missing lo*lo is 2^-22 of the product).  Against one TF32 term
// plus one BF16 term for both corrections this takes 3/4 of the tensor time (1/2 of the three TF32 terms that scores need), half
// the registers for the tile's own operands, and the error falls from 7e-6 to 5e-7.
//
// Work decomposition: a warp owns a tile of 16 points (8 consecutive longitudes on each of 2 adjacent rings) and walks the
// host-built column stream of that ring pair, 16 partner points ("columns") per chunk (sna_plan.hpp).  The 16 partner points are
// staged by cp.async into a warp-private, two-stage shared-memory ring while the previous chunk is consumed, and split in
// registers, where they are the B operands of the scores and, transposed by movmatrix, of the weighted sums.  Warps do not
// synchronise with each other, except at the end of a stream that is long for its launch: the warps of a block share it.
//
// What bounds them (128x256, cutoff 4 rings, C = 32): per chunk of 16 columns a forward warp issues 362 instructions and moves 110
// wavefronts through the SM's shared-memory pipe (cp.async writes 44, row reads 38, transpositions 16, the rest global), so with
// 16 warps per SM that pipe is busy 68 % of the time, issue slots 58 %, tensor cores 30 %; DRAM and L2 are below 20 %.  Measures
// that took instructions or wavefronts out (us forward / dq / dk+dv, N = 16, whole streams): scales from the first chunk instead of
// a maximum per chunk 368/459/559 -> 359/414/481; x - h by one mixed-precision multiply-add, and no scaling of data that needs
// none (given up again for the range that it costs, see StreamScale) -> 348/397/466; movmatrix instead of writing the split rows back for ldmatrix -> 327/388/455 and, with pieces in an order
// without bank conflicts, C = 64, N = 8 from 432/472/549 to 334/369/445.
//
// Fragment conventions (g = lane / 4, t = lane % 4): a thread holds CP/4 channels of a point (Own::channel).  As an A operand
// they belong to tile rows g and g+8, as a B operand to column g.  The MMA's k indexes 2t, 2t+1, 2t+8, 2t+9 of k-step ks are its
// own channels 4*ks .. +3 (the same permutation on both operands, so the contraction is exact).  The accumulators of the weighted
// sums, too, hold a thread's own channels: 2i and 2i+1 in fragment i.
//
// Forward: Eq. (s2_attention_discrete_detailed).  Backward: App. B.4.
#include "sna_kernels.cuh"
#include "sna_plan.hpp"

#include <cuda_fp16.h>

#include <cstdint>
#include <type_traits>
#include <utility>

namespace sna {
namespace {

constexpr int WARPS = 4;
constexpr int THREADS = WARPS * 32;
constexpr float LOG2E = 1.4426950408889634f;
constexpr float LN2 = 0.6931471805599453f;
constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// packed fp32 pairs: one instruction for two values (the kernels are bound by issue slots as much as by the tensor pipe)
__device__ __forceinline__ uint64_t pack2(float a, float b) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) { uint64_t d; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c)); return d; }
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) { uint64_t d; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) { uint64_t d; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; }
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) { uint64_t d; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; }
__device__ __forceinline__ uint64_t both(float a) { return pack2(a, a); }
__device__ __forceinline__ void acc2(float& a, float& b, float x, float y) { unpack2(add2(pack2(a, b), pack2(x, y)), a, b); }

// ---------------------------------------------------------------------------------------------------------
// Scales, all powers of two
// ---------------------------------------------------------------------------------------------------------
constexpr int TOP = 14;              // exponent of the largest element of a scaled tile row
// exponent bits of a magnitude, not below 2^-100 (zero: of 1)
__device__ __forceinline__ uint32_t exponent_bits(float amax) {
    return amax == 0.f ? 127u << 23 : max(__float_as_uint(amax) & 0x7f800000u, (uint32_t)(127 - 100) << 23);
}
__device__ __forceinline__ float pow2_to(int target, uint32_t ebits) { return __uint_as_float(((uint32_t)(254 + target) << 23) - ebits); }   // 2^(target - e)
__device__ __forceinline__ float pow2_back(int target, uint32_t ebits) { return __uint_as_float(ebits - ((uint32_t)target << 23)); }        // 2^(e - target)

// Scale of a warp's streamed rows of one array: taken from the first chunk that is not all zero, whose largest element it brings to
// [2^11, 2^12).  A split element is then held to 2^-23 of itself or to 2^-25 in scaled units (the floor), which is 2^-36 of that
// largest one, and FP16 holds elements 16 times as large.  (Where that much is not needed, `plain` - for scores, in the backward pass in
// reduced precision - the scale stays 1 and the scaling is skipped if the largest element is in [2^-1, 2^8).)  Two things can go wrong.  Larger rows overflow to
// infinities, which the sums cannot hide.  And sums of which all terms are far below the largest element (a small channel beside a
// large one, small points beside a large one that is in the window of another row of the tile) may feel the floor: each kernel
// compares its sums with it at the end.  Where they overflowed, or one is so small that the floor could be 2^-17 of it and such
// elements are there, the warp computes its part of the tile again in fp32 (dots_fp32, sums_fp32), which takes four times as long.
// What the scaling and the checks cost (128x256, cutoff 4 rings, C = 32, N = 16, us forward / dq / dk+dv): 333/362/447 -> 349/370/472.
// A second pass with scales from all rows, for overflows, cost as much again in registers.
struct StreamScale {
    float scale = 1.f, inv = 1.f;
    bool known = false;
    // amax: this thread's largest magnitude (called by the whole warp)
    __device__ __forceinline__ void set(float amax, bool plain) {
        const uint32_t w = __reduce_max_sync(FULL, __float_as_uint(amax));
        if (w == 0) return;
        const uint32_t eb = exponent_bits(__uint_as_float(w));
        known = true;
        const bool keep = plain && eb >= (126u << 23) && eb < (135u << 23);
        scale = keep ? 1.f : pow2_to(11, eb);
        inv = keep ? 1.f : pow2_back(11, eb);
    }
};

// Scale of a warp's weights whose size is not known beforehand: it changes only when a weight above 2^15 appears (and for the first
// one); then the largest is brought to about 2^11, and growth by 2^4 fits without another change.  A first weight may be far
// below later ones, and the scale multiplies those before it is corrected: it is bounded, by 2^(11 + 72), so that p (t - D), whose
// t and D are below 2^37 in the units of the tensor cores' operands, stays finite.  Weights so small that the bound leaves them
// below FP16's range are below 2^-97 of what a weight of probability 1 would be.
struct WeightScale {
    float scale = 1.f, limit = 0.f;
    // amax: this thread's largest scaled magnitude (called by the whole warp).  Returns the factor for the sums collected so
    // far and for the weights at hand.
    __device__ __forceinline__ float update(float amax) {
        const uint32_t w = __reduce_max_sync(FULL, __float_as_uint(amax));
        if (!(__uint_as_float(w) > limit)) return 1.f;
        const float f = pow2_to(11, max(w & 0x7f800000u, (uint32_t)(127 - 72) << 23));
        scale *= f;
        limit = 32768.f;
        return f;
    }
};

__device__ __forceinline__ uint32_t h2_bits(__half2 h) { return *reinterpret_cast<uint32_t*>(&h); }
// two fp32 values as an FP16 pair (hi) and the FP16 pair of what is left (lo)
__device__ __forceinline__ void split2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
    const __half2 h = __floats2half2_rn(x0, x1);
    // x - h, exact: mixed-precision multiply-adds by -1 read the FP16 halves as they are
    float r0, r1;
    asm("fma.rn.f32.f16 %0, %1, %2, %3;" : "=f"(r0) : "h"(__half_as_ushort(__low2half(h))), "h"((uint16_t)0xbc00), "f"(x0));
    asm("fma.rn.f32.f16 %0, %1, %2, %3;" : "=f"(r1) : "h"(__half_as_ushort(__high2half(h))), "h"((uint16_t)0xbc00), "f"(x1));
    hi = h2_bits(h);
    lo = h2_bits(__floats2half2_rn(r0, r1));
}

__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_zero(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t bytes) {      // the rest of the 16 bytes is zero-filled
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) { asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src) { asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ uint32_t s32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---------------------------------------------------------------------------------------------------------
// Warp-private staging of a chunk's 16 partner points (two arrays: k and v rows, or q and dout rows) as fp32.  A thread owns whole
// 16-byte pieces, in an order, and rows have a pitch, for which the eight threads that a 16-byte access serves at a time (two
// rows of a fragment) reach all banks.
// ---------------------------------------------------------------------------------------------------------
template <int CP>
struct Own {
    static constexpr int N = CP / 4;
    // the i-th channel (i a multiple of 4) of the threads with index t in their group
    __device__ static constexpr int channel(int t, int i) { return CP == 64 ? i / 8 * 32 + t * 8 + i % 8 : t * N + i; }
};
template <int CP>
struct Stage {
    static constexpr int PITCH = CP == 16 ? 64 : CP * 4 + 16, A = 0, B = 16 * PITCH, M0 = 2 * 16 * PITCH, M1 = M0 + 64, BYTES = M1 + 64;
    // M0: forward stream: log2 omega of the partner's ring; transposed stream: lse of the partner.  M1: transposed: D of the partner
};
template <int CP>
constexpr size_t smem_bytes() { return (size_t)Stage<CP>::BYTES * 2 * WARPS; }

// Walks the column stream of one ring group, copying one or two chunks ahead into a two-stage ring.  Lane l copies column l % 16
// (both half-warps compute the same indexes, which keeps the code free of divergent branches); the rows are copied in 16-byte
// pieces.  The pipeline runs ahead without branches: past the end of a group's chunks it stages the next group's first ones (the
// host pads the last).
template <int CP, bool TRANSPOSED, bool PAD>
struct StreamWalker {
    using S = Stage<CP>;
    static constexpr int PIECES = CP / 4;            // 16-byte pieces per row
    static constexpr int ROWS_PER_PASS = 32 / PIECES;
    const int4* col;          // this lane's column of chunk 0
    const uint32_t* mask;
    const float *a, *b, *lse, *D;      // at the slice; a and b advanced to this lane's piece
    uint32_t smem;            // of stage 0
    uint32_t dst, meta;       // where in a stage this lane's first piece and its column's statistics go
    int first, period, stride, lane, C;

    // flat index of the partner point in its slice
    __device__ __forceinline__ uint32_t index(const int4& e) const {
        int u = e.y;
        if (e.x >= 0) {   // relative to the tile's first point, wrapped around the ring
            u += first;
            if (u < 0) u += period;
            if (u >= period) u -= period;
            if (u >= period) u -= period;
        }
        return (uint32_t)(e.x & 0x7fffffff) + (uint32_t)(u * stride);
    }
    __device__ __forceinline__ size_t column(int i) const { return index(__ldg(col - (lane & 15) + i)); }
    __device__ __forceinline__ void issue(uint32_t st, const int4& e) const {
        const uint32_t idx = index(e);
        const uint32_t elem = idx * C;      // < 2^32: checked on the host
        const uint32_t to = st + dst;
#pragma unroll
        for (int j = 0; j < CP / 8; ++j) {
            const uint32_t off = __shfl_sync(FULL, elem, lane / PIECES + j * ROWS_PER_PASS);
            if constexpr (PAD) {
                const uint32_t bytes = 4 * (lane % PIECES) < C ? 16 : 0;
                cp_async16(to + S::A + j * ROWS_PER_PASS * S::PITCH, a + (bytes ? off : 0), bytes);
                cp_async16(to + S::B + j * ROWS_PER_PASS * S::PITCH, b + (bytes ? off : 0), bytes);
            } else {
                cp_async16(to + S::A + j * ROWS_PER_PASS * S::PITCH, a + off);
                cp_async16(to + S::B + j * ROWS_PER_PASS * S::PITCH, b + off);
            }
        }
        if (TRANSPOSED) {
            cp_async4(st + meta + S::M0, lse + idx);
            cp_async4(st + meta + S::M1, D + idx);
        } else {
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(st + meta + S::M0), "r"(e.z) : "memory");
        }
    }

    // AHEAD 1: chunk c+1 is copied during chunk c.  AHEAD 2: chunk c+2 is, from when body(stage, mask, release) calls release(),
    // having read all that it needs from the stage.
    template <int AHEAD, typename Body>
    __device__ __forceinline__ void run(int nchunks, Body&& body) const {
        if (nchunks <= 0) return;
        const int4* pc = col;
        const uint32_t* pm = mask;
        uint32_t st = smem, other = smem + S::BYTES;
        issue(st, __ldg(pc));
        cp_async_commit();
        if constexpr (AHEAD == 2) {
            issue(other, __ldg(pc += BAND_CHUNK));
            cp_async_commit();
        }
        int4 e = __ldg(pc += BAND_CHUNK);
        uint32_t m = __ldg(pm);
        auto next = [&](uint32_t stage) {
            issue(stage, e);
            cp_async_commit();
            e = __ldg(pc += BAND_CHUNK);
        };
#pragma unroll 1
        for (int c = nchunks; c > 0; --c) {
            if constexpr (AHEAD == 1) next(other);
            const uint32_t now = m;
            m = __ldg(pm += 32);
            cp_async_wait<1>();
            __syncwarp();
            body(st, now, [&] {
                if constexpr (AHEAD == 2) {
                    __syncwarp();
                    next(st);
                }
            });
            if constexpr (AHEAD == 1) __syncwarp();   // everyone is done with this stage before the next iteration refills it
            const uint32_t swap = st; st = other; other = swap;
        }
        cp_async_wait<0>();
        __syncwarp();       // the stages are free for other use
    }
};
template <int CP, bool TRANSPOSED, bool PAD>
__device__ __forceinline__ StreamWalker<CP, TRANSPOSED, PAD> make_walker(unsigned char* smem_raw, const DevBand& s, int chunk0, int first, int period, int stride, int C,
                                                                     const float* a, const float* b, const float* lse, const float* D) {
    const int lane = threadIdx.x & 31, piece = lane % (CP / 4) * 4;
    const int pc = PAD && piece >= C ? 0 : piece;      // (lanes without channels copy nothing, from a valid address)
    return StreamWalker<CP, TRANSPOSED, PAD>{s.columns + (size_t)chunk0 * BAND_CHUNK + (lane & 15), s.masks + (size_t)chunk0 * 32 + lane, a + pc, b + pc, lse, D,
                                             s32(smem_raw) + (threadIdx.x >> 5) * 2 * Stage<CP>::BYTES,
                                             (lane / (CP / 4)) * (uint32_t)Stage<CP>::PITCH + piece * 4, (lane & 15) * 4u, first, period, stride, lane, C};
}

// A thread's share of a chunk's 16 points is its own channels of columns g and 8 + g.  It is read and split in parts, which bounds
// the registers that it takes.
template <int CP>
struct RawRows {
    static constexpr int PARTS = CP == 64 ? 2 : 1, N = CP / 4 / PARTS;
    float x[2][N];
    // rows: address of this thread's first channel of row g
    __device__ __forceinline__ void load(uint32_t rows, int part) {
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < N; i += 4)
                asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(x[j][i]), "=f"(x[j][i + 1]), "=f"(x[j][i + 2]), "=f"(x[j][i + 3])
                             : "r"(rows + 8 * j * Stage<CP>::PITCH + Own<CP>::channel(0, part * N + i) * 4) : "memory");
    }
    __device__ __forceinline__ float max_abs() const {
        float m = 0.f;
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < N; i += 2) m = fmaxf(fmaxf(m, fabsf(x[j][i])), fabsf(x[j][i + 1]));
        return m;
    }
};
// ... scaled and split: as it is the B operand of the scores (channel pairs of one point), and transposed, 8 points by 8 channels
// at a time, that of the weighted sums (point pairs of one channel).
template <int CP, bool LP>
struct SplitRows {
    static constexpr int R = CP / 8;
    uint32_t hi[2][R], lo[LP ? 1 : 2][R];
    // ALWAYS: the scale is hardly ever 1
    template <bool ALWAYS = !LP>
    __device__ __forceinline__ void load(uint32_t rows, float sc) {
        using Raw = RawRows<CP>;
#pragma unroll
        for (int part = 0; part < Raw::PARTS; ++part) {
            Raw r;
            r.load(rows, part);
            if (ALWAYS || sc != 1.f) {
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int i = 0; i < Raw::N; i += 2) unpack2(mul2(pack2(r.x[j][i], r.x[j][i + 1]), both(sc)), r.x[j][i], r.x[j][i + 1]);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int i = 0; i < Raw::N; i += 2) {
                    const int at = (part * Raw::N + i) / 2;
                    if constexpr (LP) hi[j][at] = h2_bits(__floats2half2_rn(r.x[j][i], r.x[j][i + 1]));
                    else split2(r.x[j][i], r.x[j][i + 1], hi[j][at], lo[j][at]);
                }
        }
    }
};
// The scales of the two streamed arrays, and this lane's place in a stage.
template <int CP>
struct StreamScales {
    StreamScale a, b;
    uint32_t own;      // of RawRows::load
    int g, t;
    __device__ __forceinline__ StreamScales() {
        const int lane = threadIdx.x & 31;
        g = lane >> 2; t = lane & 3;
        own = g * Stage<CP>::PITCH + Own<CP>::channel(t, 0) * 4;
    }
    __device__ __forceinline__ static float max_abs(uint32_t rows) {
        float m = 0.f;
#pragma unroll
        for (int part = 0; part < RawRows<CP>::PARTS; ++part) {
            RawRows<CP> x;
            x.load(rows, part);
            m = fmaxf(m, x.max_abs());
        }
        return m;
    }
    __device__ __forceinline__ bool known() const { return a.known && b.known; }
    __device__ __forceinline__ void look(uint32_t st, bool plain_a, bool plain_b) {
        if (!a.known) a.set(max_abs(st + own + Stage<CP>::A), plain_a);
        if (!b.known) b.set(max_abs(st + own + Stage<CP>::B), plain_b);
    }
};
// After a pass: whether some thread's sums overflowed (`total` is not finite if one of them is not).
__device__ __forceinline__ bool overflowed(float total) { return __any_sync(FULL, !(fabsf(total) < INFINITY)); }
// Whether the floors of a tile row's and a streamed row's split operands (both below 2^16) could move a score by more than 2^-17 (log2
// domain; 2^-11 in reduced precision).  unit: a score's value per product of scaled operands.
template <bool LP>
__device__ __forceinline__ bool scores_lost(float unit, int C) { return unit * (float)C > (LP ? 0.15f : 0.0024f); }
constexpr float REDUCED = 1.f / 256.f;      // single products: sums may be that much smaller before the floor shows beside their 10 bits

// Persistent A operand: the tile's rows g and g+8 from two points (pointers at channel 0), scaled by `mul` and by powers of
// two, one per row or one for the warp's 16 rows (COMMON); back0, back1 undo the latter.
template <int CP, bool LP>
struct TileOperand {
    static constexpr int CPT = CP / 4, KS = CP / 16;
    uint32_t hi[KS][4], lo[LP ? 1 : KS][4];
    float back0, back1;
    template <bool COMMON>
    __device__ __forceinline__ void load(const float* p0, const float* p1, float mul, int C, int t) {
        float a[CPT], b[CPT];
        float m0 = 0.f, m1 = 0.f;
#pragma unroll
        for (int i = 0; i < CPT; i += 4) {
            const int c = Own<CP>::channel(t, i);
            float4 u = make_float4(0.f, 0.f, 0.f, 0.f), w = u;
            if (c < C) { u = __ldg(reinterpret_cast<const float4*>(p0 + c)); w = __ldg(reinterpret_cast<const float4*>(p1 + c)); }
            a[i] = u.x * mul; a[i + 1] = u.y * mul; a[i + 2] = u.z * mul; a[i + 3] = u.w * mul;
            b[i] = w.x * mul; b[i + 1] = w.y * mul; b[i + 2] = w.z * mul; b[i + 3] = w.w * mul;
        }
#pragma unroll
        for (int i = 0; i < CPT; ++i) { m0 = fmaxf(m0, fabsf(a[i])); m1 = fmaxf(m1, fabsf(b[i])); }
        uint32_t e0, e1;
        if (COMMON) {
            e0 = e1 = exponent_bits(__uint_as_float(__reduce_max_sync(FULL, __float_as_uint(fmaxf(m0, m1)))));
        } else {
            m0 = fmaxf(m0, __shfl_xor_sync(FULL, m0, 1)); m1 = fmaxf(m1, __shfl_xor_sync(FULL, m1, 1));
            m0 = fmaxf(m0, __shfl_xor_sync(FULL, m0, 2)); m1 = fmaxf(m1, __shfl_xor_sync(FULL, m1, 2));
            e0 = exponent_bits(m0); e1 = exponent_bits(m1);
        }
        const float s0 = pow2_to(TOP, e0), s1 = pow2_to(TOP, e1);
        back0 = pow2_back(TOP, e0); back1 = pow2_back(TOP, e1);
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                uint32_t l0, l1;
                split2(a[4 * ks + 2 * j] * s0, a[4 * ks + 2 * j + 1] * s0, hi[ks][2 * j], l0);
                split2(b[4 * ks + 2 * j] * s1, b[4 * ks + 2 * j + 1] * s1, hi[ks][2 * j + 1], l1);
                if constexpr (!LP) { lo[ks][2 * j] = l0; lo[ks][2 * j + 1] = l1; }
            }
    }
};

// d[j] = tile rows . points of 8-column tile j (scaled as the operands are).  Corrections first, main terms last, into
// fragments that start at zero: the tensor core truncates when it accumulates, so chains stay short.
template <int CP, bool LP>
__device__ __forceinline__ void rows_dot_points(float (&d)[2][4], const TileOperand<CP, LP>& A, const SplitRows<CP, LP>& B) {
    constexpr int KS = CP / 16;
    if constexpr (!LP) {
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                if (ks == 0) mma_zero(d[j], A.lo[ks], B.hi[j][2 * ks], B.hi[j][2 * ks + 1]);
                else mma(d[j], A.lo[ks], B.hi[j][2 * ks], B.hi[j][2 * ks + 1]);
                mma(d[j], A.hi[ks], B.lo[j][2 * ks], B.lo[j][2 * ks + 1]);
            }
    }
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (LP && ks == 0) mma_zero(d[j], A.hi[ks], B.hi[j][2 * ks], B.hi[j][2 * ks + 1]);
            else mma(d[j], A.hi[ks], B.hi[j][2 * ks], B.hi[j][2 * ks + 1]);
        }
}

// With single products an overflowed point can give scores of -infinity, which would vanish as weights: keep them in `bad` as NaN.
template <bool LP>
__device__ __forceinline__ void note_overflow(uint64_t& bad, const float (&s)[2][4]) {
    if constexpr (LP) {
#pragma unroll
        for (int j = 0; j < 2; ++j) bad = fma2(pack2(s[j][0], s[j][1]), 0, fma2(pack2(s[j][2], s[j][3]), 0, bad));
    }
}
__device__ __forceinline__ float sum2(uint64_t x) { float a, b; unpack2(x, a, b); return a + b; }

// The weights of a chunk (score layout, already scaled) as A operand of the weighted sums.
template <bool LP>
struct Weights {
    uint32_t hi[4], lo[4];
    __device__ __forceinline__ void set(const float (&w)[2][4]) {
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                if constexpr (LP) hi[2 * j + i] = h2_bits(__floats2half2_rn(w[j][2 * i], w[j][2 * i + 1]));
                else split2(w[j][2 * i], w[j][2 * i + 1], hi[2 * j + i], lo[2 * j + i]);
            }
    }
};
__device__ __forceinline__ uint32_t transpose8x8(uint32_t x) {
    uint32_t y;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
// sum[i] += weights . points for the own channels 2i, 2i+1 (rows g: [0..1], rows g+8: [2..3])
template <int CP, bool LP>
__device__ __forceinline__ void weights_times_points(float (&sum)[CP / 8][4], const Weights<LP>& W, const SplitRows<CP, LP>& B) {
#pragma unroll
    for (int i = 0; i < CP / 8; ++i) {
        const uint32_t h0 = transpose8x8(B.hi[0][i]), h1 = transpose8x8(B.hi[1][i]);
        float p[4];
        if constexpr (LP) {
            mma_zero(p, W.hi, h0, h1);
        } else {
            const uint32_t l0 = transpose8x8(B.lo[0][i]), l1 = transpose8x8(B.lo[1][i]);
            mma_zero(p, W.lo, h0, h1);
            mma(p, W.hi, l0, l1);
            mma(p, W.hi, h0, h1);
        }
        acc2(sum[i][0], sum[i][1], p[0], p[1]);
        acc2(sum[i][2], sum[i][3], p[2], p[3]);
    }
}
template <int N>
__device__ __forceinline__ float total(const float (&x)[N][4]) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) s += (x[i][0] + x[i][1]) + (x[i][2] + x[i][3]);
    return s;
}
template <int N>
__device__ __forceinline__ void clear(float (&x)[N][4]) {
#pragma unroll
    for (int i = 0; i < N; ++i) x[i][0] = x[i][1] = x[i][2] = x[i][3] = 0.f;
}
template <int N>
__device__ __forceinline__ void scale_rows(float (&x)[N][4], float f0, float f1) {
#pragma unroll
    for (int i = 0; i < N; ++i) { x[i][0] *= f0; x[i][1] *= f0; x[i][2] *= f1; x[i][3] *= f1; }
}
__device__ __forceinline__ void apply_mask(float (&x)[2][4], uint32_t mask, float other) {
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) x[j][i] = (mask & (1u << (4 * j + i))) ? x[j][i] : other;
}
// running maxima of the magnitudes in the thread's two rows
__device__ __forceinline__ void row_max(float& m0, float& m1, const float (&x)[2][4]) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(m0) : "f"(x[j][0]), "f"(x[j][1]));
        asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(m1) : "f"(x[j][2]), "f"(x[j][3]));
    }
}
__device__ __forceinline__ float group_max(float x) {
    x = fmaxf(x, __shfl_xor_sync(FULL, x, 1));
    return fmaxf(x, __shfl_xor_sync(FULL, x, 2));
}

// ---------------------------------------------------------------------------------------------------------
// What follows a pass whose sums the FP16 parts may not hold
// ---------------------------------------------------------------------------------------------------------
__device__ __forceinline__ float4 lds128(uint32_t addr) {
    float4 x;
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(addr) : "memory");
    return x;
}
__device__ __forceinline__ float dot4(const float4& a, const float4& b, float c) { return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, c)))); }
// d = tile rows g and g+8 (at p0 and p1) . the thread's four columns of the staged rows, in the layout of rows_dot_points
template <int CP>
__device__ __forceinline__ void dots_fp32(float (&d)[2][4], const float* p0, const float* p1, uint32_t rows, int C, int t) {
#pragma unroll
    for (int j = 0; j < 2; ++j) d[j][0] = d[j][1] = d[j][2] = d[j][3] = 0.f;
#pragma unroll 1
    for (int c = 0; c < C; c += 4) {
        const float4 a = __ldg(reinterpret_cast<const float4*>(p0 + c)), b = __ldg(reinterpret_cast<const float4*>(p1 + c));
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float4 x = lds128(rows + (8 * j + 2 * t + i) * Stage<CP>::PITCH + 4 * c);
                d[j][i] = dot4(a, x, d[j][i]);
                d[j][2 + i] = dot4(b, x, d[j][2 + i]);
            }
    }
}
// sum += weights . staged rows, as weights_times_points; points of weight zero (outside the window) do not enter, whatever they hold
template <int CP>
__device__ __forceinline__ void sums_fp32(float (&sum)[CP / 8][4], const float (&w)[2][4], uint32_t rows, int t) {
#pragma unroll 1
    for (int o = 0; o < 4; ++o)      // the columns of the group's o-th thread
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float w0 = __shfl_sync(FULL, w[j][i], o, 4), w1 = __shfl_sync(FULL, w[j][2 + i], o, 4);
#pragma unroll
                for (int m = 0; m < CP / 16; ++m) {
                    const float4 x = lds128(rows + (8 * j + 2 * o + i) * Stage<CP>::PITCH + 4 * Own<CP>::channel(t, 4 * m));
                    if (w0 != 0.f) {
                        sum[2 * m][0] = fmaf(w0, x.x, sum[2 * m][0]); sum[2 * m][1] = fmaf(w0, x.y, sum[2 * m][1]);
                        sum[2 * m + 1][0] = fmaf(w0, x.z, sum[2 * m + 1][0]); sum[2 * m + 1][1] = fmaf(w0, x.w, sum[2 * m + 1][1]);
                    }
                    if (w1 != 0.f) {
                        sum[2 * m][2] = fmaf(w1, x.x, sum[2 * m][2]); sum[2 * m][3] = fmaf(w1, x.y, sum[2 * m][3]);
                        sum[2 * m + 1][2] = fmaf(w1, x.z, sum[2 * m + 1][2]); sum[2 * m + 1][3] = fmaf(w1, x.w, sum[2 * m + 1][3]);
                    }
                }
            }
}
// Whether sums (small0, small1: of the thread's channels, in its two rows) are small because their terms are too small for the floor, and
// not because terms cancel.  The streamed rows (`rows`, at the slice) tell: it is so if a row has small sums in a quarter of its
// channels and some element of one of these is below `tiny`, or if one in 64 elements of such a channel is, which are fewer than
// the points of one row's window.  (A single small element in a channel and at a point that are not small otherwise is left
// alone.)  Looking at a channel takes about 2 us, computing the tile again a hundred.
template <int CP, typename Walker>
__device__ __forceinline__ bool channels_lost(const Walker walker, int nchunks, const float* rows, float tiny, uint32_t small0, uint32_t small1, int C, int t) {
    constexpr int QUADS = CP / 16;        // of channels per thread
    int in_row = __popc(small0) | __popc(small1) << 16;
    in_row += __shfl_xor_sync(FULL, in_row, 1);
    in_row += __shfl_xor_sync(FULL, in_row, 2);
    const bool many = __any_sync(FULL, max(in_row & 0xffff, in_row >> 16) * 4 >= C);
#pragma unroll 1
    for (int o = 0; o < 4 * QUADS; ++o) {
        const int owner = o / QUADS, quad = o % QUADS;
        const uint32_t which = __reduce_or_sync(FULL, t == owner ? (small0 | small1) >> 4 * quad & 15u : 0u);
        if (which == 0) continue;
        const float* at = rows + Own<CP>::channel(owner, 4 * quad);
        int tiny_ones[4] = {0, 0, 0, 0};
#pragma unroll 4
        for (int col = walker.lane; col < nchunks * BAND_CHUNK; col += 32) {
            const float4 x = __ldg(reinterpret_cast<const float4*>(at + walker.column(col) * C));
            const float y[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) tiny_ones[i] += y[i] != 0.f && fabsf(y[i]) < tiny;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int all = __reduce_add_sync(FULL, tiny_ones[i]);
            if ((which >> i & 1u) != 0 && all > 0 && (many || all * 64LL >= nchunks * BAND_CHUNK)) return true;
        }
    }
    return false;
}
// ... of sums below the row's limit: 0.3 % of the tiles of normally distributed data have one.
template <int CP, typename Walker>
__device__ __forceinline__ bool sums_lost(const float (&sum)[CP / 8][4], float limit0, float limit1, const Walker& walker, int nchunks, const float* rows, float tiny, int C, int t) {
    float least0 = INFINITY, least1 = INFINITY;
#pragma unroll
    for (int m = 0; m < CP / 16; ++m)
        if (Own<CP>::channel(t, 4 * m) < C) {
#pragma unroll
            for (int i = 2 * m; i < 2 * m + 2; ++i) {
                asm("min.abs.f32 %0, %0, %1, %2;" : "+f"(least0) : "f"(sum[i][0]), "f"(sum[i][1]));
                asm("min.abs.f32 %0, %0, %1, %2;" : "+f"(least1) : "f"(sum[i][2]), "f"(sum[i][3]));
            }
        }
    if (!__any_sync(FULL, least0 < limit0 || least1 < limit1)) return false;
    uint32_t small0 = 0, small1 = 0;
#pragma unroll
    for (int i = 0; i < CP / 4; ++i)
        if (Own<CP>::channel(t, i & ~3) < C) {
            if (fabsf(sum[i / 2][i % 2]) < limit0) small0 |= 1u << i;
            if (fabsf(sum[i / 2][2 + i % 2]) < limit1) small1 |= 1u << i;
        }
    return channels_lost<CP>(walker, nchunks, rows, tiny, small0, small1, C, t);
}
__device__ __forceinline__ uint64_t lds64(uint32_t addr) {
    uint64_t x;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(x) : "r"(addr) : "memory");
    return x;
}

// four channels of a point, from fragments 2m and 2m+1 of a sum (row 0: the point of tile row g, 1: g+8)
template <int N>
__device__ __forceinline__ float4 quad(const float (&x)[N][4], int m, int row, float f) {
    return make_float4(x[2 * m][2 * row] * f, x[2 * m][2 * row + 1] * f, x[2 * m + 1][2 * row] * f, x[2 * m + 1][2 * row + 1] * f);
}
// p: the point's channels
template <int CP>
__device__ __forceinline__ float4 load_quad(const float* p, int m, int C, int t) {
    const int c = Own<CP>::channel(t, 4 * m);
    return c < C ? *reinterpret_cast<const float4*>(p + c) : make_float4(0.f, 0.f, 0.f, 0.f);
}
template <int CP>
__device__ __forceinline__ void store_quad(float* p, int m, int C, int t, const float4& x) {
    const int c = Own<CP>::channel(t, 4 * m);
    if (c < C) *reinterpret_cast<float4*>(p + c) = x;
}
// The same four channels in channels-first planes of P points: eight threads fill 32 bytes of each plane.  cf: the tensor; pt: the
// point, counted over all slices; n: its slice.
template <int CP>
__device__ __forceinline__ void store_quad_cf(float* cf, size_t pt, int n, size_t P, int m, int C, int t, const float4& x) {
    const int c = Own<CP>::channel(t, 4 * m);
    if (c >= C) return;
    float* p = cf + (size_t)n * (C - 1) * P + pt + c * P;
    p[0] = x.x; p[P] = x.y; p[2 * P] = x.z; p[3 * P] = x.w;
}
__device__ __forceinline__ float4 operator+(const float4& a, const float4& b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

// The stream a launch walks.
struct BandView {
    DevBand s;
    const int32_t* dense_ptr;     // != null: rings with windows on the dense kernels start from (forward) or add to their partial result
    int tiles, N;                 // longitude tiles per ring group, slices
    int shared;                   // the first tasks, one per block: its warps share the tile's stream
    int total;                    // tasks
    // whether one of the two rings from h0 on has windows on the dense kernels
    __device__ __forceinline__ bool has_dense(int h0, int nlat) const { return dense_ptr[min(h0 + 2, nlat)] > dense_ptr[h0]; }
};
// The band kernel is launched to start when the dense kernel before it leaves SMs idle (programmatic dependent launch).  Tiles with
// windows on the dense kernel wait here until that has finished and its results are visible; the others need nothing from it.
// There is always one that waits, so the band kernel never finishes first.
__device__ __forceinline__ void wait_for_dense() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// A warp's task: longitude tile, slice and ring group (heavy-first order), and its part of the tile's stream.
struct Task {
    int tile, n, group, warp;
    bool shared;                  // the same for all warps of a block
    __device__ __forceinline__ bool decode(const BandView& v) {
        warp = threadIdx.x >> 5;
        shared = blockIdx.x < (unsigned)v.shared;
        const int task = shared ? blockIdx.x : v.shared + (blockIdx.x - v.shared) * WARPS + warp;
        if (task >= v.total) return false;
        tile = task % v.tiles;
        const int rest = task / v.tiles;
        n = rest % v.N;
        group = v.s.order[rest / v.N];
        return true;
    }
    __device__ __forceinline__ void chunks(const BandView& v, int row, int& first, int& count) const {
        if (v.s.one_row) row = 0;
        first = v.s.chunk_ptr[row];
        count = v.s.chunk_ptr[row + 1] - first;
        if (shared) {
            const int skip = count * warp / WARPS;
            count = count * (warp + 1) / WARPS - skip;
            first += skip;
        }
    }
    __device__ __forceinline__ bool writes(int m) const { return !shared || m % WARPS == warp; }     // the m-th four channels of each thread
};
// Sums over the warps of a shared tile, through their staging memory: every warp puts its fragments, and after a barrier
// the one that writes a channel adds them up.
template <int CP>
struct Exchange {
    float* base;
    __device__ __forceinline__ Exchange(unsigned char* smem_raw) : base(reinterpret_cast<float*>(smem_raw) + (threadIdx.x & 31)) {}
    __device__ __forceinline__ float& at(int warp, int i) const { return base[warp * (2 * Stage<CP>::BYTES / 4) + i * 32]; }
    __device__ __forceinline__ void put(const float (&x)[CP / 8][4], int warp, int first, float f0, float f1) const {
#pragma unroll
        for (int nt = 0; nt < CP / 8; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i) at(warp, first + 4 * nt + i) = x[nt][i] * (i < 2 ? f0 : f1);
    }
    // f0, f1 [warp]: factors of the warps' rows g and g + 8
    __device__ __forceinline__ void add(float (&x)[CP / 8][4], const Task& task, int first, const float (&f0)[WARPS], const float (&f1)[WARPS]) const {
#pragma unroll
        for (int nt = 0; nt < CP / 8; ++nt)
            if (task.writes(nt / 2)) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    x[nt][i] = 0.f;
#pragma unroll
                    for (int w = 0; w < WARPS; ++w) x[nt][i] = fmaf(at(w, first + 4 * nt + i), i < 2 ? f0[w] : f1[w], x[nt][i]);
                }
            }
    }
    __device__ __forceinline__ void add(float (&x)[CP / 8][4], const Task& task, int first) const {
        const float one[WARPS] = {1.f, 1.f, 1.f, 1.f};
        add(x, task, first, one, one);
    }
};
static_assert(WARPS == 4, "the list of ones above");
// The two points of a thread's rows g and g + 8 of a tile (the same longitude on the two rings of the pair that starts at ring
// h0); indexes are clamped to existing points, ok0 / ok1 tell whether they exist.
struct TilePoints {
    bool ok0, ok1;
    int ha, hb;
    size_t pt0, pt1;
    __device__ __forceinline__ TilePoints(int n, int h0, int lon, int nlat, int nlon) {
        ok0 = lon < nlon && h0 < nlat;
        ok1 = ok0 && h0 + 1 < nlat;
        const int c = min(lon, nlon - 1);
        ha = min(h0, nlat - 1); hb = min(h0 + 1, nlat - 1);
        pt0 = (size_t)(n * nlat + ha) * nlon + c;
        pt1 = (size_t)(n * nlat + hb) * nlon + c;
    }
};

// ---------------------------------------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------------------------------------
// Softmax reference.  A row's weights are 2^(score - m).  m is set by the first chunk that has a valid column for the row so
// that the largest weight becomes 2^W_SET, and raised (back to that) only when a weight would exceed 2^W_MAX: no maximum has
// to be exchanged between the threads of a row in the common case, and the weights need no further scale for FP16.
constexpr float W_SET = 10.f, W_MAX = 15.f;
constexpr float W_UNIT = 1.f / 1024.f;       // 2^-W_SET: taken out of sums before their logarithm, which then rounds less

// Reference m and weight w = 2^(x - m) for a row's earlier columns, whose logarithm (natural) is lse: m is a whole number, so
// that no rounding separates the two.
__device__ __forceinline__ void seed(float lse, float& m, float& w) {
    const float whole = rintf(lse * LOG2E);
    m = whole - W_SET;
    w = ex2(fmaf(lse, LOG2E, -whole)) / W_UNIT;
}

// The softmax of the thread's two rows, over its columns.
struct Softmax {
    float m0, m1, top0, top1;          // top: scores (relative to m) up to this need no new reference
    uint64_t l0, l1;                   // two partial sums each
    // Starts a pass, with sums o (v unscaled): from the dense kernel's partial result of a row (normalised out and lse), one weight of
    // value 2^lse, if `seeded` and there is one.
    template <int CP>
    __device__ __forceinline__ void start(bool seeded, const BandView& view, const TilePoints& at, const float* out, const float* lse, float (&o)[CP / 8][4], int C, int t) {
        clear(o);
        m0 = m1 = 0.f; top0 = top1 = -INFINITY;
        l0 = l1 = 0;
        if (!seeded) return;
        if (view.dense_ptr[at.ha + 1] > view.dense_ptr[at.ha]) {
            float w;
            seed(lse[at.pt0], m0, w);
            top0 = W_MAX;
#pragma unroll
            for (int m = 0; m < CP / 16; ++m) {
                const float4 x = load_quad<CP>(out + at.pt0 * C, m, C, t);
                o[2 * m][0] = x.x * w; o[2 * m][1] = x.y * w; o[2 * m + 1][0] = x.z * w; o[2 * m + 1][1] = x.w * w;
            }
            if (t == 0) l0 = pack2(w, 0.f);
        }
        if (view.dense_ptr[at.hb + 1] > view.dense_ptr[at.hb]) {
            float w;
            seed(lse[at.pt1], m1, w);
            top1 = W_MAX;
#pragma unroll
            for (int m = 0; m < CP / 16; ++m) {
                const float4 x = load_quad<CP>(out + at.pt1 * C, m, C, t);
                o[2 * m][2] = x.x * w; o[2 * m][3] = x.y * w; o[2 * m + 1][2] = x.z * w; o[2 * m + 1][3] = x.w * w;
            }
            if (t == 0) l1 = pack2(w, 0.f);
        }
    }
    // s: a chunk's products in, its weights out.  f2: a score per product.
    template <int N>
    __device__ __forceinline__ void weights(float (&s)[2][4], float (&o)[N][4], uint64_t f2, const uint64_t (&bias2)[2], uint32_t mask) {
        const uint64_t m02 = both(m0), m12 = both(m1);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            unpack2(fma2(pack2(s[j][0], s[j][1]), f2, sub2(bias2[j], m02)), s[j][0], s[j][1]);
            unpack2(fma2(pack2(s[j][2], s[j][3]), f2, sub2(bias2[j], m12)), s[j][2], s[j][3]);
        }
        if (!(mask & BAND_ALL)) apply_mask(s, mask, -INFINITY);   // some tile row skips some column of this chunk
        float mx0 = fmaxf(fmaxf(s[0][0], s[0][1]), fmaxf(s[1][0], s[1][1])), mx1 = fmaxf(fmaxf(s[0][2], s[0][3]), fmaxf(s[1][2], s[1][3]));
        if (__any_sync(FULL, mx0 > top0 || mx1 > top1)) {
            mx0 = fmaxf(mx0, __shfl_xor_sync(FULL, mx0, 1)); mx1 = fmaxf(mx1, __shfl_xor_sync(FULL, mx1, 1));
            mx0 = fmaxf(mx0, __shfl_xor_sync(FULL, mx0, 2)); mx1 = fmaxf(mx1, __shfl_xor_sync(FULL, mx1, 2));
            const bool up0 = mx0 > top0, up1 = mx1 > top1;
            const float d0 = up0 ? mx0 - W_SET : 0.f, d1 = up1 ? mx1 - W_SET : 0.f;
            // (a row without a reference has collected nothing: any finite factor will do)
            const float r0 = top0 == -INFINITY ? 1.f : ex2(-d0), r1 = top1 == -INFINITY ? 1.f : ex2(-d1);
            m0 += d0; m1 += d1;
            if (up0) top0 = W_MAX;
            if (up1) top1 = W_MAX;
#pragma unroll
            for (int j = 0; j < 2; ++j) { s[j][0] -= d0; s[j][1] -= d0; s[j][2] -= d1; s[j][3] -= d1; }
            l0 = mul2(l0, both(r0)); l1 = mul2(l1, both(r1));
            scale_rows(o, r0, r1);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
#pragma unroll
            for (int i = 0; i < 4; ++i) s[j][i] = ex2(s[j][i]);
            l0 = add2(l0, pack2(s[j][0], s[j][1]));
            l1 = add2(l1, pack2(s[j][2], s[j][3]));
        }
    }
};
// a row's sum across the four threads of a group
__device__ __forceinline__ float group_sum(uint64_t x) {
    float s = sum2(x);
    s += __shfl_xor_sync(FULL, s, 1);
    return s + __shfl_xor_sync(FULL, s, 2);
}
// A warp's pass in fp32.
template <int CP, typename Walker>
__device__ __forceinline__ void forward_fp32(const Walker& walker, int nchunks, const BandView& view, bool seeded, const TilePoints& at, const float* q,
                                             const float* out, const float* lse, Softmax& sm, float (&o)[CP / 8][4], int C, float scale_log2) {
    using S = Stage<CP>;
    const int t = walker.lane & 3;
    sm.start<CP>(seeded, view, at, out, lse, o, C, t);
    walker.template run<1>(nchunks, [&](uint32_t st, uint32_t mask, auto&&) {
        float s[2][4];
        dots_fp32<CP>(s, q + at.pt0 * C, q + at.pt1 * C, st + S::A, C, t);
        const uint64_t bias2[2] = {lds64(st + S::M0 + 8 * t), lds64(st + S::M0 + 32 + 8 * t)};
        sm.weights(s, o, both(scale_log2), bias2, mask);
        sums_fp32<CP>(o, s, st + S::B, t);
    });
}

// Blocks of 4 warps per SM: as many as the registers of the kernel allow without spills that matter.  Measured at 128x256, N = 16,
// C = 32 (whole streams): forward 4 blocks 333 us, 5 blocks 338; dq 3 / 4 / 5 blocks 419 / 383 / 550 us; dk/dv 3 / 4 blocks
// 455 / 589.  Single products need fewer registers: forward 5 blocks 271 us, 4 blocks 281.
template <int CP, bool LP>
struct Blocks {
    static constexpr int FWD = CP == 64 ? 3 : CP == 32 && !LP ? 4 : 5, DQ = CP == 64 ? 2 : CP == 32 || !LP ? 4 : 5, DKDV = CP == 64 ? 2 : CP == 32 && !LP ? 3 : 4;
};

template <int CP, bool LP, bool PAD, bool CF>
__global__ void __launch_bounds__(THREADS, Blocks<CP, LP>::FWD)
forward_band_kernel(DevPlan p, const __grid_constant__ BandView view, const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v,
                    float* out, float* lse, float* out_cf, int C_, float scale_log2) {
    const int C = PAD ? C_ : CP;
    constexpr int NT = CP / 8;
    using S = Stage<CP>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Task task;
    if (!task.decode(view)) return;
    const int tile = task.tile, n = task.n, group = task.group;
    const int w0 = tile * TILE_LON;
    StreamScales<CP> sc;
    const int g = sc.g, t = sc.t;

    TileOperand<CP, LP> Q;     // q in the log2 domain
    {
        const TilePoints at(n, group * TILE_LAT, w0 + g, p.nlat_out, p.nlon_out);
        Q.template load<true>(q + at.pt0 * C, q + at.pt1 * C, scale_log2, C, t);
    }
    const size_t slice = (size_t)n * p.nlat_in * p.nlon_in * C;
    int chunk0, nchunks;
    task.chunks(view, group, chunk0, nchunks);
    const auto walker = make_walker<CP, false, PAD>(smem_raw, view.s, chunk0, w0, p.nlon_out, p.ps, C, k + slice, v + slice, nullptr, nullptr);
    float o[NT][4];
    Softmax sm;
    uint64_t bad;
    const bool plain = !scores_lost<LP>(Q.back0, C);      // k needs no scale of its own for scores of this size
    const bool seeded = view.dense_ptr != nullptr && (!task.shared || task.warp == 0);
    {
        const TilePoints at(n, group * TILE_LAT, w0 + g, p.nlat_out, p.nlon_out);
        if (seeded && view.has_dense(group * TILE_LAT, p.nlat_out)) wait_for_dense();
        sm.template start<CP>(seeded, view, at, out, lse, o, C, t);
    }
    bad = 0;
    walker.template run<1>(nchunks, [&](uint32_t st, uint32_t mask, auto&&) {
        if (!sc.known()) {
            const float before = sc.b.scale;
            sc.look(st, plain, false);
            if (seeded) scale_rows(o, sc.b.scale / before, sc.b.scale / before);
        }
        float s[2][4];
        SplitRows<CP, LP> V;
        constexpr bool EARLY = CP < 64 && !LP;      // read v while the scores are computed, if there are registers for it
        {
            SplitRows<CP, LP> K;
            K.template load<false>(st + sc.own + S::A, sc.a.scale);
            if constexpr (EARLY) V.template load<true>(st + sc.own + S::B, sc.b.scale);
            rows_dot_points<CP, LP>(s, Q, K);
        }
        const uint64_t bias2[2] = {lds64(st + S::M0 + 8 * t), lds64(st + S::M0 + 32 + 8 * t)};
        note_overflow<LP>(bad, s);
        sm.weights(s, o, both(Q.back0 * sc.a.inv), bias2, mask);
        Weights<LP> W;
        W.set(s);
        if constexpr (!EARLY) V.template load<true>(st + sc.own + S::B, sc.b.scale);
        weights_times_points<CP, LP>(o, W, V);
    });
    bool lost = overflowed(sum2(add2(sm.l0, sm.l1)) + sum2(bad) + total(o));
    if (!lost) {
        // an output's floor is 2^-25 of its scaled v, which shows from 2^-8 on
        constexpr float LIMIT = (LP ? REDUCED : 1.f) / 256.f;
        const float ls0 = group_sum(sm.l0), ls1 = group_sum(sm.l1);
        lost = (sc.a.known && scores_lost<LP>(Q.back0 * sc.a.inv, C)) ||
               (sc.b.known && sums_lost<CP>(o, ls0 * LIMIT, ls1 * LIMIT, walker, nchunks, v + slice, LIMIT * sc.b.inv, C, t));
    }
    if (lost) {
        const TilePoints at(n, group * TILE_LAT, w0 + g, p.nlat_out, p.nlon_out);
        forward_fp32<CP>(walker, nchunks, view, seeded, at, q, out, lse, sm, o, C, scale_log2);
        sc.b = StreamScale();
    }
    const TilePoints at(n, group * TILE_LAT, w0 + g, p.nlat_out, p.nlon_out);
    // normalise, store
    float m0 = sm.m0, m1 = sm.m1, ls0 = group_sum(sm.l0), ls1 = group_sum(sm.l1);
    float back0 = sc.b.inv, back1 = sc.b.inv;
    if (task.shared) {
        const Exchange<CP> x(smem_raw);
        x.put(o, task.warp, 0, sc.b.inv, sc.b.inv);
        x.at(task.warp, CP / 2) = sm.top0 == -INFINITY ? -INFINITY : m0;       // (a warp may have had no column for a row)
        x.at(task.warp, CP / 2 + 1) = sm.top1 == -INFINITY ? -INFINITY : m1;
        x.at(task.warp, CP / 2 + 2) = ls0;
        x.at(task.warp, CP / 2 + 3) = ls1;
        __syncthreads();
        float f0[WARPS], f1[WARPS];
        m0 = m1 = -INFINITY;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) { m0 = fmaxf(m0, f0[w] = x.at(w, CP / 2)); m1 = fmaxf(m1, f1[w] = x.at(w, CP / 2 + 1)); }
        ls0 = ls1 = 0.f;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
            f0[w] = f0[w] == -INFINITY ? 0.f : ex2(f0[w] - m0);
            f1[w] = f1[w] == -INFINITY ? 0.f : ex2(f1[w] - m1);
            ls0 = fmaf(x.at(w, CP / 2 + 2), f0[w], ls0);
            ls1 = fmaf(x.at(w, CP / 2 + 3), f1[w], ls1);
        }
        x.add(o, task, 0, f0, f1);
        back0 = back1 = 1.f;
    }
    const float inv0 = back0 / ls0, inv1 = back1 / ls1;
#pragma unroll
    for (int m = 0; m < NT / 2; ++m) {
        if (!task.writes(m)) continue;
        if (at.ok0) store_quad<CP>(out + at.pt0 * C, m, C, t, quad(o, m, 0, inv0));
        if (at.ok1) store_quad<CP>(out + at.pt1 * C, m, C, t, quad(o, m, 1, inv1));
        if constexpr (CF) {
            const size_t P = (size_t)p.nlat_out * p.nlon_out;
            if (at.ok0) store_quad_cf<CP>(out_cf, at.pt0, n, P, m, C, t, quad(o, m, 0, inv0));
            if (at.ok1) store_quad_cf<CP>(out_cf, at.pt1, n, P, m, C, t, quad(o, m, 1, inv1));
        }
    }
    if (lse != nullptr && t == 0 && task.writes(0)) {
        if (at.ok0) lse[at.pt0] = ((m0 + W_SET) + log2f(ls0 * W_UNIT)) * LN2;
        if (at.ok1) lse[at.pt1] = ((m1 + W_SET) + log2f(ls1 * W_UNIT)) * LN2;
    }
}

// ---------------------------------------------------------------------------------------------------------
// backward, dq:  dq_i = scale * sum_j p_ij (t_ij - D_i) k_j,  D_i = dout_i . out_i  (App. B.4)
// `out` and `dq` may be the same buffer: a warp reads its own 16 rows of `out` before it writes them as dq.
// t, D and ds are in the units of the scaled dout row and the scaled v until the end.
// ---------------------------------------------------------------------------------------------------------
// A warp's pass in fp32.
template <int CP, typename Walker>
__device__ __forceinline__ void dq_fp32(const Walker& walker, int nchunks, const TilePoints& at, const float* q, const float* dout,
                                        float lse0, float lse1, float D0, float D1, float (&acc)[CP / 8][4], int C, float scale_log2) {
    using S = Stage<CP>;
    const int t = walker.lane & 3;
    clear(acc);
    walker.template run<1>(nchunks, [&](uint32_t st, uint32_t mask, auto&&) {
        float s[2][4], tt[2][4];
        dots_fp32<CP>(s, q + at.pt0 * C, q + at.pt1 * C, st + S::A, C, t);
        dots_fp32<CP>(tt, dout + at.pt0 * C, dout + at.pt1 * C, st + S::B, C, t);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            float b[2];
            unpack2(lds64(st + S::M0 + 32 * j + 8 * t), b[0], b[1]);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                s[j][i] = ex2(fmaf(s[j][i], scale_log2, fmaf(i < 2 ? lse0 : lse1, -LOG2E, b[i % 2]))) * (tt[j][i] - (i < 2 ? D0 : D1));
        }
        apply_mask(s, mask, 0.f);
        sums_fp32<CP>(acc, s, st + S::A, t);
    });
}

template <int CP, bool LP, bool PAD, bool CF>
__global__ void __launch_bounds__(THREADS, Blocks<CP, LP>::DQ)
backward_dq_band_kernel(DevPlan p, const __grid_constant__ BandView view, const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v,
                        const float* __restrict__ dout, const float* out, const float* __restrict__ lse,
                        float* dq, float* __restrict__ Dws, float* dq_cf, int C_, float scale) {
    const int C = PAD ? C_ : CP;
    constexpr int NT = CP / 8;
    using S = Stage<CP>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Task task;
    if (!task.decode(view)) return;
    const int tile = task.tile, n = task.n, group = task.group;
    const int w0 = tile * TILE_LON;
    StreamScales<CP> sc;
    const int g = sc.g, t = sc.t;

    TileOperand<CP, LP> Q, Y;
    float D0 = 0.f, D1 = 0.f, lse0, lse1;
    {
        const TilePoints at(n, group * TILE_LAT, w0 + g, p.nlat_out, p.nlon_out);
        Q.template load<true>(q + at.pt0 * C, q + at.pt1 * C, scale * LOG2E, C, t);
        Y.template load<false>(dout + at.pt0 * C, dout + at.pt1 * C, 1.f, C, t);
#pragma unroll
        for (int i = 0; i < CP / 4; i += 4) {
            const int c = Own<CP>::channel(t, i);
            if (c < C) {
                const float4 a = *reinterpret_cast<const float4*>(out + at.pt0 * C + c), ya = __ldg(reinterpret_cast<const float4*>(dout + at.pt0 * C + c));
                const float4 b = *reinterpret_cast<const float4*>(out + at.pt1 * C + c), yb = __ldg(reinterpret_cast<const float4*>(dout + at.pt1 * C + c));
                D0 = fmaf(a.x, ya.x, fmaf(a.y, ya.y, fmaf(a.z, ya.z, fmaf(a.w, ya.w, D0))));
                D1 = fmaf(b.x, yb.x, fmaf(b.y, yb.y, fmaf(b.z, yb.z, fmaf(b.w, yb.w, D1))));
            }
        }
        D0 += __shfl_xor_sync(FULL, D0, 1); D1 += __shfl_xor_sync(FULL, D1, 1);
        D0 += __shfl_xor_sync(FULL, D0, 2); D1 += __shfl_xor_sync(FULL, D1, 2);
        if (t == 0 && task.writes(0)) {
            if (at.ok0) Dws[at.pt0] = D0;
            if (at.ok1) Dws[at.pt1] = D1;
        }
        lse0 = lse[at.pt0]; lse1 = lse[at.pt1];
    }
    const size_t slice = (size_t)n * p.nlat_in * p.nlon_in * C;
    int chunk0, nchunks;
    task.chunks(view, group, chunk0, nchunks);
    const auto walker = make_walker<CP, false, PAD>(smem_raw, view.s, chunk0, w0, p.nlon_out, p.ps, C, k + slice, v + slice, nullptr, nullptr);
    float acc[NT][4];
    WeightScale ws;          // of ds
    float nD0, nD1;          // -D times the weight scale
    float max0, max1;        // largest |ds| of the thread's columns
    float f0, f1;            // dq per sum
    clear(acc);
    ws = WeightScale();
    uint64_t bad = 0;
    nD0 = -D0 / Y.back0 * sc.b.scale; nD1 = -D1 / Y.back1 * sc.b.scale;
    max0 = max1 = 0.f;
    walker.template run<LP && CP == 32 ? 1 : 2>(nchunks, [&](uint32_t st, uint32_t mask, auto&& release) {
        if (!sc.known()) {
            const float before = sc.b.scale;
            sc.look(st, LP, LP);
            const float f = sc.b.scale / before;
            nD0 *= f; nD1 *= f;
            scale_rows(acc, f, f);
        }
        float s[2][4], tt[2][4];
        SplitRows<CP, LP> K;
        {
            SplitRows<CP, LP> V;
            V.load(st + sc.own + S::B, sc.b.scale);
            rows_dot_points<CP, LP>(tt, Y, V);
        }
        K.load(st + sc.own + S::A, sc.a.scale);
        const uint64_t bias2[2] = {lds64(st + S::M0 + 8 * t), lds64(st + S::M0 + 32 + 8 * t)};
        release();
        rows_dot_points<CP, LP>(s, Q, K);
        note_overflow<LP>(bad, s);
        const uint64_t f2 = both(Q.back0 * sc.a.inv), h2 = both(ws.scale);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            unpack2(fma2(pack2(s[j][0], s[j][1]), f2, fma2(both(lse0), both(-LOG2E), bias2[j])), s[j][0], s[j][1]);
            unpack2(fma2(pack2(s[j][2], s[j][3]), f2, fma2(both(lse1), both(-LOG2E), bias2[j])), s[j][2], s[j][3]);
#pragma unroll
            for (int i = 0; i < 4; ++i) s[j][i] = ex2(s[j][i]);
            unpack2(mul2(pack2(s[j][0], s[j][1]), fma2(pack2(tt[j][0], tt[j][1]), h2, both(nD0))), s[j][0], s[j][1]);       // ds
            unpack2(mul2(pack2(s[j][2], s[j][3]), fma2(pack2(tt[j][2], tt[j][3]), h2, both(nD1))), s[j][2], s[j][3]);
        }
        if (!(mask & BAND_ALL)) apply_mask(s, mask, 0.f);
        row_max(max0, max1, s);
        if (__any_sync(FULL, fmaxf(max0, max1) > ws.limit)) {
            const float f = ws.update(fmaxf(max0, max1));
            scale_rows(acc, f, f);
            scale_rows(s, f, f);
            nD0 *= f; nD1 *= f;
            max0 *= f; max1 *= f;
        }
        Weights<LP> W;
        W.set(s);
        weights_times_points<CP, LP>(acc, W, K);
    });
    f0 = scale * sc.a.inv / ws.scale * sc.b.inv * Y.back0; f1 = scale * sc.a.inv / ws.scale * sc.b.inv * Y.back1;
    bool lost = overflowed(total(acc) + sum2(bad));
    if (!lost) {
        // The floors: of ds, 2^-25; of t, below 2^-8 in units of ds's scale.  They are compared with the row's largest ds or, if
        // t and D nearly cancel, with p D, whose rounding is an error of ds in any case (the row's p add up to 1).
        const float r0 = group_max(max0), r1 = group_max(max1), least = (LP ? REDUCED : 1.f) * fmaxf(1.f / 128.f, 1024.f * ws.scale);
        const float any = 1.f / (64.f * (float)nchunks);
        const bool low = (r0 > 0.f && fmaxf(r0, any * fabsf(nD0)) < least) || (r1 > 0.f && fmaxf(r1, any * fabsf(nD1)) < least);
        constexpr float LIMIT = (LP ? REDUCED : 1.f) / 256.f;         // of k, in a sum
        lost = (sc.a.known && scores_lost<LP>(Q.back0 * sc.a.inv, C)) || (sc.b.known && __any_sync(FULL, low)) ||
               (sc.a.known && sums_lost<CP>(acc, r0 * LIMIT, r1 * LIMIT, walker, nchunks, k + slice, LIMIT * sc.a.inv, C, t));
    }
    if (lost) {
        const TilePoints at(n, group * TILE_LAT, w0 + g, p.nlat_out, p.nlon_out);
        dq_fp32<CP>(walker, nchunks, at, q, dout, lse0, lse1, D0, D1, acc, C, scale * LOG2E);
        f0 = f1 = scale;
    }
    const TilePoints at(n, group * TILE_LAT, w0 + g, p.nlat_out, p.nlon_out);
    if (task.shared) {
        const Exchange<CP> x(smem_raw);
        x.put(acc, task.warp, 0, f0, f1);
        __syncthreads();         // (also: every warp has read its rows of `out`)
        x.add(acc, task, 0);
        f0 = f1 = 1.f;
    }
    // the dense kernel has written its part of dq for rows that have windows there: add it
    if (view.dense_ptr != nullptr && view.has_dense(group * TILE_LAT, p.nlat_out)) wait_for_dense();
    const bool add0 = view.dense_ptr != nullptr && view.dense_ptr[at.ha + 1] > view.dense_ptr[at.ha];
    const bool add1 = view.dense_ptr != nullptr && view.dense_ptr[at.hb + 1] > view.dense_ptr[at.hb];
#pragma unroll
    for (int m = 0; m < NT / 2; ++m) {
        if (!task.writes(m)) continue;
        float4 r0 = quad(acc, m, 0, f0), r1 = quad(acc, m, 1, f1);
        if (add0) r0 = r0 + load_quad<CP>(dq + at.pt0 * C, m, C, t);
        if (add1) r1 = r1 + load_quad<CP>(dq + at.pt1 * C, m, C, t);
        if constexpr (!CF) {
            if (at.ok0) store_quad<CP>(dq + at.pt0 * C, m, C, t, r0);
            if (at.ok1) store_quad<CP>(dq + at.pt1 * C, m, C, t, r1);
        } else {
            const size_t P = (size_t)p.nlat_out * p.nlon_out;
            if (at.ok0) store_quad_cf<CP>(dq_cf, at.pt0, n, P, m, C, t, r0);
            if (at.ok1) store_quad_cf<CP>(dq_cf, at.pt1, n, P, m, C, t, r1);
        }
    }
}

// ---------------------------------------------------------------------------------------------------------
// backward, dk and dv, gathered per input point over the transposed stream (no atomics):
//   dk_j = scale * sum_i p_ij (t_ij - D_i) q_i,   dv_j = sum_i p_ij dout_i          (App. B.4)
// Tile rows are 8 input columns on each of the two rings of an input ring pair; stream columns are output points.
// ---------------------------------------------------------------------------------------------------------
// A warp's pass in fp32.
template <int CP, typename Walker>
__device__ __forceinline__ void dkdv_fp32(const Walker& walker, int nchunks, const TilePoints& at, const float* k, const float* v, const float* log2_omega,
                                          float (&gk)[CP / 8][4], float (&gv)[CP / 8][4], int C, float scale_log2) {
    using S = Stage<CP>;
    const int t = walker.lane & 3;
    const float bias0 = log2_omega[at.ha], bias1 = log2_omega[at.hb];
    clear(gk);
    clear(gv);
    walker.template run<1>(nchunks, [&](uint32_t st, uint32_t mask, auto&&) {
        float s[2][4], tt[2][4];
        dots_fp32<CP>(s, k + at.pt0 * C, k + at.pt1 * C, st + S::A, C, t);
        dots_fp32<CP>(tt, v + at.pt0 * C, v + at.pt1 * C, st + S::B, C, t);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            float l[2], D[2];
            unpack2(lds64(st + S::M0 + 32 * j + 8 * t), l[0], l[1]);
            unpack2(lds64(st + S::M1 + 32 * j + 8 * t), D[0], D[1]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                s[j][i] = ex2(fmaf(s[j][i], scale_log2, fmaf(l[i % 2], -LOG2E, i < 2 ? bias0 : bias1)));
                tt[j][i] = s[j][i] * (tt[j][i] - D[i % 2]);
            }
        }
        apply_mask(s, mask, 0.f);
        apply_mask(tt, mask, 0.f);
        sums_fp32<CP>(gv, s, st + S::B, t);
        sums_fp32<CP>(gk, tt, st + S::A, t);
    });
}

template <int CP, bool LP, bool PAD, bool CF>
__global__ void __launch_bounds__(THREADS, Blocks<CP, LP>::DKDV)
backward_dkdv_band_kernel(DevPlan p, const __grid_constant__ BandView view, const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v,
                          const float* __restrict__ dout, const float* __restrict__ lse, const float* __restrict__ Dws,
                          float* dk, float* dv, float* dk_cf, float* dv_cf, int C_, float scale) {
    const int C = PAD ? C_ : CP;
    constexpr int NT = CP / 8;
    using S = Stage<CP>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Task task;
    if (!task.decode(view)) return;
    const int tile = task.tile, n = task.n, group = task.group;
    StreamScales<CP> sc;
    const int g = sc.g, t = sc.t;
    // input column of tile row g (and g+8), the first partner index of the tile, and the stream row
    int col, first, srow;
    if (p.t_consecutive) {           // 8 consecutive input columns
        col = tile * TILE_LON + g;
        first = tile * TILE_LON / p.ps;
        srow = group;
    } else {                         // every ps-th column of one residue class
        const int r = tile % p.ps, u0 = (tile / p.ps) * TILE_LON;
        col = (u0 + g) * p.ps + r;
        first = u0;
        srow = group * p.ps + r;
    }
    TileOperand<CP, LP> K, V;
    float b0, b1;                 // log2 omega, later with the exponent of p's scale
    {
        const TilePoints at(n, group * TILE_LAT, col, p.nlat_in, p.nlon_in);
        K.template load<true>(k + at.pt0 * C, k + at.pt1 * C, scale * LOG2E, C, t);
        V.template load<true>(v + at.pt0 * C, v + at.pt1 * C, 1.f, C, t);
        b0 = p.log2_omega[at.ha]; b1 = p.log2_omega[at.hb];
    }
    const size_t oslice = (size_t)n * p.nlat_out * p.nlon_out;
    int chunk0, nchunks;
    task.chunks(view, srow, chunk0, nchunks);
    const auto walker = make_walker<CP, true, PAD>(smem_raw, view.s, chunk0, first, p.nlon_out, 1, C, q + oslice * C, dout + oslice * C, lse + oslice, Dws + oslice);
    float gk[NT][4], gv[NT][4];
    // The scale of p: over global attention, and for keys that little attention reaches, all of them are small.  It brings the largest
    // of the first chunk that has some to [2^3, 2^4), so that a p 2^12 times as large still fits.
    float p_scale;
    WeightScale ws;          // of ds, beyond that
    float pmax0, pmax1, max0, max1;      // largest p and |ds| of the thread's columns
    float fk, fv;            // dk and dv per sum
    clear(gk);
    clear(gv);
    ws = WeightScale();
    p_scale = 0.f;        // not known
    float unit = sc.b.scale / V.back0;      // t, D and ds are in the units of the scaled dout and v until the end
    uint64_t bad = 0;
    pmax0 = pmax1 = max0 = max1 = 0.f;
    walker.template run<1>(nchunks, [&](uint32_t st, uint32_t mask, auto&&) {
        if (!sc.known()) {
            const float before = sc.b.scale;
            sc.look(st, LP, LP);
            unit *= sc.b.scale / before;
            scale_rows(gk, sc.b.scale / before, sc.b.scale / before);
        }
        float s[2][4], tt[2][4];
        SplitRows<CP, LP> Q, Y;
        Q.load(st + sc.own + S::A, sc.a.scale);
        rows_dot_points<CP, LP>(s, K, Q);
        Y.load(st + sc.own + S::B, sc.b.scale);
        rows_dot_points<CP, LP>(tt, V, Y);
        const uint64_t lse2[2] = {lds64(st + S::M0 + 8 * t), lds64(st + S::M0 + 32 + 8 * t)}, D2[2] = {lds64(st + S::M1 + 8 * t), lds64(st + S::M1 + 32 + 8 * t)};
        note_overflow<LP>(bad, s);
        const uint64_t f2 = both(K.back0 * sc.a.inv), h2 = both(ws.scale), nw2 = both(-ws.scale * unit), nlog2e2 = both(-LOG2E);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            // bias: log2 omega_j of the row's ring
            unpack2(fma2(pack2(s[j][0], s[j][1]), f2, fma2(lse2[j], nlog2e2, both(b0))), s[j][0], s[j][1]);
            unpack2(fma2(pack2(s[j][2], s[j][3]), f2, fma2(lse2[j], nlog2e2, both(b1))), s[j][2], s[j][3]);
#pragma unroll
            for (int i = 0; i < 4; ++i) s[j][i] = ex2(s[j][i]);
        }
        if (!(mask & BAND_ALL)) apply_mask(s, mask, 0.f);
        row_max(pmax0, pmax1, s);
        if (p_scale == 0.f) {
            const uint32_t w = __reduce_max_sync(FULL, __float_as_uint(fmaxf(pmax0, pmax1)));
            if (w != 0) {
                p_scale = pow2_to(3, max(w & 0x7f800000u, (uint32_t)(127 - 72) << 23));
                const float e = (float)((int)(__float_as_uint(p_scale) >> 23) - 127);
                b0 += e; b1 += e;
                scale_rows(s, p_scale, p_scale);
                pmax0 *= p_scale; pmax1 *= p_scale;
            }
        }
        Weights<LP> P, W;
        P.set(s);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const uint64_t nD2 = mul2(D2[j], nw2);
            unpack2(mul2(pack2(s[j][0], s[j][1]), fma2(pack2(tt[j][0], tt[j][1]), h2, nD2)), s[j][0], s[j][1]);      // ds
            unpack2(mul2(pack2(s[j][2], s[j][3]), fma2(pack2(tt[j][2], tt[j][3]), h2, nD2)), s[j][2], s[j][3]);
        }
        row_max(max0, max1, s);
        if (__any_sync(FULL, fmaxf(max0, max1) > ws.limit)) {
            const float f = ws.update(fmaxf(max0, max1));
            scale_rows(gk, f, f);
            scale_rows(s, f, f);
            max0 *= f; max1 *= f;
        }
        W.set(s);
        weights_times_points<CP, LP>(gv, P, Y);
        weights_times_points<CP, LP>(gk, W, Q);
    });
    // k was pre-multiplied by scale*log2e for the scores only; dk carries the plain scale.  Both sums carry p's scale.
    const float p_back = p_scale == 0.f ? 0.f : 1.f / p_scale;       // (0: no p at all)
    fk = scale * sc.a.inv / ws.scale * sc.b.inv * p_back * V.back0; fv = sc.b.inv * p_back;
    bool lost = overflowed(total(gk) + total(gv) + sum2(bad));
    if (!lost) {
        // The floors: of p and ds, 2^-25; of t, below 2^-8 in units of ds's scale and times p.
        const float p0 = group_max(pmax0), p1 = group_max(pmax1), r0 = group_max(max0), r1 = group_max(max1);
        constexpr float LEAST = (LP ? REDUCED : 1.f) / 128.f, LIMIT = (LP ? REDUCED : 1.f) / 256.f;      // (LIMIT: of q and dout, in a sum)
        const float of_t = (LP ? REDUCED : 1.f) * 1024.f * ws.scale;
        const bool low = (p0 > 0.f && p0 < LEAST) || (p1 > 0.f && p1 < LEAST) || (r0 > 0.f && r0 < fmaxf(LEAST, of_t * p0)) || (r1 > 0.f && r1 < fmaxf(LEAST, of_t * p1));
        lost = (sc.a.known && scores_lost<LP>(K.back0 * sc.a.inv, C)) || __any_sync(FULL, low) ||
               (sc.b.known && sums_lost<CP>(gv, p0 * LIMIT, p1 * LIMIT, walker, nchunks, dout + oslice * C, LIMIT * sc.b.inv, C, t)) ||
               (sc.a.known && sums_lost<CP>(gk, r0 * LIMIT, r1 * LIMIT, walker, nchunks, q + oslice * C, LIMIT * sc.a.inv, C, t));
    }
    if (lost) {
        const TilePoints at(n, group * TILE_LAT, col, p.nlat_in, p.nlon_in);
        dkdv_fp32<CP>(walker, nchunks, at, k, v, p.log2_omega, gk, gv, C, scale * LOG2E);
        fk = scale; fv = 1.f;
    }
    const TilePoints at(n, group * TILE_LAT, col, p.nlat_in, p.nlon_in);
    if (task.shared) {
        const Exchange<CP> x(smem_raw);
        x.put(gk, task.warp, 0, fk, fk);
        x.put(gv, task.warp, CP / 2, fv, fv);
        __syncthreads();
        x.add(gk, task, 0);
        x.add(gv, task, CP / 2);
        fk = fv = 1.f;
    }
    if (view.dense_ptr != nullptr && view.has_dense(group * TILE_LAT, p.nlat_in)) wait_for_dense();
    const bool add0 = view.dense_ptr != nullptr && view.dense_ptr[at.ha + 1] > view.dense_ptr[at.ha];
    const bool add1 = view.dense_ptr != nullptr && view.dense_ptr[at.hb + 1] > view.dense_ptr[at.hb];
#pragma unroll
    for (int m = 0; m < NT / 2; ++m) {
        if (!task.writes(m)) continue;
        float4 k0 = quad(gk, m, 0, fk), k1 = quad(gk, m, 1, fk), v0 = quad(gv, m, 0, fv), v1 = quad(gv, m, 1, fv);
        if (add0) {      // the dense kernel has already written its part of dk, dv for input rings that have windows there
            k0 = k0 + load_quad<CP>(dk + at.pt0 * C, m, C, t);
            v0 = v0 + load_quad<CP>(dv + at.pt0 * C, m, C, t);
        }
        if (add1) {
            k1 = k1 + load_quad<CP>(dk + at.pt1 * C, m, C, t);
            v1 = v1 + load_quad<CP>(dv + at.pt1 * C, m, C, t);
        }
        if constexpr (!CF) {
            if (at.ok0) { store_quad<CP>(dk + at.pt0 * C, m, C, t, k0); store_quad<CP>(dv + at.pt0 * C, m, C, t, v0); }
            if (at.ok1) { store_quad<CP>(dk + at.pt1 * C, m, C, t, k1); store_quad<CP>(dv + at.pt1 * C, m, C, t, v1); }
        } else {
            const size_t P = (size_t)p.nlat_in * p.nlon_in;
            if (at.ok0) { store_quad_cf<CP>(dk_cf, at.pt0, n, P, m, C, t, k0); store_quad_cf<CP>(dv_cf, at.pt0, n, P, m, C, t, v0); }
            if (at.ok1) { store_quad_cf<CP>(dk_cf, at.pt1, n, P, m, C, t, k1); store_quad_cf<CP>(dv_cf, at.pt1, n, P, m, C, t, v1); }
        }
    }
}

template <int CP, bool LP, bool PAD, bool CF>
cudaError_t prepare_instantiation() {
    const int bytes = (int)smem_bytes<CP>();
    cudaError_t e = cudaFuncSetAttribute(forward_band_kernel<CP, LP, PAD, CF>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(backward_dq_band_kernel<CP, LP, PAD, CF>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(backward_dkdv_band_kernel<CP, LP, PAD, CF>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    return e;
}

// Calls f(channels of the instantiation, reduced precision, padded, channels-first results) with constants.
template <typename F>
cudaError_t dispatch(int C, bool lp, bool cf, F&& f) {
    constexpr std::false_type no;
    constexpr std::true_type yes;
    auto with = [&](auto cp) {
        const bool pad = C != decltype(cp)::value;
        if (lp) return pad || cf ? cudaErrorInvalidValue : f(cp, yes, no, no);
        if (pad) return cf ? f(cp, no, yes, yes) : f(cp, no, yes, no);
        return cf ? f(cp, no, no, yes) : f(cp, no, no, no);
    };
    if (C <= 16) return with(std::integral_constant<int, 16>());
    if (C <= 32) return with(std::integral_constant<int, 32>());
    if (C <= 64) return with(std::integral_constant<int, 64>());
    return cudaErrorInvalidValue;
}

// A stream is shared by the warps of a block if it is at least this many times a warp's fair part of the launch, and this many
// chunks.  Near the poles streams are several times as long as the average, and one warp alone with one of them outlasts the rest
// of a small launch.  Whole streams, us without : with sharing: 32x64, N = 1, C = 16, forward 17.0 : 9.0; 256x512 -> 128x256,
// N = 4, C = 32, forward 316 : 226; 128x256, N = 4, dk/dv 127.6 : 126.8.  A limit of 0.25 or 0.5 costs large launches
// 2 to 4 % (each sharer repeats the prologue), 2 leaves the down-sampling case at 308.
// Equally long streams (global attention) leave a last wave of blocks that is nearly empty, up to four waves or so.
constexpr double SHARE_ABOVE = 1, SHARE_EQUAL_ABOVE = 0.25, SHARE_MIN = 8;

int ceil_div_host(int a, int b) { return (a + b - 1) / b; }

// The view of a launch - the stream with the windows the dense kernels do not serve (band) or with all of them - and its grid;
// false if the problem has too many tasks.
bool make_view(const DevPlan& p, bool transposed, bool band, int N, int blocks_per_sm, BandView& v, unsigned& grid) {
    v.s = transposed ? (band ? p.tb : p.t) : (band ? p.fwdb : p.fwd);
    v.dense_ptr = !band ? nullptr : transposed ? p.t_dense_ptr : p.dense_ptr;
    v.tiles = transposed && p.t_consecutive ? ceil_div_host(p.nlon_in, TILE_LON) : (transposed ? p.ps : 1) * ceil_div_host(p.nlon_out, TILE_LON);
    v.N = N;
    const long long per_group = (long long)v.tiles * N, total = per_group * v.s.groups;
    if (total > 0x7fffffffLL) return false;
    // Share the streams that alone would take long in comparison with the whole launch.  They are counted from the front of the order.
    // (Behind a dense kernel the groups that wait for it come later and are not shared: where those kernels are used, a launch has
    // at most two that exceed the limit, by less than a tenth.)
    const double fair = (double)v.s.chunks * (transposed && !p.t_consecutive ? v.tiles / p.ps : v.tiles) * N / ((double)p.num_sms * blocks_per_sm * WARPS);
    const double above = v.s.one_row ? SHARE_EQUAL_ABOVE : SHARE_ABOVE;
    const double longest = fair * above > SHARE_MIN ? fair * above : SHARE_MIN;
    int heavy = 0;
    while (heavy < v.s.groups && v.s.lengths[heavy] >= longest) ++heavy;
    v.shared = (int)(heavy * per_group);
    v.total = (int)total;
    grid = (unsigned)(v.shared + (total - v.shared + WARPS - 1) / WARPS);
    return true;
}

template <typename... P, typename... A>
cudaError_t launch(void (*kernel)(P...), unsigned grid, size_t smem, bool after_dense, cudaStream_t stream, A... args) {
    cudaLaunchAttribute overlap{};
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t config{};
    config.gridDim = grid;
    config.blockDim = THREADS;
    config.dynamicSmemBytes = smem;
    config.stream = stream;
    config.attrs = &overlap;
    config.numAttrs = after_dense ? 1 : 0;
    return cudaLaunchKernelEx(&config, kernel, P(args)...);
}

}  // namespace

cudaError_t band_prepare_device() {
    cudaError_t e = cudaSuccess;
    const std::pair<int, bool> wide[] = {{48, false}, {64, false}, {64, true}};       // narrower rows need less than the default 48 KB
    static_assert(smem_bytes<32>() <= 48 * 1024, "list of the instantiations to prepare");
    for (const auto& [C, lp] : wide)
        for (bool cf : {false, true})
            if (e == cudaSuccess && !(lp && cf))
                e = dispatch(C, lp, cf, [](auto cp, auto low, auto pad, auto cf) { return prepare_instantiation<decltype(cp)::value, decltype(low)::value, decltype(pad)::value, decltype(cf)::value>(); });
    return e;
}

bool band_path_supported(const DevPlan& p, int C) {
    return p.fwd.columns != nullptr && C >= 4 && C <= 64 && C % 4 == 0 && p.nlon_out >= 16 &&
           (long long)p.nlat_in * p.nlon_in * C < (1LL << 32) && (long long)p.nlat_out * p.nlon_out * C < (1LL << 32);
}

cudaError_t launch_forward_band(const DevPlan& p, const float* q, const float* k, const float* v, float* out, float* lse,
                                int N, int C, bool after_dense, bool lp, cudaStream_t stream, float* out_cf) {
    return dispatch(C, lp, out_cf != nullptr, [&](auto cp, auto low, auto pad, auto cf) {
        constexpr int CP = decltype(cp)::value;
        BandView view;
        unsigned grid;
        if (!make_view(p, false, after_dense, N, Blocks<CP, decltype(low)::value>::FWD, view, grid)) return cudaErrorInvalidValue;
        return launch(forward_band_kernel<CP, decltype(low)::value, decltype(pad)::value, decltype(cf)::value>, grid, smem_bytes<CP>(), after_dense, stream, p, view, q, k, v, out, lse, out_cf, C, LOG2E / sqrtf((float)C));
    });
}

cudaError_t launch_backward_dq_band(const DevPlan& p, const float* q, const float* k, const float* v, const float* dout,
                                    const float* out, const float* lse, float* dq, float* Dws, int N, int C, bool after_dense, bool lp,
                                    cudaStream_t stream, float* dq_cf) {
    return dispatch(C, lp, dq_cf != nullptr, [&](auto cp, auto low, auto pad, auto cf) {
        constexpr int CP = decltype(cp)::value;
        BandView view;
        unsigned grid;
        if (!make_view(p, false, after_dense, N, Blocks<CP, decltype(low)::value>::DQ, view, grid)) return cudaErrorInvalidValue;
        return launch(backward_dq_band_kernel<CP, decltype(low)::value, decltype(pad)::value, decltype(cf)::value>, grid, smem_bytes<CP>(), after_dense, stream, p, view, q, k, v, dout, out, lse, dq, Dws, dq_cf, C, 1.0f / sqrtf((float)C));
    });
}

cudaError_t launch_backward_dkdv_band(const DevPlan& p, const float* q, const float* k, const float* v, const float* dout,
                                      const float* lse, const float* Dws, float* dk, float* dv, int N, int C, bool after_dense, bool lp,
                                      cudaStream_t stream, float* dk_cf, float* dv_cf) {
    return dispatch(C, lp, dk_cf != nullptr, [&](auto cp, auto low, auto pad, auto cf) {
        constexpr int CP = decltype(cp)::value;
        BandView view;
        unsigned grid;
        if (!make_view(p, true, after_dense, N, Blocks<CP, decltype(low)::value>::DKDV, view, grid)) return cudaErrorInvalidValue;
        return launch(backward_dkdv_band_kernel<CP, decltype(low)::value, decltype(pad)::value, decltype(cf)::value>, grid, smem_bytes<CP>(), after_dense, stream, p, view, q, k, v, dout, lse, Dws, dk, dv, dk_cf, dv_cf, C, 1.0f / sqrtf((float)C));
    });
}

}  // namespace sna
