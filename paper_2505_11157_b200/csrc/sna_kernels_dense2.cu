// Dense kernels on tcgen05 / TMEM (sm_100a, C = 32) for whole-ring and wide windows.
//
// Near the poles, and in the global limit theta_cutoff = pi, an output ring attends to EVERY point of an input ring:
// that part of Eq. (s2_attention_discrete_detailed) is a dense attention block with the additive bias log omega of
// App. B.2.  A little further from the poles the windows are still hundreds of columns wide; they run here too, as the
// blocks of the ring that the tile's windows touch, with the entries outside each row's own window masked (TileWalk).
// One thread block owns 128 consecutive output longitudes of one ring (the M = 128 rows of the MMA) and walks its list of
// partner rings in blocks of 128 columns.  The work of a block is spread over specialised warps that run concurrently,
// coupled only by mbarriers:
//
//   warp 8 (one thread)  TMA: raw k and v tiles of the next blocks, 128 points x 128 bytes, 128-byte swizzle
//   warps 16-19          convert: k_lo = k - trunc19(k) (same layout as the raw tile), and v transposed and split into
//                        v_hi^T, v_lo^T (row = channel, K index = column), the K-major form the second GEMM needs
//   warp 9 (one thread)  S = Q K^T into one of two TMEM buffers: q_lo k + q k_lo + q k as TF32 UMMAs (the raw fp32 tiles
//                        serve as the hi parts: the tensor core reads only the top 19 bits)
//   warps 0-3 and 4-7    two softmax groups; thread (half, r) owns tile row r for one half of every block's columns, with
//                        its own running maximum, sum and output: it reads S from TMEM, scales, adds the bias, writes P
//                        over S and P_lo = P - trunc19(P) beside it, and folds the previous block's P V into its registers;
//                        the two halves of a row are merged at the end (a TMEM round trip costs ~130 cycles and one warp
//                        per scheduler cannot hide it, hence two groups)
//   warps 12-15 (1 each) O_part = P V over one quarter of the block's columns each (A operand from TMEM), into their own
//                        accumulators; the row's thread adds its two parts in a fixed order
//
// While the softmax threads work on block j, the tensor core computes S of block j+1 and P V of block j-1, TMA loads block
// j+2 and the converters prepare block j+1.  Every accumulator has exactly one issuing thread and all sums are taken in a
// fixed order, so results are reproducible bit for bit.  Every wait is bounded; a wait that runs out sets the plan's
// device status word and the block leaves, after another bounded wait for the copies and MMAs that it has under way.
#include <cuda.h>

#include "sna_kernels.cuh"

#include <cstdint>
#include <type_traits>

// Optional per-role wait accounting (build with -DSNA_PROF; not part of the product build): every role of block 0 writes
// its total cycles and the cycles spent in up to three kinds of waits to the plan's status area.
#ifdef SNA_PROF
#define PROF_DECL long long prof_w[3] = {0, 0, 0}; const long long prof_t0 = clock64();
#define PROF_WAIT(i, stmt) { const long long t0_ = clock64(); stmt; prof_w[i] += clock64() - t0_; }
#define PROF_DUMP(status, warp, lane, blocks) if ((lane) == 0 && blockIdx.x == 0) { long long* d_ = reinterpret_cast<long long*>((status) + 2) + (warp) * 5; \
    d_[0] = clock64() - prof_t0; d_[1] = prof_w[0]; d_[2] = prof_w[1]; d_[3] = prof_w[2]; d_[4] = (blocks); }
#else
#define PROF_DECL
#define PROF_WAIT(i, stmt) stmt
#define PROF_DUMP(status, warp, lane, blocks)
#endif

namespace sna {
namespace {

constexpr int M2 = 128;          // tile rows
constexpr int BN2 = 128;         // columns per block
constexpr int C2 = 32;           // channels
constexpr int THREADS2 = 640;        // five warpgroups: softmax (two column halves) | TMA, S issuer | four P V issuers | converters
constexpr int THREADS_DKDV = 768;    // six: element-wise (two column halves) | TMA, first GEMMs, statistics | four issuers | converters of q, of dout
constexpr int WAIT2 = 1 << 17;     // polls of one wait (each may suspend for up to ~2 us) before the thread gives up
constexpr float LOG2E_2 = 1.4426950408889634f;
constexpr float LN2_2 = 0.6931471805599453f;

// shared-memory map (bytes from a 1024-aligned base)
constexpr int TILE_B = BN2 * 128;                 // 16 KB: 128 points x 128 bytes
constexpr int OFF_Q = 0, OFF_QLO = TILE_B;
constexpr int OFF_K = 2 * TILE_B;                 // 2 stages x (raw, lo)
constexpr int OFF_VRAW = OFF_K + 4 * TILE_B;      // 2 stages
constexpr int OFF_VT = OFF_VRAW + 2 * TILE_B;     // 2 stages x (hi^T, lo^T)
constexpr int OFF_END = OFF_VT + 4 * TILE_B;      // 12 tiles = 192 KB
constexpr size_t DENSE2_SMEM = OFF_END + 1024;

// TMEM columns
constexpr int T_S0 = 0, T_S1 = 128, T_PLO = 256, T_O = 384, T_COLS = 512;   // T_O: four 32-column accumulators, one per P V issuer
constexpr int PV_ISSUERS = 4;

enum { B_KFULL = 0, B_KCONV = 2, B_KFREE = 4, B_VFULL = 6, B_VRAWFREE = 8, B_VCONV = 10, B_PVDONE = 12 /* [half][stage] */, B_SFULL = 16, B_PREADY = 18 /* [half][buffer] */, B_QFULL = 22, B_COUNT = 23 };
// The "operands ready" barriers that many threads arrive on (PREADY here, DSREADY and READY in the backward kernels) exist
// once per TMEM buffer: a warp that is a whole block ahead of another warp of its group then arrives on the OTHER buffer's
// barrier.  With one barrier per group its second arrival would be counted into the phase of the block the slow warp has
// not finished, and the second GEMM would start on that warp's stale rows (seen as run-to-run differences in 32-row
// blocks of dk / dv when the dk/dv kernel got its second buffer).  The other barriers with several arrivals are safe
// as they are: a converter thread arrives on a stage's CONV / RAWFREE barrier again only after the producer has refilled
// the stage, which waits for the stage's FREE barriers, which the GEMM issuers signal after having waited for the full CONV
// phase; an issuer commits to a buffer's DONE / STFULL barrier again only for a block whose operands-ready phase needs the
// element-wise threads to have seen the previous use of that buffer complete.
// The statistics warp of the dk/dv kernel, the third party to its QCONV barriers, waits for a stage's FREE barrier like the producer.  Of
// the six commits that it takes, the S issuer's follows QCONV's phase, and those of the second GEMMs follow both groups' READY, by which
// time the statistics have been read into registers.
// The element-wise threads read them after STFULL.  A commit orders tensor-core work, not another warp's ordinary stores, so the
// issuer of S, which has waited for QCONV, arrives on STFULL itself as well, after the commit that reports its MMAs (64x128 global,
// N = 8: 887 us without, 888 with it; a wait of the element-wise threads for QCONV costs 75 more).

// Lets a band kernel that was launched to follow this one (its programmatic dependent) take the SMs that the last blocks leave idle.
__device__ __forceinline__ void allow_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ uint32_t s32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// One lane of a whole warp, for the MMAs that one thread issues.  (With lane 0 picked by comparison the compiler does not know that
// one lane is left, and each tcgen05.mma takes 55 cycles to issue and the first eight of a batch 580, against 16 and 85.  It pays where
// many short MMAs are issued: 64x128 global, N = 8, dk/dv 971 : 880 us, a first-GEMM issuer busy 1230 of 1880 cycles per block before, 490 of
// 1630 now.  The forward kernel does without, at 457 us: with it in the P V issuers it would take 453, in the S issuer as well, whose
// 128-column MMAs keep the tensor core busy for 66 cycles each, 469.)
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(r));
    return r != 0;
}
__device__ __forceinline__ float ex2f(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float trunc19f(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

__device__ __forceinline__ void mb_init(uint32_t bar, uint32_t count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory"); }
__device__ __forceinline__ void mb_arrive(uint32_t bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory"); }
__device__ __forceinline__ void mb_expect(uint32_t bar, uint32_t bytes) { asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory"); }
// Bounded wait.  try_wait suspends the thread in hardware for up to the hinted time, so a waiting warp takes few issue
// slots from the warps that share its scheduler.  Once a wait has run out (`healthy` false) later waits give up at once.
__device__ __forceinline__ bool mb_wait_polls(uint32_t bar, uint32_t parity, int limit) {
    uint32_t done = 0;
    for (int it = 0; it < limit && !done; ++it)
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
                     : "=r"(done) : "r"(bar), "r"(parity), "r"(2000u) : "memory");
    return done != 0;
}
__device__ __forceinline__ bool mb_wait(uint32_t bar, uint32_t parity, bool healthy) {
    return mb_wait_polls(bar, parity, healthy ? WAIT2 : 4);
}
// A wait that has run out in one lane has run out for its warp: the element-wise warps go on to warp-collective instructions
// (tcgen05.ld / st, votes) and must leave their loops as one.  They agree while their TMEM loads are in flight (64x128 global, N = 8, us,
// without : with: forward 451 : 451, dq 498 : 500, dk/dv 875 : 885; directly after each wait dq takes 10 more).  The other roles
// issue nothing collective.
__device__ __forceinline__ bool all_lanes(bool ok) { return __all_sync(0xffffffffu, ok); }
__device__ __forceinline__ void tma_tile(uint32_t dst, const CUtensorMap* map, int col, int ring, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(dst), "l"(map), "r"(0), "r"(col), "r"(ring), "r"(bar) : "memory");
}
// K-major, 128-byte swizzle: rows of 128 bytes, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t desc_k(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3fff) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
__device__ __forceinline__ uint32_t idesc_tf32(int n) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(M2 >> 4) << 24);
}
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, {%5, %5, %5, %5}, p;\n\t}\n"
                 ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(0u));
}
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, {%5, %5, %5, %5}, p;\n\t}\n"
                 ::"r"(d), "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc), "r"(0u));
}
// byte offset of the 16-byte chunk c4 of row `row` in a K-major tile with 128-byte swizzle
__device__ __forceinline__ int sw_off(int row, int c4) { return row * 128 + ((c4 ^ (row & 7)) << 4); }
// Packed fp32 pairs (Blackwell f32x2 arithmetic: one instruction for two lanes of a 64-bit register pair); the element-wise
// loops are bound by issue slots, so halving their add / multiply / fma instructions pays.
__device__ __forceinline__ uint64_t pack2(float a, float b) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) { uint64_t d; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c)); return d; }
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) { uint64_t d; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) { uint64_t d; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; }
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) { uint64_t d; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; }
// hi = trunc19(x), lo = x - hi for four values, the subtractions as two packed instructions
__device__ __forceinline__ void split4(const float (&x)[4], float (&hi)[4], float (&lo)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) hi[i] = trunc19f(x[i]);
    unpack2(sub2(pack2(x[0], x[1]), pack2(hi[0], hi[1])), lo[0], lo[1]);
    unpack2(sub2(pack2(x[2], x[3]), pack2(hi[2], hi[3])), lo[2], lo[3]);
}
// x - trunc19(x) for the four components of a float4, as two packed subtractions
__device__ __forceinline__ float4 lo4p(const float4& x) {
    float4 r;
    unpack2(sub2(pack2(x.x, x.y), pack2(trunc19f(x.x), trunc19f(x.y))), r.x, r.y);
    unpack2(sub2(pack2(x.z, x.w), pack2(trunc19f(x.z), trunc19f(x.w))), r.z, r.w);
    return r;
}
// BF16 UMMA (K = 16 per instruction) for the two correction terms of a product at once: the 16 k-slots of a step hold
// [a_lo(8) | a_hi(8)] on the A side against [b_hi(8) ; b_lo(8)] on the B side, so one instruction adds a_lo*b_hi + a_hi*b_lo
// for 8 contraction indices.  The corrections are ~2^-11 of the product, so BF16's 8 bits leave ~2^-19 relative error:
// used by the backward kernels (gate 1e-4); the forward scores keep three TF32 products.  A step is 32 bytes, like a TF32 step.
__device__ __forceinline__ uint32_t idesc_bf16(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(M2 >> 4) << 24);
}
__device__ __forceinline__ void mma_ts16(uint32_t d, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, {%5, %5, %5, %5}, p;\n\t}\n"
                 ::"r"(d), "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc), "r"(0u));
}
// {low half = bf16(x0), high half = bf16(x1)}, round to nearest
__device__ __forceinline__ uint32_t bf16x2(float x0, float x1) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(x1), "f"(x0));
    return r;
}
// Stacked A operand in TMEM: per group of 8 channels, 4 words of lo pairs then 4 words of hi pairs (src: the 32 raw words).
__device__ __forceinline__ void pack_a16(const uint32_t (&src)[32], uint32_t (&dst)[32]) {
#pragma unroll
    for (int gq = 0; gq < 4; ++gq) {
        float hi[8], lo[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) { hi[i] = trunc19f(__uint_as_float(src[gq * 8 + i])); lo[i] = __uint_as_float(src[gq * 8 + i]) - hi[i]; }
#pragma unroll
        for (int i = 0; i < 4; ++i) { dst[gq * 8 + i] = bf16x2(lo[2 * i], lo[2 * i + 1]); dst[gq * 8 + 4 + i] = bf16x2(hi[2 * i], hi[2 * i + 1]); }
    }
}
// Stacked B tile beside a raw K-major tile: for point `row` and channel group `grp` (8 channels = the raw chunks 2 grp and
// 2 grp + 1) the chunk 2 grp receives the 8 hi parts and the chunk 2 grp + 1 the 8 lo parts, as BF16.
__device__ __forceinline__ void stack_b16(const unsigned char* raw, unsigned char* dst, int row, int grp) {
    const float4 a = *reinterpret_cast<const float4*>(raw + sw_off(row, 2 * grp)), b = *reinterpret_cast<const float4*>(raw + sw_off(row, 2 * grp + 1));
    const float x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    float hi[8], lo[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) hi[i] = trunc19f(x[i]);
#pragma unroll
    for (int i = 0; i < 8; i += 2) unpack2(sub2(pack2(x[i], x[i + 1]), pack2(hi[i], hi[i + 1])), lo[i], lo[i + 1]);
    *reinterpret_cast<uint4*>(dst + sw_off(row, 2 * grp)) = make_uint4(bf16x2(hi[0], hi[1]), bf16x2(hi[2], hi[3]), bf16x2(hi[4], hi[5]), bf16x2(hi[6], hi[7]));
    *reinterpret_cast<uint4*>(dst + sw_off(row, 2 * grp + 1)) = make_uint4(bf16x2(lo[0], lo[1]), bf16x2(lo[2], lo[3]), bf16x2(lo[4], lo[5]), bf16x2(lo[6], lo[7]));
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tm_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// issue only: the registers are valid after tm_ld_wait()
__device__ __forceinline__ void tm_ld32_issue(uint32_t (&r)[32], uint32_t addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]),"=r"(r[1]),"=r"(r[2]),"=r"(r[3]),"=r"(r[4]),"=r"(r[5]),"=r"(r[6]),"=r"(r[7]),"=r"(r[8]),"=r"(r[9]),"=r"(r[10]),"=r"(r[11]),"=r"(r[12]),"=r"(r[13]),"=r"(r[14]),"=r"(r[15]),
          "=r"(r[16]),"=r"(r[17]),"=r"(r[18]),"=r"(r[19]),"=r"(r[20]),"=r"(r[21]),"=r"(r[22]),"=r"(r[23]),"=r"(r[24]),"=r"(r[25]),"=r"(r[26]),"=r"(r[27]),"=r"(r[28]),"=r"(r[29]),"=r"(r[30]),"=r"(r[31]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void tm_ld16_issue(uint32_t (&r)[16], uint32_t addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]),"=r"(r[1]),"=r"(r[2]),"=r"(r[3]),"=r"(r[4]),"=r"(r[5]),"=r"(r[6]),"=r"(r[7]),"=r"(r[8]),"=r"(r[9]),"=r"(r[10]),"=r"(r[11]),"=r"(r[12]),"=r"(r[13]),"=r"(r[14]),"=r"(r[15]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void tm_st16(uint32_t addr, const uint32_t (&r)[16]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        :: "r"(addr), "r"(r[0]),"r"(r[1]),"r"(r[2]),"r"(r[3]),"r"(r[4]),"r"(r[5]),"r"(r[6]),"r"(r[7]),"r"(r[8]),"r"(r[9]),"r"(r[10]),"r"(r[11]),"r"(r[12]),"r"(r[13]),"r"(r[14]),"r"(r[15]) : "memory");
}
__device__ __forceinline__ void tm_st32(uint32_t addr, const uint32_t (&r)[32]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
        :: "r"(addr), "r"(r[0]),"r"(r[1]),"r"(r[2]),"r"(r[3]),"r"(r[4]),"r"(r[5]),"r"(r[6]),"r"(r[7]),"r"(r[8]),"r"(r[9]),"r"(r[10]),"r"(r[11]),"r"(r[12]),"r"(r[13]),"r"(r[14]),"r"(r[15]),
           "r"(r[16]),"r"(r[17]),"r"(r[18]),"r"(r[19]),"r"(r[20]),"r"(r[21]),"r"(r[22]),"r"(r[23]),"r"(r[24]),"r"(r[25]),"r"(r[26]),"r"(r[27]),"r"(r[28]),"r"(r[29]),"r"(r[30]),"r"(r[31]) : "memory");
}

__device__ __forceinline__ int fdiv(int a, int b) { const int q = a / b; return (a % b != 0 && ((a < 0) != (b < 0))) ? q - 1 : q; }
__device__ __forceinline__ int cdiv(int a, int b) { return -fdiv(-a, b); }

// Walks the blocks of partner points a tile needs.  The tile's list names partner rings, each with a window half width m
// in input columns (m < 0: the whole ring).  Partner points of a ring are addressed by an unwrapped index u (the point
// u mod period): the tile's rows together need u in [cdiv(a_lo - m, d), fdiv(a_hi + m, d)], where [a_lo, a_hi] are the
// centres of the first and last existing row and d converts input columns to partner points.  That range is cut where it
// crosses the ring's seam and each piece is covered by blocks of `step` points from its start, so a block never wraps:
// points of a block beyond the end of its piece (`seg_end`) either do not exist (TMA fills zeros) or belong to no row's
// window, and the element-wise code masks them.  Every role of a kernel walks the same sequence.
constexpr int M_WHOLE = 1 << 28;
// which turn of the ring the unwrapped index u lies in; the walks stay within (-period, 2 period) because a banded
// window is narrower than the ring
__device__ __forceinline__ int turn_of(int u, int period) { return (u >= period ? 1 : 0) - (u < 0 ? 1 : 0); }
struct TileWalk {
    const int32_t* lat;
    const int32_t* hw;
    int e, e_end, period, step, a_lo, a_hi, d;
    int ring, m, u, seg_end, uhi;        // current block: unwrapped start u, last wanted point of its piece seg_end
    __device__ __forceinline__ void load_entry() {
        if (e >= e_end) return;
        ring = lat[e];
        const int mm = hw[e];
        if (mm < 0) { m = M_WHOLE; u = 0; uhi = period - 1; }
        else if (d == 1) { m = mm; u = a_lo - mm; uhi = a_hi + mm; }
        else { m = mm; u = cdiv(a_lo - mm, d); uhi = fdiv(a_hi + mm, d); }
        seg_end = min(uhi, (turn_of(u, period) + 1) * period - 1);
    }
    __device__ __forceinline__ TileWalk(const int32_t* lat_, const int32_t* hw_, int e_begin, int e_end_, int period_, int step_,
                                        int a_lo_, int a_hi_, int d_)
        : lat(lat_), hw(hw_), e(e_begin), e_end(e_end_), period(period_), step(step_), a_lo(a_lo_), a_hi(a_hi_), d(d_),
          ring(0), m(0), u(0), seg_end(-1), uhi(-1) { load_entry(); }
    __device__ __forceinline__ int col() const { return u - turn_of(u, period) * period; }     // actual first point of the block
    __device__ __forceinline__ void advance() {
        u += step;
        if (u > seg_end) {
            u = seg_end + 1;                                  // a multiple of the period unless the ring is done
            if (u > uhi) { ++e; load_entry(); }
            else seg_end = min(uhi, u + period - 1);
        }
    }
};
// Number of blocks a TileWalk with the same arguments visits; called by one whole warp (entries spread over its lanes).
__device__ __forceinline__ int tile_block_count(const int32_t* lat, const int32_t* hw, int e_begin, int e_end, int period, int step,
                                                int a_lo, int a_hi, int d, int lane) {
    int cnt = 0;
    for (int e = e_begin + lane; e < e_end; e += 32) {
        const int mm = hw[e];
        int u = mm < 0 ? 0 : cdiv(a_lo - mm, d);
        const int uhi = mm < 0 ? period - 1 : fdiv(a_hi + mm, d);
        while (u <= uhi) {
            const int se = min(uhi, (turn_of(u, period) + 1) * period - 1);
            cnt += (se - u + step) / step;
            u = se + 1;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    return cnt;
}

// SPLIT: two instantiations of the second softmax pass, with and without the per-element window test, chosen per block.
// It pays when (nearly) every block is unmasked - plans whose windows are all whole rings: -4 % - and costs 2 % where
// masked and unmasked blocks alternate (the unrolled pass is long), so the launcher sets it for all-whole plans only.
template <bool SPLIT>
__global__ void __launch_bounds__(THREADS2, 1)
forward_dense2_kernel(DevPlan p, const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                      const __grid_constant__ CUtensorMap map_v, float* __restrict__ out, float* __restrict__ lse, int N,
                      float scale_log2, int tiles_per_row) {
    extern __shared__ unsigned char dense2_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)dense2_raw + 1023) & ~(uintptr_t)1023);
    __shared__ unsigned long long bars[B_COUNT];
    __shared__ uint32_t tmem_base_s;
    __shared__ int fail_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) allow_dependents();
    const int tile = blockIdx.x % tiles_per_row;
    const int rest = blockIdx.x / tiles_per_row;
    const int n = rest % N;
    const int h = p.dense_rows[rest / N];
    const int w0 = tile * M2;
    const int e_begin = p.dense_ptr[h], e_end = p.dense_ptr[h + 1];
    // the walk over this tile's blocks: centres of its first and last existing row, in input columns
    const int a_lo = p.ps * w0, a_hi = p.ps * (min(w0 + M2, p.nlon_out) - 1);
    __shared__ int total_s;
    if (warp == 1) {
        const int cnt = tile_block_count(p.dense_lat, p.dense_m, e_begin, e_end, p.nlon_in, BN2, a_lo, a_hi, 1, lane);
        if (lane == 0) total_s = cnt;
    }

    if (tid == 0) {
        for (int s = 0; s < 2; ++s) {
            mb_init(s32(&bars[B_KFULL + s]), 1);
            mb_init(s32(&bars[B_KCONV + s]), 128);
            mb_init(s32(&bars[B_KFREE + s]), 1);
            mb_init(s32(&bars[B_VFULL + s]), 1);
            mb_init(s32(&bars[B_VRAWFREE + s]), 128);
            mb_init(s32(&bars[B_VCONV + s]), 128);
            mb_init(s32(&bars[B_PVDONE + s]), 2);        // column half 0: two issuers
            mb_init(s32(&bars[B_PVDONE + 2 + s]), 2);    // column half 1
            mb_init(s32(&bars[B_SFULL + s]), 1);
            mb_init(s32(&bars[B_PREADY + s]), 128);      // column half 0, buffer s
            mb_init(s32(&bars[B_PREADY + 2 + s]), 128);  // column half 1, buffer s
        }
        mb_init(s32(&bars[B_QFULL]), 1);
        fail_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(&tmem_base_s)), "r"(T_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tm = tmem_base_s;
    const uint32_t sbase = s32(base);
    const int total = total_s;
    bool ok = true;

    if (warp < 8) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 152;");
        // ------------------------------------------------------------------ softmax: two groups of 128 threads; thread (half, r)
        // owns tile row r for the columns [64 half, 64 half + 64) of every block, with its own running maximum, sum and output
        const int half = warp >> 2, r = tid & 127;
        const uint32_t lanebits = (uint32_t)((warp & 3) * 32) << 16;
        const int w = w0 + r;
        const bool row_ok = w < p.nlon_out;
        constexpr int HC = BN2 / 2;                       // columns per thread and block
        float m = -INFINITY, l = 0.f, o[C2];
#pragma unroll
        for (int i = 0; i < C2; ++i) o[i] = 0.f;
        float corr_prev = 1.f;
        const int ctr = p.ps * w;                          // this row's window centre, in input columns
        TileWalk wk(p.dense_lat, p.dense_m, e_begin, e_end, p.nlon_in, BN2, a_lo, a_hi, 1);
        // folds P V of a block (this half's two partial results, fixed order); waiting for it also frees this half's P_lo columns and
        // accumulators
        auto fold = [&](int it) {
            ok = mb_wait(s32(&bars[B_PVDONE + 2 * half + (it & 1)]), (it >> 1) & 1, ok) && ok;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int c0 = 0; c0 < C2; c0 += 16) {
                uint32_t oa[16], ob[16];
                tm_ld16_issue(oa, tm + T_O + half * 64 + lanebits + c0);
                tm_ld16_issue(ob, tm + T_O + half * 64 + 32 + lanebits + c0);
                if (c0 == 0) ok = all_lanes(ok);
                tm_ld_wait();
#pragma unroll
                for (int j = 0; j < 16; j += 2)
                    unpack2(fma2(pack2(o[c0 + j], o[c0 + j + 1]), pack2(corr_prev, corr_prev),
                                 add2(pack2(__uint_as_float(oa[j]), __uint_as_float(oa[j + 1])), pack2(__uint_as_float(ob[j]), __uint_as_float(ob[j + 1])))),
                            o[c0 + j], o[c0 + j + 1]);
            }
        };
        int it = 0;
        for (; it < total && ok; ++it) {
            float corr = 1.f;
            const int b = it & 1, u = it >> 1;
            const float bias = p.log2_omega[wk.ring];
            // the columns [jl, jh] of this thread's half that exist and lie in this row's window
            int jl = max(0, ctr - wk.m - wk.u) - half * HC, jh = min(wk.seg_end - wk.u, ctr + wk.m - wk.u) - half * HC;
            if (!row_ok || jh < jl || jh < 0 || jl >= HC) { jl = HC; jh = HC; }     // none
            const uint32_t span = (uint32_t)(jh - jl);
            const bool full = __all_sync(0xffffffffu, jl <= 0 && jh >= HC - 1);     // no masking anywhere in this warp
            wk.advance();
            ok = mb_wait(s32(&bars[B_SFULL + b]), u & 1, ok) && ok;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t tS = tm + (b ? T_S1 : T_S0) + half * HC + lanebits;
            uint64_t ps2[2] = {pack2(0.f, 0.f), pack2(0.f, 0.f)};      // four running sums of P, as two packed pairs
            if constexpr (SPLIT) {
                // all-whole plans: the thread's 64 scores are loaded from TMEM once and stay in registers for both passes
                // pass 1: maximum of the raw scores (the scale is positive and the bias is the same for the whole block)
                uint32_t sq[4][16];
#pragma unroll
                for (int qd = 0; qd < 4; ++qd) tm_ld16_issue(sq[qd], tS + 16 * qd);
                ok = all_lanes(ok);
                tm_ld_wait();
                float mxr[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
                if (full) {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        mxr[j & 3] = fmaxf(mxr[j & 3], fmaxf(fmaxf(__uint_as_float(sq[0][j]), __uint_as_float(sq[1][j])),
                                                             fmaxf(__uint_as_float(sq[2][j]), __uint_as_float(sq[3][j]))));
                } else {
#pragma unroll
                    for (int qd = 0; qd < 4; ++qd)
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if ((uint32_t)(16 * qd + j - jl) <= span) mxr[j & 3] = fmaxf(mxr[j & 3], __uint_as_float(sq[qd][j]));
                }
                // (a half without any valid column keeps its state: exp2(-inf) = 0 below, and m stays -inf only if nothing was ever seen)
                const float mblk = fmaf(fmaxf(fmaxf(mxr[0], mxr[1]), fmaxf(mxr[2], mxr[3])), scale_log2, bias);
                if (it > 0) fold(it - 1);      // (not before the maximum: P V runs while it is found; 64x128, N = 8: 502 -> 457 us)
                const float mx = fmaxf(m, mblk);
                const float msafe = mx == -INFINITY ? 0.f : mx;
                corr = ex2f(m - msafe);
                m = mx;
                const float nb = bias - msafe;
                // pass 2: P over S (its top 19 bits are the hi part) and P_lo = P - trunc19(P) beside it
                auto pass2 = [&](auto unmasked) {
                    constexpr bool UNMASKED = decltype(unmasked)::value;
                    const uint64_t scale2 = pack2(scale_log2, scale_log2), nb2 = pack2(nb, nb);
#pragma unroll
                    for (int qd = 0; qd < 4; ++qd) {
                        uint32_t (&x)[16] = sq[qd];
                        const int c0 = 16 * qd;
                        uint32_t lo[16];
#pragma unroll
                        for (int j = 0; j < 16; j += 2) {
                            float x0, x1, l0, l1;
                            unpack2(fma2(pack2(__uint_as_float(x[j]), __uint_as_float(x[j + 1])), scale2, nb2), x0, x1);
                            float p0 = ex2f(x0), p1 = ex2f(x1);
                            if (!UNMASKED && !full && (uint32_t)(c0 + j - jl) > span) p0 = 0.f;
                            if (!UNMASKED && !full && (uint32_t)(c0 + j + 1 - jl) > span) p1 = 0.f;
                            const uint64_t p2 = pack2(p0, p1);
                            ps2[(j >> 1) & 1] = add2(ps2[(j >> 1) & 1], p2);
                            unpack2(sub2(p2, pack2(trunc19f(p0), trunc19f(p1))), l0, l1);
                            x[j] = __float_as_uint(p0); x[j + 1] = __float_as_uint(p1);
                            lo[j] = __float_as_uint(l0); lo[j + 1] = __float_as_uint(l1);
                        }
                        tm_st16(tS + c0, x);
                        tm_st16(tm + T_PLO + half * HC + lanebits + c0, lo);
                    }
                };
                if (SPLIT && full) pass2(std::true_type{}); else pass2(std::false_type{});
            } else {
                // plans with masked blocks: two loads per score (fewer live registers; measured 0.4 % faster there)
                // pass 1: maximum of the raw scores (the scale is positive and the bias is the same for the whole block)
                float mxr[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
                {
                    uint32_t sa[32], sb[32];
                    tm_ld32_issue(sa, tS);
                    tm_ld32_issue(sb, tS + 32);
                    ok = all_lanes(ok);
                    tm_ld_wait();
                    if (full) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) mxr[j & 3] = fmaxf(mxr[j & 3], fmaxf(__uint_as_float(sa[j]), __uint_as_float(sb[j])));
                    } else {
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            if ((uint32_t)(j - jl) <= span) mxr[j & 3] = fmaxf(mxr[j & 3], __uint_as_float(sa[j]));
                            if ((uint32_t)(32 + j - jl) <= span) mxr[j & 3] = fmaxf(mxr[j & 3], __uint_as_float(sb[j]));
                        }
                    }
                }
                // (a half without any valid column keeps its state: exp2(-inf) = 0 below, and m stays -inf only if nothing was ever seen)
                const float mblk = fmaf(fmaxf(fmaxf(mxr[0], mxr[1]), fmaxf(mxr[2], mxr[3])), scale_log2, bias);
                if (it > 0) fold(it - 1);
                const float mx = fmaxf(m, mblk);
                const float msafe = mx == -INFINITY ? 0.f : mx;
                corr = ex2f(m - msafe);
                m = mx;
                const float nb = bias - msafe;
                // pass 2: P over S (its top 19 bits are the hi part) and P_lo = P - trunc19(P) beside it
                auto pass2 = [&](auto unmasked) {
                    constexpr bool UNMASKED = decltype(unmasked)::value;
                    uint32_t bufa[16], bufb[16];
                    auto softmax16 = [&](uint32_t (&x)[16], int c0) {
                        uint32_t lo[16];
                        const uint64_t scale2 = pack2(scale_log2, scale_log2), nb2 = pack2(nb, nb);
#pragma unroll
                        for (int j = 0; j < 16; j += 2) {
                            float x0, x1, l0, l1;
                            unpack2(fma2(pack2(__uint_as_float(x[j]), __uint_as_float(x[j + 1])), scale2, nb2), x0, x1);
                            float p0 = ex2f(x0), p1 = ex2f(x1);
                            if (!UNMASKED && !full && (uint32_t)(c0 + j - jl) > span) p0 = 0.f;
                            if (!UNMASKED && !full && (uint32_t)(c0 + j + 1 - jl) > span) p1 = 0.f;
                            const uint64_t p2 = pack2(p0, p1);
                            ps2[(j >> 1) & 1] = add2(ps2[(j >> 1) & 1], p2);
                            unpack2(sub2(p2, pack2(trunc19f(p0), trunc19f(p1))), l0, l1);
                            x[j] = __float_as_uint(p0); x[j + 1] = __float_as_uint(p1);
                            lo[j] = __float_as_uint(l0); lo[j + 1] = __float_as_uint(l1);
                        }
                        tm_st16(tS + c0, x);
                        tm_st16(tm + T_PLO + half * HC + lanebits + c0, lo);
                    };
                    tm_ld16_issue(bufa, tS);
#pragma unroll
                    for (int c0 = 0; c0 < HC; c0 += 32) {
                        tm_ld_wait();
                        tm_ld16_issue(bufb, tS + c0 + 16);            // in flight while the first 16 columns are processed
                        softmax16(bufa, c0);
                        tm_ld_wait();
                        if (c0 + 32 < HC) tm_ld16_issue(bufa, tS + c0 + 32);
                        softmax16(bufb, c0 + 16);
                    }
                };
                if (SPLIT && full) pass2(std::true_type{}); else pass2(std::false_type{});
            }
            float ps[4];
            unpack2(ps2[0], ps[0], ps[1]);
            unpack2(ps2[1], ps[2], ps[3]);
            l = fmaf(l, corr, (ps[0] + ps[1]) + (ps[2] + ps[3]));
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mb_arrive(s32(&bars[B_PREADY + 2 * half + b]));
            corr_prev = corr;
        }
        if (total > 0 && ok) fold(total - 1);
        else if (it > 0) mb_wait_polls(s32(&bars[B_PVDONE + 2 * half + ((it - 1) & 1)]), ((it - 1) >> 1) & 1, WAIT2);      // P V under way
        // (here for the P V issuers too: a wait at the end of theirs cost 1 %, 451 : 455 us on 64x128 global, N = 8)
        // merge the two column halves of every row: half 1 hands its state over through shared memory
        float* xs = reinterpret_cast<float*>(base + OFF_K);         // [34][128] floats in the k stages, which are dead by now
        if (half == 1) {
#pragma unroll
            for (int j = 0; j < C2; ++j) xs[j * 128 + r] = o[j];
            xs[C2 * 128 + r] = m;
            xs[(C2 + 1) * 128 + r] = l;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");             // the two softmax groups only
        if (half == 0 && ok && row_ok) {
            const float m1 = xs[C2 * 128 + r], l1 = xs[(C2 + 1) * 128 + r];
            const float mm = fmaxf(m, m1);
            const float c0 = ex2f(m - mm), c1 = ex2f(m1 - mm);      // mm is finite: every existing row has a column in its window
            const float lt = l * c0 + l1 * c1;
            const size_t opt = (size_t)(n * p.nlat_out + h) * p.nlon_out + w;
            const float inv = 1.f / lt;
            float4* dst = reinterpret_cast<float4*>(out + opt * C2);
#pragma unroll
            for (int c4 = 0; c4 < C2 / 4; ++c4) {
                float rr[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) rr[i] = (o[4 * c4 + i] * c0 + xs[(4 * c4 + i) * 128 + r] * c1) * inv;
                dst[c4] = make_float4(rr[0], rr[1], rr[2], rr[3]);
            }
            if (lse != nullptr) lse[opt] = (mm + log2f(lt)) * LN2_2;
        }
    } else if (warp < 12) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
        // ------------------------------------------------------------------ TMA producer
        if (warp == 8 && lane == 0) {
            mb_expect(s32(&bars[B_QFULL]), TILE_B);
            tma_tile(sbase + OFF_Q, &map_q, w0, n * p.nlat_out + h, s32(&bars[B_QFULL]));
            TileWalk wk(p.dense_lat, p.dense_m, e_begin, e_end, p.nlon_in, BN2, a_lo, a_hi, 1);
            int it = 0;
            for (; it < total && ok; ++it, wk.advance()) {
                const int s = it & 1, u = it >> 1;
                const int hp = wk.ring;
                const int c0 = wk.col();
                if (u > 0) {
                    ok = mb_wait(s32(&bars[B_KFREE + s]), (u - 1) & 1, ok);
                    ok = mb_wait(s32(&bars[B_VRAWFREE + s]), (u - 1) & 1, ok) && ok;
                }
                if (!ok) break;
                mb_expect(s32(&bars[B_KFULL + s]), TILE_B);
                tma_tile(sbase + OFF_K + s * 2 * TILE_B, &map_k, c0, n * p.nlat_in + hp, s32(&bars[B_KFULL + s]));
                mb_expect(s32(&bars[B_VFULL + s]), TILE_B);
                tma_tile(sbase + OFF_VRAW + s * TILE_B, &map_v, c0, n * p.nlat_in + hp, s32(&bars[B_VFULL + s]));
            }
            ok = mb_wait_polls(s32(&bars[B_QFULL]), 0, WAIT2) && ok;
            for (int j = max(0, it - 2); j < it; ++j) {      // the copies under way
                ok = mb_wait_polls(s32(&bars[B_KFULL + j % 2]), (j / 2) & 1, WAIT2) && ok;
                ok = mb_wait_polls(s32(&bars[B_VFULL + j % 2]), (j / 2) & 1, WAIT2) && ok;
            }
        }
        // ------------------------------------------------------------------ S = Q K^T
        if (warp == 9 && lane == 0) {
            ok = mb_wait(s32(&bars[B_QFULL]), 0, ok);
            // q_lo is written by the converter warps before their first k tile: covered by KCONV of block 0
            const uint32_t idS = idesc_tf32(BN2);
            const uint64_t dq = desc_k(sbase + OFF_Q), dql = desc_k(sbase + OFF_QLO);
            int it = 0;
            for (; it < total && ok; ++it) {
                const int s = it & 1, u = it >> 1;
                ok = mb_wait(s32(&bars[B_KFULL + s]), u & 1, ok);
                ok = mb_wait(s32(&bars[B_KCONV + s]), u & 1, ok) && ok;
                if (u > 0) {   // P of block it-2 (in this S buffer) has been consumed by both column halves
                    ok = mb_wait(s32(&bars[B_PVDONE + s]), (u - 1) & 1, ok) && ok;
                    ok = mb_wait(s32(&bars[B_PVDONE + 2 + s]), (u - 1) & 1, ok) && ok;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t dk = desc_k(sbase + OFF_K + s * 2 * TILE_B), dkl = desc_k(sbase + OFF_K + s * 2 * TILE_B + TILE_B);
                const uint32_t tS = tm + (s ? T_S1 : T_S0);
#pragma unroll
                for (int ks = 0; ks < C2 / 8; ++ks) mma_ss(tS, dql + 2 * ks, dk + 2 * ks, idS, ks > 0);
#pragma unroll
                for (int ks = 0; ks < C2 / 8; ++ks) mma_ss(tS, dq + 2 * ks, dkl + 2 * ks, idS, 1);
#pragma unroll
                for (int ks = 0; ks < C2 / 8; ++ks) mma_ss(tS, dq + 2 * ks, dk + 2 * ks, idS, 1);
                mma_commit(s32(&bars[B_SFULL + s]));
                mma_commit(s32(&bars[B_KFREE + s]));
            }
            if (it > 0) ok = mb_wait_polls(s32(&bars[B_SFULL + ((it - 1) & 1)]), ((it - 1) >> 1) & 1, WAIT2) && ok;      // the MMAs under way
        }
    } else if (warp < 16) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
        // ------------------------------------------------------------------ O_part = P V over one quarter of the block's columns
        if (lane == 0) {
            const int part = warp - 12, half = part >> 1;
            constexpr int STEPS = BN2 / 8 / PV_ISSUERS;                              // 8-column steps per issuer
            const uint32_t idO = idesc_tf32(C2);
            const uint32_t tO = tm + T_O + part * 32;
            for (int it = 0; it < total && ok; ++it) {
                const int s = it & 1, u = it >> 1;
                ok = mb_wait(s32(&bars[B_VCONV + s]), u & 1, ok);
                ok = mb_wait(s32(&bars[B_PREADY + 2 * half + s]), u & 1, ok) && ok;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t tP = tm + (s ? T_S1 : T_S0), tPl = tm + T_PLO;
                const uint32_t vt = sbase + OFF_VT + s * 2 * TILE_B;
#pragma unroll
                for (int k8 = 0; k8 < STEPS; ++k8) {
                    const int ks = part * STEPS + k8;                               // 8-column step within the block
                    const uint32_t off = (uint32_t)(ks >> 2) * (C2 * 128) + (uint32_t)(ks & 3) * 32;
                    const uint64_t dvh = desc_k(vt + off), dvl = desc_k(vt + TILE_B + off);
                    mma_ts(tO, tPl + ks * 8, dvh, idO, k8 > 0);
                    mma_ts(tO, tP + ks * 8, dvl, idO, 1);
                    mma_ts(tO, tP + ks * 8, dvh, idO, 1);
                }
                mma_commit(s32(&bars[B_PVDONE + 2 * half + s]));
            }
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        // ------------------------------------------------------------------ converters (warps 16-19, 128 threads)
        const int ct = tid - 512, cw = ct >> 5;
        // q_lo once
        ok = mb_wait(s32(&bars[B_QFULL]), 0, ok);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int off = (j * 128 + ct) * 16;
            const float4 x = *reinterpret_cast<const float4*>(base + OFF_Q + off);
            *reinterpret_cast<float4*>(base + OFF_QLO + off) = lo4p(x);
        }
        for (int it = 0; it < total && ok; ++it) {
            const int s = it & 1, u = it >> 1;
            // k_lo: same swizzled position as the raw element
            ok = mb_wait(s32(&bars[B_KFULL + s]), u & 1, ok);
            unsigned char* kraw = base + OFF_K + s * 2 * TILE_B;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int off = (j * 128 + ct) * 16;
                const float4 x = *reinterpret_cast<const float4*>(kraw + off);
                *reinterpret_cast<float4*>(kraw + TILE_B + off) = lo4p(x);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mb_arrive(s32(&bars[B_KCONV + s]));
            // v transposed: this warp takes the 32 columns [32 cw, 32 cw + 32) (one K block of the transposed tiles), lane = channel
            ok = mb_wait(s32(&bars[B_VFULL + s]), u & 1, ok) && ok;
            if (u > 0) {   // the transposed tiles of block it-2 have been consumed by all four issuers
                ok = mb_wait(s32(&bars[B_PVDONE + s]), (u - 1) & 1, ok) && ok;
                ok = mb_wait(s32(&bars[B_PVDONE + 2 + s]), (u - 1) & 1, ok) && ok;
            }
            const unsigned char* vraw = base + OFF_VRAW + s * TILE_B;
            unsigned char* vth = base + OFF_VT + s * 2 * TILE_B + cw * (C2 * 128);
#pragma unroll
            for (int c8 = 0; c8 < 8; ++c8) {
                float x[4], hi[4], lo[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const float*>(vraw + sw_off(cw * 32 + c8 * 4 + i, lane >> 2) + (lane & 3) * 4);
                split4(x, hi, lo);
                *reinterpret_cast<float4*>(vth + sw_off(lane, c8)) = make_float4(hi[0], hi[1], hi[2], hi[3]);
                *reinterpret_cast<float4*>(vth + TILE_B + sw_off(lane, c8)) = make_float4(lo[0], lo[1], lo[2], lo[3]);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mb_arrive(s32(&bars[B_VRAWFREE + s]));
            mb_arrive(s32(&bars[B_VCONV + s]));
        }
    }
    if (!ok) atomicExch(&fail_s, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (fail_s && tid == 0) atomicExch(p.dev_status, 1);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"(T_COLS));
}

// ---------------------------------------------------------------------------------------------------------
// Pipelined dense part of the dq stage (App. B.4) for the whole input rings of an output ring:
//   p = exp2(s + log2 omega - lse),  ds = p (t - D),  dq += scale * dS K,   s = q.k (log2 domain),  t = dout.v.
// Same cast as the forward kernel, with blocks of 64 columns.  The tile's own operands (q, dout and their lo parts) live
// in TMEM for the whole kernel, so the two first GEMMs (S = Q K^T and T = dY V^T, one issuing thread each) read only
// the k / v blocks from shared memory.  Two groups of 128 threads turn (S, T) into dS (written over S, its top 19 bits
// are the hi part) and dS_lo (over T), each for one half of the block's columns; four threads issue dq_part = dS K over
// two 8-column steps each, into their own accumulators; the row's two threads add their parts in a fixed order and the
// two halves are merged at the end.  S and T are double-buffered, so the GEMMs of block j+1 overlap the element-wise
// work of block j and dS K of block j-1.
// ---------------------------------------------------------------------------------------------------------
constexpr int BNQ = 64;                          // columns per block
constexpr int TILE_Q = BNQ * 128;                // 8 KB: 64 points x 128 bytes
// per stage: k raw, k lo, v raw, v lo, k^T hi, k^T lo
constexpr int QST = 6 * TILE_Q;
constexpr int FOLDQ = 4;                         // dS K accumulates in TMEM over this many blocks before it is folded into registers
constexpr int NSQ = 4;                           // shared-memory stages (TMA runs three blocks ahead of the GEMMs)
constexpr size_t DQ2_SMEM = NSQ * QST + 1024;
constexpr int TQ_AQ = 0, TQ_AQL = 32, TQ_AY = 64, TQ_AYL = 96, TQ_BUF = 128 /* + 128 b: S | T */, TQ_ACC = 384 /* + 32 part */;
enum { Q_KFULL = 0, Q_VFULL = 4, Q_KCONV = 8, Q_VCONV = 12, Q_KSFREE = 16, Q_VFREE = 20, Q_KTFREE = 24 /* all [stage] */,
       Q_STFULL = 28 /* [buffer] */, Q_DSREADY = 30 /* [group][buffer] */, Q_G2DONE = 34 /* [group][buffer] */, Q_AREADY = 38, Q_COUNT = 39 };

__global__ void __launch_bounds__(THREADS2, 1)
backward_dq_dense2_kernel(DevPlan p, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                          const float* __restrict__ q, const float* __restrict__ dout, const float* __restrict__ out,
                          const float* __restrict__ lse, float* __restrict__ dq, float* __restrict__ Dws, int N, float scale,
                          int tiles_per_row) {
    extern __shared__ unsigned char dense2_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)dense2_raw + 1023) & ~(uintptr_t)1023);
    __shared__ unsigned long long bars[Q_COUNT];
    __shared__ uint32_t tmem_base_s;
    __shared__ int fail_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) allow_dependents();
    const int tile = blockIdx.x % tiles_per_row;
    const int rest = blockIdx.x / tiles_per_row;
    const int n = rest % N;
    const int h = p.dense_rows[rest / N];
    const int w0 = tile * M2;
    const int e_begin = p.dense_ptr[h], e_end = p.dense_ptr[h + 1];
    const int a_lo = p.ps * w0, a_hi = p.ps * (min(w0 + M2, p.nlon_out) - 1);     // see the forward kernel
    __shared__ int total_s;
    if (warp == 1) {
        const int cnt = tile_block_count(p.dense_lat, p.dense_m, e_begin, e_end, p.nlon_in, BNQ, a_lo, a_hi, 1, lane);
        if (lane == 0) total_s = cnt;
    }
    const float scale_log2 = scale * LOG2E_2;

    if (tid == 0) {
        for (int s = 0; s < NSQ; ++s) {
            mb_init(s32(&bars[Q_KFULL + s]), 1);
            mb_init(s32(&bars[Q_VFULL + s]), 1);
            mb_init(s32(&bars[Q_KCONV + s]), 128);
            mb_init(s32(&bars[Q_VCONV + s]), 128);
            mb_init(s32(&bars[Q_KSFREE + s]), 1);
            mb_init(s32(&bars[Q_VFREE + s]), 1);
            mb_init(s32(&bars[Q_KTFREE + s]), 4);
        }
        for (int s = 0; s < 2; ++s) {
            mb_init(s32(&bars[Q_STFULL + s]), 2);
            mb_init(s32(&bars[Q_DSREADY + s]), 128);          // group 0, buffer s
            mb_init(s32(&bars[Q_DSREADY + 2 + s]), 128);      // group 1, buffer s
            mb_init(s32(&bars[Q_G2DONE + s]), 2);
            mb_init(s32(&bars[Q_G2DONE + 2 + s]), 2);
        }
        mb_init(s32(&bars[Q_AREADY]), 128);
        fail_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(&tmem_base_s)), "r"(T_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tm = tmem_base_s;
    const uint32_t sbase = s32(base);
    const int total = total_s;
    bool ok = true;
    PROF_DECL

    if (warp < 8) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 152;");
        // ------------------------------------------------------------------ element-wise: thread (grp, r) owns tile row r for
        // the columns [32 grp, 32 grp + 32) of every block
        const int grp = warp >> 2, r = tid & 127;
        const uint32_t lanebits = (uint32_t)((warp & 3) * 32) << 16;
        const int w = w0 + r;
        const bool row_ok = w < p.nlon_out;
        const size_t opt = (size_t)(n * p.nlat_out + h) * p.nlon_out + min(w, p.nlon_out - 1);
        float D = 0.f;
        if (grp == 0) {
            // this row's q and dout into TMEM (A operands of the first GEMMs): raw words as hi parts, lo = x - trunc19(x)
            uint32_t xq[32], xy[32];
            const float4* qs = reinterpret_cast<const float4*>(q + opt * C2);
            const float4* ys = reinterpret_cast<const float4*>(dout + opt * C2);
            const float4* os = reinterpret_cast<const float4*>(out + opt * C2);
#pragma unroll
            for (int c4 = 0; c4 < C2 / 4; ++c4) {
                const float4 a = __ldg(qs + c4), b = __ldg(ys + c4), o4 = __ldg(os + c4);
                xq[4 * c4] = __float_as_uint(a.x); xq[4 * c4 + 1] = __float_as_uint(a.y); xq[4 * c4 + 2] = __float_as_uint(a.z); xq[4 * c4 + 3] = __float_as_uint(a.w);
                xy[4 * c4] = __float_as_uint(b.x); xy[4 * c4 + 1] = __float_as_uint(b.y); xy[4 * c4 + 2] = __float_as_uint(b.z); xy[4 * c4 + 3] = __float_as_uint(b.w);
                D = fmaf(b.x, o4.x, fmaf(b.y, o4.y, fmaf(b.z, o4.z, fmaf(b.w, o4.w, D))));
            }
            tm_st32(tm + TQ_AQ + lanebits, xq);
            tm_st32(tm + TQ_AY + lanebits, xy);
            {   // the stacked BF16 operands of the correction UMMAs
                uint32_t pk[32];
                pack_a16(xq, pk);
                tm_st32(tm + TQ_AQL + lanebits, pk);
                pack_a16(xy, pk);
                tm_st32(tm + TQ_AYL + lanebits, pk);
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mb_arrive(s32(&bars[Q_AREADY]));
            if (Dws != nullptr && row_ok) Dws[opt] = D;
        } else {
            const float4* ys = reinterpret_cast<const float4*>(dout + opt * C2);
            const float4* os = reinterpret_cast<const float4*>(out + opt * C2);
#pragma unroll
            for (int c4 = 0; c4 < C2 / 4; ++c4) {
                const float4 b = __ldg(ys + c4), o4 = __ldg(os + c4);
                D = fmaf(b.x, o4.x, fmaf(b.y, o4.y, fmaf(b.z, o4.z, fmaf(b.w, o4.w, D))));
            }
        }
        const float nl = -__ldg(lse + opt) * LOG2E_2;
        constexpr int GC = BNQ / 2;                       // columns per thread and block
        float acc[C2];
#pragma unroll
        for (int i = 0; i < C2; ++i) acc[i] = 0.f;
        const int ctr = p.ps * w;                          // this row's window centre, in input columns
        TileWalk wk(p.dense_lat, p.dense_m, e_begin, e_end, p.nlon_in, BNQ, a_lo, a_hi, 1);
        for (int it = 0; it <= total && ok; ++it) {
            if (it < total) {
                const int b = it & 1, u = it >> 1;
                const float nbias = p.log2_omega[wk.ring] + nl;
                // the columns [jl, jh] of this thread's half that exist and lie in this row's window
                int jl = max(0, ctr - wk.m - wk.u) - grp * GC, jh = min(wk.seg_end - wk.u, ctr + wk.m - wk.u) - grp * GC;
                if (!row_ok || jh < jl || jh < 0 || jl >= GC) { jl = GC; jh = GC; }     // none
                const uint32_t span = (uint32_t)(jh - jl);
                const bool full = __all_sync(0xffffffffu, jl <= 0 && jh >= GC - 1);     // no masking anywhere in this warp
                wk.advance();
                PROF_WAIT(0, ok = mb_wait(s32(&bars[Q_STFULL + b]), u & 1, ok) && ok);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t tS = tm + TQ_BUF + 128 * b + grp * GC + lanebits, tT = tS + BNQ;
                uint32_t sv[2][16], tv[2][16];      // two pieces: the first is stored while the second is worked on (64x128, N = 8: 518 -> 500 us)
#pragma unroll
                for (int i = 0; i < 2; ++i) { tm_ld16_issue(sv[i], tS + 16 * i); tm_ld16_issue(tv[i], tT + 16 * i); }
                ok = all_lanes(ok);
                tm_ld_wait();
                // (two instantiations: blocks in which no row of the warp is masked skip the per-element range test)
                auto elementwise = [&](auto unmasked) {
                    constexpr bool UNMASKED = decltype(unmasked)::value;
                    const uint64_t scale2 = pack2(scale_log2, scale_log2), nbias2 = pack2(nbias, nbias), D2 = pack2(D, D);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
#pragma unroll
                        for (int j = 0; j < 16; j += 2) {
                            float x0, x1, ds0, ds1, l0, l1;
                            unpack2(fma2(pack2(__uint_as_float(sv[i][j]), __uint_as_float(sv[i][j + 1])), scale2, nbias2), x0, x1);
                            float p0 = ex2f(x0), p1 = ex2f(x1);
                            if (!UNMASKED && (uint32_t)(16 * i + j - jl) > span) p0 = 0.f;
                            if (!UNMASKED && (uint32_t)(16 * i + j + 1 - jl) > span) p1 = 0.f;
                            const uint64_t ds2 = mul2(pack2(p0, p1), sub2(pack2(__uint_as_float(tv[i][j]), __uint_as_float(tv[i][j + 1])), D2));
                            unpack2(ds2, ds0, ds1);
                            unpack2(sub2(ds2, pack2(trunc19f(ds0), trunc19f(ds1))), l0, l1);
                            sv[i][j] = __float_as_uint(ds0); sv[i][j + 1] = __float_as_uint(ds1);       // dS over S
                            tv[i][j] = __float_as_uint(l0); tv[i][j + 1] = __float_as_uint(l1);         // dS_lo over T
                        }
                        tm_st16(tS + 16 * i, sv[i]);
                        tm_st16(tT + 16 * i, tv[i]);
                    }
                };
                if (full) elementwise(std::true_type{}); else elementwise(std::false_type{});
            }
            if (it > 0 && (it % FOLDQ == 0 || it == total)) {
                // fold dS K of the blocks since the last fold (this half's two parts, fixed order): the tensor core has
                // accumulated them in TMEM (chains of at most 6 * FOLDQ products); this also frees the accumulators
                const int bp = (it - 1) & 1, up = (it - 1) >> 1;
                PROF_WAIT(1, ok = mb_wait(s32(&bars[Q_G2DONE + 2 * grp + bp]), up & 1, ok) && ok);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                uint32_t oa[32], ob[32];
                tm_ld32_issue(oa, tm + TQ_ACC + grp * 64 + lanebits);
                tm_ld32_issue(ob, tm + TQ_ACC + grp * 64 + 32 + lanebits);
                ok = all_lanes(ok);
                tm_ld_wait();
#pragma unroll
                for (int j = 0; j < C2; j += 2)
                    unpack2(add2(pack2(acc[j], acc[j + 1]), add2(pack2(__uint_as_float(oa[j]), __uint_as_float(oa[j + 1])),
                                                                 pack2(__uint_as_float(ob[j]), __uint_as_float(ob[j + 1])))), acc[j], acc[j + 1]);
            }
            if (it < total) {
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                mb_arrive(s32(&bars[Q_DSREADY + 2 * grp + (it & 1)]));
            }
        }
        // merge the two column halves of every row through shared memory.  The staging tiles are reused for that, so the
        // OTHER group's second GEMMs, which may still be reading k^T tiles, must have finished too (a thread's last fold
        // only waited for its own group's).
        if (total > 0) ok = mb_wait(s32(&bars[Q_G2DONE + 2 * (grp ^ 1) + ((total - 1) & 1)]), ((total - 1) >> 1) & 1, ok) && ok;
        float* xs = reinterpret_cast<float*>(base);
        if (grp == 1) {
#pragma unroll
            for (int j = 0; j < C2; ++j) xs[j * 128 + r] = acc[j];
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (grp == 0 && ok && row_ok) {
            float4* dst = reinterpret_cast<float4*>(dq + opt * C2);
#pragma unroll
            for (int c4 = 0; c4 < C2 / 4; ++c4) {
                float rr[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) rr[i] = (acc[4 * c4 + i] + xs[(4 * c4 + i) * 128 + r]) * scale;
                dst[c4] = make_float4(rr[0], rr[1], rr[2], rr[3]);
            }
        }
    } else if (warp < 12) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
        if (warp == 8 && lane == 0) {
            // -------------------------------------------------------------- TMA producer
            TileWalk wk(p.dense_lat, p.dense_m, e_begin, e_end, p.nlon_in, BNQ, a_lo, a_hi, 1);
            int it = 0;
            for (; it < total && ok; ++it, wk.advance()) {
                const int s = it % NSQ, u = it / NSQ;
                const int hp = wk.ring;
                const int c0 = wk.col();
                if (u > 0) {   // the stage is free once both first GEMMs and all four dS K issuers of block it-NSQ are done
                    PROF_WAIT(0, ok = mb_wait(s32(&bars[Q_KSFREE + s]), (u - 1) & 1, ok));
                    PROF_WAIT(1, ok = mb_wait(s32(&bars[Q_VFREE + s]), (u - 1) & 1, ok) && ok);
                    PROF_WAIT(2, ok = mb_wait(s32(&bars[Q_KTFREE + s]), (u - 1) & 1, ok) && ok);
                }
                if (!ok) break;
                mb_expect(s32(&bars[Q_KFULL + s]), TILE_Q);
                tma_tile(sbase + s * QST, &map_k, c0, n * p.nlat_in + hp, s32(&bars[Q_KFULL + s]));
                mb_expect(s32(&bars[Q_VFULL + s]), TILE_Q);
                tma_tile(sbase + s * QST + 2 * TILE_Q, &map_v, c0, n * p.nlat_in + hp, s32(&bars[Q_VFULL + s]));
            }
            for (int j = max(0, it - NSQ); j < it; ++j) {      // the copies under way
                ok = mb_wait_polls(s32(&bars[Q_KFULL + j % NSQ]), (j / NSQ) & 1, WAIT2) && ok;
                ok = mb_wait_polls(s32(&bars[Q_VFULL + j % NSQ]), (j / NSQ) & 1, WAIT2) && ok;
            }
        }
        if ((warp == 9 || warp == 10) && elect_one()) {
            // -------------------------------------------------------------- S = Q K^T (warp 9) and T = dY V^T (warp 10)
            const bool isT = warp == 10;
            ok = mb_wait(s32(&bars[Q_AREADY]), 0, ok);
            const uint32_t idS = idesc_tf32(BNQ), idS16 = idesc_bf16(BNQ);
            const uint32_t tA = tm + (isT ? TQ_AY : TQ_AQ), tAl = tm + (isT ? TQ_AYL : TQ_AQL);
            int it = 0;
            for (; it < total && ok; ++it) {
                const int s = it % NSQ, us = it / NSQ, b = it & 1, u = it >> 1;
                PROF_WAIT(0, ok = mb_wait(s32(&bars[(isT ? Q_VFULL : Q_KFULL) + s]), us & 1, ok));
                PROF_WAIT(1, ok = mb_wait(s32(&bars[(isT ? Q_VCONV : Q_KCONV) + s]), us & 1, ok) && ok);
                if (u > 0) {   // dS / dS_lo of block it-2 (in this buffer) have been consumed by all four dS K issuers
                    PROF_WAIT(2, ok = mb_wait(s32(&bars[Q_G2DONE + b]), (u - 1) & 1, ok) && ok);
                    PROF_WAIT(2, ok = mb_wait(s32(&bars[Q_G2DONE + 2 + b]), (u - 1) & 1, ok) && ok);
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t tile0 = sbase + s * QST + (isT ? 2 * TILE_Q : 0);
                const uint64_t db = desc_k(tile0), dbl = desc_k(tile0 + TILE_Q);
                const uint32_t tD = tm + TQ_BUF + 128 * b + (isT ? BNQ : 0);
#pragma unroll
                for (int ks = 0; ks < C2 / 8; ++ks) mma_ts16(tD, tAl + ks * 8, dbl + 2 * ks, idS16, ks > 0);     // a_lo b_hi + a_hi b_lo
#pragma unroll
                for (int ks = 0; ks < C2 / 8; ++ks) mma_ts(tD, tA + ks * 8, db + 2 * ks, idS, 1);
                mma_commit(s32(&bars[Q_STFULL + b]));
                mma_commit(s32(&bars[(isT ? Q_VFREE : Q_KSFREE) + s]));
            }
            if (it > 0) ok = mb_wait_polls(s32(&bars[Q_STFULL + ((it - 1) & 1)]), ((it - 1) >> 1) & 1, WAIT2) && ok;      // the MMAs under way
        }
    } else if (warp < 16) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
        // ------------------------------------------------------------------ dq_part = dS K over two 8-column steps
        if (elect_one()) {
            const int part = warp - 12, grp = part >> 1;
            const uint32_t idO = idesc_tf32(C2);
            const uint32_t tO = tm + TQ_ACC + part * 32;
            int it = 0;
            for (; it < total && ok; ++it) {
                const int s = it % NSQ, us = it / NSQ, b = it & 1;
                PROF_WAIT(0, ok = mb_wait(s32(&bars[Q_KCONV + s]), us & 1, ok));
                PROF_WAIT(1, ok = mb_wait(s32(&bars[Q_DSREADY + 2 * grp + b]), (it >> 1) & 1, ok) && ok);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t tS = tm + TQ_BUF + 128 * b, tT = tS + BNQ;
                const uint32_t kt = sbase + s * QST + 4 * TILE_Q;
#pragma unroll
                for (int k8 = 0; k8 < 2; ++k8) {
                    const int ks = part * 2 + k8;                                   // 8-column step within the block
                    const uint32_t off = (uint32_t)(ks >> 2) * (C2 * 128) + (uint32_t)(ks & 3) * 32;
                    const uint64_t dkh = desc_k(kt + off), dkl = desc_k(kt + TILE_Q + off);
                    mma_ts(tO, tT + ks * 8, dkh, idO, (k8 > 0) || (it % FOLDQ != 0));
                    mma_ts(tO, tS + ks * 8, dkl, idO, 1);
                    mma_ts(tO, tS + ks * 8, dkh, idO, 1);
                }
                mma_commit(s32(&bars[Q_G2DONE + 2 * grp + b]));
                mma_commit(s32(&bars[Q_KTFREE + s]));
            }
            if (it > 0) ok = mb_wait_polls(s32(&bars[Q_G2DONE + 2 * grp + ((it - 1) & 1)]), ((it - 1) >> 1) & 1, WAIT2) && ok;      // the MMAs under way
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        // ------------------------------------------------------------------ converters (warps 16-19, 128 threads)
        const int ct = tid - 512, cw = ct >> 5;
        for (int it = 0; it < total && ok; ++it) {
            const int s = it % NSQ, u = it / NSQ;
            unsigned char* st = base + s * QST;
            // k_lo (same swizzled position as the raw element) and k transposed: warp cw takes the 16 columns [16 cw, 16 cw + 16),
            // lane = channel
            PROF_WAIT(0, ok = mb_wait(s32(&bars[Q_KFULL + s]), u & 1, ok));
#pragma unroll
            for (int j = 0; j < BNQ * 4 / 128; ++j) stack_b16(st, st + TILE_Q, (j * 128 + ct) >> 2, ct & 3);
            {
                unsigned char* kth = st + 4 * TILE_Q + (cw >> 1) * (C2 * 128);
#pragma unroll
                for (int c8 = 0; c8 < 4; ++c8) {
                    float x[4], hi[4], lo[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const float*>(st + sw_off(cw * 16 + c8 * 4 + i, lane >> 2) + (lane & 3) * 4);
                    split4(x, hi, lo);
                    const int chunk = (cw & 1) * 4 + c8;
                    *reinterpret_cast<float4*>(kth + sw_off(lane, chunk)) = make_float4(hi[0], hi[1], hi[2], hi[3]);
                    *reinterpret_cast<float4*>(kth + TILE_Q + sw_off(lane, chunk)) = make_float4(lo[0], lo[1], lo[2], lo[3]);
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mb_arrive(s32(&bars[Q_KCONV + s]));
            // v_lo
            PROF_WAIT(1, ok = mb_wait(s32(&bars[Q_VFULL + s]), u & 1, ok) && ok);
#pragma unroll
            for (int j = 0; j < BNQ * 4 / 128; ++j) stack_b16(st + 2 * TILE_Q, st + 3 * TILE_Q, (j * 128 + ct) >> 2, ct & 3);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mb_arrive(s32(&bars[Q_VCONV + s]));
        }
    }
    if (!ok) atomicExch(&fail_s, 1);
    PROF_DUMP(p.dev_status, warp, lane, total)
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (fail_s && tid == 0) atomicExch(p.dev_status, 1);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"(T_COLS));
}

// ---------------------------------------------------------------------------------------------------------
// Pipelined dense part of the dk/dv stage (App. B.4), transposed roles: a block owns 128 consecutive input columns of
// an input ring (tile row = input point j, its k and v rows and their lo parts live in TMEM) and walks, in blocks of 32,
// the output points i of the output rings that attend to this input ring:
//   S^T = K Q^T, T^T = V dY^T (one issuing thread each);  p = exp2(s + log2 omega_j - lse_i),  ds = p (t - D_i);
//   dV += P dY,  dK += scale * dS Q   (A operands P, dS from TMEM; B operands: q and dout blocks transposed by the converters).
// Two groups of 128 threads do the element-wise work for one half of the block's columns each and write P over S^T, dS
// over T^T and the two lo parts beside them; one warp fetches the partner points' statistics, two groups of converters prepare the q and
// the dout blocks; four threads issue the second GEMMs (dV or dK, one column half each) into their own accumulators, which collect FOLDK
// blocks in TMEM before the row's threads fold them into registers.  (One group of converters for both arrays, with the statistics'
// latency in it, was busy 1600 of the 1880 cycles that a block took.  64x128 global, N = 8: 1010 us then, 880 with the second group, the
// statistics warp and the elected issuers; without the second group alone 950, without the statistics warp alone 952, without the
// elected issuers alone 971.)  TMEM:
// 128 columns of fixed operands, two buffers of 128 (S^T, T^T, P_lo, dS_lo of 32 columns each) and 128 of accumulators.
// With two buffers the first GEMMs of block j+1 run while the element-wise threads work on block j and the second
// GEMMs on block j-1 (blocks of 64 points leave room for one buffer only, which serialised the three phases); TMA and
// the converters run up to four blocks ahead.
// ---------------------------------------------------------------------------------------------------------
constexpr int BNK = 32;                          // partner points per block
constexpr int TILE_K = BNK * 128;                // 4 KB
constexpr int FOLDK = 8;
constexpr int NSK = 5;                           // shared-memory stages
// per stage: q raw, q lo, y raw, y lo, q^T hi, q^T lo, y^T hi, y^T lo, then log2 omega - lse*log2e and D of the 32 partner points
constexpr int KST = 8 * TILE_K + 1024;
constexpr size_t DKDV2_SMEM = NSK * KST + 1024;
constexpr int TK_AK = 0, TK_AKL = 32, TK_AV = 64, TK_AVL = 96, TK_BUF = 128 /* + 128 b: S | T | P_lo | dS_lo, 32 columns each */, TK_ACC = 384 /* + 32 part */;
constexpr int TK_S = 0, TK_T = 32, TK_PLO = 64, TK_DSLO = 96;      // offsets inside a buffer
enum { K_QFULL = 0, K_YFULL = NSK, K_QCONV = 2 * NSK, K_YCONV = 3 * NSK, K_FREE = 4 * NSK /* all [stage] */, K_STFULL = 5 * NSK /* [buffer] */,
       K_READY = 5 * NSK + 2 /* [group][buffer] */, K_G2DONE = 5 * NSK + 6 /* [group][buffer] */, K_AREADY = 5 * NSK + 10, K_COUNT = 5 * NSK + 11 };

__global__ void __launch_bounds__(THREADS_DKDV, 1)
backward_dkdv_dense2_kernel(DevPlan p, const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_y,
                            const float* __restrict__ k, const float* __restrict__ v, const float* __restrict__ lse,
                            const float* __restrict__ Dws, float* __restrict__ dk, float* __restrict__ dv, int N, float scale,
                            int tiles_per_row) {
    extern __shared__ unsigned char dense2_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)dense2_raw + 1023) & ~(uintptr_t)1023);
    __shared__ unsigned long long bars[K_COUNT];
    __shared__ uint32_t tmem_base_s;
    __shared__ int fail_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) allow_dependents();
    const int tile = blockIdx.x % tiles_per_row;
    const int rest = blockIdx.x / tiles_per_row;
    const int n = rest % N;
    const int hp = p.t_dense_rows[rest / N];
    const int c0 = tile * M2;
    const int e_begin = p.t_dense_ptr[hp], e_end = p.t_dense_ptr[hp + 1];
    // the walk over this tile's blocks of output points: rows are the input columns [a_lo, a_hi]; output point w is a
    // partner of column c iff |ps w - c| <= m, so the walk runs over w with d = ps
    const int a_lo = c0, a_hi = min(c0 + M2, p.nlon_in) - 1;
    __shared__ int total_s;
    if (warp == 1) {
        const int cnt = tile_block_count(p.t_dense_lat, p.t_dense_m, e_begin, e_end, p.nlon_out, BNK, a_lo, a_hi, p.ps, lane);
        if (lane == 0) total_s = cnt;
    }
    const float scale_log2 = scale * LOG2E_2;

    if (tid == 0) {
        for (int s = 0; s < NSK; ++s) {
            mb_init(s32(&bars[K_QFULL + s]), 1);
            mb_init(s32(&bars[K_YFULL + s]), 1);
            mb_init(s32(&bars[K_QCONV + s]), 128 + 32);      // converters, statistics
            mb_init(s32(&bars[K_YCONV + s]), 128);
            mb_init(s32(&bars[K_FREE + s]), 6);         // both first GEMMs and the four second-GEMM issuers
        }
        for (int g = 0; g < 2; ++g) {
            mb_init(s32(&bars[K_STFULL + g]), 3);            // buffer g: both first GEMMs, the statistics
            mb_init(s32(&bars[K_READY + 2 * g]), 128);       // group g, buffer 0
            mb_init(s32(&bars[K_READY + 2 * g + 1]), 128);   // group g, buffer 1
            mb_init(s32(&bars[K_G2DONE + 2 * g]), 2);        // group g, buffer 0: its dV and dK issuers
            mb_init(s32(&bars[K_G2DONE + 2 * g + 1]), 2);    // group g, buffer 1
        }
        mb_init(s32(&bars[K_AREADY]), 128);
        fail_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(&tmem_base_s)), "r"(T_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tm = tmem_base_s;
    const uint32_t sbase = s32(base);
    const int total = total_s;
    bool ok = true;
    PROF_DECL

    if (warp < 8) {
        // register budget of the block: 768 threads x 80 at launch; a warpgroup can only grow by what the others give back:
        // 256 x 152 + 256 x 32 + 256 x 56 = 61440
        asm volatile("setmaxnreg.inc.sync.aligned.u32 152;");
        // ------------------------------------------------------------------ element-wise: thread (grp, r) owns tile row r (an
        // input point) for the partner columns [16 grp, 16 grp + 16) of every block
        const int grp = warp >> 2, r = tid & 127;
        const uint32_t lanebits = (uint32_t)((warp & 3) * 32) << 16;
        const int c = c0 + r;
        const bool row_ok = c < p.nlon_in;
        const size_t ipt = (size_t)(n * p.nlat_in + hp) * p.nlon_in + min(c, p.nlon_in - 1);
        if (grp == 0) {
            // this row's k and v into TMEM (A operands of the first GEMMs): raw words as hi parts, lo = x - trunc19(x)
            uint32_t xk[32], xv[32];
            const float4* ks = reinterpret_cast<const float4*>(k + ipt * C2);
            const float4* vs = reinterpret_cast<const float4*>(v + ipt * C2);
#pragma unroll
            for (int c4 = 0; c4 < C2 / 4; ++c4) {
                const float4 a = __ldg(ks + c4), b = __ldg(vs + c4);
                xk[4 * c4] = __float_as_uint(a.x); xk[4 * c4 + 1] = __float_as_uint(a.y); xk[4 * c4 + 2] = __float_as_uint(a.z); xk[4 * c4 + 3] = __float_as_uint(a.w);
                xv[4 * c4] = __float_as_uint(b.x); xv[4 * c4 + 1] = __float_as_uint(b.y); xv[4 * c4 + 2] = __float_as_uint(b.z); xv[4 * c4 + 3] = __float_as_uint(b.w);
            }
            tm_st32(tm + TK_AK + lanebits, xk);
            tm_st32(tm + TK_AV + lanebits, xv);
            {   // the stacked BF16 operands of the correction UMMAs
                uint32_t pk[32];
                pack_a16(xk, pk);
                tm_st32(tm + TK_AKL + lanebits, pk);
                pack_a16(xv, pk);
                tm_st32(tm + TK_AVL + lanebits, pk);
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mb_arrive(s32(&bars[K_AREADY]));
        }
        constexpr int GC = BNK / 2;                       // columns per thread and block
        float gk[C2], gv[C2];
#pragma unroll
        for (int i = 0; i < C2; ++i) { gk[i] = 0.f; gv[i] = 0.f; }
        TileWalk wk(p.t_dense_lat, p.t_dense_m, e_begin, e_end, p.nlon_out, BNK, a_lo, a_hi, p.ps);
        const int ps_shift = (p.ps & (p.ps - 1)) == 0 ? 31 - __clz(p.ps) : -1;      // ps a power of two: divide by shifting
        for (int it = 0; it <= total && ok; ++it) {
            if (it > 0 && (it % FOLDK == 0 || it == total)) {
                // fold the second GEMMs of the blocks since the last fold; this also frees the accumulators
                PROF_WAIT(1, ok = mb_wait(s32(&bars[K_G2DONE + 2 * grp + ((it - 1) & 1)]), ((it - 1) >> 1) & 1, ok) && ok);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                uint32_t oa[32], ob[32];
                tm_ld32_issue(oa, tm + TK_ACC + grp * 32 + lanebits);          // dV, this column half
                tm_ld32_issue(ob, tm + TK_ACC + 64 + grp * 32 + lanebits);     // dK, this column half
                ok = all_lanes(ok);
                tm_ld_wait();
#pragma unroll
                for (int j = 0; j < C2; j += 2) {
                    unpack2(add2(pack2(gv[j], gv[j + 1]), pack2(__uint_as_float(oa[j]), __uint_as_float(oa[j + 1]))), gv[j], gv[j + 1]);
                    unpack2(add2(pack2(gk[j], gk[j + 1]), pack2(__uint_as_float(ob[j]), __uint_as_float(ob[j + 1]))), gk[j], gk[j + 1]);
                }
            }
            if (it < total) {
                const int s = it % NSK, b = it & 1;
                // the partner columns [jl, jh] of this thread's half that exist and have this row's input point in their window
                const int wl = ps_shift >= 0 ? -((wk.m - c) >> ps_shift) : cdiv(c - wk.m, p.ps);      // ceil((c - m) / ps)
                const int wh = ps_shift >= 0 ? (c + wk.m) >> ps_shift : fdiv(c + wk.m, p.ps);         // floor((c + m) / ps)
                int jl = max(0, wl - wk.u) - grp * GC, jh = min(wk.seg_end - wk.u, wh - wk.u) - grp * GC;
                if (!row_ok || jh < jl || jh < 0 || jl >= GC) { jl = GC; jh = GC; }     // none
                const uint32_t span = (uint32_t)(jh - jl);
                const bool full = __all_sync(0xffffffffu, jl <= 0 && jh >= GC - 1);     // no masking anywhere in this warp
                wk.advance();
                PROF_WAIT(0, ok = mb_wait(s32(&bars[K_STFULL + b]), (it >> 1) & 1, ok) && ok);     // and the statistics of this stage (see the barrier list)
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const float* nlc = reinterpret_cast<const float*>(base + s * KST + 8 * TILE_K) + grp * GC;
                const float* Dc = nlc + BNK;
                const uint32_t tB = tm + TK_BUF + 128 * b + grp * GC + lanebits;
                const uint32_t tS = tB + TK_S, tT = tB + TK_T, tPl = tB + TK_PLO, tDl = tB + TK_DSLO;
                {
                    constexpr int hf = 0;
                    uint32_t sv[16], tv[16], pl[16], dl[16];
                    tm_ld16_issue(sv, tS + hf * 16);
                    tm_ld16_issue(tv, tT + hf * 16);
                    // the per-column statistics of this thread's 16 columns, as 16-byte loads while the TMEM loads are in flight
                    float nlv[16], Dv[16];
#pragma unroll
                    for (int q4 = 0; q4 < 4; ++q4) {
                        const float4 a = reinterpret_cast<const float4*>(nlc)[q4], d4 = reinterpret_cast<const float4*>(Dc)[q4];
                        nlv[4 * q4] = a.x; nlv[4 * q4 + 1] = a.y; nlv[4 * q4 + 2] = a.z; nlv[4 * q4 + 3] = a.w;
                        Dv[4 * q4] = d4.x; Dv[4 * q4 + 1] = d4.y; Dv[4 * q4 + 2] = d4.z; Dv[4 * q4 + 3] = d4.w;
                    }
                    ok = all_lanes(ok);
                    tm_ld_wait();
                    // (two instantiations: blocks in which no row of the warp is masked skip the per-element range test)
                    auto elementwise = [&](auto unmasked) {
                        constexpr bool UNMASKED = decltype(unmasked)::value;
                        const uint64_t scale2 = pack2(scale_log2, scale_log2);
#pragma unroll
                        for (int j = 0; j < 16; j += 2) {
                            const int col = hf * 16 + j;
                            float x0, x1, ds0, ds1, a0, a1, b0, b1;
                            unpack2(fma2(pack2(__uint_as_float(sv[j]), __uint_as_float(sv[j + 1])), scale2, pack2(nlv[j], nlv[j + 1])), x0, x1);
                            float p0 = ex2f(x0), p1 = ex2f(x1);
                            if (!UNMASKED && (uint32_t)(col - jl) > span) p0 = 0.f;
                            if (!UNMASKED && (uint32_t)(col + 1 - jl) > span) p1 = 0.f;
                            const uint64_t p2 = pack2(p0, p1);
                            const uint64_t ds2 = mul2(p2, sub2(pack2(__uint_as_float(tv[j]), __uint_as_float(tv[j + 1])), pack2(Dv[j], Dv[j + 1])));
                            unpack2(ds2, ds0, ds1);
                            unpack2(sub2(p2, pack2(trunc19f(p0), trunc19f(p1))), a0, a1);
                            unpack2(sub2(ds2, pack2(trunc19f(ds0), trunc19f(ds1))), b0, b1);
                            sv[j] = __float_as_uint(p0); sv[j + 1] = __float_as_uint(p1);
                            tv[j] = __float_as_uint(ds0); tv[j + 1] = __float_as_uint(ds1);
                            pl[j] = __float_as_uint(a0); pl[j + 1] = __float_as_uint(a1);
                            dl[j] = __float_as_uint(b0); dl[j + 1] = __float_as_uint(b1);
                        }
                    };
                    if (full) elementwise(std::true_type{}); else elementwise(std::false_type{});
                    tm_st16(tS + hf * 16, sv);
                    tm_st16(tT + hf * 16, tv);
                    tm_st16(tPl + hf * 16, pl);
                    tm_st16(tDl + hf * 16, dl);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                mb_arrive(s32(&bars[K_READY + 2 * grp + b]));
            }
        }
        // merge the two column halves of every row through shared memory.  The staging tiles are reused for that, so the
        // OTHER group's second GEMMs, which may still be reading q^T / y^T tiles, must have finished too (a thread's last
        // fold only waited for its own group's).
        if (total > 0) ok = mb_wait(s32(&bars[K_G2DONE + 2 * (grp ^ 1) + ((total - 1) & 1)]), ((total - 1) >> 1) & 1, ok) && ok;
        float* xs = reinterpret_cast<float*>(base);
        if (grp == 1) {
#pragma unroll
            for (int j = 0; j < C2; ++j) { xs[j * 128 + r] = gk[j]; xs[(C2 + j) * 128 + r] = gv[j]; }
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (grp == 0 && ok && row_ok) {
            float4* dkp = reinterpret_cast<float4*>(dk + ipt * C2);
            float4* dvp = reinterpret_cast<float4*>(dv + ipt * C2);
#pragma unroll
            for (int c4 = 0; c4 < C2 / 4; ++c4) {
                float a[4], b[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    a[i] = (gk[4 * c4 + i] + xs[(4 * c4 + i) * 128 + r]) * scale;
                    b[i] = gv[4 * c4 + i] + xs[(C2 + 4 * c4 + i) * 128 + r];
                }
                dkp[c4] = make_float4(a[0], a[1], a[2], a[3]);
                dvp[c4] = make_float4(b[0], b[1], b[2], b[3]);
            }
        }
    } else if (warp < 12) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
        if (warp == 8 && lane == 0) {
            // -------------------------------------------------------------- TMA producer: q and dout blocks of the partner rings
            TileWalk wk(p.t_dense_lat, p.t_dense_m, e_begin, e_end, p.nlon_out, BNK, a_lo, a_hi, p.ps);
            int it = 0;
            for (; it < total && ok; ++it, wk.advance()) {
                const int s = it % NSK, u = it / NSK;
                const int h = wk.ring;
                const int w0 = wk.col();
                if (u > 0) PROF_WAIT(0, ok = mb_wait(s32(&bars[K_FREE + s]), (u - 1) & 1, ok));
                if (!ok) break;
                mb_expect(s32(&bars[K_QFULL + s]), TILE_K);
                tma_tile(sbase + s * KST, &map_q, w0, n * p.nlat_out + h, s32(&bars[K_QFULL + s]));
                mb_expect(s32(&bars[K_YFULL + s]), TILE_K);
                tma_tile(sbase + s * KST + 2 * TILE_K, &map_y, w0, n * p.nlat_out + h, s32(&bars[K_YFULL + s]));
            }
            for (int j = max(0, it - NSK); j < it; ++j) {      // the copies under way
                ok = mb_wait_polls(s32(&bars[K_QFULL + j % NSK]), (j / NSK) & 1, WAIT2) && ok;
                ok = mb_wait_polls(s32(&bars[K_YFULL + j % NSK]), (j / NSK) & 1, WAIT2) && ok;
            }
        }
        if (warp == 11) {
            // -------------------------------------------------------------- the partner points' statistics, up to NSK blocks ahead
            TileWalk wk(p.t_dense_lat, p.t_dense_m, e_begin, e_end, p.nlon_out, BNK, a_lo, a_hi, p.ps);
            static_assert(BNK == 32, "one partner point per lane");
            for (int it = 0; it < total && ok; ++it, wk.advance()) {
                const int s = it % NSK, u = it / NSK;
                if (u > 0) ok = mb_wait(s32(&bars[K_FREE + s]), (u - 1) & 1, ok);
                const size_t o = (size_t)(n * p.nlat_out + wk.ring) * p.nlon_out + min(wk.col() + lane, p.nlon_out - 1);
                float* nlc = reinterpret_cast<float*>(base + s * KST + 8 * TILE_K);
                nlc[lane] = fmaf(-__ldg(lse + o), LOG2E_2, p.log2_omega[hp]);   // log2 omega_j - lse_i in the log2 domain
                nlc[BNK + lane] = __ldg(Dws + o);
                mb_arrive(s32(&bars[K_QCONV + s]));
            }
        }
        if ((warp == 9 || warp == 10) && elect_one()) {
            // -------------------------------------------------------------- S^T = K Q^T (warp 9) and T^T = V dY^T (warp 10)
            const bool isT = warp == 10;
            ok = mb_wait(s32(&bars[K_AREADY]), 0, ok);
            const uint32_t idS = idesc_tf32(BNK), idS16 = idesc_bf16(BNK);
            const uint32_t tA = tm + (isT ? TK_AV : TK_AK), tAl = tm + (isT ? TK_AVL : TK_AKL);
            int it = 0;
            for (; it < total && ok; ++it) {
                const int s = it % NSK, us = it / NSK, b = it & 1, u = it >> 1;
                PROF_WAIT(0, ok = mb_wait(s32(&bars[(isT ? K_YFULL : K_QFULL) + s]), us & 1, ok));
                PROF_WAIT(1, ok = mb_wait(s32(&bars[(isT ? K_YCONV : K_QCONV) + s]), us & 1, ok) && ok);
                if (u > 0) {   // this (S^T, T^T, P_lo, dS_lo) buffer is free once all four second-GEMM issuers of block it-2 are done
                    PROF_WAIT(2, ok = mb_wait(s32(&bars[K_G2DONE + b]), (u - 1) & 1, ok) && ok);
                    PROF_WAIT(2, ok = mb_wait(s32(&bars[K_G2DONE + 2 + b]), (u - 1) & 1, ok) && ok);
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t tile0 = sbase + s * KST + (isT ? 2 * TILE_K : 0);
                const uint64_t db = desc_k(tile0), dbl = desc_k(tile0 + TILE_K);
                const uint32_t tD = tm + TK_BUF + 128 * b + (isT ? TK_T : TK_S);
#pragma unroll
                for (int ks = 0; ks < C2 / 8; ++ks) mma_ts16(tD, tAl + ks * 8, dbl + 2 * ks, idS16, ks > 0);     // a_lo b_hi + a_hi b_lo
#pragma unroll
                for (int ks = 0; ks < C2 / 8; ++ks) mma_ts(tD, tA + ks * 8, db + 2 * ks, idS, 1);
                mma_commit(s32(&bars[K_STFULL + b]));
                if (!isT) mb_arrive(s32(&bars[K_STFULL + b]));      // passes on what QCONV has ordered: the statistics
                mma_commit(s32(&bars[K_FREE + s]));
            }
            if (it > 0) ok = mb_wait_polls(s32(&bars[K_STFULL + ((it - 1) & 1)]), ((it - 1) >> 1) & 1, WAIT2) && ok;      // the MMAs under way
        }
    } else if (warp < 16) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
        // ------------------------------------------------------------------ second GEMMs: part = (kind, column half)
        if (elect_one()) {
            const int part = warp - 12, kind = part >> 1, grp = part & 1;      // kind 0: dV = P dY, kind 1: dK = dS Q
            const uint32_t idO = idesc_tf32(C2);
            const uint32_t tO = tm + TK_ACC + part * 32;
            int it = 0;
            for (; it < total && ok; ++it) {
                const int s = it % NSK, us = it / NSK, b = it & 1;
                const uint32_t tA = tm + TK_BUF + 128 * b + (kind ? TK_T : TK_S), tAl = tm + TK_BUF + 128 * b + (kind ? TK_DSLO : TK_PLO);
                PROF_WAIT(0, ok = mb_wait(s32(&bars[(kind ? K_QCONV : K_YCONV) + s]), us & 1, ok));
                PROF_WAIT(1, ok = mb_wait(s32(&bars[K_READY + 2 * grp + b]), (it >> 1) & 1, ok) && ok);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t bt = sbase + s * KST + (kind ? 4 : 6) * TILE_K;          // q^T (dK) or y^T (dV) tiles
#pragma unroll
                for (int k8 = 0; k8 < 2; ++k8) {
                    const int ks = grp * 2 + k8;                                    // 8-column step within the block
                    const uint32_t off = (uint32_t)ks * 32;                         // the block is one K block of 32 points
                    const uint64_t dh = desc_k(bt + off), dl = desc_k(bt + TILE_K + off);
                    mma_ts(tO, tAl + ks * 8, dh, idO, (k8 > 0) || (it % FOLDK != 0));
                    mma_ts(tO, tA + ks * 8, dl, idO, 1);
                    mma_ts(tO, tA + ks * 8, dh, idO, 1);
                }
                mma_commit(s32(&bars[K_G2DONE + 2 * grp + b]));
                mma_commit(s32(&bars[K_FREE + s]));
            }
            if (it > 0) ok = mb_wait_polls(s32(&bars[K_G2DONE + 2 * grp + ((it - 1) & 1)]), ((it - 1) >> 1) & 1, WAIT2) && ok;      // the MMAs under way
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        // ------------------------------------------------------------------ converters: warps 16-19 of the q blocks, 20-23 of the dout blocks
        const bool isY = warp >= 20;
        const int ct = tid & 127, cw = ct >> 5;
        const uint32_t full = s32(&bars[isY ? K_YFULL : K_QFULL]), conv = s32(&bars[isY ? K_YCONV : K_QCONV]);
        // lo tile (same swizzled positions) and transposed hi / lo tiles of one raw tile (one K block of 32 points: row =
        // channel, 128 bytes of points): warp cw takes the 8 columns [8 cw, 8 cw + 8), lane = channel
        for (int it = 0; it < total && ok; ++it) {
            const int s = it % NSK, u = it / NSK;
            unsigned char* raw = base + s * KST + (isY ? 2 * TILE_K : 0);
            unsigned char *lo = raw + TILE_K, *th = base + s * KST + (isY ? 6 : 4) * TILE_K;
            PROF_WAIT(0, ok = mb_wait(full + 8 * s, u & 1, ok));
#pragma unroll
            for (int j = 0; j < BNK * 4 / 128; ++j) stack_b16(raw, lo, (j * 128 + ct) >> 2, ct & 3);
#pragma unroll
            for (int c8 = 0; c8 < 2; ++c8) {
                float x[4], hi[4], lw[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const float*>(raw + sw_off(cw * 8 + c8 * 4 + i, lane >> 2) + (lane & 3) * 4);
                split4(x, hi, lw);
                const int chunk = cw * 2 + c8;
                *reinterpret_cast<float4*>(th + sw_off(lane, chunk)) = make_float4(hi[0], hi[1], hi[2], hi[3]);
                *reinterpret_cast<float4*>(th + TILE_K + sw_off(lane, chunk)) = make_float4(lw[0], lw[1], lw[2], lw[3]);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mb_arrive(conv + 8 * s);
        }
    }
    if (!ok) atomicExch(&fail_s, 1);
    PROF_DUMP(p.dev_status, warp, lane, total)
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (fail_s && tid == 0) atomicExch(p.dev_status, 1);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"(T_COLS));
}

using EncodeFn2 = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                               const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                               CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn2 encode_fn2() {
    static EncodeFn2 fn = [] {
        void* sym = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess)
            sym = nullptr;
        return reinterpret_cast<EncodeFn2>(sym);
    }();
    return fn;
}
// Tensor map over a channels-last array [slices * rings][nlon][32] with boxes of box_rows points x 32 channels.
cudaError_t make_map2(CUtensorMap* map, const float* base, int rings_total, int nlon, int box_rows = BN2) {
    EncodeFn2 fn = encode_fn2();
    if (fn == nullptr) return cudaErrorNotSupported;
    const cuuint64_t dims[3] = {(cuuint64_t)C2, (cuuint64_t)nlon, (cuuint64_t)rings_total};
    const cuuint64_t strides[2] = {(cuuint64_t)C2 * 4, (cuuint64_t)nlon * C2 * 4};
    const cuuint32_t box[3] = {(cuuint32_t)C2, (cuuint32_t)box_rows, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

cudaError_t dense2_prepare_device() {
    cudaError_t e = cudaFuncSetAttribute(forward_dense2_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DENSE2_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(forward_dense2_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DENSE2_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(backward_dq_dense2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DQ2_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(backward_dkdv_dense2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DKDV2_SMEM);
    return e;
}

// The give-up path of the bounded waits, exercised without disturbing any real kernel: the last lane of a warp waits, with the
// production wait routine but only `polls` polls, on an mbarrier that nothing ever arrives on, the other lanes on one that is
// complete.  Its first lane, whose own wait is over at once, must hear of it: it records the failure in the plan's status word as the
// dense kernels do, and the kernel returns normally.
__global__ void bounded_wait_probe_kernel(int* dev_status, int polls) {
    __shared__ __align__(8) uint64_t bars[2];
    if (threadIdx.x == 0) {
        mb_init(s32(&bars[0]), 1);
        mb_init(s32(&bars[1]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mb_arrive(s32(&bars[0]));
    }
    __syncthreads();
    const bool ok = all_lanes(mb_wait_polls(s32(&bars[threadIdx.x == 31]), 0, polls));
    if (threadIdx.x == 0 && !ok) atomicExch(dev_status, 1);
}

cudaError_t launch_bounded_wait_probe(const DevPlan& p, int polls, cudaStream_t stream) {
    bounded_wait_probe_kernel<<<1, 32, 0, stream>>>(p.dev_status, polls);
    return cudaGetLastError();
}

bool dense2_path_chosen(const DevPlan& p, int C, int N) {
    if (C != C2 || p.dense_ptr == nullptr || p.n_dense_rows == 0 || p.dense_all || !band_path_supported(p, C) || encode_fn2() == nullptr) return false;
    // One block per SM walks a tile's list, so the dense kernel takes at least the longest list's time, in which the band kernel fills
    // only the SMs that it leaves idle; with too little work per SM the band kernels alone, which share long streams between warps,
    // are faster.  Measured (fwd / dq / dkdv us, with : without the dense kernels; in brackets the work in longest lists per SM):
    // 128x256, cutoff 4 rings, N = 1 (0.1) 44/40/54 : 38/41/47, N = 2 (0.2) 85/70/71 : 59/68/78, N = 4 (0.39) 101/106/126 : 103/119/137,
    // N = 8 (0.8) 169/191/234 : 182/211/254, N = 16 316/365/454 : 344/404/492; 10 rings, N = 2 (0.47) 185/185/222 : 171/190/234;
    // 256x512 -> 128x256 N = 2 (0.22) 183/136/148 : 121/139/160, N = 4 (0.44) 204/220/286 : 226/258/307; 361x720 N = 1 (0.6)
    // 230/251/316 : 252/289/352.  (N = 4 of the first grid, on the line, would gain by 2 to 12 % now; the line was drawn at 97/113/150 :
    // 88/108/123.)  The second bound is the fixed cost of another kernel: 32x64, N = 32 (0.9 lists of 3 blocks) 48/48/54 : 43/49/47.  It lies
    // too low for lists that short: N = 128, past it, takes 140/154/177 : 108/127/150.
    const long long work = (long long)((p.nlon_out + M2 - 1) / M2) * N * p.dense_blocks;
    return work * 10 >= p.num_sms * 4LL * p.dense_longest && work >= p.num_sms * 6LL;
}

bool dense2_global_supported(const DevPlan& p, int C) {
    return C == C2 && p.dense_all && p.n_dense_rows > 0 && p.n_t_dense_rows > 0 && encode_fn2() != nullptr &&
           (long long)p.nlat_in * p.nlon_in * C < (1LL << 32) && (long long)p.nlat_out * p.nlon_out * C < (1LL << 32);
}

bool dense2_global_chosen(const DevPlan& p, int C, int N, Pass pass) {
    if (!dense2_global_supported(p, C)) return false;
    if (!band_path_supported(p, C)) return true;
    // Both sides are a number of equal units of work of known duration (us).  Dense: each block walks all rings of the other grid in
    // units of `unit` columns, one block per SM at a time; rings that are no multiple of the unit leave it partly empty, and the
    // forward kernel masks then.  Band: 256 pairs per unit over the whole GPU.  Measured dense : band, fwd / dq / dkdv:
    // 24x48 N = 4 64/39/57 : 29/29/29, 32x64 N = 16 285/170/264 : 162/176/217, 51x102 N = 4 223/223/375 : 268/299/377,
    // 64x128 N = 1 119/131/230 : 174/187/264, N = 4 234/258/455 : 559/627/797, 80x160 N = 4 1626/1210/1737 : 1323/1481/1907,
    // 90x180 N = 1 737/551/942 : 623/623/813, N = 2 1122/830/1412 : 1130/1227/1540.
    // The durations are those of slower dense kernels: a unit takes 1.85, with masks 2.0 to 2.2, in dq 1.0 to 1.1, in dk/dv 0.87 to 0.94 of
    // the present ones.  So the line is on the safe side: of the problems above the forward pass of 51x102 and of 90x180, N = 2, and dk/dv
    // of 64x128, N = 1, 80x160 and 90x180, N = 2, stay on the band kernels although the dense ones are faster.
    const bool whole = p.nlon_in % M2 == 0 && p.nlon_out % M2 == 0;
    const int unit = pass == Pass::FORWARD ? 128 : pass == Pass::DQ ? 64 : 32;
    const double dense_unit = pass == Pass::FORWARD ? (whole ? 2.0 : 2.7) : pass == Pass::DQ ? 1.05 : 1.0;
    const double band_unit = pass == Pass::FORWARD ? 0.50e-3 : pass == Pass::DQ ? 0.61e-3 : 0.745e-3;
    const bool gather = pass == Pass::DKDV;      // tiles of input points, columns of output points
    const int rows = gather ? p.nlat_in : p.nlat_out, row_len = gather ? p.nlon_in : p.nlon_out;
    const int rings = gather ? p.nlat_out : p.nlat_in, ring_len = gather ? p.nlon_out : p.nlon_in;
    const long long blocks = (long long)rows * ((row_len + M2 - 1) / M2) * N, waves = (blocks + p.num_sms - 1) / p.num_sms;
    const double dense = (double)waves * rings * ((ring_len + unit - 1) / unit) * dense_unit;
    const double band = (double)rows * row_len * rings * ring_len / 256 * N * band_unit;
    return dense <= band;
}

cudaError_t launch_backward_dq_dense2(const DevPlan& p, const float* q, const float* k, const float* v, const float* dout,
                                      const float* out, const float* lse, float* dq, float* Dws, int N, int C, cudaStream_t stream) {
    if (C != C2 || out == nullptr || lse == nullptr || out == dq) return cudaErrorInvalidValue;
    const int tiles_per_row = (p.nlon_out + M2 - 1) / M2;
    const long long blocks = (long long)tiles_per_row * p.n_dense_rows * N;
    if (blocks <= 0) return cudaSuccess;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    CUtensorMap mk, mv;
    cudaError_t e = make_map2(&mk, k, N * p.nlat_in, p.nlon_in, BNQ);
    if (e == cudaSuccess) e = make_map2(&mv, v, N * p.nlat_in, p.nlon_in, BNQ);
    if (e != cudaSuccess) return e;
    backward_dq_dense2_kernel<<<(unsigned)blocks, THREADS2, DQ2_SMEM, stream>>>(p, mk, mv, q, dout, out, lse, dq, Dws, N, 1.0f / sqrtf((float)C), tiles_per_row);
    return cudaGetLastError();
}

cudaError_t launch_backward_dkdv_dense2(const DevPlan& p, const float* q, const float* k, const float* v, const float* dout,
                                        const float* lse, const float* Dws, float* dk, float* dv, int N, int C, cudaStream_t stream) {
    if (C != C2) return cudaErrorInvalidValue;
    const int tiles_per_row = (p.nlon_in + M2 - 1) / M2;
    const long long blocks = (long long)tiles_per_row * p.n_t_dense_rows * N;
    if (blocks <= 0) return cudaSuccess;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    CUtensorMap mq, my;
    cudaError_t e = make_map2(&mq, q, N * p.nlat_out, p.nlon_out, BNK);
    if (e == cudaSuccess) e = make_map2(&my, dout, N * p.nlat_out, p.nlon_out, BNK);
    if (e != cudaSuccess) return e;
    backward_dkdv_dense2_kernel<<<(unsigned)blocks, THREADS_DKDV, DKDV2_SMEM, stream>>>(p, mq, my, k, v, lse, Dws, dk, dv, N, 1.0f / sqrtf((float)C), tiles_per_row);
    return cudaGetLastError();
}

cudaError_t launch_forward_dense2(const DevPlan& p, const float* q, const float* k, const float* v, float* out, float* lse,
                                  int N, int C, cudaStream_t stream) {
    if (C != C2) return cudaErrorInvalidValue;
    const int tiles_per_row = (p.nlon_out + M2 - 1) / M2;
    const long long blocks = (long long)tiles_per_row * p.n_dense_rows * N;
    if (blocks <= 0) return cudaSuccess;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    CUtensorMap mq, mk, mv;
    cudaError_t e = make_map2(&mq, q, N * p.nlat_out, p.nlon_out);
    if (e == cudaSuccess) e = make_map2(&mk, k, N * p.nlat_in, p.nlon_in);
    if (e == cudaSuccess) e = make_map2(&mv, v, N * p.nlat_in, p.nlon_in);
    if (e != cudaSuccess) return e;
    if (p.dense_all)   // whole rings, in all but a few blocks
        forward_dense2_kernel<true><<<(unsigned)blocks, THREADS2, DENSE2_SMEM, stream>>>(p, mq, mk, mv, out, lse, N, LOG2E_2 / sqrtf((float)C), tiles_per_row);
    else
        forward_dense2_kernel<false><<<(unsigned)blocks, THREADS2, DENSE2_SMEM, stream>>>(p, mq, mk, mv, out, lse, N, LOG2E_2 / sqrtf((float)C), tiles_per_row);
    return cudaGetLastError();
}

}  // namespace sna
