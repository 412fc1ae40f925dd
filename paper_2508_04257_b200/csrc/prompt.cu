// Prompt attention (Algorithm 1's attention statement for a chunk of queries, head size 128) on the fifth-generation tensor cores.
//
// A block takes 256 rows (query token, query head) of one KV head, token-major, as two row tiles of 128, and streams the
// cache in steps of 64 tokens.  Per step the tokens' keys and values are expanded once for all 256 rows, into shared memory
// as fp16 pairs hi + lo (x' = scale * (code - zero) to ~22 bits, in units of a power of two per step), and
//   S  = Q K_hi + Q K_lo                      Q exact in TMEM (A operand), K [token][channel] in shared memory
//   O += P_hi V_hi + P_lo V_hi + P_hi V_lo    P = hi + lo over S in TMEM (A operand), V [channel][token] in shared memory
// run as tcgen05.mma with fp32 accumulators in TMEM.  Sink tokens' rows are put into the expanded tiles exactly, keys of the
// open group come from the fp16 tail, so every token takes the same softmax.  Expanding x' (instead of multiplying bare codes
// and subtracting the zero-point terms afterwards) leaves no large terms to cancel.
//
// Warps: 0-3 / 4-7 softmax of row tile 0 / 1 (a thread owns a row), 8-11 expand keys and 12-15 values (a warp owns 32 channels),
// 16 issues the outputs' and 19 the scores' matrix instructions, 17 and 18 prepare the steps' key and value parameter tables.  While one
// tile's scores are in the softmax the tensor cores run the other tile's products.
//
// What bounds it: five matrix products of 128 x 64 x 128 per row tile and step are 2560 clocks for both tiles (2816 with tile 1's
// queries in shared memory); a step takes about 3700 to 4000.  On the SMs that have a block the tensor pipe is active for 77 to 82 % of the
// time and 73 % of the issue slots are taken.  What counts is how little code the five roles have between them: at 71 KB, with the loops
// unrolled, the warps waited for instructions (1.9 of their stalls an issue; a step with a sink token, whose code was seldom there, took
// 4500 clocks more), at 54 KB hardly (0.3).  So every role is one short loop: tiles two at a time, one pass over a row's scores, parameters
// and sink rows through shared memory.  71 KB and now, append and attention, us: 4096 queries over 4096 tokens, 8 sequences of 32
// heads, 2 bit, 2749 and 2650 (the power cap holds the clock at some 1.4 GHz); 1003 queries with four heads per KV head over 7403 tokens, 4 bit, 294
// and 278; the same at 3 bit with 128-token groups 319 and 275; 2048 queries, 2 x 32 heads, 2 bit with 64-token groups 239 and 212.  Relative
// error of the outputs against 64 bits: 2.6e-6 and 8.2e-6 for the first two.
#include "common.cuh"

namespace kvsink {

namespace {

constexpr int PR_STEP = 64;                     // tokens per step
constexpr int PR_ROWS = 256;                    // rows per block
constexpr int PR_KSTAGES = 3, PR_VSTAGES = 2;   // expanded steps in flight
constexpr int PR_SBUFS = 3;                     // score buffers, taken in turn by the two row tiles
constexpr int PR_THREADS = 20 * 32;
constexpr int PR_HALF = 16384;                  // 64 tokens x 128 channels of fp16
constexpr int PR_HDRS = 8;
// A zero point up to this size is subtracted from the code in fp16 exactly; farther ones go through an additive term.
constexpr float PR_NEAR = 1000.f;
constexpr uint32_t PR_WAIT_NS = 20000;          // a poll sleeps up to this long (without the hint it comes back after some 60 clocks)
// Between 8 ms (polls of 60 clocks) and 5.2 s (polls that all sleep as long as they may): a real wait is for work of the same block, some 10 us.
// Counted in polls and not in clocks: a look at the clock every 256 polls made the kernel 6 % slower (2661 and 2825 us), since every wait
// of every role holds a copy of the loop and code is what it has least room for.
constexpr int PR_WAIT_POLLS = 1 << 18;
constexpr int PR_ROWS_KEPT = 8;                 // sink rows of a step that the parameter warps leave in shared memory

struct StepHeader {
    float k_down, k_up, v_up;                   // 2^-kappa, 2^kappa, 2^e: the step's units of K and V
    float e;
    uint32_t dead[2];                           // sink tokens that are missing from the position list
    uint32_t k_sink[2], v_sink[2];              // sink tokens of the step (once for the keys' side, once for the values')
    int k_far, v_far;                           // some zero point is beyond PR_NEAR
    int second;                                 // first tile of the step that belongs to its second key group
    int pad[3];
};

struct PromptSmem {
    unsigned char k[PR_KSTAGES][2][PR_HALF];     // [token 64][channel 128] hi, lo: two panels of 64 channels, 128-byte swizzle
    unsigned char v[PR_VSTAGES][2][PR_HALF];    // [channel 128][token 64] hi, lo: 128-byte swizzle
    unsigned char q[2 * PR_HALF];               // queries of row tile 1: [row 128][channel 128], two panels of 64 channels
    uint4 ktab[2][2][64];                       // per key group of the step (two at most) and channel pair: scale hi, lo, zero terms
    uint4 vtab[2][4][32];                       // per value channel group and token pair
    uint2 kadd[2][2][64], vadd[2][4][32];       // additive terms hi, lo of far zero points
    StepHeader hdr[PR_HDRS];
    float k_raw[2][2][2][128], v_raw[2][2][256];   // parameters as they are in memory, by the step's buffer: keys [group][scale, zero][channel], values [scale, zero][token][group]
    int k_rank[2][64], v_rank[2][64];           // side buffer rows of the step's sink tokens, in token order
    uint4 k_kept[2][PR_ROWS_KEPT][16], v_kept[2][PR_ROWS_KEPT][16];   // the first of those rows
    uint64_t k_full[PR_KSTAGES], k_empty[PR_KSTAGES], v_full[PR_VSTAGES], v_empty[PR_VSTAGES];
    uint64_t kpar_full[2], kpar_empty[2], vpar_full[2], vpar_empty[2], hdr_full[PR_HDRS];
    uint64_t s_full[PR_SBUFS], p_full[PR_SBUFS], o_done[PR_SBUFS], o_last[2], q_full[2], drained[2];
    uint32_t tmem;
    int failed;
    int odd_values;                             // a sink token of the steps so far has a value that is infinite or NaN
};

// The block holds all 512 columns of TMEM, so its addresses start at 0.  Columns: accumulators, queries of row tile 0 (with those of
// tile 1 in shared memory there is room for a third score buffer: the scores of a tile's next step are ready when its softmax
// gets there), scores (overwritten by the weights: 16 columns of hi and 16 of lo for each half of the step).
constexpr uint32_t TM_O = 0, TM_Q = 256, TM_S = 320;

__device__ __forceinline__ void bar_init(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
// Bounded wait of a whole warp; false after the limit, or soon after another warp of the block ran into its own.  All exits are
// votes, so that the warp stays converged for the matrix instructions behind it.
__device__ __forceinline__ bool bar_wait_warp(uint64_t *bar, unsigned parity, int *failed)
{
    const uint32_t a = smem_addr(bar);
#pragma unroll 1
    for (int polls = 0; polls < PR_WAIT_POLLS; ++polls) {
        unsigned ok;
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3; selp.u32 %0, 1, 0, p; }"
                     : "=r"(ok) : "r"(a), "r"(parity), "r"(PR_WAIT_NS) : "memory");
        if (__all_sync(0xffffffffu, ok != 0)) return true;
        if (__any_sync(0xffffffffu, *(volatile int *)failed)) break;
    }
    *(volatile int *)failed = 1;
    return false;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Shared-memory operand, K-major rows of 128 bytes, 128-byte swizzle, eight-row blocks 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr)
{
    return (uint64_t)((addr >> 4) & 0x3fffu) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
// kind::f16, fp16 operands, fp32 accumulators, M = 128
__host__ __device__ constexpr uint32_t instr_desc(int n) { return (1u << 4) | ((uint32_t)(n / 8) << 17) | (8u << 24); }

// Issued by one elected lane of a converged warp: under a branch on the lane number instead of elect.sync an instruction took 53
// clocks to issue, whatever its size.
__device__ __forceinline__ bool elect_one()
{
    unsigned yes;
    asm volatile("{ .reg .pred p; elect.sync _|p, 0xffffffff; selp.u32 %0, 1, 0, p; }" : "=r"(yes));
    return yes != 0;
}
__device__ __forceinline__ void tc_mma(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, bool accumulate)         // A in TMEM
{
    asm volatile("{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p; }"
                 ::"r"(d), "r"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate) : "memory");
}
__device__ __forceinline__ void tc_mma_shared(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate)  // A in shared memory
{
    asm volatile("{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p; }"
                 ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate) : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ void tm_load32(uint32_t addr, uint32_t (&r)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                   "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
                   "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
                   "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(addr) : "memory");
}
__device__ __forceinline__ void tm_load16(uint32_t addr, uint32_t (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                   "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(addr) : "memory");
}
__device__ __forceinline__ void tm_store32(uint32_t addr, const uint32_t (&r)[32])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
                 "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
                 ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
                   "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
                   "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
                   "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]) : "memory");
}
__device__ __forceinline__ void tm_store16(uint32_t addr, const uint32_t (&r)[16])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
                   "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tm_wait_load() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_wait_store() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

template <int OFF>
__device__ __forceinline__ void st_matrix(uint32_t addr, const uint32_t (&r)[4])
{
    // no memory clobber: table loads of later matrices may move up; the proxy fence that follows a step orders the stores
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0 + %5], {%1,%2,%3,%4};" ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "n"(OFF));
}

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(*(unsigned long long *)&d) : "l"(*(unsigned long long *)&a), "l"(*(unsigned long long *)&b), "l"(*(unsigned long long *)&c));
    return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(*(unsigned long long *)&d) : "l"(*(unsigned long long *)&a), "l"(*(unsigned long long *)&b));
    return d;
}

__device__ __forceinline__ float residual(__half h, float w)      // w - h, without a conversion of its own
{
    float d;
    asm("{ .reg .b16 m; mov.b16 m, 0xbc00; fma.rn.f32.f16 %0, %1, m, %2; }" : "=f"(d) : "h"(__half_as_ushort(h)), "f"(w));
    return d;
}
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ int exponent_of(float x) { return (int)((__float_as_uint(x) >> 23) & 0xffu) - 127; }
__device__ __forceinline__ float exp2i(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }
__device__ __forceinline__ float warp_top(float v)      // largest of the lanes' non-negative values
{
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}
__device__ __forceinline__ __half2 as_half2(uint32_t x) { return *reinterpret_cast<__half2 *>(&x); }
__device__ __forceinline__ uint32_t as_u32(__half2 x) { return *reinterpret_cast<uint32_t *>(&x); }
__device__ __forceinline__ bool is_finite(float x) { return fabsf(x) <= 65504.f; }       // of an fp16 value

// Fields of one 16 x 16 matrix of a packed tile, each half ORed into 1024.0: the half is 1024 + code * 2^position.
// mm: first or second of the warp's two matrices; word(s) as load_words delivers them.
template <int BITS>
__device__ __forceinline__ void matrix_fields(const uint32_t (&w)[2], int mm, bool odd_word, uint32_t (&f)[4])
{
    constexpr uint32_t ONE = 0x64006400u;
    if constexpr (BITS == 2) {
        const uint32_t x = mm ? w[0] >> 8 : w[0];
        f[0] = (x & 0x00030003u) | ONE; f[1] = (x & 0x000c000cu) | ONE; f[2] = (x & 0x00300030u) | ONE; f[3] = (x & 0x00c000c0u) | ONE;
    } else if constexpr (BITS == 4) {
        const uint32_t x = w[mm], y = x >> 8;
        f[0] = (x & 0x000f000fu) | ONE; f[1] = (x & 0x00f000f0u) | ONE; f[2] = (y & 0x000f000fu) | ONE; f[3] = (y & 0x00f000f0u) | ONE;
    } else {
        const uint32_t hh = odd_word ? w[1] << 2 : w[1];
        uint32_t me = (w[0] & 0x33333333u) | (hh & 0xccccccccu), mo = ((w[0] >> 2) & 0x33333333u) | ((hh >> 1) & 0xccccccccu);
        if (mm) { me >>= 8; mo >>= 8; }
        f[0] = (me & 0x00070007u) | ONE; f[1] = (mo & 0x00070007u) | ONE; f[2] = (me & 0x00700070u) | ONE; f[3] = (mo & 0x00700070u) | ONE;
    }
}
// log2 of the position factor of a field, by row half and column half of its matrix
template <int BITS>
__host__ __device__ constexpr int field_shift(int row_half, int col_half)
{
    return BITS == 2 ? 2 * row_half + 4 * col_half : (BITS == 4 ? 4 * row_half : 4 * col_half);
}

// The words of tile `tile` that hold the warp's matrices 2w and 2w + 1.
template <int BITS>
__device__ __forceinline__ void load_words(const uint8_t *tile, int w, int lane, uint32_t (&out)[2])
{
    const uint32_t *p = (const uint32_t *)tile;
    if constexpr (BITS == 2) {
        out[0] = __ldg(p + 4 * lane + w);
        out[1] = 0u;
    } else if constexpr (BITS == 4) {
        const uint2 v = __ldg((const uint2 *)(p + 128 * (w >> 1) + 4 * lane + ((2 * w) & 3)));
        out[0] = v.x; out[1] = v.y;
    } else {
        out[0] = __ldg(p + 4 * lane + w);
        out[1] = __ldg(p + 128 + 2 * lane + (w >> 1));
    }
}

// hi + lo = x' of one matrix: parameters of the column pairs 2t, 2t+1 (lo) and 2t+8, 2t+9 (hi).  code - zero is an exact fp16
// integer; times the fp16 scale it rounds to `hi`, whose rounding error one more FMA gives exactly; the scale's own residual
// joins that in `lo`.  Five instructions for two elements.
template <int BITS, bool FAR>
__device__ __forceinline__ void expand_matrix(const uint32_t (&f)[4], const uint4 &pl, const uint4 &ph, const uint2 &al, const uint2 &ah,
                                              uint32_t (&hi)[4], uint32_t (&lo)[4])
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int rh = i & 1, ch = i >> 1;
        const uint4 &p = ch ? ph : pl;
        const __half2 down = __half2half2(__float2half(1.f / (float)(1 << field_shift<BITS>(rh, ch))));
        const __half2 sh = as_half2(p.x), sl = as_half2(p.y);
        const __half2 c = __hfma2(as_half2(f[i]), down, as_half2(rh ? p.w : p.z));
        if constexpr (FAR) {
            const uint2 &a = ch ? ah : al;
            const __half2 h = __hfma2(c, sh, as_half2(a.x));
            const __half2 r = __hfma2(c, sh, __hneg2(__hsub2_rn(h, as_half2(a.x))));
            hi[i] = as_u32(h);
            lo[i] = as_u32(__hadd2_rn(__hfma2(c, sl, r), as_half2(a.y)));
        } else {
            const __half2 h = __hmul2_rn(c, sh);
            hi[i] = as_u32(h);
            lo[i] = as_u32(__hfma2(c, sl, __hfma2(c, sh, __hneg2(h))));
        }
    }
}

// Table entry of a column pair: scales (hi, lo) in the step's units and the zero terms for the lower and the upper row half.
template <int BITS>
__device__ __forceinline__ void table_entry(float s0, float z0, float s1, float z1, float up, int col_half, bool general, uint4 *tab, uint2 *add)
{
    const bool far0 = fabsf(z0) > PR_NEAR, far1 = fabsf(z1) > PR_NEAR;
    const float b0 = s0 * up, b1 = s1 * up;
    const __half2 h = __floats2half2_rn(b0, b1);
    const float2 hf = __half22float2(h);
    const float n0 = far0 ? 0.f : z0, n1 = far1 ? 0.f : z1;
    const float lo = (float)(1024 >> field_shift<BITS>(0, col_half)), hi = (float)(1024 >> field_shift<BITS>(1, col_half));
    *tab = make_uint4(as_u32(h), as_u32(__floats2half2_rn(b0 - hf.x, b1 - hf.y)), as_u32(__floats2half2_rn(-(lo + n0), -(lo + n1))),
                      as_u32(__floats2half2_rn(-(hi + n0), -(hi + n1))));
    if (!general) return;
    const float a0 = far0 ? -b0 * z0 : 0.f, a1 = far1 ? -b1 * z1 : 0.f;
    const __half2 ah = __floats2half2_rn(a0, a1);
    const float2 af = __half22float2(ah);
    *add = make_uint2(as_u32(ah), as_u32(__floats2half2_rn(a0 - af.x, a1 - af.y)));
}

// Power of two that puts values up to `top` into [2^14, 2^15) of fp16.
__device__ __forceinline__ int fit_exponent(float top)
{
    const int e = 14 - exponent_of(top);
    return e > 24 ? 24 : (e < -3 ? -3 : e);
}

struct PromptArgs {
    const __half *q;
    float *out, *lse;
    int64_t q_sb, q_sh, q_st;
    int T, q_pos0, blocks;
};

template <int BITS>
__global__ void __launch_bounds__(PR_THREADS, 1) prompt_kernel(Params p, kvsink_cache c, PromptArgs a)
{
    constexpr int D = 128;
    constexpr float QMAX = (float)((1 << BITS) - 1);
    extern __shared__ unsigned char smem_raw[];
    PromptSmem &sm = *reinterpret_cast<PromptSmem *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);

    // longest row blocks first over all (sequence, KV head) units: the last wave is one of short blocks
    const int units = p.B * p.Hkv, unit = blockIdx.x % units, blk = a.blocks - 1 - blockIdx.x / units;
    const int b = unit / p.Hkv, h = unit % p.Hkv;
    const int n_rows = a.T * p.rep, row0 = blk * PR_ROWS, seq_len = c.seq_len;
    const int n_body = seq_len / p.G * p.G;
    // cached tokens that row r sees, and the steps of the two row tiles
    auto row_limit = [&](int r) { return a.q_pos0 + min(r, n_rows - 1) / p.rep + 1; };
    auto tile_steps = [&](int i) {
        return row0 + 128 * i < n_rows ? (row_limit(row0 + 128 * i + 127) + PR_STEP - 1) / PR_STEP : 0;
    };
    const int n0 = tile_steps(0), n1 = tile_steps(1), n_steps = max(n0, n1);
    // every thread alike, and before anything is set up; index checks of single accesses are at the accesses
    if (!in_bounds(b < p.B && row0 < n_rows && a.q_pos0 >= 0 && a.q_pos0 + a.T <= seq_len && seq_len <= p.max_seq && p.cap >= 0, c.status)) {
        pdl_wait();
        return;
    }

    if (warp == 16) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&sm.tmem)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        if (lane == 0) {
            for (int i = 0; i < PR_KSTAGES; ++i) { bar_init(&sm.k_full[i], 4); bar_init(&sm.k_empty[i], 1); }
            for (int i = 0; i < PR_VSTAGES; ++i) { bar_init(&sm.v_full[i], 4); bar_init(&sm.v_empty[i], 1); }
            for (int i = 0; i < PR_SBUFS; ++i) { bar_init(&sm.s_full[i], 1); bar_init(&sm.p_full[i], 4); bar_init(&sm.o_done[i], 1); }
            for (int i = 0; i < 2; ++i) {
                bar_init(&sm.kpar_full[i], 1); bar_init(&sm.kpar_empty[i], 4);
                bar_init(&sm.vpar_full[i], 1); bar_init(&sm.vpar_empty[i], 4);
                bar_init(&sm.q_full[i], 4);
                bar_init(&sm.o_last[i], 1);
                bar_init(&sm.drained[i], 1);
            }
            for (int i = 0; i < PR_HDRS; ++i) bar_init(&sm.hdr_full[i], 2);
            sm.failed = 0;
            sm.odd_values = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    pdl_wait();
    pdl_release();

    // 96 registers per thread at launch: 2 x 128 threads to 128, 2 x 128 to 80, 128 to 64 add up to the same 61440
    if (warp < 8) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 128;");
        // ---------------- softmax: thread = row ----------------
        const int i = warp >> 2, steps = i ? n1 : n0;
        const int row = row0 + 128 * i + 32 * (warp & 3) + lane;
        const bool valid = row < n_rows;
        const int lim = row_limit(row), lim_min = row_limit(row - lane);
        const int qt = min(row, n_rows - 1) / p.rep, qh = h * p.rep + min(row, n_rows - 1) % p.rep;
        const uint32_t lanes = (uint32_t)(warp & 3) << 21;                   // this warp's 32 lanes of TMEM
        const uint32_t t_o = lanes + TM_O + 128 * i;
        const float qscale = 1.4426950408889634f * rsqrtf((float)D);
        bool ok = true;
        if (steps > 0) {
            const uint4 *src = (const uint4 *)(a.q + b * a.q_sb + qh * a.q_sh + qt * a.q_st);
            const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
            if (i == 0) {
#pragma unroll 1
                for (int half = 0; half < 2; ++half) {
                    uint32_t r[32];
#pragma unroll
                    for (int x = 0; x < 8; ++x) {
                        const uint4 v = valid ? __ldg(src + 8 * half + x) : zero;
                        r[4 * x] = v.x; r[4 * x + 1] = v.y; r[4 * x + 2] = v.z; r[4 * x + 3] = v.w;
                    }
                    tm_store32(lanes + TM_Q + 32 * half, r);
                }
                tm_wait_store();
                tc_fence_before();
            } else {
                const int r = tid - 128;
#pragma unroll
                for (int x = 0; x < 16; ++x)
                    *reinterpret_cast<uint4 *>(sm.q + (x >> 3) * PR_HALF + r * 128 + (((x & 7) ^ (r & 7)) << 4)) = valid ? __ldg(src + x) : zero;
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            __syncwarp();
            if (lane == 0) bar_arrive(&sm.q_full[i]);
        }
        // weights are 2^(score - M - e) with M the row's reference, moved only when a weight would leave fp16: the weights of a
        // step stay below 2^15 and the values below 2^15 in the step's units 2^-e, so that P V is in the units of 2^-M throughout
        float M = M_INIT, l = 0.f;
        // items: steps of the tiles, in turn.  Barriers are per score buffer.  Inside the loop none can run two phases ahead of a waiter:
        // the buffer's next user comes three items on, behind the same tile's next item, whose outputs need this warp's weights.
        // Behind a tile's last item the other tile may have three more, which pass through the same buffers without it, so the
        // end of a tile has a barrier of its own, completed once
        int item = i, before = 0;
#pragma unroll 1
        for (int j = 0; j < steps; before = item, item += 1 + (j + i < (i ? n0 : n1)), ++j) {
            const int sb = item % PR_SBUFS;
            const uint32_t t_s = lanes + TM_S + 64 * sb;
            if (!(ok = bar_wait_warp(&sm.s_full[sb], (item / PR_SBUFS) & 1, &sm.failed))) break;
            if (!(ok = bar_wait_warp(&sm.hdr_full[j & (PR_HDRS - 1)], (j / PR_HDRS) & 1, &sm.failed))) break;
            tc_fence_after();
            const StepHeader &hd = sm.hdr[j & (PR_HDRS - 1)];
            const float c1 = qscale * hd.k_down, ef = hd.e, vup = hd.v_up;
            const uint32_t dead0 = hd.dead[0], dead1 = hd.dead[1];
            // tokens that the row does not see: -inf over their scores, in the steps that have any
            const int left = lim - j * PR_STEP;
            if ((j + 1) * PR_STEP > lim_min || (dead0 | dead1)) {
#pragma unroll 1
                for (int x = 0; x < 64; x += 16) {
                    uint32_t v[16];
                    tm_load16(t_s + x, v);
                    tm_wait_load();
                    const int n = left - x;
                    const uint32_t gone = (x < 32 ? dead0 : dead1) >> (x & 16) | (n <= 0 ? 0xffffu : (n >= 16 ? 0u : 0xffffu << n));
#pragma unroll
                    for (int y = 0; y < 16; ++y)
                        if (gone >> y & 1u) v[y] = 0xff800000u;
                    tm_store16(t_s + x, v);
                }
                tm_wait_store();
            }
            uint32_t v0[32], v1[32];
            tm_load32(t_s, v0);
            tm_load32(t_s + 32, v1);
            tm_wait_load();
            float top = max3(__uint_as_float(v0[0]), __uint_as_float(v1[0]), -INFINITY), top2 = -INFINITY;
#pragma unroll
            for (int x = 1; x < 31; x += 2) {
                top = max3(top, __uint_as_float(v0[x]), __uint_as_float(v0[x + 1]));
                top2 = max3(top2, __uint_as_float(v1[x]), __uint_as_float(v1[x + 1]));
            }
            top = max3(max3(top, top2, __uint_as_float(v0[31])), __uint_as_float(v1[31]), -INFINITY);
            top = fmaf(top, c1, -ef);
            if (__any_sync(0xffffffffu, top > M + 15.f)) {
                const float Mn = top > M + 15.f ? top - 8.f : M, f = ex2(M - Mn);
                M = Mn;
                l *= f;
                if (j > 0) {       // not while the products of the step before are under way
                    if (!(ok = bar_wait_warp(&sm.o_done[before % PR_SBUFS], (before / PR_SBUFS) & 1, &sm.failed))) break;
                    tc_fence_after();
#pragma unroll 1
                    for (int x = 0; x < 8; ++x) {
                        uint32_t o[16];
                        tm_load16(t_o + 16 * x, o);
                        tm_wait_load();
#pragma unroll
                        for (int y = 0; y < 16; ++y) o[y] = __float_as_uint(__uint_as_float(o[y]) * f);
                        tm_store16(t_o + 16 * x, o);
                    }
                }
            }
            const float2 c2 = make_float2(c1, c1), sub2 = make_float2(-(M + ef), -(M + ef));
            float2 sum = make_float2(0.f, 0.f);
            auto weights = [&](uint32_t (&v)[32], uint32_t to) {       // the half's weights take its scores' place: hi, then lo
                uint32_t r[32];
#pragma unroll
                for (int x = 0; x < 16; ++x) {
                    float2 w = fma2(make_float2(__uint_as_float(v[2 * x]), __uint_as_float(v[2 * x + 1])), c2, sub2);
                    w.x = ex2(w.x); w.y = ex2(w.y);
                    sum = add2(sum, w);
                    const __half2 wh = __floats2half2_rn(w.x, w.y);
                    r[x] = as_u32(wh);
                    r[16 + x] = as_u32(__floats2half2_rn(residual(__low2half(wh), w.x), residual(__high2half(wh), w.y)));
                }
                tm_store32(to, r);
            };
            weights(v0, t_s);
            weights(v1, t_s + 32);
            l = fmaf(sum.x + sum.y, vup, l);
            tm_wait_store();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) bar_arrive(&sm.p_full[sb]);
        }
        if (ok && steps > 0 && bar_wait_warp(&sm.o_last[i], 0, &sm.failed)) {
            tc_fence_after();
            const float inv = l > 0.f ? 1.f / l : 0.f;
            const size_t oq = ((size_t)b * p.Hq + qh) * a.T + qt;
#pragma unroll 1
            for (int x = 0; x < 4; ++x) {
                uint32_t o[32];
                tm_load32(t_o + 32 * x, o);
                tm_wait_load();
                if (valid) {
                    float4 *dst = (float4 *)(a.out + oq * D + 32 * x);
#pragma unroll
                    for (int y = 0; y < 8; ++y)
                        dst[y] = make_float4(__uint_as_float(o[4 * y]) * inv, __uint_as_float(o[4 * y + 1]) * inv,
                                             __uint_as_float(o[4 * y + 2]) * inv, __uint_as_float(o[4 * y + 3]) * inv);
                }
            }
            if (a.lse && valid) a.lse[oq] = l > 0.f ? (M + log2f(l)) * 0.6931471805599453f : -INFINITY;
            // values of sink tokens that are infinite or NaN were left out of the products, where they would reach every row of the
            // tile; only rows that see the token get them
            if (valid && *(volatile int *)&sm.odd_values) {
#pragma unroll 1
                for (int y = 0; y < min(c.sink_count[b], p.cap); ++y) {
                    const int tok = c.sink_pos[(size_t)b * p.cap + y];
                    if (tok < 0 || tok >= lim || !mask_bit(c.sink_bitmask + (size_t)b * p.mask_words, tok)) continue;
                    const __half *v = (const __half *)c.sink_v + ((size_t)unit * p.cap + y) * D;
#pragma unroll 1
                    for (int ch = 0; ch < D; ++ch)
                        if (!is_finite(__half2float(v[ch]))) a.out[oq * D + ch] += __half2float(v[ch]);
                }
            }
        }
    } else if (warp < 16) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        // ---------------- expansion of keys (warps 8-11) and values (12-15); warp w owns channels 32 w ... 32 w + 31 ----------------
        const bool keys = warp < 12;
        const int w = warp & 3, t = lane & 3;
        const uint8_t *codes = (keys ? c.k_codes : c.v_codes) + (size_t)unit * p.max_seq * p.row_bytes;
        const int coded = keys ? n_body : seq_len;                       // tokens below it have codes
        // stmatrix: lane l gives the address of row l % 8 of the 8 x 8 matrix l / 8 (row half l/8 % 2, column half l / 16)
        const int sr = (lane & 7) + 8 * ((lane >> 3) & 1), sc = lane >> 4;
        constexpr int TILE = 16 * D * BITS / 8;
        // words of the next four tiles, each loaded when the one four before it is taken
        uint32_t words[4][2];
        auto fetch = [&](int tile, uint32_t (&to)[2]) {
            to[0] = to[1] = 0u;
            if (tile < 4 * n_steps && 16 * tile < coded && in_bounds(16 * (tile + 1) <= p.max_seq, c.status)) load_words<BITS>(codes + (size_t)tile * TILE, w, lane, to);
        };
        // keys: row = token, 16-byte chunk = eight channels, two panels of 64; values: row = channel, chunk = eight tokens
        auto place = [](int r, int ck) { return (uint32_t)((ck >> 3) * 8192 + r * 128 + (((ck & 7) ^ (r & 7)) << 4)); };
        // sink tokens: their exact rows over the expanded ones
        auto put_sinks = [&](const uint32_t (&sink)[2], const int *ranks, const uint4 (*kept)[16], uint32_t base, float up) {
            __syncwarp();
            const int ch = 32 * w + lane;
            const __half *rows = (const __half *)(keys ? c.sink_k : c.sink_v) + (size_t)unit * p.cap * D + ch, *near = (const __half *)kept + ch;
            uint64_t left = (uint64_t)sink[1] << 32 | sink[0];
#pragma unroll 1
            for (int idx = 0; left; ++idx) {
                const int tk = __ffsll((long long)left) - 1;
                left &= left - 1;
                float x = 0.f;
                if (idx < PR_ROWS_KEPT) {
                    x = __half2float(near[idx * D]);
                } else {
                    const int r = ranks[idx];
                    if (r >= 0 && in_bounds(r < p.cap, c.status)) x = __half2float(rows[(size_t)r * D]);
                }
                if (!keys && !is_finite(x)) x = 0.f;     // a weight of 0 does not hide it: added at the end
                const int r = keys ? tk : ch, col = keys ? ch : tk;
                const uint32_t at = base + place(r, col >> 3) + 2 * (col & 7);
                const unsigned short v = __half_as_ushort(__float2half_rn(x * up));
                asm volatile("st.shared.u16 [%0], %1;" ::"r"(at), "h"(v) : "memory");
                asm volatile("st.shared.u16 [%0], %1;" ::"r"(at + PR_HALF), "h"((unsigned short)0) : "memory");
            }
        };
        const __half *tail = (const __half *)c.k_tail + (size_t)unit * p.G * D;
        uint64_t *par_full = keys ? sm.kpar_full : sm.vpar_full, *par_empty = keys ? sm.kpar_empty : sm.vpar_empty;
        uint64_t *full = keys ? sm.k_full : sm.v_full, *empty = keys ? sm.k_empty : sm.v_empty;
        // byte offsets of the lane's stmatrix rows for tile tt, matrix mm, and table entries of its columns: by channel pair (keys,
        // the step's second group 64 entries on) or by token pair (values)
        const int jg = 32 * w / p.Gv;                                    // value channel group of the warp's channels
        const uint32_t at0 = keys ? place(sr, 4 * w + sc) : place(32 * w + sr, sc), at1 = keys ? place(sr, 4 * w + 2 + sc) : place(32 * w + 16 + sr, sc);
        const uint32_t add_tile = keys ? 2048 : 0, xor_tile = keys ? 0 : 32;
        const int entry0 = keys ? 16 * w + t : 32 * jg + t, entry_mm = keys ? 8 : 0;
#pragma unroll
        for (int tt = 0; tt < 4; ++tt) fetch(tt, words[tt]);
        const int stages = keys ? PR_KSTAGES : PR_VSTAGES;
        int stage = 0, phase = 0;
#pragma unroll 1
        for (int j = 0; j < n_steps; ++j) {
            const int buf = j & 1;
            if (!bar_wait_warp(&par_full[buf], (j >> 1) & 1, &sm.failed)) break;
            if (j >= stages && !bar_wait_warp(&empty[stage], phase ^ 1, &sm.failed)) break;
            const StepHeader &hd = sm.hdr[j & (PR_HDRS - 1)];
            const int second = hd.second;
            const uint32_t *sinks = keys ? hd.k_sink : hd.v_sink;
            const uint32_t sink[2] = {sinks[0], sinks[1]};
            const float up = keys ? hd.k_up : hd.v_up;
            const bool far = keys ? hd.k_far : hd.v_far;
            const uint4 *tab = keys ? &sm.ktab[buf][0][0] : &sm.vtab[buf][0][0];
            const uint32_t base = smem_addr(keys ? &sm.k[stage][0][0] : &sm.v[stage][0][0]);
#pragma unroll 2      // two tiles' chains at a time; all four are slower by a tenth, one by a twentieth
            for (int tt = 0; tt < 4; ++tt) {
                const uint32_t cur[2] = {words[0][0], words[0][1]};
#pragma unroll
                for (int x = 0; x < 3; ++x) { words[x][0] = words[x + 1][0]; words[x][1] = words[x + 1][1]; }
                fetch(4 * j + tt + 4, words[3]);
                const int entry = entry0 + (keys ? (tt >= second ? 64 : 0) : 8 * tt), tok = j * PR_STEP + 16 * tt;
                const uint32_t to0 = base + ((at0 + tt * add_tile) ^ (tt * xor_tile)), to1 = base + ((at1 + tt * add_tile) ^ (tt * xor_tile));
                if (!far && (!keys || tok < n_body)) {
#pragma unroll
                    for (int mm = 0; mm < 2; ++mm) {
                        uint32_t f[4], hi[4], lo[4];
                        matrix_fields<BITS>(cur, mm, w & 1, f);
                        const uint4 *e = tab + entry + mm * entry_mm;
                        expand_matrix<BITS, false>(f, e[0], e[4], make_uint2(0u, 0u), make_uint2(0u, 0u), hi, lo);
                        st_matrix<0>(mm ? to1 : to0, hi);
                        st_matrix<PR_HALF>(mm ? to1 : to0, lo);
                    }
                } else {                                  // far zero points, or a key tile of the open group
                    const uint2 *add = keys ? &sm.kadd[buf][0][0] : &sm.vadd[buf][0][0];
#pragma unroll 1
                    for (int mm = 0; mm < 2; ++mm) {
                        uint32_t hi[4], lo[4];
                        if (keys && tok >= n_body) {      // exact fp16 rows from the tail
                            const __half2 up2 = __half2half2(__float2half(up));
#pragma unroll
                            for (int y = 0; y < 4; ++y) {
                                const int tk = tok + (lane >> 2) + 8 * (y & 1);
                                const uint32_t v = tk < seq_len && in_bounds(tk - n_body < p.G, c.status) ? *(const uint32_t *)(tail + (size_t)(tk - n_body) * D + 16 * (2 * w + mm) + 8 * (y >> 1) + 2 * t) : 0u;
                                hi[y] = as_u32(__hmul2_rn(as_half2(v), up2));
                                lo[y] = 0u;
                            }
                        } else {
                            uint32_t f[4];
                            matrix_fields<BITS>(cur, mm, w & 1, f);
                            const int e = entry + mm * entry_mm;
                            expand_matrix<BITS, true>(f, tab[e], tab[e + 4], add[e], add[e + 4], hi, lo);
                        }
                        st_matrix<0>(mm ? to1 : to0, hi);
                        st_matrix<PR_HALF>(mm ? to1 : to0, lo);
                    }
                }
            }
            if (sink[0] | sink[1]) put_sinks(sink, keys ? sm.k_rank[buf] : sm.v_rank[buf], keys ? sm.k_kept[buf] : sm.v_kept[buf], base, up);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) { bar_arrive(&full[stage]); bar_arrive(&par_empty[buf]); }
            if (++stage == stages) { stage = 0; phase ^= 1; }
        }
    } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    if (warp == 16 || warp == 19) {
        // ---------------- matrix instructions: warp 16 the outputs', warp 19 the scores' ----------------
        // Items are the steps of the tiles, in turn: tile 0 of a step, tile 1 of it.  An item's scores go where the weights of the item
        // three before were, so they wait for its outputs: only products on one accumulator are sure to run in the order they were
        // issued.  With one warp for both kinds that wait also held up the next outputs (the two shapes above, with the append: 2887
        // and 308 us; two warps: 2707 and 287).
        // After a wait that ran out the loops go on (their waits return at once, nothing leaves the block's memory): their control
        // does not depend on the waits.
        const bool scores = warp == 19;
        const uint32_t kb = smem_addr(&sm.k[0][0][0]), vb = smem_addr(&sm.v[0][0][0]);
        const uint64_t qd = smem_desc(smem_addr(sm.q));
        const int m0 = __reduce_max_sync(0xffffffffu, n0), m1 = __reduce_max_sync(0xffffffffu, n1), items = m0 + m1;
        int i = 0, j = 0, stage = 0, phase = 0, buf = 0, bphase = 0;       // the item: tile, step; its step's stage, its score buffer
        auto next = [&](bool last, int stages) {
            if (last) {
                ++j;
                i = j < m0 ? 0 : 1;
                if (++stage == stages) { stage = 0; phase ^= 1; }
            } else {
                i = 1;
            }
            if (++buf == PR_SBUFS) { buf = 0; bphase ^= 1; }
        };
        if (!scores) {
#pragma unroll 1
            for (int it = 0; it < items; ++it) {               // O += P_hi V_lo + P_lo V_hi + P_hi V_hi
                if (i == 0 || j >= m0) bar_wait_warp(&sm.v_full[stage], phase, &sm.failed);
                bar_wait_warp(&sm.p_full[buf], bphase, &sm.failed);
                tc_fence_after();
                const uint64_t vd = smem_desc(vb + stage * 2 * PR_HALF);
                const uint32_t d = TM_O + 128 * i, w = TM_S + 64 * buf;
                const bool last = i == 1 || j >= m1;
                if (elect_one()) {
#pragma unroll 1
                    for (int part = 0; part < 3; ++part)
#pragma unroll
                        for (int x = 0; x < 4; ++x)
                            tc_mma(d, w + (part == 1 ? 16 : 0) + 32 * (x >> 1) + 8 * (x & 1), vd + (((part == 0 ? PR_HALF : 0) + x * 32) >> 4), instr_desc(128),
                                   j > 0 || part + x > 0);
                    tc_commit(&sm.o_done[buf]);
                    if (last) tc_commit(&sm.v_empty[stage]);
                    if (j == (i ? m1 : m0) - 1) tc_commit(&sm.o_last[i]);
                }
                __syncwarp();
                next(last, PR_VSTAGES);
            }
        } else {
            bar_wait_warp(&sm.q_full[0], 0, &sm.failed);
            if (m1 > 0) bar_wait_warp(&sm.q_full[1], 0, &sm.failed);
#pragma unroll 1
            for (int it = 0; it < items; ++it) {               // S = Q K_lo + Q K_hi
                if (i == 0 || j >= m0) bar_wait_warp(&sm.k_full[stage], phase, &sm.failed);
                if (it >= PR_SBUFS) bar_wait_warp(&sm.o_done[buf], bphase ^ 1, &sm.failed);
                tc_fence_after();
                const uint64_t kd = smem_desc(kb + stage * 2 * PR_HALF);
                const uint32_t d = TM_S + 64 * buf;
                const bool last = i == 1 || j >= m1;
                if (elect_one()) {
#pragma unroll 1
                    for (int part = 0; part < 4; ++part) {     // K_lo, K_hi, each by its two panels of 64 channels
                        const uint64_t kp = kd + (((part < 2 ? PR_HALF : 0) + (part & 1) * 8192) >> 4);
                        if (i == 0) {
#pragma unroll
                            for (int x = 0; x < 4; ++x) tc_mma(d, TM_Q + 32 * (part & 1) + 8 * x, kp + 2 * x, instr_desc(64), part + x > 0);
                        } else {
                            const uint64_t qp = qd + ((part & 1) * PR_HALF >> 4);
#pragma unroll
                            for (int x = 0; x < 4; ++x) tc_mma_shared(d, qp + 2 * x, kp + 2 * x, instr_desc(64), part + x > 0);
                        }
                    }
                    tc_commit(&sm.s_full[buf]);
                    if (last) tc_commit(&sm.k_empty[stage]);
                }
                __syncwarp();
                next(last, PR_KSTAGES);
            }
        }
        if (sm.failed) {       // gave up: let what was issued finish before the block goes
            int go = 0;
            if (elect_one()) tc_commit(&sm.drained[scores]);
            __syncwarp();
            bar_wait_warp(&sm.drained[scores], 0, &go);
        }
    } else {
        // ---------------- parameter tables: warp 17 of the keys, warp 18 of the values ----------------
        const bool keys = warp == 17;
        uint64_t *full = keys ? sm.kpar_full : sm.vpar_full, *empty = keys ? sm.kpar_empty : sm.vpar_empty;
        int (*rank)[64] = keys ? sm.k_rank : sm.v_rank;
        const float *ks = c.k_scale + (size_t)unit * (p.max_seq / p.G) * D, *kz = c.k_zero + (size_t)unit * (p.max_seq / p.G) * D;
        const float *vs = c.v_scale + (size_t)unit * p.max_seq * p.NGv, *vz = c.v_zero + (size_t)unit * p.max_seq * p.NGv;
        const uint32_t *bm = c.sink_bitmask + (size_t)b * p.mask_words;
        const int32_t *pos = c.sink_pos + (size_t)b * p.cap;
        const int n_pos = min(c.sink_count[b], p.cap);
        const __half *rows = (const __half *)(keys ? c.sink_k : c.sink_v) + (size_t)unit * p.cap * D + 8 * (lane & 15);
        uint4 (*kept)[PR_ROWS_KEPT][16] = keys ? sm.k_kept : sm.v_kept;
        int rank0 = 0;                                                   // sink tokens before the step
        // A step's parameters come into shared memory a step ahead, as they are: of the (at most two) key groups that meet the step (G
        // is 32, 64 or at least 128), of its tokens' values.  Entries: keys, two channel pairs a lane for each group; values, one
        // token pair a lane for each channel group.
        const float *ps = keys ? ks : vs, *pz = keys ? kz : vz;
        // group of the step's first token, tokens of the step before the next group, and the step's entries
        int g0 = 0, second = p.G;
        auto count = [&](int j, int second) {
            const int body = n_body - j * PR_STEP;
            return keys ? (body > 0 ? (min(body, PR_STEP) > second ? 4 : 2) : 0) : p.NGv;
        };
        auto fetch = [&](int j, int g) {
            const int n = keys ? (count(j, second) >> 1) : 1, chunks = keys ? 32 : 16 * p.NGv;     // 16 bytes each
            float *to = keys ? &sm.k_raw[j & 1][0][0][0] : &sm.v_raw[j & 1][0][0];
            const int half = keys ? 128 : 256;
#pragma unroll 1
            for (int y = 0; y < n; ++y, to += 256)
#pragma unroll 1
                for (int x = lane; x < chunks; x += 32) {
                    const int64_t at = keys ? (int64_t)(g + y) * D + 4 * x : (int64_t)j * PR_STEP * p.NGv + 4 * x;
                    if (keys ? !in_bounds((g + y + 1) * p.G <= n_body, c.status) : at >= (int64_t)seq_len * p.NGv) continue;
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_addr(to + 4 * x)), "l"(ps + at) : "memory");
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_addr(to + half + 4 * x)), "l"(pz + at) : "memory");
                }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        struct Pair { float s0, z0, s1, z1; };
        auto pair = [&](int j, int n) {
            Pair r = {0.f, 0.f, 0.f, 0.f};
            if (keys) {
                const float *at = &sm.k_raw[j & 1][n >> 1][0][2 * lane + 64 * (n & 1)];
                const float2 s = *(const float2 *)at, z = *(const float2 *)(at + 128);
                r.s0 = s.x; r.s1 = s.y; r.z0 = z.x; r.z1 = z.y;
            } else {
                const float *at = &sm.v_raw[j & 1][0][2 * lane * p.NGv + n];
                const int left = seq_len - (j * PR_STEP + 2 * lane);
                if (left > 0) { r.s0 = at[0]; r.z0 = at[256]; }
                if (left > 1) { r.s1 = at[p.NGv]; r.z1 = at[256 + p.NGv]; }
            }
            return r;
        };
        auto mask_word = [&](int j, int x) {
            const int left = seq_len - (j * PR_STEP + 32 * x);
            uint32_t w = left > 0 && in_bounds(2 * j + x < p.mask_words, c.status) ? __ldg(bm + 2 * j + x) : 0u;
            return left > 0 && left < 32 ? w & ((1u << left) - 1u) : w;
        };
        fetch(0, 0);
        uint32_t bits[2] = {mask_word(0, 0), mask_word(0, 1)};
#pragma unroll 1
        for (int j = 0; j < n_steps; ++j) {
            const int buf = j & 1, tok0 = j * PR_STEP;
            const uint32_t sink[2] = {bits[0], bits[1]};
            const int split = second, n_entries = count(j, second);
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();
            if (j + 1 < n_steps) {
                second -= PR_STEP;
                while (second <= 0) { second += p.G; ++g0; }
                fetch(j + 1, g0);
                bits[0] = mask_word(j + 1, 0);
                bits[1] = mask_word(j + 1, 1);
            }
            float top = 0.f;
            bool far = false, odd = false;
#pragma unroll 1
            for (int n = 0; n < n_entries; ++n) {                        // largest |scale * (code - zero)|
                const Pair r = pair(j, n);
                top = max3(top, r.s0 * fmaxf(fabsf(r.z0), fabsf(QMAX - r.z0)), r.s1 * fmaxf(fabsf(r.z1), fabsf(QMAX - r.z1)));
                far |= fabsf(r.z0) > PR_NEAR || fabsf(r.z1) > PR_NEAR;
            }
            if (j >= 2 && !bar_wait_warp(&empty[buf], ((j >> 1) - 1) & 1, &sm.failed)) break;
            // sink tokens of the step and their side buffer rows
            uint32_t dead0 = 0u, dead1 = 0u;
            const int ns0 = __popc(sink[0]), ns = ns0 + __popc(sink[1]);
            if (ns) {
#pragma unroll 1
                for (int x = 0; x < 2; ++x) {                            // a lane looks after one token of each word
                    const uint32_t word = x ? sink[1] : sink[0];
                    bool miss = false;
                    if (word >> lane & 1u) {
                        const int idx = __popc(word & ((1u << lane) - 1u)) + (x ? ns0 : 0), tok = tok0 + 32 * x + lane;
                        int r = rank0 + idx;
                        if (r >= n_pos || pos[r] != tok) {               // mask and list disagree: look for it
                            r = -1;
                            for (int y = 0; y < n_pos; ++y)
                                if (pos[y] == tok) { r = y; break; }
                            miss = r < 0;
                        }
                        rank[buf][idx] = r;
                    }
                    const uint32_t m = __ballot_sync(0xffffffffu, miss);
                    if (x) dead1 = m;
                    else dead0 = m;
                }
                __syncwarp();
                __half2 large = __float2half2_rn(0.f);
#pragma unroll 2
                for (int y = lane >> 4; y < ns; y += 2) {                // half a warp a row
                    const int r = rank[buf][y];
                    uint4 v = make_uint4(0u, 0u, 0u, 0u);
                    if (r >= 0 && in_bounds(r < p.cap, c.status)) v = *(const uint4 *)(rows + (size_t)r * D);
                    if (y < PR_ROWS_KEPT) kept[buf][y][lane & 15] = v;
                    auto look = [&](uint32_t x) {
                        const __half2 mag = __habs2(as_half2(x));
                        const uint32_t finite = __hle2_mask(mag, __float2half2_rn(65504.f));
                        odd |= finite != 0xffffffffu;
                        large = __hmax2(large, as_half2(as_u32(mag) & finite));
                    };
                    look(v.x); look(v.y); look(v.z); look(v.w);
                }
                top = max3(top, __low2float(large), __high2float(large));
                rank0 += ns;
                if (!keys && __any_sync(0xffffffffu, odd) && lane == 0) *(volatile int *)&sm.odd_values = 1;
            }
            int e = fit_exponent(warp_top(top));
            if (keys && tok0 + PR_STEP > n_body && seq_len > n_body) e = min(e, 0);    // fp16 rows of the open group, as they are
            const float up = exp2i(e);
            StepHeader &hd = sm.hdr[j & (PR_HDRS - 1)];
            far = __any_sync(0xffffffffu, far);
            uint4 *tab = keys ? &sm.ktab[buf][0][0] : &sm.vtab[buf][0][0];
            uint2 *add = keys ? &sm.kadd[buf][0][0] : &sm.vadd[buf][0][0];
#pragma unroll 1
            for (int n = 0; n < n_entries; ++n) {
                const Pair r = pair(j, n);
                table_entry<BITS>(r.s0, r.z0, r.s1, r.z1, up, (lane >> 2) & 1, far, tab + 32 * n + lane, add + 32 * n + lane);
            }
            if (lane == 0) {
                if (keys) {
                    hd.k_down = exp2i(-e); hd.k_up = up;
                    hd.k_sink[0] = sink[0]; hd.k_sink[1] = sink[1];
                    hd.dead[0] = dead0; hd.dead[1] = dead1;
                    hd.k_far = far;
                    hd.second = split / KVSINK_TILE;
                } else {
                    hd.v_up = up; hd.e = (float)e;
                    hd.v_sink[0] = sink[0]; hd.v_sink[1] = sink[1];
                    hd.v_far = far;
                }
            }
            __syncwarp();
            if (lane == 0) {
                bar_arrive(&full[buf]);
                bar_arrive(&sm.hdr_full[j & (PR_HDRS - 1)]);        // for the softmax: both warps' halves of the header
            }
        }
    }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 16) {
        tc_fence_after();
        if (lane == 0 && sm.failed) atomicOr(c.status, KVSINK_STATUS_TIMEOUT);
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sm.tmem), "r"(512) : "memory");
    }
}

template <int BITS>
int launch(const Params &p, const kvsink_cache &c, const PromptArgs &a, cudaStream_t st)
{
    auto kern = prompt_kernel<BITS>;
    constexpr int smem = sizeof(PromptSmem) + 1024;
    static_assert(smem <= 227 * 1024, "shared memory of a block");
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return KVSINK_ERR_CUDA;
    if (launch_pdl(kern, dim3((unsigned)((int64_t)a.blocks * p.B * p.Hkv)), dim3(PR_THREADS), smem, st, p, c, a) != cudaSuccess) return KVSINK_ERR_CUDA;
    return KVSINK_OK;
}

}  // namespace

// The kernel for many rows: below the line the eight-row blocks of the decode kernel (four on an SM, four warps each on a share of
// the cache) are faster.  A block here takes about 2.1 us for 64 tokens however few rows it has, one block to an SM; those blocks
// 0.6 us (2 bit) to 1 us (3, 4 bit) until some 256 of them fill the chip.  Measured at 16384 tokens, 2 bit, 32 units: 256 queries
// (1024 such blocks) 621 -> 559 us, 128 queries 387 -> 537 us; 4 bit, eight units with four rows a query: 128 queries (512
// blocks) 599 -> 556 us, 64 queries 366 -> 552 us; eight times the blocks, 13495 -> 2392 us.
bool prompt_takes(const Params &p, int T)
{
    if (p.D != 128) return false;
    const int64_t rows = (int64_t)T * p.rep, units = (int64_t)p.B * p.Hkv;
    const int64_t blocks = (rows + PR_ROWS - 1) / PR_ROWS * units, waves = (blocks + 147) / 148;
    return rows < (1 << 30) && blocks < (1 << 30) && (rows + 7) / 8 * units >= waves * (p.bits == 2 ? 1024 : 512);
}

int launch_prompt(const Params &p, const kvsink_cache &c, const __half *q, int T, int q_pos0, int64_t sb, int64_t sh, int64_t stt, float *out,
                  float *lse, cudaStream_t st)
{
    const PromptArgs a = {q, out, lse, sb, sh, stt, T, q_pos0, (int)(((int64_t)T * p.rep + PR_ROWS - 1) / PR_ROWS)};
    if (p.bits == 2) return launch<2>(p, c, a, st);
    if (p.bits == 3) return launch<3>(p, c, a, st);
    return launch<4>(p, c, a, st);
}

}  // namespace kvsink
