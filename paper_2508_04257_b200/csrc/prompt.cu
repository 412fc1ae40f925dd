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
// One block to an SM, which goes through several such work items: the roles below hand steps over through barriers that go on counting from
// one item to the next, so the expansion of the next item's first steps and its first products run beside the last ones' and the outputs'
// way to memory.  With a block for each item its set-up, first loads and outputs took 35000 of the 149000 clocks of an item of 4096 tokens in
// the mean, 16 us of the 22 us of one with 165.
//
// Warps: 0-3 / 4-7 softmax of row tile 0 / 1 (a thread owns a row), 8-11 expand keys and 12-15 values (a warp owns 32 channels),
// 16 issues the outputs' and 19 the scores' matrix instructions, 17 and 18 fetch the steps' packed tiles and parameters (bulk copies) and
// prepare the parameter tables of keys and values.  While one tile's scores are in the softmax the tensor cores run the other tile's products.
//
// What bounds it: energy where all SMs are busy for long (the power cap holds the clock at 1.4 to 1.7 GHz; the five products alone, with nothing
// else on the chip, would take 1.73 us a step there), and else the five roles' instructions, which share the issue slots: with any one role's
// work left out a step of some 3500 clocks becomes 3 to 10 % shorter, alone the products take 2800 (five of 128 x 64 x 128 for
// two row tiles), the expansion had 3000, the tables 2500, the softmax 2160.  So what counts is how little code and how few instructions the
// roles have between them: at 71 KB, with the loops unrolled, the warps waited for instructions (1.9 of their stalls an issue), at 55 KB hardly
// (0.3); matrix instructions unrolled further (2 KB more): 5 % slower; expansion of four tiles at a time 3 % slower; shared memory through
// generic addresses 6 to 9 % slower.
//
// One item a block, packed tiles through registers, suspended waits and generic addresses, and now (attention alone, us, in turn on one GPU):
// 4096 queries over 4096 tokens, 8 sequences of 32 heads, 2 bit, 2661 and 2228; 1003 queries with four heads per KV head over 7403 tokens, 4 bit,
// 276 and 251; 28 x 32 heads of 165 tokens, 2 bit, 138 and 77; of 335, 3 bit, 276 and 150; 57 x 8 KV heads with four heads each, 1064 tokens,
// 4 bit, 32-token groups 2366 and 1539; 8 KV heads with eight heads each, 100 queries over 192 tokens 23.3 and 17.0.  The outputs are the same
// bits.  Relative error of the outputs against 64 bits: 2.6e-6 and 8.2e-6 for the first two.
#include "tile_words.cuh"

namespace kvsink {

namespace {

constexpr int PR_STEP = 64;                     // tokens per step
constexpr int PR_ROWS = 256;                    // rows per block
constexpr int PR_STAGES = 2;                    // expanded steps in flight
constexpr int PR_WORDS = 4;                     // packed steps in flight: one on its way, one with the parameter warps, two with the expanding ones
constexpr int PR_SBUFS = 3;                     // score buffers, taken in turn by the two row tiles
constexpr int PR_THREADS = 20 * 32;
constexpr int PR_HALF = 16384;                  // 64 tokens x 128 channels of fp16
constexpr int PR_HDRS = 8;
constexpr int PR_GRID = 148;                    // blocks: one to an SM
constexpr int PR_ROUNDS = 95;                   // work items of a block at most
// A zero point up to this size is subtracted from the code in fp16 exactly; farther ones go through an additive term.
constexpr float PR_NEAR = 1000.f;
// Limit of a wait: 8 ms and more (a poll comes back after 60 clocks at the earliest); a real wait is for a step's work of the same block, some
// 10 us.  So nothing that goes with the number of sinks stands between two steps (a search in the ascending list of positions goes with its logarithm).
// Counted in polls and not in clocks: a look at the clock every 256 polls made the kernel 6 % slower (2661 and 2825 us), since every wait
// of every role holds a copy of the loop and code is what it has least room for.  No suspend-time hint: with one a poll is twice the
// instructions, and the waiting warps' polls take the issue slots of the working ones (the chunk above 424000 and 408000 clocks a block).
constexpr int PR_WAIT_POLLS = 1 << 18;
constexpr int PR_ROWS_KEPT = 8;                 // sink rows of a step that the parameter warps leave in shared memory

struct alignas(16) StepHeader {
    float k_down, k_up;                         // 2^-kappa, 2^kappa: the step's units of K
    uint32_t dead[2];                           // sink tokens that are missing from the position list
    uint32_t k_sink[2];                         // sink tokens of the step (once for the keys' side, once for the values')
    int k_far;                                  // some zero point is beyond PR_NEAR
    int second;                                 // first tile of the step that belongs to its second key group
    float v_up, e;                              // 2^e and e: units of V
    uint32_t v_sink[2];
    int v_far;
    int pad[3];
};

// A value that is the same in all lanes, in a uniform register: loops and branches over values from shared memory are otherwise taken for
// divergent ones
__device__ __forceinline__ int uniform(int x) { return __reduce_max_sync(0xffffffffu, x); }

struct alignas(32) Work {                       // a row block of one KV head: rows row0 ... end - 1, 256 at most
    int unit, b, h, row0, end;
    int n0, n1, n_steps;                        // steps of the two row tiles and of both; n_steps = 0: there is none
    __device__ __forceinline__ Work take() const
    {
        return {uniform(unit), uniform(b), uniform(h), uniform(row0), uniform(end), uniform(n0), uniform(n1), uniform(n_steps)};
    }
};

struct PromptSmem {
    unsigned char k[PR_STAGES][2][PR_HALF];     // [token 64][channel 128] hi, lo: two panels of 64 channels, 128-byte swizzle
    unsigned char v[PR_STAGES][2][PR_HALF];     // [channel 128][token 64] hi, lo: 128-byte swizzle
    unsigned char q[2 * PR_HALF];               // queries of row tile 1: [row 128][channel 128], two panels of 64 channels
    // from here on the first index is 0 for keys and 1 for values
    unsigned char words[2][PR_WORDS][4 * 1024]; // packed tiles of a step, as they are in memory
    uint4 tab[2][2][128];                       // scale hi, lo and zero terms: keys by the step's group (two at most) and channel pair, values by channel group and token pair
    uint2 add[2][2][128];                       // additive terms hi, lo of far zero points
    float raw[2][2][2][256];                    // scales and zero points of a step as they are in memory: keys [group][channel], values [token][group]
    StepHeader hdr[PR_HDRS];
    Work work[PR_ROUNDS + 1];                    // the block's work items, and an empty one behind them
    int rank[2][2][64];                         // side buffer rows of the step's sink tokens, in token order
    uint4 kept[2][2][PR_ROWS_KEPT][16];         // the first of those rows
    uint64_t k_full[PR_STAGES], k_empty[PR_STAGES], v_full[PR_STAGES], v_empty[PR_STAGES];
    uint64_t raw_full[2][2], par_full[2][2], par_empty[2][2], hdr_full[PR_HDRS];
    uint64_t s_full[2][PR_SBUFS], p_full[PR_SBUFS], o_done[PR_SBUFS], o_last[2], q_full[2], drained[2];
    uint32_t tmem;
    int failed;
    uint8_t odd[PR_ROUNDS + 1];                 // by work item: a sink token of its steps has a value that is infinite or NaN
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
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                     : "=r"(ok) : "r"(a), "r"(parity) : "memory");
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
// 16 lanes x 32 columns: lane l gets columns 2 (l % 4) + 8 x, + 1 of row l / 4 in r[4 x], r[4 x + 1] and of row l / 4 + 8 behind them
__device__ __forceinline__ void tm_load_rows16(uint32_t addr, uint32_t (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                   "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(addr) : "memory");
}
__device__ __forceinline__ void tm_store_rows16(uint32_t addr, const uint32_t (&r)[16])
{
    asm volatile("tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
                   "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
// Neighbouring lanes trade halves of 16-byte units: in, two words each of a unit of column block a and of one of block b (the layout of
// tm_load_rows16); out, a's unit whole in the even lane and b's in the odd one.  Lane l then has unit 2 (l % 2) + (l / 2) % 2 of the
// four that blocks a and b make.
__device__ __forceinline__ uint4 pair_up(uint32_t a0, uint32_t a1, uint32_t b0, uint32_t b1, bool odd)
{
    const uint32_t g0 = __shfl_xor_sync(0xffffffffu, odd ? a0 : b0, 1), g1 = __shfl_xor_sync(0xffffffffu, odd ? a1 : b1, 1);
    return odd ? make_uint4(g0, g1, b0, b1) : make_uint4(a0, a1, g0, g1);
}
__device__ __forceinline__ void unpair(const uint4 &u, bool odd, uint32_t &a0, uint32_t &a1, uint32_t &b0, uint32_t &b1)      // the way back
{
    const uint32_t g0 = __shfl_xor_sync(0xffffffffu, odd ? u.x : u.z, 1), g1 = __shfl_xor_sync(0xffffffffu, odd ? u.y : u.w, 1);
    a0 = odd ? g0 : u.x; a1 = odd ? g1 : u.y;
    b0 = odd ? u.z : g0; b1 = odd ? u.w : g1;
}
__device__ __forceinline__ void tm_wait_load() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_wait_store() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Untiled bulk copy into shared memory: addresses and size are multiples of 16 bytes.
__device__ __forceinline__ void bulk_copy(void *to, const void *from, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_addr(to)), "l"(from), "r"(bytes), "r"(smem_addr(bar)) : "memory");
}

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

// Fields of one 16 x 16 matrix of a packed tile, each half ORed into 1024.0: the half is 1024 + code * 2^position.  x: the matrix's
// word (4 bit), or the word of two matrices and the shift that brings this one's fields down; h: the word of the 3-bit codes' high bits.
template <int BITS>
__device__ __forceinline__ void matrix_fields(uint32_t x, uint32_t h, int shift, bool odd_word, uint32_t (&f)[4])
{
    constexpr uint32_t ONE = 0x64006400u;
    if constexpr (BITS == 2) {
        x >>= shift;
        f[0] = (x & 0x00030003u) | ONE; f[1] = (x & 0x000c000cu) | ONE; f[2] = (x & 0x00300030u) | ONE; f[3] = (x & 0x00c000c0u) | ONE;
    } else if constexpr (BITS == 4) {
        const uint32_t y = x >> 8;
        f[0] = (x & 0x000f000fu) | ONE; f[1] = (x & 0x00f000f0u) | ONE; f[2] = (y & 0x000f000fu) | ONE; f[3] = (y & 0x00f000f0u) | ONE;
    } else {
        const uint32_t hh = odd_word ? h << 2 : h;
        const uint32_t me = ((x & 0x33333333u) | (hh & 0xccccccccu)) >> shift, mo = (((x >> 2) & 0x33333333u) | ((hh >> 1) & 0xccccccccu)) >> shift;
        f[0] = (me & 0x00070007u) | ONE; f[1] = (mo & 0x00070007u) | ONE; f[2] = (me & 0x00700070u) | ONE; f[3] = (mo & 0x00700070u) | ONE;
    }
}
// log2 of the position factor of a field, by row half and column half of its matrix
template <int BITS>
__host__ __device__ constexpr int field_shift(int row_half, int col_half)
{
    return BITS == 2 ? 2 * row_half + 4 * col_half : (BITS == 4 ? 4 * row_half : 4 * col_half);
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
    uint32_t rep_mul, rep_shift;                // row / rep = row * rep_mul >> rep_shift, for rows below 2^30
};

template <int BITS>
__global__ void __launch_bounds__(PR_THREADS, 1) prompt_kernel(Params p, kvsink_cache c, PromptArgs a)
{
    constexpr int D = 128;
    constexpr float QMAX = (float)((1 << BITS) - 1);
    constexpr int TILE = KVSINK_TILE * D * BITS / 8;
    extern __shared__ unsigned char smem_raw[];
    PromptSmem &sm = *reinterpret_cast<PromptSmem *>(smem_raw + (-smem_addr(smem_raw) & 1023u));      // not through an integer: the accesses would be generic ones
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);

    const int n_rows = a.T * p.rep, seq_len = c.seq_len, n_body = seq_len / p.G * p.G;
    // cached tokens that row r sees
    auto query_of = [&](int r) { return (int)((uint64_t)(uint32_t)r * a.rep_mul >> a.rep_shift); };       // r / p.rep
    auto row_limit = [&](int r) { return a.q_pos0 + query_of(min(r, n_rows - 1)) + 1; };
    // every thread alike, and before anything is set up; index checks of single accesses are at the accesses
    if (!in_bounds(n_rows > 0 && a.q_pos0 >= 0 && a.q_pos0 + a.T <= seq_len && seq_len <= p.max_seq && p.cap >= 0, c.status)) {
        pdl_wait();
        return;
    }

    // Work items: the row blocks of all (sequence, KV head) units, longest first.  The grid's blocks take them in turn, every other
    // round the other way about, so that all get much the same number of steps.  Rows are counted off from the end, so the units' blocks
    // that are not full are their first rows and come last: behind an item without a second row tile a block has no other that has one
    // (its warps would wait for the first tile's steps of all items between).
    if (tid <= PR_ROUNDS) {
        const int units = p.B * p.Hkv, g = (int)gridDim.x, x = (int)blockIdx.x;
        const int64_t at = (int64_t)tid * g + (tid & 1 ? g - 1 - x : x);
        Work w = {0, 0, 0, 0, 0, 0, 0, 0};
        if (tid < PR_ROUNDS && at < (int64_t)units * a.blocks) {
            const int back = (int)at / units;
            w.unit = (int)at - back * units;
            w.b = w.unit / p.Hkv;
            w.h = w.unit - w.b * p.Hkv;
            w.end = n_rows - back * PR_ROWS;
            w.row0 = max(w.end - PR_ROWS, 0);
            auto tile_steps = [&](int r0) { return r0 < w.end ? (row_limit(min(r0 + 127, w.end - 1)) + PR_STEP - 1) / PR_STEP : 0; };
            w.n0 = tile_steps(w.row0);
            w.n1 = tile_steps(w.row0 + 128);
            w.n_steps = max(w.n0, w.n1);
        }
        sm.work[tid] = w;
        sm.odd[tid] = 0;
    }
    if (warp == 16) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&sm.tmem)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        if (lane == 0) {
            for (int i = 0; i < PR_STAGES; ++i) {
                bar_init(&sm.k_full[i], 4); bar_init(&sm.k_empty[i], 1);
                bar_init(&sm.v_full[i], 4); bar_init(&sm.v_empty[i], 1);
            }
            for (int i = 0; i < PR_SBUFS; ++i) { bar_init(&sm.s_full[0][i], 1); bar_init(&sm.s_full[1][i], 1); bar_init(&sm.p_full[i], 4); bar_init(&sm.o_done[i], 1); }
            for (int i = 0; i < 2; ++i) {
                for (int y = 0; y < 2; ++y) { bar_init(&sm.raw_full[i][y], 1); bar_init(&sm.par_full[i][y], 1); bar_init(&sm.par_empty[i][y], 4); }
                bar_init(&sm.q_full[i], 4);
                bar_init(&sm.o_last[i], 1);
                bar_init(&sm.drained[i], 1);
            }
            for (int i = 0; i < PR_HDRS; ++i) bar_init(&sm.hdr_full[i], 2);
            sm.failed = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        tc_fence_before();
    }
    __syncthreads();
    in_bounds(tid == 0 || tid > PR_ROUNDS || sm.work[tid].n1 == 0 || sm.work[tid - 1].n1 > 0, c.status);      // debug builds: the order of the work items
    tc_fence_after();
    pdl_wait();
    pdl_release();

    // 96 registers per thread at launch: 2 x 128 threads to 128, 2 x 128 to 80, 128 to 64 add up to the same 61440
    if (warp < 8) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 128;");
        // ---------------- softmax: thread = row ----------------
        const int i = warp >> 2, quad = lane >> 2, odd = lane & 1, unit0 = 2 * odd + ((lane >> 1) & 1);    // rows and 16-byte units of pair_up
        const uint32_t lanes = (uint32_t)(warp & 3) << 21;                   // this warp's 32 lanes of TMEM
        const uint32_t t_o = lanes + TM_O + 128 * i;
        const float qscale = 1.4426950408889634f * rsqrtf((float)D);
        // row of a.out and a.lse
        auto out_row = [&](const Work &w, int r) { const int qt = query_of(r); return (w.b * p.Hq + w.h * p.rep + r - qt * p.rep) * a.T + qt; };
        // The queries of a work item's row tile, four lanes to 64 bytes of a row (a lane to a row of its own took 4000 clocks)
        auto load_queries = [&](const Work &w) {
            if (!(i ? w.n1 : w.n0)) return;
            const int first = w.row0 + 128 * i + 32 * (warp & 3) + quad;
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {                           // rows quad, quad + 8 of the warp's lower or upper 16
                uint4 v[2][4];
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    const int row = first + 16 * half + 8 * y, r = min(row, n_rows - 1), qt = query_of(r);
                    const uint4 *src = (const uint4 *)(a.q + w.b * a.q_sb + (w.h * p.rep + r - qt * p.rep) * a.q_sh + qt * a.q_st) + unit0;
#pragma unroll
                    for (int x = 0; x < 4; ++x) v[y][x] = row < w.end ? __ldg(src + 4 * x) : make_uint4(0u, 0u, 0u, 0u);
                }
                if (i == 0) {
#pragma unroll
                    for (int x = 0; x < 4; x += 2) {
                        uint32_t r[16];
#pragma unroll
                        for (int z = 0; z < 2; ++z)
#pragma unroll
                            for (int y = 0; y < 2; ++y) unpair(v[y][x + z], odd, r[8 * z + 2 * y], r[8 * z + 2 * y + 1], r[8 * z + 4 + 2 * y], r[8 * z + 4 + 2 * y + 1]);
                        tm_store_rows16(lanes + ((uint32_t)(16 * half) << 16) + TM_Q + 16 * x, r);
                    }
                } else {
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        const int r = 32 * (warp & 3) + 16 * half + 8 * y + quad;
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int ck = 4 * x + unit0;
                            *reinterpret_cast<uint4 *>(sm.q + (ck >> 3) * PR_HALF + r * 128 + (((ck & 7) ^ (r & 7)) << 4)) = v[y][x];
                        }
                    }
                }
            }
            if (i == 0) {
                tm_wait_store();
                tc_fence_before();
            } else {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            __syncwarp();
            if (lane == 0) bar_arrive(&sm.q_full[i]);
        };
        // Counts that go on from one work item to the next: score items (steps of the tiles, in turn), steps, and this tile's score items.
        // The scores' barriers are the tile's own, taken in turn by its items: one's next use comes after three items of the tile, for which
        // this warp's weights are needed.  Weights and outputs have barriers per score buffer: the buffer's next user comes three items
        // on, behind the same tile's next item, whose outputs need this warp's weights.  Behind a tile's last item of a work item the
        // other tile may have more, which pass through the same buffers without it, so the end of a tile has a barrier of its own
        int items = 0, hdr0 = 0, own = 0, own_phase = 0, ends = 0;
        // first a work item without steps, behind which the first queries are loaded
        Work w = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll 1
        for (int round = 0;; ++round) {
            bool ok = true;
            const int steps = i ? w.n1 : w.n0;
            const int row = w.row0 + 128 * i + 32 * (warp & 3) + lane;
            const bool valid = row < w.end;
            const int lim = row_limit(row), lim_min = row_limit(row - lane);
            // weights are 2^(score - M - e) with M the row's reference, moved only when a weight would leave fp16: the weights of a
            // step stay below 2^15 and the values below 2^15 in the step's units 2^-e, so that P V is in the units of 2^-M throughout
            float M = M_INIT, l = 0.f;
            int item = items + i, before = 0;
#pragma unroll 1
            for (int j = 0; j < steps; before = item, item += 1 + (j + i < (i ? w.n0 : w.n1)), ++j) {
                const int sb = item % PR_SBUFS, hj = hdr0 + j;
                const uint32_t t_s = lanes + TM_S + 64 * sb;
                // the step's header first: it is there long before the scores.  Its barrier is never a phase behind: the tile has seen the scores
                // of one of the four steps before (two tiles end within three steps of one another), for which the header eight back was needed
                if (!(ok = bar_wait_warp(&sm.hdr_full[hj & (PR_HDRS - 1)], (hj / PR_HDRS) & 1, &sm.failed))) break;
                const StepHeader &hd = sm.hdr[hj & (PR_HDRS - 1)];
                const float c1 = qscale * hd.k_down, ef = hd.e, vup = hd.v_up;
                const uint32_t dead0 = hd.dead[0], dead1 = hd.dead[1];
                if (!(ok = bar_wait_warp(&sm.s_full[i][own], own_phase, &sm.failed))) break;
                if (++own == PR_SBUFS) { own = 0; own_phase ^= 1; }
                tc_fence_after();
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
                float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};      // four chains: one took 500 clocks
#pragma unroll
                for (int x = 0; x < 32; x += 4) {
                    m4[0] = max3(m4[0], __uint_as_float(v0[x]), __uint_as_float(v0[x + 1]));
                    m4[1] = max3(m4[1], __uint_as_float(v0[x + 2]), __uint_as_float(v0[x + 3]));
                    m4[2] = max3(m4[2], __uint_as_float(v1[x]), __uint_as_float(v1[x + 1]));
                    m4[3] = max3(m4[3], __uint_as_float(v1[x + 2]), __uint_as_float(v1[x + 3]));
                }
                float top = max3(max3(m4[0], m4[1], m4[2]), m4[3], -INFINITY);
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
            if (!ok) break;
            items += w.n0 + w.n1;
            hdr0 += w.n_steps;
            const int oq = out_row(w, min(row, n_rows - 1));
            w = sm.work[round].take();
            load_queries(w);                     // the tile's last scores are there: its queries have been read
            if (steps > 0) {
                if (!bar_wait_warp(&sm.o_last[i], ends++ & 1, &sm.failed)) break;
                tc_fence_after();
                const float inv = l > 0.f ? 1.f / l : 0.f;
                // four lanes to 64 bytes of a row; with a lane to a row of its own the stores took 8000 clocks
#pragma unroll 1
                for (int half = 0; half < 2; ++half) {
                    float f[2];
                    float4 *dst[2];
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        const int from = 16 * half + 8 * y + quad;
                        f[y] = __shfl_sync(0xffffffffu, inv, from);
                        const int to = __shfl_sync(0xffffffffu, valid ? oq : -1, from);
                        dst[y] = to < 0 ? nullptr : (float4 *)(a.out + (size_t)to * D) + unit0;
                    }
#pragma unroll 1
                    for (int x = 0; x < 4; ++x) {
                        uint32_t o[16];
                        tm_load_rows16(t_o + ((uint32_t)(16 * half) << 16) + 32 * x, o);
                        tm_wait_load();
#pragma unroll
                        for (int y = 0; y < 2; ++y)
#pragma unroll
                            for (int z = 0; z < 2; ++z) {
                                const uint4 u = pair_up(o[8 * z + 2 * y], o[8 * z + 2 * y + 1], o[8 * z + 4 + 2 * y], o[8 * z + 4 + 2 * y + 1], odd);
                                if (dst[y])
                                    dst[y][8 * x + 4 * z] = make_float4(__uint_as_float(u.x) * f[y], __uint_as_float(u.y) * f[y],
                                                                        __uint_as_float(u.z) * f[y], __uint_as_float(u.w) * f[y]);
                            }
                    }
                }
                if (a.lse && valid) a.lse[oq] = l > 0.f ? (M + log2f(l)) * 0.6931471805599453f : -INFINITY;
            }
            if (w.n_steps == 0) break;
        }
        // Values of sink tokens that are infinite or NaN were left out of the products, where they would reach every row of a tile; only rows
        // that see the token get them.  This comes behind the block's last item and not behind each: it takes as long as the list of sinks is,
        // and nobody waits for this warp any more (a wait of the other roles' is bounded by what a step takes).  A lane has four channels; the
        // sums of the tokens that a row sees go on to the next row, which sees no fewer.
        __syncwarp();
#pragma unroll 1
        for (int round = 0; uniform(sm.work[round].n_steps) > 0; ++round) {
            if (!uniform(*(volatile uint8_t *)&sm.odd[round])) continue;
            const Work w = sm.work[round].take();
            const uint32_t *bm = c.sink_bitmask + (size_t)w.b * p.mask_words;
            const int32_t *pos = c.sink_pos + (size_t)w.b * p.cap;
            const uint2 *values = (const uint2 *)((const __half *)c.sink_v + (size_t)w.unit * p.cap * D) + lane;
            const int n_pos = min(c.sink_count[w.b], p.cap), row0 = w.row0 + 128 * i + 32 * (warp & 3);
            float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
            int y = 0;
#pragma unroll 1
            for (int row = row0; row < min(row0 + 32, w.end); ++row) {
                const int lim = row_limit(row);
#pragma unroll 1
                for (; y < n_pos && pos[y] < lim; ++y) {
                    if (pos[y] < 0 || !in_bounds(pos[y] < p.max_seq, c.status) || !mask_bit(bm, pos[y])) continue;
                    const uint2 v = values[(size_t)y * (D / 4)];
                    const float2 lo = __half22float2(as_half2(v.x)), hi = __half22float2(as_half2(v.y));
                    if (!is_finite(lo.x)) sum.x += lo.x;
                    if (!is_finite(lo.y)) sum.y += lo.y;
                    if (!is_finite(hi.x)) sum.z += hi.x;
                    if (!is_finite(hi.y)) sum.w += hi.y;
                }
                if (is_finite(sum.x) && is_finite(sum.y) && is_finite(sum.z) && is_finite(sum.w)) continue;
                float4 *to = (float4 *)(a.out + (size_t)out_row(w, row) * D) + lane, o = *to;
                *to = make_float4(o.x + sum.x, o.y + sum.y, o.z + sum.z, o.w + sum.w);
            }
        }
    } else if (warp < 16) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        // ---------------- expansion of keys (warps 8-11) and values (12-15); warp w owns channels 32 w ... 32 w + 31 ----------------
        const bool keys = warp < 12;
        const int role = !keys, w = warp & 3, t = lane & 3;
        // stmatrix: lane l gives the address of row l % 8 of the 8 x 8 matrix l / 8 (row half l/8 % 2, column half l / 16)
        const int sr = (lane & 7) + 8 * ((lane >> 3) & 1), sc = lane >> 4;
        // keys: row = token, 16-byte chunk = eight channels, two panels of 64; values: row = channel, chunk = eight tokens
        auto place = [](int r, int ck) { return (uint32_t)((ck >> 3) * 8192 + r * 128 + (((ck & 7) ^ (r & 7)) << 4)); };
        // sink tokens: their exact rows over the expanded ones
        auto put_sinks = [&](int unit, const uint32_t (&sink)[2], const int *ranks, const uint4 (*kept)[16], uint32_t base, float up) {
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
        uint64_t *full = keys ? sm.k_full : sm.v_full, *empty = keys ? sm.k_empty : sm.v_empty;
        // The warp's eight matrices of a step go two at a time, with one pair of table entries: of keys, matrix x / 2 of the warp's two in tiles
        // 2 (x % 2) and the one behind; of values, both matrices of tile x.  A matrix's rows lie 32 x apart under the swizzle by its column
        // chunk (keys: the matrix, values: the tile), 2048 bytes by the other one
        const int jg = 32 * w / p.Gv;                                    // value channel group of the warp's channels
        const uint32_t at0 = keys ? place(sr, 4 * w + sc) : place(32 * w + sr, sc);
        const int entry0 = keys ? 16 * w + t : 32 * jg + t;
        const unsigned char *const word0 = &sm.words[role][0][0] + 16 * lane + (BITS == 4 ? 512 * (w >> 1) + 8 * (w & 1) : 4 * w);
        const int high = 512 + 8 * lane + 4 * (w >> 1) - (16 * lane + 4 * w);
        int stage = 0, phase = 0, s = 0;                                 // s: steps of all work items
        bool ok = true;
#pragma unroll 1
        for (int round = 0; ok; ++round) {
            const int n_steps = uniform(sm.work[round].n_steps), unit = uniform(sm.work[round].unit);
            if (n_steps == 0) break;
            const __half *tail = (const __half *)c.k_tail + (size_t)unit * p.G * D;
#pragma unroll 1
            for (int j = 0; j < n_steps; ++j, ++s) {
                const int buf = s & 1;
                if (!(ok = bar_wait_warp(&sm.par_full[role][buf], (s >> 1) & 1, &sm.failed))) break;
                if (s >= PR_STAGES && !(ok = bar_wait_warp(&empty[stage], phase ^ 1, &sm.failed))) break;
                const StepHeader &hd = sm.hdr[s & (PR_HDRS - 1)];
                const int second = hd.second;
                const uint32_t *sinks = keys ? hd.k_sink : hd.v_sink;
                const uint32_t sink[2] = {sinks[0], sinks[1]};
                const float up = keys ? hd.k_up : hd.v_up;
                const bool far = keys ? hd.k_far : hd.v_far;
                const uint4 *tab = sm.tab[role][buf] + entry0;
                const unsigned char *words = word0 + (s & (PR_WORDS - 1)) * (4 * 1024);
                const uint32_t base = smem_addr(keys ? &sm.k[stage][0][0] : &sm.v[stage][0][0]);
                // two matrices' words and table entries
                struct Two { uint32_t lo[2], hi[2]; uint4 e0, e1; };
                auto load = [&](int x, Two &o) {
                    const int out = keys ? x >> 1 : x, in = keys ? 2 * (x & 1) : 0;
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        const unsigned char *at = words + (keys ? in + y : out) * TILE;
                        o.lo[y] = *(const uint32_t *)(at + (BITS == 4 ? 4 * (keys ? out : y) : 0));
                        o.hi[y] = BITS == 3 ? *(const uint32_t *)(at + high) : 0u;
                    }
                    const uint4 *e = tab + 8 * out + (keys && in >= second ? 64 : 0);
                    o.e0 = e[0];
                    o.e1 = e[4];
                };
#pragma unroll 1
                for (int x = 0; x < 4; ++x) {
                    Two cur;
                    load(x, cur);
                    const int out = keys ? x >> 1 : x, in = keys ? 2 * (x & 1) : 0;
                    const uint32_t to = base + (at0 ^ (32 * out)) + 2048 * in;
                    const int shift[2] = {keys ? 8 * out : 0, keys ? 8 * out : 8};
                    if (!far && (!keys || (j * PR_STEP + 16 * in + 32 <= n_body && second != in + 1))) {
                        uint32_t f[2][4], hi[2][4], lo[2][4];
#pragma unroll
                        for (int y = 0; y < 2; ++y) {
                            matrix_fields<BITS>(cur.lo[y], cur.hi[y], shift[y], w & 1, f[y]);
                            expand_matrix<BITS, false>(f[y], cur.e0, cur.e1, make_uint2(0u, 0u), make_uint2(0u, 0u), hi[y], lo[y]);
                        }
                        st_matrix<0>(to, hi[0]);
                        st_matrix<PR_HALF>(to, lo[0]);
                        st_matrix<2048>(to, hi[1]);
                        st_matrix<2048 + PR_HALF>(to, lo[1]);
                    } else {                                  // far zero points, key tiles of the open group or of two groups
                        const uint2 *add = sm.add[role][buf] + entry0;
#pragma unroll 1
                        for (int y = 0; y < 2; ++y) {
                            uint32_t hi[4], lo[4];
                            const int mm = keys ? out : y, tok = j * PR_STEP + 16 * (keys ? in + y : out);
                            if (keys && tok >= n_body) {      // exact fp16 rows from the tail
                                const __half2 up2 = __half2half2(__float2half(up));
#pragma unroll
                                for (int z = 0; z < 4; ++z) {
                                    const int tk = tok + (lane >> 2) + 8 * (z & 1);
                                    const uint32_t v = tk < seq_len && in_bounds(tk - n_body < p.G, c.status) ? *(const uint32_t *)(tail + (size_t)(tk - n_body) * D + 16 * (2 * w + mm) + 8 * (z >> 1) + 2 * t) : 0u;
                                    hi[z] = as_u32(__hmul2_rn(as_half2(v), up2));
                                    lo[z] = 0u;
                                }
                            } else {
                                uint32_t f[4];
                                matrix_fields<BITS>(y ? cur.lo[1] : cur.lo[0], y ? cur.hi[1] : cur.hi[0], y ? shift[1] : shift[0], w & 1, f);
                                const int e = 8 * out + (keys && in + y >= second ? 64 : 0);
                                if (far) {
                                    expand_matrix<BITS, true>(f, tab[e], tab[e + 4], add[e], add[e + 4], hi, lo);
                                } else {
                                    expand_matrix<BITS, false>(f, tab[e], tab[e + 4], make_uint2(0u, 0u), make_uint2(0u, 0u), hi, lo);
                                }
                            }
                            st_matrix<0>(to + 2048 * y, hi);
                            st_matrix<PR_HALF>(to + 2048 * y, lo);
                        }
                    }
                }
                if (sink[0] | sink[1]) put_sinks(unit, sink, sm.rank[role][buf], sm.kept[role][buf], base, up);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) { bar_arrive(&full[stage]); bar_arrive(&sm.par_empty[role][buf]); }
                if (++stage == PR_STAGES) { stage = 0; phase ^= 1; }
            }
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
        int m0 = 0, m1 = 0, items = 0;
        int i = 0, j = 0, stage = 0, phase = 0, buf = 0, bphase = 0;       // the item: tile, step; its step's stage, its score buffer
        auto work = [&](int round) {       // the next work item; none after a wait that ran out
            m0 = uniform(sm.work[round].n0);
            m1 = uniform(sm.work[round].n1);
            items = m0 + m1;
            i = j = 0;
            return m0 > 0 && !__any_sync(0xffffffffu, *(volatile int *)&sm.failed);
        };
        auto next = [&](bool last) {
            if (last) {
                ++j;
                i = j < m0 ? 0 : 1;
                if (++stage == PR_STAGES) { stage = 0; phase ^= 1; }
            } else {
                i = 1;
            }
            if (++buf == PR_SBUFS) { buf = 0; bphase ^= 1; }
        };
        if (!scores) {
#pragma unroll 1
            for (int round = 0; work(round); ++round)
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
                    next(last);
                }
        } else {
            int seen0 = 0, seen1 = 0, own0 = 0, own1 = 0;      // queries of the tiles so far; barriers of the tiles' next scores
            bool first = true;                                 // the first PR_SBUFS items find their buffers free
#pragma unroll 1
            for (int round = 0; work(round); ++round) {
                bar_wait_warp(&sm.q_full[0], seen0++ & 1, &sm.failed);
                if (m1 > 0) bar_wait_warp(&sm.q_full[1], seen1++ & 1, &sm.failed);
#pragma unroll 1
                for (int it = 0; it < items; ++it) {               // S = Q K_lo + Q K_hi
                    if (i == 0 || j >= m0) bar_wait_warp(&sm.k_full[stage], phase, &sm.failed);
                    if (!first) bar_wait_warp(&sm.o_done[buf], bphase ^ 1, &sm.failed);
                    if (buf == PR_SBUFS - 1) first = false;
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
                        tc_commit(&sm.s_full[i][i ? own1 : own0]);
                        if (last) tc_commit(&sm.k_empty[stage]);
                    }
                    __syncwarp();
                    if (i) own1 = own1 == PR_SBUFS - 1 ? 0 : own1 + 1;
                    else own0 = own0 == PR_SBUFS - 1 ? 0 : own0 + 1;
                    next(last);
                }
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
        const int role = !keys, coded = keys ? n_body : seq_len;         // tokens below it have codes
        const size_t per_unit = keys ? (size_t)(p.max_seq / p.G) * D : (size_t)p.max_seq * p.NGv;
        const __half *all_rows = (const __half *)(keys ? c.sink_k : c.sink_v) + 8 * (lane & 15);
        const uint8_t *codes = keys ? c.k_codes : c.v_codes;
        // A step's packed tiles and parameters come into shared memory a step ahead, as they are: of the (at most two) key groups that meet
        // the step (G is 32, 64 or at least 128), of its tokens' values.  Entries: keys, two channel pairs a lane for each group; values,
        // one token pair a lane for each channel group.
        const float *ps = keys ? c.k_scale : c.v_scale, *pz = keys ? c.k_zero : c.v_zero;
        // group of the step's first token, tokens of the step before the next group, and the step's entries
        int g0 = 0, second = p.G;
        auto count = [&](int j, int second) {
            const int body = n_body - j * PR_STEP;
            return keys ? (body > 0 ? (min(body, PR_STEP) > second ? 4 : 2) : 0) : p.NGv;
        };
        auto fetch = [&](int unit, int j, int g, int s) {                // s: steps of all work items, whose buffers they take in turn
            const int left = coded - j * PR_STEP;
            const uint32_t n_code = left > 0 ? (min(left, PR_STEP) + KVSINK_TILE - 1) / KVSINK_TILE * (uint32_t)TILE : 0u;
            const uint32_t n_par = 4u * (keys ? D * (count(j, second) >> 1) : p.NGv * min(PR_STEP, p.max_seq - j * PR_STEP));
            const int64_t at = unit * per_unit + (keys ? (int64_t)g * D : (int64_t)j * PR_STEP * p.NGv);
            const bool in = in_bounds((n_code == 0 || j * PR_STEP + (int)(n_code / TILE) * KVSINK_TILE <= p.max_seq) && (!keys || (g + (int)n_par / (4 * D)) * p.G <= max(n_body, g * p.G)), c.status);
            if (elect_one()) {
                uint64_t *bar = &sm.raw_full[role][s & 1];
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(in ? n_code + 2 * n_par : 0u) : "memory");
                if (in && n_code) bulk_copy(sm.words[role][s & (PR_WORDS - 1)], codes + ((int64_t)unit * p.max_seq + j * PR_STEP) * p.row_bytes, n_code, bar);
                if (in && n_par) {
                    bulk_copy(sm.raw[role][s & 1][0], ps + at, n_par, bar);
                    bulk_copy(sm.raw[role][s & 1][1], pz + at, n_par, bar);
                }
            }
            __syncwarp();
        };
        struct Pair { float s0, z0, s1, z1; };
        auto pair = [&](int j, int n, int s) {
            Pair r = {0.f, 0.f, 0.f, 0.f};
            const float *raw = sm.raw[role][s & 1][0];
            if (keys) {
                const float *at = raw + 64 * n + 2 * lane;
                const float2 s = *(const float2 *)at, z = *(const float2 *)(at + 256);
                r.s0 = s.x; r.s1 = s.y; r.z0 = z.x; r.z1 = z.y;
            } else {
                const float *at = raw + 2 * lane * p.NGv + n;
                const int left = seq_len - (j * PR_STEP + 2 * lane);
                if (left > 0) { r.s0 = at[0]; r.z0 = at[256]; }
                if (left > 1) { r.s1 = at[p.NGv]; r.z1 = at[256 + p.NGv]; }
            }
            return r;
        };
        auto mask_word = [&](int b, int j, int x) {
            const int left = seq_len - (j * PR_STEP + 32 * x);
            const uint32_t word = left > 0 && in_bounds(2 * j + x < p.mask_words, c.status) ? __ldg(c.sink_bitmask + (size_t)b * p.mask_words + 2 * j + x) : 0u;
            return left > 0 && left < 32 ? word & ((1u << left) - 1u) : word;
        };
        uint32_t bits[2];
        int asked = 0;
        // the packed tiles, parameters and mask words of a step ahead
        auto ahead = [&](int unit, int b, int j, int s) {
            second -= PR_STEP;
            while (second <= 0) { second += p.G; ++g0; }
            if (j == 0) { second = p.G; g0 = 0; }
            fetch(unit, j, g0, s);
            asked = s + 1;
            bits[0] = mask_word(b, j, 0);
            bits[1] = mask_word(b, j, 1);
        };
        int s = 0;
        bool ok = true;
        ahead(uniform(sm.work[0].unit), uniform(sm.work[0].b), 0, 0);
#pragma unroll 1
        for (int round = 0; ok; ++round) {
            const Work w = sm.work[round].take();
            if (w.n_steps == 0) break;
            const int32_t *pos = c.sink_pos + (size_t)w.b * p.cap;
            const int n_pos = min(c.sink_count[w.b], p.cap);
            const __half *rows = all_rows + (size_t)w.unit * p.cap * D;
            int rank0 = 0;                                                   // sink tokens before the step
#pragma unroll 1
            for (int j = 0; j < w.n_steps; ++j, ++s) {
                const int buf = s & 1, tok0 = j * PR_STEP;
                const uint32_t sink[2] = {bits[0], bits[1]};
                const int split = second, n_entries = count(j, second);
                if (!(ok = bar_wait_warp(&sm.raw_full[role][buf], (s >> 1) & 1, &sm.failed))) break;
                const bool in_work = j + 1 < w.n_steps;
                // the next step, or the next work item's first
                const Work &next = sm.work[round + !in_work];
                const int unit = uniform(next.unit), b = uniform(next.b);
                if (uniform(next.n_steps) > 0) ahead(unit, b, in_work ? j + 1 : 0, s + 1);
                float top = 0.f;
                bool far = false, odd = false;
#pragma unroll 1
                for (int n = 0; n < n_entries; n += 2) {                     // largest |scale * (code - zero)|; two entries' chains at a time
                    const int n1 = min(n + 1, n_entries - 1);
                    const Pair r = pair(j, n, s), q = pair(j, n1, s);
                    const float m = max3(r.s0 * fmaxf(fabsf(r.z0), fabsf(QMAX - r.z0)), r.s1 * fmaxf(fabsf(r.z1), fabsf(QMAX - r.z1)), 0.f);
                    const float m1 = max3(q.s0 * fmaxf(fabsf(q.z0), fabsf(QMAX - q.z0)), q.s1 * fmaxf(fabsf(q.z1), fabsf(QMAX - q.z1)), 0.f);
                    top = max3(top, m, m1);
                    far |= max3(fabsf(r.z0), fabsf(r.z1), fmaxf(fabsf(q.z0), fabsf(q.z1))) > PR_NEAR;
                }
                if (s >= 2 && !(ok = bar_wait_warp(&sm.par_empty[role][buf], ((s >> 1) - 1) & 1, &sm.failed))) break;
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
                                r = find_slot(pos, n_pos, tok);
                                miss = r < 0;
                            }
                            sm.rank[role][buf][idx] = r;
                        }
                        const uint32_t m = __ballot_sync(0xffffffffu, miss);
                        if (x) dead1 = m;
                        else dead0 = m;
                    }
                    __syncwarp();
                    __half2 large = __float2half2_rn(0.f);
#pragma unroll 2
                    for (int y = lane >> 4; y < ns; y += 2) {                // half a warp a row
                        const int r = sm.rank[role][buf][y];
                        uint4 v = make_uint4(0u, 0u, 0u, 0u);
                        if (r >= 0 && in_bounds(r < p.cap, c.status)) v = *(const uint4 *)(rows + (size_t)r * D);
                        if (y < PR_ROWS_KEPT) sm.kept[role][buf][y][lane & 15] = v;
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
                    if (!keys && __any_sync(0xffffffffu, odd) && lane == 0) *(volatile uint8_t *)&sm.odd[round] = 1;
                }
                int e = fit_exponent(warp_top(top));
                if (keys && tok0 + PR_STEP > n_body && seq_len > n_body) e = min(e, 0);    // fp16 rows of the open group, as they are
                const float up = exp2i(e);
                StepHeader &hd = sm.hdr[s & (PR_HDRS - 1)];
                far = __any_sync(0xffffffffu, far);
                uint4 *tab = sm.tab[role][buf] + lane;
                uint2 *add = sm.add[role][buf] + lane;
#pragma unroll 1
                for (int n = 0; n < n_entries; n += 2) {
                    const int n1 = min(n + 1, n_entries - 1);                // an odd one out is written twice
                    const Pair r = pair(j, n, s), q = pair(j, n1, s);
                    table_entry<BITS>(r.s0, r.z0, r.s1, r.z1, up, (lane >> 2) & 1, far, tab + 32 * n, add + 32 * n);
                    table_entry<BITS>(q.s0, q.z0, q.s1, q.z1, up, (lane >> 2) & 1, far, tab + 32 * n1, add + 32 * n1);
                }
                if (lane == 0) {
                    uint4 *to = reinterpret_cast<uint4 *>(keys ? (void *)&hd.k_down : (void *)&hd.v_up);
                    to[0] = keys ? make_uint4(__float_as_uint(exp2i(-e)), __float_as_uint(up), dead0, dead1)
                                 : make_uint4(__float_as_uint(up), __float_as_uint((float)e), sink[0], sink[1]);
                    to[1] = keys ? make_uint4(sink[0], sink[1], far, split / KVSINK_TILE) : make_uint4(far, 0u, 0u, 0u);
                }
                __syncwarp();
                if (lane == 0) {
                    bar_arrive(&sm.par_full[role][buf]);
                    bar_arrive(&sm.hdr_full[s & (PR_HDRS - 1)]);        // for the softmax: both warps' halves of the header
                }
            }
        }
        if (!ok) {             // gave up: let the copies that were asked for arrive before the block goes
            int go = 0;
            for (int y = max(asked - 2, 0); y < asked; ++y) bar_wait_warp(&sm.raw_full[role][y & 1], (y >> 1) & 1, &go);
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
    const int64_t work = (int64_t)a.blocks * p.B * p.Hkv;
    const int64_t waves = (work + (int64_t)PR_GRID * PR_ROUNDS - 1) / ((int64_t)PR_GRID * PR_ROUNDS);
    const int64_t grid = work < PR_GRID ? work : waves * PR_GRID;
    if (launch_pdl(kern, dim3((unsigned)grid), dim3(PR_THREADS), smem, st, p, c, a) != cudaSuccess) return KVSINK_ERR_CUDA;
    return KVSINK_OK;
}

}  // namespace

// The kernel for many rows, or the eight-row blocks of the decode kernel, which are faster with few: a block here takes the same time however few of its
// rows there are (less with one row tile of 128 than with two), one block to an SM; those run four to an SM, each warp on a share of the cache, and slow one
// another down.  So the line is the number of them while this kernel does one round of blocks.
// Speed alone would draw it at 3 of them on an SM (2 bit, one row tile; 4 with two), 2 (3 bit), 2 and 3 (4 bit).  With 8192 tokens, us (rows x
// units, eight-row blocks on an SM, there and here):
//   2 bit: one tile   64 x 40,  3,  129 and 177;   96 x 40,  4,  192 and 179;   two tiles  512 x 8, 4,  196 and 252;   192 x 40, 7, 307 and 242
//   3 bit: one tile  128 x 16,  2,  188 and 192;   64 x 40,  3,  275 and 189;   two tiles  256 x 8, 2,  192 and 248;   384 x 8,  3, 284 and 253
//   4 bit: one tile  128 x 16,  2,  179 and 186;   96 x 40,  4,  280 and 186;   two tiles  384 x 8, 3,  186 and 249;   512 x 8,  4, 290 and 253
// There it lies at 3 bit.  At 2 and 4 bit the eight-row blocks sum the keys' products exactly, in integers, from factors of 30 bits; here keys carry 22 bits, as in
// the eight-row blocks of 3 bit, and the sums in TMEM are rounded downwards at each product.  So there this kernel has only what lies well beyond:
// from 1024 and 512 of those blocks a round on.  Relative error against 64 bits, there and here, for prompts between the lines: log-sum-exp 0.7e-7 and
// 1.8e-7 (3 bit 2e-5 and 1.9e-7); outputs 4e-5 and 1e-6 (3 bit 1.5e-4 and 1e-6) with values about zero; with values 40 to 500 from zero and ranges a
// fiftieth as wide 1e-6 and 8e-6 behind 1000 tokens, 3e-6 and 3e-5 behind 4000, at every code width.
bool prompt_takes(const Params &p, int T)
{
    if (p.D != 128) return false;
    const int64_t rows = (int64_t)T * p.rep, units = (int64_t)p.B * p.Hkv;
    const int64_t blocks = (rows + PR_ROWS - 1) / PR_ROWS * units, waves = (blocks + 147) / 148, small = (rows + 7) / 8 * units;
    return rows < (1 << 30) && blocks < (1 << 30) && (p.bits == 3 ? small > waves * 2 * 148 : small >= waves * (p.bits == 2 ? 1024 : 512));
}

int launch_prompt(const Params &p, const kvsink_cache &c, const __half *q, int T, int q_pos0, int64_t sb, int64_t sh, int64_t stt, float *out,
                  float *lse, cudaStream_t st)
{
    int shift = 30;
    while ((1ll << (shift - 30)) < p.rep) ++shift;
    const uint32_t mul = (uint32_t)(((1ull << shift) + p.rep - 1) / p.rep);
    const PromptArgs a = {q, out, lse, sb, sh, stt, T, q_pos0, (int)(((int64_t)T * p.rep + PR_ROWS - 1) / PR_ROWS), mul, (uint32_t)shift};
    if (p.bits == 2) return launch<2>(p, c, a, st);
    if (p.bits == 3) return launch<3>(p, c, a, st);
    return launch<4>(p, c, a, st);
}

}  // namespace kvsink
