// Single-token decode attention, one query head per KV head (head size 128): keys and values on the integer tensor path.
//
// What bounds it: issue slots and latency (the stream is two to four bits an element).  So (i) both sides multiply stored bytes: a
// word masked in place is the u8 A fragment of one m16n8k32 (a 2-bit word 0x03.., 0x0c.., 0x30.., 0xc0..: rows g, rows g + 8 (x4),
// the upper contraction slots (x16), both; a 4-bit word 0x0f.. and 0xf0.., two words to a fragment; 3 bit: low and high bits are first
// put together in nibbles): 16 masks and four multiplies a tile and side where fp16 operands of the values took 36 and eight.  (ii) Of
// 32 tokens every lane owns one, 8 t + g, for everything between the two products: the softmax, the parameters, the weight in
// fixed point.  With the fp16 values all lanes of a quad did the work of the quad's two tokens.
// Append and decode, us a pass, fp16 values with a warp's work on eight tokens at a time before, this kernel now: 8 x 32 units of 4096
// tokens, 2 bit, 31.0 -> 24.7 (decode alone 26.8 -> 18.1); static parameters, 3821 tokens, 27.6 -> 23.5; 16 x 32 of 8101, 3 bit, 135 -> 111;
// 64 x 32 of 8192, 4 bit, 481 -> 441; 32-token groups, 2 bit, 53.7 -> 36.8 (and 6 % less since the ring is filled by all lanes).  Error against 64 bits of these 5e-5 -> 1e-6 (the fp16
// products' accumulation truncates; 8192 tokens a warp, N(0,1), 2e-3 -> 1e-5).  Four blocks an SM; five (96 registers, a few spilled)
// are slower except at 4 bit: 26.4 against 23.9, 422 / 411.
//
// Keys: the four signed bytes of the factor q * scale in columns 0-3, and again in 4-7, so that lanes t < 2 take the first tile's sums
// and lanes t >= 2 the second's; one exchange inside a lane pair leaves each lane with its own token's sum.
// Values: a stored byte pair belongs to one channel and two tokens, and the two byte pairs of a 2- or 3-bit word (the two words of a
// 4-bit fragment) to two 16-channel matrices.  The weights' four signed bytes therefore stand in eight columns, 2 l + matrix, with
// zeros where the other matrix' codes are: lane t finds byte t of both matrices' sums in its accumulators.
//   weight = rint(2^(s - R) * scale * 2^ev), below 2^31, ev per value channel group; R and ev move only when a weight would not fit (one
//   vote a step).  The sums of a byte are exact in int32; when R or ev moves they are added to binary32 ones and start from zero.  A new
//   unit puts the largest weight into [2^28, 2^29); the upper contraction slots' tokens of 2 and 3 bit carry a weight divided by 16.  So a weight is held to
//   2^-29 of the largest, there to 2^-25; smaller ones keep their sum by a dither (next_dither).
#pragma once
#include "decode_kernel.cuh"

namespace kvsink {

__device__ __forceinline__ void imma16832(int (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// What is added to a lane's weights before they are rounded to whole units: another value in [-1/2, 1/2) for every lane and step, evenly spread
// (the golden section's multiples), so that many weights below half a unit keep their sum.  Without it a long tail of them is rounded away
// from the outputs, while its weight stays in the softmax's sum: 8192 tokens a warp 18 nats below one of them, 2 bit, error against 64 bits
// 4e-5, with it 5e-6.  It costs three instructions a step; carrying on what each weight's rounding leaves over costs three a weight, 1 to 2 %
// of the time.
// A weight of 0 stays 0.
__device__ __forceinline__ float next_dither(float d)
{
    d += 0.381966f;
    return d >= 0.5f ? d - 1.f : d;
}

// The two nibble words of a 3-bit word: rows g (me) and rows g + 8 (mo), three bits at 4 j.
__device__ __forceinline__ void nibbles3(const uint32_t *w, int i, uint32_t *me, uint32_t *mo)
{
    const uint32_t x = w[i], hh = (i & 1) ? (w[4 + i / 2] << 2) : w[4 + i / 2];
    *me = (x & 0x33333333u) | (hh & 0xccccccccu);
    *mo = ((x >> 2) & 0x33333333u) | ((hh >> 1) & 0xccccccccu);
}

// A fragment i (channels 32 i ... 32 i + 31) of a tile's words.
template <int BITS>
__device__ __forceinline__ void byte_frag(const uint32_t (&w)[2 * BITS], int i, uint32_t (&a)[4])
{
    if constexpr (BITS == 2) {
        a[0] = w[i] & 0x03030303u; a[1] = w[i] & 0x0c0c0c0cu; a[2] = w[i] & 0x30303030u; a[3] = w[i] & 0xc0c0c0c0u;
    } else if constexpr (BITS == 4) {
        const uint32_t x = w[2 * i], y = w[2 * i + 1];
        a[0] = x & 0x0f0f0f0fu; a[1] = x & 0xf0f0f0f0u; a[2] = y & 0x0f0f0f0fu; a[3] = y & 0xf0f0f0f0u;
    } else {
        uint32_t me, mo;
        nibbles3(w, i, &me, &mo);
        a[0] = me & 0x07070707u; a[1] = mo & 0x07070707u; a[2] = me & 0x70707070u; a[3] = mo & 0x70707070u;
    }
}

template <int BITS, int NGv, int CT, int PM>
__global__ void __launch_bounds__(DEC_THREADS, 4)
decode_one_kernel(Params p, kvsink_cache c, kvsink_static_params sp, const __half *__restrict__ q, float *__restrict__ out, float *__restrict__ lse,
                  float *__restrict__ part_ws, int nsplit, int groups_per_split, int seq_len, int cluster_merge)
{
    constexpr int D = 128, W = 2 * BITS, TILE_WORDS = 32 * W, CPL = D / 32;
    using Plan = DecodePlan<BITS, D, NGv, CT, 1, PM == 2>;
    constexpr int NSLOT = Plan::NSLOT, SLOT_BYTES = Plan::SLOT_BYTES, KV_BYTES = Plan::KV_BYTES, SZ_BYTES = Plan::SZ_BYTES, PS = Plan::PS;
    constexpr int TP = CT >= 2 ? 2 : 1, NP = CT / TP;                // tiles of a pair, pairs of a chunk (= softmax step)
    constexpr bool CAL = PM == 1, KT = PM == 2, FLAT = PM != 0;    // static parameters / per-token keys / either: no token groups
    constexpr int NGK = KT ? NGv : 1;                              // separate dot products per token on the key side
    static_assert(CT == 1 || CT == 2 || CT == 4, "whole pairs of tiles");
    static_assert(!KT || NGv <= 2, "per-token keys: one or two channel groups");
    constexpr float LOG2E = 1.4426950408889634f;
    constexpr float ROWF = BITS == 2 ? 0.25f : (BITS == 4 ? 0.0625f : 1.f);      // rows g + 8 of a fragment: place of their field
    constexpr float UPF = BITS == 4 ? 1.f : 0.0625f;                             // upper contraction slots: place of their field
    constexpr float WEIGHT_LIMIT = 2130706432.f;                                 // 0x7f000000: its carries still fit a signed byte

    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), g = lane >> 2, t = lane & 3;
    const bool odd = t & 1, second = TP == 2 && t >= 2;
    const int own = 8 * t + g;                                       // this lane's token of a pair
    const int split = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int64_t unit = (int64_t)b * p.Hkv + h;
    const int G = FLAT ? CT * KVSINK_TILE : p.G;                     // without token groups one ring chunk plays their part
    const int n = seq_len, n_groups = FLAT ? (n + G - 1) / G : n / G, n_body = FLAT ? n : n_groups * G;
    const int TPG = G / KVSINK_TILE, CPG = TPG / CT;                 // tiles and ring chunks per key group
    const uint32_t *bm = c.sink_bitmask + (size_t)b * p.mask_words;
    const float qscale = LOG2E * rsqrtf((float)D);

    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *qs = (float *)smem_raw;                                   // [D] q * log2e/sqrt(D)
    __half *q16 = (__half *)(qs + D);                                // [D] q as given
    uint64_t *bars = (uint64_t *)(smem_raw + Plan::Q_BYTES + DEC_WARPS * Plan::B_BYTES);   // [warps]: of the parameter slot
    unsigned char *ring_all = smem_raw + Plan::FIXED;                // [warps][WARP_RING]; later reused for the partials
    float *part = (float *)ring_all;                                 // [2*warps][D+2]

    const uint32_t pbar = smem_addr(bars + warp);
    if (lane == 0) {
        mbar_init(pbar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // everything above overlaps the tail of the kernel before this one; nothing it may have written is read before this point
    pdl_wait();
    pdl_release();
    // Sink rows are shared out over all warps of all splits and handled after the stream; the first one of this warp is fetched now
    const int sink_n = min(c.sink_count[b], p.cap);
    const int sink_worker = split * DEC_WARPS + warp, sink_workers = nsplit * DEC_WARPS;
    int sink_pos_next = -1;
    uint32_t sink_k_next[CPL / 2], sink_v_next[CPL / 2];
    auto fetch_sink = [&](int j) {
        sink_pos_next = -1;
#pragma unroll
        for (int e = 0; e < CPL / 2; ++e) sink_k_next[e] = sink_v_next[e] = 0u;
        if (j < sink_n) {
            sink_pos_next = c.sink_pos[(size_t)b * p.cap + j];
            const uint32_t *kr = (const uint32_t *)((const __half *)c.sink_k + ((size_t)unit * p.cap + j) * D + lane * CPL);
            const uint32_t *vr = (const uint32_t *)((const __half *)c.sink_v + ((size_t)unit * p.cap + j) * D + lane * CPL);
#pragma unroll
            for (int e = 0; e < CPL / 2; ++e) { sink_k_next[e] = kr[e]; sink_v_next[e] = vr[e]; }
        }
    };
    fetch_sink(sink_worker);

    unsigned char *Bs = smem_raw + Plan::Q_BYTES + (size_t)warp * Plan::B_BYTES;             // key operand of the group, 512 bytes
    const uint8_t *kc_base = c.k_codes + (size_t)unit * p.max_seq * p.row_bytes;
    const uint8_t *vc_base = c.v_codes + (size_t)unit * p.max_seq * p.row_bytes;
    const float *vs_base = c.v_scale + (size_t)unit * p.max_seq * NGv;
    const float *vz_base = c.v_zero + (size_t)unit * p.max_seq * NGv;
    const float *ktok_s_base = c.k_scale + (size_t)unit * p.max_seq * NGv;    // per-token keys: [unit][max_seq][NGv]
    const float *ktok_z_base = c.k_zero + (size_t)unit * p.max_seq * NGv;
    const float *ks_base = c.k_scale + (size_t)unit * (p.max_seq / G) * D;
    const float *kz_base = c.k_zero + (size_t)unit * (p.max_seq / G) * D;

    // ---------------- running state ----------------
    float R = M_INIT, l = 0.f;            // reference of the weights, and this lane's part of their sum
    float bv[NGv];                        // this lane's part of the sum of weight * scale * zero per value channel group
    int O[4][4];                          // [fragment][rows g: matrix 0, 1 | rows g + 8: matrix 0, 1], byte t of the sums, in units of 2^-ev
    float Of[4][4];                       // the part of them from before the last move of R or ev
    const float up = (BITS != 4 && odd) ? 0.0625f : 1.f;             // this lane's token stands in the upper contraction slots
    const float w_limit = WEIGHT_LIMIT * up;
    float dither = (lane + 0.5f) * (1.f / 32) - 0.5f;
    float evl[NGv];                       // 2^ev, a value channel group's own (groups may lie far apart in size), of this lane's slots
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int x = 0; x < 4; ++x) { O[i][x] = 0; Of[i][x] = 0.f; }
#pragma unroll
    for (int j = 0; j < NGv; ++j) { bv[j] = 0.f; evl[j] = pow2i(60) * up; }

    auto settle = [&](int j, float f) {
#pragma unroll
        for (int i = 4 / NGv * j; i < 4 / NGv * (j + 1); ++i)
#pragma unroll
            for (int x = 0; x < 4; ++x) { Of[i][x] = (Of[i][x] + (float)O[i][x]) * f; O[i][x] = 0; }
    };
    // Weights of N tokens of this lane: pw = 2^(s - R) and x = pw * scale in units of 2^-ev (plus the dither), after moving R and ev if one of the warp's
    // does not fit.  A new unit puts the largest weight into [2^28, 2^29): the next four to eight times as large still fit.
    auto weights = [&](const auto &s, const auto &sv, auto &pw, auto &x) {
        constexpr int N = sizeof(pw) / sizeof(pw[0]);
        dither = next_dither(dither);
        bool moves = false;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const float d = s[k] - R;
            pw[k] = ex2(d);
            moves |= d > 20.f;
#pragma unroll
            for (int j = 0; j < NGv; ++j) { x[k][j] = fmaf(pw[k], sv[k][j] * evl[j], dither); moves |= fabsf(x[k][j]) >= w_limit; }
        }
        if (!__any_sync(0xffffffffu, moves)) return;
        float top = R;
#pragma unroll
        for (int k = 0; k < N; ++k) top = fmaxf(top, s[k]);
        top = warp_max(top);
        const float corr = ex2(R - top);
        const int rise = max(0, -floor_log2(corr) - 1);
        const bool first = R == M_INIT;
        R = top;
        l *= corr;
#pragma unroll
        for (int k = 0; k < N; ++k) pw[k] = ex2(s[k] - R);
#pragma unroll
        for (int j = 0; j < NGv; ++j) {
            float wm = 0.f;
#pragma unroll
            for (int k = 0; k < N; ++k) wm = fmaxf(wm, pw[k] * fabsf(sv[k][j]));
            // not finer than the weights so far allow: they shrink by corr
            const int ev = floor_log2(evl[j]) - floor_log2(up), to = max(min(28 - floor_log2(warp_max(wm)), first ? 60 : min(60, ev + rise)), -60);
            settle(j, corr * pow2i(to - ev));
            evl[j] = pow2i(to) * up;
            bv[j] *= corr;
#pragma unroll
            for (int k = 0; k < N; ++k) x[k][j] = fmaf(pw[k], sv[k][j] * evl[j], dither);
        }
    };
    // The value products of a pair: this lane's token's weight and parameters, the two tiles' words.
    const int col_src = (g >> 2) * 4 + t;                            // lane that holds the byte pair of column g's byte, of token quarter 0
    const int col_byte = (g >> 1) & 1;                               // which byte of it
    const uint32_t col_sel = BITS == 4 ? (uint32_t)(col_byte | (4 + col_byte) << 4 | (2 + col_byte) << 8 | (6 + col_byte) << 12)
                             : (g & 1) ? (uint32_t)(0x4 | col_byte << 4 | 0x400 | (2 + col_byte) << 12)
                                       : (uint32_t)(col_byte | 0x40 | (2 + col_byte) << 8 | 0x4000);
    auto pair_values = [&](float pw, const float (&x)[NGv], const float (&sv)[NGv], const float (&zv)[NGv], auto words) {
        l += pw;
        uint32_t mv[NGv];
#pragma unroll
        for (int j = 0; j < NGv; ++j) {
            bv[j] = fmaf(pw, sv[j] * zv[j], bv[j]);
            // signed bytes; the transpose of the byte pairs: lane (2 t' + e, t) gets byte pair e of the weights of tokens 8 t' + 2 t, + 1
            mv[j] = movm_trans(((uint32_t)__float2int_rn(x[j]) + 0x00808080u) ^ 0x00808080u);
        }
#pragma unroll
        for (int k = 0; k < TP; ++k) {
            uint32_t vw[W];
            words(k, vw);
            uint32_t b0[NGv], b1[NGv];
#pragma unroll
            for (int j = 0; j < NGv; ++j) {
                const uint32_t lo = __shfl_sync(0xffffffffu, mv[j], col_src + 16 * k), hi = __shfl_sync(0xffffffffu, mv[j], col_src + 16 * k + 8);
                if constexpr (BITS == 4) {      // all four bytes of a word are tokens of one matrix: 2t, 2t + 8, 2t + 1, 2t + 9
                    const uint32_t v = __byte_perm(lo, hi, col_sel);
                    b0[j] = (g & 1) ? 0u : v;
                    b1[j] = (g & 1) ? v : 0u;
                } else {
                    b0[j] = __byte_perm(lo, 0u, col_sel);
                    b1[j] = __byte_perm(hi, 0u, col_sel);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint32_t a[4];
                byte_frag<BITS>(vw, i, a);
                imma16832(O[i], a, b0[i * NGv / 4], b1[i * NGv / 4]);
            }
        }
    };

    // ---- the warps take contiguous, nearly equal ranges of the split's groups; a warp's chunks (CT tiles each) are consecutive in
    //      memory and arrive through a ring of NSLOT slots filled NSLOT - 1 chunks ahead; the key parameters
    //      of a group arrive one group ahead through one more slot ----
    const int g_begin = split * groups_per_split, g_end = min(n_groups, g_begin + groups_per_split);
    const int g_cnt = max(g_end - g_begin, 0);
    const int w_begin = g_begin + (g_cnt * warp) / DEC_WARPS, w_end = g_begin + (g_cnt * (warp + 1)) / DEC_WARPS;
    const int my_groups = w_end - w_begin;
    unsigned char *ring = ring_all + (size_t)warp * Plan::WARP_RING;
    const float *kp_ring = (const float *)(ring + NSLOT * SLOT_BYTES);      // [scale D | zero D] of the next group to prepare
    const int n_chunks = my_groups * CPG;
    int iss = 0;                                                     // chunks issued so far
    uint32_t iss_kv = (uint32_t)w_begin * TPG * Plan::TILE_BYTES;    // byte offset of the next chunk in the code arrays
    uint32_t iss_sz = (uint32_t)w_begin * TPG * 16 * NGv * 4;        // and in the parameter arrays
    const uint32_t ring_s = smem_addr(ring), kp_s = smem_addr(kp_ring);
    auto issue_chunk = [&]() {
        const int slot = iss & (NSLOT - 1);
        // debug builds: the chunk must lie inside the unit's code arrays
        const bool inside = in_bounds((size_t)iss_kv + KV_BYTES <= (size_t)p.max_seq * p.row_bytes, c.status);
        const uint32_t dst = ring_s + slot * SLOT_BYTES;
        if (inside) {
            copy_words<KV_BYTES>(dst, kc_base + iss_kv, lane);
            copy_words<KV_BYTES>(dst + KV_BYTES, vc_base + iss_kv, lane);
            if constexpr (!CAL) copy_params<SZ_BYTES, KT ? 4 : 2>(dst + 2 * KV_BYTES, vs_base, vz_base, ktok_s_base, ktok_z_base, iss_sz, lane);
        }
        ++iss;
        iss_kv += KV_BYTES;
        iss_sz += SZ_BYTES;
    };
    // The caller has put the slot's last values through an operation of the whole warp: a bulk copy is not kept behind loads that are queued
    auto issue_params = [&](int gi) {
        if (lane == 0) {
            mbar_expect_tx(pbar, Plan::KP_BYTES);
            bulk_g2s(kp_s, ks_base + (size_t)(w_begin + gi) * D, D * 4, pbar);
            bulk_g2s(kp_s + D * 4, kz_base + (size_t)(w_begin + gi) * D, D * 4, pbar);
        }
    };
    auto wait_bar = [&](uint32_t bar, unsigned parity) {
        int polls = 0;
        bool ok = true;
        while (!mbar_try_wait(bar, parity)) {
            if (++polls > DEC_WAIT_LIMIT) { ok = false; break; }
        }
        return __all_sync(0xffffffffu, ok);
    };
    // sink bits of the chunk that starts at tile T: one 32-bit word covers two tiles
    auto load_mask_words = [&](int T) {
        uint2 w;
        w.x = __ldg(bm + (T >> 1));
        w.y = NP == 2 ? __ldg(bm + (T >> 1) + 1) : 0u;
        return w;
    };
    static_assert(DEC_THREADS == D, "a query value a thread");
    // The loads that come next are issued ahead of the first copies of the ring and used behind them: the copies of 16 warps keep the load unit busy,
    // and what is queued behind them waits (with the query loaded behind them, us, before and now: 8 x 32 units of 4096 tokens, 2 bit
    // 18.6 and 18.1, 3 bit, 64-token groups 32.5 and 31.6, 4 bit, 128-token groups 28.5 and 27.6)
    float cal_sv[NGv], cal_zv[NGv];       // static value parameters of the KV head
#pragma unroll
    for (int j = 0; j < NGv; ++j) { cal_sv[j] = CAL ? sp.v_scale[h * NGv + j] : 0.f; cal_zv[j] = CAL ? sp.v_zero[h * NGv + j] : 0.f; }
    const __half q_v = q[((size_t)b * p.Hq + h) * D + tid];
    uint2 mword_next = my_groups > 0 ? load_mask_words(w_begin * TPG) : make_uint2(0u, 0u);
    if (my_groups > 0) {
        if (!FLAT) issue_params(0);
        for (int i = 0; i < NSLOT - 1; ++i) {      // a group of copies a chunk, empty ones behind the last
            if (iss < n_chunks) issue_chunk();
            copies_commit();
        }
    }
    // the first copies are in flight: now the query tables
    q16[tid] = q_v;
    qs[tid] = __half2float(q_v) * qscale;
    __syncthreads();

    // Key operand: lane l prepares the bytes of one group of four contraction slots, (fragment l/8, lower or upper slots (l/4)%2, slots
    // 4(l%4) ... +3); these are its four channels and their query values.
    int i8_ch[4];
    float i8_q[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int mi = lane >> 3, c2 = (lane >> 2) & 1, tq = lane & 3;
        i8_ch[e] = BITS != 4 ? 16 * (2 * mi + (e & 1)) + 8 * c2 + 2 * tq + (e >> 1) : 16 * (2 * mi + c2) + 8 * (e & 1) + 2 * tq + (e >> 1);
        i8_q[e] = qs[i8_ch[e]];
    }

    bool stream_ok = true;
    int ci = 0;                                                      // running chunk index of this warp

    // ---- tokens of the open group: keys from the fp16 tail (last split only), one tile at a time; they come first, while the warp's
    //      first chunks are on their way (the order of the softmax steps does not matter) ----
    if (!FLAT && split == nsplit - 1) {
        const __half *tail = (const __half *)c.k_tail + (size_t)unit * G * D;
        const int T_begin = n_body / KVSINK_TILE, T_end = (n + KVSINK_TILE - 1) / KVSINK_TILE;
        for (int T = T_begin + warp; T < T_end; T += DEC_WARPS) {
            const int tok0 = T * KVSINK_TILE + g, tok1 = tok0 + 8;
            const bool in0 = tok0 < n, in1 = tok1 < n;
            const __half *r0 = tail + (size_t)(tok0 % G) * D, *r1 = tail + (size_t)(tok1 % G) * D;
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int m = 0; m < D / 16; ++m) {
                uint32_t a[4];
                a[0] = in0 ? *(const uint32_t *)(r0 + 16 * m + 2 * t) : 0u;
                a[1] = in1 ? *(const uint32_t *)(r1 + 16 * m + 2 * t) : 0u;
                a[2] = in0 ? *(const uint32_t *)(r0 + 16 * m + 2 * t + 8) : 0u;
                a[3] = in1 ? *(const uint32_t *)(r1 + 16 * m + 2 * t + 8) : 0u;
                // the query in every column: each lane finds its own token's score
                mma16816(acc, a, *(const uint32_t *)(q16 + 16 * m + 2 * t), *(const uint32_t *)(q16 + 16 * m + 2 * t + 8));
            }
            const int tok = T * KVSINK_TILE + own;                   // lanes t < 2 own the tile's 16 tokens
            const bool valid = t < 2 && tok < n && !mask_bit(bm, tok < n ? tok : 0);
            float s[1], sv[1][NGv], zv[1][NGv], pw[1], x[1][NGv];
            s[0] = valid ? (odd ? acc[2] : acc[0]) * qscale : -INFINITY;
#pragma unroll
            for (int j = 0; j < NGv; ++j) {   // tokens beyond the sequence have no parameters yet
                sv[0][j] = valid ? __ldg(vs_base + (size_t)tok * NGv + j) : 0.f;
                zv[0][j] = valid ? __ldg(vz_base + (size_t)tok * NGv + j) : 0.f;
            }
            weights(s, sv, pw, x);
            pair_values(pw[0], x[0], sv[0], zv[0], [&](int k, uint32_t (&w)[W]) {
                if (k == 0) load_tile<BITS, D>((const uint32_t *)(vc_base + (size_t)T * p.tile_bytes), lane, w);
                else {
#pragma unroll
                    for (int i = 0; i < W; ++i) w[i] = 0u;           // the pair's second tile is not there
                }
            });
        }
    }

    // state of the current key group (without token groups: set up on the first trip)
    float bias0 = 0.f, bias1 = 0.f, ck = 0.f, cr = 0.f;
    uint32_t bk[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) bk[i][0] = bk[i][1] = 0u;
#pragma unroll 1
    for (int gi = 0; gi < my_groups && stream_ok; ++gi) {
        const int grp = w_begin + gi;
        if (!FLAT || gi == 0) {
            float scv[CPL], zev[CPL];
            if constexpr (CAL) {
#pragma unroll
                for (int e = 0; e < CPL; ++e) { scv[e] = sp.k_scale[h * D + i8_ch[e]]; zev[e] = sp.k_zero[h * D + i8_ch[e]]; }
            } else if constexpr (KT) {
                // the operand is the query itself; with zero = 1 the "zero-point term" below is the sum of the query
#pragma unroll
                for (int e = 0; e < CPL; ++e) { scv[e] = 1.f; zev[e] = 1.f; }
            } else {
                if (!wait_bar(pbar, (unsigned)gi & 1u)) { stream_ok = false; break; }
#pragma unroll
                for (int e = 0; e < CPL; ++e) { scv[e] = kp_ring[i8_ch[e]]; zev[e] = kp_ring[D + i8_ch[e]]; }
            }
            // F = rint(q * scale * 2^sh) with the largest |F| in [2^29, 2^30), cut into four signed bytes (radix 256): every factor is
            // kept to 2^-30 of the group's largest one (2^-26 where it is pre-divided for the upper contraction slots).  Adding
            // 0x808080 propagates the carries of the signed digits and the exclusive-or removes the offset again.
            float v[4], amax = 0.f, bsum = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                v[e] = i8_q[e] * scv[e];
                amax = fmaxf(amax, fabsf(v[e]));
                // the zero-point term takes the unrounded factor: the limbs' rounding then meets the codes (at most
                // qmax) only, not code - zero, which is large for a channel far from zero with a narrow range
                bsum = fmaf(v[e], zev[e], bsum);
            }
            amax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(amax)));   // non-negative floats order as integers
            int sh = 29 - floor_log2(amax);
            sh = sh > 60 ? 60 : (sh < -60 ? -60 : sh);
            const float pre = pow2i(sh) * ((lane & 4) ? UPF : 1.f);
            uint32_t d[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) d[e] = ((uint32_t)__float2int_rn(v[e] * pre) + 0x00808080u) ^ 0x00808080u;
            // byte transpose: word j = byte j of the four channels, in contraction-slot order
            const uint32_t t0 = __byte_perm(d[0], d[1], 0x5140), t1 = __byte_perm(d[0], d[1], 0x7362);
            const uint32_t t2 = __byte_perm(d[2], d[3], 0x5140), t3 = __byte_perm(d[2], d[3], 0x7362);
            // table [fragment][lower / upper slots][byte, most significant first][t][slot]: this lane owns one 4-byte slot group
            uint32_t *tab = reinterpret_cast<uint32_t *>(Bs) + (lane >> 2) * 16 + (lane & 3);
            tab[0] = __byte_perm(t1, t3, 0x7632);
            tab[4] = __byte_perm(t1, t3, 0x5410);
            tab[8] = __byte_perm(t0, t2, 0x7632);
            tab[12] = __byte_perm(t0, t2, 0x5410);
            if constexpr (KT && NGv == 2) {
                // two channel groups: the query's sum over each (lanes 0-15 hold channels 0-63)
                bias0 = warp_sum(lane < 16 ? bsum : 0.f); bias1 = warp_sum(lane < 16 ? 0.f : bsum);
            } else {
                bias0 = warp_sum(bsum);
            }
            // a lane's sum is keep * ck + received * cr: even lanes keep the upper bytes' half of rows g, odd lanes the lower bytes'
            // half of rows g + 8
            const float ks = odd ? pow2i(-sh) * ROWF : pow2i(-sh);
            ck = odd ? ks : ks * 65536.f;
            cr = odd ? ks * 65536.f : ks;
            __syncwarp();
            // every lane's parameters have gone into sums over the warp: the slot can take the next group's while this one streams
            if (!FLAT && gi + 1 < my_groups) issue_params(gi + 1);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c2 = 0; c2 < 2; ++c2) bk[i][c2] = reinterpret_cast<const uint32_t *>(Bs)[(i * 2 + c2) * 16 + (g & 3) * 4 + t];
        }

#pragma unroll 1
        for (int cj = 0; cj < CPG; ++cj, ++ci) {
            const int slot = ci & (NSLOT - 1);
            // refill the slot freed by the previous chunk, then wait for this chunk's bytes
            __syncwarp();
            if (iss < n_chunks) issue_chunk();
            copies_commit();
            copies_wait<NSLOT - 1>();
            const uint2 mwords = mword_next;
            if (ci + 1 < n_chunks) mword_next = load_mask_words(grp * TPG + (cj + 1) * CT);   // the warp's chunks are consecutive
            const uint32_t *kt = (const uint32_t *)(ring + slot * SLOT_BYTES), *vt = kt + KV_BYTES / 4;
            const float *ssv = (const float *)(vt + KV_BYTES / 4) + own * NGv, *szv = ssv + SZ_BYTES / 4;
            const float *kts = szv + SZ_BYTES / 4, *ktz = kts + SZ_BYTES / 4;          // per-token keys
            const int T0 = grp * TPG + cj * CT;

            // ---- scores: each lane ends with those of its own tokens ----
            float s[NP];
#pragma unroll
            for (int pr = 0; pr < NP; ++pr) {
                int ia[TP][NGK][4];
#pragma unroll
                for (int k = 0; k < TP; ++k) {
#pragma unroll
                    for (int j = 0; j < NGK; ++j)
#pragma unroll
                        for (int x = 0; x < 4; ++x) ia[k][j][x] = 0;
                    uint32_t kw[W];
                    load_tile_shared<BITS, D>(kt + (pr * TP + k) * TILE_WORDS, lane, kw);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        uint32_t a[4];
                        byte_frag<BITS>(kw, i, a);
                        imma16832(ia[k][NGK == 2 ? (i >> 1) : 0], a, bk[i][0], bk[i][1]);
                    }
                }
                float r = 0.f;
#pragma unroll
                for (int j = 0; j < NGK; ++j) {
                    // column sums are below 2^22, two of them joined below 2^31
                    int (&last)[4] = ia[TP - 1][j];
                    const int x0 = (second ? last[0] : ia[0][j][0]) * 256 + (second ? last[1] : ia[0][j][1]);
                    const int x1 = (second ? last[2] : ia[0][j][2]) * 256 + (second ? last[3] : ia[0][j][3]);
                    const float keep = (float)(odd ? x1 : x0), got = (float)__shfl_xor_sync(0xffffffffu, odd ? x0 : x1, 1);
                    if constexpr (KT) {
                        // per-token keys: scale * (dot product - zero * sum of the query), per channel group
                        const int at = pr * 32 * NGv + j;
                        r = fmaf(kts[at], fmaf(-ktz[at], j == 0 ? bias0 : bias1, fmaf(keep, ck, got * cr)), r);
                    } else {
                        r = fmaf(keep, ck, fmaf(got, cr, -bias0));
                    }
                }
                s[pr] = r;
            }
            if (mwords.x | mwords.y) {   // sink tokens are not part of the packed stream
#pragma unroll
                for (int pr = 0; pr < NP; ++pr) {
                    const uint32_t w = TP == 1 && (T0 & 1) ? mwords.x >> 16 : (pr == 0 ? mwords.x : mwords.y);
                    if ((w >> own) & 1u) s[pr] = -INFINITY;
                }
            }
            if (TP == 1 && t >= 2) s[0] = -INFINITY;                 // no second tile
            if constexpr (FLAT) {
                if ((T0 + CT) * KVSINK_TILE > n) {   // the last tiles reach beyond the sequence: those tokens do not exist
#pragma unroll
                    for (int pr = 0; pr < NP; ++pr)
                        if (T0 * KVSINK_TILE + pr * 32 + own >= n) s[pr] = -INFINITY;
                }
            }
            // ---- one softmax step for the whole chunk, then its value products ----
            float sv[NP][NGv], zv[NP][NGv], pw[NP], x[NP][NGv];
#pragma unroll
            for (int pr = 0; pr < NP; ++pr)
#pragma unroll
                for (int j = 0; j < NGv; ++j) {
                    sv[pr][j] = CAL ? cal_sv[j] : (TP == 1 && t >= 2 ? 0.f : ssv[pr * 32 * NGv + j]);
                    zv[pr][j] = CAL ? cal_zv[j] : (TP == 1 && t >= 2 ? 0.f : szv[pr * 32 * NGv + j]);
                    if constexpr (KT) {   // tokens beyond the sequence: whatever the arrays hold there must not reach the sums
                        if (T0 * KVSINK_TILE + pr * 32 + own >= n) sv[pr][j] = zv[pr][j] = 0.f;
                    }
                }
            weights(s, sv, pw, x);
#pragma unroll
            for (int pr = 0; pr < NP; ++pr)
                pair_values(pw[pr], x[pr], sv[pr], zv[pr],
                            [&](int k, uint32_t (&w)[W]) { load_tile_shared<BITS, D>(vt + (pr * TP + k) * TILE_WORDS, lane, w); });
            // a tile adds less than 2^19 to a sum of bytes
            if ((ci & (2048 / CT - 1)) == 2048 / CT - 1) {
#pragma unroll
                for (int j = 0; j < NGv; ++j) settle(j, 1.f);
            }
        }
    }
    copies_wait<0>();      // the ring's space is used again
    if (!stream_ok && lane == 0) atomicOr(c.status, KVSINK_STATUS_TIMEOUT);

    // ---- this warp's partial record of the packed stream ----
    l = warp_sum(l);
#pragma unroll
    for (int j = 0; j < NGv; ++j) bv[j] = warp_sum(bv[j]);
    __syncthreads();   // every warp has drained its ring: the space now holds the block's partials
    float *my_part = part + (size_t)(2 * warp) * PS;
    {
        const float unit_t = pow2i(8 * t);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                float o = ((float)O[i][x] + Of[i][x]) * unit_t;      // this lane's byte; the quad's four make the sum
                o += __shfl_xor_sync(0xffffffffu, o, 1);
                o += __shfl_xor_sync(0xffffffffu, o, 2);
                if (t == x) my_part[16 * (2 * i + (x & 1)) + 8 * (x >> 1) + g] = o * (pow2i(floor_log2(up) - floor_log2(evl[i * NGv / 4])) * (x >= 2 ? ROWF : 1.f)) - bv[i * NGv / 4];
            }
        if (lane == 0) { my_part[D] = R; my_part[D + 1] = l; }
    }

    // ---------------- sink rows (fp16 side buffer), plain fp32 arithmetic ----------------
    {
        float ms = M_INIT, ls = 0.f, os[CPL];
#pragma unroll
        for (int e = 0; e < CPL; ++e) os[e] = 0.f;
        for (int j = sink_worker; j < sink_n; j += sink_workers) {
            const int pos = sink_pos_next;
            float kf[CPL], vf[CPL];
#pragma unroll
            for (int e = 0; e < CPL / 2; ++e) {
                const float2 k2 = __half22float2(*reinterpret_cast<const __half2 *>(&sink_k_next[e]));
                const float2 v2 = __half22float2(*reinterpret_cast<const __half2 *>(&sink_v_next[e]));
                kf[2 * e] = k2.x; kf[2 * e + 1] = k2.y; vf[2 * e] = v2.x; vf[2 * e + 1] = v2.y;
            }
            fetch_sink(j + sink_workers);   // the next row streams in while this one is used
            if (pos < 0 || pos >= n) continue;
            float dot = 0.f;
#pragma unroll
            for (int e = 0; e < CPL; ++e) dot += qs[lane * CPL + e] * kf[e];
            const float sc = warp_sum(dot), mnew = fmaxf(ms, sc), corr = ex2(ms - mnew), pp = ex2(sc - mnew);
            ls = ls * corr + pp;
#pragma unroll
            for (int e = 0; e < CPL; ++e) os[e] = os[e] * corr + pp * vf[e];
            ms = mnew;
        }
        float *sr = my_part + PS;
#pragma unroll
        for (int e = 0; e < CPL; ++e) sr[lane * CPL + e] = os[e];
        if (lane == 0) { sr[D] = ms; sr[D + 1] = ls; }
    }
    __syncthreads();

    // ---- merge the block's partials; write the result or this split's record ----
    static_assert(DEC_THREADS == D, "a thread per channel");
    const int ch = tid;
    const size_t oq = (size_t)b * p.Hq + h;
    auto merge = [&](int records, auto record, float *M_out, float *L_out) {
        float M = M_INIT, acc = 0.f, L = 0.f;
        for (int w = 0; w < records; ++w) M = fmaxf(M, record(w)[D]);
        for (int w = 0; w < records; ++w) {
            const float *pr = record(w);
            const float f = ex2(pr[D] - M);
            acc += pr[ch] * f;
            L += pr[D + 1] * f;
        }
        *M_out = M; *L_out = L;
        return acc;
    };
    auto write_out = [&](float acc, float M, float L) {
        out[oq * D + ch] = L > 0.f ? acc / L : 0.f;
        if (lse && ch == 0) lse[oq] = L > 0.f ? (M + log2f(L)) * 0.6931471805599453f : -INFINITY;
    };
    float M, L;
    const float acc = merge(2 * DEC_WARPS, [&](int w) { return part + (size_t)w * PS; }, &M, &L);
    if (nsplit == 1) {
        write_out(acc, M, L);
        return;
    }
    // the split's record: to the workspace for the merge kernel, or, when the splits of a unit form a thread-block cluster, to this
    // block's shared memory (the query tables are no longer needed) for the cluster's first block
    float *wsr = cluster_merge ? qs : part_ws + (oq * nsplit + split) * PS;
    wsr[ch] = acc;
    if (ch == 0) { wsr[D] = M; wsr[D + 1] = L; }
    if (cluster_merge) {
        namespace cg = cooperative_groups;
        cg::cluster_group cluster = cg::this_cluster();
        cluster.sync();
        if (split == 0) {
            const float all = merge(nsplit, [&](int s) { return (const float *)cluster.map_shared_rank(qs, s); }, &M, &L);
            write_out(all, M, L);
        }
        cluster.sync();   // nobody's shared memory goes away while the first block reads it
    }
}

}  // namespace kvsink
