// Single-token decode attention, two to four query heads per KV head (3 bit: four at a time of any number; head size 128): decode_one.cuh's
// scheme, keys and values on the integer tensor path with the weights in fixed point, for R = 2 or 4 rows of a block.
//
// What bounds it: issue slots and latency, as there.  A lane (g, t) owns tokens of one row: R = 4 tokens g, g + 8, ... of row t, R = 2 tokens
// 8 (t % 2) + g, + 16 of row t / 2.
// Keys: a row's four signed bytes in four of the eight columns of an operand (R = 4: two operands, the upper bytes and the lower).
// Values: a pair of tiles is multiplied together: the bytes of both tiles' words that belong to one 16-channel matrix are put in one word
// (4 bit: they are already), so that all 32 contraction slots are tokens and no column is spent on telling matrices apart.
//   weight = rint(2^(s - ref) * scale * 2^ev), below 2^31, ref per row and ev per row and value channel group; sums of a byte are exact in
//   int32.  When a weight does not fit (one vote a step) the references and units of the rows move by whole bits and the sums with them, in place:
//   with four rows there are 64 of them a lane, and rescaling them in binary32 (another 64 values, which only fit local memory) took 1.5 times as
//   long as everything else.
// Append and decode, us a pass, fp16 values (and the same merge and splits) before, this kernel now: 16 x 8 units of 30000 tokens, four heads
// each, 4 bit, 140 -> 127; 4 x 8 of 30000, 3 bit, 53 -> 54; 8 x 8 of 16000, groups of 32, 2 bit, 67 -> 63, groups of 64 46 -> 47; two heads,
// 2 bit 34.8 -> 30.4, 4 bit 44.2 -> 38.9 (all of these some 5 % less since the ring is filled by all lanes, behind the queries' loads).  Error against 64 bits, 8192 tokens a warp: N(0,1) 2e-3 -> 2e-5, scores with a deviation of four nats
// 4e-4 -> 1e-5; a weight keeps 22 bits of the row's largest at least, smaller ones their sum.  Three and four heads at 2 bit with one channel
// group a row stay in decode_kernel.cuh (decode_launch.cuh says why).
#pragma once
#include "decode_one.cuh"

namespace kvsink {

// Fragment of 16 value channels (matrix 2 i + e) of a pair of tiles: all 32 contraction slots are tokens.
template <int BITS>
__device__ __forceinline__ void pair_frag(const uint32_t (&va)[2 * BITS], const uint32_t (&vb)[2 * BITS], int i, int e, uint32_t (&a)[4])
{
    const uint32_t sel = e ? 0x7351u : 0x6240u;      // the matrix' bytes of both tiles' words
    if constexpr (BITS == 4) {
        const uint32_t x = va[2 * i + e], y = vb[2 * i + e];
        a[0] = x & 0x0f0f0f0fu; a[1] = x & 0xf0f0f0f0u; a[2] = y & 0x0f0f0f0fu; a[3] = y & 0xf0f0f0f0u;
    } else if constexpr (BITS == 2) {
        const uint32_t z = __byte_perm(va[i], vb[i], sel);
        a[0] = z & 0x03030303u; a[1] = z & 0x0c0c0c0cu; a[2] = z & 0x30303030u; a[3] = z & 0xc0c0c0c0u;
    } else {
        uint32_t me0, mo0, me1, mo1;
        nibbles3(va, i, &me0, &mo0);
        nibbles3(vb, i, &me1, &mo1);
        const uint32_t me = __byte_perm(me0, me1, sel), mo = __byte_perm(mo0, mo1, sel);
        a[0] = me & 0x07070707u; a[1] = mo & 0x07070707u; a[2] = me & 0x70707070u; a[3] = mo & 0x70707070u;
    }
}

template <int BITS, int NGv, int CT, int PM, int R>
__global__ void __launch_bounds__(DEC_THREADS, 4)
decode_few_kernel(Params p, kvsink_cache c, kvsink_static_params sp, const __half *__restrict__ q, float *__restrict__ out, float *__restrict__ lse,
                  float *__restrict__ part_ws, int nsplit, int groups_per_split, int qchunks, int seq_len, int cluster_merge)
{
    constexpr int D = 128, W = 2 * BITS, TILE_WORDS = 32 * W, CPL = D / 32;
    using Plan = DecodePlan<BITS, D, NGv, CT, R, PM == 2>;
    constexpr int NSLOT = Plan::NSLOT, SLOT_BYTES = Plan::SLOT_BYTES, KV_BYTES = Plan::KV_BYTES, SZ_BYTES = Plan::SZ_BYTES, PS = Plan::PS;
    constexpr int TP = CT >= 2 ? 2 : 1, NP = CT / TP;                // tiles of a pair, pairs of a chunk
    static_assert(R == 2 || R == 4, "rows of a block");
    constexpr int NT = R == 4 ? 2 : 1;                               // blocks of eight operand columns
    constexpr int SC = R;                                            // scores of a pair that a lane owns
    constexpr bool CAL = PM == 1, KT = PM == 2, FLAT = PM != 0;    // static parameters / per-token keys / either: no token groups
    constexpr int NGK = KT ? NGv : 1;                              // separate dot products per token on the key side
    static_assert(CT == 1 || CT == 2 || CT == 4, "whole pairs of tiles");
    static_assert(!KT || NGv <= 2, "per-token keys: one or two channel groups");
    constexpr float LOG2E = 1.4426950408889634f;
    constexpr float ROWF = BITS == 2 ? 0.25f : (BITS == 4 ? 0.0625f : 1.f);      // rows g + 8 of a fragment: place of their field
    constexpr float UPF = BITS == 4 ? 1.f : 0.0625f;                             // upper contraction slots: place of their field
    constexpr float WEIGHT_LIMIT = 2130706432.f;                                 // 0x7f000000: its carries still fit a signed byte
    constexpr int PLACE = BITS == 4 ? 24 : 26;                                   // a new unit puts the largest weight into [2^PLACE, 2^(PLACE + 1))

    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), g = lane >> 2, t = lane & 3;
    const bool odd = t & 1;
    // this lane's row and tokens of a pair: token own + OWN_STEP * k for score k
    const int row = R == 2 ? t >> 1 : t, own = R == 2 ? 8 * (t & 1) + g : g;
    constexpr int OWN_STEP = R == 2 ? 16 : 8;
    const int split = blockIdx.x, h = blockIdx.y / qchunks, qc = blockIdx.y % qchunks, b = blockIdx.z;
    const int nq = min(R, p.rep - R * qc), hq0 = h * p.rep + R * qc;
    const int64_t unit = (int64_t)b * p.Hkv + h;
    const int G = FLAT ? CT * KVSINK_TILE : p.G;                     // without token groups one ring chunk plays their part
    const int n = seq_len, n_groups = FLAT ? (n + G - 1) / G : n / G, n_body = FLAT ? n : n_groups * G;
    const int TPG = G / KVSINK_TILE, CPG = TPG / CT;                 // tiles and ring chunks per key group
    const uint32_t *bm = c.sink_bitmask + (size_t)b * p.mask_words;
    const float qscale = LOG2E * rsqrtf((float)D);

    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *qs = (float *)smem_raw;                                   // [R][D] q * log2e/sqrt(D)
    __half *q16 = (__half *)(qs + R * D);                            // [R][D] q as given
    uint64_t *bars = (uint64_t *)(smem_raw + Plan::Q_BYTES + DEC_WARPS * Plan::B_BYTES);   // [warps]: of the parameter slot
    unsigned char *ring_all = smem_raw + Plan::FIXED;                // [warps][WARP_RING]; later reused for the partials
    float *part = (float *)ring_all;                                 // [2*warps][nq][D+2]

    const uint32_t pbar = smem_addr(bars + warp);
    if (lane == 0) {
        mbar_init(pbar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // everything above overlaps the tail of the kernel before this one; nothing it may have written is read before this point
    pdl_wait();
    pdl_release();
    // Sink rows are shared out over all warps of all splits and handled after the stream, SB at a time: all of their loads together,
    // a batch ahead (one row at a time cost 1311 rows of eight units in 64 splits 3.6 us, five trips to memory a warp).  The first row is
    // asked for here; there are no registers for more of them to wait in.
    constexpr int SB = 4;
    const int sink_n = min(c.sink_count[b], p.cap);
    const int sink_worker = split * DEC_WARPS + warp, sink_workers = nsplit * DEC_WARPS;
    uint2 sink_k[SB], sink_v[SB];
    int sink_pos[SB];
    auto fetch_sinks = [&](int first, int from, int to) {
#pragma unroll
        for (int i = 0; i < SB; ++i) {
            if (i < from || i >= to) continue;
            const int j = first + i * sink_workers;
            sink_pos[i] = -1;
            sink_k[i] = sink_v[i] = make_uint2(0u, 0u);
            if (j < sink_n) {
                const size_t at = ((size_t)unit * p.cap + j) * D + lane * CPL;
                sink_pos[i] = c.sink_pos[(size_t)b * p.cap + j];
                sink_k[i] = *(const uint2 *)((const __half *)c.sink_k + at);
                sink_v[i] = *(const uint2 *)((const __half *)c.sink_v + at);
            }
        }
    };
    fetch_sinks(sink_worker, 0, 1);

    unsigned char *Bs = smem_raw + Plan::Q_BYTES + (size_t)warp * Plan::B_BYTES;             // key operand of the group, 512 bytes a row
    const uint8_t *kc_base = c.k_codes + (size_t)unit * p.max_seq * p.row_bytes;
    const uint8_t *vc_base = c.v_codes + (size_t)unit * p.max_seq * p.row_bytes;
    const float *vs_base = c.v_scale + (size_t)unit * p.max_seq * NGv;
    const float *vz_base = c.v_zero + (size_t)unit * p.max_seq * NGv;
    const float *ktok_s_base = c.k_scale + (size_t)unit * p.max_seq * NGv;    // per-token keys: [unit][max_seq][NGv]
    const float *ktok_z_base = c.k_zero + (size_t)unit * p.max_seq * NGv;
    const float *ks_base = c.k_scale + (size_t)unit * (p.max_seq / G) * D;
    const float *kz_base = c.k_zero + (size_t)unit * (p.max_seq / G) * D;

    // ---------------- running state ----------------
    float ref = M_INIT, l = 0.f;          // reference of the row's weights, and this lane's part of their sum
    float bv[NGv];                        // this lane's part of the sum of weight * scale * zero per value channel group
    // Byte sums in units of 2^-ev of the row: O[m] = matrix m, two columns of rows g, then of rows g + 8: two bytes of the row (R = 4: O[8 + m]
    // the lower two).
    int O[8 * NT][4];
    const float up = (BITS != 4 && odd) ? 0.0625f : 1.f;             // R = 2: this lane's tokens stand in the upper contraction slots
    auto up_of = [&](int k) { return R == 4 ? ((BITS != 4 && (k & 1)) ? 0.0625f : 1.f) : up; };
    float dither = (lane + 0.5f) * (1.f / 32) - 0.5f;
    float evf[NGv];                       // 2^ev, a value channel group's own: groups may lie far apart in size
#pragma unroll
    for (int j = 0; j < NGv; ++j) evf[j] = pow2i(60);
#pragma unroll
    for (int i = 0; i < 8 * NT; ++i)
#pragma unroll
        for (int x = 0; x < 4; ++x) O[i][x] = 0;
#pragma unroll
    for (int j = 0; j < NGv; ++j) bv[j] = 0.f;

    // The sums of value channel group j in a unit 2^k times as large (k <= 8, the same for a row's lanes): what a byte's sum loses at its lower
    // end goes to the next lower byte, and only the lowest one's is rounded.
    auto shift_sums = [&](int j, int k) {
        const int lost = (1 << k) - 1, half = (1 << k) >> 1, up = 1 << (8 - k);
#pragma unroll
        for (int i = 8 / NGv * j; i < 8 / NGv * (j + 1); ++i)
#pragma unroll
            for (int x = 0; x < 4; x += 2) {
                if constexpr (R == 2) {      // bytes 3, 2 are the even lane's, 1, 0 the odd one's
                    const int hi = O[i][x], lo = O[i][x + 1], above = __shfl_xor_sync(0xffffffffu, lo, 1);
                    O[i][x] = (hi >> k) + (odd ? (above & lost) * up : 0);
                    O[i][x + 1] = ((lo + (odd ? half : 0)) >> k) + (hi & lost) * up;
                } else {
                    int (&u)[4] = O[i], (&v)[4] = O[(8 + i) % (8 * NT)];
                    v[x + 1] = ((v[x + 1] + half) >> k) + (v[x] & lost) * up;
                    v[x] = (v[x] >> k) + (u[x + 1] & lost) * up;
                    u[x + 1] = (u[x + 1] >> k) + (u[x] & lost) * up;
                    u[x] >>= k;
                }
            }
    };
    // Carries what the sums of the lower bytes exceed a byte by to the next byte; true if a top byte's sum is large then.
    auto carry_bytes = [&]() {
        int top = 0;
        auto carry = [](int &lo, int &hi) { const int c = lo >> 8; lo -= c * 256; hi += c; };
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int x = 0; x < 4; x += 2) {
                if constexpr (R == 2) {
                    carry(O[i][x + 1], O[i][x]);
                    const int c = odd ? O[i][x] >> 8 : 0, below = __shfl_xor_sync(0xffffffffu, c, 1);
                    O[i][x] -= c * 256;
                    if (!odd) { O[i][x + 1] += below; carry(O[i][x + 1], O[i][x]); }
                    top = max(top, odd ? 0 : abs(O[i][x]));
                } else {
                    int (&u)[4] = O[i], (&v)[4] = O[(8 + i) % (8 * NT)];
                    carry(v[x + 1], v[x]);
                    carry(v[x], u[x + 1]);
                    carry(u[x + 1], u[x]);
                    top = max(top, abs(u[x]));
                }
            }
        return top > (1 << 29);
    };
    // over the lanes of a row
    auto row_max = [&](float v) {
        if (R == 2) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        return v;
    };
    auto row_sum = [&](float v) {
        if (R == 2) v += __shfl_xor_sync(0xffffffffu, v, 1);
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
    // Weights of a step's tokens of this lane: pw = 2^(s - ref) and x = pw * scale in units of 2^-ev (plus the dither), after moving the rows' references and
    // (each channel group's) units if one weight of the warp does not fit.  References are whole numbers, so that the sums so far move by
    // whole bits; a new unit puts the row's largest weight of the step into [2^PLACE, 2^(PLACE + 1)), where it is not finer than the old one: 22 bits of it also in the upper
    // slots, which take a sixteenth, and room for weights 16 (4 bit: 64) times as large.  A move costs a few hundred instructions, most of them
    // for the sums, and more room means fewer moves: 2 bits more of it and 2 (4 bit: 4) bits less, append and decode of 4 x 8 units of 30000 tokens,
    // four heads, 3 bit, 52.4 and 54.3 us; 16 x 8, 4 bit, 131.7 with four bits less.
    auto weights = [&](const auto &s, const auto &sv, auto &pw, auto &x) {
        constexpr int N = sizeof(pw) / sizeof(pw[0]);
        dither = next_dither(dither);
        bool moves = false;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const float d = s[k] - ref;
            pw[k] = ex2(d);
            moves |= d > 64.f;
#pragma unroll
            for (int j = 0; j < NGv; ++j) {
                x[k][j] = fmaf(pw[k], sv[k][j] * (evf[j] * up_of(k)), dither);
                moves |= fabsf(x[k][j]) >= WEIGHT_LIMIT * up_of(k);
            }
        }
        if (!__any_sync(0xffffffffu, moves)) return;
        float top = ref;
#pragma unroll
        for (int k = 0; k < N; ++k) top = fmaxf(top, s[k]);
        top = ceilf(row_max(top));
        const bool first = ref == M_INIT;
        const int rise = (int)fminf(top - ref, 200.f);      // of a row that has no sums yet: 200
        const float f = rise > 126 ? 0.f : pow2i(-rise);
        ref = top;
        l *= f;
#pragma unroll
        for (int k = 0; k < N; ++k) pw[k] = ex2(s[k] - ref);
#pragma unroll
        for (int j = 0; j < NGv; ++j) {
            float wm = 0.f;
#pragma unroll
            for (int k = 0; k < N; ++k) wm = fmaxf(wm, pw[k] * fabsf(sv[k][j]));
            const int ev = floor_log2(evf[j]), to = min(max(min(PLACE - floor_log2(row_max(wm)), 60), -60), ev + rise);
            // the sums are below 2^56
            for (int left = first ? 0 : min(ev + rise - to, 56); __any_sync(0xffffffffu, left > 0); left -= 8) shift_sums(j, min(max(left, 0), 8));
            evf[j] = pow2i(to);
            bv[j] *= f;
#pragma unroll
            for (int k = 0; k < N; ++k) x[k][j] = fmaf(pw[k], sv[k][j] * (evf[j] * up_of(k)), dither);
        }
    };
    // The value products of a pair: this lane's tokens' weights and parameters, and the two tiles' words.
    const uint32_t pair_sel = R == 2 && odd ? 0x4051u : 0x6273u;     // bytes of two tokens for this lane's two columns
    auto pair_values = [&](const auto &pw, const auto &x, const auto &sv, const auto &zv, auto words) {
#pragma unroll
        for (int k = 0; k < SC; ++k) {
            l += pw[k];
#pragma unroll
            for (int j = 0; j < NGv; ++j) bv[j] = fmaf(pw[k], sv[k][j] * zv[k][j], bv[j]);
        }
        auto digits = [&](float v) { return ((uint32_t)__float2int_rn(v) + 0x00808080u) ^ 0x00808080u; };      // four signed bytes
        uint32_t va[W], vb[W];
        words(0, va);
        words(1, vb);
#pragma unroll
        for (int j = 0; j < NGv; ++j) {
            uint32_t F[4];      // digits of tokens g and g + 8 of the first tile, then of the second
            if constexpr (R == 4) {
#pragma unroll
                for (int k = 0; k < 4; ++k) F[k] = digits(x[k][j]);
            } else {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const uint32_t mine = digits(x[k][j]), other = __shfl_xor_sync(0xffffffffu, mine, 1);
                    F[2 * k] = odd ? other : mine;
                    F[2 * k + 1] = odd ? mine : other;
                }
            }
            uint32_t b0[NT], b1[NT];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const uint32_t sel = nt == 0 ? pair_sel : 0x4051u;
                b0[nt] = movm_trans(__byte_perm(F[0], F[BITS == 4 ? 1 : 2], sel));
                b1[nt] = movm_trans(__byte_perm(F[BITS == 4 ? 2 : 1], F[3], sel));
            }
#pragma unroll
            for (int i = 0; i < 4 / NGv; ++i) {
                const int w = j * (4 / NGv) + i;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    uint32_t a[4];
                    pair_frag<BITS>(va, vb, w, e, a);
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) imma16832(O[nt * 8 + 2 * w + e], a, b0[nt], b1[nt]);
                }
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
    uint2 mword_next = my_groups > 0 ? load_mask_words(w_begin * TPG) : make_uint2(0u, 0u);
    // The loads that come next are issued ahead of the first copies of the ring and used behind them: the copies of 16 warps keep the load unit busy,
    // and what is queued behind them waits (with the queries loaded behind them, us, before and now: 8 x 8 units of 8000 tokens, 2 bit,
    // 64-token groups, four heads each 27.0 and 26.3, two heads each, 3000 tokens 14.2 and 13.8, static 11.9 and 11.2)
    float cal_sv[NGv], cal_zv[NGv];       // static value parameters of the KV head
#pragma unroll
    for (int j = 0; j < NGv; ++j) { cal_sv[j] = CAL ? sp.v_scale[h * NGv + j] : 0.f; cal_zv[j] = CAL ? sp.v_zero[h * NGv + j] : 0.f; }
    __half q_v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) q_v[r] = r < nq ? q[((size_t)b * p.Hq + hq0 + r) * D + tid] : __float2half(0.f);
    if (my_groups > 0) {
        if (!FLAT) issue_params(0);
        for (int i = 0; i < NSLOT - 1; ++i) {      // a group of copies a chunk, empty ones behind the last
            if (iss < n_chunks) issue_chunk();
            copies_commit();
        }
    }
    // the first copies are in flight: now the query tables
#pragma unroll
    for (int r = 0; r < R; ++r) {
        q16[r * D + tid] = q_v[r];
        qs[r * D + tid] = __half2float(q_v[r]) * qscale;
    }
    __syncthreads();

    // Key operand: lane l prepares the bytes of one group of four contraction slots, (fragment l/8, lower or upper slots (l/4)%2, slots
    // 4(l%4) ... +3); these are its four channels and their query values.
    int i8_ch[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int mi = lane >> 3, c2 = (lane >> 2) & 1, tq = lane & 3;
        i8_ch[e] = BITS != 4 ? 16 * (2 * mi + (e & 1)) + 8 * c2 + 2 * tq + (e >> 1) : 16 * (2 * mi + c2) + 8 * (e & 1) + 2 * tq + (e >> 1);
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
                // a row's query in all of its lanes' columns: each lane finds its own tokens' scores
                const __half *qr = q16 + (R == 2 ? g >> 2 : g >> 1) * D + 16 * m + 2 * t;
                mma16816(acc, a, *(const uint32_t *)qr, *(const uint32_t *)(qr + 8));
            }
            float s[SC], sv[SC][NGv], zv[SC][NGv], pw[SC], x[SC][NGv];
#pragma unroll
            for (int k = 0; k < SC; ++k) {
                // the tile's 16 tokens: R = 2 the first score, R = 4 the first two; the pair's second tile is not there
                const int tok = T * KVSINK_TILE + own + OWN_STEP * k;
                const bool valid = k < R / 2 && tok < n && !mask_bit(bm, tok < n ? tok : 0);
                s[k] = valid ? ((R == 4 ? k & 1 : odd) ? acc[2] : acc[0]) * qscale : -INFINITY;
#pragma unroll
                for (int j = 0; j < NGv; ++j) {   // tokens beyond the sequence have no parameters yet
                    sv[k][j] = valid ? __ldg(vs_base + (size_t)tok * NGv + j) : 0.f;
                    zv[k][j] = valid ? __ldg(vz_base + (size_t)tok * NGv + j) : 0.f;
                }
            }
            weights(s, sv, pw, x);
            pair_values(pw, x, sv, zv, [&](int k, uint32_t (&w)[W]) {
                if (k == 0) load_tile<BITS, D>((const uint32_t *)(vc_base + (size_t)T * p.tile_bytes), lane, w);
                else {
#pragma unroll
                    for (int i = 0; i < W; ++i) w[i] = 0u;
                }
            });
        }
    }

    // state of the current key group (without token groups: set up on the first trip)
    float bias0 = 0.f, bias1 = 0.f, ck = 0.f, cr = 0.f;
    uint32_t bk[4][2];                    // R = 2; R = 4 reads the operand from shared memory
#pragma unroll
    for (int i = 0; i < 4; ++i) bk[i][0] = bk[i][1] = 0u;
    // Word of the operand table: fragment, lower or upper slots, row, byte (most significant first), slot group.  R = 2: a row's bytes in
    // four columns; R = 4: its upper two in columns 2 r, 2 r + 1 of the first block, its lower two in those of the second, a reading lane's
    // four words together.
    auto key_word = [](int i, int c2, int r, int y, int tq) {
        return R == 2 ? ((i * 2 + c2) * R + r) * 16 + y * 4 + tq : ((i * 8 + 2 * r + (y & 1)) * 4 + tq) * 4 + (y >> 1) * 2 + c2;
    };
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
            // F = rint(q * scale * 2^sh) with the largest |F| of the row in [2^29, 2^30), cut into four signed bytes (radix 256): every
            // factor is kept to 2^-30 of the group's largest one (2^-26 where it is pre-divided for the upper contraction slots).  Adding
            // 0x808080 propagates the carries of the signed digits and the exclusive-or removes the offset again.
            uint32_t *tab = reinterpret_cast<uint32_t *>(Bs);
            float sums[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float v[4], amax = 0.f, bsum = 0.f;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    v[e] = qs[r * D + i8_ch[e]] * scv[e];
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
                const uint32_t limb[4] = {__byte_perm(t1, t3, 0x7632), __byte_perm(t1, t3, 0x5410), __byte_perm(t0, t2, 0x7632),
                                          __byte_perm(t0, t2, 0x5410)};
#pragma unroll
                for (int y = 0; y < 4; ++y) tab[key_word(lane >> 3, (lane >> 2) & 1, r, y, lane & 3)] = limb[y];
                if constexpr (KT && NGv == 2) {
                    // two channel groups: the query's sum over each (lanes 0-15 hold channels 0-63)
                    const float b0 = warp_sum(lane < 16 ? bsum : 0.f), b1 = warp_sum(lane < 16 ? 0.f : bsum);
                    if (row == r) { bias0 = b0; bias1 = b1; }
                }
                sums[r] = bsum;
                if (row == r) ck = pow2i(-sh);
            }
            if constexpr (!(KT && NGv == 2)) {
                // a lane needs its own row's sum only: rows are halved while lanes are added up
                if constexpr (R == 4) {
                    const float a0 = (odd ? sums[1] : sums[0]) + __shfl_xor_sync(0xffffffffu, odd ? sums[0] : sums[1], 1);
                    const float a1 = (odd ? sums[3] : sums[2]) + __shfl_xor_sync(0xffffffffu, odd ? sums[2] : sums[3], 1);
                    bias0 = row_sum(((t & 2) ? a1 : a0) + __shfl_xor_sync(0xffffffffu, (t & 2) ? a0 : a1, 2));
                } else {
                    bias0 = row_sum(((t & 2) ? sums[1] : sums[0]) + __shfl_xor_sync(0xffffffffu, (t & 2) ? sums[0] : sums[1], 2));
                }
            }
            // a lane's sum is keep * ck + got * cr; R = 2: even lanes keep the upper bytes' half of rows g, odd lanes the lower bytes'
            // half of rows g + 8; R = 4: the upper bytes' half
            if (R == 2) {
                const float ks = odd ? ck * ROWF : ck;
                ck = odd ? ks : ks * 65536.f;
                cr = odd ? ks * 65536.f : ks;
            } else {
                cr = ck;
                ck *= 65536.f;
            }
            __syncwarp();
            // every lane's parameters have gone into sums over the warp: the slot can take the next group's while this one streams
            if (!FLAT && gi + 1 < my_groups) issue_params(gi + 1);
            if (R == 2) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int c2 = 0; c2 < 2; ++c2) bk[i][c2] = tab[key_word(i, c2, g >> 2, g & 3, t)];
            }
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
#pragma unroll
            for (int pr = 0; pr < NP; ++pr) {
                // ---- scores: each lane ends with those of its own tokens ----
                float s[SC];
                {
                    int ia[TP][NGK][NT][4];
                    uint32_t kw[TP][W];
#pragma unroll
                    for (int k = 0; k < TP; ++k) {
                        load_tile_shared<BITS, D>(kt + (pr * TP + k) * TILE_WORDS, lane, kw[k]);
#pragma unroll
                        for (int j = 0; j < NGK * NT; ++j)
#pragma unroll
                            for (int x = 0; x < 4; ++x) ia[k][j / NT][j % NT][x] = 0;
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        uint4 kb;
                        if constexpr (R == 4) kb = *reinterpret_cast<const uint4 *>(reinterpret_cast<const uint32_t *>(Bs) + (i * 32 + lane) * 4);
                        else kb = make_uint4(bk[i][0], bk[i][1], 0u, 0u);
#pragma unroll
                        for (int k = 0; k < TP; ++k) {
                            uint32_t a[4];
                            byte_frag<BITS>(kw[k], i, a);
                            int (&acc)[NT][4] = ia[k][NGK == 2 ? (i >> 1) : 0];
                            imma16832(acc[0], a, kb.x, kb.y);
                            if constexpr (NT == 2) imma16832(acc[1], a, kb.z, kb.w);
                        }
                    }
                    // the two halves of a token's sum (column sums are below 2^22, two of them joined below 2^31), then the score
                    float keep[SC][NGK], got[SC][NGK];
#pragma unroll
                    for (int j = 0; j < NGK; ++j) {
                        if constexpr (R == 4) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const int (&acc)[NT][4] = ia[(k >> 1) < TP ? (k >> 1) : 0][j];
                                keep[k][j] = (float)(acc[0][2 * (k & 1)] * 256 + acc[0][2 * (k & 1) + 1]);
                                got[k][j] = (float)(acc[NT - 1][2 * (k & 1)] * 256 + acc[NT - 1][2 * (k & 1) + 1]);
                            }
                        } else {
#pragma unroll
                            for (int k = 0; k < SC; ++k) {
                                const int (&acc)[4] = ia[k < TP ? k : 0][j][0];
                                const int x0 = acc[0] * 256 + acc[1], x1 = acc[2] * 256 + acc[3];
                                keep[k][j] = (float)(odd ? x1 : x0);
                                got[k][j] = (float)__shfl_xor_sync(0xffffffffu, odd ? x0 : x1, 1);
                            }
                        }
                    }
#pragma unroll
                    for (int k = 0; k < SC; ++k) {
                        const float rf = (R == 4 && (k & 1)) ? ROWF : 1.f;
                        float r = 0.f;
                        if constexpr (KT) {
                            // per-token keys: scale * (dot product - zero * sum of the query), per channel group
#pragma unroll
                            for (int j = 0; j < NGK; ++j) {
                                const int at = (pr * 32 + OWN_STEP * k) * NGv + j;
                                if (TP == 2 || k < (R + 1) / 2)
                                    r = fmaf(kts[at], fmaf(-ktz[at], j == 0 ? bias0 : bias1, fmaf(keep[k][j], ck * rf, got[k][j] * (cr * rf))), r);
                            }
                        } else {
                            r = fmaf(keep[k][0], ck * rf, fmaf(got[k][0], cr * rf, -bias0));
                        }
                        s[k] = r;
                    }
                    const uint32_t mw = TP == 1 && (T0 & 1) ? mwords.x >> 16 : (pr == 0 ? mwords.x : mwords.y);
                    if (mw) {   // sink tokens are not part of the packed stream
#pragma unroll
                        for (int k = 0; k < SC; ++k)
                            if ((mw >> (own + OWN_STEP * k)) & 1u) s[k] = -INFINITY;
                    }
                    if (TP == 1) {      // no second tile
#pragma unroll
                        for (int k = 0; k < SC; ++k)
                            if (own + OWN_STEP * k >= KVSINK_TILE) s[k] = -INFINITY;
                    }
                    if constexpr (FLAT) {
                        if ((T0 + CT) * KVSINK_TILE > n) {   // the last tiles reach beyond the sequence: those tokens do not exist
#pragma unroll
                            for (int k = 0; k < SC; ++k)
                                if (T0 * KVSINK_TILE + pr * 32 + own + OWN_STEP * k >= n) s[k] = -INFINITY;
                        }
                    }
                }
                // ---- one softmax step, then its value products ----
                float sv[SC][NGv], zv[SC][NGv], pw[SC], x[SC][NGv];
#pragma unroll
                for (int k = 0; k < SC; ++k) {
                    const int at = pr * 32 + OWN_STEP * k;
                    const bool there = TP == 2 || own + at < KVSINK_TILE;
#pragma unroll
                    for (int j = 0; j < NGv; ++j) {
                        sv[k][j] = CAL ? cal_sv[j] : (there ? ssv[at * NGv + j] : 0.f);
                        zv[k][j] = CAL ? cal_zv[j] : (there ? szv[at * NGv + j] : 0.f);
                        if constexpr (KT) {   // tokens beyond the sequence: whatever the arrays hold there must not reach the sums
                            if (T0 * KVSINK_TILE + at + own >= n) sv[k][j] = zv[k][j] = 0.f;
                        }
                    }
                }
                weights(s, sv, pw, x);
                pair_values(pw, x, sv, zv, [&](int k, uint32_t (&w)[W]) {
                    if (k < TP) load_tile_shared<BITS, D>(vt + (pr * TP + k) * TILE_WORDS, lane, w);
                    else {
#pragma unroll
                        for (int i = 0; i < W; ++i) w[i] = 0u;
                    }
                });
            }
            // a tile adds less than 2^19 to a sum of bytes
            if ((ci & (2048 / CT - 1)) == 2048 / CT - 1 && __any_sync(0xffffffffu, carry_bytes())) {
#pragma unroll
                for (int j = 0; j < NGv; ++j) {
                    shift_sums(j, 1);
                    evf[j] *= 0.5f;
                }
                carry_bytes();
            }
        }
    }
    copies_wait<0>();      // the ring's space is used again
    if (!stream_ok && lane == 0) atomicOr(c.status, KVSINK_STATUS_TIMEOUT);

    fetch_sinks(sink_worker, 1, SB);

    // ---- this warp's partial records of the packed stream ----
    l = row_sum(l);
#pragma unroll
    for (int j = 0; j < NGv; ++j) bv[j] = row_sum(bv[j]);
    __syncthreads();   // every warp has drained its ring: the space now holds the block's partials
    float *my_part = part + (size_t)(2 * warp) * nq * PS;
#pragma unroll
    for (int m = 0; m < 8; ++m)
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            auto sum = [&](int i) { return fmaf((float)O[i][2 * half], 256.f, (float)O[i][2 * half + 1]); };      // two neighbouring bytes
            float o = sum(m);
            if constexpr (R == 4) o = fmaf(o, 65536.f, sum((8 + m) % (8 * NT)));
            else {      // the lane pair's halves
                o *= odd ? 1.f : 65536.f;
                o += __shfl_xor_sync(0xffffffffu, o, 1);
            }
            if (row < nq && (R == 4 || odd == (half == 1)))
                my_part[row * PS + 16 * m + 8 * half + g] = o * (pow2i(-floor_log2(evf[m * NGv / 8])) * (half ? ROWF : 1.f)) - bv[m * NGv / 8];
        }
    if (row < nq && g == 0 && (R == 4 || !odd)) { my_part[row * PS + D] = ref; my_part[row * PS + D + 1] = l; }

    // ---------------- sink rows (fp16 side buffer), plain fp32 arithmetic; a warp without one leaves no record ----------------
    if (sink_worker < sink_n) {
        float ms[R], ls[R], os[R][CPL];
#pragma unroll
        for (int i = 0; i < R; ++i) {
            ms[i] = M_INIT; ls[i] = 0.f;
#pragma unroll
            for (int e = 0; e < CPL; ++e) os[i][e] = 0.f;
        }
        for (int first = sink_worker; first < sink_n; first += SB * sink_workers) {
            // most warps have one row, if any: the work of a whole batch only where there are more
            auto rows = [&](auto batch) {
            constexpr int N = decltype(batch)::value;
            float kf[N][CPL], vf[N][CPL];
            bool seen[N];
#pragma unroll
            for (int i = 0; i < N; ++i) {
                seen[i] = sink_pos[i] >= 0 && sink_pos[i] < n;
                const uint32_t kk[2] = {sink_k[i].x, sink_k[i].y}, vv[2] = {sink_v[i].x, sink_v[i].y};
#pragma unroll
                for (int e = 0; e < CPL / 2; ++e) {
                    const float2 k2 = __half22float2(*reinterpret_cast<const __half2 *>(&kk[e]));
                    const float2 v2 = __half22float2(*reinterpret_cast<const __half2 *>(&vv[e]));
                    kf[i][2 * e] = k2.x; kf[i][2 * e + 1] = k2.y;
                    vf[i][2 * e] = seen[i] ? v2.x : 0.f; vf[i][2 * e + 1] = seen[i] ? v2.y : 0.f;
                }
            }
            if (N == SB && first + SB * sink_workers < sink_n) fetch_sinks(first + SB * sink_workers, 0, SB);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (r >= nq) break;
                const float4 qf = *(const float4 *)(qs + r * D + lane * CPL);
                float sc[N], mnew = ms[r];
#pragma unroll
                for (int i = 0; i < N; ++i)
                    sc[i] = warp_sum(fmaf(qf.w, kf[i][3], fmaf(qf.z, kf[i][2], fmaf(qf.y, kf[i][1], qf.x * kf[i][0]))));
#pragma unroll
                for (int i = 0; i < N; ++i) { sc[i] = seen[i] ? sc[i] : -INFINITY; mnew = fmaxf(mnew, sc[i]); }
                const float corr = ex2(ms[r] - mnew);
                ls[r] *= corr;
#pragma unroll
                for (int e = 0; e < CPL; ++e) os[r][e] *= corr;
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const float pp = ex2(sc[i] - mnew);
                    ls[r] += pp;
#pragma unroll
                    for (int e = 0; e < CPL; ++e) os[r][e] = fmaf(pp, vf[i][e], os[r][e]);
                }
                ms[r] = mnew;
            }
            };
            if (first + sink_workers < sink_n) rows(Count<SB>());
            else rows(Count<1>());
        }
        float *sr = my_part + (size_t)nq * PS;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            if (i >= nq) break;
#pragma unroll
            for (int e = 0; e < CPL; ++e) sr[i * PS + lane * CPL + e] = os[i][e];
            if (lane == 0) { sr[i * PS + D] = ms[i]; sr[i * PS + D + 1] = ls[i]; }
        }
    }
    __syncthreads();

    // ---- merge the block's partials; write the result or this split's record ----
    static_assert(DEC_THREADS == D, "a thread per channel");
    const int ch = tid;
    // up to eight records, absent ones left out; all loads of a pass together
    auto merge = [&](auto present, auto record, float *M_out, float *L_out) {
        float m[8], M = M_INIT, acc = 0.f, L = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            m[w] = present(w) ? record(w)[D] : M_INIT;
            M = fmaxf(M, m[w]);
        }
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const float f = ex2(m[w] - M);
            if (present(w)) {
                const float *pr = record(w);
                acc = fmaf(pr[ch], f, acc);
                L = fmaf(pr[D + 1], f, L);
            }
        }
        *M_out = M; *L_out = L;
        return acc;
    };
    auto write_out = [&](int r, float acc, float M, float L) {
        const size_t oq = (size_t)b * p.Hq + hq0 + r;
        out[oq * D + ch] = L > 0.f ? acc / L : 0.f;
        if (lse && ch == 0) lse[oq] = L > 0.f ? (M + log2f(L)) * 0.6931471805599453f : -INFINITY;
    };
    for (int r = 0; r < nq; ++r) {
        float M, L;
        static_assert(2 * DEC_WARPS == 8, "records of a block");
        const float acc = merge([&](int w) { return !(w & 1) || split * DEC_WARPS + (w >> 1) < sink_n; },
                                [&](int w) { return part + ((size_t)w * nq + r) * PS; }, &M, &L);
        if (nsplit == 1) {
            write_out(r, acc, M, L);
        } else {
            // the split's record: to the workspace for the merge kernel, or, when the splits of a unit form a thread-block cluster, to
            // this block's shared memory (the query tables are no longer needed) for the cluster
            float *wsr = cluster_merge ? qs + (size_t)r * PS : part_ws + (((size_t)b * p.Hq + hq0 + r) * nsplit + split) * PS;
            wsr[ch] = acc;
            if (ch == 0) { wsr[D] = M; wsr[D + 1] = L; }
        }
    }
    if (cluster_merge) {
        namespace cg = cooperative_groups;
        cg::cluster_group cluster = cg::this_cluster();
        cluster.sync();
        for (int r = split; r < nq; r += nsplit) {      // the rows are shared out over the blocks
            float M, L;
            const float acc = merge([&](int s) { return s < nsplit; }, [&](int s) { return (const float *)cluster.map_shared_rank(qs, s < nsplit ? s : 0) + (size_t)r * PS; }, &M, &L);
            write_out(r, acc, M, L);
        }
        cluster.sync();   // nobody's shared memory goes away while another block reads it
    }
}

}  // namespace kvsink
