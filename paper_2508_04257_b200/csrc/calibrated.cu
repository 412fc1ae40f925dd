// Static (calibrated) parameters: the paper's per-channel-key / per-token-value scheme with fixed parameters (Section 5.1),
// sink tokens left out of the calibration as well as of the quantization (Algorithm 1's remark on calibration, Section 4.1,
// Appendix C "Dynamic and static quantization").
//   calibration : global min / max per key channel and per value channel group of every KV head over all sequences and
//                 non-sink tokens, then Eq. 10-11
//   append      : every token is coded on arrival with the fixed pairs (Eq. 8, values outside the calibrated range clamp);
//                 no key tail, no per-group parameters; sink rows go to the side buffer
// The append kernels of head size 128 serve per-token keys too (PT; Section 4.1 "Per-token quantization", Section 5.1's per-token Key and
// Value dynamic scheme): keys and values alike get one (scale, zero) per token and channel group, computed on arrival from
// the token's own extremes (Eq. 10-11) and stored in the cache's parameter arrays, sink tokens (0, 0).
#include "common.cuh"
#include "tile_words.cuh"

namespace kvsink {
namespace {

// fp16 bit pattern <-> integer in value order (both zeros map to 0).
__device__ __forceinline__ int ordered(unsigned b) { return (b & 0x8000u) ? -(int)(b & 0x7fffu) : (int)b; }
__device__ __forceinline__ float unordered(int o)
{
    const unsigned b = o >= 0 ? (unsigned)o : (0x8000u | (unsigned)(-o));
    return __half2float(__ushort_as_half((unsigned short)b));
}
constexpr int NO_MIN = 0x7fffffff, NO_MAX = -0x7fffffff - 1;

// workspace: int [4][Hkv][D] = key min, key max, value min, value max per channel, in value order
__global__ void calibrate_init_kernel(int *__restrict__ ws, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait();
    if (i < n) { ws[i] = NO_MIN; ws[n + i] = NO_MAX; ws[2 * n + i] = NO_MIN; ws[3 * n + i] = NO_MAX; }
}

constexpr int CAL_THREADS = 128, CAL_SLICE = 256;   // tokens per block

// grid (token slices, Hkv, B); thread = eight channels of one of 128 / (D / 8) token lanes.
__global__ void __launch_bounds__(CAL_THREADS)
calibrate_scan_kernel(Params p, const __half *__restrict__ k, const __half *__restrict__ v, int T, int64_t sb, int64_t sh, int64_t stt,
                      const uint32_t *__restrict__ bitmask, int *__restrict__ ws)
{
    __shared__ int s_mm[4][128];
    const int D = p.D, tid = threadIdx.x, oct = D / 8, co = tid % oct, tl = tid / oct, lanes = CAL_THREADS / oct;
    const int h = blockIdx.y, b = blockIdx.z;
    const uint32_t *bm = bitmask + (size_t)b * p.mask_words;
    if (tid < D) { s_mm[0][tid] = NO_MIN; s_mm[1][tid] = NO_MAX; s_mm[2][tid] = NO_MIN; s_mm[3][tid] = NO_MAX; }
    pdl_wait();
    __syncthreads();
    constexpr uint32_t PINF2 = 0x7C007C00u, NINF2 = 0xFC00FC00u;
    uint32_t kmn[4] = {PINF2, PINF2, PINF2, PINF2}, kmx[4] = {NINF2, NINF2, NINF2, NINF2};
    uint32_t vmn[4] = {PINF2, PINF2, PINF2, PINF2}, vmx[4] = {NINF2, NINF2, NINF2, NINF2};
    bool any = false;
    const int t_end = min(T, (int)(blockIdx.x + 1) * CAL_SLICE);
    for (int t = blockIdx.x * CAL_SLICE + tl; t < t_end; t += lanes) {
        if (mask_bit(bm, t)) continue;
        const int64_t off = b * sb + h * sh + (int64_t)t * stt + co * 8;
        const uint4 a = __ldg(reinterpret_cast<const uint4 *>(k + off)), c = __ldg(reinterpret_cast<const uint4 *>(v + off));
        const uint32_t ka[4] = {a.x, a.y, a.z, a.w}, va[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            __half2 x = *reinterpret_cast<const __half2 *>(&ka[j]), y = *reinterpret_cast<const __half2 *>(&va[j]);
            __half2 r;
            r = __hmin2(*reinterpret_cast<__half2 *>(&kmn[j]), x); kmn[j] = *reinterpret_cast<uint32_t *>(&r);
            r = __hmax2(*reinterpret_cast<__half2 *>(&kmx[j]), x); kmx[j] = *reinterpret_cast<uint32_t *>(&r);
            r = __hmin2(*reinterpret_cast<__half2 *>(&vmn[j]), y); vmn[j] = *reinterpret_cast<uint32_t *>(&r);
            r = __hmax2(*reinterpret_cast<__half2 *>(&vmx[j]), y); vmx[j] = *reinterpret_cast<uint32_t *>(&r);
        }
        any = true;
    }
    if (any) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int ch = co * 8 + 2 * j + e, shft = 16 * e;
                atomicMin(&s_mm[0][ch], ordered((kmn[j] >> shft) & 0xffffu));
                atomicMax(&s_mm[1][ch], ordered((kmx[j] >> shft) & 0xffffu));
                atomicMin(&s_mm[2][ch], ordered((vmn[j] >> shft) & 0xffffu));
                atomicMax(&s_mm[3][ch], ordered((vmx[j] >> shft) & 0xffffu));
            }
    }
    __syncthreads();
    if (tid < D && s_mm[0][tid] != NO_MIN) {
        const int n = p.Hkv * D, o = h * D + tid;
        atomicMin(ws + o, s_mm[0][tid]);
        atomicMax(ws + n + o, s_mm[1][tid]);
        atomicMin(ws + 2 * n + o, s_mm[2][tid]);
        atomicMax(ws + 3 * n + o, s_mm[3][tid]);
    }
}

// One thread per key channel, then one per value channel group: Eq. 10-11 from the extremes.
__global__ void calibrate_finish_kernel(Params p, const int *__restrict__ ws, kvsink_static_params sp)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, n = p.Hkv * p.D;
    const float qmax = (float)((1 << p.bits) - 1);
    pdl_wait();
    if (i < n) {
        const bool any = ws[i] != NO_MIN;
        group_params(any, any ? unordered(ws[i]) : 0.f, any ? unordered(ws[n + i]) : 0.f, qmax, sp.k_scale + i, sp.k_zero + i);
    }
    if (i < p.Hkv * p.NGv) {
        const int h = i / p.NGv, j = i % p.NGv;
        int mn = NO_MIN, mx = NO_MAX;
        for (int e = 0; e < p.Gv; ++e) {
            mn = min(mn, ws[2 * n + h * p.D + j * p.Gv + e]);
            mx = max(mx, ws[3 * n + h * p.D + j * p.Gv + e]);
        }
        const bool any = mn != NO_MIN;
        group_params(any, any ? unordered(mn) : 0.f, any ? unordered(mx) : 0.f, qmax, sp.v_scale + i, sp.v_zero + i);
    }
}

// Eq. 8 with fixed parameters; scale 0 (nothing was calibrated) gives code 0.
__device__ __forceinline__ uint32_t code_static(float x, float s, float z, float qmax) { return s == 0.f ? 0u : code_exact(x, s, z, qmax); }

// Static pairs at head size 64: one block per (tile touched, KV head, sequence).  The new tokens' key and value codes are inserted into their tiles
// (fields of earlier tokens keep their bits; a tile whose first token arrives is written whole).
constexpr int CQ_THREADS = 128;

__global__ void __launch_bounds__(CQ_THREADS)
quantize_calibrated_kernel(Params p, kvsink_cache c, kvsink_static_params sp, const __half *__restrict__ k_src, const __half *__restrict__ v_src,
                           int first_token, int n_tokens, int64_t sb, int64_t sh, int64_t stt)
{
    constexpr int D = 64;
    __shared__ uint8_t kcode[KVSINK_TILE * D], vcode[KVSINK_TILE * D];
    __shared__ uint8_t present[KVSINK_TILE];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int h = blockIdx.y, b = blockIdx.z;
    const int64_t unit = (int64_t)b * p.Hkv + h;
    const int tile = first_token / KVSINK_TILE + blockIdx.x;
    const int t_lo = max(first_token, tile * KVSINK_TILE), t_hi = min(first_token + n_tokens, (tile + 1) * KVSINK_TILE);
    const float qmax = (float)((1 << p.bits) - 1);
    const uint32_t *bm = c.sink_bitmask + (size_t)b * p.mask_words;
    if (tid < KVSINK_TILE) present[tid] = (tile * KVSINK_TILE + tid >= t_lo && tile * KVSINK_TILE + tid < t_hi) ? 1 : 0;
    pdl_wait();
    if (!in_bounds(first_token >= 0 && first_token + n_tokens <= p.max_seq && (tile + 1) * KVSINK_TILE <= p.max_seq, c.status)) return;

    constexpr int cpl = D / 32;   // channels per lane
    float ks[cpl], kz[cpl], vs[cpl], vz[cpl];
    for (int e = 0; e < cpl; ++e) {
        const int ch = lane * cpl + e;
        ks[e] = sp.k_scale[h * D + ch]; kz[e] = sp.k_zero[h * D + ch];
        vs[e] = sp.v_scale[h * p.NGv + ch / p.Gv]; vz[e] = sp.v_zero[h * p.NGv + ch / p.Gv];
    }
    for (int pos = t_lo + warp; pos < t_hi; pos += CQ_THREADS / 32) {
        const int64_t src = b * sb + h * sh + (int64_t)(pos - first_token) * stt;
        const bool sink = mask_bit(bm, pos);
        __half kx[cpl], vx[cpl];
        for (int e = 0; e < cpl; ++e) { kx[e] = k_src[src + lane * cpl + e]; vx[e] = v_src[src + lane * cpl + e]; }
        if (sink) {
            const int count = min(c.sink_count[b], p.cap);
            const int slot = find_slot(c.sink_pos + (size_t)b * p.cap, count, pos);
            if (slot < 0) {
                if (lane == 0) atomicOr(c.status, KVSINK_STATUS_SINK_MISMATCH);
            } else {
                __half *dk = (__half *)c.sink_k + ((size_t)unit * p.cap + slot) * D;
                __half *dv = (__half *)c.sink_v + ((size_t)unit * p.cap + slot) * D;
                for (int e = 0; e < cpl; ++e) { dk[lane * cpl + e] = kx[e]; dv[lane * cpl + e] = vx[e]; }
            }
        }
        for (int e = 0; e < cpl; ++e) {
            const int o = (pos % KVSINK_TILE) * D + lane * cpl + e;
            kcode[o] = sink ? 0 : (uint8_t)code_static(__half2float(kx[e]), ks[e], kz[e], qmax);
            vcode[o] = sink ? 0 : (uint8_t)code_static(__half2float(vx[e]), vs[e], vz[e], qmax);
        }
    }
    __syncthreads();

    const int tile_words = p.tile_bytes / 4;
    const size_t tile_off = (size_t)unit * p.max_seq * p.row_bytes + (size_t)tile * p.tile_bytes;
    uint32_t *kout = (uint32_t *)(c.k_codes + tile_off), *vout = (uint32_t *)(c.v_codes + tile_off);
    const bool fresh = (t_lo % KVSINK_TILE) == 0;   // no earlier token lives in this tile
    for (int word = tid; word < tile_words; word += CQ_THREADS) {
        uint32_t fieldmask;
        // key tile: matrix element (row, col) = (token, channel); value tile: (channel, token)
        uint32_t newbits = assemble_word_masked(p.bits, D, word, [&](int m, int row, int col) {
            return present[row] ? (uint32_t)kcode[row * D + 16 * m + col] : 0x100u; }, &fieldmask);
        if (fieldmask || fresh) kout[word] = ((fresh ? 0u : kout[word]) & ~fieldmask) | newbits;
        newbits = assemble_word_masked(p.bits, D, word, [&](int m, int row, int col) {
            return present[col] ? (uint32_t)vcode[col * D + 16 * m + row] : 0x100u; }, &fieldmask);
        if (fieldmask || fresh) vout[word] = ((fresh ? 0u : vout[word]) & ~fieldmask) | newbits;
    }
}

// One token per sequence (a decode step's append): one warp per unit codes the key and the value row and sets their fields with
// word atomics.  A block per tile (as above, for any head size then) walks every word of both tiles for one token's fields: a step
// of a LLaMA2-shaped layer (append and attention) 28.7 us with it, 27.6 with this.
constexpr int CO_WARPS = 4;

template <bool PT>
__global__ void __launch_bounds__(32 * CO_WARPS)
append_one_flat_kernel(Params p, kvsink_cache c, kvsink_static_params sp, const __half *__restrict__ k_src, const __half *__restrict__ v_src, int pos,
                       int64_t sb, int64_t sh)
{
    const int D = p.D, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t unit = (int64_t)blockIdx.x * CO_WARPS + warp;
    pdl_wait();
    pdl_release();
    if (unit >= (int64_t)p.B * p.Hkv) return;
    if (!in_bounds(pos >= 0 && pos < p.max_seq, c.status)) return;
    const int b = (int)(unit / p.Hkv), h = (int)(unit % p.Hkv), cpl = D / 32;
    const float qmax = (float)((1 << p.bits) - 1);
    const int64_t src = b * sb + h * sh + lane * cpl;
    const bool sink = mask_bit(c.sink_bitmask + (size_t)b * p.mask_words, pos);
    __half kx[4], vx[4];
    float ks[4], kz[4], vs[4], vz[4];
    for (int e = 0; e < cpl; ++e) {
        const int ch = lane * cpl + e;
        kx[e] = k_src[src + e];
        vx[e] = v_src[src + e];
        if constexpr (!PT) {
            ks[e] = sp.k_scale[h * D + ch]; kz[e] = sp.k_zero[h * D + ch];
            vs[e] = sp.v_scale[h * p.NGv + ch / p.Gv]; vz[e] = sp.v_zero[h * p.NGv + ch / p.Gv];
        }
    }
    if (sink) {
        const int slot = find_slot(c.sink_pos + (size_t)b * p.cap, min(c.sink_count[b], p.cap), pos);
        if (slot < 0) {
            if (lane == 0) atomicOr(c.status, KVSINK_STATUS_SINK_MISMATCH);
        } else {
            __half *dk = (__half *)c.sink_k + ((size_t)unit * p.cap + slot) * D, *dv = (__half *)c.sink_v + ((size_t)unit * p.cap + slot) * D;
            for (int e = 0; e < cpl; ++e) { dk[lane * cpl + e] = kx[e]; dv[lane * cpl + e] = vx[e]; }
        }
    }
    if constexpr (PT) {
        float kmn = __half2float(kx[0]), kmx = kmn, vmn = __half2float(vx[0]), vmx = vmn;
        for (int e = 1; e < cpl; ++e) {
            kmn = fminf(kmn, __half2float(kx[e])); kmx = fmaxf(kmx, __half2float(kx[e]));
            vmn = fminf(vmn, __half2float(vx[e])); vmx = fmaxf(vmx, __half2float(vx[e]));
        }
        const int lanes_per_group = p.Gv / cpl;
        for (int o = 1; o < lanes_per_group; o <<= 1) {
            kmn = fminf(kmn, __shfl_xor_sync(0xffffffffu, kmn, o)); kmx = fmaxf(kmx, __shfl_xor_sync(0xffffffffu, kmx, o));
            vmn = fminf(vmn, __shfl_xor_sync(0xffffffffu, vmn, o)); vmx = fmaxf(vmx, __shfl_xor_sync(0xffffffffu, vmx, o));
        }
        float s0, z0, s1, z1;
        group_params(!sink, kmn, kmx, qmax, &s0, &z0);
        group_params(!sink, vmn, vmx, qmax, &s1, &z1);
        for (int e = 0; e < cpl; ++e) { ks[e] = s0; kz[e] = z0; vs[e] = s1; vz[e] = z1; }
        if (lane % lanes_per_group == 0) {
            const size_t o = ((size_t)unit * p.max_seq + pos) * p.NGv + lane / lanes_per_group;
            c.k_scale[o] = s0; c.k_zero[o] = z0;
            c.v_scale[o] = s1; c.v_zero[o] = z1;
        }
    }
    const int tile = pos / KVSINK_TILE, at = pos % KVSINK_TILE;
    const size_t tile_off = (size_t)unit * p.max_seq * p.row_bytes + (size_t)tile * p.tile_bytes;
    uint32_t *kout = (uint32_t *)(c.k_codes + tile_off), *vout = (uint32_t *)(c.v_codes + tile_off);
    const bool fresh = at == 0;                // a tile whose first token this is is written whole (zeros elsewhere)
    if (fresh) {
        for (int w = lane; w < p.tile_bytes / 4; w += 32) kout[w] = vout[w] = 0u;
        __syncwarp();
    }
    for (int e = 0; e < cpl; ++e) {            // key tile: element (token, channel); value tile: (channel, token)
        const int ch = lane * cpl + e;
        set_field(kout, p.bits, D, ch >> 4, at, ch & 15, sink ? 0u : code_static(__half2float(kx[e]), ks[e], kz[e], qmax), fresh);
        set_field(vout, p.bits, D, ch >> 4, ch & 15, at, sink ? 0u : code_static(__half2float(vx[e]), vs[e], vz[e], qmax), fresh);
    }
}

// Eq. 8 with fixed parameters without a division per element: r is the rounded reciprocal of the scale, so x * r is within
// 2^-22 |x / scale| of the quotient; unless it lies that close to a rounding tie, its nearest integer is that of the IEEE
// quotient.  Near a tie (fp16 inputs hit exact ties often), for huge quotients and for a reciprocal that is not finite the
// literal formula is evaluated.
__device__ __forceinline__ uint32_t code_static_fast(float x, float s, float r, float z, float qmax)
{
    const float q = x * r, c = rintf(q);
    const float room = 0.5f - fabsf(q - c);                    // distance to the nearest tie
    if (!(room > fabsf(q) * 4.76837158203125e-07f)) return code_static(x, s, z, qmax);
    return (uint32_t)(int)fminf(fmaxf(c + z, 0.f), qmax);
}

// The tiles of up to two spans of new tokens (head size 128), all of them and both spans in one launch: what a chunk has before its first
// whole group and behind its last, or a short chunk.  One block per 16-token tile: it stages the tile's new key and value rows in shared memory, and
// each of its four warps codes one side's elements of half the channels, a lane exactly those of its own pair slots of the packed tile, so
// that its words come out in the tile's own order.  Where earlier tokens live in the tile their fields are kept: a lane's words are its
// own, so that takes no atomics.
// Latency is what counts here (a few tiles a unit): a chunk's ragged ends were up to six launches, of whole tiles (a warp each) and of the tokens before and
// behind them, walking the words of both tiles field by field.  Per-token keys, 2 bit, 4 x 8 units, 91 tokens from 37: 35.0 us, one launch with a warp a
// tile 17.3, a block a tile 9.6; 14 x 4 units of 357 tokens 28.9, 19.0, 12.7.
constexpr int CF_THREADS = 128;
struct TokenSpans {
    int first[2], n[2], src[2];      // position of the first token, number of tokens, row of the first one in the source
    int tiles[2];                    // tiles that they touch
};

template <int BITS, bool PT>
__global__ void __launch_bounds__(CF_THREADS)
quantize_calibrated_tiles_kernel(Params p, kvsink_cache c, kvsink_static_params sp, const __half *__restrict__ k_src,
                                 const __half *__restrict__ v_src, TokenSpans spans, int64_t sb, int64_t sh, int64_t stt)
{
    constexpr int D = 128;
    constexpr int LO = BITS == 4 ? 4 : 2, HI = BITS == 3 ? 1 : 0;   // words of a warp's half of the channels: of whole codes or low bits, of high bits
    constexpr int ROW = D + 8;                                 // padded row (halves): conflict-free column reads
    __shared__ __align__(16) __half s_x[2][KVSINK_TILE * ROW];  // keys, values
    __shared__ float4 s_kp[PT ? 1 : D];                        // (scale, 1 / scale, zero) of the KV head's key channels
    __shared__ float4 s_pt[2][PT ? KVSINK_TILE : 1][4];        // the same per (keys / values, token, 32-channel block); static values: of the head
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int kind = warp & 1, half = warp >> 1;               // keys or values, lower or upper 64 channels
    const int h = blockIdx.y, b = blockIdx.z, ti = blockIdx.x;
    const int64_t unit = (int64_t)b * p.Hkv + h;
    const float qmax = (float)((1 << BITS) - 1);
    const uint32_t *bm = c.sink_bitmask + (size_t)b * p.mask_words;
    const int sp_i = ti >= spans.tiles[0], first = spans.first[sp_i], last = first + spans.n[sp_i];
    const int tok0 = (first / KVSINK_TILE + ti - (sp_i ? spans.tiles[0] : 0)) * KVSINK_TILE;
    pdl_wait();
    pdl_release();                                             // the whole groups' kernel of the same chunk may start beside this one
    if (!in_bounds(tok0 >= 0 && tok0 + KVSINK_TILE <= p.max_seq, c.status)) return;
    const int lo = max(first - tok0, 0), hi = min(last - tok0, KVSINK_TILE);                   // the tile's new tokens
    const uint32_t fresh16 = ((1u << hi) - 1u) & ~((1u << lo) - 1u);
    const uint32_t mask16 = (bm[tok0 >> 5] >> (tok0 & 31)) & fresh16;   // sink bits of the new tokens
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const int i = tid + CF_THREADS * x, side = i >> 8, r = (i >> 4) & 15, c8 = i & 15;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (r >= lo && r < hi)
            v = __ldg(reinterpret_cast<const uint4 *>((side ? v_src : k_src) + b * sb + h * sh + (int64_t)(spans.src[sp_i] + tok0 + r - first) * stt + c8 * 8));
        *reinterpret_cast<uint4 *>(s_x[side] + r * ROW + c8 * 8) = v;
    }
    auto triple = [](float sc, float z) { return make_float4(sc, sc == 0.f ? 0.f : __frcp_rn(sc), z, 0.f); };
    if constexpr (!PT) {
        s_kp[tid] = triple(sp.k_scale[h * D + tid], sp.k_zero[h * D + tid]);
        if (tid < 4) s_pt[1][0][tid] = triple(sp.v_scale[h * p.NGv + 32 * tid / p.Gv], sp.v_zero[h * p.NGv + 32 * tid / p.Gv]);
    }
    __syncthreads();
    // exact rows to the side buffer at the rank of their position
    if (mask16 && half == 0) {
        const int count = min(c.sink_count[b], p.cap);
        for (uint32_t rest = mask16; rest; rest &= rest - 1u) {
            const int r = __ffs((int)rest) - 1;
            const int slot = find_slot(c.sink_pos + (size_t)b * p.cap, count, tok0 + r);
            if (slot < 0) {
                if (tid == 0) atomicOr(c.status, KVSINK_STATUS_SINK_MISMATCH);
                continue;
            }
            __half *to = (__half *)(kind ? c.sink_v : c.sink_k) + ((size_t)unit * p.cap + slot) * D;
            if (lane < D / 8) *reinterpret_cast<uint4 *>(to + lane * 8) = *reinterpret_cast<const uint4 *>(s_x[kind] + r * ROW + lane * 8);
        }
    }
    if constexpr (PT) {
        // per-token parameters: a thread takes one 32-channel block of a token's keys or values; the four threads of a row put theirs together to the
        // channel group (32, 64 or 128 channels), whose first one writes the pair
        const int side = tid >> 6, tk = (tid >> 2) & 15, blk = tid & 3;
        const __half2 *row = reinterpret_cast<const __half2 *>(s_x[side] + tk * ROW + 32 * blk);
        __half2 l2 = row[0], h2 = l2;
#pragma unroll
        for (int x = 1; x < 16; ++x) { l2 = __hmin2(l2, row[x]); h2 = __hmax2(h2, row[x]); }
        float mn = fminf(__low2float(l2), __high2float(l2)), mx = fmaxf(__low2float(h2), __high2float(h2));
        for (int o = 1; 32 * o < p.Gv; o <<= 1) {
            mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        float sc, ze;
        group_params(!((mask16 >> tk) & 1u), mn, mx, qmax, &sc, &ze);
        s_pt[side][tk][blk] = triple(sc, ze);
        if (((fresh16 >> tk) & 1u) && 32 * blk % p.Gv == 0) {
            const size_t o = ((size_t)unit * p.max_seq + tok0 + tk) * p.NGv + 32 * blk / p.Gv;
            (side ? c.v_scale : c.k_scale)[o] = sc;
            (side ? c.v_zero : c.k_zero)[o] = ze;
        }
        __syncthreads();
    }
    // codes of pair slot s = 4m + r, half e: keys (token, channel) = (g + 8(r&1), 16m + 8(r>>1) + 2t + e),
    //                                        values (channel, token) = (16m + g + 8(r&1), 8(r>>1) + 2t + e)
    const uint32_t none16 = mask16 | ~fresh16;                 // code 0: sink tokens, and fields of tokens that are not this call's
    const __half *xs = s_x[kind];
    uint32_t w[LO + HI];
#pragma unroll
    for (int i = 0; i < LO + HI; ++i) w[i] = 0u;
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int s_ = 4 * m + r, row = g + 8 * (r & 1), col = 8 * (r >> 1) + 2 * t + e, ch0 = 64 * half + 16 * m;
                const int tok = kind ? col : row, ch = ch0 + (kind ? row : col);
                const float4 q = PT ? s_pt[kind][PT ? tok : 0][ch >> 5] : (kind ? s_pt[1][0][ch >> 5] : s_kp[PT ? 0 : ch]);
                const uint32_t code = ((none16 >> tok) & 1u) || q.x == 0.f ? 0u : code_static_fast(__half2float(xs[tok * ROW + ch]), q.x, q.y, q.z, qmax);
                if constexpr (BITS == 4) {
                    w[s_ / 4] |= code << (16 * e + 4 * (s_ % 4));
                } else if constexpr (BITS == 2) {
                    w[s_ / 8] |= code << (16 * e + 2 * (s_ % 8));
                } else {
                    const int i = s_ / 8, k = s_ % 8;
                    w[i] |= (code & 3u) << (16 * e + 2 * k);
                    w[LO] |= (code >> 2) << (16 * e + 4 * (k / 2) + 2 * (1 - i) + (k % 2));
                }
            }
    // the lane's words of its half: 2 and 3 bit two of the four in the plane, 4 bit the half's plane; 3 bit one of the two of the high bits
    const size_t tile_off = (size_t)unit * p.max_seq * p.row_bytes + (size_t)(tok0 / KVSINK_TILE) * p.tile_bytes;
    uint8_t *tile = (kind ? c.v_codes : c.k_codes) + tile_off;
    uint32_t *to = (uint32_t *)(tile + (BITS == 4 ? 512 * half + 16 * lane : 16 * lane + 8 * half)), *to_high = (uint32_t *)(tile + 512 + 8 * lane + 4 * half);
    if (lo > 0) {
        // earlier tokens live in the tile: their fields stay.  A slot's token: keys' by s % 2 among rows g, g + 8; values' by s / 2 % 2 among columns 2t + e, + 8
        uint32_t f[2];                                         // all ones where the word's fields of that kind are new
#pragma unroll
        for (int x = 0; x < 2; ++x)
            f[x] = kind ? ((fresh16 >> (2 * t + 8 * x)) & 1u ? 0xffffu : 0u) | ((fresh16 >> (2 * t + 1 + 8 * x)) & 1u ? 0xffff0000u : 0u)
                        : ((fresh16 >> (g + 8 * x)) & 1u ? 0xffffffffu : 0u);
        const uint32_t even = kind ? (BITS == 4 ? 0x00ff00ffu : 0x0f0f0f0fu) : (BITS == 4 ? 0x0f0f0f0fu : 0x33333333u);
        const uint32_t kept = ~((even & f[0]) | (~even & f[1]));
#pragma unroll
        for (int i = 0; i < LO; ++i) w[i] |= to[i] & kept;
        if constexpr (BITS == 3) {
            const uint32_t even_high = kind ? 0x0f0f0f0fu : 0x55555555u;
            w[LO] |= *to_high & ~((even_high & f[0]) | (~even_high & f[1]));
        }
    }
    if constexpr (BITS == 4) *reinterpret_cast<uint4 *>(to) = make_uint4(w[0], w[1], w[2], w[3]);
    else *reinterpret_cast<uint2 *>(to) = make_uint2(w[0], w[1]);
    if constexpr (BITS == 3) *to_high = w[LO];
}

}  // namespace

size_t calibrate_workspace_bytes(const Params &p) { return (size_t)4 * p.Hkv * p.D * sizeof(int) + 16; }

int launch_calibrate(const Params &p, const __half *k, const __half *v, int T, int64_t sb, int64_t sh, int64_t stt, const uint32_t *bitmask,
                     const kvsink_static_params &sp, void *workspace, cudaStream_t st)
{
    int *ws = (int *)workspace;
    const int n = p.Hkv * p.D;
    if (launch_pdl(calibrate_init_kernel, dim3((n + 255) / 256), dim3(256), 0, st, ws, n) != cudaSuccess) return KVSINK_ERR_CUDA;
    if (T > 0) {
        const dim3 grid((T + CAL_SLICE - 1) / CAL_SLICE, p.Hkv, p.B);
        if (launch_pdl(calibrate_scan_kernel, grid, dim3(CAL_THREADS), 0, st, p, k, v, T, sb, sh, stt, bitmask, ws) != cudaSuccess)
            return KVSINK_ERR_CUDA;
    }
    return launch_pdl(calibrate_finish_kernel, dim3((n + 255) / 256), dim3(256), 0, st, p, (const int *)ws, sp) == cudaSuccess ? KVSINK_OK
                                                                                                                                : KVSINK_ERR_CUDA;
}

// Up to two spans at head size 128.
template <bool PT>
static int launch_spans(const Params &p, const kvsink_cache &c, const kvsink_static_params &sp, const __half *k_src, const __half *v_src, TokenSpans s,
                        int64_t sb, int64_t sh, int64_t stt, cudaStream_t st)
{
    for (int i = 0; i < 2; ++i) s.tiles[i] = s.n[i] > 0 ? (s.first[i] + s.n[i] - 1) / KVSINK_TILE - s.first[i] / KVSINK_TILE + 1 : 0;
    const dim3 grid(s.tiles[0] + s.tiles[1], p.Hkv, p.B), block(CF_THREADS);
    if (grid.x == 0) return KVSINK_OK;
    const cudaError_t e = p.bits == 2   ? launch_pdl(quantize_calibrated_tiles_kernel<2, PT>, grid, block, 0, st, p, c, sp, k_src, v_src, s, sb, sh, stt)
                          : p.bits == 3 ? launch_pdl(quantize_calibrated_tiles_kernel<3, PT>, grid, block, 0, st, p, c, sp, k_src, v_src, s, sb, sh, stt)
                                        : launch_pdl(quantize_calibrated_tiles_kernel<4, PT>, grid, block, 0, st, p, c, sp, k_src, v_src, s, sb, sh, stt);
    return e == cudaSuccess ? KVSINK_OK : KVSINK_ERR_CUDA;
}

template <bool PT>
static int launch_tokens(const Params &p, const kvsink_cache &c, const kvsink_static_params &sp, const __half *k_src, const __half *v_src,
                         int first_token, int n_tokens, int64_t sb, int64_t sh, int64_t stt, cudaStream_t st)
{
    if (n_tokens <= 0) return KVSINK_OK;
    if (n_tokens == 1) {
        const long units = (long)p.B * p.Hkv;
        return launch_pdl(append_one_flat_kernel<PT>, dim3((unsigned)((units + CO_WARPS - 1) / CO_WARPS)), dim3(32 * CO_WARPS), 0, st, p, c, sp, k_src,
                          v_src, first_token, sb, sh) == cudaSuccess ? KVSINK_OK : KVSINK_ERR_CUDA;
    }
    if (p.D == 128) return launch_spans<PT>(p, c, sp, k_src, v_src, TokenSpans{{first_token, 0}, {n_tokens, 0}, {0, 0}, {0, 0}}, sb, sh, stt, st);
    if constexpr (PT) {
        return KVSINK_ERR_UNSUPPORTED;      // per-token keys: head size 128 alone
    } else {
        const int tiles = (first_token + n_tokens - 1) / KVSINK_TILE - first_token / KVSINK_TILE + 1;
        const dim3 grid(tiles, p.Hkv, p.B);
        return launch_pdl(quantize_calibrated_kernel, grid, dim3(CQ_THREADS), 0, st, p, c, sp, k_src, v_src, first_token, n_tokens, sb, sh, stt) ==
                       cudaSuccess ? KVSINK_OK : KVSINK_ERR_CUDA;
    }
}

// Whole G-token spans go to the bulk quantizer where it has a form for the scheme (G only shapes its work items with static parameters); the
// tokens before the first multiple of G and behind the last go ahead of it in one launch, beside which it may start (quantize_bulk.cu says why).
// Static parameters, 2859 tokens from 1237, 8 x 32 units, 2 bit: 579 us without the bulk quantizer, 105 with it.
template <bool PT>
static int launch_flat(const Params &p, const kvsink_cache &c, const kvsink_static_params &sp, const __half *k_src, const __half *v_src,
                       int first_token, int n_tokens, int64_t sb, int64_t sh, int64_t stt, cudaStream_t st)
{
    const int head = (p.G - first_token % p.G) % p.G, n_groups = (n_tokens - head) / p.G;
    if (n_tokens >= head + p.G) {
        const int64_t skip = (int64_t)head * stt;
        const int done = head + n_groups * p.G;
        const auto ends = [&] {
            return launch_spans<PT>(p, c, sp, k_src, v_src, TokenSpans{{first_token, first_token + done}, {head, n_tokens - done}, {0, done}, {0, 0}}, sb, sh, stt, st);
        };
        const LaunchBefore before = head > 0 || done < n_tokens ? launch_before(ends) : LaunchBefore{};
        const int rc = PT ? launch_quantize_pertoken_bulk(p, c, k_src + skip, v_src + skip, first_token + head, n_groups, sb, sh, stt, before, st)
                          : launch_quantize_static_bulk(p, c, sp, k_src + skip, v_src + skip, first_token + head, n_groups, sb, sh, stt, before, st);
        if (rc != KVSINK_ERR_UNSUPPORTED) return rc;
    }
    return launch_tokens<PT>(p, c, sp, k_src, v_src, first_token, n_tokens, sb, sh, stt, st);
}

int launch_quantize_calibrated(const Params &p, const kvsink_cache &c, const kvsink_static_params &sp, const __half *k_src, const __half *v_src,
                               int first_token, int n_tokens, int64_t sb, int64_t sh, int64_t stt, cudaStream_t st)
{
    return launch_flat<false>(p, c, sp, k_src, v_src, first_token, n_tokens, sb, sh, stt, st);
}

int launch_quantize_pertoken(const Params &p, const kvsink_cache &c, const __half *k_src, const __half *v_src, int first_token, int n_tokens,
                             int64_t sb, int64_t sh, int64_t stt, cudaStream_t st)
{
    const kvsink_static_params none = {nullptr, nullptr, nullptr, nullptr};
    return launch_flat<true>(p, c, none, k_src, v_src, first_token, n_tokens, sb, sh, stt, st);
}

}  // namespace kvsink
