// Asymmetric group quantization (Eq. 8-11) with sink exclusion (Algorithm 1), bit-packing into the tile
// layout, side-buffer compaction of sink rows, and the append path (Eq. 6).
#include "common.cuh"
#include "tile_words.cuh"

namespace kvsink {

// ---------------------------------------------------------------------------------------------------------
// Whole groups: one block per (token group, KV head, sequence).  Keys per channel over the group's non-sink
// tokens, values per token, sink rows to the side buffer.
// ---------------------------------------------------------------------------------------------------------
constexpr int QG_THREADS = 256;

__global__ void __launch_bounds__(QG_THREADS)
quantize_groups_kernel(Params p, kvsink_cache c, const __half *__restrict__ k_src, const __half *__restrict__ v_src,
                       int first_token, int64_t sb, int64_t sh, int64_t stt, int do_v_and_sinks)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int D = p.D, G = p.G, RS = D + 8;      // padded row stride in halves
    if (!in_bounds(first_token >= 0 && first_token + ((int)blockIdx.x + 1) * G <= p.max_seq, c.status)) return;   // every thread of the block alike
    __half *Kt = (__half *)smem;                  // [G][RS]
    __half *Vt = Kt + (size_t)G * RS;             // [G][RS]
    uint8_t *kcode = (uint8_t *)(Vt + (size_t)G * RS);   // [G][D]
    uint8_t *vcode = kcode + (size_t)G * D;               // [G][D]
    float *ks = (float *)(vcode + (size_t)G * D);         // [D] scale
    float *kz = ks + D;                                   // [D] zero
    float *vs = kz + D;                                   // [G][NGv]
    float *vz = vs + G * p.NGv;
    uint8_t *flag = (uint8_t *)(vz + G * p.NGv);          // [G] sink flags

    const int tid = threadIdx.x;
    const int grp = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int64_t unit = (int64_t)b * p.Hkv + h;
    const int p0 = first_token + grp * G;         // absolute position of the group's first token
    const int gidx = p0 / G;
    const float qmax = (float)((1 << p.bits) - 1);
    const uint32_t *bm = c.sink_bitmask + (size_t)b * p.mask_words;

    // load the tiles (16-byte chunks)
    const int chunks = D / 8;
    const __half *kbase = k_src + b * sb + h * sh + (int64_t)(grp * G) * stt;
    const __half *vbase = v_src + b * sb + h * sh + (int64_t)(grp * G) * stt;
    for (int idx = tid; idx < G * chunks; idx += QG_THREADS) {
        int t = idx / chunks, ch = (idx % chunks) * 8;
        *(uint4 *)(Kt + (size_t)t * RS + ch) = __ldg((const uint4 *)(kbase + (int64_t)t * stt + ch));
        if (do_v_and_sinks) *(uint4 *)(Vt + (size_t)t * RS + ch) = __ldg((const uint4 *)(vbase + (int64_t)t * stt + ch));
    }
    for (int t = tid; t < G; t += QG_THREADS) flag[t] = mask_bit(bm, p0 + t) ? 1 : 0;
    __syncthreads();

    // key parameters: one thread per channel
    for (int ch = tid; ch < D; ch += QG_THREADS) {
        bool any = false;
        float mn = 0.f, mx = 0.f;
        for (int t = 0; t < G; ++t) {
            if (flag[t]) continue;
            float x = __half2float(Kt[(size_t)t * RS + ch]);
            if (!any) { mn = mx = x; any = true; }
            else { mn = fminf(mn, x); mx = fmaxf(mx, x); }
        }
        float s, z;
        group_params(any, mn, mx, qmax, &s, &z);
        ks[ch] = s;
        kz[ch] = z;
        size_t o = ((size_t)unit * (p.max_seq / G) + gidx) * D + ch;
        c.k_scale[o] = s;
        c.k_zero[o] = z;
    }
    // value parameters: one thread per (token, channel group)
    if (do_v_and_sinks) {
        for (int it = tid; it < G * p.NGv; it += QG_THREADS) {
            int t = it / p.NGv, j = it % p.NGv;
            float s = 0.f, z = 0.f;
            if (!flag[t]) {
                const __half *row = Vt + (size_t)t * RS + j * p.Gv;
                float mn = __half2float(row[0]), mx = mn;
                for (int e = 1; e < p.Gv; ++e) {
                    float x = __half2float(row[e]);
                    mn = fminf(mn, x);
                    mx = fmaxf(mx, x);
                }
                group_params(true, mn, mx, qmax, &s, &z);
            }
            vs[it] = s;
            vz[it] = z;
            size_t o = ((size_t)unit * p.max_seq + p0 + t) * p.NGv + j;
            c.v_scale[o] = s;
            c.v_zero[o] = z;
        }
    }
    __syncthreads();

    // codes
    for (int idx = tid; idx < G * D; idx += QG_THREADS) {
        int t = idx / D, ch = idx % D;
        uint32_t kc = 0, vc = 0;
        if (!flag[t]) {
            kc = code_exact(__half2float(Kt[(size_t)t * RS + ch]), ks[ch], kz[ch], qmax);
            if (do_v_and_sinks) {
                int j = ch / p.Gv;
                vc = code_exact(__half2float(Vt[(size_t)t * RS + ch]), vs[t * p.NGv + j], vz[t * p.NGv + j], qmax);
            }
        }
        kcode[idx] = (uint8_t)kc;
        vcode[idx] = (uint8_t)vc;
    }
    __syncthreads();

    // pack: the group's tiles are contiguous in memory; one thread per 32-bit word
    const int tile_words = p.tile_bytes / 4, n_tiles = G / KVSINK_TILE;
    uint32_t *kout = (uint32_t *)(c.k_codes + (size_t)unit * p.max_seq * p.row_bytes + (size_t)(p0 / KVSINK_TILE) * p.tile_bytes);
    uint32_t *vout = (uint32_t *)(c.v_codes + (size_t)unit * p.max_seq * p.row_bytes + (size_t)(p0 / KVSINK_TILE) * p.tile_bytes);
    for (int idx = tid; idx < n_tiles * tile_words; idx += QG_THREADS) {
        int tile = idx / tile_words, word = idx % tile_words;
        const uint8_t *kc = kcode + (size_t)tile * KVSINK_TILE * D;
        kout[idx] = assemble_word(p.bits, D, word, [&](int m, int row, int col) { return (uint32_t)kc[row * D + 16 * m + col]; });
        if (do_v_and_sinks) {
            const uint8_t *vc = vcode + (size_t)tile * KVSINK_TILE * D;
            vout[idx] = assemble_word(p.bits, D, word, [&](int m, int row, int col) { return (uint32_t)vc[col * D + 16 * m + row]; });
        }
    }

    // sink rows: exact fp16 copies into the side buffer at the rank of their position
    if (do_v_and_sinks) {
        const int count = min(c.sink_count[b], p.cap);
        for (int t = 0; t < G; ++t) {
            if (!flag[t]) continue;
            int slot = find_slot(c.sink_pos + (size_t)b * p.cap, count, p0 + t);
            if (slot < 0) {
                if (tid == 0) atomicOr(c.status, KVSINK_STATUS_SINK_MISMATCH);
                continue;
            }
            __half *dk = (__half *)c.sink_k + ((size_t)unit * p.cap + slot) * D;
            __half *dv = (__half *)c.sink_v + ((size_t)unit * p.cap + slot) * D;
            for (int ch = tid; ch < chunks; ch += QG_THREADS) {
                *(uint4 *)(dk + ch * 8) = *(const uint4 *)(Kt + (size_t)t * RS + ch * 8);
                *(uint4 *)(dv + ch * 8) = *(const uint4 *)(Vt + (size_t)t * RS + ch * 8);
            }
        }
    }
}

static size_t groups_smem_bytes(const Params &p)
{
    size_t RS = p.D + 8;
    return 2 * (size_t)p.G * RS * 2 + 2 * (size_t)p.G * p.D + 2 * (size_t)p.D * 4 + 2 * (size_t)p.G * p.NGv * 4 + p.G + 16;
}

int launch_quantize_groups(const Params &p, const kvsink_cache &c, const __half *k_src, const __half *v_src, int first_token,
                           int n_groups, int64_t sb, int64_t sh, int64_t stt, bool do_v_and_sinks, const AppendEdges *edges, cudaStream_t st)
{
    if (n_groups <= 0) return KVSINK_OK;
    size_t smem = groups_smem_bytes(p);
    if (smem > 227 * 1024) return KVSINK_ERR_UNSUPPORTED;
    if (!allow_smem(quantize_groups_kernel, smem)) return KVSINK_ERR_CUDA;
    if (edges)
        if (const int rc = launch_append_edges(p, c, *edges, st)) return rc;
    dim3 grid(n_groups, p.Hkv, p.B);
    note_launch();
    quantize_groups_kernel<<<grid, QG_THREADS, smem, st>>>(p, c, k_src, v_src, first_token, sb, sh, stt, do_v_and_sinks ? 1 : 0);
    return cudaGetLastError() == cudaSuccess ? KVSINK_OK : KVSINK_ERR_CUDA;
}

// ---------------------------------------------------------------------------------------------------------
// Single tokens (decode-time append, and the remainder of a prefill that does not fill a group): values are
// quantized per token and inserted into their tile, keys go to the fp16 tail, sink rows to the side buffer.
// One block per (tile touched, KV head, sequence).
// ---------------------------------------------------------------------------------------------------------
constexpr int QT_THREADS = 128;

__global__ void __launch_bounds__(QT_THREADS)
quantize_tokens_kernel(Params p, kvsink_cache c, const __half *__restrict__ k_src, const __half *__restrict__ v_src, int src_offset,
                       int first_token, int n_tokens, int64_t sb, int64_t sh, int64_t stt)
{
    __shared__ uint8_t vcode[KVSINK_TILE * 128];
    __shared__ uint8_t present[KVSINK_TILE];
    const int D = p.D, G = p.G;
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

    const int cpl = D / 32;   // channels per lane (2 or 4)
    for (int pos = t_lo + warp; pos < t_hi; pos += QT_THREADS / 32) {
        const int64_t src = b * sb + h * sh + (int64_t)(src_offset + pos - first_token) * stt;
        const bool sink = mask_bit(bm, pos);
        float x[4];
        __half kx[4], vx[4];
        for (int e = 0; e < cpl; ++e) {
            vx[e] = v_src[src + lane * cpl + e];
            x[e] = __half2float(vx[e]);
            kx[e] = k_src[src + lane * cpl + e];
        }
        // key row -> tail
        __half *tail = (__half *)c.k_tail + ((size_t)unit * G + pos % G) * D;
        for (int e = 0; e < cpl; ++e) tail[lane * cpl + e] = kx[e];
        if (sink) {
            const int count = min(c.sink_count[b], p.cap);
            int slot = find_slot(c.sink_pos + (size_t)b * p.cap, count, pos);
            if (slot < 0) {
                if (lane == 0) atomicOr(c.status, KVSINK_STATUS_SINK_MISMATCH);
            } else {
                __half *dk = (__half *)c.sink_k + ((size_t)unit * p.cap + slot) * D;
                __half *dv = (__half *)c.sink_v + ((size_t)unit * p.cap + slot) * D;
                for (int e = 0; e < cpl; ++e) {
                    dk[lane * cpl + e] = kx[e];
                    dv[lane * cpl + e] = vx[e];
                }
            }
        }
        // value row: min / max over the lanes of each channel group
        float mn = x[0], mx = x[0];
        for (int e = 1; e < cpl; ++e) { mn = fminf(mn, x[e]); mx = fmaxf(mx, x[e]); }
        const int lanes_per_group = p.Gv / cpl;
        for (int o = 1; o < lanes_per_group; o <<= 1) {
            mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        float s, z;
        group_params(!sink, mn, mx, qmax, &s, &z);
        const int j = lane / lanes_per_group;
        if (lane % lanes_per_group == 0) {
            size_t o = ((size_t)unit * p.max_seq + pos) * p.NGv + j;
            c.v_scale[o] = s;
            c.v_zero[o] = z;
        }
        for (int e = 0; e < cpl; ++e)
            vcode[(pos % KVSINK_TILE) * D + lane * cpl + e] = sink ? 0 : (uint8_t)code_exact(x[e], s, z, qmax);
    }
    __syncthreads();

    // insert the new tokens' fields into the tile; fields of other tokens keep their bits
    const int tile_words = p.tile_bytes / 4;
    uint32_t *vout = (uint32_t *)(c.v_codes + (size_t)unit * p.max_seq * p.row_bytes + (size_t)tile * p.tile_bytes);
    const bool fresh = (t_lo % KVSINK_TILE) == 0;   // no earlier token lives in this tile
    for (int word = tid; word < tile_words; word += QT_THREADS) {
        uint32_t keep = fresh ? 0u : vout[word];
        uint32_t fieldmask;
        const uint32_t newbits = assemble_word_masked(p.bits, D, word, [&](int m, int row, int col) {
            return present[col] ? (uint32_t)vcode[col * D + 16 * m + row] : 0x100u; }, &fieldmask);
        if (fieldmask || fresh) vout[word] = (keep & ~fieldmask) | newbits;   // a fresh tile is written whole
    }
}

// ---------------------------------------------------------------------------------------------------------
// One token per sequence (the decode-time append): one warp per (sequence, KV head).  The value row is coded and its
// fields go straight into the tile's words: every channel's field has its own place (lane, word, bit) in the tile, so
// the lanes clear and set their fields with word atomics and nothing but the token's own fields is touched.
// ---------------------------------------------------------------------------------------------------------
constexpr int QA_WARPS = 4;

__global__ void __launch_bounds__(32 * QA_WARPS)
append_one_kernel(Params p, kvsink_cache c, const __half *__restrict__ k_src, const __half *__restrict__ v_src, int src_token, int pos,
                  int64_t sb, int64_t sh, int64_t stt)
{
    const int D = p.D, G = p.G;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t unit = (int64_t)blockIdx.x * QA_WARPS + warp;
    pdl_wait();
    if (unit >= (int64_t)p.B * p.Hkv) return;
    if (!in_bounds(pos >= 0 && pos < p.max_seq, c.status)) return;
    const int b = (int)(unit / p.Hkv), h = (int)(unit % p.Hkv);
    const float qmax = (float)((1 << p.bits) - 1);
    const int cpl = D / 32;   // channels per lane (2 or 4)
    const int64_t src = b * sb + h * sh + (int64_t)src_token * stt;
    const bool sink = mask_bit(c.sink_bitmask + (size_t)b * p.mask_words, pos);
    float x[4];
    __half kx[4], vx[4];
    for (int e = 0; e < cpl; ++e) {
        vx[e] = v_src[src + lane * cpl + e];
        x[e] = __half2float(vx[e]);
        kx[e] = k_src[src + lane * cpl + e];
    }
    // key row -> tail
    __half *tail = (__half *)c.k_tail + ((size_t)unit * G + pos % G) * D;
    for (int e = 0; e < cpl; ++e) tail[lane * cpl + e] = kx[e];
    if (sink) {
        const int count = min(c.sink_count[b], p.cap);
        const int slot = find_slot(c.sink_pos + (size_t)b * p.cap, count, pos);
        if (slot < 0) {
            if (lane == 0) atomicOr(c.status, KVSINK_STATUS_SINK_MISMATCH);
        } else {
            __half *dk = (__half *)c.sink_k + ((size_t)unit * p.cap + slot) * D;
            __half *dv = (__half *)c.sink_v + ((size_t)unit * p.cap + slot) * D;
            for (int e = 0; e < cpl; ++e) {
                dk[lane * cpl + e] = kx[e];
                dv[lane * cpl + e] = vx[e];
            }
        }
    }
    // value row: min / max over the lanes of each channel group, parameters, codes
    float mn = x[0], mx = x[0];
    for (int e = 1; e < cpl; ++e) { mn = fminf(mn, x[e]); mx = fmaxf(mx, x[e]); }
    const int lanes_per_group = p.Gv / cpl;
    for (int o = 1; o < lanes_per_group; o <<= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    float s, z;
    group_params(!sink, mn, mx, qmax, &s, &z);
    if (lane % lanes_per_group == 0) {
        const size_t o = ((size_t)unit * p.max_seq + pos) * p.NGv + lane / lanes_per_group;
        c.v_scale[o] = s;
        c.v_zero[o] = z;
    }
    // the token's fields in its tile; a tile whose first token this is is written whole (zeros elsewhere)
    const int tile = pos / KVSINK_TILE, col = pos % KVSINK_TILE;
    uint32_t *vout = (uint32_t *)(c.v_codes + (size_t)unit * p.max_seq * p.row_bytes + (size_t)tile * p.tile_bytes);
    const bool fresh = col == 0;
    if (fresh) {
        for (int w = lane; w < p.tile_bytes / 4; w += 32) vout[w] = 0u;
        __syncwarp();
    }
    for (int e = 0; e < cpl; ++e) {
        const int ch = lane * cpl + e;
        set_field(vout, p.bits, D, ch >> 4, ch & 15, col, sink ? 0u : code_exact(x[e], s, z, qmax), fresh);
    }
}

// ---------------------------------------------------------------------------------------------------------
// The ragged edges of a chunk in one kernel: the tokens that complete (or extend) an open group, the flush of that group's
// keys, and the tokens behind the last whole group.  One block per (sequence, KV head, 64 channels) has the keys; one per tile
// touched the values.  Latency bound (a few rows per block), so it is one launch instead of three that wait for one another: a 2779-token
// chunk that starts inside a group, 5 x 8 units at 3 bit, had 12 us of head tokens and 7 us of flush before its whole groups.
// The head size and the bits are the kernel's own, so that the walk over a word's fields is straight code, and the rows of codes are padded, which puts
// the lanes of a quad into different banks (walk by run-time bits, rows of 64 and 128 bytes, loads one after the other, and now, us): that chunk 26.3
// and 25.1 (20.7 without its ends), its 27 head tokens alone 7.1 and 5.9, 10 x 32 units of them 18.2 and 15.3, 8 x 32 units, 2859 tokens
// from 1237, 2 bit, 94.7 and 90.2, 4 x 8 with 64 channels, 700 from 250, 4 bit, 16.5 and 14.5.
// ---------------------------------------------------------------------------------------------------------
constexpr int QE_THREADS = 256, QE_CH = 64, QE_SHARE = QE_THREADS / QE_CH, QE_CROW = QE_CH + 4, QE_MAX_G = 128;

struct EdgeShape {
    int head_first, head_n, flush;             // tokens inside the open group; whether they complete it
    int rem_first, rem_n, rem_src;             // tokens behind the last whole group (at a group boundary), offset of the first in the source
    int head_tiles;                            // tiles the head tokens touch
};

template <int D, int BITS>
__global__ void __launch_bounds__(QE_THREADS)
append_edges_kernel(Params p, kvsink_cache c, const __half *__restrict__ k_src, const __half *__restrict__ v_src, EdgeShape e, int64_t sb, int64_t sh,
                    int64_t stt)
{
    constexpr int VROW = D + 8;                // padded row of the values' codes: a quad's tokens lie in different banks
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ float part[QE_SHARE][2][QE_CH]; // keys: extremes of the row quarters; then scale, zero
    __shared__ uint8_t flag[QE_MAX_G];         // keys: sink flags of the open group; values: tokens of the tile that are new
    __shared__ uint8_t vcode[KVSINK_TILE * VROW];
    const int G = p.G, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int h = blockIdx.y, b = blockIdx.z;
    const int64_t unit = (int64_t)b * p.Hkv + h, src0 = b * sb + h * sh;
    const float qmax = (float)((1 << BITS) - 1);
    const uint32_t *bm = c.sink_bitmask + (size_t)b * p.mask_words;
    const int32_t *sink_pos = c.sink_pos + (size_t)b * p.cap;
    pdl_wait();
    pdl_release();        // the whole groups' kernel of the same call, which touches nothing this one writes, does not even wait
    if (!in_bounds(e.head_first >= 0 && e.head_first + e.head_n <= p.max_seq && (e.rem_n == 0 || e.rem_first + e.rem_n <= p.max_seq), c.status)) return;
    const int count = min(c.sink_count[b], p.cap);

    constexpr int slices = D / QE_CH;
    if ((int)blockIdx.x < slices) {            // ---- keys: a slice of 64 channels ----
        constexpr int CHUNKS = QE_CH / 8, RS = QE_CH + 8;
        const int c0 = (int)blockIdx.x * QE_CH, old = e.head_first % G;               // rows of the open group that the tail holds
        __half *tail = (__half *)c.k_tail + (size_t)unit * G * D + c0;
        const __half *src = k_src + src0 + c0;
        if (e.flush) {
            __half *Kt = (__half *)dyn;        // [G][RS]
            uint8_t *code = (uint8_t *)(Kt + (size_t)G * RS);                         // [G][QE_CROW]
            const int g0 = e.head_first - old;
            uint4 v[QE_MAX_G * CHUNKS / QE_THREADS];                                    // all of a thread's loads on their way at once
#pragma unroll
            for (int x = 0; x < QE_MAX_G * CHUNKS / QE_THREADS; ++x) {
                const int idx = tid + x * QE_THREADS, t = idx / CHUNKS, ch = (idx % CHUNKS) * 8;
                if (t < G) v[x] = *(const uint4 *)((t < old ? tail + (size_t)t * D : src + (int64_t)(t - old) * stt) + ch);
            }
            if (tid < G) flag[tid] = mask_bit(bm, g0 + tid) ? 1 : 0;
#pragma unroll
            for (int x = 0; x < QE_MAX_G * CHUNKS / QE_THREADS; ++x) {
                const int idx = tid + x * QE_THREADS, t = idx / CHUNKS, ch = (idx % CHUNKS) * 8;
                if (t < G) *(uint4 *)(Kt + (size_t)t * RS + ch) = v[x];
            }
            __syncthreads();
            // extremes per channel: four threads with a share of the rows each, then one thread per channel
            const int ch = tid % QE_CH, qt = tid / QE_CH;
            float mn = INFINITY, mx = -INFINITY;
#pragma unroll 4
            for (int t = qt; t < G; t += QE_SHARE) {
                const float x = __half2float(Kt[(size_t)t * RS + ch]);
                mn = flag[t] ? mn : fminf(mn, x);
                mx = flag[t] ? mx : fmaxf(mx, x);
            }
            part[qt][0][ch] = mn;
            part[qt][1][ch] = mx;
            __syncthreads();
            if (tid < QE_CH) {
                for (int i = 1; i < QE_SHARE; ++i) {
                    mn = fminf(mn, part[i][0][tid]);
                    mx = fmaxf(mx, part[i][1][tid]);
                }
                float s, z;
                group_params(mn <= mx, mn, mx, qmax, &s, &z);                          // no member: +inf, -inf
                part[0][0][tid] = s;
                part[0][1][tid] = z;
                const size_t o = ((size_t)unit * (p.max_seq / G) + g0 / G) * D + c0 + tid;
                c.k_scale[o] = s;
                c.k_zero[o] = z;
            }
            __syncthreads();
            const float s = part[0][0][ch], z = part[0][1][ch];
#pragma unroll 4
            for (int t = qt; t < G; t += QE_SHARE)
                code[t * QE_CROW + ch] = flag[t] ? 0 : (uint8_t)code_exact(__half2float(Kt[(size_t)t * RS + ch]), s, z, qmax);
            __syncthreads();
            // the slice's words: per tile and lane two words of a 2-bit section, four of a 4-bit one, one of the 3-bit high section
            uint32_t *out = (uint32_t *)(c.k_codes + (size_t)unit * p.max_seq * p.row_bytes + (size_t)(g0 / KVSINK_TILE) * p.tile_bytes);
            constexpr int tile_words = 8 * D * BITS / 16, lo_bits = BITS == 4 ? 4 : 2, fields = 16 / lo_bits, lo_words = BITS == 4 ? 4 : 2, n_lo = D * lo_bits / 64;
            for (int idx = tid; idx < G / KVSINK_TILE * 32 * BITS; idx += QE_THREADS) {
                const int ln = idx % 32, i = idx / 32 % BITS, tile = idx / (32 * BITS);                 // i and tile are a warp's
                const uint8_t *rows = code + tile * KVSINK_TILE * QE_CROW;
                uint32_t word = 0;
                int m, row, col;
                if (BITS != 3 || i < lo_words) {
#pragma unroll
                    for (int k = 0; k < fields; ++k)
#pragma unroll
                        for (int x = 0; x < 2; ++x) {
                            slot_to_elem(ln, fields * i + k, x, &m, &row, &col);
                            word |= (rows[row * QE_CROW + 16 * m + col] & ((1u << lo_bits) - 1u)) << (16 * x + lo_bits * k);
                        }
                    out[tile * tile_words + section_word_offset(n_lo, ln, lo_words * (int)blockIdx.x + i)] = word;
                } else {
#pragma unroll
                    for (int k = 0; k < 16; ++k)
#pragma unroll
                        for (int x = 0; x < 2; ++x) {
                            slot_to_elem(ln, k, x, &m, &row, &col);
                            const int w = k >> 3, f = k & 7;
                            word |= (uint32_t)((rows[row * QE_CROW + 16 * m + col] >> 2) & 1) << (16 * x + 4 * (f >> 1) + 2 * (1 - w) + (f & 1));
                        }
                    out[tile * tile_words + 32 * n_lo + section_word_offset(D / 64, ln, (int)blockIdx.x)] = word;
                }
            }
        }
        // rows to the tail, as if token by token: those behind the last whole group lie over a completed group's
        for (int idx = tid; idx < e.head_n * CHUNKS; idx += QE_THREADS) {
            const int t = idx / CHUNKS, ch = (idx % CHUNKS) * 8;
            if (!e.flush || old + t >= e.rem_n) *(uint4 *)(tail + (size_t)(old + t) * D + ch) = __ldg((const uint4 *)(src + (int64_t)t * stt + ch));
        }
        for (int idx = tid; idx < e.rem_n * CHUNKS; idx += QE_THREADS) {
            const int t = idx / CHUNKS, ch = (idx % CHUNKS) * 8;
            *(uint4 *)(tail + (size_t)t * D + ch) = __ldg((const uint4 *)(src + (int64_t)(e.rem_src + t) * stt + ch));
        }
        for (int i = warp; i < e.head_n + e.rem_n; i += QE_THREADS / 32) {            // exact rows of sink tokens
            const int pos = i < e.head_n ? e.head_first + i : e.rem_first + i - e.head_n;
            if (!mask_bit(bm, pos)) continue;
            const int slot = find_slot(sink_pos, count, pos);
            if (slot < 0) continue;                                                   // the values' block reports it
            const __half *row = src + (int64_t)(i < e.head_n ? i : e.rem_src + i - e.head_n) * stt;
            __half *dk = (__half *)c.sink_k + ((size_t)unit * p.cap + slot) * D + c0;
            if (lane < CHUNKS) *(uint4 *)(dk + lane * 8) = __ldg((const uint4 *)(row + lane * 8));
        }
        return;
    }

    // ---- values of one tile ----
    const int vt = (int)blockIdx.x - slices;
    const bool head = vt < e.head_tiles;
    const int first = head ? e.head_first : e.rem_first, n = head ? e.head_n : e.rem_n, offset = head ? 0 : e.rem_src;
    const int tile = first / KVSINK_TILE + vt - (head ? 0 : e.head_tiles);
    const int t_lo = max(first, tile * KVSINK_TILE), t_hi = min(first + n, (tile + 1) * KVSINK_TILE);
    if (tid < KVSINK_TILE) flag[tid] = (tile * KVSINK_TILE + tid >= t_lo && tile * KVSINK_TILE + tid < t_hi) ? 1 : 0;
    constexpr int cpl = D / 32;   // channels per lane (2 or 4)
    for (int pos = t_lo + warp; pos < t_hi; pos += QE_THREADS / 32) {
        const __half *row = v_src + src0 + (int64_t)(offset + pos - first) * stt + lane * cpl;
        __half2 v2[2];
        v2[0] = *(const __half2 *)row;
        v2[1] = cpl == 4 ? *(const __half2 *)(row + 2) : v2[0];
        const float2 lo = __half22float2(v2[0]), hi = __half22float2(v2[1]);
        const float x[4] = {lo.x, lo.y, hi.x, hi.y};
        const bool sink = mask_bit(bm, pos);
        if (sink) {
            const int slot = find_slot(sink_pos, count, pos);
            if (slot < 0) {
                if (lane == 0) atomicOr(c.status, KVSINK_STATUS_SINK_MISMATCH);
            } else {
                __half2 *dv = (__half2 *)((__half *)c.sink_v + ((size_t)unit * p.cap + slot) * D + lane * cpl);
                dv[0] = v2[0];
                if (cpl == 4) dv[1] = v2[1];
            }
        }
        float mn = fminf(x[0], x[1]), mx = fmaxf(x[0], x[1]);
        mn = fminf(mn, fminf(x[2], x[3]));
        mx = fmaxf(mx, fmaxf(x[2], x[3]));
        const int lanes_per_group = p.Gv / cpl;
        for (int o = 1; o < lanes_per_group; o <<= 1) {
            mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        float s, z;
        group_params(!sink, mn, mx, qmax, &s, &z);
        if (lane % lanes_per_group == 0) {
            const size_t o = ((size_t)unit * p.max_seq + pos) * p.NGv + lane / lanes_per_group;
            c.v_scale[o] = s;
            c.v_zero[o] = z;
        }
        for (int i = 0; i < cpl; ++i) vcode[(pos % KVSINK_TILE) * VROW + lane * cpl + i] = sink ? 0 : (uint8_t)code_exact(x[i], s, z, qmax);
    }
    __syncthreads();
    // the new tokens' fields; fields of other tokens keep their bits, a fresh tile is written whole
    constexpr int tile_words = 8 * D * BITS / 16;
    uint32_t *vout = (uint32_t *)(c.v_codes + (size_t)unit * p.max_seq * p.row_bytes + (size_t)tile * p.tile_bytes);
    const bool fresh = t_lo % KVSINK_TILE == 0;
    for (int word = tid; word < tile_words; word += QE_THREADS) {
        const uint32_t keep = fresh ? 0u : vout[word];
        uint32_t fieldmask;
        const uint32_t newbits = assemble_word_masked(BITS, D, word, [&](int m, int row, int col) {
            return flag[col] ? (uint32_t)vcode[col * VROW + 16 * m + row] : 0x100u; }, &fieldmask);
        if (fieldmask || fresh) vout[word] = (keep & ~fieldmask) | newbits;
    }
}

// Groups of more than 128 tokens keep the kernels that go token by token (the group would not fit a block's shared memory).
int launch_append_edges(const Params &p, const kvsink_cache &c, const AppendEdges &a, cudaStream_t st)
{
    if (p.G > QE_MAX_G) return KVSINK_ERR_UNSUPPORTED;
    auto tiles = [](int first, int n) { return n > 0 ? (first + n - 1) / KVSINK_TILE - first / KVSINK_TILE + 1 : 0; };
    EdgeShape e;
    e.head_first = a.head_first;
    e.head_n = a.head_n;
    e.flush = a.head_n > 0 && (a.head_first + a.head_n) % p.G == 0;
    e.rem_first = a.head_first + a.rem_src;
    e.rem_n = a.rem_n;
    e.rem_src = a.rem_src;
    e.head_tiles = tiles(a.head_first, a.head_n);
    const dim3 grid(p.D / QE_CH + e.head_tiles + tiles(e.rem_first, e.rem_n), p.Hkv, p.B);
    const size_t smem = e.flush ? (size_t)p.G * ((QE_CH + 8) * 2 + QE_CROW) : 0;
    const auto kernel = p.D == 128 ? (p.bits == 2 ? append_edges_kernel<128, 2> : p.bits == 3 ? append_edges_kernel<128, 3> : append_edges_kernel<128, 4>)
                                   : (p.bits == 2 ? append_edges_kernel<64, 2> : append_edges_kernel<64, 4>);
    return launch_pdl(kernel, grid, dim3(QE_THREADS), smem, st, p, c, a.k_src, a.v_src, e, a.sb, a.sh, a.stt) == cudaSuccess ? KVSINK_OK : KVSINK_ERR_CUDA;
}

int launch_quantize_tokens(const Params &p, const kvsink_cache &c, const __half *k_src, const __half *v_src, int src_offset,
                           int first_token, int n_tokens, int64_t sb, int64_t sh, int64_t stt, cudaStream_t st)
{
    if (n_tokens <= 0) return KVSINK_OK;
    if (n_tokens == 1) {
        const long units = (long)p.B * p.Hkv;
        return launch_pdl(append_one_kernel, dim3((unsigned)((units + QA_WARPS - 1) / QA_WARPS)), dim3(32 * QA_WARPS), 0, st, p, c, k_src, v_src,
                          src_offset, first_token, sb, sh, stt) == cudaSuccess ? KVSINK_OK : KVSINK_ERR_CUDA;
    }
    int tiles = (first_token + n_tokens - 1) / KVSINK_TILE - first_token / KVSINK_TILE + 1;
    dim3 grid(tiles, p.Hkv, p.B);
    return launch_pdl(quantize_tokens_kernel, grid, dim3(QT_THREADS), 0, st, p, c, k_src, v_src, src_offset, first_token, n_tokens, sb, sh,
                      stt) == cudaSuccess ? KVSINK_OK : KVSINK_ERR_CUDA;
}

}  // namespace kvsink
