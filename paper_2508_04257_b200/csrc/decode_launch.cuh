// Launches of the decode kernels, included once per code width.
#pragma once
#include "decode_kernel.cuh"
#include "decode_few.cuh"
#include "decode_one.cuh"

namespace kvsink {

// ---- launch: one instantiation per (bits, head size, value groups per row, chunk size, key-side variant) ----
template <int BITS, int D, int NGV, int CT, bool PL, int I8 = 0, int PM = 0, int R = 0>
static int launch_decode_p(const Params &p, const kvsink_cache &c, const kvsink_static_params *cal, const __half *q, float *out, float *lse, float *ws,
                           cudaStream_t st)
{
    // the units the sequence is split in: key groups, or ring chunks when the parameters are static
    const int n_groups = PM != 0 ? (c.seq_len + CT * KVSINK_TILE - 1) / (CT * KVSINK_TILE) : c.seq_len / p.G;
    const kvsink_static_params sp = PM == 1 ? *cal : kvsink_static_params{nullptr, nullptr, nullptr, nullptr};
    const int nsplit = choose_splits(p, n_groups);
    const int gps = n_groups > 0 ? (n_groups + nsplit - 1) / nsplit : 0;
    const int qchunks = decode_qchunks(p);      // blocks per KV head; each serves up to NQMAX query heads
    constexpr int NQ = R ? R : (PL ? 4 : 8);
    if (qchunks * NQ < p.rep) return KVSINK_ERR_UNSUPPORTED;
    const size_t smem = DecodePlan<BITS, D, NGV, CT, NQ, PM == 2>::BYTES;
    const auto kern = [] {
        if constexpr (R == 1) return decode_one_kernel<BITS, NGV, CT, PM>;
        else if constexpr (R != 0) return decode_few_kernel<BITS, NGV, CT, PM, R>;
        else return decode_kernel<BITS, D, NGV, CT, PL, I8, PM>;
    }();
    cudaLaunchAttribute pdl[2];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    // up to eight splits (the portable cluster size): the splits of a unit are launched as one thread-block cluster and
    // merged inside the kernel through distributed shared memory, which saves the merge kernel's 2 to 3 us.  A cluster has to be placed
    // as a whole, though: where blocks by themselves would be three an SM some SMs get four, and what nearly fills the chip's 592 slots does
    // not fit in one round any more.  Decode alone, clusters and none, us: eights, 320 blocks, 40 units of 8000 tokens, 2 bit, 13.6 and 12.4;
    // sixes, 432, 72 of 6000, 15.7 and 13.9; fours, 384, 96 of 4000, 3 bit, 17.8 and 16.2, 96 of 8000, 4 bit, 35.9 and 26.1; 448, 112 of 16000, 2 bit,
    // 31.9 and 31.0; sixes, 576, 3 x 32 units of 4000, 20.3 and 14.4, 96 of 3000, 3 bit, 19.7 and 14.8; threes, 576, 192 of 1500, 3 bit,
    // 19.0 and 14.4.  512 blocks leave no SM more than it would have: eights, 64 units of 8000, four heads, 2 bit, 21.1 and 23.2, fours, 128 of 4000,
    // 3 bit, 19.6 and 20.2, 128 of 8000, four heads, 4 bit, 45.0 and 46.3; 480 are even (threes, 160 of 3000, 3 bit, 19.1 and 19.3; sixes, 80 of
    // 6000, 2 bit, 15.8 and 15.1, with four heads 23.1 and 24.5).  Up to 296 blocks clusters stay.
    // Pairs, whose second block finds room anywhere, lose beyond a round only (20 x 32 of 3000 44.9 and 39.8;
    // 592 blocks, 37 x 8 of 9000, 66.5 and 67.6); at 3 bit up to some 256 KB a block (16 x 32 of 8192, 384 KB a block, 137 and 136).
    const int64_t blocks = (int64_t)nsplit * p.Hkv * qchunks * p.B;
    const int64_t block_bytes = (int64_t)gps * (PM != 0 ? CT * KVSINK_TILE : p.G) * 2 * p.row_bytes;
    bool cluster_merge = nsplit > 1 && nsplit <= 8 && (nsplit == 2 ? blocks <= 4 * 148 && (p.bits != 3 || block_bytes < 256 * 1024) : blocks <= 2 * 148 || (blocks > 480 && blocks <= 512));
    // up to 48 KB need no leave, which costs a call
    if (smem > 48 * 1024 && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return KVSINK_ERR_CUDA;
    for (;;) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(nsplit, p.Hkv * qchunks, p.B);
        cfg.blockDim = dim3(DEC_THREADS);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cfg.attrs = pdl;
        cfg.numAttrs = 1;
        if (cluster_merge) {
            pdl[1].id = cudaLaunchAttributeClusterDimension;
            pdl[1].val.clusterDim.x = nsplit;
            pdl[1].val.clusterDim.y = 1;
            pdl[1].val.clusterDim.z = 1;
            cfg.numAttrs = 2;
        }
        cudaError_t launched;
        if constexpr (R == 1) launched = cudaLaunchKernelEx(&cfg, kern, p, c, sp, q, out, lse, ws, nsplit, gps, (int)c.seq_len, (int)cluster_merge);
        else if constexpr (R != 0) launched = cudaLaunchKernelEx(&cfg, kern, p, c, sp, q, out, lse, ws, nsplit, gps, qchunks, (int)c.seq_len, (int)cluster_merge);
        else launched = cudaLaunchKernelEx(&cfg, kern, p, c, sp, q, out, lse, ws, nsplit, gps, qchunks, (int)c.seq_len, (int)cluster_merge, PrefillShape{0, 0, 0, 0, 0});
        if (launched == cudaSuccess) {
            note_launch();
            break;
        }
        (void)cudaGetLastError();
        if (!cluster_merge) return KVSINK_ERR_CUDA;
        cluster_merge = false;   // a cluster that cannot be placed: the same launch without one, merged by the second kernel
    }
    if (nsplit > 1 && !cluster_merge) return launch_decode_merge(ws, nsplit, D, p.B * p.Hq, out, lse, st);
    return KVSINK_OK;
}

// Prompt queries (the eight-column fp16 path): one block per eight (query token, query head) rows of a KV head.
template <int BITS, int D, int NGV, int CT>
static int launch_prefill_p(const Params &p, const kvsink_cache &c, const __half *q, const PrefillShape &pre, float *out, float *lse, cudaStream_t st)
{
    const size_t smem = DecodePlan<BITS, D, NGV, CT, 8>::BYTES;
    auto kern = decode_kernel<BITS, D, NGV, CT, false, (D == 128 && BITS != 3) ? 3 : 0, 0, true>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return KVSINK_ERR_CUDA;
    const long long blocks = ((long long)pre.T * p.rep + 7) / 8;
    if (blocks > 0x7fffffffLL) return KVSINK_ERR_UNSUPPORTED;
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks, p.Hkv, p.B);
    cfg.blockDim = dim3(DEC_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = pdl;
    cfg.numAttrs = 1;
    const kvsink_static_params none = {nullptr, nullptr, nullptr, nullptr};
    if (cudaLaunchKernelEx(&cfg, kern, p, c, none, q, out, lse, (float *)nullptr, 1, 0, (int)blocks, (int)c.seq_len, 0, pre) != cudaSuccess)
        return KVSINK_ERR_CUDA;
    note_launch();
    return KVSINK_OK;
}

template <int BITS, int D, int NGV>
static int launch_prefill_n(const Params &p, const kvsink_cache &c, const __half *q, const PrefillShape &pre, float *out, float *lse, cudaStream_t st)
{
    // several channel groups per row mean G = D / NGV tokens per group: only chunk sizes that divide such a group are built;
    // four groups per row take one tile per chunk (their parameter registers would spill otherwise)
    constexpr int TPG_MAX = NGV == 1 ? 4 : D / NGV / KVSINK_TILE;
    if constexpr (TPG_MAX % 4 == 0 && 4 * (2 * 128 * (D * BITS / 64) + 2 * 16 * NGV * 4) <= 4800)
        if ((p.G / KVSINK_TILE) % 4 == 0) return launch_prefill_p<BITS, D, NGV, 4>(p, c, q, pre, out, lse, st);
    if constexpr (TPG_MAX % 2 == 0 && NGV < 4)
        if ((p.G / KVSINK_TILE) % 2 == 0) return launch_prefill_p<BITS, D, NGV, 2>(p, c, q, pre, out, lse, st);
    return launch_prefill_p<BITS, D, NGV, 1>(p, c, q, pre, out, lse, st);
}

template <int BITS, int D>
static int launch_prefill_t(const Params &p, const kvsink_cache &c, const __half *q, const PrefillShape &pre, float *out, float *lse, cudaStream_t st)
{
    if (p.NGv == 1) return launch_prefill_n<BITS, D, 1>(p, c, q, pre, out, lse, st);
    if (p.NGv == 2) return launch_prefill_n<BITS, D, 2>(p, c, q, pre, out, lse, st);
    if (p.NGv == 4) return launch_prefill_n<BITS, D, 4>(p, c, q, pre, out, lse, st);
    return KVSINK_ERR_UNSUPPORTED;
}

template <int BITS>
static int launch_prefill_bits(const Params &p, const kvsink_cache &c, const __half *q, int T, int q_pos0, int64_t sb, int64_t sh, int64_t stt,
                               float *out, float *lse, cudaStream_t st)
{
    const PrefillShape pre = {T, q_pos0, sb, sh, stt};
    if (p.D == 128) return launch_prefill_t<BITS, 128>(p, c, q, pre, out, lse, st);
    if constexpr (BITS != 3)
        if (p.D == 64) return launch_prefill_t<BITS, 64>(p, c, q, pre, out, lse, st);
    return KVSINK_ERR_UNSUPPORTED;
}

template <int BITS, int D, int NGV, int CT, int PM>
static int launch_decode_c(const Params &p, const kvsink_cache &c, const kvsink_static_params *cal, const __half *q, float *out, float *lse, float *ws,
                           cudaStream_t st)
{
    // kernel by head size, code width and query heads per KV head; only the reachable ones are built
    if constexpr (D == 128) {
        if constexpr (PM == 2 && BITS == 3)
            if (p.rep > 1) return KVSINK_ERR_UNSUPPORTED;
        if constexpr (NGV < 4 || CT == 2) {
            if (p.rep == 1) return launch_decode_p<BITS, D, NGV, CT, true, 0, PM, 1>(p, c, cal, q, out, lse, ws, st);
            if (p.rep == 2) return launch_decode_p<BITS, D, NGV, CT, true, 0, PM, 2>(p, c, cal, q, out, lse, ws, st);
            // 2 bit with one channel group a row: as many instructions as with fp16 values, and more registers (8 x 8 units of 16000 tokens,
            // static parameters, 34.0 and 32.1 us; of 8000 tokens, per-token keys, 30.1 and 27.8)
            if constexpr (BITS == 2 && NGV == 1) {
                if (p.rep <= 4) return launch_decode_p<BITS, D, NGV, CT, true, 2, PM>(p, c, cal, q, out, lse, ws, st);
            } else {
                if (p.rep <= 4 || BITS == 3) return launch_decode_p<BITS, D, NGV, CT, true, 0, PM, 4>(p, c, cal, q, out, lse, ws, st);
            }
        }
        if constexpr (PM != 2 && BITS != 3 && (NGV < 4 || CT == 1)) return launch_decode_p<BITS, D, NGV, CT, false, 3, PM>(p, c, cal, q, out, lse, ws, st);
        return KVSINK_ERR_UNSUPPORTED;           // per-token keys: at most four query heads per KV head
    } else {
        if (p.rep <= 4) return launch_decode_p<BITS, D, NGV, CT, true, 0, PM>(p, c, cal, q, out, lse, ws, st);
        return launch_decode_p<BITS, D, NGV, CT, false, 0, PM>(p, c, cal, q, out, lse, ws, st);
    }
}

template <int BITS, int D, int NGV, int PM>
static int launch_decode_n(const Params &p, const kvsink_cache &c, const kvsink_static_params *cal, const __half *q, float *out, float *lse, float *ws,
                           cudaStream_t st)
{
    // ring chunks of four tiles where a key group divides into them and two slots of that size stay below ~9 KB per
    // warp, else of two tiles (G a multiple of 32), else of one
    // several channel groups per row mean G = D / NGV tokens per group: only chunk sizes that divide such a group are built;
    // four groups per row take one tile per chunk (their parameter registers would spill otherwise)
    constexpr int TPG_MAX = NGV == 1 ? 4 : D / NGV / KVSINK_TILE;
    if constexpr (TPG_MAX % 4 == 0 && 4 * (2 * 128 * (D * BITS / 64) + (PM == 2 ? 4 : 2) * 16 * NGV * 4) <= (PM == 2 ? 5200 : 4800))
        if ((p.G / KVSINK_TILE) % 4 == 0) return launch_decode_c<BITS, D, NGV, 4, PM>(p, c, cal, q, out, lse, ws, st);
    if constexpr (TPG_MAX % 2 == 0 && NGV < 4)
        if ((p.G / KVSINK_TILE) % 2 == 0) return launch_decode_c<BITS, D, NGV, 2, PM>(p, c, cal, q, out, lse, ws, st);
    if constexpr (NGV == 4 && D == 128)      // up to four heads (3 bit: always) a lane keeps the parameters of few tokens
        if (p.rep <= 4 || BITS == 3) return launch_decode_c<BITS, D, NGV, 2, PM>(p, c, cal, q, out, lse, ws, st);
    return launch_decode_c<BITS, D, NGV, 1, PM>(p, c, cal, q, out, lse, ws, st);
}

template <int BITS, int D, int PM>
static int launch_decode_t(const Params &p, const kvsink_cache &c, const kvsink_static_params *cal, const __half *q, float *out, float *lse, float *ws,
                           cudaStream_t st)
{
    if (p.NGv == 1) return launch_decode_n<BITS, D, 1, PM>(p, c, cal, q, out, lse, ws, st);
    if constexpr (PM != 2 || BITS != 3)
        if (p.NGv == 2) return launch_decode_n<BITS, D, 2, PM>(p, c, cal, q, out, lse, ws, st);
    if constexpr (PM == 0)
        if (p.NGv == 4) return launch_decode_n<BITS, D, 4, PM>(p, c, cal, q, out, lse, ws, st);
    return KVSINK_ERR_UNSUPPORTED;
}

// Dispatch over head size for one code width; each width is compiled in a translation unit of its own.  mode 0: dynamic
// per-channel key parameters (`cal` null); 1: static parameters `cal`; 2: per-token key parameters.  Modes 1 and 2 are
// built for head size 128 with one or two channel groups per row; mode 2 for at most four query heads per KV head
// (3 bit: one, with one channel group).
template <int BITS>
static int launch_decode_bits(const Params &p, const kvsink_cache &c, const kvsink_static_params *cal, int mode, const __half *q, float *out,
                              float *lse, float *ws, cudaStream_t st)
{
    if (mode == 2) return p.D == 128 ? launch_decode_t<BITS, 128, 2>(p, c, cal, q, out, lse, ws, st) : KVSINK_ERR_UNSUPPORTED;
    if (mode == 1) return p.D == 128 && cal ? launch_decode_t<BITS, 128, 1>(p, c, cal, q, out, lse, ws, st) : KVSINK_ERR_UNSUPPORTED;
    if (p.D == 128) return launch_decode_t<BITS, 128, 0>(p, c, cal, q, out, lse, ws, st);
    if constexpr (BITS != 3)
        if (p.D == 64) return launch_decode_t<BITS, 64, 0>(p, c, cal, q, out, lse, ws, st);
    return KVSINK_ERR_UNSUPPORTED;
}

}  // namespace kvsink
