// Decode attention, host side: split heuristic, merge of the sequence splits, dispatch over the code width, and the
// entry point that keeps its scratch inside the library image.  The split kernel itself is in decode_kernel.cuh.
#include <mutex>

#include "common.cuh"

namespace kvsink {

// Merge of the sequence splits (where the splits of a unit are not launched as a cluster): one block per (sequence, query head).  Thread
// (c, sl) folds channels 2c, 2c + 1 of the records sl, sl + slices, ..., and the slices are combined in a fixed order (bit-reproducible).
// What bounds it is the latency of reading records that are in L2: a thread asks for everything it needs of up to eight records at once
// (64 splits are one round), where two passes over the records, first the maxima, waited some eight times: 3.8 -> 2.3 us for 32 rows of 64
// splits.  Few splits take few slices: eight slices for 18 records were 0.4 us slower than four.
constexpr int MERGE_SLICES = 8, MERGE_BATCH = 8;

__global__ void __launch_bounds__(64 * MERGE_SLICES) decode_merge_kernel(const float *__restrict__ part_ws, int nsplit, int D, float *__restrict__ out, float *__restrict__ lse)
{
    __shared__ float2 sh_acc[MERGE_SLICES][64];
    __shared__ float sh_m[MERGE_SLICES], sh_l[MERGE_SLICES];
    const int PS = D + 2;
    const size_t oq = blockIdx.x;
    const int c = threadIdx.x, sl = threadIdx.y, slices = blockDim.y;
    const float *base = part_ws + oq * nsplit * PS;
    // launched with programmatic stream serialization: the blocks may start while the split kernel drains, and wait
    // here until all of it has completed and its records are visible
    pdl_wait();
    float M = M_INIT, L = 0.f;
    float2 acc = make_float2(0.f, 0.f);
    for (int s0 = sl; s0 < nsplit; s0 += slices * MERGE_BATCH) {
        float m[MERGE_BATCH], l[MERGE_BATCH];
        float2 a[MERGE_BATCH];
#pragma unroll
        for (int k = 0; k < MERGE_BATCH; ++k) {
            const int s = s0 + k * slices;
            const float *r = base + (size_t)s * PS;      // 8-byte aligned: PS is even
            const bool in = s < nsplit;
            m[k] = in ? r[D] : M_INIT;
            l[k] = in ? r[D + 1] : 0.f;
            a[k] = in ? *(const float2 *)(r + 2 * c) : make_float2(0.f, 0.f);
        }
        float top = M;
#pragma unroll
        for (int k = 0; k < MERGE_BATCH; ++k) top = fmaxf(top, m[k]);
        const float f0 = ex2(M - top);
        L *= f0; acc.x *= f0; acc.y *= f0;
#pragma unroll
        for (int k = 0; k < MERGE_BATCH; ++k) {
            const float f = ex2(m[k] - top);
            L = fmaf(l[k], f, L);
            acc.x = fmaf(a[k].x, f, acc.x);
            acc.y = fmaf(a[k].y, f, acc.y);
        }
        M = top;
    }
    sh_acc[sl][c] = acc;
    if (c == 0) { sh_m[sl] = M; sh_l[sl] = L; }
    __syncthreads();
    if (sl != 0) return;
    float Mt = M_INIT, Lt = 0.f;
    float2 at = make_float2(0.f, 0.f);
    for (int i = 0; i < slices; ++i) Mt = fmaxf(Mt, sh_m[i]);
    for (int i = 0; i < slices; ++i) {
        const float f = ex2(sh_m[i] - Mt);
        const float2 v = sh_acc[i][c];
        at.x = fmaf(v.x, f, at.x);
        at.y = fmaf(v.y, f, at.y);
        Lt = fmaf(sh_l[i], f, Lt);
    }
    *(float2 *)(out + oq * D + 2 * c) = Lt > 0.f ? make_float2(at.x / Lt, at.y / Lt) : make_float2(0.f, 0.f);      // out is aligned to 16 bytes
    if (lse && c == 0) lse[oq] = Lt > 0.f ? (Mt + log2f(Lt)) * 0.6931471805599453f : -INFINITY;
}

int launch_decode_merge(const float *ws, int nsplit, int D, int n_rows, float *out, float *lse, cudaStream_t st)
{
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_rows);
    cfg.blockDim = dim3(D / 2, nsplit <= 4 ? 2 : (nsplit <= 32 ? 4 : MERGE_SLICES));
    cfg.stream = st;
    cfg.attrs = pdl;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, decode_merge_kernel, ws, nsplit, D, out, lse) != cudaSuccess) return KVSINK_ERR_CUDA;
    note_launch();
    return KVSINK_OK;
}

// ---- host side ----
constexpr int DEC_SLOTS = 148 * 4;   // resident blocks the split heuristic plans for

int max_splits(const Params &p)
{
    const int qchunks = decode_qchunks(p);
    const long units = (long)p.B * p.Hkv * qchunks;
    long ns = (2L * DEC_SLOTS + units - 1) / units;
    const long mg = p.max_seq / p.G;
    if (ns > mg) ns = mg;
    return (int)(ns < 1 ? 1 : ns);
}

// Two and four bit: whole waves of resident blocks times the groups of a warp.  At three bit an SM's time goes with the number of
// blocks it gets in all (four resident ones run at full rate, two at three quarters of it, by measurement), each with the
// groups of a warp and about one group's time for its prologue and epilogue.  Measured, microseconds, this rule's choice first and
// other split counts behind it: 16 x 32 units of 8101 tokens 2: 129 (1: 143, 3: 134; 7 blocks on the fullest SM instead of 4 of
// twice the size); 8 x 32 of 4096 4: 39 (1: 47, 2: 42); 1 x 8 of 131072 with four heads 74: 54 (37: 59, 64: 57, 96: 64);
// 4 x 8 of 30000 with four heads 18: 50 (8: 70, 12: 57, 37: 55); 37 x 8 of 9000 2: 85 (1: 98, 3: 87).
int choose_splits(const Params &p, int n_groups)
{
    const int qchunks = decode_qchunks(p);
    const long units = (long)p.B * p.Hkv * qchunks;
    const int ns_max = max_splits(p) < n_groups ? max_splits(p) : (n_groups > 0 ? n_groups : 1);
    int best = 1;
    double best_cost = 1e300;
    for (int ns = 1; ns <= ns_max; ++ns) {
        const int per_block = (n_groups + ns - 1) / ns;
        const int per_warp = (per_block + DEC_WARPS - 1) / DEC_WARPS;
        double cost;
        if (p.bits == 3) {
            static const double rate[5] = {1.0, 0.4, 0.75, 0.93, 1.0};
            const long on_sm = (units * ns + 147) / 148;
            cost = (double)on_sm / rate[on_sm < 4 ? on_sm : 4] * ((double)per_block / DEC_WARPS + 0.93) + 0.02 * ns;   // the last term: one more record to merge
        } else {
            const long waves = (units * ns + DEC_SLOTS - 1) / DEC_SLOTS;
            cost = (double)waves * (per_warp + 0.5);
        }
        if (cost < best_cost - 1e-9) { best_cost = cost; best = ns; }
    }
    // A grid that leaves most SMs without a block: a few splits more, in one cluster, bring each warp's chain down to a group or two (decode
    // alone, us, the sum above's choice and eight: 16 units of 1500 tokens, four heads each, 12.0 and 9.4, eight heads 16.0 and 13.3; 8 units
    // of 256, head size 64, 6.3 and 5.3; 32 of 500, four, 7.5 and 7.0).
    const int few = (int)(148 / units < 8 ? 148 / units : 8);
    if (best < few && best < ns_max) best = few < ns_max ? few : ns_max;
    return best;
}

size_t decode_workspace_bytes(const Params &p)
{
    return (size_t)p.B * p.Hq * max_splits(p) * (p.D + 2) * sizeof(float) + 16;
}

int launch_decode(const Params &p, const kvsink_cache &c, const kvsink_static_params *cal, int mode, const __half *q, float *out, float *lse, void *workspace,
                  size_t workspace_bytes, cudaStream_t st)
{
    if (workspace_bytes < decode_workspace_bytes(p)) return KVSINK_ERR_WORKSPACE;
    float *ws = (float *)workspace;
    if (p.bits == 2) return launch_decode_b2(p, c, cal, mode, q, out, lse, ws, st);
    if (p.bits == 3) return launch_decode_b3(p, c, cal, mode, q, out, lse, ws, st);
    if (p.bits == 4) return launch_decode_b4(p, c, cal, mode, q, out, lse, ws, st);
    return KVSINK_ERR_UNSUPPORTED;
}

// ---------------------------------------------------------------------------------------------------------
// Decode attention without caller-provided scratch: the split partials live in a fixed array inside the library
// image.  Every GPU that loads the library holds these KVSINK_STATIC_SCRATCH_BYTES until the process exits.
// ---------------------------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_decode_scratch[KVSINK_STATIC_SCRATCH_BYTES];

// In host code `g_decode_scratch` is only a handle for the runtime, not a device address; the address is looked
// up once per device (with that device current) and cached.
static void *g_scratch_ptr[64];
static bool g_scratch_known[64];
static std::mutex g_scratch_mutex;

int launch_decode_static(const Params &p, const kvsink_cache &c, const __half *q, float *out, float *lse, cudaStream_t st)
{
    if (decode_workspace_bytes(p) > (size_t)KVSINK_STATIC_SCRATCH_BYTES) return KVSINK_ERR_STATIC_SCRATCH;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return KVSINK_ERR_CUDA;
    std::lock_guard<std::mutex> guard(g_scratch_mutex);
    if (!g_scratch_known[dev]) {
        void *ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_decode_scratch) != cudaSuccess || ptr == nullptr) return KVSINK_ERR_CUDA;
        g_scratch_ptr[dev] = ptr;
        g_scratch_known[dev] = true;
    }
    // No clearing is needed: the split kernel writes every partial record the merge kernel reads.
    return launch_decode(p, c, nullptr, 0, q, out, lse, g_scratch_ptr[dev], (size_t)KVSINK_STATIC_SCRATCH_BYTES, st);
}

}  // namespace kvsink
