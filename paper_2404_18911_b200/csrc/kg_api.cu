// Host side of the C ABI declared in include/kangaroo.h: arena layout, synthetic weight fill,
// launches of the persistent decode kernel, small result copies.  No device allocation anywhere.
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/kangaroo.h"
#include "kg_engine.cuh"
#include "kg_prefill.cuh"

using namespace kg;

// ------------------------------------------------------------------------------------ generator
// Counter-based generator, implemented here independently of the host-side test generator:
//   base = mix(mix(seed) + tid); u = mix(base + i); g = bytesum(u) - 1020; x = float(g) * scale.
// mix is the SplitMix64 output function (Steele, Lea, Flood).
namespace {

__host__ __device__ inline uint64_t mix64(uint64_t z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
inline uint64_t stream_base(uint64_t seed, uint64_t tid) { return mix64(mix64(seed) + tid); }
inline float gen_scale(double std_) { return (float)(std_ / std::sqrt(43690.0)); }

__device__ __forceinline__ float gen_value(uint64_t base, uint64_t i, float scale) {
    const uint64_t u = mix64(base + i);
    const unsigned lo = (unsigned)u, hi = (unsigned)(u >> 32);
    // byte sum via two SIMD-in-register adds
    const unsigned s2 = (lo & 0x00ff00ffu) + ((lo >> 8) & 0x00ff00ffu) + (hi & 0x00ff00ffu) + ((hi >> 8) & 0x00ff00ffu);
    const int g = (int)((s2 & 0xffffu) + (s2 >> 16)) - 1020;
    return __fmul_rn((float)g, scale);
}

template <typename WT>
__global__ void fill_matrix_kernel(WT* out, uint64_t base, uint64_t count, float scale) {
    // 16 bytes of neighbouring values per thread (out is 16-byte aligned)
    constexpr int N = 16 / sizeof(WT);
    const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < count / N; j += step) {
        alignas(16) WT v[N];
#pragma unroll
        for (int k = 0; k < N; ++k) v[k] = float_to_wt<WT>(gen_value(base, j * N + k, scale));
        *reinterpret_cast<uint4*>(out + j * N) = *reinterpret_cast<const uint4*>(v);
    }
    if (blockIdx.x == 0 && threadIdx.x < count % N) { const uint64_t i = count / N * N + threadIdx.x; out[i] = float_to_wt<WT>(gen_value(base, i, scale)); }
}
__global__ void fill_gain_kernel(float* out, uint64_t base, int count, float scale) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        out[i] = __fadd_rn(1.0f, gen_value(base, (uint64_t)i, scale));
}
__global__ void fill_f32_kernel(float* out, uint64_t base, uint64_t count, float scale) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (uint64_t)gridDim.x * blockDim.x)
        out[i] = gen_value(base, i, scale);
}
// KV cache entries for positions [0, T): element index (pos*H + head)*hd + e of the stream.
template <typename WT>
__global__ void fill_cache_kernel(WT* cache, const int* page_table, uint64_t base, int T, int H, int hd, int ps, float scale) {
    const uint64_t count = (uint64_t)T * H * hd;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (uint64_t)gridDim.x * blockDim.x) {
        const int e = (int)(i % hd), head = (int)((i / hd) % H), pos = (int)(i / ((uint64_t)hd * H));
        const size_t dst = (((size_t)page_table[pos / ps] * H + head) * ps + pos % ps) * hd + e;
        cache[dst] = float_to_wt<WT>(gen_value(base, i, scale));
    }
}
// fp32 rows -> packed rows (scaled by gain) + per-slice sums of squares, sliced over the columns exactly as the
// CTAs of the decode kernel slice an operator's output (slice c = columns [K c / n, K (c+1) / n)).  One warp per row: a slice
// is a few dozen columns, so that a CTA per row and slice would spend its time in barriers.
__global__ void pack_rows_kernel(const float* x, int ldx, int M, int K, const float* gain, unsigned char* xpk, int ldpk,
                                 float* ssq, int nslices) {
    grid_dependents_launch();
    const int cta = blockIdx.x, lane = threadIdx.x & 31;
    const int k0 = (int)((unsigned)K * (unsigned)cta / (unsigned)nslices), k1 = (int)((unsigned)K * (unsigned)(cta + 1) / (unsigned)nslices);
    for (int m = threadIdx.x >> 5; m < M; m += blockDim.x >> 5) {
        float ss = 0.f;
        for (int k = k0 + lane; k < k1; k += 32) {
            const float v = x[(size_t)m * ldx + k];
            ss += v * v;
            pk_store(xpk + (size_t)m * ldpk, k, gain ? v * gain[k] : v);
        }
        ss = warp_sum(ss);
        if (lane == 0 && ssq) ssq[(size_t)m * nslices + cta] = ss;
    }
}

enum { TID_EMBED = 1, TID_HEAD = 2, TID_PROMPT = 3, TID_HIDDEN = 4, TID_GFINAL = 6, TID_DRAFT = 7, TID_LAYER_BASE = 100 };
enum { K_WQKV = 0, K_WO = 1, K_WGATE = 2, K_WUP = 3, K_WDOWN = 4, K_G1 = 5, K_G2 = 6, K_KCACHE = 8, K_VCACHE = 9 };
inline uint64_t layer_tid(int layer, int k) { return (uint64_t)TID_LAYER_BASE + 16ull * (uint64_t)layer + (uint64_t)k; }

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

struct Layout {
    size_t off_hApk, off_featApk, off_featDpk, off_abufpk, off_ssqA, off_ssqF, off_ssqAb, off_xch[2], xch_bytes;
    int xch_ld;
    size_t off_layers, off_pt, off_kc, off_vc, off_h, off_feat, off_abuf, off_po, off_ml,
        off_cnt, off_xp, xp_bytes, off_rope, off_hp, off_dbgd, off_dbgv, off_out, off_S, off_rlog, off_prompt, off_st, off_bar;
    // tensor-core prompt pass (0 bytes each when the shape cannot take it)
    size_t off_pf_h, off_pf_x, off_pf_q, off_pf_f, off_pf_rs, off_pf_part, off_pf_cnt, off_pf_err;
    size_t pf_rows, pf_part_bytes;
    size_t off_embed, off_head, off_gfinal;
    std::vector<size_t> off_w[5];     // wqkv, wo, wgate, wup, wdown
    std::vector<size_t> off_g[2];
    size_t total;
};

// The tensor-core prompt pass needs bf16 weights, a head_dim the tensor-core attention knows, and matrix sides that
// are whole tiles: N a multiple of 128, K a multiple of 64.
bool prefill_tc_shape(const kg_config* c) {
    return c->dtype == KG_BF16 && (c->head_dim == 64 || c->head_dim == 128) && c->d_model % 128 == 0 && c->d_ffn % 128 == 0 &&
           c->d_model <= PF_EW_THREADS * 4 * PF_NORM_V;      // the norm kernel keeps a row in registers
}

bool valid_config(const kg_config* c) {
    if (!c || c->struct_size != sizeof(kg_config)) return false;
    if (c->n_layers < 2 || c->exit_layer < 1 || c->exit_layer >= c->n_layers) return false;
    if (c->d_model <= 0 || c->n_heads <= 0 || c->n_heads * c->head_dim != c->d_model) return false;
    if (c->head_dim != 32 && c->head_dim != 64 && c->head_dim != 128) return false;
    if (c->d_model % 8 || c->d_ffn % 8 || c->d_ffn <= 0 || c->vocab <= 1) return false;
    if (c->dtype != KG_F32 && c->dtype != KG_BF16) return false;
    if (c->gamma_max < 1 || c->gamma_max > KG_GAMMA_MAX) return false;
    if (c->page_size < 1 || (c->page_size & (c->page_size - 1)) || c->max_seq < 2) return false;       // pages hold a power of two of tokens
    if (c->n_heads > 256) return false;
    if (c->vocab > (1 << 20) || c->d_ffn > (1 << 20)) return false;      // rows x CTAs must fit 32 bits
    // one launch may run max_seq tokens, each at most L + 5 grid barriers of at most 1024 CTAs: the arrival counter (31 bits
    // beside the abort flag) must hold them all (the bound counts five barriers a layer)
    if ((long long)c->max_seq * (5LL * (c->n_layers + 1) + 8) * 1024LL >= (1LL << 31)) return false;
    // the plain path stages all rows of an operand in shared memory
    const int kmax = c->d_ffn > c->d_model ? c->d_ffn : c->d_model;
    const bool plain_somewhere = c->dtype == KG_F32 || (c->d_model % 16) || (c->d_ffn % 16);
    if (plain_somewhere && (size_t)kmax * KG_M_MAX * 4 > (size_t)SIMPLE_XS_BYTES) return false;
    return true;
}

Layout make_layout(const kg_config* c, int own_weights, int nctas) {
    Layout L;
    const size_t es = c->dtype == KG_BF16 ? 2 : 4;
    const size_t d = c->d_model, F = c->d_ffn, V = c->vocab, H = c->n_heads, hd = c->head_dim;
    const int nl = c->n_layers;
    const size_t n_pages = (c->max_seq + c->page_size - 1) / c->page_size;
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + bytes, 256); return r; };
    L.off_st = take(sizeof(State));
    L.off_bar = take(256);
    L.off_layers = take(sizeof(LayerW) * (nl + 1));
    L.off_pt = take(sizeof(int) * n_pages);
    const size_t cache_bytes = (size_t)(nl + 1) * n_pages * H * c->page_size * hd * es;
    L.off_kc = take(cache_bytes);
    L.off_vc = take(cache_bytes);
    L.off_h = take(4 * KG_M_MAX * d);
    L.off_feat = take(4 * (KG_M_MAX + 1) * d);
    L.off_abuf = take(4 * 2 * d);
    L.xch_ld = (int)align_up(5 * d + F + nctas, 4);
    L.xch_bytes = 4 * (size_t)KG_M_MAX * L.xch_ld;
    L.off_xch[0] = take(L.xch_bytes); L.off_xch[1] = take(L.xch_bytes);
    L.off_hApk = take(4 * KG_M_MAX * d);
    L.off_featApk = take(4 * (KG_M_MAX + 1) * d);
    L.off_featDpk = take(4 * (KG_M_MAX + 1) * d);
    L.off_abufpk = take(4 * 2 * d);
    L.off_ssqA = take(4 * (size_t)KG_M_MAX * nctas);
    L.off_ssqF = take(4 * (size_t)(KG_M_MAX + 1) * nctas);
    L.off_ssqAb = take(4 * (size_t)2 * nctas);
    L.off_po = take(4 * (size_t)KG_M_MAX * H * S_CAP * hd);
    L.off_ml = take(4 * (size_t)KG_M_MAX * H * S_CAP * 2);
    L.off_cnt = take(4 * H);
    L.xp_bytes = c->dtype == KG_BF16 ? 4 * (size_t)KG_M_MAX * H * S_CAP * (hd + 4) : 0;
    L.off_xp = take(L.xp_bytes);
    L.off_rope = take(c->dtype == KG_BF16 ? 4 * (size_t)(c->max_seq + KG_M_MAX) * hd : 0);
    L.off_hp = take(sizeof(float4) * (size_t)nctas * KG_M_MAX);
    L.off_dbgd = take(c->debug_logits ? 4 * (size_t)KG_M_MAX * V : 0);
    L.off_dbgv = take(c->debug_logits ? 4 * (size_t)KG_M_MAX * V : 0);
    L.off_out = take(4 * (size_t)(c->max_seq + KG_M_MAX));
    L.off_S = take(4 * (size_t)(c->max_seq + KG_M_MAX));
    L.off_rlog = take(16 * (size_t)(c->max_seq + KG_M_MAX));
    L.off_prompt = take(4 * (size_t)c->max_seq);
    {
        // rows of a block; planes (hi, then lo) of the GEMM inputs; partial sums of the tiles that are cut along k
        const size_t R = prefill_tc_shape(c) ? align_up(c->max_seq < PF_ROWS ? c->max_seq : PF_ROWS, 256) : 0;
        L.pf_rows = R;
        L.pf_part_bytes = R ? (size_t)nctas * GM_TM * GM_NT_MAX * 4 : 0;
        L.off_pf_h = take(4 * R * d); L.off_pf_x = take(4 * R * d); L.off_pf_q = take(4 * R * d); L.off_pf_f = take(4 * R * F);
        L.off_pf_rs = take(4 * R); L.off_pf_part = take(L.pf_part_bytes);
        L.off_pf_cnt = take(R ? 4 * (size_t)nctas : 0); L.off_pf_err = take(R ? 64 : 0);
    }
    for (int k = 0; k < 5; ++k) L.off_w[k].assign(nl + 1, 0);
    for (int k = 0; k < 2; ++k) L.off_g[k].assign(nl + 1, 0);
    L.off_embed = L.off_head = L.off_gfinal = 0;
    if (own_weights) {
        L.off_embed = take(es * V * d);
        L.off_head = take(es * V * d);
        L.off_gfinal = take(4 * d);
        for (int i = 0; i <= nl; ++i) {
            L.off_w[K_WQKV][i] = take(es * 3 * d * d);
            L.off_w[K_WO][i] = take(es * d * d);
            if (i < nl) {
                L.off_w[K_WGATE][i] = take(es * F * d);
                L.off_w[K_WUP][i] = take(es * F * d);
                L.off_w[K_WDOWN][i] = take(es * d * F);
            }
            L.off_g[0][i] = take(4 * d);
            L.off_g[1][i] = take(4 * d);
        }
    }
    L.total = o;
    return L;
}

// SM count of the current device (one CTA per SM in every launch), looked up once per device.
constexpr int MAX_DEVICES = 64;
int g_sm_count[MAX_DEVICES] = {0};
int sm_count() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 148;
    if (dev >= 0 && dev < MAX_DEVICES && g_sm_count[dev] > 0) return g_sm_count[dev];
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return 148;
    if (dev >= 0 && dev < MAX_DEVICES) g_sm_count[dev] = n;
    return n;
}

// Device pointers handed in by the caller feed 16-byte bulk copies and vector loads: anything less aligned would
// fault on the device, so it is refused on the host.
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Token ids that arrive in device memory cannot be checked on the host: one thread per id records an argument
// error in the state word (the embedding lookup itself keeps every access in bounds).
__global__ void check_tokens_kernel(const int* toks, int n, int vocab, State* st) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && (unsigned)toks[i] >= (unsigned)vocab) atomicCAS(&st->status, 0, (int)KG_E_ARG);
}

}  // namespace

// Tensor maps of the prompt pass, encoded once per model: the weights in boxes of 128 rows (64 for the gate / up pair),
// the planes [R][K] in boxes of 16 * (i + 1) rows (a CTA's half of a tile), one set for K = d (x) and one for K = F (f).
struct PfMaps {
    CUtensorMap x[2][GM_NT_MAX / GM_NT_STEP], f[2][GM_NT_MAX / GM_NT_STEP];   // [hi, lo][activation rows per tile / GM_NT_STEP - 1]
    struct Layer { CUtensorMap qkv, o, gate, up, down; };
    std::vector<Layer> layer;
    CUtensorMap adapter_kv;                                    // the k and v rows of the adapter's W_qkv
    bool ready;
};

struct kg_model {
    kg_config cfg;
    PfMaps pf;
    Dev dev;
    Layout lay;
    char* arena;
    cudaStream_t stream;
    int nctas;
    size_t smem;
    bool own_weights;
    bool prefilled, pending, ar_used, dead;
    int prefill_mode;              // 0: tensor-core prompt pass when the shape and the prompt allow, 1: always the chunked pass
    unsigned long long wait_clk;   // budget of a device-side wait, in SM clocks
    int skip_arrival;              // test hook, consumed by the next launch
    cudaEvent_t ev0, ev1;          // timing of the decode loop in kg_generate, created on first use
    int gamma_pending;
    long long P_upper;      // upper bound of the device-side position P
    int force_simple;
    std::vector<LayerW> layers_host;
};

// Name and text of the CUDA error behind the last KG_E_CUDA of this thread ("" if there was none).
static thread_local char g_cuda_err[160] = "";
static bool cuda_failed(cudaError_t e, const char* what) {
    if (e == cudaSuccess) return false;
    std::snprintf(g_cuda_err, sizeof(g_cuda_err), "%s: %s (%s)", what, cudaGetErrorName(e), cudaGetErrorString(e));
    return true;
}
#define CK(x) do { if (cuda_failed((x), #x)) return KG_E_CUDA; } while (0)

extern "C" const char* kg_last_cuda_error(void) { return g_cuda_err; }

extern "C" const char* kg_strerror(int s) {
    switch (s) {
        case KG_OK: return "ok";
        case KG_E_ARG: return "invalid argument";
        case KG_E_STATE: return "call order violated";
        case KG_E_NOMEM: return "arena too small";
        case KG_E_SEQ_FULL: return "sequence would exceed max_seq";
        case KG_E_CUDA: return "CUDA runtime error";
        case KG_E_TIMEOUT: return "device-side wait timed out";
        case KG_E_LIMIT: return "size beyond the capacity of the library's static scratch (or of the operator scratch)";
        case KG_E_INTERNAL: return "a device-side index check failed (the access was skipped)";
        default: return "unknown status";
    }
}

extern "C" size_t kg_workspace_bytes(const kg_config* cfg, int own_weights) {
    if (!valid_config(cfg)) return 0;
    return make_layout(cfg, own_weights, sm_count()).total + 256;
}

// The decode kernel for a storage type, a head size and an attention (ring: bf16, 64 or 128 only)
static const void* decode_kernel(const kg_config& c, bool ring) {
    typedef __nv_bfloat16 bf;
    if (c.dtype == KG_BF16) {
        if (ring) return c.head_dim == 128 ? (const void*)kg_persistent_kernel<bf, 128, true> : (const void*)kg_persistent_kernel<bf, 64, true>;
        if (c.head_dim == 128) return (const void*)kg_persistent_kernel<bf, 128, false>;
        return c.head_dim == 64 ? (const void*)kg_persistent_kernel<bf, 64, false> : (const void*)kg_persistent_kernel<bf, 32, false>;
    }
    if (c.head_dim == 128) return (const void*)kg_persistent_kernel<float, 128, false>;
    return c.head_dim == 64 ? (const void*)kg_persistent_kernel<float, 64, false> : (const void*)kg_persistent_kernel<float, 32, false>;
}

// Before the first launch of a decode kernel.  Its warpgroups re-divide the registers that the launch gives the CTA; a budget beyond
// that pool would block the kernel at its first instruction, so that the launch allocation is checked here and never assumed.
static int prepare_decode(const kg_model* m) {
    const void* kfn = decode_kernel(m->cfg, m->dev.dm.ring != 0);
    CK(cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)m->smem));
    int occ = 0;
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kfn, DECODE_THREADS, m->smem));
    if (occ < 1) return KG_E_CUDA;
    cudaFuncAttributes fa;
    CK(cudaFuncGetAttributes(&fa, kfn));
    if ((long long)fa.numRegs * DECODE_THREADS < (long long)NTHREADS * CONSUMER_REGS + 128LL * PRODUCER_REGS) {
        std::snprintf(g_cuda_err, sizeof(g_cuda_err), "decode kernel compiled with %d registers per thread: too few for its register budgets", fa.numRegs);
        return KG_E_INTERNAL;
    }
    return KG_OK;
}

static int launch(kg_model* m, const Program& pg) {
    Program p = pg;
    p.force_simple = m->force_simple;
    p.wait_clk = m->wait_clk;
    p.skip_arrival = m->skip_arrival;
    m->skip_arrival = 0;
    void* args[] = {(void*)&m->dev, (void*)&p};
    CK(cudaLaunchCooperativeKernel(decode_kernel(m->cfg, m->dev.dm.ring != 0), dim3(m->nctas), dim3(DECODE_THREADS), args, m->smem, m->stream));
    return KG_OK;
}

// The part of the state word that a new sequence starts from; an expired wait stays recorded behind it, because such a launch leaves
// exchange words behind that the next one would take for values.
constexpr size_t SEQ_STATE_BYTES = offsetof(State, timed_out);

static int read_state(kg_model* m, State* out) {
    CK(cudaMemcpyAsync(out, m->dev.st, sizeof(State), cudaMemcpyDeviceToHost, m->stream));
    CK(cudaStreamSynchronize(m->stream));
    if (out->timed_out) { m->dead = true; return KG_E_TIMEOUT; }
    if (out->status == ST_INTERNAL) {
        std::snprintf(g_cuda_err, sizeof(g_cuda_err), "device-side index check %d failed", out->timeout_where);
        m->dead = true;
        return KG_E_INTERNAL;
    }
    if (out->status != 0) {
        // an argument error found on the device (a token id outside the vocabulary): the sequence is unusable until
        // kg_reset, which also clears the state word; the weights are untouched
        m->prefilled = m->pending = false; m->ar_used = true;
        return out->status;
    }
    return KG_OK;
}

namespace {
int prefill_tc(kg_model* m, int n);                 // the tensor-core prompt pass (end of this file)
bool prefill_tc_ok(const kg_model* m, int n);
int prefill_tc_init(kg_model* m);
bool make_tmap(CUtensorMap* tm, const void* base, uint64_t rows, uint64_t K, int box_rows);
int tmap_failed();
}

template <typename WT>
static int fill_weights(kg_model* m) {
    const kg_config& c = m->cfg;
    cudaStream_t s = m->stream;
    const uint64_t d = c.d_model, F = c.d_ffn, V = c.vocab;
    const int nl = c.n_layers;
    auto fill = [&](size_t off, uint64_t tid, uint64_t count, double std_) {
        fill_matrix_kernel<WT><<<1184, 256, 0, s>>>(reinterpret_cast<WT*>(m->arena + off), stream_base(c.seed, tid), count, gen_scale(std_));
    };
    auto gain = [&](size_t off, uint64_t tid) {
        fill_gain_kernel<<<16, 256, 0, s>>>(reinterpret_cast<float*>(m->arena + off), stream_base(c.seed, tid), (int)d, gen_scale(c.gain_std));
    };
    fill(m->lay.off_embed, TID_EMBED, V * d, c.embed_std);
    fill(m->lay.off_head, TID_HEAD, V * d, c.init_std);
    gain(m->lay.off_gfinal, TID_GFINAL);
    for (int i = 0; i <= nl; ++i) {
        const bool adapter = i == nl;
        const double os = adapter ? c.adapter_resid_scale : (i >= c.exit_layer ? c.deep_resid_scale : 1.0);
        // the output-projection std is formed in fp32 exactly as the host recipe does: float(init_std) * float(scale)
        const double std_o = (double)c.init_std * os;
        fill(m->lay.off_w[K_WQKV][i], layer_tid(i, K_WQKV), 3 * d * d, c.init_std);
        fill(m->lay.off_w[K_WO][i], layer_tid(i, K_WO), d * d, std_o);
        if (!adapter) {
            fill(m->lay.off_w[K_WGATE][i], layer_tid(i, K_WGATE), F * d, c.init_std);
            fill(m->lay.off_w[K_WUP][i], layer_tid(i, K_WUP), F * d, c.init_std);
            fill(m->lay.off_w[K_WDOWN][i], layer_tid(i, K_WDOWN), d * F, std_o);
        }
        gain(m->lay.off_g[0][i], layer_tid(i, K_G1));
        gain(m->lay.off_g[1][i], layer_tid(i, K_G2));
    }
    CK(cudaGetLastError());
    return KG_OK;
}

extern "C" int kg_init_model(const kg_config* cfg, const kg_weights* w, void* arena_dev, size_t arena_bytes,
                             void* cuda_stream, kg_model** out) {
    if (!out) return KG_E_ARG;
    *out = nullptr;
    if (!valid_config(cfg) || !arena_dev) return KG_E_ARG;
    if (w) {
        if (!w->embed_dev || !w->head_dev || !w->g_final_dev || !w->wqkv_dev || !w->wo_dev || !w->wgate_dev ||
            !w->wup_dev || !w->wdown_dev || !w->g1_dev || !w->g2_dev) return KG_E_ARG;
        if (!aligned16(w->embed_dev) || !aligned16(w->head_dev) || !aligned16(w->g_final_dev)) return KG_E_ARG;
        for (int i = 0; i <= cfg->n_layers; ++i) {
            const bool layer = i < cfg->n_layers;
            if (!w->wqkv_dev[i] || !w->wo_dev[i] || !w->g1_dev[i] || !w->g2_dev[i] ||
                (layer && (!w->wgate_dev[i] || !w->wup_dev[i] || !w->wdown_dev[i]))) return KG_E_ARG;
            if (!aligned16(w->wqkv_dev[i]) || !aligned16(w->wo_dev[i]) || !aligned16(w->g1_dev[i]) || !aligned16(w->g2_dev[i]) ||
                (layer && (!aligned16(w->wgate_dev[i]) || !aligned16(w->wup_dev[i]) || !aligned16(w->wdown_dev[i])))) return KG_E_ARG;
        }
    }
    const int nctas = sm_count();
    const int own = w ? 0 : 1;
    Layout lay = make_layout(cfg, own, nctas);
    char* base = reinterpret_cast<char*>(align_up(reinterpret_cast<size_t>(arena_dev), 256));
    if ((size_t)(base - reinterpret_cast<char*>(arena_dev)) + lay.total > arena_bytes) return KG_E_NOMEM;

    kg_model* m = new (std::nothrow) kg_model();
    if (!m) return KG_E_NOMEM;
    m->cfg = *cfg; m->lay = lay; m->arena = base; m->stream = (cudaStream_t)cuda_stream; m->nctas = nctas;
    m->own_weights = own != 0; m->prefilled = m->pending = m->ar_used = m->dead = false;
    m->gamma_pending = 0; m->P_upper = 0; m->force_simple = 0;
    m->wait_clk = WAIT_TIMEOUT_CLK; m->skip_arrival = 0; m->ev0 = m->ev1 = nullptr; m->prefill_mode = 0;
    m->smem = SMEM_TOTAL;

    const bool bf = cfg->dtype == KG_BF16;

    Dev& D = m->dev;
    std::memset(&D, 0, sizeof(D));
    D.dm.L = cfg->n_layers; D.dm.d = cfg->d_model; D.dm.H = cfg->n_heads; D.dm.hd = cfg->head_dim; D.dm.F = cfg->d_ffn;
    D.dm.V = cfg->vocab; D.dm.l = cfg->exit_layer; D.dm.eps = cfg->rms_eps; D.dm.theta = cfg->rope_theta;
    D.dm.logit_scale = cfg->logit_scale; D.dm.max_seq = cfg->max_seq; D.dm.page_size = cfg->page_size;
    D.dm.n_pages = (cfg->max_seq + cfg->page_size - 1) / cfg->page_size; D.dm.gamma_max = cfg->gamma_max;
    D.dm.n_phys = D.dm.n_pages;
    for (D.dm.ps_shift = 0; (1 << D.dm.ps_shift) < cfg->page_size; ++D.dm.ps_shift) {}
    D.dm.debug = cfg->debug_logits;
    for (int i = 0; i < cfg->head_dim / 2; ++i)
        D.inv_freq[i] = std::pow((double)cfg->rope_theta, -2.0 * (double)i / (double)cfg->head_dim);
    auto P = [&](size_t off) { return base + off; };
    D.st = (State*)P(lay.off_st); D.bar = (unsigned*)P(lay.off_bar);
    D.layers = (const LayerW*)P(lay.off_layers); D.page_table = (const int*)P(lay.off_pt);
    D.kcache = P(lay.off_kc); D.vcache = P(lay.off_vc);
    D.h = (float*)P(lay.off_h); D.feat = (float*)P(lay.off_feat); D.abuf = (float*)P(lay.off_abuf);
    D.xch[0] = (unsigned*)P(lay.off_xch[0]); D.xch[1] = (unsigned*)P(lay.off_xch[1]); D.xch_ld = lay.xch_ld;
    D.att_po = (float*)P(lay.off_po); D.att_ml = (float*)P(lay.off_ml); D.att_cnt = (unsigned*)P(lay.off_cnt);
    D.head_part = (float4*)P(lay.off_hp);
    D.hA_pk = (unsigned char*)P(lay.off_hApk);
    D.featA_pk = (unsigned char*)P(lay.off_featApk); D.featD_pk = (unsigned char*)P(lay.off_featDpk);
    D.abuf_pk = (unsigned char*)P(lay.off_abufpk);
    D.ssq_hA = (float*)P(lay.off_ssqA);
    D.ssq_feat = (float*)P(lay.off_ssqF); D.ssq_abuf = (float*)P(lay.off_ssqAb);
    D.dm.stream = (cfg->dtype == KG_BF16 && cfg->d_model % 16 == 0 && cfg->d_ffn % 16 == 0) ? 1 : 0;
    D.dbg_draft = cfg->debug_logits ? (float*)P(lay.off_dbgd) : nullptr;
    D.dbg_verify = cfg->debug_logits ? (float*)P(lay.off_dbgv) : nullptr;
    D.out_tokens = (int*)P(lay.off_out); D.S = (int*)P(lay.off_S); D.round_log = (int*)P(lay.off_rlog);
    D.prompt = (const int*)P(lay.off_prompt);

    const int nl = cfg->n_layers;
    m->layers_host.resize(nl + 1);
    if (own) {
        D.embed = P(lay.off_embed); D.head = P(lay.off_head); D.g_final = (const float*)P(lay.off_gfinal);
        for (int i = 0; i <= nl; ++i) {
            LayerW& lw = m->layers_host[i];
            lw.wqkv = P(lay.off_w[K_WQKV][i]); lw.wo = P(lay.off_w[K_WO][i]);
            lw.wgate = i < nl ? P(lay.off_w[K_WGATE][i]) : nullptr;
            lw.wup = i < nl ? P(lay.off_w[K_WUP][i]) : nullptr;
            lw.wdown = i < nl ? P(lay.off_w[K_WDOWN][i]) : nullptr;
            lw.g1 = (const float*)P(lay.off_g[0][i]); lw.g2 = (const float*)P(lay.off_g[1][i]);
        }
    } else {
        D.embed = w->embed_dev; D.head = w->head_dev; D.g_final = w->g_final_dev;
        for (int i = 0; i <= nl; ++i) {
            LayerW& lw = m->layers_host[i];
            lw.wqkv = w->wqkv_dev[i]; lw.wo = w->wo_dev[i];
            lw.wgate = i < nl ? w->wgate_dev[i] : nullptr;
            lw.wup = i < nl ? w->wup_dev[i] : nullptr;
            lw.wdown = i < nl ? w->wdown_dev[i] : nullptr;
            lw.g1 = w->g1_dev[i]; lw.g2 = w->g2_dev[i];
        }
    }
    cudaStream_t s = m->stream;
    bool ok = cudaMemcpyAsync(P(lay.off_layers), m->layers_host.data(), sizeof(LayerW) * (nl + 1), cudaMemcpyHostToDevice, s) == cudaSuccess;
    // page table: identity, or a fixed permutation (reversal within blocks of 4 pages plus a rotation)
    std::vector<int> pt(D.dm.n_pages);
    for (int i = 0; i < D.dm.n_pages; ++i) pt[i] = i;
    if (cfg->page_shuffle) {
        const int n = D.dm.n_pages;
        for (int i = 0; i < n; ++i) pt[i] = (int)(((long long)i * 7 + 3) % n);
        // i -> 7i+3 mod n is a permutation only if gcd(7, n) == 1; otherwise fall back to reversal
        if (n % 7 == 0) for (int i = 0; i < n; ++i) pt[i] = n - 1 - i;
    }
    ok = ok && cudaMemcpyAsync(P(lay.off_pt), pt.data(), sizeof(int) * pt.size(), cudaMemcpyHostToDevice, s) == cudaSuccess;
    ok = ok && cudaMemsetAsync(D.st, 0, sizeof(State), s) == cudaSuccess;
    ok = ok && cudaMemsetAsync(D.bar, 0, BAR_BYTES, s) == cudaSuccess;
    if (bf) {
        D.att_xp = (unsigned*)P(lay.off_xp);
        ok = ok && cudaMemsetAsync(D.att_xp, 0xff, lay.xp_bytes, s) == cudaSuccess;      // XCH_EMPTY
        rope_table_kernel<<<cfg->max_seq + KG_M_MAX, cfg->head_dim / 2, 0, s>>>(D, (float2*)P(lay.off_rope));
        D.rope = (const float2*)P(lay.off_rope);
        ok = ok && cudaGetLastError() == cudaSuccess;
        const uint64_t rows = (uint64_t)(cfg->n_layers + 1) * D.dm.n_pages * cfg->n_heads * cfg->page_size;
        const int box = cfg->page_size < 16 ? cfg->page_size : 16;
        D.dm.ring = D.dm.stream && (cfg->head_dim == 64 || cfg->head_dim == 128) && rows < (1ull << 31) &&
                    make_tmap(&D.tmk, D.kcache, rows, cfg->head_dim, box) && make_tmap(&D.tmv, D.vcache, rows, cfg->head_dim, box);
    }
    for (int i = 0; i < 2; ++i) ok = ok && cudaMemsetAsync(D.xch[i], 0xff, lay.xch_bytes, s) == cudaSuccess;      // XCH_EMPTY
    ok = ok && cudaMemsetAsync(D.att_cnt, 0, 4 * cfg->n_heads, s) == cudaSuccess;
    ok = ok && cudaStreamSynchronize(s) == cudaSuccess;    // pt / layers_host are host temporaries
    if (!ok) { delete m; return KG_E_CUDA; }
    if (own) {
        int r = bf ? fill_weights<__nv_bfloat16>(m) : fill_weights<float>(m);
        // the fill kernels have run to completion (and without a fault) when the model is handed out
        if (r == KG_OK && cuda_failed(cudaStreamSynchronize(s), "weight fill")) r = KG_E_CUDA;
        if (r != KG_OK) { delete m; return r; }
    }
    {
        int r = prepare_decode(m);
        if (r == KG_OK) r = prefill_tc_init(m);
        if (r != KG_OK) { delete m; return r; }
    }
    *out = m;
    return KG_OK;
}

extern "C" int kg_free_model(kg_model* m) {
    if (!m) return KG_E_ARG;
    if (m->ev0) cudaEventDestroy(m->ev0);
    if (m->ev1) cudaEventDestroy(m->ev1);
    delete m;
    return KG_OK;
}

extern "C" int kg_reset(kg_model* m) {
    if (!m) return KG_E_ARG;
    if (m->dead) return KG_E_TIMEOUT;
    CK(cudaMemsetAsync(m->dev.st, 0, SEQ_STATE_BYTES, m->stream));
    CK(cudaMemsetAsync(m->dev.att_cnt, 0, 4 * m->cfg.n_heads, m->stream));
    m->prefilled = m->pending = m->ar_used = false;
    m->P_upper = 0;
    return KG_OK;
}

static int prefill_common(kg_model* m, int32_t n) {
    int r;
    if (prefill_tc_ok(m, n)) {
        r = prefill_tc(m, n);
    } else {
        Program pg{}; pg.kind = PROG_PREFILL; pg.n = n;
        r = launch(m, pg);
    }
    if (r != KG_OK) return r;
    m->prefilled = true; m->pending = false; m->P_upper = n;
    return KG_OK;
}

extern "C" int kg_prefill(kg_model* m, const int32_t* prompt_host, int32_t n, int32_t* first_token_host) {
    if (!m || !prompt_host || n < 1) return KG_E_ARG;
    if (m->dead) return KG_E_TIMEOUT;
    if (m->prefilled || m->ar_used) return KG_E_STATE;
    if (n + 1 > m->cfg.max_seq) return KG_E_SEQ_FULL;
    for (int i = 0; i < n; ++i) if (prompt_host[i] < 0 || prompt_host[i] >= m->cfg.vocab) return KG_E_ARG;
    CK(cudaMemcpyAsync((void*)m->dev.prompt, prompt_host, sizeof(int32_t) * n, cudaMemcpyHostToDevice, m->stream));
    int r = prefill_common(m, n);
    if (r != KG_OK) return r;
    if (first_token_host) {
        State st;
        r = read_state(m, &st);
        if (r != KG_OK) return r;
        *first_token_host = st.x0;
    } else {
        // the prompt buffer is the caller's: make sure the copy has left it
        CK(cudaStreamSynchronize(m->stream));
    }
    return KG_OK;
}

extern "C" int kg_prefill_device(kg_model* m, const int32_t* prompt_dev, int32_t n) {
    if (!m || !prompt_dev || n < 1) return KG_E_ARG;
    if (m->dead) return KG_E_TIMEOUT;
    if (m->prefilled || m->ar_used) return KG_E_STATE;
    if (n + 1 > m->cfg.max_seq) return KG_E_SEQ_FULL;
    if (reinterpret_cast<uintptr_t>(prompt_dev) & 3u) return KG_E_ARG;
    CK(cudaMemcpyAsync((void*)m->dev.prompt, prompt_dev, sizeof(int32_t) * n, cudaMemcpyDeviceToDevice, m->stream));
    check_tokens_kernel<<<(n + 255) / 256, 256, 0, m->stream>>>(m->dev.prompt, n, m->cfg.vocab, m->dev.st);
    CK(cudaGetLastError());
    return prefill_common(m, n);
}

static bool bad_spec(const kg_model* m, float eta, int gamma, int mode) {
    return !(eta == eta) || gamma < 1 || gamma > m->cfg.gamma_max || (mode != KG_STOP_KEEP && mode != KG_STOP_DROP);
}

extern "C" int kg_draft(kg_model* m, float eta, int32_t gamma, int32_t stop_mode, kg_draft_out* out) {
    if (!m || bad_spec(m, eta, gamma, stop_mode)) return KG_E_ARG;
    if (m->dead) return KG_E_TIMEOUT;
    if (!m->prefilled || m->pending || m->ar_used) return KG_E_STATE;
    if (m->P_upper + gamma + 2 > m->cfg.max_seq) return KG_E_SEQ_FULL;
    Program pg{}; pg.kind = PROG_DRAFT; pg.eta = eta; pg.gamma = gamma; pg.stop_mode = stop_mode;
    int r = launch(m, pg);
    if (r != KG_OK) return r;
    m->pending = true; m->gamma_pending = gamma;
    if (out) {
        State st;
        r = read_state(m, &st);
        if (r != KG_OK) return r;
        out->n_drafted = st.n_d; out->n_steps = st.n_steps;
        for (int i = 0; i < KG_GAMMA_MAX; ++i) { out->tokens[i] = i < st.n_d ? st.draft_tok[i] : -1; out->conf[i] = i < st.n_steps ? st.conf[i] : 0.f; }
    }
    return KG_OK;
}

extern "C" int kg_verify(kg_model* m, kg_verify_out* out) {
    if (!m) return KG_E_ARG;
    if (m->dead) return KG_E_TIMEOUT;
    if (!m->prefilled || !m->pending) return KG_E_STATE;
    Program pg{}; pg.kind = PROG_VERIFY;
    int r = launch(m, pg);
    if (r != KG_OK) return r;
    m->pending = false;
    m->P_upper += m->gamma_pending + 1;
    if (out) {
        State st;
        r = read_state(m, &st);
        if (r != KG_OK) return r;
        out->n_rows = st.M; out->n_accept = st.k_acc; out->n_emitted = st.n_emit;
        for (int i = 0; i < KG_M_MAX; ++i) { out->emitted[i] = i < st.n_emit ? st.emitted[i] : -1; out->target[i] = i < st.M ? st.target[i] : -1; }
        m->P_upper = st.P;
    }
    return KG_OK;
}

static void fill_stats(kg_model* m, const State& st, const std::vector<int>& S, int max_tokens, kg_stats* out) {
    std::memset(out, 0, sizeof(*out));
    std::vector<int> s2(S);
    // truncate so that only tokens up to max_tokens (x_0 excluded from S) are counted
    long long sum = 0;
    for (size_t i = 0; i < s2.size(); ++i) {
        if (max_tokens >= 0 && sum + s2[i] > max_tokens - 1) { s2[i] = (int)(max_tokens - 1 - sum); s2.resize(s2[i] > 0 ? i + 1 : i); sum = max_tokens - 1; break; }
        sum += s2[i];
    }
    out->rounds = (int)s2.size(); out->tokens = (int)sum;
    out->draft_steps = st.draft_steps_total; out->drafted = st.drafted_total; out->accepted = st.accepted_total;
    if (!s2.empty()) {
        out->cr = (double)sum / (double)s2.size();
        for (int w = 0; w <= KG_M_MAX; ++w) {
            int cnt = 0;
            for (int v : s2) cnt += (v - w > 0);
            out->ctar[w] = (double)cnt / (double)s2.size();
        }
    }
}

static int read_S_vec(kg_model* m, int rounds, std::vector<int>& S) {
    S.assign(rounds, 0);
    if (rounds > 0) {
        CK(cudaMemcpyAsync(S.data(), m->dev.S, sizeof(int) * rounds, cudaMemcpyDeviceToHost, m->stream));
        CK(cudaStreamSynchronize(m->stream));
    }
    return KG_OK;
}

extern "C" int kg_decode(kg_model* m, int32_t max_new, float eta, int32_t gamma, int32_t stop_mode, kg_stats* stats) {
    if (!m || bad_spec(m, eta, gamma, stop_mode) || max_new < 1) return KG_E_ARG;
    if (m->dead) return KG_E_TIMEOUT;
    if (!m->prefilled || m->pending || m->ar_used) return KG_E_STATE;
    if (m->P_upper + max_new + gamma + 2 > m->cfg.max_seq) return KG_E_SEQ_FULL;
    Program pg{}; pg.kind = PROG_DECODE; pg.n = max_new; pg.eta = eta; pg.gamma = gamma; pg.stop_mode = stop_mode;
    int r = launch(m, pg);
    if (r != KG_OK) return r;
    m->P_upper += max_new + gamma + 1;
    if (stats) {
        State st;
        r = read_state(m, &st);
        if (r != KG_OK) return r;
        m->P_upper = st.P;
        std::vector<int> S;
        r = read_S_vec(m, st.rounds, S);
        if (r != KG_OK) return r;
        fill_stats(m, st, S, max_new, stats);
    }
    return KG_OK;
}

extern "C" int kg_decode_ar(kg_model* m, int32_t n_tokens, int32_t* out_host) {
    if (!m || n_tokens < 1) return KG_E_ARG;
    if (m->dead) return KG_E_TIMEOUT;
    if (!m->prefilled || m->pending) return KG_E_STATE;
    if (m->P_upper + n_tokens + 1 > m->cfg.max_seq) return KG_E_SEQ_FULL;
    Program pg{}; pg.kind = PROG_AR; pg.n = n_tokens;
    int r = launch(m, pg);
    if (r != KG_OK) return r;
    m->ar_used = true;
    m->P_upper += n_tokens;
    if (out_host) {
        State st;
        r = read_state(m, &st);
        if (r != KG_OK) return r;
        CK(cudaMemcpyAsync(out_host, m->dev.out_tokens, sizeof(int) * n_tokens, cudaMemcpyDeviceToHost, m->stream));
        CK(cudaStreamSynchronize(m->stream));
    }
    return KG_OK;
}

extern "C" int kg_read_tokens(kg_model* m, int32_t* out_host, int32_t max_n, int32_t* n_out) {
    if (!m || !out_host || max_n < 0) return KG_E_ARG;
    State st;
    int r = read_state(m, &st);
    if (r != KG_OK) return r;
    const int n = st.total < max_n ? st.total : max_n;
    if (n > 0) {
        CK(cudaMemcpyAsync(out_host, m->dev.out_tokens, sizeof(int) * n, cudaMemcpyDeviceToHost, m->stream));
        CK(cudaStreamSynchronize(m->stream));
    }
    if (n_out) *n_out = n;
    return KG_OK;
}

extern "C" int kg_read_S(kg_model* m, int32_t* out_host, int32_t max_n, int32_t* n_out) {
    if (!m || !out_host || max_n < 0) return KG_E_ARG;
    State st;
    int r = read_state(m, &st);
    if (r != KG_OK) return r;
    const int n = st.rounds < max_n ? st.rounds : max_n;
    if (n > 0) {
        CK(cudaMemcpyAsync(out_host, m->dev.S, sizeof(int) * n, cudaMemcpyDeviceToHost, m->stream));
        CK(cudaStreamSynchronize(m->stream));
    }
    if (n_out) *n_out = n;
    return KG_OK;
}

extern "C" int kg_read_round_log(kg_model* m, int32_t* out_host, int32_t max_rounds, int32_t* n_out) {
    if (!m || !out_host || max_rounds < 0) return KG_E_ARG;
    State st;
    int r = read_state(m, &st);
    if (r != KG_OK) return r;
    const int n = st.rounds < max_rounds ? st.rounds : max_rounds;
    if (n > 0) {
        CK(cudaMemcpyAsync(out_host, m->dev.round_log, sizeof(int) * 4 * n, cudaMemcpyDeviceToHost, m->stream));
        CK(cudaStreamSynchronize(m->stream));
    }
    if (n_out) *n_out = n;
    return KG_OK;
}

extern "C" int kg_generate(kg_model* m, const int32_t* prompt_host, int32_t n_prompt, int32_t max_new,
                           float eta, int32_t gamma, int32_t stop_mode,
                           int32_t* out_tokens_host, int32_t* n_out, kg_stats* stats) {
    if (!m || !prompt_host || !out_tokens_host || max_new < 1 || bad_spec(m, eta, gamma, stop_mode)) return KG_E_ARG;
    if ((long long)n_prompt + max_new + gamma + 2 > m->cfg.max_seq) return KG_E_SEQ_FULL;
    int r = kg_reset(m);
    if (r != KG_OK) return r;
    for (int i = 0; i < n_prompt; ++i) if (prompt_host[i] < 0 || prompt_host[i] >= m->cfg.vocab) return KG_E_ARG;
    if (n_prompt < 1) return KG_E_ARG;
    CK(cudaMemcpyAsync((void*)m->dev.prompt, prompt_host, sizeof(int32_t) * n_prompt, cudaMemcpyHostToDevice, m->stream));
    r = prefill_common(m, n_prompt);
    if (r != KG_OK) return r;
    const bool timed = stats != nullptr;
    if (timed) {
        if (!m->ev0) { CK(cudaEventCreate(&m->ev0)); CK(cudaEventCreate(&m->ev1)); }      // once per model
        CK(cudaEventRecord(m->ev0, m->stream));
    }
    r = kg_decode(m, max_new, eta, gamma, stop_mode, nullptr);
    if (timed && r == KG_OK) cudaEventRecord(m->ev1, m->stream);
    State st;
    if (r == KG_OK) r = read_state(m, &st);
    if (r == KG_OK) {
        if (cudaMemcpyAsync(out_tokens_host, m->dev.out_tokens, sizeof(int) * max_new, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess ||
            cudaStreamSynchronize(m->stream) != cudaSuccess) r = KG_E_CUDA;
    }
    if (r == KG_OK) {
        m->P_upper = st.P;
        if (n_out) *n_out = max_new;
        if (stats) {
            std::vector<int> S;
            r = read_S_vec(m, st.rounds, S);
            if (r == KG_OK) {
                fill_stats(m, st, S, max_new, stats);
                float ms = 0.f;
                if (cudaEventElapsedTime(&ms, m->ev0, m->ev1) == cudaSuccess) stats->ms_decode = ms;
            }
        }
    }
    return r;
}

extern "C" int kg_debug_logits(kg_model* m, int32_t which, int32_t row, float* out_host) {
    if (!m || !out_host || row < 0 || row >= KG_M_MAX || (which != 0 && which != 1)) return KG_E_ARG;
    if (!m->cfg.debug_logits) return KG_E_STATE;
    const float* src = (which == 0 ? m->dev.dbg_draft : m->dev.dbg_verify) + (size_t)row * m->cfg.vocab;
    CK(cudaMemcpyAsync(out_host, src, sizeof(float) * m->cfg.vocab, cudaMemcpyDeviceToHost, m->stream));
    CK(cudaStreamSynchronize(m->stream));
    return KG_OK;
}

extern "C" int kg_read_weight(kg_model* m, const char* name, int32_t layer, uint64_t offset, uint64_t count, float* out_host) {
    if (!m || !name || !out_host) return KG_E_ARG;
    const kg_config& c = m->cfg;
    const uint64_t d = c.d_model, F = c.d_ffn, V = c.vocab;
    const void* p = nullptr; uint64_t n = 0; bool f32 = false;
    const bool lay_ok = layer >= 0 && layer <= c.n_layers;
    if (!std::strcmp(name, "embed")) { p = m->dev.embed; n = V * d; }
    else if (!std::strcmp(name, "head")) { p = m->dev.head; n = V * d; }
    else if (!std::strcmp(name, "g_final")) { p = m->dev.g_final; n = d; f32 = true; }
    else if (!lay_ok) return KG_E_ARG;
    else if (!std::strcmp(name, "wqkv")) { p = m->layers_host[layer].wqkv; n = 3 * d * d; }
    else if (!std::strcmp(name, "wo")) { p = m->layers_host[layer].wo; n = d * d; }
    else if (!std::strcmp(name, "wgate")) { p = m->layers_host[layer].wgate; n = F * d; }
    else if (!std::strcmp(name, "wup")) { p = m->layers_host[layer].wup; n = F * d; }
    else if (!std::strcmp(name, "wdown")) { p = m->layers_host[layer].wdown; n = d * F; }
    else if (!std::strcmp(name, "g1")) { p = m->layers_host[layer].g1; n = d; f32 = true; }
    else if (!std::strcmp(name, "g2")) { p = m->layers_host[layer].g2; n = d; f32 = true; }
    else return KG_E_ARG;
    if (!p || offset > n || count > n - offset) return KG_E_ARG;
    if (f32 || c.dtype == KG_F32) {
        CK(cudaMemcpyAsync(out_host, (const float*)p + offset, 4 * count, cudaMemcpyDeviceToHost, m->stream));
        CK(cudaStreamSynchronize(m->stream));
    } else {
        std::vector<uint16_t> tmp(count);
        CK(cudaMemcpyAsync(tmp.data(), (const uint16_t*)p + offset, 2 * count, cudaMemcpyDeviceToHost, m->stream));
        CK(cudaStreamSynchronize(m->stream));
        for (uint64_t i = 0; i < count; ++i) { uint32_t b = (uint32_t)tmp[i] << 16; std::memcpy(out_host + i, &b, 4); }
    }
    return KG_OK;
}

extern "C" int kg_debug_fill_state(kg_model* m, int32_t T, int32_t n_d, uint64_t seed) {
    if (!m || T < 1 || n_d < -1 || n_d > m->cfg.gamma_max) return KG_E_ARG;
    if (m->dead) return KG_E_TIMEOUT;
    const kg_config& c = m->cfg;
    if (T + c.gamma_max + 2 > c.max_seq) return KG_E_SEQ_FULL;
    cudaStream_t s = m->stream;
    const float one = gen_scale(1.0);
    const size_t lstride = (size_t)m->dev.dm.n_pages * c.n_heads * c.page_size * c.head_dim;
    for (int i = 0; i <= c.n_layers; ++i) {
        if (c.dtype == KG_BF16) {
            fill_cache_kernel<__nv_bfloat16><<<592, 256, 0, s>>>((__nv_bfloat16*)m->dev.kcache + i * lstride, m->dev.page_table, stream_base(seed, layer_tid(i, K_KCACHE)), T, c.n_heads, c.head_dim, c.page_size, one);
            fill_cache_kernel<__nv_bfloat16><<<592, 256, 0, s>>>((__nv_bfloat16*)m->dev.vcache + i * lstride, m->dev.page_table, stream_base(seed, layer_tid(i, K_VCACHE)), T, c.n_heads, c.head_dim, c.page_size, one);
        } else {
            fill_cache_kernel<float><<<592, 256, 0, s>>>((float*)m->dev.kcache + i * lstride, m->dev.page_table, stream_base(seed, layer_tid(i, K_KCACHE)), T, c.n_heads, c.head_dim, c.page_size, one);
            fill_cache_kernel<float><<<592, 256, 0, s>>>((float*)m->dev.vcache + i * lstride, m->dev.page_table, stream_base(seed, layer_tid(i, K_VCACHE)), T, c.n_heads, c.head_dim, c.page_size, one);
        }
    }
    fill_f32_kernel<<<64, 256, 0, s>>>(m->dev.feat, stream_base(seed, TID_HIDDEN), (uint64_t)(KG_M_MAX + 1) * c.d_model, one);
    if (m->dev.dm.stream) {
        const int d = c.d_model;
        pack_rows_kernel<<<m->nctas, 256, 0, s>>>(m->dev.feat, d, KG_M_MAX + 1, d, m->layers_host[c.n_layers].g1, m->dev.featA_pk, d * 4, m->dev.ssq_feat, m->nctas);
        pack_rows_kernel<<<m->nctas, 256, 0, s>>>(m->dev.feat, d, KG_M_MAX + 1, d, m->layers_host[c.exit_layer].g1, m->dev.featD_pk, d * 4, m->dev.ssq_feat, m->nctas);
    }
    CK(cudaGetLastError());
    // tokens: x_0 and the drafts
    const uint64_t tb = stream_base(seed, TID_DRAFT);
    State st;
    std::memset(&st, 0, sizeof(st));
    st.P = T; st.len_A = T; st.total = 1; st.x0 = (int)(mix64(tb + 1000) % (uint64_t)c.vocab);
    if (n_d >= 0) {
        st.pending = 1; st.n_d = n_d; st.n_steps = n_d;
        for (int i = 0; i < n_d; ++i) { st.draft_tok[i] = (int)(mix64(tb + (uint64_t)i) % (uint64_t)c.vocab); st.conf[i] = 1.0f; }
    }
    CK(cudaMemcpyAsync(m->dev.st, &st, SEQ_STATE_BYTES, cudaMemcpyHostToDevice, s));
    CK(cudaMemsetAsync(m->dev.att_cnt, 0, 4 * c.n_heads, s));
    CK(cudaStreamSynchronize(s));
    m->prefilled = true; m->pending = n_d >= 0; m->ar_used = false; m->gamma_pending = n_d >= 0 ? n_d : 0; m->P_upper = T;
    return KG_OK;
}

extern "C" int kg_debug_force_simple(kg_model* m, int on) {
    if (!m) return KG_E_ARG;
    // the plain path stages all rows of an operand in shared memory: only shapes whose rows fit may take it
    const int kmax = m->cfg.d_ffn > m->cfg.d_model ? m->cfg.d_ffn : m->cfg.d_model;
    if (on && (size_t)kmax * KG_M_MAX * 4 > (size_t)SIMPLE_XS_BYTES) return KG_E_ARG;
    m->force_simple = on ? 1 : 0;
    return KG_OK;
}

extern "C" int kg_debug_set_wait_budget(kg_model* m, double milliseconds) {
    if (!m || !(milliseconds > 0.0) || milliseconds > 60000.0) return KG_E_ARG;
    int dev = 0, khz = 0;
    CK(cudaGetDevice(&dev));
    CK(cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, dev));
    m->wait_clk = (unsigned long long)(milliseconds * (double)khz);      // kHz = clocks per millisecond
    if (m->wait_clk < 1000ull) m->wait_clk = 1000ull;
    return KG_OK;
}

extern "C" int kg_debug_skip_barrier_arrival(kg_model* m, int cta) {
    if (!m || cta < 0 || cta >= m->nctas) return KG_E_ARG;
    m->skip_arrival = cta + 1;
    return KG_OK;
}

// ------------------------------------------------------------------------------------ single operators
namespace {

constexpr int OP_K_MAX = 32768;               // longest input row the single-operator entry points pack into scratch
constexpr size_t OP_GEMM_PART = 16u << 20;    // partial sums of the GEMM's cut tiles
constexpr int OP_GEMM_CNT = 1024;             // their arrival counters, then the error word
struct OpScratch { size_t off_hp, off_po, off_ml, off_cnt, off_xp, off_xpk, off_ssq, off_gemm, off_gcnt, total; };
OpScratch op_layout() {
    OpScratch s; size_t o = 0;
    auto take = [&](size_t b) { size_t r = o; o = align_up(o + b, 256); return r; };
    s.off_hp = take(sizeof(float4) * 1024 * KG_M_MAX);
    s.off_po = take(4 * (size_t)KG_M_MAX * S_CAP * 8192);
    s.off_ml = take(4 * (size_t)KG_M_MAX * 256 * S_CAP * 2);
    s.off_cnt = take(4 * 256);
    s.off_xp = take(4 * (size_t)KG_M_MAX * S_CAP * (8192 + 4 * 256));
    s.off_xpk = take(4 * (size_t)KG_M_MAX * OP_K_MAX);
    s.off_ssq = take(4 * (size_t)KG_M_MAX * 1024);
    s.off_gemm = take(OP_GEMM_PART);
    s.off_gcnt = take(4 * (OP_GEMM_CNT + 1));
    s.total = o;
    return s;
}

// One linear operator as a kernel of its own.  V: the row variant of the streamed tensor-core path (bf16 weights, K a multiple of
// 16), 0: the plain path; compiled one by one, because all variants in one kernel spill at its 168 registers.  FEW: lin_few().
template <typename WT, int V, bool FEW>
__global__ void __launch_bounds__(BLOCK_THREADS, 1) op_linear_kernel(const __grid_constant__ LinArgs a) {
    extern __shared__ __align__(128) char smem[];
    Ctx& c = ctx_init(smem, nullptr, nullptr, false);
    grid_dependents_launch();
    if constexpr (V == 0) {
        if (!c.producer) lin_simple<WT>(a, c);
    } else if (c.producer) {
        // launched while the kernel that packs the rows may still run: the copy warp starts on the weights at once
        if (!lin_produce<false>(a, c)) ring_drain(c);
    } else {
        grid_dependency_wait();
        lin_consume<V, FEW>(a, c);
    }
}
// one warp per row (one thread per row took 60 us: a chain of a merge per CTA)
__global__ void op_head_final_kernel(const float4* part, int nctas, int* tok, float* p) {
    grid_dependency_wait();
    const int m = threadIdx.x >> 5;
    int t; float pp;
    head_final_warp(part, nctas, m, t, pp);
    if ((threadIdx.x & 31) == 0) { tok[m] = t; p[m] = pp; }
}
// R: row groups of the tensor-core attention.  The other attention has no copy warp: without it a thread gets 255 registers and not
// 168 (three warps in one of the four register files), at which fp32 of 128 dims spilled 0.7 KB.
template <typename WT, int HD> constexpr int OP_ATT_THREADS = RING_ATT<WT, HD> ? BLOCK_THREADS : NTHREADS;
template <typename WT, int HD, int R>
__global__ void __launch_bounds__(OP_ATT_THREADS<WT, HD>, 1) op_attention_kernel(const __grid_constant__ Dev D, const __grid_constant__ AttArgs a) {
    extern __shared__ __align__(128) char smem[];
    Ctx& c = ctx_init(smem, nullptr, nullptr, false);
    if constexpr (!RING_ATT<WT, HD>) attention_impl<WT, HD / 32, true>(D, a, a.plan, c);
    else if (!c.producer) attention_ring<HD, R, false>(D, a, c);
    else if (!att_produce<HD, false>(D, a.plan, 0, c)) ring_drain(c);
}
// The arrival counters of the splits.  The attention behind it starts at once and waits where it counts its first split.  (A
// memset of the kilobyte cannot overlap the kernel behind it: 2 us a call.)
__global__ void clear_counters_kernel(unsigned* cnt) {
    grid_dependents_launch();
    cnt[threadIdx.x] = 0u;
}

// A launch that may begin before the kernel ahead of it in the stream has finished; the kernel calls grid_dependency_wait()
// before it touches anything that one writes.
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kfn)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kfn, P(args)...);
}

int g_force_simple_ops = 0;

// Lets kernel KFN use SMEM_TOTAL bytes of shared memory; the attribute belongs to the kernel and the device, so it is set at the
// first call on each device (bit `device` of `done`; two threads may both set it, to the same value).
template <auto KFN>
int set_smem() {
    static std::atomic<uint64_t> done{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return KG_E_CUDA;
    const uint64_t bit = dev >= 0 && dev < 64 ? 1ull << dev : 0;
    if (bit && (done.load(std::memory_order_relaxed) & bit)) return KG_OK;
    if (cudaFuncSetAttribute((const void*)KFN, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_TOTAL) != cudaSuccess) return KG_E_CUDA;
    done.fetch_or(bit, std::memory_order_relaxed);
    return KG_OK;
}

}  // namespace

extern "C" size_t kg_op_scratch_bytes(void) { return op_layout().total; }

extern "C" int kg_debug_force_simple_ops(int on) { g_force_simple_ops = on ? 1 : 0; return KG_OK; }

// Whether the CTAs of a streamed operator have so few stage pairs that their warps' sums are kept apart.  The kernel without that code is the
// faster one where it is not used (LM head 32000 x 4096, 16 rows, 78.6 -> 77.6 us; 12288 x 4096, 11 rows, 33.0 -> 32.0), and at 9 to 12 rows with two phases
// (4096 x 4096, 12 rows, 18.4 -> 17.2 us; with three and more phases the sums kept apart win: 2368 x 8192 22.4 -> 20.9).
template <int V>
static bool lin_few(const LinArgs& a, int nctas) {
    const int units = 2 * (((a.N + 1) / 2 + nctas - 1) / nctas), groups = (units + ST_ROWS - 1) / ST_ROWS;       // of a CTA, at most (cta_unit)
    return a.nph > (V == 12 ? 2 : 1) && (a.W2 ? groups : (groups + 1) / 2) <= LinGeom<V>::FEWP;
}
template <int V, bool FEW>
static int launch_streamed_linear(const LinArgs& a, int nctas, cudaStream_t s) {
    if (set_smem<op_linear_kernel<__nv_bfloat16, V, FEW>>() != KG_OK) return KG_E_CUDA;
    CK(launch_dependent(op_linear_kernel<__nv_bfloat16, V, FEW>, dim3(nctas), dim3(BLOCK_THREADS), SMEM_TOTAL, s, a));
    return KG_OK;
}
template <int V>
static int launch_linear(const LinArgs& a, int nctas, cudaStream_t s) {
    return lin_few<V>(a, nctas) ? launch_streamed_linear<V, true>(a, nctas, s) : launch_streamed_linear<V, false>(a, nctas, s);
}
template <typename WT>
static int launch_plain(const LinArgs& a, int nctas, cudaStream_t s) {
    if (set_smem<op_linear_kernel<WT, 0, false>>() != KG_OK) return KG_E_CUDA;
    op_linear_kernel<WT, 0, false><<<nctas, BLOCK_THREADS, SMEM_TOTAL, s>>>(a);
    return KG_OK;
}

// xpk / ssq: scratch for the packed copy of the input rows (xpk_k_max = longest row it holds) and their sums of squares
static int op_linear_common(int32_t dtype, LinArgs& a, unsigned char* xpk, int xpk_k_max, float* ssq, cudaStream_t s) {
    if (dtype != KG_F32 && dtype != KG_BF16) return KG_E_ARG;
    if (a.M < 1 || a.M > KG_M_MAX || a.N < 1 || a.N > (1 << 20) || a.K < 8 || (a.K % 8)) return KG_E_ARG;
    const bool plain = dtype == KG_F32 || g_force_simple_ops || (a.K % 16);
    if (plain && (size_t)a.K * a.M * 4 > (size_t)SIMPLE_XS_BYTES) return KG_E_ARG;
    const int nctas = sm_count();
    if (!plain) {
        if (a.K > xpk_k_max || nctas > 1024) return KG_E_LIMIT;
        pack_rows_kernel<<<nctas, 256, 0, s>>>(a.x, a.ldx, a.M, a.K, a.gain, xpk, a.K * 4, a.gain ? ssq : nullptr, nctas);
        a.xpk = xpk; a.ldpk = a.K * 4; a.ssq_in = a.gain ? ssq : nullptr; a.ld_ssq = nctas;
        lin_phases(a);
    }
    int r;
    if (dtype == KG_F32) r = launch_plain<float>(a, nctas, s);
    else if (plain) r = launch_plain<__nv_bfloat16>(a, nctas, s);
    else r = a.M <= 4 ? launch_linear<4>(a, nctas, s) : a.M <= 8 ? launch_linear<8>(a, nctas, s) : a.M <= 12 ? launch_linear<12>(a, nctas, s) : launch_linear<16>(a, nctas, s);
    if (r != KG_OK) return r;
    CK(cudaGetLastError());
    return KG_OK;
}

extern "C" int kg_op_linear(int32_t dtype, const void* W, const void* W2, int32_t N, int32_t K,
                            const float* x, int32_t M, const float* gain, float eps,
                            const float* resid, int32_t swiglu, float* out, void* scratch, void* stream) {
    if (!W || !x || !out || !scratch) return KG_E_ARG;
    if (swiglu && !W2) return KG_E_ARG;
    if (!aligned16(W) || !aligned16(W2) || !aligned16(x) || !aligned16(gain) || !aligned16(resid) || !aligned16(out) ||
        !aligned16(scratch)) return KG_E_ARG;
    LinArgs a{};
    a.W = W; a.W2 = swiglu ? W2 : nullptr; a.N = N; a.K = K; a.x = x; a.ldx = K; a.M = M; a.gain = gain; a.eps = eps;
    a.resid = resid; a.ldr = N; a.out = out; a.ldo = N;
    a.epi = swiglu ? EPI_SWIGLU : (resid ? EPI_RESID : EPI_STORE);
    OpScratch sc = op_layout();
    return op_linear_common(dtype, a, (unsigned char*)scratch + sc.off_xpk, OP_K_MAX, (float*)((char*)scratch + sc.off_ssq), (cudaStream_t)stream);
}

extern "C" int kg_op_lm_head(int32_t dtype, const void* W, int32_t V, int32_t K, const float* x, int32_t M,
                             const float* gain, float eps, float logit_scale,
                             int32_t* tok, float* p, float* logits, void* scratch, void* stream) {
    if (!W || !x || !tok || !p || !scratch) return KG_E_ARG;
    if (!aligned16(W) || !aligned16(x) || !aligned16(gain) || !aligned16(logits) || !aligned16(scratch) ||
        (reinterpret_cast<uintptr_t>(tok) & 3u) || (reinterpret_cast<uintptr_t>(p) & 3u)) return KG_E_ARG;
    if (sm_count() > 1024) return KG_E_ARG;
    OpScratch sc = op_layout();
    LinArgs a{};
    a.W = W; a.N = V; a.K = K; a.x = x; a.ldx = K; a.M = M; a.gain = gain; a.eps = eps;
    a.epi = EPI_HEAD; a.scale = logit_scale; a.head_part = (float4*)((char*)scratch + sc.off_hp);
    a.logits_dbg = logits; a.ld_dbg = V;
    int r = op_linear_common(dtype, a, (unsigned char*)scratch + sc.off_xpk, OP_K_MAX, (float*)((char*)scratch + sc.off_ssq), (cudaStream_t)stream);
    if (r != KG_OK) return r;
    CK(launch_dependent(op_head_final_kernel, dim3(1), dim3(32 * M), 0, (cudaStream_t)stream, a.head_part, sm_count(), tok, p));
    return KG_OK;
}

// ------------------------------------------------------------------------------------ no-allocation variant
// The LM-head operator keeps one partial (max, sum, arg max) per CTA and row in scratch memory.  Here that
// scratch is a fixed array inside the library image instead of caller memory.
namespace {
constexpr int NOALLOC_MAX_CTAS = 256;                        // CTAs (one per SM) the static scratch has room for
constexpr int NOALLOC_MAX_K = 8192;                          // longest input row it can pack
constexpr int NOALLOC_MAX_DEVICES = 64;
constexpr size_t NOALLOC_OFF_XPK = sizeof(float4) * NOALLOC_MAX_CTAS * KG_M_MAX;                 // head partials first: 64 KB
constexpr size_t NOALLOC_OFF_SSQ = NOALLOC_OFF_XPK + 4 * (size_t)KG_M_MAX * NOALLOC_MAX_K;        // packed input rows: 512 KB
constexpr size_t NOALLOC_BYTES = NOALLOC_OFF_SSQ + 4 * (size_t)KG_M_MAX * NOALLOC_MAX_CTAS;       // sums of squares: 16 KB
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];
static_assert(NOALLOC_MAX_DEVICES <= MAX_DEVICES, "per-device tables");
void* g_noalloc_addr[NOALLOC_MAX_DEVICES] = {nullptr};

// Device address of the static scratch on the current device.  In host code the array's name is only a
// handle for the runtime, never a pointer a kernel may use; the address comes from cudaGetSymbolAddress.
int noalloc_scratch(void** out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return KG_E_CUDA;
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return KG_E_LIMIT;
    if (!g_noalloc_addr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return KG_E_CUDA;
        g_noalloc_addr[dev] = p;
    }
    *out = g_noalloc_addr[dev];
    return KG_OK;
}
}  // namespace

extern "C" int kg_op_lm_head_noalloc(int32_t dtype, const void* W, int32_t V, int32_t K, const float* x, int32_t M,
                                     const float* gain, float eps, float logit_scale,
                                     int32_t* tok, float* p, float* logits, void* stream) {
    if (!W || !x || !tok || !p) return KG_E_ARG;
    if (!aligned16(W) || !aligned16(x) || !aligned16(gain) || !aligned16(logits) ||
        (reinterpret_cast<uintptr_t>(tok) & 3u) || (reinterpret_cast<uintptr_t>(p) & 3u)) return KG_E_ARG;
    if (M > KG_M_MAX || K > NOALLOC_MAX_K || sm_count() > NOALLOC_MAX_CTAS) return KG_E_LIMIT;
    void* scratch = nullptr;
    int r = noalloc_scratch(&scratch);
    if (r != KG_OK) return r;
    // the partials of an earlier call are stale but harmless: every CTA rewrites its rows before they are merged
    LinArgs a{};
    a.W = W; a.N = V; a.K = K; a.x = x; a.ldx = K; a.M = M; a.gain = gain; a.eps = eps;
    a.epi = EPI_HEAD; a.scale = logit_scale; a.head_part = (float4*)scratch;
    a.logits_dbg = logits; a.ld_dbg = V;
    r = op_linear_common(dtype, a, (unsigned char*)scratch + NOALLOC_OFF_XPK, NOALLOC_MAX_K, (float*)((char*)scratch + NOALLOC_OFF_SSQ),
                         (cudaStream_t)stream);
    if (r != KG_OK) return r;
    CK(launch_dependent(op_head_final_kernel, dim3(1), dim3(32 * M), 0, (cudaStream_t)stream, a.head_part, sm_count(), tok, p));
    return KG_OK;
}

template <typename WT, int HD, int R>
static int launch_attention(const Dev& D, const AttArgs& a, int nctas, cudaStream_t s) {
    if (set_smem<op_attention_kernel<WT, HD, R>>() != KG_OK) return KG_E_CUDA;
    if (a.plan.S > 1) CK(launch_dependent(op_attention_kernel<WT, HD, R>, dim3(nctas), dim3(OP_ATT_THREADS<WT, HD>), SMEM_TOTAL, s, D, a));
    else op_attention_kernel<WT, HD, R><<<nctas, OP_ATT_THREADS<WT, HD>, SMEM_TOTAL, s>>>(D, a);
    return KG_OK;
}

extern "C" int kg_op_attention(int32_t dtype, const float* qkv, int32_t M, int32_t pos0, int32_t H, int32_t hd,
                               float theta, void* kc, void* vc, const int32_t* page_table, int32_t page_size,
                               float* out, void* scratch, void* stream) {
    if (!qkv || !kc || !vc || !page_table || !out || !scratch) return KG_E_ARG;
    if (dtype != KG_F32 && dtype != KG_BF16) return KG_E_ARG;
    if (!aligned16(qkv) || !aligned16(kc) || !aligned16(vc) || !aligned16(out) || !aligned16(scratch) ||
        (reinterpret_cast<uintptr_t>(page_table) & 3u)) return KG_E_ARG;
    if (M < 1 || M > KG_M_MAX || pos0 < 0 || H < 1 || H > 256 || (hd != 32 && hd != 64 && hd != 128) || page_size < 1 ||
        (page_size & (page_size - 1))) return KG_E_ARG;
    if ((size_t)H * hd > 8192) return KG_E_ARG;
    OpScratch sc = op_layout();
    cudaStream_t s = (cudaStream_t)stream;
    Dev D;
    std::memset(&D, 0, sizeof(D));
    D.dm.H = H; D.dm.hd = hd; D.dm.d = H * hd; D.dm.page_size = page_size; D.dm.theta = theta;
    D.dm.n_pages = (pos0 + M + page_size - 1) / page_size;       // entries of page_table this call may touch
    // the caller's cache: its page count is not known here.  The ring's tensor maps count the rows of all pages in 31 bits
    const long long page_rows = (long long)H * page_size;
    D.dm.ring = dtype == KG_BF16 && hd != 32;
    if (D.dm.ring && page_rows > 0x7fffffff) return KG_E_ARG;
    D.dm.n_phys = D.dm.ring ? (int)(0x7fffffff / page_rows) : 0x7fffffff;
    for (D.dm.ps_shift = 0; (1 << D.dm.ps_shift) < page_size; ++D.dm.ps_shift) {}
    for (int i = 0; i < hd / 2; ++i) D.inv_freq[i] = std::pow((double)theta, -2.0 * (double)i / (double)hd);
    D.page_table = page_table;
    D.att_po = (float*)((char*)scratch + sc.off_po); D.att_ml = (float*)((char*)scratch + sc.off_ml);
    D.att_cnt = (unsigned*)((char*)scratch + sc.off_cnt);
    if (D.dm.ring) {
        const int box = page_size < 16 ? page_size : 16;
        if (!make_tmap(&D.tmk, kc, 0x7fffffff, hd, box) || !make_tmap(&D.tmv, vc, 0x7fffffff, hd, box)) return tmap_failed();
        D.att_xp = (unsigned*)((char*)scratch + sc.off_xp);
    }
    AttArgs a{}; a.qkv = qkv; a.ldq = 3 * H * hd; a.M = M; a.pos0 = pos0; a.kc = kc; a.vc = vc; a.out = out; a.ldo = H * hd;
    const int nctas = sm_count();
    a.plan = D.dm.ring ? ra_plan(pos0, H, nctas) : ka_plan(pos0, M, H, nctas);
    if (a.plan.S > 1) {
        clear_counters_kernel<<<1, 256, 0, s>>>(D.att_cnt);
        CK(cudaGetLastError());
    }
    typedef __nv_bfloat16 bf;
    int r;
    if (dtype == KG_F32) r = hd == 128 ? launch_attention<float, 128, 1>(D, a, nctas, s) : hd == 64 ? launch_attention<float, 64, 1>(D, a, nctas, s) : launch_attention<float, 32, 1>(D, a, nctas, s);
    else if (hd == 32) r = launch_attention<bf, 32, 1>(D, a, nctas, s);
    else if (M <= 8) r = hd == 128 ? launch_attention<bf, 128, 1>(D, a, nctas, s) : launch_attention<bf, 64, 1>(D, a, nctas, s);
    else r = hd == 128 ? launch_attention<bf, 128, 2>(D, a, nctas, s) : launch_attention<bf, 64, 2>(D, a, nctas, s);
    if (r != KG_OK) return r;
    CK(cudaGetLastError());
    return KG_OK;
}

// ------------------------------------------------------------------------------------ tensor-core prompt pass
namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// cuTensorMapEncodeTiled of the driver, looked up through the runtime (the library does not link libcuda)
EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// Tensor map of a row-major bf16 matrix [rows, K] read in boxes of 64 columns x box_rows rows with the 128-byte swizzle.
// base is 16-byte aligned and K * 2 a multiple of 16 (checked by the callers' shape test).
bool make_tmap(CUtensorMap* tm, const void* base, uint64_t rows, uint64_t K, int box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {K, rows};
    const cuuint64_t strides[1] = {K * 2};
    const cuuint32_t box[2] = {(cuuint32_t)GM_BK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
int tmap_failed() {
    std::snprintf(g_cuda_err, sizeof(g_cuda_err), "cuTensorMapEncodeTiled failed");
    return KG_E_CUDA;
}

// The kernel's warpgroups re-divide the registers of the launch: a budget beyond that pool would block them for ever, so
// what the launch allocates is checked and never assumed.
template <int EPI>
int gemm_attributes() {
    cudaFuncAttributes fa;
    CK(cudaFuncGetAttributes(&fa, (const void*)pf_gemm_kernel<EPI>));
    if ((long long)fa.numRegs * GM_THREADS < 128LL * GM_CTRL_REGS + 32LL * GM_EPI_WARPS * GM_EPI_REGS) {
        std::snprintf(g_cuda_err, sizeof(g_cuda_err), "GEMM kernel compiled with %d registers per thread: too few for its register budgets", fa.numRegs);
        return KG_E_INTERNAL;
    }
    CK(cudaFuncSetAttribute((const void*)pf_gemm_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, GM_SMEM));
    return KG_OK;
}

template <int HD>
int attention_attributes() {
    CK(cudaFuncSetAttribute((const void*)pf_attention_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, FaSm<HD>::BYTES));
    cudaFuncAttributes fa;
    CK(cudaFuncGetAttributes(&fa, (const void*)pf_attention_tc_kernel<HD>));
    if ((long long)fa.numRegs * FT_THREADS < 128LL * FT_CTRL_REGS + 32LL * FT_SOFT_WARPS * FT_SOFT_REGS) {
        std::snprintf(g_cuda_err, sizeof(g_cuda_err), "attention kernel compiled with %d registers per thread: too few for its register budgets", fa.numRegs);
        return KG_E_INTERNAL;
    }
    CK(cudaFuncSetAttribute((const void*)pf_attention_tc_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, FtSm<HD>::BYTES));
    return KG_OK;
}

int prefill_tc_init(kg_model* m) {
    m->pf.ready = false;
    if (m->dev.dm.stream == 0 || !prefill_tc_shape(&m->cfg) || encode_tiled_fn() == nullptr) return KG_OK;
    const uint64_t d = m->cfg.d_model, F = m->cfg.d_ffn, R = m->lay.pf_rows;
    const int L = m->cfg.n_layers;
    char* A = m->arena;
    bool ok = true;
    for (int p = 0; p < 2; ++p)
        for (int i = 0; i < GM_NT_MAX / GM_NT_STEP; ++i) {
            ok = ok && make_tmap(&m->pf.x[p][i], A + m->lay.off_pf_x + (size_t)p * R * d * 2, R, d, GM_NT_STEP / 2 * (i + 1));
            ok = ok && make_tmap(&m->pf.f[p][i], A + m->lay.off_pf_f + (size_t)p * R * F * 2, R, F, GM_NT_STEP / 2 * (i + 1));
        }
    m->pf.layer.resize(L);
    for (int i = 0; i < L; ++i) {
        const LayerW& lw = m->layers_host[i];
        PfMaps::Layer& t = m->pf.layer[i];
        ok = ok && make_tmap(&t.qkv, lw.wqkv, 3 * d, d, GM_TM / 2) && make_tmap(&t.o, lw.wo, d, d, GM_TM / 2) &&
             make_tmap(&t.gate, lw.wgate, F, d, GM_TM / 4) && make_tmap(&t.up, lw.wup, F, d, GM_TM / 4) && make_tmap(&t.down, lw.wdown, d, F, GM_TM / 2);
    }
    ok = ok && make_tmap(&m->pf.adapter_kv, (const __nv_bfloat16*)m->layers_host[L].wqkv + d * d, 2 * d, d, GM_TM / 2);
    if (!ok) return tmap_failed();
    int r;
    if ((r = gemm_attributes<PF_STORE>()) != KG_OK || (r = gemm_attributes<PF_QKV>()) != KG_OK || (r = gemm_attributes<PF_SWIGLU>()) != KG_OK) return r;
    if ((r = attention_attributes<128>()) != KG_OK || (r = attention_attributes<64>()) != KG_OK) return r;
    CK(cudaFuncSetAttribute((const void*)op_linear_kernel<__nv_bfloat16, 4, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_TOTAL));
    CK(cudaMemsetAsync(A + m->lay.off_pf_cnt, 0, 4 * (size_t)m->nctas, m->stream));
    m->pf.ready = true;
    return KG_OK;
}

// x_0 from the per-CTA LM-head partials; the sequence state after a prompt of n tokens (one warp)
__global__ void pf_finish_kernel(const float4* part, int nctas, State* st, int* out_tokens, int n, const int* err) {
    int tok; float p;
    head_final_warp(part, nctas, 0, tok, p);
    if (threadIdx.x == 0) {
        if (*err) { atomicCAS(&st->status, 0, ST_TIMEOUT); st->timeout_where = *err == PF_ERR_ATT ? 61 : 60; st->timed_out = 1; }      // a wait inside the attention or a GEMM gave up
        st->P = n; st->len_A = n; st->x0 = tok; st->pending = 0; st->total = 1; st->rounds = 0;
        out_tokens[0] = tok;
    }
}

// A prompt of one chunk (at most KG_M_MAX rows) takes the decode kernels, which stream every weight once and need one launch;
// from two chunks on the GEMMs are faster: 7B, 17 tokens 4.50 against 7.71 ms, 31 tokens 4.49 against 10.18; a four-layer model with
// d = 512, 17 tokens 0.232 against 0.369 ms.  One chunk of 16 takes 5.13 and 0.231 ms, of 8 tokens 3.35 and 0.218.
bool prefill_tc_ok(const kg_model* m, int n) { return m->prefill_mode == 0 && m->pf.ready && n > KG_M_MAX; }

// Tile shape and work items of a GEMM of `rows` activation rows and `wtiles` tiles of weight rows on `pairs` CTA pairs.
// Row tiles: as few as 256 columns allow, all of the same width (a multiple of 32; of
// 64 before: 7B prompts of 200, 300 and 777 tokens 8.2, 10.1 and 23.1 ms, 7.9, 9.9 and 22.3 with it).  The last wave of tiles is cut into S
// ranges of k, S the one with the shortest estimated time in units of a k block: the waves of ranges, plus what a cut
// costs (writing the partial sums and reading S of them back, which grows with the tile's columns; with 4 + S nt / 128 instead
// of 10 + S nt / 64, 7B prompts of 32, 200, 512 and 1024 tokens took 4.67, 8.79, 14.07 and 26.5 ms, now 4.43, 8.21, 13.81, 25.7).
void gm_plan(GemmArgs& g, int wtiles, int pairs, size_t part_bytes) {
    g.nrt = (g.rows + GM_NT_MAX - 1) / GM_NT_MAX;
    g.nt = ((g.rows + g.nrt - 1) / g.nrt + GM_NT_STEP - 1) / GM_NT_STEP * GM_NT_STEP;
    const int tiles = wtiles * g.nrt, nkb = g.K / GM_BK;
    const int rem = tiles % pairs;
    g.full = tiles - rem;
    g.S = 1;
    int best = nkb;
    for (int S = 2; S <= 16 && rem > 0 && nkb / S >= 4; ++S) {
        if ((size_t)rem * S * GM_TM * ((g.nt + 63) / 64 * 64) * 4 > part_bytes) break;
        const int cost = (rem * S + pairs - 1) / pairs * ((nkb + S - 1) / S) + 10 + S * g.nt / 64;
        if (cost < best) { best = cost; g.S = S; }
    }
    g.items = g.full + rem * g.S;
}

template <int EPI>
int gm_launch(GemmArgs& g, const CUtensorMap& hi, const CUtensorMap& lo, const CUtensorMap& w, const CUtensorMap& w2, int pairs, cudaStream_t s) {
    const int used = g.items < pairs ? g.items : pairs;
    CK(launch_dependent(pf_gemm_kernel<EPI>, dim3(2 * used), dim3(GM_THREADS), GM_SMEM, s, hi, lo, w, w2, g));
    return KG_OK;
}

// The attention of a block of prompt rows; tc: on tcgen05.
int launch_prompt_attention(const FaArgs& fa, int hd, bool tc, const CUtensorMap& tmk, const CUtensorMap& tmv, cudaStream_t s) {
    const dim3 grid((fa.rows + FA_ROWS - 1) / FA_ROWS * fa.H);
    static_assert(FA_ROWS == FT_ROWS, "rows of a CTA");
    if (tc) {
        if (hd == 128) CK(launch_dependent(pf_attention_tc_kernel<128>, grid, dim3(FT_THREADS), FtSm<128>::BYTES, s, tmk, tmv, fa));
        else CK(launch_dependent(pf_attention_tc_kernel<64>, grid, dim3(FT_THREADS), FtSm<64>::BYTES, s, tmk, tmv, fa));
    } else if (hd == 128) CK(launch_dependent(pf_attention_kernel<128>, grid, dim3(256), FaSm<128>::BYTES, s, fa));
    else CK(launch_dependent(pf_attention_kernel<64>, grid, dim3(256), FaSm<64>::BYTES, s, fa));
    return KG_OK;
}
bool prompt_attention_tc(const FaArgs& fa) { return fa.pos0 + fa.rows > FT_MIN_KEYS; }

// The prompt in blocks of at most PF_ROWS rows of about equal size, each block through all layers (its K / V are in the
// caches before the next block attends to them), the adapter's K / V after layer l, the LM head on the last row.
int prefill_tc(kg_model* m, int n) {
    typedef __nv_bfloat16 WT;
    const kg_config& c = m->cfg;
    const Dev& D = m->dev;
    cudaStream_t s = m->stream;
    char* A = m->arena;
    const int d = c.d_model, F = c.d_ffn, L = c.n_layers, H = c.n_heads, hd = c.head_dim;
    const size_t R = m->lay.pf_rows;
    float* h = (float*)(A + m->lay.off_pf_h);
    WT* xh = (WT*)(A + m->lay.off_pf_x); WT* xl = xh + R * d;
    WT* qh = (WT*)(A + m->lay.off_pf_q); WT* ql = qh + R * d;
    WT* fh = (WT*)(A + m->lay.off_pf_f); WT* fl = fh + R * F;
    float* rs = (float*)(A + m->lay.off_pf_rs);                     // 1/rms of the rows the planes were made from
    int* err = (int*)(A + m->lay.off_pf_err);
    const int pairs = m->nctas / 2;
    CK(cudaMemsetAsync(err, 0, 4, s));
    const size_t lstride = (size_t)D.dm.n_pages * H * c.page_size * hd;
    const int nblk = (int)((n + R - 1) / R);
    const int brows = nblk == 1 ? n : ((n + nblk - 1) / nblk + 63) / 64 * 64;
    int last = 0;
    for (int b0 = 0; b0 < n; b0 += brows) {
        const int rows = n - b0 < brows ? n - b0 : brows;
        last = rows - 1;
        pf_embed_kernel<<<rows, 256, 0, s>>>(D.prompt + b0, (const WT*)D.embed, c.vocab, d, h);
        GemmArgs base{};
        base.rows = rows; base.err = err; base.part = (float*)(A + m->lay.off_pf_part); base.cnt = (unsigned*)(A + m->lay.off_pf_cnt);
        auto norm = [&](const float* gain) { return launch_dependent(pf_norm_split_kernel, dim3(rows), dim3(PF_EW_THREADS), 0, s, h, d, d, gain, c.rms_eps, xh, xl, rs); };
        auto qkv = [&](const CUtensorMap& w, int li, int sec0) {
            GemmArgs g = base;
            g.N = (3 - sec0) * d; g.K = d; g.rowscale = rs; g.hi = qh; g.lo = ql; g.ldp = d; g.hd = hd; g.H = H; g.sec0 = sec0; g.pos0 = b0;
            g.cs = D.rope + (size_t)b0 * (hd / 2); g.page_table = D.page_table; g.ps_shift = D.dm.ps_shift; g.n_phys = D.dm.n_phys; g.st = D.st;
            g.kc = (WT*)D.kcache + (size_t)li * lstride; g.vc = (WT*)D.vcache + (size_t)li * lstride;
            g.qscale = 1.4426950408889634f / std::sqrt((float)hd);
            gm_plan(g, (g.N + GM_TM - 1) / GM_TM, pairs, m->lay.pf_part_bytes);
            return gm_launch<PF_QKV>(g, m->pf.x[0][g.nt / GM_NT_STEP - 1], m->pf.x[1][g.nt / GM_NT_STEP - 1], w, w, pairs, s);
        };
        auto resid = [&](const CUtensorMap& w, int K) {            // h += planes W^T
            GemmArgs g = base;
            g.N = d; g.K = K; g.C = h; g.resid = h; g.ldc = d;
            gm_plan(g, (d + GM_TM - 1) / GM_TM, pairs, m->lay.pf_part_bytes);
            const int i = g.nt / GM_NT_STEP - 1;
            return K == d ? gm_launch<PF_STORE>(g, m->pf.x[0][i], m->pf.x[1][i], w, w, pairs, s)
                          : gm_launch<PF_STORE>(g, m->pf.f[0][i], m->pf.f[1][i], w, w, pairs, s);
        };
        for (int i = 0; i < L; ++i) {
            const LayerW& lw = m->layers_host[i];
            const PfMaps::Layer& tm = m->pf.layer[i];
            int r;
            CK(norm(lw.g1));
            if ((r = qkv(tm.qkv, i, 0)) != KG_OK) return r;
            FaArgs fa;
            fa.qh = qh; fa.ql = ql; fa.kc = (const WT*)D.kcache + (size_t)i * lstride; fa.vc = (const WT*)D.vcache + (size_t)i * lstride;
            fa.oh = xh; fa.ol = xl; fa.page_table = D.page_table; fa.ps_shift = D.dm.ps_shift; fa.n_phys = D.dm.n_phys; fa.st = D.st;
            fa.H = H; fa.pos0 = b0; fa.rows = rows; fa.row0 = i * D.dm.n_pages * H * c.page_size; fa.err = err; fa.skip = -1;
            if ((r = launch_prompt_attention(fa, hd, D.dm.ring && prompt_attention_tc(fa), D.tmk, D.tmv, s)) != KG_OK) return r;
            if ((r = resid(tm.o, d)) != KG_OK) return r;
            CK(norm(lw.g2));
            GemmArgs g = base;
            g.N = F; g.K = d; g.rowscale = rs; g.hi = fh; g.lo = fl; g.ldp = F;
            gm_plan(g, F / (GM_TM / 2), pairs, m->lay.pf_part_bytes);
            if ((r = gm_launch<PF_SWIGLU>(g, m->pf.x[0][g.nt / GM_NT_STEP - 1], m->pf.x[1][g.nt / GM_NT_STEP - 1], tm.gate, tm.up, pairs, s)) != KG_OK) return r;
            if ((r = resid(tm.down, F)) != KG_OK) return r;
            if (i == c.exit_layer - 1) {                              // the adapter's K / V
                CK(norm(m->layers_host[L].g1));
                if ((r = qkv(m->pf.adapter_kv, L, 1)) != KG_OK) return r;
            }
        }
        CK(cudaGetLastError());
    }
    // LM head on the last prompt row (still in h): the decode path's fused head operator on one row
    {
        pack_rows_kernel<<<m->nctas, 256, 0, s>>>(h + (size_t)last * d, d, 1, d, D.g_final, D.hA_pk, d * 4, D.ssq_hA, m->nctas);
        LinArgs a{};
        a.W = D.head; a.N = c.vocab; a.K = d; a.M = 1; a.x = h + (size_t)last * d; a.ldx = d; a.gain = D.g_final; a.eps = c.rms_eps;
        a.xpk = D.hA_pk; a.ldpk = d * 4; a.ssq_in = D.ssq_hA; a.ld_ssq = m->nctas;
        a.epi = EPI_HEAD; a.scale = c.logit_scale; a.head_part = D.head_part;
        a.logits_dbg = c.debug_logits ? D.dbg_verify : nullptr; a.ld_dbg = c.vocab;
        lin_phases(a);
        op_linear_kernel<WT, 4, false><<<m->nctas, BLOCK_THREADS, SMEM_TOTAL, s>>>(a);
        pf_finish_kernel<<<1, 32, 0, s>>>(D.head_part, m->nctas, D.st, D.out_tokens, n, err);
        CK(cudaGetLastError());
    }
    return KG_OK;
}

}  // namespace

extern "C" int kg_debug_set_prefill_mode(kg_model* m, int mode) {
    if (!m || (mode != 0 && mode != 1)) return KG_E_ARG;
    m->prefill_mode = mode;
    return KG_OK;
}

extern "C" int kg_debug_prompt_attention(int32_t H, int32_t hd, int32_t pos0, int32_t rows, const void* qh, const void* ql, const void* kc, const void* vc,
                                         const int32_t* page_table, int32_t page_size, int32_t n_pages, int32_t kernel, int32_t skip,
                                         void* oh, void* ol, int32_t* err, void* stream) {
    if (!qh || !ql || !kc || !vc || !page_table || !oh || !ol || !err) return KG_E_ARG;
    for (const void* p : {qh, ql, kc, vc, (const void*)oh, (const void*)ol}) if (!aligned16(p)) return KG_E_ARG;
    if ((reinterpret_cast<uintptr_t>(page_table) & 3u) || (reinterpret_cast<uintptr_t>(err) & 3u)) return KG_E_ARG;
    if (H < 1 || H > 256 || (hd != 64 && hd != 128) || pos0 < 0 || rows < 1 || rows > PF_ROWS || pos0 > (1 << 24) || page_size < 1 || (page_size & (page_size - 1)) ||
        n_pages < 1 || kernel < 0 || kernel > 2) return KG_E_ARG;
    if ((long long)n_pages * H > 0x7fffffff / page_size) return KG_E_LIMIT;
    typedef __nv_bfloat16 WT;
    FaArgs fa;
    fa.qh = (const WT*)qh; fa.ql = (const WT*)ql; fa.kc = (const WT*)kc; fa.vc = (const WT*)vc; fa.oh = (WT*)oh; fa.ol = (WT*)ol;
    fa.page_table = page_table; fa.n_phys = n_pages; fa.st = nullptr; fa.H = H; fa.pos0 = pos0; fa.rows = rows; fa.row0 = 0; fa.err = err; fa.skip = skip;
    for (fa.ps_shift = 0; (1 << fa.ps_shift) < page_size; ++fa.ps_shift) {}
    CUtensorMap tmk, tmv;
    const uint64_t crows = (uint64_t)n_pages * H * page_size;
    const int box = page_size < 16 ? page_size : 16;
    if (!make_tmap(&tmk, kc, crows, hd, box) || !make_tmap(&tmv, vc, crows, hd, box)) return tmap_failed();
    int r = hd == 128 ? attention_attributes<128>() : attention_attributes<64>();
    if (r != KG_OK) return r;
    cudaStream_t s = (cudaStream_t)stream;
    CK(cudaMemsetAsync(err, 0, 4, s));
    return launch_prompt_attention(fa, hd, kernel == 2 || (kernel == 0 && prompt_attention_tc(fa)), tmk, tmv, s);
}

extern "C" int kg_op_gemm(const void* W, int32_t N, int32_t K, const float* x, int32_t M, const float* resid, float* out,
                          void* scratch, void* stream) {
    if (!W || !x || !out || !scratch || M < 1 || N < 1 || K < 1) return KG_E_ARG;
    if (!aligned16(W) || !aligned16(x) || !aligned16(resid) || !aligned16(out) || !aligned16(scratch)) return KG_E_ARG;
    if (N % (GM_TM / 2) || K % GM_BK) return KG_E_ARG;
    const int rows_pad = (M + 127) / 128 * 128;
    OpScratch sc = op_layout();
    if ((size_t)rows_pad * K * 4 > 4 * (size_t)KG_M_MAX * S_CAP * 8192) return KG_E_LIMIT;  // both planes live in the split-partial scratch
    if (!encode_tiled_fn()) { std::snprintf(g_cuda_err, sizeof(g_cuda_err), "cuTensorMapEncodeTiled is not available"); return KG_E_CUDA; }
    cudaStream_t s = (cudaStream_t)stream;
    __nv_bfloat16* hi = (__nv_bfloat16*)((char*)scratch + sc.off_po);
    __nv_bfloat16* lo = hi + (size_t)rows_pad * K;
    const int nctas = sm_count();
    GemmArgs g{};
    g.rows = M; g.N = N; g.K = K; g.C = out; g.resid = resid; g.ldc = N;
    g.part = (float*)((char*)scratch + sc.off_gemm); g.cnt = (unsigned*)((char*)scratch + sc.off_gcnt); g.err = (int*)g.cnt + OP_GEMM_CNT;
    CK(cudaMemsetAsync(g.cnt, 0, 4 * (OP_GEMM_CNT + 1), s));
    const int r = gemm_attributes<PF_STORE>();
    if (r != KG_OK) return r;
    gm_plan(g, (N + GM_TM - 1) / GM_TM, nctas / 2, nctas <= OP_GEMM_CNT ? OP_GEMM_PART : 0);
    pf_split_kernel<<<dim3(M, (K / 4 + PF_EW_THREADS - 1) / PF_EW_THREADS), PF_EW_THREADS, 0, s>>>(x, K, K, hi, lo);
    CUtensorMap th, tl, tw;
    if (!make_tmap(&th, hi, M, K, g.nt / 2) || !make_tmap(&tl, lo, M, K, g.nt / 2) || !make_tmap(&tw, W, N, K, GM_TM / 2)) return tmap_failed();
    return gm_launch<PF_STORE>(g, th, tl, tw, tw, nctas / 2, s);
}
