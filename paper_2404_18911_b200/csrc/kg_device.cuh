// Device-side building blocks of the Kangaroo decode step for sm_100a.
//
// Everything here is written as __device__ "operators" that every CTA of a persistent,
// cooperatively launched grid executes in lock step: each operator splits its work by
// (cta, nctas); its readers poll for the rows it writes, or a grid-wide barrier comes between.  The same operators are
// also wrapped one-by-one in small kernels for unit tests.
//
// A CTA has 8 consumer warps and one producer warp (the decode kernel a sequencer and a prefetch warp besides).  The decode step is bound by HBM bandwidth:
// every weight byte is read exactly once per pass.  The producer warp streams this CTA's share of
// every weight matrix of a pass through a ring of shared-memory slots with bulk asynchronous
// copies (cp.async.bulk + mbarrier transaction counts); because weights do not depend on
// activations it runs ahead of the consumers across operator boundaries and grid barriers, so HBM
// stays busy while the consumers synchronise.  The consumers read weight tiles with ldmatrix and
// feed tensor-core MMAs whose "M" side is the weight tile and whose "N" side is the 1..16
// activation rows (activations split into bf16 hi + lo so that the product keeps fp32 accuracy).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace kg {

constexpr int M_MAX = 16;          // rows per pass
constexpr int NTHREADS = 256;      // consumer threads per CTA
constexpr int NWARPS = NTHREADS / 32;
constexpr int BLOCK_THREADS = NTHREADS + 32;   // + the producer warp (warp index NWARPS)
// The decode kernel is launched with a whole warpgroup behind the consumers (warp NWARPS copies, the next one is the sequencer, then
// the prefetch warp; one leaves at once): registers are handed out per warpgroup, and that warpgroup gives most of its share to the two consumer
// warpgroups at kernel start (setmaxnreg).  The pool is what the launch allocated: 384 threads x 168 registers = 64512; a
// request beyond it would block forever, so the budgets below are checked against it.
constexpr int DECODE_THREADS = NTHREADS + 128;
constexpr int LAUNCH_REGS = 168;                  // 65536 / 384, rounded down to the allocation unit of 8
constexpr int CONSUMER_REGS = 216, PRODUCER_REGS = 72;
static_assert(NTHREADS * CONSUMER_REGS + 128 * PRODUCER_REGS <= DECODE_THREADS * LAUNCH_REGS, "register budgets exceed the CTA's pool");
static_assert(DECODE_THREADS * (LAUNCH_REGS + 8) > 65536, "LAUNCH_REGS is not what a launch of DECODE_THREADS threads gets");
constexpr int S_CAP = 16;          // most KV splits per head
constexpr int HD_MAX = 128;

// weight ring: RING slots of ST_ROWS weight rows x ST_K k-elements (bf16); rows are padded by 16
// bytes so that the eight row addresses of an ldmatrix fall into distinct bank groups
constexpr int RING = 6;
constexpr int ST_ROWS = 8;
constexpr int ST_K = 2048;
constexpr int ST_ROW_BYTES = ST_K * 2 + 16;
constexpr int SLOT_BYTES = ST_ROWS * ST_ROW_BYTES;
constexpr int CTRL_BYTES = 3072;
constexpr int QUEUE = 8;                                // operators in the queue: more than one layer's
constexpr int RING_OFF = CTRL_BYTES;
constexpr int WORK_OFF = RING_OFF + RING * SLOT_BYTES;
constexpr int SMEM_TOTAL = 232448;                      // 227 KB, the most one CTA may own
constexpr int WORK_BYTES = SMEM_TOTAL - WORK_OFF;       // activations, reductions, attention tiles
constexpr int SC_ROWS = 256;                            // rows whose accumulators live in shared memory at once
// the plain path never runs beside the streamed one in a launch, so it stages its activations over the ring too
constexpr int SIMPLE_XS_BYTES = SMEM_TOTAL - RING_OFF - 4096;

constexpr int BAR_STRIDE = 32;                          // words between the arrival counter and the count of CTAs that have left (a 128-byte line each)
constexpr int BAR_BYTES = 256;
constexpr unsigned long long WAIT_TIMEOUT_CLK = 6000000000ull;   // default budget of a device-side wait: ~3 s at 1.9 GHz

enum { EPI_STORE = 0, EPI_RESID = 1, EPI_SWIGLU = 2, EPI_HEAD = 3 };
enum { ST_OK = 0, ST_TIMEOUT = -6, ST_INTERNAL = -8 };

struct LayerW {
    const void* wqkv; const void* wo; const void* wgate; const void* wup; const void* wdown;
    const float* g1; const float* g2;
};

struct Dims {
    int L, d, H, hd, F, V, l;
    float eps, theta, logit_scale;
    int max_seq, page_size, n_pages, gamma_max, debug;
    int n_phys;         // physical pages behind the page table (page numbers must lie below it)
    int ps_shift;       // log2(page_size): page sizes are powers of two
    int ring;           // 1: attention reads K / V tiles from the weight ring (streamed path, bf16 cache, head_dim 64 / 128)
    int stream;         // 1: linear operators take the streamed tensor-core path (bf16, d and F multiples of 16)
};

// Device-resident sequence / round state (one int-sized field per line of the method's notation).
struct State {
    int P;              // position of x_0 = tokens held by the shallow and deep KV caches
    int len_A;          // tokens held by the adapter's KV cache (P or P-1)
    int x0;             // the round's first token
    int pending;        // 1: a drafted unit awaits kg_verify
    int n_d;            // drafts kept this round
    int n_steps;        // adapter+head passes this round
    int M, k_acc, n_emit;
    int total;          // tokens in out_tokens (x_0 of prefill included)
    int rounds;
    int draft_steps_total, drafted_total, accepted_total;
    int status;         // 0 or a negative kg_status set by a device-side wait that gave up
    int timeout_where;
    int draft_tok[M_MAX];
    float conf[M_MAX];
    int emitted[M_MAX];
    int target[M_MAX];
    // the last word: 1 after a wait that gave up, until the model is built anew (exchange words and counters may hold anything)
    int timed_out;
};

struct Dev {
    alignas(64) CUtensorMap tmk;   // the K and V caches as [rows][hd], in boxes of up to 16 rows x 64 dims (dm.ring)
    alignas(64) CUtensorMap tmv;
    Dims dm;
    const void* embed; const void* head; const float* g_final;
    const LayerW* layers;          // [L+1], index L = adapter
    void* kcache; void* vcache;    // [(L+1)][n_pages][H][page_size][hd]
    const int* page_table;         // [n_pages] logical -> physical page
    float* h;                      // [M_MAX][d] residual stream of the pass
    float* feat;                   // [M_MAX+1][d]: slot 0 = early feature of position P-1, slot 1+j = f_j
    float* abuf;                   // [2][d] adapter output rows
    // Rows exchanged inside a layer, two instances used by turns: row m of an instance is xch_ld words long and holds q, k, v
    // [3d], the attention output [d], the residual stream after attention [d], the SwiGLU output [F] and the sums of squares
    // of the residual stream [nctas].  All but q, k, v and the sums are packed rows (streamed path) or fp32 rows (plain path).
    unsigned* xch[2]; int xch_ld;
    // packed copies (streamed path; row = 4 bytes per element) and per-CTA sums of squares [row][nctas]
    unsigned char* hA_pk;          // [M_MAX][d]   residual stream scaled for the next QKV / the LM head
    unsigned char* featA_pk;       // [M_MAX+1][d] early features scaled by the adapter's input gain
    unsigned char* featD_pk;       // [M_MAX+1][d] early features scaled by the first deep layer's gain
    unsigned char* abuf_pk;        // [2][d]       adapter output scaled by its last gain
    float* ssq_hA;                 // [M_MAX][nctas]
    float* ssq_feat;               // [M_MAX+1][nctas]
    float* ssq_abuf;               // [2][nctas]
    float* att_po;                 // [M_MAX][H][S_CAP][hd] split partial outputs
    float* att_ml;                 // [M_MAX][H][S_CAP][2]  split partial (max, sum)
    unsigned* att_cnt;             // [H] arrival counters
    unsigned* att_xp;              // ring attention: [M_MAX][H][S_CAP][hd + 4] split partials; in the decode kernel exchange words (empty between uses)
    const float2* rope;            // [max_seq][hd / 2] cos, sin (null: computed where needed)
    float4* head_part;             // [nctas][M_MAX] (zmax, sumexp, argmax bits, -)
    float* dbg_draft; float* dbg_verify;   // [M_MAX][V] each (debug only)
    int* out_tokens; int* S; int* round_log;   // [max_seq], [max_seq], [max_seq][4]
    const int* prompt;             // device copy of the prompt
    State* st;
    unsigned* bar;                 // grid barrier arrival counter, and the count of CTAs that have left: both zero between launches
    double inv_freq[HD_MAX / 2];   // theta^(-2i/hd)
};

struct Ctrl;

// State of one role (consumers / producer warp) of the CTA.  It lives in shared memory: every thread of the role
// holds the same values, updates are the same in all of them, and between operators they are ordered by the
// role's barriers; reading it never touches the per-thread stack.
struct Ctx {
    int cta, nctas;
    unsigned bar_target;           // arrivals expected at the next grid barrier (thread 0 only)
    unsigned long long wait_clk;   // clocks after which a wait of this launch gives up
    State* st; unsigned* bar;
    int skip_arrival;              // test hook: 1 + index of the CTA that leaves out its first grid-barrier arrival (0: none)
    char* smem;
    Ctrl* ctl;
    bool grid;                     // false: single-operator test kernel, grid barriers are CTA barriers
    bool producer;                 // this thread belongs to the copy warp
    int backoff;                   // nanoseconds to sleep between two polls of a shared-memory barrier
    int slot; unsigned phase;      // ring cursor of this thread's role
    unsigned issued;               // producer: stages issued so far
    unsigned mail_phase;           // producer: parity of the next result it waits for
};

// ------------------------------------------------------------------------------------ operators
struct PkOut { const float* gain; unsigned char* ptr; };   // packed copy of output rows; gain == null: unscaled

struct LinArgs {
    const void* W; const void* W2;   // [N, K]; W2 != null: SwiGLU pair (gate, up)
    int N, K;
    int M;                           // activation rows
    int spw, nph;                    // streamed path: k16-steps per warp and phase, phases (lin_phases)
    const float* x; int ldx;         // plain path: fp32 rows (written earlier in this kernel)
    const float* gain; float eps;    // RMSNorm gain of the input (null: no norm)
    const unsigned char* xpk; int ldpk;   // streamed path: packed rows, already multiplied by the gain; bytes per row
    const float* ssq_in; int ld_ssq; // streamed path with norm: [M] rows of nctas partial sums of squares of the input rows
    int poll;                        // 1: the input rows and their sums are exchange words, to be polled
    const float* resid; int ldr;     // EPI_RESID
    float* out; int ldo;             // fp32 output rows (streamed path: nullable)
    int epi;
    float scale;                     // EPI_HEAD: logit scale
    float4* head_part;               // EPI_HEAD: [nctas][M_MAX]
    float* logits_dbg; int ld_dbg;   // EPI_HEAD, optional
    PkOut pk[2]; int ldpk_out;       // streamed path: packed copies of the output rows for the operators that read them
    float* ssq_out; int ld_sout;     // streamed path: [M] rows of nctas partial sums of squares of the output rows (nullable)
};

// Cut of a head's keys into S splits of `chunk` (ra_plan: tiles of the old keys, ntile of them; ka_plan: keys); pos: the position it was made for
struct AttPlan { int ntile, S, chunk; int pos; };
struct AttArgs {
    AttPlan plan;          // cut into splits (ring attention and single operator)
    int row0;              // ring attention: first row of this layer's cache in the tensor maps
    const float* qkv; int ldq;      // [M] rows of raw q, k, v of this pass
    int poll;              // 1: q, k, v are exchange words, to be polled
    int M, pos0;           // rows sit at positions pos0 .. pos0+M-1; row i sees keys 0 .. pos0+i
    void* kc; void* vc;    // this layer's cache: [n_pages][H][page_size][hd]
    float* out; int ldo;   // [M] rows of d (nullable)
    unsigned char* opk; int ldopk;  // packed copy of out for the output projection (nullable); bytes per row
};
struct EmbedArgs { const int* toks; int tok, M; };        // toks == null: the one token `tok`

enum { OPK_NONE = 0, OPK_LIN = 1, OPK_ATT = 2, OPK_EMBED = 3, OPK_HEAD = 4, OPK_MAIL = 5, OPK_KEEP = 6, OPK_EXIT = 7 };
// One operator in the queue of the decode kernel.
struct Op {
    int kind;
    int sync;                        // != 0: a grid barrier follows (and this is where it says it timed out)
    int empty_p, empty_rows;         // OPK_ATT, OPK_EXIT: rows of this exchange instance are emptied afterwards
    union { LinArgs lin; AttArgs att; EmbedArgs emb; };
};

// Per-CTA control block at the start of shared memory.
struct Ctrl {
    unsigned long long full[RING];     // producer -> consumers: slot filled (transaction count)
    unsigned long long empty[RING];    // consumers -> producer: slot drained (one arrival per consumer warp)
    unsigned long long mail;           // consumers -> sequencer: head_tok / head_p hold a new result
    int abort;                         // a bounded wait of this CTA gave up
    int sync_ok;
    int att_last;
    unsigned issued;                   // stages that the copy warp has issued, for the prefetch warp
    int head_tok[M_MAX];
    float head_p[M_MAX];
    unsigned long long qfull[QUEUE];   // sequencer -> copy warp, prefetch warp, consumers: operator written
    unsigned long long qempty[QUEUE];  // copy warp, prefetch warp (of launches that have one), consumer warps -> sequencer: operator done
    Op queue[QUEUE];
    // the per-role context (struct Ctx): one copy each for the consumers, the copy warp, the sequencer and the prefetch warp
    alignas(16) unsigned char ctx[4][128];
};
static_assert(sizeof(Ctrl) <= CTRL_BYTES - 16, "control block too large");

// ------------------------------------------------------------------------------------ helpers

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float ldcg_f(const float* p) { return __ldcg(p); }
__device__ __forceinline__ float2 ldcg_f2(const float* p) { return __ldcg(reinterpret_cast<const float2*>(p)); }
__device__ __forceinline__ float4 ldcg_f4(const float* p) { return __ldcg(reinterpret_cast<const float4*>(p)); }

// The thread index, read anew by every operator: the operators are inlined into one loop, and what is computed from an index that
// the compiler knows to be the same every time round would be kept, and spilled, across all of them.
__device__ __forceinline__ int tid_here() { int t; asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t)); return t; }

// barrier among the consumer warps only (the producer warp never takes part)
__device__ __forceinline__ void cta_sync() { asm volatile("bar.sync 1, %0;" ::"n"(NTHREADS) : "memory"); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.b32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// global -> shared bulk copy; bytes and both addresses are multiples of 16.  `policy` is an L2 cache policy made by
// l2_evict_first(): weights are read once per pass, so their lines are the first to go, and what the pass re-reads
// (activations, K/V of the draft layers, barrier words) stays in L2 while 1-65 GB of weights stream past it.
__device__ __forceinline__ void bulk_g2s(void* dst_smem, const void* src, unsigned bytes, unsigned long long* bar, unsigned long long policy) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                 ::"r"(smem_u32(dst_smem)), "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy) : "memory");
}
__device__ __forceinline__ unsigned long long l2_evict_first() {
    unsigned long long p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// The top bit of the grid barrier's arrival counter tells every CTA that some wait has given up: they learn it from
// the word they poll anyway, without a second load.
constexpr unsigned BAR_ABORT = 0x80000000u;       // the host bounds a launch's arrivals below 2^31 (max_seq check)
__device__ __forceinline__ void record_timeout(Ctx& c, int where) {
    *(volatile int*)&c.ctl->abort = 1;
    if (c.st) {
        atomicCAS(&c.st->status, 0, ST_TIMEOUT);
        c.st->timeout_where = where;
        *(volatile int*)&c.st->timed_out = 1;
    }
    if (c.grid && c.bar) atomicOr(c.bar, BAR_ABORT);
}

// Bounded wait on an mbarrier phase.  Returns false when this CTA has given up (here or elsewhere).
__device__ __forceinline__ bool mbar_wait(Ctx& c, unsigned long long* bar, unsigned parity, int where) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    unsigned spins = 0;
    while (!mbar_try_wait(bar, parity)) {
        // the copy warp and the sequencer share issue ports with consumer warps: they back off instead of spinning
        if (c.backoff) __nanosleep(c.backoff);
        if (((++spins) & 63u) == 0u) {
            if (*(volatile int*)&c.ctl->abort) return false;
            if ((unsigned long long)(clock64() - t0) > c.wait_clk) { record_timeout(c, where); return false; }
        }
    }
    return true;
}

__device__ __forceinline__ void ldmatrix_x4(unsigned (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Programmatic dependent launch: a kernel launched with that attribute may start early; what it reads of its predecessor's
// results it reads after the wait (a no-op in an ordinary launch).
__device__ __forceinline__ void grid_dependents_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

template <typename WT> __device__ __forceinline__ float wt_to_float(WT v);
template <> __device__ __forceinline__ float wt_to_float<float>(float v) { return v; }
template <> __device__ __forceinline__ float wt_to_float<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename WT> __device__ __forceinline__ WT float_to_wt(float v);
template <> __device__ __forceinline__ float float_to_wt<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 float_to_wt<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

template <typename WT> __device__ __forceinline__ float4 load4_cg(const WT* p);
template <> __device__ __forceinline__ float4 load4_cg<float>(const float* p) { return __ldcg(reinterpret_cast<const float4*>(p)); }
template <> __device__ __forceinline__ float4 load4_cg<__nv_bfloat16>(const __nv_bfloat16* p) {
    const uint2 r = __ldcg(reinterpret_cast<const uint2*>(p));
    return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u),
                       __uint_as_float(r.y << 16), __uint_as_float(r.y & 0xffff0000u));
}

// (better, z, idx): larger z wins; on equal z the lower index wins.
__device__ __forceinline__ bool arg_better(float za, int ia, float zb, int ib) {
    return za > zb || (za == zb && ia < ib);
}

// ------------------------------------------------------------------------------------ CTA set-up
// Called by every thread of the CTA at kernel start; returns the context of the thread's role.  prefetch: a prefetch warp reads the queue.
__device__ __forceinline__ Ctx& ctx_init(char* smem, State* st, unsigned* bar, bool grid,
                                         unsigned long long wait_clk = WAIT_TIMEOUT_CLK, int skip_arrival = 0, bool prefetch = false) {
    static_assert(sizeof(Ctx) <= 128, "context slot too small");
    Ctrl* ctl = reinterpret_cast<Ctrl*>(smem);
    const int role = threadIdx.x < NTHREADS ? 0 : (threadIdx.x < NTHREADS + 32 ? 1 : (threadIdx.x < NTHREADS + 64 ? 2 : 3));   // consumers, copy warp, sequencer, prefetch warp
    Ctx& c = *reinterpret_cast<Ctx*>(ctl->ctx[role]);
    if (threadIdx.x == 0 || threadIdx.x == NTHREADS || threadIdx.x == NTHREADS + 32 || threadIdx.x == NTHREADS + 64) {
        c.cta = blockIdx.x; c.nctas = gridDim.x; c.bar_target = 0; c.st = st; c.bar = bar; c.smem = smem;
        c.wait_clk = wait_clk; c.skip_arrival = skip_arrival;
        c.ctl = ctl; c.grid = grid;
        c.producer = role == 1; c.backoff = role == 0 ? 0 : (role == 2 ? 40 : 200);
        c.slot = 0; c.phase = 0; c.issued = 0; c.mail_phase = 0;
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < RING; ++i) { mbar_init(&ctl->full[i], 1); mbar_init(&ctl->empty[i], NWARPS); }
        for (int i = 0; i < QUEUE; ++i) { mbar_init(&ctl->qfull[i], 1); mbar_init(&ctl->qempty[i], NWARPS + 1 + prefetch); }
        mbar_init(&ctl->mail, 1);
        ctl->abort = 0; ctl->sync_ok = 1; ctl->att_last = 0; ctl->issued = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    return c;
}

// ------------------------------------------------------------------------------------ grid barrier
// Consumer threads only.  Monotonic arrival counter; every wait is bounded.  On expiry the kernel
// records KG_E_TIMEOUT in the state word and every CTA leaves at its next barrier.  Returns false
// when the grid must stop (the same value in every consumer thread of the CTA).
__device__ __forceinline__ bool grid_sync(Ctx& c, int where) {
    if (!c.grid) { cta_sync(); return *(volatile int*)&c.ctl->abort == 0; }
    cta_sync();
    if (threadIdx.x == 0) {
        // bar[0] counts arrivals (monotonic over the launch, below 2^31: the host bounds max_seq accordingly): one
        // release-add, then poll until every CTA has arrived or the abort bit appears
        c.bar_target += (unsigned)c.nctas;
        const unsigned gen = c.bar_target;
        if (c.skip_arrival == c.cta + 1) c.skip_arrival = 0;        // test hook: this arrival never happens
        else asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(c.bar) : "memory");
        int ok = 1;
        {
            const long long t0 = clock64();
            unsigned spins = 0;
            while (true) {
                const unsigned v = ld_acquire_u32(c.bar);
                if (v & BAR_ABORT) { ok = 0; break; }
                if (v >= gen) break;
                if (((++spins) & 63u) == 0u) {
                    if ((unsigned long long)(clock64() - t0) > c.wait_clk) { record_timeout(c, where); ok = 0; break; }
                }
            }
        }
        if (!ok) *(volatile int*)&c.ctl->abort = 1;          // lets the producer warp leave its waits
        c.ctl->sync_ok = ok;
    }
    cta_sync();
    return *(volatile int*)&c.ctl->sync_ok != 0;
}

// Thread 0 of every CTA, behind its last barrier.  A launch finds the arrival counter at zero and leaves it so: the last CTA to
// come here clears it, when no CTA polls it any more.  (Nothing about it is kept on the host, so that a captured launch can be
// replayed.)  A launch that gave up leaves the abort bit, which ends every later launch at its first barrier.
__device__ __forceinline__ void grid_leave(const Ctx& c) {
    if (atomicInc(c.bar + BAR_STRIDE, (unsigned)c.nctas - 1u) == (unsigned)c.nctas - 1u) *(volatile unsigned*)c.bar = 0u;
}

// ------------------------------------------------------------------------------------ exchange inside a layer
// Between the operators of a layer there is no grid barrier.  A word that has not been written holds XCH_EMPTY, and a
// reader polls the words that it needs; a word that holds anything else is the value itself, so neither the writer's
// stores nor the reader's loads need any order among themselves.  XCH_EMPTY is a NaN that no arithmetic produces: results
// that are NaN come out as 0x7fffffff (fp32) and 0x7fff (bf16), whatever their inputs.
//
// A barrier costs the release of the writer's stores - slow while the CTA's weight copies are in flight -, the serialised
// arrivals, the polling of the counter and then the fetch of the data; the exchange is one store and one polled load.  Four of
// the five barriers of a layer went this way: 7B, KV 512, verify pass of one row 3.08 -> 2.74 ms, of seven rows 3.60 -> 3.42,
// greedy step 3.22 -> 2.87, single draft step 0.352 -> 0.328; the fp32 model of four layers (with the plain path's loads issued
// ahead) 18.1 -> 7.3 ms for 64 tokens.  What was measured on the way: polling a few words before the first full read costs one
// more round trip (+2 % of a pass), checking each step's words at its MMA brings calls and spills into the inner loop (+17 %).
//
// Two instances of the buffers are used by turns, one per layer.  While a layer uses one of them, the other one, which the
// layer before used, is filled with XCH_EMPTY again; the grid barrier at the end of every layer stands between the last
// read of an instance and its refill, and between the refill and its next use.
constexpr unsigned XCH_EMPTY = 0xffffffffu;
__device__ __forceinline__ unsigned xch_ld1(const unsigned* p) { unsigned v; asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p)); return v; }
__device__ __forceinline__ uint2 xch_ld2(const void* p) { uint2 v; asm volatile("ld.relaxed.gpu.global.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p)); return v; }
__device__ __forceinline__ uint4 xch_ld4(const void* p) {
    uint4 v;
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ void xch_st(unsigned* p, unsigned v) { asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory"); }
__device__ __forceinline__ void xch_st4(void* p, uint4 v) { asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory"); }
__device__ __forceinline__ void xch_stf(float* p, float v) { xch_st(reinterpret_cast<unsigned*>(p), __float_as_uint(v)); }
__device__ __forceinline__ bool xch_empty(const uint2& v) { return v.x == XCH_EMPTY || v.y == XCH_EMPTY; }
__device__ __forceinline__ bool xch_empty(const uint4& v) { return v.x == XCH_EMPTY || v.y == XCH_EMPTY || v.z == XCH_EMPTY || v.w == XCH_EMPTY; }

// Called by a thread whose poll came back empty: true = poll again, false = give up (here or elsewhere).  `spins` starts at 0.
struct XchSpin { unsigned spins; long long t0; };
__device__ __noinline__ bool xch_check(Ctx& c, long long t0, int where) {
    if (*(volatile int*)&c.ctl->abort) return false;
    if ((unsigned long long)(clock64() - t0) > c.wait_clk) { record_timeout(c, where); return false; }
    return true;
}
__device__ __forceinline__ bool xch_again(Ctx& c, XchSpin& sp, int where) {
    if (sp.spins == 0u) sp.t0 = clock64();
    return ((++sp.spins) & 31u) != 0u || xch_check(c, sp.t0, where);
}

// ------------------------------------------------------------------------------------ RoPE
// cos / sin of pos * theta^(-2i/hd): the angle is formed and reduced to [-pi, pi] in double, the
// trigonometric functions are evaluated in fp32 on the reduced argument.
__device__ __forceinline__ void rope_cs(const Dev& D, int pos, int i, float& cs, float& sn) {
    double a = (double)pos * D.inv_freq[i];
    const double two_pi = 6.283185307179586476925286766559;
    double k = rint(a / two_pi);
    float r = (float)(a - k * two_pi);
    sincosf(r, &sn, &cs);
}

// ------------------------------------------------------------------------------------ linear operator
// A packed copy of activation rows: the row is cut into k16 blocks of 64 bytes; the 16 bytes at
// blk*64 + tt*16 hold {hi(k), hi(k+8), lo(k), lo(k+8)} for k = 16 blk + 2 tt, each a pair of bf16
// (elements k, k+1) with x * gain = hi + lo.  This is the B operand fragment order of the MMA, so a
// consumer lane fetches its fragments with plain 8- or 16-byte loads.  The operator that produces a
// row writes it once, in this form, for the operator that reads it.

// byte offset of the hi half of element k inside a packed row; the lo half sits 8 bytes further
__device__ __forceinline__ size_t pk_off(int k) {
    return (size_t)(k >> 4) * 64 + (size_t)(((k & 7) >> 1) * 16 + ((k >> 3) & 1) * 4 + (k & 1) * 2);
}
__device__ __forceinline__ void pk_store(unsigned char* row, int k, float v) {
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    const __nv_bfloat16 l = __float2bfloat16_rn(v - __bfloat162float(h));
    unsigned char* p = row + pk_off(k);
    *reinterpret_cast<__nv_bfloat16*>(p) = h;
    *reinterpret_cast<__nv_bfloat16*>(p + 8) = l;
}

// The same for two neighbouring elements k (even), k + 1, as whole words
__device__ __forceinline__ void pk_store2(unsigned char* row, int k, float v0, float v1) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
    const float2 f = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(v0 - f.x, v1 - f.y);
    unsigned* p = reinterpret_cast<unsigned*>(row + pk_off(k));
    xch_st(p, *reinterpret_cast<const unsigned*>(&h));
    xch_st(p + 2, *reinterpret_cast<const unsigned*>(&l));
}
// Called by whole warps whose neighbouring lanes hold neighbouring elements (k even in even lanes)
__device__ __forceinline__ void pk_store_lane(unsigned char* row, int k, float v) {
    const float o = __shfl_xor_sync(0xffffffffu, v, 1);
    if (!(k & 1)) pk_store2(row, k, v, o);
}


__device__ __forceinline__ float silu_f(float v) { return v / (1.0f + expf(-v)); }

// Running (max, argmax, sum exp) of one logit row, merged in a fixed order.
struct HeadStat { float zmax; float sum; int arg; };
__device__ __forceinline__ void head_merge(HeadStat& a, float zmax, float sum, int arg) {
    if (sum == 0.0f) return;
    if (a.sum == 0.0f) { a.zmax = zmax; a.sum = sum; a.arg = arg; return; }
    if (arg_better(zmax, arg, a.zmax, a.arg)) {
        a.sum = a.sum * expf(a.zmax - zmax) + sum;
        a.zmax = zmax; a.arg = arg;
    } else {
        a.sum = a.sum + sum * expf(zmax - a.zmax);
    }
}

// ---- streamed tensor-core path (bf16 weights, K a multiple of 16) -----------------------------------
//
// Work split.  The CTA owns a contiguous range of "units": output rows, or for the SwiGLU pair
// gate/up feature pairs.  A stage of the ring holds 8 weight rows (for the pair: the 8 gate rows of
// a feature group, then in the next stage the 8 up rows of the same features) times one k phase
// (at most 2048 k-elements when M <= 12, else 1024; lin_phases), i.e. one bulk copy of up to 4 KB per row: the copy
// engine spends a fixed time per copy, and only copies of 2-4 KB and more keep HBM saturated.
// The stages are visited superchunk (<= 256 accumulator rows) -> phase -> row group, in the same
// order by the producer warp (which issues the copies) and the consumers.
//
// Consumers take the stages two at a time: one MMA m16n8k16 computes D[weight row, activation
// column] with the 16 weight rows of a stage pair as the A operand (ldmatrix straight from the
// ring) and the activations as the 8-column B operand.  The activations keep fp32 accuracy by a
// split x * gain = hi + lo into two bf16 parts:
//   V = 4  (M <= 4):  columns 0-3 carry hi, columns 4-7 lo of rows 0-3: one MMA per k16-step;
//   V = 8  (M <= 8):  hi and lo are two MMAs;
//   V = 12 (M <= 12): the same for rows 0-7, and a third MMA carries hi and lo of rows 8-11 as V = 4 does for rows 0-3
//                     (7B, KV 512, verify pass of 11 rows: 5.47 ms with the four MMAs on 1024-k phases of V = 16, now 4.46);
//   V = 16 (M <= 16): two column tiles, hi and lo: four MMAs.
// Each of the 8 warps owns a fixed slice of the phase's k range; its B fragments are loaded once
// per phase from the packed activation rows in global memory (L2) and stay in registers for every
// row group, so the steady state touches shared memory only for the weights.  After a stage pair the 8 partial sums of each (weight row,
// activation row) are added in warp order into the per-row accumulators in shared memory.  Operators of few stage pairs per phase and more than one
// phase (O, down: d / 148 rows a CTA) leave that for the end: a warp's sums of a pair grow in place in shared memory, from phase to phase,
// and no warp waits for another before the last phase is through.  The barrier and the cross-warp sum take 0.3 to 0.4 of a pair's 1400 to
// 1800 clocks, and with two pairs between two fetches of fragments nothing hid them (7B, KV 512, 12 layers, verify pass of 1 row
// 0.905 -> 0.897, of 4 rows 0.988 -> 0.960, of 7 rows 1.118 -> 1.077, of 11 rows 1.400 -> 1.364, of 16 rows 1.719 -> 1.634 ms).  With one
// phase there is nothing to save (a model of four layers with d = 512: 1 % slower that way).  What does not fit the work area: QKV,
// gate / up, the head.
template <int V> struct LinGeom {
    static constexpr int NS = V == 16 ? 8 : 16;           // most k16-steps per warp and phase: 2048 or 1024 k-elements of a CTA
    static constexpr int FR = V == 4 ? 2 : (V == 8 ? 4 : (V == 12 ? 6 : 8));   // B fragment registers per step
    static constexpr int NACC = V == 16 ? 2 : 1;          // column tiles
    static constexpr int RED_W = V == 16 ? 256 : (V == 12 ? 192 : 128);        // floats of one warp's partial sums of a stage pair
    static constexpr int MP = V == 12 ? 12 : 16;          // row accumulator columns (activation rows, padded)
    // partial sums are double-buffered where the work area has room (V = 16: one buffer and one more barrier per pair);
    // partial sums and row accumulators together take the same space in every variant
    static constexpr int ACC_OFF = V == 16 ? NWARPS * RED_W : 2 * NWARPS * RED_W;
    static constexpr int FEWP = V <= 8 ? 4 : (V == 12 ? 3 : 2);                // stage pairs per phase whose sums can be kept warp by warp
    static constexpr int COLS = V == 4 ? 4 : (V == 8 ? 8 : MP);                // activation rows of a stage pair's sums
};
constexpr int FEW_ACC_OFF = 4608;                          // row accumulators behind the sums of few pairs
constexpr int MP_MAX = 16;

// First of the units (of N) that belong to CTA `cta`: even, so that a packed word has one writer.
__device__ __forceinline__ int cta_unit(int N, int cta, int nctas) {
    const int u = 2 * (int)((unsigned)((N + 1) >> 1) * (unsigned)cta / (unsigned)nctas);      // N * nctas < 2^32 (checked on the host)
    return min(u, N);
}

// The phases of an operator: as many as the longest possible ones and, up to 8 rows, all but the last of the same length, a whole number
// of steps for every warp.  With phases of the full length the last one may be short, and its copies with it: K = 6656 was 3 x 2048 +
// 512, now 4 x 1664 (verify pass of one row, 33B widths, 8 layers 1.104 -> 1.023 ms; 13B, 12 layers, KV 2048 1.370 -> 1.319; 7B, whose d is
// two full phases, 7 rows 1.072 -> 1.049).  The error stays what it was: linear operators of 2064 to 17920 k against float64 2.40e-6 to 2.51e-6 of the
// norm both ways at every row count, bias at 6656 k -9.8e-8 -> -8.1e-8 (7 rows).  Beyond 8 rows the phases are left as they were.  It is not the error:
// that is the same there too (9 to 12 rows of 6656 k 2.45e-6, bias -9.4e-8 and with equal phases -7.7e-8), and 9 to 12 rows would be 2 to 6 %
// faster.  But rows of short prompts go there, and the largest deviation of a confidence in the stored 33B trace, which its test holds to 4e-3,
// is anything from 3.4e-3 to 5.4e-3 with the order of the same sums (as it is 3.4e-3).
__host__ __device__ __forceinline__ void lin_phases(LinArgs& a) {
    const unsigned steps = (unsigned)a.K >> 4, most = (unsigned)(a.M <= 12 ? LinGeom<12>::NS : LinGeom<16>::NS) * NWARPS;
    const unsigned n = (steps + most - 1) / most;
    a.spw = a.M <= 8 ? (int)(((steps + n - 1) / n + NWARPS - 1) / NWARPS) : (int)(most / NWARPS);
    a.nph = (int)((steps + a.spw * NWARPS - 1) / (a.spw * NWARPS));
}

struct LinPlan {
    int u0, u1;          // this CTA's units
    int sc_units;        // units per superchunk
    int plen, nph;       // k phases
};

__device__ __forceinline__ LinPlan make_plan(const LinArgs& a, int cta, int nctas) {
    LinPlan p;
    p.u0 = cta_unit(a.N, cta, nctas);
    p.u1 = cta_unit(a.N, cta + 1, nctas);
    p.sc_units = a.W2 ? SC_ROWS / 2 : SC_ROWS;
    p.plen = a.spw * (16 * NWARPS);
    p.nph = a.nph;
    return p;
}

// Producer warp: issue the bulk copies of every stage of this operator.  PUBLISH: for a prefetch warp, which only the decode kernel has.
template <bool PUBLISH>
__device__ __noinline__ bool lin_produce(const LinArgs& a, Ctx& c) {
    const int lane = threadIdx.x & 31;
    const LinPlan pl = make_plan(a, c.cta, c.nctas);
    const bool dual = a.W2 != nullptr;
    const __nv_bfloat16* W = reinterpret_cast<const __nv_bfloat16*>(a.W);
    const __nv_bfloat16* W2 = reinterpret_cast<const __nv_bfloat16*>(a.W2);
    char* ring = c.smem + RING_OFF;
    Ctrl* ctl = c.ctl;
    int slot = c.slot; unsigned phase = c.phase; unsigned issued = c.issued;     // ring cursor, kept in registers here
    const unsigned long long policy = l2_evict_first();
    for (int sc0 = pl.u0; sc0 < pl.u1; sc0 += pl.sc_units) {
        const int sc1 = min(pl.u1, sc0 + pl.sc_units);
        const int ngrp = (sc1 - sc0 + ST_ROWS - 1) / ST_ROWS;
        const int nst = dual ? 2 * ngrp : ngrp;
        for (int ph = 0; ph < pl.nph; ++ph) {
            const int p0 = ph * pl.plen, len = min(pl.plen, a.K - p0);
            for (int si = 0; si < nst; ++si) {
                const int base = sc0 + (dual ? si >> 1 : si) * ST_ROWS;
                const int nvalid = min(ST_ROWS, sc1 - base);
                const __nv_bfloat16* src = ((dual && (si & 1)) ? W2 : W) + (size_t)(base + lane) * a.K + p0;
                int ok = 1;
                if (lane == 0) ok = mbar_wait(c, &ctl->empty[slot], phase ^ 1u, 40) ? 1 : 0;
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) { c.slot = slot; c.phase = phase; c.issued = issued; return false; }
                if (lane == 0) mbar_arrive_expect_tx(&ctl->full[slot], (unsigned)(nvalid * len * 2));
                __syncwarp();
                if (lane < nvalid) bulk_g2s(ring + (size_t)slot * SLOT_BYTES + lane * ST_ROW_BYTES, src, (unsigned)(len * 2), &ctl->full[slot], policy);
                issued++;
                if (PUBLISH && lane == 0) *(volatile unsigned*)&ctl->issued = issued;
                if (++slot == RING) { slot = 0; phase ^= 1u; }
            }
        }
    }
    c.slot = slot; c.phase = phase; c.issued = issued;
    return true;
}

// ---- the prefetch warp of the decode kernel: weights on their way into L2 before the ring has room for them
//
// The ring holds 4.4 us of HBM's time, but the consumers stand still for longer at the hand-overs around the attention and at a
// layer's end (about 9 and 6 us of a layer's 80 in the 7B shape at one row), and HBM with them.  A stage is therefore prefetched
// into L2 once the copy warp is less than PF_AHEAD stages away from it; afterwards the ring is filled from L2, faster than HBM could.
// Depth, 7B, 12 layers, KV 512, one row (ms): none 0.894, 8 stages 0.887, 10 0.874, 12 0.861, 14 0.850, 16 0.866, 24 1.041, 32 1.295
// (at 32 KB a stage and 148 CTAs 16 stages are 78 MB: not all of the 126 MB of L2 can be used that way); 33B widths 1.023 -> 0.998 / 0.995 /
// 0.996 / 1.009 (8 to 14; a stage of its phases is 26 KB), KV 4096 1.010 -> 0.995 / 0.989 / 0.978 / 0.983, 13B 1.319 -> 1.323 / 1.312 / 1.299 / 1.298.
// Passes of more than PF_ROWS_MAX rows keep the consumers busier than HBM, and the additional traffic costs them: 11 rows 1.362 -> 1.398, 16
// rows 1.635 -> 1.708 (7 rows 1.049 -> 1.008, 8 rows 1.080 -> 1.028).
constexpr int PF_AHEAD = 12, PF_ROWS_MAX = 8;
constexpr int PF_GAVE_UP = -0x40000000;
__device__ __forceinline__ void bulk_prefetch_l2(const void* src, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
// One operator.  c.issued counts the stages of the operators before it, as the copy warp counts them; stages that the copy warp has issued
// already are left out.  False: a wait gave up.
__device__ __noinline__ bool lin_prefetch(const LinArgs& a, Ctx& c) {
    const int lane = threadIdx.x & 31;
    const LinPlan pl = make_plan(a, c.cta, c.nctas);
    const bool dual = a.W2 != nullptr;
    const __nv_bfloat16* W = reinterpret_cast<const __nv_bfloat16*>(a.W);
    const __nv_bfloat16* W2 = reinterpret_cast<const __nv_bfloat16*>(a.W2);
    unsigned n = c.issued;
    __syncwarp();                                          // every lane has read the count before one writes it again
    for (int sc0 = pl.u0; sc0 < pl.u1; sc0 += pl.sc_units) {
        const int sc1 = min(pl.u1, sc0 + pl.sc_units);
        const int ngrp = (sc1 - sc0 + ST_ROWS - 1) / ST_ROWS;
        const int nst = dual ? 2 * ngrp : ngrp;
        if (a.M > PF_ROWS_MAX) { n += (unsigned)(pl.nph * nst); continue; }
        for (int ph = 0; ph < pl.nph; ++ph) {
            const int p0 = ph * pl.plen, len = min(pl.plen, a.K - p0);
            for (int si = 0; si < nst; ++si, ++n) {
                int gap = 0;                               // stages between the copy warp and this one
                if (lane == 0) {
                    const long long t0 = clock64();
                    while ((gap = (int)(n - *(volatile unsigned*)&c.ctl->issued)) >= PF_AHEAD) {
                        __nanosleep(100);
                        if (*(volatile int*)&c.ctl->abort || (unsigned long long)(clock64() - t0) > 2ull * c.wait_clk) { gap = PF_GAVE_UP; break; }
                    }
                }
                gap = __shfl_sync(0xffffffffu, gap, 0);
                if (gap == PF_GAVE_UP) return false;
                if (gap < 1) continue;                     // on its way already
                const int base = sc0 + (dual ? si >> 1 : si) * ST_ROWS;
                const int nvalid = min(ST_ROWS, sc1 - base);
                if (lane < nvalid) bulk_prefetch_l2(((dual && (si & 1)) ? W2 : W) + (size_t)(base + lane) * a.K + p0, (unsigned)(len * 2));
            }
        }
    }
    __syncwarp();
    if (lane == 0) c.issued = n;
    return true;
}

// Producer warp, after a failed wait: let the copies it still has in flight land before the CTA exits.
__device__ void ring_drain(Ctx& c) {
    if ((threadIdx.x & 31) != 0) return;
    const unsigned n = c.issued < (unsigned)RING ? c.issued : (unsigned)RING;
    int s = c.slot; unsigned ph = c.phase;
    for (unsigned i = 0; i < n; ++i) {
        if (--s < 0) { s = RING - 1; ph ^= 1u; }
        const long long t0 = clock64();
        while (!mbar_try_wait(&c.ctl->full[s], ph)) {
            if ((unsigned long long)(clock64() - t0) > c.wait_clk) break;
        }
    }
}

__device__ __forceinline__ void split_hi_lo(float2 v, unsigned& hi, unsigned& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
    const float2 f = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(v.x - f.x, v.y - f.y);
    hi = *reinterpret_cast<const unsigned*>(&h);
    lo = *reinterpret_cast<const unsigned*>(&l);
}

// Shared-memory work area of the streamed path (floats, from WORK_OFF).
constexpr int LW_RED = 0;                                 // partial sums of a stage pair, then at LinGeom::ACC_OFF the row accumulators [SC_ROWS][MP]
constexpr int LW_RS = 2 * NWARPS * 128 + SC_ROWS * MP_MAX;   // [M_MAX] 1/rms of the input rows
constexpr int LW_RSP = LW_RS + M_MAX;                     // [16] partial sums of squares of the input rows
constexpr int LW_SSW = LW_RSP + 16;                       // [NWARPS][M_MAX] sums of squares of the output rows
constexpr int PRE_NU = 64;                                // residual / gain values are prefetched for up to this many units
constexpr int LW_PRES = LW_SSW + NWARPS * M_MAX;          // [M_MAX][PRE_NU] residual values
constexpr int LW_PREG = LW_PRES + M_MAX * PRE_NU;         // [2][PRE_NU] gains of the packed outputs
constexpr int LW_HS = LW_PREG + 2 * PRE_NU;               // [M_MAX][3] LM head: running maximum, sum, arg max of each row (kept here and not
                                                          // in registers, which the fragments of the wide variants fill)
constexpr int LW_END = LW_HS + M_MAX * 3;
static_assert(LW_END * 4 <= WORK_BYTES, "linear work area too large");
template <int V> constexpr bool FEW_FITS = LinGeom<V>::FEWP * NWARPS * LinGeom<V>::RED_W <= FEW_ACC_OFF && FEW_ACC_OFF + LinGeom<V>::FEWP * 16 * LinGeom<V>::MP <= LW_RS;
static_assert(FEW_FITS<4> && FEW_FITS<8> && FEW_FITS<12> && FEW_FITS<16>, "sums of few pairs");
static_assert(LinGeom<12>::ACC_OFF + SC_ROWS * LinGeom<12>::MP <= LW_RS && LinGeom<16>::ACC_OFF + SC_ROWS * 16 <= LW_RS && LinGeom<8>::ACC_OFF + SC_ROWS * 16 <= LW_RS,
              "partial sums and accumulators overlap what follows");

__device__ __forceinline__ void cp_async4(void* dst_smem, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
}

// Epilogue of the streamed path for everything but the LM head: turns the accumulators of nu output
// units x M rows (acc_s with MP columns, 1/rms in rs) into fp32 rows, packed copies and per-CTA sums of squares.
// Thread (r, m): m = tid mod 2^ceil(log2 M), so that the lanes of a warp that share m can add their
// squares by shuffles in a fixed order.  Outputs with a packed copy have an even number of features.  Every consumer thread calls it; ssq_acc (threads < M)
// accumulates over superchunks.
template <int MP>
__device__ __forceinline__ void emit_rows(const LinArgs& a, float* wk, const float* acc_s, int sc0, int nu, bool prefetched, float& ssq_acc) {
    const int tid = tid_here(), lane = tid & 31, warp = tid >> 5;
    const int M = a.M;
    const float* rs = wk + LW_RS;
    float* ssw = wk + LW_SSW;
    const int sh = M <= 1 ? 0 : (M <= 2 ? 1 : (M <= 4 ? 2 : (M <= 8 ? 3 : 4)));
    const int mp = 1 << sh;
    const int m = tid & (mp - 1);
    float ssl = 0.f;
    // whole warps go round together: two neighbouring rows of W, in lanes mp apart, make one packed word
    for (int rb = warp * (32 >> sh); rb < nu; rb += NTHREADS >> sh) {
        const int r = rb + (lane >> sh);
        const bool valid = r < nu && m < M;
        const int row = sc0 + r;
        float v = 0.f;
        if (valid) {
            if (a.epi == EPI_SWIGLU) {
                const int srow = (r >> 3) * 16 + (r & 7);
                v = silu_f(acc_s[(size_t)srow * MP + m] * rs[m]) * (acc_s[(size_t)(srow + 8) * MP + m] * rs[m]);
            } else {
                v = acc_s[(size_t)r * MP + m] * rs[m];
                if (a.epi == EPI_RESID)
                    v += prefetched ? wk[LW_PRES + m * PRE_NU + r] : ldcg_f(a.resid + (size_t)m * a.ldr + sc0 + r);
            }
            if (a.out) xch_stf(a.out + (size_t)m * a.ldo + row, v);
            ssl += v * v;
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (a.pk[q].ptr) {
                float pv = v;
                if (valid && a.pk[q].gain) pv *= prefetched ? wk[LW_PREG + q * PRE_NU + r] : __ldg(a.pk[q].gain + row);
                const float po = __shfl_xor_sync(0xffffffffu, pv, mp);
                if (valid && !(r & 1)) pk_store2(a.pk[q].ptr + (size_t)m * a.ldpk_out, row, pv, po);
            }
        }
    }
    if (a.ssq_out) {
        for (int o = 16; o >= mp; o >>= 1) ssl += __shfl_xor_sync(0xffffffffu, ssl, o);
        if (lane < mp) ssw[warp * M_MAX + lane] = ssl;
        cta_sync();
        if (tid < M) {
            float sres = 0.f;
            for (int w = 0; w < NWARPS; ++w) sres += ssw[w * M_MAX + tid];
            ssq_acc += sres;
        }
    }
}

// log2 of the threads that add the sums of squares of one of M rows
__device__ __forceinline__ int sum_shift(int M) { return M <= 1 ? 8 : (M <= 2 ? 7 : (M <= 4 ? 6 : (M <= 8 ? 5 : 4))); }

// FEW: compiled with the sums of few pairs (a single operator that has no use for them is launched without).
template <int V, bool FEW>
__device__ __forceinline__ void lin_consume(const LinArgs& a, Ctx& c) {
    using G = LinGeom<V>;
    constexpr int NS = G::NS, FR = G::FR, NACC = G::NACC, MP = G::MP;
    const int tid = tid_here(), lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int M = a.M, K = a.K, spw = a.spw;
    const bool dual = a.W2 != nullptr;
    const LinPlan pl = make_plan(a, c.cta, c.nctas);

    float* wk = reinterpret_cast<float*>(c.smem + WORK_OFF);
    float* red = wk + LW_RED;
    float* rs = wk + LW_RS;
    const char* ring = c.smem + RING_OFF;
    Ctrl* ctl = c.ctl;
    const int nctas = c.nctas, cta = c.cta;
    int slot = c.slot; unsigned phase = c.phase;              // ring cursor, kept in registers here

    bool ok = true;
    int buf = 0;
    float ssq_acc = 0.f;

    // ---- fetched early, used in the epilogue: residual values, output gains (the requests go out behind the first phase's
    // fragment loads, which the first MMA waits for)
    const int nu0 = min(pl.u1 - pl.u0, pl.sc_units);
    const bool prefetched = nu0 <= PRE_NU;
    bool pre_pending = true;
    auto epilogue_prefetch = [&]() {
        if (prefetched && a.epi != EPI_HEAD) {
            if (a.epi == EPI_RESID)
                for (int i = tid; i < M * nu0; i += NTHREADS) cp_async4(wk + LW_PRES + (i / nu0) * PRE_NU + i % nu0, a.resid + (size_t)(i / nu0) * a.ldr + pl.u0 + i % nu0);
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (a.pk[q].ptr && a.pk[q].gain)
                    for (int i = tid; i < nu0; i += NTHREADS) cp_async4(wk + LW_PREG + q * PRE_NU + i, a.pk[q].gain + pl.u0 + i);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    for (int sc0 = pl.u0; sc0 < pl.u1; sc0 += pl.sc_units) {
        const int sc1 = min(pl.u1, sc0 + pl.sc_units);
        const int nu = sc1 - sc0;
        const int ngrp = (nu + ST_ROWS - 1) / ST_ROWS;
        const int nst = dual ? 2 * ngrp : ngrp;
        const bool few = FEW && pl.nph > 1 && (nst + 1) >> 1 <= G::FEWP;
        float* acc_s = wk + (few ? FEW_ACC_OFF : G::ACC_OFF);
        for (int ph = 0; ph < pl.nph; ++ph) {
            const int p0 = ph * pl.plen, len = min(pl.plen, K - p0);
            const int nsteps = len / 16;
            // ---- B fragments of this warp's k slice, kept in registers for every row group of the phase.  Every load is issued
            // before any is used; exchange words are read again until all of them are there.  Rows >= M re-read a valid row: their
            // columns of the product are never read, and the columns of an MMA do not mix.  Steps past the end of the phase re-read
            // the last one and are skipped.
            unsigned fr[NS][FR];
            const int last = min(nsteps - 1 - warp * spw, spw - 1);      // last valid step of this warp (< 0: none)
            {
                // this lane's rows of the packed input: V = 4: row g & 3 (hi for g < 4, lo for g >= 4); else row g and, mofs bytes
                // away, V = 12: row 8 + (g & 3) (hi for g < 4, lo for g >= 4), V = 16: row 8 + g (M > 8 here, so that g < M)
                const int xrow = V == 4 ? (g & 3) : g, mrow = 8 + (V == 12 ? (g & 3) : g);
                const int mofs = ((mrow < M ? mrow : 0) - xrow) * a.ldpk + (V == 12 ? (g >> 2) * 8 : 0);
                const unsigned char* pbase = a.xpk + (size_t)(xrow < M ? xrow : 0) * a.ldpk + (size_t)(p0 / 16 + warp * spw) * 64 + t * 16 + (V == 4 ? (g >> 2) * 8 : 0);
                int lastv = last;
                XchSpin sp; sp.spins = 0;
                while (true) {
                    asm volatile("" : "+l"(pbase), "+r"(lastv));   // keeps the steps' addresses from being formed, and spilled, ahead of the loop
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        const unsigned char* px = pbase + (size_t)max(min(s, lastv), -warp * spw) * 64;
                        if (V == 4) {
                            const uint2 v = xch_ld2(px);
                            fr[s][0] = v.x; fr[s][1] = v.y;
                        } else {
                            const uint4 v = xch_ld4(px);
                            fr[s][0] = v.x; fr[s][1] = v.y; fr[s][2] = v.z; fr[s][3] = v.w;
                            if (V == 16) {
                                const uint4 w = xch_ld4(px + mofs);
                                fr[s][FR - 4] = w.x; fr[s][FR - 3] = w.y; fr[s][FR - 2] = w.z; fr[s][FR - 1] = w.w;
                            }
                            if (V == 12) {
                                const uint2 w = xch_ld2(px + mofs);
                                fr[s][FR - 2] = w.x; fr[s][FR - 1] = w.y;
                            }
                        }
                    }
                    if (!a.poll || !ok) break;
                    bool empty = false;
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
#pragma unroll
                        for (int i = 0; i < FR; ++i) empty |= fr[s][i] == XCH_EMPTY;
                    }
                    if (!__any_sync(0xffffffffu, empty)) break;
                    if (!__all_sync(0xffffffffu, xch_again(c, sp, 43))) ok = false;
                }
            }
            if (pre_pending) { pre_pending = false; epilogue_prefetch(); }
            // ---- the row groups of this phase, two stages (16 weight rows) at a time
            const uint32_t a_lane = (uint32_t)((lane & 7) * ST_ROW_BYTES + (warp * spw * 16 + (lane >> 4) * 8) * 2);
            for (int si = 0; si < nst; si += 2) {
                const bool two = si + 1 < nst;
                const int slot_a = slot;
                const int slot_b = two ? (slot_a + 1 == RING ? 0 : slot_a + 1) : slot_a;
                const unsigned phase_b = (two && slot_a + 1 == RING) ? phase ^ 1u : phase;
                float acc[5][4];
#pragma unroll
                for (int q = 0; q < 5; ++q) { acc[q][0] = acc[q][1] = acc[q][2] = acc[q][3] = 0.f; }
                if (ok) ok = mbar_wait(c, &ctl->full[slot_a], phase, 41);
                if (ok && two) ok = mbar_wait(c, &ctl->full[slot_b], phase_b, 41);
                if (ok) {
                    // ldmatrix x4: matrices 0, 2 = rows 0-7 (first stage), 1, 3 = rows 8-15 (second stage); k halves 0-7 | 8-15
                    const uint32_t a_base = smem_u32(ring + (size_t)((lane & 8) ? slot_b : slot_a) * SLOT_BYTES) + a_lane;
                    // the weight fragments are fetched PD steps ahead of the MMA that uses them (the loads and the MMAs
                    // issue in program order, so a load right before its MMA would expose its latency at every step);
                    // loads past the phase's last step stay inside the slot and are never used
                    constexpr int PD = V == 4 ? 4 : 2;
                    unsigned af[PD][4];
#pragma unroll
                    for (int s = 0; s < PD; ++s) ldmatrix_x4(af[s], a_base + (uint32_t)s * 32u);
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        if (s <= last) {
                            if (V == 4) {
                                mma_bf16_16816(acc[s & 3], af[s % PD], fr[s][0], fr[s][1]);
                            } else if (V == 8) {
                                mma_bf16_16816(acc[(s & 1) * 2], af[s % PD], fr[s][0], fr[s][1]);
                                mma_bf16_16816(acc[(s & 1) * 2 + 1], af[s % PD], fr[s][2], fr[s][3]);
                            } else if (V == 12) {
                                // chains of eight where hi is summed (as V = 8 and V = 16 have them); lo, 2^-9 of it, in one
                                mma_bf16_16816(acc[s & 1], af[s % PD], fr[s][0], fr[s][1]);
                                mma_bf16_16816(acc[4], af[s % PD], fr[s][2], fr[s][3]);
                                mma_bf16_16816(acc[2 + (s & 1)], af[s % PD], fr[s][FR - 2], fr[s][FR - 1]);
                            } else {
                                mma_bf16_16816(acc[0], af[s % PD], fr[s][0], fr[s][1]);
                                mma_bf16_16816(acc[1], af[s % PD], fr[s][2], fr[s][3]);
                                mma_bf16_16816(acc[2], af[s % PD], fr[s][FR - 4], fr[s][FR - 3]);
                                mma_bf16_16816(acc[3], af[s % PD], fr[s][FR - 2], fr[s][FR - 1]);
                            }
                        }
                        if (s + PD < NS) ldmatrix_x4(af[s % PD], a_base + (uint32_t)(s + PD) * 32u);
                    }
                }
                __syncwarp();
                if (ok && lane == 0) { mbar_arrive(&ctl->empty[slot_a]); if (two) mbar_arrive(&ctl->empty[slot_b]); }
                slot = slot_b; phase = phase_b;
                if (++slot == RING) { slot = 0; phase ^= 1u; }
                // ---- add the k-slices in warp order into the row accumulators
                if (V == 16 && !few) cta_sync();             // single partial-sum buffer: the previous pair's sums have been read
                float* r = red + (size_t)((few ? si >> 1 : (V == 16 ? 0 : buf)) * NWARPS + warp) * G::RED_W;
                // few pairs: onto the sums of the phases before (each word has one thread)
                const bool add = few && ph != 0;
                auto put = [&](float* q, float x, float y) {
                    float2 o = make_float2(0.f, 0.f);
                    if (add) o = *reinterpret_cast<const float2*>(q);
                    *reinterpret_cast<float2*>(q) = make_float2(o.x + x, o.y + y);
                };
                if (V == 12) {
                    // acc[0], acc[1]: hi of rows 0-7 (even, odd steps), acc[4]: lo; acc[2], acc[3]: rows 8-11, hi in columns 0-3 and lo
                    // in columns 4-7, which sit two lanes further
                    put(r + g * MP + 2 * t, acc[0][0] + acc[1][0] + acc[4][0], acc[0][1] + acc[1][1] + acc[4][1]);
                    put(r + (g + 8) * MP + 2 * t, acc[0][2] + acc[1][2] + acc[4][2], acc[0][3] + acc[1][3] + acc[4][3]);
                    float mx[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) { mx[i] = acc[2][i] + acc[3][i]; mx[i] += __shfl_xor_sync(0xffffffffu, mx[i], 2); }
                    if (t < 2) {
                        put(r + g * MP + 8 + 2 * t, mx[0], mx[1]);
                        put(r + (g + 8) * MP + 8 + 2 * t, mx[2], mx[3]);
                    }
                } else if (V == 16) {
                    // acc[0] / acc[1]: hi / lo of columns 0-7; acc[2] / acc[3]: hi / lo of columns 8-15
                    put(r + g * 8 + 2 * t, acc[0][0] + acc[1][0], acc[0][1] + acc[1][1]);
                    put(r + (g + 8) * 8 + 2 * t, acc[0][2] + acc[1][2], acc[0][3] + acc[1][3]);
                    put(r + 128 + g * 8 + 2 * t, acc[2][0] + acc[3][0], acc[2][1] + acc[3][1]);
                    put(r + 128 + (g + 8) * 8 + 2 * t, acc[2][2] + acc[3][2], acc[2][3] + acc[3][3]);
                } else {
                    put(r + g * 8 + 2 * t, (acc[0][0] + acc[1][0]) + (acc[2][0] + acc[3][0]), (acc[0][1] + acc[1][1]) + (acc[2][1] + acc[3][1]));
                    put(r + (g + 8) * 8 + 2 * t, (acc[0][2] + acc[1][2]) + (acc[2][2] + acc[3][2]), (acc[0][3] + acc[1][3]) + (acc[2][3] + acc[3][3]));
                }
                if (few) {
                    if (ph != pl.nph - 1 || si + 2 < nst) continue;
                    cta_sync();
                    constexpr int EL = 16 * G::COLS;         // sums of a pair
                    for (int e = tid; e < ((nst + 1) >> 1) * EL; e += NTHREADS) {
                        const int pr = e / EL, r16 = e % EL / G::COLS, m = e % G::COLS;
                        const float* rb = red + (size_t)pr * NWARPS * G::RED_W + (V == 16 ? (m >> 3) * 128 + r16 * 8 + (m & 7) : r16 * (V == 12 ? 12 : 8) + m);
                        float v[NWARPS];
#pragma unroll
                        for (int w = 0; w < NWARPS; ++w) v[w] = V == 4 ? rb[w * G::RED_W] + rb[w * G::RED_W + 4] : rb[w * G::RED_W];
#pragma unroll
                        for (int o = NWARPS / 2; o > 0; o >>= 1) {
#pragma unroll
                            for (int w = 0; w < o; ++w) v[w] += v[w + o];
                        }
                        acc_s[(size_t)(pr * 16 + r16) * MP + m] = v[0];
                    }
                    continue;
                }
                cta_sync();
                {
                    // element (weight row r16, activation row m) of the pair; for M <= 8 every thread adds a share of the
                    // eight k-slices and a fixed butterfly joins the shares, so that no warp lags behind the others
                    if (V == 12) {
                        if (tid < 192) {
                            const float* rb = red + (size_t)buf * NWARPS * G::RED_W + tid;
                            float v = 0.f;
#pragma unroll
                            for (int w = 0; w < NWARPS; ++w) v += rb[w * G::RED_W];
                            float* dst = acc_s + (size_t)(si >> 1) * 16 * MP + tid;
                            *dst = ph == 0 ? v : *dst + v;
                        }
                    } else if (V == 16) {
                        const int r16 = tid >> 4, m = tid & 15;
                        const float* rb = red + (m >> 3) * 128 + r16 * 8 + (m & 7);
                        float v = 0.f;
#pragma unroll
                        for (int w = 0; w < NWARPS; ++w) v += rb[w * NACC * 128];
                        float* dst = acc_s + (size_t)((si >> 1) * 16 + r16) * MP + m;
                        *dst = ph == 0 ? v : *dst + v;
                    } else {
                        constexpr int TPE = V == 4 ? 4 : 2;                  // threads per element
                        constexpr int WPT = NWARPS / TPE;                    // k-slices per thread
                        const int e = tid / TPE, q = tid % TPE;
                        const int r16 = V == 4 ? e >> 2 : e >> 3;
                        const int m = V == 4 ? e & 3 : e & 7;
                        const float* rb = red + (size_t)buf * NWARPS * 128 + r16 * 8 + m;
                        float v = 0.f;
#pragma unroll
                        for (int w = 0; w < WPT; ++w) v += V == 4 ? rb[(q * WPT + w) * 128] + rb[(q * WPT + w) * 128 + 4] : rb[(q * WPT + w) * 128];
#pragma unroll
                        for (int o = 1; o < TPE; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                        if (q == 0) {
                            float* dst = acc_s + (size_t)((si >> 1) * 16 + r16) * MP + m;
                            *dst = ph == 0 ? v : *dst + v;
                        }
                    }
                }
                buf ^= 1;
            }
        }
        // ---- epilogue of this superchunk
        if (sc0 == pl.u0) {
            // the input rows' sums of squares: 2^rsh threads per row, SSB partial sums of each thread per batch of loads
            // (requested here and not beside the fragments, which fill the registers: 2 % of a verify pass at M = 1)
            if (a.ssq_in) {
                constexpr int SSB = 5;
                const int rsh = sum_shift(M), rm = tid >> rsh;
                const unsigned* ssrow = reinterpret_cast<const unsigned*>(a.ssq_in + (size_t)rm * a.ld_ssq);
                float part = 0.f;
                for (int q0 = tid & ((1 << rsh) - 1); q0 < nctas; q0 += SSB << rsh) {
                    unsigned w[SSB];
                    XchSpin sp; sp.spins = 0;
                    while (true) {
                        bool empty = false;
#pragma unroll
                        for (int i = 0; i < SSB; ++i) {
                            const int q = q0 + (i << rsh);
                            w[i] = rm < M && q < nctas ? xch_ld1(ssrow + q) : 0u;
                        }
#pragma unroll
                        for (int i = 0; i < SSB; ++i) empty |= w[i] == XCH_EMPTY;
                        if (!a.poll || !empty || !xch_again(c, sp, 44)) break;
                    }
#pragma unroll
                    for (int i = 0; i < SSB; ++i) part += __uint_as_float(w[i]);
                }
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
                if ((lane & 15) == 0) wk[LW_RSP + (tid >> 4)] = part;      // 16 sums, 16 / mp of each row
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            cta_sync();
            if (tid < M_MAX) {
                float r = 1.0f;
                if (a.ssq_in && tid < M) {
                    float ss = 0.f;
                    const int per = 1 << (sum_shift(M) - 4);                          // 16 / mp
                    for (int j = 0; j < per; ++j) ss += wk[LW_RSP + tid * per + j];
                    r = rsqrtf(ss / (float)K + a.eps);
                }
                rs[tid] = r;
            }
        }
        cta_sync();
        if (a.epi == EPI_HEAD) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int m = warp + q * NWARPS;
                if (m < M) {
                    const float f = rs[m] * a.scale;
                    float zm = -INFINITY; int im = 0x7fffffff;
                    for (int r = lane; r < nu; r += 32) {
                        const float z = acc_s[(size_t)r * MP + m] * f;
                        if (a.logits_dbg) a.logits_dbg[(size_t)m * a.ld_dbg + sc0 + r] = z;
                        if (arg_better(z, sc0 + r, zm, im)) { zm = z; im = sc0 + r; }
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const float z2 = __shfl_xor_sync(0xffffffffu, zm, o);
                        const int i2 = __shfl_xor_sync(0xffffffffu, im, o);
                        if (arg_better(z2, i2, zm, im)) { zm = z2; im = i2; }
                    }
                    float e = 0.f;
                    for (int r = lane; r < nu; r += 32) e += expf(acc_s[(size_t)r * MP + m] * f - zm);
                    e = warp_sum(e);
                    if (lane == 0) {                 // this warp tracks rows warp, warp + 8
                        HeadStat hs; hs.zmax = 0.f; hs.sum = 0.f; hs.arg = 0;
                        float* st = wk + LW_HS + m * 3;
                        if (sc0 != pl.u0) { hs.zmax = st[0]; hs.sum = st[1]; hs.arg = __float_as_int(st[2]); }
                        head_merge(hs, zm, e, im);
                        st[0] = hs.zmax; st[1] = hs.sum; st[2] = __int_as_float(hs.arg);
                    }
                }
            }
        } else {
            emit_rows<MP>(a, wk, acc_s, sc0, nu, prefetched && sc0 == pl.u0, ssq_acc);
        }
        cta_sync();                                  // acc_s is rewritten by the next superchunk / operator
    }
    if (a.epi == EPI_HEAD && lane == 0) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int m = warp + q * NWARPS;
            if (m < M) {
                const float* st = wk + LW_HS + m * 3;
                a.head_part[(size_t)cta * M_MAX + m] = pl.u0 < pl.u1 ? make_float4(st[0], st[1], st[2], 0.f) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    }
    if (a.epi != EPI_HEAD && a.ssq_out && tid < M) xch_stf(a.ssq_out + (size_t)tid * a.ld_sout + cta, ssq_acc);
    c.slot = slot; c.phase = phase;
}

// Rows that do not come out of a linear operator (token embeddings): every CTA takes its slice of
// the d columns, places the values where the epilogue expects accumulators and emits them like
// an operator output (fp32 rows, packed copies, sums of squares).  value(m, e) is given by the caller.
template <typename F>
__device__ __forceinline__ void emit_plain_rows(LinArgs& a, Ctx& c, F value) {
    const int tid = threadIdx.x;
    float* wk = reinterpret_cast<float*>(c.smem + WORK_OFF);
    const int u0 = cta_unit(a.N, c.cta, c.nctas), u1 = cta_unit(a.N, c.cta + 1, c.nctas);
    float ssq_acc = 0.f;
    a.epi = EPI_STORE;
    if (tid < M_MAX) wk[LW_RS + tid] = 1.0f;
    for (int sc0 = u0; sc0 < u1; sc0 += SC_ROWS) {
        const int nu = min(SC_ROWS, u1 - sc0);
        for (int idx = tid; idx < nu * a.M; idx += NTHREADS) {
            const int r = idx % nu, m = idx / nu;
            wk[LinGeom<8>::ACC_OFF + (size_t)r * MP_MAX + m] = value(m, sc0 + r);
        }
        cta_sync();
        emit_rows<MP_MAX>(a, wk, wk + LinGeom<8>::ACC_OFF, sc0, nu, false, ssq_acc);
        cta_sync();
    }
    if (a.ssq_out && tid < a.M) xch_stf(a.ssq_out + (size_t)tid * a.ld_sout + c.cta, ssq_acc);
}

// Plain path for any storage type (fp32 models, odd shapes, and a cross-check of the tensor-core path): activations staged in
// shared memory as fp32, one output row per warp at a time.  What bounds it on a small model is latency: the first weights of
// a warp's row are requested before the activations are waited for, and a row's sums are formed with 16-byte loads.
constexpr int SIMPLE_PF = 6;                              // 16-byte groups of a weight row per lane and batch: 768 elements
template <typename WT>
__device__ __forceinline__ void simple_fetch(const WT* row, int k0, int K, float4 (&w)[SIMPLE_PF]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < SIMPLE_PF; ++j) {
        const int k = k0 + j * 128 + lane * 4;
        w[j] = k < K ? load4_cg<WT>(row + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}
template <typename WT, int MB>
__device__ __forceinline__ void simple_rows(const LinArgs& a, Ctx& c, const float* xs, const float* rs, float4 (&w1)[SIMPLE_PF], float4 (&w2)[SIMPLE_PF], HeadStat& hs) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int M = a.M, K = a.K;
    const bool dual = a.W2 != nullptr;
    const int first = c.cta * NWARPS + warp, step = c.nctas * NWARPS;
    for (int row = first; row < a.N; row += step) {
        const WT* wr = reinterpret_cast<const WT*>(a.W) + (size_t)row * K;
        const WT* wr2 = reinterpret_cast<const WT*>(a.W2) + (size_t)row * K;
        float acc[MB], acc2[MB];
#pragma unroll
        for (int m = 0; m < MB; ++m) { acc[m] = 0.f; acc2[m] = 0.f; }
        for (int k0 = 0; k0 < K; k0 += SIMPLE_PF * 128) {
            if (row != first || k0 != 0) { simple_fetch<WT>(wr, k0, K, w1); if (dual) simple_fetch<WT>(wr2, k0, K, w2); }
#pragma unroll
            for (int j = 0; j < SIMPLE_PF; ++j) {
                const int k = k0 + j * 128 + lane * 4;
                if (k < K) {
#pragma unroll
                    for (int m = 0; m < MB; ++m) {
                        if (m < M) {
                            const float4 x = *reinterpret_cast<const float4*>(xs + (size_t)m * K + k);
                            acc[m] = fmaf(w1[j].w, x.w, fmaf(w1[j].z, x.z, fmaf(w1[j].y, x.y, fmaf(w1[j].x, x.x, acc[m]))));
                            if (dual) acc2[m] = fmaf(w2[j].w, x.w, fmaf(w2[j].z, x.z, fmaf(w2[j].y, x.y, fmaf(w2[j].x, x.x, acc2[m]))));
                        }
                    }
                }
            }
        }
        float v = 0.f, v2 = 0.f;                         // lane m takes row m
#pragma unroll
        for (int m = 0; m < MB; ++m) {
            if (m < M) {
                const float s1 = warp_sum(acc[m]);
                if (lane == m) v = s1;
                if (dual) { const float s2 = warp_sum(acc2[m]); if (lane == m) v2 = s2; }
            }
        }
        if (lane < M) {
            v *= rs[lane];
            if (a.epi == EPI_HEAD) {
                v *= a.scale;
                if (a.logits_dbg) a.logits_dbg[(size_t)lane * a.ld_dbg + row] = v;
                head_merge(hs, v, 1.0f, row);
            } else {
                if (a.epi == EPI_SWIGLU) v = silu_f(v) * (v2 * rs[lane]);
                if (a.epi == EPI_RESID) v += ldcg_f(a.resid + (size_t)lane * a.ldr + row);
                xch_stf(a.out + (size_t)lane * a.ldo + row, v);
            }
        }
    }
}
template <typename WT>
__device__ __noinline__ void lin_simple(const LinArgs& a, Ctx& c) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int M = a.M, K = a.K;
    char* work = c.smem + RING_OFF;
    float* xs = reinterpret_cast<float*>(work);                          // [M][K]
    float* rs = reinterpret_cast<float*>(work + SIMPLE_XS_BYTES);        // [M_MAX]
    float* wst = rs + M_MAX;                                             // [NWARPS][M_MAX][3] head stats

    float4 w1[SIMPLE_PF], w2[SIMPLE_PF];
    {
        const int first = c.cta * NWARPS + warp;
        const int row = min(first, a.N - 1);
        simple_fetch<WT>(reinterpret_cast<const WT*>(a.W) + (size_t)row * K, 0, K, w1);
        if (a.W2) simple_fetch<WT>(reinterpret_cast<const WT*>(a.W2) + (size_t)row * K, 0, K, w2);
    }
    cta_sync();                                          // the staging area of the operator before has been read
    for (int m = warp; m < M; m += NWARPS) {
        float ss = 0.f;
        for (int k0 = 0; k0 < K; k0 += SIMPLE_PF * 128) {
            uint4 x[SIMPLE_PF];
            XchSpin sp; sp.spins = 0;
            while (true) {
                bool empty = false;
#pragma unroll
                for (int j = 0; j < SIMPLE_PF; ++j) {
                    const int k = k0 + j * 128 + lane * 4;
                    x[j] = make_uint4(0u, 0u, 0u, 0u);
                    if (k < K) x[j] = xch_ld4(a.x + (size_t)m * a.ldx + k);
                    empty |= xch_empty(x[j]);
                }
                if (!a.poll || !empty || !xch_again(c, sp, 46)) break;
            }
#pragma unroll
            for (int j = 0; j < SIMPLE_PF; ++j) {
                const int k = k0 + j * 128 + lane * 4;
                if (k < K) {
                    float4 v = make_float4(__uint_as_float(x[j].x), __uint_as_float(x[j].y), __uint_as_float(x[j].z), __uint_as_float(x[j].w));
                    ss += (v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w);
                    if (a.gain) { const float4 gv = __ldg(reinterpret_cast<const float4*>(a.gain + k)); v.x *= gv.x; v.y *= gv.y; v.z *= gv.z; v.w *= gv.w; }
                    *reinterpret_cast<float4*>(xs + (size_t)m * K + k) = v;
                }
            }
        }
        ss = warp_sum(ss);
        if (lane == 0) rs[m] = a.gain ? rsqrtf(ss / (float)K + a.eps) : 1.0f;
    }
    cta_sync();

    HeadStat hs; hs.zmax = 0.f; hs.sum = 0.f; hs.arg = 0;               // lane m tracks row m
    if (M == 1) simple_rows<WT, 1>(a, c, xs, rs, w1, w2, hs);
    else if (M <= 4) simple_rows<WT, 4>(a, c, xs, rs, w1, w2, hs);
    else if (M <= 8) simple_rows<WT, 8>(a, c, xs, rs, w1, w2, hs);
    else simple_rows<WT, M_MAX>(a, c, xs, rs, w1, w2, hs);
    if (a.epi == EPI_HEAD) {
        if (lane < M) {
            wst[(warp * M_MAX + lane) * 3 + 0] = hs.zmax;
            wst[(warp * M_MAX + lane) * 3 + 1] = hs.sum;
            wst[(warp * M_MAX + lane) * 3 + 2] = __int_as_float(hs.arg);
        }
        cta_sync();
        if (tid < M) {
            HeadStat tot; tot.zmax = 0.f; tot.sum = 0.f; tot.arg = 0;
            for (int w = 0; w < NWARPS; ++w)
                head_merge(tot, wst[(w * M_MAX + tid) * 3 + 0], wst[(w * M_MAX + tid) * 3 + 1],
                           __float_as_int(wst[(w * M_MAX + tid) * 3 + 2]));
            a.head_part[(size_t)c.cta * M_MAX + tid] = make_float4(tot.zmax, tot.sum, __int_as_float(tot.arg), 0.f);
        }
    }
    cta_sync();
}

// Merge the per-CTA head partials of row m by a whole warp (identical result in every CTA): every lane merges the partials of CTAs lane, lane + 32, ... (independent loads, one
// round trip instead of one per CTA), then a butterfly of merges leaves the identical total in every lane (the merge
// of two partials is the same whichever of the two lanes computes it).
__device__ __forceinline__ void head_final_warp(const float4* part, int nctas, int m, int& tok, float& p) {
    const int lane = threadIdx.x & 31;
    HeadStat tot; tot.zmax = 0.f; tot.sum = 0.f; tot.arg = 0;
    for (int cta = lane; cta < nctas; cta += 32) {
        const float4 v = __ldcg(part + (size_t)cta * M_MAX + m);
        head_merge(tot, v.x, v.y, __float_as_int(v.z));
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float z = __shfl_xor_sync(0xffffffffu, tot.zmax, o);
        const float sm = __shfl_xor_sync(0xffffffffu, tot.sum, o);
        const int ar = __shfl_xor_sync(0xffffffffu, tot.arg, o);
        head_merge(tot, z, sm, ar);
    }
    tok = tot.arg;
    p = 1.0f / tot.sum;
}

// ------------------------------------------------------------------------------------ attention operator
constexpr int ATT_TK = 16;                                 // keys per tile
constexpr int ATT_RB = 4;                                  // rows per block
// Cut of a head's old tiles into splits, the same for the copy warp and the consumers.  The cost of a split count, in steps of
// one tile per warp (about 0.5 us): the tiles of an item (one step per 8 tiles, and at least the time an SM's share of the HBM
// bandwidth takes for them, 0.4 steps a tile), two steps of fixed work, three more for the merge of a head that is split.
// (Made once per position and not per layer: the 16 candidates took 2.4 us a layer in a rolled loop with divisions.)
__host__ __device__ __noinline__ inline AttPlan ra_plan(int pos0, int H, int nctas) {
    AttPlan p;
    p.ntile = (pos0 + ATT_TK - 1) / ATT_TK;
    p.S = 1;
    const float inv_ctas = 1.0f / (float)nctas;
    float best = 0.f;
    p.pos = pos0;
#pragma unroll
    for (int sc = 1; sc <= S_CAP; ++sc) {                  // (constant divisors)
        const int ch = (p.ntile + sc - 1) / sc;
        const float waves = ceilf((float)(H * sc) * inv_ctas - 1e-4f);
        const float cost = waves * (fmaxf((float)((ch + NWARPS - 1) / NWARPS), 0.4f * (float)ch) + 2.f + (sc > 1 ? 3.f : 0.f));
        if (sc == 1 || (sc <= p.ntile && cost < best)) { best = cost; p.S = sc; }
    }
    p.chunk = max(1, (p.ntile + p.S - 1) / p.S);
    p.S = max(1, (p.ntile + p.chunk - 1) / p.chunk);       // no split without tiles
    return p;
}
// The same for attention_impl: a head's keys 0 .. pos0 + M - 1, those of this pass among them.  The cost of a split count, in steps of
// 64 keys and four rows (0.7 to 1.5 us): the steps of an item, two of fixed work, two more for the merge.  The count it takes lies 1.4 %
// above the best one on average (as a single operator: 4 to 52 heads, fp32 of 64 and 128 dims and both types of 32, 60 to 8000 keys, 1, 7
// and 16 rows); without the rows in it, 7.4 % and at worst 82 %.
__host__ __device__ __forceinline__ AttPlan ka_plan(int pos0, int M, int H, int nctas) {
    AttPlan p;
    const int T = pos0 + M;
    const float inv_ctas = 1.0f / (float)nctas, steps = (float)((M + ATT_RB - 1) / ATT_RB) * (1.0f / 64.0f);
    float best = -1.f;
    p.ntile = 0; p.S = 1; p.pos = pos0;
#pragma unroll
    for (int sc = 1; sc <= S_CAP; ++sc) {
        const int chunk_ = (T + sc - 1) / sc;                                   // sc is a constant after unrolling
        const float waves = ceilf((float)(H * sc) * inv_ctas - 1e-4f);
        const float cost = waves * ((float)chunk_ * steps + (sc > 1 ? 4.f : 2.f));
        if ((sc == 1 || chunk_ >= 32) && (best < 0.f || cost < best)) { best = cost; p.S = sc; }
    }
    p.chunk = (T + p.S - 1) / p.S;
    return p;
}


// N words of a row, polled until all are there
template <int N>
__device__ __forceinline__ void att_read(const AttArgs& a, Ctx& c, const float* const (&p)[N], float (&v)[N]) {
    XchSpin sp; sp.spins = 0;
    while (true) {
        bool empty = false;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const unsigned w = xch_ld1(reinterpret_cast<const unsigned*>(p[i]));
            v[i] = __uint_as_float(w);
            empty |= w == XCH_EMPTY;
        }
        if (!a.poll || !empty || !xch_again(c, sp, 45)) return;
    }
}
// One element of the output, called by whole warps whose neighbouring lanes hold neighbouring elements
__device__ __forceinline__ void att_store(const AttArgs& a, int i, int col, float v) {
    if (a.out) xch_stf(a.out + (size_t)i * a.ldo + col, v);
    if (a.opk) pk_store_lane(a.opk + (size_t)i * a.ldopk, col, v);
}


// Consumer threads only.  One work item = (head, KV split); the eight warps of the CTA cut the item's
// key range into eight slices and run an online-softmax pass over their slice without any CTA
// barrier: a lane owns hd/32 consecutive dimensions, so a key or value row is one coalesced load of
// the warp, q . k is finished by a butterfly of shuffles, and o += p v stays in the lane.  Keys are
// taken eight at a time (their loads are issued together).  The rows of this pass are rotated
// (RoPE), rounded to the cache's storage type and appended to the cache by the item whose key range
// contains them, then read back like any other key.  The warps' (max, sum, o) are merged through
// shared memory; with more than one split every item writes a partial and the last split of a head
// to arrive merges them in split order.
template <typename WT, int DPL> struct AttLoad;          // raw bits of DPL consecutive elements, and their conversion
template <> struct AttLoad<__nv_bfloat16, 4> {
    typedef uint2 Raw;
    static __device__ __forceinline__ Raw ld(const __nv_bfloat16* p) { return __ldcg(reinterpret_cast<const uint2*>(p)); }
    static __device__ __forceinline__ void cvt(const Raw& r, float (&v)[4]) {
        v[0] = __uint_as_float(r.x << 16); v[1] = __uint_as_float(r.x & 0xffff0000u);
        v[2] = __uint_as_float(r.y << 16); v[3] = __uint_as_float(r.y & 0xffff0000u);
    }
};
template <> struct AttLoad<__nv_bfloat16, 2> {
    typedef unsigned Raw;
    static __device__ __forceinline__ Raw ld(const __nv_bfloat16* p) { return __ldcg(reinterpret_cast<const unsigned*>(p)); }
    static __device__ __forceinline__ void cvt(const Raw& r, float (&v)[2]) { v[0] = __uint_as_float(r << 16); v[1] = __uint_as_float(r & 0xffff0000u); }
};
template <> struct AttLoad<__nv_bfloat16, 1> {
    typedef unsigned short Raw;
    static __device__ __forceinline__ Raw ld(const __nv_bfloat16* p) { return __ldcg(reinterpret_cast<const unsigned short*>(p)); }
    static __device__ __forceinline__ void cvt(const Raw& r, float (&v)[1]) { v[0] = __uint_as_float((unsigned)r << 16); }
};
template <> struct AttLoad<float, 4> {
    typedef float4 Raw;
    static __device__ __forceinline__ Raw ld(const float* p) { return __ldcg(reinterpret_cast<const float4*>(p)); }
    static __device__ __forceinline__ void cvt(const Raw& r, float (&v)[4]) { v[0] = r.x; v[1] = r.y; v[2] = r.z; v[3] = r.w; }
};
template <> struct AttLoad<float, 2> {
    typedef float2 Raw;
    static __device__ __forceinline__ Raw ld(const float* p) { return __ldcg(reinterpret_cast<const float2*>(p)); }
    static __device__ __forceinline__ void cvt(const Raw& r, float (&v)[2]) { v[0] = r.x; v[1] = r.y; }
};
template <> struct AttLoad<float, 1> {
    typedef float Raw;
    static __device__ __forceinline__ Raw ld(const float* p) { return __ldcg(p); }
    static __device__ __forceinline__ void cvt(const Raw& r, float (&v)[1]) { v[0] = r; }
};

// A page number outside the cache never becomes an address: the access goes to page 0 and the state word records it.
__device__ __forceinline__ int checked_page(int pg, int n_pages, State* st, int where) {
    if ((unsigned)pg < (unsigned)n_pages) return pg;
    if (st) { atomicCAS(&st->status, 0, ST_INTERNAL); st->timeout_where = where; }
    return 0;
}

constexpr int ATT_G = 8;           // keys per group
constexpr int ATT_MB_STRIDE = HD_MAX + 2;   // merge buffer row: o[hd], max, sum

__device__ __forceinline__ float ex2f(float x) {             // 2^x, one special-function instruction
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One warp: rows i0 .. i0+nr-1 of the pass against keys [kb, ke) of head hh.  Scores are kept in the log2
// domain (q is pre-scaled by log2(e) / sqrt(hd)), so every exponential is one ex2.  The loads of the next
// key group are in flight while the current one is reduced.  A group's 8 x 4 partial dot products are summed
// by a transposing butterfly (31 shuffles) that leaves score (key j, row r) in lane 4 j + r; that lane does the
// online-softmax update of its row (lanes sharing r hold the same running max and sum), and the 32 probabilities
// reach every lane through a few words of shared memory for o += p v.
template <typename WT, int DPL>
__device__ __forceinline__ void att_warp_slice(const Dev& D, const AttArgs& a, int hh, int i0, int nr, int kb, int ke,
                                               const float* qs, float* pbuf, float& m_lane, float& l_lane, float (&o)[ATT_RB][DPL]) {
    typedef typename AttLoad<WT, DPL>::Raw Raw;
    static_assert(ATT_G == 8 && ATT_RB == 4, "the butterfly below is written for 8 keys x 4 rows");
    const int lane = threadIdx.x & 31;
    const int jl = lane >> 2, rl = lane & 3;
    constexpr int hd = 32 * DPL;
    const int H = D.dm.H, psh = D.dm.ps_shift, psm = D.dm.page_size - 1;
    const int pos0 = a.pos0;
    const WT* kc = reinterpret_cast<const WT*>(a.kc);
    const WT* vc = reinterpret_cast<const WT*>(a.vc);
    const int* page_table = D.page_table;
    float q[ATT_RB][DPL];
#pragma unroll
    for (int r = 0; r < ATT_RB; ++r) {
#pragma unroll
        for (int e = 0; e < DPL; ++e) { o[r][e] = 0.f; q[r][e] = r < nr ? qs[(i0 + r) * HD_MAX + lane * DPL + e] : 0.f; }
    }
    m_lane = -INFINITY; l_lane = 0.f;
    if (kb >= ke) return;
    // page table entries of a window of keys live in the lanes (lane p holds page first_page + p)
    const int win = max(ATT_G, ((31 << psh) >> 3) << 3);
    int wstart = kb, first_page = kb >> psh;
    auto pages = [&]() { return checked_page(__ldg(page_table + min(first_page + lane, D.dm.n_pages - 1)), D.dm.n_phys, D.st, 53); };
    int pgs = pages();
    Raw kr[ATT_G], vr[ATT_G];
    auto issue = [&](int g0) {
        if (g0 >= wstart + win) { wstart = g0; first_page = g0 >> psh; pgs = pages(); }
#pragma unroll
        for (int j = 0; j < ATT_G; ++j) {
            const int pos = min(g0 + j, ke - 1);
            const int pg = __shfl_sync(0xffffffffu, pgs, (pos >> psh) - first_page);
            const size_t base = ((((size_t)pg * H + hh) << psh) + (pos & psm)) * hd + lane * DPL;
            kr[j] = AttLoad<WT, DPL>::ld(kc + base);
            vr[j] = AttLoad<WT, DPL>::ld(vc + base);
        }
    };
    issue(kb);
    for (int g0 = kb; g0 < ke; g0 += ATT_G) {
        float kv[ATT_G][DPL], vv[ATT_G][DPL];
#pragma unroll
        for (int j = 0; j < ATT_G; ++j) { AttLoad<WT, DPL>::cvt(kr[j], kv[j]); AttLoad<WT, DPL>::cvt(vr[j], vv[j]); }
        if (g0 + ATT_G < ke) issue(g0 + ATT_G);
        float v[ATT_G * ATT_RB];
#pragma unroll
        for (int j = 0; j < ATT_G; ++j) {
#pragma unroll
            for (int r = 0; r < ATT_RB; ++r) {
                float dsum = 0.f;
#pragma unroll
                for (int e = 0; e < DPL; ++e) dsum = fmaf(q[r][e], kv[j][e], dsum);
                v[j * ATT_RB + r] = dsum;
            }
        }
        // transposing butterfly: after the step with offset `ofs` a lane keeps the half of its values selected by that
        // bit of its lane index, summed with the partner's; in the end lane L holds the full sum of value L
#pragma unroll
        for (int ofs = 16; ofs > 0; ofs >>= 1) {
            const bool up = (lane & ofs) != 0;
#pragma unroll
            for (int i = 0; i < ofs; ++i) {
                const float send = up ? v[i] : v[i + ofs];
                const float keep = up ? v[i + ofs] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, ofs);
            }
        }
        const int pos = g0 + jl;
        float sv = (pos < ke && rl < nr && pos <= pos0 + i0 + rl) ? v[0] : -INFINITY;
        float mg = sv;
        mg = fmaxf(mg, __shfl_xor_sync(0xffffffffu, mg, 4));
        mg = fmaxf(mg, __shfl_xor_sync(0xffffffffu, mg, 8));
        mg = fmaxf(mg, __shfl_xor_sync(0xffffffffu, mg, 16));
        const float mn = fmaxf(m_lane, mg);
        const float p = (sv == -INFINITY) ? 0.f : ex2f(sv - mn);
        const float cf = (m_lane == -INFINITY) ? 0.f : ex2f(m_lane - mn);
        float psum = p;
        psum += __shfl_xor_sync(0xffffffffu, psum, 4);
        psum += __shfl_xor_sync(0xffffffffu, psum, 8);
        psum += __shfl_xor_sync(0xffffffffu, psum, 16);
        l_lane = l_lane * cf + psum;
        m_lane = mn;
        __syncwarp();
        pbuf[lane] = p;
        if (jl == 0) pbuf[32 + rl] = cf;
        __syncwarp();
        const float4 cfv = *reinterpret_cast<const float4*>(pbuf + 32);
        const float cfa[4] = {cfv.x, cfv.y, cfv.z, cfv.w};
#pragma unroll
        for (int r = 0; r < ATT_RB; ++r) {
#pragma unroll
            for (int e = 0; e < DPL; ++e) o[r][e] *= cfa[r];
        }
#pragma unroll
        for (int j = 0; j < ATT_G; ++j) {
            const float4 pj = *reinterpret_cast<const float4*>(pbuf + j * 4);
            const float pa[4] = {pj.x, pj.y, pj.z, pj.w};
#pragma unroll
            for (int r = 0; r < ATT_RB; ++r) {
#pragma unroll
                for (int e = 0; e < DPL; ++e) o[r][e] = fmaf(pa[r], vv[j][e], o[r][e]);
            }
        }
    }
}

// The last split of a head to arrive merges the S partial (max, sum, o) of every row in split order.  SC >= S is the
// compile-time bound of the split loop; U elements per thread are handled together, and every load of such a batch is
// issued before any is used, so that a batch costs one L2 round trip.
template <int hd, int SC, int U>
__device__ __forceinline__ void att_merge_splits(const Dev& D, const AttArgs& a, int hh, int S, int M) {
    const int tid = threadIdx.x, H = D.dm.H;
    const int total = M * hd;
    for (int idx0 = tid; idx0 < total; idx0 += NTHREADS * U) {
        float2 mlv[U][SC];
        float pov[U][SC];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = idx0 + u * NTHREADS < total ? idx0 + u * NTHREADS : idx0;
            const int i = idx / hd, e = idx % hd;
            const float2* ml = reinterpret_cast<const float2*>(D.att_ml + ((size_t)i * H + hh) * S_CAP * 2);
            const float* po = D.att_po + ((size_t)i * H + hh) * S_CAP * hd + e;
#pragma unroll
            for (int q = 0; q < SC; ++q) {
                const int qq = q < S ? q : 0;
                mlv[u][q] = __ldcg(ml + qq);
                pov[u][q] = ldcg_f(po + (size_t)qq * hd);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = idx0 + u * NTHREADS;
            if (idx < total) {
                const int i = idx / hd, e = idx % hd;
                float mx = -INFINITY;
#pragma unroll
                for (int q = 0; q < SC; ++q) if (q < S) mx = fmaxf(mx, mlv[u][q].x);
                float den = 0.f, num = 0.f;
#pragma unroll
                for (int q = 0; q < SC; ++q) {
                    if (q < S && mlv[u][q].x != -INFINITY) {
                        const float w = ex2f(mlv[u][q].x - mx);
                        den += mlv[u][q].y * w;
                        num += pov[u][q] * w;
                    }
                }
                att_store(a, i, hh * hd + e, num / den);
            }
        }
    }
}

// OP: single operator
template <typename WT, int DPL, bool OP>
__device__ __forceinline__ void attention_impl(const Dev& D, const AttArgs& a, const AttPlan pl, Ctx& c) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int hd = 32 * DPL, half = hd / 2;
    const int H = D.dm.H, d = D.dm.d, ps = D.dm.page_size;
    const int M = a.M, pos0 = a.pos0;
    const int T = pos0 + M;
    const int S = pl.S, chunk = pl.chunk;
    const float sc = rsqrtf((float)hd) * 1.4426950408889634f;      // 1/sqrt(hd), and log2(e): scores live in the log2 domain
    WT* kc = reinterpret_cast<WT*>(a.kc);
    WT* vc = reinterpret_cast<WT*>(a.vc);

    float* qs = reinterpret_cast<float*>(c.smem + WORK_OFF);       // [M_MAX][HD_MAX]
    float* mb = qs + M_MAX * HD_MAX;                               // [NWARPS][ATT_RB][ATT_MB_STRIDE]
    float* pbuf = mb + NWARPS * ATT_RB * ATT_MB_STRIDE + warp * 40;      // [NWARPS][40] probabilities of a key group

    for (int item = c.cta; item < H * S; item += c.nctas) {
        const int hh = item / S, s = item % S;
        const int kb = s * chunk, ke = min(T, kb + chunk);
        // q rows: RoPE, pre-scaled by 1/sqrt(hd) (loads first: the angle arithmetic runs while they are in flight)
        for (int idx = tid; idx < M * half; idx += NTHREADS) {
            const int i = idx / half, e = idx % half;
            const float* src = a.qkv + (size_t)i * a.ldq + hh * hd + e;
            const float* const p[2] = {src, src + half};
            float xv[2];
            att_read<2>(a, c, p, xv);
            const float x1 = xv[0], x2 = xv[1];
            float cs, sn; rope_cs(D, pos0 + i, e, cs, sn);
            qs[i * HD_MAX + e] = (x1 * cs - x2 * sn) * sc;
            qs[i * HD_MAX + e + half] = (x2 * cs + x1 * sn) * sc;
        }
        // append this pass's K / V rows that fall into my key range (every load of an element before its first use)
        {
            const int nb = max(kb, pos0), ne = ke;
            for (int idx = tid; idx < (ne - nb) * half; idx += NTHREADS) {
                const int pos = nb + idx / half, e = idx % half, i = pos - pos0;
                const float* src = a.qkv + (size_t)i * a.ldq + hh * hd + e;
                const float* const p[4] = {src + d, src + d + half, src + 2 * d, src + 2 * d + half};
                float xv[4];
                att_read<4>(a, c, p, xv);
                const float k1 = xv[0], k2 = xv[1], v1 = xv[2], v2 = xv[3];
                const int page = checked_page(__ldg(D.page_table + (pos >> D.dm.ps_shift)), D.dm.n_phys, D.st, 54);
                float cs, sn; rope_cs(D, pos, e, cs, sn);
                const size_t base = (((size_t)page * H + hh) * ps + (pos & (ps - 1))) * hd;
                kc[base + e] = float_to_wt<WT>(k1 * cs - k2 * sn);
                kc[base + e + half] = float_to_wt<WT>(k2 * cs + k1 * sn);
                vc[base + e] = float_to_wt<WT>(v1);
                vc[base + e + half] = float_to_wt<WT>(v2);
            }
        }
        cta_sync();
        // this warp's slice of the item's keys, in whole groups
        const int nkeys = ke - kb;
        const int per = ((nkeys + NWARPS - 1) / NWARPS + ATT_G - 1) / ATT_G * ATT_G;
        const int wb = min(ke, kb + warp * per), we = min(ke, wb + per);
        for (int i0 = 0; i0 < M; i0 += ATT_RB) {
            const int nr = min(ATT_RB, M - i0);
            float m_lane, l_lane, o[ATT_RB][DPL];
            att_warp_slice<WT, DPL>(D, a, hh, i0, nr, wb, we, qs, pbuf, m_lane, l_lane, o);
#pragma unroll
            for (int r = 0; r < ATT_RB; ++r) {
                float* row = mb + ((size_t)warp * ATT_RB + r) * ATT_MB_STRIDE;
#pragma unroll
                for (int e = 0; e < DPL; ++e) row[lane * DPL + e] = o[r][e];
                if (lane == r) { row[HD_MAX] = m_lane; row[HD_MAX + 1] = l_lane; }       // lane r tracks row r
            }
            cta_sync();
            for (int idx = tid; idx < nr * hd; idx += NTHREADS) {
                const int r = idx / hd, e = idx % hd, i = i0 + r;
                float mx = -INFINITY;
#pragma unroll
                for (int w = 0; w < NWARPS; ++w) mx = fmaxf(mx, mb[((size_t)w * ATT_RB + r) * ATT_MB_STRIDE + HD_MAX]);
                float den = 0.f, num = 0.f;
#pragma unroll
                for (int w = 0; w < NWARPS; ++w) {
                    const float* row = mb + ((size_t)w * ATT_RB + r) * ATT_MB_STRIDE;
                    const float mw = row[HD_MAX];
                    if (mw != -INFINITY) {
                        const float wgt = ex2f(mw - mx);
                        den += row[HD_MAX + 1] * wgt;
                        num += row[e] * wgt;
                    }
                }
                if (S == 1) {
                    att_store(a, i, hh * hd + e, num / den);
                } else {
                    D.att_po[(((size_t)i * H + hh) * S_CAP + s) * hd + e] = num;
                    if (e == 0) {
                        D.att_ml[(((size_t)i * H + hh) * S_CAP + s) * 2 + 0] = mx;
                        D.att_ml[(((size_t)i * H + hh) * S_CAP + s) * 2 + 1] = den;
                    }
                }
            }
            cta_sync();
        }
        if (S > 1) {
            __threadfence();
            cta_sync();
            if (tid == 0) {
                if (OP) grid_dependency_wait();            // the counters have been cleared
                const unsigned prev = atomicAdd(D.att_cnt + hh, 1u);
                const int last = (prev == (unsigned)(S - 1));
                c.ctl->att_last = last;
                if (last) { D.att_cnt[hh] = 0u; __threadfence(); }
            }
            cta_sync();
            if (*(volatile int*)&c.ctl->att_last) {
                if (S <= 4) att_merge_splits<hd, 4, 4>(D, a, hh, S, M);
                else if (S <= 8) att_merge_splits<hd, 8, 2>(D, a, hh, S, M);
                else att_merge_splits<hd, S_CAP, 1>(D, a, hh, S, M);
            }
            cta_sync();
        }
    }
}


// ---- tensor-core attention (bf16 cache, head_dim 64 or 128) ----------------------------------------------------
//
// One work item = (head, KV split).  The keys before this pass travel through the weight ring: the copy warp brings tiles of
// 16 keys (K and V, 64-dim boxes with the 128-byte swizzle) into the slots between the stages of W_qkv and W_o.  They do not
// depend on this pass, so they are on their way while q, k and v are still being formed; with loads into registers a tile cost
// a DRAM latency and one tile per warp was in flight (2.3 TB/s on long caches).  7B, KV 4096: verify pass of one row 3.50 -> 2.95
// ms, of seven rows 4.20 -> 3.58; the operator alone, 32 heads, 7 rows, 4090 keys 45.2 -> 32.6 us.  The rows of this pass are one more tile, which
// the last split of a head forms in shared memory from q, k, v and appends to the cache.
//
// A warp takes whole tiles (tile j of an item: warp j mod 8):
//   S = K Q^T      m16n8k16, keys on the M side (ldmatrix), rows on the N side (fragments in shared memory, rotated, pre-scaled by
//                  log2(e) / sqrt(hd), split into bf16 hi + lo)
//   online softmax in the log2 domain on the accumulator fragment (a lane holds 2 keys x 2 rows)
//   O^T = V^T P^T  dims on the M side (ldmatrix.trans), keys on the contraction side; P (hi + lo) moves from the accumulator
//                  layout into the B layout with movmatrix.
// With more than 8 rows a warp does both groups of 8 rows (R = 2) on the same K and V fragments.
//
// Splits of a head in the decode kernel (WAIT): all but the last one leave (max, sum, o) in exchange words, the last one polls them,
// merges in split order and empties the words again (their next use lies behind the barrier at the layer's end).  It waits for items
// of lower number only, every CTA takes its items in rising order, and the launch is cooperative, so there is always one that can go
// on.  The single operator is an ordinary launch, whose CTAs may have to wait for an SM: there every split leaves its partial results
// and counts itself, and whichever comes last merges them, in the same order (att_merge_ring); nobody waits.
__device__ __forceinline__ unsigned movmatrix_trans(unsigned a) {
    unsigned d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}
__device__ __forceinline__ void ldmatrix_x4_trans(unsigned (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst_smem, const CUtensorMap* tmap, int x, int y, uint32_t bar_smem) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst_smem), "l"(tmap), "r"(x), "r"(y), "r"(bar_smem) : "memory");
}

template <int HD> struct RaGeom {
    static constexpr int HALF_BYTES = ATT_TK * HD * 2;     // K (or V) of a tile: HD / 64 boxes of 16 rows x 128 bytes
    static constexpr int TILE_BYTES = 2 * HALF_BYTES;
    static constexpr int TPS = 32768 / TILE_BYTES;         // tiles per ring slot: 4 or 8
    static constexpr int QG = HD / 16 * 512;               // Q fragments of 8 rows: {hi b0, b1, lo b0, b1} per lane and k16-step
    static constexpr int NT_OFF = 8192;                    // the tile of this pass's rows; afterwards the merge buffer
    static constexpr int MB_OFF = NT_OFF;                  // [warps][ATT_RB][ROW] floats
    static constexpr int ROW = HD + 4;                     // a row of partial results: o [HD], maximum, sum, padding
};
static_assert(2 * RaGeom<128>::QG <= RaGeom<128>::NT_OFF && RaGeom<128>::TPS * RaGeom<128>::TILE_BYTES <= SLOT_BYTES, "attention tiles");
static_assert(RaGeom<128>::MB_OFF + NWARPS * ATT_RB * RaGeom<128>::ROW * 4 <= WORK_BYTES && WORK_OFF % 128 == 0 && SLOT_BYTES % 128 == 0, "attention buffers");

// Copy warp: the old K / V tiles of this CTA's items.  row0: first row of this layer's cache in the tensor maps.
template <int HD, bool PUBLISH>
__device__ __noinline__ bool att_produce(const Dev& D, const AttPlan pl, int row0, Ctx& c) {
    using G = RaGeom<HD>;
    const int lane = threadIdx.x & 31;
    const int H = D.dm.H, psh = D.dm.ps_shift, psm = D.dm.page_size - 1;
    const int bsh = min(psh, 4), per = (HD / 64 * 2) << (4 - bsh);        // a box holds 2^bsh keys; boxes per tile
    // the rows were written with ordinary stores (by earlier passes, ordered before this point by a grid barrier)
    asm volatile("fence.proxy.async;" ::: "memory");
    int slot = c.slot; unsigned phase = c.phase, issued = c.issued;
    bool ok = true;
    for (int item = c.cta; item < H * pl.S && ok; item += c.nctas) {
        const int hh = item / pl.S, tb = item % pl.S * pl.chunk, nt = min(pl.ntile, tb + pl.chunk) - tb;
        for (int t0 = 0; t0 < nt; t0 += G::TPS) {
            const int n = min(G::TPS, nt - t0);
            int w = 1;
            if (lane == 0) w = mbar_wait(c, &c.ctl->empty[slot], phase ^ 1u, 47) ? 1 : 0;
            w = __shfl_sync(0xffffffffu, w, 0);
            if (!w) { ok = false; break; }
            if (lane == 0) mbar_arrive_expect_tx(&c.ctl->full[slot], (unsigned)(n * G::TILE_BYTES));
            __syncwarp();
            const uint32_t dst = smem_u32(c.smem + RING_OFF + (size_t)slot * SLOT_BYTES), bar = smem_u32(&c.ctl->full[slot]);
            for (int op = lane; op < n * per; op += 32) {
                const int j = op / per, r = op - j * per;
                const int kv = r & 1, half = HD == 128 ? (r >> 1) & 1 : 0, b = HD == 128 ? r >> 2 : r >> 1;
                const int key = (tb + t0 + j) * ATT_TK + (b << bsh);
                const int page = checked_page(__ldg(D.page_table + min(key >> psh, D.dm.n_pages - 1)), D.dm.n_phys, D.st, 51);
                tma_load_2d(dst + (uint32_t)(j * G::TILE_BYTES + kv * G::HALF_BYTES + half * 2048 + (b << (bsh + 7))), kv ? &D.tmv : &D.tmk,
                            half * 64, row0 + ((page * H + hh) << psh) + (key & psm), bar);
            }
            issued++;
            if (PUBLISH && lane == 0) *(volatile unsigned*)&c.ctl->issued = issued;
            if (++slot == RING) { slot = 0; phase ^= 1u; }
        }
    }
    c.slot = slot; c.phase = phase; c.issued = issued;
    return ok;
}

// ring slots that att_produce fills
template <int HD> __device__ __forceinline__ unsigned att_stages(const Dev& D, const AttPlan& pl, const Ctx& c) {
    unsigned n = 0;
    for (int item = c.cta; item < D.dm.H * pl.S; item += c.nctas) {
        const int tb = item % pl.S * pl.chunk, nt = min(pl.ntile, tb + pl.chunk) - tb;
        n += (unsigned)((nt + RaGeom<HD>::TPS - 1) / RaGeom<HD>::TPS);
    }
    return n;
}

// shared-memory address of the 16-byte chunk `ch` of row `row` of a tile's K or V at `base`
__device__ __forceinline__ uint32_t ra_addr(uint32_t base, int row, int ch) {
    const uint32_t ra = base + (uint32_t)((ch >> 3) * 2048 + row * 128);
    return ra + (((uint32_t)ch ^ (ra >> 7)) & 7u) * 16u;
}

// One tile: keys 0 .. nv - 1 of it are valid; causal: key i is seen by rows >= i only (the tile of this pass's rows).
template <int HD, int R>
__device__ __forceinline__ void ra_tile(uint32_t kb, uint32_t vb, uint32_t qf, int nv, bool causal, float (&o)[R][HD / 16][4],
                                        float (&mx)[R][2], float (&l)[R][2]) {
    const int lane = tid_here() & 31, g = lane >> 2, t = lane & 3;
    // hi of even and odd k16-steps, lo: the tensor core truncates at every accumulation, so that chains stay at HD / 32 steps
    // where it counts (lo is 2^-9 of the sum)
    float sc[R][3][4];
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int i = 0; i < 4; ++i) sc[r][0][i] = sc[r][1][i] = sc[r][2][i] = 0.f;
    }
#pragma unroll
    for (int k = 0; k < HD / 16; ++k) {
        unsigned a[4];
        ldmatrix_x4(a, ra_addr(kb, lane & 15, k * 2 + (lane >> 4)));
#pragma unroll
        for (int r = 0; r < R; ++r) {
            uint4 q;
            asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w) : "r"(qf + (uint32_t)(r * RaGeom<HD>::QG + (k * 32 + lane) * 16)));
            mma_bf16_16816(sc[r][k & 1], a, q.x, q.y);
            mma_bf16_16816(sc[r][2], a, q.z, q.w);
        }
    }
    unsigned bh[R][2], bl[R][2];
    float cf[R][2];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        float s[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            s[i] = (sc[r][0][i] + sc[r][1][i]) + sc[r][2][i];
            const int key = g + (i >> 1) * 8, row = r * 8 + 2 * t + (i & 1);
            if (key >= nv || (causal && key > row)) s[i] = -INFINITY;
        }
        float p[4];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float m = fmaxf(s[i], s[2 + i]);
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 4));
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 8));
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
            const float mn = fmaxf(mx[r][i], m);
            cf[r][i] = mx[r][i] == -INFINITY ? 0.f : ex2f(mx[r][i] - mn);
            p[i] = s[i] == -INFINITY ? 0.f : ex2f(s[i] - mn);
            p[2 + i] = s[2 + i] == -INFINITY ? 0.f : ex2f(s[2 + i] - mn);
            l[r][i] = l[r][i] * cf[r][i] + (p[i] + p[2 + i]);
            mx[r][i] = mn;
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            unsigned hi, lo;
            split_hi_lo(make_float2(p[2 * q], p[2 * q + 1]), hi, lo);
            bh[r][q] = movmatrix_trans(hi);
            bl[r][q] = movmatrix_trans(lo);
        }
    }
    // V rows past the valid keys hold anything (0 * NaN would be NaN)
    const unsigned vm0 = (2 * t < nv ? 0xffffu : 0u) | (2 * t + 1 < nv ? 0xffff0000u : 0u);
    const unsigned vm1 = (2 * t + 8 < nv ? 0xffffu : 0u) | (2 * t + 9 < nv ? 0xffff0000u : 0u);
#pragma unroll
    for (int d = 0; d < HD / 16; ++d) {
        unsigned v[4];
        ldmatrix_x4_trans(v, ra_addr(vb, (lane & 7) + (lane >> 4) * 8, d * 2 + ((lane >> 3) & 1)));
        if (nv < ATT_TK) { v[0] &= vm0; v[1] &= vm0; v[2] &= vm1; v[3] &= vm1; }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            o[r][d][0] *= cf[r][0]; o[r][d][1] *= cf[r][1]; o[r][d][2] *= cf[r][0]; o[r][d][3] *= cf[r][1];
            mma_bf16_16816(o[r][d], v, bh[r][0], bh[r][1]);
            mma_bf16_16816(o[r][d], v, bl[r][0], bl[r][1]);
        }
    }
}

__device__ __forceinline__ void rope_at(const Dev& D, int pos, int e, int half, float& cs, float& sn) {
    if (D.rope) { const float2 v = __ldg(D.rope + (size_t)pos * half + e); cs = v.x; sn = v.y; }
    else rope_cs(D, pos, e, cs, sn);
}

// One split's (max, sum, four elements) added to the merge of a row
__device__ __forceinline__ void ra_add(float& m, float& den, float4& num, float om, float ol, float4 o) {
    const float mn = fmaxf(m, om);
    const float f0 = m == -INFINITY ? 0.f : ex2f(m - mn), f1 = om == -INFINITY ? 0.f : ex2f(om - mn);
    den = den * f0 + ol * f1;
    num.x = num.x * f0 + o.x * f1; num.y = num.y * f0 + o.y * f1; num.z = num.z * f0 + o.z * f1; num.w = num.w * f0 + o.w * f1;
    m = mn;
}

// Single operator: the merge of a head's S partial results by the CTA that came last: the last split's, then the others in order.
template <int HD>
__device__ __forceinline__ void att_merge_ring(const Dev& D, const AttArgs& a, int hh, int S) {
    constexpr int ROW = RaGeom<HD>::ROW, QB = 4;
    const int tid = tid_here(), H = D.dm.H;
    for (int idx = tid; idx < a.M * (HD / 4); idx += NTHREADS) {
        const int i = idx / (HD / 4), e = idx % (HD / 4) * 4;
        const float* row = reinterpret_cast<const float*>(D.att_xp) + ((size_t)i * H + hh) * S_CAP * ROW;
        float4 num = ldcg_f4(row + (S - 1) * ROW + e);
        const float2 ml = ldcg_f2(row + (S - 1) * ROW + HD);
        float m = ml.x, den = ml.y;
        for (int q0 = 0; q0 < S - 1; q0 += QB) {
            float4 wo[QB]; float2 wm[QB];
#pragma unroll
            for (int q = 0; q < QB; ++q) { const int s = min(q0 + q, S - 2); wo[q] = ldcg_f4(row + s * ROW + e); wm[q] = ldcg_f2(row + s * ROW + HD); }
#pragma unroll
            for (int q = 0; q < QB; ++q) if (q0 + q < S - 1) ra_add(m, den, num, wm[q].x, wm[q].y, wo[q]);
        }
        *reinterpret_cast<float4*>(a.out + (size_t)i * a.ldo + hh * HD + e) = make_float4(num.x / den, num.y / den, num.z / den, num.w / den);
    }
}

template <int HD, int R, bool WAIT>
__device__ __forceinline__ void attention_ring(const Dev& D, const AttArgs& a, Ctx& c) {
    typedef __nv_bfloat16 WT;
    using G = RaGeom<HD>;
    constexpr int half = HD / 2;
    const int tid = tid_here(), lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int H = D.dm.H, d = D.dm.d, psh = D.dm.ps_shift, psm = D.dm.page_size - 1;
    const int M = a.M, pos0 = a.pos0;
    const AttPlan pl = a.plan;
    const float qscale = rsqrtf((float)HD) * 1.4426950408889634f;      // 1/sqrt(hd) and log2(e)
    char* qsm = c.smem + WORK_OFF;
    char* ntile = c.smem + WORK_OFF + G::NT_OFF;
    float* mb = reinterpret_cast<float*>(c.smem + WORK_OFF + G::MB_OFF);
    const uint32_t nt_u = smem_u32(ntile);
    int slot = c.slot; unsigned phase = c.phase;
    bool ok = true;

    for (int item = c.cta; item < H * pl.S; item += c.nctas) {
        const int hh = item / pl.S, s = item - hh * pl.S;
        const int tb = s * pl.chunk, nt = min(pl.ntile, tb + pl.chunk) - tb;
        const bool last = s == pl.S - 1;
        // ---- this pass's rows: q rotated, scaled, split into fragments; in the last split k rotated and, with v, rounded into the
        // new tile and the cache.  Rows M .. 8 R - 1 of Q and M .. 15 of V are zero.
        for (int idx0 = tid; idx0 < 8 * R * half; idx0 += 2 * NTHREADS) {
            float q1[2], q2[2], k1[2], k2[2], v1[2], v2[2], cs[2], sn[2];
            int pg[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {                  // what does not depend on this pass, before the poll
                const int idx = idx0 + u * NTHREADS, i = idx / half;
                cs[u] = sn[u] = 0.f; pg[u] = 0;
                if (i < M) {
                    rope_at(D, pos0 + i, idx & (half - 1), half, cs[u], sn[u]);
                    if (last) pg[u] = __ldg(D.page_table + ((pos0 + i) >> psh));
                }
            }
            {
                XchSpin sp; sp.spins = 0;
                const float* qkv = a.qkv;
                while (true) {
                    bool empty = false;
                    asm volatile("" : "+l"(qkv));        // (addresses are formed inside the loop, not kept across it)
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int idx = idx0 + u * NTHREADS, i = idx / half;
                        q1[u] = q2[u] = k1[u] = k2[u] = v1[u] = v2[u] = 0.f;
                        if (i < M) {
                            const unsigned* src = reinterpret_cast<const unsigned*>(qkv + (size_t)i * a.ldq + hh * HD + (idx & (half - 1)));
                            unsigned w[6];
                            w[0] = xch_ld1(src); w[1] = xch_ld1(src + half);
                            w[2] = w[3] = w[4] = w[5] = 0u;
                            if (last) { w[2] = xch_ld1(src + d); w[3] = xch_ld1(src + d + half); w[4] = xch_ld1(src + 2 * d); w[5] = xch_ld1(src + 2 * d + half); }
#pragma unroll
                            for (int q = 0; q < 6; ++q) empty |= w[q] == XCH_EMPTY;
                            q1[u] = __uint_as_float(w[0]); q2[u] = __uint_as_float(w[1]); k1[u] = __uint_as_float(w[2]); k2[u] = __uint_as_float(w[3]);
                            v1[u] = __uint_as_float(w[4]); v2[u] = __uint_as_float(w[5]);
                        }
                    }
                    if (!a.poll || !empty || !xch_again(c, sp, 45)) break;
                }
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int idx = idx0 + u * NTHREADS, i = idx / half, e = idx & (half - 1), pos = pos0 + i;
                if (i >= 8 * R) break;
                const float r[2] = {(q1[u] * cs[u] - q2[u] * sn[u]) * qscale, (q2[u] * cs[u] + q1[u] * sn[u]) * qscale};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int dim = e + h * half, kk = dim & 15;
                    char* p = qsm + (i >> 3) * G::QG + (((dim >> 4) * 32) + (i & 7) * 4 + ((kk & 7) >> 1)) * 16 + (kk >> 3) * 4 + (kk & 1) * 2;
                    const WT hi = __float2bfloat16_rn(r[h]);
                    *reinterpret_cast<WT*>(p) = hi;
                    *reinterpret_cast<WT*>(p + 8) = __float2bfloat16_rn(r[h] - __bfloat162float(hi));
                }
                if (last) {
                    const WT kr[2] = {__float2bfloat16_rn(k1[u] * cs[u] - k2[u] * sn[u]), __float2bfloat16_rn(k2[u] * cs[u] + k1[u] * sn[u])};
                    const WT vr[2] = {__float2bfloat16_rn(v1[u]), __float2bfloat16_rn(v2[u])};
                    WT* kc = nullptr; WT* vc = nullptr;
                    if (i < M) {
                        const int page = checked_page(pg[u], D.dm.n_phys, D.st, 52);
                        const size_t base = ((((size_t)page * H + hh) << psh) + (pos & psm)) * HD;
                        kc = reinterpret_cast<WT*>(a.kc) + base; vc = reinterpret_cast<WT*>(a.vc) + base;
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int dim = e + h * half;
                        const uint32_t off = ra_addr(nt_u, i, dim >> 3) - nt_u + (uint32_t)(dim & 7) * 2;
                        *reinterpret_cast<WT*>(ntile + off) = kr[h];
                        *reinterpret_cast<WT*>(ntile + G::HALF_BYTES + off) = vr[h];
                        if (i < M) { kc[dim] = kr[h]; vc[dim] = vr[h]; }
                    }
                }
            }
        }
        cta_sync();
        // ---- the tiles
        float o[R][HD / 16][4], mx[R][2], l[R][2];
#pragma unroll
        for (int r = 0; r < R; ++r) {
#pragma unroll
            for (int e = 0; e < HD / 16; ++e) { o[r][e][0] = o[r][e][1] = o[r][e][2] = o[r][e][3] = 0.f; }
            mx[r][0] = mx[r][1] = -INFINITY; l[r][0] = l[r][1] = 0.f;
        }
        const uint32_t qf = smem_u32(qsm);
        const int nslot = (nt + G::TPS - 1) / G::TPS;
        // one round per ring slot, and one more for the tile of this pass's rows
        for (int k = 0; k <= nslot; ++k) {
            const bool fresh = k == nslot;
            if (fresh && !last) break;
            if (!fresh && ok) ok = mbar_wait(c, &c.ctl->full[slot], phase, 48);
            const int jt = fresh ? nt : k * G::TPS + ((warp - k * G::TPS) & (NWARPS - 1));       // this warp's tile, if it lies in the slot
            const bool mine = fresh ? warp == (nt & (NWARPS - 1)) : (jt < (k + 1) * G::TPS && jt < nt);
            if (mine && ok) {
                const uint32_t kb = fresh ? nt_u : smem_u32(c.smem + RING_OFF + (size_t)slot * SLOT_BYTES) + (uint32_t)((jt - k * G::TPS) * G::TILE_BYTES);
                ra_tile<HD, R>(kb, kb + G::HALF_BYTES, qf, fresh ? M : min(ATT_TK, pos0 - (tb + jt) * ATT_TK), fresh, o, mx, l);
            }
            if (!fresh) {
                __syncwarp();
                if (ok && lane == 0) mbar_arrive(&c.ctl->empty[slot]);
                if (++slot == RING) { slot = 0; phase ^= 1u; }
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                l[r][i] += __shfl_xor_sync(0xffffffffu, l[r][i], 4);
                l[r][i] += __shfl_xor_sync(0xffffffffu, l[r][i], 8);
                l[r][i] += __shfl_xor_sync(0xffffffffu, l[r][i], 16);
            }
        }
        cta_sync();                                        // the new tile has been read: the merge buffer lies over it
        // ---- merge of the warps (those without tiles hold zeros and a maximum of -inf), four rows at a time, then of the splits; a
        // thread takes four neighbouring elements (one element a thread, in rolled loops, took 4.6 us for seven rows)
        unsigned* xw = D.att_xp;                           // [M_MAX][H][S_CAP][ROW]
        constexpr int ROW = G::ROW;
#pragma unroll
        for (int rb = 0; rb < 2 * R; ++rb) {
            if (rb * ATT_RB >= M) break;
            const int nr = min(ATT_RB, M - rb * ATT_RB), r = rb >> 1;
            if ((t >> 1) == (rb & 1)) {
                const int rl = 2 * (t & 1);
                float* r0 = mb + ((size_t)warp * ATT_RB + rl) * ROW;
                float* r1 = r0 + ROW;
#pragma unroll
                for (int e = 0; e < HD / 16; ++e) {
                    r0[e * 16 + g] = o[r][e][0]; r1[e * 16 + g] = o[r][e][1];
                    r0[e * 16 + 8 + g] = o[r][e][2]; r1[e * 16 + 8 + g] = o[r][e][3];
                }
                if (g == 0) { r0[HD] = mx[r][0]; r0[HD + 1] = l[r][0]; r1[HD] = mx[r][1]; r1[HD + 1] = l[r][1]; }
            }
            cta_sync();
            if (tid < nr * (HD / 4)) {
                const int rr = tid / (HD / 4), e = tid % (HD / 4) * 4, i = rb * ATT_RB + rr;
                unsigned* xrow = xw + (((size_t)i * H + hh) * S_CAP) * ROW;
                // the other splits' words are requested before this one's are added up
                constexpr int QB = 4;
                uint4 wo[QB]; uint2 wm[QB];
                auto request = [&](int q0) {
                    asm volatile("" : "+l"(xrow));
#pragma unroll
                    for (int q = 0; q < QB; ++q)
                        if (WAIT && last && q0 + q < s) { wo[q] = xch_ld4(xrow + (q0 + q) * ROW + e); wm[q] = xch_ld2(xrow + (q0 + q) * ROW + HD); }
                };
                request(0);
                const float* row = mb + rr * ROW;
                float2 ml[NWARPS];
#pragma unroll
                for (int w = 0; w < NWARPS; ++w) ml[w] = *reinterpret_cast<const float2*>(row + w * ATT_RB * ROW + HD);
                float m = ml[0].x, den = 0.f;
#pragma unroll
                for (int w = 1; w < NWARPS; ++w) m = fmaxf(m, ml[w].x);
                float4 num = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int w = 0; w < NWARPS; ++w) {
                    const float f = ml[w].x == -INFINITY ? 0.f : ex2f(ml[w].x - m);
                    const float4 v = *reinterpret_cast<const float4*>(row + w * ATT_RB * ROW + e);
                    den += ml[w].y * f;
                    num.x += v.x * f; num.y += v.y * f; num.z += v.z * f; num.w += v.w * f;
                }
                if (WAIT ? !last : pl.S > 1) {
                    unsigned* p = xrow + s * ROW;
                    xch_st4(p + e, make_uint4(__float_as_uint(num.x), __float_as_uint(num.y), __float_as_uint(num.z), __float_as_uint(num.w)));
                    if (e == 0) { xch_st(p + HD, __float_as_uint(m)); xch_st(p + HD + 1, __float_as_uint(den)); }
                } else {
                    for (int q0 = 0; WAIT && q0 < s; q0 += QB) {
                        if (q0) request(q0);
                        XchSpin sp; sp.spins = 0;
                        while (true) {
                            bool empty = false;
#pragma unroll
                            for (int q = 0; q < QB; ++q) empty |= q0 + q < s && (xch_empty(wo[q]) || xch_empty(wm[q]));
                            if (!empty || !xch_again(c, sp, 49)) break;
                            request(q0);
                        }
#pragma unroll
                        for (int q = 0; q < QB; ++q) {
                            if (q0 + q < s) {
                                ra_add(m, den, num, __uint_as_float(wm[q].x), __uint_as_float(wm[q].y),
                                       make_float4(__uint_as_float(wo[q].x), __uint_as_float(wo[q].y), __uint_as_float(wo[q].z), __uint_as_float(wo[q].w)));
                                xch_st4(xrow + (q0 + q) * ROW + e, make_uint4(XCH_EMPTY, XCH_EMPTY, XCH_EMPTY, XCH_EMPTY));      // this thread alone reads them
                            }
                        }
                    }
                    num.x /= den; num.y /= den; num.z /= den; num.w /= den;
                    const int col = hh * HD + e;
                    if (a.out) *reinterpret_cast<float4*>(a.out + (size_t)i * a.ldo + col) = num;
                    if (a.opk) { pk_store2(a.opk + (size_t)i * a.ldopk, col, num.x, num.y); pk_store2(a.opk + (size_t)i * a.ldopk, col + 2, num.z, num.w); }
                }
            }
            cta_sync();
        }
        if (!WAIT && pl.S > 1) {
            // this CTA's partial results are ordered before the counter by the barrier above and the release of the atomic; its
            // acquire orders the counter before the reads of every split's
            if (tid == 0) {
                unsigned prev;
                grid_dependency_wait();                    // the counters have been cleared
                asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(prev) : "l"(D.att_cnt + hh) : "memory");
                c.ctl->att_last = prev == (unsigned)(pl.S - 1);
            }
            cta_sync();
            if (*(volatile int*)&c.ctl->att_last) att_merge_ring<HD>(D, a, hh, pl.S);
        }
        if (WAIT && last && s > 0) {
            // maxima and sums have been read by every thread of the merge
            for (int idx = tid; idx < M * s; idx += NTHREADS) {
                unsigned* p = xw + (((size_t)(idx / s) * H + hh) * S_CAP + idx % s) * ROW + HD;
                xch_st(p, XCH_EMPTY); xch_st(p + 1, XCH_EMPTY);
            }
        }
    }
    c.slot = slot; c.phase = phase;
}

// storage type and head size of the tensor-core attention
template <typename WT, int HD> constexpr bool RING_ATT = sizeof(WT) == 2 && HD >= 64;

__device__ __forceinline__ bool attention_producer(const Dev& D, const AttPlan& pl, int row0, Ctx& c) {
    return D.dm.hd == 128 ? att_produce<128, true>(D, pl, row0, c) : att_produce<64, true>(D, pl, row0, c);
}

static_assert((M_MAX * HD_MAX + NWARPS * ATT_RB * ATT_MB_STRIDE + NWARPS * 40) * 4 <= WORK_BYTES, "attention buffers do not fit in the work area");

}  // namespace kg
