// Prompt processing on the 5th-generation tensor cores.
//
// The decode path streams every weight once per <= 16 rows; for a prompt of hundreds of rows that is the wrong
// trade.  Here a block of up to PF_ROWS prompt rows goes through a layer as real GEMMs C[rows, N] = A[rows, K] W[N, K]^T.
// The activations keep fp32 accuracy the same way as in the decode path: every value is split into two bf16 planes,
// x = hi + lo, and both planes are multiplied with the bf16 weights into the same fp32 accumulator.
//
// Every kernel but the first of a block is launched as a programmatic dependent: it may be set up while the one before still runs and
// waits (grid_dependency_wait) before it touches that one's results (7B: 77 tokens 6.22 -> 5.63 ms, 17 tokens 5.30 -> 4.60; a model of
// four layers with d = 512, 32 tokens: 0.31 -> 0.24).
//
// A layer is seven launches: RMSNorm + split into planes, QKV GEMM (epilogue: rotation, K / V rows into the cache, q
// planes), attention (reads q planes and the cache, writes planes), O GEMM (+ residual), RMSNorm + split, gate / up GEMM
// (epilogue: SwiGLU into planes), down GEMM (+ residual).
#pragma once

#include <cuda.h>

#include "kg_device.cuh"

namespace kg {

constexpr int PF_ROWS = 2048;                  // most prompt rows per pass through the layers
constexpr int GM_BK = 64;                      // k block: one 128-byte swizzle atom of bf16
constexpr int GM_CHAIN = 2;                    // k blocks summed by the tensor core before the sum goes to fp32 registers
constexpr int GM_TM = 256;                     // weight rows per CTA pair (128 in each CTA: the M side of the MMA)
constexpr int GM_NT_MAX = 256;                 // most activation rows per tile (the N side)
constexpr int GM_NT_STEP = 32;                 // widths of a tile (the N of a 256-row MMA of a CTA pair is a multiple of 32)
constexpr int GM_A_BYTES = (GM_TM / 2) * GM_BK * 2;                    // this CTA's weight rows of a k block: 16 KB
constexpr int GM_RING_BYTES = 192 * 1024;
constexpr int GM_MAX_STAGES = 8;
constexpr int GM_MAX_ACC = 4;
constexpr int GM_EPI_WARPS = 8;                // two per tensor-memory lane quadrant, every other 32 columns of the tile each
constexpr int GM_THREADS = 128 + 32 * GM_EPI_WARPS;                    // warp 0: TMA, warp 1: MMA, two idle warps, then the epilogue
constexpr int GM_STAGE_FLOATS = 32 * 32;                               // [32 columns][32 lanes] of one epilogue warp
constexpr int GM_XCH_BYTES = GM_EPI_WARPS * GM_STAGE_FLOATS * 4;
constexpr int GM_SMEM = 1024 + GM_RING_BYTES + GM_XCH_BYTES + 256;     // alignment slack, operand ring, epilogue staging, barriers
static_assert(GM_SMEM <= SMEM_TOTAL, "GEMM shared memory");
// registers: the first warpgroup needs few, the two epilogue warpgroups keep 128 sums and a batch of accumulator columns per
// thread; the pool is what the launch allocated (GM_THREADS x 168), a request beyond it would block for ever
constexpr int GM_CTRL_REGS = 56, GM_EPI_REGS = 216;
static_assert(GM_THREADS == DECODE_THREADS && 128 * GM_CTRL_REGS + 32 * GM_EPI_WARPS * GM_EPI_REGS <= GM_THREADS * LAUNCH_REGS, "register budgets exceed the CTA's pool");
constexpr unsigned long long GM_WAIT_CLK = 4000000000ull;              // ~2 s: a wait that runs this long gives up
constexpr unsigned long long GM_WAIT_CLK_FAILED = GM_WAIT_CLK / 64;    // ~30 ms: once another wait of the prompt pass gave up
enum { PF_ERR_GEMM = 1, PF_ERR_ATT = 2 };                              // the error word: whose wait gave up first

enum { PF_STORE = 0, PF_QKV = 1, PF_SWIGLU = 2 };                      // what the epilogue makes of the products

struct GemmArgs {
    int rows;                           // valid activation rows (rows of the planes beyond them hold anything)
    int N, K;                           // output features (multiple of 128; PF_SWIGLU: of each matrix) and contraction (of 64)
    int nt, nrt;                        // activation rows per tile (a multiple of 32, at most 256) and row tiles
    int full, S, items;                 // work items: `full` whole tiles, then every remaining tile cut into S ranges of k
    const float* rowscale;              // PF_QKV, PF_SWIGLU: one factor per row (1/rms of the row the planes were made from)
    float* C; const float* resid; int ldc;      // PF_STORE: C = (resid) + product; C may be resid itself
    __nv_bfloat16* hi; __nv_bfloat16* lo; int ldp;      // PF_SWIGLU: planes of SiLU(gate) * up; PF_QKV: planes of the rotated, scaled q
    int hd, H, sec0, pos0;              // PF_QKV: sec0 = first section of W's rows (0: q, k, v; 1: k, v only)
    const float2* cs;                   // PF_QKV: cos, sin [rows][hd / 2] of the block's positions
    const int* page_table; int ps_shift, n_phys; State* st;
    __nv_bfloat16* kc; __nv_bfloat16* vc;
    float qscale;
    float* part; unsigned* cnt;         // partial sums of the cut tiles, arrival counters (left at zero)
    int* err;                           // PF_ERR_GEMM when a bounded wait expired
};

// ---- TMA tile copy, tensor memory and tcgen05 MMA ----------------------------------------------------------------
// (one CTA of a pair: the copy lands in this CTA's shared memory and is counted on an mbarrier of either CTA of the pair)
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst_smem, const CUtensorMap* tmap, int x, int y, uint32_t bar_smem) {
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst_smem), "l"(tmap), "r"(x), "r"(y), "r"(bar_smem) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory operand descriptor: K-major, 128-byte swizzle (rows of 128 bytes, groups of 8 rows 1024 bytes apart).
// bits [0,14) address >> 4, [32,46) group stride >> 4, [46,48) version 1, [61,64) layout 2 = 128-byte swizzle.
// Stepping 16 k-elements inside the 64-element atom adds 32 bytes (2 units) to the address field.
constexpr uint32_t UMMA_DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t umma_desc_lo(uint32_t saddr) { return ((saddr & 0x3FFFFu) >> 4) | (1u << 16); }
// Instruction descriptor: fp32 accumulate (bit 4), bf16 A and B (bits 7, 10), both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__device__ __forceinline__ uint32_t umma_idesc(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
// one lane of a converged warp (the same one every time)
__device__ __forceinline__ bool elect_one() {
    unsigned p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
// D[256 x N] (+)= A[256 x 64] B[N x 64]^T over a CTA pair (four k16-steps), issued by one thread of the even CTA: each CTA
// holds 128 rows of A, N / 2 rows of B and its 128 rows of D
__device__ __forceinline__ void umma_kblock_pair(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %5, 0;\n\tsetp.eq.b32 q, %5, %5;\n\tmov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %4, p;\n\tadd.s64 da, da, 2;\n\tadd.s64 db, db, 2;\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %4, q;\n\tadd.s64 da, da, 2;\n\tadd.s64 db, db, 2;\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %4, q;\n\tadd.s64 da, da, 2;\n\tadd.s64 db, db, 2;\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %4, q;\n\t}"
                 ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(UMMA_DESC_HI), "r"(idesc), "r"(accumulate));
}
// the mbarrier of both CTAs of the pair receives one arrival when every MMA this thread has issued so far has completed
__device__ __forceinline__ void umma_commit_pair(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}
// shared-memory address of the same variable in the even CTA of the pair
__device__ __forceinline__ uint32_t leader_smem(uint32_t addr) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
    return r;
}
// (no cluster-scope release: what the arrival hands over is tensor memory whose reads have completed, and that fence would
// stalls while copies are in flight: a drain took 2650 clocks with it and 690 without, and 64 k blocks of a 256 x 256 tile
// 111,000 and 71,000 clocks, 66,000 being the MMAs alone)
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void named_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
// 32 consecutive accumulator columns of this thread's tensor-memory lane (lane = 32 * (warp % 4) + lane id)
// (asynchronous: tmem_ld_wait32() before the values are used)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr) : "memory");
}
// (the values pass through the wait, so that nothing can use them before it)
__device__ __forceinline__ void tmem_ld_wait32(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31]) :: "memory");
}

// Bounded wait on an mbarrier phase; on expiry the error word is set and false returned.  An error word that is set already (*failed) shortens
// the limit, so that a pass in which every kernel fails ends within seconds, but ends no wait at once: nobody waits for another CTA
// (pair), and whoever leaves has either seen what it issued complete or waited for it at least the short limit, so that no copy or
// MMA is in flight.  `failed`: the error word, or a copy from the kernel's start (the attention with heads of 64 has no register for a copy: 1999
// rows of 64 heads 124.9 us, with it 127.0.  GEMM: 7B, 12 layers, 77 tokens 2.042 to 2.051 ms; while a set word ended every wait 2.035).
__device__ __forceinline__ bool gm_wait(unsigned long long* bar, unsigned parity, int* err, const int* failed, int code = PF_ERR_GEMM) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    unsigned spins = 0;
    while (!mbar_try_wait(bar, parity)) {
        if (((++spins) & 255u) == 0u && (unsigned long long)(clock64() - t0) > (*failed ? GM_WAIT_CLK_FAILED : GM_WAIT_CLK)) {
            if (*(volatile int*)err == 0) *(volatile int*)err = code;
            return false;
        }
    }
    return true;
}

// ---- the GEMM ------------------------------------------------------------------------------------------------------
// One CTA pair (cluster of two, cta_group::2) per work item; the grid is persistent (one pair per two SMs).  The weights
// are the M side of the MMA (256 rows of a pair), the activation rows the N side (nt of them), because the weights are
// always whole tiles while a prompt may have any number of rows: nt follows the rows, and the accumulator has one weight
// row per tensor-memory lane.
//
// What bounds it: the operands of a k block.  With the activations in two planes a 128 x 128 tile of one CTA needs 48 KB for
// 4.2 MFLOP (94 bytes per clock and SM at the full MMA rate, more than L2 delivers); the pair's 256 x 256 tile needs 48 KB
// per CTA for 8.4 MFLOP, since the two CTAs share the activation planes.  With the attention below and the fused epilogues
// the prompt pass of the 7B shape (1999 tokens) went from 96.9 to 49.9 ms, of 77 tokens from 9.2 to 5.3 ms.
//
// Accumulation.  The tensor core's fp32 accumulation rounds toward zero at every MMA, by an amount that follows the size
// of the running sum, which biases long chains.  A chain of GM_CHAIN = 2 k blocks multiplies both lo planes first - sums
// about 2^-9 of the result, whose truncation does not count - and then the hi planes: eight truncations that count per
// 128 k, where one accumulator per k block with hi and lo in turn takes sixteen (N(0,1) rows, K = 4096, against float64:
// error 2.459e-6 of the norm and bias -1.06e-7, before 2.465e-6 and -1.41e-7; longer chains lose bits again).  The epilogue warps add every chain to
// fp32 registers (round to nearest) while the next ones are multiplied; the accumulators rotate through tensor memory.
//
// Work items.  Tiles are ordered row tile first, so that the pairs that run at the same time share weight tiles.  The
// last, incomplete wave of tiles is cut into S ranges of k (gm_plan on the host): each range leaves fp32 partial sums in
// global memory, and the CTA that arrives last adds them in the order of the ranges and runs the epilogue; nothing waits.
struct GmItem { int wt, rt, kb0, kb1, s, r; };            // s < 0: a whole tile
__device__ __forceinline__ GmItem gm_item(const GemmArgs& g, int idx) {
    GmItem it;
    const int nkb = g.K / GM_BK;
    int tile = idx;
    it.kb0 = 0; it.kb1 = nkb; it.s = -1; it.r = 0;
    if (idx >= g.full && g.S > 1) {
        const int j = idx - g.full;
        it.r = j / g.S; it.s = j - it.r * g.S;
        tile = g.full + it.r;
        it.kb0 = nkb * it.s / g.S; it.kb1 = nkb * (it.s + 1) / g.S;
    }
    it.wt = tile / g.nrt; it.rt = tile - it.wt * g.nrt;
    return it;
}

__device__ __forceinline__ unsigned pack_bf16(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const unsigned*>(&v);
}

// What the epilogue needs of one activation row: 1 / rms and the row's place in the caches, (physical page * heads) pages of
// page_size slots + slot.  Lane i keeps that of row i of 32 columns, loaded before the k loop.
struct GmRow { float rs; int slot; };
template <int EPI>
__device__ __forceinline__ GmRow gm_row(const GemmArgs& g, int row) {
    GmRow r{0.f, 0};
    if (EPI == PF_STORE || row >= g.rows) return r;
    r.rs = g.rowscale[row];
    if (EPI == PF_QKV) {
        const int pos = g.pos0 + row;
        r.slot = ((checked_page(__ldg(g.page_table + (pos >> g.ps_shift)), g.n_phys, g.st, 61) * g.H) << g.ps_shift) + (pos & ((1 << g.ps_shift) - 1));
    }
    return r;
}
__device__ __forceinline__ void load8(float (&v)[8], const float* p) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
// eight values as bf16, and as bf16 hi + lo planes (16-byte stores)
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float (&v)[8]) {
    *reinterpret_cast<uint4*>(p) = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
}
__device__ __forceinline__ void store8_planes(__nv_bfloat16* hi, __nv_bfloat16* lo, const float (&v)[8]) {
    uint4 h, l;
    split_hi_lo(make_float2(v[0], v[1]), h.x, l.x); split_hi_lo(make_float2(v[2], v[3]), h.y, l.y);
    split_hi_lo(make_float2(v[4], v[5]), h.z, l.z); split_hi_lo(make_float2(v[6], v[7]), h.w, l.w);
    *reinterpret_cast<uint4*>(hi) = h;
    *reinterpret_cast<uint4*>(lo) = l;
}

// The global values that the epilogue of 32 columns reads, requested before the staging: PF_STORE the residual (four columns at
// a time, four features per lane), PF_QKV (cos, sin) of eight dims of this warp's half of the columns.
template <int EPI>
__device__ __forceinline__ void gm_request(const GemmArgs& g, float4 (&rv)[8], int row0, int wt, int rank, int q, int role) {
    const int lane = threadIdx.x & 31, n = wt * GM_TM + rank * (GM_TM / 2) + q * 32;       // this warp's first row of W
    if (EPI == PF_STORE) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int row = row0 + i * 4 + (lane >> 3);
            rv[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (g.resid && row < g.rows && n < g.N) rv[i] = *reinterpret_cast<const float4*>(g.resid + (size_t)row * g.ldc + n + (lane & 7) * 4);
        }
    }
    if (EPI == PF_QKV) {
        const int half = g.hd >> 1, e = (n & (half - 1)) + (lane & 3) * 8;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int row = min(row0 + role * 16 + (i >> 2) * 8 + (lane >> 2), g.rows - 1);
            rv[i] = __ldg(reinterpret_cast<const float4*>(g.cs + (size_t)row * half + e) + (i & 3));
        }
    }
}

// Finished products of 32 columns (activation rows row0 ..) of this warp's 32 weight rows, staged as [column][lane] in
// `mine` (`theirs`: the partner warp's staging).  A lane takes eight neighbouring features of a column.  What bounds it: the
// main loop stands still meanwhile (the accumulator columns of at most nacc chains are ahead), so what counts is the chain
// of dependent steps.  With two features per lane and step, and with the row factors, page numbers and rotations loaded
// where they were used, a 256 x 256 tile's epilogue took 36,000 (QKV) and 23,000 (SwiGLU) clocks beside a k loop of 64,000;
// now 16,000 and 13,000 (7B, 77 tokens 5.6 -> 5.3 ms, 1999 tokens 53.2 -> 49.9 ms).  What is left is the latency of the rotations
// and of the residual and, for SwiGLU, the divisions (about 4,000).
template <int EPI>
__device__ __forceinline__ void gm_epilogue(const GemmArgs& g, const float* mine, const float* theirs, int row0, int wt, int rank, int q, int role,
                                            GmRow gr, const float4 (&rv)[8]) {
    const int lane = threadIdx.x & 31;
    if constexpr (EPI == PF_STORE) {
        const int n = wt * GM_TM + rank * (GM_TM / 2) + q * 32 + (lane & 7) * 4, c0 = lane >> 3;
        if (n >= g.N) return;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int row = row0 + i * 4 + c0;
            const float4 v = *reinterpret_cast<const float4*>(mine + (i * 4 + c0) * 32 + (lane & 7) * 4);
            if (row < g.rows) *reinterpret_cast<float4*>(g.C + (size_t)row * g.ldc + n) = make_float4(rv[i].x + v.x, rv[i].y + v.y, rv[i].z + v.z, rv[i].w + v.w);
        }
    } else {
        // of a pair of warps each takes half of the columns
        const int cl = lane >> 2, fe = (lane & 3) * 8;
        if constexpr (EPI == PF_SWIGLU) {
            const int f = wt * (GM_TM / 2) + rank * (GM_TM / 4) + (q & 1) * 32 + fe;
            const float* ga = role ? theirs : mine;
            const float* up = role ? mine : theirs;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int col = role * 16 + i * 8 + cl, row = row0 + col;
                float a[8], b[8];
                load8(a, ga + col * 32 + fe);
                load8(b, up + col * 32 + fe);
                const float rs = __shfl_sync(0xffffffffu, gr.rs, col);
#pragma unroll
                for (int k = 0; k < 8; ++k) a[k] = silu_f(a[k] * rs) * (b[k] * rs);
                const size_t o = (size_t)row * g.ldp + f;
                if (row < g.rows) store8_planes(g.hi + o, g.lo + o, a);
            }
        } else {
            const int d = g.H * g.hd, half = g.hd >> 1;
            const int n0 = wt * GM_TM + rank * (GM_TM / 2);                 // this CTA's 128 rows of W lie in one section
            if (n0 >= g.N) return;
            const int s0 = n0 / d, sec = s0 + g.sec0, nh = n0 - s0 * d + q * 32;     // this warp's first row within the section
            const int hh = nh >> (half == 64 ? 7 : 6), e0 = nh & (g.hd - 1);
            if (sec == 2) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int col = i * 8 + cl;
                    float v[8];
                    load8(v, mine + col * 32 + fe);
                    const float rs = __shfl_sync(0xffffffffu, gr.rs, col);
                    const int slot = __shfl_sync(0xffffffffu, gr.slot, col) + (hh << g.ps_shift);
#pragma unroll
                    for (int k = 0; k < 8; ++k) v[k] *= rs;
                    if (row0 + col < g.rows) store8(g.vc + (size_t)slot * g.hd + e0 + fe, v);
                }
            } else {
                // dims e .. e + 7 of the first half of the head and their partners half a head further
                const int e = (e0 & (half - 1)) + fe;
                const float* xa = role ? theirs : mine;
                const float* xb = role ? mine : theirs;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int col = role * 16 + i * 8 + cl, row = row0 + col;
                    float a[8], b[8];
                    load8(a, xa + col * 32 + fe);
                    load8(b, xb + col * 32 + fe);
                    const float rs = __shfl_sync(0xffffffffu, gr.rs, col);
                    const int slot = __shfl_sync(0xffffffffu, gr.slot, col) + (hh << g.ps_shift);
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float4 cs = rv[i * 4 + (k >> 1)];
                        const float c = k & 1 ? cs.z : cs.x, sn = k & 1 ? cs.w : cs.y;
                        const float xk = a[k] * rs, yk = b[k] * rs;
                        // (which product is rounded is written out: left to the compiler it changed with the surrounding code)
                        a[k] = fmaf(-yk, sn, xk * c);
                        b[k] = fmaf(xk, sn, yk * c);
                    }
                    if (sec == 0) {
#pragma unroll
                        for (int k = 0; k < 8; ++k) { a[k] *= g.qscale; b[k] *= g.qscale; }
                        const size_t o = (size_t)row * g.ldp + (size_t)hh * g.hd + e;
                        if (row < g.rows) {
                            store8_planes(g.hi + o, g.lo + o, a);
                            store8_planes(g.hi + o + half, g.lo + o + half, b);
                        }
                    } else if (row < g.rows) {
                        __nv_bfloat16* kr = g.kc + (size_t)slot * g.hd + e;
                        store8(kr, a);
                        store8(kr + half, b);
                    }
                }
            }
        }
    }
}

template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GM_THREADS, 1)
pf_gemm_kernel(const __grid_constant__ CUtensorMap tm_hi, const __grid_constant__ CUtensorMap tm_lo, const __grid_constant__ CUtensorMap tm_w,
               const __grid_constant__ CUtensorMap tm_w2, const __grid_constant__ GemmArgs g) {
    extern __shared__ __align__(128) char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw) & 0xFFFFFFu;                   // offset inside this CTA's window
    char* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);              // swizzled tiles sit on 1024-byte boundaries
    float* xch = reinterpret_cast<float*>(smem + GM_RING_BYTES);
    unsigned long long* full = reinterpret_cast<unsigned long long*>(smem + GM_RING_BYTES + GM_XCH_BYTES);   // even CTA: both CTAs' tiles have landed
    unsigned long long* empty = full + GM_MAX_STAGES;      // the stage's MMAs have completed
    unsigned long long* acc_full = empty + GM_MAX_STAGES;  // the accumulator is complete
    unsigned long long* acc_free = acc_full + GM_MAX_ACC;  // even CTA: both CTAs' epilogue warps have read the accumulator
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_free + GM_MAX_ACC);
    int* last_flag = reinterpret_cast<int*>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = blockIdx.x & 1, pair_id = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int stage_bytes = GM_A_BYTES + g.nt * 128;                       // weights, hi plane, lo plane
    const int nst = min(GM_MAX_STAGES, GM_RING_BYTES / stage_bytes);       // 4 (nt = 256) .. 8: at least a chain's stages and as many ahead
    const int nacc = g.nt <= 128 ? 4 : 2, acc_cols = g.nt <= 128 ? 128 : 256;
    if (threadIdx.x == 0) {
        for (int i = 0; i < GM_MAX_STAGES; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
        for (int i = 0; i < GM_MAX_ACC; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_free[i], 2 * GM_EPI_WARPS); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    cluster_sync_all();                                                    // both CTAs' barriers and tensor memory exist
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int failed = *(volatile int*)g.err;             // an earlier kernel of the pass gave up
    grid_dependents_launch();

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(GM_CTRL_REGS));
        if (warp == 0) {
            // ---- TMA producer of this CTA's tiles (the warp stays together, one lane issues)
            int s = 0; unsigned par = 1u;
            const int hrow = g.nt >> 1;
            bool ok = true;
            // the weights do not come from the kernel before: those of the first stages are on their way while it ends
            auto load_w = [&](const GmItem& it, int kb, int stage) {
                const uint32_t dst = smem_u32(smem + stage * stage_bytes), bar = leader_smem(smem_u32(&full[stage]));
                if (rank == 0) mbar_arrive_expect_tx(&full[stage], (unsigned)(2 * stage_bytes));
                if (EPI == PF_SWIGLU) {
                    const int y = it.wt * (GM_TM / 2) + rank * (GM_TM / 4);
                    tma_load_2d_pair(dst, &tm_w, kb * GM_BK, y, bar);
                    tma_load_2d_pair(dst + GM_A_BYTES / 2, &tm_w2, kb * GM_BK, y, bar);
                } else {
                    tma_load_2d_pair(dst, &tm_w, kb * GM_BK, it.wt * GM_TM + rank * (GM_TM / 2), bar);
                }
            };
            int early = 0;
            {
                const GmItem it = gm_item(g, pair_id);
                early = min(nst, it.kb1 - it.kb0);
                if (elect_one()) for (int i = 0; i < early; ++i) load_w(it, it.kb0 + i, i);
                __syncwarp();
            }
            grid_dependency_wait();
            for (int idx = pair_id; idx < g.items && ok; idx += npairs) {
                const GmItem it = gm_item(g, idx);
                const int y_act = it.rt * g.nt + rank * hrow;
                for (int kb = it.kb0; kb < it.kb1; ++kb) {
                    if (!(ok = gm_wait(&empty[s], par, g.err, &failed))) break;
                    if (elect_one()) {
                        if (early == 0) load_w(it, kb, s);
                        const uint32_t dst = smem_u32(smem + s * stage_bytes), bar = leader_smem(smem_u32(&full[s]));
                        const int x = kb * GM_BK;
                        tma_load_2d_pair(dst + GM_A_BYTES, &tm_hi, x, y_act, bar);
                        tma_load_2d_pair(dst + GM_A_BYTES + hrow * 128, &tm_lo, x, y_act, bar);
                    }
                    __syncwarp();
                    if (early > 0) --early;
                    if (++s == nst) { s = 0; par ^= 1u; }
                }
            }
            // every completion arrives in this CTA's shared memory before it may leave
            for (int i = 0; i < nst && ok; ++i) {
                ok = gm_wait(&empty[s], par, g.err, &failed);
                if (++s == nst) { s = 0; par ^= 1u; }
            }
        } else if (warp == 1 && rank == 0) {
            // ---- MMA issuer of the pair.  The warp stays together and one elected lane issues: with a loop that only lane 0 ran,
            // issuing took 115 clocks per instruction, which made every tile of up to 192 columns issue-bound.
            const uint32_t idesc = umma_idesc(GM_TM, g.nt);
            const uint32_t lo_off = (uint32_t)((g.nt >> 1) * 128) >> 4;          // hi plane -> lo plane, in descriptor units
            int s = 0, a = 0; unsigned par = 0u, apar = 1u;
            bool ok = true;
            for (int idx = pair_id; idx < g.items && ok; idx += npairs) {
                const GmItem it = gm_item(g, idx);
                for (int kb = it.kb0; kb < it.kb1 && ok; kb += GM_CHAIN) {
                    const int nb = min(GM_CHAIN, it.kb1 - kb);
                    const uint32_t dcol = tmem + (uint32_t)(a * acc_cols);
                    if (!(ok = gm_wait(&acc_free[a], apar, g.err, &failed))) break;
                    // the lo planes of the chain's k blocks
                    int sl = s; unsigned pl = par;
                    for (int b = 0; b < nb && ok; ++b) {
                        if (!(ok = gm_wait(&full[sl], pl, g.err, &failed))) break;
                        tc_fence_after();
                        const uint32_t base = smem_u32(smem + sl * stage_bytes);
                        const uint32_t w = umma_desc_lo(base), x = umma_desc_lo(base + GM_A_BYTES) + lo_off;
                        if (elect_one()) umma_kblock_pair(dcol, w, x, idesc, b > 0 ? 1u : 0u);
                        __syncwarp();
                        if (++sl == nst) { sl = 0; pl ^= 1u; }
                    }
                    if (!ok) break;
                    // the hi planes; a stage is free after its second pass
                    for (int b = 0; b < nb; ++b) {
                        const uint32_t base = smem_u32(smem + s * stage_bytes);
                        const uint32_t w = umma_desc_lo(base), x = umma_desc_lo(base + GM_A_BYTES);
                        if (elect_one()) {
                            umma_kblock_pair(dcol, w, x, idesc, 1u);
                            umma_commit_pair(&empty[s]);
                            if (b == nb - 1) umma_commit_pair(&acc_full[a]);
                        }
                        __syncwarp();
                        if (++s == nst) { s = 0; par ^= 1u; }
                    }
                    if (++a == nacc) { a = 0; apar ^= 1u; }
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(GM_EPI_REGS));
        grid_dependency_wait();
        // ---- epilogue: thread = one weight row (tensor-memory lane 32 * (warp % 4) + lane id) and every other 32 columns of the tile
        const int ew = warp - 4, q = warp & 3, chalf = ew >> 2, nch = ((g.nt >> 5) + 1 - chalf) >> 1;
        // the partner: the warp with the other half of a rotation (dims e and e + hd / 2) or the up rows of the same features
        const int pbit = (EPI == PF_QKV && g.hd == 64) ? 1 : 2;
        const int role = (q & pbit) ? 1 : 0, pair = pbit == 2 ? (q & 1) * 2 + chalf : (q >> 1) * 2 + chalf;
        float* mine = xch + ew * GM_STAGE_FLOATS;
        const float* theirs = xch + (ew ^ pbit) * GM_STAGE_FLOATS;
        int a = 0; unsigned apar = 0u;
        bool ok = true;                    // after a wait that gave up: the remaining work runs through without waiting (every
                                           // warp takes every named barrier), on values that nobody will use
        for (int idx = pair_id; idx < g.items; idx += npairs) {
            const GmItem it = gm_item(g, idx);
            float acc[GM_NT_MAX / 2];
#pragma unroll
            for (int i = 0; i < GM_NT_MAX / 2; ++i) acc[i] = 0.f;
            GmRow gr[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) gr[c] = gm_row<EPI>(g, it.rt * g.nt + (c * 2 + chalf) * 32 + lane);
            for (int kb = it.kb0; kb < it.kb1; kb += GM_CHAIN) {
                if (ok) ok = gm_wait(&acc_full[a], apar, g.err, &failed);
                __syncwarp();
                tc_fence_after();
                const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(a * acc_cols + chalf * 32);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if (c < nch) {
                        uint32_t v[32];
                        tmem_ld32(ta + 64u * c, v);
                        tmem_ld_wait32(v);
#pragma unroll
                        for (int i = 0; i < 32; ++i) acc[c * 32 + i] += __uint_as_float(v[i]);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(leader_smem(smem_u32(&acc_free[a])));
                if (++a == nacc) { a = 0; apar ^= 1u; }
            }
            const size_t wsize = (size_t)((g.nt + 63) >> 6) * GM_STAGE_FLOATS; // floats of one warp's products (at most)
            const size_t one = 2 * GM_EPI_WARPS * wsize;                   // ... of one range of k (both CTAs)
            float* part = g.part + (size_t)it.r * g.S * one + ((size_t)rank * GM_EPI_WARPS + ew) * wsize + lane;
            bool finish = true;
            if (it.s >= 0) {
                // a range of k: partial sums out; the last of the tile's ranges to arrive adds them in the order of the ranges
                float* dst = part + (size_t)it.s * one;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if (c < nch) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) __stcg(dst + (c * 32 + i) * 32, acc[c * 32 + i]);
                    }
                }
                __threadfence();
                named_sync(5, 32 * GM_EPI_WARPS);
                if (threadIdx.x == 128) {
                    unsigned* cn = g.cnt + it.r * 2 + rank;
                    const int last = atomicAdd(cn, 1u) == (unsigned)(g.S - 1);
                    if (last) { *cn = 0u; __threadfence(); }
                    *(volatile int*)last_flag = last;
                }
                named_sync(5, 32 * GM_EPI_WARPS);
                finish = *(volatile int*)last_flag != 0;
                named_sync(5, 32 * GM_EPI_WARPS);                          // the flag has been read by every warp
            }
            // 32 columns at a time through the staging
            auto staged = [&](int c, const float4 (&rv)[8]) {
                if (EPI == PF_STORE) __syncwarp(); else named_sync(1 + pair, 64);
                gm_epilogue<EPI>(g, mine, theirs, it.rt * g.nt + (c * 2 + chalf) * 32, it.wt, rank, q, role, c == 0 ? gr[0] : c == 1 ? gr[1] : c == 2 ? gr[2] : gr[3], rv);
                if (EPI == PF_STORE) __syncwarp(); else named_sync(1 + pair, 64);
            };
            if (it.s < 0) {
#pragma unroll 1
                for (int c = 0; c < nch; ++c) {
                    float4 rv[8];
                    gm_request<EPI>(g, rv, it.rt * g.nt + (c * 2 + chalf) * 32, it.wt, rank, q, role);
                    switch (c) {
#define KG_STAGE(C) case C: { _Pragma("unroll") for (int i = 0; i < 32; ++i) mine[i * 32 + lane] = acc[C * 32 + i]; } break
                        KG_STAGE(0); KG_STAGE(1); KG_STAGE(2); KG_STAGE(3);
#undef KG_STAGE
                    }
                    staged(c, rv);
                }
            } else if (finish) {
#pragma unroll 1
                for (int c = 0; c < nch; ++c) {
                    float4 rv[8];
                    gm_request<EPI>(g, rv, it.rt * g.nt + (c * 2 + chalf) * 32, it.wt, rank, q, role);
                    float w[32], u[32];                                    // the loads of two ranges in flight (S is at least 2)
                    const float* src = part + c * GM_STAGE_FLOATS;
#pragma unroll
                    for (int i = 0; i < 32; ++i) w[i] = __ldcg(src + i * 32);
#pragma unroll
                    for (int i = 0; i < 32; ++i) u[i] = __ldcg(src + one + i * 32);
#pragma unroll
                    for (int i = 0; i < 32; ++i) w[i] += u[i];
#pragma unroll 1
                    for (int s = 2; s < g.S; s += 2) {
                        const float* s0 = src + (size_t)s * one;
                        const bool two = s + 1 < g.S;
                        float x[32];
#pragma unroll
                        for (int i = 0; i < 32; ++i) u[i] = __ldcg(s0 + i * 32);
#pragma unroll
                        for (int i = 0; i < 32; ++i) x[i] = two ? __ldcg(s0 + one + i * 32) : 0.f;
#pragma unroll
                        for (int i = 0; i < 32; ++i) w[i] += u[i];
                        if (two) {
#pragma unroll
                            for (int i = 0; i < 32; ++i) w[i] += x[i];
                        }
                    }
#pragma unroll
                    for (int i = 0; i < 32; ++i) mine[i * 32 + lane] = w[i];
                    staged(c, rv);
                }
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    cluster_sync_all();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// ---- attention of a block of prompt rows -----------------------------------------------------------------------------
// One CTA = 128 query rows of one head (8 warps x 16 rows); key tiles of 64 travel cache -> shared memory with cp.async,
// three tiles in flight, and are read by every warp with ldmatrix.  S = Q K^T and O += P V on mma.sync.m16n8k16 with q
// and P as bf16 hi + lo, online softmax in the log2 domain (q carries log2(e) / sqrt(hd)).  CTAs with the most keys start first.
//
// What bounds it: the tensor instructions (256 per warp and tile).  The rows of a tile share K and V: with 16-row items
// (the decode path's tiles, 8 keys x 16 rows per step) every key was fetched from L2 and passed through a serial
// score - exchange - softmax chain once per 16 rows (7B, 1999 rows, one layer: 0.20 ms; with 16-row items about 0.9 ms).
constexpr int FA_ROWS = 128, FA_KEYS = 64, FA_STAGES = 3;
template <int HD> struct FaSm { static constexpr int TILE = FA_KEYS * HD * 2, BYTES = FA_STAGES * 2 * TILE; };

__device__ __forceinline__ void cp_async16(uint32_t dst_smem, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst_smem), "l"(src) : "memory");
}
struct FaArgs {
    const __nv_bfloat16* qh; const __nv_bfloat16* ql;    // [rows][d] rotated, scaled q
    const __nv_bfloat16* kc; const __nv_bfloat16* vc;    // this layer's cache
    __nv_bfloat16* oh; __nv_bfloat16* ol;                // [rows][d] planes of the output
    const int* page_table; int ps_shift, n_phys; State* st;
    int H, pos0, rows;
    int row0; int* err;                                  // pf_attention_tc_kernel: first row of the layer in the caches' tensor maps; PF_ERR_ATT when a bounded wait expired
    int skip;                                            // test hook: this CTA's first softmax warp leaves out the arrival of its first tile (-1: none)
};

template <int HD>
__global__ void __launch_bounds__(256, 1) pf_attention_kernel(const __grid_constant__ FaArgs a) {
    extern __shared__ __align__(128) char smem_raw[];
    constexpr int NK = HD / 16, CH = HD / 8;               // k16-steps of a head; 16-byte chunks of a row
    const uint32_t sm = smem_u32(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int d = a.H * HD, psm = (1 << a.ps_shift) - 1;
    const int nblk = (a.rows + FA_ROWS - 1) / FA_ROWS;
    const int rb = nblk - 1 - blockIdx.x / a.H, hh = blockIdx.x % a.H;
    const int r0 = rb * FA_ROWS, rend = min(a.rows, r0 + FA_ROWS);
    const int T = a.pos0 + rend;                           // keys any row of the block may see
    const int ntile = (T + FA_KEYS - 1) / FA_KEYS;

    auto issue = [&](int ti) {
        const uint32_t kb = sm + (uint32_t)(ti % FA_STAGES) * (2 * FaSm<HD>::TILE), vb = kb + FaSm<HD>::TILE;
#pragma unroll
        for (int i = 0; i < FA_KEYS * CH / 256; ++i) {
            const int id = tid + i * 256, r = id / CH, c = id % CH;
            const int key = min(ti * FA_KEYS + r, T - 1);
            const int page = checked_page(__ldg(a.page_table + (key >> a.ps_shift)), a.n_phys, a.st, 63);
            const size_t src = ((((size_t)page * a.H + hh) << a.ps_shift) + (key & psm)) * HD + c * 8;
            const uint32_t o = (uint32_t)(r * HD * 2 + ((c ^ (r & 7)) << 4));
            cp_async16(kb + o, a.kc + src);
            cp_async16(vb + o, a.vc + src);
        }
    };
    grid_dependents_launch();
    grid_dependency_wait();
    issue(0);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (ntile > 1) issue(1);
    asm volatile("cp.async.commit_group;" ::: "memory");

    // this warp's 16 rows: q fragments (rows past the end repeat the last row and are not stored)
    const int wr0 = r0 + warp * 16;
    const int ra = min(wr0 + g, a.rows - 1), rb8 = min(wr0 + g + 8, a.rows - 1);
    unsigned qh[NK][4], ql[NK][4];
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        const size_t o1 = (size_t)ra * d + hh * HD + k * 16 + 2 * t, o2 = (size_t)rb8 * d + hh * HD + k * 16 + 2 * t;
        qh[k][0] = *reinterpret_cast<const unsigned*>(a.qh + o1); qh[k][1] = *reinterpret_cast<const unsigned*>(a.qh + o2);
        qh[k][2] = *reinterpret_cast<const unsigned*>(a.qh + o1 + 8); qh[k][3] = *reinterpret_cast<const unsigned*>(a.qh + o2 + 8);
        ql[k][0] = *reinterpret_cast<const unsigned*>(a.ql + o1); ql[k][1] = *reinterpret_cast<const unsigned*>(a.ql + o2);
        ql[k][2] = *reinterpret_cast<const unsigned*>(a.ql + o1 + 8); ql[k][3] = *reinterpret_cast<const unsigned*>(a.ql + o2 + 8);
    }
    float o[HD / 8][4];
#pragma unroll
    for (int n = 0; n < HD / 8; ++n) { o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f; }
    float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
    const int lim0 = a.pos0 + wr0 + g, lim1 = lim0 + 8;     // last key each of the two rows may see
    const int wlast = a.pos0 + wr0 + 15;                    // no row of this warp sees a key beyond

    for (int ti = 0; ti < ntile; ++ti) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();                                    // tile ti has landed for everybody; everybody is done with tile ti - 1
        if (ti + 2 < ntile) issue(ti + 2);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const int key0 = ti * FA_KEYS;
        if (key0 > wlast || wr0 >= a.rows) continue;
        const uint32_t kb = sm + (uint32_t)(ti % FA_STAGES) * (2 * FaSm<HD>::TILE), vb = kb + FaSm<HD>::TILE;
        float s[8][4];
#pragma unroll
        for (int n = 0; n < 8; ++n) { s[n][0] = s[n][1] = s[n][2] = s[n][3] = 0.f; }
#pragma unroll
        for (int k = 0; k < NK; ++k) {
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int r = p * 16 + (lane >> 4) * 8 + (lane & 7), c = k * 2 + ((lane >> 3) & 1);
                unsigned b[4];
                ldmatrix_x4(b, kb + (uint32_t)(r * HD * 2 + ((c ^ (r & 7)) << 4)));
                mma_bf16_16816(s[2 * p], qh[k], b[0], b[1]);
                mma_bf16_16816(s[2 * p + 1], qh[k], b[2], b[3]);
                mma_bf16_16816(s[2 * p], ql[k], b[0], b[1]);
                mma_bf16_16816(s[2 * p + 1], ql[k], b[2], b[3]);
            }
        }
        if (key0 + FA_KEYS - 1 > a.pos0 + wr0) {            // the tile crosses the diagonal of this warp's rows
#pragma unroll
            for (int n = 0; n < 8; ++n) {
                const int k0 = key0 + n * 8 + 2 * t;
                if (k0 > lim0) s[n][0] = -INFINITY;
                if (k0 + 1 > lim0) s[n][1] = -INFINITY;
                if (k0 > lim1) s[n][2] = -INFINITY;
                if (k0 + 1 > lim1) s[n][3] = -INFINITY;
            }
        }
        float x0 = s[0][0], x1 = s[0][2];
#pragma unroll
        for (int n = 0; n < 8; ++n) { x0 = fmaxf(x0, fmaxf(s[n][0], s[n][1])); x1 = fmaxf(x1, fmaxf(s[n][2], s[n][3])); }
        x0 = fmaxf(x0, __shfl_xor_sync(0xffffffffu, x0, 1)); x0 = fmaxf(x0, __shfl_xor_sync(0xffffffffu, x0, 2));
        x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, 1)); x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, 2));
        // key 0 is visible to every row, so the maxima are finite from the first tile on
        const float n0 = fmaxf(m0, x0), n1 = fmaxf(m1, x1);
        const float c0 = ex2f(m0 - n0), c1 = ex2f(m1 - n1);
        m0 = n0; m1 = n1;
        float a0 = 0.f, a1 = 0.f;
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            s[n][0] = ex2f(s[n][0] - n0); s[n][1] = ex2f(s[n][1] - n0); s[n][2] = ex2f(s[n][2] - n1); s[n][3] = ex2f(s[n][3] - n1);
            a0 += s[n][0] + s[n][1]; a1 += s[n][2] + s[n][3];
        }
        l0 = l0 * c0 + a0; l1 = l1 * c1 + a1;
#pragma unroll
        for (int n = 0; n < HD / 8; ++n) { o[n][0] *= c0; o[n][1] *= c0; o[n][2] *= c1; o[n][3] *= c1; }
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            unsigned ph[4], pl[4];
            split_hi_lo(make_float2(s[2 * kk][0], s[2 * kk][1]), ph[0], pl[0]);
            split_hi_lo(make_float2(s[2 * kk][2], s[2 * kk][3]), ph[1], pl[1]);
            split_hi_lo(make_float2(s[2 * kk + 1][0], s[2 * kk + 1][1]), ph[2], pl[2]);
            split_hi_lo(make_float2(s[2 * kk + 1][2], s[2 * kk + 1][3]), ph[3], pl[3]);
#pragma unroll
            for (int n = 0; n < HD / 16; ++n) {
                const int r = kk * 16 + ((lane >> 3) & 1) * 8 + (lane & 7), c = n * 2 + (lane >> 4);
                unsigned b[4];
                ldmatrix_x4_trans(b, vb + (uint32_t)(r * HD * 2 + ((c ^ (r & 7)) << 4)));
                mma_bf16_16816(o[2 * n], ph, b[0], b[1]);
                mma_bf16_16816(o[2 * n + 1], ph, b[2], b[3]);
                mma_bf16_16816(o[2 * n], pl, b[0], b[1]);
                mma_bf16_16816(o[2 * n + 1], pl, b[2], b[3]);
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    l0 += __shfl_xor_sync(0xffffffffu, l0, 1); l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
    l1 += __shfl_xor_sync(0xffffffffu, l1, 1); l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
    const float i0 = 1.0f / l0, i1 = 1.0f / l1;
#pragma unroll
    for (int n = 0; n < HD / 8; ++n) {
        unsigned hi, lo;
        const size_t col = (size_t)hh * HD + n * 8 + 2 * t;
        if (wr0 + g < a.rows) {
            split_hi_lo(make_float2(o[n][0] * i0, o[n][1] * i0), hi, lo);
            *reinterpret_cast<unsigned*>(a.oh + (size_t)(wr0 + g) * d + col) = hi;
            *reinterpret_cast<unsigned*>(a.ol + (size_t)(wr0 + g) * d + col) = lo;
        }
        if (wr0 + g + 8 < a.rows) {
            split_hi_lo(make_float2(o[n][2] * i1, o[n][3] * i1), hi, lo);
            *reinterpret_cast<unsigned*>(a.oh + (size_t)(wr0 + g + 8) * d + col) = hi;
            *reinterpret_cast<unsigned*>(a.ol + (size_t)(wr0 + g + 8) * d + col) = lo;
        }
    }
}

// ---- the same on the 5th-generation tensor cores, for blocks of many rows and keys --------------------------------------
// One CTA = 128 query rows of one head, one row per tensor-memory lane; key tiles of 128.  Warp 0 brings K and V tiles (TMA, pages of
// the cache in boxes of up to 16 keys x 64 dims, two stages each), warp 1 issues the MMAs, eight warps do the softmax, two threads per
// row (64 keys, and HD / 2 dims of the output each).  Tensor memory: two score tiles, each overwritten by its P in two planes (the A operand of the
// second product), and the products of two tiles with V.  S(j + 1) is issued before P(j) V, so that the tensor cores work while tile
// j's softmax runs; a product is read two tiles later, beside the scores, when nobody has to wait for it.  The softmax warps of
// different rows may therefore be a tile apart, and all of them a tile ahead of the MMAs, so that P has a barrier for each of the two
// tiles: on one for all tiles, a fast warp's arrival for tile j + 1 would count for a slow one's for tile j.
//
// Precision: q and P in two bf16 planes, softmax and the sum over the tiles in fp32, as in the kernel above.  The lo planes are
// multiplied first, and a tile's P V starts from zero and is added to registers, so that fewer of the tensor core's truncations count: rows against
// float64, mean of the norm, the kernel above / this one, 300 rows 2.96e-6 / 2.88e-6, 1999 rows 4.2e-6 / 2.9e-6, 33 rows behind 2048 keys 6.1e-6 / 3.0e-6.
//
// What bounds it: per tile 2048 clocks of MMAs (both planes) beside about as many of exponentials, splits and tensor-memory traffic.  7B, one layer
// (us, the kernel above / this one): 512 rows 32.9 / 20.5, 1000 62.7 / 37.6, 1999 211 / 102; prompt pass of 1999 tokens 51.2 -> 47.9 ms.  At 1999
// rows a tile takes about 5000 clocks: what bounds it is the latency of the softmax chain (issue slots 35 % busy, tensor pipe 37 %) and, per CTA, its
// start and end (about 5 us).
constexpr int FT_ROWS = 128, FT_KEYS = 128, FT_THREADS = 384, FT_SOFT_WARPS = 8;
// Up to here the kernel above is the better one or as good (us, the kernel above / this one; 32 heads of 128: 33 rows 9.2 / 10.3, 64 10.3 / 12.3, 128 14.4 /
// 14.4, 256 20.5 / 16.4; 64 heads of 64: 64 rows 8.2 / 10.3, 128 10.3 / 10.3, 256 14.4 / 12.3).  Rows do not matter beside the keys: 1 row behind 2048
// keys 73 / 43, of 64 dims 43 / 33 (behind 128 keys of 64 dims up to 32 rows would be 1 to 2 us slower, but at least 1024 rows come before a block).
constexpr int FT_MIN_KEYS = 128;
constexpr int FT_CTRL_REGS = 56, FT_SOFT_REGS = 216;
static_assert(128 * FT_CTRL_REGS + 32 * FT_SOFT_WARPS * FT_SOFT_REGS <= FT_THREADS * LAUNCH_REGS, "register budgets exceed the CTA's pool");
template <int HD> struct FtSm {
    static constexpr int PLANE = FT_ROWS * HD * 2, TILE = FT_KEYS * HD * 2;
    static constexpr int KOFF = 2 * PLANE, VOFF = KOFF + 2 * TILE, CTRL = VOFF + 2 * TILE;
    static constexpr int BYTES = 1024 + CTRL + 2048 + 256;               // alignment slack, operands, maxima / sums of the row halves, barriers
};
constexpr uint32_t FT_S = 0, FT_O = 256;                                 // tensor-memory columns: S [2][128], each overwritten by its P (hi, lo: 64 each); P V [2][128]

__device__ __forceinline__ void umma_commit_one(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void umma_ss(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(UMMA_DESC_HI), "r"(idesc), "r"(accumulate));
}
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 db;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b64 db, {%2, %3};\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(UMMA_DESC_HI), "r"(idesc), "r"(accumulate));
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
                 : "memory");
}

template <int HD>
__global__ void __launch_bounds__(FT_THREADS, 1) pf_attention_tc_kernel(const __grid_constant__ CUtensorMap tmk, const __grid_constant__ CUtensorMap tmv,
                                                                        const __grid_constant__ FaArgs a) {
    extern __shared__ __align__(128) char smem_raw[];
    using G = FtSm<HD>;
    constexpr int HALVES = HD / 64;                        // 64-dim (128-byte) halves of a row
    const uint32_t raw = smem_u32(smem_raw);
    char* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);            // swizzled tiles sit on 1024-byte boundaries
    float* part = reinterpret_cast<float*>(smem + G::CTRL);              // [2 turns][2 halves][128 rows]
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(smem + G::CTRL + 2048);
    unsigned long long *k_full = bar, *k_empty = bar + 2, *v_full = bar + 4, *v_empty = bar + 6, *s_full = bar + 8, *o_full = bar + 10;
    unsigned long long *p_full = bar + 12, *q_full = bar + 14;
    unsigned long long* drained = bar + 15;                // the MMAs issued before a wait gave up have completed
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar + 16);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nblk = (a.rows + FT_ROWS - 1) / FT_ROWS;
    const int rb = nblk - 1 - blockIdx.x / a.H, hh = blockIdx.x % a.H;  // those with the most keys first
    const int r0 = rb * FT_ROWS, rend = min(a.rows, r0 + FT_ROWS);
    const int T = a.pos0 + rend;                           // keys any row of the block may see
    const int ntile = (T + FT_KEYS - 1) / FT_KEYS;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 16; ++i) mbar_init(bar + i, i >= 12 && i < 15 ? FT_SOFT_WARPS : 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    grid_dependents_launch();

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(FT_CTRL_REGS));
        grid_dependency_wait();
        if (warp == 0) {
            // ---- K and V tiles; boxes without a valid key are left out
            asm volatile("fence.proxy.async;" ::: "memory");
            const int bsh = min(a.ps_shift, 4), psm = (1 << a.ps_shift) - 1;      // a box holds 2^bsh keys
            bool ok = true;
            int nk = 0, nv = 0;                            // tiles on their way
            auto load = [&](const CUtensorMap* tm, int j, uint32_t dst, unsigned long long* full) {
                const int nbox = (min(FT_KEYS, T - j * FT_KEYS) + (1 << bsh) - 1) >> bsh;
                if (lane == 0) mbar_arrive_expect_tx(full, (unsigned)(nbox * HALVES * (128 << bsh)));
                __syncwarp();
                for (int i = lane; i < nbox * HALVES; i += 32) {
                    const int b = i / HALVES, half = i % HALVES, key = j * FT_KEYS + (b << bsh);
                    const int page = checked_page(__ldg(a.page_table + (key >> a.ps_shift)), a.n_phys, a.st, 64);
                    tma_load_2d(dst + (uint32_t)(half * (FT_KEYS * 128) + (b << (bsh + 7))), tm, half * 64, a.row0 + ((page * a.H + hh) << a.ps_shift) + (key & psm), smem_u32(full));
                }
                __syncwarp();
            };
            for (int j = 0; j < ntile && ok; ++j) {
                const int s = j & 1; const unsigned par = ((unsigned)(j >> 1) & 1u) ^ 1u;
                if (!(ok = __all_sync(0xffffffffu, gm_wait(&k_empty[s], par, a.err, a.err, PF_ERR_ATT)))) break;
                load(&tmk, j, smem_u32(smem + G::KOFF + s * G::TILE), &k_full[s]); ++nk;
                if (!(ok = __all_sync(0xffffffffu, gm_wait(&v_empty[s], par, a.err, a.err, PF_ERR_ATT)))) break;
                load(&tmv, j, smem_u32(smem + G::VOFF + s * G::TILE), &v_full[s]); ++nv;
            }
            // every completion arrives in this CTA's shared memory before it may leave
            for (int j = max(0, ntile - 2); j < ntile && ok; ++j)
                ok = gm_wait(&k_empty[j & 1], (unsigned)(j >> 1) & 1u, a.err, a.err, PF_ERR_ATT) && gm_wait(&v_empty[j & 1], (unsigned)(j >> 1) & 1u, a.err, a.err, PF_ERR_ATT);
            if (!ok) {                                     // no MMA may come to empty the tiles, so the copies themselves are waited for
                for (int j = max(0, nk - 2); j < nk; ++j) gm_wait(&k_full[j & 1], (unsigned)(j >> 1) & 1u, a.err, a.err, PF_ERR_ATT);
                for (int j = max(0, nv - 2); j < nv; ++j) gm_wait(&v_full[j & 1], (unsigned)(j >> 1) & 1u, a.err, a.err, PF_ERR_ATT);
            }
        } else if (warp == 1) {
            // ---- MMAs: S(j), then P(j - 1) V(j - 1).  S(j) overwrites P(j - 2), whose product must be complete
            const uint32_t sbase = smem_u32(smem);
            const uint32_t id_s = umma_idesc(FT_ROWS, FT_KEYS), id_o = umma_idesc(FT_ROWS, HD) | (1u << 16);       // V: dims are contiguous (MN-major)
            bool ok = __all_sync(0xffffffffu, gm_wait(q_full, 0u, a.err, a.err, PF_ERR_ATT));
            for (int j = 0; j <= ntile && ok; ++j) {
                if (j < ntile) {
                    const int s = j & 1; const unsigned par = (unsigned)(j >> 1) & 1u;
                    if (!(ok = __all_sync(0xffffffffu, gm_wait(&k_full[s], par, a.err, a.err, PF_ERR_ATT) && (j < 2 || gm_wait(&o_full[s], par ^ 1u, a.err, a.err, PF_ERR_ATT))))) break;
                    tc_fence_after();
                    if (elect_one()) {
#pragma unroll
                        for (int pl = 1; pl >= 0; --pl) {              // lo, hi
#pragma unroll
                            for (int k = 0; k < HD / 16; ++k) {
                                const uint32_t o = (uint32_t)((k >> 2) * (FT_KEYS * 128) + (k & 3) * 32);
                                umma_ss(tmem + FT_S + 128u * s, umma_desc_lo(sbase + pl * G::PLANE + o), umma_desc_lo(sbase + G::KOFF + s * G::TILE + o), id_s, pl == 1 && k == 0 ? 0u : 1u);
                            }
                        }
                        umma_commit_one(&k_empty[s]);
                        umma_commit_one(&s_full[s]);
                    }
                    __syncwarp();
                }
                if (j > 0) {
                    const int i = j - 1, s = i & 1;
                    if (!(ok = __all_sync(0xffffffffu, gm_wait(&v_full[s], (unsigned)(i >> 1) & 1u, a.err, a.err, PF_ERR_ATT)))) break;
                    const int nv = T - i * FT_KEYS;                    // V rows without a key hold anything (0 * NaN would be NaN)
                    if (nv < FT_KEYS) {
                        for (int x = lane; x < (FT_KEYS - nv) * HALVES * 8; x += 32) {
                            const int c = x & 7, half = (x >> 3) % HALVES, r = nv + (x >> 3) / HALVES;
                            *reinterpret_cast<uint4*>(smem + G::VOFF + s * G::TILE + half * (FT_KEYS * 128) + r * 128 + c * 16) = make_uint4(0u, 0u, 0u, 0u);
                        }
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                    }
                    if (!(ok = __all_sync(0xffffffffu, gm_wait(&p_full[s], (unsigned)(i >> 1) & 1u, a.err, a.err, PF_ERR_ATT)))) break;
                    tc_fence_after();
                    if (elect_one()) {
#pragma unroll
                        for (int pl = 1; pl >= 0; --pl) {
#pragma unroll
                            for (int k = 0; k < FT_KEYS / 16; ++k)
                                umma_ts(tmem + FT_O + 128u * s, tmem + FT_S + 128u * s + 64u * pl + 8u * k,
                                        (((sbase + G::VOFF + s * G::TILE + k * 2048) & 0x3FFFFu) >> 4) | ((uint32_t)(FT_KEYS * 128 / 16) << 16), id_o, pl == 1 && k == 0 ? 0u : 1u);
                        }
                        umma_commit_one(&v_empty[s]);
                        umma_commit_one(&o_full[s]);
                    }
                    __syncwarp();
                }
            }
            if (!ok) {                                     // tensor memory is given back after the MMAs that write it
                __syncwarp();
                if (elect_one()) umma_commit_one(drained);
                __syncwarp();
                gm_wait(drained, 0u, a.err, a.err, PF_ERR_ATT);
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(FT_SOFT_REGS));
        grid_dependency_wait();
        const int d = a.H * HD;
        {
            // q planes -> shared memory, 128-byte swizzle (rows past the end repeat the last row and are not stored)
            constexpr int CH = HD / 8;
            const int tid = threadIdx.x - 128;
#pragma unroll
            for (int pl = 0; pl < 2; ++pl) {
#pragma unroll
                for (int i = 0; i < FT_ROWS * CH / 256; ++i) {
                    const int id = tid + i * 256, r = id / CH, c = id % CH;
                    const uint4 v = *reinterpret_cast<const uint4*>((pl ? a.ql : a.qh) + (size_t)min(r0 + r, a.rows - 1) * d + hh * HD + c * 8);
                    *reinterpret_cast<uint4*>(smem + pl * G::PLANE + (c >> 3) * (FT_ROWS * 128) + r * 128 + (((c & 7) ^ (r & 7)) << 4)) = v;
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(q_full);
        }
        const int sw = warp - 4, q = sw & 3, half = sw >> 2, row = q * 32 + lane;
        const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16);             // this warp's lanes
        const int lim = min(a.pos0 + r0 + row, T - 1);                     // last key this row may see
        constexpr int OC = HD / 2;                                         // dims of the output this thread keeps
        float o[OC];
#pragma unroll
        for (int i = 0; i < OC; ++i) o[i] = 0.f;
        float m = -INFINITY, l = 0.f;
        bool ok = true;                    // after a wait that gave up the rest runs through without waiting, on values nobody will use
        // the product of tile j, columns 32 c ..
        auto request_o = [&](int j, int c, uint32_t (&v)[32]) { tmem_ld32(tl + FT_O + 128u * (j & 1) + (uint32_t)(half * OC + c * 32), v); };
        auto wait_o = [&](int j) {
            if (ok) ok = gm_wait(&o_full[j & 1], (unsigned)(j >> 1) & 1u, a.err, a.err, PF_ERR_ATT);
            __syncwarp();
            tc_fence_after();
        };
        const int skip = a.skip == (int)blockIdx.x && warp == 4 ? 0 : -1;
        float cf = 1.f;                                                    // scale of the tile before, relative to the one before that
        for (int j = 0; j < ntile; ++j) {
            const int s = j & 1, key0 = j * FT_KEYS + half * 64;
            if (ok) ok = gm_wait(&s_full[s], (unsigned)(j >> 1) & 1u, a.err, a.err, PF_ERR_ATT);
            __syncwarp();
            tc_fence_after();
            uint32_t w0[32], w1[32], v[32];
            tmem_ld32(tl + FT_S + 128u * s + 64u * half, w0);
            tmem_ld32(tl + FT_S + 128u * s + 64u * half + 32u, w1);
            // (the product of tile j - 2 is complete: S(j) comes after it)
            if (j > 1) {
                wait_o(j - 2);
                request_o(j - 2, 0, v);
            }
            tmem_ld_wait32(w0);
            tmem_ld_wait32(w1);
            float x[64];
#pragma unroll
            for (int i = 0; i < 32; ++i) { x[i] = __uint_as_float(w0[i]); x[32 + i] = __uint_as_float(w1[i]); }
            if (j * FT_KEYS + FT_KEYS - 1 > a.pos0 + r0) {                 // the tile crosses the diagonal of the block
#pragma unroll
                for (int i = 0; i < 64; ++i) if (key0 + i > lim) x[i] = -INFINITY;
            }
            float mx[4] = {x[0], x[1], x[2], x[3]};
#pragma unroll
            for (int i = 4; i < 64; ++i) mx[i & 3] = fmaxf(mx[i & 3], x[i]);
            mx[0] = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
            part[(s * 2 + half) * FT_ROWS + row] = mx[0];
            if (j > 1) {                                                   // while the other half's maximum is on its way
                tmem_ld_wait32(v);
#pragma unroll
                for (int i = 0; i < 32; ++i) o[i] = (o[i] + __uint_as_float(v[i])) * cf;
                if constexpr (OC > 32) request_o(j - 2, 1, v);
            }
            named_sync(1 + q, 64);                                         // the two warps of these rows
            // key 0 is visible to every row, so the maxima are finite from the first tile on
            const float mn = fmaxf(m, fmaxf(mx[0], part[(s * 2 + (half ^ 1)) * FT_ROWS + row]));
            const float cf_new = ex2f(m - mn);
            m = mn;
            float sum[4] = {0.f, 0.f, 0.f, 0.f};
            uint32_t ph[32], pl[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const float p0 = ex2f(x[2 * i] - mn), p1 = ex2f(x[2 * i + 1] - mn);
                sum[i & 3] += p0 + p1;
                split_hi_lo(make_float2(p0, p1), ph[i], pl[i]);
            }
            l = l * cf_new + ((sum[0] + sum[1]) + (sum[2] + sum[3]));
            if constexpr (OC > 32) {
                if (j > 1) {
                    tmem_ld_wait32(v);
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[OC - 32 + i] = (o[OC - 32 + i] + __uint_as_float(v[i])) * cf;
                }
            }
            cf = cf_new;
            // (both halves of the scores have been read: the barrier above)
            const uint32_t tp = tl + FT_S + 128u * s + 32u * half;
            tmem_st16(tp, ph); tmem_st16(tp + 16u, ph + 16);
            tmem_st16(tp + 64u, pl); tmem_st16(tp + 80u, pl + 16);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0 && j != skip) mbar_arrive(&p_full[s]);
        }
        // the products of the last two tiles (the last but one at the scale before cf)
        for (int j = max(0, ntile - 2); j < ntile; ++j) {
            wait_o(j);
#pragma unroll
            for (int c = 0; c < OC / 32; ++c) {
                uint32_t v[32];
                request_o(j, c, v);
                tmem_ld_wait32(v);
#pragma unroll
                for (int i = 0; i < 32; ++i) { o[c * 32 + i] += __uint_as_float(v[i]); if (j < ntile - 1) o[c * 32 + i] *= cf; }
            }
        }
        part[half * FT_ROWS + row] = l;                                    // (the last tile's maxima have been read, or lie in the other turn)
        named_sync(1 + q, 64);
        const float il = 1.0f / (l + part[(half ^ 1) * FT_ROWS + row]);
        if (r0 + row < rend) {
            const size_t at = (size_t)(r0 + row) * d + (size_t)hh * HD + half * OC;
#pragma unroll
            for (int i = 0; i < OC; i += 8) {
                float v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = o[i + k] * il;
                store8_planes(a.oh + at + i, a.ol + at + i, v);
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// ---- elementwise kernels around the GEMMs ----------------------------------------------------------------------------
// h[r] = E[token r], eight columns per thread (d is a multiple of 128)
__global__ void __launch_bounds__(256) pf_embed_kernel(const int* toks, const __nv_bfloat16* E, int V, int d, float* h) {
    const int r = blockIdx.x;
    int tok = toks[r];
    if ((unsigned)tok >= (unsigned)V) tok = 0;
    for (int e = threadIdx.x * 8; e < d; e += 256 * 8) {
        const uint4 v = *reinterpret_cast<const uint4*>(E + (size_t)tok * d + e);
        float4* out = reinterpret_cast<float4*>(h + (size_t)r * d + e);
        out[0] = make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
        out[1] = make_float4(__uint_as_float(v.z << 16), __uint_as_float(v.z & 0xffff0000u), __uint_as_float(v.w << 16), __uint_as_float(v.w & 0xffff0000u));
    }
}

// cos, sin of every (position, pair of dims), once per model; grid = positions, hd / 2 threads
__global__ void rope_table_kernel(const __grid_constant__ Dev D, float2* cs) {
    float c, s;
    rope_cs(D, blockIdx.x, threadIdx.x, c, s);
    cs[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = make_float2(c, s);
}

// four consecutive values -> four bf16 of each plane (8-byte stores; i is a multiple of 4)
__device__ __forceinline__ void split_store4(__nv_bfloat16* hi, __nv_bfloat16* lo, size_t i, float4 v) {
    const __nv_bfloat162 h0 = __floats2bfloat162_rn(v.x, v.y), h1 = __floats2bfloat162_rn(v.z, v.w);
    const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
    const __nv_bfloat162 l0 = __floats2bfloat162_rn(v.x - f0.x, v.y - f0.y), l1 = __floats2bfloat162_rn(v.z - f1.x, v.w - f1.y);
    uint2 hv, lv;
    hv.x = *reinterpret_cast<const unsigned*>(&h0); hv.y = *reinterpret_cast<const unsigned*>(&h1);
    lv.x = *reinterpret_cast<const unsigned*>(&l0); lv.y = *reinterpret_cast<const unsigned*>(&l1);
    *reinterpret_cast<uint2*>(hi + i) = hv;
    *reinterpret_cast<uint2*>(lo + i) = lv;
}

// planes of x[r] * gain and rs[r] = 1 / rms(x[r]): the GEMM that reads the
// planes multiplies its rows by rs afterwards, in fp32, exactly as the decode path's linear operator does (values that
// are exact in bf16, such as embedding rows under a unit gain, then stay exact).  One CTA of PF_EW_THREADS threads per
// row; the row (K a multiple of 4, at most PF_EW_THREADS * 4 * PF_NORM_V values) is read once and kept in registers.
constexpr int PF_EW_THREADS = 256;
constexpr int PF_NORM_V = 8;                  // float4 per thread: rows of up to 8192 values
__global__ void __launch_bounds__(PF_EW_THREADS) pf_norm_split_kernel(const float* x, int ldx, int K, const float* gain, float eps,
                                                                      __nv_bfloat16* hi, __nv_bfloat16* lo, float* rs) {
    __shared__ float red[32];
    grid_dependents_launch();
    grid_dependency_wait();
    const int r = blockIdx.x;
    const float4* xr = reinterpret_cast<const float4*>(x + (size_t)r * ldx);
    const int n4 = K >> 2;
    float4 v[PF_NORM_V];
#pragma unroll
    for (int j = 0; j < PF_NORM_V; ++j) {
        const int i = threadIdx.x + j * PF_EW_THREADS;
        v[j] = i < n4 ? xr[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    {
        float ss = 0.f;
#pragma unroll
        for (int j = 0; j < PF_NORM_V; ++j) ss += (v[j].x * v[j].x + v[j].y * v[j].y) + (v[j].z * v[j].z + v[j].w * v[j].w);
        ss = warp_sum(ss);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
        __syncthreads();
        if (threadIdx.x < 32) {
            float t = threadIdx.x < (PF_EW_THREADS >> 5) ? red[threadIdx.x] : 0.f;
            t = warp_sum(t);
            if (threadIdx.x == 0) rs[r] = rsqrtf(t / (float)K + eps);
        }
    }
    const float4* g4 = reinterpret_cast<const float4*>(gain);
#pragma unroll
    for (int j = 0; j < PF_NORM_V; ++j) {
        const int i = threadIdx.x + j * PF_EW_THREADS;
        if (i < n4) {
            float4 w = v[j];
            const float4 gg = g4[i];
            w.x *= gg.x; w.y *= gg.y; w.z *= gg.z; w.w *= gg.w;
            split_store4(hi, lo, (size_t)r * K + (size_t)i * 4, w);
        }
    }
}

// planes of x[r] itself; grid = (rows, ceil(K / (4 * PF_EW_THREADS))), K and ldx multiples of 4
__global__ void __launch_bounds__(PF_EW_THREADS) pf_split_kernel(const float* x, int ldx, int K, __nv_bfloat16* hi, __nv_bfloat16* lo) {
    const int r = blockIdx.x;
    const int i = blockIdx.y * PF_EW_THREADS + threadIdx.x;
    if (i < (K >> 2)) split_store4(hi, lo, (size_t)r * K + (size_t)i * 4, *reinterpret_cast<const float4*>(x + (size_t)r * ldx + (size_t)i * 4));
}

}  // namespace kg
