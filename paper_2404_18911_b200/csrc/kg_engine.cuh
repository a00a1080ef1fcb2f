// The persistent decode kernel: one cooperative grid (one CTA per SM) runs whole phases of the
// method - prefill chunks, the draft loop with its on-device exit test, the verify pass, the
// prefix accept / rollback, or many rounds back to back - with exchanges or grid barriers between
// dependent operators and no host involvement.
//
// The roles in every CTA, joined by a queue of operators in shared memory:
//   the sequencer (one thread) walks through the method - layers, draft steps, accept decisions - and writes the arguments of one
//     operator after the other into the queue.  It runs ahead of the others until the next decision that depends on a result (a
//     drafted token, its confidence, the accepted prefix), which it receives through shared memory.  Every CTA's sequencer
//     holds the same copy of the sequence state and comes to the same decisions.
//   the copy warp streams the weights and the K / V tiles of the operators in the queue, and a prefetch warp asks for weights further
//     ahead than its ring reaches;
//   the eight consumer warps do the arithmetic and take part in the grid barriers.
// The consumers' loop holds every operator once, inlined.  Before, every thread walked through the method itself and called the
// operators as functions from a dozen places: they were compiled for the 168 registers of the launch (the warpgroups' own budgets
// reach inlined code only), what the callers kept across them was spilled - beside 227 KB of shared memory there is hardly any L1,
// so that a spilled register is an L2 access -, and each layer began with one thread writing its arguments while 255 waited.
// 7B, KV 512, with the attention fed by the ring: verify pass of one row 2.74 -> 2.58 ms, of seven rows 3.42 -> 3.19, draft step
// 0.328 -> 0.300, greedy step 2.87 -> 2.70.
#pragma once

#include "kg_device.cuh"

namespace kg {

enum { PROG_PREFILL = 0, PROG_DRAFT = 1, PROG_VERIFY = 2, PROG_DECODE = 3, PROG_AR = 4 };

struct Program {
    int kind;
    int n;              // PREFILL: prompt length; DECODE / AR: total tokens wanted (x_0 included)
    float eta; int gamma; int stop_mode;
    int force_simple;   // 1: route bf16 linears through the plain path (cross-check)
    unsigned long long wait_clk;   // clocks after which a device-side wait gives up (KG_E_TIMEOUT)
    int skip_arrival;   // test hook: 1 + index of a CTA that leaves out its first grid-barrier arrival, so that a wait expires
};

// Rows handed from one operator to the next: fp32 rows (residual input, plain path), their packed copy
// scaled by the reader's norm gain, and the per-CTA sums of squares the reader's RMSNorm needs.
struct ActIn { const float* x; const unsigned char* pk; const float* ssq; };
struct ActOut { float* x; PkOut pk[2]; float* ssq; };

// linear operators on the streamed tensor-core path, for this launch
__device__ __forceinline__ bool launch_streamed(const Dev& D, const Program& pg) { return D.dm.stream != 0 && pg.force_simple == 0; }

// ---- the sequencer (one thread per CTA) ----------------------------------------------------------------------------
template <typename WT>
struct Sequencer {
    const Dev& D;
    Ctx& c;
    const Program& pg;
    const bool streamed;
    int qi = 0; unsigned qph = 0;      // queue cursor
    AttPlan plan;                      // of the last attention position
    int xp = 0;                        // exchange instance the next layer uses
    int xused = 0;                     // rows of the other instance, the one of the layer before, that hold data

    __device__ Sequencer(const Dev& d, Ctx& cx, const Program& p) : D(d), c(cx), pg(p), streamed(launch_streamed(d, p)) { plan.pos = -1; }

    // ---- the queue
    __device__ __forceinline__ Op* begin(int kind) {
        if (!mbar_wait(c, &c.ctl->qempty[qi], qph ^ 1u, 33)) return nullptr;
        Op* o = &c.ctl->queue[qi];
        o->kind = kind; o->sync = 0;
        return o;
    }
    __device__ __forceinline__ void commit() {
        mbar_arrive(&c.ctl->qfull[qi]);
        if (++qi == QUEUE) { qi = 0; qph ^= 1u; }
    }
    // waits until the consumers have come to the operator that answers
    __device__ __forceinline__ bool wait_mail() {
        const unsigned mp = c.mail_phase;
        c.mail_phase = mp ^ 1u;
        return mbar_wait(c, &c.ctl->mail, mp, 42);
    }
    // operator on the weights [N, K] with M rows
    __device__ __forceinline__ LinArgs* linear(const void* W, const void* W2, int N, int K, int M) {
        Op* o = begin(OPK_LIN);
        if (!o) return nullptr;
        LinArgs& a = o->lin;
        a.W = W; a.W2 = W2; a.N = N; a.K = K; a.M = M; a.eps = D.dm.eps;
        if (streamed) lin_phases(a);
        a.gain = nullptr; a.ssq_in = nullptr; a.poll = 0; a.resid = nullptr; a.out = nullptr;
        a.pk[0] = PkOut{nullptr, nullptr}; a.pk[1] = PkOut{nullptr, nullptr}; a.ssq_out = nullptr;
        return &a;
    }
    __device__ __forceinline__ void commit_sync(int where) { c.ctl->queue[qi].sync = where; commit(); }

    // ---- buffers
    __device__ size_t cache_layer_stride() const { return (size_t)D.dm.n_pages * D.dm.H * D.dm.page_size * D.dm.hd; }
    __device__ __forceinline__ size_t ldpk() const { return (size_t)D.dm.d * 4; }
    __device__ __forceinline__ ActIn act_h() const { return ActIn{D.h, D.hA_pk, D.ssq_hA}; }
    // the residual stream as an output, packed for a reader whose norm gain is `gain`
    __device__ __forceinline__ ActOut out_h(const float* gain) const {
        ActOut o; o.x = D.h; o.pk[0] = PkOut{gain, D.hA_pk}; o.pk[1] = PkOut{nullptr, nullptr}; o.ssq = D.ssq_hA; return o;
    }
    // norm gain of whatever reads the output of layer i: the next layer, or the LM head after the last one
    __device__ __forceinline__ const float* next_gain(int i) const { return i + 1 < D.dm.L ? D.layers[i + 1].g1 : D.g_final; }
    // the early-feature slot `slot` as an input of the adapter / of the first deep layer
    __device__ __forceinline__ ActIn feat_for_adapter(int slot) const {
        return ActIn{D.feat + (size_t)slot * D.dm.d, D.featA_pk + (size_t)slot * ldpk(), D.ssq_feat + (size_t)slot * c.nctas};
    }
    __device__ __forceinline__ ActIn feat_for_deep(int slot) const {
        return ActIn{D.feat + (size_t)slot * D.dm.d, D.featD_pk + (size_t)slot * ldpk(), D.ssq_feat + (size_t)slot * c.nctas};
    }
    // exchange rows of the layer being pushed
    __device__ __forceinline__ float* xrow(int off) const { return reinterpret_cast<float*>(D.xch[xp] + off); }
    __device__ __forceinline__ float* x_qkv() const { return xrow(0); }
    __device__ __forceinline__ float* x_attn() const { return xrow(3 * D.dm.d); }
    __device__ __forceinline__ float* x_h() const { return xrow(4 * D.dm.d); }
    __device__ __forceinline__ float* x_act() const { return xrow(5 * D.dm.d); }
    __device__ __forceinline__ float* x_ssq() const { return xrow(5 * D.dm.d + D.dm.F); }
    __device__ static __forceinline__ unsigned char* bytes(float* p) { return reinterpret_cast<unsigned char*>(p); }

    // ---- operators
    // h[i] = E[token_i]; packed for layer 0
    __device__ bool embed_rows(const int* toks, int tok, int M, int where) {
        Op* o = begin(OPK_EMBED);
        if (!o) return false;
        o->emb.toks = toks; o->emb.tok = tok; o->emb.M = M;
        commit_sync(where);
        return true;
    }
    // q, k, v and the attention of layer / adapter `li` on M rows at pos0
    __device__ bool attention_block(const LayerW& lw, int li, int M, int pos0, const ActIn& in) {
        const Dims& dm = D.dm;
        LinArgs* q = linear(lw.wqkv, nullptr, 3 * dm.d, dm.d, M);
        if (!q) return false;
        q->x = in.x; q->ldx = dm.d; q->gain = lw.g1; q->xpk = in.pk; q->ldpk = (int)ldpk(); q->ssq_in = in.ssq; q->ld_ssq = c.nctas;
        q->epi = EPI_STORE; q->out = x_qkv(); q->ldo = D.xch_ld;
        commit();
        if (D.dm.ring && plan.pos != pos0) plan = ra_plan(pos0, dm.H, c.nctas);
        Op* o = begin(OPK_ATT);
        if (!o) return false;
        AttArgs& at = o->att;
        at.plan = plan;
        at.qkv = x_qkv(); at.ldq = D.xch_ld; at.poll = 1; at.M = M; at.pos0 = pos0;
        at.kc = reinterpret_cast<WT*>(D.kcache) + (size_t)li * cache_layer_stride();
        at.vc = reinterpret_cast<WT*>(D.vcache) + (size_t)li * cache_layer_stride();
        at.row0 = li * dm.n_pages * dm.H * dm.page_size;
        at.out = streamed ? nullptr : x_attn(); at.ldo = D.xch_ld;
        at.opk = streamed ? bytes(x_attn()) : nullptr; at.ldopk = D.xch_ld * 4;
        // the instance of the layer before is emptied behind the attention (not earlier: nothing else is stored meanwhile)
        o->empty_p = xp ^ 1; o->empty_rows = xused;
        commit();
        return true;
    }
    // output projection of the attention with its residual
    __device__ LinArgs* out_proj(const LayerW& lw, int M, const ActIn& in) {
        LinArgs* o = linear(lw.wo, nullptr, D.dm.d, D.dm.d, M);
        if (!o) return nullptr;
        o->x = x_attn(); o->ldx = D.xch_ld; o->xpk = bytes(x_attn()); o->ldpk = D.xch_ld * 4; o->poll = 1;
        o->epi = EPI_RESID; o->resid = in.x; o->ldr = D.dm.d;
        return o;
    }
    __device__ __forceinline__ void turn_instance(int M) { xused = M; xp ^= 1; }

    // One decoder block on M rows at positions pos0.. (Section 3.1's M^b layers):
    //   h  = x + Wo Attn(RMSNorm(x; g1));   out = h + Wdown(SiLU(Wgate n) * Wup n), n = RMSNorm(h; g2)
    // The rows between its operators are exchange words; one grid barrier ends the layer.
    __device__ bool layer(int li, int M, int pos0, const ActIn& in, const ActOut& out) {
        const Dims& dm = D.dm;
        const LayerW& lw = D.layers[li];
        if (!attention_block(lw, li, M, pos0, in)) return false;
        // the residual stream after attention: fp32 rows of each CTA's own features, packed rows for everybody (plain path:
        // fp32 exchange rows for both)
        float* hres = streamed ? D.h : x_h();
        const int ldh = streamed ? dm.d : D.xch_ld;
        LinArgs* o = out_proj(lw, M, in);
        if (!o) return false;
        o->out = hres; o->ldo = ldh;
        o->pk[0] = PkOut{lw.g2, bytes(x_h())}; o->ldpk_out = D.xch_ld * 4;
        o->ssq_out = x_ssq(); o->ld_sout = D.xch_ld;
        commit();
        LinArgs* gu = linear(lw.wgate, lw.wup, dm.F, dm.d, M);
        if (!gu) return false;
        gu->x = x_h(); gu->ldx = D.xch_ld; gu->gain = lw.g2; gu->xpk = bytes(x_h()); gu->ldpk = D.xch_ld * 4;
        gu->ssq_in = x_ssq(); gu->ld_ssq = D.xch_ld; gu->poll = 1;
        gu->epi = EPI_SWIGLU; gu->out = streamed ? nullptr : x_act(); gu->ldo = D.xch_ld;
        gu->pk[0] = PkOut{nullptr, bytes(x_act())}; gu->ldpk_out = D.xch_ld * 4;
        commit();
        LinArgs* dn = linear(lw.wdown, nullptr, dm.d, dm.F, M);
        if (!dn) return false;
        dn->x = x_act(); dn->ldx = D.xch_ld; dn->xpk = bytes(x_act()); dn->ldpk = D.xch_ld * 4; dn->poll = 1;
        dn->epi = EPI_RESID; dn->resid = hres; dn->ldr = ldh; dn->out = out.x; dn->ldo = dm.d;
        dn->pk[0] = out.pk[0]; dn->pk[1] = out.pk[1]; dn->ldpk_out = (int)ldpk(); dn->ssq_out = out.ssq; dn->ld_sout = c.nctas;
        commit_sync(14);
        turn_instance(M);
        return true;
    }
    // Layers l0 .. l1 - 1 of a pass: `in` feeds the first one, `out` receives the last one's rows.
    __device__ __forceinline__ bool layers(int l0, int l1, int M, int pos0, const ActIn in, const ActOut out) {
        for (int i = l0; i < l1; ++i)
            if (!layer(i, M, pos0, i == l0 ? in : act_h(), i == l1 - 1 ? out : out_h(next_gain(i)))) return false;
        return true;
    }

    // Adapter A (Section 3.1, Table 2): a = f + W^A_o Attn(RMSNorm(f; g_in)) on the rows `in` at pos0..;
    // with want_out == false only the adapter's K/V are appended (prefill).
    __device__ bool adapter(int M, int pos0, const ActIn& in, bool want_out) {
        const LayerW& lw = D.layers[D.dm.L];
        if (!attention_block(lw, D.dm.L, M, pos0, in)) return false;
        if (want_out) {
            LinArgs* o = out_proj(lw, M, in);
            if (!o) return false;
            o->out = D.abuf; o->ldo = D.dm.d;
            o->pk[0] = PkOut{lw.g2, D.abuf_pk}; o->ldpk_out = (int)ldpk(); o->ssq_out = D.ssq_abuf; o->ld_sout = c.nctas;
            commit_sync(22);
        } else {
            if (!begin(OPK_NONE)) return false;
            commit_sync(21);
        }
        turn_instance(M);
        return true;
    }

    // Shared LM head on the rows `in` (norm gain `gain`), then the merged (token, p) per row: the same values in every CTA.
    __device__ __forceinline__ bool head(const ActIn in, int M, const float* gain, float* dbg, int* toks, float* ps) {
        const Dims& dm = D.dm;
        LinArgs* a = linear(D.head, nullptr, dm.V, dm.d, M);
        if (!a) return false;
        a->x = in.x; a->ldx = dm.d; a->gain = gain; a->xpk = in.pk; a->ldpk = (int)ldpk(); a->ssq_in = in.ssq; a->ld_ssq = c.nctas;
        a->epi = EPI_HEAD; a->scale = dm.logit_scale; a->head_part = D.head_part;
        a->logits_dbg = dm.debug ? dbg : nullptr; a->ld_dbg = dm.V;
        commit_sync(30);
        Op* o = begin(OPK_HEAD);
        if (!o) return false;
        o->emb.M = M;
        commit();
        if (!wait_mail()) return false;
        for (int i = 0; i < M; ++i) { toks[i] = c.ctl->head_tok[i]; ps[i] = c.ctl->head_p[i]; }
        return true;
    }

    // ---- sequence state: the same values in every CTA
    int P, len_A, x0, total, rounds;
    int n_d, n_steps;
    int dtok[M_MAX];
    float dconf[M_MAX];

    __device__ void load_state() {
        P = __ldcg(&D.st->P); len_A = __ldcg(&D.st->len_A); x0 = __ldcg(&D.st->x0);
        total = __ldcg(&D.st->total); rounds = __ldcg(&D.st->rounds);
        n_d = __ldcg(&D.st->n_d); n_steps = __ldcg(&D.st->n_steps);
        for (int i = 0; i < M_MAX; ++i) { dtok[i] = __ldcg(&D.st->draft_tok[i]); dconf[i] = __ldcg(&D.st->conf[i]); }
    }
    __device__ bool leader() const { return c.cta == 0; }

    // early feature of token `tok` at position pos -> feat slot (fp32 and packed for both of its readers)
    __device__ bool shallow_pass(int tok, int pos, int slot) {
        const Dims& dm = D.dm;
        if (!embed_rows(nullptr, tok, 1, 1)) return false;
        ActOut o;
        o.x = D.feat + (size_t)slot * dm.d;
        o.pk[0] = PkOut{D.layers[dm.L].g1, D.featA_pk + (size_t)slot * ldpk()};
        o.pk[1] = PkOut{D.layers[dm.l].g1, D.featD_pk + (size_t)slot * ldpk()};
        o.ssq = D.ssq_feat + (size_t)slot * c.nctas;
        return layers(0, dm.l, 1, pos, act_h(), o);
    }

    // Draft phase of one round (Section 3.2; Eq. 4; Figure 2).
    __device__ bool draft_phase() {
        const Dims& dm = D.dm;
        n_d = 0; n_steps = 0;
        int cur = x0;
        bool stop_after_shallow = false;
        while (true) {
            if (!shallow_pass(cur, P + n_d, 1 + n_d)) return false;                 // f[n_d]
            if (n_d == pg.gamma || stop_after_shallow) break;
            const int MA = P + n_d - len_A + 1;                                     // 1, or 2 when the adapter cache lags
            if (!adapter(MA, len_A, feat_for_adapter(1 + n_d - (MA - 1)), true)) return false;
            int tk[1]; float pp[1];
            const ActIn hin{D.abuf + (size_t)(MA - 1) * dm.d, D.abuf_pk + (size_t)(MA - 1) * ldpk(), D.ssq_abuf + (size_t)(MA - 1) * c.nctas};
            if (!head(hin, 1, D.layers[dm.L].g2, D.dbg_draft + (size_t)n_steps * dm.V, tk, pp)) return false;
            len_A += MA;
            dconf[n_steps] = pp[0];
            n_steps++;
            if (pg.stop_mode == 1 && pp[0] <= pg.eta) break;                        // drop the low-confidence token
            dtok[n_d] = tk[0];
            n_d++;
            cur = tk[0];
            if (pg.stop_mode == 0 && pp[0] <= pg.eta) stop_after_shallow = true;    // keep it; its feature is still needed
        }
        if (leader()) {
            State* st = D.st;
            st->n_d = n_d; st->n_steps = n_steps; st->len_A = len_A; st->pending = 1;
            for (int i = 0; i < M_MAX; ++i) { st->draft_tok[i] = dtok[i]; st->conf[i] = dconf[i]; }
            st->draft_steps_total += n_steps; st->drafted_total += n_d;
        }
        return true;
    }

    // Verify pass + prefix accept + rollback (Section 3: discard after the first reject; Figure 2).
    __device__ bool verify_phase() {
        const Dims& dm = D.dm;
        const int M = n_d + 1;
        if (!layers(dm.l, dm.L, M, P, feat_for_deep(1), out_h(D.g_final))) return false;
        int t[M_MAX]; float pp[M_MAX];
        if (!head(act_h(), M, D.g_final, D.dbg_verify, t, pp)) return false;
        int k = 0;
        while (k < n_d && dtok[k] == t[k]) ++k;
        const int newP = P + k + 1;
        if (len_A > newP) len_A = newP;
        if (len_A < newP) {
            // the adapter has not seen f[k] (k == n_d): keep it as the feature of position newP-1 (slot 0)
            Op* o = begin(OPK_KEEP);
            if (!o) return false;
            o->emb.M = 1 + k;
            commit();
        }
        if (leader()) {
            State* st = D.st;
            for (int i = 0; i < k; ++i) { D.out_tokens[total + i] = dtok[i]; st->emitted[i] = dtok[i]; }
            D.out_tokens[total + k] = t[k]; st->emitted[k] = t[k];
            for (int i = 0; i < M; ++i) st->target[i] = t[i];
            D.S[rounds] = k + 1;
            D.round_log[rounds * 4 + 0] = n_d; D.round_log[rounds * 4 + 1] = n_steps;
            D.round_log[rounds * 4 + 2] = k; D.round_log[rounds * 4 + 3] = P;
            st->M = M; st->k_acc = k; st->n_emit = k + 1;
            st->P = newP; st->len_A = len_A; st->x0 = t[k]; st->pending = 0;
            st->total = total + k + 1; st->rounds = rounds + 1; st->accepted_total += k;
        }
        P = newP; x0 = t[k]; total += k + 1; rounds += 1;
        return true;
    }

    __device__ bool prefill() {
        const Dims& dm = D.dm;
        const int n = pg.n;
        int tk[1]; float pp[1];
        tk[0] = 0;
        for (int c0 = 0; c0 < n; c0 += M_MAX) {
            const int M = min(M_MAX, n - c0);
            if (!embed_rows(D.prompt + c0, 0, M, 2)) return false;
            ActOut o = out_h(next_gain(dm.l - 1));
            o.pk[1] = PkOut{D.layers[dm.L].g1, D.featA_pk};    // the adapter reads the same rows
            if (!layers(0, dm.l, M, c0, act_h(), o)) return false;
            if (!adapter(M, c0, ActIn{D.h, D.featA_pk, D.ssq_hA}, false)) return false;
            if (!layers(dm.l, dm.L, M, c0, act_h(), out_h(D.g_final))) return false;
            if (c0 + M == n) {
                const ActIn hin{D.h + (size_t)(M - 1) * dm.d, D.hA_pk + (size_t)(M - 1) * ldpk(), D.ssq_hA + (size_t)(M - 1) * c.nctas};
                if (!head(hin, 1, D.g_final, D.dbg_verify, tk, pp)) return false;
            } else {
                // the next chunk attends to this one's rows: the copy warp must not run ahead of the barrier behind them
                if (!begin(OPK_MAIL)) return false;
                commit();
                if (!wait_mail()) return false;
            }
        }
        if (leader()) {
            State* st = D.st;
            st->P = n; st->len_A = n; st->x0 = tk[0]; st->pending = 0; st->total = 1; st->rounds = 0;
            D.out_tokens[0] = tk[0];
        }
        return true;
    }

    __device__ bool ar_decode() {
        int tk[1]; float pp[1];
        while (total < pg.n) {
            if (!embed_rows(nullptr, x0, 1, 3)) return false;
            if (!layers(0, D.dm.L, 1, P, act_h(), out_h(D.g_final))) return false;
            if (!head(act_h(), 1, D.g_final, D.dbg_verify, tk, pp)) return false;
            if (leader()) {
                D.out_tokens[total] = tk[0];
                D.st->P = P + 1; D.st->x0 = tk[0]; D.st->total = total + 1; D.st->len_A = -1;
            }
            P += 1; x0 = tk[0]; total += 1;
        }
        return true;
    }

    __device__ bool run_program() {
        if (pg.kind == PROG_PREFILL) return prefill();
        if (pg.kind == PROG_AR) return ar_decode();
        const bool draft = pg.kind != PROG_VERIFY, verify = pg.kind != PROG_DRAFT, once = pg.kind != PROG_DECODE;
        while (once || total < pg.n) {
            if (draft && !draft_phase()) return false;
            if (verify && !verify_phase()) return false;
            if (once) break;
        }
        return true;
    }

    __device__ void run() {
        load_state();
        if (!run_program()) return;              // a wait gave up: the abort flag ends the other roles
        // a launch finds both exchange instances empty and leaves them so
        Op* o = begin(OPK_EXIT);
        if (!o) return;
        o->empty_p = xp ^ 1; o->empty_rows = xused;
        commit();
    }
};

// ---- the copy warp ---------------------------------------------------------------------------------------------------
__device__ __forceinline__ void copy_loop(const Dev& D, Ctx& c, bool streamed) {
    Ctrl* ctl = c.ctl;
    const int lane = threadIdx.x & 31;
    int q = 0; unsigned qph = 0;
    bool ok = true, done = false;
    while (ok && !done) {
        int w = 1;
        if (lane == 0) w = mbar_wait(c, &ctl->qfull[q], qph, 34) ? 1 : 0;
        ok = __shfl_sync(0xffffffffu, w, 0) != 0;
        if (!ok) break;
        const Op& op = ctl->queue[q];
        const int kind = op.kind;
        if (streamed && kind == OPK_LIN) ok = lin_produce<true>(op.lin, c);
        else if (streamed && kind == OPK_ATT && D.dm.ring) ok = attention_producer(D, op.att.plan, op.att.row0, c);
        done = kind == OPK_EXIT;
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl->qempty[q]);
        if (++q == QUEUE) { q = 0; qph ^= 1u; }
    }
    if (!ok) ring_drain(c);
}

// ---- the prefetch warp (of launches that stream weights: the others' queue is not held up by a reader that has nothing to do)
__device__ __forceinline__ void prefetch_loop(const Dev& D, Ctx& c) {
    Ctrl* ctl = c.ctl;
    const int lane = threadIdx.x & 31;
    int q = 0; unsigned qph = 0;
    bool ok = true, done = false;
    while (!done) {
        int w = 1;                       // (a wait here that gives up ends the launch as any other does)
        if (lane == 0) w = mbar_wait(c, &ctl->qfull[q], qph, 35) ? 1 : 0;
        if (!__shfl_sync(0xffffffffu, w, 0)) return;
        const Op& op = ctl->queue[q];
        const int kind = op.kind;
        if (ok && kind == OPK_LIN) ok = lin_prefetch(op.lin, c);
        else if (kind == OPK_ATT && D.dm.ring) {
            const unsigned n = D.dm.hd == 128 ? att_stages<128>(D, op.att.plan, c) : att_stages<64>(D, op.att.plan, c);
            __syncwarp();
            if (lane == 0) c.issued += n;
        }
        done = kind == OPK_EXIT;
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl->qempty[q]);
        if (++q == QUEUE) { q = 0; qph ^= 1u; }
    }
}

// ---- the consumer warps ----------------------------------------------------------------------------------------------
// true when the predicate holds in every consumer thread (a barrier among them)
__device__ __forceinline__ bool cta_all(bool p) {
    unsigned r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(r) : "r"((unsigned)p), "n"(NTHREADS) : "memory");
    return r != 0;
}

template <typename WT>
__device__ __forceinline__ void consume_embed(const Dev& D, Ctx& c, const EmbedArgs& e, bool streamed) {
    const int d = D.dm.d, M = e.M;
    const int* toks = e.toks; const int tok1 = e.tok;
    const WT* E = reinterpret_cast<const WT*>(D.embed);
    // an id outside [0, V) never indexes the embedding table (ids that arrive in device memory are checked by a
    // kernel of their own, which records the error; here the access is merely kept in bounds)
    auto row = [&](int m) { const int tok = toks ? __ldcg(toks + m) : tok1; return E + (size_t)((unsigned)tok < (unsigned)D.dm.V ? tok : 0) * d; };
    if (!streamed) {
        for (int idx = c.cta * NTHREADS + threadIdx.x; idx < M * d; idx += c.nctas * NTHREADS) D.h[idx] = wt_to_float<WT>(row(idx / d)[idx % d]);
        return;
    }
    LinArgs a{};
    a.N = d; a.M = M; a.out = D.h; a.ldo = d;
    a.pk[0] = PkOut{D.layers[0].g1, D.hA_pk}; a.ldpk_out = d * 4; a.ssq_out = D.ssq_hA; a.ld_sout = c.nctas;
    emit_plain_rows(a, c, [&](int m, int e_) { return wt_to_float<WT>(row(m)[e_]); });
}

// The attention without the ring as a call: what a model that has the ring takes when it is told to cross-check (force_simple).
template <typename WT, int HD>
__device__ __noinline__ void attention_far(const Dev& D, const AttArgs& a, Ctx& c) {
    attention_impl<WT, HD / 32, false>(D, a, ka_plan(a.pos0, a.M, D.dm.H, c.nctas), c);
}

template <typename WT, int HD, bool RING>
__device__ __forceinline__ void consume_loop(const Dev& D, Ctx& c, bool streamed) {
    Ctrl* ctl = c.ctl;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int q = 0; unsigned qph = 0;
    while (true) {
        if (!cta_all(mbar_wait(c, &ctl->qfull[q], qph, 31))) return;
        const Op& op = ctl->queue[q];
        const int kind = op.kind;
        if (kind == OPK_LIN) {
            const LinArgs& a = op.lin;
            if (!streamed) lin_simple<WT>(a, c);
            else if constexpr (sizeof(WT) == 2) {
                if (a.M <= 4) lin_consume<4, true>(a, c); else if (a.M <= 8) lin_consume<8, true>(a, c); else if (a.M <= 12) lin_consume<12, true>(a, c); else lin_consume<16, true>(a, c);
            }
        } else if (kind == OPK_ATT) {
            const AttArgs& a = op.att;
            if constexpr (RING) {
                if (!streamed) attention_far<WT, HD>(D, a, c); else if (a.M <= 8) attention_ring<HD, 1, true>(D, a, c); else attention_ring<HD, 2, true>(D, a, c);
            } else attention_impl<WT, HD / 32, false>(D, a, ka_plan(a.pos0, a.M, D.dm.H, c.nctas), c);
        } else if (kind == OPK_EMBED) {
            consume_embed<WT>(D, c, op.emb, streamed);
        } else if (kind == OPK_HEAD) {
            const int M = op.emb.M;
            for (int m = warp; m < M; m += NWARPS) {                       // one warp per row
                int tk; float p;
                head_final_warp(D.head_part, c.nctas, m, tk, p);
                if (lane == 0) { ctl->head_tok[m] = tk; ctl->head_p[m] = p; }
            }
            cta_sync();
            if (tid == 0) mbar_arrive(&ctl->mail);
        } else if (kind == OPK_MAIL) {
            if (tid == 0) mbar_arrive(&ctl->mail);                         // (thread 0 polled the grid barrier that came before)
        } else if (kind == OPK_KEEP) {
            // early feature of slot emb.M -> slot 0
            const int s = op.emb.M, d = D.dm.d;
            const int gtid = c.cta * NTHREADS + tid, gn = c.nctas * NTHREADS;
            const float* src = D.feat + (size_t)s * d;
            for (int e = gtid; e < d; e += gn) D.feat[e] = __ldcg(src + e);
            const unsigned* psrc = reinterpret_cast<const unsigned*>(D.featA_pk + (size_t)s * d * 4);
            unsigned* pdst = reinterpret_cast<unsigned*>(D.featA_pk);
            for (int e = gtid; e < d; e += gn) pdst[e] = __ldcg(psrc + e);
            for (int e = gtid; e < c.nctas; e += gn) D.ssq_feat[e] = __ldcg(D.ssq_feat + (size_t)s * c.nctas + e);
        }
        if (kind == OPK_ATT || kind == OPK_EXIT) {
            const int n4 = op.empty_rows * (D.xch_ld >> 2);
            uint4* x = reinterpret_cast<uint4*>(D.xch[op.empty_p]);
            for (int i = c.cta * NTHREADS + tid; i < n4; i += c.nctas * NTHREADS) x[i] = make_uint4(XCH_EMPTY, XCH_EMPTY, XCH_EMPTY, XCH_EMPTY);
        }
        const int where = op.sync;
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl->qempty[q]);
        if (where && !grid_sync(c, where)) return;
        if (kind == OPK_EXIT) { if (tid == 0) grid_leave(c); return; }
        if (++q == QUEUE) { q = 0; qph ^= 1u; }
    }
}

// HD: the head size.  RING: attention from the ring; else the other attention, inlined (as a call it has the 168 registers of the launch
// and not the consumers' 216: bf16, four layers of 512 with an F that only the plain linear operators take, 32 tokens 4.13 -> 3.15 ms; fp32,
// four layers of 1024, 7.3 -> 6.7).  Compiled apart: with two head sizes in one kernel 0.9 KB of registers were spilled around the operators.
// (In the ring kernel the plain operators stay as calls.  Without them more of the row variants' registers are spilled, 460 against 240 bytes
// of loads: 7B, verify passes of 11 rows, three rounds 25.9 against 25.0 ms.)
template <typename WT, int HD, bool RING>
__global__ void __launch_bounds__(DECODE_THREADS, 1) kg_persistent_kernel(const __grid_constant__ Dev D, const __grid_constant__ Program pg) {
    extern __shared__ __align__(128) char smem[];
    Ctx& c = ctx_init(smem, D.st, D.bar, true, pg.wait_clk, pg.skip_arrival, sizeof(WT) == 2 && launch_streamed(D, pg));
    if (threadIdx.x >= NTHREADS) {
        // the third warpgroup: keeps what the copy loop and the sequencer need and returns the rest of its registers
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(PRODUCER_REGS));
        const int w = (threadIdx.x - NTHREADS) >> 5;
        if (w == 0) copy_loop(D, c, launch_streamed(D, pg));
        else if (w == 1 && (threadIdx.x & 31) == 0) {
            Sequencer<WT> seq(D, c, pg);
            seq.run();
        } else if (sizeof(WT) == 2 && w == 2 && launch_streamed(D, pg)) prefetch_loop(D, c);
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(CONSUMER_REGS));
        consume_loop<WT, HD, RING>(D, c, launch_streamed(D, pg));
    }
}

}  // namespace kg
