// Algorithm 3 (WIND beam search) for one utterance.
//
// The hypothesis map, recombination and pruning are sequential bookkeeping over a handful of hypotheses and run on
// the host; everything that touches the model runs in kernels on the caller's stream: the encoder projection once,
// and per iteration (one frame t taken from the map) the decoder update of the hypotheses that survived pruning
// (batched over the beam), the windowed joint for every hypothesis, Eq. (1) and its K best entries per hypothesis.
// Only K x K (label, offset, log-probability) triples cross to the host per iteration.  An iteration goes to one resident kernel
// (wind_beam_step.cu) that takes it as a command, or, for shapes that kernel does not take, a sequence of kernels.
//
// Decoder states live in a pool of slots in the workspace.  A hypothesis created by a label is evaluated lazily: it
// carries (parent slot, label) until it survives the pruning of its frame, so at most K decoder updates are made per
// iteration although K x K hypotheses are created.  Slots are reference-counted (a hypothesis created by the blank
// entry shares its parent's slot).
//
// An iteration waits for the one before it, but what it evaluates (a token history at a frame) rarely depends on that one: most
// hypotheses of the next frames' lists are there long before their turn.  So a command of the resident kernel is filled up with the
// histories that the following iterations will most likely ask for (struct Forecast), and an iteration whose hypotheses have all been
// evaluated needs no command.  What is evaluated is the same, in the same precision and summation order; only the guess when is not,
// and a wrong one costs a row.  Beam 4, W = 8: 1.03 evaluations per one needed, 0.33 commands per iteration.
#if defined(__x86_64__)
#include <immintrin.h>
#endif

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "wind_internal.cuh"

namespace wind {

namespace {

// pool slot -> batch row (both parities of h are not needed: the update reads parity 0, writes parity 1)
__global__ void beam_gather_kernel(const float* __restrict__ h_pool, const float* __restrict__ c_pool, const int32_t* __restrict__ src,
                                   const int32_t* __restrict__ tok, float* __restrict__ h_in, float* __restrict__ c_state,
                                   int32_t* __restrict__ emit_tok, int B, int L, int P) {
    const int b = blockIdx.x;
    const int s = src[b];
    if (threadIdx.x == 0) emit_tok[b] = s >= 0 ? tok[b] : -1;
    if (s < 0) return;
    for (int e = threadIdx.x; e < L * P; e += blockDim.x) {
        const int l = e / P, k = e - l * P;
        h_in[((size_t)l * B + b) * P + k] = h_pool[(size_t)s * L * P + e];
        c_state[((size_t)l * B + b) * P + k] = c_pool[(size_t)s * L * P + e];
    }
}

// batch row -> pool slot: new state and its pred_proj
__global__ void beam_scatter_kernel(const float* __restrict__ h_out, const float* __restrict__ c_state, const float* __restrict__ pred_proj,
                                    const int32_t* __restrict__ dst, float* __restrict__ h_pool, float* __restrict__ c_pool,
                                    float* __restrict__ g_pool, int B, int L, int P, int H) {
    const int b = blockIdx.x;
    const int s = dst[b];
    if (s < 0) return;
    for (int e = threadIdx.x; e < L * P; e += blockDim.x) {
        const int l = e / P, k = e - l * P;
        h_pool[(size_t)s * L * P + e] = h_out[((size_t)l * B + b) * P + k];
        c_pool[(size_t)s * L * P + e] = c_state[((size_t)l * B + b) * P + k];
    }
    for (int k = threadIdx.x; k < H; k += blockDim.x) g_pool[(size_t)s * H + k] = pred_proj[(size_t)b * H + k];
}

// pred_proj of the hypotheses to expand, and their frame (rows without a hypothesis sit at the utterance's end)
__global__ void beam_gather_g_kernel(const float* __restrict__ g_pool, const int32_t* __restrict__ slot, float* __restrict__ pred_proj,
                                     int32_t* __restrict__ t_cur, int t, int T, int H) {
    const int b = blockIdx.x;
    const int s = slot[b];
    if (threadIdx.x == 0) t_cur[b] = s >= 0 ? t : T;
    if (s < 0) return;
    for (int k = threadIdx.x; k < H; k += blockDim.x) pred_proj[(size_t)b * H + k] = g_pool[(size_t)s * H + k];
}

// log-probability of one label per row, from a [B][NV] table of log-softmax values (rows without a label: untouched)
__global__ void beam_pick_kernel(const float* __restrict__ logp, const int32_t* __restrict__ label, float* __restrict__ out, int B, int NV) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B && label[b] >= 0) out[b] = logp[(size_t)b * NV + label[b]];
}

__global__ void beam_fill_kernel(int32_t* a, int n, int v) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = v;
}

// Token histories are shared: a hypothesis points at the node of its last token, a node at the node before it.
struct Node {
    int32_t parent, tok, frm, len;
    uint64_t hash;          // of the token sequence up to here
};

struct Hyp {
    int32_t node = -1;      // -1: no tokens
    double score = 0.0;
    int count = 0;
    int slot = -1;          // decoder state after tok (-1: not evaluated yet)
    int parent = -1;        // slot of the state before the last token, while slot == -1
};

// Page-locked mailboxes are kept for later searches, at most eight of them.
std::mutex g_mail_mutex;
std::vector<BeamMail*> g_mail;
constexpr size_t kMailKept = 8;

// between two looks at the mailbox
inline void cpu_relax() {
#if defined(__x86_64__)
    _mm_pause();
#elif defined(__aarch64__)
    asm volatile("yield" ::: "memory");
#endif
}

// The resident kernel of one search, as the host sees it.  It holds every SM, so little of another stream fits beside it: after
// kTurn it ends with the command in hand, what waits on other streams goes first, and the next command launches it again (30 us,
// mostly its weights: 0.3 % of the search; 0.6 % with 5 ms).
constexpr std::chrono::milliseconds kTurn(10);
struct BeamDevice {
    const Call& c;
    BeamShape shape;
    float *h_pool, *c_pool, *g_pool, *logits;
    unsigned long long* relay;
    bool single;                 // other kernels run on the stream between the iterations: one launch per command
    BeamMail* mail = nullptr;
    uint32_t seq = 0, bar_base = 0;
    bool running = false;
    bool on_chip = false;        // it has given a result since its launch (which may have waited for other streams)
    std::chrono::steady_clock::time_point since{};      // the first of them

    cudaError_t open() {
        {
            std::lock_guard<std::mutex> lock(g_mail_mutex);
            if (!g_mail.empty()) { mail = g_mail.back(); g_mail.pop_back(); }
        }
        if (!mail) {
            void* q = nullptr;
            const cudaError_t e = cudaHostAlloc(&q, sizeof(BeamMail), cudaHostAllocPortable);
            if (e != cudaSuccess) return e;
            mail = static_cast<BeamMail*>(q);
        }
        std::memset(mail, 0, sizeof(BeamMail));
        return cudaMemsetAsync(relay, 0, sizeof(unsigned long long) * kBeamWords, c.stream);
    }
    int words() const { return 4 + 5 * shape.rows; }
    void post(const int32_t* words_, bool last) {
        ++seq;
        volatile unsigned long long* out = mail->cmd;
        for (int i = 0; i < words(); ++i) {
            const uint32_t flag = last && i == 1 ? kBeamLast : 0u;
            out[i] = (unsigned long long)seq << 32 | ((uint32_t)words_[i] | flag);
        }
    }
    // one command, until its result (nh * K entries) is there
    wind_status_t run(const int32_t* words, cudaError_t* err) {
        const int n_out = 2 * words[1] * c.B;
        bool last = single || (running && std::chrono::steady_clock::now() - since > kTurn);
        post(words, last);
        for (int launches = 0;;) {
            if (!running) {
                // (a kernel that ends for want of commands took every CTA with it, between two commands)
                if (++launches > 8) return WIND_ERR_TIMEOUT;
                if ((*err = beam_step(c, shape, mail, relay, seq, bar_base, h_pool, c_pool, g_pool, logits)) != cudaSuccess) return WIND_ERR_CUDA;
                running = true;
                on_chip = false;
            }
            bool there = false;
            for (uint32_t spins = 1; !there; ++spins) {
                there = true;
                for (int i = n_out - 1; i >= 0 && there; --i)
                    there = (uint32_t)(static_cast<volatile unsigned long long*>(mail->top)[i] >> 32) == seq;
                if (there) break;
                cpu_relax();
                if ((spins & 4095u) == 0u && (*err = cudaStreamQuery(c.stream)) != cudaErrorNotReady) {
                    if (*err != cudaSuccess) return WIND_ERR_CUDA;
                    running = false;
                    if (*static_cast<volatile uint32_t*>(&mail->failed)) return WIND_ERR_TIMEOUT;
                    break;
                }
            }
            if (!there) {                // it ended before it saw the command, or with the result just written
                std::atomic_thread_fence(std::memory_order_acquire);
                there = true;
                for (int i = 0; i < n_out && there; ++i) there = (uint32_t)(mail->top[i] >> 32) == seq;
                if (!there) { last = single; post(words, last); continue; }
                ++seq;               // it may have left word that no command of the next number came: that number is not used
            }
            if (!on_chip) { on_chip = true; since = std::chrono::steady_clock::now(); }
            if (last) running = false;
            bar_base += beam_step_arrivals(c, words[0]);
            return WIND_OK;
        }
    }
    // Neither the mailbox nor the caller's workspace is given back before the kernel's end.
    ~BeamDevice() {
        if (!mail) return;
        std::vector<int32_t> end((size_t)words(), -1);
        post(end.data(), false);
        cudaStreamSynchronize(c.stream);
        std::lock_guard<std::mutex> lock(g_mail_mutex);
        if (g_mail.size() < kMailKept) g_mail.push_back(mail);
        else cudaFreeHost(mail);
    }
};

// What is known and what will be asked for: per frame the evaluations made (a token history's K best entries), and a forecast of the
// lists to come.  The list of a frame is worked off in rounds (a label without a jump leads to the next round of the same frame), so
// a forecast is the K best hypotheses of each (frame, round) so far, from every evaluation made, wanted or not.
// What followed from a hypothesis that fell out goes with it: commands filled up with such leftovers brought 2 rows per one needed.
struct Eval {
    int32_t node;           // the token history
    int slot;               // its decoder state (one reference)
    int32_t label[kMaxBeam], jump[kMaxBeam];
    float logp[kMaxBeam];
};
struct Forecast {
    uint64_t hash;
    int32_t len, node;
    int slot, parent;       // as in Hyp, one reference, none once `asked`
    int count, from;        // from: frame of the hypothesis that most of its probability comes from, and that one's history
    uint64_t from_hash;
    bool asked;
    double score, most;
};
struct Round { std::vector<Forecast> best; };
struct Frame {
    int rounds = 0, open = 0;                // rounds in use; forecasts not asked for yet
    std::vector<Round> round;                // (kept from frame to frame)
    std::vector<uint64_t> hash;              // of evals
    std::vector<Eval> evals;
};

double log_add(double a, double b) {
    if (a == -INFINITY) return b;
    if (b == -INFINITY) return a;
    return a > b ? a + log1p(exp(b - a)) : b + log1p(exp(a - b));
}

}  // namespace

BeamLayout make_beam_layout(const wind_model_t& m, int T, int W, int K, int S, size_t base) {
    (void)T;
    BeamLayout L{};
    size_t off = base;
    auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes); return o; };
    L.ints = take(sizeof(int32_t) * 8 * (size_t)K);
    L.top_label = take(sizeof(int32_t) * 3 * (size_t)K * K);   // labels, offsets, log-probabilities: one block, one copy
    L.top_jump = L.top_label + sizeof(int32_t) * (size_t)K * K;
    L.top_logp = L.top_jump + sizeof(int32_t) * (size_t)K * K;
    L.relay = take(sizeof(uint64_t) * kBeamWords);
    // The pools come last: a search has them in one of two sizes, from the same place on.
    const size_t pools = off;
    auto pool = [&](BeamPools& p, int slots, int rows) {
        off = pools;
        p.slots = slots;
        p.rows = rows;
        p.h_pool = take(sizeof(float) * (size_t)slots * m.L * m.P);
        p.c_pool = take(sizeof(float) * (size_t)slots * m.L * m.P);
        p.g_pool = take(sizeof(float) * (size_t)slots * m.H);
        p.logits = take(sizeof(float) * (size_t)rows * W * (m.V + 1));
        return off;
    };
    const int s_eff = S < 32 ? S : 32;
    L.need = pool(L.own, K * (W + 2) * (s_eff + 2) + 2 * K + 2, K);
    // A workspace of `need` bytes is enough: a command then has only the hypotheses of its iteration.  (Asked for is a piece more at the
    // least, so that what is left of an unaligned block behind its first aligned address is enough too.)
    L.total = L.need + kAlign;
    const BeamShape most = beam_step_most(m, W, K);
    if (most.look > 0) L.total = pool(L.ahead, L.own.slots + 32 * most.rows, most.rows);
    return L;
}

// cb: a call bundle with B = K rows (the beam), T, W, S of the utterance, enc = the utterance's frames [T, D];
// its enc_len / out_len pointers are set here.  Outputs are HOST arrays.
wind_status_t beam_search_run(Call& cb, const BeamLayout& bl, bool ahead, int K, int prefix_search, int max_hyps, int max_out, int32_t* out_tokens,
                              int32_t* out_frames, int32_t* out_len, double* out_score, int32_t* n_hyps, int64_t* n_steps,
                              cudaError_t* cuda_err) {
    const wind_model_t& m = cb.m;
    const int T = cb.T, W = cb.W, S = cb.S, NV = m.V + 1, LP = m.L * m.P;
    cudaStream_t st = cb.stream;
    uint8_t* ws = cb.ws;
    const bool resident = beam_step_supported(cb);
    BeamShape shape = resident ? beam_step_shape(cb, ahead && !prefix_search) : BeamShape{K, 0};
    if (shape.look > 0 && shape.rows > bl.ahead.rows) shape = beam_step_shape(cb, false);
    const int R = shape.rows;
    const BeamPools& pools = shape.look > 0 ? bl.ahead : bl.own;
    float* h_pool = reinterpret_cast<float*>(ws + pools.h_pool);
    float* c_pool = reinterpret_cast<float*>(ws + pools.c_pool);
    float* g_pool = reinterpret_cast<float*>(ws + pools.g_pool);
    int32_t* ints = reinterpret_cast<int32_t*>(ws + bl.ints);   // [0] src slots, [1] tokens, [2] dst slots, [3] expand slots, [4] lengths, [5] scratch, [6] frames
    int32_t *d_src = ints, *d_tok = ints + K, *d_dst = ints + 2 * K, *d_exp = ints + 3 * K, *d_len = ints + 4 * K,
            *d_scratch = ints + 5 * K, *d_t = ints + 6 * K;
    float* logits = reinterpret_cast<float*>(ws + pools.logits);
    int32_t* d_top_label = reinterpret_cast<int32_t*>(ws + bl.top_label);
    int32_t* d_top_jump = reinterpret_cast<int32_t*>(ws + bl.top_jump);
    float* d_top_logp = reinterpret_cast<float*>(ws + bl.top_logp);
#define BEAM_CUDA(expr) do { cudaError_t e__ = (expr); if (e__ != cudaSuccess) { *cuda_err = e__; return WIND_ERR_CUDA; } } while (0)

    // ---- setup: lengths, control block, encoder projection of the one utterance, an all-zero state in slot 0 ----
    beam_fill_kernel<<<1, 256, 0, st>>>(d_len, K, T);
    cb.enc_len = d_len;
    cb.out_len = d_scratch;
    BEAM_CUDA(launch_init(cb, WIND_KERNELS_SIMT, 0, 0));
    {
        Call c1 = cb;
        c1.B = 1;
        BEAM_CUDA(simt_enc_proj(c1));
    }
    BEAM_CUDA(cudaMemsetAsync(h_pool, 0, sizeof(float) * LP, st));
    BEAM_CUDA(cudaMemsetAsync(c_pool, 0, sizeof(float) * LP, st));

    std::vector<int> refs(pools.slots, 0), free_slots;
    for (int s = pools.slots - 1; s >= 1; --s) free_slots.push_back(s);
    refs[0] = 1;   // the zero state stays
    auto release = [&](int s) { if (s > 0 && --refs[s] == 0) free_slots.push_back(s); };

    std::vector<std::vector<Hyp>> t2hyps((size_t)T + 1);
    {
        Hyp h0;            // tokens = [], score = 0: its state is "zero state fed the blank id once"
        h0.parent = 0;
        refs[0]++;
        t2hyps[0].push_back(std::move(h0));
    }
    BeamDevice dev{cb, shape, h_pool, c_pool, g_pool, logits, reinterpret_cast<unsigned long long*>(ws + bl.relay), prefix_search != 0};
    if (resident) BEAM_CUDA(dev.open());
    std::vector<int32_t> words((size_t)dev.words());
    std::vector<int32_t> host_ints(4 * (size_t)K), top(3 * (size_t)K * K);
    const int32_t* top_label = top.data();
    const int32_t* top_jump = top.data() + (size_t)K * K;
    const float* top_logp = reinterpret_cast<const float*>(top.data() + 2 * (size_t)K * K);
    int64_t steps = 0;

    std::vector<Node> nodes;
    auto node_len = [&](int32_t n) { return n < 0 ? 0 : nodes[(size_t)n].len; };
    auto node_hash = [&](int32_t n) { return n < 0 ? 0x9E3779B97F4A7C15ull : nodes[(size_t)n].hash; };
    auto same_tokens = [&](int32_t x, int32_t y) {
        if (node_len(x) != node_len(y) || node_hash(x) != node_hash(y)) return false;
        while (x != y) {   // equal lengths: the chains end together, or meet at a shared node
            if (nodes[(size_t)x].tok != nodes[(size_t)y].tok) return false;
            x = nodes[(size_t)x].parent;
            y = nodes[(size_t)y].parent;
        }
        return true;
    };
    int32_t *d_pick = ints + 7 * K;
    // decoder update of up to K (parent slot, token) pairs into fresh slots; the parents' references are released
    auto run_update = [&](int nu) -> cudaError_t {   // host_ints [0..K) src, [K..2K) tokens, [2K..3K) dst are filled
        cudaError_t e = cudaMemcpyAsync(ints, host_ints.data(), sizeof(int32_t) * 3 * K, cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) return e;
        beam_gather_kernel<<<K, 128, 0, st>>>(h_pool, c_pool, d_src, d_tok, cb.h(0), cb.c(), cb.emit_tok(), K, m.L, m.P);
        if ((e = simt_pred_step(cb, 0)) != cudaSuccess) return e;
        beam_scatter_kernel<<<K, 128, 0, st>>>(cb.h(1), cb.c(), cb.pred_proj(), d_dst, h_pool, c_pool, g_pool, K, m.L, m.P, m.H);
        for (int u = 0; u < nu; ++u) release(host_ints[u]);
        return cudaGetLastError();
    };
    auto take_slot = [&]() -> int {
        if (free_slots.empty()) return -1;
        const int s = free_slots.back();
        free_slots.pop_back();
        refs[s] = 1;
        return s;
    };
    // Step (2) of the recombination as the paper states it: for every pair (A, B) of the list with A's tokens a proper
    // prefix of B's, P(A) * prod_i P(b_i | frame t, decoder after A + b_<i) is added to B, then every such A is removed.
    // The per-label probabilities come from the same kernels as the expansion (one-row window at frame t), K pairs at a
    // time, one round per extra token; completions use the probabilities the hypotheses had when the step began.
    struct Pair { int a, b, cur; std::vector<int32_t> extra; double acc; };
    auto prefix_step = [&](std::vector<Hyp>& l, int t) -> wind_status_t {
        const int n = (int)l.size();
        if (n < 2) return WIND_OK;
        std::vector<Pair> pairs;
        for (int a = 0; a < n; ++a)
            for (int b = 0; b < n; ++b) {
                const int la = node_len(l[a].node), lb = node_len(l[b].node);
                if (a == b || la >= lb) continue;
                std::vector<int32_t> extra((size_t)(lb - la));
                int32_t x = l[b].node;
                for (int k = lb - la - 1; k >= 0; --k) { extra[(size_t)k] = nodes[(size_t)x].tok; x = nodes[(size_t)x].parent; }
                if (!same_tokens(l[a].node, x)) continue;
                pairs.push_back(Pair{a, b, -1, std::move(extra), l[a].score});
            }
        if (pairs.empty()) return WIND_OK;
        // the prefixes need their decoder state now
        std::vector<char> is_prefix((size_t)n, 0);
        for (const Pair& p : pairs) is_prefix[(size_t)p.a] = 1;
        for (int a0 = 0; a0 < n;) {
            int nu = 0;
            for (int b = 0; b < K; ++b) { host_ints[b] = -1; host_ints[K + b] = -1; host_ints[2 * K + b] = -1; }
            for (; a0 < n && nu < K; ++a0) {
                Hyp& h = l[(size_t)a0];
                if (!is_prefix[(size_t)a0] || h.slot >= 0) continue;
                const int s = take_slot();
                if (s < 0) return WIND_ERR_WORKSPACE;
                host_ints[nu] = h.parent;
                host_ints[K + nu] = h.node < 0 ? m.blank_id : nodes[(size_t)h.node].tok;
                host_ints[2 * K + nu] = s;
                h.slot = s;
                ++nu;
            }
            if (nu > 0) BEAM_CUDA(run_update(nu));
        }
        for (Pair& p : pairs) { p.cur = l[(size_t)p.a].slot; refs[p.cur]++; }
        std::vector<float> picked((size_t)K);
        size_t depth = 0;
        for (bool more = true; more; ++depth) {
            more = false;
            std::vector<size_t> act;
            for (size_t i = 0; i < pairs.size(); ++i)
                if (pairs[i].extra.size() > depth) act.push_back(i);
            for (size_t c0 = 0; c0 < act.size(); c0 += (size_t)K) {
                const int nr = (int)std::min((size_t)K, act.size() - c0);
                // log-softmax at frame t under each pair's current state, and the extra token's entry
                for (int b = 0; b < K; ++b) { host_ints[3 * K + b] = -1; host_ints[b] = -1; host_ints[K + b] = -1; host_ints[2 * K + b] = -1; }
                std::vector<int32_t> labels((size_t)K, -1);
                for (int r = 0; r < nr; ++r) {
                    Pair& p = pairs[act[c0 + (size_t)r]];
                    host_ints[3 * K + r] = p.cur;
                    labels[(size_t)r] = p.extra[depth];
                }
                BEAM_CUDA(cudaMemcpyAsync(d_exp, host_ints.data() + 3 * K, sizeof(int32_t) * K, cudaMemcpyHostToDevice, st));
                BEAM_CUDA(cudaMemcpyAsync(d_pick, labels.data(), sizeof(int32_t) * K, cudaMemcpyHostToDevice, st));
                beam_gather_g_kernel<<<K, 128, 0, st>>>(g_pool, d_exp, cb.pred_proj(), d_t, t, T, m.H);
                BEAM_CUDA(launch_set_t(cb, d_t));
                Call one = cb;
                one.W = 1;
                BEAM_CUDA(simt_joint_shared(one, logits));
                BEAM_CUDA(launch_first_output(logits, d_len, d_t, K, 1, NV, m.blank_id, 0, nullptr, nullptr, nullptr, st));
                beam_pick_kernel<<<1, 32, 0, st>>>(logits, d_pick, d_top_logp, K, NV);
                BEAM_CUDA(cudaMemcpyAsync(picked.data(), d_top_logp, sizeof(float) * K, cudaMemcpyDeviceToHost, st));
                BEAM_CUDA(cudaStreamSynchronize(st));
                // one more decoder update for the pairs that have a further token
                int nu = 0;
                for (int r = 0; r < nr; ++r) {
                    Pair& p = pairs[act[c0 + (size_t)r]];
                    p.acc += (double)picked[(size_t)r];
                    if (p.extra.size() > depth + 1) {
                        const int s = take_slot();
                        if (s < 0) return WIND_ERR_WORKSPACE;
                        host_ints[nu] = p.cur;               // released by run_update
                        host_ints[K + nu] = p.extra[depth];
                        host_ints[2 * K + nu] = s;
                        p.cur = s;
                        ++nu;
                        more = true;
                    } else {
                        release(p.cur);
                        p.cur = -1;
                    }
                }
                if (nu > 0) BEAM_CUDA(run_update(nu));
            }
        }
        std::vector<double> add((size_t)n, -INFINITY);
        for (const Pair& p : pairs) add[(size_t)p.b] = log_add(add[(size_t)p.b], p.acc);
        std::vector<Hyp> kept;
        for (int a = 0; a < n; ++a) {
            if (is_prefix[(size_t)a]) {
                release(l[(size_t)a].slot >= 0 ? l[(size_t)a].slot : l[(size_t)a].parent);
            } else {
                l[(size_t)a].score = log_add(l[(size_t)a].score, add[(size_t)a]);
                kept.push_back(l[(size_t)a]);
            }
        }
        l.swap(kept);
        return WIND_OK;
    };
    auto merge_duplicates = [&](std::vector<Hyp>& l) {
        for (size_t a = 0; a < l.size(); ++a)
            for (size_t b = a + 1; b < l.size();) {
                if (l[a].count == l[b].count && same_tokens(l[a].node, l[b].node)) {
                    const double sum = log_add(l[a].score, l[b].score);
                    if (l[b].score > l[a].score) std::swap(l[a], l[b]);
                    l[a].score = sum;
                    release(l[b].slot >= 0 ? l[b].slot : l[b].parent);
                    l.erase(l.begin() + (long)b);
                } else {
                    ++b;
                }
            }
    };
    auto prune = [&](std::vector<Hyp>& l, size_t keep) {
        std::stable_sort(l.begin(), l.end(), [](const Hyp& x, const Hyp& y) { return x.score > y.score; });
        while (l.size() > keep) {
            release(l.back().slot >= 0 ? l.back().slot : l.back().parent);
            l.pop_back();
        }
    };

    // ---- what is known of frames t .. t + look, and forecasts up to a window behind them ----
    std::vector<Frame> frames((size_t)(shape.look + W + 2));
    auto frame_at = [&](int t) -> Frame& { return frames[(size_t)t % frames.size()]; };
    auto clear_frame = [&](Frame& f) {
        for (const Eval& e : f.evals) release(e.slot);
        f.evals.clear();
        f.hash.clear();
        for (int r = 0; r < f.rounds; ++r) {
            for (const Forecast& c : f.round[(size_t)r].best)
                if (!c.asked) release(c.slot >= 0 ? c.slot : c.parent);
            f.round[(size_t)r].best.clear();
        }
        f.rounds = f.open = 0;
    };
    auto find_eval = [&](const Frame& f, int32_t node) {
        const uint64_t h = node_hash(node);
        for (size_t i = 0; i < f.hash.size(); ++i)
            if (f.hash[i] == h && same_tokens(f.evals[i].node, node)) return (int)i;
        return -1;
    };
    auto label_hash = [](uint64_t before, int label) { return (before ^ (uint64_t)(uint32_t)label) * 0x100000001B3ull + 0x9E3779B97F4A7C15ull; };
    // (history, frame) fell out of a list
    std::vector<std::pair<uint64_t, int>> fallen;
    auto remove_fallen = [&] {
        while (!fallen.empty()) {
            const auto [hash, from] = fallen.back();
            fallen.pop_back();
            for (int t = from; t <= from + W + 1 && t < T; ++t) {
                Frame& f = frame_at(t);
                for (int r = 0; r < f.rounds; ++r) {
                    std::vector<Forecast>& best = f.round[(size_t)r].best;
                    for (size_t i = 0; i < best.size();) {
                        if (best[i].from_hash != hash || best[i].from != from) { ++i; continue; }
                        if (best[i].asked) {
                            fallen.emplace_back(best[i].hash, t);
                        } else {
                            release(best[i].slot >= 0 ? best[i].slot : best[i].parent);
                            --f.open;
                        }
                        best[i] = best.back();
                        best.pop_back();
                    }
                }
            }
        }
    };
    // a hypothesis that will stand in round r of frame t: `label` (-1: none) behind the history `node`, whose state is in `slot`
    auto forecast = [&](int t, int r, int from, int32_t node, int label, int slot, int count, double score) {
        if (t >= T || r >= 64) return;
        Frame& f = frame_at(t);
        while (f.rounds <= r) {
            if ((int)f.round.size() <= f.rounds) f.round.emplace_back();
            ++f.rounds;
        }
        std::vector<Forecast>& best = f.round[(size_t)r].best;
        const uint64_t h = label < 0 ? node_hash(node) : label_hash(node_hash(node), label);
        const int len = node_len(node) + (label >= 0);
        size_t worst = 0;
        for (size_t i = 0; i < best.size(); ++i) {
            if (best[i].hash == h && best[i].len == len) {                   // (a forecast: the hash is enough)
                best[i].score = log_add(best[i].score, score);
                if (score > best[i].most) { best[i].most = score; best[i].from = from; best[i].from_hash = node_hash(node); }
                return;
            }
            if (best[i].score < best[worst].score) worst = i;
        }
        Forecast c{h, len, node, label < 0 ? slot : -1, label < 0 ? -1 : slot, count, from, node_hash(node), false, score, score};
        if ((int)best.size() < K) {
            best.emplace_back();
            worst = best.size() - 1;
        } else {
            if (!(score > best[worst].score)) return;
            if (best[worst].asked) {
                fallen.emplace_back(best[worst].hash, t);
            } else {
                release(best[worst].slot >= 0 ? best[worst].slot : best[worst].parent);
                --f.open;
            }
        }
        if (label >= 0) {
            nodes.push_back(Node{node, label, t, len, h});
            c.node = (int32_t)nodes.size() - 1;
        }
        refs[(size_t)slot]++;
        best[worst] = c;
        ++f.open;
    };
    // what follows from an evaluation of frame t, for a hypothesis of its round r
    auto forecast_children = [&](const Eval e, int t, int r, int count, double score) {
        for (int k = 0; k < K; ++k) {
            if (e.label[k] < 0 || !(e.logp[k] > -INFINITY)) continue;
            const double s = score + (double)e.logp[k];
            if (e.label[k] == m.blank_id) {
                forecast(t + std::min(W, T - t), 0, t, e.node, -1, e.slot, 0, s);
            } else {
                const int now = e.jump[k] == 0 ? count + 1 : 1, to = t + e.jump[k] + (now == S);
                forecast(to, to == t ? r + 1 : 0, t, e.node, e.label[k], e.slot, now == S ? 0 : now, s);
            }
        }
    };
    // the rows of a command: hypothesis, frame, round, score and count it counts with
    struct Row { int eval, t, round, count; double score; };
    std::vector<Row> rows;
    std::vector<int> eval_of((size_t)K);
    std::vector<int> parents;               // references to give back once the command is done

    for (int t = 0; t < T; ++t) {
        for (int round = 0; !t2hyps[t].empty(); ++round) {
            std::vector<Hyp> hyps;
            hyps.swap(t2hyps[t]);
            merge_duplicates(hyps);
            if (prefix_search) {
                const wind_status_t ps = prefix_step(hyps, t);
                if (ps != WIND_OK) return ps;
            }
            prune(hyps, (size_t)K);
            const int nh = (int)hyps.size();
            const int n = W < T - t ? W : T - t;
            ++steps;
            if (resident) {
                if ((int)free_slots.size() < K)                              // (evaluations and forecasts hold slots that the hypotheses need)
                    for (Frame& f : frames) clear_frame(f);
                std::fill(words.begin(), words.end(), -1);
                rows.clear();
                parents.clear();
                int nu = 0, reach = t + n;
                int32_t *c_src = words.data() + 4, *c_tok = c_src + R, *c_dst = c_tok + R, *c_slot = c_dst + R, *c_t = c_slot + R;
                // one more hypothesis to evaluate; false: there is no slot for its state
                auto add_row = [&](int32_t node, int slot, int parent, int at, int r, int count, double score) {
                    if (slot < 0) {
                        slot = take_slot();
                        if (slot < 0) return false;
                        c_src[nu] = parent;
                        c_tok[nu] = node < 0 ? m.blank_id : nodes[(size_t)node].tok;
                        c_dst[nu] = slot;
                        ++nu;
                    } else {
                        refs[(size_t)slot]++;
                    }
                    const size_t i = rows.size();
                    c_slot[i] = slot;
                    c_t[i] = at;
                    Frame& f = frame_at(at);
                    rows.push_back(Row{(int)f.evals.size(), at, r, count, score});
                    f.hash.push_back(node_hash(node));
                    f.evals.emplace_back();
                    f.evals.back().node = node;
                    f.evals.back().slot = slot;
                    std::fill(f.evals.back().label, f.evals.back().label + K, -1);       // (nothing follows from it yet)
                    reach = std::max(reach, std::min(at + W, T));
                    return true;
                };
                Frame& here = frame_at(t);
                for (int b = 0; b < nh; ++b) {
                    Hyp& h = hyps[b];
                    int i = find_eval(here, h.node);
                    if (i < 0) {
                        i = (int)here.evals.size();
                        if (!add_row(h.node, h.slot, h.parent, t, round, h.count, h.score)) return WIND_ERR_WORKSPACE;
                    }
                    eval_of[(size_t)b] = i;
                    if (h.slot < 0) {
                        h.slot = here.evals[(size_t)i].slot;
                        refs[(size_t)h.slot]++;
                        parents.push_back(h.parent);
                    }
                }
                // what the forecast had in this list and the list has not
                if (round < here.rounds)
                    for (const Forecast& c : here.round[(size_t)round].best) {
                        bool in = !c.asked;
                        for (int b = 0; b < nh && !in; ++b) in = node_hash(hyps[(size_t)b].node) == c.hash;
                        if (!in) fallen.emplace_back(c.hash, t);
                    }
                if (!rows.empty()) {
                    remove_fallen();
                    // the rest of the command: what comes next, frame by frame and round by round
                    for (int at = t; shape.look > 0 && at <= t + shape.look && at < T && (int)rows.size() < R; ++at) {
                        Frame& f = frame_at(at);
                        for (int r = at == t ? round + 1 : 0; r < f.rounds && f.open > 0 && (int)rows.size() < R; ++r)
                            for (size_t i = 0; i < f.round[(size_t)r].best.size(); ++i) {
                                const Forecast c = f.round[(size_t)r].best[i];
                                if (c.asked) continue;
                                const int known = find_eval(f, c.node);
                                if (known < 0) {
                                    if ((int)rows.size() == R || (int)free_slots.size() <= K) break;
                                    add_row(c.node, c.slot, c.parent, at, r, c.count, c.score);
                                }
                                f.round[(size_t)r].best[i].asked = true;
                                --f.open;
                                parents.push_back(c.slot >= 0 ? c.slot : c.parent);
                                if (known >= 0) forecast_children(f.evals[(size_t)known], at, r, c.count, c.score);
                            }
                    }
                    words[0] = nu; words[1] = (int32_t)rows.size(); words[2] = reach - t; words[3] = t;
                    const wind_status_t rs = dev.run(words.data(), cuda_err);
                    if (rs != WIND_OK) return rs;
                    for (size_t i = 0; i < rows.size(); ++i) {
                        const Row& row = rows[i];
                        Eval& e = frame_at(row.t).evals[(size_t)row.eval];
                        for (int k = 0; k < K; ++k) {
                            const size_t o = 2 * (i * (size_t)K + (size_t)k);
                            const uint32_t at = (uint32_t)dev.mail->top[o], bits = (uint32_t)dev.mail->top[o + 1];
                            e.label[k] = at == 0xffffffffu ? -1 : (int32_t)(at % (uint32_t)NV);
                            e.jump[k] = at == 0xffffffffu ? -1 : (int32_t)(at / (uint32_t)NV);
                            std::memcpy(&e.logp[k], &bits, sizeof(float));
                        }
                    }
                    if (shape.look > 0)
                        for (const Row& row : rows) forecast_children(frame_at(row.t).evals[(size_t)row.eval], row.t, row.round, row.count, row.score);
                }
                for (int q : parents) release(q);
                for (int b = 0; b < nh; ++b) {
                    const Eval& e = here.evals[(size_t)eval_of[(size_t)b]];
                    std::copy(e.label, e.label + K, top.begin() + (size_t)b * K);
                    std::copy(e.jump, e.jump + K, top.begin() + (size_t)K * K + (size_t)b * K);
                    std::memcpy(&top[2 * (size_t)K * K + (size_t)b * K], e.logp, sizeof(float) * (size_t)K);
                }
            } else {
                // ---- decoder update of the survivors that have no state yet ----
                int nu = 0;
                for (int b = 0; b < K; ++b) { host_ints[b] = -1; host_ints[K + b] = -1; host_ints[2 * K + b] = -1; host_ints[3 * K + b] = -1; }
                for (int b = 0; b < nh; ++b) {
                    Hyp& h = hyps[b];
                    if (h.slot < 0) {
                        if (free_slots.empty()) return WIND_ERR_WORKSPACE;
                        const int s = free_slots.back();
                        free_slots.pop_back();
                        refs[s] = 1;
                        host_ints[nu] = h.parent;
                        host_ints[K + nu] = h.node < 0 ? m.blank_id : nodes[(size_t)h.node].tok;
                        host_ints[2 * K + nu] = s;
                        h.slot = s;
                        ++nu;
                    }
                }
                for (int b = 0; b < nh; ++b) host_ints[3 * K + b] = hyps[b].slot;
                BEAM_CUDA(cudaMemcpyAsync(d_exp, host_ints.data() + 3 * K, sizeof(int32_t) * K, cudaMemcpyHostToDevice, st));
                beam_gather_g_kernel<<<K, 128, 0, st>>>(g_pool, d_exp, cb.pred_proj(), d_t, t, T, m.H);   // sets the frames first
                BEAM_CUDA(launch_set_t(cb, d_t));   // frames of the rows, and the control block's "active" word
                if (nu > 0) {
                    BEAM_CUDA(run_update(nu));   // (the parents are no longer needed by these hypotheses)
                    beam_gather_g_kernel<<<K, 128, 0, st>>>(g_pool, d_exp, cb.pred_proj(), d_t, t, T, m.H);
                }
                // ---- window logits of every hypothesis, Eq. (1), the K best entries each ----
                BEAM_CUDA(simt_joint_shared(cb, logits));
                BEAM_CUDA(launch_first_output(logits, d_len, d_t, K, W, NV, m.blank_id, K, d_top_label, d_top_jump, d_top_logp, st));
                BEAM_CUDA(cudaMemcpyAsync(top.data(), d_top_label, sizeof(int32_t) * 3 * K * K, cudaMemcpyDeviceToHost, st));
                BEAM_CUDA(cudaStreamSynchronize(st));
            }
            // ---- expansions ----
            for (int b = 0; b < nh; ++b) {
                const Hyp& h = hyps[b];
                for (int k = 0; k < K; ++k) {
                    const int label = top_label[(size_t)b * K + k], jump = top_jump[(size_t)b * K + k];
                    const float lp = top_logp[(size_t)b * K + k];
                    if (label < 0 || !(lp > -INFINITY)) continue;    // fewer than K entries in a small window
                    Hyp nhyp;
                    nhyp.score = h.score + (double)lp;
                    if (label != m.blank_id) {
                        int tt = t + jump;
                        Node nd;
                        nd.parent = h.node; nd.tok = label; nd.frm = tt; nd.len = node_len(h.node) + 1;
                        nd.hash = label_hash(node_hash(h.node), label);
                        nodes.push_back(nd);
                        nhyp.node = (int32_t)nodes.size() - 1;
                        nhyp.count = jump == 0 ? h.count + 1 : 1;
                        nhyp.parent = h.slot;
                        refs[h.slot]++;
                        if (nhyp.count == S) { tt += 1; nhyp.count = 0; }
                        t2hyps[tt].push_back(std::move(nhyp));
                    } else {
                        nhyp.node = h.node;
                        nhyp.count = 0;
                        nhyp.slot = h.slot;
                        refs[h.slot]++;
                        t2hyps[t + n].push_back(std::move(nhyp));
                    }
                }
            }
            for (int b = 0; b < nh; ++b) release(hyps[b].slot);
            if (shape.look == 0) clear_frame(frame_at(t));
        }
        clear_frame(frame_at(t));
    }
    std::vector<Hyp>& fin = t2hyps[T];
    merge_duplicates(fin);
    prune(fin, fin.size() > 0 ? fin.size() : 1);
    int n_out = 0;
    for (size_t a = 0; a < fin.size() && (int)a < max_hyps; ++a) {
        const Hyp& h = fin[a];
        const int len = node_len(h.node);
        out_len[a] = len;
        out_score[a] = h.score;
        int32_t nd = h.node;
        for (int k = len - 1; k >= 0; --k) {   // walk the history back from the last token
            if (k < max_out) {
                out_tokens[a * (size_t)max_out + k] = nodes[(size_t)nd].tok;
                out_frames[a * (size_t)max_out + k] = nodes[(size_t)nd].frm;
            }
            nd = nodes[(size_t)nd].parent;
        }
        ++n_out;
    }
    *n_hyps = n_out;
    if (n_steps) *n_steps = steps;
#undef BEAM_CUDA
    return WIND_OK;
}

}  // namespace wind
