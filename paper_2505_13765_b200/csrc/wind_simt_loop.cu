// The decoding loop of the plain-ALU path (fp32 models, and bf16 models outside the tensor-core set) as one persistent kernel.
//
// As separate kernels in a CUDA graph a lock step cost 20 us for a model of 64 units (launches) and 300 us for one of 640
// units in fp32 (every weight read again by kernels with one block per output).  Here the weights stay in shared memory:
//   one SM  the whole decoder fits one SM (64 units in fp32: 186 KB): a CTA decodes its utterances one after the other and
//           nothing leaves the SM but the transcripts; the phases of a step are separated by block barriers.
//   grid    otherwise: hidden units, joint units and labels are dealt out over all SMs (640 units in fp32: 143 KB each), and
//           the phases are separated by grid barriers (1.3 us each).  Models whose weights do not fit on the chip run the
//           same code and read them from L2.
//
// Phases of a lock step (Algorithm 2 for every utterance at once):
//   control   every CTA takes the decisions for all utterances from the window's keys (the same ones everywhere), CTA 0
//             records them; without an emission in the batch the two decoder phases are skipped
//   update    per layer: gates = W_ih x + W_hh h, cell update
//   project   pred_proj = W_pred h
//   joint     z = act(enc_proj + pred_proj), by every CTA for itself; logits = W_out z for this CTA's labels, the best
//             (logit, label) key of every window row
// Sums are fp32 FMA; bf16 operands (weights, enc_proj, h, z) are rounded where the per-phase kernels round them.
#include <mutex>
#include <type_traits>

#include "wind_internal.cuh"
#include "wind_loop.cuh"
#include "wind_ptx.cuh"

namespace wind {

constexpr int SL_THREADS = 512;
constexpr int SL_WARPS = SL_THREADS / 32;
constexpr int SL_UTTS = 4;          // utterances of a pass of the decoder phases
constexpr int SL_ROWS = 4;          // window rows of a joint item
constexpr int SL_MAX_B = 512;       // most utterances (their state is kept in every CTA)

struct SimtLoopParams {
    Ctrl* ctrl;
    int B, T, W, S, max_out, E, P, L, H, NV, blank, act, step_cap, extra_arrivals;
    const void* emb;
    const void* w_ih[kMaxLayers];
    const void* w_hh[kMaxLayers];
    const float* b_ih[kMaxLayers];
    const float* b_hh[kMaxLayers];
    const void* w_pred;
    const float* b_pred;
    const void* w_out;
    const float* b_out;
    const void* enc_proj;
    const int32_t* enc_len;
    float* h;                      // [2][L][B][P], a parity per utterance
    float* c;                      // [L][B][P]
    float* pred;                   // [B][H]
    unsigned long long* keys;      // [3][B * W]
    int32_t* out_tokens;
    int32_t* out_frames;
    int32_t* out_len;
};

template <typename TW> __device__ __forceinline__ float sl_round(float x);
template <> __device__ __forceinline__ float sl_round<float>(float x) { return x; }
template <> __device__ __forceinline__ float sl_round<__nv_bfloat16>(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// ---------------------------------------------------------------------------
// The decoder spread over the grid.  What a CTA owns: units, joint units and labels i * G + cta.
//
// Operands lie interleaved by four in shared memory ([k][4] weight rows, [k][4] utterances or window rows), so that a lane's step
// of a 4 x 4 block of dot products is two loads for sixteen FMAs; K is cut over the warps that would have no block of their own.
// Every CTA forms all of z for itself, which saves a barrier and costs nothing: it would have to read as much z as it reads
// enc_proj (82 KB a step at four utterances x 8 rows x 640 units: with 148 CTAs at it that is 7400 of a step's 34000 cycles, three
// barriers 8000, the joint's products 5500).  With a warp per row, generic pointers and z handed over through L2 behind a fourth
// barrier a step took 39400 cycles.  (Rows of z as they are, copied ahead while the decoder is updated: z 4700, but five loads
// instead of two per step of the products, 7900.)
// ---------------------------------------------------------------------------
struct SlPlan {
    int units, prows, labels;         // the most a CTA owns of each
    int e32, p32, h32;                // E, P, H rounded up to 32
    int k_l;                          // elements of a row of the gates, any layer: input and state, each rounded up to 32
    int zrows;                        // window rows of a joint pass
    uint32_t layer, w_l, w_pred, w_out, part, b_gate, b_pred, b_out, ints, x, z, total;   // bytes
};
template <typename TW>
static SlPlan sl_plan_grid(int G, int B, int W, int E, int P, int L, int H, int NV, bool resident, unsigned long long budget) {
    SlPlan s{};
    s.units = (P + G - 1) / G; s.prows = (H + G - 1) / G; s.labels = (NV + G - 1) / G;
    s.e32 = (E + 31) / 32 * 32; s.p32 = (P + 31) / 32 * 32; s.h32 = (H + 31) / 32 * 32;
    s.k_l = (L > 1 && s.p32 > s.e32 ? s.p32 : s.e32) + s.p32;
    const unsigned long long es = sizeof(TW);
    unsigned long long off = 0;
    auto take = [&](unsigned long long bytes) { const unsigned long long o = off; off += (bytes + 15) / 16 * 16; return (uint32_t)o; };
    auto up4 = [](int n) { return (unsigned long long)((n + 3) / 4 * 4); };
    const unsigned long long layer = es * s.units * 4 * s.k_l;
    s.layer = (uint32_t)layer;
    s.w_l = take(resident ? layer * L : 0);
    s.w_pred = take(resident ? es * up4(s.prows) * s.p32 : 0);
    s.w_out = take(resident ? es * up4(s.labels) * s.h32 : 0);
    const int groups = (s.prows + 3) / 4, blocks = s.units > groups ? s.units : groups;
    s.part = take(4ull * 16 * (blocks > SL_WARPS ? blocks : SL_WARPS));
    s.b_gate = take(4ull * L * s.units * 4);
    s.b_pred = take(4ull * s.prows);
    s.b_out = take(4ull * s.labels);
    s.ints = take(4ull * 8 * B);
    s.z = (uint32_t)off;
    const unsigned long long x = 16ull * s.k_l, row = 4ull * s.h32;
    const long long all = ((long long)B * W + SL_ROWS - 1) / SL_ROWS * SL_ROWS;
    const long long fit = off < budget ? (long long)((budget - off) / (row * SL_ROWS)) * SL_ROWS : 0;
    long long rows = fit < all ? fit : all;
    if (rows > SL_THREADS / 4) rows = SL_THREADS / 4;
    s.zrows = (int)rows;
    s.x = s.z;                        // (x and z are not needed at the same time)
    off += row * rows > x ? row * rows : x;
    s.total = rows < SL_ROWS || off > budget ? 0xffffffffu : (uint32_t)off;
    return s;
}

// Shared memory: four weight rows and four rows of x, both [k][4]; the addresses are the lane's first element.  Afterwards lane l
// holds the dot product of weight row l >> 3 and x row (l >> 1) & 3.
__device__ __forceinline__ float sl_block_sums(float* a) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int half = 8; half >= 1; half >>= 1) {
        const bool up = (lane & (2 * half)) != 0;
#pragma unroll
        for (int c = 0; c < half; ++c) {
            const float send = up ? a[c] : a[c + half], keep = up ? a[c + half] : a[c];
            a[c] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * half);
        }
    }
    return a[0] + __shfl_xor_sync(0xffffffffu, a[0], 1);
}
__device__ __forceinline__ void sl_block_step(float* a, const float* wv, uint32_t x) {
    float xv[4];
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(xv[0]), "=f"(xv[1]), "=f"(xv[2]), "=f"(xv[3]) : "r"(x));
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int n = 0; n < 4; ++n) a[4 * j + n] = fmaf(wv[j], xv[n], a[4 * j + n]);
}
template <typename TW>
__device__ __noinline__ float sl_block(uint32_t w, uint32_t x, int steps) {
    float a[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = 0.f;
#pragma unroll 4
    for (int i = 0; i < steps; ++i) {
        float wv[4];
        if constexpr (sizeof(TW) == 2) {
            uint32_t v0, v1;
            asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v0), "=r"(v1) : "r"(w + 256u * i));
            wv[0] = __uint_as_float(v0 << 16); wv[1] = __uint_as_float(v0 & 0xffff0000u);
            wv[2] = __uint_as_float(v1 << 16); wv[3] = __uint_as_float(v1 & 0xffff0000u);
        } else {
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(wv[0]), "=f"(wv[1]), "=f"(wv[2]), "=f"(wv[3]) : "r"(w + 512u * i));
        }
        sl_block_step(a, wv, x + 512u * i);
    }
    return sl_block_sums(a);
}
// the same with the weight rows in global memory (r[j] null: no such row): k = k0 + lane, ... below n
template <typename TW>
__device__ __noinline__ float sl_block_global(const TW* r0, const TW* r1, const TW* r2, const TW* r3, int k0, int n, uint32_t x, int steps) {
    float a[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = 0.f;
    const TW* const r[4] = {r0, r1, r2, r3};
#pragma unroll 4
    for (int i = 0; i < steps; ++i) {
        const int k = k0 + 32 * i + (int)(threadIdx.x & 31);
        float wv[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) wv[j] = r[j] && k < n ? (float)__ldg(r[j] + k) : 0.f;
        sl_block_step(a, wv, x + 512u * i);
    }
    return sl_block_sums(a);
}

template <typename TW, bool RES>
__global__ void __launch_bounds__(SL_THREADS, 1) simt_grid_kernel(const SimtLoopParams p, const SlPlan M) {
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ int s_stop, s_n_emit, s_n_alive;
    __shared__ int s_hist[65];
    __shared__ int s_b[SL_THREADS / 4], s_enc[SL_THREADS / 4];     // of a row of the joint pass: utterance (-1: none), enc_proj row
    __shared__ unsigned long long s_key[SL_THREADS / 4];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, grp = lane >> 3, col = (lane >> 1) & 3;
    const int G = gridDim.x, cta = blockIdx.x;
    if (p.ctrl->bad_input) return;                 // a length outside [0, T]: nothing is read through it
    const int B = p.B, P = p.P, H = p.H, W = p.W;
    const int units = (P - cta + G - 1) / G, prows = (H - cta + G - 1) / G, labels = (p.NV - cta + G - 1) / G;
    TW* w_pred = reinterpret_cast<TW*>(sm + M.w_pred);
    TW* w_out = reinterpret_cast<TW*>(sm + M.w_out);
    float* part = reinterpret_cast<float*>(sm + M.part);
    float* b_gate = reinterpret_cast<float*>(sm + M.b_gate);       // [layer][own unit][gate] b_ih + b_hh
    float* b_pred = reinterpret_cast<float*>(sm + M.b_pred);
    float* b_out = reinterpret_cast<float*>(sm + M.b_out);
    float* xs = reinterpret_cast<float*>(sm + M.x);
    float* zs = reinterpret_cast<float*>(sm + M.z);
    int* s_t = reinterpret_cast<int*>(sm + M.ints);
    int *s_len = s_t + B, *s_cnt = s_t + 2 * B, *s_pos = s_t + 3 * B, *s_tok = s_t + 4 * B, *s_hp = s_t + 5 * B, *s_list = s_t + 6 * B, *s_alive = s_t + 7 * B;
    const TW* emb = static_cast<const TW*>(p.emb);
    const TW* enc_proj = static_cast<const TW*>(p.enc_proj);

    // ---- weights ----
    auto w_layer = [&](int l) { return reinterpret_cast<TW*>(sm + M.w_l + (size_t)l * M.layer); };
    auto interleave = [&](TW* dst, const TW* r0, const TW* r1, const TW* r2, const TW* r3, int n, int n32) {   // (null: no such row)
#pragma unroll 4
        for (int k = lane; k < n32; k += 32) {
            const TW zero = (TW)0.f;
            TW* d = dst + 4 * k;
            d[0] = r0 && k < n ? __ldg(r0 + k) : zero;
            d[1] = r1 && k < n ? __ldg(r1 + k) : zero;
            d[2] = r2 && k < n ? __ldg(r2 + k) : zero;
            d[3] = r3 && k < n ? __ldg(r3 + k) : zero;
        }
    };
    auto own_row = [&](const void* w, int i, int rows, int n) { return i < rows ? static_cast<const TW*>(w) + ((size_t)i * G + cta) * n : nullptr; };
    if (RES) {
#pragma unroll 1
        for (int l = 0; l < p.L; ++l) {
            const int nin = l == 0 ? p.E : P, nin32 = l == 0 ? M.e32 : M.p32;
            const TW *wi = static_cast<const TW*>(p.w_ih[l]), *wh = static_cast<const TW*>(p.w_hh[l]);
#pragma unroll 1
            for (int i = warp; i < units; i += SL_WARPS) {
                const size_t j = (size_t)i * G + cta;
                TW* dst = w_layer(l) + 4 * i * M.k_l;
                interleave(dst, wi + j * nin, wi + (P + j) * nin, wi + (2 * (size_t)P + j) * nin, wi + (3 * (size_t)P + j) * nin, nin, nin32);
                interleave(dst + 4 * nin32, wh + j * P, wh + (P + j) * P, wh + (2 * (size_t)P + j) * P, wh + (3 * (size_t)P + j) * P, P, M.p32);
            }
        }
#pragma unroll 1
        for (int i = 4 * warp; i < prows; i += 4 * SL_WARPS)
            interleave(w_pred + i * M.p32, own_row(p.w_pred, i, prows, P), own_row(p.w_pred, i + 1, prows, P), own_row(p.w_pred, i + 2, prows, P),
                       own_row(p.w_pred, i + 3, prows, P), P, M.p32);
#pragma unroll 1
        for (int i = 4 * warp; i < labels; i += 4 * SL_WARPS)
            interleave(w_out + i * M.h32, own_row(p.w_out, i, labels, H), own_row(p.w_out, i + 1, labels, H), own_row(p.w_out, i + 2, labels, H),
                       own_row(p.w_out, i + 3, labels, H), H, M.h32);
    }
#pragma unroll 1
    for (int i = tid; i < p.L * units * 4; i += SL_THREADS) {
        const int l = i / (units * 4), r = i - l * units * 4, at = (r & 3) * P + (r >> 2) * G + cta;
        b_gate[4 * l * M.units + r] = p.b_ih[l][at] + p.b_hh[l][at];
    }
#pragma unroll 1
    for (int i = tid; i < prows; i += SL_THREADS) b_pred[i] = p.b_pred[i * G + cta];
#pragma unroll 1
    for (int i = tid; i < labels; i += SL_THREADS) b_out[i] = p.b_out[i * G + cta];
    if (tid == 0) s_stop = 0;
#pragma unroll 1
    for (int k = tid; k < 65; k += SL_THREADS) s_hist[k] = 0;

    // Barrier of all CTAs between phases.  False when the kernel is being abandoned (bounded wait).
    uint32_t epoch = 0;
    auto phase_sync = [&]() -> bool {
        __syncthreads();
        if (tid == 0) {
            epoch += (uint32_t)(G + p.extra_arrivals);
            __threadfence();
            atomicAdd(&p.ctrl->bar, 1u);
            unsigned long long t0 = 0;
#pragma unroll 1
            for (uint32_t it = 1;; ++it) {
                uint32_t v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&p.ctrl->bar) : "memory");
                if ((int32_t)(v - epoch) >= 0) break;
                if ((it & 63u) == 0u) {
                    const unsigned long long now = globaltimer_ns();
                    if (t0 == 0) t0 = now;
                    else if (now - t0 > kWaitLimitNs) { s_stop = 1; break; }
                }
            }
        }
        __syncthreads();
        return s_stop == 0;
    };
    auto h_row = [&](int par, int l, int b) { return p.h + (((size_t)par * p.L + l) * B + b) * P; };
    // rows [r0, ..) of the live utterances' windows into s_b, s_enc
    auto list_rows = [&](int r0, int nr) {
#pragma unroll 1
        for (int r = tid; r < nr; r += SL_THREADS) {
            const int i = (r0 + r) / W, w = r0 + r - i * W, b = s_alive[i], t = s_t[b] + w;
            const bool in = t < s_len[b];
            s_b[r] = in ? b : -1;
            s_enc[r] = b * p.T + (in ? t : 0);
            s_key[r] = 0ull;
        }
    };

    // ---- start of sequence ----
#pragma unroll 1
    for (int b = tid; b < B; b += SL_THREADS) {
        s_t[b] = 0;
        s_len[b] = min(max(p.enc_len[b], 0), p.T);
        s_cnt[b] = 0; s_pos[b] = 0; s_hp[b] = 0;
        s_tok[b] = s_len[b] > 0 ? p.blank : -1;
    }
    __syncthreads();
    long long n_rows = 0, n_tok = 0, n_forced = 0;                 // thread-local counts of the recording CTA
    int steps = 0;
#pragma unroll 1
    for (int step = -1;; ++step) {
        // =============================================================================
        // control: decisions for every utterance, in every CTA; lists of emitting and of live utterances
        // =============================================================================
        if (step >= 0) {
            const unsigned long long* keys = p.keys + (size_t)(step % 3) * B * W;
#pragma unroll 1
            for (int b = tid; b < B; b += SL_THREADS) {
                int t = s_t[b], tok = -1;
                const int len = s_len[b];
                if (t < len) {
                    const int n = min(p.W, len - t);
                    int first = -1, label = p.blank;
                    bool bad = false;
#pragma unroll 1
                    for (int w0 = 0; w0 < n && first < 0; w0 += 4) {
                        unsigned long long kk[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            kk[j] = 0ull;
                            if (w0 + j < n) {
                                kk[j] = __ldcg(keys + (size_t)b * p.W + w0 + j);
                            }
                        }
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (first < 0 && w0 + j < n) {
                                uint32_t lab = key_label(kk[j]);
                                if (kk[j] == 0ull || lab >= (uint32_t)p.NV) { bad = true; lab = (uint32_t)p.blank; }
                                if ((int)lab != p.blank) { first = w0 + j; label = (int)lab; }
                            }
                    }
                    const int pos = s_pos[b];
                    int cnt = s_cnt[b], jump = first < 0 ? n : first, forced = 0;
                    if (jump > 0) cnt = 0;
                    t += jump;
                    const int t_emit = t;
                    bool overflow = false;
                    if (first >= 0) {
                        if (pos < p.max_out) {
                            tok = label;
                            s_pos[b] = pos + 1;
                            if (++cnt == p.S) { ++t; cnt = 0; forced = 1; }
                        } else {
                            overflow = true;
                            t = len;                                          // this utterance stops here
                        }
                    }
                    s_t[b] = t;
                    s_cnt[b] = cnt;
                    if (blockIdx.x == 0) {                           // recorded once
                        if (tok >= 0) {
                            p.out_tokens[(size_t)b * p.max_out + pos] = label;
                            p.out_frames[(size_t)b * p.max_out + pos] = t_emit;
                            p.out_len[b] = pos + 1;
                        }
                        n_rows += n; n_tok += tok >= 0; n_forced += forced;
                        atomicAdd(&s_hist[jump < 64 ? jump : 64], 1);
                        if (overflow) set_status(p.ctrl, WIND_ERR_OUTPUT_OVERFLOW);
                        if (bad) set_status(p.ctrl, WIND_ERR_INTERNAL);
                    }
                }
                s_tok[b] = tok;
            }
            ++steps;
        }
        __syncthreads();
        if (warp == 0) {
            int ne = 0, na = 0;
#pragma unroll 1
            for (int b0 = 0; b0 < B; b0 += 32) {
                const int b = b0 + lane;
                const bool live = b < B && s_t[b] < s_len[b], em = live && s_tok[b] >= 0;   // a finished utterance needs no further state
                const uint32_t m = __ballot_sync(0xffffffffu, em), ml = __ballot_sync(0xffffffffu, live), below = (1u << lane) - 1u;
                if (em) s_list[ne + __popc(m & below)] = b;
                if (live) s_alive[na + __popc(ml & below)] = b;
                ne += __popc(m);
                na += __popc(ml);
            }
            if (lane == 0) { s_n_emit = ne; s_n_alive = na; }
        }
        __syncthreads();
        const int n_emit = s_n_emit, rows = s_n_alive * W;
        if (rows == 0) break;
        if (steps >= p.step_cap) { if (tid == 0 && cta == 0) set_status(p.ctrl, WIND_ERR_INTERNAL); break; }
        // =============================================================================
        // update and projection of the emitting utterances
        // =============================================================================
        if (n_emit > 0) {
#pragma unroll 1
            for (int l = 0; l < p.L; ++l) {
                const int nin = l == 0 ? p.E : P, nin32 = l == 0 ? M.e32 : M.p32, steps_l = (nin32 + M.p32) / 32;
                const int KS = units > 0 && units < SL_WARPS ? SL_WARPS / units : 1;
#pragma unroll 1
                for (int i0 = 0; i0 < n_emit; i0 += SL_UTTS) {
                    const int n_here = min(SL_UTTS, n_emit - i0);
                    int b4[SL_UTTS], tok[SL_UTTS], hp[SL_UTTS];
#pragma unroll
                    for (int u = 0; u < SL_UTTS; ++u) { b4[u] = s_list[i0 + min(u, n_here - 1)]; tok[u] = s_tok[b4[u]]; hp[u] = s_hp[b4[u]]; }
                    // one half of the threads the input, the other the state before; the cells' old state is requested as well
                    const int c_ui = tid / n_here, c_u = tid - c_ui * n_here;
                    const float c_first = tid < units * n_here ? p.c[((size_t)l * B + s_list[i0 + c_u]) * P + c_ui * G + cta] : 0.f;
                    if (tid < SL_THREADS / 2 && l == 0) {
#pragma unroll 3
                        for (int k = tid; k < nin32; k += SL_THREADS / 2) {
                            float x[SL_UTTS];
#pragma unroll
                            for (int u = 0; u < SL_UTTS; ++u) x[u] = k < nin ? (float)__ldg(emb + (size_t)tok[u] * p.E + k) : 0.f;
                            *reinterpret_cast<float4*>(xs + 4 * k) = make_float4(x[0], x[1], x[2], x[3]);
                        }
                    } else {
                        const bool state = tid >= SL_THREADS / 2;
                        const int n = state ? P : nin, n32 = state ? M.p32 : nin32, at = state ? nin32 : 0;
                        const float* hr[SL_UTTS];
#pragma unroll
                        for (int u = 0; u < SL_UTTS; ++u) hr[u] = state ? h_row(hp[u], l, b4[u]) : h_row(hp[u] ^ 1, l - 1, b4[u]);
#pragma unroll 3
                        for (int k = tid & (SL_THREADS / 2 - 1); k < n32; k += SL_THREADS / 2) {
                            float x[SL_UTTS];
#pragma unroll
                            for (int u = 0; u < SL_UTTS; ++u) x[u] = k < n ? sl_round<TW>(__ldcg(hr[u] + k)) : 0.f;
                            *reinterpret_cast<float4*>(xs + 4 * (at + k)) = make_float4(x[0], x[1], x[2], x[3]);
                        }
                    }
                    __syncthreads();
#pragma unroll 1
                    for (int item = warp; item < units * KS; item += SL_WARPS) {
                        const int ks = item / units, ui = item - ks * units, s0 = steps_l * ks / KS, s1 = steps_l * (ks + 1) / KS;
                        const uint32_t xa = smem_u32(xs + 4 * lane);
                        float v;
                        if constexpr (RES) {
                            v = sl_block<TW>(smem_u32(w_layer(l) + 4 * (ui * M.k_l + 32 * s0 + lane)), xa + 512u * s0, s1 - s0);
                        } else {
                            const size_t j = (size_t)ui * G + cta;
                            const TW *wi = static_cast<const TW*>(p.w_ih[l]) + j * nin, *wh = static_cast<const TW*>(p.w_hh[l]) + j * P;
                            const size_t gi = (size_t)P * nin, gh = (size_t)P * P;
                            const int mid = min(max(nin32 / 32, s0), s1);
                            v = sl_block_global<TW>(wi, wi + gi, wi + 2 * gi, wi + 3 * gi, 32 * s0, nin, xa + 512u * s0, mid - s0);
                            v += sl_block_global<TW>(wh, wh + gh, wh + 2 * gh, wh + 3 * gh, 32 * mid - nin32, P, xa + 512u * mid, s1 - mid);
                        }
                        if ((lane & 1) == 0) part[item * 16 + grp * 4 + col] = v;
                    }
                    __syncthreads();
#pragma unroll 1
                    for (int i = tid; i < units * n_here; i += SL_THREADS) {
                        const int ui = i / n_here, u = i - ui * n_here, b = s_list[i0 + u], j = ui * G + cta;
                        float* cs = p.c + ((size_t)l * B + b) * P + j;
                        const float c_old = i == tid ? c_first : *cs;
                        float a[4];
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            float s = 0.f;
#pragma unroll 1
                            for (int ks = 0; ks < KS; ++ks) s += part[(ks * units + ui) * 16 + g * 4 + u];
                            a[g] = s + b_gate[4 * (l * M.units + ui) + g];
                        }
                        const float gi = 1.f / (1.f + expf(-a[0])), gf = 1.f / (1.f + expf(-a[1])), gg = tanhf(a[2]), go = 1.f / (1.f + expf(-a[3]));
                        const float cc = cell_update_fc(gf, c_old, gi, gg);
                        *cs = cc;
                        h_row(s_hp[b] ^ 1, l, b)[j] = go * tanhf(cc);
                    }
                    if (i0 + SL_UTTS < n_emit) __syncthreads();
                }
                if (!phase_sync()) goto done;
            }
            const int pgs = (prows + 3) / 4, KS = pgs > 0 && pgs < SL_WARPS ? SL_WARPS / pgs : 1, steps_p = M.p32 / 32;
#pragma unroll 1
            for (int i0 = 0; i0 < n_emit; i0 += SL_UTTS) {
                const int n_here = min(SL_UTTS, n_emit - i0);
                int b4[SL_UTTS];
#pragma unroll
                for (int u = 0; u < SL_UTTS; ++u) b4[u] = s_list[i0 + min(u, n_here - 1)];
                const float* hr[SL_UTTS];
#pragma unroll
                for (int u = 0; u < SL_UTTS; ++u) hr[u] = h_row(s_hp[b4[u]] ^ 1, p.L - 1, b4[u]);
#pragma unroll 2
                for (int k = tid; k < M.p32; k += SL_THREADS) {
                    float x[SL_UTTS];
#pragma unroll
                    for (int u = 0; u < SL_UTTS; ++u) x[u] = k < P ? sl_round<TW>(__ldcg(hr[u] + k)) : 0.f;
                    *reinterpret_cast<float4*>(xs + 4 * k) = make_float4(x[0], x[1], x[2], x[3]);
                }
                __syncthreads();
#pragma unroll 1
                for (int item = warp; item < pgs * KS; item += SL_WARPS) {
                    const int ks = item / pgs, pg = item - ks * pgs, s0 = steps_p * ks / KS, s1 = steps_p * (ks + 1) / KS;
                    const uint32_t xa = smem_u32(xs + 4 * (32 * s0 + lane));
                    float v;
                    if constexpr (RES) v = sl_block<TW>(smem_u32(w_pred + 4 * (pg * M.p32 + 32 * s0 + lane)), xa, s1 - s0);
                    else v = sl_block_global<TW>(own_row(p.w_pred, 4 * pg, prows, P), own_row(p.w_pred, 4 * pg + 1, prows, P), own_row(p.w_pred, 4 * pg + 2, prows, P),
                                                 own_row(p.w_pred, 4 * pg + 3, prows, P), 32 * s0, P, xa, s1 - s0);
                    if ((lane & 1) == 0) part[item * 16 + grp * 4 + col] = v;
                }
                __syncthreads();
#pragma unroll 1
                for (int i = tid; i < prows * n_here; i += SL_THREADS) {
                    const int pi = i / n_here, u = i - pi * n_here;
                    float s = 0.f;
#pragma unroll 1
                    for (int ks = 0; ks < KS; ++ks) s += part[(ks * pgs + (pi >> 2)) * 16 + (pi & 3) * 4 + u];
                    p.pred[(size_t)s_list[i0 + u] * H + pi * G + cta] = s + b_pred[pi];
                }
                if (i0 + SL_UTTS < n_emit) __syncthreads();
            }
            if (!phase_sync()) goto done;
#pragma unroll 1
            for (int i = tid; i < n_emit; i += SL_THREADS) s_hp[s_list[i]] ^= 1;
        }
        // =============================================================================
        // joint
        // =============================================================================
        // three sets of keys in turn: read by the control step, raised by the joint, cleared for the joint of the next step
        unsigned long long *knext = p.keys + (size_t)((step + 1) % 3) * B * W, *kclear = p.keys + (size_t)((step + 2) % 3) * B * W;
        if (cta == 0)
#pragma unroll 1
            for (int i = tid; i < B * W; i += SL_THREADS) kclear[i] = 0ull;
#pragma unroll 1
        for (int r0 = 0; r0 < rows; r0 += M.zrows) {
            const int nr = min(M.zrows, rows - r0), nr4 = (nr + SL_ROWS - 1) / SL_ROWS;
            if (r0 > 0) __syncthreads();
            list_rows(r0, nr);
            __syncthreads();
            // z: a warp takes a group of four rows and a share of k; every load of five steps is requested before the first is used
            const int cut = nr4 < SL_WARPS ? SL_WARPS / nr4 : 1;
#pragma unroll 1
            for (int item = warp; item < nr4 * cut; item += SL_WARPS) {
                const int rg = item / cut;
                const TW* er[4];
                const float* pr[4];
                bool same = true;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int r = min(4 * rg + j, nr - 1), b = s_b[r];
                    er[j] = enc_proj + (size_t)s_enc[r] * H;
                    pr[j] = p.pred + (size_t)max(b, 0) * H;
                    same = same && (b < 0 || pr[j] == pr[0]);          // rows past an utterance's end count for nothing
                }
                auto rows4 = [&](auto one) {
#pragma unroll 5
                    for (int k = lane + 32 * (item - rg * cut); k < M.h32; k += 32 * cut) {
                        float z[4] = {0.f, 0.f, 0.f, 0.f}, g[4] = {0.f, 0.f, 0.f, 0.f};
                        if (k < H) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) z[j] = (float)__ldg(er[j] + k);
#pragma unroll
                            for (int j = 0; j < 4; ++j) g[j] = !decltype(one)::value || j == 0 ? __ldcg(pr[j] + k) : g[0];
                        }
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            z[j] += g[j];
                            if (p.act == WIND_ACT_RELU) z[j] = fmaxf(z[j], 0.f);
                        }
                        if (p.act != WIND_ACT_RELU) {
#pragma unroll 1
                            for (int j = 0; j < 4; ++j) {              // one tanh in the code
                                const float v = tanhf(z[0]);
                                z[0] = z[1]; z[1] = z[2]; z[2] = z[3]; z[3] = v;
                            }
                        }
                        *reinterpret_cast<float4*>(zs + 4 * (rg * M.h32 + k)) =
                            make_float4(sl_round<TW>(z[0]), sl_round<TW>(z[1]), sl_round<TW>(z[2]), sl_round<TW>(z[3]));
                    }
                };
                if (same) rows4(std::integral_constant<bool, true>{});
                else rows4(std::integral_constant<bool, false>{});
            }
            __syncthreads();
            const int lgs = (labels + 3) / 4;
#pragma unroll 1
            for (int item = warp; item < lgs * nr4; item += SL_WARPS) {
                const int rg = item / lgs, lg = item - rg * lgs, li = lg * 4 + grp, r = rg * 4 + col;
                const uint32_t xa = smem_u32(zs + 4 * (rg * M.h32 + lane));
                float v;
                if constexpr (RES) v = sl_block<TW>(smem_u32(w_out + 4 * (lg * M.h32 + lane)), xa, M.h32 / 32);
                else v = sl_block_global<TW>(own_row(p.w_out, 4 * lg, labels, H), own_row(p.w_out, 4 * lg + 1, labels, H), own_row(p.w_out, 4 * lg + 2, labels, H),
                                             own_row(p.w_out, 4 * lg + 3, labels, H), 0, H, xa, M.h32 / 32);
                unsigned long long key = 0ull;
                if (li < labels) {
                    v += b_out[li];
                    if (v > -INFINITY) key = pack_key(v, (uint32_t)(li * G + cta));
                }
                key = max(key, __shfl_xor_sync(0xffffffffu, key, 8));
                key = max(key, __shfl_xor_sync(0xffffffffu, key, 16));
                if ((lane & 25) == 0 && r < nr && s_b[r] >= 0 && key != 0ull) atomicMax(&s_key[r], key);
            }
            __syncthreads();
#pragma unroll 1
            for (int r = tid; r < nr; r += SL_THREADS)
                if (s_key[r] != 0ull) {
                    const int b = s_b[r], w = s_enc[r] - b * p.T - s_t[b];
                    atomicMax(&knext[(size_t)b * W + w], s_key[r]);
                }
        }
        if (!phase_sync()) goto done;
    }
    // ---- counters ----
    if (cta == 0) {
        if (tid == 0) atomicMax(&p.ctrl->step, steps);
        if (n_rows) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->joint_rows), (unsigned long long)n_rows);
        if (n_tok) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->tokens), (unsigned long long)n_tok);
        if (n_forced) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->forced), (unsigned long long)n_forced);
    }
done:
    __syncthreads();
    if (cta == 0)
#pragma unroll 1
        for (int k = tid; k < 65; k += SL_THREADS)
            if (s_hist[k]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->jump_hist[k]), (unsigned long long)s_hist[k]);
    if (tid == 0) {
        if (s_stop) { note_timeout(p.ctrl, 5, cta); set_status(p.ctrl, WIND_ERR_TIMEOUT); }
        if (cta == 0) { p.ctrl->active = 0; p.ctrl->loop_kernel = WIND_LOOP_GRID; }
    }
}

// ---------------------------------------------------------------------------
// The whole decoder inside one SM: a CTA decodes its utterances one after the other.  Everything is fp32 in shared memory
// (bf16 operands converted once), rows padded with zeros to a multiple of four and behind that by four floats per thread of
// a row, so that the 16-byte reads of neighbouring threads fall into different banks.  A row's dot product is cut over up to
// eight neighbouring threads.  A step of the 64-unit fp32 model is bound by reading its 128 KB of gate weights (1000 cycles)
// and by seven block barriers; in the grid form's code with one CTA it took 17000 cycles (8.6 us), 86 KB of instructions
// against an instruction cache of 32 KB: 427 us for an utterance of 44 steps, here 170 us.
// ---------------------------------------------------------------------------
struct SlLocal {
    int nin0, np, nh;                 // E, P, H rounded up to four
    int lg_l, lg_p, lg_j;             // log2 of the threads per row: of the gates, of W_pred, of an output of the joint
    int ld_l0, ld_l1, ld_p, ld_o;     // row pitches in floats
    int w_l0, w_l1, w_l_layer, w_pred, w_out, emb, b_gate, b_pred, b_out, x, h, c, gates, pred, z, key;   // in floats
    long long total;                  // in floats; the offsets mean something only where it fits shared memory
};
__host__ __device__ inline int sl_lg_tpr(int rows) { int l = 0; while (l < 3 && (rows << (l + 1)) <= SL_THREADS) ++l; return l; }
__host__ __device__ inline SlLocal sl_local(int W, int E, int P, int L, int H, int NV, bool emb) {
    SlLocal m{};
    m.nin0 = (E + 3) & ~3; m.np = (P + 3) & ~3; m.nh = (H + 3) & ~3;
    m.lg_l = sl_lg_tpr(4 * P); m.lg_p = sl_lg_tpr(H); m.lg_j = sl_lg_tpr(W * NV);   // (one round over the threads where that is possible)
    m.ld_l0 = m.nin0 + m.np + (4 << m.lg_l); m.ld_l1 = 2 * m.np + (4 << m.lg_l);
    m.ld_p = m.np + (4 << m.lg_p); m.ld_o = m.nh + (4 << m.lg_j);
    long long off = 0;
    auto take = [&](long long n) { const long long o = off; off += (n + 3) & ~3ll; return (int)o; };
    m.w_l0 = take(4ll * P * m.ld_l0);
    m.w_l_layer = 4 * P * m.ld_l1;
    m.w_l1 = take(4ll * P * m.ld_l1 * (L - 1));
    m.w_pred = take((long long)H * m.ld_p);
    m.w_out = take((long long)NV * m.ld_o);
    m.emb = take(emb ? (long long)NV * m.nin0 : 0);
    m.b_gate = take(4ll * L * P);
    m.b_pred = take(H);
    m.b_out = take(NV);
    m.x = take(m.nin0);
    m.h = take((long long)L * m.np);
    m.c = take((long long)L * P);
    m.gates = take(4ll * P);
    m.pred = take(H);
    m.z = take((long long)W * m.nh);
    m.key = take(2ll * W);
    m.total = off;
    return m;
}

// The share `part` of a dot product of two padded rows of n4 floats in shared memory, cut over 1 << lg threads.  One function: the
// hot code has to stay in the instruction cache.
__device__ __noinline__ float sl_local_dot(uint32_t w, uint32_t x, int n4, int part, int lg, float acc) {
    float a1 = 0.f;
    const uint32_t step = 16u << lg, end = w + 4u * (uint32_t)n4;
    w += 16u * (uint32_t)part;
    x += 16u * (uint32_t)part;
#pragma unroll 4
    for (; w < end; w += step, x += step) {
        float a[4], b[4];
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(a[0]), "=f"(a[1]), "=f"(a[2]), "=f"(a[3]) : "r"(w));
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(b[0]), "=f"(b[1]), "=f"(b[2]), "=f"(b[3]) : "r"(x));
        acc = fmaf(a[1], b[1], fmaf(a[0], b[0], acc));
        a1 = fmaf(a[3], b[3], fmaf(a[2], b[2], a1));
    }
    return acc + a1;
}

template <typename TW>
__global__ void __launch_bounds__(SL_THREADS, 1) simt_local_kernel(const SimtLoopParams p, const int emb_here) {
    extern __shared__ __align__(16) float sf[];
    __shared__ int s_tok, s_t, s_more;
    __shared__ int s_hist[65];
    if (p.ctrl->bad_input) return;                 // a length outside [0, T]: nothing is read through it
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const SlLocal M = sl_local(p.W, p.E, p.P, p.L, p.H, p.NV, emb_here != 0);
    // a matrix [rows][n] to column `at` of the padded rows at dst, with zeros up to the next multiple of four; a warp takes 32
    // elements at a time
    // (eight loads under way: a row per warp and no loads ahead took 14 us for 186 KB)
    auto load_rows = [&](float* dst, int ld, int at, const void* src_, int rows, int n) {
        const TW* src = static_cast<const TW*>(src_);
        const int n4 = (n + 3) & ~3, chunks = (n4 + 31) / 32;
#pragma unroll 8
        for (int i = warp; i < rows * chunks; i += SL_WARPS) {
            const int row = i / chunks, k = (i - row * chunks) * 32 + lane;
            const float v = k < n ? (float)__ldg(src + (size_t)row * n + k) : 0.f;
            if (k < n4) dst[row * ld + at + k] = v;
        }
    };
#pragma unroll 1
    for (int l = 0; l < p.L; ++l) {
        float* dst = sf + (l == 0 ? M.w_l0 : M.w_l1 + (l - 1) * M.w_l_layer);
        const int ld = l == 0 ? M.ld_l0 : M.ld_l1, nin = l == 0 ? p.E : p.P;
        load_rows(dst, ld, 0, p.w_ih[l], 4 * p.P, nin);
        load_rows(dst, ld, l == 0 ? M.nin0 : M.np, p.w_hh[l], 4 * p.P, p.P);
#pragma unroll 1
        for (int i = tid; i < 4 * p.P; i += SL_THREADS) sf[M.b_gate + l * 4 * p.P + i] = p.b_ih[l][i] + p.b_hh[l][i];
    }
    load_rows(sf + M.w_pred, M.ld_p, 0, p.w_pred, p.H, p.P);
    load_rows(sf + M.w_out, M.ld_o, 0, p.w_out, p.NV, p.H);
    if (emb_here) load_rows(sf + M.emb, M.nin0, 0, p.emb, p.NV, p.E);
#pragma unroll 1
    for (int i = tid; i < p.H; i += SL_THREADS) sf[M.b_pred + i] = p.b_pred[i];
#pragma unroll 1
    for (int i = tid; i < p.NV; i += SL_THREADS) sf[M.b_out + i] = p.b_out[i];
#pragma unroll 1
    for (int i = tid; i < 65; i += SL_THREADS) s_hist[i] = 0;
    unsigned long long* s_key = reinterpret_cast<unsigned long long*>(sf + M.key);

    auto share_sum = [&](float v, int lg) {
#pragma unroll 1
        for (int o = 1; o < 1 << lg; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
    const TW* enc_proj = static_cast<const TW*>(p.enc_proj);
    long long n_rows = 0, n_tok = 0, n_forced = 0;             // counts (the same in all lanes of warp 0)
    int most_steps = 0;

#pragma unroll 1
    for (int utt = blockIdx.x; utt < p.B; utt += gridDim.x) {
        const int len = min(max(p.enc_len[utt], 0), p.T);
        int cnt = 0, pos = 0, steps = 0, t = 0;                // the utterance's state (warp 0)
        __syncthreads();
#pragma unroll 1
        for (int i = tid; i < p.L * M.np; i += SL_THREADS) sf[M.h + i] = 0.f;
#pragma unroll 1
        for (int i = tid; i < p.L * p.P; i += SL_THREADS) sf[M.c + i] = 0.f;
#pragma unroll 1
        for (int i = tid; i < p.W; i += SL_THREADS) s_key[i] = 0ull;
        if (tid == 0) { s_tok = p.blank; s_t = 0; s_more = len > 0; }
        __syncthreads();
        while (s_more) {
            const int tok = s_tok, n = min(p.W, len - s_t);
            const size_t row0 = (size_t)utt * p.T + s_t;
            // this thread's first element of the window's enc_proj rows, requested before the decoder phases
            const float z_enc = tid < n * p.H ? (float)__ldg(enc_proj + row0 * p.H + tid) : 0.f;
            if (tok >= 0) {
                const float* x = sf + M.emb + tok * M.nin0;
                if (!emb_here) {
#pragma unroll 1
                    for (int k = tid; k < M.nin0; k += SL_THREADS) sf[M.x + k] = k < p.E ? (float)static_cast<const TW*>(p.emb)[(size_t)tok * p.E + k] : 0.f;
                    x = sf + M.x;
                    __syncthreads();
                }
#pragma unroll 1
                for (int l = 0; l < p.L; ++l) {
                    const float* w = sf + (l == 0 ? M.w_l0 : M.w_l1 + (l - 1) * M.w_l_layer);
                    const int ld = l == 0 ? M.ld_l0 : M.ld_l1, n_in = l == 0 ? M.nin0 : M.np, part = tid & ((1 << M.lg_l) - 1);
                    const float* xl = l == 0 ? x : sf + M.h + (l - 1) * M.np;
#pragma unroll 1
                    for (int i = tid; i - lane < 4 * p.P << M.lg_l; i += SL_THREADS) {       // whole warps: threads past the end repeat the last row
                        const int row = min(i >> M.lg_l, 4 * p.P - 1);
                        const float* wr = w + row * ld;
                        float v = sl_local_dot(smem_u32(wr), smem_u32(xl), n_in, part, M.lg_l, 0.f);
                        v = sl_local_dot(smem_u32(wr + n_in), smem_u32(sf + M.h + l * M.np), M.np, part, M.lg_l, v);
                        v = share_sum(v, M.lg_l);
                        if (part == 0) sf[M.gates + row] = v + sf[M.b_gate + l * 4 * p.P + row];
                    }
                    __syncthreads();
#pragma unroll 1
                    for (int j = tid; j < p.P; j += SL_THREADS) {
                        const float* gt = sf + M.gates + j;
                        const float gi = 1.f / (1.f + expf(-gt[0])), gf = 1.f / (1.f + expf(-gt[p.P])), gg = tanhf(gt[2 * p.P]), go = 1.f / (1.f + expf(-gt[3 * p.P]));
                        float* cs = sf + M.c + l * p.P + j;
                        const float cc = cell_update_fc(gf, *cs, gi, gg);
                        *cs = cc;
                        sf[M.h + l * M.np + j] = sl_round<TW>(go * tanhf(cc));
                    }
                    __syncthreads();
                }
                const int part = tid & ((1 << M.lg_p) - 1);
#pragma unroll 1
                for (int i = tid; i - lane < p.H << M.lg_p; i += SL_THREADS) {
                    const int row = min(i >> M.lg_p, p.H - 1);
                    const float v = share_sum(sl_local_dot(smem_u32(sf + M.w_pred + row * M.ld_p), smem_u32(sf + M.h + (p.L - 1) * M.np), M.np, part, M.lg_p, 0.f), M.lg_p);
                    if (part == 0) sf[M.pred + row] = v + sf[M.b_pred + row];
                }
                __syncthreads();
            }
#pragma unroll 1
            for (int i = tid; i < n * M.nh; i += SL_THREADS) {
                const int w = i / M.nh, k = i - w * M.nh;
                float v = 0.f;
                if (k < p.H) {
                    v = (M.nh == p.H && i == tid ? z_enc : (float)enc_proj[(row0 + w) * p.H + k]) + sf[M.pred + k];
                    v = sl_round<TW>(p.act == WIND_ACT_RELU ? fmaxf(v, 0.f) : tanhf(v));
                }
                sf[M.z + i] = v;
            }
            __syncthreads();
            {
                const int part = tid & ((1 << M.lg_j) - 1), outs = n * p.NV;
#pragma unroll 1
                for (int q = tid; q - lane < outs << M.lg_j; q += SL_THREADS) {
                    const int i = min(q >> M.lg_j, outs - 1), w = i / p.NV, v = i - w * p.NV;
                    const float s = share_sum(sl_local_dot(smem_u32(sf + M.w_out + v * M.ld_o), smem_u32(sf + M.z + w * M.nh), M.nh, part, M.lg_j, 0.f), M.lg_j) + sf[M.b_out + v];
                    unsigned long long key = s > -INFINITY ? pack_key(s, (uint32_t)v) : 0ull;
                    // one update of s_key for each window row among the warp's outputs (one or two of them)
                    for (uint32_t left = __ballot_sync(0xffffffffu, key != 0ull); left != 0u; left = __ballot_sync(0xffffffffu, key != 0ull)) {
                        const int wr = __shfl_sync(0xffffffffu, w, __ffs((int)left) - 1);
                        const unsigned long long mine = w == wr ? key : 0ull;
                        const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(mine >> 32));
                        const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(mine >> 32) == hi ? (uint32_t)mine : 0u);
                        if (lane == 0) atomicMax(&s_key[wr], ((unsigned long long)hi << 32) | lo);
                        if (w == wr) key = 0ull;
                    }
                }
            }
            __syncthreads();
            // control (Algorithm 2's branch) by warp 0: a lane looks at a window row and at the row 32 further on
            if (warp == 0) {
                const unsigned long long k0 = lane < n ? s_key[lane] : 0ull, k1 = lane + 32 < n ? s_key[lane + 32] : 0ull;
                uint32_t l0 = key_label(k0), l1 = key_label(k1);
                const bool bad0 = lane < n && (k0 == 0ull || l0 >= (uint32_t)p.NV), bad1 = lane + 32 < n && (k1 == 0ull || l1 >= (uint32_t)p.NV);
                if (bad0 || lane >= n) l0 = (uint32_t)p.blank;
                if (bad1 || lane + 32 >= n) l1 = (uint32_t)p.blank;
                const uint32_t h0 = __ballot_sync(0xffffffffu, (int)l0 != p.blank), h1 = __ballot_sync(0xffffffffu, (int)l1 != p.blank);
                const int first = h0 ? __ffs((int)h0) - 1 : (h1 ? 31 + __ffs((int)h1) : n);
                const bool hit = (h0 | h1) != 0u;
                const int label = (int)__shfl_sync(0xffffffffu, first < 32 ? l0 : l1, first & 31);
                const bool bad = __any_sync(0xffffffffu, (bad0 && lane <= first) || (bad1 && lane + 32 <= first));
                if (first > 0) cnt = 0;
                t += first;
                const int t_emit = t, at = pos;
                const bool emit = hit && pos < p.max_out;
                bool forced = false;
                if (emit) {
                    ++pos;
                    if (++cnt == p.S) { ++t; cnt = 0; forced = true; }
                } else if (hit) {
                    t = len;                                                   // no room for the token: this utterance stops here
                }
                ++steps;
                const bool stuck = steps >= p.step_cap && t < len;
                n_rows += n; n_tok += emit; n_forced += forced;
                if (lane == 0) {
                    s_tok = emit ? label : -1;
                    s_t = t;
                    s_more = t < len && !stuck;
                    s_hist[first] += 1;
                    if (emit) {
                        p.out_tokens[(size_t)utt * p.max_out + at] = label;
                        p.out_frames[(size_t)utt * p.max_out + at] = t_emit;
                    }
                    if (hit && !emit) set_status(p.ctrl, WIND_ERR_OUTPUT_OVERFLOW);
                    if (bad || stuck) set_status(p.ctrl, WIND_ERR_INTERNAL);
                    if (t >= len || stuck) p.out_len[utt] = pos;
                }
                __syncwarp();
#pragma unroll 1
                for (int w = lane; w < n; w += 32) s_key[w] = 0ull;
            }
            __syncthreads();
        }
        most_steps = max(most_steps, steps);
    }
    __syncthreads();
    if (tid == 0) {
        atomicMax(&p.ctrl->step, most_steps);
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->joint_rows), (unsigned long long)n_rows);
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->tokens), (unsigned long long)n_tok);
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->forced), (unsigned long long)n_forced);
        if (blockIdx.x == 0) { p.ctrl->active = 0; p.ctrl->loop_kernel = WIND_LOOP_ONE_SM; }
    }
#pragma unroll 1
    for (int k = tid; k < 65; k += SL_THREADS)
        if (s_hist[k]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->jump_hist[k]), (unsigned long long)s_hist[k]);
}

// ---------------------------------------------------------------------------
// One-layer models of up to 64 units, joint units and labels: the same, with the weights in registers.
//
// A step of simt_local_kernel on the 64-unit model took 5300 cycles: 128 KB of gate weights through shared memory, seven block
// barriers, and every phase's addresses worked out anew.  Here a thread keeps a gate row of W_hh (64 values), a quarter of a row of
// W_pred and of W_out for the whole decode, W_ih and the embedding have become a table of all tokens' input terms in shared memory,
// the four gates of a unit meet by shuffles, and every warp takes the decisions itself: three block barriers in a step that feeds a
// token, two in one that does not.  What is left is issue slots, so few warps are better: with 16 a step takes 3650 cycles (and the
// utterance of 44 steps 132 us in all).
// ---------------------------------------------------------------------------
constexpr int ST_MAX = 64;             // units, embedding, joint units, labels
constexpr int ST_ROWS = 32;            // window rows
constexpr int ST_THREADS = 4 * ST_MAX; // four threads a unit (its gates), a joint unit, a label (quarters of a row)
constexpr int ST_WARPS = ST_THREADS / 32;

// (ACT in the template: with both activations in the code, unrolled, its instructions do not fit the cache)
template <typename TW, int ACT>
__global__ void __launch_bounds__(ST_THREADS, 1) simt_tiny_kernel(const SimtLoopParams p) {
    extern __shared__ __align__(16) float s_table[];               // [NV][4 unit + gate] W_ih emb + b_ih + b_hh
    __shared__ __align__(16) float s_enc[2 * ST_ROWS * ST_MAX];    // enc_proj rows, a ring of 64: this window and the frames the next one may
                                                                   // reach; before that the embedding
    __shared__ __align__(16) float s_z[ACT == WIND_ACT_RELU ? 4 : ST_ROWS * ST_MAX];      // the joint's operand (ReLU: formed in registers)
    __shared__ __align__(16) float s_h[2][ST_MAX];                 // [parity of the updates]
    __shared__ __align__(16) float s_pred[ST_MAX];
    __shared__ unsigned long long s_key[ST_WARPS][ST_ROWS];        // best key of a warp's eight labels per window row
    __shared__ int s_hist[65];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int E = p.E, P = p.P, H = p.H, NV = p.NV;
    const int item = tid >> 2, part = tid & 3;                     // unit and gate; joint unit or label, and quarter of its row
    // n values of a row, 16 bytes at a time where rows allow it (element by element a matrix took 9 us); `in`: there is such a row
    auto load_row = [](float* w, const void* m, size_t row, int n, bool in) {
        constexpr int PIECE = 16 / (int)sizeof(TW);
        const TW* src = static_cast<const TW*>(m) + row * n;
        if (n % PIECE == 0 && reinterpret_cast<uintptr_t>(m) % 16 == 0) {
#pragma unroll
            for (int j = 0; j < ST_MAX; j += PIECE) {
                const uint4 v = in && j < n ? __ldg(reinterpret_cast<const uint4*>(src + j)) : make_uint4(0, 0, 0, 0);
                const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if constexpr (sizeof(TW) == 4) {
                        w[j + k] = __uint_as_float(u[k]);
                    } else {
                        w[j + 2 * k] = __uint_as_float(u[k] << 16);
                        w[j + 2 * k + 1] = __uint_as_float(u[k] & 0xffff0000u);
                    }
            }
        } else {
#pragma unroll
            for (int j = 0; j < ST_MAX; ++j) w[j] = in && j < n ? (float)__ldg(src + j) : 0.f;
        }
    };
    auto dot = [](const float* w, const float* x) {                // x in shared memory, the same for all threads
        float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < ST_MAX; j += 4) {
            const float4 v = *reinterpret_cast<const float4*>(x + j);
            a[0] = fmaf(w[j], v.x, a[0]); a[1] = fmaf(w[j + 1], v.y, a[1]); a[2] = fmaf(w[j + 2], v.z, a[2]); a[3] = fmaf(w[j + 3], v.w, a[3]);
        }
        return (a[0] + a[1]) + (a[2] + a[3]);
    };

    // ---- weights; table of the input terms ----
    const size_t g_row = (size_t)part * P + min(item, P - 1);
    float w[ST_MAX];
    {
        float e[ST_MAX * ST_MAX / ST_THREADS];                      // the embedding of all tokens
#pragma unroll
        for (int i = 0; i < ST_MAX * ST_MAX / ST_THREADS; ++i) {
            const int v = (tid >> 6) + ST_THREADS / 64 * i, k = tid & 63;
            e[i] = v < NV && k < E ? (float)__ldg(static_cast<const TW*>(p.emb) + (size_t)v * E + k) : 0.f;
        }
        load_row(w, p.w_ih[0], g_row, E, item < P);
        const float bias = item < P ? p.b_ih[0][g_row] + p.b_hh[0][g_row] : 0.f;
#pragma unroll
        for (int i = 0; i < ST_MAX * ST_MAX / ST_THREADS; ++i) s_enc[tid + ST_THREADS * i] = e[i];
        __syncthreads();
#pragma unroll 2
        for (int v = 0; v < NV; ++v) s_table[v * (4 * ST_MAX) + tid] = dot(w, s_enc + v * ST_MAX) + bias;
    }
    load_row(w, p.w_hh[0], g_row, P, item < P);
    // a quarter of a row: four pieces of four values, 16 apart, so that the quarters' pieces lie side by side
    float wp[16], wo[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int k = (j >> 2) * 16 + part * 4 + (j & 3);
        wp[j] = item < H && k < P ? (float)__ldg(static_cast<const TW*>(p.w_pred) + (size_t)item * P + k) : 0.f;
        wo[j] = item < NV && k < H ? (float)__ldg(static_cast<const TW*>(p.w_out) + (size_t)item * H + k) : 0.f;
    }
    const float b_pred = item < H ? p.b_pred[item] : 0.f, b_out = item < NV ? p.b_out[item] : 0.f;
#pragma unroll 1
    for (int i = tid; i < 65; i += ST_THREADS) s_hist[i] = 0;

    // (up to here, 11 us, under the encoder projection: the weights are the caller's)
    wait_for_previous();                           // (what follows reads nothing by __ldg)
    if (p.ctrl->bad_input) return;                 // a length outside [0, T]: nothing is read through it
    const int warps = (NV + 7) / 8;                                 // that have labels
    s_key[warp][lane] = 0ull;
    long long n_rows = 0, n_tok = 0, n_forced = 0;
    int most_steps = 0;
#pragma unroll 1
    for (int utt = blockIdx.x; utt < p.B; utt += gridDim.x) {
        const int len = min(max(p.enc_len[utt], 0), p.T);
        // the utterance's state, the same in every thread
        int t = 0, tok = p.blank, cnt = 0, pos = 0, steps = 0;
        uint32_t par = 0u;
        float c = 0.f;                                              // of unit `item`
        // what the last step decided: recorded by the last warp when the others are at the joint
        int r_first = -1, r_label = 0, r_t = 0, r_pos = 0;
        bool r_emit = false, r_overflow = false, r_bad = false;
        auto record = [&]() {
            if (lane == 0 && r_first >= 0) {
                s_hist[r_first] += 1;
                if (r_emit) {
                    p.out_tokens[(size_t)utt * p.max_out + r_pos] = r_label;
                    p.out_frames[(size_t)utt * p.max_out + r_pos] = r_t;
                }
                if (r_overflow) set_status(p.ctrl, WIND_ERR_OUTPUT_OVERFLOW);
                if (r_bad) set_status(p.ctrl, WIND_ERR_INTERNAL);
            }
        };
        const TW* enc = static_cast<const TW*>(p.enc_proj) + (size_t)utt * p.T * H;
        const int k_enc = tid & 63;
        // (an ordinary load: the kernel before this one may still have been writing enc_proj when this one began, and __ldg is only for
        // what nobody writes in a kernel's lifetime)
        auto frame = [&](int f) { return k_enc < H ? (float)enc[(size_t)f * H + k_enc] : 0.f; };
        int have = min(len, 2 * p.W);                               // frames that are in the ring or on their way
        __syncthreads();
        if (tid < ST_MAX) s_h[0][tid] = 0.f;
#pragma unroll 4
        for (int f = tid >> 6; f < have; f += ST_THREADS / 64) s_enc[f * ST_MAX + k_enc] = frame(f);
        __syncthreads();
#pragma unroll 1
        while (t < len) {
            const int n = min(p.W, len - t);
            // up to eight more frames, for the next step (a frame comes from L2: 900 cycles)
            constexpr int AT_ONCE = 8 * 64 / ST_THREADS;
            const int f0 = have + (tid >> 6);
            have = min(len, t + 2 * p.W);
            float e[AT_ONCE];
#pragma unroll
            for (int i = 0; i < AT_ONCE; ++i) e[i] = f0 + ST_THREADS / 64 * i < have ? frame(f0 + ST_THREADS / 64 * i) : 0.f;
            if (tok >= 0) {
                // ---- gates and cell: lanes 4 u + g hold gate g of a unit ----
                float s = dot(w, s_h[par]) + s_table[tok * (4 * ST_MAX) + tid];
                s = part == 2 ? tanhf(s) : 1.f / (1.f + expf(-s));
                const int base = lane & 28;
                const float gi = __shfl_sync(0xffffffffu, s, base), gf = __shfl_sync(0xffffffffu, s, base + 1), gg = __shfl_sync(0xffffffffu, s, base + 2),
                            go = __shfl_sync(0xffffffffu, s, base + 3);
                c = cell_update_fc(gf, c, gi, gg);
                const float h = sl_round<TW>(go * tanhf(c));
                par ^= 1u;
                if (part == 0) s_h[par][item] = h;                  // (units past P: zero weights, and W_pred has none there)
            }
            auto quarter = [&](const float* x, float* v) {
#pragma unroll
                for (int j = 0; j < 4; ++j) *reinterpret_cast<float4*>(v + 4 * j) = *reinterpret_cast<const float4*>(x + 16 * j + part * 4);
            };
            if (tok >= 0) {
                __syncthreads();
                // ---- pred_proj ----
                float x[16], a[4] = {0.f, 0.f, 0.f, 0.f};
                quarter(s_h[par], x);
#pragma unroll
                for (int j = 0; j < 16; ++j) a[j & 3] = fmaf(wp[j], x[j], a[j & 3]);
                float s = (a[0] + a[1]) + (a[2] + a[3]);
                s += __shfl_xor_sync(0xffffffffu, s, 1);
                s += __shfl_xor_sync(0xffffffffu, s, 2);
                if (part == 0) s_pred[item] = s + b_pred;
            }
            __syncthreads();
            // ---- joint ----
            if constexpr (ACT != WIND_ACT_RELU) {                   // the operand in a loop of its own: one tanh in the code
#pragma unroll 1
                for (int i = tid; i < n * ST_MAX; i += ST_THREADS) s_z[i] = sl_round<TW>(tanhf(s_enc[((t + (i >> 6)) & 63) * ST_MAX + (i & 63)] + s_pred[i & 63]));
                __syncthreads();
            }
            if (warp == ST_WARPS - 1) record();
            if (warp < warps) {
                float g[16];
                quarter(s_pred, g);
#pragma unroll 1
                for (int r0 = 0; r0 < n; r0 += 4) {                 // four window rows at a time (behind the last: nobody looks)
                    float a[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        float x[16], b[4] = {0.f, 0.f, 0.f, 0.f};
                        quarter(ACT == WIND_ACT_RELU ? s_enc + ((t + r0 + r) & 63) * ST_MAX : s_z + (r0 + r) * ST_MAX, x);
#pragma unroll
                        for (int j = 0; j < 16; ++j) b[j & 3] = fmaf(wo[j], ACT == WIND_ACT_RELU ? sl_round<TW>(fmaxf(x[j] + g[j], 0.f)) : x[j], b[j & 3]);
                        a[r] = (b[0] + b[1]) + (b[2] + b[3]);
                    }
                    // lane 4 v + r: label v's logit of row r
#pragma unroll
                    for (int o = 2; o >= 1; o >>= 1) {
                        const bool up = (part & o) != 0;
#pragma unroll
                        for (int r = 0; r < o; ++r) {
                            const float send = up ? a[r] : a[r + o], keep = up ? a[r + o] : a[r];
                            a[r] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                        }
                    }
                    // the best of the warp's eight labels, the lowest of equals
                    const float v = item < NV ? a[0] + b_out : -INFINITY;
                    float m = v;
#pragma unroll
                    for (int o = 4; o < 32; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                    const uint32_t equal = __ballot_sync(0xffffffffu, v == m) & (0x11111111u << part);
                    if (lane < 4) s_key[warp][r0 + part] = m > -INFINITY ? pack_key(m, (uint32_t)(8 * warp + ((__ffs((int)equal) - 1) >> 2))) : 0ull;
                }
            }
            // the frames requested above, behind those that this step looks at (the rest of them, with wide windows: now)
#pragma unroll
            for (int i = 0; i < AT_ONCE; ++i)
                if (f0 + ST_THREADS / 64 * i < have) s_enc[((f0 + ST_THREADS / 64 * i) & 63) * ST_MAX + k_enc] = e[i];
#pragma unroll 1
            for (int f = f0 + 8; f < have; f += ST_THREADS / 64) s_enc[(f & 63) * ST_MAX + k_enc] = frame(f);
            __syncthreads();
            // ---- control (Algorithm 2's branch), by every warp ----
            unsigned long long key = 0ull;                          // lane = window row; warps without labels have left 0
#pragma unroll
            for (int i = 0; i < ST_WARPS; ++i) key = max(key, s_key[i][lane]);
            uint32_t label = key_label(key);
            const bool broken = lane < n && (key == 0ull || label >= (uint32_t)NV);
            if (broken || lane >= n) label = (uint32_t)p.blank;
            const uint32_t hit = __ballot_sync(0xffffffffu, (int)label != p.blank);
            const int first = hit ? __ffs((int)hit) - 1 : n, best = (int)__shfl_sync(0xffffffffu, label, first & 31);
            const bool emit = hit && pos < p.max_out;
            if (first > 0) cnt = 0;
            t += first;
            const int t_emit = t, at = pos;
            bool forced = false;
            if (emit) {
                ++pos;
                if (++cnt == p.S) { ++t; cnt = 0; forced = true; }
            } else if (hit) {
                t = len;                                            // no room for the token: this utterance stops here
            }
            tok = emit ? best : -1;
            ++steps;
            const bool stuck = steps >= p.step_cap && t < len;
            if (stuck) t = len;
            n_rows += n; n_tok += emit; n_forced += forced;
            r_bad = __any_sync(0xffffffffu, broken && lane <= first) || stuck;
            r_first = first; r_label = best; r_t = t_emit; r_pos = at; r_emit = emit; r_overflow = hit && !emit;
        }
        if (warp == ST_WARPS - 1) {
            record();
            if (lane == 0 && len > 0) p.out_len[utt] = pos;
        }
        most_steps = max(most_steps, steps);
    }
    __syncthreads();
    if (tid == 0) {
        atomicMax(&p.ctrl->step, most_steps);
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->joint_rows), (unsigned long long)n_rows);
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->tokens), (unsigned long long)n_tok);
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->forced), (unsigned long long)n_forced);
        if (blockIdx.x == 0) { p.ctrl->active = 0; p.ctrl->loop_kernel = WIND_LOOP_ONE_SM; }
    }
#pragma unroll 1
    for (int k = tid; k < 65; k += ST_THREADS)
        if (s_hist[k]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->jump_hist[k]), (unsigned long long)s_hist[k]);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
template <typename TW>
static const void* sl_fn(bool resident) {
    return resident ? (const void*)simt_grid_kernel<TW, true> : (const void*)simt_grid_kernel<TW, false>;
}

template <typename TW>
static const void* st_fn(int act) {
    return act == WIND_ACT_RELU ? (const void*)simt_tiny_kernel<TW, WIND_ACT_RELU> : (const void*)simt_tiny_kernel<TW, WIND_ACT_TANH>;
}

static std::mutex g_sl_mutex;
static int g_sl_optin[64] = {};        // opt-in shared memory per block, 0: not asked yet

// opt-in shared memory of the current device, granted to every kernel of this file once
static cudaError_t sl_device(int* optin) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_sl_mutex);
    if (!g_sl_optin[dev]) {
        int n = 0;
        if ((e = cudaDeviceGetAttribute(&n, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
        const int dyn = n - 4096;      // the kernels' static shared memory stays below 4 KB
        for (const void* fn : {sl_fn<float>(false), sl_fn<float>(true), sl_fn<__nv_bfloat16>(false), sl_fn<__nv_bfloat16>(true),
                               (const void*)simt_local_kernel<float>, (const void*)simt_local_kernel<__nv_bfloat16>})
            if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn)) != cudaSuccess) return e;
        // (and static: 19.5 KB with ReLU, 27.7 with tanh; a block may have 227 in all)
        for (const void* fn : {st_fn<float>(WIND_ACT_RELU), st_fn<float>(WIND_ACT_TANH), st_fn<__nv_bfloat16>(WIND_ACT_RELU), st_fn<__nv_bfloat16>(WIND_ACT_TANH)})
            if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 16 * ST_MAX * ST_MAX)) != cudaSuccess) return e;
        g_sl_optin[dev] = n;
    }
    *optin = g_sl_optin[dev];
    return cudaSuccess;
}

// Which form of the kernel a decode takes; false: none (window-based decoding, batches whose state does not fit)
static bool sl_plan(const Call& c, bool* local, bool* resident, bool* emb, size_t* smem, int* grid, SlPlan* plan) {
    if (c.mode != WIND_MODE_FIRST_NONBLANK || c.B > SL_MAX_B) return false;
    int optin = 0, sms = 0;
    if (sl_device(&optin) != cudaSuccess || loop_sm_count(&sms) != cudaSuccess) { cudaGetLastError(); return false; }
    const wind_model_t& m = c.m;
    const size_t budget = (size_t)optin - 4096;
    const size_t one_sm = sizeof(float) * (size_t)sl_local(c.W, m.E, m.P, m.L, m.H, m.V + 1, false).total;
    if (one_sm <= budget) {
        *local = *resident = true;
        *smem = sizeof(float) * (size_t)sl_local(c.W, m.E, m.P, m.L, m.H, m.V + 1, true).total;
        *emb = *smem <= budget;        // the embedding table too where there is room, else its rows come from L2
        if (!*emb) *smem = one_sm;
        *grid = c.B < sms ? c.B : sms;
        return true;
    }
    *local = *emb = false;
    *grid = sms;
    for (bool res : {true, false}) {
        *resident = res;
        *plan = m.dtype == WIND_DT_BF16 ? sl_plan_grid<__nv_bfloat16>(sms, c.B, c.W, m.E, m.P, m.L, m.H, m.V + 1, res, budget)
                                        : sl_plan_grid<float>(sms, c.B, c.W, m.E, m.P, m.L, m.H, m.V + 1, res, budget);
        *smem = plan->total;
        if (plan->total <= budget) return true;
    }
    return false;
}

bool simt_loop_supported(const Call& c) {
    bool local, resident, emb;
    size_t smem;
    int grid;
    SlPlan plan;
    return sl_plan(c, &local, &resident, &emb, &smem, &grid, &plan);
}

cudaError_t simt_loop(const Call& c) {
    bool local, resident, emb;
    size_t smem;
    int grid;
    SlPlan plan;
    if (!sl_plan(c, &local, &resident, &emb, &smem, &grid, &plan)) return cudaErrorNotSupported;
    const wind_model_t& m = c.m;
    SimtLoopParams p{};
    p.ctrl = c.ctrl();
    p.B = c.B; p.T = c.T; p.W = c.W; p.S = c.S; p.max_out = c.max_out;
    p.E = m.E; p.P = m.P; p.L = m.L; p.H = m.H; p.NV = m.V + 1; p.blank = m.blank_id; p.act = m.act;
    const long long cap = (long long)c.T * (c.S + 1) + 2;
    p.step_cap = cap > 0x7fffffff ? 0x7fffffff : (int)cap;
    p.extra_arrivals = loop_extra_arrivals();
    p.emb = m.emb; p.w_pred = m.w_pred; p.b_pred = m.b_pred; p.w_out = m.w_out; p.b_out = m.b_out;
    for (int l = 0; l < m.L; ++l) {
        p.w_ih[l] = c.w_ih[l]; p.w_hh[l] = c.w_hh[l]; p.b_ih[l] = c.b_ih[l]; p.b_hh[l] = c.b_hh[l];
    }
    p.enc_proj = c.enc_proj(); p.enc_len = c.enc_len;
    p.h = c.h(0); p.c = c.c(); p.pred = c.pred_proj(); p.keys = c.keys();
    p.out_tokens = c.out_tokens; p.out_frames = c.out_frames; p.out_len = c.out_len;
    if (local && m.L == 1 && m.E <= ST_MAX && m.P <= ST_MAX && m.H <= ST_MAX && p.NV <= ST_MAX && c.W <= ST_ROWS) {
        void* args[1] = {(void*)&p};
        return launch_overlapped(m.dtype == WIND_DT_BF16 ? st_fn<__nv_bfloat16>(m.act) : st_fn<float>(m.act),
                                 dim3((unsigned)grid), dim3(ST_THREADS), args, (size_t)p.NV * 4 * ST_MAX * sizeof(float), c.stream);
    }
    if (local) {
        int emb_here = emb;
        void* args[2] = {(void*)&p, (void*)&emb_here};
        return cudaLaunchKernel(m.dtype == WIND_DT_BF16 ? (const void*)simt_local_kernel<__nv_bfloat16> : (const void*)simt_local_kernel<float>,
                                dim3((unsigned)grid), dim3(SL_THREADS), args, smem, c.stream);
    }
    const void* fn = m.dtype == WIND_DT_BF16 ? sl_fn<__nv_bfloat16>(resident) : sl_fn<float>(resident);
    void* args[2] = {(void*)&p, (void*)&plan};
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)grid), dim3(SL_THREADS), args, smem, c.stream);
}

}  // namespace wind
