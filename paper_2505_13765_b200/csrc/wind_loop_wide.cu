// The decoding loop of bf16 models with one LSTM layer whose vocabulary does not fit the other resident kernels (8193 labels and
// 1024 joint units: W_out has 65 tiles of 256 KB).
//
// loop_kernel streamed all of it every lock step: 768 KB of W_out and z through each SM for the joint and 384 KB for the decoder
// (its 128-row state tile mostly padding), 34 us a step at 32 utterances x 16 window rows; here 15.  Here every weight stays on the chip,
// because each CTA has one role only:
//   L   a W_hh tile (4 gates x 16 units, shared memory); its GEMM for the next step runs behind the projection phase
//   J   one vocabulary tile: the first 768 of K in tensor memory, the rest in shared memory; z comes through a ring
//   P   a W_pred tile (64 joint units, shared memory); builds z for all window rows
//   C   one CTA records (tokens, frames, counters) and clears the keys
// Every CTA takes the decisions of all utterances from the window's keys itself, so no decision travels; the cell state and the
// hidden state stay in the registers of the thread that updates them.
//
// What bounds a step then is z: a J CTA brings every window row into its shared memory and multiplies it from there (128 rows x 1024:
// 4600 cycles of shared-memory bandwidth, 2048 each for the copy and for the MMAs, 512 for the part of W_out that lies there).  So a lock
// step evaluates at most 128 rows: with more than 128 / W utterances alive a window is evaluated in parts, and one whose first
// part holds a label needs no second.  Where labels are so rare that the second part would often follow, 256 rows (wide_rows).
// Utterances sit in slots by length, so that the ones still decoding are a prefix and the window widens as they get fewer.
// Counters are kept per window, so they do not show the parts.
//
// Phases, behind grid barriers (1.3 us each): L control + cell update; P projection + z; J joint.
#include <mutex>

#include "wind_loop_dev.cuh"

namespace wind {

constexpr int WD_THREADS = 320;            // TMA warp, MMA warp, eight epilogue warps
constexpr int WD_EPI = 256;
constexpr int WD_NJ = 128;                 // window rows of a row group (an MMA of 64 rows takes as long as one of 128)
constexpr int WD_ROWS = 256;               // most window rows of a step
constexpr int WD_SLOTS = 64;               // most utterances
constexpr int WD_MAX_STAGES = 8;
// K blocks of a stage of z (half of them with more than 64 rows, so that a stage is 64 KB at most).  A stage costs its threads 300 to
// 450 cycles of waiting, issue and commit whatever its size: with one block each the joint of a step took 7.8 us at 32 utterances and
// 6.2 with 16 rows; with 2 / 4 blocks 6.0 and 4.2, with 4 / 8 5.9 and 3.9.
constexpr int WD_UNIT = 8;
// Most K blocks of W_out in tensor memory: 384 columns, an accumulator takes the rest (two of them up to 8 blocks).  What that leaves of
// shared memory is the ring for z: nine blocks of 128 rows.
constexpr int WD_TM_BLOCKS = 12;
constexpr uint32_t WD_Z_STAGE = WD_NJ * BK * 2;

// Window rows of a slot in the coming step.  `blanks` and `labels` are recent sums over all utterances: rows found blank, and
// rows with a label.  With blank probability q a window of w rows takes an utterance (1 - q^w) / (1 - q) rows further; a step of
// 256 rows costs 1.25 times one of 128, and q is an estimate, so it has to bring a little more: 1.35 times.  Measured with 5, 10,
// 15, 20, 30, 40 and 60 % of the frames carrying a label, 12 to 32 utterances, W = 8 to 16 (42 batches): 1.35 is within 1.7 % of the
// best of 1.25, 1.35, 1.5 and 1.7 but for one (12 utterances, 10 %: 4.1 %), 0.4 % on the average; 1.25 0.6 % (40 %, 32 x 16: 6.19 ms
// against 5.98), 1.5 1.2 % (5 %, 32 x 8: 2.59 against 2.45), 256 rows throughout 5 % (most at 60 %: 24 %), 128 throughout 4 % (5 %: 23 %).
__device__ __forceinline__ int wide_rows(int W, int live, float blanks, float labels) {
    const int n = max(live, 1), narrow = min(W, WD_NJ / n), wide = min(W, WD_ROWS / n);
    if (narrow == wide) return narrow;
    const float q = blanks / (blanks + labels + 1e-3f);
    float reach = 1.f, reach_narrow = 1.f;
    for (int w = 1; w <= wide; ++w) {
        reach *= q;
        if (w == narrow) reach_narrow = reach;
    }
    return 1.f - reach > 1.35f * (1.f - reach_narrow) ? wide : narrow;
}

struct WdMaps {
    CUtensorMap w_hh;      // [4P, P], box 16 rows x 1 block
    CUtensorMap w_pred;    // [H, P], box 64 rows x 1 block
    CUtensorMap w_out;     // [V+1, H], box 128 rows x 1 block
    // z and the state lie in blocks of 64 columns, so that a box is one contiguous piece: with rows of H columns all CTAs read the
    // same few L2 slices at a time
    CUtensorMap z[4];      // [H / 64][WD_ROWS][64], box 16, 32, 64 or 128 rows x 8, 8, 8 or 4 blocks
    CUtensorMap hb[2][2];  // [parity] [P / 64][nl][64], box all blocks of 16 or of nl rows
};

struct WdPlan {
    int n_l, n_j, n_p, grid;              // CTAs of each role; recording CTA behind J
    int nl, stages;
    uint32_t smem;
};

struct WdParams {
    Ctrl* ctrl;
    int B, T, W, S, max_out, H, P, NV, blank, act, step_cap, extra_arrivals;
    int n_l, n_j, n_p, nl, stages, kb_h, kb_p;
    const int32_t* enc_len;
    unsigned long long* keys;             // [2][WD_ROWS]
    int32_t* out_tokens;
    int32_t* out_frames;
    int32_t* out_len;
    __nv_bfloat16* hb[2];                 // [P / 64][nl][64]
    __nv_bfloat16* z;                     // [H / 64][WD_ROWS][64]
    const __nv_bfloat16* enc_proj;
    const float* g0;                      // [V+1][4P]
    const float* b_pred;
    const float* b_out;
    const __nv_bfloat16* w_out;
};

// 32 lanes x 32 columns of an accumulator, rows (lanes) spread over the warp as mma.sync spreads them: v[16 h + 4 x + 2 k + j] is lane
// 16 h + 8 k + lane / 4, column 8 x + 2 (lane % 4) + j.
__device__ __forceinline__ void wide_tmem_ld(uint32_t ta, float* v) {
    uint32_t r[32];
#pragma unroll
    for (int h = 0; h < 2; ++h)
        asm volatile(
            "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(r[16 * h]), "=r"(r[16 * h + 1]), "=r"(r[16 * h + 2]), "=r"(r[16 * h + 3]), "=r"(r[16 * h + 4]), "=r"(r[16 * h + 5]),
              "=r"(r[16 * h + 6]), "=r"(r[16 * h + 7]), "=r"(r[16 * h + 8]), "=r"(r[16 * h + 9]), "=r"(r[16 * h + 10]), "=r"(r[16 * h + 11]),
              "=r"(r[16 * h + 12]), "=r"(r[16 * h + 13]), "=r"(r[16 * h + 14]), "=r"(r[16 * h + 15])
            : "r"(ta + ((uint32_t)(16 * h) << 16))
            : "memory");
    // (the registers pass through the wait, so that nothing reads them before it)
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        asm volatile("" : "+r"(r[i]));
        v[i] = __uint_as_float(r[i]);
    }
}
// Columns [0, 2 HALF) of a lane and of the lane WITH away become HALF of either, with the better (logit, label) of the two.
template <int HALF, int WITH>
__device__ __forceinline__ void wide_exchange(float* v, int* id, int lane) {
    const bool up = (lane & WITH) != 0;
#pragma unroll
    for (int c = 0; c < HALF; ++c) {
        const float sv = up ? v[c] : v[c + HALF], kv = up ? v[c + HALF] : v[c];
        const int si = up ? id[c] : id[c + HALF], ki = up ? id[c + HALF] : id[c];
        const float rv = __shfl_xor_sync(0xffffffffu, sv, WITH);
        const int ri = __shfl_xor_sync(0xffffffffu, si, WITH);
        const bool take = (rv > kv) || (rv == kv && ri < ki);   // lowest label on equal logits
        v[c] = take ? rv : kv;
        id[c] = take ? ri : ki;
    }
}

__global__ void __launch_bounds__(WD_THREADS, 1) wide_kernel(const __grid_constant__ WdMaps M, const WdParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar[WD_MAX_STAGES], empty_bar[WD_MAX_STAGES], acc_bar[2], acc_free[2], stat_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort;
    __shared__ int s_live[2], s_blanks[2], s_labels[2];      // slots in use are [0, larger of the two); rows of the last step
    __shared__ int s_window;
    __shared__ int s_utt[WD_SLOTS], s_len[WD_SLOTS];
    __shared__ int s_tok[WD_SLOTS], s_row[WD_SLOTS], s_left[WD_SLOTS];   // this step: token (-1 none), enc_proj row of the next frame, frames left
    __shared__ int s_hist[65];
    __shared__ unsigned long long s_part[4 * WD_NJ];        // J: winners of the four lane quadrants

    const int warp = uniform_warp_index(), lane = threadIdx.x & 31;
    const int cta = blockIdx.x, G = gridDim.x;
    if (p.ctrl->bad_input) return;
    const bool is_l = cta < p.n_l, is_j = !is_l && cta < p.n_l + p.n_j, is_c = cta == p.n_l + p.n_j, is_p = cta > p.n_l + p.n_j;
    const int vt = cta - p.n_l, ut = cta, ht = cta - (p.n_l + p.n_j + 1);
    uint8_t* smem = align_smem_1024(smem_raw);
    const int kb_t = min(p.kb_h, WD_TM_BLOCKS);              // J: K blocks in tensor memory
    const uint32_t a_bytes = is_j ? (uint32_t)(p.kb_h - kb_t) * 128u * BK * 2u : (uint32_t)p.kb_p * 64u * BK * 2u;
    uint8_t* ring = smem + a_bytes;                          // J: stages of z; L, P: the state box
    float* stage = reinterpret_cast<float*>(ring + (uint32_t)p.nl * (uint32_t)p.P * 2u);   // L, P: behind the state box
    const int e = threadIdx.x - 64, sub = (warp - 2) >> 2, q = warp & 3;
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;

    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int s = 0; s < WD_MAX_STAGES; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        for (int k = 0; k < 2; ++k) { mbar_init(&acc_bar[k], 1); mbar_init(&acc_free[k], WD_EPI / 32); }
        mbar_init(&stat_bar, 1);
        fence_barrier_init();
    }
    for (int k = threadIdx.x; k < 65; k += WD_THREADS) s_hist[k] = 0;
    if (warp == 1) tmem_alloc(&tmem_slot, LOOP_TMEM_COLS);
    // slots by length, longest first (equal lengths in the caller's order)
    if (threadIdx.x < WD_SLOTS) { s_utt[threadIdx.x] = 0; s_len[threadIdx.x] = 0; }
    __syncthreads();
    for (int b = threadIdx.x; b < p.B; b += WD_THREADS) {
        const int mine = min(max(p.enc_len[b], 0), p.T);
        int rank = 0;
        for (int j = 0; j < p.B; ++j) {
            const int other = min(max(p.enc_len[j], 0), p.T);
            rank += other > mine || (other == mine && j < b);
        }
        s_utt[rank] = b;
        s_len[rank] = mine;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);
    const uint32_t tm_acc = is_j ? tmem + (uint32_t)kb_t * (BK / 2) : tmem;      // J: behind W_out's blocks
    const uint32_t two = (uint32_t)kb_t * (BK / 2) + 2 * WD_NJ <= LOOP_TMEM_COLS; // J: accumulators: row group n has number n & two

    // ---- weights ----
    const bool tile = !is_c && a_bytes > 0u;
    if (threadIdx.x == 0 && tile) {
        mbar_expect_tx(&stat_bar, a_bytes);
        if (is_l) {
            for (int kb = 0; kb < p.kb_p; ++kb)
                for (int g = 0; g < 4; ++g) tma_load_3d(smem + (kb * 64 + g * 16) * BK * 2, &M.w_hh, 0, g * p.P + ut * 16, kb, &stat_bar);
        } else if (is_p) {
            for (int kb = 0; kb < p.kb_p; ++kb) tma_load_3d(smem + kb * 64 * BK * 2, &M.w_pred, 0, ht * 64, kb, &stat_bar);
        } else {
            for (int kb = kb_t; kb < p.kb_h; ++kb) tma_load_3d(smem + (kb - kb_t) * 128 * BK * 2, &M.w_out, 0, vt * 128, kb, &stat_bar);
        }
    }
    if (is_j && warp >= 2 && warp < 6) {
        // tensor memory, lane = vocabulary entry, 32-bit column j = W_out[v, 2j], W_out[v, 2j + 1]
        const int v = vt * 128 + q * 32 + lane;
        const uint4* src = reinterpret_cast<const uint4*>(p.w_out + (size_t)(v < p.NV ? v : 0) * p.H);
        for (int c0 = 0; c0 < kb_t * (BK / 2); c0 += 16) {
            uint32_t r[16];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint4 x = v < p.NV ? src[c0 / 4 + j] : make_uint4(0, 0, 0, 0);
                r[4 * j] = x.x; r[4 * j + 1] = x.y; r[4 * j + 2] = x.z; r[4 * j + 3] = x.w;
            }
            tmem_st16(tmem + lane_off + (uint32_t)c0, r);
        }
        tmem_st_wait();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1 && tile) mbar_wait_warp(&stat_bar, 0, &s_abort);

    // ---- grid barrier ----
    uint32_t epoch = 0;
    long long clk_last = 0, cyc[3] = {0, 0, 0};
    unsigned long long ns0 = 0;
    if (cta == 0 && threadIdx.x == 0) { clk_last = clock64(); ns0 = globaltimer_ns(); }
    auto grid_sync = [&](int phase_kind) -> bool {
        __syncthreads();
        if (threadIdx.x == 0) {
            epoch += (uint32_t)(G + p.extra_arrivals);
            if (s_abort) {
                atomicExch(&p.ctrl->abort, 1);
            } else {
                __threadfence();
                atomicAdd(&p.ctrl->bar, 1u);
                unsigned long long t0 = 0;
                for (uint32_t it = 1;; ++it) {
                    if ((int32_t)(ld_acquire_u32(&p.ctrl->bar) - epoch) >= 0) break;
                    if ((it & 63u) == 0u) {
                        if (ld_volatile_i32(&p.ctrl->abort)) { s_abort = 2; break; }
                        const unsigned long long now = globaltimer_ns();
                        if (t0 == 0) t0 = now;
                        else if (now - t0 > kWaitLimitNs) { s_abort = 1; note_timeout(p.ctrl, 3, cta); atomicExch(&p.ctrl->abort, 1); break; }
                    }
                }
            }
            if (cta == 0) {
                const long long now = clock64();
                cyc[phase_kind] += now - clk_last;
                clk_last = now;
            }
        }
        __syncthreads();
        return s_abort == 0;
    };
    // ---- control state of utterance `slot` (warps 2 and 3, a lane each, the same in every CTA) ----
    const int slot = 32 * (warp - 2) + lane;
    const bool ctl = (warp == 2 || warp == 3) && slot < p.B;
    const int c_len = ctl ? s_len[slot] : 0, c_utt = ctl ? s_utt[slot] : 0;
    int c_t = 0, c_cnt = 0, c_pos = 0, c_off = 0, c_wins = 0;      // c_off: rows of the window in hand already found blank
    long long n_rows = 0, n_tok = 0, n_forced = 0;
    // ---- state of the (utterance, unit) pairs of an L thread ----
    float cell[4] = {0.f, 0.f, 0.f, 0.f};
    uint32_t hid[4] = {0u, 0u, 0u, 0u};                            // bf16
    uint4 ev[8];                                                   // P: enc_proj chunks of this thread's rows of the next window
    int kinds = 0, bw[8], bw_wi = -1;                              // 2 bits per row: 0 not written, 1 zeros, 2 a frame
    const float p_bias = is_p && e >= 0 ? p.b_pred[ht * 64 + 16 * q + (lane & 15)] : 0.f;
    float j_bias[4];                                               // J: of the thread's four vocabulary entries, lane / 4 + 8 k of its quadrant
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int v = vt * 128 + q * 32 + (lane >> 2) + 8 * k;
        j_bias[k] = is_j && e >= 0 && v < p.NV ? p.b_out[v] : 0.f;
    }

    // the CTAs start at different K blocks: not all of them on the same lines of L2
    const int kb_first = is_j ? vt % ((p.kb_h + WD_UNIT - 1) / WD_UNIT) * WD_UNIT : 0;
    uint32_t phases = warp == 0 ? 0xFFu : 0u;   // J, TMA and MMA warp: parity to wait for at each stage's barrier
    uint32_t gemm_n = 0;                  // L, P: GEMMs so far; J: row groups so far
    int wi = 0, live = 0;                 // window and slots of the joint phase just done, then of the next one
    float blanks = 0.f, labels = 0.f;     // of the last steps, fading (the same in every CTA)
    int exit_status = 0;

    // TMA and MMA of a 64-row weight tile with the state hb[par] (L and P)
    auto state_gemm = [&](int par) {
        const int n_cols = live <= 16 ? 16 : p.nl;
        const uint32_t block = (uint32_t)n_cols * BK * 2u;
        // (one box and one wait: in four, so that the first MMAs start before the last rows are there, the phase took 4.7 us instead of 4.4)
        if (warp == 0) {
            fence_proxy_async_all();
            if (elect_one()) {
                mbar_expect_tx(&full_bar[0], (uint32_t)p.kb_p * block);
                tma_load_3d(ring, &M.hb[par][n_cols != 16], 0, 0, 0, &full_bar[0]);
            }
            __syncwarp();
        } else if (warp == 1) {
            tc_fence_after();
            const uint32_t idesc = idesc_bf16(64, n_cols);
            if (mbar_wait_warp(&full_bar[0], gemm_n & 1u, &s_abort)) {
                tc_fence_after();
                if (elect_one()) {
                    for (int kb = 0; kb < p.kb_p; ++kb) {
                        const uint64_t adesc = smem_desc_sw128(smem_u32(smem) + (uint32_t)kb * 64u * BK * 2u);
                        const uint64_t bdesc = smem_desc_sw128(smem_u32(ring) + (uint32_t)kb * block);
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k) tc_mma_bf16(tm_acc, adesc + (uint64_t)(k * 2), bdesc + (uint64_t)(k * 2), idesc, (kb | k) != 0);
                    }
                    tc_commit(&acc_bar[0]);
                }
                __syncwarp();
            }
        }
        ++gemm_n;
    };

    for (int step = -1;; ++step) {
        const int par = step & 1;                                  // keys of joint phase `step`; hb[par] holds the state after step `step`
        // =====================================================================================
        // L: control in every CTA; cell update; enc_proj rows of the next window requested
        // =====================================================================================
        if (warp >= 2) {
            if (warp < 4) {
                int tok = -1, n_blank = 0;
                if (ctl && step < 0) {
                    tok = c_len > 0 ? p.blank : -1;
                } else if (ctl && c_t < c_len) {
                    const unsigned long long* kp = p.keys + (size_t)par * WD_ROWS + (size_t)slot * wi;
                    const int n = min(min(wi, p.W - c_off), c_len - c_t);
                    int first = -1, label = p.blank;
                    bool bad = false;
                    for (int w0 = 0; w0 < n && first < 0; w0 += 8) {
                        unsigned long long kk[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) kk[j] = w0 + j < n ? __ldcg(kp + w0 + j) : 0ull;
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            if (w0 + j < n && first < 0) {
                                uint32_t lab = key_label(kk[j]);
                                if (kk[j] == 0ull || lab >= (uint32_t)p.NV) { bad = true; lab = (uint32_t)p.blank; }
                                if ((int)lab != p.blank) { first = w0 + j; label = (int)lab; }
                            }
                        }
                    }
                    const int window = min(p.W, c_len - (c_t - c_off));      // rows of the whole window
                    const int pos = c_pos;
                    n_blank = first < 0 ? n : first;
                    int t = c_t + (first < 0 ? n : first);
                    const int t_emit = t, jump = c_off + (first < 0 ? n : first);
                    if (first != 0) c_cnt = 0;
                    bool forced = false, overflow = false;
                    if (first >= 0) {
                        if (pos < p.max_out) {
                            tok = label;
                            ++c_pos;
                            if (++c_cnt == p.S) { ++t; c_cnt = 0; forced = true; }
                        } else {
                            overflow = true;
                            t = c_len;                                       // no room for the token: this utterance stops here
                        }
                    }
                    c_t = t;
                    const bool whole = first >= 0 || jump >= window;         // the window is done with
                    c_off = whole ? 0 : jump;
                    c_wins += whole;
                    if (is_c) {
                        if (tok >= 0) {
                            p.out_tokens[(size_t)c_utt * p.max_out + pos] = label;
                            p.out_frames[(size_t)c_utt * p.max_out + pos] = t_emit;
                        }
                        if (c_t >= c_len) p.out_len[c_utt] = c_pos;
                        n_tok += tok >= 0; n_forced += forced;
                        if (whole) { n_rows += window; atomicAdd(&s_hist[jump < 64 ? jump : 64], 1); }
                        if (overflow) set_status(p.ctrl, WIND_ERR_OUTPUT_OVERFLOW);
                        if (bad) set_status(p.ctrl, WIND_ERR_INTERNAL);
                    }
                }
                const int left = ctl ? c_len - c_t : 0;
                if (slot < WD_SLOTS) {
                    s_tok[slot] = left > 0 ? tok : -1;                       // a finished utterance needs no further state
                    s_row[slot] = c_utt * p.T + c_t;
                    s_left[slot] = left;
                }
                const uint32_t alive = __ballot_sync(0xffffffffu, left > 0);
                const int sum_blank = __reduce_add_sync(0xffffffffu, n_blank), n_label = __popc(__ballot_sync(0xffffffffu, step >= 0 && tok >= 0));
                if (lane == 0) { s_blanks[warp - 2] = sum_blank; s_labels[warp - 2] = n_label; }
                if (lane == 0) s_live[warp - 2] = alive ? 32 * (warp - 2) + 32 - __clz((int)alive) : 0;
            }
            asm volatile("bar.sync 1, %0;" ::"n"(WD_EPI) : "memory");
            live = max(s_live[0], s_live[1]);
            blanks = 0.9f * blanks + (float)(s_blanks[0] + s_blanks[1]);
            labels = 0.9f * labels + (float)(s_labels[0] + s_labels[1]);
            wi = wide_rows(p.W, live, blanks, labels);
            if (e == 0) s_window = wi;
            if (is_l) {
                // gate-table entries of the tokens; lanes 0..15 hold the tile's accumulator rows (unit u of gate q)
                const int u = lane & 15, unit = ut * 16 + u;
                const bool gemm = step >= 0;
                if (gemm) { mbar_wait_warp(&acc_bar[0], (gemm_n - 1u) & 1u, &s_abort); tc_fence_after(); }
                for (int c0 = 16 * sub; c0 < p.nl; c0 += 32) {
                    // eight of the sixteen columns move to lanes 16..31, which hold no accumulator row
                    const int first = c0 + 8 * (lane >> 4);
                    float x[16], add[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int tok = s_tok[first + j];
                        add[j] = tok >= 0 ? __ldg(p.g0 + (size_t)tok * 4 * p.P + (size_t)q * p.P + unit) : 0.f;
                    }
                    if (gemm) {
                        tmem_ld16(tm_acc + lane_off + (uint32_t)c0, x);
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j) x[j] = 0.f;
                    }
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float hi = __shfl_sync(0xffffffffu, x[8 + j], u);
                        const float s = (lane < 16 ? x[j] : hi) + add[j];
                        stage[(q * p.nl + first + j) * 16 + u] = q == 2 ? tanhf(s) : sigmoid_f(s);
                    }
                }
                asm volatile("bar.sync 1, %0;" ::"n"(WD_EPI) : "memory");
                __nv_bfloat16* out = p.hb[(step + 1) & 1] + (size_t)(ut >> 2) * p.nl * BK + (ut & 3) * 16;
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    const int b = (e >> 4) + 16 * jj, un = e & 15;
                    if (b < p.nl && b < p.B) {
                        if (s_tok[b] >= 0) {
                            const float gi = stage[(0 * p.nl + b) * 16 + un], gf = stage[(1 * p.nl + b) * 16 + un];
                            const float gg = stage[(2 * p.nl + b) * 16 + un], go = stage[(3 * p.nl + b) * 16 + un];
                            cell[jj] = cell_update_fc(gf, cell[jj], gi, gg);
                            hid[jj] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(go * tanhf(cell[jj])));
                        }
                        out[b * BK + un] = __ushort_as_bfloat16((unsigned short)hid[jj]);
                    }
                }
                fence_proxy_async_all();
            } else if (is_p) {
                if (bw_wi != wi) {
                    bw_wi = wi;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int r = (e >> 3) + 32 * i, b = r / wi;
                        bw[i] = b < p.B ? (b << 8) | (r - b * wi) : -1;
                    }
                }
                kinds = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    ev[i] = make_uint4(0, 0, 0, 0);
                    if (bw[i] >= 0) {
                        const int b = bw[i] >> 8, w = bw[i] & 255, left = s_left[b];
                        const int kind = left <= 0 ? 0 : (w >= left ? 1 : 2);
                        kinds |= kind << (2 * i);
                        if (kind == 2) ev[i] = __ldg(reinterpret_cast<const uint4*>(p.enc_proj + ((size_t)s_row[b] + w) * p.H + ht * 64 + (e & 7) * 8));
                    }
                }
            } else if (is_c) {
                // the keys of the next joint phase (last read a step ago, by everybody)
                if (e < WD_ROWS) p.keys[(size_t)((step + 1) & 1) * WD_ROWS + e] = 0ull;
            }
        }
        if (!grid_sync(TR_L)) break;
        // (for the issuing warps; the same everywhere.  Out of a shuffle, so that the compiler knows that all lanes have the same)
        live = __shfl_sync(0xffffffffu, max(s_live[0], s_live[1]), 0);
        wi = __shfl_sync(0xffffffffu, s_window, 0);
        if (live == 0) break;
        if (step + 1 >= p.step_cap) { exit_status = WIND_ERR_INTERNAL; break; }
        // =====================================================================================
        // P: pred_proj and z; behind it the decoder's GEMM of the next step
        // =====================================================================================
        if (is_l || is_p) {
            state_gemm((step + 1) & 1);
            if (is_p && warp >= 2) {
                mbar_wait_warp(&acc_bar[0], (gemm_n - 1u) & 1u, &s_abort);
                tc_fence_after();
                for (int c0 = 16 * sub; c0 < (live <= 16 ? 16 : p.nl); c0 += 32) {
                    float g[16];
                    tmem_ld16(tm_acc + lane_off + (uint32_t)c0, g);
                    if (lane < 16) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) stage[(c0 + j) * 68 + 16 * q + lane] = g[j] + p_bias;
                    }
                }
                asm volatile("bar.sync 1, %0;" ::"n"(WD_EPI) : "memory");
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int kind = (kinds >> (2 * i)) & 3;
                    if (kind == 0) continue;
                    const float4* gs = reinterpret_cast<const float4*>(stage + (bw[i] >> 8) * 68 + (e & 7) * 8);
                    const float4 ga = gs[0], gb = gs[1];
                    const float g[8] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w};
                    const __nv_bfloat162* eb = reinterpret_cast<const __nv_bfloat162*>(&ev[i]);
                    uint32_t wds[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float2 e2 = __bfloat1622float2(eb[k]);
                        float z0 = e2.x + g[2 * k], z1 = e2.y + g[2 * k + 1];
                        z0 = p.act == WIND_ACT_RELU ? fmaxf(z0, 0.f) : tanh_fast(z0);
                        z1 = p.act == WIND_ACT_RELU ? fmaxf(z1, 0.f) : tanh_fast(z1);
                        wds[k] = kind == 2 ? pack_bf16x2(z0, z1) : 0u;
                    }
                    *reinterpret_cast<uint4*>(p.z + ((size_t)ht * WD_ROWS + (e >> 3) + 32 * i) * BK + (e & 7) * 8) = make_uint4(wds[0], wds[1], wds[2], wds[3]);
                }
                fence_proxy_async_all();
                tc_fence_before();
            }
        }
        if (!grid_sync(TR_P)) break;
        // =====================================================================================
        // J: logits of this CTA's vocabulary entries for every window row, best (logit, label) key of each row
        // =====================================================================================
        if (is_j) {
            const int rows = live * wi, groups = (rows + WD_NJ - 1) / WD_NJ, box = rows <= 16 ? 0 : (rows <= 32 ? 1 : (rows <= 64 ? 2 : 3));
            // (few rows make short stages and more of them)
            const int unit = box == 3 ? WD_UNIT / 2 : WD_UNIT, units = (p.kb_h + unit - 1) / unit;     // K blocks of a stage, stages of a row group
            const uint32_t z_block = (16u << box) * BK * 2u, z_bytes = z_block * (uint32_t)unit, stages = min((uint32_t)WD_MAX_STAGES, (uint32_t)p.stages * WD_Z_STAGE / z_bytes);
            const uint32_t loads = (uint32_t)(groups * units);
            const uint32_t used = (loads / stages & 1u ? (1u << stages) - 1u : 0u) ^ ((1u << loads % stages) - 1u);   // stages used an odd number of times
            uint32_t cur = 0, turn = 0;
            if (warp == 0) {
                fence_proxy_async_all();
                if (elect_one()) {
                    bool ok = true;
                    for (int rg = 0; rg < groups && ok; ++rg)
                        for (int i = 0, kb = kb_first; i < units; ++i, kb = kb + unit >= p.kb_h ? 0 : kb + unit) {
                            if (!(ok = mbar_wait(&empty_bar[cur], ((phases >> cur) ^ turn) & 1u, &s_abort))) break;
                            mbar_expect_tx(&full_bar[cur], z_bytes);
                            tma_load_3d(ring + cur * z_bytes, &M.z[box], 0, rg * WD_NJ, kb, &full_bar[cur]);
                            if (++cur == stages) { cur = 0; ++turn; }
                        }
                }
                __syncwarp();
                phases ^= used;
            } else if (warp == 1) {
                // (the waits stand outside the elected thread's part: behind one in it the compiler no longer keeps the MMAs' operands in
                // uniform registers, and an MMA took 50 cycles to issue)
                tc_fence_after();
                bool ok = true;
                for (int rg = 0; rg < groups && ok; ++rg, ++gemm_n) {
                    const int cols = min(WD_NJ, (rows - rg * WD_NJ + 15) / 16 * 16);
                    const uint32_t k_acc = gemm_n & two, idesc = idesc_bf16(128, cols), acc = tm_acc + k_acc * WD_NJ;
                    if (!(ok = mbar_wait_warp(&acc_free[k_acc], ((gemm_n >> two) & 1u) ^ 1u, &s_abort))) break;
                    for (int i = 0, kb = kb_first; i < units; ++i, kb = kb + unit >= p.kb_h ? 0 : kb + unit) {
                        if (!(ok = mbar_wait_warp(&full_bar[cur], ((phases >> cur) ^ turn) & 1u, &s_abort))) break;
                        tc_fence_after();
                        if (elect_one()) {
                            uint64_t bdesc = smem_desc_sw128(smem_u32(ring) + cur * z_bytes);
                            const int end = min(kb + unit, p.kb_h), end_t = min(end, kb_t);
                            uint32_t more = i > 0;
                            int b = kb;
#pragma unroll 1
                            for (; b < end_t; ++b, bdesc += z_block >> 4) {
#pragma unroll
                                for (int k = 0; k < BK / 16; ++k, more = 1u) tc_mma_bf16_ts(acc, tmem + (uint32_t)(b * (BK / 2) + k * 8), bdesc + (uint64_t)(k * 2), idesc, more);
                            }
                            uint64_t adesc = smem_desc_sw128(smem_u32(smem) + (uint32_t)(b - kb_t) * 128u * BK * 2u);
#pragma unroll 1
                            for (; b < end; ++b, bdesc += z_block >> 4, adesc += (128u * BK * 2u) >> 4) {
#pragma unroll
                                for (int k = 0; k < BK / 16; ++k, more = 1u) tc_mma_bf16(acc, adesc + (uint64_t)(k * 2), bdesc + (uint64_t)(k * 2), idesc, more);
                            }
                            tc_commit(&empty_bar[cur]);
                            if (i + 1 == units) tc_commit(&acc_bar[k_acc]);
                        }
                        __syncwarp();
                        if (++cur == stages) { cur = 0; ++turn; }
                    }
                }
                phases ^= used;
            } else {
                unsigned long long* keys = p.keys + (size_t)((step + 1) & 1) * WD_ROWS;
                const int v0 = vt * 128 + q * 32 + (lane >> 2);
                for (int rg = 0; rg < groups; ++rg, ++gemm_n) {
                    const uint32_t k_acc = gemm_n & two;
                    const bool ready = mbar_wait_warp(&acc_bar[k_acc], (gemm_n >> two) & 1u, &s_abort);
                    tc_fence_after();
                    const int here = min(WD_NJ, rows - rg * WD_NJ);
                    // A thread holds a quarter of the quadrant's entries of eight window rows: three comparisons each without an exchange,
                    // then three exchanges  (A row of entries
                    // per lane took five, with 31 instead of 7 pairs of shuffles: 3750 cycles for 128 rows against 1600.)
                    for (int c0 = 32 * sub; ready && c0 < here; c0 += 64) {
                        float x[32], val[8];
                        int id[8];
                        wide_tmem_ld(tm_acc + lane_off + k_acc * WD_NJ + (uint32_t)c0, x);
#pragma unroll
                        for (int c = 0; c < 8; ++c) { val[c] = -INFINITY; id[c] = v0; }
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (v0 + 8 * k < p.NV)
#pragma unroll
                                for (int c = 0; c < 8; ++c) {
                                    const float l = x[16 * (k >> 1) + 4 * (c >> 1) + 2 * (k & 1) + (c & 1)] + j_bias[k];
                                    if (k == 0 || l > val[c]) { val[c] = l; id[c] = v0 + 8 * k; }
                                }
                        wide_exchange<4, 16>(val, id, lane);
                        wide_exchange<2, 8>(val, id, lane);
                        wide_exchange<1, 4>(val, id, lane);
                        const int col = (lane & 16) + (lane & 8) + 2 * (lane & 3) + ((lane >> 2) & 1);
                        s_part[q * WD_NJ + c0 + col] = val[0] > -INFINITY ? pack_key(val[0], (uint32_t)id[0]) : 0ull;
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_free[k_acc]);
                    asm volatile("bar.sync 1, %0;" ::"n"(WD_EPI) : "memory");
                    if (ready && e < here) {
                        const unsigned long long* sp = s_part + e;
                        const unsigned long long key = max(max(sp[0], sp[WD_NJ]), max(sp[2 * WD_NJ], sp[3 * WD_NJ]));
                        if (key != 0ull) atomicMax(&keys[rg * WD_NJ + e], key);
                    }
                    if (rg + 1 < groups) asm volatile("bar.sync 1, %0;" ::"n"(WD_EPI) : "memory");   // s_part is written again
                }
            }
        }
        if (!grid_sync(TR_J)) break;
    }
    // L: the GEMM issued last may still run
    if (is_l && warp == 1 && gemm_n > 0u) {
        int gave_up = 0;
        mbar_wait(&acc_bar[0], (gemm_n - 1u) & 1u, &gave_up);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, LOOP_TMEM_COLS);
    }
    if (is_c && ctl) {
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->joint_rows), (unsigned long long)n_rows);
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->tokens), (unsigned long long)n_tok);
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->forced), (unsigned long long)n_forced);
        atomicMax(&p.ctrl->step, c_wins);
    }
    if (is_c)
        for (int k = threadIdx.x; k < 65; k += WD_THREADS)
            if (s_hist[k]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->jump_hist[k]), (unsigned long long)s_hist[k]);
    if (threadIdx.x == 0) {
        if (s_abort == 1) { note_timeout(p.ctrl, 4, cta); set_status(p.ctrl, WIND_ERR_TIMEOUT); }
        if (cta == 0) {
            if (exit_status) set_status(p.ctrl, exit_status);
            p.ctrl->active = 0;
            p.ctrl->loop_kernel = WIND_LOOP_WIDE;
            for (int k = 0; k < 3; ++k) p.ctrl->phase_cycles[k] = cyc[k];
            p.ctrl->loop_ns = (long long)(globaltimer_ns() - ns0);
        }
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static std::mutex g_wd_mutex;
static int g_wd_optin[64] = {};        // opt-in shared memory per block, 0: not asked yet

static cudaError_t wd_device(int* optin) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_wd_mutex);
    if (!g_wd_optin[dev]) {
        int n = 0;
        if ((e = cudaDeviceGetAttribute(&n, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
        if ((e = cudaFuncSetAttribute(wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, n - 8192)) != cudaSuccess) return e;   // static: below 8 KB
        g_wd_optin[dev] = n;
    }
    *optin = g_wd_optin[dev];
    return cudaSuccess;
}

// A CTA for every tile (and one that records), every tile in its CTA with a state box or four stages of z behind it.
static bool wd_plan(const Call& c, WdPlan* out) {
    const wind_model_t& m = c.m;
    WdPlan w{};
    if (m.L != 1 || m.P % BK || m.H % BK || c.B > WD_SLOTS || c.W > kMaxWindow || c.N > 0) return false;
    int sms = 0, optin = 0;
    if (loop_sm_count(&sms) != cudaSuccess || wd_device(&optin) != cudaSuccess) { cudaGetLastError(); return false; }
    const int budget = optin - 8192 - 1024;
    const int kb_h = m.H / BK, kb_p = m.P / BK;
    w.n_l = m.P / 16; w.n_j = (m.V + 1 + 127) / 128; w.n_p = m.H / 64;
    w.grid = w.n_l + w.n_j + 1 + w.n_p;
    if (w.grid > sms) return false;
    w.nl = c.B <= 16 ? 16 : (c.B <= 32 ? 32 : 64);
    const int tile = kb_p * 64 * BK * 2, box = w.nl * m.P * 2;
    const int l = tile + box + 4 * w.nl * 16 * 4, pp = tile + box + w.nl * 68 * 4;
    const int jw = (kb_h > WD_TM_BLOCKS ? kb_h - WD_TM_BLOCKS : 0) * 128 * BK * 2;
    w.stages = (budget - jw) / (int)WD_Z_STAGE;
    if (w.stages > 2 * WD_MAX_STAGES) w.stages = 2 * WD_MAX_STAGES;
    if (w.stages < 4) return false;
    int most = l > pp ? l : pp;
    if (most > budget) return false;
    if (jw + w.stages * (int)WD_Z_STAGE > most) most = jw + w.stages * (int)WD_Z_STAGE;
    w.smem = (uint32_t)most + 1024u;
    *out = w;
    return true;
}

// Only plain greedy decoding with the default loop options: everything else stays with loop_kernel.
bool wide_supported(const Call& c) {
    if (c.mode != WIND_MODE_FIRST_NONBLANK || c.joint_iters > 0) return false;
    const LoopOptions o = loop_get_options();
    if (!o.resident || o.dataflow >= 0 || o.joint_placement >= 0) return false;
    WdPlan w;
    return wd_plan(c, &w);
}

cudaError_t wide_loop(const Call& c) {
    WdPlan w;
    if (!wd_plan(c, &w)) return cudaErrorNotSupported;
    const wind_model_t& m = c.m;
    WdMaps M;
    cudaError_t e;
    if ((e = loop_map3(&M.w_hh, c.w_hh[0], 4ull * m.P, m.P, 16, 1)) != cudaSuccess) return e;
    if ((e = loop_map3(&M.w_pred, m.w_pred, m.H, m.P, 64, 1)) != cudaSuccess) return e;
    if ((e = loop_map3(&M.w_out, m.w_out, (uint64_t)m.V + 1, m.H, 128, 1)) != cudaSuccess) return e;
    for (int k = 0; k < 4; ++k)
        if ((e = loop_map_blocks(&M.z[k], c.z(), m.H / BK, WD_ROWS, 16 << k, k == 3 ? WD_UNIT / 2 : WD_UNIT)) != cudaSuccess) return e;
    for (int k = 0; k < 2; ++k) {
        for (int par = 0; par < 2; ++par)
            if ((e = loop_map_blocks(&M.hb[par][k], c.hb(par, 0), m.P / BK, w.nl, k ? w.nl : 16, m.P / BK)) != cudaSuccess) return e;
    }
    WdParams p{};
    p.ctrl = c.ctrl();
    p.B = c.B; p.T = c.T; p.W = c.W; p.S = c.S; p.max_out = c.max_out; p.H = m.H; p.P = m.P; p.NV = m.V + 1; p.blank = m.blank_id; p.act = m.act;
    const long long cap = (long long)c.T * (c.S + 1) + 2;       // a part of a window moves by a frame or emits, like a whole one
    p.step_cap = cap > 0x7fffffff ? 0x7fffffff : (int)cap;
    p.extra_arrivals = loop_extra_arrivals();
    p.n_l = w.n_l; p.n_j = w.n_j; p.n_p = w.n_p; p.nl = w.nl; p.stages = w.stages; p.kb_h = m.H / BK; p.kb_p = m.P / BK;
    p.enc_len = c.enc_len;
    p.keys = c.keys();
    p.out_tokens = c.out_tokens; p.out_frames = c.out_frames; p.out_len = c.out_len;
    p.hb[0] = c.hb(0, 0); p.hb[1] = c.hb(1, 0);
    p.z = c.z(); p.enc_proj = (const __nv_bfloat16*)c.enc_proj(); p.g0 = c.g0();
    p.b_pred = m.b_pred; p.b_out = m.b_out; p.w_out = (const __nv_bfloat16*)m.w_out;
    void* args[2] = {(void*)&M, (void*)&p};
    return cudaLaunchCooperativeKernel((const void*)wide_kernel, dim3((unsigned)w.grid), dim3(WD_THREADS), args, w.smem, c.stream);
}

}  // namespace wind
