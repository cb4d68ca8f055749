// The decoding loop of the bf16 path for models of one or two layers whose decoder fits one thread-block cluster (sm_100a).
//
// A lock step is a chain of small dependent products, so what it costs is the latency of handing results from SM to SM.
// Here every hand-over stays inside a cluster of 16 CTAs (st.async into distributed shared memory: about 0.25 us) instead of
// going through L2 (a barrier over the chip alone is 1.3 us), and clusters share nothing but the queue of utterances.
//
// All weights of the loop stay on chip, cut over the 16 CTAs of a cluster (large model: 5.4 MB; a CTA holds 340 KB):
//   tensor memory   W_hh rows of the CTA's first 32 hidden units (4 gates x 32 = the 128 lanes), operand A of the gates' MMA; with two
//                   layers the second one's W_ih (two more clusters hold W_hh, one a layer, for up to CL_DECODERS that decode: cl_recurrent)
//   shared memory   W_out rows of its 1/16 of the vocabulary
//   registers       W_pred rows of its 1/16 of the joint's hidden units and W_hh (W_ih) rows of its remaining hidden units, as
//                   mma.sync fragments (no register may be spilled: next to 220 KB of shared memory there is no first-
//                   level cache left, and a spilled value comes from L2)
// A cluster decodes up to 8 utterances ("slots") at a time; a lock step of a cluster is
//   keys    every CTA sends the best (logit, label) of its labels for each window row to the slot's owner (slot u: CTA u)
//   control the owner takes Algorithm 2's decision and sends (token, next frame) to every CTA, then records it; the window's
//           enc_proj rows start on their way (one TMA box per eight rows, in the layout of the joint's operand)
//   (a step in which no slot feeds a token to its decoder goes from here to the joint, and only slots that do send anything in
//   the next two phases: most steps of narrow windows emit nothing)
//   gates   W_hh h was computed a step ahead; + the token's row of the gate table, cell update, new h to every CTA (the second layer:
//           W_ih times that, + its W_hh h, computed meanwhile in another cluster)
//   pred    W_pred h, pred_proj to every CTA
//   joint   z = act(enc_proj rows + pred_proj) in place, times the CTA's W_out rows on tcgen05 (window rows on the M axis, so
//           that an accumulator lane is a window row and its argmax needs no exchange between lanes)
// W_pred h is 40 rows per CTA: as 40 dependent tcgen05.mma it would take 1000 cycles (24 each however small the tile), as
// two chains of 20 mma.sync 420.  mma.sync and tcgen05.mma accumulate a K step of 16 identically (checked bit for bit), and
// K halves, roundings and epilogue arithmetic are those of loop_kernel with resident weights: same transcripts, bit for bit.
//
// A slot whose utterance is finished takes the next one from the queue in the same lock step (its recurrent term and cell
// state count as zero in the step that feeds start-of-sequence).
//
// Every wait is bounded.  A CTA that gives up sets WIND_ERR_TIMEOUT; the others of its cluster run out of their own waits;
// all meet at the cluster barrier at the end, so no CTA leaves while another may still write into its shared memory.
#include <cudaTypedefs.h>

#include <cmath>
#include <mutex>
#include <type_traits>

#include "wind_loop_cl.cuh"
#include "wind_loop_dev.cuh"

namespace wind {

struct ClDec { int tok; uint32_t flags, row, unused; };   // what an owner sends for its slot
constexpr uint32_t CL_FRESH = 1u, CL_IDLE = 2u, CL_ODD = 4u;   // CL_ODD: parity of the step it is for

// W_hh (or the second layer's W_ih) rows of the CTA's hidden units 0..31 into tensor memory: lane 4 u + gate.  Warps 0-7.
// AT_ONCE pieces are under way: five make short decodes of two layers 0.6 % faster; with one layer the registers they take lengthen every
// step of several slots (128 utterances 8.61 -> 8.69 ms, 32 at W = 1 5.67 -> 5.71, one slot the same).
template <int AT_ONCE>
__device__ __forceinline__ void cl_gate_rows_to_tmem(const __nv_bfloat16* w, int P, int r, int warp, int lane, uint32_t tmem) {
    const int q = warp & 3, U = P / CL_SIZE, u = 8 * q + (lane >> 2), g = lane & 3;
    const bool in = u < U;
    const uint4* src = reinterpret_cast<const uint4*>(w + ((size_t)g * P + r * U + (in ? u : 0)) * P);
#pragma unroll 1
    for (int c0 = 16 * (warp >> 2); c0 < P / 2; c0 += 32 * AT_ONCE) {
        uint32_t v[AT_ONCE][16];
#pragma unroll
        for (int k = 0; k < AT_ONCE; ++k)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint4 x = in && c0 + 32 * k < P / 2 ? src[(c0 + 32 * k) / 4 + j] : make_uint4(0, 0, 0, 0);
                v[k][4 * j] = x.x; v[k][4 * j + 1] = x.y; v[k][4 * j + 2] = x.z; v[k][4 * j + 3] = x.w;
            }
#pragma unroll
        for (int k = 0; k < AT_ONCE; ++k)
            if (c0 + 32 * k < P / 2) tmem_st16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(c0 + 32 * k), v[k]);
    }
    tmem_st_wait();
}

// The recurrent terms of two-layer models.  Such a decoder (large dimensions: 12 MB) does not fit a cluster, but W_hh h of either
// layer is not needed before the next step's update, so a cluster per layer keeps that layer's W_hh and computes it for all decoding
// clusters while these go on: CTA r of a decoding cluster leaves its units of the new state in hx and adds one to req; CTA r here
// fetches the state of all units once 16 CTAs have, multiplies its rows (the units of CTA r there) and leaves the result where CTA r
// reads it (rx), every value with the number of the update: value and "ready" arrive in one load, and no write has to be waited for
// (a counter behind the writes, a copy into shared memory and their fences took 3500 cycles).  hx has two copies by parity of the
// updates: a CTA writes a copy again only two updates later, when every CTA of its cluster has had the answer to the update between;
// nothing else here needs more than one, since a CTA's next request follows its answer.  The round trip through L2 takes most of a
// step, so requests should not queue: the states of all clusters lie one behind the other as row groups of one operand, and a chain
// of MMAs serves every request that is there when it starts (its other columns go nowhere).
// Warps: 0-3 results, 4-11 remainder units (mma.sync; 4-7 for even clusters), 14 issues MMAs, 15 fetches states.
constexpr int CL_REC_SETS = 3;                            // accumulators: the results of one chain leave under the next ones
__device__ __noinline__ void cl_recurrent(const CUtensorMap& hx_map, const ClParams& p, const int layer, const int r, uint8_t* smem) {
    __shared__ uint64_t bar_full[CL_DECODERS], bar_acc[CL_REC_SETS], bar_free[CL_REC_SETS];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile uint32_t s_total[CL_DECODERS];    // updates of a decoding cluster that has left (before that: all ones)
    __shared__ volatile uint32_t s_mask[CL_REC_SETS];     // decoding clusters whose results an accumulator holds; 0: no more of them
    __shared__ volatile int s_abort;
    const int warp = uniform_warp_index(), lane = threadIdx.x & 31;
    const int n_dec = (int)gridDim.x / CL_SIZE - 2, U = p.P / CL_SIZE, NU = p.slots;
    const bool has_rem = U > 32;
    const uint32_t state = (uint32_t)p.P * 16u;           // bytes of a cluster's state: K blocks of 8 slots x 128 bytes
    const uint32_t acc_cols = (uint32_t)(8 * n_dec + 15) & ~15u;
    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int c = 0; c < CL_DECODERS; ++c) { s_total[c] = 0xFFFFFFFFu; mbar_init(&bar_full[c], 1); }
        for (int c = 0; c < CL_REC_SETS; ++c) { mbar_init(&bar_acc[c], 2); mbar_init(&bar_free[c], 4); }
        fence_barrier_init();
        prefetch_tmap(&hx_map);
    }
    if (warp == 14) tmem_alloc(&tmem_slot, LOOP_TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);
    if (warp < 8) cl_gate_rows_to_tmem<5>(p.w_rec[layer], p.P, r, warp, lane, tmem);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm_acc = tmem + CL_MAX_DIM / 2;
    auto answer = [&](int c) { return p.rx + ((size_t)(c * 2 + layer) * CL_SIZE + r) * (size_t)(NU * 4 * U); };
    uint32_t n = 0u;                                      // of cluster `lane`: updates this warp has dealt with
    // work(mask) for those of the clusters `mine` whose state is there, until all of them have left
    auto serve = [&](uint32_t mine, auto work) {
        const int c = min(lane, n_dec - 1);
        const bool on = lane < n_dec && ((mine >> lane) & 1u);
        for (;;) {
            const uint32_t total = s_total[c];
            const uint32_t ready = __ballot_sync(0xffffffffu, on && n != total && mbar_test(&bar_full[c], n & 1u));
            if (__any_sync(0xffffffffu, s_abort) || __all_sync(0xffffffffu, !on || n == total)) break;
            if (ready) {
                __syncwarp();                             // one lane has seen the barrier complete, all read what it stands for
                work(ready);
                n += (ready >> lane) & 1u;
            }
        }
    };
    if (warp < 4) {
        const int e = threadIdx.x, u = 8 * warp + (lane >> 2);
        for (uint32_t set = 0u, turn = 0u;;) {
            // (the warp that issues leaves a mask of 0 behind its last chain)
            bool there = false;
            while (!(there = __all_sync(0xffffffffu, mbar_test(&bar_acc[set], turn & 1u))) && !__any_sync(0xffffffffu, s_abort)) {}
            const uint32_t mask = there ? s_mask[set] : 0u;
            if (mask == 0u) break;
            tc_fence_after();
            n += (mask >> lane) & 1u;
            const bool alone = (mask & (mask - 1u)) == 0u;
            for (uint32_t left = mask; left; left &= left - 1u) {
                const int c = __ffs((int)left) - 1;
                const uint32_t stamp = __shfl_sync(0xffffffffu, n, c);
                float x[8];
                tmem_ld8(tm_acc + set * acc_cols + (alone ? 0u : 8u * (uint32_t)c) + ((uint32_t)(warp * 32) << 16), x);
                unsigned long long* dst = answer(c) + e;
                if (u < U)
#pragma unroll
                    for (int s = 0; s < 8; ++s)
                        if (s < NU) st_relaxed_u64(dst + s * 4 * U, (unsigned long long)stamp << 32 | __float_as_uint(x[s]));
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_free[set]);
            if (++set == CL_REC_SETS) { set = 0u; ++turn; }
        }
    } else if (warp < 12) {
        if (has_rem) {
            const int k = (warp - 4) & 3, row = 8 * k + (lane >> 2), u = 32 + (row >> 2), g = row & 3;
            uint32_t wf[40][2];
            const uint32_t* src = reinterpret_cast<const uint32_t*>(p.w_rec[layer] + ((size_t)g * p.P + r * U + min(u, U - 1)) * p.P) + (lane & 3);
#pragma unroll
            for (int s0 = 0; s0 < 40; s0 += 8)
                if (s0 < p.P / 16)
#pragma unroll
                    for (int s = s0; s < s0 + 8; ++s) { wf[s][0] = src[s * 8]; wf[s][1] = src[s * 8 + 4]; }
            serve(warp < 8 ? 0x55555555u : 0xAAAAAAAAu, [&](uint32_t mask) {
                for (uint32_t left = mask; left; left &= left - 1u) {
                    const int c = __ffs((int)left) - 1;
                    const uint32_t h_row = smem_u32(smem) + (uint32_t)c * state + (uint32_t)((lane & 7) * 128);
                    auto h_at = [&](int k32) { return h_row + (uint32_t)(k32 >> 1) * 1024u + (uint32_t)((((k32 & 1) * 4 + (lane >> 3)) ^ (lane & 7)) << 4); };
                    float acc[4] = {0.f, 0.f, 0.f, 0.f};
                    uint32_t a[2][4];
                    ldmatrix_x4(a[0], h_at(0));
#pragma unroll
                    for (int s0 = 0; s0 < 40; s0 += 8)
                        if (s0 < p.P / 16)
#pragma unroll
                            for (int s = s0; s < s0 + 8; s += 2) {
                                ldmatrix_x4(a[(s / 2 + 1) & 1], h_at(s / 2 + 1));       // (the last turn: rows nobody uses)
                                mma_16816(acc, a[(s / 2) & 1][0], 0u, a[(s / 2) & 1][1], 0u, wf[s][0], wf[s][1]);
                                mma_16816(acc, a[(s / 2) & 1][2], 0u, a[(s / 2) & 1][3], 0u, wf[s + 1][0], wf[s + 1][1]);
                            }
                    const unsigned long long stamp = (unsigned long long)(__shfl_sync(0xffffffffu, n, c) + 1u) << 32;
                    unsigned long long* dst = answer(c) + (lane >> 2) * 4 * U + 128 + k * 8 + (lane & 3) * 2;
                    if ((lane >> 2) < NU) {
                        st_relaxed_u64(dst, stamp | __float_as_uint(acc[0]));
                        st_relaxed_u64(dst + 1, stamp | __float_as_uint(acc[1]));
                    }
                }
            });
        }
    } else if (warp == 14) {
        const uint32_t id_all = idesc_bf16(128, (int)acc_cols), id_one = idesc_bf16(128, 16);
        uint32_t set = 0u, turn = 0u;                     // chains so far: turn * CL_REC_SETS + set
        auto next = [&](uint32_t mask) {                  // an accumulator for the next chain
            if (turn > 0u && !cl_wait_warp(&bar_free[set], (turn - 1u) & 1u)) { s_abort = 1; return false; }
            if (lane == 0) { s_mask[set] = mask; mbar_arrive(&bar_acc[set]); }
            __syncwarp();
            return true;
        };
        serve(0xFFFFFFFFu, [&](uint32_t mask) {
            if (!next(mask)) return;
            tc_fence_after();
            if (elect_one()) {
                // row groups (the clusters' states) `state` bytes apart.  One request alone: its state and the rows behind it (an MMA
                // has 16 columns at the least, and with 48 the chain takes half as long again)
                const bool alone = (mask & (mask - 1u)) == 0u;
                const uint32_t first = alone ? (uint32_t)(__ffs((int)mask) - 1) * state : 0u, id = alone ? id_one : id_all;
                uint64_t hd = (smem_desc_sw128(smem_u32(smem) + first) & ~((uint64_t)0x3FFF << 32)) | ((uint64_t)(state >> 4) << 32);
#pragma unroll 1
                for (int kb = 0; kb < p.P / 64; ++kb, hd += 1024 >> 4)
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        tc_mma_bf16_ts(tm_acc + set * acc_cols, tmem + (uint32_t)(kb * 32 + k * 8), hd + (uint64_t)(k * 2), id, (kb | k) != 0);
                tc_commit(&bar_acc[set]);
            }
            __syncwarp();
            if (++set == CL_REC_SETS) { set = 0u; ++turn; }
        });
        // MMAs in flight use tensor memory
        if (set > 0u || turn > 0u) cl_wait_warp(&bar_acc[set > 0u ? set - 1u : CL_REC_SETS - 1], (set > 0u ? turn : turn - 1u) & 1u);
        if (!s_abort && next(0u) && lane == 0) mbar_arrive(&bar_acc[set]);
        __syncwarp();
    } else if (warp == 15) {
        const int c = min(lane, n_dec - 1);
        bool left = lane >= n_dec;
        uint32_t beat = 0u;
        unsigned long long since = globaltimer_ns();
        for (uint32_t it = 1u;; ++it) {
            // (whether a cluster has left is asked now and then, and before what it has asked for: nothing may come after that)
            const uint32_t gone = (it & 63u) == 0u && !left ? ld_acquire_u32(p.done + c) : 0u;
            if (!left) {
                const uint32_t there = ld_acquire_u32(p.req + layer * CL_DECODERS + c) - (uint32_t)CL_SIZE * n;
                if (there >= (uint32_t)CL_SIZE) {
                    fence_proxy_async_all();              // written by generic stores
                    mbar_expect_tx(&bar_full[c], state);
                    tma_load_3d(smem + (uint32_t)c * state, &hx_map, 0, ((c * 2 + layer) * 2 + (int)(n & 1u)) * 8, 0, &bar_full[c]);
                    ++n;
                } else if (gone == (uint32_t)CL_SIZE) {
                    left = true;
                    s_total[c] = n;
                }
            }
            if (__all_sync(0xffffffffu, left)) break;
            if ((it & 1023u) == 0u) {
                // a decoding cluster may have nothing to ask for long (blanks), but it counts its steps
                const uint32_t b = left ? 0u : ld_acquire_u32(p.beat + c) + n;
                const unsigned long long now = globaltimer_ns();
                if (__any_sync(0xffffffffu, b != beat)) since = now;
                beat = b;
                if (__any_sync(0xffffffffu, now - since > 2 * kWaitLimitNs || ld_acquire_u32(reinterpret_cast<const uint32_t*>(&p.ctrl->abort)) != 0u)) { s_abort = 1; break; }
            }
        }
        if (lane < n_dec && n > 0u) cl_wait(&bar_full[lane], (n - 1u) & 1u);     // copies in flight
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 14) {
        tc_fence_after();
        tmem_dealloc(tmem, LOOP_TMEM_COLS);
    }
    if (threadIdx.x == 0 && s_abort) {
        atomicExch(&p.ctrl->abort, 1);
        note_timeout(p.ctrl, 70 + layer, blockIdx.x);
        set_status(p.ctrl, WIND_ERR_TIMEOUT);
    }
}

// Warps: 0-3 gates and z (workers), 4-9 W_pred, 10-13 remainder units, 14 issuing thread, 15 control.  Warps 0-7 also
// share the joint's epilogue.  NS: most slots in use (1, 2, 4, 8).
template <int NS, int ACT, int NL>
__global__ void __launch_bounds__(CL_THREADS, 1) cl_kernel(const __grid_constant__ CUtensorMap enc_map, const __grid_constant__ CUtensorMap hx_map, const __grid_constant__ ClParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_keys, bar_dec, bar_enc, bar_h, bar_pred, bar_z, bar_sync_mma, bar_acc_g, bar_acc_r, bar_acc_j, bar_h0, bar_rec;
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort;
    __shared__ int s_hist[65];
    __shared__ long long s_lap[4];

    const int warp = uniform_warp_index(), lane = threadIdx.x & 31;
    if (p.ctrl->bad_input || (p.choose && p.ctrl->use_grid != 0)) return;   // a length outside [0, T], or another kernel's turn: the whole grid leaves before it does anything
    const int r = (int)cl_rank();
    if constexpr (NL == 2) {
        if (blockIdx.x / CL_SIZE < 2) {                  // (these come first: nobody waits for CTAs that are not resident yet)
            cl_recurrent(hx_map, p, (int)blockIdx.x / CL_SIZE, r, align_smem_1024(smem_raw));
            return;
        }
    }
    const int cluster = (int)blockIdx.x / CL_SIZE - (NL == 2 ? 2 : 0), n_clusters = (int)gridDim.x / CL_SIZE - (NL == 2 ? 2 : 0);
    const int NU = p.slots, U = p.P / CL_SIZE, HS = p.H / CL_SIZE;
    const int kb_p = p.P / 64, kb_h = p.H / 64;
    const int wp_shift = p.wp == 8 ? 3 : (p.wp == 16 ? 4 : 5);
    const int n_groups = (NU << wp_shift) >> 3;
    const int lab_base = cl_label_base(p.NV), lab_extra = cl_label_extra(p.NV);
    const int lab0 = r * lab_base + 8 * min(r, lab_extra);              // this CTA's vocabulary entries [lab0, lab0 + labs)
    const int lab_n = lab_base + (r < lab_extra ? 8 : 0);               // the MMA's N
    const int labs = min(lab_n, max(0, p.NV - lab0));
    const int lab_rows = lab_base + (lab_extra > 0 ? 8 : 0);            // rows of a K block of the W_out tile
    const bool has_rem = U > 32;
    // Whether warps 10-13 have a part in the steps.  They then build z in every one of them: a warp that nobody waits for could fall two
    // steps behind and take one decision for another.
    const bool rem_warps = has_rem || NL == 2;

    uint8_t* smem = align_smem_1024(smem_raw);
    const ClSmem& L = p.smem;                            // (worked out on the host: there is no register to spare)
    const uint32_t sbase = smem_u32(smem);
    const ClDec* dec = reinterpret_cast<const ClDec*>(smem + L.dec);
    float* s_bout = reinterpret_cast<float*>(smem + L.b_out);
    float* s_bpred = reinterpret_cast<float*>(smem + L.b_pred);
    float* gr = reinterpret_cast<float*>(smem + L.gr);

    if (threadIdx.x == 0) {
        s_abort = 0;
        s_lap[0] = s_lap[1] = s_lap[2] = 0;
        mbar_init(&bar_keys, 1);
        mbar_init(&bar_dec, 1u + (uint32_t)p.extra_arrivals);   // extra_arrivals > 0: a test hook, the wait can then never end
        mbar_init(&bar_enc, 1);
        mbar_init(&bar_h, 1);
        mbar_init(&bar_pred, 1);
        mbar_init(&bar_z, 10u + (rem_warps ? 4u : 0u));
        mbar_init(&bar_sync_mma, 6u + (has_rem ? 4u : 0u));
        mbar_init(&bar_acc_g, 1);
        mbar_init(&bar_acc_r, 4);
        mbar_init(&bar_acc_j, 1);
        mbar_init(&bar_h0, 1);
        mbar_init(&bar_rec, 4);
        fence_barrier_init();
        // armed for their first phase (later phases: by the warp that saw the previous one complete, and only then: a barrier must
        // not be armed twice in a phase).  bar_h and bar_pred are armed in the steps that update a decoder, once it is known how many.
        mbar_expect_tx(&bar_keys, (uint32_t)(2 * CL_SIZE * p.W) * 8u);
        mbar_expect_tx(&bar_dec, (uint32_t)NU * 16u);
        prefetch_tmap(&enc_map);
    }
    if (warp == 14) tmem_alloc(&tmem_slot, LOOP_TMEM_COLS);
    for (int i = threadIdx.x; i < 65; i += CL_THREADS) s_hist[i] = 0;
    if (threadIdx.x < CL_SLOTS) *reinterpret_cast<uint4*>(smem + L.dec + threadIdx.x * 16) = make_uint4(0xFFFFFFFFu, CL_IDLE, 0u, 0u);
    for (int i = threadIdx.x; i < CL_MAX_LABELS + 8; i += CL_THREADS) s_bout[i] = i < labs ? p.b_out[lab0 + i] : -INFINITY;
    for (int i = threadIdx.x; i < 48; i += CL_THREADS) s_bpred[i] = i < HS ? p.b_pred[r * HS + i] : 0.f;
    // ---- resident weights ----
#pragma unroll 1
    for (int row = warp; row < lab_rows; row += CL_THREADS / 32)                  // W_out: K blocks of lab_rows x 128 bytes, 128-byte swizzle
        for (int c = lane; c < p.H / 8; c += 32) {                                // (asynchronously: a row's copies were three round trips)
            uint8_t* dst = smem + L.w_out + (c >> 3) * (lab_rows * 128) + row * 128 + (((c & 7) ^ (row & 7)) << 4);
            if (row < labs) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(p.w_out + (size_t)(lab0 + row) * p.H + c * 8) : "memory");
            else *reinterpret_cast<uint4*>(dst) = make_uint4(0, 0, 0, 0);
        }
    for (uint32_t i = threadIdx.x; i < (L.pred - L.h0) / 16u; i += CL_THREADS)    // h of slots nobody uses must be numbers
        *reinterpret_cast<uint4*>(smem + L.h0 + i * 16) = make_uint4(0, 0, 0, 0);
    for (int i = threadIdx.x; i < NL * CL_SLOTS * U / 8; i += CL_THREADS) *reinterpret_cast<uint4*>(smem + L.hst + i * 16) = make_uint4(0, 0, 0, 0);
    if constexpr (NL == 2)
        for (int i = threadIdx.x; i < 4 * U; i += CL_THREADS) {
            const int at = (i & 3) * p.P + r * U + (i >> 2);
            reinterpret_cast<float*>(smem + L.b_gate)[i] = p.b_gate[0][at] + p.b_gate[1][at];
        }
    // the recurrent term of layer l (two layers)
    auto rec_at = [&](int l) { return p.rx + ((size_t)(cluster * 2 + l) * CL_SIZE + r) * (size_t)(NU * 4 * U); };
    if constexpr (NL == 2)
        for (int i = threadIdx.x; i < NU * 4 * U; i += CL_THREADS) rec_at(0)[i] = rec_at(1)[i] = 0ull;   // no update has number 0
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);
    const uint32_t tm_g = tmem + CL_MAX_DIM / 2, tm_j = tm_g + 32, tm_j2 = tm_j + 80;   // gates: 16 columns; joint: two copies of up to 72
    const int q = warp & 3;                                                       // lane quadrant
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    if (warp < 8) cl_gate_rows_to_tmem<NL == 2 ? 5 : 1>(p.w_gate, p.P, r, warp, lane, tmem);
    asm volatile("cp.async.wait_all;" ::: "memory");
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    cl_barrier();                                                                 // every CTA's barriers are ready for remote stores

    bool ok = true;
    // every slot idle: all warps of the cluster leave in the same step
    auto all_idle = [&]() { return __all_sync(0xffffffffu, lane >= NU || (dec[min(lane, NU - 1)].flags & CL_IDLE) != 0u); };
    // slots that feed a token to their decoder in this step
    auto live_slots = [&]() { return __ballot_sync(0xffffffffu, lane < NU && dec[min(lane, NU - 1)].tok >= 0); };
    // ldmatrix address of the state: two K steps of 16 at a time, matrix = 8 slots x 8 columns, lane = (column piece, slot)
    constexpr uint32_t H_BLOCK = NL == 2 ? 1024u : 2048u;
    // With one slot the gates' product with the state (960 cycles, for the next step) comes behind the joint's, which it would hold up by
    // 350 of 8500.  Another CTA may be an update ahead by then, so there are two copies of the state, by parity of the updates (one more
    // update needs this CTA's h, and that this product).  With more slots a copy would lack the state of slots that sat an update out,
    // and from four on the joint's operand takes longer than the product.
    // One utterance of 100 s 2.10 -> 2.00 ms, seven short ones 0.595 -> 0.567.
    const bool late = NS == 1 && cl_gates_late(NU, NL);
    const uint32_t h_copy = late ? (uint32_t)kb_p * H_BLOCK : 0u;
    const uint32_t h_row = sbase + L.h + (uint32_t)((lane & 7) * 128);
    auto h_at = [&](int k32) { return h_row + (uint32_t)(k32 >> 1) * H_BLOCK + (uint32_t)((((k32 & 1) * 4 + (lane >> 3)) ^ (lane & 7)) << 4); };

    // The joint's operand z = act(enc_proj + pred_proj), in place, by every warp that computes (0..13).  It is bound by the shared
    // memory's bandwidth, so a 16-byte piece of pred_proj is loaded once for several window rows: a unit of work is eight threads, a
    // piece each of a K block, and p.z_rows of the rows of a group that count; units are dealt out evenly to all groups of eight threads.
    // (Eight slots, W = 8: 22 KB per group of eight rows; with pred_proj loaded for every row and rows dealt out by role it was 30 KB:
    // 128 utterances 9.75 -> 8.63 ms, 32 at W = 1 6.07 -> 5.65; one slot the same.)
    const int z_rows = p.wp == 8 ? p.W : 8;
    const int z_first = (int)(threadIdx.x >> 3) / kb_h << 8 | (int)(threadIdx.x >> 3) % kb_h;    // (group, part) << 8 | K block
    auto build_z = [&](auto which) {
        constexpr int AT_ONCE = decltype(which)::value;               // rows in flight per thread (the W_pred warps have registers for one)
        const uint32_t c = (uint32_t)(lane & 7);
#pragma unroll 1
        for (int at = z_first >> 8, kb = z_first & 255; at < n_groups << p.z_parts;) {
            const int gi = at >> p.z_parts, r0 = (at & ((1 << p.z_parts) - 1)) * p.z_rows, r1 = min(r0 + p.z_rows, z_rows);
            uint8_t* zp = smem + L.z + (uint32_t)(gi * p.H * 16 + kb * 1024);
            const uint4 y = *reinterpret_cast<const uint4*>(smem + L.pred + (uint32_t)(((gi << 3) >> wp_shift) * p.H * 2 + kb * 128) + c * 16u);
#pragma unroll 1
            for (int r = r0; r < r1; r += AT_ONCE) {
                uint4 x[AT_ONCE];
#pragma unroll
                for (int j = 0; j < AT_ONCE; ++j)
                    if (j == 0 || r + j < r1) x[j] = *reinterpret_cast<const uint4*>(zp + (uint32_t)((r + j) * 128) + ((c ^ (uint32_t)(r + j)) << 4));
#pragma unroll
                for (int j = 0; j < AT_ONCE; ++j)
                    if (j == 0 || r + j < r1)
                        *reinterpret_cast<uint4*>(zp + (uint32_t)((r + j) * 128) + ((c ^ (uint32_t)(r + j)) << 4)) =
                            make_uint4(act_add_bf16x2(x[j].x, y.x, ACT), act_add_bf16x2(x[j].y, y.y, ACT), act_add_bf16x2(x[j].z, y.z, ACT),
                                       act_add_bf16x2(x[j].w, y.w, ACT));
            }
            at += p.z_step >> 8;
            kb += p.z_step & 255;
            if (kb >= kb_h) { kb -= kb_h; ++at; }
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_z);
    };

    // Argmax of every window row over a share of this CTA's labels (HF), sent to the slots' owners.  With M = 64 accumulator row m
    // lives in lane m % 16 of quadrant m / 16.
    auto joint_argmax = [&](auto which) {
        constexpr int HF = decltype(which)::value;
        const int rows_here = (NU << wp_shift) - 16 * q;              // window rows of this warp's quadrant
        if (rows_here <= 0) return;
        constexpr int CH = HF ? 8 : 16;                                 // columns at a time (the W_pred warps have registers for eight)
        const int nh = (lab_n / 3) & ~7;                                // they take [0, nh), the workers [nh, lab_n)
        unsigned long long key;
        int row;
        bool mine;                                                      // this thread has the key of a row
        if constexpr (NS <= NL) {
            // Read as 16 lanes x 256 bits, a thread holds a quarter of the columns of rows lane / 4 and lane / 4 + 8, so that all 32 threads
            // have something to compare, and the exchanges at the end are few.  One utterance of 100 s 2.05 -> 2.00 ms, seven short ones 0.585 -> 0.572,
            // two layers with two slots 1.552 -> 1.540.
            float best[2] = {-INFINITY, -INFINITY};
            int lab[2] = {0, 0};
#pragma unroll 1
            for (int c = HF ? 0 : nh; c < (HF ? nh : lab_n); c += CH) {
                float v[CH / 2];                                        // of eight columns each: row lane / 4 twice, row lane / 4 + 8 twice
                tmem_ld_quarter<CH / 8>(tm_j + lane_off + (uint32_t)c, tm_j2 + lane_off + (uint32_t)c, v);
#pragma unroll
                for (int j = 0; j < CH / 8; ++j) {
                    const int at = c + 8 * j + 2 * (lane & 3);
                    const float2 b2 = *reinterpret_cast<const float2*>(s_bout + at); // -inf behind the last label
#pragma unroll
                    for (int k = 0; k < 2; ++k) {                       // equal logits: the lower label stays
                        const float v0 = v[4 * j + 2 * k] + b2.x, v1 = v[4 * j + 2 * k + 1] + b2.y;
                        if (v0 > best[k]) { best[k] = v0; lab[k] = at; }
                        if (v1 > best[k]) { best[k] = v1; lab[k] = at + 1; }
                    }
                }
            }
            unsigned long long keys[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                keys[k] = best[k] > -INFINITY ? pack_key(best[k], (uint32_t)(lab0 + lab[k])) : 0ull;
                if (k == 0 || rows_here > 8) {
                    keys[k] = max(keys[k], __shfl_xor_sync(0xffffffffu, keys[k], 1));
                    keys[k] = max(keys[k], __shfl_xor_sync(0xffffffffu, keys[k], 2));
                }
            }
            key = lane & 1 ? keys[1] : keys[0];
            row = 16 * q + (lane >> 2) + 8 * (lane & 1);                // lanes 4 i: row i, 4 i + 1: row i + 8
            mine = (lane & 2) == 0;
        } else {
            // A row a thread.  (Spread over the warp as above, steps of several slots took 5 % longer: 128 utterances 8.60 -> 9.04 ms, 32 at W = 1
            // 5.68 -> 5.94, two layers, 64 utterances, 12.77 -> 13.01.)  CH columns at a time: their maximum, then the lowest label that has it.
            float best = -INFINITY;
            int lab = 0;
#pragma unroll 1
            for (int c = HF ? 0 : nh; c < (HF ? nh : lab_n); c += CH) {
                float v[CH];
                if constexpr (CH == 16) tmem_ld16_sum(tm_j + lane_off + (uint32_t)c, tm_j2 + lane_off + (uint32_t)c, v);
                else tmem_ld8_sum(tm_j + lane_off + (uint32_t)c, tm_j2 + lane_off + (uint32_t)c, v);
#pragma unroll
                for (int j = 0; j < CH; j += 4) {
                    const float4 b4 = *reinterpret_cast<const float4*>(s_bout + c + j);  // -inf behind the last label
                    v[j] += b4.x; v[j + 1] += b4.y; v[j + 2] += b4.z; v[j + 3] += b4.w;
                }
                float m = v[0];
#pragma unroll
                for (int j = 1; j < CH; ++j) m = fmaxf(m, v[j]);
                int at = CH;
#pragma unroll
                for (int j = CH - 1; j >= 0; --j) at = v[j] == m ? j : at;
                if (m > best) { best = m; lab = c + at; }
            }
            key = best > -INFINITY ? pack_key(best, (uint32_t)(lab0 + lab)) : 0ull;
            row = 16 * q + (lane & 15);
            mine = lane < 16;
        }
        const int s = row >> wp_shift, w = row & (p.wp - 1);
        if (mine && s < NU && w < p.W)
            st_async_8(cl_map(sbase + L.kbuf + (uint32_t)(w * CL_KEY_PITCH + 2 * r + HF) * 8u, s), key, cl_map(smem_u32(&bar_keys), s));
    };

    if (warp < 4) {
        // =====================================================================================
        // workers: cell update, then the joint's operand
        // =====================================================================================
        const int e = threadIdx.x;                       // 0..127
        const int g = lane & 3, u = 8 * q + (lane >> 2); // gate and hidden unit (of the CTA's first 32) of this thread's accumulator lane
        const float sc = g == 2 ? 1.f : 0.5f, of = g == 2 ? 0.f : 0.5f;   // tanh, or the logistic function as 0.5 tanh(x / 2) + 0.5
        const float* g0 = p.g0 + (size_t)g * p.P + r * U + u;
        const float* g0r = p.g0 + r * U + 32 + (e & 7);
        const bool rem_on = has_rem && e < 64 && 32 + (e & 7) < U && (e >> 3) < NU;
        // h: 16-byte pieces of the CTA's part; a warp instruction serves 32 / lpd destinations with lpd lanes each
        const int h_pieces = NU * (U / 8);
        const int lpd_shift = h_pieces <= 8 ? 3 : (h_pieces <= 16 ? 4 : 5);
        const int h_first = lane & ((1 << lpd_shift) - 1);
        uint32_t h_src[2], h_dst[2];                     // h_src: slot in the top byte
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int i = h_first + 32 * k;
            const int uu = i / (U / 8), cc = i - uu * (U / 8), col = r * U + cc * 8;
            h_src[k] = (L.hst + (uint32_t)(uu * U + cc * 8) * 2u) | (uint32_t)uu << 24;
            h_dst[k] = L.h + (uint32_t)(col >> 6) * H_BLOCK + (uint32_t)(uu * 128 + ((((col >> 3) & 7) ^ (uu & 7)) << 4));
        }
        // cell state: (u, slots 2 g, 2 g + 1); (32 + (e & 7), slot e >> 3) for e < 64.  Two layers: kept in shared memory, [layer][3][e]
        float c_st[2] = {0.f, 0.f}, c_rem = 0.f;
        uint32_t updates = 0u;                           // (two layers)
        const bool timed = cluster == 0 && r == 0 && e == 0;
        unsigned long long ns0 = 0;
        if (timed) { ns0 = globaltimer_ns(); s_lap[3] = clock64(); }
        auto lap = [&](int k) { if (timed) { const long long now = clock64(); s_lap[k] += now - s_lap[3]; s_lap[3] = now; } };   // (no register to spare)

        // parities in one word (registers are short): bit 0 of the step, bit 1 of the updates so far, bit 2: there was one
        for (uint32_t st = 0u;; st ^= 1u) {
            const uint32_t par = st & 1u;
            // ---- decisions of the step; the gate table's rows are requested at once ----
            if (ok) ok = cl_wait(&bar_dec, par);
            if (ok && warp == 0 && lane == 0) mbar_expect_tx(&bar_dec, (uint32_t)NU * 16u);
            lap(0);
            const bool idle = all_idle();
            float add[NS], add_r[4];
            uint32_t fresh = 0u, live = 0u;
            {
                uint2 d[NS];                             // (token, flags); slots beyond NU never have a token
#pragma unroll
                for (int s = 0; s < NS; ++s) d[s] = *reinterpret_cast<const uint2*>(&dec[s]);
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    fresh |= (d[s].y & CL_FRESH) << s;
                    live |= (uint32_t)((int)d[s].x >= 0) << s;
                    add[s] = (int)d[s].x >= 0 && u < U ? g0[d[s].x * (uint32_t)(4 * p.P)] : 0.f;
                }
            }
            if (rem_on) {
                const int tok = dec[e >> 3].tok;
#pragma unroll
                for (int k = 0; k < 4; ++k) add_r[k] = tok >= 0 ? g0r[(uint32_t)tok * (uint32_t)(4 * p.P) + (uint32_t)(k * p.P)] : 0.f;
            }
            // ---- gates: recurrent term + gate table, cell update; the second layer: its product with the first one's new state,
            // recurrent term, biases ----
            bool leave = false;
#pragma unroll 1
            for (int l = 0; l < NL; ++l) {
            if (live != 0u) {
            __nv_bfloat16* hst = reinterpret_cast<__nv_bfloat16*>(smem + L.hst) + l * CL_SLOTS * U;
            float* c_mem = reinterpret_cast<float*>(smem + L.cell) + l * 3 * 128 + e;
            if (l == 0) {
                if (ok && warp == 0 && lane == 0) {
                    mbar_expect_tx(&bar_pred, (uint32_t)(__popc(live) * p.H) * 2u);
                    if constexpr (NL == 2) mbar_expect_tx(&bar_h0, (uint32_t)(__popc(live) * p.P) * 2u);
                }
                if (st & 4u) {
                    if constexpr (NL == 1) {
                        if (ok) ok = cl_wait(&bar_acc_g, (~st >> 1) & 1u);
                        if (has_rem && ok) ok = cl_wait(&bar_acc_r, (~st >> 1) & 1u);
                    }
                }
            }
            float rec[NS], rec_r[4] = {0.f, 0.f, 0.f, 0.f};              // two layers: the recurrent term
            if constexpr (NL == 2) {
#pragma unroll
                for (int s = 0; s < NS; ++s) rec[s] = 0.f;
                // (of slots that start afresh too, for which it does not count: the next request has to follow the answer to the last)
                const bool want_r = rem_on && ((live >> (e >> 3)) & 1u);
                if (l == 0) {
                    const float* mine = reinterpret_cast<const float*>(smem + L.rec);
                    if (st & 4u) {
                        if (ok) ok = cl_wait(&bar_rec, (~st >> 1) & 1u);
#pragma unroll
                        for (int s = 0; s < NS; ++s)
                            if (u < U && s < NU) rec[s] = mine[s * 4 * U + e];
                        if (want_r) {
                            const float4 v = *reinterpret_cast<const float4*>(mine + (e >> 3) * 4 * U + 128 + 4 * (e & 7));
                            rec_r[0] = v.x; rec_r[1] = v.y; rec_r[2] = v.z; rec_r[3] = v.w;
                        }
                    }
                } else if ((st & 4u) && ok) {
                    const unsigned long long* mine = rec_at(1);
                    ok = cl_read_stamped<NS>(mine + e, (uint32_t)(4 * U), u < U ? live : 0u, updates, rec, &p.ctrl->abort,
                                             mine + (e >> 3) * 4 * U + 128 + 4 * (e & 7), want_r, rec_r);
                }
            }
            if (l == 1) {
                if (ok) ok = cl_wait(&bar_acc_g, (st >> 1) & 1u);
                if (has_rem && ok) ok = cl_wait(&bar_acc_r, (st >> 1) & 1u);
            }
            tc_fence_after();
            {
                float x[8];
                if (NL == 1 || l == 1) tmem_ld8(tm_g + lane_off, x);
                if (NL == 2) {
                    const float bias = l == 1 && u < U ? reinterpret_cast<const float*>(smem + L.b_gate)[e] : 0.f;
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        const float rs = (fresh >> s) & 1u ? 0.f : rec[s];
                        if (l == 0) x[s] = rs;
                        else add[s] = rs + bias;
                    }
                }
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    if (s < NS) x[s] = fmaf(tanh_fast(((NL == 1 && ((fresh >> s) & 1u) ? 0.f : x[s]) + add[s]) * sc), sc, of);
                    else x[s] = 0.f;
                }
                // lane 4 u + g holds gate g of all slots; it is to hold the four gates of slots 2 g and 2 g + 1
                const bool up2 = (g & 2) != 0, up1 = (g & 1) != 0;
                float a[4], b[4];
#pragma unroll
                for (int j = 0; j < (NS < 4 ? NS : 4); ++j) {
                    a[j] = up2 ? x[4 + j] : x[j];
                    b[j] = __shfl_xor_sync(0xffffffffu, up2 ? x[j] : x[4 + j], 2);    // the same slots, gate g ^ 2
                }
#pragma unroll
                for (int j = NS < 4 ? NS : 4; j < 4; ++j) a[j] = b[j] = 0.f;
#pragma unroll
                for (int k = 0; k < (NS < 2 ? NS : 2); ++k) {
                    float own = up1 ? a[2 + k] : a[k], g2 = up1 ? b[2 + k] : b[k];
                    float g1 = __shfl_xor_sync(0xffffffffu, up1 ? a[k] : a[2 + k], 1), g3 = __shfl_xor_sync(0xffffffffu, up1 ? b[k] : b[2 + k], 1);
                    if (up1) { float t = own; own = g1; g1 = t; t = g2; g2 = g3; g3 = t; }
                    if (up2) { float t = own; own = g2; g2 = t; t = g1; g1 = g3; g3 = t; }
                    const float gi = own, gf = g1, gg = g2, go = g3;
                    const int s = 2 * g + k;
                    if (u < U && s < NU && ((live >> s) & 1u)) {
                        if constexpr (NL == 2) c_st[k] = c_mem[k * 128];
                        const float cold = (fresh >> s) & 1u ? 0.f : c_st[k];
                        const float cc = cell_update(gf, cold, gi, gg);
                        c_st[k] = cc;
                        if constexpr (NL == 2) c_mem[k * 128] = cc;
                        hst[s * U + u] = __float2bfloat16_rn(go * tanh_fast(cc));
                    }
                }
            }
            if (rem_on) {
                const int s = e >> 3;
                if ((live >> s) & 1u) {
                    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (NL == 1 || l == 1) x = *reinterpret_cast<const float4*>(gr + s * CL_GR_PITCH + 4 * (e & 7));
                    if (NL == 2) {
                        if ((fresh >> s) & 1u) rec_r[0] = rec_r[1] = rec_r[2] = rec_r[3] = 0.f;
                        if (l == 0) x = make_float4(rec_r[0], rec_r[1], rec_r[2], rec_r[3]);
                        else {
                            const float4 bias = *reinterpret_cast<const float4*>(smem + L.b_gate + 512 + 16 * (e & 7));
                            add_r[0] = rec_r[0] + bias.x; add_r[1] = rec_r[1] + bias.y; add_r[2] = rec_r[2] + bias.z; add_r[3] = rec_r[3] + bias.w;
                        }
                    } else if ((fresh >> s) & 1u) x = make_float4(0.f, 0.f, 0.f, 0.f);
                    const float gi = fmaf(tanh_fast((x.x + add_r[0]) * 0.5f), 0.5f, 0.5f);
                    const float gf = fmaf(tanh_fast((x.y + add_r[1]) * 0.5f), 0.5f, 0.5f);
                    const float gg = fmaf(tanh_fast((x.z + add_r[2]) * 1.f), 1.f, 0.f);
                    const float go = fmaf(tanh_fast((x.w + add_r[3]) * 0.5f), 0.5f, 0.5f);
                    if constexpr (NL == 2) c_rem = c_mem[2 * 128];
                    const float cold = (fresh >> s) & 1u ? 0.f : c_rem;
                    const float cc = cell_update(gf, cold, gi, gg);
                    c_rem = cc;
                    if constexpr (NL == 2) c_mem[2 * 128] = cc;
                    hst[s * U + 32 + (e & 7)] = __float2bfloat16_rn(go * tanh_fast(cc));
                }
            }
            tc_fence_before();
            }
            if (group_barrier_or<128>(1, !ok || idle)) { leave = true; break; }
            // h to all CTAs
            const uint32_t h_from = NL == 2 ? (uint32_t)(l * CL_SLOTS * U) * 2u : 0u, h_to = NL == 2 && l == 0 ? L.h0 - L.h : ((st >> 1) & 1u) * h_copy;
            const uint32_t h_bar = NL == 2 && l == 0 ? smem_u32(&bar_h0) : smem_u32(&bar_h);
#pragma unroll
            for (int k = 0; k < 2; ++k)
                if (h_first + 32 * k < h_pieces && ((live >> (h_src[k] >> 24)) & 1u)) {
                    const uint4 piece = *reinterpret_cast<const uint4*>(smem + (h_src[k] & 0xFFFFFFu) + h_from);
                    for (int d0 = warp * (32 >> lpd_shift) + (lane >> lpd_shift); d0 < CL_SIZE; d0 += 128 >> lpd_shift) {
                        const uint32_t d = (uint32_t)(d0 + r) & (CL_SIZE - 1);
                        st_async_16(cl_map(sbase, d) + h_dst[k] + h_to, piece, cl_map(h_bar, d));
                    }
                }
            if constexpr (NL == 2) {
                if (live == 0u) break;
                // and, for the next step's recurrent term, to the cluster that has the layer's W_hh
                if (warp == 3) {
#pragma unroll
                    for (int k = 0; k < 2; ++k)
                        if (lane == h_first && h_first + 32 * k < h_pieces) {
                            const uint32_t off = h_src[k] & 0xFFFFFFu, s = h_src[k] >> 24;
                            const uint32_t row = (uint32_t)((cluster * 2 + l) * 2 + (int)((st >> 1) & 1u)) * 8u + s;
                            *reinterpret_cast<uint4*>(p.hx + (size_t)row * p.P + r * U + ((off - L.hst) / 2u - s * (uint32_t)U)) = *reinterpret_cast<const uint4*>(smem + off + h_from);
                        }
                    fence_proxy_async_all();
                    __syncwarp();
                    if (lane == 0) red_release_add(p.req + l * CL_DECODERS + cluster, 1u);
                }
            }
            }
            if (leave) break;
            if (live != 0u) { st = (st ^ 2u) | 4u; ++updates; }
            lap(1);
            // ---- the joint's operand z = act(enc_proj + pred_proj), in place ----
            if (ok) ok = cl_wait(&bar_enc, par);
            if (ok) ok = cl_wait(&bar_pred, (~st >> 1) & 1u);        // of the last update: this step's, or long there
            lap(2);
            build_z(std::integral_constant<int, 4>{});
            if (ok) ok = cl_wait(&bar_acc_j, par);
            tc_fence_after();
            joint_argmax(std::integral_constant<int, 0>{});
        }
        if (timed) {
            p.ctrl->active = 0;
            p.ctrl->loop_kernel = WIND_LOOP_CLUSTERS;
            for (int k = 0; k < 3; ++k) p.ctrl->phase_cycles[k] = s_lap[k];
            p.ctrl->loop_ns = (long long)(globaltimer_ns() - ns0);
        }
    } else if (warp < 10) {
        // =====================================================================================
        // W_pred: (K half, 16 joint units) per warp, pred_proj[unit, slot] = W_pred h^T
        // =====================================================================================
        const int half = (warp - 4) / 3, mt = (warp - 4) % 3;
        const int k16s = p.P / 32;                       // K steps of 16 in a half: at most 20
        const bool mine = mt * 16 < HS;
        uint32_t wf[20][4];                              // (rows behind the last one repeat it: their results go nowhere)
        {
            const uint32_t* r0 = reinterpret_cast<const uint32_t*>(p.w_pred + (size_t)(r * HS + min(16 * mt + (lane >> 2), HS - 1)) * p.P + half * (p.P / 2)) + (lane & 3);
            const uint32_t* r1 = reinterpret_cast<const uint32_t*>(p.w_pred + (size_t)(r * HS + min(16 * mt + (lane >> 2) + 8, HS - 1)) * p.P + half * (p.P / 2)) + (lane & 3);
#pragma unroll
            for (int s0 = 0; s0 < 20; s0 += 4)
                if (s0 < k16s)
#pragma unroll
                    for (int s = s0; s < s0 + 4; ++s) { wf[s][0] = r0[s * 8]; wf[s][1] = r1[s * 8]; wf[s][2] = r0[s * 8 + 4]; wf[s][3] = r1[s * 8 + 4]; }
        }
        float4* part = reinterpret_cast<float4*>(smem + L.part) + mt * 32 + lane;
        __nv_bfloat16* pst = reinterpret_cast<__nv_bfloat16*>(smem + L.pst) + 16 * mt;     // [slot][48]
        const int halves = min(2, (HS - 16 * mt) / 8);   // 16-byte pieces of a slot in this warp's 16 units
        for (uint32_t st = 0u;; st ^= 1u) {              // bit 0: parity of the step, bit 1: of the updates so far
            const uint32_t par = st & 1u;
            if (ok) ok = cl_wait(&bar_dec, par);
            const bool idle = all_idle();
            const uint32_t live = live_slots();
            if (ok && live != 0u && warp == 4 && lane == 0) mbar_expect_tx(&bar_h, (uint32_t)(__popc(live) * p.P) * 2u);
            if (live != 0u) st ^= 2u;
            if (ok) ok = cl_wait(&bar_h, (~st >> 1) & 1u);           // of the last update: this step's, or long there
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
            if (mine && live != 0u) {
                uint32_t b[2][4];
                const uint32_t copy = ((~st >> 1) & 1u) * h_copy;
                ldmatrix_x4(b[0], h_at(half * (k16s / 2)) + copy);
                // (the state rows of the next two steps are requested a turn early; at the end they are rows nobody uses)
#pragma unroll
                for (int s0 = 0; s0 < 20; s0 += 4)
                    if (s0 < k16s)
#pragma unroll
                        for (int s = s0; s < s0 + 4; s += 2) {
                            ldmatrix_x4(b[(s / 2 + 1) & 1], h_at(half * (k16s / 2) + s / 2 + 1) + copy);
                            mma_16816(acc, wf[s][0], wf[s][1], wf[s][2], wf[s][3], b[(s / 2) & 1][0], b[(s / 2) & 1][1]);
                            mma_16816(acc, wf[s + 1][0], wf[s + 1][1], wf[s + 1][2], wf[s + 1][3], b[(s / 2) & 1][2], b[(s / 2) & 1][3]);
                        }
                if (half) *part = make_float4(acc[0], acc[1], acc[2], acc[3]);
            }
            if (group_barrier_or<192>(2, !ok || idle)) break;
            if (NL == 1 && lane == 0 && live != 0u) mbar_arrive(&bar_sync_mma);
            if (half == 0 && mine && live != 0u) {
                // the two K halves are added as loop_kernel adds its accumulators
                const float4 o = *part;
                const int m = lane >> 2, s = (lane & 3) * 2;
                const float b0 = s_bpred[16 * mt + m], b1 = s_bpred[16 * mt + m + 8];
                pst[s * 48 + m] = __float2bfloat16_rn(acc[0] + o.x + b0);
                pst[(s + 1) * 48 + m] = __float2bfloat16_rn(acc[1] + o.y + b0);
                pst[s * 48 + m + 8] = __float2bfloat16_rn(acc[2] + o.z + b1);
                pst[(s + 1) * 48 + m + 8] = __float2bfloat16_rn(acc[3] + o.w + b1);
                __syncwarp();
                // 16-byte pieces of eight units of one slot: message i = (piece, destination)
                if constexpr (NS <= 2)
                for (int i = lane; i < NU * halves * CL_SIZE; i += 32) {
                    const int pi = i >> 4, sl = halves == 2 ? pi >> 1 : pi, hh = halves == 2 ? pi & 1 : 0;
                    const uint32_t d = (uint32_t)(i + r) & (CL_SIZE - 1);
                    if ((live >> sl) & 1u) st_async_16(cl_map(sbase, d) + L.pred + (uint32_t)(sl * p.H + r * HS + 16 * mt + 8 * hh) * 2u,
                                *reinterpret_cast<const uint4*>(pst + sl * 48 + 8 * hh), cl_map(smem_u32(&bar_pred), d));
                }
            }
            if constexpr (NS > 2) {
                // many slots: all six warps send, a destination at a time each, a piece per lane
                if (live != 0u) {
                    asm volatile("bar.sync 2, 192;" ::: "memory");
                    const int per_slot = HS / 8;
#pragma unroll 1
                    for (int i = lane; i < NU * per_slot; i += 32) {
                        const int sl = i / per_slot, c = i - sl * per_slot;
                        if ((live >> sl) & 1u) {
                            const uint4 piece = *reinterpret_cast<const uint4*>(smem + L.pst + (uint32_t)(sl * 48 + 8 * c) * 2u);
                            for (int d0 = warp - 4; d0 < CL_SIZE; d0 += 6) {
                                const uint32_t d = (uint32_t)(d0 + r) & (CL_SIZE - 1);
                                st_async_16(cl_map(sbase, d) + L.pred + (uint32_t)(sl * p.H + r * HS + 8 * c) * 2u, piece, cl_map(smem_u32(&bar_pred), d));
                            }
                        }
                    }
                }
            }
            if (ok) ok = cl_wait(&bar_enc, par);
            if (ok) ok = cl_wait(&bar_pred, (~st >> 1) & 1u);
            build_z(std::integral_constant<int, 1>{});
            if (warp < 8) {
                if (ok) ok = cl_wait(&bar_acc_j, par);
                tc_fence_after();
                joint_argmax(std::integral_constant<int, 1>{});
                tc_fence_before();
            }
        }
    } else if (warp < 14) {
        // =====================================================================================
        // remainder units 32..: W_hh rows of units 32 + 2 k, + 1 (4 gates each: row 4 (u - 32) + gate) in warp 10 + k, one chain
        // over all of K (as the gates' accumulator in loop_kernel), [slot, row] = h W_hh^T.  Two layers: W_ih of the second one, and
        // behind the joint's operand these warps fetch the first layer's recurrent term, which the update of the next step begins with
        // (fetched there it cost 600 to 1000 cycles; the second layer's is fetched under the product with the first one's new state)
        // =====================================================================================
        if (rem_warps) {
            uint32_t updates = 0u;
            const int row = 8 * (warp - 10) + (lane >> 2), u = 32 + (row >> 2), g = row & 3;
            uint32_t wf[40][2];
            const uint32_t* src = reinterpret_cast<const uint32_t*>(p.w_gate + ((size_t)g * p.P + r * U + min(u, U - 1)) * p.P) + (lane & 3);
#pragma unroll
            for (int s0 = 0; s0 < 40; s0 += 8)
                if (s0 < p.P / 16)
#pragma unroll
                    for (int s = s0; s < s0 + 8; ++s) { wf[s][0] = src[s * 8]; wf[s][1] = src[s * 8 + 4]; }
            for (uint32_t st = 0u;; st ^= 1u) {          // bit 0: parity of the step, bit 1: of the updates so far
                const uint32_t par = st & 1u;
                ok = cl_wait_warp(&bar_dec, par);
                if (all_idle() || !ok) break;
                const bool update = live_slots() != 0u;
                if (update) st ^= 2u;
                if (update && has_rem) {
                ok = cl_wait_warp(NL == 2 ? &bar_h0 : &bar_h, (~st >> 1) & 1u);
                if (!ok) break;
                float acc[4] = {0.f, 0.f, 0.f, 0.f};
                uint32_t a[2][4];
                const uint32_t copy = NL == 2 ? L.h0 - L.h : ((~st >> 1) & 1u) * h_copy;     // two layers: the first one's state
                ldmatrix_x4(a[0], h_at(0) + copy);
#pragma unroll
                for (int s0 = 0; s0 < 40; s0 += 8)
                    if (s0 < p.P / 16)
#pragma unroll
                        for (int s = s0; s < s0 + 8; s += 2) {
                            ldmatrix_x4(a[(s / 2 + 1) & 1], h_at(s / 2 + 1) + copy);
                            mma_16816(acc, a[(s / 2) & 1][0], 0u, a[(s / 2) & 1][1], 0u, wf[s][0], wf[s][1]);
                            mma_16816(acc, a[(s / 2) & 1][2], 0u, a[(s / 2) & 1][3], 0u, wf[s + 1][0], wf[s + 1][1]);
                        }
                *reinterpret_cast<float2*>(gr + (lane >> 2) * CL_GR_PITCH + (warp - 10) * 8 + (lane & 3) * 2) = make_float2(acc[0], acc[1]);
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&bar_acc_r);
                    if constexpr (NL == 1) mbar_arrive(&bar_sync_mma);
                }
                }
                ok = cl_wait_warp(&bar_enc, par) && cl_wait_warp(&bar_pred, (~st >> 1) & 1u);
                if (!ok) break;
                build_z(std::integral_constant<int, 1>{});
                if constexpr (NL == 2) {
                    if (update) {
                        constexpr int AT_ONCE = NS <= 2 ? 3 : 5;
                        const unsigned long long* src = rec_at(0);
                        float* dst = reinterpret_cast<float*>(smem + L.rec);
                        ++updates;
                        for (int i = (int)threadIdx.x - 320; ok && i - lane < NU * 4 * U; i += 128 * AT_ONCE) {
                            const int n_at = (NU * 4 * U - i + 127) >> 7;             // values of this thread's from i on (may be below 1)
                            float v[AT_ONCE];
                            ok = cl_read_stamped<AT_ONCE>(src + i, 128u, n_at >= AT_ONCE ? (1u << AT_ONCE) - 1u : (1u << max(n_at, 0)) - 1u, updates, v, &p.ctrl->abort);
#pragma unroll
                            for (int k = 0; k < AT_ONCE; ++k)
                                if (k < n_at) dst[i + 128 * k] = v[k];
                        }
                        __syncwarp();
                        if (!ok) break;
                        if (lane == 0) mbar_arrive(&bar_rec);
                    }
                }
            }
        }
    } else if (warp == 14) {
        // =====================================================================================
        // issuing thread: the window's enc_proj rows, the gates' MMAs on the new state (a step ahead of their use), the joint's
        // =====================================================================================
        if (elect_one()) {
            const uint32_t id_g = idesc_bf16(128, 16), id_j = idesc_bf16(64, lab_n);
            // z: eight-row groups H * 16 bytes apart (each a TMA box: K blocks of 8 rows x 128 bytes)
            const uint64_t ad0 = (smem_desc_sw128(sbase + L.z) & ~((uint64_t)0x3FFF << 32)) | ((uint64_t)(uint32_t)p.H << 32);
            uint32_t n_g = 0u;
            for (uint32_t step = 0;; ++step) {
                const uint32_t par = step & 1u;
                if (!(ok = cl_wait(&bar_dec, par))) break;
                uint32_t idle = CL_IDLE;
                bool update = false;
#pragma unroll 1
                for (int s = 0; s < NU; ++s) { idle &= dec[s].flags; update = update || dec[s].tok >= 0; }
                if (idle) break;
                mbar_expect_tx(&bar_enc, (uint32_t)(n_groups * p.H * 16));
#pragma unroll 1
                for (int gi = 0; gi < n_groups; ++gi) {
                    const int s = (gi << 3) >> wp_shift;
                    tma_load_3d(smem + L.z + (uint32_t)(gi * p.H * 16), &enc_map, 0, (int)dec[s].row + ((gi << 3) & (p.wp - 1)), 0, &bar_enc);
                }
                auto gates = [&]() {
                    // mma.sync and tcgen05.mma exclude each other on the tensor cores: the short chains go first (when they are
                    // done, all of h is there as well)
                    if (!(ok = cl_wait(NL == 1 ? &bar_sync_mma : &bar_h0, n_g & 1u))) return;
                    fence_proxy_async_all();             // h came in through remote generic stores
                    tc_fence_after();
                    uint64_t hd = smem_desc_sw128(sbase + (NL == 2 ? L.h0 : L.h + (n_g & 1u) * h_copy));
#pragma unroll 1
                    for (int kb = 0; kb < kb_p; ++kb, hd += H_BLOCK >> 4)
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            tc_mma_bf16_ts(tm_g, tmem + (uint32_t)(kb * 32 + k * 8), hd + (uint64_t)(k * 2), id_g, (kb | k) != 0);
                    tc_commit(&bar_acc_g);
                    ++n_g;
                };
                if (!late && update) { gates(); if (!ok) break; }
                if (!(ok = cl_wait(&bar_z, par))) break;
                tc_fence_after();
                uint64_t bd = smem_desc_sw128(sbase + L.w_out), ad = ad0;
#pragma unroll 1
                for (int kb = 0; kb < kb_h; ++kb, bd += (uint64_t)(lab_rows * 8), ad += 1024 >> 4) {
                    const bool second = kb >= kb_h / 2;  // K halves in two accumulator copies, as in loop_kernel
                    const uint32_t d = second ? tm_j2 : tm_j;
                    tc_mma_bf16(d, ad, bd, id_j, kb != (second ? kb_h / 2 : 0));
#pragma unroll
                    for (int k = 1; k < 4; ++k) tc_mma_bf16(d, ad + (uint64_t)(k * 2), bd + (uint64_t)(k * 2), id_j, 1u);
                }
                tc_commit(&bar_acc_j);
                if (late && update) { gates(); if (!ok) break; }
            }
            // copies and MMAs in flight must have completed before the memory they use goes back
            if (n_g > 0u) cl_wait(&bar_acc_g, (n_g - 1u) & 1u);
            if (!ok) s_abort = 1 + 14;
        }
        __syncwarp();
        ok = true;
    } else if (r < NU) {
        // =====================================================================================
        // control: CTA u < NU owns slot u (every lane holds the same values)
        // =====================================================================================
        const bool dynamic = p.n_utt > NU * n_clusters;
        int o_utt = -1, o_t = 0, o_len = 0, o_cnt = 0, o_pos = 0;
        uint32_t o_row0 = 0u, n_steps = 0u;
        unsigned long long n_rows = 0ull, n_tok = 0ull, n_forced = 0ull;
        auto take = [&](int k) {                         // utterance k of the order, or, when it is empty or there is none, the next of the queue
            for (;;) {
                o_utt = -1; o_len = 0; o_t = 0; o_cnt = 0; o_pos = 0; o_row0 = 0u;
                if (k >= 0 && k < p.n_utt) {
                    o_utt = p.order ? p.order[k] : k;
                    o_len = min(max(p.enc_len[o_utt], 0), p.T);
                    o_row0 = (uint32_t)o_utt * (uint32_t)p.T;
                    if (o_len > 0) return;
                }
                if (!dynamic || k >= p.n_utt) { o_utt = -1; return; }
                int v = 0;
                if (lane == 0) v = atomicAdd(&p.ctrl->next_utt, 1);
                k = __shfl_sync(0xffffffffu, v, 0) - p.queue_base + NU * n_clusters;
            }
        };
        auto announce = [&](int tok, bool fresh, uint32_t odd) {       // the slot's decision to every CTA
            const bool idle = o_utt < 0;
            const uint4 m = make_uint4((uint32_t)(idle ? -1 : tok), (fresh ? CL_FRESH : 0u) | (idle ? CL_IDLE : 0u) | odd * CL_ODD,
                                       idle ? 0u : o_row0 + (uint32_t)o_t, 0u);
            if (lane < CL_SIZE) st_async_16(cl_map(sbase + L.dec + (uint32_t)r * 16u, lane), m, cl_map(smem_u32(&bar_dec), lane));
        };
        take(r * n_clusters + cluster);
        announce(p.blank, true, 0u);
        for (uint32_t step = 0;; ++step) {
            const uint32_t par = step & 1u;
            ok = cl_wait_warp(&bar_dec, par);
            // Every slot idle, as all_idle, but of this step's decisions alone: nothing waits for this warp's look at dec, so the
            // owners of the other slots may have overwritten theirs with the next step's (this slot's comes from this warp).  Where
            // there is a next step, this one is not the last.
            const bool last = __all_sync(0xffffffffu, lane >= NU || (dec[min(lane, NU - 1)].flags & (CL_IDLE | CL_ODD)) == (CL_IDLE | par * CL_ODD));
            if (last || !ok) break;
            ok = cl_wait_warp(&bar_keys, par);
            if (!ok) break;
            if (lane == 0) mbar_expect_tx(&bar_keys, (uint32_t)(2 * CL_SIZE * p.W) * 8u);
            // lane = (window row, a share of the 32 keys of that row)
            const ulonglong2* kp = reinterpret_cast<const ulonglong2*>(
                smem + L.kbuf + (uint32_t)((lane & (p.wp - 1)) * CL_KEY_PITCH + (lane >> wp_shift) * p.wp) * 8u);
            unsigned long long key = 0ull;
#pragma unroll 1
            for (int i = 0; i < p.wp / 2; i += 4) {
                const ulonglong2 k0 = kp[i], k1 = kp[i + 1], k2 = kp[i + 2], k3 = kp[i + 3];
                const unsigned long long m0 = max(max(k0.x, k0.y), max(k1.x, k1.y)), m1 = max(max(k2.x, k2.y), max(k3.x, k3.y));
                key = max(key, max(m0, m1));
            }
            for (int o = p.wp; o < 32; o <<= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
            const int n = o_utt >= 0 ? min(p.W, o_len - o_t) : 0;        // an idle slot: no rows, nothing to record
            uint32_t label = key_label(key);
            const bool broken = key == 0ull || label >= (uint32_t)p.NV;
            if (broken) label = (uint32_t)p.blank;
            const uint32_t hit = __ballot_sync(0xffffffffu, lane < n && (int)label != p.blank);
            const int first = hit ? __ffs((int)hit) - 1 : n;             // all blank: past the whole window
            const int lab = (int)__shfl_sync(0xffffffffu, label, first & 31);
            const int pos = o_pos, utt = o_utt;
            const bool emit = hit && pos < p.max_out, overflow = hit && pos >= p.max_out;
            int t = o_t + first;
            const int t_emit = t;
            if (first > 0) o_cnt = 0;
            o_cnt += emit;
            const bool forced = emit && o_cnt == p.S;
            if (forced) { ++t; o_cnt = 0; }
            o_pos += emit;
            o_t = overflow ? o_len : t;                                  // no room for the token: this utterance stops here
            n_steps += utt >= 0;
            const bool stuck = n_steps >= (uint32_t)p.step_cap;
            const bool done = utt >= 0 && (o_t >= o_len || stuck);
            if (done) {
                // finished: the slot takes the next utterance in this very step
                if (lane == 0) {
                    p.out_len[utt] = o_pos;
                    if (o_t < o_len) set_status(p.ctrl, WIND_ERR_INTERNAL);
                }
                take(dynamic && !stuck ? -1 : p.n_utt);
            }
            announce(done ? p.blank : (emit ? lab : -1), done, par ^ 1u);          // what the step decided is recorded behind the answer
            const uint32_t bad = __ballot_sync(0xffffffffu, lane < n && lane <= first && broken);   // rows after the first non-blank one do not count
            n_rows += (unsigned)n; n_tok += emit; n_forced += forced;
            if (NL == 2 && r == 0 && (step & 1023u) == 1023u && lane == 0) st_relaxed_u32(p.beat + cluster, step);
            if (lane == 0 && utt >= 0) {
                s_hist[first] += 1;
                if (emit) {
                    p.out_tokens[(size_t)utt * p.max_out + pos] = lab;
                    p.out_frames[(size_t)utt * p.max_out + pos] = t_emit;
                }
                if (overflow) set_status(p.ctrl, WIND_ERR_OUTPUT_OVERFLOW);
                if (bad) set_status(p.ctrl, WIND_ERR_INTERNAL);
            }
        }
        if (lane == 0 && n_steps > 0u) {
            atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->joint_rows), n_rows);
            atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->tokens), n_tok);
            atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->forced), n_forced);
            atomicMax(&p.ctrl->step, (int)n_steps);
#pragma unroll 1
            for (int k = 0; k < 65; ++k)
                if (s_hist[k]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->jump_hist[k]), (unsigned long long)s_hist[k]);
        }
    }
    if (!ok) s_abort = 1 + warp;
    tc_fence_before();
    __syncthreads();
    if (warp == 14) {
        tc_fence_after();
        tmem_dealloc(tmem, LOOP_TMEM_COLS);
    }
    if (threadIdx.x == 0) {
        if (s_abort) {
            note_timeout(p.ctrl, 49 + s_abort, blockIdx.x);
            set_status(p.ctrl, WIND_ERR_TIMEOUT);
            if constexpr (NL == 2) atomicExch(&p.ctrl->abort, 1);
        }
        if constexpr (NL == 2) red_release_add(p.done + cluster, 1u);
    }
    __syncwarp();
    cl_barrier();                                        // no CTA leaves while another may still write into its shared memory
}

// ---------------------------------------------------------------------------
// order of the utterances: longest first, so that the queue's tail is short (equal lengths keep their order)
// ---------------------------------------------------------------------------
constexpr int CL_ORDER_MAX = 4096;
__global__ void __launch_bounds__(1024) cl_order_kernel(const int32_t* __restrict__ enc_len, int n, int32_t* __restrict__ order) {
    __shared__ int32_t len[CL_ORDER_MAX];
    for (int i = threadIdx.x; i < n; i += 1024) len[i] = enc_len[i];
    __syncthreads();
    for (int i = blockIdx.x * 1024 + threadIdx.x; i < n; i += gridDim.x * 1024) {
        const int mine = len[i];
        int rank = 0;
        for (int j = 0; j < n; ++j) rank += len[j] > mine || (len[j] == mine && j < i);
        order[rank] = i;
    }
}

// Whether the other kernel that could take this decode (grid barriers, arrival counters or streamed weights, as the planner has it)
// is the better one for these lengths.  The clusters decode `slots` utterances at a time and take the next from the queue, longest
// first, in steps of cl_us; the other kernel decodes all `rows` at a time (refilled in the caller's order) in steps of other_us.
// Bounds of what either schedule takes mostly decide; where they overlap, a warp each plays them through: every utterance goes to
// the place that is free first.  (128 utterances of 2400 to 2500 frames, W = 8: 19.9 ms in clusters, three rounds of 56 slots,
// against 15.0; of 125 to 2500 frames: 8.3 against 13.4.)
constexpr int CL_CHOOSE_ROWS = 512;
__global__ void __launch_bounds__(256) cl_choose_kernel(Ctrl* ctrl, const int32_t* __restrict__ enc_len, const int32_t* __restrict__ order, int n, int T,
                                                        int slots, int rows, float cl_us, float other_us) {
    __shared__ uint32_t free_at[2][CL_CHOOSE_ROWS];      // frames until the place is free << 9 | place
    __shared__ uint32_t s_span[2];
    __shared__ unsigned long long s_sum;
    __shared__ int s_longest;
    if (threadIdx.x == 0) { s_sum = 0ull; s_longest = 0; }
    __syncthreads();
    auto length = [&](int u) { return min(max(enc_len[u], 0), T); };
    unsigned long long mine_sum = 0ull;
    int mine_longest = 0;
    for (int i = threadIdx.x; i < n; i += 256) { const int l = length(i); mine_sum += (unsigned long long)l; mine_longest = max(mine_longest, l); }
    atomicAdd(&s_sum, mine_sum);
    atomicMax(&s_longest, mine_longest);
    __syncthreads();
    // all rows of the other kernel wait for the slowest, a slot averages over its utterances: 1.14 times the mean number of steps
    // at 200 frames, 1.28 at 120 (128 utterances of equal length)
    auto other_cost = [&](float span) { return other_us * span * (1.f + 2.5f * rsqrtf(fmaxf(span, 1.f))); };
    const bool queue = n > rows;
    const float longest = (float)s_longest, sum = (float)s_sum, next = (float)(order && n > slots ? length(order[slots]) : s_longest);
    const float cl_lo = fmaxf(longest, sum / (float)slots), cl_hi = fmaxf(longest, sum / (float)slots + next);
    const float other_lo = queue ? fmaxf(longest, sum / (float)rows) : longest, other_hi = queue ? longest + sum / (float)rows : longest;
    const bool clusters = cl_us * cl_hi <= other_cost(other_lo), other = cl_us * cl_lo > other_cost(other_hi);
    if (clusters || other || n > CL_ORDER_MAX || (queue && rows > CL_CHOOSE_ROWS)) {
        if (threadIdx.x == 0) ctrl->use_grid = clusters ? 0 : (other ? 1 : cl_us * (cl_lo + cl_hi) > 2.f * other_cost(0.5f * (other_lo + other_hi)));
        return;
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, places = w == 0 ? slots : rows;
    if (w == 0 || (w == 1 && queue)) {
        uint32_t* f = free_at[w];
        for (int i = lane; i < CL_CHOOSE_ROWS; i += 32) f[i] = i < places ? (uint32_t)i : 0xffffffffu;
        uint32_t span = 0u, mine_free = lane < places ? (uint32_t)lane : 0xffffffffu;
        for (int j0 = 0; j0 < n; j0 += 32) {
            const int j = j0 + lane;
            const uint32_t mine = j < n ? (uint32_t)length(w == 0 && order ? order[j] : j) : 0u;
            for (int k = 0; k < 32 && j0 + k < n; ++k) {
                const uint32_t best = __reduce_min_sync(0xffffffffu, mine_free);
                const uint32_t end = min((best >> 9) + __shfl_sync(0xffffffffu, mine, k), 0x7ffffeu);
                span = max(span, end);
                if (best == mine_free) {                 // the place's lane: its places are lane, lane + 32, ...
                    f[best & 511u] = end << 9 | (best & 511u);
                    mine_free = 0xffffffffu;
                    for (int i = lane; i < places; i += 32) mine_free = min(mine_free, f[i]);
                }
            }
        }
        if (lane == 0) s_span[w] = span;
    }
    if (!queue && threadIdx.x == 32) s_span[1] = (uint32_t)s_longest;
    __syncthreads();
    if (threadIdx.x == 0) ctrl->use_grid = cl_us * (float)s_span[0] > other_cost((float)s_span[1]);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static std::mutex g_cl_mutex;
static int g_cl_clusters[64];          // per device: 0 not asked yet, -1 none, else clusters of 16 that are resident at a time

template <int ACT, int NL>
static const void* cl_fn_act(int ns) {
    switch (ns) {
        case 1: return (const void*)cl_kernel<1, ACT, NL>;
        case 2: return (const void*)cl_kernel<2, ACT, NL>;
        case 4: return (const void*)cl_kernel<4, ACT, NL>;
        default: return (const void*)cl_kernel<8, ACT, NL>;
    }
}
static const void* cl_fn(int ns, int act, int layers) {
    if (layers == 2) return act == WIND_ACT_RELU ? cl_fn_act<WIND_ACT_RELU, 2>(ns) : cl_fn_act<WIND_ACT_TANH, 2>(ns);
    return act == WIND_ACT_RELU ? cl_fn_act<WIND_ACT_RELU, 1>(ns) : cl_fn_act<WIND_ACT_TANH, 1>(ns);
}
static uint32_t cl_smem_bytes(int P, int H, int NV, int slots, int wp, int layers) {
    uint32_t bytes = cl_smem_layout(P, H, NV, slots, wp, layers).total;
    if (layers == 2) {                                   // the CTAs of cl_recurrent: what its MMAs and its last ldmatrix may read
        const uint32_t states = (uint32_t)((CL_DECODERS + 1) & ~1) * (uint32_t)P * 16u + 1024u;
        if (bytes < states) bytes = states;
    }
    return bytes + 1024u;
}
// The most that a launch asks for: what every kernel is granted.  (The window's keys grow with its padding and the states with the
// slots: with one layer one slot pair of 32 rows takes most, 219264 bytes against 212736 with eight slots of 8; with two 226944 against 224256.)
static uint32_t cl_smem_most() {
    uint32_t most = 0;
    for (int layers = 1; layers <= 2; ++layers)
        for (int wp = 8; wp <= 32; wp *= 2)
            for (int slots = 1; slots <= 8 * CL_GROUPS / wp; ++slots) {
                const uint32_t bytes = cl_smem_bytes(CL_MAX_DIM, CL_MAX_DIM, 16 * CL_MAX_LABELS, slots, wp, layers);
                if (bytes > most) most = bytes;
            }
    return most;
}
static int cl_padded_window(int W) { return W <= 8 ? 8 : (W <= 16 ? 16 : 32); }
void cl_debug_smem(const wind_model_t& m, int W, int slots, uint32_t* bytes, uint32_t* granted) {
    *bytes = cl_smem_bytes(m.P, m.H, m.V + 1, slots, cl_padded_window(W), m.L);
    *granted = cl_smem_most();
}

// clusters of 16 CTAs the current device holds at a time (one CTA per SM); 0: none
static int cl_clusters() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lock(g_cl_mutex);
    if (g_cl_clusters[dev] == 0) {
        g_cl_clusters[dev] = -1;
        int optin = 0;
        if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return 0;
        const int want = (int)cl_smem_most();
        if (want > optin - 1024) return 0;
        for (int k = 0; k < 16; ++k) {
            const void* fn = cl_fn(1 << (k & 3), k >> 2 & 1, 1 + (k >> 3));
            if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
                cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, want) != cudaSuccess) {
                cudaGetLastError();
                return 0;
            }
        }
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(CL_SIZE);
        cfg.blockDim = dim3(CL_THREADS);
        cfg.dynamicSmemBytes = (size_t)want;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = CL_SIZE; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, cl_fn(8, WIND_ACT_RELU, 2), &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
        if (n > 0) g_cl_clusters[dev] = n;
    }
    return g_cl_clusters[dev] > 0 ? g_cl_clusters[dev] : 0;
}

// What a lock step costs, in us: of a cluster with all its slots, and of the other kernel with all its rows.  Clusters: fitted to 104
// steps of one layer (13 models: P and H 128 to 640, 500 and 1024 labels, ReLU and tanh; W = 1 to 32, every slot in use) and 68 of two
// (9 models): 5.5 and 2.1 % rms for windows of up to 8 rows, 5.1 and 5.2 beyond, at most 19 off (tanh at W = 32 with few joint units).
// One layer's figures stand 2 to 7 % above its steps of today.  Chosen by these, a decode takes 1.1 % longer than by the better kernel of each
// pair on the average where weights lie on the chip (961 pairs of one layer: 18 to 300 utterances of equal and of ragged lengths; 560 of
// two: 0.8 %), 1.5 % against streamed weights (235 pairs); with 5 % less for one layer 0.6 and 1.7 %, but batches of the choice's tests
// would change sides.  With the figures of earlier kernels, 15 to 20 % above, two layers took 2.7 % longer (P = 640, H = 256, W = 1, 41
// utterances of 150 frames: 3.68 ms against 2.05).  What is lost most is 46 %: sizes where the joint of the other kernel fits well.
static float cl_step_us(const wind_model_t& m, int W, int wp) {
    const float P = (float)m.P, H = (float)m.H, NV = (float)(m.V + 1) / 1024.f, l = log2f((float)W), z = m.act == WIND_ACT_RELU ? 0.f : H;
    if (m.L == 2) return wp == 8 ? 5.45f + 0.0023f * P + (0.0001f + 0.00124f * l + 0.00074f * NV) * H + 0.00013f * (float)W * z
                                 : 5.65f + 0.0015f * P + (0.0028f + 0.0003f * NV) * H + 0.0014f * z;
    return wp == 8 ? 3.3f + 0.0014f * P + (0.0017f + 0.00045f * l) * H + 0.23f * l + 0.00017f * (float)W * z
                   : 3.77f + 0.0009f * P + 0.003f * H + 0.0015f * z;
}
// Other kernels: 430 pairs of one layer (8 % rms), 112 of two (8 %).
static float other_step_us(const wind_model_t& m, const LoopPlan& pl, int B, int W) {
    const float P = (float)m.P, H = (float)m.H, rows = (float)B * (float)W;
    if (!pl.resident) return -2.5f + 3.8f * (float)pl.mt_count + 0.0053f * rows + 0.0177f * P + 0.0145f * H;
    const int waves = (pl.rg_count + pl.rg_stride - 1) / pl.rg_stride;
    if (m.L == 2) return 12.3f + 0.0009f * H + 0.0043f * P + 0.0045f * rows + 0.018f * (float)B;
    return 10.1f + 0.005f * H + 0.002f * rows + (pl.dataflow ? 6.5f : 3.f) * (float)(waves - 1);
}

// The shapes whose decoder fits one cluster (with two layers: one, and two clusters that all share): one or two LSTM layers, P and H
// multiples of 128 (a CTA's share is then whole 16-byte pieces, and the K halves are equal) up to 640, at most 72 vocabulary entries per
// CTA, windows up to 32 rows.  Everything else, and the FULL features (logits store, window-based decoding, timeline, forced loop
// modes), stays with loop_kernel.
bool cl_fits(const wind_model_t& m, int W) {
    const int nv = m.V + 1;
    if (m.L > 2 || m.P % 128 || m.H % 128 || m.P > CL_MAX_DIM || m.H > CL_MAX_DIM || W > 32) return false;
    return cl_label_base(nv) + (cl_label_extra(nv) > 0 ? 8 : 0) <= CL_MAX_LABELS;
}
static bool cl_supported(const Call& c) {
    if (!cl_fits(c.m, c.W)) return false;
    if (c.mode != WIND_MODE_FIRST_NONBLANK || c.joint_iters > 0) return false;
    const LoopOptions o = loop_get_options();
    if (!o.resident || o.dataflow >= 0 || o.joint_placement >= 0) return false;
    return cl_clusters() > 0;
}

// Two layers: what the clusters hand one another lies in the workspace from the plain-ALU path's state (behind the utterances' order)
// to the gate table: regions of other kernels, and where they are too small (few batch rows, H far below P) the other kernel decodes.
struct ClExchange { size_t hx, rx, end; };
static ClExchange cl_exchange(const Call& c, int n, int clusters, int slots) {
    ClExchange x{};
    x.hx = c.lay.h + align_up(sizeof(int32_t) * (size_t)n);
    x.rx = align_up(x.hx + sizeof(__nv_bfloat16) * (size_t)clusters * 4 * 8 * c.m.P);
    x.end = x.rx + sizeof(unsigned long long) * (size_t)clusters * 2 * slots * 4 * c.m.P;
    return x;
}

// How a decode runs in clusters; false: it does not.  `other` is the plan by which another kernel could take it.
// Where that has the weights on the chip its transcripts are the same bit for bit, and where any lengths could favour it (the
// clusters may need as many rounds as its rows make of their slots) both are launched and the lengths decide on the device.
// Streamed weights go with other roundings; which of the two decodes must not depend on the lengths of a batch, so the shapes
// alone decide, for lengths whose mean is 0.6 of the longest, or rows that are refilled throughout.
bool cl_plan(const Call& c, const LoopPlan& other, ClPlan* out) {
    if (!cl_supported(c)) return false;
    const int n = c.N > 0 ? c.N : c.B, avail = c.m.L == 2 ? (cl_clusters() - 2 < CL_DECODERS ? cl_clusters() - 2 : CL_DECODERS) : cl_clusters();
    if (avail < 1) return false;
    ClPlan q{};
    q.wp = cl_padded_window(c.W);
    // one slot per cluster as long as there are clusters, then more slots (a lock step of eight slots costs less than two of one)
    const int most = 8 * CL_GROUPS / q.wp;
    q.clusters = n < avail ? n : avail;
    q.slots = (n + q.clusters - 1) / q.clusters < most ? (n + q.clusters - 1) / q.clusters : most;
    const int slots = q.slots * q.clusters;
    // two layers: only where the other kernel has its weights on the chip (the same roundings); the clusters exchange states and
    // recurrent terms in the regions of the other kernels' states
    if (c.m.L == 2 && !other.resident) return false;
    if (c.m.L == 2 && cl_exchange(c, n, q.clusters, q.slots).end > c.lay.g0) return false;
    q.rows = c.B < n ? c.B : n;
    q.cl_us = cl_step_us(c.m, c.W, q.wp);
    q.other_us = other_step_us(c.m, other, c.B, c.W);
    q.order = n > slots && n <= CL_ORDER_MAX && sizeof(int32_t) * (size_t)n <= sizeof(float) * 2 * (size_t)c.B * c.m.P;
    const float rounds = (float)((q.rows + slots - 1) / slots), cost = q.other_us * (1.f + 2.5f / sqrtf((float)c.T));
    if (rounds > 1.f) {
        if (!other.resident && (n > q.rows ? (float)q.rows / (float)slots : 0.6f * rounds) * q.cl_us > cost) return false;
        q.choose = other.resident && rounds * q.cl_us > cost;
    }
    *out = q;
    return true;
}

cudaError_t cl_loop(const Call& c, const ClPlan& q) {
    const wind_model_t& m = c.m;
    const int n = c.N > 0 ? c.N : c.B;
    ClParams p{};
    p.ctrl = c.ctrl();
    p.T = c.T; p.W = c.W; p.S = c.S; p.max_out = c.max_out; p.H = m.H; p.P = m.P; p.NV = m.V + 1; p.blank = m.blank_id;
    p.n_utt = n;
    p.wp = q.wp;
    p.slots = q.slots;
    p.choose = q.choose;
    {
        // units of the joint's operand: 448 threads (320 without warps 10-13) in eights; the fewer groups of rows, the fewer rows a unit
        const int kb_h = m.H / 64, units = m.L == 2 || m.P / CL_SIZE > 32 ? 56 : 40, groups = p.slots * p.wp / 8, rows = p.wp == 8 ? p.W : 8;
        p.z_parts = groups > 4 ? 1 : 2;
        while ((1 << p.z_parts) > rows) --p.z_parts;
        p.z_rows = (rows + (1 << p.z_parts) - 1) >> p.z_parts;
        p.z_step = units / kb_h << 8 | units % kb_h;
    }
    p.smem = cl_smem_layout(m.P, m.H, p.NV, p.slots, p.wp, m.L);
    const int ns = p.slots <= 1 ? 1 : (p.slots <= 2 ? 2 : (p.slots <= 4 ? 4 : 8));
    p.queue_base = n < c.B ? n : c.B;
    long long cap = (long long)c.T * (c.S + 1) + 2;
    cap = (cap + 1) * n;                      // at worst one utterance after the other in one slot
    p.step_cap = cap > 0x7fffffff ? 0x7fffffff : (int)cap;
    p.extra_arrivals = loop_extra_arrivals();
    p.enc_len = c.enc_len;
    p.g0 = c.g0();
    p.w_gate = (const __nv_bfloat16*)(m.L == 2 ? c.w_ih[1] : c.w_hh[0]); p.w_pred = (const __nv_bfloat16*)m.w_pred; p.w_out = (const __nv_bfloat16*)m.w_out;
    p.b_pred = m.b_pred; p.b_out = m.b_out;
    p.out_tokens = c.out_tokens; p.out_frames = c.out_frames; p.out_len = c.out_len;
    if (q.order) {
        int32_t* order = reinterpret_cast<int32_t*>(c.h(0));     // the plain-ALU path's state: not used by a bf16 tensor decode
        cl_order_kernel<<<(n + 1023) / 1024, 1024, 0, c.stream>>>(c.enc_len, n, order);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        p.order = order;
    }
    if (q.choose) {
        cl_choose_kernel<<<1, 256, 0, c.stream>>>(c.ctrl(), c.enc_len, p.order, n, c.T, q.slots * q.clusters, q.rows, q.cl_us, q.other_us);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    CUtensorMap enc_map, hx_map;
    cudaError_t e = loop_map3(&enc_map, c.enc_proj(), (uint64_t)n * c.T, m.H, 8);
    if (e != cudaSuccess) return e;
    hx_map = enc_map;
    if (m.L == 2) {
        const ClExchange x = cl_exchange(c, n, q.clusters, q.slots);
        for (int l = 0; l < 2; ++l) p.w_rec[l] = (const __nv_bfloat16*)c.w_hh[l];
        p.b_gate[0] = c.b_ih[1]; p.b_gate[1] = c.b_hh[1];
        p.req = c.flags(); p.done = p.req + 2 * CL_DECODERS; p.beat = p.done + CL_DECODERS;   // (23 counters at the least)
        p.hx = reinterpret_cast<__nv_bfloat16*>(c.ws + x.hx);
        p.rx = reinterpret_cast<unsigned long long*>(c.ws + x.rx);
        if ((e = loop_map3(&hx_map, p.hx, (uint64_t)q.clusters * 32, m.P, 8)) != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((q.clusters + (m.L == 2 ? 2 : 0)) * CL_SIZE));
    cfg.blockDim = dim3(CL_THREADS);
    cfg.dynamicSmemBytes = cl_smem_bytes(m.P, m.H, p.NV, p.slots, p.wp, m.L);
    cfg.stream = c.stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CL_SIZE; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeCooperative;           // two layers: clusters wait for one another, so all have to be resident
    at[1].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = m.L == 2 ? 2 : 1;
    void* args[3] = {(void*)&enc_map, (void*)&hx_map, (void*)&p};
    return cudaLaunchKernelExC(&cfg, cl_fn(ns, m.act, m.L), args);
}

}  // namespace wind
