// Parameter block and small device helpers of the cluster kernel (wind_loop_cl.cu).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "wind_internal.cuh"
#include "wind_loop.cuh"
#include "wind_ptx.cuh"

namespace wind {

constexpr int CL_SIZE = 16;            // CTAs of a cluster
constexpr int CL_SLOTS = 8;            // most utterances a cluster decodes at a time
constexpr int CL_GROUPS = 8;           // most groups of eight window rows (64 rows: the MMA's M)
constexpr int CL_MAX_DIM = 640;        // most P and H
constexpr int CL_MAX_LABELS = 72;      // most vocabulary entries of a CTA
constexpr int CL_THREADS = 512;
// two LSTM layers: one cluster per layer keeps that layer's W_hh for all the others (they hold the rest of the model)
constexpr int CL_DECODERS = 5;         // most decoding clusters beside them

// Shared-memory regions of a CTA (bytes from a 1024-byte boundary).  z comes first and is followed by the W_out tile: the
// joint's MMA always reads eight groups of rows, those beyond the ones in use are rows nobody looks at.
struct ClSmem {
    uint32_t z, w_out, h0, h, pred, kbuf, dec, b_out, b_pred, hst, gr, part, pst, b_gate, cell, rec, total;
};

struct ClParams {
    Ctrl* ctrl;
    int T, W, S, max_out, H, P, NV, blank;
    int n_utt;                         // utterances
    int slots;                         // utterances a cluster decodes at a time (NU)
    int wp;                            // window rows of a slot, padded: 8, 16 or 32
    int queue_base;                    // value of ctrl->next_utt before the first utterance is taken from the queue
    int step_cap, extra_arrivals, choose;
    ClSmem smem;
    int z_parts, z_rows, z_step;       // the joint's operand: log2 of the parts of a group of eight rows, rows of a part, (group, part) << 8 | K block from unit to unit
    const int32_t* order;              // [n_utt] order in which utterances are taken; null: 0, 1, ...
    const int32_t* enc_len;
    const float* g0;                   // [NV][4P]
    const __nv_bfloat16* w_gate;       // [4P][P] the matrix of the cluster's own gate product: W_hh; with two layers the second one's W_ih
    const __nv_bfloat16* w_pred;       // [H][P]
    const __nv_bfloat16* w_out;        // [NV][H]
    const float* b_pred;
    const float* b_out;
    int32_t* out_tokens;
    int32_t* out_frames;
    int32_t* out_len;
    // two layers (wind_loop_cl.cu, "recurrent terms"); counters in the workspace, zero at the start of the call
    const __nv_bfloat16* w_rec[2];     // W_hh of either layer
    const float* b_gate[2];            // b_ih and b_hh of the second layer
    uint32_t* req;                     // [2][CL_DECODERS] CTAs that have written their part of a layer's new state
    uint32_t* done;                    // [CL_DECODERS] CTAs of a decoding cluster that have left
    uint32_t* beat;                    // [CL_DECODERS] lock steps of a decoding cluster / 1024
    __nv_bfloat16* hx;                 // [clusters][2 layers][2 parities][8 slots][P] the states
    unsigned long long* rx;            // [clusters][2 layers][CL_SIZE][slots][4P / CL_SIZE] the recurrent terms, by CTA: number of the update << 32 | fp32
};

constexpr int CL_KEY_PITCH = 34;       // keys of a window row: two per CTA, and padding against bank conflicts
constexpr int CL_GR_PITCH = 36;        // floats: gate rows of the remainder units (at most 32) and padding

__host__ __device__ inline int cl_label_base(int NV) { return NV / 128 * 8; }              // vocabulary entries of every CTA
__host__ __device__ inline int cl_label_extra(int NV) { return (NV - 16 * cl_label_base(NV) + 7) / 8; }   // CTAs with eight more

// Bytes of a K block of the state.  The gates' MMA reads 16 rows.  One layer: rows 8 to 15 are zeros.  Two layers have two states
// and no room for that: the second group of eight rows is the next K block (its products go nowhere).
__host__ __device__ inline uint32_t cl_h_block(int layers) { return layers == 2 ? 1024u : 2048u; }

// whether the gates' product with the state follows the joint's, for which there are two copies of the state
__host__ __device__ inline bool cl_gates_late(int slots, int layers) { return layers == 1 && slots == 1; }

__host__ __device__ inline ClSmem cl_smem_layout(int P, int H, int NV, int slots, int wp, int layers) {
    ClSmem s{};
    uint32_t off = 0;
    auto take = [&](uint32_t bytes, uint32_t align) { off = (off + align - 1) / align * align; const uint32_t o = off; off += bytes; return o; };
    const uint32_t labels = (uint32_t)cl_label_base(NV) + (cl_label_extra(NV) > 0 ? 8u : 0u);
    s.z = take((uint32_t)(slots * wp) * (uint32_t)H * 2u, 1024);
    s.w_out = take(labels * (uint32_t)H * 2u, 1024);
    // eight groups of rows from the last K block of the first group on have to stay inside
    const uint32_t reach = (uint32_t)CL_GROUPS * 8u * (uint32_t)H * 2u;
    if (off < reach) off = reach;
    const uint32_t state = (uint32_t)(P / 64) * cl_h_block(layers) + (layers == 2 ? 1024u : 0u);
    s.h0 = take(layers == 2 ? state : 0u, 1024);
    s.h = take(cl_gates_late(slots, layers) ? 2u * state : state, 1024);
    s.pred = take(CL_SLOTS * (uint32_t)H * 2u, 1024);
    s.kbuf = take(CL_KEY_PITCH * (uint32_t)wp * 8u, 16);
    s.dec = take(CL_SLOTS * 16u, 16);
    s.b_out = take((CL_MAX_LABELS + 8u) * 4u, 16);
    s.b_pred = take(48u * 4u, 16);
    s.hst = take((uint32_t)layers * CL_SLOTS * (uint32_t)(P / 16) * 2u, 16);
    s.gr = take(CL_SLOTS * CL_GR_PITCH * 4u, 16);
    s.part = take(3u * 32u * 16u, 16);          // second K half of pred_proj: one accumulator fragment per lane of three warps
    s.pst = take(CL_SLOTS * 48u * 2u, 16);      // pred_proj of the CTA's joint units, bf16 [slot][48]
    s.b_gate = take(layers == 2 ? (uint32_t)(P / 4) * 4u : 0u, 16);   // biases of the second layer's gates, [4 unit + gate]
    s.cell = take(layers == 2 ? 2u * 3u * 128u * 4u : 0u, 16);
    s.rec = take(layers == 2 ? (uint32_t)slots * (uint32_t)(P / 4) * 4u : 0u, 16);   // the first layer's recurrent term, [slot][4 unit + gate]
    s.total = off;
    return s;
}

__device__ __forceinline__ uint32_t cl_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// the address in CTA `rank` of the cluster that corresponds to this CTA's shared-memory address
__device__ __forceinline__ uint32_t cl_map(uint32_t addr, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}
// asynchronous stores into another CTA's shared memory; the bytes are counted on that CTA's mbarrier
__device__ __forceinline__ void st_async_16(uint32_t addr, uint4 v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "r"(v.x),
                 "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void st_async_8(uint32_t addr, unsigned long long v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr), "l"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void cl_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// block barrier of `threads` threads that also tells each of them whether any has given up
template <int threads>
__device__ __forceinline__ bool group_barrier_or(int id, bool mine) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %2, 0;\n\t"
        "bar.red.or.pred q, %1, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(id), "r"((int)mine), "n"(threads)
        : "memory");
    return r != 0;
}
// Bounded wait for an mbarrier phase, short in code (the loop has many and its instructions have to stay in the instruction
// cache): the hardware parks the thread for up to 20 us a try, and after 2^17 tries (seconds) the wait gives up.
__device__ __forceinline__ bool cl_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .u32 n;\n\t"
        "mov.u32 n, 0;\n"
        "CL_WAIT_TRY:\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 20000;\n\t"
        "@p bra CL_WAIT_DONE;\n\t"
        "add.u32 n, n, 1;\n\t"
        "setp.lt.u32 q, n, 131072;\n\t"
        "@q bra CL_WAIT_TRY;\n"
        "CL_WAIT_DONE:\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// whether the phase is there, without waiting for it
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void st_relaxed_u32(uint32_t* p, uint32_t v) { asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory"); }
__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) { asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory"); }
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
// Bounded wait of a warp for values that carry `stamp` in their upper words: of every lane the slots of `want` (NS at most, `pitch`
// apart; out is 0 for the others), and where want_r four more.
template <int NS>
__device__ __forceinline__ bool cl_read_stamped(const unsigned long long* src, uint32_t pitch, uint32_t want, uint32_t stamp, float* out, const int32_t* abort,
                                                const unsigned long long* src_r = nullptr, bool want_r = false, float* out_r = nullptr) {
    unsigned long long t0 = 0;
    for (uint32_t it = 1u;; ++it) {
        bool there = true;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const unsigned long long v = (want >> s) & 1u ? ld_relaxed_u64(src + s * pitch) : (unsigned long long)stamp << 32;
            there = there && (uint32_t)(v >> 32) == stamp;
            out[s] = __uint_as_float((uint32_t)v);
        }
        if (want_r)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const unsigned long long v = ld_relaxed_u64(src_r + k);
                there = there && (uint32_t)(v >> 32) == stamp;
                out_r[k] = __uint_as_float((uint32_t)v);
            }
        if (__all_sync(0xffffffffu, there)) return true;
        if ((it & 255u) == 0u) {
            int gone;
            asm volatile("ld.volatile.global.u32 %0, [%1];" : "=r"(gone) : "l"(abort) : "memory");
            const unsigned long long now = globaltimer_ns();
            if (t0 == 0) t0 = now;
            if (__any_sync(0xffffffffu, gone != 0 || now - t0 > kWaitLimitNs)) return false;
        }
    }
}
// the same for a whole warp, with one answer for all its lanes
__device__ __forceinline__ bool cl_wait_warp(uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, cl_wait(bar, parity)); }

// Two accumulators of 16 rows (lanes) added, X times eight columns, rows spread over the warp as mma.sync spreads them: of columns
// 8 x ..  v[4 x], v[4 x + 1]: row lane / 4, columns 2 (lane % 4), + 1;  v[4 x + 2], v[4 x + 3]: row lane / 4 + 8.
template <int X>
__device__ __forceinline__ void tmem_ld_quarter(uint32_t ta, uint32_t tb, float* v) {
    uint32_t a[4 * X], b[4 * X];
    if constexpr (X == 1) {
        asm volatile(
            "tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%8];\n\t"
            "tcgen05.ld.sync.aligned.16x256b.x1.b32 {%4,%5,%6,%7}, [%9];\n\t"
            "tcgen05.wait::ld.sync.aligned;"
            : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3])
            : "r"(ta), "r"(tb)
            : "memory");
    } else {
        asm volatile(
            "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%16];\n\t"
            "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%17];\n\t"
            "tcgen05.wait::ld.sync.aligned;"
            : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(b[0]), "=r"(b[1]),
              "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7])
            : "r"(ta), "r"(tb)
            : "memory");
    }
#pragma unroll
    for (int i = 0; i < 4 * X; ++i) v[i] = __uint_as_float(a[i]) + __uint_as_float(b[i]);
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t* r, uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void mma_16816(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// host side (wind_loop_cl.cu)
struct ClPlan {
    int clusters, slots, wp;           // as in ClParams; the clusters that decode
    int rows;                          // utterances the other kernel decodes at a time
    bool order;                        // the utterances are taken longest first
    bool choose;                       // the other kernel has to be launched behind this one, and ctrl->use_grid tells either whether it is to run
    float cl_us, other_us;             // what a lock step of either costs
};
bool cl_plan(const Call& c, const LoopPlan& other, ClPlan* out);
cudaError_t cl_loop(const Call& c, const ClPlan& q);

}  // namespace wind
