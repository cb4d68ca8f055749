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

struct ClParams {
    Ctrl* ctrl;
    int T, W, S, max_out, H, P, NV, blank;
    int n_utt;                         // utterances
    int slots;                         // utterances a cluster decodes at a time (NU)
    int wp;                            // window rows of a slot, padded: 8, 16 or 32
    int queue_base;                    // value of ctrl->next_utt before the first utterance is taken from the queue
    int step_cap, extra_arrivals, choose;
    const int32_t* order;              // [n_utt] order in which utterances are taken; null: 0, 1, ...
    const int32_t* enc_len;
    const float* g0;                   // [NV][4P]
    const __nv_bfloat16* w_hh;         // [4P][P]
    const __nv_bfloat16* w_pred;       // [H][P]
    const __nv_bfloat16* w_out;        // [NV][H]
    const float* b_pred;
    const float* b_out;
    int32_t* out_tokens;
    int32_t* out_frames;
    int32_t* out_len;
};

// Shared-memory regions of a CTA (bytes from a 1024-byte boundary).  z comes first and is followed by the W_out tile: the
// joint's MMA always reads eight groups of rows, those beyond the ones in use are rows nobody looks at.
struct ClSmem {
    uint32_t z, w_out, h, pred, kbuf, dec, b_out, b_pred, hst, gr, part, pst, total;
};
constexpr int CL_KEY_PITCH = 34;       // keys of a window row: two per CTA, and padding against bank conflicts
constexpr int CL_GR_PITCH = 36;        // floats: gate rows of the remainder units (at most 32) and padding

__host__ __device__ inline int cl_label_base(int NV) { return NV / 128 * 8; }              // vocabulary entries of every CTA
__host__ __device__ inline int cl_label_extra(int NV) { return (NV - 16 * cl_label_base(NV) + 7) / 8; }   // CTAs with eight more

__host__ __device__ inline ClSmem cl_smem_layout(int P, int H, int NV, int slots, int wp) {
    ClSmem s{};
    uint32_t off = 0;
    auto take = [&](uint32_t bytes, uint32_t align) { off = (off + align - 1) / align * align; const uint32_t o = off; off += bytes; return o; };
    const uint32_t labels = (uint32_t)cl_label_base(NV) + (cl_label_extra(NV) > 0 ? 8u : 0u);
    s.z = take((uint32_t)(slots * wp) * (uint32_t)H * 2u, 1024);
    s.w_out = take(labels * (uint32_t)H * 2u, 1024);
    // eight groups of rows from the last K block of the first group on have to stay inside
    const uint32_t reach = (uint32_t)CL_GROUPS * 8u * (uint32_t)H * 2u;
    if (off < reach) off = reach;
    s.h = take(16u * (uint32_t)P * 2u, 1024);
    s.pred = take(CL_SLOTS * (uint32_t)H * 2u, 1024);
    s.kbuf = take(CL_KEY_PITCH * (uint32_t)wp * 8u, 16);
    s.dec = take(CL_SLOTS * 16u, 16);
    s.b_out = take((CL_MAX_LABELS + 8u) * 4u, 16);
    s.b_pred = take(48u * 4u, 16);
    s.hst = take(CL_SLOTS * (uint32_t)(P / 16) * 2u, 16);
    s.gr = take(CL_SLOTS * CL_GR_PITCH * 4u, 16);
    s.part = take(3u * 32u * 16u, 16);          // second K half of pred_proj: one accumulator fragment per lane of three warps
    s.pst = take(CL_SLOTS * 48u * 2u, 16);      // pred_proj of the CTA's joint units, bf16 [slot][48]
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
// the same for a whole warp, with one answer for all its lanes
__device__ __forceinline__ bool cl_wait_warp(uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, cl_wait(bar, parity)); }

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
    int clusters, slots, wp;           // as in ClParams
    int rows;                          // utterances the other kernel decodes at a time
    bool order;                        // the utterances are taken longest first
    bool choose;                       // the other kernel has to be launched behind this one, and ctrl->use_grid tells either whether it is to run
    float cl_us, other_us;             // what a lock step of either costs
};
bool cl_plan(const Call& c, const LoopPlan& other, ClPlan* out);
cudaError_t cl_loop(const Call& c, const ClPlan& q);

}  // namespace wind
