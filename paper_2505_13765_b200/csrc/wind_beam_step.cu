// The beam search's iterations (Algorithm 3) on the device: decoder update of the hypotheses that have no state yet, their
// projection, the window's logits under every hypothesis, Eq. (1) and the K best entries of each.
//
// As separate kernels an iteration of the 640-unit model with beam 4 took 85 us, of which 51 us were eleven kernels and copies
// (a block per hidden unit or per sixteen labels loads its weights, waits for them, and uses them once) and the rest gaps and
// the synchronisation.  Here hidden units, joint units and labels are dealt out over all SMs with their weights (67 KB each) in
// shared memory, the phases follow one another behind grid barriers, and the kernel stays for the whole search: the
// host writes each command to page-locked memory and reads the result there.  One launch per iteration
// took 42 us: 6 us of launch, the weights again, and every instruction fetched from L2 because it runs once.
// A command of 4 hypotheses at W = 8 takes 22 us, one of 12 (hypotheses of later iterations, wind_beam.cu) 30 us, before 36 us: operands
// of four elements and four rows at a time (element by element the joint's took 9 us), all updates in one pass, dot products in pairs
// and eight rows at a time.  What is left: 7 us from result to command over the host, three grid barriers (1.5 us each with
// their skew), dot products 6 us, the K best entries 6 us, and chains of a few L2 and shared-memory latencies.
//
// The kernel never depends on the host's pace: without a command for 200 us it ends, and the host launches it again with the
// next one (all state is in global memory).  So a debugger or a descheduled host thread cost the search time only.  On every SM
// it leaves 8 of 64 thousand registers, so most kernels of other streams wait for its end: the host has it end every 10 ms.
//
// A command or result word carries its 32 bits and the command's number in one 8-byte store, so no fence or flag is needed on
// either side of the bus.
//
// A dot product is summed as the per-phase kernels sum it, so that both give the same bits: 32 chains, chain r over
// k = r, r + 32, ..., then a butterfly.  A lane carries one chain of four weight rows times four operand rows.  Rows are kept
// interleaved by four ([k][4]), so that a step is two loads for sixteen products: with rows kept apart the eight loads of a step
// took 135 cycles.
#include "wind_internal.cuh"
#include "wind_loop.cuh"
#include "wind_ptx.cuh"

#include <mutex>
#include <type_traits>

namespace wind {

constexpr int BS_THREADS = 512;
constexpr int BS_WARPS = BS_THREADS / 32;
constexpr int BS_UTTS = 4;            // updates of an item
constexpr int BS_ROWS = 4;            // window rows of a joint item

constexpr unsigned long long BS_IDLE_NS = 200000ull;

// dimensions shared by the host's plan and the kernel; all sizes in elements, offsets in bytes
struct BsPlan {
    int units, prows, labels;         // the most a CTA owns of each
    int k_l, k_p;                     // row lengths, rounded up to 32: of the gates (any layer), of W_pred
    int rows, look;                   // as in BeamShape
    int quads;                        // fours of updates of a pass
    int zrows, k_z;                   // window rows of a joint pass; row length of the joint, rounded up to 32
    int resident;                     // the gates' weights of all layers stay; else a layer's are loaded in front of its use
    uint32_t layer, w_l, w_pred, w_out, bias, enc, x, z, total;   // layer: bytes of one layer's weights; z: later the window's logits
};
template <typename TW> static BsPlan bs_plan_with(int G, int W, int rows, int look, int resident, int quads, int E, int P, int L, int H, int NV, uint32_t budget) {
    BsPlan s{};
    s.units = (P + G - 1) / G; s.prows = (H + G - 1) / G; s.labels = (NV + G - 1) / G;
    const int k0 = E + P, k1 = L > 1 ? 2 * P : 0, kmax = k0 > k1 ? k0 : k1;
    s.k_l = (kmax + 31) / 32 * 32; s.k_p = (P + 31) / 32 * 32;
    s.k_z = (H + 31) / 32 * 32;
    s.rows = rows; s.look = look; s.resident = resident; s.quads = quads;
    const int all = (rows * W + BS_ROWS - 1) / BS_ROWS * BS_ROWS;
    unsigned long long off = 0;
    auto take = [&](unsigned long long bytes) { const unsigned long long o = off; off += (bytes + 15) / 16 * 16; return (uint32_t)o; };
    const unsigned long long layer = (unsigned long long)sizeof(TW) * s.units * 4 * s.k_l;
    s.layer = (uint32_t)layer;
    s.w_l = take(layer * (resident ? L : 1));
    s.w_pred = take((unsigned long long)sizeof(TW) * ((s.prows + 3) / 4 * 4) * s.k_p);
    s.w_out = take((unsigned long long)sizeof(TW) * ((s.labels + 3) / 4 * 4) * s.k_z);
    s.bias = take(4ull * (4 * L * s.units + s.prows + s.labels));
    s.enc = take((unsigned long long)sizeof(TW) * (W + look) * H);
    const unsigned long long xa = (unsigned long long)sizeof(TW) * BS_UTTS * quads * s.k_l, xb = 4ull * rows * H;
    s.x = take(xa > xb ? xa : xb);
    s.z = (uint32_t)off;
    const unsigned long long row = (unsigned long long)sizeof(TW) * s.k_z, window = 4ull * W * NV;
    const unsigned long long fit = off < budget ? (budget - off) / row / BS_ROWS * BS_ROWS : 0;
    s.zrows = fit < (unsigned long long)all ? (int)fit : all;
    off += row * s.zrows > window ? row * s.zrows : window;
    s.total = s.zrows == 0 || off > budget ? 0xffffffffu : (uint32_t)off;
    return s;
}
// The weights stay if at least four row groups fit beside them, with all updates of a command in one pass or else in several; then as
// many rows and frames ahead as fit likewise (those in one pass of updates).
template <typename TW> static BsPlan bs_plan(int G, int W, int K, bool ahead, int E, int P, int L, int H, int NV, uint32_t budget) {
    auto good = [&](const BsPlan& s) {
        const int all = (s.rows * W + BS_ROWS - 1) / BS_ROWS * BS_ROWS;
        return s.total <= budget && s.zrows >= (s.resident && all > 16 ? 16 : BS_ROWS);
    };
    auto in_one = [](int rows) { return (rows + BS_UTTS - 1) / BS_UTTS; };
    BsPlan s{};
    s.total = 0xffffffffu;
    for (int resident = 1; resident >= 0 && !good(s); --resident)
        for (int quads = in_one(K); quads >= 1; --quads)
            if (good(s = bs_plan_with<TW>(G, W, K, 0, resident, quads, E, P, L, H, NV, budget))) break;
    if (!good(s) || !ahead || K < 2) return s;
    // Where weights stay only at the price of several passes, commands twice as long as the beam are worth more than that: two layers of
    // 512 units in fp32, W = 8, K = 8: 46.2 us an iteration against 50.1 (K = 12, W = 4, where 16 rows are not twice the beam: 86 against 80).
    if (s.resident && s.quads < in_one(K))
        for (int look = kBeamLook; look >= 4 && kBeamRows >= 2 * K; look /= 2) {
            const BsPlan a = bs_plan_with<TW>(G, W, kBeamRows, look, 0, in_one(kBeamRows), E, P, L, H, NV, budget);
            if (good(a) && a.zrows >= 16) return a;
        }
    // 12 rows and 12 frames, 16 and 12, 16 and 16: 250 frames at W = 8, beam 4: 28.8, 28.1, 27.2 ms; 200 at W = 16, beam 2: 18.8, 19.0, 18.7;
    // 300 at W = 4, beam 3: 19.9, 18.9, 18.4; 100 at W = 1, beam 4: 9.4, 8.4, 9.0
    for (int rows = kBeamRows; rows >= 8 && rows >= K; rows -= 4)
        for (int look = kBeamLook; look >= 4; look /= 2) {
            const BsPlan a = bs_plan_with<TW>(G, W, rows, look, s.resident, in_one(rows), E, P, L, H, NV, budget);
            if (good(a)) return a;
        }
    return s;
}

struct BsParams {
    Ctrl* ctrl;
    BeamMail* mail;                    // page-locked host memory
    unsigned long long* relay;         // the command in device memory, read by every CTA
    uint32_t first_seq;                // number of the first command
    uint32_t bar_base;                 // arrivals at the grid barrier before this launch
    uint32_t extra_arrivals;
    BsPlan plan;
    int K;
    int E, P, L, H, NV, blank, act, W, T;
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
    float *h_pool, *c_pool, *g_pool, *logits;
};

// Two fp32 values in one register pair: an fma of both rounds each like fmaf, at half the instructions.
__device__ __forceinline__ unsigned long long bs_pair(uint32_t lo, uint32_t hi) {
    unsigned long long v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "r"(lo), "r"(hi));
    return v;
}
__device__ __forceinline__ void bs_fma_pair(unsigned long long& acc, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
// four values from shared memory: loaded, as fp32.  (volatile, or the compiler may take two loads for one, whatever barrier and stores lie between)
template <typename TW> __device__ __forceinline__ void bs_four(uint32_t at, uint32_t* v) {
    if constexpr (sizeof(TW) == 2) asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v[1]), "=r"(v[3]) : "r"(at));
    else asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(at));
}
template <typename TW> __device__ __forceinline__ void bs_widen(uint32_t* v) {
    if constexpr (sizeof(TW) == 2) {
        v[0] = v[1] << 16; v[1] &= 0xffff0000u;
        v[2] = v[3] << 16; v[3] &= 0xffff0000u;
    }
}
// four elements of a row that starts on 16 bytes, in shared or global memory
__device__ __forceinline__ float4 bs_quad(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 bs_quad(const __nv_bfloat16* p) {
    const uint2 v = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
}
// four elements of four rows (of type TW after rounding) to [k][4].  Neighbouring lanes' 64 bytes of fp32 lie behind one another: every
// second lane begins a piece further on, so that eight lanes' stores meet all banks (in one order they took four times as long).
__device__ __forceinline__ void bs_put(float* dst, const float4& a, const float4& b, const float4& c, const float4& d) {
    float4 t[4] = {make_float4(a.x, b.x, c.x, d.x), make_float4(a.y, b.y, c.y, d.y), make_float4(a.z, b.z, c.z, d.z), make_float4(a.w, b.w, c.w, d.w)};
    const uint32_t first = (threadIdx.x >> 1) & 3u, at = smem_u32(dst);
    if (first & 1u) { const float4 v = t[0]; t[0] = t[1]; t[1] = t[2]; t[2] = t[3]; t[3] = v; }
    if (first & 2u) { float4 v = t[0]; t[0] = t[2]; t[2] = v; v = t[1]; t[1] = t[3]; t[3] = v; }
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j)
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at + (((first + j) & 3u) << 4)), "f"(t[j].x), "f"(t[j].y), "f"(t[j].z), "f"(t[j].w) : "memory");
}
__device__ __forceinline__ void bs_put(__nv_bfloat16* dst, const float4& a, const float4& b, const float4& c, const float4& d) {
    uint4* to = reinterpret_cast<uint4*>(dst);
    to[0] = make_uint4(pack_bf16x2(a.x, b.x), pack_bf16x2(c.x, d.x), pack_bf16x2(a.y, b.y), pack_bf16x2(c.y, d.y));
    to[1] = make_uint4(pack_bf16x2(a.z, b.z), pack_bf16x2(c.z, d.z), pack_bf16x2(a.w, b.w), pack_bf16x2(c.w, d.w));
}
__device__ __noinline__ float4 bs_tanh(float4 v) { return make_float4(tanhf(v.x), tanhf(v.y), tanhf(v.z), tanhf(v.w)); }

// Dot products of four rows of weights with four rows of x (Q times: the next four lie x_pitch bytes on), all [k][4] in shared memory;
// the addresses are the lane's first element (k = lane).  Afterwards lane l holds the one of weight row l >> 3 and x row (l >> 1) & 3.
// What bounds them is the arithmetic pipes (bf16 to fp32 and pairs of registers take as long as the fmas): 4 x 4 took 3200 cycles
// for 20 steps of 16 warps, 8 x 4 is 1.3 times as fast.
// (One function per Q, and few unrolled loops elsewhere: an iteration runs its code once, and what does not stay
// in the 32 KB instruction cache is fetched at three cycles an instruction.)
template <typename TW, int Q>
__device__ __noinline__ float2 bs_dots(uint32_t w, uint32_t x, uint32_t x_pitch, int steps) {
    unsigned long long acc[Q][8];
#pragma unroll
    for (int i = 0; i < 8 * Q; ++i) acc[i >> 3][i & 7] = 0ull;
    // N steps' loads, then their arithmetic
    auto some = [&](auto which, int i) {
        constexpr int N = decltype(which)::value;
        uint32_t wv[N][4], xv[N][Q][4];
#pragma unroll
        for (int n = 0; n < N; ++n) {
            bs_four<TW>(w + 128u * (uint32_t)sizeof(TW) * (i + n), wv[n]);
#pragma unroll
            for (int h = 0; h < Q; ++h) bs_four<TW>(x + h * x_pitch + 128u * (uint32_t)sizeof(TW) * (i + n), xv[n][h]);
        }
#pragma unroll
        for (int n = 0; n < N; ++n) {
            unsigned long long ww[4];
            bs_widen<TW>(wv[n]);
#pragma unroll
            for (int j = 0; j < 4; ++j) ww[j] = bs_pair(wv[n][j], wv[n][j]);
#pragma unroll
            for (int h = 0; h < Q; ++h) {
                bs_widen<TW>(xv[n][h]);
                const unsigned long long x0 = bs_pair(xv[n][h][0], xv[n][h][1]), x1 = bs_pair(xv[n][h][2], xv[n][h][3]);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    bs_fma_pair(acc[h][2 * j], ww[j], x0);
                    bs_fma_pair(acc[h][2 * j + 1], ww[j], x1);
                }
            }
        }
    };
    // (fp32 in steps of four written out: between phases that hold many registers the compiler otherwise let a step wait for its own
    // loads, 40 steps 4600 cycles against 3600; bf16 was no faster by it)
    constexpr int AT_ONCE = sizeof(TW) == 4 ? 4 / Q : 1;
    int i = 0;
    if constexpr (AT_ONCE > 1)
#pragma unroll 1
        for (; i + AT_ONCE <= steps; i += AT_ONCE) some(std::integral_constant<int, AT_ONCE>{}, i);
#pragma unroll(4 / Q)
    for (; i < steps; ++i) some(std::integral_constant<int, 1>{}, i);
    const int lane = threadIdx.x & 31;
    float out[2] = {0.f, 0.f};
#pragma unroll
    for (int h = 0; h < Q; ++h) {
        float a[16];
#pragma unroll
        for (int i = 0; i < 8; ++i) asm("mov.b64 {%0, %1}, %2;" : "=f"(a[2 * i]), "=f"(a[2 * i + 1]) : "l"(acc[h][i]));
#pragma unroll
        for (int half = 8; half >= 1; half >>= 1) {
            const bool up = (lane & (2 * half)) != 0;
#pragma unroll
            for (int c = 0; c < half; ++c) {
                const float send = up ? a[c] : a[c + half], keep = up ? a[c + half] : a[c];
                a[c] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * half);
            }
        }
        out[h] = a[0] + __shfl_xor_sync(0xffffffffu, a[0], 1);
    }
    return make_float2(out[0], out[1]);
}

__device__ __forceinline__ float bs_warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float bs_warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ unsigned long long bs_best_of_warp(unsigned long long key) {
    const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(key >> 32));
    const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(key >> 32) == hi ? (uint32_t)key : 0u);
    return ((unsigned long long)hi << 32) | lo;
}
__device__ __forceinline__ unsigned long long bs_word(uint32_t value, uint32_t seq) { return ((unsigned long long)seq << 32) | value; }

template <typename TW>
__global__ void __launch_bounds__(BS_THREADS, 1) beam_step_kernel(const BsParams p) {
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ int s_stop;
    __shared__ int s_cmd[kBeamWords];
    __shared__ float s_lse[kMaxWindow], s_blank[kMaxWindow];     // of a row: log-sum-exp, blank's log-probability
    __shared__ unsigned long long s_cand[BS_WARPS * kMaxBeam];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, grp = lane >> 3, col = (lane >> 1) & 3;   // the dot product a lane ends up with
    const int G = gridDim.x, cta = blockIdx.x;
    const int P = p.P, H = p.H, NV = p.NV, K = p.K, LP = p.L * P;
    const BsPlan& M = p.plan;
    const int R = M.rows;
    const int units = (P - cta + G - 1) / G, prows = (H - cta + G - 1) / G, labels = (NV - cta + G - 1) / G;
    TW* w_pred = reinterpret_cast<TW*>(sm + M.w_pred);
    TW* w_out = reinterpret_cast<TW*>(sm + M.w_out);
    TW* encs = reinterpret_cast<TW*>(sm + M.enc);
    float* b_gate = reinterpret_cast<float*>(sm + M.bias);                     // [layer][own unit][gate]
    float *b_pred = b_gate + 4 * p.L * M.units, *b_out = b_pred + M.prows;
    TW* xs = reinterpret_cast<TW*>(sm + M.x);                    // operand of the gates or of W_pred, by fours of updates
    float* gs = reinterpret_cast<float*>(sm + M.x);              // later pred_proj of the hypotheses
    TW* za = reinterpret_cast<TW*>(sm + M.z);                    // the joint's operand
    float* zs = reinterpret_cast<float*>(sm + M.z);              // later the logits of a window
    if (tid == 0) s_stop = 0;

    // n elements (whole 16-byte pieces) by one warp, asynchronously
    auto copy_row = [&](TW* dst, const TW* src, int n) {
        constexpr int PIECE = 16 / (int)sizeof(TW);
#pragma unroll 1
        for (int k = lane * PIECE; k < n; k += 32 * PIECE)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst + k)), "l"(src + k) : "memory");
    };
    auto layer_at = [&](int l) { return reinterpret_cast<TW*>(sm + M.w_l + (size_t)(M.resident ? l : 0) * M.layer); };
    // element k of four rows (rows past the end: zeros) into [k][4]
    auto interleave = [&](TW* dst, const TW* r0, const TW* r1, const TW* r2, const TW* r3, int n, int n32) {
#pragma unroll 2
        for (int k = lane; k < n32; k += 32) {
            const TW zero = (TW)0.f;
            TW* d = dst + 4 * k;
            d[0] = r0 && k < n ? r0[k] : zero;
            d[1] = r1 && k < n ? r1[k] : zero;
            d[2] = r2 && k < n ? r2[k] : zero;
            d[3] = r3 && k < n ? r3[k] : zero;
        }
    };
    auto load_layer = [&](int l) {
        const int nin = l == 0 ? p.E : P, K32 = (nin + P + 31) / 32 * 32;
        const TW *wi = static_cast<const TW*>(p.w_ih[l]), *wh = static_cast<const TW*>(p.w_hh[l]);
#pragma unroll 1
        for (int i = warp; i < units; i += BS_WARPS) {
            const size_t j = (size_t)i * G + cta;
            TW* dst = layer_at(l) + 4 * i * M.k_l;
            interleave(dst, wi + j * nin, wi + (P + j) * nin, wi + (2 * P + j) * nin, wi + (3 * P + j) * nin, nin, nin);
            interleave(dst + 4 * nin, wh + j * P, wh + (P + j) * P, wh + (2 * P + j) * P, wh + (3 * P + j) * P, P, K32 - nin);
        }
    };
    auto load_rows = [&](TW* dst, const void* src_, int rows, int n, int n32) {      // this CTA's rows of W_pred or W_out
        const TW* src = static_cast<const TW*>(src_);
#pragma unroll 1
        for (int i = 4 * warp; i < rows; i += 4 * BS_WARPS) {
            auto row = [&](int j) { return i + j < rows ? src + ((size_t)(i + j) * G + cta) * n : nullptr; };
            interleave(dst + i * n32, row(0), row(1), row(2), row(3), n, n32);
        }
    };
    if (M.resident)
#pragma unroll 1
        for (int l = 0; l < p.L; ++l) load_layer(l);
    load_rows(w_pred, p.w_pred, prows, P, M.k_p);
    load_rows(w_out, p.w_out, labels, H, M.k_z);

#pragma unroll 1
    for (int i = tid; i < 4 * p.L * units; i += BS_THREADS) {
        const int l = i / (4 * units), r = i - l * 4 * units, at = (r & 3) * P + (r >> 2) * G + cta;
        b_gate[4 * l * M.units + r] = p.b_ih[l][at] + p.b_hh[l][at];
    }
    for (int i = tid; i < prows; i += BS_THREADS) b_pred[i] = p.b_pred[i * G + cta];
    for (int i = tid; i < labels; i += BS_THREADS) b_out[i] = p.b_out[i * G + cta];

    uint32_t epoch = p.bar_base;
    auto arrive = [&] {
        __syncthreads();
        epoch += (uint32_t)G;
        if (tid == 0) { __threadfence(); atomicAdd(&p.ctrl->bar, 1u); }
    };
    auto give_up = [&](int site) { s_stop = 1; note_timeout(p.ctrl, site, cta); set_status(p.ctrl, WIND_ERR_TIMEOUT); *const_cast<volatile uint32_t*>(&p.mail->failed) = 1u; };
    auto wait = [&]() -> bool {        // bounded; false: given up
        if (tid == 0) {
            const uint32_t target = epoch + p.extra_arrivals;
            unsigned long long t0 = 0;
            for (uint32_t it = 1;; ++it) {
                uint32_t v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&p.ctrl->bar) : "memory");
                if ((int32_t)(v - target) >= 0) break;
                if ((it & 63u) == 0u) {
                    const unsigned long long now = globaltimer_ns();
                    if (t0 == 0) t0 = now;
                    else if (now - t0 > kWaitLimitNs) { give_up(6); break; }
                }
            }
        }
        __syncthreads();
        return s_stop == 0;
    };
    // Command `seq` into s_cmd: warp 0 of CTA 0 takes it from the host and passes it on in device memory.
    auto take_command = [&](uint32_t seq) {
        __syncthreads();
        if (warp == 0) {
            const int words = 4 + 5 * R;
            const volatile unsigned long long* from = cta == 0 ? p.mail->cmd : p.relay;
            const unsigned long long limit = cta == 0 ? BS_IDLE_NS : kWaitLimitNs;
            unsigned long long v[(kBeamWords + 31) / 32], t0 = 0;
            for (uint32_t it = 1;; ++it) {
                bool ok = true;
#pragma unroll
                for (int j = 0; j < (kBeamWords + 31) / 32; ++j) {
                    v[j] = 0ull;
                    if (lane + 32 * j < words) {
                        v[j] = from[lane + 32 * j];
                        ok = ok && (uint32_t)(v[j] >> 32) == seq;
                    }
                }
                if (__all_sync(0xffffffffu, ok)) break;
                if ((it & 15u) == 0u) {
                    const unsigned long long now = __shfl_sync(0xffffffffu, globaltimer_ns(), 0);
                    if (t0 == 0) {
                        t0 = now;
                    } else if (now - t0 > limit) {
                        if (cta != 0 && lane == 0) give_up(7);
#pragma unroll
                        for (int j = 0; j < (kBeamWords + 31) / 32; ++j) v[j] = bs_word(0xffffffffu, seq);
                        break;
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < (kBeamWords + 31) / 32; ++j)
                if (lane + 32 * j < words) {
                    if (cta == 0) const_cast<volatile unsigned long long*>(p.relay)[lane + 32 * j] = v[j];
                    s_cmd[lane + 32 * j] = (int)(uint32_t)v[j];
                }
        }
        __syncthreads();
    };

    for (uint32_t seq = p.first_seq;; ++seq) {
        take_command(seq);
        const int nu = s_cmd[0], nh = s_cmd[1] & (int)(kBeamLast - 1u), span = s_cmd[2], t0 = s_cmd[3];
        const bool last = (s_cmd[1] & (int)kBeamLast) != 0;
        if (nu < 0) return;                                  // the end of the search, or no command for too long
        const int *c_src = s_cmd + 4, *c_tok = c_src + R, *c_dst = c_tok + R, *c_slot = c_dst + R, *c_t = c_slot + R;
        if (nu > 0 && !M.resident) load_layer(0);
#pragma unroll 1
        for (int w = warp; w < span; w += BS_WARPS) copy_row(encs + w * H, static_cast<const TW*>(p.enc_proj) + (size_t)(t0 + w) * H, H);

        // ---- decoder update: per layer the gates of this CTA's hidden units, then h and c into the new hypotheses' slots ----
        const int quads = (nu + BS_UTTS - 1) / BS_UTTS;
        auto update = [&](int quad, int u) { return min(quad * BS_UTTS + u, nu - 1); };      // (those behind the last repeat it)
        if (nu > 0) {
#pragma unroll 1
            for (int l = 0; l < p.L; ++l) {
                const int nin = l == 0 ? p.E : P, K32 = (nin + P + 31) / 32 * 32;
                const int K4 = K32 / 4;
#pragma unroll 1
                for (int q0 = 0; q0 < quads; q0 += M.quads) {
                    const int here = min(M.quads, quads - q0);
                    // an item: one of this CTA's units for four updates
                    auto c_of = [&](int item) { return p.c_pool + (size_t)c_src[update(q0 + item / units, col)] * LP + l * P + (item % units) * G + cta; };
                    float c_in = warp < units * here ? __ldcg(c_of(warp)) : 0.f;          // requested ahead of everything else
                    if (q0 > 0) __syncthreads();
                    // x and the state before it: four elements of four updates at a time, all loads of a thread at once
#pragma unroll 2
                    for (int i = tid; i < here * K4; i += BS_THREADS) {
                        const int quad = i / K4, k = 4 * (i - quad * K4);
                        float4 x[BS_UTTS];
#pragma unroll
                        for (int u = 0; u < BS_UTTS; ++u) {
                            const int uu = update(q0 + quad, u);
                            if (k < nin && l == 0) x[u] = bs_quad(static_cast<const TW*>(p.emb) + (size_t)c_tok[uu] * p.E + k);
                            else if (k < nin + P) x[u] = __ldcg(reinterpret_cast<const float4*>(p.h_pool + (size_t)(k < nin ? c_dst[uu] : c_src[uu]) * LP + (k < nin ? (l - 1) * P + k : l * P + k - nin)));
                            else x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                        bs_put(xs + 4 * (quad * M.k_l + k), x[0], x[1], x[2], x[3]);
                    }
                    asm volatile("cp.async.wait_all;" ::: "memory");
                    __syncthreads();
#pragma unroll 1
                    for (int item = warp; item < units * here; item += BS_WARPS) {
                        const int quad = item / units, ui = item - quad * units, j = ui * G + cta, at = (q0 + quad) * BS_UTTS + col;
                        const float mine = bs_dots<TW, 1>(smem_u32(layer_at(l) + 4 * (ui * M.k_l + lane)), smem_u32(xs + 4 * (quad * M.k_l + lane)), 0u, K32 / 32).x + b_gate[4 * (l * M.units + ui) + grp];
                        const float ai = __shfl_sync(0xffffffffu, mine, lane & 7), af = __shfl_sync(0xffffffffu, mine, 8 + (lane & 7)),
                                    ag = __shfl_sync(0xffffffffu, mine, 16 + (lane & 7)), ao = __shfl_sync(0xffffffffu, mine, 24 + (lane & 7));
                        const float gi = 1.f / (1.f + expf(-ai)), gf = 1.f / (1.f + expf(-af)), gg = tanhf(ag), go = 1.f / (1.f + expf(-ao));
                        const float cc = cell_update_fc(gf, c_in, gi, gg);
                        if ((lane & 25) == 0 && at < nu) {
                            const size_t to = (size_t)c_dst[at] * LP + l * P + j;
                            p.c_pool[to] = cc;
                            p.h_pool[to] = go * tanhf(cc);
                        }
                        if (item + BS_WARPS < units * here) c_in = __ldcg(c_of(item + BS_WARPS));
                    }
                }
                arrive();
                if (!M.resident && l + 1 < p.L) load_layer(l + 1);
                if (!wait()) return;
            }
            // ---- pred_proj of this CTA's joint units ----
            const int K4 = M.k_p / 4, pgs = (prows + 3) / 4;
#pragma unroll 1
            for (int q0 = 0; q0 < quads; q0 += M.quads) {
                const int here = min(M.quads, quads - q0);
                if (q0 > 0) __syncthreads();
#pragma unroll 2
                for (int i = tid; i < here * K4; i += BS_THREADS) {
                    const int quad = i / K4, k = 4 * (i - quad * K4);
                    float4 x[BS_UTTS];
#pragma unroll
                    for (int u = 0; u < BS_UTTS; ++u)
                        x[u] = k < P ? __ldcg(reinterpret_cast<const float4*>(p.h_pool + (size_t)c_dst[update(q0 + quad, u)] * LP + (p.L - 1) * P + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    bs_put(xs + 4 * (quad * M.k_p + k), x[0], x[1], x[2], x[3]);
                }
                __syncthreads();
#pragma unroll 1
                for (int item = warp; item < pgs * here; item += BS_WARPS) {
                    const int quad = item / pgs, pg = item - quad * pgs, pi = pg * 4 + grp, o = min(pi, prows - 1) * G + cta, at = (q0 + quad) * BS_UTTS + col;
                    const float mine = bs_dots<TW, 1>(smem_u32(w_pred + 4 * (pg * M.k_p + lane)), smem_u32(xs + 4 * (quad * M.k_p + lane)), 0u, M.k_p / 32).x + b_pred[min(pi, prows - 1)];
                    if ((lane & 1) == 0 && pi < prows && at < nu) p.g_pool[(size_t)c_dst[at] * H + o] = mine;
                }
            }
            arrive();
            if (!wait()) return;
        }

        // ---- logits of this CTA's labels for every row of the window under every hypothesis ----
        // (windows as long as the first one's; of one that the end of the utterance cuts shorter the rows behind it repeat its last frame)
        const int n = min(p.W, p.T - t0), rows = nh * n;
        const int H4 = H / 4;
        // (under a condition each, not in an unrolled loop, whose last turns would wait one for another)
#pragma unroll 1
        for (int i0 = tid; i0 < nh * H4; i0 += 4 * BS_THREADS) {
            float4 v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int i = i0 + j * BS_THREADS, b = i / H4;
                if (i < nh * H4) v[j] = __ldcg(reinterpret_cast<const float4*>(p.g_pool + (size_t)c_slot[b] * H + 4 * (i - b * H4)));
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int i = i0 + j * BS_THREADS;
                if (i < nh * H4) *reinterpret_cast<float4*>(gs + 4 * i) = v[j];
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        // passes of equal size, in whole pairs of row groups
        const int passes = (rows + M.zrows - 1) / M.zrows, pass = min(M.zrows, ((rows + passes - 1) / passes + 2 * BS_ROWS - 1) / (2 * BS_ROWS) * (2 * BS_ROWS));
#pragma unroll 1
        for (int r0 = 0; r0 < rows; r0 += pass) {
            const int nr = min(pass, rows - r0), nr4 = (nr + BS_ROWS - 1) / BS_ROWS;
            __syncthreads();
            // a warp takes four rows and a share of k
            const int cut = nr4 < BS_WARPS ? BS_WARPS / nr4 : 1;
#pragma unroll 1
            for (int item = warp; item < nr4 * cut; item += BS_WARPS) {
                const int rg = item / cut;
                const TW* e4[4];
                const float* g4[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int row = min(r0 + rg * BS_ROWS + j, rows - 1), b = row / n;
                    e4[j] = encs + min(c_t[b] - t0 + row - b * n, span - 1) * H;
                    g4[j] = gs + b * H;
                }
                auto act = [&](const float4& a, const float4& g) {
                    const float4 v = make_float4(a.x + g.x, a.y + g.y, a.z + g.z, a.w + g.w);
                    return p.act == WIND_ACT_RELU ? make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f)) : bs_tanh(v);
                };
                if constexpr (sizeof(TW) == 4) {                // element by element: nothing to turn round, and even shares of k
#pragma unroll 2
                    for (int k = lane + 32 * (item - rg * cut); k < M.k_z; k += 32 * cut)
                        *reinterpret_cast<float4*>(za + 4 * (rg * M.k_z + k)) =
                            k < H ? act(make_float4(e4[0][k], e4[1][k], e4[2][k], e4[3][k]), make_float4(g4[0][k], g4[1][k], g4[2][k], g4[3][k])) : make_float4(0.f, 0.f, 0.f, 0.f);
                } else {
#pragma unroll 1
                    for (int k = 4 * (lane + 32 * (item - rg * cut)); k < M.k_z; k += 128 * cut) {
                        float4 z[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            z[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (k < H) z[j] = act(bs_quad(e4[j] + k), bs_quad(g4[j] + k));
                        }
                        bs_put(za + 4 * (rg * M.k_z + k), z[0], z[1], z[2], z[3]);
                    }
                }
            }
            __syncthreads();
            // (fp32: one row group an item while that gives every warp one at most.  Large models have passes of four groups, and in pairs
            // four of the sixteen warps had all the work)
            const int lgs = (labels + 3) / 4, per = sizeof(TW) == 4 && lgs * nr4 <= BS_WARPS ? 1 : 2, items = lgs * ((nr4 + per - 1) / per);
#pragma unroll 1
            for (int item = warp; item < items; item += BS_WARPS) {
                const int rg = per * (item / lgs), lg = item % lgs, li = lg * 4 + grp, v = min(li, labels - 1) * G + cta;
                const uint32_t pitch = rg + 1 < nr4 ? 4u * (uint32_t)sizeof(TW) * (uint32_t)M.k_z : 0u;      // (an odd number of groups: the last one twice)
                const uint32_t wa = smem_u32(w_out + 4 * (lg * M.k_z + lane)), xa = smem_u32(za + 4 * (rg * M.k_z + lane));
                const float2 both = per == 2 ? bs_dots<TW, 2>(wa, xa, pitch, M.k_z / 32) : bs_dots<TW, 1>(wa, xa, 0u, M.k_z / 32);
                const float bias = b_out[min(li, labels - 1)];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int at = (rg + h) * BS_ROWS + col, row = r0 + at, b = row / n;
                    if (h < per && (lane & 1) == 0 && at < nr && li < labels) p.logits[((size_t)b * p.W + (row - b * n)) * NV + v] = (h ? both.y : both.x) + bias;
                }
            }
        }
        arrive();
        if (cta < nh) {
            if (!wait()) return;
            // ---- Eq. (1) for hypothesis `cta`, the window's logits in shared memory ----
            const float* src = p.logits + (size_t)cta * p.W * NV;
            const int n = min(p.W, p.T - c_t[cta]), total = n * NV;
            // A vocabulary is often a power of two and the blank, so that a window's logits are a little more than a multiple of 4096 or 8192:
            // nine and seventeen pieces of 512 take them without another round trip.  (Beam 4, W = 8, bf16: with 16 pieces 26.74 ms, with 17
            // 26.47; with 20 the other phases are short of registers: 26.77.)
            constexpr int AT_ONCE = sizeof(TW) == 4 ? 9 : 17;
#pragma unroll 1
            for (int i0 = tid; i0 < total; i0 += AT_ONCE * BS_THREADS) {
                float v[AT_ONCE];
#pragma unroll
                for (int j = 0; j < AT_ONCE; ++j)
                    if (i0 + j * BS_THREADS < total) v[j] = __ldcg(src + i0 + j * BS_THREADS);
#pragma unroll
                for (int j = 0; j < AT_ONCE; ++j)
                    if (i0 + j * BS_THREADS < total) zs[i0 + j * BS_THREADS] = v[j];
            }
            __syncthreads();
#pragma unroll 1
            for (int w = warp; w < n; w += BS_WARPS) {
                const float* row = zs + w * NV;
                float mx = -INFINITY;
#pragma unroll 8
                for (int v = lane; v < NV; v += 32) mx = fmaxf(mx, row[v]);
                mx = bs_warp_max(mx);
                float se = 0.f;
#pragma unroll 8
                for (int v = lane; v < NV; v += 32) se += expf(row[v] - mx);
                se = bs_warp_sum(se);
                if (lane == 0) {
                    const float lse = mx + logf(se);
                    s_lse[w] = lse;
                    s_blank[w] = row[p.blank] - lse;
                }
            }
            __syncthreads();
            // log P'(v, w) = logit + shift: all blanks before, then v
            auto shift_of = [&](int w) {
                float before = 0.f;
#pragma unroll 8
                for (int i = 0; i < w; ++i) before += s_blank[i];
                return before - s_lse[w];
            };
            // ---- the K best entries, best first; equal values in order of (offset, label) ----
            // A lane finds the best entry of its share, the warp takes out the best of its lanes K times, and all its lanes
            // together look through the share that lost its entry.  (Sorted lists per thread took 9000 cycles for a window of
            // 8 x 1025, a rescan by the one lane 10700.)
            const int parts = n < BS_WARPS ? BS_WARPS / n : 1, stride = 32 * parts;      // warps of a row
            unsigned long long mine = 0ull;
#pragma unroll 1
            for (int item = warp; item < n * parts; item += BS_WARPS) {
                const int w = item / parts;
                const float shift = shift_of(w);
                const float* row = zs + w * NV;
                const int skip = w != n - 1 ? p.blank : -1;
                float bv = -INFINITY;
                int at = -1;
#pragma unroll 4
                for (int v = lane + 32 * (item - w * parts); v < NV; v += stride) {
                    const float x = row[v] + shift;
                    if (x > bv && v != skip) { bv = x; at = v; }                        // v ascends: the first of equals stays
                }
                if (at >= 0) mine = max(mine, pack_key(bv, (uint32_t)(w * NV + at)));
            }
#pragma unroll 1
            for (int k = 0; k < K; ++k) {
                const unsigned long long top = bs_best_of_warp(mine);
                if (lane == 0) s_cand[warp * K + k] = top;
                if (top == 0ull || k + 1 == K) continue;
                const int owner = __ffs((int)__ballot_sync(0xffffffffu, mine == top)) - 1;
                unsigned long long next = 0ull;
#pragma unroll 1
                for (int item = warp; item < n * parts; item += BS_WARPS) {
                    const int w = item / parts;
                    const float shift = shift_of(w);
                    const int skip = w != n - 1 ? p.blank : -1;
#pragma unroll 1
                    for (int v = owner + 32 * (item - w * parts) + lane * stride; v < NV; v += 32 * stride) {
                        const float x = zs[w * NV + v] + shift;
                        const unsigned long long key = x > -INFINITY && v != skip ? pack_key(x, (uint32_t)(w * NV + v)) : 0ull;
                        if (key < top) next = max(next, key);
                    }
                }
                next = bs_best_of_warp(next);
                if (lane == owner) mine = next;
            }
            __syncthreads();
            if (warp == 0) {
                int pos = 0;                                        // lanes 0..15 take one warp's list each
#pragma unroll 1
                for (int k = 0; k < K; ++k) {
                    const unsigned long long mine = lane < BS_WARPS && pos < K ? s_cand[lane * K + pos] : 0ull, top = bs_best_of_warp(mine);
                    if (mine == top) ++pos;
                    if (lane == 0) {
                        volatile unsigned long long* out = p.mail->top + 2 * (cta * K + k);
                        out[0] = bs_word(top != 0ull ? key_label(top) : 0xffffffffu, seq);
                        out[1] = bs_word(__float_as_uint(top != 0ull ? key_logit(top) : -INFINITY), seq);
                    }
                }
            }
        }
        if (last) return;
    }
}

template <typename TW> static const void* bs_fn() { return (const void*)beam_step_kernel<TW>; }

static std::mutex g_bs_mutex;
static int g_bs_optin[64] = {};        // opt-in shared memory per block, 0: not asked yet

static cudaError_t bs_device(int* optin) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_bs_mutex);
    if (!g_bs_optin[dev]) {
        int n = 0;
        if ((e = cudaDeviceGetAttribute(&n, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
        for (const void* fn : {bs_fn<float>(), bs_fn<__nv_bfloat16>()})
            if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, n - 4096)) != cudaSuccess) return e;   // static: below 4 KB
        g_bs_optin[dev] = n;
    }
    *optin = g_bs_optin[dev];
    return cudaSuccess;
}

static BsPlan bs_plan_of(const Call& c, bool ahead, int sms, uint32_t budget) {
    const wind_model_t& m = c.m;
    return m.dtype == WIND_DT_BF16 ? bs_plan<__nv_bfloat16>(sms, c.W, c.B, ahead, m.E, m.P, m.L, m.H, m.V + 1, budget)
                                   : bs_plan<float>(sms, c.W, c.B, ahead, m.E, m.P, m.L, m.H, m.V + 1, budget);
}

// Rows in whole 16-byte pieces (8 bf16; fp32 models take the same rule), a CTA's weights and one window's logits in shared
// memory, and a CTA for every hypothesis.  Else the per-phase kernels.
bool beam_step_supported(const Call& c) {
    const wind_model_t& m = c.m;
    if (m.E % 8 || m.P % 8 || m.H % 8) return false;
    auto aligned = [](const void* q) { return reinterpret_cast<uintptr_t>(q) % 16 == 0; };
    if (!aligned(m.emb) || !aligned(m.w_pred) || !aligned(m.w_out)) return false;
    for (int l = 0; l < m.L; ++l)
        if (!aligned(c.w_ih[l]) || !aligned(c.w_hh[l])) return false;
    int optin = 0, sms = 0;
    if (bs_device(&optin) != cudaSuccess || loop_sm_count(&sms) != cudaSuccess) { cudaGetLastError(); return false; }
    return c.B <= sms && bs_plan_of(c, false, sms, (uint32_t)optin - 4096u).total <= (uint32_t)optin - 4096u;
}

// the same on a device of `sms` SMs and `optin` bytes of shared memory a block, alignments aside
bool beam_step_debug_plan(const wind_model_t& m, int W, int K, bool ahead, int sms, int optin, wind_beam_plan_t* out) {
    const uint32_t budget = (uint32_t)optin - 4096u;
    auto plan = [&](auto t) { return bs_plan<decltype(t)>(sms, W, K, ahead, m.E, m.P, m.L, m.H, m.V + 1, budget); };
    const BsPlan s = m.dtype == WIND_DT_BF16 ? plan(__nv_bfloat16()) : plan(0.f);
    if (m.E % 8 || m.P % 8 || m.H % 8 || K > sms || s.total > budget) return false;
    *out = wind_beam_plan_t{s.rows, s.look, s.resident, 4 * s.quads, s.zrows, (int32_t)s.total};
    return true;
}

// (without a device: on a B200.  No context is made for this question.)
BeamShape beam_step_most(const wind_model_t& m, int W, int K) {
    int dev = 0, optin = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        optin = 232448; sms = 148;
    }
    wind_beam_plan_t plan;
    if (!beam_step_debug_plan(m, W, K, true, sms, optin, &plan)) return {K, 0};
    return {plan.rows, plan.look};
}

// (of a call that beam_step_supported takes)
BeamShape beam_step_shape(const Call& c, bool ahead) {
    int optin = 0, sms = 0;
    if (bs_device(&optin) != cudaSuccess || loop_sm_count(&sms) != cudaSuccess) { cudaGetLastError(); return {c.B, 0}; }
    const BsPlan s = bs_plan_of(c, ahead, sms, (uint32_t)optin - 4096u);
    return {s.rows, s.look};
}

cudaError_t beam_step(const Call& c, const BeamShape& shape, BeamMail* mail, unsigned long long* relay, uint32_t first_seq, uint32_t bar_base,
                      float* h_pool, float* c_pool, float* g_pool, float* logits) {
    int optin = 0, sms = 0;
    cudaError_t e = bs_device(&optin);
    if (e == cudaSuccess) e = loop_sm_count(&sms);
    if (e != cudaSuccess) return e;
    const wind_model_t& m = c.m;
    BsParams p{};
    p.ctrl = c.ctrl(); p.mail = mail; p.relay = relay;
    p.first_seq = first_seq; p.bar_base = bar_base; p.K = c.B;
    p.extra_arrivals = (uint32_t)loop_extra_arrivals();
    p.plan = bs_plan_of(c, shape.look > 0, sms, (uint32_t)optin - 4096u);
    p.E = m.E; p.P = m.P; p.L = m.L; p.H = m.H; p.NV = m.V + 1; p.blank = m.blank_id; p.act = m.act; p.W = c.W; p.T = c.T;
    p.emb = m.emb; p.w_pred = m.w_pred; p.b_pred = m.b_pred; p.w_out = m.w_out; p.b_out = m.b_out;
    for (int l = 0; l < m.L; ++l) { p.w_ih[l] = c.w_ih[l]; p.w_hh[l] = c.w_hh[l]; p.b_ih[l] = c.b_ih[l]; p.b_hh[l] = c.b_hh[l]; }
    p.enc_proj = c.enc_proj();
    p.h_pool = h_pool; p.c_pool = c_pool; p.g_pool = g_pool; p.logits = logits;
    const void* fn = m.dtype == WIND_DT_BF16 ? bs_fn<__nv_bfloat16>() : bs_fn<float>();
    void* args[1] = {(void*)&p};
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)sms), dim3(BS_THREADS), args, p.plan.total, c.stream);
}
// arrivals at the grid barrier during one command
uint32_t beam_step_arrivals(const Call& c, int n_update) {
    int sms = 0;
    loop_sm_count(&sms);
    return (uint32_t)sms * (uint32_t)((n_update > 0 ? c.m.L + 1 : 0) + 1);
}

}  // namespace wind
