// The decoding loop of the plain-ALU path (fp32 models, and bf16 models outside the tensor-core set) as one persistent kernel.
//
// As separate kernels in a CUDA graph a lock step cost 20 us for a model of 64 units (launches) and 300 us for one of 640
// units in fp32 (every weight read again by kernels with one block per output).  Here the weights stay in shared memory:
//   LOCAL   the whole decoder fits one SM (64 units in fp32: 155 KB): a CTA decodes its utterances one after the other and
//           nothing leaves the SM but the transcripts; the phases of a step are separated by block barriers.
//   grid    otherwise: hidden units, joint units and labels are dealt out over all SMs (640 units in fp32: 117 KB each), and
//           the phases are separated by grid barriers (1.3 us each).  Models whose weights do not fit on the chip run the
//           same code and read them from L2.
//
// Phases of a lock step (Algorithm 2 for every utterance at once):
//   control   every CTA takes the decisions for all utterances from the window's keys (the same ones everywhere), CTA 0
//             records them; without an emission in the batch the two decoder phases are skipped
//   update    per layer: gates = W_ih x + W_hh h, cell update (a warp takes a hidden unit's four rows and a part of K)
//   project   pred_proj = W_pred h, then z = act(enc_proj + pred_proj) for the joint units of this CTA
//   joint     logits = W_out z for this CTA's labels, the best (logit, label) key of every window row
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
constexpr int SL_ROWS = 4;          // window rows and
constexpr int SL_LABELS = 4;        // labels of a joint item
constexpr int SL_MAX_B = 512;       // most utterances (their state is kept in every CTA)

struct SimtLoopParams {
    Ctrl* ctrl;
    int B, T, W, S, max_out, E, P, L, H, NV, blank, act, step_cap, resident, extra_arrivals;
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
    float* h;                      // [2][L][B][P], a parity per utterance          (grid mode; LOCAL: shared memory)
    float* c;                      // [L][B][P]
    void* z;                       // [B * W][H]
    unsigned long long* keys;      // [2][B * W]
    int32_t* out_tokens;
    int32_t* out_frames;
    int32_t* out_len;
};

// ---- four consecutive operands as floats; VEC: one load, else element by element ----
template <bool VEC> __device__ __forceinline__ float4 sl_load4(const float* p) {
    if (VEC) return *reinterpret_cast<const float4*>(p);
    return make_float4(p[0], p[1], p[2], p[3]);
}
template <bool VEC> __device__ __forceinline__ float4 sl_load4(const __nv_bfloat16* p) {
    if (VEC) {
        const uint2 v = *reinterpret_cast<const uint2*>(p);
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    return make_float4(__bfloat162float(p[0]), __bfloat162float(p[1]), __bfloat162float(p[2]), __bfloat162float(p[3]));
}
// of a row of n elements from element k on: zeros behind its end
template <bool VEC, typename T> __device__ __forceinline__ float4 sl_row4(const T* row, int k, int n) {
    if (VEC || k + 4 <= n) return k < n ? sl_load4<VEC>(row + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k < n) v.x = (float)row[k];
    if (k + 1 < n) v.y = (float)row[k + 1];
    if (k + 2 < n) v.z = (float)row[k + 2];
    return v;
}
// the same of data another CTA has just written (L2)
template <bool VEC> __device__ __forceinline__ float4 sl_shared4(const float* row, int k, int n) {
    if (VEC) return k < n ? __ldcg(reinterpret_cast<const float4*>(row + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k < n) v.x = __ldcg(row + k);
    if (k + 1 < n) v.y = __ldcg(row + k + 1);
    if (k + 2 < n) v.z = __ldcg(row + k + 2);
    if (k + 3 < n) v.w = __ldcg(row + k + 3);
    return v;
}
template <bool VEC> __device__ __forceinline__ float4 sl_shared4(const __nv_bfloat16* row, int k, int n) {
    if (VEC) {
        if (k >= n) return make_float4(0.f, 0.f, 0.f, 0.f);
        const uint2 v = __ldcg(reinterpret_cast<const uint2*>(row + k));
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k < n) v.x = __bfloat162float(__ldcg(row + k));
    if (k + 1 < n) v.y = __bfloat162float(__ldcg(row + k + 1));
    if (k + 2 < n) v.z = __bfloat162float(__ldcg(row + k + 2));
    if (k + 3 < n) v.w = __bfloat162float(__ldcg(row + k + 3));
    return v;
}
__device__ __forceinline__ float sl_dot(float4 a, float4 b, float acc) {
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}
template <typename TW> __device__ __forceinline__ float sl_round(float x);
template <> __device__ __forceinline__ float sl_round<float>(float x) { return x; }
template <> __device__ __forceinline__ float sl_round<__nv_bfloat16>(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
template <typename TW> __device__ __forceinline__ float4 sl_round4(float4 v) {
    return make_float4(sl_round<TW>(v.x), sl_round<TW>(v.y), sl_round<TW>(v.z), sl_round<TW>(v.w));
}
__device__ __forceinline__ void sl_store(float* p, float x) { *p = x; }
__device__ __forceinline__ void sl_store(__nv_bfloat16* p, float x) { *p = __float2bfloat16_rn(x); }

// N sums over the warp at once (N a power of two): afterwards v[0] of lane i holds the sum of column i % N
template <int N> __device__ __forceinline__ void sl_warp_sums(float* v, int lane) {
#pragma unroll
    for (int half = N / 2; half >= 1; half /= 2) {
        const bool up = (lane & half) != 0;
#pragma unroll
        for (int c = 0; c < half; ++c) {
            const float send = up ? v[c] : v[c + half], keep = up ? v[c + half] : v[c];
            v[c] = keep + __shfl_xor_sync(0xffffffffu, send, half);
        }
    }
#pragma unroll
    for (int o = N; o < 32; o *= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
}

// What a CTA owns: units, joint units and labels i * G + cta.
struct SlShare { int units, prows, labels; };
__host__ __device__ inline SlShare sl_share(int P, int H, int NV, int G, int cta) {
    return SlShare{(P - cta + G - 1) / G, (H - cta + G - 1) / G, (NV - cta + G - 1) / G};
}
// Shared memory of a CTA in bytes: weights (resident), partial sums, per-utterance state, and in LOCAL mode the exchanged data.
struct SlSmem { size_t w_lstm0, w_lstm1, w_lstm_layer, w_pred,   // layer 0's rows, layer 1's, bytes of a further layer
                        w_out, part, pred, key, ints, h, c, z, total; };
__host__ __device__ inline SlSmem sl_smem(int es, int B, int W, int E, int P, int L, int H, int NV, int G, bool resident, bool local) {
    const SlShare s = sl_share(P, H, NV, G, 0);
    SlSmem m{};
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off = (off + bytes + 15) / 16 * 16; return o; };
    m.w_lstm0 = take(resident ? (size_t)es * s.units * 4 * (E + P) : 0);
    m.w_lstm_layer = resident ? ((size_t)es * s.units * 4 * 2 * P + 15) / 16 * 16 : 0;
    m.w_lstm1 = take(m.w_lstm_layer * (L - 1));
    m.w_pred = take(resident ? (size_t)es * s.prows * P : 0);
    m.w_out = take(resident ? (size_t)es * s.labels * H : 0);
    int most = s.units > s.prows ? s.units : s.prows;
    if (most < SL_WARPS) most = SL_WARPS;
    m.part = take(sizeof(float) * (size_t)most * 4 * SL_UTTS);
    m.pred = take(sizeof(float) * (size_t)s.prows * B);
    m.key = take(sizeof(unsigned long long) * (size_t)B * W);
    m.ints = take(sizeof(int) * 7 * (size_t)B);
    m.h = take(local ? sizeof(float) * 2 * (size_t)L * P : 0);
    m.c = take(local ? sizeof(float) * (size_t)L * P : 0);
    m.z = take(local ? (size_t)es * W * H : 0);
    m.total = off;
    return m;
}

template <typename TW, bool LOCAL, bool VEC>
__global__ void __launch_bounds__(SL_THREADS, 1) simt_loop_kernel(const SimtLoopParams p) {
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ int s_stop, s_n_emit, s_n_alive, s_red[2];
    __shared__ int s_hist[65];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int G = LOCAL ? 1 : gridDim.x, cta = LOCAL ? 0 : blockIdx.x;
    if (p.ctrl->bad_input) return;                 // a length outside [0, T]: nothing is read through it
    const int B = LOCAL ? 1 : p.B;
    const SlShare own = sl_share(p.P, p.H, p.NV, G, cta);
    const SlSmem M = sl_smem((int)sizeof(TW), B, p.W, p.E, p.P, p.L, p.H, p.NV, G, p.resident != 0, LOCAL);
    float* part = reinterpret_cast<float*>(sm + M.part);
    float* s_pred = reinterpret_cast<float*>(sm + M.pred);                     // [utterance][own joint unit]
    unsigned long long* s_key = reinterpret_cast<unsigned long long*>(sm + M.key);
    int* s_t = reinterpret_cast<int*>(sm + M.ints);
    int *s_len = s_t + B, *s_cnt = s_t + 2 * B, *s_pos = s_t + 3 * B, *s_tok = s_t + 4 * B, *s_hp = s_t + 5 * B, *s_list = s_t + 6 * B;
    TW* z = LOCAL ? reinterpret_cast<TW*>(sm + M.z) : static_cast<TW*>(p.z);
    float* h = LOCAL ? reinterpret_cast<float*>(sm + M.h) : p.h;
    float* c = LOCAL ? reinterpret_cast<float*>(sm + M.c) : p.c;
    const TW* emb = static_cast<const TW*>(p.emb);
    const TW* enc_proj = static_cast<const TW*>(p.enc_proj);

    // ---- weights into shared memory ----
    auto copy_row = [&](TW* dst, const TW* src, int n) {                        // one warp, one row
        if (VEC && sizeof(TW) == 4) {
            for (int k = lane * 4; k < n; k += 128) *reinterpret_cast<float4*>(dst + k) = *reinterpret_cast<const float4*>(src + k);
        } else {
            for (int k = lane; k < n; k += 32) dst[k] = src[k];
        }
    };
    if (p.resident) {
        for (int l = 0; l < p.L; ++l) {
            const int nin = l == 0 ? p.E : p.P, K = nin + p.P;
            TW* dst = reinterpret_cast<TW*>(sm + (l == 0 ? M.w_lstm0 : M.w_lstm1 + (size_t)(l - 1) * M.w_lstm_layer));
            for (int i = warp; i < own.units * 4; i += SL_WARPS) {
                const size_t row = (size_t)(i & 3) * p.P + (size_t)(i >> 2) * G + cta;
                copy_row(dst + (size_t)i * K, static_cast<const TW*>(p.w_ih[l]) + row * nin, nin);
                copy_row(dst + (size_t)i * K + nin, static_cast<const TW*>(p.w_hh[l]) + row * p.P, p.P);
            }
        }
        for (int i = warp; i < own.prows; i += SL_WARPS)
            copy_row(reinterpret_cast<TW*>(sm + M.w_pred) + (size_t)i * p.P, static_cast<const TW*>(p.w_pred) + ((size_t)i * G + cta) * p.P, p.P);
        for (int i = warp; i < own.labels; i += SL_WARPS)
            copy_row(reinterpret_cast<TW*>(sm + M.w_out) + (size_t)i * p.H, static_cast<const TW*>(p.w_out) + ((size_t)i * G + cta) * p.H, p.H);
    }
    if (threadIdx.x == 0) s_stop = 0;
    for (int k = threadIdx.x; k < 65; k += SL_THREADS) s_hist[k] = 0;

    // Barrier between phases: the block, or all CTAs.  False when the kernel is being abandoned (bounded wait).
    uint32_t epoch = 0;
    auto phase_sync = [&]() -> bool {
        __syncthreads();
        if (LOCAL) return true;
        if (threadIdx.x == 0) {
            epoch += (uint32_t)(G + p.extra_arrivals);
            __threadfence();
            atomicAdd(&p.ctrl->bar, 1u);
            unsigned long long t0 = 0;
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
    auto fetch = [&](const auto* row, int k, int n) -> float4 {                 // data of this step from another warp or CTA
        if constexpr (LOCAL) return sl_row4<VEC>(row, k, n);
        else return sl_shared4<VEC>(row, k, n);
    };
    auto h_row = [&](int par, int l, int b) { return h + (((size_t)par * p.L + l) * B + b) * p.P; };

    // NB utterances s_list[i0 ..): partial sums of this CTA's hidden units in layer l
    auto update_partials = [&](auto nbc, int l, int i0, int n_here, int KS) {
        constexpr int NB = decltype(nbc)::value;
        const int nin = l == 0 ? p.E : p.P, K = nin + p.P;
        const int c_in = (nin + 127) / 128, chunks = c_in + (p.P + 127) / 128;
        for (int item = warp; item < own.units * KS; item += SL_WARPS) {
            const int ui = item % own.units, ks = item / own.units;
            const TW* wi[4];
            const TW* wh[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const size_t row = (size_t)g * p.P + (size_t)ui * G + cta;
                wi[g] = p.resident ? reinterpret_cast<const TW*>(sm + (l == 0 ? M.w_lstm0 : M.w_lstm1 + (size_t)(l - 1) * M.w_lstm_layer)) + (size_t)(ui * 4 + g) * K : static_cast<const TW*>(p.w_ih[l]) + row * nin;
                wh[g] = p.resident ? wi[g] + nin : static_cast<const TW*>(p.w_hh[l]) + row * p.P;
            }
            float acc[4 * NB];
#pragma unroll
            for (int j = 0; j < 4 * NB; ++j) acc[j] = 0.f;
            const int c0 = chunks * ks / KS, c1 = chunks * (ks + 1) / KS;
#pragma unroll 2
            for (int ch = c0; ch < c1; ++ch) {
                const bool in = ch < c_in;
                const int k = (in ? ch : ch - c_in) * 128 + lane * 4, n = in ? nin : p.P;
                float4 x[NB];
#pragma unroll
                for (int u = 0; u < NB; ++u) {
                    x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (u < n_here) {
                        const int b = s_list[i0 + u];
                        if (in && l == 0) x[u] = sl_row4<VEC>(emb + (size_t)s_tok[b] * p.E, k, n);
                        else x[u] = sl_round4<TW>(fetch(in ? h_row(s_hp[b] ^ 1, l - 1, b) : h_row(s_hp[b], l, b), k, n));
                    }
                }
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const float4 w = sl_row4<VEC>(in ? wi[g] : wh[g], k, n);
#pragma unroll
                    for (int u = 0; u < NB; ++u) acc[g * NB + u] = sl_dot(w, x[u], acc[g * NB + u]);
                }
            }
            sl_warp_sums<4 * NB>(acc, lane);
            if (lane < 4 * NB) part[(size_t)(ks * own.units + ui) * (4 * SL_UTTS) + (lane / NB) * SL_UTTS + lane % NB] = acc[0];
        }
    };
    auto project_partials = [&](auto nbc, int i0, int n_here, int KS) {
        constexpr int NB = decltype(nbc)::value;
        const int chunks = (p.P + 127) / 128;
        for (int item = warp; item < own.prows * KS; item += SL_WARPS) {
            const int pi = item % own.prows, ks = item / own.prows;
            const TW* w = p.resident ? reinterpret_cast<const TW*>(sm + M.w_pred) + (size_t)pi * p.P : static_cast<const TW*>(p.w_pred) + ((size_t)pi * G + cta) * p.P;
            float acc[NB];
#pragma unroll
            for (int u = 0; u < NB; ++u) acc[u] = 0.f;
#pragma unroll 2
            for (int ch = chunks * ks / KS; ch < chunks * (ks + 1) / KS; ++ch) {
                const int k = ch * 128 + lane * 4;
                const float4 wv = sl_row4<VEC>(w, k, p.P);
#pragma unroll
                for (int u = 0; u < NB; ++u)
                    if (u < n_here) {
                        const int b = s_list[i0 + u];
                        acc[u] = sl_dot(wv, sl_round4<TW>(fetch(h_row(s_hp[b] ^ 1, p.L - 1, b), k, p.P)), acc[u]);
                    }
            }
            sl_warp_sums<NB>(acc, lane);
            if (lane < NB) part[(size_t)(ks * own.prows + pi) * SL_UTTS + lane] = acc[0];
        }
    };

    // LOCAL: this CTA's utterances one after the other; grid: all utterances in one pass
    for (int u0 = LOCAL ? (int)blockIdx.x : 0; u0 < (LOCAL ? p.B : 1); u0 += LOCAL ? (int)gridDim.x : 1) {
        // ---- start of sequence ----
        __syncthreads();
        for (int b = threadIdx.x; b < B; b += SL_THREADS) {
            s_t[b] = 0;
            s_len[b] = min(max(p.enc_len[u0 + b], 0), p.T);
            s_cnt[b] = 0; s_pos[b] = 0; s_hp[b] = 0;
            s_tok[b] = s_len[b] > 0 ? p.blank : -1;
        }
        if (LOCAL) {
            for (int i = threadIdx.x; i < 2 * p.L * p.P; i += SL_THREADS) h[i] = 0.f;
            for (int i = threadIdx.x; i < p.L * p.P; i += SL_THREADS) c[i] = 0.f;
        }
        for (int i = threadIdx.x; i < B * p.W; i += SL_THREADS) s_key[i] = 0ull;
        __syncthreads();
        long long n_rows = 0, n_tok = 0, n_forced = 0;          // thread-local counts of the recording CTA
        int steps = 0;
        for (int step = -1;; ++step) {
            // =============================================================================
            // control: decisions for every utterance, in every CTA; lists of emitting and of live utterances
            // =============================================================================
            if (step >= 0) {
                const unsigned long long* keys = LOCAL ? s_key : p.keys + (size_t)(step & 1) * B * p.W;
                for (int b = threadIdx.x; b < B; b += SL_THREADS) {
                    int t = s_t[b], tok = -1;
                    const int len = s_len[b];
                    if (t < len) {
                        const int n = min(p.W, len - t);
                        int first = -1, label = p.blank;
                        bool bad = false;
                        for (int w0 = 0; w0 < n && first < 0; w0 += 4) {
                            unsigned long long kk[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                kk[j] = 0ull;
                                if (w0 + j < n) {
                                    const unsigned long long* kp = keys + (size_t)b * p.W + w0 + j;
                                    if constexpr (LOCAL) kk[j] = *kp;
                                    else kk[j] = __ldcg(kp);
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
                        if (LOCAL || blockIdx.x == 0) {                           // recorded once
                            if (tok >= 0) {
                                p.out_tokens[(size_t)(u0 + b) * p.max_out + pos] = label;
                                p.out_frames[(size_t)(u0 + b) * p.max_out + pos] = t_emit;
                                p.out_len[u0 + b] = pos + 1;
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
            // emitting utterances to the front of the list, in order (a warp scans; batches are small)
            if (warp == 0) {
                int ne = 0, na = 0;
                for (int b0 = 0; b0 < B; b0 += 32) {
                    const int b = b0 + lane;
                    const bool live = b < B && s_t[b] < s_len[b], em = live && s_tok[b] >= 0;   // a finished utterance needs no further state
                    const uint32_t m = __ballot_sync(0xffffffffu, em);
                    if (em) s_list[ne + __popc(m & ((1u << lane) - 1u))] = b;
                    ne += __popc(m);
                    na += __popc(__ballot_sync(0xffffffffu, live));
                }
                if (lane == 0) { s_n_emit = ne; s_n_alive = na; }
            }
            __syncthreads();
            const int n_emit = s_n_emit;
            if (s_n_alive == 0) break;
            if (steps >= p.step_cap) { if (threadIdx.x == 0 && (LOCAL || blockIdx.x == 0)) set_status(p.ctrl, WIND_ERR_INTERNAL); break; }
            // =============================================================================
            // update and projection of the emitting utterances
            // =============================================================================
            if (n_emit > 0) {
                for (int l = 0; l < p.L; ++l) {
                    const int KS = own.units > 0 && own.units < SL_WARPS ? SL_WARPS / own.units : 1;
                    for (int i0 = 0; i0 < n_emit; i0 += SL_UTTS) {
                        const int n_here = min(SL_UTTS, n_emit - i0);
                        if (LOCAL || n_here == 1) update_partials(std::integral_constant<int, 1>{}, l, i0, n_here, KS);
                        else update_partials(std::integral_constant<int, SL_UTTS>{}, l, i0, n_here, KS);
                        __syncthreads();
                        for (int i = threadIdx.x; i < own.units * n_here; i += SL_THREADS) {
                            const int ui = i / n_here, u = i - ui * n_here, b = s_list[i0 + u], j = ui * G + cta;
                            float a[4];
#pragma unroll
                            for (int g = 0; g < 4; ++g) {
                                float s = 0.f;
                                for (int ks = 0; ks < KS; ++ks) s += part[(size_t)(ks * own.units + ui) * (4 * SL_UTTS) + g * SL_UTTS + u];
                                a[g] = s + (p.b_ih[l][g * p.P + j] + p.b_hh[l][g * p.P + j]);
                            }
                            const float gi = 1.f / (1.f + expf(-a[0])), gf = 1.f / (1.f + expf(-a[1])), gg = tanhf(a[2]), go = 1.f / (1.f + expf(-a[3]));
                            float* cs = c + ((size_t)l * B + b) * p.P + j;
                            const float cc = gf * *cs + gi * gg;
                            *cs = cc;
                            h_row(s_hp[b] ^ 1, l, b)[j] = go * tanhf(cc);
                        }
                        if (i0 + SL_UTTS < n_emit) __syncthreads();
                    }
                    if (!phase_sync()) goto done;
                }
                const int KS = own.prows > 0 && own.prows < SL_WARPS ? SL_WARPS / own.prows : 1;
                for (int i0 = 0; i0 < n_emit; i0 += SL_UTTS) {
                    const int n_here = min(SL_UTTS, n_emit - i0);
                    if (LOCAL || n_here == 1) project_partials(std::integral_constant<int, 1>{}, i0, n_here, KS);
                    else project_partials(std::integral_constant<int, SL_UTTS>{}, i0, n_here, KS);
                    __syncthreads();
                    for (int i = threadIdx.x; i < own.prows * n_here; i += SL_THREADS) {
                        const int pi = i / n_here, u = i - pi * n_here;
                        float s = 0.f;
                        for (int ks = 0; ks < KS; ++ks) s += part[(size_t)(ks * own.prows + pi) * SL_UTTS + u];
                        s_pred[(size_t)s_list[i0 + u] * own.prows + pi] = s + p.b_pred[pi * G + cta];
                    }
                    __syncthreads();
                }
                for (int i = threadIdx.x; i < n_emit; i += SL_THREADS) s_hp[s_list[i]] ^= 1;
            }
            // z of every live utterance's window, for this CTA's joint units; the live utterances become the list
            __syncthreads();
            if (warp == 0) {
                int na = 0;
                for (int b0 = 0; b0 < B; b0 += 32) {
                    const int b = b0 + lane;
                    const bool live = b < B && s_t[b] < s_len[b];
                    const uint32_t m = __ballot_sync(0xffffffffu, live);
                    if (live) s_list[na + __popc(m & ((1u << lane) - 1u))] = b;
                    na += __popc(m);
                }
            }
            __syncthreads();
            const int n_alive = s_n_alive;
            unsigned long long* knext = LOCAL ? s_key : p.keys + (size_t)((step + 1) & 1) * B * p.W;
            for (int i = threadIdx.x; i < n_alive * p.W * own.prows; i += SL_THREADS) {
                const int pi = i % own.prows, r = i / own.prows, b = s_list[r / p.W], w = r % p.W;
                if (s_t[b] + w < s_len[b]) {
                    const int o = pi * G + cta;
                    float v = (float)enc_proj[((size_t)(u0 + b) * p.T + s_t[b] + w) * p.H + o] + s_pred[(size_t)b * own.prows + pi];
                    v = p.act == WIND_ACT_RELU ? fmaxf(v, 0.f) : tanhf(v);
                    sl_store(z + ((size_t)b * p.W + w) * p.H + o, v);
                }
            }
            for (int i = threadIdx.x; i < B * p.W; i += SL_THREADS) s_key[i] = 0ull;
            // (the other parity's keys were read by every CTA before the last barrier of the step before)
            if (!LOCAL && blockIdx.x == 0)
                for (int i = threadIdx.x; i < B * p.W; i += SL_THREADS) knext[i] = 0ull;
            if (!phase_sync()) goto done;
            // =============================================================================
            // joint: items of SL_ROWS window rows x SL_LABELS of this CTA's labels
            // =============================================================================
            {
                const int rows = n_alive * p.W, rgs = (rows + SL_ROWS - 1) / SL_ROWS, lgs = (own.labels + SL_LABELS - 1) / SL_LABELS;
                for (int item = warp; item < rgs * lgs; item += SL_WARPS) {
                    const int rg = item / lgs, lg = item - rg * lgs;
                    const TW* zr[SL_ROWS];
                    int slot[SL_ROWS];
#pragma unroll
                    for (int i = 0; i < SL_ROWS; ++i) {
                        const int row = min(rg * SL_ROWS + i, rows - 1), b = s_list[row / p.W], w = row % p.W;
                        slot[i] = rg * SL_ROWS + i < rows && s_t[b] + w < s_len[b] ? b * p.W + w : -1;
                        zr[i] = z + (size_t)(slot[i] < 0 ? b * p.W : slot[i]) * p.H;
                    }
                    const TW* wr[SL_LABELS];
#pragma unroll
                    for (int j = 0; j < SL_LABELS; ++j) {
                        const int li = min(lg * SL_LABELS + j, own.labels - 1);
                        wr[j] = p.resident ? reinterpret_cast<const TW*>(sm + M.w_out) + (size_t)li * p.H : static_cast<const TW*>(p.w_out) + ((size_t)li * G + cta) * p.H;
                    }
                    float acc[SL_ROWS * SL_LABELS];
#pragma unroll
                    for (int i = 0; i < SL_ROWS * SL_LABELS; ++i) acc[i] = 0.f;
#pragma unroll 2
                    for (int k = lane * 4; k < p.H + lane * 4; k += 128) {
                        float4 x[SL_ROWS];
#pragma unroll
                        for (int i = 0; i < SL_ROWS; ++i) x[i] = fetch(zr[i], k, p.H);
#pragma unroll
                        for (int j = 0; j < SL_LABELS; ++j) {
                            const float4 w = sl_row4<VEC>(wr[j], k, p.H);
#pragma unroll
                            for (int i = 0; i < SL_ROWS; ++i) acc[j * SL_ROWS + i] = sl_dot(w, x[i], acc[j * SL_ROWS + i]);
                        }
                    }
                    sl_warp_sums<SL_ROWS * SL_LABELS>(acc, lane);
                    // lane = (label j, row i); the best of the item's labels for each row
                    const int j = (lane >> 2) & 3, li = lg * SL_LABELS + j;
                    unsigned long long key = 0ull;
                    if (lane < 16 && li < own.labels) {
                        const int v = li * G + cta;
                        const float s = acc[0] + p.b_out[v];
                        if (s > -INFINITY) key = pack_key(s, (uint32_t)v);
                    }
                    key = max(key, __shfl_xor_sync(0xffffffffu, key, 4));
                    key = max(key, __shfl_xor_sync(0xffffffffu, key, 8));
                    int sl = -1;
#pragma unroll
                    for (int i = 0; i < SL_ROWS; ++i) sl = (lane & 3) == i ? slot[i] : sl;
                    if (lane < SL_ROWS && sl >= 0 && key != 0ull) atomicMax(&s_key[sl], key);
                }
                __syncthreads();
                if (!LOCAL)
                    for (int i = threadIdx.x; i < B * p.W; i += SL_THREADS)
                        if (s_key[i] != 0ull) atomicMax(&knext[i], s_key[i]);
            }
            if (!phase_sync()) goto done;
        }
        // ---- counters ----
        if (LOCAL || blockIdx.x == 0) {
            if (threadIdx.x == 0) atomicMax(&p.ctrl->step, steps);
            if (n_rows) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->joint_rows), (unsigned long long)n_rows);
            if (n_tok) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->tokens), (unsigned long long)n_tok);
            if (n_forced) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->forced), (unsigned long long)n_forced);
        }
    }
done:
    __syncthreads();
    if (LOCAL || blockIdx.x == 0)
        for (int k = threadIdx.x; k < 65; k += SL_THREADS)
            if (s_hist[k]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->jump_hist[k]), (unsigned long long)s_hist[k]);
    if (threadIdx.x == 0) {
        if (s_stop) set_status(p.ctrl, WIND_ERR_TIMEOUT);
        if (blockIdx.x == 0) p.ctrl->active = 0;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
template <typename TW, bool LOCAL>
static const void* sl_fn(bool vec) {
    return vec ? (const void*)simt_loop_kernel<TW, LOCAL, true> : (const void*)simt_loop_kernel<TW, LOCAL, false>;
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
        const int dyn = n - 1024;      // the kernels' static shared memory stays below 1 KB
        for (bool vec : {false, true})
            for (const void* fn : {sl_fn<float, true>(vec), sl_fn<float, false>(vec), sl_fn<__nv_bfloat16, true>(vec), sl_fn<__nv_bfloat16, false>(vec)})
                if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn)) != cudaSuccess) return e;
        g_sl_optin[dev] = n;
    }
    *optin = g_sl_optin[dev];
    return cudaSuccess;
}

// Which form of the kernel a decode takes; false: none (window-based decoding, batches whose state does not fit)
static bool sl_plan(const Call& c, bool* local, bool* resident, size_t* smem, int* grid) {
    if (c.mode != WIND_MODE_FIRST_NONBLANK || c.B > SL_MAX_B) return false;
    int optin = 0, sms = 0;
    if (sl_device(&optin) != cudaSuccess || loop_sm_count(&sms) != cudaSuccess) { cudaGetLastError(); return false; }
    const wind_model_t& m = c.m;
    const int es = m.dtype == WIND_DT_BF16 ? 2 : 4;
    const size_t budget = (size_t)optin - 1024;
    SlSmem s = sl_smem(es, 1, c.W, m.E, m.P, m.L, m.H, m.V + 1, 1, true, true);
    if (s.total <= budget) {
        *local = *resident = true;
        *smem = s.total;
        *grid = c.B < sms ? c.B : sms;
        return true;
    }
    *local = false;
    *grid = sms;
    s = sl_smem(es, c.B, c.W, m.E, m.P, m.L, m.H, m.V + 1, sms, true, false);
    *resident = s.total <= budget;
    if (!*resident) s = sl_smem(es, c.B, c.W, m.E, m.P, m.L, m.H, m.V + 1, sms, false, false);
    *smem = s.total;
    return s.total <= budget;
}

bool simt_loop_supported(const Call& c) {
    bool local, resident;
    size_t smem;
    int grid;
    return sl_plan(c, &local, &resident, &smem, &grid);
}

cudaError_t simt_loop(const Call& c) {
    bool local, resident;
    size_t smem;
    int grid;
    if (!sl_plan(c, &local, &resident, &smem, &grid)) return cudaErrorNotSupported;
    const wind_model_t& m = c.m;
    SimtLoopParams p{};
    p.ctrl = c.ctrl();
    p.B = c.B; p.T = c.T; p.W = c.W; p.S = c.S; p.max_out = c.max_out;
    p.E = m.E; p.P = m.P; p.L = m.L; p.H = m.H; p.NV = m.V + 1; p.blank = m.blank_id; p.act = m.act;
    const long long cap = (long long)c.T * (c.S + 1) + 2;
    p.step_cap = cap > 0x7fffffff ? 0x7fffffff : (int)cap;
    p.resident = resident;
    p.extra_arrivals = loop_extra_arrivals();
    p.emb = m.emb; p.w_pred = m.w_pred; p.b_pred = m.b_pred; p.w_out = m.w_out; p.b_out = m.b_out;
    // four operands at a time where every row starts on a boundary of four
    const uintptr_t mask = m.dtype == WIND_DT_BF16 ? 7 : 15;
    bool vec = m.E % 4 == 0 && m.P % 4 == 0 && m.H % 4 == 0;
    auto aligned = [&](const void* q) { return (reinterpret_cast<uintptr_t>(q) & mask) == 0; };
    vec = vec && aligned(m.emb) && aligned(m.w_pred) && aligned(m.w_out);
    for (int l = 0; l < m.L; ++l) {
        p.w_ih[l] = c.w_ih[l]; p.w_hh[l] = c.w_hh[l]; p.b_ih[l] = c.b_ih[l]; p.b_hh[l] = c.b_hh[l];
        vec = vec && aligned(c.w_ih[l]) && aligned(c.w_hh[l]);
    }
    p.enc_proj = c.enc_proj(); p.enc_len = c.enc_len;
    p.h = c.h(0); p.c = c.c(); p.z = m.dtype == WIND_DT_BF16 ? (void*)c.z() : (void*)c.zf(); p.keys = c.keys();
    p.out_tokens = c.out_tokens; p.out_frames = c.out_frames; p.out_len = c.out_len;
    const void* fn = m.dtype == WIND_DT_BF16 ? (local ? sl_fn<__nv_bfloat16, true>(vec) : sl_fn<__nv_bfloat16, false>(vec))
                                             : (local ? sl_fn<float, true>(vec) : sl_fn<float, false>(vec));
    void* args[1] = {(void*)&p};
    if (local) return cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(SL_THREADS), args, smem, c.stream);
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)grid), dim3(SL_THREADS), args, smem, c.stream);
}

}  // namespace wind
