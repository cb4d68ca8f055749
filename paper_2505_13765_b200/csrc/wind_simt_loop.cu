// The decoding loop of the plain-ALU path (fp32 models, and bf16 models outside the tensor-core set) as one persistent kernel.
//
// As separate kernels in a CUDA graph a lock step cost 20 us for a model of 64 units (launches) and 300 us for one of 640
// units in fp32 (every weight read again by kernels with one block per output).  Here the weights stay in shared memory:
//   one SM  the whole decoder fits one SM (64 units in fp32: 155 KB): a CTA decodes its utterances one after the other and
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
    float* h;                      // [2][L][B][P], a parity per utterance
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
// Shared memory of a CTA in bytes: weights (resident), partial sums, per-utterance state, biases.
struct SlSmem { size_t w_lstm0, w_lstm1, w_lstm_layer, w_pred,   // layer 0's rows, layer 1's, bytes of a further layer
                        w_out, part, pred, key, ints, b_gate, b_pred, b_out, total; };
__host__ __device__ inline SlSmem sl_smem(int es, int B, int W, int E, int P, int L, int H, int NV, int G, bool resident) {
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
    m.b_gate = take(sizeof(float) * (size_t)L * s.units * 4);
    m.b_pred = take(sizeof(float) * (size_t)s.prows);
    m.b_out = take(sizeof(float) * (size_t)s.labels);
    m.total = off;
    return m;
}

template <typename TW, bool VEC>
__global__ void __launch_bounds__(SL_THREADS, 1) simt_grid_kernel(const SimtLoopParams p) {
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ int s_stop, s_n_emit, s_n_alive;
    __shared__ int s_hist[65];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int G = gridDim.x, cta = blockIdx.x;
    if (p.ctrl->bad_input) return;                 // a length outside [0, T]: nothing is read through it
    const int B = p.B;
    const SlShare own = sl_share(p.P, p.H, p.NV, G, cta);
    const SlSmem M = sl_smem((int)sizeof(TW), B, p.W, p.E, p.P, p.L, p.H, p.NV, G, p.resident != 0);
    float* part = reinterpret_cast<float*>(sm + M.part);
    float* s_pred = reinterpret_cast<float*>(sm + M.pred);                     // [utterance][own joint unit]
    unsigned long long* s_key = reinterpret_cast<unsigned long long*>(sm + M.key);
    int* s_t = reinterpret_cast<int*>(sm + M.ints);
    int *s_len = s_t + B, *s_cnt = s_t + 2 * B, *s_pos = s_t + 3 * B, *s_tok = s_t + 4 * B, *s_hp = s_t + 5 * B, *s_list = s_t + 6 * B;
    TW* z = static_cast<TW*>(p.z);
    float *h = p.h, *c = p.c;
    float* s_bg = reinterpret_cast<float*>(sm + M.b_gate);                     // [layer][own unit][gate] b_ih + b_hh
    float* s_bp = reinterpret_cast<float*>(sm + M.b_pred);
    float* s_bo = reinterpret_cast<float*>(sm + M.b_out);
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
    for (int i = threadIdx.x; i < p.L * own.units * 4; i += SL_THREADS) {
        const int l = i / (own.units * 4), j = (i / 4) % own.units, g = i & 3;
        s_bg[i] = p.b_ih[l][g * p.P + j * G + cta] + p.b_hh[l][g * p.P + j * G + cta];
    }
    for (int i = threadIdx.x; i < own.prows; i += SL_THREADS) s_bp[i] = p.b_pred[i * G + cta];
    for (int i = threadIdx.x; i < own.labels; i += SL_THREADS) s_bo[i] = p.b_out[i * G + cta];
    if (threadIdx.x == 0) s_stop = 0;
    for (int k = threadIdx.x; k < 65; k += SL_THREADS) s_hist[k] = 0;

    // Barrier of all CTAs between phases.  False when the kernel is being abandoned (bounded wait).
    uint32_t epoch = 0;
    auto phase_sync = [&]() -> bool {
        __syncthreads();
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
    auto fetch = [&](const auto* row, int k, int n) -> float4 { return sl_shared4<VEC>(row, k, n); };   // data of this step from another CTA
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

    {
        // ---- start of sequence ----
        __syncthreads();
        for (int b = threadIdx.x; b < B; b += SL_THREADS) {
            s_t[b] = 0;
            s_len[b] = min(max(p.enc_len[b], 0), p.T);
            s_cnt[b] = 0; s_pos[b] = 0; s_hp[b] = 0;
            s_tok[b] = s_len[b] > 0 ? p.blank : -1;
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
                const unsigned long long* keys = p.keys + (size_t)(step & 1) * B * p.W;
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
            if (steps >= p.step_cap) { if (threadIdx.x == 0 && blockIdx.x == 0) set_status(p.ctrl, WIND_ERR_INTERNAL); break; }
            // =============================================================================
            // update and projection of the emitting utterances
            // =============================================================================
            if (n_emit > 0) {
                for (int l = 0; l < p.L; ++l) {
                    const int KS = own.units > 0 && own.units < SL_WARPS ? SL_WARPS / own.units : 1;
                    for (int i0 = 0; i0 < n_emit; i0 += SL_UTTS) {
                        const int n_here = min(SL_UTTS, n_emit - i0);
                        if (n_here == 1) update_partials(std::integral_constant<int, 1>{}, l, i0, n_here, KS);
                        else update_partials(std::integral_constant<int, SL_UTTS>{}, l, i0, n_here, KS);
                        __syncthreads();
                        for (int i = threadIdx.x; i < own.units * n_here; i += SL_THREADS) {
                            const int ui = i / n_here, u = i - ui * n_here, b = s_list[i0 + u], j = ui * G + cta;
                            float a[4];
#pragma unroll
                            for (int g = 0; g < 4; ++g) {
                                float s = 0.f;
                                for (int ks = 0; ks < KS; ++ks) s += part[(size_t)(ks * own.units + ui) * (4 * SL_UTTS) + g * SL_UTTS + u];
                                a[g] = s + s_bg[(l * own.units + ui) * 4 + g];
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
                    if (n_here == 1) project_partials(std::integral_constant<int, 1>{}, i0, n_here, KS);
                    else project_partials(std::integral_constant<int, SL_UTTS>{}, i0, n_here, KS);
                    __syncthreads();
                    for (int i = threadIdx.x; i < own.prows * n_here; i += SL_THREADS) {
                        const int pi = i / n_here, u = i - pi * n_here;
                        float s = 0.f;
                        for (int ks = 0; ks < KS; ++ks) s += part[(size_t)(ks * own.prows + pi) * SL_UTTS + u];
                        s_pred[(size_t)s_list[i0 + u] * own.prows + pi] = s + s_bp[pi];
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
            unsigned long long* knext = p.keys + (size_t)((step + 1) & 1) * B * p.W;
            for (int i = threadIdx.x; i < n_alive * p.W * own.prows; i += SL_THREADS) {
                const int pi = i % own.prows, r = i / own.prows, b = s_list[r / p.W], w = r % p.W;
                if (s_t[b] + w < s_len[b]) {
                    const int o = pi * G + cta;
                    float v = (float)enc_proj[((size_t)b * p.T + s_t[b] + w) * p.H + o] + s_pred[(size_t)b * own.prows + pi];
                    v = p.act == WIND_ACT_RELU ? fmaxf(v, 0.f) : tanhf(v);
                    sl_store(z + ((size_t)b * p.W + w) * p.H + o, v);
                }
            }
            for (int i = threadIdx.x; i < B * p.W; i += SL_THREADS) s_key[i] = 0ull;
            // (the other parity's keys were read by every CTA before the last barrier of the step before)
            if (blockIdx.x == 0)
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
                        const float s = acc[0] + s_bo[li];
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
                for (int i = threadIdx.x; i < B * p.W; i += SL_THREADS)
                    if (s_key[i] != 0ull) atomicMax(&knext[i], s_key[i]);
            }
            if (!phase_sync()) goto done;
        }
        // ---- counters ----
        if (blockIdx.x == 0) {
            if (threadIdx.x == 0) atomicMax(&p.ctrl->step, steps);
            if (n_rows) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->joint_rows), (unsigned long long)n_rows);
            if (n_tok) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->tokens), (unsigned long long)n_tok);
            if (n_forced) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->forced), (unsigned long long)n_forced);
        }
    }
done:
    __syncthreads();
    if (blockIdx.x == 0)
        for (int k = threadIdx.x; k < 65; k += SL_THREADS)
            if (s_hist[k]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->jump_hist[k]), (unsigned long long)s_hist[k]);
    if (threadIdx.x == 0) {
        if (s_stop) set_status(p.ctrl, WIND_ERR_TIMEOUT);
        if (blockIdx.x == 0) p.ctrl->active = 0;
    }
}

// ---------------------------------------------------------------------------
// The whole decoder inside one SM: a CTA decodes its utterances one after the other.  Everything is fp32 in shared memory
// (bf16 operands converted once), rows padded with zeros to a multiple of four and behind that by four floats per thread of
// a row, so that the 16-byte reads of neighbouring threads fall into different banks.  A row's dot product is cut over up to
// eight neighbouring threads.  A step of the 64-unit fp32 model is bound by reading its 128 KB of gate weights (1000 cycles)
// and by seven block barriers; in the grid form's code with one CTA it took 17000 cycles (8.6 us), 86 KB of instructions
// against an instruction cache of 32 KB: 427 us for an utterance of 44 steps, here 234 us.
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
    m.lg_l = sl_lg_tpr(4 * P); m.lg_p = sl_lg_tpr(H); m.lg_j = sl_lg_tpr(NV);
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

template <typename TW>
__global__ void __launch_bounds__(SL_THREADS, 1) simt_local_kernel(const SimtLoopParams p, const int emb_here) {
    extern __shared__ __align__(16) float sf[];
    __shared__ int s_tok, s_t, s_more;
    __shared__ int s_hist[65];
    if (p.ctrl->bad_input) return;                 // a length outside [0, T]: nothing is read through it
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const SlLocal M = sl_local(p.W, p.E, p.P, p.L, p.H, p.NV, emb_here != 0);
    // a matrix [rows][n] to column `at` of the padded rows at dst, with zeros up to the next multiple of four; a warp takes a row
    auto load_rows = [&](float* dst, int ld, int at, const void* src_, int rows, int n) {
        const TW* src = static_cast<const TW*>(src_);
        const int n4 = (n + 3) & ~3;
#pragma unroll 4
        for (int row = warp; row < rows; row += SL_WARPS)
            for (int k = lane; k < n4; k += 32) dst[row * ld + at + k] = k < n ? (float)src[(size_t)row * n + k] : 0.f;
    };
    for (int l = 0; l < p.L; ++l) {
        float* dst = sf + (l == 0 ? M.w_l0 : M.w_l1 + (l - 1) * M.w_l_layer);
        const int ld = l == 0 ? M.ld_l0 : M.ld_l1, nin = l == 0 ? p.E : p.P;
        load_rows(dst, ld, 0, p.w_ih[l], 4 * p.P, nin);
        load_rows(dst, ld, l == 0 ? M.nin0 : M.np, p.w_hh[l], 4 * p.P, p.P);
        for (int i = tid; i < 4 * p.P; i += SL_THREADS) sf[M.b_gate + l * 4 * p.P + i] = p.b_ih[l][i] + p.b_hh[l][i];
    }
    load_rows(sf + M.w_pred, M.ld_p, 0, p.w_pred, p.H, p.P);
    load_rows(sf + M.w_out, M.ld_o, 0, p.w_out, p.NV, p.H);
    if (emb_here) load_rows(sf + M.emb, M.nin0, 0, p.emb, p.NV, p.E);
    for (int i = tid; i < p.H; i += SL_THREADS) sf[M.b_pred + i] = p.b_pred[i];
    for (int i = tid; i < p.NV; i += SL_THREADS) sf[M.b_out + i] = p.b_out[i];
    for (int i = tid; i < 65; i += SL_THREADS) s_hist[i] = 0;
    unsigned long long* s_key = reinterpret_cast<unsigned long long*>(sf + M.key);

    // the share `part` of a dot product of two padded rows of n4 floats
    auto dot = [&](const float* w, const float* x, int n4, int part, int lg, float acc) -> float {
        float a1 = 0.f;
#pragma unroll 4
        for (int k = 4 * part; k < n4; k += 4 << lg) {
            const float4 a = *reinterpret_cast<const float4*>(w + k), b = *reinterpret_cast<const float4*>(x + k);
            acc = fmaf(a.y, b.y, fmaf(a.x, b.x, acc));
            a1 = fmaf(a.w, b.w, fmaf(a.z, b.z, a1));
        }
        return acc + a1;
    };
    auto share_sum = [&](float v, int lg) {
        for (int o = 1; o < 1 << lg; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
    const TW* enc_proj = static_cast<const TW*>(p.enc_proj);
    long long n_rows = 0, n_tok = 0, n_forced = 0;             // counts (the same in all lanes of warp 0)
    int most_steps = 0;

    for (int utt = blockIdx.x; utt < p.B; utt += gridDim.x) {
        const int len = min(max(p.enc_len[utt], 0), p.T);
        int cnt = 0, pos = 0, steps = 0, t = 0;                // the utterance's state (warp 0)
        __syncthreads();
        for (int i = tid; i < p.L * M.np; i += SL_THREADS) sf[M.h + i] = 0.f;
        for (int i = tid; i < p.L * p.P; i += SL_THREADS) sf[M.c + i] = 0.f;
        for (int i = tid; i < p.W; i += SL_THREADS) s_key[i] = 0ull;
        if (tid == 0) { s_tok = p.blank; s_t = 0; s_more = len > 0; }
        __syncthreads();
        while (s_more) {
            const int tok = s_tok, n = min(p.W, len - s_t);
            const size_t row0 = (size_t)utt * p.T + s_t;
            // this thread's first element of the window's enc_proj rows, requested before the decoder phases
            const float z_enc = tid < n * p.H ? (float)enc_proj[row0 * p.H + tid] : 0.f;
            if (tok >= 0) {
                const float* x = sf + M.emb + tok * M.nin0;
                if (!emb_here) {
                    for (int k = tid; k < M.nin0; k += SL_THREADS) sf[M.x + k] = k < p.E ? (float)static_cast<const TW*>(p.emb)[(size_t)tok * p.E + k] : 0.f;
                    x = sf + M.x;
                    __syncthreads();
                }
                for (int l = 0; l < p.L; ++l) {
                    const float* w = sf + (l == 0 ? M.w_l0 : M.w_l1 + (l - 1) * M.w_l_layer);
                    const int ld = l == 0 ? M.ld_l0 : M.ld_l1, n_in = l == 0 ? M.nin0 : M.np, part = tid & ((1 << M.lg_l) - 1);
                    const float* xl = l == 0 ? x : sf + M.h + (l - 1) * M.np;
#pragma unroll 1
                    for (int i = tid; i - lane < 4 * p.P << M.lg_l; i += SL_THREADS) {       // whole warps: threads past the end repeat the last row
                        const int row = min(i >> M.lg_l, 4 * p.P - 1);
                        const float* wr = w + row * ld;
                        float v = dot(wr, xl, n_in, part, M.lg_l, 0.f);
                        v = dot(wr + n_in, sf + M.h + l * M.np, M.np, part, M.lg_l, v);
                        v = share_sum(v, M.lg_l);
                        if (part == 0) sf[M.gates + row] = v + sf[M.b_gate + l * 4 * p.P + row];
                    }
                    __syncthreads();
                    for (int j = tid; j < p.P; j += SL_THREADS) {
                        const float* gt = sf + M.gates + j;
                        const float gi = 1.f / (1.f + expf(-gt[0])), gf = 1.f / (1.f + expf(-gt[p.P])), gg = tanhf(gt[2 * p.P]), go = 1.f / (1.f + expf(-gt[3 * p.P]));
                        float* cs = sf + M.c + l * p.P + j;
                        const float cc = gf * *cs + gi * gg;
                        *cs = cc;
                        sf[M.h + l * M.np + j] = sl_round<TW>(go * tanhf(cc));
                    }
                    __syncthreads();
                }
                const int part = tid & ((1 << M.lg_p) - 1);
#pragma unroll 1
                for (int i = tid; i - lane < p.H << M.lg_p; i += SL_THREADS) {
                    const int row = min(i >> M.lg_p, p.H - 1);
                    const float v = share_sum(dot(sf + M.w_pred + row * M.ld_p, sf + M.h + (p.L - 1) * M.np, M.np, part, M.lg_p, 0.f), M.lg_p);
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
                    const float s = share_sum(dot(sf + M.w_out + v * M.ld_o, sf + M.z + w * M.nh, M.nh, part, M.lg_j, 0.f), M.lg_j) + sf[M.b_out + v];
                    unsigned long long key = s > -INFINITY ? pack_key(s, (uint32_t)v) : 0ull;
                    if (__all_sync(0xffffffffu, w == __shfl_sync(0xffffffffu, w, 0))) {       // one row's outputs: one update for the warp
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
                        if (lane != 0) key = 0ull;
                    } else if (part != 0) {
                        key = 0ull;
                    }
                    if (key != 0ull) atomicMax(&s_key[w], key);
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
        if (blockIdx.x == 0) p.ctrl->active = 0;
    }
    for (int k = tid; k < 65; k += SL_THREADS)
        if (s_hist[k]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->jump_hist[k]), (unsigned long long)s_hist[k]);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
template <typename TW>
static const void* sl_fn(bool vec) {
    return vec ? (const void*)simt_grid_kernel<TW, true> : (const void*)simt_grid_kernel<TW, false>;
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
        for (const void* fn : {sl_fn<float>(false), sl_fn<float>(true), sl_fn<__nv_bfloat16>(false), sl_fn<__nv_bfloat16>(true),
                               (const void*)simt_local_kernel<float>, (const void*)simt_local_kernel<__nv_bfloat16>})
            if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn)) != cudaSuccess) return e;
        g_sl_optin[dev] = n;
    }
    *optin = g_sl_optin[dev];
    return cudaSuccess;
}

// Which form of the kernel a decode takes; false: none (window-based decoding, batches whose state does not fit)
static bool sl_plan(const Call& c, bool* local, bool* resident, bool* emb, size_t* smem, int* grid) {
    if (c.mode != WIND_MODE_FIRST_NONBLANK || c.B > SL_MAX_B) return false;
    int optin = 0, sms = 0;
    if (sl_device(&optin) != cudaSuccess || loop_sm_count(&sms) != cudaSuccess) { cudaGetLastError(); return false; }
    const wind_model_t& m = c.m;
    const int es = m.dtype == WIND_DT_BF16 ? 2 : 4;
    const size_t budget = (size_t)optin - 1024;
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
    SlSmem s = sl_smem(es, c.B, c.W, m.E, m.P, m.L, m.H, m.V + 1, sms, true);
    *resident = s.total <= budget;
    if (!*resident) s = sl_smem(es, c.B, c.W, m.E, m.P, m.L, m.H, m.V + 1, sms, false);
    *smem = s.total;
    return s.total <= budget;
}

bool simt_loop_supported(const Call& c) {
    bool local, resident, emb;
    size_t smem;
    int grid;
    return sl_plan(c, &local, &resident, &emb, &smem, &grid);
}

cudaError_t simt_loop(const Call& c) {
    bool local, resident, emb;
    size_t smem;
    int grid;
    if (!sl_plan(c, &local, &resident, &emb, &smem, &grid)) return cudaErrorNotSupported;
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
    if (local) {
        int emb_here = emb;
        void* args[2] = {(void*)&p, (void*)&emb_here};
        return cudaLaunchKernel(m.dtype == WIND_DT_BF16 ? (const void*)simt_local_kernel<__nv_bfloat16> : (const void*)simt_local_kernel<float>,
                                dim3((unsigned)grid), dim3(SL_THREADS), args, smem, c.stream);
    }
    const void* fn = m.dtype == WIND_DT_BF16 ? sl_fn<__nv_bfloat16>(vec) : sl_fn<float>(vec);
    void* args[1] = {(void*)&p};
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)grid), dim3(SL_THREADS), args, smem, c.stream);
}

}  // namespace wind
