// One iteration of the beam search (Algorithm 3) as one kernel: decoder update of the hypotheses that have no state yet,
// their projection, the window's logits under every hypothesis, Eq. (1) and the K best entries each, written to host memory.
//
// As separate kernels an iteration of the 640-unit model with beam 4 took 85 us, of which 51 us were eleven kernels and copies
// (a block per hidden unit or per sixteen labels loads its weights, waits for them, and uses them once) and the rest gaps and
// the synchronisation.  Here hidden units, joint units and labels are dealt out over all SMs, every CTA requests all its
// weights (67 KB) at the start, the phases follow one another behind grid barriers, and the host polls for the result.
//
// A dot product is summed as the per-phase kernels sum it, so that both give the same bits: 32 chains, chain r over
// k = r, r + 32, ..., then a butterfly.  A thread carries four neighbouring chains, so eight threads make a row, and a warp
// four rows with 8-byte reads of the weights.
#include "wind_internal.cuh"
#include "wind_loop.cuh"
#include "wind_ptx.cuh"

#include <mutex>

namespace wind {

constexpr int BS_THREADS = 512;
constexpr int BS_WARPS = BS_THREADS / 32;
constexpr int BS_UTTS = 4;            // updates of a pass
constexpr int BS_ROWS = 4;            // window rows of a joint item

// dimensions shared by the host's plan and the kernel; all sizes in elements, offsets in bytes
struct BsPlan {
    int G, units, prows, labels;      // grid, and the most a CTA owns of each
    int ld_l, ld_p, ld_o;             // row pitches: gates (any layer), W_pred, W_out
    int k_l, k_p;                     // floats of a staged x row of the gates / of h
    int zrows, ld_z;                  // window rows of a joint pass
    uint32_t w_pred, w_out, area, x, total;   // area: the gates' weights, then x behind them; later z, then the window's logits
};
template <typename TW> __host__ __device__ inline int bs_pitch(int k) {
    // eight threads read a row's 32 elements and four rows are read at a time: rows shifted by half the banks
    const int p = (k + 31) / 32 * 32;
    return sizeof(TW) == 2 ? (p % 64 == 32 ? p : p + 32) : p + 4;
}
template <typename TW> __host__ __device__ inline BsPlan bs_plan(int G, int W, int K, int E, int P, int L, int H, int NV, uint32_t budget) {
    BsPlan s{};
    s.G = G;
    s.units = (P + G - 1) / G; s.prows = (H + G - 1) / G; s.labels = (NV + G - 1) / G;
    const int k0 = E + P, k1 = L > 1 ? 2 * P : 0, kmax = k0 > k1 ? k0 : k1;
    s.ld_l = bs_pitch<TW>(kmax); s.ld_p = bs_pitch<TW>(P); s.ld_o = bs_pitch<TW>(H);
    s.k_l = (kmax + 31) / 32 * 32; s.k_p = (P + 31) / 32 * 32;
    s.ld_z = (H + 31) / 32 * 32;
    unsigned long long off = 0;
    auto take = [&](unsigned long long bytes) { const unsigned long long o = off; off += (bytes + 15) / 16 * 16; return (uint32_t)o; };
    s.w_pred = take((unsigned long long)sizeof(TW) * s.prows * s.ld_p);
    s.w_out = take((unsigned long long)sizeof(TW) * s.labels * s.ld_o);
    s.area = (uint32_t)off;
    unsigned long long gates = (unsigned long long)sizeof(TW) * s.units * 4 * s.ld_l;
    s.x = (uint32_t)(s.area + gates);
    gates += 4ull * BS_UTTS * s.k_l;
    const unsigned long long window = 4ull * W * NV;
    unsigned long long area = gates > window ? gates : window;
    const unsigned long long row = 4ull * s.ld_z;
    int rows = (K * W + BS_ROWS - 1) / BS_ROWS * BS_ROWS;
    if (off + row * BS_ROWS <= budget) {
        const unsigned long long fit = (budget - off) / row / BS_ROWS * BS_ROWS;
        if ((unsigned long long)rows > fit) rows = (int)fit;
    } else {
        rows = BS_ROWS;
    }
    s.zrows = rows;
    if (row * rows > area) area = row * rows;
    off += area;
    s.total = off > 0xffffffffull ? 0xffffffffu : (uint32_t)off;
    return s;
}

struct BsParams {
    BeamStep io;
    Ctrl* ctrl;
    uint32_t bar_base;                 // arrivals at the grid barrier before this launch
    uint32_t extra_arrivals, budget;
    int E, P, L, H, NV, blank, act, W;
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

template <typename TW> __device__ __forceinline__ float bs_round(float x);
template <> __device__ __forceinline__ float bs_round<float>(float x) { return x; }
template <> __device__ __forceinline__ float bs_round<__nv_bfloat16>(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float4 bs_load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 bs_load4(const __nv_bfloat16* p) {
    const uint2 v = *reinterpret_cast<const uint2*>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.y));
    return make_float4(a.x, a.y, b.x, b.y);
}

// N dot products of this lane group's weight row with N rows of x; w and x point at the thread's first element.  All eight
// threads of the group get the sums.
template <int N, typename TW>
__device__ __forceinline__ void bs_dots(const TW* w, const float* x, int x_pitch, int steps, float* sum) {
    float a[N][4];
#pragma unroll
    for (int n = 0; n < N; ++n)
#pragma unroll
        for (int j = 0; j < 4; ++j) a[n][j] = 0.f;
#pragma unroll 4
    for (int i = 0; i < steps; ++i) {
        const float4 wv = bs_load4(w + 32 * i);
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const float4 xv = *reinterpret_cast<const float4*>(x + n * x_pitch + 32 * i);
            a[n][0] = fmaf(wv.x, xv.x, a[n][0]);
            a[n][1] = fmaf(wv.y, xv.y, a[n][1]);
            a[n][2] = fmaf(wv.z, xv.z, a[n][2]);
            a[n][3] = fmaf(wv.w, xv.w, a[n][3]);
        }
    }
#pragma unroll
    for (int n = 0; n < N; ++n) {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
#pragma unroll
            for (int j = 0; j < 4; ++j) a[n][j] += __shfl_xor_sync(0xffffffffu, a[n][j], o);
        sum[n] = (a[n][0] + a[n][2]) + (a[n][1] + a[n][3]);
    }
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
// (value, index) as one integer: larger values first, then smaller indices; 0 where there is none
__device__ __forceinline__ unsigned long long bs_pair(float v, int i) { return v > -INFINITY ? pack_key(v, (uint32_t)i) : 0ull; }
__device__ __forceinline__ unsigned long long bs_best_of_warp(unsigned long long key) {
    const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(key >> 32));
    const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(key >> 32) == hi ? (uint32_t)key : 0u);
    return ((unsigned long long)hi << 32) | lo;
}

// KL: entries of a thread's own list of best entries (at least K)
template <typename TW, int KL>
__global__ void __launch_bounds__(BS_THREADS, 1) beam_step_kernel(const BsParams p) {
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ int s_stop;
    __shared__ float s_lse[kMaxWindow], s_before[kMaxWindow];
    __shared__ unsigned long long s_cand[BS_WARPS * KL];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, grp = lane >> 3, q = lane & 7;
    const int G = gridDim.x, cta = blockIdx.x;
    const int P = p.P, H = p.H, NV = p.NV, K = p.io.K, LP = p.L * P;
    const BsPlan M = bs_plan<TW>(G, p.W, K, p.E, P, p.L, H, NV, p.budget);
    const int units = (P - cta + G - 1) / G, prows = (H - cta + G - 1) / G, labels = (NV - cta + G - 1) / G;
    TW* w_pred = reinterpret_cast<TW*>(sm + M.w_pred);
    TW* w_out = reinterpret_cast<TW*>(sm + M.w_out);
    TW* w_l = reinterpret_cast<TW*>(sm + M.area);
    float* xs = reinterpret_cast<float*>(sm + M.x);
    float* area = reinterpret_cast<float*>(sm + M.area);
    const int nu = p.io.n_update, nh = p.io.n_hyps;
    if (tid == 0) s_stop = 0;

    // n elements (whole 16-byte pieces) by one warp, asynchronously, and zeros up to a multiple of 32
    auto copy_row = [&](TW* dst, const TW* src, int n, int n32) {
        constexpr int PIECE = 16 / (int)sizeof(TW);
        for (int k = lane * PIECE; k < n; k += 32 * PIECE)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst + k)), "l"(src + k) : "memory");
        for (int k = n + lane; k < n32; k += 32) dst[k] = (TW)0.f;
    };
    auto load_layer = [&](int l) {
        const int nin = l == 0 ? p.E : P, K32 = (nin + P + 31) / 32 * 32;
        for (int i = warp; i < units * 4; i += BS_WARPS) {
            const size_t row = (size_t)(i & 3) * P + (size_t)(i >> 2) * G + cta;
            copy_row(w_l + i * M.ld_l, static_cast<const TW*>(p.w_ih[l]) + row * nin, nin, nin);
            copy_row(w_l + i * M.ld_l + nin, static_cast<const TW*>(p.w_hh[l]) + row * P, P, K32 - nin);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (nu > 0) load_layer(0);
    if (nu > 0)
        for (int i = warp; i < prows; i += BS_WARPS)
            copy_row(w_pred + i * M.ld_p, static_cast<const TW*>(p.w_pred) + ((size_t)i * G + cta) * P, P, M.k_p);
    for (int i = warp; i < labels; i += BS_WARPS)
        copy_row(w_out + i * M.ld_o, static_cast<const TW*>(p.w_out) + ((size_t)i * G + cta) * H, H, M.ld_z);
    asm volatile("cp.async.commit_group;" ::: "memory");

    uint32_t epoch = p.bar_base;
    auto arrive = [&] {
        __syncthreads();
        epoch += (uint32_t)G;
        if (tid == 0) { __threadfence(); atomicAdd(&p.ctrl->bar, 1u); }
    };
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
                    else if (now - t0 > kWaitLimitNs) { s_stop = 1; set_status(p.ctrl, WIND_ERR_TIMEOUT); break; }
                }
            }
        }
        __syncthreads();
        return s_stop == 0;
    };

    // ---- decoder update: per layer the gates of this CTA's hidden units, then h and c into the new hypotheses' slots ----
    if (nu > 0) {
        for (int l = 0; l < p.L; ++l) {
            const int nin = l == 0 ? p.E : P, K32 = (nin + P + 31) / 32 * 32;
            for (int u0 = 0; u0 < nu; u0 += BS_UTTS) {
                const int n_here = min(BS_UTTS, nu - u0);
                if (u0 > 0) __syncthreads();
                // x and the state before it, one row per update
                for (int u = 0; u < BS_UTTS; ++u) {
                    const int uu = u0 + min(u, n_here - 1);
                    for (int k = tid; k < K32; k += BS_THREADS) {
                        float x = 0.f;
                        if (k < nin) x = l == 0 ? (float)static_cast<const TW*>(p.emb)[(size_t)p.io.tok[uu] * p.E + k]
                                                : bs_round<TW>(__ldcg(p.h_pool + (size_t)p.io.dst[uu] * LP + (l - 1) * P + k));
                        else if (k < nin + P) x = bs_round<TW>(__ldcg(p.h_pool + (size_t)p.io.src[uu] * LP + l * P + k - nin));
                        xs[u * M.k_l + k] = x;
                    }
                }
                if (u0 == 0 && l == 0) asm volatile("cp.async.wait_group 1;" ::: "memory");   // the gates' weights; the others may still come
                else asm volatile("cp.async.wait_all;" ::: "memory");
                __syncthreads();
                for (int item = warp; item < units * 2; item += BS_WARPS) {
                    const int ui = item >> 1, u = (item & 1) * 2, j = ui * G + cta;
                    if (u >= n_here) continue;
                    // c and the biases are requested ahead of the sums
                    const int me = u0 + min(u + (lane & 1), n_here - 1);
                    const float c_in = __ldcg(p.c_pool + (size_t)p.io.src[me] * LP + l * P + j);
                    const float bias = p.b_ih[l][grp * P + j] + p.b_hh[l][grp * P + j];
                    float s[2];
                    bs_dots<2>(w_l + (ui * 4 + grp) * M.ld_l + 4 * q, xs + u * M.k_l + 4 * q, M.k_l, K32 / 32, s);
                    const float mine = ((lane & 1) ? s[1] : s[0]) + bias;
                    const float ai = __shfl_sync(0xffffffffu, mine, lane & 1), af = __shfl_sync(0xffffffffu, mine, 8 + (lane & 1)),
                                ag = __shfl_sync(0xffffffffu, mine, 16 + (lane & 1)), ao = __shfl_sync(0xffffffffu, mine, 24 + (lane & 1));
                    const float gi = 1.f / (1.f + expf(-ai)), gf = 1.f / (1.f + expf(-af)), gg = tanhf(ag), go = 1.f / (1.f + expf(-ao));
                    const float cc = gf * c_in + gi * gg;
                    if (lane < 2 && u + lane < n_here) {
                        p.c_pool[(size_t)p.io.dst[me] * LP + l * P + j] = cc;
                        p.h_pool[(size_t)p.io.dst[me] * LP + l * P + j] = go * tanhf(cc);
                    }
                }
            }
            arrive();
            if (l + 1 < p.L) load_layer(l + 1);
            if (!wait()) return;
        }
        // ---- pred_proj of this CTA's joint units ----
        for (int u0 = 0; u0 < nu; u0 += BS_UTTS) {
            const int n_here = min(BS_UTTS, nu - u0);
            if (u0 > 0) __syncthreads();
            for (int u = 0; u < n_here; ++u)
                for (int k = tid; k < M.k_p; k += BS_THREADS)
                    xs[u * M.k_l + k] = k < P ? bs_round<TW>(__ldcg(p.h_pool + (size_t)p.io.dst[u0 + u] * LP + (p.L - 1) * P + k)) : 0.f;
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
            for (int item = warp; item < (prows + 3) / 4 * n_here; item += BS_WARPS) {
                const int u = item % n_here, pi = item / n_here * 4 + grp, pr = min(pi, prows - 1), o = pr * G + cta;
                const float bias = p.b_pred[o];
                float s;
                bs_dots<1>(w_pred + pr * M.ld_p + 4 * q, xs + u * M.k_l + 4 * q, M.k_l, M.k_p / 32, &s);
                if (q == 0 && pi < prows) p.g_pool[(size_t)p.io.dst[u0 + u] * H + o] = s + bias;
            }
        }
        arrive();
        if (!wait()) return;
    }

    // ---- logits of this CTA's labels for every row of the window under every hypothesis ----
    const int n = p.io.n_rows, rows = nh * n;
    asm volatile("cp.async.wait_all;" ::: "memory");
    for (int r0 = 0; r0 < rows; r0 += M.zrows) {
        const int nr = min(M.zrows, rows - r0), nr4 = (nr + BS_ROWS - 1) / BS_ROWS;
        const int h4 = M.ld_z / 4;
        __syncthreads();
#pragma unroll 2
        for (int i = tid; i < nr4 * BS_ROWS * h4; i += BS_THREADS) {
            const int r = i / h4, k = (i - r * h4) * 4, row = r0 + r, b = row / n, w = row - b * n;
            float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row < rows && k < H) {
                const float4 e = bs_load4(static_cast<const TW*>(p.enc_proj) + (size_t)(p.io.t + w) * H + k);
                const float4 g = __ldcg(reinterpret_cast<const float4*>(p.g_pool + (size_t)p.io.slot[b] * H + k));
                z = make_float4(e.x + g.x, e.y + g.y, e.z + g.z, e.w + g.w);
                if (p.act == WIND_ACT_RELU) z = make_float4(fmaxf(z.x, 0.f), fmaxf(z.y, 0.f), fmaxf(z.z, 0.f), fmaxf(z.w, 0.f));
                else z = make_float4(tanhf(z.x), tanhf(z.y), tanhf(z.z), tanhf(z.w));
                z = make_float4(bs_round<TW>(z.x), bs_round<TW>(z.y), bs_round<TW>(z.z), bs_round<TW>(z.w));
            }
            *reinterpret_cast<float4*>(area + r * M.ld_z + k) = z;
        }
        __syncthreads();
        const int lgs = (labels + 3) / 4;
        for (int item = warp; item < lgs * nr4; item += BS_WARPS) {
            const int rg = item / lgs, li = (item - rg * lgs) * 4 + grp, lr = min(li, labels - 1), v = lr * G + cta;
            const float bias = p.b_out[v];
            float s[BS_ROWS];
            bs_dots<BS_ROWS>(w_out + lr * M.ld_o + 4 * q, area + rg * BS_ROWS * M.ld_z + 4 * q, M.ld_z, M.ld_z / 32, s);
            float mine = s[0];
#pragma unroll
            for (int i = 1; i < BS_ROWS; ++i) mine = q == i ? s[i] : mine;
            const int row = r0 + rg * BS_ROWS + q, b = row / n;
            if (q < BS_ROWS && rg * BS_ROWS + q < nr && li < labels) p.logits[((size_t)b * p.W + (row - b * n)) * NV + v] = mine + bias;
        }
    }
    arrive();
    if (cta >= nh) return;
    if (!wait()) return;

    // ---- Eq. (1) for hypothesis `cta`, the window's logits in shared memory ----
    const float* src = p.logits + (size_t)cta * p.W * NV;
    const int total = n * NV;
#pragma unroll 8
    for (int i = tid; i < total; i += BS_THREADS) area[i] = __ldcg(src + i);
    __syncthreads();
    for (int w = warp; w < n; w += BS_WARPS) {
        const float* row = area + w * NV;
        float mx = -INFINITY;
#pragma unroll 4
        for (int v = lane; v < NV; v += 32) mx = fmaxf(mx, row[v]);
        mx = bs_warp_max(mx);
        float se = 0.f;
#pragma unroll 4
        for (int v = lane; v < NV; v += 32) se += expf(row[v] - mx);
        se = bs_warp_sum(se);
        if (lane == 0) s_lse[w] = mx + logf(se);
    }
    __syncthreads();
    if (tid == 0) {
        float before = 0.f;
        for (int w = 0; w < n; ++w) {
            s_before[w] = before;
            before += area[w * NV + p.blank] - s_lse[w];
        }
    }
    __syncthreads();
    // ---- the K best entries, best first; equal values in order of (offset, label): a thread's own, a warp's, the block's ----
    unsigned long long best[KL];
#pragma unroll
    for (int j = 0; j < KL; ++j) best[j] = 0ull;
    for (int w = warp; w < n; w += BS_WARPS) {
        const float shift = s_before[w] - s_lse[w];
        for (int v = lane; v < NV; v += 32) {
            const float x = area[w * NV + v] + shift;
            unsigned long long key = (v == p.blank && w != n - 1) ? 0ull : bs_pair(x, w * NV + v);
            if (key > best[KL - 1]) {
#pragma unroll
                for (int j = 0; j < KL; ++j) {
                    const unsigned long long hi = key > best[j] ? key : best[j], lo = key > best[j] ? best[j] : key;
                    best[j] = hi; key = lo;
                }
            }
        }
    }
    auto pop_best = [&]() -> unsigned long long {       // the warp's best entry, taken out of its owner's list
        const unsigned long long top = bs_best_of_warp(best[0]);
        if (top != 0ull && best[0] == top) {
#pragma unroll
            for (int j = 0; j + 1 < KL; ++j) best[j] = best[j + 1];
            best[KL - 1] = 0ull;
        }
        return top;
    };
#pragma unroll 1
    for (int k = 0; k < KL; ++k) {
        const unsigned long long top = pop_best();
        if (lane == 0) s_cand[warp * KL + k] = top;
    }
    __syncthreads();
    if (warp != 0) return;
    // lanes 0..15 take one warp's list each
#pragma unroll
    for (int j = 0; j < KL; ++j) best[j] = lane < BS_WARPS ? s_cand[lane * KL + j] : 0ull;
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
        const unsigned long long top = pop_best();
        if (lane == 0) {
            const int i = (int)key_label(top), off = top != 0ull ? i / NV : -1;
            BeamTop r;
            r.label = top != 0ull ? i - off * NV : -1;
            r.jump = off;
            r.logp = top != 0ull ? key_logit(top) : -INFINITY;
            r.pad = 0;
            p.io.top[cta * K + k] = r;
        }
    }
    if (lane == 0) {
        __threadfence_system();
        *const_cast<volatile uint32_t*>(p.io.done + cta) = p.io.seq;
    }
}

template <typename TW> static const void* bs_fn(int K) {
    return K <= 4 ? (const void*)beam_step_kernel<TW, 4> : (K <= 8 ? (const void*)beam_step_kernel<TW, 8> : (const void*)beam_step_kernel<TW, 16>);
}

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
        for (int K : {4, 8, 16})
            for (const void* fn : {bs_fn<float>(K), bs_fn<__nv_bfloat16>(K)})
                if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, n - 4096)) != cudaSuccess) return e;   // static: below 4 KB
        g_bs_optin[dev] = n;
    }
    *optin = g_bs_optin[dev];
    return cudaSuccess;
}

static BsPlan bs_plan_of(const Call& c, int sms, uint32_t budget) {
    const wind_model_t& m = c.m;
    return m.dtype == WIND_DT_BF16 ? bs_plan<__nv_bfloat16>(sms, c.W, c.B, m.E, m.P, m.L, m.H, m.V + 1, budget)
                                   : bs_plan<float>(sms, c.W, c.B, m.E, m.P, m.L, m.H, m.V + 1, budget);
}

// Rows in whole 16-byte pieces (8 bf16; fp32 models take the same rule), a CTA's weights and one window's logits in shared
// memory, every CTA the owner of something, and a CTA for every hypothesis.  Else the per-phase kernels.
bool beam_step_supported(const Call& c) {
    const wind_model_t& m = c.m;
    if (m.E % 8 || m.P % 8 || m.H % 8) return false;
    auto aligned = [](const void* q) { return reinterpret_cast<uintptr_t>(q) % 16 == 0; };
    if (!aligned(m.emb) || !aligned(m.w_pred) || !aligned(m.w_out)) return false;
    for (int l = 0; l < m.L; ++l)
        if (!aligned(c.w_ih[l]) || !aligned(c.w_hh[l])) return false;
    int optin = 0, sms = 0;
    if (bs_device(&optin) != cudaSuccess || loop_sm_count(&sms) != cudaSuccess) { cudaGetLastError(); return false; }
    return c.B <= sms && bs_plan_of(c, sms, (uint32_t)optin - 4096u).total <= (uint32_t)optin - 4096u;
}

cudaError_t beam_step(const Call& c, const BeamStep& io, float* h_pool, float* c_pool, float* g_pool, float* logits, uint32_t* bar_base) {
    int optin = 0, sms = 0;
    cudaError_t e = bs_device(&optin);
    if (e == cudaSuccess) e = loop_sm_count(&sms);
    if (e != cudaSuccess) return e;
    const wind_model_t& m = c.m;
    BsParams p{};
    p.io = io;
    p.ctrl = c.ctrl();
    p.bar_base = *bar_base;
    p.extra_arrivals = (uint32_t)loop_extra_arrivals();
    p.budget = (uint32_t)optin - 4096u;
    p.E = m.E; p.P = m.P; p.L = m.L; p.H = m.H; p.NV = m.V + 1; p.blank = m.blank_id; p.act = m.act; p.W = c.W;
    p.emb = m.emb; p.w_pred = m.w_pred; p.b_pred = m.b_pred; p.w_out = m.w_out; p.b_out = m.b_out;
    for (int l = 0; l < m.L; ++l) { p.w_ih[l] = c.w_ih[l]; p.w_hh[l] = c.w_hh[l]; p.b_ih[l] = c.b_ih[l]; p.b_hh[l] = c.b_hh[l]; }
    p.enc_proj = c.enc_proj();
    p.h_pool = h_pool; p.c_pool = c_pool; p.g_pool = g_pool; p.logits = logits;
    *bar_base += (uint32_t)sms * (uint32_t)((io.n_update > 0 ? m.L + 1 : 0) + 1);
    const void* fn = m.dtype == WIND_DT_BF16 ? bs_fn<__nv_bfloat16>(io.K) : bs_fn<float>(io.K);
    void* args[1] = {(void*)&p};
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)sms), dim3(BS_THREADS), args, bs_plan_of(c, sms, p.budget).total, c.stream);
}

}  // namespace wind
