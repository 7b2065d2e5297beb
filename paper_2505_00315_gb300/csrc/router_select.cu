// Router (F1) and TopK selection (F2) of the MoSA layer, Sec. 2.2:
//   r = sigmoid(X W^r);   r^topk, I = TopK(r, k).
//
// The selection works on an order-preserving uint32 image of the fp32 scores
// (topk_select_kernel); an in-order compaction keeps every key above the k-th
// largest plus the lowest-index keys equal to it, so I comes out ascending (the
// order the causal mask works in) and ties go to the lower token index.  Output
// positions come from block-wide prefix sums, so no sort is needed.
#include <algorithm>
#include <mutex>

#include "launch.h"
#include "profile.h"
#include "simt_gemm.cuh"
#include "tc_common.cuh"

namespace mosa {
namespace {

template <class E>
struct RouterOp {
    static constexpr bool kAKFast = true;   // X rows are contiguous along d
    static constexpr bool kBKFast = false;  // W_r rows are contiguous along H
    int M, N, K;                            // B*T tokens, H heads, d
    int T, H;
    const E *X, *Wr;
    float *r_full;
    __device__ float a(int, int m, int kk) const { return to_f32(X[(size_t)m * K + kk]); }
    __device__ float b(int, int kk, int n) const { return to_f32(Wr[(size_t)kk * N + n]); }
    __device__ void store(int, int m, int n, float logit, bool = false) const {
        const int bb = m / T, t = m % T;
        r_full[((size_t)bb * H + n) * T + t] = 1.f / (1.f + expf(-logit));
    }
};

// Router on CUDA cores (fp32 storage, and bf16 where the tensor-core router does
// not apply: H % 8 != 0 or a head size other than 64).  A CTA computes 32 or (HT =
// 64) 64 tokens x HT heads (HT = 16, 32 or 64), HT/16 x 4 per thread, each
// score one multiply-add chain over d in ascending order (so that the scores
// do not depend on HT, and match RouterOp's bit for bit).  X comes through a
// ring of kRouterStages chunks of KC columns by 16-byte cp.async and is
// read eight columns of a token at a time; W_r (rows of any alignment) goes through
// registers, 16 elements per thread, one chunk ahead, into an fp32 tile.  Measured
// alone: B4 T2048 d1024 H60 193 us with the general 64 x 64 tile product (scalar
// loads, nothing in flight across its barriers), 42 us now, most of it its issue
// slots (67% used over the kernel under ncu, the FMA pipe 46% busy, shared memory 54%; packed
// fma.rn.f32x2 on X converted in shared memory was slower, 46 us); B1 T1531 d768
// H12 129 -> 12 us; fp32 B4 T1000 d768 H12 152 -> 14 us (a short wave of 125 CTAs: 27% and 16%).
constexpr int kRouterStages = 4;
template <int HT>
struct RouterTile {
    static constexpr int THREADS = HT == 64 ? 256 : 128, TOK = THREADS / 4;
    static constexpr int ELEMS = 16 * THREADS;   // of W_r per chunk
    static constexpr int KC = ELEMS / HT;        // columns of d per chunk
};

template <class E, int HT>
constexpr int router_ld() { return RouterTile<HT>::KC + 16 / (int)sizeof(E); }   // X row stride
template <class E, int HT>
constexpr int router_smem() {
    return RouterTile<HT>::ELEMS * 4 +
           kRouterStages * RouterTile<HT>::TOK * router_ld<E, HT>() * (int)sizeof(E);
}

// Eight consecutive elements as fp32.
__device__ __forceinline__ void widen8(const float *p, float (&v)[8]) {
    const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 4);
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
}
__device__ __forceinline__ void widen8(const bf16 *p, float (&v)[8]) {
    const uint4 u = *reinterpret_cast<const uint4 *>(p);
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        v[2 * e] = __uint_as_float(w[e] << 16);
        v[2 * e + 1] = __uint_as_float(w[e] & 0xFFFF0000u);
    }
}

template <class E, int HT>
__global__ void __launch_bounds__(RouterTile<HT>::THREADS)
    router_rows_kernel(const E *__restrict__ X, const E *__restrict__ Wr, float *__restrict__ r_full,
                       int M, int T, int H, int d, uint32_t *status) {
    if (status != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *status = 0u;
    constexpr int THREADS = RouterTile<HT>::THREADS, TOK = RouterTile<HT>::TOK;
    constexpr int KC = RouterTile<HT>::KC;
    constexpr int TM = HT / 16;                    // tokens per thread
    constexpr int UE = 16 / (int)sizeof(E);        // elements of a 16-byte unit
    constexpr int UNITS = TOK * KC / UE / THREADS; // X units per thread and chunk
    constexpr int WV = RouterTile<HT>::ELEMS / THREADS;
    constexpr int XLD = router_ld<E, HT>(), S = kRouterStages;
    extern __shared__ __align__(16) uint8_t router_sm[];
    float *Ws = reinterpret_cast<float *>(router_sm);
    E *Xs = reinterpret_cast<E *>(router_sm + RouterTile<HT>::ELEMS * 4);
    const int tid = threadIdx.x;
    const int hg = tid % (HT / 4), tg = tid / (HT / 4);
    const int m0 = blockIdx.x * TOK, h0 = blockIdx.y * HT;
    const int chunks = (d + KC - 1) / KC;
    E wr[WV];
    float acc[TM][4];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    auto fetch_x = [&](int c) {   // zeros past M and d (d % 8 == 0)
        E *dst = Xs + (c % S) * TOK * XLD;
#pragma unroll
        for (int v = 0; v < UNITS; ++v) {
            const int u = tid + THREADS * v, tok = u / (KC / UE), q = u % (KC / UE);
            const int kx = c * KC + q * UE;
            const bool on = m0 + tok < M && kx < d;
            tc::cp_async16(tc::smem_u32(dst + tok * XLD + q * UE),
                           on ? X + (size_t)(m0 + tok) * d + kx : X, on ? 16u : 0u);
        }
    };
    auto load_w = [&](int c) {
#pragma unroll
        for (int v = 0; v < WV; ++v) {
            const int e = tid + THREADS * v, kx = c * KC + e / HT, h = h0 + e % HT;
            wr[v] = kx < d && h < H ? Wr[(size_t)kx * H + h] : from_f32<E>(0.f);
        }
    };
    for (int c = 0; c < S - 1; ++c) {
        if (c < chunks) fetch_x(c);
        tc::cp_async_commit();
    }
    load_w(0);
    for (int c = 0; c < chunks; ++c) {
        tc::cp_async_wait<S - 2>();
        __syncthreads();   // chunk c of X is in; chunk c - 1 has been read
#pragma unroll
        for (int v = 0; v < WV; ++v) Ws[tid + THREADS * v] = to_f32(wr[v]);
        if (c + S - 1 < chunks) fetch_x(c + S - 1);
        tc::cp_async_commit();
        __syncthreads();
        if (c + 1 < chunks) load_w(c + 1);
        const E *xs = Xs + (c % S) * TOK * XLD + tg * TM * XLD;
#pragma unroll(TM == 4 ? 2 : 4)
        for (int k8 = 0; k8 < KC; k8 += 8) {
            float a[TM][8];
#pragma unroll
            for (int i = 0; i < TM; ++i) widen8(xs + i * XLD + k8, a[i]);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float4 b = *reinterpret_cast<const float4 *>(Ws + (k8 + e) * HT + 4 * hg);
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    acc[i][0] = fmaf(a[i][e], b.x, acc[i][0]);
                    acc[i][1] = fmaf(a[i][e], b.y, acc[i][1]);
                    acc[i][2] = fmaf(a[i][e], b.z, acc[i][2]);
                    acc[i][3] = fmaf(a[i][e], b.w, acc[i][3]);
                }
            }
        }
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // scores through shared memory, so that a warp writes 32 consecutive tokens
    tc::cp_async_wait<0>();
    __syncthreads();
    constexpr int RLD = TOK + 1;
    float *Rs = Ws;
    static_assert(router_smem<E, HT>() >= HT * RLD * 4, "score tile must fit in the operand tiles");
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            Rs[(4 * hg + j) * RLD + tg * TM + i] = 1.f / (1.f + expf(-acc[i][j]));
    __syncthreads();
    const int m = m0 + tid % TOK;
    if (m < M) {
        const int bb = m / T, t = m - bb * T;
        for (int h = tid / TOK; h < HT && h0 + h < H; h += THREADS / TOK)
            r_full[((size_t)bb * H + h0 + h) * T + t] = Rs[h * RLD + tid % TOK];
    }
}

// Order-preserving map of a non-NaN float to uint32 (-0 and +0 map together).
__device__ __forceinline__ uint32_t order_key(float f) {
    uint32_t u = __float_as_uint(f);
    if (u == 0x80000000u) u = 0u;
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
constexpr int kSelThreads = 1024;
constexpr int kSelMaxVec = 4;     // float4 per thread: rows up to 16384 scores
constexpr int kSelCand = 64;      // candidates ranked directly

// Four scores s[t .. t+3] (zeros past T).  Plain loads, not __ldg, which the compiler
// may move ahead of the wait for the kernel that writes the scores.
__device__ __forceinline__ float4 load_scores(const float *s, int t, int T, bool vec) {
    if (vec && t + 4 <= T) return *reinterpret_cast<const float4 *>(s + t);
    return make_float4(t < T ? s[t] : 0.f, t + 1 < T ? s[t + 1] : 0.f, t + 2 < T ? s[t + 2] : 0.f,
                       t + 3 < T ? s[t + 3] : 0.f);
}

// One CTA per row; thread t holds the scores 4 t + 4 v blockDim .. +3, v < V, in
// registers (V blockDim 4 >= T).  The k-th largest key is found by narrowing a key
// range [lo, lo + NB 2^shift): a histogram of the keys inside it over NB = 2
// blockDim equal bins, first over the row's own range [min, max], then over the
// bin that holds the k-th key, until
//   the bin's keys are all kept (router scores with a clear gap), or
//   at most kSelCand keys are left: every warp ranks them directly, or
//   the bin is one key wide: ties, kept in token order.
// With bins over the row's range instead of fixed digits of the key (sigmoid
// scores share two or three top bytes), one histogram is the rule; a pass costs
// three barriers.  What bounds it is the latency of that chain, not the few KB a
// row has.  Alone, against four 8-bit radix passes over keys in shared memory:
// 64 x 8192 k 256 13.3 -> 9.4 us (11.1 -> 7.3 with a margin after the k-th
// score), 1024 x 1024 k 64 12.3 -> 9.0, 1024 x 4096 k 64 29.3 -> 22.4, 32 x 4096
// k 2048 10.1 -> 9.0, 48 x 1000 k 125 7.9 -> 5.5.
// With first_token, token 0 is kept and k - 1 others are chosen.
template <int V>
__global__ void __launch_bounds__(kSelThreads)
topk_select_kernel(const float *scores, int T, int k, int32_t *I, float *rsel, int B, int H,
                   int32_t *gidx, float *rsel_hm, int first_token, unsigned long long *span) {
    __shared__ uint32_t hist[2][2 * kSelThreads];
    __shared__ uint32_t wsum[32], csum[V][32], esum[V][32];
    __shared__ uint32_t wmin[32], wmax[32], sh_bin, sh_left, sh_in, sh_n;
    __shared__ uint32_t cand_key[kSelCand];
    __shared__ int cand_tok[kSelCand];
    constexpr uint32_t kAll = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x;
    const int nwarps = nthr >> 5, NB = 2 * nthr;
    const int row = blockIdx.x;
    const float *s = scores + (size_t)row * T;
    const bool vec = (T & 3) == 0 && (reinterpret_cast<uintptr_t>(scores) & 15) == 0;
    for (int i = tid; i < NB; i += nthr) hist[0][i] = 0u;
    if (tid == 0) sh_n = 0u;
    asm volatile("griddepcontrol.wait;" ::: "memory");  // scores from the router kernel
    span_begin(span);
    float4 sc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) sc[v] = load_scores(s, 4 * (tid + v * nthr), T, vec);
    uint32_t key[V][4];
    uint32_t live = 0u;   // bit 4 v + e: a token to rank
    uint32_t mn = 0xffffffffu, mx = 0u;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const float x[4] = {sc[v].x, sc[v].y, sc[v].z, sc[v].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int t = 4 * (tid + v * nthr) + e;
            key[v][e] = order_key(x[e]);
            if (t < T && !(first_token && t == 0)) {
                live |= 1u << (4 * v + e);
                mn = min(mn, key[v][e]);
                mx = max(mx, key[v][e]);
            }
        }
    }
    mn = __reduce_min_sync(kAll, mn);
    mx = __reduce_max_sync(kAll, mx);
    if (lane == 0) {
        wmin[warp] = mn;
        wmax[warp] = mx;
    }
    __syncthreads();
    mn = __reduce_min_sync(kAll, lane < nwarps ? wmin[lane] : 0xffffffffu);
    mx = __reduce_max_sync(kAll, lane < nwarps ? wmax[lane] : 0u);
    const uint32_t lg_nb = 31 - __clz(NB);   // bins used: a power of two <= NB
    uint32_t lo = mn;
    uint32_t remaining = (uint32_t)(first_token ? k - 1 : k);
    // shift: the smallest with (max - lo) >> shift < 2^lg_nb
    const uint32_t range = mx - lo;
    const int bits = range == 0u ? 0 : 32 - __clz(range);
    int shift = bits > (int)lg_nb ? bits - (int)lg_nb : 0;
    uint32_t width_m1 = range;     // keys lo .. lo + width_m1 are in the range
    // what is kept: keys above thr, and keys equal to it up to token thr_tok
    // (or, with ties, the first `left` of them in token order)
    uint32_t thr = 0u;
    int thr_tok = -1;
    bool ties = false;
    if (remaining == 0u) thr = 0xffffffffu;   // first_token with k = 1: nothing else
    for (int pass = 0; remaining > 0u; ++pass) {
        uint32_t *hc = hist[pass & 1], *hn = hist[(pass + 1) & 1];
        for (int i = tid; i < NB; i += nthr) hn[i] = 0u;   // read by no one this pass
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint32_t off = key[v][e] - lo;   // below lo wraps past the range
                if ((live >> (4 * v + e) & 1u) && off <= width_m1) atomicAdd(&hc[off >> shift], 1u);
            }
        __syncthreads();
        // warp w sums bins NB - 64 (w + 1) .. +63 (largest keys first), then every
        // warp finds the group that reaches the k-th key
        const int b0 = NB - 64 * (warp + 1);
        const uint32_t c0 = hc[b0 + 63 - 2 * lane], c1 = hc[b0 + 62 - 2 * lane];
        const uint32_t tot = __reduce_add_sync(kAll, c0 + c1);
        if (lane == 0) wsum[warp] = tot;
        __syncthreads();
        uint32_t incl = lane < nwarps ? wsum[lane] : 0u;
        const uint32_t own = incl;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(kAll, incl, off);
            if (lane >= off) incl += y;
        }
        const int g = __ffs(__ballot_sync(kAll, incl >= remaining)) - 1;
        const uint32_t before = __shfl_sync(kAll, incl - own, g);
        if (warp == g) {
            uint32_t in2 = c0 + c1;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t y = __shfl_up_sync(kAll, in2, off);
                if (lane >= off) in2 += y;
            }
            const int l = __ffs(__ballot_sync(kAll, before + in2 >= remaining)) - 1;
            if (lane == l) {
                const uint32_t b4 = before + in2 - (c0 + c1);   // keys in larger bins
                const bool second = b4 + c0 < remaining;
                sh_bin = (uint32_t)(b0 + (second ? 62 : 63) - 2 * lane);
                sh_left = remaining - b4 - (second ? c0 : 0u);
                sh_in = second ? c1 : c0;
            }
        }
        __syncthreads();
        remaining = sh_left;
        const uint32_t in = sh_in;
        lo += sh_bin << shift;
        width_m1 = shift == 0 ? 0u : min((1u << shift) - 1u, 0xffffffffu - lo);
        if (in == remaining) {   // the whole bin is kept
            thr = lo;
            thr_tok = T;
            break;
        }
        if (in <= kSelCand) {
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if ((live >> (4 * v + e) & 1u) && key[v][e] - lo <= width_m1) {
                        const uint32_t at = atomicAdd(&sh_n, 1u);
                        cand_key[at] = key[v][e];
                        cand_tok[at] = 4 * (tid + v * nthr) + e;
                    }
            __syncthreads();
            // rank of this lane's candidates; the one of rank remaining - 1 is the k-th
            uint32_t rk[2] = {0u, 0u}, ck[2];
            int ct[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int c = lane + 32 * u;
                ck[u] = c < (int)in ? cand_key[c] : 0u;
                ct[u] = c < (int)in ? cand_tok[c] : 0x7fffffff;
            }
            for (int c = 0; c < (int)in; ++c) {
                const uint32_t ok = cand_key[c];
                const int ot = cand_tok[c];
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    rk[u] += ok > ck[u] || (ok == ck[u] && ot < ct[u]) ? 1u : 0u;
            }
            const bool h0 = lane < (int)in && rk[0] == remaining - 1u;
            const bool h1 = lane + 32 < (int)in && rk[1] == remaining - 1u;
            const int src = __ffs(__ballot_sync(kAll, h0 || h1)) - 1;
            thr = __shfl_sync(kAll, h1 ? ck[1] : ck[0], src);
            thr_tok = __shfl_sync(kAll, h1 ? ct[1] : ct[0], src);
            break;
        }
        if (shift == 0) {   // more than kSelCand keys equal to lo, `remaining` of them kept
            thr = lo;
            ties = true;
            break;
        }
        shift = shift > (int)lg_nb ? shift - (int)lg_nb : 0;
    }
    // The whole-bin stop keeps every key of the bin, above lo as well as lo itself
    // (thr_tok = T); a threshold key keeps its tokens up to thr_tok.
    uint32_t take = 0u, eq = 0u;
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint32_t bit = 1u << (4 * v + e);
            const int t = 4 * (tid + v * nthr) + e;
            if (!(live & bit)) {
                if (first_token && t == 0) take |= bit;
                continue;
            }
            if (key[v][e] > thr || (key[v][e] == thr && t <= thr_tok)) take |= bit;
            if (key[v][e] == thr) eq |= bit;
        }
    if (ties) {
        // the first `remaining` tokens whose key is thr: their order from one
        // block-wide scan of the counts
        uint32_t pre[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const uint32_t n = __popc(eq >> (4 * v) & 15u);
            uint32_t in2 = n;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t y = __shfl_up_sync(kAll, in2, off);
                if (lane >= off) in2 += y;
            }
            if (lane == 31) esum[v][warp] = in2;
            pre[v] = in2 - n;
        }
        __syncthreads();
        uint32_t base = 0u;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const uint32_t w = lane < nwarps ? esum[v][lane] : 0u;
            uint32_t at = base + __reduce_add_sync(kAll, lane < warp ? w : 0u) + pre[v];
            base += __reduce_add_sync(kAll, w);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (eq >> (4 * v + e) & 1u) {
                    if (at < remaining) take |= 1u << (4 * v + e);
                    ++at;
                }
        }
    }
    uint32_t pre[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const uint32_t n = __popc(take >> (4 * v) & 15u);
        uint32_t in2 = n;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(kAll, in2, off);
            if (lane >= off) in2 += y;
        }
        if (lane == 31) csum[v][warp] = in2;
        pre[v] = in2 - n;
    }
    __syncthreads();
    const int hh = row % H, bb = row / H;
    const size_t out = (size_t)row * k, out_hm = ((size_t)hh * B + bb) * k;
    uint32_t base = 0u;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const uint32_t w = lane < nwarps ? csum[v][lane] : 0u;
        uint32_t pos = base + __reduce_add_sync(kAll, lane < warp ? w : 0u) + pre[v];
        base += __reduce_add_sync(kAll, w);
        const float x[4] = {sc[v].x, sc[v].y, sc[v].z, sc[v].w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (take >> (4 * v + e) & 1u) {
                const int t = 4 * (tid + v * nthr) + e;
                I[out + pos] = t;
                rsel[out + pos] = x[e];
                if (gidx != nullptr) {
                    gidx[out_hm + pos] = bb * T + t;
                    rsel_hm[out_hm + pos] = x[e];
                }
                ++pos;
            }
    }
    // The next kernel launches only now: launched at this kernel's start, its
    // CTAs (one per SM for the projections) sat on every SM this grid of B*H
    // CTAs leaves idle, and the side stream's copies and zeroing found no SM
    // until the attention kernel's tail (measured at B4 T4096 d1024 H16 k1024:
    // a 13 us wait before the output product, 394 -> 381 us a step).
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (span != nullptr) {
        __syncthreads();
        span_end(span);
    }
}

// Block-wide exclusive prefix sum of v (thread order); `total` receives the
// sum.  sh has 33 entries.  Two barriers.
__device__ __forceinline__ unsigned long long block_excl_scan(unsigned long long v,
                                                              unsigned long long *sh,
                                                              unsigned long long &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    unsigned long long incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) sh[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const unsigned long long w = lane < nwarps ? sh[lane] : 0ull;
        unsigned long long wi = w;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, wi, off);
            if (lane >= off) wi += y;
        }
        sh[lane] = wi - w;
        if (lane == 31) sh[32] = wi;
    }
    __syncthreads();
    total = sh[32];
    return sh[warp] + incl - v;
}

// Rows of more than 16384 scores: one CTA per row, four 8-bit radix passes over the
// scores in memory.  The passes use two histograms in turn (the next one is cleared while the
// current one fills), so a pass costs two barriers; the compaction gives each
// thread a contiguous segment of the row and places its selected keys after
// one block-wide scan of the per-segment counts.
__global__ void __launch_bounds__(kSelThreads)
topk_long_kernel(const float *scores, int T, int k, int32_t *I,
                   float *rsel, int B, int H, int32_t *gidx,
                   float *rsel_hm, int first_token, unsigned long long *span) {
    __shared__ uint32_t hist[2][256];
    __shared__ unsigned long long sh[33];
    __shared__ uint32_t sh_prefix, sh_remaining, sh_done;
    asm volatile("griddepcontrol.wait;" ::: "memory");  // scores from the router kernel
    span_begin(span);
    const int row = blockIdx.x;
    const float *s = scores + (size_t)row * T;
    const int tid = threadIdx.x;
    for (int i = tid; i < 256; i += blockDim.x) hist[0][i] = 0u;
    // token 0's key under first_token: above every score's
    auto key_of = [&](int t) -> uint32_t {
        return (first_token && t == 0) ? 0xFFFFFFFFu : order_key(s[t]);
    };
    __syncthreads();

    uint32_t prefix = 0u, mask = 0u, remaining = (uint32_t)k;
    for (int pass = 0; pass < 4; ++pass) {
        const int shift = 24 - 8 * pass;
        uint32_t *hc = hist[pass & 1], *hn = hist[(pass + 1) & 1];
        for (int i = tid; i < 256; i += blockDim.x) hn[i] = 0u;  // read by no one this pass
        // (plain shared atomics: measured at 1024 threads and 4096 keys, about
        // 700-800 cycles a pass whether the keys fall into three bins or 256;
        // aggregating equal bins per warp first (match.any) cost 1300-8100)
        for (int t = tid; t < T; t += blockDim.x) {
            const uint32_t key = key_of(t);
            if ((key & mask) == prefix) atomicAdd(&hc[(key >> shift) & 255u], 1u);
        }
        __syncthreads();
        if (tid < 32) {
            // Lane l owns the 8 bins 255-8l ... 248-8l (largest keys first).
            const int lane = tid;
            uint32_t c[8], sum = 0u;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                c[j] = hc[255 - (lane * 8 + j)];
                sum += c[j];
            }
            uint32_t incl = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += y;
            }
            const uint32_t reach = __ballot_sync(0xffffffffu, incl >= remaining);
            const int first = __ffs(reach) - 1;  // the candidates always number >= remaining
            if (lane == first) {
                uint32_t cum = incl - sum;
                int bin = 0;
                uint32_t left = remaining;
                uint32_t in_bin = 0u;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (cum + c[j] >= remaining) {
                        bin = 255 - (lane * 8 + j);
                        left = remaining - cum;
                        in_bin = c[j];
                        break;
                    }
                    cum += c[j];
                }
                sh_prefix = prefix | ((uint32_t)bin << shift);
                sh_remaining = left;
                // every key left in the bin is kept: the set is decided
                sh_done = in_bin == left ? 1u : 0u;
            }
        }
        __syncthreads();
        prefix = sh_prefix;
        remaining = sh_remaining;
        mask |= 255u << shift;
        if (sh_done) break;
    }
    // Under `mask` (the bytes decided so far) prefix is now the k-th largest
    // key; the first `remaining` keys equal to it there (in token order) are
    // kept, with every key above it.  When the passes stop early, every key
    // equal to it is kept (`remaining` of them), as the full passes would.
    const uint32_t thr = prefix;
    const int per = (T + (int)blockDim.x - 1) / (int)blockDim.x;
    const int t0 = min(T, tid * per), t1 = min(T, t0 + per);
    uint32_t n_gt = 0u, n_eq = 0u;
    for (int t = t0; t < t1; ++t) {
        const uint32_t key = key_of(t) & mask;
        n_gt += key > thr ? 1u : 0u;
        n_eq += key == thr ? 1u : 0u;
    }
    unsigned long long tot;
    const unsigned long long before =
        block_excl_scan(((unsigned long long)n_gt << 32) | n_eq, sh, tot);
    uint32_t eq_before = (uint32_t)(before & 0xffffffffu);
    uint32_t pos = (uint32_t)(before >> 32) + min(eq_before, remaining);
    const int hh = row % H, bb = row / H;
    for (int t = t0; t < t1 && pos < (uint32_t)k; ++t) {
        const uint32_t full = key_of(t), key = full & mask;
        bool take = key > thr;
        if (key == thr) take = eq_before++ < remaining;
        if (take) {
            const float v = s[t];
            I[(size_t)row * k + pos] = t;
            rsel[(size_t)row * k + pos] = v;
            if (gidx != nullptr) {
                const size_t o = ((size_t)hh * B + bb) * k + pos;
                gidx[o] = bb * T + t;
                rsel_hm[o] = v;
            }
            ++pos;
        }
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (span != nullptr) {
        __syncthreads();
        span_end(span);
    }
}

__global__ void indices_to_rows_kernel(const int32_t *I, const float *rsel, int B, int H, int T,
                                       int k, int32_t *gidx, float *rsel_hm, uint32_t *status) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int row = blockIdx.x;  // b*H + h
    const int hh = row % H, bb = row / H;
    const int32_t *Ir = I + (size_t)row * k;
    int bad = 0;
    for (int i = threadIdx.x; i < k; i += blockDim.x) {
        const int32_t t = Ir[i];
        if (t < 0 || t >= T || (i > 0 && Ir[i - 1] >= t)) bad = 1;
    }
    bad = __syncthreads_or(bad);
    if (bad && threadIdx.x == 0) atomicOr(status, kStatusBadIndex);
    for (int i = threadIdx.x; i < k; i += blockDim.x) {
        const int32_t t = bad ? i : Ir[i];
        const size_t o = ((size_t)hh * B + bb) * k + i;
        gidx[o] = bb * T + t;
        rsel_hm[o] = rsel[(size_t)row * k + i];
    }
}

// Dense heads (Sec. 2.1, Eq. mha; the dense heads of a hybrid layer,
// Sec. 2.2): every (b, h) keeps all of its k = T tokens with score 1, so row
// m = b*k + i of a head gathers X row b*T + i = m.
__global__ void dense_rows_kernel(long long n, long long rows_per_head,
                                  int32_t *__restrict__ gidx, float *__restrict__ rsel_hm) {
    for (long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x; o < n;
         o += (long long)gridDim.x * blockDim.x) {
        gidx[o] = (int32_t)(o % rows_per_head);
        rsel_hm[o] = 1.f;
    }
}

}  // namespace

template <class E, int HT>
static cudaError_t router_rows(const Dims &dm, const void *X, const void *Wr, float *r_full,
                               uint32_t *status, cudaStream_t stream) {
    const int M = dm.B * dm.T;
    constexpr int tok = RouterTile<HT>::TOK;
    const dim3 grid((M + tok - 1) / tok, (dm.H + HT - 1) / HT);
    constexpr int smem = router_smem<E, HT>();
    const cudaError_t e = allow_smem((const void *)router_rows_kernel<E, HT>, smem);
    if (e != cudaSuccess) return e;
    router_rows_kernel<E, HT><<<grid, RouterTile<HT>::THREADS, smem, stream>>>(
        (const E *)X, (const E *)Wr, r_full, M, dm.T, dm.H, dm.d, status);
    note_launches(1);
    return cudaGetLastError();
}

template <class E>
static cudaError_t router_t(const Dims &dm, const void *X, const void *Wr, float *r_full,
                            uint32_t *status, cudaStream_t stream) {
    if ((reinterpret_cast<uintptr_t>(X) & 15) != 0) {   // no 16-byte loads of its rows
        if (status != nullptr) {
            const cudaError_t e = cudaMemsetAsync(status, 0, sizeof(uint32_t), stream);
            if (e != cudaSuccess) return e;
        }
        RouterOp<E> op{dm.B * dm.T, dm.H, dm.d, dm.T, dm.H, (const E *)X, (const E *)Wr, r_full};
        return launch_simt_gemm(op, 1, stream);
    }
    if (dm.H <= 16) return router_rows<E, 16>(dm, X, Wr, r_full, status, stream);
    if (dm.H <= 32) return router_rows<E, 32>(dm, X, Wr, r_full, status, stream);
    return router_rows<E, 64>(dm, X, Wr, r_full, status, stream);
}

cudaError_t launch_router(const Dims &dm, const void *X, const void *Wr, float *r_full,
                          uint32_t *status, cudaStream_t stream) {
    return dm.bf16 ? router_t<bf16>(dm, X, Wr, r_full, status, stream)
                   : router_t<float>(dm, X, Wr, r_full, status, stream);
}

// W_r [d,H] -> Wp [d,Hp], columns H..Hp-1 zero, and the status word zeroed
// (status != nullptr).  Launched without the early-launch attribute, so it
// reads W_r and writes the status word only after all earlier work on the
// stream; it lets the router launch early at once (the router still waits for
// its completion before its first load).
__global__ void pad_wr_kernel(const bf16 *__restrict__ Wr, bf16 *__restrict__ Wp, int d, int H,
                              int Hp, uint32_t *status) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (status != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *status = 0;
    const size_t n = (size_t)d * Hp;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % Hp);
        Wp[i] = c < H ? Wr[(i / Hp) * H + c] : __float2bfloat16(0.f);
    }
}

cudaError_t launch_router_auto(const Dims &dm, const void *X, const void *Wr, float *r_full,
                               uint32_t *status, cudaStream_t stream, void *wr_pad,
                               bool zero_status) {
    cudaError_t e = cudaSuccess;
    const bool tc = use_tc(dm) && tc_router_applies(dm);
    // The tensor-core router loads W_r in blocks of 64 columns; when H is not
    // a multiple of 64 it reads a zero-padded copy, since blocks reaching past
    // column H (filled by the copy engine) ran its main loop at about 60% of
    // the in-bounds speed (10.8 against 6.3 us at B4 T4096 d1024 H8).
    const bool pad = tc && wr_pad != nullptr && dm.H % 64 != 0;
    const int hp64 = (dm.H + 63) / 64 * 64;
    if (pad) {
        const size_t n = (size_t)dm.d * hp64;
        const int grid = (int)std::min<size_t>((n + 255) / 256, 608);
        pad_wr_kernel<<<grid, 256, 0, stream>>>(static_cast<const bf16 *>(Wr),
                                                 static_cast<bf16 *>(wr_pad), dm.d, dm.H, hp64,
                                                 zero_status ? status : nullptr);
        note_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    } else if (tc && zero_status) {
        if ((e = cudaMemsetAsync(status, 0, sizeof(uint32_t), stream)) != cudaSuccess) return e;
    }
    if (tc && tc_router(dm, X, pad ? wr_pad : Wr, pad ? hp64 : dm.H, r_full, status, stream, &e))
        return e;
    // (launched without the early-launch attribute, so the status word is zeroed
    // after all earlier work on the stream)
    return launch_router(dm, X, Wr, r_full, zero_status ? status : nullptr, stream);
}

cudaError_t launch_select(int rows, int T, int k, const float *scores, int32_t *I, float *rsel,
                          int B, int H, int32_t *gidx, float *rsel_hm, cudaStream_t stream,
                          bool first_token) {
    if (rows <= 0) return cudaSuccess;
    if (T > 16 * kSelThreads) {
        const cudaError_t e = launch_pdl(topk_long_kernel, dim3(rows), dim3(kSelThreads), 0, stream,
                                         scores, T, k, I, rsel, B, H, gidx, rsel_hm,
                                         first_token ? 1 : 0, active_span());
        note_launches(1);
        return e;
    }
    // four scores per thread while all rows' threads fit the 152 SMs at once
    // (1024 each at 64 registers) and a CTA has at most 1024; else eight or sixteen
    int V = 1;
    auto threads = [&]() { return ((T + 4 * V - 1) / (4 * V) + 31) / 32 * 32; };
    while (V < kSelMaxVec && (threads() > kSelThreads || (long long)rows * threads() > 152 * 1024)) V *= 2;
    auto kern = V == 1 ? topk_select_kernel<1> : V == 2 ? topk_select_kernel<2> : topk_select_kernel<4>;
    const cudaError_t e = launch_pdl(kern, dim3(rows), dim3(threads()), 0, stream, scores, T, k, I,
                                     rsel, B, H, gidx, rsel_hm, first_token ? 1 : 0, active_span());
    note_launches(1);
    return e;
}

cudaError_t launch_indices_to_rows(const Dims &dm, const int32_t *I, const float *rsel,
                                   int32_t *gidx, float *rsel_hm, uint32_t *status,
                                   cudaStream_t stream) {
    indices_to_rows_kernel<<<dm.B * dm.H, 256, 0, stream>>>(I, rsel, dm.B, dm.H, dm.T, dm.k,
                                                           gidx, rsel_hm, status);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_dense_rows(const Dims &dm, int32_t *gidx, float *rsel_hm, cudaStream_t stream) {
    const long long n = dm.rows();
    if (n <= 0) return cudaSuccess;
    const long long blocks = (n + 255) / 256;
    dense_rows_kernel<<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, stream>>>(
        n, (long long)dm.B * dm.k, gidx, rsel_hm);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace mosa
