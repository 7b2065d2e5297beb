// Index-masked causal attention over the k selected tokens of each head
// (Sec. 2.1 Eq. attention, Sec. 2.2 mask M_ij = 0 iff I_i >= I_j) on CUDA
// cores, fp32 arithmetic: fp32 storage, and bf16 storage with a head size other
// than 64.  I is strictly ascending, so I_i >= I_j is j <= i.
//
// A CTA of 256 threads (16 x 16) owns a tile of 16 RQ rows of one (sequence,
// head) and walks over 64-row tiles of the other side in shared memory; thread
// (ty, tx) computes RQ x 4 elements of each 16 RQ x 64 score tile and RQ x
// h'/16 elements of each result, every operand read as float4.  RQ x 4 by 4
// steps take 16 RQ multiply-adds for RQ + 8 shared-memory wavefronts per
// thread row, so at RQ = 4 the FMA pipe has more to do than shared memory (16 against
// 12 cycles of an SM); smaller tiles trade that for more CTAs.  With eight or sixteen
// warps on an SM neither is full (ncu, bf16 h' = 128 B4 T1024 H16 k128: forward, RQ = 2, FMA pipe
// 29% busy, shared memory 64%; backward, RQ = 4, 34% and 47%): the barriers of a tile's loads and
// the chains between them are what is left.
//
// Forward (F4): online softmax; writes A, diag(r^topk) A and the row
// log-sum-exp.  Backward (B2): P is recomputed from the saved log-sum-exp;
//   dP = dA V^T, dS = P o (dP - D), dQ = dS K / sqrt(h'), dK = dS^T Q / sqrt(h'),
//   dV = P^T dA, with D = rowsum(dA o A);
// the CTAs of one launch take query tiles (dQ) or key tiles (dK and dV), so no
// sum crosses CTAs.
#include <cfloat>

#include "launch.h"
#include "profile.h"
#include "tc_common.cuh"

namespace mosa {
namespace {

constexpr int kThreads = 256;
constexpr int kCol = 64;          // rows of the walked side per step
constexpr int kPsLd = kCol + 4;   // row stride of the score tile (floats)

// Row stride of an operand tile in shared memory: h' + 4 floats, so that 16
// float4 reads of consecutive rows at one column fall into distinct banks.
template <int HP>
constexpr int ld_of() { return HP + 4; }

// Columns c .. c+3 of an intermediate row as stored (fp32 values, or the hi and
// lo halves), and their values.
template <class TS>
__device__ __forceinline__ uint4 ld4_raw(const void *p, size_t row, int cols, int c) {
    if constexpr (sizeof(TS) == sizeof(float)) {
        return *reinterpret_cast<const uint4 *>(static_cast<const float *>(p) + row * cols + c);
    } else {
        const bf16 *q = static_cast<const bf16 *>(p) + row * 2 * cols + c;
        const uint2 h = *reinterpret_cast<const uint2 *>(q), l = *reinterpret_cast<const uint2 *>(q + cols);
        return make_uint4(h.x, h.y, l.x, l.y);
    }
}
template <class TS>
__device__ __forceinline__ float4 values4(const uint4 &u) {
    if constexpr (sizeof(TS) == sizeof(float)) {
        return make_float4(__uint_as_float(u.x), __uint_as_float(u.y), __uint_as_float(u.z),
                           __uint_as_float(u.w));
    } else {
        auto lo16 = [](uint32_t w) { return __uint_as_float(w << 16); };
        auto hi16 = [](uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); };
        return make_float4(lo16(u.x) + lo16(u.z), hi16(u.x) + hi16(u.z), lo16(u.y) + lo16(u.w),
                           hi16(u.y) + hi16(u.w));
    }
}
template <class TS>
__device__ __forceinline__ void st4(void *p, size_t row, int cols, int c, const float (&v)[4]) {
    if constexpr (sizeof(TS) == sizeof(float)) {
        *reinterpret_cast<float4 *>(static_cast<float *>(p) + row * cols + c) =
            make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) Inter<TS>::st(p, row, cols, c + e, v[e]);
    }
}

// Rows r0 .. r0 + N - 1 of src ([., HP] intermediates; rows at or past `end`
// become zeros), read into registers by fetch() and written as fp32 into
// dst [N][HP + 4] by put(), so that all of a thread's loads are in flight at once
// (in one rolled loop of a load and a store the forward took 44 instead of 33 us
// and the backward 100 instead of 80 at bf16 h' = 128, B4 T1024 H16 k128; the
// next tile in flight during a tile's products as well gained nothing).
template <class TS, int HP, int N>
struct Tile {
    static constexpr int TOTAL = N * (HP / 4), PER = (TOTAL + kThreads - 1) / kThreads;
    uint4 raw[PER];
    __device__ __forceinline__ void fetch(const void *src, size_t base, int r0, int end) {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int e = threadIdx.x + kThreads * i, r = e / (HP / 4), c = e % (HP / 4) * 4;
            raw[i] = make_uint4(0u, 0u, 0u, 0u);
            if ((TOTAL % kThreads == 0 || e < TOTAL) && r0 + r < end)
                raw[i] = ld4_raw<TS>(src, base + r0 + r, HP, c);
        }
    }
    // True if this thread met a value that is not finite.
    __device__ __forceinline__ bool put(float *dst, float f) const {
        float bad = 0.f;   // 0 times a non-finite value is NaN
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int e = threadIdx.x + kThreads * i, r = e / (HP / 4), c = e % (HP / 4) * 4;
            const float4 v = values4<TS>(raw[i]);
            if (TOTAL % kThreads == 0 || e < TOTAL)
                *reinterpret_cast<float4 *>(dst + r * ld_of<HP>() + c) =
                    make_float4(v.x * f, v.y * f, v.z * f, v.w * f);
            bad = fmaf(v.x, 0.f, fmaf(v.y, 0.f, fmaf(v.z, 0.f, fmaf(v.w, 0.f, bad))));
        }
        return !(bad == 0.f);
    }
};

// s[r][c] = <X row ty*RQ + r, Y row tx + 16 c>
template <int HP, int RQ>
__device__ __forceinline__ void dot_tile(const float *X, const float *Y, int ty, int tx,
                                         float (&s)[RQ][4]) {
    constexpr int LD = ld_of<HP>();
#pragma unroll
    for (int r = 0; r < RQ; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) s[r][c] = 0.f;
#pragma unroll 4
    for (int p = 0; p < HP; p += 4) {
        float4 x[RQ], y[4];
#pragma unroll
        for (int r = 0; r < RQ; ++r) x[r] = *reinterpret_cast<const float4 *>(X + (ty * RQ + r) * LD + p);
#pragma unroll
        for (int c = 0; c < 4; ++c) y[c] = *reinterpret_cast<const float4 *>(Y + (tx + 16 * c) * LD + p);
#pragma unroll
        for (int r = 0; r < RQ; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c)
                s[r][c] = fmaf(x[r].w, y[c].w,
                               fmaf(x[r].z, y[c].z, fmaf(x[r].y, y[c].y, fmaf(x[r].x, y[c].x, s[r][c]))));
    }
}

// Columns of a result row that thread tx owns: h'/16 of them, in groups of
// W = min(4, h'/16) at W tx + 64 e.
template <int HP>
struct Cols {
    static constexpr int N = HP / 16, W = N < 4 ? N : 4, G = N / W;
};

// o[r][.] += sum_j P[ty*RQ + r][j] Y[j][cols of tx], j < n (n a multiple of 4)
template <int HP, int RQ>
__device__ __forceinline__ void accumulate(const float *P, const float *Y, int ty, int tx, int n,
                                           float (&o)[RQ][HP / 16]) {
    using C = Cols<HP>;
    constexpr int LD = ld_of<HP>();
#pragma unroll 2
    for (int j = 0; j < n; j += 4) {
        float4 x[RQ];
#pragma unroll
        for (int r = 0; r < RQ; ++r) x[r] = *reinterpret_cast<const float4 *>(P + (ty * RQ + r) * kPsLd + j);
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            float y[C::N];
#pragma unroll
            for (int e = 0; e < C::G; ++e) {
                const float *src = Y + (j + jj) * LD + C::W * tx + 64 * e;
                if constexpr (C::W == 4) {
                    const float4 v = *reinterpret_cast<const float4 *>(src);
                    y[4 * e] = v.x;
                    y[4 * e + 1] = v.y;
                    y[4 * e + 2] = v.z;
                    y[4 * e + 3] = v.w;
                } else {
#pragma unroll
                    for (int w = 0; w < C::W; ++w) y[w] = src[w];
                }
            }
#pragma unroll
            for (int r = 0; r < RQ; ++r) {
                const float pr = jj == 0 ? x[r].x : jj == 1 ? x[r].y : jj == 2 ? x[r].z : x[r].w;
#pragma unroll
                for (int c = 0; c < C::N; ++c) o[r][c] = fmaf(pr, y[c], o[r][c]);
            }
        }
    }
}

// The same sum without the masked elements (live(r, j) false), whose P is
// zero: needed only when Y holds a value that is not finite, since 0 times it is not 0.
template <int HP, int RQ, class Live>
__device__ __noinline__ void accumulate_masked(const float *P, const float *Y, int ty, int tx, int n,
                                               float (&o)[RQ][HP / 16], Live live) {
    using C = Cols<HP>;
    for (int j = 0; j < n; ++j)
#pragma unroll
        for (int r = 0; r < RQ; ++r) {
            if (!live(r, j)) continue;
            const float pr = P[(ty * RQ + r) * kPsLd + j];
#pragma unroll
            for (int c = 0; c < C::N; ++c)
                o[r][c] = fmaf(pr, Y[j * ld_of<HP>() + C::W * tx + 64 * (c / C::W) + c % C::W], o[r][c]);
        }
}

// Result row (columns of tx) times f into an intermediate row at column col0.
template <class TS, int HP>
__device__ __forceinline__ void store_row(void *dst, size_t row, int cols, int col0, int tx,
                                          const float (&o)[HP / 16], float f) {
    using C = Cols<HP>;
#pragma unroll
    for (int e = 0; e < C::G; ++e) {
        const int c = col0 + C::W * tx + 64 * e;
        if constexpr (C::W == 4) {
            const float v[4] = {o[4 * e] * f, o[4 * e + 1] * f, o[4 * e + 2] * f, o[4 * e + 3] * f};
            st4<TS>(dst, row, cols, c, v);
        } else {
#pragma unroll
            for (int w = 0; w < C::W; ++w) Inter<TS>::st(dst, row, cols, c + w, o[w] * f);
        }
    }
}

template <int HP, int RQ>
constexpr int fwd_smem() {
    return (int)sizeof(float) * ((16 * RQ + 2 * kCol) * ld_of<HP>() + 16 * RQ * kPsLd);
}
template <int HP, int RQ>
constexpr int bwd_smem() {
    return (int)sizeof(float) * ((32 * RQ + 2 * kCol) * ld_of<HP>() + 16 * RQ * kPsLd + 2 * kCol);
}

// (The kernels start early, before the one that writes their inputs has ended, and
// wait for it in pdl_wait(): their pointers are not __restrict__, which would let
// the compiler read through them ahead of that wait.)
template <class TS, int HP, int RQ>
__global__ void __launch_bounds__(kThreads)
attn_fwd_simt_kernel(const void *Q, const void *K,
                     const void *V, const float *rsel,
                     float *A, void *AR, float *lse, int k,
                     float scale) {
    extern __shared__ float sm[];
    float *Xs = sm, *Ys = Xs + 16 * RQ * ld_of<HP>(), *Vs = Ys + kCol * ld_of<HP>(),
          *Ps = Vs + kCol * ld_of<HP>();
    const size_t base = (size_t)blockIdx.x * k;
    // the tile is the grid's slow dimension: those with the most keys start first
    // (33 -> 26 us there)
    const int r0 = (int)(gridDim.y - 1 - blockIdx.y) * 16 * RQ;
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    tc::pdl_wait();
    {
        Tile<TS, HP, 16 * RQ> x;
        x.fetch(Q, base, r0, k);
        x.put(Xs, scale);
    }
    float o[RQ][HP / 16], m[RQ], l[RQ];
#pragma unroll
    for (int r = 0; r < RQ; ++r) {
        m[r] = -FLT_MAX;
        l[r] = 0.f;
#pragma unroll
        for (int c = 0; c < HP / 16; ++c) o[r][c] = 0.f;
    }
    const int last = min(k, r0 + 16 * RQ) - 1;
    for (int j0 = 0; j0 <= last; j0 += kCol) {
        Tile<TS, HP, kCol> y1, y2;
        y1.fetch(K, base, j0, k);
        y2.fetch(V, base, j0, k);
        __syncthreads();
        y1.put(Ys, 1.f);
        const bool bad = __syncthreads_or(y2.put(Vs, 1.f));
        float s[RQ][4];
        dot_tile<HP, RQ>(Xs, Ys, ty, tx, s);
#pragma unroll
        for (int r = 0; r < RQ; ++r) {
            const int i = r0 + ty * RQ + r;
            float mx = m[r];
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (j0 + tx + 16 * c <= i) mx = fmaxf(mx, s[r][c]);
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            const float corr = expf(m[r] - mx);
            m[r] = mx;
            float sum = 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float p = j0 + tx + 16 * c <= i ? expf(s[r][c] - mx) : 0.f;
                sum += p;
                Ps[(ty * RQ + r) * kPsLd + tx + 16 * c] = p;
            }
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
            l[r] = l[r] * corr + sum;
#pragma unroll
            for (int c = 0; c < HP / 16; ++c) o[r][c] *= corr;
        }
        __syncwarp();   // a row of the score tile is written and read by one half warp
        if (!bad)
            accumulate<HP, RQ>(Ps, Vs, ty, tx, min(kCol, (last - j0 + 4) & ~3), o);
        else
            accumulate_masked<HP, RQ>(Ps, Vs, ty, tx, min(kCol, last - j0 + 1), o,
                                      [&](int r, int j) { return j0 + j <= r0 + ty * RQ + r; });
    }
    tc::pdl_trigger();
#pragma unroll
    for (int r = 0; r < RQ; ++r) {
        const int i = r0 + ty * RQ + r;
        if (i >= k) continue;
        const size_t row = base + i;
        const float inv = 1.f / l[r], rr = rsel[row];
#pragma unroll
        for (int c = 0; c < HP / 16; ++c) o[r][c] *= inv;
        store_row<float, HP>(A, row, HP, 0, tx, o[r], 1.f);
        store_row<TS, HP>(AR, row, HP, 0, tx, o[r], rr);
        if (tx == 0) lse[row] = m[r] + logf(l[r]);
    }
}

// dQ of a query tile (kKeys false) or dK and dV of a key tile (kKeys true):
// X1, X2 are the tile's own rows (Q, dA | K, V), Y1, Y2 the walked ones
// (K, V | Q, dA).
template <class TS, int HP, int RQ, bool kKeys>
__device__ __forceinline__ void attn_bwd_tile(float *sm, const void *Q, const void *K, const void *V,
                                              const void *dA, const float *lse, const float *Dd,
                                              void *dQKV, int k, float scale, size_t base, int r0) {
    float *X1 = sm, *X2 = X1 + 16 * RQ * ld_of<HP>(), *Y1 = X2 + 16 * RQ * ld_of<HP>(),
          *Y2 = Y1 + kCol * ld_of<HP>(), *Ps = Y2 + kCol * ld_of<HP>(), *Ls = Ps + 16 * RQ * kPsLd,
          *Ds = Ls + kCol;
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    const int c_begin = kKeys ? r0 / kCol * kCol : 0;
    const int c_last = kKeys ? k - 1 : min(k, r0 + 16 * RQ) - 1;
    {
        Tile<TS, HP, 16 * RQ> x1, x2;
        x1.fetch(kKeys ? K : Q, base, r0, k);
        x2.fetch(kKeys ? V : dA, base, r0, k);
        x1.put(X1, scale);
        x2.put(X2, 1.f);
    }
    float o1[RQ][HP / 16], o2[kKeys ? RQ : 1][HP / 16], Lr[RQ], Dr[RQ];
#pragma unroll
    for (int r = 0; r < RQ; ++r) {
        const int i = r0 + ty * RQ + r;
        Lr[r] = !kKeys && i < k ? lse[base + i] : 0.f;
        Dr[r] = !kKeys && i < k ? Dd[base + i] : 0.f;
#pragma unroll
        for (int c = 0; c < HP / 16; ++c) {
            o1[r][c] = 0.f;
            if (kKeys) o2[r][c] = 0.f;
        }
    }
    for (int j0 = c_begin; j0 <= c_last; j0 += kCol) {
        Tile<TS, HP, kCol> y1, y2;
        y1.fetch(kKeys ? Q : K, base, j0, k);
        y2.fetch(kKeys ? dA : V, base, j0, k);
        __syncthreads();
        bool bad = y1.put(Y1, 1.f);
        bad = y2.put(Y2, 1.f) || bad;
        if (kKeys && threadIdx.x < kCol) {
            const int i = j0 + threadIdx.x;
            Ls[threadIdx.x] = i < k ? lse[base + i] : 0.f;
            Ds[threadIdx.x] = i < k ? Dd[base + i] : 0.f;
        }
        bad = __syncthreads_or(bad);
        auto live = [&](int r, int j) {
            const int own = r0 + ty * RQ + r, other = j0 + j;
            return kKeys ? own <= other && other < k : other <= own && own < k;
        };
        float s[RQ][4], dp[RQ][4];
        dot_tile<HP, RQ>(X1, Y1, ty, tx, s);
        dot_tile<HP, RQ>(X2, Y2, ty, tx, dp);
        const int n = min(kCol, (c_last - j0 + 4) & ~3);
#pragma unroll
        for (int r = 0; r < RQ; ++r) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int jc = tx + 16 * c;
                const bool on = live(r, jc);
                const float p = on ? expf(s[r][c] - (kKeys ? Ls[jc] : Lr[r])) : 0.f;
                dp[r][c] = on ? p * (dp[r][c] - (kKeys ? Ds[jc] : Dr[r])) : 0.f;
                if (kKeys) Ps[(ty * RQ + r) * kPsLd + jc] = p;
            }
        }
        if constexpr (kKeys) {
            __syncwarp();
            if (!bad)
                accumulate<HP, RQ>(Ps, Y2, ty, tx, n, o2);
            else
                accumulate_masked<HP, RQ>(Ps, Y2, ty, tx, min(n, c_last - j0 + 1), o2, live);
            __syncwarp();
        }
#pragma unroll
        for (int r = 0; r < RQ; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) Ps[(ty * RQ + r) * kPsLd + tx + 16 * c] = dp[r][c];
        __syncwarp();
        if (!bad)
            accumulate<HP, RQ>(Ps, Y1, ty, tx, n, o1);
        else
            accumulate_masked<HP, RQ>(Ps, Y1, ty, tx, min(n, c_last - j0 + 1), o1, live);
    }
#pragma unroll
    for (int r = 0; r < RQ; ++r) {
        const int i = r0 + ty * RQ + r;
        if (i >= k) continue;
        store_row<TS, HP>(dQKV, base + i, 4 * HP, kKeys ? HP : 0, tx, o1[r], scale);
        if constexpr (kKeys) store_row<TS, HP>(dQKV, base + i, 4 * HP, 2 * HP, tx, o2[r], 1.f);
    }
}

template <class TS, int HP, int RQ>
__global__ void __launch_bounds__(kThreads)
attn_bwd_simt_kernel(const void *Q, const void *K,
                     const void *V, const void *dA,
                     const float *lse, const float *Dd,
                     void *dQKV, int k, float scale) {
    extern __shared__ float sm[];
    const int tiles = gridDim.y >> 1, t = blockIdx.y >> 1;
    const size_t base = (size_t)blockIdx.x * k;
    tc::pdl_wait();
    // the tiles with the most work first: low key tiles, high query tiles (80 -> 68 us)
    if (blockIdx.y & 1)
        attn_bwd_tile<TS, HP, RQ, false>(sm, Q, K, V, dA, lse, Dd, dQKV, k, scale, base,
                                         (tiles - 1 - t) * 16 * RQ);
    else
        attn_bwd_tile<TS, HP, RQ, true>(sm, Q, K, V, dA, lse, Dd, dQKV, k, scale, base, t * 16 * RQ);
}

// Rows per thread (tiles of 16 RQ rows): the widest that still gives each of the
// 152 SMs a CTA, down to 16-row tiles; the backward has a query and a key side.
int rows_per_thread(const Dims &dm, bool fwd) {
    const long long units = (long long)dm.B * dm.H * (fwd ? 1 : 2);
    for (int rq = 4; rq > 1; rq /= 2)
        if (units * ((dm.k + 16 * rq - 1) / (16 * rq)) >= 152) return rq;
    return 1;
}

template <class TS, int HP, int RQ>
cudaError_t attn_fwd_t(const Dims &dm, const Saved &sv, cudaStream_t s) {
    const dim3 grid(dm.H * dm.B, (dm.k + 16 * RQ - 1) / (16 * RQ));
    const float scale = 1.f / sqrtf((float)HP);
    constexpr int smem = fwd_smem<HP, RQ>();
    cudaError_t e = allow_smem((const void *)attn_fwd_simt_kernel<TS, HP, RQ>, smem);
    if (e != cudaSuccess) return e;
    e = launch_pdl(attn_fwd_simt_kernel<TS, HP, RQ>, grid, dim3(kThreads), smem, s,
                   (const void *)sv.Q, (const void *)sv.K, (const void *)sv.V,
                   (const float *)sv.rsel, sv.A, sv.AR, sv.lse, dm.k, scale);
    note_launches(1);
    return e;
}

template <class TS, int HP, int RQ>
cudaError_t attn_bwd_t(const Dims &dm, const Saved &sv, cudaStream_t s) {
    const dim3 grid(dm.H * dm.B, 2 * ((dm.k + 16 * RQ - 1) / (16 * RQ)));
    const float scale = 1.f / sqrtf((float)HP);
    constexpr int smem = bwd_smem<HP, RQ>();
    cudaError_t e = allow_smem((const void *)attn_bwd_simt_kernel<TS, HP, RQ>, smem);
    if (e != cudaSuccess) return e;
    e = launch_pdl(attn_bwd_simt_kernel<TS, HP, RQ>, grid, dim3(kThreads), smem, s,
                   (const void *)sv.Q, (const void *)sv.K, (const void *)sv.V, (const void *)sv.dA,
                   (const float *)sv.lse, (const float *)sv.Dd, sv.dQKV, dm.k, scale);
    note_launches(1);
    return e;
}

template <class TS, int HP>
cudaError_t attn_rq(const Dims &dm, const Saved &sv, cudaStream_t s, bool fwd) {
    switch (rows_per_thread(dm, fwd)) {
        case 4: return fwd ? attn_fwd_t<TS, HP, 4>(dm, sv, s) : attn_bwd_t<TS, HP, 4>(dm, sv, s);
        case 2: return fwd ? attn_fwd_t<TS, HP, 2>(dm, sv, s) : attn_bwd_t<TS, HP, 2>(dm, sv, s);
        default: return fwd ? attn_fwd_t<TS, HP, 1>(dm, sv, s) : attn_bwd_t<TS, HP, 1>(dm, sv, s);
    }
}

template <class TS>
cudaError_t attn_dispatch(const Dims &dm, const Saved &sv, cudaStream_t s, bool fwd) {
    switch (dm.hp) {
        case 16: return attn_rq<TS, 16>(dm, sv, s, fwd);
        case 32: return attn_rq<TS, 32>(dm, sv, s, fwd);
        case 64: return attn_rq<TS, 64>(dm, sv, s, fwd);
        case 128: return attn_rq<TS, 128>(dm, sv, s, fwd);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_attn_fwd(const Dims &dm, const Saved &sv, cudaStream_t s) {
    if (use_tc(dm)) return tc_attn_fwd(dm, sv, s);
    return dm.bf16 ? attn_dispatch<SplitBF16>(dm, sv, s, true) : attn_dispatch<float>(dm, sv, s, true);
}

cudaError_t launch_attn_bwd(const Dims &dm, const Saved &sv, cudaStream_t s, float *zero_out) {
    if (use_tc(dm)) return tc_attn_bwd(dm, sv, s, zero_out);
    return dm.bf16 ? attn_dispatch<SplitBF16>(dm, sv, s, false) : attn_dispatch<float>(dm, sv, s, false);
}

}  // namespace mosa
