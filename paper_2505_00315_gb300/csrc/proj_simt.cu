// Per-head projections of the MoSA layer for fp32 storage and for bf16 with a
// head size other than 64 (and, with MOSA_FORCE_SIMT, for every shape):
//   F3  Q, K, V = X^s W^{Q,K,V}           (X^s = X[b, I, :], Sec. 2.2)
//   F5  Y[b, I, :] += diag(r^topk) A W^o  (scatter-sum over heads, Eq. mosa_mha)
//   B1  G = dY[I] W^o^T, dW^o = (diag(r) A)^T dY[I], and the row terms
//       dr = <A, G>, dA = r G, dlogit = dr r (1 - r), D = rowsum(dA o A)
//   B3  dX[b, I, :] += dQ W^Q^T + dK W^K^T + dV W^V^T + dlogit W^r[:,h]^T
//   B4  dW^{Q,K,V} = X^s^T d{Q,K,V},  dW^r[:,h] = X^s^T dlogit
// Rows of head h are m = b*k + i; gidx maps them to rows of X / Y / dY.  Each
// product is described once (an Op) and runs on the tensor cores through bf16
// planes (tc_split.cuh), or on the CUDA cores (simt_gemm.cuh) when forced or
// when a tensor's address is not 16-byte aligned.
// dQ|dK|dV rows have 4 h' columns: 3 h' of gradients, then dlogit (bf16: its
// pair at column 3 h' and the pair of what that rounded off at 3 h' + 1).
#include <algorithm>
#include <cstdlib>
#include <initializer_list>
#include <type_traits>

#include "launch.h"
#include "simt_gemm.cuh"
#include "tc_split.cuh"

namespace mosa {
namespace {

// Planes of an input tensor and of a stored intermediate of storage type T.
template <class T>
constexpr int in_planes() { return sizeof(T) == 4 ? 3 : 1; }
template <class T>
constexpr int inter_planes() { return sizeof(T) == 4 ? 3 : 2; }
// Elements per stored intermediate row of `cols` columns.
template <class T>
constexpr int inter_ld(int cols) { return sizeof(T) == 4 ? cols : 2 * cols; }

// Four consecutive columns of an intermediate row (Inter<TS>::st of each).
template <class T>
__device__ __forceinline__ void st_inter4(void *p, size_t row, int cols, int c, const float4 &v) {
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(static_cast<float *>(p) + row * cols + c) = v;
    } else {
        const float x[4] = {v.x, v.y, v.z, v.w};
        __nv_bfloat162 hi[2], lo[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const bf16 h0 = __float2bfloat16_rn(x[2 * e]), h1 = __float2bfloat16_rn(x[2 * e + 1]);
            hi[e] = __halves2bfloat162(h0, h1);
            lo[e] = __halves2bfloat162(__float2bfloat16_rn(x[2 * e] - __bfloat162float(h0)),
                                       __float2bfloat16_rn(x[2 * e + 1] - __bfloat162float(h1)));
        }
        bf16 *q = static_cast<bf16 *>(p) + row * 2 * cols + c;
        *reinterpret_cast<uint2 *>(q) = *reinterpret_cast<const uint2 *>(hi);
        *reinterpret_cast<uint2 *>(q + cols) = *reinterpret_cast<const uint2 *>(lo);
    }
}

// Weight gradients in reduction splits: split 0 (or the only one) goes to the output,
// split j to the j-th array of partial sums, laid out as the outputs one after the
// other; sum_splits_kernel adds them up, so that each gradient stays one fixed sum.
// (Added to the outputs as they came, more than two splits gave other last bits from
// call to call, and their zeroing took longer than this: fp32 steps of B4 T1000 d768 H12 k125
// 208.7 -> 202.4 us, B2 T2048 d256 H4 k512 240 -> 226.)
struct Parts {
    float *part;
    size_t stride;   // of one split's partial sums
    // where split sp puts element i of the output that starts `before` elements into the layout
    __device__ __forceinline__ float *at(float *out, size_t before, size_t i, int sp) const {
        return sp <= 0 ? out + i : part + (size_t)(sp - 1) * stride + before + i;
    }
};

template <class T>
struct QkvOp {
    using TS = typename InterOf<T>::type;
    using TA = T;
    using TB = T;
    static constexpr bool kAKFast = true, kBKFast = false;
    static constexpr int kPA = in_planes<T>(), kPB = in_planes<T>();
    static constexpr bool kAMN = false, kBMN = true, kTrans = false;
    int M, N, K;  // B*k, 3*hp, d
    int hp, lg;   // lg: log2 hp
    const T *A;   // X
    const T *Wq, *Wk, *Wv;
    const int32_t *gidx;
    void *Q, *Kp, *V;
    int lda = 0, a_lo = 0, ldb = 0, b_lo = 0;
    __device__ int a_row(int g, int m) const { return gidx[(size_t)g * M + m]; }
    __device__ const T *b_ptr(int g, int c, int n) const {
        const int w = n >> lg, p = n & (hp - 1);
        return (w == 0 ? Wq : (w == 1 ? Wk : Wv)) + ((size_t)g * K + c) * hp + p;
    }
    __device__ float a(int g, int m, int c) const { return to_f32(A[(size_t)a_row(g, m) * K + c]); }
    __device__ float b(int g, int c, int n) const { return to_f32(*b_ptr(g, c, n)); }
    __device__ void store(int g, int m, int n, float v, int) const {
        const int w = n >> lg, p = n & (hp - 1);
        Inter<TS>::st(w == 0 ? Q : (w == 1 ? Kp : V), (size_t)g * M + m, hp, p, v);
    }
    __device__ void store4(int g, int m, int n, const float4 &v, int) const {
        const int w = n >> lg, p = n & (hp - 1);
        st_inter4<T>(w == 0 ? Q : (w == 1 ? Kp : V), (size_t)g * M + m, hp, p, v);
    }
};

template <class T>
struct OutOp {
    using TS = typename InterOf<T>::type;
    using TA = T;
    using TB = T;
    static constexpr bool kAKFast = true, kBKFast = false;
    static constexpr int kPA = inter_planes<T>(), kPB = in_planes<T>();
    static constexpr bool kAMN = false, kBMN = true, kTrans = false;
    int M, N, K;  // B*k, d, hp
    const T *A;   // AR rows
    const T *Wo;
    const int32_t *gidx;
    float *Y;
    int lda = 0, a_lo = 0, ldb = 0, b_lo = 0;
    __device__ int a_row(int g, int m) const { return g * M + m; }
    __device__ const T *b_ptr(int g, int p, int n) const { return Wo + ((size_t)g * K + p) * N + n; }
    __device__ float a(int g, int m, int p) const { return Inter<TS>::ld(A, (size_t)g * M + m, K, p); }
    __device__ float b(int g, int p, int n) const { return to_f32(*b_ptr(g, p, n)); }
    __device__ void store(int g, int m, int n, float v, int) const {
        atomicAdd(Y + (size_t)gidx[(size_t)g * M + m] * N + n, v);
    }
    __device__ void store4(int g, int m, int n, const float4 &v, int) const {
        tc::red_add_v4(Y + (size_t)gidx[(size_t)g * M + m] * N + n, v.x, v.y, v.z, v.w);
    }
};

// G's reduction splits: split 0 (or the only one) goes to G, split j to the j-th h'
// columns of the rows of dQ|dK|dV (4 h' fp32 columns), which the attention backward
// writes later; out_bwd_rows_kernel adds them up, so G stays one fixed sum.
constexpr int kGSplits = 5;
__device__ __forceinline__ float *g_part(float *G, void *dQKV, size_t row, int hp, int sp) {
    return sp <= 0 ? G + row * hp : static_cast<float *>(dQKV) + row * 4 * hp + (sp - 1) * hp;
}

template <class T>
struct OutBwdGOp {
    using TA = T;
    using TB = T;
    static constexpr bool kAKFast = true, kBKFast = true;
    static constexpr int kPA = in_planes<T>(), kPB = in_planes<T>();
    static constexpr bool kAMN = false, kBMN = false, kTrans = false;
    int M, N, K;  // B*k, hp, d
    const T *A;   // dY
    const T *Wo;
    const int32_t *gidx;
    float *G;
    void *dQKV;
    int lda = 0, a_lo = 0, ldb = 0, b_lo = 0;
    __device__ int a_row(int g, int m) const { return gidx[(size_t)g * M + m]; }
    __device__ const T *b_ptr(int g, int n, int c) const { return Wo + ((size_t)g * N + n) * K + c; }
    __device__ float a(int g, int m, int c) const { return to_f32(A[(size_t)a_row(g, m) * K + c]); }
    __device__ float b(int g, int c, int n) const { return to_f32(*b_ptr(g, n, c)); }
    __device__ float *row(int g, int m, int sp) const {
        return g_part(G, dQKV, (size_t)g * M + m, N, sp);
    }
    __device__ void store(int g, int m, int n, float v, int sp) const { row(g, m, sp)[n] = v; }
    __device__ void store4(int g, int m, int n, const float4 &v, int sp) const {
        *reinterpret_cast<float4 *>(row(g, m, sp) + n) = v;
    }
};

// dW_o[h](p, c): rows c of d, columns p, reduced over the head's rows.
template <class T>
struct OutBwdWOp {
    using TS = typename InterOf<T>::type;
    using TA = T;
    using TB = T;
    static constexpr bool kAKFast = false, kBKFast = false;
    static constexpr int kPA = in_planes<T>(), kPB = inter_planes<T>();
    static constexpr bool kAMN = true, kBMN = true, kTrans = true;
    int M, N, K;  // d, hp, B*k
    const T *A;   // dY
    const T *AR;
    const int32_t *gidx;
    float *dWo;
    Parts parts;
    int lda = 0, a_lo = 0, ldb = 0, b_lo = 0;
    __device__ int a_row(int g, int m) const { return gidx[(size_t)g * K + m]; }
    __device__ const T *b_ptr(int g, int m, int p) const {
        return AR + ((size_t)g * K + m) * inter_ld<T>(N) + p;
    }
    __device__ float a(int g, int c, int m) const { return to_f32(A[(size_t)a_row(g, m) * M + c]); }
    __device__ float b(int g, int m, int p) const { return Inter<TS>::ld(AR, (size_t)g * K + m, N, p); }
    __device__ void store(int g, int c, int p, float v, int sp) const {
        *parts.at(dWo, 0, ((size_t)g * N + p) * M + c, sp) = v;
    }
    __device__ void store4(int, int, int, const float4 &, int) const {}
};

template <class T>
struct InBwdOp {
    using TS = typename InterOf<T>::type;
    using TA = T;
    using TB = T;
    static constexpr bool kAKFast = true, kBKFast = true;
    static constexpr int kPA = inter_planes<T>(), kPB = in_planes<T>();
    static constexpr bool kAMN = false, kBMN = false, kTrans = false;
    int M, N, K;  // B*k, d, 3*hp
    int hp, lg, H;   // lg: log2 hp
    const T *A;   // dQ|dK|dV rows
    const T *Wq, *Wk, *Wv, *Wr;
    const float *dlogit;
    const int32_t *gidx;
    float *dX;
    int lda = 0, a_lo = 0, ldb = 0, b_lo = 0;
    __device__ int a_row(int g, int m) const { return g * M + m; }
    __device__ const T *b_ptr(int g, int n, int kk) const {
        const int w = kk >> lg, p = kk & (hp - 1);
        return (w == 0 ? Wq : (w == 1 ? Wk : Wv)) + ((size_t)g * N + n) * hp + p;
    }
    __device__ float a(int g, int m, int kk) const { return Inter<TS>::ld(A, (size_t)g * M + m, 4 * hp, kk); }
    __device__ float b(int g, int kk, int n) const { return to_f32(*b_ptr(g, n, kk)); }
    __device__ void store(int g, int m, int n, float v, int) const {
        const size_t row = (size_t)g * M + m;
        v = fmaf(dlogit[row], to_f32(Wr[(size_t)n * H + g]), v);
        atomicAdd(dX + (size_t)gidx[row] * N + n, v);
    }
    __device__ void store4(int g, int m, int n, const float4 &v, int) const {
        const size_t row = (size_t)g * M + m;
        const float dl = dlogit[row];
        const T *w = Wr + (size_t)n * H + g;
        tc::red_add_v4(dX + (size_t)gidx[row] * N + n, fmaf(dl, to_f32(w[0]), v.x),
                       fmaf(dl, to_f32(w[H]), v.y), fmaf(dl, to_f32(w[2 * (size_t)H]), v.z),
                       fmaf(dl, to_f32(w[3 * (size_t)H]), v.w));
    }
};

// dW_{q,k,v} and, from the dlogit columns of the rows, dW_r.
template <class T>
struct WBwdOp {
    using TS = typename InterOf<T>::type;
    using TA = T;
    using TB = T;
    static constexpr bool kAKFast = false, kBKFast = false;
    static constexpr int kPA = in_planes<T>(), kPB = inter_planes<T>();
    static constexpr bool kAMN = true, kBMN = true, kTrans = false;
    static constexpr int kExtra = sizeof(T) == 4 ? 1 : 2;   // dlogit columns
    int M, N, K;  // d, 3*hp + kExtra, B*k
    int hp, lg, H;   // lg: log2 hp
    const T *A;   // X
    const T *dQKV;
    const float *dlogit;
    const int32_t *gidx;
    float *dWq, *dWk, *dWv, *dWr;
    Parts parts;
    size_t n1;   // elements of dWq (and dWk, dWv)
    int lda = 0, a_lo = 0, ldb = 0, b_lo = 0;
    __device__ int a_row(int g, int m) const { return gidx[(size_t)g * K + m]; }
    __device__ const T *b_ptr(int g, int m, int n) const {
        return dQKV + ((size_t)g * K + m) * inter_ld<T>(4 * hp) + n;
    }
    __device__ float a(int g, int c, int m) const { return to_f32(A[(size_t)a_row(g, m) * M + c]); }
    __device__ float b(int g, int m, int n) const {
        const size_t row = (size_t)g * K + m;
        if (n > 3 * hp) return 0.f;   // (dlogit's rounding remainder, in its fp32 value already)
        return n < 3 * hp ? Inter<TS>::ld(dQKV, row, 4 * hp, n) : dlogit[row];
    }
    __device__ float *dst(int g, int c, int n, int sp) const {
        if (n >= 3 * hp) return parts.at(dWr, 3 * n1, (size_t)c * H + g, sp);
        const int w = n >> lg, p = n & (hp - 1);
        return parts.at(w == 0 ? dWq : (w == 1 ? dWk : dWv), w * n1, ((size_t)g * M + c) * hp + p, sp);
    }
    __device__ void store(int g, int c, int n, float v, int sp) const {
        float *p = dst(g, c, n, sp);
        if (n <= 3 * hp)
            *p = v;
        else if (v != 0.f)   // dlogit's second column, after the first by the same thread
            *p += v;
    }
    __device__ void store4(int g, int c, int n, const float4 &v, int sp) const {
        float *p = dst(g, c, n, sp);
        if (n < 3 * hp)
            *reinterpret_cast<float4 *>(p) = v;
        else
            *p = kExtra == 2 ? v.x + v.y : v.x;
    }
};

// One warp per selected row: dr = <A, G>, dA = r G (rounded to storage),
// D = rowsum(dA o A), dlogit = dr r (1 - r).
// (Pointers without __restrict__: see attn_fwd_simt_kernel.)
template <class TS>
__global__ void out_bwd_rows_kernel(float *G, const float *A,
                                    const float *rsel, void *dA,
                                    float *Dd, float *dlogit,
                                    void *dQKV, long long rows, int hp, int splits) {
    tc::pdl_wait();
    const long long row = (long long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    const int lane = threadIdx.x & 31;
    if (row >= rows) return;
    const float r = rsel[row];
    float dr = 0.f, dd = 0.f;
    for (int p = lane; p < hp; p += 32) {
        float g = G[row * hp + p];
        for (int j = 1; j < splits; ++j) g += g_part(G, dQKV, row, hp, j)[p];
        const float a = A[row * hp + p];
        dr = fmaf(a, g, dr);
        const float da = r * g;
        Inter<TS>::st(dA, row, hp, p, da);
        dd = fmaf(da, a, dd);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        dr += __shfl_xor_sync(0xffffffffu, dr, off);
        dd += __shfl_xor_sync(0xffffffffu, dd, off);
    }
    if (lane == 0) {
        const float dl = dr * r * (1.f - r);
        Dd[row] = dd;
        dlogit[row] = dl;
        if constexpr (std::is_same<TS, float>::value) {
            static_cast<float *>(dQKV)[row * 4 * hp + 3 * hp] = dl;
        } else {
            // three bf16 parts (a non-finite value only in the first), and zeros in the rest of
            // the eight columns that the dW product loads
            bf16 *q = static_cast<bf16 *>(dQKV) + row * 8 * hp + 3 * hp;
            const bf16 h = __float2bfloat16_rn(dl);
            const float r1 = fabsf(dl) <= 3.38e38f ? dl - __bfloat162float(h) : 0.f;
            const bf16 l = __float2bfloat16_rn(r1);
            const __nv_bfloat162 hi = __halves2bfloat162(h, __float2bfloat16_rn(r1 - __bfloat162float(l)));
            *reinterpret_cast<uint4 *>(q) = make_uint4(*reinterpret_cast<const uint32_t *>(&hi), 0u, 0u, 0u);
            *reinterpret_cast<uint4 *>(q + 4 * hp) = make_uint4(__bfloat16_as_ushort(l), 0u, 0u, 0u);
        }
    }
}

// Adds the partial sums of `parts` splits, each n[0] + .. + n[3] values, to out[0] .. out[3].
struct SumSplits {
    float *out[4];
    size_t n[4];
};
__global__ void sum_splits_kernel(const SumSplits o, const float *part, size_t stride, int parts) {
    tc::pdl_wait();
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= stride) return;
    int a = 0;
    size_t at = i;
    while (at >= o.n[a]) at -= o.n[a++];
    float v = o.out[a][at];
#pragma unroll 8
    for (int j = 0; j < parts; ++j) v += part[(size_t)j * stride + i];
    o.out[a][at] = v;
}

bool aligned16(std::initializer_list<const void *> ps) {
    uintptr_t u = 0;
    for (const void *p : ps) u |= reinterpret_cast<uintptr_t>(p);
    return (u & 15) == 0;
}

// One product on the tensor cores (split), or on the CUDA cores.
template <class Op>
cudaError_t product(const Op &op, int groups, int splits, bool split, const Saved &sv,
                    cudaStream_t s) {
    return split ? launch_split_gemm(op, groups, splits, sv.status, s)
                 : launch_simt_gemm(op, groups, s);
}

int log2_of(int hp) {   // 16, 32, 64 or 128
    return hp == 16 ? 4 : hp == 32 ? 5 : hp == 64 ? 6 : 7;
}

cudaError_t zero(float *p, size_t n, cudaStream_t s) {
    return cudaMemsetAsync(p, 0, sizeof(float) * n, s);
}

// Reduction splits of dW_o and of dW_q|dW_k|dW_v|dW_r, and the values of one split's
// partial sums.
int dwo_splits(const Dims &dm) { return split_count(dm.d, dm.hp, dm.B * dm.k, dm.H); }
int dw_splits(const Dims &dm) {
    return split_count(dm.d, 3 * dm.hp + (dm.bf16 ? 2 : 1), dm.B * dm.k, dm.H);
}
size_t dwo_floats(const Dims &dm) { return (size_t)dm.H * dm.hp * dm.d; }
size_t dw_floats(const Dims &dm) { return 3 * dwo_floats(dm) + (size_t)dm.d * dm.H; }

cudaError_t sum_splits(const SumSplits &o, const Saved &sv, size_t stride, int splits, cudaStream_t s) {
    if (splits <= 1) return cudaSuccess;
    const cudaError_t e = launch_pdl(sum_splits_kernel, dim3((unsigned)((stride + 255) / 256)), dim3(256),
                                     0, s, o, (const float *)sv.wpart, stride, splits - 1);
    note_launches(1);
    return e;
}

template <class T>
cudaError_t qkv_t(const Dims &dm, const void *X, const void *Wq, const void *Wk, const void *Wv,
                  const Saved &sv, cudaStream_t s) {
    QkvOp<T> op{dm.B * dm.k, 3 * dm.hp, dm.d, dm.hp, log2_of(dm.hp), (const T *)X, (const T *)Wq, (const T *)Wk,
                (const T *)Wv, sv.gidx, sv.Q, sv.K, sv.V};
    op.lda = dm.d;
    op.ldb = dm.hp;
    return product(op, dm.H, 1, use_split() && aligned16({X, Wq, Wk, Wv}), sv, s);
}

template <class T>
cudaError_t out_t(const Dims &dm, const void *Wo, const Saved &sv, float *Y, cudaStream_t s) {
    if (!dm.accumulate) {
        const cudaError_t e = zero(Y, (size_t)dm.B * dm.T * dm.d, s);
        if (e != cudaSuccess) return e;
    }
    OutOp<T> op{dm.B * dm.k, dm.d, dm.hp, (const T *)sv.AR, (const T *)Wo, sv.gidx, Y};
    op.lda = inter_ld<T>(dm.hp);
    op.a_lo = dm.hp;
    op.ldb = dm.d;
    return product(op, dm.H, 1, use_split() && aligned16({Wo, Y}), sv, s);
}

// G has one column tile per 128 rows: as many reduction splits as the 152 SMs have
// room for, each of at least three K blocks (the last may find fewer left, none is empty).
// fp32 at B4 T1000 d768 H12 k125, 48 tiles: 28 -> 15 us on 144 CTAs, its step 225 -> 210.
// bf16 storage, whose K blocks are only copied, keeps one: at B4 T1024 d1024 H16 h'=128
// k128, 64 tiles, two splits took 17 -> 13 us here and the step 285.6 -> 286.5.  (At 4 to 48 tiles
// splits left six steps within 1% and took 203 -> 199 us off one, B2 T1024 d1024 H12 h'=128 k128, and
// 110.7 -> 105.4 off another, B2 T512 d1024 H16 h'=32 k64: not used yet.)
int g_split_count(int M, int N, int K, int groups) {
    const int tiles = (M + 127) / 128 * ((N + 127) / 128) * groups, nkb = (K + 63) / 64;
    const int sp = std::max(1, std::min({kGSplits, 152 / tiles, nkb / 3}));
    const int per = (nkb + sp - 1) / sp;
    return (nkb + per - 1) / per;
}

template <class T>
cudaError_t out_bwd_t(const Dims &dm, const void *Wo, const void *dY, const Saved &sv,
                      float *dWo, cudaStream_t s) {
    using TS = typename InterOf<T>::type;
    const bool split = use_split() && aligned16({Wo, dY, dWo});
    const int Mtok = dm.B * dm.k;
    OutBwdGOp<T> g{Mtok, dm.hp, dm.d, (const T *)dY, (const T *)Wo, sv.gidx, sv.G, sv.dQKV};
    g.lda = dm.d;
    g.ldb = dm.d;
    const int gsplits = split && sizeof(T) == 4 ? g_split_count(Mtok, dm.hp, dm.d, dm.H) : 1;
    cudaError_t e = product(g, dm.H, gsplits, split, sv, s);
    if (e != cudaSuccess) return e;
    const long long rows = dm.rows();
    const int warps = 8;
    e = launch_pdl(out_bwd_rows_kernel<TS>, dim3((unsigned)((rows + warps - 1) / warps)),
                   dim3(warps * 32), 0, s, sv.G, (const float *)sv.A,
                   (const float *)sv.rsel, sv.dA, sv.Dd, sv.dlogit, sv.dQKV, rows, dm.hp, gsplits);
    note_launches(1);
    if (e != cudaSuccess) return e;
    const int splits = split ? dwo_splits(dm) : 1;
    const size_t n = dwo_floats(dm);
    OutBwdWOp<T> w{dm.d, dm.hp, Mtok, (const T *)dY, (const T *)sv.AR, sv.gidx, dWo, {sv.wpart, n}};
    w.lda = dm.d;
    w.ldb = inter_ld<T>(dm.hp);
    w.b_lo = dm.hp;
    if ((e = product(w, dm.H, splits, split, sv, s)) != cudaSuccess) return e;
    return sum_splits({{dWo}, {n}}, sv, n, splits, s);
}

template <class T>
cudaError_t in_bwd_t(const Dims &dm, const void *Wq, const void *Wk, const void *Wv,
                     const void *Wr, const Saved &sv, float *dX, cudaStream_t s) {
    if (!dm.accumulate) {
        const cudaError_t e = zero(dX, (size_t)dm.B * dm.T * dm.d, s);
        if (e != cudaSuccess) return e;
    }
    InBwdOp<T> op{dm.B * dm.k, dm.d, 3 * dm.hp, dm.hp, log2_of(dm.hp), dm.H, (const T *)sv.dQKV, (const T *)Wq,
                  (const T *)Wk, (const T *)Wv, (const T *)Wr, sv.dlogit, sv.gidx, dX};
    op.lda = inter_ld<T>(4 * dm.hp);
    op.a_lo = 4 * dm.hp;
    op.ldb = dm.hp;
    return product(op, dm.H, 1, use_split() && aligned16({Wq, Wk, Wv, dX}), sv, s);
}

template <class T>
cudaError_t w_bwd_t(const Dims &dm, const void *X, const Saved &sv, float *dWq, float *dWk,
                    float *dWv, float *dWr, cudaStream_t s) {
    const bool split = use_split() && aligned16({X, dWq, dWk, dWv});
    const int N = 3 * dm.hp + WBwdOp<T>::kExtra, Mtok = dm.B * dm.k;
    const int splits = split ? dw_splits(dm) : 1;
    const size_t n = dwo_floats(dm), stride = dw_floats(dm);
    WBwdOp<T> op{dm.d, N, Mtok, dm.hp, log2_of(dm.hp), dm.H, (const T *)X, (const T *)sv.dQKV, sv.dlogit, sv.gidx,
                 dWq, dWk, dWv, dWr, {sv.wpart, stride}, n};
    op.lda = dm.d;
    op.ldb = inter_ld<T>(4 * dm.hp);
    op.b_lo = 4 * dm.hp;
    const cudaError_t e = product(op, dm.H, splits, split, sv, s);
    if (e != cudaSuccess) return e;
    return sum_splits({{dWq, dWk, dWv, dWr}, {n, n, n, (size_t)dm.d * dm.H}}, sv, stride, splits, s);
}

}  // namespace

size_t split_part_floats(const Dims &dm) {
    return std::max((dwo_splits(dm) - 1) * dwo_floats(dm), (dw_splits(dm) - 1) * dw_floats(dm));
}

bool use_split() {
    const char *f = std::getenv("MOSA_FORCE_SIMT");
    return f == nullptr || f[0] == '\0' || f[0] == '0';
}

bool use_tc(const Dims &dm) { return use_split() && tc_supported(dm); }

bool use_fused_forward(const Dims &dm) {
    const char *f = std::getenv("MOSA_FUSED_FWD");
    if (f != nullptr && f[0] == '0') return false;
    return use_tc(dm) && tc_fused_forward_supported(dm);
}

cudaError_t launch_qkv(const Dims &dm, const void *X, const void *Wq, const void *Wk,
                       const void *Wv, const Saved &sv, cudaStream_t s) {
    if (use_tc(dm)) return tc_qkv(dm, X, Wq, Wk, Wv, sv, s);
    return dm.bf16 ? qkv_t<bf16>(dm, X, Wq, Wk, Wv, sv, s) : qkv_t<float>(dm, X, Wq, Wk, Wv, sv, s);
}

cudaError_t launch_out(const Dims &dm, const void *Wo, const Saved &sv, float *Y, cudaStream_t s) {
    if (use_tc(dm)) return tc_out(dm, Wo, sv, Y, s, !dm.accumulate);
    return dm.bf16 ? out_t<bf16>(dm, Wo, sv, Y, s) : out_t<float>(dm, Wo, sv, Y, s);
}

cudaError_t launch_out_bwd(const Dims &dm, const void *Wo, const void *dY, const Saved &sv,
                           float *dWo, cudaStream_t s) {
    if (use_tc(dm)) {
        cudaError_t e = tc_out_bwd_g(dm, Wo, dY, sv, s);
        return e != cudaSuccess ? e : tc_out_bwd_w(dm, dY, sv, dWo, s);
    }
    return dm.bf16 ? out_bwd_t<bf16>(dm, Wo, dY, sv, dWo, s) : out_bwd_t<float>(dm, Wo, dY, sv, dWo, s);
}

cudaError_t launch_in_bwd(const Dims &dm, const void *Wq, const void *Wk, const void *Wv,
                          const void *Wr, const Saved &sv, float *dX, cudaStream_t s) {
    if (use_tc(dm)) {
        cudaError_t e = tc_transpose_wr(dm, Wr, sv, s);
        return e != cudaSuccess ? e : tc_in_bwd(dm, Wq, Wk, Wv, Wr, sv, dX, s, !dm.accumulate);
    }
    return dm.bf16 ? in_bwd_t<bf16>(dm, Wq, Wk, Wv, Wr, sv, dX, s)
                   : in_bwd_t<float>(dm, Wq, Wk, Wv, Wr, sv, dX, s);
}

cudaError_t launch_w_bwd(const Dims &dm, const void *X, const Saved &sv, float *dWq, float *dWk,
                         float *dWv, float *dWr, cudaStream_t s) {
    if (use_tc(dm)) return tc_w_bwd(dm, X, sv, dWq, dWk, dWv, dWr, s);
    return dm.bf16 ? w_bwd_t<bf16>(dm, X, sv, dWq, dWk, dWv, dWr, s)
                   : w_bwd_t<float>(dm, X, sv, dWq, dWk, dWv, dWr, s);
}

}  // namespace mosa
