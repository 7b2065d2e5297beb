// Grouped matrix product on the tensor cores (tcgen05.mma kind::f16, bf16
// planes, fp32 accumulation) for the shapes the TMA kernels do not serve: fp32
// storage, and bf16 storage with a head size other than 64.
//
// Every operand element is a sum of bf16 "planes": one for a bf16 input, two
// for a stored bf16 hi/lo pair, three for an fp32 value (its significand cut
// into three 8-bit parts, an exact decomposition: v = p0 + p1 + p2 with
// p_i = the bf16 truncation of what the parts before it left).  The product of
// two operands is the sum of the plane products that matter: 1 (bf16 x bf16),
// 2 (pair x bf16) or, for fp32 x fp32, the six of order up to 2^-16 (p0 q0,
// p0 q1, p1 q0, p1 q1, p0 q2, p2 q0); what is left out is below 2^-23 of each
// product, under the rounding of an fp32 multiply-add chain.  Each plane product
// of a K step is one MMA into the same accumulator, and the accumulator is
// drained into fp32 registers every few K blocks (kDrain), so that the tensor
// pipe's accumulation rounding acts on short partial sums only.
//
// A truncated non-finite fp32 input would turn into NaN (inf - inf) where a
// plain product gives inf, so the converting threads check every value; a CTA
// that met one recomputes its tile with plain fp32 multiply-adds.
//
// One CTA (544 threads) computes a 128 x bn tile (bn <= 128) of one group:
//   warps 0-7    drain: TMEM -> registers (two accumulators in turn), then the
//                fused output step; warp w reads TMEM lanes 32 (w % 4) .. +31
//                and columns 64 (w / 4) .. +63
//   warps 8-15   producers: gathered or plain rows, by 16-byte cp.async
//                (bf16 planes already in memory) or through registers, one K
//                block ahead (fp32, cut into planes), into the 128-byte-
//                swizzled layout
//   warp 16      TMEM allocation and the MMA issuer (one thread)
// What bounds it, fp32: six MMAs of 128 x 128 x 16 per 16-wide K step, about
// 1550 cycles per 64-wide K block, against about 1200 issue cycles for the
// conversion of its 16384 values; the CUDA-core product it replaces needed
// 4096 cycles at the FFMA rate and ran at a tenth of that.
#pragma once

#include "launch.h"
#include "profile.h"
#include "simt_gemm.cuh"
#include "tc_common.cuh"

namespace mosa {

// Contract of an Op (besides simt_gemm.cuh's M, N, K, a, b, store):
//   TA, TB                element types in memory (float or bf16)
//   kPA, kPB              planes of the operands (float: 3; bf16: 1 or 2)
//   kAMN / kBMN           the operand is contiguous along M / N in memory (else along K)
//   kTrans                outputs go out one column at a time with the lanes along M
//   A, lda, a_lo          base, row stride and offset of the second plane (elements)
//   a_row(g, r)           source row of A for strided index r (r < M or r < K)
//   b_ptr(g, r, c)        eight contiguous elements of B: strided index r (k if kBMN,
//                         else n), contiguous index c; linear in r with stride ldb; b_lo as a_lo
//   store(g, m, n, v, add)     one result; add: several reduction splits add up
//   store4(g, m, n, v4, add)   four consecutive columns (not kTrans)
struct SplitArgs {
    int bn;        // tile width, a multiple of 16, <= 128
    int nkb;       // 64-wide K blocks in the whole reduction
    int splits;    // reduction splits
    uint32_t *status;
    unsigned long long *span;
};

constexpr int kSplitThreads = 544;
constexpr int kSplitPlane = 16384;   // one 128 x 64 bf16 plane tile
constexpr int kSplitIdxMax = 2048;   // K rows of one CTA whose indices are staged

template <class Op>
constexpr bool split_f32() { return sizeof(typename Op::TA) == 4; }
template <class Op>
constexpr int split_stages() { return split_f32<Op>() ? 2 : (Op::kPA + Op::kPB == 2 ? 6 : 4); }
// K blocks between drains: at most four 16-wide steps per plane product for
// fp32, sixteen for bf16 inputs
template <class Op>
constexpr int split_drain() { return split_f32<Op>() ? 1 : 4; }
template <class Op>
constexpr int split_smem() {
    return 1024 + split_stages<Op>() * (Op::kPA + Op::kPB) * kSplitPlane + 256 + kSplitIdxMax * 4;
}

// Eight fp32 values as three planes of eight bf16 (16 bytes each); nf collects
// bit 15 / 31 for a non-finite value.
__device__ __forceinline__ void split3(const float4 &x, const float4 &y, uint4 (&pl)[3],
                                       uint32_t &nf) {
    const float v[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
    uint32_t w[3][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float a = v[2 * e], b = v[2 * e + 1];
        const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
        const float ra = a - __uint_as_float(ua & 0xFFFF0000u);
        const float rb = b - __uint_as_float(ub & 0xFFFF0000u);
        const uint32_t va = __float_as_uint(ra), vb = __float_as_uint(rb);
        const float sa = ra - __uint_as_float(va & 0xFFFF0000u);
        const float sb = rb - __uint_as_float(vb & 0xFFFF0000u);
        w[0][e] = __byte_perm(ua, ub, 0x7632);
        w[1][e] = __byte_perm(va, vb, 0x7632);
        w[2][e] = __byte_perm(__float_as_uint(sa), __float_as_uint(sb), 0x7632);
        // an exponent of all ones carries into the sign's place
        nf |= (w[0][e] & 0x7FFF7FFFu) + 0x00800080u;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) pl[i] = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
}

template <class Op>
__global__ void __launch_bounds__(kSplitThreads, 1)
    split_gemm_kernel(const __grid_constant__ Op op, const SplitArgs sa) {
    using namespace tc;
    using TA = typename Op::TA;
    using TB = typename Op::TB;
    constexpr bool kF32 = split_f32<Op>();
    constexpr int S = split_stages<Op>();
    constexpr int kStage = (Op::kPA + Op::kPB) * kSplitPlane;
    constexpr int DR = split_drain<Op>();
    extern __shared__ uint8_t smem_raw[];
    uint8_t *ring = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *bars = reinterpret_cast<uint64_t *>(ring + S * kStage);
    uint64_t *full = bars, *empty = bars + 8, *accf = bars + 16, *acce = bars + 18,
             *mdone = bars + 20;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 21);
    int *s_abort = reinterpret_cast<int *>(tmem_slot + 1);
    int *s_slow = s_abort + 1;
    int *s_row = reinterpret_cast<int *>(reinterpret_cast<uint8_t *>(bars) + 256);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = blockIdx.z / sa.splits, split = blockIdx.z - g * sa.splits;
    const int m0 = blockIdx.y * 128, n0 = blockIdx.x * sa.bn;
    const int per = (sa.nkb + sa.splits - 1) / sa.splits;
    const int kb0 = split * per;
    const int nkb = max(0, min(sa.nkb, kb0 + per) - kb0);
    const int n_end = min(op.N, n0 + sa.bn);

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(smem_u32(&full[s]), 256);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&accf[b]), 1);
            mbar_init(smem_u32(&acce[b]), 256);
        }
        mbar_init(smem_u32(mdone), 1);
        *s_abort = 0;
        *s_slow = 0;
        fence_barrier_init();
    }
    if (warp == 16) {
        tmem_alloc(smem_u32(tmem_slot), 256);
        tmem_relinquish();
    }
    pdl_wait();  // everything below may read what the previous kernel wrote
    span_begin(sa.span);
    if (Op::kAMN) {
        for (int i = threadIdx.x; i < nkb * 64; i += kSplitThreads) {
            const int r = kb0 * 64 + i;
            s_row[i] = r < op.K ? op.a_row(g, r) : -1;
        }
    } else {
        for (int i = threadIdx.x; i < 128; i += kSplitThreads)
            s_row[i] = m0 + i < op.M ? op.a_row(g, m0 + i) : -1;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    auto give_up = [&]() {
        atomicOr(sa.status, kStatusTimeout);
        *(volatile int *)s_abort = 1;
    };

    if (warp >= 8 && warp < 16) {
        // ------------------------------------------------------ producers
        const int t = threadIdx.x - 256;
        // chunk p of this thread: strided row and 16-byte unit of the tile
        const int arow = Op::kAMN ? t >> 4 : t >> 3, ach = Op::kAMN ? t & 15 : t & 7;
        const int brow = Op::kBMN ? t >> 4 : t >> 3, bch = Op::kBMN ? t & 15 : t & 7;
        constexpr int kAStep = Op::kAMN ? 16 : 32, kBStep = Op::kBMN ? 16 : 32;
        auto place = [](bool mn, int row, int ch) -> uint32_t {
            return (mn ? (uint32_t)(ch >> 3) * 8192u : 0u) + row * 128 + (((ch & 7) ^ (row & 7)) << 4);
        };
        // K-major A: the source rows of this thread's chunks, fixed for the CTA
        int ar[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) ar[p] = Op::kAMN ? 0 : s_row[arow + 32 * p];
        const bool a_on = !Op::kAMN || m0 + ach * 8 < op.M;
        auto a_src = [&](int it, int p) -> const TA * {   // nullptr: zeros
            const int r = Op::kAMN ? s_row[it * 64 + arow + 16 * p] : ar[p];
            const int col = Op::kAMN ? m0 + ach * 8 : (kb0 + it) * 64 + ach * 8;
            if (r < 0 || !a_on || (!Op::kAMN && col >= op.K)) return nullptr;
            return op.A + (size_t)r * op.lda + col;
        };
        // this thread's first B chunk of a K block; the others are kBStep rows apart
        const int bn = n0 + (Op::kBMN ? bch * 8 : brow);
        auto b_used = [&](int p) {   // inside the tile's bn columns
            return (Op::kBMN ? bch * 8 : brow + kBStep * p) < sa.bn;
        };
        auto b_first = [&](int it) -> const TB * {
            const int kk = (kb0 + it) * 64 + (Op::kBMN ? brow : bch * 8);
            if (bn >= op.N || kk >= op.K) return nullptr;
            return Op::kBMN ? op.b_ptr(g, kk, bn) : op.b_ptr(g, bn, kk);
        };
        auto b_src = [&](const TB *first, int it, int p) -> const TB * {
            if (first == nullptr || !b_used(p)) return nullptr;
            if (Op::kBMN ? (kb0 + it) * 64 + brow + kBStep * p >= op.K : bn + kBStep * p >= op.N)
                return nullptr;
            return first + (size_t)(kBStep * p) * op.ldb;
        };
        if constexpr (kF32) {
            float4 av[4][2], bv[4][2];
            uint32_t nf = 0u;
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            auto load_a = [&](int it) {
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const TA *s = a_src(it, p);
                    av[p][0] = s ? *reinterpret_cast<const float4 *>(s) : zero;
                    av[p][1] = s ? *reinterpret_cast<const float4 *>(s + 4) : zero;
                }
            };
            auto load_b = [&](int it) {
                const TB *first = b_first(it);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const TB *s = b_src(first, it, p);
                    bv[p][0] = s ? *reinterpret_cast<const float4 *>(s) : zero;
                    bv[p][1] = s ? *reinterpret_cast<const float4 *>(s + 4) : zero;
                    if (Op::kBMN && bn + 8 > op.N && s != nullptr) {   // past the last column
                        float e[8] = {bv[p][0].x, bv[p][0].y, bv[p][0].z, bv[p][0].w,
                                      bv[p][1].x, bv[p][1].y, bv[p][1].z, bv[p][1].w};
#pragma unroll
                        for (int j = 0; j < 8; ++j) e[j] = bn + j < op.N ? e[j] : 0.f;
                        bv[p][0] = make_float4(e[0], e[1], e[2], e[3]);
                        bv[p][1] = make_float4(e[4], e[5], e[6], e[7]);
                    }
                }
            };
            if (nkb > 0) {
                load_a(0);
                load_b(0);
            }
            for (int it = 0; it < nkb; ++it) {
                const int s = it % S;
                if (!mbar_wait(smem_u32(&empty[s]), ((it / S) & 1) ^ 1) || *(volatile int *)s_abort) {
                    give_up();
                    break;
                }
                uint8_t *sA = ring + s * kStage, *sB = sA + Op::kPA * kSplitPlane;
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    uint4 pl[3];
                    split3(av[p][0], av[p][1], pl, nf);
                    const uint32_t o = place(Op::kAMN, arow + kAStep * p, ach);
#pragma unroll
                    for (int i = 0; i < 3; ++i)
                        *reinterpret_cast<uint4 *>(sA + i * kSplitPlane + o) = pl[i];
                }
                if (it + 1 < nkb) load_a(it + 1);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    if (!b_used(p)) continue;
                    uint4 pl[3];
                    split3(bv[p][0], bv[p][1], pl, nf);
                    const uint32_t o = place(Op::kBMN, brow + kBStep * p, bch);
#pragma unroll
                    for (int i = 0; i < 3; ++i)
                        *reinterpret_cast<uint4 *>(sB + i * kSplitPlane + o) = pl[i];
                }
                if (it + 1 < nkb) load_b(it + 1);
                fence_proxy_async();
                mbar_arrive(smem_u32(&full[s]));
            }
            if (nf & 0x80008000u) *(volatile int *)s_slow = 1;
            named_barrier(1, 512);   // with the drain warps, which read s_slow
        } else {
            constexpr int LAG = S - 2;
            int landed = 0, issued = 0;
            for (int it = 0; it < nkb; ++it) {
                const int s = it % S;
                if (!mbar_wait(smem_u32(&empty[s]), ((it / S) & 1) ^ 1) || *(volatile int *)s_abort) {
                    give_up();
                    break;
                }
                uint8_t *sA = ring + s * kStage, *sB = sA + Op::kPA * kSplitPlane;
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const TA *src = a_src(it, p);
                    const uint32_t dst = smem_u32(sA) + place(Op::kAMN, arow + kAStep * p, ach);
#pragma unroll
                    for (int i = 0; i < Op::kPA; ++i)
                        cp_async16(dst + i * kSplitPlane, src ? src + i * op.a_lo : op.A, src ? 16u : 0u);
                }
                const TB *first = b_first(it);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    if (!b_used(p)) continue;
                    const TB *src = b_src(first, it, p);
                    const uint32_t dst = smem_u32(sB) + place(Op::kBMN, brow + kBStep * p, bch);
#pragma unroll
                    for (int i = 0; i < Op::kPB; ++i)
                        cp_async16(dst + i * kSplitPlane,
                                   src ? src + i * op.b_lo : reinterpret_cast<const TB *>(op.A),
                                   src ? 16u : 0u);
                }
                cp_async_commit();
                issued = it + 1;
                // a stage is confirmed LAG stages after its copies were issued
                if (it >= LAG) {
                    cp_async_wait<LAG>();
                    fence_proxy_async();
                    mbar_arrive(smem_u32(&full[(it - LAG) % S]));
                    ++landed;
                }
            }
            cp_async_wait<0>();
            fence_proxy_async();
            for (int it = landed; it < issued; ++it) mbar_arrive(smem_u32(&full[it % S]));
        }
    } else if (warp == 16) {
        // ----------------------------------------------------- MMA issuer
        if (elect_one()) {
            const uint32_t idesc = idesc_bf16(128, sa.bn, Op::kAMN, Op::kBMN);
            for (int it = 0; it < nkb; ++it) {
                const int s = it % S, c = it / DR;
                bool ok = mbar_wait(smem_u32(&full[s]), (it / S) & 1);
                if (ok && it % DR == 0) ok = mbar_wait(smem_u32(&acce[c & 1]), ((c >> 1) & 1) ^ 1);
                if (!ok || *(volatile int *)s_abort) {
                    give_up();
                    break;
                }
                tc_fence_after();
                const uint32_t a = smem_u32(ring + s * kStage), b = a + Op::kPA * kSplitPlane;
                const int left = op.K - (kb0 + it) * 64;
                const int steps = left >= 64 ? 4 : (left + 15) / 16;
                uint32_t acc = it % DR == 0 ? 0u : 1u;
                auto product = [&](int i, int j) {
                    for (int st = 0; st < steps; ++st) {
                        const uint32_t ai = a + i * kSplitPlane, bj = b + j * kSplitPlane;
                        const uint64_t ad = Op::kAMN ? smem_desc_sw128(ai + st * 2048, 8192, 1024)
                                                     : smem_desc_sw128(ai + st * 32, 16, 1024);
                        const uint64_t bd = Op::kBMN ? smem_desc_sw128(bj + st * 2048, 8192, 1024)
                                                     : smem_desc_sw128(bj + st * 32, 16, 1024);
                        mma_bf16(tmem + 128 * (c & 1), ad, bd, idesc, acc);
                        acc = 1u;
                    }
                };
                // small products first
                if constexpr (kF32) {
                    product(2, 0);
                    product(0, 2);
                    product(1, 1);
                }
                if constexpr (Op::kPA > 1) product(1, 0);
                if constexpr (Op::kPB > 1) product(0, 1);
                product(0, 0);
                mma_commit(smem_u32(&empty[s]));
                if (it % DR == DR - 1 || it == nkb - 1) mma_commit(smem_u32(&accf[c & 1]));
            }
            drain_mmas(smem_u32(mdone));
        }
    } else {
        // ------------------------------------------- drain and output step
        const int q = warp & 3, hf = warp >> 2;
        const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + 64 * hf;
        float v[64];
#pragma unroll
        for (int j = 0; j < 64; ++j) v[j] = 0.f;
        const int chunks = (nkb + DR - 1) / DR;
        bool ok = true;
        for (int c = 0; c < chunks; ++c) {
            ok = mbar_wait(smem_u32(&accf[c & 1]), (c >> 1) & 1);
            // warp-uniform: the TMEM loads below are warp-collective
            if (__any_sync(0xffffffffu, !ok || *(volatile int *)s_abort)) {
                give_up();
                ok = false;
                break;
            }
            tc_fence_after();
#pragma unroll
            for (int c0 = 0; c0 < 64; c0 += 16) {
                if (64 * hf + c0 >= sa.bn) continue;   // bn is a multiple of 16
                float t[16];
                tmem_ld16(tb + 128 * (c & 1) + c0, t);
#pragma unroll
                for (int j = 0; j < 16; ++j) v[c0 + j] += t[j];
            }
            tc_fence_before();
            mbar_arrive(smem_u32(&acce[c & 1]));
        }
        // main loop done: the next kernel may start its prologue
        pdl_trigger();
        bool slow = false;
        if constexpr (kF32) {
            named_barrier(1, 512);   // the producers are past their last stage
            slow = *(volatile int *)s_slow != 0;
        }
        const int nb = n0 + 64 * hf;
        if (!ok) {
            // nothing to write
        } else if (slow) {
            const int m = m0 + q * 32 + lane;
            const int k_end = min(op.K, (kb0 + nkb) * 64);
            if (m < op.M)
                for (int n = nb; n < min(n_end, nb + 64); ++n) {
                    float acc = 0.f;
                    for (int k = kb0 * 64; k < k_end; ++k) acc = fmaf(op.a(g, m, k), op.b(g, k, n), acc);
                    op.store(g, m, n, acc, sa.splits > 1);
                }
        } else if constexpr (Op::kTrans) {
            const int m = m0 + q * 32 + lane;
            if (m < op.M) {
#pragma unroll
                for (int j = 0; j < 64; ++j)
                    if (nb + j < n_end) op.store(g, m, nb + j, v[j], sa.splits > 1);
            }
        } else {
            // through a 4 KB per-warp buffer in the idle ring, so that every
            // store or reduction instruction covers whole 128-byte row pieces
            uint8_t *xb = ring + warp * 4096;
#pragma unroll
            for (int c0 = 0; c0 < 64; c0 += 32) {
                if (nb + c0 >= n_end) continue;
                stage_f32x32(xb, v + c0, 1.f, lane);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int rl = (lane >> 3) + 4 * i, m = m0 + q * 32 + rl;
                    const int n = nb + c0 + 4 * (lane & 7);
                    const float4 x = *reinterpret_cast<const float4 *>(xb + xoff128(rl, lane & 7));
                    if (m < op.M && n < n_end) op.store4(g, m, n, x, sa.splits > 1);
                }
                __syncwarp();
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    span_end(sa.span);
    if (warp == 16) {
        tc_fence_after();
        tmem_dealloc(tmem, 256);
    }
}

// Launches op over `groups` groups; splits as chosen by split_count (the
// caller zeroes the output first where it is above 1).
template <class Op>
inline cudaError_t launch_split_gemm(const Op &op, int groups, int splits, uint32_t *status,
                                     cudaStream_t stream) {
    if (op.M <= 0 || op.N <= 0 || groups <= 0) return cudaSuccess;
    constexpr int smem = split_smem<Op>();
    cudaError_t e = allow_smem((const void *)split_gemm_kernel<Op>, smem);
    if (e != cudaSuccess) return e;
    const int nt = (op.N + 127) / 128;
    SplitArgs sa;
    sa.bn = ((op.N + nt - 1) / nt + 15) / 16 * 16;
    sa.nkb = (op.K + 63) / 64;
    sa.splits = splits;
    sa.status = status;
    sa.span = active_span();
    // column tiles fastest: neighbouring CTAs read the same rows of A
    const dim3 grid(nt, (op.M + 127) / 128, groups * splits);
    e = launch_pdl(split_gemm_kernel<Op>, grid, dim3(kSplitThreads), smem, stream, op, sa);
    note_launches(1);
    return e;
}

// Reduction splits of a product with M x N outputs in `groups` groups over K:
// enough CTAs for the 152 SMs while each keeps at least four K blocks, and at
// most kSplitIdxMax K rows to a CTA.
inline int split_count(int M, int N, int K, int groups) {
    const int tiles = (M + 127) / 128 * ((N + 127) / 128) * groups;
    const int nkb = (K + 63) / 64;
    int sp = (nkb * 64 + kSplitIdxMax - 1) / kSplitIdxMax;
    while (tiles * sp * 2 <= 152 && nkb / (sp * 2) >= 4) sp *= 2;
    return sp;
}

}  // namespace mosa
