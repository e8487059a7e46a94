// Folding the shared basis into the residual experts: W_e^comb = U_r diag(S_r) V_r^T + W_e^res.
//
// Eq. 2 sums a shared and a per-expert term on the same hidden state, y = W_shared z + W_e^res z,
// so y = W_e^comb z with W_e^comb = W_shared + W_e^res, which turns the forward into one grouped
// GEMM over z (the dense FFN's arithmetic) with no basis step. This kernel forms the combined
// weights once per weight set: each CTA computes a 32 x 128 tile of W_shared = U_r diag(S_r) Vh_r in
// fp32 (products S_r[k] Vh_r[k][h] in fp32, fma over k ascending), then adds it to the same tile of
// every expert's residual (none when res[e] is null: W_shared materialised alone) and rounds once
// to the layer dtype.
//
// What bounds it: at r = 128 the fp32 products (2 d H r flops on the CUDA cores) and one read and one
// write of E matrices take about the same time. A CTA of 128 threads owns 32 x 128 outputs, each
// thread 4 rows x 2 groups of 4 columns: per k one 16-byte shared load of U and two of S Vh (conflict
// free) feed 16 packed fp32x2 FMAs; the next k chunk's operands wait in registers, and the experts'
// tiles move as 4-column vectors, the next expert's loads in flight while one is added and stored.
// 32-row tiles give 576 CTAs at 768 x 3072, about four on every SM.
// Measured (768 x 3072 bf16, E = 8, r = 128, back to back with inputs changing): 88.9 us with 64 x 64
// tiles, scalar bf16 accesses and 4 x 4 outputs per thread; 38.9 us now.
#include "common.cuh"
#include "internal.h"

namespace cm {
namespace {

constexpr int FM = 32, FN = 128;  // output tile (rows of d x columns of H)
constexpr int FK = 32;            // k chunk
constexpr int F_THREADS = 128;

template <bool BF16>
__device__ __forceinline__ float load_elem(const void* p, int64_t i) {
    if constexpr (BF16)
        return bf16_to_f32(static_cast<const uint16_t*>(p)[i]);
    else
        return static_cast<const float*>(p)[i];
}

// Four consecutive elements of a matrix: one 8-byte (bf16) or 16-byte (fp32) access with VEC, else one
// by one. T holds them as loaded.
template <bool BF16, bool VEC>
struct Quad {
    using T = float4;
    static __device__ __forceinline__ T load(const void* p, int64_t i) {
        if constexpr (VEC && !BF16) return *reinterpret_cast<const float4*>(static_cast<const float*>(p) + i);
        return make_float4(load_elem<BF16>(p, i), load_elem<BF16>(p, i + 1), load_elem<BF16>(p, i + 2), load_elem<BF16>(p, i + 3));
    }
    static __device__ __forceinline__ float4 value(T v) { return v; }
    static __device__ __forceinline__ void store(void* p, int64_t i, float4 v) {
        if constexpr (VEC && !BF16) {
            *reinterpret_cast<float4*>(static_cast<float*>(p) + i) = v;
        } else {
            const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if constexpr (BF16)
                    static_cast<uint16_t*>(p)[i + j] = f32_to_bf16(f[j]);
                else
                    static_cast<float*>(p)[i + j] = f[j];
            }
        }
    }
};
template <>
struct Quad<true, true> {
    using T = uint2;
    static __device__ __forceinline__ T load(const void* p, int64_t i) {
        return *reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(p) + i);
    }
    static __device__ __forceinline__ float4 value(T u) {
        return make_float4(bf16_lo(u.x), bf16_hi(u.x), bf16_lo(u.y), bf16_hi(u.y));
    }
    static __device__ __forceinline__ void store(void* p, int64_t i, float4 v) {
        *reinterpret_cast<uint2*>(static_cast<uint16_t*>(p) + i) = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
    }
};

// VEC: every matrix starts on a 4-element boundary (H % 4 == 0 makes every row do)
template <bool BF16, bool VEC>
__global__ void __launch_bounds__(F_THREADS, 4) fold_basis_kernel(const FoldArgs a) {
    __shared__ __align__(16) float Us[FK][FM + 4];  // U_r[i0 + i][k0 + k] at [k][i]
    __shared__ __align__(16) float Vs[FK][FN];      // S_r[k0 + k] Vh_r[k0 + k][h0 + h] at [k][h]
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int i0 = blockIdx.y * FM, h0 = blockIdx.x * FN;
    // this thread's outputs: rows i0 + 4 ty + i, columns h0 + 64 g + 4 tx + j
    float2 acc[4][2][2];  // [row][column group][pair]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int g = 0; g < 2; ++g) acc[i][g][0] = acc[i][g][1] = make_float2(0.f, 0.f);

    // operand chunk in registers: U elements tid + 128 q (32 rows x 32 k, k fastest), and S Vh vectors
    // tid + 128 q (32 k x 32 column quads, columns fastest)
    float ur[8];
    float4 vr[8];
    auto load_chunk = [&](int k0) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = tid + F_THREADS * q;
            const int i = i0 + (e >> 5), k = k0 + (e & 31);
            ur[q] = (i < a.d && k < a.r) ? load_elem<BF16>(a.U, (int64_t)i * a.r + k) : 0.f;
            const int kv = k0 + (e >> 5), h = h0 + (e & 31) * 4;
            vr[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (kv < a.r && h < a.H) {
                const float s = a.S[kv];
                const float4 v = Quad<BF16, VEC>::value(Quad<BF16, VEC>::load(a.Vh, (int64_t)kv * a.H + h));
                vr[q] = make_float4(s * v.x, s * v.y, s * v.z, s * v.w);
            }
        }
    };
    load_chunk(0);
    for (int k0 = 0; k0 < a.r; k0 += FK) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = tid + F_THREADS * q;
            Us[e & 31][e >> 5] = ur[q];
            *reinterpret_cast<float4*>(&Vs[e >> 5][(e & 31) * 4]) = vr[q];
        }
        __syncthreads();
        if (k0 + FK < a.r) load_chunk(k0 + FK);
        const int kn = min(FK, a.r - k0);
#pragma unroll 4
        for (int k = 0; k < kn; ++k) {
            const float4 av = *reinterpret_cast<const float4*>(&Us[k][4 * ty]);
            const float4 b0 = *reinterpret_cast<const float4*>(&Vs[k][4 * tx]);
            const float4 b1 = *reinterpret_cast<const float4*>(&Vs[k][64 + 4 * tx]);
            const float ar[4] = {av.x, av.y, av.z, av.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 a2 = make_float2(ar[i], ar[i]);
                acc[i][0][0] = __ffma2_rn(a2, make_float2(b0.x, b0.y), acc[i][0][0]);
                acc[i][0][1] = __ffma2_rn(a2, make_float2(b0.z, b0.w), acc[i][0][1]);
                acc[i][1][0] = __ffma2_rn(a2, make_float2(b1.x, b1.y), acc[i][1][0]);
                acc[i][1][1] = __ffma2_rn(a2, make_float2(b1.z, b1.w), acc[i][1][1]);
            }
        }
        __syncthreads();
    }
    // out[e] = W_shared + res[e]: all eight vectors of an expert's tile loaded before any is used, the
    // next expert's before this one's are stored
    const int row = i0 + 4 * ty, col = h0 + 4 * tx;
    using R = Quad<BF16, VEC>;
    typename R::T cur[4][2], nxt[4][2];
    auto load_res = [&](typename R::T (&v)[4][2], const void* res) {
        if (!res) return;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int g = 0; g < 2; ++g)
                if (row + i < a.d && col + 64 * g < a.H) v[i][g] = R::load(res, (int64_t)(row + i) * a.H + col + 64 * g);
    };
    load_res(cur, a.res[0]);
    for (int e = 0; e < a.E; ++e) {
        if (e + 1 < a.E) load_res(nxt, a.res[e + 1]);
        const bool add = a.res[e] != nullptr;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                if (row + i < a.d && col + 64 * g < a.H) {
                    const float2 p0 = acc[i][g][0], p1 = acc[i][g][1];
                    float4 o = make_float4(p0.x, p0.y, p1.x, p1.y);
                    if (add) {
                        const float4 v = R::value(cur[i][g]);
                        o = make_float4(o.x + v.x, o.y + v.y, o.z + v.z, o.w + v.w);
                    }
                    R::store(a.out[e], (int64_t)(row + i) * a.H + col + 64 * g, o);
                }
                cur[i][g] = nxt[i][g];
            }
    }
}

}  // namespace

cudaError_t launch_fold_basis(const FoldArgs& a, int dtype, cudaStream_t s) {
    const dim3 grid((unsigned)((a.H + FN - 1) / FN), (unsigned)((a.d + FM - 1) / FM));
    // 4-element accesses where every matrix allows them (the ABI states 16-byte alignment, but a call
    // with less has always been served)
    const uintptr_t mask = dtype == CLEARMOE_BF16 ? 7 : 15;
    uintptr_t low = reinterpret_cast<uintptr_t>(a.Vh);
    for (int e = 0; e < a.E; ++e) low |= reinterpret_cast<uintptr_t>(a.res[e]) | reinterpret_cast<uintptr_t>(a.out[e]);
    const bool vec = (low & mask) == 0 && a.H % 4 == 0;
    if (dtype == CLEARMOE_BF16)
        vec ? fold_basis_kernel<true, true><<<grid, F_THREADS, 0, s>>>(a) : fold_basis_kernel<true, false><<<grid, F_THREADS, 0, s>>>(a);
    else
        vec ? fold_basis_kernel<false, true><<<grid, F_THREADS, 0, s>>>(a) : fold_basis_kernel<false, false><<<grid, F_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace cm
