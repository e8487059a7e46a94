// Shared device helpers of the CLEAR-MoE library (sm_103a): status word, bounded waits,
// bf16 packing, mbarrier / TMA / tcgen05 wrappers written as inline PTX.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/clearmoe.h"

#define CM_MAX_E 16
#define CM_MAX_R 256

namespace cm {

// ------------------------------------------------------------------ status word
__device__ __forceinline__ void set_status(int32_t* status, int32_t code) {
    if (status) atomicCAS(status, 0, code);  // the first device error wins
}

__device__ __forceinline__ uint64_t globaltimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// ------------------------------------------------------------------ bf16 helpers
__device__ __forceinline__ float bf16_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t v) { return __uint_as_float(v & 0xFFFF0000u); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);  // round to nearest even
    return *reinterpret_cast<uint32_t*>(&p);
}
__device__ __forceinline__ float bf16_to_f32(uint16_t v) { return __uint_as_float((uint32_t)v << 16); }
__device__ __forceinline__ uint16_t f32_to_bf16(float v) {
    const __nv_bfloat16 b = __float2bfloat16_rn(v);  // round to nearest even
    return *reinterpret_cast<const uint16_t*>(&b);
}

__device__ __forceinline__ float gelu_erf(float u) {
    // GELU(u) = u * Phi(u) = u * (1 + erf(u / sqrt 2)) / 2, with CUDA's erff.
    return 0.5f * u * (1.0f + erff(u * 0.70710678118654752440f));
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// GELU of a pair for the bf16 layer, whose hidden state is stored in bf16: GELU(u) = max(u, 0) - |u| / 2
// erfc(|u| / sqrt 2), with erfc(t / sqrt 2) = 2^q(t) and q a polynomial of degree 6 without constant
// term, fitted here to log2 erfc(t / sqrt 2) on [0, 5.5] by reweighted least squares in the error it makes
// in GELU (8.3e-8). Past 5.5 it falls on until t = 14, where t is held and the second term is 2e-35.
// Horner's rule runs on v = -t with the odd coefficients' signs turned, and the factor 1/2 is a -1 in the
// exponent, so that the result is one fma: 7 packed fp32x2 operations and two ex2 a pair, and one more for
// the infinities. What it costs is fc1's bound in short K and its energy in long: with the rational form named
// below (12 packed operations, two reciprocals) the ViT-B layer at 50,432 tokens took 400 us under load, now
// 390, the dense FFN at 100,864 tokens 652 and 634, the 12-sublayer stack at 25,216 tokens 2,385 and 2,348, the
// DeiT-S layer at 12,608 tokens 48.8 and 48.5.
// Error against float64: at most 3.2e-7 for every u (the rational form of Abramowitz & Stegun 7.1.28 in fp32:
// 7.1e-7), in every interval below -5 smaller than that form's, and mean square below it at every width
// (tests/test_gelu_exp2.py). These are absolute bounds: down to u = -4.25 the error is at most a quarter of the
// bf16 spacing of z; the relative error reaches 0.2 % at -4.5 and 0.5 % at -5 (|z| = 1.4e-6), where half a bf16
// step is 0.2 to 0.4 %. NaN and -inf give NaN and inf gives inf, as u (1 + erf(u / sqrt 2)) / 2 does.
struct GeluE {
    static constexpr float C6 = 2.992490044562146e-05f, C5 = 0.0007398800225928426f, C4 = 0.007977480068802834f,
                           C3 = 0.05323820933699608f, C2 = -0.45891568064689636f, C1 = 1.1511471271514893f;
    static constexpr float HOLD = -14.f;
};
__device__ __forceinline__ float2 gelu_pair_bf16(float2 u) {
    const float2 v = make_float2(fmaxf(-fabsf(u.x), GeluE::HOLD), fmaxf(-fabsf(u.y), GeluE::HOLD));
    float2 q = __ffma2_rn(make_float2(GeluE::C6, GeluE::C6), v, make_float2(GeluE::C5, GeluE::C5));
    q = __ffma2_rn(q, v, make_float2(GeluE::C4, GeluE::C4));
    q = __ffma2_rn(q, v, make_float2(GeluE::C3, GeluE::C3));
    q = __ffma2_rn(q, v, make_float2(GeluE::C2, GeluE::C2));
    q = __ffma2_rn(q, v, make_float2(GeluE::C1, GeluE::C1));
    q = __ffma2_rn(q, v, make_float2(-1.f, -1.f));
    // max(u, 0) = u / 2 + |u| / 2 exactly, NaN for -inf and NaN (max.NaN(u, 0) would give 0 for -inf, and 46.7 us
    // against 46.8 for the DeiT-S layer at 12,608 tokens, 85.9 against 86.3 for the dense ViT-B FFN there)
    const float2 half = make_float2(0.5f, 0.5f);
    const float2 relu = __ffma2_rn(half, u, make_float2(0.5f * fabsf(u.x), 0.5f * fabsf(u.y)));
    return __ffma2_rn(v, make_float2(ex2_approx(q.x), ex2_approx(q.y)), relu);
}

// GELU of a pair in fp32 for the tensor-core fp32 layer: GELU(u) = max(u, 0) - |u| / 2 erfc(|u| / sqrt 2),
// with erfc(t / sqrt 2) = 2^q(t) and q a polynomial of degree 10 without constant term, fitted here to
// log2 erfc(t / sqrt 2) on [0, 5.5] by reweighted least squares in the error it makes in GELU (1.6e-10);
// it falls on past 5.5, and t is held at 20, where 2^q is 0. No cancellation in the negative tail, no
// branch and packed fp32x2 arithmetic: measured against float64 over the inputs fc1 sees, its error is
// below that of u (1 + erff(u / sqrt 2)) / 2 (largest 2.5e-7 against 4.5e-7, tests/test_gelu_approx_f32.py).
// NaN and -inf give NaN, inf gives inf, as there.
struct GeluQ {
    static constexpr float C10 = -5.3994018145431255e-08f, C9 = 1.3470461226461339e-06f, C8 = -1.4872099200147204e-05f,
                           C7 = 9.307147411163896e-05f, C6 = -0.0003201701329089701f, C5 = 5.682075789081864e-05f,
                           C4 = 0.006903232075273991f, C3 = -0.05242511257529259f, C2 = -0.45922282338142395f,
                           C1 = -1.151104211807251f;
};
__device__ __forceinline__ float2 gelu_pair_f32(float2 u) {
    const float2 t = make_float2(fminf(fabsf(u.x), 20.f), fminf(fabsf(u.y), 20.f));
    float2 q = __ffma2_rn(make_float2(GeluQ::C10, GeluQ::C10), t, make_float2(GeluQ::C9, GeluQ::C9));
    q = __ffma2_rn(q, t, make_float2(GeluQ::C8, GeluQ::C8));
    q = __ffma2_rn(q, t, make_float2(GeluQ::C7, GeluQ::C7));
    q = __ffma2_rn(q, t, make_float2(GeluQ::C6, GeluQ::C6));
    q = __ffma2_rn(q, t, make_float2(GeluQ::C5, GeluQ::C5));
    q = __ffma2_rn(q, t, make_float2(GeluQ::C4, GeluQ::C4));
    q = __ffma2_rn(q, t, make_float2(GeluQ::C3, GeluQ::C3));
    q = __ffma2_rn(q, t, make_float2(GeluQ::C2, GeluQ::C2));
    q = __ffma2_rn(q, t, make_float2(GeluQ::C1, GeluQ::C1));
    q = __fmul2_rn(q, t);
    const float2 e = make_float2(ex2_approx(q.x), ex2_approx(q.y));
    const float2 half = make_float2(0.5f, 0.5f);
    // max(u, 0) = u / 2 + |u| / 2 exactly
    const float2 relu = __ffma2_rn(half, u, make_float2(0.5f * fabsf(u.x), 0.5f * fabsf(u.y)));
    return __ffma2_rn(__fmul2_rn(make_float2(-0.5f, -0.5f), t), e, relu);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ------------------------------------------------------------------ programmatic dependent launch
// A kernel launched with programmatic stream serialisation may start while its predecessor in the
// stream is still running; it must call pdl_wait() before touching anything that predecessor
// writes (or reads, if it overwrites it). pdl_launch_dependents() lets the successor start early.
// Both are no-ops for kernels launched without the attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ------------------------------------------------------------------ mbarrier
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// By the elected lane of a converged warp (as the TMA loads below).
__device__ __forceinline__ void mbar_arrive_expect_tx_warp(uint32_t bar, uint32_t bytes) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(bar), "r"(bytes)
        : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the phase of `parity` to complete, giving up after limit_ns or when another role of
// the CTA has already given up (*abort != 0; abort may be null). Returns false on give-up; the first waiter to run
// out raises *abort and writes CLEARMOE_ETIMEOUT to the status word.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort,
                                          int32_t* status, uint64_t limit_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer();
    while (true) {
        if (abort && *abort) return false;
        if (mbar_try_wait(bar, parity)) return true;
        if (globaltimer() - t0 > limit_ns) {
            if (abort) *abort = 1;
            set_status(status, CLEARMOE_ETIMEOUT);
            return false;
        }
    }
}

// mbar_wait by a whole warp: every lane returns the same outcome. Each lane reads the clock and the abort
// flag for itself, so near the limit single lanes may give up; what follows a wait is run by the whole warp
// (tcgen05.ld, shuffles, __syncwarp, elect.sync) and needs all lanes or none.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort, int32_t* status,
                                               uint64_t limit_ns) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort, status, limit_ns));
}
// v of lane 0, as a value the compiler knows to be the same in every lane
template <typename V>
__device__ __forceinline__ V warp_uniform(V v) {
    return __shfl_sync(0xffffffffu, v, 0);
}

__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_u32(unsigned int* p, unsigned int v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// ------------------------------------------------------------------ TMA
// Called by a whole, converged warp; one elected lane issues (the reason is at the tcgen05 wrappers).
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int32_t c0,
                                            int32_t c1, uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];\n\t}" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int32_t c0, int32_t c1,
                                            int32_t c2, uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];\n\t}" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void cp_async_16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ------------------------------------------------------------------ tcgen05
__device__ __forceinline__ void tmem_alloc(uint32_t slot_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     slot_smem),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// The MMA, commit and TMA wrappers are called by a whole, converged warp; one elected lane issues.
// What bounds the issuing warp: an MMA or a tensor copy reads its descriptors from uniform registers.
// With warp-uniform control flow they are computed there; issued from a branch that only lane 0 takes,
// each instruction first pays for moving them, which bounded every kernel whose MMAs are short (K
// steps of 256 x 192 or 128 x 64 tiles; the fp32 layer's twelve MMAs per stage). Measured with lane 0
// -> the whole warp: DeiT-S layer 66.9 -> 55.5 us (basis 16.3 -> 12.3, grouped 28.7 -> 22.5 us), DeiT-B
// layer 418 -> 408 us under load (grouped 153.6 -> 141.3 us), DeiT-T fp32 layer 51.2 -> 47.5 us.
// D[tmem] (+)= A[smem] * B[smem]^T, kind::f16 (bf16 inputs, fp32 accumulator), one CTA.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                          uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Arrive once on an mbarrier when every tcgen05.mma issued so far by this warp's elected lane completes.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

#define CM_TMEM_LD_X16(taddr, r)                                                                 \
    asm volatile(                                                                                \
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13," \
        "%14,%15}, [%16];"                                                                       \
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),    \
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),             \
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])                                                  \
        : "r"(taddr))

#define CM_TMEM_LD_X8(taddr, r)                                                                  \
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"         \
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),        \
                   "=r"(r[6]), "=r"(r[7])                                                         \
                 : "r"(taddr))

__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// One warp's 32 lanes x 32 columns of tensor memory from registers (then tmem_wait_st before the
// columns are handed over).
#define CM_TMEM_ST_X32(taddr, r)                                                                       \
    asm volatile(                                                                                      \
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"           \
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),                            \
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), \
        "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), \
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), \
        "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), \
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), \
        "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), \
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), \
        "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]) \
        : "memory")

// Shared-memory matrix descriptor of a K-major bf16 tile written by TMA with 128-byte swizzle:
// rows of 128 bytes (64 elements of K), 8-row swizzle atoms 1024 bytes apart (SBO), descriptor
// version 1, layout SWIZZLE_128B. The tile base must be 1024-byte aligned; advancing along K
// inside the atom is done by adding the byte offset to the start address.
__device__ __forceinline__ uint64_t sdesc_kmajor_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;            // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;  // stride byte offset: 8 rows x 128 B
    d |= (uint64_t)1 << 46;            // descriptor version
    d |= (uint64_t)2 << 61;            // SWIZZLE_128B
    return d;
}

// The same K-major 128-byte-swizzled descriptor with 8-row atoms `sbo` bytes apart (a multiple of
// 16 below 256 KB), for tiles whose row groups are interleaved with other K blocks' in shared memory.
__device__ __forceinline__ uint64_t sdesc_kmajor_sw128_sbo(uint32_t saddr, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor of tcgen05.mma kind::f16: fp32 accumulator, bf16 A and B, both
// K-major, M x N tile.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

}  // namespace cm
