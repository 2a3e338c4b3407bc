// Helpers shared by the tensor-core kernels: bounded mbarrier waits, exp2, bf16 packing, and the
// host-side construction of TMA tensor maps.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "ptx_sm100.cuh"

namespace flat {
namespace tc {

constexpr long long WAIT_CYCLES = 2000000000ll;   // ~1 s at 2 GHz
constexpr float RESCALE_THRESHOLD = 8.0f;         // log2 units: P stays <= 2^8

// Waits for the phase of `bar` with the given parity.  Gives up when another role of the CTA has
// raised the abort flag or after WAIT_CYCLES; the first thread to time out raises the flag and
// records `code` in *status.  Never traps, never spins without limit.
__device__ __forceinline__ bool bounded_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                             int32_t* status, int code, long long limit = WAIT_CYCLES) {
    if (ptx::mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
        // The inner probes cost two instructions each; the clock and the abort flag are looked at
        // once per batch so that a waiting warp leaves the issue slots to the working ones.
#pragma unroll 1
        for (int i = 0; i < 32; ++i)
            if (ptx::mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > limit) {
            *abort_flag = 1;
            if (status) atomicExch(status, code);
            return false;
        }
    }
}

// The same wait with the barrier and the abort flag given as 32-bit shared-window addresses.
// SLEEP_NS > 0: the thread sleeps that long between probes -- for a role whose reaction time does
// not matter (a producer that runs ahead of its ring) and that should leave the issue slots and
// the shared-memory pipe to the working warps while it waits.
template <unsigned SLEEP_NS = 0>
__device__ __forceinline__ bool bounded_wait_s(uint32_t bar_addr, uint32_t parity, uint32_t abort_addr,
                                               int32_t* status, int code, long long limit = WAIT_CYCLES) {
    if (ptx::mbar_try_wait_s(bar_addr, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 32; ++i) {
            if (SLEEP_NS) __nanosleep(SLEEP_NS);
            if (ptx::mbar_try_wait_s(bar_addr, parity)) return true;
        }
        int aborted;
        asm volatile("ld.volatile.shared::cta.s32 %0, [%1];" : "=r"(aborted) : "r"(abort_addr) : "memory");
        if (aborted) return false;
        if (clock64() - t0 > limit) {
            asm volatile("st.volatile.shared::cta.s32 [%0], %1;" ::"r"(abort_addr), "r"(1) : "memory");
            if (status) atomicExch(status, code);
            return false;
        }
    }
}

// The warp's index.  The shuffle tells the compiler that it is the same in all lanes: what follows from it (roles, loops, MMA
// operands) then stays in uniform registers.  Whether that helps is a matter of each instantiation (registers, spills, which values
// the uniform datapath gets), so every kernel says at its index what was measured: with warp_wait below dK dV 3 % a step and dQ 10 %
// the other way, fused_d128 with several items 12 %, with one 3 % the other way in the softmax warps, fused_tf32 at d = 64 5 %,
// fused_decode 1 %; fused_tc3 loses 2 %, fused_tc2 1 %, fused_tf32 at d = 128 11 % and the spilling forms of proj_gemm 1 to 6 %.
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0); }

// bounded_wait by a whole warp.  The warp stays together: its lanes probe and vote as one.  (Where each lane loops by itself,
// they come back one by one after a long wait and what follows starts up to 500 cycles late.)
__device__ __forceinline__ bool warp_wait(uint32_t bar_addr, uint32_t parity, uint32_t abort_addr, int32_t* status, int code) {
    if (__all_sync(0xffffffffu, ptx::mbar_try_wait_s(bar_addr, parity))) return true;
    const long long t0 = clock64();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 32; ++i)
            if (__all_sync(0xffffffffu, ptx::mbar_try_wait_s(bar_addr, parity))) return true;
        int aborted;
        asm volatile("ld.volatile.shared::cta.s32 %0, [%1];" : "=r"(aborted) : "r"(abort_addr) : "memory");
        if (__any_sync(0xffffffffu, aborted)) return false;
        if (__any_sync(0xffffffffu, clock64() - t0 > WAIT_CYCLES)) {
            asm volatile("st.volatile.shared::cta.s32 [%0], %1;" ::"r"(abort_addr), "r"(1) : "memory");
            if (status) atomicExch(status, code);
            return false;
        }
    }
}

__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int32_t* status, int code) {
    return warp_wait(ptx::smem_u32(bar), parity, ptx::smem_u32(const_cast<int*>(abort_flag)), status, code);
}

// Teardown helper: wait for a copy this thread started, with a time limit and no side effects.
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!ptx::mbar_try_wait(bar, parity))
        if (clock64() - t0 > WAIT_CYCLES) return;
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 2^x on the FMA and integer pipes instead of the ex2 unit: x = r + f with r = round(x) and
// f in [-0.5, 0.5]; 2^f by a cubic (max relative error 7.7e-5, far below the bf16 rounding that
// the weights undergo next) and 2^r by adding r to the exponent field.  x is clamped to
// [-126, 126] so that the exponent arithmetic cannot wrap (the cubic lies in [0.70, 1.42], biased
// exponent 126 or 127, so r >= -126 keeps the field at 0 or above): below, the result is a
// denormal of about 2^-126 (as good as 0 next to a row maximum of order 1); above, it is 2^126,
// which trips the caller's overflow check exactly like the ex2 unit's +inf would.
__device__ __forceinline__ float ex2_poly(float x) {
    x = fminf(fmaxf(x, -126.f), 126.f);
    const float t = x + 12582912.f;                    // 1.5 * 2^23: the low mantissa bits now hold round(x)
    const float r = t - 12582912.f;
    const float f = x - r;
    float p = fmaf(0.05508868f, f, 0.24260405f);
    p = fmaf(p, f, 0.69327624f);
    p = fmaf(p, f, 0.99992894f);
    return __uint_as_float(__float_as_uint(p) + (__float_as_uint(t) << 23));
}

// Three-input maximum / minimum (one instruction on sm_100).
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&h);
}

// Query rows in plain fp32 FMAs, by a whole warp: for the rows whose result from split operands is not finite.  An infinity splits
// into a head and a remainder that is no number, and a weight of up to 2^40 (reference maxima are kept while they serve) may
// carry a large value past the largest number; without either, infinite values give infinite features and large ones their
// mean.  The rows are `row0` + the bits of `mask`; lane i holds the number of keys that row i sees.  Eight rows at a time share every key
// and value: a lane takes one of 32 keys' logits, then d / 32 features.  What can only be NaN is left early: rows once their
// sums are (a NaN or +infinite logit), features once all are.  Where it comes to every row of a call: B2 H16 4096^2 in fp32 with an infinite
// value in every head 37.6 ms at d = 128 and 12.3 at d = 32 (FFMA kernel 9.5 and 2.7), all queries NaN 1.4 and 0.5.
__device__ __forceinline__ void floats16(const float* p, float (&f)[4]) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
}
__device__ __forceinline__ void floats16(const __nv_bfloat16* p, float (&f)[8]) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) { f[2 * e] = __uint_as_float(w[e] << 16); f[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u); }
}
template <typename T, int D>
static __device__ __noinline__ void plain_rows(unsigned mask, int64_t row0, int own_keys, const T* Q, const T* K, const T* V, T* O, float* lse,
                                               float scale_log2e) {
    constexpr int N = 16 / sizeof(T), F = (D + 31) / 32, R = 8, UNROLL = sizeof(T) == 4 ? 4 : 2;
    const int lane = threadIdx.x & 31;
    __syncwarp();                                        // (the rows' own threads have stored them)
    while (mask) {
        int at[R], nk[R], most = 0;                      // (fewer than eight: the first one again)
        float m[R], l[R], acc[R][F];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            at[r] = mask ? __ffs(mask) - 1 : at[0];
            mask &= mask - 1;
            nk[r] = __shfl_sync(0xffffffffu, own_keys, at[r]);
            most = nk[r] > most ? nk[r] : most;
            m[r] = -INFINITY;
            l[r] = 0.f;
#pragma unroll
            for (int i = 0; i < F; ++i) acc[r][i] = 0.f;
        }
        bool done = false;                               // (the same in all lanes, as are l and m)
        for (int k0 = 0; k0 < most; k0 += 32) {
            const int key = k0 + lane;
            const T* k = K + static_cast<int64_t>(key < most ? key : k0) * D;
            float p[R];
#pragma unroll
            for (int r = 0; r < R; ++r) p[r] = 0.f;
#pragma unroll UNROLL
            for (int t = 0; t < D; t += N) {
                float b[N];
                floats16(k + t, b);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    float a[N];
                    floats16(Q + (row0 + at[r]) * D + t, a);
#pragma unroll
                    for (int e = 0; e < N; ++e) p[r] = fmaf(a[e], b[e], p[r]);
                }
            }
            bool nan = true;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float x = key < nk[r] ? p[r] * scale_log2e : -INFINITY;
                float mx = x;
#pragma unroll
                for (int s = 16; s >= 1; s >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
                const float m_new = fmaxf(m[r], mx), m_use = m_new == -INFINITY ? 0.f : m_new;
                const float alpha = exp2f(m[r] - m_use);
                p[r] = exp2f(x - m_use);
                float sum = p[r];
#pragma unroll
                for (int s = 16; s >= 1; s >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, s);
                l[r] = l[r] * alpha + sum;
                m[r] = m_new;
                nan = nan && l[r] != l[r];
#pragma unroll
                for (int i = 0; i < F; ++i) acc[r][i] *= alpha;
            }
            if (nan) break;
            if (done) continue;
            const int n = most - k0 < 32 ? most - k0 : 32;
            constexpr int JB = F > 1 ? 4 : 8;            // values in flight
            for (int j0 = 0; j0 < n; j0 += JB) {
                float v[JB][F];
#pragma unroll
                for (int j = 0; j < JB; ++j)
#pragma unroll
                    for (int i = 0; i < F; ++i)
                        v[j][i] = j0 + j < n && lane + 32 * i < D ? static_cast<float>(V[static_cast<int64_t>(k0 + j0 + j) * D + lane + 32 * i]) : 0.f;
#pragma unroll
                for (int j = 0; j < JB; ++j)
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float pj = __shfl_sync(0xffffffffu, p[r], j0 + j);
                        if (k0 + j0 + j < nk[r]) {       // (a key that the row does not see may hold anything)
#pragma unroll
                            for (int i = 0; i < F; ++i) acc[r][i] = fmaf(pj, v[j][i], acc[r][i]);
                        }
                    }
            }
            nan = true;
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int i = 0; i < F; ++i) nan = nan && (lane + 32 * i >= D || acc[r][i] != acc[r][i] || l[r] != l[r]);
            done = __all_sync(0xffffffffu, nan);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float inv = l[r] > 0.f ? 1.f / l[r] : l[r] == l[r] ? 0.f : l[r];      // (no visible key: 0; a NaN sum: NaN)
#pragma unroll
            for (int i = 0; i < F; ++i)
                if (lane + 32 * i < D) O[(row0 + at[r]) * D + lane + 32 * i] = static_cast<T>(acc[r][i] * inv);
            if (lse && lane == 0) lse[row0 + at[r]] = l[r] > 0.f ? (m[r] + log2f(l[r])) * 0.6931471805599453f : -INFINITY;
        }
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// cuTensorMapEncodeTiled through the runtime's driver entry-point lookup (no link against libcuda).
inline EncodeTiledFn get_encode_fn() {
    static EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// bf16 tensor [BH, N, d] (d contiguous) viewed as 3-D {d, N, BH}; box = 64 x rows x 1, 128-byte swizzle.
inline bool make_map(CUtensorMap* m, const void* ptr, int BH, int N, int d, int box_rows) {
    EncodeTiledFn enc = get_encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(d), static_cast<cuuint64_t>(N), static_cast<cuuint64_t>(BH)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(d) * 2, static_cast<cuuint64_t>(N) * d * 2};
    cuuint32_t box[3] = {64, static_cast<cuuint32_t>(box_rows), 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A packed tensor [tokens, H, d] bf16 (variable-length batches) as a TMA tensor {d, H, tokens} with
// boxes of 64 features x one head x box_rows tokens (in shared memory: box_rows rows of 128 bytes, as
// for the batched layout).
inline bool make_map_packed(CUtensorMap* m, const void* ptr, int64_t tokens, int H, int d, int box_rows) {
    EncodeTiledFn enc = get_encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(d), static_cast<cuuint64_t>(H), static_cast<cuuint64_t>(tokens)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(d) * 2, static_cast<cuuint64_t>(H) * d * 2};
    cuuint32_t box[3] = {64, 1, static_cast<cuuint32_t>(box_rows)};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A bias whose rows begin at any alignment, staged by TMA all the same.  Row R of all its rows (heads and batches after one
// another, Nk bf16 each) lies in group R / 8 of eight rows, groups that are 16 Nk bytes apart: a tensor map {8 Nk, groups} brings
// the rows of one phase R % 8 = b with boxes of 16 groups, from a column rounded down to 16 bytes, and 8 b columns further left
// still: in shared memory (SHIFT_ROW = 2 x box width = 0 mod 128 bytes a row) rows of different phase then start 16 bytes apart and
// the 16-byte reads of a warp's rows meet no bank conflict.  What is left, 0 to 14 bytes, a thread shifts in registers.  Rows
// beyond the last whole group (`full`: rows in whole groups) come from device memory, copied by the row's own thread.
// Measured, against 16-byte pieces straight from device memory (us): d = 64, B8 H16 1001^2 293 -> 115 (no bias: 59; 1024^2, where
// nothing is to be shifted: 80), B6 H8 2770^2 1,057 -> 278; d = 128, B8 H16 1001^2 367 -> 153, B3 H12 3247^2 1,380 -> 450.  Bound
// by the shifts (15 instructions per 8 values) and the one stage per query tile that its width leaves room for.
struct ShiftedBias {
    const uint16_t* p;
    int full;
};
// Boxes for the tile of 128 rows from row g0 of all and the keys from column col.
template <int WIDTH>
__device__ __forceinline__ void load_shifted_bias(uint8_t* dst, const void* tmap, uint64_t* bar, int g0, int col, int Nk) {
#pragma unroll
    for (int b = 0; b < 8; ++b)
        ptx::tma_load_3d(dst + b * 16 * WIDTH * 2, tmap, bar, ((b * Nk + col) & ~7) - 8 * b, (g0 + ((b - g0) & 7)) >> 3, 0);
}
// Byte offset of row R's first 16-byte piece in a tile from row g0 on, and the bytes from there to its first value (any column
// that is a multiple of 8).
template <int WIDTH>
__device__ __forceinline__ uint32_t shifted_row(int R, int g0) {
    const int b = R & 7;
    return (b * 16 + (R >> 3) - ((g0 + ((b - g0) & 7)) >> 3)) * (WIDTH * 2) + 16 * b;
}
__device__ __forceinline__ uint32_t shifted_by(int R, int Nk) { return 2 * (((R & 7) * Nk) & 7); }
// Eight values from two 16-byte pieces.
__device__ __forceinline__ void shift8(const uint32_t (&w)[8], uint32_t by, uint32_t (&o)[4]) {
    uint32_t a[6], c[5];
#pragma unroll
    for (int k = 0; k < 6; ++k) a[k] = by & 8 ? w[k + 2] : w[k];
#pragma unroll
    for (int k = 0; k < 5; ++k) c[k] = by & 4 ? a[k + 1] : a[k];
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = __funnelshift_r(c[k], c[k + 1], (by & 2) * 8);
}
// `n` values of a row into its place.
static __device__ __noinline__ void copy_bias_row(const uint16_t* src, uint32_t dst, int n) {
    for (int i = 0; i < n; ++i) asm volatile("st.shared::cta.u16 [%0], %1;" ::"r"(dst + 2 * i), "h"(src[i]) : "memory");
    ptx::fence_proxy_async_smem();       // (the tile's next copy follows)
}
inline bool make_shifted_bias_map(CUtensorMap* m, const void* ptr, int64_t groups, int Nk, int width) {
    EncodeTiledFn enc = get_encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(Nk) * 8, static_cast<cuuint64_t>(groups), 1};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(Nk) * 16, static_cast<cuuint64_t>(Nk) * 16 * groups};
    cuuint32_t box[3] = {static_cast<cuuint32_t>(width), 16, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace tc
}  // namespace flat
