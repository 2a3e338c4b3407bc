// Fused Logit-Softmax-Attend for at most sixteen queries per head (decode steps; bf16 in, fp32 accumulate, bf16 out;
// d = 64 and 128).  The paper's fused dataflow (Section 5) at its smallest row granularity: the keys and values are read
// once and meet a handful of query rows.
//
// What bounds it: device memory -- 4 d bytes per key and head, and 4 d FLOP per query of them, far below what any pipe
// delivers.  The 128-row tiles of the tcgen05 kernels spend their time on 112 to 127 padding rows instead (exponentials,
// TMEM traffic: 2.9 TB/s on B16 H16 1 x 8192, d = 128), and M = 64 would still be mostly padding; so the contractions
// go through the warp-level m16n8k16 instruction, whose sixteen rows fit the queries, and everything else is arranged
// around the stream of keys: TMA copies of 32 KB per stage, 96 KB (192 KB where a CTA has an SM to itself) in flight per
// CTA, four warps that each take a quarter of a stage's keys and keep (m, l, O) of their own in registers, no barrier
// among them until the end.  Then the four merge through shared memory and the CTAs of a cluster, which share a
// head's keys evenly, through distributed shared memory: every CTA leaves (m, l, O) in its own memory, a cluster
// barrier, and each finishes its share of the outputs from all of them in the order of the ranks (same bits every time).
// Measured (key counts uniform in [Nk / 4, Nk]): B16 H16 1 x 8192 d 128 203 -> 101 us (76,343 keys a head in the 16 batches: 625 MB, 6.2
// TB/s; all 131,072: 151 us, 7.1 TB/s), d 64 117 -> 52 (80,413 keys: 329 MB, 6.3 TB/s; all: 78 us, 6.8 TB/s); sixteen queries 190 -> 104; B32 H32 1 x 2048 181 -> 100; 4 heads x 32768 48 -> 14; B32 H8 1 x 512 29 -> 11.5.
//
// CTA = 160 threads: warps 0-3 as above, warp 4 TMA producer.  Tiles have the 128-byte swizzle; ldmatrix reads eight rows
// of a panel without bank conflicts.  A warp's logits come out with queries as rows and keys as columns, which is the
// layout of the left operand of P V.  Exact running maximum, O rescaled only when one of the warp's rows has a new one.
// Every wait is bounded; on expiry the CTA ends cleanly and reports a code (the rows it took part in become NaN).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "flat_internal.cuh"
#include "ptx_sm100.cuh"
#include "tc_common.cuh"

namespace flat {

using namespace ptx;
using namespace tc;

namespace {

constexpr int DEC_WARPS = 4, DEC_THREADS = 32 * DEC_WARPS + 32;
constexpr int DEC_MAX_Q = 16;

template <int D, int STAGES> struct LD {
    static constexpr int KEYS = 8192 / D;                // per stage: 64 (d = 128) or 128; a quarter per warp
    static constexpr int WKEYS = KEYS / DEC_WARPS;
    static constexpr int TILE_BYTES = KEYS * D * 2;      // 16 KB of K, 16 KB of V
    static constexpr int RING_BYTES = STAGES * 2 * TILE_BYTES;
    static constexpr int SMEM_BYTES = RING_BYTES + 1024;
};

__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4_t(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// c (16 x 8) += a (16 x 16) b (16 x 8)
__device__ __forceinline__ void mma16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float2 ld_cluster_f32x2(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float quad_max(float v) {
    v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
    return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}

// RG: row groups of eight queries (1: at most eight queries, 2: at most sixteen).  CS: CTAs of the cluster.
template <int D, int RG, int CS, int STAGES>
__global__ void __launch_bounds__(DEC_THREADS, STAGES > 3 ? 1 : 2)
fused_decode_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                    const __nv_bfloat16* __restrict__ Q, __nv_bfloat16* __restrict__ O, int H, int Nq, int Nk, float scale_log2e,
                    const int32_t* __restrict__ valid_len, int causal, int32_t* status, float* __restrict__ lse) {
    using LY = LD<D, STAGES>;
    constexpr int ROWS = 8 * RG;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[STAGES], empty[STAGES];
    __shared__ int abort_word;
    __shared__ float2 warp_ml[DEC_WARPS][ROWS];          // (m, l) of every warp's rows
    __shared__ float2 cta_ml[ROWS];
    volatile int* abort_flag = &abort_word;
    const int warp = warp_index(), lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int bh = blockIdx.y;
    const int crank = CS > 1 ? static_cast<int>(cluster_ctarank()) : 0;

    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], DEC_WARPS); }
        abort_word = 0;
        fence_mbar_init();
    }
    __syncthreads();
    // (launched with programmatic stream serialization: nothing in device memory is touched before the previous kernel of
    // the stream has finished)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    int n = Nk;
    if (valid_len) { n = valid_len[bh / H]; n = n < 0 ? 0 : (n > Nk ? Nk : n); }
    // this CTA's share of the tiles that hold a valid key
    const int all = (n + LY::KEYS - 1) / LY::KEYS;
    const int first = CS > 1 ? static_cast<int>(static_cast<int64_t>(all) * crank / CS) : 0;
    const int ntiles = (CS > 1 ? static_cast<int>(static_cast<int64_t>(all) * (crank + 1) / CS) : all) - first;

    float o[D / 8][4];
    float m[RG], l[RG];
    if (warp == DEC_WARPS) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            bool ok = true;
            int issued = 0;
            prefetch_tensormap(&tmK); prefetch_tensormap(&tmV);
            for (int j = 0; j < ntiles; ++j) {
                const int s = j % STAGES;
                ok = bounded_wait(&empty[s], ((j / STAGES) & 1) ^ 1, abort_flag, status, 0x900);
                if (!ok) break;
                uint8_t* kt = base + s * 2 * LY::TILE_BYTES;
                mbar_arrive_expect_tx(&full[s], 2 * LY::TILE_BYTES);
#pragma unroll
                for (int c = 0; c < D / 64; ++c) tma_load_3d(kt + c * LY::KEYS * 128, &tmK, &full[s], c * 64, (first + j) * LY::KEYS, bh);
#pragma unroll
                for (int c = 0; c < D / 64; ++c)
                    tma_load_3d(kt + LY::TILE_BYTES + c * LY::KEYS * 128, &tmV, &full[s], c * 64, (first + j) * LY::KEYS, bh);
                issued = j + 1;
            }
            if (!ok)
                for (int j = issued > STAGES ? issued - STAGES : 0; j < issued; ++j) drain_wait(&full[j % STAGES], (j / STAGES) & 1);
        }
    } else {
        // ------------------------------------------------------------ logits, softmax, attend
        // Q as the left operand: slice k of 16 features, rows g and g + 8, feature pairs at 2 t and 2 t + 8
        uint32_t qa[D / 16][4];
#pragma unroll
        for (int k = 0; k < D / 16; ++k)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int row = g + (e & 1) * 8;
                qa[k][e] = (e & 1) < RG && row < Nq
                               ? *reinterpret_cast<const uint32_t*>(Q + (static_cast<int64_t>(bh) * Nq + row) * D + k * 16 + (e >> 1) * 8 + 2 * t)
                               : 0u;
            }
        // keys that rows g and g + 8 see
        int nrow[RG];
#pragma unroll
        for (int r = 0; r < RG; ++r) {
            const long long lim = static_cast<long long>(g + 8 * r) + 1 + Nk - Nq;
            nrow[r] = causal && lim < n ? (lim < 0 ? 0 : static_cast<int>(lim)) : n;
            m[r] = -INFINITY;
            l[r] = 0.f;
        }
        const long long lim0 = 1ll + Nk - Nq;            // keys that every row sees
        const int nmin = causal && lim0 < n ? (lim0 < 0 ? 0 : static_cast<int>(lim0)) : n;
#pragma unroll
        for (int i = 0; i < D / 8; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[i][e] = 0.f;
        bool ok = true;
        constexpr int NT = LY::WKEYS / 8;                // logit blocks of eight keys
        // ldmatrix addresses: lane i gives row i % 8 (+ 8) of one of four 8 x 8 blocks.  K: blocks (keys 0-7, features 0-7),
        // (0-7, 8-15), (8-15, 0-7), (8-15, 8-15); V (transposed): (keys 0-7, columns 0-7), (8-15, 0-7), (0-7, 8-15), (8-15, 8-15)
        const int krow = warp * LY::WKEYS + (lane & 7) + ((lane >> 4) & 1) * 8, kchunk = (lane >> 3) & 1;
        const int vrow = warp * LY::WKEYS + (lane & 7) + ((lane >> 3) & 1) * 8, vchunk = (lane >> 4) & 1;
        for (int j = 0; j < ntiles; ++j) {
            const int s = j % STAGES;
            ok = warp_wait(&full[s], (j / STAGES) & 1, abort_flag, status, 0x910);
            if (!ok) break;
            const uint32_t ks = smem_u32(base + s * 2 * LY::TILE_BYTES), vs = ks + LY::TILE_BYTES;
            float c[NT][4];
#pragma unroll
            for (int i = 0; i < NT; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) c[i][e] = 0.f;
#pragma unroll
            for (int k = 0; k < D / 16; ++k)
#pragma unroll
                for (int i = 0; i < NT; i += 2) {
                    const int row = krow + i * 8, chunk = (k % 4) * 2 + kchunk;
                    uint32_t b[4];
                    ldsm4(ks + (k / 4) * LY::KEYS * 128 + row * 128 + ((chunk ^ (row & 7)) << 4), b);
                    mma16(c[i], qa[k], b[0], b[1]);
                    mma16(c[i + 1], qa[k], b[2], b[3]);
                }
            // base-2 logits; keys that a row does not see take no part
            const int key0 = (first + j) * LY::KEYS + warp * LY::WKEYS;
            const bool masked = key0 + LY::WKEYS > nmin;
            float mx[RG];
#pragma unroll
            for (int r = 0; r < RG; ++r) {
                mx[r] = -INFINITY;
#pragma unroll
                for (int i = 0; i < NT; ++i)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float x = c[i][2 * r + e] * scale_log2e;
                        if (masked && key0 + i * 8 + 2 * t + e >= nrow[r]) x = -INFINITY;
                        c[i][2 * r + e] = x;
                        mx[r] = fmaxf(mx[r], x);
                    }
                mx[r] = quad_max(mx[r]);
            }
            bool grown = mx[0] > m[0];
            if (RG == 2) grown = grown || mx[RG - 1] > m[RG - 1];
            if (__any_sync(0xffffffffu, grown)) {
#pragma unroll
                for (int r = 0; r < RG; ++r) {
                    const float mn = fmaxf(m[r], mx[r]);
                    const float a = mn == -INFINITY ? 1.f : ex2_approx(m[r] - mn);
                    m[r] = mn;
                    l[r] *= a;
#pragma unroll
                    for (int i = 0; i < D / 8; ++i) { o[i][2 * r] *= a; o[i][2 * r + 1] *= a; }
                }
            }
#pragma unroll
            for (int r = 0; r < RG; ++r) {
                const float ref = m[r] == -INFINITY ? 0.f : m[r];
#pragma unroll
                for (int i = 0; i < NT; ++i)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float p = ex2_approx(c[i][2 * r + e] - ref);
                        c[i][2 * r + e] = p;
                        l[r] += p;
                    }
            }
#pragma unroll
            for (int i = 0; i < NT; i += 2) {
                const uint32_t pa[4] = {pack_bf16x2(c[i][0], c[i][1]), RG == 2 ? pack_bf16x2(c[i][2], c[i][3]) : 0u,
                                        pack_bf16x2(c[i + 1][0], c[i + 1][1]), RG == 2 ? pack_bf16x2(c[i + 1][2], c[i + 1][3]) : 0u};
#pragma unroll
                for (int x = 0; x < D / 16; ++x) {
                    const int row = vrow + i * 8, chunk = (x % 4) * 2 + vchunk;
                    uint32_t b[4];
                    ldsm4_t(vs + (x / 4) * LY::KEYS * 128 + row * 128 + ((chunk ^ (row & 7)) << 4), b);
                    mma16(o[2 * x], pa, b[0], b[1]);
                    mma16(o[2 * x + 1], pa, b[2], b[3]);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[s]);
        }
        // (the row sums were kept per thread)
#pragma unroll
        for (int r = 0; r < RG; ++r) {
            l[r] += __shfl_xor_sync(0xffffffffu, l[r], 1);
            l[r] += __shfl_xor_sync(0xffffffffu, l[r], 2);
            if (!ok) l[r] = __int_as_float(0x7fc00000);
            if (t == 0) warp_ml[warp][g + 8 * r] = make_float2(m[r], l[r]);
        }
    }
    __syncthreads();                                     // every tile has been read: the ring's memory is free
    // ---------------------------------------------------------------- the four warps' parts: [warp][row][feature]
    float* part = reinterpret_cast<float*>(base);
    float* cta_o = part + DEC_WARPS * ROWS * D;          // [row][feature], for the cluster
    if (warp < DEC_WARPS) {
#pragma unroll
        for (int r = 0; r < RG; ++r)
#pragma unroll
            for (int i = 0; i < D / 8; ++i)
                *reinterpret_cast<float2*>(part + (warp * ROWS + g + 8 * r) * D + i * 8 + 2 * t) = make_float2(o[i][2 * r], o[i][2 * r + 1]);
    }
    __syncthreads();
    // (m, l, O) of two shares of a row's keys: m = max, l = sum of l_i 2^(m_i - m), O likewise
    for (int i = threadIdx.x; i < Nq * (D / 2); i += DEC_THREADS) {
        const int row = i / (D / 2), col = (i % (D / 2)) * 2;
        float mm = -INFINITY;
#pragma unroll
        for (int w = 0; w < DEC_WARPS; ++w) mm = fmaxf(mm, warp_ml[w][row].x);
        const float ref = mm == -INFINITY ? 0.f : mm;
        float ll = 0.f, x = 0.f, y = 0.f;
#pragma unroll
        for (int w = 0; w < DEC_WARPS; ++w) {
            const float2 ml = warp_ml[w][row];
            const float a = ex2_approx(ml.x - ref);
            const float2 v = *reinterpret_cast<const float2*>(part + (w * ROWS + row) * D + col);
            ll += ml.y * a; x += v.x * a; y += v.y * a;
        }
        if (CS == 1) {
            const float inv = ll > 0.f ? 1.f / ll : (ll == ll ? 0.f : ll);
            *reinterpret_cast<uint32_t*>(O + (static_cast<int64_t>(bh) * Nq + row) * D + col) = pack_bf16x2(x * inv, y * inv);
            if (lse && col == 0) lse[static_cast<int64_t>(bh) * Nq + row] = ll > 0.f ? (mm + log2f(ll)) * 0.6931471805599453f : -INFINITY;
        } else {
            *reinterpret_cast<float2*>(cta_o + row * D + col) = make_float2(x, y);
            if (col == 0) cta_ml[row] = make_float2(mm, ll);
        }
    }
    if (CS > 1) {
        cluster_sync_all();                              // every CTA's (m, l, O) is written
        const int pairs = Nq * (D / 2);
        const uint32_t ml_s = smem_u32(cta_ml), o_s = smem_u32(cta_o);
        for (int i = pairs * crank / CS + threadIdx.x; i < pairs * (crank + 1) / CS; i += DEC_THREADS) {
            const int row = i / (D / 2), col = (i % (D / 2)) * 2;
            float2 ml[CS], v[CS];
#pragma unroll
            for (int q = 0; q < CS; ++q) {
                ml[q] = ld_cluster_f32x2(mapa_shared(ml_s + row * 8, q));
                v[q] = ld_cluster_f32x2(mapa_shared(o_s + (row * D + col) * 4, q));
            }
            float mm = -INFINITY;
#pragma unroll
            for (int q = 0; q < CS; ++q) mm = fmaxf(mm, ml[q].x);
            const float ref = mm == -INFINITY ? 0.f : mm;
            float ll = 0.f, x = 0.f, y = 0.f;
#pragma unroll
            for (int q = 0; q < CS; ++q) {
                const float a = ex2_approx(ml[q].x - ref);
                ll += ml[q].y * a; x += v[q].x * a; y += v[q].y * a;
            }
            const float inv = ll > 0.f ? 1.f / ll : (ll == ll ? 0.f : ll);
            *reinterpret_cast<uint32_t*>(O + (static_cast<int64_t>(bh) * Nq + row) * D + col) = pack_bf16x2(x * inv, y * inv);
            if (lse && col == 0) lse[static_cast<int64_t>(bh) * Nq + row] = ll > 0.f ? (mm + log2f(ll)) * 0.6931471805599453f : -INFINITY;
        }
        cluster_sync_all();                              // nobody leaves while its memory is read
    }
}

template <int D, int RG, int CS, int STAGES>
int launch_decode(const Problem& p, cudaStream_t st) {
    using LY = LD<D, STAGES>;
    CUtensorMap tmK, tmV;
    const int BH = p.B * p.H;
    if (!make_map(&tmK, p.K, BH, p.Nk, D, LY::KEYS) || !make_map(&tmV, p.V, BH, p.Nk, D, LY::KEYS)) return FLAT_ERR_CUDA;
    auto kern = fused_decode_kernel<D, RG, CS, STAGES>;
    if (!ensure_dynamic_smem<fused_decode_kernel<D, RG, CS, STAGES>>(LY::SMEM_BYTES)) return FLAT_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CS, BH);
    cfg.blockDim = dim3(DEC_THREADS);
    cfg.dynamicSmemBytes = LY::SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = CS; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = CS > 1 ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, tmK, tmV, static_cast<const __nv_bfloat16*>(p.Q), static_cast<__nv_bfloat16*>(p.O), p.H,
                                             p.Nq, p.Nk, p.scale * 1.4426950408889634f, p.k_valid_len, p.causal, p.status, p.lse);
    return e == cudaSuccess ? FLAT_OK : FLAT_ERR_CUDA;
}

// How many CTAs share a head, and how deep their rings are.  One round of two CTAs per SM streams at full rate, so the widest split that
// stays within it; up to two rounds where a CTA still reads a megabyte, which evens out key counts that differ between the batches
// (B16 H16 1 x 8192, d = 128, 25 to 100 % filled: 6 % less time in halves; short ones
// pay for their set-up: 512 keys in halves 15.2 us against 11.7).  Sixteen, more than the portable cluster size, only while every CTA
// has an SM of its own (4 heads x 32768 keys: eight CTAs a head 20.5 us).  Six stages where that is so (8 heads x 32768: 32.2 us
// against 35.9 with three).
template <int D, int RG>
int launch_decode_split(const Problem& p, cudaStream_t st) {
    constexpr int KEYS = LD<D, 3>::KEYS;
    const int64_t heads = static_cast<int64_t>(p.B) * p.H, sms = device_sm_count();
    auto fits = [&](int cs) {
        if (p.Nk < 2 * cs * KEYS) return false;
        if (cs == 16) return heads * 16 <= sms;
        return heads * cs <= 2 * sms || (heads * cs <= 4 * sms && static_cast<int64_t>(p.Nk) * D * 4 >= cs * (1ll << 20));
    };
    if (fits(16)) {
        // (the shared-memory limit has to be raised before the device is asked)
        const int fit = ensure_dynamic_smem<fused_decode_kernel<D, RG, 16, 6>>(LD<D, 6>::SMEM_BYTES)
                            ? clusters_of_sixteen<fused_decode_kernel<D, RG, 16, 6>>(DEC_THREADS, LD<D, 6>::SMEM_BYTES) : 0;
        if (heads <= fit) {
            const int rc = launch_decode<D, RG, 16, 6>(p, st);
            if (rc == FLAT_OK) return rc;
            cudaGetLastError();                          // (refused: eight)
        }
    }
    if (fits(8)) return heads * 8 <= sms ? launch_decode<D, RG, 8, 6>(p, st) : launch_decode<D, RG, 8, 3>(p, st);
    if (fits(4)) return heads * 4 <= sms ? launch_decode<D, RG, 4, 6>(p, st) : launch_decode<D, RG, 4, 3>(p, st);
    if (fits(2)) return launch_decode<D, RG, 2, 3>(p, st);
    return launch_decode<D, RG, 1, 3>(p, st);
}

}  // namespace

bool decode_applies(const Problem& p) {
    return p.dtype == FLAT_DTYPE_BF16 && (p.d == 64 || p.d == 128) && p.Nq <= DEC_MAX_Q && !p.bias && !p.block_mask;
}

int launch_fused_decode(const Problem& p, cudaStream_t st) {
    if (!decode_applies(p)) return FLAT_ERR_UNSUPPORTED;
    if (p.d == 64) return p.Nq <= 8 ? launch_decode_split<64, 1>(p, st) : launch_decode_split<64, 2>(p, st);
    return p.Nq <= 8 ? launch_decode_split<128, 1>(p, st) : launch_decode_split<128, 2>(p, st);
}

}  // namespace flat
