// Fused Logit-Softmax-Attend for small heads (bf16 in, fp32 accumulate, bf16 out; d = 16 and 32) on the sm_100a tensor
// cores: the paper's fused dataflow (Section 5, 5.1, 5.2), one 128-row query tile per CTA, keys streamed in tiles of BN.
//
// What bounds it: the chain of a step in the softmax warps -- logits seen, TMEM load, exponentials and splits, the wait for the last
// P V, stores, arrival -- with two of them on a scheduler to hide it: the exponential unit is busy 51 % of the time, the issue slots
// 49 %, the tensor pipe 19 % (counters, B64 H8 1000^2); and 1,024 CTAs are 3.5 rounds of the 296 that run at a time.  A (query, key)
// pair costs 4 d FLOP on the tensor pipe -- at d = 32 a quarter of what d = 128 has -- and one exponential whatever the head size
// (16 per clock and SM: 4.65e12 pairs/s on 148 SMs), so the contractions are nearly free and there is room for the accuracy that the FFMA kernel gave these head sizes
// (weights kept in fp32): a weight p goes to the second contraction as TWO bf16 numbers, its rounded head and the rounded
// remainder (together 17 bits of mantissa), each with an MMA of its own against the same V, and no exponential takes
// the polynomial.  Results then sit at the rounding of the bf16 output, as before.
//
// CTA = 192 threads, two CTAs per SM: warps 0-3 softmax (thread = query row = TMEM lane), warp 4 TMA producer, warp 5
// MMA issuer.  TMEM (256 columns): S 0..95, head of P 96..143, remainder of P 144..191, O 192...  A step is 96 keys and
// not 128 because the logits, both halves of P and O then have columns of their own: S(j+1) is computed while the
// softmax works on S(j), and two CTAs fit the 512 columns of an SM.  (At 128 keys P would have to overlay S, and every
// step would wait for MMA, softmax and MMA in turn.)
// Tiles in shared memory have rows of 2 d bytes with the swizzle of that width (64 or 32 bytes): the canonical K-major
// (Q, K) and MN-major (V) layouts with one panel.
// Measured: B16 H8 1000 x 1000 at d = 32: 65 us (2.0e12 pairs/s, 0.42 of the exponential unit) against 638 us of the FFMA kernel, which keeps the fp32 tensors and the calls with a bias.
// Reference maximum as in the two-tile kernel: exact on the first and on masked steps, kept otherwise, a step whose row
// sum passes 2^40 is redone with a fresh one.  A row that does not come out finite (infinite or very large values) is computed
// again without the split (plain_rows).  Every wait is bounded; on expiry the CTA ends cleanly and reports a code.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "flat_internal.cuh"
#include "ptx_sm100.cuh"
#include "tc_common.cuh"

namespace flat {

using namespace ptx;
using namespace tc;

namespace {

constexpr int BM = 128;              // query rows per CTA
constexpr int BN = 96;               // keys per step
constexpr int STAGES = 4;            // ring depth of K and of V
constexpr int SMALL_THREADS = 192;
constexpr float OVERFLOW_SUM = 1.0995116e12f;   // 2^40

template <int D> struct LS {
    static constexpr int ROW_BYTES = 2 * D;
    static constexpr int Q_BYTES = BM * ROW_BYTES, KV_BYTES = BN * ROW_BYTES;   // multiples of 1024
    static constexpr int TILE_BYTES = Q_BYTES + 2 * STAGES * KV_BYTES;
    static constexpr int SMEM_BYTES = TILE_BYTES + 256 + 1024;
    static constexpr uint32_t S_COL = 0, P_COL = BN, R_COL = BN + BN / 2, O_COL = 2 * BN, TMEM_COLS = 256;
    static constexpr int Q_FULL = 0, K_FULL = 1, K_EMPTY = K_FULL + STAGES, V_FULL = K_EMPTY + STAGES, V_EMPTY = V_FULL + STAGES,
                         S_FULL = V_EMPTY + STAGES, S_FREE = S_FULL + 1, P_FULL = S_FREE + 1, PV_DONE = P_FULL + 1, NUM_BARS = PV_DONE + 1;
    static_assert(KV_BYTES % 1024 == 0 && O_COL + D <= TMEM_COLS, "layout");
};

// Shared-memory matrix descriptor of a one-panel tile with rows of 2 D bytes swizzled over that width; the distance
// between groups of eight rows (K-major: rows; MN-major: contraction indices) is 16 D bytes.
template <int D>
__device__ __forceinline__ uint64_t small_desc(uint32_t smem_addr) {
    return static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4) | (1ull << 16) | (static_cast<uint64_t>(16 * D >> 4) << 32) |
           (1ull << 46) | ((D == 32 ? 4ull : 6ull) << 61);
}

// p_i = 2^(s_i * scale + neg_m) of one row; heads to TMEM at p_addr, remainders at r_addr (both packed bf16); returns the
// fp32 sum of the p.  TAIL: only the first `nvalid` columns take part.
template <bool TAIL, typename BeforeStore>
__device__ __forceinline__ float exp_store_split(const uint32_t (&s)[BN], float scale_log2e, float neg_m, uint32_t p_addr,
                                                 uint32_t r_addr, int nvalid, BeforeStore&& before_store) {
    uint64_t sum0 = 0ull, sum1 = 0ull;
    const uint64_t scale2 = pack2(scale_log2e, scale_log2e), neg_m2 = pack2(neg_m, neg_m);
#pragma unroll
    for (int c = 0; c < BN / 32; ++c) {
        float p[32];
#pragma unroll
        for (int i = 0; i < 32; i += 2)
            unpack2(fma2(pack2(__uint_as_float(s[c * 32 + i]), __uint_as_float(s[c * 32 + i + 1])), scale2, neg_m2), p[i], p[i + 1]);
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            p[i] = ex2_approx(p[i]);
            if (TAIL && c * 32 + i >= nvalid) p[i] = 0.f;
        }
        uint32_t hi[16], lo[16];
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
            const uint64_t p01 = pack2(p[i], p[i + 1]), p23 = pack2(p[i + 2], p[i + 3]);
            sum0 = add2(sum0, p01);
            sum1 = add2(sum1, p23);
            hi[i / 2] = pack_bf16x2(p[i], p[i + 1]);
            hi[i / 2 + 1] = pack_bf16x2(p[i + 2], p[i + 3]);
            float r0, r1, r2, r3;
            unpack2(sub2(p01, pack2(__uint_as_float(hi[i / 2] << 16), __uint_as_float(hi[i / 2] & 0xffff0000u))), r0, r1);
            unpack2(sub2(p23, pack2(__uint_as_float(hi[i / 2 + 1] << 16), __uint_as_float(hi[i / 2 + 1] & 0xffff0000u))), r2, r3);
            lo[i / 2] = pack_bf16x2(r0, r1);
            lo[i / 2 + 1] = pack_bf16x2(r2, r3);
        }
        if (c == 0) before_store();
        tmem_st_x16(p_addr + c * 16, hi);
        tmem_st_x16(r_addr + c * 16, lo);
    }
    float a, b, cc, d;
    unpack2(sum0, a, b);
    unpack2(sum1, cc, d);
    return (a + b) + (cc + d);
}

template <int D>
__global__ void __launch_bounds__(SMALL_THREADS, 2)
fused_small_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ CUtensorMap tmV, const __nv_bfloat16* Q, const __nv_bfloat16* K, const __nv_bfloat16* V,
                   __nv_bfloat16* O, int H, int Nq, int Nk, float scale_log2e, const int32_t* __restrict__ valid_len, int coff, int32_t* status,
                   float* __restrict__ lse) {
    using LY = LS<D>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* Qs = base;
    uint8_t* Ks = Qs + LY::Q_BYTES;
    uint8_t* Vs = Ks + STAGES * LY::KV_BYTES;
    uint64_t* bars = reinterpret_cast<uint64_t*>(base + LY::TILE_BYTES);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + LY::NUM_BARS);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    // Roles by an index that the compiler knows to be the same in all lanes, the softmax warps by one that it does not; they wait by
    // whole warps, the issuer's lanes one by one (us, all known and by whole warps / so: B2 H8 16K^2 d 32 1,598 / 1,535, d 16 1,570 /
    // 1,519, B16 H8 1000^2 64.6 / 63.0 and 62.9 / 61.7; the softmax warps' waits lane by lane, too: d 16 1,548).
    const int role = warp_index(), warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bh = blockIdx.y;
    // (causal: the last rows see the most keys, so they start first)
    const int row0 = static_cast<int>(coff < (1 << 29) ? gridDim.x - 1 - blockIdx.x : blockIdx.x) * BM;

    if (threadIdx.x == 128) {
        for (int i = 0; i < LY::NUM_BARS; ++i) mbar_init(&bars[i], (i == LY::S_FREE || i == LY::P_FULL) ? 4 : 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0) { tmem_alloc(tmem_slot, LY::TMEM_COLS); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // (launched with programmatic stream serialization: the next kernel of the stream may set itself up from here on,
    // and nothing in device memory is touched before the previous one has finished)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    int n = Nk;
    if (valid_len) { n = valid_len[bh / H]; n = n < 0 ? 0 : (n > Nk ? Nk : n); }
    {
        const long long lim = static_cast<long long>(row0) + BM + coff;      // (coff = Nk - Nq under the causal mask, else 2^30)
        if (lim < n) n = lim < 0 ? 0 : static_cast<int>(lim);
    }
    const int ntiles = (n + BN - 1) / BN;

    if (role == 4) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0 && ntiles > 0) {
            prefetch_tensormap(&tmQ); prefetch_tensormap(&tmK); prefetch_tensormap(&tmV);
            mbar_arrive_expect_tx(&bars[LY::Q_FULL], LY::Q_BYTES);
            tma_load_3d(Qs, &tmQ, &bars[LY::Q_FULL], 0, row0, bh);
            bool ok = true;
            int k_issued = 0, v_issued = 0;
            for (int j = 0; j < ntiles && ok; ++j) {
                const int s = j % STAGES;
                const uint32_t ph = ((j / STAGES) & 1) ^ 1;
                ok = bounded_wait(&bars[LY::K_EMPTY + s], ph, abort_flag, status, 0x800 + s);
                if (!ok) break;
                mbar_arrive_expect_tx(&bars[LY::K_FULL + s], LY::KV_BYTES);
                tma_load_3d(Ks + s * LY::KV_BYTES, &tmK, &bars[LY::K_FULL + s], 0, j * BN, bh);
                k_issued = j + 1;
                ok = bounded_wait(&bars[LY::V_EMPTY + s], ph, abort_flag, status, 0x810 + s);
                if (!ok) break;
                mbar_arrive_expect_tx(&bars[LY::V_FULL + s], LY::KV_BYTES);
                tma_load_3d(Vs + s * LY::KV_BYTES, &tmV, &bars[LY::V_FULL + s], 0, j * BN, bh);
                v_issued = j + 1;
            }
            if (!ok) {
                drain_wait(&bars[LY::Q_FULL], 0);
                for (int j = k_issued > STAGES ? k_issued - STAGES : 0; j < k_issued; ++j)
                    drain_wait(&bars[LY::K_FULL + j % STAGES], (j / STAGES) & 1);
                for (int j = v_issued > STAGES ? v_issued - STAGES : 0; j < v_issued; ++j)
                    drain_wait(&bars[LY::V_FULL + j % STAGES], (j / STAGES) & 1);
            }
        }
    } else if (role == 5) {
        // ------------------------------------------------------------ MMA issuer (whole warp walks, one lane issues)
        if (ntiles > 0) {
            constexpr uint32_t IDESC_S = make_idesc_bf16(BM, BN, 0, 0);
            constexpr uint32_t IDESC_PV = make_idesc_bf16(BM, D, 0, 1);
            const uint64_t q_desc = small_desc<D>(smem_u32(Qs)), k_desc = small_desc<D>(smem_u32(Ks)), v_desc = small_desc<D>(smem_u32(Vs));
            bool ok = true;
            auto wait = [&](int bar, uint32_t parity, int code) {
                if (ok) ok = __all_sync(0xffffffffu, bounded_wait(&bars[bar], parity, abort_flag, status, code));
                if (ok) tc_fence_after();
            };
            auto issue_s = [&](int j) {
                const int s = j % STAGES;
                if (elect_one()) {
                    const uint64_t kd = k_desc + static_cast<uint64_t>((s * LY::KV_BYTES) >> 4);
#pragma unroll
                    for (int k = 0; k < D / 16; ++k) mma_ss(tmem + LY::S_COL, q_desc + 2 * k, kd + 2 * k, IDESC_S, k > 0);
                    tc_commit(&bars[LY::S_FULL]);
                    tc_commit(&bars[LY::K_EMPTY + s]);
                }
                __syncwarp();
            };
            auto issue_pv = [&](int j) {
                const int s = j % STAGES;
                if (elect_one()) {
                    const uint64_t vd = v_desc + static_cast<uint64_t>((s * LY::KV_BYTES) >> 4);
#pragma unroll
                    for (int k = 0; k < BN / 16; ++k) {
                        const uint64_t vk = vd + static_cast<uint64_t>((k * 16 * LY::ROW_BYTES) >> 4);
                        mma_ts(tmem + LY::O_COL, tmem + LY::R_COL + k * 8, vk, IDESC_PV, (j > 0 || k > 0));
                        mma_ts(tmem + LY::O_COL, tmem + LY::P_COL + k * 8, vk, IDESC_PV, 1);
                    }
                    tc_commit(&bars[LY::PV_DONE]);
                    tc_commit(&bars[LY::V_EMPTY + s]);
                }
                __syncwarp();
            };
            wait(LY::Q_FULL, 0, 0x820);
            wait(LY::K_FULL, 0, 0x821);
            if (ok) issue_s(0);
            for (int j = 0; j < ntiles && ok; ++j) {
                if (j + 1 < ntiles) {
                    wait(LY::K_FULL + (j + 1) % STAGES, ((j + 1) / STAGES) & 1, 0x822);
                    wait(LY::S_FREE, j & 1, 0x823);
                    if (ok) issue_s(j + 1);
                }
                wait(LY::V_FULL + j % STAGES, (j / STAGES) & 1, 0x824);
                wait(LY::P_FULL, j & 1, 0x825);
                if (ok) issue_pv(j);
            }
        }
    } else {
        // ------------------------------------------------------------ softmax + epilogue (warps 0-3)
        const int row = row0 + warp * 32 + lane;
        const uint32_t tl = tmem + (static_cast<uint32_t>(warp * 32) << 16);
        const bool neg_scale = scale_log2e < 0.f;
        float m_ref = -INFINITY, l = 0.f;
        bool ok = true;
        const long long rlim = static_cast<long long>(row) + 1 + coff;
        const int nrow = rlim < n ? (rlim < 0 ? 0 : static_cast<int>(rlim)) : n;
        const int nrow_min = __shfl_sync(0xffffffffu, nrow, 0);
        for (int j = 0; j < ntiles; ++j) {
            ok = warp_wait(&bars[LY::S_FULL], j & 1, abort_flag, status, 0x830);
            if (!ok) break;
            tc_fence_after();
            uint32_t s[BN];
#pragma unroll
            for (int c = 0; c < BN / 32; ++c) tmem_ld_x32(tl + LY::S_COL + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[c * 32]));
            tc_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars[LY::S_FREE]);
            const int col0 = j * BN;
            const bool tail = col0 + BN > nrow_min;      // (warp-uniform) some row has masked keys in this step
            const int nvalid = nrow > col0 ? (nrow - col0 < BN ? nrow - col0 : BN) : 0;
            if (tail) {
                const uint32_t excl = __float_as_uint(neg_scale ? INFINITY : -INFINITY);
#pragma unroll
                for (int i = 0; i < BN; ++i) if (i >= nvalid) s[i] = excl;
            }
            // O += P(j-1) V must have read both halves of P(j-1) before they are overwritten
            bool pv_waited = j == 0;
            auto wait_p_free = [&]() {
                if (!pv_waited) {
                    ok = warp_wait(&bars[LY::PV_DONE], (j - 1) & 1, abort_flag, status, 0x831);
                    pv_waited = true;
                    tc_fence_after();
                }
            };
            bool careful = (j == 0) || tail;
            float lt = 0.f;
            if (!careful) {
                lt = exp_store_split<false>(s, scale_log2e, -m_ref, tl + LY::P_COL, tl + LY::R_COL, BN, wait_p_free);
                if (!ok) break;
                careful = __any_sync(0xffffffffu, !(lt <= OVERFLOW_SUM));
            }
            if (careful) {
                float mx = -INFINITY;
                if (nvalid > 0) {
                    float e0 = __uint_as_float(s[0]), e1 = __uint_as_float(s[1]);
#pragma unroll
                    for (int i = 2; i < BN; i += 2) {
                        e0 = neg_scale ? fminf(e0, __uint_as_float(s[i])) : fmaxf(e0, __uint_as_float(s[i]));
                        e1 = neg_scale ? fminf(e1, __uint_as_float(s[i + 1])) : fmaxf(e1, __uint_as_float(s[i + 1]));
                    }
                    mx = (neg_scale ? fminf(e0, e1) : fmaxf(e0, e1)) * scale_log2e;
                }
                if (__any_sync(0xffffffffu, mx > m_ref + RESCALE_THRESHOLD)) {
                    const float m_new = fmaxf(m_ref, mx);
                    const float alpha = m_new == -INFINITY ? 1.f : ex2_approx(m_ref - m_new);   // 0 on the row's first keys
                    l *= alpha;
                    if (j > 0) {
                        wait_p_free();
                        if (!ok) break;
                        uint32_t r[16];
#pragma unroll
                        for (int c = 0; c < D / 16; ++c) {
                            tmem_ld_x16(tl + LY::O_COL + c * 16, r);
                            tc_wait_ld();
#pragma unroll
                            for (int i = 0; i < 16; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * alpha);
                            tmem_st_x16(tl + LY::O_COL + c * 16, r);
                        }
                    }
                    m_ref = m_new;
                }
                lt = exp_store_split<true>(s, scale_log2e, m_ref == -INFINITY ? 0.f : -m_ref, tl + LY::P_COL, tl + LY::R_COL, nvalid, wait_p_free);
                if (!ok) break;
            }
            l += lt;
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars[LY::P_FULL]);
        }
        if (ok && ntiles > 0) ok = warp_wait(&bars[LY::PV_DONE], (ntiles - 1) & 1, abort_flag, status, 0x832);
        if (ok) {
            const float inv = l > 0.f ? 1.f / l : 0.f;
            if (lse && row < Nq)
                lse[static_cast<int64_t>(bh) * Nq + row] = l > 0.f ? (m_ref + log2f(l)) * 0.6931471805599453f : -INFINITY;
            tc_fence_after();
            __nv_bfloat16* orow = O + (static_cast<int64_t>(bh) * Nq + row) * D;
            uint64_t zero[2] = {0ull, 0ull};             // (NaN once a result is not finite)
#pragma unroll
            for (int c = 0; c < D / 16; ++c) {
                uint32_t r[16];
                if (ntiles > 0) {
                    tmem_ld_x16(tl + LY::O_COL + c * 16, r);
                    tc_wait_ld();
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i) r[i] = 0u;      // no valid key: O = 0
                }
#pragma unroll
                for (int i = 0; i < 16; i += 2)
                    zero[(i >> 1) & 1] = fma2(pack2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), 0ull, zero[(i >> 1) & 1]);
                if (row < Nq) {
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        uint4 w;
                        w.x = pack_bf16x2(__uint_as_float(r[8 * v + 0]) * inv, __uint_as_float(r[8 * v + 1]) * inv);
                        w.y = pack_bf16x2(__uint_as_float(r[8 * v + 2]) * inv, __uint_as_float(r[8 * v + 3]) * inv);
                        w.z = pack_bf16x2(__uint_as_float(r[8 * v + 4]) * inv, __uint_as_float(r[8 * v + 5]) * inv);
                        w.w = pack_bf16x2(__uint_as_float(r[8 * v + 6]) * inv, __uint_as_float(r[8 * v + 7]) * inv);
                        *reinterpret_cast<uint4*>(orow + c * 16 + v * 8) = w;
                    }
                }
            }
            float z0, z1;
            unpack2(add2(zero[0], zero[1]), z0, z1);
            const unsigned again = __ballot_sync(0xffffffffu, row < Nq && z0 + z1 != 0.f);
            if (again)
                plain_rows<__nv_bfloat16, D>(again, static_cast<int64_t>(bh) * Nq + row0 + warp * 32, nrow, Q, K + static_cast<int64_t>(bh) * Nk * D,
                                             V + static_cast<int64_t>(bh) * Nk * D, O, lse, scale_log2e);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, LY::TMEM_COLS);
}

// bf16 tensor [BH, N, D] as {D, N, BH}; box = D x rows x 1, rows of 2 D bytes swizzled over that width.
template <int D>
bool small_map(CUtensorMap* m, const void* ptr, int BH, int N, int rows) {
    EncodeTiledFn enc = get_encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(D), static_cast<cuuint64_t>(N), static_cast<cuuint64_t>(BH)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(D) * 2, static_cast<cuuint64_t>(N) * D * 2};
    cuuint32_t box[3] = {static_cast<cuuint32_t>(D), static_cast<cuuint32_t>(rows), 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, D == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int D>
int launch_small_d(const Problem& p, cudaStream_t st) {
    using LY = LS<D>;
    CUtensorMap tmQ, tmK, tmV;
    const int BH = p.B * p.H;
    if (!small_map<D>(&tmQ, p.Q, BH, p.Nq, BM) || !small_map<D>(&tmK, p.K, BH, p.Nk, BN) || !small_map<D>(&tmV, p.V, BH, p.Nk, BN))
        return FLAT_ERR_CUDA;
    if (!ensure_dynamic_smem<fused_small_kernel<D>>(LY::SMEM_BYTES)) return FLAT_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((p.Nq + BM - 1) / BM, BH);
    cfg.blockDim = dim3(SMALL_THREADS);
    cfg.dynamicSmemBytes = LY::SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, fused_small_kernel<D>, tmQ, tmK, tmV, static_cast<const __nv_bfloat16*>(p.Q),
                                             static_cast<const __nv_bfloat16*>(p.K), static_cast<const __nv_bfloat16*>(p.V),
                                             static_cast<__nv_bfloat16*>(p.O), p.H, p.Nq, p.Nk, p.scale * 1.4426950408889634f, p.k_valid_len,
                                             p.causal ? p.Nk - p.Nq : (1 << 30), p.status, p.lse);
    return e == cudaSuccess ? FLAT_OK : FLAT_ERR_CUDA;
}

}  // namespace

bool small_applies(const Problem& p) {
    // (2^30 keys: the offset that stands for "no causal mask"; what lies beyond is the FFMA kernel's)
    return p.dtype == FLAT_DTYPE_BF16 && (p.d == 16 || p.d == 32) && !p.bias && !p.block_mask && p.Nk <= (1 << 30);
}

int launch_fused_small(const Problem& p, cudaStream_t st) {
    if (!small_applies(p)) return FLAT_ERR_UNSUPPORTED;
    return p.d == 32 ? launch_small_d<32>(p, st) : launch_small_d<16>(p, st);
}

}  // namespace flat
