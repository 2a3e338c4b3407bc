// Fused Logit-Softmax-Attend for d = 128 (bf16 in, fp32 accumulate, bf16 out): two query tiles of 128 rows per CTA, keys in
// steps of 64 with the logits of the step after next computed ahead.
//
// Paper mapping (Section 5, 5.1, 5.2): shared outer loops = items of (batch, head) and a slab of 256 query rows (R-granularity);
// Logit and Attend interleaved over the key steps with the streaming softmax between them (a reference maximum and a
// running sum replace the paper's full-row slice on chip; same function).
//
// What bounds it: the tensor pipe.  The two outputs take 256 of TMEM's 512 columns, so there is room for 256 columns of
// logits.  With one 128-key tile per query tile in them (fused_tc2_kernel), the weights have to overlay the logits and a
// tile's chain runs in series -- softmax, O += P V, next logits, 3,800 cycles of which the pipe works 2 x 1024 for both
// tiles.  With steps of 64 keys every query tile has TWO logit buffers: S(j + 1) is there when softmax(j) is done, and
// O += P(j) V and S(j + 2), which takes P(j)'s columns, have a whole softmax step to run in.  The price is that a
// logit MMA of N = 64 with both operands in shared memory takes 48 cycles where its arithmetic takes 32 (A alone is 4 KB of
// a port of 128 bytes a cycle): 1280 cycles of the pipe per 64 keys of both tiles, against 1024.
// Measured, against fused_tc2_kernel on the same GPU in the first 20 ms of launches (us): B4 H16 4096^2 460 -> 428, causal 347 ->
// 256; H8 64K causal 7,780 -> 6,350 (1,386 TFLOP/s; a cuBLAS GEMM of 8192^3 reaches 1,630 in a burst); B2 H16 3000 causal 120 ->
// 97; B32 H16 512^2 110 -> 106.  Since then (waits by whole warps and a uniform warp index; items taken over or dealt) 428 -> 418, 257 ->
// 244, 6,224 -> 6,052, 84 -> 78 (with lse), 90 -> 84.  After 20 ms the power cap takes the clock down: in a second of launches H8 64K causal takes 7,160
// (1,229 TFLOP/s at 1,462 MHz; cuBLAS sustained 1,376), B4 H16 4096^2 498 at 1,500 MHz.  The causal gain is also the order: the
// longest slabs first, so that short ones are left at the end.
//
// CTA = 384 threads: warps 0-3 / 4-7 softmax of tile A / B (thread = row = TMEM lane), warp 8 TMA producer, warps 9 / 10 MMA
// issuers of tile A / B (one elected lane), warp 11 idle (it completes the warpgroup for the register hand-over).
// TMEM columns: S(t, b) 128 t + 64 b (b = step parity), P over the first 32 of them, O_t 256 + 128 t.
// The softmax takes no row maximum after the first step: any reference gives the exact softmax, and a step whose row sum
// passes 2^40 is redone with a fresh maximum.  One exponential in four goes through a polynomial on the FMA pipe.
// ITEMS: a CTA has one item (batch, head, slab of 256 rows), several that are dealt in advance, or its own and those it takes over
// from CTAs that have not started; the rings and barriers go on from one to the next.
// VL: packed batches (Q, O [total_q, H, d], K, V [total_k, H, d]), an item per (sequence, head, slab of the longest sequence): a
// CTA each, or (sequences of one length) dealt.
// Every wait is bounded (tc_common.cuh); on expiry the CTA aborts cleanly and reports a code.
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

constexpr int D = 128;
constexpr int BM = 128;              // rows per query tile (two tiles per CTA)
constexpr int BN = 64;               // keys per step
constexpr int THREADS = 384;
constexpr int POLY_LANE = 3;         // element index mod 4 that takes the polynomial (none: B4 H16 4096 keys 450 us against 428)
constexpr float OVERFLOW_SUM = 1.0995116e12f;   // 2^40

constexpr int Q_BYTES = BM * D * 2, KV_BYTES = BN * D * 2;
__host__ __device__ constexpr uint32_t S_COL(int t, int b) { return 128u * t + 64u * b; }
__host__ __device__ constexpr uint32_t O_COL(int t) { return 256u + 128u * t; }
// Ring depths and barriers.  BT: with two bias tiles per query tile (2: one twice as large), which take the room of two K and two V stages.
// S_FULL / P_FULL / PV_DONE [tile][step parity], each once every second step.  (One PV_DONE a tile is not enough: a warp ahead of
// the others of its tile has its last logits when O += P V of the third last step is done, and would take that one's parity for
// the last one's.)  B_FULL / B_EMPTY [step parity][tile]: the bias tile / the four softmax warps of the tile have read it.
// Q_EMPTY / O_FREE [tile], once an item: its logit MMAs are done with the Q tile / its four softmax warps have read the output.
// ITEM_FULL / ITEM_EMPTY [2]: the next item is known / read by the ten other warps.
template <int BT> struct Layout {
    static constexpr int KS = BT ? 3 : 5, VS = KS;
    static constexpr int BIAS_BYTES = BT == 2 ? BM * SHIFTED_WIDTH(D) * 2 : BM * BN * 2;   // a bias tile: 128 rows of 64 values (2: of 128)
    static constexpr int TILE_BYTES = 2 * Q_BYTES + (KS + VS) * KV_BYTES + (BT == 2 ? 2 : BT ? 4 : 0) * BIAS_BYTES;
    static constexpr int SMEM_BYTES = TILE_BYTES + 512 + 1024;
    static constexpr int Q_FULL = 0, K_FULL = 2, K_EMPTY = K_FULL + KS, V_FULL = K_EMPTY + KS, V_EMPTY = V_FULL + VS, S_FULL = V_EMPTY + VS,
                         P_FULL = S_FULL + 4, PV_DONE = P_FULL + 4, B_FULL = PV_DONE + 4, B_EMPTY = B_FULL + 4, Q_EMPTY = B_EMPTY + 4, O_FREE = Q_EMPTY + 2, ITEM_EMPTY = O_FREE + 2,
                         ITEM_FULL = ITEM_EMPTY + 2, NUM_BARS = ITEM_FULL + 2;
    static_assert(SMEM_BYTES <= 232448 && 32 + NUM_BARS * 8 + 8 <= 512, "shared memory");
};

// p_i = 2^(s_i * scale + neg_m) of 64 logits; bf16(p) to 32 TMEM columns at `p_addr`; returns the fp32 sum of the unrounded p.
// TAIL: only the first `nvalid` take part.
template <bool TAIL>
__device__ __forceinline__ float exp_store(const uint32_t (&s)[BN], float scale_log2e, float neg_m, uint32_t p_addr, int nvalid) {
    uint64_t sum0 = 0ull, sum1 = 0ull;
    const uint64_t scale2 = pack2(scale_log2e, scale_log2e), neg_m2 = pack2(neg_m, neg_m);
#pragma unroll
    for (int c = 0; c < BN / 32; ++c) {
        uint32_t pk[16];
        float p[32];
#pragma unroll
        for (int i = 0; i < 32; i += 2)
            unpack2(fma2(pack2(__uint_as_float(s[c * 32 + i]), __uint_as_float(s[c * 32 + i + 1])), scale2, neg_m2), p[i], p[i + 1]);
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            p[i] = !TAIL && (i & 3) == POLY_LANE ? ex2_poly(p[i]) : ex2_approx(p[i]);
            if (TAIL && c * 32 + i >= nvalid) p[i] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
            sum0 = add2(sum0, pack2(p[i], p[i + 1]));
            sum1 = add2(sum1, pack2(p[i + 2], p[i + 3]));
            pk[i / 2] = pack_bf16x2(p[i], p[i + 1]);
            pk[i / 2 + 1] = pack_bf16x2(p[i + 2], p[i + 3]);
        }
        tmem_st_x16(p_addr + c * 16, pk);
    }
    float a, b, cc, d;
    unpack2(sum0, a, b);
    unpack2(sum1, cc, d);
    return (a + b) + (cc + d);
}

// s = s * scale * log2(e) + bias * log2(e), base-2 units; `brow`: shared-window address of the thread's 128-byte row of the bias
// tile, rx: the row's place in the swizzle.
// 2: `rx` is what the row is to be shifted by.
template <int BIAS>
__device__ __forceinline__ void add_bias(uint32_t (&s)[BN], float scale_log2e, uint32_t brow, int rx) {
    const uint64_t scale2 = pack2(scale_log2e, scale_log2e), log2e2 = pack2(1.4426950408889634f, 1.4426950408889634f);
    uint32_t two[8];
    auto piece = [&](int c, uint32_t& w0, uint32_t& w1, uint32_t& w2, uint32_t& w3) {
        asm volatile("ld.shared::cta.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w0), "=r"(w1), "=r"(w2), "=r"(w3) : "r"(brow + ((BIAS == 2 ? c : c ^ rx) << 4)) : "memory");
    };
    if (BIAS == 2) piece(0, two[4], two[5], two[6], two[7]);
#pragma unroll
    for (int c = 0; c < BN / 8; ++c) {
        uint32_t w[4];
        if (BIAS == 2) {
#pragma unroll
            for (int e = 0; e < 4; ++e) two[e] = two[4 + e];
            piece(c + 1, two[4], two[5], two[6], two[7]);
            shift8(two, rx, w);
        } else {
            piece(c, w[0], w[1], w[2], w[3]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int i = c * 8 + 2 * e;
            float a, b;
            unpack2(fma2(pack2(__uint_as_float(s[i]), __uint_as_float(s[i + 1])), scale2,
                         mul2(pack2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u)), log2e2)), a, b);
            s[i] = __float_as_uint(a);
            s[i + 1] = __float_as_uint(b);
        }
    }
}

__device__ __forceinline__ float row_extreme(const uint32_t (&s)[BN], bool smallest) {
    float e0 = __uint_as_float(s[0]), e1 = __uint_as_float(s[1]);
#pragma unroll
    for (int i = 2; i < BN; i += 2) {
        e0 = smallest ? fminf(e0, __uint_as_float(s[i])) : fmaxf(e0, __uint_as_float(s[i]));
        e1 = smallest ? fminf(e1, __uint_as_float(s[i + 1])) : fmaxf(e1, __uint_as_float(s[i + 1]));
    }
    return smallest ? fminf(e0, e1) : fmaxf(e0, e1);
}

// BIAS: the bias tiles (bf16, rows on 16-byte boundaries) come through TMA, one per query tile and step, two ahead.
struct Item {
    int bh, row0, n, nsteps, coff;                       // n: keys that any row of the slab sees; coff: Nk - Nq (2^30: no causal mask)
    int head, q_tok0, k_tok0, q_rows;                    // (packed batches)
};

enum { ONE_ITEM = 0, DEALT = 1, TAKEN_OVER = 2 };

template <bool VL, int BIAS, int ITEMS>
__global__ void __launch_bounds__(THREADS, 1)
fused_d128_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                  __nv_bfloat16* __restrict__ O, int BH, int H, int Nq, int Nk, float scale_log2e, const int32_t* __restrict__ valid_len,
                  int coff, int group, int32_t* status, const int32_t* __restrict__ cu_q, const int32_t* __restrict__ cu_k,
                  float* __restrict__ lse, const __grid_constant__ CUtensorMap tmBias = CUtensorMap{}, int bias_heads = 0,
                  int bias_batches = 0, const ShiftedBias sb = ShiftedBias{}) {
    using LY = Layout<BIAS>;
    constexpr bool MULTI = ITEMS != ONE_ITEM;
    constexpr int BIAS_BYTES = LY::BIAS_BYTES;
    constexpr int KS = LY::KS, VS = LY::VS;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* Qs = base;
    uint8_t* Ks = Qs + 2 * Q_BYTES;
    uint8_t* Vs = Ks + KS * KV_BYTES;
    uint8_t* Bs = Vs + VS * KV_BYTES;                    // (bias) [step parity][tile]
    uint8_t* next_item = base + LY::TILE_BYTES;          // two answers of 16 bytes
    uint64_t* bars = reinterpret_cast<uint64_t*>(next_item + 32);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + LY::NUM_BARS);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    // Roles go by an index that the compiler knows to be the same in all lanes, and so do the softmax warps where a CTA takes several
    // items (without it 12 % a step).  With one item a CTA it is better not known to them: H2 16K^2 214 -> 208 us, H16 2048^2 32.1 ->
    // 31.1, H8 4096^2 56.8 -> 55.9.
    const int role = warp_index(), warp = MULTI ? role : static_cast<int>(threadIdx.x >> 5), lane = threadIdx.x & 31;

    // (TAKEN_OVER) the r-th item, taken over from a CTA that had not started; -1: there was none, or the wait gave up.
    // The producer's one lane reads it by itself.
    auto take_item = [&](int r) {
        const int slot = (r - 1) & 1, full = smem_u32(&bars[LY::ITEM_FULL + slot]), aborts = smem_u32(const_cast<int*>(abort_flag));
        const uint32_t parity = ((r - 1) >> 1) & 1, answer = smem_u32(next_item) + 16 * slot;
        if (role == 8) {
            if (!bounded_wait_s(full, parity, aborts, status, 0xa50)) return -1;
            const int item = clc_answer(answer);
            fence_proxy_async_smem();
            return item;
        }
        if (!warp_wait(full, parity, aborts, status, 0xa51)) return -1;
        const int item = __shfl_sync(0xffffffffu, clc_answer(answer), 0);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars[LY::ITEM_EMPTY + slot]);
        __syncwarp();
        return item;
    };
    // The CTA's r-th item: (batch, head, slab of 256 rows).
    auto get_item = [&](int r, Item& it) -> bool {
        if (!MULTI && r > 0) return false;
        it.n = Nk;
        it.coff = coff;
        if (VL) {
            if (MULTI) {
                const unsigned pos = r * gridDim.x + blockIdx.x, slabs = (Nq + 2 * BM - 1) / (2 * BM);
                if (pos >= BH * slabs) return false;
                it.bh = pos / slabs;
                it.row0 = static_cast<int>(pos % slabs) * (2 * BM);
            } else {
                // the slabs of a sequence side by side; under the causal mask the last slabs (the longest) of all sequences first
                it.bh = group ? blockIdx.x : blockIdx.y;
                it.row0 = static_cast<int>(group ? gridDim.y - 1 - blockIdx.y : blockIdx.x) * (2 * BM);
            }
            const int s = it.bh / H;
            it.head = it.bh - s * H;
            const int q0 = cu_q[s], ql = cu_q[s + 1] - q0, k0 = cu_k[s], kl = cu_k[s + 1] - k0;
            if (!MULTI && it.row0 >= ql) return false;
            it.q_tok0 = q0 + it.row0; it.k_tok0 = k0; it.q_rows = ql - it.row0;
            it.n = kl < 0 || it.q_rows <= 0 ? 0 : kl;
            if (coff < (1 << 29)) it.coff = kl - ql;
        } else {
            // `group` heads at a time, their slabs side by side, the longest first under the causal mask
            const int slabs = (Nq + 2 * BM - 1) / (2 * BM), per = group * slabs;
            int pos = blockIdx.x;
            if (ITEMS == DEALT) {                        // (forth and back)
                const unsigned at = r * gridDim.x + ((r & 1) ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
                if (at >= static_cast<unsigned>(BH * slabs)) return false;
                pos = at;
            } else if (ITEMS == TAKEN_OVER && r > 0) {
                pos = take_item(r);
                if (pos < 0) return false;
            }
            const int first = pos / per * group, heads = BH - first < group ? BH - first : group, at = pos % per;
            it.bh = first + at % heads;
            it.row0 = (coff < (1 << 29) ? slabs - 1 - at / heads : at / heads) * (2 * BM);
            if (valid_len) { const int v = valid_len[it.bh / H]; it.n = v < 0 ? 0 : (v > Nk ? Nk : v); }
        }
        // Causal mask (coff = Nk - Nq; 2^30 = none): row r sees keys j < r + 1 + coff, so the last row bounds the slab's keys
        const long long lim = static_cast<long long>(it.row0) + 2 * BM + it.coff;
        if (lim < it.n) it.n = lim < 0 ? 0 : static_cast<int>(lim);
        it.nsteps = (it.n + BN - 1) / BN;
        return true;
    };
    // (bias, shifted) the slab's first row among all rows of the bias
    auto bias_row = [&](const Item& it) { return ((bias_batches ? it.bh / H : 0) * (bias_heads ? H : 1) + (bias_heads ? it.bh % H : 0)) * Nq + it.row0; };
    if (VL && !MULTI) {
        Item it;
        if (!get_item(0, it)) return;                    // (the whole CTA: nothing is set up yet)
    }

    if (threadIdx.x == 256) {
        for (int i = 0; i < LY::NUM_BARS; ++i)
            mbar_init(&bars[i], i >= LY::ITEM_FULL ? 1 : i >= LY::ITEM_EMPTY ? 10
                                : (i >= LY::P_FULL && i < LY::PV_DONE) || (i >= LY::B_EMPTY && i < LY::Q_EMPTY) || i >= LY::O_FREE ? 4
                                : (i >= LY::K_EMPTY && i < LY::V_FULL) || (i >= LY::V_EMPTY && i < LY::S_FULL) ? 2 : 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // (launched with programmatic stream serialization, packed batches aside: this set-up overlaps the tail of the previous
    // kernel of the stream, and nothing in device memory is touched before that one has finished)
    if (!VL) {
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        asm volatile("griddepcontrol.wait;" ::: "memory");
    }
    const uint32_t tmem = *tmem_slot;
    const uint32_t bars_s = smem_u32(bars), abort_s = smem_u32(const_cast<int*>(abort_flag));

    if (role >= 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
        if (role == 8) {
            // ------------------------------------------------------------ TMA producer
            if (lane == 0) {
                prefetch_tensormap(&tmQ); prefetch_tensormap(&tmK); prefetch_tensormap(&tmV);
                bool ok = true;
                int q_issued[2] = {0, 0}, k_issued = 0, v_issued = 0, b_issued = 0;
                Item it;
                int J0 = 0, q = 0;                       // key steps / items with keys so far
                auto load_q = [&](int t) {
                    if (MULTI) ok = ok && bounded_wait_s(bars_s + 8 * (LY::Q_EMPTY + t), (q & 1) ^ 1, abort_s, status, 0xa40 + t);
                    if (!ok) return;
                    mbar_arrive_expect_tx(&bars[LY::Q_FULL + t], Q_BYTES);
#pragma unroll
                    for (int c = 0; c < 2; ++c)
                        tma_load_3d(Qs + t * Q_BYTES + c * BM * 128, &tmQ, &bars[LY::Q_FULL + t], c * 64, VL ? it.head : it.row0 + t * BM, VL ? it.q_tok0 + t * BM : it.bh);
                    q_issued[t] = q + 1;
                };
                auto load_k = [&](int j) {
                    const int J = J0 + j, s = J % KS;
                    ok = ok && bounded_wait_s(bars_s + 8 * (LY::K_EMPTY + s), ((J / KS) & 1) ^ 1, abort_s, status, 0xa00 + s);
                    if (!ok) return;
                    mbar_arrive_expect_tx(&bars[LY::K_FULL + s], KV_BYTES);
#pragma unroll
                    for (int c = 0; c < 2; ++c)
                        tma_load_3d(Ks + s * KV_BYTES + c * BN * 128, &tmK, &bars[LY::K_FULL + s], c * 64, VL ? it.head : j * BN, VL ? it.k_tok0 + j * BN : it.bh);
                    k_issued = J + 1;
                };
                auto load_v = [&](int j) {
                    const int J = J0 + j, s = J % VS;
                    ok = ok && bounded_wait_s(bars_s + 8 * (LY::V_EMPTY + s), ((J / VS) & 1) ^ 1, abort_s, status, 0xa10 + s);
                    if (!ok) return;
                    mbar_arrive_expect_tx(&bars[LY::V_FULL + s], KV_BYTES);
#pragma unroll
                    for (int c = 0; c < 2; ++c)
                        tma_load_3d(Vs + s * KV_BYTES + c * BN * 128, &tmV, &bars[LY::V_FULL + s], c * 64, VL ? it.head : j * BN, VL ? it.k_tok0 + j * BN : it.bh);
                    v_issued = J + 1;
                };
                auto load_bias = [&](int j) {            // of both tiles
                    const int J = J0 + j;
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        const int s = BIAS == 2 ? t : 2 * (J & 1) + t;
                        ok = ok && bounded_wait_s(bars_s + 8 * (LY::B_EMPTY + s), ((BIAS == 2 ? J : J >> 1) & 1) ^ 1, abort_s, status, 0xa18 + t);
                        if (!ok) return;
                        mbar_arrive_expect_tx(&bars[LY::B_FULL + s], BIAS_BYTES);
                        if (BIAS == 2)
                            load_shifted_bias<SHIFTED_WIDTH(D)>(Bs + s * BIAS_BYTES, &tmBias, &bars[LY::B_FULL + s], bias_row(it) + t * BM, j * BN, Nk);
                        else
                            tma_load_4d(Bs + s * BIAS_BYTES, &tmBias, &bars[LY::B_FULL + s], j * BN, it.row0 + t * BM, bias_heads ? it.bh % H : 0, bias_batches ? it.bh / H : 0);
                        b_issued = 2 * J + t + 1;
                    }
                };
                int asked = 0;
                for (int r = 0; ok && get_item(r, it); ++r) {
                    if (it.nsteps > 0) {
                        load_q(0);
                        load_k(0);
                        load_q(1);
                        if (BIAS) load_bias(0);
                        if (it.nsteps > 1) load_k(1);
                        if (BIAS == 1 && it.nsteps > 1) load_bias(1);
                        for (int j = 0; j < it.nsteps && ok; ++j) {
                            load_v(j);
                            if (j + 2 < it.nsteps) load_k(j + 2);
                            if (BIAS && (BIAS == 2 || j > 0) && j + 1 < it.nsteps) load_bias(j + 1);
                        }
                        if (MULTI) { J0 += it.nsteps; ++q; }
                    }
                    if (ITEMS == TAKEN_OVER) {           // all copies of this item are on their way: ask for the next one
                        if (r >= 2) ok = ok && bounded_wait_s(bars_s + 8 * (LY::ITEM_EMPTY + (r & 1)), ((r >> 1) - 1) & 1, abort_s, status, 0xa52);
                        if (!ok) break;
                        mbar_arrive_expect_tx(&bars[LY::ITEM_FULL + (r & 1)], 16);
                        clc_ask(smem_u32(next_item) + 16 * (r & 1), bars_s + 8 * (LY::ITEM_FULL + (r & 1)));
                        asked = r + 1;
                    }
                }
                if (asked > 0) drain_wait(&bars[LY::ITEM_FULL + ((asked - 1) & 1)], ((asked - 1) >> 1) & 1);
                if (*abort_flag) ok = false;             // (a wait for the next item may have given up)
                if (!ok) {
                    for (int t = 0; t < 2; ++t)
                        if (q_issued[t] > 0) drain_wait(&bars[LY::Q_FULL + t], (q_issued[t] - 1) & 1);
                    for (int j = k_issued > KS ? k_issued - KS : 0; j < k_issued; ++j) drain_wait(&bars[LY::K_FULL + j % KS], (j / KS) & 1);
                    for (int j = v_issued > VS ? v_issued - VS : 0; j < v_issued; ++j) drain_wait(&bars[LY::V_FULL + j % VS], (j / VS) & 1);
                    if (BIAS)
                        for (int u = b_issued > 4 ? b_issued - 4 : 0; u < b_issued; ++u)
                            if (BIAS == 1) drain_wait(&bars[LY::B_FULL + (u & 3)], (u >> 2) & 1);
                            else if (u + 2 >= b_issued) drain_wait(&bars[LY::B_FULL + (u & 1)], (u >> 1) & 1);
                }
            }
        } else if (role <= 10) {
            // ------------------------------------------------------------ MMA issuer of tile t (whole warp walks, one lane issues)
            const int t = role - 9;
            {
                constexpr uint32_t IDESC_S = make_idesc_bf16(BM, BN, 0, 0), IDESC_PV = make_idesc_bf16(BM, D, 0, 1);
                const uint64_t q_desc = make_smem_desc_sw128(smem_u32(Qs) + t * Q_BYTES, 16, 1024);
                const uint64_t k_desc = make_smem_desc_sw128(smem_u32(Ks), 16, 1024);
                const uint64_t v_desc = make_smem_desc_sw128(smem_u32(Vs), BN * 128, 1024);
                bool ok = true;
                auto wait = [&](int bar, uint32_t parity, int code) {
                    if (ok) ok = warp_wait(bars_s + 8 * bar, parity, abort_s, status, code);
                };
                auto issue_s = [&](int j, bool last) {   // S_t(j) = Q_t K_j^T, then release the K stage
                    const uint64_t kd = k_desc + static_cast<uint64_t>(((j % KS) * KV_BYTES) >> 4);
#pragma unroll
                    for (int k = 0; k < D / 16; ++k)
                        mma_ss(tmem + S_COL(t, j & 1), q_desc + static_cast<uint64_t>(((k / 4) * (BM * 128) + (k % 4) * 32) >> 4),
                               kd + static_cast<uint64_t>(((k / 4) * (BN * 128) + (k % 4) * 32) >> 4), IDESC_S, k > 0);
                    tc_commit(&bars[LY::S_FULL + 2 * t + (j & 1)]);
                    tc_commit(&bars[LY::K_EMPTY + j % KS]);
                    if (MULTI && last) tc_commit(&bars[LY::Q_EMPTY + t]);
                };
                auto issue_pv = [&](int j, bool first) { // O_t += P_t(j) V_j, then release the V stage
                    const uint64_t vd = v_desc + static_cast<uint64_t>(((j % VS) * KV_BYTES) >> 4);
#pragma unroll
                    for (int k = 0; k < BN / 16; ++k)
                        mma_ts(tmem + O_COL(t), tmem + S_COL(t, j & 1) + k * 8, vd + static_cast<uint64_t>((k * 2048) >> 4), IDESC_PV, (!first || k > 0));
                    tc_commit(&bars[LY::PV_DONE + 2 * t + (j & 1)]);
                    tc_commit(&bars[LY::V_EMPTY + j % VS]);
                };
                Item it;
                int J = 0, q = 0;                        // the item's first key step of all; items with keys so far
                for (int r = 0; ok && get_item(r, it); ++r) {
                    const int n = it.nsteps;
                    if (n == 0) continue;
                    wait(LY::Q_FULL + t, q & 1, 0xa20);
                    for (int j = 0; j < 2 && j < n; ++j) {
                        wait(LY::K_FULL + (J + j) % KS, ((J + j) / KS) & 1, 0xa21);
                        tc_fence_after();
                        if (ok && elect_one()) issue_s(J + j, j == n - 1);
                        __syncwarp();
                    }
                    for (int j = 0; j < n && ok; ++j) {
                        const int g = J + j;
                        const bool more = j + 2 < n;
                        wait(LY::V_FULL + g % VS, (g / VS) & 1, 0xa22);
                        if (more) wait(LY::K_FULL + (g + 2) % KS, ((g + 2) / KS) & 1, 0xa23);
                        if (MULTI && j == 0) wait(LY::O_FREE + t, (q & 1) ^ 1, 0xa25);
                        wait(LY::P_FULL + 2 * t + (g & 1), (g >> 1) & 1, 0xa24);
                        if (!ok) break;
                        tc_fence_after();
                        // (S(j + 2) overwrites P(j): it goes behind the MMAs that read it)
                        if (elect_one()) { issue_pv(g, j == 0); if (more) issue_s(g + 2, j + 3 == n); }
                        __syncwarp();
                    }
                    if (MULTI) { J += n; ++q; }
                }
            }
        }
    } else {
        // ------------------------------------------------------------ softmax + epilogue (warps 0-7)
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        const int t = warp >> 2;
        const uint32_t tl = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const uint32_t my_bars = bars_s + 8 * (LY::S_FULL + 2 * t);       // S_FULL of the tile; P_FULL and PV_DONE 32 and 64 bytes on
        // (bias) the thread's row of its tile; the logits are scaled as they meet the bias
        uint32_t brow = smem_u32(Bs) + t * BIAS_BYTES + ((warp & 3) * 32 + lane) * 128;
        int rx = lane & 7;
        const float unit = BIAS ? 1.f : scale_log2e;
        const bool neg_scale = !BIAS && scale_log2e < 0.f;
        bool ok = true;
        Item it;
        int J = 0;                                       // the item's first key step of all
        for (int r = 0; ok && get_item(r, it); ++r) {
        const int n = it.n, nsteps = it.nsteps, row = it.row0 + t * BM + (warp & 3) * 32 + lane;
        const int brR = BIAS == 2 ? bias_row(it) + t * BM + (warp & 3) * 32 + lane : 0;
        const bool own_copy = BIAS == 2 && brR >= sb.full && row < Nq;      // (a row beyond the last whole group of eight)
        if (BIAS == 2) {
            brow = smem_u32(Bs) + t * BIAS_BYTES + shifted_row<SHIFTED_WIDTH(D)>(brR, bias_row(it) + t * BM);
            rx = shifted_by(brR, Nk);
        }
        float m_ref = -INFINITY, l = 0.f;
        const long long rlim = static_cast<long long>(row) + 1 + it.coff;
        const int nrow = rlim < n ? (rlim < 0 ? 0 : static_cast<int>(rlim)) : n;
        const int nrow_min = __shfl_sync(0xffffffffu, nrow, 0);
        for (int j = 0; j < nsteps; ++j) {
            const int g = J + j;
            const uint32_t s_addr = tl + S_COL(t, g & 1);
            ok = warp_wait(my_bars + 8 * (g & 1), (g >> 1) & 1, abort_s, status, 0xa30 + t);
            if (!ok) break;
            tc_fence_after();
            uint32_t s[BN];
            tmem_ld_x32(s_addr, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
            tmem_ld_x32(s_addr + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
            if (BIAS) ok = warp_wait(bars_s + 8 * (LY::B_FULL + (BIAS == 2 ? t : 2 * (g & 1) + t)), (BIAS == 2 ? g : g >> 1) & 1, abort_s, status, 0xa36 + t);
            tc_wait_ld();
            if (BIAS) {
                if (!ok) break;
                if (BIAS == 2 && own_copy) copy_bias_row(sb.p + static_cast<int64_t>(brR) * Nk + j * BN, brow + rx, Nk - j * BN < BN ? Nk - j * BN : BN);
                add_bias<BIAS>(s, scale_log2e, brow + (BIAS == 2 ? 0 : (g & 1) * (2 * BIAS_BYTES)), rx);
                __syncwarp();
                if (lane == 0) mbar_arrive_s(bars_s + 8 * (LY::B_EMPTY + (BIAS == 2 ? t : 2 * (g & 1) + t)));
            }
            const int col0 = j * BN;
            const bool tail = col0 + BN > nrow_min;      // (warp-uniform) some row has masked keys in this step
            const int nvalid = nrow > col0 ? (nrow - col0 < BN ? nrow - col0 : BN) : 0;
            if (tail) {
                const uint32_t excl = __float_as_uint(neg_scale ? INFINITY : -INFINITY);
#pragma unroll
                for (int i = 0; i < BN; ++i) if (i >= nvalid) s[i] = excl;
            }
            bool careful = j == 0 || tail;
            float lt = 0.f;
            if (!careful) {
                lt = exp_store<false>(s, unit, -m_ref, s_addr, BN);
                careful = __any_sync(0xffffffffu, !(lt <= OVERFLOW_SUM));
                if (!BIAS && careful) {  // (the weights went over the first half of the logits only: 32 registers less to keep)
                    tmem_ld_x32(s_addr + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
                    tc_wait_ld();
                }
            }
            if (careful) {
                const float mx = nvalid > 0 ? row_extreme(s, neg_scale) * unit : -INFINITY;
                if (__any_sync(0xffffffffu, mx > m_ref + RESCALE_THRESHOLD)) {
                    const float m_new = fmaxf(m_ref, mx);
                    const float alpha = m_new == -INFINITY ? 1.f : ex2_approx(m_ref - m_new);   // 0 on the row's first keys
                    l *= alpha;
                    if (j > 0) {
                        ok = warp_wait(my_bars + 64 + 8 * ((g - 1) & 1), ((g - 1) >> 1) & 1, abort_s, status, 0xa32 + t);
                        if (!ok) break;
                        tc_fence_after();
#pragma unroll 1                          // (rare; unrolled, its registers made the common path spill: 428 -> 482 us)
                        for (int c = 0; c < D / 16; ++c) {
                            uint32_t r[16];
                            tmem_ld_x16(tl + O_COL(t) + c * 16, r);
                            tc_wait_ld();
#pragma unroll
                            for (int i = 0; i < 16; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * alpha);
                            tmem_st_x16(tl + O_COL(t) + c * 16, r);
                        }
                    }
                    m_ref = m_new;
                }
                lt = exp_store<true>(s, unit, m_ref == -INFINITY ? 0.f : -m_ref, s_addr, nvalid);
            }
            l += lt;
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_s(my_bars + 32 + 8 * (g & 1));
        }
        if (ok && nsteps > 0)
            ok = warp_wait(my_bars + 64 + 8 * ((J + nsteps - 1) & 1), ((J + nsteps - 1) >> 1) & 1, abort_s, status, 0xa34 + t);
        if (MULTI) J += nsteps;
        if (ok) {
            const float inv = l > 0.f ? 1.f / l : 0.f;
            if (!VL && lse && row < Nq)
                lse[static_cast<int64_t>(it.bh) * Nq + row] = l > 0.f ? (m_ref + log2f(l)) * 0.6931471805599453f : -INFINITY;
            tc_fence_after();
            __nv_bfloat16* orow = VL ? O + ((static_cast<int64_t>(it.q_tok0) + (row - it.row0)) * H + it.head) * D
                                     : O + (static_cast<int64_t>(it.bh) * Nq + row) * D;
#pragma unroll
            for (int c = 0; c < D / 32; ++c) {
                uint32_t r[32];
                if (nsteps > 0) {
                    tmem_ld_x32(tl + O_COL(t) + c * 32, r);
                    tc_wait_ld();
                    if (MULTI && c == D / 32 - 1) {      // the next item may write its output
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_s(bars_s + 8 * (LY::O_FREE + t));
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) r[i] = 0u;      // no valid key: O = 0
                }
                if (VL ? row - it.row0 < it.q_rows : row < Nq) {
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        uint4 w;
                        w.x = pack_bf16x2(__uint_as_float(r[8 * v + 0]) * inv, __uint_as_float(r[8 * v + 1]) * inv);
                        w.y = pack_bf16x2(__uint_as_float(r[8 * v + 2]) * inv, __uint_as_float(r[8 * v + 3]) * inv);
                        w.z = pack_bf16x2(__uint_as_float(r[8 * v + 4]) * inv, __uint_as_float(r[8 * v + 5]) * inv);
                        w.w = pack_bf16x2(__uint_as_float(r[8 * v + 6]) * inv, __uint_as_float(r[8 * v + 7]) * inv);
                        *reinterpret_cast<uint4*>(orow + c * 32 + v * 8) = w;
                    }
                }
            }
        }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

template <int BIAS, int ITEMS>
int launch(const Problem& p, const CUtensorMap& tmB, int shifted_rows, cudaStream_t st) {
    constexpr int SMEM_BYTES = Layout<BIAS>::SMEM_BYTES;
    CUtensorMap tmQ, tmK, tmV;
    const int BH = p.B * p.H, slabs = (p.Nq + 2 * BM - 1) / (2 * BM);
    if (static_cast<int64_t>(slabs) * BH > 0x7fffffff) return FLAT_ERR_SHAPE;
    if (!make_map(&tmQ, p.Q, BH, p.Nq, D, BM) || !make_map(&tmK, p.K, BH, p.Nk, D, BN) || !make_map(&tmV, p.V, BH, p.Nk, D, BN))
        return FLAT_ERR_CUDA;
    if (!ensure_dynamic_smem<fused_d128_kernel<false, BIAS, ITEMS>>(SMEM_BYTES)) return FLAT_ERR_CUDA;
    // without the causal mask the slabs of a head run side by side and share K and V in L2; with it, those of as many heads as
    // fit L2 together (48 MB of K and V) go longest first: what is left at the end are the short ones
    const int64_t fit = (48ll << 20) / (static_cast<int64_t>(p.Nk) * D * 4);
    const int group = !p.causal || fit < 1 ? 1 : fit < BH ? static_cast<int>(fit) : BH;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ITEMS == DEALT ? device_sm_count() : slabs * BH);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, fused_d128_kernel<false, BIAS, ITEMS>, tmQ, tmK, tmV, static_cast<__nv_bfloat16*>(p.O), BH, p.H, p.Nq, p.Nk,
                                             p.scale * 1.4426950408889634f, p.k_valid_len, p.causal ? p.Nk - p.Nq : (1 << 30), group, p.status,
                                             static_cast<const int32_t*>(nullptr), static_cast<const int32_t*>(nullptr), p.lse, tmB, p.bias_sh ? 1 : 0, p.bias_sb ? 1 : 0,
                                             ShiftedBias{static_cast<const uint16_t*>(p.bias), shifted_rows});
    return e == cudaSuccess ? FLAT_OK : FLAT_ERR_CUDA;
}

}  // namespace

int launch_fused_d128(const Problem& p, const BiasMap& bias, cudaStream_t st) {
    if (p.dtype != FLAT_DTYPE_BF16 || p.d != D || !p.bias != !bias.map || p.block_mask) return FLAT_ERR_UNSUPPORTED;
    // More items than SMs: several items per CTA, so that one's first loads and logits overlap the last one's output.
    // Items of up to 1024 keys, and no more than three a query, that all weigh the same (no key counts, no causal mask) are dealt in
    // advance.  Otherwise a CTA that has issued an item's copies takes over another one (clusterlaunchcontrol): long and unequal items
    // end together, but every role of the CTA has to read the answer before it can go on.  us, taken over / dealt: B32 H8 300^2
    // 37.0 / 32.7, B81 H8 64^2 16.4 / 15.2, B32 H4 2000 x 500 86.0 / 80.1, B30 H8 600^2 with bias 88.0 / 83.5; B44 H4 100 x 500
    // 21.3 / 22.5, 200 x 800 32.4 / 34.8, causal B16 H16 512^2 43.9 / 49.6, key counts B12 H12 1000^2 59.9 / 61.0, B4 H16 2048^2
    // 123.0 / 124.3, H4 16K^2 412 / 424.
    // With no more items than SMs there is nothing to take over: the form for one item is the faster one at any length (us, taken over
    // / one item: B4 H8 1000^2 20.4 / 19.4, H2 16K^2 213 / 208, H1 32K^2 420 / 412, H8 4000 x 16K 217 / 211).
    // Nor does it pay where bias rows have to be shifted and an item has more than 256 keys: its steps take twice as long, and the form for one
    // item has the shorter ones (taken over / one item: B22 H6 323^2 34.6 / 34.4, B40 H6 450^2 79.2 / 78.4, B4 H16 1001^2 69.9 / 65.9, 2001^2 260 / 248,
    // causal 159 / 157; below, B50 H6 101^2 20.9 / 21.9, B80 H6 201^2 48.3 / 48.6, dealt 56.6).
    const int sms = device_sm_count(), slabs = (p.Nq + 2 * BM - 1) / (2 * BM);
    const bool shifted = bias.shifted_rows >= 0;
    const bool alike = !p.k_valid_len && !p.causal && p.Nk <= 1024 && p.Nk <= 3 * static_cast<int64_t>(p.Nq) && !shifted;
    const int items = static_cast<int64_t>(slabs) * p.B * p.H <= sms || (shifted && p.Nk > 256) ? ONE_ITEM : alike ? DEALT : TAKEN_OVER;
    const int sr = bias.shifted_rows;
    auto run = [&](auto form) {
        constexpr int BIAS = decltype(form)::value;
        const CUtensorMap tmB = bias.map ? *static_cast<const CUtensorMap*>(bias.map) : CUtensorMap{};
        if constexpr (BIAS != 2)
            if (items == DEALT) return launch<BIAS, DEALT>(p, tmB, sr, st);
        return items == ONE_ITEM ? launch<BIAS, ONE_ITEM>(p, tmB, sr, st) : launch<BIAS, TAKEN_OVER>(p, tmB, sr, st);
    };
    if (!bias.map) return run(std::integral_constant<int, 0>{});
    return sr >= 0 ? run(std::integral_constant<int, 2>{}) : run(std::integral_constant<int, 1>{});
}

int launch_fused_d128_varlen(const void* Q, const void* K, const void* V, void* O, const int32_t* cu_q, const int32_t* cu_k, int num_seqs,
                             int H, int64_t total_q, int64_t total_k, int max_seqlen_q, float scale, int causal, int32_t* status,
                             cudaStream_t st) {
    if (static_cast<int64_t>(num_seqs) * H > 65535) return FLAT_ERR_SHAPE;      // (grid y)
    CUtensorMap tmQ, tmK, tmV;
    if (!make_map_packed(&tmQ, Q, total_q, H, D, BM) || !make_map_packed(&tmK, K, total_k, H, D, BN) ||
        !make_map_packed(&tmV, V, total_k, H, D, BN))
        return FLAT_ERR_CUDA;
    const int slabs = (max_seqlen_q + 2 * BM - 1) / (2 * BM), group = causal && slabs <= 65535, sms = device_sm_count();
    const int64_t items = static_cast<int64_t>(slabs) * num_seqs * H;
    // Items that all weigh the same -- sequences of one length, without the causal mask or of one slab -- several per CTA, up to
    // 1024 tokens and from three per SM on (us, a CTA each / dealt: 100 of 256 tokens, 16 heads 146 / 129, causal
    // 142 / 116; 64 of 128, 8 heads 26.3 / 20.7; 64 of 64, 16 heads 36 / 22; 32 of 1000, 16 heads 281 / 275; with 1.7 and 2.6 per
    // SM, 16 of 512, 8 heads 26.5 / 27.5, 16 of 300, 12 heads 33.1 / 35.4).
    const bool alike = total_q == static_cast<int64_t>(num_seqs) * max_seqlen_q && total_k == total_q && (!causal || slabs == 1);
    const bool several = alike && items >= 3 * static_cast<int64_t>(sms) && items <= 0x7fffffff && max_seqlen_q <= 1024;
    if (!(several ? ensure_dynamic_smem<fused_d128_kernel<true, 0, DEALT>>(Layout<0>::SMEM_BYTES)
                  : ensure_dynamic_smem<fused_d128_kernel<true, 0, ONE_ITEM>>(Layout<0>::SMEM_BYTES)))
        return FLAT_ERR_CUDA;
    const dim3 grid(several ? sms : group ? num_seqs * H : slabs, several ? 1 : group ? slabs : num_seqs * H);
    (several ? fused_d128_kernel<true, 0, DEALT> : fused_d128_kernel<true, 0, ONE_ITEM>)<<<grid, THREADS, Layout<0>::SMEM_BYTES, st>>>(
        tmQ, tmK, tmV, static_cast<__nv_bfloat16*>(O), num_seqs * H, H, max_seqlen_q, 0, scale * 1.4426950408889634f, nullptr,
        causal ? 0 : (1 << 30), group, status, cu_q, cu_k, nullptr, CUtensorMap{}, 0, 0, ShiftedBias{});
    return cudaGetLastError() == cudaSuccess ? FLAT_OK : FLAT_ERR_CUDA;
}

}  // namespace flat
