// Fused Logit-Softmax-Attend for fp32 tensors on the tensor cores (fp32 in, fp32 out, d = 32, 64, 128).
//
// The tensor cores take 32-bit operands only as tf32 (10 mantissa bits), so every fp32 operand x is
// split into x_hi (a tf32 number close to x) and x_lo = x - x_hi (exact in fp32), and each contraction is the sum of
// three tf32 products
//     a b  ~=  a_lo b_hi + a_hi b_lo + a_hi b_hi          (the dropped a_lo b_lo is 2^-22 of the result)
// accumulated in fp32.  Both contractions of the path are done this way: S = Q K^T and, per key step,
// P V with the weights P split the same way.  The accumulation ACROSS key steps is not left to the
// tensor core: each step's P V lands in a fresh TMEM buffer and the row's owner thread adds it to the
// running output in registers, O = alpha O + P V, in round-to-nearest fp32 -- the rescaling of the
// streaming softmax then costs nothing extra, and the result does not depend on how the tensor core
// rounds a 16K-term running sum.
//
// What bounds it: the tensor pipe at d = 64 (three products at half the bf16 rate: active 77 % of the time by its counter, and
// 52 % of the shared-memory port), the chain of a 32-key step at d = 128 (59 %; its softmax warps spill 312 bytes), the softmax
// warps at d = 32.  B2 H16 4096^2, d = 32 / 64 / 128: 393 / 539 / 1,247 us in the first 20 ms of launches, 412 / 610 / 1,402 in a
// second of them (the power cap: 1,837, 1,575 and 1,717 MHz).  Before, d = 32 and 128 ran on the FFMA kernel: 2,840 and 9,600 us.
//
// Paper mapping (Section 5, 5.1, 5.2): shared outer loops = (batch, head) and a tile of 128 query rows on blockIdx.x
// (R-granularity); Logit and Attend run interleaved over steps of 64 keys (d = 128: 32) with
// the streaming softmax between them; the logits and weights never leave TMEM.
//
// CTA = 512 threads, four warpgroups:
//   warps 0-3  softmax of the even key steps (thread r <-> row r <-> TMEM lane r): Q -> TMEM once (scaled,
//              split), then per step the row maximum, p = 2^(x - m), the split of p into TMEM, and
//              O = alpha O + (P V of its step before)
//   warps 4-7  softmax of the odd key steps, the same way with a running maximum, sum and output of its own:
//              the two streams never talk until the end, where they are merged like two partial softmaxes
//   warps 8-11 converters: warps 8, 9 K tile -> (K_hi in place, K_lo); warps 10, 11 V tile -> transposed
//              (V^T_hi, V^T_lo), since a tf32 operand must have the contraction index contiguous in shared memory
//   warp  12   TMA producer (one lane): Q once, K and raw V tiles into rings
//   warps 13, 14  MMA issuers of the even / odd key steps (one elected lane each): tcgen05.mma with k-slices of 8, A
//              always from TMEM
//   warp  15   idle (it completes the warpgroup for the register hand-over)
// TMEM columns: Q_hi d, Q_lo d, then per step parity S / P_hi (as many columns as a step has keys), P_lo and P V (d); at
// d = 128, where Q takes half of TMEM, steps of 32 keys leave room for both parities of S and P and for one P V buffer:
// a step's P V waits until the one before has been read, which happens while the pipe works on the logits in between.
// An infinite operand has no finite remainder: its products are NaN.  At d = 32 and 128 a row that does not come out finite is
// computed again in plain fp32 (plain_rows), which gives what the FFMA kernel gives; at d = 64 it stays NaN.
// Every wait is bounded (see tc_common.cuh); on expiry the CTA aborts cleanly and reports a code.
#include <cuda.h>
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
constexpr int KS = 3;                // K ring (each stage: K_hi and K_lo tiles)
constexpr int VR = 2;                // raw V ring
constexpr int VS = 3;                // transposed V ring (each stage: V^T_hi and V^T_lo tiles)
constexpr int THREADS = 512;
constexpr uint32_t HI_MASK = 0xffffe000u;
constexpr uint32_t TMEM_COLS = 512;

template <int D> struct Layout {
    static constexpr int BN = D == 128 ? 32 : 64;        // keys per step
    static constexpr int TILE = BN * D * 4;              // K: D/32 panels of BN rows x 128 bytes; V^T: BN/32 panels of D rows
    static constexpr int PANEL = BN * 128, VT_PANEL = D * 128;
    static constexpr int MERGE_STRIDE = D + 4;           // floats per row of the merge scratch (outputs, m, l, padding: 16-byte rows, no bank conflicts)
    static constexpr int PVS = D == 128 ? 1 : 2;         // P V buffers
    // registers after the hand-over, of the 512 x 128 of the launch (d = 64 with 192 / 80 / 48: the converters spill, 548 us
    // against 532 on B2 H16 4096^2 in short runs)
    static constexpr int SOFT_REGS = D == 128 ? 192 : 176, CONVERT_REGS = D == 128 ? 80 : 104, ISSUE_REGS = D == 128 ? 48 : 56;
    static_assert(256 * SOFT_REGS + 128 * CONVERT_REGS + 128 * ISSUE_REGS <= THREADS * 128, "register hand-over");
    static constexpr uint32_t QH_COL = 0, QL_COL = D, S_COL = 2 * D, PL_COL = S_COL + 2 * BN, PV_COL = PL_COL + 2 * BN;
    static_assert(PV_COL + PVS * D <= TMEM_COLS, "tensor memory");
    // shared memory: K_hi[KS] K_lo[KS] Vraw[VR] VT_hi[VS] VT_lo[VS]; the Q tile is staged over the V^T rings
    static constexpr int OFF_KH = 0, OFF_KL = OFF_KH + KS * TILE, OFF_VR = OFF_KL + KS * TILE, OFF_VTH = OFF_VR + VR * TILE,
                         OFF_VTL = OFF_VTH + VS * TILE, TILE_BYTES = OFF_VTL + VS * TILE;
    static_assert(2 * VS * TILE >= BM * D * 4, "the Q tile is staged over the V^T rings");
    static_assert(2 * KS * TILE >= BM * MERGE_STRIDE * 4, "the merge scratch lies over the K rings");
    static constexpr int SMEM_BYTES = TILE_BYTES + 512 + 1024;
    static_assert(SMEM_BYTES <= 232448, "shared memory");
};

// barriers
constexpr int Q_FULL = 0, Q_READY = 1, K_FULL = 2, KC_FULL = K_FULL + KS, K_EMPTY = KC_FULL + KS, V_FULL = K_EMPTY + KS,
              VR_EMPTY = V_FULL + VR, VT_FULL = VR_EMPTY + VR, VT_EMPTY = VT_FULL + VS, S_FULL = VT_EMPTY + VS,
              P_FULL = S_FULL + 2, PV_FULL = P_FULL + 2, PV_FREE = PV_FULL + 2, NUM_BARS = PV_FREE + 2;

// D[tmem] (+)= A[tmem] * B[smem desc], tf32 operands
__device__ __forceinline__ void mma_tf32_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Instruction descriptor for kind::tf32, fp32 accumulator, both operands with the contraction index contiguous, n columns.
__host__ __device__ constexpr uint32_t idesc_tf32(int n) {
    return (1u << 4) | (2u << 7) | (2u << 10) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(BM >> 4) << 24);
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts128(uint32_t addr, uint4 v) {
    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// x_hi and x_lo = x - x_hi (exact).  NEAR: x_hi = x (1 + 0.35 * 2^-10), a third to two thirds of its unit above x, with the low
// bits cut off: nearly the nearest tf32 number (rounding the product towards zero keeps the largest numbers finite).  The mean
// square of x_lo is then a third of what cutting x off itself leaves and its mean about zero: with 32 and 128 features the
// error is that of the FFMA kernel, which ran there before (300 keys, d = 128: rms 4.8e-8 against 4.7e-8, cut off 9.3e-8; 4096
// keys, d = 32: 9.5e-9 against 3.1e-8).  It costs 2 % of the time there (B2 H16 4096^2: 1,199 us against 1,178, 432 against
// 424); 12 % at d = 64 (620 against 552), where x is cut off.
template <bool NEAR>
__device__ __forceinline__ uint32_t hi_of(uint32_t x) {
    return (NEAR ? __float_as_uint(__fmul_rz(__uint_as_float(x), 1.00034180f)) : x) & HI_MASK;
}
__device__ __forceinline__ uint32_t lo_of(uint32_t x, uint32_t hi) { return __float_as_uint(__uint_as_float(x) - __uint_as_float(hi)); }
template <bool NEAR>
__device__ __forceinline__ void split4(const uint4& v, uint4& h, uint4& l) {
    h = make_uint4(hi_of<NEAR>(v.x), hi_of<NEAR>(v.y), hi_of<NEAR>(v.z), hi_of<NEAR>(v.w));
    l = make_uint4(lo_of(v.x, h.x), lo_of(v.y, h.y), lo_of(v.z, h.z), lo_of(v.w, h.w));
}

template <int D>
__global__ void __launch_bounds__(THREADS, 1)
fused_tf32_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                  const __grid_constant__ CUtensorMap tmV, const float* Q, const float* K, const float* V, float* O, int BH, int H, int Nq,
                  int Nk, float scale_log2e, const int32_t* __restrict__ valid_len, int coff, int group, int32_t* status,
                  float* __restrict__ lse) {
    using LY = Layout<D>;
    constexpr int BN = LY::BN, TILE = LY::TILE, PANEL = LY::PANEL, OFF_KH = LY::OFF_KH, OFF_KL = LY::OFF_KL, OFF_VR = LY::OFF_VR,
                  OFF_VTH = LY::OFF_VTH, OFF_VTL = LY::OFF_VTL, TILE_BYTES = LY::TILE_BYTES;
    constexpr bool NEAR = D != 64;
    constexpr uint32_t QH_COL = LY::QH_COL, QL_COL = LY::QL_COL, S_COL = LY::S_COL, PL_COL = LY::PL_COL, PV_COL = LY::PV_COL;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(base + TILE_BYTES);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + NUM_BARS);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const uint32_t sb = smem_u32(base);

    const int warp = D == 128 ? threadIdx.x >> 5 : warp_index(), lane = threadIdx.x & 31;   // (see there; d = 32: 2 % ahead up to
    // 512 rows, from 5 % ahead to 8 % behind beyond, by the number of tiles per SM)
    auto whole_warp_wait = [&](uint64_t* bar, uint32_t parity, int code) {
        return D == 128 ? __all_sync(0xffffffffu, bounded_wait(bar, parity, abort_flag, status, code))
                        : warp_wait(bar, parity, abort_flag, status, code);
    };
    // `group` heads at a time, their tiles side by side, the longest first under the causal mask
    const int slabs = (Nq + BM - 1) / BM, per = group * slabs, first = static_cast<int>(blockIdx.x) / per * group;
    const int heads = BH - first < group ? BH - first : group, at = static_cast<int>(blockIdx.x) % per;
    const int bh = first + at % heads;
    const int row0 = (coff < (1 << 29) ? slabs - 1 - at / heads : at / heads) * BM;
    if (threadIdx.x == 384) {
        for (int i = 0; i < NUM_BARS; ++i) {
            if (i == Q_READY) { mbar_init(&bars[i], 8); continue; }
            const bool by_warps = (i >= KC_FULL && i < K_EMPTY) || (i >= VR_EMPTY && i < VT_EMPTY) ||
                                  (i >= P_FULL && i < PV_FULL) || i >= PV_FREE;
            const bool by_two = (i >= KC_FULL && i < K_EMPTY) || (i >= VR_EMPTY && i < VT_EMPTY);   // (converter warp pairs)
            mbar_init(&bars[i], by_two ? 2 : by_warps ? 4 : 1);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0) { tmem_alloc(tmem_slot, TMEM_COLS); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // (launched with programmatic stream serialization: this set-up overlaps the tail of the previous kernel of the stream, and
    // nothing in device memory is touched before that one has finished)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    int n = Nk;
    if (valid_len) { n = valid_len[bh / H]; n = n < 0 ? 0 : (n > Nk ? Nk : n); }
    {
        // Causal mask (coff = Nk - Nq; 2^30 = none): row r sees keys j < r + 1 + coff, so the CTA's
        // last row bounds the keys of all its rows.
        const long long lim = static_cast<long long>(row0) + BM + coff;
        if (lim < n) n = lim < 0 ? 0 : static_cast<int>(lim);
    }
    const int ntiles = (n + BN - 1) / BN;

    if (warp >= 12) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(LY::ISSUE_REGS));
        if (warp == 12) {
            // ------------------------------------------------------------ TMA producer
            if (lane == 0 && ntiles > 0) {
                prefetch_tensormap(&tmQ); prefetch_tensormap(&tmK); prefetch_tensormap(&tmV);
                bool ok = true;
                int k_issued = 0, v_issued = 0;
                auto load_k = [&](int j) {
                    const int s = j % KS;
                    ok = bounded_wait(&bars[K_EMPTY + s], ((j / KS) & 1) ^ 1, abort_flag, status, 0x600 + s);
                    if (!ok) return;
                    mbar_arrive_expect_tx(&bars[K_FULL + s], TILE);
#pragma unroll
                    for (int c = 0; c < D / 32; ++c)
                        tma_load_3d(base + OFF_KH + s * TILE + c * PANEL, &tmK, &bars[K_FULL + s], 32 * c, j * BN, bh);
                    k_issued = j + 1;
                };
                auto load_v = [&](int j) {
                    const int s = j % VR;
                    ok = bounded_wait(&bars[VR_EMPTY + s], ((j / VR) & 1) ^ 1, abort_flag, status, 0x610 + s);
                    if (!ok) return;
                    mbar_arrive_expect_tx(&bars[V_FULL + s], TILE);
#pragma unroll
                    for (int c = 0; c < D / 32; ++c)
                        tma_load_3d(base + OFF_VR + s * TILE + c * PANEL, &tmV, &bars[V_FULL + s], 32 * c, j * BN, bh);
                    v_issued = j + 1;
                };
                mbar_arrive_expect_tx(&bars[Q_FULL], BM * D * 4);
#pragma unroll
                for (int c = 0; c < D / 32; ++c) tma_load_3d(base + OFF_VTH + c * BM * 128, &tmQ, &bars[Q_FULL], 32 * c, row0, bh);
                load_k(0);
                if (ntiles > 1) load_k(1);
                for (int j = 0; j < ntiles && ok; ++j) {
                    load_v(j);                               // (never behind a K stage that waits for an older S)
                    if (ok && j + 2 < ntiles) load_k(j + 2);
                }
                if (!ok) {
                    drain_wait(&bars[Q_FULL], 0);
                    for (int j = k_issued > KS ? k_issued - KS : 0; j < k_issued; ++j) drain_wait(&bars[K_FULL + j % KS], (j / KS) & 1);
                    for (int j = v_issued > VR ? v_issued - VR : 0; j < v_issued; ++j) drain_wait(&bars[V_FULL + j % VR], (j / VR) & 1);
                }
            }
        } else if (warp <= 14) {
            // ------------------------------------------------------------ MMA issuers: warp 13 the even key steps, warp 14 the odd
            // ones (the whole warp runs the loop, one lane issues).  Within a parity the order P V(j), S(j+2) is program
            // order; the two parities share nothing but the tensor pipe, and one issues while the other waits.
            const int g = warp - 13;
            if (ntiles > g) {
                const uint64_t kh_desc = make_smem_desc_sw128(sb + OFF_KH, 16, 1024);
                const uint64_t kl_desc = make_smem_desc_sw128(sb + OFF_KL, 16, 1024);
                const uint64_t vh_desc = make_smem_desc_sw128(sb + OFF_VTH, 16, 1024);
                const uint64_t vl_desc = make_smem_desc_sw128(sb + OFF_VTL, 16, 1024);
                bool ok = true;
                auto wait = [&](int bar, uint32_t parity, int code) {
                    if (ok) ok = whole_warp_wait(&bars[bar], parity, code);
                    if (ok) tc_fence_after();
                };
                constexpr uint32_t IDESC_S = idesc_tf32(BN), IDESC_PV = idesc_tf32(D);
                // one product, k-slices of eight (32 bytes of a 128-byte row each): Q K^T (128 x BN x D), P V (128 x D x BN)
                auto product_s = [&](uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, bool first) {
#pragma unroll
                    for (int k = 0; k < D / 8; ++k)
                        mma_tf32_ts(d_tmem, a_tmem + k * 8, b_desc + static_cast<uint64_t>(((k >> 2) * PANEL + (k & 3) * 32) >> 4),
                                    IDESC_S, !(first && k == 0));
                };
                auto product_pv = [&](uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, bool first) {
#pragma unroll
                    for (int k = 0; k < BN / 8; ++k)
                        mma_tf32_ts(d_tmem, a_tmem + k * 8, b_desc + static_cast<uint64_t>(((k >> 2) * LY::VT_PANEL + (k & 3) * 32) >> 4),
                                    IDESC_PV, !(first && k == 0));
                };
                auto issue_s = [&](int j) {                  // S(j) = Q K_j^T, small terms first; then release the K stage
                    const int ks = j % KS, b = j & 1;
                    if (elect_one()) {
                        const uint64_t st = static_cast<uint64_t>((ks * TILE) >> 4);
                        product_s(tmem + S_COL + BN * b, tmem + QL_COL, kh_desc + st, true);
                        product_s(tmem + S_COL + BN * b, tmem + QH_COL, kl_desc + st, false);
                        product_s(tmem + S_COL + BN * b, tmem + QH_COL, kh_desc + st, false);
                        tc_commit(&bars[S_FULL + b]);
                        tc_commit(&bars[K_EMPTY + ks]);
                    }
                    __syncwarp();
                };
                auto issue_pv = [&](int j) {                 // PV(j) = P_j V_j into its own buffer; then release the V^T stage
                    const int vs = j % VS, b = j & 1;
                    if (elect_one()) {
                        const uint64_t st = static_cast<uint64_t>((vs * TILE) >> 4);
                        product_pv(tmem + PV_COL + (LY::PVS - 1) * D * b, tmem + PL_COL + BN * b, vh_desc + st, true);
                        product_pv(tmem + PV_COL + (LY::PVS - 1) * D * b, tmem + S_COL + BN * b, vl_desc + st, false);
                        product_pv(tmem + PV_COL + (LY::PVS - 1) * D * b, tmem + S_COL + BN * b, vh_desc + st, false);
                        tc_commit(&bars[PV_FULL + b]);
                        tc_commit(&bars[VT_EMPTY + vs]);
                    }
                    __syncwarp();
                };
                wait(Q_READY, 0, 0x620);
                wait(KC_FULL + g, 0, 0x621);
                if (ok) issue_s(g);
                for (int j = g; j < ntiles && ok; j += 2) {
                    wait(VT_FULL + j % VS, (j / VS) & 1, 0x630);
                    // (the buffer's last use: two steps before, or the step before, of the other issuer)
                    if (LY::PVS == 2) wait(PV_FREE + (j & 1), ((j >> 1) & 1) ^ 1, 0x631);
                    else if (j > 0) wait(PV_FREE + ((j - 1) & 1), ((j - 1) >> 1) & 1, 0x631);
                    // (the converted keys of step j + 2 are checked here, ahead of the wait for the weights, so that
                    // the check does not sit between the two batches of products)
                    if (j + 2 < ntiles) wait(KC_FULL + (j + 2) % KS, ((j + 2) / KS) & 1, 0x633);
                    wait(P_FULL + (j & 1), (j >> 1) & 1, 0x632);
                    if (ok) issue_pv(j);
                    // (S(j+2) overwrites P_hi(j): it goes behind the products that read it)
                    if (j + 2 < ntiles && ok) issue_s(j + 2);
                }
            }
        }
    } else if (warp >= 8) {
        // ------------------------------------------------------------ converters (warps 8-11)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(LY::CONVERT_REGS));
        bool ok = true;
        if (warp < 10) {
            // warps 8, 9: K tile -> K_hi (in place) and K_lo, element by element
            const int ct = threadIdx.x - 256;
            for (int j = 0; j < ntiles && ok; ++j) {
                const int s = j % KS;
                ok = whole_warp_wait(&bars[K_FULL + s], (j / KS) & 1, 0x641);
                if (!ok) break;
                const uint32_t kh = sb + OFF_KH + s * TILE, kl = sb + OFF_KL + s * TILE;
#pragma unroll
                for (int i = 0; i < TILE / 1024; ++i) {
                    const uint32_t off = (ct + 64 * i) * 16;
                    uint4 h, l;
                    split4<NEAR>(lds128(kh + off), h, l);
                    sts128(kl + off, l);
                    sts128(kh + off, h);
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars[KC_FULL + s]);
            }
        } else {
            // warps 10, 11: V tile -> transposed V^T_hi, V^T_lo.  4 x 4 blocks: a thread's blocks sit on an XOR
            // diagonal of (key block, feature block), which keeps both the 16-byte reads and the transposed
            // 16-byte writes free of bank conflicts under the 128-byte swizzle.
            const int u = lane & 7, tq = lane >> 3;
            if (ntiles > 0)
                ok = whole_warp_wait(&bars[Q_READY], 0, 0x640);   // (Q has left the V^T ring)
            for (int j = 0; j < ntiles && ok; ++j) {
                const int r = j % VR, s = j % VS;
                ok = whole_warp_wait(&bars[V_FULL + r], (j / VR) & 1, 0x642);
                if (ok) ok = whole_warp_wait(&bars[VT_EMPTY + s], ((j / VS) & 1) ^ 1, 0x643);
                if (!ok) break;
                // 32 x 32 squares (DB: of the features, KB: of the keys) in turn over the two warps
#pragma unroll
                for (int sq = 0; sq < (D / 32) * (BN / 32); sq += 2) {
                    const int DB = D == 32 ? 0 : D == 64 ? warp - 10 : sq + warp - 10, KB = D == 32 ? warp - 10 : D == 64 ? sq / 2 : 0;
                    const uint32_t vr = sb + OFF_VR + r * TILE + DB * PANEL;
                    const uint32_t vth = sb + OFF_VTH + s * TILE + KB * LY::VT_PANEL, vtl = sb + OFF_VTL + s * TILE + KB * LY::VT_PANEL;
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int dbc = u ^ (tq + 4 * i);         // feature block (chunk) within the panel; key block = u
                        uint32_t in[4][4];
#pragma unroll
                        for (int rr = 0; rr < 4; ++rr) {
                            const int krow = 32 * KB + 4 * u + rr;
                            const uint4 v = lds128(vr + krow * 128 + ((dbc ^ (krow & 7)) << 4));
                            in[rr][0] = v.x; in[rr][1] = v.y; in[rr][2] = v.z; in[rr][3] = v.w;
                        }
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const int drow = 32 * DB + 4 * dbc + c;
                            const uint32_t off = drow * 128 + ((u ^ (drow & 7)) << 4);
                            uint4 h, l;
                            split4<NEAR>(make_uint4(in[0][c], in[1][c], in[2][c], in[3][c]), h, l);
                            sts128(vth + off, h);
                            sts128(vtl + off, l);
                        }
                    }
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) { mbar_arrive(&bars[VT_FULL + s]); mbar_arrive(&bars[VR_EMPTY + r]); }
            }
        }
    } else {
        // ------------------------------------------------------------ softmax + output (warps 0-7)
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(LY::SOFT_REGS));
        const int g = warp >> 2;                             // 0: even key steps, 1: odd key steps (= TMEM buffer)
        const int r = (warp & 3) * 32 + lane;                // row of the tile <-> TMEM lane
        const int row = row0 + r;
        const uint32_t tl = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        bool ok = true;
        float o[D];
#pragma unroll
        for (int i = 0; i < D; ++i) o[i] = 0.f;
        float m = -INFINITY, l = 0.f, alpha_prev = 0.f;
        const long long rlim = static_cast<long long>(row) + 1 + coff;
        const int nrow = rlim < n ? (rlim < 0 ? 0 : static_cast<int>(rlim)) : n;
        const int nrow_min = __shfl_sync(0xffffffffu, nrow, 0);
        if (ntiles > 0) {
            // Q row -> TMEM, scaled by scale * log2(e) and split: the logits arrive in base-2 units
            // (the softmax groups take turns at the 32-feature panels of the tile)
            ok = whole_warp_wait(&bars[Q_FULL], 0, 0x650);
            if (ok) {
#pragma unroll
                for (int pn = g; pn < D / 32; pn += 2) {
                    uint32_t hi[32], lo[32];
#pragma unroll
                    for (int ch = 0; ch < 8; ++ch) {
                        const uint4 v = lds128(sb + OFF_VTH + pn * (BM * 128) + r * 128 + ((ch ^ (r & 7)) << 4));
                        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const uint32_t x = __float_as_uint(__uint_as_float(w[e]) * scale_log2e);
                            hi[ch * 4 + e] = hi_of<NEAR>(x);
                            lo[ch * 4 + e] = lo_of(x, hi[ch * 4 + e]);
                        }
                    }
                    tmem_st_x32(tl + QH_COL + pn * 32, hi);
                    tmem_st_x32(tl + QL_COL + pn * 32, lo);
                }
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars[Q_READY]);
            }
        }
        auto accumulate = [&](int k) {                       // O = alpha_k O + PV(k)  (k: a step of this group)
            ok = whole_warp_wait(&bars[PV_FULL + g], (k >> 1) & 1, 0x660 + g);
            if (!ok) return;
            tc_fence_after();
            constexpr int CH = 16;                           // (32 at a time: d = 64 1 % slower, d = 128 spills)
#pragma unroll
            for (int c = 0; c < D; c += CH) {
                uint32_t pv[CH];
                tmem_ld_x16(tl + PV_COL + (LY::PVS - 1) * D * g + c, pv);
                tc_wait_ld();
#pragma unroll
                for (int i = 0; i < CH; ++i) o[c + i] = fmaf(o[c + i], alpha_prev, __uint_as_float(pv[i]));
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars[PV_FREE + g]);
        };
        for (int j = g; j < ntiles && ok; j += 2) {
            // (the output of this group's previous step first: its products completed before S(j)'s did, and
            // P V(j) cannot be issued before that buffer is free again)
            if (j >= 2) accumulate(j - 2);
            if (!ok) break;
            ok = whole_warp_wait(&bars[S_FULL + g], (j >> 1) & 1, 0x670 + g);
            if (!ok) break;
            tc_fence_after();
            uint32_t s[BN];
#pragma unroll
            for (int c = 0; c < BN; c += 32) tmem_ld_x32(tl + S_COL + BN * g + c, *reinterpret_cast<uint32_t(*)[32]>(&s[c]));
            tc_wait_ld();
            const int col0 = j * BN;
            const int nvalid = nrow > col0 ? (nrow - col0 < BN ? nrow - col0 : BN) : 0;   // per row
            if (col0 + BN > nrow_min) {                      // (warp-uniform) some row has masked keys in this step
#pragma unroll
                for (int i = 0; i < BN; ++i) if (i >= nvalid) s[i] = __float_as_uint(-INFINITY);
            }
            float e0 = __uint_as_float(s[0]), e1 = __uint_as_float(s[1]), e2 = __uint_as_float(s[2]), e3 = __uint_as_float(s[3]);
#pragma unroll
            for (int i = 4; i < BN - 4; i += 8) {
                e0 = max3(e0, __uint_as_float(s[i]), __uint_as_float(s[i + 1]));
                e1 = max3(e1, __uint_as_float(s[i + 2]), __uint_as_float(s[i + 3]));
                e2 = max3(e2, __uint_as_float(s[i + 4]), __uint_as_float(s[i + 5]));
                e3 = max3(e3, __uint_as_float(s[i + 6]), __uint_as_float(s[i + 7]));
            }
            e0 = max3(e0, __uint_as_float(s[BN - 4]), __uint_as_float(s[BN - 3]));
            e1 = max3(e1, __uint_as_float(s[BN - 2]), __uint_as_float(s[BN - 1]));
            const float m_new = fmaxf(m, fmaxf(fmaxf(e0, e1), fmaxf(e2, e3)));
            // (a row that has seen no valid key yet has no maximum: 0 stands in, its weights are 2^-inf = 0)
            const float m_use = m_new == -INFINITY ? 0.f : m_new;
            const float alpha = ex2_approx(m - m_use);       // 0 on the row's first valid step
            m = m_new;
            const uint64_t neg_m2 = pack2(-m_use, -m_use);
            uint64_t lsum0 = 0ull, lsum1 = 0ull;
#pragma unroll
            for (int c = 0; c < BN / 16; ++c) {
                uint32_t hi[16], lo[16];
#pragma unroll
                for (int i = 0; i < 16; i += 2) {
                    float x0, x1;
                    unpack2(add2(pack2(__uint_as_float(s[c * 16 + i]), __uint_as_float(s[c * 16 + i + 1])), neg_m2), x0, x1);
                    hi[i] = __float_as_uint(ex2_approx(x0));
                    hi[i + 1] = __float_as_uint(ex2_approx(x1));
                }
#pragma unroll
                for (int i = 0; i < 16; i += 4) {
                    lsum0 = add2(lsum0, pack2(__uint_as_float(hi[i]), __uint_as_float(hi[i + 1])));
                    lsum1 = add2(lsum1, pack2(__uint_as_float(hi[i + 2]), __uint_as_float(hi[i + 3])));
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const uint32_t p = hi[i];
                    hi[i] = hi_of<NEAR>(p);
                    lo[i] = lo_of(p, hi[i]);
                }
                tmem_st_x16(tl + S_COL + BN * g + c * 16, hi);      // P_hi over the logits
                tmem_st_x16(tl + PL_COL + BN * g + c * 16, lo);
            }
            float l0, l1, l2, l3;
            unpack2(lsum0, l0, l1);
            unpack2(lsum1, l2, l3);
            l = fmaf(l, alpha, (l0 + l1) + (l2 + l3));
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars[P_FULL + g]);
            alpha_prev = alpha;
        }
        {
            // this group's last step
            const int last = ntiles - 1 - ((ntiles - 1 - g) & 1);   // largest j < ntiles with j % 2 == g (negative: none)
            if (ok && last >= 0) accumulate(last);
        }
        // Merge of the two streams.  The scratch lies over the K rings: the odd group must not write it before the even group has
        // passed its last P V too (with an odd number of key steps that one's logits are still to be computed from them when the
        // odd group is done); after that every product has completed and no copy is in flight.
        asm volatile("bar.sync 1, 256;" ::: "memory");
        float* scratch = reinterpret_cast<float*>(base + OFF_KH) + r * LY::MERGE_STRIDE;
        if (g == 1) {
#pragma unroll
            for (int v = 0; v < D / 4; ++v)
                *reinterpret_cast<float4*>(scratch + 4 * v) = make_float4(o[4 * v], o[4 * v + 1], o[4 * v + 2], o[4 * v + 3]);
            scratch[D] = ok ? m : __int_as_float(0x7fc00000);       // (a maximum is never NaN: max takes the other operand)
            scratch[D + 1] = l;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (g == 0) {
            const float m1 = scratch[D], l1 = scratch[D + 1];
            uint64_t zero[2] = {0ull, 0ull};                 // (NaN once a result is not finite)
            if (ok && m1 == m1 && row < Nq) {                // (a group that gave up leaves NaN: no output then)
                const float mt = fmaxf(m, m1);
                const float mu = mt == -INFINITY ? 0.f : mt;
                const float a0 = ex2_approx(m - mu), a1 = ex2_approx(m1 - mu);
                const float lt = l * a0 + l1 * a1;
                const float inv = lt > 0.f ? 1.f / lt : 0.f;
                if (lse) lse[static_cast<int64_t>(bh) * Nq + row] = lt > 0.f ? (mt + log2f(lt)) * 0.6931471805599453f : -INFINITY;
                const float w0 = a0 * inv, w1 = a1 * inv;
                float4* orow = reinterpret_cast<float4*>(O + (static_cast<int64_t>(bh) * Nq + row) * D);
#pragma unroll
                for (int v = 0; v < D / 4; ++v) {
                    const float4 q = *reinterpret_cast<const float4*>(scratch + 4 * v);
                    const float4 x = make_float4(o[4 * v] * w0 + q.x * w1, o[4 * v + 1] * w0 + q.y * w1, o[4 * v + 2] * w0 + q.z * w1,
                                                 o[4 * v + 3] * w0 + q.w * w1);
                    orow[v] = x;
                    if (NEAR) { zero[0] = fma2(pack2(x.x, x.y), 0ull, zero[0]); zero[1] = fma2(pack2(x.z, x.w), 0ull, zero[1]); }
                }
            }
            if (NEAR) {                                      // (at d = 64 the row stays as it is)
                float z0, z1;
                unpack2(add2(zero[0], zero[1]), z0, z1);
                const unsigned again = __ballot_sync(0xffffffffu, z0 + z1 != 0.f);
                if (again)
                    plain_rows<float, D>(again, static_cast<int64_t>(bh) * Nq + row0 + warp * 32, nrow, Q, K + static_cast<int64_t>(bh) * Nk * D,
                                         V + static_cast<int64_t>(bh) * Nk * D, O, lse, scale_log2e);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, TMEM_COLS);
}

// fp32 tensor [BH, N, D] viewed as 3-D {D, N, BH}; box = 32 floats x rows x 1 (one 128-byte-swizzled panel).
bool make_map_f32(CUtensorMap* m, const void* ptr, int BH, int N, int D, int box_rows) {
    EncodeTiledFn enc = get_encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(D), static_cast<cuuint64_t>(N), static_cast<cuuint64_t>(BH)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(D) * 4, static_cast<cuuint64_t>(N) * D * 4};
    cuuint32_t box[3] = {32, static_cast<cuuint32_t>(box_rows), 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int D>
int launch(const Problem& p, cudaStream_t st) {
    using LY = Layout<D>;
    CUtensorMap tmQ, tmK, tmV;
    const int BH = p.B * p.H, slabs = (p.Nq + BM - 1) / BM;
    if (static_cast<int64_t>(slabs) * BH > 0x7fffffff) return FLAT_ERR_SHAPE;
    if (!make_map_f32(&tmQ, p.Q, BH, p.Nq, D, BM) || !make_map_f32(&tmK, p.K, BH, p.Nk, D, LY::BN) ||
        !make_map_f32(&tmV, p.V, BH, p.Nk, D, LY::BN))
        return FLAT_ERR_CUDA;
    if (!ensure_dynamic_smem<fused_tf32_kernel<D>>(LY::SMEM_BYTES)) return FLAT_ERR_CUDA;
    // without the causal mask the tiles of a head run side by side and share K and V in L2; with it, those of as many heads as
    // fit L2 together (48 MB of K and V) go longest first: what is left at the end are the short ones
    const int64_t fit = (48ll << 20) / (static_cast<int64_t>(p.Nk) * D * 8);
    const int group = !p.causal || fit < 1 ? 1 : fit < BH ? static_cast<int>(fit) : BH;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(slabs) * BH);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = LY::SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, fused_tf32_kernel<D>, tmQ, tmK, tmV, static_cast<const float*>(p.Q), static_cast<const float*>(p.K),
                                             static_cast<const float*>(p.V), static_cast<float*>(p.O), BH, p.H, p.Nq, p.Nk,
                                             p.scale * 1.4426950408889634f, p.k_valid_len, p.causal ? p.Nk - p.Nq : (1 << 30), group, p.status, p.lse);
    return e == cudaSuccess ? FLAT_OK : FLAT_ERR_CUDA;
}

}  // namespace

bool tf32_applies(const Problem& p) {
    return p.dtype == FLAT_DTYPE_F32 && (p.d == 32 || p.d == 64 || p.d == 128) && !p.bias && !p.block_mask;
}

int launch_fused_tf32(const Problem& p, cudaStream_t st) {
    if (!tf32_applies(p)) return FLAT_ERR_UNSUPPORTED;
    return p.d == 32 ? launch<32>(p, st) : p.d == 64 ? launch<64>(p, st) : launch<128>(p, st);
}

}  // namespace flat
