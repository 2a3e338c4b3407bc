// Backward pass of the fused Logit-softmax-Attend on the sm_100a tensor cores (tcgen05 + TMEM + TMA):
// bf16 in, fp32 accumulate, bf16 gradients out.
//
// The paper stops at inference; this is the chain rule on its Section 2 steps 2-4, computed with the
// same idea as its Section 5 dataflow: the [Nq, Nk] intermediates (weights P, their gradient dP and the
// logit gradient dS) are rebuilt tile by tile on chip and never reach device memory.  With S = scale Q K^T,
// lse the row-wise log-sum-exp that the forward pass saved, P = exp(S - lse) and delta_i = sum_t dO[i,t] O[i,t]:
//     dV = P^T dO        dP = dO V^T        dS = P o (dP - delta)        dQ = scale dS K        dK = scale dS^T Q
// Two launches of one kernel template, no atomics and no workspace beyond delta [B,H,Nq]:
//   MODE_DQ : 128 query rows at a time, streaming key tiles:   S = Q K^T, dP = dO V^T, dQ += dS K.
//             Also computes delta for its rows and writes it for the second launch.
//   MODE_DKV: 128 keys at a time, streaming query tiles:       S^T = K Q^T, dP^T = V dO^T,
//             dV += P^T dO, dK += dS^T Q.
// Both are the same program: a stationary pair of tiles (X1, X2) whose rows are the TMEM lanes, a streamed
// pair (Y1, Y2) whose rows are the columns:  T1 = X1 Y1^T,  T2 = X2 Y2^T  (both operands K-major in shared
// memory), then element-wise p = 2^(c T1 - lse2), ds = p (T2 - delta) with lse2 / delta taken per lane
// (MODE_DQ) or per column (MODE_DKV), P and dS rounded to bf16 and written back to TMEM, and
// acc_a += dS Y1, acc_b += P Y2 with the bf16 tile as the TMEM A-operand and Y as an MN-major B-operand.
//
// What bounds it and how the work is arranged.  Cycles per 128 x 128 tile and launch on one SM: exponential unit 1024;
// tensor pipe 768 (dQ, d = 64), 1152 (dK dV, d = 64), 1536 and 2752 (d = 128).  Beside those two, what counts is what a
// role's loop costs while the exponential unit's queue is full (clock stamps): a barrier check 140-220 cycles even when
// the phase completed long ago.  Hence few barriers per step, wide MMAs, two issuing warps:
//  * SEP (every case but MODE_DKV at d = 128): the bf16 tiles P, dS have TMEM columns of their own, and the element-wise
//    warps pull T1 and T2 into registers and release them at once.  The next step's T1, T2 are then computed under this
//    step's exponentials, this step's accumulation under the next one's, and a warp that is ahead of the others goes on.
//    T1, T2 are whole tiles (N = 128: half as many instructions as N = 64, which with both operands in shared memory
//    also takes 48 cycles where its arithmetic takes 32: A alone is 4 KB of a port of 128 bytes a cycle).
//    MODE_DQ keeps its stationary operands in TMEM where there is room (both at d = 64, Q at d = 128).
//    What is left is the loop T seen -> in registers (470 cycles until the last warp has it) -> next T issued, computed and
//    seen (990): 1460 a step at d = 64.  Two column groups with barriers of their own, or T1 and T2 released apart, make
//    the loop shorter and the barrier checks more: 463 / 612 and 484 / 591 us against 458 / 555 (dQ / dK dV, B4 H16 4096).
//  * MODE_DKV at d = 128: the accumulators and T1, T2 fill TMEM.  P / dS overlay the columns of T they were computed
//    from, and the streamed tile is worked on in two halves of 64 columns: a half's accumulation first, then its next T
//    (the MMAs of one thread execute in issue order, so the T that overwrites P / dS needs no wait), both under the
//    element-wise work of the other half.  The streamed stage is released between the two: behind the T it came 1000
//    cycles too late for the copy after next (1243 against 965 us on B1 H4 16384).
//  * MODE_DKV: lse and delta belong to the columns.  Read from shared memory by every warp they cost 1024 cycles of the
//    port per tile (a broadcast read is one wavefront per column and warp); instead they join the contractions: one more
//    slice of 16 contraction indices, (1, 1, 1, 0 ...) on the stationary side and -lse / scale, or -delta, as the sum of
//    three bf16 numbers (24 bits) on the streamed side, gives T1 = K Q^T - lse / scale and T2 = V dO^T - delta.
//  * With more tiles than SMs a CTA that has issued the copies of its tile takes over a tile whose CTA has not started
//    (clusterlaunchcontrol), so that no tile pays for launch, allocation, barrier set-up and first loads (3,500 cycles), and the next
//    tile's operands and T are under way while this one's gradients are stored (MODE_DKV at d = 128: its operands; the warp that
//    issues T there issues the accumulations, too, and waits until the last ones have been read).  The stationary tiles come by
//    TMA and go to TMEM from shared memory, and delta's rows are read side by side: a lane per row, 16 bytes an instruction, took
//    6,600 (d = 64) and 14,300 cycles (128).
//    Between two tiles are now 3,300 / 3,800 cycles (dQ / dK dV, d = 64) and 5,800 / 7,100 (d = 128) instead of 11,100 / 6,900
//    and 20,600 / 11,000; a tile of 4096 rows has 48,000 to 98,000 cycles of steps.
//  * Waits by whole warps (warp_wait); what the compiler knows to be the same in all lanes is chosen per form (at the warp index).
//  * With no more tiles than SMs a form without any of the taking over: see launch_bwd_mode.
// Measured (both launches, us, a CTA per tile with waits lane by lane before / now): B4 H16 4096 x 4096 d 64 907 / 825, causal 551 / 458;
// B2 H16 3000 d 128 causal 287 / 235; B8 H8 512 d 64 35.7 / 27.2, d 128 55 / 39.7; B4 H8 256 d 64 13.2 / 11.5, d 128 21.3 / 15.9.
//
// CTA = 640 threads, an item at a time (a tile of the stationary operands; MULTI: its own and those it takes over): warps 0-15
// element-wise (warp w: TMEM lane quarter w % 4, 32 of a step's 128 columns: w / 4 -- four warps per scheduler), warp 16 TMA
// producer, warp 17 issues the T MMAs and warp 18 the accumulations (where P / dS overlay T, warp 17 issues both), warp 19 writes
// the slices that carry lse and delta (MODE_DKV).
// Under the causal mask the tiles of a head differ in length by a factor of their number: the longest tiles of a group of
// heads go first (launch_bwd_mode).
// Every wait is bounded (tc_common.cuh); on expiry the CTA aborts cleanly and reports a code.
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

constexpr int BT = 128;              // rows of every tile (queries or keys)
constexpr int HC = 64;               // columns (rows of the streamed tile) per half step (where the step has halves)
constexpr int EW_WARPS = 16;
constexpr int BWD_THREADS = 32 * EW_WARPS + 128;
constexpr int MODE_DQ = 0, MODE_DKV = 1;
constexpr float LOG2E = 1.4426950408889634f;

// n / d for n < 2^31 by a multiplication (Granlund and Montgomery 1994): with 2^(l - 1) < d <= 2^l and mul = ceil(2^(31 + l) / d) it is
// floor(n mul / 2^(31 + l)).  As divisions, the six places where an item is looked up took 1,000 cycles each and 9 KB of a kernel's
// instructions, which are fetched anew where kernels take turns: forward and backward, B3 H6 257^2 d 64, 26.2 -> 25.7 us; backward alone
// 14.7 -> 14.4, B4 H8 256^2 13.15 -> 12.75.
struct Divisor {
    uint32_t d, mul, shift;
    Divisor() = default;
    constexpr explicit Divisor(uint32_t d_) : d(d_), mul(0), shift(0) {
        if (d > 1) {
            uint32_t l = 1;
            while (l < 31 && (1u << l) < d) ++l;
            mul = static_cast<uint32_t>(((1ull << (31 + l)) + d - 1) / d);
            shift = l - 1;
        }
    }
    __host__ __device__ constexpr uint32_t of(uint32_t n) const {
        return d == 1 ? n : static_cast<uint32_t>((static_cast<uint64_t>(n) * mul) >> 32) >> shift;
    }
};
static_assert(Divisor(1).of(0x7fffffff) == 0x7fffffff && Divisor(2).of(0x7fffffff) == 0x3fffffff && Divisor(7).of(0x7ffffffe) == 0x12492492 &&
              Divisor(7).of(6) == 0 && Divisor(641).of(641 * 3350208u - 1) == 3350207 && Divisor(0x40000001).of(0x7fffffff) == 1 &&
              Divisor(0x7fffffff).of(0x7ffffffe) == 0 && Divisor(0x7fffffff).of(0x7fffffff) == 1, "division");

template <int D, int MODE> struct BL {
    static constexpr bool DKV = MODE == MODE_DKV;
    static constexpr bool SEP = !(D == 128 && DKV);
    static constexpr bool X1_TMEM = !DKV, X2_TMEM = !DKV && D == 64;   // stationary operand in TMEM, else in shared memory
    static constexpr int TILE_BYTES = BT * D * 2;
    static constexpr bool X_SMEM = !X1_TMEM || !X2_TMEM;                     // some stationary operand is read by MMAs from shared memory
    static constexpr int X_BYTES = 2 * TILE_BYTES;       // (an operand that goes to TMEM is staged here)
    // Rings of streamed tiles (SEP: whole ones; else halves of 64 rows), deep enough that a copy (one to two microseconds)
    // is under way for every step in work.  MODE_DQ needs Y2 = V for T2 only, so that its slots are free again early.
    static constexpr int PARTS = SEP ? 1 : 2;            // copies per step; also column groups with T, dS and barriers of their own
    static constexpr int Y_ROWS = BT / PARTS, Y_BYTES = Y_ROWS * D * 2;
    static constexpr int S1 = DKV ? 4 : D == 64 ? 5 : 3, S2 = DKV ? 4 : D == 64 ? 4 : 2;
    static constexpr int OPERAND_BYTES = X_BYTES + (S1 + S2) * Y_BYTES;
    // (MODE_DKV) slices of 16 contraction indices, 128 rows of 32 bytes: the ones; per stage (whole steps) -lse / scale and -delta
    static constexpr int AUG_BYTES = BT * 32;
    static constexpr int VSTAGES = DKV ? S1 / PARTS : 1;
    static constexpr int AUG_ALL = DKV ? (1 + 2 * VSTAGES) * AUG_BYTES : 0;
    static constexpr int DELTA_BYTES = DKV ? 0 : 2 * BT * 4;                 // delta of the rows (MODE_DQ), of two items in turn
    static constexpr int SMEM_BYTES = OPERAND_BYTES + AUG_ALL + DELTA_BYTES + 512 + 1024;
    static_assert(SMEM_BYTES <= 232448, "shared memory");
    static constexpr uint32_t T1_COL = 0, T2_COL = 128, ACC_A_COL = 256, ACC_B_COL = 256 + D;
    static constexpr uint32_t ACC_END = 256 + (DKV ? 2 : 1) * D;
    // (SEP) bf16 tiles: dS 64 columns, P 64 (MODE_DKV) or the stationary operands (MODE_DQ)
    static constexpr uint32_t P_COL = ACC_END + 64, X1_COL = ACC_END + 64, X2_COL = X1_COL + D / 2;
    static constexpr uint32_t TMEM_COLS = 512;
    static_assert(!SEP || (DKV ? P_COL + 64 : X1_COL + D / 2 + (X2_TMEM ? D / 2 : 0)) <= TMEM_COLS, "tensor memory");
    // columns of the bf16 dS / P tile that warp group g (32 of the step's columns each, 0..3) writes, and of contraction
    // slice k (16 indices, k = 0..7); without SEP each lies over the logits it came from
    __host__ __device__ static constexpr uint32_t ds_store(int g) { return SEP ? ACC_END + g * 16 : T2_COL + g * 32; }
    __host__ __device__ static constexpr uint32_t p_store(int g) { return SEP ? P_COL + g * 16 : T1_COL + g * 32; }
    __host__ __device__ static constexpr uint32_t ds_slice(int k) { return ds_store(k / 2) + (k % 2) * 8; }
    __host__ __device__ static constexpr uint32_t p_slice(int k) { return p_store(k / 2) + (k % 2) * 8; }
    static_assert(SEP || (p_slice(4) == p_slice(0) + HC && ds_slice(4) == ds_slice(0) + HC && p_slice(7) == p_slice(3) + HC), "halves");
    // barriers.  Per item: X_FULL: stationary tiles in shared memory; X_TMEM: in TMEM (one arrival per element-wise warp);
    // X_EMPTY: the T MMAs that read them from shared memory have completed (where none do: warp 17 has seen X_TMEM);
    // ACC_DONE: everything accumulated; ACC_FREE: the accumulators are in registers; ITEM_FULL / ITEM_EMPTY [2]: the next item
    // is known / read by every warp; DELTA (MODE_DQ): delta of the item's rows is in shared memory.
    // Y_FULL [S1]: the copy's Y1 and Y2 have landed (and, MODE_DKV, warp 19 has written the step's slices);
    // Y1_EMPTY [S1], Y2_EMPTY [S2] (MODE_DQ): read; ACC_STEP (SEP): the MMAs that read dS, P have completed;
    // per column group: T_FULL: T1, T2 computed; PD_FULL: dS (and P) written; T_FREE (SEP): T1, T2
    // taken into registers.  Without SEP warp 18 arrives on PD_FULL, too, once the half's next copy has landed, so that the
    // issuing warp has one barrier to look at.
    static constexpr int BAR_X_FULL = 0, BAR_X_TMEM = 1, BAR_X_EMPTY = 2, BAR_ACC_FREE = 3, BAR_ITEM_FULL = 4, BAR_ITEM_EMPTY = 6,
                         BAR_DELTA = 8, BAR_Y_FULL = 9, BAR_Y1_EMPTY = BAR_Y_FULL + S1,
                         BAR_Y2_EMPTY = BAR_Y1_EMPTY + S1, BAR_ACC_STEP = BAR_Y2_EMPTY + S2, BAR_ACC_DONE = BAR_ACC_STEP + 1,
                         BAR_T_FULL = BAR_ACC_DONE + 1, BAR_T_FREE = BAR_T_FULL + PARTS, BAR_PD_FULL = BAR_T_FREE + 1,
                         NUM_BARS = BAR_PD_FULL + PARTS;
    static constexpr int PD_ARRIVALS = SEP ? EW_WARPS : EW_WARPS / 2 + 1;
    static constexpr int READERS = EW_WARPS + (DKV ? 3 : 2);                 // warps that read an item: all but the producer
    __host__ __device__ static constexpr int arrivals(int i) {
        return i == BAR_X_TMEM || i == BAR_ACC_FREE || i == BAR_T_FREE || i == BAR_DELTA ? EW_WARPS
               : i == BAR_ITEM_EMPTY || i == BAR_ITEM_EMPTY + 1 ? READERS
               : i >= BAR_Y_FULL && i < BAR_Y1_EMPTY && DKV ? 2 : i >= BAR_PD_FULL ? PD_ARRIVALS : 1;
    }
    static_assert(NUM_BARS * 8 + 16 + 32 <= 512, "barriers");
};

// Shared-memory descriptor of a slice tile: K-major rows of 32 bytes, 32-byte swizzle, eight rows 256 bytes apart.
__device__ __forceinline__ uint64_t aug_desc(uint32_t smem_addr) {
    return static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4) | (1ull << 16) | (static_cast<uint64_t>(256 >> 4) << 32) | (1ull << 46) | (6ull << 61);
}
// Row r of a slice tile: x as the sum of three bf16 numbers, the other thirteen elements zero (the second 16 bytes of a row
// are written once, by the clearing pass).  The swizzle exchanges the two halves of a row where bit 2 of r is set.
__device__ __forceinline__ void aug_store(uint8_t* tile, int r, float x) {
    const float hi = __bfloat162float(__float2bfloat16_rn(x)), rest = x - hi, mid = __bfloat162float(__float2bfloat16_rn(rest));
    *reinterpret_cast<uint4*>(tile + r * 32 + ((r >> 2) & 1) * 16) = make_uint4(pack_bf16x2(hi, mid), pack_bf16x2(rest - mid, 0.f), 0u, 0u);
}

// What the logits are multiplied by in the exponent (base 2).  Not below 1e-30: -lse / scale must be a number, and whatever
// 1e-30 times a logit is, it is nothing beside the exponent.
__device__ __forceinline__ float exponent_factor(float scale) {
    const float c = scale * LOG2E;
    return fabsf(c) >= 1e-30f ? c : 1e-30f;
}

// How items lie in the grid: group x tiles of them at a time, heads of a group, of the last one if it has fewer; heads of a batch.
struct Places { Divisor per, group, rest, H; };

// X1, X2 / Y1, Y2 by mode:  MODE_DQ: (Q, dO) / (K, V);  MODE_DKV: (K, V) / (Q, dO).
template <int D, int MODE, bool MULTI>
__global__ void __launch_bounds__(BWD_THREADS, 1)
bwd_tc_kernel(const __grid_constant__ CUtensorMap tmX1, const __grid_constant__ CUtensorMap tmX2,
              const __grid_constant__ CUtensorMap tmY1, const __grid_constant__ CUtensorMap tmY2,
              const __nv_bfloat16* __restrict__ X1g, const __nv_bfloat16* __restrict__ X2g, const __nv_bfloat16* __restrict__ Og,
              const float* __restrict__ lse, float* __restrict__ delta,
              __nv_bfloat16* __restrict__ outA, __nv_bfloat16* __restrict__ outB,
              int BH, int Nq, int Nk, float scale, const int32_t* __restrict__ valid_len, int coff, const Places pl, int32_t* status) {
    using LY = BL<D, MODE>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* X1s = base;
    uint8_t* X2s = X1s + LY::TILE_BYTES;
    uint8_t* Y1s = base + LY::X_BYTES;                   // rings of streamed tiles
    uint8_t* Y2s = Y1s + LY::S1 * LY::Y_BYTES;
    uint8_t* aug = base + LY::OPERAND_BYTES;             // (MODE_DKV) ones, then per stage -lse / scale and -delta
    float* dls = reinterpret_cast<float*>(base + LY::OPERAND_BYTES + LY::AUG_ALL);
    uint8_t* next_item = base + LY::OPERAND_BYTES + LY::AUG_ALL + LY::DELTA_BYTES;           // two answers of 16 bytes
    uint64_t* bars = reinterpret_cast<uint64_t*>(next_item + 32);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + LY::NUM_BARS);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int* first_item = reinterpret_cast<int*>(tmem_slot + 2);

    // Roles go by an index that the compiler knows to be the same in all lanes, and so does everything else but for the roles of
    // MODE_DQ with several tiles (with it / without: 128 rows against 16384 keys, d = 64 114 / 104 us, d = 128 138 / 132; MODE_DKV 16384
    // rows against 128 keys 124 / 128 and 231 / 249; roles by the other one, too: 107).
    const int role = warp_index(), warp = MULTI && MODE == MODE_DQ ? threadIdx.x >> 5 : role, lane = threadIdx.x & 31;
    const int NX = MODE == MODE_DQ ? Nq : Nk;            // rows of the stationary tensors
    const int tiles = (NX + BT - 1) / BT;

    if (threadIdx.x == EW_WARPS * 32) {
        for (int i = 0; i < LY::NUM_BARS; ++i) mbar_init(&bars[i], LY::arrivals(i));
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0) { tmem_alloc(tmem_slot, LY::TMEM_COLS); tmem_relinquish(); }
    if (LY::DKV) {                                       // clear the slice tiles and write the ones
        for (int i = threadIdx.x; i < LY::AUG_ALL / 16; i += BWD_THREADS) {
            const int r = i >> 1;                        // (row of the first tile)
            const bool ones = i < LY::AUG_BYTES / 16 && (i & 1) == ((r >> 2) & 1);
            reinterpret_cast<uint4*>(aug)[i] = ones ? make_uint4(0x3f803f80u, 0x00003f80u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
        }
        fence_proxy_async_smem();
    }
    // Item -> (head, tile): `group` heads at a time, their tiles side by side, the longest first under the causal mask
    // (the last query tiles, the first key tiles); its range of streamed tiles, those with at least one visible (query, key)
    // pair.  Causal mask (coff = Nk - Nq; 2^30 = none): query i sees key j iff j <= i + coff.
    int bh, x0, nkeys, y_begin, nsteps;                  // nkeys: keys of this batch that take part at all
    auto place = [&](int item, int& head, int& row) {
        const uint32_t g = pl.per.of(item), at = item - g * pl.per.d, first_head = g * pl.group.d;
        const bool rest = BH - first_head < pl.group.d;  // (fewer heads in the last group)
        const uint32_t heads = rest ? pl.rest.d : pl.group.d, tile = rest ? pl.rest.of(at) : pl.group.of(at);
        head = first_head + at - tile * heads;
        row = (MODE == MODE_DQ && coff < (1 << 29) ? tiles - 1 - tile : tile) * BT;
    };
    // (the first item's here, by one thread, under the tail of the previous kernel)
    if (threadIdx.x == 0) place(blockIdx.x, first_item[0], first_item[1]);

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // (launched with programmatic stream serialization: nothing in device memory is touched before the previous kernel of
    // the stream -- the forward pass, or the dQ launch that writes delta -- has finished)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    const uint32_t bars_s = smem_u32(bars), abort_s = smem_u32(const_cast<int*>(abort_flag)), next_s = smem_u32(next_item);
    auto wait_warp = [&](int bar, uint32_t parity, int code) {
        return warp_wait(bars_s + 8 * bar, parity, abort_s, status, code);
    };

    auto decode = [&](int item) {
        if (!MULTI || item == static_cast<int>(blockIdx.x)) {
            bh = __shfl_sync(0xffffffffu, first_item[0], 0);
            x0 = __shfl_sync(0xffffffffu, first_item[1], 0);
        } else {
            place(item, bh, x0);
        }
        nkeys = Nk;
        if (valid_len) {
            nkeys = __shfl_sync(0xffffffffu, valid_len[pl.H.of(bh)], 0);
            nkeys = nkeys < 0 ? 0 : (nkeys > Nk ? Nk : nkeys);
        }
        y_begin = 0;
        int y_end;
        if (MODE == MODE_DQ) {
            const long long lim = static_cast<long long>(x0) + BT + coff;      // keys below this for the tile's last row
            const int n = lim < nkeys ? (lim < 0 ? 0 : static_cast<int>(lim)) : nkeys;
            y_end = (n + BT - 1) / BT;
        } else {
            y_end = x0 < nkeys ? (Nq + BT - 1) / BT : 0;
            const long long first = static_cast<long long>(x0) - coff;         // first query that sees key x0
            if (first > 0) y_begin = static_cast<int>(first / BT < y_end ? first / BT : y_end);
        }
        nsteps = y_end - y_begin;
    };
    // The n-th item (n > 0) that this CTA has taken over from one of the grid that had not started; -1: there was none left,
    // -2: gave up.  (The reader's fence orders its read before the next answer, which comes through the asynchronous proxy.)
    auto take_item = [&](int n) {
        if (!MULTI) return -1;
        const int slot = (n - 1) & 1;
        if (!wait_warp(LY::BAR_ITEM_FULL + slot, ((n - 1) >> 1) & 1, 0x570)) return -2;
        const int item = __shfl_sync(0xffffffffu, clc_answer(next_s + 16 * slot), 0);
        fence_proxy_async_smem();
        __syncwarp();
        if (warp != EW_WARPS && lane == 0) mbar_arrive_s(bars_s + 8 * (LY::BAR_ITEM_EMPTY + slot));
        __syncwarp();
        return item;
    };

    // Every role walks the same items; n: the item's number, gs: steps before it, ne: items before it that had steps.
    // The rings and the phases of the per-step barriers run on over the items.
    if (role >= EW_WARPS) {
      if (role == EW_WARPS) {
        // ------------------------------------------------------------ TMA producer (lane 0 issues the copies)
        if (lane == 0) { prefetch_tensormap(&tmX1); prefetch_tensormap(&tmX2); prefetch_tensormap(&tmY1); prefetch_tensormap(&tmY2); }
        // The next item is asked for some steps before the end of this one (six: early enough for what follows, late enough that
        // no CTA sits on work while another has none) and its stationary rows are brought to L2: the CTAs come to the ends of
        // their items together, and 64 to 96 KB for every SM at once take 2,500 to 5,500 cycles from DRAM.
        constexpr int LEAD = 6 * LY::PARTS;
        bool ok = true;
        int G = 0, n = 0, xs = 0, asked = 0;             // copies, items, stationary pairs and questions so far
        auto ask = [&]() {
            if (n >= 2) ok = wait_warp(LY::BAR_ITEM_EMPTY + (n & 1), ((n >> 1) - 1) & 1, 0x505);
            if (ok && lane == 0) {
                mbar_arrive_expect_tx(&bars[LY::BAR_ITEM_FULL + (n & 1)], 16);
                clc_ask(next_s + 16 * (n & 1), bars_s + 8 * (LY::BAR_ITEM_FULL + (n & 1)));
            }
            asked = n + ok;
        };
        auto answer = [&]() {
            const int next = take_item(n + 1);
            if (next >= 0 && lane == 0) {
                int head, row;
                place(next, head, row);
                const uint32_t bytes = static_cast<uint32_t>((NX - row < BT ? NX - row : BT) * D * 2);
                const int64_t at = (static_cast<int64_t>(head) * NX + row) * D;
                prefetch_l2(X1g + at, bytes);
                prefetch_l2(X2g + at, bytes);
                if (!LY::DKV) prefetch_l2(Og + at, bytes);
            }
            return next;
        };
        int item = blockIdx.x;
        while (item >= 0) {
            decode(item);
            if (MULTI && n > 0) {                        // the previous item's stationary tiles are read
                ok = wait_warp(LY::BAR_X_EMPTY, (n - 1) & 1, 0x503);
                if (ok && LY::X1_TMEM) ok = wait_warp(LY::BAR_X_TMEM, (n - 1) & 1, 0x504);
                if (!ok) break;
            }
            if (lane == 0) {
                mbar_arrive_expect_tx(&bars[LY::BAR_X_FULL], LY::X_BYTES);
#pragma unroll
                for (int c = 0; c < D / 64; ++c) {
                    tma_load_3d(X1s + c * BT * 128, &tmX1, &bars[LY::BAR_X_FULL], c * 64, x0, bh);
                    tma_load_3d(X2s + c * BT * 128, &tmX2, &bars[LY::BAR_X_FULL], c * 64, x0, bh);
                }
            }
            xs = n + 1;
            const int copies = LY::PARTS * nsteps, ask_at = copies > LEAD ? copies - LEAD : 0;
            int next = -3;                               // (not known yet)
            for (int g = 0; g < copies && ok; ++g) {
                const int s1 = G % LY::S1, s2 = G % LY::S2, y = y_begin * BT + g * LY::Y_ROWS;
                if (MULTI && g == ask_at) ask();
                if (MULTI && ok && g == ask_at + 2 * LY::PARTS) next = answer();
                if (!ok || next == -2) break;
                ok = wait_warp(LY::BAR_Y1_EMPTY + s1, ((G / LY::S1) & 1) ^ 1, 0x500);
                if (!LY::DKV && ok) ok = wait_warp(LY::BAR_Y2_EMPTY + s2, ((G / LY::S2) & 1) ^ 1, 0x501);
                if (!ok) break;
                if (lane == 0) {
                    mbar_arrive_expect_tx(&bars[LY::BAR_Y_FULL + s1], 2 * LY::Y_BYTES);
#pragma unroll
                    for (int c = 0; c < D / 64; ++c) {
                        tma_load_3d(Y1s + s1 * LY::Y_BYTES + c * LY::Y_ROWS * 128, &tmY1, &bars[LY::BAR_Y_FULL + s1], c * 64, y, bh);
                        tma_load_3d(Y2s + s2 * LY::Y_BYTES + c * LY::Y_ROWS * 128, &tmY2, &bars[LY::BAR_Y_FULL + s1], c * 64, y, bh);
                    }
                }
                ++G;
            }
            if (MULTI && ok && copies == 0) ask();
            if (ok && next == -3) next = MULTI ? answer() : -1;
            if (!ok) break;
            item = next;
            ++n;
        }
        if (lane == 0) {                                 // (where everything went well these have all completed)
            if (xs > 0) drain_wait(&bars[LY::BAR_X_FULL], (xs - 1) & 1);
            if (!ok || item == -2)
                for (int g = G > LY::S1 ? G - LY::S1 : 0; g < G; ++g) drain_wait(&bars[LY::BAR_Y_FULL + g % LY::S1], (g / LY::S1) & 1);
            if (MULTI && asked > 0) drain_wait(&bars[LY::BAR_ITEM_FULL + ((asked - 1) & 1)], ((asked - 1) >> 1) & 1);
        }
      } else if (LY::DKV && warp == EW_WARPS + 3) {
        // ------------------------------------------------------------ the slices that carry lse and delta (MODE_DKV)
        // Four queries per lane and step, fetched a step ahead.  A query that is switched off (no visible key, or past the
        // end) gets a first term so large that 2^(c T1) is 0 whatever its logits are.
        const float ce = exponent_factor(scale), inv = -LOG2E / ce, off = copysignf(3e38f, -ce);
        float l[4], dl[4];
        auto fetch = [&](int j) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = (y_begin + j) * BT + e * 32 + lane;
                l[e] = i < Nq ? lse[static_cast<int64_t>(bh) * Nq + i] : -INFINITY;
                dl[e] = i < Nq ? delta[static_cast<int64_t>(bh) * Nq + i] : 0.f;
            }
        };
        bool ok = true;
        int n = 0, gs = 0;
        for (int item = blockIdx.x; item >= 0 && ok; item = take_item(++n)) {
            decode(item);
            if (nsteps > 0) fetch(0);
            for (int j = 0; j < nsteps && ok; ++j, ++gs) {
                const int v = gs % LY::VSTAGES, g = LY::PARTS * gs + LY::PARTS - 1;   // the step's (last) copy
                float x[4], y[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    x[e] = l[e] == -INFINITY ? off : l[e] * inv;
                    x[e] = x[e] > 3e38f ? 3e38f : x[e] < -3e38f ? -3e38f : x[e];
                    y[e] = -dl[e];
                }
                if (j + 1 < nsteps) fetch(j + 1);
                // (slot v was last read by the T MMAs of step gs - VSTAGES; that step has released the stage of this step's
                // (last) copy behind its accumulation, i.e. after them)
                ok = wait_warp(LY::BAR_Y1_EMPTY + g % LY::S1, ((g / LY::S1) & 1) ^ 1, 0x502);
                if (!ok) break;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    aug_store(aug + (1 + 2 * v) * LY::AUG_BYTES, e * 32 + lane, x[e]);
                    aug_store(aug + (2 + 2 * v) * LY::AUG_BYTES, e * 32 + lane, y[e]);
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&bars[LY::BAR_Y_FULL + g % LY::S1]);
                    if (LY::PARTS == 2) mbar_arrive(&bars[LY::BAR_Y_FULL + (g - 1) % LY::S1]);
                }
            }
        }
      } else if (warp == EW_WARPS + 1 || warp == EW_WARPS + 2) {
        // ------------------------------------------------------------ MMA issuers
        //   T(j):   T1 = X1 Y1^T and T2 = X2 Y2^T (+ the slices);   ACC(j): acc_a += dS Y1 (and acc_b += P Y2).
        // SEP: warp 17 issues T(j+1) as soon as T(j) is in registers, warp 18 ACC(j) as soon as dS (and P) are written.
        // Otherwise warp 17 issues, per half, ACC(j) and behind it T(j+1).
        // The whole warp walks the loop (uniform control flow) and one elected lane issues: the MMA and
        // commit instructions take their operands from uniform registers, which the compiler can only
        // use when it knows that a single thread runs the code.
        constexpr int YR = LY::Y_ROWS;
        constexpr uint32_t IDESC_T = make_idesc_bf16(BT, YR, 0, 0), IDESC_ACC = make_idesc_bf16(BT, D, 0, 1);
        constexpr uint64_t Y16 = LY::Y_BYTES >> 4, AUG16 = LY::AUG_BYTES >> 4;           // descriptor units of 16 bytes
        // descriptors of the first feature slice of each operand (the others are constant offsets away)
        const uint64_t x1d = make_smem_desc_sw128(smem_u32(X1s), 16, 1024);            // K-major
        const uint64_t x2d = make_smem_desc_sw128(smem_u32(X2s), 16, 1024);
        const uint64_t y1k = make_smem_desc_sw128(smem_u32(Y1s), 16, 1024), y2k = make_smem_desc_sw128(smem_u32(Y2s), 16, 1024);
        const uint64_t y1m = make_smem_desc_sw128(smem_u32(Y1s), YR * 128, 1024);      // MN-major
        const uint64_t y2m = make_smem_desc_sw128(smem_u32(Y2s), YR * 128, 1024);
        const uint64_t augd = aug_desc(smem_u32(aug));
        // Consecutive MMAs into ONE accumulator wait for each other, so the slices of independent
        // products are issued in turn: T1 and T2, and the accumulations acc_a and acc_b.
        // (feature slice k of a K-major operand: panel k / 4 of 64 features, 32 bytes per slice; a panel
        // is 128 rows of 128 bytes for the stationary tiles, YR rows for the streamed ones)
        // g: the copy (of all items); where a step is two copies, their halves of the columns
        auto issue_t = [&](int g) {
            const int half = LY::PARTS == 2 ? g & 1 : 0;
            const uint64_t y1 = y1k + static_cast<uint64_t>(g % LY::S1) * Y16, y2 = y2k + static_cast<uint64_t>(g % LY::S2) * Y16;
            const uint32_t t1 = tmem + LY::T1_COL + half * HC, t2 = tmem + LY::T2_COL + half * HC;
#pragma unroll
            for (int k = 0; k < D / 16; ++k) {
                const uint64_t xoff = static_cast<uint64_t>(((k / 4) * (BT * 128) + (k % 4) * 32) >> 4);
                const uint64_t yoff = static_cast<uint64_t>(((k / 4) * (YR * 128) + (k % 4) * 32) >> 4);
                if (LY::X1_TMEM) mma_ts(t1, tmem + LY::X1_COL + k * 8, y1 + yoff, IDESC_T, k > 0);
                else             mma_ss(t1, x1d + xoff, y1 + yoff, IDESC_T, k > 0);
                if (LY::X2_TMEM) mma_ts(t2, tmem + LY::X2_COL + k * 8, y2 + yoff, IDESC_T, k > 0);
                else             mma_ss(t2, x2d + xoff, y2 + yoff, IDESC_T, k > 0);
            }
            if (LY::DKV) {
                const uint64_t av = augd + static_cast<uint64_t>(1 + 2 * ((g / LY::PARTS) % LY::VSTAGES)) * AUG16 + static_cast<uint64_t>((half * HC * 32) >> 4);
                mma_ss(t1, augd, av, IDESC_T, 1);
                mma_ss(t2, augd, av + AUG16, IDESC_T, 1);
            }
            tc_commit(&bars[LY::BAR_T_FULL + half]);
            if (!LY::DKV) tc_commit(&bars[LY::BAR_Y2_EMPTY + g % LY::S2]);
        };
        // first / last: of the item's copies
        auto issue_acc = [&](int g, bool first, bool last) {
            const uint32_t pd = tmem + (LY::PARTS == 2 ? (g & 1) * HC : 0);
            const uint64_t y1 = y1m + static_cast<uint64_t>(g % LY::S1) * Y16, y2 = y2m + static_cast<uint64_t>(g % LY::S2) * Y16;
#pragma unroll
            for (int k = 0; k < YR / 16; ++k) {
                mma_ts(tmem + LY::ACC_A_COL, pd + LY::ds_slice(k), y1 + static_cast<uint64_t>((k * 2048) >> 4), IDESC_ACC, (!first || k > 0));
                if (LY::DKV)
                    mma_ts(tmem + LY::ACC_B_COL, pd + LY::p_slice(k), y2 + static_cast<uint64_t>((k * 2048) >> 4), IDESC_ACC, (!first || k > 0));
            }
            if (LY::SEP) tc_commit(&bars[LY::BAR_ACC_STEP]);
            tc_commit(&bars[LY::BAR_Y1_EMPTY + g % LY::S1]);
            if (last) tc_commit(&bars[LY::BAR_ACC_DONE]);
        };
        auto y_full = [&](int g, int code) { return wait_warp(LY::BAR_Y_FULL + g % LY::S1, (g / LY::S1) & 1, code); };
        auto acc_free = [&](int ne) { return ne == 0 || wait_warp(LY::BAR_ACC_FREE, (ne - 1) & 1, 0x512); };
        bool ok = true;
        int n = 0, gs = 0, ne = 0;
        for (int item = blockIdx.x; item >= 0 && ok; item = take_item(++n)) {
            decode(item);
            if (warp == EW_WARPS + 1) {
                if (LY::X_SMEM) ok = wait_warp(LY::BAR_X_FULL, n & 1, 0x510);
                if (ok && LY::X1_TMEM) ok = wait_warp(LY::BAR_X_TMEM, n & 1, 0x511);
                if (!LY::X_SMEM && ok && lane == 0) mbar_arrive(&bars[LY::BAR_X_EMPTY]);
                __syncwarp();
            }
            if (LY::SEP && warp == EW_WARPS + 1) {
                for (int j = 0; j < nsteps && ok; ++j) {
                    const int g = gs + j;
                    ok = y_full(g, 0x520);
                    if (ok && g > 0) ok = wait_warp(LY::BAR_T_FREE, (g & 1) ^ 1, 0x522);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) issue_t(g);
                    __syncwarp();
                }
                if (LY::X_SMEM && ok) {
                    if (elect_one()) tc_commit(&bars[LY::BAR_X_EMPTY]);
                    __syncwarp();
                }
            } else if (LY::SEP) {
                if (nsteps > 0) ok = acc_free(ne);
                for (int j = 0; j < nsteps && ok; ++j) {
                    const int g = gs + j;
                    ok = y_full(g, 0x523);
                    if (ok) ok = wait_warp(LY::BAR_PD_FULL, g & 1, 0x530);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) issue_acc(g, j == 0, j == nsteps - 1);
                    __syncwarp();
                }
            } else if (warp == EW_WARPS + 1) {
                // (copy g of the item: half g & 1 of its columns; -2, -1: only the first T of the halves)
                const int g0 = 2 * gs, copies = 2 * nsteps;
                if (copies > 0 && ok) ok = acc_free(ne);
                for (int g = copies > 0 ? -2 : 0; g < copies && ok; ++g) {
                    ok = g < 0 ? y_full(g0 + g + 2, 0x520) : wait_warp(LY::BAR_PD_FULL + (g & 1), ((g0 + g) >> 1) & 1, 0x531);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        if (g >= 0) issue_acc(g0 + g, g == 0, g == copies - 1);
                        if (g + 2 < copies) issue_t(g0 + g + 2);
                    }
                    __syncwarp();
                    if (g + 3 == copies) {               // (behind the last T)
                        if (elect_one()) tc_commit(&bars[LY::BAR_X_EMPTY]);
                        __syncwarp();
                    }
                }
                if (copies == 0 && ok) {
                    if (elect_one()) tc_commit(&bars[LY::BAR_X_EMPTY]);
                    __syncwarp();
                }
            } else {
                // (the half's next copy: looked at here, so that the issuing warp does not have to; not before the half's
                // previous phase is over, which this arrival does not belong to)
                const int g0 = 2 * gs, copies = 2 * nsteps;
                for (int g = 0; g < copies && ok; ++g) {
                    if (g + 2 < copies) ok = y_full(g0 + g + 2, 0x521);
                    if (ok && g0 + g >= 2) ok = wait_warp(LY::BAR_PD_FULL + (g & 1), (((g0 + g) >> 1) - 1) & 1, 0x532);
                    if (ok && lane == 0) mbar_arrive(&bars[LY::BAR_PD_FULL + (g & 1)]);
                    __syncwarp();
                }
            }
            gs += nsteps;
            ne += nsteps > 0;
        }
      }
    } else {
        // ------------------------------------------------------------ element-wise + epilogue (warps 0-15)
        const int q = warp & 3, part = warp >> 2;        // lane quarter, 32 of the step's columns
        const int r = q * 32 + lane;                     // lane of the TMEM = row of the stationary tile
        const uint32_t tl = tmem + (static_cast<uint32_t>(q * 32) << 16);
        const float c2 = exponent_factor(scale);
        const bool wide = ((reinterpret_cast<uintptr_t>(outA) | (LY::DKV ? reinterpret_cast<uintptr_t>(outB) : 0)) & 31) == 0;
        bool ok = true;
        // MODE_DQ, per row: lse in base-2 units (+inf switches a row off: no key, or past the end) and delta
        float lse2_r = INFINITY, delta_r = 0.f;
        // MODE_DQ: brings the item's stationary operands from shared memory to TMEM (a quarter of the features a warp; all T
        // MMAs of the previous item have completed: their results have been seen here) and computes delta = sum_t dO O:
        // eight rows a warp, a row's features side by side in its lanes.
        constexpr int LPR = D / 8, ROWS = 32 / LPR, PASSES = 8 / ROWS;       // lanes a row, rows a pass
        auto begin_item = [&](int n) {
            if constexpr (!LY::DKV) {
                uint4 da[PASSES], db[PASSES];
#pragma unroll
                for (int i = 0; i < PASSES; ++i) {
                    const int row = x0 + warp * 8 + i * ROWS + lane / LPR;
                    da[i] = db[i] = make_uint4(0u, 0u, 0u, 0u);
                    if (row < Nq) {
                        const int64_t at = (static_cast<int64_t>(bh) * Nq + row) * D + (lane % LPR) * 8;
                        da[i] = *reinterpret_cast<const uint4*>(X2g + at);
                        db[i] = *reinterpret_cast<const uint4*>(Og + at);
                    }
                }
                const float l = x0 + r < Nq ? lse[static_cast<int64_t>(bh) * Nq + x0 + r] : -INFINITY;
                if (!wait_warp(LY::BAR_X_FULL, n & 1, 0x541)) return false;
                auto to_tmem = [&](const uint8_t* X, uint32_t col) {
                    uint32_t w[D / 8];                   // packed pairs; (16-byte chunk c of row r is at c ^ (r % 8))
                    const uint8_t* row = X + (part * (D / 4) / 64) * (BT * 128) + r * 128;
#pragma unroll
                    for (int v = 0; v < D / 32; ++v) {
                        const uint4 x = *reinterpret_cast<const uint4*>(row + ((((part * (D / 4) % 64) / 8 + v) ^ (r & 7)) << 4));
                        w[4 * v] = x.x; w[4 * v + 1] = x.y; w[4 * v + 2] = x.z; w[4 * v + 3] = x.w;
                    }
                    if constexpr (D == 64) tmem_st_x8(tl + col + part * 8, w); else tmem_st_x16(tl + col + part * 16, w);
                };
                to_tmem(X1s, LY::X1_COL);
                if (LY::X2_TMEM) to_tmem(X2s, LY::X2_COL);
                tc_wait_st();
                tc_fence_before();
                fence_proxy_async_smem();                // (read before the next item's copies)
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars[LY::BAR_X_TMEM]);
                lse2_r = l == -INFINITY ? INFINITY : l * LOG2E;
#pragma unroll
                for (int i = 0; i < PASSES; ++i) {
                    const uint32_t a[4] = {da[i].x, da[i].y, da[i].z, da[i].w}, b[4] = {db[i].x, db[i].y, db[i].z, db[i].w};
                    float sum = 0.f;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        sum = fmaf(__uint_as_float(a[e] << 16), __uint_as_float(b[e] << 16), sum);
                        sum = fmaf(__uint_as_float(a[e] & 0xffff0000u), __uint_as_float(b[e] & 0xffff0000u), sum);
                    }
#pragma unroll
                    for (int m = LPR / 2; m >= 1; m >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, m);
                    const int row = warp * 8 + i * ROWS + lane / LPR;
                    if (lane % LPR == 0) {
                        dls[(n & 1) * BT + row] = sum;
                        if (x0 + row < Nq) delta[static_cast<int64_t>(bh) * Nq + x0 + row] = sum;
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars[LY::BAR_DELTA]);
            }
            return true;
        };
        // Every warp needs what other warps computed.  One that gives up leaves the loop, so they meet at an mbarrier, in a wait
        // that gives up too: at a named barrier the rest would stand for good.
        auto finish_delta = [&](int n) {
            if constexpr (!LY::DKV) {
                if (!wait_warp(LY::BAR_DELTA, n & 1, 0x543)) return false;
                delta_r = dls[(n & 1) * BT + r];
            }
            return true;
        };
        const int cq = part * 32;                        // this warp's 32 columns of every step
        const int cgroup = LY::PARTS == 2 ? part >> 1 : 0;
        const uint32_t ds_addr = tl + LY::ds_store(0) + part * (LY::ds_store(1) - LY::ds_store(0));
        const uint32_t p_addr = tl + LY::p_store(0) + part * (LY::p_store(1) - LY::p_store(0));
        int n = 0, gs = 0, ne = 0, item = blockIdx.x;
        decode(item);
        ok = begin_item(0) && finish_delta(0);
        while (ok) {
            const int xr = x0 + r;                       // the row's index (query in MODE_DQ, key in MODE_DKV)
            // keys the row takes part with (MODE_DQ: per query row; MODE_DKV: the row IS a key)
            const long long rlim = static_cast<long long>(xr) + 1 + coff;
            const int nrow = rlim < nkeys ? (rlim < 0 ? 0 : static_cast<int>(rlim)) : nkeys;
            const bool key_live = xr < nkeys;
            const uint64_t c22 = pack2(c2, c2), nl2 = pack2(-lse2_r, -lse2_r), dl2 = pack2(delta_r, delta_r);
            for (int j = 0; j < nsteps && ok; ++j) {
                ok = wait_warp(LY::BAR_T_FULL + cgroup, (gs + j) & 1, 0x540 + cgroup);
                if (!ok) break;
                tc_fence_after();
                uint32_t t1[32], t2[32];
                tmem_ld_x32(tl + LY::T1_COL + cq, t1);
                tmem_ld_x32(tl + LY::T2_COL + cq, t2);
                const int y0 = (y_begin + j) * BT + cq;  // index of the first of the columns (key or query)
                // all 32 x 32 (row, column) pairs of this warp visible?  (then no per-element selection)
                const bool fast = __all_sync(0xffffffffu, MODE == MODE_DQ ? y0 + 32 <= nrow
                                                                          : key_live && static_cast<long long>(y0) + coff >= xr);
                // (own columns for the bf16 tiles: the MMAs that read the previous step's must be done before they are
                // overwritten.  They mostly are by now; the check here costs nothing, its result is wanted after the exponentials)
                bool acc_done = true;
                if (LY::SEP && j > 0) acc_done = mbar_test_wait_s(bars_s + 8 * LY::BAR_ACC_STEP, (gs + j - 1) & 1);
                tc_wait_ld();
                if (LY::SEP) {                           // T1, T2 may be overwritten by the next step's
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_s(bars_s + 8 * LY::BAR_T_FREE);
                }
                uint32_t pk[16], dk[16];
                // MODE_DQ:  p = 2^(c T1 - lse2), ds = p (T2 - delta);  MODE_DKV: p = 2^(c T1), ds = p T2 (lse and delta are in T1
                // and T2).  On packed pairs: two results per issue slot.
                if (fast) {
#pragma unroll
                    for (int i = 0; i < 32; i += 2) {
                        const uint64_t s2 = pack2(__uint_as_float(t1[i]), __uint_as_float(t1[i + 1]));
                        float a0, a1;
                        unpack2(LY::DKV ? mul2(s2, c22) : fma2(s2, c22, nl2), a0, a1);
                        t1[i] = __float_as_uint(ex2_approx(a0)); t1[i + 1] = __float_as_uint(ex2_approx(a1));
                    }
#pragma unroll
                    for (int i = 0; i < 32; i += 2) {
                        const uint64_t g2 = pack2(__uint_as_float(t2[i]), __uint_as_float(t2[i + 1]));
                        const float p0 = __uint_as_float(t1[i]), p1 = __uint_as_float(t1[i + 1]);
                        float d0, d1;
                        unpack2(mul2(pack2(p0, p1), LY::DKV ? g2 : sub2(g2, dl2)), d0, d1);
                        if (LY::DKV) pk[i / 2] = pack_bf16x2(p0, p1);
                        dk[i / 2] = pack_bf16x2(d0, d1);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 32; i += 2) {
                        float p[2], ds[2];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int col = y0 + i + e;
                            const bool live = MODE == MODE_DQ ? col < nrow : key_live && static_cast<long long>(col) + coff >= xr;
                            p[e] = live ? ex2_approx(fmaf(__uint_as_float(t1[i + e]), c2, LY::DKV ? 0.f : -lse2_r)) : 0.f;
                            ds[e] = p[e] * (__uint_as_float(t2[i + e]) - (LY::DKV ? 0.f : delta_r));
                        }
                        if (LY::DKV) pk[i / 2] = pack_bf16x2(p[0], p[1]);
                        dk[i / 2] = pack_bf16x2(ds[0], ds[1]);
                    }
                }
                if (LY::SEP) {
                    if (!__all_sync(0xffffffffu, acc_done)) {
                        ok = wait_warp(LY::BAR_ACC_STEP, static_cast<uint32_t>(gs + j - 1) & 1u, 0x542);
                        if (!ok) break;
                    }
                    tc_fence_after();
                }
                if (LY::DKV) tmem_st_x16(p_addr, pk);
                tmem_st_x16(ds_addr, dk);
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_s(bars_s + 8 * (LY::BAR_PD_FULL + cgroup));
            }
            if (!ok) break;
            // The next item's operands first (its T MMAs then run under what follows), then this one's gradients.
            const int bh_out = bh, xr_out = xr, steps_out = nsteps;
            item = take_item(n + 1);
            if (item == -2) break;
            gs += nsteps;
            if (item >= 0) {
                decode(item);
                ok = begin_item(n + 1);
                if (!ok) break;
            }
            if (steps_out > 0) {
                ok = wait_warp(LY::BAR_ACC_DONE, ne & 1, 0x550);
                if (!ok) break;
                tc_fence_after();
                ++ne;
            }
            // this thread's quarter of the features of its row: acc_a -> outA (dQ, or dK), acc_b -> outB (dV)
            constexpr int NO = MODE == MODE_DKV ? 2 : 1, NC = D / 64;
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                const float f = o == 0 ? scale : 1.f;
                const uint32_t col = (o == 0 ? LY::ACC_A_COL : LY::ACC_B_COL) + part * (D / 4);
                __nv_bfloat16* orow = (o == 0 ? outA : outB) + (static_cast<int64_t>(bh_out) * NX + xr_out) * D + part * (D / 4);
                uint32_t a[NC][16];
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    if (steps_out > 0) {
                        tmem_ld_x16(tl + col + c * 16, a[c]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; ++i) a[c][i] = 0u;   // nothing sees this tile: zero gradient
                    }
                }
                tc_wait_ld();
                if (o == NO - 1 && steps_out > 0) {      // the accumulators may be overwritten by the next item's
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_s(bars_s + 8 * LY::BAR_ACC_FREE);
                }
                if (xr_out < NX) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        uint32_t w[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            w[i] = pack_bf16x2(__uint_as_float(a[c][2 * i]) * f, __uint_as_float(a[c][2 * i + 1]) * f);
                        if (wide) {
                            st_global_32B(orow + c * 16, w);
                        } else {
                            *reinterpret_cast<uint4*>(orow + c * 16) = make_uint4(w[0], w[1], w[2], w[3]);
                            *reinterpret_cast<uint4*>(orow + c * 16 + 8) = make_uint4(w[4], w[5], w[6], w[7]);
                        }
                    }
                }
            }
            if (item < 0) break;
            ok = finish_delta(++n);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, LY::TMEM_COLS);
}

template <int D, int MODE, bool MULTI>
int launch_bwd_form(const BwdProblem& p, const CUtensorMap (&m)[4], cudaStream_t st) {
    using LY = BL<D, MODE>;
    if (!ensure_dynamic_smem<bwd_tc_kernel<D, MODE, MULTI>>(LY::SMEM_BYTES)) return FLAT_ERR_CUDA;
    const int BH = p.B * p.H, tiles = ((MODE == MODE_DQ ? p.Nq : p.Nk) + BT - 1) / BT;
    if (static_cast<int64_t>(tiles) * BH > 0x7fffffff) return FLAT_ERR_SHAPE;
    // Without the causal mask the tiles of a head run side by side and share its streamed tensors in L2.  With it, the
    // tiles of as many heads as fit L2 together (48 MB of streamed tensors) are dealt longest first: what is left at the
    // end are the short ones.
    const int64_t streamed = static_cast<int64_t>(MODE == MODE_DQ ? p.Nk : p.Nq) * D * 4;
    const int64_t fit = (48ll << 20) / streamed;
    const int group = !p.causal || fit < 1 ? 1 : fit < BH ? static_cast<int>(fit) : BH;
    const Places pl{Divisor(group * tiles), Divisor(group), Divisor(BH % group ? BH % group : group), Divisor(p.H)};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(tiles) * BH);
    cfg.blockDim = dim3(BWD_THREADS);
    cfg.dynamicSmemBytes = LY::SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto bf = [](const void* x) { return static_cast<const __nv_bfloat16*>(x); };
    const cudaError_t e = cudaLaunchKernelEx(
        &cfg, bwd_tc_kernel<D, MODE, MULTI>, m[0], m[1], m[2], m[3], bf(MODE == MODE_DQ ? p.Q : p.K), bf(MODE == MODE_DQ ? p.dO : p.V), bf(p.O),
        p.lse, p.delta,
        static_cast<__nv_bfloat16*>(MODE == MODE_DQ ? p.dQ : p.dK), static_cast<__nv_bfloat16*>(MODE == MODE_DQ ? nullptr : p.dV), BH,
        p.Nq, p.Nk, p.scale, p.k_valid_len, p.causal ? p.Nk - p.Nq : (1 << 30), pl, p.status);
    return e == cudaSuccess ? FLAT_OK : FLAT_ERR_CUDA;
}

// With no more tiles than SMs there is nothing to take over: a form without it has 30 KB of instructions less to fetch, and shorter steps
// (us, the other form / this one: B8 H8 128^2 d 64 11.2 / 9.8, B2 H8 256^2 d 128 16.1 / 15.0, B1 H2 8192^2 117.2 / 115.1 and
// 187.2 / 183.3; forward and backward B1 H12 512^2 d 64 26.6 / 22.9, B4 H6 629^2 d 128 45.2 / 41.0).
template <int D, int MODE>
int launch_bwd_mode(const BwdProblem& p, const CUtensorMap (&m)[4], cudaStream_t st) {
    const int64_t tiles = ((MODE == MODE_DQ ? p.Nq : p.Nk) + BT - 1) / BT * static_cast<int64_t>(p.B) * p.H;
    return tiles > device_sm_count() ? launch_bwd_form<D, MODE, true>(p, m, st) : launch_bwd_form<D, MODE, false>(p, m, st);
}

template <int D>
int launch_bwd_d(const BwdProblem& p, cudaStream_t st) {
    // stationary tiles are boxes of 128 rows; streamed ones too, or boxes of 64 rows (the dK dV launch at d = 128)
    constexpr int YR = BL<D, MODE_DKV>::Y_ROWS;
    CUtensorMap tmQ, tmK, tmV, tmdO, tmQs, tmdOs;
    const int BH = p.B * p.H;
    if (!make_map(&tmQ, p.Q, BH, p.Nq, D, BT) || !make_map(&tmdO, p.dO, BH, p.Nq, D, BT) || !make_map(&tmK, p.K, BH, p.Nk, D, BT) ||
        !make_map(&tmV, p.V, BH, p.Nk, D, BT) || !make_map(&tmQs, p.Q, BH, p.Nq, D, YR) || !make_map(&tmdOs, p.dO, BH, p.Nq, D, YR))
        return FLAT_ERR_CUDA;
    const int rc = launch_bwd_mode<D, MODE_DQ>(p, {tmQ, tmdO, tmK, tmV}, st);
    return rc != FLAT_OK ? rc : launch_bwd_mode<D, MODE_DKV>(p, {tmK, tmV, tmQs, tmdOs}, st);
}

}  // namespace

int launch_bwd_tc(const BwdProblem& p, cudaStream_t st) {
    if (p.d == 64) return launch_bwd_d<64>(p, st);
    if (p.d == 128) return launch_bwd_d<128>(p, st);
    return FLAT_ERR_UNSUPPORTED;
}

}  // namespace flat
