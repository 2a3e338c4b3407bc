// The activation-weight operators of an attention layer (Section 2, "Computation operators",
// steps 1 and 5): the Query / Key / Value projections of the input [B,N,D] into [B,H,N,d] and the
// Output projection of the concatenated heads back to [B,N,D].  Both are Y = A W^T with bf16
// operands, fp32 accumulation in TMEM and bf16 results, as one persistent tcgen05 kernel:
//   * the Q/K/V projection is ONE contraction against the stacked weights [3 H d, D]; its epilogue
//     writes each output tile straight into the head-major tensors Q, K, V [B,H,N,d] that the
//     fused attention kernel reads (no transposition pass);
//   * the Output projection reads its A operand straight from the head-major attention output
//     O [B,H,N,d]: a 64-wide slice of the contraction index h * d + c is a (head, column) box of
//     that tensor for TMA.
// CTA = 320 threads: warps 0-7 epilogue (TMEM -> bf16 -> global), warp 8 TMA producer (one lane),
// warp 9 MMA issuer (one elected lane).  The contraction runs in slices of 64 through a ring of TMA stages.  Tiles
// (launch_gemm's rule): 256 x 256 outputs as two row blocks of 128 that share every W slice (each W byte fetched feeds
// twice the MMAs), whose two accumulators fill TMEM, so that a tile's epilogue is not overlapped with the next tile's
// MMAs; 256 x 128, 128 x 128 and 128 x 64 outputs with two accumulators in turn, for problems that leave SMs empty
// with the wide tile; and 128 x 64 with the contraction split over a cluster of two or four CTAs, which leave their
// fp32 partial sums in the shared memory of the CTA that finishes the row (plain remote stores; summed in a fixed
// order), for the smallest.  A CTA walks tiles blockIdx.x, blockIdx.x + gridDim.x, ...; tiles that share their rows of
// A are neighbours, so CTAs running together share A in L2 (the weights fit L2 whole).  Launched with programmatic
// stream serialization: barriers and TMEM are set up while the previous kernel of the stream drains.
// What bounds it: large problems the tensor pipe; small ones the chain launch -> first slice -> slices -> store (about
// 3 us before the first slice's MMAs and after the last, see launch_gemm).  Every wait is bounded (tc_common.cuh).
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

constexpr int GK = 64;               // contraction slice (one 128-byte swizzle atom of bf16)
constexpr int GNM = 256;             // Nout is a multiple of this (the widest tile)
constexpr int GTHREADS = 320;        // 8 epilogue warps, TMA producer, MMA issuer

// RB: MMA row blocks of 128 per tile; TN: output columns per tile; CS: CTAs of the cluster that share a tile's contraction.
template <int RB, int TN, int CS> struct GL {
    static constexpr int GM = RB * 128;
    static constexpr int A_BYTES = GM * GK * 2;
    static constexpr int B_BYTES = TN * GK * 2;
    static constexpr int STAGES = RB == 2 ? 3 : TN == 128 ? 6 : CS > 1 ? 7 : 8;
    static constexpr int TILE_BYTES = STAGES * (A_BYTES + B_BYTES);
    // (CS > 1) partial sums of the other CTAs for the 128 / CS rows this CTA finishes: [sender][4-column vector][row]
    static constexpr int RECV_BYTES = (CS - 1) * (128 / CS) * TN * 4;
    static constexpr int SMEM_BYTES = TILE_BYTES + RECV_BYTES + 256 + 1024;
    static constexpr int NACC = RB * TN * 2 <= 512 ? 2 : 1;   // accumulators in turn: a tile's epilogue runs under the next tile's MMAs
    static constexpr uint32_t TMEM_COLS = RB * TN * NACC < 256 ? 128 : RB * TN * NACC < 512 ? 256 : 512;
    static constexpr int EC = RB == 2 ? TN : TN / 2;     // columns per epilogue thread (RB = 1: two warps share a row)
    static constexpr int FULL = 0, EMPTY = STAGES, ACC_FULL = 2 * STAGES, ACC_EMPTY = ACC_FULL + NACC, MERGE = ACC_EMPTY + NACC;
    static constexpr int NUM_BARS = MERGE + 1;
    static_assert(SMEM_BYTES <= 232448 && TMEM_COLS >= RB * TN * NACC, "layout");
};

struct GemmArgs {
    int M, Nout, Kdim;               // Y [M, Nout] = A [M, Kdim] W[Nout, Kdim]^T
    int N, H, d;                     // tokens per sequence, heads, head size (head-major sides)
    __nv_bfloat16* out0;             // token-major Y, or head-major Q
    __nv_bfloat16* out1;             // head-major K
    __nv_bfloat16* out2;             // head-major V
    int wide_stores;                 // every output pointer is 32-byte aligned: 32-byte stores
};

// A_HEADS: A is the head-major tensor [B,H,N,d] (Output projection); else token-major [M, Kdim].
// OUT_HEADS: the result goes to the head-major tensors out0..2 (Q/K/V projection); else to the
// token-major Y = out0.
template <bool A_HEADS, bool OUT_HEADS, int RB, int TN, int CS>
__global__ void __launch_bounds__(GTHREADS, 1)
proj_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW, const GemmArgs g,
                 int32_t* status) {
    using LY = GL<RB, TN, CS>;
    constexpr int STAGES = LY::STAGES, GM = LY::GM, EC = LY::EC;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* As = base;
    uint8_t* Bs = base + STAGES * LY::A_BYTES;
    float4* recv = reinterpret_cast<float4*>(base + LY::TILE_BYTES);
    uint64_t* bars = reinterpret_cast<uint64_t*>(base + LY::TILE_BYTES + LY::RECV_BYTES);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + LY::NUM_BARS);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    // Roles by an index that the compiler knows to be the same in all lanes, the epilogue by one that it does not (all known: forms of
    // four CTAs spill, M 128 K 768 -> 768 4.86 -> 5.12 us; so: 4.81).  The two forms to head-major tensors that spill even then
    // (clusters of four; 256 x 256) know it nowhere: M 128 -> 768 5.43 -> 5.12, M 8192 -> 3072 41.2 -> 40.6.
    const int warp = threadIdx.x >> 5, role = OUT_HEADS && (CS == 4 || TN == 256) ? warp : warp_index(), lane = threadIdx.x & 31;

    if (threadIdx.x == 8 * 32) {
        // (eight epilogue warps free an accumulator; the 8 / CS warps of every other CTA that hold rows of this one send)
        for (int i = 0; i < LY::NUM_BARS; ++i)
            mbar_init(&bars[i], i == LY::MERGE ? (CS > 1 ? (CS - 1) * 8 / CS : 1) : i >= LY::ACC_EMPTY ? 8 : 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0) { tmem_alloc(tmem_slot, LY::TMEM_COLS); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // (launched with programmatic stream serialization: the next kernel's set-up may start now, and nothing in device
    // memory is touched before the previous kernel of the stream has finished)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    const int crank = CS > 1 ? static_cast<int>(cluster_ctarank()) : 0;
    if (CS > 1) cluster_sync_all();                      // every CTA of the cluster has its barriers before anyone's first remote access

    const int tiles_n = g.Nout / TN, tiles_m = (g.M + GM - 1) / GM;
    const int tiles = tiles_m * tiles_n;
    // (CS > 1: one tile per cluster, this CTA's share of the contraction slices; every share has at least one)
    const int all_steps = g.Kdim / GK;
    const int k_first = CS > 1 ? all_steps * crank / CS : 0;
    const int ksteps = CS > 1 ? all_steps * (crank + 1) / CS - k_first : all_steps;
    const int tile_first = blockIdx.x / CS, tile_step = gridDim.x / CS;

    if (role == 8) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            prefetch_tensormap(&tmA); prefetch_tensormap(&tmW);
            bool ok = true;
            int issued = 0, it = 0;                      // it: ring slot counter over all tiles
            for (int tile = tile_first; tile < tiles && ok; tile += tile_step) {
                const int m0 = (tile / tiles_n) * GM, n0 = (tile % tiles_n) * TN;
                for (int kc = k_first; kc < k_first + ksteps && ok; ++kc, ++it) {
                    const int s = it % STAGES;
                    ok = bounded_wait(&bars[LY::EMPTY + s], ((it / STAGES) & 1) ^ 1, abort_flag, status, 0x500);
                    if (!ok) break;
                    mbar_arrive_expect_tx(&bars[LY::FULL + s], LY::A_BYTES + LY::B_BYTES);
                    if (A_HEADS) {
                        // each block of 128 rows holds tokens of ONE sequence (N is a multiple of 128); slice
                        // kc of the contraction index h * d + c lies in one head.  (A block past the last
                        // sequence has an out-of-range coordinate and reads zeros.)
                        const int k0 = kc * GK, h = k0 / g.d, c0 = k0 - h * g.d;
#pragma unroll
                        for (int r = 0; r < RB; ++r) {
                            const int mr = m0 + r * 128, b = mr / g.N, tok0 = mr - b * g.N;
                            tma_load_3d(As + s * LY::A_BYTES + r * 128 * GK * 2, &tmA, &bars[LY::FULL + s], c0, tok0,
                                        b * g.H + h);
                        }
                    } else {
#pragma unroll
                        for (int r = 0; r < RB; ++r)
                            tma_load_3d(As + s * LY::A_BYTES + r * 128 * GK * 2, &tmA, &bars[LY::FULL + s], kc * GK,
                                        m0 + r * 128, 0);
                    }
                    tma_load_3d(Bs + s * LY::B_BYTES, &tmW, &bars[LY::FULL + s], kc * GK, n0, 0);
                    issued = it + 1;
                }
            }
            if (!ok)
                for (int j = issued > STAGES ? issued - STAGES : 0; j < issued; ++j)
                    drain_wait(&bars[LY::FULL + j % STAGES], (j / STAGES) & 1);
        }
    } else if (role == 9) {
        // ------------------------------------------------------------ MMA issuer
        constexpr uint32_t IDESC = make_idesc_bf16(128, TN, 0, 0);
        const uint64_t ad = make_smem_desc_sw128(smem_u32(As), 16, 1024);
        const uint64_t bd = make_smem_desc_sw128(smem_u32(Bs), 16, 1024);
        bool ok = true;
        int it = 0, tcount = 0;
        for (int tile = tile_first; tile < tiles && ok; tile += tile_step, ++tcount) {
            const int a_slot = tcount % LY::NACC;
            // the epilogue must have read this accumulator's previous tile
            ok = __all_sync(0xffffffffu, bounded_wait(&bars[LY::ACC_EMPTY + a_slot], ((tcount / LY::NACC) & 1) ^ 1, abort_flag,
                                                      status, 0x510));
            if (!ok) break;
            tc_fence_after();
            for (int kc = 0; kc < ksteps && ok; ++kc, ++it) {
                const int s = it % STAGES;
                ok = __all_sync(0xffffffffu,
                                bounded_wait(&bars[LY::FULL + s], (it / STAGES) & 1, abort_flag, status, 0x520));
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t a = ad + static_cast<uint64_t>((s * LY::A_BYTES) >> 4);
                    const uint64_t b = bd + static_cast<uint64_t>((s * LY::B_BYTES) >> 4);
#pragma unroll
                    for (int k = 0; k < GK / 16; ++k)
#pragma unroll
                        for (int r = 0; r < RB; ++r)
                            mma_ss(tmem + (a_slot * RB + r) * TN, a + static_cast<uint64_t>((r * 128 * GK * 2 + k * 32) >> 4),
                                   b + static_cast<uint64_t>((k * 32) >> 4), IDESC, (kc > 0 || k > 0));
                    tc_commit(&bars[LY::EMPTY + s]);
                    if (kc == ksteps - 1) tc_commit(&bars[LY::ACC_FULL + a_slot]);
                }
                __syncwarp();
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue (warps 0-7)
        // warp w reads TMEM lanes 32 (w % 4) .. of row block w / 4, or (RB = 1) of column half w / 4
        bool ok = true;
        int tcount = 0;
        const int rb = RB == 2 ? warp >> 2 : 0, c0 = RB == 2 ? 0 : (warp >> 2) * EC;
        const int lrow = (warp & 3) * 32 + lane;         // row inside the block of 128
        const uint32_t tl = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + rb * TN + c0;
        const int HD = g.H * g.d;
        for (int tile = tile_first; tile < tiles; tile += tile_step, ++tcount) {
            const int a_slot = tcount % LY::NACC;
            const int m0 = (tile / tiles_n) * GM, n0 = (tile % tiles_n) * TN + c0;
            const int m = m0 + rb * 128 + lrow;
            ok = __all_sync(0xffffffffu, bounded_wait(&bars[LY::ACC_FULL + a_slot], (tcount / LY::NACC) & 1, abort_flag, status, 0x530));
            if (!ok && CS == 1) break;
            tc_fence_after();
            int64_t row_off = 0;                         // element offset of this thread's row in its destination
            int b = 0, tok = 0;
            if (OUT_HEADS) { b = m / g.N; tok = m - b * g.N; }
            else row_off = static_cast<int64_t>(m) * g.Nout + n0;
            // First the whole accumulator row goes to registers as packed bf16, so that the
            // accumulator is released for the next tile's MMAs before any store is issued.
            uint32_t w[EC / 2];
            bool writer = m < g.M;
            if constexpr (CS == 1) {
#pragma unroll
                for (int c = 0; c < EC / 32; ++c) {
                    uint32_t r[32];
                    tmem_ld_x32(tl + a_slot * RB * TN + c * 32, r);
                    tc_wait_ld();
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        w[c * 16 + i] = pack_bf16x2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars[LY::ACC_EMPTY + a_slot]);
            } else {
                // Partial sums: rank r finishes rows [128 r / CS, 128 (r + 1) / CS); the others store theirs into r's
                // shared memory (lanes of a warp on contiguous 16-byte vectors) and arrive on its barrier, once a warp.
                constexpr int RP = 128 / CS;             // rows per rank: whole warps
                float acc[EC];
#pragma unroll
                for (int c = 0; c < EC / 32; ++c) {
                    uint32_t r[32];
                    tmem_ld_x32(tl + c * 32, r);
                    tc_wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; ++i) acc[c * 32 + i] = ok ? __uint_as_float(r[i]) : __int_as_float(0x7fc00000);
                }
                const int owner = lrow / RP;
                if (owner != crank) {
                    const int slot = (crank - owner - 1 + CS) % CS;
                    const uint32_t dst = mapa_shared(smem_u32(recv + (slot * (TN / 4) + c0 / 4) * RP + lrow % RP), owner);
#pragma unroll
                    for (int v = 0; v < EC / 4; ++v)
                        st_cluster_v4(dst + 16 * RP * v, acc[4 * v], acc[4 * v + 1], acc[4 * v + 2], acc[4 * v + 3]);
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(mapa_shared(smem_u32(&bars[LY::MERGE]), owner));
                    writer = false;
                } else {
                    // (a sender stores and arrives whatever happened to it, at the latest when its own wait has run
                    // out, so the owner waits longer than any sender can take before it leaves)
                    const long long t0 = clock64();
                    while (!mbar_try_wait_cluster(&bars[LY::MERGE], 0)) {
                        if (clock64() - t0 > 4 * WAIT_CYCLES) {
                            writer = false;
                            if (status) atomicExch(status, 0x540);
                            break;
                        }
                    }
                    // summed in the order of the ranks, whoever finishes the row: the same bits every time
                    float sum[EC];
#pragma unroll
                    for (int r = 0; r < CS; ++r) {
                        const int slot = (r - crank - 1 + CS) % CS;
#pragma unroll
                        for (int v = 0; v < EC / 4; ++v) {
                            float4 x = make_float4(acc[4 * v], acc[4 * v + 1], acc[4 * v + 2], acc[4 * v + 3]);
                            if (r != crank) x = recv[(slot * (TN / 4) + c0 / 4 + v) * RP + lrow % RP];
                            if (r == 0) { sum[4 * v] = x.x; sum[4 * v + 1] = x.y; sum[4 * v + 2] = x.z; sum[4 * v + 3] = x.w; }
                            else { sum[4 * v] += x.x; sum[4 * v + 1] += x.y; sum[4 * v + 2] += x.z; sum[4 * v + 3] += x.w; }
                        }
                    }
#pragma unroll
                    for (int i = 0; i < EC / 2; ++i) w[i] = pack_bf16x2(sum[2 * i], sum[2 * i + 1]);
                }
            }
            if (writer) {
#pragma unroll
                for (int c = 0; c < EC / 32; ++c) {
                    __nv_bfloat16* dst;
                    if (OUT_HEADS) {
                        // 32 consecutive output columns lie in one head of one of Q, K, V (32 divides d)
                        const int n = n0 + c * 32, which = n / HD, rem = n - which * HD, h = rem / g.d, cc = rem - h * g.d;
                        __nv_bfloat16* o = which == 0 ? g.out0 : (which == 1 ? g.out1 : g.out2);
                        dst = o + ((static_cast<int64_t>(b) * g.H + h) * g.N + tok) * g.d + cc;
                    } else {
                        dst = g.out0 + row_off + c * 32;
                    }
                    if (g.wide_stores) {
                        st_global_32B(dst, *reinterpret_cast<uint32_t(*)[8]>(&w[c * 16]));
                        st_global_32B(dst + 16, *reinterpret_cast<uint32_t(*)[8]>(&w[c * 16 + 8]));
                    } else {
#pragma unroll
                        for (int v = 0; v < 4; ++v)
                            *reinterpret_cast<uint4*>(dst + v * 8) =
                                make_uint4(w[c * 16 + 4 * v], w[c * 16 + 4 * v + 1], w[c * 16 + 4 * v + 2], w[c * 16 + 4 * v + 3]);
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, LY::TMEM_COLS);
}

// [rows, cols] bf16 row-major as a TMA tensor with boxes of 64 columns x box_rows rows.
bool make_map_2d(CUtensorMap* m, const void* ptr, int rows, int cols, int box_rows) {
    return make_map(m, ptr, 1, rows, cols, box_rows);
}

// Where the operands are: A as [M, Kdim] rows, or head-major; W as [Nout, Kdim] rows.
struct GemmOperands { const void *A, *W; };

template <bool A_HEADS, bool OUT_HEADS, int RB, int TN, int CS>
int launch_gemm_tile(const GemmOperands& op, const GemmArgs& g, int32_t* status, cudaStream_t st) {
    using LY = GL<RB, TN, CS>;
    CUtensorMap tmA, tmW;
    if (!(A_HEADS ? make_map(&tmA, op.A, g.M / g.N * g.H, g.N, g.d, 128) : make_map_2d(&tmA, op.A, g.M, g.Kdim, 128)) ||
        !make_map_2d(&tmW, op.W, g.Nout, g.Kdim, TN))
        return FLAT_ERR_CUDA;
    auto kern = proj_gemm_kernel<A_HEADS, OUT_HEADS, RB, TN, CS>;
    if (!ensure_dynamic_smem<proj_gemm_kernel<A_HEADS, OUT_HEADS, RB, TN, CS>>(LY::SMEM_BYTES)) return FLAT_ERR_CUDA;
    const int tiles = ((g.M + LY::GM - 1) / LY::GM) * (g.Nout / TN);
    const int sms = device_sm_count();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CS > 1 ? tiles * CS : tiles < sms ? tiles : sms);
    cfg.blockDim = dim3(GTHREADS);
    cfg.dynamicSmemBytes = LY::SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = CS; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = CS > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, tmA, tmW, g, status) == cudaSuccess ? FLAT_OK : FLAT_ERR_CUDA;
}

// Which tile: the one whose time estimate is the smallest,
//     start + rounds x (slices x per_slice + per_tile)       (microseconds; rounds = tiles over SMs, rounded up)
// with the constants below, fitted to graph replays of this kernel in every form on 81 sizes (M 128 ... 8192, K 256 ...
// 4096, Nout 256 ... 6144; the estimate is within 12 % of them except where the power cap rules).  What lies behind:
// a slice costs the larger of its MMAs (256 x 256: 1024 cycles) and its bytes at about 66 per cycle and SM from L2
// (128 x 64: 24 KB, 128 x 128: 32 KB, 256 x 128: 48 KB), so wide tiles win once they fill the SMs and narrow ones
// while they do not; a split contraction pays about 2 us for the exchange.  M 512, K 768 -> Nout 2304: 256 x 256
// (18 CTAs) 13.2 us, 128 x 128 6.5, 128 x 64 5.9; K 3072 -> 768, M 512: 256 x 256 32.9, 128 x 64 14.0, halves of the
// contraction on two CTAs 10.1; M 8192, K 2048 -> 6144: 256 x 256 146, 256 x 128 169, 128 x 128 191.
// Clusters of four stop at 128 CTAs: with 144 they no longer all start together (9.7 us against 5.2 on clusters of two).
template <bool A_HEADS, bool OUT_HEADS>
int launch_gemm(const GemmOperands& op, const GemmArgs& g, int32_t* status, cudaStream_t st) {
    const int sms = device_sm_count(), slices = g.Kdim / GK;
    auto tiles = [&](int m, int n) { return static_cast<int64_t>((g.M + m - 1) / m) * (g.Nout / n); };
    auto estimate = [&](int m, int n, double start, double per_slice, double per_tile) {
        return start + static_cast<double>((tiles(m, n) + sms - 1) / sms) * (slices * per_slice + per_tile);
    };
    const double t[6] = {
        estimate(256, 256, 4.0, 0.555, 2.3), estimate(256, 128, 2.9, 0.392, 1.5), estimate(128, 128, 2.35, 0.253, 1.0),
        estimate(128, 64, 2.0, 0.237, 0.67),
        tiles(128, 64) * 2 <= sms && slices >= 4 ? 3.85 + slices / 2.0 * 0.237 : 1e30,
        tiles(128, 64) * 4 <= sms - sms / 8 && slices >= 8 ? 4.4 + slices / 4.0 * 0.237 : 1e30};
    int best = 0;
    for (int i = 1; i < 6; ++i)
        if (t[i] < t[best]) best = i;
    switch (best) {
        case 1: return launch_gemm_tile<A_HEADS, OUT_HEADS, 2, 128, 1>(op, g, status, st);
        case 2: return launch_gemm_tile<A_HEADS, OUT_HEADS, 1, 128, 1>(op, g, status, st);
        case 3: return launch_gemm_tile<A_HEADS, OUT_HEADS, 1, 64, 1>(op, g, status, st);
        case 4: return launch_gemm_tile<A_HEADS, OUT_HEADS, 1, 64, 2>(op, g, status, st);
        case 5: return launch_gemm_tile<A_HEADS, OUT_HEADS, 1, 64, 4>(op, g, status, st);
    }
    return launch_gemm_tile<A_HEADS, OUT_HEADS, 2, 256, 1>(op, g, status, st);
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
bool aligned32(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 31) == 0; }

}  // namespace

int launch_qkv_proj(const void* X, const void* Wqkv, void* Q, void* K, void* V, int B, int N, int H, int d, int Dm,
                    int32_t* status, cudaStream_t st) {
    if (!X || !Wqkv || !Q || !K || !V) return FLAT_ERR_NULL;
    if (B < 1 || N < 1 || H < 1 || Dm < 1) return FLAT_ERR_SHAPE;
    if (static_cast<int64_t>(B) * N > 0x7fffffff || static_cast<int64_t>(H) * d * 3 > 0x7fffffff) return FLAT_ERR_SHAPE;
    if ((d != 64 && d != 128) || (H * d) % GNM != 0 || Dm % GK != 0) return FLAT_ERR_UNSUPPORTED;
    if (!aligned16(X) || !aligned16(Wqkv) || !aligned16(Q) || !aligned16(K) || !aligned16(V)) return FLAT_ERR_ALIGN;
    GemmArgs g{B * N, 3 * H * d, Dm, N, H, d, static_cast<__nv_bfloat16*>(Q), static_cast<__nv_bfloat16*>(K),
               static_cast<__nv_bfloat16*>(V), aligned32(Q) && aligned32(K) && aligned32(V)};
    return launch_gemm<false, true>({X, Wqkv}, g, status, st);
}

int launch_out_proj(const void* O, const void* Wo, void* Y, int B, int N, int H, int d, int Dm, int32_t* status,
                    cudaStream_t st) {
    if (!O || !Wo || !Y) return FLAT_ERR_NULL;
    if (B < 1 || N < 1 || H < 1 || Dm < 1) return FLAT_ERR_SHAPE;
    if (static_cast<int64_t>(B) * N > 0x7fffffff || static_cast<int64_t>(B) * H > 0x7fffffff) return FLAT_ERR_SHAPE;
    if ((d != 64 && d != 128) || N % 128 != 0 || Dm % GNM != 0) return FLAT_ERR_UNSUPPORTED;
    if (!aligned16(O) || !aligned16(Wo) || !aligned16(Y)) return FLAT_ERR_ALIGN;
    GemmArgs g{B * N, Dm, H * d, N, H, d, static_cast<__nv_bfloat16*>(Y), nullptr, nullptr, aligned32(Y)};
    return launch_gemm<true, false>({O, Wo}, g, status, st);
}

int launch_fc(const void* X, const void* W, void* Y, int M, int Kdim, int Nout, int32_t* status, cudaStream_t st) {
    if (!X || !W || !Y) return FLAT_ERR_NULL;
    if (M < 1 || Kdim < 1 || Nout < 1) return FLAT_ERR_SHAPE;
    if (Kdim % GK != 0 || Nout % GNM != 0) return FLAT_ERR_UNSUPPORTED;
    if (!aligned16(X) || !aligned16(W) || !aligned16(Y)) return FLAT_ERR_ALIGN;
    GemmArgs g{M, Nout, Kdim, M, 1, 64, static_cast<__nv_bfloat16*>(Y), nullptr, nullptr, aligned32(Y)};
    return launch_gemm<false, false>({X, W}, g, status, st);
}

}  // namespace flat
