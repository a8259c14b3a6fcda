// cg_tc.cu -- tensor-core (tcgen05) encode of KIVI keys, head dim d = 128: gauge rotation
// (Sec. 3, Z = G X) fused with one range per channel over the 128 tokens of a key group.
//
// Persistent warp-specialized kernel, one CTA per SM, 15 warps:
//   warp 0      TMA producer: 128-token x tiles (2 x [128 rows x 64 bf16], 128-byte
//               swizzle) into a 4-stage ring;
//   warp 1      MMA issuer: z~ = G x^T on tcgen05 (M = 128 channels, N = 128 tokens, K = 128,
//               the gauge block-diagonal), G split into three bf16 terms (hi + lo + lo2, exact
//               for normal fp32 values); fp32 accumulators in tensor memory, four buffers
//               (the MMA runs one tile ahead of the three warpgroups);
//   warp 2      gauge converter: at each gauge change builds the bf16 split operand and
//               the error coefficients of the new gauge set;
//   warps 3..14 three epilogue warpgroups; warpgroup k takes tiles i = k (mod 3); one
//               thread per channel (= TMEM lane): range, fp16 scale/zero, codes, packing,
//               stores; codes are packed into the output words as they are produced.
//
// What bounds it: the epilogue's latency and issue, not memory (1.34 ms of 3.9 for 28 x 4 x 4
// heads of 32k tokens at 3 bits, keys and values). The candidates of an undecided range and
// the values near a rounding boundary are found by spreading a channel's 32 values over the
// lanes (one compare and vote) instead of by masks in every lane, and codes are made in
// packed pairs: 4.49 -> 3.89 ms; the exact rounds at one call site each: 3.85 ms. Where a CTA
// has few tiles nothing hides the chain of that search, and the extremes are looked for by
// masks (MASKS; launch_encode_bits).
//
// Exactness. The library defines z as a fixed-order fp32 sum (pairwise summation of the
// products; include/codecgauge.h). For every output channel i the converter bounds
// |z~_i - z_i| / ||x_group||_2 by
//     e_i = (c_order + c_tc) ||G_i||_2 + ||G_i - sum of split terms||_2,
// c_order = (1 + log2 g) u the rounding bound of the fixed order, c_tc a bound on the
// tensor-core fp32 accumulation, and the exact residual of the split. The MMAs accumulate
// the split's two small terms first (partial sums below 2^-8 of ||G_i|| ||x||, 2 n_hi
// K-steps) and the leading term last (n_hi = K / 16 steps), so c_tc = (n_hi + 4 + 2 n_hi /
// 128) u, 4 u covering the rounding inside each MMA and of the result; the measured
// |z~ - Gx| stays below 2.4 u ||G_i|| ||x|| (g = 32 and 128; random, Hadamard and DCT gauges). The epilogue
// turns it into E per block. A block's fp16 scale and zero are monotone functions of its
// (max, min); when every (max, min) within E of the approximate ones gives the same fp16
// results they are taken directly, otherwise the candidate extremes are recomputed
// exactly, so scales and zeros are bit-identical to the definition.
// Codes: a code taken from z~ can differ from the definition's only if the exact
// pre-rounding value t lies within mu = E/s (+ rounding slack) of a rounding boundary.
// The accepted tolerance lets a code differ by one where t lies within 1e-4 steps of a
// boundary, so blocks with mu < 1e-4 keep the z~ codes; in blocks with a larger mu the
// codes within mu of a boundary are recomputed exactly. Recomputation uses the library's
// order (as the CUDA-core kernels do): candidates go into a per-warp list in shared memory
// and teams of lanes compute them together.
#include <cuda_bf16.h>

#include "cg_sm100.cuh"
#include "cg_tc.h"
#include "cg_tc_common.cuh"
#include "cg_tc_enc.cuh"
#include "cg_tmap.h"

namespace cg {
namespace {

using namespace sm100;
using tc::kD;
using tc::kWaitLimitNs;

constexpr int kStages = 4;
constexpr int kTileBytes = 128 * kD * 2;
constexpr int kThreads = 480;
constexpr int kEpiWarp0 = 3;
constexpr int kJobCap = 8;            // exact recomputes per warp and round
constexpr int kAcc = 4;               // accumulator buffers in tensor memory
constexpr int kNPass = 3;             // bf16 terms of the gauge split
constexpr int kSegBufs = 4;
constexpr float kMagic = 12582912.0f; // 1.5 * 2^23: adding it rounds to an integer (RNE)

struct EncSmem {
    static constexpr uint32_t stages = 0;
    static constexpr uint32_t bsplit = stages + kStages * kTileBytes;  // 3 x (16 or 32 KB)
    static constexpr uint32_t queue = bsplit + kNPass * 32768;         // 12 warps x (32 values, kJobCap jobs)
    static constexpr uint32_t xch = queue + 12 * (32 + kJobCap) * 4;  // keys: 3 warpgroups x 2 x 4 warps x 4 floats
    static constexpr uint32_t misc = xch + 3 * 2 * 4 * 4 * 4;
    static constexpr uint32_t total = misc + 384;  // base is 1024-aligned (checked in-kernel)
};

struct Misc {
    uint64_t full[kStages], empty[kStages];
    uint64_t accfull[kAcc], accempty[kAcc];
    uint64_t gready[kSegBufs];
    uint64_t bfree;
    uint32_t tmem_slot;
    int abort_flag;
    float emaxb[kSegBufs][4];  // per gauge set and quantization block: max_i e_i
    float gmaxb[kSegBufs][4];  // and max_i ||G_i|| (the converter's, not read here)
    uint64_t xbar[3][2];       // keys: per warpgroup, exchange of the group-norm maxima
};

static_assert(sizeof(Misc) <= 384, "Misc outgrew its shared-memory slot");
static_assert(EncSmem::total <= 232448, "encode kernel exceeds 227 KB of shared memory");

struct EncParams {
    RowArgs a;
    tc::Sched S;
};

__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__device__ __forceinline__ float min3f(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float max3f(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

template <typename T>
__device__ __forceinline__ T pick4(const T (&v)[4], int i) {
    return i == 0 ? v[0] : i == 1 ? v[1] : i == 2 ? v[2] : v[3];
}
template <typename T>
__device__ __forceinline__ void set4(T (&v)[4], int i, T x) {
    v[0] = i == 0 ? x : v[0];
    v[1] = i == 1 ? x : v[1];
    v[2] = i == 2 ? x : v[2];
    v[3] = i == 3 ? x : v[3];
}

// The constant part of a packed word built from y = 0x4B400000 + q: the wrapping sum of
// 0x4B400000 << s over the codes of a 32-code chunk that start in word w.
template <int BITS>
__host__ __device__ constexpr uint32_t pack_bias(int w) {
    uint32_t k = 0;
    for (int c = 0; c < 32; c++)
        if ((c * BITS) >> 5 == w) k += 0x4B400000u << ((c * BITS) & 31);
    return k;
}

__device__ __forceinline__ uint32_t scale16(float mx, float mn, float qmax) {
    return f2h_bits(__fdiv_rn(__fsub_rn(mx, mn), qmax));
}

// Overwrite the BITS-bit code at bit position `bit` of a packed row in global memory
// (the row was stored by this thread; the rare exact recomputes are patched in place).
template <int BITS>
__device__ __forceinline__ void patch_code(uint8_t* rowp, int bit, uint32_t q) {
    unsigned int* wp = reinterpret_cast<unsigned int*>(rowp) + (bit >> 5);
    const int off = bit & 31;
    const uint32_t msk = (1u << BITS) - 1u;
    atomicAnd(wp, ~(msk << off));
    atomicOr(wp, q << off);
    if (off + BITS > 32) {
        const int sh = 32 - off;
        atomicAnd(wp + 1, ~(msk >> sh));
        atomicOr(wp + 1, q >> sh);
    }
}

// The MMA's operands are swapped against the row kernel's, D[channel][token] = G x^T, so a
// thread owns one channel's 128 tokens, which form its block and its packed code stream.
template <int BITS, bool KEYS, int NBK, bool MASKS>
__global__ void __launch_bounds__(kThreads, 1) tc_encode_kernel(const __grid_constant__ CUtensorMap xmap,
                                                                 const EncParams P) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    if (smem_u32(smem_raw) & 1023u) {
        // the swizzled tiles need a 1024-byte aligned base; the layout leaves no slack
        if (threadIdx.x == 0) raise_flag(P.a.status, CG_FLAG_PIPE_TIMEOUT);
        return;
    }
    unsigned char* sm = smem_raw;
    Misc* M = reinterpret_cast<Misc*>(sm + EncSmem::misc);
    unsigned char* stages = sm + EncSmem::stages;
    unsigned char* bsplit = sm + EncSmem::bsplit;
    uint32_t* queue = reinterpret_cast<uint32_t*>(sm + EncSmem::queue);
    float* xch = reinterpret_cast<float*>(sm + EncSmem::xch);

    const RowArgs& a = P.a;
    const tc::Sched& S = P.S;
    const int g = a.g, npass = kNPass;
    constexpr int blk = kD / NBK;  // quantization block: NBK blocks per row
    constexpr int nbk = NBK;
    // 6 and 8 bits: values near a rounding boundary are common (their distance mu grows with the range
    // over the scale), so every lane keeps a mask of its own and the list holds 20 of them; 2 to 4 bits:
    // rare, so a lane keeps only its largest distance and the chunk is looked through again. 3 bits, 28 x
    // 4 x 4 heads of 32k tokens: 4463 us with masks, 3888 without; 8 bits, 2 x 8 heads of 4k: 68 and 73.
    constexpr bool kMasks = BITS >= 6;
    constexpr int kJobSlots = kMasks ? 4 : 2;  // values per lane and memory round trip in the exact recompute
    // gauge operand layout: full K = 128 (block-diagonal for g < 128) for keys and g = 128,
    // else one g-wide K block per group in a 64-column tile
    const bool fullk = KEYS || g == 128;
    const uint32_t bsz = fullk ? 32768u : 16384u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    const int64_t t_begin = S.n_tiles * blockIdx.x / gridDim.x;
    const int64_t t_end = S.n_tiles * (blockIdx.x + 1) / gridDim.x;
    const int my_tiles = (int)(t_end - t_begin);
    const int64_t seg0 = my_tiles > 0 ? tc::tile_info(a, S, t_begin).seg : 0;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; i++) {
            mbar_init(&M->full[i], 1);
            mbar_init(&M->empty[i], 4);
        }
        for (int i = 0; i < kAcc; i++) {
            mbar_init(&M->accfull[i], 1);
            mbar_init(&M->accempty[i], 4);
        }
        for (int i = 0; i < kSegBufs; i++) mbar_init(&M->gready[i], 1);
        for (int w = 0; w < 3; w++) {
            mbar_init(&M->xbar[w][0], 4);
            mbar_init(&M->xbar[w][1], 4);
        }
        mbar_init(&M->bfree, 1);
        M->abort_flag = 0;
        fence_barrier_init();
    }
    for (uint32_t i = threadIdx.x; i < (uint32_t)npass * bsz / 16; i += kThreads)
        reinterpret_cast<uint4*>(bsplit)[i] = make_uint4(0, 0, 0, 0);
    if (warp == 1) {
        tmem_alloc(&M->tmem_slot, kAcc * 128);
        tmem_relinquish();
        tc_fence_before();
    }
    fence_proxy_async_smem();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = M->tmem_slot;
    volatile int* abort_flag = &M->abort_flag;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0 && my_tiles > 0) {
            prefetch_tmap(&xmap);
            int issued = 0;
            tc::TileIter it;
            it.init(a, S, t_begin);
            for (int i = 0; i < my_tiles; i++, it.step(a, 1)) {
                const int st = i % kStages;
                if (!mbar_wait(&M->empty[st], ((i / kStages) & 1) ^ 1, abort_flag, a.wait_ns)) {
                    *abort_flag = 1;
                    break;
                }
                const tc::TileInfo ti = it.info(a);
                const int64_t row0 = tc::dense_row(a, ti);
                unsigned char* dst = stages + st * kTileBytes;
                mbar_arrive_expect_tx(&M->full[st], kTileBytes);
                tma_load_2d(dst, &xmap, &M->full[st], 0, (int)row0);
                tma_load_2d(dst + 16384, &xmap, &M->full[st], 64, (int)row0);
                issued = i + 1;
            }
            if (*abort_flag) {
                const int zero = 0;
                const int from = issued > kStages ? issued - kStages : 0;
                for (int i = from; i < issued; i++)
                    mbar_wait(&M->full[i % kStages], (i / kStages) & 1, &zero, kWaitLimitNs);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0 && my_tiles > 0) {
            static_assert(KEYS, "rows are encoded by tc_rows_encode_kernel");
            constexpr uint32_t idesc = idesc_bf16_f32(128, 128);  // keys: one chain over the full K
            int64_t cur = -1;
            int committed = 0;
            tc::TileIter it;
            it.init(a, S, t_begin);
            for (int i = 0; i < my_tiles; i++, it.step(a, 1)) {
                const tc::TileInfo ti = it.info(a);
                const int64_t ls = ti.seg - seg0;
                bool ok = true;
                if (ti.seg != cur) {
                    ok = mbar_wait(&M->gready[ls & 3], (ls >> 2) & 1, abort_flag, a.wait_ns);
                    cur = ti.seg;
                }
                const int st = i % kStages, buf = i % kAcc;
                ok = ok && mbar_wait(&M->full[st], (i / kStages) & 1, abort_flag, a.wait_ns);
                ok = ok && mbar_wait(&M->accempty[buf], ((i / kAcc) & 1) ^ 1, abort_flag, a.wait_ns);
                if (!ok) {
                    *abort_flag = 1;
                    break;
                }
                tc_fence_after();
                // D[channel][token] = G x^T: the operands' K-steps lie at constant offsets, so the single
                // issuing thread spends two adds per MMA. Descriptors built in the loop cost 1 % (three
                // bit keys of the 8B-shaped cache, with their values: 4.52 -> 4.48 ms)
                const uint64_t gdesc = sdesc_sw128(smem_u32(bsplit)), xdesc = sdesc_sw128(smem_u32(stages + st * kTileBytes));
                const uint32_t d_base = tmem + buf * 128;
#pragma unroll
                for (int p = 0; p < kNPass; p++)
#pragma unroll
                    for (int ks = 0; ks < kD / 16; ks++) {
                        const uint32_t off = (uint32_t)((ks >> 2) * 16384 + (ks & 3) * 32) >> 4;
                        mma_bf16(d_base, gdesc + (uint32_t)(p * 32768 >> 4) + off, xdesc + off, idesc, (p > 0 || ks > 0) ? 1u : 0u);
                    }
                mma_commit(&M->accfull[buf]);
                const bool last_of_seg = (i + 1 == my_tiles) || it.seg_last(a);
                if (last_of_seg) mma_commit(&M->bfree);
                committed = i + 1;
            }
            if (*abort_flag && committed > 0) {
                const int zero = 0;
                const int i = committed - 1;
                mbar_wait(&M->accfull[i % kAcc], (i / kAcc) & 1, &zero, kWaitLimitNs);
            }
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------ gauge converter
        int64_t cur = -1;
        int nconv = 0;
        tc::TileIter it;
        it.init(a, S, t_begin);
        for (int i = 0; i < my_tiles; i++, it.step(a, 1)) {
            const tc::TileInfo ti = it.info(a);
            if (ti.seg == cur) continue;
            const int64_t ls = ti.seg - seg0;
            if (nconv > 0) {
                const bool ok = mbar_wait(&M->bfree, (nconv - 1) & 1, abort_flag, a.wait_ns);
                if (!__all_sync(0xffffffffu, ok)) {
                    *abort_flag = 1;
                    break;
                }
            }
            const float* Gf = a.G + tc::gauge_set(a, ti) * (int64_t)kD * g;
            tce::prefetch_next_gauges(a, ti, g, lane);
            tce::convert_gauge_set<KEYS, 4>(Gf, g, blk, nbk, fullk, bsz, bsplit, M->emaxb[ls & 3], M->gmaxb[ls & 3], 0, lane);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&M->gready[ls & 3]);
            cur = ti.seg;
            nconv++;
        }
    } else {
        // ------------------------------------------------------------ epilogue warpgroups
        const int wg = (warp - kEpiWarp0) >> 2;       // warpgroup: tiles i = wg (mod 3)
        const int q4 = warp & 3;                      // TMEM lane quadrant of this warp
        const int row = q4 * 32 + lane;               // TMEM lane: channel (and the token whose norm it takes)
        const int qw = warp - kEpiWarp0;              // job queue of this warp
        float* rowbuf = reinterpret_cast<float*>(queue) + qw * (32 + kJobCap);  // 32 values of a channel, or results
        uint32_t* jobs = reinterpret_cast<uint32_t*>(rowbuf + 32);
        const uint32_t lt = (1u << lane) - 1u;
        // The 32 values v of lane `src` spread over the lanes: lane k gets value k.
        auto spread = [&](const uint32_t (&v)[32], int src) -> float {
            __syncwarp();
            if (lane == src) {
#pragma unroll
                for (int k = 0; k < 32; k += 4)
                    *reinterpret_cast<uint4*>(rowbuf + k) = make_uint4(v[k], v[k + 1], v[k + 2], v[k + 3]);
            }
            __syncwarp();
            return rowbuf[lane];
        };
        // Appends a job for every set lane of m to the list of n (< cap) while there is room; returns the lanes left over.
        auto append = [&](uint32_t* list, int cap, uint32_t m, uint32_t word, int& n) -> uint32_t {
            const bool mine = (m >> lane) & 1u;
            const int at = n + __popc(m & lt);
            if (mine && at < cap) list[at] = word;
            const int all = n + __popc(m);
            n = all < cap ? all : cap;
            return all > cap ? __ballot_sync(0xffffffffu, mine && at >= cap) : 0u;
        };
        const float qmaxf = (float)((1 << BITS) - 1);
        const int qmax = (1 << BITS) - 1;
        int32_t flag = 0;
        tc::TileIter it;
        it.init(a, S, t_begin + wg);
        for (int i = wg; i < my_tiles; i += 3, it.step(a, 3)) {
            const tc::TileInfo ti = it.info(a);
            const int64_t ls = ti.seg - seg0;
            const int st = i % kStages, buf = i % kAcc;
            bool ok = mbar_wait(&M->accfull[buf], (i / kAcc) & 1, abort_flag, a.wait_ns);
            ok = ok && mbar_wait(&M->full[st], (i / kStages) & 1, abort_flag, a.wait_ns);
            ok = ok && mbar_wait(&M->gready[ls & 3], (ls >> 2) & 1, abort_flag, a.wait_ns);
            if (!__all_sync(0xffffffffu, ok)) {
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
            const unsigned char* stg = stages + st * kTileBytes;
            const bool valid = KEYS || row < ti.rows_valid;  // key tiles are whole token groups
            const uint32_t tacc = tmem + ((uint32_t)(q4 * 32) << 16) + buf * 128;
            const float* Gf = a.G + tc::gauge_set(a, ti) * (int64_t)kD * g;

            // ---- 1. ||x||^2 over the bound range of every block (bf16 -> fp32 exact)
            float bs[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            if (KEYS) {
                // a key block is one channel over the tile's 128 tokens: its bound uses the
                // largest group norm among those tokens. Each warp takes its own 32 token rows
                // (one per lane); the four warps of the warpgroup then exchange their per-group
                // maxima in shared memory (two buffers, alternating by tile)
                float gs[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 4
                for (int c8 = 0; c8 < 16; c8++) {
                    const uint4 xv = *reinterpret_cast<const uint4*>(stg + (c8 >> 3) * 16384 + row * 128 +
                                                                     (((c8 & 7) ^ (row & 7)) << 4));
                    float s0 = bf_lo(xv.x) * bf_lo(xv.x);
                    s0 = fmaf(bf_hi(xv.x), bf_hi(xv.x), s0);
                    s0 = fmaf(bf_lo(xv.y), bf_lo(xv.y), s0);
                    s0 = fmaf(bf_hi(xv.y), bf_hi(xv.y), s0);
                    s0 = fmaf(bf_lo(xv.z), bf_lo(xv.z), s0);
                    s0 = fmaf(bf_hi(xv.z), bf_hi(xv.z), s0);
                    s0 = fmaf(bf_lo(xv.w), bf_lo(xv.w), s0);
                    s0 = fmaf(bf_hi(xv.w), bf_hi(xv.w), s0);
                    const int r = (c8 * 8) / g;  // g >= 32: at most 4 groups
#pragma unroll
                    for (int rr = 0; rr < 4; rr++)
                        if (rr == r) gs[rr] += s0;
                }
                if (!(isfinite(gs[0]) && isfinite(gs[1]) && isfinite(gs[2]) && isfinite(gs[3]))) {
                    for (int c8 = 0; c8 < 16; c8++) {
                        const uint4 xv = *reinterpret_cast<const uint4*>(stg + (c8 >> 3) * 16384 + row * 128 +
                                                                         (((c8 & 7) ^ (row & 7)) << 4));
                        const uint32_t wv[4] = {xv.x, xv.y, xv.z, xv.w};
                        for (int k = 0; k < 4; k++)
                            if (bf16_nonfinite(wv[k] & 0xffffu) || bf16_nonfinite(wv[k] >> 16))
                                flag |= CG_FLAG_NONFINITE_INPUT;
                    }
                    // no bound for the tile's channels: the MMA's zero blocks times Inf or NaN spoil the
                    // token's z~ in every group, so all groups are undecided and every code is recomputed
                    for (int rr = 0; rr < 4; rr++) gs[rr] = INFINITY;
                }
#pragma unroll
                for (int rr = 0; rr < 4; rr++)
                    for (int off = 16; off >= 1; off >>= 1)
                        gs[rr] = fmaxf(gs[rr], __shfl_xor_sync(0xffffffffu, gs[rr], off));
                const int kx = (i - wg) / 3;  // this warpgroup's tile count
                float* xb = xch + (wg * 2 + (kx & 1)) * 16;
                if (lane == 0) {
#pragma unroll
                    for (int rr = 0; rr < 4; rr++) xb[q4 * 4 + rr] = gs[rr];
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&M->xbar[wg][kx & 1]);
                const bool okx = mbar_wait(&M->xbar[wg][kx & 1], (kx >> 1) & 1, abort_flag, a.wait_ns);
                if (!__all_sync(0xffffffffu, okx)) {
                    *abort_flag = 1;
                    break;
                }
                float gm[4];
#pragma unroll
                for (int rr = 0; rr < 4; rr++)
                    gm[rr] = fmaxf(fmaxf(xb[rr], xb[4 + rr]), fmaxf(xb[8 + rr], xb[12 + rr]));
                bs[0] = pick4(gm, row / g);
            }
            // ---- 2. approximate range of the channel from the accumulator, per 32-token chunk and whole
            static_assert(NBK == 1, "one block per channel");
            float cmn[4], cmx[4];
#pragma unroll 1
            for (int c = 0; c < 4; c++) {
                uint32_t v[32];
                tmem_ld32(tacc + c * 32, v);
                tmem_wait_ld();
                float lo = __uint_as_float(v[0]), hi = lo;
#pragma unroll
                for (int k = 1; k < 31; k += 2) {
                    lo = min3f(lo, __uint_as_float(v[k]), __uint_as_float(v[k + 1]));
                    hi = max3f(hi, __uint_as_float(v[k]), __uint_as_float(v[k + 1]));
                }
                set4(cmn, c, fminf(lo, __uint_as_float(v[31])));
                set4(cmx, c, fmaxf(hi, __uint_as_float(v[31])));
            }
            float mn[4] = {fminf(fminf(cmn[0], cmn[1]), fminf(cmn[2], cmn[3])), 0.0f, 0.0f, 0.0f};
            float mx[4] = {fmaxf(fmaxf(cmx[0], cmx[1]), fmaxf(cmx[2], cmx[3])), 0.0f, 0.0f, 0.0f};

            // ---- 3. error bound per block; scale/zero from the intervals when they agree
            float E[4];
            uint32_t s16[4], m16[4];
            int amb = 0;  // bit 2bk: scale needs the exact extremes; bit 2bk+1: zero needs the exact min
#pragma unroll
            for (int bk = 0; bk < 4; bk++) {
                E[bk] = 0.0f;
                s16[bk] = m16[bk] = 0;
                if (bk < nbk) {
                    E[bk] = sqrtf(bs[bk]) * 1.0001f * M->emaxb[ls & 3][bk] + (fabsf(mn[bk]) + fabsf(mx[bk])) * 2.4e-7f;
                    const float e = E[bk];
                    const float mn_lo = __fsub_rn(mn[bk], e), mn_hi = __fadd_rn(mn[bk], e);
                    const float mx_lo = __fsub_rn(mx[bk], e), mx_hi = __fadd_rn(mx[bk], e);
                    const uint32_t slo = f2h_bits(__fdiv_rn(fmaxf(__fsub_rn(mx_lo, mn_hi), 0.0f), qmaxf));
                    const uint32_t shi = scale16(mx_hi, mn_lo, qmaxf);
                    const uint32_t mlo = f2h_bits(mn_lo), mhi = f2h_bits(mn_hi);
                    s16[bk] = slo;
                    m16[bk] = mlo;
                    if (valid && slo != shi) amb |= 1 << (2 * bk);
                    if (valid && mlo != mhi) amb |= 2 << (2 * bk);
                }
            }

            // ---- 4. exact extremes of undecided channels: candidates are the values within 2E of the
            // approximate extreme, in chunks whose own extreme lies that close, found by one compare and
            // vote over the lanes per such chunk
            if (__any_sync(0xffffffffu, amb != 0)) {
                const int need = amb & 3;
                float ex_mn = INFINITY, ex_mx = -INFINITY;
                uint32_t m0 = 0, m1 = 0;  // MASKS: candidates of this lane's channel in chunk c, once made
                bool made = false;
                int nj = 0, c = 0;
                uint32_t todo = 0, left = 0xffffffffu;  // channels of chunk c to do; values of the first that no round has taken
                const float e2 = 2.0f * E[0], tl0 = __fadd_rn(mn[0], e2), th0 = __fsub_rn(mx[0], e2);
                do {
#pragma unroll 1
                    for (; c < 4; c++) {
                        const bool nl = need != 0 && !(pick4(cmn, c) > tl0);  // a NaN z~ is a candidate
                        const bool nh = (need & 1) && !(pick4(cmx, c) < th0);
                        if (todo == 0) todo = __ballot_sync(0xffffffffu, nl || nh);
                        if (todo == 0) continue;
                        const float tl = nl ? tl0 : -INFINITY, th = nh ? th0 : INFINITY;
                        uint32_t v[32];
                        if constexpr (MASKS) {
                            if (!made) {
                                tmem_ld32(tacc + c * 32, v);
                                tmem_wait_ld();
                                uint32_t a0 = 0, a1 = 0;  // sign bits of tl0 - z (z > tl0) and z - th0 (z < th0)
#pragma unroll
                                for (int k = 31; k >= 0; k--) {
                                    const float z = __uint_as_float(v[k]);
                                    a0 = __funnelshift_l(__float_as_uint(__fsub_rn(tl0, z)), a0, 1);
                                    a1 = __funnelshift_l(__float_as_uint(__fsub_rn(z, th0)), a1, 1);
                                }
                                m0 = nl ? ~a0 : 0u;
                                m1 = nh ? ~a1 : 0u;
                                made = true;
                            }
                            do {
                                const uint32_t m = m0 | m1, bit = m & (0u - m);
                                todo = __ballot_sync(0xffffffffu, m != 0);
                                if (!todo) break;
                                const uint32_t word = (uint32_t)(c * 32 + __ffs(m) - 1) | (uint32_t)row << 8 |
                                                      ((m0 & bit) ? 0x10000u : 0u) | ((m1 & bit) ? 0x20000u : 0u);
                                left = append(jobs, kJobCap, todo, word, nj);
                                if (!((left >> lane) & 1u)) {
                                    m0 &= ~bit;
                                    m1 &= ~bit;
                                }
                            } while (!left);
                            if (todo) break;  // the list is full
                            made = false;
                            continue;
                        }
                        tmem_ld32(tacc + c * 32, v);
                        tmem_wait_ld();
                        do {
                            const int src = __ffs(todo) - 1;
                            const float stl = __shfl_sync(0xffffffffu, tl, src), sth = __shfl_sync(0xffffffffu, th, src);
                            const float z = spread(v, src);
                            const uint32_t job = (uint32_t)(c * 32 + lane) | (uint32_t)(q4 * 32 + src) << 8 |
                                                 (z > stl ? 0u : 0x10000u) | (z < sth ? 0u : 0x20000u);
                            left = append(jobs, kJobCap, __ballot_sync(0xffffffffu, (job & 0x30000u) != 0u) & left, job, nj);
                            if (left) break;  // the list is full
                            todo &= todo - 1;
                            left = 0xffffffffu;
                        } while (todo);
                        if (todo) break;
                    }
                    if (nj) {
                        __syncwarp();
                        tce::run_jobs<kJobSlots>(jobs, rowbuf, nj, stg, Gf, g, lane);
                        __syncwarp();
#pragma unroll 1
                        for (int j = 0; j < nj; j++) {
                            const uint32_t w = jobs[j];
                            const float ze = rowbuf[j];
                            if ((int)((w >> 8) & 31u) == lane) {
                                if (w & 0x10000u) ex_mn = fminf(ex_mn, ze);
                                if (w & 0x20000u) ex_mx = fmaxf(ex_mx, ze);
                            }
                        }
                        __syncwarp();
                        nj = 0;
                    }
                } while (todo);
                if (need) {
                    m16[0] = f2h_bits(ex_mn);
                    if (need & 1) s16[0] = scale16(ex_mx, ex_mn, qmaxf);
                }
            }

            // ---- 5. code parameters per block
            float rinv[4], c0[4], lim[4];
            int fast = 0;  // bit bk: no value of the block can leave [0, qmax]
#pragma unroll
            for (int bk = 0; bk < 4; bk++) {
                rinv[bk] = c0[bk] = 0.0f;
                lim[bk] = 0.5f;
                if (bk < nbk) {
                    if (valid && (h_is_inf(s16[bk]) || h_is_inf(m16[bk]))) flag |= CG_FLAG_FP16_OVERFLOW;
                    const float sc = h2f_bits(s16[bk]), mz = h2f_bits(m16[bk]);
                    if (sc != 0.0f && !h_is_inf(s16[bk]) && !h_is_inf(m16[bk])) {
                        const float r = __frcp_rn(sc);
                        const float cc = -mz * r;
                        rinv[bk] = r;
                        c0[bk] = cc;
                        // |t~ - t| <= E/s plus roundings: the fma and its inputs r and c0 (u|z r|,
                        // 2u|c0|, u|t|) and the definition's subtract and divide (2u|t|)
                        const float zr = fmaxf(fabsf(mn[bk]), fabsf(mx[bk])) * r;
                        const float mu = E[bk] * r * 1.0001f + (zr + 2.0f * fabsf(cc) + 3.0f * (qmaxf + 1.0f)) * 6.6e-8f;
                        // mu < 1e-4: a code from z~ can only differ where the tolerance allows it
                        // (fmaxf: without a bound every code is recomputed)
                        lim[bk] = mu < 0.99e-4f ? 2.0f : fmaxf(0.5f - mu, -1.0f);
                        const float tlo = (mn[bk] - E[bk]) * r + cc, thi = (mx[bk] + E[bk]) * r + cc;
                        if (tlo > -0.49f + mu && thi < qmaxf + 0.49f - mu) fast |= 1 << bk;
                    }
                }
            }

            // ---- 6. codes from z~, stored straight from registers; near-boundary values repaired
            // rows: the token's codes; keys: the channel's 128-token stream (16 * BITS bytes)
            uint8_t* crow = KEYS ? a.codes + a.cmap.at(ti.l, ti.s, ti.b, ti.h, ti.t0) + (size_t)row * (16 * BITS)
                                 : a.codes + a.cmap.at(ti.l, ti.s, ti.b, ti.h, ti.t0 + row);
            int nj = 0;  // values within mu of a rounding boundary, to be recomputed exactly and patched
            // (with masks the row buffer serves the list: 20 jobs and their results)
            constexpr int kCodeCap = kMasks ? (32 + kJobCap) / 2 : kJobCap;
            uint32_t* cjobs = kMasks ? reinterpret_cast<uint32_t*>(rowbuf) : jobs;
            float* cres = kMasks ? rowbuf + kCodeCap : rowbuf;
            const float r = rinv[0], cc = c0[0], lm = lim[0];
#pragma unroll 1
            for (int c = 0; c < 4; c++) {
                uint32_t v[32];
                tmem_ld32(tacc + c * 32, v);
                tmem_wait_ld();
                uint32_t words[BITS];
#pragma unroll
                for (int w = 0; w < BITS; w++) words[w] = 0;
                // values within mu of a rounding boundary: whether the lane has one, or a mask of them
                float worst = 0.0f;
                uint32_t mask = 0;
                const float2 r2 = make_float2(r, r), c2 = make_float2(cc, cc), m2 = make_float2(kMagic, kMagic);
                if ((fast & 1) && lm > 1.0f) {  // no value can need a clamp or lie on the wrong side of a boundary
#pragma unroll
                    for (int k = 0; k < 32; k += 2) {
                        const float2 t = __ffma2_rn(make_float2(__uint_as_float(v[k]), __uint_as_float(v[k + 1])), r2, c2);
                        const float2 y = __fadd2_rn(t, m2);
                        tce::put_code<BITS>(words, k, __float_as_uint(y.x));
                        tce::put_code<BITS>(words, k + 1, __float_as_uint(y.y));
                    }
                } else {
                    // clamping before the rounding gives the same code as clamping after it (a dead channel: r = c0 = 0, so 0)
#pragma unroll
                    for (int k = 0; k < 32; k += 2) {
                        float2 t = __ffma2_rn(make_float2(__uint_as_float(v[k]), __uint_as_float(v[k + 1])), r2, c2);
                        t = make_float2(fminf(fmaxf(t.x, 0.0f), qmaxf), fminf(fmaxf(t.y, 0.0f), qmaxf));
                        const float2 y = __fadd2_rn(t, m2);
                        tce::put_code<BITS>(words, k, __float_as_uint(y.x));
                        tce::put_code<BITS>(words, k + 1, __float_as_uint(y.y));
                        const float2 q = __fadd2_rn(y, make_float2(-kMagic, -kMagic));
                        const float2 e = __ffma2_rn(q, make_float2(-1.0f, -1.0f), t);  // exact
                        if constexpr (kMasks)
                            mask |= (fabsf(e.x) > lm ? 1u : 0u) << k | (fabsf(e.y) > lm ? 2u : 0u) << k;
                        else
                            worst = max3f(worst, fabsf(e.x), fabsf(e.y));
                    }
                }
#pragma unroll
                for (int w = 0; w < BITS; w++) words[w] -= pack_bias<BITS>(w);
                uint32_t* dst = reinterpret_cast<uint32_t*>(crow) + c * BITS;
                if (BITS % 4 == 0) {
#pragma unroll
                    for (int w = 0; w < BITS; w += 4)
                        *reinterpret_cast<uint4*>(dst + w) = make_uint4(words[w], words[w + 1], words[w + 2], words[w + 3]);
                } else if (BITS % 2 == 0) {
#pragma unroll
                    for (int w = 0; w < BITS; w += 2) *reinterpret_cast<uint2*>(dst + w) = make_uint2(words[w], words[w + 1]);
                } else {
#pragma unroll
                    for (int w = 0; w < BITS; w++) dst[w] = words[w];
                }
                uint32_t todo = __ballot_sync(0xffffffffu, kMasks ? mask != 0 : worst > lm), left = 0xffffffffu;
                while (todo || (c == 3 && nj)) {
                    if (todo) {
                        if constexpr (kMasks) {
                            do {
                                const uint32_t word = (uint32_t)(c * 32 + __ffs(mask) - 1) | (uint32_t)row << 8;
                                left = append(cjobs, kCodeCap, todo, word, nj);
                                if (!((left >> lane) & 1u)) mask &= mask - 1;
                                todo = __ballot_sync(0xffffffffu, mask != 0);
                            } while (todo && !left);
                        } else {
                            tmem_ld32(tacc + c * 32, v);
                            tmem_wait_ld();
                            do {
                                const int src = __ffs(todo) - 1;
                                const float sr = __shfl_sync(0xffffffffu, r, src), sc = __shfl_sync(0xffffffffu, cc, src);
                                const float sl = __shfl_sync(0xffffffffu, lm, src);
                                const float z = spread(v, src);
                                const float t = fminf(fmaxf(fmaf(z, sr, sc), 0.0f), qmaxf);
                                left = append(cjobs, kCodeCap, __ballot_sync(0xffffffffu, fabsf(t - ((t + kMagic) - kMagic)) > sl) & left,
                                              (uint32_t)(c * 32 + lane) | (uint32_t)(q4 * 32 + src) << 8, nj);
                                if (left) break;  // the list is full
                                todo &= todo - 1;
                                left = 0xffffffffu;
                            } while (todo);
                        }
                        if (!todo && c < 3) break;
                    }
                    __syncwarp();
                    tce::run_jobs<kJobSlots>(cjobs, cres, nj, stg, Gf, g, lane);
                    __syncwarp();
#pragma unroll 1
                    for (int j = 0; j < nj; j++) {
                        const uint32_t w = cjobs[j];
                        const float ze = cres[j];
                        if ((int)((w >> 8) & 31u) == lane)
                            patch_code<BITS>(crow, (int)(w & 127u) * BITS, quant_code(ze, h2f_bits(s16[0]), h2f_bits(m16[0]), qmax));
                    }
                    __syncwarp();
                    nj = 0;
                }
            }

            // ---- 7. scales; release the stage and the accumulator buffer
            if (valid) {
                uint32_t* sp = KEYS ? a.scales + a.smap.at(ti.l, ti.s, ti.b, ti.h, ti.t0) + row
                                    : a.scales + a.smap.at(ti.l, ti.s, ti.b, ti.h, ti.t0 + row);
#pragma unroll
                for (int bk = 0; bk < 4; bk++)
                    if (bk < nbk) sp[bk] = s16[bk] | (m16[bk] << 16);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&M->accempty[buf]);
                mbar_arrive(&M->empty[st]);
            }
        }
        if (flag) raise_flag(a.status, flag);
    }
    __syncthreads();
    if (*abort_flag && threadIdx.x == 0) raise_flag(a.status, CG_FLAG_PIPE_TIMEOUT);
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, kAcc * 128);
    }
}

template <int BITS, bool KEYS, int NBK, bool MASKS>
cudaError_t launch_encode_nbk(const EncParams& P, const CUtensorMap& map, cudaStream_t st) {
    const size_t smem = EncSmem::total;
    cudaError_t e =
        cudaFuncSetAttribute(tc_encode_kernel<BITS, KEYS, NBK, MASKS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t grid = P.S.n_tiles < tc::num_sms() ? P.S.n_tiles : tc::num_sms();
    tc_encode_kernel<BITS, KEYS, NBK, MASKS><<<(unsigned)grid, kThreads, smem, st>>>(map, P);
    return cudaGetLastError();
}

// keys: one block (the 128-token group) per channel (block-uniform and KIVI value rows are
// encoded by cg_tc_rows.cu)
template <int BITS, bool KEYS>
cudaError_t launch_encode_bits(const EncParams& P, const CUtensorMap& map, cudaStream_t st) {
    static_assert(KEYS, "rows are encoded by tc_rows_encode_kernel");
    // one tile a CTA, masks / search: 24.2 / 25.1 us (2 bits, g = 128), 20.8 / 22.1 (6 bits, g = 64), 16.3 / 16.2 (4
    // bits, g = 32); 13 tiles: 95.9 / 93.2 us (keys and values, 2 bits, g = 32), 139.6 / 136.5 (6 bits, g = 64)
    if (P.S.n_tiles <= 4 * (int64_t)tc::num_sms()) return launch_encode_nbk<BITS, KEYS, 1, true>(P, map, st);
    return launch_encode_nbk<BITS, KEYS, 1, false>(P, map, st);
}

template <bool KEYS>
cudaError_t launch_encode(const RowArgs& a, cudaStream_t st) {
    EncParams P;
    P.a = a;
    P.S = tc::make_sched(a);
    if (P.S.n_tiles == 0) return cudaSuccess;
    CUtensorMap map;
    const uint64_t rows = (uint64_t)a.L * 2 * a.B * a.H * a.T_x;
    if (!make_tmap_bf16_sw128(&map, a.x, rows, kD, kD * 2, 128)) return cudaErrorInvalidValue;
    switch (a.bits) {
        case 2: return launch_encode_bits<2, KEYS>(P, map, st);
        case 3: return launch_encode_bits<3, KEYS>(P, map, st);
        case 4: return launch_encode_bits<4, KEYS>(P, map, st);
        case 6: return launch_encode_bits<6, KEYS>(P, map, st);
        case 8: return launch_encode_bits<8, KEYS>(P, map, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// KIVI keys as rows of the key tensor: s = 0 only, block = the 128-token key group, t_count
// = the quantized tokens (whole groups); cmap/smap address a group's first token (the
// kernel adds the channel's stream). Groups of g >= 32 channels (at most 4 per head).
bool tc_key_encode_eligible(const RowArgs& a) {
    if (a.d != kD || a.blk != 128 || a.g < 32) return false;
    if (a.t_count < 128 || a.t_count % 128) return false;
    const int64_t rows = (int64_t)a.L * 2 * a.B * a.H * a.T_x;
    if (rows + 128 >= (int64_t)1 << 31) return false;
    if ((reinterpret_cast<uintptr_t>(a.x) & 15u) || (reinterpret_cast<uintptr_t>(a.codes) & 15u)) return false;
    return tmap_encode_fn() != nullptr;
}

cudaError_t tc_launch_key_encode(const RowArgs& a, cudaStream_t st) { return launch_encode<true>(a, st); }

}  // namespace cg
