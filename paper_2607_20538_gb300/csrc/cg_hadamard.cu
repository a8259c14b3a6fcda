// cg_hadamard.cu -- Hadamard gauge by fast Walsh-Hadamard transform (the structured Hadamard control
// of Sec. 4.3, G = H_g / sqrt(g) in fp32 for every (l, s, h, r)), O(g log g) per group and no gauge
// tensor read.
//
// Every entry of G is +-c, c = fp32(1 / sqrt(g)), so the library's products are +-fl(c x_j), and the
// pairwise summation order over j (adjacent pairs first, halves last) is the butterfly order of the
// transform (stride 1 first, stride g/2 last): scaling x by c with rounding and then running the
// butterflies in fp32 gives exactly the library's z.
//
// Mapping: a lane holds 32 consecutive channels of a token row as sixteen pairs (k, k + 16), so strides
// 1..8 are packed adds and fused multiply-adds by -1 (a - b rounded once), stride 16 stays inside a
// pair, and strides 32 and 64 take one shuffle per value. d / 32 lanes share a row; a warp's 32 lane rows
// are 2 KB of the dense tensor. They come by TMA into a three-stage ring of the warp (64-byte rows in
// the 64-byte swizzle, so that the lanes' 16-byte reads meet no bank conflict) and leave the decode the
// same way; a lane's 32 codes are BITS whole words, read and written by vector accesses that are
// contiguous over the lanes. (Two rows a lane as the halves of the pairs needed 64 value registers and
// spilled around the shuffles: 0.86 ms to encode.) No division: its slow path is a call that would
// spill the row.
// Bound by instruction issue and the FP32 pipe. 8B-shaped cache (1 GiB bf16, g = 128, 4 bits), against one
// warp per row with five shuffle stages and byte-wise packing through shared memory:
// encode 2.46 -> 0.46 ms (22 instructions a value, issue slots 67 % busy), decode 1.04 -> 0.31 ms.
#include "cg_sm100.cuh"
#include "cg_tc_common.cuh"
#include "cg_tc_enc.cuh"
#include "cg_tmap.h"

namespace cg {
namespace {

using namespace sm100;
using tce::kMagic;
using tce::max3f;
using tce::min3f;
using tce::pack_bias;
using tce::put_code;

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kCtas = 4;      // per SM (64 registers; two with 116 measured 3 % slower)
constexpr int kTile = 2048;   // 32 lane rows of 32 bf16
constexpr int kStages = 3;    // encode input ring of a warp
constexpr int kOutBufs = 2;   // decode output buffers of a warp
constexpr int kDecSmem = kWarps * kOutBufs * kTile;

struct HadArgs {
    uint8_t* codes;
    uint32_t* scales;
    int32_t* status;
    uint64_t wait_ns;
    int64_t c_unit, c_tok, s_unit, s_tok;  // bytes / u32 from a unit (a token) to the next
    uint32_t rows, T;                      // token rows of this launch, tokens per unit
    uint32_t tiles;
    int g, lpr_shift;                      // gauge group, log2(lanes per row)
    int lpb, lpb_shift;                    // lanes per quantization block (1 when a lane holds whole blocks)
    float c;
};

__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }

// Butterflies over channel strides 1 .. g / 2: 32 channels of a lane as pairs (k, k + 16), then lanes.
__device__ __forceinline__ void fwht(float2 (&v)[16], int g, int lane) {
    const float2 neg = dup(-1.0f);
#pragma unroll
    for (int h = 1; h < 16; h <<= 1) {
        if (h >= 8 && h >= g) break;  // g >= 8
#pragma unroll
        for (int k = 0; k < 16; k++)
            if (!(k & h)) {
                const float2 a = v[k], b = v[k + h];
                v[k] = __fadd2_rn(a, b);
                v[k + h] = __ffma2_rn(b, neg, a);
            }
    }
    if (g > 16) {
#pragma unroll
        for (int k = 0; k < 16; k++) v[k] = make_float2(__fadd_rn(v[k].x, v[k].y), __fsub_rn(v[k].x, v[k].y));
    }
#pragma unroll 1
    for (int m = 1; 32 * m < g; m <<= 1) {
        const float2 sg = dup(lane & m ? -1.0f : 1.0f);
#pragma unroll
        for (int k = 0; k < 16; k++)
            v[k] = __ffma2_rn(v[k], sg, make_float2(__shfl_xor_sync(0xffffffffu, v[k].x, m), __shfl_xor_sync(0xffffffffu, v[k].y, m)));
    }
}

// Offsets of a lane's row of a tile.
struct LaneRow {
    bool valid;
    int64_t c, s;  // first byte of the row's codes, first word of its scales
};
__device__ __forceinline__ LaneRow lane_row(const HadArgs& a, uint32_t lane_row_index) {
    const uint32_t n = lane_row_index >> a.lpr_shift;
    LaneRow r;
    r.valid = n < a.rows;
    const uint32_t u = r.valid ? n / a.T : 0u, t = r.valid ? n - u * a.T : 0u;
    r.c = u * a.c_unit + t * a.c_tok;
    r.s = u * a.s_unit + t * a.s_tok;
    return r;
}

// The rule's code clamp(rint(fl(d / s)), 0, qmax) as 0x4B400000 + code, for any d = fl(z - m), from the
// product t = fl(d r) with r close to 1 / s (0 for s = 0). Clamping before rounding gives the same code, a NaN
// quotient codes to 0. Where t lies within `lim` of a half-integer B, the rounded quotient's side of B is
// the side of d to B s, which is exact (9 x 11 significant bits): neighbouring floats d differ by more
// than half an ulp of B in the quotient, so fl(d / s) = B only for d = B s, a tie to even.
__device__ __forceinline__ uint32_t exact_code(float d, float s, float r, float qmax, float lim) {
    const float t = fminf(fmaxf(__fmul_rn(d, r), 0.0f), qmax);
    const float y = __fadd_rn(t, kMagic);
    const float q = __fsub_rn(y, kMagic), e = __fsub_rn(t, q);
    uint32_t code = __float_as_uint(y);
    if (fabsf(e) > lim) {
        const float p = __fmul_rn(__fadd_rn(q, e > 0.0f ? 0.5f : -0.5f), s);
        const bool odd = code & 1u;
        if (e > 0.0f && (d > p || (d == p && odd))) code++;
        if (e < 0.0f && (d < p || (d == p && odd))) code--;
    }
    return code;
}

// fp16(fl(d / qmax)) for a range d >= 0, without a division (its slow path is a call, around which 64
// live values would be spilled): the products with fl(1 / qmax) widened by 8 u bracket the IEEE
// quotient; where the ends round to different fp16 values lo and hi, the quotient's side of their
// midpoint M is the side of d to M qmax, which is exact (12 x 8 significant bits), as in exact_code.
template <int BITS>
__device__ __forceinline__ uint32_t scale_bits(float d) {
    constexpr float qmaxf = (float)((1 << BITS) - 1), kRq = 1.0f / qmaxf, kU8 = 8.0f * tce::kU;
    const float t = __fmul_rn(d, kRq);
    const uint32_t lo = f2h_bits(__fmul_rn(t, 1.0f - kU8)), hi = f2h_bits(__fmul_rn(t, 1.0f + kU8));
    if (lo == hi) return lo;
    const float m = hi == 0x7c00u ? 65520.0f : 0.5f * (h2f_bits(lo) + h2f_bits(hi));
    const float p = __fmul_rn(m, qmaxf);
    return d > p || (d == p && (lo & 1u)) ? hi : lo;
}

__device__ __forceinline__ float rcp_approx(float v) {  // within one ulp (2 u)
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

template <int N>
__device__ __forceinline__ void store_words(uint32_t* dst, const uint32_t (&w)[N]) {
    if constexpr (N % 4 == 0) {
#pragma unroll
        for (int k = 0; k < N; k += 4) stg_hint_u4(dst + k, make_uint4(w[k], w[k + 1], w[k + 2], w[k + 3]), policy_evict_first());
    } else if constexpr (N % 2 == 0) {
#pragma unroll
        for (int k = 0; k < N; k += 2) *reinterpret_cast<uint2*>(dst + k) = make_uint2(w[k], w[k + 1]);
    } else {
#pragma unroll
        for (int k = 0; k < N; k++) dst[k] = w[k];
    }
}
template <int N>
__device__ __forceinline__ void load_words(const uint32_t* src, uint32_t (&w)[N]) {
    if constexpr (N % 4 == 0) {
#pragma unroll
        for (int k = 0; k < N; k += 4) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(src + k));
            w[k] = v.x; w[k + 1] = v.y; w[k + 2] = v.z; w[k + 3] = v.w;
        }
    } else if constexpr (N % 2 == 0) {
#pragma unroll
        for (int k = 0; k < N; k += 2) {
            const uint2 v = __ldg(reinterpret_cast<const uint2*>(src + k));
            w[k] = v.x; w[k + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < N; k++) w[k] = __ldg(src + k);
    }
}

// Sub-block of channel k of a lane, NSUB quantization blocks among its 32 channels (1 when a block
// spans lanes).
template <int NSUB>
__device__ constexpr int sub_of(int k) {
    return k * NSUB / 32;
}

template <int BITS, int NSUB, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, kCtas * kWarps / WARPS) hadamard_encode_kernel(const __grid_constant__ CUtensorMap xmap, const HadArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr float qmaxf = (float)((1 << BITS) - 1);
    // a product d r with r within 2 u of 1 / s is within 4 u of the IEEE quotient: closer than this to a
    // half-integer, exact_code decides
    constexpr float kLim = 0.5f - (qmaxf + 1.0f) * 2.6e-7f;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + WARPS * kStages * kTile) + warp * kStages;
    unsigned char* ring = smem + warp * kStages * kTile;
    const int zero_flag = 0;
    if (lane == 0) {
        for (int i = 0; i < kStages; i++) mbar_init(&bars[i], 1);
        fence_barrier_init();
    }
    __syncwarp();
    const uint32_t w0 = blockIdx.x * WARPS + warp, nw = gridDim.x * WARPS;
    const int n_my = w0 < a.tiles ? (int)((a.tiles - w0 + nw - 1) / nw) : 0;
    auto issue = [&](int i) {
        if (lane == 0 && i < n_my) {
            mbar_arrive_expect_tx(&bars[i % kStages], kTile);
            tma_load_2d_hint(ring + (i % kStages) * kTile, &xmap, &bars[i % kStages], 0, (int)((w0 + i * nw) * 32u), policy_evict_first());
        }
    };
    for (int i = 0; i < kStages; i++) issue(i);
    int32_t flag = 0;
    for (int i = 0; i < n_my; i++) {
        if (!__all_sync(0xffffffffu, mbar_wait(&bars[i % kStages], (i / kStages) & 1, &zero_flag, a.wait_ns))) {
            flag |= CG_FLAG_PIPE_TIMEOUT;
            for (int j = i; j < n_my && j < i + kStages; j++)  // let the copies in flight land
                mbar_wait(&bars[j % kStages], (j / kStages) & 1, &zero_flag, tc::kWaitLimitNs);
            break;
        }
        const unsigned char* src = ring + (i % kStages) * kTile + lane * 64;
        float2 v[16];
#pragma unroll
        for (int q = 0; q < 2; q++) {  // 16-byte pieces q and q + 2: channels 8 q .. and 16 + 8 q ..
            const int sw = (lane >> 1) & 3;
            const uint4 xa = *reinterpret_cast<const uint4*>(src + ((q ^ sw) << 4));
            const uint4 xb = *reinterpret_cast<const uint4*>(src + (((q + 2) ^ sw) << 4));
            const uint32_t wa[4] = {xa.x, xa.y, xa.z, xa.w}, wb[4] = {xb.x, xb.y, xb.z, xb.w};
#pragma unroll
            for (int e = 0; e < 4; e++) {
                v[8 * q + 2 * e] = make_float2(__fmul_rn(a.c, tce::bf_lo(wa[e])), __fmul_rn(a.c, tce::bf_lo(wb[e])));
                v[8 * q + 2 * e + 1] = make_float2(__fmul_rn(a.c, tce::bf_hi(wa[e])), __fmul_rn(a.c, tce::bf_hi(wb[e])));
            }
        }
        fwht(v, a.g, lane);

        // ranges of the row's blocks
        float mn[NSUB], mx[NSUB];
#pragma unroll
        for (int sb = 0; sb < NSUB; sb++) {
            constexpr int kSub = 32 / NSUB;
            auto val = [&](int k) { return k < 16 ? v[k & 15].x : v[k & 15].y; };
            float lo = val(sb * kSub), hi = lo;
#pragma unroll
            for (int k = 1; k + 1 < kSub; k += 2) {
                lo = min3f(lo, val(sb * kSub + k), val(sb * kSub + k + 1));
                hi = max3f(hi, val(sb * kSub + k), val(sb * kSub + k + 1));
            }
            lo = fminf(lo, val(sb * kSub + kSub - 1));
            hi = fmaxf(hi, val(sb * kSub + kSub - 1));
            for (int off = 1; off < a.lpb; off <<= 1) {
                lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, off));
                hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, off));
            }
            mn[sb] = lo;
            mx[sb] = hi;
        }
        // an Inf or NaN input makes all (at least 8) values of its group Inf or NaN, and this sum of one
        // value of each eight too; huge finite values can overflow as well: look at the input. The lane's
        // codes then come from exact_code, which knows NaN (min and max pass over one)
        bool plain = isfinite((v[0].x + v[8].x) + (v[0].y + v[8].y));
        if (!plain) {
            for (int q = 0; q < 4; q++) {
                const uint4 x = *reinterpret_cast<const uint4*>(src + 16 * q);
                const uint32_t w[4] = {x.x, x.y, x.z, x.w};
                for (int e = 0; e < 4; e++)
                    if (bf16_nonfinite(w[e] & 0xffffu) || bf16_nonfinite(w[e] >> 16)) flag |= CG_FLAG_NONFINITE_INPUT;
            }
        }
        __syncwarp();
        issue(i + kStages);

        // scales, and whether every code is a plain rounding (no clamp, no quotient near a half-integer)
        uint32_t sz[NSUB];
        float m[NSUB], r[NSUB];
#pragma unroll
        for (int sb = 0; sb < NSUB; sb++) {
            sz[sb] = scale_bits<BITS>(__fsub_rn(mx[sb], mn[sb])) | (f2h_bits(mn[sb]) << 16);
            if (h_is_inf(sz[sb]) || h_is_inf(sz[sb] >> 16)) flag |= CG_FLAG_FP16_OVERFLOW;
            const float s = h2f_bits(sz[sb] & 0xffffu);
            m[sb] = h2f_bits(sz[sb] >> 16);
            r[sb] = s != 0.0f ? rcp_approx(s) : 0.0f;
            plain = plain && (mn[sb] - m[sb]) * r[sb] > -0.49f && (mx[sb] - m[sb]) * r[sb] < qmaxf + 0.49f;
        }
        uint32_t cw[BITS];
#pragma unroll
        for (int w = 0; w < BITS; w++) cw[w] = 0u;
        float worst = 0.0f;
#pragma unroll
        for (int k = 0; k < 16; k++) {
            const int sa = sub_of<NSUB>(k), sb = sub_of<NSUB>(k + 16);
            const float2 d = __fadd2_rn(v[k], make_float2(-m[sa], -m[sb]));
            const float2 t = __fmul2_rn(d, make_float2(r[sa], r[sb]));
            const float2 y = __fadd2_rn(t, dup(kMagic));
            put_code<BITS>(cw, k, __float_as_uint(y.x));
            put_code<BITS>(cw, k + 16, __float_as_uint(y.y));
            const float2 e = __ffma2_rn(__fadd2_rn(y, dup(-kMagic)), dup(-1.0f), t);  // both differences exact
            worst = max3f(worst, fabsf(e.x), fabsf(e.y));
        }
        if (__any_sync(0xffffffffu, !plain || !(worst <= kLim))) {
            // clamps, exact quotients (4-bit codes: about 1 % of the tiles)
#pragma unroll
            for (int w = 0; w < BITS; w++) cw[w] = 0u;
#pragma unroll
            for (int k = 0; k < 16; k++) {
                const int sa = sub_of<NSUB>(k), sb = sub_of<NSUB>(k + 16);
                put_code<BITS>(cw, k, exact_code(__fsub_rn(v[k].x, m[sa]), h2f_bits(sz[sa] & 0xffffu), r[sa], qmaxf, kLim));
                put_code<BITS>(cw, k + 16, exact_code(__fsub_rn(v[k].y, m[sb]), h2f_bits(sz[sb] & 0xffffu), r[sb], qmaxf, kLim));
            }
        }
#pragma unroll
        for (int w = 0; w < BITS; w++) cw[w] -= pack_bias<BITS>(w);
        const LaneRow row = lane_row(a, (w0 + i * nw) * 32u + lane);
        const int q = lane & ((1 << a.lpr_shift) - 1);  // 32-channel part of the row
        if (row.valid) {
            store_words<BITS>(reinterpret_cast<uint32_t*>(a.codes + row.c) + q * BITS, cw);
            if ((q & (a.lpb - 1)) == 0) {
                const int at = NSUB > 1 ? q * NSUB : q >> a.lpb_shift;
#pragma unroll
                for (int sb = 0; sb < NSUB; sb++) a.scales[row.s + at + sb] = sz[sb];
            }
        }
    }
    if (flag) raise_flag(a.status, flag);
}

template <int BITS, int NSUB>
__global__ void __launch_bounds__(kThreads, kCtas) hadamard_decode_kernel(const __grid_constant__ CUtensorMap omap, const HadArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr uint32_t kMask = (1u << BITS) - 1u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char* bufs = smem + warp * kOutBufs * kTile;
    const uint32_t w0 = blockIdx.x * kWarps + warp, nw = gridDim.x * kWarps;
    const int n_my = w0 < a.tiles ? (int)((a.tiles - w0 + nw - 1) / nw) : 0;
    const int q = lane & ((1 << a.lpr_shift) - 1);
    const int at = NSUB > 1 ? q * NSUB : q >> a.lpb_shift;
    uint32_t cw[BITS], sz[NSUB];
    auto load = [&](int i) {  // codes and scales of this lane's row of tile i (rows that do not exist: row 0)
        const LaneRow row = lane_row(a, (w0 + i * nw) * 32u + lane);
        load_words<BITS>(reinterpret_cast<const uint32_t*>(a.codes + row.c) + q * BITS, cw);
#pragma unroll
        for (int sb = 0; sb < NSUB; sb++) sz[sb] = __ldg(a.scales + row.s + at + sb);
    };
    if (n_my > 0) load(0);
    for (int i = 0; i < n_my; i++) {
        float2 v[16];
        auto code = [&](int k) -> float {  // 2^23 + q: no integer conversion
            const int p = k * BITS;
            uint32_t y = cw[p >> 5] >> (p & 31);
            if ((p & 31) + BITS > 32) y |= cw[(p >> 5) + 1 < BITS ? (p >> 5) + 1 : 0] << (32 - (p & 31));
            return __uint_as_float((y & kMask) | 0x4B000000u);
        };
#pragma unroll
        for (int k = 0; k < 16; k++) {
            const int sa = sub_of<NSUB>(k), sb = sub_of<NSUB>(k + 16);
            const float2 f = __fadd2_rn(make_float2(code(k), code(k + 16)), dup(-8388608.0f));
            v[k] = __ffma2_rn(f, make_float2(h2f_bits(sz[sa] & 0xffffu), h2f_bits(sz[sb] & 0xffffu)),
                              make_float2(h2f_bits(sz[sa] >> 16), h2f_bits(sz[sb] >> 16)));
        }
        if (i + 1 < n_my) load(i + 1);
        fwht(v, a.g, lane);  // H is symmetric: G^T zhat = c H zhat
        unsigned char* buf = bufs + (i % kOutBufs) * kTile;
        if (lane == 0) bulk_wait_read<kOutBufs - 1>();  // the store that last used this buffer has read it
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 2; j++) {  // pieces j and j + 2
            uint32_t oa[4], ob[4];
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const float2 t0 = __fmul2_rn(dup(a.c), v[8 * j + 2 * e]), t1 = __fmul2_rn(dup(a.c), v[8 * j + 2 * e + 1]);
                const __nv_bfloat162 ba = __floats2bfloat162_rn(t0.x, t1.x), bb = __floats2bfloat162_rn(t0.y, t1.y);
                oa[e] = *reinterpret_cast<const uint32_t*>(&ba);
                ob[e] = *reinterpret_cast<const uint32_t*>(&bb);
            }
            const int sw = (lane >> 1) & 3;
            *reinterpret_cast<uint4*>(buf + lane * 64 + ((j ^ sw) << 4)) = make_uint4(oa[0], oa[1], oa[2], oa[3]);
            *reinterpret_cast<uint4*>(buf + lane * 64 + (((j + 2) ^ sw) << 4)) = make_uint4(ob[0], ob[1], ob[2], ob[3]);
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
            tma_store_2d(&omap, buf, 0, (int)((w0 + i * nw) * 32u));  // rows past the tensor are not written
            bulk_commit();
        }
    }
    if (lane == 0) bulk_wait<0>();
}

template <typename K>
cudaError_t launch_tiles(K kernel, int warps, int smem, const HadArgs& a, const CUtensorMap& map, cudaStream_t st) {
    if (smem > 48 * 1024) {  // more than a kernel may use unasked
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    const uint32_t want = (a.tiles + warps - 1) / warps, most = (uint32_t)(kCtas * kWarps / warps) * (uint32_t)tc::num_sms();
    kernel<<<want < most ? want : most, warps * 32, smem, st>>>(map, a);
    return cudaGetLastError();
}

// Encode of few tiles (all resident at once): such a call is bound by its host time, and CTAs of four
// warps stay below 48 KB of shared memory, so that the attribute call (0.2 us) is left out. 65 tokens,
// encode and decode: 19.4 -> 18.4 us. Large calls keep eight warps (four: up to 1 % slower).
template <int BITS, int NSUB>
cudaError_t launch_sub(const HadArgs& a, const CUtensorMap& map, bool enc, cudaStream_t st) {
    constexpr int kEncWarpSmem = kStages * kTile + kStages * 8;  // a warp's tiles and barriers
    if (!enc) return launch_tiles(hadamard_decode_kernel<BITS, NSUB>, kWarps, kDecSmem, a, map, st);
    if (a.tiles <= (uint32_t)(kCtas * kWarps * tc::num_sms()))
        return launch_tiles(hadamard_encode_kernel<BITS, NSUB, kWarps / 2>, kWarps / 2, kWarps / 2 * kEncWarpSmem, a, map, st);
    return launch_tiles(hadamard_encode_kernel<BITS, NSUB, kWarps>, kWarps, kWarps * kEncWarpSmem, a, map, st);
}

template <int BITS>
cudaError_t launch_bits(const HadArgs& a, int blk, const CUtensorMap& map, bool enc, cudaStream_t st) {
    if (blk == 8) return launch_sub<BITS, 4>(a, map, enc, st);
    if (blk == 16) return launch_sub<BITS, 2>(a, map, enc, st);
    return launch_sub<BITS, 1>(a, map, enc, st);
}

}  // namespace

// Block-uniform rows; the units (l, s, b, h) of x / out and of the packed history follow each other
// at a constant distance. Launches cover as many whole units as 31-bit lane-row indices allow.
cudaError_t launch_hadamard(const RowArgs& r, bool encode, cudaStream_t st) {
    const int64_t units = (int64_t)r.L * 2 * r.B * r.H;
    if (units < 1 || r.t_count < 1) return cudaSuccess;
    if (!tmap_encode_fn()) return cudaErrorNotSupported;
    HadArgs a{};
    a.status = r.status;
    a.wait_ns = r.wait_ns;
    a.c_unit = r.cmap.sH;
    a.c_tok = r.cmap.sT;
    a.s_unit = r.smap.sH;
    a.s_tok = r.smap.sT;
    a.T = (uint32_t)r.t_count;
    a.g = r.g;
    a.lpr_shift = r.d == 32 ? 0 : (r.d == 64 ? 1 : (r.d == 128 ? 2 : 3));
    a.lpb = r.blk < 32 ? 1 : r.blk / 32;
    a.lpb_shift = a.lpb == 8 ? 3 : a.lpb >> 1;
    a.c = (float)(1.0 / sqrt((double)r.g));
    const int64_t per_unit = r.t_count << a.lpr_shift;
    const int64_t most = (((int64_t)1 << 31) - 128) / per_unit;
    if (most < 1) return cudaErrorInvalidValue;
    for (int64_t u = 0; u < units; u += most) {
        const int64_t n = units - u < most ? units - u : most;
        a.codes = r.codes + r.cmap.base + u * a.c_unit;
        a.scales = r.scales + r.smap.base + u * a.s_unit;
        a.rows = (uint32_t)(n * r.t_count);
        a.tiles = (uint32_t)((n * per_unit + 31) / 32);
        CUtensorMap map;
        const uint16_t* dense = (encode ? r.x : r.out) + u * r.t_count * r.d;
        if (!make_tmap_bf16_rows32(&map, dense, (uint64_t)(n * per_unit))) return cudaErrorInvalidValue;
        cudaError_t e;
        switch (r.bits) {
            case 2: e = launch_bits<2>(a, r.blk, map, encode, st); break;
            case 3: e = launch_bits<3>(a, r.blk, map, encode, st); break;
            case 4: e = launch_bits<4>(a, r.blk, map, encode, st); break;
            case 6: e = launch_bits<6>(a, r.blk, map, encode, st); break;
            case 8: e = launch_bits<8>(a, r.blk, map, encode, st); break;
            default: e = cudaErrorInvalidValue;
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace cg
