// cg_simt.cu -- CUDA-core kernels of the encode/decode path.
//
// These kernels evaluate the gauge rotation Z = G X (Sec. 3) exactly as the library's
// quantization rule defines it (pairwise fp32 summation of the products), so scales,
// zeros and codes are reproducible to the bit. They serve every shape the library accepts and are the launch choice where a
// tile of tokens is too small or the group too small for the tensor-core kernels.
//
// Thread mapping (row kernels): a warp takes R token rows at a time; lane owns NR = d / 32
// consecutive channels of each. The (l, s, h) gauge set sits in shared memory; a CTA handles the
// rows (b, t) that share it.
#include <type_traits>

#include "cg_launch.h"

namespace cg {
namespace {

constexpr int kRowThreads = 256;
constexpr int kRowWarps = kRowThreads / 32;

__device__ __forceinline__ float seg_min(float v, int seg) {
    for (int off = seg >> 1; off >= 1; off >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, off));
    return v;
}
__device__ __forceinline__ float seg_max(float v, int seg) {
    for (int off = seg >> 1; off >= 1; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
    return v;
}

// One gauge-space coordinate sum_j G[i][j] x[j] in the library's fixed fp32 order:
// pairwise summation of the products. The 8-product leaves are summed as trees and merged
// in chunk order with a binary carry (the partial sum of 2^k chunks waits at level k), which
// reproduces the pairwise tree for a power-of-two count of chunks. Gcol[j * gstride] =
// G[i][j]; g a power of two in [8, 128].
__device__ __forceinline__ float gauge_coord(const float* Gcol, int gstride, const float* x, int g) {
    float l0 = 0.0f, l1 = 0.0f, l2 = 0.0f, l3 = 0.0f, v = 0.0f;
#pragma unroll 1
    for (int c = 0; c < g / 8; c++) {
        float a[8], b[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            a[k] = Gcol[(8 * c + k) * gstride];
            b[k] = x[8 * c + k];
        }
        v = tree8(a, b);
        if (c & 1) {
            v = __fadd_rn(l0, v);
            if (c & 2) {
                v = __fadd_rn(l1, v);
                if (c & 4) {
                    v = __fadd_rn(l2, v);
                    if (c & 8) v = __fadd_rn(l3, v);
                    else l3 = v;
                } else {
                    l2 = v;
                }
            } else {
                l1 = v;
            }
        } else {
            l0 = v;
        }
    }
    return v;
}

// Word w of the little-endian stream in which code c sits at bits [c*bits, (c+1)*bits).
__device__ __forceinline__ uint32_t pack_word(const uint8_t* q, int w, int bits) {
    int bit0 = w * 32, c0 = bit0 / bits, c1 = (bit0 + 31) / bits;
    uint32_t word = 0;
    for (int c = c0; c <= c1; c++) {
        int p = c * bits - bit0;
        uint32_t v = q[c];
        word |= p >= 0 ? (v << p) : (v >> (-p));
    }
    return word;
}

// ------------------------------------------------------------------------------------
// Rows: R token rows x NR channels of a lane at once. Bound by the FP32 pipe: the pairwise rule
// costs one multiply and one add per product, with no contraction. Each gauge value read from shared
// memory serves R rows and each x value NR channels (16-byte reads of both: 16 reads for 256
// multiplies and adds at d = 128), so shared memory stays out of the way. Gauge rows are padded by 16
// bytes and stored so that the 32 lanes' rows of one register channel are neighbours: conflict-free
// reads. x rows are padded by 16 bytes per 32 values, so that lanes of different gauge groups read
// different banks. Measured against one row per warp and two 4-byte reads per product: one token for
// 64 sequences x 32 layers x 8 heads (d = 128, g = 128, 4 bits) 250 -> 74 us, 65,536 rows of d = 256
// (g = 128) 2762 -> 472 us, their decode 1937 -> 451 us; the FP32 peak allows 27 and 107 us.
// ------------------------------------------------------------------------------------
template <int NR>
struct RowCfg {
    static constexpr int d = NR * 32;
    static constexpr int kRows = NR == 1 ? 8 : 4;                  // R
    static constexpr int kThreads = NR == 8 ? 512 : 256;           // 16 warps an SM: two CTAs, one for d = 256
    static constexpr int kWarps = kThreads / 32;
    static constexpr int kXPad = d + d / 8;                        // padded x row
    using piece_t = std::conditional_t<NR == 8, uint64_t, uint32_t>;  // a lane's NR codes of up to 8 bits
    static constexpr int kPieces = kRows * 32 * (int)(sizeof(piece_t) + 4);  // packed pieces, scales
    static constexpr int kWarpBytes = kRows * kXPad * 4 > kPieces ? kRows * kXPad * 4 : kPieces;  // x rows, then pieces
};

__device__ __forceinline__ int x_slot(int c) { return c + 4 * (c >> 5); }

// Gauge slot of channel c (lane c / NR, register c % NR).
template <int NR>
__device__ __forceinline__ int gauge_slot(int c) { return (c % NR) * 32 + c / NR; }

// out[r][k] = the library's pairwise sum over j of G[k][j] x_r[j], two channels and R rows (eight sums
// with their carry levels in registers) at a time. Gl: this lane's gauge row of channel 0, channel k
// at + k * gk; xg: the first x row, group of this lane from value x0 on. Sixteen products per step;
// binary carry of the step sums: the partial sum of 2^n steps waits at level n.
template <int NR, int R>
__device__ __forceinline__ void gauge_rows(const float* Gl, int gk, const float* xg, int xpad, int x0, int g,
                                           float (&out)[R][NR]) {
    constexpr int KB = NR < 2 ? NR : 2;
#pragma unroll
    for (int k0 = 0; k0 < NR; k0 += KB) {
        float z[R][KB], l1[R][KB], l2[R][KB], l3[R][KB];
        auto chunk = [&](int c, float (&v)[R][KB]) {  // sums of products 8 c .. 8 c + 7
            float a[KB][8];
#pragma unroll
            for (int k = 0; k < KB; k++) {
                const float4 u = *reinterpret_cast<const float4*>(Gl + (k0 + k) * gk + 8 * c);
                const float4 w = *reinterpret_cast<const float4*>(Gl + (k0 + k) * gk + 8 * c + 4);
                a[k][0] = u.x; a[k][1] = u.y; a[k][2] = u.z; a[k][3] = u.w;
                a[k][4] = w.x; a[k][5] = w.y; a[k][6] = w.z; a[k][7] = w.w;
            }
            const float* xc = xg + x_slot(x0 + 8 * c);
#pragma unroll
            for (int r = 0; r < R; r++) {
                const float4 u = *reinterpret_cast<const float4*>(xc + r * xpad);
                const float4 w = *reinterpret_cast<const float4*>(xc + r * xpad + 4);
                const float b[8] = {u.x, u.y, u.z, u.w, w.x, w.y, w.z, w.w};
#pragma unroll
                for (int k = 0; k < KB; k++) v[r][k] = tree8(a[k], b);
            }
        };
        auto each = [&](auto f) {
#pragma unroll
            for (int r = 0; r < R; r++)
#pragma unroll
                for (int k = 0; k < KB; k++) f(r, k);
        };
        if (g == 8) {
            chunk(0, z);
        } else {
            each([&](int r, int k) { l1[r][k] = l2[r][k] = l3[r][k] = 0.0f; });
#pragma unroll 1
            for (int c = 0; c < g / 16; c++) {
                float l0[R][KB];
                chunk(2 * c, l0);
                chunk(2 * c + 1, z);
                each([&](int r, int k) { z[r][k] = __fadd_rn(l0[r][k], z[r][k]); });
                if (c & 1) {
                    each([&](int r, int k) { z[r][k] = __fadd_rn(l1[r][k], z[r][k]); });
                    if (c & 2) {
                        each([&](int r, int k) { z[r][k] = __fadd_rn(l2[r][k], z[r][k]); });
                        if (c & 4) each([&](int r, int k) { z[r][k] = __fadd_rn(l3[r][k], z[r][k]); });
                        else each([&](int r, int k) { l3[r][k] = z[r][k]; });
                    } else {
                        each([&](int r, int k) { l2[r][k] = z[r][k]; });
                    }
                } else {
                    each([&](int r, int k) { l1[r][k] = z[r][k]; });
                }
            }
        }
        each([&](int r, int k) { out[r][k0 + k] = z[r][k]; });
    }
}

// (b, t) of row `row` = b * t_count + t.
__device__ __forceinline__ void row_bt(int64_t row, int64_t t_count, int& b, int64_t& t) {
    if ((row | t_count) < ((int64_t)1 << 31)) {
        b = (int)((uint32_t)row / (uint32_t)t_count);
        t = (uint32_t)row - (uint32_t)b * (uint32_t)t_count;
    } else {
        b = (int)(row / t_count);
        t = row - b * t_count;
    }
}

// Offsets of R consecutive rows in the dense tensor, the codes and the scales: the first row's, and
// constant steps where the rows are tokens of one sequence, or one token of consecutive sequences.
struct RowWalk {
    int64_t row, x, c, s, dx, dc, ds, t;
    bool linear;
    __device__ __forceinline__ RowWalk(const RowArgs& a, int l, int ss, int h, int d, int64_t row0, int n) : row(row0) {
        int b;
        row_bt(row0, a.t_count, b, t);
        at(a, l, ss, h, d, b, t);
        linear = true;
        if (a.t_count == 1) {
            dx = (int64_t)a.H * a.T_x * d;
            dc = a.cmap.sB;
            ds = a.smap.sB;
        } else {
            dx = d;
            dc = a.cmap.sT;
            ds = a.smap.sT;
            linear = t + n <= a.t_count;
        }
    }
    __device__ __forceinline__ void at(const RowArgs& a, int l, int ss, int h, int d, int b, int64_t t) {
        x = ((((int64_t)(l * 2 + ss) * a.B + b) * a.H + h) * a.T_x + t) * d;
        c = a.cmap.at(l, ss, b, h, t);
        s = a.smap.at(l, ss, b, h, t);
    }
    __device__ __forceinline__ void next(const RowArgs& a, int l, int ss, int h, int d) {
        row++;
        if (linear) {
            x += dx;
            c += dc;
            t++;
            if (a.t_count == 1 || (t & ((1 << a.smap.tshift) - 1)) == 0) s += ds;  // tiles: 16 tokens share scales
        } else {
            int b;
            row_bt(row, a.t_count, b, t);
            if (b < a.B) at(a, l, ss, h, d, b, t);
        }
    }
};

// The rule's code, clamp(rint(fl((z - m) / s)), 0, qmax), from a reciprocal product (rcp = fl(1 / s), 0
// for s = 0): the product is within a few ulp of the quotient, so it rounds to the same integer
// unless it lies within 2^-12 of a half-integer, where the exact division decides (rare). Clamping
// before the rounding gives the same code (a NaN quotient codes to 0); adding 1.5 * 2^23 rounds to
// nearest even and leaves the code in the low bits.
__device__ __forceinline__ uint32_t quant_code_rcp(float z, float s, float m, float rcp, float qmax) {
    constexpr float kMagic = 12582912.0f;
    const float d = __fsub_rn(z, m);
    float t = fminf(fmaxf(__fmul_rn(d, rcp), 0.0f), qmax);
    float y = __fadd_rn(t, kMagic);
    if (fabsf(__fsub_rn(t, __fsub_rn(y, kMagic))) > 0.49975f || !(fabsf(d) < 3.0e38f)) {
        t = s == 0.0f ? 0.0f : fminf(fmaxf(__fdiv_rn(d, s), 0.0f), qmax);
        y = __fadd_rn(t, kMagic);
    }
    return __float_as_uint(y) & 0xffu;
}

// Whether one of the two bf16 values of a word is not finite.
__device__ __forceinline__ bool pair_nonfinite(uint32_t w) { return (((w & 0x7f807f80u) + 0x00800080u) & 0x80008000u) != 0u; }

// NR consecutive bf16 values (NR * 2 bytes, naturally aligned) as packed words.
template <int NR>
__device__ __forceinline__ void load_pairs(const uint16_t* p, uint32_t (&w)[NR > 1 ? NR / 2 : 1]) {
    if constexpr (NR == 8) {
        const uint4 v = *reinterpret_cast<const uint4*>(p);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    } else if constexpr (NR == 4) {
        const uint2 v = *reinterpret_cast<const uint2*>(p);
        w[0] = v.x; w[1] = v.y;
    } else if constexpr (NR == 2) {
        w[0] = *reinterpret_cast<const uint32_t*>(p);
    } else {
        w[0] = *p;
    }
}

// Encode: Z = G X, then per-token block min/max quantization and packing (or the raw fp32 Z for the
// no-compression rows).
template <int NR>
__global__ void __launch_bounds__(RowCfg<NR>::kThreads, NR == 8 ? 1 : 2) row_encode_kernel(RowArgs a, int rows_per_cta) {
    using C = RowCfg<NR>;
    constexpr int d = C::d, R = C::kRows;
    extern __shared__ __align__(16) unsigned char smem[];
    const int g = a.g, gp = g + 4;
    float* Gs = reinterpret_cast<float*>(smem);  // [slot of channel i][j], rows padded to g + 4
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* xs = reinterpret_cast<float*>(smem + (size_t)d * gp * 4 + (size_t)warp * C::kWarpBytes);
    using piece_t = typename C::piece_t;
    piece_t* pieces = reinterpret_cast<piece_t*>(xs);  // [R][32], once the x rows are used up
    uint32_t* szs = reinterpret_cast<uint32_t*>(pieces + R * 32);  // [R][32]: scales and zeros

    const int y = blockIdx.y;
    const int h = y % a.H;
    const int s = a.s_lo + (y / a.H) % a.s_n;
    const int l = y / (a.H * a.s_n);
    const float4* Gsrc = reinterpret_cast<const float4*>(a.G + ((int64_t)(l * 2 + s) * a.H + h) * (int64_t)d * g);
    const int lq = 29 - __clz(g);  // log2(g / 4)
#pragma unroll 8
    for (int e = threadIdx.x; e < d * g / 4; e += C::kThreads)
        *reinterpret_cast<float4*>(Gs + gauge_slot<NR>(e >> lq) * gp + 4 * (e & (g / 4 - 1))) = __ldg(Gsrc + e);
    __syncthreads();

    const int64_t rows = (int64_t)a.B * a.t_count;
    const int64_t r_lo = (int64_t)blockIdx.x * rows_per_cta;
    const int64_t r_hi = r_lo + rows_per_cta < rows ? r_lo + rows_per_cta : rows;
    const int bits = a.bits, blk = a.blk;
    const float qmaxf = (float)((1 << bits) - 1);
    const int c0 = NR * lane;                       // first channel of this lane
    const int x0 = c0 & ~(g - 1);                   // its gauge group
    const int lanes_per_blk = blk / NR;             // block >= 8 >= NR
    const int lpb_shift = 31 - __clz(lanes_per_blk);
    const int nb_lane = NR * bits, nw = d * bits / 32, nb = d / blk;
    // output words w = lane, lane + 32: first piece and its bit offset in the word
    constexpr int NW = NR == 8 ? 2 : 1;
    int wp[NW], wat[NW];
#pragma unroll
    for (int q = 0; q < NW; q++) {
        wp[q] = 32 * (lane + 32 * q) / nb_lane;
        wat[q] = wp[q] * nb_lane - 32 * (lane + 32 * q);
    }
    int32_t flag = 0;

    for (int64_t r0 = r_lo + warp * R; r0 < r_hi; r0 += C::kWarps * R) {
        const int n = r_hi - r0 < R ? (int)(r_hi - r0) : R;
        const RowWalk first(a, l, s, h, d, r0, n);
        RowWalk p = first;
        bool bad = false;
#pragma unroll
        for (int r = 0; r < R; r++) {
            uint32_t w[NR > 1 ? NR / 2 : 1];
            load_pairs<NR>(a.x + p.x + c0, w);
            if (r + 1 < n) p.next(a, l, s, h, d);  // missing rows repeat the last one
            float* xr = xs + r * C::kXPad + x_slot(c0);
            float f[NR];
#pragma unroll
            for (int k = 0; k < NR; k++) {
                f[k] = k & 1 ? __uint_as_float(w[k >> 1] & 0xffff0000u) : __uint_as_float(w[k >> 1] << 16);
                if (!(k & 1)) bad = bad || pair_nonfinite(w[k >> 1]);
            }
            if constexpr (NR >= 4) {
#pragma unroll
                for (int k = 0; k < NR; k += 4) *reinterpret_cast<float4*>(xr + k) = make_float4(f[k], f[k + 1], f[k + 2], f[k + 3]);
            } else {
#pragma unroll
                for (int k = 0; k < NR; k++) xr[k] = f[k];
            }
        }
        if (bad) flag |= CG_FLAG_NONFINITE_INPUT;
        __syncwarp();
        float z[R][NR];
        gauge_rows<NR, R>(Gs + lane * gp, 32 * gp, xs, C::kXPad, x0, g, z);
        p = first;
        if (a.none_mode) {
#pragma unroll
            for (int r = 0; r < R; r++) {
                if (r >= n) break;
                float* zr = reinterpret_cast<float*>(a.codes + p.c) + c0;
#pragma unroll
                for (int k = 0; k < NR; k++) zr[k] = z[r][k];
                p.next(a, l, s, h, d);
            }
            __syncwarp();
            continue;
        }
        __syncwarp();  // the x rows have been read: their space takes the packed pieces
#pragma unroll
        for (int r = 0; r < R; r++) {
            float mn = z[r][0], mx = z[r][0];
#pragma unroll
            for (int k = 1; k < NR; k++) {
                mn = fminf(mn, z[r][k]);
                mx = fmaxf(mx, z[r][k]);
            }
            mn = seg_min(mn, lanes_per_blk);
            mx = seg_max(mx, lanes_per_blk);
            const uint32_t sz = scale_zero(mn, mx, qmaxf, &flag);
            const float sc = h2f_bits(sz & 0xffffu), mz = h2f_bits(sz >> 16);
            const float rcp = sc != 0.0f ? __frcp_rn(sc) : 0.0f;
            piece_t v = 0;
#pragma unroll
            for (int k = 0; k < NR; k++) v |= (piece_t)quant_code_rcp(z[r][k], sc, mz, rcp, qmaxf) << (k * bits);
            pieces[r * 32 + lane] = v;
            if ((lane & (lanes_per_blk - 1)) == 0) szs[r * 32 + (lane >> lpb_shift)] = sz;
        }
        __syncwarp();
        for (int r = 0; r < n; r++) {
            if (lane < nb) a.scales[p.s + lane] = szs[r * 32 + lane];
            uint32_t* cw = reinterpret_cast<uint32_t*>(a.codes + p.c);
#pragma unroll
            for (int q = 0; q < NW; q++) {
                if (lane + 32 * q >= nw) break;
                int pc = wp[q], at = wat[q];
                uint32_t word = (uint32_t)(pieces[r * 32 + pc] >> -at);
                for (at += nb_lane, pc++; at < 32; at += nb_lane, pc++) word |= (uint32_t)pieces[r * 32 + pc] << at;
                cw[lane + 32 * q] = word;
            }
            p.next(a, l, s, h, d);
        }
        __syncwarp();
    }
    if (flag) raise_flag(a.status, flag);
}

// ------------------------------------------------------------------------------------
// Block-uniform tiles: Z = G X for the 16 tokens of a tile, then one min/max range per
// tile block (16 tokens x blk channels, Sec. 4.3 with T_b = 16 from Sec. 4.2), codes and
// packing in the per-token row layout, one {scale, zero} pair per tile block.
// One warp per tile; the CTA shares the (l, s, h) gauge set in shared memory. Serves the shapes
// that the tensor-core tile encoder does not take (d other than 128, block < 32, < 64 tokens).
// ------------------------------------------------------------------------------------
constexpr int kTileTokens = CG_TILE_TOKENS;
constexpr int kTileWarpsMax = 16;
constexpr size_t kSmemOptIn = 232448;  // 227 KB of dynamic shared memory per CTA

__host__ __device__ __forceinline__ size_t tile_warp_bytes(int d) {
    return (size_t)kTileTokens * d * 4 + (size_t)kTileTokens * d + 32 * 4;
}

// Binary-carry merge of the chunk sums of one pairwise sum (see gauge_coord).
__device__ __forceinline__ void carry_push(float& l0, float& l1, float& l2, float& l3, float& v, int c) {
    if (c & 1) {
        v = __fadd_rn(l0, v);
        if (c & 2) {
            v = __fadd_rn(l1, v);
            if (c & 4) {
                v = __fadd_rn(l2, v);
                if (c & 8) v = __fadd_rn(l3, v);
                else l3 = v;
            } else {
                l2 = v;
            }
        } else {
            l1 = v;
        }
    } else {
        l0 = v;
    }
}

// gauge_coord for four tokens at once: out[t] = sum_j G[i][j] x_t[j] in the library's
// pairwise order, x_t = x0 + t * xstride (16-byte aligned rows). Each gauge value loaded
// from shared memory serves the four tokens.
__device__ __forceinline__ void gauge_coord4(const float* Gcol, int gstride, const float* x0, int xstride, int g,
                                             float (&out)[4]) {
    float l0[4] = {}, l1[4] = {}, l2[4] = {}, l3[4] = {}, v[4] = {};
#pragma unroll 1
    for (int c = 0; c < g / 8; c++) {
        float a[8];
#pragma unroll
        for (int k = 0; k < 8; k++) a[k] = Gcol[(8 * c + k) * gstride];
#pragma unroll
        for (int t = 0; t < 4; t++) {
            const float4* xp = reinterpret_cast<const float4*>(x0 + t * xstride + 8 * c);
            const float4 u0 = xp[0], u1 = xp[1];
            const float b[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
            v[t] = tree8(a, b);
            carry_push(l0[t], l1[t], l2[t], l3[t], v[t], c);
        }
    }
#pragma unroll
    for (int t = 0; t < 4; t++) out[t] = v[t];
}

template <int NR>
__global__ void __launch_bounds__(kTileWarpsMax * 32) tile_encode_kernel(RowArgs a) {
    constexpr int d = NR * 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int g = a.g;
    float* Gs = reinterpret_cast<float*>(smem);  // Gs[r][jj][i] = G_r[i][jj]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    unsigned char* wbase = smem + (size_t)d * g * 4 + (size_t)warp * tile_warp_bytes(d);
    float* buf = reinterpret_cast<float*>(wbase);                         // [16][d]: x, then z
    uint8_t* qs = wbase + (size_t)kTileTokens * d * 4;                    // [16][d] codes
    uint32_t* smw = reinterpret_cast<uint32_t*>(qs + (size_t)kTileTokens * d);  // [d/blk] scales

    const int y = blockIdx.y;
    const int h = y % a.H;
    const int s = a.s_lo + (y / a.H) % a.s_n;
    const int l = y / (a.H * a.s_n);
    const float* Gsrc = a.G + ((int64_t)(l * 2 + s) * a.H + h) * (int64_t)d * g;
    for (int e = threadIdx.x; e < d * g; e += blockDim.x) {
        int r = e / (g * g), rem = e - r * g * g, i = rem / g, jj = rem - i * g;
        Gs[r * g * g + jj * g + i] = __ldg(Gsrc + e);
    }
    __syncthreads();

    const int64_t ntc = (a.t_count + kTileTokens - 1) / kTileTokens;  // tiles per unit in this call
    const int64_t total = (int64_t)a.B * ntc;
    const int64_t chunk = (total + gridDim.x - 1) / gridDim.x;
    const int64_t k0 = (int64_t)blockIdx.x * chunk;
    const int64_t k1 = k0 + chunk < total ? k0 + chunk : total;
    const int bits = a.bits, blk = a.blk;
    const int qmax = (1 << bits) - 1;
    const float qmaxf = (float)qmax;
    const int nw = d * bits / 32;  // packed words per token row
    int32_t flag = 0;

    for (int64_t tk = k0 + warp; tk < k1; tk += nwarps) {
        const int b = (int)(tk / ntc);
        const int64_t t_lo = (tk - (int64_t)b * ntc) * kTileTokens;
        const int nt = a.t_count - t_lo < kTileTokens ? (int)(a.t_count - t_lo) : kTileTokens;
        // the tile's tokens are nt consecutive rows of x: nt * d bf16, 16-byte chunks
        const uint4* xt = reinterpret_cast<const uint4*>(
            a.x + ((((int64_t)(l * 2 + s) * a.B + b) * a.H + h) * a.T_x + t_lo) * d);
        for (int e = lane; e < nt * d / 8; e += 32) {
            const uint4 v = __ldg(xt + e);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
            float f[8];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const uint32_t lo = w[k] & 0xffffu, hi = w[k] >> 16;
                if (bf16_nonfinite(lo) || bf16_nonfinite(hi)) flag |= CG_FLAG_NONFINITE_INPUT;
                f[2 * k] = bf16_bits_to_float(lo);
                f[2 * k + 1] = bf16_bits_to_float(hi);
            }
            float4* dst = reinterpret_cast<float4*>(buf + 8 * e);
            dst[0] = make_float4(f[0], f[1], f[2], f[3]);
            dst[1] = make_float4(f[4], f[5], f[6], f[7]);
        }
        __syncwarp();
        // Z for four tokens at a time; each quad's z overwrites its x rows once all lanes
        // have read them
        for (int tq = 0; tq * 4 < nt; tq++) {
            float zq[NR][4];
#pragma unroll
            for (int k = 0; k < NR; k++) {
                const int c = lane + 32 * k, r = c / g, i = c - r * g;
                gauge_coord4(Gs + r * g * g + i, g, buf + (size_t)(4 * tq) * d + r * g, d, g, zq[k]);
            }
            __syncwarp();
#pragma unroll
            for (int t = 0; t < 4; t++)
                if (4 * tq + t < nt) {
#pragma unroll
                    for (int k = 0; k < NR; k++) buf[(4 * tq + t) * d + lane + 32 * k] = zq[k][t];
                }
            __syncwarp();
        }
        // tile block ranges: tokens per lane, then lanes (segments of min(blk, 32)), then
        // registers for blk > 32
        const int seg = blk < 32 ? blk : 32;
        const int per = blk > 32 ? blk / 32 : 1;
        float mn[NR], mx[NR];
#pragma unroll
        for (int k = 0; k < NR; k++) {
            const int c = lane + 32 * k;
            float lo = buf[c], hi = lo;
            for (int tt = 1; tt < nt; tt++) {
                const float v = buf[tt * d + c];
                lo = fminf(lo, v);
                hi = fmaxf(hi, v);
            }
            mn[k] = seg_min(lo, seg);
            mx[k] = seg_max(hi, seg);
        }
        if (per > 1) {
#pragma unroll
            for (int k = 0; k < NR; k++) {
                const int kb = (k / per) * per;
                float a0 = mn[kb], a1 = mx[kb];
                for (int kk = 1; kk < per; kk++) {
                    a0 = fminf(a0, mn[kb + kk]);
                    a1 = fmaxf(a1, mx[kb + kk]);
                }
                mn[k] = a0;
                mx[k] = a1;
            }
        }
#pragma unroll
        for (int k = 0; k < NR; k++) {
            const int c = lane + 32 * k;
            const uint32_t sz = scale_zero(mn[k], mx[k], qmaxf, &flag);
            const float sc = h2f_bits(sz & 0xffffu), mz = h2f_bits(sz >> 16);
            for (int tt = 0; tt < nt; tt++) qs[tt * d + c] = (uint8_t)quant_code(buf[tt * d + c], sc, mz, qmax);
            if ((c % blk) == 0) smw[c / blk] = sz;
        }
        __syncwarp();
        for (int e = lane; e < nt * nw; e += 32) {
            const int tt = e / nw, w = e - tt * nw;
            uint32_t* cw = reinterpret_cast<uint32_t*>(a.codes + a.cmap.at(l, s, b, h, t_lo + tt));
            cw[w] = pack_word(qs + tt * d, w, bits);
        }
        if (lane < d / blk) a.scales[a.smap.at(l, s, b, h, t_lo) + lane] = smw[lane];
        __syncwarp();
    }
    if (flag) raise_flag(a.status, flag);
}

// ------------------------------------------------------------------------------------
// Row decode: unpack, dequantize zhat = q*s + m, then Xhat = G^T Zhat, bf16 store. The rows of
// gauge_rows() are columns of G here.
// ------------------------------------------------------------------------------------
template <int NR>
__global__ void __launch_bounds__(RowCfg<NR>::kThreads, NR == 8 ? 1 : 2) row_decode_kernel(RowArgs a, int rows_per_cta) {
    using C = RowCfg<NR>;
    constexpr int d = C::d, R = C::kRows;
    extern __shared__ __align__(16) unsigned char smem[];
    const int g = a.g, gp = g + 4;
    float* Gs = reinterpret_cast<float*>(smem);  // [slot of channel i][j] = G[j][i]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* zs = reinterpret_cast<float*>(smem + (size_t)d * gp * 4 + (size_t)warp * C::kWarpBytes);

    const int y = blockIdx.y;
    const int h = y % a.H;
    const int s = a.s_lo + (y / a.H) % a.s_n;
    const int l = y / (a.H * a.s_n);
    const float* Gsrc = a.G + ((int64_t)(l * 2 + s) * a.H + h) * (int64_t)d * g;
    const int lg = 31 - __clz(g);
#pragma unroll 8
    for (int e = threadIdx.x; e < d * g; e += C::kThreads) {
        const int row = e >> lg, i = e & (g - 1);  // row = group * g + j, column i of the group
        Gs[gauge_slot<NR>((row & ~(g - 1)) + i) * gp + (row & (g - 1))] = __ldg(Gsrc + e);
    }
    __syncthreads();

    const int64_t rows = (int64_t)a.B * a.t_count;
    const int64_t r_lo = (int64_t)blockIdx.x * rows_per_cta;
    const int64_t r_hi = r_lo + rows_per_cta < rows ? r_lo + rows_per_cta : rows;
    const int bits = a.bits, blk = a.blk, nw = d * bits / 32;
    const uint32_t mask = (1u << bits) - 1u;
    const int c0 = NR * lane, x0 = c0 & ~(g - 1);
    const int bit0 = c0 * bits, wi = bit0 >> 5, sh = bit0 & 31;

    for (int64_t r0 = r_lo + warp * R; r0 < r_hi; r0 += C::kWarps * R) {
        const int n = r_hi - r0 < R ? (int)(r_hi - r0) : R;
        const RowWalk first(a, l, s, h, d, r0, n);
        RowWalk p = first;
#pragma unroll
        for (int r = 0; r < R; r++) {
            const int64_t coff = p.c, soff = p.s;
            if (r + 1 < n) p.next(a, l, s, h, d);  // missing rows repeat the last one
            float f[NR];
            if (a.none_mode) {
                const float* zr = reinterpret_cast<const float*>(a.codes + coff) + c0;
#pragma unroll
                for (int k = 0; k < NR; k++) f[k] = zr[k];
            } else {
                // this lane's NR codes: NR * bits <= 64 bits starting at bit bit0 of the row
                const uint32_t* cw = reinterpret_cast<const uint32_t*>(a.codes + coff);
                const uint32_t w0 = __ldg(cw + wi);
                const uint32_t w1 = wi + 1 < nw ? __ldg(cw + wi + 1) : 0u;
                const uint32_t w2 = NR * 8 > 32 && wi + 2 < nw ? __ldg(cw + wi + 2) : 0u;
                const uint64_t lo = (((uint64_t)w1 << 32) | w0) >> sh;
                const uint64_t cv = sh ? (lo | ((uint64_t)w2 << (64 - sh))) : lo;
                const uint32_t sz = __ldg(a.scales + soff + c0 / blk);
                const float sc = h2f_bits(sz & 0xffffu), mz = h2f_bits(sz >> 16);
#pragma unroll
                for (int k = 0; k < NR; k++) f[k] = fmaf((float)((uint32_t)(cv >> (k * bits)) & mask), sc, mz);
            }
            float* xr = zs + r * C::kXPad + x_slot(c0);
#pragma unroll
            for (int k = 0; k < NR; k++) xr[k] = f[k];
        }
        __syncwarp();
        float z[R][NR];
        gauge_rows<NR, R>(Gs + lane * gp, 32 * gp, zs, C::kXPad, x0, g, z);
        p = first;
#pragma unroll
        for (int r = 0; r < R; r++) {
            if (r >= n) break;
            uint16_t* orow = a.out + p.x + c0;
            p.next(a, l, s, h, d);
            uint32_t o[NR];
#pragma unroll
            for (int k = 0; k < NR; k++) o[k] = __bfloat16_as_ushort(__float2bfloat16_rn(z[r][k]));
            if constexpr (NR == 8) {
                *reinterpret_cast<uint4*>(orow) = make_uint4(o[0] | o[1] << 16, o[2] | o[3] << 16, o[4] | o[5] << 16, o[6] | o[7] << 16);
            } else if constexpr (NR == 4) {
                *reinterpret_cast<uint2*>(orow) = make_uint2(o[0] | o[1] << 16, o[2] | o[3] << 16);
            } else if constexpr (NR == 2) {
                *reinterpret_cast<uint32_t*>(orow) = o[0] | o[1] << 16;
            } else {
                orow[0] = (uint16_t)o[0];
            }
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------------------------
// KIVI keys: per-channel ranges over a group of Gt tokens (one CTA per (l, b, h, group)).
// ------------------------------------------------------------------------------------
template <int NR>
__global__ void __launch_bounds__(kRowThreads) key_encode_kernel(KeyArgs a) {
    constexpr int d = NR * 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int g = a.g, Gt = a.Gt, bits = a.bits;
    const int pay = Gt * bits / 8;
    float* Gs = reinterpret_cast<float*>(smem);                          // transposed
    float* Zs = reinterpret_cast<float*>(smem + (size_t)d * g * 4);      // [Gt][d]
    float* xsAll = Zs + (size_t)Gt * d;                                  // [warps][d]
    uint8_t* stage = reinterpret_cast<uint8_t*>(xsAll + kRowWarps * d);  // [d][pay]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* xs = xsAll + warp * d;

    const int64_t tg = blockIdx.x;
    const int bh = blockIdx.y % (a.B * a.H), l = blockIdx.y / (a.B * a.H);
    const int b = bh / a.H, h = bh % a.H;
    const float* Gsrc = a.G + ((int64_t)(l * 2 + 0) * a.H + h) * (int64_t)d * g;
    for (int e = threadIdx.x; e < d * g; e += kRowThreads) {
        int r = e / (g * g), rem = e - r * g * g, i = rem / g, jj = rem - i * g;
        Gs[r * g * g + jj * g + i] = __ldg(Gsrc + e);
    }
    __syncthreads();
    int32_t flag = 0;
    const uint16_t* X = a.x + ((((int64_t)(l * 2 + 0) * a.B + b) * a.H + h) * a.T + tg * Gt) * d;
    for (int t = warp; t < Gt; t += kRowWarps) {
#pragma unroll
        for (int k = 0; k < NR; k++) {
            uint32_t xb = X[(int64_t)t * d + lane + 32 * k];
            if (bf16_nonfinite(xb)) flag |= CG_FLAG_NONFINITE_INPUT;
            xs[lane + 32 * k] = bf16_bits_to_float(xb);
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < NR; k++) {
            const int c = lane + 32 * k, r = c / g, i = c - r * g;
            Zs[(size_t)t * d + c] = gauge_coord(Gs + r * g * g + i, g, xs + r * g, g);
        }
        __syncwarp();
    }
    __syncthreads();
    const int qmax = (1 << bits) - 1;
    const float qmaxf = (float)qmax;
    const int64_t bhl = (int64_t)b * a.H + h;
    for (int c = threadIdx.x; c < d; c += kRowThreads) {
        float mn = Zs[c], mx = Zs[c];
        for (int t = 1; t < Gt; t++) {
            const float v = Zs[(size_t)t * d + c];
            mn = fminf(mn, v);
            mx = fmaxf(mx, v);
        }
        const uint32_t sz = scale_zero(mn, mx, qmaxf, &flag);
        const float sc = h2f_bits(sz & 0xffffu), mz = h2f_bits(sz >> 16);
        uint8_t* st = stage + (size_t)c * pay;
        uint64_t acc = 0;
        int nacc = 0, nbytes = 0;
        for (int t = 0; t < Gt; t++) {
            acc |= (uint64_t)quant_code(Zs[(size_t)t * d + c], sc, mz, qmax) << nacc;
            nacc += bits;
            while (nacc >= 8) {
                st[nbytes++] = (uint8_t)(acc & 0xffu);
                acc >>= 8;
                nacc -= 8;
            }
        }
        a.scales[(int64_t)l * a.layer_scales + bhl * a.key_scales_per_bh + tg * d + c] = sz;
    }
    __syncthreads();
    uint32_t* dst = reinterpret_cast<uint32_t*>(a.codes + (int64_t)l * a.layer_codes + bhl * a.key_codes_per_bh +
                                                tg * (int64_t)d * pay);
    const uint32_t* src = reinterpret_cast<const uint32_t*>(stage);
    for (int w = threadIdx.x; w < d * pay / 4; w += kRowThreads) dst[w] = src[w];
    if (flag) raise_flag(a.status, flag);
}

template <int NR>
__global__ void __launch_bounds__(kRowThreads) key_decode_kernel(KeyArgs a) {
    constexpr int d = NR * 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int g = a.g, Gt = a.Gt, bits = a.bits;
    const int pay = Gt * bits / 8;
    float* Gs = reinterpret_cast<float*>(smem);                      // untransposed
    float* Zs = reinterpret_cast<float*>(smem + (size_t)d * g * 4);  // [Gt][d]
    uint8_t* stage = reinterpret_cast<uint8_t*>(Zs + (size_t)Gt * d);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    const int64_t tg = blockIdx.x;
    const int bh = blockIdx.y % (a.B * a.H), l = blockIdx.y / (a.B * a.H);
    const int b = bh / a.H, h = bh % a.H;
    const int64_t bhl = (int64_t)b * a.H + h;
    const float* Gsrc = a.G + ((int64_t)(l * 2 + 0) * a.H + h) * (int64_t)d * g;
    for (int e = threadIdx.x; e < d * g; e += kRowThreads) Gs[e] = __ldg(Gsrc + e);
    const uint32_t* src = reinterpret_cast<const uint32_t*>(a.codes + (int64_t)l * a.layer_codes +
                                                            bhl * a.key_codes_per_bh + tg * (int64_t)d * pay);
    uint32_t* stw = reinterpret_cast<uint32_t*>(stage);
    for (int w = threadIdx.x; w < d * pay / 4; w += kRowThreads) stw[w] = src[w];
    __syncthreads();
    for (int c = threadIdx.x; c < d; c += kRowThreads) {
        const uint32_t sz = a.scales[(int64_t)l * a.layer_scales + bhl * a.key_scales_per_bh + tg * d + c];
        const float sc = h2f_bits(sz & 0xffffu), mz = h2f_bits(sz >> 16);
        const uint8_t* st = stage + (size_t)c * pay;
        for (int t = 0; t < Gt; t++) {
            const int p = t * bits;
            uint32_t v = st[p >> 3] >> (p & 7);
            if ((p & 7) + bits > 8) v |= (uint32_t)st[(p >> 3) + 1] << (8 - (p & 7));
            v &= (1u << bits) - 1u;
            Zs[(size_t)t * d + c] = fmaf((float)v, sc, mz);
        }
    }
    __syncthreads();
    uint16_t* O = a.out + ((((int64_t)(l * 2 + 0) * a.B + b) * a.H + h) * a.T + tg * Gt) * d;
    for (int t = warp; t < Gt; t += kRowWarps) {
        const float* zr = Zs + (size_t)t * d;
#pragma unroll
        for (int k = 0; k < NR; k++) {
            const int c = lane + 32 * k, r = c / g, i = c - r * g;
            const float acc = gauge_coord(Gs + r * g * g + i, g, zr + r * g, g);
            O[(int64_t)t * d + c] = __bfloat16_as_ushort(__float2bfloat16_rn(acc));
        }
    }
}

__global__ void residual_copy_kernel(ResidArgs a) {
    const int64_t n16 = (a.T - a.nq) * a.d * 2 / 16;  // 16-byte chunks per unit
    for (int64_t u = blockIdx.y; u < a.units; u += gridDim.y) {
        const uint4* src;
        uint4* dst;
        if (a.to_residual) {
            src = reinterpret_cast<const uint4*>(a.src + (u * a.T + a.nq) * a.d);
            dst = reinterpret_cast<uint4*>(a.dst + u * (a.T - a.nq) * a.d);
        } else {
            src = reinterpret_cast<const uint4*>(a.src + u * (a.T - a.nq) * a.d);
            dst = reinterpret_cast<uint4*>(a.dst + (u * a.T + a.nq) * a.d);
        }
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += (int64_t)gridDim.x * blockDim.x)
            dst[i] = src[i];
    }
}

__global__ void __launch_bounds__(256) row_move_kernel(MoveArgs a) {
    const int64_t c16 = a.d / 8;  // 16-byte chunks per token row
    const int64_t rows = a.t_hi - a.t_lo;
    const int64_t n = a.units * rows * c16;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t u = i / (rows * c16), rem = i - u * rows * c16;
        const int64_t t = a.t_lo + rem / c16, c = rem % c16;
        const uint16_t* src = t < a.src_split ? a.ring_src + (u * a.W + t % a.W) * a.d
                                              : a.x + (u * a.T_x + (t - a.x_t0)) * a.d;
        uint16_t* dst = a.dst_ring ? a.dst + (u * a.W + t % a.W) * a.d : a.dst + (u * a.dst_T + (t - a.dst_t0)) * a.d;
        reinterpret_cast<uint4*>(dst)[c] = reinterpret_cast<const uint4*>(src)[c];
    }
}

}  // namespace

cudaError_t launch_row_move(const MoveArgs& a, cudaStream_t st) {
    const int64_t n = a.units * (a.t_hi - a.t_lo) * (a.d / 8);
    if (n <= 0) return cudaSuccess;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    row_move_kernel<<<(unsigned)blocks, 256, 0, st>>>(a);
    return cudaGetLastError();
}

// Warps per CTA of the tile encode kernel: as many as shared memory holds, at most 16.
static int tile_simt_warps(int d, int g) {
    if (!(d == 32 || d == 64 || d == 128 || d == 256)) return 0;
    const size_t gbytes = (size_t)d * g * 4;
    if (gbytes >= kSmemOptIn) return 0;
    const size_t n = (kSmemOptIn - gbytes) / tile_warp_bytes(d);
    return n < (size_t)kTileWarpsMax ? (int)n : kTileWarpsMax;
}

size_t tile_simt_smem(int d, int g) {
    const int nw = tile_simt_warps(d, g);
    return nw < 1 ? 0 : (size_t)d * g * 4 + (size_t)nw * tile_warp_bytes(d);
}

size_t key_simt_smem(int d, int g, int Gt, int bits) {
    if (!(d == 32 || d == 64 || d == 128 || d == 256)) return 0;
    size_t pay = (size_t)Gt * bits / 8;
    size_t enc = (size_t)d * g * 4 + (size_t)Gt * d * 4 + (size_t)kRowWarps * d * 4 + (size_t)d * pay;
    return enc;
}

// Rows per CTA: a multiple of what its warps take at once, so that the grid has about four CTAs for
// each one that is resident (a CTA stages the whole gauge set, so more rows amortize it; fewer leave
// SMs idle at the end), at most 512.
template <int NR>
static int row_simt_rows(const RowArgs& a, int64_t units) {
    using C = RowCfg<NR>;
    const int64_t step = C::kWarps * C::kRows, rows = (int64_t)a.B * a.t_count;
    int64_t per = (rows * units + 4 * 304 - 1) / (4 * 304);
    per = (per + step - 1) / step * step;
    return (int)(per < step ? step : (per > 512 ? 512 : per));
}

template <int NR>
static cudaError_t row_simt_nr(const RowArgs& a, bool enc, cudaStream_t st) {
    using C = RowCfg<NR>;
    const size_t smem = (size_t)C::d * (a.g + 4) * 4 + (size_t)C::kWarps * C::kWarpBytes;
    const auto kernel = enc ? row_encode_kernel<NR> : row_decode_kernel<NR>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t units = (int64_t)a.L * a.s_n * a.H, rows = (int64_t)a.B * a.t_count;
    const int per = row_simt_rows<NR>(a, units);
    dim3 grid((unsigned)((rows + per - 1) / per), (unsigned)units);
    kernel<<<grid, C::kThreads, smem, st>>>(a, per);
    return cudaGetLastError();
}

template <int NR>
static cudaError_t tile_encode_nr(const RowArgs& a, cudaStream_t st) {
    const int nwarps = tile_simt_warps(a.d, a.g);
    const size_t smem = tile_simt_smem(a.d, a.g);
    if (nwarps < 1) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(tile_encode_kernel<NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // two tiles per warp per CTA; the tiles of one (l, s, h) spread over grid.x
    const int64_t tiles = (int64_t)a.B * ((a.t_count + kTileTokens - 1) / kTileTokens);
    int64_t gx = (tiles + 2 * nwarps - 1) / (2 * nwarps);
    if (gx > 65535) gx = 65535;
    dim3 grid((unsigned)gx, (unsigned)(a.L * a.s_n * a.H));
    tile_encode_kernel<NR><<<grid, nwarps * 32, smem, st>>>(a);
    return cudaGetLastError();
}

template <int NR>
static cudaError_t key_encode_nr(const KeyArgs& a, cudaStream_t st) {
    size_t smem = key_simt_smem(a.d, a.g, a.Gt, a.bits);
    cudaError_t e = cudaFuncSetAttribute(key_encode_kernel<NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)(a.nq / a.Gt), (unsigned)(a.L * a.B * a.H));
    key_encode_kernel<NR><<<grid, kRowThreads, smem, st>>>(a);
    return cudaGetLastError();
}

template <int NR>
static cudaError_t key_decode_nr(const KeyArgs& a, cudaStream_t st) {
    size_t smem = key_simt_smem(a.d, a.g, a.Gt, a.bits);
    cudaError_t e = cudaFuncSetAttribute(key_decode_kernel<NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)(a.nq / a.Gt), (unsigned)(a.L * a.B * a.H));
    key_decode_kernel<NR><<<grid, kRowThreads, smem, st>>>(a);
    return cudaGetLastError();
}

#define CG_NR_SWITCH(FN, d, ...)                      \
    switch ((d) / 32) {                               \
        case 1: return FN<1>(__VA_ARGS__);            \
        case 2: return FN<2>(__VA_ARGS__);            \
        case 4: return FN<4>(__VA_ARGS__);            \
        case 8: return FN<8>(__VA_ARGS__);            \
        default: return cudaErrorInvalidValue;        \
    }

cudaError_t launch_row_encode_simt(const RowArgs& a, cudaStream_t st) { CG_NR_SWITCH(row_simt_nr, a.d, a, true, st) }
cudaError_t launch_row_decode_simt(const RowArgs& a, cudaStream_t st) { CG_NR_SWITCH(row_simt_nr, a.d, a, false, st) }
cudaError_t launch_tile_encode_simt(const RowArgs& a, cudaStream_t st) { CG_NR_SWITCH(tile_encode_nr, a.d, a, st) }

cudaError_t launch_key_encode_simt(const KeyArgs& a, cudaStream_t st) { CG_NR_SWITCH(key_encode_nr, a.d, a, st) }
cudaError_t launch_key_decode_simt(const KeyArgs& a, cudaStream_t st) { CG_NR_SWITCH(key_decode_nr, a.d, a, st) }

cudaError_t launch_residual_copy(const ResidArgs& a, cudaStream_t st) {
    const int64_t n16 = (a.T - a.nq) * a.d * 2 / 16;
    if (n16 <= 0 || a.units <= 0) return cudaSuccess;
    unsigned gx = (unsigned)((n16 + 255) / 256);
    if (gx > 1024) gx = 1024;
    dim3 grid(gx, (unsigned)(a.units < 65535 ? a.units : 65535));
    residual_copy_kernel<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace cg
