// cg_attn.cu -- attention of one decoding query per sequence, straight from the packed codes of
// a block-uniform cache: the recovered cache of Sec. 3 consumed by softmax attention (Fig. 1),
// with the inverse gauge folded out of the token loop (Sec. 3 notes that recovery can be folded
// into the surrounding computation).
//
// For KV head h and one of its n_rep query heads (grouped queries):
//   scores  q . khat_t = q . (G_K^T zhat_t) = (G_K q) . zhat_t: the query is rotated once into
//           gauge space and dotted with the dequantized codes;
//   values  sum_t p_t vhat_t = G_V^T (sum_t p_t zhat_t): the weighted sum stays in gauge space
//           and is rotated once per query at the end.
// The token loop reads only codes and scales (no bf16 cache is written or read).
//
// Kernels: attn_query_kernel (q' = scale * G_K q); a chunk kernel that writes, per (l, b, h) and
// part, the part's softmax max (base-2 logarithm), sum and gauge-space weighted value sum:
// attn_stream_kernel for 2-, 4- and 8-bit codes (both contractions on mma.sync, one warp per token
// stream), attn_chunk_kernel for 3- and 6-bit codes, whose code pairs straddle words (one
// 128-token chunk per CTA, all on CUDA cores); attn_combine_kernel (merges the parts, applies
// G_V^T).
#include "cg_launch.h"
#include "cg_sm100.cuh"
#include "cg_tc_common.cuh"

namespace cg {
namespace {

using namespace sm100;

constexpr int kAD = 128;           // head dim served
constexpr int kAThreads = 256;
constexpr int kASlices = kAThreads / 16;  // value phase: 16 channel octets x 16 token slices

// f = 1 + code * 2^-BITS for code c of a row held in registers (c known at compile time).
template <int BITS>
__device__ __forceinline__ float code_f(const uint32_t* w, int c) {
    const int bit = c * BITS, wi = bit >> 5, sh = bit & 31;
    uint32_t v = w[wi] >> sh;
    if (sh + BITS > 32) v |= w[wi + 1] << (32 - sh);
    return __uint_as_float(0x3F800000u | ((v & ((1u << BITS) - 1u)) << (23 - BITS)));
}

__device__ __forceinline__ float half_lo(uint32_t v) { return h2f_bits(v & 0xffffu); }
__device__ __forceinline__ float half_hi(uint32_t v) { return h2f_bits(v >> 16); }

constexpr int kQueries = 8;  // queries per CTA of the query rotation
constexpr int kQThreads = 256;
constexpr float kLog2e = 1.4426950408889634f;

// q' = scale * G_K q for kQueries queries of one (l, h). The gauge set is staged with rows padded by
// 16 bytes (coalesced loads, conflict-free 16-byte row reads); a thread owns one output channel and
// half of the queries, so one gauge value read from shared memory serves four of them.
__global__ void __launch_bounds__(kQThreads) attn_query_kernel(AttnArgs a) {
    extern __shared__ __align__(16) float Gs[];  // [128][g + 4], then [kQueries][128] queries
    const int g = a.g, gp = g + 4;
    float* qs = Gs + kAD * gp;
    const int l = blockIdx.x / a.H, h = blockIdx.x - l * a.H;
    const int n_all = a.B * a.n_rep;  // queries of this (l, h), sequence-major
    const int q_lo = blockIdx.y * kQueries;
    const int nq = n_all - q_lo < kQueries ? n_all - q_lo : kQueries;
    asm volatile("griddepcontrol.launch_dependents;");  // the stream kernel may take free slots and start its copies
    const float4* Gsrc = reinterpret_cast<const float4*>(a.G + ((int64_t)(l * 2 + 0) * a.H + h) * (int64_t)kAD * g);
    const int lg = 29 - __clz(g);  // log2(g / 4)
#pragma unroll 8
    for (int e = threadIdx.x; e < kAD * g / 4; e += kQThreads)
        *reinterpret_cast<float4*>(Gs + (e >> lg) * gp + 4 * (e & (g / 4 - 1))) = __ldg(Gsrc + e);
    const int i = threadIdx.x & (kAD - 1), half = threadIdx.x >> 7;
    auto row_of = [&](int k) -> int64_t {  // first element of query q_lo + k
        const int b = (q_lo + k) / a.n_rep, rq = (q_lo + k) - b * a.n_rep;
        return ((((int64_t)l * a.B + b) * a.H + h) * a.n_rep + rq) * kAD;
    };
#pragma unroll
    for (int k = 0; k < kQueries / 2; k++) {
        const int q = half * (kQueries / 2) + k;
        qs[q * kAD + i] = q < nq ? bf16_bits_to_float(a.q[row_of(q) + i]) : 0.0f;
    }
    __syncthreads();
    const float4* row = reinterpret_cast<const float4*>(Gs + i * gp);
    const float* x0 = qs + half * (kQueries / 2) * kAD + (i & ~(g - 1));
    float acc[kQueries / 2] = {};
#pragma unroll 4
    for (int j = 0; j < g / 4; j++) {
        const float4 gv = row[j];
#pragma unroll
        for (int k = 0; k < kQueries / 2; k++) {
            const float4 x = *reinterpret_cast<const float4*>(x0 + k * kAD + 4 * j);
            acc[k] = fmaf(gv.x, x.x, acc[k]);
            acc[k] = fmaf(gv.y, x.y, acc[k]);
            acc[k] = fmaf(gv.z, x.z, acc[k]);
            acc[k] = fmaf(gv.w, x.w, acc[k]);
        }
    }
#pragma unroll
    for (int k = 0; k < kQueries / 2; k++) {
        const int q = half * (kQueries / 2) + k;
        if (q < nq) a.qrot[row_of(q) + i] = a.scale * acc[k];
    }
}

// Deterministic block reduction of NV values per thread (sum or max) over NT threads, result
// in out[NV].
template <int NV, bool MAX, int NT>
__device__ __forceinline__ void block_reduce_n(float (&v)[NV], float* scratch, float* out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; k++)
        for (int off = 16; off >= 1; off >>= 1) {
            const float o = __shfl_xor_sync(0xffffffffu, v[k], off);
            v[k] = MAX ? fmaxf(v[k], o) : v[k] + o;
        }
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; k++) scratch[warp * NV + k] = v[k];
    __syncthreads();
    if (threadIdx.x < NV) {
        float r = scratch[threadIdx.x];
        for (int w = 1; w < NT / 32; w++) {
            const float o = scratch[w * NV + threadIdx.x];
            r = MAX ? fmaxf(r, o) : r + o;
        }
        out[threadIdx.x] = r;
    }
    __syncthreads();
}

template <int NV, bool MAX>
__device__ __forceinline__ void block_reduce(float (&v)[NV], float* scratch, float* out) {
    block_reduce_n<NV, MAX, kAThreads>(v, scratch, out);
}

template <int BITS, int NREP>
__global__ void __launch_bounds__(kAThreads) attn_chunk_kernel(AttnArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    float* qs = reinterpret_cast<float*>(smem);                  // [NREP][128] q'
    float* c32 = qs + NREP * kAD;                                // [NREP][4] sums of q' per 32 channels
    float* mx = c32 + NREP * 4;                                  // [NREP] chunk max
    float* sm = mx + NREP;                                       // [NREP] chunk sum of exp
    float* Wr = sm + NREP;                                       // [NREP][4] sum_t p s_V per block
    float* Zr = Wr + NREP * 4;                                   // [NREP][4] sum_t p m_V per block
    float* scratch = Zr + NREP * 4;                              // [8 warps][NREP * 4]
    uint32_t* SV = reinterpret_cast<uint32_t*>(scratch + 8 * NREP * 4);  // [chunk][4] value scales
    float* P = reinterpret_cast<float*>(SV + kAttnChunk * 4);    // [NREP][chunk] scores, then p;
                                                                 // later [16][NREP][128] partial sums
    const int tid = threadIdx.x;
    const int unit = blockIdx.y;
    const int l = unit / (a.B * a.H), bh = unit - l * a.B * a.H, b = bh / a.H, h = bh - (bh / a.H) * a.H;
    const int64_t c0 = (int64_t)blockIdx.x * kAttnChunk;
    const int n_tok = a.T - c0 < kAttnChunk ? (int)(a.T - c0) : kAttnChunk;
    const int blk = a.blk, nb = kAD / blk;
    constexpr float kTwoB = (float)(1 << BITS);

    for (int e = tid; e < NREP * kAD; e += kAThreads) qs[e] = a.qrot[(int64_t)unit * NREP * kAD + e];
    __syncthreads();
    if (tid < NREP * 4) {
        const float* src = qs + (tid >> 2) * kAD + (tid & 3) * 32;
        float s = 0.0f;
        for (int k = 0; k < 32; k++) s += src[k];
        c32[tid] = s;
    }
    __syncthreads();

    // scores: one token per thread, its packed key row in registers
    for (int tt = tid; tt < n_tok; tt += kAThreads) {
        const int64_t t = c0 + tt;
        const uint4* row = reinterpret_cast<const uint4*>(a.codes + a.cmap.at(l, 0, b, h, t));
        uint32_t w[4 * BITS + 1];
#pragma unroll
        for (int k = 0; k < BITS; k++) {
            const uint4 v = __ldg(row + k);
            w[4 * k] = v.x;
            w[4 * k + 1] = v.y;
            w[4 * k + 2] = v.z;
            w[4 * k + 3] = v.w;
        }
        w[4 * BITS] = 0u;
        const uint32_t* sk = a.scales + a.smap.at(l, 0, b, h, t);
        uint32_t sz[4];
#pragma unroll
        for (int k = 0; k < 4; k++) sz[k] = k < nb ? __ldg(sk + k) : 0u;
        float acc[NREP][4];
#pragma unroll
        for (int r = 0; r < NREP; r++)
#pragma unroll
            for (int k = 0; k < 4; k++) acc[r][k] = 0.0f;
#pragma unroll
        for (int c = 0; c < kAD; c++) {
            const float f = code_f<BITS>(w, c);
#pragma unroll
            for (int r = 0; r < NREP; r++) acc[r][c >> 5] = fmaf(qs[r * kAD + c], f, acc[r][c >> 5]);
        }
#pragma unroll
        for (int r = 0; r < NREP; r++) {
            float s = 0.0f;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const uint32_t z = sz[(32 * k) / blk];
                s += half_lo(z) * kTwoB * (acc[r][k] - c32[r * 4 + k]) + half_hi(z) * c32[r * 4 + k];
            }
            P[r * kAttnChunk + tt] = s;
        }
    }
    __syncthreads();

    // chunk softmax, and the per-block sums of p s_V and p m_V
    {
        float v[NREP];
#pragma unroll
        for (int r = 0; r < NREP; r++) {
            v[r] = -INFINITY;
            for (int tt = tid; tt < n_tok; tt += kAThreads) v[r] = fmaxf(v[r], P[r * kAttnChunk + tt]);
        }
        block_reduce<NREP, true>(v, scratch, mx);
        float ws[NREP * 4], zs[NREP * 4], es[NREP];
#pragma unroll
        for (int k = 0; k < NREP * 4; k++) ws[k] = zs[k] = 0.0f;
#pragma unroll
        for (int r = 0; r < NREP; r++) es[r] = 0.0f;
        for (int tt = tid; tt < n_tok; tt += kAThreads) {
            const int64_t t = c0 + tt;
            const uint32_t* sv = a.scales + a.smap.at(l, 1, b, h, t);
            uint32_t z[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                z[k] = k < nb ? __ldg(sv + k) : 0u;
                SV[tt * 4 + k] = z[k];
            }
#pragma unroll
            for (int r = 0; r < NREP; r++) {
                const float p = __expf(P[r * kAttnChunk + tt] - mx[r]);
                P[r * kAttnChunk + tt] = p;
                es[r] += p;
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    ws[r * 4 + k] = fmaf(p, half_lo(z[k]), ws[r * 4 + k]);
                    zs[r * 4 + k] = fmaf(p, half_hi(z[k]), zs[r * 4 + k]);
                }
            }
        }
        block_reduce<NREP, false>(es, scratch, sm);
        block_reduce<NREP * 4, false>(ws, scratch, Wr);
        block_reduce<NREP * 4, false>(zs, scratch, Zr);
    }

    // values: thread = (8 channels, token slice); sum_t (p s_V) f per channel
    const int oct = tid & 15, sl = tid >> 4;
    const int bk = (8 * oct) / blk;
    float acc[NREP][8];
#pragma unroll
    for (int r = 0; r < NREP; r++)
#pragma unroll
        for (int k = 0; k < 8; k++) acc[r][k] = 0.0f;
    {
        const int bit0 = 8 * oct * BITS, wi = bit0 >> 5, sh = bit0 & 31;
        const bool two = sh + 8 * BITS > 32;
        for (int tt = sl; tt < n_tok; tt += kASlices) {
            const uint32_t* row = reinterpret_cast<const uint32_t*>(a.codes + a.cmap.at(l, 1, b, h, c0 + tt));
            const uint32_t w0 = __ldg(row + wi);
            const uint32_t w1 = two ? __ldg(row + wi + 1) : 0u;
            const uint32_t w2 = (BITS == 8 && sh) ? __ldg(row + wi + 2) : 0u;
            const uint64_t v = ((((uint64_t)w1 << 32) | w0) >> sh) | (sh ? ((uint64_t)w2 << (64 - sh)) : 0ull);
            const float s_v = half_lo(SV[tt * 4 + bk]);
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const uint32_t q = (uint32_t)(v >> (k * BITS)) & ((1u << BITS) - 1u);
                const float f = __uint_as_float(0x3F800000u | (q << (23 - BITS)));
#pragma unroll
                for (int r = 0; r < NREP; r++) acc[r][k] = fmaf(P[r * kAttnChunk + tt] * s_v, f, acc[r][k]);
            }
        }
    }
    __syncthreads();  // all reads of P done: its space now holds the slice sums
    float* red = P;   // [16][NREP][128]
#pragma unroll
    for (int r = 0; r < NREP; r++)
#pragma unroll
        for (int k = 0; k < 8; k++) red[(sl * NREP + r) * kAD + 8 * oct + k] = acc[r][k];
    __syncthreads();
    float* part = a.part + ((int64_t)unit * a.n_parts + blockIdx.x) * NREP * (kAD + 2);
    for (int e = tid; e < NREP * kAD; e += kAThreads) {
        const int r = e / kAD, c = e - r * kAD, k = c / blk;
        float s = 0.0f;
        for (int q = 0; q < kASlices; q++) s += red[(q * NREP + r) * kAD + c];
        part[r * (kAD + 2) + 2 + c] = kTwoB * (s - Wr[r * 4 + k]) + Zr[r * 4 + k];
    }
    if (tid < NREP) {
        part[tid * (kAD + 2)] = mx[tid] * kLog2e;
        part[tid * (kAD + 2) + 1] = sm[tid];
    }
}

constexpr int kCParts = 256;     // parts whose weights are held at a time

// Merges the parts of one (l, b, h) and applies G_V^T (per gauge group): out fp32. It waits for
// memory, not arithmetic: the parts' maxima, sums and weights are taken one per thread, so that the
// loop over the parts only loads their value sums, 4 n_rep of a thread in flight; a slice's gauge
// values are loaded first. 8 units of 57 parts: 17 -> 6 us. Threads: 128 channels x SL slices of the parts and
// of the rotation (launch_combine).
template <int NREP, int SL>
__global__ void __launch_bounds__(SL * kAD) attn_combine_kernel(AttnArgs a) {
    constexpr int kCThreads = SL * kAD;
    __shared__ float red[SL][NREP][kAD], zs[NREP][kAD], Mw[kCThreads / 32][NREP], Lw[kCThreads / 32][NREP];
    __shared__ float wgt[kCParts][NREP];
    const int unit = blockIdx.x, tid = threadIdx.x, c = tid & (kAD - 1), sl = tid >> 7, lane = tid & 31;
    const int l = unit / (a.B * a.H), h = unit % a.H;
    const int g = a.g, grp = c / g, i = c - grp * g;
    constexpr int kStride = NREP * (kAD + 2);
    const float* part = a.part + (int64_t)unit * a.n_parts * kStride;
    const int n_parts = (int)(((unit + 1) * a.unit_steps - 1) / a.cta_steps - unit * a.unit_steps / a.cta_steps) + 1;
    const int per = g / SL;  // g >= 8: gauge rows of this slice
    const float* Gv = a.G + ((int64_t)(l * 2 + 1) * a.H + h) * (int64_t)kAD * g + (int64_t)grp * g * g + (int64_t)sl * per * g + i;
    float gv[32];
#pragma unroll
    for (int j = 0; j < 32; j++) gv[j] = j < per ? __ldg(Gv + (int64_t)j * g) : 0.0f;
    auto slices = [&](int r, int k) -> float {
        if constexpr (SL == 1) return red[0][r][k];
        else return (red[0][r][k] + red[1][r][k]) + (red[2][r][k] + red[3][r][k]);
    };
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the parts
    float m = -INFINITY;  // thread: query tid mod NREP
    for (int e = tid; e < n_parts * NREP; e += kCThreads) m = fmaxf(m, part[(int64_t)e * (kAD + 2)]);
#pragma unroll
    for (int off = 16; off >= NREP; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if (lane < NREP) Mw[tid >> 5][lane] = m;
    __syncthreads();
    m = Mw[0][tid % NREP];
#pragma unroll
    for (int w = 1; w < kCThreads / 32; w++) m = fmaxf(m, Mw[w][tid % NREP]);
    float o[NREP] = {}, ls = 0.0f;
    for (int j0 = 0; j0 < n_parts; j0 += kCParts) {
        const int n = n_parts - j0 < kCParts ? n_parts - j0 : kCParts;
        const float* p0 = part + (int64_t)j0 * kStride;
        for (int e = tid; e < n * NREP; e += kCThreads) {
            const float2 ml = *reinterpret_cast<const float2*>(p0 + (int64_t)e * (kAD + 2));
            const float w = exp2f(ml.x - m);
            wgt[e / NREP][tid % NREP] = w;
            ls = fmaf(ml.y, w, ls);
        }
        __syncthreads();
#pragma unroll 4
        for (int j = sl; j < n; j += SL)
#pragma unroll
            for (int r = 0; r < NREP; r++) o[r] = fmaf(p0[(int64_t)j * kStride + r * (kAD + 2) + 2 + c], wgt[j][r], o[r]);
        __syncthreads();
    }
#pragma unroll
    for (int off = 16; off >= NREP; off >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, off);
    if (lane < NREP) Lw[tid >> 5][lane] = ls;
#pragma unroll
    for (int r = 0; r < NREP; r++) red[sl][r][c] = o[r];
    __syncthreads();
    for (int e = tid; e < NREP * kAD; e += kCThreads) {
        const int r = e / kAD, k = e % kAD;
        float s = 0.0f;
#pragma unroll
        for (int w = 0; w < kCThreads / 32; w++) s += Lw[w][r];
        zs[r][k] = slices(r, k) / s;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < NREP; r++) {
        const float* z = zs[r] + grp * g + sl * per;
        float s = 0.0f;
#pragma unroll
        for (int j = 0; j < 32; j++)
            if (j < per) s = fmaf(gv[j], z[j], s);
        if constexpr (SL == 1)
            for (int j = 32; j < per; j++) s = fmaf(__ldg(Gv + (int64_t)j * g), z[j], s);
        red[sl][r][c] = s;
    }
    __syncthreads();
    for (int e = tid; e < NREP * kAD; e += kCThreads) {
        const int r = e / kAD, k = e % kAD;
        a.out[((int64_t)unit * NREP + r) * kAD + k] = slices(r, k);
    }
}

// ------------------------------------------------------------------------------------
// 2-, 4- and 8-bit codes: both contractions on tensor cores (mma.sync m16n8k16, fp16 in, fp32
// accumulate) straight from the packed words. The codes are the 16-row operand, the queries the
// 8-column one: up to four queries bring their high parts as columns 0..3 and their low parts as
// columns 4..7 of the same MMA; eight queries (Q8) take two MMAs. A code enters as the fp16
// subnormal q 2^(s - 24) (the bits of q in the mantissa, s its offset in the half word), which is
// exact; the factor 2^s is divided out of the other operand or of the result.
//   scores  D[token][query] = sum_c q_tc q'_c per quantization block: a register of the code operand
//           is two channels of one token;
//           S = sum_blocks s (D + off (C'' - C)) + m C, C = sum_c q'_c over the block.
//   values  O[channel][query] = sum_t q_tc w_t with w = p s_V: a register of the code operand is one
//           channel of two tokens (a byte permute per word and half); the weights leave the score
//           MMA as rows of tokens and become its operand by one 8x8 transpose (movmatrix);
//           sum_t p m_V is kept per block and added at the end.
// High + low carry 22 bits (w: of the value, scaled step by step; q': of hi + lo). For 2- and 4-bit codes q' is its bf16
// hi + lo pair (16 bits) and a quarter of the rest, and off = 2^b: the operands (2^b + q) against that
// pair in another form, so that results agree with those of the pair to 2e-5, with a smaller error
// (against fp64, 8 heads of 32,767 / 4,000 / 700 tokens at 4 bits: the pair as bf16 operands 1.83, 1.26,
// 1.28e-5; the pair here, with the codes' truncation, 1.94, 1.42, 1.37e-5; with a quarter of the rest 1.52, 1.15, 1.08e-5).
// For 8-bit codes q' is the fp32 value and off = 0.
// The MMA accumulators hold one step's tokens only and are added to fp32 sums in registers (rounded
// to nearest), so the tensor core's own accumulation covers at most 64 tokens.
// One warp per token stream: it has its own buffers in shared memory, its own online softmax, and
// meets the other three warps of its CTA only for the queries and at the end of the part. The next
// step's key codes are copied (bulk) while this step's values are summed, its value codes during
// the next scores; scales go through registers a step ahead (they have no 16-byte alignment) and
// are stored as fp32 records that the packed arithmetic over two queries reads directly.
// Bound by instruction issue and the ALU pipe (about 20 warp instructions a token at 4 bits and two
// blocks per row, 7.5 of them unpacking; 87 in the kernel it replaced, whose value sums ran on CUDA
// cores; with the queries as the 16-row operand instead, twice the MMAs for four queries, 308 us
// against 298). One layer, 64 sequences x 8 heads x 16,384 tokens, 4 bits, 4 queries a head: whole
// call 1043 -> 268 us (stream kernel 243 us, 5.0 TB/s, 73 % of measured HBM); one 32,767-token
// sequence at 8 bits 280 -> 42 us.
// ------------------------------------------------------------------------------------
constexpr int kSThreads = 128;
constexpr int kSWarps = kSThreads / 32;
constexpr int kSCtas = 3;  // per SM: 168 registers a thread, up to 46 bytes spilled (2 bits, four blocks, eight queries); four CTAs (128 registers) spill far more

template <int BITS, int NB>
struct StreamCfg {
    static constexpr int kTok = BITS == 8 ? 32 : 64;           // tokens of a step
    static constexpr int kRow = kAD * BITS / 8;                // packed token row
    static constexpr int kCodes = kTok * kRow;                 // one tensor's codes of a step
    static constexpr int kRecs = kTok * NB;                    // scale records {s, s, m, m} of a step
    static constexpr int kWarp = 2 * kCodes + 2 * kRecs * 16;  // a warp's K, V codes and K, V scales
    static constexpr int kBars = 128;                          // mbarriers and flags
    static constexpr int kQ = 8 * 32 * 16;                     // the score MMAs' query operand
    static constexpr int kStat = 8 * (2 * NB + 1) * 4;         // per query: C, off (C'' - C), unit
    static constexpr int kFixed = (kBars + kQ + kStat + 127) / 128 * 128;
    static constexpr int kTotal = kFixed + kSWarps * kWarp;
    static constexpr int kPass = NB == 1 ? 2 : NB;             // value passes: 16 / kPass channels each
    static constexpr int kVC = 16 / kPass;                     // codes per token, lane and pass
    static_assert(kWarp % 16 == 0 && kCodes % 16 == 0, "aligned parts");
    static_assert(kWarp >= 8 * (kAD + 2) * 4, "the merge reuses the buffers");
};

// Codes packed in half words: code i of a half word sits at bit BITS * i. It enters at a bit near the
// top of the fp16 mantissa (at most bits 2..9): the MMA aligns a subnormal's product by the lowest
// normal exponent, so a code left in the lowest mantissa bits loses the bits above it (4-bit codes in
// place: attention 5e-5 off instead of 2e-5, 2-bit ones 1.3e-4). Codes share a shift of the whole
// word where they can.
template <int BITS>
__device__ constexpr int code_shift(int i) {
    return BITS == 8 ? 2 : (BITS == 4 ? 4 : 6 + 2 * (i & 1));
}
template <int BITS>
__device__ __forceinline__ uint32_t code_pair(uint32_t x, int i) {
    constexpr uint32_t kM = ((1u << BITS) - 1u) * 0x10001u;
    const int up = code_shift<BITS>(i) - BITS * i;
    return (up >= 0 ? x << up : x >> -up) & (kM << code_shift<BITS>(i));
}

__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Transposes an 8x8 matrix of 16-bit values: lane (g, t) gives row g, columns 2t, 2t + 1 and gets
// row 2t, 2t + 1 of column g.
__device__ __forceinline__ uint32_t transpose8x8(uint32_t v) {
    uint32_t r;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
    return r;
}

__device__ __forceinline__ float ex2(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }

// (v0, v1) as fp16 high and low parts, each packed low half first.
__device__ __forceinline__ void split_f16(float v0, float v1, uint32_t& hi, uint32_t& lo) {
    const __half2 h = __floats2half2_rn(v0, v1);
    const float2 f = __half22float2(h);
    const float2 r = __fadd2_rn(make_float2(v0, v1), make_float2(-f.x, -f.y));
    const __half2 w = __floats2half2_rn(r.x, r.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&w);
}

__device__ __forceinline__ float2 scale_zero_of(uint32_t v) {
    return __half22float2(*reinterpret_cast<const __half2*>(&v));
}

template <int BITS, int NB, bool Q8>
__global__ void __launch_bounds__(kSThreads, kSCtas) attn_stream_kernel(AttnArgs a) {
    static_assert(BITS == 2 || BITS == 4 || BITS == 8, "codes that do not straddle half words");
    using C = StreamCfg<BITS, NB>;
    constexpr int kTok = C::kTok, kTiles = kTok / 16, kBlk = kAD / NB;
    constexpr int kKC = kBlk / 4;                            // key codes per token, lane and block
    constexpr int kLaneBits = BITS * kKC >= 32 ? 16 : 8;     // key pairs: half words, or bytes of one half word
    constexpr int kCL = kLaneBits / BITS;                    // codes per half word (byte)
    constexpr int kKX = kKC / (2 * kCL);                     // words per block
    constexpr int kKs = kKC / 4;                             // MMA steps per block
    constexpr int kPass = C::kPass, kVC = C::kVC;
    constexpr int kVBits = kVC * BITS;                       // value codes per token, lane and pass
    constexpr int kVL = kVBits >= 16 ? 16 / BITS : kVC;      // codes per half word
    constexpr int kVX = kVC / kVL;                           // half words
    constexpr int kItems = C::kRecs / 32;                    // scale records a lane prepares per tensor
    constexpr float kOff = BITS == 8 ? 0.0f : (float)(1 << BITS);
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem) + 2 * warp;  // this warp's K and V codes
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + 64) + 2 * warp;  // [1] stays 0 (drains)
    uint4* qb = reinterpret_cast<uint4*>(smem + C::kBars) + lane;   // [step][lane]: high b0, b1, low b0, b1
    float* stat = reinterpret_cast<float*>(smem + C::kBars + C::kQ);  // [query][C, off (C'' - C) per block, unit]
    unsigned char* kst = smem + C::kFixed + warp * C::kWarp;
    unsigned char* vst = kst + C::kCodes;
    float4* sf = reinterpret_cast<float4*>(vst + C::kCodes);  // [K, V][token][block]
    // row r of an 8-token matrix is token (r >> 1) + 4 (r & 1), so that the tokens a lane's value
    // operand takes (rows 2t, 2t + 1) are t and t + 4: fewer bank conflicts than neighbours
    const int tg = (g >> 1) + 4 * (g & 1);

    const int tsh = a.smap.tshift;
    // scale records of a lane: words lane_off + e_off of a step's rows of NB words, one row per token
    // or per 16-token tile
    const int lane_off = tsh ? (NB == 1 ? lane >> 4 : lane % NB) : lane;
    if (lane == 0) {
        abort_flag[0] = 0;
        abort_flag[1] = 0;
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        fence_barrier_init();
    }
    __syncwarp();
    uint32_t phase = 0;  // copies completed by this warp (K and V alike)
    bool dead = false;   // a wait of this warp ran out

    // this CTA's share of all units' steps: whole segments of one unit each, one part per segment
    int64_t pos = (int64_t)blockIdx.x * a.cta_steps;
    const int64_t pos_end = pos + a.cta_steps < a.all_steps ? pos + a.cta_steps : a.all_steps;
    while (pos < pos_end) {
    const int unit = (int)(pos / a.unit_steps);
    const int64_t in_unit = pos - unit * a.unit_steps;
    const int64_t seg = pos_end - pos < a.unit_steps - in_unit ? pos_end - pos : a.unit_steps - in_unit;
    const int slot = (int)(blockIdx.x - unit * a.unit_steps / a.cta_steps);
    pos += seg;
    const int l = unit / (a.B * a.H), bh = unit - l * a.B * a.H, b = bh / a.H, h = bh - (bh / a.H) * a.H;

    // tokens [lo, hi); a step of the CTA is kSWarps steps of kTok tokens, one per warp
    const int64_t lo = in_unit * (kSWarps * kTok);
    const int64_t hi = lo + seg * (kSWarps * kTok) < a.T ? lo + seg * (kSWarps * kTok) : a.T;
    const int steps_all = (int)((hi - lo + kTok - 1) / kTok);
    const int steps = steps_all > warp && !dead ? (steps_all - warp + kSWarps - 1) / kSWarps : 0;
    const uint8_t* kcodes = a.codes + a.cmap.at(l, 0, b, h, lo + warp * kTok);
    const uint8_t* vcodes = a.codes + a.cmap.at(l, 1, b, h, lo + warp * kTok);
    const uint32_t* ksc = a.scales + a.smap.at(l, 0, b, h, lo + warp * kTok) + lane_off;
    const uint32_t* vsc = a.scales + a.smap.at(l, 1, b, h, lo + warp * kTok) + lane_off;
    const int sc_step = ((kSWarps * kTok) >> tsh) * NB;  // scale words from one step of a warp to its next
    const int n_part = (int)(hi - lo);  // a part is shorter than 2^31 tokens

    auto step_tokens = [&](int i) -> int {
        const int left = n_part - (warp + i * kSWarps) * kTok;
        return left < kTok ? left : kTok;
    };
    auto load_codes = [&](int i, int which) {  // lane 0: K (0) or V (1) codes of step i
        const uint32_t bytes = (uint32_t)step_tokens(i) * C::kRow;
        mbar_arrive_expect_tx(&bars[which], bytes);
        bulk_load(which ? vst : kst, (which ? vcodes : kcodes) + (int64_t)i * (kSWarps * C::kCodes), bytes, &bars[which]);
    };
    uint32_t nsc[2][kItems];  // scales of a step: record r = (token, block)
    auto load_scales = [&](int i) {  // called for i = 0, 1, ... in turn
        const int n = step_tokens(i);
#pragma unroll
        for (int e = 0; e < kItems; e++) {
            const bool ok = n == kTok || (lane + 32 * e) / NB < n;  // tokens that do not exist: zero scale and zero
            const int at = tsh ? ((32 * e / NB) >> 4) * NB : 32 * e;
            nsc[0][e] = ok ? __ldg(ksc + at) : 0u;
            nsc[1][e] = ok ? __ldg(vsc + at) : 0u;
        }
        ksc += sc_step;
        vsc += sc_step;
    };
    if (steps > 0) {
        if (lane == 0) {
            load_codes(0, 0);
            load_codes(0, 1);
        }
        load_scales(0);
    }

    // Query operand of the scores: column g, this lane's channels (lane t: codes t * kKC .. of each
    // block); column g is query g (Q8: high and low operands), or query g & 3, high part for g < 4
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the rotated queries
    {
        const int qi = Q8 ? g : g & 3;
        const float* qrow = a.qrot + ((int64_t)unit * a.n_rep + qi) * kAD;
        auto value = [&](int ch) { return qi < a.n_rep ? qrow[ch] : 0.0f; };
        auto rounded = [&](float v) {  // the value the contraction sees
            if constexpr (BITS == 8) return v;
            const float hb = __bfloat162float(__float2bfloat16_rn(v));
            const float r = hb + __bfloat162float(__float2bfloat16_rn(v - hb));
            return fmaf(0.25f, v - r, r);
        };
        float amax = 0.0f, c1[NB], c2[NB];
#pragma unroll
        for (int k = 0; k < NB; k++) {
            c1[k] = c2[k] = 0.0f;
#pragma unroll 8
            for (int j = 0; j < kKC; j++) {
                const float v = value(k * kBlk + t * kKC + j), r = rounded(v);
                amax = fmaxf(amax, fabsf(r));
                c1[k] += v;
                c2[k] += r - v;
            }
#pragma unroll
            for (int off = 1; off < 4; off <<= 1) {
                c1[k] += __shfl_xor_sync(0xffffffffu, c1[k], off);
                c2[k] += __shfl_xor_sync(0xffffffffu, c2[k], off);
            }
        }
#pragma unroll
        for (int off = 1; off < 4; off <<= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
        // scaled by the power of two that takes the largest value into [2^14, 2^15)
        int E = (int)(__float_as_uint(amax) >> 23);
        E = E < 20 ? 20 : (E > 254 ? 254 : E);
        const float up = __uint_as_float((uint32_t)(268 - E) << 23);
        if (warp == 0 && t == 0 && (Q8 || g < 4)) {
            float* st = stat + qi * (2 * NB + 1);
#pragma unroll
            for (int k = 0; k < NB; k++) {  // in the unit of D, 2^24 / up
                st[2 * k] = c1[k] * up * 5.9604645e-08f;
                st[2 * k + 1] = kOff * c2[k] * up * 5.9604645e-08f;
            }
            // (at most 2^126: score differences beyond 2^102 leave a weight of 0 either way)
            st[2 * NB] = __uint_as_float((uint32_t)(E < 243 ? E + 10 : 253) << 23) * kLog2e;
        }
        for (int s = 2 * warp; s < 2 * warp + 2; s++) {  // two of the eight MMA steps per warp
            const int k = s / kKs, ks = s % kKs;
            uint32_t wh[2], wl[2];
#pragma unroll
            for (int hf = 0; hf < 2; hf++) {
                const int p = 2 * ks + hf, i = p % kCL, c0 = (p / kCL) * 2 * kCL + i;
                const float down = up * __uint_as_float((uint32_t)(127 - code_shift<BITS>(i)) << 23);
                const int ch = k * kBlk + t * kKC + c0;
                split_f16(rounded(value(ch)) * down, rounded(value(ch + kCL)) * down, wh[hf], wl[hf]);
            }
            if (Q8) {
                qb[32 * s] = make_uint4(wh[0], wh[1], wl[0], wl[1]);
            } else {
                const bool high = g < 4;
                qb[32 * s] = make_uint4(high ? wh[0] : wl[0], high ? wh[1] : wl[1], 0u, 0u);
            }
        }
    }
    __syncthreads();

    // this lane's score columns 2t, 2t + 1: queries q0, q0 + 1 (columns 4..7 without Q8: their low
    // parts, which take no C terms)
    const int q0 = Q8 ? 2 * t : 2 * (t & 1);
    const bool main_cols = Q8 || t < 2;
    float2 cblk[NB], eblk[NB], cF;
#pragma unroll
    for (int k = 0; k < NB; k++) {
        const float* s0 = stat + q0 * (2 * NB + 1) + 2 * k;
        cblk[k] = main_cols ? make_float2(s0[0], s0[2 * NB + 1]) : dup(0.0f);
        eblk[k] = main_cols ? make_float2(s0[1], s0[2 * NB + 2]) : dup(0.0f);
    }
    cF = make_float2(stat[q0 * (2 * NB + 1) + 2 * NB], stat[(q0 + 1) * (2 * NB + 1) + 2 * NB]);

    // columns 2t, 2t + 1: sums of w q over channels (code i of lane g's segment in pass p)
    float2 acc[kPass][kVC];
#pragma unroll
    for (int p = 0; p < kPass; p++)
#pragma unroll
        for (int i = 0; i < kVC; i++) acc[p][i] = dup(0.0f);
    float2 Mu = dup(-INFINITY), lsum = dup(0.0f), zsum[NB];
#pragma unroll
    for (int k = 0; k < NB; k++) zsum[k] = dup(0.0f);
    int kb = 0;  // acc carries a factor 2^kb, that of the last step's weights

    for (int it = 0; it < steps; it++) {
        const uint32_t par = (phase + (uint32_t)it) & 1u;
        const int n_tok = step_tokens(it);
        // The weights w = p s_V of a step take the factor 2^k that brings its largest finite value scale
        // into [2^14, 2^15) (subnormal ones below that): no w overflows fp16, and the pair of a weight is
        // off by at most 2^-23 of it or 2^-39 of that scale, whatever the scales of other steps are. The
        // sums follow by an exact power of two. (A factor from a stream's first step only, dropped when a
        // weight overflowed: up to 280 times the tests' tolerance after a prefix of zero scales; this rule
        // takes the same time or less, 62.5 -> 59.4 us for 32 x 8 x 4,000 tokens at 4 bits in one block.)
        int top = 0;
#pragma unroll
        for (int e = 0; e < kItems; e++) {
            const int x = (int)(nsc[1][e] & 0x7c00u);
            top = x == 0x7c00 ? top : max(top, x);
        }
        const int k2 = 29 - (__reduce_max_sync(0xffffffffu, top) >> 10);
        const float wup = __int_as_float((127 + k2) << 23), rescale = __int_as_float((127 + k2 - kb) << 23);
        kb = k2;
        // this step's scales to shared memory as fp32, the next step's on their way
#pragma unroll
        for (int s = 0; s < 2; s++)
#pragma unroll
            for (int e = 0; e < kItems; e++) {
                const float2 z = scale_zero_of(nsc[s][e]);
                const float f = s ? z.x * wup : z.x;
                sf[s * C::kRecs + lane + 32 * e] = make_float4(f, f, z.y, z.y);
            }
        if (it + 1 < steps) load_scales(it + 1);
        bool ok = mbar_wait(&bars[0], par, abort_flag, a.wait_ns);
        if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0) raise_flag(a.status, CG_FLAG_PIPE_TIMEOUT);
            mbar_wait(&bars[0], par, abort_flag + 1, tc::kWaitLimitNs);  // let the copies in flight land
            mbar_wait(&bars[1], par, abort_flag + 1, tc::kWaitLimitNs);
            dead = true;
            break;
        }
        __syncwarp();
        const float4* SK = sf + tg * NB;
        const float4* SV = sf + C::kRecs + tg * NB;

        // ---- scores: S[j][h] = tokens 16 j + 8 h + tg, two queries
        float2 S[kTiles][2];
#pragma unroll
        for (int j = 0; j < kTiles; j++) S[j][0] = S[j][1] = dup(0.0f);
#pragma unroll
        for (int k = 0; k < NB; k++) {
            uint32_t x[kTiles][2][kKX];
            float d[kTiles][4];
#pragma unroll
            for (int j = 0; j < kTiles; j++) {
#pragma unroll
                for (int hf = 0; hf < 2; hf++) {
                    const unsigned char* src = kst + (16 * j + 8 * hf + tg) * C::kRow + (k * kBlk + t * kKC) * BITS / 8;
                    uint32_t(&w)[kKX] = x[j][hf];
                    if constexpr (kLaneBits == 8) {
                        w[0] = __byte_perm(*reinterpret_cast<const uint16_t*>(src), 0u, 0x4140);
                    } else if constexpr (kKX % 4 == 0) {
#pragma unroll
                        for (int q = 0; q < kKX; q += 4) {
                            const uint4 v = reinterpret_cast<const uint4*>(src)[q / 4];
                            w[q] = v.x; w[q + 1] = v.y; w[q + 2] = v.z; w[q + 3] = v.w;
                        }
                    } else if constexpr (kKX == 2) {
                        const uint2 v = *reinterpret_cast<const uint2*>(src);
                        w[0] = v.x; w[1] = v.y;
                    } else {
                        w[0] = *reinterpret_cast<const uint32_t*>(src);
                    }
                }
                d[j][0] = d[j][1] = d[j][2] = d[j][3] = 0.0f;
            }
#pragma unroll
            for (int ks = 0; ks < kKs; ks++) {
                uint4 q;
                if constexpr (Q8) {
                    q = qb[32 * (k * kKs + ks)];
                } else {
                    const uint2 v = *reinterpret_cast<const uint2*>(&qb[32 * (k * kKs + ks)]);
                    q = make_uint4(v.x, v.y, 0u, 0u);
                }
                const int p0 = 2 * ks, p1 = 2 * ks + 1;
#pragma unroll
                for (int j = 0; j < kTiles; j++) {
                    const uint32_t a0 = code_pair<BITS>(x[j][0][p0 / kCL], p0 % kCL);
                    const uint32_t a1 = code_pair<BITS>(x[j][1][p0 / kCL], p0 % kCL);
                    const uint32_t a2 = code_pair<BITS>(x[j][0][p1 / kCL], p1 % kCL);
                    const uint32_t a3 = code_pair<BITS>(x[j][1][p1 / kCL], p1 % kCL);
                    mma_f16(d[j], a0, a1, a2, a3, q.x, q.y);
                    if constexpr (Q8) mma_f16(d[j], a0, a1, a2, a3, q.z, q.w);
                }
            }
#pragma unroll
            for (int j = 0; j < kTiles; j++)
#pragma unroll
                for (int hf = 0; hf < 2; hf++) {
                    const float4 z = SK[(16 * j + 8 * hf) * NB + k];
                    float2 u = make_float2(d[j][2 * hf], d[j][2 * hf + 1]);
                    if constexpr (BITS != 8) u = __fadd2_rn(u, eblk[k]);
                    S[j][hf] = __ffma2_rn(make_float2(z.z, z.w), cblk[k], S[j][hf]);
                    S[j][hf] = __ffma2_rn(make_float2(z.x, z.y), u, S[j][hf]);
                }
        }
        __syncwarp();  // all lanes have read the key codes
        if (lane == 0 && it + 1 < steps) load_codes(it + 1, 0);
        if constexpr (!Q8) {  // high + low columns
#pragma unroll
            for (int j = 0; j < kTiles; j++)
#pragma unroll
                for (int hf = 0; hf < 2; hf++)
                    S[j][hf] = __fadd2_rn(S[j][hf], make_float2(__shfl_xor_sync(0xffffffffu, S[j][hf].x, 2),
                                                                __shfl_xor_sync(0xffffffffu, S[j][hf].y, 2)));
        }
        if (n_tok < kTok) {
#pragma unroll
            for (int j = 0; j < kTiles; j++)
#pragma unroll
                for (int hf = 0; hf < 2; hf++)
                    if (16 * j + 8 * hf + tg >= n_tok) S[j][hf] = dup(-INFINITY);
        }

        // ---- online softmax of this warp's stream (the lanes of a column agree)
        float2 m = S[0][0];
#pragma unroll
        for (int j = 0; j < kTiles; j++)
#pragma unroll
            for (int hf = 0; hf < 2; hf++) {
                m.x = fmaxf(m.x, S[j][hf].x);
                m.y = fmaxf(m.y, S[j][hf].y);
            }
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) {
            m.x = fmaxf(m.x, __shfl_xor_sync(0xffffffffu, m.x, off));
            m.y = fmaxf(m.y, __shfl_xor_sync(0xffffffffu, m.y, off));
        }
        m.x = fmaxf(Mu.x, m.x);
        m.y = fmaxf(Mu.y, m.y);
        const float2 al = make_float2(ex2((Mu.x - m.x) * cF.x), ex2((Mu.y - m.y) * cF.y));  // 0 on the first step
        const float2 al_acc = make_float2(al.x * rescale, al.y * rescale);
        Mu = m;
        const float2 neg = make_float2(-m.x, -m.y);
        float2 l2 = dup(0.0f);
#pragma unroll
        for (int j = 0; j < kTiles; j++)
#pragma unroll
            for (int hf = 0; hf < 2; hf++) {
                // the difference first: it is exact near the maximum and never above 0, however large the scores
                // are (S cF less a rounded m cF is off by 2^-24 of it: NaN from scores of 2^23 on)
                const float2 e = __fmul2_rn(__fadd2_rn(S[j][hf], neg), cF);
                S[j][hf] = make_float2(ex2(e.x), ex2(e.y));
                l2 = __fadd2_rn(l2, S[j][hf]);
            }
        lsum = __ffma2_rn(lsum, al, l2);

        ok = mbar_wait(&bars[1], par, abort_flag, a.wait_ns);
        if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0) raise_flag(a.status, CG_FLAG_PIPE_TIMEOUT);
            mbar_wait(&bars[1], par, abort_flag + 1, tc::kWaitLimitNs);
            if (it + 1 < steps) mbar_wait(&bars[0], par ^ 1u, abort_flag + 1, tc::kWaitLimitNs);
            dead = true;
            break;
        }

        // ---- values: pass by pass (a pass lies in one block), 16 tokens per MMA
        uint32_t wb[kTiles][Q8 ? 4 : 2];  // weights: rows 0..7, 8..15 of the sixteen tokens (Q8: high, then low)
#pragma unroll
        for (int p = 0; p < kPass; p++) {
            const int k = NB == 1 ? 0 : p;
            if (NB > 1 || p == 0) {
                float2 z2 = dup(0.0f);
#pragma unroll
                for (int j = 0; j < kTiles; j++)
#pragma unroll
                    for (int hf = 0; hf < 2; hf++) {
                        const float4 z = SV[(16 * j + 8 * hf) * NB + k];
                        z2 = __ffma2_rn(S[j][hf], make_float2(z.z, z.w), z2);
                        const float2 w2 = __fmul2_rn(S[j][hf], make_float2(z.x, z.y));
                        uint32_t wh, wl;
                        split_f16(w2.x, w2.y, wh, wl);
                        if constexpr (Q8) {
                            wb[j][hf] = transpose8x8(wh);
                            wb[j][2 + hf] = transpose8x8(wl);
                        } else {
                            wb[j][hf] = transpose8x8(main_cols ? wh : wl);
                        }
                    }
                zsum[k] = __ffma2_rn(zsum[k], al, z2);
            }
            float d[kVC / 2][4];  // channels of codes 2 m and 2 m + 1
#pragma unroll
            for (int m2 = 0; m2 < kVC / 2; m2++) d[m2][0] = d[m2][1] = d[m2][2] = d[m2][3] = 0.0f;
            const unsigned char* vbase = vst + (NB == 1 ? 2 * g + p : 8 * p + g) * kVBits / 8;
#pragma unroll
            for (int j = 0; j < kTiles; j++) {
                // tokens t, t + 4, t + 8, t + 12 of the sixteen: MMA columns 2t, 2t + 1, 2t + 8, 2t + 9
                uint32_t w[4][kVX > 2 ? 2 : 1];
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const unsigned char* src = vbase + (16 * j + t + 4 * q) * C::kRow;
                    if constexpr (kVBits == 64) {
                        const uint2 v = *reinterpret_cast<const uint2*>(src);
                        w[q][0] = v.x;
                        w[q][kVX > 2 ? 1 : 0] = v.y;
                    } else if constexpr (kVBits == 32) {
                        w[q][0] = *reinterpret_cast<const uint32_t*>(src);
                    } else if constexpr (kVBits == 16) {
                        w[q][0] = *reinterpret_cast<const uint16_t*>(src);
                    } else {
                        w[q][0] = *src;
                    }
                }
#pragma unroll
                for (int x = 0; x < kVX; x++) {
                    const uint32_t sel = x & 1 ? 0x7632u : 0x5410u;
                    const uint32_t y0 = __byte_perm(w[0][x >> 1], w[1][x >> 1], sel);
                    const uint32_t y1 = __byte_perm(w[2][x >> 1], w[3][x >> 1], sel);
#pragma unroll
                    for (int i = 0; i < kVL; i += 2) {
                        float(&dd)[4] = d[(x * kVL + i) / 2];
                        const uint32_t a0 = code_pair<BITS>(y0, i), a1 = code_pair<BITS>(y0, i + 1);
                        const uint32_t a2 = code_pair<BITS>(y1, i), a3 = code_pair<BITS>(y1, i + 1);
                        mma_f16(dd, a0, a1, a2, a3, wb[j][0], wb[j][1]);
                        if constexpr (Q8) mma_f16(dd, a0, a1, a2, a3, wb[j][2], wb[j][3]);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < kVC; i++)
                acc[p][i] = __ffma2_rn(acc[p][i], al_acc, make_float2(d[i / 2][2 * (i & 1)], d[i / 2][2 * (i & 1) + 1]));
        }
        __syncwarp();  // all lanes have read the value codes and the scales
        if (lane == 0 && it + 1 < steps) load_codes(it + 1, 1);
    }
    phase += (uint32_t)steps;

    // ---- the part: four warp streams merged in shared memory (the buffers are free)
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) {
        lsum.x += __shfl_xor_sync(0xffffffffu, lsum.x, off);
        lsum.y += __shfl_xor_sync(0xffffffffu, lsum.y, off);
#pragma unroll
        for (int k = 0; k < NB; k++) {
            zsum[k].x += __shfl_xor_sync(0xffffffffu, zsum[k].x, off);
            zsum[k].y += __shfl_xor_sync(0xffffffffu, zsum[k].y, off);
        }
    }
    __syncthreads();
    float* mo = reinterpret_cast<float*>(smem + C::kFixed);  // [warp][query][128]
    float* ml = mo + kSWarps * 8 * kAD;                      // [warp][query][max (log2), sum]
    const float unscale = __uint_as_float((uint32_t)(127 - kb) << 23);
#pragma unroll
    for (int p = 0; p < kPass; p++)
#pragma unroll
        for (int i = 0; i < kVC; i++) {
            const float f = 16777216.0f / (float)(1 << code_shift<BITS>(i % kVL)) * unscale;
            const int ch = NB == 1 ? 16 * g + kVC * p + i : kBlk * p + kVC * g + i;
            float2 v = acc[p][i];
            if constexpr (!Q8) {
                v.x += __shfl_xor_sync(0xffffffffu, v.x, 2);
                v.y += __shfl_xor_sync(0xffffffffu, v.y, 2);
            }
            if (main_cols) {
                const float2 z = zsum[NB == 1 ? 0 : p];
                mo[(warp * 8 + q0) * kAD + ch] = fmaf(v.x, f, z.x);
                mo[(warp * 8 + q0 + 1) * kAD + ch] = fmaf(v.y, f, z.y);
            }
        }
    if (g == 0 && main_cols) {
        float* s0 = ml + (warp * 8 + q0) * 2;
        s0[0] = steps > 0 ? Mu.x * cF.x : -INFINITY;
        s0[1] = lsum.x;
        s0[2] = steps > 0 ? Mu.y * cF.y : -INFINITY;
        s0[3] = lsum.y;
    }
    __syncthreads();
    float* part = a.part + ((int64_t)unit * a.n_parts + slot) * a.n_rep * (kAD + 2);
    for (int r = 0; r < a.n_rep; r++) {
        float M = ml[r * 2];  // warp 0 has at least one step
        for (int w = 1; w < kSWarps; w++) M = fmaxf(M, ml[(w * 8 + r) * 2]);
        float o = 0.0f, ls = 0.0f;
        for (int w = 0; w < kSWarps; w++) {
            const float mw = ml[(w * 8 + r) * 2];
            if (mw == -INFINITY) continue;  // a stream without tokens
            const float e = ex2(mw - M);
            ls = fmaf(ml[(w * 8 + r) * 2 + 1], e, ls);
            o = fmaf(mo[(w * 8 + r) * kAD + tid], e, o);
        }
        part[r * (kAD + 2) + 2 + tid] = o;
        if (tid == 0) {
            part[r * (kAD + 2)] = M;
            part[r * (kAD + 2) + 1] = ls;
        }
    }
    // the buffers go back to the copies of the next segment
    fence_proxy_async_smem();
    __syncthreads();
    }
}

// Launches a kernel that may start while the one before it in the stream still runs; it waits
// (griddepcontrol.wait) before it reads what that one wrote.
template <typename K>
cudaError_t launch_dependent(K kernel, unsigned grid, unsigned threads, size_t smem, const AttnArgs& a, cudaStream_t st) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

template <int BITS, int NB, bool Q8>
cudaError_t launch_stream(AttnArgs& a, int sms, cudaStream_t st) {
    using C = StreamCfg<BITS, NB>;
    cudaError_t e = cudaFuncSetAttribute(attn_stream_kernel<BITS, NB, Q8>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kTotal);
    if (e != cudaSuccess) return e;
    // All units' steps in equal shares over the CTAs that fit at once: a share starts and ends
    // anywhere in a unit, so no SM waits for a last wave (64 sequences x 8 heads: 72 steps a CTA; whole
    // parts per CTA took 5 waves of 18). A unit's parts lie on consecutive CTAs.
    const int64_t units = (int64_t)a.L * a.B * a.H, slots = (int64_t)sms * kSCtas;
    a.unit_steps = (a.T + kSWarps * C::kTok - 1) / (kSWarps * C::kTok);
    a.all_steps = units * a.unit_steps;
    a.cta_steps = (a.all_steps + slots - 1) / slots;
    const int64_t most = (a.unit_steps + a.cta_steps - 1) / a.cta_steps + 1;
    a.n_parts = (int)(most < a.unit_steps ? most : a.unit_steps);  // at most one per 128 tokens (the workspace)
    const int64_t grid = (a.all_steps + a.cta_steps - 1) / a.cta_steps;
    return launch_dependent(attn_stream_kernel<BITS, NB, Q8>, (unsigned)grid, kSThreads, C::kTotal, a, st);
}

template <int BITS>
cudaError_t launch_stream_bits(AttnArgs& a, int sms, cudaStream_t st) {
    const bool q8 = a.n_rep > 4;
    if (a.blk == 128) return q8 ? launch_stream<BITS, 1, true>(a, sms, st) : launch_stream<BITS, 1, false>(a, sms, st);
    if (a.blk == 64) return q8 ? launch_stream<BITS, 2, true>(a, sms, st) : launch_stream<BITS, 2, false>(a, sms, st);
    return q8 ? launch_stream<BITS, 4, true>(a, sms, st) : launch_stream<BITS, 4, false>(a, sms, st);
}

template <int BITS, int NREP>
size_t chunk_smem() {
    const size_t fixed = (size_t)(NREP * kAD + NREP * 4 + 2 * NREP + 2 * NREP * 4 + 8 * NREP * 4) * 4 +
                         (size_t)kAttnChunk * 4 * 4;
    const size_t pbytes = (size_t)NREP * kAttnChunk * 4, rbytes = (size_t)kASlices * NREP * kAD * 4;
    return fixed + (pbytes > rbytes ? pbytes : rbytes);
}

template <int BITS, int NREP>
cudaError_t launch_chunks(const AttnArgs& a, cudaStream_t st) {
    const size_t smem = chunk_smem<BITS, NREP>();
    cudaError_t e = cudaFuncSetAttribute(attn_chunk_kernel<BITS, NREP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)a.n_parts, (unsigned)(a.L * a.B * a.H));
    attn_chunk_kernel<BITS, NREP><<<grid, kAThreads, smem, st>>>(a);
    return cudaGetLastError();
}

template <int BITS>
cudaError_t launch_chunks_bits(const AttnArgs& a, cudaStream_t st) {
    switch (a.n_rep) {
        case 1: return launch_chunks<BITS, 1>(a, st);
        case 2: return launch_chunks<BITS, 2>(a, st);
        case 4: return launch_chunks<BITS, 4>(a, st);
        case 8: return launch_chunks<BITS, 8>(a, st);
        default: return cudaErrorInvalidValue;
    }
}

// Few units: four slices of the parts and of the rotation per unit, for latency. More than two wide
// CTAs per SM would come in waves, so those get one slice each (768 units of 12 parts, 3 bits, whole call:
// 194.7 us with four slices, 182.5 with one; 512 units of 16,384 tokens: 280.7 and 281.4).
template <int NREP>
cudaError_t launch_combine(const AttnArgs& a, int sms, cudaStream_t st) {
    const int64_t units = (int64_t)a.L * a.B * a.H;
    if (units > 2 * (int64_t)sms) return launch_dependent(attn_combine_kernel<NREP, 1>, (unsigned)units, kAD, 0, a, st);
    return launch_dependent(attn_combine_kernel<NREP, 4>, (unsigned)units, 4 * kAD, 0, a, st);
}

}  // namespace

size_t attn_workspace_bytes(int64_t units, int n_rep, int d, int64_t T) {
    const int64_t n_chunks = (T + kAttnChunk - 1) / kAttnChunk;
    const size_t q = (((size_t)units * n_rep * d * 4) + 255) / 256 * 256;
    return q + (size_t)units * n_chunks * n_rep * (d + 2) * 4;
}

cudaError_t launch_attention(const AttnArgs& args, cudaStream_t st) {
    AttnArgs a = args;
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int queries = a.B * a.n_rep;
    const size_t qsmem = (size_t)(kAD * (a.g + 4) + kQueries * kAD) * 4;
    cudaError_t e = cudaFuncSetAttribute(attn_query_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)qsmem);
    if (e != cudaSuccess) return e;
    attn_query_kernel<<<dim3((unsigned)(a.L * a.H), (unsigned)((queries + kQueries - 1) / kQueries)), kQThreads, qsmem, st>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    a.n_parts = a.n_chunks;  // 3 and 6 bits: one chunk per part
    a.unit_steps = a.n_chunks;
    a.cta_steps = 1;
    switch (a.bits) {
        case 2: e = launch_stream_bits<2>(a, sms, st); break;
        case 3: e = launch_chunks_bits<3>(a, st); break;
        case 4: e = launch_stream_bits<4>(a, sms, st); break;
        case 6: e = launch_chunks_bits<6>(a, st); break;
        case 8: e = launch_stream_bits<8>(a, sms, st); break;
        default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    switch (a.n_rep) {
        case 1: return launch_combine<1>(a, sms, st);
        case 2: return launch_combine<2>(a, sms, st);
        case 4: return launch_combine<4>(a, sms, st);
        case 8: return launch_combine<8>(a, sms, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace cg
