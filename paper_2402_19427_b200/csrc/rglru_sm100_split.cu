// fp32 products on the sm_100a tensor cores, and the kernels around them: the forward and backward of fp32 io, the forward of bf16
// heads wider than 256 and the backward of bf16 calls that are promised fp32 between the kernels (heads wider than 256, ragged
// lengths).  Head widths that are multiples of 32.
//
// An fp32 value is the exact sum of three bf16 values ("planes": each the nearest to what the ones before leave, so that it is at most
// 2^-8 and 2^-17 of the value).  A product of two fp32 operands is the sum of six plane products; the other three are at most 2^-24 of it
// together, of either sign (planes cut off instead of rounded leave out up to 2^-21, always of the product's sign), and bf16 weights are
// a single plane, so that three products do.  They run on tcgen05 (kind::f16, bf16) and
// accumulate in fp32 tensor memory.  The accumulation rounds towards zero: measured on 128 x 128 tiles of random numbers, relative
// 2-norm error (bias) 5.5e-8 (-2.8e-8) after 64 products a result, 1.9e-7 (-1.2e-7) after 256, 8.6e-7 (-5.5e-7) after 1024, against
// 4.5e-8, 0.9e-7 and 2.1e-7 of a chain of fp32 FMAs.  So the leading product of each pair of planes has accumulators of its own, which
// take few enough terms that no output is further from the exact one than with such chains (128 in dW and du, see forward() for the
// gates), and the small ones, whose roundings are 2^-8 smaller, others.
//   1. split_weights      (fp32 io) the weights as planes
//   2. split_forward      Conv1D, planes of u, both gate products, gates, scan, chain of chunks: y, or for the backward r, i, the
//                         state before every eighth token, and the planes of u
//   3. split_reverse      reverse scan and element-wise adjoints: planes of dz, the direct part of du in fp32
//   4. split_products     du += W^T dz and dW = dz^T u, one launch
//   5. Conv1D adjoint (rglru_sm100_bwd.cu) and reductions in fixed order (rglru_generic.cu)
#include <cuda.h>
#include <cuda_bf16.h>

#include "rglru_chain.cuh"
#include "rglru_gates32.cuh"
#include "rglru_internal.h"
#include "sm100_ptx.cuh"

namespace rglru {
namespace {

using namespace ptx;

constexpr int PLANES = 3;
constexpr int SEG = 8;                        // tokens between saved states = tokens of a thread of the reverse scan
constexpr int FWD_THREADS = 320;              // eight warps of Conv1D and epilogue, one of copies, one of products
constexpr uint32_t TILE_BYTES = 128 * 128;    // 128 rows (or 2 x 64 columns) of 64 bf16: one operand tile of a K block of 64
constexpr int PROD_STAGES = 2, PROD_THREADS = 352;   // K blocks in flight; eight epilogue warps, one of products, two of copies

__device__ __forceinline__ uint32_t tops(f32x2 v) { return __byte_perm(__float_as_uint(v.x), __float_as_uint(v.y), 0x7632); }   // the upper halves, v.x's below
__device__ __forceinline__ float bound_bf16(float v) {   // the largest finite bf16 value, with v's sign, for what would round up to infinity; a NaN stays one
    float y;
    asm("min.NaN.xorsign.abs.f32 %0, %1, %2;" : "=f"(y) : "f"(v), "f"(3.38953139e38f));
    return y;
}
// The planes of two values: the nearest bf16 value to what is left, twice; what is left then (at most eight bits) is a bf16 value itself.
// An infinity leaves infinity and NaN behind itself, so that whatever it enters is NaN: gradients stay non-finite, and for the gates,
// which an infinite sum saturates, see exact_walk.
__device__ __forceinline__ void split_planes(f32x2 v, uint32_t (&w)[PLANES]) {
    w[0] = pack_bf16(bound_bf16(v.x), bound_bf16(v.y));
    v = fma2(bf2x(w[0]), pack2(-1.0f, -1.0f), v);
    w[1] = pack_bf16(v.x, v.y);
    v = fma2(bf2x(w[1]), pack2(-1.0f, -1.0f), v);
    w[2] = tops(v);
}
__device__ __forceinline__ f32x2 ld2(const float *p) { return ld2f(p); }
__device__ __forceinline__ f32x2 ld2(const __nv_bfloat16 *p) { return bf2x(*(const uint32_t *)p); }
__device__ __forceinline__ float ld1(const float *p) { return *p; }
__device__ __forceinline__ float ld1(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
__device__ __forceinline__ void st1(float *p, float v) { *p = v; }
__device__ __forceinline__ void st1(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }

// ------------------------------------------------------------------ weights as planes (fp32 io)
// out[gate][plane][n], two values a thread
__global__ void __launch_bounds__(256) split_weights_kernel(const float *Wa, const float *Wx, uint32_t *out, size_t n2) {
    dependency_wait();
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    dependency_trigger();
    if (i >= 2 * n2) return;
    const size_t gate = i >= n2, j = i - gate * n2;
    uint32_t w[PLANES];
    split_planes(ld2f((gate ? Wx : Wa) + 2 * j), w);
#pragma unroll
    for (int q = 0; q < PLANES; ++q) out[(gate * PLANES + q) * n2 + j] = w[q];
}

// One K block of 64 (four instructions, or two of its first half): the operands' descriptors advance by da and db 16-byte units an
// instruction.  Straight-line code with nothing but additions: one thread issues it, and with the descriptors built in loops it needed
// 240 cycles an instruction where the tensor core needs 49 to 65 (B4 T1024 D1024 in 4 heads, forward 72 us, products 75).
__device__ __forceinline__ void mma_block(uint32_t d_tmem, uint64_t a, uint32_t da, uint64_t b, uint32_t db, uint32_t idesc, bool accumulate, bool full) {
    mma_ss(d_tmem, a, b, idesc, accumulate);
    mma_ss(d_tmem, a + da, b + db, idesc, 1);
    if (full) {
        mma_ss(d_tmem, a + 2 * da, b + 2 * db, idesc, 1);
        mma_ss(d_tmem, a + 3 * da, b + 3 * db, idesc, 1);
    }
}

// ------------------------------------------------------------------ forward
// Block = (chunk of TOK tokens, sequence, head, 128 output channels).  Eight warps convolve 64 input channels at a time and write the
// three planes of u as the B operand (K-major, 128-byte swizzle, two stages); weight tiles of 128 channels x 64 arrive by tiled TMA as
// the A operand; z is left channel-per-lane in tensor memory, so that each of the eight warps then walks its 32 channels through half
// of the chunk's tokens in registers.  Chunks are chained as in rglru_generic.cu (block order is chunk-major).
// Two blocks fit an SM (64 tokens: 97 KB of shared memory, 256 columns of tensor memory), one's gates beside the other's products.
struct SplitFwdArgs {
    alignas(64) CUtensorMap tm_wa, tm_wx;   // [planes x H][dh][dh], box 64 x 128
    FwdArgs f;
    Chain ch;
    uint32_t *u_planes;   // SAVE: [head][plane][B T][dh] bf16
    float *h_seg;         // SAVE: [B][ceil(T / SEG)][D] state before every SEG-th token
    int nchunk, mtiles;
    int wplanes;          // 1 (bf16 weights) or 3
    int sets;             // sets of accumulators, see KSet (more than one with LATE and 32 tokens only)
    uint32_t cols;        // columns of tensor memory: those of the sets, rounded up to a power of two
};
// A set is two accumulators a gate, X and Y of TOK columns each, and the K blocks [k0, k1) that it takes.  Up to kb, leading products go to
// X and the small ones to Y, the first two planes of u as one operand of twice the width.  With LATE, the small products of the blocks
// from kb on, at most two, go to Y too, and then the leading ones: Y still is 2^-8 of the sum when they come.  See forward() for when.
struct KSet { int k0, kb, k1; };
template <bool LATE> __device__ __forceinline__ KSet k_set(int nk, int sets, int i) {
    if (!LATE) return KSet{0, nk, nk};   // one set
    const int k0 = nk * i / sets, k1 = nk * (i + 1) / sets;
    return KSet{k0, k1 - max(0, min(2, k1 - k0 - 2)), k1};
}
template <int TOK> struct FwdSmem {
    static constexpr int SLOTS = TOK == 32 ? 10 : 3;   // weight tiles in flight: two blocks of 64 tokens share an SM, one of 32 has it to itself
    static constexpr uint32_t PLANE = TOK * 128, STAGE = PLANES * PLANE, RING = 2 * STAGE, BAR = RING + SLOTS * TILE_BYTES;
    static constexpr uint32_t ALLOC = BAR + 256 + 1024;
};

// A channel on its walk through the tokens from zero state: what the Conv1D needs of it and where it stands
struct Walk {
    float ba, bx, cb, w[4], s;
    float P, h, x1, x2, x3;   // the step so far; the last three inputs
};
// Gates, decay and scan of the eight tokens from tb on: za, zx are the sums of Eq. 1 and 2 without their biases, and become the running
// steps P and h.  SAVE: r and i go to pr and pi instead.
template <bool SAVE, bool POLY>
__device__ __forceinline__ void walk_segment(Walk &k, f32x2 (&za)[4], f32x2 (&zx)[4], const float (&xs)[SEG], int tb, int T, int D, bool cv, float *pr, float *pi) {
    const bool whole = tb + SEG <= T;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const f32x2 r = sigmoid2_acc(__fadd2_rn(za[j], pack2(k.ba, k.ba)));
        const f32x2 g = sigmoid2_acc(__fadd2_rn(zx[j], pack2(k.bx, k.bx)));
        const f32x2 fr = one_minus_decay2<POLY>(r, pack2(k.s, k.s));
        f32x2 rm;
        const f32x2 m = input_scale2(fr, rm);
        float u[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float x0 = xs[2 * j + e];
            u[e] = fmaf(k.w[3], k.x3, fmaf(k.w[2], k.x2, fmaf(k.w[1], k.x1, fmaf(k.w[0], x0, k.cb))));
            k.x3 = k.x2; k.x2 = k.x1; k.x1 = x0;
        }
        const f32x2 a = fma2(fr, pack2(-1.0f, -1.0f), pack2(1.0f, 1.0f)), v = mul2(m, mul2(g, pack2(u[0], u[1])));
        const bool e0 = whole || tb + 2 * j < T, e1 = whole || tb + 2 * j + 1 < T;
        if (SAVE) {
            if (e0 && cv) { *pr = r.x; *pi = g.x; }
            pr += D; pi += D;
            if (e1 && cv) { *pr = r.y; *pi = g.y; }
            pr += D; pi += D;
        }
        // a token that does not exist holds the state
        const float a0 = e0 ? a.x : 1.0f, v0 = e0 ? v.x : 0.0f, a1 = e1 ? a.y : 1.0f, v1 = e1 ? v.y : 0.0f;
        k.P *= a0; k.h = fmaf(a0, k.h, v0);
        if (!SAVE) { za[j].x = k.P; zx[j].x = k.h; }
        k.P *= a1; k.h = fmaf(a1, k.h, v1);
        if (!SAVE) { za[j].y = k.P; zx[j].y = k.h; }
    }
}

// The walk of a warp that ended in a NaN, once more, with the sums of the gates made term by term: an infinite factor is NaN in the
// products of its planes, where a sum that ends in an infinity saturates its gate.  Slow (some hundred microseconds), and only for inputs
// or weights that are not finite (every walk of B2 T777 D5632 made again: 19 ms; nothing but NaN, where the sums end at once: 1.6; finite:
// 0.12).  Out of line: the walk that everybody takes pays a vote and some 60 bytes of spills for it (backward of B5 T1021 D1536 in 16
// heads 242.1 -> 245.5 us).  Leaves the step up to each segment (SAVE) in tensor memory, where the running steps go otherwise, and returns
// the whole one.
template <typename IOT, bool SAVE, int TOK>
__device__ __noinline__ float2 exact_walk(const SplitFwdArgs &p, uint32_t tm, int b, int head, int c, int t0, float s) {
    const FwdArgs &f = p.f;
    const int T = f.T, D = f.D, dh = D / f.H;
    const bool cv = c < dh;
    const IOT *x = (const IOT *)f.x + (size_t)b * T * D + head * dh, *cw = (const IOT *)f.conv_w + head * dh, *cs = (const IOT *)f.cs_in;
    if (cs) cs += (size_t)b * 3 * D + head * dh;
    if (!cv) c = 0;
    const size_t row = ((size_t)head * dh + c) * dh;
    const IOT *wa = (const IOT *)f.W_a + row, *wx = (const IOT *)f.W_x + row;
    auto xat = [&](int t, int k) -> float { return t >= 0 ? (t < T ? ld1(x + (size_t)t * D + k) : 0.0f) : cs ? ld1(cs + (size_t)(3 + t) * D + k) : 0.0f; };
    auto bias = [&](int k) -> float { return f.conv_b ? f.conv_b[head * dh + k] : 0.0f; };
    Walk k{f.b_a[head * dh + c], f.b_x[head * dh + c], bias(c), {}, s, 1.0f, 0.0f, xat(t0 - 1, c), xat(t0 - 2, c), xat(t0 - 3, c)};
#pragma unroll
    for (int i = 0; i < 4; ++i) k.w[i] = ld1(cw + (size_t)i * D + c);
    float segP[TOK / 2 / SEG], segH[TOK / 2 / SEG];
#pragma unroll
    for (int j = 0; j < TOK / 2 / SEG; ++j) {
        const int tb = t0 + j * SEG;
        f32x2 za[4], zx[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { za[i] = pack2(0.f, 0.f); zx[i] = pack2(0.f, 0.f); }
#pragma unroll 1
        for (int n = 0; n < dh; ++n) {
            float xv[SEG + 3], u[SEG], w[4];
            const float cb = bias(n), a = ld1(wa + n), g = ld1(wx + n);
#pragma unroll
            for (int i = 0; i < SEG + 3; ++i) xv[i] = xat(tb - 3 + i, n);
#pragma unroll
            for (int i = 0; i < 4; ++i) w[i] = ld1(cw + (size_t)i * D + n);
#pragma unroll
            for (int i = 0; i < SEG; ++i) u[i] = fmaf(w[3], xv[i], fmaf(w[2], xv[i + 1], fmaf(w[1], xv[i + 2], fmaf(w[0], xv[i + 3], cb))));
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                za[i] = fma2(pack2(a, a), pack2(u[2 * i], u[2 * i + 1]), za[i]);
                zx[i] = fma2(pack2(g, g), pack2(u[2 * i], u[2 * i + 1]), zx[i]);
            }
            if ((n & 15) == 0) {   // where the inputs themselves are NaN there is nothing to find out
                bool nan = true;
#pragma unroll
                for (int i = 0; i < 4; ++i) nan = nan && za[i].x != za[i].x && za[i].y != za[i].y && zx[i].x != zx[i].x && zx[i].y != zx[i].y;
                if (__all_sync(0xffffffffu, nan)) break;
            }
        }
        float xs[SEG];
#pragma unroll
        for (int i = 0; i < SEG; ++i) xs[i] = xat(tb + i, c);
        segP[j] = k.P; segH[j] = k.h;
        const size_t e = ((size_t)b * T + tb) * D + head * dh + c;
        walk_segment<SAVE, false>(k, za, zx, xs, tb, T, D, cv, SAVE ? f.save_r + e : nullptr, SAVE ? f.save_i + e : nullptr);
        if (!SAVE) { tmem_st8p(tm + j * SEG, za); tmem_st8p(tm + 2 * TOK + j * SEG, zx); }
    }
    if (SAVE) {
        f32x2 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = j < TOK / 2 / SEG ? pack2(segP[j], segH[j]) : pack2(0.f, 0.f);
        tmem_st8p(tm, v);
    }
    tmem_st_wait();
    return make_float2(k.P, k.h);
}

// Chain of the chunks, then the outputs: y, or (SAVE) the states before the segments
template <typename IOT, bool SAVE, int TOK>
__device__ __forceinline__ void forward_rest(const SplitFwdArgs &p, uint32_t tmem, int b, int head, int mt, int chunk, float *xch, volatile int *abort_flag, bool ok, float P, float h,
                                             const float (&segP)[TOK / 2 / SEG], const float (&segH)[TOK / 2 / SEG]) {
    constexpr int HALF = TOK / 2;
    const FwdArgs &f = p.f;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = warp & 3, half = warp >> 2;
    const int T = f.T, D = f.D, dh = D / f.H, chl = q * 32 + lane, c = mt * 128 + chl;
    const bool cv = c < dh;
    const int d = head * dh + (cv ? c : 0), t0 = chunk * TOK + half * HALF;
    const IOT *cs_in = (const IOT *)f.cs_in, *xb = (const IOT *)f.x + (size_t)b * T * D + d;
    const uint32_t tm = tmem + ((uint32_t)(q * 32) << 16) + half * HALF;
    // ---- chain: the first half's thread of a channel takes the state that the previous chunk reached and hands its own on
    float *xP = xch, *xh = xch + 128;
    if (half == 1) { xP[chl] = P; xh[chl] = h; }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    float carry = 0.0f;
    if (half == 0) {
        uint4 *slot = p.ch.slot + (size_t)b * D + d;
        const float P1 = xP[chl], h1 = xh[chl], cP = P * P1, cH = fmaf(P1, h, h1);
        float P_in = 1.0f;
        ok = !*abort_flag;
        if (ok) {
            if (chunk == 0) carry = f.h0 ? f.h0[(size_t)b * D + d] : 0.0f;
            else ok = chain_wait(p.ch, slot, cv, chunk - 1, carry, P_in);
        }
        const float hs = fmaf(cP, carry, cH), Ps = cP * P_in;
        if (ok && cv) {
            chain_put(p.ch, slot, chunk, hs, Ps);
            if (!SAVE && chunk + 1 == p.nchunk) {
                f.h_T[(size_t)b * D + d] = hs;
                if (f.a_prod) f.a_prod[(size_t)b * D + d] = Ps;
                // the last three raw inputs of concat(conv_state_in, x), bit-exact
                IOT keep[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const int t = T - 3 + k;
                    keep[k] = t >= 0 ? xb[(size_t)t * D] : cs_in ? cs_in[((size_t)b * 3 + (3 + t)) * D + d] : IOT(0.0f);
                }
#pragma unroll
                for (int k = 0; k < 3; ++k) ((IOT *)f.cs_out)[((size_t)b * 3 + k) * D + d] = keep[k];
            }
        }
        if (!ok) {
            if (cv) chain_fail(p.ch, slot, chunk);
            *abort_flag = 1;
        }
        xP[chl] = fmaf(P, carry, h);   // the state that the second half starts from
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (*abort_flag) return;
    if (half == 1) carry = xP[chl];
    if (SAVE) {
        const int nseg = (T + SEG - 1) / SEG;
#pragma unroll
        for (int j = 0; j < HALF / SEG; ++j)
            if (cv && t0 + j * SEG < T) p.h_seg[((size_t)b * nseg + t0 / SEG + j) * D + d] = fmaf(segP[j], carry, segH[j]);
        return;
    }
    const IOT *gb = (const IOT *)f.gate_branch;
#pragma unroll 1
    for (int j = 0; j < HALF / SEG; ++j) {
        f32x2 Pv[4], hv[4];
        tmem_ld8p(tm + j * SEG, Pv); tmem_ld8p(tm + 2 * TOK + j * SEG, hv);
        tmem_ld_wait();
        const int tb = t0 + j * SEG;
        const size_t e = ((size_t)b * T + tb) * D + d;
        IOT *y = (IOT *)f.y + e;
#pragma unroll
        for (int k = 0; k < SEG; ++k) {
            if (tb + k < T && cv) {
                float o = fmaf(k & 1 ? Pv[k / 2].y : Pv[k / 2].x, carry, k & 1 ? hv[k / 2].y : hv[k / 2].x);
                if (gb) o *= gelu_acc(ld1(gb + e + (size_t)k * D));   // merged output of the recurrent block (Section 2.3)
                st1(y, o);
            }
            y += D;
        }
    }
}

template <typename IOT, bool SAVE, bool LATE, int TOK, bool POLY>
__device__ __forceinline__ void forward_epilogue(const SplitFwdArgs &p, uint32_t tmem, int b, int head, int mt, int chunk, float *xch, volatile int *abort_flag, float s, uint32_t acc_bar, bool ok) {
    constexpr int HALF = TOK / 2;
    const FwdArgs &f = p.f;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = warp & 3, half = warp >> 2;
    const int T = f.T, D = f.D, dh = D / f.H, chl = q * 32 + lane, c = mt * 128 + chl;
    const bool cv = c < dh;
    const int d = head * dh + (cv ? c : 0), t0 = chunk * TOK + half * HALF;
    const IOT *x = (const IOT *)f.x, *cw = (const IOT *)f.conv_w, *cs_in = (const IOT *)f.cs_in;
    const IOT *xb = x + (size_t)b * T * D + d;
    auto xat = [&](int t) -> float { return t >= 0 ? (t < T ? ld1(xb + (size_t)t * D) : 0.0f) : cs_in ? ld1(cs_in + ((size_t)b * 3 + (3 + t)) * D + d) : 0.0f; };
    Walk k{f.b_a[d], f.b_x[d], f.conv_b ? f.conv_b[d] : 0.0f, {}, s, 1.0f, 0.0f, xat(t0 - 1), xat(t0 - 2), xat(t0 - 3)};
#pragma unroll
    for (int j = 0; j < 4; ++j) k.w[j] = ld1(cw + (size_t)j * D + d);
    const uint32_t tm = tmem + ((uint32_t)(q * 32) << 16) + half * HALF;
    float segP[HALF / SEG], segH[HALF / SEG], xn[SEG];
    auto fetch = [&](int tb) {
        if (tb + SEG <= T) {
            const IOT *px = xb + (size_t)tb * D;
#pragma unroll
            for (int k = 0; k < SEG; ++k) { xn[k] = ld1(px); px += D; }
        } else {
#pragma unroll
            for (int k = 0; k < SEG; ++k) xn[k] = xat(tb + k);
        }
    };
    fetch(t0);
    // everything above is on its way while the products run
    if (ok) ok = warp_wait(acc_bar, 0, p.ch.spin_ns, abort_flag);
    if (!ok && lane == 0) { *abort_flag = 1; atomicExch(f.status, STATUS_MAGIC | (uint32_t)RGLRU_ERR_TIMEOUT); }
    tc_fence_after();
    dependency_trigger();
#pragma unroll(SAVE ? HALF / SEG : 1)
    for (int j = 0; j < HALF / SEG; ++j) {
        f32x2 za[4], zx[4], la[4], lx[4];
        const int tb = t0 + j * SEG;
        tmem_ld8p(tm + j * SEG, za); tmem_ld8p(tm + TOK + j * SEG, la); tmem_ld8p(tm + 2 * TOK + j * SEG, zx); tmem_ld8p(tm + 3 * TOK + j * SEG, lx);
        float xs[SEG];
        if (SAVE && j > 0) fetch(tb);
#pragma unroll
        for (int i = 0; i < SEG; ++i) xs[i] = xn[i];
        if (!SAVE && j + 1 < HALF / SEG) fetch(tb + SEG);   // SAVE has no registers left for it
        tmem_ld_wait();
        if (SAVE) { segP[j] = k.P; segH[j] = k.h; }
#pragma unroll
        for (int i = 0; i < 4; ++i) { za[i] = __fadd2_rn(za[i], la[i]); zx[i] = __fadd2_rn(zx[i], lx[i]); }
        if (LATE && TOK == 32) {
#pragma unroll 1
            for (int set = 1; set < p.sets; ++set) {
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    f32x2 X[4], Y[4];
                    tmem_ld8p(tm + (4 * set + 2 * g) * TOK + j * SEG, X); tmem_ld8p(tm + (4 * set + 2 * g + 1) * TOK + j * SEG, Y);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (g == 0) za[i] = __fadd2_rn(za[i], __fadd2_rn(X[i], Y[i]));
                        else zx[i] = __fadd2_rn(zx[i], __fadd2_rn(X[i], Y[i]));
                    }
                }
            }
        }
        const size_t e = ((size_t)b * T + tb) * D + d;
        walk_segment<SAVE, POLY>(k, za, zx, xs, tb, T, D, cv, SAVE ? f.save_r + e : nullptr, SAVE ? f.save_i + e : nullptr);
        if (!SAVE) { tmem_st8p(tm + j * SEG, za); tmem_st8p(tm + 2 * TOK + j * SEG, zx); }
    }
    if (!SAVE) tmem_st_wait();
    float P = k.P, h = k.h;
    if (__any_sync(0xffffffffu, cv && (P != P || h != h))) {
        const float2 step = exact_walk<IOT, SAVE, TOK>(p, tm, b, head, c, t0, s);
        P = step.x; h = step.y;
        if (SAVE) {
            f32x2 v[4];
            tmem_ld8p(tm, v);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < HALF / SEG; ++j) { segP[j] = v[j].x; segH[j] = v[j].y; }
        }
    }
    // made again from here on: kept across the call above they would not fit the registers of the walk
    asm volatile("" : "+r"(b), "+r"(head), "+r"(mt), "+r"(chunk));
    forward_rest<IOT, SAVE, TOK>(p, tmem, b, head, mt, chunk, xch, abort_flag, ok, P, h, segP, segH);
}

template <typename IOT, bool SAVE, bool LATE, int TOK>
__global__ void __launch_bounds__(FWD_THREADS, 2) split_forward_kernel(const __grid_constant__ SplitFwdArgs p) {
    using S = FwdSmem<TOK>;
    extern __shared__ uint8_t smem_raw[];
    __shared__ float xch[2 * 128];
    __shared__ uint32_t tmem_s;
    __shared__ volatile int abort_s;
    const uint32_t raw = smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw);
    const uint32_t bar = base + S::BAR;
    auto U_FULL = [&](int i) { return bar + 8u * i; };
    auto U_EMPTY = [&](int i) { return bar + 16u + 8u * i; };
    auto W_FULL = [&](int i) { return bar + 32u + 8u * i; };
    auto W_EMPTY = [&](int i) { return bar + 32u + 8u * (S::SLOTS + i); };
    const uint32_t ACC = bar + 32u + 16u * S::SLOTS;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const FwdArgs &f = p.f;
    const int T = f.T, D = f.D, H = f.H, dh = D / H, nk = (dh + 63) / 64;
    int bid = blockIdx.x;
    const int mt = bid % p.mtiles; bid /= p.mtiles;
    const int head = bid % H; bid /= H;
    const int b = bid % f.B, chunk = bid / f.B;
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) { mbar_init(U_FULL(i), 8); mbar_init(U_EMPTY(i), 1); }
        for (int i = 0; i < S::SLOTS; ++i) { mbar_init(W_FULL(i), 1); mbar_init(W_EMPTY(i), 1); }
        mbar_init(ACC, 1);
        abort_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 8) { tmem_alloc(smem_u32(&tmem_s), p.cols); tmem_relinquish(); }
    if (warp == 9 && lane == 0) { prefetch_tensormap(&p.tm_wa); prefetch_tensormap(&p.tm_wx); }
    const unsigned long long spin = p.ch.spin_ns;
    dependency_wait();
    // u of 64 channels x TOK tokens at a time: lane = two adjacent channels, warp = TOK / 8 tokens.  The first loads are on their way
    // while the block sets itself up.
    constexpr int TW = TOK / 8;
    const int ta = chunk * TOK + warp * TW;
    const IOT *x = (const IOT *)f.x + (size_t)b * T * D + head * dh, *cw = (const IOT *)f.conv_w + head * dh, *cs = (const IOT *)f.cs_in;
    if (cs) cs += (size_t)b * 3 * D + head * dh;
    f32x2 xr[TW + 3], w[4], cb;
    const bool inside = ta >= 3 && ta + TW <= T;   // uniform over the warp
    auto fetch = [&](int kc) {
        const int k = kc * 64 + 2 * lane;
        const bool kv = k < dh;
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = kv ? ld2(cw + (size_t)j * D + k) : pack2(0.f, 0.f);
        cb = kv && f.conv_b ? ld2f(f.conv_b + head * dh + k) : pack2(0.f, 0.f);
        if (inside && kc * 64 + 64 <= dh) {
            const IOT *px = x + (size_t)(ta - 3) * D + k;
#pragma unroll
            for (int i = 0; i < TW + 3; ++i) { xr[i] = ld2(px); px += D; }
            return;
        }
#pragma unroll
        for (int i = 0; i < TW + 3; ++i) {
            const int t = ta - 3 + i;
            xr[i] = pack2(0.f, 0.f);
            if (kv) {
                if (t >= 0) { if (t < T) xr[i] = ld2(x + (size_t)t * D + k); }
                else if (cs) xr[i] = ld2(cs + (size_t)(3 + t) * D + k);
            }
        }
    };
    if (warp < 8) fetch(0);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_s;
    if (warp == 9) {
        if (lane == 0) {
            bool ok = true;
            int it = 0;
            auto load = [&](int kc, int g, int q) {
                const int s = it % S::SLOTS;
                ok = ok && mbar_wait(W_EMPTY(s), ((it / S::SLOTS) & 1) ^ 1, spin, (volatile int *)&abort_s);
                if (!ok) return;
                mbar_expect_tx(W_FULL(s), TILE_BYTES);
                tma_load_3d(base + S::RING + s * TILE_BYTES, g ? &p.tm_wx : &p.tm_wa, kc * 64, mt * 128, q * H + head, W_FULL(s));
                ++it;
            };
            for (int i = 0; i < (LATE ? p.sets : 1) && ok; ++i) {
                const KSet r = k_set<LATE>(nk, p.sets, i);
                for (int kc = r.k0; kc < r.kb; ++kc)
                    for (int g = 0; g < 2; ++g)
                        for (int q = 0; q < p.wplanes; ++q) load(kc, g, q);
                for (int g = 0; LATE && g < 2 && r.kb < r.k1; ++g) {
                    for (int kc = r.kb; kc < r.k1; ++kc)
                        for (int q = p.wplanes - 1; q > 0; --q) load(kc, g, q);
                    for (int kc = r.kb; kc < r.k1; ++kc) load(kc, g, 0);
                }
            }
            if (!ok) { abort_s = 1; atomicExch(f.status, STATUS_MAGIC | (uint32_t)RGLRU_ERR_TIMEOUT); }
        }
    } else if (warp == 8) {
        if (lane == 0) {
            // the planes of u lie one behind the other, and so do a gate's two accumulators: the first two planes are one operand of twice the width
            constexpr uint32_t idesc = make_idesc(128, TOK), idesc2 = make_idesc(128, 2 * TOK);
            constexpr int WP = sizeof(IOT) == 4 ? PLANES : 1;
            bool ok = true;
            int slot = 0, round = 0;
            auto u_full = [&](int kc) { ok = ok && mbar_wait(U_FULL(kc & 1), (kc >> 1) & 1, spin, (volatile int *)&abort_s); };
            auto w_full = [&]() {
                ok = ok && mbar_wait(W_FULL(slot), round & 1, spin, (volatile int *)&abort_s);
                tc_fence_after();
                return ok;
            };
            auto next_slot = [&]() { if (++slot == S::SLOTS) { slot = 0; ++round; } };
            auto w_tile = [&](int s) { return make_desc_sw128(base + S::RING + s * TILE_BYTES); };
            constexpr uint64_t B1 = S::PLANE >> 4, B2 = 2 * B1;
            for (int set = 0; set < (LATE ? p.sets : 1) && ok; ++set) {
                const KSet r = k_set<LATE>(nk, p.sets, set);
                const uint32_t acc0 = tmem + 4 * set * TOK;
                for (int kc = r.k0; kc < r.kb && ok; ++kc) {
                    const bool full = dh - kc * 64 >= 64;   // else the last half block
                    u_full(kc);
                    if (!ok) break;
                    const uint64_t u_desc = make_desc_sw128(base + (kc & 1) * S::STAGE);
#pragma unroll
                    for (int i = 0; i < 2 * WP; ++i) {
                        const int g = i / WP, q = i % WP;   // gate, plane of the weights
                        const uint32_t acc = acc0 + 2 * g * TOK;
                        if (!w_full()) break;
                        const uint64_t w_desc = w_tile(slot);
                        if (q == 0) {
                            mma_block(acc, w_desc, 2, u_desc, 2, idesc2, kc > r.k0, full);
                            mma_block(acc + TOK, w_desc, 2, u_desc + B2, 2, idesc, true, full);
                        } else {
                            mma_block(acc + TOK, w_desc, 2, u_desc, 2, idesc, true, full);
                            if (q == 1) mma_block(acc + TOK, w_desc, 2, u_desc + B1, 2, idesc, true, full);
                        }
                        tc_commit(W_EMPTY(slot));
                        next_slot();
                    }
                    if (ok) tc_commit(U_EMPTY(kc & 1));
                }
                if (!LATE || r.kb == r.k1) continue;
                for (int g = 0; g < 2 && ok; ++g) {
                    const uint32_t acc = acc0 + (2 * g + 1) * TOK;
                    if (WP > 1) {
                        for (int kc = r.kb; kc < r.k1 && ok; ++kc) {
                            const bool full = dh - kc * 64 >= 64;
                            const uint64_t u_desc = make_desc_sw128(base + (kc & 1) * S::STAGE);
                            if (g == 0) u_full(kc);
#pragma unroll
                            for (int q = WP - 1; q > 0; --q) {
                                if (!w_full()) break;
                                mma_block(acc, w_tile(slot), 2, u_desc, 2, idesc, true, full);
                                if (q == 1) mma_block(acc, w_tile(slot), 2, u_desc + B1, 2, idesc, true, full);
                                tc_commit(W_EMPTY(slot));
                                next_slot();
                            }
                        }
                    }
                    int first = slot;   // the tiles of the first plane stay until the leading products
                    for (int kc = r.kb; kc < r.k1 && ok; ++kc) {
                        const bool full = dh - kc * 64 >= 64;
                        const uint64_t u_desc = make_desc_sw128(base + (kc & 1) * S::STAGE);
                        if (WP == 1 && g == 0) u_full(kc);
                        if (!w_full()) break;
                        mma_block(acc, w_tile(slot), 2, u_desc + B1, 2, idesc, true, full);
                        mma_block(acc, w_tile(slot), 2, u_desc + B2, 2, idesc, true, full);
                        next_slot();
                    }
                    for (int kc = r.kb; kc < r.k1 && ok; ++kc) {
                        mma_block(acc, w_tile(first), 2, make_desc_sw128(base + (kc & 1) * S::STAGE), 2, idesc, true, dh - kc * 64 >= 64);
                        tc_commit(W_EMPTY(first));
                        if (g == 1) tc_commit(U_EMPTY(kc & 1));
                        if (++first == S::SLOTS) first = 0;
                    }
                }
            }
            if (ok) tc_commit(ACC);
            else { abort_s = 1; atomicExch(f.status, STATUS_MAGIC | (uint32_t)RGLRU_ERR_TIMEOUT); }
        }
    } else {
        bool ok = true;
        for (int kc = 0; kc < nk; ++kc) {
            const int k = kc * 64 + 2 * lane;
            const bool kv = k < dh;
            f32x2 u[TW];
#pragma unroll
            for (int i = 0; i < TW; ++i) u[i] = fma2(w[3], xr[i], fma2(w[2], xr[i + 1], fma2(w[1], xr[i + 2], fma2(w[0], xr[i + 3], cb))));
            if (kc + 1 < nk) fetch(kc + 1);
            ok = warp_wait(U_EMPTY(kc & 1), ((kc >> 1) & 1) ^ 1, spin, (volatile int *)&abort_s);
            if (!ok) break;
            uint8_t *st = smem + (kc & 1) * S::STAGE + warp * TW * 128 + (lane & 3) * 4;
            const bool own = SAVE && (kc >> 1) == mt && kv;
            const size_t plane = (size_t)f.B * T * dh / 2;
            const uint32_t row_words = (uint32_t)dh / 2;
            uint32_t *d0 = p.u_planes + (size_t)head * PLANES * plane + (((size_t)b * T + ta) * dh + k) / 2, *d1 = d0 + plane, *d2 = d1 + plane;
#pragma unroll
            for (int i = 0; i < TW; ++i) {
                uint32_t pl[PLANES];
                split_planes(u[i], pl);
                const uint32_t off = i * 128 + (((lane >> 2) ^ ((warp * TW + i) & 7)) << 4);
#pragma unroll
                for (int q = 0; q < PLANES; ++q) *(uint32_t *)(st + q * S::PLANE + off) = pl[q];
                if (SAVE) {
                    if (own && ta + i < T) { *d0 = pl[0]; *d1 = pl[1]; *d2 = pl[2]; }
                    d0 += row_words; d1 += row_words; d2 += row_words;
                }
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(U_FULL(kc & 1));
        }
        const int c = mt * 128 + (warp & 3) * 32 + lane;
        const float s = c < dh ? decay_rate_acc(f.lambda[head * dh + c], f.c) : 0.0f;
        if (__all_sync(0xffffffffu, s <= S_POLY)) forward_epilogue<IOT, SAVE, LATE, TOK, true>(p, tmem, b, head, mt, chunk, xch, &abort_s, s, ACC, ok);
        else forward_epilogue<IOT, SAVE, LATE, TOK, false>(p, tmem, b, head, mt, chunk, xch, &abort_s, s, ACC, ok);
        tc_fence_before();
    }
    __syncthreads();
    if (abort_s) {   // let copies and MMAs in flight land before shared and tensor memory are given back
        const uint64_t tw = gtimer();
        while (gtimer() - tw < 50000ull) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 8) tmem_dealloc(tmem, p.cols);
}

// ------------------------------------------------------------------ reverse scan
//   g_t = dy_t + a_{t+1} g_{t+1};  dL = g a (h_{t-1} - a v / m);  dv = g m;  di = dv u;  du = dv i;
//   dr = -s dL;  dz_a = dr r (1-r);  dz_x = di i (1-i);  dLambda += dL c r sigmoid(-Lambda).
// Block = (chunk of 64 tokens, sequence, 64 channels): a thread holds eight tokens x two adjacent channels.  h_{t-1} is run again from
// the state before the thread's tokens, u convolved again from x, so that 8 bytes of fp32 an element (r and i) are what the forward
// leaves behind.  At its 128 registers it spills some (56 and 68 bytes stored, 92 and 116 loaded, bf16 and fp32); with three blocks an SM
// it spilled more and was slower (forward and backward of B4 T1024 D1024 in 4 heads 230 -> 243 us), and with dy read again after the chain
// too (backward of B5 T1021 D1536 in 16 heads 242.6 -> 245.2).
struct SplitRevArgs {
    BwdArgs q;
    const float *conv_b, *h_seg;
    uint32_t *dz;         // [head][gate][plane][B T][dh] bf16
    Chain ch;
    int nchunk, ctiles;
};
constexpr int REV_CHUNK = 64;
struct RevShared {
    f32x2 agg[2][8][32], in_g[8][32], sums[3][8][32];
    int ok;
};

template <typename IOT, bool POLY>
__device__ __forceinline__ void reverse_chunk(const SplitRevArgs &p, RevShared &sh, int b, int link, int ct, f32x2 lam, f32x2 s, f32x2 (&r)[SEG], f32x2 (&dyv)[SEG]) {
    const BwdArgs &q = p.q;
    const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5, chunk = p.nchunk - 1 - link;
    const int T = q.T, D = q.D, dh = D / q.H, n = ct * 64 + 2 * lane;
    const bool cv = n < D;
    const int d = cv ? n : 0, t0 = chunk * REV_CHUNK + seg * SEG, nv = min(SEG, T - t0);   // nv may be <= 0
    const f32x2 ONE = pack2(1.0f, 1.0f), ZERO = pack2(0.0f, 0.0f), NEG = pack2(-1.0f, -1.0f);
    const IOT *x = (const IOT *)q.x, *cs = (const IOT *)q.cs_in, *cw = (const IOT *)q.conv_w;
    const size_t e0 = ((size_t)b * T + t0) * D + d;
    f32x2 f[SEG];
    f32x2 Q = ONE, G = ZERO;
#pragma unroll
    for (int i = SEG - 1; i >= 0; --i) {   // r = 0 for a token that does not exist: it passes g through
        f[i] = one_minus_decay2<POLY>(r[i], s);
        const f32x2 a = fma2(f[i], NEG, ONE);
        G = mul2(a, __fadd2_rn(dyv[i], G));
        Q = mul2(Q, a);
    }
    sh.agg[0][seg][lane] = Q; sh.agg[1][seg][lane] = G;
    __syncthreads();
    if (seg == 0) {
        uint4 *slot = p.ch.slot + (size_t)b * D + d;
        f32x2 cQ = ONE, cG = ZERO;   // the chunk as one step, before the wait
#pragma unroll
        for (int k = 7; k >= 0; --k) { cG = fma2(sh.agg[0][k][lane], cG, sh.agg[1][k][lane]); cQ = mul2(cQ, sh.agg[0][k][lane]); }
        f32x2 X = ZERO;
        float unused;
        bool ok = true;
        // past the last token g holds the gradient arriving on h_T (h_T = h_{T-1}, so it is carried with factor 1)
        if (link == 0) { if (q.dh_T) X = ld2f(q.dh_T + (size_t)b * D + d); }
        else ok = chain_wait(p.ch, slot, cv, link - 1, X.x, unused) && chain_wait(p.ch, slot + 1, cv, link - 1, X.y, unused);
        const f32x2 Xout = fma2(cQ, X, cG);
        if (ok && cv) {
            chain_put(p.ch, slot, link, Xout.x, 0.0f);
            chain_put(p.ch, slot + 1, link, Xout.y, 0.0f);
            if (chunk == 0 && q.dh0) *(float2 *)(q.dh0 + (size_t)b * D + d) = Xout;   // a_0 g_0: h0 enters Eq. 4 only at t = 0
        }
#pragma unroll
        for (int k = 7; k >= 0; --k) { sh.in_g[k][lane] = X; X = fma2(sh.agg[0][k][lane], X, sh.agg[1][k][lane]); }
        if (!ok) {
            if (cv) { chain_fail(p.ch, slot, link); chain_fail(p.ch, slot + 1, link); }
            sh.ok = 0;
        }
    }
    // u, i and h_{t-1} of the thread's tokens (while the first warp waits for the chain)
    f32x2 u[SEG], gi[SEG], hp[SEG];
    if (nv > 0) {
        f32x2 w[4], cb = p.conv_b ? ld2f(p.conv_b + d) : ZERO;
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = ld2(cw + (size_t)j * D + d);
        auto xat = [&](int t) -> f32x2 { return t >= 0 ? ld2(x + ((size_t)b * T + t) * D + d) : cs ? ld2(cs + ((size_t)b * 3 + (3 + t)) * D + d) : ZERO; };
        f32x2 x3 = xat(t0 - 3), x2 = xat(t0 - 2), x1 = xat(t0 - 1);
        f32x2 h = ld2f(p.h_seg + ((size_t)b * ((T + SEG - 1) / SEG) + t0 / SEG) * D + d);
        const float *pg = q.gi + e0;
        const IOT *px = x + e0;
#pragma unroll
        for (int i = 0; i < SEG; ++i) {
            gi[i] = i < nv ? ld2f(pg) : ZERO;
            u[i] = i < nv ? ld2(px) : ZERO;
            pg += D; px += D;
        }
#pragma unroll
        for (int i = 0; i < SEG; ++i) {
            const f32x2 x0 = u[i];
            u[i] = fma2(w[3], x3, fma2(w[2], x2, fma2(w[1], x1, fma2(w[0], x0, cb))));
            x3 = x2; x2 = x1; x1 = x0;
            f32x2 rm;
            hp[i] = h;
            h = fma2(fma2(f[i], NEG, ONE), h, mul2(input_scale2(f[i], rm), mul2(gi[i], u[i])));
        }
    }
    __syncthreads();
    if (!sh.ok) return;
    dependency_trigger();
    f32x2 carry = sh.in_g[seg][lane], s_lam = ZERO, s_ba = ZERO, s_bx = ZERO;
    const size_t plane = (size_t)q.B * T * dh / 2;   // of pairs
    const int head = d / dh;
    // from the last token of the segment backwards
    uint32_t *dz = p.dz + (size_t)head * 2 * PLANES * plane + (((size_t)b * T + t0 + SEG - 1) * dh + (d - head * dh)) / 2;
    float *pdu = q.hp + e0 + (size_t)(SEG - 1) * D;
    const f32x2 ns = mul2(s, NEG);
#pragma unroll
    for (int i = SEG - 1; i >= 0; --i) {
        if (i < nv && cv) {
            f32x2 rm;
            const f32x2 a = fma2(f[i], NEG, ONE), m = input_scale2(f[i], rm);
            const f32x2 g = __fadd2_rn(dyv[i], carry);
            carry = mul2(a, g);
            const f32x2 v = mul2(gi[i], u[i]);
            const f32x2 dLr = mul2(mul2(carry, fma2(mul2(a, v), mul2(rm, NEG), hp[i])), r[i]);   // dL r
            const f32x2 dv = mul2(g, m);
            const f32x2 dza = mul2(mul2(dLr, ns), fma2(r[i], NEG, ONE)), dzx = mul2(mul2(mul2(dv, u[i]), gi[i]), fma2(gi[i], NEG, ONE));
            s_lam = __fadd2_rn(s_lam, dLr);
            s_ba = __fadd2_rn(s_ba, dza); s_bx = __fadd2_rn(s_bx, dzx);
            uint32_t pa[PLANES], px[PLANES];
            split_planes(dza, pa); split_planes(dzx, px);
#pragma unroll
            for (int k = 0; k < PLANES; ++k) { dz[k * plane] = pa[k]; dz[(PLANES + k) * plane] = px[k]; }
            *(float2 *)pdu = mul2(dv, gi[i]);
        }
        dz -= dh / 2;
        pdu -= D;
    }
    sh.sums[0][seg][lane] = s_lam; sh.sums[1][seg][lane] = s_ba; sh.sums[2][seg][lane] = s_bx;
    __syncthreads();
    if (seg < 3 && cv) {
        f32x2 t = ZERO;
#pragma unroll
        for (int k = 0; k < 8; ++k) t = __fadd2_rn(t, sh.sums[seg][k][lane]);
        if (seg == 0) t = mul2(t, pack2(q.c / (1.0f + expf(lam.x)), q.c / (1.0f + expf(lam.y))));   // dL/dLambda = c r sigmoid(-Lambda)
        *(float2 *)(q.part_vec + ((size_t)(b * p.nchunk + chunk) * 3 + seg) * D + d) = t;
    }
}

template <typename IOT> __global__ void __launch_bounds__(256, 2) split_reverse_kernel(const SplitRevArgs p) {
    __shared__ RevShared sh;
    if (threadIdx.x == 0) sh.ok = 1;
    dependency_wait();
    int bid = blockIdx.x;
    const int ct = bid % p.ctiles; bid /= p.ctiles;
    const int b = bid % p.q.B, link = bid / p.q.B;   // last chunk first
    const int n = ct * 64 + 2 * (threadIdx.x & 31), D = p.q.D, t0 = (p.nchunk - 1 - link) * REV_CHUNK + (threadIdx.x >> 5) * SEG, nv = min(SEG, p.q.T - t0);
    const bool cv = n < D;
    const f32x2 lam = cv ? ld2f(p.q.lambda + n) : pack2(100.0f, 100.0f), ZERO = pack2(0.0f, 0.0f);
    f32x2 r[SEG], dyv[SEG];   // on their way while the decay rates are computed
    const size_t e0 = ((size_t)b * p.q.T + t0) * D + (cv ? n : 0);
    const float *pr = p.q.r + e0;
    const IOT *pd = (const IOT *)p.q.dy + e0;
#pragma unroll
    for (int i = 0; i < SEG; ++i) {
        r[i] = i < nv ? ld2f(pr) : ZERO;
        dyv[i] = i < nv ? ld2(pd) : ZERO;
        pr += D; pd += D;
    }
    const f32x2 s = pack2(decay_rate_acc(lam.x, p.q.c), decay_rate_acc(lam.y, p.q.c));
    // uniform over the block: every warp holds the same channels
    if (__all_sync(0xffffffffu, s.x <= S_POLY && s.y <= S_POLY)) reverse_chunk<IOT, true>(p, sh, b, link, ct, lam, s, r, dyv);
    else reverse_chunk<IOT, false>(p, sh, b, link, ct, lam, s, r, dyv);
}

// ------------------------------------------------------------------ du and dW
// Tiles of 128 x NT results, K in blocks of 64, in one launch:
//   dW: part[split][gate][head][o][n] = sum over the split's tokens of dz[tok][o] u[tok][n]   A = dz, B = u, both MN-major, K = tokens
//   du: du[tok][n] += sum over gates and o of dz[tok][o] W[o][n]                              A = dz, K-major; B = W, MN-major
// Per K block the planes of A and B arrive as tiles of 16 KB, A2 B0 first, then A1 A0 B1 B2 (bf16 weights: A1 A0), one thread copying A
// and one B, two K blocks in flight; the first two tiles are free again after A2 B0, A1 B0, A0 B0, the others after A1 B1, A0 B1, A0 B2.
// (With a barrier a tile, thirteen of them in a ring, and one thread for all copies, copies and products each cost their thread more
// than the tensor core: 72 us on B4 T1024 D1024 in 4 heads.)  After every two K blocks the epilogue warps add both accumulators to
// fp32 registers: 128 terms are what an accumulator takes (see the top of the file; with 256 dW of B1 T256 D256 was 3.9e-7 from the
// exact one, where the CUDA cores are 3.4e-7).
// Persistent blocks, one per SM, with two pairs of accumulators: a pair is drained while the products fill the other.
struct SplitProdArgs {
    alignas(64) CUtensorMap tm_dzk, tm_dzm;   // dz planes [6 H][B T][dh], boxes of 128 tokens x 64 and 64 tokens x 64
    alignas(64) CUtensorMap tm_u;             // u planes [3 H][B T][dh], box 64 tokens x 64
    alignas(64) CUtensorMap tm_wa, tm_wx;     // weights [planes x H][out][in], box 64 x 64
    int H, dh, D, NT, nt, mt, wplanes;
    int S, kb_split, dw_tiles, tiles;
    size_t ntok;
    float *du, *part;
    uint32_t *status;
    unsigned long long spin_ns;
};
constexpr uint32_t PROD_BAR = PROD_STAGES * 6 * TILE_BYTES, PROD_ALLOC = PROD_BAR + 256 + 1024;
constexpr int PROD_DRAIN = 2;

struct ProdTile { bool dw; int head, gate, split, m0, n0, kblocks; };
__device__ __forceinline__ ProdTile prod_tile(const SplitProdArgs &p, int i) {
    ProdTile t{};
    t.dw = i < p.dw_tiles;
    if (t.dw) {
        t.n0 = (i % p.nt) * p.NT; i /= p.nt;
        t.m0 = (i % p.mt) * 128; i /= p.mt;
        t.head = i % p.H; i /= p.H;
        t.gate = i & 1; t.split = i >> 1;
        const int total = (int)((p.ntok + 63) / 64);
        t.kblocks = min(p.kb_split, total - t.split * p.kb_split);
    } else {
        i -= p.dw_tiles;
        t.n0 = (i % p.nt) * p.NT; i /= p.nt;
        t.head = i % p.H; t.m0 = i / p.H * 128;
        t.kblocks = 2 * ((p.dh + 63) / 64);
    }
    return t;
}

__global__ void __launch_bounds__(PROD_THREADS, 1) split_products_kernel(const __grid_constant__ SplitProdArgs p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint32_t tmem_s;
    __shared__ volatile int abort_s;
    const uint32_t raw = smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;
    const uint32_t bar = base + PROD_BAR;
    // part 0: the tiles A2 B0 of a stage, part 1: the others
    auto FULL = [&](int st, int part) { return bar + 8u * (2 * st + part); };
    auto EMPTY = [&](int st, int part) { return bar + 8u * (2 * PROD_STAGES + 2 * st + part); };
    auto ACC_FULL = [&](int i) { return bar + 8u * (4 * PROD_STAGES + i); };
    auto ACC_EMPTY = [&](int i) { return bar + 8u * (4 * PROD_STAGES + 2 + i); };
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < 2 * PROD_STAGES; ++i) { mbar_init(FULL(i >> 1, i & 1), 2); mbar_init(EMPTY(i >> 1, i & 1), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(ACC_FULL(i), 1); mbar_init(ACC_EMPTY(i), 8); }
        abort_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 8) { tmem_alloc(smem_u32(&tmem_s), 512); tmem_relinquish(); }
    if (warp == 9 && lane == 0) { prefetch_tensormap(&p.tm_dzk); prefetch_tensormap(&p.tm_dzm); prefetch_tensormap(&p.tm_u); prefetch_tensormap(&p.tm_wa); prefetch_tensormap(&p.tm_wx); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_s;
    const int kslots = (p.dh + 63) / 64;
    dependency_wait();
    bool ok = true;
    if (warp >= 9) {
        if (lane == 0) {
            const bool is_a = warp == 9;
            int kbg = 0;   // K blocks so far
            for (int i = blockIdx.x; i < p.tiles && ok; i += gridDim.x) {
                const ProdTile t = prod_tile(p, i);
                const bool six = t.dw || p.wplanes == PLANES;
                for (int kb = 0; kb < t.kblocks && ok; ++kb, ++kbg) {
                    const int st = kbg % PROD_STAGES;
                    const uint32_t parity = ((kbg / PROD_STAGES) & 1) ^ 1, s0 = base + st * 6 * TILE_BYTES;
                    const int gate = kb >= kslots, k0 = t.dw ? (t.split * p.kb_split + kb) * 64 : (kb - gate * kslots) * 64;
                    auto load = [&](int tile, int plane, uint32_t full) {
                        const uint32_t dst = s0 + tile * TILE_BYTES;
                        if (is_a && !t.dw) tma_load_3d(dst, &p.tm_dzk, k0, t.m0, (t.head * 2 + gate) * PLANES + plane, full);
                        else {
                            const CUtensorMap *tm = t.dw ? (is_a ? &p.tm_dzm : &p.tm_u) : gate ? &p.tm_wx : &p.tm_wa;
                            const int c = is_a ? t.m0 : t.n0, row = !t.dw ? plane * p.H + t.head : (is_a ? t.head * 2 + t.gate : t.head) * PLANES + plane;
                            tma_load_3d(dst, tm, c, k0, row, full);
                            tma_load_3d(dst + TILE_BYTES / 2, tm, c + 64, k0, row, full);
                        }
                    };
                    ok = mbar_wait(EMPTY(st, 0), parity, p.spin_ns, (volatile int *)&abort_s);
                    if (!ok) break;
                    mbar_expect_tx(FULL(st, 0), TILE_BYTES);
                    load(is_a ? 0 : 1, is_a ? 2 : 0, FULL(st, 0));
                    if (!is_a && !six) { mbar_arrive(FULL(st, 1)); continue; }   // its wait is covered by the part-0 one of the next round
                    ok = mbar_wait(EMPTY(st, 1), parity, p.spin_ns, (volatile int *)&abort_s);
                    if (!ok) break;
                    mbar_expect_tx(FULL(st, 1), 2 * TILE_BYTES);
                    load(is_a ? 2 : 4, 1, FULL(st, 1));
                    load(is_a ? 3 : 5, is_a ? 0 : 2, FULL(st, 1));
                }
            }
        }
    } else if (warp == 8) {
        if (lane == 0) {
            const uint32_t id_mn = make_idesc(128, p.NT) | (1u << 15) | (1u << 16), id_bmn = make_idesc(128, p.NT) | (1u << 16);
            constexpr uint64_t TS = TILE_BYTES >> 4;
            int kbg = 0, drains = 0;   // K blocks so far, accumulator pairs handed over
            for (int i = blockIdx.x; i < p.tiles && ok; i += gridDim.x) {
                const ProdTile t = prod_tile(p, i);
                const bool six = t.dw || p.wplanes == PLANES;
                const uint32_t da = t.dw ? 2048 >> 4 : 32 >> 4, db = 2048 >> 4, id = t.dw ? id_mn : id_bmn;
                const uint64_t a_desc = t.dw ? make_desc_sw128_mn(base, TILE_BYTES / 2) : make_desc_sw128(base), b_desc = make_desc_sw128_mn(base, TILE_BYTES / 2);
                int in_acc = 0;
                for (int kb = 0; kb < t.kblocks; ++kb, ++kbg) {
                    const int st = kbg % PROD_STAGES;
                    const uint32_t parity = (kbg / PROD_STAGES) & 1, acc = tmem + (drains & 1) * 256;
                    const uint64_t A = a_desc + st * 6 * TS, B = b_desc + st * 6 * TS;
                    const bool full = t.dw || p.dh - (kb >= kslots ? kb - kslots : kb) * 64 >= 64, more = in_acc > 0;
                    if (in_acc == 0) ok = mbar_wait(ACC_EMPTY(drains & 1), ((drains >> 1) & 1) ^ 1, p.spin_ns, (volatile int *)&abort_s);
                    ok = ok && mbar_wait(FULL(st, 0), parity, p.spin_ns, (volatile int *)&abort_s);
                    if (!ok) break;
                    tc_fence_after();
                    mma_block(acc + 128, A, da, B + TS, db, id, more, full);                 // A2 B0
                    ok = mbar_wait(FULL(st, 1), parity, p.spin_ns, (volatile int *)&abort_s);
                    if (!ok) break;
                    tc_fence_after();
                    mma_block(acc + 128, A + 2 * TS, da, B + TS, db, id, true, full);        // A1 B0
                    mma_block(acc, A + 3 * TS, da, B + TS, db, id, more, full);              // A0 B0
                    tc_commit(EMPTY(st, 0));
                    if (six) {
                        mma_block(acc + 128, A + 2 * TS, da, B + 4 * TS, db, id, true, full);   // A1 B1
                        mma_block(acc + 128, A + 3 * TS, da, B + 4 * TS, db, id, true, full);   // A0 B1
                        mma_block(acc + 128, A + 3 * TS, da, B + 5 * TS, db, id, true, full);   // A0 B2
                    }
                    tc_commit(EMPTY(st, 1));
                    if (++in_acc == PROD_DRAIN || kb == t.kblocks - 1) {
                        tc_commit(ACC_FULL(drains & 1));
                        ++drains; in_acc = 0;
                    }
                }
            }
        }
    } else {
        const int q = warp & 3, half = warp >> 2;
        int drains = 0;
        for (int i = blockIdx.x; i < p.tiles && ok; i += gridDim.x) {
            const ProdTile t = prod_tile(p, i);
            const int row = t.m0 + q * 32 + lane, c0 = t.n0 + half * 64;
            const bool valid = t.dw ? row < p.dh : (size_t)row < p.ntok;
            float *dst = t.dw ? p.part + ((((size_t)t.split * 2 + t.gate) * p.H + t.head) * p.dh + row) * p.dh + c0 : p.du + (size_t)row * p.D + t.head * p.dh + c0;
            f32x2 sum[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) sum[j] = pack2(0.f, 0.f);
            if (!t.dw && valid) {   // the direct part of du, on its way while the products run
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (half * 64 + j * 8 < p.NT && c0 + j * 8 < p.dh) {
                        uint32_t o[8];
                        ld_global_v8(dst + 8 * j, o);
#pragma unroll
                        for (int e = 0; e < 4; ++e) sum[4 * j + e] = pack2(__uint_as_float(o[2 * e]), __uint_as_float(o[2 * e + 1]));
                    }
                }
            }
            const int rounds = (t.kblocks + PROD_DRAIN - 1) / PROD_DRAIN;
            for (int r = 0; r < rounds; ++r, ++drains) {
                const int acc = drains & 1;
                ok = warp_wait(ACC_FULL(acc), (drains >> 1) & 1, p.spin_ns, (volatile int *)&abort_s);
                if (!ok) break;
                tc_fence_after();
                const uint32_t tm = tmem + ((uint32_t)(q * 32) << 16) + acc * 256 + half * 64;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (half * 64 + j * 16 < p.NT) {
                        f32x2 v[8], w[8];
                        tmem_ld16(tm + j * 16, v); tmem_ld16(tm + 128 + j * 16, w);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 8; ++e) sum[8 * j + e] = __fadd2_rn(sum[8 * j + e], __fadd2_rn(v[e], w[e]));
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(ACC_EMPTY(acc));
            }
            if (valid && ok) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (half * 64 + j * 8 < p.NT && c0 + j * 8 < p.dh) {
                        uint32_t o[8];
#pragma unroll
                        for (int e = 0; e < 4; ++e) { o[2 * e] = __float_as_uint(sum[4 * j + e].x); o[2 * e + 1] = __float_as_uint(sum[4 * j + e].y); }
                        st_global_v8(dst + 8 * j, o);
                    }
                }
            }
        }
    }
    dependency_trigger();
    if (!ok && lane == 0) { abort_s = 1; atomicExch(p.status, STATUS_MAGIC | (uint32_t)RGLRU_ERR_TIMEOUT); }
    tc_fence_before();
    __syncthreads();
    if (abort_s) {   // let copies and MMAs in flight land before shared and tensor memory are given back
        const uint64_t tw = gtimer();
        while (gtimer() - tw < 50000ull) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 8) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------ host side
inline bool width_ok(int D, int H) { return H > 0 && D % H == 0 && (D / H) % 32 == 0 && D / H <= GENERIC_MAX_DH; }

bool plane_map(CUtensorMap *tm, const void *ptr, uint64_t inner, uint64_t rows, uint64_t planes, uint32_t box0, uint32_t box1) {
    const uint64_t dims[3] = {inner, rows, planes}, strides[2] = {inner * 2, inner * rows * 2};
    const uint32_t box[3] = {box0, box1, 1};
    return encode_map16_3d(tm, ptr, dims, strides, box, true);
}

// Tokens per block of the forward: 64, or 32 while that gives every block an SM of its own.  fp32 step with 64 / 32 tokens, us: B2 T100
// D1024 in 8 heads (64 blocks of 32) 58.3 / 53.3, B3 T190 D1024 in 4 (144) 83.5 / 78.8, B3 T250 (192) 91 / 107, B4 T250 (256) 108 / 124.
// Fp32 calls and backwards of heads wider than 640 too: see forward().
int fwd_tokens(int B, int T, int D, int H, bool exact) {
    const size_t blocks32 = (size_t)ceil_div(T, 32) * B * H * ceil_div(D / H, 128);
    return blocks32 <= (size_t)num_sms() || (exact && D / H > 640) ? 32 : 64;
}

template <typename IOT, bool SAVE, bool LATE, int TOK>
cudaError_t launch_forward(SplitFwdArgs &p, cudaStream_t st) {
    static PerDeviceOptIn opt_in;
    cudaError_t e = opt_in.ensure(split_forward_kernel<IOT, SAVE, LATE, TOK>, (int)FwdSmem<TOK>::ALLOC);
    if (e != cudaSuccess) return e;
    p.nchunk = ceil_div(p.f.T, TOK);
    p.sets = TOK == 32 && LATE ? ceil_div(ceil_div(p.f.D / p.f.H, 64), 4) : 1;
    for (p.cols = 4 * TOK; p.cols < (uint32_t)(4 * TOK * p.sets); p.cols *= 2) {}
    const size_t grid = (size_t)p.nchunk * p.f.B * p.f.H * p.mtiles;
    if (grid > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
    return launch_dependent(split_forward_kernel<IOT, SAVE, LATE, TOK>, dim3((unsigned)grid), dim3(FWD_THREADS), FwdSmem<TOK>::ALLOC, st, p);
}
// The weights as the products read them: the caller's (bf16), or their planes (fp32), made here in `planes`
cudaError_t weight_planes(const FwdArgs &f, int io, void *planes, const void *&wa, const void *&wx, cudaStream_t st) {
    if (io == RGLRU_BF16) { wa = f.W_a; wx = f.W_x; return cudaSuccess; }
    const size_t n = (size_t)f.D * (f.D / f.H), n2 = n / 2;
    wa = planes; wx = (const char *)planes + PLANES * n * 2;
    return launch_dependent(split_weights_kernel, dim3((unsigned)ceil_div(2 * n2, 256)), dim3(256), 0, st, (const float *)f.W_a, (const float *)f.W_x, (uint32_t *)planes, n2);
}
size_t weight_plane_bytes(int D, int H, int io) { return io == RGLRU_F32 ? up256((size_t)2 * PLANES * D * (D / H) * 2) : 0; }

// How many leading products an accumulator takes.  Fp32 calls and backwards are promised the accuracy of fp32 FMAs: no output may be
// further from the exact one than the CUDA cores' own.  The worst one's share of theirs (fp32, B40 T64, where little else hides the
// gates' error), all in one accumulator / the last two K blocks in Y / sets of at most four K blocks, 32 tokens: width 256 0.88 / 0.78 / -,
// 352 0.94 / 0.83 / -, 512 1.07 / 0.88 / 0.82, 640 1.19 / 0.98 / 0.77, 768 1.31 / 1.08 / 0.73, 1024 1.61 / 1.35 / 0.80.  Forward and
// backward of B4 T1024 D1024, us: width 256 249 / 254 / -, 512 334 / 356 / 551, 1024 526 / 540 / 931 (CUDA cores 1895).  The bf16 prefill
// has always had the first: B3 T1213 D4096 of width 1024 311 / 317 us.
template <bool SAVE>
cudaError_t forward(SplitFwdArgs &p, int io, const void *wa, const void *wx, cudaStream_t st) {
    const int dh = p.f.D / p.f.H;
    p.mtiles = ceil_div(dh, 128);
    p.wplanes = io == RGLRU_F32 ? PLANES : 1;
    if (!plane_map(&p.tm_wa, wa, dh, dh, (uint64_t)p.wplanes * p.f.H, 64, 128) || !plane_map(&p.tm_wx, wx, dh, dh, (uint64_t)p.wplanes * p.f.H, 64, 128)) return cudaErrorNotSupported;
    const bool wide = fwd_tokens(p.f.B, p.f.T, p.f.D, p.f.H, SAVE || io == RGLRU_F32) == 64, late = dh > 256;
    if (io == RGLRU_F32) {
        if (late) return wide ? launch_forward<float, SAVE, true, 64>(p, st) : launch_forward<float, SAVE, true, 32>(p, st);
        return wide ? launch_forward<float, SAVE, false, 64>(p, st) : launch_forward<float, SAVE, false, 32>(p, st);
    }
    if (SAVE && late) return wide ? launch_forward<__nv_bfloat16, SAVE, SAVE, 64>(p, st) : launch_forward<__nv_bfloat16, SAVE, SAVE, 32>(p, st);
    return wide ? launch_forward<__nv_bfloat16, SAVE, false, 64>(p, st) : launch_forward<__nv_bfloat16, SAVE, false, 32>(p, st);
}

// Token splits of dW: at least four K blocks each, at most `most` splits.  Four blocks of six products are as long as a tile of du of an
// fp32 head 128 wide; from 8192 tokens on a split is longer, since the parts are memory.  Neither the SMs nor the number of dW tiles
// enter: one narrow head leaves most SMs without one.  (One split beside the 640 tiles of du of B5 T1021 D1536 in 16 heads: 224 us, where
// the products take 61 now.)
int dw_split(size_t ntok, int most, int &kb_split) {
    const int total = ceil_div(ntok, 64);
    kb_split = ceil_div(total, most) > 4 ? ceil_div(total, most) : 4;
    return ceil_div(total, kb_split);
}

// The workspace of the backward holds r, i and du in fp32 and the planes of u and of dz, 30 bytes an element, where the CUDA cores'
// backward has 16.  So a call that would need more than 4 GiB goes through its sequences in two passes or three, one after the other in
// the same arrays, as many as it takes to need no more than they do.  Passes cost 1 to 8 % (B8 T2048 D4096 in 16 heads 2194 -> 2245 us,
// B2 T16384 in 32 heads 3469 -> 3734), which smaller calls need not pay.  (r and i in the place of dz, 22 bytes in one pass: reverse scan
// 78 -> 88 us, forward 90 -> 96 on B5 T1021 D1536 in 16 heads.)
struct BwdPlan {
    int seqs;            // of a pass
    int passes, splits;  // splits of dW over all passes
    size_t conv_rows;    // rows of part_conv over all passes
};
constexpr size_t ONE_PASS_BYTES = (size_t)4 << 30;
BwdPlan bwd_plan(int B, int T, int D) {
    BwdPlan L{};
    L.passes = 1;
    if ((size_t)B * T * D * 30 > ONE_PASS_BYTES)
        while (L.passes < B && ceil_div(B, L.passes) * 30 > B * 16) ++L.passes;
    L.seqs = ceil_div(B, L.passes);
    for (int b0 = 0; b0 < B; b0 += L.seqs) {
        const int n = B - b0 < L.seqs ? B - b0 : L.seqs;
        int kb;
        L.splits += dw_split((size_t)n * T, 32 / L.passes, kb);
        L.conv_rows += (size_t)n * conv_backward_chunks(n, T, D);
    }
    return L;
}

}  // namespace

// The fp32 forward of a few tokens is left to the CUDA cores: the weights as planes are a launch of their own and 1.5 times the bytes, and
// while the blocks of 32 tokens x 32 channels of the other kernel have an SM each (two to an SM up to width 128) it takes no longer for all
// of them than for one.  Split products / CUDA cores, us: B1 T1 D1024, widths 32 9.5 / 6.6, 128 12.1 / 10.2, 256 16.7 / 15.0, 1024 44.9 / 43.6;
// D4096, width 256, T32 (128 blocks) 19.9 / 15.8, T64 (256) 20.6 / 27.4; width 128, T64 (256) 14.3 / 14.2, T128 (512) 15.6 / 24.8; width 32,
// T64 (256) 12.6 / 8.5.  Beyond 128 tokens the two cross between 256 and 1024 (D256, width 32: T256 12.5 / 10.7, T1024 17.5 / 23.6), and
// the state of the CUDA cores' kernel is further from the exact one with every token (y: 2 times as far as this one's after 64, 4 after 500),
// so that those calls stay here; width 32, where three of four rows of a block have no channel, too (B8 T4096 D1024 755 / 717).
// The backward of any size is faster here from 32 tokens on (width 32 of D4096 from 128: T64 40.2 / 37.1), before that within 10 %
// (width 32: 8 us).
bool split_prefill_supported(int B, int T, int D, int H, int io) {
    if (!width_ok(D, H)) return false;
    const int dh = D / H;
    const size_t blocks = (size_t)B * H * ceil_div(T, 32) * ceil_div(dh, 32);
    return io != RGLRU_F32 || T > 128 || blocks > (dh <= 128 ? 296 : 148);
}
bool split_backward_supported(int D, int H) { return width_ok(D, H); }

// chain records | private copy of conv_state_in (see generic_prefill) | planes of the weights
size_t split_prefill_workspace_bytes(int B, int D, int H, int io) {
    return up256((size_t)B * D * sizeof(uint4)) + up256((size_t)B * 3 * D * (io == RGLRU_F32 ? 4 : 2)) + weight_plane_bytes(D, H, io);
}

cudaError_t split_prefill(const FwdArgs &a, int io, void *ws_body, cudaStream_t st) {
    SplitFwdArgs p{};
    p.f = a;
    char *ws = (char *)ws_body, *copy = ws + up256((size_t)a.B * a.D * sizeof(uint4));
    const size_t cs_bytes = (size_t)a.B * 3 * a.D * (io == RGLRU_F32 ? 4 : 2);
    p.ch = make_chain((uint4 *)ws, a);
    const uintptr_t ci = (uintptr_t)a.cs_in, co = (uintptr_t)a.cs_out;
    cudaError_t e;
    if (ci && ci < co + cs_bytes && co < ci + cs_bytes) {
        if ((e = cudaMemcpyAsync(copy, a.cs_in, cs_bytes, cudaMemcpyDeviceToDevice, st)) != cudaSuccess) return e;
        p.f.cs_in = copy;
    }
    const void *wa, *wx;
    if ((e = weight_planes(a, io, copy + up256(cs_bytes), wa, wx, st)) != cudaSuccess) return e;
    return forward<false>(p, io, wa, wx, st);
}

size_t split_backward_workspace_bytes(int B, int T, int D, int H, int io) {
    const BwdPlan L = bwd_plan(B, T, D);
    const size_t ntok = (size_t)L.seqs * T, dh = D / H;
    size_t bytes = 3 * up256(ntok * D * 4);                                    // r, i, du
    bytes += up256(ntok * D * PLANES * 2) + up256(ntok * D * 2 * PLANES * 2);  // planes of u and dz
    bytes += up256((size_t)L.seqs * ceil_div(T, SEG) * D * 4);
    bytes += up256((size_t)B * ceil_div(T, REV_CHUNK) * 3 * D * 4) + up256(L.conv_rows * 5 * D * 4);
    bytes += up256((size_t)L.splits * 2 * D * dh * 4) + 2 * up256((size_t)L.seqs * D * sizeof(uint4));
    return bytes + weight_plane_bytes(D, H, io);
}

cudaError_t split_backward(const FwdArgs &fwd, BwdArgs &q_all, int io, void *ws_body, cudaStream_t st) {
    const int T = fwd.T, D = fwd.D, H = fwd.H, dh = D / H, rchunks = ceil_div(T, REV_CHUNK);
    const BwdPlan L = bwd_plan(fwd.B, T, D);
    const size_t most = (size_t)L.seqs * T, wsz = (size_t)D * dh, iob = io == RGLRU_F32 ? 4 : 2;
    char *at = (char *)ws_body;
    auto take = [&](size_t bytes) { char *r = at; at += up256(bytes); return r; };
    float *rr = (float *)take(most * D * 4), *gi = (float *)take(most * D * 4), *du = (float *)take(most * D * 4);
    char *u_planes = take(most * D * PLANES * 2), *dz = take(most * D * 2 * PLANES * 2);
    float *h_seg = (float *)take((size_t)L.seqs * ceil_div(T, SEG) * D * 4);
    q_all.part_vec = (float *)take((size_t)fwd.B * rchunks * 3 * D * 4);
    q_all.part_conv = (float *)take(L.conv_rows * 5 * D * 4);
    q_all.part_dw = (float *)take((size_t)L.splits * 2 * wsz * 4);
    uint4 *slots_f = (uint4 *)take((size_t)L.seqs * D * sizeof(uint4)), *slots_r = (uint4 *)take((size_t)L.seqs * D * sizeof(uint4));
    char *planes = take(weight_plane_bytes(D, H, io));
    cudaError_t e;
    const void *wa, *wx;
    if ((e = weight_planes(fwd, io, planes, wa, wx, st)) != cudaSuccess) return e;
    const uint64_t w3 = io == RGLRU_F32 ? PLANES : 1;
    size_t splits = 0, conv_rows = 0;   // of the passes so far
    for (int b0 = 0; b0 < fwd.B; b0 += L.seqs) {
        const int B = fwd.B - b0 < L.seqs ? fwd.B - b0 : L.seqs;
        const size_t ntok = (size_t)B * T, x0 = (size_t)b0 * T * D * iob, c0 = (size_t)b0 * 3 * D * iob, h0 = (size_t)b0 * D;
        auto from = [](const void *ptr, size_t bytes) -> const void * { return ptr ? (const char *)ptr + bytes : nullptr; };
        // this pass's share of what has a batch dimension
        FwdArgs f = fwd;
        f.B = B; f.x = from(f.x, x0); f.cs_in = from(f.cs_in, c0); f.h0 = (const float *)from(f.h0, h0 * 4);
        f.gate_branch = nullptr;
        BwdArgs q = q_all;
        q.B = B; q.x = f.x; q.cs_in = f.cs_in; q.dy = from(q.dy, x0); q.dx = (void *)from(q.dx, x0);
        q.dh_T = (const float *)from(q.dh_T, h0 * 4); q.dcs_out = from(q.dcs_out, c0);
        q.dh0 = (float *)from(q.dh0, h0 * 4); q.dcs_in = (void *)from(q.dcs_in, c0);
        q.r = rr; q.gi = gi; q.hp = du;
        q.nchunk = conv_backward_chunks(B, T, D);
        q.part_vec += (size_t)b0 * rchunks * 3 * D;
        q.part_conv += conv_rows * 5 * D;
        q.part_dw += splits * 2 * wsz;
        SplitProdArgs g{};
        g.S = dw_split(ntok, 32 / L.passes, g.kb_split);
        splits += g.S; conv_rows += (size_t)B * q.nchunk;
        // forward sweep
        SplitFwdArgs p{};
        p.f = f;
        p.f.save_r = q.r; p.f.save_i = q.gi;
        p.u_planes = (uint32_t *)u_planes; p.h_seg = h_seg;
        p.ch = make_chain(slots_f, f);
        if ((e = forward<true>(p, io, wa, wx, st)) != cudaSuccess) return e;
        // reverse scan and adjoints
        SplitRevArgs r{};
        r.q = q; r.conv_b = f.conv_b; r.h_seg = h_seg; r.dz = (uint32_t *)dz; r.ch = make_chain(slots_r, f);
        r.nchunk = rchunks; r.ctiles = ceil_div(D, 64);
        const size_t rgrid = (size_t)rchunks * B * r.ctiles;
        if (rgrid > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
        if ((e = launch_dependent(io == RGLRU_F32 ? split_reverse_kernel<float> : split_reverse_kernel<__nv_bfloat16>, dim3((unsigned)rgrid), dim3(256), 0, st, r)) != cudaSuccess) return e;
        // du += W^T dz, dW = dz^T u
        if (!plane_map(&g.tm_dzk, dz, dh, ntok, (uint64_t)2 * PLANES * H, 64, 128) || !plane_map(&g.tm_dzm, dz, dh, ntok, (uint64_t)2 * PLANES * H, 64, 64) ||
            !plane_map(&g.tm_u, u_planes, dh, ntok, (uint64_t)PLANES * H, 64, 64) || !plane_map(&g.tm_wa, wa, dh, dh, w3 * H, 64, 64) || !plane_map(&g.tm_wx, wx, dh, dh, w3 * H, 64, 64))
            return cudaErrorNotSupported;
        g.H = H; g.dh = dh; g.D = D; g.wplanes = (int)w3; g.ntok = ntok;
        g.nt = ceil_div(dh, 128); g.mt = g.nt; g.NT = ceil_div(ceil_div(dh, g.nt), 32) * 32;
        g.du = q.hp; g.part = q.part_dw; g.status = f.status; g.spin_ns = g_spin_limit_ns;
        const size_t dw = (size_t)g.S * 2 * H * g.mt * g.nt, tiles = dw + (size_t)ceil_div(ntok, 128) * H * g.nt;
        if (tiles > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
        g.dw_tiles = (int)dw; g.tiles = (int)tiles;
        const int sms = num_sms();
        static PerDeviceOptIn opt_in;
        if ((e = opt_in.ensure(split_products_kernel, (int)PROD_ALLOC)) != cudaSuccess) return e;
        if ((e = launch_dependent(split_products_kernel, dim3((unsigned)(tiles < (size_t)sms ? tiles : sms)), dim3(PROD_THREADS), PROD_ALLOC, st, g)) != cudaSuccess) return e;
        if ((e = conv_backward(q, io, q.hp, false, st)) != cudaSuccess) return e;
        if ((e = state_conv_grads(q, io, q.hp, false, st)) != cudaSuccess) return e;   // after dx: it rewrites the rows conv_state_out copies
    }
    ReduceJobs jobs{};
    add_reduce_job(jobs, q_all.part_dw, (int)splits, 2 * wsz, q_all.dW_a, wsz, q_all.dW_x, wsz, nullptr, 0);
    add_reduce_job(jobs, q_all.part_vec, fwd.B * rchunks, (size_t)3 * D, q_all.dlambda, D, q_all.db_a, D, q_all.db_x, D);
    add_reduce_job(jobs, q_all.part_conv, (int)conv_rows, (size_t)5 * D, q_all.dconv_w, (size_t)4 * D, q_all.dconv_b, D, nullptr, 0);
    return run_reduce_jobs(jobs, st);
}

}  // namespace rglru
