// Shape-generic CUDA-core kernels for the RG-LRU temporal core: any head width up to
// GENERIC_MAX_DH, fp32 or bf16 io, accurate libm-grade transcendental functions, fp32 throughout.
// They serve every shape without a tensor-core kernel: head widths that are no multiple of 32, the decode step of fp32 io, and the fp32
// prefill of few tokens.
//
// Every contraction (gate products W_a u, W_x u of Eq. 1-2; du = W^T dz; dW = dz^T u) is a register-blocked fp32 product on
// packed FMAs: 128 threads own BM x 2 BM results, 2 TM NH = BM * BM / 64 each (64 for BM = 64), operands staged K-major
// through double-buffered shared memory with the next slab's global loads in flight.  At BM = 64 a thread does 64 FMAs per
// four 16-byte shared loads, so the FMA pipe and not shared memory bounds it.  BM = 32 is the same code with a quarter of the
// work per block, for problems whose 64-tiles would not fill the SMs twice (see tile_rows).
// Time is cut into chunks of BM tokens.  The forward and the reverse scan run from zero state inside a chunk, in registers,
// and the chunks of a channel are chained through one 16-byte record per (sequence, channel): block order is chunk-major, so
// a block only ever waits for blocks that were dispatched before it.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "rglru_chain.cuh"
#include "rglru_gates32.cuh"
#include "rglru_internal.h"
#include "sm100_ptx.cuh"

namespace rglru {
namespace {

using ptx::f32x2;
using ptx::fma2;
using ptx::pack2;

constexpr int NT = 256;  // threads per block of the element-wise and decode kernels
constexpr int GT = 16;   // sequences per tile of the decode kernel
constexpr int NB = 16;   // input channels per staged weight slab of the decode kernel
constexpr int MT = 128;  // threads per block of the contractions

__device__ __forceinline__ float tof(float v) { return v; }
__device__ __forceinline__ float tof(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float ldf(const float *p, size_t i) { return p[i]; }
__device__ __forceinline__ float ldf(const __nv_bfloat16 *p, size_t i) { return __bfloat162float(p[i]); }
__device__ __forceinline__ void stf(float *p, size_t i, float v) { p[i] = v; }
__device__ __forceinline__ void stf(__nv_bfloat16 *p, size_t i, float v) { p[i] = __float2bfloat16_rn(v); }
// four consecutive elements (address a multiple of four elements)
__device__ __forceinline__ void ld4(const float *p, float *v) {
    const float4 t = *(const float4 *)p;
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void ld4(const __nv_bfloat16 *p, float *v) {
    const uint2 t = *(const uint2 *)p;
    v[0] = __uint_as_float(t.x << 16); v[1] = __uint_as_float(t.x & 0xFFFF0000u);
    v[2] = __uint_as_float(t.y << 16); v[3] = __uint_as_float(t.y & 0xFFFF0000u);
}

__device__ __forceinline__ float sigmoid_acc(float z) { return 1.0f / (1.0f + expf(-z)); }

// s = c * softplus(-Lambda) = -c log sigmoid(Lambda)   (Appendix A, with a = sigmoid(Lambda))
__device__ __forceinline__ float decay_rate(float lambda, float c) {
    float z = -lambda;
    float sp = z > 0.0f ? z + log1pf(expf(-z)) : log1pf(expf(z));
    return c * sp;
}
// a_t = exp(-s r), m_t = sqrt(1 - a_t^2) = sqrt(-expm1(-2 s r))   (Eq. 3-4)
__device__ __forceinline__ void decay(float s, float r, float &a, float &m) {
    float L = -s * r;
    a = expf(L);
    m = sqrtf(fmaxf(0.0f, -expm1f(2.0f * L)));
}

// x_{tau} of sequence b for tau in [-3, T): history comes from conv_state_in (oldest first) or is zero
template <typename IOT>
__device__ __forceinline__ float x_at(const IOT *x, const IOT *cs_in, int T, int D, int b, int tau, int d) {
    if (tau >= 0) return ldf(x, ((size_t)b * T + tau) * D + d);
    if (cs_in == nullptr) return 0.0f;
    return ldf(cs_in, ((size_t)b * 3 + (3 + tau)) * D + d);
}
template <typename IOT>
__device__ __forceinline__ IOT x_raw_at(const IOT *x, const IOT *cs_in, int T, int D, int b, int tau, int d) {
    if (tau >= 0) return x[((size_t)b * T + tau) * D + d];
    if (cs_in == nullptr) return IOT(0.0f);
    return cs_in[((size_t)b * 3 + (3 + tau)) * D + d];
}

// r, i, a, m of Eq. 1-4 for one token of one channel.  A function of its own: inlined for each of a thread's 8 x 4 results it was
// some five thousand instructions, which every block fetched once.
__device__ __noinline__ float4 gates_acc(float za, float zx, float s) {
    const float r = sigmoid_acc(za), g = sigmoid_acc(zx);
    float a, m;
    decay(s, r, a, m);
    return make_float4(r, g, a, m);
}

// ------------------------------------------------------------------ register-blocked fp32 product
// Geometry of a block: 128 threads as 8 (rows) x 16 (columns); BM rows x 2 BM columns of results.  Thread (ty, tx) owns rows
// TM ty .. TM ty + TM - 1 and columns NH tx .. + NH - 1 of each half of the columns (in the forward the halves are the two
// gates of the same channels).
// A slab is BK deep: small blocks, of which an SM holds one or two, take twice the depth so that fewer rounds of load latency
// are exposed.
template <int BM> struct Tile {
    static constexpr int BN = 2 * BM, TM = BM / 8, NH = BM / 16, BK = BM == 64 ? 16 : 32;
    static constexpr int TA = BM * BK / MT, EB = BN * BK / MT;   // values of the A and B slab a thread brings in
    static constexpr int AS = BM + 4, BS = BN + 4;   // row strides in shared memory (floats): 16-byte rows, shifted by one bank group
    float As[2][BK][AS], Bs[2][BK][BS];
};

template <int BM>
__device__ __forceinline__ void mul_slab(const Tile<BM> &s, int buf, int ty, int tx, f32x2 (&acc)[Tile<BM>::TM][Tile<BM>::NH]) {
    constexpr int TM = Tile<BM>::TM, NH = Tile<BM>::NH;
#pragma unroll
    for (int k = 0; k < Tile<BM>::BK; ++k) {
        float a[TM];
        f32x2 b[NH];
#pragma unroll
        for (int i = 0; i < TM; i += 4) {
            const float4 t = *(const float4 *)&s.As[buf][k][ty * TM + i];
            a[i] = t.x; a[i + 1] = t.y; a[i + 2] = t.z; a[i + 3] = t.w;
        }
#pragma unroll
        for (int half = 0; half < 2; ++half) {
#pragma unroll
            for (int j = 0; j < NH; j += 2) b[half * (NH / 2) + j / 2] = *(const f32x2 *)&s.Bs[buf][k][half * BM + tx * NH + j];
        }
#pragma unroll
        for (int i = 0; i < TM; ++i) {
#pragma unroll
            for (int j = 0; j < NH; ++j) acc[i][j] = fma2(pack2(a[i], a[i]), b[j], acc[i][j]);
        }
    }
}
// column j (0 .. NH - 1) of half `half` of this thread's row i
template <int NH> __device__ __forceinline__ float col(const f32x2 (&row)[NH], int half, int j) {
    const f32x2 p = row[half * (NH / 2) + j / 2];
    return (j & 1) ? p.y : p.x;
}
// A BK x W block of a row-major matrix (rows = K index, W contiguous columns) on its way to shared memory: 128 threads,
// BK W / 128 values each, by fours of one row when the addresses allow it.
template <int W, int N, bool VEC, typename T>
__device__ __forceinline__ void fetch_rows(const T *src, size_t stride, int rows_valid, int cols_valid, int tid, float (&v)[N]) {
    if (VEC) {
#pragma unroll
        for (int i = 0; i < N / 4; ++i) {
            const int e = tid + MT * i, k = e / (W / 4), n = (e % (W / 4)) * 4;
            if (k < rows_valid && n < cols_valid) ld4(src + (size_t)k * stride + n, v + 4 * i);
            else { v[4 * i] = 0.f; v[4 * i + 1] = 0.f; v[4 * i + 2] = 0.f; v[4 * i + 3] = 0.f; }
        }
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int e = tid + MT * i, k = e / W, n = e % W;
            v[i] = k < rows_valid && n < cols_valid ? tof(src[(size_t)k * stride + n]) : 0.0f;
        }
    }
}
template <int W, int N, bool VEC, int K, int S>
__device__ __forceinline__ void put_rows(float (&dst)[K][S], int tid, const float (&v)[N]) {
    if (VEC) {
#pragma unroll
        for (int i = 0; i < N / 4; ++i) {
            const int e = tid + MT * i, k = e / (W / 4), n = (e % (W / 4)) * 4;
            *(float4 *)&dst[k][n] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) { const int e = tid + MT * i; dst[e / W][e % W] = v[i]; }
    }
}
// E consecutive K values of one row of a matrix whose rows run along K (it is transposed on its way to shared memory)
template <int E, bool VEC, typename T> __device__ __forceinline__ void fetch_k(const T *row, bool row_valid, int k_valid, float (&v)[E]) {
    if (VEC) {
#pragma unroll
        for (int i = 0; i < E; i += 4) {
            if (row_valid && i < k_valid) ld4(row + i, v + i);
            else { v[i] = 0.f; v[i + 1] = 0.f; v[i + 2] = 0.f; v[i + 3] = 0.f; }
        }
    } else {
#pragma unroll
        for (int i = 0; i < E; ++i) v[i] = row_valid && i < k_valid ? tof(row[i]) : 0.0f;
    }
}

// ------------------------------------------------------------------ forward
// Block = (chunk of BM tokens, sequence, head, BM output channels): Conv1D on the way into shared memory, both gate products,
// gates and decay on the results in registers, scan of each thread's TM tokens from zero state, the 8 row groups combined
// through shared memory, chain to the previous chunk, y.  u, r, i, a, v never leave the block.  With SAVE (the backward's
// forward sweep) u, r, i and h_{t-1} go to fp32 arrays instead of y.
// Against one block per (head, sequence) walking the whole of T: 4 x 1024 x 1024 (4 heads), fp32, ran at 1.8 TFLOP/s there.
template <typename IOT, bool SAVE, int BM, bool VEC>
__global__ void __launch_bounds__(MT, BM == 64 ? 3 : 6) generic_forward_kernel(FwdArgs a, Chain ch, int nchunk, int ntile) {
    ptx::dependency_wait();
    using TL = Tile<BM>;
    constexpr int TM = TL::TM, NH = TL::NH, BK = TL::BK, TA = TL::TA, EB = TL::EB;
    __shared__ __align__(16) TL s;
    __shared__ float agg_P[8][BM], agg_h[8][BM], in_h[8][BM];
    __shared__ int ok_s;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int Dh = a.D / a.H, D = a.D, T = a.T;
    int bid = blockIdx.x;
    const int nt = bid % ntile; bid /= ntile;
    const int head = bid % a.H; bid /= a.H;
    const int b = bid % a.B, chunk = bid / a.B;
    const int d0 = head * Dh, n0 = nt * BM, t0 = chunk * BM;
    const IOT *x = (const IOT *)a.x, *cw = (const IOT *)a.conv_w, *cs_in = (const IOT *)a.cs_in;
    const IOT *xb = x + (size_t)b * T * D;
    if (tid == 0) ok_s = 1;

    // A operand: this thread convolves channel kk of each slab for tokens TA seg .. + TA - 1 of the chunk
    const int kk = tid % BK, seg = tid / BK, ta = t0 + seg * TA;
    // B operand: row br of the 2 BM weight rows (both gates), EB consecutive input channels from koff
    const int br = tid % TL::BN, koff = (tid / TL::BN) * EB;
    const int bch = n0 + (br % BM);
    const IOT *wrow = (const IOT *)(br < BM ? a.W_a : a.W_x) + ((size_t)head * Dh + (bch < Dh ? bch : 0)) * Dh + koff;
    float xr[TA + 3], taps[4], cb, wv[EB];
    auto fetch = [&](int k0) {
        const int k = k0 + kk, d = d0 + k;
        const bool kv = k < Dh;
#pragma unroll
        for (int i = 0; i < TA + 3; ++i) {
            const int t = ta - 3 + i;
            float v = 0.0f;
            if (kv) {
                if (t >= 0) { if (t < T) v = ldf(xb, (size_t)t * D + d); }
                else if (cs_in) v = ldf(cs_in, ((size_t)b * 3 + (3 + t)) * D + d);
            }
            xr[i] = v;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) taps[j] = kv ? ldf(cw, (size_t)j * D + d) : 0.0f;
        cb = kv && a.conv_b ? a.conv_b[d] : 0.0f;
        fetch_k<EB, VEC>(wrow + k0, bch < Dh, Dh - k0 - koff, wv);
    };
    auto stage = [&](int buf) {
        float u[TA];
#pragma unroll
        for (int i = 0; i < TA; ++i) {
            u[i] = fmaf(taps[0], xr[i + 3], cb);
#pragma unroll
            for (int j = 1; j < 4; ++j) u[i] = fmaf(taps[j], xr[i + 3 - j], u[i]);
        }
#pragma unroll
        for (int i = 0; i < TA; i += 4) *(float4 *)&s.As[buf][kk][seg * TA + i] = make_float4(u[i], u[i + 1], u[i + 2], u[i + 3]);
#pragma unroll
        for (int i = 0; i < EB; ++i) s.Bs[buf][koff + i][br] = wv[i];
    };
    f32x2 acc[TM][NH];
#pragma unroll
    for (int i = 0; i < TM; ++i) {
#pragma unroll
        for (int j = 0; j < NH; ++j) acc[i][j] = pack2(0.f, 0.f);
    }
    const int nk = (Dh + BK - 1) / BK;
    fetch(0);
    stage(0);
    __syncthreads();
    for (int kc = 0; kc < nk; ++kc) {
        if (kc + 1 < nk) fetch((kc + 1) * BK);
        mul_slab<BM>(s, kc & 1, ty, tx, acc);
        if (kc + 1 < nk) stage((kc + 1) & 1);
        __syncthreads();
    }

    ptx::dependency_trigger();
    // ---- gates, decay, scan of this thread's TM tokens x NH channels from zero state
    const int tr = t0 + ty * TM, c0 = n0 + tx * NH, dc = d0 + c0;
    float P[TM][NH], h[TM][NH];
    {
#pragma unroll
        for (int j = 0; j < NH; ++j) {
            const bool cv = c0 + j < Dh;
            const int d = cv ? dc + j : d0;
            float u[TM];
            {
                float w[4], xv[TM + 3];
#pragma unroll
                for (int i = 0; i < TM + 3; ++i) {
                    const int t = tr - 3 + i;
                    xv[i] = t >= 0 ? (t < T ? ldf(xb, (size_t)t * D + d) : 0.0f) : (cs_in ? ldf(cs_in, ((size_t)b * 3 + (3 + t)) * D + d) : 0.0f);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) w[q] = ldf(cw, (size_t)q * D + d);
                const float cbj = a.conv_b ? a.conv_b[d] : 0.0f;
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    u[i] = fmaf(w[0], xv[i + 3], cbj);
#pragma unroll
                    for (int q = 1; q < 4; ++q) u[i] = fmaf(w[q], xv[i + 3 - q], u[i]);
                }
            }
            const float sr = decay_rate(a.lambda[d], a.c), ba = a.b_a[d], bx = a.b_x[d];
            float Pc = 1.0f, hc = 0.0f;
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const float4 gt = gates_acc(col<NH>(acc[i], 0, j) + ba, col<NH>(acc[i], 1, j) + bx, sr);
                const float r = gt.x, g = gt.y, at = gt.z, mt = gt.w;
                const bool tv = tr + i < T;
                if (SAVE) {
                    if (tv && cv) {
                        const size_t e = ((size_t)b * T + tr + i) * D + d;
                        a.save_u[e] = u[i]; a.save_r[e] = r; a.save_i[e] = g;
                    }
                    P[i][j] = Pc; h[i][j] = hc;   // state before the token
                }
                if (tv) { Pc *= at; hc = fmaf(at, hc, mt * (g * u[i])); }
                if (!SAVE) { P[i][j] = Pc; h[i][j] = hc; }
            }
            agg_P[ty][tx * NH + j] = Pc;
            agg_h[ty][tx * NH + j] = hc;
        }
    }
    __syncthreads();
    // ---- chain: one thread per channel takes the state the previous chunk reached and hands its own on
    if (tid < BM) {
        const bool cv = n0 + tid < Dh;
        const int d = cv ? d0 + n0 + tid : d0;
        uint4 *slot = ch.slot + (size_t)b * D + d;
        // the chunk as one step first, so that a link of the chain is one FMA between the record that arrives and the one that leaves
        float cP = 1.0f, cH = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q) { cH = fmaf(agg_P[q][tid], cH, agg_h[q][tid]); cP *= agg_P[q][tid]; }
        float h_in = 0.0f, P_in = 1.0f;
        bool ok = true;
        if (chunk == 0) h_in = a.h0 ? a.h0[(size_t)b * D + d] : 0.0f;
        else ok = chain_wait(ch, slot, cv, chunk - 1, h_in, P_in);
        const float hs = fmaf(cP, h_in, cH), Ps = cP * P_in;
        if (ok && cv) chain_put(ch, slot, chunk, hs, Ps);
        float hq = h_in;
#pragma unroll
        for (int q = 0; q < 8; ++q) { in_h[q][tid] = hq; hq = fmaf(agg_P[q][tid], hq, agg_h[q][tid]); }
        if (ok && cv) {
            if (!SAVE && chunk + 1 == nchunk) {
                a.h_T[(size_t)b * D + d] = hs;
                if (a.a_prod) a.a_prod[(size_t)b * D + d] = Ps;
                // the last three raw inputs of concat(conv_state_in, x), bit-exact
                IOT *cs_out = (IOT *)a.cs_out;
                IOT keep[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) keep[q] = x_raw_at(x, cs_in, T, D, b, T - 3 + q, d);
#pragma unroll
                for (int q = 0; q < 3; ++q) cs_out[((size_t)b * 3 + q) * D + d] = keep[q];
            }
        }
        if (!ok) {
            if (cv) chain_fail(ch, slot, chunk);
            ok_s = 0;
        }
    }
    __syncthreads();
    if (!ok_s) return;
    const IOT *gb = (const IOT *)a.gate_branch;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int t = tr + i;
        if (t >= T) break;
        const size_t e = ((size_t)b * T + t) * D + dc;
#pragma unroll
        for (int j = 0; j < NH; ++j) {
            if (c0 + j < Dh) {
                const float hv = fmaf(P[i][j], in_h[ty][tx * NH + j], h[i][j]);
                if (SAVE) a.save_hprev[e + j] = hv;
                // merged output of the recurrent block (Section 2.3): GeLU on the second branch, then the product
                else stf((IOT *)a.y, e + j, gb ? hv * gelu_acc(ldf(gb, e + j)) : hv);
            }
        }
    }
}

// acc_a[tt] += sum_n W_a[o][n] u_s[tt][n] (same for W_x) for this thread's output channel o.
// Weight slabs of NB input channels are staged through shared memory, transposed so that
// threads read consecutive words.  Every thread of the block must call this.
template <typename IOT>
__device__ __forceinline__ void gate_accumulate(const IOT *__restrict__ Wa, const IOT *__restrict__ Wx, int Dh, int ob,
                                                const float *u_s, float *w_s, float (&acc_a)[GT], float (&acc_x)[GT]) {
    const int tid = threadIdx.x;
    const int o = ob * NT + tid;
    constexpr int WS_STRIDE = NT + 1;
#pragma unroll
    for (int tt = 0; tt < GT; ++tt) { acc_a[tt] = 0.0f; acc_x[tt] = 0.0f; }
    for (int n0 = 0; n0 < Dh; n0 += NB) {
        __syncthreads();
        // slab W[ob*NT .. +NT)[n0 .. n0+NB): consecutive lanes read consecutive n of one row
        for (int idx = tid; idx < NT * NB; idx += NT) {
            int oo = idx / NB, nn = idx % NB;
            int orow = ob * NT + oo, n = n0 + nn;
            float va = 0.0f, vx = 0.0f;
            if (orow < Dh && n < Dh) {
                va = ldf(Wa, (size_t)orow * Dh + n);
                vx = ldf(Wx, (size_t)orow * Dh + n);
            }
            w_s[nn * WS_STRIDE + oo] = va;
            w_s[(NB + nn) * WS_STRIDE + oo] = vx;
        }
        __syncthreads();
        if (o < Dh) {
            const int nmax = min(NB, Dh - n0);
            for (int nn = 0; nn < nmax; ++nn) {
                float wa = w_s[nn * WS_STRIDE + tid], wx = w_s[(NB + nn) * WS_STRIDE + tid];
#pragma unroll
                for (int tt = 0; tt < GT; ++tt) {
                    float uv = u_s[tt * Dh + n0 + nn];
                    acc_a[tt] = fmaf(wa, uv, acc_a[tt]);
                    acc_x[tt] = fmaf(wx, uv, acc_x[tt]);
                }
            }
        }
    }
}

// One decode step.  grid = (H, ceil(B / GT)); a block handles GT sequences of one head.
template <typename IOT>
__global__ void __launch_bounds__(NT) generic_decode_kernel(FwdArgs a) {
    ptx::dependency_wait();
    extern __shared__ float smem[];
    const int Dh = a.D / a.H, D = a.D, B = a.B;
    const int k = blockIdx.x, b0 = blockIdx.y * GT, d0 = k * Dh, tid = threadIdx.x;
    const int len = min(GT, B - b0);
    float *u_s = smem, *w_s = u_s + GT * Dh + Dh;
    const IOT *x = (const IOT *)a.x, *cw = (const IOT *)a.conv_w;
    IOT *cs = (IOT *)a.cs_out;  // in/out
    const IOT *Wa = (const IOT *)a.W_a + (size_t)k * Dh * Dh, *Wx = (const IOT *)a.W_x + (size_t)k * Dh * Dh;
    IOT *y = (IOT *)a.y;
    float *h = a.h_T;  // in/out
    const int nob = (Dh + NT - 1) / NT;

    for (int idx = tid; idx < GT * Dh; idx += NT) {
        int tt = idx / Dh, n = idx % Dh, d = d0 + n;
        float u = 0.0f;
        if (tt < len) {
            const int b = b0 + tt;
            IOT *c0 = cs + ((size_t)b * 3 + 0) * D + d, *c1 = c0 + D, *c2 = c1 + D;
            IOT r0 = *c0, r1 = *c1, r2 = *c2, xn = x[(size_t)b * D + d];
            u = a.conv_b ? a.conv_b[d] : 0.0f;
            u = fmaf(ldf(cw, (size_t)0 * D + d), ldf(&xn, 0), u);
            u = fmaf(ldf(cw, (size_t)1 * D + d), ldf(&r2, 0), u);
            u = fmaf(ldf(cw, (size_t)2 * D + d), ldf(&r1, 0), u);
            u = fmaf(ldf(cw, (size_t)3 * D + d), ldf(&r0, 0), u);
            *c0 = r1; *c1 = r2; *c2 = xn;  // bit-exact shift
        }
        u_s[tt * Dh + n] = u;
    }
    __syncthreads();
    for (int ob = 0; ob < nob; ++ob) {
        float acc_a[GT], acc_x[GT];
        gate_accumulate<IOT>(Wa, Wx, Dh, ob, u_s, w_s, acc_a, acc_x);
        const int o = ob * NT + tid;
        if (o < Dh) {
            const int d = d0 + o;
            const float s = decay_rate(a.lambda[d], a.c), ba = a.b_a[d], bx = a.b_x[d];
#pragma unroll
            for (int tt = 0; tt < GT; ++tt) {
                if (tt < len) {
                    float r = sigmoid_acc(acc_a[tt] + ba), g = sigmoid_acc(acc_x[tt] + bx), at, mt;
                    decay(s, r, at, mt);
                    size_t e = (size_t)(b0 + tt) * D + d;
                    float hn = fmaf(at, h[e], mt * (g * u_s[tt * Dh + o]));
                    h[e] = hn;
                    stf(y, e, hn);
                }
            }
        }
    }
}

// ------------------------------------------------------------------ backward
// Reverse-time scan and element-wise adjoints.  Block = (chunk of 64 tokens, 32 channels, sequence): thread (lane, seg) holds
// the eight tokens of its segment in registers, runs the recurrence from zero, the segments are combined through shared
// memory, the chunks are chained last chunk first.
//   g_t = dy_t + a_{t+1} g_{t+1};  dL = g (a h_{t-1} - a^2 v / m);  dv = g m;  di = dv u;  du = dv i;
//   dr = -s dL;  dz_a = dr r (1-r);  dz_x = di i (1-i).
// In place: r -> dz_a, i -> dz_x, hprev -> du (direct part).
constexpr int RCHUNK = 64;
template <typename IOT>
__global__ void __launch_bounds__(NT) generic_bwd_scan_kernel(BwdArgs q, Chain ch, int nchunk, int ctiles) {
    ptx::dependency_wait();
    __shared__ float agg_Q[8][32], agg_g[8][32], in_g[8][32], sums[3][8][32];
    __shared__ int ok_s;
    const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5;
    int bid = blockIdx.x;
    const int ct = bid % ctiles; bid /= ctiles;
    const int b = bid % q.B, link = bid / q.B, chunk = nchunk - 1 - link;   // last chunk first
    const int T = q.T, D = q.D, d = ct * 32 + lane;
    const bool cv = d < D;
    const int dc = cv ? d : 0, t0 = chunk * RCHUNK + seg * 8;
    const IOT *dy = (const IOT *)q.dy;
    const float lam = q.lambda[dc], s = decay_rate(lam, q.c);
    const float dsdlam_neg = q.c * sigmoid_acc(-lam);  // dL/dLambda = c r sigmoid(-Lambda)
    if (threadIdx.x == 0) ok_s = 1;
    float r[8], at[8], mt[8], dyv[8];
    const size_t e0 = ((size_t)b * T + t0) * D + dc;
    const int nv = min(8, T - t0);   // tokens of the segment that exist (may be <= 0); a token that does not passes g through
#pragma unroll
    for (int i = 0; i < 8; ++i) { r[i] = i < nv ? q.r[e0 + (size_t)i * D] : 0.0f; dyv[i] = i < nv ? ldf(dy, e0 + (size_t)i * D) : 0.0f; }
    float Q = 1.0f, G = 0.0f;
#pragma unroll
    for (int i = 7; i >= 0; --i) {
        if (i < nv) decay(s, r[i], at[i], mt[i]); else { at[i] = 1.0f; mt[i] = 0.0f; }
        G = at[i] * (dyv[i] + G);
        Q *= at[i];
    }
    agg_Q[seg][lane] = Q; agg_g[seg][lane] = G;
    __syncthreads();
    if (seg == 0) {
        uint4 *slot = ch.slot + (size_t)b * D + dc;
        // past the last token g holds the gradient arriving on h_T (h_T = h_{T-1}, so it is carried with factor 1)
        float cQ = 1.0f, cG = 0.0f;   // the chunk as one step, before the wait
#pragma unroll
        for (int k = 7; k >= 0; --k) { cG = fmaf(agg_Q[k][lane], cG, agg_g[k][lane]); cQ *= agg_Q[k][lane]; }
        float X = 0.0f, unused;
        bool ok = true;
        if (link == 0) X = q.dh_T ? q.dh_T[(size_t)b * D + dc] : 0.0f;
        else ok = chain_wait(ch, slot, cv, link - 1, X, unused);
        const float Xout = fmaf(cQ, X, cG);
        if (ok && cv) {
            chain_put(ch, slot, link, Xout, 0.0f);
            if (chunk == 0 && q.dh0) q.dh0[(size_t)b * D + d] = Xout;   // a_0 g_0: h0 enters Eq. 4 only at t = 0
        }
#pragma unroll
        for (int k = 7; k >= 0; --k) { in_g[k][lane] = X; X = fmaf(agg_Q[k][lane], X, agg_g[k][lane]); }
        if (!ok) {
            if (cv) chain_fail(ch, slot, link);
            ok_s = 0;
        }
    }
    __syncthreads();
    if (!ok_s) return;
    ptx::dependency_trigger();
    float carry = in_g[seg][lane], s_lam = 0.0f, s_ba = 0.0f, s_bx = 0.0f;
#pragma unroll
    for (int i = 7; i >= 0; --i) {
        if (i < nv && cv) {
            const size_t e = e0 + (size_t)i * D;
            const float gi = q.gi[e], u = q.u[e], hp = q.hp[e], a = at[i], m = mt[i];
            const float g = dyv[i] + carry;
            const float v = gi * u;
            const float dm_term = m > 0.0f ? a * a * v / m : 0.0f;
            const float dL = g * (a * hp - dm_term);
            const float dv = g * m;
            const float di = dv * u;
            const float dr = -s * dL;
            const float dza = dr * r[i] * (1.0f - r[i]), dzx = di * gi * (1.0f - gi);
            s_lam = fmaf(dL * r[i], dsdlam_neg, s_lam);
            s_ba += dza;
            s_bx += dzx;
            q.r[e] = dza;
            q.gi[e] = dzx;
            q.hp[e] = dv * gi;
            carry = a * g;
        }
    }
    sums[0][seg][lane] = s_lam; sums[1][seg][lane] = s_ba; sums[2][seg][lane] = s_bx;
    __syncthreads();
    if (seg < 3 && cv) {
        float t = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k) t += sums[seg][k][lane];
        q.part_vec[((size_t)(b * nchunk + chunk) * 3 + seg) * D + d] = t;
    }
}

// du[tok][n] += sum_o W_a[o][n] dz_a[tok][o] + W_x[o][n] dz_x[tok][o].  Block = (BM tokens, head, 2 BM input channels); K runs
// over the output channels of both gates.
template <typename IOT, int BM, bool VEC>
__global__ void __launch_bounds__(MT, BM == 64 ? 3 : 6) generic_bwd_du_kernel(BwdArgs q, int ntile) {
    ptx::dependency_wait();
    using TL = Tile<BM>;
    constexpr int TM = TL::TM, NH = TL::NH, BK = TL::BK, EA = TL::TA;
    __shared__ __align__(16) TL s;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int Dh = q.D / q.H, D = q.D;
    int bid = blockIdx.x;
    const int n0 = (bid % ntile) * TL::BN; bid /= ntile;
    const int head = bid % q.H, d0 = head * Dh;
    const size_t ntok = (size_t)q.B * q.T, tok0 = (size_t)(bid / q.H) * BM;
    const int am = tid % BM, koff = (tid / BM) * EA;
    const bool arow = tok0 + am < ntok;
    const size_t aoff = (tok0 + (arow ? am : 0)) * D + d0 + koff;
    const int nkg = (Dh + BK - 1) / BK;   // slabs per gate
    float av[EA], bv[TL::EB];
    auto fetch = [&](int kc) {
        const int gate = kc >= nkg, k0 = (kc - gate * nkg) * BK;
        fetch_k<EA, VEC>((gate ? q.gi : q.r) + aoff + k0, arow, Dh - k0 - koff, av);
        const IOT *W = (const IOT *)(gate ? q.W_x : q.W_a) + ((size_t)head * Dh + k0) * Dh + n0;
        fetch_rows<TL::BN, TL::EB, VEC>(W, (size_t)Dh, Dh - k0, Dh - n0, tid, bv);
    };
    auto stage = [&](int buf) {
#pragma unroll
        for (int i = 0; i < EA; ++i) s.As[buf][koff + i][am] = av[i];
        put_rows<TL::BN, TL::EB, VEC>(s.Bs[buf], tid, bv);
    };
    f32x2 acc[TM][NH];
#pragma unroll
    for (int i = 0; i < TM; ++i) {
#pragma unroll
        for (int j = 0; j < NH; ++j) acc[i][j] = pack2(0.f, 0.f);
    }
    fetch(0);
    stage(0);
    __syncthreads();
    for (int kc = 0; kc < 2 * nkg; ++kc) {
        if (kc + 1 < 2 * nkg) fetch(kc + 1);
        mul_slab<BM>(s, kc & 1, ty, tx, acc);
        if (kc + 1 < 2 * nkg) stage((kc + 1) & 1);
        __syncthreads();
    }
    ptx::dependency_trigger();
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const size_t tok = tok0 + ty * TM + i;
        if (tok >= ntok) break;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int n = n0 + half * BM + tx * NH;
            float *dst = q.hp + tok * D + d0 + n;
#pragma unroll
            for (int j = 0; j < NH; ++j)
                if (n + j < Dh) dst[j] += col<NH>(acc[i], half, j);
        }
    }
}

// Partial dW_a, dW_x: part[s][gate][head][o][n] = sum over the tokens of split s of dz_gate[tok][o] u[tok][n].
// Block = (split, gate, head, BM output rows, 2 BM input columns).
template <int BM, bool VEC>
__global__ void __launch_bounds__(MT, BM == 64 ? 3 : 6) generic_bwd_dw_kernel(BwdArgs q, int mtile, int ntile) {
    ptx::dependency_wait();
    using TL = Tile<BM>;
    constexpr int TM = TL::TM, NH = TL::NH, BK = TL::BK;
    __shared__ __align__(16) TL s;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int Dh = q.D / q.H, D = q.D;
    int bid = blockIdx.x;
    const int n0 = (bid % ntile) * TL::BN; bid /= ntile;
    const int m0 = (bid % mtile) * BM; bid /= mtile;
    const int head = bid % q.H; bid /= q.H;
    const int gate = bid & 1, split = bid >> 1, d0 = head * Dh;
    const size_t ntok = (size_t)q.B * q.T, per = (ntok + q.S - 1) / q.S;
    const size_t lo = (size_t)split * per, hi = lo + per < ntok ? lo + per : ntok;
    const float *dz = (gate ? q.gi : q.r) + d0 + m0, *u = q.u + d0 + n0;
    float av[TL::TA], bv[TL::EB];
    auto fetch = [&](size_t k0) {
        const int rows = (int)(hi - k0 < (size_t)BK ? hi - k0 : (size_t)BK);
        fetch_rows<BM, TL::TA, VEC>(dz + k0 * D, (size_t)D, rows, Dh - m0, tid, av);
        fetch_rows<TL::BN, TL::EB, VEC>(u + k0 * D, (size_t)D, rows, Dh - n0, tid, bv);
    };
    auto stage = [&](int buf) {
        put_rows<BM, TL::TA, VEC>(s.As[buf], tid, av);
        put_rows<TL::BN, TL::EB, VEC>(s.Bs[buf], tid, bv);
    };
    f32x2 acc[TM][NH];
#pragma unroll
    for (int i = 0; i < TM; ++i) {
#pragma unroll
        for (int j = 0; j < NH; ++j) acc[i][j] = pack2(0.f, 0.f);
    }
    const int nk = lo < hi ? (int)((hi - lo + BK - 1) / BK) : 0;
    if (nk > 0) { fetch(lo); stage(0); }
    __syncthreads();
    for (int kc = 0; kc < nk; ++kc) {
        if (kc + 1 < nk) fetch(lo + (size_t)(kc + 1) * BK);
        mul_slab<BM>(s, kc & 1, ty, tx, acc);
        if (kc + 1 < nk) stage((kc + 1) & 1);
        __syncthreads();
    }
    ptx::dependency_trigger();
    const size_t wsz = (size_t)q.H * Dh * Dh;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int o = m0 + ty * TM + i;
        if (o >= Dh) break;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int n = n0 + half * BM + tx * NH;
            float *dst = q.part_dw + ((size_t)split * 2 + gate) * wsz + ((size_t)head * Dh + o) * Dh + n;
#pragma unroll
            for (int j = 0; j < NH; ++j)
                if (n + j < Dh) dst[j] = col<NH>(acc[i], half, j);
        }
    }
}

// Conv1D adjoint: dx_t = sum_j w[j] du_{t+j} (t+j < T); partial dw[j] = sum_t du_t x_{t-j}; partial db_c = sum_t du_t.
// One thread per (b, chunk of GENERIC_BWD_CHUNK tokens, d) walks forward with sliding windows; grid = (ceil(D/NT), nchunk, B).
template <typename IOT>
__global__ void __launch_bounds__(NT) generic_bwd_conv_kernel(BwdArgs q) {
    ptx::dependency_wait();
    const int d = blockIdx.x * NT + threadIdx.x, ch = blockIdx.y, b = blockIdx.z;
    if (d >= q.D) return;
    const int T = q.T, D = q.D;
    const IOT *x = (const IOT *)q.x, *cs_in = (const IOT *)q.cs_in, *cw = (const IOT *)q.conv_w;
    IOT *dx = (IOT *)q.dx;
    float w[4], sw[4] = {0.f, 0.f, 0.f, 0.f}, sb = 0.0f;
#pragma unroll
    for (int j = 0; j < 4; ++j) w[j] = ldf(cw, (size_t)j * D + d);
    const int t_lo = ch * GENERIC_BWD_CHUNK, t_hi = min(T, t_lo + GENERIC_BWD_CHUNK);
    const float *du = q.hp + (size_t)b * T * D + d;
    auto duat = [&](int t) -> float { return t < T ? du[(size_t)t * D] : 0.0f; };
    float x1 = x_at(x, cs_in, T, D, b, t_lo - 1, d), x2 = x_at(x, cs_in, T, D, b, t_lo - 2, d), x3 = x_at(x, cs_in, T, D, b, t_lo - 3, d);
    float g0 = duat(t_lo), g1 = duat(t_lo + 1), g2 = duat(t_lo + 2);
    for (int tb = t_lo; tb < t_hi; tb += 8) {
        float xs[8], gs[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) { xs[k] = tb + k < t_hi ? x_at(x, cs_in, T, D, b, tb + k, d) : 0.0f; gs[k] = duat(tb + k + 3); }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (tb + k < t_hi) {
                const float g3 = gs[k], x0 = xs[k];
                stf(dx, ((size_t)b * T + tb + k) * D + d, fmaf(w[3], g3, fmaf(w[2], g2, fmaf(w[1], g1, w[0] * g0))));
                sw[0] = fmaf(g0, x0, sw[0]); sw[1] = fmaf(g0, x1, sw[1]); sw[2] = fmaf(g0, x2, sw[2]); sw[3] = fmaf(g0, x3, sw[3]);
                sb += g0;
                g0 = g1; g1 = g2; g2 = g3;
                x3 = x2; x2 = x1; x1 = x0;
            }
        }
    }
    float *p = q.part_conv + ((size_t)(b * q.nchunk + ch) * 5) * D + d;
#pragma unroll
    for (int j = 0; j < 4; ++j) p[(size_t)j * D] = sw[j];
    p[(size_t)4 * D] = sb;
}

// Gradient through the carried conv inputs and through the copies in conv_state_out.  One thread per (b, d); grid (ceil(D/NT), B).
template <typename IOT, typename DUT>
__global__ void __launch_bounds__(NT) state_conv_grads_kernel(BwdArgs q, const DUT *du) {
    ptx::dependency_wait();
    const int d = blockIdx.x * NT + threadIdx.x, b = blockIdx.y;
    if (d >= q.D) return;
    const int T = q.T, D = q.D;
    const IOT *cw = (const IOT *)q.conv_w, *dcs_out = (const IOT *)q.dcs_out;
    IOT *dx = (IOT *)q.dx, *dcs_in = (IOT *)q.dcs_in;
    float w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) w[j] = ldf(cw, (size_t)j * D + d);
    auto du_at = [&](int t) -> float { return (t >= 0 && t < T) ? (float)du[((size_t)b * T + t) * D + d] : 0.0f; };
    auto dxin = [&](int t) -> float {   // gradient of the conv input at time t (t may be negative): sum_j w[j] du_{t+j}
        float acc = 0.0f;
#pragma unroll
        for (int j = 0; j < 4; ++j) acc = fmaf(w[j], du_at(t + j), acc);
        return acc;
    };
    float in_grad[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) in_grad[r] = dxin(r - 3);
    if (dcs_out) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float gk = ldf(dcs_out, ((size_t)b * 3 + k) * D + d);
            const int row = T + k;   // row of concat(conv_state_in, x) that conv_state_out[k] copies
            if (row >= 3) stf(dx, ((size_t)b * T + (row - 3)) * D + d, dxin(row - 3) + gk);
            else in_grad[row] += gk;
        }
    }
    if (dcs_in) {
#pragma unroll
        for (int r = 0; r < 3; ++r) stf(dcs_in, ((size_t)b * 3 + r) * D + d, in_grad[r]);
    }
}

// out[i] = sum over the parts of in[p * stride + i] in a fixed order (run-to-run identical results), the row of each job being
// split over up to three output arrays; all jobs of a call in one launch.  A block owns 32 columns with eight slices of the
// parts (slice k sums parts k, k + 8, ... ascending, then the slices are added in order) or, for few parts, 256 columns.
__global__ void __launch_bounds__(256) reduce_jobs_kernel(ReduceJobs jobs) {
    ptx::dependency_wait();
    __shared__ float part[8][32];
    int blk = blockIdx.x, j = 0;
    while (j + 1 < jobs.n && blk >= jobs.job[j].blocks) { blk -= jobs.job[j].blocks; ++j; }
    const ReduceJob &q = jobs.job[j];
    const size_t n = q.n0 + q.n1 + q.n2;
    const bool sliced = q.sliced != 0;
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const size_t i = sliced ? (size_t)blk * 32 + lane : (size_t)blk * 256 + threadIdx.x;
    const int p0 = sliced ? slice : 0, dp = sliced ? 8 : 1;
    float acc = 0.0f;
    if (i < n) {
        int p = p0;
        for (; p + 7 * dp < q.nparts; p += 8 * dp) {   // eight loads in flight
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = q.in[(size_t)(p + k * dp) * q.stride + i];
#pragma unroll
            for (int k = 0; k < 8; ++k) acc += v[k];
        }
        for (; p < q.nparts; p += dp) acc += q.in[(size_t)p * q.stride + i];
    }
    if (sliced) {
        part[slice][lane] = acc;
        __syncthreads();
        if (slice != 0) return;
        acc = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k) acc += part[k][lane];
    }
    if (i >= n) return;
    float *out = i < q.n0 ? (q.out0 ? q.out0 + i : nullptr) : i < q.n0 + q.n1 ? (q.out1 ? q.out1 + (i - q.n0) : nullptr) : (q.out2 ? q.out2 + (i - q.n0 - q.n1) : nullptr);
    if (out) *out = acc;
}

size_t decode_smem_bytes(int Dh) { return sizeof(float) * ((size_t)GT * Dh + Dh + 2 * NB * (NT + 1)); }

template <typename K>
cudaError_t set_smem(K kernel, size_t bytes) {
    if (bytes > 48 * 1024) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    return cudaSuccess;
}


// Rows per block of a contraction with `blocks64` blocks of 64 rows x 128 columns: three of those fit an SM, and below two per
// SM the machine is better filled by four times as many blocks of 32 x 64 (B1 T256 D256 in two heads: 8 -> 64 blocks).  Counted for
// the 148 SMs of a B200 whatever the device, like the splits below, whose number the host-only workspace size has to agree with.
constexpr int FILL_BLOCKS = 296;
inline int tile_rows(size_t blocks64) { return blocks64 >= (size_t)FILL_BLOCKS ? 64 : 32; }

// Token splits of the dW products: as many blocks as fill two waves of three per SM (one split more began a third wave), at least 128 tokens each, at most 32
int dw_splits(size_t ntok, int H, int Dh) {
    const size_t tiles = (size_t)2 * H * ceil_div(Dh, 64) * ceil_div(Dh, 128);
    size_t s = 888 / tiles;
    const size_t most = (ntok + 127) / 128;
    if (s > most) s = most;
    return (int)(s < 1 ? 1 : (s > 32 ? 32 : s));
}

}  // namespace

size_t generic_prefill_workspace_bytes(int B, int D, int io) {
    return up256((size_t)B * D * sizeof(uint4)) + up256((size_t)B * 3 * D * (io == RGLRU_F32 ? 4 : 2));
}

namespace {
template <typename IOT, bool SAVE, int BM>
cudaError_t launch_forward(const FwdArgs &a, const Chain &ch, cudaStream_t st) {
    const int Dh = a.D / a.H, nchunk = ceil_div(a.T, BM), ntile = ceil_div(Dh, BM);
    const size_t grid = (size_t)nchunk * a.B * a.H * ntile;
    if (grid > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
    return launch_dependent(Dh % 4 == 0 ? generic_forward_kernel<IOT, SAVE, BM, true> : generic_forward_kernel<IOT, SAVE, BM, false>, dim3((unsigned)grid), dim3(MT), 0, st,
                            a, ch, nchunk, ntile);
}
template <typename IOT, bool SAVE>
cudaError_t forward_any(const FwdArgs &a, const Chain &ch, cudaStream_t st) {
    const int Dh = a.D / a.H;
    const size_t blocks64 = (size_t)ceil_div(a.T, 64) * a.B * a.H * ceil_div(Dh, 64);
    return tile_rows(blocks64) == 64 ? launch_forward<IOT, SAVE, 64>(a, ch, st) : launch_forward<IOT, SAVE, 32>(a, ch, st);
}
template <typename IOT, int BM>
cudaError_t launch_du(const BwdArgs &q, cudaStream_t st) {
    const int Dh = q.D / q.H, ntile = ceil_div(Dh, 2 * BM);
    const size_t grid = (size_t)ceil_div((size_t)q.B * q.T, BM) * q.H * ntile;
    if (grid > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
    return launch_dependent(Dh % 4 == 0 ? generic_bwd_du_kernel<IOT, BM, true> : generic_bwd_du_kernel<IOT, BM, false>, dim3((unsigned)grid), dim3(MT), 0, st, q, ntile);
}
template <int BM>
cudaError_t launch_dw(const BwdArgs &q, cudaStream_t st) {
    const int Dh = q.D / q.H, mtile = ceil_div(Dh, BM), ntile = ceil_div(Dh, 2 * BM);
    const unsigned grid = (unsigned)((size_t)q.S * 2 * q.H * mtile * ntile);
    return launch_dependent(Dh % 4 == 0 ? generic_bwd_dw_kernel<BM, true> : generic_bwd_dw_kernel<BM, false>, dim3(grid), dim3(MT), 0, st, q, mtile, ntile);
}
}  // namespace

// Workspace body: chain records | private copy of conv_state_in.  The copy is used only when the caller's conv_state_out
// aliases it: blocks of the first chunk read the carried inputs of the whole head while blocks of the last chunk write theirs.
// (h0 needs none: the only block that reads a channel's h0 precedes the one that writes its h_T in the chain.)
cudaError_t generic_prefill(const FwdArgs &a, int io, void *ws_body, cudaStream_t st) {
    FwdArgs f = a;
    const Chain ch = make_chain((uint4 *)ws_body, a);
    const size_t cs_bytes = (size_t)a.B * 3 * a.D * (io == RGLRU_F32 ? 4 : 2);
    const uintptr_t ci = (uintptr_t)a.cs_in, co = (uintptr_t)a.cs_out;
    if (ci && ci < co + cs_bytes && co < ci + cs_bytes) {
        void *copy = (char *)ws_body + up256((size_t)a.B * a.D * sizeof(uint4));
        cudaError_t e = cudaMemcpyAsync(copy, a.cs_in, cs_bytes, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return e;
        f.cs_in = copy;
    }
    return io == RGLRU_F32 ? forward_any<float, false>(f, ch, st) : forward_any<__nv_bfloat16, false>(f, ch, st);
}

cudaError_t generic_decode(const FwdArgs &a, int io, cudaStream_t st) {
    const int Dh = a.D / a.H;
    const size_t smem = decode_smem_bytes(Dh);
    dim3 grid(a.H, (a.B + GT - 1) / GT);
    cudaError_t e;
    if (io == RGLRU_F32) {
        if ((e = set_smem(generic_decode_kernel<float>, smem)) != cudaSuccess) return e;
        return launch_dependent(generic_decode_kernel<float>, grid, dim3(NT), smem, st, a);
    }
    if ((e = set_smem(generic_decode_kernel<__nv_bfloat16>, smem)) != cudaSuccess) return e;
    return launch_dependent(generic_decode_kernel<__nv_bfloat16>, grid, dim3(NT), smem, st, a);
}

cudaError_t state_conv_grads(const BwdArgs &q, int io, const void *du, bool du_is_half, cudaStream_t st) {
    if (!q.dcs_in && !q.dcs_out) return cudaSuccess;
    dim3 grid((q.D + NT - 1) / NT, q.B);
    if (io == RGLRU_F32) return launch_dependent(state_conv_grads_kernel<float, float>, grid, dim3(NT), 0, st, q, (const float *)du);
    if (du_is_half) return launch_dependent(state_conv_grads_kernel<__nv_bfloat16, __half>, grid, dim3(NT), 0, st, q, (const __half *)du);
    return launch_dependent(state_conv_grads_kernel<__nv_bfloat16, float>, grid, dim3(NT), 0, st, q, (const float *)du);
}

void add_reduce_job(ReduceJobs &jobs, const float *in, int nparts, size_t stride, float *out0, size_t n0, float *out1, size_t n1, float *out2, size_t n2) {
    const size_t n = n0 + n1 + n2;
    if (n == 0 || (out0 == nullptr && out1 == nullptr && out2 == nullptr)) return;
    ReduceJob &q = jobs.job[jobs.n++];
    // Up to 16 parts are two rounds of loads for one thread; longer sums are cut into slices.  Up to 32 parts (the splits of dW) are not
    // where there are many of them: 20 parts of 295k sums in slices, 32 sums a block, took 22 us.
    q = ReduceJob{in, stride, out0, out1, out2, n0, n1, n2, nparts, nparts > 16 && (n < 65536 || nparts > 32), 0};
    q.blocks = ceil_div(n, q.sliced ? 32 : 256);
}
cudaError_t run_reduce_jobs(const ReduceJobs &jobs, cudaStream_t st) {
    int blocks = 0;
    for (int i = 0; i < jobs.n; ++i) blocks += jobs.job[i].blocks;
    if (blocks == 0) return cudaSuccess;
    return launch_dependent(reduce_jobs_kernel, dim3(blocks), dim3(256), 0, st, jobs);
}

size_t generic_backward_workspace_bytes(int B, int T, int D, int H) {
    const size_t btd = (size_t)B * T * D, Dh = D / H;
    size_t bytes = 4 * up256(btd * sizeof(float));
    bytes += up256((size_t)B * ceil_div(T, RCHUNK) * 3 * D * sizeof(float));
    bytes += up256((size_t)B * ceil_div(T, GENERIC_BWD_CHUNK) * 5 * D * sizeof(float));
    bytes += up256((size_t)dw_splits((size_t)B * T, H, (int)Dh) * 2 * H * Dh * Dh * sizeof(float));
    bytes += 2 * up256((size_t)B * D * sizeof(uint4));
    return bytes;
}

cudaError_t generic_backward(const FwdArgs &fwd_in, BwdArgs &q, int io, void *ws_body, cudaStream_t st) {
    const int B = q.B, T = q.T, D = q.D, H = q.H, Dh = D / H;
    const size_t btd = (size_t)B * T * D, wsz = (size_t)H * Dh * Dh;
    char *p = (char *)ws_body;
    auto take = [&](size_t bytes) { char *at = p; p += up256(bytes); return at; };
    q.u = (float *)take(btd * sizeof(float));
    q.r = (float *)take(btd * sizeof(float));
    q.gi = (float *)take(btd * sizeof(float));
    q.hp = (float *)take(btd * sizeof(float));
    const int rchunks = ceil_div(T, RCHUNK);
    q.nchunk = ceil_div(T, GENERIC_BWD_CHUNK);
    q.S = dw_splits((size_t)B * T, H, Dh);
    q.part_vec = (float *)take((size_t)B * rchunks * 3 * D * sizeof(float));
    q.part_conv = (float *)take((size_t)B * q.nchunk * 5 * D * sizeof(float));
    q.part_dw = (float *)take((size_t)q.S * 2 * wsz * sizeof(float));
    uint4 *slots_f = (uint4 *)take((size_t)B * D * sizeof(uint4)), *slots_r = (uint4 *)take((size_t)B * D * sizeof(uint4));
    const bool f32 = io == RGLRU_F32;

    // 1. forward sweep, keeping u, r, i and h_{t-1} in fp32
    FwdArgs f = fwd_in;
    f.save_u = q.u; f.save_r = q.r; f.save_i = q.gi; f.save_hprev = q.hp;
    const Chain chf = make_chain(slots_f, fwd_in), chr = make_chain(slots_r, fwd_in);
    cudaError_t e = f32 ? forward_any<float, true>(f, chf, st) : forward_any<__nv_bfloat16, true>(f, chf, st);
    if (e != cudaSuccess) return e;
    // 2. reverse-time scan + element-wise adjoints
    const int ctiles = ceil_div(D, 32);
    const size_t g2 = (size_t)rchunks * B * ctiles;
    if (g2 > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
    if ((e = launch_dependent(f32 ? generic_bwd_scan_kernel<float> : generic_bwd_scan_kernel<__nv_bfloat16>, dim3((unsigned)g2), dim3(NT), 0, st, q, chr, rchunks, ctiles)) != cudaSuccess)
        return e;
    // 3. du += W^T dz
    const size_t blocks3 = (size_t)ceil_div((size_t)B * T, 64) * H * ceil_div(Dh, 128);
    if (tile_rows(blocks3) == 64) e = f32 ? launch_du<float, 64>(q, st) : launch_du<__nv_bfloat16, 64>(q, st);
    else e = f32 ? launch_du<float, 32>(q, st) : launch_du<__nv_bfloat16, 32>(q, st);
    if (e != cudaSuccess) return e;
    // 4. dW partial sums
    const size_t blocks4 = (size_t)q.S * 2 * H * ceil_div(Dh, 64) * ceil_div(Dh, 128);
    if ((e = tile_rows(blocks4) == 64 ? launch_dw<64>(q, st) : launch_dw<32>(q, st)) != cudaSuccess) return e;
    // 5. Conv1D adjoint
    dim3 g5((D + NT - 1) / NT, q.nchunk, B);
    if ((e = launch_dependent(f32 ? generic_bwd_conv_kernel<float> : generic_bwd_conv_kernel<__nv_bfloat16>, g5, dim3(NT), 0, st, q)) != cudaSuccess) return e;
    if ((e = state_conv_grads(q, io, q.hp, false, st)) != cudaSuccess) return e;   // after dx: it rewrites the rows conv_state_out copies
    // 6. deterministic reductions of the partial sums
    ReduceJobs jobs{};
    add_reduce_job(jobs, q.part_dw, q.S, 2 * wsz, q.dW_a, wsz, q.dW_x, wsz, nullptr, 0);
    add_reduce_job(jobs, q.part_vec, B * rchunks, (size_t)3 * D, q.dlambda, D, q.db_a, D, q.db_x, D);
    add_reduce_job(jobs, q.part_conv, B * q.nchunk, (size_t)5 * D, q.dconv_w, (size_t)4 * D, q.dconv_b, D, nullptr, 0);
    return run_reduce_jobs(jobs, st);
}

}  // namespace rglru
