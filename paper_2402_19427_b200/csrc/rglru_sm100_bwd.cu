// sm_100a backward of the RG-LRU temporal core (bf16 io, head width a multiple of 32 up to 256 -- narrower heads in groups of
// 256 channel slots --, T a multiple of 8).
//
// The paper gives no backward; this is reverse-mode differentiation of Eq. 1-4 and the Conv1D.  The three dense
// contractions run on tcgen05 tensor cores through one small GEMM kernel, the rest is element-wise and HBM-bound:
//   1. conv_forward      u = Conv1D(x) in fp16, token-major [tok][D]; fp16 copies of the weights
//                        (every tensor-core operand here is fp16: 11 significant bits instead of bf16's 8 keep the
//                        rounding of u and dz out of the gradients; finite overflow saturates at +-65504)
//   2. GEMM              z_a | z_x = u W_a^T | u W_x^T per head (Eq. 1-2 before the sigmoid), fp16 out
//   3. scan              reverse-time scan g_t = dy_t + a_{t+1} g_{t+1} over chunks of 64 tokens, and
//                        the element-wise adjoints: dz_a, dz_x (fp16, token-major), the direct part of du (fp16), partial
//                        sums of dLambda, db_a, db_x
//   4. GEMM              du += dz_a W_a + dz_x W_x
//   5. GEMM (split K)    dW_a | dW_x = dz^T u over all tokens: both operands are read token-major as steps 1 and 3 wrote them
//                        and handed to the tensor core as MN-major operands (no transposed copies exist); fp32 partial sums
//                        per split, reduced in fixed order
//   6. Conv1D adjoint    dx, dconv_w, dconv_b with sliding windows, fixed-order reductions
// h_{t-1} comes from the forward output y (bf16); when the caller has none the forward is run first.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "rglru_internal.h"
#include "sm100_ptx.cuh"
#include "sm100_gates.cuh"

namespace rglru {
namespace {

using namespace ptx;

constexpr int DH = 256;
constexpr int SCAN_CHUNK = 64;             // tokens per block of the reverse scan (eight warps x eight tokens)
constexpr int CONV_SEG = 32;               // tokens per thread of the two Conv1D kernels ...
constexpr int CONV_CHUNK = 4 * CONV_SEG;   // ... and per block: 64 threads x 4 channels, four segments
constexpr int CONV_CH = 256;
constexpr float LOG2E = 1.44269504f;
constexpr int GEMM_THREADS = 320;          // TMA warp, MMA warp, eight epilogue warps
constexpr int GEMM_STAGES = 4;
constexpr uint32_t A_STAGE_BYTES = 128 * 128;   // 128 rows x 64 bf16
constexpr uint32_t B_STAGE_BYTES = 256 * 128;   // 256 rows x 64 bf16
constexpr uint32_t STAGE_BYTES = A_STAGE_BYTES + B_STAGE_BYTES;
constexpr uint32_t MN_BLOCK_BYTES = 64 * 128;   // one copy of 64 tokens x 64 channels for the MN-major operands of the dW product
constexpr uint32_t GEMM_SMEM_BAR = GEMM_STAGES * STAGE_BYTES;
constexpr uint32_t GEMM_SMEM_TOTAL = GEMM_SMEM_BAR + (2 * GEMM_STAGES + 4) * 8 + 16;
constexpr uint32_t GEMM_SMEM_ALLOC = GEMM_SMEM_TOTAL + 1024;

enum { MODE_Z = 0, MODE_DU = 1, MODE_DW = 2 };

struct GemmArgs {
    alignas(64) CUtensorMap tm_a;    // A rows (M side), K innermost
    alignas(64) CUtensorMap tm_b0;   // B rows (N side), K innermost
    alignas(64) CUtensorMap tm_b1;   // MODE_Z: the second gate's weights (grid.y selects)
    int mode, H, D;    // H: groups of heads
    int NS, NT;        // channel slots of a group = columns of a tile
    int hstride;       // channels of a group that exist (fewer in a partial last group) = channels from one group to the next in [.., D] arrays
    int nx, ny;        // tile grid: nx x ny x H
    int kblocks;       // MODE_DW: 64-token K blocks of a split.  MODE_Z / MODE_DU: K runs over the existing 64-slot blocks of the group
    int rows_valid;    // MODE_Z / MODE_DU: number of tokens; MODE_DW: 2 NS
    void *out;         // MODE_Z: __half z[tok][H][2][NS]; MODE_DU: __half du[tok][D] (+=); MODE_DW: float part[split][2][H][NS][NS]
    uint32_t *status;
    unsigned long long spin_ns;
};

// C[128 x NT] = A[128 x K] B[NT x K]^T per tile; A and B tiles arrive by tiled TMA in the 128-byte-swizzled K-major
// layout, accumulate in tensor memory (fp32), and leave through the eight epilogue warps.  CTAs are persistent: each
// walks tiles blockIdx.x, blockIdx.x + gridDim.x, ... with two accumulators, so that the epilogue of one tile overlaps
// the loads and MMAs of the next.  Tile number -> (x, y, z) with x fastest:
//   MODE_Z : (token tiles, 2 gates, H)        A = u[tok][h][k]        B = W_gate[h][out][k]
//   MODE_DU: (token tiles, 1, H)              A = dz[tok][h][k=2 NS]  B = W[gate][h][k=out][in], MN-major
//   MODE_DW: (2 NS / 128, splits, H)          A = dz[tok][h][row]     B = u[tok][h][in], both MN-major, K = this split's tokens

// 64-slot blocks of group h that hold channels, and the number of K blocks of a tile of that group
__device__ __forceinline__ int slot_blocks(const GemmArgs &p, int h) { return (min(p.hstride, p.D - h * p.hstride) + 63) / 64; }
__device__ __forceinline__ int tile_kblocks(const GemmArgs &p, int h) { return p.mode == MODE_DW ? p.kblocks : (p.mode == MODE_DU ? 2 : 1) * slot_blocks(p, h); }

__global__ void __launch_bounds__(GEMM_THREADS, 1) tc_gemm_kernel(const __grid_constant__ GemmArgs p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw_addr);
    const uint32_t bar0 = base + GEMM_SMEM_BAR;
    auto BAR_FULL = [&](int s) { return bar0 + 8u * s; };
    auto BAR_EMPTY = [&](int s) { return bar0 + 8u * (GEMM_STAGES + s); };
    auto BAR_ACCFULL = [&](int a) { return bar0 + 8u * (2 * GEMM_STAGES + a); };
    auto BAR_ACCEMPTY = [&](int a) { return bar0 + 8u * (2 * GEMM_STAGES + 2 + a); };
    uint32_t *tmem_base_s = (uint32_t *)(smem + GEMM_SMEM_BAR + (2 * GEMM_STAGES + 4) * 8);
    volatile int *abort_flag = (volatile int *)(tmem_base_s + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const unsigned long long spin = p.spin_ns;
    const int ntiles = p.nx * p.ny * p.H;
    // Tiles are dealt round-robin.  (Contiguous runs per CTA, with the B operand left in shared memory while head and gate
    // stay the same, measured 4 % slower on the whole backward: the operand re-reads hit L2 and were not the limit.)

    if (tid == 0) {
        for (int s = 0; s < GEMM_STAGES; ++s) { mbar_init(BAR_FULL(s), 1); mbar_init(BAR_EMPTY(s), 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(BAR_ACCFULL(a), 1); mbar_init(BAR_ACCEMPTY(a), 8); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) { tmem_alloc(smem_u32(tmem_base_s), 512); tmem_relinquish(); }
    if (warp == 0 && lane == 0) { prefetch_tensormap(&p.tm_a); prefetch_tensormap(&p.tm_b0); prefetch_tensormap(&p.tm_b1); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_base_s;
    bool ok = true;
    dependency_wait();

    if (warp == 0) {
        // ---- TMA producer
        if (lane == 0) {
            int kbg = 0;   // K blocks issued so far, over all tiles (ring position)
            const int ncopies = (p.NT + 63) / 64;   // 64-channel copies of an MN-major B operand
            const uint32_t tx_bytes = A_STAGE_BYTES + (p.mode != MODE_Z ? (uint32_t)ncopies * MN_BLOCK_BYTES : (uint32_t)p.NT * 128u);
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
                const int tx = tile % p.nx, sel = (tile / p.nx) % p.ny, h = tile / (p.nx * p.ny);   // sel: gate (MODE_Z), split (MODE_DW)
                const CUtensorMap *tb = (p.mode == MODE_Z && sel == 1) ? &p.tm_b1 : &p.tm_b0;
                const int kslots = slot_blocks(p, h), kblocks = tile_kblocks(p, h);
                for (int kb = 0; kb < kblocks; ++kb, ++kbg) {
                    const int s = kbg % GEMM_STAGES;
                    ok = mbar_wait(BAR_EMPTY(s), ((kbg / GEMM_STAGES) & 1) ^ 1, spin, abort_flag);
                    if (!ok) break;
                    mbar_expect_tx(BAR_FULL(s), tx_bytes);
                    const uint32_t a_dst = base + s * STAGE_BYTES, b_dst = a_dst + A_STAGE_BYTES;
                    if (p.mode == MODE_DW) {
                        // both operands token-major as the scan wrote them: 64 tokens (K) x 64 channels per copy, the channels
                        // innermost; tokens at or beyond B T read as zero
                        const int k0 = (sel * p.kblocks + kb) * 64;
#pragma unroll
                        for (int j = 0; j < 2; ++j) tma_load_3d(a_dst + j * MN_BLOCK_BYTES, &p.tm_a, tx * 128 + j * 64, h, k0, BAR_FULL(s));
                        for (int j = 0; j < ncopies; ++j) tma_load_3d(b_dst + j * MN_BLOCK_BYTES, tb, h * p.hstride + j * 64, k0, 0, BAR_FULL(s));
                    } else {
                        // u is read out of the layer's [tok][D] array at the group's first channel (channels past the group's own
                        // meet zero weights; past D they read as zero); dz has the groups' own [tok][group][2][NS] layout
                        const int kc = kb < kslots ? kb * 64 : p.NS + (kb - kslots) * 64;   // MODE_DU: the second gate's slots follow the first's
                        if (p.mode == MODE_Z) {
                            tma_load_3d(a_dst, &p.tm_a, h * p.hstride + kb * 64, tx * 128, 0, BAR_FULL(s));
                            tma_load_3d(b_dst, tb, kb * 64, 0, h, BAR_FULL(s));
                        } else {
                            tma_load_3d(a_dst, &p.tm_a, kc, h, tx * 128, BAR_FULL(s));
                            const int gate = kb >= kslots, o0 = (kb - gate * kslots) * 64;
                            for (int j = 0; j < ncopies; ++j) tma_load_3d(b_dst + j * MN_BLOCK_BYTES, tb, j * 64, o0, gate * p.H + h, BAR_FULL(s));
                        }
                    }
                }
            }
            if (!ok) { *abort_flag = 1; atomicExch(p.status, STATUS_MAGIC | (uint32_t)RGLRU_ERR_TIMEOUT); }
        }
    } else if (warp == 1) {
        // ---- MMA issuer
        if (lane == 0) {
            const uint32_t idesc = make_idesc_f16(128, p.NT), idesc_mn = make_idesc_f16_mn(128, p.NT), idesc_bmn = make_idesc_f16_bmn(128, p.NT);
            int kbg = 0, it = 0;
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++it) {
                const int acc = it & 1;
                ok = mbar_wait(BAR_ACCEMPTY(acc), ((it >> 1) & 1) ^ 1, spin, abort_flag);   // epilogue of tile it - 2 done
                if (!ok) break;
                const int kblocks = tile_kblocks(p, tile / (p.nx * p.ny));
                for (int kb = 0; kb < kblocks; ++kb, ++kbg) {
                    const int s = kbg % GEMM_STAGES;
                    ok = mbar_wait(BAR_FULL(s), (kbg / GEMM_STAGES) & 1, spin, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a_src = base + s * STAGE_BYTES, b_src = a_src + A_STAGE_BYTES;
                    if (p.mode == MODE_DW) {
                        // K = tokens runs along the rows of the staged blocks: 16 rows of 128 bytes per instruction
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            mma_ss(tmem + acc * 256, make_desc_sw128_mn(a_src + ks * 2048, MN_BLOCK_BYTES), make_desc_sw128_mn(b_src + ks * 2048, MN_BLOCK_BYTES),
                                   idesc_mn, (kb | ks) != 0);
                    } else if (p.mode == MODE_DU) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            mma_ss(tmem + acc * 256, make_desc_sw128(a_src + ks * 32), make_desc_sw128_mn(b_src + ks * 2048, MN_BLOCK_BYTES), idesc_bmn, (kb | ks) != 0);
                    } else {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            mma_ss(tmem + acc * 256, make_desc_sw128(a_src + ks * 32), make_desc_sw128(b_src + ks * 32), idesc, (kb | ks) != 0);
                    }
                    tc_commit(BAR_EMPTY(s));
                }
                if (ok) tc_commit(BAR_ACCFULL(acc));
            }
            if (!ok) { *abort_flag = 1; atomicExch(p.status, STATUS_MAGIC | (uint32_t)RGLRU_ERR_TIMEOUT); }
        }
    } else {
        // ---- epilogue: warp owns TMEM lanes 32 (warp & 3) .. +31 = rows of the tile, and every other 32 columns.  With four warps and
        // the du values read between the accumulator loads, the du product waited for memory once per 32 columns (118 us on B4 T4096
        // D4096); now a tile's du values are requested while its products run.
        const int q = warp & 3, half = (warp - 2) >> 2;
        int it = 0;
        for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++it) {
            const int tx = tile % p.nx, sel = (tile / p.nx) % p.ny, h = tile / (p.nx * p.ny);
            const int acc = it & 1;
            const int row = tx * 128 + q * 32 + lane;
            const bool valid = row < p.rows_valid;
            const int cv = min(p.hstride, p.D - h * p.hstride);   // channel slots of this group that exist
            const uint32_t tm_lane = tmem + ((uint32_t)(q * 32) << 16) + acc * 256;
            auto wait_acc = [&]() { ok = warp_wait(BAR_ACCFULL(acc), (it >> 1) & 1, spin, abort_flag); tc_fence_after(); };
            if (p.mode == MODE_DU) {
                // du is kept in fp16 like dz (bf16 failed the dx tolerance where the taps of the Conv1D adjoint cancel)
                __half *dst0 = (__half *)p.out + (size_t)row * p.D + h * p.hstride;
                uint32_t o[4][2][8];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c0 = j * 64 + half * 32;
                    if (valid && c0 < p.NT && c0 < cv) {   // a slot that does not exist: nothing of du belongs to it
                        ld_global_v8(dst0 + c0, o[j][0]);
                        ld_global_v8(dst0 + c0 + 16, o[j][1]);
                    }
                }
                wait_acc();
                if (!ok) break;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c0 = j * 64 + half * 32;
                    if (c0 < p.NT) {
                        f32x2 v[16];
                        tmem_ld32(tm_lane + c0, v);
                        tmem_ld_wait();
                        if (valid && c0 < cv) {
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                const float2 a0 = __half22float2(*(const __half2 *)&o[j][0][e]), a1 = __half22float2(*(const __half2 *)&o[j][1][e]);
                                o[j][0][e] = pack_f16_sat(a0.x + lo2(v[e]), a0.y + hi2(v[e]));
                                o[j][1][e] = pack_f16_sat(a1.x + lo2(v[8 + e]), a1.y + hi2(v[8 + e]));
                            }
                            st_global_v8(dst0 + c0, o[j][0]);
                            st_global_v8(dst0 + c0 + 16, o[j][1]);
                        }
                    }
                }
            } else {
                wait_acc();
                if (!ok) break;
#pragma unroll 1
                for (int c0 = half * 32; c0 < p.NT; c0 += 64) {
                    f32x2 v[16];
                    tmem_ld32(tm_lane + c0, v);
                    tmem_ld_wait();
                    if (!valid) continue;
                    if (p.mode == MODE_Z) {
                        __half *dst = (__half *)p.out + (((size_t)row * p.H + h) * 2 + sel) * p.NS + c0;
#pragma unroll
                        for (int j8 = 0; j8 < 2; ++j8) {
                            uint32_t w[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) { const __half2 hh = __floats2half2_rn(lo2(v[8 * j8 + j]), hi2(v[8 * j8 + j])); w[j] = *(const uint32_t *)&hh; }
                            st_global_v8(dst + 16 * j8, w);
                        }
                    } else {
                        const int g = row >= p.NS, o_row = row - g * p.NS;
                        float *dst = (float *)p.out + ((((size_t)sel * 2 + g) * p.H + h) * p.NS + o_row) * p.NS + c0;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            uint32_t w[8];
#pragma unroll
                            for (int e = 0; e < 4; ++e) { w[2 * e] = __float_as_uint(lo2(v[4 * j + e])); w[2 * e + 1] = __float_as_uint(hi2(v[4 * j + e])); }
                            st_global_v8(dst + 8 * j, w);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(BAR_ACCEMPTY(acc));   // this accumulator may be overwritten
        }
        if (!ok && lane == 0) { *abort_flag = 1; atomicExch(p.status, STATUS_MAGIC | (uint32_t)RGLRU_ERR_TIMEOUT); }
    }
    dependency_trigger();
    if (*abort_flag) {   // let copies and MMAs in flight land before shared and tensor memory are given back
        const uint64_t tw = gtimer();
        while (gtimer() - tw < 50000ull) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------ element-wise kernels
__device__ __forceinline__ float sigmoid_acc(float z) { return 1.0f / (1.0f + expf(-z)); }
// Hardware-approximate versions for the per-element work (relative error ~1e-6, far inside the gradient tolerance)
__device__ __forceinline__ float rsqrt_fast(float x) { float y; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
// 1 - exp(x) for x <= 0 without cancellation near 0
__device__ __forceinline__ float one_minus_exp(float x) {
    if (x > -0.25f) {   // -x (1 + x/2 + x^2/6 + x^3/24 + x^4/120 + x^5/720): relative truncation error < 2e-7
        float pl = fmaf(x, 1.0f / 720.0f, 1.0f / 120.0f);
        pl = fmaf(pl, x, 1.0f / 24.0f); pl = fmaf(pl, x, 1.0f / 6.0f); pl = fmaf(pl, x, 0.5f); pl = fmaf(pl, x, 1.0f);
        return -x * pl;
    }
    return 1.0f - __expf(x);
}
// s = c softplus(-Lambda)   (Appendix A, with a = sigmoid(Lambda))
__device__ __forceinline__ float decay_rate(float lambda, float c) {
    const float z = -lambda;
    return c * (z > 0.0f ? z + log1pf(expf(-z)) : log1pf(expf(z)));
}

struct EwArgs {
    int B, T, D, H, nchunk;
    int hstride, NS;                  // channels of a group of heads = channels from one group to the next; its channel slots
    float c;
    const __nv_bfloat16 *x, *conv_w, *cs_in, *dy, *y;
    const float *conv_b, *b_a, *b_x, *lambda, *h0;
    __half *u, *dz;
    const __half *z;                  // [tok][H][2][NS] before the sigmoid, without the bias
    __half *du;                       // [tok][D]
    uint4 *rec;                       // [nchunk][B][D] carry records of the reverse scan
    uint32_t *epoch;                  // launch counter in the workspace (any starting value): part of the records' tag
    uint32_t tag, wait_flip;          // wait_flip: see rglru_internal.h
    unsigned long long spin_ns;
    uint32_t *status;
    float *part_vec;                  // [B*S][3][D]
    const float *dh_T;                // [B][D] gradient arriving on h_T, or null
    float *dh0;                       // [B][D] gradient of h0, or null
};

// fp16 copy of the gate weights, W16[g][h][o][n] = W_g[h][o][n], eight elements per thread.  H counts groups; dh is the width of a
// head of the layer (a multiple of 32): a group holds k heads on its diagonal -- fewer in a partial last group of a layer of Hl
// heads -- and everything outside those blocks is written as zeros.  Both the z product (K-major) and the du product (MN-major)
// read this one copy.
__global__ void __launch_bounds__(256) convert_w_kernel(const __nv_bfloat16 *Wa, const __nv_bfloat16 *Wx, __half *W16, int H, int NS, int k, int dh, int Hl) {
    dependency_wait();
    const int per_row = NS / 8;
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= (size_t)2 * H * NS * per_row) return;
    const int n0 = (int)(i % per_row) * 8;
    size_t r = i / per_row;
    const int o = (int)(r % NS); r /= NS;
    const int h = (int)(r % H), g = (int)(r / H);
    const int sub = o / dh;                          // head of the group that owns this output row
    uint4 out = make_uint4(0u, 0u, 0u, 0u);
    if (sub < min(k, Hl - h * k) && n0 / dh == sub) {
        const uint4 v = *(const uint4 *)((g ? Wx : Wa) + (((size_t)h * k + sub) * dh + (o - sub * dh)) * dh + (n0 - sub * dh));
        auto cvt2 = [](uint32_t w) { return pack_f16_sat(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u)); };
        out = make_uint4(cvt2(v.x), cvt2(v.y), cvt2(v.z), cvt2(v.w));
    }
    *(uint4 *)(W16 + i * 8) = out;
}

// Fixed-order sum over the token splits of the diagonal blocks of the groups' weight gradients: one thread per
// element of dW_a / dW_x [H_layer][dh][dh].  part: [S][2 gates][G groups][NS][NS]
__global__ void reduce_dw_blocks_kernel(const float *part, int S, int G, int NS, int k, int dh, int Hl, float *dWa, float *dWx) {
    dependency_wait();
    const size_t per_gate = (size_t)Hl * dh * dh;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 2 * per_gate) return;
    const int gate = (int)(i / per_gate);
    size_t r = i % per_gate;
    const int n = (int)(r % dh); r /= dh;
    const int o = (int)(r % dh); r /= dh;
    const int head = (int)r, group = head / k, sub = head % k;
    const size_t src = (((size_t)gate * G + group) * NS + sub * dh + o) * NS + sub * dh + n;
    const size_t stride = (size_t)2 * G * NS * NS;
    float acc = 0.0f;
    for (int s = 0; s < S; ++s) acc += part[(size_t)s * stride + src];
    (gate ? dWx : dWa)[i % per_gate] = acc;
}

__device__ __forceinline__ f32x2 hf2x(uint32_t w) { return __half22float2(*(const __half2 *)&w); }

// four adjacent channels
struct f32x4 { f32x2 a, b; };
__device__ __forceinline__ f32x4 bf4x(uint2 w) { return f32x4{bf2x(w.x), bf2x(w.y)}; }
__device__ __forceinline__ f32x4 hf4x(uint2 w) { return f32x4{hf2x(w.x), hf2x(w.y)}; }
__device__ __forceinline__ f32x4 zero4() { return f32x4{pack2(0.f, 0.f), pack2(0.f, 0.f)}; }
__device__ __forceinline__ f32x4 fma4(const f32x4 &x, const f32x4 &y, const f32x4 &z) { return f32x4{fma2(x.a, y.a, z.a), fma2(x.b, y.b, z.b)}; }
__device__ __forceinline__ f32x4 mul4(const f32x4 &x, const f32x4 &y) { return f32x4{mul2(x.a, y.a), mul2(x.b, y.b)}; }

// u_t = b_c + sum_j w[j] x_{t-j} as fp16 u[B][T][D]: one thread per (sequence, 32 tokens, four adjacent channels), forward in time,
// eight tokens' loads in flight.  Bound by its 4 bytes per element: with two channels per thread and a predicate on every token it
// executed 26 instructions per element (66 % of the issue slots) and took 66 us on B4 T4096 D4096.
// grid (ceil(D/256), ceil(T/128), B)
struct ConvArgs {
    int T, D;
    const __nv_bfloat16 *x, *conv_w, *cs_in;
    const float *conv_b;
    __half *u;
    uint32_t *epoch;
};
__global__ void __launch_bounds__(256, 4) conv_forward_kernel(ConvArgs a) {
    dependency_wait();
    const int d = blockIdx.x * CONV_CH + (threadIdx.x & 63) * 4, b = blockIdx.z;
    const int T = a.T, D = a.D, t0 = blockIdx.y * CONV_CHUNK + (threadIdx.x >> 6) * CONV_SEG, t1 = min(T, t0 + CONV_SEG);
    // the scans' carry records are told apart from those an earlier launch with the same host tag (a graph replay) left behind
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) *a.epoch += 1u;
    if (d >= D || t0 >= t1) return;
    f32x4 w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) w[j] = bf4x(*(const uint2 *)(a.conv_w + (size_t)j * D + d));
    const f32x4 cb = a.conv_b ? f32x4{ld2f(a.conv_b + d), ld2f(a.conv_b + d + 2)} : zero4();
    auto xat = [&](int t) -> f32x4 {
        if (t >= 0) return bf4x(*(const uint2 *)(a.x + ((size_t)b * T + t) * D + d));
        return a.cs_in ? bf4x(*(const uint2 *)(a.cs_in + ((size_t)b * 3 + (3 + t)) * D + d)) : zero4();
    };
    f32x4 x3 = xat(t0 - 3), x2 = xat(t0 - 2), x1 = xat(t0 - 1);
    const uint32_t sD = (uint32_t)D / 4;   // token stride in groups of four channels
    const uint2 *px = (const uint2 *)(a.x + ((size_t)b * T + t0) * D + d);
    uint2 *pu = (uint2 *)(a.u + ((size_t)b * T + t0) * D + d);
    auto token = [&](uint2 xw) {
        const f32x4 x0 = bf4x(xw);
        const f32x4 uv = fma4(w[3], x3, fma4(w[2], x2, fma4(w[1], x1, fma4(w[0], x0, cb))));
        *pu = make_uint2(pack_f16_sat(uv.a.x, uv.a.y), pack_f16_sat(uv.b.x, uv.b.y));
        pu += sD;
        x3 = x2; x2 = x1; x1 = x0;
    };
    int t = t0;
#pragma unroll 1
    for (; t + 8 <= t1; t += 8) {
        uint2 xs[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) { xs[k] = *px; px += sD; }
#pragma unroll
        for (int k = 0; k < 8; ++k) token(xs[k]);
    }
#pragma unroll 1
    for (; t < t1; ++t) { token(*px); px += sD; }
}

// 1 - exp(-x) for 0 <= x <= S_POLY without cancellation: x (1 - x/2 + x^2/6 - x^3/24 + x^4/120), relative truncation error < 1.5e-6
__device__ __forceinline__ f32x2 one_minus_exp_neg2(f32x2 x) {
    f32x2 p = fma2(x, pack2(1.0f / 120.0f, 1.0f / 120.0f), pack2(-1.0f / 24.0f, -1.0f / 24.0f));
    p = fma2(p, x, pack2(1.0f / 6.0f, 1.0f / 6.0f));
    p = fma2(p, x, pack2(-0.5f, -0.5f));
    p = fma2(p, x, pack2(1.0f, 1.0f));
    return mul2(p, x);
}

// r = sigmoid(z_a + b_a) and f = 1 - a_t of two channels; a_t = 1 - f, 1 - a_t^2 = f (2 - f)
template <bool POLY> __device__ __forceinline__ void gate_f2(f32x2 za, f32x2 nba, f32x2 s2, f32x2 &r, f32x2 &f) {
    const f32x2 e = fma2(za, pack2(-LOG2E, -LOG2E), nba);   // -(z + b) log2 e
    const f32x2 q = __fadd2_rn(pack2(ex2_approx(e.x), ex2_approx(e.y)), pack2(1.0f, 1.0f));
    r = pack2(rcp_approx(q.x), rcp_approx(q.y));
    const f32x2 x = mul2(s2, r);
    f = POLY ? one_minus_exp_neg2(x) : pack2(one_minus_exp(-x.x), one_minus_exp(-x.y));
}

// The reverse scan g_t = dy_t + a_{t+1} g_{t+1} and every element-wise adjoint (derived from Eq. 1-4):
//   dL = g a (h_{t-1} - a v / m);  dv = g m;  di = dv u;  du = dv i;
//   dr = -s dL;  dz_a = dr r (1-r);  dz_x = di i (1-i);  dLambda += dL c r sigmoid(-Lambda).
// A block walks a column of 64 channels of one sequence backwards in chunks of 64 tokens; dy, y, u, z_a, z_x of the next chunk
// arrive by tiled TMA while it works on this one (two stages of 40 KB, two blocks per SM).  A thread holds two adjacent channels
// x the eight tokens of its warp's segment: fold from zero carry, segments combined through shared memory, adjoints.
// Bound by its 16 bytes per element: z and dy are read once.  (The fold, carry and apply passes of one channel per thread that
// it replaces: 79 + 5 + 309 us on B4 T4096 D4096.  One block per chunk with decoupled look-back for every chunk, all loads
// straight into registers: 525 us, each block a serial chain of load, look-back and store.)
// A column with idle SMs beside it is shared by S blocks that take its chunks round-robin: each chunk's step {Q, G} is
// published before anyone waits, and a block forms its incoming carry from the one it reached S chunks ago and the S - 1
// steps in between, in fixed order (run-to-run identical results).  The blocks of a column are neighbours in block order, so
// with at most one partly dispatched column the resident ones always finish; see carry_clock_step for other work on the GPU.
struct ScanArgs {
    alignas(64) CUtensorMap tm_dy, tm_y, tm_u;   // [B][T][D], box 64 tokens x 64 channels
    alignas(64) CUtensorMap tm_z;                // [B][T][groups x 2 x NS], the same box
    EwArgs e;
    int S;          // blocks per column
    int tiles;      // columns per group of heads
};
constexpr uint32_t SCAN_TILE_BYTES = SCAN_CHUNK * 128;
constexpr uint32_t SCAN_STAGE_BYTES = 5 * SCAN_TILE_BYTES;
constexpr uint32_t SCAN_SMEM_ALLOC = 2 * SCAN_STAGE_BYTES + 1024;
constexpr int SCAN_MAX_S = 16;
constexpr int SCAN_WINDOW = 4;   // records requested at once

struct ScanShared {
    f32x2 agg[2][8][32];   // steps of the eight segments: Q, G
    f32x2 xin[32];
    uint64_t full[2];
    int abort;
};

// Carry records of one pair of channels (two adjacent ones) of a column whose links S blocks take round-robin; this lane's records of
// link l are rec0 + l stride and the one behind it.
struct Column {
    uint4 *rec0;
    ptrdiff_t stride;
    int S;
    bool cv;               // the channels exist
    uint32_t tag, wait;    // this execution's tag, and the one waited for (another under the failure-path test flag)
    unsigned long long limit_ns;
};
__device__ __forceinline__ void mark_running(const Column &c, int first_link) {
    if (c.cv) asm volatile("st.global.b32 [%0], %1;" ::"l"(&(c.rec0 + (ptrdiff_t)first_link * c.stride)->y), "r"(c.tag ^ RUNNING) : "memory");
}
__device__ __forceinline__ void put_record(const Column &c, int link, f32x2 Q, f32x2 G) {
    uint4 *rec = c.rec0 + (ptrdiff_t)link * c.stride;
    if (!c.cv) return;
    asm volatile("st.global.v4.b32 [%0], {%1, %2, %3, %4};" ::"l"(rec), "r"(__float_as_uint(Q.x)), "r"(c.tag), "r"(__float_as_uint(G.x)), "r"(c.tag) : "memory");
    asm volatile("st.global.v4.b32 [%0], {%1, %2, %3, %4};" ::"l"(rec + 1), "r"(__float_as_uint(Q.y)), "r"(c.tag), "r"(__float_as_uint(G.y)), "r"(c.tag) : "memory");
}
// See carry_clock_step: do the blocks that write links first .. first + count - 1 run?
__device__ __noinline__ uint64_t column_clock(uint64_t state, const uint4 *rec0, ptrdiff_t stride, int S, uint32_t tag, unsigned long long limit_ns, int first, int count) {
    bool running = true;
    for (int k = 0; k < count; ++k) {
        const uint32_t v = ld_volatile_u32(&(rec0 + (ptrdiff_t)((first + k) % S) * stride)->y);
        running = running && (v == tag || v == (tag ^ RUNNING));
    }
    return carry_clock_step(state, running, limit_ns);
}
// The first W of `left` records from link `first` on, polled until every lane sees this launch's tag in both halves of each (8-byte
// words are written atomically: such a record is whole).  False if the wait ran out.
template <int W>
__device__ __forceinline__ bool read_records(const Column &c, int first, int left, uint4 (&w0)[W], uint4 (&w1)[W]) {
    uint64_t clock = 0;
    for (uint32_t npoll = 0;; ++npoll) {
        bool ready = true;
#pragma unroll
        for (int k = 0; k < W; ++k) {
            if (k < left && c.cv) {
                const uint4 *src = c.rec0 + (ptrdiff_t)(first + k) * c.stride;
                asm volatile("ld.volatile.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w0[k].x), "=r"(w0[k].y), "=r"(w0[k].z), "=r"(w0[k].w) : "l"(src) : "memory");
                asm volatile("ld.volatile.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w1[k].x), "=r"(w1[k].y), "=r"(w1[k].z), "=r"(w1[k].w) : "l"(src + 1) : "memory");
                ready = ready && w0[k].y == c.wait && w0[k].w == c.wait && w1[k].y == c.wait && w1[k].w == c.wait;
            }
        }
        if (__all_sync(0xffffffffu, ready)) return true;
        if ((npoll & 31u) == 31u) {
            clock = column_clock(clock, c.rec0, c.stride, c.S, c.tag, c.limit_ns, first, !c.cv ? 0 : left < W ? left : W);
            if (clock == ~0ull) return false;
        }
    }
}

template <bool POLY>
__device__ __forceinline__ void scan_column(const ScanArgs &p, ScanShared &sh, const uint8_t *stage, uint32_t stage_addr, int b, int k0, int group, int n0, f32x2 s2) {
    const EwArgs &a = p.e;
    const int tid = threadIdx.x, lane = tid & 31, seg = tid >> 5;
    const int T = a.T, D = a.D, S = p.S, n = n0 + 2 * lane, d = group * a.hstride + n;
    const bool cv = n < a.hstride && d < D;
    const uint32_t sD = (uint32_t)D / 2, sZ = (uint32_t)a.H * a.NS, sN = (uint32_t)a.NS / 2;   // strides in channel pairs: tokens, gates
    const f32x2 ba = cv ? ld2f(a.b_a + d) : pack2(0.f, 0.f), bx = cv ? ld2f(a.b_x + d) : pack2(0.f, 0.f);
    const f32x2 nba = mul2(ba, pack2(-LOG2E, -LOG2E)), nbx = mul2(bx, pack2(-LOG2E, -LOG2E));
    const f32x2 ONE = pack2(1.0f, 1.0f), TWO = pack2(2.0f, 2.0f), NEG = pack2(-1.0f, -1.0f), ns2 = mul2(s2, NEG);
    const uint32_t full0 = smem_u32(&sh.full[0]);
    // this block's chunks are links k0, k0 + S, ... counted from the end of the sequence
    auto issue = [&](int link, int st) {
        const int t0 = (a.nchunk - 1 - link) * SCAN_CHUNK, c = group * a.hstride + n0, zc = group * 2 * a.NS + n0;
        const uint32_t bar = full0 + 8u * st, dst = stage_addr + st * SCAN_STAGE_BYTES;
        mbar_expect_tx(bar, SCAN_STAGE_BYTES);
        tma_load_3d(dst, &p.tm_z, zc, t0, b, bar);
        tma_load_3d(dst + SCAN_TILE_BYTES, &p.tm_dy, c, t0, b, bar);
        tma_load_3d(dst + 2 * SCAN_TILE_BYTES, &p.tm_z, zc + a.NS, t0, b, bar);
        tma_load_3d(dst + 3 * SCAN_TILE_BYTES, &p.tm_u, c, t0, b, bar);
        tma_load_3d(dst + 4 * SCAN_TILE_BYTES, &p.tm_y, c, t0 - 1, b, bar);   // h_{t-1}; the row before the sequence reads as zero
    };
    if (tid == 0) {
        issue(k0, 0);
        if (k0 + S < a.nchunk) issue(k0 + S, 1);
    }
    // past the last token the carry is the gradient arriving on h_T (h_T = h_{T-1}, so it enters with factor 1), else nothing
    f32x2 X = a.dh_T && cv ? ld2f(a.dh_T + (size_t)b * D + d) : pack2(0.f, 0.f);
    f32x2 s_lam = pack2(0.f, 0.f), s_ba = s_lam, s_bx = s_lam;
    const uint32_t tag = S > 1 ? a.tag + *a.epoch * 0x9E3779B1u : 0u;
    auto column = [&]() { return Column{a.rec + ((size_t)(a.nchunk - 1) * a.B + b) * D + d, -(ptrdiff_t)a.B * D, S, cv, tag, tag ^ a.wait_flip, a.spin_ns}; };
    if (S > 1 && seg == 0) mark_running(column(), k0);
    bool ok = true;
    int it = 0;
    for (int link = k0; link < a.nchunk; link += S, ++it) {
        const int st = it & 1, chunk = a.nchunk - 1 - link, t0 = chunk * SCAN_CHUNK + seg * 8;
        const int nv = T - t0;     // tokens of the segment that exist, if fewer than eight
        ok = warp_wait(full0 + 8u * st, (it >> 1) & 1, a.spin_ns, &sh.abort);
        const uint32_t *sm = (const uint32_t *)(stage + st * SCAN_STAGE_BYTES) + seg * 8 * 32 + lane;
        constexpr int TW = SCAN_TILE_BYTES / 4;
        f32x2 r[8], f[8];
        f32x2 Q = ONE, G = pack2(0.0f, 0.0f);
        auto fold = [&](auto all) {   // all: all tokens of the chunk exist
#pragma unroll
            for (int k = 7; k >= 0; --k) {
                gate_f2<POLY>(hf2x(sm[k * 32]), nba, s2, r[k], f[k]);
                if (!decltype(all)::value && k >= nv) { r[k] = pack2(0.f, 0.f); f[k] = pack2(0.f, 0.f); }   // a token that does not exist passes the carry through (its dy reads as zero)
                const f32x2 at = fma2(f[k], NEG, ONE);
                G = mul2(at, __fadd2_rn(bf2x(sm[TW + k * 32]), G));
                Q = mul2(Q, at);
            }
        };
        const bool whole = (chunk + 1) * SCAN_CHUNK <= T;
        if (whole) fold(std::true_type{}); else fold(std::false_type{});
        sh.agg[0][seg][lane] = Q; sh.agg[1][seg][lane] = G;
        if (!ok) sh.abort = 1;
        __syncthreads();
        if (S > 1) {
            if (seg == 0 && !sh.abort) {
                f32x2 Qt = ONE, Gt = pack2(0.0f, 0.0f);
#pragma unroll
                for (int k = 7; k >= 0; --k) { Gt = fma2(sh.agg[0][k][lane], Gt, sh.agg[1][k][lane]); Qt = mul2(Qt, sh.agg[0][k][lane]); }
                const Column col = column();
                put_record(col, link, Qt, Gt);
                for (int jb = min(link, S - 1); jb > 0 && ok; jb -= SCAN_WINDOW) {   // links link - jb, link - jb + 1, ...
                    uint4 w0[SCAN_WINDOW], w1[SCAN_WINDOW];
                    ok = read_records<SCAN_WINDOW>(col, link - jb, jb, w0, w1);
                    if (!ok) break;
#pragma unroll
                    for (int k = 0; k < SCAN_WINDOW; ++k)
                        if (k < jb && cv) X = fma2(pack2(__uint_as_float(w0[k].x), __uint_as_float(w1[k].x)), X, pack2(__uint_as_float(w0[k].z), __uint_as_float(w1[k].z)));
                }
                sh.xin[lane] = X;
                if (!ok) sh.abort = 1;
            }
            __syncthreads();
            X = sh.xin[lane];
        }
        if (sh.abort) break;   // uniform: set before the barrier above
        f32x2 carry = X;
#pragma unroll
        for (int k = 7; k >= 0; --k) {
            if (k == seg) carry = X;
            X = fma2(sh.agg[0][k][lane], X, sh.agg[1][k][lane]);
        }
        uint32_t *p_dz = (uint32_t *)(a.dz + ((size_t)b * T + t0) * (size_t)(2 * sZ) + (size_t)group * 2 * a.NS + n);
        uint32_t *p_du = (uint32_t *)(a.du + ((size_t)b * T + t0) * D + d);
        auto adjoint = [&](auto all, int k) {
            const f32x2 u = hf2x(sm[3 * TW + k * 32]);
            f32x2 hp = bf2x(sm[4 * TW + k * 32]);
            if (k == 0 && t0 == 0 && a.h0 && cv) hp = ld2f(a.h0 + (size_t)b * D + d);
            const f32x2 e = fma2(hf2x(sm[2 * TW + k * 32]), pack2(-LOG2E, -LOG2E), nbx);
            const f32x2 q = __fadd2_rn(pack2(ex2_approx(e.x), ex2_approx(e.y)), ONE);
            const f32x2 gi = pack2(rcp_approx(q.x), rcp_approx(q.y));
            const f32x2 at = fma2(f[k], NEG, ONE), m2 = mul2(f[k], fma2(f[k], NEG, TWO));
            // 1 / sqrt(1 - a^2).  Where that is below 1e-15, r is below 1e-30 and makes dL r vanish as it should
            const f32x2 rm = pack2(rsqrt_fast(fmaxf(m2.x, 1e-30f)), rsqrt_fast(fmaxf(m2.y, 1e-30f)));
            const f32x2 g = __fadd2_rn(bf2x(sm[TW + k * 32]), carry);
            carry = mul2(at, g);
            const f32x2 v = mul2(gi, u);
            const f32x2 hh = fma2(mul2(at, v), mul2(rm, NEG), hp);          // h_{t-1} - a v / m
            const f32x2 dLr = mul2(mul2(carry, hh), r[k]);                   // dL r,  dL = g a (h_{t-1} - a v / m)
            const f32x2 du = mul2(mul2(g, mul2(m2, rm)), gi);
            const f32x2 dza = mul2(mul2(dLr, ns2), fma2(r[k], NEG, ONE));
            const f32x2 dzx = mul2(mul2(du, u), fma2(gi, NEG, ONE));
            s_lam = __fadd2_rn(s_lam, dLr);
            s_ba = __fadd2_rn(s_ba, dza); s_bx = __fadd2_rn(s_bx, dzx);      // tokens that do not exist add zeros (r = 0, u = 0)
            if (decltype(all)::value || k < nv) {
                if (cv) p_du[k * sD] = pack_f16_sat(du.x, du.y);
                // slots of this 64-slot block that do not exist get zeros: the du product multiplies the whole block
                p_dz[k * sZ] = cv ? pack_f16_sat(dza.x, dza.y) : 0u;
                p_dz[k * sZ + sN] = cv ? pack_f16_sat(dzx.x, dzx.y) : 0u;
            }
        };
        if (whole) {
#pragma unroll
            for (int k = 7; k >= 0; --k) adjoint(std::true_type{}, k);
        } else {
#pragma unroll
            for (int k = 7; k >= 0; --k) adjoint(std::false_type{}, k);
        }
        __syncthreads();   // everybody has read the stage and the segments' steps
        if (tid == 0 && link + 2 * S < a.nchunk) issue(link + 2 * S, st);
        if (chunk == 0 && seg == 0 && cv && a.dh0) *(float2 *)(a.dh0 + (size_t)b * D + d) = X;   // a_0 g_0, the gradient of h0
    }
    if (sh.abort) {
        if (tid == 0) {
            atomicExch(a.status, STATUS_MAGIC | (uint32_t)RGLRU_ERR_TIMEOUT);
            const uint64_t tw = gtimer();   // let copies in flight land before shared memory is given back
            while (gtimer() - tw < 50000ull) __nanosleep(1000);
        }
        __syncthreads();
        return;
    }
    dependency_trigger();
    // sums over this block's tokens, segment by segment
    f32x2(*sums)[8][32] = (f32x2(*)[8][32])stage;
    sums[0][seg][lane] = s_lam; sums[1][seg][lane] = s_ba; sums[2][seg][lane] = s_bx;
    __syncthreads();
    if (seg < 3 && cv) {
        f32x2 t = pack2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 8; ++k) t = __fadd2_rn(t, sums[seg][k][lane]);
        if (seg == 0) {   // dL/dLambda = c r sigmoid(-Lambda)
            const f32x2 lam = ld2f(a.lambda + d);
            t = mul2(t, pack2(a.c * sigmoid_acc(-lam.x), a.c * sigmoid_acc(-lam.y)));
        }
        *(float2 *)(a.part_vec + ((size_t)(b * S + k0) * 3 + seg) * D + d) = t;
    }
}

__global__ void __launch_bounds__(256, 2) scan_kernel(const __grid_constant__ ScanArgs p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ ScanShared sh;
    const uint32_t raw = smem_u32(smem_raw), base = (raw + 127u) & ~127u;
    const EwArgs &a = p.e;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&sh.full[0]), 1); mbar_init(smem_u32(&sh.full[1]), 1);
        sh.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    dependency_wait();
    int bid = blockIdx.x;
    const int k0 = bid % p.S; bid /= p.S;
    const int tile = bid % p.tiles; bid /= p.tiles;
    const int group = bid % a.H, b = bid / a.H;
    const int n = tile * 64 + (threadIdx.x & 31) * 2, d = group * a.hstride + n;
    const bool cv = n < a.hstride && d < a.D;
    const f32x2 lam = cv ? ld2f(a.lambda + d) : pack2(0.f, 0.f);
    const f32x2 s2 = cv ? pack2(decay_rate(lam.x, a.c), decay_rate(lam.y, a.c)) : pack2(0.f, 0.f);
    uint8_t *stage = smem_raw + (base - raw);
    // uniform over the block: every warp holds the same channels
    if (__all_sync(0xffffffffu, s2.x <= S_POLY && s2.y <= S_POLY)) scan_column<true>(p, sh, stage, base, b, k0, group, tile * 64, s2);
    else scan_column<false>(p, sh, stage, base, b, k0, group, tile * 64, s2);
}

// Blocks per column: two blocks fit an SM; the fewest rounds of chunks over all waves, a shared column paying for its look-back
int scan_split(int columns, int nchunk, int slots) {
    int best = 1;
    double best_cost = 1e30;
    for (int S = 1; S <= SCAN_MAX_S && S <= nchunk; ++S) {
        const double waves = (double)(((size_t)columns * S + slots - 1) / slots), rounds = (nchunk + S - 1) / S;
        const double cost = waves * (S == 1 ? rounds : 1.2 * rounds + 1.0);
        if (cost < best_cost) { best_cost = cost; best = S; }
    }
    return best;
}

// Conv1D adjoint: dx_t = sum_j w[j] du_{t+j} (t + j < T); per-chunk partial sums of dw[j] = sum_t du_t x_{t-j} and
// db_c = sum_t du_t.  One thread per (sequence, 32 tokens, four adjacent channels) walks forward with sliding windows, so that
// every du and every x is loaded once; a block adds its four segments' sums.  Bound by its 6 bytes per element (two channels per
// thread, a predicate on every token and sums per 32 tokens: 104 us on B4 T4096 D4096).  grid (ceil(D/256), ceil(T/128), B)
struct ConvBwdArgs {
    int B, T, D;
    const void *x, *conv_w, *cs_in, *du;
    void *dx;
    float *part_conv;   // [B*chunks][5][D]
};
// four adjacent channels as they lie in memory
template <typename T> struct Four { typedef uint2 raw; };
template <> struct Four<float> { typedef float4 raw; };
__device__ __forceinline__ f32x4 four(const __nv_bfloat16 *, uint2 w) { return bf4x(w); }
__device__ __forceinline__ f32x4 four(const __half *, uint2 w) { return hf4x(w); }
__device__ __forceinline__ f32x4 four(const float *, float4 w) { return f32x4{pack2(w.x, w.y), pack2(w.z, w.w)}; }
__device__ __forceinline__ uint2 four_out(const __nv_bfloat16 *, const f32x4 &v) { return make_uint2(pack_bf16(v.a.x, v.a.y), pack_bf16(v.b.x, v.b.y)); }
__device__ __forceinline__ float4 four_out(const float *, const f32x4 &v) { return make_float4(v.a.x, v.a.y, v.b.x, v.b.y); }

// LEN: tokens per thread
template <typename IOT, typename DUT, int LEN> __global__ void __launch_bounds__(256, 2) conv_backward_kernel(ConvBwdArgs a) {
    typedef typename Four<IOT>::raw XR;
    typedef typename Four<DUT>::raw GR;
    __shared__ float4 red[3][5][64];
    dependency_wait();
    const int c = threadIdx.x & 63, sg = threadIdx.x >> 6, d = blockIdx.x * CONV_CH + c * 4, b = blockIdx.z;
    const int T = a.T, D = a.D, t0 = (blockIdx.y * 4 + sg) * LEN, t1 = min(T, t0 + LEN);
    const IOT *x = (const IOT *)a.x, *cs_in = (const IOT *)a.cs_in, *cw = (const IOT *)a.conv_w;
    auto io4 = [](const IOT *p) { return four(p, *(const XR *)p); };
    auto du4 = [](const GR *p) { return four((const DUT *)p, *p); };
    f32x4 sw[5];   // four taps, bias
#pragma unroll
    for (int j = 0; j < 5; ++j) sw[j] = zero4();
    if (d < D && t0 < t1) {
        f32x4 w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = io4(cw + (size_t)j * D + d);
        auto xat = [&](int t) -> f32x4 {
            if (t >= 0) return io4(x + ((size_t)b * T + t) * D + d);
            return cs_in ? io4(cs_in + ((size_t)b * 3 + (3 + t)) * D + d) : zero4();
        };
        const uint32_t sD = (uint32_t)D / 4;
        const XR *px = (const XR *)(x + ((size_t)b * T + t0) * D + d);
        const GR *pg = (const GR *)((const DUT *)a.du + ((size_t)b * T + t0) * D + d);
        XR *pdx = (XR *)((IOT *)a.dx + ((size_t)b * T + t0) * D + d);
        f32x4 x1 = xat(t0 - 1), x2 = xat(t0 - 2), x3 = xat(t0 - 3);
        f32x4 g0 = du4(pg), g1 = t0 + 1 < T ? du4(pg + sD) : zero4(), g2 = t0 + 2 < T ? du4(pg + 2 * sD) : zero4();
        pg += 3 * (size_t)sD;
        auto token = [&](XR xw, GR gw) {   // gw: du_{t+3}, zero bits past the end
            const f32x4 x0 = four((const IOT *)nullptr, xw), g3 = four((const DUT *)nullptr, gw);
            *pdx = four_out((const IOT *)nullptr, fma4(w[3], g3, fma4(w[2], g2, fma4(w[1], g1, mul4(w[0], g0)))));
            pdx += sD;
            sw[0] = fma4(g0, x0, sw[0]); sw[1] = fma4(g0, x1, sw[1]); sw[2] = fma4(g0, x2, sw[2]); sw[3] = fma4(g0, x3, sw[3]);
            sw[4].a = __fadd2_rn(sw[4].a, g0.a); sw[4].b = __fadd2_rn(sw[4].b, g0.b);
            g0 = g1; g1 = g2; g2 = g3;
            x3 = x2; x2 = x1; x1 = x0;
        };
        constexpr int BATCH = sizeof(XR) + sizeof(GR) <= 16 ? 8 : 4;   // tokens' loads in flight
        int t = t0;
#pragma unroll 1
        for (; t + BATCH <= t1 && t + BATCH + 3 <= T; t += BATCH) {
            XR xs[BATCH];
            GR gs[BATCH];
#pragma unroll
            for (int k = 0; k < BATCH; ++k) { xs[k] = *px; px += sD; gs[k] = *pg; pg += sD; }
#pragma unroll
            for (int k = 0; k < BATCH; ++k) token(xs[k], gs[k]);
        }
#pragma unroll 1
        for (; t < t1; ++t) { token(*px, t + 3 < T ? *pg : GR{}); px += sD; pg += sD; }
    }
    // segments added in order: run-to-run identical
    if (sg > 0) {
#pragma unroll
        for (int j = 0; j < 5; ++j) red[sg - 1][j][c] = make_float4(sw[j].a.x, sw[j].a.y, sw[j].b.x, sw[j].b.y);
    }
    __syncthreads();
    if (sg == 0 && d < D) {
        float *pc = a.part_conv + ((size_t)(b * gridDim.y + blockIdx.y) * 5) * D + d;
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            float4 t = make_float4(sw[j].a.x, sw[j].a.y, sw[j].b.x, sw[j].b.y);
#pragma unroll
            for (int k = 0; k < 3; ++k) { const float4 o = red[k][j][c]; t.x += o.x; t.y += o.y; t.z += o.z; t.w += o.w; }
            *(float4 *)(pc + (size_t)j * D) = t;
        }
    }
}


unsigned gemm_grid(const GemmArgs &g) {
    const int nsm = num_sms();
    const int ntiles = g.nx * g.ny * g.H;
    return (unsigned)(ntiles < nsm ? ntiles : nsm);
}

// Groups of heads, the unit of the GEMMs and of the z / dz arrays: k = 256 / width (rounded down) consecutive heads in
// NS channel slots, their channels rounded up to K blocks of 64: one column tile (NT = NS).
struct Groups {
    int dh, k, G, hstride, NS, NT;
    size_t W16_bytes() const { return (size_t)2 * G * NS * NS * 2; }
};
Groups make_groups(int D, int H) {
    Groups g{};
    g.dh = D / H;
    g.k = DH / g.dh;
    g.G = (H + g.k - 1) / g.k;
    g.hstride = g.k * g.dh;
    g.NT = g.NS = (g.hstride + 63) / 64 * 64;
    return g;
}

struct BwdLayout {
    size_t BT, BTp, off_u, off_z, off_dz, off_du, off_y, off_hT, off_cs, off_fws, off_rec, off_pvec, off_pconv, off_pdw,
        off_w16, total;
    int nchunk, nchunk_conv, S, kb_per_split;
};

// Token splits of the dW products.  A K block (48 KB per SM) takes ~0.6 us, a tile four of them more for filling and epilogue, and
// each split's partial sums are written and read again at ~5 TB/s.  Counted in whole rounds of 148 SMs (whatever the device: the
// workspace size has to agree with the launch): 2 splits for 16 heads of 256 (64 tiles a split; eight of them took four rounds
// and 67 MB of partial sums, dW and its reduction 110 us on B4 T4096).
int dw_split(const Groups &gr, int kblocks) {
    const int tiles = gr.G * (2 * gr.NS / 128), most = kblocks < 16 ? kblocks : 16;
    const double part_us = 2.0 * 2 * gr.G * gr.NS * gr.NS * 4 / 5e6;
    int best = 1;
    double best_us = 1e30;
    for (int S = 1; S <= most; ++S) {
        const double us = ((tiles * S + 147) / 148) * 0.6 * ((kblocks + S - 1) / S + 4) + S * part_us;
        if (us < best_us) { best_us = us; best = S; }
    }
    return best;
}

BwdLayout bwd_layout(int B, int T, int D, int Hl) {
    BwdLayout L{};
    const Groups gr = make_groups(D, Hl);
    const size_t Dg = (size_t)gr.G * gr.NS;   // channel slots of all groups (>= D)
    L.BT = (size_t)B * T;
    L.BTp = (L.BT + 63) & ~(size_t)63;
    L.nchunk = (T + SCAN_CHUNK - 1) / SCAN_CHUNK;
    L.nchunk_conv = (T + CONV_CHUNK - 1) / CONV_CHUNK;
    const int kblocks = (int)(L.BTp / 64);
    L.S = dw_split(gr, kblocks);
    L.kb_per_split = (kblocks + L.S - 1) / L.S;
    size_t o = 0;
    auto take = [&](size_t bytes) { const size_t at = o; o += up256(bytes); return at; };
    L.off_u = take(L.BT * D * 2);
    L.off_z = take(L.BT * Dg * 2 * 2);
    L.off_dz = take(L.BT * Dg * 2 * 2);
    L.off_du = take(L.BT * D * 2);
    L.off_y = take(L.BT * D * 2);
    L.off_hT = take((size_t)B * D * 4);
    L.off_cs = take((size_t)B * 3 * D * 2);
    L.off_fws = take(sm100_prefill_workspace_bytes(B, T, D, Hl));
    L.off_rec = take((size_t)B * L.nchunk * D * sizeof(uint4) + 256);   // the records, then the launch counter
    L.off_pvec = take((size_t)B * (L.nchunk < SCAN_MAX_S ? L.nchunk : SCAN_MAX_S) * 3 * D * 4);
    L.off_pconv = take((size_t)B * conv_backward_chunks(B, T, D) * 5 * D * 4);
    L.off_pdw = take((size_t)L.S * 2 * gr.G * gr.NS * gr.NS * 4);
    L.off_w16 = take(gr.W16_bytes());
    L.total = o;
    return L;
}

GemmArgs gemm_args(const Groups &gr, int D, uint32_t *status) {
    GemmArgs g{};
    g.H = gr.G; g.D = D; g.NS = gr.NS; g.NT = gr.NT; g.hstride = gr.hstride; g.status = status; g.spin_ns = g_spin_limit_ns;
    return g;
}
cudaError_t run_gemm(const GemmArgs &g, cudaStream_t st) {
    static PerDeviceOptIn opt_in;
    cudaError_t e = opt_in.ensure(tc_gemm_kernel, (int)GEMM_SMEM_ALLOC);
    if (e != cudaSuccess) return e;
    return launch_dependent(tc_gemm_kernel, dim3(gemm_grid(g)), dim3(GEMM_THREADS), GEMM_SMEM_ALLOC, st, g);
}
cudaError_t convert_w(const Groups &gr, const void *Wa, const void *Wx, int Hl, __half *W16, cudaStream_t st) {
    const size_t n = (size_t)2 * gr.G * gr.NS * (gr.NS / 8);
    return launch_dependent(convert_w_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, (const __nv_bfloat16 *)Wa, (const __nv_bfloat16 *)Wx, W16, gr.G, gr.NS, gr.k, gr.dh, Hl);
}
// z = u W^T per group and gate: u [ntok][D], z [ntok][G][2][NS]
cudaError_t gemm_z(const Groups &gr, int D, size_t ntok, const __half *u, const __half *W16, __half *z, uint32_t *status, cudaStream_t st) {
    GemmArgs g = gemm_args(gr, D, status);
    const uint64_t NS = gr.NS;
    const uint64_t da[3] = {(uint64_t)D, ntok, 1}, sa[2] = {(uint64_t)D * 2, (uint64_t)D * ntok * 2};
    const uint32_t ba[3] = {64, 128, 1};
    const uint64_t db[3] = {NS, NS, (uint64_t)gr.G}, sb[2] = {NS * 2, NS * NS * 2};
    const uint32_t bb[3] = {64, (uint32_t)gr.NT, 1};
    if (!encode_map16_3d(&g.tm_a, u, da, sa, ba, true) || !encode_map16_3d(&g.tm_b0, W16, db, sb, bb, true) ||
        !encode_map16_3d(&g.tm_b1, W16 + (size_t)gr.G * NS * NS, db, sb, bb, true))
        return cudaErrorNotSupported;
    g.mode = MODE_Z; g.rows_valid = (int)ntok; g.out = z;
    g.nx = (int)((ntok + 127) / 128); g.ny = 2;
    return run_gemm(g, st);
}

}  // namespace

// Head width: a multiple of 32 up to 256.  k = 256 / width (rounded down) consecutive heads form a group whose weight matrix is
// block-diagonal; it is multiplied as a dense matrix (convert_w_kernel writes the zeros), and only the diagonal blocks of its
// gradient are kept (reduce_dw_blocks_kernel).  Slots beyond the group's channels do not exist: they meet zero weights, the scan
// writes zeros for those that share a 64-slot block with real ones, the other blocks are left out of the products, and nothing of
// them is written to du.
// T a multiple of 8, and no wider heads: those calls get the kernels with split products (rglru_sm100_split.cu), which hold u, r, i,
// h, dz and du in fp32.  These kernels run them too, twice as fast (B5 T1021 D1536 in 16 heads 133 us), but keep u, z, dz and du in
// fp16 and h_{t-1} in bf16: gradients of the parameters are then 2e-4 to 5e-4 from the exact ones (2-norm) where fp32 is below
// 1e-6, and a caller of such a shape has been promised the latter.
bool sm100_backward_supported(int B, int T, int D, int H, int io) {
    if (io != RGLRU_BF16 || B <= 0 || T <= 0 || T % 8 != 0 || H <= 0 || D % H != 0) return false;
    const int dh = D / H;
    return dh <= DH && dh % 32 == 0;
}

namespace {
// Tokens per thread: 32, or 8 while 128-token blocks would leave SMs idle (B1 T256 D256, fp32: two blocks, 11 us)
int conv_backward_len(int B, int T, int D) {
    return (size_t)B * ((T + CONV_CHUNK - 1) / CONV_CHUNK) * ((D + CONV_CH - 1) / CONV_CH) >= 148 ? CONV_SEG : 8;
}
template <typename IOT, typename DUT>
cudaError_t launch_conv_backward(const ConvBwdArgs &a, cudaStream_t st) {
    const dim3 grid((a.D + CONV_CH - 1) / CONV_CH, conv_backward_chunks(a.B, a.T, a.D), a.B);
    return launch_dependent(conv_backward_len(a.B, a.T, a.D) == CONV_SEG ? conv_backward_kernel<IOT, DUT, CONV_SEG> : conv_backward_kernel<IOT, DUT, 8>, grid, dim3(256), 0, st, a);
}
}  // namespace
int conv_backward_chunks(int B, int T, int D) {
    const int per_block = 4 * conv_backward_len(B, T, D);
    return (T + per_block - 1) / per_block;
}

cudaError_t conv_backward(const BwdArgs &q, int io, const void *du, bool du_is_half, cudaStream_t st) {
    const ConvBwdArgs a{q.B, q.T, q.D, q.x, q.conv_w, q.cs_in, du, q.dx, q.part_conv};
    if (io == RGLRU_F32) return launch_conv_backward<float, float>(a, st);
    return du_is_half ? launch_conv_backward<__nv_bfloat16, __half>(a, st) : launch_conv_backward<__nv_bfloat16, float>(a, st);
}

size_t sm100_backward_workspace_bytes(int B, int T, int D, int H) { return bwd_layout(B, T, D, H).total; }

cudaError_t sm100_backward(const FwdArgs &fwd, BwdArgs &q, const void *y_saved, void *ws_body, size_t ws_body_bytes, uint32_t *status,
                           cudaStream_t st) {
    const int B = q.B, T = q.T, D = q.D;
    const Groups gr = make_groups(D, q.H);
    const int H = gr.G, NS = gr.NS, hstride = gr.hstride;
    const BwdLayout L = bwd_layout(B, T, D, q.H);
    if (ws_body_bytes < L.total) return cudaErrorInvalidValue;
    cudaError_t e;
    char *ws = (char *)ws_body;
    __half *u = (__half *)(ws + L.off_u), *z = (__half *)(ws + L.off_z);
    __half *dz = (__half *)(ws + L.off_dz), *W16 = (__half *)(ws + L.off_w16);
    __half *du = (__half *)(ws + L.off_du);

    EwArgs a{};
    a.B = B; a.T = T; a.D = D; a.H = H; a.nchunk = L.nchunk; a.c = q.c; a.hstride = hstride; a.NS = NS;
    a.x = (const __nv_bfloat16 *)q.x; a.conv_w = (const __nv_bfloat16 *)q.conv_w; a.cs_in = (const __nv_bfloat16 *)q.cs_in;
    a.dy = (const __nv_bfloat16 *)q.dy;
    a.conv_b = fwd.conv_b; a.b_a = fwd.b_a; a.b_x = fwd.b_x; a.lambda = q.lambda; a.h0 = fwd.h0;
    a.u = u; a.dz = dz; a.z = z; a.du = du;
    a.rec = (uint4 *)(ws + L.off_rec); a.epoch = (uint32_t *)(a.rec + (size_t)B * L.nchunk * D);
    a.tag = next_call_tag(); a.wait_flip = wait_flip(fwd.flags); a.spin_ns = g_spin_limit_ns; a.status = status; a.part_vec = (float *)(ws + L.off_pvec);
    a.dh_T = q.dh_T; a.dh0 = q.dh0;

    // 0. h_{t-1} comes from the forward output.  When the caller kept none the fused prefill makes it, whose gate products stay in fp32
    // (a scan over the u and fp16 z of step 2 saves 5 % of B5 T1024 D1536 in 16 heads, and loses that)
    const void *y = y_saved;
    if (y == nullptr) {
        FwdArgs f = fwd;
        f.y = ws + L.off_y; f.h_T = (float *)(ws + L.off_hT); f.cs_out = ws + L.off_cs;
        f.gate_branch = nullptr; f.a_prod = nullptr; f.status = status;
        if ((e = sm100_prefill(f, ws + L.off_fws, sm100_prefill_workspace_bytes(B, T, D, q.H), st)) != cudaSuccess) return e;
        y = f.y;
    }
    // 1. fp16 weights, conv output
    if ((e = convert_w(gr, q.W_a, q.W_x, q.H, W16, st)) != cudaSuccess) return e;
    const dim3 grid_conv((D + CONV_CH - 1) / CONV_CH, L.nchunk_conv, B);
    if ((e = launch_dependent(conv_forward_kernel, grid_conv, dim3(256), 0, st, ConvArgs{T, D, a.x, a.conv_w, a.cs_in, a.conv_b, u, a.epoch})) != cudaSuccess) return e;

    ReduceJobs jobs{};
    const uint64_t BT = L.BT;
    // 2. z = u W^T per head and gate
    if ((e = gemm_z(gr, D, L.BT, u, W16, z, status, st)) != cudaSuccess) return e;
    GemmArgs g = gemm_args(gr, D, status);
    const unsigned mtiles = (unsigned)((L.BT + 127) / 128);
    // 3. reverse scan and element-wise adjoints
    a.y = (const __nv_bfloat16 *)y;
    ScanArgs sc{};
    sc.e = a;
    sc.tiles = (hstride + 63) / 64;
    sc.S = scan_split(B * H * sc.tiles, L.nchunk, 2 * num_sms());
    {
        const uint64_t dx[3] = {(uint64_t)D, (uint64_t)T, (uint64_t)B}, sx[2] = {(uint64_t)D * 2, (uint64_t)D * T * 2};
        const uint64_t wz = (uint64_t)H * 2 * NS, dzm[3] = {wz, (uint64_t)T, (uint64_t)B}, szm[2] = {wz * 2, wz * T * 2};
        const uint32_t box[3] = {64, SCAN_CHUNK, 1};
        if (!encode_map16_3d(&sc.tm_dy, q.dy, dx, sx, box, false) || !encode_map16_3d(&sc.tm_y, y, dx, sx, box, false) ||
            !encode_map16_3d(&sc.tm_u, u, dx, sx, box, false) || !encode_map16_3d(&sc.tm_z, z, dzm, szm, box, false))
            return cudaErrorNotSupported;
        static PerDeviceOptIn scan_opt_in;
        if ((e = scan_opt_in.ensure(scan_kernel, (int)SCAN_SMEM_ALLOC)) != cudaSuccess) return e;
    }
    const size_t scan_blocks = (size_t)B * H * sc.tiles * sc.S;
    if (scan_blocks > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
    if ((e = launch_dependent(scan_kernel, dim3((unsigned)scan_blocks), dim3(256), SCAN_SMEM_ALLOC, st, sc)) != cudaSuccess) return e;
    // 4. du += dz W
    const uint64_t K2 = 2 * (uint64_t)NS, ddz[3] = {K2, (uint64_t)H, BT}, sdz[2] = {K2 * 2, (uint64_t)H * K2 * 2};   // dz [tok][group][gate, slot]
    {
        const uint32_t ba[3] = {64, 1, 128};
        const uint64_t db[3] = {(uint64_t)NS, (uint64_t)NS, 2 * (uint64_t)H}, sb[2] = {(uint64_t)NS * 2, (uint64_t)NS * NS * 2};   // W16 [gate, group][out][in]
        const uint32_t bb[3] = {64, 64, 1};
        if (!encode_map16_3d(&g.tm_a, dz, ddz, sdz, ba, true) || !encode_map16_3d(&g.tm_b0, W16, db, sb, bb, true)) return cudaErrorNotSupported;
        g.tm_b1 = g.tm_b0;
        g.mode = MODE_DU; g.rows_valid = (int)BT; g.out = du;
        g.nx = (int)mtiles; g.ny = 1;
        if ((e = run_gemm(g, st)) != cudaSuccess) return e;
    }
    // 5. dW = dz^T u, split over the tokens, then a fixed-order sum of the splits
    {
        const uint32_t ba[3] = {64, 1, 64};
        const uint64_t db[3] = {(uint64_t)D, BT, 1}, sb[2] = {(uint64_t)D * 2, (uint64_t)D * BT * 2};         // u [tok][D]
        const uint32_t bb[3] = {64, 64, 1};
        if (!encode_map16_3d(&g.tm_a, dz, ddz, sdz, ba, true) || !encode_map16_3d(&g.tm_b0, u, db, sb, bb, true)) return cudaErrorNotSupported;
        g.tm_b1 = g.tm_b0;
        float *part = (float *)(ws + L.off_pdw);
        g.mode = MODE_DW; g.kblocks = L.kb_per_split; g.rows_valid = 2 * NS; g.out = part;
        g.nx = 2 * NS / 128; g.ny = L.S;
        if ((e = run_gemm(g, st)) != cudaSuccess) return e;
        const size_t wsz = (size_t)H * NS * NS;
        if (gr.dh == NS) {   // one head per group and every slot exists: the partial sums already have the layout of dW
            add_reduce_job(jobs, part, L.S, 2 * wsz, q.dW_a, wsz, q.dW_x, wsz, nullptr, 0);
        } else {
            const size_t nout = (size_t)2 * q.H * gr.dh * gr.dh;
            if ((e = launch_dependent(reduce_dw_blocks_kernel, dim3((unsigned)((nout + 255) / 256)), dim3(256), 0, st, part, L.S, H, NS, gr.k, gr.dh, q.H, q.dW_a, q.dW_x)) != cudaSuccess) return e;
        }
    }
    // 6. per-channel sums, Conv1D adjoint
    add_reduce_job(jobs, a.part_vec, B * sc.S, (size_t)3 * D, q.dlambda, D, q.db_a, D, q.db_x, D);
    q.part_conv = (float *)(ws + L.off_pconv);
    if ((e = conv_backward(q, RGLRU_BF16, du, true, st)) != cudaSuccess) return e;
    if ((e = state_conv_grads(q, RGLRU_BF16, du, true, st)) != cudaSuccess) return e;   // after dx: it rewrites the rows conv_state_out copies
    add_reduce_job(jobs, q.part_conv, B * conv_backward_chunks(B, T, D), (size_t)5 * D, q.dconv_w, (size_t)4 * D, q.dconv_b, D, nullptr, 0);
    return run_reduce_jobs(jobs, st);
}

}  // namespace rglru
