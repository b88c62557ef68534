// Learned vertex priority: a 12 -> 64 -> 64 -> 1 MLP over integer-derived
// per-vertex features, used in place of the edge difference (the paper's
// Alg. 4 score) when CH_PRIO_LEARNED is set. The paper has no learned
// priority; any priority yields a valid hierarchy (Alg. 5 only needs a
// strict order), so the network can only change the hierarchy's quality.
//
// Inference runs on the tensor cores: BF16 weights and activations, FP32
// accumulation (mma.sync m16n8k16), one warp per 16 vertices; layer 1's
// accumulators are re-packed in registers as layer 2's A fragments.
// Training runs forward passes with the same BF16 roundings, backward passes
// in FP32 (rounding treated as identity), gradient sums in a fixed order
// (deterministic), and Adam on FP32 master weights.
//
// Weight layout (FP32, CH_MLP_NPARAM values): W1[12][64] (input-major),
// b1[64], W2[64][64] (input-major), b2[64], W3[64], b3.

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstddef>

#include "mlp.cuh"

namespace gbch {

namespace {

constexpr int NIN = MLP_NIN, NH = MLP_NH;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NIN * NH, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NH;
static_assert(OFF_B3 + 1 == MLP_NPARAM, "parameter layout");

__device__ __forceinline__ float bf16_round(float x) {
    return __bfloat162float(__float2bfloat16_rn(x));
}

// The copy of parameter p the forward pass uses: W1 and W2 in BF16 (as the
// tensor-core inference uses them), biases and W3 in FP32.
__device__ __forceinline__ float quantised(uint32_t p, float w) {
    return (p < (uint32_t)OFF_B1 || (p >= (uint32_t)OFF_W2 && p < (uint32_t)OFF_B2)) ? bf16_round(w) : w;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// D = A * B + C for one m16n8k16 tile (A row-major BF16, B column-major BF16).
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// B fragments of W1 (K = 16 rows, 12 used) and W2 (K = 64), per lane:
// frag1[j][lane] for n-tile j (8 columns); frag2[kk][j][lane] for k-tile kk.
struct MlpFrag {
    uint2 w1[NH / 8][32];
    uint2 w2[NH / 16][NH / 8][32];
    float b1[NH], b2[NH], w3[NH], b3;
};

__global__ void k_mlp_prepare(const float *w, MlpFrag *f) {
    const uint32_t lane = threadIdx.x & 31u, grp = lane >> 2, tig = lane & 3u;
    const uint32_t warp = threadIdx.x >> 5;
    // W1: element (k, n) = W1[k][n] for k < 12, 0 above
    auto w1 = [&](uint32_t k, uint32_t n) { return k < (uint32_t)NIN ? w[OFF_W1 + k * NH + n] : 0.f; };
    for (uint32_t j = warp; j < NH / 8; j += blockDim.x >> 5) {
        const uint32_t n = 8 * j + grp;
        f->w1[j][lane] = make_uint2(pack_bf16(w1(2 * tig, n), w1(2 * tig + 1, n)),
                                    pack_bf16(w1(2 * tig + 8, n), w1(2 * tig + 9, n)));
    }
    for (uint32_t t = warp; t < (NH / 16) * (NH / 8); t += blockDim.x >> 5) {
        const uint32_t kk = t / (NH / 8), j = t % (NH / 8);
        const uint32_t n = 8 * j + grp, k0 = 16 * kk + 2 * tig;
        const float *W2 = w + OFF_W2;
        f->w2[kk][j][lane] = make_uint2(pack_bf16(W2[k0 * NH + n], W2[(k0 + 1) * NH + n]),
                                        pack_bf16(W2[(k0 + 8) * NH + n], W2[(k0 + 9) * NH + n]));
    }
    for (uint32_t i = threadIdx.x; i < (uint32_t)NH; i += blockDim.x) {
        f->b1[i] = w[OFF_B1 + i];
        f->b2[i] = w[OFF_B2 + i];
        f->w3[i] = w[OFF_W3 + i];
    }
    if (threadIdx.x == 0) f->b3 = w[OFF_B3];
}

constexpr int INF_WARPS = 4;

// y[r] = MLP(x[r]) for rows of 16 transformed features (12 used). Each warp
// takes 16 rows at a time.
__global__ void __launch_bounds__(INF_WARPS * 32)
k_mlp_infer(const float *x, uint64_t rows, const MlpFrag *fg, float *y) {
    __shared__ MlpFrag f;
    for (uint32_t i = threadIdx.x; i < sizeof(MlpFrag) / 4; i += blockDim.x)
        reinterpret_cast<uint32_t *>(&f)[i] = reinterpret_cast<const uint32_t *>(fg)[i];
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31u, grp = lane >> 2, tig = lane & 3u;
    const uint64_t warp = blockIdx.x * (uint64_t)INF_WARPS + (threadIdx.x >> 5);
    const uint64_t nwarps = (uint64_t)gridDim.x * INF_WARPS;
    for (uint64_t r0 = warp * 16; r0 < rows; r0 += nwarps * 16) {
        const uint64_t ra = r0 + grp, rb = r0 + grp + 8;
        auto xv = [&](uint64_t r, uint32_t c) { return r < rows ? x[r * 16 + c] : 0.f; };
        uint32_t a[4];
        a[0] = pack_bf16(xv(ra, 2 * tig), xv(ra, 2 * tig + 1));
        a[1] = pack_bf16(xv(rb, 2 * tig), xv(rb, 2 * tig + 1));
        a[2] = pack_bf16(xv(ra, 2 * tig + 8), xv(ra, 2 * tig + 9));
        a[3] = pack_bf16(xv(rb, 2 * tig + 8), xv(rb, 2 * tig + 9));
        // layer 1: 8 n-tiles of 8 columns
        float h1[NH / 8][4];
#pragma unroll
        for (int j = 0; j < NH / 8; ++j) {
            const float bl = f.b1[8 * j + 2 * tig], bh = f.b1[8 * j + 2 * tig + 1];
            h1[j][0] = bl;
            h1[j][1] = bh;
            h1[j][2] = bl;
            h1[j][3] = bh;
            mma_bf16(h1[j], a, f.w1[j][lane].x, f.w1[j][lane].y);
        }
        // relu, and re-pack as layer 2's A fragments (k-tile kk = n-tiles 2kk, 2kk+1)
        uint32_t a2[NH / 16][4];
#pragma unroll
        for (int kk = 0; kk < NH / 16; ++kk) {
            const float *c0 = h1[2 * kk], *c1 = h1[2 * kk + 1];
            a2[kk][0] = pack_bf16(fmaxf(c0[0], 0.f), fmaxf(c0[1], 0.f));
            a2[kk][1] = pack_bf16(fmaxf(c0[2], 0.f), fmaxf(c0[3], 0.f));
            a2[kk][2] = pack_bf16(fmaxf(c1[0], 0.f), fmaxf(c1[1], 0.f));
            a2[kk][3] = pack_bf16(fmaxf(c1[2], 0.f), fmaxf(c1[3], 0.f));
        }
        // layer 2 and layer 3 (a dot product with W3, on the CUDA cores)
        float ya = 0.f, yb = 0.f;
#pragma unroll
        for (int j = 0; j < NH / 8; ++j) {
            const float bl = f.b2[8 * j + 2 * tig], bh = f.b2[8 * j + 2 * tig + 1];
            float h2[4] = {bl, bh, bl, bh};
#pragma unroll
            for (int kk = 0; kk < NH / 16; ++kk) mma_bf16(h2, a2[kk], f.w2[kk][j][lane].x, f.w2[kk][j][lane].y);
            const float wl = f.w3[8 * j + 2 * tig], wh = f.w3[8 * j + 2 * tig + 1];
            ya += fmaxf(h2[0], 0.f) * wl + fmaxf(h2[1], 0.f) * wh;
            yb += fmaxf(h2[2], 0.f) * wl + fmaxf(h2[3], 0.f) * wh;
        }
        // sum over the 4 lanes of a group (they hold the row's 64 columns)
        ya += __shfl_xor_sync(FULL, ya, 1);
        ya += __shfl_xor_sync(FULL, ya, 2);
        yb += __shfl_xor_sync(FULL, yb, 1);
        yb += __shfl_xor_sync(FULL, yb, 2);
        if (tig == 0) {
            if (ra < rows) y[ra] = ya + f.b3;
            if (rb < rows) y[rb] = yb + f.b3;
        }
    }
}

// ----- training -----------------------------------------------------------

constexpr int TR_THREADS = 256;

// Both training kernels keep every sum in the order one thread would take it
// (k, j or the sample ascending, one fused multiply-add a term), so the
// weights do not depend on how the work is split over threads.

constexpr uint32_t TR_ROWS = 64;  // samples per forward / backward block
constexpr int TR_PITCH = 68;      // row pitch of the 64-wide tiles (16-byte aligned, no bank conflicts)

struct alignas(16) TrFwdSmem {  // every tile starts on 16 bytes (tr_tile's loads)
    float w1[NIN][TR_PITCH];
    float w2[NH][TR_PITCH];   // [k][j]
    float w2t[NH][TR_PITCH];  // [j][k]
    float xt[NIN][TR_PITCH];  // [k][sample]
    float h1t[NH][TR_PITCH];  // [j][sample]
    float h2t[NH][TR_PITCH];  // [j][sample], then the second layer's gradients
    float b1[NH], b2[NH], w3[NH], dy[TR_ROWS];
    float b3;
};
static_assert(TR_PITCH % 4 == 0, "rows of the tiles start on 16 bytes");
static_assert(offsetof(TrFwdSmem, w2) % 16 == 0 && offsetof(TrFwdSmem, w2t) % 16 == 0 &&
                  offsetof(TrFwdSmem, xt) % 16 == 0 && offsetof(TrFwdSmem, h1t) % 16 == 0 &&
                  offsetof(TrFwdSmem, h2t) % 16 == 0,
              "tiles start on 16 bytes");

// acc[a][b] += p[k][4 * pa + a] * q[k][4 * qb + b] over k ascending.
template <int K>
__device__ __forceinline__ void tr_tile(float (&acc)[4][4], const float (*p)[TR_PITCH], uint32_t pa,
                                        const float (*q)[TR_PITCH], uint32_t qb) {
#pragma unroll 8
    for (int k = 0; k < K; ++k) {
        const float4 u = *reinterpret_cast<const float4 *>(&p[k][4 * pa]);
        const float4 v = *reinterpret_cast<const float4 *>(&q[k][4 * qb]);
        const float uu[4] = {u.x, u.y, u.z, u.w}, vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) acc[x][y] = fmaf(uu[x], vv[y], acc[x][y]);
    }
}

// Forward pass with the inference's roundings (inputs, W1, W2 and the first
// hidden layer in BF16; W3, biases, the second hidden layer and the output in
// FP32), and the backward pass down to the pre-activation gradients of both
// hidden layers, for 64 samples a block. Each product with a weight matrix is
// a 64 x 64 tile in which a thread keeps 4 x 4 outputs in registers and reads
// its operands from shared memory, two 16-byte loads for 16 multiply-adds
// (a thread a sample, its layers in local memory, took 80 us for 8192
// samples; this takes 18).
__global__ void __launch_bounds__(TR_THREADS)
k_train_fwd_bwd(const float *x, const float *label, uint64_t b0, uint32_t bsz, const float *wq,
                float *h1o, float *h2o, float *g1o, float *g2o, float *dyo, float *loss_sq) {
    extern __shared__ __align__(16) unsigned char tr_raw[];
    TrFwdSmem &s = *reinterpret_cast<TrFwdSmem *>(tr_raw);
    const uint32_t tid = threadIdx.x, tj = tid % 16, ts = tid / 16;
    const uint32_t i0 = blockIdx.x * TR_ROWS;
    // the inputs do not depend on the launch before this one
    for (uint32_t t = tid; t < TR_ROWS * NIN; t += TR_THREADS) {
        const uint32_t i = t / NIN, k = t % NIN;
        s.xt[k][i] = i0 + i < bsz ? bf16_round(x[(b0 + i0 + i) * 16 + k]) : 0.f;
    }
    pdl_wait();
    pdl_launch();
    for (uint32_t t = tid; t < (uint32_t)(NIN * NH); t += TR_THREADS) s.w1[t / NH][t % NH] = wq[OFF_W1 + t];
    for (uint32_t t = tid; t < (uint32_t)(NH * NH); t += TR_THREADS) {
        const float w = wq[OFF_W2 + t];
        s.w2[t / NH][t % NH] = w;
        s.w2t[t % NH][t / NH] = w;
    }
    if (tid < (uint32_t)NH) {
        s.b1[tid] = wq[OFF_B1 + tid];
        s.b2[tid] = wq[OFF_B2 + tid];
        s.w3[tid] = wq[OFF_W3 + tid];
    }
    if (tid == 0) s.b3 = wq[OFF_B3];
    __syncthreads();
    float acc[4][4];  // [sample][output]
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int o = 0; o < 4; ++o) acc[c][o] = s.b1[4 * tj + o];
    tr_tile<NIN>(acc, s.xt, ts, s.w1, tj);
#pragma unroll
    for (int o = 0; o < 4; ++o)
#pragma unroll
        for (int c = 0; c < 4; ++c) s.h1t[4 * tj + o][4 * ts + c] = bf16_round(fmaxf(acc[c][o], 0.f));
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int o = 0; o < 4; ++o) acc[c][o] = s.b2[4 * tj + o];
    tr_tile<NH>(acc, s.h1t, ts, s.w2, tj);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint32_t i = i0 + 4 * ts + c;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            acc[c][o] = fmaxf(acc[c][o], 0.f);
            s.h2t[4 * tj + o][4 * ts + c] = acc[c][o];
        }
        if (i < bsz)
            *reinterpret_cast<float4 *>(h2o + (uint64_t)i * NH + 4 * tj) =
                make_float4(acc[c][0], acc[c][1], acc[c][2], acc[c][3]);
    }
    __syncthreads();
    if (tid < TR_ROWS) {
        const uint32_t i = i0 + tid;
        float y = s.b3;
#pragma unroll 16
        for (int j = 0; j < NH; ++j) y = fmaf(s.h2t[j][tid], s.w3[j], y);
        float dy = 0.f;
        if (i < bsz) {
            const float diff = y - label[b0 + i];
            loss_sq[i] = diff * diff;
            dy = 2.f * diff / (float)bsz;
            dyo[i] = dy;
        }
        s.dy[tid] = dy;
    }
    __syncthreads();
    // the second layer's gradients: this thread's own 4 x 4 outputs
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint32_t i = i0 + 4 * ts + c;
        float g[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            g[o] = acc[c][o] > 0.f ? s.dy[4 * ts + c] * s.w3[4 * tj + o] : 0.f;
            s.h2t[4 * tj + o][4 * ts + c] = g[o];
            acc[c][o] = 0.f;
        }
        if (i < bsz)
            *reinterpret_cast<float4 *>(g2o + (uint64_t)i * NH + 4 * tj) = make_float4(g[0], g[1], g[2], g[3]);
    }
    __syncthreads();
    tr_tile<NH>(acc, s.h2t, ts, s.w2t, tj);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint32_t i = i0 + 4 * ts + c;
        if (i >= bsz) continue;
        float h[4], g[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            h[o] = s.h1t[4 * tj + o][4 * ts + c];
            g[o] = h[o] > 0.f ? acc[c][o] : 0.f;
        }
        *reinterpret_cast<float4 *>(h1o + (uint64_t)i * NH + 4 * tj) = make_float4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<float4 *>(g1o + (uint64_t)i * NH + 4 * tj) = make_float4(g[0], g[1], g[2], g[3]);
    }
}

constexpr uint32_t TR_SLICE = 512;    // samples per partial-gradient sum
constexpr uint32_t TR_CHUNK = 64;     // samples staged at a time
constexpr uint32_t TR_PARTS = 10;     // parameter groups: W2 by 8 rows (with b2 in the first), W1 + b1, W3 + b3
constexpr int TRG_THREADS = 128;
constexpr uint32_t TR_STAGES = 4;     // chunks in shared memory: 64 columns of one operand, up to 16 of the other
constexpr int TRG_SMEM = TR_STAGES * TR_CHUNK * (NH + 16) * (int)sizeof(float);

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Partial gradients over a slice of 512 samples, each parameter's sum taken in
// sample order by one thread. A block takes one slice and one group of
// parameters and streams both operands through a ring of four chunks of 64
// samples (asynchronous copies, 80 KB, so that two blocks share an SM and the
// 160 blocks of 8192 samples run at once); a thread holds 2 x 2 sums of W2
// (or 4 x 2 of W1), so that its chains hide each other's latency. 22 us for 8192
// samples, about one block of four warps an SM: the chain of 512 dependent
// multiply-adds is about 1 us of it, the rest the latency of the staged chunks
// and of the shared-memory reads that so few warps cannot hide. (One block a
// slice, a thread a parameter reading global memory: 16 blocks and 470 us.)
__global__ void __launch_bounds__(TRG_THREADS)
k_train_grad_part(const float *x, uint64_t b0, uint32_t bsz, const float *h1, const float *h2,
                  const float *g1, const float *g2, const float *dy, float *part) {
    extern __shared__ __align__(16) unsigned char tr_raw[];
    float(*sa)[NH] = reinterpret_cast<float(*)[NH]>(tr_raw);  // [ring position][64]
    float(*sb)[16] = reinterpret_cast<float(*)[16]>(tr_raw + TR_STAGES * TR_CHUNK * NH * sizeof(float));
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t s0 = blockIdx.x * TR_SLICE, ns = min(bsz - s0, TR_SLICE);
    const uint32_t grp = blockIdx.y;
    float *out = part + (uint64_t)blockIdx.x * MLP_NPARAM;
    const float *wide = grp < 8 ? g2 : (grp == 8 ? g1 : h2);
    const uint32_t nchunk = (ns + TR_CHUNK - 1) / TR_CHUNK;
    auto stage = [&](uint32_t c) {
        if (c < nchunk) {
            const uint32_t i0 = c * TR_CHUNK, m = min(ns - i0, TR_CHUNK), r0 = (c % TR_STAGES) * TR_CHUNK;
            for (uint32_t t = tid; t < m * (NH / 4); t += TRG_THREADS) {
                const uint32_t i = t / (NH / 4), q = 4 * (t % (NH / 4));
                cp_async16(&sa[r0 + i][q], wide + (uint64_t)(s0 + i0 + i) * NH + q);
            }
            if (grp < 8) {  // 8 columns of the first hidden layer
                for (uint32_t t = tid; t < m * 2; t += TRG_THREADS) {
                    const uint32_t i = t / 2, q = 4 * (t % 2);
                    cp_async16(&sb[r0 + i][q], h1 + (uint64_t)(s0 + i0 + i) * NH + 8 * grp + q);
                }
            } else if (grp == 8) {  // the inputs
                for (uint32_t t = tid; t < m * 4; t += TRG_THREADS) {
                    const uint32_t i = t / 4, q = 4 * (t % 4);
                    cp_async16(&sb[r0 + i][q], x + (b0 + s0 + i0 + i) * 16 + q);
                }
            } else {
                for (uint32_t i = tid; i < m; i += TRG_THREADS) cp_async4(&sb[r0 + i][0], dy + s0 + i0 + i);
            }
        }
        cp_async_commit();  // one group a chunk, empty past the last
    };
    pdl_wait();
    pdl_launch();
    for (uint32_t c = 0; c + 1 < TR_STAGES; ++c) stage(c);
    const uint32_t j = 2 * lane;
    float acc[4][2] = {}, ones[2] = {};
    for (uint32_t c = 0; c < nchunk; ++c) {
        cp_async_wait<TR_STAGES - 2>();
        __syncthreads();  // chunk c has arrived, chunk c - 1 is used up
        stage(c + TR_STAGES - 1);
        const uint32_t i0 = (c % TR_STAGES) * TR_CHUNK, i1 = i0 + min(ns - c * TR_CHUNK, TR_CHUNK);
        if (grp < 8) {
            // rows 8 * grp + 2 * warp and the next one of W2
#pragma unroll 8
            for (uint32_t i = i0; i < i1; ++i) {
                const float2 g = *reinterpret_cast<const float2 *>(&sa[i][j]);
                const float2 h = *reinterpret_cast<const float2 *>(&sb[i][2 * warp]);
                acc[0][0] = fmaf(h.x, g.x, acc[0][0]);
                acc[0][1] = fmaf(h.x, g.y, acc[0][1]);
                acc[1][0] = fmaf(h.y, g.x, acc[1][0]);
                acc[1][1] = fmaf(h.y, g.y, acc[1][1]);
                ones[0] += g.x;
                ones[1] += g.y;
            }
        } else if (grp == 8) {
            // rows 4 * warp .. 4 * warp + 3 of W1 for the first three warps, b1 for the last
#pragma unroll 8
            for (uint32_t i = i0; i < i1; ++i) {
                const float2 g = *reinterpret_cast<const float2 *>(&sa[i][j]);
                const float4 v = *reinterpret_cast<const float4 *>(&sb[i][4 * warp]);
                const float vv[4] = {bf16_round(v.x), bf16_round(v.y), bf16_round(v.z), bf16_round(v.w)};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    acc[q][0] = fmaf(vv[q], g.x, acc[q][0]);
                    acc[q][1] = fmaf(vv[q], g.y, acc[q][1]);
                }
                ones[0] += g.x;
                ones[1] += g.y;
            }
        } else if (warp == 0) {
#pragma unroll 8
            for (uint32_t i = i0; i < i1; ++i) {
                const float2 h = *reinterpret_cast<const float2 *>(&sa[i][j]);
                const float v = sb[i][0];
                acc[0][0] = fmaf(h.x, v, acc[0][0]);
                acc[0][1] = fmaf(h.y, v, acc[0][1]);
                ones[0] += v;
            }
        }
    }
    if (grp < 8) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            float *o = out + OFF_W2 + (8 * grp + 2 * warp + q) * NH + j;
            o[0] = acc[q][0];
            o[1] = acc[q][1];
        }
        if (grp == 0 && warp == 0) {
            out[OFF_B2 + j] = ones[0];
            out[OFF_B2 + j + 1] = ones[1];
        }
    } else if (grp == 8) {
        if (warp < 3) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float *o = out + OFF_W1 + (4 * warp + q) * NH + j;
                o[0] = acc[q][0];
                o[1] = acc[q][1];
            }
        } else {
            out[OFF_B1 + j] = ones[0];
            out[OFF_B1 + j + 1] = ones[1];
        }
    } else if (warp == 0) {
        out[OFF_W3 + j] = acc[0][0];
        out[OFF_W3 + j + 1] = acc[0][1];
        if (lane == 0) out[OFF_B3] = ones[0];
    }
}

// Sums of the squared errors over 256 samples of a minibatch each, by a fixed
// tree: block p of minibatch q (of bsz samples, per_batch blocks) of n samples.
__global__ void __launch_bounds__(TR_THREADS)
k_train_loss(const float *sq, uint64_t n, uint32_t bsz, uint32_t per_batch, float *out) {
    __shared__ float red[TR_THREADS];
    const uint64_t m0 = (uint64_t)(blockIdx.x / per_batch) * bsz;
    const uint64_t left = n - m0;
    const uint32_t mb = left < bsz ? (uint32_t)left : bsz;
    const uint32_t i = (blockIdx.x % per_batch) * TR_THREADS + threadIdx.x;
    red[threadIdx.x] = i < mb ? sq[m0 + i] : 0.f;
    __syncthreads();
    for (uint32_t st = TR_THREADS / 2; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = red[0];
}

// grad[p] = sum of the partials in slice order; then Adam on the FP32
// master weights and a BF16-rounded copy for the next forward pass.
__global__ void k_train_adam(const float *part, uint32_t nparts, float *grad, float *w, float *wq,
                             float *m, float *v, float lr, float b1, float b2, float eps,
                             float b1t, float b2t, int apply) {
    pdl_wait();
    pdl_launch();
    for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < (uint32_t)MLP_NPARAM;
         p += gridDim.x * blockDim.x) {
        float g = 0.f;
#pragma unroll 16
        for (uint32_t k = 0; k < nparts; ++k) g += part[(uint64_t)k * MLP_NPARAM + p];
        grad[p] = g;
        if (!apply) continue;
        const float mi = b1 * m[p] + (1.f - b1) * g;
        const float vi = b2 * v[p] + (1.f - b2) * g * g;
        m[p] = mi;
        v[p] = vi;
        const float mh = mi / (1.f - b1t), vh = vi / (1.f - b2t);
        const float wi = w[p] - lr * mh / (sqrtf(vh) + eps);
        w[p] = wi;
        wq[p] = quantised(p, wi);
    }
}

__global__ void k_round_weights(const float *w, float *wq) {
    for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < (uint32_t)MLP_NPARAM;
         p += gridDim.x * blockDim.x)
        wq[p] = quantised(p, w[p]);
}

__global__ void k_log_table(float *tab) {
    const uint32_t a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a < LOG_TAB) tab[a] = feature_transform((long long)a);
}

// Transformed features of trace rows (round, vertex, 12 features).
__global__ void k_rows_to_x(const long long *rows, uint64_t n, const float *tab, float *x) {
    for (uint64_t r = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; r < n;
         r += (uint64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int k = 0; k < 16; ++k) x[r * 16 + k] = k < NIN ? feature_transform(rows[r * 14 + 2 + k], tab) : 0.f;
    }
}

// Training target of trace rows: the transformed score
// x = edge difference + 2 * hierarchy depth (features 4 and 6).
__global__ void k_targets(const long long *rows, uint64_t n, float *y) {
    for (uint64_t r = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; r < n;
         r += (uint64_t)gridDim.x * blockDim.x)
        y[r] = feature_transform(rows[r * 14 + 2 + 4] + 2 * rows[r * 14 + 2 + 6]);
}

}  // namespace

void mlp_targets(const long long *rows, uint64_t n, float *y, cudaStream_t st) {
    if (n == 0) return;
    const uint64_t blocks = std::min<uint64_t>((n + 255) / 256, (uint64_t)device_sm_count() * 8);
    k_targets<<<(unsigned)blocks, 256, 0, st>>>(rows, n, y);
    CH_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------

MlpDevice::MlpDevice() = default;
MlpDevice::~MlpDevice() = default;

void MlpDevice::load(const float *host_weights, cudaStream_t st) {
    weights.alloc(MLP_NPARAM);
    frag.alloc((sizeof(MlpFrag) + 3) / 4);
    logs.alloc(LOG_TAB);
    log_table(logs.ptr, st);
    CH_CUDA_TRY(cudaMemcpyAsync(weights.ptr, host_weights, MLP_NPARAM * sizeof(float),
                                cudaMemcpyHostToDevice, st));
    k_mlp_prepare<<<1, 256, 0, st>>>(weights.ptr, reinterpret_cast<MlpFrag *>(frag.ptr));
    CH_CHECK_LAUNCH();
}

void MlpDevice::infer(const float *x, uint64_t rows, float *y, cudaStream_t st) const {
    if (!rows) return;
    const int blocks = grid_for((rows + 15) / 16, INF_WARPS, device_sm_count() * 8);
    k_mlp_infer<<<blocks, INF_WARPS * 32, 0, st>>>(x, rows, reinterpret_cast<const MlpFrag *>(frag.ptr), y);
    CH_CHECK_LAUNCH();
}

void log_table(float *tab, cudaStream_t st) {
    k_log_table<<<LOG_TAB / 64, 64, 0, st>>>(tab);
    CH_CHECK_LAUNCH();
}

void rows_to_features(const long long *rows, uint64_t n, const float *tab, float *x, cudaStream_t st) {
    if (!n) return;
    k_rows_to_x<<<grid_for(n, 256, device_sm_count() * 8), 256, 0, st>>>(rows, n, tab, x);
    CH_CHECK_LAUNCH();
}

void mlp_train(const long long *rows, const float *labels, uint64_t n, const ch_train_params_t *tp,
               float *weights_io, float *loss_out, float *grad_out, cudaStream_t st) {
    DevBuf<float> logs, x, w, wq, m, v, grad, h1, h2, g1, g2, dy, part, sq, lpart;
    logs.alloc(LOG_TAB);
    log_table(logs.ptr, st);
    x.alloc(n * 16);
    rows_to_features(rows, n, logs.ptr, x.ptr, st);
    w.alloc(MLP_NPARAM);
    wq.alloc(MLP_NPARAM);
    m.alloc(MLP_NPARAM);
    v.alloc(MLP_NPARAM);
    grad.alloc(MLP_NPARAM);
    m.zero(st);
    v.zero(st);
    CH_CUDA_TRY(cudaMemcpyAsync(w.ptr, weights_io, MLP_NPARAM * 4, cudaMemcpyDeviceToDevice, st));
    k_round_weights<<<20, 256, 0, st>>>(w.ptr, wq.ptr);
    CH_CHECK_LAUNCH();
    const uint32_t B = std::max<uint32_t>(1, std::min<uint64_t>(tp->batch, n));
    h1.alloc((uint64_t)B * MLP_NH);
    h2.alloc((uint64_t)B * MLP_NH);
    g1.alloc((uint64_t)B * MLP_NH);
    g2.alloc((uint64_t)B * MLP_NH);
    dy.alloc(B);
    const uint32_t nparts = (B + TR_SLICE - 1) / TR_SLICE;
    part.alloc((uint64_t)nparts * MLP_NPARAM);
    float b1t = 1.f, b2t = 1.f;
    const bool apply = tp->epochs > 0;
    const uint32_t epochs = apply ? tp->epochs : 1;
    const uint64_t seen = apply ? n : B;  // samples an epoch goes over
    // squared errors of an epoch, summed and read back once at its end: no
    // step waits for the host
    const uint32_t per_batch = (B + TR_THREADS - 1) / TR_THREADS;
    const uint64_t lblocks = (seen + B - 1) / B * per_batch;
    if (lblocks > 0x7FFFFFFFull) throw Error{CH_ERANGE, "too many minibatches"};
    sq.alloc(seen);
    lpart.alloc(lblocks);
    std::vector<float> hl(lblocks);
    CH_CUDA_TRY(cudaFuncSetAttribute(k_train_fwd_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(TrFwdSmem)));
    CH_CUDA_TRY(cudaFuncSetAttribute(k_train_grad_part, cudaFuncAttributeMaxDynamicSharedMemorySize, TRG_SMEM));
    for (uint32_t ep = 0; ep < epochs; ++ep) {
        double ep_loss = 0;
        for (uint64_t b0 = 0; b0 < seen; b0 += B) {
            const uint32_t bsz = (uint32_t)std::min<uint64_t>(B, n - b0);
            launch_pdl(k_train_fwd_bwd, (bsz + TR_ROWS - 1) / TR_ROWS, TR_THREADS, sizeof(TrFwdSmem), st, x.ptr,
                       labels, b0, bsz, wq.ptr, h1.ptr, h2.ptr, g1.ptr, g2.ptr, dy.ptr, sq.ptr + b0);
            const uint32_t np = (bsz + TR_SLICE - 1) / TR_SLICE;
            launch_pdl(k_train_grad_part, dim3(np, TR_PARTS), TRG_THREADS, TRG_SMEM, st, x.ptr, b0, bsz, h1.ptr,
                       h2.ptr, g1.ptr, g2.ptr, dy.ptr, part.ptr);
            b1t *= tp->beta1;
            b2t *= tp->beta2;
            launch_pdl(k_train_adam, 20, 256, 0, st, part.ptr, np, grad.ptr, w.ptr, wq.ptr, m.ptr, v.ptr, tp->lr,
                       tp->beta1, tp->beta2, tp->eps, b1t, b2t, apply ? 1 : 0);
        }
        k_train_loss<<<(unsigned)lblocks, TR_THREADS, 0, st>>>(sq.ptr, seen, B, per_batch, lpart.ptr);
        CH_CHECK_LAUNCH();
        CH_CUDA_TRY(cudaMemcpyAsync(hl.data(), lpart.ptr, lblocks * 4, cudaMemcpyDeviceToHost, st));
        CH_CUDA_TRY(cudaStreamSynchronize(st));
        for (const float l : hl) ep_loss += l;
        if (loss_out) loss_out[ep] = (float)(ep_loss / (double)seen);
    }
    if (apply)
        CH_CUDA_TRY(cudaMemcpyAsync(weights_io, w.ptr, MLP_NPARAM * 4, cudaMemcpyDeviceToDevice, st));
    if (grad_out)
        CH_CUDA_TRY(cudaMemcpyAsync(grad_out, grad.ptr, MLP_NPARAM * 4, cudaMemcpyDeviceToDevice, st));
    CH_CUDA_TRY(cudaStreamSynchronize(st));
}

}  // namespace gbch
