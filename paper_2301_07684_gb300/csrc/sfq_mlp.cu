// sfq_mlp.cu -- the learned inverse-CDF surrogate for photon emission: a 2 -> 64 -> 64 ->
// 64 -> 1 SiLU network that maps (ln chi, u) to the paper's inverse-CDF variable w-bar
// (Eq. again), and from it xi = s / (1 + s) with s = 3 chi w-bar^3 / 2 (Eq. subs_altri).
//
//   features  x1 = (ln chi - C_CHI) / S_CHI,  x2 = L / 8 - 1,  L = -ln(1 - u)
//   output    y  = network(x1, x2),  ln w-bar = y + ln u
//
// Training runs on the GPU in binary32 (SIMT kernels written here: forward, backward with
// per-block gradient partials reduced in a fixed order, Adam).  With `quantize`, the
// forward pass rounds the weights and the inputs of layers 2-4 to bfloat16 exactly as the
// inference kernel does (the rounding is passed straight through in the backward pass).
// Inference runs layers 2-4 on the tensor cores (tcgen05.mma, bfloat16 operands staged in
// shared memory, binary32 accumulators in tensor memory, read back with tcgen05.ld); layer
// 1 and the SiLU epilogues run on the CUDA cores.  Cells
// of (ln chi, u) where the network disagrees with the plain fitted sampler by more than a
// tolerance in u (a bound on its contribution to the KS distance of the sampled energies)
// are flagged by sfq_mlp_calibrate; draws in flagged cells, and chi outside the training
// range [1e-3, 100], use the plain sampler.
#include "sfq_mlp.cuh"

namespace sfq {
namespace mlp {

// ---------------------------------------------------------------------------------------
// Initialisation: U(-1/sqrt(fan_in), 1/sqrt(fan_in)) for weights and biases (Philox).
__global__ void init_kernel(float *p, uint64_t seed) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NP) return;
    const float fan = i < O_W2 ? 2.0f : 64.0f;
    const u4 w = draws(seed, (uint64_t)i, 0, 7);
    p[i] = (2.0f * uniform<float>(w.w[0]) - 1.0f) * rsqrtf(fan);
}

// ---------------------------------------------------------------------------------------
// Training: forward and backward of TS samples per block, gradient partial per block.
// Rows of LD = 68 floats: 16-byte aligned, so that four consecutive elements of a row are one
// vector load, and 8 lanes reading 16 bytes of 8 successive rows hit all 32 banks once.
constexpr int TS = 64, TB = 256, LD = 68;
constexpr int TR = TS / (TB / 32);                 // rows of a 64 x 64 product per warp
struct TrainSmem {
    float w2[H * LD], w3[H * LD];
    float z1[TS * LD], a1[TS * LD], z2[TS * LD], a2[TS * LD], z3[TS * LD], a3[TS * LD];
    float w1[H * 2], b1[H], b2[H], b3[H], w4[H], b4;
    float x[TS * 2], yt[TS], dy[TS];
    int valid[TS];
    float red[TS];
};

struct TrainArgs {
    const float *params;
    int64_t n;
    const float *chi, *u, *lnw;
    int64_t base;          // sequential mode: first sample of block 0
    int random;            // 1: minibatch indices drawn by Philox(seed, k, step)
    uint64_t seed;
    uint32_t step;
    int quantize;
    float scale;           // d loss / d y = scale * r  (2 / batch)
    float *partial;        // [gridDim.x][NPS]
    float *partial_loss;   // [gridDim.x]
    Kind K;
};

// The three 64 x 64 x 64 products of a layer.  Each warp holds a TR x 64 strip of the result, a
// thread TR rows x 2 columns of it, and every element is summed in the order of the inner
// index with one fused multiply-add each.  What bounded them was the shared-memory pipe: with
// one row element and one column element loaded per inner index (17 loads for 16
// multiply-adds) the kernel took 44 us for 8192 samples.  Rows are read four elements at a
// time and shared by the warp (a broadcast), columns as pairs: 16 passes of the pipe for 64
// multiply-adds of a thread, 22 us.  Measured and no faster: 16 warps of 4 rows (24 passes for
// 64, 22 us); the next operands loaded ahead of the arithmetic (26 us, more moves).
__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float2 ld2(const float *p) { return *reinterpret_cast<const float2 *>(p); }

// Z[s][j] = sum_k A[s][k] W[j][k] + b[j] over the block's samples; Aout = SiLU(Z).
// The thread's columns: j = lane, lane + 32.
__device__ __forceinline__ void layer_fwd(const float *A, const float *W, const float *b, float *Z, float *Aout,
                                          bool q) {
    const int lane = threadIdx.x & 31, s0 = (threadIdx.x >> 5) * TR;
    float acc[TR][2];
#pragma unroll
    for (int r = 0; r < TR; ++r) {
        acc[r][0] = b[lane];
        acc[r][1] = b[lane + 32];
    }
#pragma unroll 4
    for (int k = 0; k < H; k += 4) {
        const float4 w0 = ld4(W + lane * LD + k), w1 = ld4(W + (lane + 32) * LD + k);
#pragma unroll
        for (int r = 0; r < TR; ++r) {
            const float4 v = ld4(A + (s0 + r) * LD + k);
            acc[r][0] = fmaf(v.w, w0.w, fmaf(v.z, w0.z, fmaf(v.y, w0.y, fmaf(v.x, w0.x, acc[r][0]))));
            acc[r][1] = fmaf(v.w, w1.w, fmaf(v.z, w1.z, fmaf(v.y, w1.y, fmaf(v.x, w1.x, acc[r][1]))));
        }
    }
#pragma unroll
    for (int r = 0; r < TR; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int e = (s0 + r) * LD + lane + 32 * c;
            Z[e] = acc[r][c];
            Aout[e] = qz(silu(acc[r][c]), q);
        }
}
// gW[j][k] = sum_s dZ[s][j] A[s][k]  (written to g[j * 64 + k]),  gb[j] = sum_s dZ[s][j].
// The thread's columns: k = 2 lane, 2 lane + 1.
__device__ __forceinline__ void layer_gw(const float *dZ, const float *A, float *g, float *gb) {
    const int k = 2 * (threadIdx.x & 31), j0 = (threadIdx.x >> 5) * TR;
    float acc[TR][2];
#pragma unroll
    for (int r = 0; r < TR; ++r) acc[r][0] = acc[r][1] = 0.0f;
#pragma unroll 8
    for (int s = 0; s < TS; ++s) {
        const float2 av = ld2(A + s * LD + k);
        const float4 d0 = ld4(dZ + s * LD + j0), d1 = ld4(dZ + s * LD + j0 + 4);
        const float d[TR] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
        for (int r = 0; r < TR; ++r) {
            acc[r][0] = fmaf(d[r], av.x, acc[r][0]);
            acc[r][1] = fmaf(d[r], av.y, acc[r][1]);
        }
    }
#pragma unroll
    for (int r = 0; r < TR; ++r) *reinterpret_cast<float2 *>(g + (j0 + r) * H + k) = make_float2(acc[r][0], acc[r][1]);
    if (threadIdx.x < H) {
        float sb = 0.0f;
#pragma unroll 16
        for (int s = 0; s < TS; ++s) sb += dZ[s * LD + threadIdx.x];
        gb[threadIdx.x] = sb;
    }
}
// dA[s][k] = sum_j dZ[s][j] W[j][k]; then dZprev[s][k] = dA[s][k] * silu'(Zprev[s][k]) in place
// (a thread owns the elements it updates).  The thread's columns: k = 2 lane, 2 lane + 1.
__device__ __forceinline__ void layer_bwd_input(const float *dZ, const float *W, float *Zprev) {
    const int k = 2 * (threadIdx.x & 31), s0 = (threadIdx.x >> 5) * TR;
    float acc[TR][2];
#pragma unroll
    for (int r = 0; r < TR; ++r) acc[r][0] = acc[r][1] = 0.0f;
#pragma unroll 4
    for (int j = 0; j < H; j += 4) {
        const float2 w0 = ld2(W + j * LD + k), w1 = ld2(W + (j + 1) * LD + k), w2 = ld2(W + (j + 2) * LD + k),
                     w3 = ld2(W + (j + 3) * LD + k);
#pragma unroll
        for (int r = 0; r < TR; ++r) {
            const float4 d = ld4(dZ + (s0 + r) * LD + j);
            acc[r][0] = fmaf(d.w, w3.x, fmaf(d.z, w2.x, fmaf(d.y, w1.x, fmaf(d.x, w0.x, acc[r][0]))));
            acc[r][1] = fmaf(d.w, w3.y, fmaf(d.z, w2.y, fmaf(d.y, w1.y, fmaf(d.x, w0.y, acc[r][1]))));
        }
    }
#pragma unroll
    for (int r = 0; r < TR; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            float *z = Zprev + (s0 + r) * LD + k + c;
            *z = acc[r][c] * dsilu(*z);
        }
}

__global__ void __launch_bounds__(TB) train_kernel(const TrainArgs a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    TrainSmem &S = *reinterpret_cast<TrainSmem *>(smraw);
    const bool q = a.quantize != 0;
    const int tid = threadIdx.x;
    const float *P = a.params;
    // the minibatch is gathered first, so that its round trip overlaps the weights' one
    float chi = 1.0f, u = 0.5f, lw = 0.0f;
    bool ok = false;
    if (tid < TS) {
        int64_t idx;
        if (a.random) {
            const u4 w = draws(a.seed, (uint64_t)blockIdx.x * TS + tid, a.step, 5);
            idx = (int64_t)(((uint64_t)w.w[0] * (uint64_t)a.n) >> 32);
            ok = true;
        } else {
            idx = a.base + (int64_t)blockIdx.x * TS + tid;
            ok = idx < a.n;
        }
        if (ok) {
            chi = a.chi[idx];
            u = a.u[idx];
            lw = a.lnw[idx];
        }
    }
#pragma unroll
    for (int e = 4 * tid; e < H * H; e += 4 * TB) {
        const int j = e >> 6, k = e & 63;
        const float4 v2 = ld4(P + O_W2 + e), v3 = ld4(P + O_W3 + e);
        *reinterpret_cast<float4 *>(S.w2 + j * LD + k) = make_float4(qz(v2.x, q), qz(v2.y, q), qz(v2.z, q), qz(v2.w, q));
        *reinterpret_cast<float4 *>(S.w3 + j * LD + k) = make_float4(qz(v3.x, q), qz(v3.y, q), qz(v3.z, q), qz(v3.w, q));
    }
    if (tid < H) {
        S.w1[2 * tid] = qz(P[O_W1 + 2 * tid], q);
        S.w1[2 * tid + 1] = qz(P[O_W1 + 2 * tid + 1], q);
        S.b1[tid] = P[O_B1 + tid];
        S.b2[tid] = P[O_B2 + tid];
        S.b3[tid] = P[O_B3 + tid];
        S.w4[tid] = qz(P[O_W4 + tid], q);
    }
    if (tid == 0) S.b4 = P[O_B4];
    if (tid < TS) {
        ok = ok && isfinite(lw);          // samples without a target (NaN) do not enter the loss
        if (!ok) { chi = 1.0f; u = 0.5f; lw = 0.0f; }
        float x1, x2;
        features(a.K, chi, u, x1, x2);
        S.x[2 * tid] = x1;
        S.x[2 * tid + 1] = x2;
        S.yt[tid] = lw - out_offset(a.K, u);
        S.valid[tid] = ok;
    }
    __syncthreads();
    // layer 1 (2 -> 64)
    {
        const int j = tid & 63, s0 = tid >> 6;
#pragma unroll
        for (int r = 0; r < TS * 64 / TB; ++r) {
            const int s = s0 + TB / 64 * r;
            const float z = fmaf(S.w1[2 * j], S.x[2 * s], fmaf(S.w1[2 * j + 1], S.x[2 * s + 1], S.b1[j]));
            S.z1[s * LD + j] = z;
            S.a1[s * LD + j] = qz(silu(z), q);
        }
    }
    __syncthreads();
    layer_fwd(S.a1, S.w2, S.b2, S.z2, S.a2, q);
    __syncthreads();
    layer_fwd(S.a2, S.w3, S.b3, S.z3, S.a3, q);
    __syncthreads();
    // layer 4 (64 -> 1): four threads per sample
    if (tid < 4 * TS) {
        const int s = tid >> 2, part = tid & 3;
        float acc = 0.0f;
        for (int k = part * 16; k < part * 16 + 16; ++k) acc = fmaf(S.a3[s * LD + k], S.w4[k], acc);
        acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 1);
        acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 2);
        if (part == 0) {
            const float y = acc + S.b4;
            const float r = S.valid[s] ? y - S.yt[s] : 0.0f;
            S.dy[s] = a.scale * r;
            S.red[s] = r * r;
        }
    }
    __syncthreads();
    float *G = a.partial + (size_t)blockIdx.x * NPS;
    if (tid == 0) {
        float l = 0.0f, gb = 0.0f;
#pragma unroll 16
        for (int s = 0; s < TS; ++s) {
            l += S.red[s];
            gb += S.dy[s];
        }
        a.partial_loss[blockIdx.x] = l;
        G[O_B4] = gb;
    }
    // layer 4 backward: gW4, and dZ3 = (dy w4) * silu'(z3) in place
    if (tid < H) {
        float g = 0.0f;
#pragma unroll 16
        for (int s = 0; s < TS; ++s) g = fmaf(S.dy[s], S.a3[s * LD + tid], g);
        G[O_W4 + tid] = g;
    }
    __syncthreads();
    {
        const int k = tid & 63, s0 = tid >> 6;
#pragma unroll
        for (int r = 0; r < TS * 64 / TB; ++r) {
            const int s = s0 + TB / 64 * r;
            S.z3[s * LD + k] = S.dy[s] * S.w4[k] * dsilu(S.z3[s * LD + k]);
        }
    }
    __syncthreads();
    layer_gw(S.z3, S.a2, G + O_W3, G + O_B3);
    layer_bwd_input(S.z3, S.w3, S.z2);          // z2 <- dZ2
    __syncthreads();
    layer_gw(S.z2, S.a1, G + O_W2, G + O_B2);
    layer_bwd_input(S.z2, S.w2, S.z1);          // z1 <- dZ1
    __syncthreads();
    if (tid < H) {
        float g0 = 0.0f, g1 = 0.0f, gb = 0.0f;
#pragma unroll 16
        for (int s = 0; s < TS; ++s) {
            const float d = S.z1[s * LD + tid];
            g0 = fmaf(d, S.x[2 * s], g0);
            g1 = fmaf(d, S.x[2 * s + 1], g1);
            gb += d;
        }
        G[O_W1 + 2 * tid] = g0;
        G[O_W1 + 2 * tid + 1] = g1;
        G[O_B1 + tid] = gb;
    }
}

// Sum of the per-block partials in a fixed order (deterministic), and with ADAM the parameter's
// Adam step from it.  A parameter is one chain of nb additions.  A block takes RP parameters:
// its RB threads fetch the terms of RC partials at a time into shared memory, all loads in
// flight together, and one thread per parameter adds them up.  So the kernel is one round
// trip to L2 per RC partials.  The loss is a block of its own, summed by a warp in binary64,
// lanes first: one thread's chain of binary64 additions (about 220 cycles each with the
// widening) had made the kernel 18 us for 128 partials and 110 us for 1025.
constexpr int RP = 64, RB = 512, RC = 128, RBLOCKS = (NP + RP - 1) / RP + 1;
template <bool ADAM>
__global__ void __launch_bounds__(RB) reduce_kernel(const float *__restrict__ partial,
                                                    const float *__restrict__ partial_loss, int nb,
                                                    float *__restrict__ grad, float *__restrict__ loss,
                                                    float loss_scale, float *__restrict__ params,
                                                    float *__restrict__ mom, float *__restrict__ var, float lr,
                                                    float b1t, float b2t) {
    if (blockIdx.x == RBLOCKS - 1) {
        if (!loss || threadIdx.x >= 32) return;
        double l = 0.0;
        for (int b = threadIdx.x; b < nb; b += 32) l += partial_loss[b];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xFFFFFFFFu, l, o);
        if (threadIdx.x == 0) *loss = (float)(l * loss_scale);
        return;
    }
    __shared__ float term[RC][RP];
    const int c = threadIdx.x & (RP - 1), p = blockIdx.x * RP + c;
    float g = 0.0f;
    for (int b0 = 0; b0 < nb; b0 += RC) {
        const int m = nb - b0 < RC ? nb - b0 : RC;
        float v[RC * RP / RB];
#pragma unroll
        for (int k = 0; k < RC * RP / RB; ++k) {
            const int b = threadIdx.x / RP + RB / RP * k;
            v[k] = b < m && p < NP ? partial[(size_t)(b0 + b) * NPS + p] : 0.0f;
        }
        if (b0) __syncthreads();                    // the previous terms have been added
#pragma unroll
        for (int k = 0; k < RC * RP / RB; ++k) term[threadIdx.x / RP + RB / RP * k][c] = v[k];
        __syncthreads();
        if (threadIdx.x < RP) {
            if (m == RC) {
#pragma unroll 32
                for (int b = 0; b < RC; ++b) g += term[b][c];
            } else {
                for (int b = 0; b < m; ++b) g += term[b][c];
            }
        }
    }
    if (threadIdx.x >= RP || p >= NP) return;
    if (!ADAM) {
        grad[p] = g;
        return;
    }
    const float mi = 0.9f * mom[p] + 0.1f * g;
    const float vi = 0.999f * var[p] + 0.001f * g * g;
    mom[p] = mi;
    var[p] = vi;
    const float mh = mi / (1.0f - b1t), vh = vi / (1.0f - b2t);
    params[p] -= lr * mh / (sqrtf(vh) + 1e-8f);
}

// ---------------------------------------------------------------------------------------
// Tensor-core inference.  One block of 128 threads handles tiles of 256 samples (two per
// thread, one row of each of two 128 x 64 activation operands).  Layers 2 and 3 are, for each,
//   D[128 x 64] (fp32, tensor memory) = A[128 x 64] (bf16, smem) * W^T (W: 64 x 64 bf16, smem)
// issued as four K = 16 steps of tcgen05.mma.kind::f16 by one thread; the output layer is
// the same with a 16 x 64 W whose row 0 is w4 (column 0 of D is the output).  Operands use the
// no-swizzle K-major layout: 8-row x 16-byte core matrices, core matrix (row group g, K
// chunk j) at ((g * 8) + j) * 128 bytes, i.e. K-adjacent core matrices 128 bytes apart
// (leading byte offset) and row groups 1024 bytes apart (stride byte offset).
constexpr uint32_t MMA_WAIT_LIMIT = 1u << 22;
constexpr int IT = 128;                       // threads of a block, rows of an activation operand
constexpr int IS = 2 * IT;                    // samples per tile: two per thread
constexpr uint32_t TMEM_COLS = 128;           // an accumulator of 64 columns for each
// kind::f16 instruction descriptor: D f32 (bit 4), A bf16 (bits 7-9 = 1), B bf16 (bits
// 10-12 = 1), both K-major, N >> 3 at bits 17-22, M >> 4 at bits 24-28.
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((64u >> 3) << 17) | ((128u >> 4) << 24);
// the output layer: N = 16 (row 0 of its B operand holds w4, rows 1-15 are zero)
constexpr uint32_t IDESC4 = (1u << 4) | (1u << 7) | (1u << 10) | ((16u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ uint32_t s_u32(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
    const uint64_t lbo = 128, sbo = 1024;
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((lbo >> 4) << 16) | ((sbo >> 4) << 32) | (1ull << 46);
}
__device__ __forceinline__ void mbar_init1(uint64_t *bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s_u32(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity) {
    const uint32_t ad = s_u32(bar);
    for (uint32_t it = 0; it < MMA_WAIT_LIMIT; ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(ad), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void mma_k16(uint32_t d_tmem, uint64_t ad, uint64_t bd, uint32_t accumulate,
                                        uint32_t idesc = IDESC) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s_u32(bar))
                 : "memory");
}
// 16 consecutive fp32 columns of this thread's lane, of two accumulators (one wait for both).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t *r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16x2(uint32_t t0, uint32_t t1, float (&v)[2][16]) {
    uint32_t r[2][16];
    tmem_ld16(t0, r[0]);
    tmem_ld16(t1, r[1]);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int k = 0; k < 16; ++k) v[h][k] = __uint_as_float(r[h][k]);
}
// Column 0 of this thread's lane.
__device__ __forceinline__ float tmem_ld1(uint32_t taddr) {
    uint32_t r;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    return __uint_as_float(r);
}
// Row m of a 128 x 64 (or 64 x 64) K-major operand: 8 chunks of 8 bf16 (16 bytes).
__device__ __forceinline__ uint32_t row_chunk_offset(int m, int j) {
    return (uint32_t)((((m >> 3) * 8) + j) * 128 + (m & 7) * 16);
}
// The finishing of queued photon emissions (APPLY): the emitter's state before the event,
// its population, and the product records (sfq_set_surrogate).
struct ApplyOut {
    const int64_t *idx;
    const float *g, *px, *py, *pz;
    float *ppx, *ppy, *ppz;
    uint8_t *flags;
    const uint64_t *id;
    uint64_t id_base;
    int64_t cap;
    float *opx, *opy, *opz;
    uint64_t *opid;
    uint32_t *ostep;
    uint8_t *ometa;
    unsigned long long *ocount;
    uint32_t step;
};

struct InferArgs {
    const float *params;
    const uint8_t *flags;     // NULL: no calibration (every in-range draw uses the network)
    const float *inv;         // plain inverse-CDF table (fallback)
    int64_t n;
    const float *chi, *r;
    float *xi, *xi_c;
    sfq_counters *counters;
    int *status;              // set to 1 when a bounded wait gave up
    Kind K;                   // photon: xi, xi_c = 1 - xi; pair: xi = electron share, xi_c = positron share
    const unsigned long long *n_dev;   // APPLY: device count of queued samples (min with n)
    ApplyOut ap;
};

// Warp-wide reservation of one slot per lane that wants one: one atomic per warp.
__device__ __forceinline__ unsigned long long warp_reserve(unsigned long long *ctr, bool want) {
    const unsigned m = __ballot_sync(0xFFFFFFFFu, want);
    const int lane = threadIdx.x & 31;
    const int leader = m ? __ffs(m) - 1 : 0;
    unsigned long long base = 0;
    if (m && lane == leader) base = atomicAdd(ctr, (unsigned long long)__popc(m));
    base = __shfl_sync(0xFFFFFFFFu, base, leader);
    return base + (unsigned long long)__popc(m & ((1u << lane) - 1u));
}

// Operands (no-swizzle K-major, 16-byte aligned): A 128 x 64 for each half of the tile, W2 and W3 64 x 64, W4 16 x 64;
// then layer 1's weights, the halved biases of layers 2 and 3, b4 and the fallback flags.
constexpr uint32_t SM_A = 0, SM_A1 = 16384, SM_B2 = 32768, SM_B3 = SM_B2 + 8192, SM_B4 = SM_B3 + 8192,
                   SM_SMALL = SM_B4 + 2048;
constexpr uint32_t SM_FLAGS = SM_SMALL + ((H * 2 + 3 * H + 1) * 4 + 15) / 16 * 16;
constexpr uint32_t SM_BYTES = SM_FLAGS + NCELL / 8;    // the fallback flags as one bit per cell
constexpr uint32_t INFER_SMEM = SM_BYTES + 128;      // + alignment slack
#ifndef SFQ_INFER_MINB
#define SFQ_INFER_MINB 4
#endif
// resident blocks per SM (registers, 53 KB of shared memory, 128 of 512 TMEM columns each)
constexpr int INFER_MINB = SFQ_INFER_MINB;

// SiLU of two units in packed registers: silu_h for each, one multiply-add for both.
__device__ __forceinline__ f32x2 silu_h2(f32x2 h) {
    float a, b, ta, tb;
    h.get(a, b);
    asm("tanh.approx.f32 %0, %1;" : "=f"(ta) : "f"(a));
    asm("tanh.approx.f32 %0, %1;" : "=f"(tb) : "f"(b));
    return fma2(h, f32x2(ta, tb), h);
}
// Eight bfloat16 (one 16-byte K chunk of an operand row) from four pairs.
__device__ __forceinline__ uint32_t pack_bf16(f32x2 v) {
    float a, b;
    v.get(a, b);
    __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&p);
}
__device__ __forceinline__ uint4 pack8_bf16(const f32x2 *v) {
    return make_uint4(pack_bf16(v[0]), pack_bf16(v[1]), pack_bf16(v[2]), pack_bf16(v[3]));
}
// Four consecutive binary32 values as two pairs (a broadcast from shared memory).
__device__ __forceinline__ void lds_pairs(const float *p, f32x2 &a, f32x2 &b) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(p);
    a = f32x2((uint64_t)v.x);
    b = f32x2((uint64_t)v.y);
}

// The epilogue of a hidden tensor-core layer for this thread's two rows, 16 accumulator columns
// of each at a time: h = (d + b) / 2 from the halved biases hb (one load for both rows),
// SiLU, and the bfloat16 rows of the next layer's operands.
__device__ __forceinline__ void epilogue(uint32_t t_row, const float *hb, unsigned char *a_base, int row) {
    const f32x2 half2(0.5f, 0.5f);
#pragma unroll
    for (int part = 0; part < 4; ++part) {
        float d[2][16];
        tmem_ld16x2(t_row + 16 * part, t_row + 64 + 16 * part, d);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            f32x2 b[4];
            lds_pairs(hb + 16 * part + 8 * c, b[0], b[1]);
            lds_pairs(hb + 16 * part + 8 * c + 4, b[2], b[3]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                f32x2 v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    v[q] = silu_h2(fma2(half2, f32x2(d[h][8 * c + 2 * q], d[h][8 * c + 2 * q + 1]), b[q]));
                *reinterpret_cast<uint4 *>(a_base + h * (SM_A1 - SM_A) + row_chunk_offset(row, 2 * part + c)) = pack8_bf16(v);
            }
        }
    }
}

// One block of 128 threads walks over tiles of 256 samples (two per thread, a row of each of
// two 128 x 64 activation operands); INFER_MINB blocks share an SM, so that the tensor
// cores of one block's layer run while the others compute their SiLU epilogues.  The
// epilogues bound it: 192 tanh per draw keep the special-function pipe 69 % busy (611 us for
// 1e7 draws; at 100 % they would take 422).  A weight or bias that every lane reads costs the
// shared-memory pipe as much as 32 different ones, so one read serves both samples (39 % of
// that pipe; 58 % with one sample per thread, 618 us), and packed registers halve the
// multiply-adds (1314 -> 943 instructions per draw and warp).  Letting the halves alternate,
// each with its own MMA group in flight, was slower (660 us: twice the barriers).
// APPLY (photon kind): the samples are the queued emissions of a Monte Carlo step; each
// sampled xi also recoils its emitter (Sec. 3: the lepton keeps (1 - xi) gamma along its
// direction) and appends the collinear photon's record.
template <bool APPLY>
__global__ void __launch_bounds__(IT, INFER_MINB) infer_tc_kernel(const InferArgs a) {
    extern __shared__ unsigned char sraw[];
    __shared__ uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ unsigned long long s_cnt[6];
    // 128-byte aligned operand area (the no-swizzle layout needs 16-byte alignment)
    const uint32_t raw = s_u32(sraw);
    unsigned char *sm = sraw + ((128u - (raw & 127u)) & 127u);
    const uint32_t sbase = s_u32(sm);
    float *w1 = reinterpret_cast<float *>(sm + SM_SMALL);
    float *b1 = w1 + 2 * H, *hb2 = b1 + H, *hb3 = hb2 + H, *b4 = hb3 + H;
    uint32_t *fl = reinterpret_cast<uint32_t *>(sm + SM_FLAGS);
    const int tid = threadIdx.x, warp = tid >> 5;
    const float *P = a.params;

    // weights: W2, W3 and W4 (row 0 of a 16-row operand, the other rows zero) as bf16 in the
    // K-major core-matrix layout; layer 1 binary32 (bf16-rounded weights); the biases of
    // layers 2 and 3 halved for the SiLU form
    for (int e = tid; e < H * H; e += IT) {
        const int n_ = e >> 6, k = e & 63;
        const uint32_t off = row_chunk_offset(n_, k >> 3) + (k & 7) * 2;
        *reinterpret_cast<__nv_bfloat16 *>(sm + SM_B2 + off) = __float2bfloat16_rn(P[O_W2 + e]);
        *reinterpret_cast<__nv_bfloat16 *>(sm + SM_B3 + off) = __float2bfloat16_rn(P[O_W3 + e]);
    }
    for (int e = tid; e < 16 * H; e += IT) {
        const int n_ = e >> 6, k = e & 63;
        const uint32_t off = row_chunk_offset(n_, k >> 3) + (k & 7) * 2;
        *reinterpret_cast<__nv_bfloat16 *>(sm + SM_B4 + off) = __float2bfloat16_rn(n_ == 0 ? P[O_W4 + k] : 0.0f);
    }
    for (int e = tid; e < H; e += IT) {
        // layer 1 halved as well (exact: a power of two), so that h = z / 2 comes out of its fmas
        w1[e] = 0.5f * bf16r(P[O_W1 + 2 * e]);
        w1[H + e] = 0.5f * bf16r(P[O_W1 + 2 * e + 1]);
        b1[e] = 0.5f * P[O_B1 + e];
        hb2[e] = 0.5f * P[O_B2 + e];
        hb3[e] = 0.5f * P[O_B3 + e];
    }
    if (tid == 0) *b4 = P[O_B4];
    for (int e = tid; e < NCELL / 32; e += IT) {
        uint32_t w = 0;
        if (a.flags)
            for (int b = 0; b < 32; ++b) w |= (a.flags[32 * e + b] ? 1u : 0u) << b;
        fl[e] = w;
    }
    if (tid < 6) s_cnt[tid] = 0;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_u32(&tmem_base)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        mbar_init1(&mbar);
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = tmem_base;
    const uint32_t t_row = taddr + ((uint32_t)(warp * 32) << 16);
    uint32_t phase = 0;
    uint32_t n_nan = 0, n_oor = 0, n_fb = 0, n_emit = 0, n_drop = 0, n_g1 = 0;
    int64_t n_all = a.n;
    if (APPLY) {
        const int64_t q = (int64_t)*a.n_dev;
        n_all = q < n_all ? q : n_all;
    }
    const int64_t ntiles = (n_all + IS - 1) / IS;
    int late = 0;                                 // this thread gave up waiting for an MMA group

    // the inputs of the block's next tile are loaded a tile ahead, so that their latency falls
    // in the current tile's work
    float chi_n[2], r_n[2];
    const auto fetch = [&](int64_t tile) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t i = tile * IS + h * IT + tid;
            chi_n[h] = 1.0f;
            r_n[h] = 0.5f;
            if (i < n_all) { chi_n[h] = a.chi[i]; r_n[h] = a.r[i]; }
        }
    };
    fetch(blockIdx.x);
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        float chi[2], r[2], u[2], x1[2], x2[2];
        bool bad[2], fallback[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) { chi[h] = chi_n[h]; r[h] = r_n[h]; }
        fetch(tile + gridDim.x);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            bad[h] = !(chi[h] >= 0.0f) || !(r[h] > 0.0f) || !(r[h] < 1.0f);
            u[h] = a.K.pair ? fabsf(2.0f * r[h] - 1.0f) : r[h];   // pair creation: |r'| (exact for r in (0, 1))
            const bool in_range = chi[h] >= a.K.chi_lo && chi[h] <= a.K.chi_hi;
            const int cell = cell_of(a.K, chi[h], u[h]);
            fallback[h] = !bad[h] && (!in_range || ((fl[cell >> 5] >> (cell & 31)) & 1u));
            features(a.K, in_range ? chi[h] : 1.0f, bad[h] ? 0.5f : u[h], x1[h], x2[h]);
        }
        // layer 1 on the CUDA cores (binary32 features, bf16-rounded weights), 8 columns at a
        // time, the weights loaded once for both samples
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            f32x2 wa[4], wb[4], b[4];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                lds_pairs(w1 + 8 * c + 4 * q, wa[2 * q], wa[2 * q + 1]);
                lds_pairs(w1 + H + 8 * c + 4 * q, wb[2 * q], wb[2 * q + 1]);
                lds_pairs(b1 + 8 * c + 4 * q, b[2 * q], b[2 * q + 1]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const f32x2 x11(x1[h], x1[h]), x22(x2[h], x2[h]);
                f32x2 v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = silu_h2(fma2(wa[q], x11, fma2(wb[q], x22, b[q])));
                *reinterpret_cast<uint4 *>(sm + SM_A + h * (SM_A1 - SM_A) + row_chunk_offset(tid, c)) = pack8_bf16(v);
            }
        }
        float y[2] = {0.0f, 0.0f};
        int stop = 0;
#pragma unroll 1
        for (int layer = 0; layer < 3; ++layer) {
            // the block meets once per layer, with every operand row written; a wait that gave up
            // in an earlier layer ends the loop for all
            fence_async_smem();
            tc_fence_before();
            stop = __syncthreads_or(late);
            if (stop) break;
            if (tid == 0) {
                tc_fence_after();
                const uint32_t bw = layer == 0 ? SM_B2 : (layer == 1 ? SM_B3 : SM_B4);
                const uint32_t idesc = layer == 2 ? IDESC4 : IDESC;
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        mma_k16(taddr + 64 * h, smem_desc(sbase + SM_A + h * (SM_A1 - SM_A) + 256 * kk),
                                smem_desc(sbase + bw + 256 * kk), kk > 0, idesc);
                mma_commit(&mbar);
            }
            // each thread goes on when the group has completed; the next group needs all of them
            if (!mbar_wait_bounded(&mbar, phase)) late = 1;
            phase ^= 1;
            tc_fence_after();
            // layers 2 and 3: the SiLU rows go to A (the MMAs that read A have completed); the
            // output layer: column 0 plus b4
            if (layer < 2) {
                epilogue(t_row, layer == 0 ? hb2 : hb3, sm + SM_A, tid);
            } else {
                y[0] = tmem_ld1(t_row) + *b4;
                y[1] = tmem_ld1(t_row + 64) + *b4;
            }
            tc_fence_before();
        }
        if (stop) break;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t i = tile * IS + h * IT + tid;
            const bool valid = i < n_all;
            float xi_v = 0.0f, xc_v = 0.0f;
            if (valid) {
                float xi, xc;
                if (bad[h]) {
                    ++n_nan;
                    xi = 0.0f;
                    xc = 0.0f;
                } else if (a.K.pair) {
                    bool oor = false;
                    if (fallback[h]) {
                        pair_shares<float>(a.inv, chi[h], r[h], xi, xc, oor);
                        n_oor += oor;
                        ++n_fb;
                    } else {
                        // 1 - v-bar = exp(-u e^y): at most 1 for any network output
                        const float small = 0.5f * expf(-expf(y[h] + logf(u[h]))), big = 1.0f - small;
                        const bool pos = 2.0f * r[h] - 1.0f >= 0.0f;
                        xi = pos ? big : small;
                        xc = pos ? small : big;
                    }
                } else {
                    float s;
                    if (fallback[h]) {
                        bool oor = false;
                        s = photon_s<float>(a.inv, chi[h], u[h], oor);
                        n_oor += oor;
                        ++n_fb;
                    } else {
                        s = 1.5f * chi[h] * expf(3.0f * (y[h] + logf(u[h])));
                    }
                    xc = 1.0f / (1.0f + s);
                    xi = s < 1e30f ? s * xc : 1.0f;
                }
                a.xi[i] = xi;
                if (a.xi_c) a.xi_c[i] = xc;
                xi_v = xi;
                xc_v = xc;
            }
            if (APPLY) {
                // recoil of the emitter and the photon's record (every lane takes part in the
                // warp-wide reservation)
                const ApplyOut &o = a.ap;
                const bool emit = valid && !bad[h];
                const unsigned long long slot = warp_reserve(o.ocount, emit);
                if (emit) {
                    // xi and 1 - xi = 1/(1 + s), the latter with relative precision (hard photons)
                    const float xi = xi_v, xc = xc_v;
                    const int64_t e = o.idx[i];
                    const float g = o.g[i], px = o.px[i], py = o.py[i], pz = o.pz[i];
                    const float pm = sqrtf(fmaf(px, px, fmaf(py, py, pz * pz)));
                    const float inv_pm = pm > 0.0f ? 1.0f / pm : 0.0f;
                    const float nx = px * inv_pm, ny = py * inv_pm, nz = pz * inv_pm;
                    const float gph = g * xi, gnew = g * xc;
                    const float q2 = fmaf(gnew, gnew, -1.0f);
                    const float pnew = q2 > 0.0f ? sqrtf(q2) : 0.0f;
                    n_g1 += !(q2 > 0.0f);
                    const uint8_t fl = o.flags[e];
                    if (slot < (unsigned long long)o.cap) {
                        o.opx[slot] = nx * gph; o.opy[slot] = ny * gph; o.opz[slot] = nz * gph;
                        o.opid[slot] = o.id ? o.id[e] : o.id_base + (uint64_t)e;
                        o.ostep[slot] = o.step;
                        o.ometa[slot] = (uint8_t)(SFQ_PHOTON | (((fl >> SFQ_TAG_SHIFT) & 3u) << 4));
                    } else {
                        ++n_drop;
                    }
                    o.ppx[e] = nx * pnew; o.ppy[e] = ny * pnew; o.ppz[e] = nz * pnew;
                    // a lepton left without momentum leaves the step (as in the step kernels)
                    if (!(pnew > 0.0f)) o.flags[e] = (uint8_t)(fl & ~SFQ_ALIVE);
                    ++n_emit;
                }
            }
        }
    }
    // a group whose wait gave up: wait once more (bounded) before the tensor memory is freed
    const int failed = __syncthreads_or(late);
    if (failed && tid == 0) {
        if (!mbar_wait_bounded(&mbar, phase ^ 1) && a.status) atomicExch(a.status, 1);
    }
    if (failed && tid == 0 && a.counters) atomicAdd(&a.counters->timeouts, 1ull);
    atomicAdd(&s_cnt[0], (unsigned long long)n_nan);
    atomicAdd(&s_cnt[1], (unsigned long long)n_oor);
    atomicAdd(&s_cnt[2], (unsigned long long)n_fb);
    if (APPLY) {
        atomicAdd(&s_cnt[3], (unsigned long long)n_emit);
        atomicAdd(&s_cnt[4], (unsigned long long)n_drop);
        atomicAdd(&s_cnt[5], (unsigned long long)n_g1);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(TMEM_COLS) : "memory");
    }
    if (tid == 0 && a.counters) {
        if (s_cnt[0]) atomicAdd(&a.counters->nan_input, s_cnt[0]);
        if (s_cnt[1]) atomicAdd(&a.counters->out_of_range, s_cnt[1]);
        if (s_cnt[2]) atomicAdd(&a.counters->surrogate_fallbacks, s_cnt[2]);
        if (APPLY) {
            if (s_cnt[3]) atomicAdd(&a.counters->emitted, s_cnt[3]);
            if (s_cnt[4]) atomicAdd(&a.counters->dropped, s_cnt[4]);
            if (s_cnt[5]) atomicAdd(&a.counters->gamma_below_one, s_cnt[5]);
        }
    }
    if (failed && tid == 0 && a.status) atomicExch(a.status, 1);
}

}  // namespace mlp

// The surrogate pass of a step: sample the queued emissions and finish them (recoil and
// records), one persistent grid over the queue's capacity (the count is read on the device).
cudaError_t launch_surrogate_apply(const sfq_ctx *ctx, const sfq_particles *p, uint32_t step, const sfq_products *out,
                                   sfq_counters *counters, cudaStream_t stream) {
    using namespace mlp;
    const sfq_mlp *m = ctx->surr;
    const sfq_event_queue &q = ctx->surr_q;
    if (q.capacity <= 0) return cudaSuccess;
    const int64_t ntiles = (q.capacity + IS - 1) / IS;
    int64_t grid = (int64_t)ctx->surr_per_sm * ctx->num_sms;
    if (ntiles < grid) grid = ntiles;
    InferArgs a{};
    a.params = m->params;
    a.flags = ctx->surr_flags ? m->flags : nullptr;
    a.inv = static_cast<const float *>(ctx->d_nlc_inv);
    a.n = q.capacity;
    a.chi = q.chi;
    a.r = q.r;
    a.xi = q.xi;
    a.xi_c = nullptr;
    a.counters = counters;
    a.status = nullptr;
    a.K = kind_of(0);
    a.n_dev = q.count;
    ApplyOut &o = a.ap;
    o.idx = q.index;
    o.g = q.gamma; o.px = q.px; o.py = q.py; o.pz = q.pz;
    o.ppx = static_cast<float *>(p->px); o.ppy = static_cast<float *>(p->py); o.ppz = static_cast<float *>(p->pz);
    o.flags = p->flags;
    o.id = p->id;
    o.id_base = p->id_base;
    o.cap = out->capacity;
    o.opx = static_cast<float *>(out->px); o.opy = static_cast<float *>(out->py); o.opz = static_cast<float *>(out->pz);
    o.opid = out->parent_id;
    o.ostep = out->step;
    o.ometa = out->meta;
    o.ocount = out->count;
    o.step = step;
    infer_tc_kernel<true><<<(unsigned)grid, IT, INFER_SMEM, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace sfq

// ---------------------------------------------------------------------------------------
// C ABI
namespace {

using namespace sfq::mlp;

sfq_status fail(sfq_ctx *ctx, sfq_status st, const char *msg) {
    if (ctx) ctx->err = msg;
    return st;
}
sfq_status cuda_fail(sfq_ctx *ctx, cudaError_t e, const char *where) {
    if (ctx) ctx->err = std::string(where) + ": " + cudaGetErrorString(e);
    return SFQ_ERR_CUDA;
}
struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        cudaGetDevice(&prev);
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DeviceGuard() {
        int cur = -1;
        cudaGetDevice(&cur);
        if (prev >= 0 && cur != prev) cudaSetDevice(prev);
    }
};
bool a16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

// Attributes of an inference kernel instance: its dynamic shared memory, and the largest
// shared-memory carveout, so that INFER_MINB blocks (4 x 53 KB) are resident on an SM.  The
// grid is then INFER_MINB blocks per SM: registers (at most 128 a thread by the launch
// bounds), shared memory and tensor memory (4 x 128 of the 512 columns) all admit them.
template <typename K>
cudaError_t set_infer_attributes(K kern) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)INFER_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    return e;
}

// The plain fitted sampler the surrogate stands for (training targets, calibration, fallback).
const float *inv_table(const sfq_mlp *m) {
    return static_cast<const float *>(m->kind ? m->ctx->d_nbw_inv : m->ctx->d_nlc_inv);
}

}  // namespace

extern "C" {

static sfq_status mlp_create(sfq_ctx *ctx, uint64_t seed, int kind, sfq_mlp **out) {
    if (!ctx || !out) return SFQ_ERR_ARG;
    *out = nullptr;
    if (ctx->cfg.precision != SFQ_FP32) return fail(ctx, SFQ_ERR_ARG, "the surrogate serves binary32 contexts");
    DeviceGuard g(ctx->device);
    sfq_mlp *m = new sfq_mlp();
    m->ctx = ctx;
    m->kind = kind;
    float **bufs[3] = {&m->params, &m->m, &m->v};
    cudaError_t e = cudaSuccess;
    for (auto b : bufs)
        if (e == cudaSuccess) e = cudaMalloc(b, NP * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&m->flags, NCELL);
    if (e == cudaSuccess) e = cudaMalloc(&m->cell_err, NCELL * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(m->m, 0, NP * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(m->v, 0, NP * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(m->flags, 0, NCELL);
    if (e == cudaSuccess) {
        init_kernel<<<(NP + 255) / 256, 256>>>(m->params, seed);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        sfq_mlp_destroy(m);
        return cuda_fail(ctx, e, "sfq_mlp_create");
    }
    *out = m;
    return SFQ_OK;
}

sfq_status sfq_mlp_create(sfq_ctx *ctx, uint64_t seed, sfq_mlp **out) { return mlp_create(ctx, seed, 0, out); }
sfq_status sfq_mlp_create_pair(sfq_ctx *ctx, uint64_t seed, sfq_mlp **out) { return mlp_create(ctx, seed, 1, out); }

void sfq_mlp_destroy(sfq_mlp *m) {
    if (!m) return;
    if (m->ctx->surr == m) m->ctx->surr = nullptr;     // detach from the context's step
    DeviceGuard g(m->ctx->device);
    void *p[5] = {m->params, m->m, m->v, m->flags, m->cell_err};
    for (void *q : p)
        if (q) cudaFree(q);
    delete m;
}

int32_t sfq_mlp_num_params(void) { return NP; }

sfq_status sfq_mlp_get_params(sfq_mlp *m, float *host) {
    if (!m || !host) return SFQ_ERR_ARG;
    DeviceGuard g(m->ctx->device);
    const cudaError_t e = cudaMemcpy(host, m->params, NP * sizeof(float), cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? SFQ_OK : cuda_fail(m->ctx, e, "sfq_mlp_get_params");
}

sfq_status sfq_mlp_set_params(sfq_mlp *m, const float *host) {
    if (!m || !host) return SFQ_ERR_ARG;
    DeviceGuard g(m->ctx->device);
    cudaError_t e = cudaMemcpy(m->params, host, NP * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(m->m, 0, NP * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(m->v, 0, NP * sizeof(float));
    m->adam_t = 0;
    m->calibrated = 0;
    return e == cudaSuccess ? SFQ_OK : cuda_fail(m->ctx, e, "sfq_mlp_set_params");
}

static sfq_status check_data(sfq_mlp *m, int64_t n, const float *chi, const float *u, const float *lnw) {
    if (n <= 0) return fail(m->ctx, SFQ_ERR_ARG, "n must be positive");
    if (n > 0xFFFFFFFFll) return fail(m->ctx, SFQ_ERR_ARG, "n above 2^32");
    if (!chi || !u || !lnw) return fail(m->ctx, SFQ_ERR_ARG, "null data buffer");
    return SFQ_OK;
}

static cudaError_t set_train_smem() {
    static bool done = false;
    if (done) return cudaSuccess;
    const cudaError_t e =
        cudaFuncSetAttribute(train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
    if (e == cudaSuccess) done = true;
    return e;
}

sfq_status sfq_mlp_loss_grad(sfq_mlp *m, int64_t n, const float *chi, const float *u, const float *lnw,
                             int32_t quantize, float *grad, float *loss, void *stream) {
    if (!m) return SFQ_ERR_ARG;
    sfq_status st = check_data(m, n, chi, u, lnw);
    if (st != SFQ_OK) return st;
    if (!grad) return fail(m->ctx, SFQ_ERR_ARG, "null gradient buffer");
    DeviceGuard g(m->ctx->device);
    const cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = set_train_smem();
    const int nb = (int)((n + TS - 1) / TS);
    float *part = nullptr;
    if (e == cudaSuccess) e = cudaMallocAsync(&part, ((size_t)nb * NPS + nb) * sizeof(float), s);
    if (e != cudaSuccess) return cuda_fail(m->ctx, e, "sfq_mlp_loss_grad");
    TrainArgs a{m->params, n, chi, u, lnw, 0, 0, 0, 0, quantize, 2.0f / (float)n, part, part + (size_t)nb * NPS,
                kind_of(m->kind)};
    train_kernel<<<nb, TB, sizeof(TrainSmem), s>>>(a);
    reduce_kernel<false><<<RBLOCKS, RB, 0, s>>>(part, part + (size_t)nb * NPS, nb, grad, loss, 1.0f / (float)n, nullptr,
                                                nullptr, nullptr, 0.0f, 0.0f, 0.0f);
    e = cudaGetLastError();
    cudaFreeAsync(part, s);
    return e == cudaSuccess ? SFQ_OK : cuda_fail(m->ctx, e, "sfq_mlp_loss_grad");
}

sfq_status sfq_mlp_train(sfq_mlp *m, int64_t n, const float *chi, const float *u, const float *lnw, int64_t steps,
                         int32_t batch, float lr, int32_t quantize, uint64_t seed, float *loss_history, void *stream) {
    if (!m) return SFQ_ERR_ARG;
    sfq_status st = check_data(m, n, chi, u, lnw);
    if (st != SFQ_OK) return st;
    if (steps <= 0 || batch < TS || batch % TS != 0) return fail(m->ctx, SFQ_ERR_ARG, "steps > 0 and batch a multiple of 64");
    if (!(lr > 0.0f)) return fail(m->ctx, SFQ_ERR_ARG, "lr must be positive");
    DeviceGuard g(m->ctx->device);
    const cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = set_train_smem();
    const int nb = batch / TS;
    float *part = nullptr;
    if (e == cudaSuccess) e = cudaMallocAsync(&part, ((size_t)nb * NPS + nb) * sizeof(float), s);
    if (e != cudaSuccess) return cuda_fail(m->ctx, e, "sfq_mlp_train");
    for (int64_t t = 0; t < steps && e == cudaSuccess; ++t) {
        TrainArgs a{m->params, n, chi, u, lnw, 0, 1, seed, (uint32_t)(m->adam_t + 1), quantize,
                    2.0f / (float)batch, part, part + (size_t)nb * NPS, kind_of(m->kind)};
        train_kernel<<<nb, TB, sizeof(TrainSmem), s>>>(a);
        m->adam_t += 1;
        // cosine schedule from lr to 0
        const float lrt = 0.5f * lr * (1.0f + cosf(3.14159265f * (float)t / (float)steps));
        const float b1t = powf(0.9f, (float)m->adam_t), b2t = powf(0.999f, (float)m->adam_t);
        reduce_kernel<true><<<RBLOCKS, RB, 0, s>>>(part, part + (size_t)nb * NPS, nb, nullptr,
                                                   loss_history ? loss_history + t : nullptr, 1.0f / (float)batch,
                                                   m->params, m->m, m->v, lrt, b1t, b2t);
        e = cudaGetLastError();
    }
    cudaFreeAsync(part, s);
    m->calibrated = 0;
    return e == cudaSuccess ? SFQ_OK : cuda_fail(m->ctx, e, "sfq_mlp_train");
}

sfq_status sfq_mlp_predict_lnw(sfq_mlp *m, int64_t n, const float *chi, const float *u, float *lnw, void *stream) {
    if (!m) return SFQ_ERR_ARG;
    if (n < 0) return fail(m->ctx, SFQ_ERR_ARG, "n < 0");
    if (n == 0) return SFQ_OK;
    if (!chi || !u || !lnw) return fail(m->ctx, SFQ_ERR_ARG, "null buffer");
    DeviceGuard g(m->ctx->device);
    const int64_t blocks = (n + 127) / 128;
    const int grid = (int)(blocks < (int64_t)m->ctx->num_sms * 8 ? blocks : (int64_t)m->ctx->num_sms * 8);
    const cudaError_t e = launch_predict(m->params, kind_of(m->kind), n, chi, u, lnw, grid, (cudaStream_t)stream);
    return e == cudaSuccess ? SFQ_OK : cuda_fail(m->ctx, e, "sfq_mlp_predict_lnw");
}

sfq_status sfq_mlp_plain_targets(sfq_mlp *m, int64_t n, const float *chi, const float *u, float *lnw, void *stream) {
    if (!m) return SFQ_ERR_ARG;
    if (n < 0) return fail(m->ctx, SFQ_ERR_ARG, "n < 0");
    if (n == 0) return SFQ_OK;
    if (!chi || !u || !lnw) return fail(m->ctx, SFQ_ERR_ARG, "null buffer");
    DeviceGuard g(m->ctx->device);
    const int64_t blocks = (n + 255) / 256;
    const int grid = (int)(blocks < (int64_t)m->ctx->num_sms * 8 ? blocks : (int64_t)m->ctx->num_sms * 8);
    const cudaError_t e =
        launch_plain_targets(inv_table(m), kind_of(m->kind), n, chi, u, lnw, grid, (cudaStream_t)stream);
    return e == cudaSuccess ? SFQ_OK : cuda_fail(m->ctx, e, "sfq_mlp_plain_targets");
}

sfq_status sfq_mlp_calibrate(sfq_mlp *m, float tol_u, int32_t *n_flagged, float *max_err, void *stream) {
    if (!m) return SFQ_ERR_ARG;
    if (!(tol_u > 0.0f)) return fail(m->ctx, SFQ_ERR_ARG, "tol_u must be positive");
    DeviceGuard g(m->ctx->device);
    const cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = launch_calibrate(m->params, kind_of(m->kind), inv_table(m), tol_u, m->flags, m->cell_err, s);
    std::vector<uint8_t> f(NCELL);
    std::vector<float> ce(NCELL);
    if (e == cudaSuccess) e = cudaMemcpyAsync(f.data(), m->flags, NCELL, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(ce.data(), m->cell_err, NCELL * sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(m->ctx, e, "sfq_mlp_calibrate");
    int32_t nf = 0;
    float mx = 0.0f;
    for (int c = 0; c < NCELL; ++c) {
        nf += f[c];
        if (!f[c] && ce[c] > mx) mx = ce[c];
    }
    if (n_flagged) *n_flagged = nf;
    if (max_err) *max_err = mx;
    m->calibrated = 1;
    return SFQ_OK;
}

static sfq_status mlp_sample(sfq_mlp *m, int64_t n, const void *chi, const void *r, void *xi, void *xi_c,
                             int32_t use_flags, sfq_counters *counters, void *stream) {
    if (!m) return SFQ_ERR_ARG;
    if (n < 0) return fail(m->ctx, SFQ_ERR_ARG, "n < 0");
    if (n == 0) return SFQ_OK;
    if (!chi || !r || !xi) return fail(m->ctx, SFQ_ERR_ARG, "null buffer");
    if (!a16(chi) || !a16(r) || !a16(xi) || (xi_c && !a16(xi_c)) || (counters && ((uintptr_t)counters & 7u)))
        return fail(m->ctx, SFQ_ERR_ARG, "misaligned buffer (16 bytes required)");
    if (use_flags && !m->calibrated) return fail(m->ctx, SFQ_ERR_ARG, "use_flags before sfq_mlp_calibrate");
    DeviceGuard g(m->ctx->device);
    static bool attr = false;
    cudaError_t e = cudaSuccess;
    if (!attr) {
        e = set_infer_attributes(infer_tc_kernel<false>);
        if (e != cudaSuccess) return cuda_fail(m->ctx, e, "sfq_mlp_sample_photon_xi: attributes");
        attr = true;
    }
    const int per_sm = INFER_MINB;
    const int64_t ntiles = (n + IS - 1) / IS;
    int64_t grid = (int64_t)per_sm * m->ctx->num_sms;
    if (ntiles < grid) grid = ntiles;
    InferArgs a{m->params, use_flags ? m->flags : nullptr, inv_table(m), n,
                static_cast<const float *>(chi), static_cast<const float *>(r), static_cast<float *>(xi),
                static_cast<float *>(xi_c), counters, nullptr, kind_of(m->kind), nullptr, ApplyOut{}};
    infer_tc_kernel<false><<<(unsigned)grid, IT, INFER_SMEM, (cudaStream_t)stream>>>(a);
    e = cudaGetLastError();
    return e == cudaSuccess ? SFQ_OK : cuda_fail(m->ctx, e, "sfq_mlp_sample_*_xi");
}

sfq_status sfq_mlp_sample_photon_xi(sfq_mlp *m, int64_t n, const void *chi, const void *r, void *xi, void *xi_c,
                                    int32_t use_flags, sfq_counters *counters, void *stream) {
    if (m && m->kind != 0) return fail(m->ctx, SFQ_ERR_ARG, "a pair-creation surrogate: use sfq_mlp_sample_pair_xi");
    return mlp_sample(m, n, chi, r, xi, xi_c, use_flags, counters, stream);
}

sfq_status sfq_mlp_sample_pair_xi(sfq_mlp *m, int64_t n, const void *chi, const void *r, void *xi_e, void *xi_p,
                                  int32_t use_flags, sfq_counters *counters, void *stream) {
    if (m && m->kind != 1) return fail(m->ctx, SFQ_ERR_ARG, "a photon-emission surrogate: use sfq_mlp_sample_photon_xi");
    return mlp_sample(m, n, chi, r, xi_e, xi_p, use_flags, counters, stream);
}

sfq_status sfq_set_surrogate(sfq_ctx *ctx, sfq_mlp *net, const sfq_event_queue *queue, int32_t use_flags) {
    if (!ctx) return SFQ_ERR_ARG;
    if (!net) {
        ctx->surr = nullptr;
        ctx->surr_q = sfq_event_queue{};
        ctx->surr_flags = 0;
        return SFQ_OK;
    }
    if (ctx->cfg.precision != SFQ_FP32) return fail(ctx, SFQ_ERR_ARG, "the surrogate needs a binary32 context");
    if (net->ctx != ctx) return fail(ctx, SFQ_ERR_ARG, "a surrogate of another context");
    if (net->kind != 0) return fail(ctx, SFQ_ERR_ARG, "a pair-creation surrogate: the step takes the photon one");
    if (use_flags && !net->calibrated) return fail(ctx, SFQ_ERR_ARG, "use_flags before sfq_mlp_calibrate");
    if (ctx->inv_tr > 0) return fail(ctx, SFQ_ERR_ARG, "truncated samplers are set: restore the full coefficients");
    if (!queue || queue->capacity < 0 || !queue->count || ((uintptr_t)queue->count & 7u))
        return fail(ctx, SFQ_ERR_ARG, "queue descriptor, capacity or counter invalid");
    if (queue->capacity > 0) {
        const void *b[8] = {queue->index, queue->chi, queue->r, queue->gamma, queue->px, queue->py, queue->pz, queue->xi};
        for (const void *q : b)
            if (!q || !a16(q)) return fail(ctx, SFQ_ERR_ARG, "queue buffer null or misaligned (16 bytes)");
    }
    DeviceGuard g(ctx->device);
    // kernel attributes and the grid of the surrogate pass, set here (outside any capture)
    cudaError_t e = sfq::prepare_step_surr_f32();
    if (e == cudaSuccess) e = set_infer_attributes(infer_tc_kernel<true>);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "sfq_set_surrogate: attributes");
    const int per_sm = INFER_MINB;
    ctx->surr = net;
    ctx->surr_q = *queue;
    ctx->surr_flags = use_flags ? 1 : 0;
    ctx->surr_per_sm = per_sm;
    return SFQ_OK;
}

}  // extern "C"
