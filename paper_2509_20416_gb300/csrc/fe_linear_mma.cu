// Linear phases of the cascade on the tensor cores (tcgen05 + TMEM), for batches of
// sequences: Y[b, m] = epilogue(sum_k W[m, k] X[b, k]) for b < B (Eq. 1 FCs; QKV, O-proj,
// gate/up and down projections of every layer L_i, Eq. 2).
//
// At batch 1 a linear phase is a matrix-vector product and the CUDA-core streaming kernel
// (fe_linear.cu) is the right tool. With many sequences it re-reads the weights once per
// batch tile; here every weight is read once for the whole batch and the products run on
// the tensor cores:
//   - xprep_kernel applies the phase's prologue (RMSNorm, concat with the token embedding,
//     storage or float32 input) and writes the activations as a bf16 B operand split into
//     hi and lo parts (x = hi + lo to ~16 significant bits, so the products keep float32
//     accuracy): rows [0, B_pad) hold hi, [B_pad, 2 B_pad) hold lo, in the 128-byte-
//     swizzled K-major layout of fe_tc.cuh, one 2 B_pad x 64 block per 64 columns.
//   - linear_mma_kernel: the weights are packed at init in 128 x 64 swizzled blocks
//     (fe_pack.cu), so one TMA bulk copy lands one A operand. The (tile of 128 output rows,
//     64-column block) units are split evenly over the CTAs in tile-major order (stream-K),
//     so every SM streams the same number of bytes whatever the matrix shape. Warp 4 issues
//     the copies (weights block + activation block per stage, a ring of S stages), warp 5
//     issues tcgen05.mma (M = 128, N = 2 B_pad, K = 16; float32 accumulators in TMEM, two
//     buffers), warps 0-3 read TMEM (thread = output row) and add hi + lo.
//   - Two forms (LinearArgs::splits). Handles of 9..32 sequences: their own weight layout (one
//     contiguous 16 KB copy per unit), two splits, one accumulation chain per tile (commit blocks
//     of up to 128 rows: linear_mma_mt). Handles of up to 8 and of 33..64 sequences (drafts of 2 to
//     16 hidden rows and commits, where linear_tc_us is below linear_stream_us): the streaming
//     kernel's tile layout, which a tensor map reads as the same operand, so that a
//     handle needs one copy of its weights for both kernels; THREE splits (hi + mid + lo are
//     all 24 bits of a float32, so the products are exact as on the CUDA cores), and every
//     unit's accumulators are drained and summed in registers with compensation: the tensor
//     core truncates its running sum at each step, which shrinks a result by ~1e-8 per step
//     of its chain. Hidden states of a 2-layer 8B-shaped cascade against 64 bits: CUDA cores
//     3.4e-7, whole-tile chains 8e-6, chains of 4 units 6.9e-7, of 1 unit 2.6e-7.
//   - A tile whose units all fall in one CTA is finished there. A tile split between CTAs
//     leaves one float32 partial per CTA in global scratch; the last CTA to finish its
//     share of the tile (an atomic counter) sums the partials in CTA order (so results do
//     not depend on timing) and applies the epilogue: store, residual add (+ copy into the
//     hidden-state buffer), or SwiGLU over the interleaved gate/up rows (the partner row
//     sits in the neighbouring lane).
#include "fe_kernels.h"
#include "fe_stream.cuh"
#include "fe_tc.cuh"
#include "fe_splitk.cuh"

namespace fe {

namespace {

// 4 epilogue warps, 1 producer warp, and 1 MMA warp, or 2 with three splits
__host__ __device__ constexpr int lin_threads(int ns) { return ns == 3 ? 224 : 192; }
constexpr size_t kXprepRowSmem = 16384 * sizeof(float);  // a finished row of up to 16384 columns
constexpr int kLinMaxStages = 8;
constexpr int kLinMaxAccs = 8;

// accumulators (TMEM buffers of N columns): a chain of one unit needs several in flight to hide
// the round trip MMA -> epilogue -> MMA; whole-tile chains alternate between two
__host__ __device__ constexpr int acc_buffers(int N, int ns, int mt) {
    return ns == 3 ? (512 / N < kLinMaxAccs ? 512 / N : kLinMaxAccs) : mt == 2 ? 1 : 2;
}

// operand rows (MMA columns): the splits' blocks of B_pad rows, to a multiple of 16
__host__ __device__ constexpr int operand_rows(int bpad, int ns) { return (ns * bpad + 15) / 16 * 16; }

struct LinMmaState {
    uint64_t full[kLinMaxStages], empty[kLinMaxStages], tfull[kLinMaxAccs], tempty[kLinMaxAccs];
    uint64_t drain[2];  // the MMA issuers', should a wait give up
    uint32_t tmem_base;
    int abort, issued;  // issued: copies the producer asked for
};

}  // namespace

// ---- activation operand ------------------------------------------------------------------
// Grid (B_pad, ceil(K / 2048)): CTA (b, y) writes row b's 16-byte chunks [256 y, 256 y + 256)
// (rows b >= B are zero); with RMSNorm every CTA of the row reads the whole row for its sum
// of squares (an L2 read of 4 d bytes). Reads what the previous kernel wrote only after
// griddep_wait(), through L2, and never through a __restrict__ pointer.
// When the previous tensor-core phase deferred its split tiles (a.prev.active), the input
// columns of those tiles are finished here first (prev_finish); with RMSNorm, one CTA per
// row (grid (B_pad, 1)) finishes the whole row into shared memory before normalising it.
constexpr int kXprepChunks = 256;  // 16-byte chunks per CTA (one per thread)

// sum of squares of 8 values, in one fixed order
__device__ __forceinline__ float sumsq8(const float (&v)[8]) {
    float s = v[0] * v[0];
#pragma unroll
    for (int e = 1; e < 8; ++e) s = fmaf(v[e], v[e], s);
    return s;
}

// Takes x's largest bf16 part out of it.
__device__ __forceinline__ uint32_t take_bf16(float& x) {
    const uint32_t h = f32_to_bf16(x);
    x -= bf16_to_f32((uint16_t)h);
    return h;
}

// The same for any x: a finite one keeps a finite part, also where it would round to infinity; an
// infinity or a NaN stays one and leaves 0.
__device__ __forceinline__ uint32_t take_bf16_any(float& x) {
    if (!(fabsf(x) < INFINITY)) {
        const uint32_t h = x == x ? __float_as_uint(x) >> 16 : 0x7fffu;
        x = 0.f;
        return h;
    }
    uint32_t h = f32_to_bf16(x);
    if ((h & 0x7fffu) == 0x7f80u) --h;
    x -= bf16_to_f32((uint16_t)h);
    return h;
}

// the bf16 operand chunk c of row b from 8 values: x = hi + lo (two splits) or hi + mid + lo,
// split q in row q * B_pad + b. Three splits stand in for a float32 product, which keeps
// infinities and NaN apart from finite values: a chunk that holds one, or a value that rounds to
// infinity (2^127 (2 - 2^-8) and above), is split by take_bf16_any.
template <int NS>
__device__ __forceinline__ void put_operand(uint16_t* xb, int N, int B_pad, int b, int c, const float (&v)[8]) {
    uint32_t w[NS][4];
    float x[8];
    uint32_t h[8], big = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        x[e] = v[e];
        big = max(big, __float_as_uint(v[e]) & 0x7fffffffu);
    }
    if (NS == 3 && big >= 0x7f7f8000u) {
#pragma unroll
        for (int e = 0; e < 8; ++e) h[e] = take_bf16_any(x[e]);
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) h[e] = take_bf16(x[e]);
    }
#pragma unroll
    for (int q = 0; q < NS; ++q) {
        if (q > 0) {
#pragma unroll
            for (int e = 0; e < 8; ++e) h[e] = take_bf16(x[e]);
        }
#pragma unroll
        for (int e = 0; e < 8; e += 2) w[q][e / 2] = h[e] | h[e + 1] << 16;
    }
    unsigned char* blk = (unsigned char*)xb + (size_t)(c / 8) * N * 128;
#pragma unroll
    for (int q = 0; q < NS; ++q)
        *reinterpret_cast<uint4*>(blk + sw128_offset(q * B_pad + b, c % 8)) = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
}

// Attention output columns k0 .. k0 + 7 of row b from its splits' partials (fe_attn.cu: value
// sum [128], base-2 max, sum of weights): sum_q w_q acc_q / sum_q w_q l_q, w_q = 2^(m_q - max).
// The 16 threads of a head form the same weights; loads go out in batches.
__device__ __forceinline__ void combine_parts(const LinearArgs& a, int b, int k0, float (&v)[8]) {
    constexpr int RS = 132, U = 4;
    const int n = a.attn_nact[b];
    const float* p = (const float*)a.x + ((size_t)b * (a.K / 128) + k0 / 128) * a.attn_splits * RS;
    float M = -INFINITY;
    for (int q0 = 0; q0 < n; q0 += 2 * U) {
        float m[2 * U];
#pragma unroll
        for (int j = 0; j < 2 * U; ++j) m[j] = q0 + j < n ? __ldcg(p + (size_t)(q0 + j) * RS + 128) : -INFINITY;
#pragma unroll
        for (int j = 0; j < 2 * U; ++j) M = fmaxf(M, m[j]);
    }
    float L = 0.f;
    for (int q0 = 0; q0 < n; q0 += U) {
        float4 x[U], y[U];
        float2 ml[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const float* r = p + (size_t)min(q0 + j, n - 1) * RS;
            x[j] = __ldcg(reinterpret_cast<const float4*>(r + k0 % 128));
            y[j] = __ldcg(reinterpret_cast<const float4*>(r + k0 % 128) + 1);
            ml[j] = __ldcg(reinterpret_cast<const float2*>(r + 128));
        }
#pragma unroll
        for (int j = 0; j < U; ++j) {
            if (q0 + j >= n || ml[j].x == -INFINITY) continue;
            const float f = exp2f(ml[j].x - M);
            L = fmaf(f, ml[j].y, L);
            v[0] = fmaf(f, x[j].x, v[0]); v[1] = fmaf(f, x[j].y, v[1]);
            v[2] = fmaf(f, x[j].z, v[2]); v[3] = fmaf(f, x[j].w, v[3]);
            v[4] = fmaf(f, y[j].x, v[4]); v[5] = fmaf(f, y[j].y, v[5]);
            v[6] = fmaf(f, y[j].z, v[6]); v[7] = fmaf(f, y[j].w, v[7]);
        }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = L > 0.f ? v[e] / L : 0.f;
}

template <int NS>
__global__ void __launch_bounds__(256) xprep_kernel(const LinearArgs a, int B_pad, uint16_t* xb, float* sq) {
    const LaunchStamp stamp(a.stamp);
    const int b = blockIdx.x, t = threadIdx.x;
    const int N = operand_rows(B_pad, NS), K = a.K, nc = K / 8;
    const int c = blockIdx.y * kXprepChunks + t;  // this thread's 16-byte chunk of row b
    const int k0 = 8 * c;
    __shared__ float red[8];
    griddep_launch_dependents();
    // weights do not depend on the previous kernel: the RMSNorm gains are loaded, and the
    // embedding row's line is prefetched into L2 (from a token id read early: a stale id
    // only warms a wrong line), before the wait
    uint4 gq = make_uint4(0, 0, 0, 0);
    if (b < a.B && c < nc) {
        if (a.pro == PRO_RMSNORM) gq = *reinterpret_cast<const uint4*>((const bf16_t*)a.gamma + k0);
        if (a.pro == PRO_CONCAT_EMB && k0 >= a.d_split) {
            const int tk = a.tok[b];
            if (tk >= 0 && tk < a.vocab)
                asm volatile("prefetch.global.L2 [%0];" ::"l"((const bf16_t*)a.embed + (size_t)tk * (K - a.d_split) +
                                                               (k0 - a.d_split)));
        }
    }
    griddep_wait();
    const int nlive = a.total ? min(a.B, *a.total - a.row0) : a.B;  // (<= 0: a block without rows)
    if (nlive <= 0) return;
    const bool live = b < nlive;
    const bool fin = live && a.prev.active;  // (without norm_post, RMSNorm inputs take xprep_row_kernel)
    const bool post = a.norm_post && a.pro == PRO_RMSNORM;  // the scale goes on the products
    int tok = 0;
    if (live && a.pro == PRO_CONCAT_EMB) {
        tok = a.tok[b];
        if (tok < 0 || tok >= a.vocab) {
            if (t == 0) atomicOr(a.status, ST_DEVICE);
            tok = -1;
        }
    }
    const float* xf = (const float*)a.x + (size_t)b * a.ldx;
    // the CTA's sum of per-thread partials in a fixed order
    auto cta_sum = [&](float ss) {
        ss = warp_sum(ss);
        if ((t & 31) == 0) red[t >> 5] = ss;
        __syncthreads();
        float tot = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) tot += red[w];
        return tot;
    };
    float rs = 1.f;
    if (live && a.pro == PRO_RMSNORM && !post) {  // 1 / sqrt(mean of squares + eps) over the whole row
        float ss = 0.f;
#pragma unroll 4
        for (int cc = t; cc < nc; cc += 256) {
            const float4 p = __ldcg(reinterpret_cast<const float4*>(xf) + 2 * cc);
            const float4 q = __ldcg(reinterpret_cast<const float4*>(xf) + 2 * cc + 1);
            const float v[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
            ss += sumsq8(v);
        }
        rs = 1.0f / sqrtf(cta_sum(ss) / (float)K + a.eps);
    }
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = 0.f;
    if (live && c < nc) {
        if (a.pro == PRO_STORAGE) {
            const bf16_t* xs = (const bf16_t*)a.x + (size_t)(a.x_row ? a.x_row[b] : b) * a.ldx + k0;
            if ((reinterpret_cast<uintptr_t>(xs) & 15) == 0) {
                Vec16<bf16_t>::widen(*reinterpret_cast<const uint4*>(xs), v);
            } else {  // (the caller's features; rows are whole 16-byte vectors apart)
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = Storage<bf16_t>::load(xs, e);
            }
        } else if (a.pro == PRO_CONCAT_EMB && k0 >= a.d_split) {
            if (tok >= 0)
                Vec16<bf16_t>::widen(*reinterpret_cast<const uint4*>((const bf16_t*)a.embed +
                                                                     (size_t)tok * (K - a.d_split) + (k0 - a.d_split)),
                                     v);
        } else if (a.pro == PRO_ATTN_PARTS) {
            combine_parts(a, b, k0, v);
        } else if (fin) {  // the previous phase's output, its split tiles finished here
            prev_finish(a.prev, B_pad, b, k0, v);
        } else {  // float32 input (PRO_F32, PRO_RMSNORM, or the float part of PRO_CONCAT_EMB)
            const float4 p = __ldcg(reinterpret_cast<const float4*>(xf + k0));
            const float4 q = __ldcg(reinterpret_cast<const float4*>(xf + k0) + 1);
            v[0] = p.x; v[1] = p.y; v[2] = p.z; v[3] = p.w; v[4] = q.x; v[5] = q.y; v[6] = q.z; v[7] = q.w;
        }
    }
    if (a.pro == PRO_RMSNORM) {
        float g[8];
        Vec16<bf16_t>::widen(gq, g);
        if (post) {  // gamma * x here; this CTA's sum of squares of x for the product kernel
            const float tot = cta_sum(sumsq8(v));
            if (t == 0) sq[blockIdx.y * B_pad + b] = tot;
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] *= g[e];
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = v[e] * rs * g[e];
        }
    }
    if (c < nc) put_operand<NS>(xb, N, B_pad, b, c, v);
}

// The split tiles of a phase that deferred them, for a reader that is no tensor-core phase and
// reads them many times (a commit's attention): grid (rows, ceil(columns / 2048)), a thread per 8
// columns. The phase's own fix-up (a CTA per tile sums all its rows at the phase's end) made the
// 8B shape's 128-row QKV projection 27 us; deferred it is 18, and this kernel 7.
__global__ void __launch_bounds__(256) finish_kernel(const LinearArgs::Prev p, int BP, int cols, const int* total, int row0) {
    griddep_launch_dependents();
    griddep_wait();
    const int b = blockIdx.x, k0 = 8 * (blockIdx.y * 256 + threadIdx.x);
    if (b >= *total - row0 || k0 >= cols) return;
    float v[8];
    prev_finish_t<false>(p, BP, b, k0, v);
}

// The deferred-input prep of an RMSNorm phase: one CTA of kRowThreads per row b finishes the
// previous phase's output over the whole row into shared memory (its split tiles, as
// prev_finish), sums its squares and writes the normalised row's operand. Thread t owns
// chunks t, t + kRowThreads, ... (the same per-thread order of the sum as xprep_kernel).
constexpr int kRowThreads = 512;

__global__ void __launch_bounds__(kRowThreads) xprep_row_kernel(const LinearArgs a, int B_pad, uint16_t* xb) {
    const LaunchStamp stamp(a.stamp);
    extern __shared__ __align__(16) float xrow[];  // the finished row [K]
    const int b = blockIdx.x, t = threadIdx.x;
    const int N = 2 * B_pad, K = a.K, nc = K / 8;
    __shared__ float red[kRowThreads / 32];
    griddep_launch_dependents();
    // the RMSNorm gains of this thread's first kPreChunks chunks (weights: loaded before the
    // wait; d <= 8192 needs no more)
    constexpr int kRowChunks = kXprepRowSmem / sizeof(float) / 8 / kRowThreads;
    constexpr int kPreChunks = 2;
    uint4 gq[kPreChunks];
#pragma unroll
    for (int j = 0; j < kPreChunks; ++j) {
        const int c = t + j * kRowThreads;
        gq[j] = b < a.B && c < nc ? *reinterpret_cast<const uint4*>((const bf16_t*)a.gamma + 8 * c) : make_uint4(0, 0, 0, 0);
    }
    griddep_wait();
    if (b >= a.B) {  // a padding row of the operand is zero
        const float z[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int c = t; c < nc; c += kRowThreads) put_operand<2>(xb, N, B_pad, b, c, z);
        return;
    }
    float ss = 0.f;
    for (int c = t; c < nc; c += kRowThreads) {
        float v[8];
        prev_finish_t<false>(a.prev, B_pad, b, 8 * c, v);  // (an RMSNorm input is never SwiGLU's output)
        ss += sumsq8(v);
        reinterpret_cast<float4*>(xrow)[2 * c] = make_float4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<float4*>(xrow)[2 * c + 1] = make_float4(v[4], v[5], v[6], v[7]);
    }
    ss = warp_sum(ss);
    if ((t & 31) == 0) red[t >> 5] = ss;
    __syncthreads();  // (also publishes xrow)
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < kRowThreads / 32; ++w) tot += red[w];
    const float rs = 1.0f / sqrtf(tot / (float)K + a.eps);
#pragma unroll
    for (int j = 0; j < kRowChunks; ++j) {
        const int c = t + j * kRowThreads;
        if (c >= nc) break;
        float v[8], g[8];
        const float4 p = reinterpret_cast<const float4*>(xrow)[2 * c];
        const float4 q = reinterpret_cast<const float4*>(xrow)[2 * c + 1];
        v[0] = p.x; v[1] = p.y; v[2] = p.z; v[3] = p.w; v[4] = q.x; v[5] = q.y; v[6] = q.z; v[7] = q.w;
        Vec16<bf16_t>::widen(j < kPreChunks ? gq[j < kPreChunks ? j : 0]
                                            : *reinterpret_cast<const uint4*>((const bf16_t*)a.gamma + 8 * c),
                             g);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = v[e] * rs * g[e];
        put_operand<2>(xb, N, B_pad, b, c, v);
    }
}

// ---- the RMSNorm scale after the product (LinearArgs::norm_post) ---------------------------
// The operand prep of an RMSNorm phase writes gamma * x and, per CTA (row b, column range
// y), the sum of squares of x over its columns in sq[y * B_pad + b]; the product kernel sums
// them (fixed order) to 1 / sqrt(mean(x^2) + eps) and multiplies its products by it. So
// the prep needs no whole-row pass and runs column-parallel like any other.
constexpr int kAuxRs = 0;      // bytes into the counter buffer: the last normalised phase's scales
constexpr int kAuxSq = 512;    // the prep's sums of squares [ny][kLinMmaMaxRows]
constexpr int kAuxEnd = 4608;  // (ny <= 8: K <= 16384)

// ---- the product ---------------------------------------------------------------------------
// Epilogue for output row m of sequences b0 .. b0 + W - 1; v[b] is b0 + b's finished product.
// SwiGLU pairs rows (2j, 2j + 1) held by neighbouring lanes of one warp.
template <int W>
__device__ __forceinline__ void lin_epilogue(const LinearArgs& a, int m, int b0, const float (&v)[W]) {
    const int lane = threadIdx.x & 31;
    // Every operand is read before any result is written: a load after a store to the same
    // buffer would wait for it, making the 32 rows one chain of L2 round trips.
    if (a.epi == EPI_SWIGLU) {
        float o[W];
#pragma unroll
        for (int b = 0; b < W; ++b) o[b] = silu(v[b]) * __shfl_xor_sync(0xffffffffu, v[b], 1);
        if ((lane & 1) || m + 1 >= a.M) return;
        float* y = a.y + (m >> 1);
#pragma unroll
        for (int b = 0; b < W; ++b)
            if (b0 + b < a.B) y[(size_t)(b0 + b) * a.ldy] = o[b];
        return;
    }
    if (m >= a.M) return;
    float* y = a.y + m;
    if (a.epi == EPI_RESID) {
        const float* base = a.ybase ? a.ybase + m : y;
        float r[W];
#pragma unroll
        for (int b = 0; b < W; ++b) r[b] = b0 + b < a.B ? __ldcg(base + (size_t)(b0 + b) * a.ldy) : 0.f;
#pragma unroll
        for (int b = 0; b < W; ++b) {
            if (b0 + b >= a.B) break;
            const float nv = r[b] + v[b];
            y[(size_t)(b0 + b) * a.ldy] = nv;
            if (a.y2) a.y2[(size_t)(b0 + b) * a.ldy2 + m] = nv;
        }
        return;
    }
#pragma unroll
    for (int b = 0; b < W; ++b)
        if (b0 + b < a.B) y[(size_t)(b0 + b) * a.ldy] = v[b];
}

// BP: B_pad, 8 .. 64 (with two splits also 96 and 128); MT: tiles to a unit; NS: splits (see the file comment; three: weights through the tensor map)
template <int BP, int NS, int MT>
__global__ void __launch_bounds__(lin_threads(NS), 1) linear_mma_kernel(const LinearArgs a, uint16_t* xb, int S,
                                                                   int stage_bytes, uint32_t tmem_cols, float* part,
                                                                   int* counters, unsigned char* aux,
                                                                   const __grid_constant__ CUtensorMap wmap) {
    const LaunchStamp stamp(a.stamp ? a.stamp + (a.prepped ? 0 : 2) : nullptr);
    constexpr int N = operand_rows(BP, NS);
    constexpr bool TM = NS == 3;  // tile layout read through the tensor map, one chain per unit
    constexpr int NA = acc_buffers(N, NS, MT);
    // one chain per unit and no more slots than accumulators: the chain's completion also
    // frees its slot (a unit S later cannot be loaded before it, so no phase is ever missed)
    const bool one_commit = TM && S <= NA;
    extern __shared__ unsigned char dsm_raw[];
    __shared__ LinMmaState st;
    __shared__ float rs_s[BP];  // norm_post: the rows' RMSNorm scales
    unsigned char* ring = (unsigned char*)(((uintptr_t)dsm_raw + 1023) & ~(uintptr_t)1023);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int G = gridDim.x, cta = blockIdx.x;
    const int nkb = a.K / 64;
    const int ntiles = (a.M + 127) / 128;
    const int64_t U = (int64_t)((ntiles + MT - 1) / MT) * nkb;
    const int64_t u0 = unit_begin(cta, U, G), u1 = unit_begin(cta + 1, U, G);
    const int tile0 = (int)(u0 / nkb), tile1 = (int)((u1 - 1) / nkb);  // tiles (pairs, MT = 2) this CTA touches
    // a commit block without rows (the plan was complete before the commit's first product
    // could start): nothing to do, no weights to read
    if (a.total && *a.total <= a.row0) {
        griddep_launch_dependents();
        griddep_wait();
        return;
    }

    if (t == 0) {
        for (int i = 0; i < S; ++i) {
            mbar_init(&st.full[i], 1);
            mbar_init(&st.empty[i], 1);
        }
        for (int i = 0; i < NA; ++i) {
            mbar_init(&st.tfull[i], 1);
            mbar_init(&st.tempty[i], 4);
        }
        mbar_init(&st.drain[0], 1);
        mbar_init(&st.drain[1], 1);
        st.abort = 0;
        mbar_fence_init();
    }
    if (warp == 0) tc_alloc(&st.tmem_base, tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = st.tmem_base;
    griddep_launch_dependents();

    // Ring positions advance by counters (slot, phase bit), not by division: the producer and
    // the MMA issuer are single threads whose every instruction is on the stream's critical
    // path.
    if (warp == 4) {  // ---- TMA producer
        if (lane == 0) {
            const int total = (int)(u1 - u0);
            const int pre = min(S, total);
            const uint32_t xbytes = (uint32_t)N * 128u;
            const unsigned char* Wsrc = (const unsigned char*)a.W + ((size_t)a.tile0 * nkb + u0) * 16384;
            const uint64_t wpol = l2_evict_first();  // weights are read once per draft
            int pt = tile0, pk = (int)(u0 - (int64_t)tile0 * nkb);  // MT: the next copy's pair and block
            int wt = (a.tile0 + tile0) * 32, wk = (int)(u0 - (int64_t)tile0 * nkb);  // TM: the next box's first group, block
            if constexpr (TM) tma_prefetch_map(&wmap);
            auto load_w = [&](unsigned char* dst, int it, uint64_t* bar) {
                if constexpr (TM) {
                    tma_load_3d(dst, &wmap, 0, wt, wk, bar, wpol);
                    if (++wk == nkb) { wk = 0; wt += 32; }
                } else if constexpr (MT == 2) {  // (a last tile without a partner: its half is not read)
                    const unsigned char* w0 = (const unsigned char*)a.W + ((size_t)(a.tile0 + 2 * pt) * nkb + pk) * 16384;
                    bulk_g2s_hint(dst, w0, 16384, bar, wpol);
                    if (2 * pt + 1 < ntiles) bulk_g2s_hint(dst + 16384, w0 + (size_t)nkb * 16384, 16384, bar, wpol);
                    if (++pk == nkb) { pk = 0; ++pt; }
                } else {
                    bulk_g2s_hint(dst, Wsrc + (size_t)it * 16384, 16384, bar, wpol);
                }
            };
            // the weights do not depend on earlier kernels: the first stages go out at once
            auto wbytes = [&]() { return MT == 2 && 2 * pt + 1 < ntiles ? 32768u : 16384u; };  // of the next copy
            for (int it = 0; it < pre; ++it) {
                mbar_arrive_expect_tx(&st.full[it], wbytes() + xbytes);
                load_w(ring + (size_t)it * stage_bytes, it, &st.full[it]);
            }
            griddep_wait();
            int kx = (int)(u0 % nkb);  // activation block of the next copy: (u0 + it) % nkb
            for (int it = 0; it < pre; ++it) {
                bulk_g2s(ring + (size_t)it * stage_bytes + MT * 16384, (const unsigned char*)xb + (size_t)kx * xbytes,
                         xbytes, &st.full[it]);
                if (++kx == nkb) kx = 0;
            }
            // iteration it >= S reuses slot it % S after the MMAs of iteration it - S: completion
            // (it - S) / S of empty[slot]
            int slot = 0, acc = 0;
            uint32_t pe = 0, pa = 0;
            int it = pre;
            for (; it < total; ++it) {
                if (!mbar_wait_abortable(one_commit ? &st.tfull[acc] : &st.empty[slot], one_commit ? pa : pe, a.status,
                                         &st.abort))
                    break;
                if (++acc == NA) { acc = 0; pa ^= 1u; }
                unsigned char* dst = ring + (size_t)slot * stage_bytes;
                mbar_arrive_expect_tx(&st.full[slot], wbytes() + xbytes);
                load_w(dst, it, &st.full[slot]);
                bulk_g2s(dst + MT * 16384, (const unsigned char*)xb + (size_t)kx * xbytes, xbytes, &st.full[slot]);
                if (++kx == nkb) kx = 0;
                if (++slot == S) { slot = 0; pe ^= 1u; }
            }
            st.issued = it;
        }
    } else if (TM && warp >= 5) {  // ---- MMA issuers: warps 5 and 6 take alternate units
        // (one thread needs ~850 cycles for a unit's waits, four MMAs and commits, more than
        // the ~680 a unit takes to arrive; the chains are independent, so two threads overlap.
        // With an odd number of slots or accumulators an issuer meets each of them at every other
        // use only, the other issuer's uses between; no wait can take the phase before last for
        // its own all the same. tempty[buf] of unit `it` follows the drain of unit it - NA, and
        // units are drained in order: so every unit up to it - NA has arrived, it - S among them
        // (NA <= S: launch_bp), and full[slot] is in the phase of unit `it`. And before, this
        // issuer waited for the drain of it - 2 - NA, so that of it - 2 NA (NA >= 2) is done and
        // tempty[buf] is in the phase that the drain of it - NA completes.)
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16_f32(128, N);
            const int total = (int)(u1 - u0);
            int slot = (warp - 5) % S, buf = (warp - 5) % NA;
            uint32_t pf = 0, pe = 1;  // phase bits of full[slot], tempty[buf] (accumulators start empty)
            for (int it = warp - 5; it < total; it += 2) {
                if (!mbar_wait_abortable(&st.tempty[buf], pe, a.status, &st.abort) ||
                    !mbar_wait_abortable(&st.full[slot], pf, a.status, &st.abort))
                    break;
                tc_fence_after();
                const uint32_t sa = smem_u32(ring + (size_t)slot * stage_bytes);
                const uint64_t adesc = sw128_desc(sa), bdesc = sw128_desc(sa + 16384);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    tc_mma(tmem + (uint32_t)(buf * N), adesc + 2 * kk, bdesc + 2 * kk, idesc, kk ? 1u : 0u);
                if (!one_commit) tc_commit(&st.empty[slot]);
                tc_commit(&st.tfull[buf]);
                if ((slot += 2) >= S) { slot -= S; pf ^= 1u; }
                if ((buf += 2) >= NA) { buf -= NA; pe ^= 1u; }
            }
            if (*(volatile int*)&st.abort) drain_mmas(&st.drain[warp - 5], a.status);
        }
    } else if (warp == 5) {  // ---- MMA issuer
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16_f32(128, N);
            int64_t u = u0;
            int slot = 0;
            uint32_t pf = 0;  // phase bit of full[slot]
            bool ok = true;
            for (int tile = tile0, j = 0; ok && tile <= tile1; ++tile, ++j) {
                const int buf = j % NA;
                const int64_t ue = min(u1, (int64_t)(tile + 1) * nkb);
                if (!mbar_wait_abortable(&st.tempty[buf], ((uint32_t)(j / NA) & 1u) ^ 1u, a.status, &st.abort)) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem + (uint32_t)(buf * MT * N);
                for (bool first = true; u < ue; ++u, first = false) {
                    if (!mbar_wait_abortable(&st.full[slot], pf, a.status, &st.abort)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(ring + (size_t)slot * stage_bytes);
                    const uint64_t bdesc = sw128_desc(sa + MT * 16384);
#pragma unroll
                    for (int h = 0; h < MT; ++h) {
                        const uint64_t adesc = sw128_desc(sa + h * 16384);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            tc_mma(d_tmem + (uint32_t)(h * N), adesc + 2 * kk, bdesc + 2 * kk, idesc, (!first || kk) ? 1u : 0u);
                    }
                    tc_commit(&st.empty[slot]);
                    if (++slot == S) { slot = 0; pf ^= 1u; }
                }
                if (ok) tc_commit(&st.tfull[buf]);
            }
            if (*(volatile int*)&st.abort) drain_mmas(&st.drain[0], a.status);
        }
    } else {  // ---- epilogue warps 0..3: TMEM lane 32 w + l = output row of the tile
        // rs_s: the per-row factor of the products (norm_post: the RMSNorm scales, else 1)
        const bool scaled = a.norm_post && a.pro == PRO_RMSNORM;
        griddep_wait();  // the epilogue reads and writes activations of earlier kernels
        if (scaled) {  // the rows' scales from the prep's sums of squares
            const float* sq = (const float*)(aux + kAuxSq);
            const int ny = (a.K / 8 + kXprepChunks - 1) / kXprepChunks;
            // row b = b0 + t / 4 sums column ranges y = t % 4, t % 4 + 4 (loads first, then in
            // order), then the four lanes combine in a fixed pattern
            const int p0 = t & 3;
#pragma unroll
            for (int b0 = 0; b0 < BP; b0 += 32) {
                const int b = b0 + (t >> 2);
                float q0 = 0.f, q1 = 0.f;
                if (b < BP) {
                    if (p0 < ny) q0 = __ldcg(sq + (size_t)p0 * BP + b);
                    if (p0 + 4 < ny) q1 = __ldcg(sq + (size_t)(p0 + 4) * BP + b);
                }
                float acc4 = q0 + q1;
                acc4 += __shfl_xor_sync(0xffffffffu, acc4, 1);
                acc4 += __shfl_xor_sync(0xffffffffu, acc4, 2);
                if (b < BP && p0 == 0) rs_s[b] = 1.0f / sqrtf(acc4 / (float)a.K + a.eps);
            }
            named_sync(1, 128);  // (the four epilogue warps)
            // a deferred split tile of this phase is finished by the next phase's prep, which
            // reads these (the previous phase's scales were read by this phase's prep,
            // complete before this kernel's griddep_wait returned)
            if (cta == 0 && t < BP) ((float*)(aux + kAuxRs))[t] = rs_s[t];
        }
        const int r = warp * 32 + lane;
        bool ok = true;
        int buf = 0;
        uint32_t pt = 0;  // phase bit of tfull[buf]
        // columns a thread holds at a time: all, or half of more than 64
        constexpr int W = BP <= 64 ? BP : BP / 2;
        for (int tile = tile0; ok && tile <= tile1; ++tile) {
            const int c_first = unit_owner((int64_t)tile * nkb, U, G);
            const int c_last = unit_owner((int64_t)(tile + 1) * nkb - 1, U, G);
            // this CTA's products (a split tile's share stays unscaled), chain by chain
            float v[W], vc[TM ? W : 1];
            if constexpr (TM) {
#pragma unroll
                for (int b = 0; b < W; ++b) vc[b] = 0.f;
            }
            // what becomes of columns b0 .. of the products: the epilogue when the whole tile was
            // ours, else this CTA's share (slot 0 for its first tile, 1 for its last)
            auto finish = [&](int b0, int h) {  // (h: which tile of a pair)
                const int m = (tile * MT + h) * 128 + r;
                if (c_first == c_last) {
                    if (scaled) {
#pragma unroll
                        for (int b = 0; b < W; ++b) v[b] *= rs_s[b0 + b];
                    }
                    lin_epilogue<W>(a, m, b0, v);
                } else {
                    float* pp = part + (((size_t)(cta * 2 + (tile == tile0 ? 0 : 1)) * MT + h) * BP + b0) * 128 + r;
#pragma unroll
                    for (int b = 0; b < W; ++b) pp[(size_t)b * 128] = v[b];
                }
            };
            const int64_t ub = max(u0, (int64_t)tile * nkb), ue = min(u1, (int64_t)(tile + 1) * nkb);
            for (int64_t u = ub; u < ue; u += TM ? 1 : ue - ub) {
                if (!mbar_wait_abortable(&st.tfull[buf], pt, a.status, &st.abort)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(buf * MT * N);
                float big = 0.f;  // the largest compensated sum
#pragma unroll 1
                for (int h = 0; h < MT; ++h)
#pragma unroll
                for (int b0 = 0; b0 < BP; b0 += W) {
#pragma unroll
                    for (int b = 0; b < W; b += 8) {
                        uint32_t x[NS][8];
#pragma unroll
                        for (int q = 0; q < NS; ++q) tc_ld8_async(taddr + h * N + q * BP + b0 + b, x[q]);
                        tc_ld_wait();
#pragma unroll
                        for (int q = 0; q < NS; ++q) tc_ld_pin(x[q]);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            float y = __uint_as_float(x[NS - 1][i]);
#pragma unroll
                            for (int q = NS - 2; q >= 0; --q) y = __uint_as_float(x[q][i]) + y;
                            if (!TM || u == ub) {
                                v[b + i] = y;
                            } else {  // compensated (Kahan): vc is what the last addition lost
                                const float x0 = y - vc[b + i], s0 = v[b + i] + x0;
                                vc[b + i] = (s0 - v[b + i]) - x0;
                                v[b + i] = s0;
                                big = fmaxf(big, fabsf(s0));
                            }
                        }
                    }
                    if (h + 1 < MT || b0 + W < BP) finish(b0, h);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&st.tempty[buf]);
                if constexpr (TM)
                    if (big == INFINITY) {  // an infinite sum has lost nothing: left alone, the next
                                            // addition would be inf - inf
#pragma unroll
                        for (int b = 0; b < W; ++b)
                            if (fabsf(v[b]) == INFINITY) vc[b] = 0.f;
                    }
                if (++buf == NA) { buf = 0; pt ^= 1u; }
            }
            if (!ok) break;
            finish(BP - W, MT - 1);
            // Rows are independent, so each warp finishes its own 32 rows of a split tile (its own
            // counter): no wait on another warp. Deferred: the next phase's operand prep does.
            if (c_first == c_last || a.defer) continue;
            // lane 0's acquire-release add publishes the warp's shares (ordered before it by
            // the warp barrier) and, in the last warp to arrive, orders the reads below
            __syncwarp();
            int last = 0;
            if (lane == 0) last = atom_add_acq_rel_gpu(&counters[tile * 4 + warp], 1) == c_last - c_first;
            last = __shfl_sync(0xffffffffu, last, 0);
            if (!last) continue;
            // (slot 1 only for c_first, when the tile is not its first: see prev_finish_t)
            const int cs_first = unit_begin(c_first, U, G) < (int64_t)tile * nkb ? 1 : 0;
#pragma unroll 1
            for (int hb = 0; hb < MT * (BP / W); ++hb) {
                const int h = hb / (BP / W), b0 = hb % (BP / W) * W;
                float s[W];
#pragma unroll
                for (int b = 0; b < W; ++b) s[b] = 0.f;
                for (int c = c_first; c <= c_last; ++c) {
                    const int cs = c == c_first ? cs_first : 0;
                    const float* q = part + (((size_t)(c * 2 + cs) * MT + h) * BP + b0) * 128 + r;
                    float x[W];
#pragma unroll
                    for (int b = 0; b < W; ++b) x[b] = __ldcg(q + (size_t)b * 128);
#pragma unroll
                    for (int b = 0; b < W; ++b) s[b] += x[b];
                }
                if (scaled) {
#pragma unroll
                    for (int b = 0; b < W; ++b) s[b] *= rs_s[b0 + b];
                }
                lin_epilogue<W>(a, (tile * MT + h) * 128 + r, b0, s);
            }
            if (lane == 0) counters[tile * 4 + warp] = 0;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (t == 0 && *(volatile int*)&st.abort) drain_copies(st.full, S, st.issued, a.status);
    if (warp == 0) tc_dealloc(tmem, tmem_cols);
}

// ---- host side -----------------------------------------------------------------------------
// Above 64 rows and with more tiles than CTAs a unit is a 64-column block of TWO tiles sharing one
// operand block: with one tile the operand (32 KB a block at 128 rows, two splits) makes an SM read
// 48 KB from L2 per 16 KB of weights, and gate/up of the 8B shape (28672 x 4096, 224 tiles on 152
// SMs) took 64 us; with two 48 (a commit of 150 rows: 1289 -> 1215 us). Their accumulators of up to
// 512 columns fill the tensor memory (no second buffer), and a pair is cut between twice as many
// CTAs: matrices of few tiles lose (O projection 15 -> 19 us, W_fuse 26 -> 31).
int linear_mma_mt(int M, int B, int splits, const DeviceInfo& dev) {
    return splits == 2 && B > kTileMaxRows && (M + 127) / 128 > dev.num_sms ? 2 : 1;
}

namespace {

template <int BP, int NS, int MT>
cudaError_t set_attr(const DeviceInfo& dev) {
    return cudaFuncSetAttribute(linear_mma_kernel<BP, NS, MT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                dev.max_smem_optin - (int)sizeof(LinMmaState) - 1024);
}

template <int BP, int NS, int MT = 1>
cudaError_t launch_bp(const LinearArgs& a, uint16_t* xb, float* part, int* counters, unsigned char* aux,
                      const DeviceInfo& dev, cudaStream_t st, int grid) {
    constexpr int N = operand_rows(BP, NS);
    const int stage_bytes = MT * 16384 + N * 128;
    const size_t budget = (size_t)dev.max_smem_optin - sizeof(LinMmaState) - 1024 - 1024;
    int S = (int)(budget / stage_bytes);
    S = S > kLinMaxStages ? kLinMaxStages : S;
    if (S < 2 || (NS == 3 && S < acc_buffers(N, NS, MT))) return cudaErrorInvalidValue;
    const size_t smem = 1024 + (size_t)S * stage_bytes;
    uint32_t cols = 32;
    while (cols < (uint32_t)(acc_buffers(N, NS, MT) * MT * N)) cols <<= 1;
    static const CUtensorMap none{};
    return launch_k(linear_mma_kernel<BP, NS, MT>, dim3(grid), dim3(lin_threads(NS)), smem, st, a.pdl, a, xb, S,
                    stage_bytes, cols, part, counters, aux, NS == 3 ? *a.wmap : none);
}

// the operand paddings: 8, 16, .. 64, and with two splits 96 and 128
constexpr int next_bp(int bp) { return bp < kTileMaxRows ? bp + 8 : bp + 32; }

template <int BP = 8>
cudaError_t prepare_bp(const DeviceInfo& dev) {
    cudaError_t e = set_attr<BP, 2, 1>(dev);
    if constexpr (BP <= kTileMaxRows) {
        if (e == cudaSuccess) e = set_attr<BP, 3, 1>(dev);
    } else {
        if (e == cudaSuccess) e = set_attr<BP, 2, 2>(dev);
    }
    if constexpr (BP < kLinMmaMaxRows)
        if (e == cudaSuccess) e = prepare_bp<next_bp(BP)>(dev);
    return e;
}

template <int BP = 8>
cudaError_t launch_product(const LinearArgs& a, uint16_t* xb, float* part, int* counters, unsigned char* aux,
                           const DeviceInfo& dev, cudaStream_t st, int grid) {
    if constexpr (BP < kLinMmaMaxRows)
        if (linear_mma_bpad(a.B) > BP) return launch_product<next_bp(BP)>(a, xb, part, counters, aux, dev, st, grid);
    if constexpr (BP <= kTileMaxRows)
        if (a.splits == 3) return launch_bp<BP, 3>(a, xb, part, counters, aux, dev, st, grid);
    if constexpr (BP > kTileMaxRows)
        if (linear_mma_mt(a.M, a.B, a.splits, dev) == 2) return launch_bp<BP, 2, 2>(a, xb, part, counters, aux, dev, st, grid);
    return launch_bp<BP, 2>(a, xb, part, counters, aux, dev, st, grid);
}

}  // namespace

int linear_mma_bpad(int B) { return B <= kTileMaxRows ? (B + 7) / 8 * 8 : (B + 31) / 32 * 32; }

bool linear_mma_ok(int M, int K, int B) { return M > 0 && K % 64 == 0 && B >= 1 && B <= kLinMmaMaxRows; }

size_t linear_mma_xb_bytes(int K, int B, int splits) { return (size_t)operand_rows(linear_mma_bpad(B), splits) * K * 2; }


int linear_mma_grid(int M, int K, const DeviceInfo& dev, int mt) {
    const int64_t U = (int64_t)(((M + 127) / 128 + mt - 1) / mt) * (K / 64);
    return (int)(U < dev.num_sms ? U : dev.num_sms);
}

size_t linear_mma_part_bytes(int B, const DeviceInfo& dev) {
    return (size_t)dev.num_sms * 2 * (B > kTileMaxRows ? 2 : 1) * linear_mma_bpad(B) * 128 * sizeof(float);
}

namespace {
// the split-tile counters' offset in the counter buffer (after the RMSNorm scales and sums)
size_t tile_counter_offset(const DeviceInfo&) { return kAuxEnd; }
}  // namespace

size_t linear_mma_counter_bytes(int M_max, const DeviceInfo& dev) {
    return tile_counter_offset(dev) + 4 * (size_t)((M_max + 127) / 128) * sizeof(int);
}

float* linear_mma_rs(int* counters) { return (float*)((unsigned char*)counters + kAuxRs); }

cudaError_t linear_mma_prepare(const DeviceInfo& dev) {
    cudaError_t e = cudaFuncSetAttribute(xprep_row_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kXprepRowSmem);
    if (e != cudaSuccess) return e;
    return prepare_bp(dev);
}

// The tensor map of a tile-layout matrix: 128 32-bit elements (a group's 4 rows x 64 columns)
// x groups x 64-column blocks, box 128 x 32 x 1: the 32 groups of a 128-row tile at one block,
// which land in shared memory as the 16 KB swizzled operand. Groups past M read zeros.
cudaError_t linear_mma_map(const void* W, int M, int K, CUtensorMap* map) {
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Encode encode = [] {  // (the library does not link the driver API)
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        const cudaError_t e =
            cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found);
        return e == cudaSuccess && found == cudaDriverEntryPointSuccess ? (Encode)fn : nullptr;
    }();
    if (!encode) return cudaErrorNotSupported;
    const cuuint64_t dims[3] = {128, (cuuint64_t)((M + 3) / 4), (cuuint64_t)(K / 64)};
    const cuuint64_t strides[2] = {(cuuint64_t)K * 8, 512};
    const cuuint32_t box[3] = {128, 32, 1}, step[3] = {1, 1, 1};
    const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, const_cast<void*>(W), dims, strides, box, step,
                                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t launch_linear_mma(const LinearArgs& a, uint16_t* xb, float* part, int* counters, const DeviceInfo& dev,
                              cudaStream_t st, cudaEvent_t after_prep) {
    if (!linear_mma_ok(a.M, a.K, a.B) || (a.splits == 3 && (!a.wmap || a.B > kTileMaxRows))) return cudaErrorInvalidValue;
    const int BP = linear_mma_bpad(a.B);
    unsigned char* aux = (unsigned char*)counters;
    int* tctr = (int*)(aux + tile_counter_offset(dev));
    const int grid = linear_mma_grid(a.M, a.K, dev, linear_mma_mt(a.M, a.B, a.splits, dev));
    // finish + normalise a row per CTA (only when the scale goes on the operand)
    const bool row_cta = !a.norm_post && a.prev.active && a.pro == PRO_RMSNORM;
    if (row_cta && ((size_t)a.K * sizeof(float) > kXprepRowSmem || a.prev.epi == EPI_SWIGLU || a.splits != 2))
        return cudaErrorInvalidValue;
    const int ny = (a.K / 8 + kXprepChunks - 1) / kXprepChunks;
    if (a.norm_post && a.pro == PRO_RMSNORM && (size_t)ny * kLinMmaMaxRows * sizeof(float) > kAuxEnd - kAuxSq)
        return cudaErrorInvalidValue;
    // (prepped: the operand is in place, the attention kernel wrote it)
    if (a.prepped) return a.prev.active ? cudaErrorInvalidValue : launch_product(a, xb, part, tctr, aux, dev, st, grid);
    float* sq = (float*)(aux + kAuxSq);
    cudaError_t e = row_cta ? launch_k(xprep_row_kernel, dim3(BP), dim3(kRowThreads), (size_t)a.K * sizeof(float), st,
                                       a.pdl, a, BP, xb)
                            : launch_k(a.splits == 3 ? xprep_kernel<3> : xprep_kernel<2>, dim3(BP, ny), dim3(256), 0, st,
                                       a.pdl, a, BP, xb, sq);
    if (e != cudaSuccess) return e;
    if (after_prep && (e = cudaEventRecord(after_prep, st)) != cudaSuccess) return e;
    return launch_product(a, xb, part, tctr, aux, dev, st, grid);
}

cudaError_t launch_linear_finish(const LinearArgs::Prev& p, int B, int cols, const int* total, int row0, bool pdl,
                                 cudaStream_t st) {
    if (cols % 8 || p.epi != EPI_STORE) return cudaErrorInvalidValue;
    return launch_k(finish_kernel, dim3(B, (cols + 2047) / 2048), dim3(256), 0, st, pdl, p, linear_mma_bpad(B), cols, total,
                    row0);
}

}  // namespace fe
