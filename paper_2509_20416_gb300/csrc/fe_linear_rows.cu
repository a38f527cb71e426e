// Linear phases of drafts of many rows on the CUDA cores, bit for bit what linear_kernel
// (fe_linear.cu) computes, with every weight streamed once for up to 64 rows.
//
// Drafts of more than 16 hidden rows round z once to bf16 before the LM head, so float32 sums
// taken in another order would show in their probabilities; these drafts therefore keep the
// streaming kernel's exact order of additions. The streaming kernel itself holds a whole
// activation row per batch row in shared memory (8 rows of 16 KB at most), streams the weights
// once per such tile and reads 2 KB of activations per 512 bytes of weights and lane group: 56
// rows of an 8B-shaped two-layer draft took 4470 us of linear phases, 4750 in all.
//
// The order (linear_kernel): the columns of a row are cut into slices of 1024; slice ks of group
// g goes to warp (phase + ks) % 8 of its CTA; lane l of a warp runs one FMA chain over the
// 16-byte vectors l, l + 32, .. of its slices; lanes add up in a butterfly (16, 8, 4, 2, 1), the
// eight warps' sums in warp order. So an output is a fixed tree over 32 chains per class (the
// slices j, j + 8, ..), and any kernel that builds the same chains and the same tree gives the
// same bits. Here:
//   - A CTA takes up to 8 row groups (32 weight rows) x all batch rows at a time and walks the
//     columns in 64-column blocks: 4 KB of weights (the tile layout) and the activations of that
//     block, both by bulk copies into a ring. xrows_kernel lays the activations out so that
//     one copy lands a block, chunk of 8 columns by chunk, rows paired for two-wide FMAs.
//   - Warp w of each of two warp groups (16 rows of weights each) takes chunk w of every block,
//     i.e. the chains of lanes w, w + 8, w + 16, w + 24; its lanes are 4 weight rows x 8 batch
//     rows, each lane 4 x NB outputs in registers. A block's loads are broadcasts (one
//     shared-memory wavefront each): 22 per 224 multiply-adds at 56 rows.
//   - Blocks come in the order of the chains: lane quarter by quarter (0, 2, 1, 3), so that the
//     butterfly's first two steps are register additions; its last three go through a small
//     exchange buffer once per class, and the classes' sums are added in warp order at the end.
// Bound by issue: at 56 rows a warp executes 312 instructions a block, 128 for the 224 multiply-adds
// (96 two-wide, 32 one-wide), 64 to widen weights, 22 for the loads above and ~98 of ring, class and
// loop overhead, and issues in 64 % of the cycles. Gate/up of the 8B shape at 56 rows (235 MB):
// streaming kernel 663 us, here 369; one-wide FMAs 450. The whole draft above: 4750 -> 2247 us.
#include <algorithm>

#include "fe_kernels.h"
#include "fe_stream.cuh"

namespace fe {

namespace {

constexpr int kRwThreads = 512;  // two groups of 8 warps
constexpr int kRwMaxStages = 6;
constexpr int kRwGroups = 8;     // row groups per CTA pass (two warp groups of 4)

struct RowsState {
    uint64_t full[kRwMaxStages], empty[kRwMaxStages];
    int last[kRwMaxStages];  // the iteration whose copies a slot last took
    int abort;
};

__host__ __device__ constexpr int quarter(int q) { return q == 1 ? 2 : q == 2 ? 1 : q; }  // 0, 2, 1, 3

// 64-column blocks in chain order: calls f(block) for class j, lane quarter h of slices [lo, hi)
template <typename F>
__device__ __forceinline__ void walk_chain(int lo, int hi, int j, int h, int nkb, F&& f) {
    for (int ks = lo + j; ks < hi; ks += 8)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int blk = ks * 16 + h + 4 * i;
            if (blk < nkb) f(blk);
        }
}

}  // namespace

// Where batch row r of a row tile sits: lane bl and index k of its NB rows. Rows 2 m and 2 m + 1
// share a lane and a two-wide FMA; the last eight of an odd NB are single.
template <int NB>
__host__ __device__ __forceinline__ int tile_row(int k, int bl) {
    return k < NB / 2 * 2 ? k / 2 * 16 + bl * 2 + (k & 1) : NB / 2 * 16 + bl;
}

// Two rows per CTA (threadIdx.y): the rows' activations exactly as linear_kernel stages them,
// into the block layout xs [row tile][K / 64][8 chunks][8 RT floats] of rows_step.
__global__ void __launch_bounds__(2 * kStreamThreads) xrows_kernel(const LinearArgs a, int RT, float* xs) {
    const LaunchStamp stamp(a.stamp);
    extern __shared__ __align__(16) float xrow[];  // [2][K]
    __shared__ float scratch[2][kWarps];
    const int y = threadIdx.y, b = min(2 * (int)blockIdx.x + y, a.B - 1), K = a.K, nkb = K / 64;
    float* mine = xrow + (size_t)y * K;
    griddep_launch_dependents();
    ProParams pp{a.pro, a.x, a.ldx, a.gamma, a.eps, a.embed, a.tok, a.d_split, a.vocab};
    const bool pre = stage_pre<bf16_t>(pp, K, mine, K, b, 1, a.status);
    griddep_wait();
    stage_activations<bf16_t>(pp, K, mine, K, b, 1, a.status, scratch[y], pre);
    __syncthreads();
    const int NP = RT / 16, r = 2 * (int)blockIdx.x % RT;  // the CTA's first row in its tile (RT is even)
    float* dst = xs + (size_t)(2 * (int)blockIdx.x / RT) * nkb * 64 * RT;
    const int t = y * kStreamThreads + threadIdx.x;
    if (r < 16 * NP) {
        for (int q = t; q < K / 2; q += 2 * kStreamThreads) {  // columns 2 q, 2 q + 1: chunk q / 4, word u = q % 4
            const float2 x = reinterpret_cast<const float2*>(xrow)[q], z = reinterpret_cast<const float2*>(xrow + K)[q];
            reinterpret_cast<float4*>(dst + (size_t)(q / 4) * 8 * RT)[(q % 4 * NP + r / 16) * 8 + r % 16 / 2] =
                make_float4(x.x, z.x, x.y, z.y);
        }
    } else {
        for (int q = threadIdx.x; q < K / 4; q += kStreamThreads)  // columns 4 q ..: chunk q / 2, half q % 2
            reinterpret_cast<float4*>(dst + (size_t)(q / 2) * 8 * RT)[(4 * NP + q % 2) * 8 + r - 16 * NP + y] =
                reinterpret_cast<const float4*>(mine)[q];
    }
}

// Two float32 multiply-adds in one instruction (each rounded as fmaf rounds it); pairs are
// (low, high) words.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// bf16 element `odd` of word r as a float32 in both halves. Two byte permutations: as a shift or
// a move the compiler puts half of them on the FMA pipe, which is the one this kernel runs out of.
__device__ __forceinline__ f32x2 widen2(uint32_t r, int odd) {
    uint32_t lo, hi;
    if (odd) {
        asm volatile("prmt.b32 %0, %1, 0, 0x3244;" : "=r"(lo) : "r"(r));
        asm volatile("prmt.b32 %0, %1, 0, 0x3244;" : "=r"(hi) : "r"(r));
    } else {
        asm volatile("prmt.b32 %0, %1, 0, 0x1044;" : "=r"(lo) : "r"(r));
        asm volatile("prmt.b32 %0, %1, 0, 0x1044;" : "=r"(hi) : "r"(r));
    }
    return (f32x2)lo | (f32x2)hi << 32;
}

// A lane's outputs for one weight row: batch rows in pairs (2 q, 2 q + 1), and the last of an odd
// NB alone.
template <int NB>
struct RowAcc {
    static constexpr int NP = NB / 2, ODD = NB % 2;
    f32x2 p[NP > 0 ? NP : 1];
    float s;
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int q = 0; q < NP; ++q) p[q] = 0ull;
        s = 0.f;
    }
    __device__ __forceinline__ float get(int k) const {  // k a constant after unrolling
        float lo, hi;
        if (k < 2 * NP) {
            unpack2(p[k / 2], lo, hi);
            return k & 1 ? hi : lo;
        }
        return s;
    }
};

// One 64-column block: this warp's chunk of 8 columns of NI weight rows per lane (row i at byte
// wo[i] of the block) against NB batch rows, FMAs in column order. xp: the chunk's activations at
// this lane, 16-byte words 8 apart: word (u, q) holds columns 2u, 2u + 1 of rows 2q and 2q + 1
// interleaved ([4][NP] words), then, for an odd NB, two words of the last row's columns.
template <int NB, int NI>
__device__ __forceinline__ void rows_step(const unsigned char* sp, const uint32_t (&wo)[4], const uint4* xp,
                                          RowAcc<NB> (&acc)[4]) {
    constexpr int NP = NB / 2, ODD = NB % 2;
#pragma unroll
    for (int h = 0; h < 2; ++h) {  // columns 4 h .. 4 h + 3
        f32x2 w2[NI][4];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const uint2 r = *reinterpret_cast<const uint2*>(sp + wo[i] + 8 * h);
#pragma unroll
            for (int j = 0; j < 4; ++j) w2[i][j] = widen2(j < 2 ? r.x : r.y, j & 1);
        }
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            const ulonglong2 x0 = *reinterpret_cast<const ulonglong2*>(xp + ((2 * h) * NP + q) * 8);
            const ulonglong2 x1 = *reinterpret_cast<const ulonglong2*>(xp + ((2 * h + 1) * NP + q) * 8);
            const f32x2 x[4] = {x0.x, x0.y, x1.x, x1.y};
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < NI; ++i) acc[i].p[q] = fma2(w2[i][j], x[j], acc[i].p[q]);
        }
        if constexpr (ODD) {
            const float4 x = *reinterpret_cast<const float4*>(xp + (4 * NP + h) * 8);
            const float xj[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < NI; ++i) {
                    float w, dup;
                    unpack2(w2[i][j], w, dup);
                    acc[i].s = fmaf(w, xj[j], acc[i].s);
                }
        }
    }
}

// The ring as a consumer sees it.
struct RowsRing {
    RowsState* st;
    const unsigned char* base;
    int S, slot, it;
    uint32_t pf;
    int* status;
};

// One class of a warp's ni row groups: its four chains (len[q] blocks each), the butterfly's
// first two steps, and the warp's sums into its exchange rows `mine`. refill(it) keeps the ring
// full.
template <int NB, typename Refill>
__device__ __forceinline__ void rows_class(RowsRing& r, const uint8_t* len, int ni, const uint32_t (&wo)[4], uint32_t xo,
                                           float* mine, int wg, int lane, Refill&& refill) {
    constexpr uint32_t STAGE = kRwGroups * 512 + 64 * 8 * NB * sizeof(float);
    RowAcc<NB> keep[4], acc[4];
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i].clear();
        const int n = len[q];
#pragma unroll 1
        for (int s = 0; s < n; ++s) {
            mbar_wait_abortable(&r.st->full[r.slot], r.pf, r.status, &r.st->abort);
            const unsigned char* sp = r.base + (size_t)r.slot * STAGE;
            const uint4* xp = reinterpret_cast<const uint4*>(sp + xo);
            switch (ni) {  // (the same for the whole warp group)
                case 4: rows_step<NB, 4>(sp, wo, xp, acc); break;
                case 3: rows_step<NB, 3>(sp, wo, xp, acc); break;
                case 2: rows_step<NB, 2>(sp, wo, xp, acc); break;
                case 1: rows_step<NB, 1>(sp, wo, xp, acc); break;
                default: break;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&r.st->empty[r.slot]);
            refill(r.it);
            ++r.it;
            if (++r.slot == r.S) { r.slot = 0; r.pf ^= 1u; }
        }
        if (q == 1) named_sync(1 + wg, 256);  // the last class's exchange has been read
        // butterfly steps 16 (quarters 0 + 2, 1 + 3) and 8
        if (!(q & 1)) {
#pragma unroll
            for (int i = 0; i < 4; ++i) keep[i] = acc[i];
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int k = 0; k < NB; ++k) {
                    float* at = mine + (i * NB + k) * 32;
                    const float v = keep[i].get(k) + acc[i].get(k);
                    *at = q == 1 ? v : *at + v;
                }
        }
    }
}

// NB: batch rows per lane (row tiles of 8 NB); n0 as linear_kernel's (slices in its first
// activation pass, 0: one pass). The warps take turns at refilling the ring: after step `it`
// warp it % 16 waits until every warp is past step it - lag (they run within a step or two of
// each other) and asks for step it + S - lag into that slot.
template <int NB>
__global__ void __launch_bounds__(kRwThreads, 1) linear_rows_kernel(const LinearArgs a, const float* xs, int S, int n0) {
    const LaunchStamp stamp(a.stamp ? a.stamp + 2 : nullptr);
    constexpr int RT = 8 * NB;
    constexpr uint32_t XB = 64 * RT * sizeof(float), WB = kRwGroups * 512, STAGE = WB + XB;
    constexpr int OUT = 4 * NB * 32;  // outputs of a warp group
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ RowsState st;
    __shared__ uint8_t chain_len[64];  // blocks of chain (class, quarter): 4 per slice, few slices
    float* xch = reinterpret_cast<float*>(smem + (size_t)S * STAGE);  // [16 warps][OUT]
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int K = a.K, nkb = K / 64, nks = (K + 1023) / 1024;
    const int GM = (a.M + kGroupRows - 1) / kGroupRows;
    const int g0 = (int)(((int64_t)blockIdx.x * GM) / gridDim.x);
    const int g1 = (int)(((int64_t)(blockIdx.x + 1) * GM) / gridDim.x);
    const int ng = g1 - g0, nch = (ng + kRwGroups - 1) / kRwGroups;
    if (n0 <= 0 || n0 > nks) n0 = nks;
    const int npass = n0 < nks ? 2 : 1, classes = min(8, n0) + (npass == 2 ? min(8, nks - n0) : 0);
    float* sums = xch + 16 * OUT;                                            // [classes][2 OUT]
    uint16_t* order = reinterpret_cast<uint16_t*>(sums + classes * 2 * OUT);  // [nkb] blocks in step order
    const int lag = S >= 4 ? 2 : 1, total = nch * nkb;
    const unsigned char* X = (const unsigned char*)xs + (size_t)blockIdx.y * nkb * XB;
    if (t == 0) {
        for (int i = 0; i < S; ++i) {
            mbar_init(&st.full[i], 1);
            mbar_init(&st.empty[i], 16);
            st.last[i] = -1;
        }
        st.abort = 0;
        mbar_fence_init();
    }
    if (warp == 0) {  // chain (class, quarter) number lane, lane + 32, ..: its place is the chains' before it
        int base = 0;
        for (int ch0 = 0; ch0 < classes * 4; ch0 += 32) {
            const int ch = ch0 + lane, cl = ch >> 2, p = cl >= min(8, n0);
            const int lo = p ? n0 : 0, hi = p ? nks : n0, j = p ? cl - min(8, n0) : cl, h = quarter(ch & 3);
            int len = 0;
            if (ch < classes * 4) walk_chain(lo, hi, j, h, nkb, [&](int) { ++len; });
            int at = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, at, o);
                if (lane >= o) at += up;
            }
            const int sum = __shfl_sync(0xffffffffu, at, 31);
            at += base - len;
            if (ch < classes * 4) {
                chain_len[ch] = (uint8_t)len;
                walk_chain(lo, hi, j, h, nkb, [&](int blk) { order[at++] = (uint16_t)blk; });
            }
            base += sum;
        }
    }
    __syncthreads();
    griddep_launch_dependents();

    // step f's copies: the weight blocks of its chunk's groups, and (act) the activations
    const uint64_t pol = l2_evict_first();
    auto ask = [&](int f, int slot, bool weights, bool act) {
        const int c = f / nkb, blk = order[f - c * nkb];
        const int cg0 = g0 + ng * c / nch, n = g0 + ng * (c + 1) / nch - cg0;
        unsigned char* dst = smem + (size_t)slot * STAGE;
        if (weights) {
            mbar_arrive_expect_tx(&st.full[slot], (uint32_t)n * 512u + XB);
            st.last[slot] = f;
            for (int i = 0; i < n; ++i)
                bulk_g2s_hint(dst + i * 512, (const unsigned char*)a.W + ((size_t)(cg0 + i) * nkb + blk) * 512, 512,
                              &st.full[slot], pol);
        }
        if (act) bulk_g2s(dst + WB, X + (size_t)blk * XB, XB, &st.full[slot]);
    };
    if (t == 0)  // the weights do not depend on the previous kernel
        for (int f = 0; f < min(S - lag, total); ++f) ask(f, f, true, false);
    griddep_wait();
    if (t == 0)
        for (int f = 0; f < min(S - lag, total); ++f) ask(f, f, false, true);

    const int wg = warp >> 3, w = warp & 7, tw = t & 255, ml = lane >> 3, bl = lane & 7;
    const int b0 = blockIdx.y * RT;
    RowsRing ring{&st, smem, S, 0, 0, 0, a.status};
    float* mine = xch + warp * OUT + lane;  // output (i, k) of this lane at (i NB + k) 32
    const float* red = xch + wg * 8 * OUT;
    const uint32_t xo = WB + (uint32_t)(2 * w * RT + bl) * 16;
    auto refill = [&](int it) {
        const int f = it + S - lag;
        if ((it & 15) != warp || f >= total) return;
        if (lane == 0) {
            const int fs = f % S, use = f / S;  // the slot's use-th filling: its last was consumed
            if (use == 0 || mbar_wait_abortable(&st.empty[fs], (uint32_t)(use - 1) & 1u, a.status, &st.abort))
                ask(f, fs, true, true);
        }
        __syncwarp();
    };
    for (int c = 0; c < nch; ++c) {
        const int cg0 = g0 + ng * c / nch, n = g0 + ng * (c + 1) / nch - cg0;
        const int gq0 = wg ? (n + 1) / 2 : 0, ni = wg ? n / 2 : (n + 1) / 2;  // this warp group's row groups
        uint32_t wo[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            wo[i] = (uint32_t)((gq0 + i) * 512 + ml * 128 + ((w ^ (4 * ((cg0 + gq0 + i) & 1) + ml)) << 4));
        for (int cls = 0; cls < classes; ++cls) {
            const uint8_t* len = chain_len + cls * 4;
            rows_class<NB>(ring, len, ni, wo, xo, mine, wg, lane, refill);
            // steps 4, 2, 1 across the warps; the class's sums
            named_sync(1 + wg, 256);
#pragma unroll
            for (int k = 0; k < (NB + 1) / 2; ++k) {
                const int o = tw + 256 * k;
                if (o < ni * NB * 32) {
                    float v[8];
#pragma unroll
                    for (int x = 0; x < 8; ++x) v[x] = red[x * OUT + o];
                    sums[(size_t)cls * 2 * OUT + wg * OUT + o] =
                        ((v[0] + v[4]) + (v[2] + v[6])) + ((v[1] + v[5]) + (v[3] + v[7]));
                }
            }
        }
        // the classes' sums in warp order (each thread reads what it wrote), then the epilogue
#pragma unroll 1
        for (int k = 0; k < (NB + 1) / 2; ++k) {
            const int o = tw + 256 * k;
            const bool on = o < ni * NB * 32;  // (whole warps: OUT and 32 NB are multiples of 32)
            if (!on) continue;
            const int i = o / (NB * 32), k8 = o / 32 % NB;
            const int g = cg0 + gq0 + i, m = g * kGroupRows + ml, b = b0 + tile_row<NB>(k8, bl);
            const int f0 = (g - g0) * n0 & 7, f1 = (ng * n0 + (g - g0) * (nks - n0)) & 7;
            const int c0 = min(8, n0), c1 = npass == 2 ? min(8, nks - n0) : 0;
            const float* sp = sums + wg * OUT + o;
            float v = 0.f;
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                const int j0 = (x - f0) & 7, j1 = (x - f1) & 7;
                float s = 0.f;
                if (j0 < c0) s += sp[(size_t)j0 * 2 * OUT];
                if (j1 < c1) s += sp[(size_t)(c0 + j1) * 2 * OUT];
                v += s;
            }
            if (a.epi == EPI_SWIGLU) {  // rows 2j (gate) and 2j + 1 (up): lanes 8 apart
                const float up = __shfl_xor_sync(0xffffffffu, v, 8);
                if (!(ml & 1) && b < a.B && m + 1 < a.M) a.y[(size_t)b * a.ldy + (m >> 1)] = silu(v) * up;
            } else if (b < a.B && m < a.M) {
                float* yp = a.y + (size_t)b * a.ldy + m;
                if (a.epi == EPI_RESID) {
                    const float nv = __ldcg(a.ybase ? a.ybase + (size_t)b * a.ldy + m : yp) + v;
                    *yp = nv;
                    if (a.y2) a.y2[(size_t)b * a.ldy2 + m] = nv;
                } else {
                    *yp = v;
                }
            }
        }
    }
    // never leave with copies in flight (only after an abort)
    __syncthreads();
    if (t == 0 && *(volatile int*)&st.abort)
        for (int i = 0; i < S; ++i)
            if (st.last[i] >= 0) mbar_wait(&st.full[i], (uint32_t)(st.last[i] / S) & 1u, a.status, 100000000LL);
}

namespace {

int rows_nb(int B) { return (B < 64 ? B + 7 : 64) / 8; }

size_t rows_smem(int NB, int S, int classes, int K) {
    return (size_t)S * (kRwGroups * 512 + 2048 * NB) + (size_t)16 * 128 * NB * 4 + (size_t)classes * 256 * NB * 4 +
           (size_t)K / 64 * 2 + 16;
}

int rows_stages(const LinearArgs& a, const DeviceInfo& dev, int n0) {
    const int nks = (a.K + 1023) / 1024, classes = n0 > 0 ? std::min(8, n0) + std::min(8, nks - n0) : std::min(8, nks);
    const size_t limit = (size_t)dev.max_smem_optin - sizeof(RowsState) - 256;
    for (int S = kRwMaxStages; S >= 2; --S)
        if (rows_smem(rows_nb(a.B), S, classes, a.K) <= limit) return S;
    return 0;
}

template <int NB>
cudaError_t launch_nb(const LinearArgs& a, const float* xs, int S, int n0, const DeviceInfo& dev, cudaStream_t st) {
    const int nks = (a.K + 1023) / 1024, classes = n0 > 0 ? std::min(8, n0) + std::min(8, nks - n0) : std::min(8, nks);
    const int GM = (a.M + kGroupRows - 1) / kGroupRows;
    const dim3 grid(GM < dev.num_sms ? GM : dev.num_sms, (a.B + 8 * NB - 1) / (8 * NB));
    return launch_k(linear_rows_kernel<NB>, grid, dim3(kRwThreads), rows_smem(NB, S, classes, a.K), st, a.pdl, a, xs, S, n0);
}

}  // namespace

size_t linear_rows_bytes(int K, int B) {
    const int RT = 8 * rows_nb(B);
    return (size_t)((B + RT - 1) / RT) * RT * K * sizeof(float);
}

bool linear_rows_ok(const LinearArgs& a, const DeviceInfo& dev) {
    if (a.K % 64 || (size_t)a.K * 2 * sizeof(float) > (size_t)dev.max_smem_optin - 1024) return false;
    const int n0 = linear_stream_passes(a, dev);
    if (n0 > 0) {
        // With few groups per CTA a warp of the streaming kernel can end its first pass in the
        // group its second pass begins with, and then runs one chain over both: not this
        // kernel's tree. Its items are warp, warp + 8, ..: the first pass's, then the second's.
        const int GM = (a.M + kGroupRows - 1) / kGroupRows, grid = GM < dev.num_sms ? GM : dev.num_sms;
        const int n1 = (a.K + 1023) / 1024 - n0;
        for (int ng = GM / grid; ng <= (GM + grid - 1) / grid; ++ng)  // groups of a CTA
            for (int w = 0; w < kWarps; ++w) {
                const int items0 = ng * n0, next = items0 + ((w - items0) & 7), last = next - 8;
                if (last >= 0 && next < ng * (n0 + n1) && last / n0 == (next - items0) / n1) return false;
            }
    }
    return rows_stages(a, dev, n0) >= 2;
}

// Issue slots of a 64-column step (NB batch rows per lane: ~24 NB of multiply-adds and their
// loads, ~130 of widening, ring and class overhead) at the measured ~62 % issue rate, or the
// weight stream, plus the second launch
float linear_rows_us(int M, int K, int B, const DeviceInfo& dev) {
    const float nb = (float)rows_nb(B), tiles = (float)((B + 63) / 64);
    const float steps = (float)M / 32.f * (float)K / 64.f * tiles / (float)dev.num_sms;
    const float issue = steps * 4.f * (24.f * nb + 130.f) / 0.62f / 1.95e3f;
    const float mem = 2.f * (float)M * (float)K * tiles / 6.0e6f;
    return (issue > mem ? issue : mem) + 8.f;
}

cudaError_t linear_rows_prepare(const DeviceInfo& dev) {
    cudaError_t e = cudaFuncSetAttribute(xrows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dev.max_smem_optin - 1024);
    const int lim = dev.max_smem_optin - (int)sizeof(RowsState) - 256;
    for (auto k : {linear_rows_kernel<1>, linear_rows_kernel<2>, linear_rows_kernel<3>, linear_rows_kernel<4>,
                   linear_rows_kernel<5>, linear_rows_kernel<6>, linear_rows_kernel<7>, linear_rows_kernel<8>})
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    return e;
}

cudaError_t launch_linear_rows(const LinearArgs& a, float* xs, const DeviceInfo& dev, cudaStream_t st,
                               cudaEvent_t after_prep) {
    const int n0 = linear_stream_passes(a, dev), S = rows_stages(a, dev, n0), NB = rows_nb(a.B);
    if (!a.tiles_sw || !linear_rows_ok(a, dev)) return cudaErrorInvalidValue;
    cudaError_t e = launch_k(xrows_kernel, dim3((a.B + 1) / 2), dim3(kStreamThreads, 2),
                             (size_t)a.K * 2 * sizeof(float), st, a.pdl, a,
                             8 * NB, xs);
    if (e != cudaSuccess) return e;
    if (after_prep && (e = cudaEventRecord(after_prep, st)) != cudaSuccess) return e;
    switch (NB) {
        case 1: return launch_nb<1>(a, xs, S, n0, dev, st);
        case 2: return launch_nb<2>(a, xs, S, n0, dev, st);
        case 3: return launch_nb<3>(a, xs, S, n0, dev, st);
        case 4: return launch_nb<4>(a, xs, S, n0, dev, st);
        case 5: return launch_nb<5>(a, xs, S, n0, dev, st);
        case 6: return launch_nb<6>(a, xs, S, n0, dev, st);
        case 7: return launch_nb<7>(a, xs, S, n0, dev, st);
        default: return launch_nb<8>(a, xs, S, n0, dev, st);
    }
}

}  // namespace fe
