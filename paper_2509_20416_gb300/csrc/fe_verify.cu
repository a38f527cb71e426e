// Lossless verification of a sampled draft tree (Sec. 2.4: the target scores the tree with
// tree attention and speculative sampling finds the longest accepted path; the paper names
// no variant). Read as recursive rejection sampling over each node's children in draw order
// (the multi-candidate form of speculative sampling: Leviathan et al. and Chen et al. 2023;
// Jeon et al. 2024), matching candidates drawn without replacement (Sec. 2.2):
//
//   at the current node, with r = the target's next-token distribution there and s = the
//   drafter's proposal of the next depth, the children are tested in draw order; child c
//   with token x is accepted iff u_acc[c] * s(x) <= r(x) (probability min(1, r(x) / s(x)));
//   on rejection r <- max(r - s, 0) renormalised and x leaves s (s renormalised over the
//   tokens not yet drawn: the law of the next draw). An accepted child becomes the current
//   node and r its own target distribution. When all children are rejected, or the node has
//   none, or N tokens were accepted, the bonus token is drawn from r by inverse CDF: the
//   smallest x with u_bonus[current] < r(0) + ... + r(x) (the last token with r > 0 when
//   rounding leaves the total below u).
//
// Two kernels. verify_cluster_kernel (vocabularies up to 131072 entries) spreads a sequence
// over a cluster of up to 8 CTAs and keeps r and q in registers; it is described there. The
// other keeps r in memory:
//
// One CTA of 512 threads per sequence. s needs no buffer: after the draws X so far it is
// q / (1 - q(X)) off X and 0 on X. r is kept as an unnormalised residual w in a per-sequence
// buffer with its sum Z (r = w / Z), so a rejection is one pass over the vocabulary (read w
// or p and q, write the new w, sum it); the up to k - 1 tokens already drawn, whose s is 0,
// are put back after the pass from values saved before it. Every thread walks the tree with
// the same values (broadcast loads, a deterministic block sum), so the decisions agree.
// Precision: the elementwise residual is float32 (one rounding per operation); the sums
// that set the scale of everything after them -- each thread's share of Z (compensated),
// the block total and q's drawn mass, the CDF of the bonus draw -- are carried in double,
// so that their error does not grow with V.
#include <float.h>
#include <limits.h>

#include "fe_common.cuh"
#include "fe_kernels.h"

namespace fe {

namespace {

constexpr int kVsThreads = 512;
constexpr int kVsWarps = kVsThreads / 32;
constexpr int kVsMaxKids = 32;

// sum of one value per thread in double, the same bits in every thread (fixed order)
__device__ __forceinline__ double block_sum(double v, double* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kVsWarps; ++w) s += red[w];
    __syncthreads();
    return s;
}

// compensated (Kahan) float accumulation: the sum's error stays near one rounding
struct KahanF {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float y = x - c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

__global__ void __launch_bounds__(kVsThreads) verify_sampled_kernel(const VerifySampledArgs a) {
    const int b = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int T = a.T, N = a.N, V = a.V;
    __shared__ int kids[kVsMaxKids];
    __shared__ int nkids;
    __shared__ double red[kVsWarps];
    __shared__ int rem_tok[kVsMaxKids];   // tokens drawn (and rejected) at this node so far
    __shared__ float saved[kVsMaxKids];   // their r before a pass
    __shared__ double chunk_sum[kVsThreads];
    __shared__ int pick_s, last_s;
    const int* tk = a.tok + (size_t)b * T;
    const int* pr = a.parent + (size_t)b * T;
    const int* dp = a.depth + (size_t)b * T;
    const int* rk = a.rank + (size_t)b * (T - 1);  // node c >= 1 -> rk[c - 1]
    float* w = a.rbuf + (size_t)b * V;
    int cur = 0, n = 0;
    bool from_p = true;  // r is p[b][cur] itself; else r = w / Z
    double Z = 1.0;
    const float* pcur = a.p + (size_t)b * T * V;
    bool bad = false;

    for (;;) {
        // ---- the children of cur, in draw order (warp 0)
        if (warp == 0) {
            int m = 0;
            for (int c0 = 1; c0 < T; c0 += 32) {
                const int c = c0 + lane;
                const bool is = c < T && pr[c] == cur;
                const unsigned bal = __ballot_sync(0xffffffffu, is);
                const int pos = m + __popc(bal & ((1u << lane) - 1u));
                if (is && pos < kVsMaxKids) kids[pos] = c;
                m += __popc(bal);
            }
            m = min(m, kVsMaxKids);
            __syncwarp();
            const int c = lane < m ? kids[lane] : -1;
            const int rc = lane < m ? rk[c - 1] : INT_MAX;
            int place = 0;
            for (int j = 0; j < m; ++j) {
                const int rj = __shfl_sync(0xffffffffu, rc, j), cj = __shfl_sync(0xffffffffu, c, j);
                if (j != lane && (rj < rc || (rj == rc && cj < c))) ++place;
            }
            __syncwarp();
            if (lane < m) kids[place] = c;
            if (lane == 0) nkids = m;
        }
        __syncthreads();
        const int m = nkids;
        if (m == 0 || n >= N) break;
        const int dcur = dp[cur];
        if (dcur < 0 || dcur >= N) {
            bad = true;
            break;
        }
        const float* qs = a.q + ((size_t)b * N + dcur) * V;
        double removed = 0.0;  // q mass of the tokens drawn so far at this node
        int nrem = 0;
        int next = -1;
        for (int i = 0; i < m; ++i) {
            const int c = kids[i], x = tk[c];
            if (x < 0 || x >= V) {
                bad = true;
                break;
            }
            const float inv = removed < 1.0 ? (float)(1.0 / (1.0 - removed)) : 0.f;
            const float invZ = Z > 0.0 ? (float)(1.0 / Z) : 0.f;
            const float sx = qs[x] * inv;
            const float rx = from_p ? pcur[x] : w[x] * invZ;
            if (a.u_acc[(size_t)b * T + c] * sx <= rx) {
                next = c;
                break;
            }
            // rejected: r <- max(r - s, 0) (renormalised through Z); x leaves s
            if (t < nrem) {
                const int v = rem_tok[t];
                saved[t] = from_p ? pcur[v] : w[v] * invZ;
            }
            __syncthreads();
            KahanF part;
            for (int v = t; v < V; v += kVsThreads) {
                const float rv = from_p ? pcur[v] : w[v] * invZ;
                const float nv = fmaxf(rv - qs[v] * inv, 0.f);
                w[v] = nv;
                part.add(nv);
            }
            double sum = block_sum(part.value(), red);
            // the tokens drawn before x have s = 0: their r stays
            for (int j = 0; j < nrem; ++j) {
                const float sj = saved[j];
                sum += (double)sj - (double)fmaxf(sj - qs[rem_tok[j]] * inv, 0.f);
            }
            if (t < nrem) w[rem_tok[t]] = saved[t];
            Z = sum;
            from_p = false;
            __syncthreads();  // everyone has read rem_tok / saved; the fix-ups are written
            if (t == 0) rem_tok[nrem] = x;
            removed += (double)qs[x];
            ++nrem;
            __syncthreads();
        }
        if (next < 0) break;  // every child rejected (or a malformed node)
        if (t == 0) a.path[(size_t)b * N + n] = next;
        ++n;
        cur = next;
        from_p = true;
        Z = 1.0;
        pcur = a.p + ((size_t)b * T + cur) * V;
        __syncthreads();  // kids[] is rebuilt for the new node
    }
    if (bad && t == 0) atomicOr(a.status, ST_DEVICE);

    // ---- the bonus token: inverse CDF of r. Thread t sums a contiguous chunk; the chunks'
    // prefix gives each its start; the first chunk whose running sum passes u holds it.
    const double u = a.u_bonus[(size_t)b * T + cur];
    const float invZ = Z > 0.0 ? (float)(1.0 / Z) : 0.f;
    const int chunk = (V + kVsThreads - 1) / kVsThreads;
    const int v0 = min(V, t * chunk), v1 = min(V, v0 + chunk);
    double cs = 0.0;
    int last = -1;
    for (int v = v0; v < v1; ++v) {
        const float rv = from_p ? pcur[v] : w[v] * invZ;
        cs += (double)rv;
        if (rv > 0.f) last = v;
    }
    chunk_sum[t] = cs;
    if (t == 0) {
        pick_s = INT_MAX;
        last_s = -1;
    }
    __syncthreads();
    if (t == 0) {  // exclusive prefix of the chunk sums, in chunk order
        double run = 0.0;
        for (int j = 0; j < kVsThreads; ++j) {
            const double cj = chunk_sum[j];
            chunk_sum[j] = run;
            run += cj;
        }
    }
    if (last >= 0) atomicMax(&last_s, last);
    __syncthreads();
    double run = chunk_sum[t];
    for (int v = v0; v < v1; ++v) {
        run += (double)(from_p ? pcur[v] : w[v] * invZ);
        if (u < run) {
            atomicMin(&pick_s, v);
            break;
        }
    }
    __syncthreads();
    for (int i = n + t; i < N; i += kVsThreads) a.path[(size_t)b * N + i] = -1;
    if (t == 0) {
        a.n_accept[b] = n;
        a.bonus[b] = pick_s != INT_MAX ? pick_s : max(last_s, 0);
    }
}

// ---- the cluster kernel ------------------------------------------------------------------
// One cluster of C CTAs (1 or 8) x 512 threads per sequence. The walk is a chain of passes
// over the vocabulary (one per rejection) and of decisions that need each pass's total, so it
// is bound by the latency of a pass: one CTA took ~10 us for 128 K entries (L2 reads and
// writes of the residual, and double additions, which this GPU issues at 1/64 rate). Here
// thread t of CTA c holds entries c S + 512 e + t (e < E) of the current residual w and of
// the proposal q in registers, loaded once per node, so a pass is E fused multiply-adds per
// thread and one exchange: every warp sends its partial total to every CTA through
// distributed shared memory (st.async, completing on the receiver's mbarrier) and sums all of
// them itself. Every warp takes every decision itself, too, from the same values, with child j
// of the node on its lane j; there is no other synchronisation in the walk. Elementwise
// arithmetic is verify_sampled_kernel's; a token that was drawn leaves s by zeroing its owner's
// q. The sums (double there):
//   - Z: compensated float shares of E entries, added as float pairs (2^-48; the shares there,
//     of V / 512 entries, are the larger error of the two);
//   - the drawn mass and the CDF of the bonus draw: 64-bit fixed point in units of 2^-62, which
//     holds a float32 of 2^-39 or more exactly (smaller ones to a unit). Integer sums do not
//     depend on their order, so the totals of CTAs, segments and entries agree to the last
//     bit and the draw never falls between two of them.
// 4 sequences, 128256 entries, 6 levels x 8 candidates: 324 us on one CTA each; here 28 us with
// the totals added in double by one warp between CTA barriers, 25 with every total a float pair
// (whose CDF could pick an entry next to its own, even one of probability 0, when the deviate
// lay within 2^-48 of a CDF edge), as much in fixed point (four seeds, one box: 26.6, 26.6, 31.4,
// 29.4 us in pairs, 25.9, 25.9, 31.1, 28.7 in fixed point).
struct FF {  // an unevaluated sum of two floats
    float h = 0.f, l = 0.f;
};

__device__ __forceinline__ FF ff_add(FF a, FF b) {
    const float s = a.h + b.h, t = s - a.h;
    const float e = (a.h - (s - t)) + (b.h - t) + (a.l + b.l);
    FF r;
    r.h = s + e;
    r.l = e - (r.h - s);
    return r;
}

__device__ __forceinline__ FF ff_shfl_xor(FF a, int o) {
    FF r;
    r.h = __shfl_xor_sync(0xffffffffu, a.h, o);
    r.l = __shfl_xor_sync(0xffffffffu, a.l, o);
    return r;
}

// A probability in units of 2^-62, rounded down: its 24 bits shifted to their place. Taken into
// [0, 2) first (0 for a NaN); sums saturate (one of 2 or more is above every deviate).
using fx64 = unsigned long long;
constexpr fx64 kFxOne = 1ull << 62;

__device__ __forceinline__ float fx_clamp(float w) { return fminf(fmaxf(w, 0.f), 1.9999999f); }

__device__ __forceinline__ fx64 fx(float w) {
    const uint32_t u = __float_as_uint(fx_clamp(w));
    fx64 r;  // (shr clamps its count: 0 from 64 on)
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"((fx64)((u & 0x7fffffu) | 0x800000u) << 39), "r"(127u - (u >> 23)));
    return r;
}

__device__ __forceinline__ fx64 fx_add(fx64 a, fx64 b) { return a + b < a ? ~0ull : a + b; }

// 1 / (a 2^-62), 0 < a <= kFxOne, rounded once from a remainder known to ~2^-48: a = M 2^(64 - s) with
// M in [1/2, 1) split into 24 + 24 + 16 bits, and the remainder of the first part's reciprocal
// is exact. (Conversions of 32-bit words: those of 64-bit ones run at a fraction of the rate, and
// every warp forms this for every rejection.)
__device__ __forceinline__ float fx_rcp(fx64 a) {
    const int s = __clzll((long long)a);
    const fx64 m = a << s;
    const float h = __uint2float_rn((uint32_t)(m >> 40)) * 0x1p-24f;
    const float l = __uint2float_rn((uint32_t)(m >> 16) & 0xffffffu) * 0x1p-48f;
    const float l2 = __uint2float_rn((uint32_t)m & 0xffffu) * 0x1p-64f;
    const float r = __frcp_rn(h);
    const float q = fmaf(r, fmaf(-r, l2, fmaf(-r, l, fmaf(-r, h, 1.f))), r);
    return q * __uint_as_float((uint32_t)(s - 2 + 127) << 23);  // (a 2^-62 = M 2^(2 - s))
}

// Transposing warp reduction: afterwards lane l holds, in v[0], the warp-wide sum of value
// l >> (5 - log2 E).
template <int N, int O>
__device__ __forceinline__ void fx_multi_sum(fx64* v, int lane) {
    if constexpr (N > 1) {
        const bool upper = (lane & O) != 0;
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            const fx64 send = upper ? v[i] : v[i + N / 2], keep = upper ? v[i + N / 2] : v[i];
            v[i] = fx_add(keep, __shfl_xor_sync(0xffffffffu, send, O));
        }
        fx_multi_sum<N / 2, O / 2>(v, lane);
    } else {
#pragma unroll
        for (int o = O; o >= 1; o >>= 1) v[0] = fx_add(v[0], __shfl_xor_sync(0xffffffffu, v[0], o));
    }
}

constexpr int kVsMaxCtas = 8;
constexpr int kVsMaxTree = 1 + 16 * 32;  // n_layers <= 16, top_k <= 32

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// every thread of every CTA of the cluster (hardware barrier; all of them get here, since no
// other wait of the kernel is unbounded)
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// 16 bytes into CTA `rank`'s copy of `slot`, completing on its copy of `bar`
__device__ __forceinline__ void st_async16(void* slot, uint64_t* bar, uint32_t rank, uint32_t x, uint32_t y, int z) {
    uint32_t rs, rb;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rs) : "r"(smem_u32(slot)), "r"(rank));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(smem_u32(bar)), "r"(rank));
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(rs),
                 "r"(x), "r"(y), "r"(z), "r"(0), "r"(rb)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// 1 / a rounded to float (the remainder of the float reciprocal is taken from both words)
__device__ __forceinline__ float ff_rcp(FF a) {
    const float r = __frcp_rn(a.h);
    return fmaf(r, fmaf(-r, a.l, fmaf(-r, a.h, 1.f)), r);
}

template <int E>
__global__ void __launch_bounds__(kVsThreads) verify_cluster_kernel(const VerifySampledArgs a, int C, int S) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int b = blockIdx.x / C, c = (int)cluster_rank();
    const int T = a.T, N = a.N, V = a.V;
    __shared__ int s_tok[kVsMaxTree], s_par[kVsMaxTree], s_dep[kVsMaxTree], s_rk[kVsMaxTree];
    __shared__ int s_kids[kVsWarps][kVsMaxKids];  // each warp's list of a node's children
    // partial totals by exchange: a float pair's words, or a fixed-point sum's and the last entry > 0
    __shared__ __align__(16) uint4 slots[2][kVsMaxCtas * kVsWarps];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ fx64 seg[E * kVsWarps];  // the bonus draw: sums of 32 consecutive entries
    __shared__ int s_seg;
    __shared__ fx64 s_before;

    if (t == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_fence_init();
    }
    for (int i = t; i < T; i += kVsThreads) {
        s_tok[i] = a.tok[(size_t)b * T + i];
        s_par[i] = a.parent[(size_t)b * T + i];
        s_dep[i] = a.depth[(size_t)b * T + i];
        s_rk[i] = i > 0 ? a.rank[(size_t)b * (T - 1) + i - 1] : 0;
    }
    cluster_sync();  // (also a CTA barrier) every CTA's barriers are ready for remote arrivals

    // Sends this warp's part (the same in all lanes) to every CTA and waits for all of them: each
    // warp then finds the partial of warp w of CTA j in its CTA's slots[x & 1][16 j + w]. Two sets of slots and barriers
    // alternate: exchange x + 2 reaches a CTA only after all of its warps, having read x, have
    // sent x + 1. False when the bounded wait ran out.
    int xch = 0;
    bool ok = true;
    auto send = [&](uint32_t lo, uint32_t hi, int last) {
        const int p = xch & 1;
        if (t == 0) mbar_arrive_expect_tx(&bar[p], 16u * kVsWarps * (uint32_t)C);
        if (lane < C) st_async16(&slots[p][c * kVsWarps + warp], &bar[p], (uint32_t)lane, lo, hi, last);
        if (!mbar_try_wait_cluster(&bar[p], (uint32_t)(xch >> 1) & 1u)) {
            const uint64_t t0 = globaltimer_ns();
            while (!mbar_try_wait_cluster(&bar[p], (uint32_t)(xch >> 1) & 1u))
                if ((int64_t)(globaltimer_ns() - t0) > kWaitBudgetNs) {
                    ok = false;
                    break;
                }
        }
        ok = __all_sync(0xffffffffu, ok);
        ++xch;
    };

    int cur = 0, n = 0;
    bool from_p = true;  // r is w itself; else r = w / Z
    float invZ = 1.f;
    bool bad = false;
    float w[E], q[E];
    for (;;) {
        const int dcur = s_dep[cur];
        const bool deeper = n < N && dcur >= 0 && dcur < N;
        // this node's distribution and the proposal of the next depth; consumed after the
        // children's own loads, so that the round trips overlap
        const float* pc = a.p + ((size_t)b * T + cur) * V;
        const float* qc = a.q + ((size_t)b * N + (deeper ? dcur : 0)) * V;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int i = e * kVsThreads + t, v = c * S + i;
            const bool in = i < S && v < V;
            w[e] = in ? __ldg(pc + v) : 0.f;
            q[e] = in && deeper ? __ldg(qc + v) : 0.f;
        }
        // ---- the children of cur, in draw order: child j on lane j
        int m = 0;
        for (int c0 = 1; c0 < T; c0 += 32) {
            const int i = c0 + lane;
            const bool is = i < T && s_par[i] == cur;
            const unsigned bal = __ballot_sync(0xffffffffu, is);
            const int pos = m + __popc(bal & ((1u << lane) - 1u));
            if (is && pos < kVsMaxKids) s_kids[warp][pos] = i;
            m += __popc(bal);
        }
        m = min(m, kVsMaxKids);
        if (m == 0 || n >= N) break;
        if (!deeper) {
            bad = true;
            break;
        }
        __syncwarp();
        const int mine = lane < m ? s_kids[warp][lane] : -1;
        const int rc = lane < m ? s_rk[mine] : INT_MAX;
        int place = 0;
        for (int j = 0; j < m; ++j) {
            const int rj = __shfl_sync(0xffffffffu, rc, j), cj = __shfl_sync(0xffffffffu, mine, j);
            if (j != lane && (rj < rc || (rj == rc && cj < mine))) ++place;
        }
        __syncwarp();
        if (lane < m) s_kids[warp][place] = mine;
        __syncwarp();
        const int kid = lane < m ? s_kids[warp][lane] : 0;
        const int kx = s_tok[kid];  // its token, and q, the residual and the deviate there
        const bool in = lane < m && kx >= 0 && kx < V;
        const float kq = in ? __ldg(qc + kx) : 0.f;
        float kw = in ? __ldg(pc + kx) : 0.f;
        const float ku = lane < m ? a.u_acc[(size_t)b * T + kid] : 0.f;
        __syncwarp();  // (s_kids is rewritten at the next node)

        fx64 left = kFxOne;  // 1 - the q mass of the tokens drawn so far at this node
        float inv = 1.f;
        int next = -1;
        for (int i = 0; i < m; ++i) {
            const int x = __shfl_sync(0xffffffffu, kx, i);
            if (x < 0 || x >= V) {
                bad = true;
                break;
            }
            const float rw = from_p ? kw : __fmul_rn(kw, invZ);
            const bool accept = __fmul_rn(ku, __fmul_rn(kq, inv)) <= rw;
            if ((__ballot_sync(0xffffffffu, accept) >> i) & 1u) {
                next = __shfl_sync(0xffffffffu, kid, i);
                break;
            }
            // rejected: r <- max(r - s, 0) (renormalised through Z); x leaves s
            KahanF part[4];
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const float rv = from_p ? w[e] : __fmul_rn(w[e], invZ);
                w[e] = fmaxf(fmaf(-q[e], inv, rv), 0.f);
                part[e & 3].add(w[e]);
            }
            const int xi = x - c * S;  // x's owner
            if (xi >= 0 && xi < S && xi % kVsThreads == t) {
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (e == xi / kVsThreads) q[e] = 0.f;
            }
            // the children's own residuals (those drawn before i have s = 0)
            kw = lane < i ? rw : fmaxf(fmaf(-kq, inv, rw), 0.f);
            FF ps[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                ps[u].h = part[u].s;
                ps[u].l = -part[u].c;
            }
            FF Z = ff_add(ff_add(ps[0], ps[1]), ff_add(ps[2], ps[3]));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) Z = ff_add(Z, ff_shfl_xor(Z, o));
            const float drop = __shfl_sync(0xffffffffu, kq, i);
            left = drop < 2.f ? left - min(left, fx(drop)) : 0ull;  // (no proposal: nothing is left)
            inv = left ? fx_rcp(left) : 0.f;
            send(__float_as_uint(Z.h), __float_as_uint(Z.l), -1);
            if (!ok) break;
            Z = FF{};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = 4 * lane + u;
                if (j < C * kVsWarps) {
                    const uint4 x = slots[(xch - 1) & 1][j];
                    FF y;
                    y.h = __uint_as_float(x.x);
                    y.l = __uint_as_float(x.y);
                    Z = ff_add(Z, y);
                }
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) Z = ff_add(Z, ff_shfl_xor(Z, o));
            invZ = Z.h > 0.f ? ff_rcp(Z) : 0.f;
            from_p = false;
        }
        if (next < 0) break;  // every child rejected (or a malformed node)
        if (c == 0 && t == 0) a.path[(size_t)b * N + n] = next;
        ++n;
        cur = next;
        from_p = true;
        invZ = 1.f;
    }
    if (bad && c == 0 && t == 0) atomicOr(a.status, ST_DEVICE);

    // ---- the bonus token: inverse CDF of r. The CTAs' totals name the CTA that holds it, the
    // sums of its 32-entry segments the segment, a warp scan the entry.
    const float uf = a.u_bonus[(size_t)b * T + cur];
    const fx64 u = uf < 2.f ? fx(uf) : ~0ull;  // (u < a sum exactly when the deviate is below it)
    fx64 mass = 0;
    float about = 0.f;
    int last = -1;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        if (!from_p) w[e] = __fmul_rn(w[e], invZ);
        mass += fx(w[e]);
        about += fx_clamp(w[e]);
        if (w[e] > 0.f) last = c * S + e * kVsThreads + t;
    }
    if (about >= 3.f) mass = ~0ull;  // (may have wrapped at 4; no deviate is between)
    int owner = -1, all_last = -1;
    fx64 prefix = 0;  // the total of the CTAs before this one
    if (ok) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            mass = fx_add(mass, __shfl_xor_sync(0xffffffffu, mass, o));
            last = max(last, __shfl_xor_sync(0xffffffffu, last, o));
        }
        send((uint32_t)mass, (uint32_t)(mass >> 32), last);
        fx64 run = 0;  // inclusive over CTAs: lanes 4 j .. 4 j + 3
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = 4 * lane + k;
            if (i < C * kVsWarps) {
                const uint4 x = slots[(xch - 1) & 1][i];
                run = fx_add(run, (fx64)x.y << 32 | x.x);
                all_last = max(all_last, (int)x.z);
            }
        }
        run = fx_add(run, __shfl_xor_sync(0xffffffffu, run, 1));
        run = fx_add(run, __shfl_xor_sync(0xffffffffu, run, 2));
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            const fx64 up = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run = fx_add(up, run);
        }
        const unsigned hit = __ballot_sync(0xffffffffu, u < run && lane % 4 == 0 && lane / 4 < C);
        owner = hit ? (__ffs(hit) - 1) / 4 : -1;
        prefix = __shfl_sync(0xffffffffu, run, max(4 * c - 4, 0));
        if (c == 0) prefix = 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) all_last = max(all_last, __shfl_xor_sync(0xffffffffu, all_last, o));
    }
    if (!ok && t == 0) atomicOr(a.status, ST_TIMEOUT);
    for (int i = n + t; i < N && c == 0; i += kVsThreads) a.path[(size_t)b * N + i] = -1;
    if (c == 0 && t == 0) {
        a.n_accept[b] = n;
        if (!ok || owner < 0) a.bonus[b] = max(all_last, 0);
    }
    if (!__syncthreads_or(!ok) && owner == c) {  // (one segment, and one entry of it, passes u)
        // the transposing reduction's first step forms the units again, two by two: held since
        // above they would spill
        fx64 v[E / 2];
#pragma unroll
        for (int e = 0; e < E / 2; ++e) {
            asm volatile("" : "+f"(w[e]), "+f"(w[e + E / 2]));
            const fx64 x = fx(w[e]), y = fx(w[e + E / 2]);
            v[e] = fx_add(lane & 16 ? y : x, __shfl_xor_sync(0xffffffffu, lane & 16 ? x : y, 16));
        }
        fx_multi_sum<E / 2, 8>(v, lane);
        constexpr int LG = 32 / E;  // lanes that hold the same sum
        if (lane % LG == 0) seg[(lane / LG) * kVsWarps + warp] = v[0];
        __syncthreads();
        if (warp == 0) {  // lane l scans segments [l E / 2, (l + 1) E / 2)
            constexpr int PL = E * kVsWarps / 32;
            fx64 sum = 0;
#pragma unroll
            for (int j = 0; j < PL; ++j) sum = fx_add(sum, seg[lane * PL + j]);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const fx64 up = __shfl_up_sync(0xffffffffu, sum, o);
                if (lane >= o) sum = fx_add(up, sum);
            }
            const fx64 inc = fx_add(prefix, sum);
            const fx64 before = __shfl_up_sync(0xffffffffu, inc, 1);
            const unsigned hit = __ballot_sync(0xffffffffu, u < inc);
            if (hit && lane == __ffs(hit) - 1) {
                fx64 run = lane ? before : prefix;
                int j = 0;
                for (; j + 1 < PL; ++j) {
                    const fx64 nx = fx_add(run, seg[lane * PL + j]);
                    if (u < nx) break;
                    run = nx;
                }
                s_seg = lane * PL + j;
                s_before = run;
            }
        }
        __syncthreads();
        if (warp == s_seg % kVsWarps) {
            const int es = s_seg / kVsWarps;
            float mine = 0.f;
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (e == es) mine = w[e];
            fx64 inc = fx_add(lane == 0 ? s_before : 0ull, fx(mine));
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const fx64 up = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc = fx_add(up, inc);
            }
            const unsigned hit = __ballot_sync(0xffffffffu, u < inc);
            if (hit && lane == 0) a.bonus[b] = c * S + es * kVsThreads + warp * 32 + __ffs(hit) - 1;
        }
    }
    cluster_sync();  // no CTA leaves while another may still write its shared memory
}

template <int E>
cudaError_t launch_cluster(const VerifySampledArgs& a, int B, int C, cudaStream_t st) {
    const int S = (a.V + C * kVsThreads - 1) / (C * kVsThreads) * kVsThreads;  // entries per CTA
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(B * C);
    cfg.blockDim = dim3(kVsThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, verify_cluster_kernel<E>, a, C, S);
}

}  // namespace

cudaError_t launch_verify_sampled(const VerifySampledArgs& a, int B, cudaStream_t st) {
    // entries per thread by the vocabulary: a small one stays in one CTA (no exchange across
    // CTAs), larger ones take 8; beyond 8 x 512 x 32 entries the registers no longer hold it.
    // (A handle's trees have at most kVsMaxTree nodes.)
    static_assert(kVerifyMaxRegV == kVsMaxCtas * kVsThreads * 32);
    if (a.V <= 8 * kVsThreads) return launch_cluster<8>(a, B, 1, st);
    if (a.V <= kVsMaxCtas * kVsThreads * 8) return launch_cluster<8>(a, B, kVsMaxCtas, st);
    if (a.V <= kVsMaxCtas * kVsThreads * 16) return launch_cluster<16>(a, B, kVsMaxCtas, st);
    if (a.V <= kVerifyMaxRegV) return launch_cluster<32>(a, B, kVsMaxCtas, st);
    if (!a.rbuf) return cudaErrorInvalidValue;
    verify_sampled_kernel<<<B, kVsThreads, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace fe
