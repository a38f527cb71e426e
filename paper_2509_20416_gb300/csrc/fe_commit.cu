// The commit step of a cycle (Sec. 2.4, "Update and Iterate"): the runtime (fe_runtime.cu)
// runs Eq. 1 and the cascade over the accepted positions' rows. On the tensor cores with head
// size 128 the plan kernel lists the rows sequence by sequence, so that blocks hold only rows
// that exist, and one attention launch per layer takes every row of a block; otherwise the
// rows of a block of row indices are gathered into a dense batch, with one attention launch
// per row index so that a row reads the rows committed before it from the cache.
#include "fe_kernels.h"
#include "fe_common.cuh"

namespace fe {

// Row r = b * nb + j of the block (j = 0 .. nb - 1, row index i = i0 + j of sequence b):
// its feature row feat[b][i] (row_bytes bytes, 16-byte aligned) and its token; rows at or
// past n_rows[b] take token 0 (their outputs are computed but never stored).
__global__ void __launch_bounds__(128) commit_gather_kernel(const unsigned char* feat, const int* tok,
                                                            const int* n_rows, int L, int i0, int nb,
                                                            int row_bytes, unsigned char* cfeat, int* ctok) {
    const int r = blockIdx.x, b = r / nb, i = i0 + r % nb;
    const uint4* src = reinterpret_cast<const uint4*>(feat + ((size_t)b * L + i) * row_bytes);
    uint4* dst = reinterpret_cast<uint4*>(cfeat + (size_t)r * row_bytes);
    for (int k = threadIdx.x; k < row_bytes / 16; k += blockDim.x) dst[k] = src[k];
    if (threadIdx.x == 0) ctok[r] = i < n_rows[b] ? tok[(size_t)b * L + i] : 0;
}

cudaError_t launch_commit_gather(const void* feat, const int* tok, const int* n_rows, int B, int L, int i0, int nb,
                                 int row_bytes, void* cfeat, int* ctok, cudaStream_t st) {
    if (B < 1 || nb < 1 || row_bytes % 16) return cudaErrorInvalidValue;
    commit_gather_kernel<<<B * nb, 128, 0, st>>>((const unsigned char*)feat, tok, n_rows, L, i0, nb, row_bytes,
                                                 (unsigned char*)cfeat, ctok);
    return cudaGetLastError();
}

// The rows of a whole commit for the multi-row path: one CTA; thread b owns sequence b, b +
// blockDim, ... The first row of sequence b in its block that has a place in the cache decides the
// cached keys all of the block's rows of b share (the rows before it are stored by then), so the
// splits follow it. Rows without a place have no splits; attn_rows_kernel leaves them out by the
// same rule (rows_in_cache).
__global__ void __launch_bounds__(256) commit_plan_kernel(const int* tok, const int* n_rows, const int* prefix_len,
                                                          int B, int L, int block_rows, int split, int max_seq,
                                                          int* off, int* total, int* x_row, int* ctok, int* nact) {
    __shared__ int so[257];
    const int t = threadIdx.x;
    int base = 0;
    for (int b0 = 0; b0 < B; b0 += 256) {
        const int b = b0 + t, n = b < B ? min(max(n_rows[b], 0), L) : 0;
        so[t] = n;
        __syncthreads();
        if (t == 0) {
            int run = base;
            for (int j = 0; j < 256; ++j) {
                const int x = so[j];
                so[j] = run;
                run += x;
            }
            so[256] = run;
        }
        __syncthreads();
        base = so[256];
        if (b < B) {
            const int o = so[t], P = prefix_len[b];
            const int2 in = rows_in_cache(P, n, max_seq);
            off[b] = o;
            for (int i = 0; i < n; ++i) {
                const int r = o + i, first = max(o + in.x, r / block_rows * block_rows) - o;
                x_row[r] = b * L + i;
                ctok[r] = tok[(size_t)b * L + i];
                nact[r] = i >= in.x && i < in.y ? (P + first) / split + 1 : 0;
            }
        }
        __syncthreads();
    }
    if (t == 0) {
        off[B] = base;
        *total = base;
    }
}

cudaError_t launch_commit_plan(const int* tok, const int* n_rows, const int* prefix_len, int B, int L, int block_rows,
                               int split, int max_seq, int* off, int* total, int* x_row, int* ctok, int* nact,
                               cudaStream_t st) {
    commit_plan_kernel<<<1, 256, 0, st>>>(tok, n_rows, prefix_len, B, L, block_rows, split, max_seq, off, total, x_row,
                                          ctok, nact);
    return cudaGetLastError();
}

}  // namespace fe
