// Per-iteration centroid preparation.
//  RBQ1 (Section 3.1 "RabitQ"): the centroid residual rho = c - m is
//  re-encoded with per-centroid SQ4 (b = min rho, s = (max rho - b)/15,
//  s = 1 when flat, ybar = clip(rint((rho - b)/s), 0, 15)) and stored as four
//  bit planes per 32-dimension word, so that sum_i xbar_i ybar_i =
//  sum_j 2^j popc(xbar & plane_j), and/or as e4m3 bytes for the tensor kernel.
//  ||rho||^2 is summed in fp64 in the library's blocked pairwise order.
//  SQ8: per-row sums of squared codes (exact int32).
#include "skm_internal.cuh"

namespace skm {

// One warp per centroid.  rho = c - m is kept in the warp's slice of shared
// memory; min/max and the code sum are exact warp reductions, the codes of
// 32 consecutive dimensions become four bit planes through __ballot_sync, and
// ||rho||^2 is summed in fp64 pairwise inside each 32-dimension block (xor
// butterfly 16, 8, 4, 2, 1) with the block sums added in order.
//
// The fp64 instructions bound this kernel (two lanes a clock and SM), so none
// is spent on a value another lane has too: CPREP_GROUP blocks go through the
// butterfly together, each exchange halving the blocks a lane still carries (9
// additions for 8 blocks instead of 40; a + b = b + a, so every block's sum is
// the butterfly's), and one warp adds up the block sums of the CTA's centroids
// side by side.  k = 4000, d = 768: 58 us before.
constexpr int CPREP_WARPS = 4;
constexpr int CPREP_GROUP = 8;

// One column's terms into its pair record (see CodePairs)
__device__ __forceinline__ void put_rbq1_pair(const CodePairs &pairs, int j, float bd, float sd, float q, float ny2) {
    float *bs = reinterpret_cast<float *>(pairs.bs + (j >> 1)) + (j & 1);
    float *qn = reinterpret_cast<float *>(pairs.qn + (j >> 1)) + (j & 1);
    bs[0] = bd;
    bs[2] = sd;
    qn[0] = q;
    qn[2] = ny2;
}

// Sums of CPREP_GROUP blocks of 32 values (v[u]: this lane's value of block
// u), each pairwise over the lanes 16, 8, 4, 2, 1 apart; the sum of block
// lane >> 2 is returned.
__device__ __forceinline__ double block_sums8(const double (&v)[CPREP_GROUP], int lane) {
    double a[4], b[2], c;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool up = (lane & 16) != 0;
        a[i] = __dadd_rn(up ? v[4 + i] : v[i], __shfl_xor_sync(0xffffffffu, up ? v[i] : v[4 + i], 16));
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const bool up = (lane & 8) != 0;
        b[i] = __dadd_rn(up ? a[2 + i] : a[i], __shfl_xor_sync(0xffffffffu, up ? a[i] : a[2 + i], 8));
    }
    {
        const bool up = (lane & 4) != 0;
        c = __dadd_rn(up ? b[1] : b[0], __shfl_xor_sync(0xffffffffu, up ? b[0] : b[1], 4));
    }
    c = __dadd_rn(c, __shfl_xor_sync(0xffffffffu, c, 2));
    return __dadd_rn(c, __shfl_xor_sync(0xffffffffu, c, 1));
}

// planes != nullptr: SQ4 codes as four bit planes per word (AND + popcount
// kernel), terms in info; yq != nullptr: the same codes as e4m3 bytes, row
// stride dq (tensor kernel), terms in the column pairs.
__global__ void __launch_bounds__(CPREP_WARPS * 32) rbq1_cprep_kernel(
    const float *__restrict__ C, int k, int d, const float *__restrict__ m,
    uint4 *__restrict__ planes, Rbq1CInfo *__restrict__ info, uint8_t *__restrict__ yq, int dq,
    float isd, const CodePairs pairs) {
    dep_sync();
    extern __shared__ __align__(8) uint8_t sh_prep[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int W = (d + 31) >> 5;
    double *bsum = reinterpret_cast<double *>(sh_prep) + (size_t)warp * W;  // [CPREP_WARPS][W]
    float *rho = reinterpret_cast<float *>(sh_prep + sizeof(double) * CPREP_WARPS * W) + (size_t)warp * d;
    __shared__ Rbq1CInfo terms[CPREP_WARPS];
    if (pairs.counters && blockIdx.x == 0 && threadIdx.x < 4) pairs.counters[threadIdx.x] = 0;
    const int j = blockIdx.x * CPREP_WARPS + warp;
    if (j < k) {  // warp-uniform
        const float *c = C + (int64_t)j * d;
        float lo = INFINITY, hi = -INFINITY;
        for (int i = lane; i < d; i += 32) {
            const float r = __fsub_rn(c[i], m[i]);
            rho[i] = r;
            lo = fminf(lo, r);
            hi = fmaxf(hi, r);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        __syncwarp();
        float sc = __fdiv_rn(__fsub_rn(hi, lo), 15.0f);
        if (!(sc > 0.0f)) sc = 1.0f;
        int32_t sy = 0;
        for (int w0 = 0; w0 < W; w0 += CPREP_GROUP) {
            double sq[CPREP_GROUP];
#pragma unroll
            for (int u = 0; u < CPREP_GROUP; ++u) {
                const int w = w0 + u, i = 32 * w + lane;
                const float r = i < d ? rho[i] : 0.0f;
                sq[u] = w < W ? __dmul_rn((double)r, (double)r) : 0.0;
                if (w >= W) continue;  // warp-uniform
                uint32_t y = 0;
                if (i < d) {
                    float q = rintf(__fdiv_rn(__fsub_rn(r, lo), sc));
                    q = (q >= 0.0f) ? q : 0.0f;
                    q = fminf(q, 15.0f);
                    y = (uint32_t)q;
                    if (yq) yq[(int64_t)j * dq + i] = e4m3_of_code(y);
                }
                sy += (int32_t)y;
                if (planes) {
                    const uint32_t p0 = __ballot_sync(0xffffffffu, y & 1u);
                    const uint32_t p1 = __ballot_sync(0xffffffffu, y & 2u);
                    const uint32_t p2 = __ballot_sync(0xffffffffu, y & 4u);
                    const uint32_t p3 = __ballot_sync(0xffffffffu, y & 8u);
                    if (lane == 0) planes[(int64_t)j * W + w] = make_uint4(p0, p1, p2, p3);
                }
            }
            const double s = block_sums8(sq, lane);
            if ((lane & 3) == 0 && w0 + (lane >> 2) < W) bsum[w0 + (lane >> 2)] = s;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sy += __shfl_xor_sync(0xffffffffu, sy, o);
        if (lane == 0) {
            Rbq1CInfo in;
            in.bd = __fmul_rn(lo, isd);
            in.sd = __fmul_rn(sc, isd);
            in.sumy = sy;
            terms[warp] = in;
        }
    }
    __syncthreads();
    if (warp == 0 && lane < CPREP_WARPS) {
        const int jj = blockIdx.x * CPREP_WARPS + lane;
        if (jj < k) {
            const double *b = bsum + (size_t)lane * W;
            double q2 = 0.0;  // the block sums in order
            for (int w = 0; w < W; ++w) q2 = __dadd_rn(q2, b[w]);
            Rbq1CInfo in = terms[lane];
            in.ny2 = __double2float_rn(q2);
            if (info) info[jj] = in;
            if (pairs.bs) put_rbq1_pair(pairs, jj, in.bd, in.sd, -(float)in.sumy, in.ny2);
        } else if (jj < pairs.kp) {
            put_rbq1_pair(pairs, jj, 0.0f, 0.0f, 0.0f, INFINITY);
        }
    }
}

static cudaError_t launch_cprep_common(const float *C, int k, int d, const float *m, uint4 *planes,
                                       Rbq1CInfo *info, uint8_t *yq, int dq, const CodePairs &pairs, cudaStream_t st) {
    const size_t smem = (size_t)CPREP_WARPS * (words_of(d) * sizeof(double) + d * sizeof(float));
    if (smem > 48 * 1024 - 1024) {
        const cudaError_t e = smem_limit(
            rbq1_cprep_kernel, (size_t)CPREP_WARPS * (words_of(MAX_D) * sizeof(double) + MAX_D * sizeof(float)));
        if (e != cudaSuccess) return e;
    }
    const int rows = k > pairs.kp ? k : pairs.kp;
    launch_dep(rbq1_cprep_kernel, (rows + CPREP_WARPS - 1) / CPREP_WARPS, CPREP_WARPS * 32, smem, st, 
        C, k, d, m, planes, info, yq, dq, rbq1_isd(d), pairs);
    return launched();
}

cudaError_t launch_rbq1_cprep(const float *C, int k, int d, const float *m, uint4 *planes,
                              Rbq1CInfo *info, cudaStream_t st) {
    return launch_cprep_common(C, k, d, m, planes, info, nullptr, 0, CodePairs{}, st);
}

cudaError_t launch_rbq1_cprep_tc(const float *C, int k, int d, const float *m, uint8_t *yq, int dq,
                                 const CodePairs &pairs, cudaStream_t st) {
    return launch_cprep_common(C, k, d, m, nullptr, nullptr, yq, dq, pairs, st);
}

// Symmetric 1-bit variant: the centroid residual rho = c - m binarized like a
// point (bit = rho_i > 0); ||rho||^2 and ||rho||_1 in fp64, pairwise inside
// 32-dimension blocks, blocks in order; fy = fl32((||rho||^2 / ||rho||_1) /
// sqrt(d)) = F_y / d (0 when rho = 0).  Outputs: e4m3 +-1 codes (yq, row
// stride dq) and/or sign words (yw), and info = (bd 0, sd fy, sumy 0, ny2), so
// the tensor epilogue's u = fma(sd, acc, bd pc) is fy (d - 2h).
__global__ void __launch_bounds__(CPREP_WARPS * 32) rbq1_cprep_sym_kernel(
    const float *__restrict__ C, int k, int d, const float *__restrict__ m, uint8_t *__restrict__ yq, int dq,
    uint32_t *__restrict__ yw, Rbq1CInfo *__restrict__ info, const CodePairs pairs) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int j = blockIdx.x * CPREP_WARPS + warp;
    if (pairs.counters && blockIdx.x == 0 && threadIdx.x < 4) pairs.counters[threadIdx.x] = 0;
    if (j >= k) {  // warp-uniform
        if (lane == 0 && j < pairs.kp) put_rbq1_pair(pairs, j, 0.0f, 0.0f, 0.0f, INFINITY);
        return;
    }
    const float *c = C + (int64_t)j * d;
    const int W = (d + 31) >> 5;
    double q2 = 0.0, l1 = 0.0;
    for (int w = 0; w < W; ++w) {
        const int i = 32 * w + lane;
        const float r = (i < d) ? __fsub_rn(c[i], m[i]) : 0.0f;
        double sq = (i < d) ? __dmul_rn((double)r, (double)r) : 0.0;
        double ab = (i < d) ? fabs((double)r) : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sq = __dadd_rn(sq, __shfl_xor_sync(0xffffffffu, sq, o));
            ab = __dadd_rn(ab, __shfl_xor_sync(0xffffffffu, ab, o));
        }
        q2 = __dadd_rn(q2, sq);
        l1 = __dadd_rn(l1, ab);
        const bool bit = (i < d) && r > 0.0f;
        if (yq && i < d) yq[(int64_t)j * dq + i] = bit ? 0x38 : 0xB8;
        const uint32_t word = __ballot_sync(0xffffffffu, bit);
        if (yw && lane == 0) yw[(int64_t)j * W + w] = word;
    }
    if (lane == 0) {
        Rbq1CInfo in;
        in.bd = 0.0f;
        in.sd = (l1 > 0.0) ? __double2float_rn(__ddiv_rn(__ddiv_rn(q2, l1), __dsqrt_rn((double)d))) : 0.0f;
        in.sumy = 0;
        in.ny2 = __double2float_rn(q2);
        if (info) info[j] = in;
        if (pairs.bs) put_rbq1_pair(pairs, j, in.bd, in.sd, 0.0f, in.ny2);
    }
}

cudaError_t launch_rbq1_cprep_sym(const float *C, int k, int d, const float *m, uint8_t *yq, int dq, uint32_t *yw,
                                  Rbq1CInfo *info, const CodePairs &pairs, cudaStream_t st) {
    const int rows = k > pairs.kp ? k : pairs.kp;
    rbq1_cprep_sym_kernel<<<(rows + CPREP_WARPS - 1) / CPREP_WARPS, CPREP_WARPS * 32, 0, st>>>(C, k, d, m, yq, dq, yw,
                                                                                           info, pairs);
    return launched();
}

// sum_i code_i^2 per row (exact, fits int32 for d <= 4096); one warp per row.
__global__ void row_sqnorm_u8_kernel(const uint8_t *__restrict__ codes, int64_t n, int d,
                                     int32_t *__restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t p = warp; p < n; p += nwarps) {
        int32_t s = 0;
        for (int i = lane; i < d; i += 32) {
            const int32_t v = codes[p * d + i];
            s += v * v;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) out[p] = s;
    }
}

cudaError_t launch_row_sqnorm_u8(const uint8_t *codes, int64_t n, int d, int32_t *out,
                                 cudaStream_t st) {
    int64_t blocks = (n * 32 + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (blocks < 1) blocks = 1;
    row_sqnorm_u8_kernel<<<(int)blocks, 256, 0, st>>>(codes, n, d, out);
    return launched();
}

}  // namespace skm
