// Centroid update, Section 2.3 STEP 3 (and the quantized-domain forms of
// Section 3.1): a sort-by-cluster segmented reduction.
//   1. histogram of assignments (shared-memory privatised counters),
//   2. exclusive scan -> per-cluster offsets,
//   3. scatter point ids (and their cluster) into cluster-contiguous order,
//   4. warps take equal runs of the sorted order and flush per-cluster register
//      sums with global atomics (load balanced whatever the cluster sizes);
//      SQ8 rows of no multiple of 16 bytes, or not 16-byte aligned: one CTA
//      per cluster;
//   5. finalise: divide by the counts (or add into caller partial sums).
// Integer representations accumulate in int64 and are exact, so their result
// does not depend on the member order produced by the scatter.
#include <algorithm>

#include "skm_internal.cuh"

namespace skm {

// ---------------------------------------------------------------- histogram
__global__ void histogram_kernel(const int32_t *__restrict__ assign, int64_t n, int k,
                                 int32_t *__restrict__ counts, int use_smem) {
    extern __shared__ int32_t sh[];
    if (use_smem) {
        for (int j = threadIdx.x; j < k; j += blockDim.x) sh[j] = 0;
        __syncthreads();
    }
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int a = assign[t];
        if (a < 0 || a >= k) continue;  // out-of-range assignments are skipped
        if (use_smem)
            atomicAdd(&sh[a], 1);
        else
            atomicAdd(&counts[a], 1);
    }
    if (use_smem) {
        __syncthreads();
        for (int j = threadIdx.x; j < k; j += blockDim.x)
            if (sh[j]) atomicAdd(&counts[j], sh[j]);
    }
}

cudaError_t launch_histogram(const int32_t *assign, int64_t n, int k, int32_t *counts32,
                             cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(counts32, 0, sizeof(int32_t) * (size_t)k, st);
    if (e != cudaSuccess) return e;
    if (n == 0) return cudaSuccess;
    const int use_smem = k <= 12288;
    const size_t smem = use_smem ? sizeof(int32_t) * (size_t)k : 0;
    // few blocks: each one adds its nonzero shared counters to the global ones,
    // so the global atomics grow with blocks x k
    int64_t blocks = (n + 4095) / 4096;
    if (blocks > 152 * 2) blocks = 152 * 2;
    histogram_kernel<<<(unsigned)blocks, 1024, smem, st>>>(assign, n, k, counts32, use_smem);
    return launched();
}

// --------------------------------------------------------------------- scan
// Exclusive scan of the counts by one block of 1024 threads, count(j) giving
// cluster j's members and put(j, offset) taking its offset.  Also the int64
// counts, and the number of empty clusters (zeros, may be NULL).  Each warp has a
// contiguous range of clusters and goes through it twice, for its sum and for the
// offsets, 32 neighbours a step, so that reads and writes are contiguous (a range a
// thread: 60,000 clusters 83 us when only offsets and counts were written, 113
// with the cursors and the empty clusters too; now 31).
template <typename Count, typename Put>
__device__ __forceinline__ void scan_block(int k, Count count, Put put, int64_t *__restrict__ offsets,
                                           int64_t *__restrict__ counts64, int accumulate,
                                           int64_t *__restrict__ zeros) {
    __shared__ int wsum[32], wzero[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int seg = (k + 1023) / 1024 * 32;
    const int lo = min(k, w * seg), hi = min(k, lo + seg);
    auto warp_incl = [&](int v) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        return v;
    };
    constexpr int U = 4;  // steps whose counts are read together
    auto read = [&](int j0, int(&c)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int j = j0 + 32 * u + lane;
            c[u] = j < hi ? count(j) : 0;
        }
    };
    int s = 0, z = 0;  // (counts add up to fewer than 2^31)
    for (int j0 = lo; j0 < hi; j0 += 32 * U) {
        int c[U];
        read(j0, c);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            s += c[u];
            z += j0 + 32 * u + lane < hi && c[u] == 0;
        }
    }
    s = __reduce_add_sync(0xffffffffu, s);
    z = __reduce_add_sync(0xffffffffu, z);
    if (lane == 0) {
        wsum[w] = s;
        wzero[w] = z;
    }
    __syncthreads();
    const int x = wsum[lane], xi = warp_incl(x);  // over the 32 warps, in each of them
    int run = __shfl_sync(0xffffffffu, xi - x, w);
    if (w == 0) {
        z = __reduce_add_sync(0xffffffffu, wzero[lane]);
        if (lane == 31) offsets[k] = xi;
        if (zeros && lane == 0) *zeros = z;
    }
    for (int j0 = lo; j0 < hi; j0 += 32 * U) {
        int c[U];
        read(j0, c);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int j = j0 + 32 * u + lane;
            const int v = warp_incl(c[u]);
            if (j < hi) {
                offsets[j] = run + v - c[u];
                put(j, run + v - c[u]);
                if (counts64) {
                    if (accumulate)
                        counts64[j] += c[u];
                    else
                        counts64[j] = c[u];
                }
            }
            run += __shfl_sync(0xffffffffu, v, 31);
        }
    }
}

// The blocks after the first clear the cluster sums (bytes a multiple of 4,
// 16-byte aligned) while the first one sorts or scans, so that the sums need
// no memset of their own.
__device__ __forceinline__ void clear_sums(void *__restrict__ sums, size_t bytes) {
    const size_t nt = (size_t)(gridDim.x - 1) * blockDim.x;
    const size_t t0 = (size_t)(blockIdx.x - 1) * blockDim.x + threadIdx.x;
    for (size_t i = t0; i < bytes / 16; i += nt) static_cast<uint4 *>(sums)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (size_t i = bytes / 16 * 4 + t0; i < bytes / 4; i += nt) static_cast<uint32_t *>(sums)[i] = 0u;
}

__global__ void __launch_bounds__(1024) scan_offsets_kernel(const int32_t *__restrict__ counts, int k,
                                                            int64_t *__restrict__ offsets,
                                                            int64_t *__restrict__ counts64, int accumulate,
                                                            int32_t *__restrict__ cursor, int64_t *__restrict__ zeros,
                                                            int32_t *__restrict__ flag, void *__restrict__ sums,
                                                            size_t sum_bytes) {
    dep_sync();
    if (flag && blockIdx.x == 0 && threadIdx.x == 0) *flag = 0;
    if (blockIdx.x > 0) {
        clear_sums(sums, sum_bytes);
        return;
    }
    scan_block(k, [&](int j) { return counts[j]; }, [&](int j, int64_t) { cursor[j] = 0; }, offsets, counts64,
               accumulate, zeros);
}

// Histogram, scan and placement of up to SORT1_MAX points in one block: a
// thread keeps its points' clusters and their ranks inside them (the values
// the shared-memory counters returned) in registers between the passes, and
// the order is put together in shared memory (16 bits a point) and written
// out in order: one SM takes 15 us for 20,000 points' scattered stores.
// Three launches and three memsets became one launch, the host's launches
// being what bounds an update of this size.
constexpr int SORT1_PER = 32;
constexpr int SORT1_MAX = 1024 * SORT1_PER;
constexpr int SORT1_MAX_K = 12288;  // 48 KiB of counters; a cluster fits 14 bits, a rank 15

__global__ void __launch_bounds__(1024) sort_one_block_kernel(const int32_t *__restrict__ assign, int n, int k,
                                                              int64_t *__restrict__ offsets,
                                                              int64_t *__restrict__ counts64, int accumulate,
                                                              int32_t *__restrict__ perm, int32_t *__restrict__ scl,
                                                              int64_t *__restrict__ zeros, int32_t *__restrict__ flag,
                                                              void *__restrict__ sums, size_t sum_bytes) {
    dep_sync();
    if (flag && blockIdx.x == 0 && threadIdx.x == 0) *flag = 0;
    if (blockIdx.x > 0) {
        clear_sums(sums, sum_bytes);
        return;
    }
    extern __shared__ int32_t cnt_sh[];
    uint16_t *perm_sh = reinterpret_cast<uint16_t *>(cnt_sh + k), *scl_sh = perm_sh + n;
    for (int j = threadIdx.x; j < k; j += 1024) cnt_sh[j] = 0;
    uint32_t place[SORT1_PER];
#pragma unroll
    for (int i = 0; i < SORT1_PER; ++i) {
        const int t = threadIdx.x + 1024 * i;
        place[i] = t < n ? (uint32_t)assign[t] : 0xffffffffu;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < SORT1_PER; ++i) {
        if (place[i] >= (uint32_t)k)  // out-of-range assignments are skipped
            place[i] = 0xffffffffu;
        else
            place[i] |= (uint32_t)atomicAdd(&cnt_sh[place[i]], 1) << 16;
    }
    __syncthreads();
    scan_block(k, [&](int j) { return cnt_sh[j]; }, [&](int j, int64_t off) { cnt_sh[j] = (int32_t)off; }, offsets,
               counts64, accumulate, zeros);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < SORT1_PER; ++i) {
        if (place[i] == 0xffffffffu) continue;
        const int a = (int)(place[i] & 0xffffu);
        const int pos = cnt_sh[a] + (int)(place[i] >> 16);
        perm_sh[pos] = (uint16_t)(threadIdx.x + 1024 * i);
        scl_sh[pos] = (uint16_t)a;
    }
    __syncthreads();
    const int nval = (int)offsets[k];  // scan_block wrote it before the barriers
    for (int i = threadIdx.x; i < nval; i += 1024) {
        perm[i] = perm_sh[i];
        scl[i] = scl_sh[i];
    }
}

// ------------------------------------------------------------------ scatter
__global__ void scatter_kernel(const int32_t *__restrict__ assign, int64_t n, int k,
                               const int64_t *__restrict__ offsets, int32_t *__restrict__ cursor,
                               int32_t *__restrict__ perm, int32_t *__restrict__ scl) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int a = assign[t];
        if (a < 0 || a >= k) continue;  // skipped consistently with the histogram
        const int pos = atomicAdd(&cursor[a], 1);
        perm[offsets[a] + pos] = (int32_t)t;
        if (scl) scl[offsets[a] + pos] = a;
    }
}

// Block-aggregated form: a block counts its SC_POINTS points per cluster in
// shared memory, reserves one range per cluster with a single global atomic,
// then places its points inside those ranges (shared-memory atomics), so the
// global atomics drop from one per point to one per (block, cluster).
constexpr int SC_POINTS = 4096;
constexpr int SC_THREADS = 512;
constexpr int SC_MAX_K = 12288;  // 48 KiB of counters

__global__ void __launch_bounds__(SC_THREADS) scatter_blocked_kernel(
    const int32_t *__restrict__ assign, int64_t n, int k, const int64_t *__restrict__ offsets,
    int32_t *__restrict__ cursor, int32_t *__restrict__ perm, int32_t *__restrict__ scl) {
    dep_sync();
    extern __shared__ int32_t cnt_sh[];
    const int64_t p0 = (int64_t)blockIdx.x * SC_POINTS;
    const int64_t p1 = min(n, p0 + SC_POINTS);
    for (int j = threadIdx.x; j < k; j += SC_THREADS) cnt_sh[j] = 0;
    __syncthreads();
    for (int64_t t = p0 + threadIdx.x; t < p1; t += SC_THREADS) {
        const int a = assign[t];
        if (a >= 0 && a < k) atomicAdd(&cnt_sh[a], 1);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < k; j += SC_THREADS) {
        const int c = cnt_sh[j];
        if (c) cnt_sh[j] = (int32_t)offsets[j] + atomicAdd(&cursor[j], c);
    }
    __syncthreads();
    for (int64_t t = p0 + threadIdx.x; t < p1; t += SC_THREADS) {
        const int a = assign[t];
        if (a < 0 || a >= k) continue;  // skipped consistently with the histogram
        const int pos = atomicAdd(&cnt_sh[a], 1);
        perm[pos] = (int32_t)t;
        if (scl) scl[pos] = a;
    }
}

cudaError_t launch_sort_by_cluster(const int32_t *assign, int64_t n, int k, int32_t *counts32, int32_t *cursor,
                                   int64_t *offsets, int64_t *counts64, int accumulate, int32_t *perm, int32_t *scl,
                                   int64_t *zeros, int32_t *flag, void *sums, size_t sum_bytes, cudaStream_t st) {
    // a block clears 32 KiB or more
    const unsigned clear = (unsigned)std::min<size_t>(152, (sum_bytes + 32767) / 32768);
    if (n <= SORT1_MAX && k <= SORT1_MAX_K) {
        const size_t smem = sizeof(int32_t) * (size_t)k + 4 * (size_t)n;  // at most 176 KiB
        if (smem > 48 * 1024 - 512) {
            const cudaError_t e = smem_limit(sort_one_block_kernel, sizeof(int32_t) * SORT1_MAX_K + 4 * SORT1_MAX);
            if (e != cudaSuccess) return e;
        }
        launch_dep(sort_one_block_kernel, 1 + clear, 1024, smem, st, 
            assign, (int)n, k, offsets, counts64, accumulate, perm, scl, zeros, flag, sums, sum_bytes);
        return launched();
    }
    cudaError_t e = launch_histogram(assign, n, k, counts32, st);
    if (e != cudaSuccess) return e;
    launch_dep(scan_offsets_kernel, 1 + clear, 1024, 0, st, counts32, k, offsets, counts64, accumulate, cursor, zeros, flag,
                                                    sums, sum_bytes);
    e = launched();
    if (e != cudaSuccess) return e;
    if (k <= SC_MAX_K) {
        const int64_t blocks = (n + SC_POINTS - 1) / SC_POINTS;
        launch_dep(scatter_blocked_kernel, (unsigned)blocks, SC_THREADS, sizeof(int32_t) * (size_t)k, st, 
            assign, n, k, offsets, cursor, perm, scl);
        return launched();
    }
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 8) blocks = 152 * 8;
    scatter_kernel<<<(unsigned)blocks, 256, 0, st>>>(assign, n, k, offsets, cursor, perm, scl);
    return launched();
}

constexpr int SEG_WARPS = 8;
constexpr int SEG_THREADS = SEG_WARPS * 32;
constexpr int SEG_CHUNK = 1024;  // columns per pass

// ------------------------------------------------------- segmented sums: SQ8
__device__ __forceinline__ uint8_t round_half_even_div(int64_t S, int64_t m) {
    int64_t q = S / m;
    const int64_t r = S - q * m;
    if (2 * r > m || (2 * r == m && (q & 1))) q += 1;
    return (uint8_t)q;
}

// Warp w takes members w, w + 8, ...; lane l sums bytes 4l..4l+3 of each
// 128-byte column group; exact integer partials are combined with shared
// memory atomics (order-independent).
__global__ void __launch_bounds__(SEG_THREADS) segsum_sq8_kernel(
    const uint8_t *__restrict__ X, int d, const int32_t *__restrict__ perm,
    const int64_t *__restrict__ offsets, uint8_t *__restrict__ C, int64_t *__restrict__ partial) {
    __shared__ unsigned long long tot[SEG_CHUNK];
    const int j = blockIdx.x;
    const int64_t lo = offsets[j], hi = offsets[j + 1];
    const int64_t cnt = hi - lo;
    if (cnt == 0) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool vec = (d % 4) == 0;
    for (int c0 = 0; c0 < d; c0 += SEG_CHUNK) {
        for (int t = threadIdx.x; t < SEG_CHUNK; t += SEG_THREADS) tot[t] = 0ull;
        __syncthreads();
        uint32_t acc[SEG_CHUNK / 32];  // columns c0 + 4*(lane + 32 g) + u
#pragma unroll
        for (int t = 0; t < SEG_CHUNK / 32; ++t) acc[t] = 0u;
        for (int64_t q = lo + warp; q < hi; q += SEG_WARPS) {
            const uint8_t *x = X + (int64_t)perm[q] * d;
#pragma unroll
            for (int g = 0; g < SEG_CHUNK / 128; ++g) {
                const int c = c0 + 4 * (lane + 32 * g);
                uint32_t w = 0;
                if (vec && c + 3 < d) {
                    w = __ldg(reinterpret_cast<const uint32_t *>(x + c));
                } else {
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (c + u < d) w |= ((uint32_t)__ldg(x + c + u)) << (8 * u);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[4 * g + u] += (w >> (8 * u)) & 0xffu;
            }
        }
#pragma unroll
        for (int g = 0; g < SEG_CHUNK / 128; ++g)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int t = 4 * (lane + 32 * g) + u;
                if (c0 + t < d && acc[4 * g + u]) atomicAdd(&tot[t], (unsigned long long)acc[4 * g + u]);
            }
        __syncthreads();
        for (int t = threadIdx.x; t < SEG_CHUNK; t += SEG_THREADS) {
            const int i = c0 + t;
            if (i >= d) break;
            const int64_t S = (int64_t)tot[t];
            if (partial)
                partial[(int64_t)j * d + i] += S;
            else
                C[(int64_t)j * d + i] = round_half_even_div(S, cnt);
        }
        __syncthreads();
    }
}

cudaError_t launch_segsum_sq8(const uint8_t *X, int d, const int32_t *perm,
                              const int64_t *offsets, int k, uint8_t *C_inout, int64_t *partial,
                              cudaStream_t st) {
    segsum_sq8_kernel<<<k, SEG_THREADS, 0, st>>>(X, d, perm, offsets, C_inout, partial);
    return launched();
}

// ------------------------------------------------------ segmented sums: RBQ1
// Fused decode-average with exact fixed-point sums: Fq = rint(F 2^e),
// T_i = sum Fq xbar_i, U = sum Fq;
// c_i = m_i + (2 T_i - U) f in fp64 -> fp32, with one factor per cluster
// f = (fl(1/sqrt(d)) 2^-e) / count.
__device__ __forceinline__ float rbq1_finish(int64_t T, int64_t U, float m, double f) {
    return __double2float_rn(__dadd_rn((double)m, __dmul_rn(__ll2double_rn(2 * T - U), f)));
}

// -------------------------------------------- chunked segmented sums (load balanced)
// Warps take `run` (at most CH_ROWS) consecutive members of the cluster-sorted order, so
// every warp has the same work whatever the cluster sizes.  A warp adds its
// rows into register accumulators and flushes them with global atomics into
// the cluster's accumulator whenever the cluster changes (and at the end).
// The member count of the sorted order is offsets[k].
constexpr int CH_WARPS = 8;
constexpr int CH_ROWS = SUM_RUN_MAX;

// fp32 / bf16 points -> float or double accumulators S[k][d], for rows without
// the alignment that the other kernels need: lane l takes columns l + 32 t, so
// that a warp's loads are contiguous whatever the row's start, CH_COLS columns a
// pass and four rows' loads in flight.  Four consecutive columns a lane and
// 1024 a pass with two rows in flight: 338k x 101 bf16 327 us, x 515 803 us.
constexpr int CH_COLS = 256;
template <bool BF16, typename ACC>
__global__ void __launch_bounds__(CH_WARPS * 32) chunk_sum_float_kernel(
    const void *__restrict__ Xv, int d, const int32_t *__restrict__ perm,
    const int32_t *__restrict__ scl, const int64_t *__restrict__ offsets, int k,
    ACC *__restrict__ S, int64_t stride, int run) {
    dep_sync();
    constexpr int NT = CH_COLS / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t nval = offsets[k];
    const int64_t q0 = ((int64_t)blockIdx.x * CH_WARPS + warp) * run;
    if (q0 >= nval) return;
    const int64_t q1 = min(nval, q0 + run);
    for (int c0 = 0; c0 < d; c0 += CH_COLS) {
        const int nc = d - c0 - lane;  // this lane's columns c0 + lane + 32 t exist for 32 t < nc
        float acc[NT];
#pragma unroll
        for (int t = 0; t < NT; ++t) acc[t] = 0.0f;
        int cur = scl[q0];
        auto flush = [&](int c) {
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                if (32 * t < nc) atomicAdd(S + (int64_t)c * stride + c0 + lane + 32 * t, (ACC)acc[t]);
                acc[t] = 0.0f;
            }
        };
        for (int64_t q = q0; q < q1; q += 4) {
            int cl[4];
            float v[4][NT];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t qq = min(q + u, q1 - 1);
                cl[u] = scl[qq];
                const int64_t at = (int64_t)perm[qq] * d + c0 + lane;
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    v[u][t] = 0.0f;
                    if (32 * t < nc) {
                        if (BF16)
                            v[u][t] = __uint_as_float((uint32_t)__ldg(static_cast<const uint16_t *>(Xv) + at + 32 * t) << 16);
                        else
                            v[u][t] = __ldg(static_cast<const float *>(Xv) + at + 32 * t);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (q + u >= q1) break;
                if (cl[u] != cur) {
                    flush(cur);
                    cur = cl[u];
                }
#pragma unroll
                for (int t = 0; t < NT; ++t) acc[t] += v[u][t];
            }
        }
        flush(cur);
    }
}

static unsigned chunk_blocks(int64_t n, int run) {
    const int64_t per = (int64_t)CH_WARPS * run;
    int64_t b = (n + per - 1) / per;
    return (unsigned)(b < 1 ? 1 : b);
}

cudaError_t launch_chunk_sum_float(const void *X, int x_is_bf16, int64_t n, int d,
                                   const int32_t *perm, const int32_t *scl,
                                   const int64_t *offsets, int k, float *S_f, double *S_d,
                                   cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const int run = sum_run(n, k, 16, SUM_WARPS, SUM_FLUSH_F32);
    const unsigned g = chunk_blocks(n, run);
    if (S_d) {
        if (x_is_bf16)
            launch_dep(chunk_sum_float_kernel<true, double>, g, CH_WARPS * 32, 0, st, X, d, perm, scl, offsets, k, S_d, d, run);
        else
            launch_dep(chunk_sum_float_kernel<false, double>, g, CH_WARPS * 32, 0, st, X, d, perm, scl, offsets, k, S_d, d, run);
    } else {
        if (x_is_bf16)
            launch_dep(chunk_sum_float_kernel<true, float>, g, CH_WARPS * 32, 0, st, X, d, perm, scl, offsets, k, S_f, d, run);
        else
            launch_dep(chunk_sum_float_kernel<false, float>, g, CH_WARPS * 32, 0, st, X, d, perm, scl, offsets, k, S_f, d, run);
    }
    return launched();
}

// fp32 sums -> centroids (clusters without members keep theirs)
__global__ void finalize_float32_kernel(const float *__restrict__ S,
                                        const int64_t *__restrict__ counts, int k, int d,
                                        float *__restrict__ C) {
    dep_sync();
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)k * d) return;
    const int64_t c = counts[t / d];
    if (c > 0) C[t] = __fdiv_rn(S[t], (float)c);
}

cudaError_t launch_finalize_float32(const float *S, const int64_t *counts, int k, int d,
                                    float *C_inout, cudaStream_t st) {
    const int64_t tot = (int64_t)k * d;
    launch_dep(finalize_float32_kernel, (unsigned)((tot + 255) / 256), 256, 0, st, S, counts, k, d, C_inout);
    return launched();
}

// --------------------------------------------------------------- finalizers
__global__ void finalize_float_kernel(const double *__restrict__ partial,
                                      const int64_t *__restrict__ counts, int k, int d,
                                      float *__restrict__ C) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)k * d) return;
    const int j = (int)(t / d);
    const int64_t c = counts[j];
    if (c > 0) C[t] = __double2float_rn(__ddiv_rn(partial[t], (double)c));
}

cudaError_t launch_finalize_float(const double *partial, const int64_t *counts, int k, int d,
                                  float *C_inout, cudaStream_t st) {
    const int64_t tot = (int64_t)k * d;
    finalize_float_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(partial, counts, k, d,
                                                                         C_inout);
    return launched();
}

__global__ void finalize_sq8_kernel(const int64_t *__restrict__ partial,
                                    const int64_t *__restrict__ counts, int k, int d,
                                    uint8_t *__restrict__ C) {
    dep_sync();
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)k * d) return;
    const int j = (int)(t / d);
    const int64_t c = counts[j];
    if (c > 0) C[t] = round_half_even_div(partial[t], c);
}

cudaError_t launch_finalize_sq8(const int64_t *partial, const int64_t *counts, int k, int d,
                                uint8_t *C_inout, cudaStream_t st) {
    const int64_t tot = (int64_t)k * d;
    launch_dep(finalize_sq8_kernel, (unsigned)((tot + 255) / 256), 256, 0, st, partial, counts, k, d,
                                                                       C_inout);
    return launched();
}

// One block per cluster: the factor f (one fp64 square root and division) is
// formed once and shared; GB300's fp64 rate makes per-element divisions the
// cost of this step otherwise.
__global__ void finalize_rbq1_kernel(const int64_t *__restrict__ partial,
                                     const int64_t *__restrict__ counts, int k, int d,
                                     const float *__restrict__ m, int e, float *__restrict__ C) {
    dep_sync();
    __shared__ double fs;
    const int j = blockIdx.x;
    const int64_t c = counts[j];
    if (c <= 0) return;  // block-uniform
    if (threadIdx.x == 0) {
        const double isd = __ddiv_rn(1.0, __dsqrt_rn((double)d));
        fs = __ddiv_rn(__dmul_rn(isd, ldexp(1.0, -e)), (double)c);
    }
    __syncthreads();
    const double f = fs;
    const int64_t *T = partial + (int64_t)j * (d + 1);
    const int64_t U = T[d];
    for (int i = threadIdx.x; i < d; i += blockDim.x) C[(int64_t)j * d + i] = rbq1_finish(T[i], U, m[i], f);
}

cudaError_t launch_finalize_rbq1(const int64_t *partial, const int64_t *counts, int k, int d,
                                 const float *m, int e, float *C_inout, cudaStream_t st) {
    launch_dep(finalize_rbq1_kernel, k, 256, 0, st, partial, counts, k, d, m, e, C_inout);
    return launched();
}

__global__ void merge_kernel(void *__restrict__ dst, const void *__restrict__ src, int64_t count,
                             int elem_type) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < count;
         t += (int64_t)gridDim.x * blockDim.x) {
        if (elem_type == 0)
            reinterpret_cast<double *>(dst)[t] += reinterpret_cast<const double *>(src)[t];
        else
            reinterpret_cast<int64_t *>(dst)[t] += reinterpret_cast<const int64_t *>(src)[t];
    }
}

cudaError_t launch_merge(void *dst, const void *src, int64_t count, int elem_type,
                         cudaStream_t st) {
    if (count == 0) return cudaSuccess;
    int64_t blocks = (count + 255) / 256;
    if (blocks > 152 * 8) blocks = 152 * 8;
    merge_kernel<<<(unsigned)blocks, 256, 0, st>>>(dst, src, count, elem_type);
    return launched();
}

}  // namespace skm

namespace skm {

// ------------------------------------------------------- empty-cluster split
// Section 2.3 STEP 3 (splitting large clusters): clusters left empty by an
// update, in increasing index order, each take the current largest cluster L
// (most members, ties to the lowest index; stop once L has fewer than 2) and
// the two become L's centroid moved by a relative 2^-10 in opposite
// directions, the sign alternating per dimension (fp32), or by one code step
// (SQ8, clipped).  L keeps ceil(n_L/2) members for later choices.  One block.
constexpr int SPLIT_THREADS = 1024;

template <typename T>
__global__ void __launch_bounds__(SPLIT_THREADS) split_empty_kernel(T *__restrict__ C,
                                                                    const int64_t *__restrict__ counts,
                                                                    int k, int d, int64_t *__restrict__ w) {
    __shared__ int64_t sv[SPLIT_THREADS / 32];
    __shared__ int si[SPLIT_THREADS / 32];
    __shared__ int sL;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int j = tid; j < k; j += SPLIT_THREADS) w[j] = counts[j];
    __syncthreads();
    for (int j = 0; j < k; ++j) {
        if (counts[j] != 0) continue;  // the same for every thread
        // argmax of w, ties to the lowest index
        int64_t bv = -1;
        int bi = 0x7fffffff;
        for (int t = tid; t < k; t += SPLIT_THREADS)
            if (w[t] > bv) {
                bv = w[t];
                bi = t;
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const int64_t ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ov > bv || (ov == bv && oi < bi)) {
                bv = ov;
                bi = oi;
            }
        }
        if (lane == 0) {
            sv[wid] = bv;
            si[wid] = bi;
        }
        __syncthreads();
        if (tid == 0) {
            int64_t v = sv[0];
            int L = si[0];
            for (int t = 1; t < SPLIT_THREADS / 32; ++t)
                if (sv[t] > v || (sv[t] == v && si[t] < L)) {
                    v = sv[t];
                    L = si[t];
                }
            sL = v >= 2 ? L : -1;
        }
        __syncthreads();
        const int L = sL;
        if (L < 0) break;  // the same for every thread
        for (int i = tid; i < d; i += SPLIT_THREADS) {
            const T c = C[(int64_t)L * d + i];
            const bool even = (i & 1) == 0;
            if constexpr (sizeof(T) == 1) {
                const int s = even ? 1 : -1;
                const int a = (int)c + s, b = (int)c - s;
                C[(int64_t)j * d + i] = (T)(a < 0 ? 0 : (a > 255 ? 255 : a));
                C[(int64_t)L * d + i] = (T)(b < 0 ? 0 : (b > 255 ? 255 : b));
            } else {
                const float up = 1.0f + 0x1p-10f, dn = 1.0f - 0x1p-10f;
                C[(int64_t)j * d + i] = __fmul_rn(c, even ? up : dn);
                C[(int64_t)L * d + i] = __fmul_rn(c, even ? dn : up);
            }
        }
        if (tid == 0) {
            w[j] = w[L] / 2;
            w[L] -= w[j];
        }
        __syncthreads();
    }
}

cudaError_t launch_split_empty(void *C, int code_bytes, const int64_t *counts, int k, int d,
                               int64_t *w, cudaStream_t st) {
    if (code_bytes == 1)
        split_empty_kernel<uint8_t><<<1, SPLIT_THREADS, 0, st>>>(static_cast<uint8_t *>(C), counts, k, d, w);
    else
        split_empty_kernel<float><<<1, SPLIT_THREADS, 0, st>>>(static_cast<float *>(C), counts, k, d, w);
    return launched();
}

}  // namespace skm

namespace skm {

// ---------------------------------------------------- stable sort by group
// Rows ordered by group, increasing row index within a group (hierarchical
// k-means' fine phase works on the meso clusters in this order, and its
// initial fine centroids are positions inside each group).  Blocks own
// SS_CHUNK consecutive rows: per-block group counts, a column scan over the
// blocks, then each block (one warp, 32 rows at a time in order) places its
// rows with __match_any_sync ranks, so the order is deterministic.
constexpr int SS_CHUNK = 4096;

static __device__ __forceinline__ int clamp_key(int g, int m) { return g < 0 ? 0 : (g >= m ? m - 1 : g); }

__global__ void ss_hist_kernel(const int32_t *__restrict__ key, int64_t n, int m, int32_t *__restrict__ hist) {
    extern __shared__ int32_t h[];
    for (int j = threadIdx.x; j < m; j += blockDim.x) h[j] = 0;
    __syncthreads();
    const int64_t r0 = (int64_t)blockIdx.x * SS_CHUNK, r1 = min(n, r0 + SS_CHUNK);
    for (int64_t r = r0 + threadIdx.x; r < r1; r += blockDim.x) atomicAdd(&h[clamp_key(key[r], m)], 1);
    __syncthreads();
    for (int j = threadIdx.x; j < m; j += blockDim.x) hist[(int64_t)blockIdx.x * m + j] = h[j];
}

// hist[b][j] (counts) -> first sorted position of block b's rows of group j;
// sizes[j] = rows in group j.  One block: a warp takes a group's counts 128
// blocks at a time (a thread walking them one by one waited for every load:
// 245 blocks x 63 groups 100 us).
__global__ void __launch_bounds__(1024) ss_scan_kernel(int32_t *__restrict__ hist, int nblk, int m,
                                                       int32_t *__restrict__ sizes) {
    extern __shared__ int32_t goff[];
    __shared__ int32_t wtot[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    auto warp_incl = [&](int32_t v) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        return v;
    };
    for (int j = wid; j < m; j += 32) {
        int32_t run = 0;
        for (int b0 = 0; b0 < nblk; b0 += 128) {
            int32_t t[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int b = b0 + 32 * u + lane;
                t[u] = b < nblk ? hist[(int64_t)b * m + j] : 0;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int b = b0 + 32 * u + lane;
                const int32_t in = warp_incl(t[u]);
                if (b < nblk) hist[(int64_t)b * m + j] = run + in - t[u];
                run += __shfl_sync(0xffffffffu, in, 31);
            }
        }
        if (lane == 0) {
            sizes[j] = run;
            goff[j] = run;
        }
    }
    __syncthreads();
    int32_t before = 0;  // goff: sizes -> exclusive sums, 1024 groups a round
    for (int j0 = 0; j0 < m; j0 += 1024) {
        const int j = j0 + threadIdx.x;
        const int32_t v = j < m ? goff[j] : 0;
        const int32_t in = warp_incl(v);
        if (lane == 31) wtot[wid] = in;
        __syncthreads();
        const int32_t w = wtot[lane];
        const int32_t wi = warp_incl(w);
        const int32_t mine = __shfl_sync(0xffffffffu, wi - w, wid);
        if (j < m) goff[j] = before + mine + in - v;
        before += __shfl_sync(0xffffffffu, wi, 31);
        __syncthreads();
    }
    for (int64_t i = threadIdx.x; i < (int64_t)nblk * m; i += 1024) hist[i] += goff[i % m];
}

__global__ void ss_place_kernel(const int32_t *__restrict__ key, int64_t n, int m,
                                const int32_t *__restrict__ starts, int32_t *__restrict__ perm,
                                int32_t *__restrict__ skey) {
    extern __shared__ int32_t cnt[];
    const int lane = threadIdx.x;  // one warp
    for (int j = lane; j < m; j += 32) cnt[j] = starts[(int64_t)blockIdx.x * m + j];
    __syncwarp();
    const int64_t r0 = (int64_t)blockIdx.x * SS_CHUNK, r1 = min(n, r0 + SS_CHUNK);
    const unsigned lt = (1u << lane) - 1u;
    // the next 8 rounds' keys are loaded together (each round waiting for its
    // own: 85 us for 1M rows)
    constexpr int PF = 8;
    int kb[PF];
    for (int64_t s = r0, at = 0; s < r1; s += 32, ++at) {
        const int64_t r = s + lane;
        if (at % PF == 0) {
#pragma unroll
            for (int u = 0; u < PF; ++u) kb[u] = r + 32 * u < r1 ? key[r + 32 * u] : 0;
        }
        int kr = kb[0];
#pragma unroll
        for (int u = 1; u < PF; ++u) kr = at % PF == u ? kb[u] : kr;
        const int g = r < r1 ? clamp_key(kr, m) : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, g);
        int pos = 0;
        if (g >= 0) pos = cnt[g] + __popc(peers & lt);
        __syncwarp();
        if (g >= 0 && (peers & lt) == 0) cnt[g] += __popc(peers);  // the group's lowest lane
        __syncwarp();
        if (g >= 0) {
            perm[pos] = (int32_t)r;
            skey[pos] = g;
        }
    }
}

cudaError_t launch_stable_sort(const int32_t *key, int64_t n, int m, int32_t *hist, int32_t *sizes,
                               int32_t *perm, int32_t *skey, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const int nblk = (int)((n + SS_CHUNK - 1) / SS_CHUNK);
    const size_t sm = sizeof(int32_t) * (size_t)m;
    ss_hist_kernel<<<nblk, 256, sm, st>>>(key, n, m, hist);
    cudaError_t e = launched();
    if (e != cudaSuccess) return e;
    // with the most groups the counters are 48 KiB, and the kernel's own words come
    // on top
    constexpr int SS_MAX_M = 12288;
    e = smem_limit(ss_scan_kernel, sizeof(int32_t) * SS_MAX_M);
    if (e != cudaSuccess) return e;
    ss_scan_kernel<<<1, 1024, sm, st>>>(hist, nblk, m, sizes);
    e = launched();
    if (e != cudaSuccess) return e;
    ss_place_kernel<<<nblk, 32, sm, st>>>(key, n, m, hist, perm, skey);
    return launched();
}

// dst row q = src row perm[q], a row being `units` units of T; one thread per
// unit, so that the writes and each row's reads are contiguous whatever the
// row's size (a warp per row left most lanes idle: 1M rows of 96 bytes 140 us,
// of one 4-byte factor as much)
template <typename T, typename I>
__global__ void gather_units_kernel(const T *__restrict__ src, int units, const int32_t *__restrict__ perm, I total,
                                    T *__restrict__ dst) {
    const I u = (I)units;
    for (I t = blockIdx.x * (I)blockDim.x + threadIdx.x; t < total; t += (I)gridDim.x * blockDim.x) {
        const I q = t / u;
        dst[t] = src[(int64_t)perm[q] * units + (int64_t)(t - q * u)];
    }
}

template <typename T>
static cudaError_t launch_gather_units(const void *src, int64_t rowbytes, const int32_t *perm, int64_t n, void *dst,
                                       cudaStream_t st) {
    const int units = (int)(rowbytes / (int64_t)sizeof(T));
    const int64_t total = n * units;
    const int64_t blocks = std::min<int64_t>(152 * 32, (total + 255) / 256);
    const T *s = static_cast<const T *>(src);
    T *d = static_cast<T *>(dst);
    if (total < (int64_t(1) << 31))  // and a last stride past it stays below 2^32
        gather_units_kernel<T, uint32_t><<<(unsigned)blocks, 256, 0, st>>>(s, units, perm, (uint32_t)total, d);
    else
        gather_units_kernel<T, int64_t><<<(unsigned)blocks, 256, 0, st>>>(s, units, perm, total, d);
    return launched();
}

cudaError_t launch_gather_rows_bytes(const void *src, int64_t rowbytes, const int32_t *perm, int64_t n,
                                     void *dst, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const uintptr_t a = reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst) | (uintptr_t)rowbytes;
    if ((a & 15) == 0) return launch_gather_units<uint4>(src, rowbytes, perm, n, dst, st);
    if ((a & 3) == 0) return launch_gather_units<uint32_t>(src, rowbytes, perm, n, dst, st);
    return launch_gather_units<uint8_t>(src, rowbytes, perm, n, dst, st);
}

// out[perm[q]] = in[q] (4-byte values)
__global__ void unpermute_kernel(const int32_t *__restrict__ in, const int32_t *__restrict__ perm, int64_t n,
                                 int32_t *__restrict__ out) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
        out[perm[q]] = in[q];
}

cudaError_t launch_unpermute(const void *in, const int32_t *perm, int64_t n, void *out, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    unpermute_kernel<<<(int)blocks, 256, 0, st>>>(static_cast<const int32_t *>(in), perm, n,
                                                  static_cast<int32_t *>(out));
    return launched();
}

}  // namespace skm
