// Projection Y = (X - mean) P on tensor cores in fp32 accuracy (Section 3.1:
// JLT / PCA, the random rotation).  x - mean and P are split into bf16 parts, x =
// x1 + x2 + x3 (each the round-to-nearest bf16 of the remainder, so the split is
// exact), and the six products with i + j <= 4 are accumulated in fp32; the
// three left out are below 2^-24 relative.
//
// One persistent CTA per SM walks output tiles of 128 rows x up to 256 columns;
// per 64-dimension slice of a tile:
//   warps 10 ..  converters: the slice of X from global memory into registers
//                (the next slice's loads in flight), minus the mean, split and
//                stored as three swizzled bf16 operands in shared memory
//   warp 0       TMA producer of P's parts, one 64 x N slice of a part a slot
//   warp 1       MMA issuer, six products a slice: x1 p1 into one TMEM
//                accumulator, the five small ones into another, so that the
//                small terms are not rounded at the size of the large one's sum
//   warps 2 ..   epilogue: the two accumulators added once and written out
// So X is read once and its parts never leave the SM.  1M x 1024 -> 256: 1.9 to
// 2.0 ms, bound by the six products (1.62 ms at the measured bf16 rate; X and Y
// take 0.68 ms at the copy bandwidth).  Split by a kernel of its own into 6
// bytes a value that a GEMM kernel then read it took 2.02 + 1.92 ms.  The error
// against 64 bits (relative 2-norm, embeddings, d = 256 .. 1536) is 2.3e-7 ..
// 1.54e-6, the accumulator's rounding, and 0.1 .. 1.3% below that of one
// accumulator for all six products.
// 128-column accumulators would let the next tile start during the epilogue,
// but an N = 128 MMA reads as many bytes of shared memory a flop as there is
// bandwidth; the epilogue is a few per cent of a tile instead.
#include <algorithm>

#include "skm_tc.cuh"
#include "tc_ptx.cuh"

namespace skm {
namespace {

constexpr int PM = 128;        // rows a tile (TMEM lanes)
constexpr int PN = 256;        // columns a tile, at most
constexpr int PK = 64;         // dimensions a slice: one 128-byte swizzle row of bf16
constexpr int PARTS = 3;
constexpr int A_PART = PM * PK * 2;           // 16 KiB
constexpr int A_BUF = PARTS * A_PART;         // a slice's three operands
constexpr int A_BUFS = 2;
constexpr int B_SLOT = PN * PK * 2;           // 32 KiB
constexpr int B_SLOTS = 4;
constexpr int EPI_WARPS = 8;
constexpr int CVT_WARPS = 8;
constexpr int CVT_THREADS = 32 * CVT_WARPS;
constexpr int THREADS = 64 + 32 * EPI_WARPS + CVT_THREADS;
constexpr int UNITS = PM * (PK / 8) / CVT_THREADS;  // 8-dimension pieces a converter thread takes a slice
constexpr size_t SMEM = 1024 + (size_t)A_BUFS * A_BUF + (size_t)B_SLOTS * B_SLOT + 256;
static_assert(SMEM <= 227 * 1024, "shared memory per CTA");

struct ProjParams {
    const float *X;
    const float *mean;  // or NULL
    void *Y;            // [n][dout], fp32 or bf16 bits
    int64_t n;
    int64_t ntiles;     // row tiles x column tiles
    int d, dout;
    int nslices;        // ceil(d / 64)
    int nct, ncols;     // column tiles and their width (a multiple of 16)
    int y_bf16;
    int vec;            // X rows and the mean can be read 16 bytes at a time
    int yvec;           // Y is 16-byte aligned
    int32_t *abort_flag;
    unsigned long long inject_wait_ns;  // fault injection: see mbar_wait below
};

// fp32 v -> bf16 parts v1 + v2 + v3 (each the round-to-nearest-even bf16 of
// the remainder; the remainders are exact in fp32)
__device__ __forceinline__ void split3(float v, uint16_t &a, uint16_t &b, uint16_t &c) {
    const __nv_bfloat16 h1 = __float2bfloat16_rn(v);
    const float r1 = __fsub_rn(v, __bfloat162float(h1));
    const __nv_bfloat16 h2 = __float2bfloat16_rn(r1);
    const float r2 = __fsub_rn(r1, __bfloat162float(h2));
    a = __bfloat16_as_ushort(h1);
    b = __bfloat16_as_ushort(h2);
    c = __bfloat16_as_ushort(__float2bfloat16_rn(r2));
}
// the same for two values, packed
__device__ __forceinline__ void split3x2(float v0, float v1, uint32_t &a, uint32_t &b, uint32_t &c) {
    auto pack = [](float lo, float hi) {
        uint32_t r;
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
        return r;
    };
    auto lo = [](uint32_t w) { return __uint_as_float(w << 16); };
    auto hi = [](uint32_t w) { return __uint_as_float(w & 0xffff0000u); };
    a = pack(v0, v1);
    const float r0 = __fsub_rn(v0, lo(a)), r1 = __fsub_rn(v1, hi(a));
    b = pack(r0, r1);
    c = pack(__fsub_rn(r0, lo(b)), __fsub_rn(r1, hi(b)));
}

__global__ void __launch_bounds__(THREADS, 1) project_tc_kernel(const __grid_constant__ CUtensorMap tmB,
                                                                const ProjParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw);
    const uint32_t sA = base, sB = base + A_BUFS * A_BUF;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + (size_t)A_BUFS * A_BUF + (size_t)B_SLOTS * B_SLOT);
    const uint32_t bar0 = smem_u32(bars);
    auto bfull = [&](uint32_t s) { return bar0 + 8u * s; };
    auto bempty = [&](uint32_t s) { return bar0 + 8u * (B_SLOTS + s); };
    auto afull = [&](uint32_t s) { return bar0 + 8u * (2 * B_SLOTS + s); };
    auto aempty = [&](uint32_t s) { return bar0 + 8u * (2 * B_SLOTS + A_BUFS + s); };
    const uint32_t tfull = bar0 + 8u * (2 * B_SLOTS + 2 * A_BUFS), tempty = tfull + 8u, drain_bar = tfull + 16u,
                   inject_bar = tfull + 24u;  // (nothing arrives on the last)
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * B_SLOTS + 2 * A_BUFS + 4);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int32_t *abort_flag = p.abort_flag;

    if (threadIdx.x == 0) {
        for (int s = 0; s < B_SLOTS; ++s) {
            mbar_init(bfull(s), 1);
            mbar_init(bempty(s), 1);
        }
        for (int s = 0; s < A_BUFS; ++s) {
            mbar_init(afull(s), CVT_WARPS);
            mbar_init(aempty(s), 1);
        }
        mbar_init(tfull, 1);
        mbar_init(tempty, EPI_WARPS);
        mbar_init(drain_bar, 1);
        mbar_init(inject_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // this CTA's tiles: t = (row tile) nct + column tile
    const int64_t t0 = blockIdx.x, tstep = gridDim.x;

    if (warp == 0) {
        if (lane == 0) {  // ---------------------------------------- TMA producer
            uint32_t it = 0;
            if (p.inject_wait_ns && !mbar_wait(inject_bar, 0u, abort_flag, p.inject_wait_ns)) goto producer_done;
            for (int64_t t = t0; t < p.ntiles; t += tstep) {
                const int col0 = (int)(t % p.nct) * p.ncols;
                for (int kc = 0; kc < p.nslices; ++kc)
                    for (int part = PARTS - 1; part >= 0; --part, ++it) {
                        const uint32_t s = it % B_SLOTS;
                        if (!mbar_wait(bempty(s), ((it / B_SLOTS) & 1u) ^ 1u, abort_flag)) goto producer_done;
                        mbar_expect_tx(bfull(s), (uint32_t)p.ncols * PK * 2);
                        tma_load_2d(sB + s * B_SLOT, &tmB, kc * PK, part * p.dout + col0, bfull(s));
                    }
            }
        producer_done:
            // the copies issued land before the CTA can exit (after a normal run
            // the MMA warp has consumed them all)
            for (uint32_t s = 0; s < (uint32_t)B_SLOTS && s < it; ++s) {
                const uint32_t last = s + ((it - 1u - s) / B_SLOTS) * B_SLOTS;
                mbar_drain(bfull(s), (last / B_SLOTS) & 1u);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {  // ------------------------------------------ MMA issuer
            // D fp32, A and B bf16, both K-major, M = 128, N = ncols
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.ncols >> 3) << 17) |
                                   ((uint32_t)(PM >> 4) << 24);
            uint32_t it = 0, ia = 0, tiles = 0;
            bool issued = false, gave_up = true;
            for (int64_t t = t0; t < p.ntiles; t += tstep, ++tiles) {
                if (!mbar_wait(tempty, (tiles & 1u) ^ 1u, abort_flag)) goto mma_done;
                tc_fence_after();
                for (int kc = 0; kc < p.nslices; ++kc, ++ia) {
                    const uint32_t ab = ia % A_BUFS;
                    if (!mbar_wait(afull(ab), (ia / A_BUFS) & 1u, abort_flag)) goto mma_done;
                    // P's part j with X's parts PARTS - 1 - j .. 0 (0-based: i + j <= 2)
                    for (int j = PARTS - 1; j >= 0; --j, ++it) {
                        const uint32_t s = it % B_SLOTS;
                        if (!mbar_wait(bfull(s), (it / B_SLOTS) & 1u, abort_flag)) goto mma_done;
                        tc_fence_after();
                        const uint64_t bd = sw128_desc(sB + s * B_SLOT);
                        for (int i = PARTS - 1 - j; i >= 0; --i) {
                            const bool large = i == 0 && j == 0;
                            const uint32_t dcol = tmem + (large ? 0u : (uint32_t)PN);
                            // the first product into an accumulator overwrites it
                            const bool fresh = kc == 0 && (large || j == PARTS - 1);
                            const uint64_t ad = sw128_desc(sA + ab * A_BUF + i * A_PART);
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk)
                                tc_mma(dcol, ad + 2u * kk, bd + 2u * kk, idesc, !(fresh && kk == 0));
                        }
                        issued = true;
                        tc_commit(bempty(s));
                    }
                    tc_commit(aempty(ab));
                }
                tc_commit(tfull);
            }
            gave_up = false;
        mma_done:
            if (gave_up && issued) {  // the MMAs issued so far complete before TMEM is released
                tc_commit(drain_bar);
                mbar_drain(drain_bar, 0u);
            }
        }
    } else if (warp < 2 + EPI_WARPS) {  // --------------------------------- epilogue
        const int q = warp & 3;                    // TMEM lane quarter this warp may access
        const int half = (warp - 2) >> 2;          // which half of the 32-column groups
        const int groups = (p.ncols + 31) / 32;
        uint32_t tiles = 0;
        // a wait ran out: this tile and those after it are written as NaN, so that
        // whoever reads Y sees it (the call has long returned)
        bool gave_up = false;
        for (int64_t t = t0; t < p.ntiles; t += tstep, ++tiles) {
            const int64_t row = (t / p.nct) * PM + q * 32 + lane;
            const int col0 = (int)(t % p.nct) * p.ncols;
            const int colw = min(p.ncols, p.dout - col0);
            if (!gave_up) gave_up = !__all_sync(0xffffffffu, mbar_wait(tfull, tiles & 1u, abort_flag));
            tc_fence_after();
            const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
            for (int g = half; g < groups; g += EPI_WARPS / 4) {
                uint32_t v[32], w[32];
                tmem_ld32(taddr + 32 * g, v);
                tmem_ld32(taddr + PN + 32 * g, w);
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    v[i] = gave_up ? 0x7fffffffu
                                   : __float_as_uint(__fadd_rn(__uint_as_float(v[i]), __uint_as_float(w[i])));
                const int c0 = 32 * g, cn = row < p.n ? min(32, colw - c0) : 0;
                if (cn <= 0) {
                    // nothing of this group inside Y
                } else if (p.y_bf16) {
                    uint16_t *y = static_cast<uint16_t *>(p.Y) + row * p.dout + col0 + c0;
                    if (cn == 32 && p.yvec && (p.dout & 7) == 0) {
#pragma unroll
                        for (int i = 0; i < 32; i += 8) {
                            uint32_t o[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                asm("cvt.rn.bf16x2.f32 %0, %1, %2;"
                                    : "=r"(o[u])
                                    : "f"(__uint_as_float(v[i + 2 * u + 1])), "f"(__uint_as_float(v[i + 2 * u])));
                            *reinterpret_cast<uint4 *>(y + i) = make_uint4(o[0], o[1], o[2], o[3]);
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (i < cn) y[i] = __bfloat16_as_ushort(__float2bfloat16_rn(__uint_as_float(v[i])));
                    }
                } else {
                    float *y = static_cast<float *>(p.Y) + row * p.dout + col0 + c0;
                    if (cn == 32 && p.yvec && (p.dout & 3) == 0) {
#pragma unroll
                        for (int i = 0; i < 32; i += 4)
                            *reinterpret_cast<uint4 *>(y + i) = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (i < cn) y[i] = __uint_as_float(v[i]);
                    }
                }
                __syncwarp();  // the next TMEM loads are the whole warp's
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0 && !gave_up) mbar_arrive(tempty);  // (no accumulator is handed on unread)
        }
    } else {  // ------------------------------------------------------- converters
        // thread ct: dimensions 8 c .. 8 c + 7 (c = ct mod 8) of the slice, rows
        // ct / 8 + 32 u of the tile
        const int ct = threadIdx.x - (64 + 32 * EPI_WARPS);
        const int c = ct & 7, rr = ct >> 3;
        constexpr int RSTEP = CVT_THREADS / 8;
        float4 x[UNITS][2], mu[2];
        auto load = [&](int64_t t, int kc) {
            const int64_t r0 = (t / p.nct) * PM + rr;
            const int i0 = kc * PK + 8 * c;
            const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            if (p.vec) {  // d % 4 == 0: a piece's float4 lies inside the row or past it
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const bool in = i0 + 4 * h < p.d;
                    mu[h] = in && p.mean ? __ldg(reinterpret_cast<const float4 *>(p.mean + i0 + 4 * h)) : z;
#pragma unroll
                    for (int u = 0; u < UNITS; ++u) {
                        const int64_t r = r0 + RSTEP * u;
                        x[u][h] = in && r < p.n ? __ldg(reinterpret_cast<const float4 *>(p.X + r * p.d + i0 + 4 * h)) : z;
                    }
                }
            } else {
                auto one = [&](const float *src, int i) { return i < p.d ? __ldg(src + i) : 0.0f; };
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int i = i0 + 4 * h;
                    mu[h] = z;
                    if (p.mean) mu[h] = make_float4(one(p.mean, i), one(p.mean, i + 1), one(p.mean, i + 2), one(p.mean, i + 3));
#pragma unroll
                    for (int u = 0; u < UNITS; ++u) {
                        const int64_t r = r0 + RSTEP * u;
                        x[u][h] = z;
                        if (r < p.n) {
                            const float *s = p.X + r * p.d;
                            x[u][h] = make_float4(one(s, i), one(s, i + 1), one(s, i + 2), one(s, i + 3));
                        }
                    }
                }
            }
        };
        uint32_t ia = 0;
        if (t0 < p.ntiles) load(t0, 0);
        for (int64_t t = t0; t < p.ntiles; t += tstep) {
            for (int kc = 0; kc < p.nslices; ++kc, ++ia) {
                const uint32_t ab = ia % A_BUFS;
                if (!__all_sync(0xffffffffu, mbar_wait(aempty(ab), ((ia / A_BUFS) & 1u) ^ 1u, abort_flag)))
                    goto cvt_done;
                uint8_t *buf = smem + (size_t)ab * A_BUF;
#pragma unroll
                for (int u = 0; u < UNITS; ++u) {
                    const int r = rr + RSTEP * u;
                    uint32_t o[PARTS][4];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float4 v = x[u][h], m = mu[h];
                        split3x2(__fsub_rn(v.x, m.x), __fsub_rn(v.y, m.y), o[0][2 * h], o[1][2 * h], o[2][2 * h]);
                        split3x2(__fsub_rn(v.z, m.z), __fsub_rn(v.w, m.w), o[0][2 * h + 1], o[1][2 * h + 1],
                                 o[2][2 * h + 1]);
                    }
                    // 128-byte swizzle: 16-byte piece c of row r at piece c ^ (r mod 8)
                    const uint32_t off = (uint32_t)r * 128u + (uint32_t)((c ^ (r & 7)) << 4);
#pragma unroll
                    for (int s3 = 0; s3 < PARTS; ++s3)
                        *reinterpret_cast<uint4 *>(buf + s3 * A_PART + off) =
                            make_uint4(o[s3][0], o[s3][1], o[s3][2], o[s3][3]);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(afull(ab));
                // the next slice's loads, in flight until its buffer is free
                if (kc + 1 < p.nslices) load(t, kc + 1);
                else if (t + tstep < p.ntiles) load(t + tstep, 0);
            }
        }
    cvt_done:;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// P [d][dout] -> parts [3][dout][dp] (transposed: K-major rows per output
// column), 32 x 32 blocks through shared memory so that both sides are
// contiguous; clears the abort flag.
__global__ void __launch_bounds__(256) proj_split_p_kernel(const float *__restrict__ P, int d, int dout, int dp,
                                                           uint16_t *__restrict__ B, int32_t *__restrict__ flag) {
    __shared__ float tile[32][33];
    const int i0 = blockIdx.x * 32, j0 = blockIdx.y * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *flag = 0;
    for (int r = ty; r < 32; r += 8)
        tile[r][tx] = i0 + r < d && j0 + tx < dout ? __ldg(P + (int64_t)(i0 + r) * dout + j0 + tx) : 0.0f;
    __syncthreads();
    const size_t part = (size_t)dout * dp;
    for (int r = ty; r < 32; r += 8) {
        const int j = j0 + r, i = i0 + tx;
        if (j >= dout || i >= dp) continue;
        uint16_t a, b, c;
        split3(tile[tx][r], a, b, c);
        uint16_t *o = B + (size_t)j * dp + i;
        o[0] = a;
        o[part] = b;
        o[2 * part] = c;
    }
}

inline int round8(int d) { return (d + 7) & ~7; }

}  // namespace

// the flag and P's parts, as tc_project carves them
size_t tc_project_ws_min(int d, int dout) {
    Carver cv(nullptr, 0);
    cv.take<int32_t>(16);
    cv.take<uint16_t>((size_t)PARTS * dout * round8(d));
    return cv.off;
}

int tc_project(const float *X, int64_t n, int d, const float *mean, const float *P, int dout, int out_bf16, void *Y,
               void *ws, size_t ws_bytes, cudaStream_t st) {
    const int dp = round8(d);
    Carver cv(ws, ws_bytes);
    int32_t *flag = cv.take<int32_t>(16);
    uint16_t *B = cv.take<uint16_t>((size_t)PARTS * dout * dp);
    if (cv.off > ws_bytes) return set_error(SKM_ERR_NO_MEMORY, "projection workspace too small");
    proj_split_p_kernel<<<dim3((unsigned)cdiv(dp, 32), (unsigned)cdiv(dout, 32)), 256, 0, st>>>(P, d, dout, dp, B, flag);
    SKM_CUDA_TRY(launched());
    ProjParams p{};
    p.X = X;
    p.mean = mean;
    p.Y = Y;
    p.n = n;
    p.d = d;
    p.dout = dout;
    p.nslices = (int)cdiv(d, PK);
    // column tiles of about equal width, a multiple of 16 (MMA N)
    p.nct = (int)cdiv(dout, PN);
    p.ncols = (int)(cdiv(cdiv(dout, p.nct), 16) * 16);
    p.ntiles = cdiv(n, PM) * p.nct;
    p.y_bf16 = out_bf16;
    p.vec = d % 4 == 0 && ((uintptr_t)X & 15) == 0 && ((uintptr_t)mean & 15) == 0;
    p.yvec = ((uintptr_t)Y & 15) == 0;
    p.abort_flag = flag;
    p.inject_wait_ns = fault_take(SKM_FAULT_WAIT) ? 1000000ull : 0ull;  // 1 ms
    CUtensorMap mb;
    SKM_TRY(make_map(&mb, B, (int64_t)PARTS * dout, d, dp, p.ncols, 2));
    SKM_CUDA_TRY(smem_limit(project_tc_kernel, SMEM));
    const int grid = (int)std::min<int64_t>(device_sms(), p.ntiles);
    tc_timer_mark(st, 0);
    project_tc_kernel<<<grid, THREADS, SMEM, st>>>(mb, p);
    tc_timer_mark(st, 1);
    SKM_CUDA_TRY(launched());
    return SKM_OK;
}

}  // namespace skm
