// dense_tc.cu -- the full field recompute of the dense instance, H = J S
// (row a4), on the 5th-generation tensor cores, from the bit matrix.
//
// J is +-1 off the diagonal, so it is stored and read as one bit per coupling
// (1.25 GB at n = 100,000 instead of the 10 GB of bytes).  A CTA takes blocks
// of 512 rows.  TMA copies 512 rows x 128 bytes (1,024 couplings) of the bit
// matrix into shared memory with the 128-byte swizzle and the population's
// 128-column slices (e4m3, replicas padded to a multiple of 16) beside them.
// Sixteen warps turn a slice's bits into e4m3 +-1 in registers and store them
// as the MMA's A operand in tensor memory, one row a lane: a column of four
// operands takes a shift and one three-input logic operation, since the K
// order within 32 couplings is free as long as both operands share it (byte b
// of column s is coupling s + 8 b).  One thread issues tcgen05.mma
// kind::f8f6f4 (M = 128, K = 32, N the padded replicas, A from tensor memory,
// B from shared memory) into fp32 accumulators.  Products are +-1 or 0 and
// partial sums integers below 2^24, so the field is exact; the clear diagonal
// bit counts as -1, which the epilogue corrects by adding the spin.
//
// The (row block, 1,024 couplings) units are dealt out as one contiguous range
// per CTA, so every SM has the same work at any n; a block cut between CTAs
// is added up with integer atomics (the fields are zeroed before).
//
// Bound: the A operands' way into tensor memory (about 28 bytes a clock and SM:
// 64 KB a slice), not HBM.  Measured at n = 100,000, R = 64: 1.12 ms (1.40 for
// TMA-fed byte couplings before); n = 5,001, R = 24: 20 us (917 for the
// mma.sync kernel that took sizes not a multiple of 16 before).
//
// Every wait is bounded; on expiry the kernel records PAMC_ERR_TIMEOUT, lets
// the copies and MMAs it issued complete (bounded), frees tensor memory and
// returns.
#include <cuda.h>

#include <mutex>

#include "pamc_device.cuh"
#include "pamc_internal.h"
#include "tc_sm100.cuh"

namespace pamc {

namespace {

constexpr int kRcTiles = 4;                        // M = 128 tiles of a row block
constexpr int kRcRows = 128 * kRcTiles;
constexpr int kRcChunk = 8;                        // 128-column slices of a unit
constexpr int kRcBitStages = 2, kRcBStages = 4, kRcAStages = 2;
constexpr int kRcBitBytes = kRcRows * 128;         // one unit's bits
constexpr int kRcBBytes = 64 * 128;                // one slice of the population
constexpr int kRcExpand = 4 * kRcTiles;            // expanding warps
constexpr int kRcThreads = (kRcExpand + 2) * 32;   // + copy and MMA warps
constexpr uint32_t kRcACol = 64 * kRcTiles;        // tensor memory: accumulators, then A stages
constexpr uint32_t kRcCols = 512;
constexpr int32_t kBoxRows = 256;                  // rows of one TMA box

__device__ __forceinline__ void tc_mma_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n}\n"
        ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void tc_st32(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
          "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]),
          "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}

// e4m3 population Sb[64][128 nk]: +-1.0, zero in the padding (rows r >= R,
// columns >= n); within 32 columns byte 4 s + b holds spin s + 8 b (the A
// operand's order).  Also clears the fields the recompute adds into.
__global__ void __launch_bounds__(256)
k_dense_spins_e4m3(int32_t n, int32_t R, int32_t nk, const int8_t *__restrict__ src,
                   const int32_t *__restrict__ parent, uint8_t *__restrict__ Sb, int32_t *__restrict__ H,
                   const DevCtl *__restrict__ ctl, int restart_t) {
    if (restart_t >= 0 ? !(ctl->restart && ctl->t == restart_t) : ctl->done != 0) return;
    const size_t stride = (size_t)gridDim.x * blockDim.x, x0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    const size_t words = (size_t)nk * 32, total = 64 * words;
    for (size_t x = x0; x < total; x += stride) {
        const int32_t r = (int32_t)(x / words), o = (int32_t)(x % words);
        uint32_t v = 0u;
        if (r < R) {
            const int8_t *row = src + (size_t)parent[r] * n;
            const int32_t k0 = (o >> 3) * 32 + (o & 7);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int32_t k = k0 + 8 * b;
                if (k < n) v |= (uint32_t)(((uint8_t)row[k] & 0x80u) | 0x38u) << (8 * b);
            }
        }
        reinterpret_cast<uint32_t *>(Sb)[x] = v;
    }
    for (size_t x = x0; x < (size_t)R * n; x += stride) H[x] = 0;
}

__global__ void __launch_bounds__(kRcThreads, 1)
k_dense_recompute_tc(const __grid_constant__ CUtensorMap tmJ, const __grid_constant__ CUtensorMap tmS, int32_t n,
                     int32_t R, const uint8_t *__restrict__ Sb, int32_t *__restrict__ H, DevCtl *__restrict__ ctl,
                     int restart_t) {
    if (restart_t >= 0 ? !(ctl->restart && ctl->t == restart_t) : ctl->done != 0) return;
    extern __shared__ uint8_t dsm[];
    __shared__ __align__(8) uint64_t full_bit[kRcBitStages], empty_bit[kRcBitStages], full_b[kRcBStages],
        empty_b[kRcBStages], full_a[kRcAStages], empty_a[kRcAStages], done, drained;
    __shared__ uint32_t s_tmem;
    __shared__ int s_err;
    uint8_t *base = dsm + ((1024u - (smem_u32(dsm) & 1023u)) & 1023u);
    uint8_t *bits = base, *Bst = base + kRcBitStages * kRcBitBytes;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t nk = (n + 127) / 128;                    // slices of a row
    const int32_t nch = (nk + kRcChunk - 1) / kRcChunk;    // units of a row block
    const int32_t nblk = (n + kRcRows - 1) / kRcRows;
    const int64_t units = (int64_t)nblk * nch;
    const int32_t lo = (int32_t)(units * blockIdx.x / gridDim.x), hi = (int32_t)(units * (blockIdx.x + 1) / gridDim.x);
    const uint32_t N = (uint32_t)((R + 15) & ~15);
    const uint32_t idesc = (1u << 4) | ((N >> 3) << 17) | ((128u >> 4) << 24);   // D f32, A and B e4m3, M = 128

    if (threadIdx.x == 0) {
        for (int s = 0; s < kRcBitStages; ++s) { mbar_init(&full_bit[s], 1); mbar_init(&empty_bit[s], kRcExpand); }
        for (int s = 0; s < kRcBStages; ++s) { mbar_init(&full_b[s], 1); mbar_init(&empty_b[s], 1); }
        for (int s = 0; s < kRcAStages; ++s) { mbar_init(&full_a[s], kRcExpand); mbar_init(&empty_a[s], 1); }
        mbar_init(&done, 1);
        mbar_init(&drained, kRcExpand);
        s_err = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tc_alloc(&s_tmem, kRcCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    // a bounded wait; false once a wait of any role has run out
    auto wait = [&](uint64_t *b, uint32_t parity) {
        if (!mbar_wait(b, parity)) {
            atomicCAS(&ctl->err, 0, (int)PAMC_ERR_TIMEOUT);
            *(volatile int *)&s_err = 1;
        }
        return *(volatile int *)&s_err == 0;
    };
    // the same for a whole warp (its next instructions need every lane)
    auto wait_warp = [&](uint64_t *b, uint32_t parity) { return __all_sync(0xffffffffu, wait(b, parity)) != 0; };
    auto slices = [&](int32_t u) { return min(kRcChunk, nk - (u % nch) * kRcChunk); };

    if (warp == kRcExpand) {
        if (lane == 0) {   // copies: a unit's bits one unit ahead, its population slices in turn
            int32_t ub = 0, sc = 0;
            auto copy_bits = [&](int32_t u) {
                const int s = ub % kRcBitStages, round = ub / kRcBitStages;
                if (round > 0 && !wait(&empty_bit[s], (uint32_t)((round - 1) & 1))) return false;
                uint8_t *dst = bits + (size_t)s * kRcBitBytes;
                mbar_expect_tx(&full_bit[s], (uint32_t)kRcBitBytes);
                for (int b = 0; b < kRcRows / kBoxRows; ++b)
                    tma_load_2d(dst + (size_t)b * kBoxRows * 128, &tmJ, (u % nch) * 128,
                                (u / nch) * kRcRows + b * kBoxRows, &full_bit[s]);
                ++ub;
                return true;
            };
            bool ok = lo < hi && copy_bits(lo);
            for (int32_t u = lo; ok && u < hi; ++u) {
                if (u + 1 < hi) ok = copy_bits(u + 1);
                const int32_t ns = slices(u);
                for (int32_t j = 0; ok && j < ns; ++j) {
                    const int s = sc % kRcBStages, round = sc / kRcBStages;
                    if (round > 0 && !wait(&empty_b[s], (uint32_t)((round - 1) & 1))) { ok = false; break; }
                    mbar_expect_tx(&full_b[s], N * 128u);
                    tma_load_2d(Bst + (size_t)s * kRcBBytes, &tmS, ((u % nch) * kRcChunk + j) * 128, 0, &full_b[s]);
                    ++sc;
                }
            }
            // every issued copy has landed before the CTA may leave (bounded)
            for (int32_t x = max(0, ub - kRcBitStages); x < ub; ++x)
                mbar_wait(&full_bit[x % kRcBitStages], (uint32_t)((x / kRcBitStages) & 1));
            for (int32_t x = max(0, sc - kRcBStages); x < sc; ++x)
                mbar_wait(&full_b[x % kRcBStages], (uint32_t)((x / kRcBStages) & 1));
        }
    } else if (warp == kRcExpand + 1) {
        if (lane == 0) {   // MMA issuer
            int32_t sc = 0, seg = 0;
            bool ok = true;
            for (int32_t u = lo; ok && u < hi; ++u) {
                const bool first = u == lo || u % nch == 0;
                if (first && seg > 0) {   // the accumulators of the last block have been read
                    if (!wait(&drained, (uint32_t)((seg - 1) & 1))) break;   // (nothing issued since the commit)
                    tc_fence_after();
                }
                const int32_t ns = slices(u);
                for (int32_t j = 0; j < ns; ++j) {
                    const int as = sc % kRcAStages, bs = sc % kRcBStages;
                    if (!wait(&full_b[bs], (uint32_t)((sc / kRcBStages) & 1)) ||
                        !wait(&full_a[as], (uint32_t)((sc / kRcAStages) & 1))) { ok = false; break; }
                    tc_fence_after();
                    const uint64_t bd = sw128_desc(smem_u32(Bst + (size_t)bs * kRcBBytes));
#pragma unroll
                    for (int tl = 0; tl < kRcTiles; ++tl)
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            tc_mma_ts(tmem + (uint32_t)(tl * 64),
                                      tmem + kRcACol + (uint32_t)(as * 32 * kRcTiles + tl * 32 + ks * 8),
                                      bd + (uint64_t)(2 * ks), idesc, (first && j == 0 && ks == 0) ? 0u : 1u);
                    tc_commit(&empty_a[as]);
                    tc_commit(&empty_b[bs]);
                    ++sc;
                }
                if (ok && (u + 1 == hi || (u + 1) % nch == 0)) {
                    tc_commit(&done);
                    ++seg;
                }
            }
            // every MMA issued has completed before tensor memory is freed (bounded):
            // first the last block's commit -- whatever became of the warps that
            // read it -- then what a wait that ran out left uncommitted
            if (seg > 0) mbar_wait(&done, (uint32_t)((seg - 1) & 1));
            if (!ok) {
                tc_commit(&done);
                mbar_wait(&done, (uint32_t)(seg & 1));
            }
        }
    } else {
        // expanding warps: tile warp / 4, rows 32 (warp % 4) .. + 31 of it
        const int tl = warp >> 2;
        const int32_t rr = tl * 128 + (warp & 3) * 32 + lane;
        const uint32_t lanes = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        int32_t ub = 0, sc = 0, seg = 0;
        int32_t first_ch = lo % nch;   // first unit of the current segment within its block
        bool ok = true;
        for (int32_t u = lo; ok && u < hi; ++u) {
            const int s = ub % kRcBitStages;
            if (!wait_warp(&full_bit[s], (uint32_t)((ub / kRcBitStages) & 1))) break;
            const uint8_t *rowb = bits + (size_t)s * kRcBitBytes + (size_t)rr * 128;
            const int32_t ns = slices(u);
            for (int32_t j = 0; j < ns; ++j) {
                const uint4 w4 = *reinterpret_cast<const uint4 *>(rowb + ((j ^ (rr & 7)) << 4));
                const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
                uint32_t v[32];
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int b = 0; b < 8; ++b) v[8 * q + b] = ((w[q] << (7 - b)) & 0x80808080u) ^ 0xB8B8B8B8u;
                const int as = sc % kRcAStages, round = sc / kRcAStages;
                if (round > 0 && !wait_warp(&empty_a[as], (uint32_t)((round - 1) & 1))) { ok = false; break; }
                tc_fence_after();
                tc_st32(lanes + kRcACol + (uint32_t)(as * 32 * kRcTiles + tl * 32), v);
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&full_a[as]);
                ++sc;
            }
            if (!ok) break;
            if (lane == 0) mbar_arrive(&empty_bit[s]);   // (read before the last arrival's warp barrier)
            ++ub;
            if (u + 1 == hi || (u + 1) % nch == 0) {   // the block's products are complete here
                if (!wait_warp(&done, (uint32_t)(seg & 1))) break;
                tc_fence_after();
                const int32_t row = (u / nch) * kRcRows + rr;
                const bool whole = first_ch == 0 && (u + 1) % nch == 0;
                for (uint32_t c0 = 0; c0 < N; c0 += 16) {
                    uint32_t v[16];
                    tc_ld16(lanes + (uint32_t)(tl * 64) + c0, v);
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const int r = (int)c0 + q;
                        if (row >= n || r >= R) continue;
                        int32_t h = __float2int_rn(__uint_as_float(v[q]));
                        if (first_ch == 0) {   // J_kk = 0: the clear bit counted as -1
                            const int32_t i = row & 31;
                            const uint8_t sv = Sb[(size_t)r * nk * 128 + (row & ~31) + 4 * (i & 7) + (i >> 3)];
                            h += (sv & 0x80u) ? -1 : 1;
                        }
                        if (whole) H[(size_t)r * n + row] = h;
                        else atomicAdd(&H[(size_t)r * n + row], h);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&drained);
                ++seg;
                first_ch = 0;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tc_dealloc(tmem, kRcCols);
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link
// against the driver library)
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

}  // namespace

bool dense_tc_supported() { return encode_fn() != nullptr; }

size_t dense_recompute_scratch(int32_t n) { return (size_t)64 * 128 * ((n + 127) / 128); }

// 2-D map over a row-major byte matrix of `rows` rows of `cols` bytes
// (cols a multiple of 16), box `box_rows` x 128 bytes, 128-byte swizzle.
cudaError_t dense_tc_map(void *map, const void *base, int32_t rows, int32_t cols, int32_t box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn || cols % 16 != 0 || (reinterpret_cast<uintptr_t>(base) & 15) != 0) return cudaErrorInvalidValue;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols};
    const cuuint32_t box[2] = {128u, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = fn(reinterpret_cast<CUtensorMap *>(map), CU_TENSOR_MAP_DATA_TYPE_UINT8, 2,
                          const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t dense_recompute_maps(int32_t n, int32_t R, const uint32_t *Jb, const uint8_t *Sb, void *mapJ,
                                 void *mapS) {
    cudaError_t e = dense_tc_map(mapJ, Jb, n, 4 * dense_bits_pitch(n), kBoxRows);
    if (e == cudaSuccess) e = dense_tc_map(mapS, Sb, 64, 128 * ((n + 127) / 128), (R + 15) & ~15);
    return e;
}

cudaError_t launch_dense_recompute(int32_t n, int32_t R, const void *mapJ, const void *mapS, const int8_t *src,
                                   const int32_t *parent, uint8_t *Sb, int32_t *H, DevCtl *ctl, cudaStream_t st,
                                   int restart_t) {
    if (R < 1 || R > 64) return cudaErrorInvalidValue;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int32_t nk = (n + 127) / 128;
    const size_t words = (size_t)64 * nk * 32;
    int grid = (int)((words + 255) / 256);
    if (grid > sms * 8) grid = sms * 8;
    k_dense_spins_e4m3<<<grid, 256, 0, st>>>(n, R, nk, src, parent, Sb, H, ctl, restart_t);
    const size_t smem = (size_t)kRcBitStages * kRcBitBytes + kRcBStages * kRcBBytes + 1024;
    cudaError_t e = allow_dynamic_smem(k_dense_recompute_tc, smem);
    if (e != cudaSuccess) return e;
    const int64_t units = (int64_t)((n + kRcRows - 1) / kRcRows) * ((nk + kRcChunk - 1) / kRcChunk);
    const CUtensorMap *mj = reinterpret_cast<const CUtensorMap *>(mapJ);
    const CUtensorMap *ms = reinterpret_cast<const CUtensorMap *>(mapS);
    k_dense_recompute_tc<<<(int)(units < sms ? units : sms), kRcThreads, smem, st>>>(*mj, *ms, n, R, Sb, H, ctl,
                                                                                    restart_t);
    return cudaGetLastError();
}

}  // namespace pamc
