// dense.cu -- the fully connected instance: J is an N x N int8 matrix in HBM
// (symmetric, +-1 off the diagonal, 0 on it).  Per temperature step:
//   k_dense_perm       the shared random order of each sweep (Sec. III.A):
//                      vertices sorted by (Philox key, index) -- bucket by the
//                      top key bits, then sort each bucket;
//   k_dense_tables     heat-bath T(h) (Eq. 4) or Metropolis T_M(2x) over the
//                      field range that does not saturate;
//   k_dense_recompute  H = J * S for the resampled population with
//                      mma.sync on e4m3 couplings (exact integer fields):
//                      the full recompute of every step when n is not a
//                      multiple of 16 (dense_tc.cu has the tcgen05 one);
// The sweeps themselves are in dense_sweep.cu.
#include "pamc_device.cuh"
#include "pamc_internal.h"

namespace pamc {

namespace {

// ------------------------------------------------------------------ order
constexpr int kPermThreads = 1024;
constexpr int kPermBucketBits = 11;   // 2048 buckets

// The order of each sweep by (Philox key, index) in two launches.  Bucketing
// (one CTA per sweep): keys, a histogram over the top 11 key bits, a
// block-wide exclusive scan and a scatter into buckets (order within a bucket
// arbitrary).  Sorting (32 buckets per CTA): each bucket is ranked in shared
// memory by (key, index), which is unique, so the result is the exact order.
__global__ void __launch_bounds__(kPermThreads)
k_dense_perm_bucket(int32_t n, uint32_t key0, uint32_t key1, int32_t t, uint32_t *__restrict__ skey,
                    int32_t *__restrict__ sidx, int32_t *__restrict__ boff, const DevCtl *__restrict__ ctl) {
    constexpr int NB = 1 << kPermBucketBits;
    __shared__ int32_t cnt[NB];
    __shared__ int32_t wsum[kPermThreads / 32];
    if (ctl->done) return;
    const int32_t sw = blockIdx.x;
    uint32_t *kk = skey + (size_t)sw * n;
    int32_t *ii = sidx + (size_t)sw * n;
    int32_t *bo = boff + (size_t)sw * (NB + 1);
    for (int b = threadIdx.x; b < NB; b += blockDim.x) cnt[b] = 0;
    __syncthreads();
    for (int32_t k = threadIdx.x; k < n; k += blockDim.x) {
        const uint32_t key = philox((uint32_t)k, (uint32_t)sw, (uint32_t)t, kTagPerm << 24, key0, key1).x;
        atomicAdd(&cnt[key >> (32 - kPermBucketBits)], 1);
    }
    __syncthreads();
    // exclusive scan of the NB counts: NB / blockDim consecutive buckets per thread
    constexpr int per = NB / kPermThreads;
    int32_t local[per], tot = 0;
#pragma unroll
    for (int i = 0; i < per; ++i) { local[i] = cnt[threadIdx.x * per + i]; tot += local[i]; }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t x = tot;
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int32_t v = lane < kPermThreads / 32 ? wsum[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += y;
        }
        if (lane < kPermThreads / 32) wsum[lane] = v;
    }
    __syncthreads();
    int32_t run = (x - tot) + (wid > 0 ? wsum[wid - 1] : 0);
#pragma unroll
    for (int i = 0; i < per; ++i) {
        const int b = threadIdx.x * per + i;
        bo[b] = run;
        cnt[b] = run;
        run += local[i];
    }
    if (threadIdx.x == 0) bo[NB] = n;
    __syncthreads();
    for (int32_t k = threadIdx.x; k < n; k += blockDim.x) {
        const uint32_t key = philox((uint32_t)k, (uint32_t)sw, (uint32_t)t, kTagPerm << 24, key0, key1).x;
        const int32_t p = atomicAdd(&cnt[key >> (32 - kPermBucketBits)], 1);
        kk[p] = key;
        ii[p] = k;
    }
}

constexpr int kSortBuckets = 32;        // buckets per sorting CTA
constexpr int kSortCap = 6144;          // items staged in shared memory (larger ranges sort in place)

__device__ __forceinline__ bool perm_before(uint32_t ka, int32_t ia, uint32_t kb, int32_t ib) {
    return ka < kb || (ka == kb && ia < ib);
}

__global__ void __launch_bounds__(256)
k_dense_perm_sort(int32_t n, const uint32_t *__restrict__ skey, const int32_t *__restrict__ sidx,
                  const int32_t *__restrict__ boff, int32_t *__restrict__ perm, const DevCtl *__restrict__ ctl) {
    constexpr int NB = 1 << kPermBucketBits;
    __shared__ uint32_t ks[kSortCap];
    __shared__ int32_t is[kSortCap];
    if (ctl->done) return;
    const int32_t sw = blockIdx.y;
    const uint32_t *kk = skey + (size_t)sw * n;
    const int32_t *ii = sidx + (size_t)sw * n;
    const int32_t *bo = boff + (size_t)sw * (NB + 1);
    int32_t *out = perm + (size_t)sw * n;
    const int b0 = blockIdx.x * kSortBuckets;
    const int32_t lo = bo[b0], hi = bo[b0 + kSortBuckets];
    const bool staged = hi - lo <= kSortCap;
    if (staged)
        for (int32_t x = lo + threadIdx.x; x < hi; x += blockDim.x) { ks[x - lo] = kk[x]; is[x - lo] = ii[x]; }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int b = b0 + warp; b < b0 + kSortBuckets; b += blockDim.x / 32) {
        const int32_t blo = bo[b], bhi = bo[b + 1];
        for (int32_t xi = blo + lane; xi < bhi; xi += 32) {
            const uint32_t kx = staged ? ks[xi - lo] : kk[xi];
            const int32_t ix = staged ? is[xi - lo] : ii[xi];
            int32_t rank = 0;
            for (int32_t y = blo; y < bhi; ++y) {
                const uint32_t ky = staged ? ks[y - lo] : kk[y];
                const int32_t iy = staged ? is[y - lo] : ii[y];
                rank += perm_before(ky, iy, kx, ix) ? 1 : 0;
            }
            out[blo + rank] = ix;
        }
    }
}

// ------------------------------------------------------------------ tables
// Heat-bath: tab[i] = T(i - Hc), i in [0, 2Hc]; Metropolis: tab[x] = T_M(2x),
// x in [0, Hc].  When Hc < n the table must reach saturation at its ends
// (T(Hc) = 2^32, T(-Hc) = 0; T_M(2Hc) = 0), else PAMC_ERR_RANGE.
__global__ void k_dense_tables(int rule, int32_t Hc, int32_t n, DevCtl *__restrict__ ctl,
                               uint64_t *__restrict__ tab) {
    if (ctl->done) return;
    const double beta = ctl->beta;
    const int32_t cntv = rule == 0 ? 2 * Hc + 1 : Hc + 1;
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cntv; i += gridDim.x * blockDim.x) {
        uint64_t v;
        if (rule == 0) v = thr_heatbath(beta, (int64_t)(i - Hc));
        else v = thr_metropolis(beta, 2 * (int64_t)i);
        tab[i] = v;
        if (Hc < n) {
            if (rule == 0 && i == 0 && v != 0) atomicCAS(&ctl->err, 0, (int)PAMC_ERR_RANGE);
            if (rule == 0 && i == 2 * Hc && v != (1ull << 32)) atomicCAS(&ctl->err, 0, (int)PAMC_ERR_RANGE);
            if (rule == 1 && i == Hc && v != 0) atomicCAS(&ctl->err, 0, (int)PAMC_ERR_RANGE);
        }
    }
}

// ------------------------------------------------------------------ recompute
// H[r][j] = sum_k J[j][k] S[r][k] with mma.m16n8k32 e4m3 x e4m3 -> f32.  J is
// stored in HBM as e4m3 bytes (+-1 and 0 are exact), the spins are converted
// to e4m3 while staged.  Every product is +-1 or 0 and every partial sum an
// integer of magnitude < 2^24, so the f32 result is the exact integer field
// (a GPU test sets a replica equal to a row of J, |h| = n - 1 up to 99,999,
// and compares every field with an exact product).
// A = J (row-major, K contiguous), B = S^T (column-major: each replica's spin
// row is K-contiguous).  One CTA per row slice of kRcRows rows and all
// (<= 64) replicas; K streamed through shared memory with cp.async.
constexpr int kRcWarps = 21;                  // 2 m16 tiles per warp
constexpr int kRcRows = kRcWarps * 32;        // 672 rows per CTA
constexpr int kRcK = 64;                      // K bytes per stage
constexpr int kRcStages = 3;                  // stages in flight
constexpr int kRcAStride = kRcK + 16;         // padded row stride (bank spread)
constexpr int kRcStageBytes = kRcRows * kRcAStride + 64 * kRcAStride;

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::); }
__device__ __forceinline__ void cp_async_wait_prior() { asm volatile("cp.async.wait_group 1;\n" ::); }

// +-1 int8 spins -> e4m3 (+1.0 = 0x38, -1.0 = 0xB8), four at a time
__device__ __forceinline__ uint32_t spins_to_e4m3(uint32_t x) { return (x & 0x80808080u) | 0x38383838u; }

// e4m3 coupling byte (0x38, 0xB8 or 0) -> +1, -1, 0
__device__ __forceinline__ int32_t e4m3_pm1(uint32_t b) {
    return ((int32_t)(int8_t)(uint8_t)b >> 7) | (int32_t)(b != 0u);
}

// stage kc of J rows and e4m3 spins into shared stage buffer `stage`
__device__ __forceinline__ void rc_load_stage(uint8_t *sm, const uint8_t *__restrict__ J,
                                              const int8_t *const *rowp, int32_t n, int32_t row0,
                                              int32_t kc, int stage) {
        uint8_t *As = sm + (size_t)stage * kRcStageBytes;
        uint8_t *Bs = As + (size_t)kRcRows * kRcAStride;
        const int32_t k0 = kc * kRcK;
        // each 16-byte piece is either copied asynchronously (aligned, in
        // range) or written synchronously -- never both
        for (int x = threadIdx.x; x < kRcRows * (kRcK / 16); x += blockDim.x) {
            const int rr = x / (kRcK / 16), cc = (x % (kRcK / 16)) * 16;
            const int32_t row = row0 + rr, col = k0 + cc;
            uint8_t *d = As + rr * kRcAStride + cc;
            if ((n & 15) == 0 && row < n && col + 16 <= n) {
                cp_async16(d, J + (size_t)row * n + col);
            } else {
                for (int q = 0; q < 16; ++q)
                    d[q] = (row < n && col + q < n) ? J[(size_t)row * n + col + q] : (uint8_t)0;
            }
        }
        for (int x = threadIdx.x; x < 64 * (kRcK / 16); x += blockDim.x) {
            const int rr = x / (kRcK / 16), cc = (x % (kRcK / 16)) * 16;
            const int32_t col = k0 + cc;
            const int8_t *p = rowp[rr];
            uint8_t *d = Bs + rr * kRcAStride + cc;
            // raw +-1 spins, converted to e4m3 when the fragments are read;
            // padding is harmless (J is zero there or the replica is unused)
            if (p != nullptr && col + 16 <= n && (((uintptr_t)(p + col)) & 15) == 0) {
                cp_async16(d, p + col);
            } else {
                for (int q = 0; q < 16; ++q) d[q] = (p != nullptr && col + q < n) ? (uint8_t)p[col + q] : (uint8_t)1;
            }
        }
        cp_async_commit();
    }

__global__ void __launch_bounds__(kRcWarps * 32, 1)
k_dense_recompute(int32_t n, int32_t R, const uint8_t *__restrict__ J, const int8_t *__restrict__ src,
                  const int32_t *__restrict__ parent, const int8_t *__restrict__ ncm_buf,
                  const int32_t *__restrict__ ncm_idx, int32_t *__restrict__ H,
                  const DevCtl *__restrict__ ctl, int restart_t) {
    extern __shared__ __align__(16) uint8_t sm[];
    // restart_t >= 0: only in the iteration whose controller restarted
    if (restart_t >= 0 ? !(ctl->restart && ctl->t == restart_t) : ctl->done != 0) return;
    const int32_t row0 = blockIdx.x * kRcRows;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, tig = lane & 3;
    __shared__ const int8_t *rowp[64];
    if (threadIdx.x < 64) {
        const int r = threadIdx.x;
        const int8_t *p = nullptr;
        if (r < R) {
            const int32_t q = ncm_idx[r];
            p = q >= 0 ? ncm_buf + (size_t)q * n : src + (size_t)parent[r] * n;
        }
        rowp[r] = p;
    }
    __syncthreads();
    float acc[2][8][4];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.f;

    const int32_t nk = (n + kRcK - 1) / kRcK;
    for (int st = 0; st < kRcStages - 1; ++st) {
        if (st < nk) rc_load_stage(sm, J, rowp, n, row0, st, st);
        else cp_async_commit();
    }
    for (int32_t kc = 0; kc < nk; ++kc) {
        // keep kRcStages-1 stages in flight
        if (kc + kRcStages - 1 < nk)
            rc_load_stage(sm, J, rowp, n, row0, kc + kRcStages - 1, (kc + kRcStages - 1) % kRcStages);
        else
            cp_async_commit();
        asm volatile("cp.async.wait_group %0;\n" ::"n"(kRcStages - 1));
        __syncthreads();
        const uint8_t *As = sm + (size_t)(kc % kRcStages) * kRcStageBytes;
        const uint8_t *Bs = As + (size_t)kRcRows * kRcAStride;
#pragma unroll
        for (int ks = 0; ks < kRcK; ks += 32) {
            uint32_t a[2][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                const uint8_t *ar = As + (size_t)(warp * 32 + mt * 16 + g) * kRcAStride + ks + tig * 4;
                a[mt][0] = *reinterpret_cast<const uint32_t *>(ar);
                a[mt][1] = *reinterpret_cast<const uint32_t *>(ar + 8 * kRcAStride);
                a[mt][2] = *reinterpret_cast<const uint32_t *>(ar + 16);
                a[mt][3] = *reinterpret_cast<const uint32_t *>(ar + 8 * kRcAStride + 16);
            }
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                const uint8_t *br = Bs + (size_t)(nt * 8 + g) * kRcAStride + ks + tig * 4;
                const uint32_t b0 = spins_to_e4m3(*reinterpret_cast<const uint32_t *>(br));
                const uint32_t b1 = spins_to_e4m3(*reinterpret_cast<const uint32_t *>(br + 16));
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    asm volatile(
                        "mma.sync.aligned.m16n8k32.row.col.f32.e4m3.e4m3.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
                        "{%8,%9}, {%0,%1,%2,%3};\n"
                        : "+f"(acc[mt][nt][0]), "+f"(acc[mt][nt][1]), "+f"(acc[mt][nt][2]),
                          "+f"(acc[mt][nt][3])
                        : "r"(a[mt][0]), "r"(a[mt][1]), "r"(a[mt][2]), "r"(a[mt][3]), "r"(b0), "r"(b1));
                }
            }
        }
        __syncthreads();
    }
    cp_async_wait_all();
    // C fragment: rows g / g+8, columns (replicas) 2*tig, 2*tig+1
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 8; ++nt)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int32_t row = row0 + warp * 32 + mt * 16 + g + (c >= 2 ? 8 : 0);
                const int r = nt * 8 + tig * 2 + (c & 1);
                if (row < n && r < R) H[(size_t)r * n + row] = __float2int_rn(acc[mt][nt][c]);
            }
}

// E_r = -1/2 sum_j s_j h_j from recomputed fields (one CTA per replica)
__global__ void k_dense_energy_from_H(int32_t n, const int32_t *__restrict__ H,
                                      const int8_t *__restrict__ spins, int64_t *__restrict__ E,
                                      const DevCtl *__restrict__ ctl, int restart_t) {
    __shared__ long long red[32];
    if (restart_t >= 0 ? !(ctl->restart && ctl->t == restart_t) : ctl->done != 0) return;
    const int r = blockIdx.x;
    long long acc = 0;
    for (int32_t j = threadIdx.x; j < n; j += blockDim.x)
        acc += (long long)spins[(size_t)r * n + j] * H[(size_t)r * n + j];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long tot = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
        E[r] = -(tot / 2);
    }
}

// Max-Cut weights -> couplings in place (J = -w), and W = sum_{i<j} w_ij.
__global__ void k_dense_negate_sum(size_t total, int8_t *__restrict__ J,
                                   unsigned long long *__restrict__ wsum) {
    long long acc = 0;
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < total;
         x += (size_t)gridDim.x * blockDim.x) {
        const int8_t v = J[x];
        acc += v;
        J[x] = (int8_t)(-v);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0 && acc != 0) atomicAdd(wsum, (unsigned long long)acc);
}

// int8 couplings (validated +-1 / 0) -> e4m3 bytes in place
__global__ void k_dense_to_e4m3(size_t total, uint8_t *__restrict__ J) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < total;
         x += (size_t)gridDim.x * blockDim.x) {
        const int8_t v = (int8_t)J[x];
        J[x] = v == 0 ? (uint8_t)0 : (v > 0 ? (uint8_t)0x38 : (uint8_t)0xB8);
    }
}

// Validation of a device-resident copy: entries in {-1, 0, +1}, zero diagonal,
// +-1 off the diagonal, symmetric.  32x32 tiles compared with their transpose.
__global__ void k_dense_validate(int32_t n, const int8_t *__restrict__ J, int *__restrict__ err) {
    __shared__ int8_t tl[32][33];
    const int32_t bi = blockIdx.y * 32, bj = blockIdx.x * 32;
    if (bj < bi) return;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int yy = ty; yy < 32; yy += blockDim.x / 32) {
        const int32_t i = bj + yy, j = bi + tx;
        tl[yy][tx] = (i < n && j < n) ? J[(size_t)i * n + j] : 0;
    }
    __syncthreads();
    for (int yy = ty; yy < 32; yy += blockDim.x / 32) {
        const int32_t i = bi + yy, j = bj + tx;
        if (i < n && j < n) {
            const int8_t v = J[(size_t)i * n + j];
            if (i == j) { if (v != 0) atomicCAS(err, 0, (int)PAMC_ERR_DIAG); }
            else if (v != 1 && v != -1) atomicCAS(err, 0, (int)PAMC_ERR_RANGE);
            else if (v != tl[tx][yy]) atomicCAS(err, 0, (int)PAMC_ERR_ASYM);
        }
    }
}

}  // namespace

cudaError_t launch_dense_validate(int32_t n, const int8_t *J, int *err, cudaStream_t st) {
    const int nt = (n + 31) / 32;
    k_dense_validate<<<dim3(nt, nt), 256, 0, st>>>(n, J, err);
    return cudaGetLastError();
}

cudaError_t launch_dense_perm(int32_t n, uint64_t seed, int32_t t, int32_t S, int32_t *perm,
                              uint32_t *skey, int32_t *sidx, int32_t *boff, const DevCtl *ctl, cudaStream_t st) {
    if (S <= 0) return cudaSuccess;
    k_dense_perm_bucket<<<S, kPermThreads, 0, st>>>(n, (uint32_t)seed, (uint32_t)(seed >> 32), t, skey, sidx,
                                                   boff, ctl);
    k_dense_perm_sort<<<dim3((1 << kPermBucketBits) / kSortBuckets, S), 256, 0, st>>>(n, skey, sidx, boff, perm,
                                                                                       ctl);
    return cudaGetLastError();
}

size_t dense_perm_offsets(int32_t S) { return (size_t)S * ((1 << kPermBucketBits) + 1); }

cudaError_t launch_dense_tables(int rule, int32_t Hc, int32_t n, DevCtl *ctl, uint64_t *tab,
                                cudaStream_t st) {
    const int32_t cntv = rule == 0 ? 2 * Hc + 1 : Hc + 1;
    int grid = (cntv + 255) / 256;
    if (grid > 304) grid = 304;
    k_dense_tables<<<grid, 256, 0, st>>>(rule, Hc, n, ctl, tab);
    return cudaGetLastError();
}

size_t dense_recompute_smem() { return (size_t)kRcStages * kRcStageBytes; }

cudaError_t launch_dense_recompute(int32_t n, int32_t R, const int8_t *J, const int8_t *src,
                                   const int32_t *parent, const int8_t *ncm_buf,
                                   const int32_t *ncm_idx, int32_t *H, const DevCtl *ctl,
                                   cudaStream_t st, int restart_t) {
    const size_t smem = dense_recompute_smem();
    cudaError_t e = allow_dynamic_smem(k_dense_recompute, smem);
    if (e != cudaSuccess) return e;
    const int grid = (n + kRcRows - 1) / kRcRows;
    k_dense_recompute<<<grid, kRcWarps * 32, smem, st>>>(n, R, reinterpret_cast<const uint8_t *>(J), src,
                                                           parent, ncm_buf, ncm_idx, H, ctl, restart_t);
    return cudaGetLastError();
}

cudaError_t launch_dense_energy(int32_t n, int32_t R, const int32_t *H, const int8_t *spins, int64_t *E,
                                const DevCtl *ctl, cudaStream_t st, int restart_t) {
    k_dense_energy_from_H<<<R, 512, 0, st>>>(n, H, spins, E, ctl, restart_t);
    return cudaGetLastError();
}

cudaError_t launch_dense_to_e4m3(size_t total, int8_t *J, cudaStream_t st) {
    k_dense_to_e4m3<<<152 * 8, 256, 0, st>>>(total, reinterpret_cast<uint8_t *>(J));
    return cudaGetLastError();
}

cudaError_t launch_dense_negate_sum(size_t total, int8_t *J, unsigned long long *wsum, cudaStream_t st) {
    k_dense_negate_sum<<<152 * 8, 256, 0, st>>>(total, J, wsum);
    return cudaGetLastError();
}

}  // namespace pamc
