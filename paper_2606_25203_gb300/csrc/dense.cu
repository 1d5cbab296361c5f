// dense.cu -- the fully connected instance: J is N x N, symmetric, +-1 off the
// diagonal and 0 on it.  Per temperature step:
//   k_dense_perm       the shared random order of each sweep (Sec. III.A):
//                      vertices sorted by (Philox key, index) -- bucket by the
//                      top key bits, then sort each bucket;
//   k_dense_tables     heat-bath T(h) (Eq. 4) or Metropolis T_M(2x) over the
//                      field range that does not saturate;
//   k_dense_energy_from_H  energies from the fields.
// The instance arrives as int8 weights and is kept as a bit matrix
// (k_dense_pack, k_dense_symmetric).  The recompute H = J S of every step is
// in dense_tc.cu, the sweeps in dense_sweep.cu.
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

// ------------------------------------------------------------------ instance
// Rows i0 .. i0 + rows - 1 of the Max-Cut weights (row pitch n) -> the bit
// matrix (bit set where J = -w = +1, i.e. w < 0; the diagonal and the padding
// clear).  Entries must be +-1 off the diagonal and 0 on it.  *neg counts the
// negative weights.  A warp packs 512 columns at a time with 16-byte loads
// where the rows allow them (n a multiple of 16, aligned base), else 32.
__global__ void __launch_bounds__(256)
k_dense_pack(int32_t n, int32_t pitch, int32_t i0, int32_t rows, const int8_t *__restrict__ w, int vec,
             uint32_t *__restrict__ Jb, unsigned long long *__restrict__ neg, int *__restrict__ err) {
    const int lane = threadIdx.x & 31;
    const int32_t gw = (int32_t)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    const int32_t nw = (int32_t)(gridDim.x * (blockDim.x >> 5));
    unsigned long long cnt = 0;
    int bad = 0;
    for (int32_t ir = gw; ir < rows; ir += nw) {
        const int32_t i = i0 + ir;
        const int8_t *row = w + (size_t)ir * n;
        uint32_t *out = Jb + (size_t)i * pitch;
        if (vec) {
            for (int32_t c0 = 0; c0 < 32 * pitch; c0 += 512) {
                const int32_t c = c0 + 16 * lane;
                uint32_t bits = 0u;
                if (c < n) {
                    const uint4 x4 = *reinterpret_cast<const uint4 *>(row + c);
                    uint32_t x[4] = {x4.x, x4.y, x4.z, x4.w};
                    if (i >= c && i < c + 16) {   // the diagonal entry: 0, then any valid value
                        const int q = (i - c) >> 2, b = 8 * ((i - c) & 3);
#pragma unroll
                        for (int p = 0; p < 4; ++p)
                            if (p == q) {
                                if ((x[p] >> b) & 0xFFu) bad = PAMC_ERR_DIAG;
                                x[p] = (x[p] & ~(0xFFu << b)) | (1u << b);
                            }
                    }
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const uint32_t m = (x[p] >> 7) & 0x01010101u;   // sign bits
                        if ((x[p] ^ (m * 0xFEu)) != 0x01010101u && !bad) bad = PAMC_ERR_RANGE;
                        bits |= ((m * 0x01020408u) >> 24 & 0xFu) << (4 * p);
                    }
                }
                const uint32_t hi = __shfl_down_sync(0xffffffffu, bits, 1);
                if (!(lane & 1) && (c >> 5) < pitch) {
                    out[c >> 5] = bits | (hi << 16);
                    cnt += __popc(bits | (hi << 16));
                }
            }
        } else {
            for (int32_t c0 = 0; c0 < 32 * pitch; c0 += 32) {
                const int32_t c = c0 + lane;
                const int8_t v = c < n ? row[c] : (int8_t)0;
                if (c < n) {
                    if (c == i) { if (v != 0) bad = PAMC_ERR_DIAG; }
                    else if (v != 1 && v != -1 && !bad) bad = PAMC_ERR_RANGE;
                }
                const uint32_t bits = __ballot_sync(0xffffffffu, c != i && v < 0);
                if (lane == 0) {
                    out[c0 >> 5] = bits;
                    cnt += __popc(bits);
                }
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
    if (lane == 0 && cnt != 0) atomicAdd(neg, cnt);
    if (bad) atomicCAS(err, 0, bad);
}

// Symmetry of the bit matrix: a warp compares a 32 x 32 block with the
// transpose of its mirror block (32 ballots).
__global__ void __launch_bounds__(256)
k_dense_symmetric(int32_t n, int32_t pitch, const uint32_t *__restrict__ Jb, int *__restrict__ err) {
    const int lane = threadIdx.x & 31;
    const int32_t nb = (n + 31) / 32;
    const int32_t bi = blockIdx.y, bj = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (bj >= nb || bj < bi) return;
    const int32_t ri = bi * 32 + lane, rj = bj * 32 + lane;
    const uint32_t a = ri < n ? Jb[(size_t)ri * pitch + bj] : 0u;
    const uint32_t b = rj < n ? Jb[(size_t)rj * pitch + bi] : 0u;
    uint32_t t = 0u;   // row lane of the mirror block, from the columns of this one
#pragma unroll
    for (int q = 0; q < 32; ++q) {
        const uint32_t col = __ballot_sync(0xffffffffu, (a >> q) & 1u);
        if (lane == q) t = col;
    }
    if (t != b) atomicCAS(err, 0, (int)PAMC_ERR_ASYM);
}

}  // namespace

cudaError_t launch_dense_pack(int32_t n, int32_t i0, int32_t rows, const int8_t *w, uint32_t *Jb,
                              unsigned long long *neg, int *err, cudaStream_t st) {
    const int vec = n % 16 == 0 && (reinterpret_cast<uintptr_t>(w) & 15) == 0 ? 1 : 0;
    int grid = (rows + 7) / 8;
    if (grid > 152 * 8) grid = 152 * 8;
    k_dense_pack<<<grid, 256, 0, st>>>(n, dense_bits_pitch(n), i0, rows, w, vec, Jb, neg, err);
    return cudaGetLastError();
}

cudaError_t launch_dense_symmetric(int32_t n, const uint32_t *Jb, int *err, cudaStream_t st) {
    const int32_t nb = (n + 31) / 32;
    k_dense_symmetric<<<dim3((nb + 7) / 8, nb), 256, 0, st>>>(n, dense_bits_pitch(n), Jb, err);
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

cudaError_t launch_dense_energy(int32_t n, int32_t R, const int32_t *H, const int8_t *spins, int64_t *E,
                                const DevCtl *ctl, cudaStream_t st, int restart_t) {
    k_dense_energy_from_H<<<R, 512, 0, st>>>(n, H, spins, E, ctl, restart_t);
    return cudaGetLastError();
}

}  // namespace pamc
