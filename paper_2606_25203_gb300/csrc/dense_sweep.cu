// dense_sweep.cu -- S sequential single-spin sweeps (Eq. 3-4) of the fully
// connected +-1 instance, every replica on its own: one thread-block cluster
// per replica holds the replica's n integer fields and spins in shared memory
// (each CTA a slice of the vertices), so no replica waits for another and
// there is no grid-wide barrier.  All replicas visit the vertices in the same
// order (the shared permutation of the sweep), so the coupling rows they need
// meet in L2.  The couplings are read from the bit matrix (one bit per
// coupling, +1 set; the diagonal bit is 0 and corrected for): a row of n =
// 100,000 is 12.5 KB instead of 100 KB.
//
// Exact batches.  A flip changes every other field by +-2.  The decisions of
// the next B positions are evaluated at once from the current fields with
// their draws; a position is a candidate when it would flip now, or when some
// field change of at most 2 m (m flips) could change its decision (the
// acceptance thresholds are monotone in the field, so comparing the draw with
// the thresholds at h - 2m and h + 2m decides that; at a negative beta they
// fall with the field, and the heat-bath decisions read the table at -h).  Every
// other position keeps its spin whatever the first m flips of the batch are.  The candidates
// (at most kCand, in order) are then decided one after the other by one warp
// from their fields and the bit tile of the couplings among them; before a
// flip m + 1 the batch ends and the next one starts at that position.  The
// flipped rows are applied to all fields of the slice in one pass.  So the
// result is the sequential sweep's, position by position.  B and m follow
// what the last batch saw.
//
// A batch's decisions are taken in every CTA of the cluster alike (margins and
// tile go to all of them), by warp 0, a candidate a lane with its tile row in
// registers.  Four warps request the slice's part of the rows that flip by bulk
// copies as they are decided; the others wait on a hardware barrier (polling
// warps took two thirds of the deciding warp's issue slots: 560 cycles a flip,
// 165 now), then count the rows bit-sliced from shared memory.
//
// Fields are kept as h / 2 in 16 bits, two a word (one parity; a field moves by
// 2): half the pass over them, and room for the rows.  Up to n = 65,000 they
// always fit.  Beyond, the largest field bounds the flips until one could not;
// when it does, the replica stops there and a second launch, otherwise empty,
// goes on with 32-bit fields from that position.
//
// Bounds.  An evaluation is one Philox call and up to three table reads per
// position; a batch with candidates adds a gather of single bits (one miss
// latency), its decisions one after the other, the latency of the last rows and a
// pass over the slice's fields.  Hot steps are bound by these per batch (of 50
// flips at n = 100,000: decisions 9, gather 10, rows and pass 20 thousand cycles),
// cold ones by the latencies of a few dozen batches.  ms of a whole step, two
// sweeps, R = 64, first (hottest) step / mean of a 20-step anneal; before: a design
// that advanced all replicas together, a grid barrier after each 256 positions, on
// byte couplings: n = 100,000 22.9 / 4.06 (24.1 / 10.7 before), n = 40,000 7.1 / 1.24
// (9.1 / 3.8), n = 10,000 1.57 / 0.33 (2.33 / 0.94), n = 2,048 0.40 / 0.13 (0.54 /
// 0.22), n = 5,001 (odd) 0.83 / 0.20 (13.2 / 2.2).
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdlib>

#include "pamc_device.cuh"
#include "pamc_internal.h"
#include "tc_sm100.cuh"

namespace cg = cooperative_groups;

namespace pamc {

namespace {

constexpr int kDsThreads = 1024;
constexpr int kEval = 4;                          // positions a thread evaluates in a batch
constexpr int kBatchMax = kDsThreads * kEval;     // positions of the largest batch
constexpr int kBatchMin = 64;
constexpr int kCand = 128;                        // candidates of a batch
constexpr int kFlipMax = 63;                      // flips of a batch (six count planes)
constexpr int kDsWin = 2048;                      // threshold entries in shared memory
constexpr int kMaxCluster = 8;
constexpr int kFetch = 4;                         // warps that request flipped rows (warp 0 decides)
constexpr int kApply = kDsThreads / 32 - 1 - kFetch;   // warps that apply them
constexpr int kWordsMax = 2 * 32 * kApply;        // row words of the widest slice: two a thread
constexpr int kRowsMax = 64;                      // rows in flight
constexpr int kChunkMax = 16;                     // chunks of rows in flight (a power of two of them)
// fields in 16 bits hold h / 2 in [-32768, 32767]: at every n up to here
constexpr int32_t kHalfAlways = 65000;

struct DenseSweepArgs {
    int32_t n, R, S, rule, Hc;
    int32_t per;              // vertices of a CTA's slice (a multiple of 32)
    int32_t pitch;            // 32-bit words of a row of the bit matrix
    int32_t t, gbase;
    PhiloxKeys K;
    const uint32_t *Jb;       // bit matrix
    const int32_t *perm;      // [S][n]
    const uint64_t *tab;
    const int8_t *src;        // previous population (resampling parents)
    const int32_t *parent;
    int32_t *H;               // [R][n] in: recomputed fields; out: fields after the sweeps
    int8_t *dst;              // [R][n]
    int64_t *E;               // [R]
    uint32_t *rowbits;        // [S][ceil(n / 32)] positions that flipped in some replica, zeroed
    int2 *resume;             // [R] n > kHalfAlways: where 32-bit fields take over (sweep, position; sweep S: nowhere)
    DevCtl *ctl;
    int32_t chunks;           // chunks of the row ring
    int32_t half_max;         // 16-bit fields: |h| / 2 stays within this, checked (0: it always does)
};

// What a batch decided (the same in every CTA of the cluster).
struct BatchOut {
    int32_t nflip, next, bsize, mcap;
    uint32_t flip[64];        // candidate | (1 << 31 when the spin turned to -1)
    uint32_t neg[2];          // the flips that turned to -1, one bit each
};

struct DsSmem {               // fixed part of a CTA's shared memory
    uint32_t win[kDsWin];
    uint32_t bm[3][kBatchMax / 32];   // candidate bits of a batch, in turn
    int32_t ck[kCand], cp[kCand];     // candidates: vertex, position
    int32_t cq[kCand];                // 2 (margin) + spin bit, see below
    uint4 tile[kCand];                // J[candidate][candidate], one bit each
    BatchOut out;
    uint64_t full[kChunkMax], empty[kChunkMax];   // the row ring's barriers
    int32_t decided, final;           // flips of the batch so far; all of them (-1: not known yet)
    int32_t lo, hi, dir, hmax, err;
    unsigned long long esum;
};

// u < T(x): x = dir h (heat-bath, dir = -1 at a negative beta: T rising with x)
// or s h (Metropolis, T falling with x).  Inside [lo, hi) the threshold lies
// strictly between 0 and 2^32.
struct Accept {
    const uint32_t *win;
    const uint64_t *tab;
    int32_t lo, hi, off, rising, dir;
    bool inwin;
    __device__ __forceinline__ bool operator()(int32_t x, uint32_t u) const {
        if (x < lo) return !rising;
        if (x >= hi) return rising;
        // all fields of a run have the parity of n - 1, so every other entry is kept
        return inwin ? u < win[(x - lo) >> 1] : (uint64_t)u < tab[dir * x + off];
    }
    // whether the visit flips spin s (0 or 1) at field h
    __device__ __forceinline__ bool flips(int32_t h, uint32_t s, uint32_t u) const {
        if (rising) return (*this)(dir * h, u) != (s != 0u);
        return (*this)(s ? h : -h, u);
    }
    // whether some field within m of h decides differently from another
    __device__ __forceinline__ bool fragile(int32_t h, uint32_t s, uint32_t u, int32_t m) const {
        const int32_t x = rising ? dir * h : s ? h : -h;
        return (*this)(x - m, u) != (*this)(x + m, u);
    }
    // margin of the decision in flips of other spins: with v = dir h (s = -1) or
    // -dir h (s = +1) the visit flips s iff v is at least some value (both rules),
    // a field changes by 2 a flip, and q >= 0 iff it flips now: the largest
    // number of adverse flips it survives, or minus the favourable ones it
    // needs; clamped to [-m - 1, m]
    __device__ __forceinline__ int32_t margin(int32_t h, uint32_t s, uint32_t u, int32_t m) const {
        int32_t lo2 = -m, hi2 = m + 1;   // smallest x in [-m, m] at which v + 2x flips, m + 1 if none
        while (lo2 < hi2) {
            const int32_t mid = (lo2 + hi2) >> 1;
            if (flips(s ? h - 2 * dir * mid : h + 2 * dir * mid, s, u)) hi2 = mid;
            else lo2 = mid + 1;
        }
        return -lo2;
    }
};

__device__ __forceinline__ void full_add(uint32_t a, uint32_t b, uint32_t c, uint32_t &sum, uint32_t &carry) {
    sum = a ^ b ^ c;
    carry = (a & b) | (c & (a ^ b));
}

__device__ __forceinline__ void st_release(int32_t *p, int32_t v) {
    asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ int32_t ld_acquire(const int32_t *p) {
    int32_t v;
    asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
// The smallest i in [0, len) with past(i), len if none (past: false, then true),
// by one warp: 32 probes at a time.
template <class F>
__device__ __forceinline__ int32_t first_past(int32_t len, int lane, F &&past) {
    int32_t lo = 0, hi = len;
    while (lo < hi) {
        const int32_t step = (hi - lo + 31) >> 5, p = lo + (lane + 1) * step - 1;
        const uint32_t m = __ballot_sync(0xffffffffu, p >= hi || past(p));
        if (m == 0u) return hi;
        const int x = __ffs(m) - 1;
        hi = min(hi, lo + (x + 1) * step - 1);
        lo += x * step;
    }
    return lo;
}

__host__ __device__ __forceinline__ int32_t ds_slice(int32_t n, int cs) { return ((n + cs - 1) / cs + 127) & ~127; }
// bytes of a slice's fields: 32 (16, two to a word) rows of a field a word
__host__ __device__ __forceinline__ size_t ds_field_bytes(int32_t nW, bool half) {
    return (size_t)(half ? 16 : 32) * (nW | 1) * 4;
}
__host__ __device__ __forceinline__ size_t ds_ring_offset(int32_t nW, bool half) {
    const size_t fixed = (sizeof(DsSmem) + 15) & ~(size_t)15;
    return (fixed + ds_field_bytes(nW, half) + (size_t)nW * 4 + 127) & ~(size_t)127;
}

// CL: clusters of more than one CTA; HALF: 16-bit fields; CH: rows of a chunk;
// RESUME: take up what 16-bit fields left.
template <bool CL, bool HALF, int CH, bool RESUME>
__global__ void __launch_bounds__(kDsThreads, 1) k_dense_sweep(DenseSweepArgs a, int cs) {
    extern __shared__ __align__(128) uint8_t smraw[];
    DsSmem &sm = *reinterpret_cast<DsSmem *>(smraw);
    const int32_t per = a.per, nW = per >> 5, nWp = nW | 1;
    // fields: vertex a0 + 32 w + b at Hs[b * nWp + w] (a thread's 32 fields of
    // one row word lie in 32 rows, consecutive words in consecutive banks); HALF:
    // (h - parity) / 2 + 32768 in half b / 16 of the word at Hs[(b % 16) * nWp + w]
    uint32_t *Hs = reinterpret_cast<uint32_t *>(smraw + ((sizeof(DsSmem) + 15) & ~(size_t)15));
    uint32_t *bits = reinterpret_cast<uint32_t *>(reinterpret_cast<uint8_t *>(Hs) + ds_field_bytes(nW, HALF));
    uint8_t *ring = smraw + ds_ring_offset(nW, HALF);   // [chunks][CH][nW] row words
    if (a.ctl->done) return;   // uniform over the grid

    const int32_t n = a.n;
    const int crank = CL ? (int)(blockIdx.x % cs) : 0;
    const int r = CL ? (int)(blockIdx.x / cs) : (int)blockIdx.x;
    int32_t sw0 = 0, p0 = 0;
    if constexpr (RESUME) {
        const int2 from = a.resume[r];
        if (from.x >= a.S) return;   // uniform over the cluster
        sw0 = from.x;
        p0 = from.y;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t a0 = min(n, crank * per), a1 = min(n, a0 + per);
    const int32_t par = (n - 1) & 1;                    // the fields' parity
    const bool checked = HALF && a.half_max != 0;       // a field may outgrow 16 bits
    auto sync_all = [&]() {
        if constexpr (CL) cg::this_cluster().sync();
        else __syncthreads();
    };
    // the same shared-memory address in CTA c of the cluster
    auto at = [&](auto *p, int c) {
        if constexpr (CL) return cg::this_cluster().map_shared_rank(p, c);
        else return p;
    };
    const int nctas = CL ? cs : 1;
    auto field = [&](int32_t j) -> int32_t {
        if constexpr (HALF) return 2 * ((int32_t)((Hs[(j & 15) * nWp + (j >> 5)] >> (j & 16)) & 0xFFFFu) - 32768) + par;
        else return (int32_t)Hs[(j & 31) * nWp + (j >> 5)];
    };

    const int appliers = min(kApply, (nW + 31) >> 5);   // apply warps with words of the slice
    // ---------------- prologue: spins, fields, thresholds
    if (threadIdx.x == 0) {
        for (int c = 0; c < a.chunks; ++c) { mbar_init(&sm.full[c], 1); mbar_init(&sm.empty[c], (uint32_t)appliers); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sm.hmax = 0;
        sm.err = 0;
    }
    const int8_t *row = RESUME ? a.dst + (size_t)r * n : a.src + (size_t)a.parent[r] * n;
    int32_t hmax = 0;   // largest |h| of the fields loaded by this thread
    for (int32_t w = warp; w < nW; w += kDsThreads / 32) {
        const int32_t k = a0 + 32 * w + lane;
        const uint32_t b = __ballot_sync(0xffffffffu, k < a1 && row[min(k, n - 1)] > 0);
        const int32_t h = k < a1 ? a.H[(size_t)r * n + k] : 0;
        if constexpr (HALF) {
            hmax = max(hmax, abs(h));
            const uint32_t q = (uint32_t)(((k < a1 ? h - par : 0) >> 1) + 32768) & 0xFFFFu;
            const uint32_t hi = __shfl_down_sync(0xffffffffu, q, 16);
            if (lane < 16) Hs[lane * nWp + w] = q | (hi << 16);
        } else {
            Hs[lane * nWp + w] = (uint32_t)h;
        }
        if (lane == 0) bits[w] = b;
    }
    for (int32_t i = threadIdx.x; i < 3 * (kBatchMax / 32); i += kDsThreads) (&sm.bm[0][0])[i] = 0u;
    // [lo, hi): where the threshold is neither 0 nor 2^32, one warp each
    if (warp < 2) {
        const int32_t last = a.rule == 0 ? 2 * a.Hc : a.Hc;
        // heat-bath: tab[i] = T(i - Hc), rising (falling at a negative beta: read
        // from its end); Metropolis: tab[x] = T_M(2x), falling from tab[0] = 2^32
        const bool back = a.rule == 0 && a.tab[0] > a.tab[last];
        const bool zero = a.rule == 0 ? warp == 0 : warp == 1;   // the end where thresholds are 0
        auto past = [&](int32_t i) {
            const uint64_t T = a.tab[back ? last - i : i];
            return a.rule == 0 ? (zero ? T > 0ull : T >= (1ull << 32)) : zero ? T == 0ull : T < (1ull << 32);
        };
        const int32_t x = first_past(last + 1, lane, past) - (a.rule == 0 ? a.Hc : 0);
        if (lane == 0) {
            if (warp == 0) {
                sm.lo = x + ((x ^ (n - 1)) & 1);   // the fields' parity
                sm.dir = back ? -1 : 1;
                sm.esum = 0ull;
            } else {
                sm.hi = x;
            }
        }
    }
    __syncthreads();
    const int32_t nwin = (max(sm.hi, sm.lo) - sm.lo + 1) >> 1;
    Accept acc{sm.win, a.tab, sm.lo, max(sm.hi, sm.lo), a.rule == 0 ? a.Hc : 0, a.rule == 0 ? 1 : 0, sm.dir,
               nwin <= kDsWin};
    if (acc.inwin)
        for (int32_t i = threadIdx.x; i < nwin; i += kDsThreads) sm.win[i] = (uint32_t)a.tab[acc.dir * (acc.lo + 2 * i) + acc.off];
    const int32_t nrw = (n + 31) >> 5;
    const uint32_t ctr3 = (kTagFlip << 24) | (uint32_t)((r >> 2) + a.gbase);
    sync_all();   // every CTA of the cluster runs before another one writes its memory
    // checked: flips until a field of the replica could outgrow its 16 bits (the
    // same in every CTA): from the largest |h| over the cluster
    int32_t room = 0x7fffffff;
    auto bound_fields = [&]() {
        const int32_t m = (int32_t)__reduce_max_sync(0xffffffffu, (unsigned)hmax);
        if (lane == 0)
            for (int c = 0; c < nctas; ++c) atomicMax(at(&sm.hmax, c), m);
        sync_all();
        room = a.half_max - (sm.hmax + 1) / 2;
        sync_all();
        if (threadIdx.x == 0) sm.hmax = 0;   // (set again after more barriers)
    };

    int32_t bsize = 512, mcap = 8, sw = sw0;
    int buf = 0;
    uint32_t chunk0 = 0;    // the ring: chunks of the batches before
    const uint32_t cmask = (uint32_t)a.chunks - 1u;
    const int clog = 31 - __clz(a.chunks);
    bool held = true, stopped = false;   // checked: the fields loaded fit 16 bits; 32-bit fields go on
    if (checked) {
        bound_fields();
        held = room >= 64;
        stopped = !held;
    }
    for (; sw < a.S && !stopped; p0 = stopped ? p0 : 0, sw += stopped ? 0 : 1) {
        const int32_t *perm = a.perm + (size_t)sw * n;
        while (p0 < n) {
            if (checked && room < 64) {   // (uniform over the cluster)
                hmax = 0;
                for (int32_t i = threadIdx.x; i < 16 * nW; i += kDsThreads) {
                    const uint32_t v = Hs[(i / nW) * nWp + i % nW];
                    hmax = max(hmax, 2 * max(abs((int32_t)(v & 0xFFFFu) - 32768), abs((int32_t)(v >> 16) - 32768)) + 1);
                }
                bound_fields();
                if (room < 64) {
                    stopped = true;
                    break;
                }
            }
            const int32_t B = min(bsize, n - p0), nbw = (B + 31) >> 5;
            uint32_t *bm = sm.bm[buf];
            // ---- evaluate the own vertices among the next B positions
            int32_t kk[kEval];
            uint32_t uu[kEval];
#pragma unroll
            for (int e = 0; e < kEval; ++e) {
                const int32_t i = e * kDsThreads + (int32_t)threadIdx.x;
                kk[e] = -1;
                uu[e] = 0u;
                if (i < B) kk[e] = perm[p0 + i];
            }
#pragma unroll
            for (int e = 0; e < kEval; ++e) {
                if (e * kDsThreads >= B) break;   // uniform
                const int32_t k = kk[e];
                bool cand = false;
                if (k >= a0 && k < a1) {
                    const u32x4 x = philox_rk((uint32_t)k, (uint32_t)sw, (uint32_t)a.t, ctr3, a.K);
                    const uint32_t u = (r & 2) ? ((r & 1) ? x.w : x.z) : ((r & 1) ? x.y : x.x);
                    const int32_t j = k - a0;
                    const int32_t h = field(j);
                    const uint32_t s = (bits[j >> 5] >> (j & 31)) & 1u;
                    uu[e] = u;
                    cand = acc.flips(h, s, u) || acc.fragile(h, s, u, 2 * mcap);
                }
                const uint32_t word = __ballot_sync(0xffffffffu, cand);
                const int32_t w = e * (kDsThreads / 32) + warp;
                if (!CL) {
                    if (lane == 0 && w < nbw) bm[w] = word;
                } else if (lane == 0 && w < nbw && word != 0u) {
                    for (int c = 0; c < cs; ++c) atomicOr(at(&bm[w], c), word);
                }
            }
            sync_all();
            // the words of the batch after next are cleared here: no CTA sets
            // them before every CTA has passed the next batch's first barrier
            const int nbuf = buf == 2 ? 0 : buf + 1;
            if (CL && (int32_t)threadIdx.x < kBatchMax / 32) sm.bm[nbuf == 2 ? 0 : nbuf + 1][threadIdx.x] = 0u;
            buf = nbuf;
            // ---- candidates of the batch, ranked in order by the warps that hold
            // positions of it: each scans the words, four a lane
            uint32_t wv[4], own, total;
            {
                const uint4 w4 = reinterpret_cast<const uint4 *>(bm)[lane];
                wv[0] = 4 * lane < nbw ? w4.x : 0u;
                wv[1] = 4 * lane + 1 < nbw ? w4.y : 0u;
                wv[2] = 4 * lane + 2 < nbw ? w4.z : 0u;
                wv[3] = 4 * lane + 3 < nbw ? w4.w : 0u;
                own = __popc(wv[0]) + __popc(wv[1]) + __popc(wv[2]) + __popc(wv[3]);
                total = __reduce_add_sync(0xffffffffu, own);
            }
            if (total == 0u) {   // every position keeps its spin
                p0 += B;
                bsize = min(2 * bsize, kBatchMax);
                mcap = max(2, mcap >> 1);
                continue;
            }
            uint32_t excl = 0u;
            if (warp < nbw) {
                uint32_t x = own;
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                excl = x - own;
            }
#pragma unroll
            for (int e = 0; e < kEval; ++e) {
                if (32 * e + warp >= nbw) break;
                // word 32 e + warp: held by lane (32 e + warp) / 4
                const int sub = warp & 3, src = e * 8 + (warp >> 2);
                uint32_t pre = excl;
                if (sub > 0) pre += __popc(wv[0]);
                if (sub > 1) pre += __popc(wv[1]);
                if (sub > 2) pre += __popc(wv[2]);
                const uint32_t w = __shfl_sync(0xffffffffu, sub == 0 ? wv[0] : sub == 1 ? wv[1] : sub == 2 ? wv[2] : wv[3], src);
                const uint32_t rank = __shfl_sync(0xffffffffu, pre, src) + __popc(w & ((1u << lane) - 1u));
                if (!((w >> lane) & 1u) || rank >= (uint32_t)kCand) continue;
                const int32_t k = kk[e];
                sm.ck[rank] = k;
                sm.cp[rank] = p0 + e * kDsThreads + (int32_t)threadIdx.x;
                if (k >= a0 && k < a1) {
                    const int32_t j = k - a0;
                    const uint32_t s = (bits[j >> 5] >> (j & 31)) & 1u;
                    const int32_t q = 2 * acc.margin(field(j), s, uu[e], mcap) + (int32_t)s;
                    for (int c = 0; c < nctas; ++c) *at(&sm.cq[rank], c) = q;
                }
            }
            __syncthreads();
            const int32_t nc = min((int32_t)total, kCand);
            if (threadIdx.x == 0) {
                sm.decided = 0;
                sm.final = -1;
            }
            // ---- the tile up to its diagonal (of row j the words 0 .. j / 32), the rows
            // dealt over the cluster's warps, two rows at a time
            {
                int32_t kc[kCand / 32];   // the lane's candidates: columns of the words
#pragma unroll
                for (int c = 0; c < kCand / 32; ++c) kc[c] = 32 * c < nc ? sm.ck[min(32 * c + lane, nc - 1)] : 0;
                const int32_t step = nctas * (kDsThreads / 32);
                for (int32_t j0 = crank * (kDsThreads / 32) + warp; j0 < nc; j0 += 2 * step) {
                    uint32_t v[2][kCand / 32];
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        const int32_t j = j0 + y * step;
                        if (j >= nc) break;
                        const uint32_t *row = a.Jb + (size_t)sm.ck[j] * a.pitch;
#pragma unroll
                        for (int c = 0; c < kCand / 32; ++c)
                            if (32 * c <= j) v[y][c] = __ldg(row + (kc[c] >> 5));
                    }
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        const int32_t j = j0 + y * step;
                        if (j >= nc) break;
#pragma unroll
                        for (int c = 0; c < kCand / 32; ++c) {
                            if (32 * c > j) break;
                            const uint32_t word = __ballot_sync(0xffffffffu, (v[y][c] >> (kc[c] & 31)) & 1u);
                            if (lane < nctas) *at(reinterpret_cast<uint32_t *>(&sm.tile[j]) + c, lane) = word;
                        }
                    }
                }
            }
            sync_all();
            // every decision is known (the requesting warps go on by themselves)
            auto decided = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(32 * (1 + kApply)) : "memory"); };
            const uint32_t row_bytes = (uint32_t)nW * 4u;
            // (up to the row's end; a slice that starts before n starts at a multiple of 128)
            const uint32_t copy_bytes = a0 < n ? (uint32_t)min(nW, a.pitch - (a0 >> 5)) * 4u : 0u;
            if (warp == 0) {
                // ---- the sequential decisions, the same in every CTA of the cluster
                int32_t q[kCand / 32];
                uint32_t sb[kCand / 32];   // the group's spin bits
                uint32_t tw[kCand / 32][kCand / 32];   // the candidate's tile row: +1 where a flip to +1 raises q
#pragma unroll
                for (int s = 0; s < kCand / 32; ++s) {
                    const int32_t j = s * 32 + lane;
                    const int32_t c = j < nc ? sm.cq[j] : -1024;
                    q[s] = c >> 1;
                    sb[s] = __ballot_sync(0xffffffffu, c & 1);
                    const uint4 t4 = sm.tile[j];   // (J is symmetric: row j is also column j)
                    const uint32_t m = 0u - ((uint32_t)(c & 1) ^ (acc.dir < 0 ? 1u : 0u));
                    tw[s][0] = t4.x ^ m; tw[s][1] = t4.y ^ m; tw[s][2] = t4.z ^ m; tw[s][3] = t4.w ^ m;
                }
                int32_t f = 0, stop = -1;
                uint64_t down = 0ull;
#pragma unroll
                for (int s = 0; s < kCand / 32; ++s) {
                    if (s * 32 >= nc || stop >= 0) break;
                    uint32_t open = 0xffffffffu;
                    while (true) {
                        const uint32_t fb = __ballot_sync(0xffffffffu, q[s] >= 0) & open;
                        if (fb == 0u) break;
                        const int o = __ffs(fb) - 1, j = s * 32 + o;
                        if (f == mcap) { stop = j; break; }
                        open = 0xfffffffeu << o;   // positions up to this one are decided
                        const uint32_t neg = (sb[s] >> o) & 1u;   // +1 turns to -1
#pragma unroll
                        for (int s3 = s; s3 < kCand / 32; ++s3)
                            q[s3] += 2 * (int32_t)(((tw[s3][s] >> o) ^ neg) & 1u) - 1;
                        if (lane == 0) sm.out.flip[f] = (uint32_t)j | (neg << 31);
                        down |= (uint64_t)neg << f;
                        ++f;
                        if (f % CH == 0 && lane == 0) st_release(&sm.decided, f);
                    }
                }
                if (lane == 0) {
                    sm.out.neg[0] = (uint32_t)down;
                    sm.out.neg[1] = (uint32_t)(down >> 32);
                    st_release(&sm.final, f);
                }
                decided();
                int32_t next = p0 + B;
                if ((int32_t)total > kCand) {   // the batch ends before candidate kCand
                    // position of the last kept candidate + 1 is at most the next one's
                    next = sm.cp[kCand - 1] + 1;
                }
                if (stop >= 0) next = sm.cp[stop];
                const int32_t done = next - p0;
                int32_t nb = (int32_t)total > kCand ? done
                             : stop >= 0            ? max(done, B >> 1)
                             : total <= kCand / 4   ? 2 * B
                             : total <= kCand / 2   ? B + (B >> 1)
                                                    : B;
                nb = min(kBatchMax, max(kBatchMin, (nb + 31) & ~31));
                const int32_t nm = stop >= 0 ? 2 * mcap : max(2, min(mcap, 2 * f + 2));
                if (lane == 0) {
                    sm.out.nflip = f;
                    sm.out.next = next;
                    sm.out.bsize = nb;
                    sm.out.mcap = min(kFlipMax, nm);
                }
                if (crank == 0)
                    for (int32_t i = lane; i < f; i += 32) {
                        const int32_t p = sm.cp[sm.out.flip[i] & 0xFFFFu];
                        // a position that flipped in some replica is counted by the first
                        const uint32_t m = 1u << (p & 31);
                        if (!(atomicOr(&a.rowbits[(size_t)sw * nrw + (p >> 5)], m) & m))
                            atomicAdd((unsigned long long *)&a.ctl->dense_rows, 1ull);
                    }
            } else if (warp <= kFetch) {
                // ---- the rows that flip, requested as they are decided: every kFetch-th
                // chunk of CH rows a warp
                int32_t first = (warp - 1) * CH;
                for (int spin = 0;;) {
                    int32_t all = 0, f = 0;   // (after an error: nothing left)
                    if (lane == 0 && *(volatile int32_t *)&sm.err == 0) {
                        all = ld_acquire(&sm.final);
                        f = all >= 0 ? all : ld_acquire(&sm.decided);
                    }
                    all = __shfl_sync(0xffffffffu, all, 0);
                    f = __shfl_sync(0xffffffffu, f, 0);
                    if (all >= 0 && first >= all) break;
                    const bool ready = f >= first + CH || all >= 0;
                    const uint32_t x = chunk0 + (uint32_t)(first / CH), slot = x & cmask, round = x >> clog;
                    bool ok = true;
                    if (!ready) {   // (bounded: about a second)
                        __nanosleep(32);
                        ok = ++spin < (1 << 24);
                    } else if (lane == 0 && round > 0) {
                        ok = mbar_wait(&sm.empty[slot], (round - 1) & 1);
                    }
                    if (!__all_sync(0xffffffffu, ok)) {
                        if (lane == 0) {
                            atomicCAS(&a.ctl->err, 0, (int)PAMC_ERR_TIMEOUT);
                            *(volatile int32_t *)&sm.err = 1;
                        }
                        break;
                    }
                    __syncwarp();
                    if (!ready) continue;
                    const int32_t rows = min(CH, f - first);
                    if (lane == 0) mbar_expect_tx(&sm.full[slot], (uint32_t)rows * copy_bytes);
                    __syncwarp();
                    if (lane < rows && copy_bytes > 0u)
                        bulk_load(ring + (size_t)(slot * CH + lane) * row_bytes,
                                     a.Jb + (size_t)sm.ck[sm.out.flip[first + lane] & 0xFFFFu] * a.pitch + (a0 >> 5),
                                     copy_bytes, &sm.full[slot]);
                    first += kFetch * CH;
                    spin = 0;
                }
            } else {
                // ---- the other warps count the requested rows once all are decided (they
                // wait on a barrier, not on the ring: polling warps would take the
                // deciding warp's issue slots), bit-sliced per row word (two words a
                // thread), and add the sum of +-2 J over the batch's flips to the slice's
                // fields at the end
                const int32_t w0 = (int32_t)threadIdx.x - 32 * (1 + kFetch);
                uint32_t c[2][6] = {};
                decided();
                const int32_t f = *(volatile int32_t *)&sm.final;
                uint64_t down = (uint64_t)sm.out.neg[1] << 32 | sm.out.neg[0];
                const bool mine =
                    __all_sync(0xffffffffu, warp - 1 - kFetch < appliers && *(volatile int32_t *)&sm.err == 0);
                for (int32_t first = 0; mine && first < f; first += CH, down >>= CH) {
                    const uint32_t x = chunk0 + (uint32_t)(first / CH), slot = x & cmask;
                    const bool late = !mbar_wait(&sm.full[slot], (x >> clog) & 1);
                    if (__any_sync(0xffffffffu, late)) {
                        if (lane == 0) {
                            atomicCAS(&a.ctl->err, 0, (int)PAMC_ERR_TIMEOUT);
                            *(volatile int32_t *)&sm.err = 1;
                        }
                        break;
                    }
                    const int32_t rows = min(CH, f - first);
                    const uint32_t *rw = reinterpret_cast<const uint32_t *>(ring) + (size_t)slot * CH * nW + w0;
                    uint32_t v[2][CH];
#pragma unroll
                    for (int q = 0; q < CH; ++q) {
                        v[0][q] = v[1][q] = 0u;
                        if (q < rows) {
                            const uint32_t m = 0u - ((uint32_t)(down >> q) & 1u);
                            if (w0 < nW) v[0][q] = rw[q * nW] ^ m;
                            if (w0 + 32 * kApply < nW) v[1][q] = rw[q * nW + 32 * kApply] ^ m;
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.empty[slot]);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if constexpr (CH == 4) {
                            uint32_t k0, k1, l0, s0;
                            full_add(c[h][0], v[h][0], v[h][1], s0, k0);
                            full_add(s0, v[h][2], v[h][3], c[h][0], k1);
                            full_add(c[h][1], k0, k1, s0, l0);
                            c[h][1] = s0;
#pragma unroll
                            for (int q = 2; q < 6; ++q) {
                                const uint32_t t2 = c[h][q] & l0;
                                c[h][q] ^= l0;
                                l0 = t2;
                            }
                        } else {
                            uint32_t l0 = v[h][0];
#pragma unroll
                            for (int q = 0; q < 6; ++q) {
                                const uint32_t t2 = c[h][q] & l0;
                                c[h][q] ^= l0;
                                l0 = t2;
                            }
                        }
                    }
                }
                if (mine && f > 0) {
                    const int np = 32 - __clz(f);   // planes a count of up to f needs
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int32_t w = w0 + h * 32 * kApply;
                        if (w >= nW) break;
                        const int32_t valid = a1 - a0 - 32 * w;   // vertices of the word
#pragma unroll
                        for (int b = 0; b < 8; ++b) {
                            uint32_t v = 0u;   // byte q: the count of bit b + 8 q
#pragma unroll
                            for (int q = 0; q < 6; ++q)
                                if (q < np) v += ((c[h][q] >> b) & 0x01010101u) << q;
                            if constexpr (HALF) {
#pragma unroll
                                for (int x = 0; x < 2; ++x) {   // vertices b + 8 x and b + 8 x + 16
                                    uint32_t *p = &Hs[(b + 8 * x) * nWp + w];
                                    const uint32_t old = *p;
                                    uint32_t nw = old + 2u * ((v >> (8 * x)) & 0x00FF00FFu) - (uint32_t)f * 0x00010001u;
                                    if (valid < 32) {   // beyond the last vertex: 0
                                        if (b + 8 * x >= valid) nw = (nw & 0xFFFF0000u) | 0x8000u;
                                        if (b + 8 * x + 16 >= valid) nw = (nw & 0xFFFFu) | 0x80000000u;
                                    }
                                    *p = nw;
                                }
                            } else {
#pragma unroll
                                for (int q = 0; q < 4; ++q)
                                    Hs[(b + 8 * q) * nWp + w] += 4u * ((v >> (8 * q)) & 0xFFu) - 2u * (uint32_t)f;
                            }
                        }
                    }
                }
            }
            __syncthreads();
            // the flipped vertices: the spin, and J_kk = 0 (the clear bit counted as -1)
            const int32_t f = sm.out.nflip;
            if ((int32_t)threadIdx.x < f) {
                const uint32_t fl = sm.out.flip[threadIdx.x];
                const int32_t j = sm.ck[fl & 0xFFFFu] - a0;
                if (j >= 0 && j < a1 - a0) {
                    if constexpr (HALF) atomicAdd(&Hs[(j & 15) * nWp + (j >> 5)], ((fl >> 31) ? ~0u : 1u) << (j & 16));
                    else Hs[(j & 31) * nWp + (j >> 5)] += (fl >> 31) ? -2 : 2;
                    atomicXor(&bits[j >> 5], 1u << (j & 31));
                }
            }
            room -= f;
            chunk0 += (uint32_t)((f + CH - 1) / CH);
            p0 = sm.out.next;
            bsize = sm.out.bsize;
            mcap = sm.out.mcap;
            __syncthreads();
        }
    }

    // ---------------- energies E_r = -1/2 sum_k s_k h_k, fields and spins back
    // a wait ran out: the copies in flight land first (bounded; a chunk never
    // requested completes no phase, which ends the wait as well)
    if (*(volatile int32_t *)&sm.err && threadIdx.x == 0)
        for (uint32_t x = chunk0 > cmask ? chunk0 - a.chunks : 0u; x < chunk0; ++x)
            mbar_wait(&sm.full[x & cmask], (x >> clog) & 1);
    long long e = 0;
    for (int32_t w = warp; w < nW; w += kDsThreads / 32) {
        const int32_t k = a0 + 32 * w + lane;
        if (k < a1) {
            const int32_t h = field(32 * w + lane);
            const bool up = (bits[w] >> lane) & 1u;
            if (held) a.H[(size_t)r * n + k] = h;   // (else as loaded)
            a.dst[(size_t)r * n + k] = up ? 1 : -1;
            e += up ? h : -h;
        }
    }
    for (int o = 16; o > 0; o >>= 1) e += __shfl_down_sync(0xffffffffu, e, o);
    if (lane == 0) atomicAdd(at(&sm.esum, 0), (unsigned long long)e);
    sync_all();
    if (crank == 0 && threadIdx.x == 0) {
        if (checked) a.resume[r] = stopped ? make_int2(sw, p0) : make_int2(a.S, 0);
        a.E[r] = -((long long)sm.esum / 2);   // (of a stopped replica: written again by 32-bit fields)
        if (r == 0 && !RESUME) a.ctl->dense_positions += (int64_t)n * a.S;
    }
}

// A slice's layout in shared memory: rows of the ring that fit beside its
// fields (0: the slice does not fit)
struct DsPlan {
    int rows = 0;
    size_t smem = 0;
};
DsPlan ds_plan(int32_t n, int cs, bool half) {
    DsPlan p;
    const int32_t nW = ds_slice(n, cs) >> 5;
    const size_t base = ds_ring_offset(nW, half), row = (size_t)nW * 4;
    if (nW > kWordsMax || base > 227 * 1024) return p;
    p.rows = (int)std::min<size_t>((227 * 1024 - base) / row, half ? kRowsMax : kChunkMax);
    p.smem = base + p.rows * row;
    return p;
}
constexpr int kHalfRows = 4;                                       // rows of a chunk, 16-bit fields
bool ds_half_fits(int32_t n, int cs) { return ds_plan(n, cs, true).rows >= 2 * kHalfRows; }

template <bool HALF, int CH, bool RESUME>
cudaError_t ds_launch(DenseSweepArgs a, int cs, cudaStream_t st) {
    const DsPlan plan = ds_plan(a.n, cs, HALF);
    a.per = ds_slice(a.n, cs);
    a.chunks = 1;
    while (2 * a.chunks * CH <= plan.rows) a.chunks *= 2;
    cudaError_t e;
    if (cs == 1) {
        e = allow_dynamic_smem(k_dense_sweep<false, HALF, CH, RESUME>, plan.smem);
        if (e != cudaSuccess) return e;
        k_dense_sweep<false, HALF, CH, RESUME><<<a.R, kDsThreads, plan.smem, st>>>(a, 1);
        return cudaGetLastError();
    }
    e = allow_dynamic_smem(k_dense_sweep<true, HALF, CH, RESUME>, plan.smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.R * cs));
    cfg.blockDim = dim3(kDsThreads);
    cfg.dynamicSmemBytes = plan.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cs;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_dense_sweep<true, HALF, CH, RESUME>, a, cs);
}

}  // namespace

// words of a row: whole 128-byte lines (the recompute copies 1,024 couplings of a row at a time)
int32_t dense_bits_pitch(int32_t n) { return ((n + 1023) / 1024) * 32; }

// The smallest cluster whose slices fit; from n = 20,000 on twice or four times
// as many CTAs a replica where every cluster still gets its own SMs: a slice's
// rows and field pass then outweigh the cluster barriers (first two-sweep step, ms,
// R = 24, 1 / 2 / 4 CTAs: n = 1,000 0.24 / 0.27 / 0.27, n = 10,000 1.56 / 1.59 / 1.50, n
// = 20,000 3.43 / 3.05 / 2.85, n = 40,000 9.0 / 7.4 / 5.8; R = 64 at 20,000: 3.45 / 3.11
// / 5.59, the last in two waves).  PAMC_DENSE_CLUSTER forces a size that fits.
int dense_sweep_cluster(int32_t n, int32_t R, int sms) {
    int cs = 1;
    while (cs <= kMaxCluster && !ds_half_fits(n, cs)) cs *= 2;
    if (cs > kMaxCluster) return 0;
    if (const char *env = getenv("PAMC_DENSE_CLUSTER")) {
        const int v = atoi(env);
        if ((v == 1 || v == 2 || v == 4 || v == 8) && v >= cs) return v;
    }
    while (n >= 20000 && cs < 4 && (int64_t)R * 2 * cs <= sms) cs *= 2;
    return cs;
}

int dense_sweep_launches(int32_t n) { return n > kHalfAlways ? 2 : 1; }

cudaError_t launch_dense_sweep(int32_t n, int32_t R, int32_t S, int32_t rule, int32_t Hc, int32_t t, uint64_t seed,
                               int cs, const uint32_t *Jb, const int32_t *perm, const uint64_t *tab,
                               const int8_t *src, const int32_t *parent, int32_t *H, int8_t *dst, int64_t *E,
                               uint32_t *rowbits, int32_t *resume, DevCtl *ctl, cudaStream_t st, int32_t rbase) {
    DenseSweepArgs a;
    a.n = n; a.R = R; a.S = S; a.rule = rule; a.Hc = Hc; a.t = t; a.gbase = rbase / 4;
    a.pitch = dense_bits_pitch(n);
    a.K = make_philox_keys(seed);
    a.Jb = Jb; a.perm = perm; a.tab = tab; a.src = src; a.parent = parent; a.H = H; a.dst = dst; a.E = E;
    a.rowbits = rowbits; a.resume = reinterpret_cast<int2 *>(resume); a.ctl = ctl;
    // PAMC_DENSE_FIELD_MAX: a smaller range for the 16-bit fields, so that small instances leave it
    const char *env = getenv("PAMC_DENSE_FIELD_MAX");
    a.half_max = env ? std::min(std::max(atoi(env), 1), 32767) : n > kHalfAlways ? 32767 : 0;
    cudaError_t e = cudaMemsetAsync(rowbits, 0, (size_t)(S > 0 ? S : 1) * ((n + 31) / 32) * 4, st);
    if (e == cudaSuccess) e = ds_launch<true, kHalfRows, false>(a, cs, st);
    if (e != cudaSuccess || a.half_max == 0) return e;
    while (cs <= kMaxCluster && ds_plan(n, cs, false).rows < 1) cs *= 2;
    if (cs > kMaxCluster) return cudaErrorInvalidValue;
    return ds_launch<false, 1, true>(a, cs, st);
}

}  // namespace pamc
