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
// fall with the field, and the heat-bath decisions read the table at -h).  Every other position
// keeps its spin whatever the first m flips of the batch are.  The candidates
// (at most kCand, in order) are then decided one after the other by one warp
// from their fields and the bit tile of the couplings among them; before a
// flip m + 1 the batch ends and the next one starts at that position.  The
// flipped rows are applied to all fields of the slice in one pass.  So the
// result is the sequential sweep's, position by position.  B and m follow
// what the last batch saw.
//
// Bounds.  An evaluation is one Philox call and up to three table reads per
// position; a batch with candidates adds a gather of single bits (one miss
// latency), at most kCand decisions of one warp, and a pass over the slice's
// fields (4 bytes read and written each at 128 bytes a clock).  Hot steps are
// bound by the flipped rows' traffic and the decisions, cold ones by the
// latencies of a few dozen batches.  Measured at n = 100,000, R = 64, two
// sweeps (a design that advanced all replicas together in blocks of 256
// positions, a grid barrier after each, before): 30.6 ms for the first, hottest
// step (22.4 before), 1.05 ms for a cold one (6.1 before), 72 ms for a 20-step
// anneal (181 before); n = 5,001, R = 24, 30 steps: 3.6 ms (16.9 before).
#include <cooperative_groups.h>

#include <cstdlib>

#include "pamc_device.cuh"
#include "pamc_internal.h"

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
    DevCtl *ctl;
};

// What the leader's warp hands to every CTA of the cluster after a batch.
struct BatchOut {
    int32_t nflip, next, bsize, mcap;
    uint32_t flip[64];        // vertex | (1 << 31 when the spin turned to -1)
};

struct DsSmem {               // fixed part of a CTA's shared memory
    uint32_t win[kDsWin];
    uint32_t bm[3][kBatchMax / 32];   // candidate bits of a batch, in turn
    int32_t ck[kCand], cp[kCand];     // candidates: vertex, position
    int32_t cq[kCand];                // (leader) 2 (margin) + spin bit, see below
    uint4 tile[kCand];                // (leader) J[candidate][candidate], one bit each
    BatchOut out;
    int32_t lo, hi, nwin, dir;
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

template <bool CL>
__global__ void __launch_bounds__(kDsThreads, 1) k_dense_sweep(DenseSweepArgs a, int cs) {
    extern __shared__ __align__(16) uint8_t smraw[];
    DsSmem &sm = *reinterpret_cast<DsSmem *>(smraw);
    const int32_t per = a.per, nW = per >> 5, nWp = nW | 1;
    // fields: vertex a0 + 32 w + b at Hs[b * nWp + w] (a thread's 32 fields of
    // one row word lie in 32 rows, consecutive words in consecutive banks)
    int32_t *Hs = reinterpret_cast<int32_t *>(smraw + ((sizeof(DsSmem) + 15) & ~(size_t)15));
    uint32_t *bits = reinterpret_cast<uint32_t *>(Hs + (size_t)32 * nWp);
    if (a.ctl->done) return;   // uniform over the grid

    const int32_t n = a.n;
    const int crank = CL ? (int)(blockIdx.x % cs) : 0;
    const int r = CL ? (int)(blockIdx.x / cs) : (int)blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t a0 = min(n, crank * per), a1 = min(n, a0 + per);
    auto sync_all = [&]() {
        if constexpr (CL) cg::this_cluster().sync();
        else __syncthreads();
    };
    // the same shared-memory address in CTA c of the cluster
    auto at = [&](auto *p, int c) {
        if constexpr (CL) return cg::this_cluster().map_shared_rank(p, c);
        else return p;
    };

    // ---------------- prologue: spins, fields, thresholds
    const int8_t *row = a.src + (size_t)a.parent[r] * n;
    for (int32_t w = warp; w < nW; w += kDsThreads / 32) {
        const int32_t k = a0 + 32 * w + lane;
        const uint32_t b = __ballot_sync(0xffffffffu, k < a1 && row[min(k, n - 1)] > 0);
        Hs[lane * nWp + w] = k < a1 ? a.H[(size_t)r * n + k] : 0;
        if (lane == 0) bits[w] = b;
    }
    for (int32_t i = threadIdx.x; i < 3 * (kBatchMax / 32); i += kDsThreads) (&sm.bm[0][0])[i] = 0u;
    if (threadIdx.x == 0) {
        // [lo, hi): where the threshold is neither 0 nor 2^32
        int32_t lo, hi;
        sm.dir = 1;
        if (a.rule == 0) {   // tab[i] = T(i - Hc), rising (falling at a negative beta: read from its end)
            const int32_t last = 2 * a.Hc;
            const bool back = a.tab[0] > a.tab[last];
            auto T = [&](int32_t i) { return a.tab[back ? last - i : i]; };
            sm.dir = back ? -1 : 1;
            int32_t l = 0, h2 = last + 1;
            while (l < h2) { const int32_t md = (l + h2) >> 1; if (T(md) > 0ull) h2 = md; else l = md + 1; }
            lo = l - a.Hc;
            h2 = last + 1;
            while (l < h2) { const int32_t md = (l + h2) >> 1; if (T(md) >= (1ull << 32)) h2 = md; else l = md + 1; }
            hi = l - a.Hc;
        } else {             // tab[x] = T_M(2x), falling from tab[0] = 2^32
            int32_t l = 0, h2 = a.Hc + 1;
            while (l < h2) { const int32_t md = (l + h2) >> 1; if (a.tab[md] < (1ull << 32)) h2 = md; else l = md + 1; }
            lo = l;
            h2 = a.Hc + 1;
            while (l < h2) { const int32_t md = (l + h2) >> 1; if (a.tab[md] == 0ull) h2 = md; else l = md + 1; }
            hi = l;
        }
        lo += (lo ^ (n - 1)) & 1;   // the fields' parity
        sm.lo = lo;
        sm.hi = max(hi, lo);
        sm.nwin = (sm.hi - lo + 1) >> 1;
        sm.esum = 0ull;
    }
    __syncthreads();
    Accept acc{sm.win, a.tab, sm.lo, sm.hi, a.rule == 0 ? a.Hc : 0, a.rule == 0 ? 1 : 0, sm.dir,
               sm.nwin <= kDsWin};
    if (acc.inwin)
        for (int32_t i = threadIdx.x; i < sm.nwin; i += kDsThreads) sm.win[i] = (uint32_t)a.tab[acc.dir * (acc.lo + 2 * i) + acc.off];
    const int32_t nrw = (n + 31) >> 5;
    const uint32_t ctr3 = (kTagFlip << 24) | (uint32_t)((r >> 2) + a.gbase);
    sync_all();   // every CTA of the cluster runs before another one writes its memory

    int32_t bsize = 512, mcap = 8;
    int buf = 0;
    for (int32_t sw = 0; sw < a.S; ++sw) {
        const int32_t *perm = a.perm + (size_t)sw * n;
        int32_t p0 = 0;
        while (p0 < n) {
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
                    const int32_t h = Hs[(j & 31) * nWp + (j >> 5)];
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
            // ---- candidates of the batch, ranked in order (the same in every
            // warp of every CTA: each scans the words, four a lane)
            uint32_t wv[4], excl, total;
            {
                const uint4 w4 = reinterpret_cast<const uint4 *>(bm)[lane];
                wv[0] = 4 * lane < nbw ? w4.x : 0u;
                wv[1] = 4 * lane + 1 < nbw ? w4.y : 0u;
                wv[2] = 4 * lane + 2 < nbw ? w4.z : 0u;
                wv[3] = 4 * lane + 3 < nbw ? w4.w : 0u;
                const uint32_t own = __popc(wv[0]) + __popc(wv[1]) + __popc(wv[2]) + __popc(wv[3]);
                uint32_t x = own;
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                excl = x - own;
                total = __shfl_sync(0xffffffffu, x, 31);
            }
            if (total == 0u) {   // every position keeps its spin
                p0 += B;
                bsize = min(2 * bsize, kBatchMax);
                mcap = max(2, mcap >> 1);
                continue;
            }
#pragma unroll
            for (int e = 0; e < kEval; ++e) {
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
                    const int32_t q = acc.margin(Hs[(j & 31) * nWp + (j >> 5)], s, uu[e], mcap);
                    *at(&sm.cq[rank], 0) = 2 * q + (int32_t)s;
                }
            }
            __syncthreads();
            const int32_t nc = min((int32_t)total, kCand), ncw = (nc + 31) >> 5;
            // ---- the tile's upper words, dealt over the cluster's warps
            {
                const int32_t words = nc * ncw, step = (CL ? cs : 1) * (kDsThreads / 32);
                for (int32_t w0 = crank * (kDsThreads / 32) + warp; w0 < words; w0 += 4 * step) {
                    uint32_t v[4];
                    int32_t kb[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int32_t wd = min(w0 + x * step, words - 1);
                        kb[x] = sm.ck[min((wd % ncw) * 32 + lane, nc - 1)];
                        v[x] = __ldg(a.Jb + (size_t)sm.ck[wd / ncw] * a.pitch + (kb[x] >> 5));
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int32_t wd = w0 + x * step;
                        if (wd >= words) break;
                        const uint32_t word = __ballot_sync(0xffffffffu, (v[x] >> (kb[x] & 31)) & 1u);
                        if (lane == 0) *at(reinterpret_cast<uint32_t *>(&sm.tile[wd / ncw]) + wd % ncw, 0) = word;
                    }
                }
            }
            sync_all();
            // ---- the sequential decisions, by the leader's first warp
            if (crank == 0 && warp == 0) {
                int32_t q[kCand / 32];
                uint32_t sb[kCand / 32];   // the group's spin bits
#pragma unroll
                for (int s = 0; s < kCand / 32; ++s) {
                    const int32_t j = s * 32 + lane;
                    const int32_t c = j < nc ? sm.cq[j] : -1024;
                    q[s] = c >> 1;
                    sb[s] = __ballot_sync(0xffffffffu, c & 1);
                }
                int32_t f = 0, stop = -1;
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
                        const uint4 tj = sm.tile[j];
                        const uint32_t neg = (sb[s] >> o) & 1u;   // +1 turns to -1
                        const uint32_t down = (0u - neg) ^ (acc.dir < 0 ? 0xFFFFFFFFu : 0u);
                        const uint32_t tw[4] = {tj.x, tj.y, tj.z, tj.w};
#pragma unroll
                        for (int s3 = s; s3 < kCand / 32; ++s3)
                            q[s3] += 2 * (int32_t)(((tw[s3] ^ sb[s3] ^ down) >> lane) & 1u) - 1;
                        if (lane == 0) sm.out.flip[f] = (uint32_t)j | (neg << 31);
                        ++f;
                    }
                }
                __syncwarp();
                for (int32_t i = lane; i < f; i += 32) {
                    const uint32_t fl = sm.out.flip[i];
                    const int32_t j = (int32_t)(fl & 0x7fffffffu), p = sm.cp[j];
                    // a position that flipped in some replica is counted by the first
                    const uint32_t m = 1u << (p & 31);
                    if (!(atomicOr(&a.rowbits[(size_t)sw * nrw + (p >> 5)], m) & m))
                        atomicAdd((unsigned long long *)&a.ctl->dense_rows, 1ull);
                    sm.out.flip[i] = (uint32_t)sm.ck[j] | (fl & 0x80000000u);
                }
                __syncwarp();
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
                                                    : B;
                nb = min(kBatchMax, max(kBatchMin, (nb + 31) & ~31));
                const int32_t nm = stop >= 0 ? 2 * mcap : max(2, min(mcap, 2 * f + 2));
                for (int c = 0; c < (CL ? cs : 1); ++c) {
                    BatchOut *o = at(&sm.out, c);
                    if (c != 0)
                        for (int32_t i = lane; i < f; i += 32) o->flip[i] = sm.out.flip[i];
                    if (lane == 0) {
                        o->nflip = f;
                        o->next = next;
                        o->bsize = nb;
                        o->mcap = min(kFlipMax, nm);
                    }
                }
            }
            sync_all();
            // ---- apply the flips to the slice: every field gets the sum of
            // +-2 J over the flipped rows, counted bit-sliced per row word
            const int32_t f = sm.out.nflip;
            if (f > 0) {
                const int np = 32 - __clz(f);   // planes a count of up to f needs
                const uint32_t *Jw = a.Jb + (a0 >> 5);
                const int32_t lim = a.pitch - (a0 >> 5);   // words of a row from a0 on
                // two row words a thread, eight rows at a time: 16 loads in flight
                for (int32_t w = threadIdx.x; w < nW; w += 2 * kDsThreads) {
                    uint32_t c[2][6] = {};
                    const bool in0 = w < lim, in1 = w + kDsThreads < min(lim, nW);
                    for (int32_t f0 = 0; f0 < f; f0 += 8) {
                        uint32_t v[2][8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            v[0][q] = v[1][q] = 0u;
                            if (f0 + q < f) {
                                const uint32_t fl = sm.out.flip[f0 + q];
                                const uint32_t *Jr = Jw + (size_t)(fl & 0x7fffffffu) * a.pitch + w;
                                if (in0) v[0][q] = __ldg(Jr) ^ (0u - (fl >> 31));
                                if (in1) v[1][q] = __ldg(Jr + kDsThreads) ^ (0u - (fl >> 31));
                            }
                        }
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t k0, k1, k2, k3, l0, l1, m0, s0, s1;
                            full_add(c[h][0], v[h][0], v[h][1], s0, k0);
                            full_add(s0, v[h][2], v[h][3], s1, k1);
                            full_add(s1, v[h][4], v[h][5], s0, k2);
                            full_add(s0, v[h][6], v[h][7], c[h][0], k3);
                            full_add(c[h][1], k0, k1, s0, l0);
                            full_add(s0, k2, k3, c[h][1], l1);
                            full_add(c[h][2], l0, l1, s0, m0);
                            c[h][2] = s0;
#pragma unroll
                            for (int q = 3; q < 6; ++q) {
                                const uint32_t t2 = c[h][q] & m0;
                                c[h][q] ^= m0;
                                m0 = t2;
                            }
                        }
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int32_t wh = w + h * kDsThreads;
                        if (wh >= nW) break;
#pragma unroll
                        for (int b = 0; b < 8; ++b) {
                            uint32_t v = 0u;   // byte q: the count of bit b + 8 q
#pragma unroll
                            for (int q = 0; q < 6; ++q)
                                if (q < np) v += ((c[h][q] >> b) & 0x01010101u) << q;
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                Hs[(b + 8 * q) * nWp + wh] += 4 * (int32_t)((v >> (8 * q)) & 0xFFu) - 2 * f;
                        }
                    }
                }
                __syncthreads();
                // the flipped vertices: the spin, and J_kk = 0 (the clear bit counted as -1)
                if ((int32_t)threadIdx.x < f) {
                    const uint32_t fl = sm.out.flip[threadIdx.x];
                    const int32_t j = (int32_t)(fl & 0x7fffffffu) - a0;
                    if (j >= 0 && j < a1 - a0) {
                        Hs[(j & 31) * nWp + (j >> 5)] += (fl >> 31) ? -2 : 2;
                        atomicXor(&bits[j >> 5], 1u << (j & 31));
                    }
                }
            }
            p0 = sm.out.next;
            bsize = sm.out.bsize;
            mcap = sm.out.mcap;
            __syncthreads();
        }
    }

    // ---------------- energies E_r = -1/2 sum_k s_k h_k, fields and spins back
    long long e = 0;
    for (int32_t w = warp; w < nW; w += kDsThreads / 32) {
        const int32_t k = a0 + 32 * w + lane;
        if (k < a1) {
            const int32_t h = Hs[lane * nWp + w];
            const bool up = (bits[w] >> lane) & 1u;
            a.H[(size_t)r * n + k] = h;
            a.dst[(size_t)r * n + k] = up ? 1 : -1;
            e += up ? h : -h;
        }
    }
    for (int o = 16; o > 0; o >>= 1) e += __shfl_down_sync(0xffffffffu, e, o);
    if (lane == 0) atomicAdd(at(&sm.esum, 0), (unsigned long long)e);
    sync_all();
    if (crank == 0 && threadIdx.x == 0) {
        a.E[r] = -((long long)sm.esum / 2);
        if (r == 0) a.ctl->dense_positions += (int64_t)n * a.S;
    }
}

size_t ds_smem(int32_t n, int cs) {
    const int32_t per = ((n + cs - 1) / cs + 31) & ~31, nW = per >> 5, nWp = nW | 1;
    return ((sizeof(DsSmem) + 15) & ~(size_t)15) + (size_t)32 * nWp * 4 + (size_t)nW * 4;
}

}  // namespace

// words of a row: whole 128-byte lines (the recompute copies 1,024 couplings of a row at a time)
int32_t dense_bits_pitch(int32_t n) { return ((n + 1023) / 1024) * 32; }

// The smallest cluster whose slices fit; from n = 32,000 on twice or four times
// as many CTAs a replica where every cluster still gets its own SMs: a slice's
// field pass then outweighs the cluster barriers (first two-sweep step, R = 24:
// n = 40,000 11.5 / 10.8 / 10.4 ms with 1 / 2 / 4 CTAs, n = 20,000 5.1 / 5.4 /
// 5.2, n = 1,000 0.24 / 0.36 / 0.36; R = 64 at 40,000: 11.2 / 10.8 / 20.2, the
// last in two waves).  PAMC_DENSE_CLUSTER forces a size that fits.
int dense_sweep_cluster(int32_t n, int32_t R, int sms) {
    int cs = 1;
    while (cs <= kMaxCluster && ds_smem(n, cs) > 227 * 1024) cs *= 2;
    if (cs > kMaxCluster) return 0;
    if (const char *env = getenv("PAMC_DENSE_CLUSTER")) {
        const int v = atoi(env);
        if ((v == 1 || v == 2 || v == 4 || v == 8) && v >= cs) return v;
    }
    while (n >= 32000 && cs < 4 && (int64_t)R * 2 * cs <= sms) cs *= 2;
    return cs;
}

cudaError_t launch_dense_sweep(int32_t n, int32_t R, int32_t S, int32_t rule, int32_t Hc, int32_t t, uint64_t seed,
                               int cs, const uint32_t *Jb, const int32_t *perm, const uint64_t *tab,
                               const int8_t *src, const int32_t *parent, int32_t *H, int8_t *dst, int64_t *E,
                               uint32_t *rowbits, DevCtl *ctl, cudaStream_t st, int32_t rbase) {
    DenseSweepArgs a;
    a.n = n; a.R = R; a.S = S; a.rule = rule; a.Hc = Hc; a.t = t; a.gbase = rbase / 4;
    a.per = ((n + cs - 1) / cs + 31) & ~31;
    a.pitch = dense_bits_pitch(n);
    a.K = make_philox_keys(seed);
    a.Jb = Jb; a.perm = perm; a.tab = tab; a.src = src; a.parent = parent; a.H = H; a.dst = dst; a.E = E;
    a.rowbits = rowbits; a.ctl = ctl;
    cudaError_t e = cudaMemsetAsync(rowbits, 0, (size_t)(S > 0 ? S : 1) * ((n + 31) / 32) * 4, st);
    if (e != cudaSuccess) return e;
    const size_t smem = ds_smem(n, cs);
    if (cs == 1) {
        e = allow_dynamic_smem(k_dense_sweep<false>, smem);
        if (e != cudaSuccess) return e;
        k_dense_sweep<false><<<R, kDsThreads, smem, st>>>(a, 1);
        return cudaGetLastError();
    }
    e = allow_dynamic_smem(k_dense_sweep<true>, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(R * cs));
    cfg.blockDim = dim3(kDsThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cs;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_dense_sweep<true>, a, cs);
}

}  // namespace pamc
