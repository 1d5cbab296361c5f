// sweep_staged.cu -- the Ising sweep (Eq. 3-4) of small populations, where one
// replica group of four has an SM to itself and a launch is bound by the
// latency of its dependency levels: one CTA per group, warps of two kinds.
//
// Producer warps run ahead of the sweep over the schedule's positions, 32 at a
// time: the block's ELL rows arrive in a ring in shared memory by a bulk copy,
// the records are copied beside them, and the draw of every position (one
// Philox call, the group's four words) is computed and stored -- none of it
// depends on spins.  Two sets of consumer warps take the passes over the levels
// in turn (a pass: as many vertices of a level as a set has lane groups): while
// one set works on its pass, the other reads the rows, records and draws of
// the next into registers, so that a level costs its own chain only -- barrier,
// shared loads of the neighbours' spin words, sum, threshold, store.  (A warp
// alone on its scheduler spends about five cycles an instruction; reading ahead
// in the same warp doubled the chain.)  A launch of 5 sweeps at N=800, degree
// 48, R=128 went from 340 to 214 us with it, one of 5 sweeps at N=2,500, degree
// 12, weights to 100 (16-bit lanes), R=250 from 624 to 175 us.  LPV lanes share
// a vertex, each sums its groups of four couplings; the partial sums are added
// across the lanes, and lane q < 4 decides replica q (two replicas a lane with LPV = 2, four with LPV
// = 1) and stores its part of the word.  Draws, orders and results are those of
// the other Ising sweeps bit for bit.
//
// Field lanes: bytes (sum_j |J_kj| <= 127: one word per vertex, byte q =
// replica q) or 16 bits (WIDE, up to 32,767: two words).
//
// Every wait is bounded; on expiry the kernel sets PAMC_ERR_TIMEOUT, the other
// waits end at once, the consumers read zeros in place of what did not arrive
// (vertex 0, coupling 0: in bounds) and run out, and nothing is written back.
#include <cstring>

#include "pamc_device.cuh"
#include "pamc_internal.h"
#include "tc_sm100.cuh"

namespace pamc {

namespace {

constexpr int kStMaxThreads = 640;
constexpr int kStRingMax = 64;   // blocks in flight (a power of two)

// (volatile: ordered against the barriers that hand the slots over)
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ int2 lds64(uint32_t a) {
    int2 v;
    asm volatile("ld.shared.v2.s32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}

// Sums over neighbours: the four replicas' fields of a vertex in byte lanes of
// one word, or in 16-bit lanes of two.
struct ByteLanes {
    using Word = uint32_t;
    using Half = uint8_t;   // one replica's part of the word
    static constexpr uint32_t kBias = 128;
    uint32_t a = 0u;
    __device__ __forceinline__ void add(uint32_t e, const Word *sp) {
        a += sp[e & 0xFFFFFFu] * (uint32_t)((int32_t)e >> 24);
    }
    __device__ __forceinline__ void join(const ByteLanes &o) { a += o.a; }
    __device__ __forceinline__ void xor_add(int o) { a += __shfl_xor_sync(0xffffffffu, a, o); }
    __device__ __forceinline__ void bias() { a += 0x80808080u; }
    __device__ __forceinline__ int32_t lane(int q) const { return (int32_t)((a >> (8 * q)) & 0xFFu); }
    __device__ static __forceinline__ uint32_t bit(Word w, int q) { return (w >> (8 * q)) & 1u; }
};
struct WideLanes {
    using Word = uint2;
    using Half = uint16_t;
    static constexpr uint32_t kBias = 32768;
    uint32_t x = 0u, y = 0u;
    __device__ __forceinline__ void add(uint32_t e, const Word *sp) {
        const uint2 w = sp[e & 0xFFFFFFu];
        const uint32_t J = (uint32_t)((int32_t)e >> 24);
        x += w.x * J;
        y += w.y * J;
    }
    __device__ __forceinline__ void join(const WideLanes &o) { x += o.x; y += o.y; }
    __device__ __forceinline__ void xor_add(int o) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    __device__ __forceinline__ void bias() { x += 0x80008000u; y += 0x80008000u; }
    __device__ __forceinline__ int32_t lane(int q) const {
        return (int32_t)(((q & 2) ? y : x) >> (16 * (q & 1)) & 0xFFFFu);
    }
    __device__ static __forceinline__ uint32_t bit(Word w, int q) {
        return (((q & 2) ? w.y : w.x) >> (16 * (q & 1))) & 1u;
    }
};

struct StLayout {   // offsets into dynamic shared memory
    uint32_t spins, ring, red, bar, total;
    uint32_t slot;  // bytes of a ring slot: the block's ELL rows, its records, its draws
};
__host__ __device__ __forceinline__ StLayout st_layout(int32_t n, int32_t H, int32_t W, int nb, bool wide,
                                                       bool tab_smem) {
    StLayout l;
    const uint32_t tab = tab_smem ? ((uint32_t)(2 * H + 1) * 8u + 127u) & ~127u : 0u;
    l.spins = tab;
    l.ring = (l.spins + (uint32_t)n * (wide ? 8u : 4u) + 127u) & ~127u;
    l.slot = 32u * (uint32_t)W * 4u + 256u + 512u;
    l.bar = l.ring + l.slot * (uint32_t)nb;
    l.red = l.bar + 2u * 8u * (uint32_t)kStRingMax;
    l.total = l.red + 64u;
    return l;
}

// LPV lanes a vertex, NV groups of four couplings a lane read ahead.
// The slow side of a bounded wait (about a second), kept out of the loops:
// polls with a pause, so that a waiting warp leaves the scheduler to the others.
__device__ __noinline__ bool st_wait_slow(uint64_t *b, uint32_t parity, uint32_t pause_ns, int *err_flag, DevCtl *ctl) {
    for (int it = 0; it < (1 << 22); ++it) {
        if (mbar_try_wait(b, parity)) return true;
        if (*(volatile int *)err_flag) return false;   // (an error elsewhere: the launch is ending)
        __nanosleep(pause_ns);
    }
    atomicCAS(&ctl->err, 0, (int)PAMC_ERR_TIMEOUT);
    *(volatile int *)err_flag = 1;
    return false;
}

template <int RULE, int LPV, int NV, class Lanes, bool TABS>
__global__ void __launch_bounds__(kStMaxThreads)
k_sweep_ising_staged(SweepDesc d, int cwarps, int nb) {
    using Word = typename Lanes::Word;
    using Half = typename Lanes::Half;
    constexpr bool WIDE = sizeof(Word) == 8;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ int s_err;
    DevCtl *ctl = const_cast<DevCtl *>(d.ctl);
    if (ctl->done) return;
    const int32_t n = d.n, H = d.H, R = d.R, S = d.S, W = d.W;
    const StLayout lay = st_layout(n, H, W, nb, WIDE, TABS);
    uint64_t *tab_s = reinterpret_cast<uint64_t *>(smem);
    Word *sp = reinterpret_cast<Word *>(smem + lay.spins);
    uint8_t *ring = smem + lay.ring;
    unsigned long long *red = reinterpret_cast<unsigned long long *>(smem + lay.red);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + lay.bar), *empty = full + kStRingMax;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int pwarps = (int)(blockDim.x >> 5) - 2 * cwarps;
    const int32_t g = blockIdx.x, r0 = g * 4;
    const int32_t nblk = (n + 31) >> 5;
    const size_t ell_stride = (size_t)nblk * 32 * W;
    const size_t sb0 = (size_t)d.slot * S;

    if (threadIdx.x == 0) {
        for (int b = 0; b < nb; ++b) { mbar_init(&full[b], 2); mbar_init(&empty[b], 2u * (uint32_t)cwarps); }
        s_err = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < 8) red[threadIdx.x] = 0ull;   // (the last two: zeros for lanes beyond a row)
    if constexpr (TABS)
        for (int i = threadIdx.x; i < 2 * H + 1; i += blockDim.x) tab_s[i] = d.tab[i];
    {   // slot r reads the NCM output if the cluster move rewrote it, else its
        // resampling parent (the replica copy of the population step)
        const int8_t *rows[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            rows[q] = nullptr;
            if (r0 + q < R) {
                const int32_t m = d.ncm_idx[r0 + q];
                rows[q] = m >= 0 ? d.ncm_buf + (size_t)m * n : d.src + (size_t)d.parent[r0 + q] * n;
            }
        }
        for (int32_t k = threadIdx.x; k < n; k += blockDim.x) {
            uint32_t b[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) b[q] = rows[q] != nullptr && rows[q][k] > 0 ? 1u : 0u;
            if constexpr (WIDE) sp[k] = make_uint2(b[0] | (b[1] << 16), b[2] | (b[3] << 16));
            else sp[k] = b[0] | (b[1] << 8) | (b[2] << 16) | (b[3] << 24);
        }
    }
    __syncthreads();
    // one lane polls, the others learn the outcome from it; the warp barrier
    // orders their accesses to the slot after what that lane acquired (a
    // shuffle orders no memory)
    auto wait = [&](uint64_t *b, uint32_t parity, uint32_t pause_ns) -> bool {
        bool ok = true;
        if (lane == 0) ok = mbar_try_wait(b, parity) || st_wait_slow(b, parity, pause_ns, &s_err, ctl);
        ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
        __syncwarp();
        return ok;
    };

    uint32_t nflip = 0;
    if (warp >= 2 * cwarps) {
        // ---- producers: every pwarps-th block of the stream of nblk blocks a
        // sweep
        const uint32_t ctr3 = (kTagFlip << 24) | (uint32_t)(g + d.gbase);
        const int32_t total = nblk * S;
        const int first = warp - 2 * cwarps;
        int32_t sw = 0, blk = first, last = -1;
        // the record of the block after this one is loaded while this one is worked on
        int2 prn = make_int2(0, 0);
        int32_t nsw = 0, nbk = blk;
        auto next_record = [&]() {
            while (nbk >= nblk) { nbk -= nblk; ++nsw; }
            if (nsw < S) prn = d.spos[(sb0 + nsw) * (size_t)n + min(nbk * 32 + lane, n - 1)];
            nbk += pwarps;
        };
        next_record();
        for (int32_t b = first; b < total; b += pwarps, blk += pwarps) {
            while (blk >= nblk) { blk -= nblk; ++sw; }
            const int2 pr = prn;
            next_record();
            const int s = b & (nb - 1);
            const int32_t round = b >> (31 - __clz(nb));
            if (round > 0 && !wait(&empty[s], (uint32_t)((round - 1) & 1), 200)) break;
            uint8_t *slot = ring + (size_t)s * lay.slot;
            const size_t sb = sb0 + sw;
            if (lane == 0) {
                mbar_expect_tx(&full[s], 128u * (uint32_t)W);
                bulk_load(slot, d.sell + sb * ell_stride + (size_t)blk * 32 * W, 128u * (uint32_t)W, &full[s]);
            }
            last = b;
            const u32x4 u = philox_rk((uint32_t)(pr.x & 0xFFFFFF), (uint32_t)sw, (uint32_t)d.t, ctr3, d.K);
            reinterpret_cast<int2 *>(slot + 128u * (uint32_t)W)[lane] = pr;
            reinterpret_cast<uint4 *>(slot + 128u * (uint32_t)W + 256u)[lane] = make_uint4(u.x, u.y, u.z, u.w);
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[s]);
        }
        // the consumers wait for every block they read; on an error this warp's
        // last copies are waited for here (bounded) before the CTA leaves
        if (*(volatile int *)&s_err)
            for (int32_t b = last; b >= 0 && b > last - nb; b -= pwarps)
                mbar_wait(&full[b & (nb - 1)], (uint32_t)((b / nb) & 1));
    } else {
        // ---- consumers
        constexpr int NVW = 32 / LPV;                 // vertices of a warp's pass
        constexpr int NQ = LPV >= 4 ? 1 : 4 / LPV;    // replicas a lane decides
        const int set = warp / cwarps, vl = (warp % cwarps) * NVW + lane % NVW, sub = lane / NVW;
        const int vpi = cwarps * NVW;                 // vertices of a pass
        const int q0 = (sub * NQ) & 3;
        const int32_t V = W >> 2, cthreads = 2 * cwarps * 32;
        const bool owner = sub * NQ < 4;
        uint32_t alive = 0u;   // the replicas of this lane that exist
#pragma unroll
        for (int q = 0; q < NQ; ++q) alive |= owner && r0 + q0 + q < R ? 1u << q : 0u;
        Half *spq = reinterpret_cast<Half *>(sp);
        int32_t rb = 0, freed = 0;   // blocks known to be full / handed back
        bool bad = false;            // a block did not arrive: zeros are read in its place, the launch reports it
        // the pass to read next: sweep, level (in the sweep, and counted over the
        // launch), first position and the end of its level; the level ends of
        // 32 levels sit across the warp's lanes, the next 32 are on their way
        int32_t fsw = 0, glev = 0, flev = 0, fL = 0, fbase = 0, fe1 = 0, lv0 = 0, lv1 = 0;
        const int32_t *flp = nullptr;
        auto open_sweep = [&]() {
            flp = d.slvl + (sb0 + fsw) * (size_t)(n + 1);
            fL = d.snlev[sb0 + fsw];
            lv0 = flp[min(1 + lane, fL)];
            lv1 = flp[min(33 + lane, fL)];
            flev = 0;
            fbase = 0;
            fe1 = __shfl_sync(0xffffffffu, lv0, 0);
        };
        // where this lane's groups of four lie in a block: byte offset and the
        // permutation of the positions (beyond the row: the zeros at zero_off)
        uint32_t goff[NV], grot[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const uint32_t x = (uint32_t)(sub + v * LPV);
            goff[v] = x < (uint32_t)V ? x * 512u : 0xFFFFFFFFu;
            grot[v] = ell_rot(x);
        }
        const uint32_t slot_bytes = lay.slot, rec_off = 128u * (uint32_t)W, nbm = (uint32_t)nb - 1u;
        const int nb_log = 31 - __clz(nb);
        const uint32_t ring0 = smem_u32(ring), zero0 = smem_u32(smem + lay.red + 32);
        struct Pass {
            int2 pr;
            uint4 e[NV];
            uint32_t u[NQ];
            uint32_t slot;   // shared address of the block's slot
            int32_t pi, base, sw, lev;   // position in the block; the pass's first position, sweep and level
            bool act;
        };
        auto advance = [&]() {   // to the next pass
            fbase += vpi;
            if (fbase < fe1 || fsw >= S) return;
            ++glev;
            if (++flev < fL) {
                fbase = fe1;
                if ((flev & 31) == 0) {
                    lv0 = lv1;
                    lv1 = flp[min(flev + 33 + lane, fL)];
                }
                fe1 = __shfl_sync(0xffffffffu, lv0, flev & 31);
            } else if (++fsw < S) {
                open_sweep();
            }
        };
        auto read = [&](Pass &P) {
            P.sw = fsw;
            if (fsw >= S) return;
            const int32_t i = fbase + vl, lastp = min(fbase + vpi, fe1) - 1, ic = min(i, lastp);
            P.act = i < fe1;
            P.base = fbase;
            P.lev = glev;
            const int32_t sblk = fsw * nblk;
            const int32_t need = sblk + (lastp >> 5);
            while (rb <= need) {
                bad |= !wait(&full[(uint32_t)rb & nbm], (uint32_t)(rb >> nb_log) & 1u, 20);
                ++rb;
            }
            const uint32_t pi = (uint32_t)ic & 31u;
            P.slot = ring0 + ((uint32_t)(sblk + (ic >> 5)) & nbm) * slot_bytes;
            P.pi = (int32_t)pi;
            P.pr = lds64(bad ? zero0 : P.slot + rec_off + 8u * pi);
#pragma unroll
            for (int v = 0; v < NV; ++v)
                P.e[v] = lds128(goff[v] != 0xFFFFFFFFu && !bad ? P.slot + goff[v] + ((pi ^ grot[v]) << 4) : zero0);
            const uint32_t ua = P.slot + rec_off + 256u + 16u * pi + 4u * (uint32_t)q0;
#pragma unroll
            for (int q = 0; q < NQ; ++q) P.u[q] = lds32(ua + 4u * q);
            advance();   // (the other set's pass)
            advance();
        };
        // every thread of both sets moves from level to level together
        int32_t cur = 0;
        auto level_barrier = [&]() {
            asm volatile("bar.sync 1, %0;" ::"r"(cthreads) : "memory");
            ++cur;
        };
        Pass pa, pb;
        open_sweep();
        if (set) advance();
        read(pa);
        // one pass: sums and decides a, reads the next one into b; true: go on
        auto step = [&](Pass &a, Pass &b) -> bool {
            if (a.sw >= S) return false;
            while (cur < a.lev) level_barrier();
            const int32_t k = a.pr.x & 0xFFFFFF;
            Lanes s0, s1;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                s0.add(a.e[v].x, sp);
                s1.add(a.e[v].y, sp);
                s0.add(a.e[v].z, sp);
                s1.add(a.e[v].w, sp);
            }
            const Word old = sp[k];
            s0.join(s1);
            if (NV == 3 && !bad) {   // rows longer than what was read ahead
                const int32_t deg = (int32_t)((uint32_t)a.pr.x >> 24);
                for (int32_t x = sub + NV * LPV; 4 * x < deg; x += LPV) {
                    const uint4 e = lds128(a.slot + (uint32_t)x * 512u + (((uint32_t)a.pi ^ ell_rot((uint32_t)x)) << 4));
                    s0.add(e.x, sp);
                    s0.add(e.y, sp);
                    s0.add(e.z, sp);
                    s0.add(e.w, sp);
                }
            }
#pragma unroll
            for (int o = NVW; o < 32; o <<= 1) s0.xor_add(o);
            s0.bias();
            const int32_t c0 = H - 2 * (int32_t)Lanes::kBias - pos_jsum(a.pr.y);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const uint32_t ob = Lanes::bit(old, q0 + q);
                const int32_t idx = 2 * s0.lane(q0 + q) + c0;   // h + H
                const int32_t ix = RULE == 0 || ob ? idx : 2 * H - idx;   // (Metropolis: s h + H)
                uint64_t T;
                if constexpr (TABS) T = tab_s[ix];
                else T = __ldg(&d.tab[ix]);
                const uint32_t nw = ((uint64_t)a.u[q] < T ? 1u : 0u) ^ (RULE == 0 ? 0u : ob);
                if (a.act && owner && nw != ob) {
                    spq[4 * k + q0 + q] = (Half)nw;
                    nflip += (alive >> q) & 1u;
                }
            }
            // the level ends here for this set unless its next pass is in it too;
            // then the next pass is read while the other set works
            if (cur < (fsw < S ? glev : glev - 1)) level_barrier();
            read(b);
            // blocks before this warp's next pass are not read by it any more: the
            // warp barrier puts every lane's reads (the long rows' loop above ends
            // at each lane's own degree) before the arrival that hands them back
            const int32_t upto = b.sw < S ? b.sw * nblk + (b.base >> 5) : S * nblk;
            __syncwarp();
            if (lane == 0)
                for (int32_t x = freed; x < upto; ++x) mbar_arrive(&empty[(uint32_t)x & nbm]);
            freed = upto;
            return true;
        };
        while (step(pa, pb) && step(pb, pa)) {}
        // the levels left to the other set
        while (cur + 1 < glev) level_barrier();
    }
    __syncthreads();
    if (s_err) return;   // (the copies have landed: the consumers wait for every block, or a wait ran out)
    unsigned long long fl = nflip;
    for (int o = 16; o > 0; o >>= 1) fl += __shfl_down_sync(0xffffffffu, fl, o);
    if (lane == 0 && fl != 0ull) atomicAdd(reinterpret_cast<unsigned long long *>(&ctl->sweep_flips), fl);

    // energy from the definition, E = -1/2 sum_k s_k h_k, by position over the
    // last sweep's rows, and the write-back
    long long acc[4] = {0, 0, 0, 0};
    const uint32_t *es = d.sell + (sb0 + (S - 1)) * ell_stride;
    const int2 *pos = d.spos + (sb0 + (S - 1)) * (size_t)n;
    for (int32_t i = threadIdx.x; i < n; i += blockDim.x) {
        const int2 pr = pos[i];
        const int32_t deg = (int32_t)((uint32_t)pr.x >> 24);
        Lanes s0;
        for (int32_t v = 0; 4 * v < deg; ++v) {
            const uint4 e = ell4(es, i, W, v);
            s0.add(e.x, sp);
            s0.add(e.y, sp);
            s0.add(e.z, sp);
            s0.add(e.w, sp);
        }
        s0.bias();
        const Word w = sp[pr.x & 0xFFFFFF];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int32_t h = 2 * (s0.lane(q) - (int32_t)Lanes::kBias) - pos_jsum(pr.y);
            acc[q] += Lanes::bit(w, q) ? h : -h;
        }
    }
    for (int32_t k = threadIdx.x; k < n; k += blockDim.x) {
        const Word w = sp[k];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (r0 + q < R) d.dst[(size_t)(r0 + q) * n + k] = Lanes::bit(w, q) ? 1 : -1;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        long long v = acc[q];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) atomicAdd(&red[q], (unsigned long long)v);
    }
    __syncthreads();
    if (threadIdx.x < 4 && r0 + (int)threadIdx.x < R) d.E_dst[r0 + threadIdx.x] = -((long long)red[threadIdx.x] / 2);
}

}  // namespace

// Ring slots for the shape: as many as fit beside the spins, 0 where they do
// not hold four passes (each set's pass at work and the one it reads).
int sweep_staged_ring(int32_t n, int32_t H, int32_t W, SweepCfg cfg) {
    const bool wide = H > kByteLaneMaxH;
    const bool ts = sweep_staged_tab_smem(H);
    const int vpi = cfg.warps_per_group * 32 / cfg.lanes_per_vertex;
    for (int nb = kStRingMax; nb >= 4 && nb >= 4 * ((vpi + 31) / 32) + 2; nb >>= 1)
        if (st_layout(n, H, W, nb, wide, ts).total <= 227 * 1024) return nb;
    return 0;
}

// (byte lanes always: H <= 127)
bool sweep_staged_tab_smem(int32_t H) { return (2 * H + 1) * 8 <= 48 * 1024; }

cudaError_t launch_sweep_ising_staged(int rule, int32_t n, int32_t H, const pamc_params &p, int32_t t, int32_t slot,
                                      SchedView sv, const uint64_t *tab, const int8_t *src, const int32_t *parent,
                                      const int8_t *ncm_buf, const int32_t *ncm_idx, int8_t *dst, int64_t *E_dst,
                                      const DevCtl *ctl, SweepCfg cfg, cudaStream_t st, int32_t rbase) {
    const int nb = sweep_staged_ring(n, H, sv.W, cfg);
    if (sv.ell == nullptr || p.sweeps < 1 || nb == 0 || cfg.lanes_per_vertex > 8) return cudaErrorInvalidValue;
    const bool wide = H > kByteLaneMaxH, ts = sweep_staged_tab_smem(H);
    SweepDesc d;
    memset(&d, 0, sizeof(d));
    d.slvl = sv.lvl_ptr; d.snlev = sv.nlev; d.sell = sv.ell; d.spos = sv.pos;
    d.tab = tab; d.src = src; d.parent = parent; d.ncm_buf = ncm_buf; d.ncm_idx = ncm_idx;
    d.dst = dst; d.E_dst = E_dst; d.ctl = ctl; d.n = n; d.H = H; d.R = p.R;
    d.S = p.sweeps; d.t = t; d.slot = slot; d.W = sv.W; d.K = make_philox_keys(p.seed);
    d.gbase = rbase / 4;
    const size_t smem = st_layout(n, H, sv.W, nb, wide, ts).total;
    const int grid = (p.R + 3) / 4, cw = cfg.warps_per_group;
    const int pw = cw <= 2 ? 2 : 4;
    const int lpv = cfg.lanes_per_vertex, nv = ((sv.W >> 2) + lpv - 1) / lpv;
    cudaError_t err = cudaErrorInvalidValue;
#define PAMC_ST_T(RU, LV, NVV, LT, TS)                                                                 \
    do {                                                                                               \
        err = allow_dynamic_smem(k_sweep_ising_staged<RU, LV, NVV, LT, TS>, smem);                     \
        if (err != cudaSuccess) return err;                                                            \
        k_sweep_ising_staged<RU, LV, NVV, LT, TS><<<grid, (2 * cw + pw) * 32, smem, st>>>(d, cw, nb);      \
    } while (0)
#define PAMC_ST(RU, LV, NVV, LT)                                                                       \
    do {                                                                                               \
        if (ts) PAMC_ST_T(RU, LV, NVV, LT, true);                                                      \
        else PAMC_ST_T(RU, LV, NVV, LT, sizeof(LT::Word) == 4);                                        \
    } while (0)
#define PAMC_ST_V(RU, LV, LT)                                                                          \
    do {                                                                                               \
        if (nv <= 1) PAMC_ST(RU, LV, 1, LT);                                                           \
        else if (nv == 2) PAMC_ST(RU, LV, 2, LT);                                                      \
        else PAMC_ST(RU, LV, 3, LT);                                                                   \
    } while (0)
#define PAMC_ST_L(RU, LT)                                                                              \
    do {                                                                                               \
        switch (lpv) {                                                                                 \
        case 8: PAMC_ST_V(RU, 8, LT); break;                                                           \
        case 4: PAMC_ST_V(RU, 4, LT); break;                                                           \
        case 2: PAMC_ST_V(RU, 2, LT); break;                                                           \
        default: PAMC_ST_V(RU, 1, LT); break;                                                          \
        }                                                                                              \
    } while (0)
    if (wide) {
        if (rule == 0) PAMC_ST_L(0, WideLanes);
        else PAMC_ST_L(1, WideLanes);
    } else {
        if (rule == 0) PAMC_ST_L(0, ByteLanes);
        else PAMC_ST_L(1, ByteLanes);
    }
#undef PAMC_ST_L
#undef PAMC_ST_V
#undef PAMC_ST
#undef PAMC_ST_T
    return cudaGetLastError();
}

}  // namespace pamc
