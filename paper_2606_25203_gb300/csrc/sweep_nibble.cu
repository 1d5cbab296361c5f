// sweep_nibble.cu -- the Ising sweep (Eq. 3-4) with EIGHT replicas per
// 32-bit word, for instances whose field range fits 4-bit lanes.
//
// Layout.  Nibble q of a vertex's word holds the spin of replica 8g + q of
// replica group g (1 = +1).  A neighbour costs one ELL word, one shared load
// and one multiply-add for eight replicas (twice the byte lanes' four), and a
// group's words take the same 4n bytes of shared memory for twice the
// replicas.
//
// Satisfied weight.  With M the weight of the negative couplings of a half-row
// (ELL slots 0..7 or 8..15), A = M 0x11111111 + sum_{j in half} J_kj word_j has
// nibble q = N_q = sum_{J > 0} J [s_j = +1] + sum_{J < 0} |J| [s_j = -1], in
// [0, 15] wherever the half's sum |J| <= 15 (every partial sum stays in range,
// so the word sums exactly), and h_q = 2 N_q - D, D = sum_j |J_kj|.  One half
// (D <= 7 on rows of at most eight slots: the +-1 torus, graphs of degree <= 7)
// keeps the nibbles; two halves are added in byte lanes (sums <= 30).  M, M'
// and D come with the position's record (pos_sums).
//
// Decision.  For a vertex of weight D the new spin depends on the draw and an
// index x in [0, D], the threshold rising with x: heat-bath x = N (s = +1 iff
// u < T(2x - D)), Metropolis x = the unsatisfied weight D - N for s = +1, N for
// s = -1 (flip iff u < T_M(D - 2x)).  At a negative beta, heat-bath, the
// threshold falls with the field: x = D - N, T(D - 2x).  Shared memory holds a row of 32-bit
// thresholds for each D, 256 bytes apart, so that the address of a replica's
// entry is the row address with its lowest byte replaced by 4 x: one byte
// permute.  A threshold of 2^32 (always) does not fit 32 bits: those entries
// hold 2^32 - 1, and the replicas with x at or beyond the first such entry are
// set by one addition over the word (nibble or byte x + 8 - x_f, + 128 - x_f:
// the top bit).  A decision then takes a permute, a shared load, a compare and
// a predicated addition.
//
// Bound: the integer pipe (half the issue rate), Philox about a third of it:
// 247 instructions a visit of eight replicas (260 with biased field lanes and
// 64-bit thresholds, whose launches took 1,247 us against 1,138 on the
// 141 x 141 torus, R = 4,096, 10 sweeps).
//
// Draws.  Replica r uses word r mod 4 of Philox(k, sweep, t, FLIP<<24 | r/4)
// as everywhere else: the eight replicas of a word take two calls, of the
// four-replica groups 2g and 2g + 1 (offset by the population's group base),
// so the results are those of the byte-lane kernel bit for bit.
//
// Order: the (t, sweep) schedule's dependency levels with position-indexed
// ELL rows, one barrier per level, as in sweep_ising.cu.
#include <cstdlib>
#include <cstring>

#include "pamc_device.cuh"
#include "pamc_internal.h"

namespace pamc {

namespace {

// Philox draws with the round keys of the seed in kernel parameter space, or
// advanced from the seed (batched launches: the key differs per member).
struct NibKeys {
    const PhiloxKeys &K;
    __device__ __forceinline__ u32x4 operator()(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3) const {
        return philox_rk(c0, c1, c2, c3, K);
    }
};
struct NibKeysSeed {
    uint32_t k0, k1;
    __device__ __forceinline__ u32x4 operator()(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3) const {
        return philox(c0, c1, c2, c3, k0, k1);
    }
};

__device__ __forceinline__ void nib_barrier(int id, int nthreads, int groups) {
    if (groups == 1) {
        __syncthreads();
    } else {
        asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
    }
}

// four couplings of a row on the neighbours' spin words
__device__ __forceinline__ uint32_t nib_add4(uint32_t A, const uint4 &e, const uint32_t *sp) {
    A += sp[e.x & 0xFFFFFFu] * (uint32_t)((int32_t)e.x >> 24);
    A += sp[e.y & 0xFFFFFFu] * (uint32_t)((int32_t)e.y >> 24);
    A += sp[e.z & 0xFFFFFFu] * (uint32_t)((int32_t)e.z >> 24);
    return A + sp[e.w & 0xFFFFFFu] * (uint32_t)((int32_t)e.w >> 24);
}

__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
// w + bit where u < T
__device__ __forceinline__ void add_if_below(uint32_t &w, uint32_t u, uint32_t T, uint32_t bit) {
    asm("{\n .reg .pred p;\n setp.lt.u32 p, %1, %2;\n @p add.u32 %0, %0, %3;\n}" : "+r"(w) : "r"(u), "r"(T), "r"(bit));
}

// bytes of the threshold rows and, per row, the word that marks the entries of
// 2^32: rows D = 0..H, 256 bytes apart (the row address has a clear low byte)
constexpr int32_t kNibRow = 64;
__host__ __device__ constexpr size_t nib_table_bytes(int32_t H) { return (size_t)(H + 1) * (kNibRow * 4 + 4) + 12 + 256; }

// The decisions of eight replicas: E, O the index of the even and the odd
// replicas in bytes, row the address of the vertex's thresholds, force its
// mark word, X the index nibbles (one half only).
template <int RULE, bool TWO>
__device__ __forceinline__ uint32_t nib_decide(uint32_t X, uint32_t E, uint32_t O, uint32_t D, uint32_t row,
                                               uint32_t force, const u32x4 &ua, const u32x4 &ub, uint32_t old) {
    if constexpr (RULE == 2) {   // the index counts the other way
        if constexpr (TWO) {
            E = D * 0x01010101u - E;
            O = D * 0x01010101u - O;
        } else {
            X = D * 0x11111111u - X;
        }
    } else if constexpr (RULE == 1) {   // the unsatisfied weight of the replicas with s = +1
        if constexpr (TWO) {
            const uint32_t me = (old & 0x01010101u) * 0xFFu, mo = ((old >> 4) & 0x01010101u) * 0xFFu;
            const uint32_t D4 = D * 0x01010101u;
            E = (E & ~me) | ((D4 - E) & me);
            O = (O & ~mo) | ((D4 - O) & mo);
        } else {
            const uint32_t m = old * 0xFu;
            X = (X & ~m) | ((D * 0x11111111u - X) & m);
        }
    }
    uint32_t e4, o4;   // 4 x of the even and the odd replicas, in bytes
    if constexpr (TWO) {
        e4 = E << 2;
        o4 = O << 2;
    } else {
        e4 = (X << 2) & 0x3C3C3C3Cu;
        o4 = (X >> 2) & 0x3C3C3C3Cu;
    }
    const uint32_t uw[8] = {ua.x, ua.y, ua.z, ua.w, ub.x, ub.y, ub.z, ub.w};
    uint32_t n0 = 0u, n1 = 0u;
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
        const uint32_t te = lds_u32(__byte_perm(e4, row, 0x7650u + (q >> 1)));
        const uint32_t to = lds_u32(__byte_perm(o4, row, 0x7650u + (q >> 1)));
        add_if_below(n0, uw[q], te, 1u << (4 * q));
        add_if_below(n1, uw[q + 1], to, 16u << (4 * q));
    }
    uint32_t nw = n0 | n1;
    if constexpr (TWO) {
        nw |= ((E + force) >> 7) & 0x01010101u;
        nw |= ((O + force) >> 3) & 0x10101010u;
    } else {
        nw |= ((X + force) >> 3) & 0x11111111u;
    }
    return RULE == 1 ? nw ^ old : nw;
}

__device__ __forceinline__ void nib_halves(uint32_t A1, uint32_t A2, uint32_t &E, uint32_t &O) {
    E = (A1 & 0x0F0F0F0Fu) + (A2 & 0x0F0F0F0Fu);
    O = ((A1 >> 4) & 0x0F0F0F0Fu) + ((A2 >> 4) & 0x0F0F0F0Fu);
}

// Whether the heat-bath thresholds fall with the field (beta < 0): RULE 2 of the
// bodies below, chosen once a launch (a branch at every visit cost 2 % of a small
// instance's launch).
__device__ __forceinline__ bool nib_falling(const SweepDesc &d) { return d.tab[0] > d.tab[2 * d.H]; }

// The sweeps of one CTA's groups of eight (groups bid*gpc .. bid*gpc+gpc-1
// of the instance), shared by the single-instance and the batched kernels;
// WC = 0: the ELL width read at run time; TWO: both halves of the rows (width 4
// to 16), else one (width 4 or 8).
template <int RULE, int WC, bool TWO, class KeyT>
__device__ __forceinline__ void
nib_body(const SweepDesc &d, const KeyT &draw, int32_t t, int32_t slot, const int8_t *__restrict__ src,
         int8_t *__restrict__ dst, int64_t *__restrict__ E_dst, int gpc, int tpg, int32_t bid) {
    extern __shared__ __align__(16) uint8_t smem[];
    const DevCtl *ctl = d.ctl;
    if (ctl->done) return;
    const int32_t n = d.n, n_pad = d.n_pad, H = d.H, R = d.R, S = d.S;
    const int32_t W = WC > 0 ? WC : d.W;
    // threshold rows at the first 256-byte boundary, the marks behind them
    const uint32_t smem0 = (uint32_t)__cvta_generic_to_shared(smem);
    const uint32_t rows0 = (smem0 + 255u) & ~255u;
    uint32_t *tab_s = reinterpret_cast<uint32_t *>(smem + (rows0 - smem0));
    uint32_t *mark_s = tab_s + (H + 1) * kNibRow;
    const uint32_t marks0 = rows0 + (uint32_t)(H + 1) * (kNibRow * 4);
    uint32_t *spins_all = reinterpret_cast<uint32_t *>(smem + ((nib_table_bytes(H) + 15) & ~(size_t)15));
    unsigned long long *red = reinterpret_cast<unsigned long long *>(spins_all + (size_t)gpc * n_pad);
    // (on its way while the spins are read; used below)
    const uint64_t first = (int)threadIdx.x < 2 * H + 1 ? d.tab[threadIdx.x] : 0ull;
    for (int i = threadIdx.x; i < gpc * 8; i += blockDim.x) red[i] = 0ull;

    const int gl = threadIdx.x / tpg, li = threadIdx.x % tpg;
    const int32_t g = bid * gpc + gl;   // group of eight replicas
    const int32_t r0 = g * 8;
    const bool active = r0 < R;
    // the spin bits (bit 4q) of the replicas r0 + q < R, for the flip count
    const uint32_t live = R - r0 >= 8 ? 0x11111111u : R - r0 <= 0 ? 0u : 0x11111111u & ((1u << (4 * (R - r0))) - 1u);
    uint32_t *sp = spins_all + (size_t)gl * n_pad;

    if (active) {
        // slot r reads the NCM output if the cluster move rewrote it, else its
        // resampling parent (the replica copy of the population step)
        const int8_t *rows[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int32_t r = r0 + q;
            if (r < R) {
                const int32_t m = d.ncm_idx[r];
                rows[q] = m >= 0 ? d.ncm_buf + (size_t)m * n : src + (size_t)d.parent[r] * n;
            } else {
                rows[q] = nullptr;
            }
        }
        for (int32_t k = li; k < n; k += tpg) {
            uint32_t w = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (rows[q] != nullptr) w |= (uint32_t)(rows[q][k] > 0) << (4 * q);
            sp[k] = w;
        }
    }
    // entries below 2^32 of the table, in rising order: row D's first one of 2^32
    // is at 2 xf - D + H >= below (D + 1: none)
    int32_t below = 0;
    for (int32_t b = 0; b < 2 * H + 1; b += blockDim.x)
        below += __syncthreads_count(b + (int)threadIdx.x < 2 * H + 1 &&
                                     (b == 0 ? first : d.tab[b + threadIdx.x]) <= 0xFFFFFFFFull);
    // tab[h + H] (heat-bath), tab[s h + H] (Metropolis): h = 2x - D (D - 2x where
    // the thresholds fall with the field, beta < 0), s h = D - 2x
    for (int i = threadIdx.x; i < (H + 1) * (H + 1); i += blockDim.x) {
        const int32_t D = i / (H + 1), x = i % (H + 1);
        if (x > D) continue;
        const uint64_t T = d.tab[RULE == 0 ? 2 * x - D + H : D - 2 * x + H];
        tab_s[D * kNibRow + x] = T > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)T;
    }
    for (int32_t D = threadIdx.x; D <= H; D += blockDim.x) {
        const int32_t xf = min(max((below + D - H + 1) >> 1, 0), D + 1);
        mark_s[D] = TWO ? (uint32_t)(128 - xf) * 0x01010101u : (uint32_t)(8 - xf) * 0x11111111u;
    }
    __syncthreads();

    if (active) {
        const size_t ell_stride = (size_t)(((n + 31) >> 5) << 5) * W;
        const uint32_t ctrA = (kTagFlip << 24) | (uint32_t)(2 * g + d.gbase);
        const uint32_t ctrB = ctrA + 1u;
        uint32_t nflip = 0;
        for (int32_t sw = 0; sw < S; ++sw) {
            const size_t sb = (size_t)slot * S + sw;
            const int32_t *lp = d.slvl + sb * (size_t)(n + 1);
            const uint32_t *es = d.sell + sb * ell_stride;
            const int2 *pos = d.spos + sb * (size_t)n;
            const int32_t L = d.snlev[sb];
            // the record and the first four couplings of a position (the first
            // eight where the rows have more) are loaded one iteration ahead --
            // for a level's first position before the previous level's barrier
            // (they do not depend on spins)
            int2 pr = make_int2(0, 0);
            uint4 e4 = make_uint4(0u, 0u, 0u, 0u), f4 = e4;
            int32_t end = 0;
            if (L > 0) {
                const int32_t i0 = min(li, n - 1);
                pr = pos[i0];
                e4 = ell4(es, i0, W, 0);
                if (W > 4) f4 = ell4(es, i0, W, 1);
            }
            for (int32_t lev = 0; lev < L; ++lev) {
                const int32_t beg = lp[lev];
                end = lp[lev + 1];
                int32_t i = beg + li;
                while (i < end) {
                    const int32_t inext = i + tpg;
                    int2 prn = make_int2(0, 0);
                    uint4 e4n = make_uint4(0u, 0u, 0u, 0u), f4n = e4n;
                    if (inext < end) {
                        prn = pos[inext];
                        e4n = ell4(es, inext, W, 0);
                        if (W > 4) f4n = ell4(es, inext, W, 1);
                    }
                    const uint32_t a0 = (uint32_t)pr.x;
                    const int32_t k = (int32_t)(a0 & 0xFFFFFFu);
                    const uint32_t ys = (uint32_t)pr.y;
                    uint32_t A = ((ys >> 16) & 15u) * 0x11111111u, A2 = 0u;
                    A = nib_add4(A, e4, sp);   // (padding slots: coupling 0)
                    if (W > 4) A = nib_add4(A, f4, sp);
                    if constexpr (TWO) {
                        // slots 8..15 into the second half, in groups of four
                        // while the degree asks for them (levels are grouped
                        // by degree, so a warp's lanes mostly agree)
                        A2 = ((ys >> 20) & 15u) * 0x11111111u;
                        const int32_t deg = (int32_t)(a0 >> 24);
                        if (W > 8 && deg > 8) {
                            A2 = nib_add4(A2, ell4(es, i, W, 2), sp);
                            if (W > 12 && deg > 12) A2 = nib_add4(A2, ell4(es, i, W, 3), sp);
                        }
                    }
                    const u32x4 ua = draw((uint32_t)k, (uint32_t)sw, (uint32_t)t, ctrA);
                    const u32x4 ub = draw((uint32_t)k, (uint32_t)sw, (uint32_t)t, ctrB);
                    const uint32_t old = sp[k];
                    const uint32_t D = ys >> 24;
                    const uint32_t row = rows0 + (D << 8), force = lds_u32(marks0 + (D << 2));
                    uint32_t E = 0u, O = 0u;
                    if constexpr (TWO) nib_halves(A, A2, E, O);
                    const uint32_t nw = nib_decide<RULE, TWO>(A, E, O, D, row, force, ua, ub, old);
                    if (nw != old) {
                        sp[k] = nw;
                        nflip += __popc((nw ^ old) & live);
                    }
                    i = inext;
                    pr = prn;
                    e4 = e4n;
                    f4 = f4n;
                }
                if (lev + 1 < L) {   // the next level's first position (clamped, see above)
                    const int32_t i2 = min(end + li, n - 1);
                    pr = pos[i2];
                    e4 = ell4(es, i2, W, 0);
                    if (W > 4) f4 = ell4(es, i2, W, 1);
                }
                nib_barrier(1 + gl, tpg, gpc);
            }
        }
        // spins that changed at a visit, summed per warp into the controller
        unsigned long long v = nflip;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0 && v != 0ull)
            atomicAdd(reinterpret_cast<unsigned long long *>(&const_cast<DevCtl *>(ctl)->sweep_flips), v);

        // energy from the definition E = -1/2 sum_k s_k h_k over the last
        // sweep's ELL rows (|s h| <= 30 per vertex: int32 per thread), and the
        // write-back of the eight rows
        int32_t acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        const size_t sb = (size_t)slot * S + (S - 1);   // S >= 1 (sweep_nibble_ok)
        const uint32_t *es = d.sell + sb * ell_stride;
        const int2 *pos = d.spos + sb * (size_t)n;
        for (int32_t i = li; i < n; i += tpg) {
            const int2 p0 = pos[i];
            const uint32_t w = sp[p0.x & 0xFFFFFF];
            const uint32_t ys = (uint32_t)p0.y;
            const int32_t D = (int32_t)(ys >> 24);
            uint32_t A = ((ys >> 16) & 15u) * 0x11111111u, A2 = TWO ? ((ys >> 20) & 15u) * 0x11111111u : 0u;
#pragma unroll
            for (int v = 0; v < (TWO ? 4 : 2); ++v) {
                if (4 * v >= W) break;
                if (v < 2) A = nib_add4(A, ell4(es, i, W, v), sp);
                else A2 = nib_add4(A2, ell4(es, i, W, v), sp);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int32_t h = 2 * (int32_t)(((A >> (4 * q)) & 0xFu) + ((A2 >> (4 * q)) & 0xFu)) - D;
                acc[q] += ((w >> (4 * q)) & 1u) ? h : -h;
            }
        }
        for (int32_t k = li; k < n; k += tpg) {
            const uint32_t w = sp[k];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (r0 + q < R) dst[(size_t)(r0 + q) * n + k] = ((w >> (4 * q)) & 1u) ? 1 : -1;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            long long v2 = acc[q];
            for (int o = 16; o > 0; o >>= 1) v2 += __shfl_down_sync(0xffffffffu, v2, o);
            if ((threadIdx.x & 31) == 0) atomicAdd(&red[gl * 8 + q], (unsigned long long)v2);
        }
    }
    __syncthreads();
    if (active && li < 8 && r0 + li < R) E_dst[r0 + li] = -((long long)red[gl * 8 + li] / 2);
}

template <int RULE, int WC, bool TWO>
__global__ void __launch_bounds__(1024) k_sweep_ising_nib(SweepDesc d, int gpc, int tpg) {
    if (RULE == 0 && nib_falling(d))
        nib_body<2, WC, TWO>(d, NibKeys{d.K}, d.t, d.slot, d.src, d.dst, d.E_dst, gpc, tpg, blockIdx.x);
    else
        nib_body<RULE, WC, TWO>(d, NibKeys{d.K}, d.t, d.slot, d.src, d.dst, d.E_dst, gpc, tpg, blockIdx.x);
}

// Many instances in one launch: CTA b works on member items[b].x, its block
// of groups items[b].y; the step index comes from the member's controller.
template <int RULE, bool TWO>
__global__ void __launch_bounds__(1024)
k_sweep_ising_nib_batched(const SweepDesc *__restrict__ descs, const int2 *__restrict__ items, int gpc, int tpg) {
    const int2 it = items[blockIdx.x];
    const SweepDesc &d = descs[it.x];
    const int32_t t = d.ctl->t;
    if (t >= d.t_end) return;
    if (RULE == 0 && nib_falling(d))
        nib_body<2, 0, TWO>(d, NibKeysSeed{d.K.k0[0], d.K.k1[0]}, t, t % d.slots, d.sp[t & 1], d.sp[(t + 1) & 1],
                            d.en[(t + 1) & 1], gpc, tpg, it.y);
    else
        nib_body<RULE, 0, TWO>(d, NibKeysSeed{d.K.k0[0], d.K.k1[0]}, t, t % d.slots, d.sp[t & 1], d.sp[(t + 1) & 1],
                               d.en[(t + 1) & 1], gpc, tpg, it.y);
}

}  // namespace

bool sweep_nibble_enabled() {
    const char *env = getenv("PAMC_SWEEP_NIBBLE");
    return !(env && env[0] == '0');
}

int nibble_halves(int32_t n, const int32_t *rp, const uint32_t *adj, int32_t H, int32_t ell_w) {
    if (H <= kNibbleMaxH && (ell_w == 4 || ell_w == 8)) return 1;
    if (!(ell_w == 4 || ell_w == 8 || ell_w == 12 || ell_w == 16) || H > kNibbleTwoMaxH) return 0;
    for (int32_t k = 0; k < n; ++k) {
        int32_t slot = 0, half[2] = {0, 0};
        for (int32_t e = rp[k]; e < rp[k + 1]; ++e) {
            const int32_t J = (int32_t)adj[e] >> 24;
            if (J == 0) continue;   // the ELL rows hold the nonzero couplings only
            half[slot < 8 ? 0 : 1] += J < 0 ? -J : J;
            ++slot;
        }
        if (slot > ell_w || half[0] > kNibbleHalfMaxH || half[1] > kNibbleHalfMaxH) return 0;
    }
    return 2;
}

bool sweep_nibble_ok(int halves, int32_t S, int lanes_per_vertex, bool global_spins) {
    return halves > 0 && S > 0 && lanes_per_vertex == 1 && !global_spins && sweep_nibble_enabled();
}

size_t sweep_nibble_smem_bytes(int32_t n, int32_t H, SweepCfg cfg) {
    const int32_t n_pad = (n + 3) & ~3;
    return ((nib_table_bytes(H) + 15) & ~(size_t)15) + (size_t)cfg.groups_per_cta * n_pad * 4 +
           (size_t)cfg.groups_per_cta * 8 * 8;
}

cudaError_t launch_sweep_ising_nib(int rule, int32_t n, int32_t H, const pamc_params &p, int32_t t, int32_t slot,
                                   SchedView sv, const uint64_t *tab, const int8_t *src, const int32_t *parent,
                                   const int8_t *ncm_buf, const int32_t *ncm_idx, int8_t *dst, int64_t *E_dst,
                                   const DevCtl *ctl, SweepCfg cfg, cudaStream_t st, int32_t rbase) {
    const bool two = sv.halves == 2;
    if (!(sv.ell != nullptr && p.sweeps > 0 &&
          (two ? (sv.W % 4 == 0 && sv.W >= 4 && sv.W <= 16 && H <= kNibbleTwoMaxH)
               : (sv.halves == 1 && (sv.W == 4 || sv.W == 8) && H <= kNibbleMaxH))))
        return cudaErrorInvalidValue;
    const int32_t groups = (p.R + 7) / 8;
    const int gpc = cfg.groups_per_cta, tpg = cfg.warps_per_group * 32;
    SweepDesc d;
    memset(&d, 0, sizeof(d));
    d.sorder = sv.order; d.slvl = sv.lvl_ptr; d.snlev = sv.nlev; d.sell = sv.ell; d.spos = sv.pos;
    d.tab = tab; d.src = src; d.parent = parent; d.ncm_buf = ncm_buf; d.ncm_idx = ncm_idx;
    d.dst = dst; d.E_dst = E_dst; d.ctl = ctl; d.n = n; d.n_pad = (n + 3) & ~3; d.H = H; d.R = p.R;
    d.S = p.sweeps; d.t = t; d.slot = slot; d.W = sv.W; d.K = make_philox_keys(p.seed);
    d.gbase = rbase / 4;
    const size_t smem = sweep_nibble_smem_bytes(n, H, cfg);
    const int grid = (groups + gpc - 1) / gpc;
    cudaError_t err = cudaSuccess;
#define PAMC_NIB(RU, WV, BI)                                                                 \
    do {                                                                                     \
        err = allow_dynamic_smem(k_sweep_ising_nib<RU, WV, BI>, smem);                       \
        if (err != cudaSuccess) return err;                                                  \
        k_sweep_ising_nib<RU, WV, BI><<<grid, gpc * tpg, smem, st>>>(d, gpc, tpg);           \
    } while (0)
#define PAMC_NIB_W(RU)                                                                       \
    do {                                                                                     \
        if (!two) {                                                                       \
            if (sv.W == 4) PAMC_NIB(RU, 4, false);                                           \
            else PAMC_NIB(RU, 8, false);                                                     \
        } else if (sv.W == 4) PAMC_NIB(RU, 4, true);                                         \
        else if (sv.W == 8) PAMC_NIB(RU, 8, true);                                           \
        else if (sv.W == 12) PAMC_NIB(RU, 12, true);                                         \
        else PAMC_NIB(RU, 16, true);                                                         \
    } while (0)
    if (rule == 0) PAMC_NIB_W(0);
    else PAMC_NIB_W(1);
#undef PAMC_NIB_W
#undef PAMC_NIB
    return cudaGetLastError();
}

cudaError_t launch_sweep_ising_nib_batched(int rule, bool two, const SweepDesc *descs, const int2 *items,
                                           int32_t nitems, size_t smem, SweepCfg cfg, cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    const int gpc = cfg.groups_per_cta, tpg = cfg.warps_per_group * 32;
    cudaError_t err;
#define PAMC_NIBB(RU, BI)                                                                    \
    do {                                                                                     \
        err = allow_dynamic_smem(k_sweep_ising_nib_batched<RU, BI>, smem);                   \
        if (err != cudaSuccess) return err;                                                  \
        k_sweep_ising_nib_batched<RU, BI><<<nitems, gpc * tpg, smem, st>>>(descs, items, gpc, tpg); \
    } while (0)
    if (rule == 0) {
        if (two) PAMC_NIBB(0, true);
        else PAMC_NIBB(0, false);
    } else {
        if (two) PAMC_NIBB(1, true);
        else PAMC_NIBB(1, false);
    }
#undef PAMC_NIBB
    return cudaGetLastError();
}

}  // namespace pamc
