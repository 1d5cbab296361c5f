// sweep_bits.cu -- the Ising sweep (Eq. 3-4) with up to 32 replicas per word,
// one bit each, for instances whose couplings are all +-1 (or 0) with at most
// 63 neighbours a vertex.
//
// Layout.  A group holds 4 nc replicas, nc = 1..8; bit m + 8b of a vertex's word is
// the spin (1 = +1) of the group's replica 4m + b, so that the four replicas of
// one Philox call lie one to a byte.
//
// Sum.  A neighbour costs one ELL word, one shared load and an exclusive or
// with the coupling's sign for all replicas of the group; the bits are counted
// by carry-save adders into P bit planes (x = their sum, up to 2^P - 1), two
// three-input logic operations a neighbour.  Heat-bath counts x = N, the
// neighbours with J_kj s_j = +1 (h = 2N - D, D the row's weight); Metropolis the
// unsatisfied ones, J_kj s_j = -s_k (one more input to the exclusive or).  At a
// negative beta, heat-bath, the threshold falls with the field: the words then
// hold the spins inverted, which makes the count x = D - N.
//
// Decision.  As in sweep_nibble.cu: shared memory holds, for each D, a row of
// 32-bit thresholds 256 bytes apart; the planes are merged into bytes 4 x (pairs
// of bits, nibbles, bytes: about one operation a replica), a replica's
// threshold address is the row's with its lowest byte replaced (one byte
// permute), and a compare and a predicated addition set its bit.  Thresholds of
// 2^32 (always) are held as 2^32 - 1; the replicas they belong to, x at or beyond
// the row's first such entry, are found by the carry of x + 2^P - x_f over the
// planes, P operations for the whole word.
//
// Bound: the integer pipe (half the issue rate; which is why the decided bits are
// collected by the floating-point adder).  On the 141 x 141 torus with 28 replicas
// a word a visit takes 614 instructions, 473 of them integer and half of
// those Philox: 17 a replica against 24 on 4-bit lanes.  us per launch of 10 sweeps at R =
// 4,096, before (4-bit or byte lanes) / now: the torus 1,139 / 818, N=7,000
// degree 5.7 751 / 503, N=10,007 degree 20 2,962 / 1,114, N=2,000 degree 20 1,097 / 455.
// Longer rows than 8 also waited for their couplings: with up to 24 slots loaded
// ahead, while the draws and decisions of the pass before run, N=10,007 went from
// 1,335 to 1,114 us, N=20,000 degree 20 R=2,048 from 2,012 to 1,567.
//
// QL lanes share a vertex where a level has fewer vertices than the group has
// lanes: they split its groups of four couplings (the partial sums are added
// plane by plane) and its Philox calls.
//
// Draws, orders and results are those of the other Ising sweeps bit for bit.
#include <cstdlib>
#include <cstring>

#include "pamc_device.cuh"
#include "pamc_internal.h"

namespace pamc {

namespace {

constexpr int32_t kBitRow = 64;   // thresholds of a row (256 bytes)

// Round keys of the seed, in kernel parameter space or advanced from the seed
// (batched launches: the key differs per member).
struct BitKeys {
    const PhiloxKeys &K;
    __device__ __forceinline__ uint32_t k0(int i) const { return K.k0[i]; }
    __device__ __forceinline__ uint32_t k1(int i) const { return K.k1[i]; }
};
struct BitKeysSeed {
    uint32_t s0, s1;
    __device__ __forceinline__ uint32_t k0(int i) const { return s0 + (uint32_t)i * 0x9E3779B9u; }
    __device__ __forceinline__ uint32_t k1(int i) const { return s1 + (uint32_t)i * 0xBB67AE85u; }
};

// Philox4x32-10 of (c0, c1, c2, c3) for several c3: what the first three rounds
// have in common is computed once (34 operations a call of 40).
struct BitDraw {
    uint32_t x2, y1, w3, h, l;
    template <class K>
    __device__ __forceinline__ BitDraw(uint32_t c0, uint32_t c1, uint32_t c2, const K &key) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c0, p1 = (uint64_t)0xCD9E8D57u * c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ key.k0(0);
        x2 = (uint32_t)(p0 >> 32) ^ key.k1(0);
        y1 = (uint32_t)p1 ^ key.k0(1);
        const uint64_t q0 = (uint64_t)0xD2511F53u * n0;
        const uint32_t z2 = (uint32_t)(q0 >> 32) ^ (uint32_t)p0 ^ key.k1(1);
        w3 = (uint32_t)q0 ^ key.k1(2);
        const uint64_t q1 = (uint64_t)0xCD9E8D57u * z2;
        h = (uint32_t)(q1 >> 32) ^ key.k0(2);
        l = (uint32_t)q1;
    }
    template <class K>
    __device__ __forceinline__ u32x4 operator()(uint32_t c3, const K &key) const {
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * (x2 ^ c3);
        const uint64_t p0 = (uint64_t)0xD2511F53u * ((uint32_t)(p1 >> 32) ^ y1);
        uint32_t a = h ^ (uint32_t)p1, b = l, c = (uint32_t)(p0 >> 32) ^ w3, e = (uint32_t)p0;
#pragma unroll
        for (int i = 3; i < 10; ++i) {
            const uint64_t r0 = (uint64_t)0xD2511F53u * a, r1 = (uint64_t)0xCD9E8D57u * c;
            a = (uint32_t)(r1 >> 32) ^ b ^ key.k0(i);
            b = (uint32_t)r1;
            c = (uint32_t)(r0 >> 32) ^ e ^ key.k1(i);
            e = (uint32_t)r0;
        }
        return {a, b, c, e};
    }
};

__device__ __forceinline__ uint32_t bl_lds(uint32_t addr) {
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint4 bl_lds4(uint32_t addr) {
    uint4 v;
    asm("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
// w + bit where u < T (the bits of a word are collected in the significand of a
// float from 2^23 up: the floating-point adder has twice the integer rate)
__device__ __forceinline__ void bl_add_if_below(float &w, uint32_t u, uint32_t T, float bit) {
    asm("{\n .reg .pred p;\n setp.lt.u32 p, %1, %2;\n @p add.rn.f32 %0, %0, %3;\n}" : "+f"(w) : "r"(u), "r"(T), "f"(bit));
}
__device__ __forceinline__ uint32_t maj(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (c & (a | b)); }

// P bit planes counting up to 2^P - 1
template <int P>
struct Planes {
    uint32_t p[P];
    // adds four bits a replica
    __device__ __forceinline__ void add4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
        const uint32_t c0 = maj(p[0], a, b), s0 = p[0] ^ a ^ b;
        const uint32_t c1 = maj(s0, c, d);
        p[0] = s0 ^ c ^ d;
        uint32_t k = maj(p[1], c0, c1);
        p[1] ^= c0 ^ c1;
#pragma unroll
        for (int i = 2; i < P; ++i) {
            const uint32_t t = p[i] & k;
            p[i] ^= k;
            k = t;
        }
    }
    // adds eight bits a replica, given as two groups of four
    __device__ __forceinline__ void add8(const uint32_t (&a)[4], const uint32_t (&b)[4]) {
        const uint32_t c0 = maj(p[0], a[0], a[1]), s0 = p[0] ^ a[0] ^ a[1];
        const uint32_t c1 = maj(s0, a[2], a[3]), s1 = s0 ^ a[2] ^ a[3];
        const uint32_t c2 = maj(s1, b[0], b[1]), s2 = s1 ^ b[0] ^ b[1];
        const uint32_t c3 = maj(s2, b[2], b[3]);
        p[0] = s2 ^ b[2] ^ b[3];
        const uint32_t d0 = maj(p[1], c0, c1), s3 = p[1] ^ c0 ^ c1;
        const uint32_t d1 = maj(s3, c2, c3);
        p[1] = s3 ^ c2 ^ c3;
        uint32_t k = maj(p[2], d0, d1);
        p[2] ^= d0 ^ d1;
#pragma unroll
        for (int i = 3; i < P; ++i) {
            const uint32_t t = p[i] & k;
            p[i] ^= k;
            k = t;
        }
    }
    // the sums of the lanes o apart (o a power of two)
    __device__ __forceinline__ void merge(int o) {
        uint32_t c = 0u;
#pragma unroll
        for (int i = 0; i < P; ++i) {
            const uint32_t q = __shfl_xor_sync(0xffffffffu, p[i], o);
            const uint32_t s = p[i] ^ q ^ c;
            c = maj(p[i], q, c);
            p[i] = s;
        }
    }
    // nibbles of the low planes of the replicas c, c + 4, ...: pairs (planes 0
    // and 1; 2 and 3) of the replicas of c's parity, then nibbles
    __device__ __forceinline__ uint32_t nibbles(int c) const {
        const uint32_t q = (c & 1) ? ((p[0] >> 1) & 0x55555555u) | (p[1] & 0xAAAAAAAAu)
                                   : (p[0] & 0x55555555u) | ((p[1] << 1) & 0xAAAAAAAAu);
        if constexpr (P == 3) {
            const uint32_t lo = (c & 2) ? (q >> 2) & 0x33333333u : q & 0x33333333u;
            const uint32_t hi = c == 0 ? p[2] << 2 : c == 1 ? p[2] << 1 : c == 2 ? p[2] : p[2] >> 1;
            return lo | (hi & 0x44444444u);
        } else {
            const uint32_t r = (c & 1) ? ((p[2] >> 1) & 0x55555555u) | (p[3] & 0xAAAAAAAAu)
                                       : (p[2] & 0x55555555u) | ((p[3] << 1) & 0xAAAAAAAAu);
            return (c & 2) ? ((q >> 2) & 0x33333333u) | (r & 0xCCCCCCCCu) : (q & 0x33333333u) | ((r << 2) & 0xCCCCCCCCu);
        }
    }
    // the bytes 4 x of call m's replicas (bits m, m + 8, m + 16, m + 24) from
    // their nibbles x = nibbles(m & 3)
    __device__ __forceinline__ uint32_t bytes4(uint32_t x, int m) const {
        uint32_t e = m < 4 ? (x << 2) & 0x3C3C3C3Cu : (x >> 2) & 0x3C3C3C3Cu;
#pragma unroll
        for (int i = 4; i < P; ++i)   // bit m of the byte to bit i + 2
            e |= (m <= i + 2 ? p[i] << (i + 2 - m) : p[i] >> (m - i - 2)) & (0x04040404u << (i > 4 ? 5 : 4));
        return e;
    }
};

// bytes of the threshold rows (D = 0..H) and, per row, of the planes of 2^P - x_f
__host__ __device__ constexpr size_t bit_rows_bytes(int32_t H) { return (size_t)(H + 1) * (kBitRow * 4 + 32); }
struct BitLayout {
    uint32_t spins, rows, red, total;   // (threshold rows at the first 256-byte boundary of the block)
};
__host__ __device__ __forceinline__ BitLayout bit_layout(int32_t n, int32_t H) {
    BitLayout l;
    l.spins = 256u + (uint32_t)bit_rows_bytes(H);
    l.rows = l.spins + (uint32_t)((n + 3) & ~3) * 4u;
    l.red = l.rows + 32u * 8u;
    l.total = l.red + 32u * 8u;
    return l;
}

__device__ __forceinline__ uint32_t sign_mask(uint32_t e) { return (uint32_t)((int32_t)e >> 31); }

// Four neighbours' bits [J_kj s_j = +1] (flip: [J_kj s_j = -1] where it is all
// ones); slots at or beyond the row's end (left of them in the group) give 0.
__device__ __forceinline__ void bit4(uint32_t (&x)[4], const uint4 &e, int32_t left, const uint32_t *sp, uint32_t flip) {
    x[0] = sp[e.x & 0xFFFFFFu] ^ sign_mask(e.x) ^ flip;
    x[1] = sp[e.y & 0xFFFFFFu] ^ sign_mask(e.y) ^ flip;
    x[2] = sp[e.z & 0xFFFFFFu] ^ sign_mask(e.z) ^ flip;
    x[3] = sp[e.w & 0xFFFFFFu] ^ sign_mask(e.w) ^ flip;
    if (left < 4) {
        if (left < 1) x[0] = 0u;
        if (left < 2) x[1] = 0u;
        if (left < 3) x[2] = 0u;
        x[3] = 0u;
    }
}

// Rows: WC = 4 or 8 the ELL width (P = 3); else it is read at run time, with two
// groups of four couplings a lane loaded ahead (WC = 0), or up to 24 slots of
// the row, 128 registers a thread, where a group has its SM to itself (kDeep).
constexpr int kDeep = 1;
template <int QL, int WC>
constexpr int kAhead = WC == 4 ? 1 : WC == 8 ? (QL == 1 ? 2 : 1) : WC == 0 ? 2 : QL == 1 ? 6 : QL == 2 ? 4 : 3;

// loads the lane's groups sub, sub + QL, ... of position i (beyond the row: any
// group of it, not used)
template <int QL, int WC>
__device__ __forceinline__ void bit_load(uint4 (&e)[kAhead<QL, WC>], const uint32_t *es, int32_t i, int32_t W, int sub) {
#pragma unroll
    for (int v = 0; v < kAhead<QL, WC>; ++v) {
        const int x = sub + v * QL;
        if (WC == 0) e[v] = ell4(es, i, W, (uint32_t)(v == 0 && QL == 1 ? 0 : min(x, (W >> 2) - 1)));
        else if (WC == kDeep ? 4 * x < W : (QL == 1 || 4 * x < WC)) e[v] = ell4(es, i, W, (uint32_t)x);
    }
}

// The bit sums of a position: the lane's groups of four couplings, the first
// given, the rest of a longer row loaded as the degree asks.
template <int P, int QL, int WC>
__device__ __forceinline__ void bit_sum(Planes<P> &x, const uint4 (&e)[kAhead<QL, WC>], const uint32_t *es, int32_t i,
                                        int32_t W, int32_t deg, int sub, const uint32_t *sp, uint32_t flip) {
    constexpr int NG = kAhead<QL, WC>;
#pragma unroll
    for (int j = 0; j < P; ++j) x.p[j] = 0u;
    auto pair = [&](const uint4 &g, const uint4 &h, int32_t left) {   // two groups, the first not empty
        uint32_t a[4], b[4];
        bit4(a, g, left, sp, flip);
        if (left > 4 * QL) {
            bit4(b, h, left - 4 * QL, sp, flip);
            x.add8(a, b);
        } else {
            x.add4(a[0], a[1], a[2], a[3]);
        }
    };
#pragma unroll
    for (int v = 0; v < NG; v += 2) {
        const int32_t left = deg - 4 * (sub + v * QL);
        if ((QL == 1 && v == 0) || left > 0) {
            if (v + 1 < NG) {
                pair(e[v], e[v + 1 < NG ? v + 1 : v], left);
            } else {
                uint32_t a[4];
                bit4(a, e[v], left, sp, flip);
                x.add4(a[0], a[1], a[2], a[3]);
            }
        }
    }
    if constexpr (WC <= kDeep) {
        for (int32_t v = sub + NG * QL; 4 * v < deg; v += 2 * QL) {
            const int32_t left = deg - 4 * v;
            const uint4 g = ell4(es, i, W, v);
            if (left > 4 * QL) {
                pair(g, ell4(es, i, W, v + QL), left);
            } else {
                uint32_t a[4];
                bit4(a, g, left, sp, flip);
                x.add4(a[0], a[1], a[2], a[3]);
            }
        }
    }
    if constexpr (QL > 1) {
        constexpr int NVW = 32 / QL;
#pragma unroll
        for (int o = NVW; o < 32; o <<= 1) x.merge(o);
    }
}

// The sweeps of one CTA's group (group g of the instance, 4 nc replicas),
// shared by the single-instance and the batched kernels.
template <int RULE, int P, int QL, int WC, class KeyT>
__device__ __forceinline__ void
bits_body(const SweepDesc &d, const KeyT &key, int32_t t, int32_t slot, const int8_t *__restrict__ src,
          int8_t *__restrict__ dst, int64_t *__restrict__ E_dst, int nc, int32_t g) {
    extern __shared__ __align__(16) uint8_t smem[];
    const DevCtl *ctl = d.ctl;
    if (ctl->done) return;
    const int32_t n = d.n, H = d.H, R = d.R, S = d.S, W = WC > kDeep ? WC : d.W;
    const BitLayout lay = bit_layout(n, H);
    const uint32_t smem0 = (uint32_t)__cvta_generic_to_shared(smem);
    const uint32_t rows0 = (smem0 + 255u) & ~255u;
    uint32_t *tab_s = reinterpret_cast<uint32_t *>(smem + (rows0 - smem0));
    uint32_t *mark_s = tab_s + (H + 1) * kBitRow;
    const uint32_t marks0 = rows0 + (uint32_t)(H + 1) * (kBitRow * 4);
    // thresholds that fall with the field: inverted spins
    const uint32_t inv = RULE == 0 && d.tab[0] > d.tab[2 * H] ? 0xFFFFFFFFu : 0u;
    // (on its way while the spins are read; used below)
    const uint64_t first = (int)threadIdx.x < 2 * H + 1 ? d.tab[threadIdx.x] : 0ull;

    const int li = threadIdx.x, tpg = blockDim.x;
    const int32_t r0 = g * 4 * nc;
    const int32_t nrep = min(4 * nc, R - r0);          // replicas of the group
    const int32_t ncg = (nrep + 3) >> 2;               // its Philox calls
    uint32_t *sp = reinterpret_cast<uint32_t *>(smem + lay.spins);
    const int8_t **rows_s = reinterpret_cast<const int8_t **>(smem + lay.rows);
    unsigned long long *red = reinterpret_cast<unsigned long long *>(smem + lay.red);
    // slot r reads the NCM output if the cluster move rewrote it, else its
    // resampling parent (the replica copy of the population step)
    for (int32_t q = li; q < 32; q += tpg) {
        const int8_t *row = nullptr;
        if (q < nrep) {
            const int32_t m = d.ncm_idx[r0 + q];
            row = m >= 0 ? d.ncm_buf + (size_t)m * n : src + (size_t)d.parent[r0 + q] * n;
        }
        rows_s[q] = row;
        red[q] = 0ull;
    }
    __syncthreads();
    {
        for (int32_t k0 = li; k0 < n; k0 += 4 * tpg) {   // four vertices of a lane at a time
            uint32_t w[4] = {0u, 0u, 0u, 0u};
            for (int32_t q = 0; q < nrep; ++q) {
                const int8_t *row = rows_s[q];
                const uint32_t bit = 1u << ((q >> 2) + 8 * (q & 3));
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (k0 + j * tpg < n && row[k0 + j * tpg] > 0) w[j] |= bit;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (k0 + j * tpg < n) sp[k0 + j * tpg] = w[j] ^ inv;
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
    const bool up = RULE == 0 && inv == 0u;
    for (int i = threadIdx.x; i < (H + 1) * (H + 1); i += blockDim.x) {
        const int32_t D = i / (H + 1), x = i % (H + 1);
        if (x > D) continue;
        const uint64_t T = d.tab[up ? 2 * x - D + H : D - 2 * x + H];
        tab_s[D * kBitRow + x] = T > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)T;
    }
    for (int32_t D = threadIdx.x; D <= H; D += blockDim.x) {
        const int32_t xf = min(max((below + D - H + 1) >> 1, 0), D + 1);
        // word 0: carry in, words 1..6: the bits of what is added to x
        const uint32_t c = xf == 0 ? 63u : (uint32_t)((1 << P) - xf);
        mark_s[D * 8] = xf == 0 ? 0xFFFFFFFFu : 0u;
        for (int i = 0; i < 7; ++i) mark_s[D * 8 + 1 + i] = 0u - ((c >> i) & 1u);
    }
    __syncthreads();

    {
        constexpr int NVW = 32 / QL;                       // vertices of a warp's pass
        const int lane = threadIdx.x & 31;
        const int sub = QL == 1 ? 0 : lane / NVW;
        const int vl = QL == 1 ? li : (li >> 5) * NVW + lane % NVW, vpi = tpg / QL;
        const size_t ell_stride = (size_t)(((n + 31) >> 5) << 5) * W;
        const uint32_t ctr = (kTagFlip << 24) | (uint32_t)(nc * g + d.gbase);
        uint32_t live = 0u;   // the bits of the group's replicas
        for (int32_t q = 0; q < nrep; ++q) live |= 1u << ((q >> 2) + 8 * (q & 3));
        uint32_t nflip = 0;
        for (int32_t sw = 0; sw < S; ++sw) {
            const size_t sb = (size_t)slot * S + sw;
            const int32_t *lp = d.slvl + sb * (size_t)(n + 1);
            const uint32_t *es = d.sell + sb * ell_stride;
            const int2 *pos = d.spos + sb * (size_t)n;
            const int32_t L = d.snlev[sb];
            // the record and the first couplings of a pass are loaded one pass
            // ahead (kDeep: the couplings once this pass's are summed, beside
            // the draws and decisions), for a level's first pass before the
            // previous level's barrier (they do not depend on spins)
            int32_t end = 0, ip = min(vl, n - 1);
            int2 pr = pos[ip];
            uint4 e[kAhead<QL, WC>];
#pragma unroll
            for (int v = 0; v < kAhead<QL, WC>; ++v) e[v] = make_uint4(0u, 0u, 0u, 0u);
            bit_load<QL, WC>(e, es, ip, W, sub);
            for (int32_t lev = 0; lev < L; ++lev) {
                const int32_t beg = end;
                end = lp[lev + 1];
                // (the lanes of a warp go through the passes together: shuffles)
                for (int32_t base = beg; base < end; base += vpi) {
                    const int32_t i = base + vl;
                    const bool act = i < end;
                    const int32_t inext = min(base + vpi < end ? i + vpi : end + vl, n - 1);
                    const int2 prn = pos[inext];
                    uint4 en[kAhead<QL, WC>];
                    if constexpr (WC != kDeep) bit_load<QL, WC>(en, es, inext, W, sub);
                    const uint32_t a0 = (uint32_t)pr.x;
                    const int32_t k = (int32_t)(a0 & 0xFFFFFFu);
                    const bool run = QL > 1 || act;   // (QL > 1: all lanes, for the shuffles)
                    uint32_t old = 0u;
                    Planes<P> x;
                    if (run) {
                        old = sp[k];
                        bit_sum<P, QL, WC>(x, e, es, ip, W, (int32_t)(a0 >> 24), sub, sp, RULE == 0 ? 0u : old);
                    }
                    if constexpr (WC == kDeep) bit_load<QL, WC>(e, es, inext, W, sub);
                    if (run) {
                        const uint32_t D = (uint32_t)pr.y >> 24;
                        const uint32_t row = rows0 + (D << 8);
                        // replicas beyond the first threshold of 2^32
                        const uint4 m0 = bl_lds4(marks0 + (D << 5));
                        uint32_t force = maj(x.p[0], m0.y, m0.x);
                        force = maj(x.p[1], m0.z, force);
                        force = maj(x.p[2], m0.w, force);
                        if constexpr (P > 3) {
                            const uint4 m1 = bl_lds4(marks0 + (D << 5) + 16u);
                            const uint32_t mk[3] = {m1.x, m1.y, m1.z};
#pragma unroll
                            for (int j = 3; j < P; ++j) force = maj(x.p[j], mk[j - 3], force);
                        }
                        if constexpr (QL > 1) {
#pragma unroll
                            for (int j = 0; j < P; ++j) x.p[j] >>= sub;
                        }
                        float n0 = 8388608.0f, n1 = 8388608.0f;
                        const BitDraw draw((uint32_t)k, (uint32_t)sw, (uint32_t)t, key);
                        uint32_t x4[4];
#pragma unroll
                        for (int m = 0; m < 4; m += QL) x4[m] = x.nibbles(m);
#pragma unroll
                        for (int m = 0; m < 8; m += QL) {
                            // (lanes of a vertex beyond the last call: bits of no replica)
                            if (m == 0 || m < ncg) {
                                const u32x4 u = draw(ctr + (uint32_t)(m + sub), key);
                                const uint32_t x4b = x.bytes4(x4[m & 3], m);
                                const float bit = (float)(1 << m);
                                bl_add_if_below(n0, u.x, bl_lds(__byte_perm(x4b, row, 0x7650u)), bit);
                                bl_add_if_below(n0, u.y, bl_lds(__byte_perm(x4b, row, 0x7651u)), 256.0f * bit);
                                bl_add_if_below(n1, u.z, bl_lds(__byte_perm(x4b, row, 0x7652u)), bit);
                                bl_add_if_below(n1, u.w, bl_lds(__byte_perm(x4b, row, 0x7653u)), 256.0f * bit);
                            }
                        }
                        uint32_t nw = __byte_perm(__float_as_uint(n0), __float_as_uint(n1), 0x5410u);
                        if constexpr (QL > 1) {
                            nw <<= sub;
#pragma unroll
                            for (int o = NVW; o < 32; o <<= 1) nw |= __shfl_xor_sync(0xffffffffu, nw, o);
                        }
                        nw |= force;
                        const uint32_t flips = (RULE == 0 ? nw ^ old ^ inv : nw) & live;
                        if (act && sub == 0 && flips != 0u) {
                            sp[k] = old ^ flips;
                            nflip += __popc(flips);
                        }
                    }
                    ip = inext;
                    pr = prn;
                    if constexpr (WC != kDeep) {
#pragma unroll
                        for (int v = 0; v < kAhead<QL, WC>; ++v) e[v] = en[v];
                    }
                }
                __syncthreads();
            }
        }
        // spins that changed at a visit, summed per warp into the controller
        unsigned long long v = nflip;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0 && v != 0ull)
            atomicAdd(reinterpret_cast<unsigned long long *>(&const_cast<DevCtl *>(ctl)->sweep_flips), v);

        // energy from the definition, E = -1/2 sum_k s_k h_k = sum_k (x_k - D_k / 2)
        // with x the unsatisfied weight, over the last sweep's ELL rows
        const size_t sb = (size_t)slot * S + (S - 1);   // S >= 1
        const uint32_t *es = d.sell + sb * ell_stride;
        const int2 *pos = d.spos + sb * (size_t)n;
        // (a warp's lanes run it together for the reduction; 1024 x 63 < 2^16)
        for (int32_t w0 = li - lane; w0 < n; w0 += 1024 * tpg) {
            const int32_t i0 = w0 + lane;
            uint32_t acc[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) acc[q] = 0u;
            uint32_t dsum = 0u;
            const int64_t lim = min((int64_t)n, (int64_t)i0 + (int64_t)1024 * tpg);
            for (int64_t ii = i0; ii < lim; ii += tpg) {
                const int32_t i = (int32_t)ii;
                const int2 p0 = pos[i];
                const int32_t deg = (int32_t)((uint32_t)p0.x >> 24);
                dsum += (uint32_t)p0.y >> 24;
                Planes<P> x;
                uint4 e[kAhead<1, WC>];
#pragma unroll
                for (int v = 0; v < kAhead<1, WC>; ++v) e[v] = make_uint4(0u, 0u, 0u, 0u);
                bit_load<1, WC>(e, es, i, W, 0);
                bit_sum<P, 1, WC>(x, e, es, i, W, deg, 0, sp, sp[p0.x & 0xFFFFFF]);
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    const uint32_t y = x.bytes4(x.nibbles(m & 3), m);
                    acc[2 * m] += (y >> 2) & 0x003F003Fu;
                    acc[2 * m + 1] += (y >> 10) & 0x003F003Fu;
                }
            }
#pragma unroll
            for (int q = 0; q < 32; ++q) {   // replica q: call q / 4, byte q % 4
                const int b = q & 3;
                int32_t s = (int32_t)((acc[2 * (q >> 2) + (b & 1)] >> (16 * (b >> 1))) & 0xFFFFu) * 2 - (int32_t)dsum;
                if (q < nrep) {   // (the same for the whole group)
                    s = __reduce_add_sync(0xffffffffu, s);
                    if (lane == 0) atomicAdd(&red[q], (unsigned long long)(long long)s);
                }
            }
        }
        // write-back, four vertices of a lane at a time
        for (int32_t k0 = li; k0 < n; k0 += 4 * tpg) {
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = k0 + j * tpg < n ? sp[k0 + j * tpg] ^ inv : 0u;
            int8_t *row = dst + (size_t)r0 * n + k0;
            for (int32_t q = 0; q < nrep; ++q, row += n) {
                const int sh = (q >> 2) + 8 * (q & 3);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (k0 + j * tpg < n) row[j * tpg] = (w[j] >> sh) & 1u ? 1 : -1;
            }
        }
    }
    __syncthreads();
    for (int32_t q = li; q < nrep; q += tpg) E_dst[r0 + q] = (long long)red[q] / 2;
}

template <int RULE, int P, int QL, int WC>
__global__ void __launch_bounds__(WC == kDeep ? 512 : 1024) k_sweep_ising_bits(SweepDesc d, int nc) {
    bits_body<RULE, P, QL, WC>(d, BitKeys{d.K}, d.t, d.slot, d.src, d.dst, d.E_dst, nc, blockIdx.x);
}

// Many instances in one launch: CTA b works on member items[b].x, its group
// items[b].y; the step index comes from the member's controller.
template <int RULE, int P, int QL>
__global__ void __launch_bounds__(1024)
k_sweep_ising_bits_batched(const SweepDesc *__restrict__ descs, const int2 *__restrict__ items, int nc) {
    const int2 it = items[blockIdx.x];
    const SweepDesc &d = descs[it.x];
    const int32_t t = d.ctl->t;
    if (t >= d.t_end) return;
    bits_body<RULE, P, QL, 0>(d, BitKeysSeed{d.K.k0[0], d.K.k1[0]}, t, t % d.slots, d.sp[t & 1], d.sp[(t + 1) & 1],
                              d.en[(t + 1) & 1], nc, it.y);
}

}  // namespace

bool bits_apply(int32_t n, const int32_t *rp, const uint32_t *adj, int32_t H, int32_t ell_w) {
    if (ell_w == 0 || H > kBitLaneMaxH) return false;
    for (int32_t e = 0; e < rp[n]; ++e) {
        const int32_t J = (int32_t)adj[e] >> 24;
        if (J < -1 || J > 1) return false;
    }
    return true;
}

int sweep_bits_planes(int32_t H) { return H <= 7 ? 3 : H <= 31 ? 5 : 6; }

size_t sweep_bits_smem_bytes(int32_t n, int32_t H) { return bit_layout(n, H).total; }

cudaError_t launch_sweep_ising_bits(int rule, int32_t n, int32_t H, const pamc_params &p, int32_t t, int32_t slot,
                                    SchedView sv, const uint64_t *tab, const int8_t *src, const int32_t *parent,
                                    const int8_t *ncm_buf, const int32_t *ncm_idx, int8_t *dst, int64_t *E_dst,
                                    const DevCtl *ctl, SweepCfg cfg, cudaStream_t st, int32_t rbase) {
    if (sv.ell == nullptr || p.sweeps < 1 || H > kBitLaneMaxH || cfg.bits < 1 || cfg.bits > 8) return cudaErrorInvalidValue;
    const int nc = cfg.bits, groups = (p.R + 4 * nc - 1) / (4 * nc);
    const int planes = sweep_bits_planes(H);
    int dev = 0, sms = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    const bool deep = planes > 3 && cfg.warps_per_group <= 16 && groups <= sms;
    const int threads = 32 * cfg.warps_per_group;
    SweepDesc d;
    memset(&d, 0, sizeof(d));
    d.slvl = sv.lvl_ptr; d.snlev = sv.nlev; d.sell = sv.ell; d.spos = sv.pos;
    d.tab = tab; d.src = src; d.parent = parent; d.ncm_buf = ncm_buf; d.ncm_idx = ncm_idx;
    d.dst = dst; d.E_dst = E_dst; d.ctl = ctl; d.n = n; d.n_pad = (n + 3) & ~3; d.H = H; d.R = p.R;
    d.S = p.sweeps; d.t = t; d.slot = slot; d.W = sv.W; d.K = make_philox_keys(p.seed);
    d.gbase = rbase / 4;
    const size_t smem = sweep_bits_smem_bytes(n, H);
#define PAMC_BITS(RU, PL, Q, WV)                                                              \
    do {                                                                                      \
        err = allow_dynamic_smem(k_sweep_ising_bits<RU, PL, Q, WV>, smem);                    \
        if (err != cudaSuccess) return err;                                                   \
        k_sweep_ising_bits<RU, PL, Q, WV><<<groups, threads, smem, st>>>(d, nc);              \
    } while (0)
#define PAMC_BITS_Q(RU, PL, WV)                                                               \
    do {                                                                                      \
        if (cfg.lanes_per_vertex == 1) PAMC_BITS(RU, PL, 1, WV);                              \
        else if (cfg.lanes_per_vertex == 2) PAMC_BITS(RU, PL, 2, WV);                         \
        else PAMC_BITS(RU, PL, 4, WV);                                                        \
    } while (0)
#define PAMC_BITS_P(RU)                                                                       \
    do {                                                                                      \
        if (planes == 3 && sv.W == 4) PAMC_BITS_Q(RU, 3, 4);                                  \
        else if (planes == 3) PAMC_BITS_Q(RU, 3, 8);                                          \
        else if (planes == 5 && deep) PAMC_BITS_Q(RU, 5, kDeep);                              \
        else if (planes == 5) PAMC_BITS_Q(RU, 5, 0);                                          \
        else if (deep) PAMC_BITS_Q(RU, 6, kDeep);                                             \
        else PAMC_BITS_Q(RU, 6, 0);                                                           \
    } while (0)
    if (rule == 0) PAMC_BITS_P(0);
    else PAMC_BITS_P(1);
#undef PAMC_BITS_P
#undef PAMC_BITS_Q
#undef PAMC_BITS
    return cudaGetLastError();
}

cudaError_t launch_sweep_ising_bits_batched(int rule, int planes, int lanes, int warps, int nc, size_t smem,
                                            const SweepDesc *descs, const int2 *items, int32_t nitems, cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    if (nc < 1 || nc > 8 || warps < 1 || warps > 16) return cudaErrorInvalidValue;
    cudaError_t err = cudaSuccess;
#define PAMC_BITB(RU, PL, Q)                                                                  \
    do {                                                                                      \
        err = allow_dynamic_smem(k_sweep_ising_bits_batched<RU, PL, Q>, smem);                \
        if (err != cudaSuccess) return err;                                                   \
        k_sweep_ising_bits_batched<RU, PL, Q><<<nitems, warps * 32, smem, st>>>(descs, items, nc); \
    } while (0)
#define PAMC_BITB_P(RU, Q)                                                                    \
    do {                                                                                      \
        if (planes == 3) PAMC_BITB(RU, 3, Q);                                                 \
        else if (planes == 5) PAMC_BITB(RU, 5, Q);                                            \
        else PAMC_BITB(RU, 6, Q);                                                             \
    } while (0)
    if (lanes == 1) {
        if (rule == 0) PAMC_BITB_P(0, 1);
        else PAMC_BITB_P(1, 1);
    } else if (lanes == 4) {
        if (rule == 0) PAMC_BITB_P(0, 4);
        else PAMC_BITB_P(1, 4);
    } else {
        return cudaErrorInvalidValue;
    }
#undef PAMC_BITB_P
#undef PAMC_BITB
    return cudaGetLastError();
}

}  // namespace pamc
