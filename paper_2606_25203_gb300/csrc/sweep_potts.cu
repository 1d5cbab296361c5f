// sweep_potts.cu -- S sweeps of the three-state Potts population (Max-3-Cut)
// with the cascaded sampler of Suppl. S3 (Eq. 6-8): with
// syn_c(k) = sum_j J_kj [sigma_j = c], label 0 iff u0 < T1(syn1-syn0, syn2-syn0),
// else label 1 iff u1 < T2(syn2-syn1), else label 2.
//
// Layout.  Four replicas form a group.  For every vertex the group keeps two
// one-hot words in shared memory: byte q of w0 (w1) is 1 iff replica q has
// label 0 (1).  A neighbour adds J to the byte lanes of both accumulators with
// one 64-bit shared load and two multiply-adds, on a bias of 128 per byte
// (bytes never carry since sum_j |J_kj| <= 127); syn2 = sum_j J_kj - syn0 -
// syn1.  Replica r's draws are words 2(r mod 2), 2(r mod 2)+1 of
// Philox(k, sweep, t, FLIP<<24 | r/2): two calls per group.  Levels of the
// (t, sweep) schedule give the exact sequential order.
//
// ELL rows (potts_ell_body): LPV = 2 lanes share a position (one where the
// level is wide and the SM crowded).  Lane s runs the Philox call of replicas 2s
// and 2s + 1, sums every second group of four couplings (one shuffle per
// accumulator adds the two partial sums) and decides and stores its own two
// replicas' halves of the one-hot words.  The record and the lane's first two
// groups are loaded one pass ahead.  The table positions (syn1 - syn0, syn2 -
// syn0) and syn2 - syn1 are linear in the two sum bytes: two multiply-adds each,
// the byte biases in the constant.  Bound: instruction issue and, at few groups
// an SM, the level's chain.  On N=2,000 degree 12, R=2,048, 10 sweeps a launch went
// from 672 to 473 us, on N=12,000 degree 5 from 2,934 to 1,379.
//
// CSR rows (no ELL, or no sweeps): one lane a position, nothing ahead.
#include <cstring>

#include "pamc_device.cuh"
#include "pamc_internal.h"

namespace pamc {

namespace {

__device__ __forceinline__ void potts_barrier(int id, int nthreads, int groups) {
    if (groups == 1) {
        __syncthreads();
    } else {
        asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
    }
}

// one-hot words of four byte labels (0..2)
__device__ __forceinline__ uint2 onehot(uint32_t labels) {
    return make_uint2(__vcmpeq4(labels, 0u) & 0x01010101u, __vcmpeq4(labels, 0x01010101u) & 0x01010101u);
}

// four couplings of a row on the neighbours' one-hot words
__device__ __forceinline__ void potts_add4(uint32_t &A0, uint32_t &A1, const uint4 &e, const uint2 *oh) {
    const uint32_t w[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint2 o = oh[w[q] & 0xFFFFFFu];
        const uint32_t J = (uint32_t)((int32_t)w[q] >> 24);
        A0 += o.x * J;
        A1 += o.y * J;
    }
}

// The sweeps of one CTA's replica groups (groups bid*gpc .. bid*gpc+gpc-1 of
// the instance), shared by the single-instance and the batched kernels.
__device__ __forceinline__ void
potts_body(int32_t n, int32_t n_pad, const int32_t *__restrict__ rp, const uint32_t *__restrict__ adj,
           int32_t H, int32_t R, int32_t S, uint32_t key0, uint32_t key1, int32_t t, int32_t slot,
           const int32_t *__restrict__ sorder, const int32_t *__restrict__ slvl,
           const int32_t *__restrict__ snlev, const uint64_t *__restrict__ tab,
           const int8_t *__restrict__ src, const int32_t *__restrict__ parent, int8_t *__restrict__ dst,
           int64_t *__restrict__ E_dst, const DevCtl *__restrict__ ctl, int64_t Wsum, int gpc, int tpg,
           int32_t bid, int32_t gbase) {
    extern __shared__ __align__(16) uint8_t smem[];
    if (ctl->done) return;
    const int32_t W1 = 4 * H + 1;
    const uint64_t *T1 = tab;                            // [(a + 2H) * W1 + (b + 2H)], read through L1
    uint64_t *T2s = reinterpret_cast<uint64_t *>(smem);  // [c + 2H]
    uint2 *oh_all = reinterpret_cast<uint2 *>(smem + (((size_t)W1 * 8 + 15) & ~(size_t)15));
    unsigned long long *red = reinterpret_cast<unsigned long long *>(oh_all + (size_t)gpc * n_pad);
    for (int i = threadIdx.x; i < W1; i += blockDim.x) T2s[i] = tab[(size_t)W1 * W1 + i];
    for (int i = threadIdx.x; i < gpc * 4; i += blockDim.x) red[i] = 0ull;

    const int gl = threadIdx.x / tpg, li = threadIdx.x % tpg;
    const int32_t g = bid * gpc + gl;
    const int32_t gk = g + gbase;   // the group's index in the whole population keys its draws
    const int32_t r0 = g * 4;
    const bool active = r0 < R;
    uint2 *oh = oh_all + (size_t)gl * n_pad;

    if (active) {
        // NCM is not defined for Potts: slot r reads its resampling parent
        const int8_t *rows[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) rows[q] = (r0 + q < R) ? src + (size_t)parent[r0 + q] * n : nullptr;
        for (int32_t k = li; k < n; k += tpg) {
            uint32_t lab = 0x03030303u;   // padding replicas: no label
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (rows[q] != nullptr) lab = (lab & ~(0xFFu << (8 * q))) | ((uint32_t)(uint8_t)rows[q][k] << (8 * q));
            oh[k] = onehot(lab);
        }
    }
    __syncthreads();

    if (active) {
        for (int32_t sw = 0; sw < S; ++sw) {
            const size_t sb = (size_t)slot * S + sw;
            const int32_t *ord = sorder + sb * (size_t)n;
            const int32_t *lp = slvl + sb * (size_t)(n + 1);
            const int32_t L = snlev[sb];
            for (int32_t lev = 0; lev < L; ++lev) {
                const int32_t beg = lp[lev], end = lp[lev + 1];
                for (int32_t i = beg + li; i < end; i += tpg) {
                    uint32_t A0 = 0x80808080u, A1 = 0x80808080u;
                    const int32_t k = ord[i] & 0xFFFFFF;
                    int32_t jsum = 0;
                    for (int32_t e = rp[k]; e < rp[k + 1]; ++e) {
                        const uint32_t a = adj[e];
                        const int32_t J = (int32_t)a >> 24;
                        const uint2 o = oh[a & 0xFFFFFFu];
                        A0 += o.x * (uint32_t)J;
                        A1 += o.y * (uint32_t)J;
                        jsum += J;
                    }
                    const u32x4 ua = philox((uint32_t)k, (uint32_t)sw, (uint32_t)t,
                                            (kTagFlip << 24) | (uint32_t)(2 * gk), key0, key1);
                    const u32x4 ub = philox((uint32_t)k, (uint32_t)sw, (uint32_t)t,
                                            (kTagFlip << 24) | (uint32_t)(2 * gk + 1), key0, key1);
                    const uint32_t u0[4] = {ua.x, ua.z, ub.x, ub.z};
                    const uint32_t u1[4] = {ua.y, ua.w, ub.y, ub.w};
                    uint32_t lab = 0x03030303u;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (r0 + q >= R) break;
                        const int32_t s0 = (int32_t)((A0 >> (8 * q)) & 0xFFu) - 128;
                        const int32_t s1 = (int32_t)((A1 >> (8 * q)) & 0xFFu) - 128;
                        const int32_t s2 = jsum - s0 - s1;
                        const uint64_t t1 = __ldg(&T1[(size_t)(s1 - s0 + 2 * H) * W1 + (s2 - s0 + 2 * H)]);
                        uint32_t c;
                        if ((uint64_t)u0[q] < t1) c = 0;
                        else if ((uint64_t)u1[q] < T2s[s2 - s1 + 2 * H]) c = 1;
                        else c = 2;
                        lab = (lab & ~(0xFFu << (8 * q))) | (c << (8 * q));
                    }
                    const uint2 nw = onehot(lab), old = oh[k];
                    if (nw.x != old.x || nw.y != old.y) oh[k] = nw;
                }
                potts_barrier(1 + gl, tpg, gpc);
            }
        }

        // energy from the definition, E = -sum_k syn_{sigma_k}(k) - W, and the write-back
        long long acc[4] = {0, 0, 0, 0};
        for (int32_t k = li; k < n; k += tpg) {
            uint32_t A0 = 0x80808080u, A1 = 0x80808080u;
            int32_t jsum = 0;
            for (int32_t e = rp[k]; e < rp[k + 1]; ++e) {
                const uint32_t a = adj[e];
                const int32_t J = (int32_t)a >> 24;
                const uint2 o = oh[a & 0xFFFFFFu];
                A0 += o.x * (uint32_t)J;
                A1 += o.y * (uint32_t)J;
                jsum += J;
            }
            const uint2 ok = oh[k];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int32_t s0 = (int32_t)((A0 >> (8 * q)) & 0xFFu) - 128;
                const int32_t s1 = (int32_t)((A1 >> (8 * q)) & 0xFFu) - 128;
                const bool l0 = (ok.x >> (8 * q)) & 1u, l1 = (ok.y >> (8 * q)) & 1u;
                const int32_t own = l0 ? s0 : (l1 ? s1 : jsum - s0 - s1);
                acc[q] += own;
                if (r0 + q < R) dst[(size_t)(r0 + q) * n + k] = (int8_t)(l0 ? 0 : (l1 ? 1 : 2));
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            long long v = acc[q];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if ((threadIdx.x & 31) == 0) atomicAdd(&red[gl * 4 + q], (unsigned long long)v);
        }
    }
    __syncthreads();
    if (active && li < 4 && r0 + li < R) E_dst[r0 + li] = -(long long)red[gl * 4 + li] - Wsum;
}

// Draws with the round keys of the seed in kernel parameter space, or advanced
// from the seed (batched launches: the key differs per member).
struct PottsKeys {
    const PhiloxKeys &K;
    __device__ __forceinline__ u32x4 operator()(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3) const {
        return philox_rk(c0, c1, c2, c3, K);
    }
};
struct PottsKeysSeed {
    uint32_t k0, k1;
    __device__ __forceinline__ u32x4 operator()(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3) const {
        return philox(c0, c1, c2, c3, k0, k1);
    }
};

template <int LPV, class KeyT>
__device__ __forceinline__ void
potts_ell_body(const SweepDesc &d, const KeyT &draw, int32_t t, int32_t slot, const int8_t *__restrict__ src,
               int8_t *__restrict__ dst, int64_t *__restrict__ E_dst, int gpc, int tpg, int32_t bid) {
    extern __shared__ __align__(16) uint8_t smem[];
    if (d.ctl->done) return;
    const int32_t n = d.n, n_pad = d.n_pad, H = d.H, R = d.R, S = d.S, W = d.W;
    const int32_t W1 = 4 * H + 1;
    const uint64_t *T1 = d.tab;                          // [(a + 2H) * W1 + (b + 2H)], read through L1
    uint64_t *T2s = reinterpret_cast<uint64_t *>(smem);  // [c + 2H]
    uint2 *oh_all = reinterpret_cast<uint2 *>(smem + (((size_t)W1 * 8 + 15) & ~(size_t)15));
    unsigned long long *red = reinterpret_cast<unsigned long long *>(oh_all + (size_t)gpc * n_pad);
    for (int i = threadIdx.x; i < W1; i += blockDim.x) T2s[i] = d.tab[(size_t)W1 * W1 + i];
    for (int i = threadIdx.x; i < gpc * 4; i += blockDim.x) red[i] = 0ull;

    const int gl = threadIdx.x / tpg, li = threadIdx.x % tpg;
    const int32_t g = bid * gpc + gl;
    const int32_t r0 = g * 4;
    const bool active = r0 < R;
    uint2 *oh = oh_all + (size_t)gl * n_pad;
    if (active) {   // NCM is not defined for Potts: slot r reads its resampling parent
        const int8_t *rows[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) rows[q] = (r0 + q < R) ? src + (size_t)d.parent[r0 + q] * n : nullptr;
        for (int32_t k = li; k < n; k += tpg) {
            uint32_t lab = 0x03030303u;   // padding replicas start without a label
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (rows[q] != nullptr) lab = (lab & ~(0xFFu << (8 * q))) | ((uint32_t)(uint8_t)rows[q][k] << (8 * q));
            oh[k] = onehot(lab);
        }
    }
    __syncthreads();
    if (active) {
        constexpr int NR = 4 / LPV;    // replicas a lane decides
        constexpr int NG = 4 / LPV;    // groups of four couplings a lane loads ahead
        const int sl = LPV == 1 ? 0 : li & 1, vi = LPV == 1 ? li : li >> 1, vpi = tpg / LPV;
        const uint32_t ctr = (kTagFlip << 24) | (uint32_t)(2 * (g + d.gbase) + sl);
        const size_t ell_stride = (size_t)(((n + 31) >> 5) << 5) * W;
        // table positions from the sum bytes b = syn + 128 of labels 0 and 1:
        // (syn1 - syn0 + 2H) W1 + syn2 - syn0 + 2H and syn2 - syn1 + 2H
        const int32_t c1 = 384 + 2 * H * (W1 + 1), m1 = W1 - 1, m0 = -(W1 + 2), c2 = 384 + 2 * H;
        for (int32_t sw = 0; sw < S; ++sw) {
            const size_t sb = (size_t)slot * S + sw;
            const int32_t *lp = d.slvl + sb * (size_t)(n + 1);
            const uint32_t *es = d.sell + sb * ell_stride;
            const int2 *pos = d.spos + sb * (size_t)n;
            const int32_t L = d.snlev[sb];
            int32_t end = 0, ip = min(vi, n - 1);
            int2 pr = pos[ip];
            uint4 ev[NG];
#pragma unroll
            for (int q = 0; q < NG; ++q)
                ev[q] = 4 * (LPV * q + sl) < W ? ell4(es, ip, W, LPV * q + sl) : make_uint4(0u, 0u, 0u, 0u);
            for (int32_t lev = 0; lev < L; ++lev) {
                const int32_t beg = end;
                end = lp[lev + 1];
                // every lane of a warp runs the same passes (the shuffles); lanes
                // beyond the level's end write nothing
                for (int32_t base = beg; base < end; base += vpi) {
                    const bool act = base + vi < end;
                    const int32_t inext = min(base + vpi < end ? base + vpi + vi : end + vi, n - 1);
                    const int2 prn = pos[inext];
                    uint4 evn[NG];
#pragma unroll
                    for (int q = 0; q < NG; ++q)
                        evn[q] = 4 * (LPV * q + sl) < W ? ell4(es, inext, W, LPV * q + sl) : make_uint4(0u, 0u, 0u, 0u);
                    if (LPV > 1 || act) {
                        const int32_t k = pr.x & 0xFFFFFF, deg = (int32_t)((uint32_t)pr.x >> 24);
                        uint32_t A0 = 0u, A1 = 0u;
#pragma unroll
                        for (int q = 0; q < NG; ++q)
                            if (q == 0 || deg > 4 * (LPV * q + sl)) potts_add4(A0, A1, ev[q], oh);
                        for (int32_t v = 4 + sl; 4 * v < deg; v += LPV) potts_add4(A0, A1, ell4(es, ip, W, v), oh);
                        if constexpr (LPV > 1) {
                            A0 += __shfl_xor_sync(0xffffffffu, A0, 1);
                            A1 += __shfl_xor_sync(0xffffffffu, A1, 1);
                        }
                        // (lanes beyond the level's end have read words that this level
                        // is changing: their sums may lie outside the tables)
                        if (act) {
                            A0 = (A0 + 0x80808080u) >> (16 * sl);
                            A1 = (A1 + 0x80808080u) >> (16 * sl);
                            const int32_t jsum = pos_jsum(pr.y);
                            uint64_t t1[NR], t2[NR];
#pragma unroll
                            for (int q = 0; q < NR; ++q) {
                                const int32_t b0 = (int32_t)((A0 >> (8 * q)) & 0xFFu), b1 = (int32_t)((A1 >> (8 * q)) & 0xFFu);
                                t1[q] = __ldg(&T1[(uint32_t)(jsum + c1 + b1 * m1 + b0 * m0)]);
                                t2[q] = T2s[jsum + c2 - b0 - 2 * b1];
                            }
                            uint32_t w0 = 0u, w1 = 0u;
#pragma unroll
                            for (int h = 0; h < NR / 2; ++h) {
                                const u32x4 u = draw((uint32_t)k, (uint32_t)sw, (uint32_t)t, ctr + (uint32_t)h);
                                const bool p0 = (uint64_t)u.x < t1[2 * h], p1 = (uint64_t)u.z < t1[2 * h + 1];
                                if (p0) w0 |= 1u << (16 * h);
                                else if ((uint64_t)u.y < t2[2 * h]) w1 |= 1u << (16 * h);
                                if (p1) w0 |= 0x100u << (16 * h);
                                else if ((uint64_t)u.w < t2[2 * h + 1]) w1 |= 0x100u << (16 * h);
                            }
                            if constexpr (LPV == 1) {
                                oh[k] = make_uint2(w0, w1);
                            } else {
                                uint16_t *half = reinterpret_cast<uint16_t *>(oh + k) + sl;
                                half[0] = (uint16_t)w0;
                                half[2] = (uint16_t)w1;
                            }
                        }
                    }
                    ip = inext;
                    pr = prn;
#pragma unroll
                    for (int q = 0; q < NG; ++q) ev[q] = evn[q];
                }
                potts_barrier(1 + gl, tpg, gpc);
            }
        }
        // energy from the definition, E = -sum_k syn_{sigma_k}(k) - W, by position
        // over the last sweep's rows, and the write-back
        const size_t sb = (size_t)slot * S + (S - 1);   // S >= 1
        const uint32_t *es = d.sell + sb * ell_stride;
        const int2 *pos = d.spos + sb * (size_t)n;
        int32_t acc[4] = {0, 0, 0, 0};   // (|syn| <= 127, n < 2^24)
        for (int32_t i = li; i < n; i += tpg) {
            const int2 pr = pos[i];
            const int32_t deg = (int32_t)((uint32_t)pr.x >> 24), jsum = pos_jsum(pr.y);
            uint32_t A0 = 0u, A1 = 0u;
            for (int32_t v = 0; 4 * v < deg; ++v) potts_add4(A0, A1, ell4(es, i, W, v), oh);
            A0 += 0x80808080u;
            A1 += 0x80808080u;
            const uint2 ok = oh[pr.x & 0xFFFFFF];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int32_t s0 = (int32_t)((A0 >> (8 * q)) & 0xFFu) - 128;
                const int32_t s1 = (int32_t)((A1 >> (8 * q)) & 0xFFu) - 128;
                acc[q] += (ok.x >> (8 * q)) & 1u ? s0 : (ok.y >> (8 * q)) & 1u ? s1 : jsum - s0 - s1;
            }
        }
        for (int32_t k = li; k < n; k += tpg) {
            const uint2 ok = oh[k];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (r0 + q < R)
                    dst[(size_t)(r0 + q) * n + k] = (ok.x >> (8 * q)) & 1u ? 0 : (ok.y >> (8 * q)) & 1u ? 1 : 2;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            long long v = acc[q];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if ((threadIdx.x & 31) == 0) atomicAdd(&red[gl * 4 + q], (unsigned long long)v);
        }
    }
    __syncthreads();
    if (active && li < 4 && r0 + li < R) E_dst[r0 + li] = -(long long)red[gl * 4 + li] - d.Wsum;
}

template <int LPV>
__global__ void __launch_bounds__(1024) k_sweep_potts_ell(SweepDesc d, int gpc, int tpg) {
    potts_ell_body<LPV>(d, PottsKeys{d.K}, d.t, d.slot, d.src, d.dst, d.E_dst, gpc, tpg, blockIdx.x);
}

__global__ void __launch_bounds__(1024)
k_sweep_potts(int32_t n, int32_t n_pad, const int32_t *__restrict__ rp, const uint32_t *__restrict__ adj,
              int32_t H, int32_t R, int32_t S, uint32_t key0, uint32_t key1, int32_t t, int32_t slot,
              const int32_t *__restrict__ sorder, const int32_t *__restrict__ slvl,
              const int32_t *__restrict__ snlev, const uint64_t *__restrict__ tab,
              const int8_t *__restrict__ src, const int32_t *__restrict__ parent, int8_t *__restrict__ dst,
              int64_t *__restrict__ E_dst, const DevCtl *__restrict__ ctl, int64_t Wsum, int gpc, int tpg,
              int32_t gbase) {
    potts_body(n, n_pad, rp, adj, H, R, S, key0, key1, t, slot, sorder, slvl, snlev, tab, src, parent, dst, E_dst, ctl,
               Wsum, gpc, tpg, blockIdx.x, gbase);
}

// Many Max-3-Cut instances in one launch: CTA b works on instance items[b].x,
// its local block items[b].y; the member's step index comes from its device
// controller (ctl->t), which picks the double-buffered labels and energies
// and the schedule slot; steps at or past t_end do nothing.  ELL members: lane
// pairs.
template <bool ELLP>
__global__ void __launch_bounds__(1024)
k_sweep_potts_batched(const SweepDesc *__restrict__ descs, const int2 *__restrict__ items, int gpc, int tpg) {
    const int2 it = items[blockIdx.x];
    const SweepDesc &d = descs[it.x];
    const DevCtl *ctl = d.ctl;
    const int32_t t = ctl->t;
    if (t >= d.t_end) return;
    if constexpr (ELLP)
        potts_ell_body<2>(d, PottsKeysSeed{d.K.k0[0], d.K.k1[0]}, t, t % d.slots, d.sp[t & 1], d.sp[(t + 1) & 1],
                          d.en[(t + 1) & 1], gpc, tpg, it.y);
    else
        potts_body(d.n, d.n_pad, d.rp, d.adj, d.H, d.R, d.S, d.K.k0[0], d.K.k1[0], t, t % d.slots, d.sorder, d.slvl,
                   d.snlev, d.tab, d.sp[t & 1], d.parent, d.sp[(t + 1) & 1], d.en[(t + 1) & 1], ctl, d.Wsum, gpc, tpg,
                   it.y, d.gbase);
}

}  // namespace

size_t sweep_potts_smem_bytes(int32_t n, int32_t H, SweepCfg cfg) {
    const int32_t n_pad = (n + 3) & ~3;
    return (((size_t)(4 * H + 1) * 8 + 15) & ~(size_t)15) + (size_t)cfg.groups_per_cta * n_pad * 8 +
           (size_t)cfg.groups_per_cta * 4 * 8;
}

cudaError_t launch_sweep_potts(int32_t n, const int32_t *rp, const uint32_t *adj, int32_t H, const pamc_params &p,
                               int32_t t, int32_t slot, SchedView sv, const uint64_t *tab, const int8_t *src,
                               const int32_t *parent, int8_t *dst, int64_t *E_dst, const DevCtl *ctl,
                               SweepCfg cfg, int64_t Wsum, cudaStream_t st, int32_t rbase) {
    const int32_t groups = (p.R + 3) / 4;
    const int gpc = cfg.groups_per_cta, tpg = cfg.warps_per_group * 32;
    const size_t smem = sweep_potts_smem_bytes(n, H, cfg);
    const int grid = (groups + gpc - 1) / gpc;
    cudaError_t err;
    if (sv.ell != nullptr && p.sweeps > 0) {
        SweepDesc d;
        memset(&d, 0, sizeof(d));
        d.slvl = sv.lvl_ptr; d.snlev = sv.nlev; d.sell = sv.ell; d.spos = sv.pos;
        d.tab = tab; d.src = src; d.parent = parent; d.dst = dst; d.E_dst = E_dst; d.ctl = ctl;
        d.n = n; d.n_pad = (n + 3) & ~3; d.H = H; d.R = p.R; d.S = p.sweeps; d.t = t; d.slot = slot; d.W = sv.W;
        d.K = make_philox_keys(p.seed); d.Wsum = Wsum; d.gbase = rbase / 4;
        err = cfg.lanes_per_vertex == 2 ? allow_dynamic_smem(k_sweep_potts_ell<2>, smem)
                                        : allow_dynamic_smem(k_sweep_potts_ell<1>, smem);
        if (err != cudaSuccess) return err;
        if (cfg.lanes_per_vertex == 2) k_sweep_potts_ell<2><<<grid, gpc * tpg, smem, st>>>(d, gpc, tpg);
        else k_sweep_potts_ell<1><<<grid, gpc * tpg, smem, st>>>(d, gpc, tpg);
        return cudaGetLastError();
    }
    err = allow_dynamic_smem(k_sweep_potts, smem);
    if (err != cudaSuccess) return err;
    k_sweep_potts<<<grid, gpc * tpg, smem, st>>>(n, (n + 3) & ~3, rp, adj, H, p.R, p.sweeps, (uint32_t)p.seed,
                                                 (uint32_t)(p.seed >> 32), t, slot, sv.order, sv.lvl_ptr, sv.nlev, tab, src,
                                                 parent, dst, E_dst, ctl, Wsum, gpc, tpg, rbase / 4);
    return cudaGetLastError();
}

}  // namespace pamc

namespace pamc {

cudaError_t launch_sweep_potts_batched(bool ell, const SweepDesc *descs, const int2 *items, int32_t nitems,
                                       int32_t n_max, SweepCfg cfg, cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    const int gpc = cfg.groups_per_cta, tpg = cfg.warps_per_group * 32;
    const size_t smem = sweep_potts_smem_bytes(n_max, 127, cfg);
    cudaError_t err;
    if (ell) {
        err = allow_dynamic_smem(k_sweep_potts_batched<true>, smem);
        if (err != cudaSuccess) return err;
        k_sweep_potts_batched<true><<<nitems, gpc * tpg, smem, st>>>(descs, items, gpc, tpg);
    } else {
        err = allow_dynamic_smem(k_sweep_potts_batched<false>, smem);
        if (err != cudaSuccess) return err;
        k_sweep_potts_batched<false><<<nitems, gpc * tpg, smem, st>>>(descs, items, gpc, tpg);
    }
    return cudaGetLastError();
}

}  // namespace pamc
