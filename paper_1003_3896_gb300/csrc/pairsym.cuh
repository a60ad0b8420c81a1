// pairsym.cuh -- the symmetric pair kernels' common frame (Newton's third law).
//
// Each unordered pair is evaluated once and its force added to both bodies.
// The pair term costs 3 differences, 3 FMAs for r^2 + eps^2, a reciprocal
// square root and its cube (2 multiplies); both bodies' sums take 3 FMAs each.
// So two interactions cost 14 FMA-pipe operations in the equal-mass float
// form, 7 per interaction, where the full N x N kernel of pair.cu needs 11.
//
// Work: SymRows' tiles (one unordered pair of i-blocks of ipb = TILE * I
// bodies each), cut into units of jt j bodies; the units of all clusters are
// split into equal contiguous runs, one per block (Decomp).
//
// A block of four warps holds one i-block at a time: warp w owns a row of
// 32 kw consecutive bodies, lane l bodies l, l + 32, ... of it, whose sums stay
// in registers for the whole run.  The j bodies come in chunks of 32, staged
// twice in a row in a warp-private shared-memory buffer, so that in step t of
// 32 lane l reads body (l + t) mod 32 at a fixed offset from its own address:
// every lane works on another j body, and the sums of the j bodies travel
// with them, one shuffle to the neighbouring lane per step and word.  After 32
// steps each j body's sums over the warp's row are back in its own lane.  No
// atomics and no reduction over lanes are needed, and the order of every sum
// is fixed by the decomposition: results are bit-reproducible.
//
// The warps' j sums of a unit meet in a slab in shared memory, one unit later
// (three slabs; phase_wait, so no warp stops for the others); each j body's four
// are added in warp order and go to the partial slot of the tile's delta.  The i
// sums go to a slot per (row, block).  The consumers (the kick, the acceleration
// output) add a body's slots in order.
//
// The tile of a block with itself: the chunk's bodies lie in the row of one
// warp r.  That warp sums them without the j side (so its own row is a full
// square, 32 kw of the n bodies); the rows' six unordered pairs are taken by
// the warps r - 1 (all) and r - 2 (the first two), counted mod 4.
#pragma once

#include "arith.cuh"
#include "nb_internal.cuh"
#include "split.cuh"

namespace nb {

constexpr int SWARPS = TILE / 32;   // warps per block

// Per-cluster values by value (kernel parameter): uniform across the block.
// The widest table also carries the blocks' launch order (nperm = 0: index
// order).
template <int KC>
struct SymTab {
    int32_t K;
    int32_t nperm;
    uint16_t perm[KC >= PARAM_CLUSTERS ? PERM_CAP : 1];
    int64_t uoff[KC + 1];
    int64_t boff[KC];
    int64_t poff[KC];
    double mu[KC];
    int32_t nk[KC];
    float eps2f[KC];
};
template <int KC>
using SymTabOf = SymTab<KC == 0 ? 1 : KC>;

// The units of a row in order: unit `sub` of tile delta covers the j bodies
// [j0, j1) of block b + delta; j1 <= j0 past the cluster's end (a ragged last
// block).
struct SymUnit {
    int32_t delta, sub, c, j0, j1;
    __device__ __forceinline__ void range(const Decomp &d, int32_t n)
    {
        j0 = c * d.ipb + sub * d.jt;
        j1 = j0 + d.jt < n ? j0 + d.jt : n;
    }
    __device__ __forceinline__ void at(const Decomp &d, const SymRows &sr, int32_t b, int32_t t,
                                       int32_t upt, int32_t n)
    {
        delta = t / upt;
        sub = t - delta * upt;
        c = b + delta < sr.nb ? b + delta : b + delta - sr.nb;
        range(d, n);
    }
    __device__ __forceinline__ void next(const Decomp &d, const SymRows &sr, int32_t upt, int32_t n)
    {
        if (++sub == upt) {
            sub = 0;
            ++delta;
            c = c + 1 == sr.nb ? 0 : c + 1;
        }
        range(d, n);
    }
};

// Block-wide phases without a stop: a warp arrives when its part of a unit's
// slab is written and waits for a unit's phase one unit later, when the other
// warps have long arrived.  The wait is bounded: a phase that does not come
// (it cannot: every warp of the block runs the same units) leaves a mark in
// the result flag.
__device__ __forceinline__ void phase_arrive(uint32_t bar)
{
    asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.shared::cta.b64 t, [%0];\n\t}" ::"r"(bar)
                 : "memory");
}
__device__ __forceinline__ void phase_wait(uint32_t bar, uint32_t parity, int *flag)
{
    for (int tries = 0; tries < (1 << 22); ++tries) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(bar), "r"(parity)
                     : "memory");
        if (ok) return;
    }
    atomicOr(flag, 2);
}

// Block of the decomposition that launch position q runs: sets of clusters carry
// an order by estimated work, largest first (block_order), so that the cheap
// blocks (ragged rows, tiles of blocks with themselves) set the kernel's tail;
// units and slots stay with the block's index.  Float-float kernel of 200 clusters
// of 100 to 1500 bodies 277 -> 266 us, of 48 79 -> 77 us.  For one system such an
// order changed nothing (16384 bodies 109 -> 112 us).
template <int KC>
__device__ __forceinline__ int64_t sym_block(const SymTabOf<KC> &t)
{
    if (KC >= PARAM_CLUSTERS && t.nperm > 0) return t.perm[blockIdx.x];
    return blockIdx.x;
}

// A: the arithmetic.  It gives
//   I          bodies per thread; groups(kw): how many groups of them hold bodies
//   JSUM       whether the j side is summed (not for the potential)
//   Stage      a warp's staged chunk; Pre: one lane's j body on its way there
//   IState     the thread's i bodies and their sums; JSum: its j body's sums
//   pass<SYM, MASK, PA>   32 steps over the chunk for the first PA groups
//   Slab, ACC  type of the warps' j sums; floats of running sums per thread in
//              shared memory
template <class A>
struct SymShared {
    typename A::Stage stage[SWARPS];
    typename A::Slab slab[A::JSUM ? 3 : 1][SWARPS][3][A::JSUM ? TILE : 1];
    float acc[A::ACC > 0 ? A::ACC : 1][TILE];
    uint64_t bar;
};

template <class A, int KC>
__global__ void __launch_bounds__(TILE, A::MINB) pair_sym_kernel(
    const __grid_constant__ DevState s, const __grid_constant__ SymTabOf<KC> tab,
    const __grid_constant__ Decomp d, double G)
{
    constexpr int I = A::I, CH = 32 * A::JL;
    extern __shared__ __align__(16) unsigned char smem[];
    SymShared<A> &sh = *reinterpret_cast<SymShared<A> *>(smem);

    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int w = tid >> 5;
    typename A::Stage &st = sh.stage[w];
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&sh.bar);
    if (A::JSUM) {
        if (tid == 0)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(SWARPS) : "memory");
        __syncthreads();
    }
    const int64_t g = sym_block<KC>(tab);
    int64_t u = d.U(g);
    const int64_t uend = d.U(g + 1);
    const int32_t upt = d.ipb / d.jt;
    int32_t phase = 0, buf = 0;   // units summed so far; phase mod 3

    while (u < uend) {
        const int32_t k = KC == 1 ? 0
                          : KC > 0 ? find_in(tab.uoff, tab.K, u)
                                   : find_cluster(s.cl.uoff, s.cl.K, u);
        const int64_t u0 = KC > 0 ? tab.uoff[k] : s.cl.uoff[k];
        const int32_t n = KC > 0 ? tab.nk[k] : (int32_t)s.cl.nk[k];
        const int64_t base = KC > 0 ? tab.boff[k] : s.cl.boff[k];
        const int64_t prow = 3 * (KC > 0 ? tab.poff[k] : s.cl.poff[k]);
        const double mu = KC > 0 ? tab.mu[k] : s.cl.mu[k];
        const typename A::Eps eps(KC > 0 ? tab.eps2f[k] : s.cl.eps2f[k], s.cl.eps2d + k);
        const SymRows sr(n, d.ipb);
        const int64_t lu = u - u0;
        const int32_t b = sr.row_of(lu / upt);
        const int64_t rf = sr.row_first(b) * upt;
        const int32_t t0 = (int32_t)(lu - rf);
        const int32_t nt = sr.row_tiles(b) * upt;
        const int32_t t1 = uend - u < nt - t0 ? t0 + (int32_t)(uend - u) : nt;
        const int32_t slot_i = (int32_t)(g - d.owner(u0 + rf)) + (A::JSUM ? sr.jslots(b) : 0);
        typename A::Part *const part = reinterpret_cast<typename A::Part *>(s.part) + prow;

        // the block's bodies, spread over the four warps: rows of 32 kw
        const int32_t ib0 = b * d.ipb;
        const int32_t rem = n - ib0 < d.ipb ? n - ib0 : d.ipb;
        const int32_t kw = (rem + TILE * A::JL - 1) / (TILE * A::JL) * A::JL;
        const int32_t rw = 32 * kw;
        const int32_t nw = (rem + rw - 1) / rw;   // warps with bodies
        const int32_t r0 = ib0 + w * rw;
        const bool live = w < nw;
        const int32_t pact = A::groups(kw);
        // both sides' scale: a_i += G m_j d / r^3, a_j -= G m_i d / r^3
        const typename A::Wide::Scale gmi(A::UM ? G * mu : G), gmj = gmi.negated();

        typename A::IState is;
        is.load(s, base, r0 + lane, n, kw);
#pragma unroll
        for (int r = 0; r < A::ACC; ++r) sh.acc[r][tid] = 0.f;

        // the j sums of one unit, all warps' in warp order, to its slot
        auto combine = [&](int32_t slab, int32_t delta, int32_t j0, int32_t j1) {
            const int32_t j = j0 + tid;
            if (j >= j1) return;
            int32_t who = (1 << nw) - 1;   // warps that summed this body
            if (delta == 0) {
                const int32_t r = (j - ib0) / rw;
                who = 1 << ((r - 1) & (SWARPS - 1));
                if (r >= 2) who |= 1 << (r - 2);
                who &= (1 << nw) - 1;
            }
            typename A::Part *o = part + (int64_t)delta * 3 * n + j;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                typename A::Wide v;
                v.zero();
#pragma unroll
                for (int q = 0; q < SWARPS; ++q)
                    if (who >> q & 1) v.add(sh.slab[slab][q][c][tid]);
                o[(int64_t)c * n] = v.scaled(gmj);
            }
        };

        SymUnit un;
        un.at(d, sr, b, t0, upt, n);
        typename A::Pre pre;
        pre.load(s, base, un.j0 + lane, n);
        int32_t folded = 0;
        int32_t pend = -1, pend_buf = 0, pend_j0 = 0, pend_j1 = 0;   // delta of the unit to combine
        for (int32_t t = t0; t < t1; ++t) {
            SymUnit nx = un;
            if (t + 1 < t1) nx.next(d, sr, upt, n);
            for (int32_t j0 = un.j0; j0 < un.j1; j0 += CH) {
                A::put(st, lane, pre);
                __syncwarp();
                // the next chunk's bodies on their way
                pre.load(s, base, (j0 + CH < un.j1 ? j0 + CH : nx.j0) + lane, n);
                typename A::JSum js;
                js.zero();
                if (live) {
                    bool own = false, sym = true;
                    if (un.delta == 0) {
                        const int32_t rel = ((j0 - ib0) / rw - w) & (SWARPS - 1);
                        own = rel == 0;
                        sym = rel == 1 || (rel == 2 && w < 2);
                    }
                    if (own) {
                        const int32_t kd = (j0 - r0) >> 5;
                        if (A::SELF || d.mask_self)
                            A::template run<false, true>(pact, st, lane, is, js, eps, kd);
                        else
                            A::template run<false, false>(pact, st, lane, is, js, eps, 0);
                    } else if (sym) {
                        A::template run<A::JSUM, false>(pact, st, lane, is, js, eps, 0);
                    }
                    if (++folded == A::FOLD_CHUNKS) {
                        is.fold(sh.acc, tid);
                        folded = 0;
                    }
                }
                if (A::JSUM) {
                    const int32_t jj = j0 - un.j0 + lane;
#pragma unroll
                    for (int c = 0; c < 3; ++c)
#pragma unroll
                        for (int h = 0; h < A::JL; ++h)
                            sh.slab[buf][w][c][jj + 32 * h] = js.get(c, h);
                }
                __syncwarp();
            }
            if (un.j1 <= un.j0) {
                pre.load(s, base, nx.j0 + lane, n);
            } else if (A::JSUM) {
                // the unit before this one (its phase long complete), then this
                // one's arrival: whoever waits for it knows that the slab of the
                // unit before is free, so three slabs are enough
                if (pend >= 0) {
                    phase_wait(bar, (phase - 1) & 1, s.flag);
                    combine(pend_buf, pend, pend_j0, pend_j1);
                }
                __syncwarp();
                if (lane == 0) phase_arrive(bar);
                pend = un.delta;
                pend_buf = buf;
                pend_j0 = un.j0;
                pend_j1 = un.j1;
                ++phase;
                buf = buf == 2 ? 0 : buf + 1;
            }
            un = nx;
        }
        if (A::JSUM && pend >= 0) {
            phase_wait(bar, (phase - 1) & 1, s.flag);
            combine(pend_buf, pend, pend_j0, pend_j1);
        }
        if (live) {
            is.fold(sh.acc, tid);
            typename A::Part *o = part + (int64_t)slot_i * 3 * n;
#pragma unroll
            for (int kk = 0; kk < I; ++kk) {
                const int32_t i = r0 + lane + 32 * kk;
                if (kk < kw && i < n) {
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        if (c == 0 || A::JSUM)
                            o[(int64_t)c * n + i] = is.sum(sh.acc, tid, kk, c).scaled(gmi);
                }
            }
        }
        u += t1 - t0;
    }
}

// Lane l's value moves to lane l - 1: after it a lane holds its neighbour's.
__device__ __forceinline__ float rot1(float v, int next) { return __shfl_sync(0xffffffffu, v, next); }
__device__ __forceinline__ float2 rot1(float2 v, int next)
{
    return make_float2(rot1(v.x, next), rot1(v.y, next));
}
__device__ __forceinline__ double rot1(double v, int next)
{
    return __shfl_sync(0xffffffffu, v, next);
}

// Double-single and double running values of a partial sum.
struct WideDS {
    float h, l;
    __device__ __forceinline__ void zero() { h = l = 0.f; }
    __device__ __forceinline__ void add(float t) { ds_add(h, l, t); }
    struct Scale {
        float gh, gl;
        __device__ __forceinline__ explicit Scale(double Gm)
        {
            gh = __double2float_rn(Gm);
            gl = __double2float_rn(Gm - (double)gh);
        }
        __device__ __forceinline__ Scale negated() const
        {
            Scale r(*this);
            r.gh = -gh;
            r.gl = -gl;
            return r;
        }
    };
    // times the scale in float-float (FMA-exact h gh plus the cross terms),
    // normalised
    __device__ __forceinline__ float2 scaled(const Scale &g) const
    {
        const float p = __fmul_rn(h, g.gh);
        float e = __fmaf_rn(h, g.gh, -p);
        e = __fmaf_rn(h, g.gl, __fmaf_rn(l, g.gh, e));
        const float r = __fadd_rn(p, e);
        return make_float2(r, __fsub_rn(e, __fsub_rn(r, p)));
    }
};
struct WideF64 {
    double v;
    __device__ __forceinline__ void zero() { v = 0.0; }
    __device__ __forceinline__ void add(double t) { v += t; }
    struct Scale {
        double g;
        __device__ __forceinline__ explicit Scale(double Gm) : g(Gm) {}
        __device__ __forceinline__ Scale negated() const { return Scale(-g); }
    };
    __device__ __forceinline__ double scaled(const Scale &k) const { return k.g * v; }
};

// Variants over 48 KB of shared memory need the limit raised on the device.
template <class A, int KC>
cudaError_t sym_shared_limit()
{
    if (sizeof(SymShared<A>) <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(pair_sym_kernel<A, KC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(SymShared<A>));
}

// Host side: fill the by-value table and launch.
template <class A, int KC>
cudaError_t launch_sym(const DevState &s, const PairLaunch &pl, const HostTab &ht, double G,
                       cudaStream_t st)
{
    SymTabOf<KC> t{};
    if (KC > 0) {
        if (ht.K > KC) return cudaErrorInvalidValue;
        t.K = ht.K;
        if (KC >= PARAM_CLUSTERS && ht.perm && ht.nperm == pl.d.G && ht.nperm <= PERM_CAP) {
            t.nperm = ht.nperm;
            for (int32_t q = 0; q < ht.nperm; ++q) t.perm[q] = ht.perm[q];
        }
        for (int32_t q = 0; q < ht.K; ++q) {
            t.uoff[q] = ht.uoff[q];
            t.boff[q] = ht.boff[q];
            t.poff[q] = ht.poff[q];
            t.nk[q] = (int32_t)ht.nk[q];
            t.eps2f[q] = ht.eps2f[q];
            t.mu[q] = ht.mu ? ht.mu[q] : 0.0;
        }
        t.uoff[ht.K] = ht.uoff[ht.K];
    }
    const cudaError_t e = sym_shared_limit<A, KC>();
    if (e != cudaSuccess) return e;
    pair_sym_kernel<A, KC><<<(unsigned)pl.d.G, TILE, sizeof(SymShared<A>), st>>>(s, t, pl.d, G);
    return cudaGetLastError();
}

template <class A, int KC>
int occupancy_sym()
{
    int nb = 0;
    if (sym_shared_limit<A, KC>() != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pair_sym_kernel<A, KC>, TILE,
                                                      sizeof(SymShared<A>)) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

template <class A>
cudaError_t launch_sym_any(const DevState &s, const PairLaunch &pl, const HostTab &ht, double G,
                           cudaStream_t st)
{
    if (ht.K == 1) return launch_sym<A, 1>(s, pl, ht, G, st);
    if (ht.K <= PARAM_CLUSTERS) return launch_sym<A, PARAM_CLUSTERS>(s, pl, ht, G, st);
    return launch_sym<A, 0>(s, pl, ht, G, st);
}
template <class A>
int occupancy_sym_any()
{
    const int a = occupancy_sym<A, 1>(), b = occupancy_sym<A, PARAM_CLUSTERS>(),
              c = occupancy_sym<A, 0>();
    return a < b ? (a < c ? a : c) : (b < c ? b : c);
}

// the variants (pairsym_sp.cu, pairsym_wide.cu)
cudaError_t launch_sym_sp(const DevState &s, const PairLaunch &pl, const HostTab &ht, double G,
                          cudaStream_t st);
int occupancy_sym_sp(int mode, int I, bool um);
cudaError_t launch_sym_wide(const DevState &s, const PairLaunch &pl, const HostTab &ht, double G,
                            cudaStream_t st);
int occupancy_sym_wide(int mode, int I);

}  // namespace nb
