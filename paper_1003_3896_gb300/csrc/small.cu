// small.cu -- whole steps of a small system in one kernel.
//
// A step of a few hundred bodies is a chain of five kernels (frame moments,
// frame, drift, pair sums, kick) that each last a few microseconds, most of it
// their start and the memory latency between them; the pair arithmetic of 480
// bodies is one microsecond.  Here one thread-block cluster of 16 blocks on 16 SMs
// runs all steps of the call: every block holds all bodies' split coordinates
// in shared memory and owns a sixteenth of the bodies, the blocks write the
// split of their bodies into each other's shared memory (two sets in turn, so
// one cluster barrier per exchange) and meet at hardware cluster barriers.
//
// The sums are those of the separate kernels, operation for operation: the float
// partial sums of each run of the full decomposition (a thread per two bodies,
// packed, and run), folded, scaled, added in run order, the frame's moments by
// the same tree.  So results do not depend on which path ran a step.
//
// What bounds it: up to about 500 bodies the barriers, exchanges and the chain of
// double-precision operations between them (4 to 5 us per force evaluation);
// above, the FP32 pipes of 16 SMs.
//
// The lines, measured (us; separate kernels -> here, mixed mode without a field):
//   bodies   one leapfrog call   64 leapfrogs, each   sixth-order call
//     384       27.5 -> 22.2        18.2 ->  8.6        71.0 -> 53.0
//     512       28.0 -> 22.2        18.9 ->  8.9        71.7 -> 54.1
//     704       29.1 -> 25.5        19.6 -> 11.5        75.9 -> 71.4
//     768       28.5 -> 26.3        19.6 -> 12.7        74.8 -> 79.3
//    1024       29.4 -> 29.3        20.0 -> 15.5        76.1 -> 99.4
// pure float: 1024 leapfrogs 19.5 -> 12.6, sixth order 768 70.5 -> 67.8, 896 73.0
// -> 75.7.  So leapfrogs up to SMALL_MAX = 1024, where the shared memory ends, and
// sixth-order steps, which spread the launch and the frame over seven
// evaluations, up to SMALL_SI6_DS and SMALL_SI6_FP32.
#include <cooperative_groups.h>

#include "arith.cuh"
#include "engine.h"
#include "step.cuh"

namespace nb {
constexpr int SMALL_SI6_DS = 704, SMALL_SI6_FP32 = 832;

namespace {

namespace cg = cooperative_groups;

constexpr int SB = 16;                       // blocks of the cluster
constexpr int SMT = 512;                     // threads per block
constexpr int OWN = SMALL_MAX / SB;          // bodies per block, at most (even)
constexpr int SRT = 256;                     // threads of a reduction segment (integrate.cu)
constexpr int SEGS = (SMALL_MAX + SEG_BODIES - 1) / SEG_BODIES;

struct SmallShared {
    float4 hi[2][SMALL_MAX], lo[2][SMALL_MAX];   // split coordinates (and mass), two sets
    float2 run[3][SMALL_SLOTS][OWN];             // each run's scaled sums of own bodies
    double seg[4][SEG_BODIES];                   // segment `rank`: m, x, y, z
    double tree[5][SRT];
    double mom[SEGS][5];                         // every segment's moments
    int J0[2][SMALL_SLOTS], J1[2][SMALL_SLOTS];  // runs of the (at most two) rows
    int nrun[2], c8[2];                          // their number, slots per part
};

struct SmallArgs {
    DevState s;
    Decomp d;
    ExtField ext;
    int n, ntiles;
    int64_t base;           // first body's index
    float eps2f;
    double eps2d, dt;       // softening squared, scale of the step length
    double h;
    double wk[7];
    int stages;
    int64_t steps;
    double Gm;
};

// q / n for 0 <= q < 4096 and n <= OWN (a multiplication: the quotients are taken
// in every force evaluation).
__device__ __forceinline__ unsigned reciprocal(int n) { return n ? ((1u << 20) + n - 1) / n : 0u; }
__device__ __forceinline__ int over(int q, unsigned r) { return (int)((unsigned)q * r >> 20); }

template <bool FULL, bool UM, bool EXT>
__global__ void __launch_bounds__(SMT, 1) small_step_kernel(const __grid_constant__ SmallArgs a)
{
    extern __shared__ __align__(16) unsigned char raw[];
    SmallShared &sh = *reinterpret_cast<SmallShared *>(raw);
    const cg::cluster_group cluster = cg::this_cluster();
    const DevState &s = a.s;
    const Decomp &d = a.d;
    const int tid = threadIdx.x, rank = (int)cluster.block_rank();
    const int n = a.n;
    const int64_t base = a.base;
    const int own = 2 * ((n + 2 * SB - 1) / (2 * SB));   // even: pairs of bodies share a row
    const int i0 = rank * own < n ? rank * own : n, i1 = i0 + own < n ? i0 + own : n;
    const int nown = i1 - i0;
    const float eps2 = a.eps2f;
    const int np8 = slot_parts(d, n);
    const double dt = a.dt, hstep = a.h;
    const float gh = __double2float_rn(a.Gm), gl = __double2float_rn(a.Gm - (double)gh);

    // own bodies' state: one thread each
    const bool mine = tid < nown;
    const int64_t gi = base + i0 + tid;
    double x = 0, y = 0, z = 0, vx = 0, vy = 0, vz = 0;
    float m = 0.f;
    if (mine) {
        x = s.x[gi];
        y = s.y[gi];
        z = s.z[gi];
        vx = s.vx[gi];
        vy = s.vy[gi];
        vz = s.vz[gi];
        m = s.mf[gi];
    }
    // the reduction segment of this block, and the one of this thread's body
    const int S = (n + SEG_BODIES - 1) / SEG_BODIES;
    const int ns = rank < S ? (n - rank * SEG_BODIES < SEG_BODIES ? n - rank * SEG_BODIES
                                                                 : SEG_BODIES)
                            : 0;
    for (int t = tid; t < ns; t += SMT) {
        const int64_t i = base + rank * SEG_BODIES + t;
        sh.seg[0][t] = s.m[i];
        sh.seg[1][t] = s.x[i];
        sh.seg[2][t] = s.y[i];
        sh.seg[3][t] = s.z[i];
    }
    // the runs of the rows that hold own bodies
    const int row0 = i0 / d.ipb;
    for (int r = 0; r < 2; ++r) {
        const int64_t nt = d.units_per_iblock(a.ntiles);
        const int64_t u0 = (int64_t)(row0 + r) * nt, u1 = u0 + nt;
        if ((int64_t)(row0 + r) * d.ipb >= n) {
            if (tid == 0) sh.nrun[r] = 0;
            continue;
        }
        const int64_t first = d.owner(u0);
        const int nr = (int)(d.owner(u1 - 1) - first) + 1;   // <= d.slots <= SMALL_SLOTS
        if (tid == 0) {
            sh.nrun[r] = nr;
            sh.c8[r] = (nr + np8 - 1) / np8;
        }
        if (tid < nr) {
            const int64_t ua = d.U(first + tid), ub = d.U(first + tid + 1);
            sh.J0[r][tid] = (int)(((ua > u0 ? ua : u0) - u0) * d.jt);
            const int64_t J1 = ((ub < u1 ? ub : u1) - u0) * d.jt;
            sh.J1[r][tid] = (int)(J1 < n ? J1 : n);   // padding adds exactly zero
        }
    }
    const int sl = (i0 + tid) % SEG_BODIES;
    SmallShared *const so =
        cluster.map_shared_rank(&sh, mine ? (i0 + tid) / SEG_BODIES : 0);
    int buf = 0;
    cluster.sync();   // every block of the cluster runs
    const int np = (nown + 1) / 2, row1 = (row0 + 1) * d.ipb;
    const unsigned by_np = reciprocal(np), by_nown = reciprocal(nown);
    const int most = sh.nrun[0] > sh.nrun[1] ? sh.nrun[0] : sh.nrun[1];

    for (int64_t step = 0; step < a.steps; ++step) {
        // the frame's moments, a segment per block: 256 threads' sums, then the
        // reduction tree of integrate.cu, a warp per moment
        if (rank < S) {
            if (tid < SRT) {
                double v[5] = {0, 0, 0, 0, 0};
                for (int t = tid; t < ns; t += SRT)
                    moment_add(v, sh.seg[0][t], sh.seg[1][t], sh.seg[2][t], sh.seg[3][t]);
                for (int q = 0; q < 5; ++q) sh.tree[q][tid] = v[q];
            }
            __syncthreads();
            const int q = tid >> 5, lane = tid & 31;
            if (q < 5) {
                double t[8];
#pragma unroll
                for (int w = 0; w < 8; ++w) t[w] = sh.tree[q][32 * w + lane];
#pragma unroll
                for (int w = 4; w > 0; w >>= 1)
#pragma unroll
                    for (int r = 0; r < w; ++r) t[r] += t[r + w];
                double u = t[0];
                for (int w = 16; w > 0; w >>= 1) u += __shfl_down_sync(0xffffffffu, u, w);
                u = __shfl_sync(0xffffffffu, u, 0);
                if (lane < SB) cluster.map_shared_rank(&sh, lane)->mom[rank][q] = u;
            }
        }
        cluster.sync();
        Frame f{};
        if (mine) {
            double v[5];
            for (int q = 0; q < 5; ++q) v[q] = sh.mom[0][q];
            for (int g = 1; g < S; ++g)
                for (int q = 0; q < 5; ++q) v[q] += sh.mom[g][q];
            f = frame_of(v, a.eps2d);
        }

        for (int k = -1; k < a.stages; ++k) {
            if (k >= 0) {
                // pair sums: own bodies 2p, 2p + 1 (packed) against one run
                for (int q = tid; q < np * most; q += SMT) {
                    const int g = over(q, by_np), il = 2 * (q - g * np), i = i0 + il;
                    const int r = i >= row1;
                    if (g >= sh.nrun[r]) continue;
                    const int J0 = sh.J0[r][g], J1 = sh.J1[r][g];
                    const bool two = il + 1 < nown;
                    const float4 ha = sh.hi[buf][i], hb = sh.hi[buf][two ? i + 1 : i];
                    const float2 nx = make_float2(-ha.x, -hb.x), ny = make_float2(-ha.y, -hb.y),
                                 nz = make_float2(-ha.z, -hb.z);
                    float2 nlx, nly, nlz;
                    if (FULL) {
                        const float4 la = sh.lo[buf][i], lb = sh.lo[buf][two ? i + 1 : i];
                        nlx = make_float2(-la.x, -lb.x);
                        nly = make_float2(-la.y, -lb.y);
                        nlz = make_float2(-la.z, -lb.z);
                    }
                    const float2 e2 = make_float2(eps2, eps2);
                    float h[2][3] = {}, l[2][3] = {};
                    for (int ja = J0; ja < J1; ja += 4 * TILE) {
                        const int jb = ja + 4 * TILE < J1 ? ja + 4 * TILE : J1;
                        float2 ax = make_float2(0.f, 0.f), ay = ax, az = ax;
#pragma unroll 8
                        for (int j = ja; j < jb; ++j) {
                            const float4 A = sh.hi[buf][j];
                            float2 dx = __fadd2_rn(make_float2(A.x, A.x), nx);
                            float2 dy = __fadd2_rn(make_float2(A.y, A.y), ny);
                            float2 dz = __fadd2_rn(make_float2(A.z, A.z), nz);
                            if (FULL) {
                                const float4 B = sh.lo[buf][j];
                                dx = __fadd2_rn(dx, __fadd2_rn(make_float2(B.x, B.x), nlx));
                                dy = __fadd2_rn(dy, __fadd2_rn(make_float2(B.y, B.y), nly));
                                dz = __fadd2_rn(dz, __fadd2_rn(make_float2(B.z, B.z), nlz));
                            }
                            float2 r2 = __ffma2_rn(dx, dx, e2);
                            r2 = __ffma2_rn(dy, dy, r2);
                            r2 = __ffma2_rn(dz, dz, r2);
                            const float2 ri = make_float2(rsqrt_mufu(r2.x), rsqrt_mufu(r2.y));
                            float2 sp = __fmul2_rn(
                                UM ? ri : __fmul2_rn(make_float2(A.w, A.w), ri), __fmul2_rn(ri, ri));
                            if (d.mask_self) {
                                if (j == i) sp.x = 0.f;
                                if (j == i + 1) sp.y = 0.f;
                            }
                            ax = __ffma2_rn(dx, sp, ax);
                            ay = __ffma2_rn(dy, sp, ay);
                            az = __ffma2_rn(dz, sp, az);
                        }
                        const float t[2][3] = {{ax.x, ay.x, az.x}, {ax.y, ay.y, az.y}};
#pragma unroll
                        for (int b = 0; b < 2; ++b)
#pragma unroll
                            for (int c = 0; c < 3; ++c) {
                                if (FULL)
                                    ds_add(h[b][c], l[b][c], t[b][c]);
                                else
                                    h[b][c] = __fadd_rn(h[b][c], t[b][c]);
                            }
                    }
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        float2 o[2];
#pragma unroll
                        for (int b = 0; b < 2; ++b) {
                            const float pr = __fmul_rn(h[b][c], gh);
                            float e = __fmaf_rn(h[b][c], gh, -pr);
                            e = __fmaf_rn(h[b][c], gl, __fmaf_rn(l[b][c], gh, e));
                            const float t = __fadd_rn(pr, e);
                            o[b] = make_float2(t, __fsub_rn(e, __fsub_rn(t, pr)));
                        }
                        // (a lone body's pair slot is its own: il + 1 < OWN)
                        *reinterpret_cast<float4 *>(&sh.run[c][g][il]) =
                            make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
                    }
                }
                __syncthreads();
                // the runs' sums, a thread per body and part (slot_parts)
                for (int q = tid; q < nown * np8; q += SMT) {
                    const int p = over(q, by_nown), il = q - p * nown;
                    const int r = i0 + il >= row1, nr = sh.nrun[r], c8 = sh.c8[r], g0 = p * c8;
                    if (g0 >= nr) continue;
                    float h[3] = {0.f, 0.f, 0.f}, l[3] = {0.f, 0.f, 0.f};
                    for (int g = g0; g < nr && g < g0 + c8; ++g)
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            const float2 t = sh.run[c][g][il];
                            ff_add(h[c], l[c], t.x, t.y);
                        }
#pragma unroll
                    for (int c = 0; c < 3; ++c) sh.run[c][g0][il] = make_float2(h[c], l[c]);
                }
                __syncthreads();
            }
            const bool last = k + 1 == a.stages;
            if (mine) {
                if (k >= 0) {
                    const int r = i0 + tid >= row1, nr = sh.nrun[r], c8 = sh.c8[r];
                    float H[3] = {0.f, 0.f, 0.f}, L[3] = {0.f, 0.f, 0.f};
                    for (int g = 0; g < nr; g += c8)
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            const float2 p = sh.run[c][g][tid];
                            ff_add(H[c], L[c], p.x, p.y);
                        }
                    double ax = widen(H[0]) + widen(L[0]), ay = widen(H[1]) + widen(L[1]),
                           az = widen(H[2]) + widen(L[2]);
                    if (EXT) field_accel(a.ext, x, y, z, ax, ay, az);
                    const double hk = (a.wk[k] * hstep) * dt;
                    vx = moved(hk, ax, vx);
                    vy = moved(hk, ay, vy);
                    vz = moved(hk, az, vz);
                }
                const double w0 = k >= 0 ? a.wk[k] : 0.0, w1 = last ? 0.0 : a.wk[k + 1];
                const double hd = (k < 0 ? 0.5 * w1 * hstep : 0.5 * (w0 + w1) * hstep) * dt;
                x = moved(hd, vx, x);
                y = moved(hd, vy, y);
                z = moved(hd, vz, z);
                if (last && step + 1 == a.steps) {
                    s.x[gi] = x;
                    s.y[gi] = y;
                    s.z[gi] = z;
                    s.vx[gi] = vx;
                    s.vy[gi] = vy;
                    s.vz[gi] = vz;
                } else if (last) {
                    so->seg[1][sl] = x;
                    so->seg[2][sl] = y;
                    so->seg[3][sl] = z;
                }
            }
            if (!last) {
                // the split into the other set, then to every block's copy
                const int to = buf ^ 1;
                if (mine) {
                    float4 hv, lv;
                    split_ds(x - f.cx, hv.x, lv.x);
                    split_ds(y - f.cy, hv.y, lv.y);
                    split_ds(z - f.cz, hv.z, lv.z);
                    hv.w = m;
                    lv.w = 0.f;
                    sh.hi[to][i0 + tid] = hv;
                    sh.lo[to][i0 + tid] = lv;
                }
                __syncthreads();
                for (int q = tid; q < nown * SB; q += SMT) {
                    const int r = over(q, by_nown), i = i0 + q - r * nown;
                    if (r == rank) continue;
                    SmallShared *o = cluster.map_shared_rank(&sh, r);
                    o->hi[to][i] = sh.hi[to][i];
                    if (FULL) o->lo[to][i] = sh.lo[to][i];
                }
                buf = to;
            }
            // the splits (or, after the last stage, the positions) of all blocks
            cluster.sync();
        }
    }
}

using Kernel = void (*)(SmallArgs);

Kernel kernel_of(bool full, bool um, bool ext)
{
    if (full) {
        if (um) return ext ? small_step_kernel<true, true, true> : small_step_kernel<true, true, false>;
        return ext ? small_step_kernel<true, false, true> : small_step_kernel<true, false, false>;
    }
    if (um) return ext ? small_step_kernel<false, true, true> : small_step_kernel<false, true, false>;
    return ext ? small_step_kernel<false, false, true> : small_step_kernel<false, false, false>;
}

cudaLaunchConfig_t config(cudaLaunchAttribute *at, cudaStream_t st)
{
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = SB;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(SB);
    c.blockDim = dim3(SMT);
    c.dynamicSmemBytes = sizeof(SmallShared);
    c.stream = st;
    c.attrs = at;
    c.numAttrs = 1;
    return c;
}

// Whether the device can hold the cluster (16 blocks: above the portable 8).
bool fits(Kernel kernel)
{
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t c = config(at, nullptr);
    int clusters = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(SmallShared)) != cudaSuccess ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&clusters, kernel, &c) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return clusters >= 1;
}

}  // namespace

bool small_ok(const ClusterSet &C, const Plan &pl, const Phys &ph)
{
    const Decomp &d = pl.pl.d;
    if (C.K != 1 || C.n > SMALL_MAX || d.sym || d.rows || d.b0 || d.slots > SMALL_SLOTS)
        return false;
    // a block's bodies lie in at most two rows
    if (d.ipb < OWN || !d.fpart) return false;
    if (pl.pl.mode != PM_DS_FULL && pl.pl.mode != PM_FP32) return false;
    return fits(kernel_of(pl.pl.mode == PM_DS_FULL, pl.pl.um, ph.ext.on));
}

bool small_order(const ClusterSet &C, const Plan &pl, int order)
{
    return order == 2 || C.n <= (pl.pl.mode == PM_FP32 ? SMALL_SI6_FP32 : SMALL_SI6_DS);
}

int small_steps(const Pool &P, const ClusterSet &C, const Plan &pl, const Phys &ph, int order,
                double h, int64_t steps, cudaStream_t st)
{
    SmallArgs a{};
    a.s = view(P, C, pl);
    a.d = pl.pl.d;
    a.ext = ph.ext;
    a.n = (int)C.n;
    a.ntiles = C.ntiles[0];
    a.base = C.boff[0];
    a.eps2f = C.eps2f[0];
    a.eps2d = C.eps2d[0];
    a.dt = C.dts[0];
    a.h = h;
    a.stages = stage_weights(order, a.wk);
    a.Gm = pl.pl.um ? ph.G * C.mu[0] : ph.G;
    const Kernel kernel = kernel_of(pl.pl.mode == PM_DS_FULL, pl.pl.um, ph.ext.on);
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t c = config(at, st);
    // a launch lasts a fraction of a second at most
    constexpr int64_t RUN = 4096;
    for (int64_t k = 0; k < steps; k += RUN) {
        a.steps = steps - k < RUN ? steps - k : RUN;
        NB_TRY(cudaLaunchKernelEx(&c, kernel, a));
    }
    return NB_OK;
}

}  // namespace nb
