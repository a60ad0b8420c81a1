// integrate.cu -- O(N) kernels over a set of clusters: state layout
// conversion, the per-cluster float frame and split, the fused kick(+external
// field)/drift substep of the symplectic schemes (Sect. 3.1), and
// deterministic per-cluster reductions for the diagnostics of Sect. 5.1.
// All state arithmetic is double precision (Sect. 4.2: the time advance is
// the round-off sensitive part).
//
// Per-body kernels run over linear body indices t (cluster after cluster);
// the set's body -> cluster map gives t's cluster k, and its pool slot is
// boff[k] + t - noff[k].
// Reductions run per segment (a run of one cluster's bodies), then one block
// per cluster adds its segments in a fixed tree order.
#include "arith.cuh"
#include "nb_internal.cuh"
#include "split.cuh"
#include "step.cuh"

namespace nb {

constexpr int RT = 256;   // threads per reduction block
constexpr int OT = 256;   // threads per block of the per-body kernels, at most

static inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// Threads per block of a per-body kernel over n bodies: OT, or fewer (a
// multiple of 32) when n is small, so the blocks spread over at least ~300
// SMs' worth of slots; these kernels carry FP64 arithmetic and dependent
// loads, and a small system on a few SMs waits on one SM's FP64 pipe.
static inline int ot_for(int64_t n)
{
    int t = 32;
    while (t < OT && (int64_t)t * 304 < n) t *= 2;
    return t;
}

struct BodyRef {
    int32_t k;     // cluster
    int64_t li;    // index inside the cluster
    int64_t gi;    // pool slot
};

__device__ __forceinline__ BodyRef body_at(const Clusters &c, int64_t t)
{
    BodyRef r;
    r.k = cluster_of(c, t);
    r.li = t - c.noff[r.k];
    r.gi = c.boff[r.k] + r.li;
    return r;
}

__device__ __forceinline__ double field_phi(const ExtField &e, double x, double y, double z)
{
    const double R2 = x * x + y * y;
    const double q = e.ad + sqrt(z * z + e.bd * e.bd);
    const double ph = e.Mbh > 0 ? e.G * e.Mbh * rsqrt(R2 + z * z + e.eps2bh) : 0.0;
    return -e.G * e.Md * rsqrt(R2 + q * q) - e.G * e.Mb * rsqrt(R2 + z * z + e.ab * e.ab) - ph;
}

// Tree reduction of NV doubles over a block of RT threads; fixed order.
template <int NV>
__device__ void block_sum(double (&v)[NV], double *sh)
{
    const int t = threadIdx.x;
    __syncthreads();
    for (int k = 0; k < NV; ++k) sh[k * RT + t] = v[k];
    __syncthreads();
    for (int w = RT / 2; w > 0; w >>= 1) {
        if (t < w)
            for (int k = 0; k < NV; ++k) sh[k * RT + t] += sh[k * RT + t + w];
        __syncthreads();
    }
    for (int k = 0; k < NV; ++k) v[k] = sh[k * RT];
}

// Sum of the NV segment partials of cluster blockIdx.x (fixed order).
template <int NV>
__device__ void cluster_sum(const DevState &s, double (&v)[NV], double *sh)
{
    const int k = blockIdx.x;
    for (int q = 0; q < NV; ++q) v[q] = 0.0;
    for (int sg = s.cl.seg_off[k] + threadIdx.x; sg < s.cl.seg_off[k + 1]; sg += RT)
        for (int q = 0; q < NV; ++q) v[q] += s.red[(int64_t)sg * 16 + q];
    block_sum<NV>(v, sh);
}

// ---- layout ------------------------------------------------------------------

__global__ void unpack_kernel(DevState s, const double *__restrict__ pos,
                              const double *__restrict__ vel, const double *__restrict__ mass)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= s.n) return;
    const int64_t i = body_at(s.cl, t).gi;
    s.x[i] = pos[3 * t];
    s.y[i] = pos[3 * t + 1];
    s.z[i] = pos[3 * t + 2];
    s.vx[i] = vel[3 * t];
    s.vy[i] = vel[3 * t + 1];
    s.vz[i] = vel[3 * t + 2];
    s.m[i] = mass[t];
    s.mf[i] = __double2float_rn(mass[t]);   // masses never change after load
}

// Positions and / or velocities (NULL: kept) of a loaded state.
__global__ void set_state_kernel(DevState s, const double *__restrict__ pos,
                                 const double *__restrict__ vel)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= s.n) return;
    const int64_t i = body_at(s.cl, t).gi;
    if (pos) {
        s.x[i] = pos[3 * t];
        s.y[i] = pos[3 * t + 1];
        s.z[i] = pos[3 * t + 2];
    }
    if (vel) {
        s.vx[i] = vel[3 * t];
        s.vy[i] = vel[3 * t + 1];
        s.vz[i] = vel[3 * t + 2];
    }
}

__global__ void pack_kernel(DevState s, double *__restrict__ pos, double *__restrict__ vel)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= s.n) return;
    const int64_t i = body_at(s.cl, t).gi;
    if (pos) {
        pos[3 * t] = s.x[i];
        pos[3 * t + 1] = s.y[i];
        pos[3 * t + 2] = s.z[i];
    }
    if (vel) {
        vel[3 * t] = s.vx[i];
        vel[3 * t + 1] = s.vy[i];
        vel[3 * t + 2] = s.vz[i];
    }
}

// cid[t] = cluster of linear body t (binary search once per layout).
__global__ void cluster_map_kernel(Clusters c, int32_t *cid, int64_t n)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t < n) cid[t] = find_cluster(c.noff, c.K, t);
}

cudaError_t launch_cluster_map(const Clusters &c, int32_t *cid, int64_t n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    cluster_map_kernel<<<blocks_for(n, ot_for(n)), ot_for(n), 0, st>>>(c, cid, n);
    return cudaGetLastError();
}

cudaError_t launch_unpack(const DevState &s, const double *pos, const double *vel,
                          const double *mass, cudaStream_t st)
{
    unpack_kernel<<<blocks_for(s.n, ot_for(s.n)), ot_for(s.n), 0, st>>>(s, pos, vel, mass);
    return cudaGetLastError();
}

cudaError_t launch_set_state(const DevState &s, const double *pos, const double *vel,
                             cudaStream_t st)
{
    set_state_kernel<<<blocks_for(s.n, ot_for(s.n)), ot_for(s.n), 0, st>>>(s, pos, vel);
    return cudaGetLastError();
}

cudaError_t launch_pack(const DevState &s, double *pos, double *vel, cudaStream_t st)
{
    pack_kernel<<<blocks_for(s.n, ot_for(s.n)), ot_for(s.n), 0, st>>>(s, pos, vel);
    return cudaGetLastError();
}

// ---- frame and split ---------------------------------------------------------

__global__ void frame_partial_kernel(DevState s)
{
    __shared__ double sh[5 * RT];
    const int sg = blockIdx.x;
    const int32_t k = s.cl.seg_k[sg];
    const int64_t base = s.cl.boff[k] - s.cl.noff[k];
    double v[5] = {0, 0, 0, 0, 0};
    for (int64_t t = s.cl.seg_lo[sg] + threadIdx.x; t < s.cl.seg_hi[sg]; t += RT) {
        const int64_t i = base + t;
        moment_add(v, s.m[i], s.x[i], s.y[i], s.z[i]);
    }
    block_sum<5>(v, sh);
    if (threadIdx.x == 0)
        for (int q = 0; q < 5; ++q) s.red[(int64_t)sg * 16 + q] = v[q];
}

__global__ void frame_final_kernel(DevState s, double near_frac)
{
    __shared__ double sh[5 * RT];
    double v[5];
    cluster_sum<5>(s, v, sh);
    if (threadIdx.x == 0) {
        const int k = blockIdx.x;
        const Frame f = frame_of(v, s.cl.eps2d[k]);
        s.cl.frame[k] = f;
    }
}

// Smallest and largest mass per segment, then per cluster (into diag[k][0..1]).
__global__ void mass_range_partial_kernel(DevState s)
{
    __shared__ double lo_sh[RT], hi_sh[RT];
    const int sg = blockIdx.x;
    const int32_t k = s.cl.seg_k[sg];
    const int64_t base = s.cl.boff[k] - s.cl.noff[k];
    double lo = INFINITY, hi = -INFINITY;
    for (int64_t t = s.cl.seg_lo[sg] + threadIdx.x; t < s.cl.seg_hi[sg]; t += RT) {
        const double m = s.m[base + t];
        lo = fmin(lo, m);
        hi = fmax(hi, m);
    }
    lo_sh[threadIdx.x] = lo;
    hi_sh[threadIdx.x] = hi;
    __syncthreads();
    for (int w = RT / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            lo_sh[threadIdx.x] = fmin(lo_sh[threadIdx.x], lo_sh[threadIdx.x + w]);
            hi_sh[threadIdx.x] = fmax(hi_sh[threadIdx.x], hi_sh[threadIdx.x + w]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        s.red[(int64_t)sg * 16] = lo_sh[0];
        s.red[(int64_t)sg * 16 + 1] = hi_sh[0];
    }
}

__global__ void mass_range_final_kernel(DevState s)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= s.cl.K) return;
    double lo = INFINITY, hi = -INFINITY;
    for (int sg = s.cl.seg_off[k]; sg < s.cl.seg_off[k + 1]; ++sg) {
        lo = fmin(lo, s.red[(int64_t)sg * 16]);
        hi = fmax(hi, s.red[(int64_t)sg * 16 + 1]);
    }
    s.diag[(int64_t)k * DIAG_STRIDE] = lo;
    s.diag[(int64_t)k * DIAG_STRIDE + 1] = hi;
}

cudaError_t launch_mass_range(const DevState &s, cudaStream_t st)
{
    mass_range_partial_kernel<<<s.cl.S, RT, 0, st>>>(s);
    mass_range_final_kernel<<<(s.cl.K + 127) / 128, 128, 0, st>>>(s);
    return cudaGetLastError();
}

// Harmonic moment about the frame origin: sum m / |x - c| (per segment),
// with a floor of 1e-3 R_rms on the distance.
__global__ void frame_harmonic_kernel(DevState s)
{
    __shared__ double sh[2 * RT];
    const int sg = blockIdx.x;
    const int32_t k = s.cl.seg_k[sg];
    const int64_t base = s.cl.boff[k] - s.cl.noff[k];
    const Frame f = s.cl.frame[k];
    const double floor2 = 1e-6 * f.r2rms + 1e-300;
    double v[2] = {0, 0};
    for (int64_t t = s.cl.seg_lo[sg] + threadIdx.x; t < s.cl.seg_hi[sg]; t += RT) {
        const int64_t i = base + t;
        const double dx = s.x[i] - f.cx, dy = s.y[i] - f.cy, dz = s.z[i] - f.cz;
        v[0] += s.m[i] * rsqrt(dx * dx + dy * dy + dz * dz + floor2);
        v[1] += s.m[i];
    }
    block_sum<2>(v, sh);
    if (threadIdx.x == 0)
        for (int q = 0; q < 2; ++q) s.red[(int64_t)sg * 16 + q] = v[q];
}

// Near-pair radius d_th = near_frac * S / N^{1/3}: a mean-spacing scale like
// the paper's softening rule (Sect. 2), so the expected number of near
// neighbours per body does not grow with N.  S = min(R_rms, 3 R_h) with the
// harmonic radius R_h = M / sum(m / |x - c|): for centrally concentrated
// clusters (Plummer: R_rms = 2.6 R_h; uniform sphere: 1.2 R_h) S is the rms
// radius, but once escapers or a disrupted halo inflate R_rms, S follows the
// bound core instead, so the core does not crowd into a few cells.
__global__ void frame_scale_kernel(DevState s, double near_frac)
{
    __shared__ double sh[2 * RT];
    double v[2];
    cluster_sum<2>(s, v, sh);
    if (threadIdx.x == 0) {
        const int k = blockIdx.x;
        Frame f = s.cl.frame[k];
        double scale2 = f.r2rms;
        if (v[0] > 0) {
            const double rh = v[1] / v[0];
            if (9.0 * rh * rh < scale2) scale2 = 9.0 * rh * rh;
        }
        const double nk = (double)s.cl.nk[k];
        const double spacing2 = scale2 / cbrt(nk * nk);
        f.th2 = (float)(near_frac * near_frac * spacing2 + s.cl.eps2d[k]);
        f.dth = (float)(near_frac * sqrt(spacing2));
        f.hx = scale2 > 0 ? HV_X * (float)(v[1] / scale2) : INFINITY;
        s.cl.frame[k] = f;
    }
}

cudaError_t launch_frame(const DevState &s, double near_frac, bool near, cudaStream_t st)
{
    frame_partial_kernel<<<s.cl.S, RT, 0, st>>>(s);
    frame_final_kernel<<<s.cl.K, RT, 0, st>>>(s, near_frac);
    if (near) {
        frame_harmonic_kernel<<<s.cl.S, RT, 0, st>>>(s);
        frame_scale_kernel<<<s.cl.K, RT, 0, st>>>(s, near_frac);
    }
    return cudaGetLastError();
}

// hi = fl32(x - c), lo = fl32((x - c) - hi): the double-single representation
// of Sect. 5.2, taken relative to the cluster's frame origin.
// MASS: also write the mass words of the j-stream copies (m and its float
// rounding residue); the kick's per-substep splits leave them as the step's
// first split wrote them (masses never change).
// JS: write the j-stream copies (the symmetric kernels read the planes).
template <bool MASS, bool JS = true>
__device__ __forceinline__ void split_one(const DevState &s, const Frame &f, int64_t i,
                                          double x, double y, double z)
{
    float hx, hy, hz, lx, ly, lz;
    split_ds(x - f.cx, hx, lx);
    split_ds(y - f.cy, hy, ly);
    split_ds(z - f.cz, hz, lz);
    s.xh[i] = hx;
    s.yh[i] = hy;
    s.zh[i] = hz;
    s.xl[i] = lx;
    s.yl[i] = ly;
    s.zl[i] = lz;
    if (!JS) return;
    s.jd[2 * i] = make_float4(hx, hx, hy, hy);
    s.jl[2 * i] = make_float4(lx, lx, ly, ly);
    if (MASS) {
        const float m = s.mf[i];
        const float ml = __double2float_rn(s.m[i] - (double)m);   // mass lo part (float-float)
        s.jd[2 * i + 1] = make_float4(hz, hz, m, m);
        s.jl[2 * i + 1] = make_float4(lz, lz, ml, ml);
    } else {
        *reinterpret_cast<float2 *>(&s.jd[2 * i + 1]) = make_float2(hz, hz);
        *reinterpret_cast<float2 *>(&s.jl[2 * i + 1]) = make_float2(lz, lz);
    }
}

__global__ void split_kernel(DevState s)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= s.n) return;
    const BodyRef r = body_at(s.cl, t);
    const int64_t i = r.gi;
    s.mf[i] = __double2float_rn(s.m[i]);
    split_one<true>(s, s.cl.frame[r.k], i, s.x[i], s.y[i], s.z[i]);
}

cudaError_t launch_split(const DevState &s, cudaStream_t st)
{
    split_kernel<<<blocks_for(s.n, ot_for(s.n)), ot_for(s.n), 0, st>>>(s);
    return cudaGetLastError();
}

// ---- substep -----------------------------------------------------------------

// Sum of a run of slots.  Float-pair partial sums (Decomp::fpart) are added in
// float-float arithmetic on the FP32 pipes and widened to double from their bits
// at the end (the conversion instruction runs on the FP64 pipe, 1/77 of the
// FP32 rate here); others in double.
template <bool FP>
struct SlotSum;
template <>
struct SlotSum<true> {
    float hx = 0.f, lx = 0.f, hy = 0.f, ly = 0.f, hz = 0.f, lz = 0.f;
    __device__ __forceinline__ void add(const SlotSum &o)
    {
        ff_add(hx, lx, o.hx, o.lx);
        ff_add(hy, ly, o.hy, o.ly);
        ff_add(hz, lz, o.hz, o.lz);
    }
    __device__ __forceinline__ void get(double &ax, double &ay, double &az) const
    {
        ax = widen(hx) + widen(lx);
        ay = widen(hy) + widen(ly);
        az = widen(hz) + widen(lz);
    }
};
template <>
struct SlotSum<false> {
    double x = 0.0, y = 0.0, z = 0.0;
    __device__ __forceinline__ void add(const SlotSum &o)
    {
        x += o.x;
        y += o.y;
        z += o.z;
    }
    __device__ __forceinline__ void get(double &ax, double &ay, double &az) const
    {
        ax = x;
        ay = y;
        az = z;
    }
};

// Slots [k0, k1) in order, four of them loaded together (more would cost resident
// warps, which hide the memory latency better).
template <bool FP>
__device__ __forceinline__ SlotSum<FP> sum_run(const DevState &s, const SlotRun &run, int64_t k0,
                                               int64_t k1)
{
    constexpr int SB = 4;
    const int64_t ps = run.stride;
    int64_t at = run.base + 3 * k0 * ps;
    SlotSum<FP> a;
    for (; k0 < k1; k0 += SB) {
        SlotSum<FP> b[SB];
#pragma unroll
        for (int q = 0; q < SB; ++q) {
            if (k0 + q >= k1) continue;
            if constexpr (FP) {
                const float2 *p = reinterpret_cast<const float2 *>(s.part) + at;
                const float2 x = p[0], y = p[ps], z = p[2 * ps];
                b[q].hx = x.x;
                b[q].lx = x.y;
                b[q].hy = y.x;
                b[q].ly = y.y;
                b[q].hz = z.x;
                b[q].lz = z.y;
            } else {
                const double *p = s.part + at;
                b[q].x = p[0];
                b[q].y = p[ps];
                b[q].z = p[2 * ps];
            }
            at += 3 * ps;
        }
#pragma unroll
        for (int q = 0; q < SB; ++q)
            if (k0 + q < k1) a.add(b[q]);
    }
    return a;
}

// A body in a close encounter: its whole sum is in corr.
template <bool FP>
__device__ __forceinline__ bool is_heavy(const DevState &s, const Decomp &d, int64_t t)
{
    return FP && d.sym && s.hv_flag && s.hv_flag[t] && *s.hv_count <= hv_limit(s.n);
}

// One thread per body (slot_parts = 1): float-pair partial sums in slot order.  SB:
// slots loaded together (a grid run in waves gives an i-block tens of slots; an
// ensemble of small clusters a few, where a narrower batch keeps registers, and so
// resident warps, for the memory latency).
template <int SB>
__device__ __forceinline__ void sum_slots_ff(const DevState &s, const SlotRun &run,
                                             double &ax, double &ay, double &az)
{
    const int64_t count = run.count, ps = run.stride;
    const float2 *part2 = reinterpret_cast<const float2 *>(s.part) + run.base;
    float hx = 0.f, lx = 0.f, hy = 0.f, ly = 0.f, hz = 0.f, lz = 0.f;
    for (int64_t k0 = 0; k0 < count; k0 += SB) {
        float2 bx[SB], by[SB], bz[SB];
#pragma unroll
        for (int q = 0; q < SB; ++q) {
            bx[q] = by[q] = bz[q] = make_float2(0.f, 0.f);
            if (k0 + q < count) {
                const float2 *p = part2 + ((k0 + q) * 3) * ps;
                bx[q] = p[0];
                by[q] = p[ps];
                bz[q] = p[2 * ps];
            }
        }
#pragma unroll
        for (int q = 0; q < SB; ++q)
            if (k0 + q < count) {
                ff_add(hx, lx, bx[q].x, bx[q].y);
                ff_add(hy, ly, by[q].x, by[q].y);
                ff_add(hz, lz, bz[q].x, bz[q].y);
            }
    }
    ax = widen(hx) + widen(lx);
    ay = widen(hy) + widen(ly);
    az = widen(hz) + widen(lz);
}

template <int SB, bool FP>
__device__ __forceinline__ void sum_slots(const DevState &s, const Decomp &d, const BodyRef &r,
                                          int64_t t, double &ax, double &ay, double &az)
{
    if (is_heavy<FP>(s, d, t)) {
        ax = s.corr[r.gi];
        ay = s.corr[s.cap + r.gi];
        az = s.corr[2 * s.cap + r.gi];
        return;
    }
    const SlotRun run = slot_run(d, s.cl, r.k, r.li, t, s.pstride);
    const int64_t count = run.count, ps = run.stride;
    if (FP) {
        sum_slots_ff<SB>(s, run, ax, ay, az);
        if (s.corr) {
            ax += s.corr[r.gi];
            ay += s.corr[s.cap + r.gi];
            az += s.corr[2 * s.cap + r.gi];
        }
        return;
    }
    ax = ay = az = 0.0;
    // slots in order, SB at a time so the loads are in flight together
    for (int64_t k0 = 0; k0 < count; k0 += SB) {
        double bx[SB], by[SB], bz[SB];
#pragma unroll
        for (int q = 0; q < SB; ++q) {
            bx[q] = by[q] = bz[q] = 0.0;
            if (k0 + q < count) {
                const double *p = s.part + run.base + ((k0 + q) * 3) * ps;
                bx[q] = p[0];
                by[q] = p[ps];
                bz[q] = p[2 * ps];
            }
        }
#pragma unroll
        for (int q = 0; q < SB; ++q)
            if (k0 + q < count) {
                ax += bx[q];
                ay += by[q];
                az += bz[q];
            }
    }
    if (s.corr) {
        ax += s.corr[r.gi];
        ay += s.corr[s.cap + r.gi];
        az += s.corr[2 * s.cap + r.gi];
    }
}

// A body's state and what its update reads besides the sums: a kernel that waits
// at a barrier for the sums loads them ahead (the others gain nothing by it: at
// a million bodies the registers it holds cost 2 us of 86).
struct BodyState {
    double x, y, z, vx, vy, vz, dt;
    Frame f;
};
__device__ __forceinline__ BodyState load_body(const DevState &s, int32_t k, int64_t i)
{
    BodyState b;
    b.x = s.x[i];
    b.y = s.y[i];
    b.z = s.z[i];
    b.vx = s.vx[i];
    b.vy = s.vy[i];
    b.vz = s.vz[i];
    b.dt = s.cl.dts[k];
    return b;
}

// One body's update: kick (KICK) by (ax, ay, az) plus the field, drift, split
// (AHEAD: in the frame loaded with the state).  TWO: the first half drift of the
// next step may follow (wd2 not zero; FP64 only, the others take a frame between
// steps).  What a launch does is fixed at compile time where it can be: every
// double-precision operation, comparisons included, costs a set of a million
// bodies 2 us.
template <bool EXT, bool KICK, bool TWO, bool AHEAD, bool SYM>
__device__ __forceinline__ void advance(const DevState &s, const BodyState &b, int32_t k, int64_t i,
                                        double ax, double ay, double az, double wk, double wd,
                                        double wd2, int do_split, const ExtField &ext)
{
    const double dt = b.dt;
    double x = b.x, y = b.y, z = b.z, vx = b.vx, vy = b.vy, vz = b.vz;
    if (KICK) {
        if (EXT) field_accel(ext, x, y, z, ax, ay, az);
        const double hk = wk * dt;
        vx = moved(hk, ax, vx);
        vy = moved(hk, ay, vy);
        vz = moved(hk, az, vz);
        s.vx[i] = vx;
        s.vy[i] = vy;
        s.vz[i] = vz;
    }
    const double hd = wd * dt;
    x = moved(hd, vx, x);
    y = moved(hd, vy, y);
    z = moved(hd, vz, z);
    if (TWO && wd2 != 0.0) {
        const double h2 = wd2 * dt;
        x = moved(h2, vx, x);
        y = moved(h2, vy, y);
        z = moved(h2, vz, z);
    }
    s.x[i] = x;
    s.y[i] = y;
    s.z[i] = z;
    const Frame &f = AHEAD ? b.f : s.cl.frame[k];
    // 1: coordinates, 2: and masses, 3: planes only (the symmetric kernels read no
    // more).  A branch of its own for each decomposition: with all three in one
    // kernel the stores of a million bodies took 78 us instead of 57
    if (SYM) {
        if (do_split) split_one<false, false>(s, f, i, x, y, z);
    } else if (do_split == 2) {
        split_one<true>(s, f, i, x, y, z);
    } else if (do_split) {
        split_one<false>(s, f, i, x, y, z);
    }
}

// A drift alone.
template <bool SYM>
__global__ void drift_kernel(DevState s, double wd, int do_split, int64_t t0, int64_t t1)
{
    const int64_t t = t0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= t1) return;
    const BodyRef r = body_at(s.cl, t);
    advance<false, false, false, false, SYM>(s, load_body(s, r.k, r.gi), r.k, r.gi, 0.0, 0.0, 0.0,
                                             0.0, wd, 0.0, do_split, ExtField());
}

// EXT: the external field is on (a separate variant keeps its registers out
// of the field-free kick).
template <bool EXT, int SB, bool FP, bool SYM>
__global__ void kick_drift_kernel(DevState s, Decomp dd, double wk, double wd, double wd2,
                                  int do_split, ExtField ext, int64_t t0, int64_t t1)
{
    const int64_t t = t0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= t1) return;
    Decomp d = dd;
    d.sym = SYM ? 1 : 0;   // the other decomposition's indexing costs registers
    const BodyRef r = body_at(s.cl, t);
    double ax, ay, az;
    sum_slots<SB, FP>(s, d, r, t, ax, ay, az);
    advance<EXT, true, !FP, false, SYM>(s, load_body(s, r.k, r.gi), r.k, r.gi, ax, ay, az, wk, wd,
                                        wd2, do_split, ext);
}

// The sums with a warp per run of slots, 32 bodies per block: true, and the
// sums, in the first warp.
template <int NP, bool FP, typename Ahead>
__device__ __forceinline__ bool split_sum(const DevState &s, const Decomp &d, int64_t t,
                                          int64_t t1, BodyRef &r, Ahead ahead, double &ax,
                                          double &ay, double &az)
{
    __shared__ SlotSum<FP> part[NP - 1][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    SlotSum<FP> a;
    double cx = 0.0, cy = 0.0, cz = 0.0;
    bool heavy = false;
    if (t < t1) {
        r = body_at(s.cl, t);
        if (w == 0) {
            ahead(r);
            heavy = is_heavy<FP>(s, d, t);
            if (s.corr) {
                cx = s.corr[r.gi];
                cy = s.corr[s.cap + r.gi];
                cz = s.corr[2 * s.cap + r.gi];
            }
        }
        const SlotRun run = slot_run(d, s.cl, r.k, r.li, t, s.pstride);
        const int64_t c = (run.count + NP - 1) / NP;
        const int64_t k0 = w * c, k1 = k0 + c < run.count ? k0 + c : run.count;
        a = sum_run<FP>(s, run, k0, k1);
        if (w > 0) part[w - 1][lane] = a;
    }
    __syncthreads();
    if (w > 0 || t >= t1) return false;
    for (int q = 0; q < NP - 1; ++q) a.add(part[q][lane]);
    ax = ay = az = 0.0;
    if (!heavy) a.get(ax, ay, az);
    if (s.corr) {
        ax += cx;
        ay += cy;
        az += cz;
    }
    return true;
}

// Blocks per SM that hold SUM_WARPS warps.
template <bool EXT, int NP, bool FP, bool SYM>
__global__ void __launch_bounds__(32 * NP, SUM_WARPS / NP) kick_split_kernel(
    DevState s, Decomp dd, double wk, double wd, double wd2, int do_split, ExtField ext, int64_t t0,
    int64_t t1)
{
    const int64_t t = t0 + blockIdx.x * (int64_t)32 + (threadIdx.x & 31);
    Decomp d = dd;
    d.sym = SYM ? 1 : 0;
    BodyRef r{};
    BodyState b{};
    double ax, ay, az;
    if (split_sum<NP, FP>(
            s, d, t, t1, r,
            [&](const BodyRef &q) {
                b = load_body(s, q.k, q.gi);
                if (do_split) b.f = s.cl.frame[q.k];
            },
            ax, ay, az))
        advance<EXT, true, !FP, true, SYM>(s, b, r.k, r.gi, ax, ay, az, wk, wd, wd2, do_split, ext);
}

// Blocks of at most 128 threads: with ~100 registers a thread, 128-thread
// blocks pack 20 warps on an SM against 16 for 256 (the kick waits on memory;
// the ensemble's kick ran 8% faster).
static cudaError_t kick_drift(const DevState &s, const Decomp &d, double wk, double wd, double wd2,
                              int do_kick, int do_split, const ExtField &ext, int64_t t0,
                              int64_t t1, cudaStream_t st)
{
    if (t1 <= t0) return cudaSuccess;
    const int64_t m = t1 - t0;
    const int t = ot_for(m) < 128 ? ot_for(m) : 128;
    const unsigned nb = blocks_for(m, t);
    if (!do_kick) {
        if (d.sym)
            drift_kernel<true><<<nb, t, 0, st>>>(s, wd, do_split, t0, t1);
        else
            drift_kernel<false><<<nb, t, 0, st>>>(s, wd, do_split, t0, t1);
        return cudaGetLastError();
    }
    const int parts = slot_parts(d, s.n);
    if (parts > 1) {
        const unsigned ns = blocks_for(m, 32);
#define NB_KS(E, P, F, S) kick_split_kernel<E, P, F, S><<<ns, 32 * P, 0, st>>>(s, d, wk, wd, wd2, do_split, ext, t0, t1)
#define NB_KP(E, F, S) \
    if (parts == 8) NB_KS(E, 8, F, S); else if (parts == 4) NB_KS(E, 4, F, S); else NB_KS(E, 2, F, S)
#define NB_KE(F, S) \
    if (ext.on) { NB_KP(true, F, S); } else { NB_KP(false, F, S); }
        if (d.fpart && d.sym) {
            NB_KE(true, true)
        } else if (d.fpart) {
            NB_KE(true, false)
        } else if (d.sym) {
            NB_KE(false, true)
        } else {
            NB_KE(false, false)
        }
#undef NB_KE
#undef NB_KP
#undef NB_KS
        return cudaGetLastError();
    }
    const bool narrow = d.slots <= 4;   // every i-block has at most 4 slots
#define NB_KD(E, B, F, S) kick_drift_kernel<E, B, F, S><<<nb, t, 0, st>>>(s, d, wk, wd, wd2, do_split, ext, t0, t1)
#define NB_KB(E, F, S) \
    if (narrow) NB_KD(E, 4, F, S); else NB_KD(E, 8, F, S)
    if (d.fpart && d.sym) {
        if (ext.on) { NB_KB(true, true, true); } else { NB_KB(false, true, true); }
    } else if (d.fpart) {
        if (ext.on) { NB_KB(true, true, false); } else { NB_KB(false, true, false); }
    } else if (d.sym) {
        if (ext.on) { NB_KB(true, false, true); } else { NB_KB(false, false, true); }
    } else {
        if (ext.on) { NB_KB(true, false, false); } else { NB_KB(false, false, false); }
    }
#undef NB_KB
#undef NB_KD
    return cudaGetLastError();
}

cudaError_t launch_kick_drift(const DevState &s, const Decomp &d, double wk, double wd,
                              int do_kick, int do_split, const ExtField &ext, cudaStream_t st,
                              double wd2)
{
    return kick_drift(s, d, wk, wd, wd2, do_kick, do_split, ext, 0, s.n, st);
}

cudaError_t launch_kick_drift_range(const DevState &s, const Decomp &d, double wk, double wd,
                                    int do_kick, int do_split, const ExtField &ext, int64_t t0,
                                    int64_t t1, cudaStream_t st)
{
    return kick_drift(s, d, wk, wd, 0.0, do_kick, do_split, ext, t0, t1, st);
}

// Loads the code of the kernels of a field-free step (a kernel's first launch
// otherwise does, and waits for it).
cudaError_t load_step_kernels()
{
    const void *all[] = {
        (const void *)frame_partial_kernel, (const void *)frame_final_kernel,
        (const void *)frame_harmonic_kernel, (const void *)frame_scale_kernel,
        (const void *)drift_kernel<true>, (const void *)drift_kernel<false>,
        (const void *)unpack_kernel, (const void *)pack_kernel, (const void *)cluster_map_kernel,
#define NB_LD(F, S)                                                                              \
    (const void *)kick_drift_kernel<false, 4, F, S>,                                             \
        (const void *)kick_drift_kernel<false, 8, F, S>,                                         \
        (const void *)kick_split_kernel<false, 2, F, S>,                                         \
        (const void *)kick_split_kernel<false, 4, F, S>,                                         \
        (const void *)kick_split_kernel<false, 8, F, S>
        NB_LD(true, true), NB_LD(true, false), NB_LD(false, true), NB_LD(false, false)
#undef NB_LD
    };
    for (const void *f : all) {
        cudaFuncAttributes at;
        const cudaError_t e = cudaFuncGetAttributes(&at, f);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Row q of the output: the internal sum plus the field at the body.
__device__ __forceinline__ void put_accel(const DevState &s, const ExtField &ext, int64_t gi,
                                          int64_t q, double ax, double ay, double az,
                                          double *__restrict__ out)
{
    if (ext.on) field_accel(ext, s.x[gi], s.y[gi], s.z[gi], ax, ay, az);
    out[3 * q] = ax;
    out[3 * q + 1] = ay;
    out[3 * q + 2] = az;
    if (!isfinite(ax) || !isfinite(ay) || !isfinite(az)) atomicOr(s.flag, 1);
}

template <bool FP, bool SYM>
__global__ void accel_out_kernel(DevState s, Decomp dd, ExtField ext, double *__restrict__ out,
                                 int64_t t0, int64_t t1)
{
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t t = t0 + q;
    if (t >= t1) return;
    Decomp d = dd;
    d.sym = SYM ? 1 : 0;   // as in kick_drift_kernel
    const BodyRef r = body_at(s.cl, t);
    double ax, ay, az;
    sum_slots<8, FP>(s, d, r, t, ax, ay, az);
    put_accel(s, ext, r.gi, q, ax, ay, az, out);
}

template <int NP, bool FP, bool SYM>
__global__ void __launch_bounds__(32 * NP, SUM_WARPS / NP) accel_split_kernel(
    DevState s, Decomp dd, ExtField ext, double *__restrict__ out, int64_t t0, int64_t t1)
{
    const int64_t q = blockIdx.x * (int64_t)32 + (threadIdx.x & 31);
    Decomp d = dd;
    d.sym = SYM ? 1 : 0;
    BodyRef r{};
    double ax, ay, az;
    if (split_sum<NP, FP>(s, d, t0 + q, t1, r, [](const BodyRef &) {}, ax, ay, az))
        put_accel(s, ext, r.gi, q, ax, ay, az, out);
}

cudaError_t launch_accel_out(const DevState &s, const Decomp &d, const ExtField &ext,
                             double *out_aos, cudaStream_t st)
{
    return launch_accel_out_range(s, d, ext, out_aos, 0, s.n, st);
}

cudaError_t launch_accel_out_range(const DevState &s, const Decomp &d, const ExtField &ext,
                                   double *out_aos, int64_t t0, int64_t t1, cudaStream_t st)
{
    const int parts = slot_parts(d, s.n);
    if (parts > 1) {
        const unsigned ns = blocks_for(t1 - t0, 32);
#define NB_AS(P, F, S) accel_split_kernel<P, F, S><<<ns, 32 * P, 0, st>>>(s, d, ext, out_aos, t0, t1)
#define NB_AP(F, S) \
    if (parts == 8) NB_AS(8, F, S); else if (parts == 4) NB_AS(4, F, S); else NB_AS(2, F, S)
        if (d.fpart) {
            if (d.sym) { NB_AP(true, true); } else { NB_AP(true, false); }
        } else {
            if (d.sym) { NB_AP(false, true); } else { NB_AP(false, false); }
        }
#undef NB_AP
#undef NB_AS
        return cudaGetLastError();
    }
    const int t = ot_for(t1 - t0);
    const unsigned nb = blocks_for(t1 - t0, t);
#define NB_AO(F, S) accel_out_kernel<F, S><<<nb, t, 0, st>>>(s, d, ext, out_aos, t0, t1)
    if (d.fpart) {
        if (d.sym) NB_AO(true, true); else NB_AO(true, false);
    } else {
        if (d.sym) NB_AO(false, true); else NB_AO(false, false);
    }
#undef NB_AO
    return cudaGetLastError();
}

// ---- diagnostics -------------------------------------------------------------

// Per segment: K, sum m_i phi_i, W_ext, P, L, non-finite count (10 values).
// d is the potential kernel's decomposition (s.cl.uoff and poff must be its).
__global__ void energy_partial_kernel(DevState s, Decomp d, ExtField ext)
{
    __shared__ double sh[10 * RT];
    const int sg = blockIdx.x;
    const int32_t k = s.cl.seg_k[sg];
    double v[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t t = s.cl.seg_lo[sg] + threadIdx.x; t < s.cl.seg_hi[sg]; t += RT) {
        BodyRef r;
        r.k = k;
        r.li = t - s.cl.noff[k];
        r.gi = s.cl.boff[k] + r.li;
        const int64_t i = r.gi;
        const double m = s.m[i], x = s.x[i], y = s.y[i], z = s.z[i];
        const double vx = s.vx[i], vy = s.vy[i], vz = s.vz[i];
        const SlotRun run = slot_run(d, s.cl, k, r.li, t, s.pstride);
        const int64_t count = run.count;
        double phi = 0.0;
        for (int64_t q0 = 0; q0 < count; q0 += 8) {
            double bp[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                bp[q] = q0 + q < count ? s.part[run.base + ((q0 + q) * 3) * run.stride] : 0.0;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q0 + q < count) phi += bp[q];
        }
        v[0] += 0.5 * m * (vx * vx + vy * vy + vz * vz);
        v[1] += m * phi;
        if (ext.on) v[2] += m * field_phi(ext, x, y, z);
        v[3] += m * vx;
        v[4] += m * vy;
        v[5] += m * vz;
        v[6] += m * (y * vz - z * vy);
        v[7] += m * (z * vx - x * vz);
        v[8] += m * (x * vy - y * vx);
        if (!isfinite(phi) || !isfinite(x) || !isfinite(y) || !isfinite(z) || !isfinite(vx) ||
            !isfinite(vy) || !isfinite(vz))
            v[9] += 1.0;
    }
    block_sum<10>(v, sh);
    if (threadIdx.x == 0)
        for (int q = 0; q < 10; ++q) s.red[(int64_t)sg * 16 + q] = v[q];
}

__global__ void energy_final_kernel(DevState s, double G)
{
    __shared__ double sh[10 * RT];
    double v[10];
    cluster_sum<10>(s, v, sh);
    if (threadIdx.x == 0) {
        double *o = s.diag + (int64_t)blockIdx.x * DIAG_STRIDE;
        const double W = -G * v[1];   // each unordered pair once
        o[0] = v[0];
        o[1] = W;
        o[2] = v[2];
        o[3] = v[0] + W + v[2];
        for (int q = 0; q < 6; ++q) o[4 + q] = v[3 + q];
        if (v[9] != 0.0 || !isfinite(o[3])) atomicOr(s.flag, 1);
    }
}

cudaError_t launch_energy_reduce(const DevState &s, const Decomp &d, const ExtField &ext,
                                 double G, cudaStream_t st)
{
    energy_partial_kernel<<<s.cl.S, RT, 0, st>>>(s, d, ext);
    energy_final_kernel<<<s.cl.K, RT, 0, st>>>(s, G);
    return cudaGetLastError();
}

// External torque of eq. 8: sum m_i r_i x a_ext(r_i), per cluster.
__global__ void torque_partial_kernel(DevState s, ExtField ext)
{
    __shared__ double sh[3 * RT];
    const int sg = blockIdx.x;
    const int32_t k = s.cl.seg_k[sg];
    const int64_t base = s.cl.boff[k] - s.cl.noff[k];
    double v[3] = {0, 0, 0};
    for (int64_t t = s.cl.seg_lo[sg] + threadIdx.x; t < s.cl.seg_hi[sg]; t += RT) {
        const int64_t i = base + t;
        const double m = s.m[i], x = s.x[i], y = s.y[i], z = s.z[i];
        double ax = 0.0, ay = 0.0, az = 0.0;
        field_accel(ext, x, y, z, ax, ay, az);
        v[0] += m * (y * az - z * ay);
        v[1] += m * (z * ax - x * az);
        v[2] += m * (x * ay - y * ax);
    }
    block_sum<3>(v, sh);
    if (threadIdx.x == 0)
        for (int q = 0; q < 3; ++q) s.red[(int64_t)sg * 16 + q] = v[q];
}

__global__ void torque_final_kernel(DevState s)
{
    __shared__ double sh[3 * RT];
    double v[3];
    cluster_sum<3>(s, v, sh);
    if (threadIdx.x == 0)
        for (int q = 0; q < 3; ++q) s.diag[(int64_t)blockIdx.x * DIAG_STRIDE + 10 + q] = v[q];
}

cudaError_t launch_torque(const DevState &s, const ExtField &ext, cudaStream_t st)
{
    torque_partial_kernel<<<s.cl.S, RT, 0, st>>>(s, ext);
    torque_final_kernel<<<s.cl.K, RT, 0, st>>>(s);
    return cudaGetLastError();
}

}  // namespace nb
