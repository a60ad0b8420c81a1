// near.cu -- near-pair correction of the mixed-precision pair sum (NB_DS).
//
// The mixed pair kernel evaluates every pair in float on coordinates taken
// relative to the cluster's frame origin c (hi = fl(x - c)).  For pairs
// closer than the near radius d_th the rounding of hi dominates the error of
// the coordinate difference (Sect. 5.2's "delicate evaluation of coordinate
// difference"), so this pass finds them with a spatial grid and adds, per
// body i,
//     corr_i = G sum_{j near i, j != i} [ f(d_ij^ds) - f(d_ij^float) ]
// where d^ds = (hi_j - hi_i) + (lo_j - lo_i) is the double-single difference
// and f(d^float) is recomputed with exactly the operations of the pair
// kernel, so it cancels that kernel's float contribution to within the
// rounding of its running sum.  Cells carry the cluster index, so bodies of
// different clusters never pair.
//
// Grid: cubic cells of side h = CELL_SCALE d_th.  Since h > 2 d_th, the
// d_th-ball around a body reaches, along each axis, only its own cell and the
// neighbour on the side of the cell half the body sits in, so each body looks
// at 2 x 2 x 2 cells.  The 10% margin in CELL_SCALE absorbs the float rounding
// of x / h for every cell coordinate the key can hold.  Occupied cells live
// in an open-addressing table (linear probing, at most one cell per four
// slots, so that probes for the many empty neighbour cells end fast) whose
// slot records carry the cell's range in a cell-ordered copy of
// the bodies, so a probe costs one 16-byte load and never walks another
// cell's bodies.  Each cluster k owns the slots [4 noff[k], 4 noff[k+1]):
// its bodies' probes stay in a region proportional to its size (cache
// locality for ensembles of small clusters), and probing wraps inside it.  Near pairs are rare (a few tenths per body in a Plummer
// sphere), so the pass is dominated by these probes.
//
// Pass: clear the table (one memset), insert cells and count arrivals, let
// each cell's first arrival claim its range of the cell-ordered copies (one
// atomic add on a running total), scatter, order each cell by body index and
// write the copies, correct.
//
// On the way each body's strongest single pull decides whether it is in a
// close encounter (Heavy, nb_internal.cuh).
//
// Deterministic: within a cell the bodies are ordered by linear index, and
// every body visits its 8 cells in a fixed order, so the FP64 correction sums
// do not depend on timing (which slot a cell lands in, and where its range
// lands, may vary; the sums do not depend on either).
#include "arith.cuh"
#include "nb_internal.cuh"
#include "split.cuh"

namespace nb {

__device__ __forceinline__ float near_rsqrt(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

constexpr int CELL_BITS = 15;                 // per coordinate
constexpr int CELL_OFF = 1 << (CELL_BITS - 1);
constexpr int CELL_MAX = CELL_OFF - 2;        // |cell| <= CELL_MAX, neighbours <= CELL_OFF - 1
constexpr float CELL_SCALE = 2.2f;            // h / d_th
constexpr unsigned long long NG_EMPTY = ~0ull;

__device__ __forceinline__ uint64_t cell_key(int32_t k, int cx, int cy, int cz)
{
    return ((uint64_t)(uint32_t)k << (3 * CELL_BITS)) |
           ((uint64_t)(cx + CELL_OFF) << (2 * CELL_BITS)) |
           ((uint64_t)(cy + CELL_OFF) << CELL_BITS) | (uint64_t)(cz + CELL_OFF);
}

// Region of cluster k's cells in the slot table.
constexpr int SLOTS_PER_BODY = 4;

struct Region {
    int64_t base;   // first slot
    uint32_t size;  // slots (SLOTS_PER_BODY n_k)
};

__device__ __forceinline__ Region region_of(const Clusters &c, int32_t k)
{
    Region r;
    r.base = SLOTS_PER_BODY * c.noff[k];
    r.size = (uint32_t)(SLOTS_PER_BODY * c.nk[k]);
    return r;
}

// Multiplicative (Fibonacci) hash of the key (the middle bits of
// key * 2^64/phi), reduced to the region by a multiply-shift.
__device__ __forceinline__ int64_t slot_of(uint64_t key, const Region &r)
{
    const uint32_t h = (uint32_t)((key * 0x9E3779B97F4A7C15ull) >> 32);
    return r.base + (int64_t)(((uint64_t)h * r.size) >> 32);
}

// Next slot of the linear probe, wrapping inside the region.
__device__ __forceinline__ int64_t next_slot(int64_t b, const Region &r)
{
    return b + 1 == r.base + r.size ? r.base : b + 1;
}

// Cell coordinate of v (clamped to the key's range) and the side, -1 or +1,
// of the neighbour its d_th-interval can reach.
__device__ __forceinline__ int cell_coord(float v, float inv_h, int &side)
{
    const float q = v * inv_h;
    const float f = floorf(q);
    side = q - f < 0.5f ? -1 : 1;
    return (int)fminf(fmaxf(f, -(float)CELL_MAX), (float)CELL_MAX);
}

// Per body: the cell key, insertion of the cell into the slot table and the
// body's rank among its cell's arrivals.
// LIST (where a kernel for close encounters follows): the cell's bodies form a
// list instead (the slot's end its head, ng_entry the links), from which the
// claim pass takes each body's rank by index, so no scatter pass is needed;
// the lists are short (at most ~10 bodies in the core of a Plummer sphere).
template <bool LIST>
__global__ void near_cell_kernel(DevState s)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= s.n) return;
    if (LIST && t < hv_limit(s.n)) s.hv_done[t] = 0;
    if (t == 0) {
        *s.ng_total = 0;   // read only by the claim pass, which follows
        if (s.hv_count) *s.hv_count = 0;
    }
    const int32_t k = cluster_of(s.cl, t);
    const int64_t i = s.cl.boff[k] + t - s.cl.noff[k];
    const float dth = s.cl.frame[k].dth;
    if (!(dth > 0.f)) {   // no pair can pass the test r^2 + eps^2 < eps^2
        s.ng_bucket[t] = -1;
        return;
    }
    const float ih = 1.0f / (CELL_SCALE * dth);
    int sx, sy, sz;
    const int cx = cell_coord(s.xh[i], ih, sx), cy = cell_coord(s.yh[i], ih, sy),
              cz = cell_coord(s.zh[i], ih, sz);
    const uint64_t key = cell_key(k, cx, cy, cz);
    // the region has more slots than the cluster has bodies, so a free or
    // matching slot always exists; the bound only caps the loop
    const Region rg = region_of(s.cl, k);
    int64_t b = slot_of(key, rg);
    for (uint32_t p = 0; p < rg.size; ++p) {
        const unsigned long long prev = atomicCAS(&s.ng_slot[b].key, NG_EMPTY, key);
        if (prev == NG_EMPTY || prev == key) break;
        b = next_slot(b, rg);
    }
    s.ng_bucket[t] = (int)b;
    if (LIST) {
        s.ng_entry[t] = atomicExch(&s.ng_slot[b].end, (int)t);   // -1 (empty): the list's end
        return;
    }
    // the slot's end counts arrivals from -1 (the empty record) until the
    // claim pass turns it into the range end
    s.ng_rank[t] = atomicAdd(&s.ng_slot[b].end, 1) + 1;
}

// After all insertions: the first arrival of each cell claims the cell's
// range of the cell-ordered copies.  A block sums its claims (warp-shuffle
// scan, then across the warps) and takes one range of the running total with
// a single atomic add; a claim per atomic on one address would serialise.
// Ranges land in the order the blocks claim them; only their contents,
// ordered by body index, enter the sums.  The slot keeps [start, end).
// LIST: the body of the cell's least index claims, and each body's rank is the
// number of lesser indices; the claiming body's is kept as minus the cell's
// count, for the copy pass.
constexpr int CLAIM_T = 256;

template <bool LIST>
__global__ void __launch_bounds__(CLAIM_T) near_claim_kernel(DevState s)
{
    __shared__ int wsum[CLAIM_T / 32];
    __shared__ int base;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int b = -1, cnt = 0;
    if (t < s.n) {
        b = s.ng_bucket[t];
        if (LIST && b >= 0) {
            int r = 0;
            for (int e = s.ng_slot[b].end; e >= 0; e = s.ng_entry[e]) {
                ++cnt;
                r += e < (int)t ? 1 : 0;
            }
            s.ng_rank[t] = r > 0 ? r : -cnt;
            if (r > 0) {
                b = -1;
                cnt = 0;
            }
        } else if (b >= 0 && s.ng_rank[t] == 0)
            cnt = s.ng_slot[b].end + 1;   // arrivals counted from -1
        else
            b = -1;
    }
    int x = cnt;   // inclusive scan over the warp
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        int run = 0;
        for (int q = 0; q < CLAIM_T / 32; ++q) {
            const int v = wsum[q];
            wsum[q] = run;
            run += v;
        }
        base = run > 0 ? atomicAdd(s.ng_total, run) : 0;
    }
    __syncthreads();
    if (b >= 0) {
        const int st = base + wsum[w] + x - cnt;
        s.ng_slot[b].start = st;
        if (!LIST) s.ng_slot[b].end = st + cnt;
    }
}

// Bodies into their cell's range, in arrival order.
__global__ void near_scatter_kernel(DevState s)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= s.n) return;
    const int b = s.ng_bucket[t];
    if (b < 0) return;
    s.ng_entry[s.ng_slot[b].start + s.ng_rank[t]] = (int)t;
}

// Final place of each body in its cell = number of cell members with a
// smaller linear index; writes the cell-ordered copies of its float planes
// (lo.w = t) and, from the cell's first body, the slot's range.  Bodies
// outside the grid get their (zero) correction here.  LIST: the place is known,
// and the cell's first body leaves the range's end in the slot.
template <bool LIST>
__global__ void near_rank_kernel(DevState s)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= s.n) return;
    const int b = s.ng_bucket[t];
    const int32_t k = cluster_of(s.cl, t);
    const int64_t i = s.cl.boff[k] + t - s.cl.noff[k];
    if (b < 0) {   // not in the grid (no near radius): no correction
        if (s.hv_flag) s.hv_flag[t] = 0;
        s.corr[i] = 0.0;
        s.corr[s.cap + i] = 0.0;
        s.corr[2 * s.cap + i] = 0.0;
        return;
    }
    const int lo = s.ng_slot[b].start;
    int r = 0;
    if (LIST) {
        r = s.ng_rank[t];
        if (r < 0) {
            s.ng_slot[b].end = lo - r;
            r = 0;
        }
    } else {
        const int hi = s.ng_slot[b].end;
        for (int e = lo; e < hi; ++e) r += s.ng_entry[e] < (int)t ? 1 : 0;
    }
    s.ng_spos[lo + r] = make_float4(s.xh[i], s.yh[i], s.zh[i], s.mf[i]);
    s.ng_slo[lo + r] = make_float4(s.xl[i], s.yl[i], s.zl[i], __int_as_float((int)t));
}

// One thread per body in cell order (entry e of the cell-ordered copies), so
// that the threads of a warp share cells, probes and member lists: probe its
// 8 cells (first loads issued together), then visit their bodies in cell
// order.  The cell and side are recomputed from the copy's float position
// with the cell kernel's arithmetic.  Bodies outside the grid got a zero
// correction from near_rank_kernel.  UM: the pair kernel left the common
// mass out of the pair term (multiplying its sums by it afterwards); the
// correction repeats exactly that and scales by the cluster's mass.
constexpr int NC_T = 256;   // threads per block of the correction

// HEAVY: bodies in a close encounter are listed.
template <bool UM, bool HEAVY>
__global__ void __launch_bounds__(NC_T) near_correct_kernel(DevState s, double G)
{
    // per thread: the ranges of its 8 probed cells (empty: start = end), so
    // that one flat loop walks all its candidates; a loop per cell would
    // run as long as the warp's longest member list for every cell
    __shared__ int2 rng[8][NC_T];
    const int tid = threadIdx.x;
    const int64_t e0 = blockIdx.x * (int64_t)blockDim.x + tid;
    if (e0 >= *s.ng_total) return;   // bodies in the grid
    const float4 P = s.ng_spos[e0];
    const float4 Lo = s.ng_slo[e0];
    const int t = __float_as_int(Lo.w);
    const int32_t k = cluster_of(s.cl, t);
    double ax = 0.0, ay = 0.0, az = 0.0;
    int total = 0;
    {
        const float ih = 1.0f / (CELL_SCALE * s.cl.frame[k].dth);
        int sx, sy, sz;
        const int cx = cell_coord(P.x, ih, sx), cy = cell_coord(P.y, ih, sy),
                  cz = cell_coord(P.z, ih, sz);
        const Region rg = region_of(s.cl, k);
        uint64_t key[8];
        int64_t slot[8];
        NgSlot v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            key[q] = cell_key(k, cx + (q & 1 ? sx : 0), cy + (q & 2 ? sy : 0),
                              cz + (q & 4 ? sz : 0));
            slot[q] = slot_of(key[q], rg);
            v[q] = s.ng_slot[slot[q]];
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            NgSlot c = v[q];
            int64_t b = slot[q];
            for (uint32_t p = 1; p < rg.size && c.key != key[q] && c.key != NG_EMPTY; ++p) {
                b = next_slot(b, rg);
                c = s.ng_slot[b];
            }
            const bool hit = c.key == key[q];
            rng[q][tid] = hit ? make_int2(c.start, c.end) : make_int2(0, 0);
            total += hit ? c.end - c.start : 0;
        }
    }
    const float eps2 = s.cl.eps2f[k];
    const float th2 = s.cl.frame[k].th2;
    float pull = 0.f;   // largest m_j / (r^2 + eps^2) met
    const float xi = P.x, yi = P.y, zi = P.z;
    const float lxi = Lo.x, lyi = Lo.y, lzi = Lo.z;
    // candidates in cell order 0..7, each cell's members in body order,
    // NBT at a time: their indices are resolved first, so their position
    // loads are in flight together; only the few candidates inside the near
    // radius load their lo words (one candidate in twenty on a Plummer
    // sphere).  The body itself is the candidate at its own cell-ordered
    // position e0.
    constexpr int NBT = 4;
    int q = 0;
    int2 r = rng[0][tid];
    int e = r.x;
    for (int it = 0; it < total; it += NBT) {
        int ee[NBT];
#pragma unroll
        for (int b = 0; b < NBT; ++b) {
            ee[b] = -1;
            if (it + b < total) {
                while (e >= r.y) {
                    r = rng[++q][tid];
                    e = r.x;
                }
                ee[b] = e++;
            }
        }
        float4 Pb[NBT];
#pragma unroll
        for (int b = 0; b < NBT; ++b)
            Pb[b] = s.ng_spos[ee[b] >= 0 ? ee[b] : e0];
#pragma unroll
        for (int b = 0; b < NBT; ++b) {
            if (ee[b] < 0) break;
            const float4 Pj = Pb[b];
            // the pair kernel's float contribution, operation for operation
            const float mj = Pj.w;
            const float ddx = __fadd_rn(Pj.x, -xi);
            const float ddy = __fadd_rn(Pj.y, -yi);
            const float ddz = __fadd_rn(Pj.z, -zi);
            float r2 = __fmaf_rn(ddx, ddx, eps2);
            r2 = __fmaf_rn(ddy, ddy, r2);
            r2 = __fmaf_rn(ddz, ddz, r2);
            if (ee[b] == (int)e0 || !(r2 < th2)) continue;
            const float4 Lj = s.ng_slo[ee[b]];
            const float ri = near_rsqrt(r2);
            const float sf = UM ? __fmul_rn(ri, __fmul_rn(ri, ri))
                                : __fmul_rn(__fmul_rn(mj, ri), __fmul_rn(ri, ri));
            // the same pair with the double-single coordinate difference
            const float ex = __fadd_rn(ddx, __fsub_rn(Lj.x, lxi));
            const float ey = __fadd_rn(ddy, __fsub_rn(Lj.y, lyi));
            const float ez = __fadd_rn(ddz, __fsub_rn(Lj.z, lzi));
            float e2 = __fmaf_rn(ex, ex, eps2);
            e2 = __fmaf_rn(ey, ey, e2);
            e2 = __fmaf_rn(ez, ez, e2);
            const float re = near_rsqrt(e2);
            if (HEAVY) pull = fmaxf(pull, mj * re * re);
            const float se = UM ? __fmul_rn(re, __fmul_rn(re, re))
                                : __fmul_rn(__fmul_rn(mj, re), __fmul_rn(re, re));
            ax += (double)__fmul_rn(ex, se) - (double)__fmul_rn(ddx, sf);
            ay += (double)__fmul_rn(ey, se) - (double)__fmul_rn(ddy, sf);
            az += (double)__fmul_rn(ez, se) - (double)__fmul_rn(ddz, sf);
        }
    }
    const int64_t i = s.cl.boff[k] + t - s.cl.noff[k];
    if (HEAVY) {
        const bool heavy = pull > s.cl.frame[k].hx;
        s.hv_flag[t] = heavy ? 1 : 0;
        if (heavy) {
            const int q = atomicAdd(s.hv_count, 1);
            if (q < hv_limit(s.n)) s.hv_list[q] = t;
        }
    }
    const double Gm = UM ? G * s.cl.mu[k] : G;
    s.corr[i] = Gm * ax;
    s.corr[s.cap + i] = Gm * ay;
    s.corr[2 * s.cap + i] = Gm * az;
}

// ---- bodies in a close encounter (Heavy) ----------------------------------------
// Each listed body's internal acceleration as the full single-precision kernel
// and the kick give it, near-pair correction included, into corr: the float
// partial sums over 512 j bodies of every block of the full decomposition, each
// in j order, then the blocks' double-single sums, scaled, and their sum in
// block order.  A block takes HVG partial sums of one body: its threads form
// their pair terms HVS j at a time (a warp 32 consecutive j of a plane, the next
// slice's loads in flight) and stage them in shared memory, from where one
// thread per partial sum adds its terms in order; the body's last block to
// finish adds up.  What bounds it is latency: 512 additions in order per partial
// sum, in 16 slices of one load latency each.
constexpr int HVT = 256;       // threads per block
constexpr int HVG = HV_PART;   // partial sums per block
constexpr int HVS = 32;        // j bodies per slice
constexpr int HVK = HVG * HVS / HVT;

// The runs of body t's row in the full decomposition: j range of run sg and its
// number of partial sums.
struct HeavyRow {
    int64_t u0, u1, first;
    int nseg;
    __device__ __forceinline__ HeavyRow(const Decomp &f, int64_t nt, int64_t t)
    {
        u0 = (t / f.ipb) * nt;
        u1 = u0 + nt;
        first = f.owner(u0);
        nseg = (int)(f.owner(u1 - 1) - first) + 1;   // <= f.slots <= MAX_PART_SLOTS
    }
    __device__ __forceinline__ int range(const Decomp &f, int64_t n, int sg, int &J0, int &J1) const
    {
        const int64_t ua = f.U(first + sg), ub = f.U(first + sg + 1);
        const int64_t a = ua > u0 ? ua : u0, b = ub < u1 ? ub : u1;
        const int64_t jend = (n + 31) & ~(int64_t)31;
        J0 = (int)((a - u0) * f.jt);
        J1 = (int)((b - u0) * f.jt < jend ? (b - u0) * f.jt : jend);
        return J1 > J0 ? (J1 - J0 + 4 * TILE - 1) / (4 * TILE) : 0;
    }
};

__global__ void __launch_bounds__(HVT) near_encounter_kernel(DevState s, Heavy h, double Gm, int um)
{
    constexpr int FOLD = 4 * TILE;
    __shared__ float4 term[HVG][HVS + 1];
    __shared__ int2 grp[HVG];                        // j range of each partial sum
    __shared__ int seg0[MAX_PART_SLOTS + 2];         // first partial sum of each block's run
    __shared__ float2 segsum[3][MAX_PART_SLOTS + 1];
    __shared__ bool last;
    const int tid = threadIdx.x;
    const int cnt = *s.hv_count;
    if (cnt > hv_limit(s.n)) return;
    const Decomp &f = h.full;
    const int64_t n = s.cl.nk[0], base = s.cl.boff[0];
    const int64_t nt = f.units_per_iblock(s.cl.ntiles[0]);
    const float eps2 = s.cl.eps2f[0];
    const float gh = __double2float_rn(Gm), gl = __double2float_rn(Gm - (double)gh);
    for (int item = blockIdx.x; item < cnt * h.parts; item += gridDim.x) {
        const int q = item / h.parts, part = item - q * h.parts;
        const int t = s.hv_list[q];
        const HeavyRow row(f, nt, t);
        const int nseg = row.nseg;
        __syncthreads();   // the last item's tables have been read
        for (int sg = tid; sg < nseg; sg += HVT) {
            int J0, J1;
            seg0[sg + 1] = row.range(f, n, sg, J0, J1);
        }
        __syncthreads();
        if (tid < 32) {   // prefix sums, one warp
            int run = 0;
            for (int b0 = 0; b0 < nseg; b0 += 32) {
                int v = b0 + tid < nseg ? seg0[b0 + tid + 1] : 0;
                for (int d = 1; d < 32; d <<= 1) {
                    const int w = __shfl_up_sync(0xffffffffu, v, d);
                    if (tid >= d) v += w;
                }
                if (b0 + tid < nseg) seg0[b0 + tid + 1] = run + v;
                run += __shfl_sync(0xffffffffu, v, 31);
            }
            if (tid == 0) seg0[0] = 0;
        }
        __syncthreads();
        const int ng = seg0[nseg];
        const int g0 = part * HVG, gn = ng - g0 < HVG ? ng - g0 : HVG;   // gn <= 0: none left
        for (int sg = tid; sg < nseg; sg += HVT) {
            if (seg0[sg + 1] <= g0 || seg0[sg] >= g0 + HVG) continue;
            int J0, J1;
            row.range(f, n, sg, J0, J1);
            for (int e = seg0[sg]; e < seg0[sg + 1]; ++e) {
                const int ja = J0 + (e - seg0[sg]) * FOLD;
                const int jb = ja + FOLD < J1 ? ja + FOLD : J1;
                // padding adds exactly zero
                if (e >= g0 && e < g0 + HVG) grp[e - g0] = make_int2(ja, jb < n ? jb : (int)n);
            }
        }
        for (int e = tid; e < HVG; e += HVT)
            if (e >= gn) grp[e] = make_int2(0, 0);
        __syncthreads();
        const float xi = s.xh[base + t], yi = s.yh[base + t], zi = s.zh[base + t];
        // term k of this thread: partial sum tid / HVS + k (HVT / HVS), j body
        // tid % HVS of the slice
        const int jj = tid % HVS, gg = tid / HVS;
        int2 rk[HVK];
        float x[HVK], y[HVK], z[HVK], m[HVK];
        auto fetch = [&](int sl) {
#pragma unroll
            for (int k = 0; k < HVK; ++k) {
                const int j = rk[k].x + sl + jj;
                x[k] = y[k] = z[k] = m[k] = 0.f;
                if (j < rk[k].y) {
                    x[k] = s.xh[base + j];
                    y[k] = s.yh[base + j];
                    z[k] = s.zh[base + j];
                    if (!um) m[k] = s.mf[base + j];
                }
            }
        };
        int longest = 0;
#pragma unroll
        for (int k = 0; k < HVK; ++k) {
            rk[k] = grp[gg + k * (HVT / HVS)];
            longest = max(longest, rk[k].y - rk[k].x);
        }
        fetch(0);
        float ax = 0.f, ay = 0.f, az = 0.f;
        const int2 mine = tid < HVG ? grp[tid] : make_int2(0, 0);
        for (int sl = 0; sl < FOLD; sl += HVS) {
            if (!__syncthreads_or(sl < longest)) break;   // and the last slice's terms are added
#pragma unroll
            for (int k = 0; k < HVK; ++k) {
                const float dx = __fadd_rn(x[k], -xi);
                const float dy = __fadd_rn(y[k], -yi);
                const float dz = __fadd_rn(z[k], -zi);
                float r2 = __fmaf_rn(dx, dx, eps2);
                r2 = __fmaf_rn(dy, dy, r2);
                r2 = __fmaf_rn(dz, dz, r2);
                const float ri = rsqrt_mufu(r2);
                float sp = __fmul_rn(um ? ri : __fmul_rn(m[k], ri), __fmul_rn(ri, ri));
                if (rk[k].x + sl + jj == t) sp = 0.f;   // exactly zero for eps > 0 as well
                term[gg + k * (HVT / HVS)][jj] = make_float4(dx, dy, dz, sp);
            }
            fetch(sl + HVS);
            __syncthreads();
            if (tid < HVG) {
                const int left = mine.y - mine.x - sl;
                if (left >= HVS) {
#pragma unroll 8
                    for (int e = 0; e < HVS; ++e) {
                        const float4 v = term[tid][e];
                        ax = __fmaf_rn(v.x, v.w, ax);
                        ay = __fmaf_rn(v.y, v.w, ay);
                        az = __fmaf_rn(v.z, v.w, az);
                    }
                } else {
                    for (int e = 0; e < left; ++e) {
                        const float4 v = term[tid][e];
                        ax = __fmaf_rn(v.x, v.w, ax);
                        ay = __fmaf_rn(v.y, v.w, ay);
                        az = __fmaf_rn(v.z, v.w, az);
                    }
                }
            }
        }
        float *out = s.hv_sum + (int64_t)q * 3 * h.parts * HVG;
        if (tid < gn) {
            out[3 * (g0 + tid)] = ax;
            out[3 * (g0 + tid) + 1] = ay;
            out[3 * (g0 + tid) + 2] = az;
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) last = atomicAdd(s.hv_done + q, 1) == h.parts - 1;
        __syncthreads();
        if (!last) continue;
        __threadfence();
        for (int e = tid; e < 3 * nseg; e += HVT) {
            const int c = e / nseg, sg = e - c * nseg;
            float hi = 0.f, lo = 0.f;
            for (int g = seg0[sg]; g < seg0[sg + 1]; ++g) ds_add(hi, lo, __ldcg(out + 3 * g + c));
            const float pr = __fmul_rn(hi, gh);
            float er = __fmaf_rn(hi, gh, -pr);
            er = __fmaf_rn(hi, gl, __fmaf_rn(lo, gh, er));
            const float r = __fadd_rn(pr, er);
            segsum[c][sg] = make_float2(r, __fsub_rn(er, __fsub_rn(r, pr)));
        }
        __syncthreads();
        if (tid < 3) {
            float H = 0.f, L = 0.f;
            for (int sg = 0; sg < nseg; ++sg) ff_add(H, L, segsum[tid][sg].x, segsum[tid][sg].y);
            s.corr[tid * s.cap + base + t] += widen(H) + widen(L);
        }
    }
}

cudaError_t load_near_kernels()
{
    const void *all[] = {(const void *)near_cell_kernel<true>,
                         (const void *)near_cell_kernel<false>,
                         (const void *)near_claim_kernel<true>,
                         (const void *)near_claim_kernel<false>,
                         (const void *)near_scatter_kernel,
                         (const void *)near_rank_kernel<true>,
                         (const void *)near_rank_kernel<false>,
                         (const void *)near_correct_kernel<true, true>,
                         (const void *)near_correct_kernel<true, false>,
                         (const void *)near_correct_kernel<false, true>,
                         (const void *)near_correct_kernel<false, false>,
                         (const void *)near_encounter_kernel};
    for (const void *f : all) {
        cudaFuncAttributes at;
        const cudaError_t e = cudaFuncGetAttributes(&at, f);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

int64_t near_table_size(int64_t n)
{
    return SLOTS_PER_BODY * n;
}

template <bool UM>
static void correct(const DevState &s, double G, bool heavy, cudaStream_t st)
{
    const unsigned nb = (unsigned)((s.n + NC_T - 1) / NC_T);
    if (heavy)
        near_correct_kernel<UM, true><<<nb, NC_T, 0, st>>>(s, G);
    else
        near_correct_kernel<UM, false><<<nb, NC_T, 0, st>>>(s, G);
}

cudaError_t launch_near_correct(const DevState &s, double G, bool um, cudaStream_t st,
                                const Heavy *hv)
{
    const int64_t H = near_table_size(s.n);
    if (H > s.ng_hcap) return cudaErrorInvalidValue;
    const unsigned nbn = (unsigned)((s.n + 255) / 256);
    const bool list = hv && hv->blocks > 0 && s.hv_flag;
    if (list && s.cl.K != 1) return cudaErrorInvalidValue;
    DevState q = s;
    if (!list) q.hv_flag = nullptr;
    // empty records: key all ones, start = end = -1
    cudaError_t e = cudaMemsetAsync(s.ng_slot, 0xff, (size_t)H * sizeof(NgSlot), st);
    if (e != cudaSuccess) return e;
    if (list) {
        near_cell_kernel<true><<<nbn, 256, 0, st>>>(q);
        near_claim_kernel<true><<<nbn, CLAIM_T, 0, st>>>(q);
        near_rank_kernel<true><<<nbn, 256, 0, st>>>(q);
    } else {
        near_cell_kernel<false><<<nbn, 256, 0, st>>>(q);
        near_claim_kernel<false><<<nbn, CLAIM_T, 0, st>>>(q);
        near_scatter_kernel<<<nbn, 256, 0, st>>>(q);
        near_rank_kernel<false><<<nbn, 256, 0, st>>>(q);
    }
    if (um)
        correct<true>(q, G, list, st);
    else
        correct<false>(q, G, list, st);
    if (list) {
        // the scale as the pair kernel forms it: G, times the common mass
        near_encounter_kernel<<<hv->blocks, HVT, 0, st>>>(q, *hv, um ? G * hv->mu : G, um ? 1 : 0);
    }
    return cudaGetLastError();
}

}  // namespace nb
