// engine.cu -- state pool, cluster-set tables, launch plans and the enqueue
// functions shared by the context API and the serving loop.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "engine.h"

namespace nb {

namespace {
thread_local std::string g_err;
}

int set_error(int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

const char *last_error() { return g_err.c_str(); }

// ---- pool --------------------------------------------------------------------

int device_sms(int device)
{
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return 0;
    return v;
}

// Partial sums of the full decomposition: a set of n bodies needs about
// G * ipb / n + 2 slots per body, where G * ipb <= SMs * MAX_WAVES *
// (resident blocks * i-block width) and the last factor is at most 3072 for
// every compiled variant (8 x 256, 6 x 512, 3 x 1024).  The planes are laid
// out per set (stride n, linear body index), so 3 (giw + 2 n) doubles give
// its n bodies (giw + 2 n) / n slots whatever the pool's size.  make_decomp
// shrinks a grid that would need more than a set has.
int64_t part_elems_for(int sms, int64_t n)
{
    const int64_t giw = (int64_t)sms * MAX_WAVES * 3072;
    const int64_t slots_n = giw + 2 * n, cap_n = MAX_PART_SLOTS * n;
    return 3 * (slots_n < cap_n ? slots_n : cap_n);
}

int pool_create(Pool &P, int device, int64_t cap)
{
    P.device = device;
    P.cap = cap;
    P.num_sms = device_sms(device);
    if (P.num_sms < 1) return set_error(NB_ECUDA, "cudaDeviceGetAttribute failed");
    DevState &s = P.s;
    s.cap = cap;
    s.part_slots = 0;
    s.pstride = 0;
    s.red_len = 0;
    bool ok = true;
    auto A = [&](void **q, size_t bytes) {
        if (ok && cudaMalloc(q, bytes) != cudaSuccess) {
            *q = nullptr;
            ok = false;
        }
    };
    const size_t c8 = (size_t)cap * 8, c4 = (size_t)cap * 4;
    A((void **)&s.x, c8); A((void **)&s.y, c8); A((void **)&s.z, c8);
    A((void **)&s.vx, c8); A((void **)&s.vy, c8); A((void **)&s.vz, c8); A((void **)&s.m, c8);
    A((void **)&s.xh, c4); A((void **)&s.yh, c4); A((void **)&s.zh, c4); A((void **)&s.mf, c4);
    A((void **)&s.xl, c4); A((void **)&s.yl, c4); A((void **)&s.zl, c4);
    A((void **)&s.jd, 2 * (size_t)cap * sizeof(float4));
    A((void **)&s.jl, 2 * (size_t)cap * sizeof(float4));
    A((void **)&s.corr, 3 * c8);
    A((void **)&P.stage, 7 * c8);
    if (!ok) {
        cudaGetLastError();
        pool_destroy(P);
        return set_error(NB_ENOMEM, "device allocation failed for %lld bodies",
                         (long long)cap);
    }
    return NB_OK;
}

void pool_destroy(Pool &P)
{
    DevState &s = P.s;
    void *ptrs[] = {s.x,  s.y,  s.z,  s.vx, s.vy, s.vz, s.m,    s.xh,    s.yh,
                    s.zh, s.mf, s.xl, s.yl, s.zl, s.jd, s.jl, s.part, s.corr, P.stage};
    for (void *q : ptrs)
        if (q) cudaFree(q);
    s = DevState();
    P.stage = nullptr;
    P.cap = 0;
}

// ---- cluster sets ------------------------------------------------------------

namespace {
inline size_t al(size_t b) { return (b + 255) / 256 * 256; }
}

int set_create(ClusterSet &C, int32_t kcap, int64_t body_cap, int priority)
{
    C.kcap = kcap;
    C.scap = (body_cap + SEG_BODIES - 1) / SEG_BODIES + kcap;
    const size_t k8 = (size_t)kcap * 8, k81 = (size_t)(kcap + 1) * 8;
    const size_t bytes = al(k8) * 2 + al(k81) * 3 + al((size_t)kcap * 4) * 2 + al(k8) * 2 +
                         al((size_t)C.scap * 4) + al((size_t)C.scap * 8) * 2 +
                         al((size_t)(kcap + 1) * 4) + al((size_t)kcap * sizeof(Frame)) +
                         al((size_t)kcap * DIAG_STRIDE * 8) + al(k8) * 3;
    if (cudaMalloc(&C.dmem, bytes) != cudaSuccess) {
        cudaGetLastError();
        C.dmem = nullptr;
        return set_error(NB_ENOMEM, "cluster tables: device allocation failed");
    }
    // reduction partials (one row of 16 doubles per segment), the near-pair
    // cell table and body copies, and the non-finite flag
    C.body_cap = body_cap;
    C.ng_hcap = near_table_size(body_cap);
    bool ok = true;
    auto A = [&](void **q, size_t b) {
        if (ok && cudaMalloc(q, b) != cudaSuccess) {
            *q = nullptr;
            ok = false;
        }
    };
    A((void **)&C.red, (size_t)C.scap * 16 * 8);
    A((void **)&C.ng_bucket, (size_t)body_cap * 4);
    A((void **)&C.ng_entry, (size_t)body_cap * 4);
    A((void **)&C.ng_rank, (size_t)body_cap * 4);
    A((void **)&C.ng_total, sizeof(int));
    A((void **)&C.flag, sizeof(int));
    A((void **)&C.cid, (size_t)body_cap * 4);
    A((void **)&C.ng_spos, (size_t)body_cap * 16);
    A((void **)&C.ng_slo, (size_t)body_cap * 16);
    A((void **)&C.ng_slot, (size_t)C.ng_hcap * sizeof(NgSlot));
    if (!ok) {
        cudaGetLastError();
        set_destroy(C);
        return set_error(NB_ENOMEM, "cluster tables: device allocation failed");
    }
    if (cudaStreamCreateWithPriority(&C.side, cudaStreamNonBlocking, priority) != cudaSuccess ||
        cudaEventCreateWithFlags(&C.fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&C.join, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        set_destroy(C);
        return set_error(NB_ECUDA, "cluster tables: stream or event creation failed");
    }
    cudaMemset(C.dmem, 0, bytes);
    return NB_OK;
}

// Storage of at least need elements at p (have of them there), grown by half or
// more, within most where that is enough: freed and allocated on the stream (ordered) or by the plain calls, which
// wait for all work of the device.
template <typename T>
static int reserve(T *&p, int64_t &have, int64_t need, int64_t most, bool ordered,
                   cudaStream_t st)
{
    if (have >= need) return NB_OK;
    const int64_t want = p ? std::max(need, std::min(have * 3 / 2, most)) : need;
    if (p) {
        NB_TRY(ordered ? cudaFreeAsync(p, st) : cudaFree(p));
        p = nullptr;
        have = 0;
    }
    for (const int64_t e : {want, need}) {
        void *q = nullptr;
        const size_t bytes = (size_t)e * sizeof(T);
        if ((ordered ? cudaMallocAsync(&q, bytes, st) : cudaMalloc(&q, bytes)) == cudaSuccess) {
            p = static_cast<T *>(q);
            have = e;
            return NB_OK;
        }
        cudaGetLastError();
    }
    return set_error(NB_ENOMEM, "partial-sum storage: %lld bytes not available",
                     (long long)(need * (int64_t)sizeof(T)));
}

int set_reserve_part(ClusterSet &C, int64_t elems, cudaStream_t st)
{
    return reserve(C.part, C.part_elems, elems, C.part_limit / 8, C.part_ordered, st);
}

int set_release_part(ClusterSet &C, cudaStream_t st)
{
    double *const p = C.part;
    C.part = nullptr;
    C.part_elems = 0;
    if (p) NB_TRY(C.part_ordered ? cudaFreeAsync(p, st) : cudaFree(p));
    return NB_OK;
}

void set_destroy(ClusterSet &C)
{
    void *ptrs[] = {C.dmem,    C.red,   C.ng_bucket, C.ng_entry, C.ng_total, C.flag,
                    C.cid,     C.ng_spos, C.ng_slo,  C.ng_slot,  C.ng_rank,
                    C.hv_mem};
    for (void *q : ptrs)
        if (q) cudaFree(q);
    if (C.part) cudaFree(C.part);
    if (C.fork) cudaEventDestroy(C.fork);
    if (C.join) cudaEventDestroy(C.join);
    if (C.side) cudaStreamDestroy(C.side);
    C = ClusterSet();
}

int set_define(ClusterSet &C, int32_t K, const int64_t *boff, const int64_t *nk,
               const double *eps, const double *dts)
{
    if (K < 1 || K > C.kcap) return set_error(NB_EINVAL, "cluster count %d outside [1, %d]", K, C.kcap);
    C.K = K;
    C.boff.assign(boff, boff + K);
    C.nk.assign(nk, nk + K);
    C.eps.assign(K, 0.0);
    C.dts.assign(K, 1.0);
    C.noff.assign(K + 1, 0);
    for (int32_t k = 0; k < K; ++k) {
        if (nk[k] < 1) return set_error(NB_EINVAL, "cluster %d has no bodies", k);
        C.eps[k] = eps ? eps[k] : 0.0;
        if (dts) C.dts[k] = dts[k];
        C.noff[k + 1] = C.noff[k] + nk[k];
    }
    C.n = C.noff[K];
    // widest cluster in j-tiles (independent of the i-block width; part of
    // the tuned-shape key, so known before the layout)
    C.max_ntiles = 0;
    for (int32_t k = 0; k < K; ++k) {
        const int64_t nt = (C.nk[k] + TILE - 1) / TILE;
        if (nt > C.max_ntiles) C.max_ntiles = nt;
    }
    C.eps2d.resize(K);
    C.eps2f.resize(K);
    for (int32_t k = 0; k < K; ++k) {
        C.eps2d[k] = C.eps[k] * C.eps[k];
        C.eps2f[k] = (float)C.eps2d[k];
    }
    C.ipb = 0;   // layout pending
    return NB_OK;
}

int set_units(ClusterSet &C, int ipb, int jt, bool sym)
{
    if (jt < 32 || jt > TILE || TILE % jt != 0)
        return set_error(NB_EINVAL, "j-range width %d must divide %d and be >= 32", jt, TILE);
    const int64_t per_tile = TILE / jt;
    const int32_t K = C.K;
    C.ipb = ipb;
    C.ntiles.resize(K);
    C.uoff.assign(K + 1, 0);
    C.poff.assign(K, 0);
    C.poff_pot.assign(K, 0);
    C.max_ntiles = 0;
    for (int32_t k = 0; k < K; ++k) {
        const int64_t nt = (C.nk[k] + TILE - 1) / TILE;
        C.ntiles[k] = (int32_t)nt;
        if (nt > C.max_ntiles) C.max_ntiles = nt;
        C.uoff[k + 1] = C.uoff[k] + ((C.nk[k] + ipb - 1) / ipb) * nt * per_tile;
    }
    if (sym) sym_units(C.nk.data(), K, ipb, jt, C.uoff.data());
    C.uoff_pot.assign(K + 1, 0);
    sym_units(C.nk.data(), K, TILE * POT_I, POT_JT, C.uoff_pot.data());
    return NB_OK;
}

int set_layout(ClusterSet &C, cudaStream_t st)
{
    const int32_t K = C.K;
    C.seg_off.assign(K + 1, 0);
    C.seg_k.clear();
    C.seg_lo.clear();
    C.seg_hi.clear();
    for (int32_t k = 0; k < K; ++k) {
        for (int64_t lo = C.noff[k]; lo < C.noff[k + 1]; lo += SEG_BODIES) {
            C.seg_k.push_back(k);
            C.seg_lo.push_back(lo);
            C.seg_hi.push_back(lo + SEG_BODIES < C.noff[k + 1] ? lo + SEG_BODIES : C.noff[k + 1]);
        }
        C.seg_off[k + 1] = (int32_t)C.seg_k.size();
    }
    const int64_t S = (int64_t)C.seg_k.size();
    if (S > C.scap) return set_error(NB_EINVAL, "too many reduction segments");
    // frames and diagnostics at fixed places, then the tables, gathered on the host
    // and copied at once (a copy each took 2 us); set_create's size covers them
    C.frame = (Frame *)C.dmem;
    C.diag = (double *)(C.dmem + al((size_t)C.kcap * sizeof(Frame)));
    char *const dev = (char *)C.diag + al((size_t)C.kcap * DIAG_STRIDE * 8);
    if ((int32_t)C.mu.size() != K) C.mu.assign(K, 0.0);
    std::vector<char> host;
    auto put = [&](const auto &v, size_t count) {
        const size_t at = (host.size() + 15) / 16 * 16, bytes = count * sizeof(v[0]);
        host.resize(at + bytes);
        if (bytes) std::memcpy(host.data() + at, v.data(), bytes);
        return dev + at;
    };
    int64_t *d_boff = (int64_t *)put(C.boff, K);
    int64_t *d_nk = (int64_t *)put(C.nk, K);
    int64_t *d_noff = (int64_t *)put(C.noff, K + 1);
    int64_t *d_uoff = (int64_t *)put(C.uoff, K + 1);
    int64_t *d_uoffp = (int64_t *)put(C.uoff_pot, K + 1);
    int32_t *d_ntiles = (int32_t *)put(C.ntiles, K);
    float *d_eps2f = (float *)put(C.eps2f, K);
    double *d_eps2d = (double *)put(C.eps2d, K);
    double *d_dts = (double *)put(C.dts, K);
    int32_t *d_segk = (int32_t *)put(C.seg_k, S);
    int64_t *d_seglo = (int64_t *)put(C.seg_lo, S);
    int64_t *d_seghi = (int64_t *)put(C.seg_hi, S);
    int32_t *d_segoff = (int32_t *)put(C.seg_off, K + 1);
    double *d_mu = (double *)put(C.mu, K);
    int64_t *d_poff = (int64_t *)put(C.poff, K);
    int64_t *d_poffp = (int64_t *)put(C.poff_pot, K);
    NB_TRY(cudaMemcpyAsync(dev, host.data(), host.size(), cudaMemcpyHostToDevice, st));
    Clusters &c = C.cl;
    c.K = K;
    c.boff = d_boff;
    c.nk = d_nk;
    c.noff = d_noff;
    c.uoff = d_uoff;
    c.ntiles = d_ntiles;
    c.eps2f = d_eps2f;
    c.eps2d = d_eps2d;
    c.dts = d_dts;
    c.mu = d_mu;
    c.poff = d_poff;
    c.frame = C.frame;
    c.S = (int32_t)S;
    c.seg_k = d_segk;
    c.seg_lo = d_seglo;
    c.seg_hi = d_seghi;
    c.seg_off = d_segoff;
    c.cid = C.cid;
    if (K > 1) NB_TRY(launch_cluster_map(c, C.cid, C.n, st));
    // pageable copies are staged before returning; make the tables visible
    // to kernels launched on other streams too
    NB_TRY(cudaStreamSynchronize(st));
    C.cl_pot = c;
    C.cl_pot.uoff = d_uoffp;
    C.cl_pot.poff = d_poffp;
    return NB_OK;
}

// ---- plans -------------------------------------------------------------------

bool sp_family(int mode) { return mode == PM_DS_NEAR || mode == PM_DS_FULL || mode == PM_FP32; }

int mode_of(int precision)
{
    switch (precision) {
    case NB_FP64: return PM_FP64;
    case NB_FP32: return PM_FP32;
    case NB_DS_FULL: return PM_DS_FULL;
    case NB_DD: return PM_DD;
    default: return PM_DS_NEAR;
    }
}

bool float_planes(int precision) { return precision != NB_FP64; }

// Launch order of the pair kernel's blocks over set C: largest estimated work
// first, so that the blocks handed out last, which set the kernel's tail
// when the grid runs in waves, are the cheap ones (longest-processing-time
// first).  A unit's work is its j count (the cluster's last j-tile clipped
// to its bodies rounded up to 32) times the packed i-pairs its i-block
// evaluates per warp (sp: the pairs holding bodies; the float-float kernel
// evaluates all of them), each warp's pairs plus half a pair for its share
// of the j-stream loads; each segment (a run of one i-block's units) adds
// the cost of 16 j of a full i-block for its set-up and write-out.  Only the
// order depends on these estimates: any order gives the same sums.
void block_order(ClusterSet &C, const Decomp &d, int I, bool partial)
{
    const int64_t G = d.G;
    const double full = (TILE / 32) * (I / 2 + 0.5);
    std::vector<double> cost((size_t)G, 0.0);
    for (int64_t g = 0; g < G && d.sym; ++g)
        for (int64_t u = d.U(g); u < d.U(g + 1);) {
            const int32_t k = (int32_t)(std::upper_bound(C.uoff.begin(),
                                                         C.uoff.begin() + C.K + 1, u) -
                                        C.uoff.begin()) - 1;
            const SymRows sr(C.nk[k], d.ipb);
            const int32_t upt = d.ipb / d.jt;
            const int32_t b = sr.row_of((u - C.uoff[k]) / upt);
            const int64_t rf = C.uoff[k] + sr.row_first(b) * upt;
            const int64_t n = C.nk[k], rem = std::min<int64_t>(d.ipb, n - (int64_t)b * d.ipb);
            const double rows = (double)rem / TILE;   // of full width, per warp
            for (; u < d.U(g + 1) && u < rf + (int64_t)sr.row_tiles(b) * upt; ++u) {
                const int32_t t = (int32_t)(u - rf), delta = t / upt;
                const int32_t c = b + delta < sr.nb ? b + delta : b + delta - sr.nb;
                const int64_t j0 = (int64_t)c * d.ipb + (t % upt) * d.jt;
                const int64_t js = std::max<int64_t>(0, std::min<int64_t>(d.jt, n - j0));
                // the tile of a block with itself: 10 of 16 rows' worth
                cost[(size_t)g] += (delta ? 1.0 : 0.625) * rows * (double)((js + 31) / 32 * 32);
            }
            cost[(size_t)g] += 16.0 * I;
        }
    for (int64_t g = 0; g < G && !d.sym; ++g) {
        int64_t u = d.U(g);
        const int64_t uend = d.U(g + 1);
        double c = 0.0;
        while (u < uend) {
            const int32_t k = (int32_t)(std::upper_bound(C.uoff.begin(),
                                                         C.uoff.begin() + C.K + 1, u) -
                                        C.uoff.begin()) - 1;
            const int64_t nt = d.units_per_iblock(C.ntiles[k]);
            const int64_t lu = u - C.uoff[k];
            const int64_t rb = lu / nt, t0 = lu - rb * nt;
            const int64_t t1 = std::min(nt, t0 + (uend - u));
            const int64_t n = C.nk[k], ib0 = rb * d.ipb;
            double act = full;
            if (partial) {
                act = 0.0;
                for (int w = 0; w < TILE / 32; ++w) {
                    const int64_t lw = ib0 + 32 * w;
                    int64_t kmax = n > lw ? (n - lw + TILE - 1) / TILE : 0;
                    if (kmax > I) kmax = I;
                    if (kmax > 0) act += (kmax + 1) / 2 + 0.5;
                }
            }
            const int64_t jend = (n + 31) / 32 * 32;
            const int64_t j0 = t0 * d.jt, j1 = std::min(t1 * d.jt, jend);
            if (j1 > j0) c += act * (double)(j1 - j0);
            c += 16.0 * full;
            u += t1 - t0;
        }
        cost[(size_t)g] = c;
    }
    std::vector<int64_t> idx((size_t)G);
    for (int64_t g = 0; g < G; ++g) idx[(size_t)g] = g;
    std::stable_sort(idx.begin(), idx.end(),
                     [&](int64_t a, int64_t b) { return cost[(size_t)a] > cost[(size_t)b]; });
    C.bperm.resize((size_t)G);
    for (int64_t q = 0; q < G; ++q) C.bperm[(size_t)q] = (uint16_t)idx[(size_t)q];
    C.bperm_G = G;
    C.bperm_W = d.W;
    C.bperm_jt = d.jt;
    C.bperm_ipb = d.ipb;
}

// Whether a set takes the symmetric kernels, where their slots fit.  The modes
// of FP64-class accuracy do: the order of their sums moves results by 1e-14 at
// most.  So does the two-pass mixed mode on one system: there the order moves
// velocities by 1e-10 a step (bodies in an encounter apart, Heavy).  On many
// small clusters it is 1e-9 (fewer, larger float partial sums) with encounters
// in every cluster, and the modes without the near-pair pass do not find their
// encounters: those keep the full kernels and their results.
//
// Small systems and sets of small clusters keep the full kernels too: a unit of
// the symmetric kernels (a j range against every body of one row) lasts longer by
// both sides' sums, and their tiles of an i-block with itself save nothing, which
// counts until every SM has several units.  Measured, full / symmetric (us):
//   double precision, one leapfrog: 512 bodies 23.6 / 28.2, 720 25.0 / 36.4, 768
//   23.6 / 28.3, 800 33.4 / 28.3, 1300 61.9 / 50.1
//   float-float, one SI6A step: 200 bodies 104 / 133, 1024 110 / 139, 1280 147 /
//   139; clusters of 400 to 700 bodies, 2 of them 119 / 145; of 600 to 1000, 2
//   144 / 151; of 300 to 1000, 8 243 / 223; of 300 to 600, 12 183 / 218, 40 396 /
//   414; of 100 to 900, 40 458 / 434; of 100 to 600, 40 315 / 350, 100 590 / 584,
//   800 4040 / 3464; of 300 to 400, 400 1909 / 1502; of 100 to 300, 200 433 / 482,
//   800 1528 / 1659
//   mixed, explicitly two-pass, one SI6A step: 500 bodies 230 / 279, 4096 324 /
//   346, 8192 418 / 465, 11000 537 / 544, 12000 593 / 550: from the size on where
//   NB_DS takes that form
static bool use_sym(const ClusterSet &C, int mode)
{
    double n2 = 0;
    for (int32_t k = 0; k < C.K; ++k) n2 += (double)C.nk[k] * (double)C.nk[k];
    if (mode == PM_DS_NEAR) return C.K == 1 && n2 > (double)DS_FULL_MAX_PAIRS;
    if (mode == PM_FP64) return n2 > 784.0 * 784.0;
    if (mode != PM_DD) return false;
    const double wn = n2 / (double)C.n;   // mean size, by work
    return n2 > 1200.0 * 1200.0 && wn > 250 && (wn > 700 || n2 > 3300.0 * 3300.0);
}

// Bodies per thread without a tuned entry, full decomposition.
static int full_default_I(const ClusterSet &C, int mode)
{
    const int64_t mean = C.n / (C.K > 0 ? C.K : 1);
    switch (mode) {
    case PM_FP64: return 1;
    case PM_DD: return 2;   // measured fastest at N = 262144
    case PM_DS_FULL: return mean < 16384 ? 2 : 4;
    default:
        // float pairs (mixed and pure float): 8 bodies per thread measured
        // fastest at N = 65536 and N = 262144 and on the 512-cluster
        // ensemble (mean N 2519); small clusters keep 2 so the i-blocks
        // stay narrow enough to give every resident block a unit
        return mean < 2048 ? 2 : 8;
    }
}

// The same for the symmetric one, by the work-weighted mean cluster size.
static int sym_default_I(const ClusterSet &C, int mode)
{
    double n2 = 0;
    for (int32_t k = 0; k < C.K; ++k) n2 += (double)C.nk[k] * (double)C.nk[k];
    const double wn = n2 / (double)C.n;
    // an evaluation of 16384 bodies takes 110 / 116 us with 4 / 8, of 20000 156
    // / 147 us, of 24576 bodies 8 bodies 197 us
    if (mode == PM_DS_NEAR) return wn < 4096 ? 2 : wn < 18432 ? 4 : 8;
    if (mode == PM_FP64) return wn < 32768 ? 1 : 2;
    return wn < 6144 ? 2 : 4;   // measured: pairsym_wide.cu
}

// The search for bodies in a close encounter (Heavy) of a symmetric plan in the
// mixed mode: the full kernels' untuned decomposition of the set, and storage for
// the sums.
static int plan_heavy(const Pool &P, ClusterSet &C, int mode, int waves, cudaStream_t st, Heavy &h)
{
    const int fI = full_default_I(C, mode);
    const int64_t resident = (int64_t)P.num_sms * std::max(1, pair_occupancy(mode, fI));
    const int64_t ib = (C.n + TILE * fI - 1) / (TILE * fI), tiles = (C.n + TILE - 1) / TILE;
    int j = TILE;
    while (j > 32 && ib * tiles * (TILE / j) < resident) j /= 2;
    const int64_t W = ib * tiles * (TILE / j);
    const int64_t G = resident * (waves > 0 ? std::min(waves, MAX_WAVES) : DEFAULT_WAVES);
    const int64_t cap = std::min<int64_t>(part_elems_for(P.num_sms, C.n) / (3 * C.n),
                                          MAX_PART_SLOTS);
    h = Heavy{};
    h.full = make_decomp(W, tiles, TILE * fI, std::min(G, W), cap, j);
    h.mu = C.mu[0];
    const int64_t groups = C.n / 512 + h.full.slots + 1;
    if (groups > HV_GROUPS)
        return set_error(NB_EINVAL, "%lld bodies: too many for the search for encounters",
                         (long long)C.n);
    h.parts = (int)((groups + HV_PART - 1) / HV_PART);
    h.blocks = (int)std::min<int64_t>(hv_limit(C.n) * h.parts, 2 * P.num_sms);
    const int64_t listed = hv_limit(C.n), sums = listed * h.parts * HV_PART * 3;
    const int rc = reserve(C.hv_mem, C.hv_bytes, 4 * (sums + 2 * listed + 1) + C.n, INT64_MAX,
                           C.part_ordered, st);
    if (rc) return rc;
    C.hv_sum = (float *)C.hv_mem;
    C.hv_list = (int *)(C.hv_sum + sums);
    C.hv_done = C.hv_list + listed;
    C.hv_count = C.hv_done + listed;
    C.hv_flag = (unsigned char *)(C.hv_count + 1);
    return NB_OK;
}

int plan_make(const Pool &P, ClusterSet &C, int precision, cudaStream_t st, Plan &out,
              const PairShape *force, bool use_table, int waves)
{
    Plan pl;
    pl.precision = precision;
    pl.pl.mode = plan_mode(C, precision);
    bool sym = use_sym(C, pl.pl.mode);
    int I, bps = 0, jt = 0;
    bool untuned = false;
    PairShape tuned;
    if (force) {
        I = force->I;
        bps = force->blocks_per_sm;
        jt = force->jt;
    } else if (use_table && tune_lookup(tune_key(P, C, precision), &tuned) &&
               pair_variant_exists(pl.pl.mode, tuned.I)) {
        I = tuned.I;
        bps = tuned.blocks_per_sm;
        jt = tuned.jt;
    } else {
        I = sym ? sym_default_I(C, pl.pl.mode) : full_default_I(C, pl.pl.mode);
        untuned = true;
    }
    if (!pair_variant_exists(pl.pl.mode, I))
        return set_error(NB_EINVAL, "no pair kernel with %d bodies per thread for this precision",
                         I);
    pl.pl.I = I;
    pl.pl.um = true;
    for (int32_t k = 0; k < C.K && pl.pl.um; ++k) pl.pl.um = C.mu[k] > 0;
    int64_t rows = 0;   // partial sums needed
    for (;;) {
        int occ = sym ? sym_occupancy(pl.pl.mode, I, pl.pl.um) : pair_occupancy(pl.pl.mode, I);
        if (occ < 1) occ = 1;
        int b = bps;
        if (waves > 0) b = (waves < MAX_WAVES ? waves : MAX_WAVES) * occ;
        // the symmetric mixed kernel's blocks: units are coarse (i-blocks of
        // 1024), so the most waves even out (an evaluation of 24576 / 65536 /
        // 131072 bodies 212 / 1104 / 4155 us with 4 of them, 197 / 1097 / 4131
        // us with 6), except where the near-pair pass would wait for the last
        // of them (32768 / 49152 / 57344 bodies 320 / 650 / 828 us with 4, 343
        // / 651 / 860 us with 6)
        int dw = DEFAULT_WAVES;
        if (sym && pl.pl.mode == PM_DS_NEAR && (C.n < 25000 || C.n > 60000)) dw = MAX_WAVES;
        pl.pl.blocks_per_sm = b > 0 ? (b < MAX_WAVES * occ ? b : MAX_WAVES * occ) : dw * occ;
        const int64_t want = (int64_t)P.num_sms * pl.pl.blocks_per_sm;
        const int64_t resident = (int64_t)P.num_sms * occ;
        int j = jt;
        const int least = sym ? sym_jt_least(pl.pl.mode) : 32;
        if (j > 0 && j < least) j = least;
        if (j == 0) {
            // full-width j-tiles, halved while the units are too few to give
            // every resident block one (small clusters)
            j = TILE;
            for (;;) {
                int rc = set_units(C, TILE * I, j, sym);
                if (rc) return rc;
                if (j == least || C.uoff[C.K] >= resident) break;
                j /= 2;
            }
        }
        int rc = set_units(C, TILE * I, j, sym);
        if (rc) return rc;
        const int64_t W = C.uoff[C.K];
        const int64_t G = want < W ? want : W;   // at least one unit per block
        const int64_t full = part_elems_for(P.num_sms, C.n);
        if (!sym) {
            rc = set_reserve_part(C, full, st);
            if (rc) return rc;
            pl.pl.d = make_decomp(W, C.max_ntiles, TILE * I, G, part_slot_cap(C), j);
            break;
        }
        const int64_t limit = C.part_limit / 24;
        if (make_sym_decomp(C.nk.data(), C.K, C.uoff.data(), TILE * I, j, G, limit, true, pl.pl.d,
                            C.poff.data(), &rows) &&
            set_reserve_part(C, 3 * rows > full ? 3 * rows : full, st) == NB_OK &&
            (pl.pl.mode != PM_DS_NEAR ||
             plan_heavy(P, C, pl.pl.mode, waves, st, pl.heavy) == NB_OK))
            break;
        pl.heavy = Heavy{};
        sym = false;   // the slots do not fit: the full kernels, in their own shape
        if (untuned) pl.pl.I = I = full_default_I(C, pl.pl.mode);
    }
    pl.pl.d.fpart = sp_family(pl.pl.mode) ? 1 : 0;
    // several clusters by value: launch the blocks largest-work first.  Not
    // with the near-pair pass beside the pair kernel: its kernels get SMs as
    // the pair kernel's blocks drain, and on the 512-cluster ensemble the
    // tighter tail left them less room (pair kernel 2.5% faster, step 2%
    // slower); in the other modes it made the step 0.5-2.6% faster
    C.bperm_G = -1;
    if (pl.pl.mode != PM_FP64 && pl.pl.mode != PM_DS_NEAR && C.K > 1 && C.K <= PARAM_CLUSTERS &&
        pl.pl.d.G <= PERM_CAP && (!pl.pl.d.sym || pl.pl.d.W <= 4 * PERM_CAP))
        block_order(C, pl.pl.d, I, sp_family(pl.pl.mode));
    for (int32_t k = 0; k < C.K; ++k)
        if (C.eps2d[k] == 0.0) pl.pl.d.mask_self = 1;
    int occ_pot = potential_occupancy();
    if (occ_pot < 1) occ_pot = 1;
    const int64_t Gp = (int64_t)P.num_sms * occ_pot;
    // at most ceil(T G / W) + 1 <= T + 1 slots per body of a row of T units,
    // (G / rows + 2) n in all: always within the full kernels' storage
    int rc = NB_OK;
    if (!make_sym_decomp(C.nk.data(), C.K, C.uoff_pot.data(), TILE * POT_I, POT_JT, Gp,
                         C.part_elems / 3, false, pl.pot, C.poff_pot.data(), &rows))
        rc = set_reserve_part(C, 3 * rows, st);
    if (!rc) rc = set_layout(C, st);
    if (rc) return rc;
    out = pl;
    return NB_OK;
}

int plan_mode(const ClusterSet &C, int precision)
{
    const int m = mode_of(precision);
    if (m != PM_DS_NEAR || precision == NB_DS_NEAR) return m;
    double pairs = 0;
    for (int32_t k = 0; k < C.K; ++k) pairs += (double)C.nk[k] * (double)C.nk[k];
    return pairs <= DS_FULL_MAX_PAIRS ? PM_DS_FULL : PM_DS_NEAR;
}

DevState view(const Pool &P, const ClusterSet &C, const Plan &pl)
{
    DevState s = view(P, C, (int)pl.precision);
    if (pl.pl.mode != PM_DS_NEAR) s.corr = nullptr;
    if (pl.heavy.blocks > 0) {
        s.hv_flag = C.hv_flag;
        s.hv_list = C.hv_list;
        s.hv_count = C.hv_count;
        s.hv_done = C.hv_done;
        s.hv_sum = C.hv_sum;
    }
    return s;
}

// A symmetric plan's shape is no measure for these launches: its i-blocks are
// wider where each unordered pair is evaluated once (float-float from 6144 bodies,
// double precision from 32768), which here halves the blocks.  The first eighth of
// 65536 bodies in float-float takes 10.6 ms with 2 bodies per thread, 21.1 with
// 4; of 32768 in double precision 19.3 with 1, 33.0 with 2.  The mixed mode takes
// the symmetric kernel's choice where that is the narrower, 2048 to 18432 bodies.
PairLaunch range_launch(const Pool &P, const ClusterSet &C, const Plan &pl, int64_t i0, int64_t i1,
                        int64_t &W)
{
    PairLaunch r = pl.pl;
    if (pl.pl.d.sym) r.I = full_default_I(C, r.mode);
    if (r.mode == PM_DS_NEAR) r.I = std::min(r.I, sym_default_I(C, r.mode));
    if (pl.pl.d.sym || r.I != pl.pl.I)
        r.blocks_per_sm = DEFAULT_WAVES * std::max(1, pair_occupancy(r.mode, r.I));
    const int ipb = TILE * r.I;
    const int64_t b0 = i0 / ipb, b1 = (i1 + ipb - 1) / ipb;
    W = b1 - b0;
    const int64_t G = std::min((int64_t)P.num_sms * r.blocks_per_sm, W);
    r.d = make_decomp(W, C.max_ntiles, ipb, G, part_slot_cap(C), TILE, 1);
    r.d.b0 = b0;
    r.d.mask_self = pl.pl.d.mask_self;
    r.d.fpart = pl.pl.d.fpart;
    return r;
}

int64_t part_slot_cap(const ClusterSet &C)
{
    const int64_t per = C.n > 0 ? C.part_elems / (3 * C.n) : MAX_PART_SLOTS;
    return per < MAX_PART_SLOTS ? per : MAX_PART_SLOTS;
}

DevState view(const Pool &P, const ClusterSet &C, int precision)
{
    DevState s = P.s;
    s.cl = C.cl;
    s.n = C.n;
    s.part = C.part;
    s.part_elems = C.part_elems;
    s.pstride = C.n > 0 ? C.n : 1;
    s.part_slots = part_slot_cap(C);
    s.diag = C.diag;
    s.red = C.red;
    s.red_len = C.scap * 16;
    s.ng_bucket = C.ng_bucket;
    s.ng_entry = C.ng_entry;
    s.ng_total = C.ng_total;
    s.ng_hcap = C.ng_hcap;
    s.ng_spos = C.ng_spos;
    s.ng_slo = C.ng_slo;
    s.ng_slot = C.ng_slot;
    s.ng_rank = C.ng_rank;
    s.flag = C.flag;
    if (precision != NB_DS && precision != NB_DS_NEAR) s.corr = nullptr;
    return s;
}

// ---- enqueue -----------------------------------------------------------------

namespace {
void count(int64_t *k, int64_t v)
{
    if (k) *k += v;
}
constexpr int64_t NEAR_KERNELS = 5;   // launch_near_correct (memsets not counted)
}  // namespace

int enq_split(const Pool &P, const ClusterSet &C, const Plan &pl, const Phys &ph,
              cudaStream_t st, int64_t *kernels)
{
    if (!float_planes(pl.precision)) return NB_OK;
    const DevState s = view(P, C, pl);
    const bool near = pl.pl.mode == PM_DS_NEAR;
    NB_TRY(launch_frame(s, ph.near_frac, near, st));
    NB_TRY(launch_split(s, st));
    count(kernels, near ? 5 : 3);
    return NB_OK;
}

int enq_force(const Pool &P, const ClusterSet &C, const Plan &pl, const Phys &ph,
              cudaStream_t st, cudaEvent_t ev0, cudaEvent_t ev1, int64_t *kernels)
{
    const DevState s = view(P, C, pl);
    // inside a stream capture an event record must be an external node to
    // time anything; outside it is a plain record
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    NB_TRY(cudaStreamIsCapturing(st, &cs));
    const unsigned evf =
        cs == cudaStreamCaptureStatusActive ? cudaEventRecordExternal : cudaEventRecordDefault;
    if (ev0) NB_TRY(cudaEventRecordWithFlags(ev0, st, evf));
    HostTab ht;
    ht.K = C.K;
    ht.uoff = C.uoff.data();
    ht.boff = C.boff.data();
    ht.noff = C.noff.data();
    ht.nk = C.nk.data();
    ht.ntiles = C.ntiles.data();
    ht.eps2f = C.eps2f.data();
    ht.mu = C.mu.data();
    ht.poff = C.poff.data();
    const Decomp &d = pl.pl.d;
    if (C.bperm_G == d.G && C.bperm_W == d.W && C.bperm_jt == d.jt && C.bperm_ipb == d.ipb) {
        ht.perm = C.bperm.data();
        ht.nperm = (int32_t)C.bperm.size();
    }
    // the near-pair pass (mixed mode) forks onto the set's side stream and
    // runs beside the pair kernel: both read only the float planes, and they
    // write different buffers (corr, part), so the overlap cannot change a
    // result; the join orders it before whatever follows on st
    const bool near = pl.pl.mode == PM_DS_NEAR;
    if (near) {
        NB_TRY(cudaEventRecord(C.fork, st));
        NB_TRY(cudaStreamWaitEvent(C.side, C.fork, 0));
        NB_TRY(launch_near_correct(s, ph.G, pl.pl.um, C.side, &pl.heavy));
        NB_TRY(cudaEventRecord(C.join, C.side));
        count(kernels, NEAR_KERNELS);
    }
    NB_TRY(launch_pair(s, pl.pl, ht, ph.G, st));
    if (ev1) NB_TRY(cudaEventRecordWithFlags(ev1, st, evf));
    count(kernels, 1);
    if (near) NB_TRY(cudaStreamWaitEvent(st, C.join, 0));
    return NB_OK;
}

int stage_weights(int order, double *w)
{
    if (order == 2) {
        w[0] = 1.0;
        return 1;
    }
    const double w0 = 1.0 - 2.0 * (SI6_W1 + SI6_W2 + SI6_W3);
    const double seq[7] = {SI6_W3, SI6_W2, SI6_W1, w0, SI6_W1, SI6_W2, SI6_W3};
    for (int k = 0; k < 7; ++k) w[k] = seq[k];
    return 7;
}

bool ahead_ok(const Plan &pl) { return !float_planes(pl.precision); }

int enq_step(const Pool &P, const ClusterSet &C, const Plan &pl, const Phys &ph, int order,
             double h, cudaStream_t st, const std::vector<cudaEvent_t> *evs, int64_t *kernels,
             bool ahead, bool next)
{
    const bool sp = float_planes(pl.precision);
    const DevState s = view(P, C, pl);
    double wk[7];
    const int K = stage_weights(order, wk);
    if (sp) {
        const bool near = pl.pl.mode == PM_DS_NEAR;
        NB_TRY(launch_frame(s, ph.near_frac, near, st));
        count(kernels, near ? 4 : 2);
    }
    // drift of the first leapfrog's half step (and the split it feeds, mass
    // words included: the later splits of the step rewrite coordinates only)
    const int first_split = pl.pl.d.sym ? 3 : 2, split = pl.pl.d.sym ? 3 : 1;
    const double hd0 = 0.5 * wk[0] * h;
    if (!ahead) {
        NB_TRY(launch_kick_drift(s, pl.pl.d, 0.0, hd0, 0, sp ? first_split : 0, ph.ext, st));
        count(kernels, 1);
    }
    for (int k = 0; k < K; ++k) {
        // adjacent half drifts of consecutive leapfrogs merge
        const double hd = 0.5 * (wk[k] + (k + 1 < K ? wk[k + 1] : 0.0)) * h;
        const bool last = (k + 1 == K);
        cudaEvent_t e0 = evs ? (*evs)[2 * k] : nullptr, e1 = evs ? (*evs)[2 * k + 1] : nullptr;
        int rc = enq_force(P, C, pl, ph, st, e0, e1, kernels);
        if (rc) return rc;
        NB_TRY(launch_kick_drift(s, pl.pl.d, wk[k] * h, hd, 1, sp && !last ? split : 0, ph.ext, st,
                                 last && next ? hd0 : 0.0));
        count(kernels, 1);
    }
    return NB_OK;
}

int enq_accel_out(const Pool &P, const ClusterSet &C, const Plan &pl, const Phys &ph,
                  double *out, cudaStream_t st, int64_t *kernels)
{
    const DevState s = view(P, C, pl);
    NB_TRY(launch_accel_out(s, pl.pl.d, ph.ext, out, st));
    count(kernels, 1);
    return NB_OK;
}

int enq_energy(const Pool &P, const ClusterSet &C, const Plan &pl, const Phys &ph,
               cudaStream_t st, int64_t *kernels)
{
    DevState s = view(P, C, pl);
    s.cl = C.cl_pot;
    HostTab ht;
    ht.K = C.K;
    ht.uoff = C.uoff_pot.data();
    ht.boff = C.boff.data();
    ht.nk = C.nk.data();
    ht.eps2f = C.eps2f.data();
    ht.poff = C.poff_pot.data();
    NB_TRY(launch_potential(s, pl.pot, ht, st));
    NB_TRY(launch_energy_reduce(s, pl.pot, ph.ext, ph.G, st));
    count(kernels, 3);
    return NB_OK;
}

int enq_torque(const Pool &P, const ClusterSet &C, const Phys &ph, cudaStream_t st,
               int64_t *kernels)
{
    const DevState s = view(P, C, NB_FP64);
    NB_TRY(launch_torque(s, ph.ext, st));
    count(kernels, 2);
    return NB_OK;
}

}  // namespace nb
