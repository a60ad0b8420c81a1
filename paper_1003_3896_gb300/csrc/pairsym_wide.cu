// pairsym_wide.cu -- symmetric pair kernels of FP64-class accuracy: float-float
// on the FP32 pipes (NB_DD), plain double precision (NB_FP64), and the softened
// potential sums of the energy diagnostic.  The frame is pairsym.cuh.
#include "pairsym.cuh"

namespace nb {
namespace {

// ---- float-float ---------------------------------------------------------------
// The pair term of pair_ff_kernel (pair.cu) with its force added to both
// bodies; the product s d is formed once, so a pair costs 71 + 12 + 2 x 24
// FMA-pipe operations (equal masses) for two interactions, 65.5 each instead of
// 107.  Both sides' float-float sums hold at most 32 P terms per half (32 j
// bodies on the i side, a chunk's 2 P bodies of 32 lanes on the j side) before
// they are added in double.  The FP32 FMA pipe bounds it (74% busy, ncu, at P =
// 1, N = 20000; FP64 pipe 29% with the folds).  Kernel rate at N = 50021: 470
// Gpair/s with equal masses, 411 with a mass spectrum (P = 2; P = 1 385), where
// the full kernel's are 306 and 302; one evaluation with a mass spectrum went
// from 8.49 to 6.21 ms.  Four steps unrolled: 2% over two, 4% over one at P = 1;
// a cap of 4 resident blocks at P = 1 (128 registers) lost 1%.  P = 2 halves the
// shuffles and staged reads per pair, P = 1's narrower i-blocks win below ~6000
// bodies, where few units per block are left (N = 3000: 35 against 43 us).
template <int P, bool UM_>
struct Dd {
    static constexpr int I = 2 * P, JL = 1;
    static constexpr bool UM = UM_, JSUM = true, SELF = false;
    static constexpr int ACC = 0, FOLD_CHUNKS = 1;
    static constexpr int MINB = P == 1 ? 3 : 2;
    typedef double Slab, Part;
    typedef WideF64 Wide;

    struct Eps {
        float2 h, l;
        __device__ __forceinline__ Eps(float f, const double *e2)
        {
            const float r = __double2float_rn(*e2 - (double)f);
            h = make_float2(f, f);
            l = make_float2(r, r);
        }
    };

    struct Stage {
        float4 xy[64], zm[64], lxy[64], lzm[64];
    };
    struct Pre {
        float x, y, z, m, lx, ly, lz, lm;
        __device__ __forceinline__ void load(const DevState &s, int64_t base, int32_t j, int32_t n)
        {
            x = y = z = FAR_F;
            m = lx = ly = lz = lm = 0.f;
            if (j < n) {
                const int64_t q = base + j;
                x = __ldg(s.xh + q);
                y = __ldg(s.yh + q);
                z = __ldg(s.zh + q);
                lx = __ldg(s.xl + q);
                ly = __ldg(s.yl + q);
                lz = __ldg(s.zl + q);
                if (!UM) {
                    m = __ldg(s.mf + q);
                    lm = __double2float_rn(__ldg(s.m + q) - (double)m);
                }
            }
        }
    };
    static __device__ __forceinline__ void put(Stage &st, int lane, const Pre &p)
    {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = lane + h * 32;
            st.xy[e] = make_float4(p.x, p.x, p.y, p.y);
            st.zm[e] = make_float4(p.z, p.z, p.m, p.m);
            st.lxy[e] = make_float4(p.lx, p.lx, p.ly, p.ly);
            st.lzm[e] = make_float4(p.lz, p.lz, p.lm, p.lm);
        }
    }

    struct IState {
        float2 xh[P], yh[P], zh[P], xl[P], yl[P], zl[P];
        float2 mh[UM ? 1 : P], ml[UM ? 1 : P];
        float2 axh[P], axl[P], ayh[P], ayl[P], azh[P], azl[P];   // sums of one chunk
        double dax[I], day[I], daz[I];

        __device__ __forceinline__ void zero()
        {
#pragma unroll
            for (int p = 0; p < P; ++p)
                axh[p] = axl[p] = ayh[p] = ayl[p] = azh[p] = azl[p] = make_float2(0.f, 0.f);
        }
        __device__ __forceinline__ void load(const DevState &s, int64_t base, int32_t i, int32_t n,
                                             int32_t kw)
        {
#pragma unroll
            for (int p = 0; p < P; ++p) {
                float v[8][2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int kk = 2 * p + h;
                    v[0][h] = v[1][h] = v[2][h] = -FAR_F;   // padding; j padding sits at +FAR
                    v[3][h] = v[4][h] = v[5][h] = v[6][h] = v[7][h] = 0.f;
                    if (kk < kw && i + 32 * kk < n) {
                        const int64_t q = base + i + 32 * kk;
                        v[0][h] = s.xh[q];
                        v[1][h] = s.yh[q];
                        v[2][h] = s.zh[q];
                        v[3][h] = s.xl[q];
                        v[4][h] = s.yl[q];
                        v[5][h] = s.zl[q];
                        if (!UM) {
                            v[6][h] = s.mf[q];
                            v[7][h] = __double2float_rn(s.m[q] - (double)v[6][h]);
                        }
                    }
                    dax[kk] = day[kk] = daz[kk] = 0.0;
                }
                xh[p] = make_float2(v[0][0], v[0][1]);
                yh[p] = make_float2(v[1][0], v[1][1]);
                zh[p] = make_float2(v[2][0], v[2][1]);
                xl[p] = make_float2(v[3][0], v[3][1]);
                yl[p] = make_float2(v[4][0], v[4][1]);
                zl[p] = make_float2(v[5][0], v[5][1]);
                if (!UM) {
                    mh[p] = make_float2(v[6][0], v[6][1]);
                    ml[p] = make_float2(v[7][0], v[7][1]);
                }
            }
            zero();
        }
        __device__ __forceinline__ void fold(float (*)[TILE], int)
        {
#pragma unroll
            for (int p = 0; p < P; ++p) {
                dax[2 * p] += (double)axh[p].x + (double)axl[p].x;
                dax[2 * p + 1] += (double)axh[p].y + (double)axl[p].y;
                day[2 * p] += (double)ayh[p].x + (double)ayl[p].x;
                day[2 * p + 1] += (double)ayh[p].y + (double)ayl[p].y;
                daz[2 * p] += (double)azh[p].x + (double)azl[p].x;
                daz[2 * p + 1] += (double)azh[p].y + (double)azl[p].y;
            }
            zero();
        }
        __device__ __forceinline__ WideF64 sum(float (*)[TILE], int, int kk, int c) const
        {
            WideF64 v;
            v.v = c == 0 ? dax[kk] : c == 1 ? day[kk] : daz[kk];
            return v;
        }
    };

    struct JSum {
        float2 xh, xl, yh, yl, zh, zl;
        __device__ __forceinline__ void zero()
        {
            xh = xl = yh = yl = zh = zl = make_float2(0.f, 0.f);
        }
        static __device__ __forceinline__ double both(float2 h, float2 l)
        {
            return ((double)h.x + (double)h.y) + ((double)l.x + (double)l.y);
        }
        __device__ __forceinline__ double get(int c, int) const
        {
            return c == 0 ? both(xh, xl) : c == 1 ? both(yh, yl) : both(zh, zl);
        }
    };

    static __device__ __forceinline__ int32_t groups(int32_t kw) { return (kw + 1) / 2; }

    // (h, l) += (f, g): two-sum of the high words, the rest into the low word
    static __device__ __forceinline__ void acc(float2 &h, float2 &l, float2 f, float2 g)
    {
        float2 t, e;
        two_sum2(h, f, t, e);
        h = t;
        l = __fadd2_rn(l, __fadd2_rn(e, g));
    }

    template <bool SYM, bool MASK, int PA>
    static __device__ __forceinline__ void pass(const Stage &st, int lane, IState &q, JSum &js,
                                                const Eps &eps, int32_t kd)
    {
        const float2 one = make_float2(1.f, 1.f);
        const float2 c32 = make_float2(1.5f, 1.5f), c158 = make_float2(1.875f, 1.875f);
        const int next = (lane + 1) & 31;
#pragma unroll 4
        for (int t = 0; t < 32; ++t) {
            const int e = lane + t;
            const float4 A = st.xy[e], B = st.zm[e], C = st.lxy[e], D = st.lzm[e];
            const float2 xjh = make_float2(A.x, A.y), yjh = make_float2(A.z, A.w);
            const float2 zjh = make_float2(B.x, B.y), mjh = make_float2(B.z, B.w);
            const float2 xjl = make_float2(C.x, C.y), yjl = make_float2(C.z, C.w);
            const float2 zjl = make_float2(D.x, D.y), mjl = make_float2(D.z, D.w);
#pragma unroll
            for (int p = 0; p < PA; ++p) {
                float2 dxh, dxl, dyh, dyl, dzh, dzl;
                ff_diff(xjh, xjl, q.xh[p], q.xl[p], dxh, dxl);
                ff_diff(yjh, yjl, q.yh[p], q.yl[p], dyh, dyl);
                ff_diff(zjh, zjl, q.zh[p], q.zl[p], dzh, dzl);
                float2 px, ex, py, ey, pz, ez;
                ff_sq(dxh, dxl, px, ex);
                ff_sq(dyh, dyl, py, ey);
                ff_sq(dzh, dzl, pz, ez);
                float2 s1, t1, s2, t2, s3, t3;   // all terms >= 0
                pos_two_sum2(px, py, s1, t1);
                pos_two_sum2(s1, pz, s2, t2);
                pos_two_sum2(s2, eps.h, s3, t3);
                const float2 err = __fadd2_rn(__fadd2_rn(__fadd2_rn(ex, ey), __fadd2_rn(ez, eps.l)),
                                              __fadd2_rn(__fadd2_rn(t1, t2), t3));
                // (r^2 + eps^2)^(-3/2) as in pair_ff_kernel
                const float2 y0 = make_float2(rsqrt_mufu(s3.x), rsqrt_mufu(s3.y));
                const float2 qh = __fmul2_rn(y0, y0);
                const float2 qe = __ffma2_rn(y0, y0, f2neg(qh));
                float2 v = __ffma2_rn(f2neg(s3), qh, one);
                v = __ffma2_rn(f2neg(s3), qe, v);
                v = __ffma2_rn(f2neg(err), qh, v);
                float2 sh = __fmul2_rn(qh, y0);
                float2 ce = __ffma2_rn(qh, y0, f2neg(sh));
                ce = __ffma2_rn(qe, y0, ce);
                const float2 kv = __fmul2_rn(__ffma2_rn(v, c158, c32), v);
                float2 sl = __ffma2_rn(sh, kv, ce);
                if (MASK) {
                    if (t == 0 && kd == 2 * p) sh.x = sl.x = 0.f;
                    if (t == 0 && kd == 2 * p + 1) sh.y = sl.y = 0.f;
                }
                float2 fh, fl;
                if (UM) {
                    ff_mul(sh, sl, dxh, dxl, fh, fl);
                    acc(q.axh[p], q.axl[p], fh, fl);
                    if (SYM) acc(js.xh, js.xl, fh, fl);
                    ff_mul(sh, sl, dyh, dyl, fh, fl);
                    acc(q.ayh[p], q.ayl[p], fh, fl);
                    if (SYM) acc(js.yh, js.yl, fh, fl);
                    ff_mul(sh, sl, dzh, dzl, fh, fl);
                    acc(q.azh[p], q.azl[p], fh, fl);
                    if (SYM) acc(js.zh, js.zl, fh, fl);
                } else {
                    float2 mh, ml;
                    ff_mul(mjh, mjl, sh, sl, mh, ml);
                    ff_mul(mh, ml, dxh, dxl, fh, fl);
                    acc(q.axh[p], q.axl[p], fh, fl);
                    ff_mul(mh, ml, dyh, dyl, fh, fl);
                    acc(q.ayh[p], q.ayl[p], fh, fl);
                    ff_mul(mh, ml, dzh, dzl, fh, fl);
                    acc(q.azh[p], q.azl[p], fh, fl);
                    if (SYM) {
                        ff_mul(q.mh[p], q.ml[p], sh, sl, mh, ml);
                        ff_mul(mh, ml, dxh, dxl, fh, fl);
                        acc(js.xh, js.xl, fh, fl);
                        ff_mul(mh, ml, dyh, dyl, fh, fl);
                        acc(js.yh, js.yl, fh, fl);
                        ff_mul(mh, ml, dzh, dzl, fh, fl);
                        acc(js.zh, js.zl, fh, fl);
                    }
                }
            }
            if (SYM) {
                js.xh = rot1(js.xh, next);
                js.xl = rot1(js.xl, next);
                js.yh = rot1(js.yh, next);
                js.yl = rot1(js.yl, next);
                js.zh = rot1(js.zh, next);
                js.zl = rot1(js.zl, next);
            }
        }
    }

    template <bool SYM, bool MASK>
    static __device__ __forceinline__ void run(int32_t pact, const Stage &st, int lane, IState &is,
                                               JSum &js, const Eps &eps, int32_t kd)
    {
        if (pact >= P)
            pass<SYM, MASK, P>(st, lane, is, js, eps, kd);
        else
            pass<SYM, MASK, 1>(st, lane, is, js, eps, kd);
    }
};

// ---- double precision and potential -------------------------------------------
// The pair term of pair_fp64_kernel: 3 differences, 3 FMAs, 3 operations for
// (r^2 + eps^2)^(-3/2) (split.cuh), 3 FMAs per side: 15 FP64-pipe operations for
// two interactions (equal masses) instead of 24.  The FP64 pipe bounds it: 75
// Gpair/s at N = 16384 (72 at 4096) where the full kernel ran 38 with six
// operations for the power, one evaluation 7.45 -> 3.83 ms.  One and two bodies
// per thread run alike at N = 16384; one keeps i-blocks narrow for small systems
// (N = 1024: 25 against 43 us), two halves the j slots of large ones.  POT: the potential
// m_j / sqrt(r^2 + eps^2) of eq. 4 summed on the i side alone, each unordered
// pair once: a pair inside a warp's own row, which both of its bodies
// evaluate, counts half, so sum_i m_i phi_i is the sum over unordered pairs:
// half the full sum's pairs at 10 operations, the energy of N = 32768 in 9.7
// instead of 25.4 ms.
template <int I_, bool UM_, bool POT>
struct F64 {
    static constexpr int I = I_, JL = 1;
    static constexpr bool UM = UM_, JSUM = !POT, SELF = POT;
    static constexpr int ACC = 0, FOLD_CHUNKS = 1 << 30;
    static constexpr int MINB = 4;
    typedef double Slab, Part;
    typedef WideF64 Wide;

    struct Eps {
        double e2;
        __device__ __forceinline__ Eps(float, const double *p) : e2(*p) {}
    };
    struct Stage {
        double x[64], y[64], z[64], m[UM ? 1 : 64];
    };
    struct Pre {
        double x, y, z, m;
        __device__ __forceinline__ void load(const DevState &s, int64_t base, int32_t j, int32_t n)
        {
            x = y = z = FAR_D;
            m = 0.0;
            if (j < n) {
                const int64_t q = base + j;
                x = __ldg(s.x + q);
                y = __ldg(s.y + q);
                z = __ldg(s.z + q);
                if (!UM) m = __ldg(s.m + q);
            }
        }
    };
    static __device__ __forceinline__ void put(Stage &st, int lane, const Pre &p)
    {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = lane + h * 32;
            st.x[e] = p.x;
            st.y[e] = p.y;
            st.z[e] = p.z;
            if (!UM) st.m[e] = p.m;
        }
    }

    struct IState {
        double x[I], y[I], z[I], m[UM || POT ? 1 : I], ax[I], ay[I], az[I];
        __device__ __forceinline__ void load(const DevState &s, int64_t base, int32_t i, int32_t n,
                                             int32_t kw)
        {
#pragma unroll
            for (int kk = 0; kk < I; ++kk) {
                x[kk] = y[kk] = z[kk] = -FAR_D;
                if (!UM && !POT) m[kk] = 0.0;
                if (kk < kw && i + 32 * kk < n) {
                    const int64_t q = base + i + 32 * kk;
                    x[kk] = s.x[q];
                    y[kk] = s.y[q];
                    z[kk] = s.z[q];
                    if (!UM && !POT) m[kk] = s.m[q];
                }
                ax[kk] = ay[kk] = az[kk] = 0.0;
            }
        }
        __device__ __forceinline__ void fold(float (*)[TILE], int) {}
        __device__ __forceinline__ WideF64 sum(float (*)[TILE], int, int kk, int c) const
        {
            WideF64 v;
            v.v = c == 0 ? ax[kk] : c == 1 ? ay[kk] : az[kk];
            return v;
        }
    };
    struct JSum {
        double x, y, z;
        __device__ __forceinline__ void zero() { x = y = z = 0.0; }
        __device__ __forceinline__ double get(int c, int) const { return c == 0 ? x : c == 1 ? y : z; }
    };

    static __device__ __forceinline__ int32_t groups(int32_t kw) { return kw; }

    template <bool SYM, bool MASK, int PA>
    static __device__ __forceinline__ void pass(const Stage &st, int lane, IState &is, JSum &js,
                                                const Eps &eps, int32_t kd)
    {
        const int next = (lane + 1) & 31;
#pragma unroll 2
        for (int t = 0; t < 32; ++t) {
            const int e = lane + t;
            const double xj = st.x[e], yj = st.y[e], zj = st.z[e];
            const double mj = UM ? 1.0 : st.m[e];
#pragma unroll
            for (int kk = 0; kk < PA; ++kk) {
                const double dx = xj - is.x[kk], dy = yj - is.y[kk], dz = zj - is.z[kk];
                double r2 = fma(dx, dx, eps.e2);
                r2 = fma(dy, dy, r2);
                r2 = fma(dz, dz, r2);
                if (POT) {
                    double ri = rsqrt_pow<true>(r2);
                    if (MASK && t == 0 && kd == kk) ri = 0.0;
                    is.ax[kk] = fma(MASK ? 0.5 * mj : mj, ri, is.ax[kk]);
                } else {
                    double sp = rsqrt_pow<false>(r2);
                    if (MASK && t == 0 && kd == kk) sp = 0.0;
                    const double si = UM ? sp : mj * sp;
                    is.ax[kk] = fma(dx, si, is.ax[kk]);
                    is.ay[kk] = fma(dy, si, is.ay[kk]);
                    is.az[kk] = fma(dz, si, is.az[kk]);
                    if (SYM) {
                        const double sj = UM ? sp : is.m[kk] * sp;
                        js.x = fma(dx, sj, js.x);
                        js.y = fma(dy, sj, js.y);
                        js.z = fma(dz, sj, js.z);
                    }
                }
            }
            if (SYM) {
                js.x = rot1(js.x, next);
                js.y = rot1(js.y, next);
                js.z = rot1(js.z, next);
            }
        }
    }

    template <bool SYM, bool MASK>
    static __device__ __forceinline__ void run(int32_t pact, const Stage &st, int lane, IState &is,
                                               JSum &js, const Eps &eps, int32_t kd)
    {
        if (pact >= I)
            pass<SYM, MASK, I>(st, lane, is, js, eps, kd);
        else
            pass<SYM, MASK, 1>(st, lane, is, js, eps, kd);
    }
};

// The double-precision kernels wait on the FP64 pipe, not on loop bounds: one
// system's values by value, any ensemble's from the device tables.
template <class A>
cudaError_t launch_f64(const DevState &s, const PairLaunch &pl, const HostTab &ht, double G,
                       cudaStream_t st)
{
    return ht.K == 1 ? launch_sym<A, 1>(s, pl, ht, G, st) : launch_sym<A, 0>(s, pl, ht, G, st);
}
template <class A>
int occupancy_f64()
{
    const int a = occupancy_sym<A, 1>(), b = occupancy_sym<A, 0>();
    return a < b ? a : b;
}

}  // namespace

cudaError_t launch_sym_wide(const DevState &s, const PairLaunch &pl, const HostTab &ht, double G,
                            cudaStream_t st)
{
#define NB_S(M, II, L, ...)                                                   \
    if (pl.mode == M && pl.I == II)                                           \
        return pl.um ? L<__VA_ARGS__, true>>(s, pl, ht, G, st) : L<__VA_ARGS__, false>>(s, pl, ht, G, st);
    NB_S(PM_DD, 2, launch_sym_any, Dd<1)
    NB_S(PM_DD, 4, launch_sym_any, Dd<2)
#undef NB_S
#define NB_S(II)                                                                \
    if (pl.mode == PM_FP64 && pl.I == II)                                       \
        return pl.um ? launch_f64<F64<II, true, false>>(s, pl, ht, G, st)       \
                     : launch_f64<F64<II, false, false>>(s, pl, ht, G, st);
    NB_S(1) NB_S(2)
#undef NB_S
    return cudaErrorInvalidValue;
}

int occupancy_sym_wide(int mode, int I)
{
    int a = 0, b = 0;
    if (mode == PM_DD && I == 2) {
        a = occupancy_sym_any<Dd<1, true>>();
        b = occupancy_sym_any<Dd<1, false>>();
    } else if (mode == PM_DD && I == 4) {
        a = occupancy_sym_any<Dd<2, true>>();
        b = occupancy_sym_any<Dd<2, false>>();
    } else if (mode == PM_FP64 && I == 1) {
        a = occupancy_f64<F64<1, true, false>>();
        b = occupancy_f64<F64<1, false, false>>();
    } else if (mode == PM_FP64 && I == 2) {
        a = occupancy_f64<F64<2, true, false>>();
        b = occupancy_f64<F64<2, false, false>>();
    }
    return a < b ? a : b;
}

cudaError_t launch_potential(const DevState &s, const Decomp &d, const HostTab &ht,
                             cudaStream_t st)
{
    PairLaunch pl{};
    pl.d = d;
    return launch_f64<F64<POT_I, false, true>>(s, pl, ht, 1.0, st);
}

int potential_occupancy() { return occupancy_f64<F64<POT_I, false, true>>(); }

}  // namespace nb
