// pairsym_sp.cu -- symmetric pair kernel of the mixed mode's float pairs (its
// close pairs are corrected by near.cu).  The frame is pairsym.cuh.
//
// The FP32 FMA pipe bounds it: 14 operations per unordered pair with equal
// masses (17 with a mass spectrum) cap it at 5.75e12 interactions/s.  At N =
// 65536 it runs 4.1e12 (1.047 ms; the full kernel 1.451 ms at 82% of its cap of
// 3.66e12), at N = 15360 3.1e12 (76 us).  What is lost is operand supply: a
// packed FMA with three different register pairs takes the register file more
// than the two cycles it holds the pipe (alone it reaches 54% of the pipe's
// rate, with one operand repeated 86%), and both sides' accumulations, six of
// the fourteen, are of that kind; unpacked FMAs were slower (1.12-1.25 ms, issue
// slots).  Packing two j bodies of a lane, not two i bodies of a thread, halves
// the shuffles and staged reads per pair at the same registers and i-block
// width: 1.047 against 1.092 ms; eight i bodies against four 1.047 : 1.098, with
// four steps unrolled (one 1.059, two 1.094, eight 1.140).  With a mass spectrum
// 1.276 ms at N = 65536 (FMA pipe 76% busy), 19.1 at 262144; with the cube of the
// inverse distance shared by both sides, one operation fewer, 18.9 at 262144, but
// that cube leaves the float range beyond 4e12 length units.
#include "pairsym.cuh"

namespace nb {
namespace {

// I bodies per thread; a lane's two j bodies, q and q + 32 of a chunk of 64, are
// the halves of a packed f32x2 operand.  UM_: all masses of a cluster equal; the
// pair term is d / r^3, scaled after.
template <int I_, bool UM_>
struct Sp {
    static constexpr int I = I_, JL = 2;
    static constexpr bool UM = UM_, JSUM = true, SELF = false;
    static constexpr int ACC = 6 * I;           // double-single running sums
    static constexpr int FOLD_CHUNKS = 8;       // 512 j bodies, 256 per float partial sum
    // resident blocks: the mass spectrum's registers (each i body's mass as both
    // halves) do not fit those of one block more; spilled, an evaluation's kernel
    // took 19.8 instead of 19.1 ms at N = 262144 (I = 8), 65 instead of 61 us at
    // 12000 (I = 4)
    static constexpr int MINB = I == 8 ? (UM ? 3 : 2) : UM ? 4 : 3;
    typedef float Slab;
    typedef float2 Part;
    typedef WideDS Wide;
    struct Eps {
        float e2;
        __device__ __forceinline__ Eps(float f, const double *) : e2(f) {}
    };
    // the chunk's bodies q and q + 32 as one packed operand, twice in a row
    struct Stage {
        float4 xy[64];
        float2 z[64];
        float2 m[UM ? 1 : 64];
    };
    struct Pre {
        float x[2], y[2], z[2], m[2];
        __device__ __forceinline__ void load(const DevState &s, int64_t base, int32_t j, int32_t n)
        {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                x[h] = y[h] = z[h] = FAR_F;
                m[h] = 0.f;
                if (j + 32 * h < n) {
                    const int64_t q = base + j + 32 * h;
                    x[h] = __ldg(s.xh + q);
                    y[h] = __ldg(s.yh + q);
                    z[h] = __ldg(s.zh + q);
                    if (!UM) m[h] = __ldg(s.mf + q);
                }
            }
        }
    };
    static __device__ __forceinline__ void put(Stage &st, int lane, const Pre &p)
    {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = lane + 32 * h;
            st.xy[e] = make_float4(p.x[0], p.x[1], p.y[0], p.y[1]);
            st.z[e] = make_float2(p.z[0], p.z[1]);
            if (!UM) st.m[e] = make_float2(p.m[0], p.m[1]);
        }
    }
    struct IState {
        float nx[I], ny[I], nz[I];                          // negated hi coordinates
        float mi[UM ? 1 : I];
        float2 ax[I], ay[I], az[I];                          // float partial sums
        __device__ __forceinline__ void load(const DevState &s, int64_t base, int32_t i, int32_t n,
                                             int32_t kw)
        {
#pragma unroll
            for (int k = 0; k < I; ++k) {
                nx[k] = ny[k] = nz[k] = FAR_F;
                if (!UM) mi[k] = 0.f;
                if (k < kw && i + 32 * k < n) {
                    const int64_t q = base + i + 32 * k;
                    nx[k] = -s.xh[q];
                    ny[k] = -s.yh[q];
                    nz[k] = -s.zh[q];
                    if (!UM) mi[k] = s.mf[q];
                }
                ax[k] = ay[k] = az[k] = make_float2(0.f, 0.f);
            }
        }
        // fold the float partial sums into the double-single running sums
        __device__ __forceinline__ void fold(float (*acc)[TILE], int tid)
        {
#pragma unroll
            for (int k = 0; k < I; ++k) {
                const float2 t[3] = {ax[k], ay[k], az[k]};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    float *hi = &acc[c * I + k][tid];
                    float *lo = &acc[(3 + c) * I + k][tid];
                    float a = *hi, b = *lo;
                    ds_add(a, b, t[c].x);
                    ds_add(a, b, t[c].y);
                    *hi = a;
                    *lo = b;
                }
                ax[k] = ay[k] = az[k] = make_float2(0.f, 0.f);
            }
        }
        __device__ __forceinline__ WideDS sum(float (*acc)[TILE], int tid, int kk, int c) const
        {
            WideDS v;
            v.h = acc[c * I + kk][tid];
            v.l = acc[(3 + c) * I + kk][tid];
            return v;
        }
    };
    struct JSum {
        float2 x, y, z;
        __device__ __forceinline__ void zero() { x = y = z = make_float2(0.f, 0.f); }
        __device__ __forceinline__ float get(int c, int h) const
        {
            const float2 v = c == 0 ? x : c == 1 ? y : z;
            return h ? v.y : v.x;
        }
    };
    static __device__ __forceinline__ int32_t groups(int32_t kw) { return kw; }   // even

    // MASK: lane l's i bodies kd and kd + 1 are its own two j bodies of the chunk
    // (the warp's own row); they meet at t = 0.
    template <bool SYM, bool MASK, int PA>
    static __device__ __forceinline__ void pass(const Stage &st, int lane, IState &is, JSum &js,
                                                const Eps &eps, int32_t kd)
    {
        const float2 e2 = make_float2(eps.e2, eps.e2);
        const int next = (lane + 1) & 31;
#pragma unroll 4
        for (int t = 0; t < 32; ++t) {
            const int e = lane + t;
            const float4 xy = st.xy[e];
            const float2 xx = make_float2(xy.x, xy.y), yy = make_float2(xy.z, xy.w), zz = st.z[e];
            float2 mm;
            if (!UM) mm = st.m[e];
#pragma unroll
            for (int p = 0; p < PA; ++p) {
                const float2 dx = __fadd2_rn(xx, make_float2(is.nx[p], is.nx[p]));
                const float2 dy = __fadd2_rn(yy, make_float2(is.ny[p], is.ny[p]));
                const float2 dz = __fadd2_rn(zz, make_float2(is.nz[p], is.nz[p]));
                float2 r2 = __ffma2_rn(dx, dx, e2);
                r2 = __ffma2_rn(dy, dy, r2);
                r2 = __ffma2_rn(dz, dz, r2);
                const float2 ri = make_float2(rsqrt_mufu(r2.x), rsqrt_mufu(r2.y));
                const float2 q2 = __fmul2_rn(ri, ri);
                // the masses on one factor first (pair.cu): a shared 1 / r^3 would
                // save a multiplication, but not its range
                float2 si = __fmul2_rn(UM ? ri : __fmul2_rn(mm, ri), q2);
                if (MASK) {
                    if (t == 0 && kd == p) si.x = 0.f;
                    if (t == 0 && kd + 1 == p) si.y = 0.f;
                }
                is.ax[p] = __ffma2_rn(dx, si, is.ax[p]);
                is.ay[p] = __ffma2_rn(dy, si, is.ay[p]);
                is.az[p] = __ffma2_rn(dz, si, is.az[p]);
                if (SYM) {
                    const float2 sj =
                        UM ? si : __fmul2_rn(__fmul2_rn(make_float2(is.mi[p], is.mi[p]), ri), q2);
                    js.x = __ffma2_rn(dx, sj, js.x);
                    js.y = __ffma2_rn(dy, sj, js.y);
                    js.z = __ffma2_rn(dz, sj, js.z);
                }
            }
            if (SYM) {
                js.x = rot1(js.x, next);
                js.y = rot1(js.y, next);
                js.z = rot1(js.z, next);
            }
        }
    }
    // i bodies that exist: a variant per count keeps the loops unrolled
    template <bool SYM, bool MASK>
    static __device__ __forceinline__ void run(int32_t pact, const Stage &st, int lane, IState &is,
                                               JSum &js, const Eps &eps, int32_t kd)
    {
        if (pact >= I)
            pass<SYM, MASK, I>(st, lane, is, js, eps, kd);
        else if (I > 2 && pact == (I > 2 ? I - 2 : 2))
            pass<SYM, MASK, (I > 2 ? I - 2 : 2)>(st, lane, is, js, eps, kd);
        else if (I > 4 && pact == (I > 4 ? I - 4 : 2))
            pass<SYM, MASK, (I > 4 ? I - 4 : 2)>(st, lane, is, js, eps, kd);
        else if (I > 6)
            pass<SYM, MASK, 2>(st, lane, is, js, eps, kd);
    }
};

}  // namespace

// One system: its values by value.
cudaError_t launch_sym_sp(const DevState &s, const PairLaunch &pl, const HostTab &ht, double G,
                          cudaStream_t st)
{
    if (ht.K != 1) return cudaErrorInvalidValue;
#define NB_S(II)                                                          \
    if (pl.mode == PM_DS_NEAR && pl.I == II)                              \
        return pl.um ? launch_sym<Sp<II, true>, 1>(s, pl, ht, G, st)      \
                     : launch_sym<Sp<II, false>, 1>(s, pl, ht, G, st);
    NB_S(2) NB_S(4) NB_S(8)
#undef NB_S
    return cudaErrorInvalidValue;
}

int occupancy_sym_sp(int mode, int I, bool um)
{
#define NB_O(II)                                                                          \
    if (mode == PM_DS_NEAR && I == II)                                                    \
        return um ? occupancy_sym<Sp<II, true>, 1>() : occupancy_sym<Sp<II, false>, 1>();
    NB_O(2) NB_O(4) NB_O(8)
#undef NB_O
    return 0;
}

}  // namespace nb
