// pairsym.cu -- decomposition and dispatch of the symmetric pair kernels
// (pairsym.cuh).
#include "pairsym.cuh"

namespace nb {

void sym_units(const int64_t *nk, int32_t K, int ipb, int jt, int64_t *uoff)
{
    uoff[0] = 0;
    for (int32_t k = 0; k < K; ++k)
        uoff[k + 1] = uoff[k] + SymRows(nk[k], ipb).tiles() * (ipb / jt);
}

bool make_sym_decomp(const int64_t *nk, int32_t K, const int64_t *uoff, int ipb, int jt,
                     int64_t G, int64_t limit, bool jsum, Decomp &d, int64_t *poff,
                     int64_t *rows)
{
    d = Decomp();
    d.sym = 1;
    d.jsum = jsum ? 1 : 0;
    d.ipb = ipb;
    d.jt = jt;
    const int64_t W = uoff[K];
    d.W = W > 0 ? W : 1;
    if (G > d.W) G = d.W;
    if (G < 1) G = 1;
    const int64_t least = G / 4;
    for (;;) {
        // a row's units touch at most ceil(T G / W) + 1 blocks; its bodies get
        // a slot from each, and one per tile whose j side they are
        int64_t need = 0, most = 0;
        for (int32_t k = 0; k < K; ++k) {
            const SymRows sr(nk[k], ipb);
            const int64_t T = (int64_t)sr.D * (ipb / jt);
            int64_t slots = (T * G + d.W - 1) / d.W + 1;
            if (slots > T) slots = T;
            if (jsum) slots += sr.D;
            poff[k] = need;
            need += slots * nk[k];
            if (slots > most) most = slots;
        }
        d.G = G;
        d.slots = most;
        *rows = need;
        if (need <= limit) break;
        if (G <= least || G == 1) return false;
        G = G - G / 8 - 1;
    }
    d.narrow = (double)(d.W + 1) * (double)(d.G + 1) < 4294967296.0 ? 1 : 0;
    return true;
}

cudaError_t launch_pair_sym(const DevState &s, const PairLaunch &pl, const HostTab &ht, double G,
                            cudaStream_t st)
{
    if (!ht.poff) return cudaErrorInvalidValue;
    return sp_family(pl.mode) ? launch_sym_sp(s, pl, ht, G, st)
                              : launch_sym_wide(s, pl, ht, G, st);
}

int sym_occupancy(int mode, int I, bool um)
{
    return sp_family(mode) ? occupancy_sym_sp(mode, I, um) : occupancy_sym_wide(mode, I);
}

}  // namespace nb
