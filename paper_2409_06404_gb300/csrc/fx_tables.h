// Host side of the fixed-point reaction tables (fx_tables.cu): what nk_mechanism_load builds from
// a mechanism for the kernels that work on base-2 logarithms in 64-bit fixed point (nk_fx.cuh).
#pragma once

#include <vector>

#include "nk_internal.cuh"

namespace nk {

struct FxTables {
    bool ok = false;                     // the mechanism's numbers fit the fixed-point ranges
    int eff_shift = 0;
    struct Set {
        FxSet s{};                       // (pointers left to the caller)
        std::vector<unsigned char> chunks;
        std::vector<FxSpecies> sp;
    } set[kFxSets];
    double log2_maxinvW = 0.0;
    std::vector<uint32_t> tab;           // exp and log tables (kFxTabBytes)
    Set set32[3];
    std::vector<int32_t> slot32;         // [K]
    std::vector<FxExtra> extra;
    std::vector<int32_t> nu1;
    std::vector<FxTroe> troe;
    std::vector<FxEff> eff;
    int th_lo = 0;                       // thermo polynomials: low range in T/2^th_lo; 0: none
    std::vector<FxThermo> th;
};

// order32: for the rounds of 1, 2 and 4 parts, the reactions (device order) in the order their terms are
// summed; lin_boff: DevMech::lin_boff.  rxn: the mechanism's reactions in device order; nasa: [K][2][kNasaStride].
FxTables build_fx_tables(int K, const std::vector<RxnRec>& rxn, const std::vector<TroeRec>& troe,
                         const std::vector<int32_t>& eff_sp, const std::vector<double>& eff_m1,
                         const std::vector<double>& nasa, const double* W, const double* Tmid,
                         const std::vector<int> (&order32)[3], const std::vector<int32_t>& lin_boff);

}  // namespace nk
