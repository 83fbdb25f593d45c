// Host side of the fixed-point reaction tables (fx_tables.cu): what nk_mechanism_load builds from
// a mechanism for the kernels that work on base-2 logarithms in 64-bit fixed point (nk_fx.cuh).
#pragma once

#include <vector>

#include "nk_internal.cuh"

namespace nk {

struct FxTables {
    bool ok = false;                     // the mechanism's numbers fit the fixed-point ranges
    int rows = 0, nchunk = 0, eff_shift = 0;
    int image = 0, image_parts = 0, image_spec = 0, image_list = 0;
    double log2_maxinvW = 0.0;
    std::vector<uint32_t> tab;           // exp and log tables (kFxTabBytes)
    std::vector<unsigned char> chunks;   // [nchunk][image]
    std::vector<FxExtra> extra;
    std::vector<FxTroe> troe;
    std::vector<FxSpecies> sp;
    std::vector<FxEff> eff;
};

// rxn: the mechanism's reactions in device order; nasa: [K][2][kNasaStride].
FxTables build_fx_tables(int K, const std::vector<RxnRec>& rxn, const std::vector<TroeRec>& troe,
                         const std::vector<int32_t>& eff_sp, const std::vector<double>& eff_m1,
                         const std::vector<double>& nasa, const double* W, const double* Tmid);

}  // namespace nk
