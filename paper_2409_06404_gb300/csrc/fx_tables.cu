// Fixed-point reaction tables: a mechanism's logarithms as 64-bit integers (nk_fx.cuh), the check
// that they fit, and the chunks in which the kernels sum rates of progress into species.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "fx_tables.h"
#include "nk_fx.cuh"

namespace nk {
namespace {

constexpr double kLimit = 15000.0;        // |coefficient|, well inside 2^14
constexpr double kMaxX = 2900.0;          // |log2| of a rate constant over the temperature window
constexpr long double kL2E = 1.44269504088896340735992468100189214L;

int64_t fx(long double v) { return (int64_t)llroundl(v * 281474976710656.0L); }   // 2^48

// The exp and log tables, from their definitions in extended precision (built once).
const std::vector<uint32_t>& math_tables() {
    static const std::vector<uint32_t> t = [] {
        // exp entries {float T_j, d_j}; log entries -log2(c_j/1024) and the reciprocals c_j
        std::vector<uint32_t> tab(kFxTabBytes / 4, 0);
        for (int j = 0; j < kFxExpTab; ++j) {
            const long double t = exp2l((long double)j / kFxExpTab);
            float c = (float)t;
            if ((long double)c > t) c = nextafterf(c, 0.0f);
            std::memcpy(&tab[2 * j], &c, 4);
            tab[2 * j + 1] = (uint32_t)llroundl(((long double)j / kFxExpTab - log2l((long double)c)) * 281474976710656.0L);
        }
        for (int j = 0; j < kFxLogTab; ++j) {
            const long double c = rintl(1024.0L / (1.0L + ((long double)j + 0.5L) / kFxLogTab));
            const int64_t l = fx(-log2l(c / 1024.0L));
            std::memcpy(&tab[2 * kFxExpTab + 2 * j], &l, 8);
            tab[2 * kFxExpTab + 2 * kFxLogTab + j] = (uint32_t)c;
        }
        return tab;
    }();
    return t;
}

// One kernel family's schedule: species slots and chunk images.
bool schedule(int set, int K, const std::vector<RxnRec>& rxn, const std::vector<FxRxn>& rec,
              const std::vector<FxSpecies>& species, const std::vector<int32_t>& eff_sp,
              const std::vector<double>& eff_w, FxTables::Set& out) {
    const int R = (int)rxn.size(), NP = fx_parts(K, set);
    FxSet& f = out.s;
    bool ok = true;
    f.np = NP;
    f.row = set == 0 ? kFxRow : set == 1 ? kFxDRow : 256;
    if (NP == 0) return true;              // (the family does not take this mechanism)

    // species slots: by decreasing number of molecules over all reactions, dealt to the parts with
    // the fewest so far that still have a place
    std::vector<int> slot(K);
    {
        std::vector<int> count(K, 0), by(K);
        for (const RxnRec& r : rxn)
            for (int e = 0; e < 2 * kMaxSide; ++e)
                if (e < r.nr || (e >= kMaxSide && e < kMaxSide + r.np)) count[r.sp[e]] += r.nu[e];
        for (int k = 0; k < K; ++k) by[k] = k;
        std::stable_sort(by.begin(), by.end(), [&](int a, int b) { return count[a] > count[b]; });
        std::vector<int> load(NP, 0), used(NP, 0);
        out.sp.resize(K);
        for (int k : by) {
            int b = -1;
            for (int q = 0; q < NP; ++q)
                if (q + NP * used[q] < K && (b < 0 || load[q] < load[b])) b = q;
            slot[k] = b + NP * used[b]++;
            out.sp[slot[k]] = species[k];
            load[b] += count[k];
        }
    }

    // Chunks of about equal size with the costlier kinds spread evenly over them; within a chunk
    // the reactions go to the parts by decreasing cost, each to the part with the least so far.
    const int chunk = set != 1 || NP > 12 ? 48 : 36;   // (derivatives: their rows share the memory)
    f.nchunk = (R + chunk - 1) / chunk;
    std::vector<std::vector<int>> members(f.nchunk);
    for (int kind = 2, next = 0; kind >= 0; --kind)
        for (int q = 0; q < R; ++q)
            if (rxn[q].type == kind) members[next++ % f.nchunk].push_back(q);
    const int cost[3] = {10, 17, 50};      // elementary, third-body, Troe (instructions, roughly)
    std::vector<std::vector<int>> order(f.nchunk);
    std::vector<std::vector<unsigned char>> first(f.nchunk);
    std::vector<std::vector<std::vector<uint16_t>>> add(f.nchunk), sub(f.nchunk);
    std::vector<std::vector<std::vector<FxEffTerm>>> effs(f.nchunk);
    size_t most = 0, most_eff = 0;
    for (int c = 0; c < f.nchunk; ++c) {
        std::vector<std::vector<int>> part(NP);
        std::vector<int> load(NP, 0);
        for (int q : members[c]) {         // (already by decreasing cost)
            const int b = (int)(std::min_element(load.begin(), load.end()) - load.begin());
            part[b].push_back(q);
            load[b] += cost[rxn[q].type];
        }
        for (int b = 0; b < NP; ++b) {
            first[c].push_back((unsigned char)order[c].size());
            order[c].insert(order[c].end(), part[b].begin(), part[b].end());
        }
        first[c].push_back((unsigned char)order[c].size());
        f.rows = std::max(f.rows, (int)order[c].size());
        add[c].resize(K);
        sub[c].resize(K);
        size_t entries = 0, neff = 0;
        effs[c].resize(K);
        int nx = 0;
        for (size_t i = 0; i < order[c].size(); ++i) {
            const RxnRec& r = rxn[order[c][i]];
            if (r.type != NK_RXN_ELEMENTARY) {
                for (int j = r.eff0; j < r.eff1; ++j, ++neff) effs[c][slot[eff_sp[j]]].push_back(FxEffTerm{eff_w[j], nx, 0});
                ++nx;
            }
            for (int side = 0; side < 2; ++side)
                for (int e = 0; e < (side ? r.np : r.nr); ++e)
                    for (int j = 0; j < r.nu[side * kMaxSide + e]; ++j, ++entries)
                        (side ? add : sub)[c][slot[r.sp[side * kMaxSide + e]]].push_back((uint16_t)(i * 256));
        }
        for (int k = 0; k < K; ++k) ok = ok && add[c][k].size() < 256 && sub[c][k].size() < 256;
        most = std::max(most, entries);
        most_eff = std::max(most_eff, neff);
        f.xrows = std::max(f.xrows, nx);
    }
    auto up = [](int v) { return (v + 15) / 16 * 16; };
    f.image_parts = f.rows * (int)sizeof(FxRxn);
    f.image_spec = f.image_parts + up(NP + 1);
    f.image_list = f.image_spec + up(4 * K);
    f.image_eff = f.image_list + up(2 * (int)most);
    f.image_effl = f.image_eff + (set != 1 ? 0 : up(4 * K));
    f.image = f.image_effl + (set != 1 ? 0 : (int)(most_eff * sizeof(FxEffTerm)));
    ok = ok && f.xrows < 64;
    out.chunks.assign((size_t)f.nchunk * f.image, 0);
    for (int c = 0; c < f.nchunk; ++c) {
        unsigned char* im = out.chunks.data() + (size_t)c * f.image;
        int nx = 0;
        for (size_t i = 0; i < order[c].size(); ++i) {
            FxRxn x = rec[order[c][i]];
            for (uint32_t& o : x.off) o = (o == (uint32_t)K ? (uint32_t)K : (uint32_t)slot[o]) * (uint32_t)f.row;
            if (rxn[order[c][i]].type != NK_RXN_ELEMENTARY) x.info |= (nx++ & 63) << 10;
            std::memcpy(im + i * sizeof(FxRxn), &x, sizeof x);
        }
        if (set == 1) {
            uint32_t at = 0;
            for (int k = 0; k < K; ++k) {
                ok = ok && effs[c][k].size() < 256;
                const uint32_t w = at << 8 | (uint32_t)(effs[c][k].size() & 255);
                std::memcpy(im + f.image_eff + 4 * k, &w, 4);
                for (const FxEffTerm& t : effs[c][k]) std::memcpy(im + f.image_effl + (at++) * sizeof(FxEffTerm), &t, sizeof t);
            }
        }
        std::memcpy(im + f.image_parts, first[c].data(), NP + 1);
        uint32_t at = 0;
        for (int k = 0; k < K; ++k) {
            const uint32_t w = at << 16 | (uint32_t)(add[c][k].size() & 255) << 8 | (uint32_t)(sub[c][k].size() & 255);
            std::memcpy(im + f.image_spec + 4 * k, &w, 4);
            for (const std::vector<uint16_t>* l : {&add[c][k], &sub[c][k]})
                for (uint16_t o : *l) std::memcpy(im + f.image_list + 2 * at++, &o, 2);
        }
    }
    return ok;
}

// The single-precision products' chunks of consecutive reactions of `order`.
bool schedule32(int K, const std::vector<RxnRec>& rxn, const std::vector<int>& order, const std::vector<int32_t>& boff,
                const std::vector<int32_t>& slot, FxTables::Set& out) {
    const int R = (int)order.size(), NP = fx_parts(K, 2), chunk = 48;
    FxSet& f = out.s;
    bool ok = true;
    f.np = NP;
    f.row = 128;
    f.nchunk = (R + chunk - 1) / chunk;
    const int per = (R + f.nchunk - 1) / f.nchunk;
    f.rows = per;
    std::vector<std::vector<std::vector<FxTerm32>>> terms(f.nchunk);
    size_t most = 0;
    auto up = [](int v) { return (v + 15) / 16 * 16; };
    for (int c = 0; c < f.nchunk; ++c) {
        terms[c].resize(K);
        size_t n = 0;
        for (int i = c * per; i < std::min(R, (c + 1) * per); ++i) {
            const RxnRec& r = rxn[order[i]];
            for (int side = 0; side < 2; ++side)
                for (int e = 0; e < (side ? r.np : r.nr); ++e, ++n)
                    terms[c][slot[r.sp[side * kMaxSide + e]]].push_back(
                        FxTerm32{(uint32_t)(i - c * per) * 256u, (float)r.nud[side * kMaxSide + e]});
        }
        most = std::max(most, n);
    }
    f.image_parts = per * (int)sizeof(FxRxn32);
    f.image_spec = f.image_parts + up(NP + 1);
    f.image_list = f.image_spec + up(4 * K);
    f.image = f.image_list + up((int)(most * sizeof(FxTerm32)));
    out.chunks.assign((size_t)f.nchunk * f.image, 0);
    for (int c = 0; c < f.nchunk; ++c) {
        unsigned char* im = out.chunks.data() + (size_t)c * f.image;
        const int n = std::min(R, (c + 1) * per) - c * per;
        for (int i = 0; i < n; ++i) {
            const int q = order[c * per + i];
            const RxnRec& r = rxn[q];
            FxRxn32 x;
            std::memset(&x, 0, sizeof x);
            for (int e = 0; e < r.nr; ++e) x.off[e] = (uint16_t)(slot[r.sp[e]] * 128);
            for (int e = 0; e < r.np; ++e) x.off[4 + e] = (uint16_t)(slot[r.sp[kMaxSide + e]] * 128);
            x.info = r.nr | r.np << 4 | r.type << 8;
            x.r = q;
            x.boff = boff[q];
            x.eff0 = r.eff0;
            x.eff1 = r.eff1;
            std::memcpy(im + i * sizeof x, &x, sizeof x);
        }
        for (int p = 0; p <= NP; ++p) im[f.image_parts + p] = (unsigned char)(n * p / NP);
        uint32_t at = 0;
        for (int k = 0; k < K; ++k) {
            ok = ok && terms[c][k].size() < 256;
            const uint32_t w = at << 8 | (uint32_t)(terms[c][k].size() & 255);
            std::memcpy(im + f.image_spec + 4 * k, &w, 4);
            for (const FxTerm32& t : terms[c][k]) std::memcpy(im + f.image_list + (at++) * sizeof t, &t, sizeof t);
        }
    }
    return ok;
}

}  // namespace

FxTables build_fx_tables(int K, const std::vector<RxnRec>& rxn, const std::vector<TroeRec>& troe,
                         const std::vector<int32_t>& eff_sp, const std::vector<double>& eff_m1,
                         const std::vector<double>& nasa, const double* W, const double* Tmid,
                         const std::vector<int> (&order32)[3], const std::vector<int32_t>& lin_boff) {
    FxTables f;
    const int R = (int)rxn.size();
    bool ok = true;
    auto put = [&](long double v) {
        if (!(fabsl(v) < kLimit)) {
            ok = false;
            return (int64_t)0;
        }
        return fx(v);
    };

    f.tab = math_tables();

    // species
    long double maxInv = 0.0L;
    for (int k = 0; k < K; ++k) maxInv = std::max(maxInv, 1.0L / (long double)W[k]);
    f.log2_maxinvW = (double)log2l(maxInv);
    std::vector<FxSpecies> spec(K);
    const long double s = 8192.0L;        // fx_mul halves: T/4096 enters as T/8192, 128/T as 64/T, log2(T)/16 as log2(T)/32
    const long double l2RP0 = log2l((long double)kR / (long double)kP0);
    for (int k = 0; k < K; ++k) {
        FxSpecies& x = spec[k];
        std::memset(&x, 0, sizeof x);
        x.k = k;
        x.lw = put(log2l(1.0L / (long double)W[k]));
        x.w = (int64_t)llroundl(1.0L / (long double)W[k] / maxInv * 4611686018427387904.0L);   // 2^62
        x.Tmid = Tmid[k];
        for (int r = 0; r < 2; ++r) {
            const double* a = nasa.data() + ((size_t)k * 2 + r) * kNasaStride;
            int64_t* c = x.c[r];
            c[0] = put(kL2E * ((long double)a[0] - a[6]) + l2RP0) + 4;       // (+4: fx_mul cuts)
            c[1] = put(32.0L * (1.0L - (long double)a[0]));
            c[2] = put(-kL2E * a[1] / 2.0L * s);
            c[3] = put(-kL2E * a[2] / 6.0L * s * s);
            c[4] = put(-kL2E * a[3] / 12.0L * s * s * s);
            c[5] = put(-kL2E * a[4] / 20.0L * s * s * s * s);
            c[6] = put(kL2E * a[5] / 64.0L);
            c[8] = put(a[0]);
            c[9] = put((long double)a[1] / 2.0L * s);
            c[10] = put((long double)a[2] / 3.0L * s * s);
            c[11] = put((long double)a[3] / 4.0L * s * s * s);
            c[12] = put((long double)a[4] / 5.0L * s * s * s * s);
            c[13] = put((long double)a[5] / 64.0L);
            c[14] = put((long double)a[1] * s / kFxCpScale);
            c[15] = put((long double)a[2] * s * s / kFxCpScale);
            c[16] = put((long double)a[3] * s * s * s / kFxCpScale);
            c[17] = put((long double)a[4] * s * s * s * s / kFxCpScale);
            c[7] = put((long double)a[0] / kFxCpScale);
        }
    }

    // thermo polynomials: per species and quantity the finest unit its coefficients allow
    {
        double tm = 0.0;
        for (int k = 0; k < K; ++k) tm = std::max(tm, Tmid[k]);
        f.th_lo = 7;
        while (std::ldexp(1.0 - 1e-9, f.th_lo) <= tm && f.th_lo < 13) ++f.th_lo;
        bool th = f.th_lo <= 12;
        f.th.resize(K);
        for (int k = 0; k < K; ++k) {
            FxThermo& x = f.th[k];
            std::memset(&x, 0, sizeof x);
            x.Tmid = Tmid[k];
            long double c[2][18], most[3] = {1.0L, 1.0L, 1.0L};
            for (int r = 0; r < 2; ++r) {
                const double* a = nasa.data() + ((size_t)k * 2 + r) * kNasaStride;
                const long double b = ldexpl(1.0L, (r ? 12 : f.th_lo) + 1), R0 = (long double)kR;
                long double bj = 1.0L;
                for (int j = 0; j < 5; ++j, bj *= b) {
                    c[r][j] = R0 * a[j] * bj;
                    c[r][6 + j] = R0 * a[j] * bj * b / (j + 1);
                    if (j) c[r][13 + j] = -R0 * a[j] * bj * b / (j * (j + 1));
                }
                c[r][5] = c[r][11] = R0 * a[5];
                c[r][12] = R0 * b * ((long double)a[0] - a[6]);
                c[r][13] = -R0 * b * a[0] * 32.0L;
                for (int j = 0; j < 18; ++j) {
                    long double& m = most[j < 5 ? 0 : j < 11 ? 1 : 2];
                    m = std::max(m, fabsl(c[r][j]));
                    th = th && std::isfinite((double)c[r][j]);      // (a NaN or infinite coefficient: doubles)
                }
            }
            for (int q = 0; q < 3; ++q) {
                int e = 0;
                frexpl(most[q], &e);
                x.sh[q] = 60 - e;          // (sums of up to six terms stay below 2^63)
                th = th && x.sh[q] > 20;
            }
            for (int r = 0; r < 2; ++r)
                for (int j = 0; j < 18; ++j)
                    x.c[r][j] = th ? (int64_t)llroundl(ldexpl(c[r][j], x.sh[j < 5 ? 0 : j < 11 ? 1 : 2])) : 0;
        }
        if (!th) f.th_lo = 0;
    }

    // reactions: flattened molecules (a coefficient nu repeats its species nu times)
    std::vector<FxRxn> rec(R);
    for (int q = 0; q < R; ++q) {
        const RxnRec& r = rxn[q];
        FxRxn& x = rec[q];
        std::memset(&x, 0, sizeof x);
        x.lnA = put(kL2E * r.lnA) + 2;    // (fx_mul cuts about 1.25 units)
        x.beta = put(32.0L * r.beta);
        x.Ea = put(-kL2E * r.EaR / 64.0L);
        x.orig = r.orig | q << 16;
        f.nu1.push_back(r.nu[0] | r.nu[kMaxSide] << 4);
        int cnt[2] = {0, 0};
        for (int e = 0; e < 8; ++e) x.off[e] = (uint32_t)K;          // (species; offsets per set below)
        for (int side = 0; side < 2; ++side) {
            const int b = side * kMaxSide, ne = side ? r.np : r.nr;
            for (int e = 0; e < ne; ++e)
                for (int j = 0; j < r.nu[b + e]; ++j) {
                    if (cnt[side] == kMaxSide) {
                        ok = false;       // more than four molecules on a side
                        break;
                    }
                    x.off[b + cnt[side]++] = (uint32_t)r.sp[b + e];
                }
        }
        x.info = cnt[0] | cnt[1] << 4 | r.type << 8;
        if (r.type != NK_RXN_ELEMENTARY) {
            x.info |= (int32_t)f.extra.size() << 16;
            f.extra.push_back(FxExtra{r.eff0, r.eff1, r.aux, 0});
        }
    }
    f.troe.resize(troe.size());
    for (size_t j = 0; j < troe.size(); ++j) {
        f.troe[j].lnA0 = put(kL2E * troe[j].lnA0) + 2;
        f.troe[j].beta0 = put(32.0L * troe[j].beta0);
        f.troe[j].Ea0 = put(-kL2E * troe[j].Ea0R / 64.0L);
        f.troe[j].l3 = put(troe[j].a < 1.0 ? log2l(1.0L - (long double)troe[j].a) : 0.0L);
        f.troe[j].l1 = put(troe[j].a > 0.0 ? log2l((long double)troe[j].a) : 0.0L);
        f.troe[j].x3 = -kL2E * 8192.0L * troe[j].invT3 > -kLimit ? fx(-kL2E * 8192.0L * troe[j].invT3) : 0;
        f.troe[j].x1 = -kL2E * 8192.0L * troe[j].invT1 > -kLimit ? fx(-kL2E * 8192.0L * troe[j].invT1) : 0;
        f.troe[j].x2 = troe[j].hasT2 != 0.0 ? put(-kL2E * troe[j].T2 / 64.0L) : 0;
        // 0 < a < 1 with exponents in range: F_cent in fixed point
        f.troe[j].flags = (troe[j].a > 0.0 && troe[j].a < 1.0 && f.troe[j].x3 != 0 && f.troe[j].x1 != 0 ? 1 : 0) |
                          (troe[j].hasT2 != 0.0 ? 2 : 0);
    }
    // (eps - 1)/W relative to the largest 1/W, in units of 2^(eff_shift - 62)
    long double m = 1.0L;
    for (size_t j = 0; j < eff_sp.size(); ++j) {
        m = std::max(m, fabsl((long double)eff_m1[j]) / (long double)W[eff_sp[j]] / maxInv);
        ok = ok && std::isfinite(eff_m1[j]);                        // (std::max passes a NaN over)
    }
    while (ldexpl(1.0L, f.eff_shift) <= m && f.eff_shift < 32) ++f.eff_shift;
    if (f.eff_shift >= 20) ok = false;
    std::vector<double> eff_w(eff_sp.size());
    for (size_t j = 0; j < eff_sp.size(); ++j)
        eff_w[j] = (double)((long double)eff_m1[j] / (long double)W[eff_sp[j]] / maxInv);
    f.eff.resize(eff_sp.size());
    for (size_t j = 0; j < eff_sp.size(); ++j) {
        f.eff[j].w = ok ? (int64_t)llroundl(ldexpl((long double)eff_m1[j] / (long double)W[eff_sp[j]] / maxInv, 62 - f.eff_shift)) : 0;
        f.eff[j].sp = eff_sp[j];
        f.eff[j].pad = 0;
        f.eff[j].wd = eff_w[j];
        f.eff[j].pad2 = 0;
    }

    // Ranges over the temperature window: rate constants and reaction Gibbs energies together
    // below kMaxX (so that sums stay inside the format and a zero concentration underflows).
    const int NT = 64;
    std::vector<double> G(K);
    for (int it = 0; it <= NT && ok; ++it) {
        const double T = kFxTmin * std::pow(kFxTmax / kFxTmin, (double)it / NT), lT = std::log(T), l2e = (double)kL2E;
        for (int k = 0; k < K; ++k) {
            const double* a = nasa.data() + ((size_t)k * 2 + (T <= Tmid[k] ? 0 : 1)) * kNasaStride;
            G[k] = l2e * (a[0] * (1.0 - lT) - T * (a[1] / 2 + T * (a[2] / 6 + T * (a[3] / 12 + T * a[4] / 20))) +
                          a[5] / T - a[6] + lT) + (double)l2RP0;
        }
        for (int q = 0; q < R && ok; ++q) {
            const RxnRec& r = rxn[q];
            double g = 0.0;
            for (int e = 0; e < r.nr; ++e) g -= r.nu[e] * G[r.sp[e]];
            for (int e = kMaxSide; e < kMaxSide + r.np; ++e) g += r.nu[e] * G[r.sp[e]];
            const double lk = std::fabs(l2e * (r.lnA + r.beta * lT - r.EaR / T));
            double l0 = 0.0;
            if (r.aux >= 0) l0 = std::fabs(l2e * (troe[r.aux].lnA0 + troe[r.aux].beta0 * lT - troe[r.aux].Ea0R / T));
            ok = lk + std::fabs(g) < kMaxX && l0 < kMaxX;
        }
    }

    for (int set = 0; set < kFxSets; ++set) ok = schedule(set, K, rxn, rec, spec, eff_sp, eff_w, f.set[set]) && ok;
    f.slot32.assign(K, 0);
    for (int q = 0; q < K; ++q) f.slot32[f.set[2].sp[q].k] = q;
    for (int v = 0; v < 3; ++v) ok = schedule32(K, rxn, order32[v], lin_boff, f.slot32, f.set32[v]) && ok;
    f.ok = ok;
    return f;
}

}  // namespace nk
