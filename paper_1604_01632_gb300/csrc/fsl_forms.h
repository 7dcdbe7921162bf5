// fsl_forms.h -- the stream-collide forms and the tuner's choice among them:
// plain host code without CUDA.
#pragma once

#include "../../include/fsl.h"

namespace fsl {

// Stream-collide kernel forms (the autotuner picks one per workload): the split
// form (interface blocks first, then one block per liquid tile), the
// persistent form with 1, 2 or 4 tiles per liquid item, the slab form, the
// two-kernel form (liquid kernel, then one thread per interface cell), the
// tile-fused form with 2 or 4 tiles per block, and the two kernels run side by
// side on two streams.
enum { SC_SPLIT = 0, SC_PERS1 = 1, SC_PERS2 = 2, SC_PERS4 = 3, SC_SLAB = 4, SC_TWO = 5, SC_TILE2 = 6, SC_TILE4 = 7,
       SC_TWOC = 8, SC_FORMS = 9 };

// In FP32 and 16-bit storage the forms fall into three families that round the
// PDFs rebuilt at the interface differently in the last bit (in FP64 every form
// gives the same bits).  A chaotic flow makes another state of that bit within
// tens of steps, so which family a workload runs must not depend on a timing.
enum { FAM_SHARED = 0,   // forms 0-4: several threads per interface cell, normals in shared memory
       FAM_TWO = 1,      // forms 5 and 8
       FAM_TILE = 2 };   // forms 6 and 7
inline int form_family(int form) {
    if (form == SC_TWO || form == SC_TWOC) return FAM_TWO;
    return form == SC_TILE2 || form == SC_TILE4 ? FAM_TILE : FAM_SHARED;
}

// The family the tuner chooses from: a function of the storage precision, one or many
// domains, the padded cells and the interface cells among them (in 1/64).  No timing,
// and nothing that ran before in the process, enters it.  The lines are where the
// fastest form of one family became that of another when each family still had a
// kernel of its own, so that a workload stays on the states it has had.
// Stream-collide work of a step at the lines (us, fastest form of each family,
// SHARED / TWO / TILE; one domain unless said otherwise):
//   few interface cells: FP16-s 1.4 M cells, 1.7/64 interface  51 /  63 /  76
//                                8.0 M cells, 1.7/64           277 / 292 / 313
//                        FP32    8.0 M cells, 1.7/64           303 / 357 / 357
//   small lattices:      FP16-s 137 k cells, 8.2/64             24 /  24 /  29
//                               266 k cells, 7.2/64             34 /  27 /  29
//                        FP32   152 k cells, 8.3/64             22 /  26 /  27
//                               285 k cells, 8.3/64             36 /  28 /  29
//   TWO against TILE (equal since both run as the same tile-fused kernel):
//                        FP32   3.4 M cells, 5.5/64            240 / 207 / 207
//                               3.0 M cells, 7.0/64            254 / 193 / 193
//                        batch, FP16-s 15.8 M cells, 8.1/64   1830 / 857 / 838
inline int family_of(int prec, bool multi, long long cells, int ifrac) {
    const bool wide = prec == FSL_P_FP32;
    // cells from which forms 0-4 no longer hide the interface work, at that share of the
    // cells, behind the liquid tiles of the same launch
    long long shared_below = wide ? 1LL << 18 : 200000;
    if (ifrac < 5) shared_below = wide ? 1LL << 23 : 1LL << 21;
    if (ifrac < 3) shared_below = wide ? 1LL << 62 : 1LL << 24;
    if (ifrac < 2) shared_below = 1LL << 62;
    if (cells < shared_below) return FAM_SHARED;
    if (wide) return !multi && cells >= 1LL << 20 && ifrac < 6 ? FAM_TWO : FAM_TILE;
    return multi && cells >= 1LL << 23 ? FAM_TWO : FAM_TILE;
}

// A tuning decision holds for one shape of workload: storage precision, one or
// many domains, SM count, lattice size (floor of log2 of the padded cells), the
// interface cells among them (in 1/64) and the family the form is chosen from (0 in
// FP64, where any form may be).
struct TuneKey {
    int prec, multi, sms, lsize, ifrac, family;
    TuneKey(int prec_, bool multi_, int sms_, long long cells, long long interface_cells)
        : prec(prec_), multi(multi_ ? 1 : 0), sms(sms_), lsize(0),
          ifrac((int)(64 * interface_cells / (cells > 0 ? cells : 1))) {
        while ((1LL << (lsize + 1)) <= cells) ++lsize;
        family = prec == FSL_P_FP64 ? 0 : family_of(prec, multi_, cells, ifrac);
    }
    bool operator<(const TuneKey& o) const {
        if (prec != o.prec) return prec < o.prec;
        if (multi != o.multi) return multi < o.multi;
        if (sms != o.sms) return sms < o.sms;
        if (lsize != o.lsize) return lsize < o.lsize;
        if (ifrac != o.ifrac) return ifrac < o.ifrac;
        return family < o.family;
    }
};

// The fastest measured form (ms: best time per form, 0 where it did not run) of
// those the workload may run; usable[f]: form f can run on this handle now.
inline int choose_form(const TuneKey& k, const double* ms, const bool* usable) {
    int best = -1, first = -1;
    for (int f = 0; f < SC_FORMS; ++f) {
        if (!usable[f] || (k.prec != FSL_P_FP64 && form_family(f) != k.family)) continue;
        if (first < 0) first = f;
        if (ms[f] > 0.0 && (best < 0 || ms[f] < ms[best])) best = f;
    }
    return best >= 0 ? best : first;
}

// The form a handle takes from the cache.  The key does not hold the order of the
// interface list, which an option sets per handle and which the slab form needs: a
// handle with the list in appended order takes the split form, of the same family,
// in its place.
inline int cached_form(int form, const bool* usable) { return usable[form] ? form : SC_SPLIT; }

}  // namespace fsl
