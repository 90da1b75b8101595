// C entry point over the window product's plan (csrc/xd_window.h) for the CPU tests (no CUDA).
#include "xd_window.h"

using namespace xd;

// The plan of a graph on 152 CTAs with couplings J: fit[form]: every pass fits in shared memory; listed[0], [1]:
// passes listed coupling by coupling and with the bond.  Returns the number of passes, -1 where a pair is not in
// exactly one of them.
extern "C" int window_fit(int N, int nup, const int32_t *bonds, int nb, const double *J, int32_t *fit, int32_t *listed) {
    std::vector<int> of;
    const auto pairs = win_pairs(bonds, nb, &of);
    std::vector<double> Jp(pairs.size(), 0.0);
    for (int b = 0; b < nb; ++b) Jp[of[b]] += J[b];
    const bool wide = win_wide(n_choose_k(N, nup));
    std::vector<int> covered(pairs.size(), 0);
    listed[0] = listed[1] = 0;
    std::fill(fit, fit + kWinForms, 1);
    const std::vector<WinPlan> plan = win_plan(N, nup, pairs, 152);
    for (const WinPlan &d : plan) {
        std::vector<double> vals;
        std::vector<int> gid;
        for (int b : d.p.bonds) {
            ++covered[b];
            size_t g = std::find(vals.begin(), vals.end(), Jp[b]) - vals.begin();
            if (g == vals.size()) vals.push_back(Jp[b]);
            gid.push_back((int)g);
        }
        const int ng = (int)vals.size() <= kWinMaxGroups ? (int)vals.size() : 0;
        if (!ng) gid.assign(gid.size(), 0);
        WinTables T;
        bool f[kWinForms];
        const int used = win_fitting_lists(d.p, pairs, d.nbase, wide, gid, ng, &T, f);
        ++listed[used ? 0 : 1];
        for (int q = 0; q < kWinForms; ++q) {
            const WinSmem s = win_smem(d.p.rows, T.maxslots, T.maxlist, T.maxstep, used ? used : kWinMaxBonds + 1, d.nbase[q], wide);
            if (f[q] && s.total > 227 * 1024 - 1536) return -2;  // what a CTA can have, less the kernel's own
            fit[q] = fit[q] && f[q];
        }
    }
    for (int c : covered)
        if (c != 1) return -1;
    return (int)plan.size();
}
