// C entry point over the ring search of xd_orbit.h for the CPU tests (no CUDA).
#include "xd_orbit.h"

extern "C" void shim_ring_orbit(int N, int dih, int64_t n, const uint64_t *words, uint64_t *rep, int *cand, int *cnt) {
    for (int64_t i = 0; i < n; ++i) {
        const xd::RingOrbit o = xd::ring_orbit(N, dih, words[i]);
        rep[i] = o.rep;
        cand[i] = o.cand;
        cnt[i] = o.cnt;
    }
}
