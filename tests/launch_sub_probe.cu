// Calls launch_sub (csrc/kcl_sub.cu) for tests/test_launches.py.
#include "../paper_2203_13512_gb300/csrc/kcl_internal.cuh"

// n roots of class c, whose out-degrees reach maxd; warps: the call's cta_warps.
extern "C" int probe_launch_sub(unsigned k, int c, unsigned n, unsigned maxd, int listing, unsigned warps) {
    kcl_graph g;
    g.num_sms = 152;
    kcl::Workspace w;
    kcl::ListArgs la;
    la.listing = listing;
    la.max_outdeg = maxd;
    return kcl::launch_sub(&g, k, w, c, 0, n, nullptr, la, warps, nullptr);
}
