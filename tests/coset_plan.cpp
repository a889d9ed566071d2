// Prints how sv_expect's expectation passes of a Hamiltonian run: linked with
// the library, so that tests can ask which variant and which codes a set of
// strings reaches.  stdin: n g complex128 nterms, then x z per string.
// Per pass: "pass <run bits> <span> <strings> unit <codes...> phases <codes of
// each item...> rest <groups left to the general kernels>".
#include <cstdio>
#include <string>
#include <vector>

#include "sv_internal.h"

int main() {
    int n, g, wide;
    long m;
    if (std::scanf("%d %d %d %ld", &n, &g, &wide, &m) != 4) return 1;
    std::vector<sv_pauli> s(m);
    for (auto &p : s) {
        unsigned long long x, z;
        if (std::scanf("%llu %llu", &x, &z) != 2) return 1;
        p.x = x;
        p.z = z;
    }
    sv_options o;
    sv_options_default(wide ? SV_C128 : SV_C64, &o);
    sv::PlanOptions po;
    po.evc_low_bits = o.evc_low_bits;
    po.evc_span = o.evc_span;
    po.pad_highest = o.pad_highest != 0;
    std::vector<int32_t> l2p(n);
    for (int q = 0; q < n; ++q) l2p[q] = q;
    const std::vector<double> c(m, 1.0);
    sv::EvcPlan P;
    const std::string err = sv::plan_evc(n, g, s.data(), c.data(), m, true, po, l2p, P);
    if (!err.empty()) return std::puts(err.c_str()), 1;
    sv::plan_evc_kernels(P, wide ? SV_C128 : SV_C64);
    for (auto &cp : P.passes) {
        std::printf("pass %d %d %d unit", cp.kl, cp.m, cp.s_end - cp.s_begin);
        for (int i = cp.u_begin; i < cp.u_end; ++i) std::printf(" %u", P.uitems[i].code);
        std::printf(" phases");
        for (int i = cp.ri_begin; cp.rp_end > cp.rp_begin && i < cp.ri_end; ++i)
            std::printf(" %u", P.ritems[i].ctl >> 8 & 255u);
        std::printf(" rest %d\n", cp.u_end > cp.u_begin ? 0 : cp.g_end - cp.g_reg);
    }
    return 0;
}
