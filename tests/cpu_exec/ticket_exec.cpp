// ticket_exec.cpp -- TEST-ONLY CPU scaffold: the ticket order of split regions
// (planner.h) decoded as the region kernel decodes it, region by region, and
// compared with the successor patterns.  Compiled by the tests, never part of
// libsp.so.
#include <cstdint>
#include <cstdio>
#include <set>
#include <string>
#include <vector>

#include "planner.h"

extern "C" {

// bands bands of a grid of J positions per axis at base B; reuse: one mailbox
// slot.  planted: 1 = the inverted pyramids before the last wedges,
// 2 = a predecessor's offset with the wrong sign, 3 = one predecessor missing.
int tx_check(int B, int J0, int J1, int J2, int bands, int reuse, int planted, char *msg, int msglen)
{
    auto err = [&](const std::string &m) {
        std::snprintf(msg, msglen, "%s", m.c_str());
        return -1;
    };
    sp::TileTables t;
    sp::PredTables p;
    std::string e = sp::build_tables(B, &t);
    if (e.empty()) e = sp::build_preds(t, &p);
    if (!e.empty()) return err(e);
    const int J[3] = {J0, J1, J2}, Jtot = J0 * J1 * J2;
    const unsigned phases = planted == 1 ? 0x36574210u : sp::kPhaseOrder;
    auto wrap_sum = [&](int jl, const int *d) {
        int jc = 0, mul = 1;
        const int j[3] = {jl % J0, (jl / J0) % J1, jl / (J0 * J1)};
        for (int k = 0; k < 3; ++k) {
            int v = j[k] + d[k];
            v += v < 0 ? J[k] : 0;
            v -= v >= J[k] ? J[k] : 0;
            jc += v * mul;
            mul *= J[k];
        }
        return jc;
    };
    const int total = bands * sp::kTypes * Jtot;
    auto id_of = [&](int band, int S, int jl) { return (band * sp::kTypes + S) * Jtot + jl; };
    // the successor patterns, inverted
    std::vector<std::set<int>> want(total);
    for (int b = 0; b < bands; ++b)
        for (int S = 0; S < sp::kTypes; ++S)
            for (int jl = 0; jl < Jtot; ++jl) {
                auto edge = [&](int band, const sp::Succ &s) {
                    const int d[3] = {s.e[0], s.e[1], s.e[2]};
                    if (band < bands) want[id_of(band, s.type, wrap_sum(jl, d))].insert(id_of(b, S, jl));
                };
                for (const sp::Succ &s : t.same_succ[S]) edge(b, s);
                if (S == sp::kTypes - 1)
                    for (const sp::Succ &s : t.next_succ[(b + 1) & 1]) edge(b + 1, s);
                if (reuse)
                    for (const sp::Succ &s : t.reuse_succ[S]) edge(b + 1, s);
            }
    std::vector<int> ticket(total, -1);
    for (int k = 0; k < total; ++k) {
        const int run = k / Jtot, S = (int)(phases >> (4 * (run & 7))) & 7;
        const int id = id_of(run >> 3, S, k - run * Jtot);
        if (ticket[id] >= 0) return err("a region has two tickets");
        ticket[id] = k;
    }
    for (int b = 0; b < bands; ++b)
        for (int S = 0; S < sp::kTypes; ++S)
            for (int jl = 0; jl < Jtot; ++jl) {
                const int me = id_of(b, S, jl);
                std::set<int> got;
                int n = p.n[S][b == 0 ? 0 : reuse ? 2 : 1];
                if (planted == 3 && S == 7) --n;
                for (int i = 0; i < n; ++i) {
                    const sp::Pred &q = p.preds[(size_t)((b & 1) * sp::kTypes + S) * sp::kMaxPreds + i];
                    int d[3] = {q.e[0], q.e[1], q.e[2]};
                    if (planted == 2)
                        for (int &v : d) v = -v;
                    const int from = id_of(b - (q.type_prev >> 3), q.type_prev & 7, wrap_sum(jl, d));
                    if (from < 0 || from >= total) return err("a predecessor outside the launch");
                    if (ticket[from] >= ticket[me]) return err("a predecessor holds a later ticket");
                    got.insert(from);
                }
                if (got != want[me]) return err("predecessors differ from the inverted successors");
            }
    return 0;
}

}  // extern "C"
