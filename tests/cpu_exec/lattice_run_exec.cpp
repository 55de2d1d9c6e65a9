// lattice_run_exec.cpp -- TEST-ONLY CPU scaffold: runs lattice regions from the
// lists that the GPU kernels read (imp_run, and cell_wide where a size has it;
// lattice_exec.cpp runs imp_all and cell, whose accesses it checks against the
// dependency DAG).  Compiled by the tests, never part of libsp.so.
//
// What a region loads from imp_run and does not need -- the other half of a
// pair whose level the region does not compute, the other slot of a 16-byte
// pair copy -- is poisoned (NaN, no level) unless another load of that slot by
// the region needs the same site, so that a list, a filter or a flag that
// makes a level read such a value, or read a slot nothing filled, is reported.
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <limits>
#include <random>
#include <string>
#include <vector>

#include "lattice.h"
#include "sp_update.h"

using sp::f2;

namespace {

int sext8(uint32_t w, int byte) { return (int)(int8_t)(uint8_t)(w >> (8 * byte)); }

// A cell of a level as its kernel decodes it.
struct Cell {
    int slot, row, pc, nb[7];
    bool exp_phi, exp_pc;
};

Cell decode(const sp::LatticeTables &t, int i)
{
    Cell c;
    if (!t.cell_wide.empty()) {
        const uint32_t w0 = t.cell_wide[2 * i], w1 = t.cell_wide[2 * i + 1];
        const int a = t.bank_a, b = t.bank_b, sl = (int)(w0 & sp::kLatWideSlotMask);
        c.slot = sl, c.row = (int)((w0 >> sp::kLatWideRowShift) & sp::kLatRowMask), c.pc = sl + 16 * sext8(w0, 3);
        const int nb[7] = {sl, sl - 1, sl + 1, sl - a + 16 * sext8(w1, 0), sl + a + 16 * sext8(w1, 1), sl - b + 16 * sext8(w1, 2),
                           sl + b + 16 * sext8(w1, 3)};
        std::copy(nb, nb + 7, c.nb);
        c.exp_phi = (w0 & sp::kLatWideExpPhi) != 0, c.exp_pc = (w0 & sp::kLatWideExpPc) != 0;
    } else {
        const uint32_t e = t.cell[i];
        const int sl = sp::lat_slot(e);
        const uint64_t rn = t.row_nb[sp::lat_row(e)];
        c.slot = sl, c.row = sp::lat_row(e), c.pc = sl + t.row_pc[c.row];
        const int nb[7] = {sl, sl - 1, sl + 1, sl + sp::lat_dym(rn), sl + sp::lat_dyp(rn), sl + sp::lat_dzm(rn), sl + sp::lat_dzp(rn)};
        std::copy(nb, nb + 7, c.nb);
        c.exp_phi = (e & sp::kLatExpPhi) != 0, c.exp_pc = (e & sp::kLatExpPc) != 0;
    }
    return c;
}

// Planted mistakes: one field of every entry that has it.
bool plant(int which, sp::LatticeTables *t)
{
    bool any = false;
    for (size_t i = 0; i < t->imp_run.size(); i += 2) {
        uint32_t &e = t->imp_run[i], &w = t->imp_run[i + 1];
        const uint32_t before_e = e, before = w;
        switch (which) {
        case 1: w &= ~sp::kLatRunPair; break;
        case 2: w &= ~sp::kLatRunFull2; break;
        case 3: w += 1; break;                       // first level
        case 4: w -= 1 << 8; break;                  // last level
        case 5: w += 1u << sp::kLatRunPcShift; break;
        case 6: e &= ~sp::kLatImpFull; break;
        case 7: e ^= sp::kLatImpBuf; break;
        case 8: e |= sp::kLatImpPair; break;         // pair copies for every import
        }
        any = any || e != before_e || w != before;
    }
    for (size_t i = 0; i < t->cell_wide.size(); i += 2) {
        uint32_t &w0 = t->cell_wide[i], &w1 = t->cell_wide[i + 1];
        switch (which) {
        case 9: w1 += 1; break;
        case 10: w1 -= 1u << 24; break;
        case 11: w0 &= ~sp::kLatWideExpPhi; break;
        case 12: w0 &= ~sp::kLatWideExpPc; break;
        case 13: w0 += 1u << 24; break;              // (pi, c) step
        default: continue;
        }
        any = true;
    }
    return any;
}

}  // namespace

extern "C" {

// One call of nsteps levels; aligned: whether phi starts on 16 bytes; mode 0:
// ticket order, 1: random topological order.  0; -1 with msg; 1: nothing to plant.
int lxr_run(int s, int nx, int ny, int nz, int nsteps, int mode, uint64_t seed, int aligned, int planted, const float *coef4,
            float dt, float inv_dx2, float eta2, float *phi, float *pc, char *msg, int msglen)
{
    auto err = [&](const char *m) {
        std::snprintf(msg, msglen, "%s", m);
        return -1;
    };
    sp::LatticeTables t;
    const std::string e = sp::build_lattice_tables(s, &t);
    if (!e.empty()) return err(e.c_str());
    if (planted && !plant(planted, &t)) return 1;
    sp::LatGeom g;
    g.s = s, g.M[0] = nx / (4 * s), g.M[1] = ny / (4 * s), g.M[2] = nz / (4 * s);
    const int n[3] = {nx, ny, nz}, Lmin = sp::lat_min_layer(), Lcount = sp::lat_layer_count(s, nsteps);
    const int64_t sites = (int64_t)nx * ny * nz, per_layer = sp::lat_per_layer(g), nreg = per_layer * Lcount;
    const sp::PhysConst q = {dt, inv_dx2, eta2, 0.0f};
    const float nan = std::numeric_limits<float>::quiet_NaN();

    std::vector<f2> P[2];
    std::vector<int> tagP[2], tagG((size_t)sites, 0);
    for (int p = 0; p < 2; ++p) P[p].assign((size_t)sites, f2{0.0f, 0.0f}), tagP[p].assign((size_t)sites, -1000000);
    std::memcpy(P[0].data(), phi, sites * 8);
    std::fill(tagP[0].begin(), tagP[0].end(), 0);
    std::vector<float> G(pc, pc + 4 * sites);

    // the order
    std::vector<int64_t> order;
    if (mode == 0) {
        for (int64_t id = 0; id < nreg; ++id) order.push_back(id);
    } else {
        std::mt19937_64 rng(seed);
        std::vector<int> cnt((size_t)nreg, 4);
        std::vector<int64_t> ready;
        for (int64_t id = 0; id < per_layer; ++id) ready.push_back(id);
        while (!ready.empty()) {
            const size_t pick = (size_t)(rng() % ready.size());
            const int64_t id = ready[pick];
            ready[pick] = ready.back();
            ready.pop_back();
            order.push_back(id);
            if (id + per_layer >= nreg) continue;
            int a[3];
            sp::lat_centre(g, Lmin + (int)(id / per_layer), id % per_layer, a);
            for (int i = 0; i < 4; ++i) {
                int d[3], b[3];
                sp::lat_pred_shift(i, d);
                for (int k = 0; k < 3; ++k) b[k] = sp::lat_wrap(a[k] - d[k], 4 * g.M[k]);
                const int64_t sid = (id / per_layer + 1) * per_layer + sp::lat_index<int64_t>(g, b);
                if (--cnt[sid] == 0) ready.push_back(sid);
            }
        }
    }

    const int slots = (t.n_slots + 1) & ~1;
    std::vector<f2> ps[2];
    std::vector<int> tps[2], tpc;
    std::vector<int64_t> need[2], need_pc;  // by slot: the site that a load the region needs puts there, or -1
    std::vector<float> pcs;
    for (const int64_t id : order) {
        const int L = Lmin + (int)(id / per_layer);
        int a[3];
        sp::lat_centre(g, L, id % per_layer, a);
        const int tau_b = 1 + s * L, k_lo = std::max(0, 1 - tau_b), k_hi = std::min(t.K - 1, nsteps - tau_b);
        auto site = [&](int slot, int row) {
            int r[3];
            t.offset_of(slot, row, &r[0], &r[1], &r[2]);
            int64_t v = 0;
            for (int d = 2; d >= 0; --d) v = v * n[d] + sp::lat_wrap(s * a[d] + r[d], n[d]);
            return v;
        };
        for (int p = 0; p < 2; ++p) {
            ps[p].assign(slots, f2{nan, nan}), tps[p].assign(slots, -999), need[p].assign(slots, -1);
        }
        pcs.assign(4 * (size_t)t.n_foot, nan), tpc.assign(t.n_foot, -999), need_pc.assign(t.n_foot, -1);
        // what it needs, from the lists that are not under test
        std::vector<std::vector<int>> level(2, std::vector<int>(slots, -1));  // import level by buffer and slot
        if (k_lo > 0)
            for (int i = t.cell_off[k_lo - 1]; i < t.cell_off[k_lo - 1] + t.cell_n[k_lo - 1]; ++i) {
                const int sl = sp::lat_slot(t.cell[i]), row = sp::lat_row(t.cell[i]);
                need[(k_lo - 1) & 1][sl] = site(sl, row), need_pc[sl + t.row_pc[row]] = site(sl, row);
            }
        for (size_t i = 0; i < t.imp_all.size(); i += 2) {
            const uint32_t en = t.imp_all[i];
            const int k = (int)t.imp_all[i + 1], sl = sp::lat_slot(en), row = sp::lat_row(en);
            level[(k - 1) & 1][sl] = k;
            if (k < k_lo || k > k_hi) continue;
            need[(k - 1) & 1][sl] = site(sl, row);
            if (en & sp::kLatImpFull) need_pc[sl + t.row_pc[row]] = site(sl, row);
        }
        // phi of site v into a slot of buffer b, as the value of local level k - 1
        // (k < 0: whatever the array holds)
        auto put_phi = [&](int b, int sl, int64_t v, int k) {
            if (sl < 0 || sl >= slots) return false;
            if (need[b][sl] >= 0) {
                if (need[b][sl] != v) return false;
                k = level[b][sl] >= k_lo && level[b][sl] <= k_hi ? level[b][sl] : k_lo;
            } else if (k >= 0) {
                k = -1;
            }
            const int par = (tau_b + b) & 1;  // local levels of parity b
            if (k >= 0 && tagP[par][v] != tau_b + k - 1) return false;
            ps[b][sl] = k >= 0 ? P[par][v] : f2{nan, nan};
            tps[b][sl] = k >= 0 ? k - 1 : -999;
            return true;
        };
        auto put_pc = [&](int at, int64_t v) {
            if (at < 0 || at >= t.n_foot) return false;
            if (need_pc[at] < 0) {
                std::fill(&pcs[4 * at], &pcs[4 * at] + 4, nan), tpc[at] = -999;
                return true;
            }
            if (need_pc[at] != v) return false;
            std::memcpy(&pcs[4 * at], &G[4 * v], 16);
            tpc[at] = tagG[v] - tau_b;
            return true;
        };
        if (k_lo > 0)
            for (int i = t.cell_off[k_lo - 1]; i < t.cell_off[k_lo - 1] + t.cell_n[k_lo - 1]; ++i) {
                const Cell c = decode(t, i);
                const int64_t v = site(c.slot, c.row);
                if (!put_phi((k_lo - 1) & 1, c.slot, v, k_lo) || !put_pc(c.pc, v)) return err("own cell of a cut region");
            }
        for (size_t i = 0; i < t.imp_run.size(); i += 2) {
            const uint32_t en = t.imp_run[i], w = t.imp_run[i + 1];
            if (sp::lat_run_last(w) < k_lo || sp::lat_run_first(w) > k_hi) continue;
            const int sl = sp::lat_slot(en), row = sp::lat_row(en), b = (en & sp::kLatImpBuf) ? 1 : 0;
            const int64_t v = site(sl, row);
            const bool same = aligned && ((sl ^ (int)v) & 1) == 0, both = t.run_pairs && (w & sp::kLatRunPair);
            if (!put_phi(b, sl, v, 0)) return err("import into a slot that needs another value");
            if (same && (both || (en & (k_lo == 0 ? sp::kLatImpPair : sp::kLatImpPairRow)))) {
                if (!put_phi(b, sl ^ 1, v ^ 1, 0)) return err("pair copy into a slot that needs another value");
            } else if (both) {
                if (!put_phi(b, sl + 1, site(sl + 1, row), 0)) return err("second import of a pair into a slot that needs another value");
            }
            const int at = sl + sp::lat_run_pc(w);
            if ((en & sp::kLatImpFull) && !put_pc(at, v)) return err("(pi, c) import into a place that needs another value");
            if (both && (w & sp::kLatRunFull2) && !put_pc(at + 1, site(sl + 1, row))) return err("second (pi, c) import of a pair");
        }
        for (int k = k_lo; k <= k_hi; ++k) {
            const int tau = tau_b + k, rp = (k - 1) & 1, wp = k & 1, par = tau & 1;
            const float *cf = coef4 + 4 * (tau - 1);
            const sp::LevelCoef co = {cf[0], cf[1], cf[2], 0.0f};
            for (int i = t.cell_off[k]; i < t.cell_off[k] + t.cell_n[k]; ++i) {
                const Cell c = decode(t, i);
                for (const int nb : c.nb)
                    if (nb < 0 || nb >= t.n_slots || tps[rp][nb] != k - 1) return err("level reads a phi slot without its value");
                if (c.pc < 0 || c.pc >= t.n_foot || tpc[c.pc] != k - 1) return err("level reads (pi, c) without its value");
                f2 p = {pcs[4 * c.pc], pcs[4 * c.pc + 1]}, cc = {pcs[4 * c.pc + 2], pcs[4 * c.pc + 3]};
                const f2 out = sp::site_update(ps[rp][c.nb[0]], ps[rp][c.nb[1]], ps[rp][c.nb[2]], ps[rp][c.nb[3]], ps[rp][c.nb[4]],
                                               ps[rp][c.nb[5]], ps[rp][c.nb[6]], p, cc, co, q);
                ps[wp][c.slot] = out, tps[wp][c.slot] = k;
                const float v4[4] = {p.x, p.y, cc.x, cc.y};
                std::copy(v4, v4 + 4, &pcs[4 * c.pc]);
                tpc[c.pc] = k;
                const int64_t v = site(c.slot, c.row);
                if (c.exp_phi || k == k_hi) P[par][v] = out, tagP[par][v] = tau;
                if (c.exp_pc || k == k_hi) std::copy(v4, v4 + 4, &G[4 * v]), tagG[v] = tau;
            }
        }
    }
    for (int64_t v = 0; v < sites; ++v)
        if (tagP[nsteps & 1][v] != nsteps || tagG[v] != nsteps) return err("final state incomplete");
    std::memcpy(phi, P[nsteps & 1].data(), sites * 8);
    std::memcpy(pc, G.data(), sites * 16);
    return 0;
}

}  // extern "C"
