// kt_coop_tables.cu -- per-lane programs of the kernels with G lanes per cell, and the
// Jacobian program of the larger-network kernels (host code).
//
// A program is a list of terms per lane; the G lists run side by side, padded to the
// longest.  Rows of f (and entries of the iteration matrix) are dealt to the lanes
// longest first, each to the lane with the least so far, so the padded length stays near
// the average (combustion network, 300 row terms: 60 steps for G >= 8, where the
// temperature row alone has one term per reaction, and 75 for G = 4).  The terms of one row or entry
// stay on one lane in the order in which kt_lane.cuh adds them.
#include <algorithm>
#include <cstring>
#include <vector>

#include "kt_internal.h"

namespace kt {
namespace {

using Terms = std::vector<unsigned>;

// Deals the lists to G lanes, at most `cap` lists each; returns the lane of each list.
std::vector<int> deal(const std::vector<Terms> &lists, int G, int cap)
{
    std::vector<int> order(lists.size()), lane(lists.size()), load(G, 0), count(G, 0);
    for (size_t i = 0; i < order.size(); ++i) order[i] = static_cast<int>(i);
    std::stable_sort(order.begin(), order.end(),
                     [&](int x, int y) { return lists[x].size() > lists[y].size(); });
    for (int i : order) {
        int best = -1;
        for (int l = 0; l < G; ++l)
            if (count[l] < cap && (best < 0 || load[l] < load[best])) best = l;
        lane[i] = best;
        load[best] += static_cast<int>(lists[i].size());
        ++count[best];
    }
    return lane;
}

// Interleaves the lanes' lists as [step][G]; every list ends with its end marker.
int pack(const std::vector<Terms> &lists, const std::vector<int> &lane, int G, unsigned pad,
         std::vector<unsigned> *prog)
{
    std::vector<Terms> per(G);
    for (size_t i = 0; i < lists.size(); ++i)
        per[lane[i]].insert(per[lane[i]].end(), lists[i].begin(), lists[i].end());
    size_t steps = 0;
    for (const Terms &p : per) steps = std::max(steps, p.size());
    prog->assign((steps + kCoopPad) * G, pad);
    for (int l = 0; l < G; ++l)
        for (size_t e = 0; e < per[l].size(); ++e) (*prog)[e * G + l] = per[l][e];
    return static_cast<int>(steps);
}

}  // namespace

bool coop_tables(int N, int ns, int nr, int energy, const int *nin, const int *nout, const int (*in)[kMaxSide],
                 const int (*out)[kMaxSide], const double *dH, int fp32, int G, CoopTab *tab,
                 std::vector<unsigned char> *bytes)
{
    if (N > kLaneMaxN || nr < 1 || nr > kCoopMaxReactions) return false;
    const int NM = coop_nm(N, energy), NC = (NM + G - 1) / G, LD = coop_ld(NM);
    const unsigned rb = fp32 ? 4 : 8;   // bytes of a partial derivative
    std::vector<Terms> rows(N), ent(static_cast<size_t>(N) * N);
    int nin_max = 1;
    for (int r = 0; r < nr; ++r) nin_max = std::max(nin_max, nin[r]);
    auto coef = [](int i) { return static_cast<unsigned>(8 * i) << 16; };          // 0, 1, -1, -dH_r
    for (int r = 0; r < nr; ++r) {
        const unsigned w = 8u * r;
        for (int j = 0; j < nin[r]; ++j) rows[in[r][j]].push_back(w | coef(2));
        for (int j = 0; j < nout[r]; ++j) rows[out[r][j]].push_back(w | coef(1));
        if (energy) rows[ns].push_back(w | coef(3 + r));
    }
    auto partial = [&](int kind, int r) { return rb * static_cast<unsigned>(kCoopConst + kind * nr + r); };
    for (int r = 0; r < nr; ++r)
        for (int c = 0; c < nin[r] + (energy ? 1 : 0); ++c) {
            // column of reactant c, or of the temperature: M = I - h J gains +d in the
            // reactants' rows, -d in the products', + heat * d in the temperature row
            const bool tcol = c == nin[r];
            const int col = tcol ? ns : in[r][c];
            const unsigned d = partial(tcol ? nin_max : c, r);
            for (int j = 0; j < nin[r]; ++j) ent[in[r][j] * N + col].push_back(d | (rb << 16));
            for (int j = 0; j < nout[r]; ++j) ent[out[r][j] * N + col].push_back(d | (2 * rb << 16));
            if (energy) ent[ns * N + col].push_back(d | (partial(nin_max + 1, r) << 16));
        }
    const unsigned pad_row = 8u * nr;   // rate 0 with coefficient 0; partial 0 with coefficient 0
    auto close = [](Terms &list, unsigned pad) {
        if (list.empty()) list.push_back(pad);
        list.back() |= kCoopEnd;
    };
    for (int i = 0; i < N; ++i) {
        close(rows[i], pad_row);
        ent[i * N + i].push_back(rb | (rb << 16));   // the identity: + 1 * 1 after the updates
        for (int j = 0; j < N; ++j) close(ent[i * N + j], 0u);
    }
    const std::vector<int> row_lane = deal(rows, G, NC), ent_lane = deal(ent, G, N * N);
    std::vector<unsigned> rp, jp;
    *tab = CoopTab{};
    tab->nin_max = nin_max;
    tab->ld = LD;
    tab->n_row = pack(rows, row_lane, G, pad_row, &rp);
    tab->n_jac = pack(ent, ent_lane, G, 0u, &jp);
    std::vector<std::vector<unsigned char>> to(G);
    for (int i = 0; i < N; ++i)
        for (int j = 0; j < N; ++j) to[ent_lane[i * N + j]].push_back(static_cast<unsigned char>(i * LD + j));
    size_t n_to = 0;
    for (const auto &t : to) n_to = std::max(n_to, t.size());
    auto align16 = [](size_t x) { return (x + 15) & ~static_cast<size_t>(15); };
    tab->off_row = static_cast<int>(align16(static_cast<size_t>(G) * NC));
    tab->off_jac = static_cast<int>(align16(tab->off_row + 4 * rp.size()));
    tab->off_to = static_cast<int>(align16(tab->off_jac + 4 * jp.size()));
    tab->off_coef = static_cast<int>(align16(tab->off_to + n_to * G));
    tab->bytes = static_cast<int>(align16(tab->off_coef + 8 * (3 + static_cast<size_t>(nr))));
    bytes->assign(tab->bytes, 0);
    std::vector<signed char> own(static_cast<size_t>(G) * NC, -1);
    std::vector<int> have(G, 0);
    for (int i = 0; i < N; ++i) own[row_lane[i] * NC + have[row_lane[i]]++] = static_cast<signed char>(i);
    std::memcpy(bytes->data(), own.data(), own.size());
    std::memcpy(bytes->data() + tab->off_row, rp.data(), 4 * rp.size());
    std::memcpy(bytes->data() + tab->off_jac, jp.data(), 4 * jp.size());
    for (int l = 0; l < G; ++l)
        for (size_t k = 0; k < to[l].size(); ++k) (*bytes)[tab->off_to + k * G + l] = to[l][k];
    std::vector<double> cf{0.0, 1.0, -1.0};
    for (int r = 0; r < nr; ++r) cf.push_back(-dH[r]);
    std::memcpy(bytes->data() + tab->off_coef, cf.data(), 8 * cf.size());
    return true;
}

int team_jacobian(int ns, int nr, int energy, const int *nin, const int (*in)[kMaxSide], const std::vector<int> &rp,
                  const std::vector<int> &re, int LD, int T, std::vector<unsigned> *prog)
{
    const int N = ns + energy;
    int nin_max = 1;
    for (int r = 0; r < nr; ++r) nin_max = std::max(nin_max, nin[r]);
    const int zero = nr * (nin_max + energy);   // the partial that is always 0
    if (zero > static_cast<int>(kTermIndex) || N * LD > static_cast<int>(kTermIndex)) return 0;
    std::vector<Terms> ent(static_cast<size_t>(ns) * N);
    for (int s = 0; s < ns; ++s)
        for (int e = rp[s]; e < rp[s + 1]; ++e) {
            const int r = re[e] >> 8;
            const unsigned sign = (re[e] & 0x80) ? kTermMinus : 0u;
            for (int c = 0; c < nin[r]; ++c)
                ent[s * N + in[r][c]].push_back(sign | static_cast<unsigned>(c * nr + r));
            if (energy) ent[s * N + ns].push_back(sign | static_cast<unsigned>(nin_max * nr + r));
        }
    for (int s = 0; s < ns; ++s)
        for (int m = 0; m < N; ++m) {
            Terms &list = ent[s * N + m];
            if (list.empty()) list.push_back(static_cast<unsigned>(zero));
            list.back() |= kTermEnd | (static_cast<unsigned>(m * LD + s) << kTermPlace);
        }
    const int steps = pack(ent, deal(ent, T, ns * N), T, static_cast<unsigned>(zero), prog);
    const int padded = (steps + 7) & ~7;
    prog->resize(static_cast<size_t>(padded + 8) * T, static_cast<unsigned>(zero));
    std::fill(prog->begin() + static_cast<size_t>(steps) * T, prog->end(), static_cast<unsigned>(zero));
    return padded;
}

}  // namespace kt
