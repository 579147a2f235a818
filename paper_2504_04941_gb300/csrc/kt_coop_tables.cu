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
#include <array>
#include <cstdint>
#include <cstring>
#include <vector>

#include "kt_internal.h"

namespace kt {
namespace {

// The lists' terms one list after the other: of[i] .. of[i + 1] are list i's.
struct Lists {
    std::vector<int> of;
    std::vector<unsigned> terms;

    int size() const { return static_cast<int>(of.size()) - 1; }
    int length(int i) const { return of[i + 1] - of[i]; }
};

// Fills n lists from a source that is run twice, source(add) calling add(list, term) in the
// order of the terms within a list: once to count, once to place.  An empty list gets `pad`;
// mark(i, last) finishes a list's last term.
template <typename Source, typename Mark>
Lists gather(int n, unsigned pad, const Source &source, const Mark &mark)
{
    Lists l;
    l.of.assign(n + 1, 0);
    source([&](int i, unsigned) { ++l.of[i + 1]; });
    std::vector<int> at(n);
    for (int i = 0; i < n; ++i) {
        at[i] = l.of[i];
        l.of[i + 1] = l.of[i] + std::max(l.of[i + 1], 1);
    }
    l.terms.assign(l.of[n], pad);
    source([&](int i, unsigned term) { l.terms[at[i]++] = term; });
    for (int i = 0; i < n; ++i) mark(i, &l.terms[l.of[i + 1] - 1]);
    return l;
}

// Deals the lists to G lanes, at most `cap` lists each, longest first, each to the lane with
// the least so far (the lowest of equals); returns the lane of each list.
std::vector<int> deal(const Lists &lists, int G, int cap)
{
    const int n = lists.size();
    int longest = 0;
    for (int i = 0; i < n; ++i) longest = std::max(longest, lists.length(i));
    std::vector<int> start(longest + 2, 0), order(n), lane(n), count(G, 0);
    for (int i = 0; i < n; ++i) ++start[longest - lists.length(i) + 1];
    for (int k = 0; k <= longest; ++k) start[k + 1] += start[k];
    for (int i = 0; i < n; ++i) order[start[longest - lists.length(i)]++] = i;
    // with[w]: the lanes (G <= 128) with load w that take more lists; loads only grow, so does the least
    std::vector<std::array<uint64_t, 2>> with(1, std::array<uint64_t, 2>{});
    for (int l = 0; l < G; ++l) with[0][l >> 6] |= uint64_t{1} << (l & 63);
    size_t least = 0;
    for (int i : order) {
        while (!(with[least][0] | with[least][1])) ++least;
        const int half = with[least][0] ? 0 : 1, l = 64 * half + __builtin_ctzll(with[least][half]);
        with[least][half] &= with[least][half] - 1;
        lane[i] = l;
        const size_t load = least + lists.length(i);
        if (with.size() <= load) with.resize(load + 1, std::array<uint64_t, 2>{});
        if (++count[l] < cap) with[load][half] |= uint64_t{1} << (l & 63);
    }
    return lane;
}

// Interleaves the lanes' lists as [step][G], each lane's in the order of their numbers.
int pack(const Lists &lists, const std::vector<int> &lane, int G, unsigned pad, std::vector<unsigned> *prog)
{
    std::vector<int> at(G, 0);
    for (int i = 0; i < lists.size(); ++i) at[lane[i]] += lists.length(i);
    const int steps = *std::max_element(at.begin(), at.end());
    prog->assign(static_cast<size_t>(steps + kCoopPad) * G, pad);
    std::fill(at.begin(), at.end(), 0);
    for (int i = 0; i < lists.size(); ++i) {
        const int l = lane[i];
        for (int e = lists.of[i]; e < lists.of[i + 1]; ++e) (*prog)[static_cast<size_t>(at[l]++) * G + l] = lists.terms[e];
    }
    return steps;
}

}  // namespace

bool coop_tables(int N, int ns, int nr, int energy, const int *nin, const int *nout, const int (*in)[kMaxSide],
                 const int (*out)[kMaxSide], const double *dH, int fp32, int G, CoopTab *tab,
                 std::vector<unsigned char> *bytes)
{
    if (N > kLaneMaxN || nr < 1 || nr > kCoopMaxReactions) return false;
    const int NM = coop_nm(N, energy), NC = (NM + G - 1) / G, LD = coop_ld(NM);
    const unsigned rb = fp32 ? 4 : 8;   // bytes of a partial derivative
    int nin_max = 1;
    for (int r = 0; r < nr; ++r) nin_max = std::max(nin_max, nin[r]);
    auto coef = [](int i) { return static_cast<unsigned>(8 * i) << 16; };          // 0, 1, -1, -dH_r
    auto row_terms = [&](auto add) {
        for (int r = 0; r < nr; ++r) {
            const unsigned w = 8u * r;
            for (int j = 0; j < nin[r]; ++j) add(in[r][j], w | coef(2));
            for (int j = 0; j < nout[r]; ++j) add(out[r][j], w | coef(1));
            if (energy) add(ns, w | coef(3 + r));
        }
    };
    auto partial = [&](int kind, int r) { return rb * static_cast<unsigned>(kCoopConst + kind * nr + r); };
    auto ent_terms = [&](auto add) {
        for (int r = 0; r < nr; ++r)
            for (int c = 0; c < nin[r] + (energy ? 1 : 0); ++c) {
                // column of reactant c, or of the temperature: M = I - h J gains +d in the
                // reactants' rows, -d in the products', + heat * d in the temperature row
                const bool tcol = c == nin[r];
                const int col = tcol ? ns : in[r][c];
                const unsigned d = partial(tcol ? nin_max : c, r);
                for (int j = 0; j < nin[r]; ++j) add(in[r][j] * N + col, d | (rb << 16));
                for (int j = 0; j < nout[r]; ++j) add(out[r][j] * N + col, d | (2 * rb << 16));
                if (energy) add(ns * N + col, d | (partial(nin_max + 1, r) << 16));
            }
        for (int i = 0; i < N; ++i) add(i * N + i, rb | (rb << 16));   // the identity: + 1 * 1 after the updates
    };
    const unsigned pad_row = 8u * nr;   // rate 0 with coefficient 0; partial 0 with coefficient 0
    auto end = [](int, unsigned *last) { *last |= kCoopEnd; };
    const Lists rows = gather(N, pad_row, row_terms, end), ent = gather(N * N, 0u, ent_terms, end);
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
    auto terms = [&](auto add) {
        for (int s = 0; s < ns; ++s)
            for (int e = rp[s]; e < rp[s + 1]; ++e) {
                const int r = re[e] >> 8;
                const unsigned sign = (re[e] & 0x80) ? kTermMinus : 0u;
                for (int c = 0; c < nin[r]; ++c) add(s * N + in[r][c], sign | static_cast<unsigned>(c * nr + r));
                if (energy) add(s * N + ns, sign | static_cast<unsigned>(nin_max * nr + r));
            }
    };
    const Lists ent = gather(ns * N, static_cast<unsigned>(zero), terms, [&](int i, unsigned *last) {
        *last |= kTermEnd | (static_cast<unsigned>(i % N * LD + i / N) << kTermPlace);
    });
    const int steps = pack(ent, deal(ent, T, ns * N), T, static_cast<unsigned>(zero), prog);
    const int padded = (steps + 7) & ~7;
    prog->resize(static_cast<size_t>(padded + 8) * T, static_cast<unsigned>(zero));
    std::fill(prog->begin() + static_cast<size_t>(steps) * T, prog->end(), static_cast<unsigned>(zero));
    return padded;
}

}  // namespace kt
