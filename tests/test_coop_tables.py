"""Per-lane programs of the kernels that give a cell several lanes (csrc/kt_coop_tables.cu).

The larger networks' Jacobian program is laid out by the same file and replayed too.

Replayed here on random rates for random networks (repeated species, one to three
reactants, up to three products, with and without temperature): every row of f and every
entry of I - h J must come out bit for bit as the reaction-by-reaction loop of the
lane-per-cell kernels forms it, each component owned by exactly one lane.  Host compiler
only; no GPU.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2504_04941_gb300", "csrc")

PROBE = r"""
#include "kt_coop_tables.cu"
extern "C" int probe(int N, int ns, int nr, int energy, const int *nin, const int *nout, const int *in,
                     const int *out, const double *dH, int fp32, int G, int *tab, unsigned char *bytes, int cap)
{
    kt::CoopTab t;
    std::vector<unsigned char> b;
    if (!kt::coop_tables(N, ns, nr, energy, nin, nout, reinterpret_cast<const int(*)[3]>(in),
                         reinterpret_cast<const int(*)[3]>(out), dH, fp32, G, &t, &b))
        return -1;
    const int v[9] = {t.n_row, t.n_jac, t.off_row, t.off_jac, t.off_to, t.off_coef, t.nin_max,
                      kt::coop_nm(N), kt::coop_ld(kt::coop_nm(N))};
    std::memcpy(tab, v, sizeof v);
    if (static_cast<int>(b.size()) > cap) return -2;
    std::memcpy(bytes, b.data(), b.size());
    return static_cast<int>(b.size());
}
extern "C" int team(int ns, int nr, int energy, const int *nin, const int *in, const int *rp, const int *re, int LD, int T,
                    unsigned *prog, int cap)
{
    std::vector<unsigned> p;
    const int steps = kt::team_jacobian(ns, nr, energy, nin, reinterpret_cast<const int(*)[3]>(in),
                                        std::vector<int>(rp, rp + ns + 1), std::vector<int>(re, re + rp[ns]), LD, T, &p);
    if (static_cast<int>(p.size()) > cap) return -2;
    std::memcpy(prog, p.data(), 4 * p.size());
    return steps ? steps << 16 | static_cast<int>(p.size()) / T : 0;
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("coop")
    src, so = d / "probe.cpp", d / "probe.so"
    src.write_text(PROBE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True,
                   capture_output=True)
    return ctypes.CDLL(str(so))


def _network(rng, ns, nr):
    nin, nout = rng.integers(1, 4, nr), rng.integers(0, 4, nr)
    species = lambda k: [int(v) for v in rng.integers(0, ns, k)]
    return [species(k) for k in nin], [species(k) for k in nout]


@pytest.mark.parametrize("N,energy,nr,G,fp32", [(1, 0, 1, 4, 0), (2, 1, 3, 8, 1), (3, 0, 3, 4, 1), (11, 1, 60, 8, 1),
                                                (11, 1, 60, 16, 0), (11, 1, 60, 32, 1), (7, 1, 33, 16, 0),
                                                (12, 0, 29, 4, 1), (16, 1, 400, 16, 0), (16, 0, 1, 32, 1)])
def test_programs_replay_the_reaction_loop(probe, N, energy, nr, G, fp32):
    rng = np.random.default_rng(N * 1000 + nr + G)
    ns = N - energy
    ins, outs = _network(rng, ns, nr)
    ity = np.int32
    nin, nout = np.array([len(i) for i in ins], ity), np.array([len(o) for o in outs], ity)
    pad = lambda ls: np.array([(l + [-1] * 3)[:3] for l in ls], ity)
    pin, pout, dH = pad(ins), pad(outs), rng.standard_normal(nr)
    tab, buf = np.zeros(9, ity), np.zeros(1 << 20, np.uint8)
    p = lambda a: ctypes.c_void_p(a.ctypes.data)
    size = probe.probe(N, ns, nr, energy, p(nin), p(nout), p(pin), p(pout), p(dH), fp32, G, p(tab), p(buf), buf.size)
    assert size > 0 and size % 16 == 0
    n_row, n_jac, off_row, off_jac, off_to, off_coef, nin_max, NM, LD = (int(v) for v in tab)
    assert nin_max == nin.max()
    NC, rb, ft = -(-NM // G), 4 if fp32 else 8, np.float32 if fp32 else np.float64
    own = buf[:G * NC].view(np.int8).reshape(G, NC)
    assert sorted(own[own >= 0].tolist()) == list(range(N))
    rows = buf[off_row:off_row + 4 * (n_row + 2) * G].view(np.uint32).reshape(-1, G)
    jac = buf[off_jac:off_jac + 4 * (n_jac + 2) * G].view(np.uint32).reshape(-1, G)
    to = buf[off_to:off_coef].copy()
    coef = buf[off_coef:off_coef + 8 * (3 + nr)].view(np.float64)
    w = np.append(rng.standard_normal(nr), 0.0)
    part = np.concatenate([[0.0, 1.0, -1.0, 0.0], rng.standard_normal(nr * (nin_max + 2))]).astype(ft)
    # references: one reaction at a time, each product rounded before its add on both sides
    f = np.zeros(N)
    M = np.zeros((N, N), ft)
    P = lambda kind, r: part[4 + kind * nr + r]
    for r in range(nr):
        for i in ins[r]:
            f[i] -= w[r]
        for o in outs[r]:
            f[o] += w[r]
        if energy:
            f[ns] += -dH[r] * w[r]
        for c, col in list(enumerate(ins[r])) + ([(nin_max, ns)] if energy else []):
            for i in ins[r]:
                M[i, col] += P(c, r)
            for o in outs[r]:
                M[o, col] -= P(c, r)
            if energy:
                M[ns, col] += P(nin_max + 1, r) * P(c, r)
    M += np.eye(N, dtype=ft)
    gotf, gotM, seen = np.full(N, np.nan), np.full((N, N), np.nan, ft), 0
    for l in range(G):
        s, k = 0.0, 0
        for u in rows[:n_row, l].tolist():
            s += coef[(u >> 16) // 8] * w[(u & 0x3fff) // 8]
            if u & 0x8000:
                gotf[own[l, k]] = s
                s, k = 0.0, k + 1
        v, k = ft(0), 0
        for u in jac[:n_jac, l].tolist():
            v = ft(v + part[((u >> 16) & 0x3fff) // rb] * part[(u & 0x3fff) // rb])
            if u & 0x8000:
                at = int(to[k * G + l])
                gotM[at // LD, at % LD] = v
                v, k, seen = ft(0), k + 1, seen + 1
    assert seen == N * N
    assert np.array_equal(gotf, f) and np.array_equal(gotM, M)
    # the two steps past the end add nothing: rate 0 (or partial 0) times coefficient 0
    assert np.all(rows[n_row:] == 8 * nr) and np.all(jac[n_jac:] == 0)


def test_networks_beyond_the_programs_are_left_to_the_lane_kernels(probe):
    tab, buf, nr = np.zeros(9, np.int32), np.zeros(16, np.uint8), 401
    one, sp, dH = np.ones(nr, np.int32), np.zeros((nr, 3), np.int32), np.zeros(nr)
    p = lambda a: ctypes.c_void_p(a.ctypes.data)
    for N, n in ((4, 401), (17, 10), (4, 0)):
        assert probe.probe(N, N, n, 0, p(one), p(one), p(sp), p(sp), p(dH), 0, 8, p(tab), p(buf), buf.size) == -1


@pytest.mark.parametrize("ns,energy,nr,LD,T", [(1, 0, 1, 4, 32), (16, 1, 75, 20, 32), (31, 1, 400, 36, 32), (32, 0, 90, 36, 32),
                                               (33, 1, 500, 36, 128), (95, 1, 64, 100, 128)])
def test_team_program_replays_the_row_lists(probe, ns, energy, nr, LD, T):
    rng = np.random.default_rng(ns + nr)
    N = ns + energy
    ins, outs = _network(rng, ns, nr)
    nin_max = max(map(len, ins))
    lists = [[] for _ in range(ns)]
    for r in range(nr):
        for i in ins[r]:
            lists[i].append(r << 8 | 0xff)
        for o in outs[r]:
            lists[o].append(r << 8 | 1)
    ity = np.int32
    nin, pin = np.array([len(i) for i in ins], ity), np.array([(i + [-1] * 3)[:3] for i in ins], ity)
    rp, re = np.cumsum([0] + [len(l) for l in lists]).astype(ity), np.array(sum(lists, []) + [0], ity)
    prog = np.zeros(1 << 18, np.uint32)
    p = lambda a: ctypes.c_void_p(a.ctypes.data)
    got = probe.team(ns, nr, energy, p(nin), p(pin), p(rp), p(re), LD, T, p(prog), prog.size)
    assert got > 0
    steps, total = got >> 16, got & 0xffff
    assert steps % 8 == 0 and total == steps + 8
    prog = prog[:total * T].reshape(total, T)
    zero = nr * (nin_max + energy)
    D = np.append(rng.standard_normal(zero), 0.0).astype(np.float32)
    J = np.zeros((ns, N), np.float32)     # one list entry after the other
    for s in range(ns):
        for ent in lists[s]:
            r, sg = ent >> 8, np.float32(-1 if ent & 0x80 else 1)
            for c, col in list(enumerate(ins[r])) + ([(nin_max, ns)] if energy else []):
                J[s, col] += sg * D[c * nr + r]
    gotJ, seen = np.full((ns, N), np.nan, np.float32), 0
    for t in range(T):
        v = np.float32(0)
        for u in prog[:steps, t].tolist():
            d = D[u & 0x3fff]
            v = np.float32(v + (-d if u >> 31 else d))
            if u >> 28 & 1:
                at = u >> 14 & 0x3fff
                gotJ[at % LD, at // LD] = v
                v, seen = np.float32(0), seen + 1
    assert seen == ns * N and np.array_equal(gotJ, J)
    assert np.all(prog[steps:] == zero)


def test_team_program_is_left_out_beyond_its_indices(probe):
    nr = 8200     # 2 partials each: more than 14 bits hold
    one, sp, prog = np.ones(nr, np.int32), np.zeros((nr, 3), np.int32), np.zeros(1, np.uint32)
    rp, re = np.zeros(3, np.int32), np.zeros(1, np.int32)
    p = lambda a: ctypes.c_void_p(a.ctypes.data)
    assert probe.team(2, nr, 1, p(one), p(sp), p(rp), p(re), 4, 32, p(prog), 1) == 0
