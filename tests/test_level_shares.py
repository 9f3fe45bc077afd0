"""The equal shares of the OPF's block updates (level_shares; host code, no device) against the update lists they
deal out: every update of every target once and in one place, targets cut between groups only on levels
of one column, their slots within what the kernel has room for."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2512_08465_gb300 import build, synth

HARNESS = r"""
#include "symbolic.cu"
static Symbolic S;
extern "C" int shares_of(int n, int m, const int* f, const int* t, int ref, int groups) {
    S = Symbolic();
    if (!symbolic_analysis(n, std::vector<int>(f, f + m), std::vector<int>(t, t + m), ref, S).empty()) return -1;
    level_shares(groups, S);
    return S.nlevels;
}
extern "C" int get(const char* name, int* out) {
    const std::string k = name;
    const std::vector<int>& v = k == "lev_ptr" ? S.lev_ptr : k == "lev_col" ? S.lev_col : k == "tgt_ptr" ? S.tgt_ptr :
        k == "tgt" ? S.tgt : k == "upd_ptr" ? S.upd_ptr : k == "upd_a" ? S.upd_a : k == "upd_b" ? S.upd_b :
        k == "rn_ptr" ? S.rn_ptr : k == "rn_first" ? S.rn_first : k == "rn_end" ? S.rn_end : k == "sh_a" ? S.sh_a :
        k == "sh_b" ? S.sh_b : k == "off_ptr" ? S.off_ptr : k == "off" ? S.off : k == "Lcol" ? S.Lcol : S.Lrow;
    if (out) std::copy(v.begin(), v.end(), out);
    return (int)v.size();
}
"""
NAMES = ("lev_ptr lev_col tgt_ptr tgt upd_ptr upd_a upd_b rn_ptr rn_first rn_end sh_a sh_b off_ptr off Lcol").split()


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("shares")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", build.SRC, "-I", build.INC, str(src),
                    "-o", str(so)], check=True)
    return ctypes.CDLL(os.fspath(so))


def _shares(lib, net, groups):
    f, t = (np.ascontiguousarray(a, np.int32) for a in (net.f, net.t))
    ptr = ctypes.POINTER(ctypes.c_int)
    levels = lib.shares_of(net.n_bus, f.size, f.ctypes.data_as(ptr), t.ctypes.data_as(ptr), int(net.ref_bus), groups)
    out = {}
    for k in NAMES:
        out[k] = np.empty(lib.get(k.encode(), None), np.int32)
        lib.get(k.encode(), out[k].ctypes.data_as(ptr))
    return levels, out


NETS = [("tree", lambda: synth.make_network(9, 8, 3, 4, 0, seed=1)), ("14", lambda: synth.make_network(14, 20, 5, 11, 1, seed=3)),
        ("57", lambda: synth.make_network(57, 80, 9, 40, 0, seed=3)), ("118", synth.case118),
        ("300", lambda: synth.case_scaled(300, seed=300))]


@pytest.mark.parametrize("groups", [2, 4, 8, 16])
@pytest.mark.parametrize("make", [m for _, m in NETS], ids=[k for k, _ in NETS])
def test_every_update_is_dealt_once(lib, make, groups):
    net = make()
    n = net.n_bus
    levels, S = _shares(lib, net, groups)
    assert S["rn_ptr"].size == levels * groups + 1 and S["rn_first"].size == S["rn_end"].size + 1
    assert (np.diff(S["rn_ptr"]) >= 0).all() and (np.diff(S["rn_first"]) > 0).all()     # no empty run
    assert S["rn_first"][-1] == S["sh_a"].size == S["upd_a"].size                      # nothing twice
    cut_targets = 0
    for h in range(levels):
        targets = S["tgt"][S["tgt_ptr"][h]:S["tgt_ptr"][h + 1]]
        columns = S["lev_ptr"][h + 1] - S["lev_ptr"][h]
        one = columns == 1 and groups > 2
        off = S["off"].reshape(-1, 4)[S["off_ptr"][h]:S["off_ptr"][h + 1]]
        owner = {}                                                                     # slot -> target
        for q, col, first, slots in off:
            assert col == S["Lcol"][q]
            for p in range(first, first + slots):
                assert p not in owner
                owner[p] = n + q
        assert sorted(owner) == list(range(len(owner))) and len(owner) <= 2 * groups
        assert one or not owner
        assert sorted(n + q for q in off[:, 0]) == sorted(t for t in targets if t >= n)
        dealt, sizes = {int(t): [] for t in targets}, []
        for g in range(groups):
            r0, r1 = S["rn_ptr"][h * groups + g], S["rn_ptr"][h * groups + g + 1]
            if one and g < 2:
                assert r1 - r0 <= 1
            sizes.append(int(S["rn_first"][r1] - S["rn_first"][r0]))
            for r in range(r0, r1):
                end = int(S["rn_end"][r])
                tg = owner.pop(-1 - end) if end < 0 else end
                if one:                                # the pivot is for groups 0 and 1, the rest for the others
                    assert (tg < n) == (g < 2)
                u = slice(S["rn_first"][r], S["rn_first"][r + 1])
                dealt[tg] += list(zip(S["sh_a"][u], S["sh_b"][u]))
        assert not owner                               # every slot that is read was written
        cut_targets += sum(s > 0 for s in off[:, 3])
        for tg, got in dealt.items():                  # in the order of the target's own list
            u = slice(S["upd_ptr"][tg], S["upd_ptr"][tg + 1])
            assert got == list(zip(S["upd_a"][u], S["upd_b"][u])), (h, tg)
        if one:                                        # equal shares, to one update
            for part in (sizes[:2], sizes[2:]):
                assert max(part) - min(part) <= 1
    if net.n_bus >= 118 and groups > 2:
        assert cut_targets > 0
