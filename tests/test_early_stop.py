"""The early stop of infeasible OPFs rests on a bound: no interior-point iteration takes z . mu down by more
than 2^29 (a step keeps at least the fraction 5e-5 of every z and of every mu).  The oracle's histories have
to keep it, and none that meets the stop's condition may converge.  On the GPU, counts and classes are the
oracle's at several caps, also where a scenario converges in its last iteration."""
import math

import numpy as np
import pytest

from oracle import grid, opf, pipeline
from paper_2512_08465_gb300 import synth

LOSS, STATE = 30, 100                   # bits: of z . mu per iteration, of the largest state


def _net():
    return synth.make_network(14, 20, 5, 11, 1, seed=3, levels=(0.5,))


INFEASIBLE = [(20, 22), (20, 23), (21, 23), (22, 24)]          # two of the five units out
FEASIBLE = [(-1, -1), (12, 22), (22, -1), (7, 23)]              # 13, 23, 20 and 19 iterations
SEEDS = [(6, 9, 3, 4, 1, s) for s in range(4)] + [(14, 20, 5, 11, 1, s) for s in range(3)]


@pytest.mark.parametrize("nb,nbr,ng,nl,nt,seed", SEEDS)
@pytest.mark.parametrize("load", [0.5, 1.3])
def test_the_bound_holds_in_the_oracle(nb, nbr, ng, nl, nt, seed, load):
    net = synth.make_network(nb, nbr, ng, nl, nt, seed=seed, levels=(load,))
    units = [(-1, -1)] + [(nbr + a, nbr + b) for a in range(ng) for b in range(a + 1, ng)]
    for i, j in units:
        with np.errstate(all="ignore"):
            r = opf.solve(net, grid.make_scenario(net, 0, i, j), trace=True)
        niq = r["z"].size
        zmu = [row[3] / 0.1 * niq for row in r["hist"]]        # gamma = 0.1 z . mu / niq after each step
        for k, (a, b) in enumerate(zip(zmu, zmu[1:])):
            if a > 0 and math.isfinite(a) and math.isfinite(b):
                assert b >= a * 2.0 ** -29, (i, j, k)
                left = 50 - (k + 1)
                if math.frexp(a)[1] > math.frexp(opf.TOL)[1] + STATE + LOSS * left:
                    assert not r["converged"], (i, j, k)


@pytest.mark.gpu
@pytest.mark.parametrize("cap", [10, 20, 23, 50])
def test_counts_are_the_oracle_s(cap):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_08465_gb300 import cs
    net = _net()
    net.opf_max_it = cap
    sc = INFEASIBLE + FEASIBLE
    ei, ej = (torch.tensor([s[q] for s in sc], dtype=torch.int32, device="cuda:0") for q in (0, 1))
    ctx = cs.Context()
    out = ctx.alloc_results(len(sc), "cuda:0")
    ctx.evaluate_device(ctx.load_network(net), 0, ei, ej, out)
    ctx.sync()
    got = {k: v.cpu().numpy() for k, v in out.items()}
    ctx.close()
    for q, (i, j) in enumerate(sc):
        with np.errstate(all="ignore"):
            r = opf.solve(net, grid.make_scenario(net, 0, i, j), max_it=cap)
        assert int(got["opf_iters"][q]) == r["iterations"], (i, j)
        assert (int(got["klass"][q]) == pipeline.OPF_NONCONV) == (not r["converged"]), (i, j)
    assert (got["opf_iters"][:len(INFEASIBLE)] == cap).all()
