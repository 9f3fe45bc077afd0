"""State orders around the register pass of the Hessenberg reduction in global memory (384 columns: longer
rows make a second pass over memory), and the batched Risk Index over several words of its bit rows and at the
sample counts and element counts where another kernel takes over.

Tolerances are those of the parity suite: eigen statistics 1e-6 in FP64 and 2e-3 on the mixed form's path
without refinement, cost 1e-6 relative; Risk Index exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2512_08465_gb300 import cs, synth  # noqa: E402
from oracle import pipeline, risk  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _run(ctx, nid, ei, ej):
    out = ctx.alloc_results(len(ei), DEV)
    ctx.evaluate_device(nid, 0, torch.as_tensor(np.asarray(ei, np.int32), device=DEV),
                        torch.as_tensor(np.asarray(ej, np.int32), device=DEV), out)
    ctx.sync()
    return {k: v.cpu().numpy() for k, v in out.items()}


# state orders 384, 389 and 479, 5 less with a unit out
@pytest.mark.parametrize("n_gen", [77, 78, 96])
def test_orders_around_384_columns(n_gen):
    net = synth.make_network(100, 150, n_gen, 80, 4, seed=2, levels=(0.3,))
    ei, ej = [-1, 0, net.n_branch + n_gen - 1, 4], [-1, -1, -1, 60]
    refs = [pipeline.evaluate(net, 0, i, j) for i, j in zip(ei, ej)]
    for prec, tol in ((cs.PREC_FP64, 1e-6), (cs.PREC_MIXED, 2e-3)):
        ctx = cs.Context(precision=prec)
        got = _run(ctx, ctx.load_network(net), ei, ej)
        ctx.close()
        for q, ref in enumerate(refs):
            assert int(got["klass"][q]) == ref["klass"] and int(got["opf_iters"][q]) == ref["opf_iters"]
            assert abs(got["cost"][q] - ref["cost"]) <= 1e-6 * abs(ref["cost"])
            assert abs(got["max_re"][q] - ref["max_re"]) <= tol, (prec, q)
            assert abs(got["min_zeta"][q] - ref["min_zeta"]) <= tol, (prec, q)


# 32, 33, 64, 65, 240 and 822 elements: one, two, three, eight and 26 words; 930: more than a tile holds
@pytest.mark.parametrize("n_bus,n_branch,n_gen", [(14, 27, 5), (14, 28, 5), (30, 54, 10), (30, 55, 10),
                                                  (118, 186, 54), (400, 622, 200), (460, 700, 230)])
def test_batched_risk_index_over_words(n_bus, n_branch, n_gen):
    """Every sample equals the single-vector reduction bit for bit, and the oracle's exact sum."""
    net = synth.make_network(n_bus, n_branch, n_gen, n_bus // 2, 0, seed=4, levels=(0.3,))
    E = net.n_elem
    ii, jj = synth.all_pairs(E)
    if E > 100:                                    # complete rows at the ends and in the middle
        keep = np.isin(ii, (0, E // 2, E - 2)) | np.isin(jj, (E // 2, E - 1)) & (ii % 7 == 0)
        ii, jj = ii[keep][:1500], jj[keep][:1500]
    one = np.arange(E)
    ei, ej = np.concatenate([one, ii]), np.concatenate([np.full(E, -1), jj])
    ctx = cs.Context()
    nid = ctx.load_network(net)
    sev = _run(ctx, nid, ei, ej)["severe"]
    S2 = np.zeros((E, E), np.uint8)
    S2[ii, jj] = S2[jj, ii] = sev[E:]
    assert S2.any()
    for n_samples in (15, 16, 17, 32, 33):
        lam = 2.0 ** np.random.default_rng(n_samples).uniform(-30, 10, (n_samples, E))
        d = torch.as_tensor(lam, device=DEV)
        for mode in (cs.RISK_EQ3, cs.RISK_ORDERED):
            R = torch.empty_like(d)
            ctx.risk_index_batch(nid, 0, d, R, mode)
            ctx.sync()
            got = R.cpu().numpy()
            for s in range(n_samples):
                np.testing.assert_array_equal(got[s], ctx.risk_index(nid, 0, lam[s], mode)[0])
        s = n_samples - 1
        np.testing.assert_array_equal(got[s], risk.risk_index(lam[s], sev[:E], S2, risk.ORDERED))
    ctx.close()
