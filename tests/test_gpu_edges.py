"""Edges of the kernels' tiles against the oracle and the single reductions: state orders around the
windows of the QR sweeps (8 steps in FP64, 12 in FP32, 32 columns) and of the register passes of the
Hessenberg reductions, sample counts around the tile of the batched Risk Index, and infeasible
scenarios that stop early but report the iteration cap.

Tolerances are those of the parity suite: eigen statistics 1e-6 (both forms), cost 1e-6 relative;
Risk Index and integers exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2512_08465_gb300 import cs, synth  # noqa: E402
from oracle import pipeline  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _run(ctx, nid, ei, ej):
    out = ctx.alloc_results(len(ei), DEV)
    ctx.evaluate_device(nid, 0, torch.as_tensor(np.asarray(ei, np.int32), device=DEV),
                        torch.as_tensor(np.asarray(ej, np.int32), device=DEV), out)
    ctx.sync()
    return {k: v.cpu().numpy() for k, v in out.items()}


@pytest.fixture(autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# state orders 5 n_gen - 1 (and 5 less with a unit out): 9, 14, 19 on 6 buses; 29, 34, 39, 49, 69 on 14
@pytest.mark.parametrize("n_gen", [2, 3, 4, 6, 7, 8, 10, 14])
@pytest.mark.parametrize("prec", [cs.PREC_FP64, cs.PREC_MIXED], ids=["fp64", "mixed"])
def test_eigen_screen_at_window_edges(n_gen, prec):
    if n_gen < 6:
        net = synth.make_network(6, 9, n_gen, 4, 1, seed=1, levels=(0.4,))
        ei, ej = [-1, 0, 4, 2], [-1, -1, -1, 7]
    else:
        net = synth.make_network(14, 20, n_gen, 11, 1, seed=3, levels=(0.3,))
        ei, ej = [-1, 0, 4, 9, net.n_branch + n_gen - 1], [-1, -1, -1, 13, -1]
    ctx = cs.Context(precision=prec)
    got = _run(ctx, ctx.load_network(net), ei, ej)
    ctx.close()
    for q in range(len(ei)):
        ref = pipeline.evaluate(net, 0, ei[q], ej[q])
        assert int(got["klass"][q]) == ref["klass"], (q, got["klass"][q], ref["klass"])
        if ref["converged"]:
            assert abs(got["cost"][q] - ref["cost"]) <= 1e-6 * abs(ref["cost"])
        if np.isfinite(ref["max_re"]):
            assert abs(got["max_re"][q] - ref["max_re"]) <= 1e-6, q
            assert abs(got["min_zeta"][q] - ref["min_zeta"]) <= 1e-6, q


# state orders 59, 64, 84, 109 (and 5 less with a unit out) around the blocks of 60 from which the FP32 QR
# runs two sweeps at a time, 48 steps apart
@pytest.mark.parametrize("n_gen", [12, 13, 17, 22])
@pytest.mark.parametrize("prec", [cs.PREC_FP64, cs.PREC_MIXED], ids=["fp64", "mixed"])
def test_two_sweeps_at_a_time(n_gen, prec):
    net = synth.make_network(24, 36, n_gen, 20, 1, seed=5, levels=(0.3,))
    ei, ej = [-1, 0, 4, net.n_branch + n_gen - 1, 9], [-1, -1, -1, -1, 13]
    ctx = cs.Context(precision=prec)
    got = _run(ctx, ctx.load_network(net), ei, ej)
    reruns = ctx.eigen_reruns()
    ctx.close()
    for q in range(len(ei)):
        ref = pipeline.evaluate(net, 0, ei[q], ej[q])
        assert int(got["klass"][q]) == ref["klass"]
        assert abs(got["max_re"][q] - ref["max_re"]) <= 1e-6, q
        assert abs(got["min_zeta"][q] - ref["min_zeta"]) <= 1e-6, q
    assert reruns == 0


@pytest.mark.parametrize("mode", [cs.RISK_EQ3, cs.RISK_ORDERED])
@pytest.mark.parametrize("n_samples", [1, 2, 31, 32, 33, 65])
def test_batched_risk_index_at_tile_edges(n_samples, mode):
    """Every sample equals the single-vector reduction bit for bit; a rate out of range makes
    its sample NaN, leaves the others alone and is reported."""
    net = synth.make_network(14, 20, 5, 11, 1, seed=3, levels=(0.5,))
    ii, jj = synth.all_pairs(net.n_elem)
    one = np.arange(net.n_elem)
    ctx = cs.Context()
    nid = ctx.load_network(net)
    _run(ctx, nid, np.concatenate([one, ii[:200]]), np.concatenate([np.full(one.size, -1), jj[:200]]))
    rng = np.random.default_rng(n_samples)
    lam = 2.0 ** rng.uniform(-30, 10, (n_samples, net.n_elem))
    lam[0, :2] = [2.0 ** -30, 2.0 ** 10]
    d = torch.as_tensor(lam, device=DEV)
    R = torch.empty_like(d)
    ctx.risk_index_batch(nid, 0, d, R, mode)
    ctx.sync()
    got = R.cpu().numpy()
    for s in range(n_samples):
        np.testing.assert_array_equal(got[s], ctx.risk_index(nid, 0, lam[s], mode)[0])
    bad = n_samples // 2
    d[bad, 7] = float("nan")
    ctx.risk_index_batch(nid, 0, d, R, mode)
    with pytest.raises(cs.CSError):
        ctx.sync()
    again = R.cpu().numpy()
    assert np.isnan(again[bad]).all()
    np.testing.assert_array_equal(np.delete(again, bad, 0), np.delete(got, bad, 0))
    ctx.close()


@pytest.mark.parametrize("cap", [1, 20, 50])
def test_infeasible_scenarios_report_the_cap(cap):
    """Two of the five units out: the load cannot be served, the multipliers grow until the iteration
    stops, and the record states the cap, as a full run of it would."""
    net = synth.make_network(14, 20, 5, 11, 1, seed=3, levels=(0.5,))
    net.opf_max_it = cap
    g = net.n_branch
    ei, ej = [g, g, g + 1, g + 2], [g + 2, g + 3, g + 3, g + 4]
    ctx = cs.Context()
    got = _run(ctx, ctx.load_network(net), ei, ej)
    ctx.close()
    np.testing.assert_array_equal(got["klass"], 2)
    np.testing.assert_array_equal(got["opf_iters"], cap)
    assert np.isnan(got["cost"]).all()
