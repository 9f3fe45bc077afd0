"""How much scratch the small-signal blocks take: four per SM where that stays within bounds, else two; and a
device short of memory gets the records all the same."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2512_08465_gb300 import cs, synth  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _net(n_bus):
    return synth.case118() if n_bus == 118 else synth.case_scaled(n_bus, seed=n_bus, levels=(0.6,), vband=(0.85, 1.15))


# 118 buses: within the OPF's scratch; 300: 1.35 GB for four, 0.74 GB budgeted; 520: 3.9 GB for four
@pytest.mark.parametrize("n_bus,budget,blocks", [(118, 0, 4), (118, 64 << 30, 4), (300, 0, 4), (300, 64 << 30, 2),
                                                 (520, 0, 2)])
def test_blocks_per_sm(n_bus, budget, blocks):
    ctx = cs.Context(hbm_budget=budget)
    assert ctx.network_stats(ctx.load_network(_net(n_bus)))["dyn_ctas_per_sm"] == blocks
    ctx.close()


def test_short_device_memory():
    """600 pairs of 300 buses need 1.35 GB of scratch with four blocks per SM and 0.74 GB with two; with 1 GB free
    every record is as with all the memory, bit for bit (they do not depend on the shape)."""
    net = _net(300)
    ii, jj = synth.all_pairs(net.n_elem)
    sel = np.random.default_rng(5).choice(ii.size, 600, replace=False)
    ei, ej = torch.as_tensor(ii[sel], device=DEV), torch.as_tensor(jj[sel], device=DEV)
    got = []
    for short in (False, True):
        ctx = cs.Context()
        nid = ctx.load_network(net)                  # (the base case: every kernel has run once)
        out = ctx.alloc_results(600, DEV)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        rest = torch.empty(torch.cuda.mem_get_info()[0] - (1 << 30) if short else 1, dtype=torch.uint8, device=DEV)
        ctx.evaluate_device(nid, 0, ei, ej, out)
        ctx.sync()
        got.append({k: v.cpu().numpy() for k, v in out.items()})
        ctx.close()
        del rest
        torch.cuda.empty_cache()
    for k in got[0]:
        np.testing.assert_array_equal(got[0][k], got[1][k], err_msg=k)
