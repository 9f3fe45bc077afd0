"""Two contexts of networks of different size, each used by its own host thread (distinct contexts are
independent): no call of one may fail because of the other's, and every record is the one that a thread
alone gets, bit for bit."""
import threading

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


def test_batched_risk_index_of_two_threads():
    """25 and 240 elements: tiles of 7 KB and 63 KB of dynamic shared memory, the larger one above the 48 KB
    that a kernel has without opting in."""
    work = []
    for q, net in enumerate((synth.make_network(14, 20, 5, 11, 1, seed=3, levels=(0.5,)), synth.case118())):
        ctx = cs.Context()
        nid = ctx.load_network(net)
        ii, jj = synth.all_pairs(net.n_elem)
        ei = torch.as_tensor(ii[:64], device=DEV)
        ej = torch.as_tensor(jj[:64], device=DEV)
        ctx.evaluate_device(nid, 0, ei, ej, ctx.alloc_results(64, DEV))
        lam = torch.as_tensor(np.random.default_rng(q).uniform(0.01, 1.0, (64, net.n_elem)), device=DEV)
        R, alone = torch.empty_like(lam), torch.empty_like(lam)
        ctx.risk_index_batch(nid, 0, lam, alone)
        ctx.sync()
        work.append((ctx, nid, lam, R, alone))
    start, wrong = threading.Barrier(2), []

    def loop(ctx, nid, lam, R, alone):
        start.wait()
        try:
            for _ in range(3000):
                ctx.risk_index_batch(nid, 0, lam, R)
            ctx.sync()
        except cs.CSError as e:
            wrong.append(str(e))

    threads = [threading.Thread(target=loop, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong
    for ctx, _, _, R, alone in work:
        np.testing.assert_array_equal(R.cpu().numpy(), alone.cpu().numpy())
        ctx.close()
