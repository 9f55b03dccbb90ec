"""One slot serving requests of every degree class in turn (the slot's captured
round is pointed at another element kernel between them): each solution is
bitwise what a fresh server gives, and meets its tolerance."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2202_12477_gb300 import hb  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.lib()


def test_one_slot_every_degree_class():
    reqs = [dict(ex=3, ey=2, ez=2, N=N, perturb=0.1, seed=N, rhs_seed=N, lam=0.1, rtol=1e-10)
            for N in (11, 3, 8, 7, 11, 10, 9, 1, 11)]
    ng = [(3 * q["N"] - 1) * (2 * q["N"] - 1) ** 2 for q in reqs]
    srv = hb.Server(4 << 30, max_slots=1, iters_per_launch=4)
    tickets = [srv.submit(**q, keep_x=True) for q in reqs]
    got = [srv.wait(t, n) for t, n in zip(tickets, ng)]
    srv.close()
    for q, n, (res, x) in zip(reqs, ng, got):
        assert res.status == hb.HB_OK and res.rel_res <= 1e-10
        fresh = hb.Server(4 << 30, max_slots=1, iters_per_launch=4)
        _, x1 = fresh.wait(fresh.submit(**q, keep_x=True), n)
        fresh.close()
        assert np.array_equal(x, x1)
