"""Batched solves whose CTAs hold many members (one CTA per instance: a
half-warp per child, draws behind the evaluation): every instance equals its
solve alone, for tournaments of one, two and four shuffle steps and longer
ones, elites found by one warp and by all, odd populations, both precisions."""
import numpy as np
import pytest

from paper_2511_20511_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_20511_gb300 import binding, build

    build.build()
    binding.lib()
    return binding


@pytest.mark.parametrize("L,K,N,E,tour,prec", [(7, 4, 128, 2, 3, 0), (7, 8, 101, 0, 1, 0),
                                               (7, 5, 70, 9, 5, 0), (7, 4, 99, 8, 8, 0),
                                               (19, 10, 128, 2, 12, 0), (7, 4, 66, 3, 6, 1)])
def test_one_cta_per_instance(B, L, K, N, E, tour, prec):
    n, G = 160, 12  # more instances than SMs: clusters of one CTA
    insts = [inputs.instance(L, K, seed=s, dtype=np.float32) for s in range(8)]
    items = []
    for i in range(n):
        d = insts[i % 8]
        cfg = B.pa_config_default(L, K, prec=prec, mode=1, M=256.0, rho=d["rho"], N=N, E=E,
                                  tour=tour, seed=i, pm_thresh=B.pa_prob_to_thresh(0.2))
        items.append(dict(cfg=cfg, beta=d["beta"], user_xy_mm=d["user_xy_mm"],
                          bs_xy_mm=d["bs_xy_mm"]))
    batch = B.Batch(items)
    assert (batch.groups()[0] == 1).all()
    rows, fit = batch.solve(G)
    for i in (0, 1, 77, n - 1):
        d = items[i]
        with B.Context(d["cfg"], d["beta"], d["user_xy_mm"], d["bs_xy_mm"]) as ctx:
            best, bf = ctx.solve(G)
        assert (rows[i] == best).all() and fit[i] == bf
    batch.close()
