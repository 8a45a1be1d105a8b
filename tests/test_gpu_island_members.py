"""Re-clustering of many members of few users (the cluster K-means with the
members split over its CTAs) against the oracle, bit for bit: on both sides of the
lines between the forms, more clusters than one lane sums at once, odd cluster
counts, a partial last word of users, members that do not divide by the CTAs,
clusters that empty, rows with pilots out of range (read as the last one)."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("N,L,K,C", [(81, 2, 2, 9), (80, 2, 2, 9), (1000, 2, 2, 64), (393, 7, 4, 17),
                                     (392, 7, 4, 17), (841, 7, 4, 8), (840, 7, 4, 8), (4096, 7, 4, 2),
                                     (4001, 5, 5, 63), (2003, 3, 7, 16), (1441, 7, 10, 33),
                                     (4000, 7, 10, 64), (4095, 2, 16, 5)])
def test_members_split(B, oracle, N, L, K, C):
    rng = np.random.default_rng(N + C)
    beta = np.exp(rng.normal(-20.0, 1.0, size=(L, L, K)))
    cfg = B.pa_config_default(L, K, prec=1, N=N, islands=C, island_iter=25, seed=N + C)
    base = np.argsort(rng.random((2 * C, L, K)), axis=-1).astype(np.uint8)
    pop = base[rng.integers(0, 2 * C, size=N)].copy()
    mix = rng.integers(0, N, size=N)  # rows of another member: several passes
    rows = rng.random((N, L)) < 0.3
    pop[rows] = pop[mix][rows]
    pop[N // 2, L - 1, K - 1] = 200
    ctx = B.pa_create(cfg, beta)
    try:
        dpop = torch.from_numpy(pop).cuda()
        labels = torch.full((N,), -7, dtype=torch.int32, device="cuda")
        for gen in (0, 6):
            passes = B.pa_island_cluster(ctx, dpop, gen, labels)
            want, wpasses = oracle.pop_kmeans(np.minimum(pop, K - 1), C, 25, cfg.seed, gen)
            assert passes == wpasses
            assert (labels.cpu().numpy() == want).all()
    finally:
        B.pa_destroy(ctx)
