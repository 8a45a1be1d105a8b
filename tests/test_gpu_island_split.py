"""The cluster K-means of the island GA with the users split over the CTAs:
labels and pass counts against the oracle, bit for bit, at the sizes where the
split can go wrong -- fewer words of users than CTAs, a partial last word,
members that do not divide by the CTAs, more clusters than one pushed chunk
holds, more than a warp's lanes, odd cluster counts, and every CTA's slice
below a warp."""
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


@pytest.mark.parametrize("N,L,K,C", [(64, 2, 2, 2), (4096, 2, 2, 64), (3723, 4, 2, 33),
                                     (2153, 2, 5, 63), (257, 3, 5, 17), (300, 7, 3, 16),
                                     (1001, 7, 4, 50), (1024, 19, 10, 5), (100, 13, 9, 3),
                                     (128, 37, 16, 40), (70, 61, 32, 7), (999, 2, 64, 9)])
def test_cluster_kmeans_split(B, oracle, N, L, K, C):
    full = next(r for r in (7, 19, 37, 61) if r >= L)
    beta = np.ascontiguousarray(inputs.instance(full, K, seed=1)["beta"][:L, :L])
    cfg = B.pa_config_default(L, K, prec=1, N=N, islands=C, island_iter=25, seed=N + C)
    rng = np.random.default_rng(N)
    base = inputs.random_population(2 * C, L, K, seed=C)
    pop = base[rng.integers(0, 2 * C, size=N)].copy()
    mix = rng.integers(0, N, size=N)  # rows of another member: several passes
    rows = rng.random((N, L)) < 0.3
    pop[rows] = pop[mix][rows]
    ctx = B.pa_create(cfg, beta)
    try:
        dpop = torch.from_numpy(pop).cuda()
        labels = torch.full((N,), -7, dtype=torch.int32, device="cuda")
        for gen in (0, 6):
            passes = B.pa_island_cluster(ctx, dpop, gen, labels)
            want, wpasses = oracle.pop_kmeans(pop, C, 25, cfg.seed, gen)
            assert passes == wpasses
            assert (labels.cpu().numpy() == want).all()
    finally:
        B.pa_destroy(ctx)


@pytest.mark.parametrize("N,L,K,C,E", [(48, 7, 4, 5, 8), (100, 7, 5, 7, 3), (256, 19, 10, 12, 2)])
def test_island_solve_trajectory(B, oracle, N, L, K, C, E):
    """Whole FP64 island solves: the split K-means inside the fused launch, and
    each elite found by its own slot's warp."""
    inst = inputs.instance(L, K, seed=4)
    cfg = B.pa_config_default(L, K, prec=1, mode=1, M=256.0, rho=inst["rho"], N=N, E=E,
                              islands=C, seed=21)
    G = 13
    ctx = B.pa_create(cfg, inst["beta"], inst["user_xy_mm"], inst["bs_xy_mm"])
    try:
        best = np.zeros((L, K), dtype=np.uint8)
        bf = B.pa_solve(ctx, G, best)
        pop = np.zeros((N, L, K), dtype=np.uint8)
        B.pa_get_population(ctx, pop, None)
        sp = oracle.sinr_params(cfg.mode, cfg.tau_p, cfg.M, cfg.rho, cfg.sigma2)
        gp = oracle.ga_params(N, E, cfg.tour, cfg.pc_thresh, cfg.pm_thresh, cfg.seed)
        ref = oracle.solve_islands(inst["beta"], sp, gp, G, C, cfg.recluster, cfg.island_iter,
                                   inst["user_xy_mm"], inst["bs_xy_mm"])
        assert (pop == ref["pop"]).all() and bf == ref["best_fit"]
    finally:
        B.pa_destroy(ctx)
