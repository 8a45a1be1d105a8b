"""One GA generation through pa_ga_step against the oracle, bit for bit, where
the warp-per-child kernel branches: units of 16, 4 and 1 bytes (L*K and the
buffers' alignment), tournaments that fit a half-warp and longer ones, elites
within and beyond the values a thread caches, no elites, nearly all elites,
ties, and shared memory above the default limit."""
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


@pytest.mark.parametrize("L,K,N,E,tour,shift", [
    (61, 32, 2048, 2, 3, 0), (61, 32, 70, 2, 3, 4), (19, 10, 256, 2, 3, 0), (7, 4, 33, 32, 16, 0),
    (7, 4, 40, 0, 17, 1), (7, 5, 2049, 5, 64, 0), (16, 16, 5000, 64, 2, 0), (3, 1, 9, 1, 1, 0),
    (150, 27, 64, 3, 3, 0)])
@pytest.mark.parametrize("prec", [0, 1])
def test_ga_step(B, oracle, L, K, N, E, tour, shift, prec):
    rng = np.random.default_rng(L * K + N)
    beta = np.exp(rng.normal(-20.0, 1.0, size=(L, L, K)))
    if prec == 0 and L == 150:
        beta = beta.astype(np.float32).astype(np.float64)
    cfg = B.pa_config_default(L, K, prec=prec, N=N, E=E, tour=tour, seed=77,
                              pm_thresh=B.pa_prob_to_thresh(0.4))
    pop = inputs.random_population(N, L, K, seed=N)
    fit = rng.integers(0, max(2, N // 3), size=N).astype(np.float64) + 0.25  # ties
    ctx = B.pa_create(cfg, beta)
    try:
        size = N * L * K
        src = torch.zeros(size + 16, dtype=torch.uint8, device="cuda")
        dst = torch.zeros(size + 16, dtype=torch.uint8, device="cuda")
        p = src[shift:shift + size].view(N, L, K)
        q = dst[shift:shift + size].view(N, L, K)
        p.copy_(torch.from_numpy(pop))
        f = torch.from_numpy(fit).cuda().to(torch.float64 if prec else torch.float32)
        gp = oracle.ga_params(N, E, tour, cfg.pc_thresh, cfg.pm_thresh, cfg.seed)
        for gen in (0, 9):
            B.pa_ga_step(ctx, p, f, gen, q)
            want = oracle.ga_step(pop, fit, gp, gen)
            assert (q.cpu().numpy() == want).all()
        assert dst[shift + size:].sum().item() == 0 and dst[:shift].sum().item() == 0
    finally:
        B.pa_destroy(ctx)
