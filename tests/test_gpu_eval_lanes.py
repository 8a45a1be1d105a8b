"""The throughput FP32 evaluation (a lane per chromosome, a warp per pilot)
against the kernels that small calls take, bit for bit, and against the
oracle: the same population evaluated in one large call and in small chunks.
Shapes at the edges of its column shares (12, 13, 24, 25, 48 columns), of the
load widths (K = 16, 17), of the row alignments the decoders tell apart, and
column-tiled tables (16, 8 and 4 columns; whole inverses and chunks of cells);
ragged counts; populations off 16-byte alignment."""
import numpy as np
import pytest

from paper_2511_20511_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WORDS = 12_500_000  # table words from which one call takes the throughput kernel


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_20511_gb300 import binding, build

    build.build()
    binding.lib()
    return binding


def _instance(L, K):
    if L > 61:  # beyond the layouts: log-normal gains
        rng = np.random.default_rng(L * 64 + K)
        b = np.exp(rng.normal(-20.0, 2.0, size=(L, L, K)))
        b[np.arange(L), np.arange(L)] *= 50.0
        return b.astype(np.float32).astype(np.float64)
    full = next(r for r in (7, 19, 37, 61) if r >= L)
    inst = inputs.instance(full, K, seed=L * 64 + K, dtype=np.float32)
    return np.ascontiguousarray(inst["beta"][:L, :L])


def _cfg(B, L, K, mode, obj):
    return B.pa_config_default(L, K, mode=mode, objective=obj, M=256.0)


def _eval(B, ctx, pop):
    fit = torch.empty(pop.shape[0], dtype=torch.float32, device="cuda")
    B.pa_eval_population(ctx, pop, fit)
    return fit


def _chunks(B, ctx, pop, step):
    return torch.cat([_eval(B, ctx, pop[i:i + step].contiguous().clone())
                      for i in range(0, pop.shape[0], step)])


@pytest.mark.parametrize("L,K", [(2, 2), (7, 4), (12, 16), (13, 7), (19, 10), (19, 16), (24, 5),
                                 (25, 16), (37, 13), (37, 16), (48, 3), (19, 17), (13, 32), (7, 40),
                                 (33, 20), (61, 12), (53, 20), (49, 9), (61, 32), (49, 17),
                                 (61, 56), (150, 27), (120, 32)])
@pytest.mark.parametrize("mode,obj", [(1, 0), (0, 0), (1, 1)])
def test_large_call_equals_small_calls(B, oracle, L, K, mode, obj):
    beta = _instance(L, K)
    n = max(WORDS // (L * L * K) + 1, 50001) | 1  # odd: a ragged last tile
    cfg = _cfg(B, L, K, mode, obj)
    ctx = B.pa_create(cfg, beta)
    try:
        pop = inputs.random_population_torch(n, L, K, 5, "cuda")
        fit = _eval(B, ctx, pop)
        step = min(1000, max(1, WORDS // (2 * L * L * K)))
        assert torch.equal(fit, _chunks(B, ctx, pop, step))
        raw = torch.zeros(n * L * K + 16, dtype=torch.uint8, device="cuda")
        view = raw[3:3 + n * L * K].view(n, L, K)
        view.copy_(pop)
        assert torch.equal(fit, _eval(B, ctx, view))
        idx = np.r_[0:40, n - 40:n]
        sp = oracle.sinr_params(cfg.mode, cfg.tau_p, cfg.M, cfg.rho, cfg.sigma2, objective=obj)
        ref = oracle.fitness_batch(beta, pop.cpu().numpy()[idx], sp)
        got = fit.cpu().numpy()[idx].astype(np.float64)
        assert (np.abs(got - ref) / ref).max() <= 1e-5
    finally:
        B.pa_destroy(ctx)


def test_invalid_rows_stay_their_own(B):
    L, K, n = 19, 10, 8192
    ctx = B.pa_create(_cfg(B, L, K, 1, 0), _instance(L, K))
    try:
        pop = inputs.random_population_torch(n, L, K, 6, "cuda")
        good = _eval(B, ctx, pop)
        bad = pop.clone()
        hit = [0, 31, 32, 4097, n - 1]
        for i, h in enumerate(hit):
            bad[h, (5 * i) % L, i % K] = (10, 127, 128, 200, 255)[i]
            bad[h, L - 1, :] = i
        got = _eval(B, ctx, bad)
        keep = torch.ones(n, dtype=torch.bool)
        keep[hit] = False
        assert torch.equal(got.cpu()[keep], good.cpu()[keep])
    finally:
        B.pa_destroy(ctx)


def test_noalloc_large_call(B):
    L, K, n = 19, 10, 20001
    beta = _instance(L, K)
    cfg = _cfg(B, L, K, 1, 0)
    ctx = B.pa_create(cfg, beta)
    try:
        pop = inputs.random_population_torch(n, L, K, 7, "cuda")
        fit = torch.empty(n, dtype=torch.float32, device="cuda")
        B.pa_eval_population_noalloc(cfg, beta, pop, fit)
        assert torch.equal(fit, _eval(B, ctx, pop))
    finally:
        B.pa_destroy(ctx)
