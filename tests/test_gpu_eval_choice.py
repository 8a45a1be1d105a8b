"""The kernel of an FP32 evaluation is chosen by both kernels' estimated times,
so a call may change sides at any count: every count around such changes gives
the fitness that other counts give, bit for bit, and the oracle's (1e-5, as every
FP32 fitness).  Resident tables with float2 and scalar rows, one block per SM,
column tiles with whole inverses and with chunks of cells."""
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


@pytest.mark.parametrize("L,K", [(2, 16), (7, 4), (19, 10), (24, 16), (43, 6), (37, 13), (2, 36),
                                 (7, 40), (19, 24), (61, 4), (61, 12), (61, 20), (61, 32)])
@pytest.mark.parametrize("mode,obj", [(1, 0), (0, 1)])
def test_same_values_at_every_count(B, oracle, L, K, mode, obj):
    rng = np.random.default_rng(L * 64 + K)
    beta = np.exp(rng.normal(-20.0, 1.0, size=(L, L, K)))
    beta[np.arange(L), np.arange(L)] *= 50.0  # own cell: SINRs of order one
    beta = beta.astype(np.float32).astype(np.float64)
    cfg = B.pa_config_default(L, K, mode=mode, M=256.0, rho=1e9, objective=obj)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per_sm = [0.02, 0.2, 0.3, 0.5, 0.75, 1.0] if L == 61 else \
        [0.02, 0.3, 0.7, 1.0, 1.25, 1.5, 2.0, 2.5, 3.5, 5.0, 8.0]
    counts = sorted({1, 31, 33} | {max(1, int(32 * sms * f) - d) for f in per_sm for d in (0, 13)})
    ctx = B.pa_create(cfg, beta)
    try:
        pop = inputs.random_population_torch(counts[-1], L, K, 9, "cuda")
        full = torch.empty(counts[-1], dtype=torch.float32, device="cuda")
        B.pa_eval_population(ctx, pop, full)
        for n in counts:
            fit = torch.full((n + 1,), -1.0, dtype=torch.float32, device="cuda")
            B.pa_eval_population(ctx, pop[:n], fit[:n])
            assert torch.equal(fit[:n], full[:n])
            assert fit[n].item() == -1.0
        sp = oracle.sinr_params(cfg.mode, cfg.tau_p, cfg.M, cfg.rho, cfg.sigma2, objective=obj)
        ref = oracle.fitness_batch(beta, pop[:48].cpu().numpy(), sp)
        assert (np.abs(full[:48].cpu().numpy().astype(np.float64) - ref) / ref).max() <= 1e-5
    finally:
        B.pa_destroy(ctx)
