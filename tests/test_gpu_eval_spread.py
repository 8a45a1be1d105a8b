"""Small FP32 evaluations, whose tiles are cut so that they spread over the
SMs: counts at the edges of the tiles against the same chromosomes in one full
call (bit for bit) and the oracle (1e-5, as every FP32 fitness)."""
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


# members per bulk copy: 8, 4, 16, 1; more than 24 cells; more than 16 users
@pytest.mark.parametrize("L,K", [(19, 10), (7, 4), (7, 5), (16, 16), (37, 13), (19, 24), (2, 1)])
@pytest.mark.parametrize("obj", [0, 1])
def test_small_calls(B, oracle, L, K, obj):
    rng = np.random.default_rng(L + K)
    beta = np.exp(rng.normal(-20.0, 1.0, size=(L, L, K))).astype(np.float32).astype(np.float64)
    cfg = B.pa_config_default(L, K, mode=B.PA_SINR_FINITE_M, M=256.0, rho=1e9, objective=obj)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 300 * sms  # every block full
    ctx = B.pa_create(cfg, beta)
    try:
        pop = inputs.random_population_torch(n, L, K, 9, "cuda")
        full = torch.empty(n, dtype=torch.float32, device="cuda")
        B.pa_eval_population(ctx, pop, full)
        for m in (1, 7, 8, 9, sms - 1, sms, sms + 1, 256, 2 * sms + 1, 8 * sms, 8 * sms + 1,
                  24 * sms - 1, 24 * sms + 1, 64 * sms):
            for first in (0, 1):  # 1: rows that need not start at 16 bytes
                fit = torch.full((m + 1,), -1.0, dtype=torch.float32, device="cuda")
                B.pa_eval_population(ctx, pop[first:first + m], fit[:m])
                assert torch.equal(fit[:m], full[first:first + m])
                assert fit[m].item() == -1.0
        sp = oracle.sinr_params(cfg.mode, cfg.tau_p, cfg.M, cfg.rho, cfg.sigma2, objective=obj)
        ref = oracle.fitness_batch(beta, pop[:64].cpu().numpy(), sp)
        assert (np.abs(full[:64].cpu().numpy().astype(np.float64) - ref) / ref).max() <= 1e-5
    finally:
        B.pa_destroy(ctx)
