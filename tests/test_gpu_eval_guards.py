"""What the large-call FP32 evaluation kernels do outside the ordinary path:
rows that are no permutations (pilots >= K, repeated pilots) leave every other
chromosome's fitness as it was, and copies that never arrive end in
PA_ETIMEOUT within seconds, after which the same context evaluates as before.
The counts are a multiple of the SM count far above those at which these
kernels take over (by estimated times, from one to ten tiles of 32 per SM), so that
other estimates do not move a case to another kernel."""
import time

import numpy as np
import pytest

from paper_2511_20511_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# lanes: row loads of 1, 8 and 4 bytes' alignment, float2 and scalar rows;
# column tiles; chunks of cells: 16-, 4- and 1-byte row loads, 16 and 8 columns
LANES = [(19, 10), (19, 8), (19, 16), (37, 13), (19, 24)]
TILED = [(61, 12), (61, 16)]
CHUNK = [(61, 32), (61, 28), (49, 17), (61, 56)]


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_20511_gb300 import binding, build

    build.build()
    binding.lib()
    return binding


def _beta(L, K):
    rng = np.random.default_rng(L * 64 + K)
    return np.exp(rng.normal(-20.0, 1.0, size=(L, L, K))).astype(np.float32).astype(np.float64)


def _count(L, K):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return (64 if L <= 37 else 2) * 32 * sms + 5  # a ragged last tile


def _eval(B, ctx, pop):
    fit = torch.empty(pop.shape[0], dtype=torch.float32, device="cuda")
    B.pa_eval_population(ctx, pop, fit)
    return fit


@pytest.mark.parametrize("L,K", LANES + TILED + CHUNK)
@pytest.mark.parametrize("shift", [0, 3])
def test_invalid_rows_stay_their_own(B, L, K, shift):
    n = _count(L, K)
    ctx = B.pa_create(B.pa_config_default(L, K, mode=1, M=256.0, rho=1e9), _beta(L, K))
    try:
        raw = torch.zeros(n * L * K + 16, dtype=torch.uint8, device="cuda")
        bad = raw[shift:shift + n * L * K].view(n, L, K)
        bad.copy_(inputs.random_population_torch(n, L, K, 6, "cuda"))
        good = _eval(B, ctx, bad)
        hit = [0, 31, 32, 4097, n - 6, n - 1]
        for i, h in enumerate(hit):
            bad[h, (5 * i) % L, i % K] = (K, 127, 128, 200, 255, 64)[i]
            bad[h, (5 * i + 3) % L, K - 1] = 255
            bad[h, L - 1, :] = i if i < K else 0
        got = _eval(B, ctx, bad)
        keep = torch.ones(n, dtype=torch.bool, device="cuda")
        keep[hit] = False
        assert torch.equal(got[keep], good[keep])
    finally:
        B.pa_destroy(ctx)


# a resident table; column tiles; chunks, added by the last block (2,048) and
# by a reduction
@pytest.mark.parametrize("L,K,n", [(19, 10, None), (19, 24, None), (61, 12, None), (61, 32, 2048),
                                   (61, 32, None)])
def test_stalled_copies_time_out_and_context_recovers(B, L, K, n):
    n = n or _count(L, K)
    beta = _beta(L, K)
    cfg = B.pa_config_default(L, K, mode=B.PA_SINR_FINITE_M, M=256.0, rho=1e9)
    plain = B.pa_create(cfg, beta)
    cfg.flags = B.PA_FLAG_TEST_STALL_COPIES
    ctx = B.pa_create(cfg, beta)
    try:
        pop = inputs.random_population_torch(n, L, K, 11, "cuda")
        want = _eval(B, plain, pop).cpu().numpy()
        rows = pop.cpu().numpy()
        fit = np.zeros(n, dtype=np.float32)
        t0 = time.monotonic()
        with pytest.raises(B.PaError) as e:
            B.pa_eval_population_host(ctx, rows, fit)
        assert e.value.status == B.PA_ETIMEOUT
        # at most seven waits of 2e9 cycles in a row: two for a copy, then one
        # for each buffer in flight (up to five) before the block ends
        assert time.monotonic() - t0 < 8.5
        for _ in range(2):
            B.pa_eval_population_host(ctx, rows, fit)
            assert (fit == want).all()
        small = _eval(B, plain, pop[-40:].contiguous())  # the small calls' kernel
        assert (fit[-40:] == small.cpu().numpy()).all()
    finally:
        B.pa_destroy(ctx)
        B.pa_destroy(plain)
