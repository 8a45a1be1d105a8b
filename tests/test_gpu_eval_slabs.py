"""Column-tiled evaluations with more than 16 pilots decode at most 256 MB of
inverses at once: calls of several such slabs with a ragged last one against the
same chromosomes in calls of one slab and, around the slabs' edges, in small
calls (another kernel), bit for bit; the device memory a context keeps for them."""
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


def _beta(L, K):
    rng = np.random.default_rng(L * 64 + K)
    return np.exp(rng.normal(-20.0, 1.0, size=(L, L, K))).astype(np.float32).astype(np.float64)


def _eval(B, ctx, pop):
    fit = torch.empty(pop.shape[0], dtype=torch.float32, device="cuda")
    B.pa_eval_population(ctx, pop, fit)
    return fit


# bytes of 32 chromosomes' inverses: 32 pilots x ceil(L/4) words rounded to pairs
@pytest.mark.parametrize("L,K,ntile", [(61, 48, 8), (150, 27, 19)])
def test_several_slabs(B, L, K, ntile):
    tile = 32 * K * 8 * ((L + 7) // 8)
    slab = (256 << 20) // tile * 32
    n = 2 * slab + 1005
    ctx = B.pa_create(B.pa_config_default(L, K, mode=1, M=256.0, rho=1e9, N=32), _beta(L, K))
    try:
        pop = inputs.random_population_torch(n, L, K, 3, "cuda")
        _eval(B, ctx, pop[:64])
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        fit = torch.empty(n, dtype=torch.float32, device="cuda")
        before = torch.cuda.mem_get_info()[0]
        B.pa_eval_population(ctx, pop, fit)
        torch.cuda.synchronize()
        kept = before - torch.cuda.mem_get_info()[0]
        # inverses and tickets, one partial sum per column tile, allocation units
        assert kept <= (256 << 20) + 4 * n * ntile + (16 << 20)
        step = 20001
        for i in range(0, n, step):
            assert torch.equal(_eval(B, ctx, pop[i:i + step].contiguous()), fit[i:i + step])
        for edge in (0, slab, 2 * slab, n):
            a, b = max(0, edge - 20), min(n, edge + 20)
            assert torch.equal(_eval(B, ctx, pop[a:b].contiguous()), fit[a:b])
    finally:
        B.pa_destroy(ctx)


def test_no_memory_for_the_inverses(B):
    """Where the inverses cannot be had the call takes a kernel that needs none,
    again and again, also while its stream is being captured."""
    L, K, n = 61, 32, 1 << 16
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        cfg = B.pa_config_default(L, K, mode=1, M=256.0, rho=1e9, N=32)
        beta = _beta(L, K)
        plain, ctx = B.pa_create(cfg, beta, stream=st), B.pa_create(cfg, beta, stream=st)
        hold = None
        try:
            pop = inputs.random_population_torch(n, L, K, 3, "cuda")
            fit = torch.empty(n, dtype=torch.float32, device="cuda")
            B.pa_eval_population(plain, pop, fit)
            want = fit.clone()
            B.pa_eval_population(ctx, pop[:64], fit[:64])  # its kernel is loaded
            warm = torch.cuda.CUDAGraph()
            st.synchronize()
            with torch.cuda.graph(warm, stream=st):
                B.pa_eval_population(ctx, pop[:64], fit[:64])
            st.synchronize()
            torch.cuda.empty_cache()
            # 128 MB and a little would be needed
            hold = torch.empty(torch.cuda.mem_get_info()[0] - (100 << 20), dtype=torch.uint8,
                               device="cuda")
            for _ in range(2):
                fit.fill_(-1.0)
                B.pa_eval_population(ctx, pop, fit)
                assert torch.equal(fit, want)
            st.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=st):
                B.pa_eval_population(ctx, pop, fit)
            fit.fill_(-1.0)
            graph.replay()
            assert torch.equal(fit, want)
        finally:
            del hold
            st.synchronize()
            B.pa_destroy(ctx)
            B.pa_destroy(plain)
            torch.cuda.empty_cache()
