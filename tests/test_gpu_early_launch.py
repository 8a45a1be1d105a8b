"""Generations whose kernels may start while their predecessor still runs
(evaluation of column tiles, GA step), against the same calls with a
synchronisation behind each one, and captured into a graph: equal bit for bit."""
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


# chunks with tickets; chunks and a reduction; a small call's kernel; no elites
@pytest.mark.parametrize("L,K,N,E", [(61, 32, 2048, 2), (61, 32, 6001, 5), (61, 32, 40, 2),
                                     (61, 32, 2047, 0), (19, 10, 256, 2)])
def test_back_to_back_equals_synchronised(B, L, K, N, E):
    rng = np.random.default_rng(7)
    beta = np.exp(rng.normal(-20.0, 1.0, size=(L, L, K))).astype(np.float32).astype(np.float64)
    st = torch.cuda.Stream()
    cfg = B.pa_config_default(L, K, N=N, E=E, seed=5, pm_thresh=B.pa_prob_to_thresh(0.3))
    with torch.cuda.stream(st):
        start = inputs.random_population_torch(N, L, K, 3, "cuda")
        ctx = B.pa_create(cfg, beta, stream=st)
        try:
            pops = [torch.empty_like(start), torch.empty_like(start)]
            fit = torch.empty(N, dtype=torch.float32, device="cuda")

            def run(gens, sync):
                pops[0].copy_(start)
                for g in range(gens):
                    B.pa_eval_population(ctx, pops[g & 1], fit)
                    if sync:
                        st.synchronize()
                    B.pa_ga_step(ctx, pops[g & 1], fit, g, pops[1 - (g & 1)])
                    if sync:
                        st.synchronize()
                B.pa_eval_population(ctx, pops[gens & 1], fit)
                return pops[gens & 1].clone(), fit.clone()

            want = run(12, True)
            for _ in range(5):
                got = run(12, False)
                assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
            st.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=st):
                got = run(12, False)
            for _ in range(2):
                graph.replay()
                st.synchronize()
                assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
        finally:
            st.synchronize()
            B.pa_destroy(ctx)
