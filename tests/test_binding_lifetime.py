"""Device addresses handed out by the binding keep the context, and so the
memory they point into, alive: a view of a context's resident population is
read after the Context (or Batch) it came from has been dropped.  On the CPU
against a stand-in for the library that records what is destroyed; on a GPU
through torch."""
import ctypes as C

import numpy as np
import pytest

from paper_2511_20511_gb300 import binding as B
from paper_2511_20511_gb300 import inputs


class FakeLib:
    def __init__(self):
        self.live, self.next = set(), 0x1000

    def new(self, out):
        self.next += 0x1000
        self.live.add(self.next)
        C.cast(out, C.POINTER(C.c_void_p))[0] = self.next
        return B.PA_OK

    def pa_create(self, cfg, beta, u, b, stream, out):
        return self.new(out)

    def pa_batch_create(self, n, cfgs, betas, u, b, stream, out):
        return self.new(out)

    def pa_destroy(self, h):
        self.live.remove(h.value)

    pa_batch_destroy = pa_destroy

    def pa_batch_context(self, batch, i, out):
        assert batch.value in self.live
        C.cast(out, C.POINTER(C.c_void_p))[0] = batch.value + 0x10
        return B.PA_OK

    def pa_population_device(self, h, pop, fit):
        C.cast(pop, C.POINTER(C.c_void_p))[0] = h.value + 0x100
        C.cast(fit, C.POINTER(C.c_void_p))[0] = h.value + 0x200
        return B.PA_OK


@pytest.fixture
def fake(monkeypatch):
    f = FakeLib()
    monkeypatch.setattr(B, "lib", lambda: f)
    return f


def _cfg():
    cfg = B.pa_config()
    cfg.L, cfg.K, cfg.N = 2, 2, 4
    return cfg


def test_address_outlives_dropped_context(fake):
    ctx = B.Context(_cfg(), np.ones((2, 2, 2)))
    pop, fit = B.pa_population_device(ctx.handle)
    assert isinstance(pop, int) and pop == 0x2100 and fit == 0x2200
    seen = {pop: 1}
    assert B.pa_population_device(ctx.handle)[0] in seen
    view = {"data": (pop, False)}
    del ctx, pop, fit, seen
    assert len(fake.live) == 1
    del view
    assert not fake.live


def test_dropped_and_closed_contexts_are_destroyed_once(fake):
    ctx = B.Context(_cfg(), np.ones((2, 2, 2)))
    del ctx
    assert not fake.live
    with B.Context(_cfg(), np.ones((2, 2, 2))) as ctx:
        pop = B.pa_population_device(ctx.handle)[0]
    assert not fake.live  # close() frees whatever is still referenced
    ctx.close()
    del ctx, pop
    raw = B.pa_create(_cfg(), np.ones((2, 2, 2)))  # a bare handle stays the caller's
    again = raw.value
    del raw
    assert fake.live == {again}


def test_address_outlives_dropped_batch(fake):
    batch = B.Batch([dict(cfg=_cfg(), beta=np.ones((2, 2, 2)))])
    pop = B.pa_population_device(batch.context(0))[0]
    del batch
    assert len(fake.live) == 1
    del pop
    assert not fake.live


class _View:
    def __init__(self, ptr, shape):
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "|u1", "data": (ptr, False),
                                         "version": 2}


@pytest.mark.gpu
def test_view_of_a_dropped_context_reads_its_population():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_20511_gb300 import build

    build.build()
    inst = inputs.instance(7, 4, seed=1)
    cfg = B.pa_config_default(7, 4, N=32, rho=inst["rho"])
    ctx = B.Context(cfg, inst["beta"], inst["user_xy_mm"], inst["bs_xy_mm"])
    ctx.solve(5)
    want, _, _ = ctx.get_population(with_fitness=False)
    view = torch.as_tensor(_View(B.pa_population_device(ctx.handle)[0], (32, 7, 4)),
                           device="cuda")
    held = ctx.handle.value
    del ctx
    other = B.Context(cfg, inst["beta"], inst["user_xy_mm"], inst["bs_xy_mm"])
    other.solve(9)
    assert other.handle.value != held
    assert (view.cpu().numpy() == want).all()
