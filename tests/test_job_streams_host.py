"""Stream order and lifetimes of run_ftlm and lanczos, without a GPU: torch's streams and
caching allocator are stood in for by vector clocks, and every queued call, allocation and
drop is checked against the allocator's contract:

  - a block belongs to the stream that was current when it was allocated; it is free for
    that stream's next work from the moment it is dropped, so every use on another stream
    has to precede the owner's queue by then, or be recorded on the block;
  - a use on another stream has to come after the owner's earlier work (the block's last
    owner), and after the writes it reads.
"""
import math
import types

import numpy as np
import pytest
import torch as real

from paper_2605_26261_gb300 import ftlm


class World:
    def __init__(self):
        self.errors, self.done, self.count = [], {}, 0
        self.held, self.peak, self.built = 0, 0, []  # bytes of tables now and at most; (sector, bytes held before it)
        self.tables = lambda N, two_sz: 1 << 20
        Stream.world, Stream.clocks = self, {}
        self.here = Stream()
        self.current = self.here

    def synchronize(self, *_):
        self.done = {s: n for s, n in Stream.clocks.items()}

    def reached(self, stream, other, n):
        """Whether the work that `stream` queues now runs after operation n of `other`."""
        return other is stream or self.done.get(other, 0) >= n or stream.clock.get(other, 0) >= n

    def tensor(self, shape=(), dtype=None, device=None):
        return Tensor(self, shape, dtype)


class Stream:
    world, clocks = None, {}

    def __init__(self, *_):
        self.clock = {}
        self.world.count += 1
        self.cuda_stream = 1000 + self.world.count
        Stream.clocks[self] = 0

    def op(self):
        Stream.clocks[self] += 1
        self.clock[self] = Stream.clocks[self]
        return Stream.clocks[self]

    def wait_stream(self, other):
        for s, n in {**other.clock, other: Stream.clocks[other]}.items():
            self.clock[s] = max(self.clock.get(s, 0), n)


class Tensor:
    is_cuda = True
    device = "cuda"

    def __init__(self, world, shape, dtype):
        self.world, self.shape, self.owner = world, shape, world.current
        self.start = Stream.clocks[self.owner]
        self.uses, self.recorded, self.written = [], set(), None

    def numel(self):
        return int(np.prod(self.shape))

    def element_size(self):
        return 1

    def record_stream(self, stream):
        self.recorded.add(stream)

    def use(self, stream, n, what, write=False):
        w = self.world
        if not w.reached(stream, self.owner, self.start):
            w.errors.append(f"{what}: before the last use of its block")
        if not write and self.written and not w.reached(stream, *self.written):
            w.errors.append(f"{what}: read before it is written")
        self.uses.append((stream, n, what))
        if write:
            self.written = (stream, n)

    def __del__(self):
        for stream, n, what in self.uses:
            if stream not in self.recorded and not self.world.reached(self.owner, stream, n):
                self.world.errors.append(f"{what}: dropped under queued work")


def make(monkeypatch, needs):
    """ftlm over the stand-ins; needs: workspace bytes of the sector 2 S^z = key."""
    w = World()

    class on:
        def __init__(self, s):
            self.s = s

        def __enter__(self):
            self.was = w.current
            w.current = self.s or w.current

        def __exit__(self, *exc):
            w.current = self.was

    cuda = types.SimpleNamespace(current_stream=lambda *_: w.current, current_device=lambda: 0, stream=on,
                                 Stream=Stream, synchronize=w.synchronize)
    fake = types.SimpleNamespace(
        cuda=cuda, device=lambda *a: a, empty=w.tensor, empty_like=lambda t: w.tensor(t.shape),
        is_tensor=lambda t: isinstance(t, Tensor), uint8=real.uint8, int32=real.int32, float32=real.float32,
        float64=real.float64)

    def as_tensor(a, **kw):
        t = w.tensor(a.shape)
        t.use(w.current, w.current.op(), "T", write=True)
        return t
    fake.as_tensor = as_tensor

    class Basis:
        def __init__(self, N, two_sz, bonds, mode=0, stream=None, wait=True):
            self.two_sz, self.handle, self.dim = two_sz, self, 100
            self.table_bytes = w.tables(N, two_sz)
            w.held += self.table_bytes
            w.peak = max(w.peak, w.held)
            w.built.append((two_sz, w.held - self.table_bytes))
            self.table = w.tensor((1,))
            self.table.owner = stream
            self.table.use(stream, stream.op(), "tables", write=True)
            if wait:
                w.synchronize()

        @classmethod
        def sectors(cls, N, two_sz, bonds, mode=0, stream=None, two_s=1, wait=True):
            return [cls(N, tz, bonds, mode, stream, wait) for tz in two_sz]

        def release(self, stream):
            if self.table:
                w.held -= self.table_bytes
                self.table.owner, self.table = stream, None

        def close(self):
            w.synchronize()
            w.held -= self.table_bytes
            self.table = None

        def __enter__(self):
            return self

        def __exit__(self, *exc):
            self.close()

    def lanczos(handle, R, M, seed, dist, code, work, theta, weight, m_eff, alpha=None, beta=None, stream=None):
        stream = stream or w.current
        n, tz = stream.op(), handle.two_sz
        handle.table.use(stream, n, f"tables {tz}")
        assert work.numel() >= needs[tz]
        work.use(stream, n, f"workspace {tz}", write=True)
        for t in (theta, weight, m_eff, alpha, beta):
            if t is not None:
                t.use(stream, n, f"outputs {tz}", write=True)

    def lanczos_from(handle, R, M, start, code, *args, stream=None):
        start.use(stream or w.current, Stream.clocks[stream or w.current] + 1, "start vectors")
        lanczos(handle, R, M, 0, 0, code, *args, stream=stream)

    def thermo(two_sz, dims, R, M, thetas, weights, m_effs, mirror, g, h, T, E, C, chi, mag, stream=None):
        stream = stream or w.current
        n = stream.op()
        for t in (T, *thetas, *weights, *m_effs):
            t.use(stream, n, "inputs of the sums")
        for t in (E, C, chi, mag):
            t.use(stream, n, "observables", write=True)

    monkeypatch.setattr(ftlm, "torch", fake)
    monkeypatch.setattr(ftlm, "Basis", Basis)
    monkeypatch.setattr(ftlm, "ftlm_lanczos_workspace_bytes", lambda h, R, M, code: needs[h.two_sz])
    monkeypatch.setattr(ftlm, "ftlm_lanczos", lanczos)
    monkeypatch.setattr(ftlm, "ftlm_lanczos_from", lanczos_from)
    monkeypatch.setattr(ftlm, "ftlm_thermo", thermo)
    monkeypatch.setattr(ftlm, "_dtype_code", lambda dt: ftlm.F32)
    return w


SIDE, HELD = 1 << 20, ftlm.SIDE_BYTES + 1  # a workspace beside others; one of a small sector on the job's stream
# N = 30: 2 S^z <= 10 has more rows than run beside others, 2 S^z >= 12 fewer
BRANCHES = {"one side sector": {20: SIDE}, "side by side": {18: SIDE, 20: SIDE, 22: SIDE, 24: SIDE, 26: SIDE, 28: SIDE},
            "held": {14: HELD}, "held and side": {14: HELD, 16: HELD, 20: SIDE, 22: SIDE}, "large": {0: HELD},
            "all": {0: HELD, 2: HELD, 14: HELD, 20: SIDE, 22: SIDE, 24: SIDE}}


@pytest.mark.parametrize("keep", ["all", "observables", "nothing"])
@pytest.mark.parametrize("other", [False, True])
@pytest.mark.parametrize("branch", list(BRANCHES))
def test_run_ftlm_keeps_its_memory_until_it_is_free(monkeypatch, branch, other, keep):
    needs = BRANCHES[branch]
    w = make(monkeypatch, needs)
    stream = ftlm.torch.cuda.Stream() if other else None
    T = w.tensor((5,))
    T.use(w.here, w.here.op(), "T", write=True)  # still being produced on the current stream
    obs = ftlm.run_ftlm(30, ((), (), ()), 8, 10, T, sectors=list(needs), keep_coeffs=True, stream=stream)
    del T
    on = stream or w.here
    for t in (obs["E"], *(t for s in obs["sectors"] for t in s[2].values())):  # all of it joined to the stream
        t.use(on, on.op(), "results on the job's stream")
    if keep == "observables":
        obs = {k: obs[k] for k in ("E", "C", "chi", "mag")}
    if keep == "nothing":
        obs = None
    assert w.errors == []
    if obs:
        w.here.wait_stream(on)
        obs["E"].use(w.here, w.here.op(), "results on the caller's stream")
        obs = None
    assert w.errors == []


def test_host_temperatures(monkeypatch):
    w = make(monkeypatch, {20: SIDE})
    ftlm.run_ftlm(30, ((), (), ()), 8, 10, np.ones(4), sectors=[20], stream=ftlm.torch.cuda.Stream())
    assert w.errors == []


@pytest.mark.parametrize("own_work", [False, True])
@pytest.mark.parametrize("own_start", [False, True])
def test_lanczos_keeps_its_memory_until_it_is_free(monkeypatch, own_work, own_start):
    w = make(monkeypatch, {20: SIDE})
    s = ftlm.torch.cuda.Stream()
    b = ftlm.Basis(30, 20, None, stream=w.here)
    work = w.tensor((SIDE,)) if own_work else None
    start = w.tensor((8, 100)) if own_start else None
    out = ftlm.lanczos(b, 8, 10, start=start, work=work, keep_coeffs=True, stream=s)
    del work, start
    assert w.errors == []
    w.here.wait_stream(s)
    out["theta"].use(w.here, w.here.op(), "outputs on the caller's stream")
    del out
    assert w.errors == []


def test_any_object_with_a_stream_handle(monkeypatch):
    w = make(monkeypatch, {20: SIDE, 22: SIDE})
    wrapped = {}

    def external(handle):
        wrapped[handle] = ftlm.torch.cuda.Stream()
        return wrapped[handle]
    ftlm.torch.cuda.ExternalStream = external
    ftlm.run_ftlm(30, ((), (), ()), 8, 10, np.ones(4), sectors=[20, 22], stream=types.SimpleNamespace(cuda_stream=77))
    assert set(wrapped) == {77} and w.errors == []


@pytest.mark.parametrize("N", [20, 26, 28, 30, 32])
def test_tables_held_at_once(monkeypatch, N):
    """All sectors of a job: the tables held at once stay within TABLE_BYTES (one sector's where
    that is larger), and none is held when a large sector's chains start."""
    two = ftlm.computed_two_sz(N)
    dims = {tz: math.comb(N, (N + tz) // 2) for tz in two}
    w = make(monkeypatch, {tz: 2 * 8 * 4 * d for tz, d in dims.items()})
    lookup = (1 << N) // 4
    w.tables = lambda N, tz: lookup + 4 * dims[tz] if dims[tz] < 1 << 20 else 1 << 18
    ftlm.run_ftlm(N, ((), (), ()), 8, 10, np.ones(4))
    assert w.errors == [] and w.held == 0 and len(w.built) == len(two)
    assert w.peak <= max(ftlm.TABLE_BYTES + lookup, w.tables(N, two[-1]) + (1 << 23))
    for tz, held in w.built:
        if 8 * dims[tz] > ftlm.SIDE_BYTES:
            assert held == 0, tz
