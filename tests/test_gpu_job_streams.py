"""run_ftlm's small sectors share the device over side streams: the results are those of
the sectors one after another, bit for bit, on the default and on another stream, with
sectors above the side-by-side size in the mix, and the call leaves its stream ordered
after all of them."""
import pytest
import torch

from paper_2605_26261_gb300 import ftlm, inputs

pytestmark = pytest.mark.gpu


def one_by_one(N, bonds, R, M, T, **kw):
    res = []
    for tz in ftlm.computed_two_sz(N):
        with ftlm.Basis(N, tz, bonds) as b:
            res.append((tz, b.dim, ftlm.lanczos(b, R, M, keep_coeffs=True, **kw)))
            torch.cuda.synchronize()
    return ftlm.thermo(res, T, R, M), res


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("side_bytes", [None, 1 << 17, 0])
def test_side_by_side_sectors_match_one_by_one(cuda_dev, dtype, side_bytes, monkeypatch):
    if side_bytes is not None:  # some, or all, sectors above the limit
        monkeypatch.setattr(ftlm, "SIDE_BYTES", side_bytes)
    N, R, M = 15, 5, 25
    bonds = inputs.random_graph(N, seed=2)
    T = torch.logspace(-1, 1, 20, dtype=torch.float64, device=cuda_dev)
    ref, secs = one_by_one(N, bonds, R, M, T, seed=4, dtype=dtype)
    for stream in (None, torch.cuda.Stream()):
        if stream is not None:
            stream.wait_stream(torch.cuda.current_stream())
        got = ftlm.run_ftlm(N, bonds, R, M, T, seed=4, dtype=dtype, keep_coeffs=True, stream=stream)
        (stream or torch.cuda.current_stream()).synchronize()  # nothing else is waited for
        for k in ("E", "C", "chi", "mag"):
            assert torch.equal(got[k], ref[k]), k
        assert [s[:2] for s in got["sectors"]] == [s[:2] for s in secs]
        for a, b in zip(got["sectors"], secs):
            for k in ("alpha", "beta", "theta", "weight", "m_eff"):
                assert torch.equal(a[2][k], b[2][k]), k


def test_bad_sector_raises_and_leaves_the_device_usable(cuda_dev):
    T = torch.ones(1, dtype=torch.float64, device=cuda_dev)
    for bad in ([0, 3], [12], [2, 99]):
        with pytest.raises(ftlm.FtlmError) as e:
            ftlm.run_ftlm(10, inputs.ring(10), 2, 10, T, sectors=bad)
        assert e.value.status == ftlm.FTLM_EINVAL
    ok = ftlm.run_ftlm(10, inputs.ring(10), 2, 10, T, sectors=[0, 2])
    assert torch.isfinite(ok["E"]).all()


@pytest.mark.parametrize("sectors", [[0, 8, 14, 18, 20, 26],  # 10.4 M rows; 3.1 M; 0.23 M and fewer, side by side
                                     [14],                     # one sector, workspace below SIDE_BYTES
                                     [8]])                     # one sector, workspace above
def test_jobs_on_two_streams_without_a_wait(cuda_dev, sectors):
    N, R, M = 26, 8, 10
    bonds = inputs.random_graph(N, seed=3)
    T = torch.logspace(-1, 1, 20, dtype=torch.float64, device=cuda_dev)
    want = []
    for seed in (1, 2):
        want.append(ftlm.run_ftlm(N, bonds, R, M, T, seed=seed, sectors=sectors, keep_coeffs=True))
        torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for seed, s in zip((1, 2), streams):
        got.append(ftlm.run_ftlm(N, bonds, R, M, T * 1.0, seed=seed, sectors=sectors, keep_coeffs=True, stream=s))
        # the caller's next allocations do not share memory with the queued job
        junk = [torch.full((n << 20,), 255, dtype=torch.uint8, device=cuda_dev) for n in (700, 220, 220, 64, 16, 16, 4)]
        del junk
    torch.cuda.synchronize()
    for g, w in zip(got, want):
        for k in ("E", "C", "chi", "mag"):
            assert torch.equal(g[k], w[k]), k
        for a, b in zip(g["sectors"], w["sectors"]):
            for k in ("alpha", "beta", "theta", "weight", "m_eff"):
                assert torch.equal(a[2][k], b[2][k]), (a[0], k)
