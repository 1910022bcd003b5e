"""Plans whose streaming tiles outnumber the H.v tiles: a unit's partial sums take the
larger of the two counts, so no unit's sums reach into its neighbour's vectors."""
import pytest
import torch

from paper_2605_26261_gb300 import ftlm, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile_rows,stream_rows", [(4096, 0), (8192, 256), (1 << 20, 256), (256, 1 << 20)])
def test_streaming_tiles_may_outnumber_hv_tiles(cuda_dev, tile_rows, stream_rows):
    M = 12
    bases = [ftlm.Basis(N, N % 2, inputs.random_graph(N, seed=N)) for N in (15, 16, 17, 18)]
    entries = [(b, 16, 5 + i, 0) for i, b in enumerate(bases)]
    with ftlm.Batch(entries, M, plan=ftlm.BatchPlan(8, 1, tile_rows, stream_rows)) as odd, \
            ftlm.Batch(entries, M, plan=ftlm.BatchPlan(8, 1, 0, 0)) as plain:
        got, want = odd.run(), plain.run()
        torch.cuda.synchronize()
        for g, w in zip(got, want):
            assert torch.equal(g["m_eff"], w["m_eff"])
            # only the order of the FP64 sums of the tiles differs; it enters the FP32
            # vectors through their scales, M times
            scale = w["theta"].abs().max()
            assert (g["theta"] - w["theta"]).abs().max() <= M * 2.0**-22 * scale
    for b in bases:
        b.close()
