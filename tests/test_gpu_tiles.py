"""Sizes where the split of a matrix over warps, CTAs and clusters changes: one warp tile is 32 blocks; up to 8 tiles run in
one CTA, up to 768 in a cluster, more in a grid whose tiles stay in shared memory up to ten a warp and stream beyond."""
import numpy as np
import pytest
import torch

from oracle import soar_ref as R
from paper_2605_12245_b200 import api
from paper_2605_12245_b200 import workloads as WL
from tests import parity as P

pytestmark = pytest.mark.gpu


# blocks: a lone one, a ragged tile, 8 and 9 tiles, one tile a warp and one block more, 768 and 769 tiles
@pytest.mark.parametrize("blocks", [1, 31, 33, 8 * 32, 8 * 32 + 1, 256 * 32, 256 * 32 + 1, 768 * 32, 768 * 32 + 1])
@pytest.mark.parametrize("ld_extra", [0, 24])
@pytest.mark.parametrize("cfgkw", [dict(), dict(max_iters=0), dict(max_iters=2, early_stop_rel=0.0, n_dq=2, n_beta=1)])
def test_matrices_at_the_edges_of_the_split(blocks, ld_extra, cfgkw):
    rows = next(r for r in (7, 3, 2, 1) if blocks % r == 0 and blocks >= 4 * r) if blocks > 1 else 1
    w = WL.small_case(rows, 16 * (blocks // rows), blocks, outlier_entry_frac=0.002, outlier_scale=30.0)
    cfg, ref_cfg = P.cfg_pair(**cfgkw)
    gpu = P.run_gpu(w, cfg, w.shape[1] + ld_extra if ld_extra else None)
    P.assert_parity(gpu, R.quantize(w, ref_cfg), mismatch_cap=max(1, blocks // 10000))


@pytest.mark.parametrize("rows", [5920, 5921])   # 23680 tiles of 2048 columns: exactly ten a warp of 148 CTAs, then more
def test_the_last_matrix_that_stays_in_shared_memory_and_the_first_that_does_not(rows):
    w = np.tile(WL.small_case(592, 2048, 5, dist="laplace"), (11, 1))[:rows]
    cfg, _ = P.cfg_pair(max_iters=3)
    one = P.run_gpu(w, cfg)
    (batched, _) = P.run_gpu_batch([w, w[:1]], cfg)      # the streaming kernel of a batch
    assert np.array_equal(one.packed, batched.packed) and np.array_equal(one.scales, batched.scales)
    assert one.alpha == batched.alpha and one.result.iters_run == batched.result.iters_run
    assert one.result.sse == pytest.approx(batched.result.sse, rel=1e-12)


@pytest.mark.parametrize("rows,cols", [(2, 128), (16, 8192), (16, 8224), (200, 2064)])
def test_a_cluster_call_replays_and_repeats(rows, cols):
    """The replay of a captured call, and calls on a workspace that held anything, give what a first call gives."""
    w = WL.small_case(rows, cols, rows + cols)
    cfg, _ = P.cfg_pair()
    W = P.to_device(w)
    want = api.soar_quantize(W, cfg)
    out = api.alloc_buffers(rows, cols, cfg)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        api.soar_quantize(W, cfg, out, side)
    for fill in (0, 255, 170):
        out.workspace.fill_(fill)
        out.packed.zero_()
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out.packed, want.packed) and torch.equal(out.scales, want.scales)
        assert torch.equal(out.alpha, want.alpha)
        assert out.read_result().sse == want.read_result().sse
