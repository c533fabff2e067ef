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


@pytest.mark.parametrize("seed", range(6))
def test_the_error_of_a_resident_matrix_keeps_its_bits_beside_one_large_weight(seed):
    """One weight stands a hundred thousand times above the others (4096 and some hundredths), so that a CTA's share of the
    error is a small part of what bounds it.  All rows but one are alike and every warp has nine of them, so that what the CTAs
    round off their shares adds up.  (Both layouts: the last meeting is then one by sums too.)"""
    rows = 9 * 16 * torch.cuda.get_device_properties(0).multi_processor_count    # a tile a row
    row = WL.small_case(1, 512, seed)[0]
    odd = row.copy()
    odd[511] = WL.f32_to_bf16_bits(np.float32([4096.0]))[0]       # the maximum: 2^12, the others about 2^-5
    w = np.tile(row, (rows, 1))
    w[-1] = odd                                    # few additions follow in its lane
    cfg = api.soar_default_cfg(api.PRESET_PAPER, max_iters=2, early_stop_rel=0.0,
                               scale_layout=api.SCALES_LINEAR | api.SCALES_SWIZZLED)
    gpu = P.run_gpu(w, cfg)
    for r in (1, rows // 2, rows - 2):             # equal blocks have equal codes
        assert np.array_equal(gpu.packed[r], gpu.packed[0]) and np.array_equal(gpu.scales[r], gpu.scales[0])
    each = [R.dequant_error(w[r:r + 1], gpu.packed[r:r + 1], gpu.scales[r:r + 1], gpu.alpha) for r in (0, rows - 1)]
    sse, sumsq = ((rows - 1) * each[0][i] + each[1][i] for i in (0, 1))
    # The report is sum W^2 plus (error minus sum W^2), either off by some twenty roundings of 2^-53: nine additions in the lane
    # with the large weight, ten over its CTA's warps, a few over the CTAs.
    assert abs(gpu.result.sse - sse) <= 2.0 ** -47 * sumsq


@pytest.mark.parametrize("rows,cols,ld_extra", [(5003, 2352, 0), (1025, 1040, 8), (127, 6416, 0)])
@pytest.mark.parametrize("cfgkw", [dict(), dict(max_iters=1, early_stop_rel=0.0, n_dq=2, n_beta=1)])
def test_tiled_scales_of_a_resident_matrix_with_ragged_edges(rows, cols, ld_extra, cfgkw):
    """Grids whose CTAs lay their own scales out: rows that end within a tile of 128, block columns that end within four, a last
    warp tile that is not full; the bytes of the row-major layout, and zeroes in the padding."""
    w = WL.small_case(rows, cols, rows)
    w[5, :16] = 0
    lin, _ = P.cfg_pair(**cfgkw)
    both, _ = P.cfg_pair(**cfgkw)
    both.scale_layout = api.SCALES_LINEAR | api.SCALES_SWIZZLED
    tiled, _ = P.cfg_pair(**cfgkw)
    tiled.scale_layout = api.SCALES_SWIZZLED
    W = P.to_device(w, cols + ld_extra)
    want = api.soar_quantize(W, lin)
    r, c = np.meshgrid(np.arange(rows), np.arange(cols // 16), indexing="ij")
    at = (r // 128 * ((cols // 16 + 3) // 4) + c // 4) * 512 + r % 32 * 16 + r % 128 // 32 * 4 + c % 4
    for cfg in (both, tiled):
        out = api.alloc_buffers(rows, cols, cfg)
        out.scales_sw.fill_(255)
        api.soar_quantize(W, cfg, out)
        torch.cuda.synchronize()
        expect = np.zeros(out.scales_sw.numel(), np.uint8)
        expect[at] = want.scales.cpu().numpy()
        assert np.array_equal(out.scales_sw.cpu().numpy(), expect)
        assert torch.equal(out.packed, want.packed) and torch.equal(out.alpha, want.alpha)
        assert out.scales is None or torch.equal(out.scales, want.scales)


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


def test_the_count_of_wide_candidates_of_a_pass_does_not_end_at_32_bits():
    """Blocks below 2^-110 take the binary64 sums for each of the 512 x 16 candidates of the coupled arm, once in the start and
    once a candidate in the iteration: 4.36e9 in one pass.  One matrix alone and in a batch."""
    W = torch.full((1024, 16 * 520), 2.0 ** -115, dtype=torch.bfloat16, device="cuda")
    W[0, :16] = 2.0 ** -90
    cfg = api.soar_default_cfg(api.PRESET_PAPER, max_iters=1, early_stop_rel=0.0, n_dq=16, n_beta=512, beta_step_pct=0,
                               flags=api.FLAG_COUPLED_SCALE)
    one = api.soar_quantize(W, cfg)
    outs = [api.alloc_buffers(*x.shape, cfg) for x in (W, W[:1])]
    api.soar_quantize_batch([W, W[:1]], cfg, outs)
    for o, blocks in ((one, 1024 * 520), (outs[0], 1024 * 520), (outs[1], 520)):
        res = o.read_result()
        assert res.status == 0 and res.iters_run == 1
        assert res.wide_candidates == (blocks - 1) * (1 + 512 * 16)


@pytest.mark.parametrize("preset", [api.PRESET_RTN, api.PRESET_SINGLE_PASS, api.PRESET_PAPER])
def test_the_last_blocks_of_a_row_of_more_than_2_32_weights(preset):
    """A row that ends in a ragged tile beyond weight 2^32, zero but for that tile: it comes out as on its own."""
    tail = P.to_device(WL.small_case(1, 128, 17, outlier_entry_frac=0.05, outlier_scale=10.0))
    W = torch.zeros((1, 2 ** 32 + 128), dtype=torch.bfloat16, device="cuda")
    W[:, 2 ** 32:] = tail
    cfg = api.soar_default_cfg(preset)
    want, got = api.soar_quantize(tail, cfg), api.soar_quantize(W, cfg)
    res = got.read_result()
    assert res.status == 0 and res.zero_blocks == 2 ** 28
    assert torch.equal(got.alpha, want.alpha)
    assert torch.equal(got.packed[:, -64:], want.packed) and torch.equal(got.scales[:, -8:], want.scales)
    assert res.sse == pytest.approx(want.read_result().sse, rel=1e-12)
    if preset == api.PRESET_RTN:
        want, got = api.soar_mx_quantize(tail, n_beta=0), api.soar_mx_quantize(W, n_beta=0)
        assert torch.equal(got.packed[:, -64:], want.packed) and torch.equal(got.scales[:, -4:], want.scales)


# words of four scale bytes of padding below one row: a little under 2^32 and above it, with and without a ragged last word
@pytest.mark.parametrize("nbc", [4 * 33818630, 4 * 33818641 - 1, 4 * 33900000])
def test_padding_of_one_long_row_of_tiled_scales(nbc):
    cfg = api.soar_default_cfg(api.PRESET_RTN, scale_layout=api.SCALES_LINEAR | api.SCALES_SWIZZLED)
    W = torch.zeros((1, 16 * nbc), dtype=torch.bfloat16, device="cuda")
    W[0, ::16 * 1021] = 1.5
    W[0, -1] = -3.0
    out = api.alloc_buffers(1, 16 * nbc, cfg)
    out.scales_sw.fill_(255)
    api.soar_quantize(W, cfg, out)
    assert out.read_result().status == 0 and out.read_result().zero_blocks == nbc - len(range(0, nbc, 1021)) - 1 + ((nbc - 1) % 1021 == 0)
    tiles = out.scales_sw.view(-1, 512)                   # a tile: row 0's four scales, then the padding
    assert torch.equal(tiles[:, :4].reshape(-1)[:nbc], out.scales[0])
    assert not tiles[-1, nbc - 4 * (len(tiles) - 1):4].any()
    assert not any(bool(part[:, 4:].any()) for part in tiles.split(1 << 20))


def test_every_kind_of_launch_replays_from_one_graph():
    """Chained, cluster and cooperative launches behind memsets and each other, captured once, replayed on other inputs."""
    cfg = api.soar_default_cfg(api.PRESET_PAPER, max_iters=2, scale_layout=api.SCALES_LINEAR | api.SCALES_SWIZZLED)
    rtn = api.soar_default_cfg(api.PRESET_RTN, scale_layout=api.SCALES_SWIZZLED)
    big, small = (torch.empty(s, dtype=torch.bfloat16, device="cuda") for s in ((1300, 4096), (70, 4096)))
    h = torch.rand(4096, device="cuda") + 0.5

    def fill(seed):
        for i, W in enumerate((big, small)):
            W.copy_(P.to_device(WL.small_case(W.shape[0], 4096, seed + i)))

    def buffers():
        b = [api.alloc_buffers(*W.shape, c) for W, c in ((big, rtn), (small, rtn), (big, cfg), (small, cfg), (big, cfg), (small, cfg))]
        b.append(api.alloc_buffers(*big.shape, cfg, weighted=True))
        return b, [api.soar_mx_quantize(W) for W in (big, small)], torch.empty(2, dtype=torch.float64, device="cuda")

    fill(1)
    want, got = buffers(), buffers()
    ws = torch.empty(api.soar_batch_workspace_bytes([big, small], want[0][4:6], cfg), dtype=torch.uint8, device="cuda")

    def calls(b, mx, err):
        for o in b + mx:
            o.packed.zero_()
        for W, c, o in ((big, rtn, b[0]), (small, rtn, b[1]), (big, cfg, b[2]), (small, cfg, b[3])):
            api.soar_quantize(W, c, o)
        api.soar_quantize_batch([big, small], cfg, b[4:6], ws)
        api.soar_quantize_weighted(big, h, cfg, b[6])
        for W, o in zip((big, small), mx):
            api.soar_mx_quantize(W, out=o)
        api.soar_dequant_error(big, b[2].packed, b[2].scales, b[2].alpha, out=err)
        api.soar_quantize(big, rtn, b[0])                     # once more behind the error check

    calls(*got)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls(*got)
    for seed in (10, 20):
        fill(seed)
        graph.replay()
        graph.replay()
        calls(*want)
        torch.cuda.synchronize()
        for a, b in zip(want[0] + want[1], got[0] + got[1]):
            assert torch.equal(a.packed, b.packed) and a.read_result().status == b.read_result().status == 0
            assert a.scales is None or torch.equal(a.scales, b.scales)
        for a, b in zip(want[0], got[0]):
            assert torch.equal(a.alpha, b.alpha) and torch.equal(a.scales_sw, b.scales_sw)
        assert got[2].cpu().numpy() == pytest.approx(want[2].cpu().numpy(), rel=1e-12)


# one warp tile is 32 blocks of 16: a lone block, a ragged tile, a whole one, one block more, more tiles than warps of a device
EDGES = [(1, 16), (1, 16 * 31), (2, 16 * 16), (3, 16 * 11), (1, 16 * 4097), (9, 16 * 8421)]


@pytest.mark.parametrize("rows,cols", EDGES)
@pytest.mark.parametrize("ld_extra", [0, 8])
@pytest.mark.parametrize("cfgkw", [dict(max_iters=2), dict(max_iters=1, early_stop_rel=0.0, n_dq=2, n_beta=1)])
def test_weighted_calls_at_the_edges_of_a_tile(rows, cols, ld_extra, cfgkw):
    w = WL.small_case(rows, cols, cols, outlier_entry_frac=0.002, outlier_scale=30.0)
    h = WL.column_weights(cols, rows)
    cfg, ref_cfg = P.cfg_pair(**cfgkw)
    out = api.soar_quantize_weighted(P.to_device(w, cols + ld_extra), torch.from_numpy(h).cuda(), cfg)
    torch.cuda.synchronize()
    gpu = P.GpuOut(out.packed.cpu().numpy(), out.scales.cpu().numpy(), float(out.alpha.cpu()[0]), out.read_result(), out)
    P.assert_parity(gpu, R.quantize(w, ref_cfg, h=h), mismatch_cap=max(1, w.size // 160000))


# A lane has a block of 32: a lone block, a warp's ragged, whole and overfull turn, one CTA's and one more, and two matrices that
# give the lanes of a device (two CTAs of 256 an SM, 75,776; three would be 113,664) a second turn, the last one partly filled.
@pytest.mark.parametrize("rows,cols", [(1, 32), (1, 32 * 15), (2, 32 * 16), (1, 32 * 33), (1, 32 * 257), (1, 32 * 2049), (9, 32 * 4211),
                                       (3, 32 * 18945), (1021, 32 * 149), (3, 32 * 50527)])
@pytest.mark.parametrize("ld_extra", [0, 8])
@pytest.mark.parametrize("cfgkw", [dict(n_beta=0), dict(), dict(n_dq=1, n_beta=5), dict(n_dq=4)])
def test_mxfp4_calls_at_the_edges_of_a_tile(rows, cols, ld_extra, cfgkw):
    w = WL.small_case(rows, cols, cols)
    n = rows * cols // 32
    for i, b in enumerate({0, n // 2, n - 1} if n > 100_000 else ()):      # irregular blocks in the first turn and the last
        part = w.reshape(-1, 32)[b]
        part[:] = 0 if i == 0 else WL.f32_to_bf16_bits(WL.bf16_bits_to_f32(part) * np.float32(2.0 ** (-70 if i == 1 else 75)))
    out = api.soar_mx_quantize(P.to_device(w, cols + ld_extra), **cfgkw)
    torch.cuda.synchronize()
    ref, res = R.mx_quantize(w, **cfgkw), out.read_result()
    bad = (out.packed.cpu().numpy() != ref.packed).reshape(rows, cols // 32, 16).any(axis=2) | (out.scales.cpu().numpy() != ref.scales)
    assert not (bad & ~ref.tie_flags.astype(bool)).any() and bad.sum() <= max(1, bad.size // 10000)
    assert res.sse == pytest.approx(ref.sse, rel=P.SSE_RTOL) and res.sumsq == pytest.approx(ref.sumsq, rel=1e-12)


# a lane has a block of 32: the edges of a warp's 32 blocks, and of a turn of a device's warps over them
@pytest.mark.parametrize("rows,cols", [(1, 32 * 31), (1, 32 * 32), (3, 32 * 11), (1, 32 * 65), (37, 32 * 2048), (41, 32 * 1849)])
@pytest.mark.parametrize("offset,ld_extra", [(0, 0), (8, 0), (0, 8)])    # 32-byte aligned, 16-byte aligned, rows apart
@pytest.mark.parametrize("cfgkw", [dict(n_beta=0), dict()])
def test_mxfp4_irregular_blocks_between_regular_ones(rows, cols, offset, ld_extra, cfgkw):
    """Zero, vanishing and very small or large blocks anywhere in a lane's share, the first and the last ones among them."""
    w = WL.small_case(rows, cols, cols + rows)
    rng = np.random.default_rng(cols)
    blocks = w.reshape(-1, 32)
    n = len(blocks)
    pick = np.unique(np.concatenate([[0, 30, n - 1], rng.integers(0, n, max(4, n // 50))]))
    for i, b in enumerate(pick):
        v = WL.bf16_bits_to_f32(blocks[b]).astype(np.float64)
        v = v * (0.0, 2.0 ** -118, 2.0 ** -70, 2.0 ** 75)[i % 4]
        blocks[b] = WL.f32_to_bf16_bits(v.astype(np.float32))
    ld = cols + ld_extra
    buf = torch.zeros(rows * ld + offset, dtype=torch.bfloat16, device="cuda")
    W = buf[offset:offset + rows * ld].view(rows, ld)[:, :cols]
    W.copy_(P.to_device(w))
    out = api.soar_mx_quantize(W, **cfgkw)
    torch.cuda.synchronize()
    ref, res = R.mx_quantize(w, **cfgkw), out.read_result()
    bad = (out.packed.cpu().numpy() != ref.packed).reshape(rows, cols // 32, 16).any(axis=2) | (out.scales.cpu().numpy() != ref.scales)
    assert not (bad & ~ref.tie_flags.astype(bool)).any() and bad.sum() <= max(1, bad.size // 10000)
    # (the large blocks' terms differ by 2^75 squared from the others': both sides add in binary64)
    assert res.sse == pytest.approx(ref.sse, rel=P.SSE_RTOL) and res.sumsq == pytest.approx(ref.sumsq, rel=1e-12)
    assert res.zero_blocks == int((ref.scales == 0).sum())


@pytest.mark.parametrize("rows,cols", EDGES + [(127, 16 * 5), (129, 16 * 4)])
@pytest.mark.parametrize("ld_extra", [0, 8])
def test_error_check_at_the_edges_of_a_tile(rows, cols, ld_extra):
    w = WL.small_case(rows, cols, cols)
    h = WL.column_weights(cols, rows)
    W, H = P.to_device(w, cols + ld_extra), torch.from_numpy(h).cuda()
    cfg = api.soar_default_cfg(api.PRESET_SINGLE_PASS, scale_layout=api.SCALES_LINEAR | api.SCALES_SWIZZLED)
    b = api.soar_quantize(W, cfg)
    packed, scales, alpha = b.packed.cpu().numpy(), b.scales.cpu().numpy(), float(b.alpha.cpu()[0])
    for layout, sc in ((api.SCALES_LINEAR, b.scales), (api.SCALES_SWIZZLED, b.scales_sw)):
        for e, want in ((api.soar_dequant_error(W, b.packed, sc, b.alpha, layout), R.dequant_error(w, packed, scales, alpha)),
                        (api.soar_dequant_error_weighted(W, H, b.packed, sc, b.alpha, layout),
                         R.dequant_error(w, packed, scales, alpha, h=h))):
            assert e.cpu().numpy() == pytest.approx(np.array(want), rel=1e-11)    # the oracle adds term after term
